"""Two-buffer cavities of the sizes whose plain steps run in place by twos
(inplace_pays), and the flat numbering of the paired kernels, against the
one-cell two-buffer kernels, bitwise."""

import numpy as np
import pytest

from paper_1511_04633_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1511_04633_gb300 import dmrt
    return dmrt


def _cavity(dm, grid, wall, storage, cpt, K):
    cav = dm.Cavity(grid, 1e5, wall_type=wall, storage=storage, cells_per_thread=cpt, residual_interval=K)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, np.float32)[:, None, None, None]
    f = w * (19 * inputs.random_populations(grid, 19, seed=3, spread=0.02))
    cav.set_populations(f, inputs.random_thermal_populations(grid, seed=4))
    return cav


# the smallest and largest working sets of the rule (433,000 cells FP32, 2.2
# million 16-bit), row tiles and flat blocks, odd rows; odd and even residual
# intervals; then boxes outside the rule for the flat numbering: thin, two
# cells wide, few blocks, a last block with one pair
@pytest.mark.parametrize("grid,wall,storage,K", [
    ((130, 96, 48), 2, 0, 6), ((96, 96, 48), 1, 0, 7), ((114, 96, 100), 3, 0, 2), ((190, 80, 60), 3, 1, 5),
    ((128, 128, 128), 1, 2, 4), ((101, 75, 61), 2, 0, 7), ((129, 90, 80), 3, 1, 6), ((127, 97, 121), 1, 2, 3),
    ((12, 250, 250), 2, 1, 6), ((2, 300, 129), 1, 0, 5), ((36, 36, 36), 3, 2, 4), ((130, 130, 3), 2, 0, 3),
])
def test_bitwise_the_one_cell_kernels(dm, grid, wall, storage, K):
    a = _cavity(dm, grid, wall, storage, 0, K)
    b = _cavity(dm, grid, wall, storage, 1, K)
    for n in (1, 2, 3, 2 * K, K + 3):
        a.step(n)
        b.step(n)
        for p, q in zip(a.populations(), b.populations()):
            assert np.array_equal(p, q)
    for p, q in zip(a.fields(), b.fields()):
        assert np.array_equal(p, q)
    assert a.nusselt(1) == b.nusselt(1)
    assert abs(a.residual() - b.residual()) <= 1e-12 * b.residual()
    # a checkpoint of either continues in the other
    blob = a.save()
    b.load(blob)
    a.step(3)
    b.step(3)
    for p, q in zip(a.populations(), b.populations()):
        assert np.array_equal(p, q)
    a.close()
    b.close()


# shape groups whose plain steps run in place by twos: two chains of mixed
# shapes (the rule's FP32 and 16-bit ranges), one chain, one shape in two
# launches; even and odd residual intervals, graph-replayed and launched singly
@pytest.mark.parametrize("shapes,each,storage,K", [
    ([(50, 41, 33), (70, 64, 30)], 3, 0, 6), ([(50, 41, 33), (70, 64, 30)], 5, 1, 7), ([(36, 50, 42)], 12, 2, 5),
    ([(24, 24, 24)], 70, 1, 2), ([(24, 24, 24), (2, 40, 60)], 65, 2, 4),
])
def test_ensembles_bitwise_the_one_cell_kernels(dm, shapes, each, storage, K):
    cav = [{"grid": shapes[k % len(shapes)], "Ra": 10 ** (3 + 2 * k / 130), "wall": 1 + k % 3}
           for k in range(each * len(shapes))]
    a = dm.Ensemble(cav, storage=storage, residual_interval=K)
    b = dm.Ensemble(cav, storage=storage, residual_interval=K, cells_per_thread=1)
    for n in (1, 2, 3, 2 * K, K + 3):
        a.step(n)
        b.step(n)
        for k in (0, 1, len(cav) // 2, len(cav) - 1):
            for p, q in zip(a.populations(k), b.populations(k)):
                assert np.array_equal(p, q), (n, k)
    assert np.array_equal(np.asarray(a.residual()), np.asarray(b.residual()))
    assert np.array_equal(np.asarray(a.nusselt(1)), np.asarray(b.nusselt(1)))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", [1, 2])
def test_checkpoint_bytes_do_not_depend_on_the_scheme(dm, storage):
    """Header, populations and counter of a saved state: the same bytes
    whichever kernels took the steps and however the calls divided them."""
    grid = (114, 96, 100)
    a = _cavity(dm, grid, 2, storage, 0, 20)
    b = _cavity(dm, grid, 2, storage, 0, 20)
    c = _cavity(dm, grid, 2, storage, 1, 20)
    a.step(7)
    for n in (1, 1, 1, 1, 1, 2):
        b.step(n)
    c.step(7)
    cells = grid[0] * grid[1] * grid[2]
    blobs = [cav.save() for cav in (a, b, c)]
    head = len(blobs[0]) - 16 * cells - 64  # up to the residual's snapshot and sums
    assert all(blob[:head] == blobs[2][:head] for blob in blobs)
    for cav in (a, b, c):
        cav.close()
