"""Boxes with odd rows: the kernels that pair cells of neighbouring slabs
(csrc/step_split.cu) against the one-cell kernels, bitwise."""

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


def _cavity(dm, grid, wall, storage, streaming, cpt, rounding=0):
    cav = dm.Cavity(grid, 1e5, wall_type=wall, storage=storage, streaming=streaming, cells_per_thread=cpt,
                    residual_interval=5, rounding=rounding)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, np.float32)[:, None, None, None]
    f = w * (19 * inputs.random_populations(grid, 19, seed=3, spread=0.02))
    cav.set_populations(f, inputs.random_thermal_populations(grid, seed=4))
    return cav


# (an odd and an even number of slabs, two slabs only, rows of 3 cells, rows
# longer than a block, one round of blocks and several)
@pytest.mark.parametrize("grid", [(41, 40, 37), (33, 64, 30), (201, 151, 2), (3, 250, 81), (301, 9, 23), (101, 75, 61)])
@pytest.mark.parametrize("wall,storage,streaming,rounding", [
    (1, 0, 0, 0), (2, 0, 1, 0), (3, 1, 0, 0), (1, 1, 1, 0), (2, 2, 0, 0), (3, 2, 1, 0), (2, 1, 1, 1), (1, 2, 0, 1),
])
def test_bitwise_the_one_cell_kernels(dm, grid, wall, storage, streaming, rounding):
    """Populations, fields and Nu after single steps, graph-replayed intervals
    of an odd length and a broken one; the residual to the rounding of its
    double-float sums."""
    a = _cavity(dm, grid, wall, storage, streaming, 0, rounding)
    b = _cavity(dm, grid, wall, storage, streaming, 1, rounding)
    for n in (1, 4, 15, 2, 1):
        a.step(n)
        b.step(n)
        for p, q in zip(a.populations(), b.populations()):
            assert np.array_equal(p, q)
    for p, q in zip(a.fields(), b.fields()):
        assert np.array_equal(p, q)
    assert a.nusselt(0) == b.nusselt(0) and a.nusselt_flux(1) == b.nusselt_flux(1)
    assert abs(a.residual() - b.residual()) <= 1e-12 * b.residual()
    a.close()
    b.close()


@pytest.mark.parametrize("streaming", [0, 1])
def test_two_slabs_bitwise_the_one_cell_kernels(dm, streaming):
    a = _cavity(dm, (33, 1000, 2), 3, 1, streaming, 0)
    b = _cavity(dm, (33, 1000, 2), 3, 1, streaming, 1)
    for n in (1, 4, 15, 2):
        a.step(n)
        b.step(n)
        for p, q in zip(a.populations(), b.populations()):
            assert np.array_equal(p, q)
    assert abs(a.residual() - b.residual()) <= 1e-12 * b.residual()
    a.close()
    b.close()
