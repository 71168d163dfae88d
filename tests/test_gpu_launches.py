"""Seen through a stand-in for the launch call: a launch that the runtime refuses
between the two in-place steps of a two-buffer state (the handle then has no
state, says so, and takes a new one), and the kernels that the autotuner times."""

import pytest

from launch_shim import run_child

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


HELPERS = """
    def status(f, *a):
        try:
            f(*a)
        except dm.DmrtError as e:
            return e.status
        return dm.OK

    start = inputs.random_fields
"""


@pytest.mark.parametrize("grid", [(130, 96, 48), (101, 75, 61)])
def test_cavity(tmp_path, grid):
    run_child(tmp_path, HELPERS + f"""
    grid = {grid}
    fresh = lambda: dm.Cavity(grid, 1e5, wall_type=2, residual_interval=20)
    a, ref = fresh(), fresh()
    for cav in (a, ref):
        cav.init_fields(*start(grid, 3))
        cav.step(4)
    # the first launch refused: nothing has happened
    shim.shim_refuse(1)
    assert status(a.step, 4) == dm.ERR_CUDA
    for p, q in zip(a.fields(), ref.fields()):
        assert np.array_equal(p, q)
    # the second one refused: no state
    shim.shim_refuse(2)
    assert status(a.step, 4) == dm.ERR_CUDA
    for f in (a.fields, a.populations, a.save, lambda: a.nusselt(0), lambda: a.nusselt_flux(0), lambda: a.step(1)):
        assert status(f) == dm.ERR_CUDA
    # a new state, and a loaded one
    blob = ref.save()
    for renew in (lambda cav: cav.init_fields(*start(grid, 5)), lambda cav: cav.load(blob),
                  lambda cav: cav.set_populations(*[np.copy(v) for v in pops])):
        pops = ref.populations()
        shim.shim_refuse(2)
        status(a.step, 4)
        assert status(a.fields) == dm.ERR_CUDA
        shim.shim_refuse(0)
        renew(a)
        renew(ref)
        for cav in (a, ref):
            cav.step(5)
        for p, q in zip(a.populations(), ref.populations()):
            assert np.array_equal(p, q)
    """)


@pytest.mark.parametrize("refused", [2, 3, 4])
def test_ensemble(tmp_path, refused):
    run_child(tmp_path, HELPERS + f"""
    shapes = [(50, 41, 33), (70, 64, 30)]
    cav = [dict(grid=shapes[k % 2], Ra=1e4 * (1 + k), wall=1 + k % 3) for k in range(6)]
    a, ref = [dm.Ensemble(cav, residual_interval=20) for _ in range(2)]
    for e in (a, ref):
        for k in range(6):
            e.init_fields(k, *start(cav[k]["grid"], k))
        e.step(4)
    shim.shim_refuse(1)
    assert status(a.step, 4) == dm.ERR_CUDA
    for k in range(6):
        assert np.array_equal(a.populations(k)[0], ref.populations(k)[0])
    shim.shim_refuse({refused})
    assert status(a.step, 4) == dm.ERR_CUDA
    for f in (lambda: a.fields(1), lambda: a.populations(5), lambda: a.nusselt(0), lambda: a.step(1), lambda: a.autotune(1)):
        assert status(f) == dm.ERR_CUDA
    for k in range(6):
        assert status(a.step, 1) == dm.ERR_CUDA
        for e in (a, ref):
            e.init_fields(k, *start(cav[k]["grid"], 20 + k))
        assert np.array_equal(a.populations(k)[0], ref.populations(k)[0])
    for e in (a, ref):
        e.step(7)
    for k in range(6):
        assert np.array_equal(a.populations(k)[0], ref.populations(k)[0])
    """)


@pytest.mark.parametrize("each,storage,twos", [(3, 0, True), (5, 1, True), (5, 2, True), (1, 0, False)])
def test_autotune_times_the_kernels_that_step(tmp_path, each, storage, twos):
    """The step kernels that dmrt_ensemble_autotune launches are those of the
    interval's plain steps, and the state stays as it was."""
    run_child(tmp_path, f"""
    shapes = [(50, 41, 33), (70, 64, 30)]
    cav = [dict(grid=shapes[k % 2], Ra=1e4 * (1 + k), wall=1 + k % 3) for k in range(2 * {each})]
    a, ref = [dm.Ensemble(cav, storage={storage}, residual_interval=20) for _ in range(2)]
    names = lambda: set(n for n in shim.shim_names().decode().split() if "pair_kernel" in n)
    for e in (a, ref):
        e.step(5)
    shim.shim_forget()
    a.step(4)
    stepped = names()
    assert len(stepped) == ({2 if twos else 1}), stepped
    a.sync()
    shim.shim_forget()
    report = a.autotune(3)
    assert names() == stepped, (names(), stepped)
    assert "chosen threads=128" in report
    ref.step(4)
    for k in range(len(cav)):
        assert np.array_equal(a.populations(k)[0], ref.populations(k)[0])
    a.step(18)
    ref.step(18)
    for k in range(len(cav)):
        assert np.array_equal(a.populations(k)[0], ref.populations(k)[0])
    """)


@pytest.mark.parametrize("grid,split", [
    ((47, 47, 47), False), ((49, 49, 49), False), ((165, 11, 55), False), ((217, 183, 3), False), ((39, 39, 39), False),
    ((45, 45, 45), True), ((55, 55, 55), True), ((33, 1000, 2), True), ((69, 69, 69), True), ((101, 75, 61), True),
])
@pytest.mark.parametrize("streaming", [0, 1])
def test_boxes_with_odd_rows_take_the_faster_kernel(tmp_path, grid, split, streaming):
    """By the blocks that either kernel would have per SM."""
    run_child(tmp_path, f"""
    for storage in (0, 1, 2):
        cav = dm.Cavity({grid}, 1e4, wall_type=1, storage=storage, streaming={streaming}, residual_interval=20)
        shim.shim_forget()
        cav.step(4)
        names = shim.shim_names().decode().split()
        assert names and all(("split" in n) == {split} for n in names), names
    """)


# flat numbering shows as the kernel's last template argument
@pytest.mark.parametrize("grid,streaming,flat", [
    ((54, 54, 54), 0, (0, 1, 1)), ((54, 54, 54), 1, (0, 0, 0)), ((108, 77, 19), 0, (0, 1, 1)), ((30, 30, 30), 1, (1, 0, 0)),
    ((110, 15, 17), 1, (1, 0, 0)), ((28, 46, 24), 1, (1, 0, 0)), ((206, 8, 96), 0, (1, 1, 1)), ((12, 40, 58), 1, (1, 1, 1)),
    ((58, 58, 58), 1, (1, 1, 1)), ((30, 30, 30), 0, (1, 1, 1)), ((70, 70, 70), 0, (1, 1, 1)), ((48, 48, 48), 0, (0, 0, 0)),
])
def test_boxes_with_even_rows_take_the_faster_numbering(tmp_path, grid, streaming, flat):
    run_child(tmp_path, f"""
    for storage, flat in enumerate({flat}):
        cav = dm.Cavity({grid}, 1e4, wall_type=1, storage=storage, streaming={streaming}, residual_interval=20)
        shim.shim_forget()
        cav.step(4)
        names = shim.shim_names().decode().split()
        assert names and all("pair_kernel" in n and f"Lb{{flat}}EEEv" in n for n in names), names
    """)


@pytest.mark.parametrize("grid,kw,name", [
    ((32, 32, 32), {}, "step_pair_kernel"), ((32, 32, 32), {"cells_per_thread": 1}, "step_kernel"),
    ((32, 32, 32), {"streaming": 1}, "step_inplace_pair_kernel"), ((31, 32, 32), {"streaming": 1}, "step_inplace_kernel"),
    ((64, 64, 64), {"storage": 1, "pair_loads": 2}, "step_pair_tma_kernel"),
    ((96, 96, 96), {"storage": 2}, "step_inplace_pair_kernel by twos"),
    ((96, 96, 96), {"storage": 2, "residual_interval": 2}, "step_pair_kernel"),
    ((101, 75, 61), {}, "step_inplace_split_kernel by twos"), ((101, 75, 61), {"storage": 1}, "step_split_kernel"),
    ((101, 75, 61), {"streaming": 1}, "step_inplace_split_kernel"), ((130, 130, 130), {"wall_type": 0}, "step_kernel"),
])
def test_cavities_name_the_kernel_that_steps(tmp_path, grid, kw, name):
    run_child(tmp_path, f"""
    cav = dm.Cavity({grid}, 1e4, **{{"wall_type": 1, **{kw}}})
    shim.shim_forget()
    cav.step(6 if cav.params["residual_interval"] > 6 else 1)
    names = shim.shim_names().decode().split()
    base = {name!r}.split(" ")[0]
    assert cav.step_kernel == {name!r}
    # (mangled names carry their length)
    assert names and all(f"{{len(base)}}{{base}}I" in n for n in names), names
    """)


@pytest.mark.parametrize("grids,kw,name", [
    ([(48, 48, 48)] * 3, {}, "ensemble_group_pair_kernel"), ([(48, 48, 48)] * 3, {"streaming": 1}, "ensemble_group_inplace_pair_kernel"),
    ([(48, 48, 48)] * 5, {}, "ensemble_group_inplace_pair_kernel by twos"),
    ([(48, 48, 48)] * 5, {"residual_interval": 2}, "ensemble_group_pair_kernel"),
    ([(31, 20, 20), (32, 20, 20)], {}, "ensemble_step_kernel"), ([(31, 20, 20)] * 2, {"streaming": 1}, "ensemble_inplace_kernel"),
    ([(2 * k, 8, 8) for k in range(1, 41)], {}, "ensemble_pair_kernel"),
])
def test_ensembles_name_the_kernel_that_steps(tmp_path, grids, kw, name):
    run_child(tmp_path, f"""
    ens = dm.Ensemble([dict(grid=g, Ra=1e4, wall=1) for g in {grids}], **{kw})
    shim.shim_forget()
    ens.step(6 if ens.params(0)["residual_interval"] > 6 else 1)
    names = [n for n in shim.shim_names().decode().split() if "residual" not in n]
    base = {name!r}.split(" ")[0]
    assert ens.step_kernel == {name!r}
    assert names and all(f"{{len(base)}}{{base}}I" in n for n in names), names
    """)
