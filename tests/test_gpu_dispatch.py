"""Both sides of the sizes at which a call changes its kernel, and what the change costs."""
import numpy as np
import pytest

from gpu_util import ctx, cuda, host, torch

pytestmark = pytest.mark.gpu


def _sms():
    return torch().cuda.get_device_properties(0).multi_processor_count


def _best_us(f, reps=20):
    """Shortest of five means over `reps` calls, by events."""
    T = torch()
    f()
    best = 1e30
    for _ in range(5):
        a, b = T.cuda.Event(enable_timing=True), T.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            f()
        b.record()
        T.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / reps)
    return best


def _moments_and_matching(sizes, seed=6):
    """Moments and matched velocities of cells of these sizes: (starts, moments, velocities)."""
    C, rng = ctx(), np.random.default_rng(seed)
    cs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    x = [cuda(v) for v in 1e3 * rng.standard_normal((3, int(cs[-1]))) + 50.0]
    mom = C.cell_moments(cuda(cs), *x)
    y = [c * 1.5 - 7.0 for c in x]
    C.moment_match(cuda(cs), mom, *y)
    assert C.sync_status() == 0
    return cs, host(mom), [host(c) for c in y]


@pytest.mark.parametrize("per_sm,more", [(0, 40), (8, 1), (96, 0), (96, 1)])
def test_cells_longer_than_a_lane_group_holds(per_sm, more):
    """Cells of up to ten times what a group's lanes hold in registers (32 and 128 particles), around every
    multiple that the batches of four loads have: bit for bit what the claiming kernel gives, whatever the size."""
    ends = [[k + d for k in (32, 64, 96, 128, 160) for d in (-1, 0, 1)],
            [k + d for k in (256, 384, 512, 640, 1280) for d in (-1, 0, 1)] + [0, 7]]
    out = []
    for nc in (per_sm * _sms() + more, 400 * _sms()):
        sizes = np.zeros(nc, np.int64)
        sizes[:15], sizes[-17:] = ends
        _, mom, v = _moments_and_matching(sizes)
        out.append([mom[:15], mom[-17:]] + v)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_dense_cells_cost_no_more_by_groups_than_by_claims():
    """Matching of 1,300 cells of about 1,000 particles (by groups of cells) against the same cells before 20,000
    empty ones (by claims, which visit those too): not above 1.4 times (one load at a time for the particles
    beyond the held ones took twice the time)."""
    T, C = torch(), ctx()
    sizes = np.random.default_rng(1).poisson(1000, 1300)
    took = []
    for nc in (1300, 21300):
        starts = cuda(np.concatenate([[0], np.cumsum(np.pad(sizes, (0, nc - 1300)))]).astype(np.int32))
        v = [T.randn(int(sizes.sum()), dtype=T.float64, device="cuda") for _ in range(3)]
        mom = C.cell_moments(starts, *v)
        took.append(_best_us(lambda: C.moment_match(starts, mom, *v)))
    assert took[0] <= 1.4 * took[1], took


@pytest.mark.parametrize("path,nx,per,scale", [("vhs", 64, 20, 2000.0), ("vhs", 65, 20, 2000.0), ("table", 288, 20, 1000.0),
                                               ("table", 289, 20, 1000.0), ("vhs", 0, 470, 1500.0), ("vhs", 0, 600, 1500.0),
                                               ("table", 0, 470, 1500.0), ("table", 0, 600, 1500.0), ("vhs", 64, 75, 300.0),
                                               ("table", 288, 65, 300.0)])
def test_step_on_both_sides_of_the_cell_groups(path, nx, per, scale):
    """A step on each side of every limit of the update by groups of cells (cells per SM; particles per cell, three
    cells; particles per SM) against the collide call: the same bits."""
    import test_gpu_variants as V
    V.test_step_by_cell_groups_equals_the_collide_calls(path, nx * _sms() if nx else 3, 1, per, scale)


def _uniform_gas(n_cells, per):
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C = torch(), ctx()
    n = n_cells * per
    gas = D.make_gas(dict(W.couette()["gas"], b_max=4.17e-10, fn_over_vc=3e20, dt=1e-7, model=0))
    st = D.StepState(C, n, n_cells, 4 * n)
    for c in (st.vx, st.vy, st.vz):
        c.copy_(T.randn(n, dtype=T.float64, device="cuda") * 400)
    st.cell_id.copy_(T.arange(n, device="cuda", dtype=T.int32) % n_cells)
    st.sigma_g_max.copy_(C.sigma_g_max_init(gas, T.full((n_cells,), 300.0, dtype=T.float64, device="cuda")))
    return gas, D.make_path(D.PATH_VHS), st


def test_autotune_times_the_kernels_that_take_the_shapes():
    """A gas whose step takes the moments one group of cells per warp, without a shape: the trials are of the
    claiming kernel, which a quarter of the blocks slows down by more than 15 %; by the other kernel all
    would take the same time."""
    from paper_2602_21244_gb300 import dsmc as D
    C = ctx()
    gas, path, st = _uniform_gas(300 * _sms(), 30)
    try:
        trials = C.autotune_step(gas, path, st, step=0, reps=20)
        ms = {t["blocks_per_sm"]: t["ms"] for t in trials if t["kernel"] == "moments"}
        assert sorted(ms) == [1, 2, 3, 4] and ms[1] > 1.15 * ms[4], ms
    finally:
        for k in range(len(D.TUNE_KERNELS)):
            C.tune_set(k)


def test_autotune_keeps_the_builtin_shape_where_all_launch_alike():
    """A gas of fewer cells than a block per SM: one launch, one time, and no shape chosen by noise."""
    from paper_2602_21244_gb300 import dsmc as D
    C = ctx()
    gas, path, st = _uniform_gas(8 * _sms(), 20)
    kernels = [D.TUNE_KERNELS.index(k) for k in ("moments", "moment_match")]
    for k in kernels:
        C.tune_set(k)
    default = [C.tune_get(k) for k in kernels]
    try:
        trials = C.autotune_step(gas, path, st, step=0, reps=2)
        for k in ("moments", "moment_match"):
            assert len({t["ms"] for t in trials if t["kernel"] == k}) == 1
        assert [C.tune_get(k) for k in kernels] == default
    finally:
        for k in range(len(D.TUNE_KERNELS)):
            C.tune_set(k)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("pad", [1024, 1025, 2048, 2049, 8192, 8193, 2048 * 4096, 2048 * 4096 + 1])
def test_selection_on_both_sides_of_its_launches(pad, order):
    """One tile and two of the one-block word counts, their last size (2,048 cells) and the first of two launches, the
    last one-block scan (8,192 counts), the last scan whose blocks sum the ones before them (2,048 blocks)."""
    import test_gpu_variants as V
    V.test_selection_variants_by_cell_count(pad, order)
