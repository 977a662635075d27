"""Kernel variants chosen by size: every variant gives what the others give."""
import numpy as np
import pytest

from gpu_util import ctx, cuda, host, torch

pytestmark = pytest.mark.gpu


def _sms():
    return torch().cuda.get_device_properties(0).multi_processor_count


def _cells(n_cells, seed=4):
    """Ragged cells at both ends of n_cells cells (32 and 128 are the particles that a cell's lanes
    hold in registers), empty ones between: the same particles whatever n_cells."""
    rng = np.random.default_rng(seed)
    ends = [[0, 1, 2, 31, 32, 33, 127], [128, 129, 1024, 5, 0, 3]]
    sizes = np.zeros(n_cells, np.int64)
    sizes[:7], sizes[-6:] = ends
    n = int(sizes.sum())
    v = (rng.uniform(-1e4, 1e4, (n, 3)) + 10.0 ** rng.uniform(-3, 3, (n, 1)) * rng.standard_normal((n, 3))).T
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), [np.ascontiguousarray(c) for c in v]


@pytest.mark.parametrize("per_sm,more", [(0, 13), (8, 0), (8, 1), (128, 0), (128, 1), (320, 0), (320, 1)])
def test_cell_kernels_agree_across_sizes(per_sm, more):
    """Moments and moment matching: the per-cell results are exact integer sums converted by the same
    FP64 operations, so the one-group-per-warp kernels equal the claiming kernel bit for bit."""
    C = ctx()
    out = []
    for nc in (per_sm * _sms() + more, 400 * _sms()):
        cs, v = _cells(nc)
        x = [cuda(c) for c in v]
        mom = C.cell_moments(cuda(cs), *x)
        y = [c * 1.25 + 3.0 for c in x]
        C.moment_match(cuda(cs), mom, *y)
        assert C.sync_status() == 0
        m = host(mom)
        assert not m[7:-6].any()
        out.append([m[:7], m[-6:]] + [host(c) for c in y])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_one_group_per_warp_moments_report_nonfinite():
    from paper_2602_21244_gb300 import dsmc as D
    C = ctx()
    cs, v = _cells(40)
    v[1][3] = np.nan
    C.cell_moments(cuda(cs), *[cuda(c) for c in v])
    assert C.sync_status() == D.DSMC_ERR_NONFINITE


@pytest.mark.parametrize("n_nodes", [8, 33, 128])
def test_chi_does_not_depend_on_the_warp_it_runs_in(n_nodes):
    """The chi batch shares the bracket scan and the nodes of a warp's low-energy pairs between its lanes
    while few of them are low; the sums keep the order of the nodes, so a pair's chi is the same bits in
    warps of any mix (0, 1, 8, 9, 20, 21, 28, 29 and 32 low pairs), with head-on, motionless and
    core-penetrating pairs among them, and in a batch that ends inside a warp."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    C = ctx()
    gas = D.make_gas(dict(mass=W.M_AR, fn_over_vc=1.0, dt=1.0, model=1, b_max=1.2e-9))
    pot = D.make_potential(W.JAGER_SYNTHETIC_AR)
    rng = np.random.default_rng(n_nodes)
    g, b = [], []
    for low in (0, 1, 8, 9, 20, 21, 28, 29, 32, 3):
        gg = np.where(rng.permutation(32) < low, rng.uniform(100, 400, 32), rng.uniform(500, 15000, 32))
        g.append(gg)
        b.append(12.0 * np.sqrt(rng.random(32)))
    g, b = (np.concatenate(a).astype(np.float32)[:-5] for a in (g, b))
    g[40], g[41], b[42], g[70], b[70] = 0.0, 9.0e4, 0.0, 9.0e4, 0.5
    whole = host(C.jager_chi(gas, pot, cuda(b), cuda(g), n_nodes=n_nodes))
    assert C.sync_status() == 0 and np.isfinite(whole).all() and whole[42] == np.float32(np.pi) and whole[40] == 0
    for order in (np.argsort(g), rng.permutation(len(g))):
        again = host(C.jager_chi(gas, pot, cuda(b[order]), cuda(g[order]), n_nodes=n_nodes))
        assert np.array_equal(again, whole[order])
    one = [float(host(C.jager_chi(gas, pot, cuda(b[q:q + 1]), cuda(g[q:q + 1]), n_nodes=n_nodes))[0])
           for q in range(0, len(g), 7)]
    assert np.array_equal(np.float32(one), whole[::7])


@pytest.mark.parametrize("n", [4096, 65536, 65537, 2500000, 2500001])
def test_sort_variants_by_particle_count(n):
    """16 and 17 chunks of the radix sort (the scatter sums few chunks' counts itself) and both sides of
    the gather's switch from one launch to one per component: the stable order, bit for bit."""
    C = ctx()
    rng = np.random.default_rng(n)
    nc = 1000
    cid = rng.integers(0, nc, n).astype(np.int32)
    v = [rng.standard_normal(n) for _ in range(3)]
    out = C.sort_cells(cuda(cid), *[cuda(c) for c in v], nc)
    assert C.sync_status() == 0
    perm = np.argsort(cid, kind="stable")
    assert np.array_equal(host(out["perm"]), perm)
    assert np.array_equal(host(out["cell_start"]), np.concatenate([[0], np.cumsum(np.bincount(cid, minlength=nc))]))
    for k, c in zip(("svx", "svy", "svz"), v):
        assert np.array_equal(host(out[k]), c[perm])


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("pad", [4096, 4097, 8192, 8193])
def test_selection_variants_by_cell_count(pad, order):
    """One-block and two-launch word counts and scans: the same cells followed by empty ones give the same
    selection, whatever the number of cells."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    C = ctx()
    w = W.hypersonic(scale=0.05)
    gas = D.make_gas(w["gas"])
    got = []
    for nc in (w["n_cells"], pad):
        o = C.sort_cells(cuda(w["cell_id"]), cuda(w["vx"]), cuda(w["vy"]), cuda(w["vz"]), nc)
        sg = C.sigma_g_max_init(gas, cuda(np.concatenate([w["T_cell"], np.full(nc - w["n_cells"], 300.0)])))
        sel = C.select_pairs(gas, o["cell_start"], o["svx"], o["svy"], o["svz"], sg, 5, 1 << 18, order=order)
        assert C.sync_status() == 0
        info = host(sel["info"])
        n, R = int(info[0]), int(info[2])
        assert n > 1000 and R > 3
        got.append([info, host(sel["pairs"])[:n], host(sel["deps"])[:n], host(sel["round_offsets"])[:R + 1],
                    host(sg)[:w["n_cells"]]])
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_collide_accepts_a_workspace_at_any_word():
    """The done stamps are cleared 16 bytes at a time only from an aligned workspace."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    C = ctx()
    w = W.hypersonic(scale=0.05, model=0)
    gas = D.make_gas(w["gas"])
    o = C.sort_cells(cuda(w["cell_id"]), cuda(w["vx"]), cuda(w["vy"]), cuda(w["vz"]), w["n_cells"])
    sg = C.sigma_g_max_init(gas, cuda(w["T_cell"]))
    sel = C.select_pairs(gas, o["cell_start"], o["svx"], o["svy"], o["svz"], sg, 1, 1 << 18)
    n = len(w["cell_id"])
    got = []
    for shift in (0, 4, 12):
        ws = torch().full((4 * n + 1024,), 255, dtype=torch().uint8, device="cuda")[shift:]
        v = [o[k].clone() for k in ("svx", "svy", "svz")]
        C.collide_vhs(gas, 1, sel, *v, ws=ws)
        assert C.sync_status() == 0
        got.append(host(torch().stack(v)))
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


@pytest.mark.parametrize("n_hidden", [1, 3, 4])
@pytest.mark.parametrize("cells,dt", [(1, 1e-9), (3, 1e-7), (40, 1e-7)])
def test_neural_collide_does_not_depend_on_the_order_of_its_tiles(cells, dt, n_hidden):
    """A single pair, fewer than a tile, and chains of many levels: the rounds' and the claim levels' lists hold
    the same pairs in other tiles, and each pair's arithmetic is its own, so the velocities agree bit for bit."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C = torch(), ctx()
    w = W.couette(seed=3, n_cells=cells, per_cell=150)
    gas = D.make_gas(dict(w["gas"], fn_over_vc=4e19, dt=dt, model=1))
    wts = W.mlp_weights(n_hidden=n_hidden)
    mlp = D.make_mlp(8, 128, n_hidden, 3, 0, W.sigma_v(), 273.0, 1e-12)
    bits, bias = cuda(wts["W_bits"].view(np.int16)), cuda(wts["bias"].astype(np.float32))
    o = C.sort_cells(cuda(w["cell_id"]), cuda(w["vx"]), cuda(w["vy"]), cuda(w["vz"]), cells)
    mom = C.cell_moments(o["cell_start"], o["svx"], o["svy"], o["svz"])
    got, pairs = [], None
    for order in (0, 1):
        sg = C.sigma_g_max_init(gas, cuda(w["T_cell"]))
        sel = C.select_pairs(gas, o["cell_start"], o["svx"], o["svy"], o["svz"], sg, 2, 1 << 18, order=order)
        v = [o[k].clone() for k in ("svx", "svy", "svz")]
        C.collide_neural(gas, mlp, bits, bias, 2, mom, sel, *v)
        assert C.sync_status() == 0
        got.append(host(T.stack(v)))
        pairs = int(host(sel["info"])[0])
    assert np.array_equal(got[0], got[1])
    start = np.stack([host(o[k]) for k in ("svx", "svy", "svz")])
    assert np.array_equal(got[0], start) == (pairs == 0)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("runs", [1, 16, 17, 32, 0])
@pytest.mark.parametrize("n", [4096, 4097, 12287, 17 * 4096 + 31])
def test_sort_is_stable_for_every_run_length(n, runs, offset):
    """Batches of 32 with 1, 16, 17 or 32 runs of equal cells (0: a mix, run lengths changing inside a
    warp) take the ranks from match or from ballots; whole and partial chunks, ids at any word; ids out
    of range in both.  Whole numbers: the order is the stable one."""
    from paper_2602_21244_gb300 import dsmc as D
    C, rng = ctx(), np.random.default_rng(n + runs)
    n_cells = 70000
    i = np.arange(n)
    group = i * runs // 32 if runs else np.cumsum(rng.random(n) < np.repeat(rng.random(n // 64 + 1), 64)[:n])
    ids = rng.integers(0, n_cells, int(group[-1]) + 1)[group].astype(np.int32)
    ids[[0, n // 2, n - 1]] = [0, n_cells - 1, 0]
    buf = cuda(np.concatenate([np.zeros(offset, np.int32), ids]))[offset:]
    v = [cuda(rng.standard_normal(n)) for _ in range(3)]
    o = C.sort_cells(buf, *v, n_cells)
    assert C.sync_status() == 0
    order = np.argsort(ids, kind="stable")
    assert np.array_equal(host(o["perm"]), order)
    assert np.array_equal(host(o["cell_start"]), np.concatenate([[0], np.cumsum(np.bincount(ids, minlength=n_cells))]))
    assert np.array_equal(host(o["svx"]), host(v[0])[order])
    buf[n // 3] = -1
    buf[n // 5] = n_cells
    o = C.sort_cells(buf, *v, n_cells)
    assert C.sync_status() == D.DSMC_ERR_ARG
    keep = host(buf)
    keep = np.where((keep < 0) | (keep >= n_cells), n_cells, keep)
    assert np.array_equal(host(o["perm"])[:n - 2], np.argsort(keep, kind="stable")[:n - 2])


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_jager_rotation_along_an_axis(axis):
    """Relative velocities along one axis: along x the rotation's frame is the degenerate one.  Velocities
    within 1e-12 of max(|v|, c_ref) of the oracle's rotation by the kernel's own chi, as for the random gas."""
    from gpu_util import c_ref
    import test_gpu_parity as P
    W = P.W
    from paper_2602_21244_gb300 import dsmc as D
    w = W.hypersonic(scale=0.04)
    for c in range(3):
        if c != axis:
            w[("vx", "vy", "vz")[c]][:] = 0.0
    gas = P.O.make_gas(**w["gas"])
    sg0 = P._sgmax0(w, gas)
    perm, cs, *x = P.oracle_sorted(w)
    pr = P.O.select_pairs(gas, cs, *x, sg0, 4, capacity=1 << 22)
    Dg, srt, mom, sg, sel = P.gpu_step_pieces(w, sg0, step=4)
    C = ctx()
    n = int(host(sel["info"])[0])
    assert n == pr["n_pairs"] > 0
    chi = torch().zeros(n, dtype=torch().float32, device="cuda")
    C.collide_jager(Dg, D.make_potential(P.JP), 4, sel, srt["svx"], srt["svy"], srt["svz"], n_nodes=32, chi_out=chi)
    assert C.sync_status() == 0
    p = P.sel_host(sel)["pairs"]
    order = np.lexsort((p[:, 3], p[:, 2]))
    want = P.O.collide_given_chi(gas, pr, 4, host(chi)[order].astype(np.float64), *x)
    for a, r in zip(("svx", "svy", "svz"), want):
        assert (np.abs(host(srt[a]) - r) / np.maximum(np.abs(r), c_ref(W.M_AR))).max() <= 1e-12


@pytest.mark.parametrize("path", ["vhs", "table"])
@pytest.mark.parametrize("nx,ny,per,scale", [(1, 1, 300, 2000.0), (3, 1, 200, 5000.0), (33, 31, 20, 300.0),
                                             (-64, 1, 20, 7000.0), (-64, 1, 4, 2000.0), (-64, 1, 4, 0.0)])
def test_step_by_cell_groups_equals_the_collide_calls(path, nx, ny, per, scale):
    """The step's pair update by groups of cells against the collide call that takes any pair list: more
    rounds than a warp has lanes, one cell, more groups than warps, the last size that goes by groups
    (VHS: 64 cells per SM, nx = -64), fewer pairs than cells and none at all.  The same functions on the same pairs in the
    same order of each particle's pairs: the same bits."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C = torch(), ctx()
    nx = nx if nx > 0 else -nx * _sms()
    nc, rng = nx * ny, np.random.default_rng(nx + per)
    counts = rng.poisson(per, nc)
    cid = rng.permutation(np.repeat(np.arange(nc, dtype=np.int32), counts))
    n = len(cid)
    v = [cuda(c) for c in 400.0 * rng.standard_normal((3, n))]
    gas = D.make_gas(dict(W.couette()["gas"], b_max=4.17e-10, fn_over_vc=max(scale, 1e-6) * 2e18, dt=1e-7,
                          model=1 if path == "table" else 0))
    cells = cuda(cid)
    sg0 = C.sigma_g_max_init(gas, cuda(np.full(nc, 300.0)))
    o = C.sort_cells(cells, *v, nc)
    x = [o[k] for k in ("svx", "svy", "svz")]
    mom = C.cell_moments(o["cell_start"], *x)
    cap = 1 << 22
    sel = C.select_pairs(gas, o["cell_start"], *x, sg0.clone(), 7, cap)
    chi = cuda(np.linspace(0.1, 3.0, 64 * 64).astype(np.float32).reshape(64, 64))
    tab = D.ChiTable(chi, 2.0, 12.0)
    if path == "vhs":
        C.collide_vhs(gas, 7, sel, *x)
    else:
        C.collide_table(gas, tab, 7, sel, *x)
    C.moment_match(o["cell_start"], mom, *x)
    info = host(sel["info"])
    st = D.StepState(C, n, nc, cap)
    for a, b in zip((st.vx, st.vy, st.vz), v):
        a.copy_(b)
    st.cell_id.copy_(cells)
    st.sigma_g_max.copy_(sg0)
    C.step(gas, D.make_path(D.PATH_VHS) if path == "vhs" else D.make_path(D.PATH_TABLE, table=tab), st, 7)
    assert C.sync_status() == 0
    assert np.array_equal(host(st.info), info)
    assert (info[0] > 0) == (scale > 0) and (per < 200 or (info[2] & 0xFFFFFFFF) > 32)
    for a, b in zip((st.svx, st.svy, st.svz), x):
        assert np.array_equal(host(a), host(b))


@pytest.mark.parametrize("n", [16, 128, 144, 4096])
@pytest.mark.parametrize("act", [0, 1])
def test_training_takes_parameters_and_workspace_at_any_word(n, act):
    """Weights read 16 bytes or a word at a time, partial gradients written 16 bytes or a word at a time: the
    same values, so loss and gradient agree bit for bit; part of a tile, one, more than one, many."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C, rng = torch(), ctx(), np.random.default_rng(n)
    mlp = D.make_mlp(8, 128, 3, 3, act, W.sigma_v(), 273.0, 1e-12)
    theta = (0.1 * rng.standard_normal(D_PARAMS)).astype(np.float32)
    pairs = [cuda(400.0 * rng.standard_normal((n, 3))) for _ in range(4)]
    temp = cuda(rng.uniform(200.0, 400.0, n))
    nb = C.train_workspace("cuda").numel()
    got = []
    for off in (0, 1, 2):
        th = T.zeros(D_PARAMS + off, device="cuda")[off:]
        th.copy_(cuda(theta))
        ws = T.zeros(nb + 4 * off, dtype=T.uint8, device="cuda")[4 * off:]
        g, l = C.train_loss_grad(mlp, th, 5, 1, pairs[0], pairs[1], temp, pairs[2], pairs[3], ws=ws)
        assert C.sync_status() == 0
        got.append((host(g), host(l)))
    assert np.isfinite(got[0][0]).all() and np.abs(got[0][0]).max() > 0
    for g, l in got[1:]:
        assert np.array_equal(g, got[0][0]) and np.array_equal(l, got[0][1])


D_PARAMS = 34563   # weights and biases of the operator (d_in 8, width 128, 3 hidden layers, 3 outputs)


@pytest.mark.parametrize("copies", [False, True])
@pytest.mark.parametrize("n", [16, 144])
def test_training_step_is_gradient_then_adam(n, copies):
    """The step applies Adam where the gradient is summed: the same formulas on the same sums in FP32, whose
    multiply-adds either kernel may contract: within four roundings (4 x 2^-24) of the larger term."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C, rng = torch(), ctx(), np.random.default_rng(n)
    mlp = D.make_mlp(8, 128, 3, 3, 0, W.sigma_v(), 273.0, 1e-12)
    pairs = [cuda(400.0 * rng.standard_normal((n, 3))) for _ in range(4)]
    temp = cuda(rng.uniform(200.0, 400.0, n))
    start = [cuda((s * np.abs(rng.standard_normal(D_PARAMS))).astype(np.float32)) for s in (0.1, 1e-3, 1e-6)]
    weights, ws, res = D_PARAMS - 387, C.train_workspace("cuda"), []
    for fused in (True, False):
        th, m, v = (t.clone() for t in start)
        wb = T.zeros(weights, dtype=T.int16, device="cuda") if copies else None
        bias = T.zeros(387, device="cuda") if copies else None
        grad, loss = T.zeros(D_PARAMS, device="cuda"), T.zeros(1, dtype=T.float64, device="cuda")
        if fused:
            C.train_step(mlp, th, m, v, 3, 1e-3, 9, pairs[0], pairs[1], temp, pairs[2], pairs[3], grad, loss, ws, wb, bias)
        else:
            grad, loss = C.train_loss_grad(mlp, th, 9, 3, pairs[0], pairs[1], temp, pairs[2], pairs[3], ws=ws)
            C.adam_step(weights, grad, th, m, v, 3, w_bits=wb, bias=bias)
        assert C.sync_status() == 0
        res.append([host(t) for t in (grad, loss, th, m, v)])
        if copies:
            assert np.array_equal(host(bias), res[-1][2][weights:])
            bits = host(wb).view(np.uint16).astype(np.uint32) << 16
            assert np.abs(bits.view(np.float32) - res[-1][2][:weights]).max() <= np.abs(res[-1][2]).max() * 2.0 ** -8
    (g0, l0, *a), (g1, l1, *b) = res
    assert np.array_equal(g0, g1) and np.array_equal(l0, l1)
    for x, y, s in zip(a, b, start):
        assert np.abs(x - y).max() <= 4 * 2.0 ** -24 * max(np.abs(y).max(), float(s.abs().max()))
