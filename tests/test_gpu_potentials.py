"""Hard spheres and the inverse power law through the kernels compiled for them."""
import numpy as np
import pytest

from gpu_util import c_ref, ctx, cuda, host, torch
import test_gpu_dispatch as G
import test_gpu_parity as P

pytestmark = pytest.mark.gpu

W = P.W
SPECS = [dict(kind=1, d_hs=3.6), dict(kind=2, kappa=1.3e9, p=12.0)]


def _setup(spec):
    from paper_2602_21244_gb300 import dsmc as D
    gas = D.make_gas(dict(mass=W.M_AR, fn_over_vc=1.0, dt=1.0, model=1, b_max=1.2e-9))
    return D, ctx(), gas, D.make_potential(spec)


@pytest.mark.parametrize("n_nodes", [8, 33, 128])
@pytest.mark.parametrize("spec", SPECS)
def test_chi_does_not_depend_on_its_place(spec, n_nodes):
    """One pair, a part of a warp and several blocks, in any order, head-on and motionless pairs among them: every
    pair's angle is the same bits."""
    D, C, gas, pot = _setup(spec)
    rng = np.random.default_rng(n_nodes)
    n = 128 * 5 - 3
    g = np.exp(rng.uniform(np.log(100), np.log(15000), n)).astype(np.float32)
    b = (12.0 * np.sqrt(rng.random(n))).astype(np.float32)
    g[40], b[42] = 0.0, 0.0
    whole = host(C.jager_chi(gas, pot, cuda(b), cuda(g), n_nodes=n_nodes))
    assert C.sync_status() == 0 and np.isfinite(whole).all() and whole[40] == 0 and whole[42] == np.float32(np.pi)
    order = rng.permutation(n)
    assert np.array_equal(host(C.jager_chi(gas, pot, cuda(b[order]), cuda(g[order]), n_nodes=n_nodes)), whole[order])
    one = [float(host(C.jager_chi(gas, pot, cuda(b[q:q + 1]), cuda(g[q:q + 1]), n_nodes=n_nodes))[0]) for q in range(0, n, 37)]
    assert np.array_equal(np.float32(one), whole[::37])


@pytest.mark.parametrize("spec", SPECS)
def test_collide_rotates_by_its_own_chi(spec):
    """Velocities within 1e-12 of max(|v|, c_ref) of the oracle's rotation by the kernel's own chi, the bound of the
    Jager form."""
    from paper_2602_21244_gb300 import dsmc as D
    w = W.hypersonic(scale=0.04)
    gas = P.O.make_gas(**w["gas"])
    sg0 = P._sgmax0(w, gas)
    perm, cs, *x = P.oracle_sorted(w)
    pr = P.O.select_pairs(gas, cs, *x, sg0, 4, capacity=1 << 22)
    Dg, srt, mom, sg, sel = P.gpu_step_pieces(w, sg0, step=4)
    C = ctx()
    n = int(host(sel["info"])[0])
    assert n == pr["n_pairs"] > 0
    chi = torch().zeros(n, dtype=torch().float32, device="cuda")
    C.collide_jager(Dg, D.make_potential(spec), 4, sel, srt["svx"], srt["svy"], srt["svz"], n_nodes=32, chi_out=chi)
    assert C.sync_status() == 0
    p = P.sel_host(sel)["pairs"]
    order = np.lexsort((p[:, 3], p[:, 2]))
    assert (host(chi) != 0).any()
    want = P.O.collide_given_chi(gas, pr, 4, host(chi)[order].astype(np.float64), *x)
    for a, r in zip(("svx", "svy", "svz"), want):
        assert (np.abs(host(srt[a]) - r) / np.maximum(np.abs(r), c_ref(W.M_AR))).max() <= 1e-12


def test_hard_sphere_batch_does_not_pay_for_the_jager_form():
    """2^22 hard-sphere pairs with 128 nodes of a few operations take less time than the same pairs of the Jager form
    with 32 nodes (0.6 of it; through a kernel that holds the Jager form's code too, 1.15)."""
    D, C, gas, hs = _setup(SPECS[0])
    jager = D.make_potential(W.JAGER_SYNTHETIC_AR)
    b, g = (cuda(a) for a in W.chi_pairs(1 << 22, seed=1))
    chi = torch().empty_like(b)
    took = [G._best_us(lambda: C.jager_chi(gas, p, b, g, n_nodes=n, chi=chi), reps=3) for p, n in ((hs, 128), (jager, 32))]
    assert took[0] < 0.85 * took[1], took
