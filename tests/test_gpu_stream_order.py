"""Calls that follow one another on a stream without a synchronisation between them."""
import numpy as np
import pytest

from gpu_util import ctx, cuda, host, torch

pytestmark = pytest.mark.gpu


def test_chi_batch_follows_the_call_before_it():
    """The chi batch reads what the pair update before it on the stream writes last (its angles, here taken as
    impact parameters), and writes where that one wrote: the same angles as with a synchronisation before it."""
    from paper_2602_21244_gb300 import dsmc as D
    from paper_2602_21244_gb300 import workloads as W
    T, C = torch(), ctx()
    w = W.hypersonic(scale=0.3, model=1)
    gas = D.make_gas(w["gas"])
    pot = D.make_potential(W.JAGER_SYNTHETIC_AR)
    o = C.sort_cells(cuda(w["cell_id"]), cuda(w["vx"]), cuda(w["vy"]), cuda(w["vz"]), w["n_cells"])
    sel = C.select_pairs(gas, o["cell_start"], o["svx"], o["svy"], o["svz"], C.sigma_g_max_init(gas, cuda(w["T_cell"])),
                         1, 1 << 22)
    n = int(host(sel["info"])[0])
    assert n > 10000 and C.sync_status() == 0
    angles = cuda(np.linspace(0.1, 3.0, 64 * 64).astype(np.float32).reshape(64, 64))
    tab = D.ChiTable(angles, 2.0, 12.0)
    g = T.full((n,), 800.0, device="cuda")
    C.jager_chi(gas, pot, g * 1e-3, g)   # (host constants of the potential: kept, so that the next launch is prompt)
    near, want = g * 2e-3, None
    for wait in (True, False, False, False):
        v = [o[k].clone() for k in ("svx", "svy", "svz")]
        b = T.full((n,), 9.0, device="cuda")
        chi = T.empty(n, device="cuda")
        T.cuda.synchronize()
        C.collide_table(gas, tab, 1, sel, *v, chi_out=b)
        if wait:
            T.cuda.synchronize()
        C.jager_chi(gas, pot, b, g, chi=chi)
        C.collide_table(gas, tab, 1, sel, *v, chi_out=b)
        C.jager_chi(gas, pot, near, g, chi=b)   # over the angles just written
        assert C.sync_status() == 0
        got = host(chi), host(b)
        assert want is None or all(np.array_equal(x, y) for x, y in zip(got, want))
        want = got
