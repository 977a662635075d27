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
