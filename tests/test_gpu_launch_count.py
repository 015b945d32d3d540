"""stats.kernel_launches of batches that one pack launch cannot take (it takes 64 systems)."""
import pytest

import synth

pytestmark = pytest.mark.gpu

M = torch = None


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


@pytest.mark.parametrize('n,more', [(1, 0), (64, 0), (65, 6), (129, 12)])
def test_pack_launches_are_counted(n, more):
    """Equal systems take the same chunks and updates whatever their number; each group of 64 adds a launch per parity
    to the two packings of the sources and to the unpacking of the solutions."""
    dims, L5 = (2, 2, 2, 2), 2
    ctx = M.mdwf_create(dims, 0)
    M.mdwf_load_gauge(ctx, 0, synth.random_gauge(dims, 7, 0.3), 1)
    M.mdwf_set_action(ctx, 0, 1.3, 1.5, 0.5, 0.05, L5)
    b = torch.from_numpy(synth.gaussian_spinor((L5,) + tuple(reversed(dims)) + (4, 3), 5)).cuda()

    def launches(k):
        xs = [torch.empty_like(b) for _ in range(k)]
        torch.cuda.synchronize()
        st = M.mdwf_solve_batch_dev(ctx, 0, [b] * k, xs, 1e-8, opts=M.mdwf_default_opts(precision='double'))
        assert all(s['iters'] == st[0]['iters'] for s in st)
        return st[0]['kernel_launches']

    try:
        assert launches(n) - launches(2) == more
    finally:
        M.mdwf_destroy(ctx)
