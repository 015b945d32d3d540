"""Output arrays of one batch that coincide or overlap: what they share holds the values of the last
system that covers it, as if the systems were written one after the other."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

M = torch = None
DIMS, L5, ACT = (4, 2, 2, 6), 5, (1.3, 1.5, 0.5, 0.05)
SHAPE = (L5,) + tuple(reversed(DIMS)) + (4, 3)
MASSES = [0.03 + 0.02 * k for k in range(5)]


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


@pytest.fixture
def ctx():
    c = M.mdwf_create(DIMS, 0)
    M.mdwf_load_gauge(c, 0, synth.random_gauge(DIMS, 7, 0.3), 1)
    M.mdwf_set_action(c, 0, *ACT, L5)
    yield c
    torch.cuda.synchronize()
    M.mdwf_destroy(c)


def _views(offsets):
    """Fields at the given offsets (in doubles) of one buffer."""
    n = 2 * int(np.prod(SHAPE))
    buf = torch.zeros(n + max(offsets), dtype=torch.float64, device='cuda')
    return buf, [buf[o:o + n].view(*SHAPE, 2) for o in offsets]


def _in_order(buf, alone, offsets):
    want = torch.zeros_like(buf)
    for x, o in zip(alone, offsets):
        want[o:o + 2 * x.numel()] = torch.view_as_real(x).reshape(-1)
    return want


N = 2 * int(np.prod(SHAPE))
# one array for all; two arrays in turn; every array a site further on than the last, which moves it to the other parity
OFFSETS = {'same': [0] * 5, 'in turn': [0, N, 0, N, 0], 'a site apart': [0, 24, 48, 72, 96]}


@pytest.mark.parametrize('case', list(OFFSETS))
@pytest.mark.parametrize('entry', ['schur', 'noalloc', 'solve'])
def test_shared_outputs(ctx, case, entry):
    srcs = [torch.from_numpy(synth.gaussian_spinor(SHAPE, 70 + k)).cuda() for k in range(5)]
    opts = M.mdwf_default_opts(precision='half')

    def call(ins, outs, masses):
        if entry == 'solve':
            M.mdwf_solve_batch_dev(ctx, 0, ins, outs, 1e-8, masses=masses, opts=opts)
        else:
            f = M.mdwf_apply_schur_batch_dev if entry == 'schur' else M.mdwf_apply_schur_batch_dev_noalloc
            f(ctx, 0, ins, outs, masses=masses, precision='single')
        torch.cuda.synchronize()

    alone = [torch.empty_like(s) for s in srcs]
    torch.cuda.synchronize()
    for s, x, m in zip(srcs, alone, MASSES):
        call([s], [x], [m])
    buf, outs = _views(OFFSETS[case])
    torch.cuda.synchronize()
    call(srcs, outs, MASSES)
    assert torch.equal(buf, _in_order(buf, alone, OFFSETS[case]))
