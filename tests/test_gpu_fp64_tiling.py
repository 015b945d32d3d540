"""Sites per block of the FP64 hop: the caller's choice (opts.nsb, bits 8 to 15 of the batched operator's
hop_variant) gives the bits of the library's own, and mdwf_autotune reports the latter."""
import pytest

import synth
from oracle import mdwf_oracle as O

pytestmark = pytest.mark.gpu

M = torch = None
ACT = (1.3, 1.5, 0.5, 0.05)


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


def _ctx(dims, L5):
    ctx = M.mdwf_create(dims, 0)
    M.mdwf_load_gauge(ctx, 0, synth.random_gauge(dims, 7, 0.3), 1)
    M.mdwf_set_action(ctx, 0, *ACT, L5)
    return ctx


@pytest.mark.parametrize('L5,n', [(2, 1), (5, 1), (8, 1), (8, 3), (12, 4)])
def test_autotune_reports_the_fp64_tiling(L5, n):
    """32 units per block, whole sites, on a lattice with more blocks than the device runs at a time."""
    ctx = _ctx((8, 8, 8, 16), L5)
    try:
        t = M.mdwf_autotune(ctx, 0, n, 'double')
        assert t['nsb'] == max(1, 32 // (L5 * n)) and t['hop_variant'] == M.HOP_DIRECT and t['ms_per_pair'] > 0
    finally:
        M.mdwf_destroy(ctx)


@pytest.mark.parametrize('L5,n', [(2, 1), (5, 4), (32, 17)])
def test_sites_per_block_do_not_change_the_bits(L5, n):
    """Up to more sites than the shared-memory tile holds."""
    dims = (4, 2, 2, 6)
    ctx = _ctx(dims, L5)
    try:
        shape = (L5,) + tuple(reversed(dims)) + (4, 3)
        xs = [torch.from_numpy(O.restrict(synth.gaussian_spinor(shape, 80 + k), O.parity_mask(dims))).cuda()
              for k in range(n)]
        masses = [0.02 + 0.01 * (k % 7) for k in range(n)]
        ref = None
        for nsb in (0, 1, 2, 5, 64, 255):
            for dagger in (0, 1):
                outs = [torch.empty_like(x) for x in xs]
                torch.cuda.synchronize()
                M.mdwf_apply_schur_batch_dev(ctx, 0, xs, outs, masses=masses, dagger=dagger, precision='double',
                                             hop_variant=M.HOP_DIRECT | (nsb << 8))
                torch.cuda.synchronize()
                if nsb == 0:
                    ref = (ref or []) + [outs]
                assert all(torch.equal(a, b) for a, b in zip(ref[dagger], outs))
        for nsb in (0, 3):
            y = torch.empty_like(xs[0])
            torch.cuda.synchronize()
            M.mdwf_solve_batch_dev(ctx, 0, xs[:1], [y], 1e-8, opts=M.mdwf_default_opts(precision='double', nsb=nsb))
            torch.cuda.synchronize()
            if nsb == 0:
                first = y
        assert torch.equal(first, y)
    finally:
        M.mdwf_destroy(ctx)
