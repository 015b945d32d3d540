"""Residual-mass correlators on lattices of few and of many time slices: the number of blocks per slice
follows both the slice's size and their number.

A correlator sums squares: u times (the terms of a component's square + the depth of the sums) of the sum
itself, below 64 u for these sizes.  Lattices of the same volume read the same bytes, so their times are alike
wherever the blocks fill the device; a factor of two is left for the shorter rows of the smaller slices."""
import time

import numpy as np
import pytest

import synth
from oracle import mdwf_oracle as O

pytestmark = pytest.mark.gpu

M = torch = None
U64 = 2.0 ** -53


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


def _ctx(dims, L5):
    ctx = M.mdwf_create(dims, 0)
    M.mdwf_load_gauge(ctx, 0, synth.unit_gauge(dims), 1)
    M.mdwf_set_action(ctx, 0, 1.3, 1.5, 0.5, 0.05, L5)
    return ctx


# blocks per slice: 608 of 608 (all), 608 of 768, 39 and 38 on both sides of Lt = 32, 32 of 32 slots of the sum
@pytest.mark.parametrize('dims', [(18, 18, 20, 2), (16, 16, 32, 2), (8, 8, 8, 32), (8, 8, 8, 40), (4, 2, 2, 64)])
def test_correlators_of_few_and_many_slices(dims):
    L5, n = 2, 2
    xs = [synth.gaussian_spinor((L5,) + tuple(reversed(dims)) + (4, 3), 20 + k) for k in range(n)]
    ctx = _ctx(dims, L5)
    got = M.mdwf_mres_correlators_dev(ctx, 0, [torch.from_numpy(x).cuda() for x in xs])
    M.mdwf_destroy(ctx)
    for a, b in zip(got, O.mres_correlators(xs)):
        assert np.all(np.abs(a - b) <= 64 * U64 * b)


def test_time_does_not_depend_on_the_number_of_slices():
    best = []
    for dims in ((32, 32, 32, 2), (16, 16, 16, 16)):
        ctx = _ctx(dims, 2)
        xs = [torch.ones((2,) + tuple(reversed(dims)) + (4, 3), dtype=torch.complex128, device='cuda') for _ in range(12)]
        torch.cuda.synchronize()
        t = []
        for _ in range(20):
            t0 = time.perf_counter()
            M.mdwf_mres_correlators_dev(ctx, 0, xs)
            t.append(time.perf_counter() - t0)
        best.append(min(t))
        M.mdwf_destroy(ctx)
    assert best[0] <= 2.0 * best[1]
