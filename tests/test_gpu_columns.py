"""The FP64 hop's recursions along the fifth dimension at lengths on both sides of those it holds in registers
(4, 6, 8, 10, 12, 16), in all of its column epilogues: B A^-1 and A^-+ B^+ (the Schur operator), A^-1 of a
source (preparation and reconstruction) and the two forms of the symmetric operator (a solve with schur = 1).

Elementwise bound of the operator: 16 u max |oracle| (the roundings that reach one component)."""
import numpy as np
import pytest

import synth
from oracle import mdwf_oracle as O

pytestmark = pytest.mark.gpu

M = torch = None
U64 = 2.0 ** -53
DIMS, ACT = (4, 2, 2, 4), (1.3, 1.5, 0.5, 0.05)


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


@pytest.mark.parametrize('L5', [2, 3, 4, 6, 8, 9, 10, 12, 14, 16, 17, 20, 24])
def test_fp64_columns(L5):
    U = synth.random_gauge(DIMS, 7, 0.3)
    shape = (L5,) + tuple(reversed(DIMS)) + (4, 3)
    b = synth.gaussian_spinor(shape, 5)
    e = O.restrict(b, O.parity_mask(DIMS))
    ctx = M.mdwf_create(DIMS, 0)
    try:
        M.mdwf_load_gauge(ctx, 0, U, 1)
        M.mdwf_set_action(ctx, 0, *ACT, L5)
        for dagger, op in ((0, O.schur_op), (1, O.schur_op_dag)):
            ref = op(U, e, *ACT)
            got = M.mdwf_apply_schur(ctx, 0, e, dagger, M.MDWF_PREC_DOUBLE)
            assert np.abs(got - ref).max() <= 16 * U64 * np.abs(ref).max()
        for schur in (0, 1):
            xs, _ = M.mdwf_solve_batch(ctx, 0, [b], 1e-10, opts=M.mdwf_default_opts(precision='double', schur=schur))
            assert O.true_residual(U, b, xs[0], *ACT) <= 1e-10
    finally:
        M.mdwf_destroy(ctx)
