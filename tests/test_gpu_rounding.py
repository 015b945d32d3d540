"""Rounding errors of the FP64 hop, against extended precision.

The hop: its error is at most that of the plainest order of the same operations, both products of a
direction rounded by themselves and the eight of them added one after the other.  The kernel adds them
as a tree, which leaves 0.93 of that order's error in a model of both; over 24,576 reals the ratio
scatters by less than 0.01.
"""
import numpy as np
import pytest

import synth
from oracle import mdwf_oracle as O

pytestmark = pytest.mark.gpu

M = torch = None
LD, CLD = np.longdouble, np.clongdouble


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


def _dag(W):
    return np.conj(np.swapaxes(W, -1, -2))


def _rms(a):
    return float(np.sqrt(np.mean(a.real ** 2 + a.imag ** 2)))


def _fma(a, b, c):
    return (a.astype(LD) * b + c).astype(np.float64)


def _product(W, v):
    """W v in FP64: one multiply and five multiply-adds per real."""
    out = np.empty_like(v)
    for a in range(3):
        for b in range(3):
            u, x = W[..., None, a, b], v[..., b]
            re = _fma(u.real, x.real, re) if b else u.real * x.real
            im = _fma(u.real, x.imag, im) if b else u.real * x.imag
            re, im = _fma(-u.imag, x.imag, re), _fma(u.imag, x.real, im)
        out[..., a] = re + 1j * im
    return out


def _exact_product(W, v):
    return (W[..., None, :, :].astype(CLD) * v[..., None, :]).sum(-1)


def _hop(U, psi, dagger, product, dtype):
    """The hopping term, its eight products added one after the other."""
    out, s = np.zeros(psi.shape, dtype=dtype), 1.0 if dagger else -1.0
    for mu in range(4):
        ax = (-3, -4, -5, -6)[mu]
        W = U[..., mu, :, :].copy()
        if mu == 3:
            W[-1] *= -1.0
        v = psi.astype(dtype)
        out = out + product(W, O.spin_mul(O.ID4 + s * O.GAMMA[mu], np.roll(v, -1, ax)))
        out = out + product(_dag(np.roll(W, 1, ax)), O.spin_mul(O.ID4 - s * O.GAMMA[mu], np.roll(v, 1, ax)))
    return out


@pytest.mark.parametrize('dagger', [0, 1])
def test_hop_rounds_no_more_than_the_plain_order(dagger):
    dims, L5 = (4, 4, 4, 8), 4
    U = synth.random_gauge(dims, 3, 0.4)
    psi = synth.gaussian_spinor((L5,) + tuple(reversed(dims)) + (4, 3), 4)
    ctx = M.mdwf_create(dims, 0)
    M.mdwf_load_gauge(ctx, 0, U, 1)
    M.mdwf_set_action(ctx, 0, 1.3, 1.5, 0.5, 0.05, L5)
    got = M.mdwf_apply_dslash(ctx, 0, psi, -1, dagger)
    M.mdwf_destroy(ctx)
    exact = _hop(U, psi, dagger, _exact_product, CLD)
    plain = _hop(U, psi, dagger, _product, np.complex128)
    for spins in (slice(0, 2), slice(2, 4)):
        assert _rms((got - exact)[..., spins, :]) <= _rms((plain - exact)[..., spins, :])
