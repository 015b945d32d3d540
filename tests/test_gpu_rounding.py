"""Rounding errors of the FP64 hop and of the flow, against extended precision.

The hop: its error is at most that of the plainest order of the same operations, both products of a
direction rounded by themselves and the eight of them added one after the other.  The kernel adds them
as a tree, which leaves 0.93 of that order's error in a model of both; over 24,576 reals the ratio
scatters by less than 0.01.

The flow: of U <- exp(X) U with |X| << 1 only the sum U + (exp(X) - 1) U is rounded at the size of U,
once per stage.  A real of size 1/2 to 1 is then off by at most 2^-54 per stage, with rms 2^-54 / sqrt(3); the
bound allows two such roundings per stage.
"""
import numpy as np
import pytest

import synth
from oracle import flow as F
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


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _force(U, eps):
    out, ax = np.empty_like(U), (3, 2, 1, 0)
    for mu in range(4):
        u, w = U[..., mu, :, :], 0
        for nu in set(range(4)) - {mu}:
            v = U[..., nu, :, :]
            vp, un = np.roll(v, -1, ax[mu]), np.roll(u, -1, ax[nu])
            um, vm, vpm = np.roll(u, 1, ax[nu]), np.roll(v, 1, ax[nu]), np.roll(vp, 1, ax[nu])
            w = w + _mm(u, _mm(vp, _mm(_dag(un), _dag(v))) + _mm(_dag(vpm), _mm(_dag(um), vm)))
        a = (w - _dag(w)) / 2
        tr = np.trace(a, axis1=-2, axis2=-1)[..., None, None] / LD(3)
        out[..., mu, :, :] = -eps * (a - tr * np.eye(3, dtype=CLD))
    return out


def _exp_times(X, U):
    term, out = U, U
    for k in range(1, 18):
        term = _mm(X, term) / LD(k)
        out = out + term
    return out


def test_flow_rounds_the_links_once_per_stage():
    dims, eps, steps = (4, 4, 2, 4), 0.02, 2
    U0 = synth.random_gauge(dims, 5, 0.1)
    ctx = M.mdwf_create(dims, 0)
    d = torch.from_numpy(U0).cuda()
    M.mdwf_wilson_flow_dev(ctx, d, eps, steps)
    got = d.cpu().numpy()
    M.mdwf_destroy(ctx)
    U = U0.astype(CLD)
    e = LD(eps)
    for _ in range(steps):
        z0 = _force(U, e)
        U = _exp_times(z0 / 4, U)
        z1 = _force(U, e)
        U = _exp_times(LD(8) / 9 * z1 - LD(17) / 36 * z0, U)
        z2 = _force(U, e)
        U = _exp_times(LD(3) / 4 * z2 - LD(8) / 9 * z1 + LD(17) / 36 * z0, U)
    i = np.arange(3)
    diag = U[..., i, i].real
    assert float(diag.min()) > 0.5
    err = (got[..., i, i].real - diag).astype(np.float64)
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(2 * 3 * steps) * 2.0 ** -54 / np.sqrt(3)


def test_flow_of_large_steps():
    """|X| above 1/2: exp(X) - 1 by squarings of a scaled one."""
    dims, eps = (4, 2, 2, 4), 0.5
    U = synth.random_gauge(dims, 6, 0.7)
    assert 3.0 * eps / 4 * np.sqrt(np.sum(np.abs(F.flow_generator(U)) ** 2, axis=(-2, -1))).max() > 1.0
    ctx = M.mdwf_create(dims, 0)
    d = torch.from_numpy(U).cuda()
    M.mdwf_wilson_flow_dev(ctx, d, eps, 1)
    got = d.cpu().numpy()
    M.mdwf_destroy(ctx)
    assert np.abs(got - F.wilson_flow(U, eps, 1)).max() <= 1e-12
