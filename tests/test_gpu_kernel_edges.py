"""The kernels at the sizes and arrays where their splits can go wrong: ragged tiles and slot
groups, arrays aligned to a double only, overlapping arrays, both sides of the lines that choose a form.

Elementwise bound of an FP64 result: C u max |oracle| with C = 16 (the roundings that reach one
component, as in test_gpu_parity).  A smearing step adds 6 products of 3 terms: 16 u per step.  A
correlator sums squares: u times (the terms of a component's square + the depth of the sums) of the
sum itself, below 64 u for these sizes.  A norm of n terms summed as a tree is exact to a few tens of u;
a residual of 1e-6 is the difference of terms of the size of |D| |x|, here below 1e4 |b|, so it agrees with
the oracle's to 1e4 u / 1e-6 x 100 = 1e-4.
"""
import numpy as np
import pytest

import synth
from oracle import mdwf_oracle as O

pytestmark = pytest.mark.gpu

M = torch = None
U64 = 2.0 ** -53
ACT = (1.3, 1.5, 0.5, 0.05)


def setup_module(module):
    global M, torch
    from paper_1701_07559_gb300 import build
    build.build()
    from paper_1701_07559_gb300 import mdwf
    import torch as _torch
    M, torch = mdwf, _torch


class Lat:
    def __init__(self, dims, L5, eps=0.5, seed=7):
        self.dims, self.L5 = dims, L5
        self.U = synth.random_gauge(dims, seed, eps)
        self.ctx = M.mdwf_create(dims, 0)
        M.mdwf_load_gauge(self.ctx, 0, self.U, 1)
        M.mdwf_set_action(self.ctx, 0, *ACT, L5)
        self.shape4 = tuple(reversed(dims)) + (4, 3)
        self.shape = (L5,) + self.shape4

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        M.mdwf_destroy(self.ctx)


def _odd(shape, a=None, shift=1):
    """A float64 view [..., 2] `shift` doubles into a buffer of its own."""
    n = int(np.prod(shape)) * 2
    buf = torch.zeros(n + 2 * shift + 2, dtype=torch.float64, device='cuda')
    v = buf[shift:shift + n].view(*shape, 2)
    if a is not None:
        v.copy_(torch.view_as_real(torch.from_numpy(a)))
    return v


def _c(v):
    return torch.view_as_complex(v.contiguous().clone()).cpu().numpy()


def _close(got, ref, c=16.0):
    assert np.abs(got - ref).max() <= c * U64 * np.abs(ref).max()


SIZES = [((2, 2, 2, 2), 2), ((6, 4, 2, 4), 3), ((4, 2, 6, 10), 7), ((2, 4, 2, 6), 32)]


@pytest.mark.parametrize('dims,L5', SIZES)
@pytest.mark.parametrize('arrays', ['odd', 'in place', 'overlapping'])
def test_operators_on_the_callers_arrays(dims, L5, arrays):
    with Lat(dims, L5) as L:
        psi = synth.gaussian_spinor(L.shape, 5)
        mask = O.parity_mask(dims)
        n = psi.size * 2

        def run(f):
            if arrays == 'odd':
                x, y = _odd(L.shape, psi), _odd(L.shape, shift=3)
            else:
                buf = torch.zeros(n + 8, dtype=torch.float64, device='cuda')
                x = buf[:n].view(*L.shape, 2)
                x.copy_(torch.view_as_real(torch.from_numpy(psi)))
                k = 0 if arrays == 'in place' else 5
                y = buf[k:k + n].view(*L.shape, 2)
            f(x, y)
            torch.cuda.synchronize()
            return _c(y)

        for dagger in (0, 1):
            h = O.hopping(L.U, psi, True, bool(dagger))
            for par in (-1, 0, 1):
                got = run(lambda x, y: M.mdwf_apply_dslash_dev(L.ctx, 0, x, y, par, dagger))
                _close(got, h if par < 0 else O.restrict(h, mask if par == 0 else 1 - mask))
            f = O.mobius_dag if dagger else O.mobius
            _close(run(lambda x, y: M.mdwf_apply_mdwf_dev(L.ctx, 0, x, y, dagger)), f(L.U, psi, *ACT))


@pytest.mark.parametrize('dims,L5', SIZES)
def test_fifth_dimension_operators(dims, L5):
    with Lat(dims, L5) as L:
        psi = synth.gaussian_spinor(L.shape, 6)
        for dagger in (False, True):
            for op, ref in ((0, O.op_A(psi, *ACT, dagger)), (1, O.op_B(psi, ACT[1], ACT[2], ACT[3], dagger)),
                            (2, O.op_A_inv(psi, *ACT, dagger))):
                _close(M.mdwf_apply_5d(L.ctx, 0, op, psi, int(dagger)), ref)


@pytest.mark.parametrize('dims,L5', SIZES)
@pytest.mark.parametrize('shift', [None, 0, 3])
def test_wall_source(dims, L5, shift):
    """Arrays aligned to a double; eta inside the source's array."""
    with Lat(dims, L5) as L:
        eta = synth.gaussian_spinor(L.shape4, 8)
        src = _odd(L.shape)
        if shift is None:
            e = _odd(L.shape4, eta)
        else:
            e = src.view(-1)[shift:shift + 2 * eta.size].view(*L.shape4, 2)
            e.copy_(torch.view_as_real(torch.from_numpy(eta)))
        M.mdwf_make_source_dev(L.ctx, 0, e, src)
        torch.cuda.synchronize()
        _close(_c(src), O.make_source(L.U, eta, ACT[0], ACT[2], L5))


@pytest.mark.parametrize('dims', [(2, 2, 2, 2), (6, 2, 4, 10), (10, 6, 2, 4)])
@pytest.mark.parametrize('slices', ['one', 'some', 'all'])
def test_smearing_of_some_slices(dims, slices):
    with Lat(dims, 2) as L:
        eta = synth.gaussian_spinor(L.shape4, 9)
        keep = {'one': [dims[3] - 1], 'some': [0, dims[3] - 1], 'all': range(dims[3])}[slices]
        for t in range(dims[3]):
            if t not in keep:
                eta[t] = 0
        d = _odd(L.shape4, eta)
        for n in (1, 4):
            d.copy_(torch.view_as_real(torch.from_numpy(eta)))
            M.mdwf_smear_source_dev(L.ctx, 0, d, 1.7, n)
            torch.cuda.synchronize()
            _close(_c(d), O.gaussian_smear(L.U, eta, 1.7, n), 16.0 * n)


@pytest.mark.parametrize('dims,L5', SIZES)
@pytest.mark.parametrize('n', [1, 3])
def test_residual_mass_correlators(dims, L5, n):
    with Lat(dims, L5) as L:
        xs = [synth.gaussian_spinor(L.shape, 20 + k) for k in range(n)]
        got = M.mdwf_mres_correlators_dev(L.ctx, 0, [_odd(L.shape, x) for x in xs])
        for a, b in zip(got, O.mres_correlators(xs)):
            assert np.all(np.abs(a - b) <= 64 * U64 * b)


@pytest.mark.parametrize('dims', [(2, 2, 2, 2), (6, 2, 4, 10)])
def test_flow_and_plaquette_of_unaligned_links(dims):
    """The same bits as on aligned arrays."""
    U = synth.random_gauge(dims, 10, 0.5)
    with Lat(dims, 2) as L:
        a = torch.from_numpy(U).cuda()
        b = _odd(U.shape, U)
        M.mdwf_wilson_flow_dev(L.ctx, a, 0.01, 2)
        M.mdwf_wilson_flow_dev(L.ctx, b, 0.01, 2)
        torch.cuda.synchronize()
        assert np.array_equal(a.cpu().numpy(), _c(b))
        assert M.mdwf_plaquette_dev(L.ctx, a) == M.mdwf_plaquette_dev(L.ctx, b)


@pytest.mark.parametrize('dims,L5,n', [((2, 2, 2, 2), 2, 67), ((4, 2, 2, 6), 5, 9), ((2, 4, 2, 2), 32, 14)])
@pytest.mark.parametrize('dagger', [0, 1])
def test_fp64_schur_of_many_systems(dims, L5, n, dagger):
    """More systems than one pack launch or one slot group of the FP64 hop takes."""
    with Lat(dims, L5) as L:
        masses = [0.02 + 0.01 * (k % 5) for k in range(n)]
        xs = [O.restrict(synth.gaussian_spinor(L.shape, 30 + k), O.parity_mask(dims)) for k in range(n)]
        outs = [_odd(L.shape) for _ in xs]
        M.mdwf_apply_schur_batch_dev(L.ctx, 0, [_odd(L.shape, x) for x in xs], outs, masses=masses, dagger=dagger,
                                     precision='double')
        torch.cuda.synchronize()
        f = O.schur_op_dag if dagger else O.schur_op
        for k in {0, 1, n // 2, n - 4, n - 3, n - 1}:
            _close(_c(outs[k]), f(L.U, xs[k], *ACT[:3], masses[k]))


@pytest.mark.parametrize('dims', [(8, 8, 8, 16), (8, 8, 6, 22), (2, 2, 2, 4)])
@pytest.mark.parametrize('precision', ['half', 'double'])
def test_norms_on_both_sides_of_the_cluster_sum(dims, precision):
    """4096 even sites are summed by one block per system, 4224 by a cluster."""
    with Lat(dims, 2, eps=0.2) as L:
        b = [synth.gaussian_spinor(L.shape, 40 + k) for k in range(2)]
        xs, st = M.mdwf_solve_batch(L.ctx, 0, b, 1e-6, opts=M.mdwf_default_opts(precision=precision))
        for k in range(2):
            res = O.true_residual(L.U, b[k], xs[k], *ACT)
            assert res <= 1e-6 and abs(st[k]['rel_true_resid'] - res) <= 1e-4 * res


@pytest.mark.parametrize('precision,n', [('half', 10), ('single', 6), ('double', 3)])
@pytest.mark.parametrize('chunk', [4, 7])
def test_grouped_steps_give_the_bits_of_single_ones(precision, n, chunk):
    """The vectors of n systems exceed the line of the grouped update of x, those of one don't.  The
    masses make the systems stop at different iterations of a group."""
    with Lat((8, 8, 8, 16), 8, eps=0.15) as L:
        masses = [0.05 + 0.05 * k for k in range(n)]
        b = [torch.from_numpy(synth.gaussian_spinor(L.shape, 50 + k)).cuda() for k in range(n)]
        opts = M.mdwf_default_opts(precision=precision, chunk=chunk)
        x = [torch.empty_like(v) for v in b]
        st = M.mdwf_solve_batch_dev(L.ctx, 0, b, x, 1e-8, masses=masses, opts=opts)
        assert len({s['iters'] for s in st}) > 1
        for k in (0, n - 1):
            y = torch.empty_like(b[k])
            one = M.mdwf_solve_batch_dev(L.ctx, 0, [b[k]], [y], 1e-8, masses=[masses[k]], opts=opts)
            torch.cuda.synchronize()
            assert one[0]['iters'] == st[k]['iters'] and torch.equal(x[k], y)


@pytest.mark.parametrize('dims,L5,n', [((2, 2, 2, 2), 3, 1), ((6, 4, 2, 6), 5, 4), ((4, 2, 2, 4), 32, 20)])
def test_fp64_solves_of_ragged_tiles(dims, L5, n):
    """FP64 updates with four lanes per unit: the same bits alone and in a batch, and the oracle's residual."""
    with Lat(dims, L5, eps=0.3) as L:
        masses = [0.05 + 0.02 * k for k in range(n)]
        b = [synth.gaussian_spinor(L.shape, 60 + k) for k in range(n)]
        opts = M.mdwf_default_opts(precision='double')
        xs, _ = M.mdwf_solve_batch(L.ctx, 0, b, 1e-9, masses=masses, opts=opts)
        for k in {0, n - 1}:
            assert O.true_residual(L.U, b[k], xs[k], *ACT[:3], masses[k]) <= 1e-9
            one, _ = M.mdwf_solve_batch(L.ctx, 0, [b[k]], 1e-9, masses=[masses[k]], opts=opts)
            assert np.array_equal(one[0], xs[k])


@pytest.mark.parametrize('n,L5,nsb', [(24, 12, 2), (24, 12, 1), (12, 6, 4), (12, 12, 4), (6, 5, 8)])
def test_half_hop_with_part_of_the_systems_per_block(n, L5, nsb):
    """Blocks that take a divisor of the systems to fill their warps: the bits of each system alone."""
    with Lat((4, 2, 2, 6), L5) as L:
        masses = [0.02 + 0.01 * (k % 7) for k in range(n)]
        xs = [torch.from_numpy(O.restrict(synth.gaussian_spinor(L.shape, 80 + k), O.parity_mask(L.dims))).cuda()
              for k in range(n)]
        for form in (M.HOP_DIRECT, M.HOP_PAIR_PF):
            for dagger in (0, 1):
                outs = [torch.empty_like(x) for x in xs]
                M.mdwf_apply_schur_batch_dev(L.ctx, 0, xs, outs, masses=masses, dagger=dagger, precision='half',
                                             hop_variant=form | (nsb << 8))
                for k in {0, n // 3, n // 2 - 1, n - 1}:
                    one = torch.empty_like(xs[k])
                    M.mdwf_apply_schur_batch_dev(L.ctx, 0, [xs[k]], [one], masses=[masses[k]], dagger=dagger,
                                                 precision='half', hop_variant=form | (1 << 8))
                    torch.cuda.synchronize()
                    assert torch.equal(one, outs[k])
