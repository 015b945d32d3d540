"""Measured cases: what a user of the library has it do, through its public entry points.

Each case is one call (or one short loop) of a valence-quark measurement on one gauge
configuration: batched propagator solves, the serving session, the FP64 operators, source
construction and smearing, the gradient flow of the links, and the residual-mass contraction.
Lattices and actions are the shapes of the paper's tuned ensembles and of this repository's
workloads and tests, down to a 4^3 x 8 lattice and up to 16^3 x 48; links are random SU(3)
matrices near the identity (as smooth as flowed links) or, for the flow, rough ones.

listed() gives the cases, draw(rng) another case of the same ranges, prepare(case, seed) what a
program holds before the call (context, links, action, inputs, output buffers), run(state) one
pass, work(case) the bytes and flops a pass cannot do without, and exact(case, seed) the same
outputs from plain 64-bit torch arithmetic where that takes seconds (None elsewhere).
"""
import math
import weakref

import torch

from paper_1701_07559_gb300 import mdwf as M

# (M5, b5, c5) of the tuned actions: a15m310, a12m310
ACTIONS = {'a15': (1.3, 1.5, 0.5), 'a12': (1.2, 1.25, 0.25)}


def listed():
    return [
        # the propagator of one configuration: 12 spin-colour point sources, L5 = 12, in one batch
        # (the a15m310 action; the largest call)
        dict(name='propagator 16x32', kind='solve', dims='16,16,16,32', L5=12, action='a15', n=12, masses='0.0158',
             precision='half', source='point', eps=0.1),
        # several masses in one batch (the a12m310 action's quark masses)
        dict(name='two masses 12x24', kind='solve', dims='12,12,12,24', L5=8, action='a12', n=6,
             masses='0.0126,0.0102', precision='half', source='z2', eps=0.1),
        # one right-hand side of a small lattice: short launches, where latency counts
        dict(name='one source 8x16', kind='solve', dims='8,8,8,16', L5=8, action='a12', n=1, masses='0.0102',
             precision='half', source='point', eps=0.1),
        # plain FP64 CG on the smallest lattice (the check of a new installation against a CPU code)
        dict(name='fp64 solve 4x8', kind='solve', dims='4,4,4,8', L5=4, action='a15', n=1, masses='0.1',
             precision='double', source='point', eps=0.3),
        # the serving loop: stochastic sources entering and leaving a session with continuous batching
        dict(name='session 8x24', kind='session', dims='8,8,8,24', L5=6, action='a15', slots=4, requests=6,
             masses='0.0102,0.0158,0.0216', precision='half', source='z2', eps=0.1),
        # the 5D operator on a whole lattice (residual checks, deflation set-up)
        dict(name='mobius 16x48', kind='apply', op='mobius', dims='16,16,16,48', L5=12, action='a15', dagger=0, eps=0.1),
        # the adjoint hopping term on a small ragged lattice (odd L5): the shortest call
        dict(name='hopping 6x10', kind='apply', op='dslash', dims='6,4,2,10', L5=5, action='a12', dagger=1, eps=0.5),
        # the even-odd operator on several fields in FP64
        dict(name='schur fp64 8x16', kind='schur', dims='8,8,8,16', L5=8, action='a12', n=4, masses='0.0126,0.0102',
             dagger=1, eps=0.1),
        # a 5D source from a 4D noise field
        dict(name='wall source 16x48', kind='source', dims='16,16,16,48', L5=12, action='a15', source='z2', eps=0.1),
        # gauge-covariant Gaussian smearing of a point source
        dict(name='smearing 16x48', kind='smear', dims='16,16,16,48', sigma=3.0, steps=30, eps=0.1),
        # gradient flow of rough links (ten of the steps to t = 1) and the plaquette it ends with
        dict(name='flow 16x48', kind='flow', dims='16,16,16,48', step=0.01, steps=10, eps=0.4),
        # residual-mass correlators of a propagator's 12 solutions
        dict(name='residual mass 16x48', kind='mres', dims='16,16,16,48', L5=12, n=12),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, sites):
    """Even extents whose product is near `sites` (at least 2 in each direction)."""
    for _ in range(200):
        d = [2 * max(1, round(_log(rng, 2, 16) / 2)) for _ in range(3)]
        t = 2 * max(1, round(sites / (d[0] * d[1] * d[2]) / 2))
        if 2 <= t <= 64 and t >= max(d) // 2:
            return ','.join(str(v) for v in d + [t])
    return '4,4,4,8'


def draw(rng):
    kind = rng.choice(['solve', 'solve', 'solve', 'session', 'apply', 'schur', 'source', 'smear', 'flow', 'mres'])
    act = rng.choice(['a15', 'a12'])
    L5 = rng.choice([4, 5, 6, 7, 8, 9, 10, 12, 12, 16])
    eps = round(rng.uniform(0.05, 0.3), 3)
    mass = ','.join('%.4f' % _log(rng, 0.01, 0.1) for _ in range(rng.choice([1, 2, 3])))
    if kind == 'solve':
        prec = rng.choice(['half', 'half', 'half', 'bf16', 'single', 'double'])
        n = rng.choice([1, 2, 3, 5, 8, 12])
        hi = 2000 if prec == 'double' else 40000
        dims = _dims(rng, _log(rng, 256, max(512, hi // n if prec == 'double' else 3e6 / (n * L5))))
        return dict(kind=kind, dims=dims, L5=L5, action=act, n=n, masses=mass, precision=prec,
                    source=rng.choice(['point', 'z2', 'gauss']), eps=eps)
    if kind == 'session':
        slots = rng.choice([1, 2, 3, 4])
        return dict(kind=kind, dims=_dims(rng, _log(rng, 256, 2e4)), L5=L5, action=act, slots=slots,
                    requests=slots + rng.choice([0, 1, 3]), masses=mass, precision=rng.choice(['half', 'half', 'single']),
                    source=rng.choice(['point', 'z2']), eps=eps)
    if kind == 'apply':
        return dict(kind=kind, op=rng.choice(['mobius', 'mobius', 'dslash']), dims=_dims(rng, _log(rng, 128, 1.6e5)),
                    L5=L5, action=act, dagger=rng.choice([0, 1]), eps=eps)
    if kind == 'schur':
        n = rng.choice([1, 2, 3, 5, 8, 12])
        return dict(kind=kind, dims=_dims(rng, _log(rng, 128, 6e4 / n)), L5=L5, action=act, n=n, masses=mass,
                    dagger=rng.choice([0, 1]), eps=eps)
    if kind == 'source':
        return dict(kind=kind, dims=_dims(rng, _log(rng, 256, 1.6e5)), L5=L5, action=act,
                    source=rng.choice(['point', 'z2', 'gauss']), eps=eps)
    if kind == 'smear':
        return dict(kind=kind, dims=_dims(rng, _log(rng, 256, 1.9e5)), sigma=round(rng.uniform(1.0, 4.0), 2),
                    steps=rng.randint(1, 40), eps=eps)
    if kind == 'flow':
        return dict(kind=kind, dims=_dims(rng, _log(rng, 256, 1.9e5)), step=rng.choice([0.01, 0.02, 0.05]),
                    steps=rng.randint(1, 12), eps=round(rng.uniform(0.2, 0.7), 3))
    return dict(kind='mres', dims=_dims(rng, _log(rng, 256, 1.6e5)), L5=L5, n=rng.choice([1, 3, 12]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _lat(case):
    return tuple(int(v) for v in case['dims'].split(','))


def _masses(case, n):
    m = [float(v) for v in case['masses'].split(',')]
    return [m[i % len(m)] for i in range(n)]


def _gen(seed, stream):
    g = torch.Generator(device='cuda')
    g.manual_seed(int(seed) * 16 + stream)
    return g


def _randc(shape, g):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device='cuda', generator=g))


def _links(dims, eps, seed):
    """Random SU(3) links [t, z, y, x, mu, 3, 3] near the identity: 1 + i eps H + (i eps H)^2 / 2 with H
    Hermitian and Gaussian, its first two rows orthonormalised, the third their conjugate cross product."""
    Lx, Ly, Lz, Lt = dims
    h = _randc((Lt, Lz, Ly, Lx, 4, 3, 3), _gen(seed, 1))
    a = (0.5j * eps) * (h + h.mH)
    a = torch.eye(3, dtype=torch.complex128, device='cuda') + a + 0.5 * (a[..., :, :, None] * a[..., None, :, :]).sum(-2)
    r0 = a[..., 0, :] / a[..., 0, :].abs().square().sum(-1, keepdim=True).sqrt()
    r1 = a[..., 1, :] - (r0.conj() * a[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], dim=-2).contiguous()


def _eta(case, dims, seed, k):
    """The k-th 4D source: a spin-colour point source, Z2 noise or a Gaussian field."""
    Lx, Ly, Lz, Lt = dims
    shape = (Lt, Lz, Ly, Lx, 4, 3)
    g = _gen(seed, 4 + k % 12)
    if case['source'] == 'point':
        eta = torch.zeros(shape, dtype=torch.complex128, device='cuda')
        at = seed % (Lx * Ly * Lz * Lt)
        eta.view(-1, 4, 3)[at, (k % 12) // 3, k % 3] = 1.0
        return eta
    if case['source'] == 'z2':
        return (2.0 * torch.randint(0, 2, shape, device='cuda', generator=g) - 1.0).to(torch.complex128)
    return _randc(shape, g)


def _inputs(case, seed):
    """(links, fields) of a case, without this library: the fields are what run() is given or, for the
    solves, the 4D sources."""
    dims = _lat(case)
    kind = case['kind']
    Lx, Ly, Lz, Lt = dims
    s4 = (Lt, Lz, Ly, Lx, 4, 3)
    if kind == 'mres':
        return None, [_randc((case['L5'],) + s4, _gen(seed, 4 + k)) for k in range(case['n'])]
    U = _links(dims, case['eps'], seed)
    if kind == 'flow':
        return U, []
    if kind == 'smear':
        return U, [_eta(dict(source='point'), dims, seed, seed % 12)]
    if kind == 'source':
        return U, [_eta(case, dims, seed, seed % 12)]
    if kind == 'apply':
        return U, [_randc((case['L5'],) + s4, _gen(seed, 2))]
    if kind == 'schur':
        return U, [_randc((case['L5'],) + s4, _gen(seed, 4 + k)) for k in range(case['n'])]
    n = case['n'] if kind == 'solve' else case['requests']
    return U, [_eta(case, dims, seed, k) for k in range(n)]


class State:
    """A program's handles and buffers; the library's context goes with it."""

    def __init__(self, case, ctx, ins=(), outs=()):
        self.case, self.ctx, self.ins, self.outs = case, ctx, list(ins), list(outs)
        self.session = self.opts = self.masses = None


def _release(ctx, sessions):
    torch.cuda.synchronize()
    for s in sessions:
        M.mdwf_session_destroy(s)
    M.mdwf_destroy(ctx)


# relative residual of every solve: a digit below the 1e-10 of the examples, so that the solution
# itself is defined to better than 1e-9
TOL = 1e-11


def prepare(case, seed):
    dims, kind = _lat(case), case['kind']
    U, fields = _inputs(case, seed)
    torch.cuda.synchronize()
    ctx = M.mdwf_create(dims, 0)
    sessions = []
    state = State(case, ctx)
    weakref.finalize(state, _release, ctx, sessions)
    if kind == 'flow':
        state.ins = [U]
        return state
    if kind != 'mres':
        M.mdwf_load_gauge(ctx, 0, U.cpu().numpy(), 1)
    if kind == 'smear':
        state.ins = fields
        return state
    L5 = case['L5']
    mf = _masses(case, 1)[0] if 'masses' in case else 0.0158
    if kind == 'mres':
        M.mdwf_load_gauge(ctx, 0, torch.eye(3, dtype=torch.complex128).expand(dims[3], dims[2], dims[1], dims[0], 4, 3, 3).contiguous().numpy(), 1)
        M.mdwf_set_action(ctx, 0, *ACTIONS['a15'], mf, L5)
        state.ins = fields
        return state
    M.mdwf_set_action(ctx, 0, *ACTIONS[case['action']], mf, L5)
    shape5 = (L5, dims[3], dims[2], dims[1], dims[0], 4, 3)

    def field():
        return torch.empty(shape5, dtype=torch.complex128, device='cuda')

    if kind in ('solve', 'session'):
        srcs = []
        for eta in fields:
            srcs.append(field())
            M.mdwf_make_source_dev(ctx, 0, eta, srcs[-1])
        state.ins, state.masses = srcs, _masses(case, len(srcs))
        state.outs = [field() for _ in srcs]
        state.opts = M.mdwf_default_opts(precision=case['precision'])
        if kind == 'session':
            state.session = M.mdwf_session_create(ctx, 0, case['slots'], TOL, opts=state.opts)
            sessions.append(state.session)
        return state
    state.ins = fields
    state.outs = [field() for _ in fields]
    if kind == 'source':
        state.outs = [field()]
    if kind == 'schur':
        state.masses = _masses(case, case['n'])
    return state


def run(state):
    case, ctx = state.case, state.ctx
    kind = case['kind']
    if kind == 'solve':
        M.mdwf_solve_batch_dev(ctx, 0, state.ins, state.outs, TOL, masses=state.masses, opts=state.opts)
        return state.outs
    if kind == 'session':
        sess, k, left = state.session, 0, len(state.ins)
        while left:
            while k < len(state.ins) and M.mdwf_session_occupied(sess) < case['slots']:
                M.mdwf_session_submit(sess, state.ins[k], state.masses[k], state.outs[k], k)
                k += 1
            M.mdwf_session_launch(sess)
            left -= len(M.mdwf_session_poll(sess))
        return state.outs
    if kind == 'apply':
        if case['op'] == 'mobius':
            M.mdwf_apply_mdwf_dev(ctx, 0, state.ins[0], state.outs[0], case['dagger'])
        else:
            M.mdwf_apply_dslash_dev(ctx, 0, state.ins[0], state.outs[0], -1, case['dagger'])
        return state.outs[0]
    if kind == 'schur':
        M.mdwf_apply_schur_batch_dev(ctx, 0, state.ins, state.outs, masses=state.masses, dagger=case['dagger'],
                                     precision='double')
        return state.outs
    if kind == 'source':
        M.mdwf_make_source_dev(ctx, 0, state.ins[0], state.outs[0])
        return state.outs[0]
    if kind == 'smear':
        eta = state.ins[0].clone()           # the smearing is in place: the point source stays in hand
        torch.cuda.current_stream().synchronize()
        M.mdwf_smear_source_dev(ctx, 0, eta, case['sigma'], case['steps'])
        return eta
    if kind == 'flow':
        U = state.ins[0].clone()             # in place as well: the unflowed links stay in hand
        torch.cuda.current_stream().synchronize()
        M.mdwf_wilson_flow_dev(ctx, U, case['step'], case['steps'])
        return U, M.mdwf_plaquette_dev(ctx, U)
    pp, j5 = M.mdwf_mres_correlators_dev(ctx, 0, state.ins)
    return pp, j5


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# CG iterations a solve takes at these masses and links, for the flops of a solve
ITERS = 250


def work(case):
    dims, kind = _lat(case), case['kind']
    V = dims[0] * dims[1] * dims[2] * dims[3]
    field4 = V * 24 * 8
    links = V * 4 * 18 * 8
    if kind == 'flow':
        # per link and stage: six staples of two matrix products, their product with the link, X^2 for the
        # exponential and its product with the link (198 flops each), and the sums
        return dict(bytes=2 * links, flops=case['steps'] * 3 * V * 4 * (15 * 198 + 400))
    if kind == 'smear':
        return dict(bytes=2 * field4 + links * 3 // 4, flops=case['steps'] * V * 4 * (6 * 66 + 48))
    L5 = case['L5']
    field5 = L5 * field4
    if kind == 'mres':
        return dict(bytes=case['n'] * 2 * field4, flops=case['n'] * V * 96)
    if kind == 'source':
        # only the two walls carry a source; the other slices are zero
        return dict(bytes=field4 + links + field5, flops=V * 1400)
    if kind == 'apply':
        return dict(bytes=2 * field5 + links, flops=L5 * V * (1320 + (144 if case['op'] == 'mobius' else 0)))
    if kind == 'schur':
        return dict(bytes=case['n'] * field5 + links, flops=case['n'] * L5 * V * (1320 + 150))
    n = case['n'] if kind == 'solve' else case['requests']
    per_unit = 4 * 1320 + 96 * L5 + 6 * 72 + 240
    return dict(bytes=n * 2 * field5 + links, flops=ITERS * n * (V // 2) * L5 * per_unit)


# ---------------------------------------------------------------------------
# the same outputs in plain 64-bit torch arithmetic
# ---------------------------------------------------------------------------
_AX = (-3, -4, -5, -6)     # axis of direction x, y, z, t in [..., t, z, y, x, spin, colour]
_GAMMA = [[[0, 0, 0, 1j], [0, 0, 1j, 0], [0, -1j, 0, 0], [-1j, 0, 0, 0]],
          [[0, 0, 0, -1], [0, 0, 1, 0], [0, 1, 0, 0], [-1, 0, 0, 0]],
          [[0, 0, 1j, 0], [0, 0, 0, -1j], [-1j, 0, 0, 0], [0, 1j, 0, 0]],
          [[0, 0, 1, 0], [0, 0, 0, 1], [1, 0, 0, 0], [0, 1, 0, 0]]]


def _gamma(mu):
    return torch.tensor(_GAMMA[mu], dtype=torch.complex128, device='cuda')


def _colour(W, psi):
    return (W[..., None, :, :] * psi[..., None, :]).sum(-1)


def _hop(U, psi, dagger=False):
    """H psi, or H^+ psi, with antiperiodic time."""
    out = torch.zeros_like(psi)
    one = torch.eye(4, dtype=torch.complex128, device='cuda')
    s = 1.0 if dagger else -1.0
    for mu in range(4):
        W = U[..., mu, :, :]
        if mu == 3:
            W = W.clone()
            W[-1] *= -1.0
        f = _colour(W, torch.roll(psi, -1, _AX[mu]))
        b = torch.roll(_colour(W.mH, psi), 1, _AX[mu])
        out += torch.einsum('ij,...jc->...ic', one + s * _gamma(mu), f)
        out += torch.einsum('ij,...jc->...ic', one - s * _gamma(mu), b)
    return out


def _p5(psi, m, dagger=False):
    """(P psi)_s = P_+ psi_{s-1} + P_- psi_{s+1} with wall factor -m; the adjoint exchanges the shifts."""
    dn, up = torch.roll(psi, 1, 0), torch.roll(psi, -1, 0)
    dn[0] *= -m
    up[-1] *= -m
    if dagger:
        dn, up = up, dn
    return torch.cat([dn[..., :2, :], up[..., 2:, :]], dim=-2)


class _Op:
    def __init__(self, U, action, m):
        self.U, self.m = U, m
        M5, self.b5, self.c5 = action
        self.d = 4.0 - M5

    def A(self, v, dagger=False):
        return (self.b5 * self.d + 1.0) * v + (self.c5 * self.d - 1.0) * _p5(v, self.m, dagger)

    def B(self, v, dagger=False):
        return self.b5 * v + self.c5 * _p5(v, self.m, dagger)

    def Ainv(self, v, dagger=False):
        """Solved along s: (alpha + beta S) y = x is a dense L5 x L5 system per chirality."""
        L5 = v.shape[0]
        eye = torch.eye(L5, dtype=torch.complex128, device='cuda')
        out = []
        for chi in (0, 1):
            f = torch.zeros((L5, L5, 4, 1), dtype=torch.complex128, device='cuda')
            f[:, :, 2 * chi] = eye[:, :, None]
            mat = self.A(f, dagger)[:, :, 2 * chi, 0]
            part = v[..., 2 * chi:2 * chi + 2, :]
            out.append(torch.linalg.solve(mat, part.reshape(L5, -1)).reshape(part.shape))
        return torch.cat(out, dim=-2)

    def D(self, v, dagger=False):
        if dagger:
            return self.A(v, True) - 0.5 * self.B(_hop(self.U, v, True), True)
        return self.A(v) - 0.5 * _hop(self.U, self.B(v))


def _cg(op, b):
    """x with D x = b by conjugate gradient on D^+ D x = D^+ b, to the rounding floor."""
    x = torch.zeros_like(b)
    r = op.D(b, True)
    p, g = r.clone(), r.abs().square().sum()
    stop = 1e-28 * g
    for _ in range(3000):
        if not bool(g > stop):
            break
        q = op.D(p)
        a = g / q.abs().square().sum()
        x += a * p
        r -= a * op.D(q, True)
        g, g0 = r.abs().square().sum(), g
        p = r + (g / g0) * p
    return x


def _source(U, eta, action, L5):
    M5, _, c5 = action
    w = torch.zeros((L5,) + tuple(eta.shape), dtype=torch.complex128, device='cuda')
    w[0, ..., :2, :] = eta[..., :2, :]
    w[-1, ..., 2:, :] = eta[..., 2:, :]
    return (1.0 - c5 * (4.0 - M5)) * w + 0.5 * c5 * _hop(U, w)


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _loop_sum(U, mu):
    """Sum of the six plaquettes that start with U_mu(x)."""
    ax = (3, 2, 1, 0)
    u = U[..., mu, :, :]
    acc = 0
    for nu in range(4):
        if nu == mu:
            continue
        v = U[..., nu, :, :]
        vp, un = torch.roll(v, -1, ax[mu]), torch.roll(u, -1, ax[nu])
        acc = acc + _mm(_mm(_mm(u, vp), un.mH), v.mH)
        um, vm, vpm = torch.roll(u, 1, ax[nu]), torch.roll(v, 1, ax[nu]), torch.roll(vp, 1, ax[nu])
        acc = acc + _mm(_mm(_mm(u, vpm.mH), um.mH), vm)
    return acc


def _force(U, step):
    out = torch.empty_like(U)
    eye = torch.eye(3, dtype=torch.complex128, device='cuda')
    for mu in range(4):
        w = _loop_sum(U, mu)
        a = 0.5 * (w - w.mH)
        out[..., mu, :, :] = -step * (a - (torch.diagonal(a, dim1=-2, dim2=-1).sum(-1) / 3.0)[..., None, None] * eye)
    return out


def _expm(X):
    """exp(X) by its Taylor series after scaling by 2^-4, squared four times (|X| is far below one here)."""
    Y = X / 16.0
    out = torch.eye(3, dtype=torch.complex128, device='cuda').expand(X.shape).clone()
    term = out.clone()
    for k in range(1, 13):
        term = _mm(term, Y) / k
        out = out + term
    for _ in range(4):
        out = _mm(out, out)
    return out


def exact(case, seed):
    dims, kind = _lat(case), case['kind']
    V = dims[0] * dims[1] * dims[2] * dims[3]
    if kind in ('solve', 'session') and V * case['L5'] * case.get('n', case.get('requests')) > 150000:
        return None
    U, fields = _inputs(case, seed)
    if kind == 'flow':
        for _ in range(case['steps']):
            z0 = _force(U, case['step'])
            U = _mm(_expm(0.25 * z0), U)
            z1 = _force(U, case['step'])
            U = _mm(_expm(8.0 / 9.0 * z1 - 17.0 / 36.0 * z0), U)
            z2 = _force(U, case['step'])
            U = _mm(_expm(0.75 * z2 - 8.0 / 9.0 * z1 + 17.0 / 36.0 * z0), U)
        plaq = 0.0
        ax = (3, 2, 1, 0)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                u, v = U[..., mu, :, :], U[..., nu, :, :]
                w = _mm(_mm(_mm(u, torch.roll(v, -1, ax[mu])), torch.roll(u, -1, ax[nu]).mH), v.mH)
                plaq += float(torch.diagonal(w, dim1=-2, dim2=-1).real.sum())
        return U, plaq / (18.0 * V)
    if kind == 'smear':
        eta = fields[0]
        k = case['sigma'] ** 2 / (4.0 * case['steps'])
        for _ in range(case['steps']):
            acc = (1.0 - 6.0 * k) * eta
            for mu in range(3):
                W = U[..., mu, :, :]
                acc = acc + k * (_colour(W, torch.roll(eta, -1, _AX[mu])) + torch.roll(_colour(W.mH, eta), 1, _AX[mu]))
            eta = acc
        return eta
    if kind == 'mres':
        L5, m = case['L5'], case['L5'] // 2
        pp = j5 = 0
        for x in fields:
            pp = pp + x[0, ..., 2:, :].abs().square().sum((1, 2, 3, 4, 5)) + x[-1, ..., :2, :].abs().square().sum((1, 2, 3, 4, 5))
            j5 = j5 + x[m - 1, ..., :2, :].abs().square().sum((1, 2, 3, 4, 5)) + x[m, ..., 2:, :].abs().square().sum((1, 2, 3, 4, 5))
        return pp.cpu().numpy(), j5.cpu().numpy()
    action, L5 = ACTIONS[case['action']], case['L5']
    if kind == 'source':
        return _source(U, fields[0], action, L5)
    if kind == 'apply':
        if case['op'] == 'dslash':
            return _hop(U, fields[0], bool(case['dagger']))
        return _Op(U, action, 0.0158).D(fields[0], bool(case['dagger']))
    if kind == 'schur':
        t, z, y, x = torch.meshgrid(*(torch.arange(n, device='cuda') for n in reversed(dims)), indexing='ij')
        even = (((t + z + y + x) % 2) == 0).to(torch.float64)[..., None, None]
        out = []
        for v, m in zip(fields, _masses(case, case['n'])):
            op, e = _Op(U, action, m), even * v
            if case['dagger']:
                w = 0.25 * op.B(_hop(U, op.Ainv(op.B((1 - even) * _hop(U, e, True), True), True), True), True)
                out.append(even * (op.A(e, True) - w))
            else:
                w = 0.25 * _hop(U, op.B(op.Ainv((1 - even) * _hop(U, op.B(e)))))
                out.append(even * (op.A(e) - w))
        return out
    return [_cg(_Op(U, action, m), _source(U, eta, action, L5)) for eta, m in zip(fields, _masses(case, len(fields)))]
