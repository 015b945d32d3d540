"""The grouped update of x (a step of four CG iterations at once) where the batch's vectors exceed its line: the
bits of single steps in every 16-bit storage type and Schur form that takes it, and in a session whose slots
fill and empty between chunks.  The batches check that the grouped kernels ran: equal systems take the same
chunks and updates alone and in a batch, so a batch puts more kernels on the GPU only through the groups.  The
session holds as many slots of the same types."""
import pytest

import synth

pytestmark = pytest.mark.gpu

M = torch = None
DIMS, L5, N = (8, 8, 8, 16), 8, 10        # 10 systems: 126 MB of 16-bit vectors with the FP32 solution; the line is 120 MB


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
    M.mdwf_load_gauge(c, 0, synth.random_gauge(DIMS, 7, 0.15), 1)
    M.mdwf_set_action(c, 0, 1.3, 1.5, 0.5, 0.05, L5)
    yield c
    torch.cuda.synchronize()
    M.mdwf_destroy(c)


def _source(k):
    return torch.from_numpy(synth.gaussian_spinor((L5,) + tuple(reversed(DIMS)) + (4, 3), 50 + k)).cuda()


def _solve(ctx, b, masses, opts):
    x = [torch.empty_like(v) for v in b]
    torch.cuda.synchronize()
    st = M.mdwf_solve_batch_dev(ctx, 0, b, x, 1e-8, masses=masses, opts=opts)
    torch.cuda.synchronize()
    return x, st


@pytest.mark.parametrize('precision,schur', [('half', 0), ('bf16', 0), ('half', 1), ('bf16', 1)])
def test_grouped_batch(ctx, precision, schur):
    opts = M.mdwf_default_opts(precision=precision, schur=schur, chunk=7)
    b = [_source(k) for k in range(N)]
    masses = [0.05 + 0.05 * k for k in range(N)]
    x, st = _solve(ctx, b, masses, opts)
    assert len({s['iters'] for s in st}) > 1
    for k in (0, N - 1):
        y, one = _solve(ctx, [b[k]], [masses[k]], opts)
        assert one[0]['iters'] == st[k]['iters'] and torch.equal(x[k], y[0])
    _, same = _solve(ctx, [b[0]] * N, [masses[0]] * N, opts)
    _, one = _solve(ctx, [b[0]], [masses[0]], opts)
    more = same[0]['kernel_launches'] - one[0]['kernel_launches']
    assert more > 0 and more % 2 == 0         # two groups (of 4 and 3) per chunk of 7


@pytest.mark.parametrize('precision', ['half', 'bf16'])
def test_grouped_session(ctx, precision):
    """Requests enter and leave while others iterate (two more slots in use each turn), in chunks of 7 iterations."""
    opts = M.mdwf_default_opts(precision=precision, chunk=7)
    reqs = [(_source(k % 4), 0.05 + 0.03 * (k % 7)) for k in range(N + 5)]

    def serve(slots, todo, first):
        sess = M.mdwf_session_create(ctx, 0, slots, 1e-8, opts=opts)
        out, left, k, turn = [torch.empty_like(b) for b, _ in todo], len(todo), 0, 0
        torch.cuda.synchronize()
        iters = {}
        while left:
            while k < len(todo) and M.mdwf_session_occupied(sess) < min(slots, first + 2 * turn):
                M.mdwf_session_submit(sess, todo[k][0], todo[k][1], out[k], k)
                k += 1
            M.mdwf_session_launch(sess, 7)
            done = M.mdwf_session_poll(sess)
            left -= len(done)
            turn += 1
            iters.update({tag: s['iters'] for tag, s in done})
        M.mdwf_session_destroy(sess)
        torch.cuda.synchronize()
        return out, iters

    out, iters = serve(N, reqs, 4)
    assert len(set(iters.values())) > 1
    for k in (0, 5, N - 1, N + 4):
        one, it = serve(1, [reqs[k]], 1)
        assert it[0] == iters[k] and torch.equal(one[0], out[k])
