#!/usr/bin/env python
"""Benchmark of the even-odd preconditioned Moebius domain-wall solve on GB300.

One step = one batched mixed-precision solve (fp16 storage with a power-of-two
scale per stored spinor, FP32 arithmetic, FP64 reliable updates / accumulator /
sums) of all right-hand sides of a workload, to a true FP64 residual
|b - D x| / |b| <= 1e-10.  The default workload ('16x48', the headline line) is
the 12 spin-colour point sources of 16^3 x 48, L5 = 12 with the a15m310 action
of the paper's Table II (M5 = 1.3, b5 = 1.5, c5 = 0.5, m_f = 0.0158) on
near-identity random SU(3) links smoothed by Wilson flow to t = 1.
``--workload`` selects the others: '4x8' (the oracle-sized plain FP64 case, timed
beside a full oracle solve), '24x64' (a12m310 action, 24 RHS over two masses in
one batch) and '48x64' (a12m130-shaped light quark).

Prints one JSON line (rank 0): solves/s, time to solution, iterations, updates,
the FP64 certificate and the oracle's check of a solution, the per-phase device
time, the dominant hop kernel against the HBM roofline (algorithmic bytes) and
the FP32 roofline, the FP64 single-RHS GPU CG on the same input, the oracle on
the host cores (one core and all cores), and the same metric end to end through
the host-pointer call.  ``--impl reference`` times the FP64 CPU oracle on a
bounded sample of the same workload instead.  Other modes: ``--mode op``
applies the batched Schur operator only (a short driver for kernel profiles);
``--mode serve`` serves a Poisson stream of solve requests over three resident
configurations and reports p50/p99 latency and solves/s.  ``--schur sym`` solves
through the symmetric Schur form.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "MDWF solves/s to 1e-10 (batched mixed vs FP64 CG); Dslash HBM GB/s; p50/p99"
# The workloads: synthetic stand-ins shaped like the paper's ensembles (Table II
# actions); '16x48' is the headline line.
WORKLOADS = {
    '4x8': dict(name='4^3x8 L5=4, exp(0.3 i H) links (no flow), one point source (spin 0, colour 0, origin), '
                     'plain FP64 CG, tol 1e-10',
                dims=(4, 4, 4, 8), L5=4, M5=1.3, b5=1.5, c5=0.5, masses=[0.1], seed=1, eps=0.3, flow_t=0.0,
                flow_eps=0.01, sources='point1', tol=1e-10, precision='double'),
    '16x48': dict(name='16^3x48 L5=12 a15m310-action, flowed SU(3), 12 spin-colour point sources, tol 1e-10',
                  dims=(16, 16, 16, 48), L5=12, M5=1.3, b5=1.5, c5=0.5, masses=[0.0158] * 12, seed=2, eps=0.4,
                  flow_t=1.0, flow_eps=0.01, sources='point12', tol=1e-10, precision='half'),
    '24x64': dict(name='24^3x64 L5=8 a12m310-action, flowed SU(3), 12 spin-colour point sources x m_f '
                       '{0.0126, 0.0102} in one 24-RHS batch, tol 1e-10',
                  dims=(24, 24, 24, 64), L5=8, M5=1.2, b5=1.25, c5=0.25, masses=[0.0126] * 12 + [0.0102] * 12,
                  seed=3, eps=0.4, flow_t=1.0, flow_eps=0.01, sources='point12', tol=1e-10, precision='half'),
    '48x64': dict(name='48^3x64 L5=8 a12m130-shaped light quark m_f=0.0022, flowed SU(3), spin-colour point '
                       'sources, tol 1e-10',
                  dims=(48, 48, 48, 64), L5=8, M5=1.2, b5=1.25, c5=0.25, masses=[0.0022] * 12, seed=4, eps=0.4,
                  flow_t=1.0, flow_eps=0.01, sources='point12', tol=1e-10, precision='half', batch_default=3),
}
WORKLOAD = WORKLOADS['16x48']
# algorithmic bytes of one stored real (input + output spinor, 24 reals each, and the
# link share 8 links x 18 reals of each output site over its L5 x N units; FP32 links here)
REAL_BYTES = {'half': 2, 'single': 4, 'bf16': 2, 'double': 8}
LINK_REAL_BYTES = {'half': 4, 'single': 4, 'bf16': 4, 'double': 8}
# what a hop launch of the solver moves in its storage format: input, output and, in two of the
# four launches of an iteration, the `same` field, plus the fp16 scale of each stored spinor
BYTES_PER_UNIT = {'half': 48 + 4, 'single': 96, 'bf16': 48, 'double': 192}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument('--gpus', type=int, default=1)
    ap.add_argument('--steps', type=int, default=5)
    ap.add_argument('--warmup', type=int, default=3)
    ap.add_argument('--impl', default='ours', choices=['ours', 'reference'])
    ap.add_argument('--precision', default=None, choices=['half', 'single', 'bf16', 'double'],
                    help="inner storage precision (default: the workload's)")
    ap.add_argument('--no-fp64', action='store_true', help='skip the FP64 single-RHS GPU CG comparison')
    ap.add_argument('--no-cpu', action='store_true', help='skip the oracle cpu_baseline sample')
    ap.add_argument('--workload', default='16x48', choices=sorted(WORKLOADS),
                    help='4x8: the oracle-sized FP64 case; 16x48 (default, the headline line): a15m310; '
                         '24x64: a12m310, 24 RHS over two masses; 48x64: a12m130-shaped light quark')
    ap.add_argument('--rhs', type=int, default=0, help='right-hand sides per step (0: the workload\'s)')
    ap.add_argument('--batch', type=int, default=0,
                    help='right-hand sides per solve call (0: the workload\'s; all of a step where they fit in HBM)')
    ap.add_argument('--mode', default='solve', choices=['solve', 'op', 'serve'],
                    help="'op': only apply the batched Schur operator (the solver's hop kernels), for profiling")
    ap.add_argument('--lattice', default=None, help="Lx,Ly,Lz,Lt instead of the workload's (profiling captures)")
    ap.add_argument('--hop-variant', type=int, default=0,
                    help='0 autotuned (CUDA-core forms), 1 CUDA-core direct loads, 2 CUDA-core staged, '
                         '3 tensor-core (fp16), 4 autotuned including the staged and tensor-core forms, '
                         '6 CUDA-core direct, one unit per thread, 7 as 1 with prefetching (fp16)')
    ap.add_argument('--nsb', type=int, default=0, help='sites per thread block (0: chosen by the library)')
    ap.add_argument('--link-recon', type=int, default=18, choices=[18, 12],
                    help='reals per link read by the inner hops (12: third row rebuilt in the kernel)')
    ap.add_argument('--schur', default='asym', choices=['asym', 'sym'],
                    help='Schur form of the solve: asymmetric (default) or symmetric')
    ap.add_argument('--profile-steps', default='all', choices=['all', 'extra'],
                    help="'all': the timed solves carry the per-launch hop events and phase timers; "
                         "'extra': the timed solves run without them and one more solve is profiled")
    ap.add_argument('--requests', type=int, default=300, help='serve mode: requests per arrival rate')
    ap.add_argument('--rates', default='0.5,0.9,1.2', help='serve mode: arrival rates as fractions of capacity')
    ap.add_argument('--serve-lattices', default='16,16,16,48:12;24,24,24,64:8;32,32,32,96:6',
                    help='serve mode: the resident configurations, Lx,Ly,Lz,Lt:L5 separated by ;')
    ap.add_argument('--slots', type=int, default=12, help='serve mode: maximum slots of one session')
    ap.add_argument('--hbm-budget-gb', type=float, default=0.0, help='serve mode: HBM budget (0: 85%% of free)')
    ap.add_argument('--profile-region', action='store_true',
                    help='bracket the timed solves with cudaProfilerStart/Stop (for ncu --profile-from-start off)')
    ap.add_argument('--priorities', action='store_true',
                    help='serve mode: rank the configurations\' streams by the cost of one request')
    return ap.parse_args()


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ('index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,'
              'clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,'
              'clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap')

    def __init__(self, device_index):
        self.dev = str(device_index)
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(['nvidia-smi', '-i', self.dev, '--query-gpu=' + self.FIELDS,
                                          '--format=csv,noheader,nounits', '-lms', '200'],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.th = threading.Thread(target=self._read, daemon=True)
            self.th.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {'sm_mhz': None, 'sm_max_mhz': None, 'reasons': ['nvidia-smi unavailable']}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, power, reasons = [], None, [], set()
        names = ['hw_slowdown', 'hw_thermal_slowdown', 'sw_thermal_slowdown', 'sw_power_cap']
        for ln in self.lines:
            f = [x.strip() for x in ln.split(',')]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
                power.append(float(f[3]))
            except ValueError:
                continue
            for name, v in zip(names, f[5:9]):
                if v.lower() == 'active':
                    reasons.add(name)
        return {'sm_mhz': statistics.median(sm) if sm else None, 'sm_max_mhz': smax,
                'reasons': sorted(reasons), 'samples': len(sm), 'power_w_max': max(power) if power else None}


# ---------------------------------------------------------------------------
# helpers
# ---------------------------------------------------------------------------
def dist_setup(args):
    rank = int(os.environ.get('RANK', '0'))
    world = int(os.environ.get('WORLD_SIZE', '1'))
    local = int(os.environ.get('LOCAL_RANK', '0'))
    return rank, world, local


def measured_peaks():
    try:
        with open(os.path.join(ROOT, 'MEASURED_PEAKS.json')) as f:
            p = json.load(f)
        return float(p['hbm_gbs']), 'measured'
    except (OSError, KeyError, ValueError):
        return 6800.0, 'fallback'


HOP_SOURCES = ('hop_pair.cu', 'hop_common.cuh', 'mdwf_internal.h')


def hop_sources_sha256():
    import hashlib
    h = hashlib.sha256()
    for name in HOP_SOURCES:
        with open(os.path.join(ROOT, 'paper_1701_07559_gb300', 'csrc', name), 'rb') as f:
            h.update(f.read())
    return h.hexdigest()


def ncu_traffic(kernel_key):
    """Per-launch DRAM bytes of the hop kernel from the committed ncu record, if the
    kernel's sources have not changed since it was captured (else None)."""
    path = os.path.join(ROOT, 'profiles', 'hop_pair_kernel_ncu.json')
    try:
        with open(path) as f:
            rec = json.load(f)
        if rec.get('sources_sha256') != hop_sources_sha256():
            return None
        return rec['workloads'][kernel_key]['dram_bytes_per_launch']
    except (OSError, KeyError, ValueError):
        return None


def flowed_links(M, dims, seed, eps, flow_t, flow_eps, device=0):
    """Random links exp(i eps H) (host generator) flowed to flow_t on the device."""
    import synth
    if flow_t <= 0:
        return synth.random_gauge(dims, seed, eps)
    ctx = M.mdwf_create(dims, device)
    try:
        return M.flowed_gauge_dev(ctx, synth.random_gauge(dims, seed, eps), flow_t, flow_eps)
    finally:
        M.mdwf_destroy(ctx)


def workload(args):
    W = dict(WORKLOADS[args.workload])
    W['key'] = args.workload
    W['precision'] = args.precision or W['precision']
    if args.lattice:    # a smaller lattice of the same workload (profiling captures)
        W['dims'] = tuple(int(v) for v in args.lattice.split(','))
        W['name'] = W['name'] + ' (lattice %s)' % args.lattice
    n = args.rhs or W.get('rhs_default', len(W['masses']))
    W['masses'] = [W['masses'][k % len(W['masses'])] for k in range(n)]
    W['nsrc'] = n
    W['batch'] = min(n, args.batch or W.get('batch_default', n))
    W['lattice'] = '%d^3x%d' % (W['dims'][0], W['dims'][3]) if W['dims'][0] == W['dims'][1] == W['dims'][2] \
        else 'x'.join(str(d) for d in W['dims'])
    return W


def source_4d(W, k):
    """k-th 4D source of the workload: the spin-colour point sources at the origin,
    spin k // 3 and colour k % 3 of the k % 12-th (the 12 repeat for each mass)."""
    import synth
    j = k % 12 if W['sources'] == 'point12' else 0
    return synth.point_source_4d(W['dims'], j // 3, j % 3)


def make_inputs(M, ctx, W):
    return [M.mdwf_make_source(ctx, 0, source_4d(W, k)) for k in range(W['nsrc'])]


def _oracle_apply_worker(task):
    """One FP64 oracle Schur-operator application (run in a spawned process)."""
    import synth
    from oracle import mdwf_oracle as O
    W, U, seed = task
    Lx, Ly, Lz, Lt = W['dims']
    ev = O.parity_mask(W['dims'])
    psi = O.restrict(synth.gaussian_spinor((W['L5'], Lt, Lz, Ly, Lx, 4, 3), seed), ev)
    t0 = time.perf_counter()
    O.schur_op(U, psi, W['M5'], W['b5'], W['c5'], W['masses'][0])
    return time.perf_counter() - t0


def oracle_timing(W, U, n_iter, procs):
    """The oracle as it stands on the host cores: one Schur-operator application
    on one core, then `procs` of them at once (one per process, spawned); a CGNR
    iteration is two applications, a solve n_iter iterations."""
    import multiprocessing as mp
    t1 = _oracle_apply_worker((W, U, 1))
    out = {'apply_s_1core': t1, 'solves_per_s_1core': 1.0 / (2.0 * t1 * n_iter) if n_iter else None}
    if procs > 1:
        ctx = mp.get_context('spawn')
        t0 = time.perf_counter()
        with ctx.Pool(procs) as pool:
            pool.map(_oracle_apply_worker, [(W, U, 1 + k) for k in range(procs)])
        tp = time.perf_counter() - t0
        out.update({'procs': procs, 'apply_wall_s_all': tp,
                    'solves_per_s_all': procs / (2.0 * tp * n_iter) if n_iter else None})
    return out


def host_mem_available():
    """MemAvailable of the host in bytes (None where /proc/meminfo is absent)."""
    try:
        with open('/proc/meminfo') as fh:
            for line in fh:
                if line.startswith('MemAvailable:'):
                    return int(line.split()[1]) * 1024
    except OSError:
        pass
    return None


def oracle_procs(W, n):
    """Processes for the all-cores oracle leg: one per core, at most one per RHS
    and 16, and at most as many as half the free host memory holds at about
    twenty full 5D FP64 fields per process (the oracle's temporaries)."""
    procs = min(host_cores(), n, 16)
    avail = host_mem_available()
    if avail:
        per = 20 * W['L5'] * W['dims'][0] * W['dims'][1] * W['dims'][2] * W['dims'][3] * 12 * 16
        procs = max(1, min(procs, int(0.5 * avail // per)))
    return procs


def host_cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


# ---------------------------------------------------------------------------
# reference arm: the FP64 CPU oracle
# ---------------------------------------------------------------------------
def run_reference(args):
    rank, world, _ = dist_setup(args)
    if rank != 0:
        return 0
    import numpy as np  # noqa: F401
    import synth
    W = workload(args)
    U = synth.flowed_gauge(W['dims'], W['seed'], W['eps'], W['flow_t'], W['flow_eps']) if W['flow_t'] > 0 \
        else synth.random_gauge(W['dims'], W['seed'], W['eps'])
    rec = iteration_record(W['key'])
    n_iter = rec['fp64_cgnr_iters'] if rec else None
    for _ in range(max(0, min(args.warmup, 1))):
        _oracle_apply_worker((W, U, 1))
    times = [_oracle_apply_worker((W, U, 1)) for _ in range(max(1, args.steps))]
    t = statistics.median(times)
    per_solve = 2.0 * t * n_iter if n_iter else None
    value = (1.0 / per_solve) if per_solve else None
    sample = ('one FP64 oracle Schur-operator application (numpy, one RHS, the full %s x %d lattice, one core) '
              'per step; a CGNR iteration is two such applications; solves/s = 1/(2 t n_iter) with n_iter = %s, '
              'the iteration count of FP64 CGNR on this workload' % (W['lattice'], W['L5'], n_iter))
    line = {'impl': 'reference', 'metric': METRIC, 'value': value, 'unit': 'solves/s', 'n_gpus': args.gpus,
            'steps': len(times), 'warmup': args.warmup, 'ms_per_step': 1e3 * statistics.mean(times),
            'higher_is_better': True, 'scaling': 'weak', 'vs_baseline': None, 'dtype': 'f64', 'data': 'synthetic',
            'config': config_of(W, W['nsrc'], 'single process'),
            'cpu_baseline': {'value': value, 'unit': 'solves/s', 'cores': 1, 'kind': 'oracle', 'sample': sample},
            'e2e': {'value': value, 'unit': 'solves/s', 'h2d_bytes_per_step': 0, 'd2h_bytes_per_step': 0}}
    print(json.dumps(line), flush=True)
    return 0


def cgnr_flops_per_unit_iteration(L5):
    """Algorithmic flops of one CGNR iteration on the asymmetric Schur operator per
    (half-lattice site, slice, RHS) unit: four Wilson hops of 1320, two A^-1 of
    48 L5, four B and two A of 72, and about 240 in the vector updates."""
    return 4 * 1320 + 2 * 48 * L5 + 6 * 72 + 240


def solver_tflops(vh, L5, iters, seconds):
    """Sustained solver TFLOP/s of a step: the algorithmic flops of every RHS's
    own iterations (vh * L5 units each) over the step's device time."""
    return cgnr_flops_per_unit_iteration(L5) * vh * L5 * sum(iters) / seconds / 1e12


def iteration_record(key='16x48'):
    """FP64 CGNR iteration count of the workload (profiles/workload_iterations.json,
    written from bench lines), used to scale oracle timing samples to solves/s."""
    try:
        with open(os.path.join(ROOT, 'profiles', 'workload_iterations.json')) as f:
            return json.load(f).get(key)
    except (OSError, ValueError):
        return None


def config_of(W, n, parallelism):
    """The workload as both arms name it (the same keys and values at one process)."""
    Lx, Ly, Lz, Lt = W['dims']
    units = (Lx * Ly * Lz * Lt // 2) * W['L5'] * W.get('batch', n)
    return {'workload': W['name'], 'lattice': W['lattice'], 'L5': W['L5'], 'rhs_per_step': n,
            'action': {'M5': W['M5'], 'b5': W['b5'], 'c5': W['c5'], 'masses': sorted(set(W['masses']))},
            'gauge': 'exp(i %.1f H)%s' % (W['eps'], ', Wilson flow t=%g (RK3, eps %g, FP64)' % (
                W['flow_t'], W['flow_eps']) if W['flow_t'] > 0 else ', no flow'),
            'precision': W['precision'], 'parallelism': parallelism,
            'l2': l2_note(6 * units * BYTES_PER_UNIT[W['precision']])}


def l2_note(nbytes):
    if nbytes > 129e6:
        return 'inputs larger than L2: %.2f GB of inner vectors per batch' % (nbytes / 1e9)
    return 'inputs fit in L2: %.2f MB of inner vectors per batch, no flush between steps' % (nbytes / 1e6)


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------
def run_ours(args):
    import numpy as np
    import torch
    rank, world, local = dist_setup(args)
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group('nccl')
    import __graft_entry__
    __graft_entry__.build()
    from paper_1701_07559_gb300 import mdwf as M
    W = workload(args)
    prec = W['precision']
    U = flowed_links(M, W['dims'], W['seed'], W['eps'], W['flow_t'], W['flow_eps'], local)
    ctx = M.mdwf_create(W['dims'], local)
    M.mdwf_load_gauge(ctx, 0, U, 1)
    M.mdwf_set_action(ctx, 0, W['M5'], W['b5'], W['c5'], W['masses'][0], W['L5'])
    n = W['nsrc']
    masses = W['masses']
    stream = torch.cuda.current_stream()
    # the RHS of a step go through the solver in batches of W['batch'] (all at once
    # where their FP64 source and solution fields fit in HBM next to the solver)
    batch = W['batch']
    chunks = [list(range(i, min(i + batch, n))) for i in range(0, n, batch)]
    Lx, Ly, Lz, Lt = W['dims']
    if len(chunks) == 1:
        srcs = make_inputs(M, ctx, W)
        dsrc = [torch.from_numpy(s).to('cuda') for s in srcs]
        eta = None
    else:
        # batches share `batch` device source and solution fields; each batch's 5D
        # sources are built on the device (mdwf_make_source_dev) from its 4D point
        # sources, inside the step
        srcs = None
        dsrc = [torch.empty((W['L5'], Lt, Lz, Ly, Lx, 4, 3), dtype=torch.complex128, device='cuda')
                for _ in range(batch)]
        eta = torch.zeros((Lt, Lz, Ly, Lx, 4, 3), dtype=torch.complex128, device='cuda')
    dx = [torch.empty_like(s) for s in dsrc]

    def load_chunk(c):
        if eta is None:
            return
        for j, k in enumerate(c):
            sp = (k % 12 if W['sources'] == 'point12' else 0)
            eta.zero_()
            eta[0, 0, 0, 0, sp // 3, sp % 3] = 1.0
            M.mdwf_make_source_dev(ctx, 0, eta, dsrc[j], stream=stream)
    schur = 1 if args.schur == 'sym' else 0
    opts = M.mdwf_default_opts(precision=prec, profile=1, hop_variant=args.hop_variant, nsb=args.nsb, schur=schur,
                               link_recon=args.link_recon)
    opts_timed = opts if args.profile_steps == 'all' else M.mdwf_default_opts(
        precision=prec, profile=0, hop_variant=args.hop_variant, nsb=args.nsb, schur=schur,
        link_recon=args.link_recon)

    def barrier():
        if dist is not None:
            dist.barrier()

    def solve(o):
        # per-RHS stats of the step, batch after batch (a list per batch)
        out = []
        for c in chunks:
            load_chunk(c)
            out.append(M.mdwf_solve_batch_dev(ctx, 0, dsrc[:len(c)], dx[:len(c)], W['tol'],
                                              masses=[masses[k] for k in c], opts=o, stream=stream))
        return out

    for _ in range(args.warmup):
        solve(opts)
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(local)
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    stats = []
    if args.profile_region:
        torch.cuda.profiler.start()
    t0 = time.perf_counter()
    for i in range(args.steps):
        ev[i][0].record(stream)
        stats.append(solve(opts_timed))
        ev[i][1].record(stream)
    torch.cuda.synchronize()
    barrier()
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    if args.profile_region:
        torch.cuda.profiler.stop()
    clk = clocks.stop()
    timed = stats
    if args.profile_steps == 'extra':
        stats = [solve(opts)]
    step_ms = [a.elapsed_time(b) for a, b in ev]
    from paper_1701_07559_gb300 import replicas
    # independent replicas: solves of all ranks over the slowest rank's time
    value = replicas.job_throughput(n * args.steps, sum(step_ms) / 1e3, dist, 'cuda')
    total_s = replicas.max_over_ranks(sum(step_ms) / 1e3, dist, 'cuda')

    # correctness of what was timed: every system of the last step reports its
    # FP64 full-lattice residual (the library's certificate)
    last = [s for ch in timed[-1] for s in ch]
    resid_max = max(s['rel_true_resid'] for s in last)
    assert all(s['converged'] for s in last), last
    iters = [s['iters'] for s in last]

    # dominant kernel: the inner-precision hop (4 launches per CG iteration)
    hop_launches = sum(ch[0]['hop_launches'] for st in stats for ch in st)
    hop_ms = sum(ch[0]['hop_ms'] for st in stats for ch in st)
    units = timed[-1][0][0]['hop_units']
    L5, V = W['L5'], W['dims'][0] * W['dims'][1] * W['dims'][2] * W['dims'][3]
    hop_avg_s = (hop_ms / hop_launches) / 1e3 if hop_launches else None
    # algorithmic bytes: input and output spinor (24 reals each) per unit, plus
    # 8 links of 18 reals per output site shared by its L5 x N units
    w, wg = REAL_BYTES[prec], LINK_REAL_BYTES[prec]
    link_reals = args.link_recon if prec != 'double' else 18
    bytes_per_unit = 48 * w + 8 * link_reals * wg / (L5 * len(chunks[0]))
    bytes_per_launch = units * bytes_per_unit
    # what the launches store and load: + the fp16 scales, + `same` in half of the launches
    stored_per_launch = units * 2.5 * BYTES_PER_UNIT[prec] + (V // 2) * 8 * link_reals * wg
    achieved = bytes_per_launch / hop_avg_s / 1e9 if hop_avg_s else None
    peak, peak_kind = measured_peaks()
    gflops = units * 1320 / hop_avg_s / 1e9 if hop_avg_s else None
    # FP32 CUDA-core peak at the measured clock: 152 SMs x 128 lanes x 2 flops (FMA)
    mhz = clk.get('sm_mhz') or 2070.0
    fp32_peak_tflops = 152 * 128 * 2 * mhz * 1e6 / 1e12
    gpu_launches = sum(ch[0]['kernel_launches'] for st in timed for ch in st)
    tuned = M.mdwf_autotune(ctx, 0, len(chunks[0]), prec, include_tensor_core=args.hop_variant == 4) \
        if args.hop_variant in (0, 4) and args.nsb == 0 else None
    variant = tuned['hop_variant'] if tuned else (args.hop_variant or 1)
    kernel_name = {1: 'hop_pair_kernel' if prec != 'double' else 'hop64_kernel',
                   2: 'hop_staged_kernel', 3: 'hop_mma_kernel', 6: 'hop_fast_kernel'}.get(variant, 'hop_pair_kernel')
    hop_form = 'prefetching' if (variant == 7 and prec == 'half' and args.link_recon == 18) else 'plain'

    field_bytes = L5 * V * 24 * 8
    # the first solution of the last batch and its source, on the host, for the
    # oracle's checks below (the device fields are freed before the end-to-end leg)
    x0 = b0 = None
    m0 = masses[chunks[-1][0]]
    if rank == 0 and not args.no_cpu and world == 1:
        x0 = dx[0].cpu().numpy()
        b0 = srcs[chunks[-1][0]] if srcs is not None else dsrc[0].cpu().numpy()

    # plain FP64 single-RHS GPU CG on the same input, like for like: device
    # pointers, one warm-up solve, CUDA events around each timed solve
    fp64 = None
    if not args.no_fp64:
        o64 = M.mdwf_default_opts(precision='double', hop_variant=1)
        one = lambda: M.mdwf_solve_batch_dev(ctx, 0, dsrc[:1], dx[:1], W['tol'], masses=[m0], opts=o64,
                                             stream=stream)
        one()
        k64 = max(1, min(args.steps, 2))
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k64)]
        for a, b in evs:
            a.record(stream)
            st64 = one()
            b.record(stream)
        torch.cuda.synchronize()
        t64 = statistics.mean(a.elapsed_time(b) for a, b in evs) / 1e3
        fp64 = {'solves_per_s': 1.0 / t64, 'time_s': t64, 'iters': st64[0]['iters'], 'timed_solves': k64,
                'rel_true_resid': st64[0]['rel_true_resid'],
                'precision': 'FP64 storage and arithmetic, 1 RHS, device pointers, warmed'}

    # end to end through the host-pointer C ABI call, pinned host buffers.  Batched
    # workloads: the first batch (at most as many RHS as 40 % of the free host
    # memory holds twice), after the device fields are freed for the library's copies
    e2e_idx = chunks[0]
    if eta is None:
        pin_src = [torch.from_numpy(s).pin_memory().numpy() for s in srcs]
    else:
        avail = host_mem_available()
        if avail:
            e2e_idx = e2e_idx[:max(1, min(len(e2e_idx), int(0.4 * avail // (2 * field_bytes))))]
        load_chunk(e2e_idx)
        pin_src = []
        for j in range(len(e2e_idx)):
            t = torch.empty(tuple(dsrc[j].shape), dtype=torch.complex128, pin_memory=True)
            t.copy_(dsrc[j])
            pin_src.append(t.numpy())
        del dsrc, dx
        torch.cuda.empty_cache()
    pin_x = [torch.empty(s.shape, dtype=torch.complex128).pin_memory().numpy() for s in pin_src]
    m_e2e = [masses[k] for k in e2e_idx]
    opts_e2e = M.mdwf_default_opts(precision=prec, hop_variant=args.hop_variant, nsb=args.nsb, schur=schur,
                                   link_recon=args.link_recon)
    M.mdwf_solve_batch(ctx, 0, pin_src, W['tol'], masses=m_e2e, opts=opts_e2e, out=pin_x)
    torch.cuda.synchronize()
    barrier()
    e2e_t = []
    for _ in range(args.steps):
        t1 = time.perf_counter()
        M.mdwf_solve_batch(ctx, 0, pin_src, W['tol'], masses=m_e2e, opts=opts_e2e, out=pin_x)
        e2e_t.append(time.perf_counter() - t1)
    e2e_value = replicas.job_throughput(len(e2e_idx) * args.steps, sum(e2e_t), dist, 'cuda')
    del pin_src, pin_x

    out = None
    if rank == 0:
        cpu = None
        oracle_check = None
        if not args.no_cpu and world == 1:
            # the oracle as it stands, on the host cores: a full solve where it takes
            # seconds (the 4^3 x 8 workload), else a bounded sample of applications
            from oracle import mdwf_oracle as O
            from oracle import sampled
            if V <= 4096:
                t1 = time.perf_counter()
                xref, it_or = O.solve_schur(U, b0, W['M5'], W['b5'], W['c5'], m0, tol=W['tol'])
                t_or = time.perf_counter() - t1
                cpu = {'value': 1.0 / t_or, 'unit': 'solves/s', 'cores': 1, 'kind': 'oracle',
                       'sample': 'one full FP64 oracle solve (Schur CGNR, %d iterations) of the first source, '
                                 '%.2f s on one host core' % (it_or, t_or)}
                oracle_check = {'err_vs_oracle_solution': float(np.linalg.norm((x0 - xref).ravel()) /
                                                                np.linalg.norm(xref.ravel())),
                                'oracle_true_residual': float(O.true_residual(U, b0, x0, W['M5'], W['b5'],
                                                                              W['c5'], m0))}
            else:
                n_iter = fp64['iters'] if fp64 else (iteration_record(W['key']) or {}).get('fp64_cgnr_iters')
                ot = oracle_timing(W, U, n_iter, oracle_procs(W, n))
                cpu = {'value': ot['solves_per_s_1core'], 'unit': 'solves/s', 'cores': 1, 'kind': 'oracle',
                       'sample': ('one FP64 oracle Schur-operator application on one RHS of this workload (%.1f s '
                                  'on one core); a CGNR iteration is two, a solve %s iterations (FP64 CGNR here)'
                                  % (ot['apply_s_1core'], n_iter)),
                       'all_cores': {'value': ot.get('solves_per_s_all'), 'cores': ot.get('procs'),
                                     'apply_wall_s': ot.get('apply_wall_s_all'),
                                     'sample': 'the same application in %s spawned processes at once'
                                               % ot.get('procs')},
                       'host_cores': host_cores()}
                # the oracle's own D on the first solution at sampled sites: |b - D x|(site) / |b|
                rng = np.random.default_rng(W['seed'])
                sites = [(0, 0, 0, 0)] + [tuple(int(rng.integers(d)) for d in W['dims']) for _ in range(3)]
                bn = np.linalg.norm(b0.ravel())
                worst = max(np.linalg.norm(sampled.residual_at_site(U, b0, x0, s, W['M5'], W['b5'], W['c5'],
                                                                    m0).ravel()) / bn for s in sites)
                oracle_check = {'sampled_sites': len(sites), 'max_site_residual_over_norm_b': float(worst),
                                'note': 'no oracle solve is feasible at this size; the error against the solution '
                                        'is bounded by kappa x 1e-10'}
        lat = sorted(step_ms)
        p99 = lat[min(len(lat) - 1, int(np.ceil(0.99 * len(lat))) - 1)]
        phases = {k: statistics.mean(sum(ch[0]['phase_ms'][k] for ch in st) for st in stats) for k in M.PHASES}
        out = {
            'metric': METRIC, 'value': value, 'unit': 'solves/s', 'n_gpus': world, 'steps': args.steps,
            'warmup': args.warmup, 'ms_per_step': total_s * 1e3 / args.steps, 'higher_is_better': True,
            'scaling': 'weak', 'vs_baseline': None, 'dtype': 'f64' if prec == 'double' else 'f32',
            'storage': {'half': 'fp16 + power-of-two scale per (site, slice, RHS)', 'single': 'fp32',
                        'bf16': 'bf16', 'double': 'fp64'}[prec] +
                       ' inner vectors; FP64 accumulator, reliable updates and sums',
            'data': 'synthetic',
            'config': config_of(W, n, 'replicas' if world > 1 else 'single process'),
            'solver': {'rhs_per_batch': len(chunks[0]), 'batches_per_step': len(chunks), 'schur': args.schur,
                       'link_reals': link_reals, 'device': 'one GPU per process'},
            'latency_ms': {'p50': statistics.median(step_ms), 'p99': p99, 'per_step': step_ms},
            'time_to_solution_s': {'p50': statistics.median(step_ms) / 1e3, 'p99': p99 / 1e3},
            'iters': iters, 'rel_true_resid_max': resid_max,
            'solver_tflops': solver_tflops(V // 2, L5, iters, total_s / args.steps),
            'reliable_updates': [s['reliable_updates'] for s in last],
            'fp32_updates': [s['fp32_updates'] for s in last],
            'fp64_rerefs': [s['fp64_rerefs'] for s in last],
            'restarts': max(s['restarts'] for s in last),
            'phases_ms_per_step': phases,
            'hop_ms_per_step': hop_ms / len(stats),
            'profiled_steps': args.profile_steps,
            'oracle_check': oracle_check,
            'fp64_gpu_cg': fp64,
            'speedup_vs_fp64_gpu_cg': (value / fp64['solves_per_s']) if fp64 else None,
            'autotuned': tuned,
            'dslash': {'kernel': '%s<%s>' % (kernel_name, prec), 'form': hop_form, 'launches_timed': hop_launches,
                       'avg_launch_us': hop_avg_s * 1e6 if hop_avg_s else None,
                       'GB_per_s': achieved, 'eff_GFLOP_per_s': gflops,
                       'units_per_launch': units, 'algorithmic_bytes_per_unit': bytes_per_unit,
                       'bytes_per_launch': bytes_per_launch,
                       'stored_bytes_per_launch': stored_per_launch,
                       'stored_GB_per_s': stored_per_launch / hop_avg_s / 1e9 if hop_avg_s else None},
            'roofline': {'bound': 'hbm', 'achieved': achieved, 'peak': peak, 'unit': 'GB/s',
                         'frac': achieved / peak if achieved else None, 'peak_kind': peak_kind,
                         'traffic': ncu_traffic('%s_%s' % (W['key'], prec))},
            'alu_roofline': {'bound': 'alu', 'achieved': gflops / 1e3 if gflops else None,
                             'peak': fp32_peak_tflops, 'unit': 'TFLOP/s',
                             'frac': gflops / 1e3 / fp32_peak_tflops if gflops else None,
                             'peak_kind': 'derived: 152 SMs x 128 FP32 lanes x 2 flops x %.0f MHz' % mhz,
                             'flops_per_unit': 1320},
            'cpu_baseline': cpu,
            'e2e': dict({'value': e2e_value, 'unit': 'solves/s', 'h2d_bytes_per_step': len(e2e_idx) * field_bytes,
                         'd2h_bytes_per_step': len(e2e_idx) * field_bytes},
                        **({} if len(e2e_idx) == n else
                           {'rhs_per_step': len(e2e_idx), 'note': 'one batch of the workload per host-pointer call'})),
            'gpu_launches': gpu_launches,
            'clocks': clk,
            'wall_s': wall,
        }
        print(json.dumps(out), flush=True)
    M.mdwf_destroy(ctx)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def run_op(args):
    """Apply Mhat and Mhat^+ to --rhs random fields of the workload, warmup + steps
    times, through the batched C-ABI call (a short driver for kernel profiles)."""
    import numpy as np  # noqa: F401
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import synth
    from paper_1701_07559_gb300 import mdwf as M
    W = dict(WORKLOAD)
    args.precision = args.precision or 'half'
    args.rhs = args.rhs or 12
    if args.lattice:
        W['dims'] = tuple(int(v) for v in args.lattice.split(','))
    U = synth.flowed_gauge(W['dims'], W['seed'], W['eps'], W['flow_t'], W['flow_eps'])
    ctx = M.mdwf_create(W['dims'], 0)
    M.mdwf_load_gauge(ctx, 0, U, 1)
    M.mdwf_set_action(ctx, 0, W['M5'], W['b5'], W['c5'], W['masses'][0], W['L5'])
    Lx, Ly, Lz, Lt = W['dims']
    shape = (W['L5'], Lt, Lz, Ly, Lx, 4, 3)
    variant = args.hop_variant | (args.nsb << 8)
    ins = [torch.from_numpy(synth.gaussian_spinor(shape, 50 + i)).to('cuda') for i in range(args.rhs)]
    outs = [torch.empty_like(x) for x in ins]
    t = []
    for i in range(args.warmup + args.steps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        M.mdwf_apply_schur_batch_dev(ctx, 0, ins, outs, dagger=0, precision=args.precision, hop_variant=variant)
        M.mdwf_apply_schur_batch_dev(ctx, 0, outs, ins, dagger=1, precision=args.precision, hop_variant=variant)
        torch.cuda.synchronize()
        if i >= args.warmup:
            t.append(time.perf_counter() - t0)
    M.mdwf_destroy(ctx)
    print(json.dumps({'mode': 'op', 'rhs': args.rhs, 'precision': args.precision, 'lattice': W['dims'],
                      'hop_variant': args.hop_variant, 'nsb': args.nsb,
                      'ms_per_pair_of_applies': 1e3 * statistics.mean(t) if t else None}), flush=True)
    return 0


# the serving mix: three resident flowed configurations (seeds 5, 6, 7); the
# 24^3 x 64 one carries the a12m310 action of Table II, the others the a15m310 one
SERVE_ACTIONS = {12: (1.3, 1.5, 0.5), 8: (1.2, 1.25, 0.25), 6: (1.3, 1.5, 0.5)}
SERVE_MASSES = (0.0102, 0.0158, 0.0216)


def serve_requests(serving, names, dims, n, seed):
    """n requests: configuration and mass uniform, Z2 noise or point source 50/50."""
    import numpy as np
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(n):
        k = int(rng.integers(len(names)))
        mass = float(SERVE_MASSES[int(rng.integers(3))])
        if rng.random() < 0.5:
            src = ('z2', int(rng.integers(1 << 62)))
        else:
            src = ('point', int(rng.integers(4)), int(rng.integers(3)), tuple(int(rng.integers(d)) for d in dims[k]))
        out.append(serving.Request(names[k], mass, src))
    return out


def run_serve(args):
    """Continuous-batching serving of a Poisson stream of solve requests over the
    resident configurations: capacity from a closed-loop run, then p50/p99 latency
    and solves/s at the given fractions of it."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1701_07559_gb300 import serving
    from paper_1701_07559_gb300 import mdwf as M
    torch.cuda.set_device(0)
    args.precision = args.precision or 'half'
    budget = int(args.hbm_budget_gb * 1e9) if args.hbm_budget_gb > 0 else None
    srv = serving.Server(device=0, hbm_budget=budget, tol=1e-10, precision=args.precision, max_slots=args.slots,
                         priorities=args.priorities)
    names, dims = [], []
    t0 = time.perf_counter()
    for i, spec in enumerate(args.serve_lattices.split(';')):
        lat, l5 = spec.split(':')
        d = tuple(int(v) for v in lat.split(','))
        l5 = int(l5)
        M5, b5, c5 = SERVE_ACTIONS.get(l5, (1.3, 1.5, 0.5))
        U = flowed_links(M, d, 5 + i, 0.4, 1.0, 0.01)
        name = '%dx%dx%dx%d L5=%d' % (d + (l5,))
        srv.add_config(name, d, U, M5, b5, c5, SERVE_MASSES[1], l5)
        names.append(name)
        dims.append(d)
    setup_s = time.perf_counter() - t0
    # warm-up: one request per configuration (sessions, graphs)
    srv.run(serve_requests(serving, names, dims, 2 * len(names), 1))
    # capacity: everything queued at once
    ncap = max(2 * args.slots, args.requests // 3)
    clocks = ClockSampler(0)
    clocks.start()
    done = srv.run(serve_requests(serving, names, dims, ncap, 7))
    cap = serving.Server.metrics(done)
    capacity = cap['solves_per_s']
    runs = []
    for j, frac in enumerate(float(f) for f in args.rates.split(',')):
        reqs = serve_requests(serving, names, dims, args.requests, 8 + j)
        arr = serving.poisson_arrivals(len(reqs), frac * capacity, 8 + j)
        done = srv.run(reqs, arr)
        m = serving.Server.metrics(done)
        m['rate_fraction'] = frac
        m['offered_per_s'] = frac * capacity
        m['per_config'] = {}
        for name in names:
            sub = [r for r in done if r.config == name]
            if sub:
                mm = serving.Server.metrics(sub)
                m['per_config'][name] = {'requests': len(sub), 'p50_s': mm['p50_s'], 'p99_s': mm['p99_s'],
                                         'iters_mean': mm['iters_mean']}
        runs.append(m)
    clk = clocks.stop()
    peak_bytes = max(s[3] for s in srv.samples)
    queue_max = max(s[1] for s in srv.samples)
    srv.close()
    print(json.dumps({'mode': 'serve', 'metric': 'p50/p99 latency and solves/s of a Poisson stream of solves to 1e-10',
                      'precision': args.precision, 'priorities': args.priorities, 'configs': names,
                      'masses': SERVE_MASSES, 'requests_per_rate': args.requests,
                      'sources': 'Z2 noise or point, 50/50', 'slots_max': args.slots,
                      'hbm_budget_bytes': srv.budget, 'hbm_peak_accounted_bytes': peak_bytes, 'queue_max': queue_max,
                      'capacity_solves_per_s': capacity, 'capacity_run': cap, 'runs': runs, 'setup_s': setup_s,
                      'clocks': clk, 'data': 'synthetic'}), flush=True)
    return 0


def main():
    args = parse()
    if args.impl == 'reference':
        return run_reference(args)
    if args.mode == 'op':
        return run_op(args)
    if args.mode == 'serve':
        return run_serve(args)
    return run_ours(args)


if __name__ == '__main__':
    sys.exit(main())
