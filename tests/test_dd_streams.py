"""A GPU sub-domain's calls and torch's stream, with a stand-in for the library and the device (no GPU):
the library runs on a stream of its own, so each call has to come after a wait for what torch has queued
for its arrays, the ones the call allocates included."""
import types

import torch

from paper_1701_07559_gb300 import dd


def test_subdomain_waits_for_torch_before_each_library_call(monkeypatch):
    log = []
    wait = types.SimpleNamespace(synchronize=lambda: log.append('wait'))
    monkeypatch.setattr(torch.cuda, 'current_stream', lambda device=None: wait)
    for name in ('empty', 'empty_like'):
        def alloc(*a, _f=getattr(torch, name), **k):
            log.append('alloc')
            return _f(*a, **k)
        monkeypatch.setattr(torch, name, alloc)
    sub = dd.GPUSubdomain.__new__(dd.GPUSubdomain)
    sub.M = types.SimpleNamespace(mdwf_dd_pack_faces_dev=lambda *a: log.append('pack'),
                                  mdwf_dd_apply_dev=lambda *a: log.append('apply'))
    sub.ctx, sub.cfg_id, sub.fshape, sub.device = None, 0, (2, 2, 2, 2, 2, 3), torch.device('cpu')
    x = torch.zeros(4, dtype=torch.complex128)
    fp, fn = sub.pack(0, 0, x)
    sub.apply(0, 0, x, fn, fp, 1.0, -1.0)
    assert log == ['alloc', 'alloc', 'wait', 'pack', 'alloc', 'wait', 'apply']
