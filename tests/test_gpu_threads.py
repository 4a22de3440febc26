"""Gradients from several host threads, each with its own stream and workspace: none may fail for what another asks for."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_2309_12252_b200 import binding as bd
from paper_2309_12252_b200 import synth

pytestmark = pytest.mark.gpu


# one kernel launched with shared memory of two sizes: with and without dx; two sizes of cell
@pytest.mark.parametrize("jobs", [((64, 6, True), (64, 6, False)), ((32, 32, True), (32, 32, False)), ((60, 72, True), (62, 100, False))])
def test_gradients_in_threads(jobs):
    from bench import read_profile
    B, T, count, failed = 1, 65, 300, []
    done = {}

    def work(k, n, m, want_dx):
        p = bd.GruParamsDev.from_numpy(synth.gru_params(n, m, seed=1, tag="th/gru"))
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        x, y0 = dev(synth.x_gaussian(B, T, m, seed=1, tag="th/x")), torch.zeros((B, n), device="cuda")
        y, gy = dev(synth.normal(1, "th/y", (B, T, n)) * np.float32(0.3)), dev(synth.normal(1, "th/gy", (B, T, n)))
        out = [torch.empty(s, device="cuda") for s in ((3 * n, m), (3 * n, n), (3 * n,), (3 * n,))]
        dx, ws, st = torch.empty_like(x) if want_dx else None, bd.alloc_workspace(bd.DEER_OP_VJP, B, T, n, m), torch.cuda.Stream()
        torch.cuda.synchronize()
        ps, gs = p.c_struct(), bd._Grads(*(t.data_ptr() for t in out))
        args = [ctypes.byref(ps)] + [bd._ptr(t) for t in (x, y0, y, gy)] + [B, T, ctypes.byref(gs), bd._ptr(dx), None, bd._ptr(ws), ws.numel(), 0,
                                                                          ctypes.c_void_p(st.cuda_stream)]
        for i in range(count):                           # (the call without the interpreter's part, so that the threads meet in it)
            rc = bd.lib().deer_gru_vjp(*args)
            if rc:
                failed.append((n, m, want_dx, rc))
            if i % 16 == 15:
                st.synchronize()
        st.synchronize()
        done.setdefault((n, m, want_dx), []).append([t.cpu() for t in out])

    threads = [threading.Thread(target=work, args=(k, *jobs[k % 2])) for k in range(4)]
    bd.lib().deer_profile_enable(1)                      # (its events widen the time between a kernel's set-up and its launch)
    try:
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        bd.lib().deer_profile_enable(0)
        read_profile(bd)
    assert not failed, (len(failed), failed[:3])
    for same in done.values():
        assert len(same) == 2 and all(torch.equal(a, b) for a, b in zip(*same))
