"""Handles of their own from host threads of their own."""
import ctypes
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_two_set_lists_from_several_threads(cuda_ok):
    """Two-set lists on grids of 27 and of 613 stencil entries at once, each
    thread with its handle, stream and buffers: every call succeeds with the
    pairs it finds alone. (The stencil sits in the kernels' shared memory, whose
    limit belongs to the kernel and not to the call.)"""
    import paper_2202_06427_gb300 as P
    from paper_2202_06427_gb300 import _lib
    lib = _lib.lib()
    rng = np.random.default_rng(5)
    h = np.eye(3) * 20.0
    x = torch.from_numpy(rng.uniform(0, 20, size=(2500, 3))).cuda()
    y = torch.from_numpy(rng.uniform(0, 20, size=(8, 3))).cuda()
    rounds, threads, failed = 3000, [], []
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())

    def work(args, stream, want, a):
        n = ctypes.c_longlong(0)
        for _ in range(rounds):
            code = lib.cl_cross_pairlist(*args, ctypes.byref(n), ctypes.c_void_p(stream.cuda_stream))
            if code != 0 or n.value != want.numel():
                failed.append((code, n.value))
                return
        if not torch.equal(a, want):
            failed.append("pairs")

    keep = []
    for lcell in (1, 4, 1, 4):
        cl = P.cl_build(x, h, 2.0, lcell)
        want = P.cl_cross_pairlist(cl, y)["a"]
        a, b, d = (torch.zeros(want.numel(), dtype=t, device="cuda") for t in (torch.int32, torch.int32, torch.float32))
        stream = torch.cuda.Stream()
        keep.append((cl, a, b, d, stream))
        args = (cl.handle, ptr(y), y.shape[0], want.numel(), ptr(a), ptr(b), ptr(d))
        threads.append(threading.Thread(target=work, args=(args, stream, want, a)))
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
