"""Two contexts of one device, each used by its own host thread: calls of different
launch sizes run side by side through the same kernels, so neither thread's launch may
depend on what the other asked of a kernel (its shared-memory limit belongs to the
kernel, not to the call).  Every call succeeds and gives the values it gives alone.
"""
import ctypes
import threading

import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

CALLS = 800
M = dict(workloads.BASE_MODEL)


@pytest.fixture(scope="module")
def simr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2402_12111_gb300 as simr

    simr.load()
    return simr


class Ctx:
    """A library context, a stream and device buffers of its own."""

    def __init__(self, S, n):
        self.S, self.L = S, S.load()
        self.h = ctypes.c_void_p()
        S.check(self.L.simr_create(ctypes.byref(self.h), 0))
        self.stream = torch.cuda.Stream()
        self.p = torch.zeros(n, dtype=torch.float64, device="cuda")
        self.g = torch.zeros(n, 7, dtype=torch.float64, device="cuda")

    def close(self):
        self.L.simr_destroy(self.h)

    def args(self):
        return ctypes.c_void_p(self.p.data_ptr()), ctypes.c_void_p(self.g.data_ptr()), \
            ctypes.c_void_p(self.stream.cuda_stream)


def _strikes(n):
    return torch.linspace(80.0, 120.0, n, dtype=torch.float64, device="cuda")


def _price(S, steps, paths, n=256):
    K, H = _strikes(n), S.as_heston(M)

    def call(c):
        p, _, st = c.args()
        return c.L.simr_price(c.h, ctypes.byref(H), ctypes.c_void_p(K.data_ptr()), n, 0, steps, paths, 1, 0, p, None, st)
    return n, call


def _adjoint(S, steps, paths, every, n=32):
    K, H = _strikes(n), S.as_heston(M)

    def call(c):
        p, g, st = c.args()
        return c.L.simr_greeks_adjoint(c.h, ctypes.byref(H), ctypes.c_void_p(K.data_ptr()), n, 0, steps, paths, 1, 0,
                                       every, p, None, g, st)
    return n, call


def _paths_adjoint(S, steps, every, n=64):
    H = S.as_heston(M)

    def call(c):
        p, g, st = c.args()  # (both buffers are larger than n floats and 5 n floats)
        return c.L.simr_paths_adjoint(c.h, ctypes.byref(H), steps, 0, n, 1, 0, every, p, g, st)
    return n, call


def _book(S, steps, paths, adjoint, n=8):
    opts = (S.Option * n)()
    for o in opts:
        o.m, o.K, o.is_put, o.steps, o.paths = S.as_heston(M), 100.0, 0, steps, paths
    flags = S.BATCH_NO_AUTOTUNE | (S.BATCH_ADJOINT if adjoint else 0)

    def call(c):
        p, g, st = c.args()
        return c.L.simr_batch_submit(c.h, opts, n, 1, flags, p, None, g if adjoint else None, st)
    return n, call


def _basket(S, paths, n=256):
    K, H = _strikes(n), (S.Heston * 2)(S.as_heston(M), S.as_heston(M))
    C, w = np.eye(2), np.full(2, 0.5)

    def call(c):
        p, _, st = c.args()
        return c.L.simr_basket_price(c.h, H, 2, C.ctypes.data_as(ctypes.c_void_p), w.ctypes.data_as(ctypes.c_void_p),
                                     ctypes.c_void_p(K.data_ptr()), n, 0, 2, paths, 1, p, None, st)
    return n, call


def _lsm(S, steps, paths):
    H = S.as_heston(M)

    def call(c):
        p, _, st = c.args()
        return c.L.simr_lsm_price(c.h, ctypes.byref(H), 100.0, 1, steps, 1, paths, 1, 0, p, None, None, None, st)
    return 1, call


# each pair: the same kernel with less and with more shared memory
PAIRS = {
    "price": lambda S: (_price(S, 2, 64 * 152 * 30), _price(S, 2, 64 * 152 * 60)),
    "adjoint, global segments": lambda S: (_adjoint(S, 172, 64, 0), _adjoint(S, 1024, 64, 0)),
    "adjoint, shared segments": lambda S: (_adjoint(S, 16, 64, 2), _adjoint(S, 64, 64, 64)),
    "adjoint paths": lambda S: (_paths_adjoint(S, 8, 8), _paths_adjoint(S, 64, 64)),
    "price book": lambda S: (_book(S, 4, 64, False), _book(S, 1024, 64, False)),
    "adjoint book": lambda S: (_book(S, 4, 64, True), _book(S, 1024, 64, True)),
    "basket": lambda S: (_basket(S, 64), _basket(S, 32 * 152 * 8)),
    "lsm": lambda S: (_lsm(S, 2, 64), _lsm(S, 256, 64)),
}


@pytest.mark.parametrize("kind", PAIRS)
def test_two_contexts_on_two_threads(simr, kind):
    from paper_2402_12111_gb300 import _simr as S

    jobs = PAIRS[kind](S)
    ctxs = [Ctx(S, n) for n, _ in jobs]
    torch.cuda.synchronize()
    try:
        alone = []
        for c, (_, call) in zip(ctxs, jobs):
            S.check(call(c))
            c.stream.synchronize()
            alone.append((c.p.clone(), c.g.clone()))
            torch.cuda.synchronize()
        failed = [[], []]
        gate = threading.Barrier(2)

        def work(i):
            c, (_, call) = ctxs[i], jobs[i]
            gate.wait()
            for k in range(CALLS):
                rc = call(c)
                if rc != S.SIMR_OK:
                    failed[i].append((k, rc, c.L.simr_last_error()))
                if k % 16 == 15:
                    c.stream.synchronize()
            c.stream.synchronize()

        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert not failed[0] and not failed[1], [(len(f), f[:1]) for f in failed]
        for c, (p, g) in zip(ctxs, alone):
            assert torch.equal(c.p, p) and torch.equal(c.g, g)
    finally:
        torch.cuda.synchronize()
        for c in ctxs:
            c.close()
