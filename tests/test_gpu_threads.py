"""Two host threads, each with its own context, plan and stream, evaluate calls of different
shared-memory sizes on one GPU at the same time (needs a GB300; marked gpu)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = 1500


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04269_gb300 import build
    build.build()


def fields(T, V3):
    f = np.random.default_rng(V3).standard_normal((2, 1, T, V3, 12, 12, 2)).view(np.complex128)[..., 0]
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in f]


class Caller:
    """One thread's context, plan, fields and stream; call() evaluates them once."""

    def __init__(self, kind, op, prec, T, L):
        from paper_2201_04269_gb300 import Context
        self.ctx = Context(0)
        self.stream = torch.cuda.Stream()
        self.U, self.D = fields(T, L ** 3)
        self.C = torch.zeros(1, T, dtype=torch.complex128, device="cuda")
        s = self.stream.cuda_stream
        if kind in ("blocks", "blocks_local"):
            self.plan = self.ctx.block_plan(op, prec)
            self.call = (lambda: self.plan.correlator(self.U, self.D, self.C, L, stream=s)) if kind == "blocks" else \
                (lambda: self.plan.correlator_local(self.U, self.D, self.C, stream=s))
        else:
            self.plan = self.ctx.plan_operator(op, "egraph", prec)
            if kind == "batch":
                items = [dict(plan=self.plan.handle, U=self.U, D=self.D, n_sets=1, T=T, V3=L ** 3, C=self.C)]
                self.call = lambda: self.ctx.batch(items, s)
            else:
                self.call = lambda: self.plan.correlator(self.U, self.D, self.C, stream=s)
        torch.cuda.synchronize()
        self.call()
        torch.cuda.synchronize()
        self.first = self.C.cpu().numpy().copy()
        self.error = None

    def loop(self, barrier):
        try:
            barrier.wait()
            for _ in range(CALLS):
                self.call()
        except Exception as e:                   # reported by the main thread
            self.error = e

    def close(self):
        torch.cuda.synchronize()
        self.plan.destroy()
        self.ctx.close()


GUARDS = [
    ("call", ("proton", "fp32", 1, 24), ("proton", "fp32", 1, 4)),             # slice guard: 55 KB and 256 bytes
    ("batch", ("proton", "fp32", 1, 24), ("proton", "fp32", 1, 4)),            # its batched form
]
PLANS = [
    ("call", ("he3_II_s", "fp32", 1, 1), ("he3_I", "fp32", 1, 1)),             # FP32 kernel
    ("call", ("dinucleon_I", "mixed", 1, 2), ("proton", "mixed", 1, 2)),       # double-float and FP64 kernels
    ("call", ("dinucleon_I", "fp64", 1, 2), ("proton", "fp64", 1, 2)),
    ("batch", ("dinucleon_I", "mixed", 1, 2), ("proton", "mixed", 1, 2)),
    ("blocks", ("dinucleon_I", "fp64", 1, 2), ("proton", "fp64", 1, 2)),       # projection and block tree
    ("blocks", ("dinucleon_I", "mixed", 1, 2), ("proton", "mixed", 1, 2)),
    ("blocks_local", ("dinucleon_I", "fp64", 1, 2), ("proton", "fp64", 1, 2)),
]


@pytest.mark.parametrize("kind,a,b", GUARDS + PLANS)
def test_threads_do_not_share_shared_memory_limits(kind, a, b):
    """A kernel's shared-memory limit belongs to the kernel, not to a context: no call may be refused
    because another thread's call of a smaller size came in between."""
    callers = [Caller(kind, *a), Caller(kind, *b)]
    barrier = threading.Barrier(2)
    threads = [threading.Thread(target=c.loop, args=(barrier,)) for c in callers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    got = [c.C.cpu().numpy() for c in callers]
    for c in callers:
        c.close()
    assert [c.error for c in callers] == [None, None]
    for c, x in zip(callers, got):
        assert np.array_equal(x, c.first)
