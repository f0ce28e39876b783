"""Contexts are independent: what one thread does with its context does not depend on
another thread that is capturing a CUDA graph at the same time (thread-local mode).
"""
import ctypes
import threading

import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class _Capturing(threading.Thread):
    """Captures one addition on a stream of its own; stays in capture between
    `begun` and `finish`."""

    def __init__(self, blocking=False):
        super().__init__()
        if blocking:  # a stream that waits for the legacy default stream
            handle = ctypes.c_void_p()
            assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(handle))) == 0
            self.stream = torch.cuda.ExternalStream(handle.value)
        else:
            self.stream = torch.cuda.Stream()
        self.begun, self.finish = threading.Event(), threading.Event()
        self.x = torch.ones(256, device="cuda")
        self.y = torch.zeros(256, device="cuda")
        self.graph = torch.cuda.CUDAGraph()
        self.error = None

    def run(self):
        try:
            with torch.cuda.stream(self.stream):
                torch.add(self.x, 1.0, out=self.y)
                torch.cuda.synchronize()
                self.graph.capture_begin(capture_error_mode="thread_local")
                torch.add(self.x, 2.0, out=self.y)
                self.begun.set()
                self.finish.wait(60)
                self.graph.capture_end()
        except Exception as e:  # (reported by the main thread)
            self.error = e
        finally:
            self.begun.set()

    def __enter__(self):
        torch.cuda.synchronize()
        self.start()
        assert self.begun.wait(60)
        return self

    def __exit__(self, *exc):
        self.finish.set()
        self.join()
        if exc[0] is None:
            assert self.error is None
            self.graph.replay()
            torch.cuda.synchronize()
            assert bool((self.y == 3.0).all())


def test_clover_rebuild_while_another_thread_captures():
    from paper_1109_4279_gb300 import binding as B
    dims, block = (4, 4, 4, 8), (2, 2, 2, 2)
    fields = [synth.gauge_field(dims, 0.5, k)[0] for k in (51, 52)]
    Us = [torch.from_numpy(U).cuda() for U in fields]
    psi = torch.from_numpy(synth.gaussian_spinor(dims, synth.gauge_field(dims, 0.5, 53)[1])).cuda()
    outs = [torch.empty_like(psi) for _ in range(4)]
    lat = B.Lattice(dims, block, 0.1, 1.3)
    lat.load_gauge(Us[0])
    with _Capturing():
        lat.load_gauge(Us[1])        # new links: the FP64 records are used again
        B.qcd_apply_D(lat.ctx, psi, outs[0])
        B.qcd_build_clover(lat.ctx)  # the same links once more
        B.qcd_apply_D(lat.ctx, psi, outs[1])
    for k, U in enumerate(Us):
        fresh = B.Lattice(dims, block, 0.1, 1.3)
        fresh.load_gauge(U)
        B.qcd_apply_D(fresh.ctx, psi, outs[2 + k])
        fresh.close()
    assert torch.equal(outs[0], outs[3]) and torch.equal(outs[1], outs[3]) and not torch.equal(outs[2], outs[3])
    lat.close()


def test_first_solve_while_another_thread_captures_a_blocking_stream():
    """The first solve of a context allocates its workspace; nothing of that may go
    through the default stream, which the captured stream waits for."""
    from paper_1109_4279_gb300 import binding as B
    dims, block = (4, 4, 4, 8), (2, 2, 2, 2)
    U, rng = synth.gauge_field(dims, 0.5, 54)
    U = torch.from_numpy(U).cuda()
    b = torch.from_numpy(synth.gaussian_spinor(dims, rng)).cuda()
    sp = B.solver_params(tol=1e-10, solver="cg")
    xs = [torch.zeros_like(b) for _ in range(3)]
    contexts = [B.Lattice(dims, block, 0.1, 1.3) for _ in range(2)]
    for lat in contexts:
        lat.load_gauge(U)
    _, want = B.qcd_solve(contexts[0].ctx, b, xs[0], 1, sp)
    side = torch.cuda.Stream()
    with _Capturing(blocking=True):
        with torch.cuda.stream(side):
            st, _ = B.qcd_solve(contexts[1].ctx, b, xs[1], 1, sp, raise_on_fail=False)
    torch.cuda.synchronize()
    assert st == 0
    _, info = B.qcd_solve(contexts[1].ctx, b, xs[2], 1, sp)
    assert info[0]["cg_iterations"] == want[0]["cg_iterations"]
    assert torch.equal(xs[1], xs[0]) and torch.equal(xs[2], xs[0])
    for lat in contexts:
        lat.close()


def test_force_and_operator_of_one_context_from_several_threads():
    """qcd_apply_D and qcd_force of one context at once, each thread on its own stream:
    the staging memory of a call is its own until it returns (bit for bit)."""
    from paper_1109_4279_gb300 import binding as B
    dims, block, n = (8, 8, 8, 8), (4, 4, 4, 4), 4
    U, rng = synth.gauge_field(dims, 0.5, 55)
    lat = B.Lattice(dims, block, 0.1, 1.3)
    lat.load_gauge(torch.from_numpy(U).cuda())
    psi = torch.from_numpy(synth.gaussian_spinor(dims, rng, nrhs=n + 1)).cuda()
    D = [torch.empty_like(psi[0]) for _ in range(n)]
    F = [torch.empty((lat.V, 4, 8), dtype=torch.float64, device="cuda") for _ in range(n)]
    for k in range(n):
        B.qcd_apply_D(lat.ctx, psi[k], D[k], prec="f32")
        B.qcd_force(lat.ctx, psi[k], psi[k + 1], F[k])
    got = [[(torch.empty_like(D[k]), torch.empty_like(F[k])) for _ in range(8)] for k in range(n)]
    streams = [torch.cuda.Stream() for _ in range(n)]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            with torch.cuda.stream(streams[k]):
                for d, f in got[k]:
                    B.qcd_apply_D(lat.ctx, psi[k], d, prec="f32")
                    B.qcd_force(lat.ctx, psi[k], psi[k + 1], f)
        except Exception as e:  # (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(torch.equal(d, D[k]) and torch.equal(f, F[k]) for k in range(n) for d, f in got[k])
    lat.close()
