"""Entry points that stage fields in memory kept by the context: calls of
changing size and precision one after another, on two streams, one whose
fields exceed what is kept, and calls from several threads at the same time,
give what a fresh context gives.
"""
import threading

import pytest

from paper_1109_4279_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lattice(dims, block, U):
    from paper_1109_4279_gb300 import binding
    lat = binding.Lattice(dims, block, 0.0, 1.5)
    lat.load_gauge(U)
    return lat


def test_changing_sizes_and_streams():
    from paper_1109_4279_gb300 import binding
    dims, block = (8, 8, 8, 8), (4, 4, 2, 2)
    U, rng = synth.gauge_field(dims, 0.5, 31)
    U = torch.from_numpy(U).cuda()
    psi = torch.from_numpy(synth.gaussian_spinor(dims, rng, nrhs=3)).cuda()
    lat = _lattice(dims, block, U)
    side = torch.cuda.Stream()
    for k, (prec, nrhs) in enumerate((("f16", 1), ("f64", 3), ("f32", 2), ("df64", 1), ("bf16", 3), ("f64", 1))):
        p = psi[:nrhs].contiguous()
        with torch.cuda.stream(side if k % 2 else torch.cuda.current_stream()):
            side.wait_stream(torch.cuda.default_stream())
            out = lat.apply_D(p, prec=prec)
            F = torch.empty((lat.V, 4, 8), dtype=torch.float64, device="cuda")
            binding.qcd_force(lat.ctx, psi[0].contiguous(), psi[1].contiguous(), F)
        torch.cuda.synchronize()
        fresh = _lattice(dims, block, U)
        G = torch.empty_like(F)
        binding.qcd_force(fresh.ctx, psi[0].contiguous(), psi[1].contiguous(), G)
        assert torch.equal(out, fresh.apply_D(p, prec=prec)) and torch.equal(F, G)
        fresh.close()
    lat.close()


def test_fields_beyond_what_is_kept():
    """Three FP64 right-hand sides of 32^4 stage 1.2 GB, more than the 1 GiB kept."""
    dims = (32, 32, 32, 32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    V = 32 ** 4
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    psi = torch.view_as_complex(torch.randn((3, V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
    lat = _lattice(dims, (4, 4, 4, 4), U)
    from paper_1109_4279_gb300 import binding
    out = torch.empty_like(psi)
    free0 = torch.cuda.mem_get_info()[0]
    binding.qcd_apply_D(lat.ctx, psi, out, nrhs=3)
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)  # given back
    for k in range(3):
        one = torch.empty_like(psi[0])
        binding.qcd_apply_D(lat.ctx, psi[k].contiguous(), one)
        assert torch.equal(one, out[k])
    lat.close()


def test_threads_do_not_share_the_memory():
    """Four threads apply D of one context on their own streams at the same time;
    each gets its own answer (the kernels sum in a fixed order: bit for bit)."""
    from paper_1109_4279_gb300 import binding
    dims, block, n = (16, 8, 8, 8), (4, 4, 4, 4), 4
    U, rng = synth.gauge_field(dims, 0.5, 32)
    lat = _lattice(dims, block, torch.from_numpy(U).cuda())
    psi = torch.from_numpy(synth.gaussian_spinor(dims, rng, nrhs=n)).cuda()
    want = [lat.apply_D(psi[k], prec="f64") for k in range(n)]
    outs = [[torch.empty_like(psi[k]) for _ in range(12)] for k in range(n)]
    streams = [torch.cuda.Stream() for _ in range(n)]
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            with torch.cuda.stream(streams[k]):
                for o in outs[k]:
                    binding.qcd_apply_D(lat.ctx, psi[k], o)
        except Exception as e:  # (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(n)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors
    assert all(torch.equal(o, want[k]) for k in range(n) for o in outs[k])
    lat.close()
