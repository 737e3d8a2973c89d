"""Read-back of distinct velocity components, through the records in the idle
particle set (device, 64 MiB and more) and the direct scatter (host), with
either set idle: bits move, so what was uploaded comes back.  dt = 0: a step
only sorts."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,prec,np_", [(2, "fp32", (64 << 20) // 20 + 1), (3, "fp32", (64 << 20) // 28 + 259),
                                        (2, "fp64", (64 << 20) // 40 + 3), (3, "fp64", (64 << 20) // 56 + 257)])
def test_velocities_bit_exact(torch_cuda, d, prec, np_):
    from paper_2008_09441_gb300 import Run
    torch = torch_cuda
    dt = torch.float32 if prec == "fp32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(np_)
    u = torch.rand(d, np_, generator=g, device="cuda", dtype=dt)
    v = torch.randn(d, np_, generator=g, device="cuda", dtype=dt)
    w = torch.rand(np_, generator=g, device="cuda", dtype=dt) - 0.5
    torch.cuda.synchronize()
    run = Run((1.0,) * d, 5, list(u), list(v), w, 0.0, precision=prec, sort_every=1)
    for _ in range(3):
        out = [torch.full_like(x, 7.0) for x in (u, v, w)]
        torch.cuda.synchronize()
        run.particles_device(list(out[0]), list(out[1]), out[2])
        assert all(torch.equal(a, b) for a, b in zip(out, (u, v, w)))
        hu, hv, hw = run.particles()
        assert np.array_equal(hu, u.T.cpu().numpy()) and np.array_equal(hv, v.T.cpu().numpy())
        assert np.array_equal(hw, w.cpu().numpy())
        run.step(1)
    run.close()
