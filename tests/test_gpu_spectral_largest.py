"""The regular-grid transforms where their launches change form: the filter's
solve with one block for all components and the estimator with more masks than
its half spectra hold (2D n = 12, 3D n = 8), and the estimator of an FP32 run.
The references start from the run's own densities."""
import numpy as np
import pytest

from oracle import sgpic_oracle as O
from test_gpu_parity import TOL, nrmse, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def run_of(d, n, prec, **kw):
    from paper_2008_09441_gb300 import Run
    rng = np.random.default_rng(10 * d + n)
    u = 0.5 + 0.15 * rng.normal(size=(40009, d))  # a few large modes
    return Run((2.0,) * d, n, u - np.floor(u), np.zeros((40009, d)), -rng.random(40009), 0.01, precision=prec, **kw)


@pytest.mark.parametrize("d,n,prec", [(2, 12, "fp32"), (2, 12, "fp64"), (3, 8, "fp32")])
def test_filter_field(torch_cuda, d, n, prec):
    r = run_of(d, n, prec, mode="filter", tau=n - 1)
    rho, E = r.density(), r.field()
    r.close()
    N = 1 << n
    f = np.fft.rfftn(rho)
    k = np.fft.fftfreq(N, 1.0 / N) * (2 * np.pi / 2.0)
    ks = [k.reshape([-1 if a == m else 1 for a in range(d)]) for m in range(d)]
    ks[d - 1] = ks[d - 1][..., :N // 2 + 1]
    k2 = sum(x * x for x in ks)
    k2[(0,) * d] = 1.0
    f[(0,) * d] = 0.0
    for m in range(d):
        km = ks[m].copy()
        np.moveaxis(km, m, 0)[N // 2] = 0.0  # no field of the axis's Nyquist plane
        assert nrmse(E[m], np.fft.irfftn(-1j * km * f / k2, s=rho.shape, axes=range(d))) < TOL[prec], m


@pytest.mark.parametrize("d,n,prec", [(2, 12, "fp64"), (3, 8, "fp32"), (2, 6, "fp32"), (3, 5, "fp32")])
def test_estimates(torch_cuda, d, n, prec):
    r = run_of(d, n, prec, alpha=0.02, pc_ref=1.0, tau=n - 1)
    tau, g, z = r.select_tau()
    rho, q = r.regular_charge(), r.diagnostics()["charge_total"]
    r.close()
    ref, table, _ = O.tau_estimator(rho, Np=40009, L=2.0, alpha=0.02, pc_ref=1.0, Qe=q, constants="paper")
    assert tau == ref
    for t, ge, ze in table:
        assert g[t - 1] == pytest.approx(ge, rel=1e-9) and z[t - 1] == pytest.approx(ze, rel=1e-9)
