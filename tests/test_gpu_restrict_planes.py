"""The restriction of 3D runs, plane by plane (and by axis where the plane
does not fit shared memory), against the oracle's matrices applied to the
run's own regular density.

Bound: a halving step averages with three roundings of at most u of the
largest value, n steps per axis, three axes: 9 n u <= 64 u of the largest
deviation from the mean (u = 2^-24, FP64 2^-53)."""
import numpy as np
import pytest

from oracle import sgpic_oracle as O
from paper_2008_09441_gb300 import workloads
from test_gpu_parity import make_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tau,centring,prec", [
    (2, 1, "node", "fp32"), (2, 2, "cell", "fp64"), (3, 1, "cell", "fp32"), (3, 3, "node", "fp32"),
    (4, 3, "cell", "fp32"), (5, 1, "node", "fp64"), (6, 1, "cell", "fp32"), (6, 5, "cell", "fp64"),
    (7, 1, "node", "fp32"), (7, 6, "node", "fp32"), (7, 1, "cell", "fp32"), (7, 2, "node", "fp64")])
def test_component_densities(torch_cuda, n, tau, centring, prec):
    wl = workloads.twostream3d(n_particles=20011, n=n, tau=tau, seed=60 + n)
    run, _ = make_run(wl, prec, torch_cuda, centring=centring)
    reg, got = run.regular_charge(), run.grid_charges()
    run.close()
    u = 2.0 ** -24 if prec == "fp32" else 2.0 ** -53
    bound = 64 * u * np.max(np.abs(reg - np.mean(reg))) + 4 * u * abs(np.mean(reg))
    for l, _ in O.combination_grids(3, n, tau):
        assert np.max(np.abs(got[l] - O.restrict(reg, n, l, centring))) <= bound, l
