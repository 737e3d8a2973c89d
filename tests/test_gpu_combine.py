"""The combination against sum_i c_i P_i E_i in float64 of the run's own
component fields, at the edges of its kernels: lines of 4 to 2048 nodes (the
thread's run of 4 up to several blocks per line), single grids and many, both
centrings, both precisions and accumulations, and 3D runs whose planes of
pairs go in several launches (large tau).

Bound: a grid's interpolated term takes at most 6 roundings (3D: two along z,
the pair's rounding, two along y, the split's), each at most u = 2^-24 (FP32;
FP64 and the prolongation's 12 levels: 2^-53) of the grid's largest value, so
no node is off by more than 8 u sum_i |c_i| max |E_i| (FP64: 64 u)."""
import numpy as np
import pytest

from oracle import sgpic_oracle as O
from paper_2008_09441_gb300 import workloads
from test_gpu_parity import make_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,tau,centring,prec,combine", [
    (2, 2, 1, "node", "fp32", "float-float"), (2, 2, 2, "cell", "fp32", "float-float"),
    (2, 3, 1, "cell", "fp64", "float-float"), (2, 4, 4, "node", "fp32", "float-float"),
    (2, 5, 2, "cell", "fp32", "fp64"), (2, 7, 1, "cell", "fp32", "float-float"),
    (2, 9, 1, "node", "fp64", "float-float"), (2, 10, 3, "node", "fp32", "float-float"),
    (2, 11, 1, "cell", "fp32", "float-float"), (2, 11, 10, "node", "fp32", "float-float"),
    (3, 2, 1, "cell", "fp32", "float-float"), (3, 2, 2, "node", "fp64", "float-float"),
    (3, 3, 3, "cell", "fp32", "float-float"), (3, 4, 2, "node", "fp32", "fp64"),
    (3, 5, 1, "cell", "fp32", "float-float"), (3, 5, 1, "node", "fp64", "float-float"),
    (3, 6, 5, "node", "fp32", "float-float"), (3, 7, 1, "node", "fp32", "float-float"),
    (3, 7, 6, "cell", "fp32", "float-float")])
def test_combination_of_own_fields(torch_cuda, d, n, tau, centring, prec, combine):
    gen = workloads.landau2d if d == 2 else workloads.twostream3d
    wl = gen(n_particles=3001, n=n, tau=tau, seed=17 + n)
    run, _ = make_run(wl, prec, torch_cuda, centring=centring, combine=combine)
    comps = run.grid_fields()
    got, dens, rho = run.field(), run.density(), run.grid_charges()
    mean = -1.0 if prec == "fp64" else np.float64(np.mean(next(iter(rho.values()))))
    run.close()
    u = 8 * 2.0 ** -24 if prec == "fp32" else 64 * 2.0 ** -53
    grids = O.combination_grids(d, n, tau)
    for m in range(d):
        ref = sum(c * O.prolong(comps[l][m], n, l, centring) for l, c in grids)
        scale = sum(abs(c) * np.max(np.abs(comps[l][m])) for l, c in grids)
        assert np.max(np.abs(got[m] - ref)) <= u * scale
    ref = sum(c * O.prolong(rho[l] - mean, n, l, centring) for l, c in grids) + mean
    scale = sum(abs(c) * np.max(np.abs(rho[l] - mean)) for l, c in grids)
    assert np.max(np.abs(dens - ref)) <= u * scale + 2.0 ** -50 * abs(mean)
