"""The deposit's two block sizes at their edges (chunks of 512 and 2048
particles, the line between them at 304 chunks of 2048 on a 152-SM GPU)
against the oracle, with the tolerance of the parity tests."""
import numpy as np
import pytest

from oracle import sgpic_oracle as O
from paper_2008_09441_gb300 import workloads
from test_gpu_parity import TOL, make_run, nrmse, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,prec,np_", [(2, "fp64", 511), (2, "fp64", 513), (3, "fp64", 2049), (2, "fp32", 515),
                                        (3, "fp32", 5123), (2, "fp64", 304 * 2048 - 2048), (2, "fp32", 304 * 2048 - 1),
                                        (2, "fp32", 304 * 2048 + 3), (3, "fp64", 304 * 2048 + 1)])
def test_density_at_block_edges(torch_cuda, d, prec, np_):
    gen = workloads.landau2d if d == 2 else workloads.twostream3d
    wl = gen(n_particles=np_, n=5, tau=1, seed=np_ % 1000)
    run, (u, _, q) = make_run(wl, prec, torch_cuda)
    got = run.regular_charge()
    run.close()
    ref = O.deposit_cic(O.wrap_unit(u), q, (5,) * d, wl.L)
    assert nrmse(got, ref) < TOL[prec]
