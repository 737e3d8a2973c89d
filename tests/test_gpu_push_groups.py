"""The 3D FP32 push at the edges of its 64-particle groups (the remainder goes
one particle per thread to the first block) against the oracle, over an
ordinary and a sort step, with the tolerances of the trajectory tests."""
import pytest

from paper_2008_09441_gb300 import workloads
from test_gpu_parity import torch_cuda, trajectory_check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_", [63, 64, 65, 127, 511, 513, 2048 + 63])
def test_steps_at_group_edges(torch_cuda, np_):
    wl = workloads.twostream3d(n_particles=np_, n=4, tau=1, seed=np_)
    trajectory_check(wl, "fp32", torch_cuda, 2, sort_every=2)
