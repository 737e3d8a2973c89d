"""The stand-alone cell sort at the edges of its tiles (4096 keys), digit
widths (2 to 24 key bits in one to three passes) and runs, bit for bit."""
import ctypes as C

import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,level,n,spread", [
    (2, 1, 1, 1.0), (2, 1, 4097, 1.0), (3, 1, 31, 1.0), (2, 4, 4096, 1.0), (3, 3, 8191, 0.1), (2, 5, 12289, 1.0),
    (3, 5, 40000, 1e-3), (2, 9, 70001, 1.0), (3, 7, 123457, 1.0), (2, 12, 65537, 1.0), (3, 8, 33333, 1.0),
    (2, 10, 300001, 0.0)])
def test_sort_edges(torch_cuda, d, level, n, spread):
    from oracle import sgpic_oracle as O
    from paper_2008_09441_gb300.sgpic import sg_cell_sort
    torch = torch_cuda
    rng = np.random.default_rng(n + level)
    u = (0.37 + spread * rng.uniform(-1.0, 1.0, (n, d))).astype(np.float32)  # outside the box too
    u[:: 7] = u[0]
    cols = [torch.from_numpy(np.ascontiguousarray(u[:, m])).cuda() for m in range(d)]
    keys, perm, counts = (x.cpu().numpy().view(np.uint32) for x in sg_cell_sort(cols, level))
    w = u - np.floor(u)
    w[w >= 1] = 0
    ref = O.cell_keys(w.astype(np.float64), level)
    order = np.argsort(ref, kind="stable")
    assert np.array_equal(keys, ref[order]) and np.array_equal(perm, order)
    assert np.array_equal(counts, np.bincount(ref.astype(np.int64), minlength=1 << (d * level)))
