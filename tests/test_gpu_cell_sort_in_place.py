"""The cell sort's outputs may lie where its positions are: sorted keys over a
position array, counts over another (two and three passes, both precisions)."""
import ctypes as C

import numpy as np
import pytest

from oracle import sgpic_oracle as O
from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d,level,n", [(2, 4, 70001), (2, 7, 70001), (3, 5, 40003), (3, 6, 262144)])
def test_outputs_over_the_positions(torch_cuda, d, level, n, prec, static):
    from paper_2008_09441_gb300 import _lib as L
    torch = torch_cuda
    dt, code = (np.float32, L.SG_FP32) if prec == "fp32" else (np.float64, L.SG_FP64)
    u = np.random.default_rng(n + level).random((n, d)).astype(dt)
    cols = [torch.from_numpy(np.ascontiguousarray(u[:, m])).cuda() for m in range(d)]
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    cells = 1 << (d * level)
    over = cells * 4 <= cols[1].numel() * cols[1].element_size()
    counts = cols[1] if over else torch.empty(cells, dtype=torch.int32, device="cuda")
    arr = (C.c_void_p * 3)(*([c.data_ptr() for c in cols] + [None] * (3 - d)))
    lib = L.lib()
    fn = lib.sg_cell_sort_static if static else lib.sg_cell_sort
    assert fn(code, d, level, n, arr, C.c_void_p(cols[0].data_ptr()), C.c_void_p(perm.data_ptr()),
              C.c_void_p(counts.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream)) == L.SG_OK
    torch.cuda.synchronize()
    p_ref, k_ref, c_ref = O.sort_by_key(O.cell_keys(u.astype(np.float64), level), level, d)
    assert np.array_equal(cols[0].cpu().numpy().view(np.uint32)[:n], k_ref)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), p_ref)
    assert np.array_equal(counts.cpu().numpy().view(np.uint32)[:cells], c_ref)
