"""What the FP32 combination may round: a grid's own value, once per
interpolated axis but x (a product and a fused multiply-add per axis).
Everything after it -- the sum over the grids, cell midpoints, the prolongation
along x -- runs in float pairs, so the combined field equals the same
expression in 64 bits up to 2^-42 of the terms' magnitudes (a pair carries 48
bits, and fewer than 2^5 rounded pair operations follow one another on the way
to a node).  The field energy adds the squares of the high parts, each rounded
once, in float pairs and doubles.  The component fields are read back from the
run itself."""
import numpy as np
import pytest

from test_gpu_parity import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def fma32(w, b, t):
    """float32(w b + t), rounded once: the product is exact in 64 bits, the sum is rounded to odd."""
    p, t = w.astype(np.float64) * b, t.astype(np.float64)
    s = p + t
    bb = s - p
    err = (p - (s - bb)) + (t - bb)
    odd = (s.view(np.int64) & 1) == 1
    return np.where((err == 0) | odd, s, np.nextafter(s, np.where(err > 0, np.inf, -np.inf))).astype(np.float32)


def lerp32(w0, a, w1, b):
    return fma32(w1, b, (w0 * a).astype(np.float32))


def bracket(n, lev, cell):
    y, r = np.arange(1 << n), n - lev
    if not cell:
        k0, f = y >> r, (y & ((1 << r) - 1)) / (1 << r)
    else:
        num = 2 * y + 1 - (1 << r)
        fl = num >> (r + 1)
        k0, f = fl & ((1 << lev) - 1), (num - fl * (2 << r)) / (2 << r)
    return k0, (k0 + 1) & ((1 << lev) - 1), f.astype(np.float32)


def ref_combination(grids, n, cell):
    """grids: {levels: (coeff, float32 array indexed [i_1, .., i_d])} -> sums and magnitudes on the regular nodes."""
    total = mag = 0.0
    for lev, (c, e) in grids.items():
        t, c = e, np.float32(c)
        for axis in range(len(lev) - 1, 0, -1):  # rounded axes, the last one first
            k0, k1, f = bracket(n, lev[axis], cell)
            f = f.reshape((-1,) + (1,) * (t.ndim - 1 - axis))
            t = lerp32(c * (1 - f), t.take(k0, axis), c * f, t.take(k1, axis))
            c = np.float32(1)
        t = t.astype(np.float64)
        k0, k1, f = bracket(n, lev[0], cell)
        f = f.astype(np.float64).reshape((-1,) + (1,) * (t.ndim - 1))
        total = total + (1 - f) * t[k0] + f * t[k1]
        mag = mag + np.abs(t).max()
    return total, mag


def make_run(torch, d, n, tau, cell, mode="combine", np_=20011):
    from paper_2008_09441_gb300 import Run
    rng = np.random.default_rng(100 * d + n)
    u, v = rng.random((np_, d)), rng.normal(size=(np_, d))
    return Run((2.0,) * d, n, u, v, -rng.random(np_), 0.01, tau=tau, centring="cell" if cell else "node", mode=mode)


def check_energy(r, E):
    hi = E.astype(np.float32)
    h = (2.0 / 2 ** r.n) ** r.d
    assert abs(r.diagnostics()["field_energy"] / (0.5 * h * np.sum((hi * hi).astype(np.float64))) - 1) <= 2.0 ** -42


CASES = [(2, 2, 1), (2, 5, 1), (2, 6, 2), (2, 8, 1), (2, 10, 3), (2, 11, 1), (3, 2, 1), (3, 4, 1), (3, 5, 2), (3, 6, 1)]


@pytest.mark.parametrize("cell", [False, True])
@pytest.mark.parametrize("d,n,tau", CASES)
def test_field_is_the_pair_sum(torch_cuda, d, n, tau, cell):
    r = make_run(torch_cuda, d, n, tau, cell)
    r.step(1)
    coeff = dict(r.grids())
    E, fields = r.field(), r.grid_fields()
    for m in range(d):
        ref, mag = ref_combination({l: (coeff[l], e[m].astype(np.float32)) for l, e in fields.items()}, n, cell)
        assert np.abs(E[m] - ref).max() <= 2.0 ** -42 * mag, (m, np.abs(E[m] - ref).max() / mag)
    check_energy(r, E)
    r.close()


@pytest.mark.parametrize("cell", [False, True])
@pytest.mark.parametrize("d,n,tau", [(2, 6, 1), (2, 9, 2), (3, 5, 1), (3, 6, 2)])
def test_filtered_density_is_the_pair_sum(torch_cuda, d, n, tau, cell):
    """The same kernels on one component, whose result is stored as one float:
    deviations from the mean, which the getters add back in 64 bits."""
    r = make_run(torch_cuda, d, n, tau, cell, mode="filter")
    coeff, rho = dict(r.grids()), r.density()
    mean = np.float64(np.float32(r.diagnostics()["charge_total"] / 2.0 ** d))
    ref, mag = ref_combination({l: (coeff[l], (e - mean).astype(np.float32)) for l, e in r.grid_charges().items()}, n,
                               cell)
    assert np.all(np.abs(rho - mean - ref) <= 2.0 ** -24 * (1 + 2.0 ** -10) * np.abs(ref) + 2.0 ** -42 * mag
                  + 2.0 ** -52 * abs(mean))
    r.close()


@pytest.mark.parametrize("d,n", [(2, 5), (2, 9), (2, 11), (3, 4), (3, 6)])
def test_filter_mode_energy(torch_cuda, d, n):
    r = make_run(torch_cuda, d, n, 1, False, mode="filter")
    r.step(1)
    check_energy(r, r.field())
    r.close()
