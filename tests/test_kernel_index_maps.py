"""Index arithmetic of the kernels, restated on the CPU: the line kernel's
storage order, the deposit's divisions, the one-block solve's stages without
reordering, the pairing of real rows in one complex transform, and the tile
scatter's numbering with parts of tiles."""
import numpy as np
import pytest


def line_pos(x, l, n):
    if l == n:
        return ((x & 3) << (l - 2)) + (x >> 2)
    return ((x & 1) << (l - 1)) + (x >> 1) if l == n - 1 else x


@pytest.mark.parametrize("n", range(2, 13))
def test_line_order_and_the_runs_read_from_it(n):
    for l in range(n + 1):
        assert sorted(line_pos(x, l, n) for x in range(1 << l)) == list(range(1 << l))
    for l, R in ((n, 4), (n - 1, 2)):  # a thread reads R nodes and the one past them
        LR = R.bit_length() - 1
        for a in range(0, 1 << l, R):
            for j in range(R):
                assert (j << (l - LR)) + (a >> LR) == line_pos(a + j, l, n)
            b = (a + R) & ((1 << l) - 1)
            assert b >> LR == line_pos(b, l, n)
            if R == 2:  # cell-centred: and the one before
                b = (a - 1) & ((1 << l) - 1)
                assert ((b & 1) << (l - 1)) + (b >> 1) == line_pos(b, l, n)


def test_deposit_divisions():
    """A box has at most 51,200 nodes and 224 along an axis."""
    r = np.arange(51201, dtype=np.uint64)
    for n in range(2, 225):
        m = np.uint64(0xFFFFFFFF // n + 1)
        assert np.array_equal((r * m) >> np.uint64(32), r // np.uint64(n)), n


def bitrev(t, bits):
    return int(format(t, f"0{bits}b")[::-1], 2) if bits else 0


def one_block_axis(buf, logn, ls, inverse):
    """The stages of the one-block solve along an axis of stride 2^ls: pairs of
    stages over elements t, t + q, t + 2q, t + 3q, and one of span 2 for odd logn."""
    S, smask = buf.size, (1 << ls) - 1

    def radix2():
        j = np.arange(S >> 1)
        i0 = ((j >> ls) << (ls + 1)) + (j & smask)
        i1 = i0 + (1 << ls)
        buf[i0], buf[i1] = buf[i0] + buf[i1], buf[i0] - buf[i1]

    if inverse and logn & 1:
        radix2()
    for k in (range(logn & 1, logn - 1, 2) if inverse else range(logn - 2, -1, -2)):
        q = 1 << k
        j = np.arange(S >> 2)
        p, st = j >> ls, q << ls
        pos = p & (q - 1)
        i0 = ((((p >> k) << (k + 2)) + pos) << ls) + (j & smask)
        a0, a1, a2, a3 = (buf[i0 + m * st] for m in range(4))
        sign = 1 if inverse else -1
        w1, w2 = np.exp(sign * 2j * np.pi * pos / (2 * q)), np.exp(sign * 2j * np.pi * pos / (4 * q))
        w3 = (1j if inverse else -1j) * w2  # w2's turned by a quarter
        if inverse:
            b0, b1, b2, b3 = a0 + w1 * a1, a0 - w1 * a1, a2 + w1 * a3, a2 - w1 * a3
            x = b0 + w2 * b2, b1 + w3 * b3, b0 - w2 * b2, b1 - w3 * b3
        else:
            b0, b1, b2, b3 = a0 + a2, a1 + a3, (a0 - a2) * w2, (a1 - a3) * w3
            x = b0 + b1, (b0 - b1) * w1, b2 + b3, (b2 - b3) * w1
        for m in range(4):
            buf[i0 + m * st] = x[m]
    if not inverse and logn & 1:
        radix2()


@pytest.mark.parametrize("logs", [(1, 1), (2, 5), (7, 1), (3, 4), (1, 2, 3), (4, 1, 2)])
def test_one_block_transforms_without_reordering(logs):
    rng = np.random.default_rng(sum(logs))
    x = rng.normal(size=1 << sum(logs)).astype(complex)
    shape = tuple(1 << l for l in reversed(logs))  # x fastest
    buf = x.copy()
    for a, l in enumerate(logs):
        one_block_axis(buf, l, sum(logs[:a]), False)
    rev = np.ix_(*[[bitrev(t, l) for t in range(1 << l)] for l in reversed(logs)])
    # position t holds frequency bitrev(t) of every axis
    assert np.allclose(buf.reshape(shape), np.fft.fftn(x.reshape(shape))[rev], atol=1e-12 * x.size)
    for a in reversed(range(len(logs))):
        one_block_axis(buf, logs[a], sum(logs[:a]), True)
    assert np.allclose(buf, x * x.size, atol=1e-12 * x.size)


@pytest.mark.parametrize("N", [2, 4, 32])
def test_pairs_of_real_rows(N):
    rng = np.random.default_rng(N)
    r = rng.normal(size=(2, N))
    z = np.fft.fft(r[0] + 1j * r[1])
    k = np.arange(N // 2 + 1)
    m = np.conj(z[-k % N])
    H = (z[k] + m) / 2, (z[k] - m) / 2j
    assert np.allclose(H, np.fft.rfft(r))
    full = np.zeros(N, complex)
    for j in k:
        a, b = H[0][j], H[1][j]
        if j in (0, N // 2):
            full[j] = a.real + 1j * b.real
        else:
            full[j], full[N - j] = a + 1j * b, np.conj(a) + 1j * np.conj(b)
    assert np.allclose(np.fft.ifft(full), r[0] + 1j * r[1])


@pytest.mark.parametrize("d,shift,spread", [(3, 9, 4096), (3, 9, 3), (3, 0, 4096), (3, 3, 100), (2, 8, 4096), (2, 0, 1)])
def test_tile_scatter_numbering(d, shift, spread):
    """A block numbers the tiles that occur and, in 3D, splits each into as many
    parts as its 4096 counters allow: its particles come out ordered by tile, in
    one run per tile that starts where the tile's cursor was."""
    rng = np.random.default_rng(shift + spread)
    n = 2048 - 5
    keys = rng.integers(0, spread, n) << shift | rng.integers(0, 1 << shift, n)
    tiles = np.unique(keys >> shift)
    R = tiles.size
    number = {t: i for i, t in enumerate(tiles)}
    logf = min(shift if d == 3 else 0, 12 - ((R - 1).bit_length() if R > 1 else 0))
    assert logf >= 0 and R << logf <= 4096
    fine = (1 << shift) - 1
    bucket = np.array([(number[k >> shift] << logf) + ((k & fine) >> (shift - logf)) for k in keys])
    count = np.bincount(bucket, minlength=R << logf)
    start = np.cumsum(count) - count
    rank = np.array([np.sum(bucket[:i] == b) for i, b in enumerate(bucket)])  # any order within a bucket serves
    at = start[bucket] + rank
    assert sorted(at) == list(range(n))
    out = np.empty(n, int)
    out[at] = keys
    assert np.all(np.diff(out >> shift) >= 0)
    for q, t in enumerate(tiles):
        a = start[q << logf]
        e = start[(q + 1) << logf] if q + 1 < R else n
        assert e - a == np.sum(keys >> shift == t) and np.all(out[a:e] >> shift == t)
