"""The opening of a wide context's basis (rows of more than 17 words: up to
1,024 rows in registers, then up to 32 further rows one at a time) at its
edges: widths around the words and the kernel's smallest, row counts around a
group of four, a warp, the 1,024 rows and the 32 further ones, low and full
rank, rows that contradict earlier ones among the first rows and among the
further ones, ranks that grow in the further rows, the last of 1,025 pivots
when every thread holds one, and a second call on the learned store.  Bit-exact
against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_basis_equal, cuda_device, dev_arrays, lib

pytestmark = pytest.mark.gpu

WIDTHS = (543, 544, 545, 575, 576, 800, 1023, 1024)
ROWS = (1, 3, 4, 5, 31, 33, 1023, 1024, 1025, 1055, 1056, 1057, 1400)


def _bits(rng, n, T, kind):
    """T rows of n features: in the span of a few vectors, of a few and more from row 1,030 on, dense, or independent
    up to the last pivot."""
    if kind == "dense":
        return rng.integers(0, 2, (T, n))
    if kind == "last":  # 1,024 independent rows, then the one that completes 1,025 (with the constant)
        x = np.tril(rng.integers(0, 2, (T, n)), -1)
        x[np.arange(min(T, n)), np.arange(min(T, n))] = 1
        x[n:] = rng.integers(0, 2, (max(T - n, 0), n))
        if T > n:
            x[n] = 0
        return x
    r = int(rng.integers(2, 40))
    G = rng.integers(0, 2, (r, n))
    x = (rng.integers(0, 2, (T, r)) @ G) & 1
    if kind == "grows":
        late = np.arange(T) >= 1030
        x[late] ^= rng.integers(0, 2, (int(late.sum()), 1)) * rng.integers(0, 2, (int(late.sum()), n))
    return x


def _batch(rng, n_bits, counts, kinds, maps):
    W = [(n + 31) // 32 for n in n_bits]
    row_off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    x_off = np.concatenate([[0], np.cumsum([t * w for t, w in zip(counts, W)])[:-1]]).astype(np.int64)
    x = np.zeros(int(sum(t * w for t, w in zip(counts, W))), np.uint32)
    y = np.zeros((int(row_off[-1]), 4), np.uint32)
    for c, (n, T) in enumerate(zip(n_bits, counts)):
        xb = np.zeros((T, 32 * W[c]), np.uint8)
        xb[:, :n] = _bits(rng, n, T, kinds[c])
        A, b = maps[c]
        yb = ((xb[:, :n].astype(np.float32) @ A).astype(np.int64) + b) & 1
        for i in (T // 2, 600, 1000, 1023, 1024, 1026, 1040, 1055, 1056, T - 1):
            if c % 3 and 0 <= i < T and rng.random() < 0.5:  # independent rows only plant another map
                yb[i, int(rng.integers(128))] ^= 1
        x[x_off[c]:x_off[c] + T * W[c]] = np.packbits(xb, axis=1, bitorder="little").view(np.uint32).reshape(-1)
        y[row_off[c]:row_off[c + 1]] = np.packbits(yb.astype(np.uint8), axis=1, bitorder="little").view(np.uint32)
    return row_off, x_off, x, y


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("kind", ["few", "grows", "dense", "last"])
def test_opening(kind, raw):
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(41 + raw)
    n_bits = [n for n in WIDTHS for _ in ROWS]
    counts = [T for _ in WIDTHS for T in ROWS]
    again = [(0, 1, 40, 1100)[c % 4] for c in range(len(n_bits))]
    maps = [(rng.integers(0, 2, (n, 128)).astype(np.float32), 0 if raw else rng.integers(0, 2, 128)) for n in n_bits]
    nb = np.array(n_bits, np.int32)
    st = binding.Store(nb, raw=raw, device=dev)
    O = oracle.Oracle(nb, raw=raw)
    for cnt, kinds in ((counts, [kind] * len(n_bits)), (again, ["dense"] * len(n_bits))):
        ro, xo, x, y = _batch(rng, n_bits, cnt, kinds, maps)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        O.learn(ro, xo, x, y)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        ref = O.export()
        assert_basis_equal(binding, st.basis(), ref)
    if kind == "last" and not raw:
        full = [c for c, (n, T) in enumerate(zip(n_bits, counts)) if n == 1024 and T > 1024]
        assert (ref["rank"][full] == 1025).all()
    st.close()


def test_timing_includes_the_opening():
    """The elimination's time of a wide context runs from its opening: 1,000
    dense rows, which all go into it, take hundreds of microseconds there and a
    few in the kernel after it."""
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(4)
    n_bits, counts = [1024, 40], [1000, 1000]
    maps = [(rng.integers(0, 2, (n, 128)).astype(np.float32), rng.integers(0, 2, 128)) for n in n_bits]
    st = binding.Store(np.array(n_bits, np.int32), device=dev)
    st.set_option(binding.F2_OPT_TIMING, 1)
    ro, xo, x, y = _batch(rng, n_bits, counts, ["dense"] * 2, maps)
    ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
    st.learn(ro_t, x_t, xo_t, y_t)
    times = st.learn_timing()
    start, end = int(times[0, 2]), int(times[0, 3])
    assert start and end - start > 200_000  # ns; 1,000 pivots of about 0.7 us
    st.close()
