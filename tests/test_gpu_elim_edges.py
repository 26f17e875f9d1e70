"""Elimination at the edges of its tiles: row counts around the 32 rows of a
warp round, the 128 rows of a first block and the 256 of a CTA round, widths
around the word and kernel boundaries, low-rank rows (so that later rounds run
against a lookup table) and dense ones, rows that contradict earlier ones and a
second call on the learned store.  Every array is bit-exact against the CPU
oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_basis_equal, csr_from_rows, cuda_device, dev_arrays, lib

pytestmark = pytest.mark.gpu

ROWS = (1, 31, 32, 33, 64, 127, 128, 129, 160, 257, 520, 900)
WIDTHS = (1, 8, 31, 32, 48, 63, 64, 70, 95, 96, 127, 128, 160, 255, 287)


def _rows(rng, n, count, gens, flip):
    """`count` rows of x in the span of `gens` random vectors plus an offset, y planted; a few repeats, some with a
    flipped word bit."""
    W = (n + 31) // 32
    A = rng.integers(0, 2, (n, 128)).astype(np.uint8)
    b = rng.integers(0, 2, 128).astype(np.uint8)
    G = rng.integers(0, 2, (gens, n)).astype(np.uint8)
    x = (rng.integers(0, 2, (count, gens)).astype(np.int64) @ G + rng.integers(0, 2, n)) & 1
    y = ((x @ A) + b) & 1
    for i in range(1, count):
        if rng.random() < 0.2:  # a repeat
            j = int(rng.integers(i))
            x[i], y[i] = x[j], y[j]
            if flip and rng.random() < 0.3:
                y[i, int(rng.integers(128))] ^= 1
    xw = np.zeros((count, W * 32), np.uint8)
    xw[:, :n] = x
    xw = np.packbits(xw, axis=1, bitorder="little").view(np.uint32).reshape(count, W)
    yw = np.packbits(y.astype(np.uint8), axis=1, bitorder="little").view(np.uint32).reshape(count, 4)
    return list(zip(xw, yw))


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("mode", ["default", "cta", "no_tables", "no_dedup"])
def test_edges(mode, raw):
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(77)
    n_bits, batches = [], [[], []]
    for n in WIDTHS:
        for k, count in enumerate(ROWS):
            gens = int(rng.integers(1, n + 1)) if k % 2 else n
            n_bits.append(n)
            rows = _rows(rng, n, count + count // 3, gens, flip=k % 3 == 0)
            batches[0].append(rows[:count])
            batches[1].append(rows[count:])
    n_bits = np.array(n_bits, np.int32)
    st = binding.Store(n_bits, raw=raw, device=dev)
    if mode == "cta":
        st.set_option(binding.F2_OPT_HEAVY_ROWS, 1)
    else:
        st.set_option(binding.F2_OPT_HEAVY_ROWS, 4096)  # a warp each (the store is small enough for a CTA each)
        st.set_option(binding.F2_OPT_WARP_WORK, 1 << 40)
    if mode == "no_tables":
        st.set_option(binding.F2_OPT_ELIM_TABLES, 0)
    if mode == "no_dedup":
        st.set_option(binding.F2_OPT_DEDUP, 0)
    O = oracle.Oracle(n_bits, raw=raw)
    for rows in batches:
        ro, xo, x, y = csr_from_rows(n_bits, rows)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        O.learn(ro, xo, x, y)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        assert_basis_equal(binding, st.basis(), O.export())
    st.close()
