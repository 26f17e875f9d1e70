"""The duplicate pass of 10..16-word feature rows at its edges: row counts
around the warp, quad, CTA and piece sizes, rows that nearly all repeat, that
never do and that outgrow the numbered distinct rows, feature rows at odd word
offsets, repeats with a flipped word bit, contexts split over CTAs and not.
Bit-exact against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_basis_equal, cuda_device, dev_arrays, lib

pytestmark = pytest.mark.gpu

COUNTS = (129, 256, 257, 1000, 4096, 4097, 16384, 16500, 40000)
WIDTHS = (289, 320, 352, 383, 448, 481, 512)


@pytest.mark.parametrize("shards", [1, 4])
@pytest.mark.parametrize("shift", [0, 1])
def test_wide_rows(shards, shift):
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(9 + shift)
    n_bits, counts = [], []
    for j, T in enumerate(COUNTS):
        for k in range(3):  # few distinct rows, many, all
            n_bits.append(WIDTHS[(3 * j + k) % len(WIDTHS)])
            counts.append(T)
    W = [(n + 31) // 32 for n in n_bits]
    row_off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    x_off = (shift + np.concatenate([[0], np.cumsum([t * w for t, w in zip(counts, W)])[:-1]])).astype(np.int64)
    x = rng.integers(0, 2 ** 32, int(x_off[-1] + counts[-1] * W[-1]), dtype=np.uint64).astype(np.uint32)
    y = np.zeros((int(row_off[-1]), 4), np.uint32)
    for c, (n, T) in enumerate(zip(n_bits, counts)):
        distinct = (max(2, T // 50), max(2, T // 2), T)[c % 3]
        A = rng.integers(0, 2, (24, 128)).astype(np.uint8)
        G = rng.integers(0, 2, (24, n)).astype(np.uint8)
        sel = rng.integers(0, 2, (distinct, 24)).astype(np.uint8)
        xb = np.zeros((distinct, W[c] * 32), np.uint8)
        xb[:, :n] = (sel.astype(np.int64) @ G) & 1
        yb = ((sel.astype(np.int64) @ A) & 1).astype(np.uint8)
        src = rng.integers(0, distinct, T) if c % 3 < 2 else np.arange(T)
        xc = np.packbits(xb, axis=1, bitorder="little").view(np.uint32)[src]
        if n % 32:  # bits above n are ignored: a repeat may differ there
            xc[:, -1] |= rng.integers(0, 2 ** 32, T, dtype=np.uint64).astype(np.uint32) & ~np.uint32((1 << (n % 32)) - 1)
        yc = np.packbits(yb, axis=1, bitorder="little").view(np.uint32)[src].copy()
        for i in rng.integers(1, T, 3):
            yc[i, 1] ^= 4
        x[x_off[c]:x_off[c] + T * W[c]] = xc.reshape(-1)
        y[row_off[c]:row_off[c + 1]] = yc
    nb = np.array(n_bits, np.int32)
    st = binding.Store(nb, device=dev)
    st.set_option(binding.F2_OPT_DEDUP_SHARDS, shards)
    ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, row_off, x, x_off, y)
    st.learn(ro_t, x_t, xo_t, y_t)
    torch.cuda.synchronize()
    assert st.device_status() == binding.F2_OK
    O = oracle.Oracle(nb)
    O.learn(row_off, x_off, x, y)
    assert_basis_equal(binding, st.basis(), O.export())
    st.close()
