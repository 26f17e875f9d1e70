"""The check of handed-off contexts at its edges: more contexts than a warp
looks at in one step, chunks of one row and of all, feature rows at word
offsets that allow four-, two- and one-word loads, bases of single-bit rows
and of rows with other columns, rows of features with and without the
constant, rows outside the span in the check.  Bit-exact against the CPU
oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_20532_gb300 import workloads
from gpu_util import KEYS, as_bytes, assert_basis_equal, cuda_device, dev_arrays, gpu_learn_workload, lib

pytestmark = pytest.mark.gpu

WIDTHS = (1, 20, 31, 32, 33, 64, 127, 128, 192, 255, 256, 287, 288, 320, 384, 415, 512, 543)


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_check(shift, raw):
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(70 + shift + 10 * raw)
    n_bits = [n + (raw and n == 543) for n in WIDTHS for _ in range(4)]
    counts = [int(rng.choice([512, 513, 800, 1023, 1025, 1700])) for _ in n_bits]
    W = [(n + 31) // 32 for n in n_bits]
    row_off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    x_off, at = [], 0
    for t, w in zip(counts, W):  # the same alignment for every context: `shift` words off a 16-byte boundary
        x_off.append(at + shift)
        at = (at + shift + t * w + 3) // 4 * 4
    x_off = np.array(x_off, np.int64)
    x = rng.integers(0, 2 ** 32, at, dtype=np.uint64).astype(np.uint32)
    y = np.zeros((int(row_off[-1]), 4), np.uint32)
    for c, (n, T) in enumerate(zip(n_bits, counts)):
        r = min(n, 1 + c % 9)
        G = np.zeros((r, n), np.uint8)
        if c % 4 < 2:
            G[np.arange(r), rng.permutation(n)[:r]] = 1
        else:
            G[:] = rng.integers(0, 2, (r, n))
        base = rng.integers(0, 2, n) if c % 2 else np.zeros(n, np.int64)
        A = rng.integers(0, 2, (n, 128)).astype(np.int64)
        xb = np.zeros((T, 32 * W[c]), np.uint8)
        xb[:, :n] = (base + rng.integers(0, 2, (T, r)) @ G.astype(np.int64)) & 1
        if c % 3 == 0:  # a row outside the span, late
            xb[T - 1 - c % 7, rng.integers(0, n)] ^= 1
        yb = ((xb[:, :n].astype(np.int64) @ A) & 1).astype(np.uint8)
        xc = np.packbits(xb, axis=1, bitorder="little").view(np.uint32)
        if n % 32:  # bits above n are ignored
            xc[:, -1] |= rng.integers(0, 2 ** 32, T, dtype=np.uint64).astype(np.uint32) & ~np.uint32((1 << (n % 32)) - 1)
        yc = np.packbits(yb, axis=1, bitorder="little").view(np.uint32).copy()
        for i in rng.integers(T // 2, T, c % 4):
            yc[i, 2] ^= 16
        x[x_off[c]:x_off[c] + T * W[c]] = xc.reshape(-1)
        y[row_off[c]:row_off[c + 1]] = yc
    nb = np.array(n_bits, np.int32)
    O = oracle.Oracle(nb, raw=raw)
    O.learn(row_off, x_off, x, y)
    for opts in ({binding.F2_OPT_DEDUP: 0}, {}):
        st = binding.Store(nb, device=dev, raw=raw)
        for k, v in {binding.F2_OPT_HEAVY_ROWS: 1, binding.F2_OPT_HANDOFF_REPS: 8, **opts}.items():
            st.set_option(k, v)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, row_off, x, x_off, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        assert_basis_equal(binding, st.basis(), O.export())
        st.close()


def test_default_without_memory():
    """A call that would hand off by default goes without where the check's
    records cannot be allocated: nothing that the caller did not ask for may
    fail the call."""
    dev = cuda_device()
    binding = lib()
    cfg = dict(num_ctx=16, layout=workloads.LAYOUT_UNIFORM_BITS, n_fixed=300, rows_fixed=66000, dup_frac=0.5,
               density=0.05, n_contra=3)
    wl = workloads.generate(cfg, 31)
    assert wl.total_rows >= 1 << 20
    got = []
    for fail_at in (-1, 2):  # after the two lists of the duplicate pass
        st = binding.Store(wl.n_bits, device=dev)
        st.set_option(binding.F2_OPT_FAIL_ALLOC, fail_at)
        gpu_learn_workload(binding, st, wl, dev)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        got.append({k: as_bytes(binding.to_numpy(v)).copy() for k, v in st.basis().items()})
        st.close()
    for k in KEYS:
        assert np.array_equal(got[0][k], got[1][k]), k


def test_default_of_a_mixed_store():
    """The default hand-off of a store that mixes contexts of every width, long
    contexts of low rank (which walk their pivots) and of high rank (which run
    against a lookup table), some with a row outside the span late; and the
    option set and set back to the default."""
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(88)
    n_bits, ranks = [], []
    for n in (40, 64, 95, 128, 200, 287, 320, 500):
        for r in (3, 9, n // 3, n - 2):
            n_bits.append(n)
            ranks.append(r)
    T = 33000
    nb = np.array(n_bits, np.int32)
    W = (nb.astype(np.int64) + 31) // 32
    row_off = np.arange(len(n_bits) + 1, dtype=np.int64) * T
    assert int(row_off[-1]) >= 1 << 20
    x_off = np.concatenate([[0], np.cumsum(T * W)[:-1]]).astype(np.int64)
    x = np.zeros(int(T * W.sum()), np.uint32)
    y = np.zeros((int(row_off[-1]), 4), np.uint32)
    for c, (n, r) in enumerate(zip(n_bits, ranks)):
        G = rng.integers(0, 2, (r, n)).astype(np.float32)
        A = rng.integers(0, 2, (n, 128)).astype(np.float32)
        xb = np.zeros((T, 32 * int(W[c])), np.uint8)
        xb[:, :n] = (rng.integers(0, 2, (T, r)).astype(np.float32) @ G).astype(np.int64) & 1
        if c % 3 == 0:
            xb[T - 1 - 7 * c, int(rng.integers(n))] ^= 1
        yb = ((xb[:, :n].astype(np.float32) @ A).astype(np.int64) & 1).astype(np.uint8)
        yc = np.packbits(yb, axis=1, bitorder="little").view(np.uint32).copy()
        for i in rng.integers(T // 2, T, c % 4):
            yc[i, 2] ^= 16
        x[x_off[c]:x_off[c] + T * W[c]] = np.packbits(xb, axis=1, bitorder="little").view(np.uint32).reshape(-1)
        y[row_off[c]:row_off[c + 1]] = yc
    O = oracle.Oracle(nb)
    O.learn(row_off, x_off, x, y)
    ref = O.export()
    st = binding.Store(nb, device=dev)
    ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, row_off, x, x_off, y)
    for option in (None, 0, -1, 2048):
        if option is not None:
            st.set_option(binding.F2_OPT_HANDOFF_REPS, option)
        st.reset()
        st.learn(ro_t, x_t, xo_t, y_t)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        assert_basis_equal(binding, st.basis(), ref)
    with pytest.raises(binding.F2Error):
        st.set_option(binding.F2_OPT_HANDOFF_REPS, -2)
    st.close()
