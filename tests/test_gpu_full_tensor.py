"""The full-rank check on the tensor cores at the edges of its tiles: feature
counts around the 256-feature chunks and the smallest it takes, row counts
around 128-row tiles and 2,048-row chunks, feature rows at odd word offsets,
garbage above the last feature, contradicting rows in the first, last and
ragged tiles, and contexts left to the table kernel beside it.  Bit-exact
against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_basis_equal, cuda_device, dev_arrays, lib

pytestmark = pytest.mark.gpu

NS = (191, 192, 255, 256, 257, 300, 512, 513, 767, 1000, 1023, 1024)
ROWS = (2047, 2048, 2049, 2176, 4300)


def _batch(rng, n_bits, counts, maps, flips, shift):
    """Uniform rows of each context's planted map; rows listed in flips[c] get a flipped word bit.  Feature rows
    start `shift` words into x, and bits above n are set at random."""
    W = [(n + 31) // 32 for n in n_bits]
    row_off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    x_off = (shift + np.concatenate([[0], np.cumsum([k * w for k, w in zip(counts, W)])[:-1]])).astype(np.int64)
    x = rng.integers(0, 2 ** 32, int(x_off[-1] + counts[-1] * W[-1]), dtype=np.uint64).astype(np.uint32)
    y = np.zeros((int(row_off[-1]), 4), np.uint32)
    for c, n in enumerate(n_bits):
        A, b = maps[c]
        xc = x[x_off[c]:x_off[c] + counts[c] * W[c]].reshape(counts[c], W[c])
        bits = np.unpackbits(xc.view(np.uint8), axis=1, bitorder="little")[:, :n]
        yb = (bits.astype(np.float32) @ A + b).astype(np.int64) & 1
        yc = np.packbits(yb.astype(np.uint8), axis=1, bitorder="little").view(np.uint32)
        for i in flips[c]:
            if i < counts[c]:
                yc[i, int(rng.integers(4))] ^= np.uint32(1 << int(rng.integers(32)))
        y[row_off[c]:row_off[c + 1]] = yc
    return row_off, x_off, x, y


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("shift", [0, 3])
def test_full_rank_by_tensor(raw, shift):
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(5 + shift)
    n_bits, counts = [], []
    for j, n in enumerate(NS):
        n_bits += [n, n, 40]
        counts += [ROWS[j % 5], ROWS[(j + 2) % 5], 3000]  # the narrow one is left to the table kernel
    maps = [(rng.integers(0, 2, (n, 128)).astype(np.float32), 0 if raw else rng.integers(0, 2, 128)) for n in n_bits]
    none = [() for _ in n_bits]
    flips = [() if c % 4 == 0 else (0, 127, 128, 2047, 2048, counts[c] - 1) for c in range(len(n_bits))]
    st = binding.Store(np.array(n_bits, np.int32), raw=raw, device=dev)
    O = oracle.Oracle(np.array(n_bits, np.int32), raw=raw)
    for cnt, fl in (([n + 80 for n in n_bits], none), (counts, flips), ([k + 1 for k in counts], flips)):
        ro, xo, x, y = _batch(rng, n_bits, cnt, maps, fl, shift)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        O.learn(ro, xo, x, y)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        assert_basis_equal(binding, st.basis(), O.export())
    assert int((st.basis()["rank"].cpu().numpy() == np.array(n_bits) + (0 if raw else 1)).sum()) >= len(n_bits) - 2
    st.close()


@pytest.mark.parametrize("shift", [0, 1])
def test_by_features_and_rows(shift):
    """The smallest contexts that go to the tensor cores and the largest that
    stay with the tables, by features (whole and begun chunks, feature rows of
    whole 16-byte pieces and not) and by rows."""
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(25 + shift)
    n_bits, counts = [], []
    for n in (455, 456, 480, 481, 512, 513, 609, 640, 641, 680, 681, 736, 768, 769, 807, 808, 864, 865, 1023, 1024):
        for T in (2047, 2048, 5000):
            n_bits.append(n)
            counts.append(T)
    maps = [(rng.integers(0, 2, (n, 128)).astype(np.float32), rng.integers(0, 2, 128)) for n in n_bits]
    flips = [() if c % 5 == 0 else (0, 129, 2047, 2048, counts[c] - 1) for c in range(len(n_bits))]
    nb = np.array(n_bits, np.int32)
    st = binding.Store(nb, device=dev)
    O = oracle.Oracle(nb)
    for cnt, fl in (([n + 80 for n in n_bits], [()] * len(n_bits)), (counts, flips)):
        ro, xo, x, y = _batch(rng, n_bits, cnt, maps, fl, shift)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        O.learn(ro, xo, x, y)
        torch.cuda.synchronize()
        assert st.device_status() == binding.F2_OK
        assert_basis_equal(binding, st.basis(), O.export())
    st.close()


@pytest.mark.parametrize("raw", [False, True])
def test_a_wait_that_gives_up_commits_nothing(raw):
    """A call whose check gives up reports it and leaves the contradiction
    records and row counts of the contexts it was checking as they were (the
    narrow context, checked by the table kernel, is counted); the next call
    goes on from there."""
    dev = cuda_device()
    binding = lib()
    rng = np.random.default_rng(15)
    n_bits = [500, 768, 1024, 40]
    wide = np.array(n_bits) >= 500
    maps = [(rng.integers(0, 2, (n, 128)).astype(np.float32), 0 if raw else rng.integers(0, 2, 128)) for n in n_bits]
    st = binding.Store(np.array(n_bits, np.int32), raw=raw, device=dev)
    O = oracle.Oracle(np.array(n_bits, np.int32), raw=raw)

    def learn(counts, flips, learner):
        ro, xo, x, y = _batch(rng, n_bits, counts, maps, flips, 0)
        ro_t, x_t, xo_t, y_t = dev_arrays(binding, dev, ro, x, xo, y)
        st.learn(ro_t, x_t, xo_t, y_t)
        torch.cuda.synchronize()
        if learner is not None:
            learner.learn(ro, xo, x, y)

    def state():
        return {k: binding.to_numpy(v).copy() for k, v in st.basis().items()}

    learn([n + 80 for n in n_bits], [(), (840,), (), ()], O)  # one recorded already
    before = state()
    assert (before["rank"] == np.array(n_bits) + (0 if raw else 1)).all()
    st.set_option(binding.F2_OPT_FAIL_WAIT, 1)
    learn([4300, 3000, 9000, 3000], [(0, 2100)] * 4, None)
    assert st.device_status() == binding.F2_ERR_TIMEOUT
    after = state()
    for k in ("contra", "first_contra", "n_contra", "rows_seen"):
        assert np.array_equal(after[k][wide], before[k][wide]), k
        assert (after[k][~wide] != before[k][~wide]).all(), k
    for k in ("rank", "pivot_mask", "basis_x", "basis_z"):
        assert np.array_equal(after[k], before[k]), k
    st.set_option(binding.F2_OPT_FAIL_WAIT, 0)
    learn([4300, 2731, 9000, 0], [(7, 4000)] * 4, O)
    assert st.device_status() == binding.F2_OK
    ref, got = O.export(), state()
    for k in ("rank", "contra", "first_contra", "n_contra", "rows_seen"):
        assert np.array_equal(got[k][wide].astype(np.int64), ref[k][wide].astype(np.int64)), k
    st.close()
