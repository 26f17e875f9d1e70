"""Every call of the binding on a store reaches the library with the store's
device current and that device's stream, whatever device the caller is on
(the library and torch.cuda are stand-ins: no GPU needed)."""
import contextlib
import ctypes
import types

import numpy as np
import pytest
import torch

from paper_2608_20532_gb300 import binding

HERE, STORE = 0, 1  # the caller's device and the store's


class FakeCuda:
    def __init__(self):
        self.current = HERE
        self.Event = lambda: types.SimpleNamespace(query=lambda: True, record=lambda s: None)

    def current_device(self):
        return self.current

    @contextlib.contextmanager
    def device(self, d):
        before, self.current = self.current, d.index if isinstance(d, torch.device) else d
        yield
        self.current = before

    def current_stream(self, d=None):
        d = self.current if d is None else (d.index if isinstance(d, torch.device) else d)
        return types.SimpleNamespace(cuda_stream=1000 + d)


class FakeLib:
    """Records the device that is current in each call, and the stream it gets."""

    def __init__(self, cuda):
        self.cuda, self.calls = cuda, []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append((name, self.cuda.current, args[-1] if args else None))
            if name == "f2_create":
                args[0]._obj.value = 77
            if name == "f2_merge_bases":
                args[4]._obj.value = 78
            return 0

        return call


@pytest.fixture
def env(monkeypatch):
    cuda = FakeCuda()
    lib = FakeLib(cuda)
    where = []
    fake = types.SimpleNamespace(
        cuda=cuda, device=torch.device, Tensor=torch.Tensor, int32=torch.int32, int64=torch.int64, uint8=torch.uint8,
        empty=lambda *a, device=None, **k: where.append(device) or torch.empty(*a, **k))
    monkeypatch.setattr(binding, "torch", fake)
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    monkeypatch.setattr(binding, "_dptr", lambda t: 0)
    monkeypatch.setattr(binding, "_current_stream", lambda i: 1000 + i)
    return cuda, lib, where


@pytest.mark.parametrize("device", [torch.device("cuda", STORE), f"cuda:{STORE}"])
def test_every_call_is_made_on_the_stores_device(env, device):
    cuda, lib, where = env
    st = binding.Store(np.array([8, 8], np.int32), device=device)
    i64, i32 = torch.zeros(3, dtype=torch.int64), torch.zeros(8, dtype=torch.int32)
    q, u8 = torch.zeros((2, 1), dtype=torch.int32), torch.zeros(2, dtype=torch.uint8)
    y = torch.zeros((2, 4), dtype=torch.int32)
    st.reset()
    st.learn(i64, i32, i64[:2], y)
    st.learn_host(i64, i32, i64[:2], y)
    st.basis()
    st.solve()
    st.encode(i32[:2], q)
    st.encode_epilogue(i32[:2], u8, y)
    st.encode_host(i32[:2], q, y, u8)
    st.learn_timing()
    st.device_status()
    st.import_state(st.export_state())
    merged, _ = st.merge([0, 0], 1)
    merged.reset()
    merged.close()
    st.close()
    on_stream = {"f2_create", "f2_reset", "f2_learn_batched", "f2_learn_host", "f2_get_basis", "f2_solve_affine",
                 "f2_encode_batched", "f2_encode_epilogue", "f2_encode_host", "f2_learn_timing", "f2_device_status",
                 "f2_store_export", "f2_store_import", "f2_merge_bases"}
    assert on_stream | {"f2_destroy"} <= {name for name, _, _ in lib.calls}
    for name, current, stream in lib.calls:
        if name in on_stream or name == "f2_destroy":
            assert current == STORE, name
        if name in on_stream:
            assert stream == 1000 + STORE, name
    assert cuda.current == HERE
    assert where and all((d.index if isinstance(d, torch.device) else d) == STORE for d in where)


def test_a_store_without_an_index_stays_on_its_device(env):
    """device="cuda" is the device that is current when the store is made."""
    cuda, lib, _ = env
    st = binding.Store(np.array([8], np.int32), device="cuda")
    cuda.current = STORE
    st.reset()
    assert lib.calls[-1] == ("f2_reset", HERE, 1000 + HERE)
    assert cuda.current == STORE
    cuda.current = HERE
    st.close()
    assert ctypes.c_void_p().value == st._h.value
