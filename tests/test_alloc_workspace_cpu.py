"""alloc_workspace never holds two buffers: a workspace of more than half the free memory must not fail for its alignment."""
import weakref

import torch


def test_one_buffer_at_a_time(monkeypatch):
    from paper_2412_05781_b200 import build_library
    build_library()
    from paper_2412_05781_b200 import binding as B
    real, alive = torch.empty, []

    def empty(n, **kw):
        assert all(r() is None for r in alive)
        raw = real(n + 2048, **kw)
        start = (-raw.data_ptr()) % 1024 + 512           # never aligned to 1024 bytes
        t = raw[start:start + n]
        alive.append(weakref.ref(t))
        return t

    monkeypatch.setattr(B.torch, "empty", empty)
    ws = B.alloc_workspace(5000, device="cpu")
    assert ws.numel() == 5000 and ws.data_ptr() % 1024 == 0 and len(alive) == 2
