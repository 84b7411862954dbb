"""The size of the adjoint's workspace (kept by a Problem for its lifetime): all units where that is little,
at most 2 GiB more than the forward's, and the forward's size where the growth is above 256 MiB and more than
a sixteenth of the free memory, or the caller gave a cap.  Host only: the device's free memory is made up."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2311_12134_gb300 import conductivity as C

MB, GB = 1 << 20, 1 << 30


def _size(monkeypatch, forward, mn, al, free, cached=0, capped=False):
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda device=None: (free, 280 * GB))
    monkeypatch.setattr(torch.cuda, "memory_reserved", lambda device=None: cached + GB)
    monkeypatch.setattr(torch.cuda, "memory_allocated", lambda device=None: GB)
    monkeypatch.setattr(torch, "empty", lambda n, **kw: types.SimpleNamespace(numel=lambda: n))
    p = types.SimpleNamespace(workspace=types.SimpleNamespace(numel=lambda: forward), _capped=capped, device="cuda:0")
    return C.Problem._adjoint_workspace(p, mn, al).numel()


def test_adjoint_workspace_is_bounded(monkeypatch):
    assert _size(monkeypatch, 3 * MB, 7 * MB, 19 * MB, 200 * GB) == 19 * MB
    assert _size(monkeypatch, 160 * MB, 161 * MB, 494 * MB, 200 * GB) == 494 * MB
    assert _size(monkeypatch, 500 * MB, 300 * MB, 10 * GB, 200 * GB) == 2 * GB + 500 * MB  # not 8 GB
    assert _size(monkeypatch, 3 * GB, 2 * GB, 3 * GB + 600 * MB, 200 * GB) == 3 * GB + 600 * MB
    assert _size(monkeypatch, 160 * MB, 161 * MB, 494 * MB, 200 * GB, capped=True) == 161 * MB


def test_adjoint_workspace_leaves_the_rest_of_a_full_device(monkeypatch):
    assert _size(monkeypatch, 160 * MB, 161 * MB, 494 * MB, 4 * GB) == 161 * MB
    assert _size(monkeypatch, 160 * MB, 161 * MB, 494 * MB, 1 * GB, cached=20 * GB) == 494 * MB
    assert _size(monkeypatch, 3 * MB, 7 * MB, 19 * MB, 4 * GB) == 19 * MB
    assert _size(monkeypatch, 3 * MB, 7 * MB, 263 * MB, 0) == 263 * MB  # 256 MB are taken without asking
    assert _size(monkeypatch, 3 * MB, 7 * MB, 264 * MB, 0) == 7 * MB
