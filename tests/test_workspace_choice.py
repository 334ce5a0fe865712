"""The binding's workspace: of the preferred size where memory reaches that far, of the needed one where it does not, and then kept
without asking again on every call.  No device: the allocator is a stand-in that refuses above a limit."""
import torch

from paper_2503_13089_b200 import binding as cc


class _Room:
    def __init__(self, nbytes):
        self.nbytes = nbytes

    def numel(self):
        return self.nbytes


def _context(monkeypatch, limit):
    asked, told = [], []

    def empty(nbytes, dtype=None, device=None):
        asked.append(nbytes)
        if nbytes > limit:
            raise torch.OutOfMemoryError("refused")
        return _Room(nbytes)

    monkeypatch.setattr(cc.torch, "empty", empty)
    monkeypatch.setattr(cc, "cc_set_workspace", lambda ctx, ws, n: told.append(n))
    c = object.__new__(cc.Context)
    c._h, c.device, c._ws, c._ws_refused = None, 0, None, None
    return c, asked, told


def test_a_refused_size_is_not_asked_for_again(monkeypatch):
    N, g, K = 4 << 20, 4, 65536
    need, want = cc.cc_workspace_bytes(N, g, K), cc.cc_workspace_bytes_preferred(N, g, K)
    assert want > need
    c, asked, told = _context(monkeypatch, (need + want) // 2)
    c.ensure_workspace(N, g, K)
    assert asked == [want, need] and told == [need] and c._ws.numel() == need
    for _ in range(3):
        c.ensure_workspace(N, g, K)
    assert asked == [want, need] and told == [need]                     # kept
    c.ensure_workspace(2 * N, g, K)                                     # larger: only what it needs
    assert asked[2:] == [cc.cc_workspace_bytes(2 * N, g, K)]
    n0 = len(asked)
    c.ensure_workspace(N // 8, g, K)                                    # smaller: there already
    assert len(asked) == n0


def test_with_memory_the_preferred_size_is_taken(monkeypatch):
    N, g, K = 4 << 20, 4, 65536
    c, asked, told = _context(monkeypatch, 1 << 40)
    c.ensure_workspace(1000, g, 16)
    c.ensure_workspace(N, g, K)
    c.ensure_workspace(N, g, K)
    assert asked[1:] == [cc.cc_workspace_bytes_preferred(N, g, K)] == told[1:]


def test_a_call_that_cannot_be_served_raises(monkeypatch):
    c, asked, _ = _context(monkeypatch, 1 << 20)
    try:
        c.ensure_workspace(4 << 20, 4, 65536)
    except torch.OutOfMemoryError:
        pass
    else:
        raise AssertionError("no error")
    assert c._ws is None
