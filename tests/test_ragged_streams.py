"""solve_ragged's streams when a group fails, with the CUDA calls replaced (no GPU needed)."""
import contextlib

import pytest

torch = pytest.importorskip("torch")
from paper_1510_04686_gb300 import negf as B  # noqa: E402


class _Stream:
    def __init__(self, name):
        self.name, self.device, self.waits = name, "dev", []

    def wait_stream(self, other):
        self.waits.append(other)


@pytest.mark.parametrize("host_check", [0, 4])  # one host thread, a thread per group
@pytest.mark.parametrize("bad", [0, 1, 2])
def test_a_failing_group_leaves_no_stream_behind(monkeypatch, host_check, bad):
    cur, side = _Stream("cur"), []

    def stream(device=None):
        side.append(_Stream(f"side{len(side)}"))
        return side[-1]

    null = lambda *a, **k: contextlib.nullcontext()  # noqa: E731
    monkeypatch.setattr(B.torch.cuda, "current_stream", lambda *a: cur)
    monkeypatch.setattr(B.torch.cuda, "Stream", stream)
    monkeypatch.setattr(B.torch.cuda, "stream", null)
    monkeypatch.setattr(B.torch.cuda, "device", null)
    monkeypatch.setattr(B, "_RAGGED_STREAMS", {})
    monkeypatch.setattr(B, "library", lambda: None)
    monkeypatch.setattr(B, "Device", lambda Hd, Hu: Hd.shape[-1])
    sizes, started = [8, 6, 4], []

    def lead(dev, E, sys_idx, opt):
        started.append(dev)
        if dev == sizes[bad]:
            raise B.NegfError(2, "lead")
        return {"sigma_R": None, "sigma_L": None}

    monkeypatch.setattr(B, "lead_selfenergy", lead)
    monkeypatch.setattr(B, "rgf_solve", lambda dev, E, *a, **k: {"density": E.clone()})
    systems = [(torch.zeros(2, b, b), torch.zeros(1, b, b), torch.zeros(1)) for b in sizes]
    with pytest.raises(B.NegfError):
        B.solve_ragged(systems, B._Opt(sr_host_check=host_check))
    assert started and len(side) == 3
    # the calling stream waits for every side stream that may have work in flight
    assert cur.waits == side
