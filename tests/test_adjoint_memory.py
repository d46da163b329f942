"""Which workspace the binding asks for: every alpha kept only where it leaves the memory to others (no GPU: the
library's sizes, the allocator and the driver's answer are stand-ins)."""
import pytest
import torch

from paper_2211_00621_gb300 import api, _lib

GB = 1 << 30


class _Sizes:
    def __init__(self, full, small):
        self.full, self.small = full, small

    def hmm_adjoint_workspace_size(self, *a):
        return self.full

    def hmm_adjoint_min_workspace_size(self, *a):
        return self.small


@pytest.fixture
def memory(monkeypatch):
    state = dict(free=0, reserved=0, allocated=0, asked=[], refuse=None)

    def ws(n, device):
        state["asked"].append(n)
        if state["refuse"] is not None and n >= state["refuse"]:
            raise torch.OutOfMemoryError("no")
        return n

    monkeypatch.setattr(api, "_ws", ws)
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda d=None: (state["free"], 280 * GB))
    monkeypatch.setattr(torch.cuda, "memory_reserved", lambda d=None: state["reserved"])
    monkeypatch.setattr(torch.cuda, "memory_allocated", lambda d=None: state["allocated"])
    return state


def _ask(full, small):
    return api._adjoint_ws(_Sizes(full, small), _lib.accel_hmm_model(), 8, 100, 50, "cuda")


@pytest.mark.parametrize("full,free,cached,kept", [
    (3 * GB, 270 * GB, 0, True), (3 * GB, 20 * GB, 0, False), (3 * GB, 20 * GB, 4 * GB, True), (32 * GB, 256 * GB, 0, True),
    (32 * GB, 255 * GB, 0, False), (256 << 20, 300 << 20, 0, True), ((256 << 20) + 1, 1 * GB, 0, False)])
def test_every_alpha_only_with_room_to_spare(memory, full, free, cached, kept):
    memory.update(free=free, reserved=10 * GB + cached, allocated=10 * GB)
    assert _ask(full, full // 6) == (full if kept else full // 6)
    assert len(memory["asked"]) == 1                # near the limit no large allocation is tried


def test_graphs_held_at_once_leave_the_memory_to_others(memory):
    # twenty graphs of a program, whose checkpoints fitted into the memory with 100 GB to spare
    memory.update(free=250 * GB)
    for _ in range(20):
        memory["free"] -= _ask(30 * GB, 5 * GB)
    assert memory["free"] >= 100 * GB


def test_an_allocator_without_figures(memory, monkeypatch):
    def none(d=None):
        raise RuntimeError("not supported")

    monkeypatch.setattr(torch.cuda, "memory_reserved", none)
    memory.update(free=20 * GB)
    assert _ask(3 * GB, 1 * GB) == 1 * GB and _ask(2 * GB, 1 * GB) == 2 * GB


def test_a_refused_allocation_falls_back(memory):
    memory.update(free=270 * GB, refuse=2 * GB)
    assert _ask(3 * GB, 1 * GB) == 1 * GB
    assert memory["asked"] == [3 * GB, 1 * GB]
