"""Memory a ground state with its vector takes beside its workspace: bounded over all
calls, kept between calls while a handle of the device lives, and given back."""
import os
import subprocess
import sys
import threading
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]
GIB = 1 << 30
SLACK = 128 << 20                                       # tables, scratch and CUDA's own


def _sector():
    import paper_1204_3425_gb300 as hub
    from workload import ring
    return hub, hub.hubbard_sector_create(13, ring(13), 6, 6, 1.0, 4.0)


def _state(hub, H):
    v = torch.rand(H.D, dtype=torch.float64, device="cuda") - 0.5
    return v, torch.empty_like(v), torch.empty(hub.lanczos_workspace_bytes(H), dtype=torch.uint8, device="cuda")


CHILD = """
import torch
import tests.test_gpu_store as T
hub, H = T._sector()
v, psi, ws = T._state(hub, H)
torch.cuda.synchronize()
free = [torch.cuda.mem_get_info()[0]]
hub.lanczos_ground_state(H, v, 1000, 1e-10, workspace=ws, psi_out=psi)
torch.cuda.synchronize()
free.append(torch.cuda.mem_get_info()[0])
H.close()
torch.cuda.synchronize()
free.append(torch.cuda.mem_get_info()[0])
print(*free)
"""


def test_memory_is_given_back_with_the_last_handle():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]          # a process of its own: no handle of another test is alive
    before, held, after = map(int, r.stdout.split())
    assert before - held <= GIB + SLACK
    assert before - after <= SLACK


def test_concurrent_calls_share_one_bound():
    states, streams = [], [torch.cuda.Stream() for _ in range(3)]
    for _ in streams:
        hub, H = _sector()
        states.append((H,) + _state(hub, H))
    want = []
    for H, v, psi, ws in states:
        hub.lanczos_ground_state(H, v, 1000, 1e-10, workspace=ws, psi_out=psi)
        want.append(psi.clone())
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]               # the pool holds at most its bound already
    low, stop = [before], threading.Event()

    def watch():
        while not stop.is_set():
            low[0] = min(low[0], torch.cuda.mem_get_info()[0])
            time.sleep(0.0005)

    def solve(k):
        H, v, psi, ws = states[k]
        with torch.cuda.stream(streams[k]):
            for _ in range(4):
                hub.lanczos_ground_state(H, v, 1000, 1e-10, workspace=ws, psi_out=psi, stream=streams[k])

    w = threading.Thread(target=watch)
    ts = [threading.Thread(target=solve, args=(k,)) for k in range(3)]
    w.start()
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    stop.set()
    w.join()
    torch.cuda.synchronize()
    assert before - low[0] <= SLACK                     # three calls at once: no more than one had
    for (H, v, psi, ws), p in zip(states, want):        # kept or replayed, the same vector
        assert torch.equal(psi, p)
        H.close()
