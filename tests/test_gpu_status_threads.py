"""sweep_status keeps a word of page-locked memory per thread: a thread that read
a status may end while another one captures a graph in the global mode (torch's
default), without spoiling that capture."""
import os
import threading
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_thread_ends_during_another_threads_capture():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14189_gb300 import sweep
    ws = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    read, leave, codes = threading.Event(), threading.Event(), []

    def reader():
        codes.append(sweep.status(ws))
        read.set()
        leave.wait(30)

    t = threading.Thread(target=reader)
    t.start()
    assert read.wait(30)
    task = f"/proc/self/task/{t.native_id}"  # gone once the thread's own data is freed
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x.add_(1)
        leave.set()
        t.join()
        end = time.monotonic() + 10
        while os.path.exists(task) and time.monotonic() < end:
            time.sleep(0.01)
        assert not os.path.exists(task)
        x.add_(1)
    g.replay()
    torch.cuda.synchronize()
    assert codes == [sweep.OK] and x.tolist() == [2.0] * 8
