"""What the library remembers of its kernels holds for other threads and after the
device was reset."""
import os
import subprocess
import sys
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
ap = pytest.importorskip("paper_2108_02416_gb300")
DEV = torch.device("cuda:0")


def test_aggregation_after_a_device_reset():
    here = os.path.dirname(os.path.abspath(__file__))
    p = subprocess.run([sys.executable, os.path.join(here, "_reset_worker.py")], capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0 and p.stdout.strip() == "done", p.stdout + p.stderr


# one kernel each, with different amounts of shared memory
@pytest.mark.parametrize("clusters,d,mode", [([(22, 3), (24, 3), (26, 3)], 64, 0),
                                             ([(28, 3), (30, 3), (31, 3)], 64, 0),
                                             ([(16, 3), (18, 3), (12, 5)], 64, 0),
                                             ([(9, 3), (15, 3), (24, 3)], 64, 1)])
def test_threads_with_other_numbers_of_files(clusters, d, mode):
    errors = []
    torch.cuda.synchronize()

    def run(K, r):
        try:
            a = ap.aspis_assign(K, r)
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                copies = torch.randn((a.f, r, d), device=DEV)
                sel = torch.zeros(a.f, dtype=torch.int8, device=DEV)
                buf = ap.RoundBuffers(a, d, DEV)
                for k in range(1000):
                    ap.aspis_aggregate(copies, d, a, sel, buf.det, buf.out, mode, stream)
                    if k % 100 == 99:
                        stream.synchronize()
                want = copies[:, 0].sort(0).values[(a.f - 1) // 2] if mode == 0 else copies[:, 0].double().mean(0)
                stream.synchronize()
                err = (buf.out - want).abs().max().item()
                if err > (0.0 if mode == 0 else 1e-6):
                    errors.append(f"K={K}: off by {err}")
        except Exception as e:                                   # (raised in the thread, reported below)
            errors.append(f"K={K}: {e}")

    threads = [threading.Thread(target=run, args=c) for c in clusters for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
