"""The host's thread loops when memory or threads run out (CPU): no range is
lost or run twice, an exception reaches the caller and no thread is left
running (a joinable thread that is destroyed ends the process)."""
import os
import subprocess

from paper_2102_01366_gb300 import _build


def test_loops_survive_failed_allocations_and_thread_starts(tmp_path):
    exe = str(tmp_path / "host_threads")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_threads.cpp")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", _build.CSRC, src, "-o", exe, "-ldl"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    word, done, refused = r.stdout.split()
    # 16 failures planted 50 times: each leaves a loop done or refused, some of either kind
    assert word == "ok" and int(done) + int(refused) == 800 and int(done) > 0 and int(refused) > 0
