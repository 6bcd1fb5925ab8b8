"""The kernels' FP64 <-> FP32 conversions on the integer pipe (gks_device.cuh)
compiled for the host: widen, narrow and both parts of split_pair equal the
compiler's conversions over every binade, ties, carries into the next binade,
the edges of the range the bit forms cover, denormals, zeros, infinities and
NaN."""
import os
import subprocess

from paper_2102_01366_gb300 import _build


def test_conversions_over_the_whole_range(tmp_path):
    exe = str(tmp_path / "host_conversions")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_conversions.cpp")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I", _build.CSRC, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.stdout, r.stderr)
    assert int(r.stdout.split()[1]) > 4_800_000
