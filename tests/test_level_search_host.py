"""The search of one level on the host, for sets that hold vertices of the graph
only and for sets with bits at or above n (tw_expand_level_static takes its sets
unchecked): every loop ends, bits at or above n count as vertices without edges,
and the results are those of plain closures (tests/c/level_search_host.cu)."""
import os
import subprocess

from paper_1709_09990_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_search_ends_and_is_exact_for_any_set(tmp_path):
    exe = tmp_path / "level_search_host"
    subprocess.check_call([build._nvcc(), *build.ARCH, "-std=c++17", "-O1", "-I", build.INCLUDE,
                           os.path.join(HERE, "c", "level_search_host.cu"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.startswith("ok "), out.stdout + out.stderr
