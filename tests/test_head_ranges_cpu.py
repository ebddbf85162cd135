"""The ranges of heads that the host-tensor step works by: alignment of everything that is accessed in 16-byte pieces, and what the first kernel of
an update clears, for odd numbers of tokens and ranges that begin at odd heads, on both paths of the planner."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_range_of_heads_is_aligned_and_clears_its_own_words(tmp_path):
    from paper_2602_01801_b200 import build
    build.build_library()
    own = ("update_kernels.cu", "fastar_api.cu")           # the program includes these
    objs = [os.path.join(build.LIB_DIR, "obj", s.replace(".cu", ".o")) for s in build.SOURCES if s not in own]
    exe = str(tmp_path / "head_ranges")
    # PTX only: no device code runs, and assembling it is most of the build
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-Xcicc", "-O0", os.path.join(ROOT, "tests", "head_ranges.cu")] + objs + ["-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
