"""Host-side pieces of the native library that need no GPU, compiled by the
host compiler alone."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_04981_gb300", "csrc")


def _run(tmp_path, source, stdin=""):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)])
    return subprocess.run([str(exe)], input=stdin, capture_output=True, text=True, check=True).stdout.split()


def test_step_cap_of_large_trees(tmp_path):
    """64 steps per node and triangle in 64 bits, held below 2^31 (the library
    takes up to 2^27 triangles; 64 x 2 x 16.8M already leaves 32 bits)."""
    sizes = [1, 2, 165_000, 16_700_000, 16_777_215, 16_777_217, 16_800_000, 1 << 25, 1 << 27]
    src = '#include <cstdio>\n#include "step_cap.h"\nint main() { long long n; int c;\n' \
          'while (scanf("%d %lld", &c, &n) == 2) printf("%d\\n", hdof::step_cap(c, n > 1 ? n - 1 : 1, n)); }'
    lines = [(c, n) for n in sizes for c in (0, 1, 1000, 2 ** 31 - 1)]
    got = [int(x) for x in _run(tmp_path, src, "\n".join(f"{c} {n}" for c, n in lines))]
    top = 2 ** 31 - 2
    for (c, n), g in zip(lines, got):
        assert g == min(c if c else 64 * (max(n - 1, 1) + n) + 64, top), (c, n)
    # every call takes its cap from there
    for f in ("trace.cu", "gbuffer.cu", "bvh.cu"):
        assert open(os.path.join(CSRC, f)).read().count("step_cap(") == 1
