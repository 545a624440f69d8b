"""Host-side pieces of the native library that need no GPU, compiled by the
host compiler alone."""
import os
import subprocess
from fractions import Fraction

import numpy as np

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


def test_three_float_sums(tmp_path):
    """Sum3 against the exact sum: its value is within one rounding of a double
    (2^-52 of the sum of magnitudes leaves room for the last addition too),
    term by term, with rounding errors handed in, and over a tree of partial
    sums, where a pair of floats would drop what lies 2^-48 below."""
    rng = np.random.default_rng(0)
    sets = [np.float32([1.0, 2.0 ** -25, 2.0 ** -49]), np.float32([1.0, 2.0 ** -25, 2.0 ** -28, -1.0, -2.0 ** -25]),
            rng.uniform(0, 1, 96).astype(np.float32), rng.normal(size=400).astype(np.float32),
            (rng.normal(size=400) * np.exp2(rng.uniform(-30, 30, 400))).astype(np.float32)]
    src = """#include <cstdio>
#include "sum3.cuh"
int main() {
    int n;
    while (scanf("%d", &n) == 1) {
        hdof::Sum3 s{}, part[32] = {}, sq{};
        for (int k = 0; k < n; ++k) {
            float x;
            if (scanf("%a", &x) != 1) return 1;
            s.add(x);
            part[k % 32].add(x);
            const double d = (double)x * x;
            const float p = (float)d;
            sq.add(p, (float)(d - p));
        }
        for (int o = 16; o; o >>= 1) {
            hdof::Sum3 t[32];
            for (int k = 0; k < 32; ++k) { t[k] = part[k]; t[k].add(part[k ^ o]); }
            for (int k = 0; k < 32; ++k) part[k] = t[k];
        }
        printf("%a %a %a\\n", s.value(), part[0].value(), sq.value());
    }
}"""
    got = _run(tmp_path, src, "\n".join(f"{len(x)} " + " ".join(float(v).hex() for v in x) for x in sets))
    for x, g in zip(sets, np.reshape([float.fromhex(v) for v in got], (-1, 3))):
        ex = [Fraction(float(v)) for v in x]
        for k, terms in ((0, ex), (1, ex), (2, [v * v for v in ex])):
            assert abs(Fraction(float(g[k])) - sum(terms)) <= Fraction(1, 2 ** 52) * sum(map(abs, terms)), (k, len(x))
    # where a double is exact, so is the sum
    assert float.fromhex(got[0]) == 1.0 + 2.0 ** -25 + 2.0 ** -49 and float.fromhex(got[4]) == 2.0 ** -28


def test_mask_strips_of_an_image_and_of_a_batch(tmp_path):
    """Strips are cut shorter only while all the warps of a launch are too few:
    alone, a 256x256 view takes 8 rows, among 64 of them 32."""
    src = """#include <cstdio>
#include <vector>
#include "mask_rows.h"
int main() {
    int n, sms;
    while (scanf("%d %d", &sms, &n) == 2) {
        std::vector<int> s(2 * n);
        for (int& v : s) if (scanf("%d", &v) != 1) return 1;
        printf("%d\\n", hdof::sweep_rows([&](int r) {
            long long t = 0;
            for (int k = 0; k < n; ++k) t += hdof::sweep_warps(s[2 * k], s[2 * k + 1], r);
            return t; }, sms));
    }
}"""
    cases = [(152, [(256, 256)]), (152, [(128, 128)]), (152, [(1920, 1080)]), (152, [(640, 480)]), (152, [(1, 1)]),
             (152, [(1280, 720)]), (152, [(256, 256)] * 12), (152, [(256, 256)] * 64), (152, [(640, 480)] * 4),
             (152, [(1920, 1080), (256, 256)]), (8, [(256, 256)]), (1000, [(1920, 1080)]), (152, [(16384, 16384)] * 64)]
    got = [int(g) for g in _run(tmp_path, src, "\n".join(f"{m} {len(s)} " + " ".join(f"{w} {h}" for w, h in s)
                                                         for m, s in cases))]
    for (m, s), g in zip(cases, got):
        warps = [sum(-(-w // 26) * -(-h // r) for w, h in s) for r in (32, 16, 8)]
        assert g == next((r for r, t in zip((32, 16, 8), warps) if t >= 8 * m), 8), (m, s[:2], len(s))
    assert got[0] == 8 and got[7] == 32  # a 256x256 view alone, and 64 of them


def test_default_trace_rule(tmp_path):
    """Form and ray order of a view: packets below 0.1 of the view's height,
    earlier rays for a batch's small views; sorted by lens bin from 0.01 and
    from a lens that spreads rays over more than a packet's pixel block on
    (K sqrt(spp) of 14, in a batch 36)."""
    src = """#include <cstdio>
#include "trace_rule.h"
int main() {
    float kh; int H, spp, batch;
    while (scanf("%f %d %d %d", &kh, &H, &spp, &batch) == 4) {
        const hdof::TraceRule r = hdof::trace_rule(kh, H, spp, batch != 0);
        printf("%d%d\\n", (int)r.packets, (int)r.binned);
    }
}"""
    P, R = "10", "00"  # packets, rays; "11" and "01" sorted
    cases = [((0.012, 256, 16, 1), P), ((0.025, 256, 16, 1), P), ((0.05, 256, 16, 1), "11"),
             ((0.08, 256, 16, 1), "01"), ((0.012, 480, 16, 1), P), ((0.08, 480, 16, 1), "11"),
             ((0.12, 480, 16, 1), "01"), ((0.012, 1080, 16, 1), "11"), ((0.012, 1080, 4, 1), P),
             ((0.0099, 1080, 16, 1), P), ((0.2, 256, 1, 1), "01"), ((0.2, 64, 1, 1), R),
             ((0.08, 256, 16, 0), "11"), ((0.0148, 136, 4, 0), P), ((0.0241, 175, 8, 0), P),
             ((0.0231, 231, 16, 0), "11"), ((0.012, 1080, 8, 0), "11"), ((0.0099, 1080, 255, 0), P),
             ((0.0043, 2160, 16, 0), P), ((0.2, 128, 16, 0), "01"), ((0.2, 10, 1, 0), R), ((0.0, 1080, 255, 0), P)]
    got = _run(tmp_path, src, "\n".join(" ".join(map(str, c)) for c, _ in cases))
    assert got == [w for _, w in cases], [(c, w, g) for (c, w), g in zip(cases, got) if w != g]
