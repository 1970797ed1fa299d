"""The word by which the two threads of a row in the audit's epilogue exchange their best
values (csrc/twk_bound.cuh), on the CPU: whatever word of the last or next seven segments a
reader sees, and nothing orders it with the writer, it gets a lower bound on what was
published in its own segment, or none.  The word is one 32-bit object, so no state in between
can be seen; as separate value and stamp words every mixture of two publications could."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2608_27128_gb300 import build as B   # noqa: E402

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "twk_bound.cuh"
using namespace twk;
static uint32_t bits(float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; }
static float val(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
int main()
{
    const float v[] = {1e-45f, 3e-39f, 1.17549435e-38f, 9.7e-4f, 1.0f, 1.0009765625f, 1.5f,
                       1.99999988f, 2.0009765625f, 3.4e38f, val(0x7F800000u)};
    static_assert(sizeof(bound_word(0u, 0u)) == 4, "one 32-bit word");
    for (uint32_t s = 0; s < 200; ++s)
        for (int far = -7; far <= 7; ++far) {
            const uint32_t owner = s + far + 7, reader = s + 7;   // stamps of both threads
            if (bound_bits(bound_word(kNoBound, owner), reader) != kNoBound) return 1;
            for (float x : v) {
                const float got = val(bound_bits(bound_word(bits(x), owner), reader));
                if (far != 0 && got != val(kNoBound)) return 2;   // another segment's value
                if (far == 0 && !(got <= x)) return 3;            // not a lower bound
                if (far == 0 && x > 1e-30f && x < 1e38f && got < x * (1.f - 8e-6f)) return 4;
            }
        }
    std::puts("ok");
    return 0;
}
"""


def test_bound_word(tmp_path):
    src, exe = tmp_path / "bound.cu", tmp_path / "bound"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.returncode
