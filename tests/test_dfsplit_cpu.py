"""The integer split of an FP64 value into a double word (csrc/dfsplit.h), bit for
bit against hi = (float)x, lo = (float)(x - hi) in hardware arithmetic: random
significands over all exponents, ties and their neighbours at the cut, carries into
the exponent, zeros, subnormals, infinities and NaN."""
import pathlib
import shutil
import subprocess

import pytest

ROOT = pathlib.Path(__file__).resolve().parents[1]
HDR = ROOT / "paper_2212_06635_gb300" / "csrc" / "dfsplit.h"

DRIVER = r"""
#include <cstdio>
#include "dfsplit.h"
static uint64_t s = 0x9E3779B97F4A7C15ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static int check(uint64_t b) {
    double x;
    memcpy(&x, &b, 8);
    volatile float h = (float)x;
    volatile double r = x - (double)h;
    float want[2] = {h, (float)r}, got[2];
    tmk::df_split(x, got[0], got[1]);
    const bool nan = got[0] != got[0] && want[0] != want[0] && got[1] != got[1] && want[1] != want[1];
    if (!nan && memcmp(want, got, 8)) { std::printf("FAIL %016llx\n", (unsigned long long)b); return 1; }
    return 0;
}
int main() {
    int bad = 0;
    const uint64_t low[] = {0, 1, 0x0fffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull, 0x1ffffff0ull};
    const uint64_t high[] = {0, 1, 2, 0x7ffffeull, 0x7fffffull, 0x400000ull};
    for (uint64_t e = 0; e < 2048; ++e)
        for (uint64_t sg = 0; sg < 2; ++sg) {
            for (uint64_t h : high)
                for (uint64_t l : low) bad |= check(sg << 63 | e << 52 | h << 29 | l);
            for (int k = 0; k < 2000; ++k) bad |= check(sg << 63 | e << 52 | (rnd() & 0xfffffffffffffull));
        }
    if (!bad) std::printf("OK\n");
    return bad;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_split_matches_the_arithmetic_form(tmp_path):
    src = tmp_path / "split.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "split"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", f"-I{HDR.parent}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout[:400]
