"""The integer square root of I-LayerNorm (csrc/isqrt.cuh) compiled for the host and run over every radicand of its range, and the
promise that it is part of: no floating point on the device."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_01405_b200", "csrc")

SOURCE = r"""
#include <cstdio>
#include "isqrt.cuh"

int main() {
  unsigned r = 0;
  for (unsigned n = 0; n < (1u << 26); ++n) {
    if ((r + 1) * (r + 1) <= n) ++r;
    if (ivit::isqrt26(n) != r) { std::printf("%u: %u, not %u\n", n, ivit::isqrt26(n), r); return 1; }
  }
  return 0;
}
"""


def test_every_radicand(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover", "-I", CSRC, str(tmp_path / "t.cpp"),
                    "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_no_floating_point_in_device_code():
    """No floating-point type, PTX suffix or root in the kernel sources (host code counts work in doubles and hands out
    milliseconds as float: host.cu and probe.cu)."""
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
        if name in ("host.cu", "probe.cu"):
            text = re.sub(r"\bfloat\s*\*?\s*ms\b", "", text)
        bad = re.search(r"\bfloat\d?\b|__half|bfloat|\.b?f(16|32|64)\b|\br?sqrtf?\s*\(|__f[a-z]+_r[nzud]", text)
        assert not bad, f"{name}: {bad.group(0)}"
