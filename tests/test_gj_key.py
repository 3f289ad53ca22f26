"""Host check of the pivot key of the FP64 Gauss-Jordan eliminations.

gj_key_bits (paper_1504_05090_gb300/csrc/gj_key.cuh) rounds |x| to FP32 with
integer instructions.  The header also compiles as plain C++; a small program
compares it bit for bit with the conversion that k_gj_cluster compares, on
random numbers over the exponent range, ties, carries into the next power of
two and to infinity, and numbers that differ below the 20 leading bits.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1504_05090_gb300", "csrc")

PROGRAM = r"""
#include "gj_key.cuh"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
int main() {
  std::mt19937_64 rng(3);
  long long n = 0, bad = 0, unused = 0;
  auto check = [&](uint64_t b) {
    double x;
    std::memcpy(&x, &b, 8);
    const float f = static_cast<float>(std::fabs(x));
    uint32_t ref;
    std::memcpy(&ref, &f, 4);
    bool ok;
    const uint32_t k = dqmc::gj_key_bits(b, ok);
    ++n;
    if (!ok) ++unused;
    if (ok && k != ref) ++bad;
    if (!ok && std::isnormal(f) && std::fabs(x) >= 0x1p-126 && std::fabs(x) < 0x1p128) ++bad;
  };
  for (int it = 0; it < 300000; ++it) check(rng());
  for (uint64_t E = 0; E < 2048; ++E)
    for (uint64_t m : {0ull, 1ull, 0x10000000ull, 0x0FFFFFFFull, 0x10000001ull, 0x30000000ull, 0x1FFFFFFFull,
                       0xFFFFFFFFFFFFFull, 0xFFFFFF0000000ull, 0xFFFFFEFFFFFFFull, 0xFFFFF00000000ull})
      for (uint64_t s = 0; s < 2; ++s) check((s << 63) | (E << 52) | m);
  const uint64_t one = 1023ull << 52;
  for (uint64_t d = 0; d < 64; ++d) check(one + (d << 27));
  std::printf("%lld %lld %lld\n", n, bad, unused);
  return 0;
}
"""


def test_key_is_the_fp32_rounding(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "key.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "key"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    n, bad, unused = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert n > 340000 and bad == 0 and unused < n


@pytest.mark.gpu
def test_pivots_do_not_depend_on_the_matrices_in_flight():
    """A field (U = 4, beta = 5, one of 20000 random ones) whose middle matrix
    has two pivot candidates that agree to 20 bits and not to 24: the kernels
    in shared memory (8 and 4 CTAs) and on global memory take the same one, so
    G agrees bit for bit in every chain of 2, 20 and 40."""
    import numpy as np

    import paper_1504_05090_gb300 as pkg
    bits = np.unpackbits(np.load(os.path.join(HERE, "golden", "gj_pivot_field_16x16.npy")))
    field = (2 * bits.astype(np.int8) - 1).reshape(1, 20, 256)
    first = None
    for C in (2, 20, 40):
        g = pkg.Group(Lx=16, Ly=16, t=0.25, U=4.0, beta=5.0, dtau=0.25, n_chains=C, stab_interval=5,
                      delay_k=8, precision="fp64")
        with pkg.DQMC([g], seed=0) as sim:
            sim.set_field([np.repeat(field, C, axis=0)])
            for c in range(C):
                G = sim.G(c, 0)
                if first is None:
                    first = G
                assert np.array_equal(G, first), (C, c)
