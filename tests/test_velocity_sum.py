"""The velocity combination of the mixed path (csrc/velsum.cuh) on the host. It
stands for a sum of double-precision products rounded to a float at the end, and
its error against the exact sum is never larger than that one's: also where terms
cancel, and where the sum lies next to the middle between two floats. Beyond half
a unit it is off by at most 2^-69 of the terms (three floats of 24 bits)."""
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "velsum.cuh"
#include <stdio.h>
#include <string.h>
int main() {
  int nc;
  while (scanf("%d", &nc) == 1) {
    reg::FloatSum<float> s, q;
    bool one = true;
    for (int l = 0; l < nc; ++l) {
      double w;
      float u;
      if (scanf("%la %a", &w, &u) != 2) return 1;
      s.add<false>(l, reg::split_weight(w), u);
      q.add<true>(l, reg::split_weight(w), u);
      one = one && reg::split_weight(w).mid == 0.f;
    }
    float r;
    (one ? q : s).rounded(&r);  // as the kernel chooses
    unsigned i;
    memcpy(&i, &r, sizeof i);
    printf("%08x\n", i);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("velsum")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1408_6299_gb300", "csrc"), "-o", str(d / "velsum"), str(d / "main.cpp")],
                   check=True)
    return str(d / "velsum")


def sums(program, cases):
    text = "".join("%d %s\n" % (len(c), " ".join(f"{float(w).hex()} {float(u).hex()}" for w, u in c)) for c in cases)
    out = subprocess.run([program], input=text, capture_output=True, text=True, check=True).stdout.split()
    return [struct.unpack("<f", struct.pack("<I", int(x, 16)))[0] for x in out]


def cases(kind, nc, n_t, count, seed):
    r = np.random.default_rng(seed)
    nodes = [np.polynomial.chebyshev.chebval(2.0 * j / n_t - 1.0, np.eye(nc)) for j in range(n_t + 1)]
    out = []
    for _ in range(count):
        w = nodes[r.integers(len(nodes))]
        u = np.float32(r.standard_normal(nc) * 10.0 ** r.uniform(-4, 1, nc))
        if kind == "cancel":  # the last term takes away all but a few bits of the others
            l = int(np.argmax(np.abs(w[1:]))) + 1
            rest = sum(w[m] * float(u[m]) for m in range(nc) if m != l)
            if w[l]:
                u[l] = np.float32(-rest / w[l])
        elif kind == "middle":  # the sum next to the middle between two floats
            rest = sum(w[m] * float(u[m]) for m in range(1, nc))
            f = np.float32(r.standard_normal())
            u[0] = np.float32(float(f) + 0.5 * float(np.spacing(f)) - rest)
        out.append([(w[l], u[l]) for l in range(nc)])
    return out


@pytest.mark.parametrize("kind", ["random", "cancel", "middle"])
@pytest.mark.parametrize("nc,n_t", [(2, 16), (3, 32), (3, 12), (4, 7), (16, 100)])
def test_no_further_off_than_a_sum_of_doubles(program, kind, nc, n_t):
    cs = cases(kind, nc, n_t, 2000, nc * 1000 + n_t)
    for c, got in zip(cs, sums(program, cs)):
        terms = [Fraction(float(w)) * Fraction(float(u)) for w, u in c]
        err, doubles = abs(Fraction(got) - sum(terms)), 0.0
        for w, u in c:
            doubles += float(w) * float(u)
        assert err <= abs(Fraction(float(np.float32(doubles))) - sum(terms)), (c, got)
        assert err <= Fraction(float(np.spacing(np.abs(np.float32(got))))) / 2 + sum(abs(x) for x in terms) / 2**69, (c, got)


def test_infinities_and_nan(program):
    inf, nan = float("inf"), float("nan")
    got = sums(program, [[(1.0, inf), (0.3, 1.0)], [(1.0, 1.0), (-0.3, inf)], [(1.0, inf), (-1.0, inf)],
                         [(1.0, 1.0), (0.1, nan), (0.5, 2.0)], [(1.0, 0.0), (0.0, -1.0), (0.3, 0.0)]])
    assert got[0] == inf and got[1] == -inf and np.isnan(got[2]) and np.isnan(got[3]) and got[4] == 0.0
