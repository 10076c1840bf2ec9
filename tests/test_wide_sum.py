"""The three-word FP32 sum of the weight gradient's reduction (csrc/wide_sum.cuh), compiled for the host: on sums whose
terms cancel it is no further from the exact value than the FP64 chain it stands for, up to the final rounding to FP64."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_01216_gb300", "csrc")
MAIN = """
#include <cstdio>
#include <cstring>
#include "wide_sum.cuh"
int main() {   // records: a count, then that many floats; out: the value and whether the words are finite
  int n;
  while (fread(&n, 4, 1, stdin) == 1) {
    fr3d::WideSum s;
    for (int i = 0; i < n; ++i) { float x; if (fread(&x, 4, 1, stdin) != 1) return 1; s.add(x); }
    printf("%a %d\\n", s.value(), (int)s.finite());
  }
}
"""


@pytest.fixture(scope="module")
def summed(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("wide")
    (d / "m.cc").write_text(MAIN)
    subprocess.run([cxx, "-O2", "-x", "c++", "-I", CSRC, str(d / "m.cc"), "-o", str(d / "m")], check=True)

    def run(seqs):
        data = b"".join(np.int32(len(s)).tobytes() + np.asarray(s, np.float32).tobytes() for s in seqs)
        out = subprocess.run([str(d / "m")], input=data, capture_output=True, check=True).stdout.decode().split()
        return [(float.fromhex(v), f == "1") for v, f in zip(out[::2], out[1::2])]
    return run


def fp64_chain(s):
    t = 0.0
    for x in s:
        t += float(x)
    return t


def test_no_further_off_than_an_fp64_chain(summed):
    rng = np.random.default_rng(7)
    seqs = [rng.standard_normal(n).astype(np.float32) for n in (1, 2, 33, 1040)]
    for scale in (12, 24, 36):      # terms over many binades, in any order
        seqs.append((rng.standard_normal(700) * 2.0 ** rng.integers(-scale, scale, 700)).astype(np.float32))
    for big in (2.0 ** 20, 2.0 ** 40, 2.0 ** 55):    # large terms that cancel: what is left was in the low words
        tail = rng.standard_normal(200).astype(np.float32)
        seqs.append(np.concatenate([[big], tail, [-big]]).astype(np.float32))
        seqs.append(np.concatenate([rng.permutation(np.concatenate([big * np.ones(40), -big * np.ones(40)])), tail]).astype(np.float32))
    for s, (got, finite) in zip(seqs, summed(seqs)):
        exact = math.fsum(float(x) for x in s)
        assert finite
        assert abs(got - exact) <= max(abs(fp64_chain(s) - exact), 2.0 ** -53 * abs(exact)), (len(s), got, exact)


def test_sums_that_leave_the_range_say_so(summed):
    big = np.float32(3e38)
    for s in ([big, big, -big], [np.inf, 1.0], [np.nan], [1.0, -np.inf, np.inf]):
        assert not summed([s])[0][1]
