"""The merge of partial softmax sums (fc_merge.cuh), compiled for the host and
checked against float64: parts in rounds of eight, parts without a key that
counts, and parts that gave up, whose row is left alone."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_17139_gb300", "csrc")

HARNESS = """
#include "fc_merge.cuh"
extern "C" int merge(const float2* ml, const float4* o, int parts, float* out) {  // one row, eight columns
  FcRowMerge<8> row;
  for (int h0 = 0; h0 < parts; h0 += 8) {
    float2 v[8];
    float4 x[8][2] = {};
    for (int q = 0; q < 8; ++q) {
      v[q] = make_float2(-INFINITY, 0.f);
      if (h0 + q >= parts) continue;
      v[q] = ml[h0 + q];
      x[q][0] = o[2 * (h0 + q)], x[q][1] = o[2 * (h0 + q) + 1];
    }
    row.round(v, x, parts - h0, h0 == 0);
  }
  if (!row.whole) return 0;
  for (int u = 0; u < 8; ++u) out[u] = row.acc[u] / row.l;
  return 1;
}
extern "C" void no_part(float2* ml) { *ml = FC_NO_PART; }
"""


@pytest.fixture(scope="module")
def merge(tmp_path_factory):
    from paper_2502_17139_gb300 import build
    d = tmp_path_factory.mktemp("merge")
    (d / "m.cpp").write_text(HARNESS)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", cuda, str(d / "m.cpp"), "-o", str(d / "m.so")],
                   check=True)
    lib = C.CDLL(str(d / "m.so"))

    def call(ml, o):
        out = np.full(8, 7.0, np.float32)
        ok = lib.merge(ml.ctypes.data_as(C.c_void_p), o.ctypes.data_as(C.c_void_p), len(ml), out.ctypes.data_as(C.c_void_p))
        return ok, out

    call.lib = lib
    return call


def parts(n, dead, seed=0):
    rng = np.random.default_rng([n, seed])
    ml = np.stack([rng.normal(0, 8, n), rng.uniform(0.5, 200, n)], 1).astype(np.float32)
    o = (rng.normal(0, 1, (n, 8)) * ml[:, 1:]).astype(np.float32)
    for t in dead:
        ml[t] = -np.inf, 0.0
        o[t] = 0.0
    return ml, o


@pytest.mark.parametrize("n", [2, 7, 8, 9, 16, 17, 19])
@pytest.mark.parametrize("dead", ["none", "seven", "eight", "all_but_last", "later_round"])
def test_merge_against_float64(merge, n, dead):
    at = {"none": [], "seven": range(7), "eight": range(8), "all_but_last": range(n - 1), "later_round": range(8, 16)}[dead]
    ml, o = parts(n, [t for t in at if t < n - 1])
    ok, out = merge(ml, o)
    w = np.exp2(ml[:, 0].astype(np.float64) - ml[:, 0].max())
    ref = (o.astype(np.float64) * w[:, None]).sum(0) / (ml[:, 1] * w).sum()
    # n products, sums and weights in 32 bits: (n + 4) roundings of terms whose absolute sum is the first factor
    bound = (np.abs(o) * w[:, None]).sum(0) / (ml[:, 1] * w).sum() * (n + 4) * 2.0 ** -22
    assert ok and (np.abs(out - ref) <= bound).all()


@pytest.mark.parametrize("n,lost", [(2, 0), (2, 1), (9, 3), (17, 8), (17, 16)])
def test_row_of_a_lost_part_is_left_alone(merge, n, lost):
    ml, o = parts(n, [])
    merge.lib.no_part(ml[lost].ctypes.data_as(C.c_void_p))
    o[lost] = np.nan  # its slot holds whatever the workspace held
    ok, out = merge(ml, o)
    assert not ok and (out == 7.0).all()
