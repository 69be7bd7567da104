"""The query stage's plan (csrc/query_plan.h) compiled by the host compiler."""
import ctypes
import functools
import os
import subprocess
import tempfile

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")
CODE = r"""
#include "query_plan.h"
extern "C" int plan(int d, int nkv, int lin, int fc, int slices, int gen, int N, int BH, int sms, int* out) {
  AsUnits u;
  const AsLoop l{d, nkv, lin, fc, slices, gen};
  const int whole = as_plan_units(u, N, BH, sms), parts = as_plan_parts(u, l, N, BH, sms);
  const int v[] = {parts > 0 ? parts : whole, parts > 0, u.n_pairs, u.n_rounds, u.share, as_threads_per_row(u, l)};
  for (int i = 0; i < 6; ++i) out[i] = v[i];
  return parts;
}
extern "C" int deal(int n_pairs, int n_rounds, int share, int nkv, int lin, int fc, int slices, int n, int c, int* out) {
  AsPart p[2];
  const int np = as_deal_parts(n_pairs, n_rounds, share, nkv, lin, fc, slices, n, c, p);
  for (int i = 0; i < np; ++i) {
    const int v[] = {p[i].unit, p[i].k0, p[i].k1, p[i].leaves, p[i].merges, p[i].at_items, p[i].at_s, p[i].at_p, p[i].at_pf, p[i].at_tail};
    for (int j = 0; j < 10; ++j) out[10 * i + j] = v[j];
  }
  return np;
}
"""


@functools.lru_cache(None)
def _library():
    with tempfile.TemporaryDirectory() as where:
        source, library = os.path.join(where, "plan.cpp"), os.path.join(where, "plan.so")
        with open(source, "w") as f:
            f.write(CODE)
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, source, "-o", library], check=True)
        return ctypes.CDLL(library)


def plan(N, BH, rate, d, F, hidden=0, gen=False, sms=148, n_keys=None):
    """{"ctas", "parts", "pairs", "rounds", "share", "threads", "nkv"} of a layer; one softmax token in `rate`, or `n_keys` of them."""
    keys = n_keys if n_keys is not None else -(-N // rate)
    nkv, lin = -(-keys // 128), int(rate != 1)
    fc, slices = -(-F // 128), hidden // d if lin else 0
    out = (ctypes.c_int * 6)()
    _library().plan(d, nkv, lin, fc, slices, int(gen and lin), N, BH, sms, out)
    return dict(zip(("ctas", "parts", "pairs", "rounds", "share", "threads"), out), nkv=nkv)


def deal(n_pairs, n_rounds, share, nkv, lin, fc, slices, n, c):
    """The parts of CTA c of n, as (unit, k0, k1, leaves, merges, at_items, at_s, at_p, at_pf, at_tail)."""
    out = (ctypes.c_int * 20)()
    count = _library().deal(n_pairs, n_rounds, share, nkv, lin, fc, slices, n, c, out)
    return [tuple(out[10 * i:10 * i + 10]) for i in range(count)]
