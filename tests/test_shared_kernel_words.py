"""The words that the kernels with a point's tensors shared out over warps read and
write in the same array.  The last block's spare threads repeat the last point
without storing anything: they must not read the words that this point's own
threads are storing.

Words that a launch also writes are read with ordinary loads, not through the
read-only path.

The update of k_reconstruct_shared (StageUpdate) runs here on the host, compiled
from its source text against stand-ins that count every read."""

import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_3408_gb300", "csrc")

_HARNESS = r"""
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
static std::vector<const double*> reads, cached;  // all reads; those through the read-only path
static double __ldg(const double* p) { reads.push_back(p); cached.push_back(p); return *p; }
template <class T> struct S { static T c(double x) { return x; } static double to_double(T x) { return x; } };
template <class T, bool F> struct Store {
  static T ld(const double* b, long long i) { return __ldg(b + i); }
  static T ld_rw(const double* b, long long i) { reads.push_back(b + i); return b[i]; }
  static void st(double* b, long long i, T v) { b[i] = v; }
};
template <class T> constexpr bool kIn = PAIRS;
static bool finite_s(double) { return true; }
static double twice(double x) { return 2 * x; }
%s
template <int KIND> void run(bool live) {
  double dst[8] = {}, u[8], U[8] = {}, k[8], uf[8];
  for (int i = 0; i < 8; ++i) u[i] = k[i] = uf[i] = i + 1;
  StageUpdate<double, KIND> up{dst, u, U, k, uf, 4, 3, KIND == 2 ? 3 : 1, live, false, 0.5, 0.25};
  reads.clear();
  cached.clear();
  up.put(1, 10.0, up.fetch(1));
  // reads of arrays that this kind of update writes
  auto written = [&](const std::vector<const double*>& v) {
    int n = 0;
    for (const double* p : v)
      for (const double* a : {KIND == 1 ? k : u, KIND == 1 ? U : uf}) n += p >= a && p < a + 8;
    return n;
  };
  const int r = written(reads), c = written(cached);
  std::printf("%%d %%d %%g %%g %%g %%g %%g\n", c, r, dst[7], u[7], U[7], k[7], uf[7]);
}
int main() { run<0>(true); run<1>(true); run<2>(true); run<0>(false); run<1>(false); run<2>(false); }
"""


def _source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return fh.read()


def _struct(src, name):
    a = src.index("template <class T, int KIND>\nstruct " + name)
    return src[a:src.index("\n};", a) + 3]


@pytest.mark.parametrize("pairs", [0, 1])
def test_spare_threads_read_no_word_that_the_stage_update_stores(tmp_path, pairs):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src = _source("pointwise.cu")
    cpp = tmp_path / "u.cpp"
    cpp.write_text(_HARNESS % (_struct(src, "StateWords") + "\n" + _struct(src, "StageUpdate")))
    subprocess.check_call([gxx, "-std=c++17", f"-DPAIRS={pairs}", "-o", str(tmp_path / "u"), str(cpp)])
    got = [line.split() for line in subprocess.check_output([str(tmp_path / "u")], text=True).splitlines()]
    words = [[float(x) for x in row[2:]] for row in got]
    # live: filtered result; stage 2 (U = u + dt k, acc += 2 k); last stage (u += (acc + k) dt / 6)
    assert words[0] == [10, 8, 0, 8, 10 if pairs else 8]
    assert words[1] == [0, 8, 13, 28, 8] and words[2] == [0, 12.5, 0, 8, 12.5 if pairs else 8]
    # spare: nothing stored, and nothing read where the live threads store
    assert words[3:] == [[0, 8, 0, 8, 8]] * 3
    assert [int(row[1]) for row in got] == [0, 1, 1, 0, 0, 0]
    assert [int(row[0]) for row in got] == [0] * 6  # none through the read-only path


def test_spare_threads_read_no_source_word_that_is_stored():
    src = _source("rhs.cu")
    a = src.index("k_rhs_quad_shared(const double*")
    body = src[a:src.index("\n}\n", a)]
    after = body[body.index("__syncthreads();"):]
    # rows 40..49 (alpha, beta^i, gamma^ij) are only read by this kernel
    assert re.findall(r"ldA\w*<T, kInt<T>>\((\w+), P, p, ([^)]*)\)", after) == [("part_src", "s")]
    assert "part_src = live ? src : src + 40 * P;" in after


@pytest.mark.parametrize("name,kernel,words", [
    ("rhs.cu", "k_rhs_quad(const double*", r"\(src, P, p, s\)"),
    ("rhs.cu", "k_rhs_quad_shared(const double*", r"\(part_src, P, p, s\)"),
    ("nest.cu", "k_interface(const double*", r"\(S[AB], \(long long\)f \* P[AB] \+ p[ab]\)"),
])
def test_words_that_the_launch_writes_take_ordinary_loads(name, kernel, words):
    src = _source(name)
    a = src.index(kernel)
    reads = re.findall(r"(ld\w*)(?:<T, kInt<T>>)?" + words, src[a:src.index("\n}\n", a)])
    assert reads and all(r.endswith("_rw") for r in reads), reads
