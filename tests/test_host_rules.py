"""Layouts and launch rules that the host code fixes, checked without a GPU by
compiling small programs against the kernel headers."""
import os
import subprocess

from paper_2609_02876_gb300 import build as B


def run(tmp_path, body):
    src, exe = tmp_path / "t.cu", str(tmp_path / "t")
    src.write_text(body)
    r = subprocess.run([B.nvcc()] + B.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I",
                                              os.path.join(B.ROOT, "include"), str(src), "-o", exe],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return subprocess.run([exe], capture_output=True, text=True, timeout=600)


def test_nrob_stage_data_is_aligned_for_its_vector_accesses(tmp_path):
    """A local copy of the group form's stage data is read and written 16 bytes
    at a time, as is its place in a segment and in a side block."""
    r = run(tmp_path, r"""
#include "gs_internal.h"
#include "gs_nrob.cuh"
using G = gs::NeuralRobertsonGroup;
static_assert(alignof(G::Data) % 16 == 0 && sizeof(G::Data) % 16 == 0, "local copies");
static_assert((3 + G::D) % 2 == 0 && G::ACT % 2 == 0 && gs::NRG_STAGE_DOUBLES % 2 == 0, "segments and side blocks");
static_assert(G::ACT + sizeof(G::Data) / 8 == gs::NRG_STAGE_DOUBLES, "payload");
struct Holder { double x; G::Data d; };
int main() { Holder h[3]; for (auto& v : h) if (reinterpret_cast<size_t>(&v.d) % 16) return 1; return 0; }
""")
    assert r.returncode == 0


def test_stiff_records_run_in_the_fewest_rounds(tmp_path):
    """ctas_by_rounds against its definition by counting: c CTAs per SM take the
    ensemble round by round, a round costing c; the cheaper of the two, lo on a tie."""
    r = run(tmp_path, r"""
#include "gs_internal.h"
static long long cost(long long lanes, long long wave, int c) {
  long long t = 0;
  for (; lanes > 0; lanes -= c * wave) t += c;
  return t;
}
int main() {
  const int pairs[][2] = {{2, 3}, {4, 5}};
  for (long long wave : {1ll, 128ll, 19456ll})
    for (auto& p : pairs)
      for (long long w = 0; w < 64; ++w)
        for (long long d : {-1ll, 0ll, 1ll}) {
          const long long n = w * wave + d;
          if (n < 1) continue;
          const int want = cost(n, wave, p[1]) < cost(n, wave, p[0]) ? p[1] : p[0];
          if (gs::ctas_by_rounds(n, wave, p[0], p[1]) != want) return 1;
        }
  // Robertson on 152 SMs, where a rule for some of the waves only was the slower choice
  const auto c = [](long long n) { return gs::ctas_by_rounds(n, 19456, 2, 3); };
  return !(c(66000) == 2 && c(78000) == 2 && c(140000) == 2 && c(160000) == 3 && c(58368) == 3 && c(58369) == 2);
}
""")
    assert r.returncode == 0
