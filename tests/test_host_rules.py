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
