"""The TMA step kernel's compile-time layout under its build options (compiled
here, not run): what its pipeline and its stores take for granted."""

import os
import subprocess

import pytest

from paper_2502_20049_gb300 import build as B


def compiles(tmp_path, defines, asserts):
    """nvcc's front end and ptxas on a translation unit of static assertions; its messages if they fail."""
    src = tmp_path / "layout.cu"
    src.write_text('#include "psm_internal.h"\n#include "psm_kernels.cuh"\nusing namespace psm;\n' + asserts)
    cmd = [B.nvcc()] + B.ARCH + ["-std=c++17", "-I", B.CSRC] + [f"-D{d}" for d in defines] + \
        ["-c", str(src), "-o", os.devnull]
    r = subprocess.run(cmd, capture_output=True, text=True)
    return r.stderr if r.returncode else ""


KINDS = [(s, q, m, f) for s in ("__half", "__nv_bfloat16", "float", "double") for q in (19, 27) for m in (0, 1, 2)
         for f in (0, 2) if not (f == 2 and q == 27)]


def test_tensor_stores_come_with_one_cell_per_thread(tmp_path):
    """PSM_TMA_STORE: the AA even step's warps write boxes of 32 neighbouring
    cells, so no storage or operator may give their threads two cells there."""
    asserts = "".join(
        f"static_assert(TmaLayout<{s}, {q}, {m}, {f}>::STORE_TMA == ({m} == MODE_AA_EVEN));\n"
        f"static_assert(!TmaLayout<{s}, {q}, {m}, {f}>::STORE_TMA || (!tile_pairs<{s}, {f}, {m}>() && "
        f"TmaLayout<{s}, {q}, {m}, {f}>::CPT == 1));\n" for s, q, m, f in KINDS)
    assert compiles(tmp_path, ["PSM_TMA_STORE=1", "PSM_TMA_CPT16=1"], asserts) == ""


@pytest.mark.parametrize("defines", [[], ["PSM_TMA_MAX_STAGES=2"], ["PSM_TMA_MAX_STAGES=4"], ["PSM_TMA_MAX_STAGES=5"],
                                     ["PSM_TMA_MAX_STAGES=7", "PSM_TMA_REFILL_LAG=1"], ["PSM_TMA_REFILL_LAG=3"]])
def test_a_stage_belongs_to_one_group_of_warps(tmp_path, defines):
    """Where two groups of warps take alternate tiles, tiles k and k + stages
    share a stage and must fall to one group, and so must a tile and the one at
    whose reading its stage is refilled: both counts even, whatever the limits."""
    asserts = "template <class L, bool P> constexpr bool ok() {\n" \
              "  return L::NST >= 2 && L::LAG >= 0 && L::LAG < L::NST && (!P || (L::NST % 2 == 0 && L::LAG % 2 == 0));\n}\n"
    asserts += "".join(f"static_assert(ok<TmaLayout<{s}, {q}, {m}, {f}>, tile_pairs<{s}, {f}, {m}>()>());\n"
                       for s, q, m, f in KINDS)
    assert compiles(tmp_path, defines, asserts) == ""
