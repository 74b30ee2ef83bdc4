"""CPU: the bench line names the kernels that run at the timed rank and precision, and the
sliced FP64 products are held against the MMA rate, not the FP64 pipe."""
import glob
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

PEAKS = {"f64": 1.1, "f32": 80.0, "bf16": 1900.0, "tf32": 900.0}


def test_named_kernels_are_in_the_sources():
    text = "".join(open(p).read() for p in glob.glob(
        os.path.join(ROOT, "paper_2311_00921_gb300", "csrc", "*.cu")))
    for prec in ("f64", "f32"):
        for rank in (8, 16, 17, 32, 33, 64, 128, 129):
            for kind in bench.KERNEL_SOURCES:
                for name in bench.kernels_of(kind, prec, rank):
                    assert re.search(rf"\b{name}\(", text), name


@pytest.mark.parametrize("dominant,rank,kernel,peak", [
    ("gemm_skinny.f64", 128, "fx_gemm_kernel, fx_skinny_kernel", 1900.0 / 36),
    ("gemm.f64", 8, "fx_gemm_kernel", 1900.0 / 36),
    ("ql.f64", 17, "ql_panel_kernel", 1.1), ("ql.f64", 16, "ql_basis_kernel", 1.1),
    ("pchol.f64", 8, "chol64_kernel", 1.1), ("trsv_fwd.f64", 16, "trsv_fwd_kernel", 1.1),
    ("trsv_fwd.f32", 128, "narrow32_kernel", 80.0), ("trsv_fwd.f32", 32, "trsv_fwd_kernel", 80.0),
    ("ql.f32", 128, "ql_basis_kernel, ql_panel_kernel", 80.0), ("pair_gemm.f32", 128, "df_gemm_kernel",
                                                               80.0 / bench.PAIR_OPS_PER_FLOP)])
def test_roofline_follows_rank_and_precision(dominant, rank, kernel, peak):
    r = bench.roofline_of({dominant: (5.0, 10, 24.1e9), "other.f64": (0.1, 1, 0.0)}, PEAKS, 1,
                          rank=rank)
    assert r["kernel"].rsplit(" (", 1)[0] == kernel
    assert r["peak"] == pytest.approx(peak) and r["frac"] == pytest.approx(r["achieved"] / peak)
    assert r["peak_source"]
