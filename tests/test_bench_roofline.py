"""The benchmark's headline roofline names the kernel that ran and divides by the peak of its pipe."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

PEAKS = {"bf16_tflops": 2000.0, "bf16_tflops_sustained": 1700.0}


def _stats(exec_chi0, exec_ec, ms_chi0=350.0, ms_ec=200.0):
    return {"ms_gemm_chi0": ms_chi0, "flop_gemm_chi0": 6.4e12, "n_gemm_chi0": 480, "flop_exec_gemm_chi0": exec_chi0,
            "ms_gemm_ec": ms_ec, "flop_gemm_ec": 3.0e12, "n_gemm_ec": 144, "flop_exec_gemm_ec": exec_ec}


def test_planes():
    """FP64 on digit planes: 6.4e12 FP64 flops in 0.35 s are no 18 TFLOP/s of a 1.1 TFLOP/s pipe."""
    r = bench.roofline(_stats(2.4e14, 1.0e14), PEAKS, "measured", 1.1, "FP64", True)
    assert r["kernel"] == "k_ozgemm (chi0 GEMMs)" and r["peak"] == 2000.0 and r["traffic"] is None
    assert r["achieved"] == pytest.approx(2.4e14 / 0.35 / 1e12) and r["frac"] < 1.0


@pytest.mark.parametrize("ms_ec,kernel,flop", [(5000.0, "k_dgemm_nt", 6.4e12), (9000.0, "k_zgemm, k_dgemm_tri", 3.0e12)])
def test_pipes(ms_ec, kernel, flop):
    r = bench.roofline(_stats(0.0, 0.0, 8000.0, ms_ec), PEAKS, "measured", 1.1, "FP64", False)
    assert r["kernel"] == kernel and r["peak"] == 1.1 and r["flop"] == flop and r["peak_note"] == "FP64"


def test_each_leg_by_its_own_pipe():
    """A small cell: contraction on planes, ln det on the FP64 pipes."""
    assert bench.roofline(_stats(2.4e14, 0.0, 1.0, 2.0), PEAKS, "measured", 1.1, "FP64", False)["kernel"] == "k_zgemm, k_dgemm_tri"
    assert bench.roofline(_stats(2.4e12, 0.0, 2.0, 1.0), PEAKS, "measured", 1.1, "FP64", False)["kernel"] == "k_ozgemm (chi0 GEMMs)"
