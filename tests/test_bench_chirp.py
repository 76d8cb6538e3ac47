"""The roofline of bench.py for the kernels that take the contraction's place on k grids uniform in ln k:
their operation counts, the peak they are divided by, and the recomputed forward pass.  No GPU."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

PEAKS = {"hbm_gbs": 6777.3, "bf16_tflops": 1890.6, "bf16_tflops_sustained": 1739.2}


@pytest.fixture(scope="module")
def n5k():
    return bench.make_inputs(1, 0, 1)[0]


def test_counts_of_the_chirp_transforms(n5k):
    # N = 2048, 1024 k points, 15 tracers, 103 multipoles: both directions fit 2048 points; two FFTs of 5 M
    # log2 M and the products with a_n, the filter and b_q
    rows = 103 * 15
    work = bench.algorithmic_work(n5k, 1, 1)
    assert work["chirp fwd f32"][1] == rows * (10 * 2048 * 11 + 6 * (961 + 2048 + 1024))
    assert work["chirp fwd fp64"][1] == rows * (10 * 2048 * 11 + 6 * (1024 + 2048 + 1024))
    assert work["chirp adj f32"][1] == work["chirp adj fp64"][1] == rows * (10 * 2048 * 11 + 6 * (1025 + 2048 + 1024))
    assert work["basis head"][1:] == (4 * 64 * 1024 * rows, 6)
    assert work["k-quadrature f32"][1] == 103 * 1024 * (15 + 15 * 16)
    # ragged lists count the listed multipoles; two profile rows take two transforms
    assert bench.algorithmic_work(n5k, 2, 1, n_ell_useful=103)["chirp adj f32"][1] == work["chirp adj f32"][1]
    assert bench.algorithmic_work(n5k, 1, 2)["chirp adj f32"][1] == 2 * work["chirp adj f32"][1]


def test_rooflines_have_a_bound(n5k):
    flops = bench.algorithmic_work(n5k, 1, 1)["chirp fwd f32"][1]
    r = bench.roofline({"chirp fwd f32": (10, 10 * 0.02)}, n5k, 1, "bf16x9", PEAKS, "measured", 1, "n5k", 10)
    assert r["bound"] == "alu32" and r["peak"] == pytest.approx(bench.FP32_PEAK_TFLOPS)
    assert r["achieved"] == pytest.approx(flops / 0.02e-3 / 1e12)
    r = bench.roofline({"chirp fwd fp64": (10, 10 * 0.46)}, n5k, 1, "fp64", PEAKS, "measured", 1, "n5k", 10)
    assert r["bound"] == "alu" and r["peak"] == pytest.approx(bench.FP64_PEAK_TFLOPS)
    # five steps of three chunks, each contracted once more in the VJP
    for name in ("chirp fwd f32", "basis head"):
        stats = {name: (30, 30 * 0.01)}
        a = bench.roofline(stats, n5k, 1, "bf16x9", PEAKS, "measured", 1, "n5k", 5, True)
        b = bench.roofline(stats, n5k, 1, "bf16x9", PEAKS, "measured", 1, "n5k", 5, False)
        assert a["achieved"] == pytest.approx(2 * b["achieved"])
