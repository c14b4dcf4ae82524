"""The streaming gradient kernel at row lengths around every change of its
variants (lanes per row, warps per row, chunks per lane) and at row counts
around its batches and stages, against the fp64 oracle.

Tolerance: every sum is fp32 with at most d (rows: m) terms per lane group and
fixed-order combinations, so a gradient is off by a few hundred ulps of
mean |r x| at most; 2e-5 of the largest entry leaves that ten times over."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import generate, make_gpu, rel_err, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = 2e-5
BASE = W.WORKLOADS["cr_n8_logistic_d1024"].replace(n=3, s=1, lr=0.01)

D32 = [1, 4, 5, 31, 32, 33, 63, 65, 129, 255, 257, 385, 511, 513, 700, 770, 1025, 1500, 1540, 2047, 2049, 3001, 4097, 5121,
       6145, 7200, 8193, 10300, 12289, 14337, 16383]
D16 = [1, 8, 9, 64, 65, 130, 257, 513, 769, 1000, 1025, 1600, 2000, 2049, 3100, 4097, 6145, 8193, 10241, 12289, 16000, 20481]


@pytest.mark.parametrize("dtype,d", [("f32", d) for d in D32] + [("bf16", d) for d in D16])
def test_row_lengths(libpgc, cuda, dtype, d):
    w = BASE.replace(dtype=dtype, d=d, m=(70, 1, 37), loss="lsq" if d % 2 else "logistic")
    w = w.replace(lr=0.01 / (1.0 + d / 36.0))
    Xs, ys, masks = generate(w, 4)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks)
    for a, b in zip(recs, run_oracle(w, Xs, ys, masks)):
        assert rel_err(a["grad"], b["grad"]) < TOL
        assert a["loss"] == pytest.approx(b["loss"], rel=1e-5)
    g.close()


@pytest.mark.parametrize("d", [60, 600, 1900, 3001])
@pytest.mark.parametrize("m", [(600, 599, 1), (2049, 33, 1024), (5000, 4999, 7)])
def test_row_counts(libpgc, cuda, d, m):
    w = BASE.replace(d=d, m=m)
    Xs, ys, masks = generate(w, 3)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks)
    for a, b in zip(recs, run_oracle(w, Xs, ys, masks)):
        assert rel_err(a["grad"], b["grad"]) < TOL
    g.close()


@pytest.mark.parametrize("dtype,d", [("f32", 70), ("f32", 1100), ("f32", 3001), ("bf16", 70), ("bf16", 2100)])
def test_rows_next_to_a_row_do_not_reach_it(libpgc, cuda, dtype, d):
    """Rows lie back to back: a partition beside one full of infinities and NaN
    keeps its gradient, and a row's unused lanes read nothing of the next row."""
    w = BASE.replace(dtype=dtype, d=d, m=(33, 40, 20))
    Xs, ys, masks = generate(w, 1)
    clean = make_gpu(libpgc, w, Xs, ys)
    clean.step(masks[0])
    bad = [X.copy() for X in Xs]
    junk = np.resize(np.float32([np.inf, np.nan]), bad[1].shape)
    bad[1][:] = W.f32_to_bf16_bits(junk) if dtype == "bf16" else junk
    g = make_gpu(libpgc, w, bad, ys)
    g.step(masks[0])
    np.testing.assert_array_equal(g.store(0, 0), clean.store(0, 0))   # worker 0, slot 0: partition 0
    assert not np.isfinite(g.store(0, 1)).any()                        # slot 1: partition 1
    g.close()
    clean.close()
