"""Single-precision softmax on the tensor cores (up to 128 classes, operands
split into bf16 parts) against the fp64 oracle, at the edges of its tiles:
class counts around the multiples of 16 and 64 that its MMAs are built from,
feature counts around its 64-wide K blocks and 256-wide feature units, row
counts around its 64-, 128- and 256-row blocks.

Tolerance: products of parts are exact in the MMA; a leading sum is cut off
after each of the 8 K steps (16 products each) of an accumulator, at most
2^-23 of the sum so far, and the 128-product chunks are added in fp32, as the
CUDA-core kernels add single products.  So a logit is off by less than about
1e-6 of sum |w x|, and with |g| a few times smaller than the mean |r x| its
relative error stays below 1e-5 (2e-7 measured)."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import (CUDA_CORE_LAUNCHES, SPLIT_LAUNCHES, compare_runs, generate, gradient_launches, make_gpu, rel_err,
                    run_gpu, run_oracle)

pytestmark = pytest.mark.gpu

TOL = 1e-5
BASE = W.WORKLOADS["cr_n128_softmax_k1000"].replace(n=4, s=1, lr=0.1)

SHAPES = [
    # K, d, rows per partition
    (2, 1, (1, 2, 63, 64)),
    (16, 64, (65, 128, 129, 30)),
    (17, 65, (255, 256, 257, 1)),
    (33, 320, (400, 64, 127, 513)),
    (64, 256, (130, 129, 1, 64)),
    (65, 257, (90, 300, 3, 128)),
    (81, 130, (700, 700, 650, 701)),
    (112, 600, (128, 256, 200, 31)),
    (128, 1000, (257, 100, 64, 1)),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,d,m", SHAPES)
def test_split_softmax_edges(libpgc, cuda, monkeypatch, dtype, K, d, m):
    monkeypatch.setenv("PGC_NO_SMALLK", "1")     # bf16 with K <= 16 too
    monkeypatch.setenv("PGC_NO_TC", "1")         # and K = 128
    w = BASE.replace(dtype=dtype, K=K, d=d, m=m)
    Xs, ys, masks = generate(w, 4)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks)
    assert g.gradient_path == "softmax_cc"
    ora = run_oracle(w, Xs, ys, masks)
    compare_runs(w, recs, ora)
    for a, b in zip(recs, ora):
        assert rel_err(a["grad"], b["grad"]) < TOL
    assert gradient_launches(libpgc, g, masks[0]) == SPLIT_LAUNCHES
    g.close()


@pytest.mark.parametrize("scheme,mode,n,s", [("FR", "pgc", 6, 2), ("FR", "gc", 4, 1), ("CR", "is_sgd", 5, 2), ("CR", "pgc", 3, 2)])
def test_split_softmax_schemes(libpgc, cuda, scheme, mode, n, s):
    """Every destination rule of the new gradients, with partials (700 rows
    split over several units) and without (200 rows)."""
    for rows in (700, 200):
        w = BASE.replace(scheme=scheme, n=n, s=s, dtype="f32", K=20, d=200, m=rows)
        Xs, ys, masks = generate(w, 5)
        g, recs = run_gpu(libpgc, w, Xs, ys, masks, mode=mode)
        ora = run_oracle(w, Xs, ys, masks, mode=mode)
        for a, b in zip(recs, ora):
            assert rel_err(a["grad"], b["grad"]) < TOL
        assert gradient_launches(libpgc, g, masks[0]) == SPLIT_LAUNCHES
        g.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_rows_past_a_partition_do_not_reach_it(libpgc, cuda, dtype):
    """The last tile of a partition reads past its rows; what the next
    partition holds there (here infinities and NaN) must not enter its sums."""
    w = BASE.replace(dtype=dtype, K=20, d=100, m=70)
    Xs, ys, masks = generate(w, 1)
    clean = make_gpu(libpgc, w, Xs, ys)
    clean.step(masks[0])
    bad = [X.copy() for X in Xs]
    bad[1][:5] = W.f32_to_bf16_bits(np.float32([np.inf, np.nan] * 50)) if dtype == "bf16" else [np.inf, np.nan] * 50
    g = make_gpu(libpgc, w, bad, ys)
    g.step(masks[0])
    np.testing.assert_array_equal(g.store(0, 0), clean.store(0, 0))   # worker 0, slot 0: partition 0
    assert not np.isfinite(g.store(0, 1)).any()                        # slot 1: partition 1
    g.close()
    clean.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_set_weights_and_restore_refresh_the_parts(libpgc, cuda, dtype):
    """Parameters set from the host, and a restored checkpoint, reach the
    split copy of W that the kernels read."""
    w = BASE.replace(dtype=dtype, K=24, d=90, m=50)
    Xs, ys, masks = generate(w, 3)
    beta = np.random.default_rng(3).standard_normal((w.K, w.d)).astype(np.float32)
    a, b = make_gpu(libpgc, w, Xs, ys), make_gpu(libpgc, w, Xs, ys)
    a.set_weights(beta)
    ga, gb = (np.zeros(w.K * w.d, np.float32) for _ in range(2))
    a.step(masks[0], ga)
    saved = a.checkpoint()
    a.step(masks[1], ga)
    b.restore(saved)
    b.step(masks[1], gb)
    np.testing.assert_array_equal(ga, gb)
    from oracle import pgc_oracle as O
    o = O.PGCOracle(O.CR, w.n, w.s, O.SOFTMAX, [W.features_as_float(X, w.dtype) for X in Xs], ys, w.lr, beta0=beta, K=w.K)
    o.step(masks[0])
    assert rel_err(ga.reshape(w.K, w.d), o.step(masks[1])["grad"]) < TOL
    a.close()
    b.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_cuda_core_softmax_matches_oracle(libpgc, cuda, monkeypatch, dtype):
    """The CUDA-core kernels (more than 128 classes in single precision, and
    runs whose memory does not hold the split residuals)."""
    monkeypatch.setenv("PGC_NO_SPLIT", "1")
    w = BASE.replace(dtype=dtype, K=20, d=100, m=(60, 1, 130, 64))
    Xs, ys, masks = generate(w, 4)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks)
    assert g.gradient_path == "softmax_cc"
    for a, b in zip(recs, run_oracle(w, Xs, ys, masks)):
        assert rel_err(a["grad"], b["grad"]) < TOL
    assert gradient_launches(libpgc, g, masks[0]) == CUDA_CORE_LAUNCHES
    g.close()


@pytest.mark.parametrize("d,m,path", [(64, 2000, "softmax_cc"), (64, 40, "softmax_rows"), (300, 4000, "softmax_cc"),
                                      (300, 100, "softmax_rows"), (1100, 300, "softmax_rows")])
@pytest.mark.parametrize("mode", ["pgc", "naive_cr"])
def test_few_classes_take_the_faster_path(libpgc, cuda, d, m, path, mode):
    """bf16 with up to 16 classes: whole rows, or split operands where rows are
    short and many; both against the oracle (whole rows round W and R to bf16)."""
    w = W.WORKLOADS["fr_n32_softmax_k10"].replace(scheme="CR", n=6, s=2, m=m, d=d)
    if mode == "pgc":
        Xs, ys, masks = generate(w, 4)
        g, recs = run_gpu(libpgc, w, Xs, ys, masks)
        compare_runs(w, recs, run_oracle(w, Xs, ys, masks))
    else:
        from test_gpu_naive_cr import run_and_compare
        run_and_compare(libpgc, w, 5)                # steps, so that later ones read the parts the weighted decode wrote
        g = make_gpu(libpgc, w, *generate(w, 1)[:2], mode=mode)
        g.set_gc_encoding(W.make_gc_draws(w, 5))
        masks = W.make_masks(w, 1, 7)
    assert g.gradient_path == path
    assert gradient_launches(libpgc, g, masks[0]) == (SPLIT_LAUNCHES if path == "softmax_cc" else 1)
    g.close()


@pytest.mark.parametrize("dtype,K", [("f32", 10), ("bf16", 40)])
@pytest.mark.parametrize("m", [100, 900])
@pytest.mark.parametrize("mode", ["naive_cr", "gc"])
def test_split_softmax_with_the_weighted_decode(libpgc, cuda, dtype, K, m, mode):
    """GC-CR's decode writes beta's parts anew each step; rows in one unit per
    partition (100) and in several with partials (900)."""
    from test_gpu_naive_cr import run_and_compare
    w = BASE.replace(scheme="CR", n=6, s=2, dtype=dtype, K=K, d=150, m=m, lr=0.02)
    worst, _ = run_and_compare(libpgc, w, 5, mode=mode)
    assert worst < TOL                               # relative to the decode's own scale, sum |alpha| max |store|
