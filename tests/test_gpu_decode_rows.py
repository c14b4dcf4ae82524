"""The standalone decode at the parameter counts where it changes the thread
rows a column's terms are split over (8, 4, 2; 152 SMs: 38,912 and 77,824 float4
columns) and where one thread takes a column (2^18), on both sides, with the
commit in the same launch (700 rows: several partials per partition) and without
(40 rows), against the fp64 oracle.

Tolerance: the gradients meet 1e-5 of their norm (single-precision softmax
kernels); the decode adds at most n + c + s c <= 30 fp32 terms to each, below
2e-6 of the sum of their magnitudes."""

import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import SPLIT_LAUNCHES, compare_runs, generate, gradient_launches, rel_err, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = 1.2e-5
BASE = W.WORKLOADS["cr_n128_softmax_k1000"].replace(dtype="bf16", lr=0.1)

SIZES = [(100, 1556), (100, 1560), (120, 2592), (120, 2600), (128, 8184), (128, 8200)]


@pytest.mark.parametrize("rows", [40, 700])
@pytest.mark.parametrize("K,d", SIZES)
def test_decode_thread_rows(libpgc, cuda, monkeypatch, K, d, rows):
    monkeypatch.setenv("PGC_NO_TC", "1")         # K = 128 too
    for scheme, n, s in (("CR", 5, 2), ("FR", 4, 1)):
        w = BASE.replace(scheme=scheme, n=n, s=s, K=K, d=d, m=rows)
        Xs, ys, masks = generate(w, 4)
        g, recs = run_gpu(libpgc, w, Xs, ys, masks)
        ora = run_oracle(w, Xs, ys, masks)
        compare_runs(w, recs, ora)
        for a, b in zip(recs, ora):
            assert rel_err(a["grad"], b["grad"]) < TOL
        assert gradient_launches(libpgc, g, masks[0]) == SPLIT_LAUNCHES
        g.close()
