"""Streaming runs that evaluate more partitions than the GPU has SMs: every
partition takes part in every step that the schedule gives it, whatever the
row length (rows of 16 KB and more are split over the SMs by another rule
where there are fewer partitions).

Tolerance: as for the row lengths, sums of fp32 products in a fixed order;
2e-5 of the largest entry is ten times what they are off."""

import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import compare_runs, generate, rel_err, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

TOL = 2e-5
BASE = W.WORKLOADS["cr_n64_lsq_d16384"].replace(lr=1e-3)

CASES = [
    # mode, scheme, n, s, dtype, d, rows (n = 160: the warm-up and gradient coding evaluate all, a steady FR step 80)
    ("pgc", "CR", 160, 1, "f32", 4096, 8),
    ("pgc", "CR", 200, 1, "f32", 4093, tuple(1 + k % 3 for k in range(200))),
    ("pgc", "CR", 320, 0, "f32", 16384, 1),
    ("is_sgd", "CR", 200, 3, "f32", 8192, 5),
    ("pgc", "FR", 160, 1, "f32", 4096, 4),
    ("gc", "FR", 160, 1, "f32", 5000, tuple(1 + 7 * (k % 5) for k in range(160))),
    ("pgc", "CR", 200, 1, "bf16", 8192, 3),
    ("pgc", "CR", 700, 1, "f32", 100, 2),
]


@pytest.mark.parametrize("mode,scheme,n,s,dtype,d,m", CASES)
def test_more_partitions_than_sms(libpgc, cuda, mode, scheme, n, s, dtype, d, m):
    w = BASE.replace(scheme=scheme, n=n, s=s, dtype=dtype, d=d, m=m)
    Xs, ys, masks = generate(w, 4)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks, mode=mode)
    ora = run_oracle(w, Xs, ys, masks, mode=mode)
    if mode == "pgc":
        compare_runs(w, recs, ora)
    for a, b in zip(recs, ora):
        assert rel_err(a["grad"], b["grad"]) < TOL
        assert rel_err(a["beta"], b["beta"]) < TOL
    assert all((g.store(i, 0) != 0).any() for i in range(n))
    g.close()


@pytest.mark.parametrize("per_sm", ["1", "3"])
@pytest.mark.parametrize("n,s,dtype,d,m", [(200, 1, "f32", 4096, 7), (3, 1, "f32", 600, (2049, 33, 1024)), (5, 1, "bf16", 1000, 700)])
def test_items_handed_out_dynamically(libpgc, cuda, monkeypatch, per_sm, n, s, dtype, d, m):
    """PGC_ITEMS_PER_SM: the CTAs take items of one length as they get free."""
    monkeypatch.setenv("PGC_ITEMS_PER_SM", per_sm)
    w = BASE.replace(n=n, s=s, dtype=dtype, d=d, m=m)
    Xs, ys, masks = generate(w, 4)
    g, recs = run_gpu(libpgc, w, Xs, ys, masks)
    for a, b in zip(recs, run_oracle(w, Xs, ys, masks)):
        assert rel_err(a["grad"], b["grad"]) < TOL
    g.close()
