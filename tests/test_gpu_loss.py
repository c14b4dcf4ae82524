"""pgc_loss against the fp64 oracle: softmax on the tensor cores (class blocks
of 128, row tiles of 256) and its CUDA-core form, logistic and least squares
at ragged row lengths.  A row's logits are fp32 sums of d products (relative
error below 1e-6 of sum |w x|), the rows are summed in fp64, so the mean
over the rows stays within 2e-6."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import generate, make_gpu

pytestmark = pytest.mark.gpu

SOFTMAX = W.WORKLOADS["cr_n128_softmax_k1000"].replace(n=3, s=1)
ROWS = W.WORKLOADS["cr_n8_logistic_d1024"].replace(n=3, s=1)


def check(libpgc, w):
    from oracle import pgc_oracle as O
    Xs, ys, _ = generate(w, 1)
    shape = (w.K, w.d) if w.loss == "softmax" else (w.d,)
    beta = (np.random.default_rng(7).standard_normal(shape) / np.sqrt(w.d)).astype(np.float32)
    g = make_gpu(libpgc, w, Xs, ys)
    g.set_weights(beta)
    loss = {"logistic": O.LOGISTIC, "lsq": O.LSQ, "softmax": O.SOFTMAX}[w.loss]
    want = O.full_loss(loss, [W.features_as_float(X, w.dtype).astype(np.float64) for X in Xs], ys, beta.astype(np.float64))
    for _ in range(2):
        assert g.loss() == pytest.approx(want, rel=2e-6)
    g.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,d,m", [(2, 3, (1, 254, 1)), (16, 100, (255, 1, 1)), (20, 64, (300, 7, 64)),
                                   (127, 130, (90, 90, 90)), (128, 257, (256, 256, 1)), (129, 320, (70, 200, 3)),
                                   (300, 500, (129, 400, 77)), (1000, 96, (100, 100, 101)), (2050, 64, (40, 30, 50))])
def test_softmax_loss(libpgc, cuda, dtype, K, d, m):
    check(libpgc, SOFTMAX.replace(dtype=dtype, K=K, d=d, m=m))


@pytest.mark.parametrize("K", [20, 300])
def test_softmax_loss_on_cuda_cores(libpgc, cuda, monkeypatch, K):
    monkeypatch.setenv("PGC_NO_SPLIT", "1")
    check(libpgc, SOFTMAX.replace(dtype="f32", K=K, d=100, m=(90, 1, 65)))


@pytest.mark.parametrize("loss", ["logistic", "lsq"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [1, 33, 1000, 3001, 5000])
def test_rows_loss(libpgc, cuda, loss, dtype, d):
    check(libpgc, ROWS.replace(loss=loss, dtype=dtype, d=d, m=(300, 1, 65)))


@pytest.mark.parametrize("K", [20, 300])
def test_softmax_loss_without_dependent_launches(libpgc, cuda, monkeypatch, K):
    monkeypatch.setenv("PGC_NO_PDL", "1")
    check(libpgc, SOFTMAX.replace(dtype="bf16", K=K, d=100, m=(300, 1, 65)))
