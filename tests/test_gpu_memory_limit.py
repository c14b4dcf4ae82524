"""A run that fits the GPU's free memory only without the buffers of the
tensor-core loss (12 bytes per row and more) is created without them, takes
its steps and computes its loss the other way.

The rest of the memory is held by a tensor for the length of the test; what
the run needs without those buffers is measured first, with them switched off."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20
ROWS, D, K, N = 1_000_000, 256, 128, 4                      # 2 GB of features, 2 GB of residuals, 48 MB of row statistics


def _free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_run_that_fits_only_without_the_loss_buffers(libpgc, cuda, monkeypatch):
    torch = cuda
    torch.cuda.empty_cache()

    def make(rows=ROWS):
        return libpgc.PGC("CR", N, 1, "softmax", "bf16", D, K=K, rows=[rows] * N, lr=0.1)

    def use(g, rows):
        """Load rows that are all alike, e_0 with label 3, and check a step and both losses."""
        X = np.zeros((rows, D), np.uint16)
        X[:, 0] = W.f32_to_bf16_bits(np.float32([1.0]))[0]
        g.load([X] * N, [np.full(rows, 3, np.int32)] * N)
        assert g.loss() == pytest.approx(np.log(K), rel=1e-6)
        g.step(np.array([0, 1, 0, 0], np.uint8))
        w = g.weights()
        want = np.full(K, -0.1 / K)
        want[3] += 0.1
        np.testing.assert_allclose(w[:, 0], want, rtol=2e-2)
        p = np.exp(w[:, 0].astype(np.float64))
        assert g.loss() == pytest.approx(np.log(p.sum()) - np.log(p[3]), rel=1e-5)
        g.close()

    # what the kernels themselves need is allocated at their first use, on both ways of the loss
    use(make(100), 100)
    with monkeypatch.context() as mp:
        mp.setenv("PGC_NO_SPLIT", "1")
        use(make(100), 100)
    make().close()
    before = _free(torch)
    with monkeypatch.context() as mp:
        mp.setenv("PGC_NO_SPLIT", "1")
        g = make()
        without = before - _free(torch)
        g.close()
    g = make()
    assert g.gradient_path == "tc_fused"
    with_all = before - _free(torch)
    g.close()
    assert with_all > without + 16 * MB
    hold = torch.empty(_free(torch) - without - 10 * MB, dtype=torch.uint8, device="cuda")
    try:
        assert without < _free(torch) < with_all
        g = make()
        assert g.gradient_path == "tc_fused"
        use(g, ROWS)
    finally:
        del hold
        torch.cuda.empty_cache()
