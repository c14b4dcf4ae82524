"""Outputs of a step in every layout the decode writes them in: rows without
padding, one class whose array ends inside a 16-byte column, padded rows, with
aligned and unaligned destinations, on the device, in pinned and in pageable
host memory.  All hold what the library keeps (get_weights), bit for bit, and
nothing is written past their ends."""

import numpy as np
import pytest

from paper_2607_20739_gb300 import workloads as W

from parity import generate, make_gpu

pytestmark = pytest.mark.gpu

WL = W.WORKLOADS
CASES = {
    # K = 1: fused decode, standalone decode (6 copies of 30000 floats), GC-CR decode
    "rows_fused_d33": (WL["cr_n8_logistic_d1024"].replace(n=4, s=1, m=20, d=33), "pgc"),
    "rows_fused_bf16_d1001": (WL["cr_n8_logistic_d1024"].replace(n=4, s=1, m=20, d=1001, dtype="bf16"), "pgc"),
    "rows_decode_d14999": (WL["cr_n64_lsq_d16384"].replace(n=6, s=2, m=9, d=14999, lr=1e-4), "pgc"),
    "rows_naive_d70": (WL["cr_n8_logistic_d1024"].replace(n=5, s=1, m=20, d=70), "naive_cr"),
    # K > 1: whole-row few-class kernel (fused), split softmax, tensor cores (both decodes)
    "few_d700": (WL["fr_n32_softmax_k10"].replace(n=8, m=50, d=700), "pgc"),
    "few_d701": (WL["fr_n32_softmax_k10"].replace(n=8, m=50, d=701), "pgc"),
    "few_d768": (WL["fr_n32_softmax_k10"].replace(n=8, m=50, d=768), "pgc"),
    "split_d90": (WL["cr_n128_softmax_k1000"].replace(n=4, s=1, K=21, d=90, m=40), "pgc"),
    "tc_d301": (WL["cr_n128_softmax_k1000"].replace(n=4, s=1, K=130, d=301, m=40), "pgc"),
    "tc_wide_d4093": (WL["cr_n128_softmax_k1000"].replace(n=3, s=1, K=260, d=4093, m=30), "pgc"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_outputs(libpgc, cuda, name):
    torch = cuda
    w, mode = CASES[name]
    Xs, ys, masks = generate(w, 4)
    size, guard = w.K * w.d, 8
    g = make_gpu(libpgc, w, Xs, ys, mode=mode)
    ref = make_gpu(libpgc, w, Xs, ys, mode=mode)
    if mode == "naive_cr":
        draws = W.make_gc_draws(w, 5)
        g.set_gc_encoding(draws)
        ref.set_gc_encoding(draws)
    for t in range(4):
        want = np.zeros(size, np.float32)                    # pageable: padded copies
        ref.step(masks[t], want)
        # aligned device, device one float off, pinned host, pinned one float off
        make = (lambda n: torch.full((n,), 7.0, device="cuda")) if t < 2 else \
            (lambda n: torch.full((n,), 7.0).pin_memory())
        off = t % 2
        gb, wb = make(size + off + guard), make(size + off + guard)
        g.step(masks[t], gb[off:off + size], wb[off:off + size])
        g.sync()
        got = gb[off:off + size].cpu().numpy()
        if name.startswith("tc"):
            # two runs differ: U[o_t] is summed in the order the CTAs finish (a few
            # fp32 roundings of the largest entry)
            assert np.abs(got - want).max() <= 1e-6 * np.abs(want).max()
        else:
            np.testing.assert_array_equal(got, want)
        np.testing.assert_array_equal(wb[off:off + size].cpu().numpy(), g.weights().reshape(-1))
        for b in (gb, wb):
            assert (b[:off] == 7.0).all() and (b[off + size:] == 7.0).all()
    # one output only
    only = torch.full((size,), 7.0, device="cuda")
    g.step(masks[0], None, only)
    g.sync()
    np.testing.assert_array_equal(only.cpu().numpy(), g.weights().reshape(-1))
    g.close()
    ref.close()


@pytest.mark.parametrize("K,d,off", [(130, 2538, 0), (130, 2539, 0), (130, 2540, 1), (130, 2540, 0), (1000, 333, 0)])
def test_host_rows_around_the_size_that_copies_take(libpgc, cuda, K, d, off):
    """Pinned rows that start off 16 bytes: written by the decode up to 330,000
    floats, copied from there on."""
    torch = cuda
    w = WL["cr_n128_softmax_k1000"].replace(n=3, s=1, K=K, d=d, m=20)
    Xs, ys, masks = generate(w, 2)
    g, size = make_gpu(libpgc, w, Xs, ys), K * d
    for t in range(2):
        gb, wb = (torch.full((size + off + 8,), 7.0).pin_memory() for _ in range(2))
        before = g.weights().reshape(-1)
        g.step(masks[t], gb[off:off + size], wb[off:off + size])
        np.testing.assert_array_equal(wb[off:off + size].numpy(), g.weights().reshape(-1))
        moved = before - np.float32(w.lr) * gb[off:off + size].numpy()
        assert np.abs(moved - g.weights().reshape(-1)).max() <= 1e-6 * np.abs(moved).max()   # one rounding more than the fused update
        for b in (gb, wb):
            assert (b[:off] == 7.0).all() and (b[off + size:] == 7.0).all()
    g.close()


def test_large_unaligned_host_rows_do_not_hold_up_the_decode(libpgc, cuda):
    """Float by float over the link, three million floats took the decode
    fifteen times as long as on the device; with copies it takes the same time."""
    torch = cuda
    w = WL["cr_n128_softmax_k1000"].replace(n=3, s=1, K=1000, d=3001, m=20)
    Xs, ys, masks = generate(w, 1)
    g, ms = make_gpu(libpgc, w, Xs, ys), {}
    for where in ("device", "host"):
        make = (lambda: torch.zeros(w.K * w.d, device="cuda")) if where == "device" else \
            (lambda: torch.zeros(w.K * w.d).pin_memory())
        a, b = make(), make()
        for _ in range(4):
            g.step(masks[0], a, b)
        g.timing(True)
        for _ in range(10):
            g.step(masks[0], a, b)
        ms[where] = g.timing_read()["ms"][libpgc.KERNEL_GROUPS.index("decode")]
        g.timing(False)
    g.close()
    assert ms["host"] < 4 * ms["device"], ms
