"""Infinities and NaN in x on the CUDA-core family, whichever kernel runs the batch: they reach
only the outputs whose row keeps the column.  Integer-valued weights and the other x make every
finite sum exact, so finite results must match bit for bit."""
import numpy as np
import pytest

from paper_2405_03594_gb300 import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

BAD = [np.inf, -np.inf, np.nan]


def _expected(x, w, mask):
    """x . (w o mask)^T over kept columns only, each product and sum as IEEE has it."""
    fin = np.isfinite(x)
    y = np.where(fin, x, 0.0) @ np.where(mask, w, 0.0).T
    with np.errstate(invalid="ignore"):
        for m, k in zip(*np.nonzero(~fin)):
            keep = mask[:, k] != 0
            y[m, keep] += w[keep, k] * x[m, k]
    return y


# a CTA per row block, clusters that push and that read their sums, many and few chunks
@pytest.mark.parametrize("N,K", [(130, 72), (1003, 1096), (40000, 64), (64, 11008), (4096, 6400), (22016, 1152)])
@pytest.mark.parametrize("int8,M", [(False, 1), (False, 2), (False, 3), (False, 8), (False, 9), (False, 10),
                                    (True, 1), (True, 2), (True, 5), (True, 13)])
def test_dropped_columns_take_no_part(N, K, int8, M):
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N + K + M)
    mask = (g.random((N, K)) < 0.4).astype(np.uint8)
    x = g.integers(-2, 3, size=(M, K)).astype(np.float64)
    for i in range(max(1, M // 2)):  # tokens 0, 2, 4, ...: one to three values each, the last column too
        cols = np.append(g.choice(K - 1, i % 3, replace=False), K - 1)
        x[2 * i % M, cols] = g.choice(BAD, len(cols))
    with np.errstate(invalid="ignore"):
        xb = synth.bf16_from_f32(x.astype(np.float32))
    if int8:
        w = g.integers(-128, 128, size=(N, K))
        s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
        h = sp.compress(gu.i8_to_dev(w.astype(np.int8)), gu.u8_to_dev(mask), gu.f32_to_dev(s))
        want = _expected(x, w.astype(np.float64), mask) * s
    else:
        w = g.integers(-4, 5, size=(N, K)).astype(np.float32)
        h = sp.compress(gu.bf16_to_dev(synth.bf16_from_f32(w)), gu.u8_to_dev(mask))
        want = _expected(x, w.astype(np.float64), mask)
    assert np.isfinite(want).any() and not np.isfinite(want).all()
    xd = gu.bf16_to_dev(xb)
    y = h.linear(xd)
    sp.check()
    got = gu.bf16_from_dev(y)
    fin = np.isfinite(want)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    assert np.array_equal(gu.bf16_bits_from_dev(y)[fin], synth.bf16_from_f32(want[fin].astype(np.float32)))
    # an epilogue takes the same sums
    h0 = torch.zeros_like(y)
    assert h.linear_epi(xd, h0, "residual", torch.zeros(N, dtype=torch.bfloat16, device=y.device))
    sp.check()
    res = gu.bf16_from_dev(h0)
    assert np.array_equal(np.isnan(res), np.isnan(want)) and np.array_equal(res[~np.isnan(want)], got[~np.isnan(want)])
