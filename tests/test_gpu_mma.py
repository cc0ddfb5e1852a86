"""Batches of 2 to 32 rows on linear_mma_kernel against the float64 oracle: every token-tile
width (8, 16, 32 tokens, full and ragged), row blocks and K-tiles that end inside a tile, one
chunk per CTA up to more chunks than ring slots, dense and nearly empty rows, both value types.
Integer-valued inputs make every sum exact, so they must match bit for bit."""
import numpy as np
import pytest

from paper_2405_03594_gb300 import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SHAPES = [(1, 8), (130, 72), (128, 64), (257, 136), (1003, 1096), (64, 11008), (12288, 256), (40000, 64)]


@pytest.mark.parametrize("N,K", SHAPES)
@pytest.mark.parametrize("M", [2, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("int8", [False, True])
def test_integer_sums_bit_exact(oracle, N, K, M, int8):
    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N * K + M)
    keep = g.uniform(0.0, 1.0, size=(N, 1))  # rows from empty to dense
    mask = (g.random((N, K)) < keep).astype(np.uint8)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    if int8:
        q = g.integers(-128, 128, size=(N, K)).astype(np.int8)
        s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
        h = sp.compress(gu.i8_to_dev(q), gu.u8_to_dev(mask), gu.f32_to_dev(s))
        ref = oracle.linear_int8(x, q, mask, s)
    else:
        W = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
        h = sp.compress(gu.bf16_to_dev(W), gu.u8_to_dev(mask))
        ref = oracle.linear_bf16(x, W, mask)
    for path in ("auto", "cuda_core") if M <= 16 else ("auto",):
        assert h.kernel_name(M, path) == "linear_mma_kernel"
        y = h.linear(gu.bf16_to_dev(x), path=path)
        sp.check()
        assert np.array_equal(gu.bf16_bits_from_dev(y), synth.bf16_from_f32(ref.astype(np.float32))), path


@pytest.mark.parametrize("N,K", [(22016, 1152), (4096, 6400)])
@pytest.mark.parametrize("M", [3, 16, 32])
@pytest.mark.parametrize("least", [0.4, 1.0])
def test_large_chunks_at_lower_occupancy(oracle, N, K, M, least):
    """More than 20 chunks per SM whose size leaves fewer CTAs per SM than the kernel allows."""
    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N + M)
    mask = (g.random((N, K)) < g.uniform(least, 2 * least, size=(N, 1))).astype(np.uint8)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    W = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
    h = sp.compress(gu.bf16_to_dev(W), gu.u8_to_dev(mask))
    assert h.kernel_name(M) == "linear_mma_kernel"
    y = h.linear(gu.bf16_to_dev(x))
    sp.check()
    ref = oracle.linear_bf16(x, W, mask)
    assert np.array_equal(gu.bf16_bits_from_dev(y), synth.bf16_from_f32(ref.astype(np.float32)))


@pytest.mark.parametrize("N,K", [(22016, 1152), (4096, 6408)])
@pytest.mark.parametrize("keep", [0.30, 0.36, 0.5, 1.0])  # either side of the lines at 0.36 and 0.26
@pytest.mark.parametrize("M", [1, 2])
def test_one_and_two_rows_of_many_int8_weights(oracle, N, K, keep, M):
    """INT8 matrices that keep many weights: the products and the residual epilogue."""
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N + M)
    mask = (g.random((N, K)) < keep).astype(np.uint8)
    q = g.integers(-128, 128, size=(N, K)).astype(np.int8)
    s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    h = sp.compress(gu.i8_to_dev(q), gu.u8_to_dev(mask), gu.f32_to_dev(s))
    many = h.info.nnz >= (0.36 if M == 1 else 0.26) * N * K
    assert (h.kernel_name(M) == "linear_mma_kernel") == many
    ws = torch.zeros(max(h.workspace_size(M), 256), dtype=torch.uint8, device=gu.dev())
    y = h.linear(gu.bf16_to_dev(x), workspace=ws)
    ref = oracle.linear_int8(x, q, mask, s)
    assert np.array_equal(gu.bf16_bits_from_dev(y), synth.bf16_from_f32(ref.astype(np.float32)))
    h0 = gu.bf16_to_dev(synth.activations(M, N, g))
    r = gu.bf16_to_dev(synth.activations(1, N, g)[0])
    h1 = h0.clone()
    assert h.linear_epi(gu.bf16_to_dev(x), h1, "residual", r, workspace=ws)
    sp.residual_add(h0, y, r)
    sp.check()
    assert np.array_equal(gu.bf16_bits_from_dev(h1), gu.bf16_bits_from_dev(h0))
