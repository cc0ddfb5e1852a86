"""Large batches (the matrix expanded once, then a dense product) against the float64 oracle:
one and several token tiles, a ragged last one, an odd number of row blocks (half a CTA pair's
tile empty), K-tiles that end inside a tile, fewer tiles than CTA pairs and several waves with
a split rest, y rows that TMA stores cannot address, both value types.  Integer-valued inputs
make every sum exact, so they must match bit for bit."""
import numpy as np
import pytest

from paper_2405_03594_gb300 import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _matrix(sp, N, K, int8, g):
    keep = g.uniform(0.0, 1.0, size=(N, 1))  # rows from empty to dense
    mask = (g.random((N, K)) < keep).astype(np.uint8)
    if int8:
        q = g.integers(-128, 128, size=(N, K)).astype(np.int8)
        s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
        return (q, mask, s), sp.compress(gu.i8_to_dev(q), gu.u8_to_dev(mask), gu.f32_to_dev(s))
    W = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
    return (W, mask, None), sp.compress(gu.bf16_to_dev(W), gu.u8_to_dev(mask))


@pytest.mark.parametrize("N,K,M", [(256, 512, 40), (1150, 1096, 33), (2048, 1024, 300), (1500, 2056, 513), (19520, 64, 70),
                                   (6000, 328, 2049), (128, 11008, 100)])
@pytest.mark.parametrize("int8", [False, True])
def test_integer_sums_bit_exact(oracle, N, K, M, int8):
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N * K + M)
    (v, mask, s), h = _matrix(sp, N, K, int8, g)
    assert h.launch_count(M) == 2 and h.kernel_name(M) == "expand_kernel + dense_kernel"
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    ws = torch.zeros(h.workspace_size(M), dtype=torch.uint8, device=gu.dev())
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=gu.dev())
    h.linear(gu.bf16_to_dev(x), out=y, workspace=ws)
    # the workspace also serves the calls that need its arrival counters at zero
    y1 = h.linear(gu.bf16_to_dev(x[:1]), workspace=ws)
    sp.check()
    assert not ws[:4096].any()
    toks = np.unique(np.concatenate([[0, M - 1], g.choice(M, 14, replace=False)]))
    xt = np.ascontiguousarray(x[toks])
    ref = oracle.linear_int8(xt, v, mask, s) if int8 else oracle.linear_bf16(xt, v, mask)
    want = synth.bf16_from_f32(ref.astype(np.float32))
    assert np.array_equal(gu.bf16_bits_from_dev(y)[toks], want)
    assert np.array_equal(gu.bf16_bits_from_dev(y1)[0], want[0])
    rows = np.unique(np.concatenate([[0, N - 1], g.choice(N, 30, replace=False)]))
    ref = oracle.linear_int8(x, v[rows], mask[rows], s[rows]) if int8 else oracle.linear_bf16(x, v[rows], mask[rows])
    assert np.array_equal(gu.bf16_bits_from_dev(y)[:, rows], synth.bf16_from_f32(ref.astype(np.float32)))


@pytest.mark.parametrize("int8", [False, True])
@pytest.mark.parametrize("N,K", [(8960, 8192), (2048, 1024), (1024, 1200), (1024, 512), (256, 512)])
def test_one_workspace_size_above_240_rows(N, K, int8):
    """A workspace sized for one batch of more than 240 rows serves every other one, and none
    of fewer rows needs more: matrices of 16 chunks and more, of fewer chunks than SMs too."""
    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(9)
    _, h = _matrix(sp, N, K, int8, g)
    size = h.workspace_size(241)
    assert {h.workspace_size(m) for m in (249, 250, 256, 257, 2048, (1 << 24) + 1)} == {size}
    assert max(h.workspace_size(m) for m in (1, 2, 16, 32, 33, 100, 200, 240)) <= size


def test_workspace_sized_at_241_rows_runs_2048(oracle):
    """64 chunks, fewer than SMs: linear_tc_kernel would need more at 2048 rows than at 241."""
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(3)
    (W, mask, _), h = _matrix(sp, 1024, 512, False, g)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(2048, 512)).astype(np.float32))
    ws = torch.zeros(h.workspace_size(241), dtype=torch.uint8, device=gu.dev())
    y = h.linear(gu.bf16_to_dev(x), workspace=ws)
    sp.check()
    ref = oracle.linear_bf16(np.ascontiguousarray(x[::64]), W, mask)
    assert np.array_equal(gu.bf16_bits_from_dev(y)[::64], synth.bf16_from_f32(ref.astype(np.float32)))


def test_fewer_than_16_chunks_need_more_for_more_rows(oracle):
    """15 chunks stay on linear_tc_kernel: each batch's own size serves it and every smaller one."""
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(4)
    (W, mask, _), h = _matrix(sp, 384, 320, False, g)
    Ms = (1, 32, 33, 240, 241, 300, 2048, 5000)
    sizes = [h.workspace_size(m) for m in Ms]
    assert sizes == sorted(sizes) and h.launch_count(2048) == 1
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(2048, 320)).astype(np.float32))
    for M in (241, 2048):
        ws = torch.zeros(h.workspace_size(M), dtype=torch.uint8, device=gu.dev())
        y = h.linear(gu.bf16_to_dev(x[:M]), workspace=ws)
        sp.check()
        ref = oracle.linear_bf16(np.ascontiguousarray(x[:M:48]), W, mask)
        assert np.array_equal(gu.bf16_bits_from_dev(y)[::48], synth.bf16_from_f32(ref.astype(np.float32)))


def test_update_then_large_batch_on_one_stream(oracle):
    """The expansion reads the values that a masked update before it on the stream wrote."""
    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(5)
    (W, mask, _), h = _matrix(sp, 2048, 1024, False, g)
    grad = g.integers(-3, 4, size=W.shape).astype(np.float32)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(200, 1024)).astype(np.float32))
    xd, gd = gu.bf16_to_dev(x), gu.f32_to_dev(grad)
    h.masked_update(gd, 1.0)
    y = h.linear(xd)
    sp.check()
    w = synth.bf16_from_f32(synth.bf16_to_f32(W) - grad)
    ref = oracle.linear_bf16(x[:16], w, mask)
    assert np.array_equal(gu.bf16_bits_from_dev(y)[:16], synth.bf16_from_f32(ref.astype(np.float32)))
