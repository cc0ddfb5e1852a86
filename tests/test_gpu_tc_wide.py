"""Batches of 33 to 249 rows of wide matrices on linear_tc_kernel, whose CTAs share row blocks:
segments of two and three CTAs, finished by one that runs it last or by one of several that end
together, one and several token blocks, both value types.  Integer-valued inputs make every sum
exact, so they must match bit for bit; the workspace's counters return to zero."""
import numpy as np
import pytest

from paper_2405_03594_gb300 import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,Ms", [(22016, 4096, (33, 64, 100, 199)), (12288, 4096, (40, 46)), (12280, 4104, (33, 46)),
                                    (12283, 4096, (33, 46))])
@pytest.mark.parametrize("int8", [False, True])
def test_shared_segments_bit_exact(oracle, N, K, Ms, int8):
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N + K)
    mask = (g.random((N, K)) < 0.3).astype(np.uint8)
    if int8:
        v = g.integers(-128, 128, size=(N, K)).astype(np.int8)
        s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
        h = sp.compress(gu.i8_to_dev(v), gu.u8_to_dev(mask), gu.f32_to_dev(s))
    else:
        v = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
        h = sp.compress(gu.bf16_to_dev(v), gu.u8_to_dev(mask))
    rows = np.unique(np.concatenate([[0, N - 1], g.choice(N, 200, replace=False)]))
    for M in Ms:
        assert h.launch_count(M) == 1 and h.kernel_name(M) == "linear_tc_kernel"
        x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
        ws = torch.zeros(h.workspace_size(M), dtype=torch.uint8, device=gu.dev())
        ref = oracle.linear_int8(x, v[rows], mask[rows], s[rows]) if int8 else oracle.linear_bf16(x, v[rows], mask[rows])
        want = synth.bf16_from_f32(ref.astype(np.float32))
        first = None
        for _ in range(4):
            y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=gu.dev())
            h.linear(gu.bf16_to_dev(x), out=y, workspace=ws)
            got = gu.bf16_bits_from_dev(y)
            assert np.array_equal(got[:, rows], want)
            first = got if first is None else first
            assert np.array_equal(got, first)
        sp.check()
        assert not ws[:4096].any()
