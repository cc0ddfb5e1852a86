"""Calls without a workspace of their own: they may overlap on several streams, come from several
threads, be captured into a graph and grow the workspace between replays.  Large batches expand
the matrix into the workspace by one launch and multiply by the next, so a shared one would give
wrong products.  Integer-valued inputs make every sum exact, so results must match bit for bit."""
import threading

import numpy as np
import pytest

from paper_2405_03594_gb300 import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _case(sp, oracle, N, K, M, seed):
    g = np.random.default_rng(seed)
    mask = (g.random((N, K)) < 0.3).astype(np.uint8)
    W = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    h = sp.compress(gu.bf16_to_dev(W), gu.u8_to_dev(mask))
    want = synth.bf16_from_f32(oracle.linear_bf16(x, W, mask).astype(np.float32))
    return h, gu.bf16_to_dev(x), want


def test_one_workspace_per_stream_thread_and_capture():
    import torch

    from paper_2405_03594_gb300 import sp

    sp.release_workspaces()
    dev = gu.dev()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    a, b, c = sp.workspace_for(4096, dev), sp.workspace_for(4096, dev, s1), sp.workspace_for(4096, dev, s2)
    assert len({a.data_ptr(), b.data_ptr(), c.data_ptr()}) == 3
    assert sp.workspace_for(2048, dev, s1) is b  # kept
    with torch.cuda.stream(s1):
        assert sp.workspace_for(4096, dev) is b  # the current stream is the same stream
    grown = sp.workspace_for(200000, dev, s1)
    s1.synchronize()
    assert grown.numel() >= 200000 and not grown[:65536].any() and sp.workspace_for(4096, dev, s1) is grown
    other = []
    t = threading.Thread(target=lambda: other.append(sp.workspace_for(4096, dev)))
    t.start()
    t.join()
    assert other[0].data_ptr() != a.data_ptr()
    g = torch.cuda.CUDAGraph()
    captured = []
    with torch.cuda.graph(g, stream=s2):
        captured += [sp.workspace_for(4096, dev), sp.workspace_for(2048, dev)]
    assert captured[0] is captured[1] and captured[0].data_ptr() not in (a.data_ptr(), c.data_ptr())
    assert sp.workspace_for(4096, dev, s2) is c  # not the graph's
    for _ in range(20):
        sp.workspace_for(4096, dev, torch.cuda.Stream())
    assert len(sp._workspaces.kept) <= 8
    sp.release_workspaces()
    assert not sp._workspaces.kept


def test_calls_on_two_streams(oracle):
    import torch

    from paper_2405_03594_gb300 import sp

    cases = [_case(sp, oracle, N, K, M, N) for N, K, M in ((4096, 2048, 300), (4096, 1024, 257))]
    streams = [torch.cuda.Stream() for _ in cases]
    torch.cuda.synchronize()
    ys = []
    for _ in range(12):
        for (h, x, want), s in zip(cases, streams):
            y = torch.empty((x.shape[0], h.n), dtype=torch.bfloat16, device=x.device)
            ys.append((y, want))
            s.wait_stream(torch.cuda.current_stream())
            h.linear(x, out=y, stream=s)
    sp.check()
    torch.cuda.synchronize()
    for y, want in ys:
        assert np.array_equal(gu.bf16_bits_from_dev(y), want)


def test_calls_from_threads_on_one_stream(oracle):
    import torch

    from paper_2405_03594_gb300 import sp

    cases = [_case(sp, oracle, 2048, 1024, 300 + i, i) for i in range(4)]
    stream = torch.cuda.current_stream()
    out = [[] for _ in cases]
    start = threading.Barrier(len(cases))

    def work(i):
        h, x, _ = cases[i]
        start.wait()
        for _ in range(8):
            out[i].append(h.linear(x, stream=stream))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    sp.check()
    torch.cuda.synchronize()
    for (_, _, want), ys in zip(cases, out):
        assert len(ys) == 8
        for y in ys:
            assert np.array_equal(gu.bf16_bits_from_dev(y), want)


@pytest.mark.parametrize("M", [1, 300])
def test_a_graph_keeps_its_workspace(oracle, M):
    """Replays beside a larger call that outgrows what the thread keeps, and beside calls on
    another stream."""
    import torch

    from paper_2405_03594_gb300 import sp

    h, x, want = _case(sp, oracle, 2048, 1024, M, 7)
    big, xb, want_big = _case(sp, oracle, 4096, 2048, 400, 8)
    h.linear(x)  # per-device kernel attributes are set outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y = h.linear(x)
    other = torch.cuda.Stream()
    for _ in range(4):
        yb = big.linear(xb)
        sp.release_workspaces()
        torch.cuda.empty_cache()
        junk = torch.full((64 << 20,), 255, dtype=torch.uint8, device=gu.dev())
        other.wait_stream(torch.cuda.current_stream())
        y.zero_()
        g.replay()
        yo = torch.empty_like(yb)
        big.linear(xb, out=yo, stream=other)
        sp.check()
        torch.cuda.synchronize()
        del junk
        assert np.array_equal(gu.bf16_bits_from_dev(y), want)
        assert np.array_equal(gu.bf16_bits_from_dev(yb), want_big)
        assert np.array_equal(gu.bf16_bits_from_dev(yo), want_big)


@pytest.mark.parametrize("int8", [False, True])
@pytest.mark.parametrize("N,K,M", [(4096, 4096, 33), (9000, 2056, 300)])
def test_large_batch_without_room_for_the_expanded_matrix(oracle, N, K, M, int8):
    """A workspace of the one-launch kernels' size is accepted, and one byte less is not."""
    import torch

    from paper_2405_03594_gb300 import sp

    g = np.random.default_rng(N + M)
    mask = (g.random((N, K)) < 0.3).astype(np.uint8)
    x = synth.bf16_from_f32(g.integers(-2, 3, size=(M, K)).astype(np.float32))
    rows = np.unique(np.concatenate([[0, N - 1], g.choice(N, 200, replace=False)]))
    if int8:
        v = g.integers(-128, 128, size=(N, K)).astype(np.int8)
        s = np.exp2(g.integers(-3, 4, size=N)).astype(np.float32)
        h = sp.compress(gu.i8_to_dev(v), gu.u8_to_dev(mask), gu.f32_to_dev(s))
        ref = oracle.linear_int8(x, v[rows], mask[rows], s[rows])
    else:
        v = synth.bf16_from_f32(g.integers(-4, 5, size=(N, K)).astype(np.float32))
        h = sp.compress(gu.bf16_to_dev(v), gu.u8_to_dev(mask))
        ref = oracle.linear_bf16(x, v[rows], mask[rows])
    want = synth.bf16_from_f32(ref.astype(np.float32))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    counters = (32 * sms + 255) // 256 * 256
    ntok = min(256, (M + 15) // 16 * 16)
    # split-K partials of 128 rows: two per CTA, of 16 tokens on up to four CTAs per SM (its first
    # 16 rows' kernels) or of the token tile on one
    size = max(h.workspace_size(1), counters + 2 * sms * 128 * ntok * 4)
    assert size < h.workspace_size(M)
    xd = gu.bf16_to_dev(x)
    ws = torch.zeros(size, dtype=torch.uint8, device=gu.dev())
    y = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device=gu.dev())
    h.linear(xd, out=y, workspace=ws)
    sp.check()
    assert not ws[:counters].any()
    assert np.array_equal(gu.bf16_bits_from_dev(y)[:, rows], want)
    with pytest.raises(sp.SpError) as e:
        h.linear(xd, out=y, workspace=ws[:size - 1])
    assert e.value.code == 8
    if int8:  # activations that are whole numbers widen exactly with unit scales
        xb = (M * K * 2 + 255) // 256 * 256
        ws = torch.zeros((size + 255) // 256 * 256 + xb, dtype=torch.uint8, device=gu.dev())
        assert ws.numel() < h.w8a8_workspace_size(M)
        y.fill_(float("nan"))
        qx = gu.i8_to_dev(synth.bf16_to_f32(x).astype(np.int8))
        h.linear_w8a8(qx, gu.f32_to_dev(np.ones(M, dtype=np.float32)), out=y, workspace=ws)
        sp.check()
        assert np.array_equal(gu.bf16_bits_from_dev(y)[:, rows], want)
