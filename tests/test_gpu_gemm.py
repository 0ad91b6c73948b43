"""bpdq_gemm (TMA + tcgen05 tensor-core kernel) against the checker, same bound as every linear kernel."""
import numpy as np
import pytest

import oracle
from paper_2602_04163_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,g,out,in_,M", [
    (2, 128, 128, 128, 16),      # one tile, one 128-column block, two stages
    (2, 128, 128, 1024, 32),     # more k-blocks than pipeline stages: every barrier wraps
    (3, 128, 256, 512, 33),      # 48 token columns, the last fifteen beyond M
    (1, 128, 128, 256, 5),
    (2, 64, 128, 384, 64),       # a coefficient group per k-block
    (3, 256, 256, 768, 100),     # a coefficient group every four k-blocks, 112 token columns
    (2, 128, 160, 640, 130),     # ragged last row tile (160 = 128 + 32), several token tiles, the last one ragged
    (3, 128, 384, 2048, 257),    # an odd number of tokens, the last tile ragged
    (2, 128, 1024, 1024, 300),
    (2, 128, 128, 128, 1),       # a single token through the tensor-core path
    (4, 128, 256, 512, 40),      # sixteen candidates per group (the paper's W4-G128): two byte-permutes and a select
    (4, 64, 128, 384, 300),
    (2, 128, 256, 4096, 40),     # few row tiles, long rows: four CTAs share a tile
    (3, 64, 128, 8192, 64),      # eight shares
    (4, 128, 384, 2048, 7),      # two shares per tile, ragged token columns
    (2, 128, 256, 4096, 100),    # 112 token columns: one accumulator pair, four shares per tile
    (3, 128, 384, 2048, 128),    # two shares per tile, all 128 token columns in use
    (2, 256, 160, 640, 24),      # g = 256 with a short last group: TMEM kernel
    (3, 256, 272, 1152, 200),    # ... prefill kernel, one token tile
    (2, 256, 160, 1664, 600),    # ... several token tiles (six and a half groups)
    (2, 128, 256, 384, 20500),   # more token tiles than SMs: a second tile for some CTAs, odd number of blocks per tile
    (4, 128, 128, 640, 38000),   # the same with the largest packed blocks (K = 4)
    (3, 64, 160, 640, 24),       # TMEM kernel, ragged last row tile (the tensor maps fill the missing rows), two groups per block
    (1, 256, 144, 1024, 100),    # TMEM kernel with 112 token columns, ragged row tile, a group every two blocks
    (2, 128, 400, 1152, 9),      # 16 token columns, odd number of blocks, rings wrap at different blocks
    (2, 128, 256, 512, 256),     # prefill kernel, 64-column stages
    (3, 128, 384, 2048, 200),    # prefill kernel, ragged token tile
    (2, 64, 160, 640, 700),      # prefill kernel, several token tiles, ragged row tile, a group per half block
    (3, 256, 272, 1024, 513),    # an odd number of tokens over 512; a group every two blocks
    (1, 128, 128, 256, 1030),    # two blocks per tile, several token tiles
    (4, 128, 256, 384, 300),     # prefill kernel with sixteen candidates (largest packed blocks), odd number of blocks per tile
])
def test_gemm_kernel(K, g, out, in_, M):
    h, bits, coef = G.make_layer(60 + K, out, in_, K, g, max_M=M)
    x = synth.activations(70 + K, M, in_)
    rows = None
    if M > 4096:                 # many tokens: every token, rows sampled from every 32-row quadrant of every row tile
        rows = np.unique(np.concatenate([np.arange(0, out, 37), [0, 31, 32, 127, out - 128, out - 1]]))
    G.check_linear(h, bits, coef, x, g, binding.KERNEL_GEMM, rows=rows, what="gemm")
    y1 = G.run_linear(h, x, binding.KERNEL_GEMM)
    y2 = G.run_linear(h, x, binding.KERNEL_GEMM)
    if M > 128 or in_ < 2048:
        assert np.array_equal(y1, y2)                    # one CTA per output tile, fixed accumulation order: bit-identical reruns
    else:                                                # CTAs that share a tile add their parts in a free order: last binary16 digit
        assert np.allclose(y1, y2, rtol=2.0 ** -9, atol=1e-5)


@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_gemm_equals_dequant_times_x(K):
    """The decoded operand is W^ itself: with one-hot tokens the kernel must return columns of bpdq_dequant exactly."""
    g, out, in_ = 128, 256, 512
    h, bits, coef = G.make_layer(5, out, in_, K, g, max_M=in_)
    w = G.run_dequant(h).view(np.float16)
    x = np.eye(in_, dtype=np.float16)                    # token t selects column t
    y = G.run_linear(h, x.view(np.uint16), binding.KERNEL_GEMM)
    assert np.array_equal(y.astype(np.float16), w.T)


def test_dispatch_sends_large_m_to_the_tensor_core_kernel():
    K, g, out, in_, M = 2, 128, 256, 512, 48
    h, bits, coef = G.make_layer(9, out, in_, K, g, max_M=M)
    x = synth.activations(10, M, in_)
    G.check_linear(h, bits, coef, x, g, binding.KERNEL_AUTO, what="auto")
    assert np.array_equal(G.run_linear(h, x, binding.KERNEL_AUTO), G.run_linear(h, x, binding.KERNEL_GEMM))


@pytest.mark.parametrize("name,out,in_,K,M", [("gate", 29568, 8192, 3, 2048), ("down", 8192, 29568, 2, 512)])
def test_gemm_full_size_sampled(name, out, in_, K, M):
    """72B-shaped layers generated on the device; a row of every few tiles, every token, against the checker."""
    g = 128
    h = binding.Handle(out, in_, K, g, None, 950 + K, M)
    x = synth.activations(951, M, in_)
    y = G.run_linear(h, x, binding.KERNEL_GEMM)
    rows = np.unique(np.concatenate([np.arange(0, out, 997), [0, 127, 128, out - 129, out - 128, out - 1]]))
    y_ref, a_ref = oracle.linear(synth.plane_bits(950 + K, out, in_, K, rows),
                                 synth.coefficients(950 + K, out, in_, K, g, rows), x, g)
    G.assert_linear_close(y[:, rows], y_ref, a_ref, name)
    assert np.all(np.isfinite(y))


@pytest.mark.parametrize("K,g,M", [(2, 128, 48), (2, 256, 100), (3, 64, 40), (4, 128, 128), (3, 64, 300)])
def test_gemm_packed_ring_under_load(K, g, M):
    """A layer that keeps every SM's packed ring turning, several launches: a slot that is refilled before the last load from it
    has returned shows as rows that are off by a few columns' worth.  Weights from bpdq_dequant, sums in binary32."""
    import torch
    out, in_ = 18944, 3584
    h = binding.Handle(out, in_, K, g, None, 17, M)
    x = synth.activations(18, M, in_)
    w = torch.from_numpy(G.run_dequant(h).view(np.float16)).cuda().float()
    ref = (G.x_tensor(x).float() @ w.T).cpu().numpy()
    for _ in range(8):
        y = G.run_linear(h, x, binding.KERNEL_GEMM)
        # binary16 rounding of the result (2^-11) and binary32 sums of 3584 terms of size up to 0.2 in another order
        assert np.all(np.abs(y - ref) <= 2.0 ** -10 * np.abs(ref) + 2e-3)


@pytest.mark.parametrize("K,g,shapes,M", [
    (2, 128, [(4096, 2048), (528, 2048), (512, 2048)], 5),       # rows of one length, fewer tiles than SMs: all are cut
    (3, 64, [(20000, 2048), (272, 2048)], 16),                   # a whole tile per CTA and shared ones, across a linear's end
    (2, 256, [(400, 1152), (272, 640), (16, 2176)], 3),          # rows of different lengths, ragged tiles
    (4, 128, [(144, 384), (160, 384)], 9),                       # short rows: whole tiles only
])
def test_gemm_batch(K, g, shapes, M):
    """Several linears in one launch of the tensor-core kernel, each against the checker; a second call finds clean state."""
    import torch
    hs, ref, xs, ys = [], [], [], []
    for k, (o, i) in enumerate(shapes):
        h, bits, coef = G.make_layer(400 + k, o, i, K, g, max_M=M)
        x = synth.activations(410 + k, M, i)
        rows = np.unique(np.concatenate([np.arange(0, o, 1 + o // 200), [0, o - 17 if o > 16 else 0, o - 1]]))
        bias = np.random.RandomState(k).randn(o).astype(np.float16)
        if k == 1:
            h.bpdq_set_bias(bias.view(np.uint16))
        r, a = oracle.linear(bits[:, rows], coef[:, rows], x, g)
        ref.append((rows, r + (bias[rows].astype(np.float64) if k == 1 else 0.0), a + (np.abs(bias[rows].astype(np.float64)) if k == 1 else 0.0)))
        hs.append(h)
        xs.append(G.x_tensor(x))
        ys.append(torch.full((M, o), float("nan"), dtype=torch.float16, device="cuda"))
    for _ in range(2):
        n0 = sum(h.bpdq_launch_count() for h in hs)
        binding.bpdq_linear_batch(hs, [x.data_ptr() for x in xs], [y.data_ptr() for y in ys], M, G.stream_ptr())
        torch.cuda.synchronize()
        hs[0].bpdq_get_status(G.stream_ptr())
        assert sum(h.bpdq_launch_count() for h in hs) == n0 + 1
        for y, (rows, r, a) in zip(ys, ref):
            G.assert_linear_close(y.cpu().numpy().astype(np.float64)[:, rows], r, a, "batch")


@pytest.mark.parametrize("K,g,out,in_,M", [(2, 128, 2064, 2048, 17), (3, 64, 528, 896, 100), (4, 128, 272, 4096, 128), (2, 128, 40000, 256, 33)])
def test_gated_unit_up_to_128_tokens_in_one_launch(K, g, out, in_, M):
    """silu(gate) * up from unrounded sums: shared tiles, whole tiles and short rows."""
    import torch
    hg, bg, cg = G.make_layer(420, out, in_, K, g, max_M=M)
    hu, bu, cu = G.make_layer(421, out, in_, K, g, max_M=M)
    x = synth.activations(422, M, in_)
    rows = np.unique(np.concatenate([np.arange(0, out, 1 + out // 100), [127, 128, out - 1]]))
    gy, ga = oracle.linear(bg[:, rows], cg[:, rows], x, g)
    uy, ua = oracle.linear(bu[:, rows], cu[:, rows], x, g)
    want = oracle.swiglu(gy, uy)
    dg, du = G.TOL_REL * ga + G.TOL_ABS, G.TOL_REL * ua + G.TOL_ABS
    silu_g = oracle.swiglu(gy, np.ones_like(gy))
    bound = 1.1 * (np.abs(uy) + du) * dg + (np.abs(silu_g) + 1.1 * dg) * du + 2.0 ** -10 * np.abs(want) + 1e-4
    xt = G.x_tensor(x)
    for _ in range(2):
        hout = torch.full((M, out), float("nan"), dtype=torch.float16, device="cuda")
        n0 = hg.bpdq_launch_count() + hu.bpdq_launch_count()
        binding.bpdq_gate_up_swiglu(hg, hu, xt.data_ptr(), hout.data_ptr(), M, G.stream_ptr())
        torch.cuda.synchronize()
        hg.bpdq_get_status(G.stream_ptr())
        assert hg.bpdq_launch_count() + hu.bpdq_launch_count() == n0 + 1
        assert np.all(np.abs(hout.cpu().numpy().astype(np.float64)[:, rows] - want) <= bound)


@pytest.mark.parametrize("K,g,in_,M", [(2, 128, 256, 17), (3, 64, 128, 64), (4, 128, 384, 64), (2, 256, 1024, 65), (3, 64, 896, 128), (2, 128, 1152, 100)])
def test_short_rows_in_more_tiles_than_sms(K, g, in_, M):
    """Either side of the lines where up to 128 tokens of short rows go to the prefill kernel; a tile more than SMs, the last one
    ragged.  Weights from bpdq_dequant, sums in binary32."""
    import torch
    out = 128 * torch.cuda.get_device_properties(0).multi_processor_count + 48
    h = binding.Handle(out, in_, K, g, None, 23, M)
    bias = np.random.RandomState(3).randn(out).astype(np.float16)
    h.bpdq_set_bias(bias.view(np.uint16))
    x = synth.activations(24, M, in_)
    w = torch.from_numpy(G.run_dequant(h).view(np.float16)).cuda().float()
    ref = (G.x_tensor(x).float() @ w.T).cpu().numpy() + bias.astype(np.float32)
    for kernel in (binding.KERNEL_AUTO, binding.KERNEL_GEMM):
        y = G.run_linear(h, x, kernel)
        # binary16 rounding of the result (2^-11) and binary32 sums of up to 1152 terms of size up to 0.2 in another order
        assert np.all(np.abs(y - ref) <= 2.0 ** -10 * np.abs(ref) + 2e-3)


@pytest.mark.parametrize("K,g,out,in_,M", [
    (2, 128, 512, 3584, 777),        # halves of 16 tokens: four decode groups
    (3, 64, 160, 384, 9000),         # halves of 64: three blocks per tile, a ragged row tile and a ragged last token tile
    (1, 256, 128, 640, 20000),       # halves of 80: an odd number of blocks, a short last group
    (2, 128, 3584, 1152, 777),       # halves of 80 with two decode groups
    (3, 128, 1024, 512, 4096),       # halves of 128: the widest MMA
    (4, 128, 144, 256, 2100),        # sixteen candidates: two decode groups at any half
])
def test_whole_tiles_of_up_to_256_tokens(K, g, out, in_, M):
    """One MMA for a whole token tile, one tile per CTA.  Weights from bpdq_dequant, sums in binary32; every call returns the same bits."""
    check_against_dequant(K, g, out, in_, M)


@pytest.mark.parametrize("K,g,in_,M,half,groups", G.TILE_WALKS)
def test_ctas_walk_over_several_tiles(K, g, in_, M, half, groups):
    """Four or five tiles per CTA: stage and packed slots run on from tile to tile, the two accumulators of whole tiles are used again (from the
    third tile on) while the other is drained, and the one of longer tiles after its drain."""
    check_against_dequant(K, g, G.TILE_WALK_ROWS, in_, M)


def check_against_dequant(K, g, out, in_, M):
    import torch
    h = binding.Handle(out, in_, K, g, None, 29, M)
    x = G.x_tensor(synth.activations(30, M, in_))
    w = torch.from_numpy(G.run_dequant(h).view(np.float16)).cuda().float()
    ref = x.float() @ w.T
    first = None
    for _ in range(4):
        y = torch.full((M, out), float("nan"), dtype=torch.float16, device="cuda")
        h.bpdq_linear_ex(x.data_ptr(), y.data_ptr(), M, binding.KERNEL_GEMM, G.stream_ptr())
        torch.cuda.synchronize()
        h.bpdq_get_status(G.stream_ptr())
        if first is None:
            first = y
            # binary16 rounding of the result (2^-11) and binary32 sums of up to 3584 terms of size up to 0.2 in another order
            assert bool(torch.all((y.float() - ref).abs() <= 2.0 ** -10 * ref.abs() + 2e-3))
        assert torch.equal(first, y)
