"""The few-token kernel (weights decoded in registers, warp-level tensor-core instructions) against the checker,
with the bound every linear kernel is held to."""
import numpy as np
import pytest

import oracle
from paper_2602_04163_b200 import binding, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,g,out,in_,M", [
    (2, 128, 160, 640, 5),        # five 32-row groups, a ragged second slice (one block)
    (3, 128, 96, 384, 16),        # a single ragged slice (three blocks)
    (2, 128, 4096, 4096, 8),      # benchmark config 1 with eight tokens: several segments per CTA
    (3, 128, 1024, 2048, 13),
    (2, 256, 64, 1024, 3),        # a coefficient group every two blocks
    (1, 128, 32, 128, 1),
    (4, 128, 48, 1536, 9),        # sixteen candidates; 48 rows: the last row group holds 16 rows
    (2, 128, 272, 896, 17),       # two token tiles, the second holds one token
    (3, 128, 144, 512, 32),       # the most tokens this kernel takes
    (2, 128, 16, 128, 4),         # smallest supported shape
    (2, 64, 80, 384, 6),          # a coefficient group per half block (the paper's W2-G64)
    (3, 64, 272, 896, 24),        # W3-G64, two token tiles
    (4, 64, 48, 1536, 11),
    (1, 64, 1024, 2048, 2),
    (2, 128, 1040, 8192, 16),     # sixteen slices: four column ranges accumulate through the workspace
    (4, 128, 2064, 2048, 16),     # sixteen candidates with tasks of two row groups: several segments per CTA, ragged last task
    (4, 64, 1040, 4096, 20),      # the same with two token tiles and a coefficient group per half block
    (2, 256, 160, 640, 7),        # g = 256 with a short last group (the last slice holds one block of it)
    (3, 256, 272, 1152, 20),      # four and a half groups, two token tiles
])
def test_few_token_kernel(K, g, out, in_, M):
    h, bits, coef = G.make_layer(140 + K, out, in_, K, g, max_M=M)
    x = synth.activations(150 + K, M, in_)
    rows = None
    if out * in_ > 2 ** 22:
        rows = np.unique(np.concatenate([np.arange(0, out, 61), [15, 16, 31, 32, out - 17, out - 16, out - 1]]))
    G.check_linear(h, bits, coef, x, g, binding.KERNEL_FEW, rows=rows, what="few")
    # partial sums of different column ranges meet in binary32 atomic adds whose order is free: two calls may differ
    # by the last binary16 digit, no more (and workspace and counters must come back clean for the second call)
    y1 = G.run_linear(h, x, binding.KERNEL_FEW)
    y2 = G.run_linear(h, x, binding.KERNEL_FEW)
    assert np.allclose(y1, y2, rtol=2.0 ** -9, atol=1e-5)


@pytest.mark.parametrize("K", [1, 2, 3, 4])
def test_few_token_kernel_multiplies_the_dequantized_weights(K):
    """The operand is W^ itself: with one-hot tokens the kernel returns columns of bpdq_dequant exactly."""
    g, out, in_ = 128, 96, 640
    h, bits, coef = G.make_layer(7, out, in_, K, g, max_M=32)
    w = G.run_dequant(h).view(np.float16)
    for c0 in (0, 96, 608):
        x = np.zeros((32, in_), dtype=np.float16)
        x[np.arange(32), c0 + np.arange(32)] = 1.0
        y = G.run_linear(h, x.view(np.uint16), binding.KERNEL_FEW)
        assert np.array_equal(y.astype(np.float16), w[:, c0:c0 + 32].T)


@pytest.mark.parametrize("name,out,in_,K,M", [("gate", 29568, 8192, 2, 16), ("down", 8192, 29568, 3, 8), ("gate", 29568, 8192, 3, 32),
                                               ("down", 8192, 29568, 2, 5), ("7b_down", 3584, 18944, 2, 16), ("gate", 29568, 8192, 4, 12)])
def test_few_token_kernel_full_size_sampled(name, out, in_, K, M):
    """Benchmark-sized layers generated on the device; sampled rows against the checker."""
    g = 128
    h = binding.Handle(out, in_, K, g, None, 960 + K, M)
    x = synth.activations(961, M, in_)
    y = G.run_linear(h, x, binding.KERNEL_FEW)
    rows = np.unique(np.concatenate([np.arange(0, out, max(1, out // 40)), [0, 15, 16, 31, 32, out - 32, out - 16, out - 1]]))
    y_ref, a_ref = oracle.linear(synth.plane_bits(960 + K, out, in_, K, rows), synth.coefficients(960 + K, out, in_, K, g, rows), x, g)
    G.assert_linear_close(y[:, rows], y_ref, a_ref, name)
    assert np.all(np.isfinite(y))


@pytest.mark.parametrize("K,g", [(2, 128), (3, 64), (4, 128), (4, 64)])
def test_dispatcher_on_default_settings(K, g):
    """Which kernel takes how many tokens: the look-up-table kernel up to 2 (3 at K = 4 and g >= 128; two tokens per pass), the
    tensor-core kernels above.  Bit for bit: rows of 14 blocks are not cut between CTAs, and the kernels that a wrong choice would take
    add in another order (some of 2064 x M results differ)."""
    out, in_ = 2064, 1792
    h, bits, coef = G.make_layer(171 + K, out, in_, K, g, max_M=129)
    lut = 3 if K == 4 and g >= 128 else 2
    rows = np.unique(np.concatenate([np.arange(0, out, 61), [127, 128, out - 1]]))
    for M in (1, 2, 3, 4, 16, 17, 33, 128, 129):
        x = synth.activations(172 + M, M, in_)
        n0 = h.bpdq_launch_count()
        ya = G.run_linear(h, x, binding.KERNEL_AUTO)
        assert h.bpdq_launch_count() - n0 == ((M + 1) // 2 if M <= lut else 1)
        y_ref, a_ref = oracle.linear(bits[:, rows], coef[:, rows], x, g)
        G.assert_linear_close(ya[:, rows], y_ref, a_ref, f"auto M={M}")
        gemm = G.run_linear(h, x, binding.KERNEL_GEMM)
        if M > lut:
            assert np.array_equal(ya, gemm)
            if 16 <= M <= binding.FEW_MAX_M:
                assert not np.array_equal(ya, G.run_linear(h, x, binding.KERNEL_FEW))
        else:
            assert not np.array_equal(ya, gemm)
            # four slices meet in binary32 adds in the order of their arrival: the last binary16 digit may differ
            assert np.allclose(ya, G.run_linear(h, x, binding.KERNEL_GEMV), rtol=2.0 ** -9, atol=1e-5)


def test_few_token_kernel_on_request():
    """bpdq_set_few_max_m: single, batched and gated calls with a bias and a permutation, twice in a row, against the checker; one launch
    each beside the gathers.  The kernel's own sums: a batch equals single calls but for the order of adds."""
    import torch
    K, g, M, in_ = 3, 128, 13, 896
    outs = (2064, 144, 2064)
    layers = [G.make_layer(181 + k, o, in_, K, g, max_M=20) for k, o in enumerate(outs)]
    hs = [L[0] for L in layers]
    perm = np.random.RandomState(5).permutation(in_).astype(np.int32)
    bias = np.random.RandomState(6).randn(outs[1]).astype(np.float16)
    hs[0].bpdq_set_input_permutation(perm)
    hs[1].bpdq_set_bias(bias.view(np.uint16))
    x = synth.activations(185, M, in_)
    refs, sums = [], []
    for k, (_, bits, coef) in enumerate(layers):
        y, a = oracle.linear(bits, coef, np.ascontiguousarray(x[:, perm]) if k == 0 else x, g)
        refs.append(y + (bias.astype(np.float64) if k == 1 else 0.0))
        sums.append(a + (np.abs(bias.astype(np.float64)) if k == 1 else 0.0))
    default = [G.run_linear(h, x) for h in hs]
    for h in hs:
        h.bpdq_set_few_max_m(16)
    few = [G.run_linear(h, x, binding.KERNEL_FEW) for h in hs]
    assert any(not np.array_equal(f, d) for f, d in zip(few, default))
    xt = G.x_tensor(x)
    launches = lambda: sum(h.bpdq_launch_count() for h in hs)          # noqa: E731
    for _ in range(2):
        for h, y, a, f in zip(hs, refs, sums, few):
            ya = G.run_linear(h, x)
            G.assert_linear_close(ya, y, a, "single")
            assert np.allclose(ya, f, rtol=2.0 ** -9, atol=1e-5)
        ys = [torch.full((M, o), float("nan"), dtype=torch.float16, device="cuda") for o in outs]
        n0 = launches()
        binding.bpdq_linear_batch(hs, [xt.data_ptr()] * 3, [y.data_ptr() for y in ys], M, G.stream_ptr())
        torch.cuda.synchronize()
        hs[0].bpdq_get_status(G.stream_ptr())
        assert launches() - n0 == 2                                     # one gather, one launch over the three
        for y, r, a, f in zip(ys, refs, sums, few):
            y = y.cpu().numpy().astype(np.float64)
            G.assert_linear_close(y, r, a, "batch")
            assert np.allclose(y, f, rtol=2.0 ** -9, atol=1e-5)
        unit = torch.full((M, outs[0]), float("nan"), dtype=torch.float16, device="cuda")
        n0 = launches()
        binding.bpdq_gate_up_swiglu(hs[0], hs[2], xt.data_ptr(), unit.data_ptr(), M, G.stream_ptr())
        torch.cuda.synchronize()
        hs[0].bpdq_get_status(G.stream_ptr())
        assert launches() - n0 == 2
        want = oracle.swiglu(refs[0], refs[2])
        dg, du = G.TOL_REL * sums[0] + G.TOL_ABS, G.TOL_REL * sums[2] + G.TOL_ABS
        silu_g = oracle.swiglu(refs[0], np.ones_like(refs[0]))
        bound = 1.1 * (np.abs(refs[2]) + du) * dg + (np.abs(silu_g) + 1.1 * dg) * du + 2.0 ** -10 * np.abs(want) + 1e-4
        assert np.all(np.abs(unit.cpu().numpy().astype(np.float64) - want) <= bound)
    for h in hs:
        h.bpdq_set_few_max_m(0)                                         # switched off: the tensor-core kernel takes over
        assert np.array_equal(G.run_linear(h, x), G.run_linear(h, x, binding.KERNEL_GEMM))


def test_few_token_kernel_rejects_what_it_cannot_take():
    h, _, _ = G.make_layer(173, 32, 128, 2, 128, max_M=40)
    import torch
    x = torch.zeros((40, 128), dtype=torch.float16, device="cuda")
    y = torch.zeros((40, 32), dtype=torch.float16, device="cuda")
    n0 = h.bpdq_launch_count()
    with pytest.raises(binding.BpdqError) as ei:
        h.bpdq_linear_ex(x.data_ptr(), y.data_ptr(), binding.FEW_MAX_M + 1, binding.KERNEL_FEW, G.stream_ptr())
    assert ei.value.code == binding.ERR_INVALID and h.bpdq_launch_count() == n0


@pytest.mark.parametrize("g", [128, 64])
def test_dispatcher_with_sixteen_candidates(g):
    """K = 4 through bpdq_linear at the token counts either side of its threshold (look-up-table kernel up to 3 tokens, 2 at
    g = 64; tensor-core kernel beyond): every choice within the checker's bound."""
    K, out, in_ = 4, 272, 1536
    h, bits, coef = G.make_layer(190 + g, out, in_, K, g, max_M=20)
    for M in (1, 2, 3, 4, 16, 17):
        x = synth.activations(191 + M, M, in_)
        n0 = h.bpdq_launch_count()
        G.check_linear(h, bits, coef, x, g, binding.KERNEL_AUTO, what=f"K=4 g={g} M={M}")
        lut_max = 2 if g == 64 else 3
        passes = (M + 1) // 2 if M <= lut_max else 1      # the look-up-table kernel takes two tokens per pass
        assert h.bpdq_launch_count() - n0 == passes
    h.bpdq_destroy()


@pytest.mark.parametrize("K,g,M", [(2, 128, 16), (4, 64, 9), (3, 128, 32)])
def test_few_token_landing_areas_under_load(K, g, M):
    """A layer that keeps every warp refilling its landing area, several launches: a copy that overtook the loads from the area would
    show as rows off by a task's worth of columns.  Weights from bpdq_dequant, sums in binary32."""
    import torch
    out, in_ = 18944, 3584
    h = binding.Handle(out, in_, K, g, None, 17, M)
    x = synth.activations(18, M, in_)
    w = torch.from_numpy(G.run_dequant(h).view(np.float16)).cuda().float()
    ref = (G.x_tensor(x).float() @ w.T).cpu().numpy()
    for _ in range(8):
        y = G.run_linear(h, x, binding.KERNEL_FEW)
        # binary16 rounding of the result (2^-11) and binary32 sums of 3584 terms of size up to 0.2 in another order
        assert np.all(np.abs(y - ref) <= 2.0 ** -10 * np.abs(ref) + 2e-3)
