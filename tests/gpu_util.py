"""Helpers for the GPU parity tests: device buffers via PyTorch, expected values via the checker."""
import numpy as np
import torch

import oracle
from paper_2602_04163_b200 import binding, synth

TOL_REL, TOL_ABS = 4e-3, 1e-3     # |y - y_ref| <= 4e-3 * sum|x_j w_j| + 1e-3

# Prefill launches in which a CTA of the 148 takes four tiles and the first CTA five, the last of them ragged: (K, group, columns, tokens, tokens of a half tile,
# decode groups).  test_rings.py checks that the tile rule and the group rule give these.
TILE_WALK_ROWS = 128 * 4 * 148 + 48
TILE_WALKS = [(2, 128, 640, 100, 64, 4), (3, 64, 640, 129, 80, 4), (3, 128, 640, 200, 112, 4), (1, 256, 384, 250, 128, 4), (2, 128, 640, 200, 112, 2),
              (2, 64, 384, 250, 128, 2), (4, 128, 384, 250, 128, 2), (4, 64, 256, 33, 32, 2), (2, 256, 640, 330, 176, 2), (3, 128, 384, 500, 256, 2)]


def stream_ptr() -> int:
    return torch.cuda.current_stream().cuda_stream


def make_layer(seed, out, in_, K, g, max_M=1, on_device=False):
    """Returns (handle, bits, coef).  With on_device=True the blob is generated by the library's
    device filler; bits/coef then come from the host generator, which must describe the same tensors."""
    bits = synth.plane_bits(seed, out, in_, K)
    coef = synth.coefficients(seed, out, in_, K, g)
    if on_device:
        h = binding.Handle(out, in_, K, g, None, seed, max_M)
    else:
        h = binding.Handle(out, in_, K, g, binding.bpdq_pack(bits, coef, g), 0, max_M)
    return h, bits, coef


def x_tensor(x_bits: np.ndarray) -> torch.Tensor:
    return torch.from_numpy(x_bits.view(np.int16).copy()).cuda().view(torch.float16)


def run_linear(h, x_bits: np.ndarray, kernel=binding.KERNEL_AUTO) -> np.ndarray:
    M = x_bits.shape[0]
    x = x_tensor(x_bits)
    y = torch.full((M, h.out), float("nan"), dtype=torch.float16, device="cuda")
    h.bpdq_linear_ex(x.data_ptr(), y.data_ptr(), M, kernel, stream_ptr())
    torch.cuda.synchronize()
    h.bpdq_get_status(stream_ptr())
    return y.cpu().numpy().astype(np.float64)


def run_dequant(h) -> np.ndarray:
    w = torch.empty((h.out, h.in_), dtype=torch.float16, device="cuda")
    h.bpdq_dequant(w.data_ptr(), stream_ptr())
    torch.cuda.synchronize()
    return w.view(torch.int16).cpu().numpy().view(np.uint16)


def assert_linear_close(y_gpu, y_ref, a_ref, what=""):
    err = np.abs(y_gpu - y_ref)
    bound = TOL_REL * a_ref + TOL_ABS
    bad = np.argwhere(~(err <= bound))
    assert bad.size == 0, f"{what}: {bad.shape[0]} elements out of tolerance, first {bad[:5].tolist()}, " \
                          f"max err/bound {np.nanmax(err / bound):.3g}"
    return float(np.max(err / bound))


def check_linear(h, bits, coef, x_bits, g, kernel=binding.KERNEL_AUTO, rows=None, what=""):
    y = run_linear(h, x_bits, kernel)
    if rows is not None:
        y_ref, a_ref = oracle.linear(bits[:, rows], coef[:, rows], x_bits, g)
        return assert_linear_close(y[:, rows], y_ref, a_ref, what)
    y_ref, a_ref = oracle.linear(bits, coef, x_bits, g)
    return assert_linear_close(y, y_ref, a_ref, what)
