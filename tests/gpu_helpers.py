"""Shared helpers of the GPU parity tests: device buffers through torch (memory
plumbing only), oracle set-up from the seeded generators, tolerances."""
from __future__ import annotations

import numpy as np

import synth
from oracle import model as M
from oracle import quant

# Tolerances of the parity bar: max |gpu - ref| <= tau * max |ref| per tensor,
# 2e-2 on bf16 / int8 weight paths, 5e-2 on int4 weight paths (GPTQ4 is int4).
TAU = {0: 2e-2, 1: 2e-2, 2: 5e-2, 3: 5e-2}


def torch_mod():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


# Every device buffer a test makes stays referenced until the test ends, so a
# pointer taken from a temporary (ptr(dev(x))) cannot be recycled by torch's
# caching allocator before the kernel reading it has run.
KEEP = []


def dev(a: np.ndarray):
    """Host numpy array -> device tensor with the same bytes."""
    torch = torch_mod()
    a = np.ascontiguousarray(a)
    view = {np.dtype(np.uint16): np.int16, np.dtype(np.uint32): np.int32}.get(a.dtype)
    t = torch.from_numpy(a.view(view) if view else a).to("cuda")
    KEEP.append(t)
    return t


def host(t, dtype):
    torch = torch_mod()
    torch.cuda.synchronize()
    a = t.detach().cpu().numpy()
    return a.view(dtype)


def empty(n_bytes_or_shape, dtype=np.uint8):
    torch = torch_mod()
    tmap = {np.dtype(np.uint8): torch.uint8, np.dtype(np.int8): torch.int8, np.dtype(np.uint16): torch.int16,
            np.dtype(np.int16): torch.int16, np.dtype(np.int32): torch.int32, np.dtype(np.float32): torch.float32}
    shape = n_bytes_or_shape if isinstance(n_bytes_or_shape, tuple) else (n_bytes_or_shape,)
    t = torch.zeros(shape, dtype=tmap[np.dtype(dtype)], device="cuda")
    KEEP.append(t)
    return t


def ptr(t):
    return t.data_ptr() if t is not None else None


def rel_err(gpu, ref):
    gpu = np.asarray(gpu, np.float64)
    ref = np.asarray(ref, np.float64)
    return float(np.max(np.abs(gpu - ref)) / max(np.max(np.abs(ref)), 1e-30))


# ---------------------------------------------------------------- linears
def check_decode_linear(fp, wq, m, n, k, epi):
    """fp_op_linear (m <= 64) on seeded weights against the oracle; the residual in place."""
    w = synth.weight_bf16(70 + wq, 0, 1, (n, k))
    x = synth.uniform_bf16(71, m, (m, k), -2.0, 2.0)
    nout = n // 2 if epi == 2 else n
    r = synth.uniform_bf16(72, m, (m, nout), -1.0, 1.0)
    codes, scales, zeros = empty(n * k * 2), empty(n * (k // 128), np.uint16), empty(n * (k // 128), np.uint16)
    fp.fp_op_quantize(wq, ptr(dev(w)), n, k, ptr(codes), ptr(scales), ptr(zeros))
    out = dev(r) if epi == 1 else empty(m * nout * (4 if epi == 3 else 2))
    ws_b = fp.fp_op_linear_workspace_bytes(wq, m, n, k)
    ws = empty(max(ws_b, 16))
    fp.fp_op_linear(wq, epi, ptr(dev(x)), m, n, k, ptr(codes), ptr(scales), ptr(zeros), ptr(out if epi == 1 else dev(r)),
                    ptr(out), ptr(ws), ws_b)
    got = host(out, np.float32) if epi == 3 else quant.bf16_to_f32(host(out, np.uint16))
    wd = quant.quantize_weight(w, wq)[1]
    if wq == 2 and m >= 17:  # the tcgen05 path multiplies bf16((q - z) s)
        wd = quant.bf16_to_f32(synth.f32_to_bf16_bits(wd.astype(np.float32))).astype(np.float64)
    ref = quant.bf16_to_f32(x).astype(np.float64) @ wd.T
    if epi == 1:
        ref = ref + quant.bf16_to_f32(r).astype(np.float64)
    elif epi == 2:
        ref = M.silu(ref[:, :nout]) * ref[:, nout:]
    # fp32 sums; int8 codes carry an offset of 1152 that is taken out of the sum
    # (2^-24 of 1152 sum|x| against sum|q x|, q up to 127); one rounding to bf16
    err = rel_err(got.reshape(m, nout), ref)
    assert err <= (1e-4 if epi == 3 else 1.05 * 2.0 ** -8 + 1e-4), err


# ---------------------------------------------------------------- weights
def arch_dict(a: M.Arch):
    return dict(n_layers=a.n_layers, hidden=a.hidden, n_heads=a.n_heads, n_kv_heads=a.n_kv_heads,
                head_dim=a.head_dim, ffn=a.ffn, vocab=a.vocab, rms_eps=a.rms_eps, rope_base=a.rope_base)


def weight_getter(seed, gains="random", scale=1.0):
    """bf16 tensors for both sides: seeded N(0, 0.02)-like matrices (times
    ``scale``) and random gains in [0.5, 1.5) so a dropped gain shows."""

    def get(layer, t, shape):
        if len(shape) == 1:
            if gains == "ones":
                return synth.f32_to_bf16_bits(np.ones(shape, np.float32))
            return synth.uniform_bf16(seed, 900 + 16 * (layer + 1) + t, shape, 0.5, 1.5)
        w = synth.weight_bf16(seed, layer, t, shape)
        if scale != 1.0:
            w = synth.f32_to_bf16_bits(quant.bf16_to_f32(w) * np.float32(scale))
        return w

    return get


def upload_weights(fp, h, arch: M.Arch, get):
    for t in range(3):
        fp.fp_set_weight(h, -1, t, get(-1, t, M.tensor_shape(arch, -1, t)).reshape(-1))
    for l in range(arch.n_layers):
        for t in range(9):
            fp.fp_set_weight(h, l, t, get(l, t, M.tensor_shape(arch, l, t)).reshape(-1))
