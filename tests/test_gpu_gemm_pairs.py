"""The prefill GEMM on single CTAs (128 x 256 tiles; small matrices) and on pairs of
them (256 x 256; a long K): ragged rows around
one and two tiles (the odd CTA of a pair with no or few rows), ragged columns (half a
weight tile past N), K tails, every epilogue; the expansion of int8, int4 and GPTQ4
weights for K around its blocks of 4096 elements and its rows that share one."""
import numpy as np
import pytest

import synth
from oracle import model as M
from oracle import quant
from tests.gpu_helpers import TAU, dev, empty, host, ptr, rel_err, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


def _check(fp, m, n, k, epi, w):
    x = synth.uniform_bf16(6, m, (m, k), -2.0, 2.0)
    nout = n // 2 if epi == 2 else n
    r = synth.uniform_bf16(7, m, (m, nout), -1.0, 1.0)
    out = empty(m * nout * (4 if epi == 3 else 2))
    for _ in range(2):
        fp.fp_op_linear(0, epi, ptr(dev(x)), m, n, k, ptr(dev(w)), None, None, ptr(dev(r)), ptr(out))
    got = host(out, np.float32) if epi == 3 else quant.bf16_to_f32(host(out, np.uint16))
    ref = quant.bf16_to_f32(x).astype(np.float64) @ quant.bf16_to_f32(w).astype(np.float64).T
    if epi == 1:
        ref = ref + quant.bf16_to_f32(r).astype(np.float64)
    elif epi == 2:
        ref = M.silu(ref[:, :nout]) * ref[:, nout:]
    # fp32 sums of exact products, a step of the tensor core adding 16 of them and dropping
    # less than a unit in the last place (2^-23) of the sum; one rounding to bf16 (2^-8)
    assert rel_err(got.reshape(m, nout), ref) <= (max(1e-5, k / 16 * 2.0 ** -23) if epi == 3 else 1.05 * 2.0 ** -8)


@pytest.mark.parametrize("epi", [0, 1, 2, 3])
@pytest.mark.parametrize("m,n,k", [(65, 256, 64), (128, 520, 192), (129, 392, 72), (256, 1024, 4160), (257, 264, 128),
                                   (513, 776, 328), (300, 20000, 64), (2100, 2304, 256)])
def test_tiles(fp, m, n, k, epi):
    _check(fp, m, n, k, epi, synth.weight_bf16(5, 0, 1, (n, k)))


# one round of pairs from K 3072 and 2^24 weights, two from K 1024 (with SwiGLU 1536), and 79 pairs of
# tiles, a round more than the single CTAs need
@pytest.mark.parametrize("n,k,ms", [(5464, 3080, (65, 128, 129, 256, 257, 300)), (5440, 3080, (129, 300)),
                                    (5496, 3064, (257,)), (4104, 8200, (300,)),
                                    (2304, 1544, (2100,)), (2304, 1024, (2049,)), (2304, 1016, (2100,)),
                                    (20000, 1032, (129, 300))])
def test_pairs_of_ctas(fp, n, k, ms):
    w = synth.weight_bf16(5, 0, 1, (n, k))
    for i, m in enumerate(ms):
        for epi in ((i, i + 2) if len(ms) > 2 else range(4)):
            _check(fp, m, n, k, epi % 4, w)


@pytest.mark.parametrize("wq,k", [(1, 16), (1, 4096), (1, 4112), (1, 8208), (2, 128), (2, 4096), (2, 4224), (3, 4224),
                                  (1, 272), (1, 1040), (1, 2064), (2, 256), (2, 1152), (2, 2048), (3, 256), (3, 1152)])
def test_expansion(fp, wq, k):
    m, n = 96, 264
    w = synth.weight_bf16(8, 0, 1, (n, k))
    x = synth.uniform_bf16(9, m, (m, k), -2.0, 2.0)
    out = empty(m * n * 4)
    codes = empty(n * k)
    scales, zeros = empty(n * max(1, k // 128), np.uint16), empty(n * max(1, k // 128), np.uint16)
    if wq == 3:
        order = np.random.default_rng(1).permutation(k).astype(np.int32)
        perm = dev(order)
        fp.fp_op_quantize_gptq4(ptr(dev(w)), n, k, ptr(perm), ptr(codes), ptr(scales), ptr(zeros))
        b = fp.fp_op_linear_gptq4_workspace_bytes(m, n, k)
        ws = empty(b)
        fp.fp_op_linear_gptq4(3, ptr(dev(x)), m, n, k, ptr(perm), ptr(codes), ptr(scales), ptr(zeros), None, ptr(out),
                              ptr(ws), b)
        wd = np.empty((n, k))
        wd[:, order] = quant.quantize_weight(np.ascontiguousarray(w[:, order]), 2)[1]
    else:
        fp.fp_op_quantize(wq, ptr(dev(w)), n, k, ptr(codes), ptr(scales), ptr(zeros))
        b = fp.fp_op_linear_workspace_bytes(wq, m, n, k)
        ws = empty(b)
        fp.fp_op_linear(wq, 3, ptr(dev(x)), m, n, k, ptr(codes), ptr(scales), ptr(zeros), None, ptr(out), ptr(ws), b)
        wd = quant.quantize_weight(w, wq)[1]
    if wq != 1:  # int4 weights enter as bf16((q - z) s)
        wd = quant.bf16_to_f32(synth.f32_to_bf16_bits(wd.astype(np.float32))).astype(np.float64)
    ref = quant.bf16_to_f32(x).astype(np.float64) @ wd.T
    assert rel_err(host(out, np.float32).reshape(m, n), ref) <= 2e-5
