"""int8 linears at 17 to 32 tokens on the tcgen05 kernel: ragged rows and tokens around
the rule's edges (2^24 weights, K 3072, a K that is a power of two, SwiGLU, 33 tokens), and
the report of an x beyond the fp16 range, which the mma.sync kernel they came from makes."""
import numpy as np
import pytest

import synth
from oracle import model as M
from oracle import quant
from tests.gpu_helpers import arch_dict, dev, empty, host, ptr, rel_err, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("wq", [1])
@pytest.mark.parametrize("m,n,k,epi", [
    (17, 4104, 5376, 1), (24, 3336, 5120, 0), (32, 1544, 11008, 3), (31, 8200, 5504, 1), (33, 4104, 5376, 1),
    (20, 8328, 5504, 0), (18, 4104, 8192, 0), (32, 6152, 5376, 2), (16, 4104, 5376, 1),
    (17, 5464, 3072, 0), (32, 5456, 3072, 1), (24, 16392, 3200, 3), (20, 6152, 2944, 0), (31, 1032, 16256, 1)])
def test_int8_linear(fp, wq, m, n, k, epi):
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
    assert rel_err(got.reshape(m, nout), ref) <= (1e-4 if epi == 3 else 1.05 * 2.0 ** -8 + 1e-4)


def test_x_beyond_fp16_is_reported(fp):
    """A norm gain of 300 leaves the inputs of the first linears within the fp16 range and
    takes the down projection's, products of two sums of that size, beyond it."""
    arch = M.Arch(1, 3328, 26, 26, 128, 5376, 32000)
    batch = 17
    h = fp.fp_create(arch_dict(arch), 1, 0, batch, 32, seed=9)
    try:
        toks = synth.tokens(9, batch * 4, arch.vocab).reshape(batch, 4)
        step = synth.tokens(10, batch, arch.vocab)
        fp.fp_prefill(h, toks)
        fp.fp_decode_step(h, step)
        fp.fp_set_weight(h, 0, fp.FP_T_FFN_NORM, synth.f32_to_bf16_bits(np.full(arch.hidden, 300.0, np.float32)))
        with pytest.raises(fp.FPError) as e:
            for _ in range(3):
                fp.fp_decode_step(h, step)
        assert e.value.code == fp.FP_ERR_DEVICE_ASSERT and "fp16" in str(e.value)
        fp.fp_set_weight(h, 0, fp.FP_T_FFN_NORM, synth.f32_to_bf16_bits(np.ones(arch.hidden, np.float32)))
        fp.fp_prefill(h, toks)
        fp.fp_decode_step(h, step)
    finally:
        fp.fp_destroy(h)
