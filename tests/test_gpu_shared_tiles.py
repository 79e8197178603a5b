"""The tcgen05 decode linears at 17 to 64 tokens where many CTAs share a row tile:
their sums are added several CTAs and 8 or 16 tokens at a time, so the numbers of CTAs
and tokens lie around those."""
import numpy as np
import pytest

import synth
from oracle import model as M
from oracle import quant
from tests.gpu_helpers import dev, empty, host, ptr, rel_err, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("wq", [0, 2])
@pytest.mark.parametrize("m", [17, 24, 31, 33, 48, 49, 64])
@pytest.mark.parametrize("n,k,epi", [(6400, 4096, 0), (3328, 8192, 3), (2056, 13824, 1), (4104, 8192, 2)])
def test_shared_row_tiles(fp, wq, m, n, k, epi):
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
