"""int8 linears at 17 to 32 tokens on the tcgen05 kernel: ragged rows and tokens around
the rule's edges (2^24 weights, K 3072, a K that is a power of two, SwiGLU, 33 tokens), and
the report of an x beyond the fp16 range, which the mma.sync kernel they came from makes."""
import numpy as np
import pytest

import synth
from oracle import model as M
from tests.gpu_helpers import arch_dict, check_decode_linear, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("m,n,k,epi", [
    (17, 4104, 5376, 1), (24, 3336, 5120, 0), (32, 1544, 11008, 3), (31, 8200, 5504, 1), (33, 4104, 5376, 1),
    (20, 8328, 5504, 0), (18, 4104, 8192, 0), (32, 6152, 5376, 2), (16, 4104, 5376, 1),
    (17, 5464, 3072, 0), (32, 5456, 3072, 1), (24, 16392, 3200, 3), (20, 6152, 2944, 0), (31, 1032, 16256, 1)])
def test_int8_linear(fp, m, n, k, epi):
    check_decode_linear(fp, 1, m, n, k, epi)


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
