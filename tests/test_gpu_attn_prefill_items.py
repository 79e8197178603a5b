"""Prefill attention where its work items can go wrong: prompts around one and two
tiles of 128 rows, KV groups of even and odd size (pairs of heads, pairs of row
tiles, single tiles with their keys cut in two), few items and many (one block of heads and several), both caches."""
import numpy as np
import pytest

from oracle import model as M
from oracle import quant
from tests.gpu_helpers import TAU, dev, empty, host, ptr, rel_err, torch_mod
from tests.test_gpu_ops import Cache
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


@pytest.mark.parametrize("kvq", [0, 1])
@pytest.mark.parametrize("B,H,Hkv,S", [
    (2, 3, 3, 128), (2, 3, 3, 129), (1, 3, 1, 256), (2, 3, 1, 257), (1, 6, 6, 385),  # odd groups, ragged second tiles
    (2, 4, 2, 128), (3, 4, 2, 255), (1, 8, 2, 641),                                   # pairs of heads
    (20, 16, 16, 300), (41, 32, 4, 129), (64, 32, 32, 257), (300, 32, 4, 130),        # several rounds of SMs, many
    (1, 8, 2, 300), (1, 2, 2, 1153), (1, 40, 40, 520), (3, 8, 8, 1024),               # a query tile's keys cut in two
    (76, 4, 2, 128), (77, 4, 2, 100), (229, 4, 2, 33), (40, 64, 8, 128), (310, 3, 3, 17)])  # one tile: both kernels
def test_work_items(fp, kvq, B, H, Hkv, S):
    hd = 128
    c = Cache(fp, kvq, B, S + 7, Hkv, hd, seed=S + H + kvq)
    width = (H + 2 * Hkv) * hd  # q read in place from the fused rows
    q = synth.uniform_bf16(41, S, (B * S, width), -2, 2)
    out, err = empty(B * S * H * hd, np.uint16), empty(1, np.int32)
    fp.fp_op_attention_prefill(ptr(dev(q)), width, B, S, H, c.view, ptr(out), ptr(err))
    got = quant.bf16_to_f32(host(out, np.uint16)).reshape(B, S, H, hd)
    assert host(err, np.int32)[0] == 0
    qf = quant.bf16_to_f32(q).astype(np.float64).reshape(B, S, -1, hd)
    for b in sorted({0, B // 2, B - 1}):
        k, v = c.seq("k", b, S), c.seq("v", b, S)
        for h in sorted({0, 1, H // 2, H - 1}):
            g = h // (H // Hkv)
            ref = M.attention(qf[b][:, h:h + 1], np.arange(S), k[:, g:g + 1], v[:, g:g + 1])
            assert rel_err(got[b][:, h:h + 1], ref) <= TAU[0] / 2, (b, h, rel_err(got[b][:, h:h + 1], ref))


@pytest.mark.parametrize("kvq", [0, 1])
@pytest.mark.parametrize("S", [100, 700])
def test_growing_scores_move_the_reference(fp, kvq, S):
    """Scores that rise along the keys by far more than the 2^8 the running maximum
    may lag behind: the output is rescaled again and again, and stays exact."""
    B, H, Hkv, hd = 1, 4, 2, 128
    c = Cache(fp, kvq, B, S, Hkv, hd, seed=5)
    q = synth.uniform_bf16(3, S, (B * S, H * hd), 0.5, 1.0)
    ramp = np.linspace(0.0, 4.0, S)
    pages, slot = c.table[0, np.arange(S) // 16], np.arange(S) % 16
    if kvq == 0:
        kf = quant.bf16_to_f32(c.k)
        kf[pages, :, slot] = np.abs(kf[pages, :, slot]) * ramp[:, None, None]
        c.k = synth.f32_to_bf16_bits(kf.astype(np.float32))
        c.kd.copy_(dev(c.k))
    else:
        c.k = np.abs(c.k)
        c.kd.copy_(dev(c.k))
        c.ksc[pages, :, slot] = (0.02 * ramp[:, None]).astype(np.float32)
        c.ks.copy_(dev(c.ksc))
    out = empty(B * S * H * hd, np.uint16)
    fp.fp_op_attention_prefill(ptr(dev(q)), H * hd, B, S, H, c.view, ptr(out))
    got = quant.bf16_to_f32(host(out, np.uint16)).reshape(S, H, hd)
    ref = M.attention(quant.bf16_to_f32(q).astype(np.float64).reshape(S, H, hd), np.arange(S), c.seq("k", 0, S),
                      c.seq("v", 0, S))
    assert np.isfinite(got).all() and rel_err(got, ref) <= TAU[0] / 2, rel_err(got, ref)
