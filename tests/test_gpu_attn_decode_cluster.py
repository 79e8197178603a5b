"""Decode attention with a cluster of CTAs per (sequence, KV head): sequences shorter
than the cluster has CTAs or the blocks that it shares out, lengths around those
blocks, clusters of two to eight, both kernels; and splits through the workspace where
the context is too long for eight CTAs or the clusters would not all fit at once."""
import numpy as np
import pytest

import synth
from oracle import model as M
from oracle import quant
from tests.gpu_helpers import TAU, dev, empty, host, ptr, rel_err, torch_mod
from tests.test_gpu_ops import Cache

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


def _check(fp, kvq, hd, H, Hkv, lens, T):
    B = len(lens)
    c = Cache(fp, kvq, B, T, Hkv, hd, seed=T + H + kvq)
    q = synth.uniform_bf16(33, B, (B, H * hd), -2, 2)
    out, err = empty(B * H * hd, np.uint16), empty(1, np.int32)
    wsb = fp.fp_op_attention_decode_workspace_bytes(B, H, hd, T)
    ws = empty(wsb)
    fp.fp_op_attention_decode(ptr(dev(q)), H * hd, B, H, c.view, ptr(dev(np.array(lens, np.int32))), T, ptr(out),
                              ptr(ws), wsb, ptr(err))
    got = quant.bf16_to_f32(host(out, np.uint16)).reshape(B, H, hd)
    assert host(err, np.int32)[0] == 0
    qf = quant.bf16_to_f32(q).astype(np.float64).reshape(B, H, hd)
    for b, L in enumerate(lens):
        ref = M.attention(qf[b][None], np.array([L - 1]), c.seq("k", b, L), c.seq("v", b, L))[0]
        assert rel_err(got[b], ref) <= TAU[0] / 2, (b, rel_err(got[b], ref))
    return ws


@pytest.mark.parametrize("kvq,hd", [(0, 64), (0, 128), (1, 64), (1, 128)])
@pytest.mark.parametrize("H,Hkv,lens,T", [
    (8, 8, [1], 130), (8, 1, [64, 65], 130), (16, 4, [1, 2, 63, 64, 65, 500], 512),  # ranks without a block
    (2, 2, [16, 17, 511, 512, 513], 520), (64, 8, [300, 1, 229], 300),
    (16, 8, [7, 1290, 640], 1300), (4, 4, [2400, 2561], 2561),                       # eight CTAs for more splits
    (32, 32, [130, 200, 3, 128], 200), (8, 4, [700] * 6 + [90] * 6, 700)])           # two CTAs; five or six
def test_cluster_ranges(fp, kvq, hd, H, Hkv, lens, T):
    _check(fp, kvq, hd, H, Hkv, lens, T)


@pytest.mark.parametrize("kvq,hd,H,Hkv,lens,T", [
    (1, 128, 64, 8, [5000], 5000), (1, 128, 8, 8, [5000, 4990], 5003), (1, 128, 4, 2, [1, 6000], 6000),  # page streaming
    (0, 128, 16, 2, [3000, 17], 3000), (0, 64, 8, 8, [4100], 4100), (1, 64, 16, 4, [3001, 64], 3001),    # tile kernel
    (0, 128, 32, 8, [224] * 30 + [1] + [150] * 29, 224), (1, 128, 32, 32, [420] * 10 + [5] + [64] * 10, 420)])
def test_splits_through_the_workspace(fp, kvq, hd, H, Hkv, lens, T):
    assert host(_check(fp, kvq, hd, H, Hkv, lens, T), np.uint8).any()  # the partials


def test_lengths_past_the_table_are_clipped_and_reported(fp):
    B, H, Hkv, hd, T = 2, 8, 2, 128, 512
    c = Cache(fp, 0, B, T, Hkv, hd, seed=3)
    q = synth.uniform_bf16(34, B, (B, H * hd), -2, 2)
    wsb = fp.fp_op_attention_decode_workspace_bytes(B, H, hd, T)
    ws, outs, errs = empty(wsb), [], []
    for lens in ([T, 100], [T + 9, 100]):
        out, err = empty(B * H * hd, np.uint16), empty(1, np.int32)
        fp.fp_op_attention_decode(ptr(dev(q)), H * hd, B, H, c.view, ptr(dev(np.array(lens, np.int32))), T, ptr(out),
                                  ptr(ws), wsb, ptr(err))
        outs.append(host(out, np.uint16))
        errs.append(host(err, np.int32)[0])
    assert errs == [0, 1] and np.array_equal(outs[0], outs[1])
