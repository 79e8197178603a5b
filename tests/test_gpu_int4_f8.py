"""The int4 decode linear with 8-bit operands (large matrices at up to 16
tokens, the largest SwiGLU at up to 32) against the oracle's dequantisation, on
sampled output columns; against the general decode path; and, beyond 16 tokens, an x
of a wide range, which the bf16 expansion takes over."""
import numpy as np
import pytest

import synth
from oracle import model as M
from oracle import quant
from tests.gpu_helpers import dev, empty, host, ptr, rel_err, torch_mod

pytestmark = pytest.mark.gpu

# One rounding of the result to bf16 (8 significant bits: half a unit of 1 is
# 2^-8); the sums are fp32 and x is carried to 2^-22 of the largest value of its group
# of 128, both far below.
TOL = 1.05 * 2.0 ** -8


@pytest.fixture(scope="module")
def fp():
    torch_mod()
    import paper_2501_13111_gb300 as fp

    return fp


def _weights(fp, n, k, seed, perm=None):
    w = empty(n * k, np.uint16)
    fp.fp_op_init_weights(ptr(w), n * k, seed, 3)
    codes, scales, zeros = empty(n * k // 2), empty(n * k // 128, np.uint16), empty(n * k // 128, np.uint16)
    if perm is None:
        fp.fp_op_quantize(2, ptr(w), n, k, ptr(codes), ptr(scales), ptr(zeros))
    else:
        fp.fp_op_quantize_gptq4(ptr(w), n, k, ptr(perm), ptr(codes), ptr(scales), ptr(zeros))
    return codes, scales, zeros


def _rows(n, k, seed, rows):
    """The oracle's dequantised weights of some rows of that matrix."""
    w = np.stack([synth.normal_bf16(seed, 3, int(r) * k, k) for r in rows])
    return quant.quantize_weight(w, 2)[1]


def _x(m, k, seed):
    """Rows with small elements, one large one in the last row, a zero row where there are several."""
    x = quant.bf16_to_f32(synth.uniform_bf16(seed, m, (m, k), -2.0, 2.0))
    x[:, 1::7] *= 2.0 ** -11
    x[-1, 5] = 300.0
    if m > 2:
        x[1] = 0.0
    return synth.f32_to_bf16_bits(x)


# ragged row tiles, an odd number of groups (a half item at each row's end), CTAs
# that cover whole tiles and tiles shared by several, every token tile
@pytest.mark.parametrize("m,n,k,epi", [
    (1, 4104, 4096, 0), (8, 12008, 1408, 1), (9, 4104, 4096, 1), (16, 8240, 2176, 2), (7, 140000, 128, 0),
    (16, 1200, 14080, 1), (5, 65664, 256, 2), (16, 65600, 4096, 2), (9, 67096, 4096, 2),
    (32, 65536, 4096, 2), (17, 57352, 4864, 2), (24, 21848, 12416, 2)])
def test_matches_oracle(fp, m, n, k, epi):
    codes, scales, zeros = _weights(fp, n, k, 9)
    x, nout = _x(m, k, 8), n // 2 if epi == 2 else n
    r = synth.uniform_bf16(7, m, (m, nout), -1.0, 1.0)
    rd = dev(r)
    ws_b = fp.fp_op_linear_workspace_bytes(2, m, n, k)
    ws = empty(ws_b)
    out = dev(r) if epi == 1 else empty(m * nout, np.uint16)  # the residual may be the output
    for _ in range(2 if epi != 1 else 1):  # the workspace serves a second call
        fp.fp_op_linear(2, epi, ptr(dev(x)), m, n, k, ptr(codes), ptr(scales), ptr(zeros),
                        ptr(out if epi == 1 else rd), ptr(out), ptr(ws), ws_b)
    got = quant.bf16_to_f32(host(out, np.uint16)).reshape(m, nout).astype(np.float64)
    assert not host(ws, np.uint8)[:16384].any()  # the tickets are zero again
    cols = np.unique(np.concatenate([[0, 1, nout - 1], np.random.default_rng(m).integers(0, nout, 60)]))
    xf = quant.bf16_to_f32(x).astype(np.float64)
    ref = xf @ _rows(n, k, 9, cols).T
    if epi == 1:
        ref = ref + quant.bf16_to_f32(r).astype(np.float64)[:, cols]
    elif epi == 2:
        ref = M.silu(ref) * (xf @ _rows(n, k, 9, cols + nout).T)
    for i in range(m):  # row by row: the row with the large element must not hide the others
        assert rel_err(got[i:i + 1][:, cols], ref[i:i + 1]) <= TOL, (i, rel_err(got[i:i + 1][:, cols], ref[i:i + 1]))


@pytest.mark.parametrize("m,epi", [(1, 0), (8, 1), (13, 2)])
def test_agrees_with_the_general_path(fp, m, epi):
    """Scales at an address that is not a multiple of 16 keep the mma.sync path."""
    n, k = 8200, 4096
    codes, scales, zeros = _weights(fp, n, k, 11)
    nout = n // 2 if epi == 2 else n
    x, r = dev(_x(m, k, 3)), dev(synth.uniform_bf16(4, m, (m, nout), -1.0, 1.0))
    shifted = dev(np.concatenate([np.zeros(1, np.uint16), host(scales, np.uint16)]))
    ws_b = fp.fp_op_linear_workspace_bytes(2, m, n, k)
    ws, res = empty(ws_b), []
    for sc in (ptr(scales), ptr(shifted) + 2):
        out = empty(m * nout, np.uint16)
        fp.fp_op_linear(2, epi, ptr(x), m, n, k, ptr(codes), sc, ptr(zeros), ptr(r), ptr(out), ptr(ws), ws_b)
        res.append(quant.bf16_to_f32(host(out, np.uint16)).reshape(m, nout).astype(np.float64))
    for a, b in zip(*res):
        assert rel_err(a[None], b[None]) <= 2 * TOL


@pytest.mark.parametrize("shift", [1, 2, 4])
@pytest.mark.parametrize("m,epi", [(17, 0), (40, 2), (64, 1)])
def test_scales_at_any_address_beyond_16_tokens(fp, m, epi, shift):
    """The tcgen05 expansion reads scales and zeros in up to 16 bytes: those at other
    addresses take the mma.sync path, whose weights are exact."""
    n, k = 520, 1024
    codes, scales, zeros = _weights(fp, n, k, 11)
    nout = n // 2 if epi == 2 else n
    x, r = _x(m, k, 3), synth.uniform_bf16(4, m, (m, nout), -1.0, 1.0)
    pad = np.zeros(shift, np.uint16)
    sd, zd = (dev(np.concatenate([pad, host(t, np.uint16)])) for t in (scales, zeros))
    ws_b = fp.fp_op_linear_workspace_bytes(2, m, n, k)
    ws = empty(ws_b)
    xf, wd = quant.bf16_to_f32(x).astype(np.float64), _rows(n, k, 11, range(n))
    ref = xf @ wd.T
    if epi == 1:
        ref = ref + quant.bf16_to_f32(r).astype(np.float64)
    elif epi == 2:
        ref = M.silu(ref[:, :nout]) * ref[:, nout:]
    for sc, ze in ((ptr(sd) + 2 * shift, ptr(zeros)), (ptr(scales), ptr(zd) + 2 * shift)):
        out = empty(m * nout, np.uint16)
        fp.fp_op_linear(2, epi, ptr(dev(x)), m, n, k, ptr(codes), sc, ze, ptr(dev(r)), ptr(out), ptr(ws), ws_b)
        got = quant.bf16_to_f32(host(out, np.uint16)).reshape(m, nout).astype(np.float64)
        for i in range(m):
            assert rel_err(got[i:i + 1], ref[i:i + 1]) <= TOL, (i, rel_err(got[i:i + 1], ref[i:i + 1]))


def test_gptq4_reads_x_through_the_act_order(fp):
    m, n, k = 6, 4608, 4096
    order = np.random.default_rng(5).permutation(k).astype(np.int32)
    perm = dev(order)
    codes, scales, zeros = _weights(fp, n, k, 12, perm)
    x = _x(m, k, 6)
    ws_b = max(fp.fp_op_linear_gptq4_workspace_bytes(m, n, k), fp.fp_op_linear_workspace_bytes(2, m, n, k))
    ws, err, a, b = empty(ws_b), empty(1, np.int32), empty(m * n, np.uint16), empty(m * n, np.uint16)
    fp.fp_op_linear_gptq4(0, ptr(dev(x)), m, n, k, ptr(perm), ptr(codes), ptr(scales), ptr(zeros), None, ptr(a),
                          ptr(ws), ws_b, ptr(err))
    fp.fp_op_linear(2, 0, ptr(dev(np.ascontiguousarray(x[:, order]))), m, n, k, ptr(codes), ptr(scales), ptr(zeros),
                    None, ptr(b), ptr(ws), ws_b)
    assert np.array_equal(host(a, np.uint16), host(b, np.uint16)) and host(err, np.int32)[0] == 0
    # an entry outside [0, K) reads as zero and is reported
    order[7] = k
    x0 = x.copy()
    lost = int(np.setdiff1d(np.arange(k), order)[0])
    x0[:, lost] = 0
    fp.fp_op_linear_gptq4(0, ptr(dev(x)), m, n, k, ptr(dev(order)), ptr(codes), ptr(scales), ptr(zeros), None, ptr(a),
                          ptr(ws), ws_b, ptr(err))
    order[7] = lost
    fp.fp_op_linear(2, 0, ptr(dev(np.ascontiguousarray(x0[:, order]))), m, n, k, ptr(codes), ptr(scales), ptr(zeros),
                    None, ptr(b), ptr(ws), ws_b)
    assert np.array_equal(host(a, np.uint16), host(b, np.uint16)) and host(err, np.int32)[0] == 1


def test_beyond_fp16_is_reported_as_on_the_general_path(fp):
    m, n, k = 4, 4608, 4096
    perm = dev(np.arange(k, dtype=np.int32))
    codes, scales, zeros = _weights(fp, n, k, 12)
    x = _x(m, k, 6)
    x[2, 100] = synth.f32_to_bf16_bits(np.array([7e4], np.float32))[0]
    ws_b = fp.fp_op_linear_gptq4_workspace_bytes(m, n, k)
    ws, err, out = empty(ws_b), empty(1, np.int32), empty(m * n, np.uint16)
    fp.fp_op_linear_gptq4(0, ptr(dev(x)), m, n, k, ptr(perm), ptr(codes), ptr(scales), ptr(zeros), None, ptr(out),
                          ptr(ws), ws_b, ptr(err))
    assert host(err, np.int32)[0] == 3


def _large_swiglu(fp, m, n, k, x, zeroed, cols, perm=None):
    """Rows of x through the SwiGLU of an n x k int4 matrix with the weights of channels
    `zeroed` zero: the result, and the oracle's weights of the gate and up rows of `cols`."""
    w = empty(n * k, np.uint16)
    fp.fp_op_init_weights(ptr(w), n * k, 9, 3)
    w.view(n, k)[:, zeroed] = 0
    codes, scales, zeros = empty(n * k // 2), empty(n * k // 128, np.uint16), empty(n * k // 128, np.uint16)
    nout = n // 2
    out, xd = empty(m * nout, np.uint16), dev(synth.f32_to_bf16_bits(x))
    if perm is None:
        fp.fp_op_quantize(2, ptr(w), n, k, ptr(codes), ptr(scales), ptr(zeros))
        ws_b = fp.fp_op_linear_workspace_bytes(2, m, n, k)
        ws = empty(ws_b)
        fp.fp_op_linear(2, 2, ptr(xd), m, n, k, ptr(codes), ptr(scales), ptr(zeros), None, ptr(out), ptr(ws), ws_b)
    else:
        pd = dev(perm)
        fp.fp_op_quantize_gptq4(ptr(w), n, k, ptr(pd), ptr(codes), ptr(scales), ptr(zeros))
        ws_b = fp.fp_op_linear_gptq4_workspace_bytes(m, n, k)
        ws = empty(ws_b)
        fp.fp_op_linear_gptq4(2, ptr(xd), m, n, k, ptr(pd), ptr(codes), ptr(scales), ptr(zeros), None, ptr(out), ptr(ws), ws_b)
    got = quant.bf16_to_f32(host(out, np.uint16)).reshape(m, nout).astype(np.float64)
    assert not host(ws, np.uint8)[:16384].any()  # the tickets are zero again
    rows = np.stack([synth.normal_bf16(9, 3, int(c) * k, k) for c in np.concatenate([cols, cols + nout])])
    rows[:, zeroed] = 0
    wd = quant.quantize_weight(rows if perm is None else np.ascontiguousarray(rows[:, perm]), 2)[1]
    if perm is not None:
        back = np.empty_like(wd)
        back[:, perm] = wd
        wd = back
    return got, wd[:len(cols)], wd[len(cols):]


def _rounded(wd):
    return quant.bf16_to_f32(synth.f32_to_bf16_bits(wd.astype(np.float32))).astype(np.float64)


@pytest.mark.parametrize("m,gptq", [(17, False), (32, False), (20, True)])
def test_beyond_16_tokens_x_keeps_the_range_of_bf16(fp, m, gptq):
    """The largest SwiGLU matrices at 17 tokens and more: an element of 2^18 whose weights
    are zero must not cost the row's other elements their bits, and an infinity is the
    infinity that its column's weights make of it."""
    n, k, big, inf = 65536, 4096, 1003, 2010
    x = quant.bf16_to_f32(synth.uniform_bf16(8, m, (m, k), -2.0, 2.0))
    x[:, big] = 2.0 ** 18
    x[m - 1, inf] = np.inf
    cols = np.unique(np.concatenate([[0, 1, n // 2 - 1], np.random.default_rng(m).integers(0, n // 2, 120)]))
    perm = np.random.default_rng(3).permutation(k).astype(np.int32) if gptq else None
    got, g, u = _large_swiglu(fp, m, n, k, x, [big], cols, perm)
    g, u = _rounded(g), _rounded(u)  # the expansion multiplies the weights rounded to bf16, x as it is
    xf = x[:m - 1].astype(np.float64)
    ref = M.silu(xf @ g.T) * (xf @ u.T)
    for i in range(m - 1):
        assert rel_err(got[i:i + 1][:, cols], ref[i:i + 1]) <= TOL + 1e-4, (i, rel_err(got[i:i + 1][:, cols], ref[i:i + 1]))
    both = (g[:, inf] > 0) & (u[:, inf] != 0)
    assert both.sum() > 10 and np.array_equal(got[m - 1, cols][both], np.sign(u[both, inf]) * np.inf)


@pytest.mark.parametrize("amp", [0.0, 300.0, 2.0 ** 14, 2.0 ** 15, 2.0 ** 16, 2.0 ** 17, 2.0 ** 24])
def test_beyond_16_tokens_around_the_line(fp, amp):
    """One token with a large element (its weights zero): up to where the two pieces lose as
    much as the bf16 rounding of the weights does they are kept, and every token's error stays
    at either path's: exact weights and x to 2^-10, or x exact and the weights to bf16."""
    m, n, k, big = 19, 65536, 4096, 1003
    x = quant.bf16_to_f32(synth.uniform_bf16(8, m, (m, k), -2.0, 2.0))
    x[m - 2, big] = amp
    cols = np.unique(np.random.default_rng(m).integers(0, n // 2, 150))
    got, g, u = _large_swiglu(fp, m, n, k, x, [big], cols)
    xf = x.astype(np.float64)
    ref = M.silu(xf @ g.T) * (xf @ u.T)
    # 2-norm: the result's rounding (2^-8 at most), and 2^-9.8 (2^-10 of the pieces) of each of
    # two factors; without the large element exact weights and x to 2^-22, the rounding alone
    bound = TOL if amp <= 300.0 else 2.0 ** -8 + 2 * 1.1 * 2.0 ** -9.8
    for i in range(m):
        e = np.linalg.norm(got[i, cols] - ref[i]) / np.linalg.norm(ref[i])
        assert e <= bound, (i, e)


def _dominated(fp, m, n, k, big, zeroed, amp):
    """Rows of small elements and one of `amp`, the weights of channels `zeroed` zero: the
    results of the 8-bit operands and of mma.sync (scales at an address that is not a
    multiple of 16), some columns, and the oracle's weights of those."""
    w = empty(n * k, np.uint16)
    fp.fp_op_init_weights(ptr(w), n * k, 9, 3)
    w.view(n, k)[:, zeroed] = 0
    codes, scales, zeros = empty(n * k // 2), empty(n * k // 128, np.uint16), empty(n * k // 128, np.uint16)
    fp.fp_op_quantize(2, ptr(w), n, k, ptr(codes), ptr(scales), ptr(zeros))
    shifted = dev(np.concatenate([np.zeros(1, np.uint16), host(scales, np.uint16)]))
    x = quant.bf16_to_f32(synth.uniform_bf16(8, m, (m, k), -0.1, 0.1))
    x[:, big] = amp
    ws_b = fp.fp_op_linear_workspace_bytes(2, m, n, k)
    ws, res = empty(ws_b), []
    for sc in (ptr(scales), ptr(shifted) + 2):
        out = empty(m * n, np.uint16)
        fp.fp_op_linear(2, 0, ptr(dev(synth.f32_to_bf16_bits(x))), m, n, k, ptr(codes), sc, ptr(zeros), None, ptr(out),
                        ptr(ws), ws_b)
        res.append(quant.bf16_to_f32(host(out, np.uint16)).reshape(m, n).astype(np.float64))
    cols = np.unique(np.random.default_rng(m).integers(0, n, 100))
    rows = np.stack([synth.normal_bf16(9, 3, int(c) * k, k) for c in cols])
    rows[:, zeroed] = 0
    return [r[:, cols] for r in res], x.astype(np.float64), quant.quantize_weight(rows, 2)[1]


@pytest.mark.parametrize("m,n,k", [(1, 4104, 4096), (8, 1160, 14592), (16, 4104, 4096), (4, 65536, 256)])
def test_a_large_element_costs_the_other_groups_nothing(fp, m, n, k):
    """The large element lies in a group whose weights are all zero (scale 0)."""
    (got, general), x, wd = _dominated(fp, m, n, k, 131, slice(128, 256), 30000.0)
    ref = x @ wd.T
    for i in range(m):
        assert rel_err(got[i:i + 1], ref[i:i + 1]) <= TOL, (i, rel_err(got[i:i + 1], ref[i:i + 1]))
        assert rel_err(general[i:i + 1], ref[i:i + 1]) <= TOL


@pytest.mark.parametrize("amp", [8000.0, 30000.0, 65280.0])
@pytest.mark.parametrize("m,n,k", [(1, 4104, 4096), (8, 1160, 14592), (16, 4104, 4096), (4, 65536, 256)])
def test_a_large_element_among_small_ones(fp, m, n, k, amp):
    """Its own weights are zero (the code is the zero point), its group's are not."""
    (got, general), x, wd = _dominated(fp, m, n, k, 131, [131], amp)
    ref = x @ wd.T
    group = wd[:, 128:256]
    # the group's x to 2^-22 of its largest; its fp32 sum of up to 15 amp s, then less z amp s: a unit in
    # the last place each (group's scale from its smallest step); the result's rounding to bf16
    step = np.array([np.diff(np.unique(r)).min() for r in group])
    bound = 2.0 ** -22 * amp * np.abs(group).sum(1) + 4 * 2.0 ** -23 * 15 * amp * step + 1.05 * 2.0 ** -8 * np.abs(ref)
    assert (np.abs(got - ref) <= bound + 2.0 ** -20 * np.abs(ref).max()).all()
    # and no further off than the operands of 16 bits, whose sums hold (1024 + q) amp
    norm = lambda y: np.linalg.norm(y - ref) / np.linalg.norm(ref)
    assert norm(got) <= norm(general), (norm(got), norm(general))
