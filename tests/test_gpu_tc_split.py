"""Tensor-core convolution on exact bf16 planes of the operands (fp32 and
qint8): channel counts that are no multiple of a block, of eight or of four,
ragged tiles, stride 2 on odd extents, several accumulator drains, residuals,
infinities, and a wait that runs out."""
import zlib

import numpy as np
import pytest

import synth
from oracle import q8
from oracle.net import run_layer
from paper_2110_06037_gb300 import SN_OPT_CHECK, SN_OPT_WAIT_LIMIT, SnError, _sn, build_graph, routine_name

from gpu_helpers import from_device, to_device
from test_gpu_q8 import F32, _out_scales, _ref_codes, codes_from_device, codes_to_device, conv_layer

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, k, s, pad, dil
    (1, 3, 9, 9, 16, 3, 1, 1, 1),       # channels padded from 3 to 8
    (2, 64, 8, 8, 64, 1, 1, 0, 1),      # plain, one K step
    (1, 132, 5, 7, 68, 1, 1, 0, 1),     # plain, ragged rows, K past a tile
    (2, 40, 9, 11, 66, 3, 1, 1, 1),     # K % 4 != 0: element stores
    (1, 72, 13, 7, 24, 5, 2, 2, 1),     # stride 2 on odd extents
    (3, 24, 12, 12, 8, 3, 1, 2, 2),     # dilation
    (1, 328, 7, 7, 136, 3, 1, 1, 1),    # 54 K steps: fourteen drains in fp32, four in qint8
    (5, 64, 28, 28, 200, 3, 1, 1, 1),   # more tiles than SMs: both accumulator buffers in turn
]


def tc_candidates(g, layer):
    t = g.cost_table()
    return [int(c) for c in np.flatnonzero(t["layer"] == layer) if " [tc " in g.candidate_desc(int(c))], t


def force(g, t, layer, c):
    path = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])]
    path[layer] = c
    g.set_path(path)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("residual", [False, True])
def test_f32(case, residual):
    """Error bound, per output, against fp64: a drain covers 128 products in 8
    accumulation steps of 16 products; allowing a truncated unit (2^-23) for
    each step and one for its alignment, 2^-19 of sum |x w| covers a drain, and
    2^-18 the round-to-nearest sums of the drains (at most 27, 2^-24 each) and the
    dropped plane products (2^-25) besides; bias and residual add two roundings
    of the result."""
    import torch
    N, C, H, W, K, k, s, pd, dil = case
    sch = ("f32", "nhwc")
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    layer = synth.conv(C, K, k, s, pd, act="none", d=dil)
    layer["weight"] = rng.standard_normal((K, C, k, k)).astype(np.float32)
    layer["bias"] = rng.standard_normal(K).astype(np.float32)
    other = dict(layer, weight=rng.standard_normal((K, C, k, k)).astype(np.float32))
    mag = run_layer(dict(layer, weight=np.abs(layer["weight"]), bias=np.zeros(K, np.float32)), [np.abs(x).astype(np.float64)])
    ref = run_layer(layer, [x.astype(np.float64)])
    net, li = [dict(layer, inputs=[-1])], 1
    if residual:  # another convolution of the same input joins the layer
        net, li = [dict(other, inputs=[-1]), dict(layer, inputs=[-1, 0])], 2
    g = build_graph(net, x.shape, sch, sch, [sch])
    cands, t = tc_candidates(g, li)
    assert cands
    for c in cands:
        force(g, t, li, c)
        xd = to_device(x, sch)
        if residual:  # the joined value is the library's own first layer
            g1 = build_graph(net[:1], x.shape, sch, sch, [sch])
            force(g1, g1.cost_table(), 1, int(np.flatnonzero(g1.cost_table()["layer"] == 1)[0]))
            want = ref + from_device(g1.run(xd), sch).reshape(ref.shape)
        else:
            want = ref
        y = g.run(xd)
        torch.cuda.synchronize()
        got = from_device(y, sch).reshape(want.shape)
        bound = 2.0 ** -18 * mag + 2.0 ** -22 * np.abs(want) + 2.0 ** -22
        assert (np.abs(got - want) <= bound).all(), (g.candidate_desc(c), float((np.abs(got - want) / bound).max()))
        # far below the bound in the mean: the error of an fp32 sum, not of a 16-bit one
        assert np.linalg.norm(got - want) <= 2e-6 * np.linalg.norm(want), g.candidate_desc(c)


@pytest.mark.parametrize("C,k", [(128, 1), (256, 1), (384, 1), (512, 1), (16, 3), (128, 3)])
def test_f32_operands_of_one_sign(C, k):
    """The tensor core's truncation does not cancel: of each of a drain's 8
    accumulation steps half a unit (2^-24) of the partial sum in the mean, and the
    partial sums come to 4.5 times the drain's, so 4.5 * 2^-24 of the result; from
    256 products on, no more than the fp32 multiply-adds of the direct kernel."""
    import torch
    sch = ("f32", "nhwc")
    rng = np.random.default_rng(C + k)
    x = np.abs(rng.standard_normal((2, C, 14, 14))).astype(np.float32)
    layer = synth.conv(C, 64, k, 1, k // 2, act="none")
    layer["weight"] = np.abs(rng.standard_normal((64, C, k, k))).astype(np.float32)
    layer["bias"] = np.zeros(64, np.float32)
    want = run_layer(layer, [x.astype(np.float64)])
    g = build_graph([dict(layer, inputs=[-1])], x.shape, sch, sch, [sch])
    cands, t = tc_candidates(g, 1)
    direct = [int(c) for c in np.flatnonzero(t["layer"] == 1) if routine_name(int(t["routine"][c])) == "conv2/direct"]
    err = []
    for c in direct + cands:
        force(g, t, 1, c)
        y = g.run(to_device(x, sch))
        torch.cuda.synchronize()
        err.append(np.linalg.norm(from_device(y, sch).reshape(want.shape) - want) / np.linalg.norm(want))
    assert max(err[1:]) <= 4.5 * 2.0 ** -24, err
    assert C * k * k < 256 or max(err[1:]) <= err[0], err


def test_f32_infinities_and_large_values():
    """Operands that the planes cannot carry give what plain fp32 arithmetic gives."""
    import torch
    sch = ("f32", "nhwc")
    rng = np.random.default_rng(3)
    x = rng.standard_normal((1, 16, 6, 6)).astype(np.float32)
    x[0, 3, 1, 1] = np.inf
    x[0, 5, 4, 4] = -np.inf
    x[0, 7, 4, 0] = np.nan
    x[0, 2, 0, 4] = 3.4e38  # above the largest bf16
    layer = synth.conv(16, 8, 3, 1, 1, act="none")
    layer["weight"] = (rng.standard_normal((8, 16, 3, 3)) * 0.25).astype(np.float32)
    layer["weight"][0, 3] = 0.5  # a plane of this weight is zero
    layer["bias"] = np.zeros(8, np.float32)
    g = build_graph([dict(layer, inputs=[-1])], x.shape, sch, sch, [sch])
    cands, t = tc_candidates(g, 1)
    direct = [int(c) for c in np.flatnonzero(t["layer"] == 1) if routine_name(int(t["routine"][c])) == "conv2/direct"]
    outs = []
    for c in direct + cands:
        force(g, t, 1, c)
        y = g.run(to_device(x, sch))
        torch.cuda.synchronize()
        outs.append(from_device(y, sch))
    for o in outs[1:]:
        assert np.array_equal(np.isnan(o), np.isnan(outs[0])) and np.array_equal(np.isinf(o), np.isinf(outs[0]))
        fine = np.isfinite(outs[0])
        assert np.array_equal(np.sign(o[~np.isnan(o)]), np.sign(outs[0][~np.isnan(outs[0])]))
        assert np.allclose(o[fine], outs[0][fine], rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("sx,sw", [(2.0 ** -120, 2.0 ** 100), (2.0 ** -130, 2.0 ** 30), (1e-36, 1.0), (2.0 ** -60, 2.0 ** -60),
                                   (2.0 ** 60, 2.0 ** 10), (2.0 ** 106, 2.0 ** -90), (1.0, 2.0 ** 105)])
def test_f32_tiny_and_huge_operands(sx, sw):
    """The bound of test_f32 for operands and results over fp32's whole range (a
    subnormal operand or result counts with its own spacing, 2^-149)."""
    import torch
    sch = ("f32", "nhwc")
    rng = np.random.default_rng(6)
    x = (rng.standard_normal((1, 40, 7, 7)).astype(np.float32) * np.float32(sx)).astype(np.float32)
    layer = synth.conv(40, 24, 3, 1, 1, act="none")
    layer["weight"] = (rng.standard_normal((24, 40, 3, 3)).astype(np.float32) * np.float32(sw)).astype(np.float32)
    layer["bias"] = np.zeros(24, np.float32)
    mag = run_layer(dict(layer, weight=np.abs(layer["weight"])), [np.abs(x).astype(np.float64)])
    want = run_layer(layer, [x.astype(np.float64)])
    g = build_graph([dict(layer, inputs=[-1])], x.shape, sch, sch, [sch])
    cands, t = tc_candidates(g, 1)
    for c in cands:
        force(g, t, 1, c)
        y = g.run(to_device(x, sch))
        torch.cuda.synchronize()
        got = from_device(y, sch).reshape(want.shape)
        bound = 2.0 ** -18 * mag + 2.0 ** -148
        assert (np.abs(got - want) <= bound).all(), (g.candidate_desc(c), float((np.abs(got - want) / bound).max()))


@pytest.mark.parametrize("case", [c for c in CASES if c[1] % 4 == 0 and c[4] % 4 == 0])
@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("out_dt", ["qi8", "f16", "f32"])
def test_q8_bit_exact(case, extreme, out_dt):
    import torch
    N, C, H, W, K, k, s, pd, dil = case
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    # another qint8 layer of the same input joins, as a shortcut does
    short = conv_layer(rng, C, K, k, s, pd, dil, act="none")
    layer = dict(conv_layer(rng, C, K, k, s, pd, dil, act="relu"), inputs=[-1, 0])
    q_in = rng.integers(-127, 128, (N, C, H, W)).astype(np.int8)
    if extreme:  # every product 127 * 127: the sums come closest to 2^24
        q_in[:] = 127
        layer["weight"][:] = np.abs(layer["weight"]).max()
    s_in = F32(0.02)
    scales = _out_scales([short, layer], q_in, s_in)
    lam = [("qi8", "nhwc")] + ([(out_dt, "nhwc")] if out_dt != "qi8" else [])
    g = build_graph([short, layer], q_in.shape, ("qi8", "nhwc"), (out_dt, "nhwc"), lam)
    for i, v in zip((-1, 0, 1), [s_in] + scales):
        g.set_qscale(i, float(v))
    cands, t = tc_candidates(g, 2)
    cands = [c for c in cands if t["schema"][c] == 0 and t["out_schema"][c] == len(lam) - 1]
    assert cands
    first = [int(c) for c in np.flatnonzero(t["layer"] == 1) if t["schema"][c] == 0 and t["out_schema"][c] == 0][0]
    q_s = q8.run_layer(short, [q_in], [s_in], scales[0])
    want = q8.run_layer(layer, [q_in, q_s], [s_in, scales[0]], scales[1],
                        **({} if out_dt == "qi8" else {"out_dtype": out_dt}))
    for c in cands:
        path = [int(np.flatnonzero(t["layer"] == 0)[0]), first, c, int(np.flatnonzero(t["layer"] == 3)[0])]
        g.set_path(path)
        y = g.run(codes_to_device(q_in, "nhwc"))
        torch.cuda.synchronize()
        got = codes_from_device(y, "nhwc") if out_dt == "qi8" else from_device(y, (out_dt, "nhwc"))
        assert np.array_equal(got.reshape(want.shape), want.astype(got.dtype)), g.candidate_desc(c)


def test_q8_refuses_an_infinite_scale_in_every_variant():
    """Calibration of a layer whose sums overflow leaves an infinite scale: every
    way to run the layer says so (zeros with a good status are no answer)."""
    rng = np.random.default_rng(8)
    sch = ("f32", "nhwc")
    layers = [dict(conv_layer(rng, 16, 16, 1, 1, 0, 1), inputs=[-1]), dict(conv_layer(rng, 16, 16, 1, 1, 0, 1), inputs=[0])]
    layers[0]["weight"][:] = 3e38
    g = build_graph(layers, (1, 16, 8, 8), sch, sch, [sch, ("qi8", "nhwc")])
    t = g.cost_table()
    t["cost"] = np.where(t["routine"] == 0, 0, 1).astype(np.int64)
    t["adapt"] = np.where(np.eye(t["adapt"].shape[1], dtype=bool), 0, 1).astype(np.int64) * np.ones_like(t["adapt"])
    g.set_cost_table(t)
    xd = to_device(np.ones((1, 16, 8, 8), np.float32), sch)
    g.calibrate(xd)
    assert np.isfinite(g.get_qscale(-1)) and g.get_qscale(0) == np.inf

    def of(layer, out):
        return [int(c) for c in np.flatnonzero((t["layer"] == layer) & (t["schema"] == 1) & (t["out_schema"] == out))]

    io = [int(np.flatnonzero(t["layer"] == i)[0]) for i in (0, 3)]
    last = [c for c in of(2, 0) if " [tc " in g.candidate_desc(c)][0]  # codes in, fp32 out: no adapt reads the scale
    names = {c: g.candidate_desc(c) for c in of(1, 1)}
    assert sum("dp4a" in d for d in names.values()) > 1 and any("direct" in d for d in names.values())
    for c, d in names.items():
        g.set_path([io[0], c, last, io[1]])
        with pytest.raises(SnError):
            g.run(xd)
            pytest.fail(d)


def test_expired_wait_reports_timeout_and_recovers():
    import torch
    x, layers = synth.single_conv(2, 14, 64, 128, 3, 1)
    sch = ("f32", "nhwc")
    g = build_graph(layers, x.shape, sch, sch, [sch])
    cands, t = tc_candidates(g, 1)
    force(g, t, 1, cands[0])
    g.set_option(SN_OPT_CHECK, 1)
    xd = to_device(x, sch)
    y0 = g.run(xd).clone()
    g.set_option(SN_OPT_WAIT_LIMIT, 1)
    with pytest.raises(SnError) as e:
        g.run(xd)
    assert e.value.status == _sn.SN_ETIMEOUT
    g.set_option(SN_OPT_WAIT_LIMIT, 0)
    y1 = g.run(xd)
    torch.cuda.synchronize()
    assert torch.equal(y0, y1)
