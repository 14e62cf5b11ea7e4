"""The vectorised pooling, scale and dense kernels (float and qint8) and the
qint8 depthwise kernel at the sizes where their splits can go wrong: fewer
pixels or features than a block has slices, a channel count that ends inside a
block's vectors, column counts that are no multiple of a thread's columns, one
and several images per warp, and sizes that fall back to the general kernels."""
import zlib

import numpy as np
import pytest

import synth
from oracle.net import run_layer
from paper_2110_06037_gb300 import build_graph

from gpu_helpers import TOL, from_device, maxrel, stored_values, to_device
from test_gpu_q8 import F32, _out_scales, _ref_codes, conv_layer, run_q8

pytestmark = pytest.mark.gpu


def run_float(layers, x, schema):
    import torch
    g = build_graph(layers, x.shape, schema, schema, [schema])
    t = g.cost_table()
    g.set_path([int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])])
    y = g.run(to_device(x, schema))
    torch.cuda.synchronize()
    return from_device(y, schema)


@pytest.mark.parametrize("n,c,h,w", [(1, 8, 1, 1), (2, 72, 3, 5), (3, 120, 28, 28), (1, 200, 31, 33), (2, 10, 9, 9)])
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
def test_gap_then_scale(n, c, h, w, dt):
    rng = np.random.default_rng(zlib.crc32(repr((n, c, h, w, dt)).encode()))
    x = rng.standard_normal((n, c, h, w)).astype(np.float32)
    xs = stored_values(x, dt)
    net = [dict(synth.gap(), inputs=[-1])]
    pooled = run_layer(net[0], [xs], dt)
    assert maxrel(run_float(net, x, (dt, "nhwc")), pooled) <= TOL[dt]
    net.append(dict(synth.mul(act="none"), inputs=[-1, 0]))
    assert maxrel(run_float(net, x, (dt, "nhwc")), run_layer(net[1], [xs, pooled], dt)) <= TOL[dt]


@pytest.mark.parametrize("n,i,o", [(1, 8, 1), (1, 1032, 9), (6, 1024, 520), (9, 24, 120), (3, 520, 1001), (33, 264, 333), (2, 100, 7)])
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
def test_dense(n, i, o, dt):
    rng = np.random.default_rng(zlib.crc32(repr((n, i, o, dt)).encode()))
    x = rng.standard_normal((n, i, 1, 1)).astype(np.float32)
    layer = dict(synth.dense(i, o, act="hsigmoid"), inputs=[-1])
    layer["weight"] = (rng.standard_normal((o, i)) / np.sqrt(i)).astype(np.float32)
    layer["bias"] = rng.standard_normal(o).astype(np.float32)
    ref = run_layer(layer, [stored_values(x, dt)], dt)
    assert maxrel(run_float([layer], x, (dt, "nhwc")), ref) <= TOL[dt]


@pytest.mark.parametrize("ks,st", [(3, 1), (3, 2), (5, 1), (5, 2)])
@pytest.mark.parametrize("c,h,w", [(4, 1, 1), (20, 7, 5), (36, 9, 18), (6, 8, 8)])
@pytest.mark.parametrize("act", ["relu6", "hswish"])
def test_q8_depthwise_vectors(ks, st, c, h, w, act):
    rng = np.random.default_rng(zlib.crc32(repr((ks, st, c, h, w)).encode()))
    layer = conv_layer(rng, c, c, ks, st, ks // 2, act=act, dw=True)
    q_in = rng.integers(-127, 128, (3, c, h, w)).astype(np.int8)
    s_in = F32(0.05)
    scales = _out_scales([layer], q_in, s_in)
    got, _ = run_q8([layer], q_in, s_in, scales, "nhwc", ["dwconv2/direct"])
    assert np.array_equal(got, _ref_codes([layer], q_in, s_in, scales))


@pytest.mark.parametrize("n,c,h,w", [(1, 4, 1, 1), (2, 36, 3, 5), (3, 48, 27, 29), (2, 6, 9, 9)])
def test_q8_pool_gap_add_mul_vectors(n, c, h, w):
    rng = np.random.default_rng(zlib.crc32(repr((n, c, h, w)).encode()))
    q_in = rng.integers(-127, 128, (n, c, h, w)).astype(np.int8)
    s_in = F32(0.03)
    nets = [
        [{"type": "maxpool", "inputs": [-1], "params": dict(kh=3, kw=3, sh=2, sw=2, ph=1, pw=1)}],
        [{"type": "gap", "inputs": [-1]}],
        [{"type": "add", "inputs": [-1, -1], "params": dict(act="hswish")}],
        [{"type": "gap", "inputs": [-1]}, {"type": "mul", "inputs": [-1, 0], "params": dict(act="none")}],
    ]
    for layers in nets:
        scales = _out_scales(layers, q_in, s_in)
        got, _ = run_q8(layers, q_in, s_in, scales, "nhwc", [])
        assert np.array_equal(got, _ref_codes(layers, q_in, s_in, scales)), layers[-1]["type"]


@pytest.mark.parametrize("n,i,o", [(1, 4, 1), (8, 168, 672), (3, 1032, 1024), (9, 2048, 520), (40, 20, 2000)])
def test_q8_dense_words(n, i, o):
    rng = np.random.default_rng(n * 1000 + i)
    layer = {"type": "dense", "inputs": [-1], "params": dict(in_features=i, out_features=o, act="hsigmoid"),
             "weight": (rng.standard_normal((o, i)) / np.sqrt(i)).astype(F32),
             "bias": rng.standard_normal(o).astype(F32)}
    q_in = rng.integers(-127, 128, (n, i, 1, 1)).astype(np.int8)
    s_in = F32(0.01)
    scales = _out_scales([layer], q_in, s_in)
    got, _ = run_q8([layer], q_in, s_in, scales, "nhwc", ["dense/simt"])
    assert np.array_equal(got, _ref_codes([layer], q_in, s_in, scales))


@pytest.mark.parametrize("ks,st,dil", [(5, 1, 1), (5, 2, 1), (3, 1, 1), (3, 2, 1), (7, 1, 1)])
@pytest.mark.parametrize("c,h,w", [(8, 1, 1), (24, 7, 5), (40, 9, 18)])
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
def test_depthwise_windows(ks, st, dil, c, h, w, dt):
    rng = np.random.default_rng(zlib.crc32(repr((ks, st, c, h, w, dt)).encode()))
    x = rng.standard_normal((3, c, h, w)).astype(np.float32)
    layer = dict(synth.dwconv(c, ks, st, act="hswish"), inputs=[-1])
    layer["weight"] = (rng.standard_normal((c, 1, ks, ks)) / ks).astype(np.float32)
    layer["bias"] = rng.standard_normal(c).astype(np.float32)
    ref = run_layer(layer, [stored_values(x, dt)], dt)
    assert maxrel(run_float([layer], x, (dt, "nhwc")), ref) <= TOL[dt]


@pytest.mark.parametrize("ks,st,pd", [(3, 2, 1), (3, 2, 0), (2, 2, 0), (2, 2, 1), (3, 1, 1)])
@pytest.mark.parametrize("n,c,h,w", [(1, 8, 3, 3), (2, 24, 7, 9), (3, 264, 10, 35), (8, 64, 113, 112)])
@pytest.mark.parametrize("dt", ["f32", "f16", "bf16"])
def test_maxpool_windows(ks, st, pd, n, c, h, w, dt):
    # one row a thread and (the last size) four, the last group cut short;
    # windows over every edge, infinities and a NaN (which the maximum passes over)
    rng = np.random.default_rng(ks + h)
    x = rng.standard_normal((n, c, h, w)).astype(np.float32)
    x[0, 0] = -np.inf
    x[-1, 1, 0, 0] = np.inf
    x[0, 2, 1, 1] = np.nan
    net = [{"type": "maxpool", "inputs": [-1], "params": dict(kh=ks, kw=ks, sh=st, sw=st, ph=pd, pw=pd)}]
    xs = stored_values(x, dt)
    ref = run_layer(net[0], [np.where(np.isnan(xs), -np.inf, xs)], dt)
    np.testing.assert_array_equal(run_float(net, x, (dt, "nhwc")), ref)


@pytest.mark.parametrize("c,w", [(264, 37), (1032, 5), (8, 130)])
@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_depthwise_general_path_rows(c, w, dt):
    """Blocks that stay in a row: rows of several blocks, the last one partly idle, and short rows."""
    rng = np.random.default_rng(c + w)
    x = rng.standard_normal((2, c, 4, w)).astype(np.float32)
    layer = dict(synth.dwconv(c, 7, 1, act="relu6"), inputs=[-1])
    layer["weight"] = (rng.standard_normal((c, 1, 7, 7)) / 7).astype(np.float32)
    layer["bias"] = rng.standard_normal(c).astype(np.float32)
    ref = run_layer(layer, [stored_values(x, dt)], dt)
    assert maxrel(run_float([layer], x, (dt, "nhwc")), ref) <= TOL[dt]
