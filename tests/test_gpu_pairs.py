"""A pointwise convolution and its depthwise reader in one launch: equal bit for
bit to the two launches, over kernels, strides, types, activations, channel
counts that end inside a block or a slice, maps of one tile and of several,
bands of one row and whole maps; only where the depthwise layer alone reads the
convolution; buffers of a longer net; a wait that runs out."""
import zlib

import numpy as np
import pytest

import synth
from oracle.net import run_net
from paper_2110_06037_gb300 import (SN_OPT_CHECK, SN_OPT_PAIR, SN_OPT_WAIT_LIMIT, SnError, _sn, build_graph,
                                    routine_name)

from gpu_helpers import TOL, from_device, maxrel, to_device

pytestmark = pytest.mark.gpu


def weights(layers, seed):
    rng = np.random.default_rng(seed)
    for l in layers:
        p = l["params"]
        if l["type"] in ("conv2", "dwconv2"):
            shp = (p["c_out"], p["c_in"] // p["groups"], p["kh"], p["kw"])
            l["weight"] = (rng.standard_normal(shp) * np.sqrt(2.0 / np.prod(shp[1:]))).astype(np.float32)
            l["bias"] = rng.standard_normal(p["c_out"]).astype(np.float32)
    return layers


def graph(layers, x, sch):
    g = build_graph(layers, x.shape, sch, sch, [sch])
    t = g.cost_table()
    path = []
    for i in range(t["n_layers"]):
        idx = np.flatnonzero(t["layer"] == i)
        tc = [int(c) for c in idx if routine_name(int(t["routine"][c])) == "conv2/igemm_tc"]
        path.append(tc[0] if tc else int(idx[0]))
    g.set_path(path)
    return g


CASES = [
    # N, C, H, W, E, k, s
    (1, 8, 1, 1, 8, 3, 1),
    (1, 24, 14, 14, 72, 3, 1),     # channels past a slice
    (2, 96, 7, 7, 576, 3, 1),      # two blocks of input channels
    (1, 160, 9, 11, 200, 5, 1),
    (3, 16, 28, 28, 64, 3, 2),
    (2, 40, 15, 27, 120, 5, 2),    # odd extents
    (1, 16, 112, 112, 96, 3, 2),   # bands of a row or two, three tiles and more
    (1, 24, 40, 130, 80, 3, 1),    # a row takes more than a tile
    (32, 32, 28, 28, 192, 3, 1),   # close to all the CTAs the GPU holds
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("acts", [("relu6", "relu6"), ("hswish", "relu"), ("none", "hswish")])
def test_pair_equals_two_launches(case, dt, acts):
    import torch
    N, C, H, W, E, k, s = case
    sch = (dt, "nhwc")
    layers = weights([dict(synth.conv(C, E, 1, act=acts[0]), inputs=[-1]),
                      dict(synth.dwconv(E, k, s, act=acts[1]), inputs=[0])], zlib.crc32(repr(case).encode()))
    x = np.random.default_rng(1).standard_normal((N, C, H, W)).astype(np.float32)
    g = graph(layers, x, sch)
    xd = to_device(x, sch)
    assert g.plan_stats() == (2, 1)
    y = g.run(xd).clone()
    g.set_option(SN_OPT_PAIR, 0)
    assert g.plan_stats() == (2, 2)
    y2 = g.run(xd)
    torch.cuda.synchronize()
    assert torch.equal(y.view(torch.int16), y2.view(torch.int16))
    if N * H * W * E < 1 << 18:
        assert maxrel(from_device(y, sch), run_net(layers, x, dt)) <= TOL[dt]


def test_pair_within_a_net():
    """Inverted residual blocks: the pair's input lives on as the residual, and
    buffers are shared; a convolution with a second reader stays on its own."""
    import torch
    sch = ("f16", "nhwc")
    layers = weights([
        dict(synth.conv(16, 96, 1, act="relu6"), inputs=[-1]),
        dict(synth.dwconv(96, 3, 1), inputs=[0]),
        dict(synth.conv(96, 16, 1, act="none"), inputs=[1, -1]),   # + residual
        dict(synth.conv(16, 96, 1, act="relu6"), inputs=[2]),
        dict(synth.dwconv(96, 5, 1), inputs=[3]),
        dict(synth.conv(96, 96, 1, act="none"), inputs=[4, 3]),    # reads the expanded map again
    ], 5)
    x = np.random.default_rng(2).standard_normal((2, 16, 20, 20)).astype(np.float32)
    g = graph(layers, x, sch)
    assert g.plan_stats()[1] == 5  # the first pair only
    y = g.run(to_device(x, sch)).clone()
    g.set_option(SN_OPT_PAIR, 0)
    y2 = g.run(to_device(x, sch))
    torch.cuda.synchronize()
    assert torch.equal(y, y2)
    assert maxrel(from_device(y, sch), run_net(layers, x, "f16")) <= TOL["f16"]


def test_unaligned_output_and_expired_wait():
    import torch
    sch = ("bf16", "nhwc")
    layers = weights([dict(synth.conv(16, 64, 1), inputs=[-1]), dict(synth.dwconv(64, 3, 1), inputs=[0])], 7)
    x = np.random.default_rng(3).standard_normal((1, 16, 12, 12)).astype(np.float32)
    g = graph(layers, x, sch)
    xd = to_device(x, sch)
    y = g.run(xd).clone()
    flat = torch.zeros(y.numel() + 1, dtype=torch.bfloat16, device="cuda")
    g.run(xd, flat[1:].view(y.shape))
    torch.cuda.synchronize()
    assert torch.equal(flat[1:].view(y.shape), y)
    g.set_option(SN_OPT_CHECK, 1)
    g.set_option(SN_OPT_WAIT_LIMIT, 1)
    with pytest.raises(SnError) as e:
        g.run(xd)
    assert e.value.status == _sn.SN_ETIMEOUT
    g.set_option(SN_OPT_WAIT_LIMIT, 0)
    assert torch.equal(g.run(xd), y)


def test_larger_layers_stay_two_launches():
    """More than one wave of CTAs: the two layers keep their launches."""
    sch = ("f16", "nhwc")
    layers = weights([dict(synth.conv(16, 192, 1), inputs=[-1]), dict(synth.dwconv(192, 3, 1), inputs=[0])], 9)
    x = np.zeros((64, 16, 56, 56), np.float32)
    g = graph(layers, x, sch)
    assert g.plan_stats() == (2, 2)


@pytest.mark.parametrize("case", [(1, 96, 14, 14, 72, 3, 1), (2, 160, 7, 7, 200, 5, 1), (1, 200, 9, 11, 136, 3, 2),
                                  (1, 512, 7, 7, 256, 3, 1), (1, 16, 1, 300, 24, 3, 1)])
@pytest.mark.parametrize("dt", ["f16", "bf16"])
def test_pair_equals_two_launches_of_any_variants(case, dt):
    """Whatever variants the path selected: clusters group the K steps among their
    CTAs, and so does the pair; variants that group them otherwise, and the fp16
    3x3 depthwise kernel that adds in fp32 (wide rows), stay two launches."""
    import torch
    N, C, H, W, E, k, s = case
    sch = (dt, "nhwc")
    layers = weights([dict(synth.conv(C, E, 1, act="relu6"), inputs=[-1]),
                      dict(synth.dwconv(E, k, s, act="hswish"), inputs=[0])], zlib.crc32(repr(case).encode()))
    x = np.random.default_rng(4).standard_normal((N, C, H, W)).astype(np.float32)
    g = build_graph(layers, x.shape, sch, sch, [sch])
    t = g.cost_table()
    xd = to_device(x, sch)
    tc = [int(c) for c in np.flatnonzero(t["layer"] == 1) if routine_name(int(t["routine"][c])) == "conv2/igemm_tc"]
    dw = [int(c) for c in np.flatnonzero(t["layer"] == 2)]
    seen = set()
    for c in tc:
        for d in dw if c in (tc[0], tc[-1]) else dw[:1]:
            g.set_option(SN_OPT_PAIR, 1)
            g.set_path([int(np.flatnonzero(t["layer"] == 0)[0]), c, d, int(np.flatnonzero(t["layer"] == 3)[0])])
            what = g.candidate_desc(c) + " + " + g.candidate_desc(d)
            split = "ksplit=1" not in what and "cluster=" not in what or "csk=2" in what or "streamk" in what
            one = g.plan_stats()[1] == 1
            assert not (one and split), what
            assert one or split or "cluster=8" in what or W == 300, what
            seen.add((one, what.split("cluster=")[-1][:1] if "cluster=" in what else split))
            y = g.run(xd).clone()
            g.set_option(SN_OPT_PAIR, 0)
            y2 = g.run(xd)
            torch.cuda.synchronize()
            assert torch.equal(y.view(torch.int16), y2.view(torch.int16)), what
    assert (True, False) in seen and ((True, "2") in seen or C <= 64)
    if W == 300 and dt == "f16":
        assert any(not one for one, _ in seen)
