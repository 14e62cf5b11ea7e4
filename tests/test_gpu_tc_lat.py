"""Small-layer tensor-core tiles (a cluster of 1, 2, 4 or 8 CTAs per tile, the K
steps split among them): K steps that do not divide by the cluster, more K steps
per CTA than stages, output channels that end inside a CTA's columns, ragged
rows, stride 2, residuals, repeatability, and a wait that runs out in a cluster."""
import zlib

import numpy as np
import pytest

import synth
from oracle.net import run_layer
from paper_2110_06037_gb300 import SN_OPT_CHECK, SN_OPT_WAIT_LIMIT, SnError, _sn, build_graph

from gpu_helpers import TOL, from_device, maxrel, stored_values, to_device

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, k, s, pad
    (1, 64, 1, 1, 8, 1, 1, 0),       # one pixel, one K step: clusters of one
    (1, 200, 7, 7, 72, 1, 1, 0),     # four K steps, the second channel tile holds eight channels
    (1, 328, 14, 14, 40, 1, 1, 0),   # six K steps among 1, 2 and 4
    (2, 136, 9, 11, 104, 3, 1, 1),   # 27 K steps: stages reused
    (1, 64, 16, 16, 128, 3, 2, 1),   # stride 2
    (1, 1024, 14, 14, 256, 1, 1, 0),  # sixteen K steps among eight
]


def lat(g, layer):
    t = g.cost_table()
    return [int(c) for c in np.flatnonzero(t["layer"] == layer) if "cluster=" in g.candidate_desc(int(c))], t


def path(t, layer, c):
    p = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])]
    p[layer] = c
    return p


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("residual", [False, True])
def test_cluster_tiles(case, dt, residual):
    import torch
    N, C, H, W, K, k, s, pd = case
    sch = (dt, "nhwc")
    rng = np.random.default_rng(zlib.crc32(repr((case, dt)).encode()))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    layer = synth.conv(C, K, k, s, pd, act="hswish")
    layer["weight"] = (rng.standard_normal((K, C, k, k)) * np.sqrt(2.0 / (C * k * k))).astype(np.float32)
    layer["bias"] = rng.standard_normal(K).astype(np.float32)
    other = dict(layer, params=dict(layer["params"], act="none"), weight=layer["weight"][:, ::-1].copy())
    net = [dict(other, inputs=[-1]), dict(layer, inputs=[-1, 0])] if residual else [dict(layer, inputs=[-1])]
    g = build_graph(net, x.shape, sch, sch, [sch])
    xd = to_device(x, sch)
    ins = [stored_values(x, dt)]
    if residual:  # the value that joins is the library's own first layer
        g1 = build_graph(net[:1], x.shape, sch, sch, [sch])
        t1 = g1.cost_table()
        g1.set_path(path(t1, 0, 0))
        ins.append(from_device(g1.run(xd), sch))
    ref = run_layer(layer, ins, dt)
    cands, t = lat(g, len(net))
    assert cands
    for c in cands:
        g.set_path(path(t, len(net), c))
        y = g.run(xd).clone()
        y2 = g.run(xd)
        torch.cuda.synchronize()
        assert maxrel(from_device(y, sch), ref) <= TOL[dt] / 4, g.candidate_desc(c)
        assert torch.equal(y, y2), g.candidate_desc(c)


@pytest.mark.parametrize("size", [1, 4])
def test_expired_wait_in_a_cluster_reports_timeout_and_recovers(size):
    import torch
    x, layers = synth.single_conv(1, 14, 256, 64, 1, 1)
    sch = ("bf16", "nhwc")
    g = build_graph(layers, x.shape, sch, sch, [sch])
    cands, t = lat(g, 1)
    c = [c for c in cands if f"cluster={size} " in g.candidate_desc(c)][0]
    g.set_path(path(t, 1, c))
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


@pytest.mark.parametrize("size", [2, 8])
def test_expired_wait_in_every_cta_of_a_cluster(size):
    """Every CTA gives up with its peers' sums under way, many times in a row;
    the next run has its values."""
    import torch
    x, layers = synth.single_conv(2, 14, 512, 128, 1, 1)
    sch = ("f16", "nhwc")
    g = build_graph(layers, x.shape, sch, sch, [sch])
    cands, t = lat(g, 1)
    c = [c for c in cands if f"cluster={size} " in g.candidate_desc(c)][0]
    g.set_path(path(t, 1, c))
    g.set_option(SN_OPT_CHECK, 1)
    xd = to_device(x, sch)
    y0 = g.run(xd).clone()
    for _ in range(20):
        g.set_option(SN_OPT_WAIT_LIMIT, 1)
        with pytest.raises(SnError) as e:
            g.run(xd)
        assert e.value.status == _sn.SN_ETIMEOUT
    g.set_option(SN_OPT_WAIT_LIMIT, 0)
    y1 = g.run(xd)
    torch.cuda.synchronize()
    assert torch.equal(y0, y1)
