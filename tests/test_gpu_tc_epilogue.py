"""The epilogue's packed pairs: relu and relu6 after the rounding, sums past the
16-bit range, infinities and NaNs, with and without a residual, in the tiles of
every kind (full, half, cluster, split along K, NCHW writer)."""
import numpy as np
import pytest

import synth
from paper_2110_06037_gb300 import SnError, build_graph

from gpu_helpers import from_device, stored_values, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("dt", ["f16", "bf16"])
def test_values_of_the_epilogue(act, residual, dt):
    import torch
    # a permutation of the channels with power-of-two weights and zero bias: each
    # sum has one non-zero product (and a residual equal to it, which doubles it),
    # so every sum is exact and the result known
    C, H = 128, 16
    rng = np.random.default_rng(3)
    x = (rng.standard_normal((1, C, H, H)) * 4).astype(np.float32)
    x[0, :, 0, 0] = 6.0
    x[0, :, 1, 1] = 40000.0  # doubled: past the largest f16 value
    x[0, :, 2, 2] = -0.0
    x[0, 5, 3, 3] = np.inf  # times zero in every other channel: a NaN
    x[0, 6, 4, 4] = np.nan
    perm = rng.permutation(C)
    w = np.zeros((C, C, 1, 1), np.float32)
    w[np.arange(C), perm] = 1.0
    conv = dict(synth.conv(C, C, 1, 1, 0, act=act), weight=w, bias=np.zeros(C, np.float32))
    first = dict(conv, params=dict(conv["params"], act="none"))
    sch = (dt, "nhwc")
    net = [dict(first, inputs=[-1]), dict(conv, inputs=[-1, 0])] if residual else [dict(conv, inputs=[-1])]
    xs = stored_values(x, dt)
    with np.errstate(invalid="ignore"):
        f = xs[:, perm]
        f[:, :, 4, 4] = np.nan
        f[:, perm != 5, 3, 3] = np.nan
        if residual:
            f = f + f
        if act != "none":  # a NaN becomes 0, as fmaxf has it
            f = np.where(np.isnan(f), 0.0, np.clip(f, 0.0, 6.0 if act == "relu6" else np.inf)).astype(np.float32)
        ref = stored_values(f, dt)
    g = build_graph(net, x.shape, sch, sch, [sch])
    t = g.cost_table()
    li = len(net)
    p = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])]
    if residual:
        p[1] = [int(c) for c in np.flatnonzero(t["layer"] == 1) if "igemm_tc" in g.candidate_desc(int(c))][0]
    xd = to_device(x, sch)
    seen = 0
    for c in np.flatnonzero(t["layer"] == li):
        if f"conv2/igemm_tc {dt}" not in g.candidate_desc(int(c)):
            continue
        p[li] = int(c)
        try:
            g.set_path(p)
        except SnError:  # a candidate of another schema does not join this path
            continue
        y = from_device(g.run(xd), sch)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(y, ref, err_msg=g.candidate_desc(int(c)))
        seen += 1
    assert seen > 4


@pytest.mark.parametrize("dt", ["f16", "bf16"])
@pytest.mark.parametrize("c,k", [(64, 136), (72, 320)])
def test_residual_over_many_tiles(c, k, dt):
    # several tiles a CTA, the last ones ragged in pixels and channels: the
    # residual of the next tile is loaded while this one is stored
    import torch
    rng = np.random.default_rng(k)
    x = rng.standard_normal((9, c, 57, 57)).astype(np.float32)
    pick = rng.integers(0, c, k)
    w = np.zeros((k, c, 1, 1), np.float32)
    w[np.arange(k), pick] = 1.0
    bias = rng.integers(-2, 3, k).astype(np.float32)
    first = dict(synth.conv(c, k, 1, 1, 0, act="none"), weight=w, bias=np.zeros(k, np.float32), inputs=[-1])
    conv = dict(synth.conv(c, k, 1, 1, 0, act="relu"), weight=w, bias=bias, inputs=[-1, 0])
    sch = (dt, "nhwc")
    f = stored_values(x, dt)[:, pick]
    # the library's order: (sum + bias) + residual, each rounded to fp32
    v = (f.astype(np.float32) + bias[None, :, None, None]).astype(np.float32) + f.astype(np.float32)
    ref = stored_values(np.maximum(v, 0.0), dt)
    g = build_graph([first, conv], x.shape, sch, sch, [sch])
    t = g.cost_table()
    p = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])]
    desc = {int(c): g.candidate_desc(int(c)) for c in np.flatnonzero((t["layer"] == 1) | (t["layer"] == 2))}
    p[1] = [i for i, d in desc.items() if t["layer"][i] == 1 and f"conv2/igemm_tc {dt}.nhwc [" in d][0]
    xd = to_device(x, sch)
    seen = 0
    for i, d in desc.items():
        if t["layer"][i] != 2 or f"conv2/igemm_tc {dt}.nhwc [" not in d:
            continue
        p[2] = i
        g.set_path(p)
        y = from_device(g.run(xd), sch)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(y, ref, err_msg=d)
        seen += 1
    assert seen > 4
