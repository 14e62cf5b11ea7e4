"""Tensor-core convolution with stride 2 on odd extents: an odd extent's even
sub-lattice has one more row or column than its odd one.  Every variant of the
routine against the oracle, at the extents where a sub-lattice is
smallest and where the last output row or column reads the map's last row."""
import zlib

import numpy as np
import pytest

import synth
from oracle.net import run_layer
from paper_2110_06037_gb300 import build_graph, routine_name

from gpu_helpers import TOL, from_device, maxrel, stored_values, to_device

pytestmark = pytest.mark.gpu

CASES = [
    # N, C, H, W, K, k, pad
    (1, 64, 3, 3, 64, 3, 1),      # smallest odd map: sub-lattices of 2 and 1
    (2, 64, 2, 3, 64, 1, 0),      # even rows, odd columns
    (3, 72, 35, 35, 120, 5, 2),   # 5x5, channels past a 64-channel block
    (2, 128, 7, 13, 136, 3, 1),   # two blocks per stage
    (1, 24, 9, 8, 40, 3, 0),      # valid padding: the last odd row is read by no tap
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("residual", [False, True])
def test_stride2_odd_extents(case, residual):
    import torch
    N, C, H, W, K, k, pd = case
    schema = ("f16", "nhwc")
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    x = rng.standard_normal((N, C, H, W)).astype(np.float32)
    main = synth.conv(C, K, k, 2, pd, act="relu")
    proj = synth.conv(C, K, k, 2, pd, act="none")
    for l in (main, proj):
        l["weight"] = (rng.standard_normal((K, C, k, k)) * np.sqrt(2.0 / (C * k * k))).astype(np.float32)
        l["bias"] = (rng.standard_normal(K) * 0.1).astype(np.float32)
    xs = stored_values(x, "f16")
    if residual:  # the projection of a stage's first block: its output joins the main conv
        layers = [dict(proj, inputs=[-1]), dict(main, inputs=[-1, 0])]
        ref = run_layer(main, [xs, run_layer(proj, [xs], "f16")], "f16")
    else:
        layers = [dict(main, inputs=[-1])]
        ref = run_layer(main, [xs], "f16")
    g = build_graph(layers, x.shape, schema, schema, [schema])
    t = g.cost_table()
    n = t["n_layers"]
    xd = to_device(x, schema)
    first = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(n)]  # per layer: its first routine
    tc = [c for c in np.flatnonzero(t["layer"] == n - 2) if routine_name(int(t["routine"][c])) == "conv2/igemm_tc_odd"]
    assert tc
    for c in tc:
        path = list(first)
        path[n - 2] = int(c)
        g.set_path(path)
        y = g.run(xd)
        torch.cuda.synchronize()
        err = maxrel(from_device(y, schema), ref)
        assert err <= TOL["f16"], (g.candidate_desc(int(c)), err)
