"""Host-side behaviour of the C ABI: validation, call order, cost-table and
plan-file round trips.  CPU only (no kernel is launched)."""
import numpy as np
import pytest

import synth
from paper_2110_06037_gb300 import SN_SELECT_DPRS, SnError, build_graph, _sn
from paper_2110_06037_gb300.api import Graph

S2 = [("f32", "nchw"), ("f32", "nhwc")]


def tiny():
    x, layers = synth.tiny_cnn()
    return x, build_graph(layers, x.shape, ("f32", "nchw"), ("f32", "nchw"), S2, torch_alloc=False)


def test_shapes_and_candidates():
    x, g = tiny()
    t = g.cost_table()
    assert t["n_layers"] == 8 and t["n_schemas"] == 2
    assert g.layer_shape(1) == (1, 16, 32, 32)
    assert g.layer_shape(2) == (1, 32, 16, 16)
    assert g.layer_shape(6) == (1, 10, 1, 1)
    assert g.layer_shape(7) == (1, 10, 1, 1)
    # Winograd only on the 3x3 stride-1 conv, tensor cores never in fp32
    names = {(int(t["layer"][c]), _sn.routine_name(int(t["routine"][c]))) for c in range(len(t["cost"]))}
    assert (1, "conv2/wino_f2x2_3x3") in names and (2, "conv2/wino_f2x2_3x3") not in names
    assert not any(n == "conv2/igemm_tc" for _, n in names)
    assert np.all(t["cost"][t["routine"] != 0] == _sn.COST_INF)


def test_invalid_layers_rejected():
    g = Graph((1, 3, 8, 8), ("f32", "nchw"), ("f32", "nchw"), S2, torch_alloc=False)
    bad = dict(c_in=4, c_out=8, kh=3, kw=3, sh=1, sw=1, ph=1, pw=1)
    with pytest.raises(SnError) as e:
        g.add_layer(_sn.SN_L_CONV2, bad, (-1,), np.zeros((8, 4, 3, 3)), None)
    assert e.value.status == _sn.SN_EINVAL
    with pytest.raises(SnError):
        g.add_layer(_sn.SN_L_CONV2, dict(bad, c_in=3), (5,), np.zeros((8, 3, 3, 3)), None)
    with pytest.raises(SnError):
        g.add_layer(_sn.SN_L_CONV2, dict(bad, c_in=3, kh=11, ph=0), (-1,), np.zeros((8, 3, 11, 3)), None)
    with pytest.raises(SnError):
        g.add_layer(_sn.SN_L_DENSE, dict(in_features=3, out_features=2), (-1,), np.zeros((2, 3)), None)
    l0 = g.add_layer(_sn.SN_L_CONV2, dict(bad, c_in=3), (-1,), np.zeros((8, 3, 3, 3)), None)
    with pytest.raises(SnError):  # shapes differ
        g.add_layer(_sn.SN_L_ADD, {"act": "none"}, (-1, l0))


def test_dead_end_layer_is_rejected():
    g = Graph((1, 4, 4, 4), ("f32", "nchw"), ("f32", "nchw"), S2, torch_alloc=False)
    p = dict(c_in=4, c_out=4, kh=1, kw=1, sh=1, sw=1, ph=0, pw=0)
    g.add_layer(_sn.SN_L_CONV2, p, (-1,), np.zeros((4, 4, 1, 1)), None)
    g.add_layer(_sn.SN_L_CONV2, p, (-1,), np.zeros((4, 4, 1, 1)), None)  # layer 0 is now a dead end
    with pytest.raises(SnError) as e:
        g.cost_table()
    assert e.value.status == _sn.SN_EINVAL


def test_call_order():
    x, g = tiny()
    with pytest.raises(SnError) as e:
        _sn.check(_sn.lib().sn_run(g.h, 1, 1, None))
    assert e.value.status == _sn.SN_ESTATE
    with pytest.raises(SnError) as e:  # all costs unknown -> infeasible
        g.select_path(SN_SELECT_DPRS)
    assert e.value.status == _sn.SN_EINFEASIBLE
    with pytest.raises(SnError) as e:  # finalised: no more layers
        g.add_layer(_sn.SN_L_GAP, None, (0,))
    assert e.value.status == _sn.SN_ESTATE


def test_cost_table_validation_and_roundtrip(tmp_path):
    x, g = tiny()
    t = g.cost_table()
    rng = np.random.default_rng(0)
    t["cost"] = np.where(t["routine"] == 0, 0, rng.integers(1, 100, len(t["cost"]))).astype(np.int64)
    a = rng.integers(1, 50, t["adapt"].shape).astype(np.int64)
    for e in range(a.shape[0]):
        np.fill_diagonal(a[e], 0)
    t["adapt"] = a
    g.set_cost_table(t)
    t2 = g.cost_table()
    assert np.array_equal(t2["cost"], t["cost"]) and np.array_equal(t2["adapt"], a)
    bad = dict(t)
    bad["adapt"] = a.copy()
    bad["adapt"][0, 0, 0] = 5  # void adapt must be 0
    with pytest.raises(SnError):
        g.set_cost_table(bad)
    bad = dict(t)
    bad["schema"] = t["schema"].copy()
    bad["schema"][3] ^= 1
    with pytest.raises(SnError):
        g.set_cost_table(bad)
    assert np.array_equal(g.cost_table()["cost"], t["cost"])  # unchanged after errors
    tot, sch, cand = g.select_path(SN_SELECT_DPRS)
    p = tmp_path / "plan.json"
    g.save_plan(p)
    x2, g2 = tiny()
    g2.load_plan(p)
    t3 = g2.cost_table()
    assert np.array_equal(t3["cost"], t["cost"]) and np.array_equal(t3["adapt"], a)
    g2.save_plan(tmp_path / "plan2.json")
    assert open(p).read() == open(tmp_path / "plan2.json").read()


def test_set_path_validation():
    x, g = tiny()
    t = g.cost_table()
    with pytest.raises(SnError):
        g.set_path(np.zeros(t["n_layers"], np.int32))  # candidate 0 belongs to layer 0 only
    first = [int(np.flatnonzero(t["layer"] == i)[0]) for i in range(t["n_layers"])]
    g.set_path(first)


def test_tc_not_offered_where_it_cannot_run():
    for C, dt, lay, s, H in [(3, "f16", "nhwc", 1, 8), (64, "f32", "nhwc", 1, 8), (64, "f16", "nchw", 1, 8),
                             (64, "bf16", "nhwc", 2, 7)]:
        layer = synth.conv(C, 64, 3, s, 1)
        layer["weight"] = np.zeros((64, C, 3, 3), np.float32)
        layer["bias"] = np.zeros(64, np.float32)
        g = build_graph([dict(layer, inputs=[-1])], (1, C, H, H), (dt, lay), (dt, lay), [(dt, lay)],
                        torch_alloc=False)
        t = g.cost_table()
        assert not any(_sn.routine_name(int(r)) == "conv2/igemm_tc" for r in t["routine"])


def test_qint8_candidates_and_scales():
    """The qint8 schema offers exactly the routines with an int8 kernel, and
    blob scales are validated and kept across finalisation."""
    x, layers = synth.tiny_cnn()
    g = build_graph(layers, x.shape, ("f32", "nchw"), ("f32", "nchw"), [("f32", "nhwc"), ("qi8", "nhwc")],
                    torch_alloc=False)
    g.set_qscale(-1, 0.5)
    t = g.cost_table()  # finalises
    q8_names = {_sn.routine_name(int(t["routine"][c])) for c in range(len(t["cost"]))
                if t["schema"][c] == 1}
    assert q8_names <= {"io", "conv2/direct", "conv2/igemm_dp4a", "dwconv2/direct", "maxpool/direct", "gap/reduce",
                        "add/eltwise", "mul/eltwise", "dense/simt"}
    assert "conv2/direct" in q8_names
    f_names = {_sn.routine_name(int(t["routine"][c])) for c in range(len(t["cost"])) if t["schema"][c] == 0}
    assert "conv2/igemm_dp4a" not in f_names
    assert g.get_qscale(-1) == 0.5 and g.get_qscale(0) == 0.0
    g.set_qscale(2, 0.125)
    assert g.get_qscale(2) == 0.125
    for bad in (0.0, -1.0, float("inf"), float("nan")):
        with pytest.raises(SnError) as e:
            g.set_qscale(0, bad)
        assert e.value.status == _sn.SN_EINVAL
    with pytest.raises(SnError):
        g.set_qscale(len(layers), 1.0)
    with pytest.raises(SnError):
        g.get_qscale(-2)


def test_convert_needs_a_scale_for_qint8():
    import ctypes as C
    shp = (C.c_int64 * 4)(1, 2, 3, 4)
    fake = C.c_void_p(256)  # validation fails before any device access
    st = _sn.lib().sn_convert(fake, _sn.schema(("f16", "nchw")), fake, _sn.schema(("qi8", "nchw")), shp, None)
    assert st == _sn.SN_EINVAL
    st = _sn.lib().sn_convert_q(fake, _sn.schema(("f16", "nchw")), fake, _sn.schema(("f16", "nhwc")), shp,
                                C.c_float(1.0), None)
    assert st == _sn.SN_EINVAL  # no qint8 side
    st = _sn.lib().sn_convert_q(fake, _sn.schema(("f16", "nchw")), fake, _sn.schema(("qi8", "nchw")), shp,
                                C.c_float(0.0), None)
    assert st == _sn.SN_EINVAL  # bad scale


def test_calibration_needs_costs_and_a_single_input():
    import ctypes as C
    x, layers = synth.tiny_cnn()
    g = build_graph(layers, x.shape, ("f32", "nchw"), ("f32", "nchw"), [("f32", "nhwc"), ("qi8", "nhwc")],
                    torch_alloc=False)
    fake = C.c_void_p(256)  # refused before any device access
    assert _sn.lib().sn_calibrate(g.h, fake, None) == _sn.SN_ESTATE  # nothing profiled: no finite float path
    g2 = Graph((1, 4, 3, 3), ("f32", "nchw"), ("f32", "nchw"), [("f32", "nchw")], torch_alloc=False)
    g2.add_input((1, 4, 3, 3))
    w = np.zeros((4, 4, 1, 1), np.float32)
    p = dict(c_in=4, c_out=4, kh=1, kw=1, sh=1, sw=1, ph=0, pw=0)
    g2.add_layer(_sn.SN_L_CONV2, p, (-1,), w, None)
    g2.add_layer(_sn.SN_L_CONV2, p, (-2,), w, None)
    g2.add_layer(_sn.SN_L_ADD, dict(act="none"), (0, 1), None, None)
    assert _sn.lib().sn_calibrate(g2.h, fake, None) == _sn.SN_EUNSUPPORTED
    assert g2.io_counts() == (2, 1)
    # a second input's scale is set by its id
    g2.set_qscale(-2, 0.25)
    assert g2.get_qscale(-2) == 0.25 and g2.get_qscale(-1) == 0.0
    with pytest.raises(SnError):
        g2.set_qscale(-3, 1.0)


def test_candidate_descriptors():
    """Every candidate has a descriptor naming its routine, the schema it reads
    and, for the tensor-core routine, the parameter values that tell its
    variants apart (section III-C: routine descriptor + routine parameters)."""
    x, layers = synth.single_conv(2, 14, 64, 128, 3, 1)
    g = build_graph(layers, x.shape, ("bf16", "nhwc"), ("bf16", "nhwc"), [("bf16", "nhwc")], torch_alloc=False)
    t = g.cost_table()
    descs = [g.candidate_desc(c) for c in range(len(t["cost"]))]
    for c, d in enumerate(descs):
        assert d.startswith(_sn.routine_name(int(t["routine"][c]))), d
        assert "bf16.nhwc" in d or t["routine"][c] == 0, d
    tc = [d for c, d in enumerate(descs) if _sn.routine_name(int(t["routine"][c])) == "conv2/igemm_tc"]
    assert len(tc) > 4 and len(set(tc)) == len(tc), tc  # distinct parameter values per variant
    assert all("bn=" in d and "tile=" in d for d in tc)
    with pytest.raises(SnError):
        g.candidate_desc(len(t["cost"]))


def test_plan_file_of_a_build_with_fewer_candidates(tmp_path):
    """A plan file that lists a subset of the graph's candidates (written before
    a routine or a routine parameter was added) loads: the path names the same
    routines, the candidates it does not list stay unprofiled."""
    import json

    import synth
    from paper_2110_06037_gb300._sn import COST_INF
    layer = synth.conv(16, 16, 3, 1)
    layer["weight"] = np.ones((16, 16, 3, 3), np.float32)

    def make():
        sch = [("f16", "nchw"), ("f16", "nhwc")]
        return build_graph([dict(layer, inputs=[-1])], (1, 16, 8, 8), sch[0], sch[0], sch)

    g = make()
    t = g.cost_table()
    t["cost"] = np.arange(len(t["cost"])) + 100
    t["adapt"][t["adapt"] > 0] = 7
    g.set_cost_table(t)
    mine = np.flatnonzero(t["layer"] == 1)
    path = [int(np.flatnonzero(t["layer"] == 0)[0]), int(mine[-1]), int(np.flatnonzero(t["layer"] == 2)[0])]
    g.set_path(path)
    f = tmp_path / "plan.json"
    g.save_plan(f)
    doc = json.loads(f.read_text())
    drop = int(mine[1])  # the file never heard of this candidate
    del doc["candidates"][drop]
    doc["n_candidates"] -= 1
    doc["path"] = [c - (c > drop) for c in doc["path"]]
    f.write_text(json.dumps(doc))
    g2 = make()
    g2.load_plan(f)
    t2 = g2.cost_table()
    want = np.asarray(t["cost"]).copy()
    want[drop] = COST_INF
    assert list(t2["cost"]) == list(want)
    g2.save_plan(tmp_path / "back.json")
    assert json.loads((tmp_path / "back.json").read_text())["path"] == path
    doc["candidates"][drop][1] = 9999  # a candidate that this build does not have
    f.write_text(json.dumps(doc))
    with pytest.raises(Exception):
        g2.load_plan(f)


def _one_conv_net(n, c, k, hw=8):
    import synth
    layer = synth.conv(c, k, 3, 1)
    layer["weight"] = np.ones((k, c, 3, 3), np.float32)
    sch = [("f16", "nchw"), ("f16", "nhwc"), ("f32", "nhwc"), ("qi8", "nhwc")]
    g = build_graph([dict(layer, inputs=[-1])], (n, c, hw, hw), sch[0], sch[0], sch)
    t = g.cost_table()
    t["cost"] = np.arange(len(t["cost"])) + 100
    t["adapt"][t["adapt"] > 0] = 7
    g.set_cost_table(t)
    mine = np.flatnonzero(t["layer"] == 1)
    g.set_path([int(np.flatnonzero(t["layer"] == 0)[0]), int(mine[5]), int(np.flatnonzero(t["layer"] == 2)[0])])
    return g


def _first_format(doc, keep):
    """The document as the first format had it: five numbers a candidate, those in `keep` only."""
    doc = dict(doc, format="softneuro-gb300-plan-1", n_candidates=len(keep),
               candidates=[doc["candidates"][i][:5] for i in keep])
    doc["path"] = [keep.index(c) for c in doc["path"]]
    return doc


def test_plan_file_of_the_first_format(tmp_path):
    """Without ids, a list must be this net's or the one that the builds of that
    format made of it; any other is another net's."""
    import json

    from paper_2110_06037_gb300._sn import COST_INF
    g = _one_conv_net(2, 128, 64)
    f = tmp_path / "plan.json"
    g.save_plan(f)
    doc = json.loads(f.read_text())
    desc = [g.candidate_desc(c) for c in range(doc["n_candidates"])]
    later = [d for d in desc if "cluster=" in d or "igemm_tc_odd" in d or "igemm_tc_f32" in d or " [tc " in d]
    assert any("cluster=" in d for d in later) and any("igemm_tc_f32" in d for d in later) and any("dp4a" in d for d in later)
    old = [i for i, d in enumerate(desc) if d not in later]
    for keep in (list(range(len(desc))), old):
        f.write_text(json.dumps(_first_format(doc, keep)))
        g2 = _one_conv_net(2, 128, 64)
        g2.load_plan(f)
        cost = list(g2.cost_table()["cost"])
        assert cost == [doc["candidates"][i][4] if i in keep else COST_INF for i in range(len(desc))]
        g2.save_plan(tmp_path / "back.json")
        assert json.loads((tmp_path / "back.json").read_text())["path"] == doc["path"]
    for drop in (old[-2], [i for i in range(len(desc)) if i not in old][0]):
        for keep in (list(range(len(desc))), old):
            if drop in keep and drop not in doc["path"]:
                f.write_text(json.dumps(_first_format(doc, [i for i in keep if i != drop])))
                with pytest.raises(SnError):
                    g.load_plan(f)


def test_plan_file_of_another_net_with_a_shorter_list(tmp_path):
    """Same layers, another batch or channel count: fewer variants apply there, and
    those of the same index are other tiles here."""
    import json
    f = tmp_path / "plan.json"
    here = _one_conv_net(1, 64, 128, 14)
    shorter = 0
    for other in (_one_conv_net(32, 64, 128, 14), _one_conv_net(1, 64, 64, 14), _one_conv_net(1, 256, 128, 14)):
        other.save_plan(f)
        doc = json.loads(f.read_text())
        keys = [tuple(c[:4]) for c in doc["candidates"]]
        here.save_plan(tmp_path / "here.json")
        mine = [tuple(c[:4]) for c in json.loads((tmp_path / "here.json").read_text())["candidates"]]
        assert keys != mine
        shorter += all(keys.count(k) <= mine.count(k) for k in keys)
        with pytest.raises(SnError):
            here.load_plan(f)
        f.write_text(json.dumps(_first_format(doc, list(range(len(keys))))))
        with pytest.raises(SnError):
            here.load_plan(f)
    assert shorter
    # a layer without candidates, and candidates in another order
    here.save_plan(f)
    doc = json.loads(f.read_text())
    for cands in ([c for c in doc["candidates"] if c[3] != 1], doc["candidates"][:1] + doc["candidates"][2:0:-1] + doc["candidates"][3:]):
        bad = dict(doc, candidates=cands, n_candidates=len(cands), path=[])
        f.write_text(json.dumps(bad))
        with pytest.raises(SnError):
            here.load_plan(f)
