"""The FP32 photon pass works on two photons per thread where the field does
not depend on the position; here at odd and even counts around its tiles, with
dead photons among them, against the FP64 oracle and against the same photons
pushed in another arrangement."""
import numpy as np
import pytest

import oracle
from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


def _photons(n, seed, dead=0.0):
    r = np.random.default_rng(seed)
    v = r.standard_normal((n, 3))
    k = np.exp(r.uniform(np.log(3.0), np.log(3000.0), n))
    v *= (k / np.linalg.norm(v, axis=1))[:, None]
    d = {c: r.uniform(-3, 3, n).astype(np.float32).astype(float) for c in ("x", "y", "z")}
    d.update({c: v[:, i].astype(np.float32).astype(float) for i, c in enumerate(("px", "py", "pz"))})
    d["w"] = np.where(r.random(n) < dead, 0.0, 1.0)
    d["id"] = np.arange(n, dtype=np.uint64)
    return d


def _push(photons, kind, prm, steps, capacity):
    g = q.Generator(q.make_config(precision=q.QED_FP32, seed=5, push_photons=1))
    ens = q.DeviceEnsemble.from_host([W._empty(), W._empty(), photons], [200000, 200000, capacity], q.QED_FP32)
    st = g.push(ens, q.make_field(kind, prm), W.TWO_PI / 100, steps, 3, auto_grow=False)
    out = [ens.to_host(s) for s in range(3)]
    g.close()
    return out, st


FIELDS = {"rotating_e": (W.FIELD_ROTATING_E, [2500.0]), "uniform_b": (W.FIELD_UNIFORM, [0, 0, 0, 0, 900.0, 1500.0]),
          "uniform_eb": (W.FIELD_UNIFORM, [700.0, 0, -300.0, 200.0, 900.0, 1500.0])}


@pytest.mark.parametrize("field", FIELDS)
@pytest.mark.parametrize("n", [1, 2, 511, 513, 30001])
def test_one_step_against_oracle(field, n):
    """Photons that did not convert fly straight at c: positions within the
    rounding of one FP32 addition (2^-23 of 3.1 each coordinate, with the
    direction's own few ulp); those that convert are the oracle's, except
    draws within the FP32 rate's error (3e-5 relative) of the boundary: none
    expected among 3e4 photons of which some hundreds convert."""
    kind, prm = FIELDS[field]
    ph = _photons(n, 7, dead=0.1)
    out, st = _push(ph, kind, prm, 1, n + 5000)
    oens = oracle.Ensemble.from_arrays([W._empty(), W._empty(), ph], [200000] * 3)
    ost = oracle.push_and_generate(oens, oracle.build_tables(), oracle.make_cfg(seed=5, push_photons=1, field_kind=kind,
                                                                                field_prm=prm), W.TWO_PI / 100, 1, 3)
    o = oens.view(2)
    live = o["w"] > 0
    assert abs(st["pair_events"] - ost["pair_events"]) <= 1
    common, a, b = np.intersect1d(out[2]["id"], o["id"][live], return_indices=True)
    assert len(common) >= max(len(out[2]["id"]), live.sum()) - 2
    for c in ("x", "y", "z"):
        assert np.max(np.abs(out[2][c][a] - o[c][live][b]), initial=0.0) < 1e-6


@pytest.mark.parametrize("field", FIELDS)
def test_arrangement_does_not_matter(field):
    """The same photons in another order, so in other pairs: bit for bit the
    same results after three steps."""
    kind, prm = FIELDS[field]
    ph = _photons(20001, 9)
    order = np.random.default_rng(1).permutation(20001)
    a, sa = _push(ph, kind, prm, 3, 60000)
    b, sb = _push({k: v[order] for k, v in ph.items()}, kind, prm, 3, 60000)
    assert sa["pair_events"] == sb["pair_events"] > 0
    for s in range(3):
        i, j = np.argsort(a[s]["id"]), np.argsort(b[s]["id"])
        for k in a[s]:
            assert np.array_equal(a[s][k][i], b[s][k][j]), (s, k)
