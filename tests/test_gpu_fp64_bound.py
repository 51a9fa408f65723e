"""FP64 photons whose flight to the step end, and FP64 leptons whose step
without an event, is decided by a bound in FP32: against the oracle, decision by decision, over photon energies and directions
from far below the pair threshold to chi of several hundred, in every analytic
field (along and across the field, at rest-frame extremes)."""
import numpy as np
import pytest

import oracle
from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

FIELDS = [(W.FIELD_ROTATING_E, [2500.0]), (W.FIELD_STANDING_CP, [2500.0]),
          (W.FIELD_UNIFORM, [0, 0, 0, 0, 900.0, 1500.0]), (W.FIELD_UNIFORM, [700.0, 0, -300.0, 200.0, 900.0, 1500.0])]


@pytest.mark.parametrize("kind,prm", FIELDS)
@pytest.mark.parametrize("n", [1, 257, 40000])
def test_photons_fp64(kind, prm, n):
    r = np.random.default_rng(n)
    k = np.exp(r.uniform(np.log(1e-3), np.log(1e5), n))
    v = r.standard_normal((n, 3))
    v[: n // 5] *= [1.0, 1e-9, 1e-9]                       # nearly along an axis
    v *= (k / np.linalg.norm(v, axis=1))[:, None]
    ph = {c: r.uniform(-40, 40, n) for c in ("x", "y", "z")}
    ph.update({c: v[:, i] for i, c in enumerate(("px", "py", "pz"))})
    ph.update(w=np.ones(n), id=np.arange(n, dtype=np.uint64))
    cap = [200000, 200000, n + 200000]
    g = q.Generator(q.make_config(precision=q.QED_FP64, seed=5, push_photons=1))
    ens = q.DeviceEnsemble.from_host([W._empty(), W._empty(), ph], cap, q.QED_FP64)
    st = g.push(ens, q.make_field(kind, prm), W.TWO_PI / 100, 2, 3, auto_grow=False)
    g.close()
    o = oracle.Ensemble.from_arrays([W._empty(), W._empty(), ph], cap)
    ost = oracle.push_and_generate(o, oracle.build_tables(), oracle.make_cfg(seed=5, push_photons=1, field_kind=kind,
                                                                             field_prm=prm), W.TWO_PI / 100, 2, 3)
    assert (st["pair_events"], st["emit_events"]) == (ost["pair_events"], ost["emit_events"])
    assert n < 1000 or st["pair_events"] > 50
    a, b = ens.to_host(2), o.view(2)
    i, j = np.argsort(a["id"]), np.argsort(b["id"])
    assert np.array_equal(a["id"][i], b["id"][j])
    for c in ("x", "y", "z"):
        assert np.allclose(a[c][i], b[c][j], rtol=0, atol=1e-12)


@pytest.mark.parametrize("kind,prm", FIELDS)
@pytest.mark.parametrize("n,steps,photons", [(1, 3, 1), (129, 3, 0), (20000, 2, 1), (20000, 3, 0)])
def test_leptons_fp64(kind, prm, n, steps, photons):
    r = np.random.default_rng(n + steps)
    k = np.exp(r.uniform(np.log(1e-4), np.log(1e5), n))
    k[::11] = 0.0                                          # at rest
    v = r.standard_normal((n, 3))
    v[: n // 5] *= [1.0, 1e-9, 1e-9]
    v *= (k / np.linalg.norm(v, axis=1))[:, None]
    sp = []
    for s in range(2):
        d = {c: r.uniform(-40, 40, n) for c in ("x", "y", "z")}
        d.update({c: v[:, i] for i, c in enumerate(("px", "py", "pz"))})
        d.update(w=np.ones(n), id=np.arange(n, dtype=np.uint64) + (s << 40))
        sp.append(d)
    cap = [n + 50000, n + 50000, 400000]
    g = q.Generator(q.make_config(precision=q.QED_FP64, seed=6, push_photons=photons))
    ens = q.DeviceEnsemble.from_host(sp + [W._empty()], cap, q.QED_FP64)
    st = g.push(ens, q.make_field(kind, prm), W.TWO_PI / 100, steps, 3, auto_grow=False)
    g.close()
    o = oracle.Ensemble.from_arrays(sp + [W._empty()], cap)
    ost = oracle.push_and_generate(o, oracle.build_tables(),
                                   oracle.make_cfg(seed=6, push_photons=photons, field_kind=kind, field_prm=prm),
                                   W.TWO_PI / 100, steps, 3)
    for key in ("particle_steps", "emit_events", "pair_events"):
        assert st[key] == ost[key], key
    for s in range(2):
        a, b = ens.to_host(s), o.view(s)
        i, j = np.argsort(a["id"]), np.argsort(b["id"])
        assert np.array_equal(a["id"][i], b["id"][j]) and np.array_equal(a["nevents"][i], b["nevents"][j])
        pa, pb = (np.stack([d[c][m] for c in ("px", "py", "pz")]) for d, m in ((a, i), (b, j)))
        assert np.max(np.linalg.norm(pa - pb, axis=0) / np.maximum(np.linalg.norm(pb, axis=0), 1e-3)) < 1e-5
