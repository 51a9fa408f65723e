"""Emission runs of several steps take one launch while the leptons fit the
resident threads (a few times over in FP32) and a launch per step beyond; both
sides of the line give the results of steps taken one call at a time."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

STEPS = 12


def _run(prec, n, calls):
    w = W.uniform_b_emission(n=n, seed=3, chi0=1.0, steps_per_period=400, nsteps=STEPS)
    w.species[0]["w"][::7] = 0.0
    g = q.Generator(q.make_config(precision=prec, seed=3, push_photons=0))
    ens = q.DeviceEnsemble.from_host(w.species, [n, 4, n], prec)
    st = [g.push(ens, q.make_field(w.field_kind, w.field_prm), w.dt, STEPS if calls == "one" else 1, k, auto_grow=False)
          for k in range(1 if calls == "one" else STEPS)]
    out = [ens.to_host(s) for s in (0, 2)]
    g.close()
    return out, {k: sum(s[k] for s in st) for k in ("particle_steps", "emit_events", "launches")}


@pytest.mark.parametrize("prec,n,one", [(q.QED_FP32, 70000, True), (q.QED_FP32, 220001, True), (q.QED_FP32, 400001, False),
                                        (q.QED_FP64, 30001, True), (q.QED_FP64, 200001, False)])
def test_both_sides_of_the_line(prec, n, one):
    a, sa = _run(prec, n, "one")
    b, sb = _run(prec, n, "each")
    assert (sa["launches"] < STEPS) == one
    assert sa["particle_steps"] == sb["particle_steps"] and sa["emit_events"] == sb["emit_events"] > 0
    tol = 1e-5 if prec == q.QED_FP32 else 1e-12
    for u, v in zip(a, b):
        i, j = np.argsort(u["id"]), np.argsort(v["id"])
        assert np.array_equal(u["id"][i], v["id"][j]) and np.array_equal(u["nevents"][i], v["nevents"][j])
        for k in ("px", "py"):
            assert np.max(np.abs(u[k][i] - v[k][j])) < tol * 1000
