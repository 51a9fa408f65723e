"""Every step after one that ran out of capacity or of generations does nothing:
a call of several steps that stops in its first leaves the particles, the
demand and the statistics of a call of that step alone."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

SAME = ("particle_steps", "lepton_steps", "photon_steps", "emit_events", "pair_events", "max_subevents", "passes",
        "overflow")


def _photons(n):
    """Photons that mostly fly on, so that a step opens with all three species."""
    r = np.random.default_rng(9)
    d = {k: np.zeros(n) for k in ("x", "y", "z", "py", "pz")}
    d.update(px=r.uniform(500, 2000, n), w=np.ones(n), id=np.arange(n, dtype=np.uint64) + (7 << 32))
    return d


def _run(prec, capacity, steps, calls, thin_cap, **cfg):
    """(status, statistics, leptons in the order of their ids) of the steps, without a snapshot."""
    w = W.uniform_b_emission(n=3000, seed=5, p0=1e5, chi0=50.0, steps_per_period=20, nsteps=1)
    sp = [w.species[0], {k: (v + (1 << 33) if k == "id" else v) for k, v in w.species[0].items()}, _photons(500)]
    g = q.Generator(q.make_config(precision=prec, seed=w.seed, restore_on_overflow=0, thin_cap=thin_cap, **cfg))
    ens = q.DeviceEnsemble.from_host(sp, capacity, prec)
    field = q.make_field(w.field_kind, w.field_prm)
    rc = q.QED_OK
    for k in range(steps if calls == "each" else 1):
        g.push_async(ens, field, w.dt, 1 if calls == "each" else steps, k)
    try:
        st = g.wait(ens)
    except q.QedError as e:
        rc, st = e.status, e.stats
    lep = []
    for s in range(2):
        d = ens.to_host(s)
        order = np.argsort(d["id"])
        lep.append({k: v[order] for k, v in d.items()})
    g.close()
    return rc, st, lep, list(ens.count)


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("calls", ["one", "each"])
@pytest.mark.parametrize("thin_cap", [0, 100000])
@pytest.mark.parametrize("profile", [0, 1])
def test_steps_after_an_overflow_do_nothing(prec, calls, thin_cap, profile):
    cap = [40000, 40000, 600]
    rc1, st1, lep1, n1 = _run(prec, cap, 1, "one", thin_cap, profile=profile)
    rc, st, lep, n = _run(prec, cap, 4, calls, thin_cap, profile=profile)
    assert rc1 == rc == q.QED_ERR_CAPACITY and st1["needed_capacity"][2] > 600
    assert st["needed_capacity"] == st1["needed_capacity"] and n == n1
    for k in SAME:
        assert st[k] == st1[k], k
    for a, b in zip(lep1, lep):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("calls", ["one", "each"])
def test_steps_after_a_timeout_do_nothing(prec, calls):
    cap = [200000, 200000, 400000]
    rc1, st1, lep1, n1 = _run(prec, cap, 1, "one", 0, pass_limit=1)
    rc, st, lep, n = _run(prec, cap, 4, calls, 0, pass_limit=1)
    assert rc1 == rc == q.QED_ERR_TIMEOUT
    assert n == n1
    for k in SAME:
        assert st[k] == st1[k], k
    for a, b in zip(lep1, lep):
        for k in a:
            assert np.array_equal(a[k], b[k]), k
