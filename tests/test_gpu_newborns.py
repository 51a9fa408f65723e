"""Newborns of a step (Algorithm 2): avalanches inside one long step, against
the FP64 oracle particle by particle.  Electrons at chi0 = 300 emit several
times in the step and most of their photons convert, so newborns have newborns
of their own over many generations, and blocks with many electrons create more
pairs than their newborn lists hold (the rest take further launches)."""
import numpy as np
import pytest

import oracle
from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

CAP = 1000000


def _avalanche(n):
    return W.uniform_b_emission(n=n, seed=5, p0=1e5, chi0=300.0, steps_per_period=1, nsteps=1)


def _push(w, prec):
    g = q.Generator(q.make_config(precision=prec, seed=w.seed, push_photons=1))
    ens = q.DeviceEnsemble.from_host(w.species, [CAP] * 3, prec)
    st = g.push(ens, q.make_field(w.field_kind, w.field_prm), w.dt, 1, 0, auto_grow=False)
    out = [ens.to_host(s) for s in range(3)]
    g.close()
    return out, st


def _oracle(w):
    ot = oracle.build_tables()
    ens = oracle.Ensemble.from_arrays(w.species, [CAP] * 3)
    st = oracle.push_and_generate(ens, ot, oracle.make_cfg(seed=w.seed, push_photons=1, field_kind=w.field_kind,
                                                           field_prm=w.field_prm), w.dt, 1, 0)
    return [ens.view(s) for s in range(3)], st


@pytest.mark.parametrize("n", [1, 127, 129, 1000])
def test_avalanche_in_one_step_fp64(n):
    w = _avalanche(n)
    g, gs = _push(w, q.QED_FP64)
    o, os_ = _oracle(w)
    for k in ("particle_steps", "emit_events", "pair_events", "max_subevents"):
        assert gs[k] == os_[k], k
    assert gs["passes"] >= (2 if n > 1 else 0)
    if n == 1000:                    # block lists overflowed: launches beyond those of the one-electron step
        assert gs["launches"] > _push(_avalanche(1), q.QED_FP64)[1]["launches"]
    for s in range(3):
        a, b = np.argsort(g[s]["id"]), np.argsort(o[s]["id"])
        assert np.array_equal(g[s]["id"][a], o[s]["id"][b]), s
        assert np.array_equal(g[s]["nevents"][a], o[s]["nevents"][b]), s
        gp = np.stack([g[s][k][a] for k in ("x", "y", "z", "px", "py", "pz")])
        op = np.stack([o[s][k][b] for k in ("x", "y", "z", "px", "py", "pz")])
        for v in (slice(0, 3), slice(3, 6)):
            size = np.maximum(np.linalg.norm(op[v], axis=0), 1e-3)
            if gp.shape[1]:
                assert np.max(np.linalg.norm(gp[v] - op[v], axis=0) / size) < 1e-5, s


def test_avalanche_in_one_step_fp32():
    """The same numbers of events as the oracle's within five standard
    deviations: an electron's avalanche is independent of the others', and
    its number of pairs has a spread below three times its mean."""
    w = _avalanche(1000)
    g, gs = _push(w, q.QED_FP32)
    _, os_ = _oracle(w)
    for k in ("emit_events", "pair_events"):
        mean = os_[k] / 1000
        assert abs(gs[k] - os_[k]) < 5 * 3 * mean * np.sqrt(2 * 1000), k
    # charge and count: every pair is one electron and one positron
    assert len(g[0]["id"]) == 1000 + gs["pair_events"] and len(g[1]["id"]) == gs["pair_events"]
    assert len(g[2]["id"]) == gs["emit_events"] - gs["pair_events"]
