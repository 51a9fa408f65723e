"""FP64 mode where the FP32 bound that decides steps without an event leaves
FP32's range (a product of momentum and field, or a momentum, beyond 3.4e38:
infinities, whose differences are NaN): such particles are decided in FP64,
with the oracle's events."""
import numpy as np
import pytest

import oracle
from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

N, CAP = 1500, 60000


def _particles(p):
    d = {k: np.zeros(N) for k in ("x", "y", "z")}
    d.update({k: np.full(N, p) for k in ("px", "py", "pz")}, w=np.ones(N), id=np.arange(N, dtype=np.uint64))
    return d


def _both(sp, b, dt, steps, photons):
    prm = [0.0, 0.0, 0.0, b, 2 * b, 3 * b]               # no electric field: an emitter that stops stays
    g = q.Generator(q.make_config(precision=q.QED_FP64, seed=8, push_photons=photons))
    ens = q.DeviceEnsemble.from_host(sp, [CAP] * 3, q.QED_FP64)
    st = g.push(ens, q.make_field(W.FIELD_UNIFORM, prm), dt, steps, 0, auto_grow=False)
    g.close()
    o = oracle.Ensemble.from_arrays(sp, [CAP] * 3)
    cfg = oracle.make_cfg(seed=8, push_photons=photons, field_kind=W.FIELD_UNIFORM, field_prm=prm)
    return st, oracle.push_and_generate(o, oracle.build_tables(), cfg, dt, steps, 0)


# momentum per axis, field, steps in which about a third of the leptons emit (and stop) and a few percent of the
# photons convert: small avalanches by the oracle's count
RANGES = [(1e22, 1e17, 1e-4, 3e-5), (1e18, 1e21, 3e-9, 1e-9), (1e39, 1e17, 20.0, 6.0)]


@pytest.mark.parametrize("p,b,dt,_", RANGES)
@pytest.mark.parametrize("steps", [1, 2])
def test_leptons_beyond_fp32_range(p, b, dt, _, steps):
    st, ost = _both([_particles(p), W._empty(), W._empty()], b, dt, steps, 0)
    assert ost["emit_events"] > N // 10
    assert st["emit_events"] == ost["emit_events"] and st["max_subevents"] == ost["max_subevents"]


@pytest.mark.parametrize("p,b,_,dt", RANGES)
def test_photons_beyond_fp32_range(p, b, _, dt):
    st, ost = _both([W._empty(), W._empty(), _particles(p)], b, dt, 1, 1)
    assert ost["pair_events"] > 20
    for k in ("pair_events", "emit_events", "particle_steps"):
        assert st[k] == ost[k], k
