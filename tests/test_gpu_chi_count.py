"""qed_stats.chi_fp64 counts evaluations of particles that are pushed: places
with dead photons (and the place past an odd count) add nothing to it."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


def _count(ph, steps):
    g = q.Generator(q.make_config(precision=q.QED_FP32, seed=5))
    ens = q.DeviceEnsemble.from_host([W._empty(), W._empty(), ph], [4000, 4000, 60000], q.QED_FP32)
    # photons along E x B cancel: their chi takes the FP64 form
    st = g.push(ens, q.make_field(W.FIELD_UNIFORM, [0, 1000.0, 0, 0, 0, 1000.0]), W.TWO_PI / 100, steps, 3, auto_grow=False)
    g.close()
    return st


@pytest.mark.parametrize("n", [1, 512, 20001])
@pytest.mark.parametrize("steps", [1, 3])
def test_dead_photons_are_not_counted(n, steps):
    r = np.random.default_rng(n)
    k = r.uniform(3, 30, n)
    ph = {c: r.uniform(-3, 3, n) for c in ("x", "y", "z")}
    ph.update(px=k, py=k * r.uniform(-1e-3, 1e-3, n), pz=np.zeros(n), w=np.ones(n), id=np.arange(n, dtype=np.uint64))
    dead = r.random(n) < 0.2                                 # few enough to stay in place (deferred removal)
    dead[0] = n == 1
    some = {c: (np.where(dead, 0.0, v) if c == "w" else v) for c, v in ph.items()}
    live = {c: v[~dead] for c, v in ph.items()}
    a, b = _count(some, steps), _count(live, steps)
    assert a["chi_fp64"] == b["chi_fp64"] and a["photon_steps"] == b["photon_steps"]
    assert n == 1 or b["chi_fp64"] > 0.9 * b["photon_steps"]
