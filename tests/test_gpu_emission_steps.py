"""An emission run (photons recorded, no leveling) takes all steps of a call in
one launch; here against the same steps taken one call at a time, at sizes
around its tiles and beyond one wave of blocks, with positrons and dead
entries, and when the photons run out of room."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

STEPS = 4


def _leptons(n, seed):
    r = np.random.default_rng(seed)
    d = {k: r.uniform(-3, 3, n).astype(np.float32).astype(float) for k in ("x", "y", "z")}
    d.update({k: r.normal(0, 800, n).astype(np.float32).astype(float) for k in ("px", "py", "pz")})
    d["w"] = np.where(r.random(n) < 0.1, 0.0, 1.0)
    d["id"] = np.arange(n, dtype=np.uint64) + (seed << 32)
    return d


def _run(sp, prec, field, calls, capacity):
    g = q.Generator(q.make_config(precision=prec, seed=4, push_photons=0))
    ens = q.DeviceEnsemble.from_host(sp, capacity, prec)
    events = 0
    for k in range(STEPS if calls == "each" else 1):
        st = g.push(ens, field, W.TWO_PI / 100, 1 if calls == "each" else STEPS, 2 + k, auto_grow=False)
        events += st["emit_events"]
    out = [ens.to_host(s) for s in range(3)]
    g.close()
    return out, events


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("kind,prm", [(W.FIELD_UNIFORM, [0, 0, 0, 0, 0, 900.0]), (W.FIELD_STANDING_CP, [1500.0])])
@pytest.mark.parametrize("n,m", [(1, 0), (0, 127), (129, 257), (120001, 3)])
def test_one_call_against_single_steps(prec, kind, prm, n, m):
    """The same draws, so the same events (a last-bit difference between the
    two launches' code would have to fall on a decision: 5e5 decisions times
    1e-7); momenta and positions within a few roundings per step."""
    sp = [_leptons(n, 1), _leptons(m, 2), W._empty()]
    field = q.make_field(kind, prm)
    cap = [max(n, 1), max(m, 1), 4 * (n + m) + 64]
    a, ea = _run(sp, prec, field, "one", cap)
    b, eb = _run(sp, prec, field, "each", cap)
    assert ea == eb and (ea > 0 or n + m < 10)
    tol = 1e-5 if prec == q.QED_FP32 else 1e-12
    for s in range(3):
        i, j = np.argsort(a[s]["id"]), np.argsort(b[s]["id"])
        assert np.array_equal(a[s]["id"][i], b[s]["id"][j])
        assert np.array_equal(a[s]["nevents"][i], b[s]["nevents"][j])
        for keys in (("x", "y", "z"), ("px", "py", "pz")):
            u = np.stack([a[s][k][i] for k in keys]) if len(i) else np.zeros((3, 0))
            v = np.stack([b[s][k][j] for k in keys]) if len(j) else np.zeros((3, 0))
            assert np.max(np.linalg.norm(u - v, axis=0) / np.maximum(np.linalg.norm(v, axis=0), 1e-2), initial=0.0) < tol


def test_out_of_room_restores():
    sp = [_leptons(3000, 1), W._empty(), W._empty()]
    g = q.Generator(q.make_config(precision=q.QED_FP32, seed=4, push_photons=0))
    field = q.make_field(W.FIELD_UNIFORM, [0, 0, 0, 0, 0, 900.0])
    ens = q.DeviceEnsemble.from_host(sp, [3000, 8, 16], q.QED_FP32)
    before = ens.to_host(0)
    P = ens.struct()
    rc, st = q.qed_push_and_generate(g.ctx, P, field, W.TWO_PI / 100, STEPS, 2)
    ens.pull_counts(P)
    assert rc == q.QED_ERR_CAPACITY and st["needed_capacity"][2] > 16 and ens.count == [3000, 0, 0]
    after = ens.to_host(0)
    assert all(np.array_equal(before[k], after[k]) for k in before)
    g.push(ens, field, W.TWO_PI / 100, STEPS, 2)             # grows and replays
    ref, _ = _run(sp, q.QED_FP32, field, "one", [3000, 8, 20000])
    g.close()
    i, j = np.argsort(ens.to_host(2)["id"]), np.argsort(ref[2]["id"])
    assert np.array_equal(ens.to_host(2)["px"][i], ref[2]["px"][j])
