"""Emission runs of several steps whose photons run out of room.  Without a
snapshot every lepton stands at the end of the step in which that happened, as
after the same steps taken one by one; with one, the demand is that of the whole
call, whatever the timing of its blocks."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

STEPS = 6
STATS = ("particle_steps", "lepton_steps", "emit_events", "max_subevents", "needed_capacity", "chi_fp64")


def _run(prec, n, room, calls, restore):
    """(status, statistics, electrons) of STEPS steps in one batch."""
    w = W.uniform_b_emission(n=n, seed=3, chi0=1.0, steps_per_period=100, nsteps=STEPS)
    g = q.Generator(q.make_config(precision=prec, seed=3, push_photons=0, restore_on_overflow=restore))
    ens = q.DeviceEnsemble.from_host(w.species, [n, 4, room], prec)
    field = q.make_field(w.field_kind, w.field_prm)
    for k in range(0, STEPS, 1 if calls == "each" else STEPS if calls == "one" else STEPS // 2):
        g.push_async(ens, field, w.dt, {"each": 1, "one": STEPS, "halves": STEPS // 2}[calls], k)
    rc = q.QED_OK
    try:
        st = g.wait(ens)
    except q.QedError as e:
        rc, st = e.status, e.stats
    out = ens.to_host(0)
    g.close()
    return rc, st, out, list(ens.count)


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("n", [700, 120001])
@pytest.mark.parametrize("calls", ["one", "halves"])
def test_without_a_snapshot_all_stop_at_the_same_step(prec, n, calls):
    _, full, _, _ = _run(prec, n, n, "each", 0)
    room = int(0.4 * full["emit_events"])                    # runs out in the third of six steps
    rc1, st1, e1, n1 = _run(prec, n, room, "each", 0)
    rc, st, e, c = _run(prec, n, room, calls, 0)
    assert rc1 == rc == q.QED_ERR_CAPACITY and c == n1
    assert st1["particle_steps"] == 3 * n and st1["needed_capacity"][2] > room
    for k in STATS:
        assert st[k] == st1[k], k
    for k in e:
        assert np.array_equal(e[k], e1[k]), k


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("n", [700, 60001])                  # few enough for all steps to be taken in one launch
def test_with_a_snapshot_the_demand_is_that_of_the_call(prec, n):
    rc0, full, _, c0 = _run(prec, n, n, "one", 1)
    assert rc0 == q.QED_OK
    w = W.uniform_b_emission(n=n).species[0]
    for room in (8, int(0.4 * c0[2]), c0[2] - 1):
        rc, st, e, c = _run(prec, n, room, "one", 1)
        assert rc == q.QED_ERR_CAPACITY and c == [n, 0, 0]
        assert st["needed_capacity"][2] == c0[2]
        for k in ("particle_steps", "lepton_steps", "emit_events", "max_subevents"):
            assert st[k] == full[k], k
        assert all(np.array_equal(e[k], w[k]) for k in ("x", "px", "py", "pz", "id"))
    # a later call of the batch does nothing more
    rc, st, _, c = _run(prec, n, 8, "halves", 1)
    assert rc == q.QED_ERR_CAPACITY and c == [n, 0, 0] and st["particle_steps"] == n * STEPS // 2
