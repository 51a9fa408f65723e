"""qed_batch_push: the photons of every ensemble are recorded in that
ensemble's own arrays, also where a block works on tiles of several ensembles
at once.  Each ensemble's photons equal those of a call with it alone."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


def _push(gen, ws, prec, steps):
    ens = [q.DeviceEnsemble.from_host(w.species, [len(w.species[0]["id"]), 1, 60 * len(w.species[0]["id"]) + 64], prec)
           for w in ws]
    arr, fields = (q.QedParticles * len(ws))(), (q.QedFieldDesc * len(ws))()
    for k, e in enumerate(ens):
        arr[k] = e.struct()
        fields[k] = q.make_field(ws[k].field_kind, ws[k].field_prm)
    rc, st = q.qed_batch_push(gen.ctx, arr, fields, ws[0].dt, steps, 0)
    assert rc == q.QED_OK
    for k, e in enumerate(ens):
        e.pull_counts(arr[k])
    return [e.to_host(2) for e in ens], st


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("n_ens", [2, 400])
def test_photons_stay_with_their_ensemble(prec, n_ens):
    ws = W.batched_uniform_b(n_ens=n_ens, seed=6, size_lo=30, size_hi=3000, chi_lo=0.3, chi_hi=30.0)
    g = q.Generator(q.make_config(precision=prec, seed=8, push_photons=0))
    together, st = _push(g, ws, prec, 5)          # 400: more tiles than resident blocks, so blocks mix ensembles
    assert st["emit_events"] == sum(len(p["id"]) for p in together)
    for k in range(0, n_ens, 1 + n_ens // 40):
        (alone,), _ = _push(g, [ws[k]], prec, 5)
        i, j = np.argsort(together[k]["id"]), np.argsort(alone["id"])
        assert len(i) == len(j), k
        for f in ("id", "px", "py", "pz", "x", "w"):
            assert np.array_equal(together[k][f][i], alone[f][j]), (k, f)
    g.close()
