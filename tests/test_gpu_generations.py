"""qed_stats.passes is the depth of the step's avalanche (generations of
newborns), whatever a full block list leaves to further launches and in which
order: the depth of the deepest of the same electrons pushed a few at a time,
where no list fills, and the least pass_limit with which the step completes."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

CAP = 2000000


@pytest.mark.parametrize("prec,n", [(q.QED_FP64, 1000), (q.QED_FP32, 1000)])
@pytest.mark.parametrize("profile", [0, 1])
def test_depth_does_not_depend_on_the_launches(prec, n, profile):
    w = W.uniform_b_emission(n=n, seed=5, p0=1e5, chi0=300.0, steps_per_period=1, nsteps=1)
    field = q.make_field(w.field_kind, w.field_prm)

    def push(sel, ens, **cfg):
        g = gens.setdefault(tuple(cfg.items()), None) or q.Generator(q.make_config(precision=prec, seed=w.seed, profile=profile, **cfg))
        gens[tuple(cfg.items())] = g
        e = w.species[0]
        for k in ens.arr[0]:
            if k in e:
                v = e[k][sel]
                ens.arr[0][k][:len(v)].copy_(torch.from_numpy(v.view(np.int64) if k == "id" else v))
        ens.arr[0]["nevents"].zero_()
        ens.count = [len(e["id"][sel]), 0, 0]
        P = ens.struct()
        try:
            return q.qed_push_and_generate(g.ctx, P, field, w.dt, 1, 0)
        except q.QedError as err:
            return err.status, None

    gens = {}
    few = q.DeviceEnsemble([20000] * 3, prec)
    alone = [push(slice(i, i + 8), few)[1] for i in range(0, n, 8)]
    depth = max(st["passes"] for st in alone)
    ens = q.DeviceEnsemble([CAP] * 3, prec)
    for _ in range(4):
        rc, st = push(slice(None), ens)
        assert rc == q.QED_OK and st["pair_events"] == sum(a["pair_events"] for a in alone)
        assert st["launches"] > alone[0]["launches"]             # some pairs took further launches
        assert st["passes"] == depth >= 3
    assert push(slice(None), ens, pass_limit=depth)[0] == q.QED_OK
    assert push(slice(None), ens, pass_limit=depth - 1)[0] == q.QED_ERR_TIMEOUT
    for g in gens.values():
        g.close()
