"""The captured step keeps no address of a work buffer that another call on the
same context has replaced: steps of a small ensemble, then a merge of a larger
one (its work buffers grow), then more steps of the small one, against a
context that saw the small one only."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


def _large(prec):
    r = np.random.default_rng(3)
    sp = []
    for s, n in enumerate((900001, 700003, 800002)):
        d = {k: r.normal(0, 1, n) for k in ("x", "y", "z", "px", "py", "pz")}
        d.update(w=np.where(r.random(n) < 0.3, 0.0, 1.0), id=np.arange(n, dtype=np.uint64) + (s << 40))
        sp.append(d)
    return q.DeviceEnsemble.from_host(sp, [900001, 700003, 800002], prec)


def _steps(prec, between):
    w = W.rotating_e_cascade(n=2000, seed=1, thin_cap=0)
    g = q.Generator(q.make_config(precision=prec, seed=w.seed))
    ens = q.DeviceEnsemble.from_host(w.species, [20000, 20000, 200000], prec)
    field = q.make_field(w.field_kind, w.field_prm)
    g.push(ens, field, w.dt, 30, 60, auto_grow=False)
    if between == "compact":
        g.compact(_large(prec), 0)
    elif between == "level":
        big = _large(prec)
        P = big.struct()
        q.qed_level_apply(g.ctx, P, 2, 2.0, 5)
        big.pull_counts(P)
    torch.cuda.synchronize()
    fill = [torch.full((4 << 20,), 7, dtype=torch.int32, device="cuda") for _ in range(4)]   # whoever gets the old buffers
    g.push(ens, field, w.dt, 30, 90, auto_grow=False)
    out = []
    for s in range(3):
        d = ens.to_host(s)
        order = np.argsort(d["id"])
        out.append({k: v[order] for k, v in d.items()})
    g.close()
    assert all(bool((f == 7).all()) for f in fill)
    return out


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("between", ["compact", "level"])
def test_steps_after_a_larger_merge(prec, between):
    for a, b in zip(_steps(prec, None), _steps(prec, between)):
        for k in a:
            assert np.array_equal(a[k], b[k]), k
