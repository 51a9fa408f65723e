"""A wait inside the leveling that runs out (its limit set low enough on
purpose) is reported by every call that levels, changes no particle, and leaves
nothing behind that a later leveling or shard evaluation of the context counts."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

CAP = 50000


def _ensemble(prec, n):
    r = np.random.default_rng(4)
    sp = []
    for s in range(3):
        d = {k: r.normal(0, 1, n).astype(np.float32).astype(float) for k in ("x", "y", "z", "px", "py", "pz")}
        d.update(w=r.integers(1, 9, n) / 8.0, id=np.arange(n, dtype=np.uint64) + (s << 40))
        d["w"][r.random(n) < 0.1] = 0.0
        sp.append(d)
    return q.DeviceEnsemble.from_host(sp, [2 * n] * 3, prec)


def _check_sums(g, ens, s):
    """A shard's sums (weights are multiples of 1/8: exact in any order)."""
    w = ens.to_host(s)["w"]
    A, C, N, M = q.qed_level_eval(g.ctx, ens.struct().s[s], s, 0.7)
    assert (A, C, N, M) == (w[w < 0.7].sum(), int((w >= 0.7).sum()), int((w > 0).sum()), w.max())


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
def test_compact_reports_a_wait_that_ran_out(prec):
    g = q.Generator(q.make_config(precision=prec, thin_cap=CAP, level_polls=1))
    ens = _ensemble(prec, 200003)
    before = [ens.to_host(s) for s in range(3)]
    for rnd in range(3):
        with pytest.raises(q.QedError) as e:
            g.compact(ens, rnd)
        assert e.value.status == q.QED_ERR_TIMEOUT
        for s in range(3):
            after = ens.to_host(s)
            assert all(np.array_equal(before[s][k], after[k]) for k in after)
            _check_sums(g, ens, s)
    g.close()


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("profile", [0, 1])
def test_push_reports_a_wait_that_ran_out(prec, profile):
    w = W.rotating_e_cascade(n=1000, seed=1)
    field = q.make_field(w.field_kind, [1e-3])           # nothing happens to the particles but the leveling
    g = q.Generator(q.make_config(precision=prec, thin_cap=CAP, level_polls=1, profile=profile))
    ens = _ensemble(prec, 200003)
    weights = [ens.to_host(s)["w"] for s in range(3)]
    for rnd in range(2):
        g.push_async(ens, field, w.dt, 2, rnd)
        with pytest.raises(q.QedError) as e:
            g.wait(ens)
        assert e.value.status == q.QED_ERR_TIMEOUT
        for s in range(3):
            assert np.array_equal(ens.to_host(s)["w"], weights[s])
            _check_sums(g, ens, s)
    g.close()
