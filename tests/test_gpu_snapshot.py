"""The state copied aside when a call opens comes back after an overflow, array
by array, at sizes that are no multiple of 16 bytes and with optical-depth
arrays that are only aligned to their elements."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("sizes", [(1, 0, 3), (1023, 4097, 70001)])
@pytest.mark.parametrize("method", [q.QED_METHOD_SUBSTEP, q.QED_METHOD_OPTICAL_DEPTH])
def test_overflow_restores_every_array(prec, sizes, method):
    r = np.random.default_rng(1)
    sp = []
    for s, n in enumerate(sizes):
        d = {k: r.normal(0, 300.0, n).astype(np.float32).astype(float) for k in ("x", "y", "z", "px", "py", "pz")}
        d.update(w=np.ones(n), id=np.arange(n, dtype=np.uint64) + (s << 40),
                 nevents=r.integers(0, 5, n).astype(np.uint32), od=r.uniform(1e-6, 1e-5, n))
        sp.append(d)
    g = q.Generator(q.make_config(precision=prec, seed=2, event_method=method))
    cap = [sizes[0] + 2, sizes[1] + 2, sizes[2]]             # no room for a photon
    ens = q.DeviceEnsemble.from_host(sp, cap, prec, optical_depth=True)
    for s in range(3):                                       # one element past a 16-byte boundary
        od = torch.zeros(cap[s] + 1, dtype=ens.fdtype, device="cuda")[1:]
        od.copy_(ens.arr[s]["od"])
        ens.arr[s]["od"] = od
    before = [ens.to_host(s) for s in range(3)]
    g._bind(ens)
    P = ens.struct()
    rc, _ = q.qed_push_and_generate(g.ctx, P, q.make_field(W.FIELD_UNIFORM, [0, 0, 0, 0, 900.0, 2e6]), 0.5, 3, 0)
    assert rc == q.QED_ERR_CAPACITY
    ens.pull_counts(P)
    assert ens.count == list(sizes)
    for s in range(3):
        after = ens.to_host(s)
        assert all(np.array_equal(before[s][k], after[k]) for k in before[s]), s
    g.close()
