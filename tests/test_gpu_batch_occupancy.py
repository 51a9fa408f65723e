"""qed_batch_push in FP32 has two copies of its kernel per block shape: one for
calls with at most one tile per block, one with more warps per SM beyond that.
A particle's result does not depend on the copy: the same leptons pushed in one
call around that limit and in small calls end bit for bit the same."""
import numpy as np
import pytest

from paper_2409_17299_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


def _push(gen, w, sl, steps):
    sp = [{k: v[sl] for k, v in w.species[0].items()}, w.species[1], w.species[2]]
    n = len(sp[0]["id"])
    e = q.DeviceEnsemble.from_host(sp, [n, 1, 8 * n + 64], q.QED_FP32)
    arr, fields = (q.QedParticles * 1)(e.struct()), (q.QedFieldDesc * 1)(q.make_field(w.field_kind, w.field_prm))
    rc, _ = q.qed_batch_push(gen.ctx, arr, fields, w.dt, steps, 0)
    assert rc == q.QED_OK
    e.pull_counts(arr[0])
    return e.to_host(0)


# blocks per SM of the first copy (at most): 128 threads 7, 256 threads 2, 512 threads 1
@pytest.mark.parametrize("threads,per_sm", [(128, 7), (256, 2), (512, 1)])
@pytest.mark.parametrize("extra", [0, 1])
def test_copies_agree(threads, per_sm, extra):
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm * threads + extra
    (w,) = W.batched_uniform_b(n_ens=1, seed=3, size_lo=n, size_hi=n, chi_lo=1.0, chi_hi=3.0)
    total = len(w.species[0]["id"])
    assert abs(total - n) <= 1
    g = q.Generator(q.make_config(precision=q.QED_FP32, seed=4, push_photons=0, block_threads=threads))
    whole = _push(g, w, slice(0, total), 6)
    parts = [_push(g, w, slice(a, min(a + total // 3, total)), 6) for a in range(0, total, total // 3)]
    i = np.argsort(whole["id"])
    j = np.argsort(np.concatenate([p["id"] for p in parts]))
    assert whole["nevents"].sum() > n // 4
    for f in ("id", "x", "y", "z", "px", "py", "pz", "nevents"):
        assert np.array_equal(whole[f][i], np.concatenate([p[f] for p in parts])[j]), f
    g.close()
