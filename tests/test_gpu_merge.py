"""The merge step over all species at once (one launch per pass): removal of
dead entries entry by entry at the edges of its tiles (4096 entries) and of
its scan (1024 tiles), and leveling of several species in one launch against
the defining equation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402

FIELDS = ("x", "y", "z", "px", "py", "pz", "w")


def _species(n, dead, seed, prec):
    r = np.random.default_rng(seed)
    f = np.float32 if prec == q.QED_FP32 else np.float64
    d = {k: r.standard_normal(n).astype(f).astype(np.float64) for k in FIELDS[:6]}
    d["w"] = r.uniform(0.5, 2.0, n).astype(f).astype(np.float64)
    if n:
        d["w"][r.random(n) < dead] = 0.0
    d["id"] = r.permutation(n).astype(np.uint64)
    d["nevents"] = r.integers(0, 9, n).astype(np.uint32)
    return d


def _expected(d):
    """The r-th dead slot below the alive count takes the r-th alive entry at or above it."""
    alive = d["w"] > 0
    a = int(alive.sum())
    holes, movers = np.nonzero(~alive[:a])[0], a + np.nonzero(alive[a:])[0]
    out = {k: v[:a].copy() for k, v in d.items()}
    for k in out:
        out[k][holes] = d[k][movers]
    return out


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
@pytest.mark.parametrize("sizes,dead", [((0, 1, 4095), 0.3), ((4096, 4097, 8193), 0.5), ((1, 4095, 0), 1.0),
                                        ((70000, 12289, 4096), 0.02), ((3, 1024 * 4096 + 5, 4097), 0.3)])
def test_removal_over_all_species(prec, sizes, dead):
    sp = [_species(n, dead, 10 + s, prec) for s, n in enumerate(sizes)]
    g = q.Generator(q.make_config(precision=prec))
    ens = q.DeviceEnsemble.from_host(sp, [n + 8 for n in sizes], prec)
    g.compact(ens, 0)
    g.close()
    for s in range(3):
        want, got = _expected(sp[s]), ens.to_host(s)
        assert ens.count[s] == len(want["id"])
        for k in want:
            assert np.array_equal(got[k], want[k]), (s, k)


@pytest.mark.parametrize("prec", [q.QED_FP32, q.QED_FP64])
def test_leveling_of_several_species_in_one_launch(prec):
    """Electrons and photons above the cap, positrons below it (left alone).
    Each leveled species ends within six standard deviations of the cap (a
    sum of independent keep decisions), with weights w* below and unchanged
    above the threshold of the defining equation; twice, so that the second
    iteration starts at a warm start."""
    cap, sizes = 50000, (120001, 40000, 200003)
    g = q.Generator(q.make_config(precision=prec, thin_cap=cap, seed=3))
    for rnd in range(2):
        sp = [_species(n, 0.05, 20 + 3 * rnd + s, prec) for s, n in enumerate(sizes)]
        ens = q.DeviceEnsemble.from_host(sp, sizes, prec)
        g.compact(ens, rnd)
        for s in range(3):
            w0 = {int(i): v for i, v in zip(sp[s]["id"], sp[s]["w"]) if v > 0}
            got = ens.to_host(s)
            assert set(map(int, got["id"])) <= set(w0)
            before = np.array([w0[int(i)] for i in got["id"]])
            if len(w0) <= cap:
                assert ens.count[s] == len(w0) and np.array_equal(got["w"], before)
                continue
            w = np.array(list(w0.values()))
            lo, hi = w.min(), w.sum() / cap * 4
            for _ in range(200):                    # sum min(1, w / t) falls with t
                t = 0.5 * (lo + hi)
                lo, hi = (t, hi) if np.minimum(1.0, w / t).sum() > cap else (lo, t)
            assert abs(ens.count[s] - cap) < 6 * np.sqrt(cap)
            tol = 1e-6 if prec == q.QED_FP32 else 1e-12
            assert np.allclose(got["w"], np.maximum(before, t), rtol=tol, atol=0)
    g.close()
