"""The gradient sum over the CTAs has a fixed order, so training and gradient
calls of the same inputs give the same bits every time: with one CTA, with few
(a thread holds several groups of parameters), with several threads to a group,
and with a CTA on every SM and two tiles each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2409_17299_gb300 as q  # noqa: E402


@pytest.mark.parametrize("batch", [128, 384, 640, 8192, 19456, 38912])
def test_training_twice_gives_the_same_bits(batch):
    runs = []
    for _ in range(2):
        g = q.Generator(q.make_config(precision=q.QED_FP32, seed=1))
        for _ in range(2):
            loss = q.qed_train_surrogate(g.ctx, 24 * batch, batch, 4e-3, 78)
            runs.append((loss, q.qed_mlp_get_params(g.ctx)))
        g.close()
    for loss, P in runs[1:]:
        assert loss == runs[0][0]
        assert np.array_equal(P, runs[0][1])


@pytest.mark.parametrize("n", [1, 129, 20000])
def test_gradient_twice_gives_the_same_bits(n):
    g = q.Generator(q.make_config(precision=q.QED_FP32, seed=1))
    r = np.random.default_rng(n)
    q.qed_mlp_set_params(g.ctx, r.normal(0, 0.2, q.MLP_NPARAMS))
    feat = torch.from_numpy(r.uniform(-1, 1, (n, 2)).astype(np.float32)).cuda()
    target = torch.from_numpy(r.uniform(0, 1, n).astype(np.float32)).cuda()
    runs = [q.qed_mlp_grad(g.ctx, feat.data_ptr(), target.data_ptr(), n) for _ in range(4)]
    g.close()
    for grad, loss in runs[1:]:
        assert loss == runs[0][1]
        assert np.array_equal(grad, runs[0][0])
