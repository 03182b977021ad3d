"""A training step after a backward call with a given output gradient: the step's
own output gradient fills 2 dim of the 16 columns and clears the others, so the
update is that of a network that never saw the other call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1911_13255_gb300 as pkg  # noqa: E402
from oracle import mpnn as M  # noqa: E402


@pytest.mark.parametrize("dim,shape,R", [(2, (13, 7), 3), (3, (5, 3, 3), 1)])
def test_train_step_after_backward_equals_a_fresh_one(dim, shape, R):
    rng = np.random.default_rng(5)
    axes = np.meshgrid(*[np.arange(k) for k in shape], indexing="ij")
    r0 = np.stack([a.ravel() for a in axes], 1) * 0.01
    graph = M.build_graph(r0, 0.01, dim)
    theta = M.init_params(dim, seed=1).astype(np.float32)
    rows = R * len(r0)
    x = np.zeros((rows, M.FIN), np.float32)
    x[:, :M.n_features(dim)] = rng.normal(size=(rows, M.n_features(dim)))
    target = rng.normal(size=(rows, M.NOUT)).astype(np.float32)
    out = []
    for given in (True, False):
        net = pkg.Mpnn(dim, graph, replicas=R)
        net.set_params(theta)
        if given:
            net.forward(x)
            net.backward(rng.normal(size=(rows, M.NOUT)))
        out.append((net.train_step(x, target, lr=1e-3), net.get_params()))
        net.close()
    (la, a), (lb, b) = out
    # the loss differs by the order of an FP32 sum
    assert abs(la - lb) <= 1e-5 * abs(lb)
    # Adam's first update is lr in size wherever the gradient is well above its
    # epsilon: only parameters with a gradient of rounding size may differ
    far = np.abs(a.astype(np.float64) - b) > 1e-4
    assert far.mean() < 0.01, far.mean()
