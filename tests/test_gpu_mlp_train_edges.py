"""Training and gradients of the opening-angle network at the edges of the
cluster kernel's split: batches that are not whole 16-sample tiles, fewer
tiles than blocks, more than one tile per block, and more steps than one
launch covers, against the FP64 oracle with the same BF16 operands.

Tolerances: gradients as in the main test (2e-2 of a block's norm, BF16
operands).  After k Adam steps a parameter may differ by a rounding flip's
effect on the update direction; the training test bounds the summed loss of
every epoch (1 %) and the parameters' distance by 5 % of the distance
travelled.  Over the 520 steps that pass a launch's end the two trajectories
would part at a training rate, so that case takes a rate that moves each
parameter by at most 520 x 2e-6 = 1e-3: the network, and with it the
gradients, then stay those of the start to about 1 %.
"""
import numpy as np
import pytest

from oracle import mlp
from tests.test_gpu_mlp import BLOCKS, data, params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("n", [1, 15, 17, 255, 257, 600])
def test_gradient_of_ragged_batches(n):
    import paper_0909_0541_gb300 as nb
    p = params(5)
    f, y = data(n, 40 + n)
    g, loss = nb.mlp_grad(_dev(p), _dev(f), _dev(y))
    L, want = mlp.backward(p, f[:, :12], y, bf=True)
    assert abs(loss.item() / n - L) <= 1e-3 * L + 1e-9
    g = g.cpu().numpy()
    for name, a, b in BLOCKS:
        err = np.linalg.norm(g[a:b] - want[a:b]) / max(np.linalg.norm(want[a:b]), 1e-12)
        assert err < 2e-2, (name, err)
    assert not g[9472:9920].any() and not g[9921:].any()   # unused slots, mean and spread


@pytest.mark.parametrize("n,batch,epochs", [(50, 16, 2), (230, 100, 3), (700, 300, 2),
                                            (64, 16, 130)])
def test_training_follows_the_oracle(n, batch, epochs):
    import paper_0909_0541_gb300 as nb
    p0 = params(6)
    f, y = data(n, 50 + n)
    rng = np.random.default_rng(n)
    order = np.stack([rng.permutation(n) for _ in range(epochs)]).astype(np.int32)
    # parameters at an odd offset: no alignment is asked of them
    buf = torch.zeros(len(p0) + 1, dtype=torch.float32, device="cuda")
    P = buf[1:]
    P.copy_(_dev(p0))
    lr = 1e-3 if epochs < 100 else 2e-6
    hist = nb.mlp_train(P, _dev(f), _dev(y), _dev(order), epochs, batch, lr).cpu().numpy()
    p, m, v, t = p0.astype(np.float64), np.zeros(len(p0)), np.zeros(len(p0)), 0
    want = np.zeros(epochs)
    for e in range(epochs):
        for k in range(n // batch):
            i = order[e, k * batch:(k + 1) * batch]
            L, g = mlp.backward(p, f[i, :12], y[i], bf=True)
            want[e] += L * batch
            t += 1
            p, m, v = mlp.adam(p, m, v, g, t, lr)
    assert np.allclose(hist, want, rtol=1e-2), (hist[-1], want[-1])
    got = P.cpu().numpy().astype(np.float64)
    used = np.r_[0:9472, 9920:9921]
    moved = np.linalg.norm((p - p0)[used])
    assert np.linalg.norm((got - p)[used]) <= 5e-2 * moved
    rest = np.r_[9472:9920, 9921:len(p0)]
    assert np.array_equal(got[rest], p0[rest].astype(np.float64))
