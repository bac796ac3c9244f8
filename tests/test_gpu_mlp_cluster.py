"""The 8-block form of the training and gradient kernels (two owner slots a
block), which the library takes where a 16-block cluster does not fit, against
the 16-block form.  Both sum every gradient over the batch in sample order
(the output bias and the loss: lane l of a warp the samples l, l + 32, ...), so
gradients, parameters, moments and losses agree bit for bit.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from tests.test_gpu_mlp import data, params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import paper_0909_0541_gb300 as nb
    from paper_0909_0541_gb300 import build as B
    out = str(tmp_path_factory.mktemp("cluster") / "libcluster.so")
    r = subprocess.run([B.nvcc(), *B.NVFLAGS, "-shared", "-Xlinker", "-Bsymbolic", "-o", out,
                        os.path.join(HERE, "mlp_cluster.cu"), nb.library_path(), "-Xlinker",
                        "-rpath=" + os.path.dirname(nb.library_path()), "-lcudart"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    vp, i64, i32 = C.c_void_p, C.c_int64, C.c_int
    L.cluster_train.argtypes = [i32, vp, vp, vp, vp, vp, vp, i64, i32, i64, C.c_float, vp, vp, vp]
    L.cluster_grad.argtypes = [i32, vp, vp, vp, i64, vp, vp, vp, vp]
    return L


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _work():
    import paper_0909_0541_gb300 as nb
    return torch.empty(int(nb._lib.nb_mlp_workspace_size(16)), dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("n", [1, 15, 17, 128, 129, 255, 257, 600])
def test_gradient(lib, n):
    p = _dev(params(5))
    f, y = data(n, 40 + n)
    f, y = _dev(f), _dev(y)
    out = []
    for blocks in (16, 8):
        g = torch.zeros_like(p)
        loss = torch.zeros(1, device="cuda")
        work = _work()
        assert lib.cluster_grad(blocks, p.data_ptr(), f.data_ptr(), y.data_ptr(), n, g.data_ptr(),
                                loss.data_ptr(), work.data_ptr(), None) == 0
        torch.cuda.synchronize()
        out.append((g.cpu().numpy(), loss.item()))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    for a, b in ((0, 1024), (1088, 5184), (5248, 9344), (9408, 9472), (9920, 9921)):
        assert out[0][0][a:b].any()


@pytest.mark.parametrize("n,batch,epochs", [(50, 16, 2), (400, 128, 3), (700, 300, 2),
                                            (64, 16, 70)])
def test_training(lib, n, batch, epochs):
    p0 = params(6)
    f, y = data(n, 50 + n)
    rng = np.random.default_rng(n)
    order = np.stack([rng.permutation(n) for _ in range(epochs)]).astype(np.int32)
    f, y, o = _dev(f), _dev(y), _dev(order)
    out = []
    for blocks in (16, 8):
        p = _dev(p0)
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        loss = torch.zeros(epochs, device="cuda")
        work = _work()
        assert lib.cluster_train(blocks, p.data_ptr(), m.data_ptr(), v.data_ptr(), f.data_ptr(),
                                 y.data_ptr(), o.data_ptr(), n, epochs, batch, 1e-3,
                                 loss.data_ptr(), work.data_ptr(), None) == 0
        torch.cuda.synchronize()
        out.append([t.cpu().numpy() for t in (p, m, v, loss)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert not np.array_equal(out[0][0], p0)
