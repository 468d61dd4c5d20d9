"""The network's kernels at the edges of their tiles, against the FP64 reference.

The fused row tiles hold 16 or 48 rows and serve n_hidden <= 256 as far as the weights fit in
shared memory; other networks run one GEMM per product.  The weight gradients are accumulated
by whole tiles or left in split-K parts.  Sizes: one row, tiles one short and one over, outputs
that fill no step of 16, odd numbers of inputs, every n_hidden / 64, the first shapes that no
longer fit.  Tolerance: with weights and inputs that BF16 holds exactly five roundings to BF16
remain (h1, h2, dY, dZ2, dZ1), each at most 2^-9 relative and at most doubled on its way through
the tanh derivative, so a gradient is within 5 * 2^-8 = 2e-2 (L2, per tensor)."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0911_0459_gb300.mlp import MLP, _lib, _ptr  # noqa: E402
from test_gpu_mlp import bf16_round  # noqa: E402


@pytest.mark.parametrize("nin,nh,nout,members,n", [
    (4, 256, 64, 5, 1), (4, 256, 64, 5, 1457), (3, 256, 88, 2, 47), (16, 256, 128, 1, 33), (1, 256, 136, 1, 17),
    (5, 192, 8, 3, 49), (7, 128, 24, 16, 300), (2, 64, 200, 1, 95), (4, 320, 40, 2, 129), (16, 1024, 8, 1, 65)])
def test_gradients_and_predictions_at_the_edges_of_the_tiles(nin, nh, nout, members, n):
    rng = np.random.default_rng(nh + nout + n)
    net = MLP(nin, nh, nout, members=members, max_batch=n + 3, seed=1)
    x = bf16_round(rng.uniform(-1, 1, (n, nin)))
    y = rng.normal(0, 1, (n, nout)).astype(np.float32)
    params = [bf16_round(net.get_params(k) + rng.normal(0, 0.02, net.P).astype(np.float32)) for k in range(members)]
    for k, p in enumerate(params):
        net.set_params(k, p)
    net.set_data(x, y)
    _, _, out = net.predict(x, members=True)
    for k in {0, members - 1}:
        p = params[k].astype(np.float64)
        loss, g = net.gradients(k)
        rloss, rg = ref.loss_and_grads(p, x.astype(np.float64), y, nin, nh, nout)
        assert abs(loss / rloss - 1) < 2e-2
        for name, a, b in zip(("W1", "b1", "W2", "b2", "W3", "b3"), ref.unpack(g, nin, nh, nout),
                              ref.unpack(rg, nin, nh, nout)):
            err = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert err < 2e-2, (k, name, err)
        yr, _ = ref.forward(p, x.astype(np.float64), nin, nh, nout)
        assert np.linalg.norm(out[k] - yr) < 2e-2 * np.linalg.norm(yr)
    net.close()


@pytest.mark.parametrize("nin,nh,nout,members,n", [
    (4, 256, 64, 5, 8192), (4, 256, 64, 5, 20011), (3, 64, 200, 1, 14593), (16, 192, 24, 16, 45000), (2, 128, 8, 7, 70000)])
def test_large_predictions_equal_those_of_their_rows(nin, nh, nout, members, n):
    """Results above 4 MB reach host arrays that exist in parts; a row's outputs do not depend
    on the rows beside it, so they are the bytes that short predictions give (no tolerance)."""
    rng = np.random.default_rng(n)
    net = MLP(nin, nh, nout, members=members, max_batch=n, seed=2)
    x = rng.uniform(-1, 1, (n, nin)).astype(np.float32)
    out = [np.full((n, nout), np.nan, np.float32), np.full((n, nout), np.nan, np.float32),
           np.full((members, n, nout), np.nan, np.float32)]
    assert _lib().lb_mlp_predict(net.h, n, _ptr(x), *(_ptr(a) for a in out)) == 0
    fresh = net.predict(x, members=True)
    for a, b in zip(out, fresh):
        assert np.array_equal(a, b)
    for r in (0, n // 3, n // 2 - 7, n - 301):
        mean, sd, each = net.predict(x[r:r + 301], members=True)
        assert np.array_equal(mean, out[0][r:r + 301]) and np.array_equal(sd, out[1][r:r + 301])
        assert np.array_equal(each, out[2][:, r:r + 301])
    net.close()
