"""Networks of one n_hidden and different n_out, used from two threads at once (needs a GPU)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0911_0459_gb300.mlp import MLP  # noqa: E402


def test_two_threads_with_networks_that_share_their_kernels():
    """Each thread's calls succeed and predictions are the bytes that they give alone (a row's
    outputs depend on nothing but its inputs and the weights)."""
    rng = np.random.default_rng(0)
    x = rng.uniform(-1, 1, (2048, 4)).astype(np.float32)
    nets = [MLP(4, 256, nout, members=4, max_batch=2048, seed=3, stream=torch.cuda.Stream()) for nout in (128, 8)]
    alone = [[net.predict(x[:n]) for n in (16, 2048)] for net in nets]
    errors = []

    def use(net, ref):
        try:
            for k in range(300):
                for n, r in zip((16, 2048), ref):
                    got = net.predict(x[:n])
                    if not (np.array_equal(got[0], r[0]) and np.array_equal(got[1], r[1])):
                        raise AssertionError(f"predictions of {n} rows differ in pass {k}")
            net.set_data(x[:512], np.zeros((512, net.n_out), np.float32))
            for k in range(20):
                if not np.isfinite(net.train(20)).all():
                    raise AssertionError("loss not finite")
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=use, args=a) for a in zip(nets, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for net in nets:
        net.close()
    assert not errors, errors
