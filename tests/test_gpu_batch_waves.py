"""FP16-block sweeps with a little more tiles than one wave of CTAs holds (needs a GPU)."""
import numpy as np
import pytest

import workloads as W
from paper_0911_0459_gb300 import STORAGE_F16_BLOCKED, Batch, Lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


# rows on block boundaries and inside blocks; 510 and 684 tiles, 1.12 waves of three and four CTAs an SM
@pytest.mark.parametrize("nx", [1280, 1276])
@pytest.mark.parametrize("tx,n", [(128, 17), (64, 12)])
@pytest.mark.parametrize("variant", [2, 3])
def test_the_body_for_more_ctas_gives_the_bits_of_single_lattices(nx, tx, n, variant):
    caps = [W.Capillary("b", nx, 24, 160, nx - 160, 1, 22, 32, 10, W.binary_params(nu_l=0.5, nu_g=0.05 + 0.01 * k),
                        theta_deg=45.0 + k) for k in range(n)]
    b = Batch(caps, storage=STORAGE_F16_BLOCKED)
    b.set_kernel(variant)
    b.set_tile(tx, 8)
    b.step(9)
    for k in (0, n // 2, n - 1):
        lat = Lattice.from_workload(caps[k], storage=STORAGE_F16_BLOCKED)
        lat.step(9)
        for x, y in zip(b.populations(k, rested=False), lat.populations(rested=False)):
            assert np.array_equal(x, y), k
        lat.close()
    b.close()
