"""The two forms of the sliding-window variant where one gives way to the other (needs a GPU)."""
import numpy as np
import pytest

import workloads as W
from paper_0911_0459_gb300 import STORAGE_F16DEV, STORAGE_F32, STORAGE_F64, Lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


# bands on both sides of the strips' second wave: 64 and 128 columns on the 2304-wide lattice,
# CTAs of 256 on the 1024-wide one
@pytest.mark.parametrize("nx,ny,tiles", [(2304, 128, ((64, 3), (64, 4), (128, 4), (256, 4))),
                                         (1024, 64, ((256, 1), (256, 2), (128, 2)))])
@pytest.mark.parametrize("model,storage", [(W.BINARY, STORAGE_F32), (W.BINARY, STORAGE_F16DEV), (W.LG, STORAGE_F32),
                                           (W.BINARY, STORAGE_F64), (W.LG, STORAGE_F64)])
def test_every_tile_of_the_sliding_window_gives_the_bits_of_the_staged_kernel(nx, ny, tiles, model, storage):
    p = W.lg_params(storage=storage) if model == W.LG else W.binary_params(nu_l=0.5, nu_g=0.05, storage=storage)
    cap = W.Capillary("t", nx, ny, nx // 2, nx - nx // 2, 1, ny - 3, 8, 3, p, wall_grad=-0.1)
    ref = Lattice.from_workload(cap)
    ref.set_kernel(2)
    ref.set_tile(128, 16)
    ref.step(7)
    want = ref.moments()
    for tx, ty in tiles:
        lat = Lattice.from_workload(cap)
        lat.set_kernel(1)
        lat.set_tile(tx, ty)
        lat.step(7)
        assert np.array_equal(lat.moments(), want), (tx, ty)
        lat.close()
    ref.close()
