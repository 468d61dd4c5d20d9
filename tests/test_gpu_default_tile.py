"""The tile a new lattice starts with: valid at every size, and the bits of any other tile."""
import numpy as np
import pytest

import workloads as W
from paper_0911_0459_gb300 import (STORAGE_F16_BLOCKED, STORAGE_F16DEV, STORAGE_F32, STORAGE_F32_BLOCKED,
                                   STORAGE_F64, STORAGE_MOMENTS, Lattice)

pytestmark = pytest.mark.gpu


# narrow and low lattices, rows that fill half a tile, rows that are no multiple of 8, one wave, many waves
@pytest.mark.parametrize("nx,ny", [(8, 700), (65, 12), (130, 9), (257, 40), (700, 40), (2048, 64), (4096, 200)])
@pytest.mark.parametrize("model,storage", [(W.LG, STORAGE_F64), (W.BINARY, STORAGE_F64), (W.BINARY, STORAGE_F32),
                                           (W.BINARY, STORAGE_F32_BLOCKED), (W.BINARY, STORAGE_F16_BLOCKED),
                                           (W.BINARY, STORAGE_F16DEV), (W.BINARY, STORAGE_MOMENTS)])
def test_default_tile_is_valid_and_gives_the_same_bits(nx, ny, model, storage):
    p = W.lg_params(storage=storage) if model == W.LG else W.binary_params(nu_l=0.5, nu_g=0.05, storage=storage)
    cap = W.Capillary("t", nx, ny, nx // 2, nx - nx // 2, 1, ny - 3, 2, 3, p, wall_grad=-0.1)
    a, b = Lattice.from_workload(cap), Lattice.from_workload(cap)
    tx, ty = a.tile()
    assert tx in (64, 128, 256) and 1 <= ty <= ny and (tx == 64 or nx > tx // 2)
    b.set_tile(128, min(16, ny))
    a.step(67)  # a replayed graph and single launches
    b.step(67)
    assert np.array_equal(a.moments(), b.moments()), (tx, ty)
    a.close()
    b.close()
