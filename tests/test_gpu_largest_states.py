"""Node addresses of the planar step kernels at the largest lattices (needs a GPU, about 12 GB of
host memory)."""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from paper_0911_0459_gb300 import STORAGE_F32, Lattice
from paper_0911_0459_gb300.lb import _check, library

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

NX, NY, SEAM = 65536, 7282, 12
PX, PY = 97, 89  # periods of the state; neither divides 65536


@pytest.fixture(scope="module")
def state():
    """Density and velocity that differ between any two nodes whose distance is not a multiple of
    both periods."""
    rng = np.random.default_rng(7)
    x, y = np.arange(NX) % PX, np.arange(NY) % PY
    rho, u = 3.4 + 0.1 * rng.random((PY, PX)), 0.02 * (rng.random((PY, PX)) - 0.5)
    out = [np.empty((NY, NX)), np.empty((NY, NX))]
    for full, table in zip(out, (rho, u)):
        rows = np.ascontiguousarray(table[:, x])
        for r in range(NY):
            full[r] = rows[y[r]]
    return out


def stepped(rho, u, kernel):
    ny = rho.shape[0]
    lat = Lattice.from_workload(W.periodic_box(NX, ny, W.lg_params(storage=STORAGE_F32)))
    lat.set_kernel(kernel)
    lat.init_fields(rho, u, u)
    lat.step(2)
    out = np.empty((ny, NX))
    _check(library().lb_fields(lat.h, out.ctypes.data_as(C.c_void_p), None, None, None), lat.h)
    lat.close()
    torch.cuda.empty_cache()
    return out


# 65536 x 7281 is the last lattice of the 32-bit offsets (9 N < 2^32): strips (1) and the staged
# kernel (2); one more row runs the shared window
@pytest.mark.parametrize("ny,kernel", [(7281, 1), (7281, 2), (7282, 1)])
def test_rows_at_the_end_of_the_largest_lattices(state, ny, kernel):
    """The first populations take in the rows beside their own and a step moves nothing further than
    two rows, so after two steps the rows around the seam equal, bit for bit, those of a small
    lattice made of the last and the first rows, but for its outer five."""
    rho, u = (a[:ny] for a in state)
    around = [np.ascontiguousarray(np.concatenate((a[-SEAM:], a[:SEAM]))) for a in (rho, u)]
    want = stepped(*around, kernel=2)
    got = stepped(rho, u, kernel)
    inner = slice(5, 2 * SEAM - 5)
    seen = np.concatenate((got[-SEAM:], got[:SEAM]))
    assert np.isfinite(want).all() and np.array_equal(seen[inner], want[inner])
    assert len(np.unique(want[inner])) > 1000
    # and rows in the middle, which hold the same values as others a period away
    mid = ny // 2
    assert np.array_equal(got[mid:mid + 5], got[mid + PY:mid + PY + 5])
