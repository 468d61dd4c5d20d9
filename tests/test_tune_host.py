"""lb_autotune's choice with launches of known times, without a GPU (fake_cudart.cpp)."""
import pytest

from fake_cuda import run

TUNE = r'''
h = lattice({nx}, {ny}, W.{model}, {storage})
if {tile}: assert L.lb_set_tile(h, *{tile}) == 0
if {kernel}: assert L.lb_set_kernel(h, {kernel}) == 0
log()
assert L.lb_step(h, 1) == 0
grid, block, name = launches("_kernel")[0]
if {fast}: grid, block, name = {fast}
fake.fake_cost(name.split("<")[0].split()[-1].encode(), grid, block, 7.0)  # every other launch: 10
before = [tile(h), kernel(h)]
a, b, us = C.c_int(), C.c_int(), C.c_double()
assert L.lb_autotune(h, C.byref(a), C.byref(b), C.byref(us)) == 0
print(json.dumps([before, [tile(h), kernel(h)], [a.value, b.value], us.value]))
'''


def tune(tmp_path, nx, ny, model, storage, tile=None, kernel=0, fast=None):
    return run(tmp_path, TUNE.format(nx=nx, ny=ny, model=model, storage=storage, tile=tile, kernel=kernel, fast=fast))


@pytest.mark.parametrize("nx,ny,model,storage,tile,kernel", [
    (256, 32, "BINARY", "lb.STORAGE_MOMENTS", None, 0),        # as created: one row, no candidate
    (1000, 200, "BINARY", "lb.STORAGE_F32", None, 0),          # as created: three rows
    (704, 40, "BINARY", "lb.STORAGE_F32", (64, 3), 0),         # as set
    (704, 40, "LG", "lb.STORAGE_F64", (128, 10), 2),
    (704, 40, "BINARY", "lb.STORAGE_F16_BLOCKED", (128, 6), 3)])
def test_the_choice_in_use_is_kept_unless_a_candidate_is_faster(tmp_path, nx, ny, model, storage, tile, kernel):
    before, after, told, us = tune(tmp_path, nx, ny, model, storage, tile, kernel)
    assert after == before and told == before[0] and us == pytest.approx(7.0)


@pytest.mark.parametrize("nx,ny,storage,fast,best", [
    (256, 32, "lb.STORAGE_MOMENTS", (3 * 8, 128, "lbk::moment_step_kernel<"), [[128, 4], 4]),
    (704, 40, "lb.STORAGE_F32", (6 * 5, 160, "lbk::step_tma_kernel<"), [[128, 8], 2])])
def test_a_faster_candidate_is_taken(tmp_path, nx, ny, storage, fast, best):
    _, after, told, us = tune(tmp_path, nx, ny, "BINARY", storage, fast=fast)
    assert after == best and told == best[0] and us == pytest.approx(7.0)
