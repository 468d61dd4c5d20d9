"""The batch's choice of body by its number of tiles, without a GPU (fake_cudart.cpp)."""
from fake_cuda import run


def test_a_sweep_just_over_one_wave_runs_the_body_that_holds_it(tmp_path):
    """FP16 blocks, tiles of 128 columns, three CTAs an SM and five by the second body: 456 tiles
    fill a wave; from a tenth to three tenths more the second body takes all tiles at once, one
    CTA each.  FP32 blocks have no second body."""
    seen = run(tmp_path, r'''
for name, per in ((b"SF16B, 128, 4, false", 3), (b"SF16B, 128, 4, true", 5), (b"SF32B, 128, 4, false", 3)):
    fake.fake_resident(b"batch_tma_kernel<lbk::" + name, per)
seen = []
for st in (lb.STORAGE_F16_BLOCKED, lb.STORAGE_F32_BLOCKED):
    for n in (14, 15, 16, 17, 18, 19, 20, 30):
        caps = [W.Capillary("b", 1280, 24, 160, 1120, 1, 22, 32, 10, W.binary_params(storage=st), theta_deg=45.0)] * n
        s = [lb._structs_for(c) for c in caps]
        h = C.c_void_p()
        assert L.lb_batch_create(n, (lb.LbGrid * n)(*[x[0] for x in s]), (lb.LbWalls * n)(*[x[1] for x in s]),
                                 (lb.LbParams * n)(*[x[2] for x in s]), None, None, C.byref(h)) == 0
        assert L.lb_batch_set_tile(h, 128, 8) == 0
        log()
        assert L.lb_batch_step(h, 2) == 0
        (grid, block, name), = launches("batch_tma_kernel")
        seen.append([st, 30 * n, grid, block, "true" in name.split("(")[0]])
        L.lb_batch_destroy(h)
print(json.dumps(seen))
''')
    for st, tiles, grid, block, many in seen:
        assert block == 160
        assert many == (st == 7 and 1.1 * 456 < tiles <= 1.3 * 456), (st, tiles)
        assert grid == (tiles if many else min(tiles, 456)), (st, tiles)
    assert [t for st, t, _, _, many in seen if many] == [510, 540, 570]
