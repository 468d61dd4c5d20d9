"""The step kernel behind the automatic choice, by lattice and tile, without a GPU (fake_cudart.cpp)."""
import json
import os
import subprocess

from fake_cuda import ROOT, run


def test_tall_bands_on_small_block_lattices_run_the_staged_kernel(tmp_path):
    """A tile given to a small lattice under the automatic choice.  In the block storages the
    bands for which the staged kernel is faster run staged: FP16 at any height where rows start
    on block boundaries and above two rows where they don't, FP32 above 16 rows on block
    boundaries.  Other storages keep the sliding window at every height.  lb_get_kernel tells
    what is launched."""
    seen = run(tmp_path, r'''
seen = []
for nx in (1024, 1000, 612):
    for st in (lb.STORAGE_F64, lb.STORAGE_F32, lb.STORAGE_F16DEV, lb.STORAGE_F32_BLOCKED, lb.STORAGE_F16_BLOCKED):
        h = lattice(nx, 64, W.LG if st == lb.STORAGE_F64 else W.BINARY, st)
        for t in [None] + [(x, y) for x in (64, 128, 256) for y in (1, 2, 3, 16, 17, 64)]:
            if t: assert L.lb_set_tile(h, *t) == 0
            log()
            assert L.lb_step(h, 1) == 0
            names = [n for _, _, n in launches("_kernel")]
            assert len(names) == 1
            seen.append([nx, st, tile(h)[1], kernel(h), "step_tma_kernel" in names[0]])
        L.lb_destroy(h)
print(json.dumps(seen))
''')
    for nx, st, ty, kernel, staged in seen:
        assert kernel == (2 if staged else 1)
        aligned = nx % 32 == 0
        if st == 7:  # FP16 blocks (612 x 64: fewer than 40000 fluid nodes, staged at every tile)
            expect = nx == 612 or ty > (0 if aligned else 2)
        else:
            expect = st == 6 and aligned and ty > 16
        assert staged == expect, (nx, st, ty)


def test_sliding_window_runs_the_kernel_whose_tiles_fit_in_one_wave(tmp_path):
    """Strips of 30 columns against tiles of 32 a warp: where the tiles fit in one wave of 16
    warps on each of the 152 SMs and the strips don't, the planes run the shared window."""
    seen = run(tmp_path, r'''
seen = []
for nx, ny in ((1024, 64), (700, 40), (2304, 128), (1000, 200)):
    for model, st in ((W.LG, lb.STORAGE_F64), (W.LG, lb.STORAGE_F32), (W.BINARY, lb.STORAGE_F64), (W.BINARY, lb.STORAGE_F32),
                      (W.BINARY, lb.STORAGE_F16DEV), (W.BINARY, lb.STORAGE_F32_BLOCKED)):
        h = lattice(nx, ny, model, st)
        assert L.lb_set_kernel(h, 1) == 0
        for t in [(x, y) for x in (64, 128, 256) for y in (1, 2, 3, 4, 8)]:
            assert L.lb_set_tile(h, *t) == 0
            log()
            assert L.lb_step(h, 1) == 0
            (grid, block, name), = launches("_kernel")
            assert kernel(h) == 1 and block == t[0]
            seen.append([nx, ny, model, st, t, grid, "strip_kernel" in name])
        L.lb_destroy(h)
print(json.dumps(seen))
''')
    windows = set()
    for nx, ny, model, st, (tx, ty), grid, strip in seen:
        bands = -(-ny // ty)
        strips, window = -(-nx // (tx // 32 * 30)) * bands, -(-nx // tx) * bands
        assert grid == (strips if strip else window)
        wave = 152 * 16 // (tx // 32)
        one = window <= wave < strips
        if st == 6:
            expect = True
        elif model == 0 and st == 1:
            expect = not (tx == 256 and one)
        else:
            expect = not (one or (tx == 256 and window <= wave and -(-strips // 152) > -(-window // 152)))
            if st == 0 and ty > 2:
                expect = False
        assert strip == expect, (nx, ny, model, st, tx, ty)
        if not strip:
            windows.add((nx, tx, ty, st))
    assert {(2304, 128, 4, 1), (2304, 64, 4, 2), (1024, 256, 2, 0)} <= windows


def test_staged_launches_that_let_the_next_step_in_early(tmp_path):
    """TmaArgs::early: off for long CTAs between half of one and five (64 columns), three (128), two
    (256) on each of the 152 SMs: FP64 bands from six rows, FP32 blocks from three, FP16 blocks
    from six; on for everything else."""
    from paper_0911_0459_gb300 import build
    kinds = [(m, s) for m, s in ((0, "SF64"), (1, "SF64"), (1, "SF32"), (0, "SF32"), (1, "SF16"), (1, "SF32B"), (1, "SF16B"))]
    probe = tmp_path / "offsets.cu"
    probe.write_text('#include <stddef.h>\n#include <stdio.h>\n#include "lb_step_tma.cuh"\nint main() {\n' + "".join(
        f'  {{ using T = lbk::TmaArgs<{m}, lbk::{s}>; printf("%zu\\n", offsetof(T, early)); }}\n' for m, s in kinds) + "}\n")
    subprocess.run([build.nvcc(), "-std=c++17", *build.ARCH, "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, "-o",
                    str(tmp_path / "offsets"), str(probe)], check=True, capture_output=True)
    at = subprocess.run([str(tmp_path / "offsets")], capture_output=True, text=True, check=True).stdout.split()
    watch = {f"step_tma_kernel<{m}, lbk::{s}, ": int(o) for (m, s), o in zip(kinds, at)}
    seen = run(tmp_path, "for k, o in " + json.dumps(watch) + ".items(): fake.fake_watch(k.encode(), o)\n" + r'''
seen = []
for nx, ny in ((1024, 64), (1000, 200), (4096, 128)):
    for model, st in ((W.LG, lb.STORAGE_F64), (W.BINARY, lb.STORAGE_F64), (W.BINARY, lb.STORAGE_F32), (W.LG, lb.STORAGE_F32),
                      (W.BINARY, lb.STORAGE_F16DEV), (W.BINARY, lb.STORAGE_F32_BLOCKED), (W.BINARY, lb.STORAGE_F16_BLOCKED)):
        h = lattice(nx, ny, model, st)
        for v in (2, 3):
            assert L.lb_set_kernel(h, v) == 0
            for t in [(x, y) for x in (64, 128, 256) for y in (1, 2, 3, 5, 6, 12, 32)]:
                assert L.lb_set_tile(h, *t) == 0
                log()
                assert L.lb_step(h, 1) == 0
                lines = log()
                (i, l), = [(i, l) for i, l in enumerate(lines) if l[0] == "launch"]
                assert "step_tma_kernel" in l[5] and lines[i - 1][0] == "word"
                seen.append([st, t, int(l[2]), int(lines[i - 1][1])])
        L.lb_destroy(h)
print(json.dumps(seen))
''')
    late = 0
    for st, (tx, ty), grid, early in seen:
        rows, full = {0: 6, 6: 3, 7: 6}.get(st), {64: 5, 128: 3, 256: 2}[tx]
        expect = rows is None or ty < rows or not 76 <= grid < full * 152
        assert early == expect, (st, tx, ty, grid)
        late += not early
    assert late > 30
