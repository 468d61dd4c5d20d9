"""The host side of the surrogate network's calls, without a GPU (fake_cudart.cpp)."""
from fake_cuda import run


def test_networks_that_share_a_kernel_share_its_shared_memory_limit(tmp_path):
    """The dynamic shared memory limit belongs to a kernel, and networks of one n_hidden run the
    same kernels whatever their n_out: whichever network sets the limit last, also from another
    thread between the first one's setting and its launch, every launch has to stay within it."""
    seen = run(tmp_path, r'''
x, y = np.zeros((4096, 4), np.float32), np.zeros((4096, 128), np.float32)
log()
for nout in (128, 8, 64):
    for n in (16, 4096):
        h = network(4, 256, nout, 2, 4096)
        out = [np.zeros((n, nout), np.float32) for _ in range(2)]
        assert M.lb_mlp_predict(h, n, ptr(x), ptr(out[0]), ptr(out[1]), None) == 0
        assert M.lb_mlp_set_data(h, n, ptr(x), ptr(y)) == 0
        assert M.lb_mlp_train(h, 2, 1e-3, 1e-4, 0.0, None) == 0
        M.lb_mlp_destroy(h)
limits, used = {}, {}
for l in log():
    if l[0] == "limit":
        limits.setdefault(" ".join(l[2:]), set()).add(int(l[1]))
    elif l[0] == "launch" and int(l[4]) > 48 << 10:
        used[l[5]] = max(used.get(l[5], 0), int(l[4]))
print(json.dumps([{k: sorted(v) for k, v in limits.items()}, used]))
''')
    limits, used = seen
    assert len(used) >= 4 and any("predict_kernel" in k for k in used) and any("rows_kernel" in k for k in used)
    for name, most in used.items():
        assert min(limits[name]) >= most, (name, limits[name], most)
