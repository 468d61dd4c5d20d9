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


def test_no_copy_of_a_failed_prediction_outlives_the_call(tmp_path):
    """A large prediction copies its results on a second stream, in parts.  Whichever runtime call
    fails, every stream that was given a copy into the caller's arrays is waited for before the
    call returns, and again before the network's memory goes back."""
    runs = run(tmp_path, r'''
n, nout, K = 16384, 64, 5
x = np.zeros((n, 4), np.float32)
out = [np.zeros((n, nout), np.float32), np.zeros((n, nout), np.float32), np.zeros((K, n, nout), np.float32)]
runs = []
for fn in ("cudaMemcpyAsync", "cudaStreamWaitEvent", "cudaEventRecord", "cudaLaunchKernelExC", "cudaStreamSynchronize"):
    for k in range(100):
        h = network(4, 256, nout, K, n)
        log()
        fake.fake_fail(fn.encode(), k)
        st = M.lb_mlp_predict(h, n, ptr(x), *(ptr(a) for a in out))
        called = log()
        M.lb_mlp_destroy(h)
        if st == 0:  # a prediction makes no more than k of these calls
            fake.fake_fail(fn.encode(), 1 << 30)
            break
        runs.append([fn, k, st, called, log()])
print(json.dumps(runs))
''')
    copied = 0
    for fn, k, st, called, after in runs:
        assert st == 2, (fn, k)  # LB_ERR_CUDA
        last = {}
        for i, l in enumerate(called):
            if l[0] in ("d2h", "sync"):
                last.setdefault(l[1], {})[l[0]] = i
        for stream, at in last.items():
            copied += "d2h" in at
            assert at.get("sync", -1) > at.get("d2h", -1), (fn, k, stream, called)
        gone = [l[1] for l in after if l[0] == "destroy"]
        assert gone and all(["sync", s] in after[:after.index(["destroy", s])] for s in gone), (fn, k, after)
    assert copied > 20 and len({r[0] for r in runs}) == 5
