"""Tuning cache file (krr_tune_save / krr_tune_load): the autotuner's picks
(kernel variant and split scale per product shape) written on one handle and
read into another give the same products bit for bit; the file round-trips;
malformed files, missing files and files from a device with another SM count
are refused with KRR_ERR_INVALID_ARG.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1408_1237_gb300 import binding
    return binding


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _tuned_handle(K):
    h = K.Handle()
    K.krr_set_option(K.KRR_OPT_AUTOTUNE, 1, handle=h)
    return h


def test_tune_cache_round_trip(K, tmp_path):
    rng = np.random.default_rng(11)
    X = _dev(rng.random((60000, 2)).astype(np.float32))
    q = _dev(rng.standard_normal(60000).astype(np.float32))
    Q = _dev(rng.standard_normal((12, 60000)).astype(np.float32))
    path = tmp_path / "tune.txt"
    h1 = _tuned_handle(K)
    try:
        for arg in (q, Q):
            K.krr_kernel_mvp(X, arg, 0.05, 1e-3, handle=h1)  # tunes this shape
        ref = [K.krr_kernel_mvp(X, arg, 0.05, 1e-3, handle=h1).cpu().numpy() for arg in (q, Q)]
        K.krr_tune_save(path, handle=h1)
    finally:
        h1.close()
    lines = path.read_text().splitlines()
    assert lines[0].startswith("krr-tune 1 sms ") and len(lines) >= 3
    h2 = _tuned_handle(K)
    try:
        K.krr_tune_load(path, handle=h2)
        got = [K.krr_kernel_mvp(X, arg, 0.05, 1e-3, handle=h2).cpu().numpy() for arg in (q, Q)]
        path2 = tmp_path / "tune2.txt"
        K.krr_tune_save(path2, handle=h2)
    finally:
        h2.close()
    for a, b in zip(ref, got):
        np.testing.assert_array_equal(a, b)
    assert path2.read_text().splitlines()[0] == lines[0]
    assert sorted(path2.read_text().splitlines()[1:]) == sorted(lines[1:])


def test_tune_cache_refuses_bad_files(K, tmp_path):
    h = K.Handle()
    try:
        good = tmp_path / "good.txt"
        K.krr_tune_save(good, handle=h)
        header = good.read_text().splitlines()[0]
        sms = int(header.split()[-1])
        cases = {
            "missing": None,
            "not_a_cache": "hello\n",
            "other_device": f"krr-tune 1 sms {sms + 1}\n",
            "bad_scale": header + "\nmvp|1|1|3|0|1|0|0|3|0|0\t-2\t1\n",
            "bad_variant": header + "\nmvp|1|1|3|0|1|0|0|3|0|0\t1\t99\n",
            "missing_field": header + "\nmvp|1|1|3|0|1|0|0|3|0|0\t1\n",
        }
        for name, text in cases.items():
            p = tmp_path / f"{name}.txt"
            if text is not None:
                p.write_text(text)
            with pytest.raises(K.KrrError) as ei:
                K.krr_tune_load(p, handle=h)
            assert ei.value.status == K.KRR_ERR_INVALID_ARG, name
        K.krr_tune_load(good, handle=h)  # an empty cache loads
    finally:
        h.close()


def test_gradient_keeps_its_own_kernel_choice(K, tmp_path):
    """krr_mll_grad chooses its block solves' kernel by a wider margin than the
    solvers do: neither takes the other's choice for one shape (a compact cloud,
    the same counts in both orders)."""
    rng = np.random.default_rng(12)
    X = _dev(0.01 * rng.random((600, 4)).astype(np.float32))
    B = _dev(rng.standard_normal((16, 600)).astype(np.float32))
    path = tmp_path / "tune.txt"
    keys = []
    with K.Handle() as h:
        opts = K.default_opts(tol=1e-4)
        K.krr_mll_grad(X, B[0].contiguous(), 0.1, 0.5, n_probes=15, opts=opts, handle=h)
        for _ in range(2):
            K.krr_tune_save(path, handle=h)
            keys.append({line.split("\t")[0] for line in path.read_text().splitlines()[1:]})
            K.krr_fgmres_solve(X, B, 0.1, 0.5, opts=opts, handle=h)
    mine = {k for k in keys[0] if k.endswith("|g")}
    assert mine and {k[:-2] for k in mine} <= keys[1] - keys[0]


def test_tuning_of_other_shapes_brings_no_wait(K, tmp_path):
    """A small single-column product waits for the device only if its own shape
    may have been tuned."""
    import time
    import torch
    rng = np.random.default_rng(13)
    X = _dev(rng.random((3000, 3)).astype(np.float32))
    Y = _dev(rng.random((2000, 3)).astype(np.float32))
    q, p = (_dev(rng.standard_normal(n).astype(np.float32)) for n in (3000, 2000))
    path = tmp_path / "tune.txt"
    with _tuned_handle(K) as h:
        K.krr_kernel_mvp(Y, p, 0.1, 1e-3, handle=h)
        tuned = K.krr_kernel_mvp(Y, p, 0.1, 1e-3, handle=h)
        K.krr_tune_save(path, handle=h)
    with K.Handle() as h:
        want = K.krr_kernel_mvp(X, q, 0.1, 1e-3, handle=h)
        K.krr_tune_load(path, handle=h)
        for A, w, ref, waits in ((X, q, want, False), (Y, p, tuned, True)):
            K.krr_kernel_mvp(A, w, 0.1, 1e-3, handle=h)
            torch.cuda.synchronize()
            torch.cuda._sleep(600_000_000)  # about 0.3 s
            t0 = time.perf_counter()
            y = K.krr_kernel_mvp(A, w, 0.1, 1e-3, handle=h)
            held = time.perf_counter() - t0 > 0.1
            torch.cuda.synchronize()
            assert held == waits and torch.equal(y, ref)
