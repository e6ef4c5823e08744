"""Small single-column products run as one launch: the same bits as gather,
product and finalize (the form that a profiled handle takes), call after call,
with shards, and against the FP64 oracle."""
import numpy as np
import pytest

from conftest import f32

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


def _data(N, d, seed):
    import torch
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.rand(N, d, device="cuda", generator=g), torch.randn(N, device="cuda", generator=g)


@pytest.mark.parametrize("N,d", [(1, 1), (32, 3), (33, 2), (257, 8), (2048, 4), (4095, 3), (16384, 2), (16384, 7),
                                 (16385, 3)])
@pytest.mark.parametrize("family", [0, 1])
def test_one_launch_equals_three(K, oracle_mod, N, d, family):
    import torch
    X, q = _data(N, d, N + d)
    sigma, gamma = 0.1 * d ** 0.5, 1e-2
    h, g = K.Handle(), K.Handle()
    for x in (h, g):
        K.krr_set_option(K.KRR_OPT_KERNEL, family, handle=x)
    K.krr_profile_enable(True, handle=g)
    for _ in range(3):  # arrival counters are left at zero
        y = K.krr_kernel_mvp(X, q, sigma, gamma, handle=h)
        three = K.krr_kernel_mvp(X, q, sigma, gamma, handle=g)
        torch.cuda.synchronize()
        assert torch.equal(y, three)
    with K.Points(X, sigma, handle=h) as P:
        assert torch.equal(K.krr_kernel_mvp_points(P, q, gamma), y)
    K.krr_set_option(K.KRR_OPT_SHARD_COUNT, 3, handle=h)
    parts = torch.full_like(y, float("nan"))
    for k in range(3):
        K.krr_set_option(K.KRR_OPT_SHARD_INDEX, k, handle=h)
        K.krr_kernel_mvp(X, q, sigma, gamma, out=parts, handle=h)
    assert torch.equal(parts, y)
    if family == 0 and N <= 4096:
        X64, q64 = X.cpu().numpy().astype(np.float64), q.cpu().numpy().astype(np.float64)
        ref = oracle_mod.mvp(X64, q64, f32(sigma), f32(gamma))
        scale = oracle_mod.mvp(X64, np.abs(q64), f32(sigma), f32(gamma))
        assert np.max(np.abs(y.cpu().numpy() - ref) / scale) <= 1e-5
    h.close()
    g.close()



@pytest.mark.parametrize("N,d", [(12288, 2), (12289, 2), (16384, 4), (20000, 3), (24576, 2), (24577, 4), (32001, 1)])
@pytest.mark.parametrize("family", [0, 1])
def test_products_in_one_and_in_several_waves(K, oracle_mod, N, d, family):
    """Both depths of unrolling of the one-target kernel, against the oracle on
    sampled rows."""
    X, q = _data(N, d, N + d)
    sigma, gamma = 0.1 * d ** 0.5, 1e-2
    with K.Handle() as h:
        K.krr_set_option(K.KRR_OPT_KERNEL, family, handle=h)
        y = K.krr_kernel_mvp(X, q, sigma, gamma, handle=h).cpu().numpy()
    rows = np.random.default_rng(N).choice(N, 64, replace=False)
    X64, q64 = X.cpu().numpy().astype(np.float64), q.cpu().numpy().astype(np.float64)
    kernel = "matern32" if family else "gaussian"
    ref = oracle_mod.mvp(X64, q64, f32(sigma), f32(gamma), rows=rows, kernel=kernel)
    scale = oracle_mod.mvp(X64, np.abs(q64), f32(sigma), f32(gamma), rows=rows, kernel=kernel)
    assert np.max(np.abs(y[rows] - ref) / scale) <= 1e-5
