"""Source tiles whose kernel values are all exact zeros are left out of the
compact blocks' products; the sums must be the same bit for bit.  A weight of
f16's largest size keeps its tile, so a column of such weights (or one such
weight per tile, against the same weights halved) gives the product with every
tile evaluated."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BIG = 65504.0  # f16's largest: its tile is kept


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1408_1237_gb300 import binding
    return binding


def _cloud(name, N, seed):
    import torch
    rng = np.random.default_rng(seed)
    if name == "clusters":  # two far clusters: whole tiles at distances around the cut
        X = 0.02 * rng.standard_normal((N, 2)) + np.where(rng.random((N, 1)) < 0.5, 0.0, 0.3)
        return torch.from_numpy(X.astype(np.float32)).cuda(), 0.03
    X = rng.random((N, 3)) + (1000.0 if name == "offset" else 0.0)  # offset: boxes rounded to 6e-5
    return torch.from_numpy(X.astype(np.float32)).cuda(), 0.05


@pytest.mark.parametrize("cloud,N", [("cube", 150001), ("clusters", 40007), ("offset", 131073)])
@pytest.mark.parametrize("m,tc,prec", [(2, 0, "fp32"), (16, 0, "fp32"), (16, 1, "fp32"), (3, 0, "fp16"),
                                       (9, 1, "fp16"), (4, 0, "bf16"), (16, 1, "bf16")])
def test_columns_do_not_change_with_every_tile_kept(K, cloud, N, m, tc, prec):
    import torch
    X, sigma = _cloud(cloud, N, 5)
    h = K.Handle()
    K.krr_set_option(K.KRR_OPT_TCGEN05, tc, handle=h)
    Q = torch.randn(m, N, device="cuda", generator=torch.Generator("cuda").manual_seed(6))
    Q[m - 1] = 0.0
    y = K.krr_kernel_mvp(X, Q, sigma, 1e-3, prec=prec, handle=h)
    Q[m - 1] = BIG
    kept = K.krr_kernel_mvp(X, Q, sigma, 1e-3, prec=prec, handle=h)
    torch.cuda.synchronize()
    assert torch.equal(y[: m - 1], kept[: m - 1])
    assert torch.isfinite(kept).all()
    h.close()


@pytest.mark.parametrize("cloud,N", [("cube", 150001), ("clusters", 40007), ("offset", 131073)])
def test_single_column_is_the_same_with_every_tile_kept(K, cloud, N):
    import torch
    X, sigma = _cloud(cloud, N, 7)
    q = torch.randn(N, device="cuda", generator=torch.Generator("cuda").manual_seed(8)) * BIG
    q = torch.where(q.abs() < BIG, torch.sign(q) * 1.0, torch.sign(q) * BIG)  # about 80 kept weights per tile
    y = K.krr_kernel_mvp(X, q, sigma, 1e-3)
    half = K.krr_kernel_mvp(X, q * 0.5, sigma, 1e-3)  # exact scaling; no weight keeps its tile
    torch.cuda.synchronize()
    assert torch.equal(y, 2.0 * half)


@pytest.mark.parametrize("m", [1, 4])
def test_infinite_weight_and_nan_point_reach_every_compact_row(K, m):
    """0 * inf and a value at a point that is not a number are NaN, at any distance."""
    import torch
    X, sigma = _cloud("clusters", 40007, 9)
    Q = torch.randn(m, 40007, device="cuda", generator=torch.Generator("cuda").manual_seed(10))
    Q[0, 17] = float("inf")
    y = K.krr_kernel_mvp(X, Q[0] if m == 1 else Q, sigma, 1e-3).reshape(m, -1)
    assert torch.isnan(y[0]).float().mean() > 0.4  # the rows of the other cluster too
    X2 = X.clone()
    X2[23, 1] = float("nan")
    y = K.krr_kernel_mvp(X2, torch.ones(40007, device="cuda"), sigma, 1e-3)
    torch.cuda.synchronize()
    assert torch.isnan(y).float().mean() > 0.9
