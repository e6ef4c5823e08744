"""Which targets share a super-block decides the form a 16-bit product rounds
their kernel values in, so 16-bit products (Gaussian, d <= 8) sort their points
in Morton order.  The row shards show the order: with as many shards as
super-blocks, shard k writes exactly the rows of super-block k."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SB = 256


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1408_1237_gb300 import binding
    return binding


def morton_order(X):
    """Stable order by interleaved cells, coordinate 0 lowest."""
    N, d = X.shape
    bits = max(1, min(16, 30 // d))
    lo, hi = X.min(0), X.max(0)
    cells = ((X - lo) / (hi - lo) * np.float32(1 << bits)).clip(0, (1 << bits) - 1).astype(np.uint32)
    key = np.zeros(N, dtype=np.uint32)
    for b in range(bits):
        for k in range(d):
            key |= ((cells[:, k] >> np.uint32(b)) & np.uint32(1)) << np.uint32(b * d + k)
    return np.argsort(key, kind="stable")


def rows_of_shards(K, h, product, N):
    import torch
    nsb = -(-N // SB)
    K.krr_set_option(K.KRR_OPT_SHARD_COUNT, nsb, handle=h)
    label = np.full(N, -1)
    for k in range(nsb):
        K.krr_set_option(K.KRR_OPT_SHARD_INDEX, k, handle=h)
        Y = torch.full((N,), float("nan"), device="cuda")
        product(Y)
        label[~torch.isnan(Y).cpu().numpy()] = k
    K.krr_set_option(K.KRR_OPT_SHARD_INDEX, 0, handle=h)
    K.krr_set_option(K.KRR_OPT_SHARD_COUNT, 1, handle=h)
    return label


def _data(N, d, seed):
    import torch
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, d)).astype(np.float32)
    q = torch.from_numpy(rng.standard_normal(N).astype(np.float32)).cuda()
    return X, torch.from_numpy(X).cuda(), q


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("N,d", [(2049, 8), (3000, 3), (257, 2)])
def test_products_in_16_bits_keep_morton_blocks(K, N, d, prec):
    X, Xd, q = _data(N, d, N + d)
    want = np.empty(N, dtype=int)
    want[morton_order(X)] = np.arange(N) // SB
    with K.Handle() as h:
        got = rows_of_shards(K, h, lambda Y: K.krr_kernel_mvp(Xd, q, 1.0, 1e-2, prec=prec, out=Y, handle=h), N)
        assert np.array_equal(got, want)
        with K.Points(Xd, 1.0, handle=h) as P:
            got = rows_of_shards(K, h, lambda Y: K.krr_kernel_mvp_points(P, q, 1e-2, prec=prec, out=Y), N)
        assert np.array_equal(got, want)


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("m", [1, 3])
def test_prediction_in_16_bits_is_the_square_product_at_the_same_points(K, m, prec):
    import torch
    X, Xd, _ = _data(3000, 4, 3)
    Q = torch.randn(m, 3000, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    Q = Q[0].contiguous() if m == 1 else Q
    y = K.krr_kernel_mvp(Xd, Q, 0.8, 0.0, prec=prec)
    assert torch.equal(K.krr_kernel_mvp_rect(Xd, Xd, Q, 0.8, prec=prec), y)


def test_point_set_holds_both_orders(K):
    """Products in 16 bits and in float32 over one object do not disturb each
    other; the first one in 16 bits is refused under capture, and the object
    works afterwards."""
    import torch
    N, d = 4000, 3
    X, Xd, q = _data(N, d, 9)
    with K.Handle() as h:
        f32 = K.krr_kernel_mvp(Xd, q, 0.7, 1e-2, handle=h)
        f16 = K.krr_kernel_mvp(Xd, q, 0.7, 1e-2, prec="fp16", handle=h)
        P = K.Points(Xd, 0.7, handle=h)
        out = torch.empty_like(q)
        one = K.krr_kernel_mvp_points(P, q, 1e-2)
        s = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            with pytest.raises(RuntimeError):
                K.krr_kernel_mvp_points(P, q, 1e-2, prec="fp16", out=out)
            K.krr_kernel_mvp_points(P, q, 1e-2, out=out)
        g.replay()
        two = K.krr_kernel_mvp_points(P, q, 1e-2, prec="fp16")
        g2 = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g2, stream=s):
            K.krr_kernel_mvp_points(P, q, 1e-2, prec="fp16", out=out)
        torch.cuda.synchronize()
        assert torch.equal(one, f32) and torch.equal(out, f32) and torch.equal(two, f16)
        g2.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, f16)
        assert torch.equal(K.krr_kernel_mvp_points(P, q, 1e-2), f32)
        P.close()
