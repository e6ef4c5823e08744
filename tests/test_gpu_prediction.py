"""Prediction products of several columns (krr_kernel_mvp_rect): as accurate as
their single columns whatever the handle's kernel options."""
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


def errors(oracle_mod, Xt, Xs, Q, Y, sigma):
    """Largest error per column, scaled by sum_j |Q_j| K_tj."""
    Xt, Xs = Xt.astype(np.float64), Xs.astype(np.float64)
    out = []
    for q, y in zip(np.atleast_2d(Q).astype(np.float64), np.atleast_2d(Y)):
        ref = oracle_mod.mvp_rect(Xt, Xs, q, f32(sigma))
        out.append(np.max(np.abs(y - ref) / oracle_mod.mvp_rect(Xt, Xs, np.abs(q), f32(sigma))))
    return np.array(out)


def _clouds(d, Nt, Ns, seed):
    rng = np.random.default_rng(seed)
    return rng.random((Nt, d)).astype(np.float32), rng.random((Ns, d)).astype(np.float32), rng


@pytest.mark.parametrize("m", [9, 16])
def test_kernel_options_do_not_change_a_prediction(K, oracle_mod, m):
    """The tcgen05 kernels sum less exactly than single columns: predictions
    take none of them.  (The tuner may choose other splits.)"""
    import torch
    Xt, Xs, rng = _clouds(3, 1500, 1201, m)
    Q = rng.standard_normal((m, 1201)).astype(np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (Xt, Xs, Q)]
    ys = []
    for tc in (0, 1, 2, 3):
        with K.Handle() as h:
            K.krr_set_option(K.KRR_OPT_TCGEN05, tc, handle=h)
            ys.append(K.krr_kernel_mvp_rect(*dev, 0.3, handle=h))
            assert torch.equal(ys[0], ys[-1])
    with K.Handle() as h:
        K.krr_set_option(K.KRR_OPT_AUTOTUNE, 1, handle=h)
        tuned = K.krr_kernel_mvp_rect(*dev, 0.3, handle=h)
        assert torch.equal(K.krr_kernel_mvp_rect(*dev, 0.3, handle=h), tuned)
    for y in (ys[0], tuned):
        assert errors(oracle_mod, Xt, Xs, Q[:2], y[:2].cpu().numpy(), 0.3).max() <= 1e-5


# The bar of the float32 products is 1e-5.  A pass of several columns drops
# Pl Ql and sums three tf32 products per term: 3 * 2^-20 on top of the error of
# the same columns alone.  Ten widths out the exponent is 72 and more: rounding
# its f16 hi + lo operands (72 * 2^-23, and 2^-23 * 17 * 2.8 for the cross term)
# and truncating in its float32 accumulator (120 * 2^-23) moves it by at most
# 4e-5, single columns too.
TOL, SPLIT, TOL_FAR = 1e-5, 3 * 2.0 ** -20, 4e-5


@pytest.mark.parametrize("m", [1, 3, 4, 8, 9, 16, 17])
@pytest.mark.parametrize("scale", [1e-6, 1.0, 1e5, 1e30, "mixed"])
def test_weights_of_any_size(K, oracle_mod, m, scale):
    """Compact blocks (sigma 0.3), direct-form blocks (0.02) and both (0.14)."""
    import torch
    Xt, Xs, rng = _clouds(3, 1801, 1501, m)
    Q = rng.standard_normal((m, 1501)).astype(np.float32)
    Q *= np.float32(scale) if scale != "mixed" else np.float32(10.0) ** rng.uniform(-6, 5, Q.shape).astype(np.float32)
    Qd = torch.from_numpy(Q if m > 1 else Q[0]).cuda()
    for sigma in (0.3, 0.14, 0.02):
        y = K.krr_kernel_mvp_rect(torch.from_numpy(Xt).cuda(), torch.from_numpy(Xs).cuda(), Qd, sigma)
        y = y.cpu().numpy().reshape(m, -1)
        for c in {0, m // 2, m - 1}:
            assert errors(oracle_mod, Xt, Xs, Q[c], y[c], sigma)[0] <= TOL, (sigma, c)


@pytest.mark.parametrize("d,sigma", [(1, 0.05), (2, 0.15), (3, 0.2), (4, 0.25), (8, 0.5)])
@pytest.mark.parametrize("m", [3, 16])
def test_targets_away_from_all_sources(K, oracle_mod, m, d, sigma):
    import torch
    Xt0, Xs, rng = _clouds(d, 301, 1501, d)
    Q = rng.standard_normal((m, 1501)).astype(np.float32)
    Xsd, Qd = torch.from_numpy(Xs).cuda(), torch.from_numpy(Q).cuda()
    for out in (0, 2, 3, 4, 5, 6, 10):
        Xt = (1.5 * sigma * Xt0).astype(np.float32)  # one compact block and a remainder
        Xt[:, 0] += np.float32(1.0 + out * sigma)
        Xtd = torch.from_numpy(Xt).cuda()
        got = errors(oracle_mod, Xt, Xs, Q[:3], K.krr_kernel_mvp_rect(Xtd, Xsd, Qd, sigma)[:3].cpu().numpy(), sigma)
        alone = np.stack([K.krr_kernel_mvp_rect(Xtd, Xsd, Qd[c].contiguous(), sigma).cpu().numpy() for c in range(3)])
        one = errors(oracle_mod, Xt, Xs, Q[:3], alone, sigma)
        assert max(got.max(), one.max()) <= (TOL if out <= 6 else TOL_FAR), (out, got, one)
        if out <= 3:
            assert (got <= one + SPLIT).all(), (out, got, one)


def test_infinite_weight_stays_in_its_column(K):
    import torch
    Xt, Xs, rng = _clouds(2, 700, 1100, 5)
    dev = [torch.from_numpy(a).cuda() for a in (Xt, Xs)]
    Q = torch.from_numpy(rng.standard_normal((3, 1100)).astype(np.float32)).cuda()
    y = K.krr_kernel_mvp_rect(*dev, Q, 0.2)
    Q[0, 17] = float("inf")
    z = K.krr_kernel_mvp_rect(*dev, Q, 0.2)
    torch.cuda.synchronize()
    assert torch.equal(y[1:], z[1:]) and not torch.isfinite(z[0]).any()


@pytest.mark.parametrize("family", ["gaussian", "matern32"])
@pytest.mark.parametrize("d,width", [(2, 0.2), (5, 0.5), (12, 1.2), (33, 1.4)])
@pytest.mark.parametrize("m", [2, 5, 17])
def test_columns_together_and_alone(K, oracle_mod, m, d, width, family):
    """Every route of several columns (two kernel families, d above 8, one and
    two passes) against the oracle and the same columns alone."""
    import torch
    Xt, Xs, rng = _clouds(d, 1237, 1411, m + d)
    Q = rng.standard_normal((m, 1411)).astype(np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (Xt, Xs, Q)]
    with K.Handle() as h:
        K.krr_set_option(K.KRR_OPT_KERNEL, {"gaussian": K.KRR_KERNEL_GAUSSIAN, "matern32": K.KRR_KERNEL_MATERN32}[family],
                         handle=h)
        y = K.krr_kernel_mvp_rect(*dev, width, handle=h).cpu().numpy()
        for c in {0, m - 1}:
            alone = K.krr_kernel_mvp_rect(dev[0], dev[1], dev[2][c].contiguous(), width, handle=h).cpu().numpy()
            q = Q[c].astype(np.float64)
            args = (Xt.astype(np.float64), Xs.astype(np.float64))
            ref = oracle_mod.mvp_rect(*args, q, f32(width), kernel=family)
            scale = oracle_mod.mvp_rect(*args, np.abs(q), f32(width), kernel=family)
            got, one = (np.max(np.abs(v - ref) / scale) for v in (y[c], alone))
            assert one <= TOL and got <= min(TOL, one + SPLIT), (got, one)


def test_many_targets_take_the_same_kernels(K, oracle_mod):
    """From 131,072 targets and 9 columns on the automatic choice of the square
    products is a tcgen05 kernel."""
    import torch
    Xt, Xs, rng = _clouds(3, 131073, 1501, 8)
    Q = rng.standard_normal((9, 1501)).astype(np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (Xt, Xs, Q)]
    y = K.krr_kernel_mvp_rect(*dev, 0.1)
    with K.Handle() as h:
        K.krr_set_option(K.KRR_OPT_TCGEN05, 0, handle=h)
        assert torch.equal(K.krr_kernel_mvp_rect(*dev, 0.1, handle=h), y)
    rows = rng.choice(131073, 64, replace=False)
    assert errors(oracle_mod, Xt[rows], Xs, Q, y[:, torch.from_numpy(rows).cuda()].cpu().numpy(), 0.1).max() <= TOL
