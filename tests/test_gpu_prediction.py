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
