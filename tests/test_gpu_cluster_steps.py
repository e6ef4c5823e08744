"""Solves at the sizes where the cluster kernels of the CG and Arnoldi steps
change their rows per thread (2048, 4096, 8192, 16384 padded rows) and where
the kernels of larger problems take over, with one and several columns (one of
them zero, inactive from the start): the FP64 oracle's residual meets the
tolerance, and the graph and the host loop give the same bits."""
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


@pytest.mark.parametrize("N", [1, 255, 2048, 2049, 4097, 8193, 16384, 16385])
@pytest.mark.parametrize("m", [1, 3])
def test_solve_at_the_row_boundaries(K, oracle_mod, N, m):
    import torch
    rng = np.random.default_rng(N + m)
    X = rng.random((N, 2)).astype(np.float32)
    B = rng.standard_normal((m, N)).astype(np.float32)
    if m > 1:
        B[1] = 0.0
    sigma, gamma = 0.02, 0.5
    Xd, Bd = torch.from_numpy(X).cuda(), torch.from_numpy(B[0] if m == 1 else B).cuda()
    sols = []
    for graph in (1, 0):
        opts = K.default_opts(delta=0.5, inner_tol=1e-2, use_graph=graph)
        x, info = K.krr_fgmres_solve(Xd, Bd, sigma, gamma, opts=opts)
        assert all(i["status"] == K.KRR_OK for i in info)
        sols.append(x.cpu().numpy().reshape(m, N))
    assert np.array_equal(sols[0], sols[1])
    X64 = X.astype(np.float64)
    for c in range(m):
        b = B[c].astype(np.float64)
        r = b - oracle_mod.mvp(X64, sols[0][c], f32(sigma), f32(gamma))
        assert np.linalg.norm(r) <= 1e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("N,m", [(12288, 1), (12289, 1), (12288, 4), (12289, 4), (12289, 5), (16384, 5), (16385, 5)])
def test_steps_at_the_boundaries_of_few_and_many_columns(K, oracle_mod, N, m):
    test_solve_at_the_row_boundaries(K, oracle_mod, N, m)
