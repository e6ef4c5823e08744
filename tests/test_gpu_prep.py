"""Point preparation at the sizes where its sort changes form: one cluster in
shared memory with 1 to 16 items per thread up to 131072 points, three launches
per pass above; each against the FP64 oracle on sampled rows, with repeated
points (equal keys) and a constant coordinate."""
import numpy as np
import pytest

from paper_1408_1237_gb300 import inputs

from conftest import f32

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-5


@pytest.fixture(scope="module")
def K():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1408_1237_gb300 import binding
    return binding


@pytest.mark.parametrize("N,d", [(1, 3), (31, 1), (257, 5), (8192, 2), (8193, 3), (16385, 9), (32769, 8),
                                 (65537, 2), (131072, 3), (131073, 3), (200001, 31)])
def test_preparation_at_the_sort_boundaries(K, oracle_mod, N, d):
    import torch
    rng = np.random.default_rng(N)
    X = rng.random((N, d)).astype(np.float32)
    X[: N // 3] = X[0]          # equal keys: ties keep every point exactly once
    if d > 1:
        X[:, d - 1] = 0.25      # an empty extent
    q = rng.standard_normal(N).astype(np.float32)
    sigma, gamma = 0.05 * np.sqrt(d), 1e-3
    got = K.krr_kernel_mvp(torch.from_numpy(X).cuda(), torch.from_numpy(q).cuda(), sigma, gamma).cpu().numpy()
    rows = inputs.sample_rows(N, 64, seed=1)
    X64, q64 = X.astype(np.float64), q.astype(np.float64)
    ref = oracle_mod.mvp(X64, q64, f32(sigma), f32(gamma), rows=rows)
    scale = oracle_mod.mvp(X64, np.abs(q64), f32(sigma), f32(gamma), rows=rows)
    assert np.max(np.abs(got[rows] - ref) / scale) <= TOL_FP32
