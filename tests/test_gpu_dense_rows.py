"""The dense row and column chains (asynchronous ring of stages) at the edges
of their 32-row groups, their stages (32 FP64 or 64 FP32 columns) and their two
copy forms (rows on 16-byte boundaries or not), against the FP64 oracle and,
in FP32, against the chain written out."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 2), (31, 40), (33, 31), (64, 64), (65, 129), (300, 255), (5000, 32), (40000, 33), (97, 3001)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_dense_residual_equals_oracle(cuda_ok, m, n, dtype):
    """Each row is one chain in column order: equal bit for bit."""
    s = W.gaussian_dense(m, n, seed=m + n, num_blocks=max(1, m // 200), lam=1.0)
    s.dense = np.ascontiguousarray(s.dense.astype(dtype))
    x = np.random.default_rng(1).standard_normal(n)
    with B.Handle.from_system(s) as h:
        r = torch.empty(m, dtype=torch.float64, device="cuda")
        xd = torch.zeros(n + 1, dtype=torch.float64, device="cuda")[1:]     # not on a 16-byte boundary
        xd.copy_(torch.as_tensor(x))
        h.residual(torch.as_tensor(s.b, device="cuda"), xd, r)
    np.testing.assert_array_equal(r.cpu().numpy(), oracle.residual(s, s.b, x)[0])


@pytest.mark.parametrize("m,n", [(33, 31), (65, 129), (200, 64)])
def test_dense_residual32_is_the_fp32_chain(cuda_ok, m, n):
    """FP32 fused chain over the columns: one rounding per link, so a chain of n
    links stays within n units of 2^-24 of the magnitudes summed."""
    s = W.gaussian_dense(m, n, seed=3, num_blocks=1, lam=1.0)
    x, b = (np.random.default_rng(k).standard_normal(v).astype(np.float32) for k, v in ((1, n), (2, m)))
    with B.Handle.from_system(s, precision=B.PREC_MIXED) as h:
        r = torch.empty(m, dtype=torch.float32, device="cuda")
        h.residual32(torch.as_tensor(b, device="cuda"), torch.as_tensor(x, device="cuda"), r)
    A = s.dense.astype(np.float32).astype(np.float64)
    bound = (n + 1) * 2.0 ** -24 * (np.abs(A) @ np.abs(x.astype(np.float64)) + np.abs(b))
    assert np.all(np.abs(r.cpu().numpy() - (b - A @ x.astype(np.float64))) <= bound)


@pytest.mark.parametrize("m,n,k", [(70, 75, 2), (640, 333, 5), (66, 2050, 2)])
def test_dense_iterations_at_ragged_sizes(cuda_ok, m, n, k):
    """Static updates, top-K, dynamic update: 8 iterations equal the oracle's,
    with more sampled updates per iteration than the grid launches take too."""
    s = W.gaussian_dense(m, n, seed=9, num_blocks=k, lam=1e-4)
    for n_static in (3, 5):
        o = oracle.solve(s, maxit=8, tol=0.0, seed=6, n_static=n_static)
        with B.Handle.from_system(s) as h:
            x = torch.zeros(n, dtype=torch.float64, device="cuda")
            h.solve(torch.as_tensor(s.b, device="cuda"), x, tol=0.0, maxit=8, seed=6, n_static=n_static)
        np.testing.assert_array_equal(x.cpu().numpy(), o.x)
