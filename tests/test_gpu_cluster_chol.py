"""The dynamic block's factor and solves in one thread-block cluster, against
the FP64 oracle's dynamic update, at the edges of its 32-column panels, of its
cluster sizes (4, 8 and 16 blocks) and of its largest order (543), above which
other kernels take over.  Every entry sees the definition's operations in the
definition's order, so the updated x is equal bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(s):
    rng = np.random.default_rng(s.m)
    x0 = rng.standard_normal(s.n)
    r = rng.standard_normal(s.m)
    I = np.arange(s.m, dtype=np.int32)              # one block: all rows
    with B.Handle.from_system(s) as h:
        assert h.info.dyn_rows == s.m < s.n
        x = torch.as_tensor(x0, device="cuda")
        h.dynamic_update(torch.as_tensor(I, device="cuda"), torch.as_tensor(r, device="cuda"), x)
    xo = oracle.update_with_cholesky(s, I, s.lam, r, x0)
    np.testing.assert_array_equal(x.cpu().numpy(), xo)


@pytest.mark.parametrize("K", [1, 2, 31, 32, 33, 64, 65, 128, 129, 256, 543, 544])
def test_dense_dynamic_update(cuda_ok, K):
    _check(W.gaussian_dense(K, K + 3, seed=K, num_blocks=1, lam=1e-3))


@pytest.mark.parametrize("K", [33, 64, 65, 129, 287, 543, 544])
def test_sparse_dynamic_update_with_one_large_component(cuda_ok, K):
    _check(W.random_sparse(K, 2 * K, 0.06, seed=K, num_blocks=1, lam=1e-3, empty_rows=K // 16))


@pytest.mark.parametrize("nr", [2, 16])
def test_columns_with_large_components(cuda_ok, nr):
    """One cluster per column: K = 270 rows on 1,200 columns, every column the
    library's one-column solve bit for bit (FP64 and mixed)."""
    s = W.random_sparse(1080, 1200, 0.01, seed=5, num_blocks=4, lam=1e-3)
    Bm = torch.as_tensor(W.rhs_block(s, nr, 3), device="cuda")
    for prec in (B.PREC_FP64, B.PREC_MIXED):
        with B.Handle.from_system(s, precision=prec) as h, h.multi(nr) as hm:
            X = torch.zeros(s.n, nr, dtype=torch.float64, device="cuda")
            hm.solve_multi(Bm, X, tol=0.0, maxit=6, seed=2, precision=prec)
            for j in (0, nr - 1):
                x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
                h.solve(Bm[:, j].contiguous(), x, tol=0.0, maxit=6, seed=2, precision=prec)
                assert torch.equal(X[:, j], x)
