"""Paths of the set-up and of the value refresh that depend on the shape: rows of
the centroids' Gram in shared memory (up to 24,576 blocks) and in global memory,
columns in more than 32 blocks, and refreshes of dense systems, of blocks in the
s >= n form and of blocks with more than 65,536 entries.  A refreshed handle
equals a fresh one bit for bit; C's row sums are compared with scipy's within the
rounding of sums of non-negative terms (one unit of 2^-53 per term)."""
import numpy as np
import pytest

from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu


def _rowsum(s, k):
    """sum_j C(t, j) for blocks of equal size."""
    A = sp.csr_matrix((s.values_f64(), s.col_idx, s.row_ptr), shape=(s.m, s.n))
    rows = s.m // k
    C = sp.csr_matrix((np.ones(s.m), np.arange(s.m), np.arange(0, s.m + 1, rows)), shape=(k, s.m)) @ A
    G = (C @ C.T).tocsr()
    nrm = np.sqrt(G.diagonal())
    D = sp.diags(1.0 / nrm)
    return np.asarray(abs(D @ G @ D).sum(axis=1)).ravel(), int(np.diff(G.indptr).max())


def _linked(m, k, n, wide, seed):
    """Three entries per row; column 0 holds an entry of `wide` blocks' first rows."""
    rng = np.random.default_rng(seed)
    first = np.zeros(m, dtype=bool)
    first[rng.choice(k, wide, replace=False) * (m // k)] = True
    cols = [np.concatenate([[0] if first[i] else [], 1 + rng.choice(n - 1, 3, replace=False)]) for i in range(m)]
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])])
    ci = np.concatenate([np.sort(c) for c in cols]).astype(np.int32)
    return W.System("linked", m, n, row_ptr=ptr, col_idx=ci, values=rng.standard_normal(ci.size),
                    b=rng.standard_normal(m), num_blocks=k, lam=1e-3)


@pytest.mark.parametrize("m,k,wide", [(640, 320, 2), (640, 320, 33), (640, 320, 320), (24576, 24576, 100),
                                      (24577, 24577, 3000)])
def test_row_sums_and_their_refresh(cuda_ok, m, k, wide):
    s = _linked(m, k, 4 * m, wide, m + wide)
    v2 = np.random.default_rng(3).standard_normal(s.values.size)
    s2 = W.System("linked2", s.m, s.n, row_ptr=s.row_ptr, col_idx=s.col_idx, values=v2, b=s.b, num_blocks=k, lam=s.lam)
    with B.Handle.from_system(s) as h, B.Handle.from_system(s2) as fresh:
        first = h.proposal()[1]
        h.update_values(torch.as_tensor(v2, device="cuda"))
        cdf, second = h.proposal()
        np.testing.assert_array_equal(cdf, fresh.proposal()[0])
        np.testing.assert_array_equal(second, fresh.proposal()[1])
    for system, got in ((s, first), (s2, second)):
        ref, terms = _rowsum(system, k)
        np.testing.assert_allclose(got, ref, rtol=(terms + 16) * 2.0 ** -52)


DENSE = {"dense": lambda: W.gaussian_dense(640, 333, seed=9, num_blocks=5, lam=1e-4),
         "dense_odd_blocks": lambda: W.gaussian_dense(643, 700, seed=9, num_blocks=5, lam=1e-4),
         "dense_s_ge_n": lambda: W.gaussian_dense(600, 100, seed=4, num_blocks=5, lam=1e-4),
         "sparse_s_ge_n": lambda: W.random_sparse(600, 100, 0.05, seed=4, num_blocks=5, lam=1e-4),
         "sparse_long_blocks": lambda: W.random_sparse(1000, 900, 0.15, seed=4, num_blocks=2, lam=1e-4)}


@pytest.mark.parametrize("kind", sorted(DENSE))
@pytest.mark.parametrize("where", ["device", "host"])
def test_refreshed_handle_equals_a_fresh_one(cuda_ok, kind, where):
    s = DENSE[kind]()
    rng = np.random.default_rng(8)
    if s.is_dense:
        v2 = s.dense * (1.0 + 0.25 * rng.standard_normal(s.dense.shape))
        s2 = W.System("v2", s.m, s.n, dense=v2, b=s.b, num_blocks=s.num_blocks, lam=s.lam)
    else:
        v2 = s.values * (1.0 + 0.25 * rng.standard_normal(s.values.size))
        s2 = W.System("v2", s.m, s.n, row_ptr=s.row_ptr, col_idx=s.col_idx, values=v2, b=s.b,
                      num_blocks=s.num_blocks, lam=s.lam)
    if kind == "sparse_long_blocks":
        assert np.diff(s.row_ptr[::500]).max() > 65536
    b = torch.as_tensor(s.b, device="cuda")
    with B.Handle.from_system(s, precision=B.PREC_MIXED) as h, B.Handle.from_system(s2, precision=B.PREC_MIXED) as fresh:
        h.update_values(torch.as_tensor(v2, device="cuda") if where == "device" else v2)
        for a, c in zip(h.proposal(), fresh.proposal()):
            np.testing.assert_array_equal(a, c)
        for t in range(s.num_blocks):
            xs = []
            for one in (h, fresh):
                x = torch.ones(s.n, dtype=torch.float64, device="cuda")
                one.static_update(t, b, x)
                xs.append(x)
            assert torch.equal(xs[0], xs[1])
        if kind == "sparse_long_blocks":                 # (its dynamic set is beyond the workspace)
            return
        for prec in (B.PREC_FP64, B.PREC_MIXED):
            xs = []
            for one in (h, fresh):
                x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
                one.solve(b, x, tol=0.0, maxit=6, seed=4, precision=prec)
                xs.append(x)
            assert torch.equal(xs[0], xs[1])
