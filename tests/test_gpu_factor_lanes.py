"""Factors of the dynamic block whose lanes take different paths: pivots and
entries on both sides of the exponents between which roots and quotients come
from fused remainders, so that some lanes of a warp call sqrt or the division
while others do not.  Every entry still receives the definition's operations in
the definition's order: the updated x equals the FP64 oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _groups(sizes, seed):
    """Rows in groups that share one column each, with a column of their own
    besides: row i of a group holds t_i there and a_i in the group's column, with
    exponents up to +-380, so that the Gram's entries a_i a_j and its pivots spread
    over twice that.  |a_i| <= 2 |t_i|: well conditioned after scaling."""
    rng = np.random.default_rng(seed)
    cols, vals, ptr = [], [], [0]
    m = sum(sizes)
    row = 0
    for g, size in enumerate(sizes):
        for _ in range(size):
            e = rng.uniform(-380, 380) if rng.random() < 0.5 else rng.uniform(-4, 4)
            t = 2.0 ** e * rng.uniform(1, 2)
            a = t * rng.uniform(0.2, 1.0) * rng.choice([-1, 1])
            cols += [row, m + g]
            vals += [t, a]
            ptr.append(len(cols))
            row += 1
    return W.System("groups", m, m + len(sizes) + 1, row_ptr=np.array(ptr), col_idx=np.array(cols, dtype=np.int32),
                    values=np.array(vals), b=np.ones(m), num_blocks=1, lam=0.0)


def _check(s):
    rng = np.random.default_rng(s.m)
    r = rng.standard_normal(s.m) * np.sqrt(np.add.reduceat(s.values ** 2, s.row_ptr[:-1]))
    I = np.arange(s.m, dtype=np.int32)
    with B.Handle.from_system(s) as h:
        assert h.info.dyn_rows == s.m
        x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
        h.dynamic_update(torch.as_tensor(I, device="cuda"), torch.as_tensor(r, device="cuda"), x)
    xo = oracle.update_with_cholesky(s, I, s.lam, r, np.zeros(s.n))
    assert np.all(np.isfinite(xo))
    np.testing.assert_array_equal(x.cpu().numpy(), xo)


@pytest.mark.parametrize("sizes", [(2,), (3, 32, 31, 2, 17), (32,) * 8])
@pytest.mark.parametrize("seed", [1, 2])
def test_small_components_with_lanes_apart(cuda_ok, sizes, seed):
    _check(_groups(sizes, seed))


@pytest.mark.parametrize("sizes", [(33,), (64, 40), (150, 5, 1), (300,)])
def test_cluster_with_lanes_apart(cuda_ok, sizes):
    """Components above 32 rows: the same in the cluster (4, 8 and 16 blocks)."""
    _check(_groups(sizes, 3))


@pytest.mark.parametrize("half", [17, 40, 150])
def test_singular_component_is_reported(cuda_ok, half):
    """Rows i and half + i are equal, in different sampled blocks (each regular
    with lambda = 0) but in one dynamic set and one component: a pivot of exactly
    0 ends the update with NOT_SPD, x as it was, and the handle goes on."""
    m = 2 * half
    rng = np.random.default_rng(half)
    # 1 in the pair's own column, 2 in one that all rows share
    cols = np.array([[i % half, half] for i in range(m)], dtype=np.int32)
    vals = np.array([[1.0, 2.0]] * m)
    s = W.System("pairs", m, m + 3, row_ptr=2 * np.arange(m + 1), col_idx=cols.ravel(), values=vals.ravel(),
                 b=np.ones(m), num_blocks=2, lam=0.0)
    # K = half rows: with num_blocks = 2 the dynamic set holds both of some pairs
    I = np.sort(np.concatenate([np.arange(half // 2), half + np.arange(half - half // 2)])).astype(np.int32)
    x0 = rng.standard_normal(s.n)
    r = torch.as_tensor(rng.standard_normal(m), device="cuda")
    with B.Handle.from_system(s) as h:
        x = torch.as_tensor(x0.copy(), device="cuda")
        with pytest.raises(B.RorbkError) as e:
            h.dynamic_update(torch.as_tensor(I, device="cuda"), r, x)
        assert e.value.status == -4
        np.testing.assert_array_equal(x.cpu().numpy(), x0)
        I2 = np.arange(half, dtype=np.int32)
        h.dynamic_update(torch.as_tensor(I2, device="cuda"), r, x)
    xo = oracle.update_with_cholesky(s, I2, s.lam, r.cpu().numpy()[:half], x0)
    np.testing.assert_array_equal(x.cpu().numpy(), xo)
