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
