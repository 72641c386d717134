"""Large components of the dynamic block that are shallow trees are factored in
place, level by level; deeper trees, rows with two larger ones and other
components go to the cluster.  On both sides of the rule, and with components of
both kinds in one update, the updated x equals the FP64 oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _system(links, m, seed, scale=0.0):
    """Rows 0 .. m - 1 with a column of their own each, and one column per linked
    pair of rows; values over `scale` binary exponents."""
    rng = np.random.default_rng(seed)
    cols = [[] for _ in range(m)]
    for c, pair in enumerate(links):
        for i in pair:
            cols[i].append(c)
    n0 = len(links)
    ptr, ci, va = [0], [], []
    for i in range(m):
        f = 2.0 ** rng.uniform(-scale, scale)
        ci += cols[i] + [n0 + i]
        va += list(f * rng.choice([-1, 1], len(cols[i]) + 1) * rng.uniform(0.5, 2.0, len(cols[i]) + 1))
        ptr.append(len(ci))
    n = n0 + m + 1
    return W.System("links", m, n, row_ptr=np.array(ptr), col_idx=np.array(ci, dtype=np.int32), values=np.array(va),
                    b=rng.standard_normal(m), num_blocks=1, lam=0.0)


def star(first, size, hub):
    return [(i, first + hub) for i in range(first, first + size) if i != first + hub]


def heap(first, size):
    """Row i (from the end) hangs from row (i - 1) // 2: smaller rows are the leaves."""
    return [(first + size - 1 - i, first + size - 1 - (i - 1) // 2) for i in range(1, size)]


def chain(first, size):
    return [(i, i + 1) for i in range(first, first + size - 1)]


CASES = {
    "star_33": (star(0, 33, 32), 33),
    "star_256": (star(0, 256, 255), 256),
    "star_180_pairs_twice": (star(0, 180, 179) + star(0, 180, 179), 180),
    "hub_first": (star(0, 40, 0), 40),
    "hub_inside": (star(0, 60, 30), 60),
    "heap_250": (heap(0, 250), 250),
    "six_stars": (sum((star(40 * g, 40, 39) for g in range(6)), []), 240),
    "chain_40": (chain(0, 40), 40),
    "levels_12": (star(0, 30, 29) + chain(29, 11), 41),          # 0 .. 11: the deepest handled in place
    "levels_13": (star(0, 30, 29) + chain(29, 12), 42),
    "star_chain_small": (star(0, 50, 49) + chain(50, 60) + heap(110, 20) + chain(140, 5), 150),
    "above_the_limit": (star(0, 257, 256), 257),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("scale", [0.0, 330.0])
def test_update_equals_oracle(cuda_ok, name, scale):
    links, m = CASES[name]
    s = _system(links, m, 5, scale)
    r = np.random.default_rng(7).standard_normal(m) * np.sqrt(np.add.reduceat(s.values ** 2, s.row_ptr[:-1]))
    I = np.arange(m, dtype=np.int32)
    with B.Handle.from_system(s) as h:
        x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
        for _ in range(2):
            x.zero_()
            h.dynamic_update(torch.as_tensor(I, device="cuda"), torch.as_tensor(r, device="cuda"), x)
    xo = oracle.update_with_cholesky(s, I, 0.0, r, np.zeros(s.n))
    assert np.all(np.isfinite(xo))
    np.testing.assert_array_equal(x.cpu().numpy(), xo)


def test_mixed_form_converges_and_columns_agree(cuda_ok):
    links, m = CASES["six_stars"]
    s = _system(links, m, 3)
    s.lam = 1e-6
    xt = np.random.default_rng(1).standard_normal((s.n, 2))
    Bm = torch.as_tensor(np.ascontiguousarray(s.to_dense() @ xt), device="cuda")
    with B.Handle.from_system(s, precision=B.PREC_MIXED) as h, h.multi(2) as hm:
        X = torch.zeros(s.n, 2, dtype=torch.float64, device="cuda")
        hm.solve_multi(Bm, X, tol=0.0, maxit=6, seed=2, precision=B.PREC_MIXED)
        for j in range(2):
            b = Bm[:, j].contiguous()
            x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
            h.solve(b, x, tol=0.0, maxit=6, seed=2, precision=B.PREC_MIXED)
            assert torch.equal(X[:, j], x)
            assert h.solve(b, x, tol=1e-10, maxit=200, seed=2, precision=B.PREC_MIXED).converged
