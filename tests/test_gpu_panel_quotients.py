"""Quotients next to the middle between two numbers, in the panel of the cluster's
factor: a dense system whose Gram has the pivot d and, below it, numerators v
chosen so that v / sqrt(d) lies as near to a middle as quotients can.  The updated x
equals the FP64 oracle's bit for bit."""
import math

import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hard_numerators(l, count, rng):
    """V in [2^52, 2^53) with V 2^s - M L = j for small odd j and odd 54-bit M, L the
    mantissa of l (odd)."""
    L = int(math.ldexp(l, 52))
    out = []
    j = 1
    while len(out) < count:
        for s in (53, 54):
            for k in (j, -j):
                M = -k * pow(L, -1, 2 ** s) % 2 ** s
                M = M + 2 ** 53 if s == 53 else M
                V, rest = divmod(M * L + k, 2 ** s)
                if 2 ** 53 <= M < 2 ** 54 and rest == 0 and 2 ** 52 <= V < 2 ** 53:
                    out.append(float(V) if rng.random() < 0.5 else -float(V))
        j += 2
    return np.array(out[:count])


@pytest.mark.parametrize("seed", range(12))
def test_panel_quotients_next_to_a_middle(cuda_ok, seed):
    K, n = 256, 260
    rng = np.random.default_rng(seed)
    while True:
        d = rng.uniform(1.0, 4.0)
        if int(math.ldexp(math.sqrt(d), 52)) % 2:
            break
    v = _hard_numerators(math.sqrt(d), K - 1, rng) * 2.0 ** -52
    c = 2.0 ** -30                                   # c^2 is below half a unit of d
    A = np.zeros((K, n))
    A[0, 0] = c
    A[1:, 0] = v / c                                 # Gram: g_00 = d, g_i0 = v_i exactly
    A[np.arange(1, K), np.arange(1, K)] = 2.0 ** 30
    s = W.System("quotients", K, n, dense=A, b=np.ones(K), num_blocks=1, lam=d)
    G = oracle.block_gram(s, np.arange(K), d)
    assert G[0, 0] == d and np.array_equal(G[1:, 0], v)
    I = np.arange(K, dtype=np.int32)
    r = np.zeros(K)
    r[0] = 1.0
    with B.Handle.from_system(s) as h:
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        h.dynamic_update(torch.as_tensor(I, device="cuda"), torch.as_tensor(r, device="cuda"), x)
    xo = oracle.update_with_cholesky(s, I, d, r, np.zeros(n))
    np.testing.assert_array_equal(x.cpu().numpy(), xo)
