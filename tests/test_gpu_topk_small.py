"""The one-block top-K of short residuals (up to 16,384 rows) at its edges and
with ties: the set of an iteration's first residual, r = b with no sampled
updates, equals the definition's (larger |r| first, ties to the lower row)."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k", [(3, 3), (1023, 1), (1025, 5), (16383, 16), (16384, 16), (16385, 17)])
@pytest.mark.parametrize("kind", ["normal", "few_values", "wide"])
def test_first_iteration_set(cuda_ok, m, k, kind):
    rng = np.random.default_rng(m)
    # ("wide": as far as the squares that ||b|| sums are representable)
    b = {"normal": rng.standard_normal(m),
         "few_values": rng.choice([0.0, 1.0, -1.0, 2.0], m, p=[0.1, 0.44, 0.44, 0.02]),
         "wide": rng.standard_normal(m) * 10.0 ** rng.uniform(-150, 150, m)}[kind]
    n = m + 1                                        # K < n
    s = W.System("diagonal", m, n, row_ptr=np.arange(m + 1), col_idx=np.arange(m, dtype=np.int32),
                 values=np.ones(m), b=b, num_blocks=k, lam=1.0)
    with B.Handle.from_system(s) as h:
        K = h.info.dyn_rows
        tr = B.Trace()
        I = torch.full((K,), -1, dtype=torch.int32, device="cuda")
        tr.capacity, tr.I = 1, I.data_ptr()
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        h.solve(torch.as_tensor(b, device="cuda"), x, tol=0.0, maxit=1, seed=1, n_static=0, trace=tr)
    np.testing.assert_array_equal(I.cpu().numpy(), oracle.topk(b, K))
