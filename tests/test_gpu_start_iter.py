"""Any 64-bit start_iter is a Philox counter, -1 (whose successor is 0) among
them: the draws of the iterations before, at and after the wrap are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SYSTEMS = {"sparse": lambda: W.powerlaw(n=2048, num_blocks=16, seed=3, lam=1e-8),
           "dense": lambda: W.gaussian_dense(640, 333, seed=9, num_blocks=16, lam=1e-4)}


@pytest.mark.parametrize("kind", ["sparse", "dense"])
@pytest.mark.parametrize("start", [-2, -1, 0, 2 ** 63 - 4])
@pytest.mark.parametrize("host_loop", [0, 1])
def test_draws_from_any_counter(cuda_ok, kind, start, host_loop):
    s = SYSTEMS[kind]()
    tau = torch.full((3, 3), -1, dtype=torch.int64, device="cuda")
    tr = B.Trace()
    tr.capacity, tr.tau = 3, tau.data_ptr()
    with B.Handle.from_system(s) as h:
        x = torch.zeros(s.n, dtype=torch.float64, device="cuda")
        h.solve(torch.as_tensor(s.b, device="cuda"), x, tol=0.0, maxit=3, seed=5, start_iter=start, trace=tr,
                host_loop=host_loop)
    o = oracle.solve(s, maxit=3, tol=0.0, seed=5, start_iter=start, trace_tau=True)
    np.testing.assert_array_equal(tau.cpu().numpy(), o.tau)
    np.testing.assert_array_equal(x.cpu().numpy(), o.x)
