"""The dense residual at every number of pairs of warps per SM that its rows lead
to (one, two, three, four, five and more groups of 32 rows per SM), for each value
type and both precisions: FP64 equal to the FP64 oracle bit for bit, FP32 within
the rounding of its chain (n links: n + 1 units of 2^-24 of the magnitudes)."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [1, 2, 3, 4, 5, 6, 7, 8, 10.5])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_residuals(cuda_ok, groups, dtype):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m, n = int(32 * sms * groups) - 5, 131
    s = W.gaussian_dense(m, n, seed=m, num_blocks=max(1, m // 200), lam=1.0)
    s.dense = np.ascontiguousarray(s.dense.astype(dtype))
    rng = np.random.default_rng(1)
    x, b = rng.standard_normal(n), rng.standard_normal(m)
    with B.Handle.from_system(s, precision=B.PREC_MIXED) as h:
        r = torch.empty(m, dtype=torch.float64, device="cuda")
        rr = h.residual(torch.as_tensor(b, device="cuda"), torch.as_tensor(x, device="cuda"), r)
        x32, b32 = x.astype(np.float32), b.astype(np.float32)
        r32 = torch.empty(m, dtype=torch.float32, device="cuda")
        h.residual32(torch.as_tensor(b32, device="cuda"), torch.as_tensor(x32, device="cuda"), r32)
    ref = oracle.residual(s, b, x)[0]
    np.testing.assert_array_equal(r.cpu().numpy(), ref)
    assert rr == pytest.approx(float(ref @ ref), rel=1e-12)
    A = s.dense.astype(np.float32).astype(np.float64)
    bound = (n + 1) * 2.0 ** -24 * (np.abs(A) @ np.abs(x32.astype(np.float64)) + np.abs(b32))
    assert np.all(np.abs(r32.cpu().numpy() - (b32 - A @ x32.astype(np.float64))) <= bound)
