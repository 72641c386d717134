"""What a value refresh takes from the device while it runs: the scratch of the
set-up (the operators' in the place of the centroids'), and a copy of the values
only where they are not on the device yet, given back before the set-up's
scratch is taken."""
import threading

import numpy as np
import pytest

from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _peak(call):
    """Most device memory in use during call(), above the use before it (polled
    from another thread: the library's calls run without the interpreter lock)."""
    torch.cuda.synchronize()
    free0, low, stop = torch.cuda.mem_get_info()[0], [], threading.Event()

    def poll():
        while not stop.is_set():
            low.append(torch.cuda.mem_get_info()[0])
    t = threading.Thread(target=poll)
    t.start()
    try:
        call()
    finally:
        stop.set()
        t.join()
    return free0 - min(low)


def test_refresh_holds_no_copy_of_the_values_beside_the_scratch(cuda_ok):
    m, n = 49152, 2048                               # 768 MB of values; operators of 256 rows
    g = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randn(m, n, generator=g, device="cuda", dtype=torch.float64)
    host = v.cpu().numpy()
    s = W.System("gaussian", m, n, dense=host, b=np.ones(m), num_blocks=m // 256, lam=1e-3)
    size = v.numel() * 8
    with B.Handle.from_system(s) as h:
        h.update_values(v)                           # (kernels loaded)
        on_device = _peak(lambda: h.update_values(v))
        on_host = _peak(lambda: h.update_values(host))
    assert on_device < size / 4                      # 192 operators of 512 KB and small change
    assert on_host < size + on_device / 2


def test_refresh_scratch_of_a_sparse_system_is_shared(cuda_ok):
    """4,096 blocks of 64 rows that share a column: the centroids' Gram and the
    operators take 128 MB each."""
    m, k = 1 << 18, 4096
    rows = np.arange(m)
    cols = np.stack([rows, m + rows // 64], 1).astype(np.int32)
    vals = np.stack([np.full(m, 2.0), np.random.default_rng(1).uniform(1, 2, m)], 1)
    s = W.System("blocks", m, m + k, row_ptr=2 * np.arange(m + 1), col_idx=cols.ravel(), values=vals.ravel(),
                 b=np.ones(m), num_blocks=k, lam=1e-3)
    v = torch.as_tensor(vals.ravel(), device="cuda")
    with B.Handle.from_system(s) as h, B.Handle.from_system(s) as fresh:
        h.update_values(v)
        assert _peak(lambda: h.update_values(v)) < 200e6
        np.testing.assert_array_equal(h.proposal()[0], fresh.proposal()[0])
        for t in (0, 2049, k - 1):
            np.testing.assert_array_equal(h.static_operator(t, 64), fresh.static_operator(t, 64))
