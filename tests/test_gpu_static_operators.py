"""Static operators on both sides of what decides how they are formed: up to 64
coupled rows in shared memory and above in global memory, blocks whose entries are
staged or not (8,192 entries; rows of up to eight entries), blocks of both kinds in
one system, and block transposes by sorting or searching (8,192 entries).  W_t
equals the FP64 oracle's bit for bit, as do updates with it."""
import numpy as np
import pytest

import oracle
from paper_2510_02156_gb300 import binding as B
from paper_2510_02156_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _blocks(coupled, rows, length, seed):
    """Blocks of `rows` rows of `length` entries; block t's first coupled[t] rows share
    columns of the block (any two of them a few), the others have columns of their own."""
    rng = np.random.default_rng(seed)
    k = len(coupled)
    shared = max(2, 2 * length)
    n = k * shared + k * rows * length
    cols = []
    for t, c in enumerate(coupled):
        for i in range(rows):
            if i < c:
                own = t * shared + np.concatenate([[0], 1 + rng.choice(shared - 1, length - 1, replace=False)])
            else:
                own = k * shared + (t * rows + i) * length + np.arange(length)
            cols.append(np.sort(own))
    ci = np.concatenate(cols).astype(np.int32)
    m = k * rows
    return W.System("blocks", m, n, row_ptr=length * np.arange(m + 1), col_idx=ci,
                    values=rng.standard_normal(ci.size), b=rng.standard_normal(m), num_blocks=k, lam=1e-3)


CASES = {"edges_of_small": ([0, 2, 63, 64, 65, 100, 1, 64], 100, 12),
         "short_rows": ([65, 200, 0, 3], 200, 8),
         "nine_entries": ([65, 200, 0, 3], 200, 9),
         "small_only": ([64, 63, 2, 0], 80, 5),
         "large_only": ([200, 300], 300, 10),
         "entries_8192": ([70, 128], 128, 64),
         "entries_8256": ([70, 129], 129, 64),
         "entries_8320": ([40, 70], 160, 52)}


@pytest.mark.parametrize("name", sorted(CASES))
def test_operators_equal_oracle(cuda_ok, name):
    coupled, rows, length = CASES[name]
    s = _blocks(coupled, rows, length, 7)
    k = s.num_blocks
    v2 = s.values * np.random.default_rng(2).uniform(0.5, 2.0, s.values.size)
    s2 = W.System("blocks2", s.m, s.n, row_ptr=s.row_ptr, col_idx=s.col_idx, values=v2, b=s.b, num_blocks=k, lam=s.lam)
    x0 = np.random.default_rng(3).standard_normal(s.n)
    with B.Handle.from_system(s) as h:
        for system in (s, s2):
            if system is s2:
                h.update_values(torch.as_tensor(v2, device="cuda"))
            for t in range(k):
                Wo = oracle.static_operator(system, k, t, s.lam)
                np.testing.assert_array_equal(h.static_operator(t, rows), Wo)
                x = torch.as_tensor(x0.copy(), device="cuda")
                h.static_update(t, torch.as_tensor(s.b, device="cuda"), x)
                xo = oracle.update_with_inverse(system, np.arange(t * rows, (t + 1) * rows), Wo, s.b, x0)
                np.testing.assert_array_equal(x.cpu().numpy(), xo)
