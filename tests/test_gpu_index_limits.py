"""Operators of 2^31 - 1 rows or entries, the most that a handle takes: indices
that run a batch or a few rows ahead of the last one must not wrap.  The
reference is exact (small integers) and computed from the structure; a test
is skipped where the device has not the memory it needs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LIMIT = 2 ** 31 - 1
SEED = 3


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    return mlt


def _need(gb):
    import gc

    import torch
    from paper_2103_10516_gb300 import mlt
    gc.collect()
    torch.cuda.empty_cache()
    mlt.mlt_release_cached()
    if torch.cuda.mem_get_info()[0] < gb * 1e9:
        pytest.skip("needs %d GB of free device memory" % gb)


class _Csr:
    pass


def _device_csr(nrows, ncols, rowptr, col):
    m = _Csr()
    m.nrows, m.ncols, m.nnz, m.rowptr, m.col, m.val = nrows, ncols, int(col.numel()), rowptr, col, None
    return m


def _rows(n, entries):
    """CUDA CSR arrays of an n-row pattern whose entries (row, column), in order,
    lie in a few rows."""
    import torch
    r = torch.tensor([i for i, _ in entries], device="cuda")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    for i in range(len(entries)):
        rowptr[int(r[i]) + 1:].add_(1)
    return rowptr, torch.tensor([j for _, j in entries], dtype=torch.int32, device="cuda")


def _sign(O, p, i):
    return int(O.lib().orc_rademacher(SEED, p, i))


def test_rows(L, O):
    """A square operator with edges between its first and last vertices; V_1 = A z
    and both moments are small integers."""
    _need(225)
    n = LIMIT
    edges = [(0, n - 1), (1, n - 2), (n - 3, n - 40), (n - 35, n - 300)]
    e = sorted(edges + [(j, i) for i, j in edges])
    with L.Matrix(_device_csr(n, n, *_rows(n, e))) as M:
        mu = M.moments(-1.0, 1.0, SEED, 0, np.full(3, 2, dtype=np.int32), precision="fp32")
    for p in range(3):
        assert mu[p, 0] == n
        assert mu[p, 1] == sum(2 * _sign(O, p, i) * _sign(O, p, j) for i, j in edges)
        assert mu[p, 2] == 2 * len(e) - n
