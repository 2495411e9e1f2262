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


def _release():
    import gc

    import torch
    from paper_2103_10516_gb300 import mlt
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    mlt.mlt_release_cached()


@pytest.fixture(autouse=True)
def _give_back(L):
    yield
    _release()


def _need(gb):
    import torch
    _release()
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


def test_gram_rows(L, O):
    """X^T X for an X whose entries lie in its first and last rows: the product
    X V runs over 2^31 - 1 rows.  With the interval [-8, 8] the moments are
    multiples of 1/64."""
    _need(225)
    n, d, probes = LIMIT, 64, 3
    rows = list(range(4)) + list(range(n - 44, n))
    e = [(r, c) for i, r in enumerate(rows) for c in sorted(((5 * i) % d, (7 * i + 3) % d)) if (5 * i) % d != (7 * i + 3) % d]
    x = np.zeros((len(rows), d))
    for r, c in e:
        x[rows.index(r), c] = 1.0
    at = x.T @ x / 8.0
    assert np.linalg.eigvalsh(at)[-1] < 1.0
    z = np.array([[_sign(O, p, i) for i in range(d)] for p in range(probes)], dtype=np.float64).T
    want = np.array([np.full(probes, float(d)), np.sum(z * (at @ z), axis=0), 2.0 * np.sum((at @ z) ** 2, axis=0) - d]).T
    with L.Matrix(_device_csr(n, d, *_rows(n, e)), gram=True) as M:
        for precision in ("fp64", "df64", "fp32"):
            mu = M.moments(-8.0, 8.0, SEED, 0, np.full(probes, 2, dtype=np.int32), precision=precision)
            assert np.array_equal(mu, want), precision


def _entries(d, width):
    """A d-row pattern of LIMIT entries: row i holds `width` consecutive columns
    from _first(i) on, the last row one fewer."""
    import torch
    col = torch.empty(LIMIT, dtype=torch.int32, device="cuda")
    j = torch.arange(width, dtype=torch.int32, device="cuda")
    step = 4096
    for r in range(0, d, step):
        i = torch.arange(r, min(r + step, d), dtype=torch.int64, device="cuda")
        block = (_first(i, d, width).to(torch.int32)[:, None] + j).reshape(-1)
        col[r * width:r * width + block.numel()] = block[:min(block.numel(), LIMIT - r * width)]
    rowptr = torch.arange(d + 1, dtype=torch.int64, device="cuda") * width
    rowptr[d] = LIMIT
    return rowptr, col


def _first(i, d, width):
    return (i * 977) % (d - width)


def _apply(v, d, width):
    s = np.concatenate([[0.0], np.cumsum(v)])
    f = _first(np.arange(d), d, width)
    e = f + width
    e[-1] -= 1
    return s[e] - s[f]


@pytest.mark.parametrize("width", [2 ** 11, 2 ** 13], ids=["rows", "segments"])
def test_entries(L, O, width):
    """Rows shorter and longer than a segment (4096 entries at this size), up to
    the last entry.  With the interval [-2^k, 2^k] the first step is exact in
    FP64 and double-float; FP32 dots are within 2^-23 of the sum of their terms'
    magnitudes.  The Lanczos interval's first step is exact but for its square
    roots and quotients."""
    d = 2 ** 31 // width
    _need(60)
    probes = 66
    z = np.array([O.rademacher(SEED, p, d) for p in range(probes)], dtype=np.float64)
    y = np.array([_apply(v, d, width) for v in z])
    b = 4.0 * width
    want = np.array([np.full(probes, float(d)), np.sum(z * y, axis=1) / b, 2.0 * np.sum(y * y, axis=1) / b ** 2 - d]).T
    size = np.array([np.zeros(probes), np.sum(np.abs(y), axis=1) / b, 2.0 * np.sum(y * y, axis=1) / b ** 2]).T
    with L.Matrix(_device_csr(d, d, *_entries(d, width))) as M:
        for precision in ("fp64", "df64", "fp32"):
            for w in (1, 3, 8, 16, 32, 66):
                mu = M.moments(-b, b, SEED, 0, np.full(w, 2, dtype=np.int32), precision=precision)
                err = np.abs(mu - want[:w])
                assert np.all(err <= (2.0 ** -23 * size[:w] if precision == "fp32" else 0.0)), (precision, w, err.max())
        lo, hi = L.mlt_spectrum_bounds(M.handle, L.MLT_BOUNDS_LANCZOS, 2, SEED)
    # two steps by hand, in the library's order
    q0 = z[0] / np.sqrt(d)
    w0 = _apply(q0, d, width)
    a0 = q0 @ w0
    w0 = w0 - a0 * q0
    b0 = np.linalg.norm(w0)
    q1 = w0 / b0
    w1 = _apply(q1, d, width)
    a1 = q1 @ w1
    b1 = np.linalg.norm(w1 - a1 * q1 - b0 * q0)
    th, S = np.linalg.eigh(np.array([[a0, b0], [b0, a1]]))
    e0, e1 = th[0] - b1 * abs(S[1, 0]), th[1] + b1 * abs(S[1, 1])
    # prefix sums of d terms up to sqrt(d): 2^-53 d per entry of the products here
    assert abs(lo - (e0 - 0.01 * abs(e0))) <= 1e-9 * abs(e1)
    assert abs(hi - (e1 + 0.01 * abs(e1))) <= 1e-9 * abs(e1)
