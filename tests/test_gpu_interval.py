"""Lanczos intervals (mlt_spectrum_bounds) against the same recurrence in numpy,
on operators whose rows take each of the product's paths: rows shorter and
longer than a segment (128 entries for small operators), empty rows, a hub row
of several segments with a remainder, patterns and values, X^T X, relabelled
handles, and column arrays that do not start on a 16-byte boundary.  Four
steps: further Ritz pairs would converge on these small operators, and the
residual of a converged pair is rounding noise."""
import numpy as np
import pytest

from paper_2103_10516_gb300 import synth

pytestmark = pytest.mark.gpu
STEPS, SEED = 4, 9


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    return mlt


def _hub(d, deg, val):
    """A star-like symmetric matrix: vertex 0 joined to 1..deg, a ring over the
    next d/2 vertices, the rest isolated."""
    a = np.zeros((d, d))
    a[0, 1:deg + 1] = a[1:deg + 1, 0] = 1.0
    for i in range(1, d // 2):
        a[i, i + 1] = a[i + 1, i] = 1.0
    if val:
        rng = np.random.default_rng(deg)
        w = rng.standard_normal((d, d))
        a *= w + w.T
    r, c = np.nonzero(a)
    return synth._from_coo(d, d, r, c, a[r, c] if val else None)


def _reference(mul, d, z, gram):
    q, prev, bprev, al, be = z / np.sqrt(d), np.zeros(d), 0.0, [], []
    for _ in range(min(STEPS, d)):
        w = mul(q)
        a = q @ w
        w = w - a * q - bprev * prev
        b = np.linalg.norm(w)
        al.append(a)
        be.append(b)
        prev, q, bprev = q, w / b, b
    n = len(al)
    th, S = np.linalg.eigh(np.diag(al) + np.diag(be[:n - 1], 1) + np.diag(be[:n - 1], -1))
    lo, hi = th[0] - be[-1] * abs(S[-1, 0]), th[-1] + be[-1] * abs(S[-1, -1])
    lo, hi = lo - 0.01 * abs(lo), hi + 0.01 * abs(hi)
    return (max(lo, 1e-6 * hi) if gram else lo), hi


@pytest.mark.parametrize("case", ["ring", "hub127", "hub128", "hub129", "hub700", "hub700_val", "rmat", "stencil",
                                  "gram", "gram_wide"])
@pytest.mark.parametrize("form", ["host", "reorder", "unaligned"])
def test_lanczos_interval(L, O, case, form):
    import torch
    gram = case.startswith("gram")
    if gram and form == "reorder":
        pytest.skip("relabelling needs a square operator")
    m = {"ring": lambda: _hub(64, 1, False), "rmat": lambda: synth.rmat_adjacency(11, 16, seed=3),
         "stencil": lambda: synth.diffusion_3d(9, shift=0.2, seed=1),
         "gram": lambda: synth.sparse_gaussian(900, 300, 0.02, seed=2),
         "gram_wide": lambda: synth.sparse_gaussian(40, 700, 0.4, seed=2)}.get(
        case, lambda: _hub(1000, int(case[3:].split("_")[0]), case.endswith("val")))()
    d = m.ncols
    a = m.to_dense()
    z = np.asarray(O.rademacher(SEED, 0, d), dtype=np.float64)
    lo, hi = _reference((lambda v: a.T @ (a @ v)) if gram else (lambda v: a @ v), d, z, gram)
    if form == "unaligned":
        class T:
            pass
        t = T()
        t.nrows, t.ncols, t.nnz = m.nrows, m.ncols, m.nnz
        t.rowptr = torch.from_numpy(m.rowptr).cuda()
        buf = torch.empty(m.nnz + 1, dtype=torch.int32, device="cuda")
        buf[1:] = torch.from_numpy(m.col).cuda()
        t.col = buf[1:]
        t.val = None if m.val is None else torch.from_numpy(m.val).cuda()
        M = L.Matrix(t, gram=gram)
    else:
        M = L.Matrix(m, gram=gram, reorder=form == "reorder")
    with M:
        got = L.mlt_spectrum_bounds(M.handle, L.MLT_BOUNDS_LANCZOS, STEPS, SEED)
    # four steps of FP64 sums over at most 1000 terms: 1e-11 of the interval's
    # size leaves a factor of about 100 over their roundings
    assert abs(got[0] - lo) <= 1e-11 * max(abs(lo), abs(hi)), (got, lo, hi)
    assert abs(got[1] - hi) <= 1e-11 * max(abs(lo), abs(hi)), (got, lo, hi)



def _profiled_interval(L, M, steps):
    import torch
    L.mlt_profile_start()
    iv = L.mlt_spectrum_bounds(M.handle, L.MLT_BOUNDS_LANCZOS, steps, SEED)
    torch.cuda.synchronize()
    return tuple(iv), L.mlt_profile_stop()


def test_rows_are_sorted_only_where_it_pays(L):
    """A call on rows of even length prepares nothing but its vectors."""
    for m, gram in ((synth.diffusion_3d(24, shift=0.2, seed=1), False), (synth.sparse_gaussian(3000, 2000, 0.01, seed=2), True)):
        with L.Matrix(m, gram=gram) as M:
            _profiled_interval(L, M, 2)
            assert "lanczos_setup" not in _profiled_interval(L, M, 2)[1]


def test_order_of_rows_changes_no_bit(L):
    """Rows in storage order (5 steps), sorted (40) and in the order of a relabelled
    handle: each row is summed on its own, in entry order."""
    m = synth.rmat_adjacency(16, 16, seed=3)
    with L.Matrix(m) as M, L.Matrix(m, reorder=True) as R:
        for steps, is_sorted in ((5, False), (40, True)):
            iv, prof = _profiled_interval(L, M, steps)
            assert ("lanczos_setup" in prof) == is_sorted
            assert iv == _profiled_interval(L, R, steps)[0]


@pytest.mark.parametrize("deg", [1024, 1400, 4500])
def test_hub_of_many_segments(L, O, deg):
    """8 segments, 11, and 36: the loop over a row's segments takes eight at a time."""
    m = _hub(max(1500, deg + 300), deg, True)
    a, d = m.to_dense(), m.ncols
    z = np.asarray(O.rademacher(SEED, 0, d), dtype=np.float64)
    lo, hi = _reference(lambda v: a @ v, d, z, False)
    with L.Matrix(m) as M:
        got = L.mlt_spectrum_bounds(M.handle, L.MLT_BOUNDS_LANCZOS, STEPS, SEED)
    # sums of up to 4500 terms: five times the bound for 1000 terms above
    assert abs(got[0] - lo) <= 5e-11 * max(abs(lo), abs(hi)), (got, lo, hi)
    assert abs(got[1] - hi) <= 5e-11 * max(abs(lo), abs(hi)), (got, lo, hi)
