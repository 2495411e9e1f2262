"""The moment step over the widths where its kernels change: 1 to 66 live
probes (groups of 1 to 32 lanes, one or several column classes), patterns and
values, short, long and empty rows, X^T X, and column arrays that do not start
on a 16-byte boundary, each precision against the oracle.  Tolerances are those
of the other parity tests: 1e-10 d for FP64 and double-float, 64 2^-24 d for
FP32 (degrees up to 128)."""
import numpy as np
import pytest

from paper_2103_10516_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "df64": 1e-10, "fp32": 64 * 2.0 ** -24}
WIDTHS = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 18, 23, 33, 36, 42, 50, 66]


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    return mlt


MATS = {"rmat": (lambda: synth.rmat_adjacency(10, 12, seed=5), False),          # rows of 0 to several hundred entries
        "values": (lambda: synth.random_symmetric(300, 0.03, seed=6), False),
        "dense_rows": (lambda: synth.random_symmetric(180, 0.9, seed=6), False),   # every row longer than a segment
        "stencil": (lambda: synth.diffusion_3d(7, shift=0.3, seed=2), False),
        "gram": (lambda: synth.sparse_gaussian(400, 150, 0.03, seed=4), True)}


class _Dev:
    """CUDA copies of a CSR, the column array `shift` entries off its allocation's start."""

    def __init__(self, m, shift):
        import torch
        self.nrows, self.ncols, self.nnz = m.nrows, m.ncols, m.nnz
        self.rowptr = torch.from_numpy(m.rowptr).cuda()
        buf = torch.zeros(m.nnz + shift, dtype=torch.int32, device="cuda")
        buf[shift:] = torch.from_numpy(m.col).cuda()
        self.col = buf[shift:]
        self.val = None if m.val is None else torch.from_numpy(m.val).cuda()


@pytest.mark.parametrize("name", list(MATS))
@pytest.mark.parametrize("precision", list(TOL))
def test_widths(L, O, name, precision):
    make, gram = MATS[name]
    m = make()
    sc = 1.0 if gram else 1.0 / max(1.0, float(np.max(np.diff(m.rowptr))))
    a, b = O.interval(m, scale=sc, gram=gram)
    d = m.ncols
    ref = O.moments(m, a, b, 5, 40, np.full(max(WIDTHS), 16, dtype=np.int32), gram=gram, scale=sc)
    for shift in (0, 1):
        with L.Matrix(_Dev(m, shift), gram=gram, scale=sc) as M:
            for w in WIDTHS if shift == 0 else WIDTHS[:9]:
                # ragged: half of the probes stop at a lower degree, odd or even
                deg = np.where(np.arange(w) % 2 == 0, 16, w % 16).astype(np.int32)
                got = M.moments(a, b, 5, 40, deg, precision=precision)
                for p in range(w):
                    err = np.max(np.abs(got[p, :deg[p] + 1] - ref[p, :deg[p] + 1]))
                    assert err <= TOL[precision] * d, (w, p, err / d)
                    assert not got[p, deg[p] + 1:].any()


@pytest.mark.parametrize("deg", [4095, 4097, 5000])
@pytest.mark.parametrize("precision", list(TOL))
def test_hub_row_of_many_segments(L, O, deg, precision):
    """A vertex whose row has 32 segments of 128 entries, 33, and 40 (rows of 32
    or more take a whole CTA of the long-row kernel), next to a row of two."""
    d = 5200
    e = [(0, j) for j in range(1, deg + 1)] + [(deg + 1, j) for j in range(1, 180)] + [(j, j + 1) for j in range(1, 900)]
    r, c = np.array([x for x, _ in e] + [y for _, y in e]), np.array([y for _, y in e] + [x for x, _ in e])
    key = np.unique(r.astype(np.int64) * d + c)
    m = synth._from_coo(d, d, key // d, key % d)
    sc = 1.0 / deg
    a, b = O.interval(m, scale=sc)
    for w in (1, 3, 16, 65, 130):
        degs = np.full(w, 8, dtype=np.int32)
        ref = O.moments(m, a, b, 5, 7, degs[:3], scale=sc)
        with L.Matrix(m, scale=sc) as M:
            got = M.moments(a, b, 5, 7, degs, precision=precision)
        assert np.max(np.abs(got[:3] - ref[:w])) <= TOL[precision] * d
