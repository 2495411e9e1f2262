"""Operators whose rows are cut into 32 segments and more (128 entries each on
these sizes), a few such rows (a CTA each in the long-row kernel) and more of
them than CTAs (groups take them), rows of one segment fewer, and the kernel's
three uses (recurrence, Clenshaw step, X V of X^T X), every column against
numpy.  Tolerances are those of the other parity
tests: 1e-10 d for FP64 and double-float, 64 2^-24 d for FP32; a segment
left out of one hub row moves the moments by many times that (checked here on
the CPU, with the mistake in the reference)."""
import numpy as np
import pytest

from paper_2103_10516_gb300 import synth

TOL = {"fp64": 1e-10, "df64": 1e-10, "fp32": 64 * 2.0 ** -24}
D, DEG, SEED, OFF = 4200, 8, 5, 7
WIDTHS = (1, 3, 8, 16, 33, 65, 130)


@pytest.fixture(scope="module")
def L():
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    return mlt


def _hub_rows(nh):
    """Symmetric, entries +-1: the first nh rows and columns full, else diagonal;
    with the scale that brings its spectrum into (-1, 1)."""
    rng = np.random.default_rng(nh)
    a = np.sign(rng.standard_normal((D, D)))
    a = np.triu(a, 1)
    a = a + a.T
    a[nh:, nh:] = 0.0
    np.fill_diagonal(a, 1.0)
    return a, 0.9 / (np.sqrt(D) * (2.0 if nh == D else 1.0 + np.sqrt(nh / D)) + 1.0)


def _one_hub(deg):
    """Symmetric, entries +-1: vertex 0 joined to 1 .. deg, and a diagonal."""
    rng = np.random.default_rng(deg)
    a = np.eye(D)
    a[0, 1:deg + 1] = a[1:deg + 1, 0] = np.sign(rng.standard_normal(deg))
    return a, 0.9 / (np.sqrt(deg) + 1.0)


def _csr(a):
    r, c = np.nonzero(a)
    return synth._from_coo(a.shape[0], a.shape[1], r, c, a[r, c])


def _moments(a, scale, z):
    """z^T T_j(scale a) z for j <= DEG (the interval is [-1, 1])."""
    v0, v1 = z, scale * (a @ z)
    mu = [np.sum(z * z, axis=0), np.sum(z * v1, axis=0)]
    for _ in range(DEG - 1):
        v0, v1 = v1, 2.0 * scale * (a @ v1) - v0
        mu.append(np.sum(z * v1, axis=0))
    return np.array(mu).T


def _probes(O, n):
    return np.array([O.rademacher(SEED, OFF + p, D) for p in range(n)], dtype=np.float64).T


@pytest.mark.parametrize("nh", [20, D])
def test_a_lost_segment_shows(O, nh):
    a, sc = _hub_rows(nh)
    z = _probes(O, 130)
    ref = _moments(a, sc, z)
    row = a[0].copy()
    for s in (0, 1, 16, 31, 32):          # the first, inner ones, and the remainder
        a[0, 128 * s:128 * (s + 1)] = 0.0
        assert np.max(np.abs(_moments(a, sc, z) - ref)) > 4 * TOL["fp32"] * D, s
        a[0] = row


@pytest.mark.gpu
@pytest.mark.parametrize("nh", [20, D])
@pytest.mark.parametrize("precision", list(TOL))
def test_moments(L, O, nh, precision):
    a, sc = _hub_rows(nh)
    ref = _moments(a, sc, _probes(O, max(WIDTHS)))
    with L.Matrix(_csr(a), scale=sc) as M:
        for w in WIDTHS:
            got = M.moments(-1.0, 1.0, SEED, OFF, np.full(w, DEG, dtype=np.int32), precision=precision)
            assert np.max(np.abs(got - ref[:w])) <= TOL[precision] * D, w


# 31 segments with the diagonal entry, 32, 33 of which the last has one entry
HUBS = [31 * 128 - 1, 32 * 128 - 1, 32 * 128]


@pytest.mark.parametrize("deg", HUBS)
def test_a_lost_segment_of_one_hub_shows(O, deg):
    a, sc = _one_hub(deg)
    z = _probes(O, 130)
    ref = _moments(a, sc, z)
    row = a[0].copy()
    for s in (1, deg // 128):             # an inner segment and the last
        a[0, 128 * s:128 * (s + 1)] = 0.0
        assert np.max(np.abs(_moments(a, sc, z) - ref)) > 2 * TOL["fp32"] * D, s
        a[0] = row


@pytest.mark.gpu
@pytest.mark.parametrize("deg", HUBS)
@pytest.mark.parametrize("precision", list(TOL))
def test_moments_around_the_threshold(L, O, deg, precision):
    a, sc = _one_hub(deg)
    ref = _moments(a, sc, _probes(O, max(WIDTHS)))
    with L.Matrix(_csr(a), scale=sc) as M:
        for w in WIDTHS:
            got = M.moments(-1.0, 1.0, SEED, OFF, np.full(w, DEG, dtype=np.int32), precision=precision)
            assert np.max(np.abs(got - ref[:w])) <= TOL[precision] * D, w


@pytest.mark.gpu
@pytest.mark.parametrize("make", [lambda: _hub_rows(20), lambda: _hub_rows(D), lambda: _one_hub(31 * 128 - 1)],
                         ids=["20", "all", "31"])
def test_clenshaw(L, make):
    """p(At) X through Clenshaw's recurrence; the tolerance is that of the other
    polynomial applications, 1e-10 sum|c| max|X|."""
    a, sc = make()
    c = np.random.default_rng(3).standard_normal(DEG + 1)
    for w in (1, 5, 40, 130):
        x = np.random.default_rng(w).standard_normal((D, w))
        t0, t1 = x, sc * (a @ x)
        want = c[0] * t0 + c[1] * t1
        for k in range(2, DEG + 1):
            t0, t1 = t1, 2.0 * sc * (a @ t1) - t0
            want += c[k] * t1
        with L.Matrix(_csr(a), scale=sc) as M:
            got = L.mlt_poly_apply(M.handle, -1.0, 1.0, c, x)
        assert np.max(np.abs(got - want)) <= 1e-10 * np.sum(np.abs(c)) * np.max(np.abs(x)), w


@pytest.mark.gpu
@pytest.mark.parametrize("tall", [False, True], ids=["wide", "tall"])
@pytest.mark.parametrize("precision", list(TOL))
def test_gram_moments(L, O, tall, precision):
    """X^T X for an X with rows of 33 and 31 segments, and for its transpose."""
    rng = np.random.default_rng(4)
    x = np.where(rng.random((60, D)) < 0.01, rng.standard_normal((60, D)), 0.0)
    x[0] = np.sign(rng.standard_normal(D))
    x[7, :31 * 128] = np.sign(rng.standard_normal(31 * 128))
    if tall:
        x = x.T
    d = x.shape[1]
    n = 1.01 * np.linalg.norm(x, 2) ** 2
    z = np.array([O.rademacher(SEED, OFF + p, d) for p in range(max(WIDTHS))], dtype=np.float64).T
    at = 2.0 / n * (x.T @ x) - np.eye(d)
    ref = _moments(at, 1.0, z)
    with L.Matrix(_csr(x), gram=True) as M:
        for w in WIDTHS:
            got = M.moments(0.0, n, SEED, OFF, np.full(w, DEG, dtype=np.int32), precision=precision)
            assert np.max(np.abs(got - ref[:w])) <= TOL[precision] * d, w


@pytest.mark.gpu
def test_many_long_rows_do_not_queue(L):
    """With more such rows than CTAs, adding up their segments costs less than
    computing them, whatever the width (a CTA a row, one row after another, took
    six times as long for one FP64 probe)."""
    import torch
    a, sc = _hub_rows(D)
    with L.Matrix(_csr(a), scale=sc) as M:
        for w in (1, 8):
            ms = {}
            for _ in range(4):
                L.mlt_profile_start()
                M.moments(-1.0, 1.0, SEED, OFF, np.full(w, DEG, dtype=np.int32))
                torch.cuda.synchronize()
                for k, (n, t) in L.mlt_profile_stop().items():
                    ms[k] = min(t, ms.get(k, t))
            assert ms["cheb_step_long"] < ms["cheb_step"], (w, ms)
