"""A CTA's running dots are merged without losing the precision they have.

One row a thread: a diagonal operator of 256 double-float values a_i in (0.5,
1) with the interval [-1, 1], so that V_1 = a z and every thread's dot V_1 . z
is a_i exactly.  mu_1 is then the sum of 256 numbers of 48 bits, added at most
14 deep (3 in a lane, 3 between lanes, 8 between warps): with the precision of
FP64 that is 14 2^-53 of it.  The seed is one for which adding them as
double-float pairs loses 1.0e-14, seven times that."""
import math

import numpy as np
import pytest

from paper_2103_10516_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "df64"])
def test_dots_merge_with_the_precision_of_fp64(precision):
    import torch
    assert torch.cuda.is_available()
    from paper_2103_10516_gb300 import build, mlt
    build.build()
    x = np.random.default_rng(934).uniform(0.5, 1.0, 256)
    hi = x.astype(np.float32).astype(np.float64)
    a = hi + (x - hi).astype(np.float32).astype(np.float64)
    i = np.arange(256)
    with mlt.Matrix(synth._from_coo(256, 256, i, i, a)) as M:
        mu = M.moments(-1.0, 1.0, 1, 0, np.array([1], dtype=np.int32), precision=precision)
    want = math.fsum(a)
    assert abs(mu[0, 1] - want) <= 14 * 2.0 ** -53 * want
