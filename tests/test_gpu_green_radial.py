"""Green's function samples of problems with two unbounded-like directions, taken from Chebyshev series in the
distance where that costs fewer evaluations, against the oracle's quadrature at every sample."""
import math

import numpy as np
import pytest

import oracle
from paper_2211_07777_gb300 import flups as F

pytestmark = pytest.mark.gpu

E, O, P, U = F.EVEN, F.ODD, F.PER, F.UNB

# large enough for the series (several hundred samples per panel's evaluations); spectral direction x, y, z;
# unequal spacings; a short smoothing length
CASES = [
    ((8, 96, 96), ((P, P), (U, U), (U, U)), "hej2", 2.0, (1 / 96, 1 / 96, 1 / 96)),
    ((128, 8, 64), ((U, U), (E, O), (U, O)), "hej4", 2.0, (1 / 128, 1 / 64, 1 / 128)),
    ((96, 72, 8), ((E, U), (U, U), (O, O)), "hej10", 2.0, (1 / 96, 1 / 72, 1 / 48)),
    ((192, 192, 6), ((U, U), (U, U), (E, E)), "hej2", 1.0, (1 / 192,) * 3),
]


@pytest.mark.parametrize("n,bc,kernel,eps,h", CASES, ids=["per-x", "quarter-y", "unequal-z", "eps-h"])
def test_samples_match_the_oracle(n, bc, kernel, eps, h):
    L = tuple(n[d] * h[d] for d in range(3))
    unb = [U in b for b in bc]
    ext, wn = [], []
    for d in range(3):
        l, r = bc[d]
        N = n[d]
        ext.append(N // 2 + 1 if l == P else N + 1 if l == r else 2 * N + 1 if U in bc[d] else N)
        g = np.arange(ext[d])
        wn.append(2 * math.pi * g / L[d] if l == P else math.pi * (g + (0.5 if l != r else 0.0)) / L[d])
    s = F.Solver(n, bc, h=h, L=L, prec=F.F64, green=kernel, eps_over_h=eps)
    try:
        samples, _ = F.flups_debug_green(s._s, int(np.prod(ext)))
    finally:
        s.close()
    got = samples.reshape(ext[2], ext[1], ext[0])
    ds = unb.index(False)
    da, db = [d for d in range(3) if d != ds]
    ra, rb = np.arange(ext[da]) * h[da], np.arange(ext[db]) * h[db]
    r = np.sqrt(rb[:, None] ** 2 + ra[None, :] ** 2)
    for k in {0, 1, ext[ds] - 1}:
        ref = oracle.green.hej_mixed(int(kernel[3:]) // 2, 2, np.full_like(r, wn[ds][k]), r, eps * max(h))
        out = np.take(got, k, axis=2 - ds)
        # both sides carry their quadrature's rounding (a few 1e-15 of the wavenumber's largest value), and the
        # device drops integrands below e^-50 over a range of at most 40, which is 1e-11 of the largest value at
        # the shortest waves (e^-20)
        tol = 2e-14 * np.abs(ref).max() + 40 * math.exp(-50.0) / (4 * math.pi)
        assert np.abs(out - ref).max() < tol, (k, np.abs(out - ref).max(), tol)
