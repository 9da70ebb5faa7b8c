"""CPU model of the separable tile transforms (csrc/sep_common.cuh) against
the direct phase factors.

Over a 32 x 32 tile, exp(-i C.Z) = Y(v) X(u) exp(-i r) with the mixed terms
r = u R1(v) + u^2 R2(v) + u^3 R3(v) taken about the middle row of one of 2^k
row strips, and exp(-i r) as a cubic in u whose u^4 term enters as u^2. The
model follows the choice of k in k_sep_params and the cubic of the kernels, in
float64, for every order and mode set that they accept, on odd grids with
ragged tiles and for aberrations that need 1 to 32 strips. Bound, by the rule
itself: 1e-6 per pixel, and below a tenth of that for the orders its estimate
leaves out (R1^6 / 720 where R1^4 / 96 < 1e-6).
"""
from math import comb

import numpy as np
import pytest

from oracle import zernike

TOL = 1e-6
EXPS = [(a, b) for a in range(5) for b in range(5 - a)]


def _monomials(noll):
    rng = np.random.default_rng(0)
    x, y = rng.uniform(-1, 1, (2, 400))
    V = np.stack([x**a * y**b for a, b in EXPS], 1)
    Z = np.stack([zernike.zernike_polar(*zernike.noll_to_nm(j), np.hypot(x, y), np.arctan2(y, x)) for j in noll], 1)
    return np.linalg.lstsq(V, Z, rcond=None)[0]          # [15, D]


def _dropped(R1, R2, R3):
    s = R1 * R1
    e4 = s * s / 24 + 0.5 * s * R2 + 0.5 * R2 * R2
    e5 = s * s * R1 / 120 + s * R1 * R2 / 6 + 0.5 * R1 * R2 * R2 + 0.5 * s * R3 + R2 * R3
    return 0.25 * e4 + R1 * R3 + e5


def _strips(p):
    a11, a21, a12, a22, a31, a13 = (abs(p[k]) for k in ((1, 1), (2, 1), (1, 2), (2, 2), (3, 1), (1, 3)))
    if _dropped(a11 + a12 + a13, a21 + a22, a31) <= TOL:
        return 0
    for k in range(1, 5):
        f = 0.5**k
        if _dropped(f * (a11 + 2 * a12 + 3 * a13), f * (a21 + 2 * a22), f * a31) <= TOL:
            return k
    return 5


@pytest.mark.parametrize("nx,ny", [(71, 45), (33, 130), (131, 131), (1, 40)])
@pytest.mark.parametrize("noll", [[2, 3], [4], [2, 3, 4, 5, 6], list(range(2, 11)), list(range(2, 16)), [5, 14, 11]])
def test_strips_and_cubic_reproduce_the_phase_factors(nx, ny, noll):
    rng = np.random.default_rng(nx + 10 * len(noll))
    mono, R = _monomials(noll), min(nx, ny) / 2.0
    Z = zernike.basis(nx, ny, noll).reshape(len(noll), ny, nx)
    m = np.arange(-16, 16) / 16.0
    seen = set()
    for scale in (1e-3, 1e-2, 0.1, 0.5, 2.0, 1e-4, 1e-5):
        c = scale * rng.normal(size=len(noll))
        direct = np.exp(-1j * np.tensordot(c, Z, 1))
        for ty in range(0, ny, 32):
            for tx in range(0, nx, 32):
                xc, yc = (tx + 16 - (nx - 1) / 2) / R, (ty + 16 - (ny - 1) / 2) / R
                p = {(k, l): 0.0 for k, l in EXPS}
                for (a, b), w in zip(EXPS, mono @ c):
                    for k in range(a + 1):
                        for l in range(b + 1):
                            p[k, l] += w * comb(a, k) * comb(b, l) * xc**(a - k) * yc**(b - l) * (16 / R)**(k + l)
                X = sum(p[k, 0] * m**k for k in range(1, 5))
                Y = np.exp(-1j * sum(p[0, l] * m**l for l in range(5)))
                rows = lambda v: (p[1, 1] * v + p[1, 2] * v**2 + p[1, 3] * v**3,     # noqa: E731
                                  p[2, 1] * v + p[2, 2] * v**2, p[3, 1] * v)
                k = _strips(p)
                seen.add(k)
                n = 32 >> k
                got = np.empty((32, 32), complex)
                for row in range(32):
                    mid = 0.0 if k == 0 else ((row // n) * n - 16 + 0.5 * (n - 1)) / 16
                    M = rows(mid)
                    R1, R2, R3 = (a - b for a, b in zip(rows(m[row]), M))
                    q2 = -R1**2 / 2 + R1**4 / 24 - R2**2 / 2 + 1j * R2 * (R1**2 / 2 - 1)
                    q3 = -R1 * R2 + 1j * (R1**3 / 6 - R3)
                    col = np.exp(-1j * (X + M[0] * m + M[1] * m**2 + M[2] * m**3))
                    got[row] = Y[row] * col * (1 - 1j * R1 * m + q2 * m**2 + q3 * m**3)
                ref = direct[ty:ty + 32, tx:tx + 32]
                err = np.abs(got[:ref.shape[0], :ref.shape[1]] - ref).max()
                assert err <= 1.1 * TOL, (scale, tx, ty, k, err)
    if len(noll) > 3 and min(nx, ny) > 1:
        assert len(seen) > 1, seen                    # tiles of one strip and of several both occur
    if noll in ([2, 3], [4]):
        assert seen == {0}                            # no mixed terms
