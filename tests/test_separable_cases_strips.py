"""The GPU tests that set strong coefficients on a separable handle
(test_gpu_separable_choice.py) reach every number of row strips, 1 to 32: the
choice of k_sep_params, over the tiles and spots of their problems, on the CPU."""
from math import comb

import numpy as np

from test_separable_model import EXPS, TOL, _dropped, _monomials
from workloads import random_problem

MIXED = ((1, 1), (2, 1), (1, 2), (2, 2), (3, 1), (1, 3))


def _strips(nx, ny, noll, C):
    """log2 of the strips of every (tile, spot)."""
    mono, R = _monomials(noll), min(nx, ny) / 2.0
    out = []
    for ty in range(0, ny, 32):
        for tx in range(0, nx, 32):
            xc, yc = (tx + 16 - (nx - 1) / 2) / R, (ty + 16 - (ny - 1) / 2) / R
            row = {q: 0.0 for q in MIXED}
            for (a, b), w in zip(EXPS, mono):
                for k, l in MIXED:
                    if k <= a and l <= b:
                        row[k, l] = row[k, l] + w * comb(a, k) * comb(b, l) * xc**(a - k) * yc**(b - l) * (16 / R)**(k + l)
            a11, a21, a12, a22, a31, a13 = (np.abs(C @ row[q]) for q in MIXED)
            k = np.full(len(C), 5)
            for q in range(4, 0, -1):
                f = 0.5**q
                k[_dropped(f * (a11 + 2 * a12 + 3 * a13), f * (a21 + 2 * a22), f * a31) <= TOL] = q
            k[_dropped(a11 + a12 + a13, a21 + a22, a31) <= TOL] = 0
            out.append(k)
    return np.concatenate(out)


def test_strong_coefficients_reach_every_strip_count():
    seen = set()
    for nx, ny, N, scale in ((577, 590, 100, 30.0), (640, 600, 97, 6.0), (905, 903, 161, 30.0)):
        p = random_problem(nx + 3 * ny + N, nx, ny, N, list(range(2, 12)), defocus_max=5.0)
        seen |= set(_strips(nx, ny, p.noll, p.coeff.astype(np.float64) * scale).tolist())
    assert seen == {0, 1, 2, 3, 4, 5}
