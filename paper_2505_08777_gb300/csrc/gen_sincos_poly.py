"""Coefficients of the FP32-pipe sine / cosine (sincos2_poly in common.cuh).

With t = x / (2 pi), r = t - rint(t) in [-1/2, 1/2] and h = pi r (the half
angle), the device evaluates
    S(u) ~ sqrt(2) sin(pi r) / r,   C(u) ~ sqrt(2) cos(pi r),   u = r^2,
as polynomials of degree 4 in u, and then
    sin x = 2 sin h cos h = (r S) C,    cos x = 2 cos^2 h - 1 = C^2 - 1.
The coefficients are a weighted least-squares fit on Chebyshev nodes of r
(near-minimax for these smooth functions), computed in float64 and rounded
to float32. Running this file prints them and the worst absolute error of
sin x and cos x over r in [-1/2, 1/2], evaluated with float32 rounding after
every operation (an upper bound for the fused multiply-adds of the device).

It also prints the coefficients of cis2_turns (sep_common.cuh), whose error over
a turn has to vanish on average as well: with the zeros of sine and cosine
taken out,
    sin 2 pi r = r (1/4 - u) P(u),    cos 2 pi r = (1 - 16 u) Q(u),
P of degree 5 and Q of degree 6, evaluated with a rounding per fused
multiply-add as the device does.
"""
import numpy as np

DEG_S, DEG_C = 4, 4


def fit():
    k = np.arange(4000)
    r = 0.5 * np.cos(np.pi * (k + 0.5) / len(k))      # Chebyshev nodes on [-1/2, 1/2]
    r = r[np.abs(r) > 1e-6]
    u = r * r
    s_target = np.sqrt(2.0) * np.sin(np.pi * r) / r
    c_target = np.sqrt(2.0) * np.cos(np.pi * r)
    # weight the sine fit by |r| (its error enters sin x multiplied by r)
    Vs = np.vander(u, DEG_S + 1, increasing=True)
    Vc = np.vander(u, DEG_C + 1, increasing=True)
    s = np.linalg.lstsq(Vs * np.abs(r)[:, None], s_target * np.abs(r), rcond=None)[0]
    c = np.linalg.lstsq(Vc, c_target, rcond=None)[0]
    return s.astype(np.float32), c.astype(np.float32)


def evaluate(s, c, n=200001):
    f = np.float32
    r = np.linspace(-0.5, 0.5, n).astype(np.float32)
    u = (r * r).astype(f)
    S = np.full_like(u, s[-1])
    for a in s[-2::-1]:
        S = (S * u + a).astype(f)
    C = np.full_like(u, c[-1])
    for a in c[-2::-1]:
        C = (C * u + a).astype(f)
    sinx = ((r * S).astype(f) * C).astype(f)
    cosx = (C * C - f(1.0)).astype(f)
    x = 2.0 * np.pi * r.astype(np.float64)
    return float(np.max(np.abs(sinx - np.sin(x)))), float(np.max(np.abs(cosx - np.cos(x))))


ZEROS_S, ZEROS_C = 5, 6


def fit_zeros():
    k = np.arange(6000)
    r = 0.5 * np.cos(np.pi * (k + 0.5) / len(k))
    u = r * r
    wp, wq = r * (0.25 - u), 1.0 - 16.0 * u
    p = np.linalg.lstsq(np.vander(u, ZEROS_S + 1, increasing=True) * wp[:, None], np.sin(2 * np.pi * r), rcond=None)[0]
    q = np.linalg.lstsq(np.vander(u, ZEROS_C + 1, increasing=True) * wq[:, None], np.cos(2 * np.pi * r), rcond=None)[0]
    return p.astype(np.float32), q.astype(np.float32)


def evaluate_zeros(p, q, n=2000001):
    """Max and rms error of the sine, the same of the cosine, mean error of the cosine."""
    f = np.float32

    def fma(a, b, c):
        return (np.float64(a) * np.float64(b) + np.float64(c)).astype(f)
    r = np.linspace(-0.5, 0.5, n).astype(f)
    u = r * r
    P, Q = np.full_like(u, p[-1]), np.full_like(u, q[-1])
    for a in p[-2::-1]:
        P = fma(P, u, a)
    for a in q[-2::-1]:
        Q = fma(Q, u, a)
    x = 2.0 * np.pi * r.astype(np.float64)
    es, ec = (r * (f(0.25) - u)) * P - np.sin(x), fma(u, f(-16.0), f(1.0)) * Q - np.cos(x)
    return np.abs(es).max(), np.sqrt(np.mean(es * es)), np.abs(ec).max(), np.sqrt(np.mean(ec * ec)), np.mean(ec)


if __name__ == "__main__":
    s, c = fit()
    es, ec = evaluate(s, c)
    print("S:", ", ".join(f"{v:.9e}f" for v in s))
    print("C:", ", ".join(f"{v:.9e}f" for v in c))
    print(f"max |sin error| {es:.3e}, max |cos error| {ec:.3e}")
    p, q = fit_zeros()
    print("P:", ", ".join(f"{v:.9e}f" for v in p))
    print("Q:", ", ".join(f"{v:.9e}f" for v in q))
    print("sin max %.2e rms %.2e, cos max %.2e rms %.2e mean %.1e" % evaluate_zeros(p, q))
