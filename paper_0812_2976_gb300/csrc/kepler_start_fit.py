"""Coefficients of the solve's start in kc_pair.cuh (start_constants).

With s the real root of Mikkola's (1987) cubic, the start is

    E0 = M + e s (3 + c1 x + c2 x^2 + c3 x^3 + c4 x^4),   x = s^2,

c_i cubics in e.  One Newton step from E0 errs by (E0 - E)^2 e sin E /
(2 (1 - e cos E)) to leading order, so the fit minimises the largest
|E0 - E| sqrt(e sin E / (1 - e cos E)) over a grid of (M, e) by least squares
with weights moved towards the largest error.  Prints the 4 x 4 coefficients
(rows c1 .. c4, columns powers of e) and, with them rounded to four places, the
largest error of the start and of the Newton step for |M| up to pi, to the fit's
end and to what the kernels' mean anomalies reach (1.038 pi in kc_pair.cuh, 1.057
pi in kc_f64.cuh).  numpy only, under a minute.
"""
import numpy as np

MEAN = np.concatenate([np.geomspace(1e-6, 0.05, 400), np.linspace(0.05, 1.02 * np.pi, 1200)])
ECC = np.concatenate([np.linspace(0.0, 0.95, 58)[1:], 1.0 - np.geomspace(0.05, 1e-6, 16)[1:]])


def eccentric(M, e):
    E = np.minimum(M + 0.85 * e, np.pi + 0.3)
    for _ in range(12):
        s, c = np.sin(E), np.cos(E)
        f, f1 = E - e * s - M, 1.0 - e * c
        d = -f / f1
        d = -f / (f1 + 0.5 * d * e * s)
        d = -f / (f1 + 0.5 * d * e * s + d * d * e * c / 6.0)
        E = E + d
    return E


def cubic_root(M, e):
    r = 1.0 / (4.0 * e + 0.5)
    sa = np.sqrt((1.0 - e) * r)
    b = 0.5 * M * r / sa ** 3
    z = np.cbrt(b + np.sqrt(b * b + 1.0))
    return sa * (z - 1.0 / z)


def errors(coef, top):
    """Largest error of the start and of the Newton step for 0 < M <= top."""
    M = np.concatenate([MEAN[MEAN <= top], np.linspace(0.9 * top, top, 400)])
    start = step = 0.0
    for e in ECC:
        s, root = cubic_root(M, e), eccentric(M, e)
        c = [np.polyval(row[::-1], e) for row in coef]
        E = M + e * s * (3.0 + sum(k * s ** (2 * i + 2) for i, k in enumerate(c)))
        E1 = E - (E - e * np.sin(E) - M) / (1.0 - e * np.cos(E))
        start = max(start, float(np.abs(E - root).max()))
        step = max(step, float(np.abs(E1 - root).max()))
    return start, step


def fit(iterations=150):
    rows, rhs, weight = [], [], []
    for e in ECC:
        E, s = eccentric(MEAN, e), cubic_root(MEAN, e)
        rows.append(np.stack([s ** (2 * i) * e ** k for i in range(1, 5) for k in range(4)], 1)
                    * (e * s)[:, None])
        rhs.append(E - MEAN - 3.0 * e * s)
        weight.append(np.sqrt(e * np.abs(np.sin(E)) / (1.0 - e * np.cos(E)) + 1e-3))
    A, y, W = (np.concatenate(x) for x in (rows, rhs, weight))
    w, best = W.copy(), None
    for _ in range(iterations):
        scale = np.linalg.norm(A * w[:, None], axis=0)
        c = np.linalg.lstsq(A * w[:, None] / scale, y * w, rcond=1e-14)[0] / scale
        r = np.abs(A @ c - y) * W
        if best is None or r.max() < best[0]:
            best = (r.max(), c)
        w = np.maximum(w * (r / r.max() + 0.02) ** 0.25, 1e-9)
        w /= w.max()
    return best[1].reshape(4, 4)


if __name__ == "__main__":
    coef = np.round(fit(), 4)
    print(coef)
    for top in (1.0, 1.02, 1.038, 1.057):
        print("|M| <= %.3f pi: largest error of the start %.2e rad, of the Newton step %.2e"
              % (top, *errors(coef, top * np.pi)))
