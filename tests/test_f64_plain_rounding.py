"""Host check of the FP64 forward kernels' arithmetic: an Endpoint deposit formed as
OpsF64Plain forms it (reciprocal root and reciprocal by a Householder step, fused
operations) is no further from the long-double value than the formulas written out, operation
for operation, as OpsF64 has them."""
import numpy as np
import pytest

from paper_2309_03717_gb300 import synth

LD = np.longdouble


def fma(a, b, c):
    return (LD(a) * LD(b) + LD(c)).astype(np.float64)


def approx(x, rng):
    """An approximation good to 20 bits, as the hardware's."""
    return (x * (1 + LD(2.0) ** -20 * rng.uniform(-1.0, 1.0, np.shape(x)))).astype(np.float64)


def rsqrt_f64(x, rng):
    y = approx(1 / np.sqrt(LD(x)), rng)
    e = fma(-(x * y), y, 1.0)
    return fma(fma(e, 0.375, 0.5), y * e, y)


def rcp_f64(x, rng):
    y = approx(1 / LD(x), rng)
    e = fma(-x, y, 1.0)
    return fma(y, fma(e, e, e), y)


def formulas(p, a, b, E, med, T):
    """The deposit's vector V/(D R), every operation in T."""
    p, a, b = ([T(v) for v in x] for x in (p, a, b))
    d = [a[k] - p[k] for k in range(3)]
    R = np.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
    inv = T(1) / R
    rh = [x * inv for x in d]
    n = T(1) + T(med["N0"]) * T(E) if "N0" in med else T(med["n"])
    c = b[0] * rh[0] + b[1] * rh[1] + b[2] * rh[2]
    D = T(1) - n * c
    s = T(1) / (D * R)
    return [s * (c * rh[k] - b[k]) for k in range(3)], D


def plain(p, a, b, E, med, rng):
    d = [a[k] - p[k] for k in range(3)]
    S = fma(d[2], d[2], fma(d[1], d[1], d[0] * d[0]))
    iR = rsqrt_f64(S, rng)
    rh = [x * iR for x in d]
    c = fma(b[2], rh[2], fma(b[1], rh[1], b[0] * rh[0]))
    n = fma(med["N0"], E, 1.0) if "N0" in med else np.full_like(c, med["n"])
    D = fma(-n, c, 1.0)
    s = iR * rcp_f64(D, rng)
    return [s * fma(c, rh[k], -b[k]) for k in range(3)], D


@pytest.mark.parametrize("zenith", [0.0, 50.0])
@pytest.mark.parametrize("medium", [synth.AIR_EXPONENTIAL, {"kind": "uniform", "n": 1.000292}])
def test_deposit_no_further_off_than_the_formulas(medium, zenith):
    n = 50_000
    t = {f: x.astype(np.float64) for f, x in synth.make_tracks(n, 31, zenith, dtype=np.float64).items()}
    rng = np.random.default_rng(2)
    old, new = [], []
    for ant in ([25.0, 0.0, 0.0], [150.0, 80.0, 0.0], [400.0, -300.0, 30.0]):
        for e in "01":
            p = [t[c + e] for c in "xyz"]
            b = [t["b" + c] for c in "xyz"]
            E = np.exp(-p[2] / medium["H"]) if "H" in medium else np.ones(n)
            exact, D = formulas(p, ant, b, E, medium, lambda v: np.asarray(v, LD))
            far = np.abs(D) >= 1e-3  # (the others take the midpoint)
            size = np.sqrt(sum(x * x for x in exact))
            for (got, _), out in ((formulas(p, ant, b, E, medium, lambda v: np.asarray(v, np.float64)), old),
                             (plain(p, ant, b, E, medium, rng), new)):
                out.append(np.sqrt(sum((LD(g) - x) ** 2 for g, x in zip(got, exact)))[far] / size[far])
    rms = [float(np.sqrt(np.mean(np.concatenate(v).astype(np.float64) ** 2))) for v in (old, new)]
    assert rms[1] <= rms[0], rms
