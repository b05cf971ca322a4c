"""How many bits the diagnostics sweep keeps: its terms against the oracle's in extended
precision (80 or 128 bits), on seeded FP32 states whose populations both sides share."""
import numpy as np
import pytest

from oracle import lbm_oracle as O
from paper_2101_04847_gb300 import lbm
from tests import inputs

pytestmark = pytest.mark.gpu

GRIDS = [(97, 60), (124, 48), (64, 90), (130, 71), (33, 120), (200, 40), (77, 77), (150, 33)]


def seeded_flow(seed, nx, ny, minority=0.08):
    """FP32 equilibrium populations of a tanh interface in a field of vortices with speeds up
    to 0.02."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:ny, 0:nx].astype(float)
    H = 0.5 * (1.0 + np.tanh((y - ny / 2 - 3.0 * np.sin(2 * np.pi * x / nx + rng.uniform(0, 6))) / 1.5))
    ux, uy = np.zeros_like(H), np.zeros_like(H)
    for kx, ky, a, p in zip(rng.integers(1, 4, 4), rng.integers(1, 4, 4), rng.uniform(-0.01, 0.01, 4), rng.uniform(0, 6, 4)):
        ux += a * np.cos(2 * np.pi * kx * x / nx + p) * np.cos(np.pi * ky * y / ny)
        uy += a * np.sin(2 * np.pi * kx * x / nx + p) * np.sin(np.pi * ky * y / ny)
    rho = (1.0 * (minority + (1 - minority) * H), 0.9 * (minority + (1 - minority) * (1 - H)))
    return np.stack([O.equilibrium(r, ux, uy) for r in rho]).astype(np.float32)


def extended_fields(f, p):
    """Densities and physical velocity (j + F / 2) / rho of FP32 populations, no wall forces,
    in extended precision (the oracle forms its forces in FP64)."""
    f = f.astype(np.longdouble)
    rho = f.sum(axis=1)
    j = [sum(int(O.C[i, k]) * (f[0, i] + f[1, i]) for i in range(9)) for k in range(2)]
    F = [0, 0]
    for s, sign in ((0, -1), (1, 1)):
        r = np.pad(rho[1 - s], ((1, 1), (0, 0)))
        for k in range(2):
            n = sum(int(O.C[i, k]) * np.longdouble((16, 4, 1)[abs(O.C[i]).sum()]) / 36
                    * np.roll(r[1 + O.C[i, 1]:1 + O.C[i, 1] + p.ny], -O.C[i, 0], axis=1) for i in range(9))
            F[k] = F[k] + rho[s] * (-np.longdouble(p.G) * n + (sign * np.longdouble(p.g) if k == 1 else 0))
    return rho[0], rho[1], (j[0] + F[0] / 2) / (rho[0] + rho[1]), (j[1] + F[1] / 2) / (rho[0] + rho[1])


@pytest.fixture(scope="module")
def samples(gpu):
    """(diagnostics, profile, the oracle's terms of the extended-precision fields, those of the
    extracted fields) of 32 states, the oracle's arithmetic in extended precision."""
    out = []
    for k in range(32):
        nx, ny = GRIDS[k % len(GRIDS)]
        d = inputs.params(inputs.C0, nx=nx, ny=ny, g=1e-4, crop_rows=5, G=(1.4, 1.2)[k % 2])
        f = seeded_flow(k, nx, ny)
        p = O.Params(**{q: v for q, v in d.items() if q in O.Params.__dataclass_fields__})
        with lbm.Solver(**d) as s:
            s.set_populations(f)
            got, rows, fld = s.diagnostics(), s.profile(), s.fields()
        fld = {q: fld[q].astype(np.longdouble) for q in ("rhoA", "rhoB", "ux", "uy")}
        out.append((got, rows, O.field_diagnostics(*extended_fields(f, p), p), O.field_diagnostics(*fld.values(), p)))
    return out


# The extracted fields carry the velocity as a double-float quotient rounds it.  A term taken
# from them in extended precision is off by that velocity's error alone; the sweep may add the
# roundings of its own products and sums, of either sign at 2^-48 each and averaged over
# thousands of sites: 2^-50 is allowed for them.  A quotient by a rounded reciprocal
# has 1.6 times the velocity error, and products without the low parts' own product
# make every square too small by 2^-50 to 2^-49.
@pytest.mark.parametrize("term", ["E_k", "enstrophy", "viscous", "flux_K", "flux_tau"])
def test_terms_are_as_accurate_as_the_fields(samples, term):
    def rms(k):
        return float(np.sqrt(np.mean([((s[k][term] - s[2][term]) / s[2][term]) ** 2 for s in samples])))

    assert rms(0) <= rms(3) + 2.0 ** -50, (rms(0), rms(3))


# A row's phi are added in double-float by 16 threads, 8 columns each, and in FP64 from
# there on.  The low part of a double-float sum S lies evenly within 2^-25 |S|, so its two
# roundings in an addition have a standard deviation of about 0.15 * 2^-48 |S|; over
# partial sums of 2 .. 8 values of size 1 that makes 2.2 * 2^-48 per thread, 8.8 * 2^-48
# over 16 threads and 2^-51.8 in the mean of a block's 124 columns.  With double-float
# partial sums of up to 124 values it is 2^-50.4.  Allowed: 2^-51 beside the error of the
# densities, which the extracted fields carry too.
def test_row_means_are_as_accurate_as_the_fields(gpu):
    errors = []
    for k in range(24):
        d = inputs.params(inputs.C0, nx=124, ny=64, g=1e-4, crop_rows=5, G=0.0, minority=0.0)
        f = seeded_flow(100 + k, 124, 64, minority=0.0)
        p = O.Params(**{q: v for q, v in d.items() if q in O.Params.__dataclass_fields__})
        with lbm.Solver(**d) as s:
            s.set_populations(f)
            s.diagnostics()
            rows, fld = s.profile(), s.fields()
        A, B = extended_fields(f, p)[:2]
        means = [np.mean((a - b)[5:-5], axis=1, dtype=np.longdouble)
                 for a, b in ((A, B), (fld["rhoA"].astype(np.longdouble), fld["rhoB"].astype(np.longdouble)))]
        errors.append((rows - means[0], means[1] - means[0]))
    sweep, fields = (float(np.sqrt(np.mean(np.square([e[q] for e in errors])))) for q in range(2))
    assert sweep <= fields + 2.0 ** -51, (sweep, fields)
