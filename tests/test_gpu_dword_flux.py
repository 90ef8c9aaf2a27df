"""The sums of products of csrc/dword.cuh (mul_add, dot2, dot2_add, dot3) and the
double-word face flux made of them (csrc/physics_dw.cuh) on the GPU against
60-digit arithmetic; tests/dword_flux_probe.cu evaluates them.

Sums, u = 2^-24: the high products and their sum are exact, every low-order term
passes at most six FP32 roundings of quantities of at most 4u of the sum of the
magnitudes of the terms (the low parts of up to three products and two sums, and
one renormalisation, which under cancellation loses no more): 24 u^2 of that sum.
A dropped or misplaced correction term gives errors near u, 2^24 / 24 times that.

Flux: 64 u^2 of the row's scale, the sum of the magnitudes of both sides'
convective fluxes and of the terms of the dissipation (chains of fewer than
twenty operations of at most 6.5 u^2, most on terms below the scale), and for the
central pressure term of the momentum rows
- in binary64 (the split sweeps, and all from P = 1 on): the conversion of the
  row's sum, which drops less than 2^-46 = 4 u^2 of it;
- in double-word (one-launch sweeps of P = 0 levels): the conversions (4 u^2
  each) of three summands, two products (6.5 u^2), two sums of one sign or below
  the scale (3 u^2) and the last sum: 64 u^2 of the term again.
Inputs: the vortex's, the cylinder's and a Mach number of 0.3, and states whose
gauge pressure is a million times the dynamic pressure, where the momentum rows
are the pressure term.
"""
import os
import shutil
import subprocess
from decimal import Decimal, localcontext
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U2 = Fraction(1, 2 ** 48)
HERE = os.path.dirname(os.path.abspath(__file__))
GAMMA = 1.4
#          Ma, speed, cut-off, gauge pressure, jumps
FLOWS = {"vortex": (0.005, 2.0 ** 0.5, 0.0, 0.3, 1e-3), "cylinder": (0.001, 1.0, 0.001, 0.3, 1e-5),
         "Ma 0.3": (0.3, 1.0, 0.0, 0.5, 0.1), "pressure": (1e-5, 1.0, 0.0, 1e6, 1e-3)}


def _inputs(flow, n=600):
    Ma, speed, _, gp, jump = FLOWS[flow]
    rng = np.random.default_rng(sorted(FLOWS).index(flow))
    T = speed ** 2 / (GAMMA * Ma ** 2)
    x = np.empty((n, 21))
    x[:, :6] = 10.0 ** rng.uniform(-6, 6, (n, 6)) * rng.choice([-1.0, 1.0], (n, 6))
    k = n // 3                                             # a b + c, a b + c d cancel
    x[:k, 2] = -x[:k, 0] * x[:k, 1] * (1 + 10.0 ** rng.uniform(-12, -2, k))
    x[k:2 * k, 3] = -x[k:2 * k, 0] * x[k:2 * k, 1] / x[k:2 * k, 2] * (1 + 10.0 ** rng.uniform(-12, -2, k))
    x[k:2 * k, 4] *= 1e-6
    sgn = rng.choice([-1.0, 1.0], n)
    x[:, 6] = gp * rng.uniform(0.1, 1.0, n) * sgn
    x[:, 7] = T * (1 + 0.1 * Ma ** 2 * rng.uniform(-1, 1, n))
    base = np.stack([jump * rng.uniform(-1, 1, n), speed * rng.uniform(0.3, 1.0, n) * rng.choice([-1.0, 1.0], n),
                     speed * rng.uniform(-0.5, 0.5, n), jump * rng.uniform(-1, 1, n)], axis=1)
    x[:, 8:12] = base
    x[:, 12:16] = base + jump * rng.uniform(-1, 1, (n, 4))
    th = rng.uniform(0, 2 * np.pi, n)
    x[:, 16], x[:, 17], x[:, 18] = np.cos(th), np.sin(th), 0.1 * 10.0 ** rng.uniform(-1, 1, n)
    x[:, 19:] = 0.0
    return x, T


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("dwflux") / "probe")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-o", out,
                    os.path.join(HERE, "dword_flux_probe.cu")], check=True)
    return out


def _run(exe, tmp_path, flow):
    x, T = _inputs(flow)
    with open(tmp_path / "in.bin", "wb") as f:
        f.write(np.int32(x.shape[0]).tobytes())
        f.write(np.array([GAMMA, FLOWS[flow][2], T], "<f8").tobytes())
        f.write(x.astype("<f8").tobytes())
    subprocess.run([exe, str(tmp_path / "in.bin"), str(tmp_path / "out.bin")], check=True)
    return x, T, np.fromfile(tmp_path / "out.bin", "<f4").reshape(x.shape[0], 18, 2)


def _val(w):
    return Fraction(float(w[0])) + Fraction(float(w[1]))


def _flux(row, T0, eps_min):
    """Convective flux with dissipation, its scale, and the pressure term (momentum rows), in Decimals."""
    D = lambda v: Decimal(float(v))
    g = D(GAMMA)
    Cp, gm1 = g / (g - 1), g - 1
    ref, sm, sp, (nx, ny, dS) = (D(row[6]), D(0), D(0), D(row[7])), row[8:12], row[12:16], map(D, row[16:19])
    qm = [ref[v] + D(sm[v]) for v in range(4)]
    qp = [ref[v] + D(sp[v]) for v in range(4)]
    h = dS / 2
    pc = (qm[0] + qp[0]) * h
    qm[0] += D(T0)
    qp[0] += D(T0)
    out, scale = [Decimal(0)] * 4, [Decimal(0)] * 4
    for q in (qm, qp):
        m = q[0] / q[3] * (q[1] * nx + q[2] * ny) * h
        H = Cp * q[3] + (q[1] ** 2 + q[2] ** 2) / 2
        # the mass flux is a sum of two products: its scale is that of the terms
        ma = abs(q[0] / q[3]) * (abs(q[1] * nx) + abs(q[2] * ny)) * h
        for v, f in enumerate((1, q[1], q[2], H)):
            out[v] += m * f
            scale[v] += abs(ma * f)
    dp, du, dv, dT = (b - a for a, b in zip(qm, qp))
    p, u, w, T = ((a + b) / 2 for a, b in zip(qm, qp))
    rho, c2, vv = p / T, g * T, u * u + w * w
    e2 = min(Decimal(1), max(D(eps_min) ** 2, vv / c2))
    un, dun = u * nx + w * ny, du * nx + dv * ny
    # |B| on (p, u_n) by its two eigenvalues; the T row through (B - u_n)^-1
    b = (1 - e2) * un
    c = ((b / 2) ** 2 + e2 * c2).sqrt()
    lp, lm = un - b / 2 + c, un - b / 2 - c
    a1 = (abs(lp) - abs(lm)) / (2 * c)
    a0 = abs(lp) - a1 * lp
    B = lambda x, y: (e2 * (un * x + rho * c2 * y), x / rho + un * y)
    zp, zu = (a0 * s + a1 * t for s, t in zip((dp, dun), B(dp, dun)))
    w0, w1 = rho * dun, (b * dun + dp / rho) / (e2 * c2)
    y0, y1 = ((a0 - abs(un)) * s + a1 * t for s, t in zip((w0, w1), B(w0, w1)))
    xT = -b / (rho * Cp) * y0 + e2 * gm1 * T * y1 + abs(un) * dT
    yp = zp / e2
    yT = (1 / e2 - 1) / (rho * Cp) * zp + xT
    drho = (yp - rho * yT) / T
    zn = zu - abs(un) * dun
    xu, xv = abs(un) * du + zn * nx, abs(un) * dv + zn * ny
    H = Cp * T + vv / 2
    diss = (drho, u * drho + rho * xu, w * drho + rho * xv, H * drho - yp + rho * (u * xu + w * xv + Cp * yT))
    mag = (abs(yp) + rho * abs(yT)) / T
    amp = (mag, abs(u) * mag + rho * (abs(un * du) + abs(zn)), abs(w) * mag + rho * (abs(un * dv) + abs(zn)),
           H * mag + abs(yp) + rho * (abs(u * xu) + abs(w * xv) + Cp * abs(yT)))
    for v in range(4):
        out[v] -= h * diss[v]
        scale[v] += h * amp[v]
    return [Fraction(v) for v in out], [Fraction(v) for v in scale], [Fraction(0), Fraction(pc * nx),
                                                                      Fraction(pc * ny), Fraction(0)]


@pytest.mark.parametrize("flow", list(FLOWS))
def test_sums_of_products_and_face_flux(exe, tmp_path, flow):
    x, T, words = _run(exe, tmp_path, flow)
    for i in range(x.shape[0]):
        a, b, c, d, e, f = (_val(words[i, j]) for j in range(6))
        for j, terms in ((6, (a * b, c)), (7, (a * b, c * d)), (8, (a * b, c * d, e)), (9, (a * b, c * d, e * f))):
            assert abs(_val(words[i, j]) - sum(terms)) <= 24 * U2 * sum(abs(t) for t in terms), (i, j)
    with localcontext() as ctx:
        ctx.prec = 60
        for i in range(x.shape[0]):
            conv, scale, press = _flux(x[i], T, FLOWS[flow][2])
            for v in range(4):
                exact = conv[v] + press[v]
                tail = 4 * U2 * abs(exact)
                assert abs(_val(words[i, 10 + v]) - exact) <= 64 * U2 * scale[v] + (tail if v in (1, 2) else 0), (i, v)
                assert abs(_val(words[i, 14 + v]) - exact) <= 64 * U2 * (scale[v] + abs(press[v])), (i, v)
