"""MRT with general rates (no two-rate structure): the moment-space collision,
whose every rounding is fixed, so that no kernel and no compilation of it gives
a node other bits, and its agreement with the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
XI = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
RATES = [0.3, 1.31, 0.77, 0.1, 1.7, 0.2, 0.9, 1.23, 1.57]
NX, NY, ETA = 300, 70, 1e-7


@pytest.fixture(scope="module", autouse=True)
def _lib():
    global V
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1812_05401_gb300 import build as B
    B.build()
    from paper_1812_05401_gb300 import vplbm
    V = vplbm
    yield


F = np.float32


def _mad(a, b, c):
    """FP32 a b + c, rounded once: the FP64 product is exact, the FP64 sum
    (Knuth's two-sum) is rounded to odd before the last rounding."""
    p, c = np.broadcast_arrays(np.float64(a) * np.float64(b), np.float64(c))
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    bits = np.ascontiguousarray(s).view(np.int64)
    odd = np.where((err != 0) & (bits % 2 == 0), bits + np.where((err > 0) == (s > 0), 1, -1), bits)
    return np.where(s == 0, s, odd.view(np.float64)).astype(F)


def _mul(a, b):
    return (np.float64(a) * np.float64(b)).astype(F)


def _step_fp32(h, solid, us, g):
    """One periodic step of FP32 offsets h with the roundings of the printed
    moment-space operator as the library makes them."""
    h = [np.roll(h[a], (XI[a][1], XI[a][0]), (0, 1)) for a in range(9)]
    a_s, kap = (np.where(solid, F(v), F(0)) for v in (1 / (2 * ETA), (1 / ETA) / (1 + 0.5 / ETA)))
    usx, usy = (np.where(solid, u.astype(F), F(0)) for u in us)
    gx, gy = F(g[0]), F(g[1])
    drho = h[0] + (((h[1] + h[3]) + (h[2] + h[4])) + ((h[5] + h[7]) + (h[6] + h[8])))
    rho = F(1) + drho
    d57, d68 = h[5] - h[7], h[6] - h[8]
    half = F(0.5) * rho
    dx = _mad(-rho, usx, _mad(half, gx, (h[1] - h[3]) + (d57 - d68)))
    dy = _mad(-rho, usy, _mad(half, gy, (h[2] - h[4]) + (d57 + d68)))
    inv = (1 / np.float64(_mul(rho, F(1) + a_s))).astype(F)
    ux, uy = _mad(dx, inv, usx), _mad(dy, inv, usy)
    Fx, Fy = _mad(rho, gx, _mul(-kap, dx)), _mad(rho, gy, _mul(-kap, dy))

    s1, s2, s4, s6, s7, s8 = (F(RATES[i]) for i in (1, 2, 4, 6, 7, 8))
    c1, c2, c4, c6, c7, c8 = (F(1) - F(0.5) * s for s in (s1, s2, s4, s6, s7, s8))
    s14, s58 = (h[1] + h[2]) + (h[3] + h[4]), (h[5] + h[6]) + (h[7] + h[8])
    e = F(-4) * h[0] - s14 + F(2) * s58
    eps = F(4) * h[0] - F(2) * s14 + s58
    jx = (h[1] - h[3]) + (h[5] - h[6]) + (h[8] - h[7])
    qx = F(2) * (h[3] - h[1]) + (h[5] - h[6]) + (h[8] - h[7])
    jy = (h[2] - h[4]) + (h[5] + h[6]) - (h[7] + h[8])
    qy = F(2) * (h[4] - h[2]) + (h[5] + h[6]) - (h[7] + h[8])
    pxx, pxy = (h[1] - h[2]) + (h[3] - h[4]), (h[5] - h[6]) + (h[7] - h[8])
    uu, uF = _mad(ux, ux, _mul(uy, uy)), _mad(ux, Fx, _mul(uy, Fy))
    rho3, rux = _mul(F(3), rho), _mul(rho, ux)
    es = _mad(_mul(c1, F(6)), uF, _mad(-s1, e - _mad(rho3, uu, F(-2) * drho), e))
    epss = _mad(-_mul(c2, F(6)), uF, _mad(-s2, eps - _mad(-rho3, uu, drho), eps))
    qxs = _mad(-c4, Fx, _mad(-s4, qx + rux, qx))
    qys = _mad(-c6, Fy, _mad(-s6, _mad(rho, uy, qy), qy))
    pxxs = _mad(c7 * F(2), _mad(ux, Fx, -_mul(uy, Fy)),
                _mad(-s7, _mad(-rho, _mad(ux, ux, -_mul(uy, uy)), pxx), pxx))
    pxys = _mad(c8, _mad(ux, Fy, _mul(uy, Fx)), _mad(-s8, _mad(-rux, uy, pxy), pxy))
    a0, a1, a2 = _mul(drho, F(1 / 9)), _mul(es, F(1 / 36)), _mul(epss, F(1 / 36))
    a4, a6, a7, a8 = _mul(qxs, F(1 / 12)), _mul(qys, F(1 / 12)), pxxs * F(0.25), pxys * F(0.25)
    x14, x58 = _mad(jx + Fx, F(1 / 6), F(-2) * a4), _mad(jx + Fx, F(1 / 6), a4)
    y14, y58 = _mad(jy + Fy, F(1 / 6), F(-2) * a6), _mad(jy + Fy, F(1 / 6), a6)
    b14, b58 = a0 - a1 - F(2) * a2, a0 + F(2) * a1 + a2
    return np.stack([a0 - F(4) * a1 + F(4) * a2, b14 + x14 + a7, b14 + y14 - a7, b14 - x14 + a7, b14 - y14 - a7,
                     b58 + x58 + y58 + a8, b58 - x58 + y58 - a8, b58 - x58 - y58 + a8, b58 + x58 - y58 - a8])


def _solver(storage, g, streaming="ab", rows=0, stream=None, rounding="stochastic"):
    cfg = V.make_config(NX, NY, "mrt", storage, 0.62, eta=ETA, body_force=g, rates=RATES, ring_len=64,
                        streaming=streaming, tile_rows=rows, stream=stream, rounding=rounding)
    s = V.Solver(cfg)
    s.set_mask(I.random_mask(NX, NY, 3, 0.3), I.random_solid_velocity(NX, NY, 4, 0.03))
    s.set_populations(I.random_populations(NX, NY, 17, 0.05))
    return s


@pytest.mark.parametrize("g", [(0.0, 0.0), (1e-3, -7e-4)])
@pytest.mark.parametrize("streaming", ["ab", "aa"])
@pytest.mark.parametrize("rows", [8, 32])  # one node per thread; a vector of nodes
@pytest.mark.parametrize("grouped", [False, True])
def test_fp32_bits_of_every_kernel(g, streaming, rows, grouped):
    """Two steps (in place: a push and a local one), bit for bit."""
    import torch
    with _solver("f32", g, streaming, rows, torch.cuda.Stream()) as s:
        h = (s.populations() - W).astype(F)
        solid, us = s.mask() != 0, I.random_solid_velocity(NX, NY, 4, 0.03)
        for _ in range(2):
            if grouped:
                V.vplbm_group_step([s.h], [1])
            else:
                s.step(1)
            h = _step_fp32(h, solid, us, g)
            assert np.array_equal((s.populations() - W).astype(F), h)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("streaming", ["ab", "aa"])
@pytest.mark.parametrize("rows", [8, 32])
@pytest.mark.parametrize("g", [(0.0, 0.0), (1e-6, -2e-6)])
def test_kernels_agree_and_match_the_oracle(storage, streaming, rows, g):
    """Unequal rates, random solids, with and without a body force: alone and
    grouped bitwise alike over three steps; the first within the oracle's
    one-step bounds (FP64 1e-14 relative, FP32 4e-7, 16-bit one rounding step
    of |h| <= 0.06 beside it)."""
    import torch
    chi, us = I.random_mask(NX, NY, 3, 0.3), I.random_solid_velocity(NX, NY, 4, 0.03)
    ocfg = O.Config(nx=NX, ny=NY, collision=O.MRT, tau=0.62, g=g, chi=chi, us=us, rates=RATES)
    out = []
    for grouped in (False, True):
        with _solver(storage, g, streaming, rows, torch.cuda.Stream()) as s:
            got = []
            ref = s.populations()
            O.run(ocfg, ref, 1)
            for n in (1, 2):
                if grouped:
                    V.vplbm_group_step([s.h], [n])
                else:
                    s.step(n)
                got.append(s.populations())
            tol = {"f64": 1e-14 * np.abs(ref).max(), "f32": 4e-7, "f16": 0.06 * 2.0 ** -10 + 1e-6,
                   "bf16": 0.06 * 2.0 ** -7 + 1e-6}[storage]
            assert np.abs(got[0] - ref).max() < tol
            out.append([*got, *s.forces(), *s.moments()])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
