"""Two steps in one launch against single steps: a call of several steps takes
pairs (FP32, two-rate collision, larger grids), calls of one step do not, and
the two must give bitwise the same populations, records and moments."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BCS = {"periodic": (0, 0), "channel": (1, 2), "channel-convective": (3, 2),
       "inlet-periodic": (1, 0), "convective-periodic": (3, 0), "periodic-slip": (0, 2)}


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


def _compare(nx, ny, bc, calls, coll="mrt", force=(0.0, 0.0), moving=False, solid=0.05):
    chi, us = I.random_mask(nx, ny, 3, solid), I.random_solid_velocity(nx, ny, 4, 0.02)
    f0 = I.random_populations(nx, ny, 17, 0.05)
    out = []
    for paired in (False, True):
        cfg = V.make_config(nx, ny, coll, "f32", 0.62, bc=BCS[bc], u_in=(0.04, 0.01), body_force=force, ring_len=256)
        bodies = [I.BodySpec(0.4 * nx, 0.5 * ny, 0.1 * ny, 0.0, 6.0 * moving, 40.0 * moving, 0.001, False)]
        with V.Solver(cfg, bodies) as s:
            if solid:
                s.set_mask(chi, us)
            s.set_populations(f0)
            n0 = s.launches
            for n in calls:
                for k in [n] if paired else [1] * n:
                    s.step(k)
            if not moving:
                want = sum(n // 2 + n % 2 for n in calls) if paired else sum(calls)
                assert s.launches - n0 == want
            out.append([s.populations(), *s.forces(), *s.moments(), s.mask()])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


# tiles of 128 x 16: whole ones, one column or row over, one short, two columns
# of tiles, two rows of tiles
@pytest.mark.parametrize("nx,ny", [(4096, 1024), (2049, 2017), (4095, 1023), (129, 32002), (160001, 26)])
@pytest.mark.parametrize("bc", list(BCS))
def test_pair_equals_single_steps(nx, ny, bc):
    _compare(nx, ny, bc, (5, 2, 1))


@pytest.mark.parametrize("bc", ["channel-convective", "periodic"])
@pytest.mark.parametrize("coll,force", [("srt", (0.0, 0.0)), ("mrt", (1e-6, -2e-6))])
def test_pair_options(bc, coll, force):
    _compare(2801, 1701, bc, (66, 3), coll, force, solid=0.0)


@pytest.mark.parametrize("bc,solid", [("channel", 0.0), ("channel-convective", 0.02)])
def test_pair_moving_body(bc, solid):
    _compare(4000, 1100, bc, (9, 1, 4), moving=True, solid=solid)


def test_pair_tile_forms():
    """6144 x 2016: tiles of 32 rows, which a pair takes in two parts."""
    _compare(6144, 2016, "channel", (4,), solid=0.0)
