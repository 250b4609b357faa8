"""One node per thread (small grids) against the vector kernel: a solver's own
steps take the first below a size, grouped steps always the second, and the two
must give bitwise the same populations, records and moments."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BCS = {"periodic": (0, 0), "channel": (1, 2), "channel-convective": (3, 2),
       "inlet-periodic": (1, 0), "convective-periodic": (3, 0), "periodic-slip": (0, 2)}
RATES = [0.0, 1.1, 1.3, 0.0, 1.2, 0.0, 1.25, 1.6, 1.5]


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


def _compare(nx, ny, storage, bc, steps, streaming="ab", coll="mrt", rates=None, force=(0.0, 0.0), tile_rows=0,
             rounding="stochastic", solid=0.1):
    import torch
    shared = torch.cuda.Stream()
    chi, us = I.random_mask(nx, ny, 3, solid), I.random_solid_velocity(nx, ny, 4, 0.02)
    out = []
    for grouped in (False, True):
        cfg = V.make_config(nx, ny, coll, storage, 0.62, bc=BCS[bc], u_in=(0.04, 0.01), body_force=force,
                            rates=rates, ring_len=64, tile_rows=tile_rows, rounding=rounding, streaming=streaming,
                            stream=shared)
        with V.Solver(cfg, [I.BodySpec(0.4 * nx, 0.5 * ny, 0.1 * ny, omega=0.001)]) as s:
            s.set_mask(chi, us)
            s.set_populations(I.random_populations(nx, ny, 17, 0.05))
            for n in steps:
                if grouped:
                    V.vplbm_group_step([s.h], [n])
                else:
                    s.step(n)
            out.append([s.populations(), *s.forces(), *s.moments(), np.array(s.momentum_exchange())])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f64"])
@pytest.mark.parametrize("streaming", ["ab", "aa"])
@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (5, 1), (1, 9), (127, 8), (129, 7), (130, 33), (645, 171)])
def test_nodewise_equals_vector_kernel(storage, streaming, bc, nx, ny):
    _compare(nx, ny, storage, bc, (3, 1), streaming, force=(1e-6, -2e-6) if nx == 130 else (0.0, 0.0))


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
@pytest.mark.parametrize("rows", [8, 16, 32])
@pytest.mark.parametrize("rates", [None, RATES])
def test_nodewise_tile_heights_and_rates(storage, rows, rates):
    """Taller tiles give a unit several rows (a block of several rows, or the
    vector kernel where the unit is too large); no solids beside the body."""
    _compare(400, 100, storage, "channel", (5,), rates=rates, tile_rows=rows, rounding="nearest", solid=0.0)
