"""The vector kernel (a lane takes two or four nodes of a row) against the FP64
oracle on ragged grids: tiles of 32 rows, which no solver of any size runs one
node per thread for storages of 128-node tiles; FP64 tiles of 32 rows run one
node per thread alone, so the grouped step, always the vector kernel, is
compared there and everywhere."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as O
from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = {"periodic": (0, 0), "channel": (1, 2), "inlet-periodic": (1, 0), "periodic-slip": (0, 2)}
OBC_X = {0: O.BC_PERIODIC, 1: O.BC_INLET_OUTLET}
OBC_Y = {0: O.BC_PERIODIC, 2: O.BC_FREE_SLIP}


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


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("coll", ["srt", "mrt"])
@pytest.mark.parametrize("bc", list(BC))
@pytest.mark.parametrize("g", [(0.0, 0.0), (1e-6, -2e-6)])
def test_one_step(storage, coll, bc, g):
    """One step of a random state with solids and a rotating body: populations
    within one storage rounding step (FP64 1e-14 relative, FP32 4e-7, 16-bit
    one step of |h| <= 0.06 and FP32 arithmetic), the force within 1e-5
    relative (FP64 1e-11)."""
    import torch
    nx, ny = 301, 71
    chi, us = I.random_mask(nx, ny, 11, 0.15), I.random_solid_velocity(nx, ny, 12, 0.03)
    body = I.BodySpec(200.5, 38.0, 9.0, omega=0.002)
    bx, by = BC[bc]
    ocfg = O.Config(nx=nx, ny=ny, collision=O.SRT if coll == "srt" else O.MRT, tau=0.62, bc_x=OBC_X[bx], bc_y=OBC_Y[by],
                    u_in=(0.04, 0.0), g=g, chi=chi, us=us, bodies=[O.Body(body.cx, body.cy, body.radius, omega=body.omega)])
    cfg = V.make_config(nx, ny, coll, storage, 0.62, bc=(bx, by), u_in=(0.04, 0.0), body_force=g, tile_rows=32,
                        ring_len=8, stream=torch.cuda.Stream())
    with V.Solver(cfg, [body]) as s:
        assert storage == "f64" or V.vplbm_step_kernel(s.h) == "fused_step_kernel"
        s.set_mask(chi, us)
        s.set_populations(I.random_populations(nx, ny, 13, 0.05))
        ref = s.populations()
        fx, fy, mass = O.run(ocfg, ref, 1)
        V.vplbm_group_step([s.h], [1])
        f, got = s.populations(), s.forces()
    tol = {"f64": 1e-14 * np.abs(ref).max(), "f32": 4e-7, "f16": 0.06 * 2.0 ** -10 + 1e-6,
           "bf16": 0.06 * 2.0 ** -7 + 1e-6}[storage]
    assert np.abs(f - ref).max() < tol
    rel, small = (1e-11, 0.0) if storage == "f64" else (1e-5, 1e-6)
    assert got[0][0] == pytest.approx(fx[0], rel=rel, abs=small) and got[1][0] == pytest.approx(fy[0], rel=rel, abs=small)
    assert got[2][0] == pytest.approx(mass[0], rel=1e-14 if storage == "f64" else 1e-7)
