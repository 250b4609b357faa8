"""Steps inside CUDA graph capture: the step's launches are dependent launches
(programmatic), which a captured graph must keep in order."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
def test_captured_steps_equal_launched_steps(storage):
    """vplbm_step captured (its launches replayed once by the graph) against
    the same steps launched: populations and records bit for bit."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1812_05401_gb300 import vplbm as V
    w = I.cylinder_channel(700, 300, 24.0, 0.05, 150.0, 0, storage=storage, seed=5)
    st = torch.cuda.Stream()
    with V.Solver.from_workload(w) as a, V.Solver.from_workload(w, stream=st) as b:
        a.step(70)
        b.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            b.step(70)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(a.populations(), b.populations())
        for x, y in zip(a.forces(), b.forces()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("nx,ny,storage", [(4001, 1100, "f32"), (2100, 300, "f32"), (2100, 300, "bf16")])
@pytest.mark.parametrize("n", [2, 4, 6, 3])
def test_captured_steps_replay_from_their_own_result(nx, ny, storage, n):
    """A graph of an even number of steps, replayed, goes on from its own
    result (static body, nearest rounding: every step does the same): grids
    whose steps run in pairs and grids of the vector kernel. An odd number is
    replayed once."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1812_05401_gb300 import vplbm as V
    st = torch.cuda.Stream()
    out = []
    for graph in (False, True):
        cfg = V.make_config(nx, ny, "mrt", storage, 0.56, bc="channel-convective", u_in=(0.05, 0.0), ring_len=16,
                            rounding="nearest", stream=st)
        with V.Solver(cfg, [I.BodySpec(nx / 4, ny / 2, ny / 12)], perturbation=(0.05, 0.0, 1e-3, 3)) as s:
            s.synchronize()
            replays = 3 if n % 2 == 0 else 1
            if graph:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=st):
                    s.step(n)
                for _ in range(replays):
                    g.replay()
                torch.cuda.synchronize()
            else:
                s.step(n * replays)
            records = np.stack(s.forces())[:, -n:]
            out.append((s.populations(), records))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
