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
