"""Per-step records (force, mass): the tile partials of a call's steps are
summed by one launch per window of 64 steps. Records must not depend on how
the steps were batched, on the ring's length or on the grouping, and several
chunks of tiles must add to the whole."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu


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


def _wake(storage, **kw):
    w = I.cylinder_channel(300, 75, 12.0, 0.05, 150.0, 0, xc=100.0, storage=storage, seed=7)
    return V.Solver.from_workload(w, **kw)


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
@pytest.mark.parametrize("calls", [(1,) * 66, (63, 2, 1), (64, 2), (65, 1), (66,)])
def test_records_do_not_depend_on_batching(storage, calls):
    with _wake(storage) as a, _wake(storage, ring_len=5) as b:
        parts = []
        for n in calls:
            a.step(n)
            parts.append(np.stack(a.forces()))
            assert parts[-1].shape[1] == n
        b.step(66)  # the ring keeps the latest five
        last = np.stack(b.forces())
        assert last.shape[1] == 5
        assert np.array_equal(np.concatenate(parts, axis=1)[:, -5:], last)
    with _wake(storage) as c:
        c.step(66)
        assert np.array_equal(np.stack(c.forces()), np.concatenate(parts, axis=1))


def test_grouped_windows_equal_alone():
    import torch
    shared = torch.cuda.Stream()
    steps = [130, 64, 65, 1, 0]
    with _wake("f32") as a:
        a.step(130)
        ref = np.stack(a.forces())
    group = [_wake("f32", stream=shared, ring_len=256) for _ in steps]
    try:
        V.vplbm_group_step([s.h for s in group], steps)
        for s, n in zip(group, steps):
            got = np.stack(s.forces())
            assert got.shape[1] == n and np.array_equal(got, ref[:, :n])
    finally:
        for s in group:
            s.close()


def test_several_chunks_of_tiles():
    """4128 x 520 in tiles of 8 rows: 33 x 65 = 2145 tiles, two chunks. The
    density of the uniform rest state is exact; the force of a body far from
    the first chunk's tiles equals that of 32-row tiles up to the order of the
    FP32 and FP64 sums (some 1e4 nodes: 1e-5)."""
    out = []
    for rows in (8, 32):
        cfg = V.make_config(4128, 520, "srt", "f32", 0.6, bc="channel", u_in=(0.04, 0.0), u0=(0.04, 0.0),
                            tile_rows=rows)
        with V.Solver(cfg, [I.BodySpec(3000.0, 480.0, 30.0)]) as s:
            s.step(3)
            out.append(np.stack(s.forces()))
    assert np.allclose(out[0], out[1], rtol=1e-5, atol=1e-5 * np.abs(out[1][0]).max())
    with V.Solver(V.make_config(4128, 520, "srt", "f32", 0.6, tile_rows=8)) as s:
        s.step(2)
        assert np.array_equal(s.forces()[2], [4128.0 * 520.0] * 2)
