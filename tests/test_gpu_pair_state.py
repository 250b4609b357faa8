"""Paired steps through changes of a solver's state between calls: everything
that the second mask of moving bodies, or the choice between pairs and single
steps, depends on. Each against single steps, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1812_05401_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NX, NY = 2801, 1701


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


def _bodies(x, amp=6.0):
    return [I.BodySpec(x, 0.5 * NY, 0.1 * NY, 0.0, amp, 400.0, 0.001, False)]


def _run(act, paired, allocator=None, rows=0, force=(0.0, 0.0), bc=(3, 2)):
    cfg = V.make_config(NX, NY, "mrt", "f32", 0.62, bc=bc, u_in=(0.04, 0.01) if bc[0] else (0.0, 0.0),
                        body_force=force, ring_len=256, allocator=allocator, tile_rows=rows)
    with V.Solver(cfg, _bodies(0.4 * NX)) as s:
        s.set_populations(I.random_populations(NX, NY, 17, 0.05))

        def step(n):
            for k in [n] if paired else [1] * n:
                s.step(k)

        extra = act(s, step) or []
        return [s.populations(), *s.forces(), *s.moments(), s.mask(), *extra]


def _same(act, **kw):
    for a, b in zip(_run(act, False, **kw), _run(act, True, **kw)):
        assert np.array_equal(a, b)


def _layer(seed, solid=0.05):
    return I.random_mask(NX, NY, seed, solid), I.random_solid_velocity(NX, NY, seed + 1, 0.02)


def test_static_layer_replaced_between_pairs():
    def act(s, step):
        step(5)
        s.set_mask(*_layer(3))
        step(4)
        s.set_mask(*_layer(7, 0.02))
        step(3)
    _same(act)


@pytest.mark.parametrize("rows", [16, 32])
def test_bodies_replaced_between_pairs(rows):
    def act(s, step):
        s.set_mask(*_layer(3))
        step(4)
        s.set_bodies(_bodies(0.6 * NX))
        step(3)
        s.set_bodies(_bodies(0.5 * NX, amp=0.0))  # at rest
        step(4)
        s.set_bodies(_bodies(0.3 * NX, amp=9.0))
        step(4)
    _same(act, rows=rows)


def test_state_restored_between_pairs():
    def act(s, step):
        s.set_mask(*_layer(3))
        step(3)
        state = V.vplbm_save_state(s.h)
        s.set_mask(*_layer(7, 0.02))
        step(6)
        V.vplbm_load_state(s.h, state)
        step(5)
    _same(act)


def test_single_and_grouped_steps_between_pairs():
    def act(s, step):
        step(4)
        s.step(1)
        V.vplbm_group_step([s.h], [3])
        step(6)
    _same(act)


def test_restart_between_pairs():
    def act(s, step):
        step(7)
        s.set_initial_velocity()
        step(4)
    _same(act)


def test_momentum_exchange_switched_between_pairs():
    def act(s, step):
        step(4)
        s.record_momentum_exchange(True)
        step(4)
        got = list(s.momentum_exchange_forces())
        s.record_momentum_exchange(False)
        step(4)
        return got
    _same(act)


@pytest.mark.parametrize("bc", [(0, 0), (1, 2), (3, 2)])
def test_body_force_through_solids(bc):
    """The porous flow: a body force, static solids with a velocity, bodies."""
    def act(s, step):
        s.set_mask(*_layer(3, 0.15))
        step(5)
    _same(act, force=(2e-6, -1e-6), bc=bc)


def test_refused_second_mask_steps_singly():
    import torch
    A = V.TorchAllocator()
    inner = A._do_alloc
    plane = NY * ((NX + 31) // 32 * 32)
    refused = []

    def alloc(nbytes, ctx):
        if refused and nbytes == plane:
            refused.append(nbytes)
            return None
        return inner(nbytes, ctx)

    A._alloc = V.DEV_ALLOC_FN(alloc)

    def act(s, step):
        refused.append(0)  # from here on
        n0 = s.launches
        step(6)
        assert s.launches - n0 >= 6
        assert V.vplbm_step_kernel(s.h) == "fused_step_kernel"
    got = _run(act, True, allocator=A)
    assert len(refused) == 2  # asked for once
    for a, b in zip(got, _run(lambda s, step: step(6), True)):
        assert np.array_equal(a, b)
    torch.cuda.synchronize()
    assert A.live_bytes == 0


def test_timed_launches_count_their_steps():
    def act(s, step):
        V.vplbm_enable_timing(s.h, True)
        step(7)
        ms, n = V.vplbm_fused_timing(s.h)
        assert n == 7 and ms > 0
    _run(act, True)
