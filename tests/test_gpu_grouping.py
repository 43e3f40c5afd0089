"""The two ways from keys to work items agree: a context's first step sorts,
the steps that reuse its page-table boxes count (group.cu).

Outputs of both against the FP64 oracle within the FP32 bounds of
test_gpu_parity.py (v 1e-5 of max|v|, C 1e-4 of the C scale), or, beyond the
oracle's reach in time, against each other within twice those bounds; the
counts of items and multi-body nodes are equal.  The blocks that stencils reach
are told per run of one body in one block when counting, and per 32 sorted
particles of such a run after the sort, so counting may flag a few more.
"""
import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu

TOL_V, TOL_C = 1e-5, 1e-4


@pytest.fixture(scope="module")
def apic():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    return apic


def _step(apic, ctx, s, dtype=np.float32, body=None, **kw):
    import torch

    f = s.astype(dtype)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    r = apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body if body is None else body), s.h, s.mu,
                          s.n_iter, n_bodies=s.n_bodies, stats=True, **kw)
    torch.cuda.synchronize()
    return r.v.cpu().double().numpy(), r.C.cpu().double().numpy(), r.stats


def _scales(s, C):
    return np.abs(s.v).max(), max(np.linalg.norm(s.C.reshape(-1, 9), axis=1).max(),
                                  np.linalg.norm(C.reshape(-1, 9), axis=1).max(), 2 * np.abs(s.v).max() / s.h)


def _near(s, got, ref, times=1.0):
    vs, cs = _scales(s, ref[1])
    assert np.abs(got[0] - ref[0]).max() <= times * TOL_V * vs
    assert np.abs(got[1] - ref[1]).max() <= times * TOL_C * cs


def _same_counts(counted, by_sort):
    for k in ("work_items", "multibody_nodes"):
        assert counted[k] == by_sort[k], k
    assert counted["active_blocks"] >= by_sort["active_blocks"]


CLOUDS = {
    "one": dict(n=1, n_bodies=1),
    "forty": dict(n=40, n_bodies=2),
    "a warp less one": dict(n=31, n_bodies=1, spread=0.3),
    "one full item and one particle": dict(n=129, n_bodies=1, spread=0.2),
    "runs of thousands": dict(n=9000, n_bodies=2, spread=0.3),
    "32 bodies, negative": dict(n=20_000, n_bodies=32, origin=(-1.7, -0.4, -3.1), h=0.07),
    "sparse": dict(n=3000, n_bodies=3, spread=6.0),
}


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_counted_step_matches_sorted_step_and_oracle(apic, name, dtype):
    s = scenes.random_cloud(seed=5, **CLOUDS[name])
    ref = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=s.n_bodies)
    with apic.Context(0) as ctx:
        ctx.set_variant(5)  # (the autotuner's variants differ in their largest item)
        got = [_step(apic, ctx, s, dtype) for _ in range(4)]  # sorted, counted, captured, replayed
    for g in got:
        _near(s, g, ref)
        _same_counts(g[2], got[0][2])


def test_ordered_counting_of_more_particles_than_l2_order_needs(apic):
    """Above 2^20 particles the counting kernels look back for their places."""
    s = scenes.random_cloud((1 << 20) + 77, n_bodies=3, seed=9, h=0.02, n_iter=1)
    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        first = _step(apic, ctx, s)
        for _ in range(3):
            g = _step(apic, ctx, s)
            _near(s, g, first, 2.0)
            _same_counts(g[2], first[2])


def test_more_pairs_than_the_step_before_left_room_for(apic):
    """Two clumps at the corners of a box, then the same particles spread over
    it: thousands of (block, body) pairs where a few were; then back."""
    wide = scenes.random_cloud(6000, n_bodies=4, seed=3, h=0.02, n_iter=2)
    clumps = scenes.random_cloud(6000, n_bodies=4, seed=4, h=0.02, n_iter=2, spread=0.05)
    clumps.x[::2] += 0.95
    with apic.Context(0) as ctx:
        for s in (clumps, clumps, wide, wide, clumps):
            ref = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=4)
            _near(s, _step(apic, ctx, s), ref)


def test_bad_particles_are_refused_in_a_step_that_reuses_its_boxes(apic):
    s = scenes.random_cloud(3000, n_bodies=3, seed=6)
    ref = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=3)
    bad = s.body.copy()
    bad[17], bad[99] = 3, 1 << 30
    with apic.Context(0) as ctx:
        for _ in range(2):
            _near(s, _step(apic, ctx, s), ref)
            _near(s, _step(apic, ctx, s), ref)
            with pytest.raises(apic.ApicError, match="body id out of range"):
                _step(apic, ctx, s, body=bad)


@pytest.mark.parametrize("slack", [1.0, 1.02, 1.1])
def test_a_budget_that_holds_a_sorted_step_holds_every_later_one(apic, slack):
    """A context whose budget is what its first step needs (scratch grows by a
    quarter more than asked while the budget allows) goes on without it."""
    s = scenes.random_cloud(20_000, n_bodies=3, seed=8, h=0.02, n_iter=2)
    ref = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=3)
    with apic.Context(0) as ctx:
        _near(s, _step(apic, ctx, s), ref)
        budget = int(ctx.scratch_bytes() * slack)
    with apic.Context(0, hbm_budget_bytes=budget) as ctx:
        ctx.set_variant(5)
        for _ in range(4):
            _near(s, _step(apic, ctx, s), ref)
        assert ctx.scratch_bytes() <= budget
