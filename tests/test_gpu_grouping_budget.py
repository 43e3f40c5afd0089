"""A context's budget and the tables of grouping by counting: whatever a context
that only sorts has room for is not refused because earlier steps counted."""
import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu

H = 0.05
SIDE = 21  # grid blocks a side between the two particles that span the box


@pytest.fixture(scope="module")
def apic():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    return apic


def _clusters(blocks, per, seed):
    """`per` particles of one body in each of the given grid blocks, and one in
    each corner block (so the page-table box does not depend on the blocks)."""
    rng = np.random.default_rng(seed)
    b = np.concatenate([np.repeat(blocks, per, axis=0), [[0, 0, 0], [SIDE - 1] * 3]])
    n = len(b)
    x = (b + rng.uniform(0.02, 0.98, (n, 3))) * 4 * H
    nrm = rng.normal(size=(n, 3))
    return scenes.Scene(x, rng.normal(size=(n, 3)), rng.normal(size=(n, 3, 3)), rng.uniform(0.5, 2.0, n),
                        nrm / np.linalg.norm(nrm, axis=1, keepdims=True), np.zeros(n, np.int32), 1, H, 0.3, 2)


def _grid(k, stride, start):
    r = np.arange(k)
    return start + stride * np.stack(np.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)


def _fits(apic, budget, *steps):
    import torch

    with apic.Context(0, hbm_budget_bytes=budget) as ctx:
        ctx.set_variant(5)
        out = []
        for s in steps:
            f = s.astype(np.float32)
            t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
            try:
                r = apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body), s.h, s.mu, s.n_iter,
                                      n_bodies=1, stats=True)
            except apic.ApicError as e:
                assert e.code == apic.APIC_ERR_OUT_OF_MEMORY
                return None
            torch.cuda.synchronize()
            out.append((r.v.cpu().double().numpy(), r.C.cpu().double().numpy()))
        assert ctx.scratch_bytes() <= budget
        return out


@pytest.mark.parametrize("pairs", ["as many pairs", "more pairs"])
def test_bodies_that_spread_inside_their_boxes(apic, pairs):
    """The grid of a later step is several times the first one's.  The budget is
    the least (to 0.5%) that a first step on the spread particles, which sorts,
    has room in."""
    per = 32
    close = _clusters(_grid(5, 1, 8), per, 1)
    wide = _clusters(_grid(5, 4, 2), per, 2)
    if pairs == "more pairs":  # (than the step before left room for: 125 and 2 and a quarter more and 256)
        wide = _clusters(_grid(10, 2, 1), per * 125 // 1000, 3)
    assert close.x.shape == wide.x.shape
    hi = 1 << 28
    assert _fits(apic, hi, wide)
    lo = 0
    while hi - lo > hi // 200:
        mid = (lo + hi) // 2
        if _fits(apic, mid, wide):
            hi = mid
        else:
            lo = mid
    ref = {id(s): oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=1)
           for s in (close, wide)}
    steps = [close, close, close, wide, wide, close, wide]
    got = _fits(apic, hi, *steps)
    assert got is not None
    for s, (v, C) in zip(steps, got):
        rv, rC, _ = ref[id(s)]
        vs = np.abs(s.v).max()
        cs = max(np.linalg.norm(s.C.reshape(-1, 9), axis=1).max(), np.linalg.norm(rC.reshape(-1, 9), axis=1).max(),
                 2 * vs / s.h)
        assert np.abs(v - rv).max() <= 1e-5 * vs and np.abs(C - rC).max() <= 1e-4 * cs


def test_other_calls_find_the_room_that_counting_tables_held(apic):
    """A call that needs scratch of its own on a context that has counted."""
    import torch

    s = _clusters(_grid(5, 4, 2), 32, 4)
    f = s.astype(np.float32)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    x = torch.zeros(100, 3, dtype=torch.float64, device="cuda:0")
    tri = torch.zeros(0, 3, dtype=torch.int32, device="cuda:0")

    def steps(ctx, k):
        for _ in range(k):
            apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body), s.h, s.mu, s.n_iter, n_bodies=1)
        torch.cuda.synchronize()

    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        steps(ctx, 1)
        sorted_only = ctx.scratch_bytes()
        steps(ctx, 2)
        counted = ctx.scratch_bytes()
    assert counted > sorted_only
    with apic.Context(0, hbm_budget_bytes=counted) as ctx:
        ctx.set_variant(5)
        steps(ctx, 3)
        # (what is left of the budget holds 100 nodes, not ten thousand: the tables make way)
        big = torch.zeros((counted - sorted_only) // 48, 3, dtype=torch.float64, device="cuda:0")
        for q in (x, big):
            nrm = apic.node_normals(ctx, q, tri)
            torch.cuda.synchronize()
            assert float(nrm.abs().max()) == 0.0
        steps(ctx, 3)
        assert ctx.scratch_bytes() <= counted
