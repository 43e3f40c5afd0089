"""Which way a step finds its work items, told by the context's count of sorts:
the first step sorts, steps that reuse its boxes count, refused sizings sort again,
the deterministic mode always sorts.  And counting with 64-bit keys."""
import numpy as np
import pytest

from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def apic():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    return apic


def _sorts(apic, ctx, s, flags=0):
    """Sorts of one step on the scene."""
    import torch

    f = s.astype(np.float32)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    before = ctx.profile()["sort_launches"]
    apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body), s.h, s.mu, s.n_iter,
                      n_bodies=s.n_bodies, flags=flags)
    torch.cuda.synchronize()
    return ctx.profile()["sort_launches"] - before


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("cloud", [dict(n=40, n_bodies=2), dict(n=9000, n_bodies=2, spread=0.3),
                                   dict(n=20_000, n_bodies=32, origin=(-1.7, -0.4, -3.1), h=0.07),
                                   dict(n=(1 << 20) + 77, n_bodies=3, h=0.02, n_iter=1)])
def test_steps_that_reuse_their_boxes_count(apic, cloud, graphs):
    s = scenes.random_cloud(seed=5, **cloud)
    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        ctx.set_graphs(graphs)
        assert [_sorts(apic, ctx, s) for _ in range(4)] == [1, 0, 0, 0]
        assert _sorts(apic, ctx, s, apic.APIC_DETERMINISTIC) == 1
        assert _sorts(apic, ctx, s) == 0


@pytest.mark.parametrize("graphs", [False, True])
def test_more_pairs_than_room_and_a_box_left_sort_again(apic, graphs):
    wide = scenes.random_cloud(6000, n_bodies=4, seed=3, h=0.02, n_iter=2)
    clumps = scenes.random_cloud(6000, n_bodies=4, seed=4, h=0.02, n_iter=2, spread=0.05)
    clumps.x[::2] += 0.95
    # (both spread clouds have over 3,300 pairs, so a quarter more and 256 are over
    # 4,096 and over a quarter of the particles: such steps go on sorting, and where
    # a box is left they sort twice, in the refused sizing and in the fresh one)
    away = scenes.random_cloud(6000, n_bodies=4, seed=4, h=0.02, n_iter=2, origin=(7.0, 0.0, 0.0))
    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        ctx.set_graphs(graphs)
        got = [_sorts(apic, ctx, s) for s in (clumps, clumps, clumps, wide, wide, wide, away, away)]
    assert got == [1, 0, 0, 1, 1, 1, 2, 1]


def test_counting_with_64_bit_keys(apic):
    """20 M particles in a box of more than 2^26 (page, body) pairs, 17 of one of
    32 bodies in each occupied block: the first step, by sorting, against the
    counted ones, within twice the FP32 bounds (v 1e-5, C 1e-4)."""
    import torch

    per, side, h = 17, 128, 1.0
    k = 20_000_000 // per
    g = torch.Generator(device="cuda").manual_seed(5)
    r = lambda *sh: torch.rand(*sh, generator=g, device="cuda")  # noqa: E731
    b = torch.randperm(side ** 3 - 2, generator=g, device="cuda")[:k - 2] + 1
    b = torch.cat([b, torch.tensor([0, side ** 3 - 1], device="cuda")])  # (the corners, for the box)
    blk = torch.stack([b // side ** 2, b // side % side, b % side], 1).double()
    n = k * per
    X = (blk.repeat_interleave(per, 0) + r(n, 3).double() * 0.999) * (4 * h)
    B = torch.randint(0, 32, (k,), generator=g, device="cuda", dtype=torch.int32).repeat_interleave(per)
    V, Cc, M, N = r(n, 3) - 0.5, r(n, 3, 3) - 0.5, 0.5 + r(n), torch.zeros(n, 3, device="cuda")
    assert 64 * 32 * (side + 6) ** 3 > 2 ** 32 and 32 * (side + 6) ** 3 <= 4 * n
    vo, Co = torch.empty_like(V), torch.empty_like(Cc)
    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        for i in range(4):
            apic.contact_step(ctx, X, V, Cc, M, N, B, h, 0.3, 1, n_bodies=32, v_out=vo, C_out=Co)
            torch.cuda.synchronize()
            if i == 0:
                v0, C0 = vo.clone(), Co.clone()
            assert float((vo - v0).abs().max()) <= 2e-5 * 0.5
            assert float((Co - C0).abs().max()) <= 2e-4 * float(C0.flatten(1).norm(dim=1).max())
            vo.zero_(), Co.zero_()
        assert ctx.profile()["sort_launches"] == 1
