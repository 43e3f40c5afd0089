"""The active grid blocks of a step are those that some stencil reaches, however
the step finds its work items: counted here from the positions."""
import numpy as np
import pytest

from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu


def _reached(s):
    cell = np.floor(s.x / s.h).astype(np.int64)
    blocks = set()
    for d in np.stack(np.meshgrid([-1, 2], [-1, 2], [-1, 2], indexing="ij"), -1).reshape(-1, 3):
        blocks.update(map(tuple, (cell + d) >> 2))  # (a 4-node stencil spans at most two blocks an axis: its corners)
    return len(blocks)


CLOUDS = {
    "one": dict(n=1, n_bodies=1),
    "two thousand in a few blocks": dict(n=2000, n_bodies=2, spread=0.2),
    "32 bodies, negative": dict(n=20_000, n_bodies=32, origin=(-1.7, -0.4, -3.1), h=0.07),
    "sparse": dict(n=3000, n_bodies=3, spread=6.0),
    "a surface's worth": dict(n=30_000, n_bodies=1, h=0.013),
}


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("name", list(CLOUDS))
def test_active_blocks_are_the_reached_ones(name, dt):
    import torch

    from paper_2108_02259_gb300 import apic, build

    build.build()
    s = scenes.random_cloud(seed=5, **CLOUDS[name])
    want = _reached(s)
    f = s.astype(dt)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    with apic.Context(0) as ctx:
        ctx.set_variant(5)
        for flags in (0, 0, 0, 0, apic.APIC_DETERMINISTIC if dt == np.float32 else 0):
            r = apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body), s.h, s.mu, s.n_iter,
                                  n_bodies=s.n_bodies, flags=flags, stats=True)
            torch.cuda.synchronize()
            assert r.stats["active_blocks"] == want
