"""Deterministic mode: what a node sum of a small scene still resolves.

The scene's unit is the largest power of two u with n B <= 2^62 u (n particles,
B the largest term): 2^-60 for two unit masses.  A node's weight above it must
not vanish, in the mass nor in the body mask, however the shared tile holds its
sums."""
import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2_weight", [-40, -53, -56, -58])
@pytest.mark.parametrize("flags", ["default", "deterministic"])
def test_a_node_of_small_weight_keeps_both_bodies(flags, log2_weight):
    """Two particles of two bodies at one place, offset t from the lower corner
    of their cell: the weight of the farthest of their 64 nodes is (t^2 / 4)^3."""
    import torch

    from paper_2108_02259_gb300 import apic, build

    build.build()
    t = 2.0 ** ((log2_weight / 3 + 2) / 2)
    x = np.full((2, 3), 5 + t)  # (h = 1: cell 5; t to the 2^-32 that the cell kernel keeps)
    v = np.array([[1.0, 0.5, -0.25], [-0.5, 0.25, 1.0]])
    nrm = np.array([[1.0, 0, 0], [-1.0, 0, 0]])
    s = scenes.Scene(x, v, np.zeros((2, 3, 3)), np.ones(2), nrm, np.arange(2, dtype=np.int32), 2, 1.0, 0.3, 1)
    rv, _, rst = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=2)
    assert rst["multibody_nodes"] == 64
    f = s.astype(np.float32)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    with apic.Context(0) as ctx:
        r = apic.contact_step(ctx, d(f.x), d(f.v), d(f.C), d(f.m), d(f.nrm), d(f.body), s.h, s.mu, s.n_iter, n_bodies=2,
                              flags=apic.APIC_DETERMINISTIC if flags == "deterministic" else 0, stats=True)
        torch.cuda.synchronize()
    assert r.stats["multibody_nodes"] == 64
    assert np.abs(r.v.cpu().double().numpy() - rv).max() <= 1e-5
