"""Augury dynamics at rest: where the forces cancel in exact arithmetic and in
correctly rounded FP64 arithmetic, the acceleration is exactly zero.

The positions are multiples of 1/8, so squared lengths are exact; numpy's square
root, product and quotient are correctly rounded, and so are the ones a step
needs (a spring at its rest length: sqrt(l2) - rest; a hanging particle:
f / m + g)."""
import numpy as np
import pytest

from paper_2108_02259_gb300 import scenes  # noqa: F401  (the package's tests import it first)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2108_02259_gb300 import apic, build

    build.build()
    c = apic.Context(0)
    yield apic, c, torch
    c.close()


def _accelerations(env, x, m, springs, rest, k, dt, gravity=(0.0, 0.0, 0.0), h=0.1):
    """(av, aC) of the initial acceleration from rest."""
    apic, ctx, torch = env
    n = len(x)
    td = torch.float64 if dt == np.float64 else torch.float32
    d = lambda a, ty: torch.as_tensor(np.ascontiguousarray(a), dtype=ty, device="cuda")  # noqa: E731
    z = lambda c: torch.zeros(n, c, dtype=td, device="cuda")  # noqa: E731
    av, aC = z(3), z(9)
    apic.augury_steps(ctx, d(x, torch.float64), z(3), z(9), av, aC, d(m, td), d(np.zeros(n), torch.int32),
                      d(springs, torch.int32), d(rest, torch.float64), d(k, torch.float64),
                      torch.zeros(0, 3, dtype=torch.int32, device="cuda"), h, 0.3, 1, 1e-3, 1e-3, 0, gravity=gravity,
                      n_bodies=1, init=True)
    torch.cuda.synchronize()
    return av.cpu().double().numpy(), aC.cpu().double().numpy()


@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_springs_at_their_rest_length_pull_nothing(env, dt):
    rng = np.random.default_rng(1)
    n = 3000
    x = rng.permutation(24 ** 3)[:n]
    x = np.stack([x // 576, x // 24 % 24, x % 24], 1) / 8.0
    springs = np.stack([rng.permutation(n), rng.permutation(n)], 1)
    springs = springs[springs[:, 0] != springs[:, 1]].astype(np.int32)
    rest = np.sqrt(((x[springs[:, 1]] - x[springs[:, 0]]) ** 2).sum(1))
    av, aC = _accelerations(env, x, np.ones(n), springs, rest, rng.uniform(10, 100, len(springs)), dt)
    assert np.abs(av).max() == 0.0 and np.abs(aC).max() == 0.0
