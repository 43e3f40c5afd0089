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


@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_a_particle_that_hangs_in_balance_stays(env, dt):
    """Each particle hangs on a spring of length 1 and rest length 0 whose force
    is fl(m g), from an anchor of its own a metre (ten cells) above."""
    rng = np.random.default_rng(2)
    g = 9.81
    m = rng.uniform(0.5, 2.0, 4000).astype(np.float32).astype(np.float64)
    m = m[(m * g) / m == g][:1000]
    assert len(m) == 1000
    i = np.arange(len(m))
    low = np.stack([i % 10 * 2.0, i // 100 * 4.0, i // 10 % 10 * 2.0], 1) + 0.5
    x = np.concatenate([low, low + [0.0, 1.0, 0.0]])
    springs = np.stack([i, i + len(m)], 1).astype(np.int32)
    av, _ = _accelerations(env, x, np.concatenate([m, m]), springs, np.zeros(len(m)), m * g, dt, gravity=(0.0, -g, 0.0))
    assert np.abs(av[:len(m)]).max() == 0.0
    assert np.abs(av[len(m):, 1] + 2 * g).max() <= (1e-4 if dt == np.float32 else 1e-10) * g


def test_a_subnormal_mass_falls(env):
    """f / m where 1 / m overflows.  The grid's sums of m = 1e-310 hold 2^-31 of it
    at the smallest weight, 1/16^3."""
    x = np.array([[0.05, 0.05, 0.05]]) + np.array([[0.0, 0, 0], [2.0, 0, 0]])
    av, _ = _accelerations(env, x, np.full(2, 1e-310), np.zeros((0, 2), np.int32), np.zeros(0), np.zeros(0), np.float64,
                           gravity=(0.0, -9.81, 0.0))
    assert np.abs(av - [0.0, -9.81, 0.0]).max() <= 1e-6
