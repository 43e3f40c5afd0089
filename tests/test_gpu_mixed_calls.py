"""Calls of different kinds on one context: what a context keeps from one call
(page-table boxes, captured launch sequences) must not reach the next call's
results.  References: the FP64 oracle, within test_gpu_parity.py's bounds."""
import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu

TOL = {np.float32: (1e-5, 1e-4), np.float64: (1e-11, 1e-11)}


@pytest.fixture(scope="module")
def apic():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    return apic


def _t(a, dt):
    import torch

    return torch.as_tensor(np.ascontiguousarray(a), device="cuda:0", dtype=dt)


def _dev(s, dt):
    import torch

    f, td = s.astype(dt), torch.float32 if dt == np.float32 else torch.float64
    return (_t(f.x, torch.float64), _t(f.v, td), _t(f.C, td), _t(f.m, td), _t(f.nrm, td), _t(f.body, torch.int32))


def _near(s, dt, v, C, ref):
    vs = np.abs(s.v).max()
    cs = max(np.linalg.norm(s.C.reshape(-1, 9), axis=1).max(), np.linalg.norm(ref[1].reshape(-1, 9), axis=1).max(),
             2 * vs / s.h)
    assert np.abs(v.cpu().double().numpy() - ref[0]).max() <= TOL[dt][0] * vs
    assert np.abs(C.cpu().double().numpy() - ref[1]).max() <= TOL[dt][1] * cs


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("order", ["nsnsnsnn", "ssnsnnss"])
def test_mass_normals_between_steps_on_the_same_particles(apic, order, dt):
    """n: apic_mass_normals, s: a step with its own normals, on the same arrays
    and so with the same sizes: each sequence is captured and replayed as its
    own."""
    import torch

    s = scenes.random_cloud(4000, n_bodies=5, seed=42, h=0.08, n_iter=2, origin=(-1.2, 0.4, 2.0))
    ref = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=s.n_bodies)
    X, V, Cc, M, NR, B = _dev(s, dt)
    with apic.Context(0) as one:
        nref = apic.mass_normals(one, X, M, B, s.h, n_bodies=s.n_bodies).cpu().double().numpy()
    with apic.Context(0) as ctx:
        ctx.set_variant(5)  # (the autotuner's variants differ in their largest item)
        for kind in order:
            if kind == "n":
                got = apic.mass_normals(ctx, X, M, B, s.h, n_bodies=s.n_bodies)
                torch.cuda.synchronize()
                # (near the threshold a sum's last bits decide: few particles)
                far = np.abs(got.cpu().double().numpy() - nref).max(axis=1) > TOL[dt][0]
                assert far.mean() <= 1e-3
            else:
                r = apic.contact_step(ctx, X, V, Cc, M, NR, B, s.h, s.mu, s.n_iter, n_bodies=s.n_bodies)
                torch.cuda.synchronize()
                _near(s, dt, r.v, r.C, ref)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("empty", [0, 1, 2])
def test_a_scene_that_was_empty_when_the_boxes_were_sized(apic, empty, dt):
    """A batch in which one scene gains its particles in a later call, with as
    many scenes: boxes are sized afresh for it."""
    import torch

    sc = [scenes.random_cloud(700 + 300 * i, n_bodies=2 + i, seed=i, h=0.1, n_iter=2, origin=(-3.0 * i, 1.0, 0.4))
          for i in range(3)]
    refs = [oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=s.n_bodies) for s in sc]
    args = [_dev(s, dt) for s in sc]
    none = tuple(a[:0] for a in args[empty])

    def batch(a):
        return [apic.BatchScene(*b, s.h, s.mu, n_bodies=s.n_bodies) for s, b in zip(sc, a)]

    with apic.Context(0) as ctx:
        for full in (False, False, True, True, True, False, True):
            b = batch(args if full else args[:empty] + [none] + args[empty + 1:])
            apic.contact_step_batched(ctx, b, 2)
            torch.cuda.synchronize()
            for i, s in enumerate(sc):
                if full or i != empty:
                    _near(s, dt, b[i].v_out, b[i].C_out, refs[i])


def test_mass_normals_take_no_part_in_tuning(apic):
    """apic_mass_normals runs one pass of the step's N + 2: its time must not
    choose the variant of the size class's steps."""
    import torch

    s = scenes.random_cloud(4000, n_bodies=5, seed=42, h=0.08, n_iter=2)
    X, _, _, M, _, B = _dev(s, np.float32)
    with apic.Context(0) as ctx:
        for _ in range(2 * len(apic.variants()) + 2):
            apic.mass_normals(ctx, X, M, B, s.h, n_bodies=s.n_bodies)
            torch.cuda.synchronize()
        assert ctx.variant(s.n) == (0, False) and ctx.tuning() == {}
