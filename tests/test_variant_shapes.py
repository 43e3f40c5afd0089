"""The transfer kernel's variants exist in their own shapes with the PIC and
Sec. 2.3 options as without (the host stubs' names in the built library tell
which shapes were compiled), and each gives the oracle's PIC step."""
import re
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

TOL_V, TOL_C = 1e-5, 1e-4


@pytest.fixture(scope="module")
def apic():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    return apic


def test_every_variant_has_its_shape_with_the_options(apic):
    if shutil.which("nm") is None:
        pytest.skip("no nm to list the library's own names")
    names = subprocess.run(["nm", "-C", apic.LIB_PATH], capture_output=True, text=True, check=True).stdout
    shapes = {}  # (mode, options) -> {(CTAs per SM, threads, row weights, rows per lane, persistent)}
    for m in re.finditer(r"k_items<float, (\d+), (\d+), (\d+), (\w+), false, (\d+), (\w+), (\w+)>", names):
        mode, minb, threads, rowtab, rpl, persist, gen = m.groups()
        shapes.setdefault((int(mode), gen == "true"), set()).add((minb, threads, rowtab, rpl, persist))
    modes = {mode for mode, gen in shapes if gen}
    assert len(modes) == 5  # first, middle, last and only pass, and the mass pass
    for mode in modes:
        assert shapes[mode, True] == shapes[mode, False]
        assert len(shapes[mode, True]) == len(apic.variants())


@pytest.mark.gpu
def test_every_variant_gives_the_pic_step(apic):
    import torch

    s = scenes.random_cloud(6000, n_bodies=4, seed=17, h=0.05, n_iter=4)
    rv, rC, _ = oracle.contact_step(s.x, s.v, s.C, s.m, s.nrm, s.body, s.h, s.mu, s.n_iter, n_bodies=s.n_bodies,
                                    flags=oracle.FLAG_PIC)
    f = s.astype(np.float32)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")  # noqa: E731
    vs = np.abs(s.v).max()
    cs = max(np.linalg.norm(s.C.reshape(-1, 9), axis=1).max(), np.linalg.norm(rC.reshape(-1, 9), axis=1).max())
    with apic.Context(0) as ctx:
        for var in range(len(apic.variants())):
            ctx.set_variant(var)
            for _ in range(3):
                r = apic.contact_step(ctx, t(f.x), t(f.v), t(f.C), t(f.m), t(f.nrm), t(f.body), s.h, s.mu, s.n_iter,
                                      n_bodies=s.n_bodies, flags=apic.APIC_VARIANT_PIC)
                torch.cuda.synchronize()
                assert np.abs(r.v.cpu().double().numpy() - rv).max() <= TOL_V * vs
                assert np.abs(r.C.cpu().double().numpy() - rC).max() <= TOL_C * cs
