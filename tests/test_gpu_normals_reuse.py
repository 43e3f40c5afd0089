"""apic_node_normals keeps its sums clear between calls instead of clearing them
first: calls of growing, shrinking and failing meshes on one context each match
the FP64 oracle (FP32 within 1e-6, as in test_gpu_normals.py)."""
import numpy as np
import pytest

import oracle
from paper_2108_02259_gb300 import scenes

pytestmark = pytest.mark.gpu


def test_calls_on_one_context_leave_no_sums_behind():
    import torch

    from paper_2108_02259_gb300 import apic, build

    build.build()
    meshes = [scenes.box_lattice_surface(*d, 0.1) for d in ((3, 3, 3), (12, 11, 10), (2, 5, 1024), (4, 4, 4), (30, 9, 40))]
    with apic.Context(0) as ctx:
        for rep in range(2):
            for x, tri in meshes:
                X, T = torch.as_tensor(x, device="cuda"), torch.as_tensor(tri, device="cuda")
                got = apic.node_normals(ctx, X, T).cpu().double().numpy()
                assert np.abs(got - oracle.node_normals(x, tri)).max() <= 1e-6
                bad = T.clone()
                bad[-1, 1] = len(x)
                with pytest.raises(apic.ApicError, match="triangle index"):
                    apic.node_normals(ctx, X, bad)
                assert not apic.node_normals(ctx, X, T[:0]).any()
