"""Node normals of triangles whose sums are exact (integer corners, one triangle
a node): FP64 normals are the sum times the rounded quotient 1 / sqrt(|s|^2), FP32
normals the nearest FP32 numbers, to a few parts in 10^8 of their last place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_normals_of_exact_sums():
    import torch

    from paper_2108_02259_gb300 import apic, build

    build.build()
    rng = np.random.default_rng(3)
    n = 30000
    x = rng.integers(-999, 1000, (n, 3)).astype(np.float64)
    tri = np.arange(n, dtype=np.int32).reshape(-1, 3)
    s = 0.5 * np.cross(x[1::3] - x[::3], x[2::3] - x[::3])
    s = np.repeat(s, 3, axis=0)
    len2 = (s * s).sum(1)
    assert len2.min() > 0
    want = s * (1.0 / np.sqrt(len2))[:, None]
    exact = (s.astype(np.longdouble) / np.sqrt(len2.astype(np.longdouble))[:, None]).astype(np.longdouble)
    d = lambda a: torch.as_tensor(a, device="cuda:0")  # noqa: E731
    with apic.Context(0) as ctx:
        for _ in range(2):
            got = apic.node_normals(ctx, d(x), d(tri), fp64=True).cpu().numpy()
            assert np.array_equal(got, want)
            got = apic.node_normals(ctx, d(x), d(tri)).cpu().numpy()
            ulp = np.spacing(np.abs(got)).astype(np.float64)
            assert (np.abs(got - exact.astype(np.float64)) <= ulp * (0.5 + 1e-7)).all()
