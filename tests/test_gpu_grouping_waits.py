"""A bounded wait of the grouping by counting that runs out (the bounds-checking
build, whose limits can be set): the call fails with a status, the kernels after
the wait touch nothing out of range, no result is written, and the next calls
are as ever.  In a child process, for the environment switch that selects the
library."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import torch
sys.path.insert(0, ROOT)
from paper_2108_02259_gb300 import apic, build
build.build(debug=True)
assert apic.load().apic_debug_build() == 1
n = (1 << 20) + 77  # (look-back from 2^20 particles on)
g = torch.Generator(device="cuda").manual_seed(3)
r = lambda *s: torch.rand(*s, generator=g, device="cuda")
X, V, Cc, M = r(n, 3).double(), r(n, 3) - 0.5, r(n, 3, 3) - 0.5, 0.5 + r(n)
B = (r(n) * 3).int()
N = torch.zeros(n, 3, device="cuda")
vo, Co = torch.empty(n, 3, device="cuda"), torch.empty(n, 3, 3, device="cuda")
def step(ctx):
    apic.contact_step(ctx, X, V, Cc, M, N, B, 0.02, 0.3, 1, n_bodies=3, v_out=vo, C_out=Co)
    torch.cuda.synchronize()
    return vo.clone(), Co.clone()
apic.debug_flags(clear=True)
with apic.Context(0) as ctx:
    ctx.set_variant(5)
    ctx.set_graphs(GRAPHS)
    first = step(ctx)
    for limits in (dict(pairs=-1), dict(items=-1), dict(pairs=-1, items=-1)):
        for _ in range(3):
            step(ctx)  # sizes afresh after a failed call; counts; replays
        apic.debug_wait_limit(**limits)
        vo.fill_(7.0); Co.fill_(7.0)
        try:
            step(ctx)
            raise SystemExit(f"no error with {limits}")
        except apic.ApicError as e:
            assert e.code == apic.APIC_ERR_TIMEOUT and "grouping" in str(e), e
        torch.cuda.synchronize()
        assert bool((vo == 7.0).all()) and bool((Co == 7.0).all())
        apic.debug_wait_limit()
    for _ in range(3):
        v, C = step(ctx)
        assert float((v - first[0]).abs().max()) <= 2e-5 * float(V.abs().max())
        assert float((C - first[1]).abs().max()) <= 2e-4 * max(float(first[1].abs().max()), float(V.abs().max()) / 0.01)
assert apic.debug_flags(clear=True) == 0
print("DONE")
"""


@pytest.mark.gpu
@pytest.mark.parametrize("graphs", [False, True])
def test_a_wait_that_runs_out_fails_the_call(graphs):
    env = dict(os.environ, APIC_DEBUG_BOUNDS="1")
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}; GRAPHS = {graphs}\n" + CHILD], env=env,
                       capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "DONE" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


def test_the_normal_build_has_no_wait_limit():
    from paper_2108_02259_gb300 import apic, build

    build.build()
    with pytest.raises(apic.ApicError, match="bounds-checking"):
        apic.debug_wait_limit(-1, -1)
