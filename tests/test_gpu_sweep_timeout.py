"""Form 11's wait for a tile's copies running out: with a limit of 0 every CTA
gives up on copies that are still in flight, waits for them to land, and ends
normally; the call reports IBM_E_TIMEOUT and the device goes on working."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ALONE = """
import torch
from paper_2402_17337_gb300 import IBM_E_TIMEOUT, Batch, IbmError, Solver, build, workloads as W
build.build()
cfgs = W.batch_small(3)
for shape in range(37, 43):
    s = Solver.from_config(cfgs[0], precision=1)
    s.set_sor_shape(shape)
    s.set_wait_limit(0.0)
    b = torch.tensor(W.random_field((s.ny, s.nx), seed=1), device="cuda")
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    rc, _, _ = s.poisson_solve(b.data_ptr(), x.data_ptr(), 1e-8, 8, 4000)
    assert rc == IBM_E_TIMEOUT, (shape, rc)
    s.close()
ss = [Solver.from_config(c, precision=1) for c in cfgs]
ss[1].set_wait_limit(0.0)
B = Batch(ss)
for shape in range(37, 43):
    B.set_sor_shape(shape)
    try:
        B.step(1)
        raise SystemExit("no error")
    except IbmError as e:
        assert "gave up" in str(e), e
x = torch.arange(1 << 20, device="cuda", dtype=torch.float64)
assert float(x.sum()) == (1 << 19) * float((1 << 20) - 1)
print("ended normally")
"""


def test_copies_in_flight_are_waited_for():
    out = subprocess.run([sys.executable, "-c", ALONE], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert out.returncode == 0 and "ended normally" in out.stdout, (out.stdout, out.stderr)
