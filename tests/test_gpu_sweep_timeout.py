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


def test_a_wait_that_runs_out_fails_the_solve_that_ran_it_and_no_other():
    """One context's sweeps give up (limit 0, form 11): its solve reports
    IBM_E_TIMEOUT.  Contexts of every precision and a batch go on, and with the
    default limit the context itself solves as a new one does.  A batch one of
    whose cases has the limit 0 fails, its cases and other batches do not."""
    import numpy as np
    import torch
    from paper_2402_17337_gb300 import IBM_E_TIMEOUT, Batch, IbmError, Solver, build
    from paper_2402_17337_gb300 import workloads as W
    build.build()
    cfg = W.batch_small(1)[0]

    def solve(s, check=8):
        xf, yf = s.grid()
        b, vol = W.random_field((s.ny, s.nx), seed=1), np.outer(np.diff(yf), np.diff(xf))
        b = torch.tensor(b - (b * vol).sum() / vol.sum(), device="cuda")  # a compatible right-hand side
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        rc, n, res = s.poisson_solve(b.data_ptr(), x.data_ptr(), 1e-6, check, 20000)
        return (rc, n, res), x

    def fresh(precision):
        s = Solver.from_config(cfg, precision=precision)
        if precision == 1:
            s.set_sor_shape(38)
        return s

    others = [fresh(p) for p in (0, 1, 2)]
    want = [solve(s) for s in others]
    assert all(w[0][0] == 0 for w in want)
    late = fresh(1)
    B, Blate = Batch([fresh(1)]), Batch([fresh(1), fresh(1)])
    for b in (B, Blate):
        b.set_sor_shape(38)
    Blate.solvers[0].set_wait_limit(0.0)
    for _ in range(2):
        late.set_wait_limit(0.0)
        assert solve(late)[0][0] == IBM_E_TIMEOUT
        with pytest.raises(IbmError) as e:
            Blate.step(1)
        assert e.value.code == IBM_E_TIMEOUT
        for s, w in zip(others, want):
            got = solve(s)
            assert got[0][0] == 0 and (s.P.precision == 2 or got[0] == w[0]), (s.P.precision, got[0], w[0])
            assert s.P.precision == 2 or torch.equal(got[1], w[1])
        B.step(1)
        late.set_wait_limit(-1.0)
        got = solve(late)
        assert got[0] == want[1][0] and torch.equal(got[1], want[1][1])


def test_the_autotuner_leaves_out_shapes_that_do_not_run():
    """A shape whose launches give up has a short time and no result.  With the
    limit 0 all of form 11 does: the tuners of a context and of a batch take
    another form, and the solves that follow converge."""
    from paper_2402_17337_gb300 import Batch, Solver, build
    from paper_2402_17337_gb300 import workloads as W
    build.build()
    ss = [Solver.from_config(c, precision=1) for c in W.batch_small(3)]
    for s in ss:
        s.set_wait_limit(0.0)
    for s in ss[:2]:
        st = s.step(1)
        assert 3 <= s.profile()["sor_form"] <= 10 and st["div_max"] <= 1e-8
    B = Batch(ss)
    for st in B.step(1):
        assert st["div_max"] <= 1e-8
    assert 3 <= B.profile()["sor_form"] <= 10
