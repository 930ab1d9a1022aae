"""FP64 sweeps kept on chip (k_sor64.cu) against the oracle: one cluster, tiles
over all SMs, and the sizes where a grid goes from one to the other; strips and
tiles of a few rows, odd sizes, sweep caps between two checks.  The kernels and
the oracle share their arithmetic, so sweep counts agree exactly; fields are
compared at 1e-13 of their largest value, above the rounding that 8 operations
an update could leave in 60 sweeps (8 x 60 x 1.1e-16)."""
import numpy as np
import pytest

import oracle
from paper_2402_17337_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (9, 200), (64, 15), (33, 16), (17, 17), (128, 93), (129, 95), (41, 300),
                                   (300, 41), (191, 129), (513, 257), (500, 500), (547, 548), (548, 549), (75, 100), (76, 100),
                                   (105, 100), (106, 100)])
@pytest.mark.parametrize("m,cap", [(8, 60), (3, 20), (1, 2), (7, 49)])
def test_sweeps_on_chip_match_oracle(nx, ny, m, cap):
    import torch
    from paper_2402_17337_gb300 import Solver, build
    build.build()
    kw = dict(x0=0.0, x1=2.0 + nx / ny, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    g, o = Solver(**kw), oracle.Sim(**kw)
    b = W.random_field((ny, nx), seed=nx + 3 * ny)
    b -= b.mean()
    phi0 = W.random_field((ny, nx), seed=5, scale=0.1)
    rc, phio, so, ro = o.poisson(b, phi0=phi0, tol=1e-300, check=m, maxs=cap)
    bd, pd = torch.tensor(b, device="cuda"), torch.tensor(phi0, device="cuda")
    torch.cuda.synchronize()
    rg, sg, rr = g.poisson_solve(bd.data_ptr(), pd.data_ptr(), 1e-300, m, cap)
    assert rc == rg == -3 and sg == cap // m * m
    assert abs(rr - ro) <= 1e-10 * ro
    assert np.abs(pd.cpu().numpy() - phio).max() <= 1e-13 * np.abs(phio).max()


def test_two_streams_and_threads_solve_at_once():
    """Cooperative launches of two contexts from two threads do not wait on each other for good."""
    import threading

    import torch
    from paper_2402_17337_gb300 import Solver, build
    build.build()
    nx, ny = 384, 200
    kw = dict(x0=0.0, x1=3.0, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    b = W.random_field((ny, nx), seed=1)
    b -= b.mean()
    out = {}

    def work(k):
        g = Solver(**kw)
        bd = torch.tensor(b, device="cuda")
        for _ in range(4):
            pd = torch.zeros_like(bd)
            torch.cuda.synchronize()
            rc = g.poisson_solve(bd.data_ptr(), pd.data_ptr(), 1e-300, 8, 400)
        out[k] = rc, pd.cpu().numpy()
        g.close()

    ts = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert all(out[k][0][0] == -3 and np.array_equal(out[k][1], out[0][1]) for k in range(3))


@pytest.mark.parametrize("nx,ny", [(105, 100), (106, 100), (131, 67), (384, 193), (547, 548), (548, 549)])
@pytest.mark.parametrize("m,cap", [(8, 60), (7, 49)])
def test_allocation_free_solve_repeats_the_context_bit_for_bit(nx, ny, m, cap):
    """Tiles in the static scratch, from the smallest grid that takes them to the first that does not; two calls,
    the second on buffers that hold the first one's exchanges."""
    import ctypes as C

    import torch
    import paper_2402_17337_gb300 as ibm
    from paper_2402_17337_gb300 import build
    build.build()
    g = ibm.Solver(x0=0.0, x1=2.0 + nx / ny, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    xf, yf = g.grid()
    fn, D = ibm.lib().ibm_poisson_solve_noalloc, C.POINTER(C.c_double)
    fn.argtypes = [C.c_int, C.c_int, D, D, C.c_void_p, C.c_void_p, C.c_double, C.c_double, C.c_int, C.c_int,
                   C.c_void_p, C.POINTER(C.c_int), C.POINTER(C.c_double)]
    for seed in (1, 2):
        bd = torch.tensor(W.random_field((ny, nx), seed=seed), device="cuda")
        p, q = torch.zeros_like(bd), torch.zeros_like(bd)
        torch.cuda.synchronize()
        rc, sg, rg = g.poisson_solve(bd.data_ptr(), p.data_ptr(), 1e-300, m, cap)
        sn, rn = C.c_int(-1), C.c_double(-1.0)
        assert fn(nx, ny, xf.ctypes.data_as(D), yf.ctypes.data_as(D), bd.data_ptr(), q.data_ptr(), g.P.omega_p, 1e-300,
                  m, cap, None, C.byref(sn), C.byref(rn)) == rc == -3
        assert sn.value == sg and rn.value == rg
        assert torch.equal(p, q)


@pytest.mark.parametrize("nx,ny", [(70, 45), (513, 257)])
@pytest.mark.parametrize("m,cap", [(3000, 20000), (65537, 131084)])
def test_launches_between_checks_do_not_change_the_iterates(nx, ny, m, cap):
    """A solve takes several launches whatever the interval between checks (here
    longer than a launch, and no multiple of one): the same iterates bit for
    bit as with a check every 8 sweeps, by the context and by the
    allocation-free call.  The relaxation factor is small, so the iterates
    still change at the end."""
    import ctypes as C

    import torch
    import paper_2402_17337_gb300 as ibm
    from paper_2402_17337_gb300 import build
    build.build()
    g = ibm.Solver(x0=0.0, x1=2.0 + nx / ny, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0, omega_p=0.05)
    xf, yf = g.grid()
    fn, D = ibm.lib().ibm_poisson_solve_noalloc, C.POINTER(C.c_double)
    fn.argtypes = [C.c_int, C.c_int, D, D, C.c_void_p, C.c_void_p, C.c_double, C.c_double, C.c_int, C.c_int,
                   C.c_void_p, C.POINTER(C.c_int), C.POINTER(C.c_double)]
    b = W.random_field((ny, nx), seed=1)
    b -= b.mean()
    bd = torch.tensor(b, device="cuda")
    out = []
    for every in (8, m):
        p = torch.zeros_like(bd)
        torch.cuda.synchronize()
        g.set_profiling(True)
        rc, sweeps, res = g.poisson_solve(bd.data_ptr(), p.data_ptr(), 1e-300, every, cap)
        assert (rc, sweeps) == (-3, cap // every * every)
        assert g.profile()["sweep_launches"] >= cap // 8192
        q = torch.zeros_like(bd)
        torch.cuda.synchronize()
        sn, rn = C.c_int(-1), C.c_double(-1.0)
        assert fn(nx, ny, xf.ctypes.data_as(D), yf.ctypes.data_as(D), bd.data_ptr(), q.data_ptr(), g.P.omega_p, 1e-300,
                  every, cap, None, C.byref(sn), C.byref(rn)) == rc
        assert (sn.value, rn.value) == (sweeps, res)
        assert torch.equal(p, q)
        out.append(p)
    assert torch.equal(*out)
    p = torch.zeros_like(bd)
    torch.cuda.synchronize()
    g.poisson_solve(bd.data_ptr(), p.data_ptr(), 1e-300, 8, cap - 8)
    assert not torch.equal(p, out[0])
    g.close()


@pytest.mark.parametrize("nx,ny,cap,launches", [(192, 96, 4096, 8), (192, 96, 4100, 9), (513, 257, 1500, 3),
                                                (70, 45, 4096, 1)])
def test_a_solve_on_every_SM_is_cut_into_short_launches(nx, ny, cap, launches):
    """Tiles hold every SM, so a launch of theirs ends after 512 sweeps and lets
    other streams' kernels in; a cluster leaves SMs free and goes on."""
    import torch
    from paper_2402_17337_gb300 import Solver, build
    build.build()
    g = Solver(x0=0.0, x1=2.0 + nx / ny, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    bd = torch.tensor(W.random_field((ny, nx), seed=1), device="cuda")
    p = torch.zeros_like(bd)
    torch.cuda.synchronize()
    g.set_profiling(True)
    rc, sweeps, _ = g.poisson_solve(bd.data_ptr(), p.data_ptr(), 1e-300, 8, cap)
    assert (rc, sweeps) == (-3, cap // 8 * 8)
    assert g.profile()["sweep_launches"] == launches
    g.close()


@pytest.mark.parametrize("nx,ny", [(192, 96), (513, 257)])
def test_a_wait_that_runs_out_ends_the_solve_and_leaves_the_context_usable(nx, ny):
    """With a limit of 0 a tile gives up at the first neighbour that has not
    posted yet: the kernel ends normally, the call reports IBM_E_TIMEOUT, and
    with the default limit the same context solves as a new one does."""
    import torch
    from paper_2402_17337_gb300 import IBM_E_TIMEOUT, Solver, build
    build.build()
    kw = dict(x0=0.0, x1=2.0 + nx / ny, y0=0.0, y1=1.5, nx=nx, ny=ny, hmin=0.0, dt=1.0)
    bd = torch.tensor(W.random_field((ny, nx), seed=1), device="cuda")

    def solve(g):
        p = torch.zeros_like(bd)
        torch.cuda.synchronize()
        return g.poisson_solve(bd.data_ptr(), p.data_ptr(), 1e-300, 8, 400), p

    g, fresh = Solver(**kw), Solver(**kw)
    want = solve(fresh)
    for _ in range(3):
        g.set_wait_limit(0.0)
        assert solve(g)[0][0] == IBM_E_TIMEOUT
        g.set_wait_limit(-1.0)
        got = solve(g)
        assert got[0] == want[0] and torch.equal(got[1], want[1])
    g.close()
    fresh.close()
