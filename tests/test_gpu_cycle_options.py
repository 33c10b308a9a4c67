"""V-cycle options that the default V(2,2) cycle does not reach: adaptive inner cycles that
stop after any number of sweeps."""
import numpy as np
import pytest

import oracle
import workloads as W
from _sbm import cuda, gpu_grid, host, oracle_problem, random_workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2212_02362_gb300 import build
    build.build()
    oracle.build()


def _sweeps(g, f, e, count, omega):
    for _ in range(count):
        e = g.smooth(g.finest, f, e, "jacobi", omega, fp32=True)
    return e


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("nu1,nu2", [(1, 1), (1, 2), (2, 1), (2, 2), (1, 0), (3, 2)])
@pytest.mark.parametrize("dim,n", [(2, (33, 49)), (3, (17, 25, 17)), (3, (33, 33, 41))])
def test_gate_that_closes_after_the_pre_smoothing(dim, n, nu1, nu2, use_graph):
    """The correction is what the gate's residual was taken of, on a grid whose buffers hold
    another solve: after the pre-smoothing of the first cycle, and of the second."""
    wk = random_workload(dim, n, 170, moduli=W.iso_cubic(1.0, 0.2))
    P, omega = oracle_problem(wk), 0.5
    g = gpu_grid(wk, precision="mixed")
    f, u0 = cuda(wk.f), cuda(wk.u0)
    zero = torch.zeros_like(u0)
    kw = dict(omega=omega, nu1=nu1, nu2=nu2, tol=0.0, max_cycles=1, use_graph=use_graph, raise_on_fail=False)

    def dirty():
        g.set_source(cuda(W.uniform(171, P.ndofs, -1e3, 1e3)))
        g.solve(zero.clone(), omega=omega, max_cycles=3, tol=0.0, raise_on_fail=False)
        g.set_source(f)

    def check(u, e):
        d = host(u) - wk.u0
        assert np.abs(d - host(e)).max() <= 1e-5 * np.abs(host(e)).max()

    r, _ = g.residual(g.finest, f, u0)
    dirty()
    u = u0.clone()
    info = g.solve(u, inner_cycles=4, inner_rtol=1e3, **kw)      # closes in the first cycle
    assert info.cycles == 1 and info.vcycles == 1
    check(u, _sweeps(g, r, zero, nu1, omega))
    dirty()
    u1 = u0.clone()
    g.solve(u1, inner_cycles=1, inner_rtol=0.0, **kw)            # one whole cycle
    e1 = cuda(host(u1) - wk.u0)
    for rtol in 0.9 ** np.arange(1, 60):
        dirty()
        u = u0.clone()
        info = g.solve(u, inner_cycles=4, inner_rtol=float(rtol), **kw)
        if info.vcycles == 2:
            break
    assert info.vcycles == 2
    check(u, _sweeps(g, r, e1, nu1, omega))
