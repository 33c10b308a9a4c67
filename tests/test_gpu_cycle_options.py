"""V-cycle options that the default V(2,2) cycle does not reach: adaptive inner cycles that
stop after any number of sweeps, other counts of sweeps on levels of every kind (fused
small ones, per-node, tiled), and cycles whose arithmetic is all FP64 instructions."""
import numpy as np
import pytest

import oracle
import workloads as W
import test_gpu_amr as amr
from _amr import dense_solve
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


COUNTS = [(0, 1), (1, 0), (0, 2), (2, 0), (1, 1), (1, 2), (2, 1), (3, 2), (1, 3)]
# 2D: fused levels only, and unfused ones above them; 3D: per-node levels and a tiled one
GRIDS = [(2, (33, 49)), (2, (161, 193)), (3, (17, 25, 17)), (3, (33, 33, 25))]


def _err(u, ref, u0):
    return np.abs(u - ref).max() / np.abs(ref - u0).max()


@pytest.mark.parametrize("nu1,nu2", COUNTS)
@pytest.mark.parametrize("dim,n", GRIDS)
def test_sweep_counts(dim, n, nu1, nu2):
    """Two cycles from the boundary data, as the oracle's."""
    wk = random_workload(dim, n, 180, moduli=W.iso_cubic(1.0, 0.2))
    P, psi = oracle_problem(wk), oracle.floor_psi(wk.psi, wk.psi_min)
    for smoother in ("jacobi", "gs"):
        kw = dict(nu1=nu1, nu2=nu2, omega=0.5, smoother=smoother, tol=0.0, max_cycles=2)
        ref = oracle.mg_solve(P, psi, wk.f, wk.u0, **kw)
        for precision, tol in (("fp64", 1e-11), ("mixed", 1e-4)):
            g = gpu_grid(wk, precision=precision)
            u = cuda(wk.u0)
            info = g.solve(u, raise_on_fail=False, **kw)
            assert _err(host(u), ref.u, wk.u0) <= tol, (smoother, precision)
            assert np.allclose(info.history, ref.history[:3], rtol=1e-9 if precision == "fp64" else 1e-3)


@pytest.mark.parametrize("nu1,nu2", [(0, 2), (1, 1), (1, 2), (2, 1), (3, 0)])
@pytest.mark.parametrize("case", ["2d_multibox", "3d_two_slabs"])
@pytest.mark.parametrize("precision,inner", [("fp64", 1), ("mixed", 1), ("mixed", 4)])
def test_sweep_counts_on_patches(case, precision, inner, nu1, nu2):
    wk = amr.SMALL[case]()
    A, psis = amr._oracle(wk)
    us0 = [np.ascontiguousarray(wk.level_u0(a)) for a in range(A.nlev)]
    ref = dense_solve(A, psis, amr._zeros_f(A), us0)
    for smoother in ("jacobi", wk.smoother):
        g = amr._gpu(wk, precision)
        us = [cuda(u) for u in us0]
        g.amr_solve(us, tol=1e-10, omega=wk.omega, smoother=smoother, nu1=nu1, nu2=nu2, inner_cycles=inner)
        num = np.sqrt(sum(((host(us[a]) - ref[a]) ** 2).sum() for a in range(A.nlev)))
        assert num <= 1e-8 * np.sqrt(sum((r ** 2).sum() for r in ref))


@pytest.mark.parametrize("smoother", ["jacobi", "gs"])
@pytest.mark.parametrize("dim,n", GRIDS)
def test_cycles_in_fp64_instructions(dim, n, smoother):
    """Moduli beyond the integer form's range: every kernel of the cycle takes its FP64 branch, and
    with the load scaled alike the iterates are those of moderate moduli."""
    wk = random_workload(dim, n, 190, moduli=W.iso_cubic(1.0, 0.2))
    kw = dict(omega=0.5, smoother=smoother, tol=0.0, max_cycles=3, raise_on_fail=False)
    g = gpu_grid(wk)
    u = cuda(wk.u0)
    info = g.solve(u, **kw)
    wk.moduli, wk.f = tuple(1e70 * m for m in wk.moduli), 1e70 * wk.f
    g = gpu_grid(wk)
    v = cuda(wk.u0)
    big = g.solve(v, **kw)
    assert _err(host(v), host(u), wk.u0) <= 1e-12
    assert np.allclose(big.history, info.history, rtol=1e-9)
