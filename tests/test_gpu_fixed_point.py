"""The FP64 3D sweep in integer arithmetic (k_sweep3_fix) against the oracle where its
tiles, its plane ring and its hand-over to FP64 instructions can go wrong."""
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


def _rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


# one tile holds 32 x 10 cells: one cell, exactly a tile, a tile and a remainder of one
# cell on either axis, one plane per block and long segments
# (with the norm; apply and smoothing of up to 12000 nodes take eight threads a node, (97, 41, 25) the tiles)
@pytest.mark.parametrize("n", [(2, 2, 2), (3, 2, 17), (33, 11, 2), (34, 12, 3), (33, 11, 15), (66, 12, 6), (9, 31, 33),
                               (97, 41, 25)])
def test_tile_edges(n):
    wk = random_workload(3, n, 90)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = wk.u0 + W.uniform(91, P.ndofs, -1e-2, 1e-2) * ~oracle.dirichlet_mask(P)
    psi = oracle.floor_psi(wk.psi, wk.psi_min)
    assert _rel(host(g.apply(g.finest, cuda(u))), oracle.apply(P, psi, u)) <= 1e-13
    r, nrm = g.residual(g.finest, cuda(wk.f), cuda(u))
    ref = oracle.residual(P, psi, wk.f, u)
    assert _rel(host(r), ref) <= 1e-13 and np.isclose(nrm, oracle.norm_free(P, ref), rtol=1e-13)
    got = host(g.smooth(g.finest, cuda(wk.f), cuda(u), "jacobi", 0.6))
    assert _rel(got - u, oracle.jacobi_sweep(P, psi, wk.f, u, 0.6) - u) <= 1e-12


@pytest.mark.parametrize("scale", [1e-200, 1e-130, 1e-100, 1.0, 1e140, 1e150])
def test_magnitudes(scale):
    """In and beyond the range of the integer form (2^-423 to 2^477)."""
    wk = random_workload(3, (35, 13, 12), 92)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = scale * W.uniform(93, P.ndofs, -1, 1)
    assert _rel(host(g.apply(g.finest, cuda(u))) / scale, oracle.apply(P, oracle.floor_psi(wk.psi, wk.psi_min), u) / scale) <= 1e-13


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e250, 1e-250])
@pytest.mark.parametrize("plane", [0, 9, 20])
def test_planes_that_do_not_fit(value, plane):
    """One node's value sends the rest of its block's planes to FP64 instructions: every
    other value is as before, and the neighbourhood of a NaN or infinity is not finite."""
    wk = random_workload(3, (35, 13, 21), 94)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = W.uniform(95, P.ndofs, -1, 1)
    v = u.reshape(3, 21, 13, 35)
    if value == 1e-250:
        v[:, plane] = 0.0
    v[1, plane, 6, 17] = value
    with np.errstate(invalid="ignore", over="ignore"):
        ref = oracle.apply(P, oracle.floor_psi(wk.psi, wk.psi_min), u)
    got = host(g.apply(g.finest, cuda(u)))
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(got))
    fin &= np.abs(ref) < 1e10
    assert fin.sum() > 20000 and np.abs(got - ref)[fin].max() <= 1e-12 * np.abs(ref[fin]).max()


def test_planes_of_different_size():
    """Each plane has its own unit: neighbouring planes nine decades apart."""
    wk = random_workload(3, (37, 13, 31), 96)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = W.uniform(97, P.ndofs, -1, 1).reshape(3, 31, 13, 37)
    u *= (10.0 ** np.array([0, -9, -3, 0, 6, 6, -2, 0, 0, 3] * 3 + [0]))[None, :, None, None]
    ref = oracle.apply(P, oracle.floor_psi(wk.psi, wk.psi_min), u.reshape(-1)).reshape(3, 31, -1)
    got = host(g.apply(g.finest, cuda(u.reshape(-1)))).reshape(3, 31, -1)
    big = np.abs(ref).max(axis=(0, 2))
    near = np.maximum(big, np.maximum(np.roll(big, 1), np.roll(big, -1)))
    assert np.all(np.abs(got - ref).max(axis=(0, 2)) <= 1e-13 * near)


def test_zero_psi_and_wide_psi():
    """Cells without force beside cells of full stiffness, psi over eight decades."""
    wk = random_workload(3, (35, 13, 11), 98, psi_lo=1e-8)
    wk.psi = 10.0 ** W.uniform(99, wk.ncells, -8, 0)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = W.uniform(100, P.ndofs, -1, 1)
    assert _rel(host(g.apply(g.finest, cuda(u))), oracle.apply(P, oracle.floor_psi(wk.psi, 1e-8), u)) <= 1e-13
    assert np.all(host(g.apply(g.finest, cuda(np.repeat([0.3, -0.7, 1.1], P.nnodes)))) == 0.0)


# 2D: tiles of 32 x 8 or 32 x 4 cells (from 152 tiles on the taller ones), colour tiles of
# 16 or (from 304 tiles of 32 on) 32 nodes
@pytest.mark.parametrize("n", [(2, 2), (33, 5), (34, 6), (17, 16), (16, 33), (65, 49), (609, 521)])
def test_2d_tile_edges(n):
    wk = random_workload(2, n, 110)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = wk.u0 + W.uniform(111, P.ndofs, -1e-2, 1e-2) * ~oracle.dirichlet_mask(P)
    psi = oracle.floor_psi(wk.psi, wk.psi_min)
    assert _rel(host(g.apply(g.finest, cuda(u))), oracle.apply(P, psi, u)) <= 1e-13
    r, nrm = g.residual(g.finest, cuda(wk.f), cuda(u))
    ref = oracle.residual(P, psi, wk.f, u)
    assert _rel(host(r), ref) <= 1e-13 and np.isclose(nrm, oracle.norm_free(P, ref), rtol=1e-13)
    got = host(g.smooth(g.finest, cuda(wk.f), cuda(u), "jacobi", 0.6))
    assert _rel(got - u, oracle.jacobi_sweep(P, psi, wk.f, u, 0.6) - u) <= 1e-12
    for desc in (False, True):
        got = host(g.smooth(g.finest, cuda(wk.f), cuda(u), "gs", descending=desc))
        assert _rel(got - u, oracle.gs_sweep(P, psi, wk.f, u, desc) - u) <= 1e-11


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e250, 1e-250])
def test_2d_values_that_do_not_fit(value):
    wk = random_workload(2, (49, 33), 112)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u = W.uniform(113, P.ndofs, -1, 1)
    v = u.reshape(2, 33, 49)
    if value == 1e-250:
        v[:, 13:20, 20:27] = 0.0
    v[1, 16, 23] = value
    psi = oracle.floor_psi(wk.psi, wk.psi_min)
    with np.errstate(invalid="ignore", over="ignore"):
        pairs = [(oracle.apply(P, psi, u), host(g.apply(g.finest, cuda(u)))),
                 (oracle.gs_sweep(P, psi, wk.f, u), host(g.smooth(g.finest, cuda(wk.f), cuda(u), "gs")))]
    for ref, got in pairs:
        fin = np.isfinite(ref)
        assert np.array_equal(fin, np.isfinite(got))
        fin &= np.abs(ref) < 1e10
        assert fin.sum() > 3000 and np.abs((got - ref)[fin]).max() <= 1e-11 * np.abs(ref[fin]).max()


@pytest.mark.parametrize("dim,n", [(2, (65, 41)), (3, (17, 17, 21))])
def test_solve_after_a_new_psi(dim, n):
    """The FP64 Jacobi scaling kept per level follows the psi: solves on one grid with a
    first and a second psi equal solves on fresh grids."""
    wk, w2 = random_workload(dim, n, 114, moduli=W.iso_cubic(1.0, 0.2)), random_workload(dim, n, 115, moduli=W.iso_cubic(1.0, 0.2))
    g = gpu_grid(wk)
    for psi in (wk.psi, w2.psi, wk.psi):
        g.set_psi(cuda(psi), wk.psi_min)
        fresh = gpu_grid(wk)
        fresh.set_psi(cuda(psi), wk.psi_min)
        u, v = cuda(wk.u0), cuda(wk.u0)
        a, b = g.solve(u, omega=0.5), fresh.solve(v, omega=0.5)
        assert a.cycles == b.cycles and np.array_equal(host(u), host(v))


@pytest.mark.parametrize("dim,n", [(2, (41, 33)), (3, (19, 13, 11))])
def test_steps_on_overlapping_arrays(dim, n):
    """apply and residual read and write the caller's arrays in place of copies; an output
    that is one of the inputs gives the same values as one that is not."""
    import paper_2212_02362_gb300 as sbm
    wk = random_workload(dim, n, 120)
    g, P = gpu_grid(wk), oracle_problem(wk)
    u, f = cuda(W.uniform(121, P.ndofs, -1, 1)), cuda(wk.f)
    ref, (r, nrm) = g.apply(g.finest, u), g.residual(g.finest, f, u)
    import ctypes as C
    v = u.clone()
    assert sbm.lib().sbm_apply(g._h, g.finest, 0, v.data_ptr(), v.data_ptr()) == 0 and torch.equal(v, ref)
    for inout in (u.clone(), f.clone()):
        a, b = (f, inout) if torch.equal(inout, u) else (inout, u)
        norm = C.c_double()
        st = sbm.lib().sbm_residual(g._h, g.finest, 0, a.data_ptr(), b.data_ptr(), inout.data_ptr(), C.byref(norm))
        assert st == 0 and torch.equal(inout, r) and norm.value == nrm


@pytest.mark.parametrize("dim,n", [(2, (65, 33)), (3, (25, 9, 9))])
def test_decaying_field(dim, n):
    """A displacement that decays from one node over thirty decades: cells whose values
    are a unit or two of the integer form, of either sign."""
    wk = random_workload(dim, n, 130)
    g, P = gpu_grid(wk), oracle_problem(wk)
    psi = oracle.floor_psi(wk.psi, wk.psi_min)
    X = W.node_coords(dim, wk.n, wk.h)
    r2 = sum((X[a] - c) ** 2 for a, c in zip(range(dim), (0.9, 0.2, 0.2)))
    for rate in (20.0, 60.0, 85.0):
        u = np.concatenate([s * np.exp(-rate * r2) for s in (0.0, -1.0, 0.3)[:dim]])
        assert _rel(host(g.apply(g.finest, cuda(u))), oracle.apply(P, psi, u)) <= 1e-13
        if dim == 2:
            ref = oracle.gs_sweep(P, psi, wk.f, u)
            assert _rel(host(g.smooth(g.finest, cuda(wk.f), cuda(u), "gs")) - u, ref - u) <= 1e-11


def _residual(wk, psi, u):
    """Residual and norm without a hierarchy (any size, psi as given)."""
    import ctypes as C

    import paper_2212_02362_gb300 as sbm
    nx, ny, nz = wk.n
    nodal = np.zeros((nz, ny, nx))
    nodal[:max(nz - 1, 1), :ny - 1, :nx - 1] = psi.reshape(max(nz - 1, 1), ny - 1, nx - 1)
    psi_d, f_d, u_d = cuda(nodal.reshape(-1)), cuda(wk.f), cuda(u)
    r_d, norm = torch.full_like(u_d, float("nan")), C.c_double()
    st = sbm.lib().sbm_residual_noalloc(wk.dim, (C.c_int * 3)(*wk.n), wk.h, (C.c_double * 3)(*wk.moduli),
                                        (C.c_uint * 3)(*wk.dirichlet_bits()), psi_d.data_ptr(), f_d.data_ptr(),
                                        u_d.data_ptr(), r_d.data_ptr(), C.byref(norm), None)
    assert st == 0, sbm.lib().sbm_last_error(None)
    return host(r_d), norm.value


@pytest.mark.parametrize("n", [(321, 101, 5), (257, 91, 6), (193, 121, 7), (161, 111, 3)])
def test_blocks_of_several_tiles(n):
    """Shallow grids with more tiles than SMs: a block goes from the top of one tile to the
    bottom of the next, whose planes go into ring slots that the last step's copy (a plane
    above the grid: zeros) was issued for."""
    wk = random_workload(3, n, 140)
    P = oracle_problem(wk)
    u = W.uniform(141, P.ndofs, -1, 1)
    ref = oracle.residual(P, wk.psi, wk.f, u)
    for _ in range(5):
        r, nrm = _residual(wk, wk.psi, u)
        assert _rel(r, ref) <= 1e-13 and np.isclose(nrm, oracle.norm_free(P, ref), rtol=1e-13)


def _scale(P, psi, u, n):
    """(|K| |u|) of every dof: the sum over its cells of |psi K_e| |u|."""
    nx, ny, nz = n
    Ke = np.abs(oracle.element_matrix(P))
    v, out = np.abs(u).reshape(3, nz, ny, nx), np.zeros((3, nz, ny, nx))
    at = lambda a: (slice(a >> 2, nz - 1 + (a >> 2)), slice((a >> 1) & 1, ny - 1 + ((a >> 1) & 1)),
                    slice(a & 1, nx - 1 + (a & 1)))
    U = np.stack([v[(p,) + at(a)] for a in range(8) for p in range(3)])
    F = np.tensordot(Ke, U, axes=([1], [0])) * psi.reshape(nz - 1, ny - 1, nx - 1)
    for a in range(8):
        for p in range(3):
            out[(p,) + at(a)] += F[a * 3 + p]
    return out.reshape(-1)


# FP64 forms of the operator differ in a dof by their rounding: 24 terms a cell and 8 cells, each
# off by 2^-53 of its share of |K||u|, in either of the two
LOCAL = 2 * 32 * 2.0 ** -53


@pytest.mark.parametrize("field", ["x2", "x3", "x4", "x8", "decay", "spot", "checker", "halves", "tiny"])
def test_fields_of_many_sizes_in_a_tile(field):
    """Displacements that vary by many powers of two within a tile of the 3D sweep: every
    dof's error against its own |K||u|, and the same values wherever the tiles lie."""
    n = (75, 27, 23)
    wk = random_workload(3, n, 150, bits=(0, 0, 0))
    P = oracle_problem(wk)
    wk.f = np.zeros(P.ndofs)
    X = W.node_coords(3, wk.n, wk.h)
    x, y, z = (c / wk.h for c in X)
    w = {"x2": ((1 + x) / 75) ** 2, "x3": ((1 + x) / 75) ** 3, "x4": ((1 + x) / 75) ** 4, "x8": ((1 + x) / 75) ** 8,
         "decay": np.exp(-0.5 * x - 0.3 * y), "spot": np.exp(-0.1 * ((x - 40) ** 2 + (y - 13) ** 2 + (z - 11) ** 2)),
         "checker": np.where((x + y + z) % 2 > 0, 1.0, 1e-9), "halves": np.where(x > 20, 1.0, 1e-12),
         "tiny": np.where(y > 13, 1.0, 1e-140)}[field]
    u = np.tile(w, 3) * W.uniform(151, P.ndofs, 0.5, 1) * np.sign(W.uniform(152, P.ndofs, -1, 1))
    r, _ = _residual(wk, wk.psi, u)
    ref, scale = oracle.residual(P, wk.psi, wk.f, u), _scale(P, wk.psi, u, n)
    free = ~oracle.dirichlet_mask(P)
    assert free.sum() == P.ndofs
    assert (np.abs(r - ref) / scale).max() <= LOCAL


@pytest.mark.parametrize("dim,n", [(2, (49, 33)), (3, (35, 13, 29))])
def test_psi_of_negative_zero(dim, n):
    """psi as given may be a zero of either sign: no force."""
    wk = random_workload(dim, n, 160)
    u = W.uniform(161, dim * wk.nnodes, -1, 1)
    psi = wk.psi.copy()
    psi[::3] = 0.0
    neg = np.where(psi == 0.0, -0.0, psi)
    (r, nrm), (r0, nrm0) = _residual(wk, neg, u), _residual(wk, psi, u)
    assert np.array_equal(r, r0) and nrm == nrm0
    assert _rel(r, oracle.residual(oracle_problem(wk), psi, wk.f, u)) <= 1e-13
    r, _ = _residual(wk, 0.0 * psi * -1.0, u)
    free = ~oracle.dirichlet_mask(oracle_problem(wk))
    assert np.array_equal(r[free], wk.f[free])


def _check_local(wk, psi, u):
    """The residual dof by dof where it is finite, and its norm."""
    P = oracle_problem(wk)
    with np.errstate(invalid="ignore", over="ignore"):
        ref = oracle.residual(P, psi, wk.f, u)
        norm = oracle.norm_free(P, ref)
        scale = np.nan_to_num(_scale(P, np.abs(psi), np.abs(u), wk.n), posinf=np.inf)   # fixed dofs beside a NaN: exact
    r, nrm = _residual(wk, psi, u)
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(r))
    assert np.all(np.abs(r - ref)[fin] <= (LOCAL * scale + 2.0 ** -51 * np.abs(wk.f))[fin])
    assert np.isclose(nrm, norm, rtol=1e-13) if np.isfinite(norm) else not np.isfinite(nrm)


# the tiled sweep: 24 tiles of 32 x 10 cells, six or seven planes a block
TILED = (129, 61, 40)


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e250, 1e-250])
@pytest.mark.parametrize("plane", [0, 17, 39])
def test_tiled_values_that_do_not_fit(value, plane):
    """A cell that does not fit, at the bottom, inside and at the top of the blocks' ranges: the blocks
    that hold it finish with FP64 instructions, their partial norms in two parts."""
    wk = random_workload(3, TILED, 200)
    u = W.uniform(201, 3 * wk.nnodes, -1, 1)
    v = u.reshape(3, 40, 61, 129)
    if value == 1e-250:
        v[:, max(plane - 2, 0):plane + 3, 26:33, 60:68] = 0.0
    v[1, plane, 29, 64] = value                   # a corner of four tiles
    _check_local(wk, wk.psi, u)


@pytest.mark.parametrize("value", [-0.5, np.inf, np.nan, 1e-70, 1e70])
@pytest.mark.parametrize("layer", [0, 17, 38])
def test_tiled_psi_that_does_not_fit(value, layer):
    wk = random_workload(3, TILED, 202)
    psi = wk.psi.copy()
    psi.reshape(39, 60, 128)[layer, 29, 63] = value
    _check_local(wk, psi, W.uniform(203, 3 * wk.nnodes, -1, 1))


@pytest.mark.parametrize("moduli", [(1e70, 0.6e70, 0.5e70), (1e-70, 0.6e-70, 0.5e-70), (1.0, 0.0, 1e-3)])
def test_moduli_that_do_not_fit(moduli):
    for n in ((97, 41, 25), (65, 49, 1)):
        wk = random_workload(3 if n[2] > 1 else 2, n, 204, moduli=moduli)
        wk.f = moduli[0] * wk.f
        P, u = oracle_problem(wk), W.uniform(205, (3 if n[2] > 1 else 2) * wk.nnodes, -1, 1)
        if wk.dim == 3:
            _check_local(wk, wk.psi, u)
        else:
            r, nrm = _residual(wk, wk.psi, u)
            ref = oracle.residual(P, wk.psi, wk.f, u)
            assert _rel(r, ref) <= 1e-13 and np.isclose(nrm, oracle.norm_free(P, ref), rtol=1e-13)


def test_wide_psi_and_rigid_motion_on_tiles():
    """psi over eight decades, cells without force beside full ones; a translation gives none."""
    wk = random_workload(3, TILED, 206)
    psi = 10.0 ** W.uniform(207, wk.ncells, -8, 0)
    psi[::5] = 0.0
    _check_local(wk, psi, W.uniform(208, 3 * wk.nnodes, -1, 1))
    r, _ = _residual(wk, psi, np.repeat([0.3, -0.7, 1.1], wk.nnodes))
    free = ~oracle.dirichlet_mask(oracle_problem(wk))
    assert np.array_equal(r[free], wk.f[free])


@pytest.mark.parametrize("scale", [1e-150, 1e-120, 1.0, 1e140, 1e150])
def test_tiled_magnitudes(scale):
    wk = random_workload(3, (97, 41, 25), 210)
    wk.f = scale * wk.f
    P, u = oracle_problem(wk), scale * W.uniform(211, 3 * wk.nnodes, -1, 1)
    r, _ = _residual(wk, wk.psi, u)
    assert _rel(r / scale, oracle.residual(P, wk.psi, wk.f, u) / scale) <= 1e-13


def test_hand_over_with_fp32_output():
    """The residual of a mixed solve is written in FP32: a start with a value below the range of
    the integer form gives the iterates of one without."""
    wk = random_workload(3, (65, 33, 41), 212, moduli=W.iso_cubic(1.0, 0.2))
    g = gpu_grid(wk, precision="mixed")
    kw = dict(omega=0.5, tol=0.0, max_cycles=2, raise_on_fail=False)
    u = cuda(wk.u0)
    v = u.clone()
    v.view(3, 41, 33, 65)[1, 20, 16, 32] = 1e-140
    a, b = g.solve(u, **kw), g.solve(v, **kw)
    assert np.allclose(a.history, b.history, rtol=1e-6) and _rel(host(v), host(u)) <= 1e-6
