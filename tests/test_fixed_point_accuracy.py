"""Accuracy of the integer cell arithmetic (csrc/sbm_fix.cuh), compiled for the host: the
corner forces and the energy of single cells against long double, beside the same formula
in FP64, over the values, moduli and psi of the kernels.  An error counts against the
cell's largest |K||u|, and componentwise against that component's own."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2212_02362_gb300", "csrc")

SHIM = r"""
namespace sbm { inline long double madd(long double a, long double b, long double c) { return a * b + c; } }
#include "sbm_fix.cuh"
using namespace sbm;
typedef long double Q;
static Coef<Q> wide(const Coef<double> &c)
{
    Coef<Q> q;
    q.a11 = c.a11; q.a12 = c.a12; q.a44 = c.a44; q.ad = c.ad; q.b1 = c.b1; q.b12 = c.b12; q.b44 = c.b44; q.c2 = c.c2;
    return q;
}
static Coef<double> coef(int dim, const double *m) { return make_coef<double>(dim, 1.0 / 64, m[0], m[1], m[2]); }
template <int D, int N> static unsigned largest(const double (&v)[D][N])
{
    unsigned k = 0;
    for (auto &r : v)
        for (double x : r) k = fix::exp_key(x) > k ? fix::exp_key(x) : k;
    return k;
}
static int unit(unsigned key) { return (int)(key >> 20) > fix::kExpLo ? (int)(key >> 20) : fix::kExpLo; }

extern "C" int usable(int dim, const double *m) { return fix::level_consts(dim, coef(dim, m)).ok; }

// err: [way][corner dof] of the integer forms (0: by faces, 1: by corners) and of FP64 (2); scale:
// |K||u| of the dof; top: the largest |force| as an integer, over 2^61 (2D: the same)
extern "C" void errors3(const double *m, const double *uu, double psi, double *err, double *scale, double *top)
{
    const Coef<double> c = coef(3, m);
    const fix::Consts fc = fix::make_consts(3, c);
    double u[3][8], d[3][8];
    Q q[3][8];
    memcpy(u, uu, sizeof(u));
    memcpy(d, uu, sizeof(d));
    for (int i = 0; i < 24; ++i) q[i / 8][i % 8] = u[i / 8][i % 8];
    cell_forces3<double>(d, psi, c);
    cell_forces3<Q>(q, (Q)psi, wide(c));
    const int E = unit(largest(u));
    fix::i64 T[2][3][4], Fb[3][4], Ft[3][4], U[3][8], F[3];
    int e, ec, eu;
    for (int z = 0; z < 2; ++z)
        for (int p = 0; p < 3; ++p) {
            for (int k = 0; k < 4; ++k) T[z][p][k] = fix::to_fix(u[p][4 * z + k], E);
            bfly4xy(T[z][p]);
        }
    fix::cell_faces3(T[0], T[1], E, psi, fc, Fb, Ft, e);
    bool none;
    fix::transform_cell3(u, U, none, eu);
    *top = 0.0;
    for (int p = 0; p < 3; ++p) {
        bfly4xyT(Fb[p]);
        bfly4xyT(Ft[p]);
    }
    for (int i = 0; i < 24; ++i) {
        const int p = i / 8, a = i % 8;
        const fix::i64 f = a < 4 ? Fb[p][a] : Ft[p][a - 4];
        fix::corner_force3(U, none, eu, a, psi, fc, F, ec);
        *top = fmax(*top, ldexp(fmax(fabs((double)f), fabs((double)F[p])), -61));
        err[i] = (double)fabsl(fix::to_double(f, e) - q[p][a]);
        err[24 + i] = (double)fabsl(fix::to_double(F[p], ec) - q[p][a]);
        err[48 + i] = (double)fabsl(d[p][a] - q[p][a]);
    }
    for (int i = 0; i < 24; ++i) scale[i] = 0.0;
    for (int j = 0; j < 24; ++j) {
        double k[3][8] = {};
        k[j / 8][j % 8] = 1.0;
        cell_forces3<double>(k, psi, c);
        for (int i = 0; i < 24; ++i) scale[i] += fabs(k[i / 8][i % 8] * u[j / 8][j % 8]);
    }
}

extern "C" void errors2(const double *m, const double *uu, double psi, double *err, double *scale, double *top)
{
    const Coef<double> c = coef(2, m);
    const fix::Consts fc = fix::make_consts(2, c);
    double u[2][4], d[2][4];
    Q q[2][4];
    memcpy(u, uu, sizeof(u));
    memcpy(d, uu, sizeof(d));
    for (int i = 0; i < 8; ++i) q[i / 4][i % 4] = u[i / 4][i % 4];
    cell_forces2<double>(d, psi, c);
    cell_forces2<Q>(q, (Q)psi, wide(c));
    const int E = unit(largest(u));
    fix::i64 I[2][4], F[2][4], G[2];
    int e, eg;
    for (int i = 0; i < 8; ++i) I[i / 4][i % 4] = fix::to_fix(u[i / 4][i % 4], E);
    fix::cell_forces2(I, E, psi, fc, F, e);
    *top = 0.0;
    for (int i = 0; i < 8; ++i) {
        const int p = i / 4, a = i % 4;
        fix::corner_force2(I, a, E, psi, fc, G, eg);
        *top = fmax(*top, ldexp(fmax(fabs((double)F[p][a]), 2.0 * fabs((double)G[p])), -61));
        err[i] = (double)fabsl(fix::to_double(F[p][a], e) - q[p][a]);
        err[8 + i] = (double)fabsl(fix::to_double(G[p], eg) - q[p][a]);
        err[16 + i] = (double)fabsl(d[p][a] - q[p][a]);
    }
    for (int i = 0; i < 8; ++i) scale[i] = 0.0;
    for (int j = 0; j < 8; ++j) {
        double k[2][4] = {};
        k[j / 4][j % 4] = 1.0;
        cell_forces2<double>(k, psi, c);
        for (int i = 0; i < 8; ++i) scale[i] += fabs(k[i / 4][i % 4] * u[j / 4][j % 4]);
    }
}

// The 3D forces by faces, each on its own unit as the tiled sweep stages it
extern "C" void errors_staged(const double *m, const double *uu, double psi, double *err)
{
    const Coef<double> c = coef(3, m);
    double u[3][8];
    Q q[3][8];
    memcpy(u, uu, sizeof(u));
    for (int i = 0; i < 24; ++i) q[i / 8][i % 8] = u[i / 8][i % 8];
    cell_forces3<Q>(q, (Q)psi, wide(c));
    fix::i64 T[2][3][4], Fb[3][4], Ft[3][4];
    int E[2], e;
    for (int z = 0; z < 2; ++z) {
        unsigned key = 0;
        for (int i = 0; i < 12; ++i) {
            const unsigned k = fix::exp_key(u[i / 4][4 * z + i % 4]);
            key = k > key ? k : key;
        }
        E[z] = fix::face_exp(key);
        for (int p = 0; p < 3; ++p) {
            for (int k = 0; k < 4; ++k) T[z][p][k] = fix::to_fix(u[p][4 * z + k], E[z]);
            bfly4xy(T[z][p]);
        }
    }
    fix::cell_faces3(T[0], E[0], T[1], E[1], psi, fix::make_consts(3, c), Fb, Ft, e);
    for (int p = 0; p < 3; ++p) {
        bfly4xyT(Fb[p]);
        bfly4xyT(Ft[p]);
        for (int a = 0; a < 4; ++a) {
            err[p * 8 + a] = (double)fabsl(fix::to_double(Fb[p][a], e) - q[p][a]);
            err[p * 8 + a + 4] = (double)fabsl(fix::to_double(Ft[p][a], e) - q[p][a + 4]);
        }
    }
}

// v^T S u: the errors of the integer form and of FP64, and |v|^T |S| |u|
extern "C" void errors_work(const double *m, const double *uu, const double *vv, double *err)
{
    const Coef<double> c = coef(3, m);
    double u[3][8], v[3][8], d[3][8];
    Q q[3][8], ref = 0;
    memcpy(u, uu, sizeof(u));
    memcpy(v, vv, sizeof(v));
    memcpy(d, uu, sizeof(d));
    for (int i = 0; i < 24; ++i) q[i / 8][i % 8] = u[i / 8][i % 8];
    cell_forces3<double>(d, 1.0, c);
    cell_forces3<Q>(q, (Q)1, wide(c));
    fix::i64 U[3][8], V[3][8];
    bool nu, nv;
    int eu, ev;
    fix::transform_cell3(u, U, nu, eu);
    fix::transform_cell3(v, V, nv, ev);
    double s = 0.0;
    err[2] = 0.0;
    for (int a = 0; a < 8; ++a)
        for (int p = 0; p < 3; ++p) {
            s += v[p][a] * d[p][a];
            ref += v[p][a] * q[p][a];
        }
    for (int j = 0; j < 24; ++j) {
        double k[3][8] = {};
        k[j / 8][j % 8] = 1.0;
        cell_forces3<double>(k, 1.0, c);
        for (int i = 0; i < 24; ++i) err[2] += fabs(v[i / 8][i % 8] * k[i / 8][i % 8] * u[j / 8][j % 8]);
    }
    err[0] = (double)fabsl((nu || nv ? 0.0 : fix::cell_work3(U, eu, V, ev, fix::make_consts(3, c))) - ref);
    err[1] = (double)fabsl(s - ref);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("acc")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def _p(a):
    return a.ctypes.data_as(C.POINTER(C.c_double))


def _errors(lib, dim, mod, u, psi):
    n = dim << dim
    mod, u, err, scale, top = np.array(mod, float), np.ascontiguousarray(u, float), np.zeros((3, n)), np.zeros(n), C.c_double()
    (lib.errors3 if dim == 3 else lib.errors2)(_p(mod), _p(u), C.c_double(psi), _p(err), _p(scale), C.byref(top))
    return err, scale, top.value


KINDS = ("random", "smooth", "stretch", "components", "hourglass")
MODULI = [(1.0, 0.6, 0.5), (1.2, 0.4, 0.4), (1.0, -0.3, 0.4), W.iso_cubic(1480.0, 0.22), W.iso_cubic(1.0, 0.4999)]


def _cells(kind, dim, count, seed):
    """(count, dim, 2^dim) nodal values."""
    nc = 1 << dim
    x = np.array([[(a >> m) & 1 for m in range(dim)] for a in range(nc)], float)
    r = W.uniform(seed, count * dim * nc, -1, 1).reshape(count, dim, nc)
    g = W.uniform(seed + 1, count * dim * (dim + 1), -1, 1).reshape(count, dim, dim + 1)
    if kind == "random":
        return r
    if kind == "smooth":                          # a linear displacement with a little noise
        return g[:, :, -1:] + 0.02 * np.einsum("cpm,am->cpa", g[:, :, :dim], x) + 1e-4 * r
    if kind == "stretch":
        return 1.0 + 1e-5 * r
    if kind == "components":                      # components decades apart
        return r * 10.0 ** (3.0 * W.uniform(seed + 2, count * dim, -1, 1)).reshape(count, dim, 1)
    sign = np.prod(2.0 * x - 1.0, axis=1)
    return sign * g[:, :, :1] + 1e-3 * r


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("mod", MODULI)
@pytest.mark.parametrize("kind", KINDS)
def test_forces_are_no_further_off_than_in_fp64(lib, dim, mod, kind):
    assert lib.usable(dim, _p(np.array(mod, float))) == 1
    count = 800
    psi = 10.0 ** W.uniform(301, count, -4, 0)
    whole, own = np.zeros((3, count)), np.zeros((3, count))
    for i, u in enumerate(_cells(kind, dim, count, 302)):
        err, scale, top = _errors(lib, dim, mod, u, psi[i])
        assert top <= 1.0
        whole[:, i], own[:, i] = err.max(axis=1) / scale.max(), (err / scale).max(axis=1)
    for e in (whole, own):
        rms = np.sqrt((e ** 2).mean(axis=1))
        assert rms[0] <= rms[2] and rms[1] <= rms[2], rms


@pytest.mark.parametrize("kind", KINDS)
def test_faces_on_units_of_their_own(lib, kind):
    """Cells staged face by face, every scale modulo the units' steps, the faces up to 2^70 apart."""
    count = 400
    mod = np.array(MODULI[0], float)
    psi = 10.0 ** W.uniform(341, count, -4, 0)
    for scale in (1.0, 2.0, 4.0, 8.0):
        for above in (0, 1, 2, 3, 4, 5, 7, 10, 30, 59, 60, 61, 70):
            for face in (0, 1):
                whole, own = np.zeros((2, count)), np.zeros((2, count))
                for i, u in enumerate(_cells(kind, 3, count, 342)):
                    u, err = scale * u, np.zeros(24)
                    u[:, 4 * face:4 * face + 4] *= 2.0 ** -above
                    lib.errors_staged(_p(mod), _p(u), C.c_double(psi[i]), _p(err))
                    ref, k, _ = _errors(lib, 3, mod, u, psi[i])
                    for j, e in enumerate((err, ref[2])):
                        whole[j, i], own[j, i] = e.max() / k.max(), (e / k).max()
                for e in (whole, own):
                    rms = np.sqrt((e ** 2).mean(axis=1))
                    assert rms[0] <= rms[1], (scale, above, face, rms)


@pytest.mark.parametrize("kind", KINDS)
def test_energies_are_no_further_off_than_in_fp64(lib, kind):
    count = 800
    for mod in MODULI:
        mod, e = np.array(mod, float), np.zeros((count, 3))
        for i, (u, v) in enumerate(zip(_cells(kind, 3, count, 310), _cells(kind, 3, count, 320))):
            u, v = np.ascontiguousarray(u), np.ascontiguousarray(v)
            lib.errors_work(_p(mod), _p(u), _p(v), _p(e[i]))
        rms = np.sqrt(((e[:, :2] / e[:, 2:]) ** 2).mean(axis=0))
        assert rms[0] <= rms[1], (mod, rms)


@pytest.mark.parametrize("dim", [2, 3])
def test_sums_stay_in_range(lib, dim):
    """Values and psi at the ends of their binades, in every pattern of signs along an axis and in
    random ones, moduli at the ends of what is positive definite: a corner force keeps below 2^61."""
    big = 2.0 - 2.0 ** -52
    nc = 1 << dim
    pats = [np.sign(W.uniform(330 + i, dim * nc, -1, 1)) for i in range(200)]
    for p in range(nc):
        s = np.array([(-1.0) ** bin(a & p).count("1") for a in range(nc)])
        pats += [np.tile(s, dim), np.concatenate([s * (-1.0) ** q for q in range(dim)])]
        pats += [np.concatenate([s if q == r else 0 * s for q in range(dim)]) for r in range(dim)]
    for mod in MODULI + [(1.0, 0.999, 1e-3), (1.0, 0.0, 1e-3), (1.0, -0.499, 1e-3), (1.0, -0.499, 5.0), (1.0, 0.999, 5.0)]:
        for s in pats:
            for psi in (1.0, big, 0.5 * big):
                err, scale, top = _errors(lib, dim, mod, big * s, psi)
                assert top <= 1.0
                assert err[:2].max() <= 8 * 2.0 ** -53 * scale.max()


@pytest.mark.parametrize("dim", [2, 3])
def test_weakly_coupled_moduli_take_fp64(lib, dim):
    """Forces along one axis far below those along another, whose bound sets the unit."""
    for mod, ok in (((1.0, 0.0, 0.5), 1), ((1.0, 0.5, 1e-3), 1), ((1.0, 0.0, 1e-3), 0), ((1.0, 1e-3, 1e-2), 0)):
        assert lib.usable(dim, _p(np.array(mod))) == ok
