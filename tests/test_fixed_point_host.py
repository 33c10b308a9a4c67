"""The integer cell arithmetic of the FP64 3D sweep (csrc/sbm_fix.cuh), compiled for the
host: the corner forces of single cells against the oracle's cell matrix, over the
magnitudes and moduli the kernel takes."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2212_02362_gb300", "csrc")

SHIM = r"""
#include "sbm_fix.cuh"
using namespace sbm;
extern "C" int cell3(double h, const double *mod, const double *u, double psi, double *F)
{
    const fix::Consts fc = fix::make_consts(3, make_coef<double>(3, h, mod[0], mod[1], mod[2]));
    if (!fc.ok || !fix::psi_ok(psi)) return 1;
    unsigned key[2] = {0, 0};
    for (int p = 0; p < 3; ++p)
        for (int b = 0; b < 8; ++b) {
            const unsigned k = fix::exp_key(u[p * 8 + b]);
            if (k > key[b / 4]) key[b / 4] = k;
        }
    int E[2];
    for (int z = 0; z < 2; ++z) {
        if (!fix::key_ok(key[z])) return 1;
        E[z] = (int)(key[z] >> 20) > fix::kExpLo ? (int)(key[z] >> 20) : fix::kExpLo;
    }
    const int Em = E[0] > E[1] ? E[0] : E[1];
    fix::i64 T[2][3][4], Fb[3][4], Ft[3][4];
    int e;
    for (int z = 0; z < 2; ++z)
        for (int p = 0; p < 3; ++p) {
            for (int q = 0; q < 4; ++q) T[z][p][q] = fix::to_fix(u[p * 8 + 4 * z + q], E[z]);
            bfly4xy(T[z][p]);
            for (int q = 0; q < 4; ++q) T[z][p][q] = fix::down(T[z][p][q], Em - E[z]);
        }
    fix::cell_faces3(T[0], T[1], Em, psi, fc, Fb, Ft, e);
    for (int p = 0; p < 3; ++p) {
        bfly4xyT(Fb[p]);
        bfly4xyT(Ft[p]);
        for (int q = 0; q < 4; ++q) {
            F[p * 8 + q] = fix::to_double(Fb[p][q], e);
            F[p * 8 + 4 + q] = fix::to_double(Ft[p][q], e);
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def cell3(tmp_path_factory):
    oracle.build()
    d = tmp_path_factory.mktemp("fix")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    fn = C.CDLL(str(so)).cell3
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))

    def call(h, mod, u, psi):
        mod, u, F = np.array(mod, float), np.array(u, float), np.zeros(24)
        return fn(C.c_double(h), ptr(mod), ptr(u), C.c_double(psi), ptr(F)), F
    return call


@pytest.mark.parametrize("mod", [(1.0, 0.6, 0.5), W.iso_cubic(1480.0, 0.22), (1.0, -0.3, 0.4), (1.0, 0.0, 1e-3)])
@pytest.mark.parametrize("scale", [1.0, 1e-120, 1e120])
def test_cell_forces(cell3, mod, scale):
    h = 1.0 / 64
    P = oracle.Problem(3, (2, 2, 2), h, *mod)
    for seed, kind in enumerate(("random", "stretch", "rigid", "zero", "spread")):
        u = W.uniform(40 + seed, 24, -1, 1)
        if kind == "stretch":                     # small strain on a large displacement
            u = 1.0 + 1e-5 * u
        elif kind == "rigid":
            u = np.repeat(u[:3], 8)
        elif kind == "zero":
            u = np.zeros(24)
        elif kind == "spread":                    # components and corners of very different size
            u = u * 10.0 ** W.uniform(60, 24, -9, 0)
        u = u * scale
        for psi in (1.0, 0.37, 1e-8, 0.0):
            ref = oracle.apply(P, np.array([psi]), u)
            st, F = cell3(h, mod, u, psi)
            assert st == 0
            # the oracle's own rounding: 24 terms of |K| |u|, K's largest entries of order max(mod) / h^2
            bound = 24 * 2.0 ** -52 * 3.0 * max(mod) / h ** 2 * psi * np.abs(u).max()
            assert np.abs(F - ref).max() <= bound, (kind, psi)
            if kind in ("rigid", "zero") or psi == 0.0:
                assert np.all(F == 0.0)


def test_values_outside_the_range_are_refused(cell3):
    u = W.uniform(41, 24, -1, 1)
    for bad in (np.inf, -np.inf, np.nan, 1e200, 5e-324):
        v = np.zeros(24) if bad == 5e-324 else u.copy()
        v[11] = bad
        assert cell3(1.0, (1.0, 0.6, 0.5), v, 1.0)[0] == 1
    assert cell3(1.0, (1.0, 0.6, 0.5), u * 1e-200, 1.0)[0] == 1
    for psi in (-1.0, np.nan, np.inf, 1e-90, 1e90):
        assert cell3(1.0, (1.0, 0.6, 0.5), u, psi)[0] == 1
    assert cell3(1e-40, (1.0, 0.6, 0.5), u, 1.0)[0] == 1


def test_psi_of_negative_zero(cell3):
    st, F = cell3(1.0, (1.0, 0.6, 0.5), W.uniform(42, 24, -1, 1), -0.0)
    assert st == 0 and np.all(F == 0.0)
