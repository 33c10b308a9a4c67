// k_source.cu — the source terms of eq. SBMLinearElasticity (Sec. 2.1),
//     div(psi C (grad u - eps0)) - psi b = t |grad psi|,
// brought to the form K u = f of the cell-flux operator:
//     f_n = h^-d sum_{cells c of n} psi_c int_c B_n^T C eps0_c  -  w_n (psi_n b_n + t_n |grad psi|_n).
// For an eigenstrain that is constant in each cell the cell integral is closed form:
// int_c dN_n/dx_q = s_q h^(d-1) / 2^(d-1), s_q = +1 when the cell lies below the node
// along q, -1 above, so the eigenstrain load is sum_c sum_q s_q (psi_c C eps0_c)_pq /
// (2^(d-1) h).  psi_n is the mean of the 2^d cells around the node, the gradient along
// a the mean of (psi_+ - psi_-) / h over the cell pairs facing each other across the
// node; cells beyond a face of the box take the value of their mirror image (no
// normal gradient at the box), and w_n = (cells of the grid around n) / 2^d is the
// node's share of the volume.  The diffuse traction t is given at the nodes (the
// traction of the closest point of the boundary).  FP64, packed arrays; a cell pass
// forms each cell's eigenstrain stress once, then one thread per node gathers from
// its cells (no atomics).  This is setup work, run once per load: not part of the
// V-cycle.
//
// Bound by FP64 issue (about two lanes per SM and clock): the gather's 72 + 32 additions a
// node run on 64-bit integers instead, the node's values turned into them on the
// largest exponent of the stress rows (53 bits kept down to 2^-5 of it); 16 FP64 instructions a node are
// left, and the square root where psi is not constant around the node.  Values that do
// not fit (infinities, NaN, extreme exponents) are added in FP64.
#include "sbm_common.cuh"
#include "sbm_fix.cuh"

namespace sbm {

namespace {

constexpr int kThr = 256;

struct SourceArgs {
    int nx, ny, nz;
    double inv;            // 1 / (2^(d-1) h)
    double c11, c12, c44;
};

// Voigt slot of the symmetric pair (a, b): 2D (xx, yy, xy), 3D (xx, yy, zz, yz, xz, xy).
template <int D>
__device__ __forceinline__ int vslot(int a, int b)
{
    if (a == b) return a;
    if (D == 2) return 2;
    return 6 - a - b;        // (1,2) -> 3, (0,2) -> 4, (0,1) -> 5
}

// Pass 1: the eigenstrain stress of every cell, sig_c = psi_c C eps0_c (Voigt slots,
// slot-major like eps0).
template <int D>
__global__ void __launch_bounds__(kThr) k_cell_stress(const SourceArgs A, const double *__restrict__ psi,
                                                      const double *__restrict__ eps0, double *__restrict__ sig)
{
    const int NC = (A.nx - 1) * (A.ny - 1) * (D == 3 ? A.nz - 1 : 1);
    const int c = blockIdx.x * kThr + threadIdx.x;
    if (c >= NC) return;
    double e[D == 3 ? 6 : 3];
#pragma unroll
    for (int v = 0; v < (D == 3 ? 6 : 3); ++v) e[v] = eps0[v * NC + c];
    double tr = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) tr += e[a];
    // cubic C: sigma_pp = (c11 - c12) e_pp + c12 tr, sigma_pq = 2 c44 e_pq (tensor shear)
    const double pc = psi[c], l = A.c12 * tr, sh = pc * (2.0 * A.c44);
#pragma unroll
    for (int a = 0; a < D; ++a) sig[a * NC + c] = pc * madd(A.c11 - A.c12, e[a], l);
#pragma unroll
    for (int v = D; v < (D == 3 ? 6 : 3); ++v) sig[v * NC + c] = sh * e[v];
}

// Pass 2 (or the only pass without eigenstrain): one thread per node gathering its
// 2^d cells: the eigenstrain load sum_c sum_q s_q sig_pq(c) / (2^(d-1) h) from the
// cell stresses, psi_n, |grad psi|_n and the volume share for the body force and
// the traction.  The sums over the cells run on 64-bit integers (sbm_fix.cuh): with FP64
// instructions their issue bound the kernel.  All three terms at 129^3: 0.66 -> 0.30 ms, the
// node's own FP64 instructions (|grad psi|, the products with b and t) being most of it.
template <int D>
__global__ void __launch_bounds__(kThr) k_source_terms(const SourceArgs A, const double *__restrict__ psi,
                                                       const double *__restrict__ sig, const double *__restrict__ b,
                                                       const double *__restrict__ t, double *__restrict__ f)
{
    const int N = A.nx * A.ny * A.nz;          // < 2^31 (checked by the launcher)
    const int n = blockIdx.x * kThr + threadIdx.x;
    if (n >= N) return;
    const int nxy = A.nx * A.ny;
    const int nd[3] = {n % A.nx, (n % nxy) / A.nx, n / nxy};
    const int mc[3] = {A.nx - 1, A.ny - 1, D == 3 ? A.nz - 1 : 1};
    const int NC = mc[0] * mc[1] * mc[2];
    constexpr int NV = D == 3 ? 6 : 3, NK = 1 << D;
    double sv[NK][NV], pv[NK];                    // the cells' stresses (0 outside the grid) and psi (mirrored)
    unsigned kv[NV], kp = 0;                      // largest exponents: of each stress component, of psi
#pragma unroll
    for (int v = 0; v < NV; ++v) kv[v] = 0;
    int inside = 0;
#pragma unroll
    for (int c = 0; c < NK; ++c) {
        int cc[3] = {0, 0, 0};
        bool in = true;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            int v = nd[a] - 1 + ((c >> a) & 1);
            if (v < 0 || v >= mc[a]) in = false;
            cc[a] = min(max(v, 0), mc[a] - 1);
        }
        const int cid = cc[0] + mc[0] * (cc[1] + mc[1] * cc[2]);
        pv[c] = psi[cid];
        kp = max(kp, fix::exp_key(pv[c]));
        inside += in ? 1 : 0;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            sv[c][v] = (in && sig) ? sig[v * NC + cid] : 0.0;
            kv[v] = max(kv[v], fix::exp_key(sv[c][v]));
        }
    }
    double acc[D], ps, g[D];
    bool flat;                                    // no gradient of psi
    if (fix::key_ok(kp)) {
        const int E = max((int)(kp >> 20), fix::kExpLo);
        fix::i64 s = 0, d[D];
#pragma unroll
        for (int a = 0; a < D; ++a) d[a] = 0;
#pragma unroll
        for (int c = 0; c < NK; ++c) {
            const fix::i64 v = fix::to_fix(pv[c], E);
            s += v;
#pragma unroll
            for (int a = 0; a < D; ++a) d[a] += ((c >> a) & 1) ? v : -v;
        }
        ps = fix::to_double(s, E - fix::kFixUnit);
        fix::i64 any = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) any |= d[a];
        flat = any == 0;
#pragma unroll
        for (int a = 0; a < D; ++a) g[a] = flat ? 0.0 : fix::to_double(d[a], E - fix::kFixUnit);
    } else {
        ps = 0.0;
        flat = false;
#pragma unroll
        for (int a = 0; a < D; ++a) g[a] = 0.0;
#pragma unroll
        for (int c = 0; c < NK; ++c) {
            ps += pv[c];
#pragma unroll
            for (int a = 0; a < D; ++a) g[a] += ((c >> a) & 1) ? pv[c] : -pv[c];
        }
    }
    // s_q = +1 when the cell lies below the node along q (bit clear), -1 above.  A component of the
    // force sums a row of the stress; rows within 2^2 of each other share a unit (their own
    // largest values then keep 56 bits), others take one each.
    unsigned kr[D], ks = 0;
#pragma unroll
    for (int p = 0; p < D; ++p) {
        kr[p] = 0;
#pragma unroll
        for (int q = 0; q < D; ++q) kr[p] = max(kr[p], kv[vslot<D>(p, q)]);
        ks = max(ks, kr[p]);
    }
    bool shared = fix::key_ok(ks), each = true;
#pragma unroll
    for (int p = 0; p < D; ++p) {
        each = each && fix::key_ok(kr[p]);
        shared = shared && (kr[p] == 0u || (kr[p] >> 20) + 2u >= (ks >> 20));
    }
    if (shared) {
        const int E = max((int)(ks >> 20), fix::kExpLo);
        fix::i64 s[D];
#pragma unroll
        for (int p = 0; p < D; ++p) s[p] = 0;
#pragma unroll
        for (int c = 0; c < NK; ++c) {
            fix::i64 v[NV];
#pragma unroll
            for (int m = 0; m < NV; ++m) v[m] = fix::to_fix<5>(sv[c][m], E);     // 24 terms at most
#pragma unroll
            for (int p = 0; p < D; ++p)
#pragma unroll
                for (int q = 0; q < D; ++q) s[p] += ((c >> q) & 1) ? -v[vslot<D>(p, q)] : v[vslot<D>(p, q)];
        }
#pragma unroll
        for (int p = 0; p < D; ++p) acc[p] = fix::to_double(s[p], E - fix::kFixUnit + 2);
    } else if (each) {
#pragma unroll
        for (int p = 0; p < D; ++p) {
            const int E = max((int)(kr[p] >> 20), fix::kExpLo);
            fix::i64 s = 0;
#pragma unroll
            for (int c = 0; c < NK; ++c)
#pragma unroll
                for (int q = 0; q < D; ++q) {
                    const fix::i64 v = fix::to_fix<5>(sv[c][vslot<D>(p, q)], E);
                    s += ((c >> q) & 1) ? -v : v;
                }
            acc[p] = fix::to_double(s, E - fix::kFixUnit + 2);
        }
    } else {
#pragma unroll
        for (int p = 0; p < D; ++p) {
            acc[p] = 0.0;
#pragma unroll
            for (int c = 0; c < NK; ++c)
#pragma unroll
                for (int q = 0; q < D; ++q) {
                    const double v = sv[c][vslot<D>(p, q)];
                    acc[p] += ((c >> q) & 1) ? -v : v;
                }
        }
    }
    const double inv = A.inv;
    const double pn = ps * (1.0 / (1 << D));
    double gn = 0.0;
    if (!flat) {
        double gg = 0.0;
#pragma unroll
        for (int a = 0; a < D; ++a) gg += (g[a] * inv) * (g[a] * inv);
        gn = sqrt(gg);
    }
    const double w = (double)inside * (1.0 / (1 << D));
#pragma unroll
    for (int p = 0; p < D; ++p) {
        double s = 0.0;
        if (b) s += pn * b[p * N + n];
        if (t) s += t[p * N + n] * gn;
        f[p * N + n] = acc[p] * inv - w * s;
    }
}

}  // namespace

cudaError_t launch_source_terms(int dim, const int n[3], double h, const double mod[3], const double *psi,
                                const double *eps0, const double *b, const double *t, double *f, double *sig,
                                cudaStream_t s)
{
    SourceArgs A;
    A.nx = n[0];
    A.ny = n[1];
    A.nz = dim == 3 ? n[2] : 1;
    A.inv = 1.0 / ((dim == 3 ? 4.0 : 2.0) * h);
    A.c11 = mod[0];
    A.c12 = mod[1];
    A.c44 = mod[2];
    const long long N = (long long)A.nx * A.ny * A.nz;
    if (N * (dim == 3 ? 6 : 3) >= (1ll << 31)) return cudaErrorInvalidValue;   // 32-bit indexing
    const long long NC = (long long)(A.nx - 1) * (A.ny - 1) * (dim == 3 ? A.nz - 1 : 1);
    if (eps0) {
        if (!sig) return cudaErrorInvalidValue;
        const dim3 cgrid((unsigned)((NC + kThr - 1) / kThr));
        if (dim == 3) k_cell_stress<3><<<cgrid, kThr, 0, s>>>(A, psi, eps0, sig);
        else k_cell_stress<2><<<cgrid, kThr, 0, s>>>(A, psi, eps0, sig);
        ++g_launches;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)((N + kThr - 1) / kThr));
    if (dim == 3) k_source_terms<3><<<grid, kThr, 0, s>>>(A, psi, eps0 ? sig : nullptr, b, t, f);
    else k_source_terms<2><<<grid, kThr, 0, s>>>(A, psi, eps0 ? sig : nullptr, b, t, f);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace sbm
