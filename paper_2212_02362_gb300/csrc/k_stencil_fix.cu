// k_stencil_fix.cu — FP64 apply / residual / damped-Jacobi sweep and the 2D FP64 colour
// Gauss-Seidel sweep with the cell arithmetic in 64-bit integers (sbm_fix.cuh).
//
// What bounds it (3D).  With FP64 instructions the sweep is bound by their issue rate (about
// two lanes per SM and clock on GB300): some 180 of them per cell.  In block floating
// point a cell takes some 1100 integer instructions, conversions included, which issue 64
// times as fast, and leaves some ten FP64 instructions per node (the conversion of the
// node's force, f - K u, the norm), which run on the FP64 pipe beside them.
//
// Work split.  A block owns a tile of 32 x 10 cells in x/y (33 x 11 threads, one per cell
// column with the halo column and row; 12 warps, so 168 registers a thread) and a
// contiguous range of (tile, node plane) units, which it streams along z, one cell layer
// a step.  Node planes pass through a four-slot shared-memory ring, so that nothing
// inside a step waits for global memory and one barrier a step suffices.  In step lz
//   plane lz+4  is copied by cp.async (into the slot that plane lz left in step lz - 1)
//   plane lz+3  has arrived: each thread takes the largest exponent of each node it copied
//   plane lz+1  is read by the cells of layer lz, each turning its face's values into
//               integers on a unit of its own (the exponents of its four nodes), kept
//               for the layer above; where a cell's two faces differ, both are shifted to
//               the larger of their units
// The forces a layer sends to its top plane are carried in registers in the transformed
// basis with their exponent; those of the four columns around a node are exchanged
// through a double-buffered shared array with the exponents beside them.
//
// A cell or a psi that the integer form does not take (sbm_fix.cuh) ends the integer
// loop before any node that depends on it; the block finishes its range with the FP64
// body below, which also runs when the level's constants do not fit.
//
// A unit per staged plane and tile instead (values converted once, in place, instead of by
// the four cells around a column) took 213 us for a 129^3 residual call, 231 now, but lost the digits
// of cells far below the tile's largest value.
//
// Measured (kernel time, FP64 instructions -> this form): residual with norm at 129^3
// 812 -> 204 us (0.84 TB/s), Jacobi sweep with kept scaling at 65^3 155 -> 35 us, at 33^3 46 ->
// 11.5 us; issue and latency of one block of 12 warps per SM (registers).
#include <algorithm>

#include "sbm_common.cuh"
#include "sbm_bodies.cuh"
#include "sbm_fix.cuh"

namespace sbm {

namespace {

using fix::i64;

constexpr int TX = 32, TY = 10;                   // cells of a tile
constexpr int BX = TX + 1, BY = TY + 1, NT = BX * BY;
constexpr int PX = TX + 2, PY = TY + 2, PP = PX * PY;
// ring of node planes (4 x 3 components); two buffers of 9 exchanged forces, psi of the
// cells below + above and the exponent (the FP64 body: 12 forces and psi); the ring's node keys
constexpr size_t kSmem = sizeof(double) * (12 + 2 * (9 + 1)) * PP + (2 + 4) * sizeof(int) * PP;

// 8-byte global -> shared copy; ok = false fills zeros (src must still be valid).
__device__ __forceinline__ void cp_async8(void *sdst, const void *gsrc, bool ok)
{
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(sdst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gsrc), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Deterministic block reduction of ssq into *out.
template <int N>
__device__ __forceinline__ void block_partial(double ssq, double *out, double *red)
{
    constexpr int NW = (N + 31) / 32;
    const int tid = threadIdx.x;
    red[tid] = ssq;
    if (tid < NW * 32 - N) red[N + tid] = 0.0;
    __syncthreads();
    if (tid < 32) {
        double s = 0.0;
        for (int w = 0; w < NW; ++w) s += red[w * 32 + tid];
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (tid == 0) *out = s;
    }
}

// Index of cell (i, j, k) in a.psi.
template <typename TO>
__device__ __forceinline__ long long pidx(const SweepArgs<double, TO> &a, int i, int j, int k)
{
    return i + (long long)(a.psx ? a.psx : a.g.sx) * j + (a.psx ? a.psy : a.g.sy) * k;
}

// One tile's share of the grid for this thread.
struct Tile {
    int x0, y0;            // first owned node
    int gx, gy;            // the thread's node; its cell is (gx - 1, gy - 1)
    bool own, cell_ok;
};

__device__ __forceinline__ Tile make_tile(const Geom &g, int t, int ntx, int tx, int ty)
{
    Tile T;
    T.x0 = (t % ntx) * TX;
    T.y0 = (t / ntx) * TY;
    T.gx = T.x0 + tx;
    T.gy = T.y0 + ty;
    T.own = T.gx < g.nx && T.gy < g.ny && (tx < TX || T.gx == g.nx - 1) && (ty < TY || T.gy == g.ny - 1);
    T.cell_ok = T.gx >= 1 && T.gx < g.nx && T.gy >= 1 && T.gy < g.ny;
    return T;
}

// The staged nodes of this thread (tid and, for the first few threads, tid + NT): their
// offset within a plane, -1 outside the grid.
struct Stage {
    int o0, o1;
};

__device__ __forceinline__ Stage make_stage(const Geom &g, const Tile &T)
{
    auto off = [&](int s) {
        const int gx = T.x0 - 1 + s % PX, gy = T.y0 - 1 + s / PX;
        return (s < PP && gx >= 0 && gx < g.nx && gy >= 0 && gy < g.ny) ? gx + g.sx * gy : -1;
    };
    return {off(threadIdx.x), off(threadIdx.x + NT)};
}
static_assert(PP <= 2 * NT, "two staged nodes a thread at most");

// Node plane k of a tile into the shared array dst[3][PP] (zeros outside the grid).
__device__ __forceinline__ void load_plane(const double *u, const Geom &g, const Stage &S, int k, double *dst)
{
    const bool in = k >= 0 && k < g.nz;
    const double *pl = u + (in ? g.sy * k : 0);
    auto node = [&](int o, int s) {
        const bool ok = in && o >= 0;
        const double *q = ok ? pl + o : u;
#pragma unroll
        for (int p = 0; p < 3; ++p) cp_async8(dst + p * PP + s, q + (ok ? p * g.cs : 0), ok);
    };
    node(S.o0, threadIdx.x);
    if (threadIdx.x + NT < PP) node(S.o1, threadIdx.x + NT);
    cp_async_commit();
}

// The units [ub, ue) with FP64 instructions: what the integer form does not take.  A node
// plane's in-plane transform is shared by the two cell layers it bounds, and planes come
// through a three-slot ring two steps ahead.
template <typename TO, int MODE>
__device__ __noinline__ double sweep_dp(const SweepArgs<double, TO> &a, long long ub, long long ue, double *up)
{
    double *fc = up + 12 * PP, *ps = fc + 12 * PP;
    const Geom &g = a.g;
    const int tid = threadIdx.x;
    int tx, ty;
    row_warp_xy<BY>(tid, tx, ty);
    cp_async_wait_all();
    __syncthreads();
    for (int s = tid; s < PP; s += NT) {
        const int lx = s % PX, ly = s / PX;
        if (lx == BX || ly == BY) {
            for (int q = 0; q < 12; ++q) fc[q * PP + s] = 0.0;
            ps[s] = 0.0;
        }
    }
    const int ntx = (g.nx - 1 + TX - 1) / TX;
    double ssq = 0.0;
    for (long long su = ub; su < ue;) {
        const int kz0 = (int)(su % g.nz);
        const int kend = (int)min((long long)g.nz, kz0 + (ue - su)) - 1;   // last node plane finalised
        const Tile T = make_tile(g, (int)(su / g.nz), ntx, tx, ty);
        const Stage S = make_stage(g, T);
        su += kend + 1 - kz0;
        const int kfirst = kz0 > 0 ? kz0 - 1 : 0;
        const int me = ty * PX + tx;
        auto corners = [&](int k, double (&C)[3][4]) {
            const double *pl = up + (k % 3) * 3 * PP;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                C[p][0] = pl[p * PP + me];
                C[p][1] = pl[p * PP + me + 1];
                C[p][2] = pl[p * PP + me + PX];
                C[p][3] = pl[p * PP + me + PX + 1];
                bfly4xy(C[p]);
            }
        };
        auto cell_psi = [&](int lz) {
            return (T.cell_ok && lz <= g.nz - 2) ? a.psi[pidx(a, T.gx - 1, T.gy - 1, lz)] : 0.0;
        };
        double Tb[3][4], Cf[3][4];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int s = 0; s < 4; ++s) Cf[p][s] = 0.0;
        double psi_prev = 0.0;
        double psi = cell_psi(kfirst);
        load_plane(a.u, g, S, kfirst, up + (kfirst % 3) * 3 * PP);
        load_plane(a.u, g, S, kfirst + 1, up + ((kfirst + 1) % 3) * 3 * PP);
        cp_async_wait_all();
        __syncthreads();
        corners(kfirst, Tb);
        for (int lz = kfirst; lz <= kend; ++lz) {
            load_plane(a.u, g, S, lz + 2, up + ((lz + 2) % 3) * 3 * PP);   // slot of plane lz - 1
            const double psi_next = cell_psi(lz + 1);
            const bool fin = T.own && lz >= kz0;
            double fv[3];
            const long long on = gidx(g, T.gx, T.gy, lz);
#pragma unroll
            for (int p = 0; p < 3; ++p) fv[p] = (MODE != kApply && fin) ? a.f[p * g.cs + on] : 0.0;
            double Tt[3][4], Fb[3][4], Ft[3][4];
            corners(lz + 1, Tt);
            cell_faces3<double>(Tb, Tt, psi, a.c, Fb, Ft);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    Fb[p][s] += Cf[p][s];   // plane lz: top face of layer lz-1 + bottom face of layer lz
                    Cf[p][s] = Ft[p][s];
                    Tb[p][s] = Tt[p][s];
                }
                bfly4xyT(Fb[p]);
#pragma unroll
                for (int q = 0; q < 4; ++q) fc[(p * 4 + q) * PP + me] = Fb[p][q];
            }
            ps[me] = psi_prev + psi;
            psi_prev = psi;
            psi = psi_next;
            __syncthreads();
            if (fin) {
                double Ku[3], uv[3];
                const double *pl = up + (lz % 3) * 3 * PP;
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    Ku[p] = (fc[(p * 4 + 3) * PP + me] + fc[(p * 4 + 2) * PP + me + 1]) +
                            (fc[(p * 4 + 1) * PP + me + PX] + fc[(p * 4 + 0) * PP + me + PX + 1]);
                    uv[p] = pl[p * PP + me + PX + 1];
                }
                const double ip = MODE == kJacobi ? 1.0 / ((ps[me] + ps[me + 1]) + (ps[me + PX] + ps[me + PX + 1])) : 0.0;
                body::finalize_f<double, TO, MODE>(a, T.gx, T.gy, lz, Ku, ip, uv, fv, ssq);
            }
            cp_async_wait_all();                              // plane lz + 2 in this thread's copies
            __syncthreads();
        }
    }
    return ssq;
}

template <typename TO, int MODE>
__global__ void __launch_bounds__(NT, 1) k_sweep3_fix(const SweepArgs<double, TO> a, const fix::Consts fc)
{
    pdl_begin();
    if (a.gate && *a.gate) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *up = reinterpret_cast<double *>(smem_raw);        // [4][3][PP] ring of node planes
    i64 *X2 = reinterpret_cast<i64 *>(up + 12 * PP);           // [2][9][PP]: corner forces 0..2 of a plane
    double *ps2 = up + 30 * PP;                                // [2][PP]
    int *Xe2 = reinterpret_cast<int *>(ps2 + 2 * PP);          // [2][PP]: exponents of the forces
    unsigned *node_keys = reinterpret_cast<unsigned *>(Xe2 + 2 * PP);   // [4][PP]: of the ring's nodes
    __shared__ double red[((NT + 31) / 32) * 32];

    const Geom &g = a.g;
    const int tid = threadIdx.x;
    int tx, ty;
    row_warp_xy<BY>(tid, tx, ty);
    for (int s = tid; s < PP; s += NT) {
        const int lx = s % PX, ly = s / PX;
        if (lx == BX || ly == BY) {                            // no cells there
            for (int q = 0; q < 18; ++q) X2[q * PP + s] = 0;
            Xe2[s] = Xe2[PP + s] = fix::kNoExp;
            ps2[s] = ps2[PP + s] = 0.0;
        }
    }
    const int ntx = (g.nx - 1 + TX - 1) / TX, nty = (g.ny - 1 + TY - 1) / TY;
    const long long U = (long long)ntx * nty * g.nz;
    const long long ub = U * blockIdx.x / gridDim.x, ue = U * (blockIdx.x + 1) / gridDim.x;
    const int me = ty * PX + tx;
    double ssq = 0.0;
    int buf = 0;
    long long rest = fc.ok ? ue : ub;          // units from here on are left to the FP64 body

    auto slot = [&](int k) { return up + (k & 3) * 3 * PP; };
    // the largest exponent key of each node this thread copied
    auto take_key = [&](int k) {
        const double *pl = slot(k);
        unsigned *nk = node_keys + (k & 3) * PP;
        auto node = [&](int s) {
            nk[s] = max(max(fix::exp_key(pl[s]), fix::exp_key(pl[PP + s])), fix::exp_key(pl[2 * PP + s]));
        };
        node(tid);
        if (tid + NT < PP) node(tid + NT);
    };
    // and of the four nodes of this thread's face
    auto face_key = [&](int k) {
        const unsigned *nk = node_keys + (k & 3) * PP;
        return max(max(nk[me], nk[me + 1]), max(nk[me + PX], nk[me + PX + 1]));
    };
    // the face's values as integers on E, transformed
    auto corners = [&](int k, int E, i64 (&C)[3][4]) {
        const double *pl = slot(k);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            C[p][0] = fix::to_fix(pl[p * PP + me], E);
            C[p][1] = fix::to_fix(pl[p * PP + me + 1], E);
            C[p][2] = fix::to_fix(pl[p * PP + me + PX], E);
            C[p][3] = fix::to_fix(pl[p * PP + me + PX + 1], E);
            bfly4xy(C[p]);
        }
    };

    for (long long su = ub; su < ue && rest == ue;) {
        const int t = (int)(su / g.nz), kz0 = (int)(su % g.nz);
        const int kend = (int)min((long long)g.nz, kz0 + (ue - su)) - 1;   // last node plane finalised
        const long long seg = su - kz0;                                    // unit of the tile's plane 0
        const Tile T = make_tile(g, t, ntx, tx, ty);
        su += kend + 1 - kz0;
        const int kfirst = kz0 > 0 ? kz0 - 1 : 0;
        // the cell column's psi from here on (advanced a layer at a time)
        const double *pp = a.psi + (T.cell_ok ? pidx(a, T.gx - 1, T.gy - 1, kfirst) : 0);
        const long long psy = a.psx ? a.psy : g.sy;
        auto cell_psi = [&](int lz) { return (T.cell_ok && lz <= g.nz - 2) ? *pp : 0.0; };
        const Stage S = make_stage(g, T);
        // the last step of a segment leaves a copy (plane kend + 4) in flight; copies are not
        // ordered among each other, so it has to land before its slot is loaded again
        cp_async_wait_all();
        // planes kfirst to kfirst + 2 with their keys, kfirst + 3 on its way
        for (int k = kfirst; k < kfirst + 3; ++k) load_plane(a.u, g, S, k, slot(k));
        double psi = cell_psi(kfirst), psi_prev = 0.0;
        cp_async_wait_all();
        __syncthreads();
        load_plane(a.u, g, S, kfirst + 3, slot(kfirst + 3));
        for (int k = kfirst; k < kfirst + 3; ++k) take_key(k);
        if (__syncthreads_or(!fix::psi_ok(psi))) {
            rest = seg + kz0;
            break;
        }
        i64 Tb[3][4], Cf[3][4];
        unsigned kb = face_key(kfirst);                        // the bottom face: its key, its unit
        int Eb = fix::face_exp(kb), ecf = fix::kNoExp;
        corners(kfirst, Eb, Tb);
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) Cf[p][q] = 0;
        __syncthreads();                                       // plane kfirst's slot is free
#pragma unroll 1
        for (int lz = kfirst; lz <= kend; ++lz) {
            cp_async_wait_all();                               // plane lz + 3 in this thread's copies
            take_key(lz + 3);
            load_plane(a.u, g, S, lz + 4, slot(lz + 4));
            i64 *X = X2 + buf * 9 * PP;
            int *Xe = Xe2 + buf * PP;
            double *ps = ps2 + buf * PP;
            pp += psy;
            const double psi_next = cell_psi(lz + 1);
            const bool fin = T.own && lz >= kz0;
            double fv[3], uv[3];
            const long long on = fin ? gidx(g, T.gx, T.gy, lz) : 0;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                fv[p] = (MODE != kApply && fin) ? a.f[p * g.cs + on] : 0.0;
                uv[p] = (MODE == kJacobi && fin) ? a.u[p * g.cs + on] : 0.0;
            }
            double ip = (MODE == kJacobi && a.dinv && fin) ? a.dinv[on] : 0.0;
            // the cell of layer lz
            const unsigned kt = face_key(lz + 1);
            const bool fits = fix::key_ok(max(kb, kt));
            const int Et = fix::face_exp(kt);
            i64 Tt[3][4], Fb[3][4], Ft[3][4];
            corners(lz + 1, Et, Tt);
            int e;
            fix::cell_faces3(Tb, Eb, Tt, Et, psi, fc, Fb, Ft, e);
#pragma unroll
            for (int p = 0; p < 3; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) Tb[p][q] = Tt[p][q];
            kb = kt;
            Eb = Et;
            // plane lz: top face of layer lz - 1 + bottom face of layer lz
            const int en = max(e, ecf), s0 = en - ecf, s1 = en - e;
            i64 N[3][4];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    N[p][q] = fix::down(Cf[p][q], s0) + fix::down(Fb[p][q], s1);
                    Cf[p][q] = Ft[p][q];
                }
                bfly4xyT(N[p]);
#pragma unroll
                for (int q = 0; q < 3; ++q) X[(p * 3 + q) * PP + me] = N[p][q];
            }
            Xe[me] = en;
            ecf = e;
            if (MODE == kJacobi && !a.dinv) ps[me] = psi_prev + psi;
            psi_prev = psi;
            psi = psi_next;
            if (__syncthreads_or(!fits || (!fix::psi_ok(psi) && lz < kend))) {
                rest = seg + max(lz, kz0);                     // this plane's cells, or the next psi
                break;
            }
            buf ^= 1;
            if (fin) {
                const int e1 = Xe[me + 1], e2 = Xe[me + PX], e3 = Xe[me + PX + 1];
                const int ee = max(max(en, e1), max(e2, e3)) + fix::kNodeBits3;
                const int d0 = ee - en, d1 = ee - e1, d2 = ee - e2, d3 = ee - e3;
                double Ku[3];
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const i64 s = (fix::down(N[p][3], d0) + fix::down(X[(p * 3 + 2) * PP + me + 1], d1)) +
                                  (fix::down(X[(p * 3 + 1) * PP + me + PX], d2) +
                                   fix::down(X[(p * 3 + 0) * PP + me + PX + 1], d3));
                    Ku[p] = fix::to_double(s, ee);
                }
                if (MODE == kJacobi && !a.dinv)
                    ip = 1.0 / ((ps[me] + ps[me + 1]) + (ps[me + PX] + ps[me + PX + 1]));
                body::finalize_f<double, TO, MODE>(a, T.gx, T.gy, lz, Ku, ip, uv, fv, ssq);
            }
        }
    }
    if (rest < ue) ssq += sweep_dp<TO, MODE>(a, rest, ue, up);
    if (MODE == kResidual && a.part) {
        __syncthreads();
        block_partial<NT>(ssq, a.part + blockIdx.x, red);
    }
}

// Small 3D levels: eight consecutive threads per node, thread c evaluating the cell of which
// the node is corner c; exponents and forces are combined by shuffles and the first three
// lanes finalise a component each.  A cell that does not fit sends its warp to FP64
// instructions.  No shared memory, no barrier, no plane ring: what is left is one round
// of loads and one cell's chain (7 us at 17^3 against 12 us tiled; see kNode64MaxNodes).
constexpr int kNode64Threads = 128;

template <int MODE>
__global__ void __launch_bounds__(kNode64Threads) k_sweep3_node64(const SweepArgs<double, double> a, const fix::Consts fc)
{
    const Geom &g = a.g;
    const int n = g.nx * g.ny * g.nz;
    const int node = blockIdx.x * (kNode64Threads / 8) + (threadIdx.x >> 3);
    const int c = threadIdx.x & 7;
    const bool valid = node < n;
    const int i = node % g.nx, j = node / g.nx % g.ny, k = node / (g.nx * g.ny);
    const int ci = i - (c & 1), cj = j - ((c >> 1) & 1), ck = k - (c >> 2);
    const bool has = valid && ci >= 0 && cj >= 0 && ck >= 0 && ci < g.nx - 1 && cj < g.ny - 1 && ck < g.nz - 1;
    const long long on = valid ? gidx(g, i, j, k) : 0;
    const int p = c < 3 ? c : 0;                          // the component this lane finalises (lanes 0..2)
    // what no kernel of the cycle writes is read before the wait for the predecessor
    const double psi = has ? a.psi[pidx(a, ci, cj, ck)] : 0.0;
    double ip = (MODE == kJacobi && a.dinv) ? a.dinv[on] : 0.0;
    pdl_begin();
    if (a.gate && *a.gate) return;
    double V[3][8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const long long o = has ? gidx(g, ci + (b & 1), cj + ((b >> 1) & 1), ck + (b >> 2)) : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) V[q][b] = has ? a.u[q * g.cs + o] : 0.0;
    }
    const double uv = MODE == kJacobi ? a.u[p * g.cs + on] : 0.0;
    const double fv = MODE != kApply ? a.f[p * g.cs + on] : 0.0;
    i64 U[3][8], F[3];
    bool none;
    int eu, e;
    const bool ok = fix::transform_cell3(V, U, none, eu) && fix::psi_ok(psi) && fc.ok;
    double Ku = 0.0;
    if (__all_sync(0xffffffffu, ok)) {
        fix::corner_force3(U, none, eu, c, psi, fc, F, e);
        int ee = e;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) ee = max(ee, __shfl_xor_sync(0xffffffffu, ee, off));
        ee += fix::kNodeBits3;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            F[q] = fix::down(F[q], ee - e);
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) F[q] += __shfl_xor_sync(0xffffffffu, F[q], off);
        }
        Ku = fix::to_double(p == 0 ? F[0] : p == 1 ? F[1] : F[2], ee);
    } else {
        cell_forces3<double>(V, psi, a.c);
        double f[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            f[q] = V[q][0];
#pragma unroll
            for (int b = 1; b < 8; ++b) f[q] = c == b ? V[q][b] : f[q];
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) f[q] += __shfl_xor_sync(0xffffffffu, f[q], off);
        }
        Ku = p == 0 ? f[0] : p == 1 ? f[1] : f[2];
    }
    if (MODE == kJacobi && !a.dinv) {
        double s = psi;                                   // over z, x, y: the order of dinv
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        ip = 1.0 / s;
    }
    if (!valid || c >= 3) return;
    const bool dir = is_dir(g, p, i, j, k);
    double r;
    if (MODE == kJacobi) r = dir ? uv : uv + (fv - Ku) * ip * (p == 0 ? a.wk[0] : p == 1 ? a.wk[1] : a.wk[2]);
    else if (MODE == kResidual) r = dir ? 0.0 : fv - Ku;
    else r = Ku;
    a.out[p * g.cs + on] = r;
}

// ------------------------------------------------------------------------- 2D
//
// One thread per cell of a 32 x TY2 tile (the first row and column the halo), which
// turns its own four corners into integers on their largest exponent: no staging and no
// block-wide unit, one barrier for the exchange of the corner forces.  A block with a
// value that does not fit evaluates its cells with FP64 instructions.  What is left is
// latency (one round of loads, one barrier), so small grids take the flat tile, which
// spreads the FP64 instructions of the update over twice as many SMs.  A Jacobi sweep took
// 9.6 us at 65^2 and 40 us at 513^2 with FP64 instructions; 2.9 and 12 us here.
constexpr int TX2 = 32;

// PRO: u is taken as u + P ec, ec the correction on the coarse level gc (a prolongation
// launch less; on large grids its FP64 additions, repeated by the cells around a node, cost
// more than the launch).
template <typename TO, int MODE, int TY2, bool PRO>
__global__ void __launch_bounds__((TX2 + 1) * (TY2 + 1))
    k_sweep2_fix(const SweepArgs<double, TO> a, const fix::Consts fc, const Geom gc, const double *__restrict__ ec)
{
    constexpr int BX2 = TX2 + 1, BY2 = TY2 + 1, NT2 = BX2 * BY2, PX2 = TX2 + 2, PP2 = PX2 * (TY2 + 2);
    __shared__ i64 X[2][4][PP2];                   // corner forces (integers, or doubles where they do not fit)
    __shared__ int Xe[PP2];
    __shared__ double ps[PP2];
    __shared__ double red[((NT2 + 31) / 32) * 32];
    const Geom &g = a.g;
    const int tid = threadIdx.x;
    int tx, ty;
    row_warp_xy<BY2>(tid, tx, ty);
    for (int s = tid; s < PP2; s += NT2) {
        if (s % PX2 == BX2 || s / PX2 == BY2) {
            for (int q = 0; q < 8; ++q) (&X[0][0][0])[q * PP2 + s] = 0;
            Xe[s] = fix::kNoExp;
            ps[s] = 0.0;
        }
    }
    const int gx = blockIdx.x * TX2 + tx, gy = blockIdx.y * TY2 + ty;
    const bool own = gx < g.nx && gy < g.ny && (tx < TX2 || gx == g.nx - 1) && (ty < TY2 || gy == g.ny - 1);
    const bool cell_ok = gx >= 1 && gx < g.nx && gy >= 1 && gy < g.ny;
    const long long on = gidx(g, gx, gy, 0);
    // what no kernel of the cycle writes is read before the wait for the predecessor
    if (a.foreign_psi) pdl_wait();
    const double psi = cell_ok ? a.psi[pidx(a, gx - 1, gy - 1, 0)] : 0.0;
    double ip = (MODE == kJacobi && a.dinv && own) ? a.dinv[on] : 0.0;
    pdl_begin();
    if (a.gate && *a.gate) return;
    double D[2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = gx - 1 + (q & 1), j = gy - 1 + (q >> 1);
        const bool ok = i >= 0 && i < g.nx && j >= 0 && j < g.ny;
        const long long o = ok ? gidx(g, i, j, 0) : 0;
#pragma unroll
        for (int p = 0; p < 2; ++p) D[p][q] = ok ? a.u[p * g.cs + o] : 0.0;
    }
    if (PRO) {
        // the coarse cell around this cell; along an axis an even cell holds its first node
        // and the midpoint, an odd one the midpoint and its second node
        const bool ox = ((gx - 1) & 1) != 0, oy = ((gy - 1) & 1) != 0;
        double C[2][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = ((gx - 1) >> 1) + (q & 1), j = ((gy - 1) >> 1) + (q >> 1);
            const bool ok = i >= 0 && i < gc.nx && j >= 0 && j < gc.ny;
            const long long o = ok ? gidx(gc, i, j, 0) : 0;
#pragma unroll
            for (int p = 0; p < 2; ++p) C[p][q] = ok ? ec[p * gc.cs + o] : 0.0;
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
#pragma unroll
            for (int r = 0; r < 4; r += 2) {
                const double m = 0.5 * (C[p][r] + C[p][r + 1]);
                C[p][r + (ox ? 0 : 1)] = m;
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const double m = 0.5 * (C[p][r] + C[p][r + 2]);
                C[p][r + (oy ? 0 : 2)] = m;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = gx - 1 + (q & 1), j = gy - 1 + (q >> 1);
                if (i >= 0 && i < g.nx && j >= 0 && j < g.ny) D[p][q] += C[p][q];
            }
        }
    }
    double fv[2] = {0.0, 0.0};
    if (MODE != kApply && own) {
        fv[0] = a.f[on];
        fv[1] = a.f[g.cs + on];
    }
    const double uv[2] = {D[0][3], D[1][3]};
    const int me = ty * PX2 + tx;
    unsigned key = 0;
    i64 I[2][4], F[2][4];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) key = max(key, fix::exp_key(D[p][q]));
    const bool ok = fc.ok && fix::key_ok(key) && fix::psi_ok(psi);
    const int E = max((int)(key >> 20), fix::kExpLo);
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) I[p][q] = fix::to_fix(D[p][q], E);
    int e;
    fix::cell_forces2(I, E, psi, fc, F, e);
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) X[p][q][me] = F[p][q];
    Xe[me] = e;
    ps[me] = psi;
    const bool all = __syncthreads_and(ok) != 0;
    double Ku[2] = {0.0, 0.0};
    if (all) {
        if (own) {
            const int e1 = Xe[me + 1], e2 = Xe[me + PX2], e3 = Xe[me + PX2 + 1];
            const int ee = max(max(e, e1), max(e2, e3)) + fix::kNodeBits2;
#pragma unroll
            for (int p = 0; p < 2; ++p)
                Ku[p] = fix::to_double((fix::down(F[p][3], ee - e) + fix::down(X[p][2][me + 1], ee - e1)) +
                                           (fix::down(X[p][1][me + PX2], ee - e2) +
                                            fix::down(X[p][0][me + PX2 + 1], ee - e3)),
                                       ee);
        }
    } else {
        cell_forces2<double>(D, psi, a.c);
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) X[p][q][me] = fix::bits_of(D[p][q]);
        __syncthreads();
        if (own)
#pragma unroll
            for (int p = 0; p < 2; ++p)
                Ku[p] = fix::of_bits(X[p][3][me]) + fix::of_bits(X[p][2][me + 1]) + fix::of_bits(X[p][1][me + PX2]) +
                        fix::of_bits(X[p][0][me + PX2 + 1]);
    }
    double ssq = 0.0;
    if (own) {
        if (MODE == kJacobi && !a.dinv) ip = 1.0 / (ps[me] + ps[me + 1] + ps[me + PX2] + ps[me + PX2 + 1]);
        body::finalize_f<double, TO, MODE>(a, gx, gy, 0, Ku, ip, uv, fv, ssq);
    }
    if (MODE == kResidual && a.part)
        block_partial<NT2>(ssq, a.part + blockIdx.x + (long long)gridDim.x * blockIdx.y, red);
}

// Rows of cells per block: 8, on grids that would give fewer blocks than SMs 4.
int rows2(const Geom &g)
{
    return ((g.nx + 30) / 32) * (long long)((g.ny + 6) / 8) >= 152 ? 8 : 4;
}

// Small 2D levels: the residual with its full weighting and the coarse level's first sweep
// in one launch.  A block takes CT x CT coarse nodes: the forces of the (2 CT + 2)^2 cells
// around them, the residuals of the (2 CT + 1)^2 fine nodes, then the weighted sums.
constexpr int CT = 4, RC = 2 * CT + 2, RN = 2 * CT + 1, kRrThreads = 128;
static_assert(RC * RC <= kRrThreads, "one thread a cell");

__global__ void __launch_bounds__(kRrThreads) k_resid_restrict2(const SweepArgs<double, double> a, const fix::Consts fc,
                                                                const Geom gc, double *__restrict__ rhs,
                                                                const FirstSweep<double> first)
{
    __shared__ i64 X[2][4][RC * RC];
    __shared__ int Xe[RC * RC];
    __shared__ double R[2][RN * RN];
    const Geom &g = a.g;
    const int tid = threadIdx.x;
    const int I0 = blockIdx.x * CT, J0 = blockIdx.y * CT;
    const int lx = tid % RC, ly = tid / RC;
    const int cx = 2 * I0 - 2 + lx, cy = 2 * J0 - 2 + ly;          // this thread's cell
    const bool cell = tid < RC * RC;
    const bool cell_ok = cell && cx >= 0 && cx < g.nx - 1 && cy >= 0 && cy < g.ny - 1;
    const double psi = cell_ok ? a.psi[gidx(g, cx, cy, 0)] : 0.0;
    const int I = I0 + tid % CT, J = J0 + tid / CT;                // this thread's coarse node
    const bool coarse = tid < CT * CT && I < gc.nx && J < gc.ny;
    double ip = 0.0;
    if (first.u && coarse) ip = first.dinv ? first.dinv[gidx(gc, I, J, 0)] : body::inv_psi_sum<double, 2>(gc, first.psi, I, J, 0);
    pdl_begin();
    if (a.gate && *a.gate) return;
    double D[2][4];
    unsigned key = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = cx + (q & 1), j = cy + (q >> 1);
        const bool ok = cell && i >= 0 && i < g.nx && j >= 0 && j < g.ny;
        const long long o = ok ? gidx(g, i, j, 0) : 0;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            D[p][q] = ok ? a.u[p * g.cs + o] : 0.0;
            key = max(key, fix::exp_key(D[p][q]));
        }
    }
    const int nx = tid % RN, ny = tid / RN;                        // this thread's fine node
    const int gi = 2 * I0 - 1 + nx, gj = 2 * J0 - 1 + ny;
    const bool node = tid < RN * RN && gi >= 0 && gi < g.nx && gj >= 0 && gj < g.ny;
    double fv[2] = {0.0, 0.0};
#pragma unroll
    for (int p = 0; p < 2; ++p)
        if (node) fv[p] = a.f[p * g.cs + gidx(g, gi, gj, 0)];
    const int E = max((int)(key >> 20), fix::kExpLo);
    i64 U[2][4], F[2][4];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) U[p][q] = fix::to_fix(D[p][q], E);
    int e;
    fix::cell_forces2(U, E, psi, fc, F, e);
    const bool all = __syncthreads_and(fc.ok && fix::key_ok(key) && fix::psi_ok(psi)) != 0;
    if (!all) cell_forces2<double>(D, psi, a.c);
    if (cell) {
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) X[p][q][tid] = all ? F[p][q] : fix::bits_of(D[p][q]);
        Xe[tid] = e;
    }
    __syncthreads();
    if (tid < RN * RN) {
        const int c3 = ny * RC + nx, c2 = c3 + 1, c1 = c3 + RC, c0 = c1 + 1;   // the node's corner in its cells
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            double Ku;
            if (all) {
                const int ee = max(max(Xe[c0], Xe[c1]), max(Xe[c2], Xe[c3])) + fix::kNodeBits2;
                Ku = fix::to_double((fix::down(X[p][3][c3], ee - Xe[c3]) + fix::down(X[p][2][c2], ee - Xe[c2])) +
                                        (fix::down(X[p][1][c1], ee - Xe[c1]) + fix::down(X[p][0][c0], ee - Xe[c0])),
                                    ee);
            } else {
                Ku = fix::of_bits(X[p][3][c3]) + fix::of_bits(X[p][2][c2]) + fix::of_bits(X[p][1][c1]) +
                     fix::of_bits(X[p][0][c0]);
            }
            R[p][tid] = (!node || is_dir(g, p, gi, gj, 0)) ? 0.0 : fv[p] - Ku;
        }
    }
    __syncthreads();
    if (coarse) {
        const int m = (2 * (tid / CT) + 1) * RN + 2 * (tid % CT) + 1;   // the coincident fine node
        double f[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            double r[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double *row = R[p] + m + (d - 1) * RN;
                r[d] = row[0] + 0.5 * (row[-1] + row[1]);
            }
            f[p] = is_dir(gc, p, I, J, 0) ? 0.0 : 0.25 * (r[1] + 0.5 * (r[0] + r[2]));
            rhs[p * gc.cs + gidx(gc, I, J, 0)] = f[p];
        }
        if (first.u) body::first_sweep<double, 2>(first, gc, I, J, 0, ip, f);
    }
}

// 2D colour Gauss-Seidel in FP64, one launch per sweep.  A block owns a TILE x TILE tile of
// nodes and stages u, f and psi on the tile plus a four-node halo; the four colour phases
// then run in shared memory, phase q relaxing its colour on the tile grown by 3 - q nodes,
// so every value a phase reads was produced by the phases before it exactly as in four
// separate colour passes.  Only the tile is written, to a second buffer.  A phase is a
// chain of one node's update, so its work is spread: a thread takes one of a node's four
// cells (the corner force in integers), then, after a barrier, one thread per node adds
// the four and updates.  A node with a value that does not fit takes its row of K in FP64.
// The diagonal blocks follow from psi sums: every corner of the unit-psi cell matrix has
// the same diagonal entry, and the same coupling up to its sign (+ at corners 0 and 3).
// A sweep of the refinement levels (1 to 49 tiles) took 51 us with FP64 instructions and a
// thread per node, 11 to 14 us here; what is left is the four phases' chain.
constexpr int kGsThreads = 512;

template <int TILE>
__global__ void __launch_bounds__(kGsThreads) k_gs2_fix(const Geom g, const fix::Consts fc,
                                                        const double *__restrict__ psi, const double *__restrict__ Ke,
                                                        const double *__restrict__ f, const double *__restrict__ uin,
                                                        double *__restrict__ uout, int descending, const int *gate)
{
    constexpr int H = 4, SN = TILE + 2 * H, SC = SN - 1, SF = SN - 2;
    constexpr int NQ = (TILE + 6) / 2 * ((TILE + 6) / 2);  // nodes of the largest phase
    constexpr int kBad = 1 << 20;                          // exponent of a cell that does not fit
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *su = reinterpret_cast<double *>(smem_raw);   // [2][SN][SN] staged nodes
    double *sf = su + 2 * SN * SN;                        // [2][SF][SF] right-hand side of staged nodes 1 .. SN-2
    double *sw = sf + 2 * SF * SF;                        // [2][SF][SF] 1 / diagonal and coupling of the node's block
    double *sp = sw + 2 * SF * SF;                        // [SC][SC] psi of the staged cells (0 outside the grid)
    i64 *X = reinterpret_cast<i64 *>(sp + SC * SC);       // [4][2][NQ] corner forces of a phase
    int *Xe = reinterpret_cast<int *>(X + 8 * NQ);        // [4][NQ] their exponents
    const int tid = threadIdx.x, nt = kGsThreads;
    const int x0 = blockIdx.x * TILE - H, y0 = blockIdx.y * TILE - H;   // global node of staged (0, 0)
    // psi and the diagonal blocks, which no kernel of the cycle writes, before the wait for
    // the predecessor: the divisions run while it drains
    for (int s = tid; s < SC * SC; s += nt) {
        const int i = x0 + s % SC, j = y0 + s / SC;
        const bool ok = i >= 0 && i < g.nx - 1 && j >= 0 && j < g.ny - 1;
        sp[s] = ok ? psi[gidx(g, i, j, 0)] : 0.0;
    }
    const double kd = Ke[0], k01 = Ke[1];                 // corner 0: diagonal and coupling
    __syncthreads();
    for (int s = tid; s < SF * SF; s += nt) {
        const int lx = s % SF, ly = s / SF;               // cells below and above staged node (lx + 1, ly + 1)
        const double p3 = sp[ly * SC + lx], p2 = sp[ly * SC + lx + 1], p1 = sp[(ly + 1) * SC + lx],
                     p0 = sp[(ly + 1) * SC + lx + 1];
        const int i = x0 + 1 + lx, j = y0 + 1 + ly;
        if (i < 0 || i >= g.nx || j < 0 || j >= g.ny) continue;
        sw[s] = 1.0 / (kd * ((p0 + p1) + (p2 + p3)));
        sw[SF * SF + s] = k01 * ((p0 + p3) - (p1 + p2));
    }
    pdl_begin();
    if (gate && *gate) return;
    for (int s = tid; s < SN * SN; s += nt) {
        const int i = x0 + s % SN, j = y0 + s / SN;
        const bool ok = i >= 0 && i < g.nx && j >= 0 && j < g.ny;
        const long long o = ok ? gidx(g, i, j, 0) : 0;
        su[s] = ok ? uin[o] : 0.0;
        su[SN * SN + s] = ok ? uin[g.cs + o] : 0.0;
    }
    for (int s = tid; s < SF * SF; s += nt) {
        const int i = x0 + 1 + s % SF, j = y0 + 1 + s / SF;
        const bool ok = i >= 0 && i < g.nx && j >= 0 && j < g.ny;
        const long long o = ok ? gidx(g, i, j, 0) : 0;
        sf[s] = ok ? f[o] : 0.0;
        sf[SF * SF + s] = ok ? f[g.cs + o] : 0.0;
    }
    __syncthreads();
    for (int q = 0; q < 4; ++q) {
        const int c = descending ? 3 - q : q;
        const int h = 3 - q;                              // halo still relaxed in this phase
        const int lo = H - h, nr = (TILE + 2 * h) / 2;    // first staged index, colour nodes per row
        const int nq = nr * nr;
        const int lx0 = lo + (((c & 1) - lo) & 1), ly0 = lo + (((c >> 1) - lo) & 1);
        for (int t = tid; t < 4 * nq; t += nt) {
            const int a = t / nq, n = t - a * nq;         // the node is corner a of the cell
            const int cx = lx0 + 2 * (n % nr) - (a & 1), cy = ly0 + 2 * (n / nr) - (a >> 1);
            const double pc = sp[cy * SC + cx];
            double v[2][4];
            unsigned key = 0;
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    v[p][b] = su[p * SN * SN + (cy + (b >> 1)) * SN + cx + (b & 1)];
                    key = max(key, fix::exp_key(v[p][b]));
                }
            int e = kBad;
            if (fc.ok && fix::key_ok(key) && fix::psi_ok(pc)) {
                const int E = max((int)(key >> 20), fix::kExpLo);
                i64 I[2][4], F[2];
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int b = 0; b < 4; ++b) I[p][b] = fix::to_fix(v[p][b], E);
                fix::corner_force2(I, a, E, pc, fc, F, e);
                X[(a * 2) * NQ + n] = F[0];
                X[(a * 2 + 1) * NQ + n] = F[1];
            }
            Xe[a * NQ + n] = e;
        }
        __syncthreads();
        for (int n = tid; n < nq; n += nt) {
            const int lx = lx0 + 2 * (n % nr), ly = ly0 + 2 * (n / nr);
            const int i = x0 + lx, j = y0 + ly;
            if (i < 0 || j < 0 || i >= g.nx || j >= g.ny) continue;
            const int me = ly * SN + lx, mf = (ly - 1) * SF + lx - 1;
            const double w = sw[mf], s01 = sw[SF * SF + mf];
            int e[4], ee = fix::kNoExp;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                e[a] = Xe[a * NQ + n];
                ee = max(ee, e[a]);
            }
            double Ku[2] = {0.0, 0.0};
            if (ee != kBad) {
#pragma unroll
                for (int p = 0; p < 2; ++p)
                    Ku[p] = fix::to_double(
                        (fix::down(X[p * NQ + n], ee - e[0]) + fix::down(X[(2 + p) * NQ + n], ee - e[1])) +
                            (fix::down(X[(4 + p) * NQ + n], ee - e[2]) + fix::down(X[(6 + p) * NQ + n], ee - e[3])),
                        ee);
            } else {
                for (int a = 0; a < 4; ++a)
                    for (int p = 0; p < 2; ++p) {
                        double t = 0.0;
                        for (int b = 0; b < 4; ++b)
                            for (int r = 0; r < 2; ++r)
                                t = madd(Ke[(a * 2 + p) * 8 + b * 2 + r],
                                         su[r * SN * SN + me + ((b >> 1) - (a >> 1)) * SN + (b & 1) - (a & 1)], t);
                        Ku[p] = madd(sp[(ly - (a >> 1)) * SC + lx - (a & 1)], t, Ku[p]);
                    }
            }
            if (!is_dir(g, 0, i, j, 0)) {
                const double du = (sf[mf] - Ku[0]) * w;
                su[me] += du;
                Ku[1] = madd(s01, du, Ku[1]);
            }
            if (!is_dir(g, 1, i, j, 0)) su[SN * SN + me] += (sf[SF * SF + mf] - Ku[1]) * w;
        }
        __syncthreads();
    }
    for (int s = tid; s < TILE * TILE; s += nt) {
        const int lx = H + s % TILE, ly = H + s / TILE;
        const int i = x0 + lx, j = y0 + ly;
        if (i >= g.nx || j >= g.ny) continue;
        const long long o = gidx(g, i, j, 0);
        uout[o] = su[ly * SN + lx];
        uout[g.cs + o] = su[SN * SN + ly * SN + lx];
    }
}

template <int TILE>
cudaError_t launch_gs2_tile(const Geom &g, const fix::Consts &fc, const double *psi, const double *Ke, const double *f,
                            const double *uin, double *uout, int descending, cudaStream_t s, const int *gate)
{
    constexpr int SN = TILE + 8, NQ = (TILE + 6) / 2 * ((TILE + 6) / 2);
    constexpr size_t sm = sizeof(double) * (2 * SN * SN + 4 * (SN - 2) * (SN - 2) + (SN - 1) * (SN - 1) + 8 * NQ) +
                          sizeof(int) * 4 * NQ;
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = smem_attr_once(reinterpret_cast<const void *>(k_gs2_fix<TILE>), sm, attr_done);
    if (e != cudaSuccess) return e;
    const dim3 gr((g.nx + TILE - 1) / TILE, (g.ny + TILE - 1) / TILE, 1);
    e = launch_pdl(k_gs2_fix<TILE>, gr, dim3(kGsThreads), sm, s, g, fc, psi, Ke, f, uin, uout, descending, gate);
    if (e != cudaSuccess) return e;
    ++g_launches;
    return cudaGetLastError();
}

__global__ void k_inv_psi(const Geom g, const double *__restrict__ psi, double *__restrict__ dinv)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z * blockDim.z + threadIdx.z;
    if (i >= g.nx || j >= g.ny || k >= g.nz) return;
    dinv[gidx(g, i, j, k)] =
        g.dim == 3 ? body::inv_psi_sum<double, 3>(g, psi, i, j, k) : body::inv_psi_sum<double, 2>(g, psi, i, j, k);
}

template <typename TO, int MODE>
cudaError_t launch_fix_mode(const SweepArgs<double, TO> &a, cudaStream_t s)
{
    const fix::Consts fc = fix::level_consts(a.g.dim, a.c);
    cudaError_t e;
    if (a.g.dim == 3) {
        static std::atomic<unsigned long long> attr_done{0};
        e = smem_attr_once(reinterpret_cast<const void *>(k_sweep3_fix<TO, MODE>), kSmem, attr_done);
        if (e != cudaSuccess) return e;
        e = launch_pdl(k_sweep3_fix<TO, MODE>, dim3((unsigned)(a.max_ctas ? std::min<long long>(sweep_blocks_fix(a.g), a.max_ctas) : sweep_blocks_fix(a.g))),
                       dim3(NT), kSmem, s, a, fc);
    } else {
        const int ty = rows2(a.g);
        const dim3 gr((a.g.nx + 30) / 32, (a.g.ny - 2 + ty) / ty), b(33 * (ty + 1));
        const double *none = nullptr;
        e = ty == 8 ? launch_pdl(k_sweep2_fix<TO, MODE, 8, false>, gr, b, 0, s, a, fc, a.g, none)
                    : launch_pdl(k_sweep2_fix<TO, MODE, 4, false>, gr, b, 0, s, a, fc, a.g, none);
    }
    if (e != cudaSuccess) return e;
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace

// 3D: one block per SM of the 152, at most one per (tile, node plane) unit.  2D: the tiles.
long long sweep_blocks_fix(const Geom &g)
{
    if (g.dim == 2) {
        const int ty = rows2(g);
        return ((g.nx + 30) / 32) * (long long)((g.ny - 2 + ty) / ty);
    }
    const long long units = (long long)((g.nx - 1 + TX - 1) / TX) * ((g.ny - 1 + TY - 1) / TY) * g.nz;
    return std::min<long long>(152, units);
}

cudaError_t launch_sweep_node64(int mode, const SweepArgs<double, double> &a, cudaStream_t s)
{
    if (a.g.dim != 3 || (long long)a.g.nx * a.g.ny * a.g.nz >= (1 << 24)) return cudaErrorInvalidValue;
    const int n = a.g.nx * a.g.ny * a.g.nz;
    const dim3 gr((n + kNode64Threads / 8 - 1) / (kNode64Threads / 8)), b(kNode64Threads);
    const fix::Consts fc = fix::level_consts(3, a.c);
    cudaError_t e;
    switch (mode) {
    case kApply: e = launch_pdl(k_sweep3_node64<kApply>, gr, b, 0, s, a, fc); break;
    case kResidual: e = launch_pdl(k_sweep3_node64<kResidual>, gr, b, 0, s, a, fc); break;
    case kJacobi: e = launch_pdl(k_sweep3_node64<kJacobi>, gr, b, 0, s, a, fc); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_prolong_sweep(const SweepArgs<double, double> &a, const Geom &gc, const double *ec, cudaStream_t s)
{
    if (a.g.dim != 2 || a.u == a.out) return cudaErrorInvalidValue;
    const fix::Consts fc = fix::level_consts(2, a.c);
    const int ty = rows2(a.g);
    const dim3 gr((a.g.nx + 30) / 32, (a.g.ny - 2 + ty) / ty), b(33 * (ty + 1));
    cudaError_t e = ty == 8 ? launch_pdl(k_sweep2_fix<double, kJacobi, 8, true>, gr, b, 0, s, a, fc, gc, ec)
                            : launch_pdl(k_sweep2_fix<double, kJacobi, 4, true>, gr, b, 0, s, a, fc, gc, ec);
    if (e != cudaSuccess) return e;
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_resid_restrict(const SweepArgs<double, double> &a, const Geom &gc, double *fc,
                                  const FirstSweep<double> &first, cudaStream_t s)
{
    if (a.g.dim != 2) return cudaErrorInvalidValue;
    const dim3 gr((gc.nx + CT - 1) / CT, (gc.ny + CT - 1) / CT);
    cudaError_t e = launch_pdl(k_resid_restrict2, gr, dim3(kRrThreads), 0, s, a, fix::level_consts(2, a.c), gc, fc, first);
    if (e != cudaSuccess) return e;
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_inv_psi(const Geom &g, const double *psi, double *dinv, cudaStream_t s)
{
    const dim3 b(32, 4, 2), gr((g.nx + 31) / 32, (g.ny + 3) / 4, (g.nz + 1) / 2);
    k_inv_psi<<<gr, b, 0, s>>>(g, psi, dinv);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_gs2_fix(const Geom &g, const Coef<double> &c, const double *psi, const double *Ke, const double *f,
                           const double *uin, double *uout, int descending, cudaStream_t s, const int *gate)
{
    const fix::Consts fc = fix::level_consts(2, c);
    const long long b32 = ((g.nx + 31) / 32) * (long long)((g.ny + 31) / 32);
    if (b32 >= 304) return launch_gs2_tile<32>(g, fc, psi, Ke, f, uin, uout, descending, s, gate);
    return launch_gs2_tile<16>(g, fc, psi, Ke, f, uin, uout, descending, s, gate);
}

template <typename TO>
cudaError_t launch_sweep_fix(int mode, const SweepArgs<double, TO> &a, cudaStream_t s)
{
    switch (mode) {
    case kApply: return launch_fix_mode<TO, kApply>(a, s);
    case kResidual: return launch_fix_mode<TO, kResidual>(a, s);
    case kJacobi: return launch_fix_mode<TO, kJacobi>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

template cudaError_t launch_sweep_fix<double>(int, const SweepArgs<double, double> &, cudaStream_t);
template cudaError_t launch_sweep_fix<float>(int, const SweepArgs<double, float> &, cudaStream_t);

}  // namespace sbm
