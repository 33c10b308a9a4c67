// sbm_fix.cuh — the FP64 cell arithmetic of the operator in 64-bit integers.
//
// GB300 issues about one FP64 instruction for every 64 integer ones, so the FP64 stencil,
// evaluated with FP64 instructions, is bound by the FP64 pipe.  Here the same cell
// formula (sbm_cell.cuh) is evaluated in block floating point: a 64-bit integer mantissa
// per value and one power of two per cell.
//
//   1. The nodal values around a cell become integers |u| < 2^60 on a common power of
//      two, which follows the largest of the cell's own values: a double keeps all of its
//      53 bits down to 2^-7 (in the tiled 3D sweep 2^-6, see face_exp) of that value.
//   2. The mean/difference transform is exact (additions of integers).
//   3. The cell's 21 transformed values are shifted left until the largest reaches
//      2^60, so the products below keep the cell's own leading digits, however small
//      its strain is beside its displacement.
//   4. The constants psi C / h^2 are 62-bit fractions (psi as mantissa and exponent);
//      a product keeps its upper 64 bits.  A corner force of the cell stays
//      below 2^61, its bound over all values of step 3 (row sums of the stress map).
//   5. Forces of neighbouring cells are added after a shift to the larger of their
//      exponents and by the bits that the sum needs (kNodeBits); the sum is converted to
//      a double once per node.
//
// Errors.  Step 2 has none.  A product is off by 1.5 at most in units of 2^-61 of the
// cell's bound on a corner force, a sum over a node's cells by one unit of 2^-59 of the
// largest of their bounds for every cell.  Measured against 113-bit arithmetic, 20 000
// cells each, rms of a cell's largest corner error over its largest |K||u| (the formula in
// FP64 with FMAs in brackets), moduli (1, 0.6, 0.5): random values 3.5e-17 (8.5e-17),
// hourglass patterns 2.3e-17 (4.6e-17), components decades apart 4.3e-17 (1.0e-16),
// smooth displacements 1.2e-18 (4.1e-17).  Step 1 truncates values below 2^-7 of the largest.
// Values that do not fit the scheme
// (infinities, NaN, exponents beyond the range below, negative psi) are recognised while
// they are staged, and the caller evaluates those planes with FP64 instructions.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "sbm_cell.cuh"

namespace sbm {
namespace fix {

typedef long long i64;

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ int clz64(unsigned long long v) { return __clzll((long long)v); }
__device__ __forceinline__ i64 bits_of(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ double of_bits(i64 b) { return __longlong_as_double(b); }
#else
inline int clz64(unsigned long long v) { return v ? __builtin_clzll(v) : 64; }
inline i64 bits_of(double v) { i64 b; memcpy(&b, &v, 8); return b; }
inline double of_bits(i64 b) { double v; memcpy(&v, &b, 8); return v; }
#endif

// Biased exponents a staged value may have; with the bounds on the constants below, every
// result is then a normal number.  Zero is allowed as well.
constexpr int kExpLo = 600, kExpHi = 1500;
constexpr int kNoExp = -(1 << 20);      // exponent of a cell without force

// The exponent field of a value's magnitude as an ordered key: 0 for zero, key >> 20 the
// biased exponent otherwise (a denormal, with exponent 0, gives a key of at least 1).
__host__ __device__ __forceinline__ unsigned exp_key(double v)
{
    const i64 b = bits_of(v);
    return ((unsigned)(b >> 32) & 0x7fffffffu) | ((unsigned)b != 0u ? 1u : 0u);
}
__host__ __device__ __forceinline__ bool key_ok(unsigned key)
{
    return key == 0u || (key >= ((unsigned)kExpLo << 20) && key < ((unsigned)kExpHi << 20));
}

// The exponent that a face's values are staged on, from the key of the largest: rounded up to
// an odd one, so that the two faces of a cell mostly share it (a 129^3 residual of values all
// of one size 236 us, as with steps of four; 249 us without).  The values then keep 59 or 60
// bits of the largest: the residual of a solved displacement (45 x 37 x 41) is 5.0e-17 off against
// long double, 4.3e-17 of that the rounding of the result; 1.1e-16 with steps of four.
__host__ __device__ __forceinline__ int face_exp(unsigned key)
{
    const int e = (int)(key >> 20);
    return (e > kExpLo ? e : kExpLo) | 1;
}

// v as an integer on the unit 2^(E - 1023 - 52 - UP), E >= the biased exponent of v: below
// 2^(53 + UP).  UP = 7 unless sums of more than eight values follow.
template <int UP = 7>
__host__ __device__ __forceinline__ i64 to_fix(double v, int E)
{
    const i64 b = bits_of(v);
    const int ex = (int)((unsigned)(b >> 52) & 0x7ffu);
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    const unsigned sh = (unsigned)(E - ex);
    const i64 a = (i64)((m << UP) >> (sh < 63u ? sh : 63u));
    return b < 0 ? -a : a;
}
constexpr int kFixUnit = 1023 + 59;     // to_fix<7>'s unit is 2^(E - kFixUnit)

// a * 2^e as a double (e such that the result is normal; a may be zero).
__host__ __device__ __forceinline__ double to_double(i64 a, int e)
{
    const double v = (double)a;
    return a == 0 ? 0.0 : of_bits(bits_of(v) + ((i64)e << 52));
}

// A constant below 2^60 in two signed 32-bit parts, hi 2^32 + lo.
struct Frac {
    int hi, lo;
};
__host__ __device__ __forceinline__ Frac split(i64 k)
{
    Frac f;
    f.lo = (int)(unsigned)(unsigned long long)k;
    f.hi = (int)(k >> 32) + (f.lo < 0 ? 1 : 0);
    return f;
}

// (a k) / 2^64, off by -1.5 to 0.5 (the fraction and a_lo k_lo are dropped): three 32 x 32 -> 64
// bit products.  k >= 0 and |a| / 2 + k below 2^63, which keeps the sum of the cross products in
// 64 bits (psi's mantissa 2^62 + 2^61; the trace 1.6 2^61 + 1.8 2^61, a12 being at most 0.22 of
// the bound; any other value 2^62 + 2^62 at most, where k is far below that).
__host__ __device__ __forceinline__ i64 mul(i64 a, Frac k)
{
    const int ah = (int)(a >> 32);
    const unsigned al = (unsigned)(unsigned long long)a;
    const i64 t = (i64)((unsigned long long)((i64)ah * k.lo) + (unsigned long long)al * (unsigned)k.hi);
    return (i64)ah * k.hi + (t >> 32);
}

// Moduli constants of a level, prepared on the host as fractions of 2^ec.
// c[]: ad, |a12|, a44, (b1 + b12)/2, (b1 - b12)/2, b44, c2 of Coef (2D: a11 - a12, |a12|,
// a44, b1); neg12: a12 < 0.
struct Consts {
    Frac c[7];              // value = c 2^(ec - 63), c at most 2^61
    Frac d[7];              // 2 c, for products without psi
    int neg12;
    int ec;
    int ok;                 // the constants fit; otherwise the FP64 kernel is used
};

// Scale: with transformed values below 2^61 the corner forces stay below 2^61 and the
// constants times psi (scaled) below 2^62.
inline Consts make_consts(int dim, const Coef<double> &c)
{
    Consts r;
    memset(&r, 0, sizeof(r));
    const double a12 = fabs(c.a12), b12 = fabs(c.b12);
    double v[7], bound, big;
    if (dim == 3) {
        v[0] = c.ad; v[1] = a12; v[2] = c.a44;
        v[3] = 0.5 * (c.b1 + c.b12); v[4] = 0.5 * (c.b1 - c.b12);
        v[5] = c.b44; v[6] = c.c2;
        // the rows of the stress map that reach a corner's force along one axis
        bound = (c.ad + 3.0 * a12) + 4.0 * c.a44 + 2.0 * (c.b1 + b12) + 4.0 * c.b44 + c.c2;
    } else {
        v[0] = c.a11 - c.a12; v[1] = a12; v[2] = c.a44; v[3] = c.b1;
        v[4] = v[5] = v[6] = 0.0;
        bound = v[0] + 2.0 * a12 + 2.0 * c.a44 + c.b1;
    }
    big = 0.0;
    for (int i = 0; i < 7; ++i) {
        if (!(v[i] >= 0.0)) return r;
        big = fmax(big, v[i]);
    }
    bound = 1.0000001 * fmax(bound, 4.0 * big);      // (its own rounding)
    r.neg12 = c.a12 < 0.0;
    if (!(bound > ldexp(1.0, -200)) || !(bound < ldexp(1.0, 200))) return r;
    int eb;
    frexp(bound, &eb);                       // bound < 2^eb
    i64 k[7];
    for (int i = 0; i < 7; ++i) k[i] = (i64)rint(ldexp(v[i], 63 - eb));
    if (dim == 3) {                          // the sum and the difference without the rounding of a double
        const i64 p = (i64)rint(ldexp(c.b1, 62 - eb)), q = (i64)rint(ldexp(c.b12, 62 - eb));
        k[3] = p + q;
        k[4] = p - q;
    }
    for (int i = 0; i < 7; ++i) {
        r.c[i] = split(k[i]);
        r.d[i] = split(2 * k[i]);
    }
    r.ec = eb;
    r.ok = 1;
    return r;
}

// The constants a level's kernels run with.  The unit of a cell's forces goes with the bound
// on all of them, so where a12 and a44 are both far below it, the force along one axis from
// displacements along another would keep fewer digits than in FP64 (|a12|, a44 = bound / 64:
// components decades apart 1.0e-16 of the component's own |K||u|, FP64 1.3e-16): FP64 then.
inline Consts level_consts(int dim, const Coef<double> &c)
{
    Consts r = make_consts(dim, c);
    if (fmax(fabs(c.a12), c.a44) < ldexp(1.0, r.ec - 6)) r.ok = 0;
    return r;
}

// The constants of a cell: c times psi's mantissa, such that a normalised value times k
// over 2^64 is a force on the unit 2^(value's + psi's exponent + ec).
template <int N>
__host__ __device__ __forceinline__ void cell_consts(i64 pm, const Consts &c, Frac (&k)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) k[i] = split((i64)((unsigned long long)mul(pm, c.c[i]) << 2));
}

// Bits by which the corner forces of a node's 8 (3D) or 4 (2D) cells are shifted down
// before they are added.
constexpr int kNodeBits3 = 2, kNodeBits2 = 1;

// psi the scheme takes: 0 of either sign, or positive and within 2^+-200.
__host__ __device__ __forceinline__ bool psi_ok(double psi)
{
    const unsigned h = (unsigned)(bits_of(psi) >> 52);      // sign and exponent
    return psi == 0.0 || (h >= 823u && h < 1223u);
}

// psi > 0 as mantissa in [2^62, 2^63) and exponent: psi = m 2^(e - 63); mantissa 0 for 0.
__host__ __device__ __forceinline__ i64 psi_mantissa(double psi, int &e)
{
    const i64 b = bits_of(psi);
    e = (int)((unsigned)(b >> 52) & 0x7ffu) - 1022;
    return (b << 1) == 0 ? 0 : (i64)((((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull) << 10);
}

// The upper word of v's magnitude (less one for v < 0).
__host__ __device__ __forceinline__ unsigned mag_hi(i64 v)
{
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}

// Shift of the transformed values: all of them below 2^61 in magnitude afterwards.
// m: the OR of their magnitudes.
__host__ __device__ __forceinline__ int norm_shift(unsigned long long m) { return clz64(m) - 3; }

__host__ __device__ __forceinline__ i64 down(i64 v, int s) { return v >> (s > 63 ? 63 : s); }

// The 21 transformed values of a 3D cell that carry force (U[p][1..7] of bfly8), shifted up
// to 2^61 at most.  Returns the shift (-3 at least); none: all are zero.
// mh: the OR of their mag_hi.
__host__ __device__ __forceinline__ int normalize3(i64 (&U)[3][8], unsigned mh, bool &none)
{
    unsigned long long m = (unsigned long long)mh << 32 | 0xffffffffu;
    if (mh == 0u) {                          // all below 2^32: the magnitudes themselves decide
        m = 0;
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int s = 1; s < 8; ++s) m |= (unsigned long long)(U[p][s] < 0 ? -U[p][s] : U[p][s]);
    }
    none = m == 0ull;
    const int sh = norm_shift(m);
    int up = sh;
    if (sh < 0) {                            // sums of opposite corners near the bound
        up += 3;
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int s = 1; s < 8; ++s) U[p][s] >>= 3;
    }
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int s = 1; s < 8; ++s) U[p][s] = (i64)((unsigned long long)U[p][s] << (up & 63));
    return sh;
}

// The stress map of a 3D cell on normalised values, constants k (cell_consts, or Consts
// itself): dU[p][s], dU[p][0] = 0; the sum of a component's is below 2^61 in magnitude.
__host__ __device__ __forceinline__ void stress3(const i64 (&U)[3][8], const Frac (&k)[7], int neg12, i64 (&dU)[3][8])
{
    i64 ltr = mul(U[0][1] + U[1][2] + U[2][4], k[1]);
    ltr = neg12 ? -ltr : ltr;
    const i64 sxx = mul(U[0][1], k[0]) + ltr, syy = mul(U[1][2], k[0]) + ltr, szz = mul(U[2][4], k[0]) + ltr;
    const i64 sxy = mul(U[1][1] + U[0][2], k[2]);
    const i64 sxz = mul(U[2][1] + U[0][4], k[2]);
    const i64 syz = mul(U[2][2] + U[1][4], k[2]);
    const i64 S = U[2][3] + U[1][5] + U[0][6];
    // (b1 x + b12 y, b1 y + b12 x) from the sum and the difference of x and y
    i64 a, d;
    a = mul(U[0][3] + U[2][6], k[3]); d = mul(U[0][3] - U[2][6], k[4]);
    const i64 d03 = a + d, d26 = a - d;
    a = mul(U[1][3] + U[2][5], k[3]); d = mul(U[1][3] - U[2][5], k[4]);
    const i64 d13 = a + d, d25 = a - d;
    a = mul(U[0][5] + U[1][6], k[3]); d = mul(U[0][5] - U[1][6], k[4]);
    const i64 d05 = a + d, d16 = a - d;
    const i64 d23 = mul(S + U[2][3], k[5]), d15 = mul(S + U[1][5], k[5]), d06 = mul(S + U[0][6], k[5]);
    const i64 d07 = mul(U[0][7], k[6]), d17 = mul(U[1][7], k[6]), d27 = mul(U[2][7], k[6]);
    const i64 r[3][8] = {{0, sxx, sxy, d03, sxz, d05, d06, d07},
                         {0, sxy, syy, d13, syz, d15, d16, d17},
                         {0, sxz, syz, d23, szz, d25, d26, d27}};
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int s = 0; s < 8; ++s) dU[p][s] = r[p][s];
}

// One 3D cell: in-plane transforms (bfly4xy of the integers) of its bottom and top faces
// on the units 2^(Eb - kFixUnit) and 2^(Et - kFixUnit), its psi.  Returns the transformed
// face forces, the unit of which is 2^e (e = kNoExp: no force, Fb = Ft = 0).
__host__ __device__ __forceinline__ void cell_faces3(const i64 (&Tb)[3][4], int Eb, const i64 (&Tt)[3][4], int Et,
                                                     double psi, const Consts &c, i64 (&Fb)[3][4], i64 (&Ft)[3][4], int &e)
{
    i64 U[3][8], dU[3][8];
    const int E = Eb > Et ? Eb : Et;
    if (Eb == Et) {
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                U[p][s] = Tb[p][s] + Tt[p][s];
                U[p][s + 4] = Tt[p][s] - Tb[p][s];
            }
    } else {
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const i64 b = down(Tb[p][s], E - Eb), t = down(Tt[p][s], E - Et);
                U[p][s] = b + t;
                U[p][s + 4] = t - b;
            }
    }
    unsigned mh = 0;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            if (s > 0) mh |= mag_hi(U[p][s]);
            mh |= mag_hi(U[p][s + 4]);
        }
    bool none;
    const int sh = normalize3(U, mh, none);
    int ep;
    const i64 pm = psi_mantissa(psi, ep);
    e = (none || pm == 0) ? kNoExp : E - kFixUnit - sh + ep + c.ec;
    Frac k[7];
    cell_consts(pm, c, k);
    stress3(U, k, c.neg12, dU);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        Fb[p][0] = -dU[p][4];
        Ft[p][0] = dU[p][4];
#pragma unroll
        for (int s = 1; s < 4; ++s) {
            Fb[p][s] = dU[p][s] - dU[p][s + 4];
            Ft[p][s] = dU[p][s] + dU[p][s + 4];
        }
    }
}

__host__ __device__ __forceinline__ void cell_faces3(const i64 (&Tb)[3][4], const i64 (&Tt)[3][4], int E, double psi,
                                                     const Consts &c, i64 (&Fb)[3][4], i64 (&Ft)[3][4], int &e)
{
    cell_faces3(Tb, E, Tt, E, psi, c, Fb, Ft, e);
}

// Nodal values of a 3D cell as transformed, normalised integers: v = U 2^(e), e returned.
// False when a value does not fit.
__host__ __device__ __forceinline__ bool transform_cell3(const double (&v)[3][8], i64 (&U)[3][8], bool &none, int &e)
{
    unsigned key = 0;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const unsigned q = exp_key(v[p][a]);
            key = q > key ? q : key;
        }
    if (!key_ok(key)) return false;
    const int E = (int)(key >> 20) > kExpLo ? (int)(key >> 20) : kExpLo;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
#pragma unroll
        for (int a = 0; a < 8; ++a) U[p][a] = to_fix(v[p][a], E);
        bfly8(U[p]);
    }
    unsigned mh = 0;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int s = 1; s < 8; ++s) mh |= mag_hi(U[p][s]);
    e = E - kFixUnit - normalize3(U, mh, none);
    return true;
}

// Force on corner a of a 3D cell with transformed, normalised values U (transform_cell3,
// exponent eu) and psi: F on the unit 2^e (e = kNoExp: none).
__host__ __device__ __forceinline__ void corner_force3(const i64 (&U)[3][8], bool none, int eu, int a, double psi,
                                                       const Consts &c, i64 (&F)[3], int &e)
{
    i64 dU[3][8];
    int ep;
    const i64 pm = psi_mantissa(psi, ep);
    e = (none || pm == 0) ? kNoExp : eu + ep + c.ec;
    Frac k[7];
    cell_consts(pm, c, k);
    stress3(U, k, c.neg12, dU);
    // the transform's row of basis function s at corner a: the product over the axes of s of
    // +1 (corner bit set) or -1
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        i64 f = 0;
#pragma unroll
        for (int s = 1; s < 8; ++s) {
            const int m = s & ~a;                                  // axes of s whose corner bit is clear
            const bool neg = ((m ^ (m >> 1) ^ (m >> 2)) & 1) != 0;
            f += neg ? -dU[p][s] : dU[p][s];
        }
        F[p] = f;
    }
}

// v^T S u of a 3D cell (S the unit-psi cell matrix of the constants c), u and v given as
// transform_cell3 leaves them: the sum, in 128 bits, of 21 products of the stress of u with
// the transform of v, in the basis where the cell's rigid motion has dropped out.
__host__ __device__ __forceinline__ double cell_work3(const i64 (&U)[3][8], int eu, const i64 (&V)[3][8], int ev,
                                                      const Consts &c)
{
    i64 dU[3][8];
    stress3(U, c.d, c.neg12, dU);
    __int128 s = 0;                          // 3 x 2^61 x 2^61 at most
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 1; q < 8; ++q) s += (__int128)dU[p][q] * V[p][q];
    const i64 hi = (i64)(s >> 64);
    const unsigned long long lo = (unsigned long long)s;
    if (s == 0) return 0.0;
    // dU = U c / 2^63 with c in units of 2^(ec - 63)
    const double d = (double)hi * 18446744073709551616.0 + (double)lo;
    const int e = eu + ev + c.ec, f = (int)((unsigned)(bits_of(d) >> 52) & 0x7ffu) + e;
    return f > 0 && f < 2047 ? of_bits(bits_of(d) + ((i64)e << 52)) : ldexp(d, e);
}

// The six transformed values of a 2D cell that carry force, in the order U[0][1..3],
// U[1][1..3] of bfly4, shifted up to 2^61 at most.  Returns the shift.
__host__ __device__ __forceinline__ int transform2(const i64 (&u)[2][4], i64 (&U)[2][4], bool &none)
{
    unsigned long long m = 0;
    i64 any = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
#pragma unroll
        for (int q = 0; q < 4; ++q) U[p][q] = u[p][q];
        bfly4(U[p]);
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            any |= U[p][q];
            m |= (unsigned long long)(U[p][q] ^ (U[p][q] >> 63));   // 0 for -1 as for 0
        }
    }
    none = any == 0;
    const int sh = norm_shift(m);            // |U| <= 4 2^60: at least -2
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 1; q < 4; ++q)
            U[p][q] = sh >= 0 ? (i64)((unsigned long long)U[p][q] << (sh & 63)) : U[p][q] >> (-sh & 63);
    return sh;
}

// One 2D cell: nodal integers on the unit 2^(E - kFixUnit) -> corner forces on 2^e.
__host__ __device__ __forceinline__ void cell_forces2(const i64 (&u)[2][4], int E, double psi, const Consts &c,
                                                      i64 (&F)[2][4], int &e)
{
    i64 U[2][4];
    bool none;
    const int sh = transform2(u, U, none);
    int ep;
    const i64 pm = psi_mantissa(psi, ep);
    e = (none || pm == 0) ? kNoExp : E - kFixUnit - sh + ep + c.ec;
    Frac k[4];
    cell_consts(pm, c, k);
    i64 ltr = mul(U[0][1] + U[1][2], k[1]);
    ltr = c.neg12 ? -ltr : ltr;
    const i64 sxy = mul(U[1][1] + U[0][2], k[2]);
    F[0][0] = 0; F[0][1] = mul(U[0][1], k[0]) + ltr; F[0][2] = sxy; F[0][3] = mul(U[0][3], k[3]);
    F[1][0] = 0; F[1][1] = sxy; F[1][2] = mul(U[1][2], k[0]) + ltr; F[1][3] = mul(U[1][3], k[3]);
    bfly4T(F[0]);
    bfly4T(F[1]);
}

// The same for the force on corner a alone; psi multiplies the two forces, which come out
// below 2^60 (no bits to make room for before they are added).
__host__ __device__ __forceinline__ void corner_force2(const i64 (&u)[2][4], int a, int E, double psi, const Consts &c,
                                                       i64 (&F)[2], int &e)
{
    i64 U[2][4];
    bool none;
    const int sh = transform2(u, U, none);
    int ep;
    const i64 pm = psi_mantissa(psi, ep);
    e = (none || pm == 0) ? kNoExp : E - kFixUnit - sh + ep + c.ec + 1;
    i64 ltr = mul(U[0][1] + U[1][2], c.d[1]);
    ltr = c.neg12 ? -ltr : ltr;
    const i64 sxx = mul(U[0][1], c.d[0]) + ltr, syy = mul(U[1][2], c.d[0]) + ltr;
    const i64 sxy = mul(U[1][1] + U[0][2], c.d[2]);
    const i64 d0 = mul(U[0][3], c.d[3]), d1 = mul(U[1][3], c.d[3]);
    const bool px = (a & 1) != 0, py = (a & 2) != 0;
    const Frac k = split(pm >> 1);
    F[0] = mul(2 * ((px ? sxx : -sxx) + (py ? sxy : -sxy) + (px == py ? d0 : -d0)), k);
    F[1] = mul(2 * ((px ? sxy : -sxy) + (py ? syy : -syy) + (px == py ? d1 : -d1)), k);
}

}  // namespace fix
}  // namespace sbm
