// dpde_device.cuh -- device-side building blocks of the DPDE step (sm_103a).
//
// Precision is a template parameter T of positions, momenta, forces and pair
// arithmetic: double (FP64 mode) or float (mixed mode). Internal energies use
// the type E: double in FP64 mode, a compensated float pair (hi + lo, about
// 48 significant bits) in the mixed mode, so that the small per-pair energy
// reinjections are not lost against eps ~ C_v T.
//
// Particle data are cell-sorted structures of arrays (slot order):
//   q   : (ox, oy, oz, id bits) -- offset of the particle inside its cell,
//                                  o in [0, l) with l = L / ncell per axis
//   cc  : packed cell coordinates cx | cy << 10 | cz << 20
//   p   : (px, py, pz, beta)    -- beta_i = C_v / eps_i, Eq. (DPDE_internalEOS)
//   eps : E
// Cell-relative offsets keep float positions at ~1e-7 absolute resolution
// whatever the box size; the distance between particles of cells c and
// c + d is (o_i - o_j) - d * l, which also gives the periodic image.
#pragma once

#include <cmath>

#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

namespace dpde {

// 32-byte aligned four-double vector (one 256-bit access per particle).
struct __align__(32) d4 {
    double x, y, z, w;
};

// Compensated float pair: value = hi + lo with |lo| <= ulp(hi)/2.
struct __align__(8) ff {
    float hi, lo;
};

template <class T> struct V;
template <> struct V<double> { using t = d4; using e = double; };
template <> struct V<float> { using t = float4; using e = ff; };
template <class T> using vec_t = typename V<T>::t;
template <class T> using eps_t = typename V<T>::e;

__device__ __forceinline__ uint32_t id_of(const float4& q) { return __float_as_uint(q.w); }
__device__ __forceinline__ uint32_t id_of(const d4& q) {
    return (uint32_t)__double_as_longlong(q.w);
}
__device__ __forceinline__ void set_id(float4& q, uint32_t id) { q.w = __uint_as_float(id); }
__device__ __forceinline__ void set_id(d4& q, uint32_t id) {
    q.w = __longlong_as_double((long long)id);
}

// ---------------------------------------------------------------------------
// compensated float arithmetic (Knuth's two-sum; Dekker's normalisation)
// ---------------------------------------------------------------------------
__device__ __forceinline__ ff ff_add(ff a, float b) {
    const float s = __fadd_rn(a.hi, b);
    const float bb = __fsub_rn(s, a.hi);
    const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    const float lo = __fadd_rn(a.lo, err);
    const float hi = __fadd_rn(s, lo);
    return {hi, __fsub_rn(lo, __fsub_rn(hi, s))};
}
// Knuth's two-sum: a + b = s + err exactly
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}
// compensated pair + compensated pair (normalised)
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    float e;
    const float s = two_sum(a.hi, b.hi, e);
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    const float hi = __fadd_rn(s, e);
    return {hi, __fsub_rn(e, __fsub_rn(hi, s))};
}
// (p1 - p0)(p1 + p0) of two floats as hi + lo, to a few units of 2^-46 of
// its size: both factors by two-sum, their leading product by the FMA
// two-product (its rounding error exactly), the cross terms in float.
__device__ __forceinline__ float diff_of_squares(float p1, float p0, float& lo) {
    float ea, eb;
    const float a = two_sum(p1, -p0, ea);
    const float b = two_sum(p1, p0, eb);
    const float h = __fmul_rn(a, b);
    lo = __fadd_rn(__fmaf_rn(a, b, -h), __fadd_rn(__fmul_rn(a, eb), __fmul_rn(ea, b)));
    return h;
}
__device__ __forceinline__ double eps_value(double e) { return e; }
__device__ __forceinline__ double eps_value(ff e) { return (double)e.hi + (double)e.lo; }
__device__ __forceinline__ void eps_from(double v, double& e) { e = v; }
__device__ __forceinline__ void eps_from(double v, ff& e) {
    e.hi = (float)v;
    e.lo = (float)(v - (double)e.hi);
}
__device__ __forceinline__ double eps_add(double e, double d) { return e + d; }
__device__ __forceinline__ ff eps_add(ff e, float d) { return ff_add(e, d); }

// Per-replica constants (one independent periodic system each).
struct RepInfo {
    double L[3];     // box lengths
    double ell[3];   // cell size L_d / ncell_d
    double s[3];     // ncell_d / L_d
    float ellf[3];
    int nc[3];       // cells per axis
    int k[3];        // cells per brick per axis
    int B[3];        // bricks (Hybrid domains) per axis
    int cell_off;    // first global cell index of the replica
    int ncells;
    int part_off;    // first particle slot of the replica
    int n;
    int brick_off;   // first global brick index of the replica
    int tab_off;     // offset of the replica's cell tables
    double cv;       // C_v
    float cvf;
    int walls;       // 1: specular walls along z (not periodic along z)
    double wall_u;   // velocity of the upper wall along z (walls = 1)
};

// Position of the upper wall of a walled replica for the current step's
// drift, as a cell index and an offset in it: z_w = c ell_z + o.
struct WallPos {
    double o;
    int c;
    int pad;
};

// Cell tables of a replica, at tab_off: lin_x[nc0] | lin_y[nc1] | lin_z[nc2]
// | brick_x[nc0] | brick_y[nc1] | brick_z[nc2]. The brick-major linear cell
// index is cell_off + lin_x[cx] + lin_y[cy] + lin_z[cz]; brick_d[c] = c / k_d.
__device__ __forceinline__ int cell_index(const int* __restrict__ tab, const RepInfo& R, int cx,
                                          int cy, int cz) {
    const int* t = tab + R.tab_off;
    return R.cell_off + __ldg(t + cx) + __ldg(t + R.nc[0] + cy) + __ldg(t + R.nc[0] + R.nc[1] + cz);
}
__device__ __forceinline__ const int* brick_tab(const int* __restrict__ tab, const RepInfo& R) {
    return tab + R.tab_off + R.nc[0] + R.nc[1] + R.nc[2];
}

__device__ __forceinline__ int pack_cell(int cx, int cy, int cz) { return cx | (cy << 10) | (cz << 20); }
__device__ __forceinline__ int cell_x(int c) { return c & 1023; }
__device__ __forceinline__ int cell_y(int c) { return (c >> 10) & 1023; }
__device__ __forceinline__ int cell_z(int c) { return (c >> 20) & 1023; }

template <class T> __device__ __forceinline__ T cell_len(const RepInfo& R, int d);
template <> __device__ __forceinline__ double cell_len<double>(const RepInfo& R, int d) { return R.ell[d]; }
template <> __device__ __forceinline__ float cell_len<float>(const RepInfo& R, int d) { return R.ellf[d]; }

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds; each round
// multiplies counter words 0 and 2 by the two round constants, keeps the full
// 64-bit products, and xors the high halves with words 1 / 3 and the key;
// the key is advanced by the two Weyl constants before every later round.
// ---------------------------------------------------------------------------
//
// The ten round keys of a handle's seed are launch constants (kernel
// parameters): bumping the key in every draw was 18 of its ~300 instructions.
// tab: the tables of the double-precision Gaussians (gauss_tables).
struct PhiloxKeys {
    uint32_t x[10], y[10];
    const double2* tab;
};

__host__ __device__ __forceinline__ PhiloxKeys philox_keys(uint2 k, const double2* tab = nullptr) {
    PhiloxKeys K;
    K.tab = tab;
    for (int r = 0; r < 10; ++r) {
        K.x[r] = k.x + (uint32_t)r * 0x9E3779B9u;
        K.y[r] = k.y + (uint32_t)r * 0xBB67AE85u;
    }
    return K;
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const PhiloxKeys& K) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ K.x[r], lo1, hi0 ^ c.w ^ K.y[r], lo0);
    }
    return c;
}

template <class T> struct T3 { T x, y, z; };

// Box-Muller on 24-bit uniforms u in (0, 1] and t in [0, 1) (exact in float):
// G = (R1 cos 2 pi t1, R1 sin 2 pi t1, R2 cos 2 pi t2), R = sqrt(-2 ln u).
__device__ __forceinline__ T3<float> gauss3(uint4 x, const double2*, float) {
    const float u1 = (float)((x.x >> 8) + 1u) * 0x1p-24f;
    const float t1 = (float)(x.y >> 8) * 0x1p-24f;
    const float u2 = (float)((x.z >> 8) + 1u) * 0x1p-24f;
    const float t2 = (float)(x.w >> 8) * 0x1p-24f;
    const float R1 = sqrtf(-2.0f * logf(u1));
    const float R2 = sqrtf(-2.0f * logf(u2));
    float s1, c1;
    sincospif(2.0f * t1, &s1, &c1);
    const float c2 = cospif(2.0f * t2);
    return {R1 * c1, R1 * s1, R2 * c2};
}

// In double the chip does two operations a clock and SM, so their count is the
// time (log, sincospi and cospi were ~120 of a draw's): both functions are
// table-driven (P. T. P. Tang, ACM TOMS 15 (1989) and 16 (1990)), which the
// 24-bit arguments suit.
//   -2 ln(K / 2^24): K = 2^e m, m in [1, 2) in 512 intervals with reciprocals
//     c of 26 bits, so that r = m c - 1, |r| < 2^-9, is exact; the sum of
//     -2 E ln 2 and -2 L (L = -ln c, less ln 2 from sqrt(2) on, where E counts
//     one more) is exact in the tables' high parts, multiples of 2^-42.
//   angle 2 pi T / 2^24: folded to an eighth of a turn, 512 steps, and the
//     Taylor series of sine and cosine for the rest, at most 7.7e-4.
// Errors of ln, cos and sin: 1 to 2 ulp, as CUDA's. Us per pass in FP64: ten
// Hybrid steps of 1,000 particles 5445 -> 5024, two of 108,000 2183 -> 2030.
constexpr int GT_TRIG = 0, GT_TRIG_N = 513;             // (cos, sin)
constexpr int GT_EXP = GT_TRIG + GT_TRIG_N, GT_EXP_N = 25;   // (high, low) of 2 (24 - E) ln 2, E = 0..24
constexpr int GT_LOG = GT_EXP + GT_EXP_N, GT_LOG_N = 512;    // (c, high), (low, 0)
constexpr int GT_SIZE = GT_LOG + 2 * GT_LOG_N;
constexpr int GT_FOLD = 212;                             // first interval beyond sqrt(2)

// the tables, built on the host once (0.7 ms where long double is software)
inline std::vector<double2> make_gauss_tables() {
    std::vector<double2> t(GT_SIZE);
    const long double pi = 3.14159265358979323846264338327950288L, ln2 = std::log(2.0L);
    auto split = [](long double x) {
        const double hi = (double)(std::nearbyint(x * 0x1p42L) * 0x1p-42L);
        return make_double2(hi, (double)(x - (long double)hi));
    };
    for (int i = 0; i < GT_TRIG_N; ++i)
        t[GT_TRIG + i] = make_double2((double)std::cos(pi * i / 2048), (double)std::sin(pi * i / 2048));
    for (int e = 0; e < GT_EXP_N; ++e) t[GT_EXP + e] = split(2 * (24 - e) * ln2);
    for (int i = 0; i < GT_LOG_N; ++i) {
        // c = 1 and 1/2 at the ends, so that ln 1 = 0 is met without cancellation
        const double c = i == 0 ? 1.0 : (i == GT_LOG_N - 1 ? 0.5 : std::nearbyint(0x1p26 / (1.0 + (i + 0.5) / 512)) * 0x1p-26);
        const double2 l = split(2 * std::log((long double)c * (i < GT_FOLD ? 1 : 2)));
        t[GT_LOG + 2 * i] = make_double2(c, l.x);
        t[GT_LOG + 2 * i + 1] = make_double2(l.y, 0.0);
    }
    return t;
}
inline const std::vector<double2>& gauss_tables() {
    static const std::vector<double2> t = make_gauss_tables();
    return t;
}

__device__ __forceinline__ double neg2_log24(uint32_t K, const double2* __restrict__ tab) {   // 1 <= K <= 2^24
    const uint32_t f = __float_as_uint((float)K);   // exact
    const uint32_t mant = f & 0x7fffffu, i = mant >> 14;
    const int E = (int)(f >> 23) - 127 + (i >= (uint32_t)GT_FOLD ? 1 : 0);
    const double m = __hiloint2double((int)(0x3ff00000u | (mant >> 3)), (int)(mant << 29));
    const double2 a = tab[GT_LOG + 2 * i], x = tab[GT_EXP + E];
    const double lo = tab[GT_LOG + 2 * i + 1].x + x.y;
    const double r = fma(m, a.x, -1.0);
    double q = fma(r, 2.0 / 6, -2.0 / 5);   // -2 log1p(r) / r
    q = fma(r, q, 2.0 / 4);
    q = fma(r, q, -2.0 / 3);
    q = fma(r, q, 1.0);
    q = fma(r, q, -2.0);
    return (x.x + a.y) + fma(r, q, lo);
}

// cos and sin of 2 pi T / 2^24, T < 2^24
__device__ __forceinline__ double2 cos_sin24(uint32_t T, const double2* __restrict__ tab) {
    const uint32_t quad = T >> 22;
    uint32_t f = T & 0x3fffffu;
    const bool fold = f > 0x200000u;   // beyond 45 degrees: the complement
    f = fold ? 0x400000u - f : f;
    const uint32_t i = (f + 2048u) >> 12;
    const double2 a = tab[GT_TRIG + i];
    // times 2 pi / 2^24 in two parts, the first of 40 bits: an exact product
    const double n = (double)((int)f - (int)(i << 12)), b = fma(n, 0x1.a308d313198a3p-63, n * 0x1.921fb54442000p-22);
    const double b2 = b * b;
    const double sb = fma(b * b2, fma(b2, 1.0 / 120, -1.0 / 6), b);
    const double cb = b2 * fma(b2, 1.0 / 24, -0.5);   // cos b - 1
    double c = fma(-a.y, sb, fma(a.x, cb, a.x));
    double s = fma(a.x, sb, fma(a.y, cb, a.y));
    const bool swap = fold != ((quad & 1) != 0);   // odd quadrants: (cos, sin) -> (-sin, cos)
    const double c1 = swap ? s : c, s1 = swap ? c : s;
    return make_double2(quad == 1 || quad == 2 ? -c1 : c1, quad >= 2 ? -s1 : s1);
}

__device__ __forceinline__ T3<double> gauss3(uint4 x, const double2* __restrict__ tab, double) {
    const double R1 = sqrt(neg2_log24((x.x >> 8) + 1u, tab));
    const double R2 = sqrt(neg2_log24((x.z >> 8) + 1u, tab));
    const double2 t1 = cos_sin24(x.y >> 8, tab);
    return {R1 * t1.x, R1 * t1.y, R2 * cos_sin24(x.w >> 8, tab).x};
}

// G_ij for particle i (id_i) and neighbour j (id_j): drawn for the ordered
// pair (min id, max id) and negated when id_i > id_j, so G_ji = -G_ij.
template <class T>
__device__ __forceinline__ T3<T> pair_gauss(const PhiloxKeys& key, uint32_t step, uint32_t rep, uint32_t id_i,
                                            uint32_t id_j) {
    const bool lo = id_i < id_j;
    const uint4 x = philox4x32_10(make_uint4(lo ? id_i : id_j, lo ? id_j : id_i, step, rep), key);
    T3<T> g = gauss3(x, key.tab, T(0));
    if (!lo) {
        g.x = -g.x;
        g.y = -g.y;
        g.z = -g.z;
    }
    return g;
}

// ---------------------------------------------------------------------------
// Pair potential: the soft repulsion v = (a r_c/2)(1 - r/r_c)^2, or the
// shifted, splined, truncated Lennard-Jones potential of Eq. (Ep),
// v = 4 eps((r_LJ/r)^12 - (r_LJ/r)^6) - eps_sh - f_sp (r - r_c) with eps_sh =
// v_LJ(r_c), f_sp = v_LJ'(r_c) so that v(r_c) = v'(r_c) = 0.
// ---------------------------------------------------------------------------
template <class T> struct PotT {
    int kind;                       // DPDE_POT_SOFT or DPDE_POT_LJ
    T a, rc, inv_rc, half_arc;      // soft: a, r_c, 1/r_c, a r_c / 2
    T lj4e, ljr2, ljesh, ljfsp;     // LJ: 4 eps, r_LJ^2, eps_sh, f_sp
};

// For 0 < r2 < r_c^2 and ir = 1/sqrt(r2): v(r), fr = -v'(r)/r (so that the
// force on i is fr (q_i - q_j)) and lap = v''(r) + 2 v'(r)/r.
template <class T>
__device__ __forceinline__ void pair_pot_soft(const PotT<T>& P, T r2, T ir, T& v, T& fr, T& lap) {
    const T w = T(1) - r2 * ir * P.inv_rc;
    v = P.half_arc * w * w;
    fr = P.a * w * ir;
    lap = P.a * P.inv_rc - T(2) * P.a * w * ir;
}
template <class T>
__device__ __forceinline__ void pair_pot(const PotT<T>& P, T r2, T ir, T& v, T& fr, T& lap) {
    const T r = r2 * ir;
    if (P.kind == 1) {
        const T ir2 = ir * ir;
        const T s2 = P.ljr2 * ir2, s6 = s2 * s2 * s2, s12 = s6 * s6;
        const T dv = P.lj4e * (T(6) * s6 - T(12) * s12) * ir - P.ljfsp;
        v = P.lj4e * (s12 - s6) - P.ljesh - P.ljfsp * (r - P.rc);
        fr = -dv * ir;
        lap = P.lj4e * (T(156) * s12 - T(42) * s6) * ir2 + T(2) * dv * ir;
    } else {
        pair_pot_soft(P, r2, ir, v, fr, lap);
    }
}

// Constants of the pair potential from the parameters (host side, double).
inline PotT<double> make_pot(int kind, double a, double rc, double lj_eps, double lj_r) {
    PotT<double> P{};
    P.kind = kind;
    P.a = a;
    P.rc = rc;
    P.inv_rc = 1.0 / rc;
    P.half_arc = 0.5 * a * rc;
    if (kind == 1) {
        const double s6 = std::pow(lj_r / rc, 6.0), s12 = s6 * s6;
        P.lj4e = 4.0 * lj_eps;
        P.ljr2 = lj_r * lj_r;
        P.ljesh = 4.0 * lj_eps * (s12 - s6);                  // v_LJ(r_c)
        P.ljfsp = 4.0 * lj_eps * (6.0 * s6 - 12.0 * s12) / rc;  // v_LJ'(r_c)
    }
    return P;
}

template <class T> inline PotT<T> cast_pot(const PotT<double>& P) {
    return PotT<T>{P.kind, (T)P.a, (T)P.rc, (T)P.inv_rc, (T)P.half_arc, (T)P.lj4e, (T)P.ljr2, (T)P.ljesh, (T)P.ljfsp};
}

// v at r = 0: the soft potential's maximum; no LJ term
template <class T>
__device__ __forceinline__ T pair_pot_at_zero(const PotT<T>& P) { return P.kind == 1 ? T(0) : P.half_arc; }

// Status bits raised by the kernels (read and cleared by the host).
enum : unsigned int {
    ST_NEG_EPS = 1u, ST_NONFINITE = 2u, ST_CAPACITY = 4u, ST_DOMAIN = 8u, ST_WALL = 16u, ST_TIMEOUT = 32u
};

}  // namespace dpde
