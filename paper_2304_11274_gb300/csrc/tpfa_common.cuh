// tpfa_common.cuh -- device-side building blocks shared by the TPFA kernels.
//
// Physics (arXiv 2304.11274, Section 3): Eq. density for rho(p), Eq. flux-calc
// for the two-point flux with single-point upwinding, Eq. vk for the
// accumulation term.  Every link function here is written with explicit
// round-to-nearest intrinsics so that the naive, tiled and batched kernels,
// whichever cell computes a link, produce bit-identical values.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tpfa_grid.h"

namespace tpfa {

// ---------------------------------------------------------------- geometry

// Links of cell index i along an axis of n cells: to i-1 and to i+1.
__host__ __device__ __forceinline__ int axis_links(int i, int n) { return (i > 0) + (i < n - 1); }

// Links from all cells i' < i along an axis of n cells.
__host__ __device__ __forceinline__ long long axis_links_before(int i, int n) {
    return (long long)(i > 1 ? i - 1 : 0) + (i < n - 1 ? i : n - 1);
}

// CSR offset of the first entry of row (i, j, k).  A row holds the cell
// itself and adj(K) (Section 5.1), so its length is
//   1 + ex(i) + ey(j) + ez(k) + diag * ex(i) * ey(j);
// summing that over all cells before (i, j, k) in x-fastest order gives this
// closed form, so the kernels never read row_ptr.
__host__ __device__ __forceinline__ long long row_start(const GridGeom& g, int i, int j, int k) {
    const long long nx = g.nx, ny = g.ny;
    const long long Ex = 2 * (nx - 1), Ey = 2 * (ny - 1);
    const long long D = g.diag;
    const long long plane = nx * ny + Ex * ny + nx * Ey + D * Ex * Ey;
    const int ez = axis_links(k, g.nz), ey = axis_links(j, g.ny);
    long long s = (long long)k * plane + nx * ny * axis_links_before(k, g.nz);
    s += (long long)j * (nx + Ex + nx * ez) + axis_links_before(j, g.ny) * (nx + D * Ex);
    s += (long long)i * (1 + ey + ez) + axis_links_before(i, g.nx) * (1 + D * ey);
    return s;
}

__host__ __device__ __forceinline__ long long total_nnz(const GridGeom& g) {
    return row_start(g, 0, 0, g.nz);
}

__host__ __device__ __forceinline__ int row_length(const GridGeom& g, int i, int j, int k) {
    const int ex = axis_links(i, g.nx), ey = axis_links(j, g.ny), ez = axis_links(k, g.nz);
    return 1 + ex + ey + ez + g.diag * ex * ey;
}

// ---------------------------------------------------------------- FP32 -> FP64

// Exact widening of a float to a double done on the integer pipe.  On GB300
// the float->double convert instruction issues on the FP64 unit (about two
// per clock per SM), which the mixed kernels cannot afford per link; this
// rebuilds the IEEE-754 binary64 bit pattern of normal numbers and zeros
// (sign kept, exponent rebiased by 1023 - 127 = 896, 23-bit fraction moved up
// by 29 bits) and leaves subnormals, infinities and NaNs to the hardware.
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t a = u & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u) {  // normal: 0x00800000 <= a < 0x7f800000
        const uint32_t hi = ((a >> 3) + 0x38000000u) | (u & 0x80000000u);
        return __hiloint2double((int)hi, (int)(u << 29));
    }
    if (a == 0u) return __hiloint2double((int)u, 0);  // signed zero
    return (double)x;
}

// Narrowing of a finite, normal-range double to a float by truncating the
// fraction (error below one float ulp), on the integer pipe.  Used only where
// the value is a small additive term of a compensated FP32 sum.
__device__ __forceinline__ float narrow_rz(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const uint32_t lo = (uint32_t)__double2loint(x);
    const uint32_t ex = (hi >> 20) & 0x7ffu;
    if (ex > 896u && ex < 1151u) {
        const uint32_t f = ((hi & 0x000fffffu) << 3) | (lo >> 29);
        return __uint_as_float((hi & 0x80000000u) | ((ex - 896u) << 23) | f);
    }
    return (float)x;
}

// The two conversions above without the conversion instruction: it is
// predicated, not jumped over, and takes its time on the FP64 pipe even when no
// lane needs it.  Measured without it: the two-cell assembly at 512 x 512 x 256
// 1430 -> 1378 us, an ensemble of 20 models 1692 -> 1624 us.
//   narrow_flush, widen_flush: |x| < 2^128; what would be or is an FP32
//     subnormal gives zero;
//   narrow_any: every x, with the bits of narrow_rz (NaN payloads aside); the
//     rare values by integer operations behind a branch.
__device__ __forceinline__ float narrow_flush(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const uint32_t lo = (uint32_t)__double2loint(x);
    const uint32_t a = hi & 0x7fffffffu;
    const uint32_t f = ((a - 0x38000000u) << 3) | (lo >> 29);
    return __uint_as_float((hi & 0x80000000u) | (a >= 0x38100000u ? f : 0u));
}
// The same for any x: from 2^128 on an infinity or NaN.
__device__ __forceinline__ float narrow_sat(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const uint32_t a = min(hi & 0x7fffffffu, 0x47f00000u);
    const uint32_t f = ((a - 0x38000000u) << 3) | ((uint32_t)__double2loint(x) >> 29);
    return __uint_as_float((hi & 0x80000000u) | (a >= 0x38100000u ? f : 0u));
}
// Magnitude bits of (float)x for |x| outside [2^-126, 2^128), from its words.
__device__ __forceinline__ uint32_t narrow_rare(uint32_t a, uint32_t lo) {
    if (a >= 0x47f00000u) return a > 0x7ff00000u || (a == 0x7ff00000u && lo) ? 0x7fc00000u : 0x7f800000u;
    // units of 2^-149, rounded to nearest even: x = m 2^-149 / 2^s
    const int s = 926 - (int)(a >> 20);
    if (s > 53) return 0u;
    const uint64_t m = ((uint64_t)((a & 0x000fffffu) | 0x00100000u) << 32) | lo;
    const uint64_t rest = m & ((1ull << s) - 1u), half = 1ull << (s - 1);
    const uint32_t n = (uint32_t)(m >> s);
    return n + (rest > half || (rest == half && (n & 1u)));
}
__device__ __forceinline__ float narrow_any(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const uint32_t lo = (uint32_t)__double2loint(x);
    const uint32_t a = hi & 0x7fffffffu;
    uint32_t f = a ? ((a - 0x38000000u) << 3) | (lo >> 29) : 0u;
    if (a - 0x38100000u >= 0x0fe00000u && a) f = narrow_rare(a, lo);
    return __uint_as_float((hi & 0x80000000u) | f);
}
__device__ __forceinline__ double widen_flush(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint32_t a = u & 0x7fffffffu;
    const bool n = a >= 0x00800000u;
    const uint32_t hi = (n ? (a >> 3) + 0x38000000u : 0u) | (u & 0x80000000u);
    return __hiloint2double((int)hi, n ? (int)(u << 29) : 0);
}
__device__ __forceinline__ bool finite_f32(float x) { return fabsf(x) < __int_as_float(0x7f800000); }
// Below kSubnormal: x is subnormal (twice its bits: no sign; zero wraps round).
constexpr uint32_t kSubnormal = 2u * 0x007fffffu;
__device__ __forceinline__ uint32_t sub_word(float x) { return 2u * __float_as_uint(x) - 2u; }

__device__ __forceinline__ float rcp_approx(float x) {  // 1/x within 2^-23
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// A double as an unevaluated FP32 pair v = hi + lo (hi the truncation of v,
// lo the exact remainder narrowed; |lo| < ulp(hi)), so differences of nearby
// values can be formed in FP32: (hi_a - hi_b) + (lo_a - lo_b) is accurate to
// a few float ulps of a - b itself (hi_a - hi_b is exact when a and b are
// within a factor of two).
struct F2Split {
    float hi, lo;
};
__device__ __forceinline__ F2Split split_f2(double v) {
    F2Split r;
    r.hi = narrow_rz(v);
    r.lo = narrow_rz(__dadd_rn(v, -widen(r.hi)));
    return r;
}

// a - b for two split doubles, in FP32.
__device__ __forceinline__ float diff_f2(const F2Split& a, const F2Split& b) {
    return __fadd_rn(__fsub_rn(a.hi, b.hi), __fsub_rn(a.lo, b.lo));
}

// Distance over area of each link direction, the geometric factor of the
// two-point transmissibility (x faces, y faces, z faces, in-plane diagonals).
struct LinkGeo {
    float cx, cy, cz, cd;
};
struct LinkGeoD {
    double cx, cy, cz, cd;
};

// ---------------------------------------------------------------- Kahan

struct Kahan32 {
    float s = 0.f, c = 0.f;  // running sum and compensation; value = s - c
    __device__ __forceinline__ void add(float x) {
        const float y = __fsub_rn(x, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
};

// ---------------------------------------------------------------- cell state

template <typename T>
struct CellVal {
    T p, z, rho, drho;  // pressure, depth, density, d rho / dp
};
// The FP64 path carries the mobility rho / mu instead of the density (one
// product per cell instead of one per link); its derivative c_f rho / mu
// only appears inside the link.
template <>
struct CellVal<double> {
    double p, z, lam;  // pressure, depth, rho / mu
};

struct PhysF {
    float rho_ref, p_ref, c_f, inv_mu, g, half_g, V_dt, c_r;
};
// FP64 constants, combined once on the host.
struct PhysD {
    double p_ref, c_f;
    double lam_ref;  // rho_ref / mu
    double hg, chg;  // g mu / 2 and c_f g mu / 2: (rho_a + rho_b) g / 2 = (lam_a + lam_b) hg
    double vol;      // (V/dt) mu
    double vol_cr;   // (V/dt) mu c_r
    double cc, cs;   // c_f c_r and c_f + c_r
};
inline PhysD make_phys_d(double rho_ref, double p_ref, double c_f, double mu, double g, double V_dt, double c_r) {
    PhysD q;
    q.p_ref = p_ref, q.c_f = c_f;
    q.lam_ref = rho_ref / mu;
    q.hg = 0.5 * g * mu, q.chg = c_f * (0.5 * g * mu);
    q.vol = V_dt * mu, q.vol_cr = V_dt * mu * c_r;
    q.cc = c_f * c_r, q.cs = c_f + c_r;
    return q;
}

// exp(x) and expm1(x) in FP64 for the small arguments the state equation
// meets (|x| < 2^-5: c_f (p - p_ref) with c_f ~ 1e-9 / Pa and pressures
// within tens of MPa of p_ref) by their Taylor series, cut after x^8 (exp)
// and x^9 (expm1): the remainder is below 2^-60 of the value, so the result
// is the function's within the few roundings of the Horner steps.  Larger
// arguments (and NaN or infinity) take exp() / expm1().  The FP64 path is
// bound by the FP64 pipe (two operations per clock per multiprocessor), and
// these series need fewer FP64 instructions per call; smaller arguments still
// fewer: below 2^-6 the terms of exp from x^5 / 5! on are less than 2^-36 of
// the value, so their sum over x^5 is taken in FP32 (its error stays below
// 2^-59 of the value) and five FP64 operations remain of eight; below 2^-10 the
// terms of expm1 from x^4 / 4! on are less than 2^-34 of it, and four of ten
// remain.  Against 80-bit values over 4 million arguments of each binade the errors
// are those of the all-FP64 series to four digits in the mean (exp 5.05e-17, expm1
// 6.80e-17 rms) and below 2^-8 in the largest (1.11e-16, 2.20e-16); at 2^-6 exp's
// largest is 1.116e-16.  The range tests read the high word (integer pipe).
__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ double exp_fp64(double x) {
    const uint32_t a = abs_hi(x);
    double r;
    if (a < 0x3f900000u) {  // |x| < 2^-6
        const float xf = narrow_flush(x);
        const float t = __fmaf_rn(__fmaf_rn(xf, 1.f / 5040.f, 1.f / 720.f), xf, 1.f / 120.f);
        r = __fma_rn(widen_flush(t), x, 1.0 / 24.0);
    } else if (a < 0x3fa00000u) {  // |x| < 2^-5
        r = 1.0 / 40320.0;  // 1/8!
        r = __fma_rn(r, x, 1.0 / 5040.0);
        r = __fma_rn(r, x, 1.0 / 720.0);
        r = __fma_rn(r, x, 1.0 / 120.0);
        r = __fma_rn(r, x, 1.0 / 24.0);
    } else {
        return exp(x);
    }
    r = __fma_rn(r, x, 1.0 / 6.0);
    r = __fma_rn(r, x, 0.5);
    r = __fma_rn(r, x, 1.0);
    return __fma_rn(r, x, 1.0);
}
__device__ __forceinline__ double expm1_fp64(double x) {
    const uint32_t a = abs_hi(x);
    double r;
    if (a < 0x3f500000u) {  // |x| < 2^-10
        const float t = __fmaf_rn(narrow_flush(x), 1.f / 120.f, 1.f / 24.f);
        r = __fma_rn(widen_flush(t), x, 1.0 / 6.0);
    } else if (a < 0x3fa00000u) {  // |x| < 2^-5
        r = 1.0 / 362880.0;  // 1/9!: expm1(x) = x (1 + x/2! + x^2/3! + ... + x^8/9!)
        r = __fma_rn(r, x, 1.0 / 40320.0);
        r = __fma_rn(r, x, 1.0 / 5040.0);
        r = __fma_rn(r, x, 1.0 / 720.0);
        r = __fma_rn(r, x, 1.0 / 120.0);
        r = __fma_rn(r, x, 1.0 / 24.0);
        r = __fma_rn(r, x, 1.0 / 6.0);
    } else {
        return expm1(x);
    }
    r = __fma_rn(r, x, 0.5);
    r = __fma_rn(r, x, 1.0);
    return __dmul_rn(r, x);
}

// Eq. density: rho = rho_ref exp(c_f (p - p_ref)), and its derivative.
__device__ __forceinline__ CellVal<float> make_cell(const PhysF& q, float p, float z) {
    CellVal<float> c;
    c.p = p;
    c.z = z;
    c.rho = __fmul_rn(q.rho_ref, expf(__fmul_rn(q.c_f, __fsub_rn(p, q.p_ref))));
    c.drho = __fmul_rn(q.c_f, c.rho);
    return c;
}
__device__ __forceinline__ CellVal<double> make_cell(const PhysD& q, double p, double z) {
    CellVal<double> c;
    c.p = p;
    c.z = z;
    c.lam = __dmul_rn(q.lam_ref, exp_fp64(__dmul_rn(q.c_f, __dsub_rn(p, q.p_ref))));
    return c;
}

// ---------------------------------------------------------------- one link

template <typename T>
struct LinkOut {
    T F;   // F_ab: mass outflow from a to b
    T Da;  // dF_ab / dp_a
    T Db;  // dF_ab / dp_b
};
// FP64 path: also the gravity parts, which the sums below need.
template <>
struct LinkOut<double> {
    double F, Da, Db;
    double u, rs;  // T lam_up c_f (g mu / 2)(z_a - z_b) and lam_a + lam_b
};

// Two-point flux of Eq. flux-calc seen from row a (z = depth, positive down):
//   dPhi = (p_a - p_b) - rho_avg g (z_a - z_b)
//   upstream = a if dPhi > 0 else b,  F = T (rho_up / mu) dPhi
// and its two pressure derivatives.  rho_avg g dz is formed as
// (rho_a + rho_b)(g/2 dz): halving is exact, so the fused product equals
// the one of rho_avg and g dz bit for bit, with two multiplications fewer;
// T/mu is formed once and scales both rho_up and dPhi.  Negating every input
// that changes sign between the two ends of a link negates every output, so
// F_ba = -F_ab exactly (except the derivatives at an exact tie dPhi == 0,
// where each end takes the other cell as upstream).
__device__ __forceinline__ LinkOut<float> link(const PhysF& q, float T, const CellVal<float>& a,
                                               const CellVal<float>& b) {
    const float dp = __fsub_rn(a.p, b.p);
    const float hgdz = __fmul_rn(q.half_g, __fsub_rn(a.z, b.z));
    const float dphi = __fmaf_rn(-__fadd_rn(a.rho, b.rho), hgdz, dp);
    const bool up_a = dphi > 0.f;
    const float Tm = __fmul_rn(T, q.inv_mu);
    const float Tl = __fmul_rn(Tm, up_a ? a.rho : b.rho);
    const float w = __fmul_rn(Tm, dphi);
    LinkOut<float> r;
    r.F = __fmul_rn(Tl, dphi);
    const float dda = __fmaf_rn(-a.drho, hgdz, 1.f);
    const float ddb = __fmaf_rn(-b.drho, hgdz, -1.f);
    r.Da = __fmaf_rn(Tl, dda, up_a ? __fmul_rn(a.drho, w) : 0.f);
    r.Db = __fmaf_rn(Tl, ddb, up_a ? 0.f : __fmul_rn(b.drho, w));
    return r;
}

// FP64: the same flux with the mobility lam = rho / mu,
//   F = T lam_up dPhi,  dF/dp_a =  T lam_up (1 - c_f lam_a hg dz) + [up = a] c_f F
//                       dF/dp_b = -T lam_up (1 + c_f lam_b hg dz) + [up = b] c_f F
// (d lam / dp = c_f lam, so the mobility's term is c_f F).  Cells at one depth
// have no gravity terms: FLAT leaves them out, which gives the same bits as
// evaluating them with dz = 0 (a sum with an exact zero), so a kernel may
// choose it for any set of links that link_flat() admits.
template <bool FLAT>
__device__ __forceinline__ LinkOut<double> link_d(const PhysD& q, double T, const CellVal<double>& a,
                                                  const CellVal<double>& b) {
    LinkOut<double> r;
    double dphi = __dsub_rn(a.p, b.p);
    double dz = 0.0;
    r.rs = 0.0;
    if (!FLAT) {
        dz = __dsub_rn(a.z, b.z);
        r.rs = __dadd_rn(a.lam, b.lam);
        dphi = __fma_rn(-r.rs, __dmul_rn(q.hg, dz), dphi);
    }
    // dphi > 0 on the integer pipe: positive, not zero, not NaN
    const long long bits = __double_as_longlong(dphi);
    const bool up_a = bits > 0 && bits <= 0x7ff0000000000000ll;
    const double Tl = __dmul_rn(T, up_a ? a.lam : b.lam);
    r.F = __dmul_rn(Tl, dphi);
    r.u = 0.0;
    double da = Tl, db = -Tl;
    if (!FLAT) {
        r.u = __dmul_rn(__dmul_rn(q.chg, dz), Tl);
        da = __fma_rn(-r.u, a.lam, Tl);
        db = -__fma_rn(r.u, b.lam, Tl);
    }
    r.Da = __fma_rn(q.c_f, up_a ? r.F : 0.0, da);
    r.Db = __fma_rn(q.c_f, up_a ? 0.0 : r.F, db);
    return r;
}
// Whether FLAT gives the link's bits: equal finite depths and finite mobilities.
__device__ __forceinline__ bool link_flat(const CellVal<double>& a, const CellVal<double>& b) {
    return __double_as_longlong(a.z) == __double_as_longlong(b.z) && abs_hi(a.z) < 0x7ff00000u &&
           abs_hi(a.lam) < 0x7ff00000u && abs_hi(b.lam) < 0x7ff00000u;
}
__device__ __forceinline__ LinkOut<double> link(const PhysD& q, double T, const CellVal<double>& a,
                                                const CellVal<double>& b) {
    return link_d<false>(q, T, a, b);
}
// The link seen from its other end: exact except at a tie dPhi == 0, where
// each end takes the other cell as upstream.
__device__ __forceinline__ LinkOut<double> flip(const LinkOut<double>& l) {
    return LinkOut<double>{-l.F, -l.Db, -l.Da, -l.u, l.rs};
}
// Whether a link may be an exact tie (zero flux; harmlessly also underflow).
__device__ __forceinline__ bool zero_flux(const LinkOut<double>& l) {
    return (__double_as_longlong(l.F) << 1) == 0;
}

// ---------------------------------------------------------------- packed FP32x2
//
// Two links evaluated at once with the FP32x2 instructions of sm_100+ (each
// half rounds exactly like the scalar instruction, so link2() returns, in
// each half, the bits link() returns for that link).

__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

struct Link2 {
    float2 F, Da, Db;  // .x: first link, .y: second link
};

__device__ __forceinline__ Link2 link2(const PhysF& q, float2 T, const CellVal<float>& a, const CellVal<float>& b0,
                                       const CellVal<float>& b1) {
    const float2 dp = __fadd2_rn(f2(a.p), neg2(f2(b0.p, b1.p)));
    const float2 hgdz = __fmul2_rn(f2(q.half_g), __fadd2_rn(f2(a.z), neg2(f2(b0.z, b1.z))));
    const float2 dphi = __ffma2_rn(neg2(__fadd2_rn(f2(a.rho), f2(b0.rho, b1.rho))), hgdz, dp);
    const bool u0 = dphi.x > 0.f, u1 = dphi.y > 0.f;
    const float2 Tm = __fmul2_rn(T, f2(q.inv_mu));
    const float2 Tl = __fmul2_rn(Tm, f2(u0 ? a.rho : b0.rho, u1 ? a.rho : b1.rho));
    const float2 w = __fmul2_rn(Tm, dphi);
    Link2 r;
    r.F = __fmul2_rn(Tl, dphi);
    const float2 dda = __ffma2_rn(neg2(f2(a.drho)), hgdz, f2(1.f));
    const float2 ddb = __ffma2_rn(neg2(f2(b0.drho, b1.drho)), hgdz, f2(-1.f));
    const float2 ta = __fmul2_rn(f2(a.drho), w);
    const float2 tb = __fmul2_rn(f2(b0.drho, b1.drho), w);
    r.Da = __ffma2_rn(Tl, dda, f2(u0 ? ta.x : 0.f, u1 ? ta.y : 0.f));
    r.Db = __ffma2_rn(Tl, ddb, f2(u0 ? 0.f : tb.x, u1 ? 0.f : tb.y));
    return r;
}

// Kahan summation of two independent sums at once (.x and .y), each half
// identical to Kahan32 on its own.  The three subtractions are written as
// fused multiply-adds by -1 (a - b = fma(b, -1, a): the product is exact, so
// the one rounding is the subtraction's).  Written as paired additions of a
// negated operand, they gave sums differing from the scalar Kahan32 by an
// ulp in the two-cell march (found by comparing variants against the naive
// kernel; the fused form matches it bit for bit in every kernel).
struct Kahan2 {
    float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
    __device__ __forceinline__ void add(float2 x) {
        const float2 m1 = make_float2(-1.f, -1.f);
        const float2 y = __ffma2_rn(c, m1, x);
        const float2 t = __fadd2_rn(s, y);
        c = __ffma2_rn(y, m1, __ffma2_rn(s, m1, t));
        s = t;
    }
};

// ---------------------------------------------------------------- accumulation

// expm1(x) in FP32.  The accumulation term's argument c_f (p - p^n) is tiny
// (|x| ~ 1e-4 for a time step's pressure change of 0.1 MPa at c_f = 1e-9 /
// Pa), so below 2^-7 it takes the Taylor series x (1 + x/2 (1 + x/3 (1 +
// x/4))): the first omitted term is x^5 / 120, below 2^-30 of the value, so
// the error is the rounding of three fused multiply-adds and a product (a
// few ulps); larger arguments take expm1f().  Every FP32 kernel calls this,
// so they still agree bit for bit.
__device__ __forceinline__ float expm1_f32(float x) {
    if (fabsf(x) < 0.0078125f) {
        float r = __fmaf_rn(x, 1.f / 24.f, 1.f / 6.f);
        r = __fmaf_rn(x, r, 0.5f);
        r = __fmaf_rn(x, r, 1.f);
        return __fmul_rn(r, x);
    }
    return expm1f(x);
}

// Accumulation term of Eq. vk, A = (V/dt)(phi(p) rho(p) - phi^n rho^n), and
// dA/dp.  With mn = (V/dt) phi(p^n) rho(p^n) precomputed in FP64:
//   phi(p) rho(p) - phi^n rho^n = phi0 c_r (p - p^n) rho(p) + phi^n rho^n expm1(c_f (p - p^n)),
// which forms the small difference without cancellation.
struct AccF {
    double A;  // FP64 accumulation term
    float dA;  // its pressure derivative (a term of the FP32 diagonal sum)
    // PLAIN (below): the least sub_word and the sum of A's FP32 factors
    uint32_t low;
    float all;
};

// expm1 of the accumulation term with its value as a double: in PLAIN rows
// (below) the series' result takes the cheap widening.
template <bool PLAIN>
__device__ __forceinline__ float expm1_wide(float x, double& w) {
    const float r = expm1_f32(x);
    w = PLAIN && fabsf(x) < 0.0078125f ? widen_flush(r) : widen(r);
    return r;
}

template <bool CR, bool PLAIN = false>
__device__ __forceinline__ AccF accumulation(const PhysF& q, float p, float pn, double mn, float rho,
                                             float phi0) {
    const float dpn = __fsub_rn(p, pn);
    AccF r;
    double e64;
    const float e = expm1_wide<PLAIN>(__fmul_rn(q.c_f, dpn), e64);
    r.A = __dmul_rn(mn, e64);
    if (PLAIN) r.low = sub_word(e), r.all = e;
    if (CR) {
        // (V/dt) phi0 c_r (p - p^n) rho(p), and dA = (V/dt)(phi0 c_r rho + phi(p) c_f rho)
        const float vphi = __fmul_rn(q.V_dt, phi0);
        const float g = __fmul_rn(__fmul_rn(vphi, q.c_r), __fmul_rn(dpn, rho));
        r.A = __dadd_rn(r.A, PLAIN ? widen_flush(g) : widen(g));
        if (PLAIN) r.low = min(r.low, sub_word(g)), r.all = __fadd_rn(e, g);
        const float phi_rel = __fmaf_rn(q.c_r, __fsub_rn(p, q.p_ref), 1.f);
        r.dA = __fmul_rn(__fmul_rn(vphi, rho), __fmaf_rn(phi_rel, q.c_f, q.c_r));
    } else {
        // phi = phi0: (V/dt) phi0 rho(p) = mn exp(c_f (p - p^n))
        r.dA = __fmul_rn(__fmul_rn(q.c_f, PLAIN ? narrow_flush(mn) : narrow_any(mn)), __fadd_rn(1.f, e));
    }
    return r;
}

// The marches (PLAIN) form a row's FP64 results, R = (A + s) - c and the
// diagonal s - c, from its compensated FP32 sums (s, c), A = mn expm1(x) and mn
// with the cheap conversions, which are exact for normal values and zero.  Rows
// with another value among them, odd rows, are computed again after the march
// by the naive kernel's row code, as tie rows are, which also reports
// non-finite values.  The tests are on these values themselves, two integer
// instructions each and no branch: sub_word of the sums and of A's factors, one
// finiteness test of their sum, and odd_mass.  A sum that is merely small or zero
// (cells of next to no permeability, no change of pressure) makes no row odd;
// a compensation is subnormal where fluxes are below 1e-31 (k below 1e-43 m^2).
// (Testing the results' size instead, with these tests behind a branch, took
// 3 % of an ensemble's time.)
__device__ __forceinline__ bool odd_mass(double mn) {  // outside FP32's normal range, not zero
    const uint32_t w = 2u * (uint32_t)__double2hiint(mn);
    return w - 2u * 0x38100000u >= 2u * 0x0fe00000u && w != 0u;
}

struct AccD {
    double A, dA;
};

// `lam` is rho(p) / mu.  With c_r == 0, dA = c_f mn exp(c_f (p - p^n)) = c_f (mn + A).
template <bool CR>
__device__ __forceinline__ AccD accumulation(const PhysD& q, double p, double pn, double mn, double lam,
                                             double phi0) {
    const double dpn = __dsub_rn(p, pn);
    const double e = expm1_fp64(__dmul_rn(q.c_f, dpn));
    AccD r;
    r.A = __dmul_rn(mn, e);
    if (CR) {
        r.A = __fma_rn(__dmul_rn(phi0, q.vol_cr), __dmul_rn(dpn, lam), r.A);
        r.dA = __dmul_rn(__dmul_rn(__dmul_rn(phi0, q.vol), lam), __fma_rn(q.cc, __dsub_rn(p, q.p_ref), q.cs));
    } else {
        r.dA = __dmul_rn(q.c_f, __dadd_rn(mn, r.A));
    }
    return r;
}

// Sums of an FP64 row over its links, in slot order.  The diagonal needs no
// term of its own per link: dF/dp_a + dF/dp_b = c_f F - u (lam_a + lam_b), so
//   sum dF/dp_a = -sum dF/dp_b + (c_f sum F - sum u rs),
// the bracket and dA small beside the first sum, which they join last.  (Against
// 80-bit values the diagonals are 2 % closer than with a term per link while
// c_f |dPhi| <= 0.1; the bracket cancels by 1 + c_f |dPhi|, so they are 7 % further
// off at c_f |dPhi| = 1, a density that changes e-fold from cell to cell.)
struct RowAccD {
    double F = 0.0, d = 0.0, grav = 0.0;  // sum F, -sum dF/dp_b, -sum u rs
    template <bool JAC, bool FLAT = false>
    __device__ __forceinline__ void add(const LinkOut<double>& l) {
        F = __dadd_rn(F, l.F);
        if (JAC) d = __dsub_rn(d, l.Db);
        if (!FLAT) grav = __fma_rn(-l.u, l.rs, grav);
    }
    // sum dF/dp_a + sum dF/dp_b + dA, and the row's diagonal dR_K/dp_K
    __device__ __forceinline__ double excess(const PhysD& q, double dA) const {
        return __dadd_rn(__fma_rn(q.c_f, F, grav), dA);
    }
    __device__ __forceinline__ double diagonal(const PhysD& q, double dA) const {
        return __dadd_rn(d, excess(q, dA));
    }
};

// Non-finite test on the integer pipe (exponent all ones).
__device__ __forceinline__ bool nonfinite(double x) {
    return ((uint32_t)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}

}  // namespace tpfa
