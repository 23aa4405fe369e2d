// tpfa_setup.cu -- per-grid and per-time-step setup kernels (not on the
// per-Newton-iteration path): owned transmissibilities, the CSR pattern,
// field conversion and the previous-step mass m^n.
#include <cuda_runtime.h>

#include "tpfa_common.cuh"
#include "tpfa_impl.h"
#include "tpfa_tile.h"

namespace tpfa {

namespace {

constexpr int kThreads = 256;

inline unsigned blocks_for(long long n) {
    long long b = (n + kThreads - 1) / kThreads;
    if (b > (1LL << 30)) b = 1LL << 30;  // grid-stride loops cover the rest
    return (unsigned)(b > 0 ? b : 1);
}

// Two-point transmissibility (the paper names Upsilon_KL without a formula):
// half-transmissibilities k area / (d/2) in series, i.e.
// 2 k_K k_L / (k_K + k_L) * area / d; zero if either cell is impermeable.
__device__ __forceinline__ double two_point(double kK, double kL, double area_over_d) {
    if (!(kK > 0.0) || !(kL > 0.0)) return 0.0;
    return (2.0 * kK * kL / (kK + kL)) * area_over_d;
}

struct Geo {
    double ax, ay, az, ad;  // area / distance of x, y, z faces and of an in-plane diagonal
    float2 px, py, pz, pd;  // twice that as FP32 pairs, zero outside their range
};

// Permeability of cell c: the stored value, or exp of the stored natural
// log (the adjoint's parameterisation, k = exp(ln k)).
template <bool LOG>
__device__ __forceinline__ double perm_at(const double* __restrict__ perm, long long c) {
    return LOG ? exp(perm[c]) : perm[c];
}

// ---- reciprocal permeabilities and links without the FP64 pipe
//
// With r = 1/k the harmonic two-point value is 2 (area/d) / (r_K + r_L), and
// from ln k the reciprocal is one exponential, r = exp(-ln k).  The FP64
// pipe does two operations per clock per multiprocessor, so the first form
// of this kernel (six exponentials and five divisions per cell, all FP64)
// took 638 us from ln k on a 128^3 grid, 33 times its memory traffic.  Here
// a block computes r once per cell of its tile (and its one-cell halo) in
// shared memory; on the mixed path r, the sum and the quotient are FP32
// pairs (value = h + l, about 45 bits), which the FP32 pipe does 64 times
// faster.  The stored FP32 value is accepted only if every number within
// 2^-40 of the pair's value rounds to it (Ziv's rounding test); FP64 rounding
// errors and the pair's own are far below that, so the accepted values are
// those of the FP64 evaluation bit for bit, and the rest (about one link in
// 10^5, and every input outside the pairs' range, zero and NaN included) are
// evaluated by the FP64 formula.

struct Pair32 {
    float h, l;
};
__device__ __forceinline__ Pair32 fast_two_sum(float a, float b) {  // |a| >= |b|
    const float h = __fadd_rn(a, b);
    return {h, __fsub_rn(b, __fsub_rn(h, a))};
}
__device__ __forceinline__ Pair32 pair_mul(Pair32 a, Pair32 b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ Pair32 pair_add(Pair32 a, Pair32 b) {
    const float h = __fadd_rn(a.h, b.h);
    const float t = __fsub_rn(h, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(h, t)), __fsub_rn(b.h, t));
    return {h, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
// c + t s for a constant c with |c| >= |t s|
__device__ __forceinline__ Pair32 pair_step(float c, Pair32 t, Pair32 s) {
    const float p = __fmul_rn(t.h, s.h);
    float e = __fmaf_rn(t.h, s.h, -p);
    e = __fmaf_rn(t.h, s.l, e);
    e = __fmaf_rn(t.l, s.h, e);
    const float h = __fadd_rn(c, p);
    return {h, __fadd_rn(__fsub_rn(p, __fsub_rn(h, c)), e)};
}
// num / d: the quotient h of the leading parts and the remainder over d
__device__ __forceinline__ Pair32 pair_div(Pair32 num, Pair32 d) {
    const float q = rcp_approx(d.h);
    const float h = __fmul_rn(num.h, q);
    const float rem = __fmaf_rn(-h, d.l, __fadd_rn(__fmaf_rn(-h, d.h, num.h), num.l));
    return {h, __fmul_rn(rem, q)};
}
// Pairs are used for magnitudes in [2^-90, 2^90]; NaN fails the test.
__device__ __forceinline__ bool pair_range(float h) { return h >= 0x1p-90f && h <= 0x1p90f; }

// The FP32 value every number within 2^-40 of v (relative) rounds to, or
// false if there is none.
__device__ __forceinline__ bool round_pair(Pair32 v, float& out) {
    const float d = __fmul_rn(v.h, 0x1p-40f);
    const float a = __fadd_rn(v.h, __fadd_rn(v.l, d)), b = __fadd_rn(v.h, __fsub_rn(v.l, d));
    out = a;
    return a == b && pair_range(v.h);
}

constexpr float kNoPair = -1.f;  // h of a cell whose reciprocal has no pair

// 2^(j/8), j = 0..7
__constant__ const double kEighth[8] = {1.0,
                                        1.0905077326652577,
                                        1.1892071150027210,
                                        1.2968395546510096,
                                        1.4142135623730951,
                                        1.5422108254079407,
                                        1.6817928305074290,
                                        1.8340080864093424};

// exp(-x) for |x| < 60: -x = n ln2 / 8 + t, |t| < 0.0434; exp(t) by its Taylor
// series up to t^7 / 7! (the next term is below 2^-51), the terms from t^4 on in
// FP32 (they are below 2^-22 of the sum), the others in pairs; times 2^(n/8).
// `eighth` holds 2^(j/8) as pairs (shared memory).
__device__ __forceinline__ Pair32 split_pair(double v) {
    const float h = narrow_flush(v);
    return {h, narrow_flush(__dadd_rn(v, -widen_flush(h)))};
}
__device__ __forceinline__ Pair32 exp_neg_pair(double x, const float2* eighth) {
    const float nf = rintf(__fmul_rn(narrow_flush(x), -11.541560327111708f));  // -8 / ln 2
    const int n = (int)nf;
    const Pair32 t = split_pair(__fma_rn(widen_flush(-nf), 0.086643397569993164, -x));  // ln 2 / 8
    float u = __fmaf_rn(t.h, 1.f / 5040.f, 1.f / 720.f);
    u = __fmaf_rn(t.h, u, 1.f / 120.f);
    u = __fmaf_rn(t.h, u, 1.f / 24.f);
    constexpr float s6 = (float)(1.0 / 6.0), s6l = (float)(1.0 / 6.0 - (double)s6);
    Pair32 s = fast_two_sum(s6, __fmul_rn(t.h, u));
    s.l = __fadd_rn(s.l, s6l);
    s = pair_step(0.5f, t, s);
    s = pair_step(1.f, t, s);
    s = pair_step(1.f, t, s);
    const float2 e = eighth[n & 7];
    const Pair32 r = pair_mul(s, Pair32{e.x, e.y});
    const float scale = __int_as_float(((n >> 3) + 127) << 23);
    return {__fmul_rn(r.h, scale), __fmul_rn(r.l, scale)};
}

// r = 1/k of cell c as a pair, h = kNoPair where k lies outside the pairs' range.
template <bool LOG>
__device__ __forceinline__ Pair32 recip_pair(double v, const float2* eighth) {
    if (LOG) {
        if (((uint32_t)__double2hiint(v) & 0x7fffffffu) >= 0x404e0000u) return {kNoPair, 0.f};  // |v| >= 60, NaN
        return exp_neg_pair(v, eighth);
    }
    const uint32_t ex = (uint32_t)__double2hiint(v) >> 20;  // sign and exponent
    if (!(ex > 1023u - 90u && ex < 1023u + 90u)) return {kNoPair, 0.f};
    return pair_div(Pair32{1.f, 0.f}, split_pair(v));
}

// num / s in FP64 for s inside the pairs' range: the FP32 reciprocal refined to
// y = 1/s by y (1 + e + e^2), e = 1 - s y (the third-order iteration for the
// reciprocal; e is below 2^-22), then the quotient with its remainder folded
// in once, which rounds it correctly (Markstein's final step).
__device__ __forceinline__ double quotient(double num, double s) {
    const double y0 = widen_flush(rcp_approx(narrow_flush(s)));
    const double e = __fma_rn(-s, y0, 1.0);
    const double y = __fma_rn(y0, __fma_rn(e, e, e), y0);
    const double q = __dmul_rn(num, y);
    return __fma_rn(__fma_rn(-s, q, num), y, q);
}

// What a tile holds per cell: 1/k as a pair (mixed path) or k (FP64 path).
template <typename Real>
struct Tile;
template <>
struct Tile<float> {
    using type = float2;
    template <bool LOG>
    static __device__ __forceinline__ double pre(double v) { return v; }
    template <bool LOG>
    static __device__ __forceinline__ float2 of(double v, const float2* eighth) {
        const Pair32 r = recip_pair<LOG>(v, eighth);
        return make_float2(r.h, r.l);
    }
    // 2 (area/d) / (r_K + r_L); false if the FP64 formula has to decide
    static __device__ __forceinline__ bool link(float2 a, float2 b, float2 ap, double, float& T) {
        if (a.x == kNoPair || b.x == kNoPair) return false;
        return round_pair(pair_div(Pair32{ap.x, ap.y}, pair_add(Pair32{a.x, a.y}, Pair32{b.x, b.y})), T);
    }
};
template <>
struct Tile<double> {
    using type = double;
    template <bool LOG>
    static __device__ __forceinline__ double pre(double v) { return LOG ? exp(v) : v; }
    template <bool LOG>
    static __device__ __forceinline__ double of(double k, const float2*) { return k; }
    // two_point() with the quotient above
    static __device__ __forceinline__ bool link(double a, double b, float2, double area, double& T) {
        const uint32_t ea = (uint32_t)__double2hiint(a) >> 20, eb = (uint32_t)__double2hiint(b) >> 20;
        if (!(min(ea, eb) > 1023u - 90u && max(ea, eb) < 1023u + 90u)) return false;
        T = __dmul_rn(quotient(__dmul_rn(__dadd_rn(a, a), b), __dadd_rn(a, b)), area);
        return true;
    }
};

// Whether the grid still holds the tagged permeability; else counts this launch.
// (The count only grows, so a block that reads it after block 0 has counted
// decides as the others.)
__device__ __forceinline__ bool still_held(const PermTag& tag) {
    if (tag.held && *tag.held == *static_cast<const volatile unsigned long long*>(tag.set)) return true;
    if (tag.set && blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long n = *tag.set + 1;
        *tag.set = n;
        if (tag.take) *tag.take = n;
    }
    return false;
}

// The FP64 formula, a thread per cell: for planes of so few cells that a tile
// of theirs leaves most of its warp idle.  Measured against the tile kernel below
// (us, from k and from ln k): FP64 100000 cells of 1 x 1 planes 64 -> 6 and 269 ->
// 12, 50000 2 x 2 planes, 10 links 152 -> 33 and 254 -> 72, 20000 4 x 4 planes 64 ->
// 49 and 105 -> 106 (8 x 4: 31 and 49, 47 and 107 this way); mixed 1 x 1 planes 41 ->
// 8 and 59 -> 14 (2 x 2: 28 and 37, 27 and 57 this way).
template <typename Real, bool LOG>
__global__ void k_trans_cells(GridGeom g, Geo geo, const double* __restrict__ perm, Real* Tx, Real* Ty, Real* Tz,
                              Real* Tpp, Real* Tmp, Real* kperm, PermTag tag) {
    if (still_held(tag)) return;
    const long long nx = g.nx, nxy = nx * g.ny, N = nxy * g.nz;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
         c += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(c / nxy), j = (int)((c - k * nxy) / nx), i = (int)(c - k * nxy - j * nx);
        const bool xp = i + 1 < g.nx, yp = j + 1 < g.ny;
        const double kc = perm_at<LOG>(perm, c);
        // an absent link's neighbour is the cell itself, so every address is in range
        auto T = [&](bool there, long long d, double a) {
            return there ? (Real)two_point(kc, perm_at<LOG>(perm, there ? d : c), a) : Real(0);
        };
        Tx[c] = T(xp, c + 1, geo.ax);
        Ty[c] = T(yp, c + nx, geo.ay);
        Tz[c] = T(k + 1 < g.nz, c + nxy, geo.az);
        if (g.diag) {
            Tpp[c] = T(xp && yp, c + nx + 1, geo.ad);
            Tmp[c] = T(i > 0 && yp, c + nx - 1, geo.ad);
        }
        if (kperm) kperm[c] = (Real)kc;
    }
}

constexpr int kTileThreads = 256;  // cells of a tile at most (one thread each)
constexpr int kTransRun = 4;      // planes a block walks at most (its next plane's own cells are already there)

// Owned transmissibilities of a tile of TX x TY cells over kTransRun planes,
// and (kperm != null) the adjoint's copy of k.  Per plane the tile's
// reciprocals with the cells its links reach (one more row above, one more
// column on each side) sit
// in shared memory: 1.2 per cell instead of six.  Measured from ln k with the
// copy of k (a kernel of its own before): mixed 128^3 704 -> 42 us, FP64
// 97 x 83 x 50 144 -> 68 us (bound by the FP64 pipe: 1.5 exponentials and five
// quotients per cell).  Runs of 8 planes instead of 4 measured the same on the
// mixed path and 7 % slower in FP64 (fewer blocks); shorter ones where the tiles are
// too few for the multiprocessors (20^3, FP64, 10 links, from ln k 24.7 -> 10.4 us).
template <typename Real, bool LOG>
__global__ void __launch_bounds__(kTileThreads)
    k_trans(GridGeom g, Geo geo, int TX, int TY, int run, const double* __restrict__ perm, Real* Tx, Real* Ty, Real* Tz,
            Real* Tpp, Real* Tmp, Real* kperm, PermTag tag) {
    if (still_held(tag)) return;
    using R = Tile<Real>;
    using RT = typename R::type;
    // (TX + 2)(TY + 1) with TX TY <= 256 and TX <= 128 is at most 3 * 257
    constexpr int kPlane = 3 * (kTileThreads + 1);
    __shared__ RT tile[2][kPlane];
    __shared__ float2 eighth[8];
    const int PX = TX + 2;
    const int t = threadIdx.x, nt = blockDim.x;
    const bool in = t < TX * TY;
    const int ty = in ? t / TX : 0, tx = in ? t - ty * TX : 0;
    if (sizeof(Real) == 4 && LOG && t < 8) {
        const float h = (float)kEighth[t];
        eighth[t] = make_float2(h, (float)(kEighth[t] - (double)h));
    }
    if (sizeof(Real) == 4 && LOG) __syncthreads();
    const int nx = g.nx, ny = g.ny;
    const long long nxy = (long long)nx * ny;
    const unsigned bx = (unsigned)(nx + TX - 1) / TX, by = (unsigned)(ny + TY - 1) / TY;
    const unsigned bt = blockIdx.x / bx;
    const int i0 = (int)(blockIdx.x - bt * bx) * TX, j0 = (int)(bt % by) * TY;
    const int i = i0 + tx, j = j0 + ty;
    const bool act = in && i < nx && j < ny;
    // in-range cell of tile position (x, y), x = 0 the cell left of the tile
    auto cell = [&](int x, int y) {
        const int ci = min(max(i0 + x - 1, 0), nx - 1), cj = min(j0 + y, ny - 1);
        return ci + (long long)nx * cj;
    };
    const long long own = cell(tx + 1, ty);
    const int sp = ty * PX + tx + 1;
    const int k0 = (int)(bt / by) * run, k1 = min(k0 + run, g.nz);
    double vc = R::template pre<LOG>(perm[own + nxy * k0]);  // own k (FP64 path) or the stored value
    RT rc = R::template of<LOG>(vc, eighth);
    for (int k = k0; k < k1; ++k) {
        RT* const P = tile[(k - k0) & 1];
        const long long base = nxy * k;
        if (in) P[sp] = rc;
        // the row above and the columns left and right of the tile
        for (int h = t; h < PX + 2 * TY; h += nt) {
            const int x = h < PX ? h : (((h - PX) & 1) ? PX - 1 : 0), y = h < PX ? TY : (h - PX) / 2;
            P[y * PX + x] = R::template of<LOG>(R::template pre<LOG>(perm[base + cell(x, y)]), eighth);
        }
        const bool zp = k + 1 < g.nz;
        const double vn = zp ? R::template pre<LOG>(perm[base + nxy + own]) : vc;
        const RT rn = zp ? R::template of<LOG>(vn, eighth) : rc;
        __syncthreads();
        const long long c = base + own;
        auto put = [&](Real* T, bool there, RT rb, float2 ap, double a, long long d) {
            Real v = Real(0);
            if (there && !R::link(rc, rb, ap, a, v))
                v = (Real)two_point(perm_at<LOG>(perm, c), perm_at<LOG>(perm, d), a);
            T[c] = v;
        };
        if (act) {
            const bool xp = i + 1 < nx, yp = j + 1 < ny;
            put(Tx, xp, P[sp + 1], geo.px, geo.ax, xp ? c + 1 : c);
            put(Ty, yp, P[sp + PX], geo.py, geo.ay, yp ? c + nx : c);
            put(Tz, zp, rn, geo.pz, geo.az, zp ? c + nxy : c);
            if (g.diag) {
                const bool pp = yp && xp, mp = yp && i > 0;
                put(Tpp, pp, P[sp + PX + 1], geo.pd, geo.ad, pp ? c + nx + 1 : c);
                put(Tmp, mp, P[sp + PX - 1], geo.pd, geo.ad, mp ? c + nx - 1 : c);
            }
            if (kperm) {
                Real kv;
                if constexpr (sizeof(Real) == 4 && LOG) {
                    if (rc.x == kNoPair || !round_pair(pair_div(Pair32{1.f, 0.f}, Pair32{rc.x, rc.y}), kv))
                        kv = (Real)exp(vc);
                } else {
                    kv = (Real)vc;
                }
                kperm[c] = kv;
            }
        }
        vc = vn;
        rc = rn;
    }
}

// The library's own exponentials, one argument per element: exp_fp64,
// expm1_fp64, and expm1_f32 of the argument rounded to FP32 (its result
// widened exactly).  Only tpfa_math_eval launches it.
__global__ void k_math_eval(int fn, const double* __restrict__ x, double* __restrict__ y, long long n) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const double a = x[c];
        double r;
        if (fn == TPFA_MATH_EXP_FP64) r = exp_fp64(a);
        else if (fn == TPFA_MATH_EXPM1_FP64) r = expm1_fp64(a);
        else r = (double)expm1_f32(__double2float_rn(a));
        y[c] = r;
    }
}

Geo make_geo(const SetupPhys& s) {
    Geo q;
    q.ax = s.dy * s.dz / s.dx;
    q.ay = s.dx * s.dz / s.dy;
    q.az = s.dx * s.dy / s.dz;
    // diagonal: distance sqrt(dx^2 + dy^2), area dz dx dy / distance
    q.ad = s.dz * s.dx * s.dy / (s.dx * s.dx + s.dy * s.dy);
    // outside the pairs' range (pair_range): zero, whose links the FP64 formula decides
    auto pair = [](double v) {
        if (!(v >= 0x1p-90 && v <= 0x1p90)) return make_float2(0.f, 0.f);
        const float h = (float)v;
        return make_float2(h, (float)(v - (double)h));
    };
    q.px = pair(2.0 * q.ax), q.py = pair(2.0 * q.ay), q.pz = pair(2.0 * q.az), q.pd = pair(2.0 * q.ad);
    return q;
}

__global__ void k_to_f32(const double* __restrict__ in, float* out, long long n) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        out[c] = (float)in[c];
}

__global__ void k_copy_f64(const double* __restrict__ in, double* out, long long n) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        out[c] = in[c];
}

// m^n = (V/dt) phi(p^n) rho(p^n), phi(p) = phi0 (1 + c_r (p - p_ref)),
// rho(p) = rho_ref exp(c_f (p - p_ref))  (Eq. density), in FP64.
template <typename Real>
__global__ void k_prev_mass(SetupPhys s, const Real* __restrict__ pn, const double* __restrict__ phi0, double* mn,
                            long long n) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const double p = (double)pn[c];
        const double dp = p - s.p_ref;
        const double phi = phi0[c] * (1.0 + s.c_r * dp);
        const double rho = s.rho_ref * exp(s.c_f * dp);
        mn[c] = s.V_dt * (phi * rho);
    }
}

// One thread per row: row_ptr[row] from the closed form, then the valid
// neighbours in ascending column order (the slot order of tpfa_row.cuh).
__global__ void k_pattern(GridGeom g, long long* row_ptr, int* col_idx) {
    const long long nx = g.nx, nxy = nx * g.ny, N = nxy * g.nz;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
         c += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(c / nxy);
        const int j = (int)((c - k * nxy) / nx);
        const int i = (int)(c - k * nxy - j * nx);
        const long long rs = row_start(g, i, j, k);
        row_ptr[c] = rs;
        if (c == N - 1) row_ptr[N] = total_nnz(g);
        const bool xm = i > 0, xp = i + 1 < g.nx, ym = j > 0, yp = j + 1 < g.ny, zm = k > 0, zp = k + 1 < g.nz;
        const bool d = g.diag != 0;
        long long e = rs;
        if (zm) col_idx[e++] = (int)(c - nxy);
        if (d && xm && ym) col_idx[e++] = (int)(c - nx - 1);
        if (ym) col_idx[e++] = (int)(c - nx);
        if (d && xp && ym) col_idx[e++] = (int)(c - nx + 1);
        if (xm) col_idx[e++] = (int)(c - 1);
        col_idx[e++] = (int)c;
        if (xp) col_idx[e++] = (int)(c + 1);
        if (d && xm && yp) col_idx[e++] = (int)(c + nx - 1);
        if (yp) col_idx[e++] = (int)(c + nx);
        if (d && xp && yp) col_idx[e++] = (int)(c + nx + 1);
        if (zp) col_idx[e++] = (int)(c + nxy);
    }
}

}  // namespace

template <typename Real>
static cudaError_t launch_trans_t(const GridGeom& g, const SetupPhys& s, const double* perm, Real* Tx, Real* Ty,
                                  Real* Tz, Real* Tpp, Real* Tmp, Real* kperm, cudaStream_t st, bool log_k,
                                  const PermTag& tag) {
    // one block index for tiles and z-runs: any grid shape of fewer than 2^31 cells fits
    int TX = 1, TY = 1;
    tile_shape(g.nx, g.ny, kTileThreads, TX, TY);
    const long long tiles = (long long)((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY);
    // shorter runs where the long ones would leave multiprocessors idle
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int run = kTransRun;
    while (run > 1 && tiles * ((g.nz + run - 1) / run) < 2LL * sms) run /= 2;
    const long long nb = tiles * ((g.nz + run - 1) / run);
    const int block = (TX * TY + 31) / 32 * 32;
    const Geo q = make_geo(s);
    if (TX * TY <= (sizeof(Real) == 8 ? 16 : 2)) {
        const unsigned cells = blocks_for((long long)g.nx * g.ny * g.nz);
        if (log_k) k_trans_cells<Real, true><<<cells, kThreads, 0, st>>>(g, q, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, tag);
        else k_trans_cells<Real, false><<<cells, kThreads, 0, st>>>(g, q, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, tag);
        return cudaGetLastError();
    }
    if (log_k) k_trans<Real, true><<<(unsigned)nb, block, 0, st>>>(g, q, TX, TY, run, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, tag);
    else k_trans<Real, false><<<(unsigned)nb, block, 0, st>>>(g, q, TX, TY, run, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, tag);
    return cudaGetLastError();
}

cudaError_t launch_transmissibility_f32(const GridGeom& g, const SetupPhys& s, const double* perm, float* Tx,
                                        float* Ty, float* Tz, float* Tpp, float* Tmp, float* kperm, cudaStream_t st,
                                        bool log_k, const PermTag& tag) {
    return launch_trans_t<float>(g, s, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, st, log_k, tag);
}

cudaError_t launch_transmissibility_f64(const GridGeom& g, const SetupPhys& s, const double* perm, double* Tx,
                                        double* Ty, double* Tz, double* Tpp, double* Tmp, double* kperm,
                                        cudaStream_t st, bool log_k, const PermTag& tag) {
    return launch_trans_t<double>(g, s, perm, Tx, Ty, Tz, Tpp, Tmp, kperm, st, log_k, tag);
}

cudaError_t launch_convert_f32(const double* in, float* out, long long n, cudaStream_t st) {
    k_to_f32<<<blocks_for(n), kThreads, 0, st>>>(in, out, n);
    return cudaGetLastError();
}

cudaError_t launch_copy_f64(const double* in, double* out, long long n, cudaStream_t st) {
    k_copy_f64<<<blocks_for(n), kThreads, 0, st>>>(in, out, n);
    return cudaGetLastError();
}

cudaError_t launch_prev_mass_f32(const SetupPhys& s, const float* pn, const double* phi0, double* mn, long long n,
                                 cudaStream_t st) {
    k_prev_mass<float><<<blocks_for(n), kThreads, 0, st>>>(s, pn, phi0, mn, n);
    return cudaGetLastError();
}

cudaError_t launch_prev_mass_f64(const SetupPhys& s, const double* pn, const double* phi0, double* mn, long long n,
                                 cudaStream_t st) {
    k_prev_mass<double><<<blocks_for(n), kThreads, 0, st>>>(s, pn, phi0, mn, n);
    return cudaGetLastError();
}

cudaError_t launch_pattern(const GridGeom& g, long long* row_ptr, int* col_idx, cudaStream_t st) {
    const long long N = (long long)g.nx * g.ny * g.nz;
    k_pattern<<<blocks_for(N), kThreads, 0, st>>>(g, row_ptr, col_idx);
    return cudaGetLastError();
}

cudaError_t launch_math_eval(int fn, const double* x, double* y, long long n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    k_math_eval<<<blocks_for(n), kThreads, 0, st>>>(fn, x, y, n);
    return cudaGetLastError();
}

}  // namespace tpfa
