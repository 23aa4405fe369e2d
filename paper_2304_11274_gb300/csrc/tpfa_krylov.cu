// tpfa_krylov.cu -- preconditioned BiCGStab on the assembled Jacobian (the
// linear solve of a Newton step on Eq. vk), sm_103a.
//
// BiCGStab (van der Vorst, 1992) with right preconditioning by M, the
// tridiagonal part of J along z (default) or its diagonal (Jacobi):
//   r = b, r^ = b, x = 0, rho = (r^, r)
//   repeat:  p = r + beta (p - omega v)            (p = r on the first pass)
//            p^ = M^-1 p,  v = J p^,  alpha = rho / (r^, v)
//            s = r - alpha v,  s^ = M^-1 s,  t = J s^,  omega = (t, s) / (t, t)
//            x += alpha p^ + omega s^,  r = s - omega t
//            rho' = (r^, r),  beta = (rho' / rho)(alpha / omega),  rho = rho'
//   until ||r||_2 <= rtol ||b||_2.
// Five kernels per iteration: the update of p fused with M^-1 (p^), the product
// with J and its dot product, the update of s (stored over r) fused with M^-1
// (s^), the product again, and the update of x and r.  Every scalar lives in a
// device-side KrylovScalars record: each dot product is reduced per block into
// a partial-sum array, and the block that finishes last sums the partials in a
// fixed order and advances the scalars, so results are deterministic and the
// host only polls the record.  Once `done` is set every kernel returns at
// entry, so the host may enqueue several iterations between polls.
//
// What bounds it: HBM (0.83 GB per iteration at 128^3 of which the L2 keeps
// some) and the FP64 pipe (two operations per clock and multiprocessor;
// 24 per cell and iteration).  So the matrix is copied once per solve from its
// CSR order to slot-major groups of 32 cells (the CSR rows of 11 values would
// cost eleven times the L1 wavefronts in each of the two products of every
// iteration), dot products are accumulated per thread
// over a run of planes before the warp reduction (whose ten FP64 additions per
// warp would otherwise equal ten per cell), and conversions avoid the FP64 pipe.
// Measured at 128^3 (mixed, z-line): 0.331 -> 0.175 ms per iteration; the
// product 69 -> 36 us (168 MB: 4.7 TB/s), the line solve with its update 62
// (p) and 59 (s) -> 38 and 34 us, the last update 31 us either way, three
// one-block reduction kernels of 13 us each gone.
//
// FP64 path: products and sums in FP64.  Mixed path: the FP32 off-diagonal
// values times the vector split into FP32 pairs (written by the update
// kernels), exact two-float products summed as a double-float, plus the FP64
// diagonal times the FP64 vector.
#include <cuda_runtime.h>

#include <type_traits>

#include "tpfa_impl.h"
#include "tpfa_row.cuh"

namespace tpfa {

namespace {

constexpr int kThreads = 256;
constexpr int kVecBlocks = 152 * 5;   // blocks of the vector kernels, at most
constexpr int kMaxBlocks = 152 * 4;   // blocks of the products: one wave

// v as an FP32 pair hi + lo without the FP64 pipe: hi the truncation of v, lo the
// 29 fraction bits it leaves, rounded to 24 (below 2^-126 to a multiple of
// 2^-149).  A v below 2^-126 is rounded to a subnormal hi alone, beyond the FP32
// range hi is infinite (the solve then breaks down, as it must).
__device__ __forceinline__ float2 split_pair(double v) {
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const uint32_t a = h & 0x7fffffffu, sign = h & 0x80000000u;
    uint32_t hi = ((a - 0x38000000u) << 3) | (l >> 29);
    // lo = low bits 2^-52 times the power of two of hi
    float lo = __fmul_rn(__fmul_rn(__uint2float_rn(l & 0x1fffffffu), 0x1p-52f),
                         __uint_as_float((hi & 0x7f800000u) | sign));
    if (a - 0x38100000u >= 0x0fe00000u) {
        hi = a ? narrow_rare(a, l) : 0u;
        lo = 0.f;
    }
    return make_float2(__uint_as_float(hi | sign), lo);
}

__device__ __forceinline__ bool finite(double x) { return !nonfinite(x); }

// Advance the scalars.  stage 0: after k_init; 1: after v = J p^; 2: after
// t = J s^; 3: after k_update_xr.
__device__ __forceinline__ void advance(int stage, double d0, double d1, KrylovScalars* S) {
    switch (stage) {
        case 0:  // rho = (r^, r) = (b, b)
            S->bb = d0;
            S->rho = d0;
            S->rr = d0;
            S->iter = 0;
            S->breakdown = 0;
            S->alpha = S->omega = 1.0;
            S->beta = 0.0;
            S->done = (d0 == 0.0) ? 1 : 0;  // b = 0: x = 0 is exact
            if (!finite(d0)) S->done = S->breakdown = 1;
            break;
        case 1:  // alpha = rho / (r^, v)
            if (d0 == 0.0 || !finite(d0)) {
                S->done = S->breakdown = 1;
            } else {
                S->alpha = S->rho / d0;
            }
            break;
        case 2:  // omega = (t, s) / (t, t); t = 0 means s = 0: the half step solved it
            S->omega = (d1 > 0.0 && finite(d1) && finite(d0)) ? d0 / d1 : 0.0;
            break;
        default: {  // rho' = (r^, r), rr = (r, r)
            S->iter += 1;
            S->rr = d1;
            if (!finite(d0) || !finite(d1)) {
                S->done = S->breakdown = 1;
            } else if (d1 <= S->tol2 * S->bb) {
                S->done = 1;
            } else if (S->omega == 0.0 || d0 == 0.0) {
                S->done = S->breakdown = 1;
            } else {
                S->beta = (d0 / S->rho) * (S->alpha / S->omega);
                S->rho = d0;
                if (S->iter >= S->max_iters) S->done = 1;
            }
        }
    }
}

// Sums d0 and d1 over the block; the sums are returned to thread 0.  The two
// half-warps carry one sum each after the first step: five FP64 additions
// per warp instead of ten.
__device__ __forceinline__ void block_sum(double& d0, double& d1) {
    __shared__ double sh[2][kThreads / 32];
    const int t = threadIdx.x, lane = t & 31;
    const double other = __shfl_xor_sync(0xffffffffu, lane < 16 ? d1 : d0, 16);
    double d = (lane < 16 ? d0 : d1) + other;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o, 16);
    if ((lane & 15) == 0) sh[lane >> 4][t >> 5] = d;
    __syncthreads();
    if (t < 32) {  // half-warp 0 sums d0's parts, half-warp 1 d1's
        d = (lane & 15) < kThreads / 32 ? sh[lane >> 4][lane & 15] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o, 16);
        d0 = d;
        d1 = __shfl_sync(0xffffffffu, d, 16);
    }
}

// The end of every reducing kernel (all threads of all blocks): per-block
// partials, and in the last block to arrive their sum in block order and the
// next scalars.  The counter goes back to zero for the next kernel.
__device__ __forceinline__ void reduce_and_advance(double d0, double d1, int stage, const KrylovSums& k) {
    __shared__ bool last;
    block_sum(d0, d1);
    if (threadIdx.x == 0) {
        k.part[2 * blockIdx.x] = d0;
        k.part[2 * blockIdx.x + 1] = d1;
        __threadfence();
        last = atomicAdd(k.arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    d0 = d1 = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kThreads) {
        d0 += __ldcg(k.part + 2 * b);
        d1 += __ldcg(k.part + 2 * b + 1);
    }
    __syncthreads();  // block_sum's buffer is free again
    block_sum(d0, d1);
    if (threadIdx.x == 0) {
        *k.arrived = 0u;
        advance(stage, d0, d1, k.S);
    }
}

// ---------------------------------------------------------------- the matrix by slots

// Slot arrays present with the grid's connectivity, in slot order.
template <bool DIAG>
__host__ __device__ constexpr int slot_array(int s) {
    if (DIAG) return s < SLOT_SELF ? s : s - 1;
    return s == 0 ? 0 : s == 2 ? 1 : s == 4 ? 2 : s == 6 ? 3 : s == 8 ? 4 : 5;
}

// Values per cell (off-diagonals), and the position of cell c's entry n: groups
// of 32 consecutive cells hold their entries slot by slot, so a warp reads each
// slot as one coalesced run at a constant offset from its first.
template <bool DIAG>
constexpr int kSlots = DIAG ? 10 : 6;
template <bool DIAG>
__device__ __forceinline__ long long slot_at(long long c) {
    return (c >> 5) * (kSlots<DIAG> * 32) + (c & 31);
}

// CSR rows to slots (entries of links that do not exist are zero) and, on the
// FP64 path, the diagonal.
template <typename Real, bool DIAG>
__global__ void __launch_bounds__(kThreads) k_by_slots(GridGeom g, const Real* __restrict__ vals, Real* __restrict__ dia,
                                                       double* __restrict__ diag) {
    const long long nxy = (long long)g.nx * g.ny, N = nxy * g.nz;
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < N; c += (long long)gridDim.x * kThreads) {
        const int k = (int)(c / nxy), q = (int)(c - nxy * k), j = q / g.nx, i = q - j * g.nx;
        const unsigned mask = slot_mask(g, i, j, k);
        const Real* row = vals + row_start(g, i, j, k);
        Real* out = dia + slot_at<DIAG>(c);
        int pos = 0;
#pragma unroll
        for (int s = 0; s < NSLOT; ++s) {
            const bool there = (mask >> s) & 1u;
            const Real v = there ? row[pos] : Real(0);
            pos += there;
            if (s == SLOT_SELF) {
                if constexpr (sizeof(Real) == 8) diag[c] = v;
            } else if (DIAG || !((0x28au >> s) & 1u)) {
                out[slot_array<DIAG>(s) * 32] = v;
            }
        }
    }
}

__device__ __forceinline__ double as_f64(float x) { return widen(x); }
__device__ __forceinline__ double as_f64(double x) { return x; }

// y = J x and the partials of (a, y) and, with YY, (y, y).  One thread per
// column of a run of planes: it keeps x of planes k - 1, k and k + 1, and loads
// the row operands of plane k + 1 (off-diagonals, diagonal, x, a) before it works
// on plane k, so that about 2 KB per warp are on their way from HBM at any time.
// Mixed path: x also as split pairs hi + lo (FP32), the FP32 off-diagonals v:
// each v hi is formed exactly as p + e (e = fma(v, hi, -p)), v lo is added to e,
// and the terms are summed as a double-float (TwoSum on the leading parts, the
// trailing parts summed apart), about 48 bits; the FP64 diagonal times the
// FP64 x is added in FP64.  Four FP64 operations per row with the dot products
// instead of thirteen, the product as accurate as an FP64 one for the Krylov
// iteration.
template <typename Real, bool DIAG, bool YY>
__global__ void __launch_bounds__(kThreads, sizeof(Real) == 4 ? 4 : 2)
    k_spmv(GridGeom g, int run, long long items, const Real* __restrict__ dia, const double* __restrict__ diag,
           const double* __restrict__ x, const float2* __restrict__ xp, double* __restrict__ y,
           const double* __restrict__ a, KrylovSums sums) {
    if (sums.S->done) return;  // uniform over the grid
    constexpr bool MIXED = sizeof(Real) == 4;
    constexpr int NA = kSlots<DIAG>;
    using X = typename std::conditional<MIXED, float2, double>::type;
    const X* __restrict__ xv;
    if constexpr (MIXED) xv = xp;
    else xv = x;
    const int nx = g.nx, nxy = nx * g.ny;
    const int runs = (g.nz + run - 1) / run;
    double d0 = 0.0, d1 = 0.0;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const long long qt = it / runs;
        const int k0 = (int)(it - qt * runs) * run, k1 = min(k0 + run, g.nz);
        const long long q = qt * kThreads + threadIdx.x;
        if (q >= nxy) continue;
        const int j = (int)q / nx, i = (int)q - j * nx;
        const bool xm = i > 0, xpl = i + 1 < nx, ym = j > 0, yp = j + 1 < g.ny;
        struct Row {
            Real v[NA];
            double d, x, a;
        };
        auto load_row = [&](Row& w, long long c) {
            const Real* D = dia + slot_at<DIAG>(c);
#pragma unroll
            for (int n = 0; n < NA; ++n) w.v[n] = __ldcs(D + n * 32);  // read once per product
            w.d = diag[c];
            w.x = MIXED ? x[c] : 0.0;
            w.a = a[c];
        };
        long long c = q + (long long)nxy * k0;
        X zero{};
        X pm = k0 > 0 ? xv[c - nxy] : zero, pc = xv[c];
        Row next;
        load_row(next, c);
        for (int k = k0; k < k1; ++k, c += nxy) {
            const Row w = next;
            const X* const xc = xv + c;
            const X pp = k + 1 < g.nz ? xc[nxy] : zero;
            const X x2 = ym ? xc[-nx] : zero, x4 = xm ? xc[-1] : zero, x6 = xpl ? xc[1] : zero, x8 = yp ? xc[nx] : zero;
            X x1 = zero, x3 = zero, x7 = zero, x9 = zero;
            if (DIAG) {
                x1 = xm && ym ? xc[-nx - 1] : zero;
                x3 = xpl && ym ? xc[-nx + 1] : zero;
                x7 = xm && yp ? xc[nx - 1] : zero;
                x9 = xpl && yp ? xc[nx + 1] : zero;
            }
            if (k + 1 < k1) load_row(next, c + nxy);
            float ah = 0.f, al = 0.f;
            double acc = 0.0;
            auto term = [&](int n, X xn) {
                const Real v = w.v[n];
                if constexpr (MIXED) {
                    const float p = __fmul_rn(v, xn.x);
                    const float t = __fmaf_rn(v, xn.y, __fmaf_rn(v, xn.x, -p));
                    const float sum = __fadd_rn(ah, p);
                    const float bb = __fsub_rn(sum, ah);
                    const float err = __fadd_rn(__fsub_rn(ah, __fsub_rn(sum, bb)), __fsub_rn(p, bb));
                    ah = sum;
                    al = __fadd_rn(al, __fadd_rn(err, t));
                } else {
                    acc = __fma_rn(v, xn, acc);
                }
            };
            // absent neighbours: a zero entry times zero
            term(slot_array<DIAG>(0), pm);
            if (DIAG) term(slot_array<DIAG>(1), x1);
            term(slot_array<DIAG>(2), x2);
            if (DIAG) term(slot_array<DIAG>(3), x3);
            term(slot_array<DIAG>(4), x4);
            term(slot_array<DIAG>(6), x6);
            if (DIAG) term(slot_array<DIAG>(7), x7);
            term(slot_array<DIAG>(8), x8);
            if (DIAG) term(slot_array<DIAG>(9), x9);
            term(slot_array<DIAG>(10), pp);
            double yc;
            if constexpr (MIXED) {
                // a subnormal or non-finite part would not survive the cheap widening
                double off;
                if (min(sub_word(ah), sub_word(al)) >= kSubnormal && finite_f32(ah))
                    off = __dadd_rn(widen_flush(ah), widen_flush(al));
                else
                    off = __dadd_rn(widen(ah), widen(al));
                yc = __fma_rn(w.d, w.x, off);
            } else {
                yc = __fma_rn(w.d, pc, acc);
            }
            y[c] = yc;
            d0 = __fma_rn(w.a, yc, d0);
            if (YY) d1 = __fma_rn(yc, yc, d1);
            pm = pc;
            pc = pp;
        }
    }
    reduce_and_advance(d0, d1, YY ? 2 : 1, sums);
}

// M^-1 = 1 / diag(J) (1 where the diagonal is zero).
__global__ void __launch_bounds__(kThreads) k_dinv(long long n, const double* __restrict__ diag,
                                                   double* __restrict__ dinv) {
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < n; c += (long long)gridDim.x * kThreads) {
        const double d = diag[c];
        dinv[c] = d != 0.0 ? 1.0 / d : 1.0;
    }
}

// ---------------------------------------------------------------- z-line preconditioner
//
// M = the tridiagonal part of J along z (each cell's diagonal and its two
// vertical couplings), inverted exactly column by column: the vertical links of
// 10 x 10 x 2 m cells carry 25 times the transmissibility of the horizontal
// ones, so M captures most of J.  The columns are few (nx ny: 512 warps of a
// 128 x 128 grid, less than one per scheduler) and a sweep is a chain of
// dependent steps, so each column is eliminated from both ends at once (the
// twisted factorisation, "burn at both ends"): warp 0 of a block takes its 32
// columns from plane 0 up to the middle plane m, warp 1 from plane nz - 1 down
// to it, the two meet in row m and substitute back outwards, with the same
// operation count as the one-ended Thomas algorithm.  The factorisation
// (once per solve) stores per cell the multiplier l (of the row before it in
// its half), the inverse pivot 1 / b' and u, the coupling to the row after it
// over the pivot (row m has two rows before it and none after: l and u hold
// its two multipliers).  Elimination: y = in - l y_before; back: z = y / b' - u
// z_after; one dependent FP64 operation per step each.  The sweep's input, p or
// s, is formed on the way (its update needs no kernel of its own).  Operands
// are on their way into a shared-memory ring kLineDepth steps ahead (8-byte
// cp.async per value) in chunks of kChunk: a chunk's independent operations are
// issued together.

constexpr int kLineDepth = 16;  // steps in flight per half column
constexpr int kChunk = 4;       // steps read together

// The rows of half w (0: from plane 0, 1: from plane nz - 1) without row m.
struct Half {
    int m, len, first, dir;
    __device__ __forceinline__ Half(int nz, int w)
        : m(nz / 2), len(w == 0 ? m : nz - 1 - m), first(w == 0 ? 0 : nz - 1), dir(w == 0 ? 1 : -1) {}
};

template <typename Real, bool DIAG>
__global__ void __launch_bounds__(64) k_line_factor(GridGeom g, const Real* __restrict__ dia,
                                                    const double* __restrict__ diag, double* __restrict__ inv_b,
                                                    double* __restrict__ lmul, double* __restrict__ up) {
    __shared__ double end[2][32];  // coupling of row m's neighbour to row m over that neighbour's pivot
    const long long nxy = (long long)g.nx * g.ny;
    const int w = threadIdx.y, l = threadIdx.x;
    const long long col = blockIdx.x * 32LL + l;
    const bool on = col < nxy;
    const Half h(g.nz, w);
    // coupling of row k to the row before / after it in this half's order
    const int before = (w == 0 ? slot_array<DIAG>(0) : slot_array<DIAG>(10)) * 32;
    const int after = (w == 0 ? slot_array<DIAG>(10) : slot_array<DIAG>(0)) * 32;
    double u = 0.0, inv = 0.0;  // of the row before
    double a_prev = 0.0;
    if (on) {
#pragma unroll 4
        for (int e = 0; e < h.len; ++e) {
            const long long c = col + nxy * (h.first + h.dir * e);
            const Real* D = dia + slot_at<DIAG>(c);
            const double a = as_f64(D[after]), bf = e > 0 ? as_f64(D[before]) : 0.0;
            const double lm = bf * inv;
            const double b = fma(-lm, a_prev, diag[c]);
            inv = b != 0.0 ? 1.0 / b : 1.0;
            u = a * inv;
            inv_b[c] = inv;
            lmul[c] = lm;
            up[c] = u;
            a_prev = a;
        }
    }
    end[w][l] = h.len > 0 ? inv : 0.0;
    __shared__ double cpl[2][32];
    cpl[w][l] = h.len > 0 ? a_prev : 0.0;
    __syncthreads();
    if (w == 0 && on) {  // row m
        const long long c = col + nxy * h.m;
        const Real* D = dia + slot_at<DIAG>(c);
        const double l0 = h.m > 0 ? as_f64(D[slot_array<DIAG>(0) * 32]) * end[0][l] : 0.0;
        const double l1 = h.m + 1 < g.nz ? as_f64(D[slot_array<DIAG>(10) * 32]) * end[1][l] : 0.0;
        const double b = fma(-l1, cpl[1][l], fma(-l0, cpl[0][l], diag[c]));
        inv_b[c] = b != 0.0 ? 1.0 / b : 1.0;
        lmul[c] = l0;
        up[c] = l1;
    }
}

__device__ __forceinline__ void cp8_async(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The vector the preconditioner is applied to, formed from its update:
// p = r + beta (p - omega v) (p = r on the first pass), or s = r - alpha v,
// which replaces r.
struct Update {
    bool is_p, first;
    double beta, omega, alpha;
    __device__ __forceinline__ Update(bool p, const KrylovScalars* S)
        : is_p(p), first(S->iter == 0), beta(S->beta), omega(S->omega), alpha(S->alpha) {}
    __device__ __forceinline__ double operator()(double r, double v, double p) const {
        if (is_p) return first ? r : fma(beta, fma(-omega, v, p), r);
        return fma(-alpha, v, r);
    }
};

// (p or s), out = M^-1 (p or s), and on the mixed path out as FP32 pairs.
// Each lane copies and reads back only its own ring entries; a chunk's slots
// are refilled after its operands are in registers.
template <bool IS_P>
__global__ void __launch_bounds__(64)
    k_line_apply(GridGeom g, const double* __restrict__ inv_b, const double* __restrict__ lmul,
                 const double* __restrict__ up, double* __restrict__ r, const double* __restrict__ v,
                 double* __restrict__ p, double* __restrict__ out, float2* __restrict__ pair, const KrylovScalars* S) {
    constexpr int CH = kChunk, NCH = kLineDepth / kChunk;
    static_assert((NCH & (NCH - 1)) == 0, "ring index by mask");
    __shared__ __align__(16) double ring_all[2][NCH][CH][4][32];
    __shared__ double meet[2][32];
    if (S->done) return;
    const long long nxy = (long long)g.nx * g.ny;
    const int w = threadIdx.y, l = threadIdx.x;
    const long long col = blockIdx.x * 32LL + l;
    const bool on = col < nxy;
    const Half h(g.nz, w);
    const int len = on ? h.len : 0, chunks = (len + CH - 1) / CH, full = len / CH;
    const long long st = h.dir * nxy;  // elements from one row to the next
    double(*const ring)[CH][4][32] = ring_all[w];
    const Update upd(IS_P, S);

    // ---- elimination towards row m
    long long ci = col + nxy * h.first;  // cell of the next chunk to request
    auto issue_f = [&](int ch) {
        if (ch < chunks) {
            auto& R = ring[ch & (NCH - 1)];
#pragma unroll
            for (int e = 0; e < CH; ++e) {
                if (ch < full || ch * CH + e < len) {
                    const long long c = ci + e * st;
                    cp8_async(&R[e][0][l], r + c);
                    cp8_async(&R[e][1][l], v + c);
                    if (IS_P) cp8_async(&R[e][2][l], p + c);
                    cp8_async(&R[e][3][l], lmul + c);
                }
            }
            ci += CH * st;
        }
        cp_commit();
    };
    for (int ch = 0; ch < NCH; ++ch) issue_f(ch);
    double y = 0.0;
    long long c0 = col + nxy * h.first;
    for (int ch = 0; ch < chunks; ++ch, c0 += CH * st) {
        cp_wait<NCH - 1>();
        auto& R = ring[ch & (NCH - 1)];
        double in[CH], m[CH];
#pragma unroll
        for (int e = 0; e < CH; ++e) {
            in[e] = upd(R[e][0][l], R[e][1][l], IS_P ? R[e][2][l] : 0.0);
            m[e] = R[e][3][l];
        }
        issue_f(ch + NCH);
#pragma unroll
        for (int e = 0; e < CH; ++e) {
            if (ch < full || ch * CH + e < len) {
                y = fma(-m[e], y, in[e]);
                (IS_P ? p : r)[c0 + e * st] = in[e];
                out[c0 + e * st] = y;
            }
        }
    }
    cp_wait<0>();
    meet[w][l] = y;
    __syncthreads();  // also: y stored above is read back below by the same thread
    double z = 0.0;
    if (on) {  // row m, by both halves; the first one stores it
        const long long c = col + nxy * h.m;
        const double in = upd(r[c], v[c], IS_P ? p[c] : 0.0);
        const double ym = fma(-up[c], meet[1][l], fma(-lmul[c], meet[0][l], in));
        z = ym * inv_b[c];
    }
    __syncthreads();  // row m's operands are read before they are replaced
    if (on && w == 0) {
        const long long c = col + nxy * h.m;
        (IS_P ? p : r)[c] = upd(r[c], v[c], IS_P ? p[c] : 0.0);
        out[c] = z;
        if (pair) pair[c] = split_pair(z);
    }

    // ---- back substitution away from row m
    ci = col + nxy * (h.m - h.dir);
    auto issue_b = [&](int ch) {
        if (ch < chunks) {
            auto& R = ring[ch & (NCH - 1)];
#pragma unroll
            for (int e = 0; e < CH; ++e) {
                if (ch < full || ch * CH + e < len) {
                    const long long c = ci - e * st;
                    cp8_async(&R[e][0][l], out + c);
                    cp8_async(&R[e][1][l], up + c);
                    cp8_async(&R[e][2][l], inv_b + c);
                }
            }
            ci -= CH * st;
        }
        cp_commit();
    };
    for (int ch = 0; ch < NCH; ++ch) issue_b(ch);
    c0 = col + nxy * (h.m - h.dir);
    for (int ch = 0; ch < chunks; ++ch, c0 -= CH * st) {
        cp_wait<NCH - 1>();
        auto& R = ring[ch & (NCH - 1)];
        double yi[CH], u[CH];
#pragma unroll
        for (int e = 0; e < CH; ++e) {
            yi[e] = R[e][0][l] * R[e][2][l];
            u[e] = R[e][1][l];
        }
        issue_b(ch + NCH);
#pragma unroll
        for (int e = 0; e < CH; ++e) {
            if (ch < full || ch * CH + e < len) {
                z = fma(-u[e], z, yi[e]);
                out[c0 - e * st] = z;
                if (pair) pair[c0 - e * st] = split_pair(z);
            }
        }
    }
    cp_wait<0>();
}

// The same with M^-1 = 1 / diag(J).
template <bool IS_P>
__global__ void __launch_bounds__(kThreads) k_diag_apply(long long n, const double* __restrict__ dinv,
                                                         double* __restrict__ r, const double* __restrict__ v,
                                                         double* __restrict__ p, double* __restrict__ out,
                                                         float2* __restrict__ pair, const KrylovScalars* S) {
    if (S->done) return;
    const Update upd(IS_P, S);
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < n; c += (long long)gridDim.x * kThreads) {
        const double in = upd(r[c], v[c], IS_P ? p[c] : 0.0);
        (IS_P ? p : r)[c] = in;
        const double z = in * dinv[c];
        out[c] = z;
        if (pair) pair[c] = split_pair(z);
    }
}

// x = 0, r = r^ = sign * b; rho = (b, b).
__global__ void __launch_bounds__(kThreads) k_init(long long n, const double* __restrict__ b, double sign,
                                                   double* __restrict__ x, double* __restrict__ r,
                                                   double* __restrict__ rh, KrylovSums sums) {
    double d0 = 0.0;
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < n; c += (long long)gridDim.x * kThreads) {
        const double bc = sign * b[c];
        x[c] = 0.0;
        r[c] = bc;
        rh[c] = bc;
        d0 = fma(bc, bc, d0);
    }
    reduce_and_advance(d0, 0.0, 0, sums);
}

// x += alpha p^ + omega s^, r = s - omega t (s is held in r); (r^, r) and (r, r).
__global__ void __launch_bounds__(kThreads) k_update_xr(long long n, double* __restrict__ x,
                                                        const double* __restrict__ ph, const double* __restrict__ sh,
                                                        const double* __restrict__ t, double* __restrict__ r,
                                                        const double* __restrict__ rh, KrylovSums sums) {
    if (sums.S->done) return;
    const double alpha = sums.S->alpha, omega = sums.S->omega;
    double d0 = 0.0, d1 = 0.0;
#pragma unroll 4
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < n; c += (long long)gridDim.x * kThreads) {
        x[c] = fma(omega, sh[c], fma(alpha, ph[c], x[c]));
        const double rc = fma(-omega, t[c], r[c]);
        r[c] = rc;
        d0 = fma(rh[c], rc, d0);
        d1 = fma(rc, rc, d1);
    }
    reduce_and_advance(d0, d1, 3, sums);
}

// p = p + delta, rounded to the field type.
template <typename Real>
__global__ void __launch_bounds__(kThreads) k_add_delta(long long n, Real* p, const double* __restrict__ d) {
    for (long long c = blockIdx.x * (long long)kThreads + threadIdx.x; c < n; c += (long long)gridDim.x * kThreads)
        p[c] = (Real)((double)p[c] + d[c]);
}

unsigned vec_blocks(long long n) {
    const long long b = (n + kThreads - 1) / kThreads;
    return (unsigned)(b < 1 ? 1 : (b > kVecBlocks ? kVecBlocks : b));
}

template <typename Real, bool DIAG, bool YY>
cudaError_t launch_spmv(const GridGeom& g, const KrylovWork& w, const double* x, double* y, const double* a,
                        cudaStream_t st) {

    // runs of planes: the busiest block's planes are minimised (a run's start
    // costs about one more)
    const long long tiles = ((long long)g.nx * g.ny + kThreads - 1) / kThreads;
    long long run = 1, best = -1;
    for (int r = 1; r <= g.nz && r <= 64; ++r) {
        const long long cost = (tiles * ((g.nz + r - 1) / r) + kMaxBlocks - 1) / kMaxBlocks * (r + 1);
        if (best < 0 || cost < best) best = cost, run = r;
    }
    const long long items = tiles * ((g.nz + run - 1) / run);
    const unsigned nb = (unsigned)(items < kMaxBlocks ? items : kMaxBlocks);
    k_spmv<Real, DIAG, YY><<<nb, kThreads, 0, st>>>(g, (int)run, items, (const Real*)w.dia, w.diag, x, w.pair, y, a,
                                                    w.sums);
    return cudaGetLastError();
}

template <typename Real, bool DIAG>
cudaError_t iteration(const GridGeom& g, long long n, const KrylovWork& w, bool line, cudaStream_t st) {
    const unsigned nl = (unsigned)(((long long)g.nx * g.ny + 31) / 32), nb = vec_blocks(n);
    const dim3 halves(32, 2, 1);
    float2* pair = sizeof(Real) == 4 ? w.pair : nullptr;
    if (line) k_line_apply<true><<<nl, halves, 0, st>>>(g, w.dinv, w.lmul, w.up, w.r, w.v, w.p, w.ph, pair, w.sums.S);
    else k_diag_apply<true><<<nb, kThreads, 0, st>>>(n, w.dinv, w.r, w.v, w.p, w.ph, pair, w.sums.S);
    cudaError_t e = launch_spmv<Real, DIAG, false>(g, w, w.ph, w.v, w.rh, st);
    if (e != cudaSuccess) return e;
    if (line) k_line_apply<false><<<nl, halves, 0, st>>>(g, w.dinv, w.lmul, w.up, w.r, w.v, w.p, w.sh, pair, w.sums.S);
    else k_diag_apply<false><<<nb, kThreads, 0, st>>>(n, w.dinv, w.r, w.v, w.p, w.sh, pair, w.sums.S);
    e = launch_spmv<Real, DIAG, true>(g, w, w.sh, w.t, w.r, st);
    if (e != cudaSuccess) return e;
    k_update_xr<<<nb, kThreads, 0, st>>>(n, w.x, w.ph, w.sh, w.t, w.r, w.rh, w.sums);
    return cudaGetLastError();
}

template <typename Real, bool DIAG>
void prepare(const GridGeom& g, long long n, const void* vals, const KrylovWork& w, bool line, cudaStream_t st) {
    k_by_slots<Real, DIAG><<<vec_blocks(n), kThreads, 0, st>>>(g, (const Real*)vals, (Real*)w.dia, w.diag);
    if (line) {
        const unsigned nb = (unsigned)(((long long)g.nx * g.ny + 31) / 32);
        k_line_factor<Real, DIAG><<<nb, dim3(32, 2, 1), 0, st>>>(g, (const Real*)w.dia, w.diag, w.dinv, w.lmul, w.up);
    } else {
        k_dinv<<<vec_blocks(n), kThreads, 0, st>>>(n, w.diag, w.dinv);
    }
}

}  // namespace

long long krylov_partials() { return kMaxBlocks > kVecBlocks ? kMaxBlocks : kVecBlocks; }

long long krylov_slot_values(const GridGeom& g, long long n) { return (n + 31) / 32 * 32 * (g.diag ? 10 : 6); }

cudaError_t krylov_start(const GridGeom& g, long long n, bool mixed, const void* vals, const double* b, double sign,
                         const KrylovWork& w, bool line, cudaStream_t st) {
    if (mixed) g.diag ? prepare<float, true>(g, n, vals, w, line, st) : prepare<float, false>(g, n, vals, w, line, st);
    else g.diag ? prepare<double, true>(g, n, vals, w, line, st) : prepare<double, false>(g, n, vals, w, line, st);
    k_init<<<vec_blocks(n), kThreads, 0, st>>>(n, b, sign, w.x, w.r, w.rh, w.sums);
    return cudaGetLastError();
}

cudaError_t krylov_iteration(const GridGeom& g, long long n, bool mixed, const KrylovWork& w, bool line,
                             cudaStream_t st) {
    if (mixed) return g.diag ? iteration<float, true>(g, n, w, line, st) : iteration<float, false>(g, n, w, line, st);
    return g.diag ? iteration<double, true>(g, n, w, line, st) : iteration<double, false>(g, n, w, line, st);
}

cudaError_t krylov_add_delta(long long n, bool mixed, void* p, const double* d, cudaStream_t st) {
    if (mixed) k_add_delta<float><<<vec_blocks(n), kThreads, 0, st>>>(n, (float*)p, d);
    else k_add_delta<double><<<vec_blocks(n), kThreads, 0, st>>>(n, (double*)p, d);
    return cudaGetLastError();
}

}  // namespace tpfa
