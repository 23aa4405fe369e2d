// tpfa_fp64.cu -- the FP64 path on structured grids: residual, residual +
// Jacobian, J w and adjoint (sm_103a).
//
// GB300 does two FP64 operations per clock and multiprocessor: a warp's FP64
// instruction holds its scheduler's pipe for 64 cycles, so everything else
// (integer work, shared memory, loads) is free as long as it runs beside it,
// and the time is the number of FP64 instructions.  The kernel below is
// arranged around that count:
//
//   * densities: a block owns a tile of TX x TY cells (one thread each) and
//     walks a run of z-planes; p, depth and mobility of the tile and of its
//     one-cell rim sit in shared memory, so a mobility is evaluated about 1.3
//     times per cell instead of once per neighbour;
//   * in-plane links are evaluated from both ends (6 FP64 operations each with
//     its sums; exchanging them would save three and cost the tile's rim), the
//     vertical link once: a thread carries it from plane k to plane k + 1 and
//     takes it from its other end there (flip(), or link() again at an exact
//     tie, where the ends disagree);
//   * neighbours at the same depth (any flat layer) skip the gravity terms: a
//     warp whose valid in-plane links are all flat takes that path, with the
//     same bits (link_d);
//   * the diagonal is summed from the off-diagonals (RowAccD);
//   * lanes past the end of a row cost as much as others, so TX and TY are
//     chosen per grid to fill the warps (tile_shape), and the run length to
//     fill the multiprocessors evenly (run_length).
//
// Double buffers: plane k + 1 is written into one half of the tile (and of the
// CSR staging rows) while plane k is read from the other, one block barrier per
// plane.  Measured against the kernels before it (a 32-lane y-march for the
// assembly, one thread per cell with a density per neighbour for J w and the
// adjoint): R + J of 256^3, 10 links 7.79 -> 3.13 ms (95 FP64 operations per cell
// instead of 230, at 84 % of the pipe's rate), of 32^3, 6 links 223 -> 12.3 us (one
// plane per block instead of a serial march of 32 rows), J w of 161 x 119 x 67,
// 6 links 615 -> 234 us, the adjoint call of 97 x 83 x 50, 10 links 449 -> 160 us (142
// with k_L / (k_K + k_L) from T alone: see Perm), R alone there 283 -> 71 us.  Three
// blocks per multiprocessor (80 registers, a few spilled values) instead of two:
// 3.39 -> 3.13 ms for R + J; the adjoint needs the registers of two.
//
// The rows are those of naive_row<double> bit for bit (same link, same sums in
// slot order).
#include <cuda_runtime.h>

#include <type_traits>

#include "tpfa_impl.h"
#include "tpfa_row.cuh"
#include "tpfa_tile.h"

namespace tpfa {

namespace {

enum class Op64 { Jacobian, Residual, Jvp, Vjp };

constexpr int kMaxThreads = 256;

struct Args64 {
    GridGeom g;
    PhysD q;
    AsmFields<double> f;
    AsmOut<double> o;
    int TX, TY;           // tile
    int bx, by;           // tiles along x and y
    int run, k0, k1;      // planes per block; planes [k0, k1) of the grid
    const double* dir;    // w (J w) or v (adjoint)
    double* out;          // J w or g_p
    double* g_lnk;        // adjoint, or null
    const double* kperm;  // adjoint
    LinkGeoD lg;          // adjoint
};

// The adjoint's k_L / (k_K + k_L) of a link without a division: T (d/A) / (2 k_K)
// is that ratio but for T's four roundings, and for the ones of (d/A) / (2 k_K);
// one correction by its remainder takes them out again,
//   q0 = T (d/A) / (2 k_K),  q = q0 + q0 (k_L - (k_K + k_L) q0) / k_L,
// the last quotient in FP32: it is below 2^-38, or the division is taken.  Four
// FP64 operations per link.  Against 80-bit values, 10 links, log-normal k, the
// sums' error in the 2-norm is 1.77e-16, with the rounded quotient 1.95e-16,
// with q0 alone 2.35e-16.
struct Perm {
    double k = 0.0, cx = 0.0, cy = 0.0, cz = 0.0, cd = 0.0;  // k_K, (d/A) / (2 k_K)
    // x 2^60 as FP32 (m^2 are small numbers); NaN from x = 2^65 on
    static __device__ __forceinline__ float up60(double x) {
        const float r = narrow_flush(__hiloint2double(__double2hiint(x) + (60 << 20), __double2loint(x)));
        return abs_hi(x) < 0x44000000u ? r : __int_as_float(0x7fffffff);
    }
    __device__ __forceinline__ void set(const LinkGeoD& lg, double kK) {
        k = kK;
        // 1 / (2 k) to about 2^-44: any error is corrected per link
        const double y = widen_flush(__fmul_rn(rcp_approx(up60(kK)), 0.5f));
        const double y60 = __hiloint2double(y != 0.0 ? __double2hiint(y) + (60 << 20) : 0, __double2loint(y));
        const double i2k = __fma_rn(y60, __fma_rn(-2.0 * k, y60, 1.0), y60);
        cx = __dmul_rn(lg.cx, i2k), cy = __dmul_rn(lg.cy, i2k), cz = __dmul_rn(lg.cz, i2k), cd = __dmul_rn(lg.cd, i2k);
    }
    // ok: false for k = 0 (a link without flux, T = 0) and outside up60's range
    template <int S>
    __device__ __forceinline__ double ratio(double T, double kL, bool& ok) const {
        const double q0 = __dmul_rn(T, (S == 0 || S == 10) ? cz : (S == 2 || S == 8) ? cy : (S == 4 || S == 6) ? cx : cd);
        const double rem = __fma_rn(-kL, q0, __fma_rn(-k, q0, kL));
        const float kf = up60(kL), d = __fmul_rn(up60(rem), rcp_approx(kf));
        ok = fabsf(d) <= 0x1p-38f && kf >= 0x1p-60f;
        return ok ? __fma_rn(q0, widen_flush(d), q0) : 0.0;
    }
};

// The sum over cell (i, j, k)'s links with divisions, from global memory: for the
// rows with a permeability outside ratio()'s range.
__device__ __noinline__ double lnk_by_division(const Args64& a, int i, int j, int k) {
    const int nx = a.g.nx, nxy = nx * a.g.ny, c = i + nx * j + nxy * k;
    const unsigned mask = slot_mask(a.g, i, j, k);
    const CellVal<double> me = make_cell(a.q, a.f.p[c], a.f.z[c]);
    double sum = 0.0;
#pragma unroll 1
    for (int s = 0; s < NSLOT; ++s) {
        // a link that does not exist is formed from the cell itself: every address is in range
        const bool there = s != SLOT_SELF && ((mask >> s) & 1u);
        const bool z = s == 0 || s == 10;
        const int x = z ? 0 : (s - 1) % 3 - 1, y = z ? 0 : (s - 1) / 3 - 1;
        const int d = !there ? c : s == 0 ? c - nxy : s == 10 ? c + nxy : c + x + nx * y;
        const double* T = z ? a.f.Tz : x == 0 ? a.f.Ty : y == 0 ? a.f.Tx : x == y ? a.f.Tpp : a.f.Tmp;
        const double F = link(a.q, T[s < SLOT_SELF ? d : c], me, make_cell(a.q, a.f.p[d], a.f.z[d])).F;
        const double kk = __dadd_rn(a.kperm[c], a.kperm[d]);
        const double ratio = kk > 0.0 ? a.kperm[d] / kk : 0.0;
        if (there) sum = __fma_rn(__dmul_rn(F, __dsub_rn(a.dir[c], a.dir[d])), ratio, sum);
    }
    return sum;
}

// One cell's sums over its links.
template <Op64 OP>
struct Sums {
    RowAccD row;
    double acc = 0.0;  // J w: sum dF/dp_L (w_L - w_K); adjoint: g_p
    double lnk = 0.0;  // adjoint: sum F (v_K - v_L) k_L / (k_K + k_L)
    bool divide = false;  // ... a ratio of which has to be divided

    // dv: w_L - w_K or v_K - v_L; adjoint: T and k_L of the link (0 if g_lnk is not wanted)
    template <int S, bool FLAT>
    __device__ __forceinline__ void add(const LinkOut<double>& l, double T, double dv, const Perm& pm, double kL) {
        if constexpr (OP == Op64::Jacobian) row.add<true, FLAT>(l);
        if constexpr (OP == Op64::Residual) row.add<false, FLAT>(l);
        if constexpr (OP == Op64::Jvp) {
            row.add<false, FLAT>(l);
            acc = __fma_rn(l.Db, dv, acc);
        }
        if constexpr (OP == Op64::Vjp) {
            acc = __fma_rn(l.Da, dv, acc);
            bool ok;
            lnk = __fma_rn(__dmul_rn(l.F, dv), pm.ratio<S>(T, kL, ok), lnk);
            divide = divide || !(ok || zero_flux(l));
        }
    }
    // adjoint: v_L (dF_KL/dp_K + dF_LK/dp_K) of a tie (zero otherwise)
    __device__ __forceinline__ void tie(double Da, double Db_other, double vL) {
        acc = __fma_rn(vL, __dadd_rn(Da, Db_other), acc);
    }
};

template <Op64 OP, bool DIAG, bool CRK>
__global__ void __launch_bounds__(kMaxThreads, OP == Op64::Vjp ? 2 : 3) k_cells_fp64(const __grid_constant__ Args64 a) {
    constexpr bool JAC = OP == Op64::Jacobian, JVP = OP == Op64::Jvp, VJP = OP == Op64::Vjp;
    constexpr bool DIR = JVP || VJP;
    constexpr int NF = VJP ? 5 : DIR ? 4 : 3;  // tile fields: p, depth, mobility, direction, k
    constexpr int L = DIAG ? 11 : 7;        // values of an interior row
    extern __shared__ __align__(16) double sm64[];
    const GridGeom& g = a.g;
    const PhysD& q = a.q;
    const int nx = g.nx, ny = g.ny, nxy = nx * ny;
    const int TX = a.TX, TY = a.TY, PX = TX + 2, NP = PX * (TY + 2);
    const int t = threadIdx.x, nt = blockDim.x, cells = TX * TY;
    double* const stage0 = sm64 + 2 * NF * NP;  // two buffers of cells * L values

    unsigned b = blockIdx.x;
    const int i0 = (int)(b % (unsigned)a.bx) * TX;
    b /= (unsigned)a.bx;
    const int j0 = (int)(b % (unsigned)a.by) * TY;
    const int kA = a.k0 + (int)(b / (unsigned)a.by) * a.run, kB = min(kA + a.run, a.k1);

    // this thread's cell; a thread without one works on a cell of the grid and
    // stores nothing, so every address formed is in range
    const bool in = t < cells;
    const int ly = in ? t / TX : 0, lx = in ? t - ly * TX : 0;
    const int i = min(i0 + lx, nx - 1), j = min(j0 + ly, ny - 1);
    const bool act = in && i0 + lx < nx && j0 + ly < ny;
    const int own = i + nx * j;
    const int sp = (ly + 1) * PX + lx + 1;
    const bool xm = i > 0, xp = i + 1 < nx, ym = j > 0, yp = j + 1 < ny;

    const bool lnk = VJP && a.g_lnk;
    auto load_cell = [&](int c) { return make_cell(q, a.f.p[c], a.f.z[c]); };
    auto put_cell = [&](double* P, int s, const CellVal<double>& v) {
        P[s] = v.p;
        P[NP + s] = v.z;
        P[2 * NP + s] = v.lam;
    };
    // the tile's rim on plane k: rows -1 and TY, columns -1 and TX
    auto fill_rim = [&](double* P, int k) {
        for (int h = t; h < 2 * PX + 2 * TY; h += nt) {
            int x, y;
            if (h < 2 * PX) {
                y = h < PX ? 0 : TY + 1;
                x = h < PX ? h : h - PX;
            } else {
                y = 1 + (h - 2 * PX) / 2;
                x = ((h - 2 * PX) & 1) ? TX + 1 : 0;
            }
            const int ci = min(max(i0 + x - 1, 0), nx - 1), cj = min(max(j0 + y - 1, 0), ny - 1);
            const int c = ci + nx * cj + nxy * k;
            put_cell(P, y * PX + x, load_cell(c));
            if (DIR) P[3 * NP + y * PX + x] = a.dir[c];
            if (VJP && lnk) P[4 * NP + y * PX + x] = a.kperm[c];
        }
    };

    CellVal<double> me = load_cell(own + nxy * kA);
    double dme = DIR ? a.dir[own + nxy * kA] : 0.0;
    double kme = VJP && lnk ? a.kperm[own + nxy * kA] : 0.0, kdn = 0.0;  // k of this cell and the one below
    // the vertical link below this plane, from this cell's side
    LinkOut<double> zl{};
    double Tzm = 0.0, ddn = 0.0;  // its T; the direction's difference (and v_L, tie partner) for it
    double vdn = 0.0, zl_other = 0.0;
    if (kA > 0) {
        const int c = own + nxy * (kA - 1);
        const CellVal<double> dn = load_cell(c);
        Tzm = a.f.Tz[c];
        const LinkOut<double> up = link(q, Tzm, dn, me);
        zl = zero_flux(up) ? link(q, Tzm, me, dn) : flip(up);
        if (DIR) {
            vdn = a.dir[c];
            ddn = JVP ? __dsub_rn(vdn, dme) : __dsub_rn(dme, vdn);
        }
        if (VJP && lnk) kdn = a.kperm[c];
        zl_other = up.Db;
    }
    if (in) {
        put_cell(sm64 + (kA & 1) * NF * NP, sp, me);
        if (DIR) sm64[((kA & 1) * NF + 3) * NP + sp] = dme;
        if (VJP && lnk) sm64[((kA & 1) * NF + 4) * NP + sp] = kme;
    }
    fill_rim(sm64 + (kA & 1) * NF * NP, kA);

    // the staged CSR rows of plane k, one contiguous stretch per tile row
    auto write_rows = [&](int k) {
        const double* S = stage0 + (k & 1) * cells * L;
        const int iend = min(i0 + TX, nx);
        for (int r = t >> 5; r < TY && j0 + r < ny; r += nt >> 5) {
            const long long s0 = row_start(g, i0, j0 + r, k);
            const int len = (int)(row_start(g, iend, j0 + r, k) - s0);
            double* dst = a.o.vals + s0;
            for (int e = t & 31; e < len; e += 32) dst[e] = S[r * TX * L + e];
        }
    };

    for (int k = kA; k < kB; ++k) {
        double* const P = sm64 + (k & 1) * NF * NP;
        __syncthreads();  // plane k's tile and plane k - 1's staged rows are complete
        if (JAC && k > kA) write_rows(k - 1);
        const int c = own + nxy * k;
        const bool zm = k > 0, zp = k + 1 < g.nz;
        unsigned mask = (1u << SLOT_SELF) | (unsigned)zm | (unsigned)ym << 2 | (unsigned)xm << 4 | (unsigned)xp << 6 |
                        (unsigned)yp << 8 | (unsigned)zp << 10;
        if (DIAG)
            mask |= (unsigned)(xm && ym) << 1 | (unsigned)(xp && ym) << 3 | (unsigned)(xm && yp) << 7 |
                    (unsigned)(xp && yp) << 9;
        const double pn = a.f.pn[c], mn = a.f.mn[c], phi = CRK ? a.f.phi0[c] : 0.0, Tz = a.f.Tz[c];
        double T[NSLOT];
        T[2] = a.f.Ty[ym ? c - nx : c];
        T[4] = a.f.Tx[xm ? c - 1 : c];
        T[6] = a.f.Tx[c];
        T[8] = a.f.Ty[c];
        if (DIAG) {
            T[1] = a.f.Tpp[xm && ym ? c - nx - 1 : c];
            T[3] = a.f.Tmp[xp && ym ? c - nx + 1 : c];
            T[7] = a.f.Tmp[c];
            T[9] = a.f.Tpp[c];
        }
        // the cell above: the vertical link's other end now, this thread's cell next
        CellVal<double> up = me;
        double dup = dme, kup = kme;
        if (zp) {
            up = load_cell(c + nxy);
            if (DIR) dup = a.dir[c + nxy];
            if (VJP && lnk) kup = a.kperm[c + nxy];
        }

        // staging position of this row's values
        const int ey = (int)ym + (int)yp, ez = (int)zm + (int)zp;
        const int per = 1 + ey + ez, perx = 1 + g.diag * ey;
        double* const row = stage0 + (k & 1) * cells * L + ly * TX * L + lx * per +
                            (int)(axis_links_before(i, nx) - axis_links_before(i0, nx)) * perx;

        Sums<OP> sum;
        Perm pm;
        if (VJP && lnk) pm.set(a.lg, kme);
        auto neighbour = [&](int s) {
            return CellVal<double>{P[s], P[NP + s], P[2 * NP + s]};
        };
        auto slot = [&](auto flat, auto slot_c, int off) {
            constexpr int S = decltype(slot_c)::value;
            constexpr bool FLAT = decltype(flat)::value;
            if (mask & (1u << S)) {
                const CellVal<double> nb = neighbour(sp + off);
                const LinkOut<double> l = link_d<FLAT>(q, T[S], me, nb);
                double dv = 0.0;
                if (DIR) {
                    const double dn = P[3 * NP + sp + off];
                    dv = JVP ? __dsub_rn(dn, dme) : __dsub_rn(dme, dn);
                    // (a flat tie has equal pressures: its term is zero)
                    if (VJP && !FLAT && zero_flux(l)) sum.tie(l.Da, link(q, T[S], nb, me).Db, dn);
                }
                sum.template add<S, FLAT>(l, T[S], dv, pm, VJP && lnk ? P[4 * NP + sp + off] : 0.0);
                if (JAC && act) row[slot_pos(mask, S)] = l.Db;
            }
        };
        using std::integral_constant;
        auto in_plane = [&](auto flat) {
            if (DIAG) slot(flat, integral_constant<int, 1>{}, -PX - 1);
            slot(flat, integral_constant<int, 2>{}, -PX);
            if (DIAG) slot(flat, integral_constant<int, 3>{}, -PX + 1);
            slot(flat, integral_constant<int, 4>{}, -1);
            slot(flat, integral_constant<int, 6>{}, 1);
            if (DIAG) slot(flat, integral_constant<int, 7>{}, PX - 1);
            slot(flat, integral_constant<int, 8>{}, PX);
            if (DIAG) slot(flat, integral_constant<int, 9>{}, PX + 1);
        };

        if (zm) {  // slot 0
            sum.template add<0, false>(zl, Tzm, ddn, pm, kdn);
            if (VJP && zero_flux(zl)) sum.tie(zl.Da, zl_other, vdn);
            if (JAC && act) row[0] = zl.Db;
        }
        // rim cells are clamped copies where the neighbour does not exist, so
        // all eight (four) may be tested
        bool flat = link_flat(me, neighbour(sp - 1)) && link_flat(me, neighbour(sp + 1)) &&
                    link_flat(me, neighbour(sp - PX)) && link_flat(me, neighbour(sp + PX));
        if (DIAG)
            flat = flat && link_flat(me, neighbour(sp - PX - 1)) && link_flat(me, neighbour(sp - PX + 1)) &&
                   link_flat(me, neighbour(sp + PX - 1)) && link_flat(me, neighbour(sp + PX + 1));
        if (__all_sync(0xffffffffu, flat)) in_plane(integral_constant<bool, true>{});
        else in_plane(integral_constant<bool, false>{});
        if (zp) {  // slot 10, and the next plane's slot 0
            const LinkOut<double> l = link(q, Tz, me, up);
            const bool tie = zero_flux(l);
            zl = tie ? link(q, Tz, up, me) : flip(l);
            double dv = 0.0;
            if (DIR) dv = JVP ? __dsub_rn(dup, dme) : __dsub_rn(dme, dup);
            sum.template add<10, false>(l, Tz, dv, pm, kup);
            if (VJP && tie) sum.tie(l.Da, zl.Db, dup);
            if (JAC && act) row[slot_pos(mask, 10)] = l.Db;
            Tzm = Tz;
            ddn = -dv;
            vdn = dme;
            zl_other = l.Db;
        }

        const AccD A = accumulation<CRK>(q, me.p, pn, mn, me.lam, phi);
        bool bad = false;
        if constexpr (JAC) {
            const double R = __dadd_rn(sum.row.F, A.A), d = sum.row.diagonal(q, A.dA);
            bad = nonfinite(R) || nonfinite(d);
            if (act) {
                row[slot_pos(mask, SLOT_SELF)] = d;
                if (a.o.R) a.o.R[c] = R;
            }
        } else if constexpr (OP == Op64::Residual) {
            const double R = __dadd_rn(sum.row.F, A.A);
            bad = nonfinite(R);
            if (act) a.o.R[c] = R;
        } else if constexpr (JVP) {
            const double jw = __fma_rn(sum.row.excess(q, A.dA), dme, sum.acc);
            bad = nonfinite(jw);
            if (act) a.out[c] = jw;
            if (a.o.R) {
                const double R = __dadd_rn(sum.row.F, A.A);
                bad = bad || nonfinite(R);
                if (act) a.o.R[c] = R;
            }
        } else {
            const double gp = __fma_rn(dme, A.dA, sum.acc);
            bad = nonfinite(gp);
            if (act) a.out[c] = gp;
            if (a.g_lnk) {
                const double gk = act && sum.divide ? lnk_by_division(a, i, j, k) : sum.lnk;
                bad = bad || nonfinite(gk);
                if (act) a.g_lnk[c] = gk;
            }
        }
        if (act && bad) atomicOr(a.o.status, STATUS_NONFINITE);

        if (k + 1 < kB) {  // the next plane's tile
            double* const N = sm64 + ((k + 1) & 1) * NF * NP;
            if (in) {
                put_cell(N, sp, up);
                if (DIR) N[3 * NP + sp] = dup;
                if (VJP && lnk) N[4 * NP + sp] = kup;
            }
            fill_rim(N, k + 1);
        }
        me = up;
        dme = dup;
        kdn = kme;
        kme = kup;
    }
    if (JAC) {
        __syncthreads();
        write_rows(kB - 1);
    }
}

// Planes per block: a longer run saves its first plane's extra vertical link
// and density (about 25 operations against 80 per plane), a shorter one
// spreads the blocks evenly.  The busiest multiprocessor's work is minimised;
// a block that runs there alone takes about a third longer than one of a pair.
int run_length(long long tiles, int planes, int sms) {
    int best = 1;
    double cost = 1e300;
    for (int r = 1; r <= 32 && r <= planes; ++r) {
        const long long n = (tiles * ((planes + r - 1) / r) + sms - 1) / sms;
        const double c = ((double)n + (n & 1) * 0.35) * (80.0 * r + 25.0);
        if (c < cost) cost = c, best = r;
    }
    return best;
}

template <Op64 OP, bool DIAG, bool CRK>
cudaError_t launch64(Args64& a, cudaStream_t st) {
    constexpr int NF = OP == Op64::Vjp ? 5 : OP == Op64::Jvp ? 4 : 3, L = DIAG ? 11 : 7;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    tile_shape(a.g.nx, a.g.ny, kMaxThreads, a.TX, a.TY);
    a.bx = (a.g.nx + a.TX - 1) / a.TX;
    a.by = (a.g.ny + a.TY - 1) / a.TY;
    const int planes = a.k1 - a.k0;
    a.run = run_length((long long)a.bx * a.by, planes, sms);
    const long long blocks = (long long)a.bx * a.by * ((planes + a.run - 1) / a.run);
    if (blocks >= (1LL << 31)) return cudaErrorInvalidConfiguration;
    const int threads = (a.TX * a.TY + 31) / 32 * 32;
    const int np = (a.TX + 2) * (a.TY + 2);
    const int smem = 8 * (2 * NF * np + (OP == Op64::Jacobian ? 2 * a.TX * a.TY * L : 0));
    // the limit for the largest tile: (TX + 2)(TY + 2) with TX TY <= 256 is largest for one row or column
    constexpr int most = 8 * (2 * NF * 3 * (kMaxThreads + 2) + (OP == Op64::Jacobian ? 2 * kMaxThreads * L : 0));
    e = ensure_smem_limit(reinterpret_cast<const void*>(&k_cells_fp64<OP, DIAG, CRK>), most);
    if (e != cudaSuccess) return e;
    k_cells_fp64<OP, DIAG, CRK><<<(unsigned)blocks, threads, smem, st>>>(a);
    return cudaGetLastError();
}

template <Op64 OP>
cudaError_t launch64_op(Args64& a, bool crk, cudaStream_t st) {
    if (a.g.diag) return crk ? launch64<OP, true, true>(a, st) : launch64<OP, true, false>(a, st);
    return crk ? launch64<OP, false, true>(a, st) : launch64<OP, false, false>(a, st);
}

Args64 args64(const GridGeom& g, const PhysD& q, const AsmFields<double>& f, const AsmOut<double>& o) {
    Args64 a{};
    a.g = g, a.q = q, a.f = f, a.o = o;
    a.k0 = 0, a.k1 = g.nz;
    return a;
}

}  // namespace

cudaError_t launch_cells_fp64(const GridGeom& g, const PhysD& q, bool crk, const AsmFields<double>& f,
                              const AsmOut<double>& o, cudaStream_t st, int k0, int k1) {
    Args64 a = args64(g, q, f, o);
    a.k0 = k0, a.k1 = k1;
    return o.vals ? launch64_op<Op64::Jacobian>(a, crk, st) : launch64_op<Op64::Residual>(a, crk, st);
}

cudaError_t launch_jvp_fp64(const GridGeom& g, const PhysD& q, bool crk, const AsmFields<double>& f, const double* w,
                            double* Jw, double* R, unsigned int* status, cudaStream_t st) {
    Args64 a = args64(g, q, f, AsmOut<double>{R, nullptr, nullptr, status});
    a.dir = w, a.out = Jw;
    return launch64_op<Op64::Jvp>(a, crk, st);
}

cudaError_t launch_vjp_fp64(const GridGeom& g, const PhysD& q, bool crk, const AsmFields<double>& f,
                            const double* kperm, const LinkGeoD& lg, const double* v, double* g_p, double* g_lnk,
                            unsigned int* status, cudaStream_t st) {
    Args64 a = args64(g, q, f, AsmOut<double>{nullptr, nullptr, nullptr, status});
    a.dir = v, a.out = g_p, a.g_lnk = g_lnk, a.kperm = kperm, a.lg = lg;
    return launch64_op<Op64::Vjp>(a, crk, st);
}

}  // namespace tpfa
