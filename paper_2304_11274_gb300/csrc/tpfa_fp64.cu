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
// 6 links 615 -> 234 us, the adjoint of 97 x 83 x 50 436 -> 135 us, R alone there
// 283 -> 71 us.  Three blocks per multiprocessor (80 registers, a few spilled
// values) instead of two: 3.39 -> 3.13 ms for R + J, the adjoint the other way
// round (380 against 383 us for the whole gradient call).
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

// One cell's sums over its links.
template <Op64 OP>
struct Sums {
    RowAccD row;
    double acc = 0.0;                                // J w: sum dF/dp_L (w_L - w_K); adjoint: g_p
    double gx = 0.0, gy = 0.0, gz = 0.0, gd = 0.0;  // adjoint: sum F (v_K - v_L) T per link direction

    // dv: w_L - w_K or v_K - v_L; vL: v_L; lt: the link from L's side at a tie
    template <int S, bool FLAT>
    __device__ __forceinline__ void add(const LinkOut<double>& l, double T, double dv) {
        if constexpr (OP == Op64::Jacobian) row.add<true, FLAT>(l);
        if constexpr (OP == Op64::Residual) row.add<false, FLAT>(l);
        if constexpr (OP == Op64::Jvp) {
            row.add<false, FLAT>(l);
            acc = __fma_rn(l.Db, dv, acc);
        }
        if constexpr (OP == Op64::Vjp) {
            acc = __fma_rn(l.Da, dv, acc);
            const double h = __dmul_rn(l.F, dv);
            double& s = (S == 0 || S == 10) ? gz : (S == 2 || S == 8) ? gy : (S == 4 || S == 6) ? gx : gd;
            s = __fma_rn(h, T, s);
        }
    }
    // adjoint: v_L (dF_KL/dp_K + dF_LK/dp_K) of a tie (zero otherwise)
    __device__ __forceinline__ void tie(double Da, double Db_other, double vL) {
        acc = __fma_rn(vL, __dadd_rn(Da, Db_other), acc);
    }
};

template <Op64 OP, bool DIAG, bool CRK>
__global__ void __launch_bounds__(kMaxThreads, OP == Op64::Vjp ? 2 : 3) k_cells_fp64(const Args64 a) {
    constexpr bool JAC = OP == Op64::Jacobian, JVP = OP == Op64::Jvp, VJP = OP == Op64::Vjp;
    constexpr bool DIR = JVP || VJP;
    constexpr int NF = DIR ? 4 : 3;         // tile fields: p, depth, mobility, direction
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
        }
    };

    CellVal<double> me = load_cell(own + nxy * kA);
    double dme = DIR ? a.dir[own + nxy * kA] : 0.0;
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
        zl_other = up.Db;
    }
    if (in) {
        put_cell(sm64 + (kA & 1) * NF * NP, sp, me);
        if (DIR) sm64[((kA & 1) * NF + 3) * NP + sp] = dme;
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
        double dup = dme;
        if (zp) {
            up = load_cell(c + nxy);
            if (DIR) dup = a.dir[c + nxy];
        }

        // staging position of this row's values
        const int ey = (int)ym + (int)yp, ez = (int)zm + (int)zp;
        const int per = 1 + ey + ez, perx = 1 + g.diag * ey;
        double* const row = stage0 + (k & 1) * cells * L + ly * TX * L + lx * per +
                            (int)(axis_links_before(i, nx) - axis_links_before(i0, nx)) * perx;

        Sums<OP> sum;
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
                    if (VJP && zero_flux(l)) sum.tie(l.Da, link(q, T[S], nb, me).Db, dn);
                }
                sum.template add<S, FLAT>(l, T[S], dv);
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
            sum.template add<0, false>(zl, Tzm, ddn);
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
            sum.template add<10, false>(l, Tz, dv);
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
                // k_L / (k_K + k_L) = T (d/A) / (2 k_K); an impermeable cell's links have T = 0
                const double kk = a.kperm[c];
                double gk = __dmul_rn(sum.gx, a.lg.cx);
                gk = __fma_rn(sum.gy, a.lg.cy, gk);
                gk = __fma_rn(sum.gz, a.lg.cz, gk);
                gk = __fma_rn(sum.gd, a.lg.cd, gk);
                gk = gk != 0.0 ? gk / (2.0 * kk) : 0.0;
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
            }
            fill_rim(N, k + 1);
        }
        me = up;
        dme = dup;
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
    constexpr int NF = OP == Op64::Jvp || OP == Op64::Vjp ? 4 : 3, L = DIAG ? 11 : 7;
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
