// tpfa_mesh.cu -- residual and Jacobian of Eq. vk on a general mesh given as a
// list of connections (K, L, Upsilon_KL), the extension to arbitrary mesh
// topologies (corner-point grids with faults, unstructured meshes) that the
// paper names as future work (Section 8).  sm_103a.
//
// Gather form: one thread per row K walks row K of the pattern (columns
// ascending) and evaluates every link from K's side with the same link() and
// accumulation() arithmetic as the structured kernels, so a structured grid
// passed as a connection list sums in the same (ascending-column) order.  No
// atomics: each link is evaluated once from each side (bit-exact
// antisymmetry of F).  A block's 128 rows own one contiguous stretch of the
// CSR arrays: its columns and T are read into shared memory, and its values
// written from there, with consecutive lanes (read by the rows themselves, 44
// bytes apart, they cost eleven L1 wavefronts per load instead of one); each
// value takes the place of its T.  Rows longer than the buffer fall back to
// direct access.  Neighbour gathers go through a checked index, one entry ahead.
// Measured (mixed, 10 links): a faulted mesh of 1.75 M cells 98.7 -> 86.4 us,
// of 0.42 M cells 30.7 -> 28.7 us; issue bound (about 116 instructions per entry:
// the link, the neighbour's density, the Kahan sums).  Two entries at a time
// as FP32x2 pairs were slower (92 us: register pairs to assemble, fewer warps).
#include <cuda_runtime.h>

#include <type_traits>

#include "tpfa_impl.h"
#include "tpfa_row.cuh"

namespace tpfa {

namespace {

constexpr int kRows = 128;
constexpr int kStage = kRows * 16;  // staged CSR entries per block

template <typename Real, bool CRK, bool JAC>
__global__ void __launch_bounds__(kRows) k_mesh_assemble(MeshFields<Real> f, long long n,
                                                         typename PhysOf<Real>::type q, AsmOut<Real> o) {
    __shared__ Real stage[kStage];  // the block's T, each replaced by its value
    __shared__ int cols[kStage];
    const long long r0 = (long long)blockIdx.x * kRows;
    const long long r = r0 + threadIdx.x;
    const long long rl = min(r0 + kRows, n);
    const long long e0 = f.row_ptr[r0], e1 = f.row_ptr[rl];
    const bool staged = (e1 - e0) <= kStage;  // block-uniform
    if (staged) {
        const int len = (int)(e1 - e0);
        const int* col = f.col + e0;
        const Real* Tc = f.Tc + e0;
#pragma unroll 4
        for (int e = threadIdx.x; e < len; e += kRows) {
            cols[e] = __ldg(col + e);
            stage[e] = __ldg(Tc + e);
        }
        __syncthreads();
    }
    if (r < n) {
        const long long rs = f.row_ptr[r], re = f.row_ptr[r + 1];
        const int a = (int)(rs - e0), b = (int)(re - e0);  // the row within the block's stretch
        const CellVal<Real> me = make_cell(q, f.p[r], f.z[r]);
        RowSums out;
        const int self = (int)r;
        // p and z of cell c; an index outside the mesh is recorded and reads nothing
        auto gather = [&](int c, Real& pv, Real& zv) {
            const bool ok = (unsigned)c < (unsigned)n;
            if (!ok) atomicOr(o.status, STATUS_DEVICE_CHECK);
            pv = ok ? __ldg(f.p + c) : Real(0);
            zv = ok ? __ldg(f.z + c) : Real(0);
        };
        auto row = [&](auto in_smem) {
            constexpr bool SMEM = decltype(in_smem)::value;
            // entry e of the block's stretch
            auto col_of = [&](int e) { return SMEM ? cols[e] : f.col[e0 + e]; };
            auto T_of = [&](int e) { return SMEM ? stage[e] : f.Tc[e0 + e]; };
            auto put = [&](int e, Real v) {
                if (SMEM) stage[e] = v;
                else o.vals[e0 + e] = v;
            };
            int dpos = a;
            if constexpr (sizeof(Real) == 4) {
                // the next neighbour is on its way while this link is
                // evaluated; F and dF/dp_K share one FP32x2 Kahan sum
                Kahan2 sum;
                int c = col_of(a);
                float pv, zv;
                gather(c, pv, zv);
                for (int e = a; e < b; ++e) {
                    const int cc = c;
                    const CellVal<float> nb = make_cell(q, pv, zv);
                    if (e + 1 < b) {
                        c = col_of(e + 1);
                        gather(c, pv, zv);
                    }
                    if (cc == self) {
                        dpos = e;
                    } else {
                        const LinkOut<float> L = link(q, T_of(e), me, nb);
                        sum.add(f2(L.F, JAC ? L.Da : 0.f));
                        if (JAC) put(e, L.Db);
                    }
                }
                const AccF acc = accumulation<CRK>(q, me.p, f.pn[r], f.mn[r], me.rho, CRK ? f.phi0[r] : 0.f);
                out.R = __dadd_rn(__dadd_rn(acc.A, widen(sum.s.x)), -widen(sum.c.x));
                out.diag64 = 0.0;
                if (JAC) {
                    Kahan32 d{sum.s.y, sum.c.y};
                    d.add(acc.dA);
                    out.diag64 = __dadd_rn(widen(d.s), -widen(d.c));
                    put(dpos, __fsub_rn(d.s, d.c));
                }
            } else {
                RowAccD sum;
                for (int e = a; e < b; ++e) {
                    const int c = col_of(e);
                    if (c == self) {
                        dpos = e;
                        continue;
                    }
                    double pv, zv;
                    gather(c, pv, zv);
                    const LinkOut<double> L = link(q, T_of(e), me, make_cell(q, pv, zv));
                    sum.add<JAC>(L);
                    if (JAC) put(e, L.Db);
                }
                const AccD acc = accumulation<CRK>(q, me.p, f.pn[r], f.mn[r], me.lam, CRK ? f.phi0[r] : 0.0);
                out.R = __dadd_rn(sum.F, acc.A);
                out.diag64 = 0.0;
                if (JAC) {
                    out.diag64 = sum.diagonal(q, acc.dA);
                    put(dpos, out.diag64);
                }
            }
        };
        if (staged) row(std::integral_constant<bool, true>{});
        else row(std::integral_constant<bool, false>{});
        if (o.R) o.R[r] = out.R;
        if (JAC && o.diag64) o.diag64[r] = out.diag64;
        if (nonfinite(out.R) || (JAC && nonfinite(out.diag64))) atomicOr(o.status, STATUS_NONFINITE);
    }
    if (JAC && staged) {
        __syncthreads();
        const int len = (int)(e1 - e0);
        Real* vals = o.vals + e0;
        for (int e = threadIdx.x; e < len; e += kRows) vals[e] = stage[e];
    }
}

// (V / dt) phi0 per cell in FP64, and in the field type when c_r != 0.
template <typename Real>
__global__ void k_mesh_vphi(long long n, double inv_dt, const double* __restrict__ V, const double* __restrict__ poro,
                            double* vphi_d, Real* vphi_r) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const double v = (V[c] * inv_dt) * poro[c];
        vphi_d[c] = v;
        if (vphi_r) vphi_r[c] = (Real)v;
    }
}

unsigned blocks_of(long long n, int per) {
    long long b = (n + per - 1) / per;
    return (unsigned)(b < 1 ? 1 : (b > (1LL << 30) ? (1LL << 30) : b));
}

template <typename Real>
cudaError_t launch_mesh_t(const MeshFields<Real>& f, long long n, const typename PhysOf<Real>::type& q, bool crk,
                          const AsmOut<Real>& o, cudaStream_t st) {
    const unsigned nb = (unsigned)((n + kRows - 1) / kRows);
    const bool jac = o.vals != nullptr;
    if (crk) {
        if (jac) k_mesh_assemble<Real, true, true><<<nb, kRows, 0, st>>>(f, n, q, o);
        else k_mesh_assemble<Real, true, false><<<nb, kRows, 0, st>>>(f, n, q, o);
    } else {
        if (jac) k_mesh_assemble<Real, false, true><<<nb, kRows, 0, st>>>(f, n, q, o);
        else k_mesh_assemble<Real, false, false><<<nb, kRows, 0, st>>>(f, n, q, o);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_mesh_vphi(long long n, double dt, bool mixed, const double* V, const double* poro,
                             double* vphi_d, void* vphi_r, cudaStream_t st) {
    if (mixed)
        k_mesh_vphi<float><<<blocks_of(n, 256), 256, 0, st>>>(n, 1.0 / dt, V, poro, vphi_d, (float*)vphi_r);
    else
        k_mesh_vphi<double><<<blocks_of(n, 256), 256, 0, st>>>(n, 1.0 / dt, V, poro, vphi_d, (double*)vphi_r);
    return cudaGetLastError();
}

cudaError_t launch_mesh_mixed(const MeshFields<float>& f, long long n, const PhysF& q, bool crk,
                              const AsmOut<float>& o, cudaStream_t st) {
    return launch_mesh_t<float>(f, n, q, crk, o, st);
}

cudaError_t launch_mesh_fp64(const MeshFields<double>& f, long long n, const PhysD& q, bool crk,
                             const AsmOut<double>& o, cudaStream_t st) {
    return launch_mesh_t<double>(f, n, q, crk, o, st);
}

}  // namespace tpfa
