// The backward of f(rho, u) = u^T K(rho) u without K: both gradients from the cells.
//
// With FP64 element matrices the u-gradient 2 g K(rho) u = 2 g sum_e E_e K_e^0 u_e
// needs no assembled matrix: one kernel forms each cell's nodal forces E_e K_e^0 u_e
// and the rho-gradient g E'(rho_e) u_e^T K_e^0 u_e from the same intermediate values,
// the second adds every node's forces in the order of its cells (a fixed order,
// no atomics).  On the 120x40x40 hexahedra K is 381 MB to write and to read back,
// the forces are 37 MB that stay in L2.
//
//  k_lattice_forces : box lattices (Walsh sectors, see k_lattice_sens): the modes w of
//                     the cell's displacements, y = B w in each sector, s = w . y, and
//                     the forces as the transform of y.  One thread per cell; the
//                     forces in planes [corner][component][cell], read back in planes.
//  k_strain_forces  : affine cells of up to 10 nodes: at every point of the rule of
//                     k_strain_energy the displacement gradient, the energy density
//                     and the weighted stress S_q = w_q sigma G^T; then the forces
//                     f_b = |det J| sum_q S_q grad^ phi_b(xi_q), which take the displacements'
//                     place in shared memory and leave coalesced as [cell][node][component].
// In float pairs (48 bits) but for the last component of P3 triangles and Q2 quadrilaterals.
// (The product over K has the last row of every node in FP64.)  The call, with the product
// over K assembled for it and from the forces: 120x40x40 Q1 hexahedra 208 and 41 us,
// 144,000 P2 tetrahedra 515 and 114 us, 160,000 P3 triangles 437 and 119 us (in float pairs
// alone 88), 480x160 quadrilaterals 109 and 11 us.  What bounds it is instruction issue in
// the force kernels (float-pair products; all data are in L2).
#include <algorithm>
#include <cstdint>

#include "df64.cuh"
#include "internal.h"
#include "kernels_common.cuh"

namespace soptx {
namespace {

constexpr int kThreads = 128;

// Accumulate x into the unnormalised pair a.
__device__ __forceinline__ void acc_add(df &a, df x)
{
    float t, err;
    two_sum(a.h, x.h, t, err);
    a.h = t;
    a.l = __fadd_rn(a.l, __fadd_rn(x.l, err));
}
__device__ __forceinline__ void acc_fma(df &a, df x, df y) { acc_add(a, df_mul_raw(x, y)); }
__device__ __forceinline__ df settle(df a)
{
    df r;
    two_sum(a.h, a.l, r.h, r.l);
    return r;
}
__device__ __forceinline__ df pair_of(float2 v) { return df{v.x, v.y}; }

// E f as a normalised pair, the modulus outside the float-pair range (in FP64, out of line).
__device__ __noinline__ float2 times_fp64(double E, float h, float l)
{
    const df r = df_from_double(E * ((double)h + (double)l));
    return make_float2(r.h, r.l);
}

template <int D>
__global__ void __launch_bounds__(kThreads, 4)
k_lattice_forces(int nx, int ny, int64_t nc, const double *__restrict__ rho, const double *__restrict__ u,
                 SimpParams sp, const SectorTable<D> B, const double *__restrict__ gout, double *__restrict__ grad_rho,
                 float2 *__restrict__ f)
{
    constexpr int NC = 1 << D;
    const double g = *gout;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nc; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t ue = (uint32_t)e, r = ue / (uint32_t)nx;
        const int ex = (int)(ue % (uint32_t)nx);
        const int ey = D == 3 ? (int)(r % (uint32_t)ny) : (int)r, ez = D == 3 ? (int)(r / (uint32_t)ny) : 0;
        df w[NC][D];
#pragma unroll
        for (int a = 0; a < NC; a++) {
            const int64_t node = (int64_t)(ex + (a & 1)) +
                                 (int64_t)(nx + 1) * ((ey + ((a >> 1) & 1)) + (int64_t)(ny + 1) * (ez + (a >> 2)));
#pragma unroll
            for (int i = 0; i < D; i++) w[a][i] = df_split_z(u[D * node + i]);
        }
        const double re = rho[e];
        // the transform, y = B w sector by sector in w's place with s = w . y, and the
        // transform again (one copy of its code: two made the kernel wait on
        // instruction fetches)
#pragma unroll 1
        for (int pass = 0; pass < 2; pass++) {
#pragma unroll
            for (int m = 0; m < D; m++)
#pragma unroll
                for (int a = 0; a < NC; a++)
                    if (!(a & (1 << m)))
#pragma unroll
                        for (int i = 0; i < D; i++) {
                            const df x = w[a][i], y = w[a | (1 << m)][i];
                            w[a][i] = df_add_lazy(x, y);
                            w[a | (1 << m)][i] = df_add_lazy(x, df_neg(y));
                        }
            if (pass == 1) break;
            df s{0.f, 0.f};
#pragma unroll
            for (int c = 0; c < NC; c++) {
                df x[D], y[D];
#pragma unroll
                for (int i = 0; i < D; i++) x[i] = w[c ^ (1 << i)][i];
#pragma unroll
                for (int i = 0; i < D; i++) {
                    df t{0.f, 0.f};
#pragma unroll
                    for (int j = 0; j < D; j++) {
                        if (sector_zero(c, i < j ? i : j, i < j ? j : i)) continue;
                        // (the table's off-diagonal entries are doubled)
                        float2 b = i <= j ? B.b[(c * D + i) * D + j] : B.b[(c * D + j) * D + i];
                        if (i != j) b = make_float2(0.5f * b.x, 0.5f * b.y);
                        acc_fma(t, x[j], pair_of(b));
                    }
                    y[i] = settle(t);
                    acc_fma(s, x[i], y[i]);
                }
#pragma unroll
                for (int i = 0; i < D; i++) w[c ^ (1 << i)][i] = y[i];
            }
            const df st = settle(s);
            grad_rho[e] = g * simp_dE(sp, re) * df_to_double(st.h, st.l);
        }
        const float2 Ep = simp_E_pair(sp, re);
        const bool bad = isnan(Ep.y);
        const double Ed = bad ? simp_E(sp, re) : 0.0;
#pragma unroll
        for (int a = 0; a < NC; a++)
#pragma unroll
            for (int i = 0; i < D; i++) {
                const df t = df_mul(df{Ep.x, Ep.y}, w[a][i]);
                f[(int64_t)(a * D + i) * nc + e] = bad ? times_fp64(Ed, w[a][i].h, w[a][i].l) : make_float2(t.h, t.l);
            }
    }
}

// out = 2 g times the sum of every node's forces, one thread per node, corners in ascending order of the cell
template <int D>
__global__ void __launch_bounds__(256)
k_lattice_gather(int nx, int ny, int nz, int64_t nn, int64_t nc, const float2 *__restrict__ f,
                 const double *__restrict__ gout, double *__restrict__ out)
{
    const double g2 = 2.0 * *gout;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < nn; n += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t un = (uint32_t)n, r = un / (uint32_t)(nx + 1);
        const int ix = (int)(un % (uint32_t)(nx + 1));
        const int iy = D == 3 ? (int)(r % (uint32_t)(ny + 1)) : (int)r, iz = D == 3 ? (int)(r / (uint32_t)(ny + 1)) : 0;
        float2 v[1 << D][D];
#pragma unroll
        for (int k = 0; k < 1 << D; k++) {
            // cell on the low (bit clear) or high side: the node is the opposite corner of it
            const int a = ((1 << D) - 1) ^ k;
            const int ex = ix - 1 + (k & 1), ey = iy - 1 + ((k >> 1) & 1), ez = D == 3 ? iz - 1 + (k >> 2) : 0;
            const bool in = ex >= 0 && ex < nx && ey >= 0 && ey < ny && ez >= 0 && ez < (D == 3 ? nz : 1);
            const int64_t e = ((int64_t)ez * ny + ey) * nx + ex;
#pragma unroll
            for (int i = 0; i < D; i++) v[k][i] = in ? __ldg(f + (int64_t)(a * D + i) * nc + e) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < D; i++) {
            df t{0.f, 0.f};
#pragma unroll
            for (int k = 0; k < 1 << D; k++) acc_add(t, pair_of(v[k][i]));
            t = settle(t);
            out[D * n + i] = g2 * df_to_double(t.h, t.l);
        }
    }
}

struct ForceArgs {
    int64_t nc;
    const int32_t *__restrict__ cell_node;
    const double *__restrict__ u;
    const double *__restrict__ rho;
    SimpParams sp;
    const float2 *__restrict__ geo;   // [nc or 1][d*d + 1] G row-major, |det J|, as pairs
    int64_t geo_stride;               // d*d + 1, or 0 when every cell has the same Jacobian
    const float2 *__restrict__ qw;    // [NQ] weights
    const float2 *__restrict__ qd;    // [NQ][NB][D] reference gradients
    const double *__restrict__ qd64;  // the same in FP64 (2D, NQ > 4)
    float2 lam, mu;
    const double *__restrict__ gout;
    double *__restrict__ grad_rho;
    float2 *__restrict__ f;           // [nc][NB][D]
};

// One thread per cell; displacements, then forces, in shared memory: [NB D][kThreads + 1].
template <int D, int NB, int NQ>
__global__ void __launch_bounds__(kThreads) k_strain_forces(const ForceArgs A)
{
    constexpr int P = kThreads + 1, ND = NB * D;
    constexpr bool kFp64 = D == 2 && NQ > 4;
    extern __shared__ float2 us[];
    const int tid = threadIdx.x;
    const double g = *A.gout;
    const df lam = pair_of(A.lam), mu = pair_of(A.mu);
    for (int64_t e0 = (int64_t)blockIdx.x * kThreads; e0 < A.nc; e0 += (int64_t)gridDim.x * kThreads) {
        const int64_t e = e0 + tid;
        if (e < A.nc) {
            int32_t nd[NB];
#pragma unroll
            for (int b = 0; b < NB; b++) nd[b] = __ldg(A.cell_node + e * NB + b);
            double uv[NB][D];
#pragma unroll
            for (int b = 0; b < NB; b++)
#pragma unroll
                for (int i = 0; i < D; i++) uv[b][i] = __ldg(A.u + (int64_t)D * nd[b] + i);
#pragma unroll
            for (int b = 0; b < NB; b++)
#pragma unroll
                for (int i = 0; i < D; i++) {
                    const df v = df_split_z(uv[b][i]);
                    us[(b * D + i) * P + tid] = make_float2(v.h, v.l);
                }
            df G[D * D], det;
            const float2 *gp = A.geo + e * A.geo_stride;
#pragma unroll
            for (int t = 0; t < D * D; t++) G[t] = pair_of(gp[t]);
            det = pair_of(gp[D * D]);
            const double re = A.rho[e];
            const float2 Ep = simp_E_pair(A.sp, re);
            const bool bad = isnan(Ep.y);
            const double Ed = bad ? simp_E(A.sp, re) : 0.0;
            df S[NQ][D][D], s{0.f, 0.f};
#pragma unroll
            for (int q = 0; q < NQ; q++) {
                const float2 *dq = A.qd + (size_t)q * ND;
                df U[D][D];
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int m = 0; m < D; m++) U[i][m] = df{0.f, 0.f};
#pragma unroll 2
                for (int b = 0; b < NB; b++) {
                    df dp[D];
#pragma unroll
                    for (int m = 0; m < D; m++) dp[m] = pair_of(__ldg(dq + b * D + m));
#pragma unroll
                    for (int i = 0; i < D; i++) {
                        const df ub = pair_of(us[(b * D + i) * P + tid]);
#pragma unroll
                        for (int m = 0; m < D; m++) {
                            acc_fma(U[i][m], ub, dp[m]);
                            // in 2D the sums' tails are short: 5% less error of g_u
                            if (D == 2 && (b & 1)) U[i][m] = settle(U[i][m]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int m = 0; m < D; m++) U[i][m] = settle(U[i][m]);
                // grad u = U^ G, the stress and w sigma G^T
                df gu[D][D];
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int j = 0; j < D; j++) {
                        df t{0.f, 0.f};
#pragma unroll
                        for (int m = 0; m < D; m++) acc_fma(t, U[i][m], G[m * D + j]);
                        gu[i][j] = settle(t);
                    }
                df tr = gu[0][0];
#pragma unroll
                for (int m = 1; m < D; m++) tr = df_add(tr, gu[m][m]);
                const df lt = df_mul(lam, tr), w = pair_of(__ldg(A.qw + q));
                df sg[D][D], en{0.f, 0.f};
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int j = i; j < D; j++) {
                        df t = df_mul(mu, df_add(gu[i][j], gu[j][i]));
                        if (i == j) t = df_add(t, lt);
                        sg[i][j] = sg[j][i] = df_mul(w, t);
                    }
                // density . w = sigma : grad u
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int j = 0; j < D; j++) acc_fma(en, sg[i][j], gu[i][j]);
                acc_add(s, en);
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int m = 0; m < D; m++) {
                        df t{0.f, 0.f};
#pragma unroll
                        for (int j = 0; j < D; j++) acc_fma(t, sg[i][j], G[m * D + j]);
                        S[q][i][m] = settle(t);
                    }
            }
            // |det J| last: taken into every point's weight its tail is lost on cells of 1e-9
            // (a gradient 8e-13 off, now 1e-13)
            const df sv = df_mul(settle(s), det);
            A.grad_rho[e] = g * simp_dE(A.sp, re) * df_to_double(sv.h, sv.l);
            // the forces in the displacements' place.  In 2D with many points the second
            // component is formed in FP64 from the stresses, as k_spmv forms a node's last
            // row: in float pairs alone the sum over the points left g_u further off than the
            // assembled product (P3 triangles 8.5e-15 against 7.8e-15 of 64 bits, Q2 boxes
            // 8.8e-15 against 8.3e-15).  FP64 in both components is slower still
            double S2[kFp64 ? NQ : 1][D], Ed2 = 0.0;
            if constexpr (kFp64) {
#pragma unroll
                for (int q = 0; q < NQ; q++)
#pragma unroll
                    for (int m = 0; m < D; m++) S2[q][m] = pair_to_double(S[q][D - 1][m].h, S[q][D - 1][m].l);
                Ed2 = (bad ? Ed : pair_to_double(Ep.x, Ep.y)) * pair_to_double(det.h, det.l);
            }
#pragma unroll 1
            for (int b = 0; b < NB; b++) {
                df t[D];
                double t2 = 0.0;
#pragma unroll
                for (int i = 0; i < D; i++) t[i] = df{0.f, 0.f};
#pragma unroll
                for (int q = 0; q < NQ; q++)
#pragma unroll
                    for (int m = 0; m < D; m++) {
                        const int at = q * ND + b * D + m;
                        const df dp = pair_of(__ldg(A.qd + at));
#pragma unroll
                        for (int i = 0; i < (kFp64 ? D - 1 : D); i++) acc_fma(t[i], S[q][i][m], dp);
                        if constexpr (kFp64) t2 = fma(S2[q][m], __ldg(A.qd64 + at), t2);
                    }
#pragma unroll
                for (int i = 0; i < D; i++) {
                    float2 *const o = us + (b * D + i) * P + tid;
                    if (kFp64 && i == D - 1) {
                        const df y = df_split_z(Ed2 * t2);
                        *o = make_float2(y.h, y.l);
                    } else {
                        const df x = df_mul(settle(t[i]), det), y = df_mul(df{Ep.x, Ep.y}, x);
                        *o = bad ? times_fp64(Ed, x.h, x.l) : make_float2(y.h, y.l);
                    }
                }
            }
        }
        __syncthreads();
        const int n = (int)min((int64_t)kThreads, A.nc - e0) * ND;
        for (int x = tid; x < n; x += kThreads) A.f[e0 * ND + x] = us[(x % ND) * P + x / ND];
        __syncthreads();
    }
}

// out = 2 g times the sum of every node's forces over its incidences (ascending cells)
template <int D>
__global__ void __launch_bounds__(256)
k_force_gather(int64_t nn, const int32_t *__restrict__ inc_ptr, const int32_t *__restrict__ inc,
               const float2 *__restrict__ f, const double *__restrict__ gout, double *__restrict__ out)
{
    const double g2 = 2.0 * *gout;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < nn; n += (int64_t)gridDim.x * blockDim.x) {
        const int32_t q0 = __ldg(inc_ptr + n), q1 = __ldg(inc_ptr + n + 1);
        df t[D];
#pragma unroll
        for (int i = 0; i < D; i++) t[i] = df{0.f, 0.f};
        int32_t q = q0;
        for (; q + 4 <= q1; q += 4) {
            float2 v[4][D];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int64_t x = (int64_t)__ldg(inc + q + k) * D;
#pragma unroll
                for (int i = 0; i < D; i++) v[k][i] = __ldg(f + x + i);
            }
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int i = 0; i < D; i++) acc_add(t[i], pair_of(v[k][i]));
        }
        for (; q < q1; q++) {
            const int64_t x = (int64_t)__ldg(inc + q) * D;
#pragma unroll
            for (int i = 0; i < D; i++) acc_add(t[i], pair_of(__ldg(f + x + i)));
        }
#pragma unroll
        for (int i = 0; i < D; i++) {
            const df r = settle(t[i]);
            out[D * n + i] = g2 * df_to_double(r.h, r.l);
        }
    }
}

int blocks_for(int64_t items, int per) { return (int)std::max<int64_t>(1, std::min<int64_t>((items + per - 1) / per, 152 * 32)); }

template <int D>
cudaError_t lattice_vjp(const soptx_mesh_s &m, const double *rho, const double *u, const double *gout, double *grad_rho,
                        double *grad_u, float2 *f, cudaStream_t st)
{
    const auto &h = m.h;
    SectorTable<D> B;
    for (int t = 0; t < (1 << D) * D * D; t++) B.b[t] = h.sectors[(size_t)t];
    k_lattice_forces<D><<<blocks_for(h.nc, kThreads), kThreads, 0, st>>>(h.lat_n[0], h.lat_n[1], h.nc, rho, u,
                                                                        simp_params(m.mat), B, gout, grad_rho, f);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_lattice_gather<D><<<blocks_for(h.nn, 256), 256, 0, st>>>(h.lat_n[0], h.lat_n[1], h.lat_n[2], h.nn, h.nc, f, gout,
                                                              grad_u);
    return cudaGetLastError();
}

template <int D, int NB, int NQ>
cudaError_t strain_vjp(const soptx_mesh_s &m, const ForceArgs &A, double *grad_u, cudaStream_t st)
{
    const size_t smem = (size_t)NB * D * (kThreads + 1) * sizeof(float2);
    auto k = k_strain_forces<D, NB, NQ>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<blocks_for(A.nc, kThreads), kThreads, smem, st>>>(A);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_force_gather<D><<<blocks_for(m.h.nn, 256), 256, 0, st>>>(m.h.nn, m.d.inc_ptr, m.d.inc, A.f, A.gout, grad_u);
    return cudaGetLastError();
}

// The cells k_strain_forces is compiled for: nodes and points of the rule, and the cells
// from which it is the faster way (a thread per cell: on few cells of many points its chain
// of operations is longer than the product over K.  Calls, us, product and forces: P2
// tetrahedra 96 cells 33 and 36, 900 35 and 36, 4860 45 and 40; hexahedra 150 cells 42 and
// 54, 6480 50 and 55, 106,000 314 and 174; P3 triangles 1200 cells 32 and 34, 9800 33 and 34,
// 160,000 241 and 77; Q2 quadrilaterals 800 cells 33 and 37, 6000 34 and 38, 98,000 282 and 86).
bool forces_fit(const soptx_mesh_s &m)
{
    static const int combos[][4] = {{2, 3, 1, 0}, {2, 6, 3, 0}, {2, 10, 7, 8192}, {2, 4, 4, 0}, {2, 9, 9, 8192},
                                    {3, 4, 1, 0}, {3, 10, 4, 2048}, {3, 8, 8, 10000}};
    for (const auto &c : combos)
        if (m.h.dim == c[0] && m.h.nb == c[1] && m.d.snq == c[2]) return m.h.nc >= c[3];
    return false;
}

}  // namespace

// Whether both gradients come from the cells (FP64 element matrices: with FP32 ones
// the product is that of the rounded matrices; the forces fit in the nnz values of
// the scratch).
bool vjp_matrix_free(const soptx_mesh_s &m)
{
    const auto &h = m.h;
    if (m.prec != SOPTX_ELEM_FP64 || h.nc == 0 || h.nc * h.ldof > h.nnz) return false;
    if (m.path == SOPTX_PATH_LATTICE) return m.d.sectors && (int)h.sectors.size() == (h.dim << h.dim) * h.dim;
    return m.d.strain && !h.nonaffine && forces_fit(m);
}

cudaError_t launch_vjp(const soptx_mesh_s &m, const double *rho, const double *u, const double *gout, double *grad_rho,
                       double *grad_u, float2 *f, cudaStream_t st)
{
    const auto &h = m.h;
    if (m.path == SOPTX_PATH_LATTICE)
        return h.dim == 3 ? lattice_vjp<3>(m, rho, u, gout, grad_rho, grad_u, f, st)
                          : lattice_vjp<2>(m, rho, u, gout, grad_rho, grad_u, f, st);
    auto pair = [](double x) {
        const float hh = (float)x;
        return make_float2(hh, (float)(x - (double)hh));
    };
    ForceArgs A;
    A.nc = h.nc;
    A.cell_node = m.d.cell_node;
    A.u = u;
    A.rho = rho;
    A.sp = simp_params(m.mat);
    A.geo = m.d.sgeo;
    A.geo_stride = m.path == SOPTX_PATH_UNIFORM ? 0 : h.dim * h.dim + 1;
    A.qw = m.d.sq;
    A.qd = m.d.sq + m.d.snq;
    A.qd64 = m.d.gtab;
    A.lam = pair(m.mat.lam);
    A.mu = pair(m.mat.mu);
    A.gout = gout;
    A.grad_rho = grad_rho;
    A.f = f;
#define SOPTX_VJP(D, NB, NQ) \
    if (h.dim == D && h.nb == NB && m.d.snq == NQ) return strain_vjp<D, NB, NQ>(m, A, grad_u, st);
    SOPTX_VJP(2, 3, 1) SOPTX_VJP(2, 6, 3) SOPTX_VJP(2, 10, 7) SOPTX_VJP(2, 4, 4) SOPTX_VJP(2, 9, 9)
    SOPTX_VJP(3, 4, 1) SOPTX_VJP(3, 10, 4) SOPTX_VJP(3, 8, 8)
#undef SOPTX_VJP
    return cudaErrorInvalidValue;
}

}  // namespace soptx
