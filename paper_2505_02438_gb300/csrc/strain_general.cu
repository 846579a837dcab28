// The sensitivities of general (bilinear and trilinear, non-affine) cells with FP64
// element matrices: s_e = u_e^T K_e^0 u_e = sum_q w_q |det J_q| (lam (tr g)^2 +
// mu sum_ij g_ij (g_ij + g_ji)), g = grad u at point q of the Gauss rule that defines
// K_e^0.  dc_e = -E'(rho_e) s_e, c = sum_e E(rho_e) s_e (fixed-order block partials).
// The points' energies are added in FP64, as the gather over the cached matrices adds
// its node partials.
//
//  k_strain_corners : order 1, a thread per cell, in float pairs.  The 2^d Gauss points
//                     are the corners of a box, so the reference displacement gradient at
//                     all of them is a Walsh transform each way.
//  k_strain_tensor  : orders 2 and 3, a lane per point, in FP64, by sum factorisation.
// Orders 2 and 3 were in float pairs first: with the tables rounded to pairs and some
// hundred operations in a row their error, 4.2e-15 .. 6.0e-15 of dc against 64 bits, was up
// to three times that of the gather (1.8e-15 .. 4.2e-15).
#include <algorithm>
#include <cstdint>

#include "df64.cuh"
#include "internal.h"
#include "kernels_common.cuh"

namespace soptx {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 128;

struct GeneralArgs {
    int64_t nc;
    const int32_t *__restrict__ cell_node;
    const double *__restrict__ u;
    const double *__restrict__ rho;
    SimpParams sp;
    // G = J^-1 row-major and w |det J| of every point, 8 bytes each.  k_strain_corners: G as
    // float pairs, w |det J| in FP64, a plane over the cells per (point, entry);
    // k_strain_tensor: all in FP64, per cell [entry][point]
    const float2 *__restrict__ geo;
    const double *__restrict__ tab;   // k_strain_tensor: 1D basis values [n][n], derivatives
                                      // [n][n], lattice index of each local node [n^d]
    int rounds;                       // k_strain_tensor: see there
    double lam, mu;   // at E = 1
    const double *__restrict__ gscale;
    double *__restrict__ out;
    double *__restrict__ partial;
    unsigned *__restrict__ counter;
    double *__restrict__ c;
};

// Product with the term of both tails: of squares it always has the same sign, and left
// out it was a bias of 1e-15 in every energy.
__device__ __forceinline__ df mul_full(df a, df b)
{
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.l, b.l, __fmaf_rn(a.h, b.h, -p));
    e = __fmaf_rn(a.h, b.l, e);
    return df{p, __fmaf_rn(a.l, b.h, e)};
}
struct Acc {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(df x)
    {
        float t, err;
        two_sum(s, x.h, t, err);
        s = t;
        c = __fadd_rn(c, __fadd_rn(x.l, err));
    }
    __device__ __forceinline__ df val() const
    {
        df r;
        two_sum(s, c, r.h, r.l);
        return r;
    }
};

// The cell's results from its energy at unit modulus.
__device__ __forceinline__ void put_cell(const GeneralArgs &A, int64_t e, double g, double sd, double &mine)
{
    const double r = A.rho[e];
    A.out[e] = g * simp_dE(A.sp, r) * sd;
    mine += simp_E(A.sp, r) * sd;
}

// Order 1.  With the differences (bit set) and sums (bit clear) of the corner values along
// the axes, w_b, and a = 1 / sqrt(3), the derivative along axis 1 at the signs (s2, s3) of a
// hexahedron's points is
//     (w_100 + s2 a w_110 + s3 a w_101 + s2 s3 a^2 w_111) / 4
// (and so on), about 150 float-pair sums in place of 576 multiply-adds; the square of that
// quarter is applied at the end.  Every sum is normalised: products of unnormalised pairs
// lose a term of 2^-46 (dc of hexahedra against 64 bits 5.8e-15, now 3.0e-15; the gather
// over the cached matrices 3.2e-15).  The derivative of component i along axis m at the
// signs s of the other axes lies at us[((m D + i) 2^(D-1) + s) kThreads + thread]: in
// registers, with the points unrolled, the kernel waited on instruction fetches (80 us in
// place of 68 on 192,000 hexahedra).  Bound by instruction issue (55% of the slots, 45% with
// the last wave) and the latency of the geometry's loads at 15 warps per SM, 36 KB of shared
// memory a block; the 123 MB of geometry alone take 18 us.
template <int D>
__global__ void __launch_bounds__(kThreads, 5) k_strain_corners(const GeneralArgs A)
{
    constexpr int NB = 1 << D, NS = NB / 2;
    __shared__ float2 us[D * D * NS * kThreads];
    const int tid = threadIdx.x;
    const double g = A.gscale ? *A.gscale : -1.0;
    const df lam = df_from_double(A.lam), mu = df_from_double(A.mu);
    const df a1 = df_from_double(0.57735026918962576451), a2 = df_from_double(1.0 / 3.0);
    double mine = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * kThreads + tid; e < A.nc; e += (int64_t)gridDim.x * kThreads) {
        int32_t nd[NB];
#pragma unroll
        for (int b = 0; b < NB; b++) nd[b] = __ldg(A.cell_node + e * NB + b);
#pragma unroll 1
        for (int i = 0; i < D; i++) {
            df w[NB];
#pragma unroll
            for (int b = 0; b < NB; b++) w[b] = df_split_z(__ldg(A.u + D * (int64_t)nd[b] + i));
#pragma unroll
            for (int m = 0; m < D; m++)
#pragma unroll
                for (int b = 0; b < NB; b++)
                    if (!(b & (1 << m))) {
                        const df lo = w[b], hi = w[b | (1 << m)];
                        w[b] = df_add(lo, hi);
                        w[b | (1 << m)] = df_add(hi, df_neg(lo));
                    }
#pragma unroll
            for (int b = 3; b < NB; b++)   // two bits set: a; three: a^2
                if (b != 4) w[b] = df_mul(w[b], b == 7 ? a2 : a1);
#pragma unroll
            for (int m = 0; m < D; m++) {
                const int p = m == 0 ? 1 : 0, r = m == 2 ? 1 : 2;   // the other axes
                float2 *o = us + (m * D + i) * NS * kThreads + tid;
                const df c0 = w[1 << m], cp = w[1 << m | 1 << p];
                df v[NS];
                const df pl = df_add(c0, df_neg(cp)), ph = df_add(c0, cp);
                if constexpr (D == 2) {
                    v[0] = pl;
                    v[1] = ph;
                } else {
                    const df cr = w[1 << m | 1 << r], cc = w[7];
                    const df ql = df_add(cr, df_neg(cc)), qh = df_add(cr, cc);
                    v[0] = df_add(pl, df_neg(ql));
                    v[1] = df_add(ph, df_neg(qh));
                    v[2] = df_add(pl, ql);
                    v[3] = df_add(ph, qh);
                }
#pragma unroll
                for (int k = 0; k < NS; k++) o[k * kThreads] = make_float2(v[k].h, v[k].l);
            }
        }
        double s = 0.0;
        const float2 *gp = A.geo + e;
#pragma unroll 1
        for (int q = 0; q < NB; q++, gp += (D * D + 1) * A.nc) {
            df G[D * D], gu[D][D];
#pragma unroll
            for (int t = 0; t < D * D; t++) {
                const float2 v = __ldcs(gp + t * A.nc);
                G[t] = df{v.x, v.y};
            }
            const double wd = __ldcs(reinterpret_cast<const double *>(gp + D * D * A.nc));
#pragma unroll
            for (int i = 0; i < D; i++) {
                df U[D];
#pragma unroll
                for (int m = 0; m < D; m++) {
                    const int k = (q & ((1 << m) - 1)) | ((q >> (m + 1)) << m);
                    const float2 v = us[((m * D + i) * NS + k) * kThreads + tid];
                    U[m] = df{v.x, v.y};
                }
#pragma unroll
                for (int j = 0; j < D; j++) {
                    Acc a;
#pragma unroll
                    for (int m = 0; m < D; m++) a.add(df_mul_raw(U[m], G[m * D + j]));
                    gu[i][j] = a.val();
                }
            }
            df tr = gu[0][0];
#pragma unroll
            for (int m = 1; m < D; m++) tr = df_add_lazy(tr, gu[m][m]);
            Acc sh, dens;
#pragma unroll
            for (int i = 0; i < D; i++)
#pragma unroll
                for (int j = 0; j < D; j++) sh.add(mul_full(gu[i][j], df_add_lazy(gu[i][j], gu[j][i])));
            const df t2 = mul_full(tr, tr);
            df tn;
            fast_two_sum(t2.h, t2.l, tn.h, tn.l);
            dens.add(df_mul_raw(lam, tn));
            dens.add(df_mul_raw(mu, sh.val()));
            s = fma(wd, (double)dens.s + (double)dens.c, s);
        }
        put_cell(A, e, g, s * (D == 3 ? 0.0625 : 0.25), mine);
    }
    if (A.c) grid_sum_last_block(mine, A.partial, A.counter, A.c);
}

__device__ __forceinline__ double density(const double (&gu)[2][2], double lam, double mu)
{
    const double tr = gu[0][0] + gu[1][1], sh = gu[0][1] + gu[1][0];
    return fma(lam * tr, tr, mu * fma(sh, sh, 2.0 * fma(gu[0][0], gu[0][0], gu[1][1] * gu[1][1])));
}
__device__ __forceinline__ double density(const double (&gu)[3][3], double lam, double mu)
{
    const double tr = gu[0][0] + gu[1][1] + gu[2][2];
    const double s0 = gu[0][1] + gu[1][0], s1 = gu[1][2] + gu[2][1], s2 = gu[2][0] + gu[0][2];
    const double d = fma(gu[0][0], gu[0][0], fma(gu[1][1], gu[1][1], gu[2][2] * gu[2][2]));
    return fma(lam * tr, tr, mu * fma(s0, s0, fma(s1, s1, fma(s2, s2, 2.0 * d))));
}

// Order K = 2, 3 by sum factorisation: the basis is a tensor product of 1D polynomials and
// the rule one of n = K + 1 points, so the reference gradient at the n^d points is d passes
// of 1D contractions through shared memory.  A lane per point (two for the 64 of a
// hexahedron), its rows of the 1D tables in registers; a warp holds 3 quadrilaterals of 9
// points, 2 of 16 or one hexahedron.  Bound by the FP64 pipe (81 .. 84% busy, 16 cycles of it
// an instruction).  A thread per quadrilateral took 111 us on 97,000 cells of order 2 (103
// here) and 56 us on any small mesh of order 3, a chain of 1300 operations (9 here).
template <int D, int K>
__global__ void __launch_bounds__(kThreads) k_strain_tensor(const GeneralArgs A)
{
    constexpr int n = K + 1, P = D == 2 ? n * n : n * n * n, NG = D * D + 1;
    constexpr int GL = P < 32 ? P : 32, NP = P / GL, NC = 32 / GL;   // lanes and points a lane of a cell, cells of a warp
    constexpr int NS = D == 2 ? 3 : 6;                               // staged arrays [D][P] of a cell
    extern __shared__ double ud[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gi = lane / GL, r = lane - gi * GL, base = gi * GL;
    double *const us = ud + (size_t)(warp * NC + min(gi, NC - 1)) * NS * D * P;
    double *const av = us + D * P, *const ad = av + D * P;
    const int q1 = r % n, q2 = (r / n) % n;
    double v1[n], d1[n], v2[n], d2[n], v3[D == 3 ? NP : 1][n], d3[D == 3 ? NP : 1][n];
    int lat[NP];
#pragma unroll
    for (int b = 0; b < n; b++) {
        v1[b] = A.tab[q1 * n + b];
        d1[b] = A.tab[n * n + q1 * n + b];
        v2[b] = A.tab[q2 * n + b];
        d2[b] = A.tab[n * n + q2 * n + b];
#pragma unroll
        for (int p = 0; p < (D == 3 ? NP : 0); p++) {
            const int q3 = (r + GL * p) / (n * n);
            v3[p][b] = A.tab[q3 * n + b];
            d3[p][b] = A.tab[n * n + q3 * n + b];
        }
    }
#pragma unroll
    for (int p = 0; p < NP; p++) lat[p] = (int)A.tab[2 * n * n + r + GL * p];
    const double g = A.gscale ? *A.gscale : -1.0;
    double mine = 0.0;
    // a warp takes A.rounds times its cells in a row and finishes them together, a lane per
    // cell: their moduli in FP64 cost about a fifth of a quadrilateral's energy
    const int64_t take = (int64_t)NC * A.rounds;
    for (int64_t c0 = ((int64_t)blockIdx.x * (kThreads / 32) + warp) * take; c0 < A.nc;
         c0 += (int64_t)gridDim.x * (kThreads / 32) * take) {
        double mys = 0.0;   // of cell c0 + lane
        for (int j = 0; j < A.rounds && c0 + j * NC < A.nc; j++) {
            const int64_t e = c0 + j * NC + gi;
            const bool on = gi < NC && e < A.nc;
            __syncwarp();
            if (on)
#pragma unroll
                for (int p = 0; p < NP; p++) {
                    const int64_t nd = __ldg(A.cell_node + e * P + r + GL * p);
#pragma unroll
                    for (int i = 0; i < D; i++) us[i * P + lat[p]] = __ldg(A.u + D * nd + i);
                }
            __syncwarp();
            // first index: av, ad at (q1, b2, b3) = sum_b1 l, l'_(b1)(q1) u(b1, b2, b3)
            if (on)
#pragma unroll
                for (int p = 0; p < NP; p++)
#pragma unroll
                    for (int i = 0; i < D; i++) {
                        const int o = i * P + r + GL * p;
                        double sv = 0.0, sd = 0.0;
#pragma unroll
                        for (int b = 0; b < n; b++) {
                            const double x = us[o - q1 + b];
                            sv = fma(v1[b], x, sv);
                            sd = fma(d1[b], x, sd);
                        }
                        av[o] = sv;
                        ad[o] = sd;
                    }
            __syncwarp();
            double s = 0.0;
            if constexpr (D == 2) {
                if (on) {
                    double U[2][2], gu[2][2], G[NG];
                    const double *gp = reinterpret_cast<const double *>(A.geo) + e * P * NG + r;
#pragma unroll
                    for (int t = 0; t < NG; t++) G[t] = __ldcs(gp + t * P);
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const int o = i * P + q1;
                        U[i][0] = U[i][1] = 0.0;
#pragma unroll
                        for (int b = 0; b < n; b++) {
                            U[i][0] = fma(v2[b], ad[o + n * b], U[i][0]);
                            U[i][1] = fma(d2[b], av[o + n * b], U[i][1]);
                        }
#pragma unroll
                        for (int j = 0; j < 2; j++) gu[i][j] = fma(U[i][0], G[j], U[i][1] * G[2 + j]);
                    }
                    s = G[4] * density(gu, A.lam, A.mu);
                }
                // the lanes' sum in the cell's first lane, in a fixed order
                if constexpr (GL == 9) {
                    const double x = __shfl_sync(kFull, s, min(base + 8, 31));
                    if (r == 0) s += x;
                }
#pragma unroll
                for (int o = GL == 16 ? 8 : 4; o > 0; o >>= 1)
                    s += __shfl_sync(kFull, s, min(base + ((r + o) & (GL == 16 ? 15 : 7)), 31));
            } else {
                double *const bvv = ad + D * P, *const bvd = bvv + D * P, *const bdv = bvd + D * P;
                // second index, at (q1, q2, b3)
#pragma unroll
                for (int p = 0; p < NP; p++)
                    if (on)
#pragma unroll
                        for (int i = 0; i < D; i++) {
                            const int o = i * P + r + GL * p;
                            double vv = 0.0, vd = 0.0, dv = 0.0;
#pragma unroll
                            for (int b = 0; b < n; b++) {
                                const double x = av[o + n * (b - q2)], y = ad[o + n * (b - q2)];
                                vv = fma(v2[b], x, vv);
                                vd = fma(d2[b], x, vd);
                                dv = fma(v2[b], y, dv);
                            }
                            bvv[o] = vv;
                            bvd[o] = vd;
                            bdv[o] = dv;
                        }
                __syncwarp();
                // third index at the points, and the energy there
                if (on)
#pragma unroll
                    for (int p = 0; p < NP; p++) {
                        const double *gp = reinterpret_cast<const double *>(A.geo) + e * P * NG + r + GL * p;
                        double G[NG], gu[D][D];
#pragma unroll
                        for (int t = 0; t < NG; t++) G[t] = __ldcs(gp + t * P);
#pragma unroll
                        for (int i = 0; i < D; i++) {
                            const int o = i * P + q1 + n * q2;
                            double U[D] = {};
#pragma unroll
                            for (int b = 0; b < n; b++) {
                                U[0] = fma(v3[p][b], bdv[o + n * n * b], U[0]);
                                U[1] = fma(v3[p][b], bvd[o + n * n * b], U[1]);
                                U[2] = fma(d3[p][b], bvv[o + n * n * b], U[2]);
                            }
#pragma unroll
                            for (int j = 0; j < D; j++) gu[i][j] = fma(U[0], G[j], fma(U[1], G[3 + j], U[2] * G[6 + j]));
                        }
                        s = fma(G[9], density(gu, A.lam, A.mu), s);
                    }
                s = warp_sum(s);
            }
            const double x = __shfl_sync(kFull, s, lane % NC * GL);
            if (lane / NC == j) mys = x;
        }
        if (lane < take && c0 + lane < A.nc) put_cell(A, c0 + lane, g, mys, mine);
    }
    if (A.c) grid_sum_last_block(mine, A.partial, A.counter, A.c);
}

// At mesh creation: G = J^-1 and w |det J| at the Gauss points, in FP64 (PAIRS: G as float pairs).
template <int D, bool PAIRS>
__global__ void k_point_geometry(int64_t nc, int nq, const double *__restrict__ xcell, const double *__restrict__ qw,
                                 const double *__restrict__ dgeo, int64_t cell, int64_t point, int64_t entry, float2 *__restrict__ geo)
{
    constexpr int NV = 1 << D;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nc * nq; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = x / nq;
        const int q = (int)(x - e * nq);
        const double *xv = xcell + e * NV * D;
        double J[D][D] = {};   // from the edge vectors: the rounding does not grow with the cell's distance from the origin
        for (int v = 1; v < NV; v++)
            for (int i = 0; i < D; i++)
                for (int m = 0; m < D; m++) J[i][m] += (xv[v * D + i] - xv[i]) * dgeo[(q * NV + v) * D + m];
        double G[D * D], det;
        if constexpr (D == 2) {
            det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
            G[0] = J[1][1] / det;
            G[1] = -J[0][1] / det;
            G[2] = -J[1][0] / det;
            G[3] = J[0][0] / det;
        } else {
            double C[3][3];   // cofactors
            for (int i = 0; i < 3; i++)
                for (int m = 0; m < 3; m++) {
                    const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, m1 = (m + 1) % 3, m2 = (m + 2) % 3;
                    C[i][m] = J[i1][m1] * J[i2][m2] - J[i1][m2] * J[i2][m1];
                }
            det = J[0][0] * C[0][0] + J[0][1] * C[0][1] + J[0][2] * C[0][2];
            for (int i = 0; i < 3; i++)
                for (int m = 0; m < 3; m++) G[m * 3 + i] = C[i][m] / det;
        }
        float2 *o = geo + e * cell + q * point;
        for (int t = 0; t < D * D; t++) {
            if (PAIRS) {
                const float h = __double2float_rn(G[t]);
                o[t * entry] = make_float2(h, __double2float_rn(G[t] - (double)h));
            } else {
                *reinterpret_cast<double *>(o + t * entry) = G[t];
            }
        }
        *reinterpret_cast<double *>(o + D * D * entry) = qw[q] * fabs(det);
    }
}

}  // namespace

cudaError_t launch_point_geometry(const soptx_mesh_s &m, cudaStream_t st)
{
    const auto &h = m.h;
    const auto &d = m.d;
    const int64_t ng = h.dim * h.dim + 1;
    // order 1: planes over the cells; else a cell's entries one after another, each over its points
    const int64_t cell = h.order == 1 ? 1 : d.snq * ng, point = h.order == 1 ? ng * h.nc : 1,
                  entry = h.order == 1 ? h.nc : d.snq;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((h.nc * d.snq + 255) / 256, 152 * 16));
    auto k = h.dim == 2 ? (h.order == 1 ? k_point_geometry<2, true> : k_point_geometry<2, false>)
                        : (h.order == 1 ? k_point_geometry<3, true> : k_point_geometry<3, false>);
    k<<<grid, 256, 0, st>>>(h.nc, d.snq, d.xcell, d.qw, d.qdgeo, cell, point, entry, d.sgeo);
    return cudaGetLastError();
}

// max_grid > 0 caps the blocks (the kernels loop over the cells): all of it for
// k_strain_corners, a quarter for quadrilaterals of order 2 and 3 (beside the gather, steps
// of 97,000 cells of order 2 499 us at one block per SM, 549 at two, 580 at four), no cap for
// hexahedra of order 2 and 3 (197 us at one, 187 from three on).
cudaError_t launch_general_sensitivity(const soptx_mesh_s &m, const double *rho, const double *u, double *out,
                                       double *c, const double *gscale, cudaStream_t st, int max_grid)
{
    const auto &h = m.h;
    GeneralArgs A;
    A.nc = h.nc;
    A.cell_node = m.d.cell_node;
    A.u = u;
    A.rho = rho;
    A.sp = simp_params(m.mat);
    A.geo = m.d.sgeo;
    A.tab = m.d.gtab;
    A.lam = m.mat.lam;
    A.mu = m.mat.mu;
    A.gscale = gscale;
    A.out = out;
    A.partial = m.d.scratch;
    A.counter = m.d.counter;
    A.c = c;
    void (*k)(GeneralArgs);
    int64_t per = kThreads;   // cells of a block
    A.rounds = 1;
    size_t smem = 0;
    if (h.order == 1) {
        k = h.dim == 3 ? k_strain_corners<3> : k_strain_corners<2>;
    } else {
        per = kThreads / 32 * (h.dim == 3 ? 1 : 32 / h.nb);
        k = h.dim == 2 ? (h.order == 2 ? k_strain_tensor<2, 2> : k_strain_tensor<2, 3>)
                       : (h.order == 2 ? k_strain_tensor<3, 2> : k_strain_tensor<3, 3>);
        smem = (size_t)per * (h.dim == 2 ? 3 : 6) * h.dim * h.nb * sizeof(double);
        // several rounds where four blocks per SM have them
        A.rounds = (int)std::max<int64_t>(1, std::min<int64_t>(8, h.nc / ((int64_t)per * 4 * 152)));
        per *= A.rounds;
        max_grid = h.dim == 2 ? (max_grid + 3) / 4 : 0;
    }
    int64_t grid = std::max<int64_t>(1, std::min<int64_t>((h.nc + per - 1) / per, m.d.scratch_len));
    if (max_grid > 0) grid = std::min<int64_t>(grid, max_grid);
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    k<<<(int)grid, kThreads, smem, st>>>(A);
    return cudaGetLastError();
}

}  // namespace soptx
