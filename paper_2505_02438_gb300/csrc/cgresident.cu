// Conjugate gradients with the matrix resident in shared memory (solve.cu has the
// general loop and the start of both).
//
// The general loop is three dependent launches per iteration, each of a few
// microseconds however small the matrix.  When every SM can hold its share of K in
// shared memory (up to about 30 MB of it), one cooperative launch runs the iterations
// instead: each block owns consecutive nodes, keeps their rows (d-1 of a node's d as float pairs), their
// u, r and 1/diag, and a copy of p at all nodes its rows name (the halo), and an
// iteration exchanges only what other blocks need:
//
//   q = K p on the own rows; p.q          -> the block's term to every block
//   alpha; u, r, z = r/diag; r.z, r.r     -> z to memory, the terms to every block
//   beta; p = z + beta p on own and halo nodes (the same operation in every block)
//
// An exchange is a release-add to one counter after the block's terms (and z) are
// stored, an acquire wait for all blocks' adds, and the same sum of all terms in every
// block: every block takes the same decisions, no block waits for one that does the
// sums, and the iterates are bitwise reproducible.  1.5 us for 152 blocks without the
// sums; words of value and iteration number that the readers poll, which need neither
// counter nor fence, took 2.0 us, and 3.2 us with words of its own for every reader.
// Every wait is bounded: a block that waits too long raises the error word and leaves,
// and the others' waits run out after it.
//
// What bounds it is latency: two exchanges, and some 40 FP64 operations in a row (an FP64
// instruction also occupies the SM's FP64 pipe for 16 cycles, so only one lane tests the
// residual and divides).  Per iteration, the general loop and this kernel: 60x20x4 Q1
// hexahedra 20.2 and 9.8 us, 36x14x14 22.5 and 11.2, 60x20 Q1 quadrilaterals 14.6 and 8.0,
// 160x60 18.3 and 9.8, 260x150 29.3 and 16; 4x2 19 and 10: where it fits it is the faster
// one.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "df64.cuh"
#include "internal.h"
#include "kernels_common.cuh"

namespace soptx {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kHaloStride = kThreads - 32;
constexpr int kMaxBlocks = 160, kSlotsPerLane = kMaxBlocks / 32;
constexpr int kWaitLimit = 1 << 20;       // polls of about a microsecond each
constexpr int kItersPerLaunch = 4096;
constexpr int kNodeWeight = 24;           // a node's cost beside its entries, in entries (6 .. 24 measured alike)
constexpr int32_t kFixed = INT32_MIN;     // flag of a constrained dof in the halo's list of dofs

// Shared memory of a block with n nodes, e entries (row blocks) and h halo nodes (the own
// ones among them), as the kernel lays it out.  A node's values start at
// roundup(D D entry, 16) + 24 node doubles: node starts differ by 8 modulo 16, so the two
// nodes a half warp reads lie in different banks.
__host__ __device__ inline int vals_base(int dd, int entry, int node) { return ((dd * entry + 15) & ~15) + 24 * node; }
size_t smem_bytes(int D, int64_t n, int64_t e, int64_t h)
{
    return (size_t)vals_base(D * D, (int)e, (int)n) * 8 + (size_t)h * D * 16 + (size_t)n * D * 6 * 8 + (size_t)h * D * 4 +
           (size_t)(n + 1) * 4 + (size_t)e * D * 2 + 32;
}

struct Args {
    const int64_t *node_off;
    const double *vals;
    const uint8_t *fixed;
    const double *dinv;
    double *u, *r, *p, *rz;         // rz: (r.z) carried between launches
    const int32_t *n0, *hoff, *halo;
    const uint16_t *lidx;
    double *z;
    double2 *terms;                 // [2][blocks] the two sums of each exchange
    unsigned *arrived;              // blocks that have published, over all exchanges since the start
    int it0, it1, check_every, max_iter;
    double stop;                    // converged when sqrt(r.r) <= stop at a check
    CgResidentOut *out;
};

// Two sums over the warp's lanes by one butterfly: the total of the first in lanes 0 .. 15,
// that of the second in lanes 16 .. 31 (five FP64 additions in a row, not ten; each is
// about 100 cycles of latency here with its shuffle).
__device__ __forceinline__ double sum_pair(double s0, double s1)
{
    const bool up = threadIdx.x & 16;
    double s = (up ? s1 : s0) + __shfl_xor_sync(kFull, up ? s0 : s1, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    return s;
}

// Warp 0's exchange of two sums: the rows' terms t[0 .. n) and t[n .. 2 n) are added and
// published, and all blocks' pairs added in a fixed order once every block has arrived
// (*arrived counts them, want after this exchange).  What the block wrote to memory before
// its barrier is visible to a block whose wait has ended; with wake the other warps wait
// for that at the block's barrier, to read it while the terms are added.  The totals are
// in out[0] and out[1]; false when the wait ran out.
__device__ __forceinline__ bool exchange(const double *t, int n, double2 *terms, unsigned *arrived, unsigned want,
                                         bool wake, double *out)
{
    const int lane = threadIdx.x & 31, nblk = gridDim.x;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 1
    for (int r0 = lane; r0 < n; r0 += 128) {
        double v0[4], v1[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const bool on = r0 + 32 * j < n;
            v0[j] = on ? t[r0 + 32 * j] : 0.0;
            v1[j] = on ? t[n + r0 + 32 * j] : 0.0;
        }
        s0 += (v0[0] + v0[1]) + (v0[2] + v0[3]);
        s1 += (v1[0] + v1[1]) + (v1[2] + v1[3]);
    }
    double s = sum_pair(s0, s1);
    if ((lane & 15) == 0) __stcg((double *)(terms + blockIdx.x) + (lane >> 4), s);
    __syncwarp();
    if (lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
    for (int tries = 0;; tries++) {
        unsigned c;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(arrived) : "memory");
        if (__all_sync(kFull, (int)(c - want) >= 0)) break;
        if (tries > kWaitLimit) {
            if (wake) __syncthreads();
            return false;
        }
    }
    if (wake) __syncthreads();
    double2 v[kSlotsPerLane];
#pragma unroll
    for (int k = 0; k < kSlotsPerLane; k++) v[k] = __ldcg(terms + min(lane + 32 * k, nblk - 1));
#pragma unroll
    for (int k = 0; k < kSlotsPerLane; k++)
        if (lane + 32 * k >= nblk) v[k] = make_double2(0.0, 0.0);
    static_assert(kSlotsPerLane == 5, "the tree below");
    s = sum_pair(((v[0].x + v[1].x) + (v[2].x + v[3].x)) + v[4].x, ((v[0].y + v[1].y) + (v[2].y + v[3].y)) + v[4].y);
    if ((lane & 15) == 0) out[lane >> 4] = s;
    __syncwarp();
    return true;
}

__device__ __forceinline__ float2 pair_of(double v)
{
    const df s = df_split_z(v);
    return make_float2(s.h, s.l);
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1) k_cg_resident(const Args a)
{
    constexpr int DD = D * D;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double s_coef, s_sum[2], s_inv;
    __shared__ int s_fail, s_done;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, blk = blockIdx.x, nblk = gridDim.x;
    const int64_t n0 = a.n0[blk];
    const int ln = (int)(a.n0[blk + 1] - n0), rows = D * ln;
    const int64_t e0 = a.node_off[n0];
    const int ne = (int)(a.node_off[n0 + ln] - e0);
    const int h0 = a.hoff[blk], nh = a.hoff[blk + 1] - h0;
    // p at the halo's dofs: the value, and split
    double *xd = reinterpret_cast<double *>(smem);
    float2 *xp = reinterpret_cast<float2 *>(xd + (size_t)nh * D);
    float2 *val = xp + (size_t)nh * D;
    double *us = reinterpret_cast<double *>(val + vals_base(DD, ne, ln)), *rs = us + rows, *ds = rs + rows,
           *qs = ds + rows, *ts = qs + rows;   // ts [2][rows]: the rows' terms of the two sums
    int32_t *dof = reinterpret_cast<int32_t *>(ts + 2 * rows);   // the halo's dofs, flagged when constrained
    int32_t *noff = dof + nh * D;
    uint16_t *col = reinterpret_cast<uint16_t *>(noff + ln + 1);

    if (tid == 0) s_fail = s_done = 0, s_sum[0] = s_sum[1] = 0.0;
#pragma unroll 1
    for (int n = tid; n <= ln; n += kThreads) noff[n] = (int)(a.node_off[n0 + n] - e0);
#pragma unroll 1
    for (int i = tid; i < nh; i += kThreads) {
        const int32_t node = a.halo[h0 + i];
        for (int c = 0; c < D; c++) {
            const int32_t k = D * node + c;
            const double pv = a.p[k];
            xd[i * D + c] = pv;
            xp[i * D + c] = pair_of(pv);
            dof[i * D + c] = a.fixed[k] ? k | kFixed : k;
        }
    }
#pragma unroll 1
    for (int row = tid; row < rows; row += kThreads) {
        us[row] = a.u[D * n0 + row];
        rs[row] = a.r[D * n0 + row];
        ds[row] = a.dinv[D * n0 + row];
    }
#pragma unroll 1
    for (int row = tid; row < 2 * rows; row += kThreads) ts[row] = 0.0;
    double rz = *a.rz;
    __syncthreads();
#pragma unroll 1
    for (int n = warp; n < ln; n += kWarps) {
        const int eo = noff[n], cnt = noff[n + 1] - eo, len = D * cnt, base = vals_base(DD, eo, n);
        const double *src = a.vals + DD * (e0 + eo);
#pragma unroll 1
        for (int t = lane; t < DD * cnt; t += 32) {
            const double v = src[t];   // rows 0 .. d-2 split
            if (t < (D - 1) * len) val[base + t] = pair_of(v);
            else reinterpret_cast<double *>(val)[base + t] = v;
        }
#pragma unroll 1
        for (int t = lane; t < len; t += 32) col[D * eo + t] = (uint16_t)(D * a.lidx[e0 + eo + t / D] + t % D);
    }
    __syncthreads();

    const int g = lane >> 3, c = lane & 7;
    int it = a.it0;
    const int nx = nh * D;
    int until = a.check_every - it % a.check_every;   // iterations to the next check
    for (;;) {
        // q = K p: eight lanes a node, columns c, c + 8, ... of its d rows; rows 0 .. d-2 in
        // float pairs, row d-1 in FP64, as k_spmv (all rows in float pairs: 0.5 us less, but
        // solutions up to 50 times as far from the exact ones).  Four columns a pass, its
        // loads before its arithmetic.  (Elsewhere loops are kept rolled: unrolled by
        // default the iteration was 75 KB of code.)
#pragma unroll 1
        for (int nb = warp * 4; nb < ln; nb += kWarps * 4) {
            const int n = nb + g;
            float S[D], C[D];
            double Sd = 0.0;
#pragma unroll
            for (int i = 0; i < D - 1; i++) S[i] = C[i] = 0.f;
            if (n < ln) {
                const int eo = noff[n], len = D * (noff[n + 1] - eo);
                const uint16_t *cp = col + D * eo;
                const float2 *vf = val + vals_base(DD, eo, n);
                const double *vd = reinterpret_cast<const double *>(vf + (D - 1) * len);
#pragma unroll 1
                for (int t0 = c; t0 < len; t0 += 32) {
                    float2 w[4], v[4][D];
                    double wd[4], vl[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const bool on = t0 + 8 * k < len;
                        const int j = on ? cp[t0 + 8 * k] : 0;
                        w[k] = on ? xp[j] : make_float2(0.f, 0.f);
                        wd[k] = on ? xd[j] : 0.0;
                        vl[k] = on ? vd[t0 + 8 * k] : 0.0;
#pragma unroll
                        for (int i = 0; i < D - 1; i++) v[k][i] = on ? vf[i * len + t0 + 8 * k] : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        Sd = fma(vl[k], wd[k], Sd);
#pragma unroll
                        for (int i = 0; i < D - 1; i++) {
                            const df pr = df_mul_raw(df{v[k][i].x, v[k][i].y}, df{w[k].x, w[k].y});
                            float s2, err;
                            two_sum(S[i], pr.h, s2, err);
                            S[i] = s2;
                            C[i] = __fadd_rn(C[i], __fadd_rn(pr.l, err));
                        }
                    }
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                Sd += __shfl_xor_sync(kFull, Sd, o);
#pragma unroll
                for (int i = 0; i < D - 1; i++) {
                    const float Sp = __shfl_xor_sync(kFull, S[i], o), Cp = __shfl_xor_sync(kFull, C[i], o);
                    float s2, err;
                    two_sum(S[i], Sp, s2, err);   // exact, so the partners' operand order does not matter
                    S[i] = s2;
                    C[i] = __fadd_rn(__fadd_rn(C[i], Cp), err);
                }
            }
            if (n < ln && c < D) {
                float h = 0.f, l = 0.f;
#pragma unroll
                for (int i = 0; i < D - 1; i++)
                    if (i == c) two_sum(S[i], C[i], h, l);
                const int row = D * n + c;
                const double q = dof[row] < 0 ? 0.0 : c == D - 1 ? Sd : df_to_double(h, l);
                qs[row] = q;
                ts[row] = xd[row] * q;
            }
        }
        bool ok = true;
        double zv[4];
        int at[4];
#pragma unroll 1
        for (int ph = 0; ph < 2; ph++) {
            __syncthreads();   // the rows' terms (and z) are complete
            if (warp == 0) {
                ok = exchange(ts, rows, a.terms + ph * nblk, a.arrived, (unsigned)nblk * (2u * it + ph + 1u), ph == 1,
                              s_sum) && ok;
                if (lane == 0) {
                    s_coef = ph ? s_sum[0] * s_inv : ok && s_sum[0] != 0.0 ? rz / s_sum[0] : 0.0;
                    if (!ok) s_fail = 1;
                    // (one lane tests: FP64 in every warp would fill the FP64 pipe)
                    if (ph == 1 && (--until == 0 || it + 1 == a.max_iter)) {
                        until = a.check_every;
                        s_done = sqrt(s_sum[1]) <= a.stop;
                    }
                }
            } else if (ph == 0) {
                if (tid == 32) s_inv = rz != 0.0 ? 1.0 / rz : 0.0;   // for beta, off the chain
            } else {
                __syncthreads();   // every block's z is out: the first of it while warp 0 adds the terms
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    at[k] = nx > 0 ? dof[min(tid - 32 + k * kHaloStride, nx - 1)] : 0;
                    zv[k] = __ldcg(a.z + (at[k] & INT32_MAX));
                }
            }
            __syncthreads();
            if (ph == 0) {
                const double alpha = s_coef;
                double *zw = a.z + D * n0;
#pragma unroll 1
                for (int row = tid; row < rows; row += kThreads) {
                    double rn = 0.0, zv = 0.0;
                    if (dof[row] >= 0) {
                        rn = fma(-alpha, qs[row], rs[row]);
                        zv = rn * ds[row];
                        rs[row] = rn;
                        us[row] = fma(alpha, xd[row], us[row]);
                    }
                    __stcg(zw + row, zv);
                    ts[row] = rn * zv;
                    ts[rows + row] = rn * rn;
                }
            }
        }
        // p at the own and halo nodes, by all warps but the first
        if (warp > 0) {
            const double beta = s_coef;
#pragma unroll 1
            for (int i0 = tid - 32; i0 < nx; i0 += 4 * kHaloStride) {
                if (i0 >= 4 * kHaloStride) {
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        at[k] = dof[min(i0 + k * kHaloStride, nx - 1)];
                        zv[k] = __ldcg(a.z + (at[k] & INT32_MAX));
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const int i = i0 + k * kHaloStride;
                    if (i >= nx) continue;
                    const double pv = at[k] < 0 ? 0.0 : fma(beta, xd[i], zv[k]);
                    xd[i] = pv;
                    xp[i] = pair_of(pv);
                }
            }
        }
        __syncthreads();
        rz = s_sum[0];
        it++;
        if (s_fail) break;
        if (s_done || it >= a.it1) break;
    }
#pragma unroll 1
    for (int row = tid; row < rows; row += kThreads) {
        a.u[D * n0 + row] = us[row];
        a.r[D * n0 + row] = rs[row];
        a.p[D * n0 + row] = xd[row];
    }
    if (tid == 0) {
        if (s_fail) {
            a.out->error = 1;
        } else if (blk == 0) {
            a.out->it = it;
            a.out->converged = s_done;
            a.out->rr = s_sum[1];
            *a.rz = rz;
        }
    }
}

cudaError_t launch(const soptx_mesh_s &m, const Args &a, cudaStream_t st)
{
    const auto &d = m.d;
    Args args = a;
    void *params[] = {&args};
    const void *k = m.h.dim == 3 ? (const void *)k_cg_resident<3> : (const void *)k_cg_resident<2>;
    return cudaLaunchCooperativeKernel(k, dim3(d.rblocks), dim3(kThreads), params, (size_t)d.rsmem, st);
}

// The partition: consecutive nodes by weight (entries and kNodeWeight a node), per block the nodes its rows name, the own ones first, and every entry's place in that list.
struct Plan {
    std::vector<int32_t> n0, hoff, halo;
    std::vector<uint16_t> lidx;
    size_t smem = 0;
};

bool make_plan(const HostMesh &h, int blocks, size_t most, Plan &P)
{
    const int D = h.dim;
    if (h.ndof > INT32_MAX || h.node_off[(size_t)h.nn] > INT32_MAX) return false;
    const int64_t W = h.node_off[(size_t)h.nn] + kNodeWeight * h.nn;
    P.n0.assign((size_t)blocks + 1, (int32_t)h.nn);
    for (int64_t n = 0, b = 0; n < h.nn && b <= blocks; n++)
        while (b < blocks && h.node_off[(size_t)n] + kNodeWeight * n >= W * b / blocks) P.n0[(size_t)b++] = (int32_t)n;
    P.hoff.assign(1, 0);
    P.lidx.resize((size_t)h.node_off[(size_t)h.nn]);
    std::vector<int32_t> seen((size_t)h.nn, -1), place((size_t)h.nn, 0);
    for (int b = 0; b < blocks; b++) {
        const int32_t n0 = P.n0[(size_t)b], n1 = P.n0[(size_t)b + 1];
        const int64_t e0 = h.node_off[(size_t)n0], e1 = h.node_off[(size_t)n1];
        const size_t first = P.halo.size();
        if (smem_bytes(D, n1 - n0, e1 - e0, n1 - n0) > most) return false;
        auto add = [&](int32_t n) {
            if (seen[(size_t)n] == b) return;
            seen[(size_t)n] = b;
            place[(size_t)n] = (int32_t)(P.halo.size() - first);
            P.halo.push_back(n);
        };
        for (int32_t n = n0; n < n1; n++) add(n);
        for (int64_t e = e0; e < e1; e++) add(h.nbr[(size_t)e]);
        const int64_t nh = (int64_t)(P.halo.size() - first);
        const size_t need = smem_bytes(D, n1 - n0, e1 - e0, nh);
        if (need > most || nh * D > 65535) return false;
        P.smem = std::max(P.smem, need);
        for (int64_t e = e0; e < e1; e++) P.lidx[(size_t)e] = (uint16_t)place[(size_t)h.nbr[(size_t)e]];
        P.hoff.push_back((int32_t)P.halo.size());
    }
    return true;
}

size_t up16(size_t b) { return (b + 15) & ~(size_t)15; }

}  // namespace

// Decides once per mesh whether the solve is resident and lays out its tables; false
// (the general loop) when the matrix does not fit the SMs' shared memory, when the
// device cannot launch cooperatively, or when the memory cannot be had.
bool cg_resident_ready(soptx_mesh_s &m, cudaStream_t st)
{
    auto &d = m.d;
    const auto &h = m.h;
    if (d.rstate != 0) return d.rstate > 0;
    d.rstate = -1;
    int dev = 0, sms = 0, coop = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || !coop) {
        cudaGetLastError();
        return false;
    }
    const int blocks = (int)std::min<int64_t>(std::min(sms, kMaxBlocks), (h.nn + 7) / 8);
    const size_t most = (size_t)optin - 1024;   // less the kernel's static words
    if ((size_t)h.nnz * 8 > most * blocks) return false;
    Plan P;
    if (!make_plan(h, blocks, most, P)) return false;
    const void *k = h.dim == 3 ? (const void *)k_cg_resident<3> : (const void *)k_cg_resident<2>;
    int per_sm = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, P.smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return false;
    }
    // one allocation: the exchanged terms and their counter, the result, the tables
    const size_t sb = (size_t)2 * blocks * 16 + 128, ob = up16(sizeof(CgResidentOut));
    const size_t nb = up16(P.n0.size() * 4), hb = up16(P.hoff.size() * 4), lb = up16(P.halo.size() * 4),
                 ib = up16(P.lidx.size() * 2), bytes = sb + ob + nb + hb + lb + ib;
    unsigned char *p = nullptr;
    cudaError_t e = dev_alloc((void **)&p, bytes);
    unsigned char *t = p + sb + ob;
    if (e == cudaSuccess) e = cudaMemcpyAsync(t, P.n0.data(), P.n0.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(t + nb, P.hoff.data(), P.hoff.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(t + nb + hb, P.halo.data(), P.halo.size() * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(t + nb + hb + lb, P.lidx.data(), P.lidx.size() * 2, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (p) cudaFree(p);
        return false;
    }
    m.device_bytes += (int64_t)bytes;
    d.rbuf = p;
    d.rtables = t;
    d.rhoff = nb;
    d.rhalo = nb + hb;
    d.rlidx = nb + hb + lb;
    d.rblocks = blocks;
    d.rsmem = (int)P.smem;
    d.rstate = 1;
    return true;
}

// Iterations it < max_iter until the residual test holds; *launched stays false when the
// first launch was refused (nothing has changed then).
cudaError_t cg_resident_run(const soptx_mesh_s &m, const double *vals, const uint8_t *fixed, const double *dinv,
                            double *u, double *r, double *z, double *p, double *rz, int check_every, int max_iter,
                            double stop, cudaStream_t st, CgResidentOut *res, bool *launched)
{
    const auto &d = m.d;
    const size_t sb = (size_t)2 * d.rblocks * 16 + 128;
    Args a{};
    a.node_off = d.node_off;
    a.vals = vals;
    a.fixed = fixed;
    a.dinv = dinv;
    a.u = u;
    a.r = r;
    a.p = p;
    a.rz = rz;
    a.n0 = (const int32_t *)d.rtables;
    a.hoff = (const int32_t *)(d.rtables + d.rhoff);
    a.halo = (const int32_t *)(d.rtables + d.rhalo);
    a.lidx = (const uint16_t *)(d.rtables + d.rlidx);
    a.z = z;
    a.terms = (double2 *)d.rbuf;
    a.arrived = (unsigned *)(d.rbuf + sb - 128);
    a.out = (CgResidentOut *)(d.rbuf + sb);
    a.check_every = check_every;
    a.max_iter = max_iter;
    a.stop = stop;
    *launched = false;
    *res = CgResidentOut{};
    cudaError_t e = cudaMemsetAsync(d.rbuf, 0, sb + sizeof(CgResidentOut), st);
    while (e == cudaSuccess && res->it < max_iter && !res->converged && !res->error) {
        a.it0 = res->it;
        a.it1 = (int)std::min<int64_t>(max_iter, (int64_t)res->it + kItersPerLaunch);
        e = launch(m, a, st);
        if (e != cudaSuccess) break;
        *launched = true;
        e = cudaMemcpyAsync(res, a.out, sizeof *res, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    return e;
}

}  // namespace soptx
