// K(rho) = sum_e E(rho_e) K_e^0 on 3D meshes off the box lattice, by chunks of
// complete rows.
//
// A chunk is a set of nodes that are close together (consecutive along a
// Hilbert curve through the cells), with all of their rows.  One CTA assembles
// a chunk: one lane per node pair {a, b} that shares a cell walks the cells
// that hold both, sums the 3 x 3 block in float pairs in registers (no atomics,
// a fixed order), and puts it into the chunk's rows, staged in shared memory
// -- with FP64 element matrices transposed as well when b is in the chunk too,
// since K is symmetric, so those blocks are formed and converted once for two
// places (FP32 ones are symmetric only to their rounding).  The finished rows
// of a node are contiguous in the CSR values and leave by one bulk copy each
// (cp.async.bulk), so every sector is written whole, whatever the order of the
// chunks.  A pair of more than `cap` cells is shared by 2, 4, ... lanes whose sums a
// fixed shuffle tree adds, so no lane of a tile walks much further than the others.
//
// Nothing in the pair loop waits on global memory: one warp of the CTA moves the
// data.  A chunk's record (its nodes' places, cell list, pairs and their cells)
// is copied to shared memory two chunks ahead (cp.async.bulk) and its cells'
// data one chunk ahead (cp.async).  The other warps take tiles of 32 pairs from
// the chunk's counter and go on to the next chunk when there are none, so they
// never wait for one another (with a barrier of the whole CTA around each chunk,
// the kernel ran at 51% issue, now 65%: P2 tets 60x20x20 in FP32 243 -> 205 us).
// A persistent grid takes the chunks from a counter; a CTA that starts late
// beside another kernel simply takes fewer.
//
// Assembly call, us, against the kernels this one replaced (row and node gathers of
// the cache, a node-owner contraction, the pair kernel without symmetry): P2 tets
// 60x20x20 FP64 350 -> 296, FP32 283 -> 216; jittered hexahedra Q1 120x40x40 337 -> 249,
// Q2 40x14x14 316 -> 166, Q3 26x9x9 699 -> 265; boxes Q2 195 -> 118, Q3 282 -> 197.
// What bounds it (a capture each): kContract the FP32 instructions at 16 warps per SM (65%
// issue); kUniform no pipe alone (issue 52%, L1 data pipe 53%, the conversions' FP64 pipe
// 50%) but the latency of K^0's blocks and the dependences at those warps; kStream the latency
// of its one read of the blocks, at 4.9 TB/s.
//
// A block K_e^0[(a,.),(b,.)] comes from one of the following (SRC):
//   kContract : FP32 element matrices of affine cells, never stored: the
//               reference integrals M^{kl}_{ab} in FP32 contracted with the cell's
//               G and |det J| in shared memory (Sec. 3.2.2), then E K as an exact
//               FP32 product pair.
//   kUniform  : one element matrix for every cell (boxes of order 2 and 3): the
//               float-pair blocks of K^0, read through L1.
//   kStream   : cached FP64 element matrices: at mesh creation every record's
//               block is laid down in the order in which the lanes meet it, so a
//               warp reads whole 512-byte pieces, one record row ahead (in
//               registers; through two buffers in shared memory filled by the
//               copy engine it was slower, 344 against 296 us on the P2 tets: one CTA per
//               SM, and less in flight).  Bound by that read and by writing K.
//
// Record of a chunk (32-bit words, a whole number of 16-byte units):
//   0 cells | nodes << 16;  1 tiles | record rows << 16;  2 first word of the tiles |
//   of the pairs << 16;  3 first word of the records;  4 record rows before this chunk
//   nodes  : [nodes][2] row block offset of the node in K; staged place | degree << 16
//   cells  : [cells] cell ids
//   tiles  : [tiles] first record row | rows << 16
//   pairs  : [tiles * 32][2] staged place of the block | row length << 16 | cells(0-4) << 27;
//            of the transpose (0xffff: none) | row length << 16 | (cells(5-6) | lg lanes << 2) << 27
//   records: [rows][32] 16 bits: cell of the chunk (cell_bits) | (a nb + b) << cell_bits
#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "df64.cuh"
#include "internal.h"
#include "kernels_common.cuh"

namespace soptx {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int D = 3;
constexpr int kContract = kBlockContract, kUniform = kBlockUniform, kStream = kBlockStream;

// Bytes of a cell in shared memory, its modulus included.
template <int SRC> constexpr int kCellBytes = SRC == kContract ? 48 : 8;
// Bytes of a record row of streamed blocks: 32 blocks of 9 float pairs.
constexpr int kRowBytes = 32 * 9 * 8;

struct BlockArgs {
    int64_t nchunks;
    unsigned *__restrict__ ticket;        // [0] chunks handed out, [1] CTAs done (both zero between calls)
    volatile unsigned *expired;           // host memory: set when a wait ran out (the next call reports it)
    int tries;                            // limit of the data-moving warp's waits
    const uint4 *__restrict__ blob;
    const uint32_t *__restrict__ coff;    // [nchunks + 1] chunk starts in 16-byte units
    int max_blob, max_cells, max_stage, cell_bits;   // 16-byte units, cells, values; of a record
    const float4 *__restrict__ cdata;     // kContract: [nc][3] G row-major, |det J|
    const float *__restrict__ M;          // kContract: reference integrals [nb nb][12]
    int nm;                               // floats in M
    const float4 *__restrict__ kblk;      // kUniform: [nb nb][5] float pairs, two per float4; kStream: the blocks
    const float2 *__restrict__ Edf;
    const double *__restrict__ rho;
    const float2 *__restrict__ K;         // kStream: the cached element matrices (FP64 redo)
    int nb;
    SimpParams sp;
    float lam, mu;
    double *__restrict__ vals;
};

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *sdst, const void *gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void *sdst, const void *gsrc)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// shared -> global by the copy engine: both addresses 16-byte aligned, size a multiple of 16
__device__ __forceinline__ void bulk_store(double *gdst, const double *ssrc, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_addr(ssrc)),
                 "r"(bytes)
                 : "memory");
}

// Shared-memory barriers (mbarrier).  Every wait is bounded: after kBlockWaitTries tries (the
// data-moving warp: BlockArgs::tries, the same but in tests) of up to 20 us each the whole
// warp gives up, raises the error word and leaves.  The data-moving warp then ends the
// chunks of the others and still waits, with the full limit, for the copies that it has in
// flight; when another warp gives up, its waits run out after it.
__device__ __forceinline__ void mbar_init(uint64_t *b, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint64_t *b, unsigned parity, int tries)
{
    for (int i = 0; i < tries; i++) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\n\tselp.u32 %0, 1, 0, "
            "p;\n\t}"
            : "=r"(done)
            : "r"(smem_addr(b)), "r"(parity)
            : "memory");
        if (__all_sync(kFull, (int)done)) return true;   // (the lanes decide alike)
    }
    return false;
}
// global -> shared by the copy engine, counted on b (one arrival and the bytes)
__device__ __forceinline__ void bulk_load(void *sdst, const void *gsrc, uint32_t bytes, uint64_t *b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_addr(b)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(sdst)),
                 "l"(gsrc), "r"(bytes), "r"(smem_addr(b))
                 : "memory");
}

// Accumulate x into the unnormalised pair (s, c).
__device__ __forceinline__ void acc_add(float &s, float &c, df x)
{
    float t, err;
    two_sum(s, x.h, t, err);
    s = t;
    c = __fadd_rn(c, __fadd_rn(x.l, err));
}
// E k as an unnormalised pair, k FP32 (exact head, one rounding in the tail).
__device__ __forceinline__ df times(df E, float k)
{
    const float p = __fmul_rn(E.h, k);
    return df{p, __fmaf_rn(E.l, k, __fmaf_rn(E.h, k, -p))};
}

// max that keeps a NaN
__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// The FP32 block of a pair and cell: P = |det J| G^T M G, K = lam P + mu P^T + mu tr P I.
// cell: G row-major; g2: its last entry, |det J| and the cell's modulus.
__device__ __forceinline__ void contract(const float4 *cell, const float4 g2, const float *Mp, float lam, float mu,
                                         float (&K)[9])
{
    const float4 g0 = cell[0], g1 = cell[1];
    const float4 m0 = *reinterpret_cast<const float4 *>(Mp), m1 = *reinterpret_cast<const float4 *>(Mp + 4);
    const float G[9] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w, g2.x};
    const float M[9] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w, Mp[8]};
    float T[3][3], P[3][3];
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int j = 0; j < 3; j++)
            T[k][j] = fmaf(M[3 * k + 2], G[6 + j], fmaf(M[3 * k + 1], G[3 + j], M[3 * k] * G[j]));
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) P[i][j] = fmaf(G[6 + i], T[2][j], fmaf(G[3 + i], T[1][j], G[i] * T[0][j]));
    const float tr = P[0][0] + P[1][1] + P[2][2];
    const float l2 = g2.y * lam, m2 = g2.y * mu;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) K[3 * i + j] = fmaf(l2, P[i][j], m2 * (i == j ? P[j][i] + tr : P[j][i]));
}

__device__ __forceinline__ int pair_cells(uint2 p) { return (int)((p.x >> 27) | (((p.y >> 27) & 3u) << 5)); }

// Plain-FP64 redo of one pair (a modulus outside the float-pair range): the records
// of its lanes, each block times E(rho_e) in FP64.
template <int SRC>
__device__ __noinline__ void block_fp64(const BlockArgs &A, const uint32_t *B, const float *Ms, const uint16_t *rec,
                                        const uint2 *pair, int lanes, double *acc)
{
    const uint32_t *cells = B + kBlockHead + 2 * (B[0] >> 16);
    for (int p = 0; p < 9; p++) acc[p] = 0.0;
    for (int l = 0; l < lanes; l++) {
        const int cnt = pair_cells(pair[l]);
        for (int k = 0; k < cnt; k++) {
            const uint32_t r = rec[32 * k + l];
            const int64_t e = cells[r & ((1u << A.cell_bits) - 1u)];
            const int code = (int)(r >> A.cell_bits);
            const double E = simp_E(A.sp, A.rho[e]);
            if constexpr (SRC == kContract) {
                float4 cell[3];
                for (int w = 0; w < 3; w++) cell[w] = A.cdata[3 * e + w];
                float K[9];
                contract(cell, cell[2], Ms + code * 12, A.lam, A.mu, K);
                for (int p = 0; p < 9; p++) acc[p] += E * (double)K[p];
            } else if constexpr (SRC == kUniform) {
                const float2 *kb = reinterpret_cast<const float2 *>(A.kblk + (int64_t)code * 5);
                for (int p = 0; p < 9; p++) acc[p] += E * ((double)kb[p].x + (double)kb[p].y);
            } else {
                const int ld = D * A.nb;
                const float2 *kb = A.K + (e * ld + D * (code / A.nb)) * ld + D * (code % A.nb);
                for (int p = 0; p < 9; p++) acc[p] += E * KLoad<float2>::get64(kb + (p / 3) * ld + p % 3);
            }
        }
    }
}

// One record row's blocks of a stream, this lane's: whole 16-byte pieces lane by lane, then the ninth entries.
struct Blocks {
    float2 k[9];
    __device__ __forceinline__ void load(const unsigned char *stream, int row, int lane)
    {
        const float4 *b = reinterpret_cast<const float4 *>(stream + (int64_t)row * kRowBytes);
#pragma unroll
        for (int w = 0; w < 4; w++) {
            const float4 f = __ldcs(b + 32 * w + lane);
            k[2 * w] = make_float2(f.x, f.y);
            k[2 * w + 1] = make_float2(f.z, f.w);
        }
        k[8] = __ldcs(reinterpret_cast<const float2 *>(b + 128) + lane);
    }
};

// W warps assemble, one more moves data.  In step k that warp waits until the others
// have left chunk k - 2 and hands its rows to the copy engine, starts the copy of
// record k + 2 into the place that chunk k - 2 had,
// gathers the cells of chunk k + 1 and opens it, and frees the place of chunk
// k's rows once the copy engine has read the rows staged there.  The assembling warps
// look for the freed place only before their first rows of a chunk.  They are never
// more than two chunks apart (chunk k + 2 opens once all have left chunk k - 1).
template <int SRC, int W, int MINB>
__global__ void __launch_bounds__(32 * (W + 1), MINB) k_block_rows(const BlockArgs A)
{
    constexpr int CB = kCellBytes<SRC>;
    extern __shared__ uint4 sm4[];
    double *const stages = reinterpret_cast<double *>(sm4);
    const int sstride = (A.max_stage + 1) & ~1;
    uint4 *const blobs = sm4 + sstride;
    unsigned char *const cbuf = reinterpret_cast<unsigned char *>(blobs + 4 * A.max_blob);
    const int cstride = (A.max_cells * CB + 15) & ~15;
    float *const Ms = reinterpret_cast<float *>(cbuf + 3 * cstride);   // kContract: the reference integrals
    // record there; record and cells there; place of the rows free; chunk assembled
    __shared__ uint64_t s_rec[4], s_full[3], s_free[2], s_done[4];
    __shared__ int s_more[3], s_tile[3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if constexpr (SRC == kContract)
        for (int t = tid; t < A.nm; t += 32 * (W + 1)) Ms[t] = A.M[t];
    if (tid == 0) {
        for (int q = 0; q < 4; q++) {
            mbar_init(&s_rec[q], 1);
            mbar_init(&s_done[q], W);
        }
        for (int q = 0; q < 3; q++) mbar_init(&s_full[q], 1);
        for (int q = 0; q < 2; q++) mbar_init(&s_free[q], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    auto raise = [&]() {
        if (lane == 0) {
            *A.expired = 1u;
            __threadfence_system();
        }
    };
    if (warp == W) {
        const bool al16 = (reinterpret_cast<uintptr_t>(A.vals) & 15u) == 0;
        auto grab = [&]() -> int64_t {
            unsigned t = 0;
            if (lane == 0) t = atomicAdd(A.ticket, 1u);
            return (int64_t)__shfl_sync(kFull, t, 0);
        };
        auto bounds = [&](int64_t c, uint32_t &u0, uint32_t &u1) {
            u0 = u1 = 0u;
            if (c < A.nchunks) {
                u0 = __ldg(A.coff + c);
                u1 = __ldg(A.coff + c + 1);
            }
        };
        int issued = 0, landed = 0;   // records on their way, and waited for: record i in place i mod 4
        auto load_record = [&](uint32_t u0, uint32_t u1) {
            if (u1 <= u0) return;
            const int q = issued++ & 3;
            if (lane == 0) bulk_load(blobs + q * A.max_blob, A.blob + u0, 16u * (u1 - u0), &s_rec[q]);
        };
        auto wait_record = [&](int tries) {
            if (!mbar_wait(&s_rec[landed & 3], (landed >> 2) & 1, tries)) return false;
            landed++;
            return true;
        };
        auto record = [&](int k) { return reinterpret_cast<const uint32_t *>(blobs + (k & 3) * A.max_blob); };
        // the staged rows of the chunk with record B to the CSR values
        auto store_rows = [&](const uint32_t *B, const double *stage) {
            const int nn = (int)(B[0] >> 16);
            if (al16) {
                for (int i = lane; i < nn; i += 32) {
                    const uint32_t off = B[kBlockHead + 2 * i], w = B[kBlockHead + 1 + 2 * i];
                    const int n = D * D * (int)(w >> 16);
                    const double *src = stage + (w & 0xffffu);
                    double *dst = A.vals + (int64_t)D * D * off;
                    // a value at an odd 8-byte place at either end goes out by a plain store
                    const int head = (int)(off & 1u), mid = (n - head) & ~1;
                    if (mid > 0) bulk_store(dst + head, src + head, 8u * (uint32_t)mid);
                    if (head) __stcs(dst, src[0]);
                    if (n - head - mid) __stcs(dst + n - 1, src[n - 1]);
                }
            } else {
                // values at an odd 8-byte address: plain stores
                for (int i = 0; i < nn; i++) {
                    const uint32_t off = B[kBlockHead + 2 * i], w = B[kBlockHead + 1 + 2 * i];
                    const int n = D * D * (int)(w >> 16);
                    for (int t = lane; t < n; t += 32)
                        __stcs(A.vals + (int64_t)D * D * off + t, stage[(w & 0xffffu) + t]);
                }
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            __syncwarp();
        };
        auto gather_cells = [&](const uint32_t *B, unsigned char *dst) {
            const uint32_t nc = B[0] & 0xffffu;
            const uint32_t *cells = B + kBlockHead + 2 * (B[0] >> 16);
            if constexpr (SRC == kContract) {
                for (uint32_t t = lane; t < 4 * nc; t += 32) {
                    const uint32_t i = t >> 2, w = t & 3u;
                    const int64_t e = cells[i];
                    unsigned char *d = dst + CB * i;
                    if (w < 2) cp_async16(d + 16 * w, A.cdata + 3 * e + w);
                    else if (w == 2) cp_async8(d + 32, A.cdata + 3 * e + 2);
                    else cp_async8(d + 40, A.Edf + e);
                }
            } else {
                for (uint32_t t = lane; t < nc; t += 32) cp_async8(dst + 8 * t, A.Edf + cells[t]);
            }
            cp_async_commit();
        };
        auto open = [&](int q, bool more) {
            __syncwarp();
            if (lane == 0) {
                s_more[q] = more;
                s_tile[q] = 0;
                mbar_arrive(&s_full[q]);
            }
        };
        uint32_t u0, u1;
        int64_t c = grab();
        bounds(c, u0, u1);
        load_record(u0, u1);
        bool more = c < A.nchunks, ok = true;
        c = grab();
        bounds(c, u0, u1);
        load_record(u0, u1);
        bool more1 = c < A.nchunks;   // chunk k + 1 exists
        c = grab();
        bounds(c, u0, u1);            // chunk k + 2
        if (more) {
            ok = wait_record(A.tries);
            if (ok) gather_cells(record(0), cbuf);
            cp_async_wait_all();
        }
        int q = 0, last = more ? 1 : 0;   // (k + 1) mod 3; chunks known to exist
        more = more && ok;
        open(0, more);
        for (int k = 0; ok && k < last + 2; k++) {
            const int s = k & 1;
            q = q == 2 ? 0 : q + 1;
            if (k >= 2) {
                ok = mbar_wait(&s_done[(k - 2) & 3], ((k - 2) >> 2) & 1, A.tries);
                if (!ok) break;
                store_rows(record(k - 2), stages + s * sstride);
            }
            if (!more) continue;
            load_record(u0, u1);
            const bool more2 = c < A.nchunks;
            if (more1) {
                ok = wait_record(A.tries);
                if (!ok) break;
                gather_cells(record(k + 1), cbuf + q * cstride);
                last++;
                c = grab();
                bounds(c, u0, u1);
            }
            // the rows staged two chunks ago have been read: their place is free
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_free[s]);
            cp_async_wait_all();
            open(q, more1);
            more = more1;
            more1 = more2;
        }
        if (!ok) {
            raise();
            __syncwarp();
            if (more && lane == 0) {   // the next chunk, which is not there
                s_more[q] = 0;
                mbar_arrive(&s_full[q]);
            }
            while (landed < issued && wait_record(kBlockWaitTries)) {
            }
        }
        cp_async_wait_all();
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        // the last CTA to finish sets the counter back to zero for the next call
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            if (atomicAdd(A.ticket + 1, 1u) == gridDim.x - 1u) {
                A.ticket[0] = 0u;
                A.ticket[1] = 0u;
            }
        }
        return;
    }

    const uint32_t cmask = (1u << A.cell_bits) - 1u;
    int q = 0;
    unsigned pq = 0;   // parity of s_full[q]
    for (int k = 0;; k++) {
        const int s = k & 1;
        if (!mbar_wait(&s_full[q], pq, kBlockWaitTries)) return raise();
        if (!s_more[q]) return;
        const uint32_t *B = reinterpret_cast<const uint32_t *>(blobs + (k & 3) * A.max_blob);
        const unsigned char *const cb = cbuf + q * cstride;
        bool free = false;   // the place of this chunk's rows is known to be free
        double *const stage = stages + s * sstride;
        const int ntiles = (int)(B[1] & 0xffffu);
        const uint32_t *const tiles = B + (B[2] & 0xffffu);
        const uint2 *const pairs = reinterpret_cast<const uint2 *>(B + (B[2] >> 16));
        const uint16_t *const recs = reinterpret_cast<const uint16_t *>(B + B[3]);
        int tk = 0;
        if (lane == 0) tk = atomicAdd(&s_tile[q], 1);
        int t = __shfl_sync(kFull, tk, 0);
        Blocks next;   // kStream: the row after the one being added, across the ends of tiles
        const unsigned char *const stream =
            reinterpret_cast<const unsigned char *>(A.kblk) + (int64_t)B[4] * kRowBytes;
        if constexpr (SRC == kStream)
            if (t < ntiles) next.load(stream, (int)(tiles[t] & 0xffffu), lane);
        while (t < ntiles) {
            if (lane == 0) tk = atomicAdd(&s_tile[q], 1);   // the tile after this one
            const uint32_t tw = tiles[t];
            const uint2 pr = pairs[32 * t + lane];
            const int row0 = (int)(tw & 0xffffu), rows = (int)(tw >> 16);
            const uint16_t *const rec = recs + 32 * row0 + lane;
            const int cnt = pair_cells(pr), lg = (int)(pr.y >> 29);
            float2 v[9];
#pragma unroll
            for (int p = 0; p < 9; p++) v[p] = make_float2(0.f, 0.f);
            uint32_t rn = rec[0];
            for (int r_ = 0; r_ < rows; r_++) {
                const uint32_t r = rn;
                rn = rec[32 * min(r_ + 1, rows - 1)];
                Blocks cur;
                if constexpr (SRC == kStream) {
                    cur = next;
                    if (r_ + 1 < rows) {
                        next.load(stream, row0 + r_ + 1, lane);
                    } else {
                        const int tn = __shfl_sync(kFull, tk, 0);
                        if (tn < ntiles) next.load(stream, (int)(tiles[tn] & 0xffffu), lane);
                    }
                }
                if (r_ >= cnt) continue;
                const unsigned char *const cell = cb + CB * (r & cmask);
                const uint32_t code = r >> A.cell_bits;
                if constexpr (SRC == kContract) {
                    const float4 *cf = reinterpret_cast<const float4 *>(cell);
                    const float4 g2 = cf[2];
                    float K[9];
                    contract(cf, g2, Ms + 12 * code, A.lam, A.mu, K);
#pragma unroll
                    for (int p = 0; p < 9; p++) acc_add(v[p].x, v[p].y, times(df{g2.z, g2.w}, K[p]));
                } else {
                    const float2 E2 = *reinterpret_cast<const float2 *>(cell);
                    const df E{E2.x, E2.y};
                    if constexpr (SRC == kUniform) {
                        const float4 *kb = A.kblk + (int64_t)code * 5;
                        float4 f[5];
#pragma unroll
                        for (int w = 0; w < 5; w++) f[w] = __ldg(kb + w);
#pragma unroll
                        for (int p = 0; p < 9; p++)
                            cur.k[p] = (p & 1) ? make_float2(f[p / 2].z, f[p / 2].w) : make_float2(f[p / 2].x, f[p / 2].y);
                    }
#pragma unroll
                    for (int p = 0; p < 9; p++) acc_add(v[p].x, v[p].y, df_mul_raw(E, df{cur.k[p].x, cur.k[p].y}));
                }
            }
            // a modulus outside the float-pair range has a NaN tail, which the sums keep
            bool bad = isnan(v[0].y);
            // the lanes of a shared pair, in a fixed tree (the first lane ends with the sum)
            if (__any_sync(kFull, lg > 0)) {
#pragma unroll 1
                for (int o = 0; o < 5; o++) {
                    if (!__any_sync(kFull, lg > o)) break;
                    const bool badp = __shfl_down_sync(kFull, (int)bad, 1 << o) != 0;
                    const bool add = lg > o;
                    bad |= add && badp;
#pragma unroll
                    for (int p = 0; p < 9; p++) {
                        const float x = __shfl_down_sync(kFull, v[p].x, 1 << o),
                                    l = __shfl_down_sync(kFull, v[p].y, 1 << o);
                        if (add) acc_add(v[p].x, v[p].y, df{x, l});
                    }
                }
            }
            // the largest head of the block (NaN when one is): beyond the floats it is redone
            // in FP64 too; below kRebiasMin the fast conversion would add up to 2^-126 to
            // entries that are not far above it
            float big = 0.f;
#pragma unroll
            for (int p = 0; p < 9; p++) big = max_nan(big, fabsf(v[p].x));
            bad |= !(big <= FLT_MAX);
            if (!free) {
                if (!mbar_wait(&s_free[s], (k >> 1) & 1, kBlockWaitTries)) return raise();
                free = true;
            }
            const uint32_t o1 = pr.x & 0xffffu;
            if (o1 != 0xffffu && !(lane & ((1 << lg) - 1))) {
                double dv[9];
                if (bad) {
                    // (a copy: dv itself stays in registers)
                    double acc[9];
                    block_fp64<SRC>(A, B, Ms, rec, pairs + 32 * t + lane, 1 << lg, acc);
#pragma unroll
                    for (int p = 0; p < 9; p++) dv[p] = acc[p];
                } else if (big < kRebiasMin) {
#pragma unroll
                    for (int p = 0; p < 9; p++) dv[p] = (double)v[p].x + (double)v[p].y;
                } else {
#pragma unroll
                    for (int p = 0; p < 9; p++) dv[p] = pair_to_double_rebias(v[p].x, v[p].y);
                }
                double *const d1 = stage + o1;
                const int rl1 = (int)((pr.x >> 16) & 0x7ffu);
#pragma unroll
                for (int i = 0; i < D; i++)
#pragma unroll
                    for (int j = 0; j < D; j++) d1[i * rl1 + j] = dv[D * i + j];
                const uint32_t o2 = pr.y & 0xffffu;
                if (o2 != 0xffffu) {
                    double *const d2 = stage + o2;
                    const int rl2 = (int)((pr.y >> 16) & 0x7ffu);
#pragma unroll
                    for (int j = 0; j < D; j++)
#pragma unroll
                        for (int i = 0; i < D; i++) d2[j * rl2 + i] = dv[D * i + j];
                }
            }
            __syncwarp();
            t = __shfl_sync(kFull, tk, 0);
        }
        // the rows this warp staged, before the copy engine reads them (the others may
        // still be in chunk k - 2: each of the last four chunks has its own count)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&s_done[k & 3]);
        if (++q == 3) {
            q = 0;
            pq ^= 1u;
        }
    }
}

// At mesh creation: every record's block of the cached element matrices in the order
// of the stream, one block of threads per chunk.
__global__ void k_block_stream(int64_t nchunks, const uint4 *__restrict__ blob, const uint32_t *__restrict__ coff,
                               int cell_bits, int nb, const float2 *__restrict__ K, unsigned char *__restrict__ out)
{
    const int ld = D * nb;
    for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const uint32_t *B = reinterpret_cast<const uint32_t *>(blob + coff[c]);
        const uint32_t *cells = B + kBlockHead + 2 * (B[0] >> 16);
        const uint16_t *recs = reinterpret_cast<const uint16_t *>(B + B[3]);
        const int n = 32 * (int)(B[1] >> 16);
        unsigned char *o = out + (int64_t)B[4] * kRowBytes;
        for (int x = threadIdx.x; x < 9 * n; x += blockDim.x) {
            const int p = x % 9, i = x / 9, lane = i & 31;
            const uint32_t r = recs[i];
            const int64_t e = cells[r & ((1u << cell_bits) - 1u)];
            const int code = (int)(r >> cell_bits);
            float2 *row = reinterpret_cast<float2 *>(o + (int64_t)(i >> 5) * kRowBytes);
            // whole 16-byte pieces lane by lane, then the ninth entries
            row[p == 8 ? 8 * 32 + lane : (p / 2) * 64 + 2 * lane + p % 2] =
                K[(e * ld + D * (code / nb) + p / 3) * ld + D * (code % nb) + p % 3];
        }
    }
}

template <int SRC, int W, int MINB>
cudaError_t block_launch(const soptx_mesh_s &m, const double *rho, double *vals, cudaStream_t st)
{
    const auto &h = m.h;
    const auto &d = m.d;
    BlockArgs A;
    A.nchunks = d.bchunks;
    A.ticket = d.cticket;
    A.expired = d.bexpired;
    A.tries = d.btries;
    A.blob = d.bblob;
    A.coff = d.bcoff;
    A.max_blob = d.bmax_blob;
    A.max_cells = d.bmax_cells;
    A.max_stage = d.bmax_stage;
    A.cell_bits = d.bcell_bits;
    A.cdata = d.bcell;
    A.M = d.bM;
    A.nm = SRC == kContract ? h.nb * h.nb * 12 : 0;
    A.kblk = d.bkblk;
    A.Edf = d.Edf;
    A.rho = rho;
    A.K = SRC == kStream ? static_cast<const float2 *>(d.K) : nullptr;
    A.nb = h.nb;
    A.sp = simp_params(m.mat);
    A.lam = (float)(m.mat.lam);
    A.mu = (float)(m.mat.mu);
    A.vals = vals;
    auto kern = k_block_rows<SRC, W, MINB>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, d.bsmem);
    if (err != cudaSuccess) return err;
    int dev = 0, sms = 0, per_sm = 0;
    err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err == cudaSuccess)
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * (W + 1), (size_t)d.bsmem);
    if (err != cudaSuccess) return err;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(A.nchunks, (int64_t)sms * std::max(per_sm, 1)));
    kern<<<grid, 32 * (W + 1), d.bsmem, st>>>(A);
    return cudaGetLastError();
}

}  // namespace

int64_t block_row_bytes() { return kRowBytes; }

// Shared memory of a CTA: two chunks' staged rows, four chunk records, three chunks' cells,
// then the reference integrals (kContract).
int64_t block_smem(int src, int nb, const BlockTables &T)
{
    const int64_t cb = src == kContract ? kCellBytes<kContract> : kCellBytes<kUniform>;
    const int64_t more = src == kContract ? (int64_t)nb * nb * 12 * 4 : 0;
    return (int64_t)((T.max_stage + 1) & ~1) * 16 + 64 * (int64_t)T.max_blob + 3 * ((T.max_cells * cb + 15) & ~(int64_t)15) +
           more;
}

cudaError_t launch_block_stream(const soptx_mesh_s &m, cudaStream_t st)
{
    if (m.d.bchunks <= 0) return cudaSuccess;
    k_block_stream<<<(int)std::min<int64_t>(m.d.bchunks, 152 * 16), 256, 0, st>>>(
        m.d.bchunks, m.d.bblob, m.d.bcoff, m.d.bcell_bits, m.h.nb, static_cast<const float2 *>(m.d.K),
        reinterpret_cast<unsigned char *>(m.d.bkblk));
    return cudaGetLastError();
}

// Element moduli as float pairs (k_prep), then the block rows.
cudaError_t launch_block_rows(const soptx_mesh_s &m, const double *rho, double *vals, cudaStream_t st)
{
    cudaError_t err = launch_prep(m, rho, nullptr, st);
    if (err != cudaSuccess || m.d.bchunks == 0) return err;
    if (m.d.bsrc == kContract && m.h.nb == 4) return block_launch<kContract, 4, 4>(m, rho, vals, st);
    if (m.d.bsrc == kContract) return block_launch<kContract, 8, 2>(m, rho, vals, st);
    if (m.d.bsrc == kUniform) return block_launch<kUniform, 8, 2>(m, rho, vals, st);
    return block_launch<kStream, 8, 2>(m, rho, vals, st);
}

}  // namespace soptx
