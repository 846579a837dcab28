// Host tables of the block-row kernel (blockrows.cu): the nodes of a mesh cut
// into chunks of complete rows, and for each chunk everything its CTA needs
// (its nodes' places in the CSR values, its cells, its node pairs and their
// cells), as one contiguous record that is copied into shared memory whole.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <thread>

#include "internal.h"

namespace soptx {
namespace {

// Index along the Hilbert curve of the point p (b bits per axis), by Skilling's
// transpose algorithm ("Programming the Hilbert curve", AIP Conf. Proc. 707,
// 2004): consecutive indices are neighbouring cells, so a run of them is compact.
uint64_t hilbert_index(uint32_t *x, int b, int d)
{
    const uint32_t top = 1u << (b - 1);
    for (uint32_t q = top; q > 1; q >>= 1) {
        const uint32_t p = q - 1;
        for (int i = 0; i < d; i++) {
            if (x[i] & q) {
                x[0] ^= p;
            } else {
                const uint32_t t = (x[0] ^ x[i]) & p;
                x[0] ^= t;
                x[i] ^= t;
            }
        }
    }
    for (int i = 1; i < d; i++) x[i] ^= x[i - 1];
    uint32_t t = 0;
    for (uint32_t q = top; q > 1; q >>= 1)
        if (x[d - 1] & q) t ^= q - 1;
    for (int i = 0; i < d; i++) x[i] ^= t;
    uint64_t h = 0;
    for (int k = b - 1; k >= 0; k--)
        for (int i = 0; i < d; i++) h = (h << 1) | ((x[i] >> k) & 1u);
    return h;
}

int64_t shares_for(int64_t items, int64_t least)
{
    return std::max<int64_t>(1, std::min<int64_t>({16, (int64_t)std::thread::hardware_concurrency(), items / least}));
}

// f(0) .. f(n - 1), one per thread; those whose thread cannot be had run in this one.  f does not throw.
template <typename F>
void in_threads(int64_t n, const F &f)
{
    std::vector<std::thread> pool;
    int64_t here = 1;
    try {
        pool.reserve((size_t)n);
        for (; here < n; here++) pool.emplace_back(f, here);
    } catch (const std::exception &) {
    }
    f(0);
    for (int64_t k = here; k < n; k++) f(k);
    for (auto &t : pool) t.join();
}

// Processing order of the nodes: by the place of their first cell along a
// Hilbert curve through the cells' centroids, so consecutive nodes are close
// together, share most of their cells and are each other's neighbours.
std::vector<int32_t> node_order(const HostMesh &h, const double *coords, const int32_t *cv)
{
    const int d = h.dim, nvc = h.nvc, bits = d == 2 ? 16 : 10;
    const int64_t shares = shares_for(h.nc, 4096);
    std::vector<double> cen((size_t)h.nc * d), lo_s((size_t)shares * d, HUGE_VAL), hi_s((size_t)shares * d, -HUGE_VAL);
    in_threads(shares, [&](int64_t k) {
        for (int64_t e = h.nc * k / shares; e < h.nc * (k + 1) / shares; e++)
            for (int i = 0; i < d; i++) {
                double s = 0.0;
                for (int v = 0; v < nvc; v++) s += coords[(int64_t)cv[e * nvc + v] * d + i];
                s /= nvc;
                cen[(size_t)e * d + i] = s;
                lo_s[(size_t)k * d + i] = std::min(lo_s[(size_t)k * d + i], s);
                hi_s[(size_t)k * d + i] = std::max(hi_s[(size_t)k * d + i], s);
            }
    });
    double lo[3] = {0, 0, 0}, ext = 0.0;
    for (int i = 0; i < d; i++) {
        double a = HUGE_VAL, b = -HUGE_VAL;
        for (int64_t k = 0; k < shares; k++) {
            a = std::min(a, lo_s[(size_t)k * d + i]);
            b = std::max(b, hi_s[(size_t)k * d + i]);
        }
        lo[i] = a;
        ext = std::max(ext, b - a);
    }
    const double scale = ext > 0.0 ? ((1u << bits) - 1) / ext : 0.0;
    std::vector<std::pair<uint64_t, int32_t>> key((size_t)h.nc);
    in_threads(shares, [&](int64_t k) {
        for (int64_t e = h.nc * k / shares; e < h.nc * (k + 1) / shares; e++) {
            uint32_t x[3] = {0, 0, 0};
            for (int i = 0; i < d; i++) x[i] = (uint32_t)((cen[(size_t)e * d + i] - lo[i]) * scale);
            key[(size_t)e] = {hilbert_index(x, bits, d), (int32_t)e};
        }
        std::sort(key.begin() + h.nc * k / shares, key.begin() + h.nc * (k + 1) / shares);
    });
    for (int64_t w = 1; w < shares; w *= 2)   // merges of sorted shares
        in_threads((shares + 2 * w - 1) / (2 * w), [&](int64_t k) {
            auto at = [&](int64_t q) { return key.begin() + h.nc * std::min(q, shares) / shares; };
            std::inplace_merge(at(2 * w * k), at(2 * w * k + w), at(2 * w * k + 2 * w));
        });
    std::vector<int32_t> order;
    order.reserve((size_t)h.nn);
    std::vector<char> seen((size_t)h.nn, 0);
    for (auto &k : key)
        for (int a = 0; a < h.nb; a++) {
            const int32_t n = h.cell_node[(size_t)k.second * h.nb + a];
            if (!seen[(size_t)n]) {
                seen[(size_t)n] = 1;
                order.push_back(n);
            }
        }
    return order;   // nodes of no cell have no rows
}

// The records of chunks c0 .. c1 - 1.  False when one does not fit the record's fields.
bool build_chunks(const HostMesh &h, const BlockLimits &L, const std::vector<int32_t> &order,
                  const std::vector<size_t> &start, const std::vector<int32_t> &node_chunk,
                  const std::vector<int32_t> &node_loc, const std::vector<int32_t> &cinc, int64_t c0, int64_t c1,
                  BlockTables &T)
{
    const int d = h.dim, nb = h.nb;
    T.coff.push_back(0);
    T.blob.resize(1);
    std::vector<int32_t> cell_chunk((size_t)h.nc, -1), cell_loc((size_t)h.nc, 0);
    std::vector<int32_t> cells;
    struct Pair {
        uint32_t o1, rl1, o2, rl2;   // places of the block and of its transpose (o2 = 0xffff: none)
        uint32_t lg, rows;           // 2^lg lanes of `rows` cells each share the pair
        uint32_t r0, cnt;            // its records
    };
    std::vector<Pair> pairs;
    std::vector<uint32_t> prec, soff;
    std::vector<int32_t> scnt, sstart, sfill;
    std::vector<uint32_t> idx, key_start, trows, tsort;
    std::vector<std::pair<uint32_t, uint32_t>> lane;   // (pair, share) of each lane
    bool ok = true;
    constexpr uint32_t kNone = 0xffffu;
    for (int64_t chunk = c0; chunk < c1 && ok; chunk++) {
        const int32_t *const nodes = order.data() + start[(size_t)chunk];
        const size_t nnode = start[(size_t)chunk + 1] - start[(size_t)chunk];
        cells.clear();
        for (size_t i = 0; i < nnode; i++)
            for (int32_t q = h.inc_ptr[(size_t)nodes[i]]; q < h.inc_ptr[(size_t)nodes[i] + 1]; q++) {
                const int32_t e = h.inc_e[(size_t)q];
                if (cell_chunk[(size_t)e] != chunk) {
                    cell_chunk[(size_t)e] = (int32_t)chunk;
                    cell_loc[(size_t)e] = (int32_t)cells.size();
                    cells.push_back(e);
                }
            }
        // the staged rows of each node start at the 16-byte phase of their place in the CSR values
        uint32_t s = 0;
        soff.clear();
        for (size_t i = 0; i < nnode; i++) {
            const int32_t n = nodes[i];
            const int64_t off = h.node_off[(size_t)n], deg = h.node_off[(size_t)n + 1] - off;
            if (((int64_t)d * d * off - s) & 1) s++;
            soff.push_back(s);
            s += (uint32_t)(d * d * deg);
        }
        if (s > 0xfffeu) ok = false;
        T.max_stage = std::max(T.max_stage, (int)s);
        T.max_nodes = std::max(T.max_nodes, (int)nnode);
        T.max_cells = std::max(T.max_cells, (int)cells.size());
        pairs.clear();
        prec.clear();
        for (size_t i = 0; i < nnode; i++) {
            const int32_t a = nodes[i];
            const int32_t q0 = h.inc_ptr[(size_t)a], q1 = h.inc_ptr[(size_t)a + 1];
            const int64_t off = h.node_off[(size_t)a];
            const int deg = (int)(h.node_off[(size_t)a + 1] - off);
            // the node's records grouped by column block; a block whose other node comes
            // earlier in the chunk is that node's (written transposed)
            auto mine = [&](int32_t b) { return !L.sym || node_chunk[(size_t)b] != chunk || node_loc[(size_t)b] >= (int32_t)i; };
            scnt.assign((size_t)deg, 0);
            for (int32_t q = q0; q < q1; q++) {
                const int32_t *cn = &h.cell_node[(size_t)h.inc_e[(size_t)q] * nb];
                for (int j = 0; j < nb; j++)
                    if (mine(cn[j])) scnt[h.pos[(size_t)q * nb + j]]++;
            }
            sstart.assign((size_t)deg + 1, 0);
            for (int p = 0; p < deg; p++) sstart[(size_t)p + 1] = sstart[(size_t)p] + scnt[(size_t)p];
            sfill.assign(sstart.begin(), sstart.end() - 1);
            const uint32_t base = (uint32_t)prec.size();
            prec.resize(base + (size_t)sstart[(size_t)deg]);
            for (int32_t q = q0; q < q1; q++) {
                const int32_t e = h.inc_e[(size_t)q];
                const int32_t *cn = &h.cell_node[(size_t)e * nb];
                const uint32_t al = h.inc_a[(size_t)q];
                for (int j = 0; j < nb; j++)
                    if (mine(cn[j]))
                        prec[base + (size_t)sfill[h.pos[(size_t)q * nb + j]]++] =
                            (uint32_t)cell_loc[(size_t)e] | (al * nb + (uint32_t)j) << 16;
            }
            for (int p = 0; p < deg; p++) {
                const uint32_t c = (uint32_t)scnt[(size_t)p];
                if (c == 0) continue;
                const int32_t b = h.nbr[(size_t)(off + p)];
                Pair w{soff[i] + (uint32_t)(d * p), (uint32_t)(d * deg), kNone, 0u, 0u, c, base + (uint32_t)sstart[(size_t)p], c};
                if (L.sym && b != a && node_chunk[(size_t)b] == chunk) {
                    // the place of a in b's rows, from the pair's first cell
                    const uint32_t r = prec[w.r0], code = r >> 16;
                    const int32_t e = cells[r & 0xffffu];
                    const int pba = h.pos[(size_t)cinc[(size_t)e * nb + code % nb] * nb + code / nb];
                    const int degb = (int)(h.node_off[(size_t)b + 1] - h.node_off[(size_t)b]);
                    w.o2 = soff[(size_t)node_loc[(size_t)b]] + (uint32_t)(d * pba);
                    w.rl2 = (uint32_t)(d * degb);
                }
                while (w.rows > (uint32_t)L.cap && w.lg < 5) {
                    w.lg++;
                    w.rows = (c + (1u << w.lg) - 1) >> w.lg;
                }
                if (w.rows > 127) ok = false;
                pairs.push_back(w);
            }
        }
        // pairs shared by most lanes first (so a pair's lanes are aligned to their
        // number), then by the cells per lane
        const uint32_t nk = 6 * 128;
        key_start.assign(nk + 1, 0);
        auto key = [&](const Pair &w) { return (5 - w.lg) * 128 + (127 - std::min(w.rows, 127u)); };
        for (auto &w : pairs) key_start[key(w) + 1]++;
        for (uint32_t k = 0; k < nk; k++) key_start[k + 1] += key_start[k];
        idx.resize(pairs.size());
        for (uint32_t k = 0; k < pairs.size(); k++) idx[key_start[key(pairs[k])]++] = k;
        if (L.by_code)
            std::stable_sort(idx.begin(), idx.end(), [&](uint32_t x, uint32_t y) {
                const uint32_t kx = key(pairs[x]), ky = key(pairs[y]);
                return kx != ky ? kx < ky : (prec[pairs[x].r0] >> 16) < (prec[pairs[y].r0] >> 16);
            });
        // lanes: (pair, share) in tiles of 32
        std::vector<uint32_t> &B = T.blob[0];
        const size_t b0 = B.size();
        size_t lanes = 0;
        for (auto &w : pairs) lanes += (size_t)1 << w.lg;
        const uint32_t ntiles = (uint32_t)((lanes + 31) / 32);
        // the lanes' pairs and shares, and the record rows of each tile
        lane.assign((size_t)ntiles * 32, {UINT32_MAX, 0});
        trows.assign(ntiles, 0);
        {
            size_t np = 0;
            uint32_t share = 0;
            for (size_t l = 0; l < lanes; l++) {
                const Pair &w = pairs[idx[np]];
                lane[l] = {idx[np], share};
                trows[l / 32] = std::max(trows[l / 32], std::min(w.rows, w.cnt - std::min(w.cnt, share * w.rows)));
                if (++share == 1u << w.lg) {
                    share = 0;
                    np++;
                }
            }
        }
        // tiles with the most rows first: the warps take them in this order
        tsort.resize(ntiles);
        for (uint32_t t = 0; t < ntiles; t++) tsort[t] = t;
        std::stable_sort(tsort.begin(), tsort.end(), [&](uint32_t x, uint32_t y) { return trows[x] > trows[y]; });
        const uint32_t nnodes = (uint32_t)nnode;
        const uint32_t wn = kBlockHead, wc = wn + 2 * nnodes, wt = wc + (uint32_t)cells.size();
        uint32_t wp = wt + ntiles;
        wp += wp & 1;
        const uint32_t wr = wp + 64 * ntiles;
        B.resize(b0 + wr, 0u);
        B[b0] = (uint32_t)cells.size() | nnodes << 16;
        B[b0 + 1] = ntiles;
        B[b0 + 2] = wt | wp << 16;
        B[b0 + 3] = wr;
        if (T.rows > (int64_t)UINT32_MAX) ok = false;
        B[b0 + 4] = (uint32_t)T.rows;
        if (wp > 0xffffu || ntiles > 0xffffu) ok = false;
        for (size_t i = 0; i < nnodes; i++) {
            B[b0 + wn + 2 * i] = (uint32_t)h.node_off[(size_t)nodes[i]];
            B[b0 + wn + 2 * i + 1] = soff[i] | (uint32_t)(h.node_off[(size_t)nodes[i] + 1] - h.node_off[(size_t)nodes[i]]) << 16;
        }
        for (size_t i = 0; i < cells.size(); i++) B[b0 + wc + i] = (uint32_t)cells[i];
        uint32_t row = 0, place = 0;
        for (uint32_t t : tsort) {
            const uint32_t rows = trows[t];
            for (uint32_t l = 0; l < 32; l++) {
                const auto &ln = lane[32 * (size_t)t + l];
                uint32_t x = kNone, y = kNone;
                if (ln.first != UINT32_MAX) {
                    const Pair &q = pairs[ln.first];
                    const uint32_t n = std::min(q.rows, q.cnt - std::min(q.cnt, ln.second * q.rows));
                    x = q.o1 | q.rl1 << 16 | (n & 31u) << 27;
                    y = q.o2 | q.rl2 << 16 | (((n >> 5) & 3u) | q.lg << 2) << 27;
                }
                B[b0 + wp + 2 * (32 * place + l)] = x;
                B[b0 + wp + 2 * (32 * place + l) + 1] = y;
            }
            if (row + rows > 0xffffu) ok = false;
            B[b0 + wt + place] = row | rows << 16;
            const size_t r0 = B.size();
            B.resize(r0 + 16 * (size_t)rows, 0u);
            for (uint32_t l = 0; l < 32; l++) {
                const auto &ln = lane[32 * (size_t)t + l];
                if (ln.first == UINT32_MAX) continue;
                const Pair &q = pairs[ln.first];
                const uint32_t first = ln.second * q.rows, n = std::min(q.rows, q.cnt - std::min(q.cnt, first));
                // a lane past its cells repeats its last record (its result is not used)
                for (uint32_t k = 0; k < rows; k++) {
                    const uint32_t r = prec[q.r0 + (n ? first + std::min(k, n - 1) : 0u)];
                    B[r0 + 16 * k + l / 2] |= ((r & 0xffffu) | (r >> 16) << T.cell_bits) << (16 * (l & 1));
                }
            }
            row += rows;
            place++;
        }
        B[b0 + 1] |= row << 16;
        T.rows += row;
        B.resize((B.size() + 3) & ~(size_t)3, 0u);
        T.max_blob = std::max(T.max_blob, (int)((B.size() - b0) / 4));
        if (B.size() / 4 > (size_t)UINT32_MAX) ok = false;
        T.coff.push_back((uint32_t)(B.size() / 4));
    }
    return ok;
}

}  // namespace

bool build_block_tables(const HostMesh &h, const double *coords, const int32_t *cv, const BlockLimits &L,
                        BlockTables &T)
{
    const int d = h.dim, nb = h.nb;
    if (h.node_off[(size_t)h.nn] > (int64_t)UINT32_MAX || d * h.max_deg > 2047 || nb > 255) return false;
    const std::vector<int32_t> order = node_order(h, coords, cv);
    // the incidence of each (cell, local node)
    std::vector<int32_t> cinc((size_t)h.nc * nb, 0);
    for (int64_t n = 0; n < h.nn; n++)
        for (int32_t q = h.inc_ptr[(size_t)n]; q < h.inc_ptr[(size_t)n + 1]; q++)
            cinc[(size_t)h.inc_e[(size_t)q] * nb + h.inc_a[(size_t)q]] = q;
    T = BlockTables{};
    int code_bits = 1;
    while (nb * nb > 1 << code_bits) code_bits++;
    if (code_bits > 14) return false;
    const int cell_bits = 16 - code_bits;
    // the chunks: consecutive nodes of the order
    const int most_cells = std::min(L.cells, 1 << cell_bits);
    std::vector<size_t> start;   // [chunks + 1] places in the order
    std::vector<int32_t> node_chunk((size_t)h.nn, -1), node_loc((size_t)h.nn, 0);
    {
        std::vector<int32_t> cell_chunk((size_t)h.nc, -1);
        int32_t chunk = -1;
        int blocks = 0, cells = 0;
        for (size_t i = 0; i < order.size(); i++) {
            const int32_t n = order[i];
            const int deg = (int)(h.node_off[(size_t)n + 1] - h.node_off[(size_t)n]);
            const int32_t q0 = h.inc_ptr[(size_t)n], q1 = h.inc_ptr[(size_t)n + 1];
            int fresh = 0;
            for (int32_t q = q0; q < q1; q++) fresh += cell_chunk[(size_t)h.inc_e[(size_t)q]] != chunk;
            if (chunk < 0 || blocks + deg > L.blocks || cells + fresh > most_cells || (int)(i - start.back()) >= L.nodes) {
                if (q1 - q0 > 1 << cell_bits) return false;
                chunk++;
                start.push_back(i);
                blocks = cells = 0;
                fresh = q1 - q0;
            }
            node_chunk[(size_t)n] = chunk;
            node_loc[(size_t)n] = (int32_t)(i - start.back());
            blocks += deg;
            cells += fresh;
            for (int32_t q = q0; q < q1; q++) cell_chunk[(size_t)h.inc_e[(size_t)q]] = chunk;
        }
        start.push_back(order.size());
        T.nchunks = chunk + 1;
    }
    // their records, in shares of consecutive chunks, one per thread
    const int64_t shares = shares_for(T.nchunks, 64);
    std::vector<BlockTables> part((size_t)shares);
    std::vector<char> good((size_t)shares, 0);   // 0: failed, 1: built, 2: out of memory
    auto run = [&](int64_t k) {
        try {
            part[(size_t)k].cell_bits = cell_bits;
            good[(size_t)k] = build_chunks(h, L, order, start, node_chunk, node_loc, cinc, T.nchunks * k / shares,
                                           T.nchunks * (k + 1) / shares, part[(size_t)k]);
        } catch (const std::bad_alloc &) {
            good[(size_t)k] = 2;
        }
    };
    in_threads(shares, run);
    T.cell_bits = cell_bits;
    T.coff.push_back(0);
    for (int64_t k = 0; k < shares; k++) {
        BlockTables &P = part[(size_t)k];
        if (good[(size_t)k] == 2) throw std::bad_alloc();
        if (!good[(size_t)k] || T.rows + P.rows > (int64_t)UINT32_MAX ||
            (T.words + (int64_t)P.blob[0].size()) / 4 > (int64_t)UINT32_MAX)
            return false;
        const uint32_t base = T.coff.back();
        for (size_t c = 0; c + 1 < P.coff.size(); c++) P.blob[0][4 * (size_t)P.coff[c] + 4] += (uint32_t)T.rows;
        for (size_t c = 1; c < P.coff.size(); c++) T.coff.push_back(base + P.coff[c]);
        T.words += (int64_t)P.blob[0].size();
        T.blob.push_back(std::move(P.blob[0]));
        T.rows += P.rows;
        T.max_blob = std::max(T.max_blob, P.max_blob);
        T.max_cells = std::max(T.max_cells, P.max_cells);
        T.max_stage = std::max(T.max_stage, P.max_stage);
        T.max_nodes = std::max(T.max_nodes, P.max_nodes);
    }
    return true;
}

}  // namespace soptx
