// Resize on the device: one meta operator of Section 3.3.2 (project, extend,
// double, merge, product, swap of sizes) applied to many walkers' schemes at
// once, each result written into a walker of the population of the result
// format (the Resize step of the exploratory search, Section 3.4).
//
// Every operator is a coefficient re-indexing of the source term (product: of
// a source and an aux term, multiplied): the host builds, per block of output
// terms, a map from each output coefficient to a source (and aux) coefficient
// in the u | v | w row layout, and the kernel evaluates it term by term,
// restores the sign normalisation (Section 3.6), drops terms with a zero
// factor (project), and packs the terms into the destination's slot layout.
#include <climits>
#include <cstdint>
#include <vector>

#include "tfg_internal.h"

namespace tfg {

// ---------------------------------------------------------------------------
// Host: coefficient maps.  Row layout of a term of (m, n, p): u[i*n + k] at 0,
// v[k*p + j] at m*n, w[j*m + i] at m*n + n*p.
namespace {

struct Fmt {
    int m, n, p;
    int lu() const { return m * n; }
    int lv() const { return n * p; }
    int lt() const { return m * n + n * p + p * m; }
    int iu(int i, int k) const { return i * n + k; }
    int iv(int k, int j) const { return lu() + k * p + j; }
    int iw(int j, int i) const { return lu() + lv() + j * m + i; }
};

// block concatenation along `axis`: out = (a | b); maps of a's and b's terms
void merge_maps(const Fmt &a, const Fmt &b, int axis, Fmt &o, std::vector<int16_t> &ma, std::vector<int16_t> &mb) {
    o = Fmt{a.m + (axis == 0 ? b.m : 0), a.n + (axis == 1 ? b.n : 0), a.p + (axis == 2 ? b.p : 0)};
    const int oi = axis == 0 ? a.m : 0, ok = axis == 1 ? a.n : 0, oj = axis == 2 ? a.p : 0;
    ma.assign(o.lt(), -1);
    mb.assign(o.lt(), -1);
    for (int i = 0; i < o.m; ++i)
        for (int k = 0; k < o.n; ++k) {
            if (i < a.m && k < a.n) ma[o.iu(i, k)] = (int16_t)a.iu(i, k);
            if (i >= oi && i < oi + b.m && k >= ok && k < ok + b.n) mb[o.iu(i, k)] = (int16_t)b.iu(i - oi, k - ok);
        }
    for (int k = 0; k < o.n; ++k)
        for (int j = 0; j < o.p; ++j) {
            if (k < a.n && j < a.p) ma[o.iv(k, j)] = (int16_t)a.iv(k, j);
            if (k >= ok && k < ok + b.n && j >= oj && j < oj + b.p) mb[o.iv(k, j)] = (int16_t)b.iv(k - ok, j - oj);
        }
    for (int j = 0; j < o.p; ++j)
        for (int i = 0; i < o.m; ++i) {
            if (j < a.p && i < a.m) ma[o.iw(j, i)] = (int16_t)a.iw(j, i);
            if (j >= oj && j < oj + b.p && i >= oi && i < oi + b.m) mb[o.iw(j, i)] = (int16_t)b.iw(j - oj, i - oi);
        }
}

// remove index `idx` along `axis`
void project_map(const Fmt &f, int axis, int idx, Fmt &o, std::vector<int16_t> &mp) {
    o = Fmt{f.m - (axis == 0), f.n - (axis == 1), f.p - (axis == 2)};
    auto src = [&](int x, int ax) { return (axis == ax && x >= idx) ? x + 1 : x; };
    mp.assign(o.lt(), -1);
    for (int i = 0; i < o.m; ++i)
        for (int k = 0; k < o.n; ++k) mp[o.iu(i, k)] = (int16_t)f.iu(src(i, 0), src(k, 1));
    for (int k = 0; k < o.n; ++k)
        for (int j = 0; j < o.p; ++j) mp[o.iv(k, j)] = (int16_t)f.iv(src(k, 1), src(j, 2));
    for (int j = 0; j < o.p; ++j)
        for (int i = 0; i < o.m; ++i) mp[o.iw(j, i)] = (int16_t)f.iw(src(j, 2), src(i, 0));
}

// Kronecker product: row index i = i1*m2 + i2, and so on for k and j
void product_maps(const Fmt &a, const Fmt &b, Fmt &o, std::vector<int16_t> &ma, std::vector<int16_t> &mb) {
    o = Fmt{a.m * b.m, a.n * b.n, a.p * b.p};
    ma.assign(o.lt(), -1);
    mb.assign(o.lt(), -1);
    for (int i1 = 0; i1 < a.m; ++i1)
        for (int i2 = 0; i2 < b.m; ++i2)
            for (int k1 = 0; k1 < a.n; ++k1)
                for (int k2 = 0; k2 < b.n; ++k2) {
                    const int e = o.iu(i1 * b.m + i2, k1 * b.n + k2);
                    ma[e] = (int16_t)a.iu(i1, k1);
                    mb[e] = (int16_t)b.iu(i2, k2);
                }
    for (int k1 = 0; k1 < a.n; ++k1)
        for (int k2 = 0; k2 < b.n; ++k2)
            for (int j1 = 0; j1 < a.p; ++j1)
                for (int j2 = 0; j2 < b.p; ++j2) {
                    const int e = o.iv(k1 * b.n + k2, j1 * b.p + j2);
                    ma[e] = (int16_t)a.iv(k1, j1);
                    mb[e] = (int16_t)b.iv(k2, j2);
                }
    for (int j1 = 0; j1 < a.p; ++j1)
        for (int j2 = 0; j2 < b.p; ++j2)
            for (int i1 = 0; i1 < a.m; ++i1)
                for (int i2 = 0; i2 < b.m; ++i2) {
                    const int e = o.iw(j1 * b.p + j2, i1 * b.m + i2);
                    ma[e] = (int16_t)a.iw(j1, i1);
                    mb[e] = (int16_t)b.iw(j2, i2);
                }
}

// (AB)^T = B^T A^T: (m,n,p) -> (p,n,m), u' = v^T, v' = u^T, w' = w^T
void transpose_map(const Fmt &f, Fmt &o, std::vector<int16_t> &mp) {
    o = Fmt{f.p, f.n, f.m};
    mp.assign(o.lt(), -1);
    for (int j = 0; j < f.p; ++j)
        for (int k = 0; k < f.n; ++k) mp[o.iu(j, k)] = (int16_t)f.iv(k, j);
    for (int k = 0; k < f.n; ++k)
        for (int i = 0; i < f.m; ++i) mp[o.iv(k, i)] = (int16_t)f.iu(i, k);
    // w'[j'*m' + i'] with j' < p' = m, i' < m' = p: c'_{j'i'} ... = w[i' * m + j']
    for (int jp = 0; jp < o.p; ++jp)
        for (int ip = 0; ip < o.m; ++ip) mp[o.iw(jp, ip)] = (int16_t)f.iw(ip, jp);
}

// (u, v, w) -> (v, w, u): (m,n,p) -> (n,p,m), rows unchanged
void cyclic_map(const Fmt &f, Fmt &o, std::vector<int16_t> &mp) {
    o = Fmt{f.n, f.p, f.m};
    mp.assign(o.lt(), -1);
    for (int e = 0; e < f.lv(); ++e) mp[e] = (int16_t)(f.lu() + e);
    for (int e = 0; e < f.p * f.m; ++e) mp[f.lv() + e] = (int16_t)(f.lu() + f.lv() + e);
    for (int e = 0; e < f.lu(); ++e) mp[f.lv() + f.p * f.m + e] = (int16_t)e;
}

// out[e] = first[second[e]] (second maps the output to the intermediate term)
std::vector<int16_t> compose(const std::vector<int16_t> &first, const std::vector<int16_t> &second) {
    std::vector<int16_t> r(second.size(), -1);
    for (size_t e = 0; e < second.size(); ++e) r[e] = second[e] < 0 ? (int16_t)-1 : first[second[e]];
    return r;
}

const int kSwapTargets[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};

// the order of the sizes after transpose^t then cyclic^c
void order_after(int t, int c, int out[3]) {
    int o[3] = {0, 1, 2};
    if (t) { const int x = o[0]; o[0] = o[2]; o[2] = x; }
    for (int q = 0; q < c; ++q) { const int x = o[0]; o[0] = o[1]; o[1] = o[2]; o[2] = x; }
    for (int q = 0; q < 3; ++q) out[q] = o[q];
}

bool swap_map(const Fmt &f, int perm, Fmt &o, std::vector<int16_t> &mp) {
    for (int t = 0; t < 2; ++t)
        for (int c = 0; c < 3; ++c) {
            int ord[3];
            order_after(t, c, ord);
            if (ord[0] != kSwapTargets[perm][0] || ord[1] != kSwapTargets[perm][1] || ord[2] != kSwapTargets[perm][2])
                continue;
            Fmt cur = f;
            std::vector<int16_t> total(f.lt());
            for (int e = 0; e < f.lt(); ++e) total[e] = (int16_t)e;
            if (t) {
                Fmt nx;
                std::vector<int16_t> m1;
                transpose_map(cur, nx, m1);
                total = compose(total, m1);
                cur = nx;
            }
            for (int q = 0; q < c; ++q) {
                Fmt nx;
                std::vector<int16_t> m1;
                cyclic_map(cur, nx, m1);
                total = compose(total, m1);
                cur = nx;
            }
            o = cur;
            mp = total;
            return true;
        }
    return false;
}

}  // namespace

// Builds the plan of one resize operator on the host (maps and blocks; the
// caller uploads maps and aux terms).  Returns false for an unsupported
// operator or argument.
bool build_resize_plan(int op, int axis, int index, const tfg_format &src, const tfg_format *aux, int aux_rank,
                       tfg_format &out, ResizePlan &plan, std::vector<int16_t> &maps) {
    const Fmt f{src.m, src.n, src.p};
    Fmt o{0, 0, 0};
    maps.clear();
    plan = ResizePlan{};
    plan.lt_src = f.lt();
    plan.mn_src = f.lu();
    plan.np_src = f.lv();
    plan.canon = src.mode == TFG_MODE_ZT;
    std::vector<int16_t> a, b;
    auto add_block = [&](int kind, const std::vector<int16_t> *ma, const std::vector<int16_t> *mb) {
        ResizeBlock &bk = plan.blk[plan.nblk++];
        bk.kind = kind;
        bk.map_a = -1;
        bk.map_b = -1;
        if (ma) { bk.map_a = (int32_t)maps.size(); maps.insert(maps.end(), ma->begin(), ma->end()); }
        if (mb) { bk.map_b = (int32_t)maps.size(); maps.insert(maps.end(), mb->begin(), mb->end()); }
    };
    auto set_aux = [&](const Fmt &g) {
        plan.lt_aux = g.lt();
        plan.mn_aux = g.lu();
        plan.np_aux = g.lv();
    };
    const bool ax_ok = axis >= 0 && axis < 3;
    switch (op) {
    case TFG_RESIZE_PROJECT: {
        const int size = axis == 0 ? f.m : (axis == 1 ? f.n : f.p);
        if (!ax_ok || index < 0 || index >= size || size < 2) return false;
        project_map(f, axis, index, o, a);
        add_block(kResizeSrc, &a, nullptr);
        plan.drop_zero = 1;
        break;
    }
    case TFG_RESIZE_EXTEND: {
        if (!ax_ok) return false;
        const Fmt blk{axis == 0 ? 1 : f.m, axis == 1 ? 1 : f.n, axis == 2 ? 1 : f.p};
        merge_maps(f, blk, axis, o, a, b);
        add_block(kResizeSrc, &a, nullptr);
        add_block(kResizeAux, nullptr, &b);   // the naive scheme of the block, uploaded as aux
        set_aux(blk);
        plan.aux_rank = blk.m * blk.n * blk.p;
        break;
    }
    case TFG_RESIZE_DOUBLE: {
        if (!ax_ok) return false;
        merge_maps(f, f, axis, o, a, b);
        add_block(kResizeSrc, &a, nullptr);
        add_block(kResizeSrc, &b, nullptr);
        break;
    }
    case TFG_RESIZE_MERGE: {
        if (!ax_ok || !aux) return false;
        const Fmt g{aux->m, aux->n, aux->p};
        const bool agree = axis == 0 ? (g.n == f.n && g.p == f.p) : axis == 1 ? (g.m == f.m && g.p == f.p)
                                                                            : (g.m == f.m && g.n == f.n);
        if (!agree) return false;
        merge_maps(f, g, axis, o, a, b);
        add_block(kResizeSrc, &a, nullptr);
        add_block(kResizeAux, nullptr, &b);
        set_aux(g);
        plan.aux_rank = aux_rank;
        break;
    }
    case TFG_RESIZE_PRODUCT: {
        if (!aux) return false;
        const Fmt g{aux->m, aux->n, aux->p};
        product_maps(f, g, o, a, b);
        add_block(kResizeProduct, &a, &b);
        set_aux(g);
        plan.aux_rank = aux_rank;
        break;
    }
    case TFG_RESIZE_SWAP: {
        if (index < 0 || index >= 6 || !swap_map(f, index, o, a)) return false;
        add_block(kResizeSrc, &a, nullptr);
        break;
    }
    default:
        return false;
    }
    out = tfg_format{o.m, o.n, o.p, src.mode};
    plan.lt_out = o.lt();
    plan.mn_out = o.lu();
    plan.np_out = o.lv();
    return true;
}

// ---------------------------------------------------------------------------
// Device
namespace {

// One warp per walker, one lane per output term, many walkers per block.  A source
// coefficient goes to at most one output coefficient, so a term is built from its
// few non-zero coefficients: the block first inverts the maps into tables (source
// coefficient -> bit of the packed result; of a product the bit is the sum of a
// source and an aux entry) and packs the aux terms, then every term scatters its
// set bits into a row of packed words in shared memory, twice: once for the leading
// coefficients (sign normalisation, zero factors), once with the final signs.
// Bound by the writes of the result (live and best slots).  Evaluating every output
// coefficient of every term from the maps, by one block per walker, took 0.91 ms for
// 65536 walkers (3,3,3) -> (3,3,4); now 0.2 ms.
constexpr int kResizeWarps = 8;
constexpr int kResizeThreads = 32 * kResizeWarps;
constexpr int kMaxLT = 3 * 128;

// f(coefficient, negative) for the non-zero coefficients of bits [lo, lo + len) of packed 32-bit words
template <class F>
__device__ __forceinline__ void each_set(const uint32_t *pos, const uint32_t *neg, int lo, int len, F f) {
    for (int w = lo >> 5; (w << 5) < lo + len; ++w) {
        const uint32_t nw = neg ? neg[w] : 0u;
        uint32_t nz = pos[w] | nw;
        const int o0 = lo - (w << 5), o1 = lo + len - (w << 5);
        if (o0 > 0) nz &= ~((1u << o0) - 1u);
        if (o1 < 32) nz &= (1u << o1) - 1u;
        while (nz) {
            const int o = __ffs(nz) - 1;
            nz &= nz - 1u;
            f((w << 5) + o - lo, (bool)((nw >> o) & 1u));
        }
    }
}

// shared memory: tables [2][kMaxLT] int16, aux terms [aux_rank][2][aw] words, term rows [nw32][threads]
__global__ void __launch_bounds__(kResizeThreads) resize_kernel(const SegDesc src, int64_t src_first, const SegDesc dst,
                                                                int64_t dst_first, int64_t count, const ResizePlan pl,
                                                                unsigned long long *skipped) {
    extern __shared__ __align__(16) unsigned char rsm[];
    int16_t(*tab)[kMaxLT] = reinterpret_cast<int16_t(*)[kMaxLT]>(rsm);
    const int aw = (pl.lt_aux + 31) >> 5;
    const int aux_rank = min(pl.aux_rank, kResizeMaxTerms + 1);   // more: every walker is skipped
    const int aux_held = aux_rank > kResizeMaxTerms ? 0 : aux_rank;
    uint32_t *aux = reinterpret_cast<uint32_t *>(rsm + 2 * kMaxLT * sizeof(int16_t));
    uint32_t *rows = aux + (size_t)aux_held * 2 * aw;
    const int tid = threadIdx.x, lane = tid & 31;
    const int nw32 = dst.nws * dst.word_bits / 32, sign32 = dst.tw * dst.word_bits / 32;   // words per slot / per sign
    const bool zt = src.tw * 2 == src.nws;   // Z_T: negative words present
    const bool product = pl.blk[0].kind == kResizeProduct;
    const int src_start[3] = {0, pl.mn_src, pl.mn_src + pl.np_src};
    const int src_len[3] = {pl.mn_src, pl.np_src, pl.lt_src - pl.mn_src - pl.np_src};
    const int aux_start[3] = {0, pl.mn_aux, pl.mn_aux + pl.np_aux};
    const int aux_len[3] = {pl.mn_aux, pl.np_aux, pl.lt_aux - pl.mn_aux - pl.np_aux};
    // ---- tables: tab[block][coefficient of its terms] -> bit of the packed result (-1: gone)
    for (int e = tid; e < 2 * kMaxLT; e += kResizeThreads) tab[0][e] = -1;
    __syncthreads();
    for (int e = tid; e < pl.lt_out; e += kResizeThreads) {
        const int f = e < pl.mn_out ? 0 : (e < pl.mn_out + pl.np_out ? 1 : 2);
        const int bit = dst.fbase[f] + e - (f == 0 ? 0 : (f == 1 ? pl.mn_out : pl.mn_out + pl.np_out));
        if (product) {
            const int qa = pl.maps[pl.blk[0].map_a + e], qb = pl.maps[pl.blk[0].map_b + e];
            if (qb == aux_start[f]) tab[0][qa] = (int16_t)bit;
            if (qa == src_start[f]) tab[1][qb] = (int16_t)(bit - dst.fbase[f]);
        } else {
            for (int b = 0; b < pl.nblk; ++b) {
                const int q = pl.maps[(pl.blk[b].kind == kResizeAux ? pl.blk[b].map_b : pl.blk[b].map_a) + e];
                if (q >= 0) tab[b][q] = (int16_t)bit;
            }
        }
    }
    for (int e = tid; e < aux_held * aw; e += kResizeThreads) {
        const int l = e / aw, w = e - l * aw;
        uint32_t ps = 0u, ng = 0u;
        for (int q = 32 * w; q < min(pl.lt_aux, 32 * w + 32); ++q) {
            const int v = pl.aux[(int64_t)l * pl.lt_aux + q];
            ps |= (v > 0 ? 1u : 0u) << (q & 31);
            ng |= (v < 0 ? 1u : 0u) << (q & 31);
        }
        aux[(2 * l) * aw + w] = ps;
        aux[(2 * l + 1) * aw + w] = ng;
    }
    __syncthreads();
    uint32_t *row = rows + tid;   // word q of this lane's term at row[q * kResizeThreads]
    const int ssign32 = src.tw * src.word_bits / 32, snw32 = src.nws * src.word_bits / 32;
    for (int64_t k = (int64_t)blockIdx.x * kResizeWarps + (tid >> 5); k < count; k += (int64_t)gridDim.x * kResizeWarps) {
        const int64_t ws = src_first + k, wd = dst_first + k;
        const tfg_walker_info &hs = src.hdr[ws];
        const int r_src = pl.use_best ? hs.best_r : hs.r;
        const uint32_t *sw = reinterpret_cast<const uint32_t *>(pl.use_best ? src.best : src.slots) + (size_t)ws * src.R * snw32;
        const int n0 = pl.blk[0].kind == kResizeAux ? aux_rank : (product ? r_src * aux_rank : r_src);
        const int n1 = pl.nblk < 2 ? 0 : (pl.blk[1].kind == kResizeAux ? aux_rank : r_src);
        const int r_raw = n0 + n1;
        // f(factor, bit of the result, negative) for the non-zero coefficients of output term o
        auto scatter = [&](int o, auto f) {
            const int b = o >= n0 ? 1 : 0, loc = o - (b ? n0 : 0);
            if (product) {
                const int t = loc / aux_rank, l = loc - t * aux_rank;
                const uint32_t *sp = sw + (size_t)t * snw32, *ap = aux + (size_t)(2 * l) * aw;
                for (int x = 0; x < 3; ++x)
                    each_set(sp, zt ? sp + ssign32 : nullptr, src.fbase[x], src_len[x], [&](int e, bool ne) {
                        const int base = tab[0][src_start[x] + e];
                        each_set(ap, ap + aw, aux_start[x], aux_len[x],
                                 [&](int g, bool ng) { f(x, base + tab[1][aux_start[x] + g], ne != ng); });
                    });
            } else if (pl.blk[b].kind == kResizeAux) {
                const uint32_t *ap = aux + (size_t)(2 * loc) * aw;
                // an aux coefficient's factor in the result is its own
                for (int x = 0; x < 3; ++x)
                    each_set(ap, ap + aw, aux_start[x], aux_len[x], [&](int e, bool ne) { f(x, tab[b][aux_start[x] + e], ne); });
            } else {
                const uint32_t *sp = sw + (size_t)loc * snw32;
                // a size swap permutes the factors: the result's factor is where the bit lands
                for (int x = 0; x < 3; ++x)
                    each_set(sp, zt ? sp + ssign32 : nullptr, src.fbase[x], src_len[x], [&](int e, bool ne) {
                        const int bit = tab[b][src_start[x] + e];
                        if (bit >= 0) f(bit < dst.fbase[1] ? 0 : (bit < dst.fbase[2] ? 1 : 2), bit, ne);
                    });
            }
        };
        // leading coefficients of term o: bit 0 / 1 of the result: u / v starts with -1; bits 2, 3, 4: u, v, w not zero
        auto look = [&](int o) -> unsigned {
            int lu = INT_MAX, lv = INT_MAX;
            unsigned z = 0u;
            scatter(o, [&](int x, int bit, bool ne) {
                const int key = 2 * bit + (int)ne;
                if (x == 0) lu = min(lu, key);
                if (x == 1) lv = min(lv, key);
                z |= 4u << x;
            });
            return z | (pl.canon ? (unsigned)((lu != INT_MAX && (lu & 1)) | ((lv != INT_MAX && (lv & 1)) << 1)) : 0u);
        };
        // terms with a zero factor go; project may bring a larger scheme below the capacity that way
        bool skip = r_src < 1 || r_src > src.R || r_raw > kResizeMaxTerms || (!pl.drop_zero && r_raw > dst.R);
        if (!skip && r_raw > dst.R) {
            int stay = 0;
            for (int o0 = 0; o0 < r_raw; o0 += 32)
                stay += __popc(__ballot_sync(0xffffffffu, o0 + lane < r_raw && (look(o0 + lane) >> 2) == 7u));
            skip = stay > dst.R;
        }
        if (skip) {
            if (lane == 0) atomicAdd(skipped, 1ull);
            continue;
        }
        uint32_t *live = reinterpret_cast<uint32_t *>(dst.slots) + (size_t)wd * dst.R * nw32;
        uint32_t *best = reinterpret_cast<uint32_t *>(dst.best) + (size_t)wd * dst.R * nw32;
        int nnz = 0, at = 0;
        for (int o0 = 0; o0 < r_raw; o0 += 32) {
            const int o = o0 + lane;
            const unsigned lk = o < r_raw ? look(o) : 0u;
            const bool keep = (lk >> 2) == 7u;
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int slot = at + __popc(kept & ((1u << lane) - 1u));
                // Section 3.6: first non-zero of u, then of v, made +1; w absorbs the signs
                const bool su = lk & 1u, sv = (lk >> 1) & 1u;
                for (int q = 0; q < nw32; ++q) row[q * kResizeThreads] = 0u;
                scatter(o, [&](int x, int bit, bool ne) {
                    const bool neg = ne != (x == 0 ? su : (x == 1 ? sv : su != sv));
                    row[((bit >> 5) + (neg ? sign32 : 0)) * kResizeThreads] |= 1u << (bit & 31);
                    nnz += 1;
                });
                if (nw32 == 4) {
                    const uint4 v = make_uint4(row[0], row[kResizeThreads], row[2 * kResizeThreads], row[3 * kResizeThreads]);
                    reinterpret_cast<uint4 *>(live)[slot] = v;
                    reinterpret_cast<uint4 *>(best)[slot] = v;
                } else if (nw32 == 2) {
                    const uint2 v = make_uint2(row[0], row[kResizeThreads]);
                    reinterpret_cast<uint2 *>(live)[slot] = v;
                    reinterpret_cast<uint2 *>(best)[slot] = v;
                } else {
                    for (int q = 0; q < nw32; ++q) {
                        const uint32_t v = row[q * kResizeThreads];
                        live[slot * nw32 + q] = v;
                        best[slot * nw32 + q] = v;
                    }
                }
            }
            at += __popc(kept);
        }
        const int r_new = at;
        if (r_new == 0) {   // nothing written: left as it was
            if (lane == 0) atomicAdd(skipped, 1ull);
            continue;
        }
        // unused slots cleared
        for (int q = r_new * nw32 + lane; q < dst.R * nw32; q += 32) {
            live[q] = 0u;
            best[q] = 0u;
        }
        nnz = __reduce_add_sync(0xffffffffu, nnz);
        if (lane == 0) {
            tfg_walker_info &h = dst.hdr[wd];
            h.r = r_new;
            h.best_r = r_new;
            h.plateau = 0;
            h.best_t = h.t;
            h.best_nnz = (uint32_t)nnz;
        }
    }
}

}  // namespace

void launch_resize(const SegDesc &src, int64_t src_first, const SegDesc &dst, int64_t dst_first, int64_t count,
                   const ResizePlan &plan, unsigned long long *d_skipped, cudaStream_t st) {
    if (count <= 0) return;
    const size_t smem = (size_t)2 * kMaxLT * sizeof(int16_t) + (plan.aux_rank > kResizeMaxTerms ? (size_t)0 : (size_t)plan.aux_rank * 2 * ((plan.lt_aux + 31) / 32) * 4) +
                        (size_t)dst.nws * dst.word_bits / 32 * 4 * kResizeThreads;
    // the most of any launch: another thread may be about to launch the kernel with more
    constexpr int most_smem = 2 * kMaxLT * (int)sizeof(int16_t) + kResizeMaxTerms * 2 * (kMaxLT / 32) * 4 +
                              2 * (kMaxLT / 32) * 4 * kResizeThreads;
    cudaFuncSetAttribute(resize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most_smem);
    int dev = 0, sms = 1, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, resize_kernel, kResizeThreads, smem);
    const int64_t blocks = (count + kResizeWarps - 1) / kResizeWarps, most = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    resize_kernel<<<(unsigned)(blocks < most ? blocks : most), kResizeThreads, smem, st>>>(src, src_first, dst, dst_first,
                                                                                       count, plan, d_skipped);
}

}  // namespace tfg
