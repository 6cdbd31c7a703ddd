// Wide-term flip-graph walk kernel for sm_103a: formats whose terms have more
// than 64 coefficients (m*n + n*p + p*m > 64), with factors of up to 128.
//
// Layout.  A term is factor-aligned: factor f (u, v, w) is words f*FW ..
// f*FW+FW-1 of the positive-coefficient words and the same words of the
// negative ones (Section 3.5.1's digits/signs masks, FW = 1 or 2 words of 64
// bits per factor and sign), so every operation of Section 3.5.2 works word
// by word and needs no mask.
//
// Mapping.  Eight lanes per walker, four walkers a warp, with the factor classes of walk_link.cuh kept in shared memory: per factor the
// slots of equal factors (w up to sign) form a cyclic list in ascending order, and
// the slots' 8-bit factor hashes are held bit-sliced.  A step reads the sampled
// term's three lists (a lane each); an accepted flip moves two slots to other
// classes: the lanes share the hash words of the new factor's scan, check the
// hits on the full words, and one lane per moved slot relinks it.  The arithmetic
// of a flip, a merge or a plus transition works on one word per lane (lane q < 3*FW
// holds word q, of factor q / FW, of each term involved): additions and
// normalisation are a handful of lane-parallel instructions and ballots.  All
// walker-uniform bookkeeping is replicated in the walker's lanes.  The four walkers
// of a warp stay converged: what only some of them do is entered when any does
// and predicated on their lanes (`on`), since shuffles and ballots on the lanes of one
// walker alone split the warp into four that run one after another (32 us
// a step of 32768 walkers at 351 terms, converged 27, and 18 with the scan, the
// snapshots and the build as they are now).
//
// Bound by the latency of a step, the reads of terms from L2 and memory first; 3.3 KB
// of shared memory per walker at 354 slots let 64 walkers reside on an SM (8 blocks, 16 warps).
// The kernel it replaces searched all slots' 32-bit signatures with a warp per walker in
// every step (1186 instructions a walker-step at 351 terms, now 280).  Measured, Z_T, 32768
// walkers, 400 steps (classes built at each launch), before / now: (4,5,12) 10.7 / 5.4 ms,
// (5,6,10) 10.7 / 6.3, (6,7,9) 12.7 / 8.2, (4,5,5) 7.8 / 3.7; (9,8,2) 16384 walkers 5.9 / 3.1.
//
// The step contract (draws, candidate order, flip, rejection, removal,
// normalisation, reduction cascade, best/plateau bookkeeping, plus
// transitions, trajectory digest) is the one of the lane-group and
// thread-per-walker kernels.
#include <cstdint>
#include <type_traits>

#include "tfg_internal.h"
#include "pterm.cuh"
#include "walk_link.cuh"
#include "walk_wide_search.cuh"

namespace tfg {
namespace dev {

// PG: the walk policy is read from the descriptor (policies 1 and 2); without
// it the plateau policy is compiled in alone.
// FW: 64-bit words per factor (1: factors of at most 64 coefficients, 2: at most 128).
// GM: the terms stay in the walker's device-memory slots, else they are staged in shared
// memory for the launch.
template <int MODE, bool PG, int FW, bool GM>
struct WideWalker {
    static constexpr int G = 8;   // lanes per walker
    static_assert(FW == 1 || FW == 2, "one or two words per factor");
    static_assert(G >= 3 * FW && G >= 5 && G < 32, "a lane per word of a term and per list of the reduction test");
    static constexpr bool ZT = (MODE == TFG_MODE_ZT);
    __device__ __forceinline__ static int policy_of(const SegDesc &d) { return PG ? d.walk_policy : 0; }
    static constexpr int TW = 3 * FW;                          // words per sign
    static constexpr int NWG = ZT ? 2 * TW : TW;               // words per slot (p words [n words])
    static constexpr unsigned FM = (1u << FW) - 1u;            // a factor's lanes / words in a ballot
    static_assert(G >= kHashBits, "a lane per hash slice");
    static constexpr int NL = 32 / G;                          // hash words per lane at 1023 slots
    static constexpr int kNone = 1 << 20;

    uint64_t *W;      // this walker's slots [R][NWG], in device (GM) or shared memory
    uint16_t *nx;     // next of (k, f) = nx[f * R + k]
    uint32_t *hs;     // hash slices: bit b of factor f, slots 32 q .. 32 q + 31 = hs[(f * 8 + b) * KW + q]
    int lane, gb;     // lane within the walker's G lanes; the first of them
    int KW;           // hash words: ceil(R / 32)
    int r, best_r, R;
    int64_t t, plateau, best_t;
    uint64_t dig;
    uint32_t wid, key0, key1;
    uint32_t c_acc, c_rej, c_noc, c_drp, c_mrg, c_pls, c_red;
    int qlen, q0, q1, q2;
    uint32_t nnz, best_nnz;   // non-zero coefficients of the live (walk policy 2) / best scheme

    __host__ __device__ static constexpr size_t walker_bytes(int R) {
        return term_bytes(R) + (((size_t)R * 6 + 15) & ~(size_t)15) + (size_t)3 * kHashBits * ((R + 31) / 32) * 4;
    }
    __host__ __device__ static constexpr size_t term_bytes(int R) {   // in shared memory
        return GM ? (size_t)0 : ((size_t)R * NWG * 8 + 15) & ~(size_t)15;
    }
    // slots: the walker's device-memory slots
    __device__ __forceinline__ void attach(unsigned char *at, uint64_t *slots) {
        W = GM ? slots : reinterpret_cast<uint64_t *>(at);
        at += term_bytes(R);
        nx = reinterpret_cast<uint16_t *>(at);
        hs = reinterpret_cast<uint32_t *>(at + (((size_t)R * 6 + 15) & ~(size_t)15));
    }

    // ---- group communication
    __device__ __forceinline__ unsigned vote(bool p) const {
        return (__ballot_sync(kFull, p) >> gb) & ((1u << G) - 1u);
    }
    template <class V>
    __device__ __forceinline__ V from(V v, int l) const { return __shfl_sync(kFull, v, gb + l); }
    __device__ __forceinline__ static bool any(bool p) { return __any_sync(kFull, p); }

    __device__ __forceinline__ static uint32_t sum(uint32_t v) {   // over the walker's lanes
#pragma unroll
        for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
        return v;
    }

    // ---- one word per lane: lane q < 3*FW holds word q (factor q / FW) of each
    // term involved; the other lanes mirror word 0 and never store
    struct DF { uint64_t p, n; };
    int fq;   // this lane's word (0 on lanes past the words)
    __device__ __forceinline__ bool owns(int f) const { return (lane >> (FW - 1)) == f; }   // holds a word of factor f
    __device__ __forceinline__ bool fown() const { return lane < 3 * FW; }

    bool live;   // these lanes have a walker; without one they hold zero terms and read no one's slots or classes
    __device__ __forceinline__ DF dget(int s) const {
        if (!live) return DF{0ull, 0ull};
        return DF{W[(size_t)s * NWG + fq], ZT ? W[(size_t)s * NWG + TW + fq] : 0ull};
    }
    // res = a with factor f := a_f + b_f (neg: a_f - b_f); false when a
    // coefficient leaves the coefficient set (Section 3.5.2)
    __device__ __forceinline__ bool dadd(const DF &a, const DF &b, int f, bool neg, DF &res) const {
        const bool me = owns(f);
        bool bad = false;
        if constexpr (ZT) {
            const uint64_t bp = neg ? b.n : b.p, bn = neg ? b.p : b.n;
            res.p = me ? ((a.p | bp) & ~(a.n | bn)) : a.p;
            res.n = me ? ((a.n | bn) & ~(a.p | bp)) : a.n;
            bad = me && ((a.p & bp) | (a.n & bn)) != 0ull;
        } else {
            res.p = me ? (a.p ^ b.p) : a.p;
            res.n = 0ull;
        }
        return vote(bad) == 0u;
    }
    __device__ __forceinline__ bool dzero(const DF &a, int f) const {
        return ((vote((a.p | a.n) == 0ull) >> (f * FW)) & FM) == FM;
    }
    __device__ __forceinline__ void dtake(DF &dst, const DF &src, int f) const {
        if (owns(f)) dst = src;
    }
    // Sign flags of the leading coefficient of every factor: bit f*FW (of the
    // returned ballot) is set when factor f's first non-zero coefficient is negative.
    __device__ __forceinline__ unsigned dlead(const DF &a) const {
        const uint64_t d = a.p | a.n;
        const unsigned ng = vote((a.n & d & (0ull - d)) != 0ull);
        if constexpr (FW == 1) {
            return ng;
        } else {
            // a factor's second word decides only when its first word is zero
            const unsigned nz = vote(d != 0ull);
            return (ng & nz & 0x15u) | ((ng >> 1) & ~nz & 0x15u);
        }
    }
    // Section 3.6: first non-zero of u, then of v, made +1; w absorbs the signs
    __device__ __forceinline__ void dcanon(DF &a) const {
        if constexpr (ZT) {
            const unsigned neg = dlead(a);
            const bool f0 = neg & 1u, f1 = (neg >> FW) & 1u;
            const bool sw = (owns(0) && f0) || (owns(1) && f1) || (owns(2) && f0 != f1);
            const uint64_t p = sw ? a.n : a.p, n = sw ? a.p : a.n;
            a.p = p; a.n = n;
        }
    }
    // non-zero coefficients of a term held one word per lane
    __device__ __forceinline__ uint32_t dnnz(const DF &a) const {
        const uint32_t c = fown() ? (uint32_t)__popcll(a.p | a.n) : 0u;
        return sum(c);
    }
    // w of a equals -w of b
    __device__ __forceinline__ bool dwneg(const DF &a, const DF &b) const {
        return ZT && ((vote(a.p == b.n && a.n == b.p) >> (2 * FW)) & FM) == FM;
    }
    __device__ __forceinline__ void dput(bool on, int s, const DF &a) {
        if (on && fown()) {
            W[(size_t)s * NWG + lane] = a.p;
            if constexpr (ZT) W[(size_t)s * NWG + TW + lane] = a.n;
        }
        __syncwarp();
    }

    // ---- factor classes
    __device__ __forceinline__ uint16_t &next(int k, int f) const { return nx[f * R + k]; }
    // symmetric in the two signs: w's class is up to sign
    __device__ __forceinline__ static uint32_t fold(uint64_t x) {
        const uint64_t a = (uint64_t)(uint32_t)x * 0x9E3779B1u + (uint64_t)(uint32_t)(x >> 32) * 0x85EBCA77u;
        return (uint32_t)a ^ (uint32_t)(a >> 32);
    }
    __device__ __forceinline__ static uint32_t word_hash(uint64_t p, uint64_t n, int h) {
        const uint32_t x = fold(p) + (ZT ? fold(n) : 0u);
        return h ? x * 0xC2B2AE35u : x;
    }
    // hash of factor f of a term held one word per lane
    __device__ __forceinline__ uint32_t dhash(const DF &a, int f) const {
        const uint32_t x = word_hash(a.p, a.n, FW == 1 ? 0 : lane & 1);
        uint32_t h = from(x, f * FW);
        if constexpr (FW == 2) h += from(x, f * FW + 1);
        return h;
    }
    // live slots of hash word q
    __device__ __forceinline__ static uint32_t live_word(int r, int q) {
        const int lo = r - 32 * q;
        return lo >= 32 ? ~0u : (lo > 0 ? (1u << lo) - 1u : 0u);
    }
    __device__ __forceinline__ static void spreads(uint32_t h, uint32_t (&sp)[kHashBits]) {
        sp[0] = sign_spread<0>(h); sp[1] = sign_spread<1>(h); sp[2] = sign_spread<2>(h); sp[3] = sign_spread<3>(h);
        const uint32_t h1 = h << 1;
        sp[4] = sign_spread<0>(h1); sp[5] = sign_spread<1>(h1); sp[6] = sign_spread<2>(h1); sp[7] = sign_spread<3>(h1);
    }
    // This lane's share (words lane, lane + G, ...) of the slots that may hold the factor f
    // of hash h, slot s aside; s's own slices := the hash.
    __device__ __forceinline__ void scan(bool on, int s, int f, uint32_t h, uint32_t (&c)[NL]) const {
        uint32_t sp[kHashBits];
        spreads(h, sp);
        const uint32_t sb = 1u << (s & 31);
        uint32_t *base = hs + f * kHashBits * KW;
#pragma unroll
        for (int a = 0; a < NL; ++a) c[a] = 0u;
#pragma unroll
        for (int a = 0; a < NL; ++a) {
            if (a * G >= KW) break;   // the same for all lanes
            const int q = a * G + lane;
            if (on && q < KW) {
                uint32_t dd = 0u;
#pragma unroll
                for (int b = 0; b < kHashBits; ++b) dd |= base[b * KW + q] ^ sp[b];
                c[a] = ~dd & live_word(r, q) & (q == (s >> 5) ? ~sb : ~0u);
            }
        }
        __syncwarp();
        // a lane per slice
        if (on && lane < kHashBits) {
            uint32_t mine = sp[0];
#pragma unroll
            for (int b = 1; b < kHashBits; ++b) mine = lane == b ? sp[b] : mine;
            uint32_t &w = base[lane * KW + (s >> 5)];
            w = (w & ~sb) | (mine & sb);
        }
    }
    // this lane's lowest slot of c, removed from it (-1: none)
    __device__ __forceinline__ int take(uint32_t (&c)[NL]) const {
        int k = -1;
#pragma unroll
        for (int a = 0; a < NL; ++a) {
            const bool here = k < 0 && c[a] != 0u;
            k = here ? 32 * (a * G + lane) + __ffs(c[a]) - 1 : k;
            c[a] = here ? c[a] & (c[a] - 1u) : c[a];
        }
        return k;
    }
    // factor f of slot s of the slots w equals (vp, vn) up to sign
    __device__ __forceinline__ static bool fsame(const uint64_t *w, int s, int f, const uint64_t (&vp)[FW],
                                                 const uint64_t (&vn)[FW]) {
        bool ep = true, en = ZT;
#pragma unroll
        for (int h = 0; h < FW; ++h) {
            const uint64_t p = w[(size_t)s * NWG + f * FW + h], n = ZT ? w[(size_t)s * NWG + TW + f * FW + h] : 0ull;
            ep = ep && p == vp[h] && n == vn[h];
            en = en && p == vn[h] && n == vp[h];
        }
        return ep || en;
    }
    // slot s out of its class of factor f, then into the class of slot `hit` (-1: a class of
    // its own); by one lane
    __device__ __forceinline__ void move_class(int s, int f, int hit) const {
        const int o = next(s, f);
        int p = s, q = o;
#pragma unroll 1
        for (int n = 0; n < R && q != s; ++n) {   // a class has at most R members
            p = q;
            q = next(q, f);
        }
        next(p, f) = (uint16_t)o;
        p = hit >= 0 ? hit : s;
        q = hit >= 0 ? (int)next(hit, f) : s;
#pragma unroll 1
        for (int n = 0; n < R && !(p < q ? (p < s && s < q) : (s >= p || s <= q)); ++n) {
            p = q;
            q = next(q, f);
        }
        next(p, f) = (uint16_t)s;
        next(s, f) = (uint16_t)q;
    }
    // One or (TWO) two slots change their class: slot sa's factor fa is now va's, slot sb's
    // factor fb (fb != fa) now vb's (both stored already).
    template <bool TWO>
    __device__ __forceinline__ void relink(bool on, int sa, int fa, const DF &va, int sb, int fb, const DF &vb) const {
        uint32_t ca[NL], cb[NL];
        scan(on, sa, fa, dhash(va, fa), ca);
        if constexpr (TWO) {
            scan(on, sb, fb, dhash(vb, fb), cb);
        } else {
#pragma unroll
            for (int a = 0; a < NL; ++a) cb[a] = 0u;
        }
        uint64_t ap[FW], an[FW], bp[FW], bn[FW];
#pragma unroll
        for (int h = 0; h < FW; ++h) {
            ap[h] = from(va.p, fa * FW + h);
            an[h] = ZT ? from(va.n, fa * FW + h) : 0ull;
            bp[h] = TWO ? from(vb.p, fb * FW + h) : 0ull;
            bn[h] = TWO && ZT ? from(vb.n, fb * FW + h) : 0ull;
        }
        int ha = -1, hb = -1;   // a slot of the new class
#pragma unroll 1
        for (int n = 0; n <= R; ++n) {
            const int ka = ha < 0 ? take(ca) : -1, kb = TWO && hb < 0 ? take(cb) : -1;
            if (!any(ka >= 0 || kb >= 0)) break;
            const bool oa = ka >= 0 && fsame(W, ka, fa, ap, an);
            const bool ob = TWO && kb >= 0 && fsame(W, kb, fb, bp, bn);
            const unsigned ma = vote(oa);
            const int fa2 = from(ka, ma ? __ffs(ma) - 1 : 0);
            ha = ma ? fa2 : ha;
            if constexpr (TWO) {
                const unsigned mb = vote(ob);
                const int fb2 = from(kb, mb ? __ffs(mb) - 1 : 0);
                hb = mb ? fb2 : hb;
            }
        }
        if constexpr (TWO) {
            if (on && lane < 2) move_class(lane ? sb : sa, lane ? fb : fa, lane ? hb : ha);
        } else {
            if (on && lane == 0) move_class(sa, fa, ha);
        }
        __syncwarp();
    }
    // slot s := term v, every class anew
    __device__ __forceinline__ void put(bool on, int s, const DF &v) {
        dput(on, s, v);
#pragma unroll 1
        for (int f = 0; f < 3; ++f) relink<false>(on, s, f, v, s, f, v);
    }
    __device__ __forceinline__ void unlink(bool on, int s) const {
        if (on && lane < 3) move_class(s, lane, -1);
        __syncwarp();
    }

    // ---- reduction queue (slot indices), walker-uniform
    __device__ __forceinline__ void q_push(int s) {
        q0 = (qlen == 0) ? s : q0;
        q1 = (qlen == 1) ? s : q1;
        q2 = (qlen == 2) ? s : q2;
        qlen += 1;
    }
    __device__ __forceinline__ int q_pop() {
        const int s = q0;
        q0 = q1; q1 = q2;
        qlen -= 1;
        return s;
    }
    __device__ __forceinline__ void q_remove(int s) {
        const bool k0 = qlen > 0 && q0 != s, k1 = qlen > 1 && q1 != s, k2 = qlen > 2 && q2 != s;
        const int n0 = k0 ? q0 : (k1 ? q1 : q2);
        const int n1 = k0 ? (k1 ? q1 : q2) : q2;
        q0 = n0; q1 = n1;
        qlen = (int)k0 + (int)k1 + (int)k2;
    }
    __device__ __forceinline__ void q_rename(int from_, int to) {
        q0 = (qlen > 0 && q0 == from_) ? to : q0;
        q1 = (qlen > 1 && q1 == from_) ? to : q1;
        q2 = (qlen > 2 && q2 == from_) ? to : q2;
    }

    // Remove slot h: the last live term moves into the hole.
    __device__ __forceinline__ void drop(bool on, int h) {
        const int last = r - 1;
        const bool mv = on && h != last;
        if (on) q_remove(h);
        unlink(on, h);
        unlink(mv, last);
        if (on) r -= 1;
        if (any(mv)) {
            put(mv, mv ? h : 0, dget(mv ? last : 0));
            if (mv) q_rename(last, h);
        }
    }

    // Slot k against the term v (held one word per lane): which factors are equal, negated,
    // and where the sum / difference leaves the coefficient set (bit f).
    struct Against { unsigned eq, ne, cp, cn; };
    __device__ __forceinline__ static unsigned by_factor_all(unsigned b) {
        if constexpr (FW == 1) return b & 7u;
        else return ((b & (b >> 1)) & 1u) | (((b & (b >> 1)) >> 1) & 2u) | (((b & (b >> 1)) >> 2) & 4u);
    }
    __device__ __forceinline__ static unsigned by_factor_any(unsigned b) {
        if constexpr (FW == 1) return b & 7u;
        else return ((b | (b >> 1)) & 1u) | (((b | (b >> 1)) >> 1) & 2u) | (((b | (b >> 1)) >> 2) & 4u);
    }
    __device__ __forceinline__ Against against(int k, const DF &v) const {
        const DF c = dget(k);
        Against a;
        a.eq = by_factor_all(vote(c.p == v.p && c.n == v.n));
        a.ne = ZT ? by_factor_all(vote(c.p == v.n && c.n == v.p)) : 0u;
        a.cp = ZT ? by_factor_any(vote(((v.p & c.p) | (v.n & c.n)) != 0ull)) : 0u;
        a.cn = ZT ? by_factor_any(vote(((v.p & c.n) | (v.n & c.p)) != 0ull)) : 0u;
        return a;
    }

    // Reduction of the term in slot s with the lowest slot sharing (u,v), else
    // (u,w), else (v,w), whose merged third factor stays in the coefficient set; the
    // merged term keeps s's pair factors and goes to the lower slot.
    __device__ __forceinline__ void reduce_one(bool on, int s) {   // s valid in every lane
        const DF dv = dget(s);
        int k0 = kNone, k1 = kNone, k2 = kNone;
        bool n1 = false, n2 = false;
        int k = on ? (int)next(s, 0) : s;
        bool act = on && k != s;
#pragma unroll 1
        for (int n = 0; n < R && any(act); ++n) {
            const Against a = against(k, dv);
            const bool ev = a.eq & 2u, ewp = a.eq & 4u, ewn = !ewp && (a.ne & 4u);
            if (act && ev && k < k0 && !(a.cp & 4u)) k0 = k;
            if (act && (ewp || ewn) && k < k1 && !((ewn ? a.cn : a.cp) & 2u)) { k1 = k; n1 = ewn; }
            k = act ? (int)next(k, 0) : k;
            act = act && k != s;
        }
        k = on ? (int)next(s, 1) : s;
        act = on && k0 == kNone && k1 == kNone && k != s;
#pragma unroll 1
        for (int n = 0; n < R && any(act); ++n) {
            const Against a = against(k, dv);
            const bool ewp = a.eq & 4u, ewn = !ewp && (a.ne & 4u);
            if (act && (ewp || ewn) && k < k2 && !((ewn ? a.cn : a.cp) & 1u)) { k2 = k; n2 = ewn; }
            k = act ? (int)next(k, 1) : k;
            act = act && k != s;
        }
        const bool has = k0 != kNone || k1 != kNone || k2 != kNone;
        if (!any(has)) return;
        const int P = k0 != kNone ? 0 : (k1 != kNone ? 1 : 2);
        k = !has ? s : (P == 0 ? k0 : (P == 1 ? k1 : k2));
        const bool kneg = P == 1 ? n1 : (P == 2 ? n2 : false);
        const int F = 2 - P;   // third factor: w, v, u
        DF mv;
        dadd(dv, dget(k), F, kneg, mv);
        const bool z = dzero(mv, F);
        dcanon(mv);
        const int lo = s < k ? s : k;
        const int hi = s < k ? k : s;
        if (has) q_remove(k);
        dput(has, lo, mv);
        relink<false>(has, lo, F, mv, lo, F, mv);   // s and k share the other two factors
        c_mrg += has;
        drop(has, hi);
        if (any(has && z)) drop(has && z, lo);
        c_drp += has && z;
        if (has && !z) q_push(lo);
    }

    __device__ __forceinline__ void cascade() {
#pragma unroll 1
        while (any(qlen > 0)) {
            const bool on = qlen > 0;
            int s = 0;
            if (on) s = q_pop();
            reduce_one(on, s);
        }
    }

    // Live slots to the best slots of the walkers that want it, one after another by the
    // whole warp (8 lanes alone wait for memory 66 times at 351 terms).
    __device__ __forceinline__ void snapshots(bool want, uint64_t *bestp) const {
        unsigned pend = __ballot_sync(kFull, want && lane == 0);
        using V = typename std::conditional<NWG % 2 == 0, ulonglong2, unsigned long long>::type;
        constexpr int PV = NWG * 8 / (int)sizeof(V);   // vectors per slot
#pragma unroll 1
        while (pend) {
            const int a = __ffs(pend) - 1;
            pend &= pend - 1u;
            const int ra = __shfl_sync(kFull, r, a);
            const V *src = reinterpret_cast<const V *>(__shfl_sync(kFull, reinterpret_cast<unsigned long long>(W), a));
            V *dst = reinterpret_cast<V *>(__shfl_sync(kFull, reinterpret_cast<unsigned long long>(bestp), a));
#pragma unroll 8
            for (int e = threadIdx.x & 31; e < ra * PV; e += 32) dst[e] = src[e];
        }
    }

    // Expansion (Section 3.3.1): plus (three new terms), or split under walk policy 1
    // when y3 >= 2^31; the changed terms are queued for the cascade;
    // returns the digest record (0 when no attempt passed).
    __device__ __forceinline__ uint64_t plus_setup(const SegDesc &d, bool on) {
        uint64_t rec = 0;
        bool pend = on;
#pragma unroll 1
        for (int a = 1; a <= d.plus_attempts && any(pend); ++a) {
            const U4 y = philox10((uint32_t)t, (uint32_t)(t >> 32), wid, (uint32_t)a, key0, key1);
            const int pi = pend ? (int)__umulhi(y.x, (uint32_t)r) : 0;
            const int pj = pend ? (pi + 1 + (int)__umulhi(y.y, (uint32_t)(r - 1))) % r : 0;
            const int perm = (int)__umulhi(y.z, 6u);
            int A, B, C;
            plus_roles(perm, A, B, C);
            const DF ti = dget(pi), tj = dget(pj);
            const bool split = policy_of(d) == 1 && y.w >= 0x80000000u;
            DF nw, ti2, tj2;   // the new term, terms i and j afterwards
            bool ok = dadd(ti, tj, B, false, ti2);   // (A_i, B_i + B_j, C_i)
            ok &= dadd(tj, ti, C, true, tj2);        // (A_i, B_j, C_j - C_i)
            ok &= dadd(tj, ti, A, true, nw);         // (A_j - A_i, B_j, C_j)
            const bool zb = dzero(ti2, B), zc = dzero(tj2, C), za = dzero(nw, A);
            ok = ok && !(zb || zc || za);
            dtake(tj2, ti, A);
            if constexpr (PG) {
                // split: term i = (A_j, B_i, C_i), new term (A_i - A_j, B_i, C_i), term j unchanged
                DF sw;
                const bool sok = dadd(ti, tj, A, true, sw);
                const bool sz = dzero(sw, A);
                if (split) {
                    ok = sok && !sz;
                    nw = sw;
                    ti2 = ti;
                    dtake(ti2, tj, A);
                    tj2 = tj;
                }
            }
            const bool go = pend && ok;
            pend = pend && !ok;
            if (!any(go)) continue;
            dcanon(nw);
            dcanon(ti2);
            dcanon(tj2);
            r += go;
            put(go, go ? r - 1 : 0, nw);
            put(go && !split, pj, tj2);
            put(go, pi, ti2);
            c_pls += go;
            if (go) {
                plateau = 0;
                qlen = 0;
                q_push(pi);
                if (!split) q_push(pj);
                q_push(r - 1);
                rec = plus_record(a, perm, pi, pj, split ? 1 : 0);
            }
        }
        return rec;
    }

    // Classes and hash slices of one walker's live slots from scratch, by the whole warp: a
    // lane per slot, 32 slots at a time (once per launch).  Per factor, chained hash
    // buckets first (heads in the slices' space, chains in the factor's next array,
    // entries slot | 6 more hash bits << 10); every slot walks its bucket for the next
    // member above it, or the lowest one, by hash, checks that one on the words, and
    // only after a mismatch checks every entry.  (Comparing every slot with all slots by
    // the slices took 3.6 ms of a launch of 32768 walkers at 351 terms, this 0.9.)
    __device__ __forceinline__ static void build(const uint64_t *w, int rr, int R, uint16_t *nx, uint32_t *hs) {
        const int l = threadIdx.x & 31, KW = (R + 31) >> 5;
        const int heads = 3 * kHashBits * KW;
        constexpr uint32_t kEnd = 0xffffu;
        auto factor = [&](int s, int f, uint64_t (&p)[FW], uint64_t (&n)[FW]) -> uint32_t {
            uint32_t x = 0u;
#pragma unroll
            for (int h = 0; h < FW; ++h) {
                p[h] = s < rr ? w[(size_t)s * NWG + f * FW + h] : 0ull;
                n[h] = ZT && s < rr ? w[(size_t)s * NWG + TW + f * FW + h] : 0ull;
                x += word_hash(p[h], n[h], h);
            }
            return x;
        };
        uint64_t p[FW], n[FW];
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
            uint16_t *chain = nx + f * R;
            for (int e = l; e < heads; e += 32) hs[e] = kEnd;
            __syncwarp();
#pragma unroll 4
            for (int s = l; s < rr; s += 32) {
                const uint32_t x = factor(s, f, p, n) * 0x9E3779B1u;
                chain[s] = (uint16_t)atomicExch(&hs[__umulhi(x, (uint32_t)heads)], (uint32_t)s | ((x & 63u) << 10));
            }
            __syncwarp();
            uint16_t found[32];   // by chunk
#pragma unroll 1
            for (int q = 0; 32 * q < rr; ++q) {
                const int s = 32 * q + l;
                int nxt = s;
                if (s < rr) {
                    const uint32_t x = factor(s, f, p, n) * 0x9E3779B1u, tag = x & 63u;
                    const uint32_t head = hs[__umulhi(x, (uint32_t)heads)];
                    int above = kNone, below = kNone;
                    for (uint32_t e = head; e != kEnd; e = chain[e & 1023u]) {
                        const int k = (int)(e & 1023u);
                        const bool hit = (e >> 10) == tag;
                        above = hit && k > s ? min(above, k) : above;
                        below = hit && k < s ? min(below, k) : below;
                    }
                    nxt = above != kNone ? above : (below != kNone ? below : s);
                    if (nxt != s && !fsame(w, nxt, f, p, n)) {
                        above = below = kNone;
                        for (uint32_t e = head; e != kEnd; e = chain[e & 1023u]) {
                            const int k = (int)(e & 1023u);
                            if (k == s || (e >> 10) != tag || !fsame(w, k, f, p, n)) continue;
                            if (k > s) above = min(above, k);
                            else below = min(below, k);
                        }
                        nxt = above != kNone ? above : (below != kNone ? below : s);
                    }
                }
                found[q] = (uint16_t)nxt;
            }
            __syncwarp();
            for (int q = 0; 32 * q < R; ++q)
                if (32 * q + l < R) chain[32 * q + l] = 32 * q + l < rr ? found[q] : (uint16_t)(32 * q + l);
            __syncwarp();
        }
#pragma unroll 2
        for (int q = 0; q < KW; ++q)
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const uint32_t x = factor(32 * q + l, f, p, n);
                uint32_t word = 0u;
#pragma unroll
                for (int b = 0; b < kHashBits; ++b) {
                    // slice order of spreads(): top bits of bytes 0 .. 3, then the next bits
                    const unsigned m = __ballot_sync(kFull, (x >> (8 * (b & 3) + 7 - (b >> 2))) & 1u);
                    word = l == b ? m : word;
                }
                if (l < kHashBits) hs[(f * kHashBits + l) * KW + q] = word;
            }
        __syncwarp();
    }

    // the sampled term's class sizes and members below it, one factor per lane 0 .. 2
    __device__ __forceinline__ void classes(int i, int &n0, int &n1, int &n2, int &mine_below) const {
        int n = 0, b = 0;
        if (live && lane < 3) {
            int p = next(i, lane);
#pragma unroll 1
            for (; n < R && p != i; ++n) {
                b += p < i;
                p = next(p, lane);
            }
        }
        __syncwarp();
        n0 = from(n, 0); n1 = from(n, 1); n2 = from(n, 2);
        mine_below = b;
    }

    // w: the walker; lanes without one take part in the warp's votes only
    __device__ __forceinline__ void run(const SegDesc &d, int64_t w, int32_t steps) {
        fq = lane < 3 * FW ? lane : 0;
        tfg_walker_info *H = d.hdr + w;
        r = live ? min(max(H->r, 0), R) : 0;   // in range whatever a restored state holds
        best_r = live ? H->best_r : -1;        // without a walker: no candidate, no best, no expansion
        t = H->t; plateau = H->plateau; best_t = H->best_t;
        dig = H->digest; wid = H->walker_id;
        key0 = d.key0; key1 = d.key1;
        best_nnz = H->best_nnz;
        c_acc = c_rej = c_noc = c_drp = c_mrg = c_pls = c_red = 0;
        qlen = 0; q0 = q1 = q2 = 0;
        uint64_t *bestp = reinterpret_cast<uint64_t *>(d.best) + (size_t)w * R * NWG;
        nnz = 0;
        if (policy_of(d) == 2) {
            uint32_t mine = 0;
#pragma unroll 1
            for (int e = lane; e < r * TW; e += G) {
                const int s = e / TW, q = e - s * TW;
                mine += (uint32_t)__popcll(W[(size_t)s * NWG + q] | (ZT ? W[(size_t)s * NWG + TW + q] : 0ull));
            }
            __syncwarp();
            nnz = sum(mine);
        }

        uint32_t xr0 = 0, xr1 = 0, xr2 = 0, xr3 = 0;
        int kb = G;
#pragma unroll 1
        for (int32_t step = 0; step < steps; ++step) {
            // ---- draw: lane l holds the Philox output of step (batch start + l)
            if (kb == G) {
                const uint64_t tl = (uint64_t)t + (uint64_t)lane;
                const U4 x = philox10((uint32_t)tl, (uint32_t)(tl >> 32), wid, 0u, key0, key1);
                xr0 = x.x; xr1 = x.y; xr2 = x.z; xr3 = x.w;
                kb = 0;
            }
            const uint32_t x0 = from(xr0, kb), x1 = from(xr1, kb), x2 = from(xr2, kb), x3 = PG ? from(xr3, kb) : 0u;
            kb += 1;

            const int r_before = r;
            const int i = (int)__umulhi(x0, (uint32_t)r);
            const DF di = dget(i);   // on its way during the walk over the lists
            // ---- try_flip: candidates (X, j) with X_j = +-X_i, ordered (X, slot)
            int nU, nV, nW, below;
            classes(i, nU, nV, nW, below);
            const int K = live ? 2 * (nU + nV + nW) : 0;
            const int c = (int)__umulhi(x1, (uint32_t)K);
            const int mi = c >> 1;
            int action = kNoCand, X = 0, j = 0, rho = 0, sneg = 0;
            if (K > 0) {
                rho = c & 1;
                X = (int)(mi >= nU) + (int)(mi >= nU + nV);
            }
            const int idx = mi - (X == 0 ? 0 : (X == 1 ? nU : nU + nV));
            const int bX = from(below, X);
            if (K > 0) {
                // the idx-th candidate of factor X in slot order: the cycle after i has the
                // members above i, then those below
                const int n = X == 0 ? nU : (X == 1 ? nV : nW);
                int go = idx < bX ? n - bX + idx : idx - bX;
                j = next(i, X);
#pragma unroll 1
                for (; go > 0; --go) j = next(j, X);
            }
            __syncwarp();
            const DF dj = dget(j);
            const bool wneg = dwneg(dj, di);
            sneg = (X == 2 && wneg && K > 0) ? 1 : 0;
            // flip: (Y, Z) cyclic after X, rho swaps; Y_i += Y_j, Z_j -= s Z_i
            const int X1 = X == 2 ? 0 : X + 1, X2 = X == 0 ? 2 : X - 1;
            const int Y = rho ? X2 : X1, Z = rho ? X1 : X2;
            DF ti2, tj2;
            bool ok = dadd(di, dj, Y, false, ti2);
            ok &= dadd(dj, di, Z, sneg == 0, tj2);
            const bool acc = K > 0 && ok;
            if (K > 0) action = ok ? kAccept : kReject;
            c_noc += K == 0;
            c_rej += action == kReject;
            c_acc += acc;
            qlen = 0;
            if (any(acc)) {
                const bool zi = dzero(ti2, Y);
                const bool zj = dzero(tj2, Z);
                if (policy_of(d) == 2) {
                    const uint32_t ci = dnnz(ti2), cj = dnnz(tj2), bi = dnnz(di), bj = dnnz(dj);
                    if (acc) nnz += (zi ? 0u : ci) + (zj ? 0u : cj) - bi - bj;
                }
                dcanon(ti2);
                dcanon(tj2);
                dput(acc, i, ti2);
                dput(acc, j, tj2);
                // of the other factors the normalisation changes the sign of w at most
                relink<true>(acc, i, Y, ti2, j, Z, tj2);
                const bool zz = acc && (zi || zj);
                if (policy_of(d) != 2) {
                    // A third slot shares a pair with the new term i iff it is in two of its
                    // classes x, e1, z, with the new term j iff in two of x, e2, e3: the five
                    // classes' members (j aside in x) modulo 32, a lane each, as a superset
                    // test (the cascade checks exactly).
                    uint32_t mask = 0u;
                    if (acc && !zz && lane < 5) {
                        const int s = lane < 3 ? i : j;
                        const int f = lane == 0 ? X : ((lane == 1 || lane == 4) ? Z : Y);
                        int p = next(s, f);
#pragma unroll 1
                        for (int q = 0; q < R && p != s; ++q) {
                            mask |= lane == 0 && p == j ? 0u : 1u << (p & 31);
                            p = next(p, f);
                        }
                    }
                    __syncwarp();
                    const uint32_t cx = from(mask, 0), cz = from(mask, 1), e1 = from(mask, 2), e2 = from(mask, 3),
                                   e3 = from(mask, 4);
                    if ((cx & cz) | (e1 & (cx | cz)) | (e2 & (cx | e3)) | (cx & e3)) {
                        q_push(i);
                        q_push(j);
                    }
                }
                if (any(zz)) {
                    if (zz) {
                        q_push(i);
                        q_push(j);
                    }
                    const int hi = i > j ? i : j, lo = i > j ? j : i;
                    const bool zhi = zz && ((hi == i) ? zi : zj), zlo = zz && ((lo == i) ? zi : zj);
                    if (any(zhi)) drop(zhi, hi);
                    if (any(zlo)) drop(zlo, lo);
                    c_drp += (uint32_t)zhi + (uint32_t)zlo;
                    if (policy_of(d) == 2) qlen = 0;   // no reduction edges
                }
            }
            cascade();
            // ---- digest, best scheme, plateau
            c_red += r < r_before;
            dig = digest_mix(dig, flip_record(action, X, rho, sneg, i, j, r));
            // walk policy 1: a failed try_flip expands and ends the step (no best update)
            const bool failed = policy_of(d) == 1 && action != kAccept;
            // best scheme: always when better, with probability 0.01 when equal
            // (policy 2: better = least (rank, non-zero coefficients))
            const bool better = !failed && (r < best_r || (policy_of(d) == 2 && r == best_r && nnz < best_nnz));
            const bool again = !failed && r == best_r && (policy_of(d) != 2 || nnz == best_nnz) && x2 < d.refresh_thresh;
            plateau += 1;
            if (better) {
                best_r = r;
                if (policy_of(d) == 2) best_nnz = nnz;
                best_t = t;
                plateau = 0;
            }
            if (any(better || again)) snapshots(better || again, bestp);
            // expansion: plus on a plateau near the best rank (policy 0), or Algorithm 1's
            // expand after a failed try_flip / with probability p_expand (policy 1)
            bool expand;
            if (policy_of(d) == 2)
                expand = false;
            else if (policy_of(d) == 1)
                expand = failed ? (r < R && r >= 2) : (x3 < d.expand_thresh && r <= best_r + 2 && r < R && r >= 2);
            else
                expand = d.plus_enabled && plateau >= d.plateau_len && r <= best_r + 2 && r < R && r >= 2;
            __syncwarp();
            if (any(expand)) {
                const uint64_t rec = plus_setup(d, expand);
                cascade();
                if (rec) dig = digest_mix(dig, rec | ((uint64_t)(uint32_t)r << 44));
            }
            t += 1;
        }

        // ---- write back (the slots were written in place)
        if (live && lane == 0) {
            H->r = r; H->best_r = best_r;
            H->t = t; H->plateau = plateau; H->best_t = best_t;
            H->digest = dig;
            H->accepted += c_acc; H->rejected += c_rej; H->nocand += c_noc;
            H->drops += c_drp; H->merges += c_mrg; H->plus += c_pls; H->reductions += c_red;
            H->best_nnz = best_nnz;
        }
    }
};

constexpr int kWideBlock = 64;

// per: walkers per warp (1 .. 4), the first of its four groups of lanes
template <int MODE, bool PG, int FW, bool GM>
__global__ void __launch_bounds__(kWideBlock, 10) walk_wide_kernel(const SegDesc d, const int32_t steps, const int per) {
    extern __shared__ __align__(16) unsigned char wide_sm[];
    using WW = WideWalker<MODE, PG, FW, GM>;
    const int wl = threadIdx.x & 31, group = wl / WW::G;
    const size_t bytes = WW::walker_bytes(d.R);
    unsigned char *at = wide_sm + bytes * per * (threadIdx.x >> 5);
    const int64_t first = ((int64_t)blockIdx.x * (kWideBlock / 32) + (threadIdx.x >> 5)) * per;
    if (first >= d.n_walkers) return;   // no block-wide barrier is used
    const int here = (int)min((int64_t)per, d.n_walkers - first);   // the warp's walkers
    WW wk;
    wk.R = d.R;
    wk.KW = (d.R + 31) >> 5;
    const int words = d.R * WW::NWG;
    uint64_t *slots = reinterpret_cast<uint64_t *>(d.slots) + (size_t)first * words;
    // the whole warp stages its walkers and builds their classes, one after another
#pragma unroll 1
    for (int a = 0; a < here; ++a) {
        wk.attach(at + bytes * a, slots + (size_t)a * words);
        if constexpr (!GM) {
#pragma unroll 4
            for (int e = wl; e < words; e += 32) wk.W[e] = slots[(size_t)a * words + e];
            __syncwarp();
        }
        WW::build(wk.W, min(max(d.hdr[first + a].r, 0), d.R), d.R, wk.nx, wk.hs);
    }
    wk.lane = wl % WW::G;
    wk.gb = wl - wk.lane;
    wk.live = group < here;
    const int a = wk.live ? group : 0;
    wk.attach(at + bytes * a, slots + (size_t)a * words);
    wk.run(d, first + a, steps);
    if constexpr (!GM) {
        __syncwarp();
#pragma unroll 1
        for (int b = 0; b < here; ++b) {
            wk.attach(at + bytes * b, slots);
#pragma unroll 4
            for (int e = wl; e < words; e += 32) slots[(size_t)b * words + e] = wk.W[e];
        }
    }
}

}  // namespace dev

namespace {

template <int MODE, int FW>
void prepare_walk_wide() {
    prepare_walk_search<MODE, FW>();
    static bool attr = [] {
        auto set = [](auto kernel) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinkSmem);
        };
        set(dev::walk_wide_kernel<MODE, false, FW, false>);
        set(dev::walk_wide_kernel<MODE, false, FW, true>);
        set(dev::walk_wide_kernel<MODE, true, FW, false>);
        set(dev::walk_wide_kernel<MODE, true, FW, true>);
        return true;
    }();
    (void)attr;
}

// When keeping the classes pays.  They are built at every launch (about 60 steps' worth at
// 351 terms), a step with four walkers a warp takes longer than a warp's on one walker
// unless the warps are many, and an expansion (walk policy 1) changes three terms.
// Measured, every step searching / keeping classes, ms: policy 0, (4,5,5) Z_T 300 steps 1000
// walkers 0.39 / 0.43, 4000 0.98 / 0.76, 16000 3.0 / 1.8; (5,6,10) Z_T 16000 walkers 60 steps
// 0.92 x, 300 steps 1.35 x; policy 2, (4,5,5) Z_2 300 steps 4000 walkers 0.96 x, 8000 1.48 x;
// policy 1, 300 steps, 8000 walkers: (4,5,5) Z_T 1.21 x, Z_2 0.98 x, (6,7,9) 1.54 x, 60 steps 0.91 x.
template <int MODE>
bool classes_pay(const SegDesc &d, int32_t steps) {
    const bool large = d.R >= 256;
    if (d.walk_policy == 0) return d.population >= 4000 && steps >= (large ? 120 : 40);
    if (d.walk_policy == 2) return d.population >= 8000 && steps >= (large ? 200 : 60);
    return d.population >= 8000 && steps >= 300 && (MODE == TFG_MODE_ZT || d.R >= 128);
}

// Walkers per warp: four, unless that leaves an SM's schedulers without two warps each; a
// warp takes the changing part of a step when any of its walkers does, so a lone
// walker's step is shorter.  The terms go to shared memory when the whole population
// resides at once that way.
struct WidePlan {
    int per;   // walkers per warp
    unsigned grid;
    bool shared;
    size_t smem;
};
template <int MODE, int FW>
WidePlan wide_plan(const SegDesc &d) {
    using Shared = dev::WideWalker<MODE, false, FW, false>;
    using Device = dev::WideWalker<MODE, false, FW, true>;
    int per = 32 / Shared::G;
    while (per > 1 && (d.population + per - 1) / per < (int64_t)sm_count() * 8) per /= 2;
    const int walkers = dev::kWideBlock / 32 * per;   // of a block
    const unsigned grid = (unsigned)((d.n_walkers + walkers - 1) / walkers);
    const bool shared = link_terms_shared(Shared::walker_bytes(d.R) * walkers, (d.population + walkers - 1) / walkers);
    return {per, grid, shared, (shared ? Shared::walker_bytes(d.R) : Device::walker_bytes(d.R)) * walkers};
}
template <int MODE, int FW>
LaunchShape wide_shape(const SegDesc &d, int /*block*/) {
    if (!classes_pay<MODE>(d, INT32_MAX)) return search_shape(d);
    return {dev::WideWalker<MODE, false, FW, true>::G, dev::kWideBlock, wide_plan<MODE, FW>(d).grid};
}

template <int MODE, int FW>
void launch_walk_wide(const SegDesc &d, int32_t steps, int /*grid*/, int /*block*/, cudaStream_t st) {
    if (!classes_pay<MODE>(d, steps)) {
        launch_walk_search<MODE, FW>(d, steps, st);
        return;
    }
    prepare_walk_wide<MODE, FW>();
    if (d.n_walkers <= 0) return;
    const WidePlan k = wide_plan<MODE, FW>(d);
    if (k.shared) {
        if (d.walk_policy == 0) dev::walk_wide_kernel<MODE, false, FW, false><<<k.grid, dev::kWideBlock, k.smem, st>>>(d, steps, k.per);
        else dev::walk_wide_kernel<MODE, true, FW, false><<<k.grid, dev::kWideBlock, k.smem, st>>>(d, steps, k.per);
    } else {
        if (d.walk_policy == 0) dev::walk_wide_kernel<MODE, false, FW, true><<<k.grid, dev::kWideBlock, k.smem, st>>>(d, steps, k.per);
        else dev::walk_wide_kernel<MODE, true, FW, true><<<k.grid, dev::kWideBlock, k.smem, st>>>(d, steps, k.per);
    }
}

// G = 32 is the mapping's name in tfg_params and tfg_mapping; the kernel sets its own launch shape.
template <int MODE, int FW>
WalkVariant wide_variant() {
    return WalkVariant{MODE, 64, 3 * FW, 32, 0, 0, &launch_walk_wide<MODE, FW>,
                       reinterpret_cast<const void *>(&dev::walk_wide_kernel<MODE, false, FW, true>),
                       &prepare_walk_wide<MODE, FW>, &wide_shape<MODE, FW>, 1023};
}

}  // namespace

// Factor-aligned terms: 3 (factors of at most 64 coefficients) or 6 (at most
// 128) words of 64 bits per sign; capacity 1023 slots (74 KB of shared memory for a
// block's eight walkers).
const WalkVariant *walk_variants_wide(int *n) {
    static const WalkVariant v[] = {wide_variant<TFG_MODE_ZT, 1>(), wide_variant<TFG_MODE_Z2, 1>(),
                                    wide_variant<TFG_MODE_ZT, 2>(), wide_variant<TFG_MODE_Z2, 2>()};
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}

}  // namespace tfg
