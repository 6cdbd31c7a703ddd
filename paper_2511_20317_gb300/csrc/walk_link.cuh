// Thread-per-walker flip-graph walk kernel with incremental factor classes, for
// sm_103a: terms of at most 64 coefficients, at most 96 slots.
//
// try_flip asks, for a sampled term, which other slots hold an equal factor u, v
// or w (w up to sign).  A step changes at most two factors of the scheme (and
// most steps, rejected ones, change none), so the answer is kept instead of
// being searched for: per factor the slots form classes of equal factors, and
// only an accepted flip moves two slots to other classes.
//   NW = 1 (at most 32 slots): one 32-bit row per slot and factor, bit k = slot
//     k holds an equal factor (ROWS);
//   NW > 1, or LIST: the slots of a class form a cyclic list in ascending order, one byte
//     per slot and factor (the next member), so that a walker needs 4 bytes
//     per slot instead of 3 * 4 * NW (link_lists_pay says when at most 32 slots take lists).
// Where a changed factor goes is found by its 8-bit hash: the hashes of all
// slots are held bit-sliced (word q of slice b: bit b of the hashes of slots
// 32 q .. 32 q + 31), so that one pass over the 8 NW words of the factor compares
// with all slots and rewrites the slot's own bits; every slot the hashes leave
// over (about r / 256 false ones) is checked on the terms, so classes are exact.
//
// Slots, classes and slices sit in shared memory as [row][lane], a row of every
// lane's words side by side: a thread's accesses at a row of its own never
// conflict with another lane's.  GM: the packed terms stay in the walker's
// device-memory slots.  PG: the walk policy is read from the descriptor (policies 1
// and 2); without it the plateau policy is compiled in alone.  CNT (window mode): lists
// at any capacity, and every slot's number of matches (u, v and w) is kept too.
//
// What bounds it: the latency of a warp's step (600 to 1300 instructions, most of them in
// the accepting lanes' short dependent loops, 13 of 32 lanes active; at 62% of the issue
// rate with 14 warps an SM, 35% with 7 to 9).  The kernel it replaces tested every slot in every
// step (5500 instructions a warp-step at 83 slots, two thirds of the ALU pipe).
// Measured, Z_T, steps/s before / now: (2,3,4) 65536 walkers 1.43e10 / 2.60e10, (3,3,4)
// 40330 4.9e9 / 1.24e10, (3,4,5) 40330 4.3e9 / 1.12e10, (4,4,4) 80660 4.0e9 / 1.07e10,
// (4,4,5) 80660 2.6e9 / 9.5e9; Z_2 (4,4,5) 2.4e9 / 6.8e9; Algorithm 1 policy (3,3,4)
// 10007 walkers 6.9e8 / 3.1e9; (2,2,2) 1024 walkers 8.9e8 / 1.7e9.
//
// Step order and every tie-break are those of the lane-group kernel and of the
// CPU reference:
//   draw -> sample term i -> try_flip candidates ordered (factor, slot, rho)
//   -> flip + ternary validity -> zero-term removal -> sign normalisation ->
//   reduction cascade -> best/plateau -> plus transition (+ cascade).
#pragma once
#include <algorithm>
#include <cstdint>

#include "pterm.cuh"

namespace tfg {
namespace dev {

constexpr int kHashBits = 8;
constexpr int kLane = 32;   // stride of a thread's rows in its warp's shared memory

// The lanes of this thread's warp that hold walkers (the first ones), taken by all threads of
// a block, of whole warps or of fewer than 32 threads, before those past the population
// return.  Not read off the hardware where it is used: loading a walker runs loops of
// different lengths, after which a warp need not be together.
__device__ __forceinline__ unsigned walker_lanes(const SegDesc &d, int64_t w) {
    return __ballot_sync(blockDim.x < 32 ? (1u << blockDim.x) - 1u : ~0u, w < d.n_walkers);
}

// all four bytes = the sign of byte B (compile-time) of x: a word of 0 or of ones
template <int B>
__device__ __forceinline__ uint32_t sign_spread(uint32_t x) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %1, %2;" : "=r"(r) : "r"(x), "n"((8 | B) * 0x1111));
    return r;
}

template <int MODE, class Wd, int NW, bool GM, bool PG, bool CNT = false, bool LIST = false>
struct LinkWalker {
    static constexpr bool ZT = (MODE == TFG_MODE_ZT);
    static constexpr int NWS = ZT ? 2 : 1;   // words per slot
    static constexpr bool ROWS = NW == 1 && !CNT && !LIST;
    static constexpr bool kCounts = CNT;
    using T = PTerm<Wd, 1, ZT>;
    using O = Ops<Wd, 1, ZT>;
    using M = Masks<Wd, 1>;

    Wd *sm;           // slot k at sm[k * RS]: this thread's shared-memory column, or (GM) the walker's own slots
    uint32_t *ix;     // ROWS: row of slot k, factor f at ix[(3 k + f) * kLane]; lists: next of (k, f) = byte f of ix[k * kLane]
    uint32_t *cn;     // CNT: matches of slots 2k and 2k + 1 in the halves of cn[k * kLane]
    int matches;      // CNT: their sum
    uint32_t *hs;     // hash slices: bit b of factor f, word q at hs[((f * 8 + b) * NW + q) * kLane]
    M mk;
    int r, best_r, R;
    int64_t t, best_t;
    int64_t t_zero;             // plateau (steps without a better best scheme) after the step at t: t - t_zero
    int64_t t_exp;              // the step from which the plateau policy expands: t_zero + plateau_len
    uint64_t dig;
    uint32_t wid, key0, key1;
    uint32_t c_acc, c_rej, c_drp, c_mrg, c_pls, c_red;
    int qlen, q0, q1, q2;
    uint32_t nnz, best_nnz;     // non-zero coefficients of the live / best scheme (nnz: policy 2 only)

    static constexpr int RS = GM ? NWS : kLane * NWS;

    // words of shared memory of a thread
    __host__ __device__ static constexpr size_t thread_bytes(int R) {
        return (GM ? (size_t)0 : (size_t)R * NWS * sizeof(Wd)) + (size_t)R * (ROWS ? 12 : 4) +
               (CNT ? (size_t)(R + 1) / 2 * 4 : (size_t)0) + (size_t)3 * kHashBits * NW * 4;
    }

    __device__ __forceinline__ static int popc_word(Wd x) {
        if constexpr (sizeof(Wd) == 8) return __popcll(x);
        else return __popc(x);
    }
    __device__ __forceinline__ static uint32_t nnz_of(const T &v) {
        if constexpr (ZT) return (uint32_t)popc_word(v.p[0] | v.n[0]);
        else return (uint32_t)popc_word(v.p[0]);
    }

    // ---- packed terms
    __device__ __forceinline__ static T ld_at(const Wd *a) {
        T v;
        if constexpr (ZT) {
            if constexpr (sizeof(Wd) == 4) {
                const uint2 q = *reinterpret_cast<const uint2 *>(a);
                v.p[0] = q.x; v.n[0] = q.y;
            } else {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(a);
                v.p[0] = q.x; v.n[0] = q.y;
            }
        } else {
            v.p[0] = a[0];
            v.n[0] = 0;
        }
        return v;
    }
    __device__ __forceinline__ T ld(int k) const { return ld_at(sm + (size_t)(k * RS)); }
    __device__ __forceinline__ void st(int k, const T &v) {
        Wd *a = sm + (size_t)(k * RS);
        if constexpr (ZT) {
            if constexpr (sizeof(Wd) == 4) *reinterpret_cast<uint2 *>(a) = make_uint2(v.p[0], v.n[0]);
            else *reinterpret_cast<ulonglong2 *>(a) = make_ulonglong2(v.p[0], v.n[0]);
        } else {
            a[0] = v.p[0];
        }
    }

    // ---- factor classes
    __device__ __forceinline__ uint32_t &row(int k, int f) const { return ix[(3 * k + f) * kLane]; }
    __device__ __forceinline__ uint8_t &next(int k, int f) const { return reinterpret_cast<uint8_t *>(ix)[k * (kLane * 4) + f]; }

    // CNT: slot k's number of matches changes by n
    __device__ __forceinline__ void count(int k, int n) {
        if constexpr (CNT) {
            reinterpret_cast<uint16_t *>(cn)[(k >> 1) * (kLane * 2) + (k & 1)] += (uint16_t)n;
            matches += n;
        }
    }
    // f(k) for every other slot of slot s's class of factor fc
    template <class F>
    __device__ __forceinline__ void each_match(int s, int fc, F f) const {
        if constexpr (ROWS) {
            uint32_t m = row(s, fc);
#pragma unroll 1
            while (m) {
                f(__ffs(m) - 1);
                m &= m - 1u;
            }
        } else {
#pragma unroll 1
            for (int p = next(s, fc); p != s; p = next(p, fc)) f(p);
        }
    }

    // Symmetric in the two signs, so that w's class (up to sign) has one hash; u and
    // v are sign-normalised and never meet their negatives.
    __device__ __forceinline__ static uint32_t fold(Wd x) {
        if constexpr (sizeof(Wd) == 4) {
            const uint64_t a = (uint64_t)x * 0x9E3779B1u;
            return (uint32_t)a ^ (uint32_t)(a >> 32);
        } else {
            const uint64_t a = (uint64_t)(uint32_t)x * 0x9E3779B1u + (uint64_t)(uint32_t)(x >> 32) * 0x85EBCA77u;
            return (uint32_t)a ^ (uint32_t)(a >> 32);
        }
    }
    __device__ __forceinline__ static uint32_t factor_hash(const T &v, Wd m) {
        uint32_t h = fold(v.p[0] & m);
        if constexpr (ZT) h += fold(v.n[0] & m);
        return h;
    }
    // The same with the product of the two parts mixed in: the sum alone gives a + b and
    // a - b nearly the same hash, which 8 bits do not notice and 16 do (at 64 slots, 65%
    // of the walkers had two factors of one 16-bit hash, now 3%).
    __device__ __forceinline__ static uint32_t factor_hash16(const T &v, Wd m) {
        const uint32_t a = fold(v.p[0] & m), b = ZT ? fold(v.n[0] & m) : 0u;
        const uint64_t c = (uint64_t)a * b;
        return a + b + ((uint32_t)c ^ (uint32_t)(c >> 32));
    }
    // the factors of a and b under mask m are equal up to sign
    __device__ __forceinline__ static bool same(const T &a, const T &b, Wd m) {
        if constexpr (ZT)
            return ((((a.p[0] ^ b.p[0]) | (a.n[0] ^ b.n[0])) & m) == Wd(0)) ||
                   ((((a.p[0] ^ b.n[0]) | (a.n[0] ^ b.p[0])) & m) == Wd(0));
        else
            return ((a.p[0] ^ b.p[0]) & m) == Wd(0);
    }
    // Slots that may hold the factor f of hash h, slot s aside; s's own slices := the hash.
    __device__ __forceinline__ void scan(int s, int f, uint32_t h, uint32_t (&c)[NW]) const {
        uint32_t d[NW];
#pragma unroll
        for (int q = 0; q < NW; ++q) d[q] = 0u;
        uint32_t *base = hs + f * (kHashBits * NW * kLane);
        const uint32_t sb = 1u << (s & 31);
        uint32_t sp[kHashBits];
        sp[0] = sign_spread<0>(h); sp[1] = sign_spread<1>(h); sp[2] = sign_spread<2>(h); sp[3] = sign_spread<3>(h);
        const uint32_t h1 = h << 1;
        sp[4] = sign_spread<0>(h1); sp[5] = sign_spread<1>(h1); sp[6] = sign_spread<2>(h1); sp[7] = sign_spread<3>(h1);
        if constexpr (ROWS) {
#pragma unroll
            for (int b = 0; b < kHashBits; ++b) {
                const uint32_t w = base[b * kLane];
                d[0] |= w ^ sp[b];
                base[b * kLane] = (w & ~sb) | (sp[b] & sb);
            }
        } else {
            uint32_t *own = base + (s >> 5) * kLane;
#pragma unroll
            for (int b = 0; b < kHashBits; ++b) {
#pragma unroll
                for (int q = 0; q < NW; ++q) d[q] |= base[(b * NW + q) * kLane] ^ sp[b];
            }
#pragma unroll
            for (int b = 0; b < kHashBits; ++b) {
                const uint32_t w = own[b * NW * kLane];
                own[b * NW * kLane] = (w & ~sb) | (sp[b] & sb);
            }
        }
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const int lo = r - 32 * q;
            uint32_t live = lo >= 32 ? ~0u : (lo > 0 ? (1u << lo) - 1u : 0u);
            if (ROWS || (s >> 5) == q) live &= ~sb;
            c[q] = ~d[q] & live;
        }
    }
    // the lowest set slot of c, removed from it (c not empty)
    __device__ __forceinline__ static int take_lowest(uint32_t (&c)[NW]) {
        if constexpr (NW == 1) {
            const int k = __ffs(c[0]) - 1;
            c[0] &= c[0] - 1u;
            return k;
        } else {
            int k = 0;
            bool done = false;
#pragma unroll
            for (int q = 0; q < NW; ++q) {
                const bool here = !done && c[q] != 0u;
                k = here ? 32 * q + __ffs(c[q]) - 1 : k;
                c[q] = here ? c[q] & (c[q] - 1u) : c[q];
                done = done || here;
            }
            return k;
        }
    }
    __device__ __forceinline__ static bool some(const uint32_t (&c)[NW]) {
        uint32_t o = c[0];
#pragma unroll
        for (int q = 1; q < NW; ++q) o |= c[q];
        return o != 0u;
    }
    // One or (TWO) two slots change their class: slot sa's factor fa is now va's, slot
    // sb's factor fb (fb != fa) now vb's.  The two moves run side by side: they touch
    // different factors' classes, and a thread's time is the latency of these short
    // dependent loops.  ROWS: returns the new classes.
    template <bool TWO>
    __device__ __forceinline__ void relink_pair(int sa, int fa, const T &va, int sb, int fb, const T &vb, uint32_t &ea,
                                                uint32_t &eb) {
        const Wd ma = mk.of(fa, 0), mb = TWO ? mk.of(fb, 0) : Wd(0);
        uint32_t ca[NW], cb[NW];
        scan(sa, fa, factor_hash(va, ma), ca);
        if constexpr (TWO) {
            scan(sb, fb, factor_hash(vb, mb), cb);
        } else {
#pragma unroll
            for (int q = 0; q < NW; ++q) cb[q] = 0u;
        }
        if constexpr (ROWS) {
            ea = eb = 0u;
#pragma unroll 1
            while (ca[0] | cb[0]) {
                const uint32_t la = ca[0] & (0u - ca[0]), lb = cb[0] & (0u - cb[0]);
                const T xa = ld(ca[0] ? __ffs(ca[0]) - 1 : 0);
                ea |= same(xa, va, ma) ? la : 0u;
                ca[0] ^= la;
                if constexpr (TWO) {
                    const T xb = ld(cb[0] ? __ffs(cb[0]) - 1 : 0);
                    eb |= same(xb, vb, mb) ? lb : 0u;
                    cb[0] ^= lb;
                }
            }
            // rows that gain or lose the slot
            uint32_t ha = row(sa, fa) ^ ea, hb = 0u;
            row(sa, fa) = ea;
            if constexpr (TWO) {
                hb = row(sb, fb) ^ eb;
                row(sb, fb) = eb;
            }
            const uint32_t ba = 1u << sa, bb = 1u << sb;
#pragma unroll 1
            while (ha | hb) {
                if (ha) {
                    row(__ffs(ha) - 1, fa) ^= ba;
                    ha &= ha - 1u;
                }
                if constexpr (TWO) {
                    if (hb) {
                        row(__ffs(hb) - 1, fb) ^= bb;
                        hb &= hb - 1u;
                    }
                }
            }
        } else {
            // a slot of the new class: the lowest one with the same factor
            int ga = -1, gb = -1;
            bool na = some(ca), nb = some(cb);
#pragma unroll 1
            while (na || nb) {
                if (na) {
                    const int k = take_lowest(ca);
                    const bool ok = same(ld(k), va, ma);
                    ga = ok ? k : ga;
                    na = !ok && some(ca);
                }
                if (TWO && nb) {
                    const int k = take_lowest(cb);
                    const bool ok = same(ld(k), vb, mb);
                    gb = ok ? k : gb;
                    nb = !ok && some(cb);
                }
            }
            // out of the old cycles: find the members before the slots
            const int oa = next(sa, fa), ob = TWO ? next(sb, fb) : sb;
            int pa = sa, qa = oa, pb = sb, qb = ob;   // q = next of p
#pragma unroll 1
            while (qa != sa || (TWO && qb != sb)) {
                if (qa != sa) { pa = qa; count(pa, -1); count(sa, -1); qa = next(pa, fa); }
                if (TWO && qb != sb) { pb = qb; count(pb, -1); count(sb, -1); qb = next(pb, fb); }
            }
            next(pa, fa) = (uint8_t)oa;
            if (TWO) next(pb, fb) = (uint8_t)ob;
            // into the new ones: between p < s < n, or at the wrap (n <= p)
            pa = ga >= 0 ? ga : sa;
            qa = ga >= 0 ? next(ga, fa) : sa;
            if (TWO) { pb = gb >= 0 ? gb : sb; qb = gb >= 0 ? next(gb, fb) : sb; }
            auto seek = [](int p, int q, int s) { return !(p < q ? (p < s && s < q) : (s >= p || s <= q)); };
            bool ma2 = seek(pa, qa, sa), mb2 = TWO && seek(pb, qb, sb);
#pragma unroll 1
            while (ma2 || mb2) {
                if (ma2) { pa = qa; qa = next(pa, fa); ma2 = seek(pa, qa, sa); }
                if (TWO && mb2) { pb = qb; qb = next(pb, fb); mb2 = seek(pb, qb, sb); }
            }
            next(pa, fa) = (uint8_t)sa;
            next(sa, fa) = (uint8_t)qa;
            if (TWO) { next(pb, fb) = (uint8_t)sb; next(sb, fb) = (uint8_t)qb; }
            if constexpr (CNT) {
#pragma unroll 1
                while (qa != sa || (TWO && qb != sb)) {
                    if (qa != sa) { count(qa, 1); count(sa, 1); qa = next(qa, fa); }
                    if (TWO && qb != sb) { count(qb, 1); count(sb, 1); qb = next(qb, fb); }
                }
            }
        }
    }
    __device__ __forceinline__ void relink(int s, int f, const T &v) {
        uint32_t ea, eb;
        relink_pair<false>(s, f, v, s, f, v, ea, eb);
    }
    // Lists: slot s (a class of its own) into the class of slot m
    __device__ __forceinline__ void link(int s, int f, int m) {
        int p = m, n = next(p, f);
#pragma unroll 1
        while (!(p < n ? (p < s && s < n) : (s > p || s < n))) {
            p = n;
            n = next(p, f);
        }
        next(p, f) = (uint8_t)s;
        next(s, f) = (uint8_t)n;
        if constexpr (CNT) {
#pragma unroll 1
            for (; n != s; n = next(n, f)) {
                count(n, 1);
                count(s, 1);
            }
        }
    }
    // take slot s out of its class of factor f (it becomes a class of its own)
    __device__ __forceinline__ void unlink(int s, int f) {
        if constexpr (ROWS) {
            uint32_t ch = row(s, f);
            const uint32_t sb = 1u << s;
            row(s, f) = 0u;
#pragma unroll 1
            while (ch) {
                row(__ffs(ch) - 1, f) ^= sb;
                ch &= ch - 1u;
            }
        } else {
            const int n = next(s, f);
            if (n != s) {
                int p = s, q = n;
#pragma unroll 1
                while (q != s) {
                    p = q;
                    count(p, -1);
                    count(s, -1);
                    q = next(p, f);
                }
                next(p, f) = (uint8_t)n;
                next(s, f) = (uint8_t)s;
            }
        }
    }
    // ---- reduction queue (slot indices)
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
    __device__ __forceinline__ void q_rename(int from, int to) {
        q0 = (qlen > 0 && q0 == from) ? to : q0;
        q1 = (qlen > 1 && q1 == from) ? to : q1;
        q2 = (qlen > 2 && q2 == from) ? to : q2;
    }

    // Slot h (in no class) takes slot last's term and place in its classes; last leaves them.
    __device__ __forceinline__ void move_slot(int last, int h) {
        st(h, ld(last));
        // hash bits
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
            uint32_t *from = hs + (f * kHashBits * NW + (last >> 5)) * kLane, *to = hs + (f * kHashBits * NW + (h >> 5)) * kLane;
#pragma unroll
            for (int b = 0; b < kHashBits; ++b) {
                const uint32_t v = (from[b * NW * kLane] >> (last & 31)) & 1u, w = to[b * NW * kLane];
                to[b * NW * kLane] = (w & ~(1u << (h & 31))) | (v << (h & 31));
            }
            if constexpr (ROWS) {
                uint32_t e = row(last, f);
                row(last, f) = 0u;
                row(h, f) = e;
                const uint32_t both = (1u << last) | (1u << h);
#pragma unroll 1
                while (e) {
                    row(__ffs(e) - 1, f) ^= both;
                    e &= e - 1u;
                }
            } else {
                const int m = next(last, f);
                unlink(last, f);
                if (m != last) link(h, f, m);
            }
        }
    }
    // Remove slot h: the last live term moves into the hole.
    __device__ __forceinline__ void drop(int h) {
        const int last = r - 1;
        q_remove(h);
#pragma unroll 1
        for (int f = 0; f < 3; ++f) unlink(h, f);
        r -= 1;
        if (h != last) {
            move_slot(last, h);
            q_rename(last, h);
        }
    }

    // validity of a_f + (neg ? -b_f : b_f)
    __device__ __forceinline__ bool sum_ok(const T &a, const T &b, Wd m, bool neg) const {
        if constexpr (ZT) {
            const Wd bp = neg ? b.n[0] : b.p[0], bn = neg ? b.p[0] : b.n[0];
            return (((a.p[0] & bp) | (a.n[0] & bn)) & m) == Wd(0);
        } else {
            return true;
        }
    }

    // Reduction of slot s with the lowest partner sharing (u,v), else (u,w),
    // else (v,w), whose merged third factor stays in the coefficient set.
    __device__ __forceinline__ void reduce_one(int s) {
        const T v = ld(s);
        constexpr int kNone = 1 << 20;
        int k0 = kNone, k1 = kNone, k2 = kNone;
        bool n1 = false, n2 = false;
        each_match(s, 0, [&](int k) {
            const T c = ld(k);
            bool eu, ev, ewp, ewn;
            O::compare(c, v, mk, eu, ev, ewp, ewn);
            if (ev && k < k0 && sum_ok(v, c, mk.m[2][0], false)) k0 = k;
            if ((ewp || ewn) && k < k1 && sum_ok(v, c, mk.m[1][0], ewn)) { k1 = k; n1 = ewn; }
        });
        if (k0 == kNone && k1 == kNone)
            each_match(s, 1, [&](int k) {
                const T c = ld(k);
                bool eu, ev, ewp, ewn;
                O::compare(c, v, mk, eu, ev, ewp, ewn);
                if ((ewp || ewn) && k < k2 && sum_ok(v, c, mk.m[0][0], ewn)) { k2 = k; n2 = ewn; }
            });
        if (k0 == kNone && k1 == kNone && k2 == kNone) return;
        const int P = k0 != kNone ? 0 : (k1 != kNone ? 1 : 2);
        const int k = P == 0 ? k0 : (P == 1 ? k1 : k2);
        const bool kneg = P == 1 ? n1 : (P == 2 ? n2 : false);
        const int F = 2 - P;   // third factor: w, v, u
        const T kv = ld(k);
        T mv;
        O::add(v, kv, F, kneg, mk, mv);
        const bool zero = O::zero(mv, F, mk);
        O::canon(mv, mk);
        const int lo = s < k ? s : k;
        const int hi = s < k ? k : s;
        q_remove(k);
        st(lo, mv);
        relink(lo, F, mv);   // s and k share the other two factors
        c_mrg += 1;
        drop(hi);
        if (zero) {
            drop(lo);
            c_drp += 1;
        } else {
            q_push(lo);
        }
    }

    // Reduction cascade of every thread of the warp: the loop runs while any
    // thread still has queued terms, so the warp is converged afterwards.
    __device__ __forceinline__ void cascade_all(unsigned wmask) {
#pragma unroll 1
        while (__any_sync(wmask, qlen > 0)) {
            if (qlen > 0) reduce_one(q_pop());
        }
    }

    // Warp-cooperative best snapshot: lanes copy consecutive slots of each
    // requesting walker to its best buffer (coalesced stores).
    __device__ __forceinline__ void coop_snapshot(unsigned wmask, int lane, int nl, bool want, Wd *bestp) const {
        unsigned pend = __ballot_sync(wmask, want);
        if (pend == 0u) return;
        __syncwarp(wmask);   // the slots as their owners left them, and (below) left alone until they are read
#pragma unroll 1
        while (pend) {
            const int a = __ffs(pend) - 1;
            pend &= pend - 1;
            const int ra = __shfl_sync(wmask, r, a);
            Wd *dst = reinterpret_cast<Wd *>(__shfl_sync(wmask, reinterpret_cast<unsigned long long>(bestp), a));
            const Wd *col;
            if constexpr (GM)
                col = reinterpret_cast<const Wd *>(__shfl_sync(wmask, reinterpret_cast<unsigned long long>(sm), a));
            else
                col = sm + (a - lane) * NWS;
#pragma unroll 1
            for (int k = lane; k < ra; k += nl) {
                const T v = ld_at(col + (size_t)(k * RS));
                if constexpr (ZT) {
                    if constexpr (sizeof(Wd) == 4) reinterpret_cast<uint2 *>(dst)[k] = make_uint2(v.p[0], v.n[0]);
                    else reinterpret_cast<ulonglong2 *>(dst)[k] = make_ulonglong2(v.p[0], v.n[0]);
                } else {
                    dst[k] = v.p[0];
                }
            }
        }
        __syncwarp(wmask);
    }

    // Expansion (Section 3.3.1): plus (three terms from the pair) or, under
    // walk policy 1 when y3 >= 2^31, split (term i = (A_j, B_i, C_i), new term
    // (A_i - A_j, B_i, C_i)); writes the new terms, queues them for the cascade
    // and returns the digest record (0 when no attempt passed).
    __device__ __forceinline__ uint64_t plus_setup(const SegDesc &d) {
#pragma unroll 1
        for (int a = 1; a <= d.plus_attempts; ++a) {
            const U4 y = philox10((uint32_t)t, (uint32_t)(t >> 32), wid, (uint32_t)a, key0, key1);
            const int pi = (int)__umulhi(y.x, (uint32_t)r);
            const int pj = (pi + 1 + (int)__umulhi(y.y, (uint32_t)(r - 1))) % r;
            const int perm = (int)__umulhi(y.z, 6u);
            const bool split = PG && d.walk_policy == 1 && y.w >= 0x80000000u;
            int A, B, C;
            plus_roles(perm, A, B, C);
            const T ti = ld(pi), tj = ld(pj);
            T nx, ti2, tj2;   // the new term, terms i and j afterwards
            if (split) {
                const bool ok = O::add(ti, tj, A, true, mk, nx);   // (A_i - A_j, B_i, C_i)
                if (!ok || O::zero(nx, A, mk)) continue;
                ti2 = ti;                                          // (A_j, B_i, C_i)
                O::take(ti2, tj, A, mk);
                tj2 = tj;
            } else {
                bool ok = O::add(ti, tj, B, false, mk, ti2);       // (A_i, B_i + B_j, C_i)
                ok &= O::add(tj, ti, C, true, mk, tj2);            // (A_i, B_j, C_j - C_i)
                ok &= O::add(tj, ti, A, true, mk, nx);             // (A_j - A_i, B_j, C_j)
                ok = ok && !O::zero(ti2, B, mk) && !O::zero(tj2, C, mk) && !O::zero(nx, A, mk);
                if (!ok) continue;
                O::take(tj2, ti, A, mk);
                O::canon(tj2, mk);
            }
            O::canon(nx, mk);
            O::canon(ti2, mk);
            // Slots i and j and the new one are stored, then enter their classes factor by
            // factor (a split leaves term j, and of term i only A changes): of each factor
            // the slot that had a class before comes first, the new slot, still alone, last.
            const int n = r;
            r += 1;
            st(pi, ti2);
            st(n, nx);
            uint32_t e0, e1;
            if (split) {
                relink_pair<true>(pi, A, ti2, n, B, nx, e0, e1);
                relink_pair<true>(n, A, nx, n, C, nx, e0, e1);
            } else {
                st(pj, tj2);
#pragma unroll 1
                for (int h = 0; h < 3; ++h) {
                    const bool h0 = h == 0, h1 = h == 1;
                    relink_pair<true>(h0 ? pi : (h1 ? pj : n), h0 ? B : (h1 ? C : B), h0 ? ti2 : (h1 ? tj2 : nx),
                                      h0 ? pj : n, h0 ? A : (h1 ? A : C), h0 ? tj2 : nx, e0, e1);
                }
            }
            restart(d);
            c_pls += 1;
            qlen = 0;
            q_push(pi);
            if (!split) q_push(pj);
            q_push(r - 1);
            return plus_record(a, perm, pi, pj, split ? 1 : 0);
        }
        return 0;
    }

    // ---- walker record and slots: HBM -> registers / shared memory
    __device__ __forceinline__ void load(const SegDesc &d, int64_t w) {
        const tfg_walker_info *H = d.hdr + w;
        R = d.R;
        const int rr = min(max(H->r, 0), R);   // in range whatever a restored state holds
        best_r = H->best_r;
        t = H->t; best_t = H->best_t;
        t_zero = t - H->plateau - 1;
        t_exp = t_zero + d.plateau_len;
        dig = H->digest; wid = H->walker_id;
        key0 = d.key0; key1 = d.key1;
        best_nnz = H->best_nnz;
        mk.load(d);
        c_acc = c_rej = c_drp = c_mrg = c_pls = c_red = 0;
        qlen = 0; q0 = q1 = q2 = 0;
        nnz = 0;
        if constexpr (!GM) {
            const Wd *src = reinterpret_cast<const Wd *>(d.slots) + (size_t)w * R * NWS;
#pragma unroll 4
            for (int k = 0; k < R; ++k) st(k, ld_at(src + (size_t)k * NWS));
        }
#pragma unroll 4
        for (int k = 0; k < R; ++k) {
            if constexpr (ROWS) row(k, 0) = row(k, 1) = row(k, 2) = 0u;
            else ix[k * kLane] = (uint32_t)k * 0x010101u;
        }
        if constexpr (CNT) {
            matches = 0;
            for (int k = 0; k < (R + 1) / 2; ++k) cn[k * kLane] = 0u;
        }
#pragma unroll
        for (int q = 0; q < 3 * kHashBits * NW; ++q) hs[q * kLane] = 0u;
        // the slots enter their classes one after another
#pragma unroll 1
        for (r = 1; r <= rr; ++r) {
            const T v = ld(r - 1);
            if (PG && d.walk_policy == 2) nnz += nnz_of(v);
#pragma unroll 1
            for (int f = 0; f < 3; ++f) relink(r - 1, f, v);
        }
        r = rr;
    }

    __device__ __forceinline__ void store(const SegDesc &d, int64_t w, uint32_t steps) {
        if constexpr (!GM) {   // GM: the slots were written in place
            Wd *dst = reinterpret_cast<Wd *>(d.slots) + (size_t)w * R * NWS;
#pragma unroll 4
            for (int k = 0; k < R; ++k) {
                const T v = ld(k);
                dst[(size_t)k * NWS] = v.p[0];
                if constexpr (ZT) dst[(size_t)k * NWS + 1] = v.n[0];
            }
        }
        tfg_walker_info *H = d.hdr + w;
        H->r = r; H->best_r = best_r;
        H->t = t; H->plateau = t - 1 - t_zero; H->best_t = best_t;
        H->digest = dig;
        H->accepted += c_acc; H->rejected += c_rej; H->nocand += steps - c_acc - c_rej;
        H->drops += c_drp; H->merges += c_mrg; H->plus += c_pls; H->reductions += c_red;
        H->best_nnz = best_nnz;
    }

    // plateau := 0 by the step at t
    __device__ __forceinline__ void restart(const SegDesc &d) {
        t_zero = t;
        t_exp = t + d.plateau_len;
    }

    // The sampled term of the next step, fetched ahead: its slot, its words and
    // its row / list entries.
    struct Sample {
        int i;
        T ti;
        uint32_t l[ROWS ? 3 : 1];
    };
    __device__ __forceinline__ void fetch(uint32_t x0, Sample &s) const {
        s.i = (int)__umulhi(x0, (uint32_t)r);
        s.ti = ld(s.i);
        if constexpr (ROWS) {
            s.l[0] = row(s.i, 0); s.l[1] = row(s.i, 1); s.l[2] = row(s.i, 2);
        } else {
            s.l[0] = ix[s.i * kLane];
        }
    }
    // Candidate classes of the sampled term: sizes, and (lists) how many members lie below it.
    struct Cand {
        int n0, n1, n2, b0, b1, b2;
    };
    __device__ __forceinline__ void candidates(const Sample &s, Cand &c) const {
        if constexpr (ROWS) {
            c.n0 = __popc(s.l[0]); c.n1 = __popc(s.l[1]); c.n2 = __popc(s.l[2]);
            c.b0 = c.b1 = c.b2 = 0;
        } else {
            const int i = s.i;
            int p0 = (int)(s.l[0] & 255u), p1 = (int)((s.l[0] >> 8) & 255u), p2 = (int)((s.l[0] >> 16) & 255u);
            c.n0 = c.n1 = c.n2 = c.b0 = c.b1 = c.b2 = 0;
#pragma unroll 1
            while ((p0 ^ i) | (p1 ^ i) | (p2 ^ i)) {
                if (p0 != i) { c.n0 += 1; c.b0 += p0 < i; p0 = next(p0, 0); }
                if (p1 != i) { c.n1 += 1; c.b1 += p1 < i; p1 = next(p1, 1); }
                if (p2 != i) { c.n2 += 1; c.b2 += p2 < i; p2 = next(p2, 2); }
            }
        }
    }
    // the idx-th (0-based) member, in ascending order, of the sampled term's class X without it
    __device__ __forceinline__ int member(const Sample &s, int X, int idx, const Cand &c) const {
        if constexpr (ROWS) {
            uint32_t y = X == 0 ? s.l[0] : (X == 1 ? s.l[1] : s.l[2]);
            int pos = 0, n = idx;
            // halving: skip the lower half when it holds at most n members
#pragma unroll
            for (int h = 16; h >= 1; h >>= 1) {
                const int k = __popc(y & ((1u << h) - 1u));
                const bool up = n >= k;
                n -= up ? k : 0;
                pos += up ? h : 0;
                y >>= up ? h : 0;
            }
            return pos;
        } else {
            const int n = X == 0 ? c.n0 : (X == 1 ? c.n1 : c.n2), b = X == 0 ? c.b0 : (X == 1 ? c.b1 : c.b2);
            // the cycle after i: the members above i, then those below
            int go = idx < b ? n - b + idx : idx - b;
            int p = (int)((s.l[0] >> (8 * X)) & 255u);
#pragma unroll 1
            for (; go > 0; --go) p = next(p, X);
            return p;
        }
    }
    // first non-zero of factor f (0, 1) of a made +1, w absorbing the sign; f = 2: nothing
    // (the other factors are normalised already)
    __device__ __forceinline__ void canon_factor(T &a, int f) const {
        if constexpr (ZT) {
            const Wd m = f == 0 ? mk.m[0][0] : (f == 1 ? mk.m[1][0] : Wd(0));
            const Wd dd = (a.p[0] | a.n[0]) & m;
            const Wd neg = (a.n[0] & dd & (Wd(0) - dd)) != Wd(0) ? (m | mk.m[2][0]) : Wd(0);
            const Wd sw = (a.p[0] ^ a.n[0]) & neg;
            a.p[0] ^= sw;
            a.n[0] ^= sw;
        }
    }

    // What a step did: the candidate it drew and what became of it.
    struct Step {
        int action, i, j, X, rho, sneg;
    };

    // ---- the flip (Section 3.3.1) of candidate (X, j, rho) on term i = s.i with the
    // ternary validity test; on acceptance the terms are normalised and stored,
    // zero terms are removed, and terms that may share a pair of factors with
    // another slot are queued for the cascade.
    __device__ __forceinline__ void flip(const T &ti, const T &tj, int policy, Step &s) {
        const int i = s.i, j = s.j, X = s.X;
        // (Y, Z) cyclic after X, rho swaps; Y_i += Y_j, Z_j -= s Z_i
        const int X1 = X == 2 ? 0 : X + 1, X2 = X == 0 ? 2 : X - 1;
        const int Y = s.rho ? X2 : X1, Z = s.rho ? X1 : X2;
        s.sneg = (ZT && X == 2) ? (int)(((ti.p[0] ^ tj.p[0]) & mk.m[2][0]) != Wd(0)) : 0;
        T ti2, tj2;
        bool ok = O::add(ti, tj, Y, false, mk, ti2);
        ok &= O::add(tj, ti, Z, s.sneg == 0, mk, tj2);
        s.action = ok ? kAccept : kReject;
        if (!ok) return;
        const bool zi = O::zero(ti2, Y, mk);
        const bool zj = O::zero(tj2, Z, mk);
        if (policy == 2) nnz += (zi ? 0u : nnz_of(ti2)) + (zj ? 0u : nnz_of(tj2)) - nnz_of(ti) - nnz_of(tj);
        canon_factor(ti2, Y);
        canon_factor(tj2, Z);
        st(i, ti2);
        st(j, tj2);
        // of the other factors the normalisation changes the sign of w at most
        uint32_t e1, e3;
        relink_pair<true>(i, Y, ti2, j, Z, tj2, e1, e3);
        if (zi || zj) {
            q_push(i);
            q_push(j);
            const int hi = i > j ? i : j, lo = i > j ? j : i;
            const bool zhi = (hi == i) ? zi : zj, zlo = (lo == i) ? zi : zj;
            if (zhi) { drop(hi); c_drp += 1; }
            if (zlo) { drop(lo); c_drp += 1; }
            if (policy == 2) qlen = 0;   // no reduction edges
        } else if (policy != 2) {
            // A third slot shares a pair with i' = (X_i, Y_i + Y_j, Z_i) iff it is in two of
            // its classes x, e1, z, and with j' = (X_j, Y_j, Z_j - s Z_i), X_j = +-X_i, iff in
            // two of x, e2, e3.  i' and j' share X and never another factor: that
            // would need Y_i = 0, or Z_j equal to 0 or to +-2 Z_i.
            if constexpr (ROWS) {
                const uint32_t cx = row(i, X) & ~(1u << j), cz = row(i, Z), e2 = row(j, Y);
                if ((cx & cz) | (e1 & (cx | cz)) | (e2 & (cx | e3)) | (cx & e3)) { q_push(i); q_push(j); }
            } else {
                // sets of members modulo 32 (a superset test: the cascade checks exactly)
                uint32_t cx = 0u, cz = 0u, a1 = 0u, a2 = 0u, a3 = 0u;
                int px = next(i, X), pz = next(i, Z), p1 = next(i, Y), p2 = next(j, Y), p3 = next(j, Z);
#pragma unroll 1
                while ((px ^ i) | (pz ^ i) | (p1 ^ i) | (p2 ^ j) | (p3 ^ j)) {
                    if (px != i) { cx |= px != j ? 1u << (px & 31) : 0u; px = next(px, X); }
                    if (pz != i) { cz |= 1u << (pz & 31); pz = next(pz, Z); }
                    if (p1 != i) { a1 |= 1u << (p1 & 31); p1 = next(p1, Y); }
                    if (p2 != j) { a2 |= 1u << (p2 & 31); p2 = next(p2, Y); }
                    if (p3 != j) { a3 |= 1u << (p3 & 31); p3 = next(p3, Z); }
                }
                if ((cx & cz) | (a1 & (cx | cz)) | (a2 & (cx | a3)) | (cx & a3)) { q_push(i); q_push(j); }
            }
        }
    }

    // ---- rest of a step, warp-converged, after the cascade of its flip: digest, best
    // scheme, plateau, expansion (and its cascade).  x2, x3: the step's third and
    // fourth draw.  Returns whether any lane's scheme changed here.
    __device__ __forceinline__ bool finish(const SegDesc &d, unsigned wmask, int lane, int nl, Wd *bestp, int policy,
                                           uint32_t x2, uint32_t x3, const Step &s) {
        dig = digest_mix(dig, ((uint64_t)((uint32_t)r << 8) << 32) |
                                  ((uint32_t)s.action | ((uint32_t)s.X << 4) | ((uint32_t)s.rho << 6) |
                                   ((uint32_t)s.sneg << 7) | ((uint32_t)s.i << 8) | ((uint32_t)s.j << 24)));
        // walk policy 1: a failed try_flip expands and ends the step (no best update)
        const bool failed = policy == 1 && s.action != kAccept;
        // the best scheme is the one of least rank (policy 2: least (rank, non-zero coefficients))
        const bool better = !failed && (r < best_r || (policy == 2 && r == best_r && nnz < best_nnz));
        const bool again = !failed && r == best_r && (policy != 2 || nnz == best_nnz) && x2 < d.refresh_thresh;
        bool expand;
        if (policy == 0) expand = t >= t_exp;   // and more, below
        else if (policy == 1) expand = failed || x3 < d.expand_thresh;
        else expand = false;
        if (!__any_sync(wmask, better | again | expand)) return false;
        if (better) {
            best_r = r;
            if (policy == 2) best_nnz = nnz;
            best_t = t;
            restart(d);
        }
        coop_snapshot(wmask, lane, nl, better | again, bestp);
        if (policy == 0) expand = d.plus_enabled && t >= t_exp;
        expand = expand && r < R && r >= 2 && (failed || r <= best_r + 2);
        if (!__any_sync(wmask, expand)) return false;
        uint64_t rec = 0;
        if (expand) rec = plus_setup(d);
        cascade_all(wmask);
        if (rec) dig = digest_mix(dig, rec | ((uint64_t)(uint32_t)r << 44));
        return true;
    }

    // wmask: walker_lanes
    __device__ __forceinline__ void run(const SegDesc &d, int64_t w, unsigned wmask, int32_t steps) {
        load(d, w);
        __syncwarp(wmask);
        Wd *bestp = reinterpret_cast<Wd *>(d.best) + (size_t)w * R * NWS;
        const int lane = threadIdx.x & 31;
        const int nl = __popc(wmask);
        const int policy = PG ? d.walk_policy : 0;
        U4 x = philox10((uint32_t)t, (uint32_t)(t >> 32), wid, 0u, key0, key1);
        Sample s;
        fetch(x.x, s);
#pragma unroll 1
        for (int32_t step = 0; step < steps; ++step) {
            const int64_t tn = t + 1;
            const U4 xn = philox10((uint32_t)tn, (uint32_t)(tn >> 32), wid, 0u, key0, key1);   // the next step's draws
            // ---- try_flip (Algorithm 1): candidates X_j = +-X_i, ordered (X, slot, rho)
            const int r_before = r;
            Step did{kNoCand, s.i, 0, 0, 0, 0};
            Cand c;
            candidates(s, c);
            const int n01 = c.n0 + c.n1, K = 2 * (n01 + c.n2);
            if (K > 0) {
                const int ch = (int)__umulhi(x.y, (uint32_t)K);
                did.rho = ch & 1;
                const int mi = ch >> 1;
                const int X = (int)(mi >= c.n0) + (int)(mi >= n01);
                did.X = X;
                did.j = member(s, X, mi - (X == 0 ? 0 : (X == 1 ? c.n0 : n01)), c);
                flip(s.ti, ld(did.j), policy, did);
            }
            c_acc += did.action == kAccept;
            c_rej += did.action == kReject;
            cascade_all(wmask);
            // ---- the next step's term, unless this one still expands
            fetch(xn.x, s);
            c_red += r < r_before;
            if (finish(d, wmask, lane, nl, bestp, policy, x.z, x.w, did)) fetch(xn.x, s);
            x = xn;
            t = tn;
        }
        store(d, w, (uint32_t)steps);
    }
};

// Rows of a thread's warp in shared memory: terms (unless in device memory), classes,
// counts, slices.
template <class LW, class Wd>
__device__ __forceinline__ void link_rows(LW &wk, const SegDesc &d, int64_t w, bool in_device, unsigned char *smem) {
    const int lane = threadIdx.x & 31;
    unsigned char *at = smem + (size_t)(threadIdx.x >> 5) * (LW::thread_bytes(d.R) * 32);
    if (in_device) {
        wk.sm = reinterpret_cast<Wd *>(d.slots) + (size_t)w * d.R * LW::NWS;
    } else {
        wk.sm = reinterpret_cast<Wd *>(at) + lane * LW::NWS;
        at += (size_t)d.R * 32 * LW::NWS * sizeof(Wd);
    }
    wk.ix = reinterpret_cast<uint32_t *>(at) + lane;
    uint32_t *after = wk.ix + (size_t)d.R * 32 * (LW::ROWS ? 3 : 1);
    wk.cn = after;
    wk.hs = after + (LW::kCounts ? (size_t)(d.R + 1) / 2 * 32 : (size_t)0);
}

// Blocks of any whole number of warps (kLinkMaxBlock threads at most): a warp's
// rows are its own.
constexpr int kLinkMaxBlock = 160;
template <int MODE, class Wd, int NW, bool GM, bool PG, bool LIST = false>
__global__ void __launch_bounds__(kLinkMaxBlock, 3) walk_link_kernel(const SegDesc d, const int32_t steps) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned wmask = walker_lanes(d, w);
    if (w >= d.n_walkers) return;   // no block-wide barrier is used
    using LW = LinkWalker<MODE, Wd, NW, GM, PG, false, LIST>;
    LW wk;
    link_rows<LW, Wd>(wk, d, w, GM, smem_raw);
    wk.run(d, w, wmask, steps);
}

}  // namespace dev

constexpr int kLinkSmem = 227 * 1024;   // shared memory of an SM's blocks

template <int MODE, class Wd, int NW>
void prepare_walk_link() {
    static bool attr = [] {
        auto set = [](auto kernel) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinkSmem);
        };
        set(dev::walk_link_kernel<MODE, Wd, NW, false, false>);
        set(dev::walk_link_kernel<MODE, Wd, NW, false, true>);
        if constexpr (NW == 1 && sizeof(Wd) == 4) {
            set(dev::walk_link_kernel<MODE, Wd, NW, false, false, true>);
            set(dev::walk_link_kernel<MODE, Wd, NW, false, true, true>);
        }
        if constexpr (sizeof(Wd) == 8) {
            set(dev::walk_link_kernel<MODE, Wd, NW, true, false>);
            set(dev::walk_link_kernel<MODE, Wd, NW, true, true>);
        }
        return true;
    }();
    (void)attr;
}

// Where the packed terms sit.  A term of 64-bit words takes 16 bytes a slot (Z_T), four
// times the slot's list entry, so keeping the terms in the walker's device-memory
// slots lets about three times as many walkers reside on an SM; a step then waits
// for two or three reads from L2.  Steps are bound by latency, so the terms go to
// shared memory exactly when the whole population resides at once that way.
// Measured, Z_T, shared / device memory, steps/s: (2,4,5) 20165 walkers (all
// resident) 9.2e9 / 7.0e9; (3,3,4) 40330 walkers (1.1 times what fits) 1.02e10 /
// 1.24e10; (4,4,5) 80660 walkers (4.5 times) 5.3e9 / 9.5e9.  32-bit terms (at
// most 32 slots of 8 bytes) always go to shared memory.
// Blocks an SM's shared memory holds (1 KB a block is the system's), over all SMs
inline int64_t link_resident(size_t block_bytes) {
    return (int64_t)sm_count() * (int64_t)(kLinkSmem / (block_bytes + 1024));
}
inline bool link_terms_shared(size_t block_bytes, int64_t grid) {
    return block_bytes <= (size_t)kLinkSmem && grid <= link_resident(block_bytes);
}

// Launch shape of a class walker and the place of its terms (thread_bytes with the terms in
// shared / device memory; device 0: shared only).  A population too small to fill the
// GPU takes blocks of one warp with walkers in few lanes (walk_lanes), as many warps as
// reside at once; their columns are a full warp's.  Terms in device memory leave
// room for more warps, which outweighs the reads from L2 when that means a quarter of
// the lanes, eight at most: (4,4,5), 500 steps, shared / device, 2048 walkers 0.99 (8 lanes)
// / 0.82 (2), 4096 1.17 (16) / 1.19 (4), 10000 1.36 (32) / 1.75 (16).
struct LinkShape {
    int grid, block;
    bool shared;
    size_t smem;
};
inline LinkShape link_shape(const SegDesc &d, int block, size_t shared_bytes, size_t device_bytes) {
    auto blocks = [&](int walkers) { return (int)((d.n_walkers + walkers - 1) / walkers); };
    auto lanes = [&](size_t bytes) {
        return walk_lanes(d, std::min(spread_warps(d), link_resident(32 * bytes)));
    };
    const int ls = lanes(shared_bytes), lg = device_bytes ? lanes(device_bytes) : 32;
    const bool spread_device = 4 * lg <= ls && ls <= 8;
    const bool shared = device_bytes == 0 ||
                        (!spread_device && (ls < 32 || link_terms_shared(shared_bytes * block, (d.population + block - 1) / block)));
    const int l = shared ? ls : lg;
    const size_t bytes = shared ? shared_bytes : device_bytes;
    if (l == 32) return {blocks(block), block, shared, bytes * block};
    return {blocks(l), l, shared, bytes * 32};
}

// At most 32 slots: classes as rows (12 bytes a slot) or as lists (4).  A row is read at
// once, a list member by member, so rows are the faster where as many walkers reside;
// lists let up to twice as many (16 warps an SM, by their registers), and pay when rows
// need half as many waves of blocks again, under policy 1 twice as many.  Not
// where a factor is so short that many slots share it (lists grow long): at least
// six coefficients.  Measured, rows / lists, ms per 1000 steps: (2,3,4) 20000 walkers (one
// wave) Z_T 1.55 / 1.81, 65536 (two / one) Z_T 3.03 / 2.52, Z_2 3.82 / 2.81, 131072 (three /
// two) Z_T 4.79 / 4.46, Z_2 5.84 / 5.07, policy 1 Z_T 100000 (three / two) 7.0 / 7.9, 65536
// Z_2 (two / one) 12.0 / 10.1, policy 2 Z_T 65536 3.13 / 2.20; (2,3,3) 65536 Z_T (two /
// one) 2.79 / 2.32, 262144 (five / four) 7.3 / 7.8; (2,2,6) Z_T 65536 (two / one) 3.16 /
// 3.17, 131072 (three / two) 5.02 / 5.62.
inline bool link_lists_pay(const SegDesc &d, size_t rows_bytes, size_t lists_bytes, int block) {
    const int64_t grid = (d.population + block - 1) / block;
    const int shortest = std::min(d.m * d.n, std::min(d.n * d.p, d.p * d.m));
    if (shortest < 6) return false;
    auto waves = [&](size_t bytes) {   // of at most 16 warps an SM
        const size_t room = std::max(bytes, (size_t)kLinkSmem / (512 / block) - 1024);
        return (grid + link_resident(room) - 1) / std::max<int64_t>(link_resident(room), 1);
    };
    const int64_t rows = waves(rows_bytes), lists = waves(lists_bytes);
    return d.walk_policy == 1 ? rows >= 2 * lists : 2 * rows >= 3 * lists;
}

struct LinkPlan {
    LinkShape k;
    bool lists;   // at most 32 slots: classes as lists
};
template <int MODE, class Wd, int NW>
LinkPlan link_plan(const SegDesc &d, int block) {
    using Shared = dev::LinkWalker<MODE, Wd, NW, false, false>;
    using Device = dev::LinkWalker<MODE, Wd, NW, true, false>;
    const LinkShape k = link_shape(d, block, Shared::thread_bytes(d.R),
                                   sizeof(Wd) == 8 ? Device::thread_bytes(d.R) : (size_t)0);
    if constexpr (NW == 1 && sizeof(Wd) == 4) {
        const size_t lists = dev::LinkWalker<MODE, Wd, NW, false, false, false, true>::thread_bytes(d.R) * block;
        if (k.block == block && link_lists_pay(d, k.smem, lists, block)) return {{k.grid, block, true, lists}, true};
    }
    return {k, false};
}
template <int MODE, class Wd, int NW>
LaunchShape link_launch_shape(const SegDesc &d, int block) {
    const LinkShape k = link_plan<MODE, Wd, NW>(d, block).k;
    return {1, k.block, k.grid};
}

template <int MODE, class Wd, int NW>
void launch_walk_link(const SegDesc &d, int32_t steps, int /*grid*/, int block, cudaStream_t st) {
    prepare_walk_link<MODE, Wd, NW>();
    const LinkPlan plan = link_plan<MODE, Wd, NW>(d, block);
    const LinkShape &k = plan.k;
    if constexpr (NW == 1 && sizeof(Wd) == 4) {
        if (plan.lists) {
            if (d.walk_policy == 0)
                dev::walk_link_kernel<MODE, Wd, NW, false, false, true><<<k.grid, k.block, k.smem, st>>>(d, steps);
            else
                dev::walk_link_kernel<MODE, Wd, NW, false, true, true><<<k.grid, k.block, k.smem, st>>>(d, steps);
            return;
        }
    }
    if (k.shared) {
        if (d.walk_policy == 0) dev::walk_link_kernel<MODE, Wd, NW, false, false><<<k.grid, k.block, k.smem, st>>>(d, steps);
        else dev::walk_link_kernel<MODE, Wd, NW, false, true><<<k.grid, k.block, k.smem, st>>>(d, steps);
    } else if constexpr (sizeof(Wd) == 8) {
        if (d.walk_policy == 0) dev::walk_link_kernel<MODE, Wd, NW, true, false><<<k.grid, k.block, k.smem, st>>>(d, steps);
        else dev::walk_link_kernel<MODE, Wd, NW, true, true><<<k.grid, k.block, k.smem, st>>>(d, steps);
    }
}

}  // namespace tfg
