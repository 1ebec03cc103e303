// sssp_small.cuh -- the kernel that runs a single query's small rounds (Garg,
// arXiv 1812.10499, Sec. V-VI) back to back in one thread-block cluster.
//
// A round whose frontier and active set hold a few thousand vertices is not
// bound by bandwidth or arithmetic but by the chain of instructions and memory
// round trips from one phase to the next.  This kernel shortens that chain:
//   - The work lists live in the CTAs' shared memory.  An active vertex stays
//     in one CTA's list, with its edge ranges and outWeight, until it is fixed;
//     a newly discovered vertex is written into the list of a CTA chosen by a
//     hash of its id, through distributed shared memory (230 cycles, where a
//     global counter takes 350-760).  No global counter, list or offset array
//     is read between the phases.
//   - A list entry is handled by a group of lanes (as many as the length of
//     the list allows), so that a round's few vertices spread over all warps
//     and an entry's edges are read side by side; a larger entry is read by its
//     whole warp, a very large one by its whole CTA.
//   - The minima (Lemmas 7 and 8) and the counts that end a round travel with
//     the cluster barrier: each CTA writes one slot into every other CTA's
//     shared memory before it arrives.
// Per round there are two such barriers (450 cycles each, 1000 with stores to
// complete): after the lower bounds and fixing (steps (b), (c)) and after the
// relaxation (step (a)) of the fixed vertices.  Global memory holds what the
// rounds of the other kernels hold, except the work lists and the control
// block, which are written when the kernel hands over (or the query ends).
//
// Measured (GB300, 2070 MHz) against k_tail, which keeps its lists in global
// memory and gives a warp 32 vertices: 1024 x 1024 weighted grid 13.4 -> 6.4 us
// a round, unit grid 2001 x 1500 13.0 -> 6.7; a solve of random n = 4096 (26 rounds)
// 389 -> 199 us.
// 512 threads per CTA: 256 are 5-8% slower (two passes over the lists), 1024
// 25% (barriers).
#pragma once
#include "sssp_round.cuh"

namespace sssp {

constexpr u32 kSmallCTAs = kTailCTAs;
constexpr u32 kSmallThreads = 512;
constexpr u32 kSmallWarps = kSmallThreads / 32;
constexpr u32 kSmallCap = 1024;      // entries of a CTA's active list, and of its frontier
static_assert(kSmallEntries == kSmallCTAs * (kSmallCap * 3 / 4),
              "a quarter of a list is left for the vertices that a round discovers");
// Edges in flight per lane.  1: random n = 4096 and R-MAT tails 7-17% slower
// (degrees above the group's lanes); 4: grids 7% slower (empty slots).
constexpr u32 kSmallU = 2;
constexpr u32 kGroupDeg = 32;        // entries up to this are always read by their group
constexpr u32 kCtaDeg = 512;         // entries above are read by the whole CTA ...
constexpr u32 kBigCap = 64;          // ... up to this many, the rest by their warps

struct __align__(16) ActEntry {      // an active vertex
    u32 g, deg;                      // record (= vertex) id, in-degree
    u64 ib, ob;                      // first in-edge, first out-edge
    u32 odeg, ow;                    // out-degree, outWeight (kNoOutW: none)
};
struct __align__(16) FrontEntry {    // a vertex to relax
    u32 g, deg;                      // bit 31 of g: kFixedEntry, fixed in the last round
    u64 ob;                          // first out-edge
};
constexpr u32 kFixedEntry = 1u << 31;
constexpr u64 kLiveEntry = 1ull << 63;   // in ob: the vertex relaxes (not only fixed)

// What one CTA tells the others at a barrier.
struct __align__(16) SmallSlot {
    u64 minD, thr;                   // after the relaxation
    u32 nfront, nact;                // list entries it added in the phase
    u32 chunks, nfix;                // hub chunks among its entries; vertices fixed
    u32 flags, pad[3];               // 1: a list overflowed, 2: the target is fixed
};

// The CTA's counts that a decided vertex adds to: entries of the two active lists,
// frontier entries, those that relax, those fixed.
enum : u32 { kActive0 = 0, kActive1 = 1, kFront = 2, kLive = 3, kNewFixed = 4, kCounts = 5 };

struct SmallShared {
    ActEntry act[2][kSmallCap];
    FrontEntry fr[kSmallCap];
    u64 fdist[kSmallCap];            // distance a frontier entry relaxes with
    SmallSlot xa[kSmallCTAs], xb[kSmallCTAs];
    u64 wd[kSmallWarps], wt[kSmallWarps];      // the warps' folds ...
    u32 wpush[kSmallWarps], wchunk[kSmallWarps];   // ... and discoveries
    u64 bigmin;
    u32 big[kBigCap];                // entries for the whole CTA
    u32 cnt[kCounts];
    u32 nbig, chunks, fchunks, flags;
};

// --------------------------------------------------- distributed shared memory

__device__ __forceinline__ u32 map_cta(u32 addr, u32 cta) {
    u32 r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(cta));
    return r;
}
__device__ __forceinline__ u32 dsm_add(u32 addr, u32 v) {
    u32 r;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;\n"
                 : "=r"(r)
                 : "r"(addr), "r"(v)
                 : "memory");
    return r;
}
__device__ __forceinline__ void dsm_st4(u32 addr, u32 a, u32 b, u32 c, u32 d) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(a), "r"(b),
                 "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
}

// Barrier of the cluster; the aligned form needs converged warps.
__device__ __forceinline__ void small_sync() {
    __syncwarp();
    cluster_sync_all();
}

// ------------------------------------------------------------------ layouts

// State access of the two layouts.  Records, filter words and change marks are
// written by other CTAs during the kernel, so they are read from L2.
struct SmallWide {
    typedef VRec Rec;
    typedef u64 Dist;
    static constexpr bool kNarrow = false;
    static constexpr u64 kInf = kInf64;
    static constexpr u64 kTermInf = kInf64;
    __device__ static Rec* rec(const RoundParams& P) { return P.rec; }
    __device__ static u32 shift(const RoundParams& P) { return P.vbits; }
    __device__ static Dist none(const RoundParams& P) { return P.dinf; }
    __device__ static Dist clip(u64 v) { return v; }
    struct Nbr {
        u64 d, c;
    };
    __device__ static Nbr load(const Rec* p, u32 cur) {
        return Nbr{__ldcg(&p->dp), __ldcg(&p->cf[cur])};
    }
    __device__ static Dist term(const RoundParams& P, const Nbr& s, u32 w, Dist thr, Dist minD) {
        const u64 d = s.d >> P.vbits, c = s.c & kCMask;
        u64 lb;
        if (P.rule == 0) lb = umax64(c, umin64(d, thr));
        else lb = (s.c & kFixed) ? c : umax64(c, minD);
        return umin64(lb + w, P.dinf);
    }
    __device__ static void own(const RoundParams& P, const Nbr& s, Dist& d, Dist& c) {
        d = s.d >> P.vbits;
        c = s.c & kCMask;
    }
    __device__ static void set_c(Rec* p, u32 slot, Dist c, bool fixed) {
        p->cf[slot] = c | (fixed ? kFixed : 0ull);
    }
    __device__ static Dist fixed_dist(const Rec* p, u32 cur) {
        return __ldcg(&p->cf[cur]) & kCMask;
    }
    __device__ static Dist wmin(Dist v) { return warp_min64(v); }
    // A relaxation target: open (not fixed), its packed D, outWeight, in-degree.
    struct Tgt {
        u64 d, c;
        u32 outw, indeg;
    };
    __device__ static Tgt target(const RoundParams&, const Rec* p, u32 cur) {
        const ulonglong2 lo = __ldcg(reinterpret_cast<const ulonglong2*>(p));
        const ulonglong2 hi = __ldcg(reinterpret_cast<const ulonglong2*>(p) + 1);
        return Tgt{lo.x, cur ? hi.x : lo.y, (u32)hi.y, (u32)(hi.y >> 32)};
    }
    __device__ static bool open(const Tgt& t) { return (t.c & kFixed) == 0; }
};
struct SmallNarrow {
    typedef VRecN Rec;
    typedef u32 Dist;
    static constexpr bool kNarrow = true;
    static constexpr u32 kInf = kFull;
    static constexpr u32 kTermInf = kInf31;
    __device__ static Rec* rec(const RoundParams& P) { return P.recn; }
    __device__ static u32 shift(const RoundParams&) { return 32u; }
    __device__ static Dist none(const RoundParams&) { return kFull; }
    __device__ static Dist clip(u64 v) { return v < kFull ? (u32)v : kFull; }
    struct Nbr {
        u32 d, c;
    };
    __device__ static Nbr load(const Rec* p, u32 cur) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p));
        return Nbr{v.y, cur ? v.w : v.z};
    }
    __device__ static Dist term(const RoundParams& P, const Nbr& s, u32 w, Dist thr, Dist minD) {
        const u32 c = s.c & ~kFixedN;
        u32 lb;
        if (P.rule == 0) lb = max(c, min(s.d, min(thr, kInf31)));
        else lb = (s.c & kFixedN) ? c : max(c, min(minD, kInf31));
        return min(lb + w, kInf31);
    }
    __device__ static void own(const RoundParams&, const Nbr& s, Dist& d, Dist& c) {
        d = s.d;
        c = s.c & ~kFixedN;
    }
    __device__ static void set_c(Rec* p, u32 slot, Dist c, bool fixed) {
        p->cf[slot] = c | (fixed ? kFixedN : 0u);
    }
    __device__ static Dist fixed_dist(const Rec* p, u32 cur) {
        return __ldcg(&p->cf[cur]) & ~kFixedN;
    }
    __device__ static Dist wmin(Dist v) { return __reduce_min_sync(kFull, v); }
    struct Tgt {
        u64 d;
        u32 c;
    };
    __device__ static Tgt target(const RoundParams&, const Rec* p, u32 cur) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p));
        return Tgt{((u64)v.y << 32) | v.x, cur ? v.w : v.z};
    }
    __device__ static bool open(const Tgt& t) { return (t.c & kFixedN) == 0; }
};

// outWeight word of the compact layout without its in-hub flag.
__device__ __forceinline__ u32 plain_outw(u32 packed) {
    const u32 w = packed & kInf31;
    return w == kInf31 ? kNoOutW : w;
}

// ------------------------------------------------------------------ relaxation

// What a thread carries through the rounds.
template <class S>
struct SmallAcc {
    typename S::Dist fd, ft;             // folds of D and D + outWeight
    u32 pushed, chunks;                  // discoveries of the phase, their hub chunks
    u64 out, in, act, front;             // work counters
};

// A full list: the vertex goes to the global list, and the cluster hands the
// round over at the next barrier.
static __device__ __noinline__ void push_overflow(const RoundParams& P, u32* flags, u32 cur, u32 y,
                                                  u32 deg) {
    if (deg > P.hub) put_hub(P, &P.ctl->AHpk[cur], P.L.AH[cur], P.L.AC[cur], y, deg);
    else put_small(P, P.L.AS[cur], atomicAdd(&P.ctl->nAS[cur], 1u), y);
    atomicOr(flags, 1u);
}

// Relaxes kSmallU edges per lane, out of one frontier vertex per lane (id x,
// distance dx): targets, atomics, discoveries, in three waves of loads.  Only
// the first nu (warp-uniform) of the U edges are looked at.
template <class S, bool WIN>
__device__ __forceinline__ void small_relax(const RoundParams& P, SmallShared& s, u32 p, u32 cur,
                                            const uint2 (&e)[kSmallU], bool (&ev)[kSmallU],
                                            typename S::Dist dx, u32 x, u32 nu, SmallAcc<S>& a) {
    typedef typename S::Dist Dist;
    constexpr u32 U = kSmallU;
    typename S::Rec* rec = S::rec(P);
    u32 ow[U];
    bool ok[U], unseen[U];
    if (S::kNarrow && !WIN && P.gf) {
        uint2 fw[U];
#pragma unroll
        for (u32 i = 0; i < U; ++i) {
            fw[i] = make_uint2(0u, 0u);
            if (i < nu && ev[i]) fw[i] = __ldcg(P.gf + e[i].x);
        }
#pragma unroll
        for (u32 i = 0; i < U; ++i) {
            ok[i] = false;
            if (i >= nu) break;
            ok[i] = ev[i] && dx + e[i].y <= fw[i].x;
            unseen[i] = ok[i] && fw[i].x == kRelaxUnseen;
            ow[i] = plain_outw(fw[i].y);
        }
    } else {
        typename S::Tgt t[U];
        u32 w[U];
#pragma unroll
        for (u32 i = 0; i < U; ++i) {
            w[i] = 0;
            if (i < nu && ev[i]) {
                t[i] = S::target(P, rec + e[i].x, cur);
                if constexpr (S::kNarrow) w[i] = __ldg(P.g.outw + e[i].x);
            }
        }
#pragma unroll
        for (u32 i = 0; i < U; ++i) {
            ok[i] = false;
            if (i >= nu) break;
            const u64 cand = ((u64)(dx + e[i].y) << S::shift(P)) | x;
            ok[i] = ev[i] && S::open(t[i]) && cand < t[i].d;
            unseen[i] = ok[i] && t[i].d == kInf64;
            if constexpr (S::kNarrow) ow[i] = plain_outw(w[i]);
            else ow[i] = t[i].outw;
            // D changes this round (to at most cand): it must relax again.
            if (WIN && ok[i]) P.chg[e[i].x] = 1u;
        }
    }
    // The edge ranges of a vertex that may be new are loaded beside the atomic
    // that tells.
    u64 old[U], i0[U], o0[U];
    u32 id[U], od[U];
#pragma unroll
    for (u32 i = 0; i < U; ++i) {
        old[i] = 0;
        if (i < nu && ok[i]) {
            const Dist dd = dx + e[i].y;
            const u64 cand = ((u64)dd << S::shift(P)) | x;
            if (unseen[i]) {
                old[i] = atomicMin(&rec[e[i].x].dp, cand);
                i0[i] = __ldg(P.g.in_off + e[i].x);
                id[i] = (u32)(__ldg(P.g.in_off + e[i].x + 1) - i0[i]);
                o0[i] = __ldg(P.g.out_off + e[i].x);
                od[i] = (u32)(__ldg(P.g.out_off + e[i].x + 1) - o0[i]);
            } else {
                atomicMin(&rec[e[i].x].dp, cand);
            }
            const Dist t = ow[i] == kNoOutW ? S::none(P) : dd + ow[i];
            a.fd = dd < a.fd ? dd : a.fd;
            a.ft = t < a.ft ? t : a.ft;
        }
    }
#pragma unroll
    for (u32 i = 0; i < U; ++i) {
        if (i >= nu) break;
        if (old[i] != kInf64) continue;
        // Newly discovered: it joins the active list of one CTA.
        const u32 y = e[i].x;
        const u32 cta = (y * 0x9E3779B1u) >> 28;
        static_assert(kSmallCTAs == 16, "the owner is the hash's upper 4 bits");
        const u32 pos = dsm_add(map_cta(smem_addr(&s.cnt[p]), cta), 1u);
        // Its edges are read from the next phase on.  (It has an in-edge; a vertex
        // without out-edges may stand at the very end of the array.)
        prefetch_l2(P.g.in_adj + i0[i]);
        if (od[i]) prefetch_l2(P.g.out_adj + o0[i]);
        ++a.pushed;
        if (id[i] > P.hub) a.chunks += (id[i] + P.chunk - 1) / P.chunk;
        if (pos < kSmallCap) {
            const u32 at = map_cta(smem_addr(&s.act[p][pos]), cta);
            dsm_st4(at, y, id[i], (u32)i0[i], (u32)(i0[i] >> 32));
            dsm_st4(at + 16, (u32)o0[i], (u32)(o0[i] >> 32), od[i], ow[i]);
        } else {
            push_overflow(P, &s.flags, cur, y, id[i]);
        }
    }
}

// Lanes per list entry (as a power of two): as many as the CTA's threads
// allow for n entries, at most 16.
__device__ __forceinline__ u32 group_shift(u32 n) {
    constexpr u32 lt = 9;
    static_assert(kSmallThreads == 1u << lt, "");
    const u32 ln = n > 1 ? 32u - __clz(n - 1) : 0u;      // log2, rounded up
    return ln >= lt ? 0u : min(4u, lt - ln);
}

// Hands a list entry to the whole CTA, if its list of such entries has room.
__device__ __forceinline__ bool take_big(SmallShared& s, u32 idx) {
    const u32 k = atomicAdd(&s.nbig, 1u);
    if (k < kBigCap) s.big[k] = idx;
    return k < kBigCap;
}

// Step (a): the CTA's frontier.  One loop serves the three ways an entry is
// read (its group of lanes, its warp, the CTA): the phases' code has to stay
// in the instruction caches, because each round runs through all of it.
template <class S, bool WIN>
__device__ __forceinline__ void small_phase_relax(const RoundParams& P, SmallShared& s, u32 p,
                                                  u32 cur, u32 lane, u32 wib, SmallAcc<S>& a) {
    typedef typename S::Dist Dist;
    constexpr u32 U = kSmallU;
    const u32 n = s.cnt[kFront];
    const u32 gs = group_shift(n), sub = lane & ((1u << gs) - 1u);
    const u32 lim = max(kGroupDeg, (4 * U) << gs);
    typename S::Rec* rec = S::rec(P);
    u32 base = wib << (5 - gs), b = 0, nb = 0;
    bool tiles = true;
    for (;;) {
        const uint2* adj;
        u32 x, deg, len, k, step, todo = 0;
        Dist dx;
        if (tiles) {
            if (base >= n) {
                tiles = false;
                __syncthreads();
                nb = min(s.nbig, kBigCap);
                continue;
            }
            const u32 idx = base + (lane >> gs);
            base += kSmallWarps << (5 - gs);
            FrontEntry f = {0, 0, 0};
            dx = 0;
            if (idx < n) {
                f = s.fr[idx];
                dx = (Dist)s.fdist[idx];
            }
            x = f.g & ~kFixedEntry;
            deg = f.deg;
            adj = P.g.out_adj + (f.ob & ~kLiveEntry);
            bool cta = false;
            if (idx < n && sub == 0) {
                // The word of the other parity becomes "fixed" too.
                if (f.g & kFixedEntry) S::set_c(rec + x, cur ^ 1u, dx, true);
                a.out += deg;
                if (deg > kCtaDeg) cta = take_big(s, idx);
            }
            len = deg <= lim ? deg : 0u;
            k = sub;
            step = 1u << gs;
            todo = __ballot_sync(kFull, sub == 0 && deg > lim && !cta);
        } else {
            if (b >= nb) break;
            const FrontEntry f = s.fr[s.big[b]];
            dx = (Dist)s.fdist[s.big[b]];
            ++b;
            x = f.g & ~kFixedEntry;
            deg = len = f.deg;
            adj = P.g.out_adj + (f.ob & ~kLiveEntry);
            k = threadIdx.x;
            step = kSmallThreads;
        }
        const uint2* adj0 = adj;
        const u32 x0 = x;
        const Dist dx0 = dx;
        for (;;) {
#pragma unroll 1
            for (; __any_sync(kFull, k < len); k += step * U) {
                uint2 e[U];
                bool ev[U];
                // A second edge per lane only where some lane has one: the
                // instructions of an empty slot cost 0.2 us a phase.
                const u32 nu = __any_sync(kFull, k + step < len) ? U : 1u;
#pragma unroll
                for (u32 i = 0; i < U; ++i) {
                    ev[i] = k + i * step < len;
                    e[i] = make_uint2(0u, 0u);
                    if (ev[i]) e[i] = __ldg(adj + k + i * step);
                }
                small_relax<S, WIN>(P, s, p, cur, e, ev, dx, x, nu, a);
            }
            if (todo == 0) break;
            // The next larger entry of the tile, by the whole warp.
            const u32 own = __ffs(todo) - 1;
            todo &= todo - 1;
            adj = reinterpret_cast<const uint2*>(__shfl_sync(kFull, (u64)adj0, own));
            x = __shfl_sync(kFull, x0, own);
            dx = __shfl_sync(kFull, dx0, own);
            len = __shfl_sync(kFull, deg, own);
            k = lane;
            step = 32;
        }
    }
}

// ---------------------------------------------------------- lower bounds, fixing

// Decides one active vertex (all lanes of the warp; `in`: this lane holds a
// vertex): its new lower bound, and its entry in the next lists.
template <class S, bool WIN>
__device__ __forceinline__ void small_decide(const RoundParams& P, SmallShared& s, u32 q, u32 r,
                                             bool in, bool fix_now, const ActEntry& en,
                                             typename S::Dist dy, typename S::Dist cy,
                                             typename S::Dist m, typename S::Dist thr,
                                             typename S::Dist minD, u32 target, u32 lane,
                                             SmallAcc<S>& a) {
    typedef typename S::Dist Dist;
    const u32 cur = r & 1u, nxt = cur ^ 1u;
    typename S::Rec* rec = S::rec(P);
    bool fix = false;
    if (in) {
        Dist cn = dy;
        if (fix_now) {
            fix = true;
        } else {
            const Dist self = (P.rule == 0) ? max(cy, min(dy, thr)) : max(cy, minD);
            cn = max(self, m);
            fix = cn == dy || (P.rule == 1 && dy <= thr);
            if (fix) cn = dy;
        }
        S::set_c(rec + en.g, nxt, cn, fix);
        if (fix) P.fround[en.g] = (int)r;
        if (S::kNarrow && !WIN && P.gf) P.gf[en.g].x = fix ? 0u : (u32)dy;
        if (fix && en.g == target) atomicOr(&s.flags, 2u);
    }
    // Windowed: the frontier is the fixed vertices and, while D < minD +
    // delta, the survivors, each only if its D changed since it last relaxed.
    bool fx = fix;
    const bool sv = in && !fix;
    if (WIN) {
        fx = false;
        if (in && (fix || (u64)dy < win_limit((u64)minD, P.delta))) {
            fx = __ldcg(P.chg + en.g) != 0;
            if (fx) {
                P.chg[en.g] = 0;
                P.snap[en.g] = dy;
            }
        }
    }
    const bool fl = fx || fix;                 // a windowed fixed vertex may have nothing to relax
    const u32 below = (1u << lane) - 1u;
    const u32 ms = __ballot_sync(kFull, sv), mf = __ballot_sync(kFull, fl);
    const u32 mx = WIN ? __ballot_sync(kFull, fx) : mf;
    const u32 mfix = WIN ? __ballot_sync(kFull, fix) : mf;
    // Lanes 0 to 3 reserve the places and count, side by side.
    u32 got = 0;
    static_assert(kFront == 2 && kLive == 3 && kNewFixed == 4, "of lanes 1 to 3");
    {
        const u32 cnt = __popc(lane == 0 ? ms : lane == 1 ? mf : lane == 2 ? mx : mfix);
        if (lane < 4 && cnt) got = atomicAdd(&s.cnt[lane == 0 ? q : lane + 1], cnt);
    }
    const u32 bs = __shfl_sync(kFull, got, 0), bf = __shfl_sync(kFull, got, 1);
    if (sv) {
        const u32 k = bs + __popc(ms & below);
        s.act[q][k] = en;
        const Dist t = en.ow == kNoOutW ? S::none(P) : dy + en.ow;
        a.fd = dy < a.fd ? dy : a.fd;
        a.ft = t < a.ft ? t : a.ft;
        if (en.deg > P.hub) atomicAdd(&s.chunks, (en.deg + P.chunk - 1) / P.chunk);
    }
    if (fl) {
        const u32 k = bf + __popc(mf & below);
        const u32 od = fx ? en.odeg : 0u;
        s.fr[k] = FrontEntry{en.g | (fix ? kFixedEntry : 0u), od,
                             en.ob | (fx ? kLiveEntry : 0ull)};
        s.fdist[k] = dy;
        if (od > P.hub) atomicAdd(&s.fchunks, (od + P.chunk - 1) / P.chunk);
    }
}

// Steps (b) and (c): the CTA's active list p; survivors go to list p ^ 1.
template <class S, bool WIN>
__device__ __forceinline__ void small_phase_bounds(const RoundParams& P, SmallShared& s, u32 p,
                                                   u32 r, typename S::Dist thr,
                                                   typename S::Dist minD, u32 target, u32 lane,
                                                   u32 wib, SmallAcc<S>& a) {
    typedef typename S::Dist Dist;
    constexpr u32 U = kSmallU;
    const u32 cur = r & 1u;
    const u32 n = s.cnt[p];
    const u32 gs = group_shift(n), sub = lane & ((1u << gs) - 1u);
    const u32 lim = max(kGroupDeg, (4 * U) << gs);
    const typename S::Rec* rec = S::rec(P);
    u32 base = wib << (5 - gs), b = 0, nb = 0;
    bool tiles = true;
    for (;;) {
        ActEntry en = {0, 0, 0, 0, 0, kNoOutW};
        bool lead, fix_now = false;
        u32 deg, len, k, step, todo = 0;
        if (tiles) {
            if (base >= n) {
                tiles = false;
                __syncthreads();
                nb = min(s.nbig, kBigCap);
                continue;
            }
            const u32 idx = base + (lane >> gs);
            base += kSmallWarps << (5 - gs);
            const bool in = idx < n;
            if (in) en = s.act[p][idx];
            lead = in && sub == 0;
            deg = en.deg;
            if (P.cheap && in) {
                Dist d, c;
                S::own(P, S::load(rec + en.g, cur), d, c);
                fix_now = cheap_rules_fix((u64)d, __ldg(P.g.inw + en.g), (u64)thr, (u64)minD);
                if (fix_now) deg = 0;              // its in-edges are not read
            }
            bool cta = false;
            if (lead) {
                a.in += deg;
                a.act++;
                if (deg > kCtaDeg) cta = take_big(s, idx);
            }
            len = deg <= lim ? deg : 0u;
            k = sub;
            step = 1u << gs;
            todo = __ballot_sync(kFull, lead && deg > lim && !cta);
            lead = lead && !cta;
        } else {
            if (b >= nb) break;
            if (threadIdx.x == 0) s.bigmin = kInf64;
            __syncthreads();
            en = s.act[p][s.big[b]];
            ++b;
            deg = len = en.deg;
            k = threadIdx.x;
            step = kSmallThreads;
            lead = threadIdx.x == 0;
        }
        // The vertex's own state, beside its edges.
        typename S::Nbr me = {0, 0};
        if (lead) me = S::load(rec + en.g, cur);
        const uint2* adj = P.g.in_adj + en.ib;
        u32 own = 32;                              // row owner (32: groups or the CTA)
        Dist m = S::kTermInf;
        for (;;) {
            Dist w = S::kTermInf;
#pragma unroll 1
            for (; __any_sync(kFull, k < len); k += step * U) {
                uint2 e[U];
                typename S::Nbr v[U];
                const u32 nu = __any_sync(kFull, k + step < len) ? U : 1u;
#pragma unroll
                for (u32 i = 0; i < U; ++i) {
                    e[i] = make_uint2(0u, 0u);
                    if (i < nu && k + i * step < len) e[i] = __ldg(adj + k + i * step);
                }
#pragma unroll
                for (u32 i = 0; i < U; ++i)
                    if (i < nu && k + i * step < len) v[i] = S::load(rec + e[i].x, cur);
#pragma unroll
                for (u32 i = 0; i < U; ++i)
                    if (i < nu && k + i * step < len)
                        w = min(w, S::term(P, v[i], e[i].y, thr, minD));
            }
            if (tiles && own == 32) {
                for (u32 d = step >> 1; d; d >>= 1)
                    w = min(w, (Dist)__shfl_xor_sync(kFull, w, d));
                m = w;
            } else {
                w = S::wmin(w);
                if (lane == own) m = w;
            }
            if (todo == 0) {
                if (!tiles) m = w;
                break;
            }
            own = __ffs(todo) - 1;
            todo &= todo - 1;
            adj = P.g.in_adj + __shfl_sync(kFull, en.ib, own);
            len = __shfl_sync(kFull, deg, own);
            k = lane;
            step = 32;
        }
        if (!tiles) {
            if (lane == 0) atomicMin(&s.bigmin, (u64)m);
            __syncthreads();
            m = S::clip(s.bigmin);
        }
        Dist dy, cy;
        S::own(P, me, dy, cy);
        small_decide<S, WIN>(P, s, p ^ 1u, r, lead, fix_now, en, dy, cy, m, thr, minD, target, lane,
                             a);
        if (!tiles) __syncthreads();
    }
}

// ------------------------------------------------------------------- the kernel

// Whether round ctl->round starts in this kernel: the loop is running and not
// past its stop round, the frontier and the active set each make at most
// P.tail_items work items (32-entry tiles plus hub chunks) and fit the lists,
// and few of them are hub chunks (P.tail_chunks).  Every CTA takes the same decision.
__device__ __forceinline__ bool small_fits(const RoundParams& P, u32 items, u32 entries,
                                           u32 chunks) {
    return items <= P.tail_items && entries <= kSmallEntries && chunks <= P.tail_chunks;
}

template <class S, bool WIN>
__global__ void __launch_bounds__(kSmallThreads, 1)
    k_small(const __grid_constant__ RoundParams P) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    SmallShared& s = *reinterpret_cast<SmallShared*>(s_raw);
    typedef typename S::Dist Dist;
    Ctl* ctl = P.ctl;
    InstVar* iv = P.ivar;
    const u32 rank = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, wib = tid >> 5;
    const bool lead = rank == 0 && tid == 0;
    u32 r = ld_volatile(&ctl->round);
    const u32 stop_round = ld_volatile(&ctl->stop_round);
    const u32 limit = ld_volatile(&ctl->round_limit);
    const u32 c0 = r & 1u;
    const u32 nfs = ld_volatile(&ctl->nFS[c0]), nas = ld_volatile(&ctl->nAS[c0]);
    const u64 fhpk = ld_volatile(&ctl->FHpk[c0]), ahpk = ld_volatile(&ctl->AHpk[c0]);
    const u32 nfh = (u32)(fhpk >> 32), nah = (u32)(ahpk >> 32);
    const bool go = ld_volatile(&ctl->status) == kRunning && r <= stop_round &&
                    small_fits(P, ((nfs + 31) >> 5) + (u32)fhpk, nfs + nfh, (u32)fhpk) &&
                    small_fits(P, ((nas + 31) >> 5) + (u32)ahpk, nas + nah, (u32)ahpk);
    if (!go) {
        if (lead && P.cond)
            cudaGraphSetConditional(
                P.cond, (ld_volatile(&ctl->status) == kRunning && r <= stop_round) ? 1u : 0u);
        return;
    }
    const u64 d0 = ld_volatile(&iv->minD[c0]), t0 = ld_volatile(&iv->thr[c0]);
    const u32 target = iv->target, start_round = iv->start_round, max_rounds = iv->max_rounds;
    typename S::Rec* rec = S::rec(P);

    // The lists, dealt round-robin over the CTAs.
    if (tid == 0) {
        s.nbig = s.chunks = s.fchunks = s.flags = s.cnt[kNewFixed] = 0;
        s.cnt[0] = (nas + nah + kSmallCTAs - 1 - rank) / kSmallCTAs;
        s.cnt[1] = 0;
        s.cnt[kFront] = s.cnt[kLive] = (nfs + nfh + kSmallCTAs - 1 - rank) / kSmallCTAs;
    }
    for (u32 i = tid; rank + kSmallCTAs * i < nfs + nfh; i += kSmallThreads) {
        const u32 k = rank + kSmallCTAs * i;
        const u32 g = k < nfs ? P.L.FS[c0][k] : P.L.FH[c0][k - nfs].x;
        const u64 o0 = P.g.out_off[g], o1 = P.g.out_off[g + 1];
        s.fr[i] = FrontEntry{g | (WIN ? 0u : kFixedEntry), (u32)(o1 - o0), o0 | kLiveEntry};
        s.fdist[i] = WIN ? P.snap[g] : (u64)S::fixed_dist(rec + g, c0);
    }
    for (u32 i = tid; rank + kSmallCTAs * i < nas + nah; i += kSmallThreads) {
        const u32 k = rank + kSmallCTAs * i;
        const u32 g = k < nas ? P.L.AS[c0][k] : P.L.AH[c0][k - nas].x;
        const u64 i0 = P.g.in_off[g], i1 = P.g.in_off[g + 1];
        const u64 o0 = P.g.out_off[g], o1 = P.g.out_off[g + 1];
        u32 ow;
        if constexpr (S::kNarrow) ow = plain_outw(P.g.outw[g]);
        else ow = rec[g].outw;
        s.act[0][i] = ActEntry{g, (u32)(i1 - i0), i0, o0, (u32)(o1 - o0), ow};
    }
    if (WIN) {
        // Vertices fixed in the last round: their fixed word goes to the other
        // parity (the frontier need not hold them).
        const u32 nfx = min(ld_volatile(&ctl->nFX[c0]), P.L.capS);
        for (u32 i = rank * kSmallThreads + tid; i < nfx; i += kSmallCTAs * kSmallThreads) {
            const u32 g = P.L.FX[c0][i];
            S::set_c(rec + g, c0 ^ 1u, S::fixed_dist(rec + g, c0), true);
        }
    }
    small_sync();
    if (lead) {
        // The global lists are empty from here on; a hand-over fills them again.
        for (u32 i = 0; i < 2; ++i) {
            ctl->nFS[i] = ctl->nAS[i] = ctl->nFX[i] = 0;
            ctl->FHpk[i] = ctl->AHpk[i] = 0;
            iv->minD[i] = iv->thr[i] = kInf64;
        }
    }
    small_sync();

    SmallAcc<S> a = {S::kInf, S::kInf, 0, 0, 0, 0, 0, 0};
    if (lead) {                                // the survivors' folds of the round before
        a.fd = S::clip(d0);
        a.ft = S::clip(t0);
    }
    u64 reached = 0;
    u32 p = 0, surv = nas + nah, schunks = (u32)ahpk;
    // How the kernel ends: a status of the query, or the round to hand over.
    u32 end_status = kRunning;
    bool cup_only = false, err_rounds = false;
    Dist thr = S::kInf, minD = S::kInf;
    for (;;) {
        const u32 cur = r & 1u;
        // Step (a) of round r, then the minima over the active set.
        if (tid == 0) s.cnt[p ^ 1u] = 0;
        small_phase_relax<S, WIN>(P, s, p, cur, lane, wib, a);
        {
            const Dist d = S::wmin(a.fd), t = S::wmin(a.ft);
            const u32 np = __reduce_add_sync(kFull, a.pushed);
            const u32 nc = __reduce_add_sync(kFull, a.chunks);
            a.fd = a.ft = S::kInf;
            a.pushed = a.chunks = 0;
            if (lane == 0) {
                s.wd[wib] = d == S::kInf ? kInf64 : (u64)d;
                s.wt[wib] = t == S::kInf ? kInf64 : (u64)t;
                s.wpush[wib] = np;
                s.wchunk[wib] = nc;
            }
        }
        __syncthreads();
        if (wib == 0) {
            const bool in = lane < kSmallWarps;
            const u64 d = warp_min64(in ? s.wd[lane] : kInf64);
            const u64 t = warp_min64(in ? s.wt[lane] : kInf64);
            const u32 np = __reduce_add_sync(kFull, in ? s.wpush[lane] : 0u);
            const u32 nc = __reduce_add_sync(kFull, in ? s.wchunk[lane] : 0u);
            const u32 flags = s.flags;
            if (lane < kSmallCTAs) {
                const u32 at = map_cta(smem_addr(&s.xb[rank]), lane);
                dsm_st4(at, (u32)d, (u32)(d >> 32), (u32)t, (u32)(t >> 32));
                dsm_st4(at + 16, 0u, np, nc, 0u);
                dsm_st4(at + 32, flags, 0u, 0u, 0u);
            }
        } else if (wib == 1 && lane == 0) {
            a.front += s.cnt[kLive];
            s.chunks = s.fchunks = s.nbig = 0;
            s.cnt[kFront] = s.cnt[kLive] = s.cnt[kNewFixed] = 0;
        }
        small_sync();
        u32 nact = surv, chunks = schunks;
        {
            const bool in = lane < kSmallCTAs;
            const u64 d = in ? s.xb[lane].minD : kInf64, t = in ? s.xb[lane].thr : kInf64;
            minD = S::wmin(S::clip(d));
            thr = S::wmin(S::clip(t));
            nact += __reduce_add_sync(kFull, in ? s.xb[lane].nact : 0u);
            chunks += __reduce_add_sync(kFull, in ? s.xb[lane].chunks : 0u);
            const u32 flags = __reduce_or_sync(kFull, in ? s.xb[lane].flags : 0u);
            if ((flags & 1u) || !small_fits(P, ((nact + 31) >> 5) + chunks, nact, chunks)) {
                cup_only = true;               // the full grid finishes the round
                break;
            }
        }
        // Steps (b) and (c).
        small_phase_bounds<S, WIN>(P, s, p, r, thr, minD, target, lane, wib, a);
        __syncthreads();
        if (wib == 0) {
            const u32 ns = s.cnt[p ^ 1u], nl = s.cnt[kLive], nf = s.cnt[kNewFixed], ch = s.chunks,
                      fch = s.fchunks, flags = s.flags;
            if (lane < kSmallCTAs) {
                const u32 at = map_cta(smem_addr(&s.xa[rank]), lane);
                dsm_st4(at, fch, 0u, 0u, 0u);
                dsm_st4(at + 16, nl, ns, ch, nf);
                dsm_st4(at + 32, flags, 0u, 0u, 0u);
            }
            __syncwarp();
            if (lane == 0) s.nbig = s.chunks = 0;
        }
        small_sync();
        const bool in = lane < kSmallCTAs;
        const u32 nfront = __reduce_add_sync(kFull, in ? s.xa[lane].nfront : 0u);
        const u32 fchunks = __reduce_add_sync(kFull, in ? (u32)s.xa[lane].minD : 0u);
        surv = __reduce_add_sync(kFull, in ? s.xa[lane].nact : 0u);
        schunks = __reduce_add_sync(kFull, in ? s.xa[lane].chunks : 0u);
        reached += __reduce_add_sync(kFull, in ? s.xa[lane].nfix : 0u);
        const u32 flags = __reduce_or_sync(kFull, in ? s.xa[lane].flags : 0u);
        // End of round r (the decisions of round_epilogue, in its order).
        if (nfront == 0 && !(WIN && surv != 0)) end_status = kDone;
        else if (flags & 2u) end_status = kStopped;
        else if (max_rounds != 0 && r - start_round + 1 >= max_rounds) end_status = kStopped;
        else if (r + 1 > limit) err_rounds = true;
        p ^= 1u;
        ++r;
        if (end_status != kRunning || err_rounds || r > stop_round ||
            !small_fits(P, ((nfront + 31) >> 5) + fchunks, nfront, fchunks))
            break;
    }

    // Hand over.  After the relaxation (cup_only): round r's active list and
    // minima.  At the end of a round: round r's frontier, its active list and
    // the survivors' folds.  (r already counts the next round there.)
    const u32 cu = r & 1u;
    if (end_status == kRunning && !err_rounds) {
        const u32 n = s.cnt[p] < kSmallCap ? s.cnt[p] : kSmallCap;
        for (u32 i = tid; i < n; i += kSmallThreads) {
            const ActEntry en = s.act[p][i];
            if (en.deg > P.hub)
                put_hub(P, &ctl->AHpk[cu], P.L.AH[cu], P.L.AC[cu], en.g, en.deg);
            else
                put_small(P, P.L.AS[cu], atomicAdd(&ctl->nAS[cu], 1u), en.g);
        }
        if (!cup_only) {
            for (u32 i = tid; i < s.cnt[kFront]; i += kSmallThreads) {
                const FrontEntry f = s.fr[i];
                const u32 g = f.g & ~kFixedEntry;
                if (f.g & kFixedEntry) S::set_c(rec + g, cu ^ 1u, (Dist)s.fdist[i], true);
                if (!(f.ob & kLiveEntry)) continue;
                if (f.deg > P.hub)
                    put_hub(P, &ctl->FHpk[cu], P.L.FH[cu], P.L.FC[cu], g, f.deg);
                else
                    put_small(P, P.L.FS[cu], atomicAdd(&ctl->nFS[cu], 1u), g);
            }
            const Dist d = S::wmin(a.fd), t = S::wmin(a.ft);
            if (lane == 0 && d != S::kInf) atomicMin(&iv->minD[cu], (u64)d);
            if (lane == 0 && t != S::kInf) atomicMin(&iv->thr[cu], (u64)t);
        }
    }
    {
        const u64 o = warp_sum64(a.out), i = warp_sum64(a.in), ac = warp_sum64(a.act),
                  fr = warp_sum64(a.front);
        if (lane == 0) {
            if (o) atomicAdd(&ctl->stats[0].v, o);
            if (i) atomicAdd(&ctl->stats[1].v, i);
            if (ac) atomicAdd(&ctl->stats[2].v, ac);
            if (fr) atomicAdd(&ctl->stats[3].v, fr);
        }
    }
    if (lead) {
        ctl->stats[4].v += reached;
        ctl->round = r;
        ctl->cup_only = cup_only ? 1u : 0u;
        ctl->work[0].v = 0;
        u32 st = kRunning;
        if (end_status != kRunning) {
            iv->rounds = r - start_round;
            iv->status = end_status;
            ctl->running = 0;
            st = kDone;
        } else if (err_rounds) {
            st = kErrRounds;
        }
        ctl->status = st;
        if (cup_only) {
            // What the skipped relaxation launch would have opened; the minima.
            iv->minD[cu] = minD == S::kInf ? kInf64 : (u64)minD;
            iv->thr[cu] = thr == S::kInf ? kInf64 : (u64)thr;
            iv->nfix[cu ^ 1u] = 0;
            ctl->work[1].v = 0;
            ctl->done_ctas = 0;
        }
        if (P.cond) cudaGraphSetConditional(P.cond, (st == kRunning && r <= stop_round) ? 1u : 0u);
    }
    // No CTA leaves while another may still write to its shared memory (the
    // last such writes were before the last barrier, so none can).
}

}  // namespace sssp
