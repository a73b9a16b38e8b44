// cand_eval.cuh -- the exact verdict of one candidate priority order, by one
// group of LG lanes (16 or 32), lane r holding the chain of rank r (0 = highest
// priority).  Used by the search (analyze_cand.cu) and the Audsley-style seed
// (audsley.cu).
//
// The analysis is that of analyze_lazy.cu (Theorem 1, Eq. 6, with Eqs. 1-5, in
// the 32-bit narrow sums), asked for less: not every chain's R, only whether all
// of them (or one target chain) are schedulable.  Issue-bound, so it is arranged
// to execute little:
//  - In rank order "higher priority" is "lower lane": the sets hps(c), Lemma 2's
//    lower bound (a prefix sum of S*) and the same-bucket blocking (a suffix
//    maximum of M*) need no sets or sorted copies.  What does not depend on the
//    order (the aggregates, whether the system is inside the 32-bit and narrow
//    bounds, whether any core is shared) is read from the chain records.
//    Executors without a second chain on their core need no relations at all.
//  - Every chain's R is at least low = B + E + own + delta eps + f sum_{hps} S* + 2
//    sum_{hp, hpp} w: every arrival count is at least f or 2, Lemma 2's sum at
//    least own + f delta sum S* (f = 2 when A* + blk >= 1, else 1), and w is the
//    same bound on an interferer's E + H* (E + delta eps for a suspending hpp).  A
//    chain whose bound is above its deadline is not schedulable, and one vote over
//    the lanes rejects the candidate before any recurrence: 84% of the random
//    orders of the 16-chain search workload (88% fail), 99.8% of uneven systems'.
//  - For the others every lane takes its own chain's recurrence at once: one
//    evaluation of all chains reads the bounds on H* that the evaluation before
//    it gave, so the R's and H*'s rise together to the least fixed point that
//    the chains one after another would reach (their order has no cycle), and a
//    vote ends it when an R passes its deadline.  H* stops at Lemma 2's lower
//    bound; a chain whose Eq. 4 sum passes that (one or two of 16) and those
//    whose DEP-rule set holds it are then taken one by one, with Lemma 2's exact
//    sum, smallest slack first, up to the first failure.  Which chains are
//    evaluated before a failure does not change the verdict, and every
//    recurrence starts at or below its least fixed point.
//  - The part of that bound that needs no relation (E + own + delta eps + f sum S*)
//    is voted on first: it rejects 40% of the first workload's orders and nearly
//    all that fail of the uneven systems', whose shared executors make the
//    relations long.
#pragma once

#include "reg_common.cuh"

namespace paam_cand {
using namespace paam_reg;

// Word 11 of a chain record (chain_records_kernel): the chain's own flag and
// those of its system (systems of up to 32 chains).
constexpr uint32_t kRecFit = 1u;        // every chain of the system is inside the 32-bit bound
constexpr uint32_t kRecSpin = 2u;       // this chain busy-waits
constexpr uint32_t kRecNarrow16 = 4u;   // every deadline below 2^27 - 16
constexpr uint32_t kRecNarrow32 = 8u;   // ... below 2^27 - 32
constexpr uint32_t kRecCounted = 16u;   // the iteration bound passes kIterCap: count evaluations
constexpr uint32_t kRecShared = 32u;    // some core runs two chains or more
constexpr uint32_t kRecTwoExec = 64u;   // some core runs chains of two executors or more

// Joint evaluations at most before the chains are taken one by one (some 4 suffice
// for the workloads; a system with very short periods could take millions).
constexpr int kJointIters = 48;

template <int LG>
struct CandSmem {
    uint4 rel[LG]; // {hp, hpp, deps = delta eps, first segment relative to the system's first}
    uint4 rec[LG]; // {D, base = B + E, own = S* + delta blk (capped at D + 1), R's start}
    uint4 dvu[LG]; // by rank among the users: {2 (T - 1), magic, l, S*} (a server interferer's term)
    uint4 dvc[LG]; // by rank: {2 (T - 1), magic, l, E + H*'s bound} (an hp interferer's term)
    uint32_t whpp[LG]; // by rank: the same as an hpp interferer
    uint4 seg[LG]; // {delta, lb (Lemma 2's lower bound past own), blk, 0}
    uint32_t xm[LG];   // by the first chain of an executor: the ranks of its chains
    uint32_t ym[LG];   // the same for a core
    uint32_t sx[LG];   // by rank: the ranks on the same executor
    uint32_t emax[LG]; // by rank: longest callback (Lemma 4)
    uint32_t ord[LG];  // by rank: the chain
};

// ceil(t / T) + 1 (Lemma 1) times c, capped at 2^27 - 1 so that the group's sum fits 32 bits
__device__ __forceinline__ uint32_t term_of(uint32_t mu, uint32_t c)
{
    const uint64_t v = (uint64_t)mu * c;
    return v < kNarrow - 1 ? (uint32_t)v : kNarrow - 1;
}

// Every lane of the group calls it; chain: the local index of the chain of rank
// `lane` (lane < n).  recs: the system's records.  TGT: the verdict of the chain
// of rank tgt alone; otherwise of all chains.  The system is inside the narrow
// bound of LG lanes.
template <int LG, bool TGT>
__device__ __forceinline__ bool cand_eval(const BatchDev &b, int32_t n_buckets, uint64_t kappa2, uint64_t eps,
                                          int n, int64_t seg_base, const uint4 *__restrict__ recs, int chain,
                                          int tgt, CandSmem<LG> &s, int lane, unsigned gm)
{
    const unsigned sh = LG == 32 ? 0u : (threadIdx.x & 16u); // the group's first lane in the warp
    const uint32_t self = 1u << lane, lt = self - 1u;
    const uint32_t all = n >= 32 ? ~0u : (1u << n) - 1u;
    const bool val = lane < n;
    uint32_t tm2 = 0, mg = 0, lg = 0, D = 0, E = 0, S = 0, Emax = 0, M = 0, Amin = 0, dl = 0, seg0 = 0, fl = 0;
    uint32_t cx = 0, cy = 0; // chains (by index) on the same executor, on the same core
    if (val) {
        const uint4 *r = recs + 4 * chain;
        const uint4 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3];
        tm2 = r0.x, mg = r0.y, lg = r0.z, D = r0.w;
        E = r1.x, S = r1.y, Emax = r1.z, M = r1.w;
        Amin = r2.x, dl = r2.y, seg0 = r2.z, fl = r2.w;
        cx = r3.z, cy = r3.w;
    }
    const uint32_t sysfl = __shfl_sync(gm, fl, 0, LG);
    const bool user = dl != 0, sp = (fl & kRecSpin) != 0;

    // ---- Lemma 2's lower bound and the same-bucket blocking
    uint32_t sums = user ? umin(S, kNarrow - 1) : 0u; // sum of S* over the users of higher priority
#pragma unroll
    for (int d = 1; d < LG; d <<= 1) {
        const uint32_t w = __shfl_up_sync(gm, sums, d, LG);
        if (lane >= d) sums = umin(sums + w, kNarrow);
    }
    sums = __shfl_up_sync(gm, sums, 1, LG);
    if (lane == 0) sums = 0u;
    uint32_t blk = user ? M : 0u;
    if (n_buckets == 1) { // every user shares the bucket: the longest lower-priority request (R2-R3)
#pragma unroll
        for (int d = 1; d < LG; d <<= 1) {
            const uint32_t w = __shfl_down_sync(gm, blk, d, LG);
            if (lane + d < LG) blk = umax(blk, w);
        }
        blk = __shfl_down_sync(gm, blk, 1, LG);
        if (lane + 1 >= LG || !user) blk = 0u;
    } else { // bucket = floor(rank among the users * n_buckets / |U|) (R2), rising along the lanes
        const uint32_t users = __ballot_sync(gm, user) >> sh;
        const uint32_t nu = (uint32_t)__popc(users), ur = (uint32_t)__popc(users & lt);
        const uint32_t nb = umin((uint32_t)n_buckets, nu); // from |U| buckets on every user has its own
        const uint32_t key = ur < nu ? ur * nb / nu : 0xFFFFFFFFu; // a lane without a segment takes the next user's
#pragma unroll
        for (int d = 1; d < LG; d <<= 1) {
            const uint32_t w = __shfl_down_sync(gm, blk, d, LG), kk = __shfl_down_sync(gm, key, d, LG);
            if (lane + d < LG && kk == key) blk = umax(blk, w);
        }
        blk = __shfl_down_sync(gm, blk, 1, LG);
        const uint32_t kk = __shfl_down_sync(gm, key, 1, LG);
        if (lane + 1 >= LG || !user || kk != key) blk = 0u;
    }

    // ---- own terms; the lower bound of R without CPU blocking and interference
    const uint32_t deps = (uint32_t)((uint64_t)dl * eps);
    const uint64_t own64 = (uint64_t)S + (uint64_t)dl * blk;
    const uint32_t own = own64 < (uint64_t)D + 1 ? (uint32_t)own64 : D + 1; // above D: as D + 1
    const uint32_t f = ((uint64_t)Amin + blk) >= 1 ? 2u : 1u;
    const uint32_t dem = E + (user ? own + deps + f * sums : 0u); // E + H*, below 2^32: each part is
    if (__any_sync(gm, val && (!TGT || lane == tgt) && dem > D)) return false;

    // ---- relations (Lemma 4, Theorem 1): only where a core is shared
    uint32_t hp = 0, hpp = 0, needs = 0, Bv = 0;
    if (sysfl & kRecShared) {
        s.xm[lane] = 0u;
        s.ym[lane] = 0u;
        s.emax[lane] = Emax;
        const uint32_t spins = __ballot_sync(gm, sp) >> sh;
        __syncwarp(gm);
        const int xi = val ? __ffs(cx) - 1 : 0, yi = val ? __ffs(cy) - 1 : 0;
        if (val) {
            atomicOr(&s.xm[xi], self);
            atomicOr(&s.ym[yi], self);
        }
        __syncwarp(gm);
        const uint32_t samex = val ? s.xm[xi] : self;
        hp = samex & lt;
        for (uint32_t lo = samex & ~lt & ~self; lo; lo &= lo - 1) // Lemma 4: one LP callback on the executor
            Bv = umax(Bv, s.emax[__ffs(lo) - 1]);
        if (sysfl & kRecTwoExec) {
            // criticality-as-priority: an executor's priority is that of its first rank
            const int top = __ffs(samex) - 1;
            const uint32_t tops = __ballot_sync(gm, val && top == lane) >> sh;
            s.sx[lane] = samex;
            __syncwarp(gm);
            if (val)
                for (uint32_t m = s.ym[yi] & tops & ((1u << top) - 1u); m; m &= m - 1) hpp |= s.sx[__ffs(m) - 1];
        }
        needs = hp | (hpp & spins); // the DEP rule
    }

    // ---- the lower bound of R
    const uint32_t base = Bv + E;
    uint32_t low = umin(Bv + umin(dem, kNarrow), 1u << 31);
    // E + H* as a CPU interferer's coefficient, from below (capped: above every deadline)
    const uint32_t esus = umin(E + deps, kNarrow); // a suspending chain in hpp: delta eps only
    uint32_t whp = umin(dem, kNarrow), whpp = sp ? whp : esus;
    const bool shared = (sysfl & kRecShared) != 0;
    if (shared) {
        s.dvc[lane] = make_uint4(tm2, mg, lg, whp);
        s.whpp[lane] = whpp;
        __syncwarp(gm);
        uint32_t cs = 0;
        for (uint32_t m = hp; m; m &= m - 1) cs = umin(cs + 2u * s.dvc[__ffs(m) - 1].w, kNarrow);
        for (uint32_t m = hpp; m; m &= m - 1) cs = umin(cs + 2u * s.whpp[__ffs(m) - 1], kNarrow);
        low += cs;
    }
    const bool over = val && low > D;
    uint32_t todo = all, sched = 0;
    uint32_t Ehp = E, Ehpp = E + (sp ? 0u : deps);
    if (TGT) { // the target and, through the DEP rule, the chains its verdict rests on
        todo = 1u << tgt;
        if (shared)
            for (;;) {
                const uint32_t more = todo | __reduce_or_sync(gm, ((todo >> lane) & 1) ? needs : 0u);
                if (more == todo) break;
                todo = more;
            }
        if (__any_sync(gm, over && ((todo >> lane) & 1))) return false;
    } else if (__any_sync(gm, over)) {
        return false;
    }
    const uint64_t lb64 = (uint64_t)f * dl * sums;
    const uint32_t lb = lb64 < kNarrow ? (uint32_t)lb64 : kNarrow;
    uint32_t R0 = low; // where the chain's recurrence starts: at or below its least fixed point
    if (!TGT && !(sysfl & kRecCounted)) {
        const uint32_t users = __ballot_sync(gm, user) >> sh;
        const int above = __popc(users & lt), nu = __popc(users);
        if (user) s.dvu[above] = make_uint4(tm2, mg, lg, S);
        __syncwarp(gm);
        bool left = false, settled = false;
        for (int it = 0; it < kJointIters; ++it) {
            uint64_t sum = 0;
#pragma unroll 4
            for (int h = 0; h < nu - 1; ++h) {
                const uint4 dv = s.dvu[h];
                if (h < above) sum += (uint64_t)rarrivals(R0, dv.x, dv.y, dv.z) * dv.w;
            }
            const uint32_t as = sum < kNarrow ? (uint32_t)sum : kNarrow;
            left = user && as > lb;
            const uint32_t hs = user ? umin(own + umin(as, lb) + deps, kNarrow) : 0u; // Eq. 1
            uint32_t Rn = base + hs;
            if (shared) {
                whp = umin(E + hs, kNarrow);
                whpp = sp ? whp : esus;
                __syncwarp(gm);
                s.dvc[lane].w = whp;
                s.whpp[lane] = whpp;
                __syncwarp(gm);
                uint64_t cs = 0;
                for (uint32_t m = hp; m; m &= m - 1) {
                    const uint4 dv = s.dvc[__ffs(m) - 1];
                    cs += (uint64_t)rarrivals(R0, dv.x, dv.y, dv.z) * dv.w;
                }
                for (uint32_t m = hpp; m; m &= m - 1) {
                    const int h = __ffs(m) - 1;
                    const uint4 dv = s.dvc[h];
                    cs += (uint64_t)rarrivals(R0, dv.x, dv.y, dv.z) * s.whpp[h];
                }
                Rn += cs < kNarrow ? (uint32_t)cs : kNarrow;
            }
            const bool moved = val && Rn != R0;
            R0 = val ? Rn : R0;
            const uint32_t vote = __reduce_or_sync(gm, (val && R0 > D ? 2u : 0u) | (moved ? 1u : 0u));
            if (vote & 2u) return false;
            if (!vote) {
                settled = true;
                break;
            }
        }
        if (settled) {
            // chains that Lemma 2's exact sum may still lower, and those that rest on them
            uint32_t open = __ballot_sync(gm, left) >> sh;
            if (!open) return true;
            if (shared)
                for (;;) {
                    const uint32_t more = open | (__ballot_sync(gm, (needs & open) != 0) >> sh);
                    if (more == open) break;
                    open = more;
                }
            sched = all & ~open;
            if ((sched >> lane) & 1) {
                Ehp = whp;
                Ehpp = whpp;
            }
        }
    }
    if (((todo & ~sched) >> lane) & 1) {
        s.rel[lane] = make_uint4(hp, hpp, deps, seg0);
        s.rec[lane] = make_uint4(D, base, own, R0);
        s.seg[lane] = make_uint4(dl, lb, blk, 0u);
    }
    __syncwarp(gm);

    // ---- Theorem 1 (Eq. 6), smallest slack first among the chains that are ready
    const uint32_t key = ((D - R0) << (LG == 32 ? 5 : 4)) | (uint32_t)lane; // D < 2^27 - LG: fits, below ~0
    const uint32_t k2 = (uint32_t)kappa2;
    auto chains = [&](auto counted_tag) -> bool {
        constexpr bool CNT = decltype(counted_tag)::value;
        while (sched != todo) {
            const bool ready = (((todo & ~sched) >> lane) & 1) && !(needs & ~sched);
            const uint32_t pick = __reduce_min_sync(gm, ready ? key : 0xFFFFFFFFu);
            if (pick == 0xFFFFFFFFu) return false; // cannot happen: the DEP rule has no cycle
            const int c = (int)(pick & (LG - 1));
            const uint4 rl = s.rel[c], rc = s.rec[c], sg = s.seg[c];
            const uint32_t D32 = rc.x, base_c = rc.y, own_c = rc.z, deps_c = rl.z, dl_c = sg.x;
            const uint32_t ccoef = ((rl.x >> lane) & 1) ? Ehp : (((rl.y >> lane) & 1) ? Ehpp : 0u);
            const bool cpu = (rl.x | rl.y) != 0; // the same in every lane of the group
            const uint32_t acoef = (user && lane < c) ? S : 0u;
            uint32_t R = rc.w, hs = 0, ev = 0;
            uint32_t lbc = dl_c ? sg.y : kInfR; // kInfR once the fixed points are taken
            uint32_t Hs = kInfR;               // Lemma 2's per-segment sum: unbounded, or not needed yet
            bool ok = false;
            for (;;) { // twice at most: before and after the fixed points are taken
                bool need = false;
                for (;;) {
                    if (CNT && ev++ == kIterCap) break;
                    const uint32_t mu = rarrivals(R, tm2, mg, lg);
                    uint32_t Rn = base_c;
                    if (dl_c) {
                        const uint32_t as = umin(__reduce_add_sync(gm, term_of(mu, acoef)), kNarrow);
                        if (as > lbc) { // this evaluation is taken again once Lemma 2's sum is known
                            need = true;
                            if (CNT) --ev;
                            break;
                        }
                        hs = umin(Hs, own_c + as) + deps_c; // Eq. 1 with min(Eq. 3, Eq. 4)
                        Rn += umin(hs, kNarrow);
                    }
                    if (cpu) Rn += umin(__reduce_add_sync(gm, term_of(mu, ccoef)), kNarrow);
                    if (Rn == R) {
                        ok = true;
                        break;
                    }
                    R = Rn;
                    if (R > D32) break;
                }
                if (!need) break;
                lbc = kInfR;
                // the sum matters only below Eq. 4 at R = D (and below D + 1)
                const uint32_t hchd =
                    umin(__reduce_add_sync(gm, term_of(rarrivals(D32, tm2, mg, lg), acoef)), kNarrow);
                const uint32_t lim = umin(own_c + hchd, D32 + 1);
                const int64_t qb = seg_base + rl.w;
                uint32_t H32 = 0;
                bool inf = false, capped = false;
                for (uint32_t q = 0; q < dl_c && !inf; ++q) {
                    const uint32_t hb = (uint32_t)b.A[qb + q] + k2 + sg.z;
                    uint32_t h = hb; // the recurrence starts with the first two terms
                    uint32_t evs = 0;
                    for (;;) {
                        if (h > D32 || H32 + h >= lim) {
                            inf = true;
                            break;
                        }
                        if (CNT && evs++ == kIterCap) {
                            inf = capped = true;
                            break;
                        }
                        const uint32_t nh =
                            hb + umin(__reduce_add_sync(gm, term_of(rarrivals(h, tm2, mg, lg), acoef)), kNarrow);
                        if (nh == h) break; // strictly increasing until here, bounded by D
                        h = nh;
                    }
                    H32 += h;
                }
                if (capped) return false; // no bound (PAAM_ST_ITERCAP)
                if (!inf) Hs = H32;
            }
            if (!ok) return false;
            sched |= 1u << c;
            if (TGT && c == tgt) return true;
            if (lane == c) {
                Ehp = E + hs;
                if (sp) Ehpp = E + hs;
            }
        }
        return true;
    };
    return (sysfl & kRecCounted) ? chains(std::true_type{}) : chains(std::false_type{});
}

} // namespace paam_cand
