// analyze_lazy_big.cu -- the lazy register-table analysis of the larger systems
// under the two options that analyze_lazy64.cu does not serve: segments on
// several accelerators (rule R1: one server per accelerator, analysed on its
// own), and the safe reading of Lemma 4 (blocking_mode 1).  One warp per system,
// CPL chains per lane (chain j = lane + 32 k, slot k): CPL = 1 for up to 32
// chains, CPL = 2 for up to 64, over the deferral list of the 16-lane kernels
// (analyze_lazy_acc.cu, the safe instantiation of analyze_lazy.cu).
//
// The mathematics and the order of work are those kernels' (see there) and, for
// two slots per lane, analyze_lazy64.cu's: the relations from priority slots and
// suffix scans, the blocking and Lemma 2's lower bound from scans in priority
// order (per accelerator), the chains one after another in the analysis order,
// Lemma 2's exact per-segment fixed points only at the first evaluation that
// needs them; under the safe reading every segment's bound beforehand, one per
// lane, then each chain's longest hold and Eq. 3's exact sum.  32-bit narrow sums
// (every deadline below 2^27 - 32 CPL); what is not narrow, outside the 32-bit
// bound or, under the safe reading, above kBigSegs segments goes to the int64
// kernel's list.  That kernel took all of them before: 200,000 uneven systems of
// 2-64 chains (17% above 16) with three accelerators 3.36 -> 0.67 ms, under the
// safe reading 1.47 -> 0.68 ms (both with the 16-lane pass; the passes here 0.16 +
// 0.12 and 0.17 + 0.19 ms).  Bound by issue at one chain per lane (55-58% of the
// slots) and by latency at two (27-37%, few systems in flight).
#include "reg_common.cuh"

namespace {
using namespace paam_reg;

constexpr unsigned kFull = 0xffffffffu;

template <int CPL>
using MaskOf = typename std::conditional<CPL == 1, uint32_t, uint64_t>::type;

template <int CPL>
struct BigSafe {
    static constexpr int N = 32 * CPL;
    uint4 dv[N];              // by chain: {2 (T - 1), magic, l, S*} (the interferer's term)
    MaskOf<CPL> hps[N];       // by chain
    uint2 ch[N];              // by chain: {D, blk}
    uint32_t hq[kBigSegs];    // by segment (relative to the system's first): its bound; kInfR none, kCapR cut short
    uint8_t segc[kBigSegs];   // by segment: its chain
};
struct BigNoSafe {};

template <int CPL, int NACC, bool SAFE>
struct BigSmem {
    static constexpr int N = 32 * CPL;
    using Mask = MaskOf<CPL>;
    Mask hp[N], hpp[N];       // by analysis position
    Mask hps[N][NACC];        // by analysis position, per accelerator
    uint4 rec[N];             // by position: {D, base = B + E, deps = delta eps, delta (all segments)}
    uint4 acc[N][NACC];       // by position: {own = S*_u + delta_u blk_u (capped at D + 1), lb_u (safe: Eq. 3's sum), blk_u, delta_u}
    uint2 at[N];              // by position: {chain, first segment relative to the system's first}
    Mask needs[N];            // by chain: its DEP-rule set
    uint32_t emax[N];         // by chain: longest callback, or hold (Lemma 4)
    uint32_t m[NACC][N];      // by chain: M*_u (same-bucket blocking with several buckets)
    int32_t bucket[NACC][N];  // by chain
    uint32_t msort[NACC][N];  // by priority rank: M*_u of the users of u (0 for the others)
    uint32_t ssort[NACC][N];  // by priority rank: S*_u of the users of u (capped at 2^27 - 1)
    Mask xms[N], cms[N];      // by executor / core index: its chains
    Mask exm[N], inv[N];      // by executor / chain priority value: the chains of that priority
    int32_t xep[N];           // by executor index: its highest chain priority
    typename std::conditional<SAFE, BigSafe<CPL>, BigNoSafe>::type x;
};

// ---- values of 32 CPL slots, slot lane + 32 k in element k of every lane -----
template <typename V>
__device__ __forceinline__ V shfl_any(V v, int src)
{
    if constexpr (sizeof(V) == 8) {
        const uint32_t lo = __shfl_sync(kFull, (uint32_t)v, src), hi = __shfl_sync(kFull, (uint32_t)((uint64_t)v >> 32), src);
        return (V)(((uint64_t)hi << 32) | lo);
    } else {
        return __shfl_sync(kFull, v, src);
    }
}

template <int CPL, typename V>
__device__ __forceinline__ V slot_value(const V (&a)[CPL], int v)
{
    V x = shfl_any(a[0], v & 31);
    if constexpr (CPL == 2) {
        const V y = shfl_any(a[1], v & 31);
        x = v < 32 ? x : y;
    }
    return x;
}

// exclusive scans over the slots: from above (later slots) or below; op(a, b) with identity zero
template <int CPL, typename V, typename F>
__device__ __forceinline__ void scan_above(V (&a)[CPL], int lane, F op)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const V w = shfl_any(a[k], (lane + d) & 31);
            if (lane + d < 32) a[k] = op(a[k], w);
        }
    V upper = 0;
    if constexpr (CPL == 2) {
        upper = shfl_any(a[1], 0);
        a[0] = op(a[0], upper);
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const V nx = shfl_any(a[k], (lane + 1) & 31);
        a[k] = lane < 31 ? nx : (k == 0 ? upper : (V)0);
    }
}

template <int CPL, typename V, typename F>
__device__ __forceinline__ void scan_below(V (&a)[CPL], int lane, F op)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const V w = shfl_any(a[k], (lane - d) & 31);
            if (lane >= d) a[k] = op(a[k], w);
        }
    V lower = 0;
    if constexpr (CPL == 2) {
        lower = shfl_any(a[0], 31);
        a[1] = op(a[1], lower);
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const V pv = shfl_any(a[k], (lane - 1) & 31);
        a[k] = lane > 0 ? pv : (k == 0 ? (V)0 : lower);
    }
}

template <int CPL>
__device__ __forceinline__ MaskOf<CPL> ballot_slots(const bool (&v)[CPL])
{
    MaskOf<CPL> m = __ballot_sync(kFull, v[0]);
    if constexpr (CPL == 2) m |= (MaskOf<CPL>)__ballot_sync(kFull, v[1]) << 32;
    return m;
}

// the warp's sum of every slot's arrivals(mu) times coefficient, each lane's part
// capped at 2^27 - 1 so that the sum fits 32 bits
template <int CPL>
__device__ __forceinline__ uint32_t slots_sum(const uint32_t (&mu)[CPL], const uint32_t (&c)[CPL])
{
    uint32_t v = 0;
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const uint64_t t = (uint64_t)mu[k] * c[k];
        v = umin(v + (t < kNarrow - 1 ? (uint32_t)t : kNarrow - 1), kNarrow - 1);
    }
    return umin(__reduce_add_sync(kFull, v), kNarrow);
}

template <int NACC>
__device__ __forceinline__ int acc_of(const BatchDev &b, int64_t q)
{
    if constexpr (NACC == 1) {
        return 0;
    } else { // validated: 0 .. PAAM_MAX_ACC - 1; the launch covers the largest
        const int u = b.acc[q];
        return u < NACC ? u : NACC - 1;
    }
}

// a term of a segment's recurrence under the safe reading, capped far above every deadline
constexpr uint64_t kTermCap = 1ull << 40;
// a hold without a bound, and any hold at or above it: every deadline is below it
constexpr uint32_t kHoldInf = (uint32_t)kFitR;

template <int CPL, int NACC, bool SAFE>
__device__ void big_system(const BatchDev &b, const AnalysisParams &p, int64_t item, BigSmem<CPL, NACC, SAFE> &s,
                           int lane, int64_t *__restrict__ R_out, uint8_t *__restrict__ st_out,
                           uint8_t *__restrict__ verdict, int32_t *wide_list, int32_t *wide_count)
{
    using Mask = MaskOf<CPL>;
    constexpr int N = 32 * CPL;
    int64_t sys;
    int32_t cand;
    item_of(p, item, sys, cand);
    if (p.K > 0 && p.early) { // candidate above the best schedulable one found so far
        const int pruned = __shfl_sync(kFull, cand_pruned(p, sys, cand) ? 1 : 0, 0);
        if (pruned) return;
    }
    const int64_t c0 = b.sys_chain_off[sys];
    const int n = (int)(b.sys_chain_off[sys + 1] - c0);
    if (CPL == 1 ? n > N : n <= 32) return; // the other width's
    const int64_t row = p.K > 0 ? sys * p.Kc + cand_of(p, sys, cand) : 0;
    const int16_t *rank_row = p.K > 0 ? p.ranks + row * p.nmax : nullptr;
    const int32_t *xprio = p.K > 0 ? nullptr : b.exec_prio; // candidates: criticality-as-priority
    const int64_t x0 = b.sys_exec_off[sys];
    const uint64_t kappa2 = 2 * (uint64_t)p.kappa, eps = (uint64_t)p.eps;
    const int64_t seg_base = n > 0 ? b.cb_seg_off[b.chain_cb_off[c0]] : 0;
    __syncwarp();

    // ---- per-chain aggregates (Sec. II-C), per accelerator -------------------
    uint32_t tm2[CPL], mg[CPL], lg[CPL], Dv[CPL], Ev[CPL], Emx[CPL], dlt[CPL], seg0[CPL];
    uint32_t Sa[CPL][NACC], Ma[CPL][NACC], Amn[CPL][NACC], dla[CPL][NACC];
    int32_t pr[CPL], ep[CPL], ex[CPL], co[CPL];
    bool sp[CPL], val[CPL];
    unsigned fit = 1, rank_ok = 1;
    Mask rbit = 0;
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int j = lane + 32 * k;
        val[k] = j < n;
        tm2[k] = mg[k] = lg[k] = Dv[k] = Ev[k] = Emx[k] = dlt[k] = seg0[k] = 0;
#pragma unroll
        for (int u = 0; u < NACC; ++u) Sa[k][u] = Ma[k][u] = Amn[k][u] = dla[k][u] = 0;
        pr[k] = ep[k] = INT32_MIN;
        ex[k] = co[k] = -1 - j;
        sp[k] = false;
        if (!val[k]) continue;
        const int64_t g = c0 + j;
        const int64_t T = b.T[g], D = b.D[g];
        ex[k] = b.exec[g];
        if (rank_row) { // candidate priority order: rank 0 is the highest priority
            const int r = rank_row[j];
            const bool ok = r >= 0 && r < n;
            rank_ok &= ok ? 1u : 0u;
            rbit |= ok ? (Mask)1 << r : 0;
            pr[k] = n - 1 - r;
        } else {
            pr[k] = b.prio[g];
        }
        co[k] = b.exec_core[x0 + ex[k]];
        if (xprio) ep[k] = xprio[x0 + ex[k]];
        sp[k] = b.spin[g] != 0;
        const int64_t cb0 = b.chain_cb_off[g], cb1 = b.chain_cb_off[g + 1];
        const int64_t q0 = b.cb_seg_off[cb0], q1 = b.cb_seg_off[cb1];
        // sums and extremes in 32 bits over values capped at 2^30 (a capped value
        // takes its chain's sum to the 32-bit bound, and the system to the int64 kernel)
        const int64_t *Ep = b.E + cb0;
        const int ncb = (int)(cb1 - cb0);
        uint32_t E = 0, Emax = 0;
#pragma unroll 4
        for (int i = 0; i < ncb; ++i) {
            const uint32_t e = (uint64_t)Ep[i] < kFitR ? (uint32_t)Ep[i] : (uint32_t)kFitR;
            E = umin(E + e, (uint32_t)kFitR);
            Emax = umax(Emax, e);
        }
        const int64_t nq = q1 - q0;
        const uint32_t k2c = kappa2 < kFitR ? (uint32_t)kappa2 : (uint32_t)kFitR;
        uint32_t Amin[NACC];
#pragma unroll
        for (int u = 0; u < NACC; ++u) Amin[u] = 0xFFFFFFFFu;
#pragma unroll 2
        for (int64_t q = q0; q < q1; ++q) {
            const uint32_t a = ((uint64_t)b.A[q] < kFitR ? (uint32_t)b.A[q] : (uint32_t)kFitR) + k2c; // A* = A + 2 kappa
            const int uq = acc_of<NACC>(b, q);
#pragma unroll
            for (int u = 0; u < NACC; ++u)
                if (u == uq) {
                    Sa[k][u] = umin(Sa[k][u] + a, (uint32_t)kFitR);
                    Ma[k][u] = umax(Ma[k][u], a);
                    Amin[u] = umin(Amin[u], a);
                    dla[k][u] += 1;
                }
        }
        uint32_t Stot = 0;
#pragma unroll
        for (int u = 0; u < NACC; ++u) Stot = umin(Stot + Sa[k][u], (uint32_t)kFitR);
        const uint64_t dl = (uint64_t)nq;
        const bool f = (uint64_t)T < kFitR && (uint64_t)D < kFitR && E < kFitR && Stot < kFitR && dl < kFitR &&
                       (eps == 0 || dl <= (kFitR - 1) / eps);
        fit &= f ? 1u : 0u;
        if (f) rdivisor((uint32_t)T, tm2[k], mg[k], lg[k]);
        Dv[k] = (uint32_t)D;
        Ev[k] = E;
        Emx[k] = Emax;
        dlt[k] = (uint32_t)dl;
        seg0[k] = (uint32_t)(q0 - seg_base);
#pragma unroll
        for (int u = 0; u < NACC; ++u) Amn[k][u] = dla[k][u] ? (Amin[u] < kFitR ? Amin[u] : 0u) : 0u;
    }
    Mask users[NACC];
#pragma unroll
    for (int u = 0; u < NACC; ++u) {
        bool us[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) us[k] = val[k] && dla[k][u] != 0;
        users[u] = ballot_slots<CPL>(us);
    }
    const Mask spins = ballot_slots<CPL>(sp);
    const Mask all = n >= N ? ~(Mask)0 : (((Mask)1 << n) - 1);
    if (rank_row) { // a candidate must be a permutation of 0..n-1
        rank_ok = __reduce_and_sync(kFull, rank_ok);
        Mask rb = __reduce_or_sync(kFull, (uint32_t)rbit);
        if constexpr (CPL == 2) rb |= (Mask)__reduce_or_sync(kFull, (uint32_t)((uint64_t)rbit >> 32)) << 32;
        if (!rank_ok || rb != all) {
            if (lane == 0) {
                atomicExch(p.err, PAAM_E_INVAL);
                if (p.cand_ok) p.cand_ok[row] = 0;
            }
            return;
        }
    }
    bool wide = !__reduce_and_sync(kFull, fit); // outside the 32-bit bound
    uint32_t dpart = 0, spart = 0;
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        dpart = umax(dpart, Dv[k]);
        if (val[k]) spart += umin(dlt[k], (uint32_t)kBigSegs + 1);
    }
    const uint32_t dmax = __reduce_max_sync(kFull, dpart);
    const uint32_t nseg = __reduce_add_sync(kFull, spart);
    wide |= dmax >= kNarrow - N; // inside it but not narrow
    if (SAFE) wide |= nseg > (uint32_t)kBigSegs;
    if (wide) {
        if (lane == 0) wide_list[atomicAdd(wide_count, 1)] = (int32_t)item;
        return;
    }
    // The system's iteration bound (as in analyze_lazy.cu): no recurrence of Eq. 3 or
    // Eq. 6 takes more than L = sum_h ceil(Dmax / T_h) + 2 evaluations; with L within
    // kIterCap the loops run without counters, otherwise every loop stops at kIterCap.
    uint32_t lpart = 0;
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        if (val[k]) lpart += umin(rarrivals(dmax, tm2[k], mg[k], lg[k]) - 1u, kIterCap + 1u);
    const bool counted = __reduce_add_sync(kFull, lpart) + 2u > kIterCap;

    // ---- relations (Lemma 4, Theorem 1, Eq. 3), analysis order ---------------
    Mask samex[CPL], corem[CPL], eqx[CPL], higher[CPL], ehigher[CPL];
    bool inside = true;
#pragma unroll
    for (int k = 0; k < CPL; ++k)
        inside &= !val[k] || ((uint32_t)ex[k] < N && (uint32_t)co[k] < N && (uint32_t)pr[k] < N &&
                              (!xprio || (uint32_t)ep[k] < N));
    if (__all_sync(kFull, inside)) {
        // keys below N index slots of shared memory into which each chain ORs its bit;
        // the set above a priority value is the OR of the slots past it
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int v = lane + 32 * k;
            s.xms[v] = s.cms[v] = s.exm[v] = s.inv[v] = 0;
            s.xep[v] = INT32_MIN;
        }
        __syncwarp();
        auto or_into = [](Mask *at, Mask bit) {
            if constexpr (CPL == 1) atomicOr((unsigned int *)at, (unsigned int)bit);
            else atomicOr((unsigned long long *)at, (unsigned long long)bit);
        };
#pragma unroll
        for (int k = 0; k < CPL; ++k)
            if (val[k]) {
                const Mask bit = (Mask)1 << (lane + 32 * k);
                or_into(&s.xms[ex[k]], bit);
                or_into(&s.cms[co[k]], bit);
                if (!xprio) atomicMax(&s.xep[ex[k]], pr[k]);
            }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const Mask bit = (Mask)1 << (lane + 32 * k);
            samex[k] = val[k] ? s.xms[ex[k]] : bit;
            corem[k] = val[k] ? s.cms[co[k]] : bit;
            if (!xprio && val[k]) ep[k] = s.xep[ex[k]]; // criticality-as-priority
            if (val[k]) {
                s.inv[pr[k]] = bit; // distinct priorities: one chain per slot
                or_into(&s.exm[ep[k]], bit);
            }
        }
        __syncwarp();
        Mask a[CPL], e[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            eqx[k] = val[k] ? s.exm[ep[k]] : (Mask)1 << (lane + 32 * k);
            a[k] = s.inv[lane + 32 * k];
            e[k] = s.exm[lane + 32 * k];
        }
        auto orop = [](Mask x, Mask y) { return x | y; };
        scan_above<CPL>(a, lane, orop);
        scan_above<CPL>(e, lane, orop);
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            higher[k] = slot_value<CPL>(a, val[k] ? pr[k] : 0);
            ehigher[k] = slot_value<CPL>(e, val[k] ? ep[k] : 0);
            if (!val[k]) higher[k] = ehigher[k] = all;
        }
    } else { // one comparison each per chain pair
        if (!xprio) { // criticality-as-priority: the highest chain priority on the executor
            int32_t best[CPL];
#pragma unroll
            for (int k = 0; k < CPL; ++k) best[k] = INT32_MIN;
            for (int t = 0; t < n; ++t) {
                const int32_t pt = slot_value<CPL>(pr, t), xt = slot_value<CPL>(ex, t);
#pragma unroll
                for (int k = 0; k < CPL; ++k)
                    if (xt == ex[k] && pt > best[k]) best[k] = pt;
            }
#pragma unroll
            for (int k = 0; k < CPL; ++k) ep[k] = best[k];
        }
#pragma unroll
        for (int k = 0; k < CPL; ++k) samex[k] = corem[k] = eqx[k] = higher[k] = ehigher[k] = 0;
        for (int t = 0; t < n; ++t) {
            const int32_t pt = slot_value<CPL>(pr, t), et = slot_value<CPL>(ep, t);
            const int32_t xt = slot_value<CPL>(ex, t), kt = slot_value<CPL>(co, t);
            const Mask bit = (Mask)1 << t;
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                samex[k] |= xt == ex[k] ? bit : 0;
                corem[k] |= kt == co[k] ? bit : 0;
                eqx[k] |= et == ep[k] ? bit : 0;
                higher[k] |= pt > pr[k] ? bit : 0;
                ehigher[k] |= et > ep[k] ? bit : 0;
            }
        }
#pragma unroll
        for (int k = 0; k < CPL; ++k)
            if (!val[k]) { // past n: only itself on its executor and core
                const Mask bit = (Mask)1 << (lane + 32 * k);
                samex[k] = corem[k] = eqx[k] = bit;
                higher[k] = ehigher[k] = all;
            }
    }
    const bool one_bucket = p.n_buckets == 1;
    int pos[CPL], prank[CPL];
    Mask hp[CPL], hpp[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int j = lane + 32 * k;
        // position in the analysis order: executor priority, then chain priority
        pos[k] = rpopc(ehigher[k]) + rpopc((Mask)(eqx[k] & higher[k] & all));
        hp[k] = samex[k] & higher[k];               // hp(c), Lemma 4
        hpp[k] = corem[k] & ~samex[k] & ehigher[k]; // hpp(c), Theorem 1
        prank[k] = rpopc(higher[k]);                // rank by chain priority, 0 = highest
        s.emax[j] = Emx[k];
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
            s.m[u][j] = Ma[k][u];
            if (val[k]) {
                s.ssort[u][prank[k]] = umin(Sa[k][u], kNarrow - 1); // 0 for a chain without segments on u
                s.msort[u][prank[k]] = Ma[k][u];
            }
        }
    }
    __syncwarp();
    uint32_t Bv[CPL], blk[CPL][NACC], sums[CPL][NACC];
    if constexpr (!SAFE) {
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            Bv[k] = 0;
            const Mask jb = (Mask)1 << (lane + 32 * k);
            for (Mask lo = samex[k] & ~higher[k] & ~jb & all; lo; lo &= lo - 1) // Lemma 4: one LP callback
                Bv[k] = umax(Bv[k], s.emax[rlowest(lo)]);
        }
    }
#pragma unroll
    for (int u = 0; u < NACC; ++u) {
        // sum_h S*_{h,u} over hps_u(c): a prefix sum in priority order, saturating at 2^27
        uint32_t a[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) a[k] = lane + 32 * k < n ? s.ssort[u][lane + 32 * k] : 0u;
        scan_below<CPL>(a, lane, [](uint32_t x, uint32_t y) { return umin(x + y, kNarrow); });
#pragma unroll
        for (int k = 0; k < CPL; ++k) sums[k][u] = slot_value<CPL>(a, prank[k] < N ? prank[k] : 0);
        if (one_bucket) { // every user of u shares its bucket: the longest lower-priority request (R2-R3)
#pragma unroll
            for (int k = 0; k < CPL; ++k) a[k] = lane + 32 * k < n ? s.msort[u][lane + 32 * k] : 0u;
            scan_above<CPL>(a, lane, [](uint32_t x, uint32_t y) { return umax(x, y); });
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                const uint32_t below = slot_value<CPL>(a, prank[k] < N ? prank[k] : 0);
                blk[k][u] = dla[k][u] ? below : 0u;
            }
        }
    }
    if (!one_bucket) { // bucket = floor(rank * n_buckets / |U_u|), rank among the users of u (R2)
#pragma unroll
        for (int u = 0; u < NACC; ++u)
#pragma unroll
            for (int k = 0; k < CPL; ++k)
                s.bucket[u][lane + 32 * k] =
                    dla[k][u] ? (int32_t)((uint32_t)rpopc((Mask)(users[u] & higher[k])) * (uint32_t)p.n_buckets /
                                          (uint32_t)rpopc(users[u]))
                              : -1;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < NACC; ++u)
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                blk[k][u] = 0;
                const int32_t bk = s.bucket[u][lane + 32 * k];
                if (dla[k][u])
                    for (Mask lo = users[u] & ~higher[k] & ~((Mask)1 << (lane + 32 * k)); lo; lo &= lo - 1) {
                        const int l = rlowest(lo);
                        if (s.bucket[u][l] == bk) blk[k][u] = umax(blk[k][u], s.m[u][l]);
                    }
            }
    }

    uint32_t hsum[CPL] = {}; // safe reading: Eq. 3's exact sum over the chain's segments (kInfR none, kCapR cut short)
    if constexpr (SAFE) {
        static_assert(NACC == 1, "the safe reading here: one accelerator");
        // every segment's fixed point h = A* + blk + sum over hps(c) of (ceil(h / T_t)
        // + 1) S*_t (Lemma 2), one segment per lane
#pragma unroll
        for (int k = 0; k < CPL; ++k)
            if (val[k]) {
                const int j = lane + 32 * k;
                s.x.dv[j] = make_uint4(tm2[k], mg[k], lg[k], Sa[k][0]);
                s.x.hps[j] = users[0] & higher[k];
                s.x.ch[j] = make_uint2(Dv[k], blk[k][0]);
                for (uint32_t i = 0; i < dlt[k]; ++i) s.x.segc[seg0[k] + i] = (uint8_t)j;
            }
        __syncwarp();
        for (uint32_t q = lane; q < nseg; q += 32) {
            const int c = s.x.segc[q];
            const Mask hps = s.x.hps[c];
            const uint2 ch = s.x.ch[c];
            const uint64_t base = (uint64_t)b.A[seg_base + q] + kappa2 + ch.y;
            uint64_t h = base; // the recurrence starts with the first two terms
            uint32_t out, evs = 0;
            for (;;) {
                if (h > ch.x) {
                    out = kInfR;
                    break;
                }
                if (counted && evs++ == kIterCap) {
                    out = kCapR;
                    break;
                }
                uint64_t sum = 0;
                for (Mask m = hps; m; m &= m - 1) {
                    const uint4 dv = s.x.dv[rlowest(m)];
                    const uint64_t term = (uint64_t)rarrivals((uint32_t)h, dv.x, dv.y, dv.z) * dv.w;
                    sum += term < kTermCap ? term : kTermCap;
                }
                const uint64_t nh = base + sum;
                if (nh == h) { // strictly increasing until here, bounded by D
                    out = (uint32_t)h;
                    break;
                }
                h = nh;
            }
            s.x.hq[q] = out;
        }
        __syncwarp();
        // the lane's chains: their callbacks' holds E_i + sum over the callback's segments
        // of (bound + eps), and Eq. 3's sum over all the chain's segments; a chain
        // without segments holds its executor for its longest callback
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            uint32_t hold = Emx[k];
            if (val[k] && dlt[k]) {
                const int64_t g = c0 + lane + 32 * k;
                const int64_t cb1 = b.chain_cb_off[g + 1];
                uint64_t Hsum = 0, hl = 0;
                bool seg_inf = false, hold_inf = false, capped = false;
                for (int64_t cb = b.chain_cb_off[g]; cb < cb1; ++cb) {
                    uint64_t t = (uint64_t)b.E[cb];
                    bool t_inf = false;
                    const uint32_t k1 = (uint32_t)(b.cb_seg_off[cb + 1] - seg_base);
                    for (uint32_t q = (uint32_t)(b.cb_seg_off[cb] - seg_base); q < k1; ++q) {
                        const uint32_t h = s.x.hq[q];
                        if (h >= kCapR) { // no bound
                            seg_inf = t_inf = true;
                            capped |= h == kCapR;
                        } else {
                            Hsum += h;
                            t += h + eps;
                        }
                    }
                    if (t_inf) hold_inf = true;
                    else if (t > hl) hl = t;
                }
                const uint64_t cap = (uint64_t)Dv[k] + 1;
                hsum[k] = capped ? kCapR : seg_inf ? kInfR : (uint32_t)(Hsum < cap ? Hsum : cap);
                hold = hold_inf || hl >= kHoldInf ? kHoldInf : (uint32_t)hl;
            }
            s.emax[lane + 32 * k] = hold;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            Bv[k] = 0;
            const Mask jb = (Mask)1 << (lane + 32 * k);
            for (Mask lo = samex[k] & ~higher[k] & ~jb & all; lo; lo &= lo - 1) // safe Lemma 4: the longest LP hold
                Bv[k] = umax(Bv[k], s.emax[rlowest(lo)]);
        }
    }

    // ---- own recurrence terms; chains known not to be schedulable --------------
    // (the bound of analyze_lazy.cu, its accelerator part summed over the
    // accelerators; not under the safe reading, whose blocking mostly decides)
    uint32_t own[CPL][NACC];
    Mask needs[CPL];
    uint32_t low[CPL];
    bool dead_[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        needs[k] = hp[k] | (hpp[k] & spins);
        low[k] = 0;
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
            const uint64_t own64 = (uint64_t)Sa[k][u] + (uint64_t)dla[k][u] * blk[k][u];
            own[k][u] = own64 < (uint64_t)Dv[k] + 1 ? (uint32_t)own64 : Dv[k] + 1; // above D: as D + 1
            const uint32_t f = ((uint64_t)Amn[k][u] + blk[k][u]) >= 1 ? 2u : 1u;
            if (dla[k][u]) low[k] = umin(low[k] + own[k][u] + f * sums[k][u], kNarrow);
        }
        low[k] = umin(Ev[k] + low[k] + (uint32_t)((uint64_t)dlt[k] * eps), kNarrow);
    }
    Mask alive = all;
    if (!SAFE && !counted) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < CPL; ++k) s.ssort[0][lane + 32 * k] = low[k]; // the scans above have read it
        __syncwarp();
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            low[k] += Bv[k];
            for (Mask m = hp[k]; m; m &= m - 1) low[k] = umin(low[k] + 2u * s.ssort[0][rlowest(m)], 1u << 31);
            dead_[k] = val[k] && low[k] > Dv[k];
        }
        Mask dead = ballot_slots<CPL>(dead_);
        for (;;) {
#pragma unroll
            for (int k = 0; k < CPL; ++k) dead_[k] = (needs[k] & dead) != 0;
            const Mask more = dead | ballot_slots<CPL>(dead_);
            if (more == dead) break;
            dead = more;
        }
        alive = all & ~dead;
    }
    Mask steps = 0; // the positions that take a step (none in a candidate that has failed already)
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int j = lane + 32 * k, at = pos[k];
        if (val[k]) s.needs[j] = needs[k];
        if (!((alive >> j) & 1)) continue;
        steps |= (Mask)1 << at;
        s.hp[at] = hp[k];
        s.hpp[at] = hpp[k];
        s.at[at] = make_uint2((uint32_t)j, seg0[k]);
        s.rec[at] = make_uint4(Dv[k], Bv[k] + Ev[k], (uint32_t)((uint64_t)dlt[k] * eps), dlt[k]);
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
            // Lemma 2's sum over the segments on u is at least own_u + lb_u, lb_u =
            // f delta_u sum_h S*_{h,u} (f = 2 if A*_u + blk_u >= 1)
            const uint64_t lb = (((uint64_t)Amn[k][u] + blk[k][u]) >= 1 ? 2 : 1) * (uint64_t)dla[k][u] * sums[k][u];
            s.acc[at][u] = make_uint4(own[k][u], SAFE ? hsum[k] : (lb < kNarrow ? (uint32_t)lb : kNarrow), blk[k][u],
                                      dla[k][u]);
            s.hps[at][u] = users[u] & higher[k];
        }
    }
    {
        uint32_t lo = __reduce_or_sync(kFull, (uint32_t)steps), hi = 0;
        if constexpr (CPL == 2) hi = __reduce_or_sync(kFull, (uint32_t)((uint64_t)steps >> 32));
        steps = (Mask)lo;
        if constexpr (CPL == 2) steps |= (Mask)hi << 32;
        if (rank_row && alive != all) steps = 0;
    }
    __syncwarp();

    // ---- Theorem 1 (Eq. 6), chain by chain -----------------------------------
    uint32_t Ehp[CPL], Ehpp[CPL], Rv[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        Ehp[k] = Ev[k];
        Ehpp[k] = Ev[k] + (sp[k] ? 0u : (uint32_t)((uint64_t)dlt[k] * eps));
        Rv[k] = 0;
    }
    Mask sched = 0;
    const uint32_t k2 = (uint32_t)kappa2;
    auto chains = [&](auto counted_tag) {
    constexpr bool CNT = decltype(counted_tag)::value;
    for (Mask left = steps; left; left &= left - 1) {
        const int step = rlowest(left);
        const uint2 at = s.at[step];
        const int c = (int)at.x;
        if (s.needs[c] & ~sched) { // a needed H*_h is not available (the chain is DEP)
            if (rank_row) break; // a candidate fails at its first unschedulable chain
            continue;
        }
        const uint4 rc = s.rec[step];
        const uint32_t D32 = rc.x, base = rc.y, deps = rc.z, dl = rc.w;
        const Mask hpc = s.hp[step], hppc = s.hpp[step];
        uint32_t cc[CPL], ac[NACC][CPL], ow[NACC], lb[NACC], Hs[NACC];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int j = lane + 32 * k;
            cc[k] = ((hpc >> j) & 1) ? Ehp[k] : (((hppc >> j) & 1) ? Ehpp[k] : 0u);
        }
        uint32_t h0 = 0, uses = 0; // uses: the accelerators of the chain's segments
        bool capped = false;
#pragma unroll
        for (int u = 0; u < NACC; ++u) {
            const uint4 ar = s.acc[step][u];
            const Mask hs_u = s.hps[step][u];
            ow[u] = ar.x;
            lb[u] = ar.w && !SAFE ? ar.y : kInfR; // kInfR: u unused by the chain, or its fixed points taken
            Hs[u] = ar.w && SAFE ? ar.y : kInfR;
            capped |= SAFE && ar.w && ar.y == kCapR; // a segment recurrence was cut short
#pragma unroll
            for (int k = 0; k < CPL; ++k) ac[u][k] = ((hs_u >> (lane + 32 * k)) & 1) ? Sa[k][u] : 0u;
            uses |= ar.w ? 1u << u : 0u;
            if (ar.w) h0 += ow[u]; // Lemma 2's sum on u is never below own_u
        }
        const bool cpu = (hpc | hppc) != 0; // the same in every lane
        // start: B + E + H* with the interference parts of Eq. 4 empty
        uint32_t R = base + (dl ? umin(h0, kNarrow) + deps : 0u);
        uint32_t hs = 0, ev = 0;
        bool ok = false;
        if (!capped && R <= D32) {
            for (;;) { // until no accelerator's fixed points are newly needed
                int need = -1;
                for (;;) {
                    if (CNT && ev++ == kIterCap) break;
                    uint32_t mu[CPL];
#pragma unroll
                    for (int k = 0; k < CPL; ++k) mu[k] = rarrivals(R, tm2[k], mg[k], lg[k]);
                    const uint32_t cs = cpu ? slots_sum<CPL>(mu, cc) : 0u;
                    hs = 0;
#pragma unroll
                    for (int u = 0; u < NACC; ++u) {
                        if (!((uses >> u) & 1)) continue; // the same in every lane
                        const uint32_t as = slots_sum<CPL>(mu, ac[u]);
                        if (as > lb[u] && need < 0) need = u;
                        hs += umin(Hs[u], ow[u] + as); // min(Eq. 3, Eq. 4) on u, summed (R1)
                    }
                    if (need >= 0) { // this evaluation is taken again once that sum is known
                        if (CNT) --ev;
                        break;
                    }
                    if (dl) hs = umin(hs, kNarrow) + deps; // Eq. 1
                    const uint32_t Rn = base + umin(hs, kNarrow) + cs;
                    if (Rn == R) {
                        ok = true;
                        break;
                    }
                    R = Rn;
                    if (R > D32) break;
                }
                if (need < 0) break;
                // Lemma 2 over the chain's segments on accelerator `need`: the sum matters
                // only below Eq. 4 at R = D on it (and below D + 1)
#pragma unroll
                for (int u = 0; u < NACC; ++u) {
                    if (u != need) continue;
                    lb[u] = kInfR;
                    uint32_t mu[CPL];
#pragma unroll
                    for (int k = 0; k < CPL; ++k) mu[k] = rarrivals(D32, tm2[k], mg[k], lg[k]);
                    const uint32_t lim = umin(ow[u] + slots_sum<CPL>(mu, ac[u]), D32 + 1);
                    const uint32_t blkc = s.acc[step][u].z;
                    const int64_t qb = seg_base + at.y;
                    uint32_t H32 = 0;
                    bool inf = false;
                    for (uint32_t q = 0; q < dl && !inf; ++q) {
                        if (acc_of<NACC>(b, qb + q) != u) continue; // the chain's segments on u
                        const uint32_t hb = (uint32_t)b.A[qb + q] + k2 + blkc;
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
#pragma unroll
                            for (int k = 0; k < CPL; ++k) mu[k] = rarrivals(h, tm2[k], mg[k], lg[k]);
                            const uint32_t nh = hb + slots_sum<CPL>(mu, ac[u]);
                            if (nh == h) break; // strictly increasing until here, bounded by D
                            h = nh;
                        }
                        H32 += h;
                    }
                    if (!inf) Hs[u] = H32;
                }
                if (capped) break; // a segment recurrence was cut short
            }
        }
        if (capped) { // no bound (PAAM_ST_ITERCAP)
#pragma unroll
            for (int k = 0; k < CPL; ++k)
                if (lane + 32 * k == c) Rv[k] = kCapR;
            if (rank_row) break;
            continue;
        }
        if (ok) {
            sched |= (Mask)1 << c;
#pragma unroll
            for (int k = 0; k < CPL; ++k)
                if (lane + 32 * k == c) {
                    Rv[k] = R;
                    Ehp[k] = Ev[k] + hs;
                    if (sp[k]) Ehpp[k] = Ev[k] + hs;
                }
        } else {
#pragma unroll
            for (int k = 0; k < CPL; ++k)
                if (ev > kIterCap && lane + 32 * k == c) Rv[k] = kCapR; // cut short (PAAM_ST_ITERCAP)
            if (rank_row) break;
        }
    }
    };
    if (counted)
        chains(std::true_type{});
    else
        chains(std::false_type{});

    // ---- outputs -------------------------------------------------------------
    if (rank_row) {
        if (lane == 0) {
            const bool ok = sched == all;
            if (p.cand_ok) p.cand_ok[row] = ok ? 1 : 0;
            if (ok) atomicMin(p.first_ok + sys, cand);
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        if (!val[k]) continue;
        const int j = lane + 32 * k;
        const bool ok = (sched >> j) & 1;
        R_out[c0 + j] = ok ? (int64_t)Rv[k] : -1;
        // DEP: skipped at its step, i.e. some chain of its DEP-rule set (all earlier in
        // the analysis order) is not schedulable
        st_out[c0 + j] = ok ? PAAM_ST_SCHED
                            : (Rv[k] == kCapR ? PAAM_ST_ITERCAP
                                              : ((s.needs[j] & ~sched) ? PAAM_ST_DEP : PAAM_ST_OVERRUN));
    }
    if (lane == 0 && verdict) verdict[sys] = sched == all ? 1 : 0;
}

constexpr int kWarps = 4; // systems per block
// The block's tables: 63.5 KB with four accelerators and 51.2 KB under the safe reading
// (up to 64 chains), above the 48 KB that need no attribute.
constexpr size_t kBigTables = 64 << 10;
static_assert(sizeof(BigSmem<2, PAAM_MAX_ACC, false>) * kWarps <= kBigTables &&
                  sizeof(BigSmem<2, 1, true>) * kWarps <= kBigTables,
              "the largest tables of a block");

template <int CPL, int NACC, bool SAFE>
__global__ void __launch_bounds__(32 * kWarps) analyze_lazy_big_kernel(const __grid_constant__ BatchDev b,
                                                                      const __grid_constant__ AnalysisParams p,
                                                                      int64_t *R, uint8_t *st, uint8_t *verdict,
                                                                      const int32_t *list, const int32_t *count,
                                                                      int32_t *wide_list, int32_t *wide_count)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BigSmem<CPL, NACC, SAFE> &s = reinterpret_cast<BigSmem<CPL, NACC, SAFE> *>(smem_raw)[threadIdx.x / 32];
    const int lane = threadIdx.x % 32;
    const int64_t n_items = (int64_t)*count;
    for_each_item<32>(p, n_items, threadIdx.x / 32, kWarps, lane, kFull, [&](int64_t i) {
        big_system<CPL, NACC, SAFE>(b, p, (int64_t)list[i], s, lane, R, st, verdict, wide_list, wide_count);
    });
}

template <int CPL, int NACC, bool SAFE>
int launch_big(const paam_batch *bt, const AnalysisParams &p, int64_t *R, uint8_t *st, uint8_t *verdict,
               int64_t max_items, cudaStream_t stream)
{
    const size_t smem = sizeof(BigSmem<CPL, NACC, SAFE>) * kWarps;
    auto kern = analyze_lazy_big_kernel<CPL, NACC, SAFE>;
    PAAM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    PAAM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kWarps, smem));
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (max_items + kWarps - 1) / kWarps;
    const int64_t cap = (int64_t)per_sm * bt->ctx->n_sm;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    AnalysisParams pq = p;
    if (pq.queue_batch > 0) pq.queue_batch = 1; // few systems per warp
    kern<<<(unsigned)blocks, 32 * kWarps, smem, stream>>>(batch_dev(bt), pq, R, st, verdict, bt->list_big, bt->counts,
                                                          bt->list_wide, bt->counts + 1);
    PAAM_CUDA_TRY(cudaGetLastError());
    return PAAM_OK;
}

template <int CPL>
int launch_width(const paam_batch *bt, const AnalysisParams &p, int64_t *R, uint8_t *st, uint8_t *verdict,
                 int64_t max_items, cudaStream_t stream)
{
    if (p.blocking_mode == 1) return launch_big<CPL, 1, true>(bt, p, R, st, verdict, max_items, stream);
    const unsigned long long used = bt->stats[ST_ACCMAX] + 1;
    static_assert(PAAM_MAX_ACC == 4, "instantiations below cover 2..4 accelerators");
    if (used >= 4) return launch_big<CPL, 4, false>(bt, p, R, st, verdict, max_items, stream);
    if (used == 3) return launch_big<CPL, 3, false>(bt, p, R, st, verdict, max_items, stream);
    return launch_big<CPL, 2, false>(bt, p, R, st, verdict, max_items, stream);
}

} // namespace

int paam_launch_lazy_big(const paam_batch *bt, int cpl, const AnalysisParams &p, int64_t *R, uint8_t *st,
                         uint8_t *verdict, int64_t max_items, cudaStream_t stream)
{
    return cpl == 1 ? launch_width<1>(bt, p, R, st, verdict, max_items, stream)
                    : launch_width<2>(bt, p, R, st, verdict, max_items, stream);
}
