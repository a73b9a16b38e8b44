// analyze_cand.cu -- the candidate mode of the priority search (search.cu) for
// systems of up to 32 chains with chain records: one (system, candidate) item per
// group of 16 or 32 lanes, decided by cand_eval.cuh.  The 16-lane pass takes
// every item; systems of more than 16 chains or outside its narrow bound go to
// the deferral list for the 32-lane pass and, above 32 chains, the 64-chain
// kernel, systems outside the 32-bit bound to the int64 kernel's list.
// Bound by issue (310 executed warp instructions per order, 68% of the issue
// slots).  10,000 systems x 256 orders of 16 chains: 3.03 -> 0.96 ms against the
// lazy kernel's candidate mode on the same records; four blocks per SM (64
// registers) beat five with spills by 7% and three by 16%.
#include "cand_eval.cuh"

namespace {
using namespace paam_cand;

template <int LG>
__device__ __forceinline__ void cand_item(const BatchDev &b, const AnalysisParams &p, int64_t item, CandSmem<LG> &s,
                                          int lane, unsigned gm, int32_t *big_list, int32_t *big_count,
                                          int32_t *wide_list, int32_t *wide_count)
{
    int64_t sys;
    int32_t cand;
    item_of(p, item, sys, cand);
    if (p.early) { // a candidate above the best schedulable one found so far
        const int pruned = __shfl_sync(gm, cand_pruned(p, sys, cand) ? 1 : 0, 0, LG);
        if (pruned) return;
    }
    const int64_t c0 = b.sys_chain_off[sys];
    const int n = (int)(b.sys_chain_off[sys + 1] - c0);
    if (n > LG) { // the 64-chain kernel's; the first pass appends it to its list
        if (LG == 16 && lane == 0) big_list[atomicAdd(big_count, 1)] = (int32_t)item;
        return;
    }
    const int64_t row = sys * p.Kc + cand_of(p, sys, cand);
    const uint4 *recs = p.chain_recs + c0 * 4;
    // the ranks: a permutation of 0..n-1; lane r then takes the chain of rank r
    const bool val = lane < n;
    const int r = val ? p.ranks[row * p.nmax + lane] : -1;
    const bool in = r >= 0 && r < n;
    const uint32_t sysfl = n > 0 ? recs[2].w : (kRecFit | kRecNarrow16 | kRecNarrow32);
    const int64_t seg_base = n > 0 ? b.cb_seg_off[b.chain_cb_off[c0]] : 0;
    __syncwarp(gm);
    if (in) s.ord[r] = (uint32_t)lane;
    const uint32_t bits = __reduce_or_sync(gm, in ? 1u << r : 0u);
    if (bits != (n >= 32 ? ~0u : (1u << n) - 1u)) {
        if (lane == 0) {
            atomicExch(p.err, PAAM_E_INVAL);
            if (p.cand_ok) p.cand_ok[row] = 0;
        }
        return;
    }
    if (!(sysfl & kRecFit)) { // outside the 32-bit bound
        if (lane == 0) wide_list[atomicAdd(wide_count, 1)] = (int32_t)item;
        return;
    }
    if (!(sysfl & (LG == 16 ? kRecNarrow16 : kRecNarrow32))) { // inside it but not narrow
        if (lane == 0) {
            if (LG == 16) big_list[atomicAdd(big_count, 1)] = (int32_t)item;
            else wide_list[atomicAdd(wide_count, 1)] = (int32_t)item;
        }
        return;
    }
    __syncwarp(gm);
    const int chain = val ? (int)s.ord[lane] : 0;
    const bool ok = cand_eval<LG, false>(b, p.n_buckets, 2 * (uint64_t)p.kappa, (uint64_t)p.eps, n, seg_base, recs,
                                         chain, 0, s, lane, gm);
    if (lane == 0) {
        if (p.cand_ok) p.cand_ok[row] = ok ? 1 : 0;
        if (ok) atomicMin(p.first_ok + sys, cand);
    }
}

template <int LG>
__global__ void __launch_bounds__(256, 4)
    analyze_cand_kernel(const __grid_constant__ BatchDev b, const __grid_constant__ AnalysisParams p,
                        const int32_t *list, const int32_t *count, int32_t *big_list, int32_t *big_count,
                        int32_t *wide_list, int32_t *wide_count)
{
    __shared__ CandSmem<LG> sm[256 / LG];
    const int groups = 256 / LG, grp = threadIdx.x / LG, lane = threadIdx.x % LG;
    const unsigned gm = rgroup_mask<LG>();
    const int64_t n_items = list ? (int64_t)*count : b.n_sys * p.K;
    for_each_item<LG>(p, n_items, grp, groups, lane, gm, [&](int64_t i) {
        cand_item<LG>(b, p, list ? (int64_t)list[i] : i, sm[grp], lane, gm, big_list, big_count, wide_list,
                      wide_count);
    });
}

} // namespace

template <int LG>
int launch_cand(const paam_batch *bt, const AnalysisParams &p, const int32_t *list, const int32_t *count,
                int64_t max_items, cudaStream_t stream)
{
    auto kern = analyze_cand_kernel<LG>;
    int per_sm = 0;
    PAAM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, 0));
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (max_items + 256 / LG - 1) / (256 / LG);
    const int64_t cap = (int64_t)per_sm * bt->ctx->n_sm;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    AnalysisParams pc = p;
    // items per queue fetch: a candidate is short, and with 2 the fetches cost 4%; 8
    // cost an early-exit search of few systems 5%
    if (pc.queue_batch > 0) pc.queue_batch = 4;
    kern<<<(unsigned)blocks, 256, 0, stream>>>(batch_dev(bt), pc, list, count, bt->list_big, bt->counts,
                                               bt->list_wide, bt->counts + 1);
    PAAM_CUDA_TRY(cudaGetLastError());
    return PAAM_OK;
}

template int launch_cand<16>(const paam_batch *, const AnalysisParams &, const int32_t *, const int32_t *, int64_t,
                             cudaStream_t);
template int launch_cand<32>(const paam_batch *, const AnalysisParams &, const int32_t *, const int32_t *, int64_t,
                             cudaStream_t);
