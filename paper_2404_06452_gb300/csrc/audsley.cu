// audsley.cu -- Audsley-style priority seed on the GPU: a greedy assignment
// of chain priorities from the lowest level up, each step decided by the
// exact analysis (Sec. IV-F, Theorem 1) of trial orders.
//
// At step j of a system with n chains (level l = n - 1 - j, rank 0 highest)
// every unassigned chain c is a trial: the chains already placed keep their
// ranks (all below l), c takes rank l and the other unassigned chains take
// ranks 0 .. l-1 in deadline-monotonic order (D ascending, ties by index).  A
// trial's verdict is whether c itself is schedulable.  The first passing c in
// index order takes level l; if none passes, the unassigned chain with the
// largest D (ties: highest index) does.  The admission test is not
// OPA-compatible (bucket ranks, blocking and the DEP rule depend on the whole
// order), so the result is a seed for the exact search, not an optimum.
//
// Systems of up to 32 chains inside the narrow 32-bit bound (one accelerator,
// Lemma 4 as printed) run the whole greedy in one kernel (seed_kernel below).
// The others take one launch per level, every trial analysed by the exact int64
// kernel in target mode.
#include "cand_eval.cuh"

namespace {

using namespace paam_cand;

// ---- the whole greedy of a system in one kernel -----------------------------
// GPS groups of LG lanes work on one system: they try GPS candidates of a level at
// a time, in index order, and the first that passes ends the level, so few trials
// past it are run (a 16-chain system of the search workload passes after 37 trials
// on average, where a launch per level runs all 136).  A trial's ranks are built in
// registers: lane c holds chain c's place among the placed chains, or the set of
// chains before it in deadline-monotonic order, of which those still unassigned
// are counted.  Nothing of a trial goes to memory, and cand_eval.cuh evaluates
// only the chains that the target's verdict rests on.  The last level has one
// chain left, which takes it whether it passes or not: no trial.
//
// With many systems the trials themselves are the limit (issue, 58% of the slots,
// and the last systems' levels): one group per system.  A batch too small to fill
// the chip is bound by one system's chain of levels: two groups, or a whole block
// of 16 (LG = 16) or 8 (LG = 32).  10,000 systems of 16 chains: 0.37 ms, where the
// launches per level took 3.8 ms (trial rows 0.6, trials 3.0, picks 0.15).
template <int LG, int GPS>
__global__ void __launch_bounds__(256, LG == 16 ? 4 : 3)
    seed_kernel(const __grid_constant__ BatchDev b, int32_t n_buckets, uint64_t kappa2, uint64_t eps,
                const uint4 *__restrict__ recs_all, int32_t rec_stride, int32_t nmax, int16_t *__restrict__ rank_out,
                uint8_t *__restrict__ done)
{
    constexpr int GROUPS = 256 / LG;
    static_assert(GPS == 1 || GPS * LG == 32 || GPS == GROUPS, "groups of a warp, or of the block");
    __shared__ CandSmem<LG> sm[GROUPS];
    __shared__ int passed[GROUPS];
    const int grp = threadIdx.x / LG, lane = threadIdx.x % LG, sub = grp % GPS;
    const unsigned gm = rgroup_mask<LG>();
    CandSmem<LG> &s = sm[grp];
    const int64_t stride = (int64_t)gridDim.x * (GROUPS / GPS);
    for (int64_t sys = (int64_t)blockIdx.x * (GROUPS / GPS) + grp / GPS; sys < b.n_sys; sys += stride) {
        const int64_t c0 = b.sys_chain_off[sys];
        const int n = (int)(b.sys_chain_off[sys + 1] - c0);
        if (n == 0 || n > LG || (LG == 32 && n <= 16)) continue; // the other width's, or the launches per level
        const uint4 *recs = recs_all + sys * rec_stride * 4;
        const uint32_t sysfl = recs[2].w;
        if (!(sysfl & kRecFit) || !(sysfl & (LG == 16 ? kRecNarrow16 : kRecNarrow32))) continue;
        const int64_t seg_base = b.cb_seg_off[b.chain_cb_off[c0]];
        const bool val = lane < n;
        const uint32_t D = val ? recs[4 * lane].w : 0xFFFFFFFFu;
        uint32_t before = 0; // chains ahead of this one in deadline-monotonic order
        for (int t = 0; t < n; ++t) {
            const uint32_t Dt = __shfl_sync(gm, D, t, LG);
            before |= (Dt < D || (Dt == D && t < lane)) ? 1u << t : 0u;
        }
        uint32_t un = n >= 32 ? ~0u : (1u << n) - 1u; // unassigned chains
        int rank = 0;                                 // of a placed chain
        for (int level = n - 1; level > 0; --level) {
            int pick = -1;
            uint32_t rest = un;
            // every group of the system keeps the same un, rest and pick
            while (rest && pick < 0) {
                uint32_t mine = rest; // this group's trial: the sub-th unassigned chain not tried yet
                for (int k = 0; k < sub && mine; ++k) mine &= mine - 1;
                bool ok = false;
                int c = -1;
                if (mine) {
                    c = __ffs(mine) - 1;
                    __syncwarp(gm);
                    const int r = ((un >> lane) & 1) ? (lane == c ? level : __popc(before & un & ~(1u << c))) : rank;
                    if (val) s.ord[r] = (uint32_t)lane;
                    __syncwarp(gm);
                    const int chain = val ? (int)s.ord[lane] : 0;
                    ok = cand_eval<LG, true>(b, n_buckets, kappa2, eps, n, seg_base, recs, chain, level, s, lane, gm);
                }
                if (GPS == 1) {
                    if (ok) pick = c;
                } else {
                    if (lane == 0) passed[grp] = ok ? c : -1;
                    if (GPS == GROUPS) __syncthreads();
                    else __syncwarp();
                    for (int k = 0; k < GPS; ++k) {
                        const int v = passed[grp - sub + k];
                        if (pick < 0 && v >= 0) pick = v;
                    }
                    if (GPS == GROUPS) __syncthreads();
                    else __syncwarp();
                }
                for (int k = 0; k < GPS; ++k) rest &= rest - 1;
            }
            if (pick < 0) { // the largest deadline, ties: the highest index (D < 2^27)
                const uint32_t key = ((un >> lane) & 1) ? (D << 5) | (uint32_t)lane : 0u;
                pick = (int)(__reduce_max_sync(gm, key) & 31u);
            }
            un &= ~(1u << pick);
            if (lane == pick) rank = level;
        }
        if (sub == 0) {
            if (val) rank_out[sys * nmax + lane] = (int16_t)rank; // the last unassigned chain: rank 0
            if (lane == 0) done[sys] = 1;
        }
    }
}

template <int LG, int GPS>
int launch_seed(const paam_batch *bt, const paam_analysis_opts *o, const uint4 *recs, int32_t rec_stride, int32_t nmax,
                int16_t *rank, uint8_t *done, int64_t blocks_cap, cudaStream_t stream)
{
    const int64_t per_block = 256 / LG / GPS;
    int64_t blocks = (bt->n_sys + per_block - 1) / per_block;
    if (blocks > blocks_cap) blocks = blocks_cap;
    seed_kernel<LG, GPS><<<(unsigned)blocks, 256, 0, stream>>>(batch_dev(bt), o->n_buckets, 2 * (uint64_t)o->kappa_ns,
                                                               (uint64_t)o->eps_ns, recs, rec_stride, nmax, rank, done);
    PAAM_CUDA_TRY(cudaGetLastError());
    return PAAM_OK;
}

// Groups per system by how many systems there are for the resident groups.
template <int LG>
int launch_seed_width(const paam_batch *bt, const paam_analysis_opts *o, const uint4 *recs, int32_t rec_stride,
                      int32_t nmax, int16_t *rank, uint8_t *done, cudaStream_t stream)
{
    const int64_t cap = (LG == 16 ? 4 : 3) * (int64_t)bt->ctx->n_sm; // resident blocks
    if (bt->n_sys <= cap) return launch_seed<LG, 256 / LG>(bt, o, recs, rec_stride, nmax, rank, done, cap, stream);
    if (LG == 16 && bt->n_sys * 2 <= cap * 16)
        return launch_seed<LG, 32 / LG>(bt, o, recs, rec_stride, nmax, rank, done, cap, stream);
    return launch_seed<LG, 1>(bt, o, recs, rec_stride, nmax, rank, done, cap, stream);
}

// ---- a launch per level -------------------------------------------------------
// trial t of system s at step j: ranks row and target chain (none for a system
// the kernel above has done)
__global__ void audsley_trials(BatchDev b, int32_t j, int32_t Kc, int32_t nmax, const uint8_t *__restrict__ done,
                               const int16_t *__restrict__ rank, int16_t *__restrict__ trial,
                               int16_t *__restrict__ target)
{
    const int64_t items = b.n_sys * (int64_t)Kc;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += stride) {
        const int64_t s = i / Kc;
        const int t = (int)(i - s * Kc);
        const int64_t c0 = b.sys_chain_off[s];
        const int n = (int)(b.sys_chain_off[s + 1] - c0);
        const int16_t *rs = rank + s * nmax;
        if (j >= n || t >= n - j || done[s]) {
            target[i] = -1;
            continue;
        }
        int c = -1; // the t-th unassigned chain by index
        for (int k = 0, seen = 0; k < n; ++k)
            if (rs[k] < 0 && seen++ == t) {
                c = k;
                break;
            }
        const int level = n - 1 - j;
        int16_t *row = trial + i * nmax;
        for (int k = 0; k < n; ++k) {
            int16_t r;
            if (rs[k] >= 0) {
                r = rs[k];
            } else if (k == c) {
                r = (int16_t)level;
            } else { // position among the other unassigned chains, deadline-monotonic
                const int64_t Dk = b.D[c0 + k];
                int pos = 0;
                for (int u = 0; u < n; ++u) {
                    if (u == c || u == k || rs[u] >= 0) continue;
                    const int64_t Du = b.D[c0 + u];
                    pos += (Du < Dk || (Du == Dk && u < k));
                }
                r = (int16_t)pos;
            }
            row[k] = r;
        }
        target[i] = (int16_t)c;
    }
}

// step j: the first passing trial, else the largest deadline, takes level n-1-j
__global__ void audsley_pick(BatchDev b, int32_t j, int32_t Kc, int32_t nmax, const uint8_t *__restrict__ done,
                             int16_t *__restrict__ rank, const int16_t *__restrict__ target,
                             const uint8_t *__restrict__ ok)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < b.n_sys; s += stride) {
        const int64_t c0 = b.sys_chain_off[s];
        const int n = (int)(b.sys_chain_off[s + 1] - c0);
        if (j >= n || done[s]) continue;
        int16_t *rs = rank + s * nmax;
        int chosen = -1;
        for (int t = 0; t < n - j && chosen < 0; ++t)
            if (ok[s * Kc + t]) chosen = target[s * Kc + t];
        if (chosen < 0)
            for (int k = 0; k < n; ++k)
                if (rs[k] < 0 && (chosen < 0 || b.D[c0 + k] >= b.D[c0 + chosen])) chosen = k;
        rs[chosen] = (int16_t)(n - 1 - j);
    }
}

constexpr size_t kTrialBytes = (size_t)512 << 20; // chain records and trial rank rows held at once

} // namespace

extern "C" int paam_rta_audsley_order(paam_ctx *ctx, const paam_batch *b, const paam_analysis_opts *o,
                                      int32_t nmax, int16_t *ranks_out, void *stream_)
{
    if (!ctx || !b || !o) return PAAM_E_INVAL;
    if (b->ctx != ctx) return PAAM_E_STATE;
    if (o->n_buckets < 1 || o->eps_ns < 0 || o->kappa_ns < 0) return PAAM_E_INVAL;
    if (o->eps_ns > PAAM_MAX_OVERHEAD || o->kappa_ns > PAAM_MAX_OVERHEAD) return PAAM_E_RANGE;
    if (o->blocking_mode != 0 && o->blocking_mode != 1) return PAAM_E_INVAL;
    if (nmax < 1 || nmax < b->max_chains || (b->n_sys > 0 && !ranks_out)) return PAAM_E_INVAL;
    if (b->n_sys == 0) return PAAM_OK;
    PAAM_CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t stream = (cudaStream_t)stream_;
    const int32_t Kc = b->max_chains > 0 ? b->max_chains : 1; // trials per system at step 0
    // the kernel for the whole greedy serves one accelerator, Lemma 4 as printed and
    // up to 32 chains; the launches per level follow unless it is known to take all
    const bool fused = !b->acc && o->blocking_mode == 0;
    const bool levels = !fused || b->max_chains > 32 || !paam_batch_fits_32(b, o) ||
                        b->stats[ST_DMAX] >= kLazyNarrowD - 16;
    const size_t rec_row = fused ? 64 * (size_t)Kc : 0;
    const size_t per_sys =
        rec_row + 1 + (levels ? (size_t)Kc * ((size_t)nmax * sizeof(int16_t) + sizeof(int16_t) + 1) : 0);
    int64_t chunk = (int64_t)(kTrialBytes / per_sys);
    if (chunk < 1) chunk = 1;
    if (chunk > b->n_sys) chunk = b->n_sys;
    if (chunk * (int64_t)Kc > (int64_t)INT32_MAX) chunk = INT32_MAX / Kc;

    void *tmp = nullptr;
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t rec_bytes = up((size_t)chunk * rec_row), done_bytes = up((size_t)chunk);
    const size_t trial_bytes = levels ? up((size_t)chunk * Kc * nmax * sizeof(int16_t)) : 0;
    const size_t target_bytes = levels ? up((size_t)chunk * Kc * sizeof(int16_t)) : 0;
    const size_t ok_bytes = levels ? up((size_t)chunk * Kc) : 0;
    if (cudaMallocAsync(&tmp, rec_bytes + done_bytes + trial_bytes + target_bytes + ok_bytes + 256, stream) !=
        cudaSuccess) {
        cudaGetLastError();
        return PAAM_E_NOMEM;
    }
    uint4 *recs = (uint4 *)tmp;
    uint8_t *done = (uint8_t *)tmp + rec_bytes;
    int16_t *trial = (int16_t *)(done + done_bytes);
    int16_t *target = (int16_t *)((char *)trial + trial_bytes);
    uint8_t *ok = (uint8_t *)target + target_bytes;
    int32_t *err = (int32_t *)(ok + ok_bytes);

    int rc = PAAM_OK;
    unsigned launches = 0;
    const int threads = 256;
    const int cap = 8 * ctx->n_sm;
    if (cudaMemsetAsync(err, 0, sizeof(int32_t), stream) != cudaSuccess ||
        cudaMemsetAsync(ranks_out, 0xff, (size_t)b->n_sys * nmax * sizeof(int16_t), stream) != cudaSuccess) // -1
        rc = PAAM_E_CUDA;
    for (int64_t s0 = 0; s0 < b->n_sys && rc == PAAM_OK; s0 += chunk) {
        paam_batch sub = *b; // systems [s0, s0 + m): chain offsets stay absolute
        const int64_t m = b->n_sys - s0 < chunk ? b->n_sys - s0 : chunk;
        sub.n_sys = m;
        sub.sys_chain_off = b->sys_chain_off + s0;
        sub.sys_exec_off = b->sys_exec_off + s0;
        sub.sys_order = nullptr; // the whole batch's order does not index a chunk
        const BatchDev bd = batch_dev(&sub);
        int16_t *rank = ranks_out + s0 * nmax;
        AnalysisParams p = {};
        p.n_buckets = o->n_buckets;
        p.eps = o->eps_ns;
        p.kappa = o->kappa_ns;
        p.blocking_mode = o->blocking_mode;
        if (levels && cudaMemsetAsync(done, 0, (size_t)m, stream) != cudaSuccess) rc = PAAM_E_CUDA;
        if (fused && rc == PAAM_OK) {
            rc = paam_launch_chain_records(&sub, p, recs, stream, Kc);
            if (rc == PAAM_OK) rc = launch_seed_width<16>(&sub, o, recs, Kc, nmax, rank, done, stream);
            launches += 1;
            if (rc == PAAM_OK && b->max_chains > 16) {
                rc = launch_seed_width<32>(&sub, o, recs, Kc, nmax, rank, done, stream);
                launches += 1;
            }
        }
        if (!levels) continue;
        p.K = Kc;
        p.Kc = Kc;
        p.ranks = trial;
        p.n_sys = m;
        p.nmax = nmax;
        p.cand_ok = ok;
        p.err = err;
        p.target = target;
        const int64_t items = m * (int64_t)Kc;
        int tb = (int)((items + threads - 1) / threads);
        if (tb > cap) tb = cap;
        int sb = (int)((m + threads - 1) / threads);
        if (sb > cap) sb = cap;
        for (int32_t j = 0; j < b->max_chains && rc == PAAM_OK; ++j) {
            audsley_trials<<<tb, threads, 0, stream>>>(bd, j, Kc, nmax, done, rank, trial, target);
            if (cudaGetLastError() != cudaSuccess) rc = PAAM_E_CUDA;
            if (rc == PAAM_OK) rc = paam_launch_wide(&sub, p, nullptr, nullptr, nullptr, nullptr, nullptr, items, stream);
            if (rc == PAAM_OK) {
                audsley_pick<<<sb, threads, 0, stream>>>(bd, j, Kc, nmax, done, rank, target, ok);
                if (cudaGetLastError() != cudaSuccess) rc = PAAM_E_CUDA;
            }
            launches += 3;
        }
    }
    paam_count_launch(launches);
    int32_t herr = 0;
    if (cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, stream) != cudaSuccess) rc = PAAM_E_CUDA;
    cudaFreeAsync(tmp, stream);
    if (cudaStreamSynchronize(stream) != cudaSuccess) rc = PAAM_E_CUDA;
    if (rc == PAAM_OK && herr != 0) rc = herr;
    return rc;
}
