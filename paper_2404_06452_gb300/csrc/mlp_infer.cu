// mlp_infer.cu -- the surrogate's four layers over many rows and each row's score in one
// persistent kernel (tcgen05 + TMA + TMEM on sm_103a), for inputs of up to 256 columns.
//
// A kernel per layer reads and writes 512 bytes of activations per row between any two
// layers and runs at that traffic's rate: 2.56 M rows took 3 x 390 + 217 us at 6.7 TB/s.
// Here a row's activations stay in shared memory from its features to its score.  Each
// CTA has two tiles of 128 rows in turn: while the tensor core works on one tile, the
// epilogue warps turn the other's accumulator (256 TMEM columns each) into its next
// operand, in place.  2.56 M rows of 256 features: 960 us.  What bounds it are the
// activation's two special-function results per element (3,070 of the 3,500 cycles of a
// tile and layer) and, once per tile, the way from the last activations to the next tile's
// first accumulator, 6,400 cycles of which the other tile's activations hide half.  Weights
// stream through a ring from L2, once per tile and layer: both tiles' activations and a
// whole layer's weights together do not fit in shared memory.
//
// With one lane of the MMA warp waiting and issuing by itself each step's 16 MMAs took
// 4,400 cycles to issue (1,265 us in all); the whole warp waiting and one elected lane
// issuing takes 2,200.
//
//   warp 0       weights, stages of 64 columns of a layer (32 KB)
//   warp 1       MMAs, in the order  L0 L0 | L1 L1 L2 L2 L3 L0' L3 L0' | ... of the two tiles
//   warp 2       the tiles' features, each block as soon as the tile before has left it
//   warps 4-19   bias, activation and bf16 operand of layers 0 to 2, in the tiles' turn
//   warps 20-23  the outputs' maximum (beside the other tile's activations)
//
// The sums are those of a kernel per layer, in the same order: the scores' bits are the same.
#include "gelu.cuh"
#include "mlp.cuh"
#include "tc.cuh"

namespace {
using namespace paam_gelu;

constexpr int BM = 128, BK = 64, kHidden = 256, kIn = 1024, kOutCols = 16;
constexpr int kBlocks = kHidden / BK;                // operand blocks of a tile
constexpr int kA = BM * BK * 2, kTile = kBlocks * kA; // a tile's activations
constexpr int kStages = 3, kStage = kHidden * BK * 2, kOutBlock = kOutCols * BK * 2;
constexpr int kTiles = 2 * kTile + kStages * kStage;
constexpr int kSmem = kTiles + 256 + 1024; // barriers and flags, alignment slack
static_assert(kSmem <= 227 * 1024, "one CTA's shared memory");
constexpr int kEpiWarps = 16, kEpi0 = 4, kOut0 = kEpi0 + kEpiWarps, kThreads = 32 * (kOut0 + 4);
constexpr uint64_t kWaitNs = 2000000000ull; // 2 s: far above any legitimate wait

struct ScoreMaps {
    CUtensorMap X;    // [rows][kx]
    CUtensorMap W[4]; // [out][in]
};

// The CTA's u-th tile in place t (0, 1); past the last: m_tiles or more
__device__ __forceinline__ int tile_of(int u, int t) { return (int)blockIdx.x + (2 * u + t) * (int)gridDim.x; }

// The order of the layers' MMAs: f(layer, place, u) for each, until one fails
template <class F>
__device__ __forceinline__ bool walk(int m_tiles, F f)
{
    for (int t = 0; t < 2; ++t)
        if (tile_of(0, t) < m_tiles && !f(0, t, 0)) return false;
    for (int u = 0; tile_of(u, 0) < m_tiles; ++u) {
        for (int i = 0; i < 8; ++i) {
            // 1 1 2 2 3 0' 3 0'
            const int t = i < 4 ? (i & 1) : (i - 4) >> 1;
            const int l = i < 4 ? 1 + (i >> 1) : ((i & 1) ? 0 : 3), v = u + (l == 0);
            if (tile_of(v, t) < m_tiles && !f(l, t, v)) return false;
        }
    }
    return true;
}

__global__ void __launch_bounds__(kThreads, 1)
    score_chain_kernel(const __grid_constant__ ScoreMaps maps, const __grid_constant__ ScoreChain c)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *ring = smem + 2 * kTile;
    uint64_t *full = (uint64_t *)(smem + kTiles);
    uint64_t *empty = full + kStages;
    uint64_t *xfull = empty + kStages;     // [place][block]: features have landed
    uint64_t *xfree = xfull + 2 * kBlocks; // [place][block]: layer 3 has read the block
    uint64_t *acc = xfree + 2 * kBlocks;   // [place]: layer 0, 1 or 2 is complete
    uint64_t *acc_out = acc + 2;           // [place]: layer 3 is
    uint64_t *ready = acc_out + 2;         // [place]: the accumulator is read, the next operand written
    uint64_t *out_read = ready + 2;        // [place]: the outputs are read
    uint64_t *fin = out_read + 2;
    uint32_t *tmem_slot = (uint32_t *)(fin + 1);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    volatile int *issued = abort_flag + 1, *x_issued = abort_flag + 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m_tiles = (c.rows + BM - 1) / BM, kb0 = c.kx / BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2 * kBlocks; ++i) {
            tc::mbar_init(&xfull[i], 1);
            tc::mbar_init(&xfree[i], 1);
        }
        for (int t = 0; t < 2; ++t) {
            tc::mbar_init(&acc[t], 1);
            tc::mbar_init(&acc_out[t], 1);
            tc::mbar_init(&ready[t], kEpiWarps);
            tc::mbar_init(&out_read[t], 4);
        }
        tc::mbar_init(fin, 1);
        *abort_flag = 0;
        *issued = 0;
        *x_issued = 0;
        tc::fence_barrier_init();
        tc::prefetch_tmap(&maps.X);
        for (int l = 0; l < 4; ++l) tc::prefetch_tmap(&maps.W[l]);
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, 2 * kHidden);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    auto give_up = [&]() {
        *abort_flag = 1;
        atomicExch(c.err, PAAM_E_TIMEOUT);
    };

    if (warp == 0 && lane == 0) { // ---- weights
        int it = 0;
        const bool ok = walk(m_tiles, [&](int l, int, int) {
            const int stages = l == 0 ? kb0 : (l == 3 ? 1 : kBlocks);
            for (int i = 0; i < stages; ++i, ++it) {
                const int s = it % kStages, r = it / kStages;
                if (*abort_flag || (r > 0 && !tc::mbar_wait(&empty[s], (r - 1) & 1, kWaitNs))) return false;
                uint8_t *w = ring + s * kStage;
                tc::mbar_expect_tx(&full[s], l == 3 ? kBlocks * kOutBlock : kStage);
                if (l == 3) // all of it in one stage
                    for (int kb = 0; kb < kBlocks; ++kb) tc::tma_load_2d(w + kb * kOutBlock, &maps.W[3], &full[s], kb * BK, 0);
                else
                    tc::tma_load_2d(w, &maps.W[l], &full[s], i * BK, 0);
            }
            return true;
        });
        *issued = it;
        if (!ok) give_up();
    } else if (warp == 1) { // ---- MMA issuer: the warp waits as one, one lane issues
        int s = 0;
        uint32_t round = 0;
        const uint32_t lead = tc::elect_one();
        const uint32_t a0 = tc::smem_u32(smem), w0 = tc::smem_u32(ring);
        const uint32_t d0 = __shfl_sync(0xffffffffu, tmem, 0);
        const bool ok = walk(m_tiles, [&](int l, int t, int u) {
            // no vote here: the warp executes nothing together before the __syncwarp at the
            // end, where a lane that gives up waits for the others
            if (*abort_flag) return false;
            if (l > 0 ? !tc::mbar_wait(&ready[t], (3 * u + l - 1) & 1, kWaitNs)
                      : (u > 0 && !tc::mbar_wait(&out_read[t], (u - 1) & 1, kWaitNs)))
                return false;
            tc::fence_after_sync();
            const uint32_t idesc = l == 3 ? tc::idesc_bf16(BM, kOutCols) : tc::idesc_bf16(BM, kHidden);
            const int blocks = l == 0 ? kb0 : kBlocks;
            for (int kb = 0; kb < blocks; ++kb) {
                if (l == 0 && !tc::mbar_wait(&xfull[t * kBlocks + kb], u & 1, kWaitNs)) return false;
                if ((l < 3 || kb == 0) && !tc::mbar_wait(&full[s], round, kWaitNs)) return false;
                if (lead) {
                    const uint64_t a = tc::desc_sw128(a0 + t * kTile + kb * kA);
                    const uint64_t w = tc::desc_sw128(w0 + s * kStage + (l == 3 ? kb * kOutBlock : 0));
#pragma unroll
                    for (int j = 0; j < BK / 16; ++j)
                        tc::mma_bf16(d0 + (uint32_t)(t * kHidden), a + 2 * j, w + 2 * j, idesc, (kb > 0 || j > 0) ? 1u : 0u);
                    if (l < 3 || kb == kBlocks - 1) tc::mma_commit(&empty[s]);
                    if (l == 3) tc::mma_commit(&xfree[t * kBlocks + kb]);
                }
                if ((l < 3 || kb == kBlocks - 1) && ++s == kStages) {
                    s = 0;
                    round ^= 1;
                }
            }
            if (lead) tc::mma_commit(l == 3 ? &acc_out[t] : &acc[t]);
            return true;
        });
        if (!ok && lead) give_up();
        // every MMA issued has completed before TMEM can be released
        if (lead) {
            tc::mma_commit(fin);
            tc::mbar_wait(fin, 0, kWaitNs);
        }
        __syncwarp();
    } else if (warp == 2 && lane == 0) { // ---- features
        int n = 0;
        bool ok = true;
        for (int u = 0; ok && tile_of(u, 0) < m_tiles; ++u)
            for (int t = 0; ok && t < 2; ++t) {
                const int tile = tile_of(u, t), ahead = tile_of(u + 1, t);
                if (tile >= m_tiles) continue;
                if (ahead < m_tiles) // the place's next tile comes into L2 meanwhile
                    for (int kb = 0; kb < kb0; ++kb) tc::tma_prefetch_2d(&maps.X, kb * BK, ahead * BM);
                for (int kb = 0; kb < kb0; ++kb, ++n) {
                    if (*abort_flag || (u > 0 && !tc::mbar_wait(&xfree[t * kBlocks + kb], (u - 1) & 1, kWaitNs))) {
                        give_up();
                        ok = false;
                        break;
                    }
                    tc::mbar_expect_tx(&xfull[t * kBlocks + kb], kA);
                    tc::tma_load_2d(smem + t * kTile + kb * kA, &maps.X, &xfull[t * kBlocks + kb], kb * BK, tile * BM);
                }
            }
        *x_issued = n;
    } else if (warp >= kEpi0 && warp < kOut0) { // ---- activations: one row per thread, 64 columns per warp
        const int q = warp & 3, cg = (warp - kEpi0) >> 2; // TMEM lane quadrant, operand block
        const int tr = 32 * q + lane;
        bool ok = true;
        for (int u = 0; ok && tile_of(u, 0) < m_tiles; ++u)
            for (int i = 0; i < 6; ++i) {
                const int l = i >> 1, t = i & 1;
                if (tile_of(u, t) >= m_tiles) continue;
                if (!tc::warp_ok(!*abort_flag && tc::mbar_wait(&acc[t], (3 * u + l) & 1, kWaitNs))) {
                    give_up();
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t tile = tc::smem_u32(smem + t * kTile);
                const uint32_t from = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(t * kHidden + BK * cg);
                const float4 *b4 = reinterpret_cast<const float4 *>(c.bias[l] + BK * cg);
                // 16 columns at a time, the next 16 on their way meanwhile
                uint32_t v[2][16];
                tc::tmem_ld16(from, v[0]);
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    float4 b[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) b[e] = __ldg(b4 + 4 * h + e);
                    tc::tmem_wait_ld();
                    if (h < 3) tc::tmem_ld16(from + 16 * (h + 1), v[(h + 1) & 1]);
                    const uint32_t(&z)[16] = v[h & 1];
                    __nv_bfloat162 out[8];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 g0 = gelu2(add2(pack2(__uint_as_float(z[4 * e]), __uint_as_float(z[4 * e + 1])), pack2(b[e].x, b[e].y)));
                        const float2 g1 = gelu2(add2(pack2(__uint_as_float(z[4 * e + 2]), __uint_as_float(z[4 * e + 3])), pack2(b[e].z, b[e].w)));
                        out[2 * e] = __floats2bfloat162_rn(g0.x, g0.y);
                        out[2 * e + 1] = __floats2bfloat162_rn(g1.x, g1.y);
                    }
                    const uint4 *o4 = reinterpret_cast<const uint4 *>(out);
#pragma unroll
                    for (int k = 0; k < 2; ++k) tc::st_shared(tc::sw128_piece(tile, tr, BK * cg, 2 * h + k), o4[k]);
                }
                tc::fence_before_sync();
                tc::fence_proxy_async_smem(); // the operand is read by the tensor core
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&ready[t]);
            }
    } else if (warp >= kOut0) { // ---- scores: one row per thread
        const int q = warp & 3;
        float bias[kOutCols];
#pragma unroll
        for (int i = 0; i < kOutCols; ++i) bias[i] = __ldg(c.bias[3] + i);
        bool ok = true;
        for (int u = 0; ok && tile_of(u, 0) < m_tiles; ++u)
            for (int t = 0; t < 2; ++t) {
                const int tile = tile_of(u, t);
                if (tile >= m_tiles) continue;
                const int row = tile * BM + 32 * q + lane;
                int n = 0; // the system's chains: the valid columns
                if (row < c.rows) {
                    const int64_t at = c.sys0 + row / c.rows_per_sys;
                    const int64_t sys = c.sys_list ? (int64_t)c.sys_list[at] : at;
                    n = (int)(c.sys_off[sys + 1] - c.sys_off[sys]);
                }
                if (!tc::warp_ok(!*abort_flag && tc::mbar_wait(&acc_out[t], u & 1, kWaitNs))) {
                    give_up();
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                uint32_t v[32];
                tc::tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(t * kHidden), v);
                tc::tmem_wait_ld();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&out_read[t]);
                float m = 0.0f;
#pragma unroll
                for (int i = 0; i < kOutCols; ++i)
                    if (i < n) m = fmaxf(m, __uint_as_float(v[i]) + bias[i]); // a NaN prediction is ignored
                if (row < c.rows) c.score[row] = m > 0.0f ? m : 0.0f;
            }
    }
    __syncthreads();
    if (warp == 0 && lane == 0 && *abort_flag) {
        // let TMA copies already issued land before this CTA's shared memory is released
        const int n = *issued, x = *x_issued;
        for (int s = 0; s < kStages && s < n; ++s) {
            const int last = ((n - 1 - s) / kStages) * kStages + s;
            tc::mbar_wait(&full[s], (last / kStages) & 1, kWaitNs / 4);
        }
        for (int i = 0; i < 2 * kb0 && i < x; ++i) // copy i went to place i / kb0 % 2, block i % kb0
            tc::mbar_wait(&xfull[i / kb0 * kBlocks + i % kb0], ((x - 1 - i) / (2 * kb0)) & 1, kWaitNs / 4);
    }
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 2 * kHidden);
    }
}

} // namespace

bool paam_score_chain_takes(int kx) { return kx > 0 && kx <= kHidden && kx % BK == 0; }

int paam_score_chain(const ScoreChain &c, const __nv_bfloat16 *X, const __nv_bfloat16 *const (&W)[4],
                     cudaStream_t stream)
{
    if (!paam_score_chain_takes(c.kx) || c.rows <= 0 || c.n_sm < 1) return PAAM_E_INVAL;
    ScoreMaps m;
    bool ok = tc_make_map(&m.X, X, c.rows, c.kx, c.kx, BM);
    for (int l = 0; l < 4; ++l) {
        const int in = l == 0 ? kIn : kHidden, out = l == 3 ? kOutCols : kHidden;
        ok = ok && tc_make_map(&m.W[l], W[l], out, l == 0 ? c.kx : in, in, out);
    }
    if (!ok) return PAAM_E_CUDA;
    const int tiles = (c.rows + BM - 1) / BM;
    PAAM_CUDA_TRY(cudaFuncSetAttribute(score_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    score_chain_kernel<<<(unsigned)(tiles < c.n_sm ? tiles : c.n_sm), kThreads, kSmem, stream>>>(m, c);
    PAAM_CUDA_TRY(cudaGetLastError());
    paam_count_launch();
    return PAAM_OK;
}
