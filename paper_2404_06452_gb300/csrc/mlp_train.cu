// mlp_train.cu -- a training step's chain of layers in one kernel (tcgen05 + TMA +
// TMEM on sm_103a): for a tile of 128 minibatch rows, the four layers forward,
// the loss and its gradient, and the three input gradients back.
//
// A minibatch of a few thousand rows is too small for a kernel per layer: each of
// those (8,192 x 256 x 256) has 0.5 us of tensor work behind 8 us of launch, set-up,
// first loads and drain, and every layer waits for the one before it.  Here a pair of
// CTAs (a cluster) keeps 128 rows, each CTA half of every layer's columns: it reads its
// accumulator from tensor memory, applies the activation and writes the result to its
// own and its partner's shared memory as the next layer's A operand (128-byte swizzle,
// four blocks of 64 columns), while the next layers' weights stream into a ring.  To
// memory goes only what others read: the activations and gradients that the weight-
// gradient GEMMs contract over, by TMA from the operand tiles (those GEMMs read them
// transposed, so nothing is stored transposed), and the first layer's pre-activations,
// which come back for its gradient (the other two layers' stay in shared memory).
// The loss leaves as sums of 32 rows and half of the columns.
//
//   phase 0 1 2   H_l = gelu(H_(l-1) W_l^T + b_l)
//         3       Y = H_2 W_3^T + b_3, loss, dY
//         4 5 6   dZ_l = (dZ_(l+1) W_(l+1)) gelu'(Z_l), l = 2, 1, 0
//
// Warp 0 streams the operands (3 stages of 16 + 16 KB), one lane of warp 1 issues
// the MMAs (128 x 128 or 128 x 32 x 16, fp32 accumulator in TMEM) and the stores, 16
// warps run the epilogues (four per TMEM lane quadrant, 32 columns each).  A phase's
// MMAs of both CTAs are complete before either epilogue writes operand tiles, and both
// epilogues are before either's next MMAs.  The sums are those of a kernel per layer,
// in the same order.  Bound by the epilogues: the activation's two special-function
// results per element take 1 us per phase.  8,192 rows: seven kernels 75 us, one CTA
// per 128 rows 51-60, a pair 41 us (about 10,000 cycles per phase, 1,200 of them MMAs,
// 2,900 arithmetic, 4,000 the operand writes into both CTAs and the fence behind them);
// 44 with one lane of the MMA warp waiting by itself.
#include "gelu.cuh"
#include "mlp.cuh"
#include "tc.cuh"

namespace {
using namespace paam_gelu;

constexpr int BM = 128, BK = 64, kHidden = 256, kOut = 64, kIn = 1024;
constexpr int kPhases = 7, kStages = 3;
constexpr int kHalf = kHidden / 2; // columns per CTA of the pair
constexpr int kA = BM * BK * 2, kB = kHalf * BK * 2, kStage = kA + kB;
constexpr int kH = 4 * kA; // the activations of 128 rows: four blocks of 64 columns
constexpr int kZ = 2 * kA; // the CTA's half of a layer's pre-activations
constexpr int kTiles = kStages * kStage + kH + 2 * kZ;
constexpr int kSmem = kTiles + 256 + 1024; // barriers and flags, alignment slack
static_assert(kSmem <= 227 * 1024, "one CTA's shared memory");
constexpr int kEpiWarps = 16, kThreads = 32 * (2 + kEpiWarps);
constexpr uint64_t kWaitNs = 2000000000ull; // 2 s: far above any legitimate wait

__host__ __device__ constexpr int blocks_of(int p) { return p == 0 ? kIn / BK : (p == 4 ? kOut / BK : kHidden / BK); }
__host__ __device__ constexpr int cols_of(int p) { return p == 3 ? kOut : kHidden; }
__host__ __device__ constexpr int mine_of(int p) { return cols_of(p) / 2; } // columns per CTA

struct ChainMaps {
    CUtensorMap X;          // [rows][1024]
    CUtensorMap W[kPhases]; // the B operand of each phase
    CUtensorMap O[kPhases]; // what each phase's epilogue leaves: H, dY, dZ
    CUtensorMap Z;          // the first layer's pre-activations
};

__device__ __forceinline__ uint4 get_piece(uint32_t at)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
    return v;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    train_chain_kernel(const __grid_constant__ ChainMaps maps, const __grid_constant__ TrainChain c)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *hs = smem + kStages * kStage; // the A operand, all columns
    uint8_t *zs = hs + kH;                 // two tiles of pre-activations: Z_2 (first Z_0), Z_1
    uint64_t *full = (uint64_t *)(smem + kTiles);
    uint64_t *empty = full + kStages;
    uint64_t *done = empty + kStages; // a phase's MMAs are complete, in both CTAs
    uint64_t *ready = done + 1;       // its epilogues are: accumulator read, next operand written
    uint64_t *stored = ready + 1;     // the stores of the phase before have read their tiles, in both CTAs
    uint64_t *zbar = stored + 1;      // Z_0 is back
    uint64_t *fin = zbar + 1;
    uint32_t *tmem_slot = (uint32_t *)(fin + 1);
    volatile int *abort_flag = (volatile int *)(tmem_slot + 1);
    volatile int *issued = abort_flag + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = tc::cluster_rank();
    const int m0 = (blockIdx.x >> 1) * BM;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(done, 2);
        tc::mbar_init(ready, 2 * kEpiWarps);
        tc::mbar_init(stored, 2);
        tc::mbar_init(zbar, 1);
        tc::mbar_init(fin, 1);
        *abort_flag = 0;
        *issued = 0;
        tc::fence_barrier_init();
        tc::prefetch_tmap(&maps.X);
        for (int p = 0; p < kPhases; ++p) {
            tc::prefetch_tmap(&maps.W[p]);
            tc::prefetch_tmap(&maps.O[p]);
        }
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, kHalf);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::cluster_sync(); // both CTAs' barriers exist
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) { // ---- TMA producer
        int it = 0;
        bool ok = true;
        for (int p = 0; p < kPhases && ok; ++p)
            for (int kb = 0; kb < blocks_of(p); ++kb) {
                const int s = it % kStages, r = it / kStages;
                if (*abort_flag || (r > 0 && !tc::mbar_wait(&empty[s], (r - 1) & 1, kWaitNs))) {
                    *abort_flag = 1;
                    atomicExch(c.err, PAAM_E_TIMEOUT);
                    ok = false;
                    break;
                }
                uint8_t *a = smem + s * kStage;
                tc::mbar_expect_tx(&full[s], (uint32_t)(mine_of(p) * BK * 2 + (p == 0 ? kA : 0)));
                if (p == 0) tc::tma_load_2d(a, &maps.X, &full[s], kb * BK, m0);
                tc::tma_load_2d(a + kA, &maps.W[p], &full[s], kb * BK, (int)rank * mine_of(p));
                ++it;
            }
        *issued = it;
    } else if (warp == 1) { // ---- MMA issuer, stores: the warp waits as one, one lane issues
        bool ok = true, zload = false;
        int s = 0;
        uint32_t round = 0;
        const uint32_t lead = tc::elect_one(), d = __shfl_sync(0xffffffffu, tmem, 0);
        // phase p's results, complete in the operand tiles, to memory: each CTA its own
        // columns (the output gradient's 64 are one block: the first CTA)
        auto store = [&](int p) {
            if (p == 3) {
                if (rank == 0) tc::tma_store_2d(&maps.O[p], hs, 0, m0);
            } else {
                for (int kb = 2 * (int)rank; kb < 2 * (int)rank + 2; ++kb)
                    tc::tma_store_2d(&maps.O[p], hs + kb * kA, kb * BK, m0);
            }
            if (p == 0)
                for (int kb = 0; kb < 2; ++kb) tc::tma_store_2d(&maps.Z, zs + kb * kA, (2 * (int)rank + kb) * BK, m0);
            tc::bulk_commit();
        };
        for (int p = 0; p < kPhases && ok; ++p) {
            if (p > 0) {
                if (!tc::warp_ok(!*abort_flag && tc::mbar_wait_cluster(ready, (p - 1) & 1, kWaitNs))) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                if (p == 5) { // Z_2's tile has been read: Z_0 comes back into it
                    if (lead) {
                        tc::bulk_wait_all();
                        tc::mbar_expect_tx(zbar, kZ);
                        for (int kb = 0; kb < 2; ++kb)
                            tc::tma_load_2d(zs + kb * kA, &maps.Z, zbar, (2 * (int)rank + kb) * BK, m0);
                    }
                    zload = true;
                }
            }
            const uint32_t idesc = p == 3 ? tc::idesc_bf16(BM, kOut / 2) : tc::idesc_bf16(BM, kHalf);
            for (int kb = 0; kb < blocks_of(p); ++kb) {
                ok = tc::mbar_wait(&full[s], round, kWaitNs);
                if (!ok) break; // to the vote below
                const uint32_t st = tc::smem_u32(smem + s * kStage);
                const uint64_t a = tc::desc_sw128(p == 0 ? st : tc::smem_u32(hs + kb * kA));
                const uint64_t w = tc::desc_sw128(st + kA);
                if (lead) {
#pragma unroll
                    for (int j = 0; j < BK / 16; ++j)
                        tc::mma_bf16(d, a + 2 * j, w + 2 * j, idesc, (kb > 0 || j > 0) ? 1u : 0u);
                    tc::mma_commit(&empty[s]);
                }
                if (++s == kStages) {
                    s = 0;
                    round ^= 1;
                }
            }
            ok = tc::warp_ok(ok);
            if (!ok) break;
            if (lead) {
                tc::mma_commit_multicast(done, 3);
                // the stores run beside the MMAs and the epilogues' arithmetic
                if (p > 0) {
                    store(p - 1);
                    tc::bulk_wait_read_all();
                }
                tc::mbar_arrive_cluster(tc::map_rank(tc::smem_u32(stored), 0));
                tc::mbar_arrive_cluster(tc::map_rank(tc::smem_u32(stored), 1));
            }
            __syncwarp();
        }
        ok = ok && tc::warp_ok(tc::mbar_wait_cluster(ready, (kPhases - 1) & 1, kWaitNs));
        if (lead) {
            if (ok) store(kPhases - 1);
            tc::bulk_wait_all();
            if (!ok) {
                *abort_flag = 1;
                atomicExch(c.err, PAAM_E_TIMEOUT);
                if (zload) tc::mbar_wait(zbar, 0, kWaitNs / 4); // the copy has landed
            }
            // every MMA issued has completed before TMEM can be released
            tc::mma_commit(fin);
            tc::mbar_wait(fin, 0, kWaitNs);
        }
        __syncwarp();
    } else if (warp >= 2) { // ---- epilogues: one row per thread, 32 of the CTA's columns per warp
        const int q = warp & 3, cg = (warp - 2) >> 2; // TMEM lane quadrant, column group
        const int tr = 32 * q + lane;
        const int64_t row = m0 + tr;
        const uint32_t hme = tc::smem_u32(hs), hpeer = tc::map_rank(hme, rank ^ 1);
        const uint32_t ready_peer = tc::map_rank(tc::smem_u32(ready), rank ^ 1);
#pragma unroll 1
        for (int p = 0; p < kPhases; ++p) {
            if (!tc::warp_ok(!*abort_flag && tc::mbar_wait_cluster(done, p & 1, kWaitNs) &&
                             (p < 6 || tc::mbar_wait(zbar, 0, kWaitNs)))) {
                *abort_flag = 1;
                atomicExch(c.err, PAAM_E_TIMEOUT);
                break;
            }
            tc::fence_after_sync();
            __nv_bfloat162 out[16];
            int col0 = 0;
            if (p != 3 || cg == 0) {
                const int here = 32 * cg; // of the CTA's columns
                col0 = (int)rank * mine_of(p) + here; // of the layer's
                uint32_t v[32];
                tc::tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)here, v);
                if (p < 3) { // bias, pre-activation, activation
                    const float4 *b4 = reinterpret_cast<const float4 *>(c.bias[p] + col0);
                    const uint32_t zt = tc::smem_u32(zs + (p == 1 ? kZ : 0));
                    tc::tmem_wait_ld();
                    uint4 zb[4];
                    __nv_bfloat162 *z2 = reinterpret_cast<__nv_bfloat162 *>(zb);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 b = __ldg(b4 + i);
                        const uint64_t za = add2(pack2(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1])), pack2(b.x, b.y));
                        const uint64_t zc = add2(pack2(__uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3])), pack2(b.z, b.w));
                        const float2 a0 = unpack2(za), a2 = unpack2(zc), g0 = gelu2(za), g2 = gelu2(zc);
                        z2[2 * i] = __floats2bfloat162_rn(a0.x, a0.y);
                        z2[2 * i + 1] = __floats2bfloat162_rn(a2.x, a2.y);
                        out[2 * i] = __floats2bfloat162_rn(g0.x, g0.y);
                        out[2 * i + 1] = __floats2bfloat162_rn(g2.x, g2.y);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) tc::st_shared(tc::sw128_piece(zt, tr, here, k), zb[k]);
                } else if (p == 3) { // outputs, masked squared error and its gradient
                    const float4 *b4 = reinterpret_cast<const float4 *>(c.bias[3] + col0);
                    const float4 *l4 = reinterpret_cast<const float4 *>(c.L + row * kOut + col0);
                    const float inv = 1.0f / fmaxf(*c.count, 1.0f);
                    tc::tmem_wait_ld();
                    float acc = 0.0f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 b = __ldg(b4 + i), l = l4[i];
                        const float y[4] = {__uint_as_float(v[4 * i]) + b.x, __uint_as_float(v[4 * i + 1]) + b.y,
                                            __uint_as_float(v[4 * i + 2]) + b.z, __uint_as_float(v[4 * i + 3]) + b.w};
                        const float ll[4] = {l.x, l.y, l.z, l.w};
                        float g[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float d = ll[e] >= 0.0f ? y[e] - ll[e] : 0.0f;
                            acc += d * d;
                            g[e] = 2.0f * d * inv;
                        }
                        out[2 * i] = __floats2bfloat162_rn(g[0], g[1]);
                        out[2 * i + 1] = __floats2bfloat162_rn(g[2], g[3]);
                    }
                    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                    if (lane == 0) c.loss_part[2 * (row >> 5) + rank] = acc * inv;
                } else { // through the activation
                    const uint32_t zt = tc::smem_u32(zs + (p == 5 ? kZ : 0));
                    uint4 zb[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) zb[k] = get_piece(tc::sw128_piece(zt, tr, here, k));
                    const __nv_bfloat162 *z2 = reinterpret_cast<const __nv_bfloat162 *>(zb);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float2 zf = __bfloat1622float2(z2[i]);
                        out[i] = __floats2bfloat162_rn(__uint_as_float(v[2 * i]) * gelu_grad(zf.x),
                                                       __uint_as_float(v[2 * i + 1]) * gelu_grad(zf.y));
                    }
                }
                if (!tc::warp_ok(tc::mbar_wait_cluster(stored, p & 1, kWaitNs))) {
                    *abort_flag = 1; // the warp leaves at its next phase
                    atomicExch(c.err, PAAM_E_TIMEOUT);
                }
                const uint4 *o4 = reinterpret_cast<const uint4 *>(out);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t at = tc::sw128_piece(0, tr, col0, k);
                    tc::st_shared(hme + at, o4[k]);
                    if (p < kPhases - 1) tc::st_cluster(hpeer + at, o4[k]);
                }
            }
            tc::fence_before_sync();
            tc::fence_proxy_async_cluster(); // the tiles are read by the tensor core and by TMA, here and in the partner
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive_cluster(tc::map_rank(tc::smem_u32(ready), rank));
                tc::mbar_arrive_cluster(ready_peer);
            }
        }
    }
    __syncthreads();
    if (warp == 0 && lane == 0 && *abort_flag) {
        // let TMA copies already issued land before this CTA's shared memory is released
        const int n = *issued;
        for (int s = 0; s < kStages && s < n; ++s) {
            const int last = ((n - 1 - s) / kStages) * kStages + s;
            tc::mbar_wait(&full[s], (last / kStages) & 1, kWaitNs / 4);
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kHalf);
    }
    tc::cluster_sync(); // the partner no longer writes to this CTA's shared memory
}

} // namespace

int paam_train_chain(const TrainChain &c, const __nv_bfloat16 *X, const __nv_bfloat16 *const (&W)[4],
                     const __nv_bfloat16 *const (&WT)[4], cudaStream_t stream)
{
    if (c.rows <= 0 || c.rows % BM) return PAAM_E_INVAL;
    ChainMaps m;
    bool ok = tc_make_map(&m.X, X, c.rows, kIn, kIn, BM);
    for (int p = 0; p < 4; ++p) { // W_p [out][in]
        const int in = p == 0 ? kIn : kHidden, out = p == 3 ? kOut : kHidden;
        ok = ok && tc_make_map(&m.W[p], W[p], out, in, in, out / 2);
    }
    for (int p = 4; p < kPhases; ++p) { // W_l^T [in][out], l = 3, 2, 1
        const int l = 7 - p, out = l == 3 ? kOut : kHidden;
        ok = ok && tc_make_map(&m.W[p], WT[l], kHidden, out, out, kHalf);
    }
    for (int p = 0; p < kPhases; ++p) {
        __nv_bfloat16 *o = p < 3 ? c.H[p] : (p == 3 ? c.dY : c.dZ[6 - p]);
        ok = ok && tc_make_map(&m.O[p], o, c.rows, cols_of(p), cols_of(p), BM);
    }
    ok = ok && tc_make_map(&m.Z, c.Z, c.rows, kHidden, kHidden, BM);
    if (!ok) return PAAM_E_CUDA;
    PAAM_CUDA_TRY(cudaFuncSetAttribute(train_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    train_chain_kernel<<<(unsigned)(2 * (c.rows / BM)), kThreads, kSmem, stream>>>(m, c);
    PAAM_CUDA_TRY(cudaGetLastError());
    paam_count_launch();
    return PAAM_OK;
}
