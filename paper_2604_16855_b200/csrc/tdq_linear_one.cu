// The W4A4 linear layer with one accumulator per output element over the whole contraction: one token-group per token
// (g = C_pad) and the power-of-two variant, whose group scales ride in the operands.  y must be one that bulk tensor stores
// can write.  Same integer sums as the general kernel (tdq_linear.cu), same float operations on them.
//
// What bounds it.  Without a per-group pass this is a plain 8-bit GEMM, bound by the tensor pipe if the operands arrive.  What
// kept the general kernel at half of it is shared-memory bandwidth (128 bytes a clock): a 128 x 128 x 32 instruction takes
// 64 clocks and reads 8 KB, and the 8 KB of operands it uses up are written by the copy engine meanwhile, together 128 clocks.
// Two CTAs of a cluster therefore work on one 256 x 256 tile with cta_group::2 instructions: each CTA holds 128 rows of A and
// 128 of B (8 KB per K-step for 128 clocks of tensor time), its own 128 x 256 half of the accumulator in TMEM, and the other's
// B half reaches it through the pair's own path.  Two accumulators (all 512 TMEM columns) let the tensor core run a tile
// ahead of the epilogue.  Warp roles, per CTA:
//
//   warps 0, 3  producers: this CTA's K-steps of A and of B, four (16 KB) each per ring stage
//   warp 1      CTA 0: issues the instructions, commits to both CTAs' barriers; CTA 1: passes the landing of its stages on
//               (with the arrival's default semantics: a release at cluster scope costs about 800 clocks a stage here, and the
//               data it would order, written by the copy engine, is in shared memory once its barrier has completed)
//   warp 2      allocates TMEM
//   warps 4-11  epilogue: 32 rows x 128 columns each, 32 columns at a time (sixteen warps of half the width: 10 % slower)
//
// Measured, with the operand expansion in front (general kernel -> this one): 16384 x 4096 -> 4096 bf16 242 -> 157 us (134 of
// them here, against 115 at the instruction's own rate), 18464 x 768 -> 3072 bf16 49.3 -> 40.8, fp32 61.4 -> 52.4, power-of-two
// steps bf16 54.0 -> 44.6, 9216 x 320 -> 320 12.4 -> 8.2.
#include "tdq_tc.cuh"

namespace tdq {
namespace {

constexpr int kOneN = 256;                             // columns of a cluster's tile; 256 rows, 128 in each CTA
constexpr int kOneSteps = 4;                                   // K-steps per ring stage
constexpr uint32_t kOneStageBytes = 2 * kOneSteps * kBlock;    // of 128 rows of A, then of 128 rows of B
constexpr int kOneMaxStages = 6;
constexpr uint32_t kOneCtrl = 1024;
constexpr int kOneEpiWarp0 = 4, kOneEpiWarps = 8;
constexpr int kOneCols = kOneN / (kOneEpiWarps / 4);   // columns per epilogue warp
constexpr int kOneThreads = (kOneEpiWarp0 + kOneEpiWarps) * 32;
constexpr uint32_t kOneWsb = kOneEpiWarps * kOneCols * 8;   // per warp: its columns' scales and biases
constexpr uint32_t kOneShape = ((uint32_t)(kOneN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
constexpr uint32_t kOneIdescI8 = (2u << 4) | (1u << 7) | (1u << 10) | kOneShape;
constexpr uint32_t kOneIdescF8 = (1u << 4) | kOneShape;

struct OneCtrl {
    uint64_t full[kOneMaxStages], empty[kOneMaxStages];
    uint64_t peer[kOneMaxStages];            // CTA 0: the other CTA's half of the stage has landed
    uint64_t tfull[2], tempty[2];            // accumulator n & 1 of tile n (tempty: CTA 0 only)
};
static_assert(sizeof(Ctrl) + sizeof(OneCtrl) <= kOneCtrl, "control block outgrew its reservation");

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// lane 0 of a converged warp arrives on CTA 0's barrier of this address
__device__ __forceinline__ void arrive_cta0_lane0(uint32_t bar_s, int lane) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 ra;\n\tsetp.eq.s32 p, %1, 0;\n\tmapa.shared::cluster.u32 ra, %0, 0;\n\t"
        "@p mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}"
        ::"r"(bar_s), "r"(lane) : "memory");
}
template <bool I8>
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    if (I8)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(kOneIdescI8), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(kOneIdescF8), "r"(accumulate) : "memory");
}
// arrives on the barrier of this address in both CTAs once this thread's instructions so far have completed
__device__ __forceinline__ void commit_both(uint32_t bar_s) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar_s), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void bulk_wait_group_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }

template <bool I8, bool YBF16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kOneThreads, 1)
w4a4_one_kernel(const LinArgs a, const __grid_constant__ CUtensorMap ymap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    Ctrl* c = reinterpret_cast<Ctrl*>(smem_raw);            // its abort flag and TMEM address; the barriers are g's
    OneCtrl* g = reinterpret_cast<OneCtrl*>(smem_raw + sizeof(Ctrl));
    const uint32_t sm_s = smem_u32(smem_raw);
    const uint32_t ring_s = sm_s + kOneCtrl;
    const uint32_t n_stages = (uint32_t)a.n_stages;
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 0) {
        for (int i = 0; i < kOneMaxStages; ++i) { mbar_init(&g->full[i], 2); mbar_init(&g->empty[i], 1); mbar_init(&g->peer[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&g->tfull[i], 1); mbar_init(&g->tempty[i], 2 * kOneEpiWarps); }
        c->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                                        // both CTAs' barriers are initialised
    tc_fence_after();
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.status + 2, 1u);   // the call's epoch (see expand_pow2_kernel)
    const uint32_t tmem_base = c->tmem_base;
    const int tiles_m = (a.tiles_m + 1) / 2, tiles_n = (a.tiles_n + 1) / 2;   // in units of 256
    const int n_tiles = tiles_m * tiles_n, n_clusters = (int)gridDim.x / 2, first = (int)blockIdx.x / 2;
    const int n_chunks = (a.n_steps + kOneSteps - 1) / kOneSteps;

    if (warp == 0 || warp == 3) {
        // ------------------------------------------------------------ operand blocks: A by warp 0, B by warp 3
        const bool is_a = warp == 0;
        const uint32_t empty_s = smem_u32(&g->empty[0]);
        const uint32_t dst0 = ring_s + (is_a ? 0u : kOneSteps * kBlock);
        uint32_t s = 0, ph = 1;
        for (int tile = first; tile < n_tiles && !c->abort_flag; tile += n_clusters) {
            const int mt = tile / tiles_n, nt = tile - mt * tiles_n;
            // an odd number of blocks: the last pair's second half repeats the first and is clipped when stored
            const int64_t blk = is_a ? min(2 * mt + (int)rank, a.tiles_m - 1) : min(2 * nt + (int)rank, a.tiles_n - 1);
            const uint8_t* src = (is_a ? a.a_blocks : a.b_blocks) + blk * a.n_steps * kBlock;
#pragma unroll 1
            for (int k0 = 0; k0 < a.n_steps; k0 += kOneSteps) {
                const uint32_t bytes = (uint32_t)min(kOneSteps, a.n_steps - k0) * kBlock;
                wait_hot(empty_s + s * 8, ph, c, a.status, 5u);
                if (c->abort_flag) break;
                if (elect_one()) {
                    mbar_expect_tx(&g->full[s], bytes);
                    bulk_load(dst0 + s * kOneStageBytes, src, bytes, &g->full[s]);
                }
                __syncwarp();
                src += kOneSteps * kBlock;
                if (++s == n_stages) { s = 0; ph ^= 1; }
            }
        }
    } else if (warp == 1 && rank == 1) {
        // ------------------------------------------------------------ this CTA's landings, passed on to CTA 0
        const uint32_t full_s = smem_u32(&g->full[0]), peer_s = smem_u32(&g->peer[0]);
        uint32_t s = 0, ph = 0;
        for (int tile = first; tile < n_tiles && !c->abort_flag; tile += n_clusters)
#pragma unroll 1
            for (int kc = 0; kc < n_chunks; ++kc) {
                wait_hot(full_s + s * 8, ph, c, a.status, 4u);
                if (c->abort_flag) break;
                __syncwarp();
                arrive_cta0_lane0(peer_s + s * 8, lane);
                if (++s == n_stages) { s = 0; ph ^= 1; }
            }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issue
        const uint32_t full_s = smem_u32(&g->full[0]), peer_s = smem_u32(&g->peer[0]), empty_s = smem_u32(&g->empty[0]);
        const uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        const uint32_t a_lo = desc_lo(ring_s), b_lo = desc_lo(ring_s + kOneSteps * kBlock);
        uint32_t s = 0, ph = 0, n = 0;
        for (int tile = first; tile < n_tiles && !c->abort_flag; tile += n_clusters, ++n) {
            const uint32_t slot = n & 1u, d = tmem_base + slot * kOneN;
            wait_hot(tempty_s + slot * 8, ((n >> 1) & 1u) ^ 1u, c, a.status, 3u);
#pragma unroll 1
            for (int kc = 0; kc < n_chunks; ++kc) {
                wait_hot(full_s + s * 8, ph, c, a.status, 4u);
                wait_hot(peer_s + s * 8, ph, c, a.status, 6u);
                if (c->abort_flag) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t so = s * (kOneStageBytes >> 4);
#pragma unroll
                    for (int k = 0; k < kOneSteps; ++k)
                        if (kc * kOneSteps + k < a.n_steps) mma_pair<I8>(d, desc_of(a_lo + so + k * (kBlock >> 4)), desc_of(b_lo + so + k * (kBlock >> 4)), (kc | k) != 0 ? 1u : 0u);
                    commit_both(empty_s + s * 8);
                    if (kc == n_chunks - 1) commit_both(tfull_s + slot * 8);
                }
                __syncwarp();
                if (++s == n_stages) { s = 0; ph ^= 1; }
            }
        }
    } else if (warp >= kOneEpiWarp0) {
        // ------------------------------------------------------------ epilogue
        const int ew = warp - kOneEpiWarp0, quarter = warp & 3, half = ew >> 2;
        const int row = quarter * 32 + lane;
        constexpr uint32_t kStrip = 32 * 32 * (YBF16 ? 2 : 4);
        const uint32_t bufs = (uint32_t)a.n_ibuf;              // strips per warp
        const uint32_t strips_s = ((ring_s + n_stages * kOneStageBytes + 1023u) & ~1023u) + (uint32_t)ew * bufs * kStrip;
        const uint32_t wsb_s = ((ring_s + n_stages * kOneStageBytes + 1023u) & ~1023u) + kOneEpiWarps * bufs * kStrip + (uint32_t)ew * (kOneCols * 8);
        float* wsb = reinterpret_cast<float*>(smem_raw + (wsb_s - sm_s));   // scales, then biases
        const uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        uint32_t va[32], vb[32];
#pragma unroll
        for (int q = 0; q < 32; ++q) { va[q] = 0u; vb[q] = 0u; }
        uint32_t n = 0, buf = 0;
        for (int tile = first; tile < n_tiles && !c->abort_flag; tile += n_clusters, ++n) {
            const int mt = tile / tiles_n, nt = tile - mt * tiles_n;
            const int64_t m0 = (int64_t)mt * 256 + rank * kBM + quarter * 32, n0 = (int64_t)nt * kOneN + half * kOneCols;
            const int64_t mb = min(2 * mt + (int)rank, a.tiles_m - 1);
            const float delta = __ldg(reinterpret_cast<const float*>(a.s_blocks) + mb * kBM + row);
            const uint64_t delta2 = pack2(__float_as_uint(delta), __float_as_uint(delta));
            __syncwarp();                                  // the last tile's constants have been read
#pragma unroll
            for (int i = 0; i < kOneCols / 32; ++i) {
                const int64_t col = n0 + 32 * i + lane;
                wsb[32 * i + lane] = col < a.O ? __fmul_rn(__ldg(a.wscale + col), a.out_scale) : 0.f;
                wsb[kOneCols + 32 * i + lane] = (a.bias && col < a.O) ? __ldg(a.bias + col) : 0.f;
            }
            __syncwarp();
            const uint32_t slot = n & 1u;
            wait_hot(tfull_s + slot * 8, (n >> 1) & 1u, c, a.status, 2u);
            tc_fence_after();
            const uint32_t tm = tmem_base + ((uint32_t)(quarter * 32) << 16) + slot * kOneN + half * kOneCols;
            tmem_ld32(tm, va);
#pragma unroll
            for (int i = 0; i < kOneCols / 32; ++i) {
                uint32_t* const v = (i & 1) ? vb : va;
                tmem_ld_wait_on(v);
                if (i < kOneCols / 32 - 1) {
                    tmem_ld32(tm + 32 * (i + 1), (i & 1) ? va : vb);
                } else {
                    tc_fence_before();                     // the accumulator is drained
                    __syncwarp();
                    arrive_cta0_lane0(tempty_s + slot * 8, lane);
                }
                if (lane == 0) {                           // the strip has been read
                    if (bufs == 2) bulk_wait_group_read1();
                    else bulk_wait_group_read0();
                }
                __syncwarp();
                const uint32_t strip = strips_s + buf * kStrip + (uint32_t)lane * (YBF16 ? 64u : 128u);
                const float4* s4 = reinterpret_cast<const float4*>(wsb + 32 * i);
                const float4* b4 = reinterpret_cast<const float4*>(wsb + kOneCols + 32 * i);
#pragma unroll
                for (int j = 0; j < 4; ++j) {              // eight columns
                    const float4 sa = s4[2 * j], sb = s4[2 * j + 1], ba = b4[2 * j], bb = b4[2 * j + 1];
                    const float* const ss[2] = {reinterpret_cast<const float*>(&sa), reinterpret_cast<const float*>(&sb)};
                    const float* const bs[2] = {reinterpret_cast<const float*>(&ba), reinterpret_cast<const float*>(&bb)};
                    float o[8];
#pragma unroll
                    for (int q = 0; q < 8; q += 2) {       // y = s (delta sum) + b, two columns an instruction
                        uint32_t f0 = v[8 * j + q], f1 = v[8 * j + q + 1];
                        if (I8) {
                            f0 = __float_as_uint((float)(int32_t)f0);
                            f1 = __float_as_uint((float)(int32_t)f1);
                        }
                        uint64_t t = pack2(f0, f1), y2 = pack2(__float_as_uint(bs[q >> 2][q & 3]), __float_as_uint(bs[q >> 2][(q & 3) + 1]));
                        asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(t) : "l"(delta2));
                        fma2(y2, t, pack2(__float_as_uint(ss[q >> 2][q & 3]), __float_as_uint(ss[q >> 2][(q & 3) + 1])));
                        unpack2(y2, o[q], o[q + 1]);
                    }
                    if (!YBF16) {
                        const uint32_t x7 = (uint32_t)lane & 7u;
                        sts128(strip + (((uint32_t)(2 * j) ^ x7) << 4), __float_as_uint(o[0]), __float_as_uint(o[1]), __float_as_uint(o[2]), __float_as_uint(o[3]));
                        sts128(strip + (((uint32_t)(2 * j + 1) ^ x7) << 4), __float_as_uint(o[4]), __float_as_uint(o[5]), __float_as_uint(o[6]), __float_as_uint(o[7]));
                    } else {
                        sts128(strip + (((uint32_t)j ^ (((uint32_t)lane >> 1) & 3u)) << 4), pack16(o[0], o[1], a.y_f16), pack16(o[2], o[3], a.y_f16),
                               pack16(o[4], o[5], a.y_f16), pack16(o[6], o[7], a.y_f16));
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the engine's reads
                __syncwarp();
                if (lane == 0) {
                    if (m0 < a.M && n0 + 32 * i < a.O) tma_store_2d(&ymap, strips_s + buf * kStrip, (int32_t)(n0 + 32 * i), (int32_t)m0);
                    bulk_commit_group();
                }
                if (bufs == 2) buf ^= 1u;
            }
        }
        tmem_ld_wait();
        if (lane == 0) bulk_wait_group0();                 // no store may still be reading this CTA's shared memory at exit
    }

    tc_fence_before();
    __syncthreads();
    if (c->abort_flag) __nanosleep(1000000);               // a wait gave up: give the tensor core a moment
    cluster_sync();                                        // neither CTA leaves while the other may still signal it
    if (warp == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
}

}  // namespace

// The caller has run the operand expansion and encoded y's map with boxes of 32 x 32.
tdq_status launch_linear_one(LinArgs a, const CUtensorMap& ymap, int n_sm, int dev, bool i8, bool ybf, cudaStream_t stream) {
    void (*const kernels[4])(LinArgs, CUtensorMap) = {w4a4_one_kernel<false, false>, w4a4_one_kernel<false, true>,
                                                      w4a4_one_kernel<true, false>, w4a4_one_kernel<true, true>};
    const int inst = (ybf ? 1 : 0) + (i8 ? 2 : 0);
    // Two strips per epilogue warp, or one and another ring stage: the stage for fp32 output (5 instead of 4; 18464 x 768 ->
    // 3072 57.8 -> 53.3 us) and long contractions (16384 x 4096 -> 4096 bf16 164 -> 156 us), the strip else (43.9 -> 40.4 us).
    a.n_ibuf = (ybf && a.n_steps < 64) ? 2 : 1;
    const int strips = kOneEpiWarps * a.n_ibuf * 32 * 32 * (ybf ? 2 : 4);
    a.n_stages = (kSmemLimit - (int)kOneCtrl - 1024 - strips - (int)kOneWsb) / (int)kOneStageBytes;
    if (a.n_stages > kOneMaxStages) a.n_stages = kOneMaxStages;
    const uint32_t smem = kOneCtrl + (uint32_t)a.n_stages * kOneStageBytes + 1024 + (uint32_t)strips + kOneWsb;
    static std::atomic<uint64_t> smem_done[4];
    if (allow_smem(kernels[inst], kSmemLimit, smem_done[inst], dev) != cudaSuccess) return TDQ_ERR_CUDA;
    const int64_t tiles = (int64_t)((a.tiles_m + 1) / 2) * ((a.tiles_n + 1) / 2);
    const unsigned clusters = (unsigned)(tiles < n_sm / 2 ? tiles : n_sm / 2);
    if (launch_pdl(kernels[inst], dim3(2 * clusters), dim3(kOneThreads), smem, stream, a, ymap) != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

}  // namespace tdq
