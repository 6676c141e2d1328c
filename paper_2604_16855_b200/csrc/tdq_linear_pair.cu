// The W4A4 linear layer at the paper's group size g = 32 for contractions of up to about 1536 channels (Algorithm S1 step 10
// with Eq. 9 and Eq. 4 substituted), and of any length where y is not one that bulk tensor stores can write.
// The arithmetic is tdq_linear_g32.cu's, bit for bit:
//
//   acc[m,o,k] = sum_{i in group k} q_x[m,i] q_w[o,i]      one tcgen05.mma (E4M3 operands, exact) per group
//   y[m,o]     = s_o * sum_k Delta[m,k] * acc[m,o,k] + b_o  fp32 in registers ("promotion")
//
// What bounds it.  Every K-step of the tensor core ends an accumulator.  Per 128 x 128 group the SM needs 64 clocks of
// tensor time, 64 of TMEM reads (1 KB per clock) and about 145 of its FMA pipes (packed multiply-adds at 1.13 clocks an
// element and scheduler), and TMEM holds four such groups, each of which spends most of its stay in signalling (arrival to
// MMA warp, issue, commit to barrier, notice, load: about 800 clocks).  One block per SM with all of TMEM
// (tdq_linear_g32.cu) adds to that, per tile, everything the epilogue takes, because nothing is promoted meanwhile: a
// third of a 768-channel tile, nearly all of a 64-channel one.
//
// So: two thread blocks per SM, each with half of TMEM, that drift against each other: one's loads, waits, epilogue and
// output run under the other's multiply-adds.  A block is persistent, works on 128 x 64 tiles and takes a tile's groups two
// at a time, a pair of 64-column slots with one barrier each way, since the handshake and not the data is what costs (a
// barrier per slot: 7 % slower):
//
//   warp 0      producer: operand blocks and steps Delta of 4 groups (16 KB of A, 8 KB of B, 2 KB) through a ring of stages
//   warps 1-2   MMA issue, one pair of slots each
//   warp 3      stores: starts a staged tile's bulk tensor stores, hands the area back when the engine has read it,
//               and fetches the next tile's channel constants meanwhile
//   warps 4-7   promotion and epilogue: warp = 32 TMEM lanes (rows), all 64 columns: 64 float sums, 128 landing registers
//
// Groups of 64 and 128 codes take the same kernel (template argument SPG) for short contractions, narrow layers and few
// tiles; larger ones are bound by the operands' way through shared memory, which the general kernel's wider tiles halve.
//
// Measured against the other kernel (us; with the operand expansion): 73728 x 64 -> 64 fp32 16.2 -> 11.0, 73728 x 64 -> 192
// 25.0 -> 18.0, 9216 x 64 -> 256 8.4 -> 7.2, 16384 x 512 -> 2048 bf16 63.8 -> 51.4, 16384 x 1024 -> 2048 92.7 -> 86.6,
// 18464 x 768 -> 3072 fp32 119.7 -> 115.4; above 48 groups the other one is 2-10 % faster (narrower tiles read A twice
// as often and the older of an SM's two blocks runs an eighth faster than the other; both sides in tdq_linear.cu).
#include "tdq_tc.cuh"

namespace tdq {
namespace {

constexpr int kN = 64;                       // columns per tile = one TMEM slot
constexpr int kBHalf = kN * 32;              // operand bytes of 64 rows of B and one K-step
constexpr int kPairThreads = 256;
constexpr int kPairStages = 3;
static_assert(kPairStages * kChunk == kPairRing);
constexpr uint32_t kPairScales = kChunk * (kBlock + kBHalf);   // offset of a stage's scales: 4 groups x 128 rows
constexpr uint32_t kPairStageBytes = kPairScales + kChunk * kScaleBlock;
constexpr uint32_t kPairCtrl = 512;
constexpr int kProducerWarp = 0, kFirstMmaWarp = 1, kPairStoreWarp = 3, kFirstPromoWarp = 4, kPairPromoWarps = 4;
constexpr int kRegsPairCtl = 40, kRegsPairPromo = 216;     // 128 * 40 + 128 * 216 = 256 * 128
constexpr uint32_t kIdescN64 = (1u << 4) | ((uint32_t)(kN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
constexpr uint32_t kPairBoxF32 = 128 * 128, kPairBoxBF16 = 128 * 64;   // one 32-column box of 128 rows in the staging area

struct PairCtrl {
    uint64_t full[kPairStages], empty[kPairStages];
    uint64_t tfull[2], tempty[2];            // per pair of slots
    uint64_t sfull, sfree;                   // the staged output tile is complete / has been read by the copy engine
};
static_assert(sizeof(Ctrl) + sizeof(PairCtrl) <= kPairCtrl, "control block outgrew its reservation");

// The operands of a block's only tile straight from the packed codes (DIRECT; contractions that the ring holds whole): 128 rows
// of A, 64 of B and the rows' steps, stage by stage.  A lane takes a row, so that the 16-byte stores of a quarter warp fill a
// core matrix; the loads of neighbouring K-steps share sectors.  STAGES: how many stages' loads are in flight together.
template <int STAGES>
__device__ __forceinline__ void fill_stages(const LinArgs& a, int mt, int nt, uint32_t ring_s) {
    const int t = threadIdx.x, ra = t & 127, rb = t & 63;
    const int64_t ma = (int64_t)mt * kBM + ra, ob = (int64_t)nt * kN + rb;
    const uint4* sa = reinterpret_cast<const uint4*>(a.xcodes + ma * a.row_bytes);
    const uint4* sb = reinterpret_cast<const uint4*>(a.wcodes + ob * a.row_bytes);
    const float* sx = a.xscale + ma * a.n_steps;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    uint4 pa[STAGES][2], pb[STAGES];
    float d[STAGES][2];
#pragma unroll
    for (int i = 0; i < STAGES; ++i) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int ks = kChunk * i + (t >> 7) + 2 * j;
            const bool on = ks < a.n_steps && ma < a.M;
            pa[i][j] = on ? __ldg(sa + ks) : zero;
            d[i][j] = on ? __ldg(sx + ks) : 0.0f;
        }
        const int ks = kChunk * i + (t >> 6);
        pb[i] = (ks < a.n_steps && ob < a.O) ? __ldg(sb + ks) : zero;
    }
    auto put = [&](uint32_t dst, const uint4& p) {
        uint4 c0, c1;
        expand8<false>(p.x, c0.x, c0.y);
        expand8<false>(p.y, c0.z, c0.w);
        expand8<false>(p.z, c1.x, c1.y);
        expand8<false>(p.w, c1.z, c1.w);
        sts128(dst, c0.x, c0.y, c0.z, c0.w);
        sts128(dst + 128, c1.x, c1.y, c1.z, c1.w);
    };
#pragma unroll
    for (int i = 0; i < STAGES; ++i) {
        const uint32_t st = ring_s + i * kPairStageBytes;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int k = (t >> 7) + 2 * j;
            if (kChunk * i + k < a.n_steps) {
                put(st + (uint32_t)k * kBlock + (uint32_t)((ra >> 3) * 256 + (ra & 7) * 16), pa[i][j]);
                sts32(st + kPairScales + (uint32_t)k * kScaleBlock + (uint32_t)ra * 4, __float_as_uint(d[i][j]));
            }
        }
        const int k = t >> 6;
        if (kChunk * i + k < a.n_steps) put(st + kChunk * kBlock + (uint32_t)k * kBHalf + (uint32_t)((rb >> 3) * 256 + (rb & 7) * 16), pb[i]);
    }
}

// DIRECT: at most 12 groups (the ring holds them all) and one tile per block; the operands come from the packed codes
// (fill_stages), and the call is one launch instead of an expansion and this.  SPG: K-steps per group (1, 2 or 4).  With
// one, a stage holds two pairs of groups and their steps; with more, a pair of groups is one stage or two, one MMA warp
// takes them all, and the row's steps come from global memory a pair ahead.
template <bool YBF16, bool DBG, int SPG, bool DIRECT = false>
__global__ void __launch_bounds__(kPairThreads, 2) w4a4_pair_kernel(const LinArgs a, const __grid_constant__ CUtensorMap ymap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    Ctrl* c = reinterpret_cast<Ctrl*>(smem_raw);            // its abort flag and TMEM address; the barriers are g's
    PairCtrl* g = reinterpret_cast<PairCtrl*>(smem_raw + sizeof(Ctrl));
    const uint32_t sm_s = smem_u32(smem_raw);
    const uint32_t ring_s = sm_s + kPairCtrl;
    const uint32_t stage_s = (ring_s + kPairStages * kPairStageBytes + 1023u) & ~1023u;   // the swizzle patterns repeat every 1024 bytes
    const uint32_t wsb_s = stage_s + (YBF16 ? 2 * kPairBoxBF16 : 2 * kPairBoxF32);   // [64] channel scales, [64] biases of the current tile
    const int warp = uniform_warp(), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kPairStages; ++i) { mbar_init(&g->full[i], 1); mbar_init(&g->empty[i], SPG == 1 ? 2 + kPairPromoWarps : 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&g->tfull[i], 1); mbar_init(&g->tempty[i], kPairPromoWarps); }
        mbar_init(&g->sfull, kPairPromoWarps);
        mbar_init(&g->sfree, 1);
        c->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kFirstMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem_base)),
                     "r"(kSlots * kN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();          // barrier set-up and the TMEM allocation overlap the tail of the kernel before this one
    pdl_trigger();
    const uint32_t tmem_base = c->tmem_base;
    const int n_tiles = a.tiles_m * a.tiles_n;
    const int n_steps = a.n_steps;
    if (DIRECT) {
        if (blockIdx.x == 0 && threadIdx.x < 4) a.status[threadIdx.x] = 0u;   // the expansion's job otherwise
        const int mt = (int)blockIdx.x / a.tiles_n;
        const int nt = (int)blockIdx.x - mt * a.tiles_n;
        if (n_steps <= kChunk) fill_stages<1>(a, mt, nt, ring_s);
        else fill_stages<kPairStages>(a, mt, nt, ring_s);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // written through the generic proxy, read by the tensor core
        __syncthreads();
    }

    if (warp < kFirstPromoWarp) {
        setmaxnreg_dec<kRegsPairCtl>();
        if (warp == kProducerWarp) {
            // ------------------------------------------------------------ operand blocks
            const uint32_t empty_s = smem_u32(&g->empty[0]);
            uint32_t s = 0, ph = 1;
            for (int tile = blockIdx.x; !DIRECT && tile < n_tiles && !c->abort_flag; tile += gridDim.x) {
                const int mt = tile / a.tiles_n, nt = tile - mt * a.tiles_n;
                const uint8_t* a_src = a.a_blocks + (int64_t)mt * n_steps * kBlock;
                const uint8_t* b_src = a.b_blocks + (int64_t)nt * n_steps * kBHalf;
                const uint8_t* s_src = a.s_blocks + (int64_t)mt * n_steps * kScaleBlock;
#pragma unroll 1
                for (int k0 = 0; k0 < n_steps; k0 += kChunk) {
                    const uint32_t nk = (uint32_t)min(kChunk, n_steps - k0);
                    wait_hot(empty_s + s * 8, ph, c, a.status, 5u);
                    if (c->abort_flag) break;
                    if (elect_one()) {
                        const uint32_t st = ring_s + s * kPairStageBytes;
                        mbar_expect_tx(&g->full[s], nk * (kBlock + kBHalf + (SPG == 1 ? kScaleBlock : 0)));
                        bulk_load(st, a_src, nk * kBlock, &g->full[s]);
                        bulk_load(st + kChunk * kBlock, b_src, nk * kBHalf, &g->full[s]);
                        if (SPG == 1) bulk_load(st + kPairScales, s_src, nk * kScaleBlock, &g->full[s]);
                    }
                    __syncwarp();
                    a_src += kChunk * kBlock;
                    b_src += kChunk * kBHalf;
                    s_src += kChunk * kScaleBlock;
                    if (++s == kPairStages) { s = 0; ph ^= 1; }
                }
            }
        } else if (warp < kPairStoreWarp) {
            // ------------------------------------------------------------ MMA issue
            // Warp `me` owns slots 2 me and 2 me + 1, one group each, and reports a pair with one commit.
            const uint32_t me = (uint32_t)(warp - kFirstMmaWarp);
            const uint32_t full_s = smem_u32(&g->full[0]), empty_s = smem_u32(&g->empty[0]);
            const uint32_t tfull_s = smem_u32(&g->tfull[me]), tempty_s = smem_u32(&g->tempty[me]);
            const uint32_t tm = tmem_base + 2 * me * kN;
            const uint32_t a_lo = desc_lo(ring_s) + (SPG == 1 ? 2 * me * (kBlock >> 4) : 0u);
            const uint32_t b_lo = desc_lo(ring_s + kChunk * kBlock) + (SPG == 1 ? 2 * me * (kBHalf >> 4) : 0u);
            uint32_t s = 0, ph = 0;
            uint32_t q = 1;                      // parity to wait for on tempty; a fresh barrier passes parity 1
            for (int tile = blockIdx.x; SPG == 1 && tile < n_tiles && !c->abort_flag; tile += gridDim.x) {   // steps 2 me and 2 me + 1 of every stage
#pragma unroll 1
                for (int k0 = 0; k0 < n_steps; k0 += kChunk) {
                    const int mine = n_steps - k0 - 2 * (int)me;         // steps left from this warp's first one on
                    const uint32_t so = s * (kPairStageBytes >> 4);
                    const bool rf = DIRECT || mbar_test_s(full_s + s * 8, ph);    // the two tests are in flight together
                    const bool rt = mbar_test_s(tempty_s, q);
                    if (!rf) wait_cold(full_s + s * 8, ph, c, a.status, 4u);
                    if (mine > 0) {
                        if (!rt) wait_cold(tempty_s, q, c, a.status, 3u);
                        q ^= 1u;
                        tc_fence_after();
                        if (elect_one()) {
                            mma_f8(tm, desc_of(a_lo + so), desc_of(b_lo + so), kIdescN64);
                            if (mine > 1) mma_f8(tm + kN, desc_of(a_lo + so + (kBlock >> 4)), desc_of(b_lo + so + (kBHalf >> 4)), kIdescN64);
                            mma_commit(tfull_s);
                            if (!DIRECT) mma_commit(empty_s + s * 8);
                        }
                    } else if (!DIRECT && elect_one()) {
                        mma_commit(empty_s + s * 8);
                    }
                    __syncwarp();
                    if (++s == kPairStages) { s = 0; ph ^= 1; }
                }
            }
            // SPG > 1: one warp takes all the pairs.  (Two in turn would each skip stages of the ring, and a parity wait cannot
            // tell the phase a warp means from the one two phases before it that its neighbour has not got to yet.)
            uint32_t n = 0;                      // pairs of groups so far; pair n uses slots 2 (n & 1) and the next
            for (int tile = blockIdx.x; SPG > 1 && me == 0 && tile < n_tiles && !c->abort_flag; tile += gridDim.x) {
#pragma unroll 1
                for (int g0 = 0; g0 < a.Kg; g0 += 2, ++n) {
                    const int groups = min(2, a.Kg - g0), stages = SPG == 4 ? groups : 1;
                    const uint32_t p = n & 1u, d = tmem_base + 2 * p * kN;
                    const bool rt = mbar_test_s(tempty_s + p * 8, ((n >> 1) & 1u) ^ 1u);
                    bool rf = mbar_test_s(full_s + s * 8, ph);
                    if (!rt) wait_cold(tempty_s + p * 8, ((n >> 1) & 1u) ^ 1u, c, a.status, 3u);
#pragma unroll
                    for (int j = 0; j < (SPG == 4 ? 2 : 1); ++j) {
                        if (j >= stages) break;
                        if (!rf) wait_cold(full_s + s * 8, ph, c, a.status, 4u);
                        tc_fence_after();
                        if (elect_one()) {
                            const uint32_t so = s * (kPairStageBytes >> 4);
#pragma unroll
                            for (int k = 0; k < kChunk; ++k) {
                                const int slot = SPG == 4 ? j : k >> 1;
                                if (SPG == 4 || slot < groups)
                                    mma_f8(d + slot * kN, desc_of(a_lo + so + k * (kBlock >> 4)), desc_of(b_lo + so + k * (kBHalf >> 4)), kIdescN64,
                                           (k & (SPG - 1)) != 0 ? 1u : 0u);
                            }
                            if (j == stages - 1) mma_commit(tfull_s + p * 8);
                            mma_commit(empty_s + s * 8);
                        }
                        __syncwarp();
                        if (++s == kPairStages) { s = 0; ph ^= 1; }
                        if (j + 1 < stages) rf = mbar_test_s(full_s + s * 8, ph);
                    }
                }
            }
        } else {
            // ------------------------------------------------------------ output stores, channel constants
            // A staged tile is two boxes of 32 columns x 128 rows; the copy engine clips them at the edges of y.
            // The staging area goes back to the promotion warps when the engine has read it.  The same hand-over
            // carries the next tile's channel scales (times the accumulator's power of two) and biases: phase n of
            // `sfree` says that tile n of this CTA may be staged and that its constants are in place.
            constexpr uint32_t box_bytes = YBF16 ? kPairBoxBF16 : kPairBoxF32;
            float* wsb = reinterpret_cast<float*>(smem_raw + (wsb_s - sm_s));
            auto fetch = [&](int nt) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int64_t col = (int64_t)nt * kN + 32 * i + lane;
                    wsb[32 * i + lane] = col < a.O ? __fmul_rn(__ldg(a.wscale + col), a.out_scale) : 0.f;
                    wsb[kN + 32 * i + lane] = (a.bias && col < a.O) ? __ldg(a.bias + col) : 0.f;
                }
                __syncwarp();
            };
            uint32_t sph = 0;
            if ((int)blockIdx.x < n_tiles) {
                fetch((int)blockIdx.x % a.tiles_n);
                mbar_arrive_lane0(&g->sfree, lane);
            }
            for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
                const int mt = tile / a.tiles_n, nt = tile - mt * a.tiles_n;
                wait_hot(smem_u32(&g->sfull), sph, c, a.status, 8u);
                if (c->abort_flag) break;
                sph ^= 1u;
                if (lane == 0 && a.tma_ok) {
                    const int64_t n0 = (int64_t)nt * kN;
#pragma unroll
                    for (int cb = 0; cb < 2; ++cb)
                        if (n0 + 32 * cb < a.O)
                            tma_store_2d(&ymap, stage_s + (uint32_t)cb * box_bytes, (int32_t)n0 + 32 * cb, mt * kBM);
                    bulk_commit_group();
                }
                const int next = tile + (int)gridDim.x;
                if (next < n_tiles) fetch(next % a.tiles_n);
                if (lane == 0) bulk_wait_group_read0();
                __syncwarp();
                mbar_arrive_lane0(&g->sfree, lane);
            }
            if (lane == 0) bulk_wait_group0();   // no store may still be reading this CTA's shared memory at exit
        }
    } else {
        setmaxnreg_inc<kRegsPairPromo>();
        // ------------------------------------------------------------ promotion + epilogue
        const int quarter = warp & 3;                 // TMEM lanes 32 * quarter .. + 31
        const int row = quarter * 32 + lane;
        uint64_t yacc[kN / 2];                        // 64 floats of one output row, packed in pairs
        uint32_t va[32], vb[32], vc[32], vd[32];      // landing buffers: columns 0-31 and 32-63 of an even and of an odd slot
#pragma unroll
        for (int q = 0; q < 32; ++q) { va[q] = 0u; vb[q] = 0u; vc[q] = 0u; vd[q] = 0u; }
        uint32_t p_full = 0u;                         // bit p: parity of the completion of tfull[p] to wait for next
        uint32_t sf_par = 0u;                         // parity to wait for on sfree
        uint32_t rs = 0, rph = 0;                     // ring stage and its phase
        int tile = blockIdx.x, mt = 0, nt = 0;
        uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        const uint32_t full_s = smem_u32(&g->full[0]), empty_s = smem_u32(&g->empty[0]);
        uint32_t tmem_row = tmem_base + ((uint32_t)(quarter * 32) << 16);
        // opaque to the compiler: kept in registers instead of being recomputed from the thread index at every use
        asm volatile("" : "+r"(tfull_s), "+r"(tempty_s), "+r"(tmem_row));

        auto wait_pair = [&](uint32_t p, bool ready) {
            if (!ready) wait_cold(tfull_s + p * 8, (p_full >> p) & 1u, c, a.status, 2u);
            p_full ^= 1u << p;
            tc_fence_after();
        };
        auto load_lo = [&](uint32_t slot) { tmem_ld32(tmem_row + slot * kN, va); tmem_ld32(tmem_row + slot * kN + 32, vb); };
        auto load_hi = [&](uint32_t slot) { tmem_ld32(tmem_row + slot * kN, vc); tmem_ld32(tmem_row + slot * kN + 32, vd); };
        auto fold = [&](const uint32_t* x, const uint32_t* z, uint32_t dbits) {
            const uint64_t d2 = pack2(dbits, dbits);
#pragma unroll
            for (int q = 0; q < 16; ++q) fma2(yacc[q], pack2(x[2 * q], x[2 * q + 1]), d2);
#pragma unroll
            for (int q = 0; q < 16; ++q) fma2(yacc[16 + q], pack2(z[2 * q], z[2 * q + 1]), d2);
        };
        auto debug = [&](const uint32_t* x, const uint32_t* z, int k) {
            const int64_t m = (int64_t)mt * kBM + row;
            if (a.acc_debug && m < a.M) {
                debug_store<false>(a, x, m, (int64_t)nt * kN, k);
                debug_store<false>(a, z, m, (int64_t)nt * kN + 32, k);
            }
        };
        // The four steps Delta of the current ring stage for this row; then the stage is this warp's no longer.  (The
        // stage's scales came with its operands, so they are there when the first accumulator of the stage is.)
        uint32_t d[4];
        auto take_steps = [&](bool ready) {
            if (!DIRECT && !ready) wait_cold(full_s + rs * 8, rph, c, a.status, 7u);
            const uint32_t src = ring_s + rs * kPairStageBytes + kPairScales + (uint32_t)row * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) d[j] = lds32(src + j * kScaleBlock);
        };
        auto leave_stage = [&]() {
            if (!DIRECT) {
                // read through the generic proxy, refilled through the async proxy: only a proxy fence orders the two
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                mbar_arrive_lane0_s(empty_s + rs * 8, lane);
            }
            if (++rs == kPairStages) { rs = 0; rph ^= 1; }
        };

        // SPG > 1: the steps of groups k and k + 1 of row block `block` (zero past the end)
        auto global_steps = [&](uint32_t (&e)[4], int block, int k) {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(a.s_blocks) + ((int64_t)block * a.Kg + k) * kBM + row;
            e[0] = __ldg(src);
            e[1] = k + 1 < a.Kg ? __ldg(src + kBM) : 0u;
        };
        uint32_t n = 0;                               // SPG > 1: pairs of groups so far; pair n uses slots 2 (n & 1) and the next

        // A tile's groups are taken two at a time (a pair of slots): wait for the pair's landing, hand both slots back
        // with one arrival, fold the first group in, start the next pair's first load into the registers that frees, fold
        // the second, start the second load.
        if (tile < n_tiles) {
            mt = tile / a.tiles_n;
            nt = tile - mt * a.tiles_n;
            wait_pair(0, mbar_test_s(tfull_s, p_full & 1u));
            load_lo(0);
            if (a.Kg > 1) load_hi(1);
            if (SPG == 1) take_steps(mbar_test_s(full_s, 0u));
            else global_steps(d, mt, 0);
#pragma unroll 1
            while (!c->abort_flag) {
                // one tile; the load of its first pair is in flight, its first steps are in d
#pragma unroll
                for (int j = 0; j < kN / 2; ++j) yacc[j] = 0ull;
                const int next = tile + (int)gridDim.x;
                const bool another = next < n_tiles;
                const int mt_next = another ? next / a.tiles_n : mt;
#pragma unroll 1
                for (int k = 0; SPG > 1 && k < a.Kg; k += 2, ++n) {
                    const bool tile_end = k + 2 >= a.Kg, more = !tile_end || another;
                    const uint32_t p = (n + 1) & 1u;      // the next pair's slots
                    const bool r = more ? mbar_test_s(tfull_s + p * 8, (p_full >> p) & 1u) : true;
                    uint32_t e[4] = {0u, 0u, 0u, 0u};
                    if (more) global_steps(e, tile_end ? mt_next : mt, tile_end ? 0 : k + 2);
                    tmem_ld_wait_on(va); tmem_ld_wait_on(vb); tmem_ld_wait_on(vc); tmem_ld_wait_on(vd);
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0_s(tempty_s + (n & 1u) * 8, lane);
                    if (DBG) { debug(va, vb, k); if (k + 1 < a.Kg) debug(vc, vd, k + 1); }
                    fold(va, vb, d[0]);
                    if (more) { wait_pair(p, r); load_lo(2 * p); }
                    if (k + 1 < a.Kg) fold(vc, vd, d[1]);
                    if (more && (tile_end ? a.Kg > 1 : k + 3 < a.Kg)) load_hi(2 * p + 1);
                    d[0] = e[0];
                    d[1] = e[1];
                }
                int left = n_steps;                       // groups not yet folded in
#pragma unroll 1
                for (; SPG == 1;) {
                    // first pair of the stage: slots 0 and 1
                    const bool second = left > 2;         // the stage has another pair
                    bool r1 = true;
                    if (second) r1 = mbar_test_s(tfull_s + 8, (p_full >> 1) & 1u);
                    tmem_ld_wait_on(va); tmem_ld_wait_on(vb); tmem_ld_wait_on(vc); tmem_ld_wait_on(vd);
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0_s(tempty_s, lane);
                    if (DBG) { debug(va, vb, n_steps - left); if (left > 1) debug(vc, vd, n_steps - left + 1); }
                    fold(va, vb, d[0]);
                    if (second) { wait_pair(1, r1); load_lo(2); }
                    leave_stage();
                    if (left > 1) fold(vc, vd, d[1]);
                    if (!second) break;
                    if (left > 3) load_hi(3);
                    // second pair: slots 2 and 3
                    const bool more = left > 4;
                    bool r0 = true, rf = true;
                    if (more) {
                        r0 = mbar_test_s(tfull_s, p_full & 1u);
                        rf = mbar_test_s(full_s + rs * 8, rph);
                    }
                    tmem_ld_wait_on(va); tmem_ld_wait_on(vb); tmem_ld_wait_on(vc); tmem_ld_wait_on(vd);
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_lane0_s(tempty_s + 8, lane);
                    if (DBG) { debug(va, vb, n_steps - left + 2); if (left > 3) debug(vc, vd, n_steps - left + 3); }
                    fold(va, vb, d[2]);
                    if (more) { wait_pair(0, r0); load_lo(0); }
                    if (left > 3) fold(vc, vd, d[3]);
                    if (!more) break;
                    if (left > 5) load_hi(1);
                    take_steps(rf);
                    left -= 4;
                }
                if (SPG == 1 && another) {                // the next tile's first pair lands under the epilogue
                    wait_pair(0, mbar_test_s(tfull_s, p_full & 1u));
                    load_lo(0);
                    if (n_steps > 1) load_hi(1);
                    take_steps(mbar_test_s(full_s + rs * 8, rph));
                }

                // y = (s_o * 2^18) * sum + bias, parked as the source of the bulk tensor stores: box cb = columns
                // 32 cb .. + 31 of all 128 rows, rows of 128 bytes whose 16-byte chunk j sits at j ^ (row & 7) (fp32), or
                // rows of 64 bytes with chunk j at j ^ ((row >> 1) & 3) (16-bit types).
                wait_hot(smem_u32(&g->sfree), sf_par, c, a.status, 9u);   // the previous tile's stores have read the area
                sf_par ^= 1u;
                const float4* wsb4 = reinterpret_cast<const float4*>(smem_raw + (wsb_s - sm_s));
#pragma unroll
                for (int cb = 0; cb < 2; ++cb) {
                    const uint32_t row_s = stage_s + (uint32_t)cb * (YBF16 ? kPairBoxBF16 : kPairBoxF32) + (uint32_t)row * (YBF16 ? 64u : 128u);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {          // eight columns
                        const float4 sa = wsb4[8 * cb + 2 * j], sb = wsb4[8 * cb + 2 * j + 1];
                        const float4 ba = wsb4[kN / 4 + 8 * cb + 2 * j], bb = wsb4[kN / 4 + 8 * cb + 2 * j + 1];
                        float o[8];
                        unpack2(yacc[16 * cb + 4 * j], o[0], o[1]);
                        unpack2(yacc[16 * cb + 4 * j + 1], o[2], o[3]);
                        unpack2(yacc[16 * cb + 4 * j + 2], o[4], o[5]);
                        unpack2(yacc[16 * cb + 4 * j + 3], o[6], o[7]);
                        o[0] = __fmaf_rn(sa.x, o[0], ba.x); o[1] = __fmaf_rn(sa.y, o[1], ba.y);
                        o[2] = __fmaf_rn(sa.z, o[2], ba.z); o[3] = __fmaf_rn(sa.w, o[3], ba.w);
                        o[4] = __fmaf_rn(sb.x, o[4], bb.x); o[5] = __fmaf_rn(sb.y, o[5], bb.y);
                        o[6] = __fmaf_rn(sb.z, o[6], bb.z); o[7] = __fmaf_rn(sb.w, o[7], bb.w);
                        if (!YBF16) {
                            const uint32_t x7 = (uint32_t)lane & 7u;
                            sts128(row_s + (((uint32_t)(2 * j) ^ x7) << 4), __float_as_uint(o[0]), __float_as_uint(o[1]), __float_as_uint(o[2]), __float_as_uint(o[3]));
                            sts128(row_s + (((uint32_t)(2 * j + 1) ^ x7) << 4), __float_as_uint(o[4]), __float_as_uint(o[5]), __float_as_uint(o[6]), __float_as_uint(o[7]));
                        } else {
                            sts128(row_s + (((uint32_t)j ^ (((uint32_t)lane >> 1) & 3u)) << 4), pack16(o[0], o[1], a.y_f16), pack16(o[2], o[3], a.y_f16),
                                   pack16(o[4], o[5], a.y_f16), pack16(o[6], o[7], a.y_f16));
                        }
                    }
                }
                if (a.tma_ok) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the engine's reads
                    __syncwarp();
                } else {
                    // y off the 16-byte grid: the warp writes its own 32 rows, a row's columns side by side (two columns a
                    // lane where a pair of 16-bit values is one aligned word).  9217 x 160 -> 63 fp32 9.3 -> 8.6 us against
                    // the general kernel when both had the expansion in front.
                    __syncwarp();
                    const int64_t m0 = (int64_t)mt * kBM + quarter * 32, c0 = (int64_t)nt * kN;
                    const int rows = (int)min((int64_t)32, a.M - m0), cols = (int)min((int64_t)kN, a.O - c0);
                    uint8_t* out = reinterpret_cast<uint8_t*>(a.y) + (m0 * a.y_stride + c0) * (YBF16 ? 2 : 4);
                    const uint8_t* tile_sm = smem_raw + (stage_s - sm_s) + (uint32_t)(quarter * 32) * (YBF16 ? 64u : 128u);
                    // eight rows at a time: all their reads, then all their writes
                    constexpr int kBatch = 8;
#pragma unroll 1
                    for (int r0 = 0; r0 < rows; r0 += kBatch) {
                        uint32_t lo[kBatch], hi[kBatch];
#pragma unroll
                        for (int i = 0; i < kBatch; ++i) {
                            const uint32_t r = (uint32_t)(r0 + i);
                            if (!YBF16) {
                                const uint8_t* at = tile_sm + r * 128u + ((((uint32_t)lane >> 2) ^ (r & 7u)) << 4) + ((uint32_t)lane & 3u) * 4u;
                                lo[i] = *reinterpret_cast<const uint32_t*>(at);
                                hi[i] = *reinterpret_cast<const uint32_t*>(at + kPairBoxF32);
                            } else if (a.y_words) {
                                const uint32_t w = (uint32_t)lane & 15u;
                                lo[i] = *reinterpret_cast<const uint32_t*>(tile_sm + r * 64u + ((uint32_t)lane >> 4) * kPairBoxBF16 +
                                                                           (((w >> 2) ^ ((r >> 1) & 3u)) << 4) + (w & 3u) * 4u);
                                hi[i] = 0u;
                            } else {
                                const uint8_t* at = tile_sm + r * 64u + ((((uint32_t)lane >> 3) ^ ((r >> 1) & 3u)) << 4) + ((uint32_t)lane & 7u) * 2u;
                                lo[i] = *reinterpret_cast<const uint16_t*>(at);
                                hi[i] = *reinterpret_cast<const uint16_t*>(at + kPairBoxBF16);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < kBatch; ++i) {
                            if (r0 + i >= rows) break;
                            uint8_t* dst = out + (int64_t)(r0 + i) * a.y_stride * (YBF16 ? 2 : 4);
                            if (!YBF16) {
                                if (lane < cols) reinterpret_cast<uint32_t*>(dst)[lane] = lo[i];
                                if (lane + 32 < cols) reinterpret_cast<uint32_t*>(dst)[lane + 32] = hi[i];
                            } else if (a.y_words) {
                                if (2 * lane + 1 < cols) reinterpret_cast<uint32_t*>(dst)[lane] = lo[i];
                                else if (2 * lane < cols) reinterpret_cast<uint16_t*>(dst)[2 * lane] = (uint16_t)lo[i];
                            } else {
                                if (lane < cols) reinterpret_cast<uint16_t*>(dst)[lane] = (uint16_t)lo[i];
                                if (lane + 32 < cols) reinterpret_cast<uint16_t*>(dst)[lane + 32] = (uint16_t)hi[i];
                            }
                        }
                    }
                    __syncwarp();
                }
                mbar_arrive_lane0(&g->sfull, lane);
                if (!another) break;
                tile = next;
                mt = mt_next;
                nt = tile - mt * a.tiles_n;
            }
        }
        tmem_ld_wait();            // nothing may still be landing when TMEM is released
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kFirstMmaWarp) {
        // all MMAs this CTA issued have completed unless a wait gave up; in that case give the
        // tensor core a moment before the columns are handed back
        if (c->abort_flag) __nanosleep(1000000);
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kSlots * kN) : "memory");
    }
}

}  // namespace

// a.tiles_n and a.b_blocks are in units of 64 columns here (see ExpandArgs::b_rows).
tdq_status launch_linear_pair(const LinArgs& a, const CUtensorMap& ymap, int n_sm, int dev, bool ybf, bool dbg, bool direct,
                              cudaStream_t stream) {
    constexpr int kInst = 14;
    void (*const kernels[kInst])(LinArgs, CUtensorMap) = {
        w4a4_pair_kernel<false, false, 1>, w4a4_pair_kernel<true, false, 1>, w4a4_pair_kernel<false, true, 1>, w4a4_pair_kernel<true, true, 1>,
        w4a4_pair_kernel<false, false, 2>, w4a4_pair_kernel<true, false, 2>, w4a4_pair_kernel<false, true, 2>, w4a4_pair_kernel<true, true, 2>,
        w4a4_pair_kernel<false, false, 4>, w4a4_pair_kernel<true, false, 4>, w4a4_pair_kernel<false, true, 4>, w4a4_pair_kernel<true, true, 4>,
        w4a4_pair_kernel<false, false, 1, true>, w4a4_pair_kernel<true, false, 1, true>};
    const int inst = direct ? 12 + (ybf ? 1 : 0) : (ybf ? 1 : 0) + (dbg ? 2 : 0) + 4 * (a.steps_per_grp >> 1);
    if (inst >= kInst) return TDQ_ERR_UNSUPPORTED;
    void (*const kernel)(LinArgs, CUtensorMap) = kernels[inst];
    const uint32_t smem = kPairCtrl + kPairStages * kPairStageBytes + 1024 + 2 * (ybf ? kPairBoxBF16 : kPairBoxF32) + 2 * kN * 4;
    static_assert(kPairCtrl + kPairStages * kPairStageBytes + 1024 + 2 * kPairBoxF32 + 2 * kN * 4 <= 113 * 1024, "two CTAs per SM");
    static std::atomic<uint64_t> smem_done[kInst];
    if (allow_smem(kernel, 113 * 1024, smem_done[inst], dev) != cudaSuccess) return TDQ_ERR_CUDA;
    const int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
    const unsigned grid = (unsigned)(direct || tiles < 2 * n_sm ? tiles : 2 * n_sm);
    if (launch_pdl(kernel, dim3(grid), dim3(kPairThreads), smem, stream, a, ymap) != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

}  // namespace tdq
