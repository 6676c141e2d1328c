// The W4A4 linear layer (Algorithm S1 step 10 with Eq. 9 and Eq. 4 substituted) for groups of 32, 64 and 128 where there are
// several 128 x 128 tiles per SM:
//
//   acc[m,o,k] = sum_{i in group k} q_x[m,i] q_w[o,i]      SPG tcgen05.mma (E4M3 operands, exact) per group of 32 SPG codes
//   y[m,o]     = s_o * sum_k Delta[m,k] * acc[m,o,k] + b_o  fp32 in registers ("promotion")
//
// The arithmetic is that of tdq_linear_pair.cu and tdq_linear_g32.cu, bit for bit.
//
// What bounds it.  A tile costs its groups (per 128 x 128 group 160 clocks of packed multiply-adds, 2.5 clocks each, and the
// hand-over of a TMEM slot, of which there are four) and its epilogue, about 2000 clocks of shared-memory traffic for eight
// promotion warps.  The two-blocks-per-SM kernel (tdq_linear_pair.cu) spends 285 clocks a group and 2700 a tile: a block that
// is in its epilogue leaves its half of TMEM idle.  Here one block has all of TMEM, and a tile's epilogue is done during the
// next tile: its finished sums move to a second set of registers, and sixteen columns of them are scaled and parked along
// with each of the next tile's first four groups, under the waits for TMEM.  270 clocks a group, 1900 a tile.
//
//   warps 0, 1   operand blocks of A and of B, four K-steps a stage, through a ring
//   warps 2-5    MMA issue; group k of a tile goes to TMEM slot k & 3.  With one K-step per group warp 2 + j owns slot j; with
//                more, warp 2 takes all groups
//   warp 6       the staged tile's bulk tensor stores, and the next tile's channel constants
//   warp 7       the steps Delta of a tile (two tiles' in flight where they fit)
//   warps 8-15   promotion: 32 rows x 64 columns each; 64 sums, 64 finished sums and two 32-register landing buffers
//
// The hot loop has compile-time slots and nothing else in it: with the slot, the ring stage and the end of the tile as run-time
// values it ran 1.3 to 3 times slower (the scalar instructions are serial, and the compiler then copies the landing buffers).
//
// Measured (B200, with the expansion, from a graph), us against the kernels that took these layers before: 18464 x 768 -> 3072
// g = 32 fp32 117.9 -> 103.8, bf16 112.4 -> 101.7, g = 64 fp32 97.3 -> 81.5, g = 128 fp32 84.3 -> 79.9; 4616 x 768 -> 3072 g = 128
// fp16 23.8 -> 20.8; 18464 x 1024 -> 3072 g = 32 fp32 146.3 -> 129.8.
// Not kept: the epilogue in 32 KB of staging and two passes (the wait for the stores between them: 118.8 us on the first of
// these), its pieces spread over eight groups (111.8: the next tile then waits for the stores), sixteen promotion warps of 32
// columns (111.8), two sets of four promotion warps on tiles in turn (116.0), TMEM slots handed over by halves (103.7), ring
// stages of two K-steps (104.4); three ring stages instead of four are 119.3.
#include "tdq_tc.cuh"

namespace tdq {
namespace {

constexpr int kDeferCtlWarps = 8, kDeferPromoWarps = 8;
constexpr int kDeferThreads = (kDeferCtlWarps + kDeferPromoWarps) * 32;   // 512
constexpr int kRegsDeferCtl = 32, kRegsDeferPromo = 224;                  // 256 * 32 + 256 * 224 = 512 * 128
constexpr int kDeferProdA = 0, kDeferProdB = 1, kDeferMma0 = 2, kDeferStore = 6, kDeferProdS = 7;
constexpr int kDeferCols = 64;                                            // of a row, per promotion thread
constexpr uint32_t kDeferStageBytes = 2 * kChunk * kBlock;                // four K-steps of A, then of B
constexpr int kDeferMaxStages = 6;
constexpr uint32_t kDeferCtrl = 1024;
constexpr uint32_t kDeferBoxF32 = 128 * 128, kDeferBox16 = 128 * 64;      // one 32-column box of 128 rows in the staging area
// shared memory without the ring: control block, the steps of `bufs` tiles, the staged tile (on a 1 KB boundary) and its
// channel constants
constexpr int64_t defer_fixed(bool y16, int64_t Kg, int bufs) {
    return kDeferCtrl + bufs * Kg * kScaleBlock + 1024 + 4 * (y16 ? kDeferBox16 : kDeferBoxF32) + 2 * kBN * 4;
}
constexpr int64_t defer_stages(bool y16, int64_t Kg, int bufs) { return (kSmemLimit - defer_fixed(y16, Kg, bufs)) / kDeferStageBytes; }

struct DeferCtrl {
    uint64_t full[kDeferMaxStages], empty[kDeferMaxStages];
    uint64_t dfull[2], dempty[2];
    uint64_t tfull[kSlots], tempty[kSlots];
    uint64_t sfull, sfree;
};
static_assert(sizeof(Ctrl) + sizeof(DeferCtrl) <= kDeferCtrl, "control block outgrew its reservation");

template <bool YBF16, int SPG>
__global__ void __launch_bounds__(kDeferThreads, 1) w4a4_defer_kernel(const LinArgs a, const __grid_constant__ CUtensorMap ymap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    constexpr int kPer = kChunk / SPG;                       // groups per chunk (a ring stage: four K-steps)
    Ctrl* c = reinterpret_cast<Ctrl*>(smem_raw);             // its abort flag and TMEM address; the barriers are g's
    DeferCtrl* g = reinterpret_cast<DeferCtrl*>(smem_raw + sizeof(Ctrl));
    const uint32_t sm_s = smem_u32(smem_raw);
    const uint32_t ring_s = sm_s + kDeferCtrl;
    const uint32_t n_stages = (uint32_t)a.n_stages;
    const uint32_t steps_s = ring_s + n_stages * kDeferStageBytes, steps_bytes = (uint32_t)a.Kg * kScaleBlock;
    const uint32_t stage_s = (steps_s + (uint32_t)a.n_ibuf * steps_bytes + 1023u) & ~1023u;   // the swizzle patterns repeat every 1024 bytes
    const uint32_t wsb_s = stage_s + 4 * (YBF16 ? kDeferBox16 : kDeferBoxF32);        // [128] channel scales, [128] biases
    const int warp = uniform_warp(), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kDeferMaxStages; ++i) { mbar_init(&g->full[i], 2); mbar_init(&g->empty[i], SPG == 1 ? kSlots : 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&g->dfull[i], 1); mbar_init(&g->dempty[i], kDeferPromoWarps); }
        for (int i = 0; i < kSlots; ++i) { mbar_init(&g->tfull[i], 1); mbar_init(&g->tempty[i], kDeferPromoWarps); }
        mbar_init(&g->sfull, kDeferPromoWarps);
        mbar_init(&g->sfree, 1);
        c->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kDeferMma0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();          // barrier set-up and the TMEM allocation overlap the tail of the kernel before this one
    pdl_trigger();
    const uint32_t tmem_base = c->tmem_base;
    const uint32_t buf_mask = (uint32_t)a.n_ibuf - 1u, buf_shift = buf_mask;   // tile n's steps are in buffer n & mask, phase n >> shift
    const int n_tiles = a.tiles_m * a.tiles_n, n_steps = a.n_steps;

    if (warp < kDeferCtlWarps) {
        setmaxnreg_dec<kRegsDeferCtl>();
        if (warp == kDeferProdA || warp == kDeferProdB) {
            // ------------------------------------------------------------ operand blocks of A or of B
            const bool is_b = warp == kDeferProdB;
            const uint32_t empty_s = smem_u32(&g->empty[0]);
            const uint32_t dst = ring_s + (is_b ? kChunk * kBlock : 0u);
            uint32_t s = 0, ph = 1;
            for (int tile = blockIdx.x; tile < n_tiles && !c->abort_flag; tile += gridDim.x) {
                const int mt = tile / a.tiles_n;
                const uint8_t* src = (is_b ? a.b_blocks : a.a_blocks) + (int64_t)(is_b ? tile - mt * a.tiles_n : mt) * n_steps * kBlock;
#pragma unroll 1
                for (int k0 = 0; k0 < n_steps; k0 += kChunk) {
                    const uint32_t bytes = (uint32_t)min(kChunk, n_steps - k0) * kBlock;
                    wait_hot(empty_s + s * 8, ph, c, a.status, 5u);
                    if (c->abort_flag) break;
                    if (elect_one()) {
                        mbar_expect_tx(&g->full[s], bytes);
                        bulk_load(dst + s * kDeferStageBytes, src, bytes, &g->full[s]);
                    }
                    __syncwarp();
                    src += kChunk * kBlock;
                    if (++s == n_stages) { s = 0; ph ^= 1; }
                }
            }
        } else if (warp == kDeferProdS) {
            // ------------------------------------------------------------ steps Delta, a tile at a time, two in flight
            uint32_t n = 0;
            for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++n) {
                const uint8_t* src = a.s_blocks + (int64_t)(tile / a.tiles_n) * steps_bytes;
                const uint32_t buf = n & buf_mask;
                wait_hot(smem_u32(&g->dempty[buf]), ((n >> buf_shift) & 1u) ^ 1u, c, a.status, 6u);
                if (c->abort_flag) break;
                if (elect_one()) {
                    mbar_expect_tx(&g->dfull[buf], steps_bytes);
                    for (uint32_t off = 0; off < steps_bytes; off += 16384u)
                        bulk_load(steps_s + buf * steps_bytes + off, src + off, min(16384u, steps_bytes - off), &g->dfull[buf]);
                }
                __syncwarp();
            }
        } else if (warp < kDeferStore) {
            // ------------------------------------------------------------ MMA issue
            // Group k of a tile goes to slot k & 3.  One K-step per group: this warp owns slot `me`.  More: one warp takes all
            // groups.
            const uint32_t me = (uint32_t)(warp - kDeferMma0);
            const uint32_t full_s = smem_u32(&g->full[0]), empty_s = smem_u32(&g->empty[0]);
            const uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
            const uint32_t a_lo = desc_lo(ring_s) + (SPG == 1 ? me * (kBlock >> 4) : 0u);
            const uint32_t b_lo = desc_lo(ring_s + kChunk * kBlock) + (SPG == 1 ? me * (kBlock >> 4) : 0u);
            uint32_t s = 0, ph = 0;
            uint32_t q = SPG == 1 ? 1u : 15u;      // parity to wait for on tempty (SPG > 1: bit s for slot s); a fresh barrier passes parity 1
            for (int tile = blockIdx.x; (SPG == 1 || me == 0) && tile < n_tiles && !c->abort_flag; tile += gridDim.x) {
#pragma unroll 1
                for (int k0 = 0; k0 < n_steps; k0 += kChunk) {
                    const int left = n_steps - k0;         // K-steps of the tile from this chunk on
                    const uint32_t so = s * (kDeferStageBytes >> 4);
                    if (SPG == 1) {
                        const bool mine = (int)me < left;
                        const bool rf = mbar_test_s(full_s + s * 8, ph);   // the two tests are in flight together
                        const bool rt = mbar_test_s(tempty_s + me * 8, q);
                        if (!rf) wait_cold(full_s + s * 8, ph, c, a.status, 4u);
                        if (mine) {
                            if (!rt) wait_cold(tempty_s + me * 8, q, c, a.status, 3u);
                            q ^= 1u;
                        }
                        tc_fence_after();
                        if (elect_one()) {
                            if (mine) {
                                mma_f8(tmem_base + me * kBN, desc_of(a_lo + so), desc_of(b_lo + so), kIdescF8);
                                mma_commit(tfull_s + me * 8);
                            }
                            mma_commit(empty_s + s * 8);
                        }
                        __syncwarp();
                    } else {
                        wait_hot(full_s + s * 8, ph, c, a.status, 4u);
#pragma unroll
                        for (int u = 0; u < kPer; ++u) {
                            if (u * SPG < left) {
                                const uint32_t slot = (uint32_t)((k0 / SPG + u) & (kSlots - 1));
                                wait_hot(tempty_s + slot * 8, (q >> slot) & 1u, c, a.status, 3u);
                                q ^= 1u << slot;
                                tc_fence_after();
                                if (elect_one()) {
#pragma unroll
                                    for (int k = 0; k < SPG; ++k)
                                        mma_f8(tmem_base + slot * kBN, desc_of(a_lo + so + (u * SPG + k) * (kBlock >> 4)),
                                               desc_of(b_lo + so + (u * SPG + k) * (kBlock >> 4)), kIdescF8, k ? 1u : 0u);
                                    mma_commit(tfull_s + slot * 8);
                                }
                                __syncwarp();
                            }
                        }
                        if (elect_one()) mma_commit(empty_s + s * 8);
                        __syncwarp();
                    }
                    if (++s == n_stages) { s = 0; ph ^= 1; }
                }
            }
        } else {
            // ------------------------------------------------------------ output stores, channel constants
            // A staged tile is four boxes of 32 columns x 128 rows; the copy engine clips them at the edges of y.  Phase n
            // of sfree says that tile n of this block may be staged: the engine has read the tile before it, and the
            // tile's constants are in place.
            constexpr uint32_t box_bytes = YBF16 ? kDeferBox16 : kDeferBoxF32;
            float* wsb = reinterpret_cast<float*>(smem_raw + (wsb_s - sm_s));
            auto fetch = [&](int nt) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int64_t col = (int64_t)nt * kBN + 32 * i + lane;
                    wsb[32 * i + lane] = col < a.O ? __fmul_rn(__ldg(a.wscale + col), a.out_scale) : 0.f;
                    wsb[kBN + 32 * i + lane] = (a.bias && col < a.O) ? __ldg(a.bias + col) : 0.f;
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
                if (lane == 0) {
                    const int64_t n0 = (int64_t)nt * kBN;
#pragma unroll
                    for (int cb = 0; cb < 4; ++cb)
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
        setmaxnreg_inc<kRegsDeferPromo>();
        // ------------------------------------------------------------ promotion + epilogue
        const int quarter = warp & 3;                 // TMEM lanes 32 * quarter .. + 31
        const int half = (warp - kDeferCtlWarps) >> 2;   // columns 64 * half .. + 63 of the tile
        const int row = quarter * 32 + lane;
        uint64_t yacc[kDeferCols / 2];                // this tile's sums, packed in pairs
        uint64_t done[kDeferCols / 2];                // the finished sums of the tile before it
        uint32_t va[32], vb[32];                      // landing buffers: columns 0-31 and 32-63 of this thread's share of a slot
#pragma unroll
        for (int q = 0; q < 32; ++q) { va[q] = 0u; vb[q] = 0u; yacc[q] = 0ull; done[q] = 0ull; }
        uint32_t p_full[kSlots] = {0u, 0u, 0u, 0u};   // parity of the completion of tfull[s] to wait for next
        uint32_t sf_par = 0u;                         // parity to wait for on sfree
        uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        uint32_t tmem_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * kDeferCols);
        uint32_t my_row = stage_s + (uint32_t)(2 * half) * (YBF16 ? kDeferBox16 : kDeferBoxF32) + (uint32_t)row * (YBF16 ? 64u : 128u);
        const uint32_t swz = YBF16 ? ((uint32_t)lane >> 1) & 3u : (uint32_t)lane & 7u;
        uint32_t wsb_half = wsb_s + (uint32_t)half * (kDeferCols * 4);
        // opaque to the compiler: kept in registers instead of being recomputed from the thread index at every use
        asm volatile("" : "+r"(tfull_s), "+r"(tempty_s), "+r"(tmem_row), "+r"(my_row), "+r"(wsb_half));
        int tile = blockIdx.x;

        // Eight columns (8 i .. 8 i + 7) of the finished tile: y = (s_o * 2^18) * sum + bias, parked as the source of the bulk
        // tensor stores: box cb = columns 32 cb .. + 31 of all 128 rows, rows of 128 bytes whose 16-byte chunk j sits at
        // j ^ (row & 7) (fp32), or rows of 64 bytes with chunk j at j ^ ((row >> 1) & 3) (16-bit types).
        uint64_t cs[4], cb[4];                        // their constants, fetched ahead of their use
        auto fetch = [&](int i) {
            lds128(wsb_half + 32 * i, cs[0], cs[1]);
            lds128(wsb_half + 32 * i + 16, cs[2], cs[3]);
            lds128(wsb_half + kBN * 4 + 32 * i, cb[0], cb[1]);
            lds128(wsb_half + kBN * 4 + 32 * i + 16, cb[2], cb[3]);
        };
        auto park = [&](int i) {
            float f[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                fma2(cb[q], done[4 * i + q], cs[q]);
                unpack2(cb[q], f[2 * q], f[2 * q + 1]);
            }
            const uint32_t at = my_row + (uint32_t)(i >> 2) * (YBF16 ? kDeferBox16 : kDeferBoxF32);
            const uint32_t w = (uint32_t)(i & 3);
            if (!YBF16) {
                sts128(at + (((2 * w) ^ swz) << 4), __float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
                sts128(at + (((2 * w + 1) ^ swz) << 4), __float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]), __float_as_uint(f[7]));
            } else {
                sts128(at + ((w ^ swz) << 4), pack16(f[0], f[1], a.y_f16), pack16(f[2], f[3], a.y_f16), pack16(f[4], f[5], a.y_f16), pack16(f[6], f[7], a.y_f16));
            }
        };
        auto stage_begin = [&]() {                    // the previous tile's stores have read the area, the constants are there
            wait_hot(smem_u32(&g->sfree), sf_par, c, a.status, 9u);
            sf_par ^= 1u;
        };
        auto stage_end = [&]() {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the engine's reads
            __syncwarp();
            mbar_arrive_lane0(&g->sfull, lane);
        };
        auto flush = [&]() {
            stage_begin();
#pragma unroll
            for (int i = 0; i < 8; ++i) { fetch(i); park(i); }
            stage_end();
        };

        // Starts the load of the first half of a tile's first group (slot 0) into va.
        auto first_load = [&]() {
            wait_hot(tfull_s, p_full[0], c, a.status, 2u);
            p_full[0] ^= 1u;
            tc_fence_after();
            tmem_ld32(tmem_row, va);
        };
        // One group (slot U) whose first half is on its way into va: start the second half, fold the first in, hand the slot
        // back once the second has landed, start the next group's first half (`more`), fold the second in.  P: the part of the
        // finished tile's epilogue that runs along (sixteen columns), or -1.  A barrier test answers about a hundred clocks
        // after it is issued and a shared-memory load after about thirty, so both are issued well before their results are
        // needed.
        uint32_t dnext = 0u;
        auto group = [&](auto u_tag, auto p_tag, uint32_t scale_q, bool more) {
            constexpr uint32_t U = decltype(u_tag)::value, N = (U + 1) & (kSlots - 1);
            constexpr int P = decltype(p_tag)::value;
            const bool rn = more ? mbar_test_s(tfull_s + N * 8, p_full[N]) : true;
            const uint64_t d2 = pack2(dnext, dnext);
            if (P == 0) stage_begin();
            if (P >= 0) fetch(2 * P);
            tmem_ld_wait_on(va);
            tmem_ld32(tmem_row + U * kBN + 32, vb);
#pragma unroll
            for (int q = 0; q < 16; ++q) fma2(yacc[q], pack2(va[2 * q], va[2 * q + 1]), d2);
            if (P >= 0) { park(2 * P); fetch(2 * P + 1); }
            tmem_ld_wait_on(vb);
            tc_fence_before();                            // the slot is drained
            __syncwarp();
            mbar_arrive_lane0_s(tempty_s + U * 8, lane);
            if (more) {
                if (!rn) wait_cold(tfull_s + N * 8, p_full[N], c, a.status, 2u);
                p_full[N] ^= 1u;
                tc_fence_after();
                tmem_ld32(tmem_row + N * kBN, va);
            }
            // the step of the group after this one (past the tile's last group this reads the start of the next region of
            // shared memory; the value is then replaced before it is used)
            dnext = lds32(scale_q + (U + 1) * kScaleBlock);
#pragma unroll
            for (int q = 0; q < 16; ++q) fma2(yacc[16 + q], pack2(vb[2 * q], vb[2 * q + 1]), d2);
            if (P >= 0) park(2 * P + 1);
            if (P == 3) stage_end();
        };
        const std::integral_constant<int, 0> u0{};
        const std::integral_constant<int, 1> u1{};
        const std::integral_constant<int, 2> u2{};
        const std::integral_constant<int, 3> u3{};
        const std::integral_constant<int, -1> none{};
        if (tile < n_tiles) {
            bool pending = false;                         // a finished tile waits in `done`
            uint32_t n = 0;                               // tiles so far
            first_load();
#pragma unroll 1
            while (!c->abort_flag) {
                // one tile; the first half of its first group is in flight
                const int Kg = a.Kg;
                const uint32_t buf = n & buf_mask;
                uint32_t scale_q = steps_s + buf * steps_bytes + (uint32_t)row * 4;
                wait_hot(smem_u32(&g->dfull[buf]), (n >> buf_shift) & 1u, c, a.status, 7u);
                dnext = lds32(scale_q);
                int k = 0;
                if (pending) {
                    if (Kg > 4) {
                        group(u0, u0, scale_q, true);
                        group(u1, u1, scale_q, true);
                        group(u2, u2, scale_q, true);
                        group(u3, u3, scale_q, true);
                        k = 4;
                        scale_q += 4 * kScaleBlock;
                    } else {
                        flush();
                    }
                }
#pragma unroll 1
                for (; k + 4 < Kg; k += 4, scale_q += 4 * kScaleBlock) {   // four groups, and more behind them
                    group(u0, none, scale_q, true);
                    group(u1, none, scale_q, true);
                    group(u2, none, scale_q, true);
                    group(u3, none, scale_q, true);
                }
                const int rem = Kg - k;                   // the last one to four groups
                group(u0, none, scale_q, rem > 1);
                if (rem > 1) {
                    group(u1, none, scale_q, rem > 2);
                    if (rem > 2) {
                        group(u2, none, scale_q, rem > 3);
                        if (rem > 3) group(u3, none, scale_q, false);
                    }
                }
                // the steps were read through the generic proxy and are overwritten through the async proxy: only a proxy fence
                // orders the two
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                mbar_arrive_lane0(&g->dempty[buf], lane);
                ++n;
                tile += (int)gridDim.x;
                if (tile < n_tiles) first_load();
#pragma unroll
                for (int q = 0; q < kDeferCols / 2; ++q) { done[q] = yacc[q]; yacc[q] = 0ull; }
                pending = true;
                if (tile >= n_tiles) break;
            }
            if (pending && !c->abort_flag) flush();
        }
        tmem_ld_wait();            // nothing may still be landing when TMEM is released
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kDeferMma0) {
        // all MMAs this CTA issued have completed unless a wait gave up; in that case give the
        // tensor core a moment before the columns are handed back
        if (c->abort_flag) __nanosleep(1000000);
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

}  // namespace

// The steps of one tile and three ring stages have to fit: up to 128 groups (fp32 y) or 192.
bool linear_defer_fits(bool y16, int32_t Kg) { return defer_stages(y16, Kg, 1) >= 3; }

tdq_status launch_linear_defer(LinArgs a, const CUtensorMap& ymap, int n_sm, int dev, bool ybf, cudaStream_t stream) {
    constexpr int kInst = 6;
    void (*const kernels[kInst])(LinArgs, CUtensorMap) = {
        w4a4_defer_kernel<false, 1>, w4a4_defer_kernel<true, 1>, w4a4_defer_kernel<false, 2>,
        w4a4_defer_kernel<true, 2>, w4a4_defer_kernel<false, 4>, w4a4_defer_kernel<true, 4>};
    const int inst = (ybf ? 1 : 0) + 2 * (a.steps_per_grp >> 1);
    if (inst >= kInst || !a.tma_ok || !linear_defer_fits(ybf, a.Kg)) return TDQ_ERR_UNSUPPORTED;
    a.n_ibuf = defer_stages(ybf, a.Kg, 2) >= 3 ? 2 : 1;
    const int64_t stages = defer_stages(ybf, a.Kg, a.n_ibuf);
    a.n_stages = (int32_t)(stages < kDeferMaxStages ? stages : kDeferMaxStages);
    const uint32_t smem = (uint32_t)(defer_fixed(ybf, a.Kg, a.n_ibuf) + (int64_t)a.n_stages * kDeferStageBytes);
    static std::atomic<uint64_t> smem_done[kInst];
    if (allow_smem(kernels[inst], kSmemLimit, smem_done[inst], dev) != cudaSuccess) return TDQ_ERR_CUDA;
    const int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
    if (launch_pdl(kernels[inst], dim3((unsigned)(tiles < n_sm ? tiles : n_sm)), dim3(kDeferThreads), smem, stream, a, ymap) != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

}  // namespace tdq
