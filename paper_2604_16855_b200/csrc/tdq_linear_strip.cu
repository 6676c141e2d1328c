// The W4A4 linear layer at the paper's group size g = 32 (Algorithm S1 step 10 with Eq. 9 and Eq. 4 substituted) for
// contractions of up to 512 channels (768 with a single column tile) with a few 128 x 128 tiles per SM, from the packed codes in
// one launch:
//
//   acc[m,o,k] = sum_{i in group k} q_x[m,i] q_w[o,i]      one tcgen05.mma (E4M3 operands, exact) per group
//   y[m,o]     = s_o * sum_k Delta[m,k] * acc[m,o,k] + b_o  fp32 in registers ("promotion")
//
// bit for bit what the other kernels of the layer compute.
//
// What bounds it.  These layers have a few microseconds of work per SM, and an expansion kernel in front costs five: a gap, its
// own three, and the wait of the kernel behind it for blocks that come back out of L2.  So a block makes its operands
// from the packed codes itself.  That only pays if a row of A is not expanded again for every column tile: a block takes a run of
// tiles that are neighbours in a row block, and a row block's operands stay in shared memory while the columns of B pass by.
// The two 64-column halves of a tile have a pipeline each (operands, ring, MMA warp, four TMEM slots, promotion warps, staging
// area) that only share A, so one's waits and epilogue run under the other's multiply-adds.
//
//   warps 0, 1    MMA issue for half 0 and half 1; group k of a chunk of four goes to slot k of 64 columns
//   warps 2, 3    a staged half's bulk tensor stores, and the next tile's channel constants
//   warps 4-11    operands: four warps per half bring the half's B through a ring, and every other chunk (four K-steps) of A and
//                 of the steps Delta when a new row block begins
//   warps 12-19   promotion and epilogue: 32 rows x 64 columns each; 64 sums and two 32-register landing buffers
//
// Measured (B200, quantizer and layer through the binding), us, against the expansion and the kernels behind it: 73728 x 64 -> 256
// fp32 32.5 -> 28.0, 18432 x 128 -> 384 20.5 -> 16.9, 9216 x 320 -> 960 bf16 24.6 -> 22.9, 1152 x 384 -> 1536 14.5 -> 12.1, 73728 x 320 -> 128
// bf16 45.1 -> 38.9; the encoder's 32 layers at batch 8 672 -> 625.  Both sides at more sizes are beside the rule in tdq_linear.cu.  A group
// of 128 x 128 takes 330 clocks and a tile 2000 more, against 270 and 1900 in tdq_linear_defer.cu, whose issue slots the
// operands' warps do not share: 18464 x 768 -> 3072 is 105 us there and 133 here.
// Not kept: 32 columns per promotion thread, eight slots and the epilogue along with the next tile (400 clocks per 128 x 64
// group, all in the instructions around the multiply-adds: 9216 x 320 -> 960 24.3 us for the layer alone, now 16.4); weights as sign
// and magnitude (19.3); each chunk of A split between the halves (16.5, and 0.2 to 0.4 slower with 512 channels).
#include "tdq_tc.cuh"

namespace tdq {
namespace {

constexpr int kStripN = 64;                                 // columns of half a tile = one TMEM slot
constexpr int kStripCtlWarps = 4, kStripExpWarps = 8, kStripPromoWarps = 8;
constexpr int kStripThreads = (kStripCtlWarps + kStripExpWarps + kStripPromoWarps) * 32;   // 640
constexpr int kRegsStripCtl = 40, kRegsStripExp = 48, kRegsStripPromo = 168;               // 128 * 40 + 256 * 48 + 256 * 168 <= 640 * 96
constexpr int kStripMaxStages = 3, kStripMaxChunks = 8;     // of B, per half; of A, all row blocks that are held
// K-steps are 32 bytes off a multiple of 128 bytes apart, so that the four lanes that write a row's four K-steps meet different banks
constexpr uint32_t kStripABlk = kBlock + 32, kStripBBlk = kStripN * 32 + 32;
constexpr uint32_t kStripSteps = kChunk * kStripABlk;       // of a chunk of A: four K-steps' operands, then the steps Delta
constexpr uint32_t kStripABytes = kStripSteps + kChunk * kScaleBlock, kStripBBytes = kChunk * kStripBBlk;
constexpr uint32_t kStripCtrl = 1024;
constexpr uint32_t kStripBoxF32 = 128 * 128, kStripBox16 = 128 * 64;   // one 32-column box of 128 rows in the staging area
constexpr uint32_t kStripConsts = 2 * kStripN * 4;          // channel scales and biases of half a tile
constexpr uint32_t kIdescStrip = (1u << 4) | ((uint32_t)(kStripN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);

struct StripCtrl {
    uint64_t afull[kStripMaxChunks], aempty[kStripMaxChunks];
    uint64_t full[2][kStripMaxStages], empty[2][kStripMaxStages];
    uint64_t tfull[2][kChunk], tempty[2][kChunk];
    uint64_t sfull[2], sfree[2];
};
static_assert(sizeof(Ctrl) + sizeof(StripCtrl) <= kStripCtrl, "control block outgrew its reservation");

// 32 packed codes -> operand bytes (E4M3).  The channels of a group may be summed in any order, so the two nibbles of a byte stay
// apart in both operands: even channels, then odd ones.  Activations, expanded once per row block, become sign and magnitude
// in units of 2^-9.  The byte n is the number n 2^-9 for n = 0..15, so a weight takes one bit operation as q + 8, and an
// instruction with a constant block of -8 in front takes 8 sum q_x off again (exact: everything is below 2^12 in units
// of 2^-18); sign and magnitude would cost five times as much, for every column tile.
__device__ __forceinline__ void put_acts(uint32_t dst, const uint4& p) {
    const uint32_t w[4] = {p.x, p.y, p.z, p.w};
    uint32_t e[4], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        e[i] = to_sign_magnitude((w[i] << 4) & 0xF0F0F0F0u);
        o[i] = to_sign_magnitude(w[i] & 0xF0F0F0F0u);
    }
    sts128(dst, e[0], e[1], e[2], e[3]);
    sts128(dst + 128, o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ void put_weights(uint32_t dst, const uint4& p) {
    const uint32_t w[4] = {p.x, p.y, p.z, p.w};
    uint32_t e[4], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        e[i] = (w[i] & 0x0F0F0F0Fu) ^ 0x08080808u;
        o[i] = ((w[i] >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
    }
    sts128(dst, e[0], e[1], e[2], e[3]);
    sts128(dst + 128, o[0], o[1], o[2], o[3]);
}

// Row block `rb` (counted from the block's first) and chunk i: its place among the chunks of A, and how often the place was used
// before.
struct AChunks {
    uint32_t buf = 0, use = 0;
    __device__ __forceinline__ void next(uint32_t bufs) { if (++buf == bufs) { buf = 0; use ^= 1u; } }
};

// a.n_stages: stages of B in each half's ring; a.n_ibuf: row blocks of A held
template <bool Y16>
__global__ void __launch_bounds__(kStripThreads, 1) w4a4_strip_kernel(const LinArgs a, const __grid_constant__ CUtensorMap ymap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    constexpr uint32_t kBox = Y16 ? kStripBox16 : kStripBoxF32;
    Ctrl* c = reinterpret_cast<Ctrl*>(smem_raw);             // its abort flag and TMEM address; the barriers are g's
    StripCtrl* g = reinterpret_cast<StripCtrl*>(smem_raw + sizeof(Ctrl));
    const int n_steps = a.n_steps, chunks = (n_steps + kChunk - 1) / kChunk;
    const uint32_t n_stages = (uint32_t)a.n_stages, n_bufs = (uint32_t)a.n_ibuf;
    const uint32_t sm_s = smem_u32(smem_raw);
    const uint32_t minus_s = sm_s + kStripCtrl;              // an operand block of -8
    const uint32_t a_s = minus_s + kStripN * 32, buf_bytes = (uint32_t)chunks * kStripABytes;
    const uint32_t b_s = a_s + n_bufs * buf_bytes;
    const uint32_t stage_s = (b_s + 2 * n_stages * kStripBBytes + 1023u) & ~1023u;   // the swizzle patterns repeat every 1024 bytes
    const uint32_t wsb_s = stage_s + 4 * kBox;
    const int t = threadIdx.x, warp = uniform_warp(), lane = t & 31;

    if (t == 0) {
        for (int i = 0; i < kStripMaxChunks; ++i) { mbar_init(&g->afull[i], 4); mbar_init(&g->aempty[i], kStripPromoWarps); }
        for (int h = 0; h < 2; ++h) {
            for (int i = 0; i < kStripMaxStages; ++i) { mbar_init(&g->full[h][i], 4); mbar_init(&g->empty[h][i], 1); }
            for (int i = 0; i < kChunk; ++i) { mbar_init(&g->tfull[h][i], 1); mbar_init(&g->tempty[h][i], 4); }
            mbar_init(&g->sfull[h], 4);
            mbar_init(&g->sfree[h], 1);
        }
        c->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem_base)), "r"(2 * kChunk * kStripN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t >= 128 && t < 128 + kStripN * 2) {
        sts128(minus_s + (uint32_t)(t - 128) * 16, 0x88888888u, 0x88888888u, 0x88888888u, 0x88888888u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // written through the generic proxy, read by the tensor core
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();          // barrier set-up and the TMEM allocation overlap the tail of the kernel before this one
    pdl_trigger();
    if (blockIdx.x == 0 && t < 4) a.status[t] = 0u;
    const uint32_t tmem_base = c->tmem_base;
    // this block's run of tiles, column tiles of a row block next to each other
    const int64_t n_tiles = (int64_t)a.tiles_m * a.tiles_n;
    const int t0 = (int)(n_tiles * blockIdx.x / gridDim.x), t1 = (int)(n_tiles * (blockIdx.x + 1) / gridDim.x);
    const int mt0 = t0 / a.tiles_n, nt0 = t0 - mt0 * a.tiles_n;
    const uint32_t afull_s = smem_u32(&g->afull[0]), aempty_s = smem_u32(&g->aempty[0]);

    if (warp < kStripCtlWarps) {
        setmaxnreg_dec<kRegsStripCtl>();
        const int h = warp & 1;
        if (warp < 2) {
            // ------------------------------------------------------------ MMA issue
            const uint32_t full_s = smem_u32(&g->full[h][0]), empty_s = smem_u32(&g->empty[h][0]);
            const uint32_t tfull_s = smem_u32(&g->tfull[h][0]), tempty_s = smem_u32(&g->tempty[h][0]);
            const uint32_t d = tmem_base + (uint32_t)h * (kChunk * kStripN);
            const uint32_t m_lo = desc_lo(minus_s), a_lo = desc_lo(a_s), b_lo = desc_lo(b_s + (uint32_t)h * n_stages * kStripBBytes);
            uint32_t s = 0, ph = 0;
            uint32_t q = 15u;                        // bit i: parity to wait for on tempty[i]; a fresh barrier passes parity 1
            AChunks ac;
            int nt = nt0;
            for (int tile = t0; tile < t1 && !c->abort_flag; ++tile) {
                const bool fresh = nt == 0 || tile == t0;                // the row block's first tile in this block
                uint32_t a_at = a_lo + ac.buf * (buf_bytes >> 4), slot = ac.buf * (uint32_t)chunks;
#pragma unroll 1
                for (int k0 = 0; k0 < n_steps; k0 += kChunk, ++slot) {
                    const uint32_t b_at = b_lo + s * (kStripBBytes >> 4);
                    if (fresh) wait_hot(afull_s + slot * 8, ac.use, c, a.status, 6u);
                    wait_hot(full_s + s * 8, ph, c, a.status, 4u);
#pragma unroll
                    for (int u = 0; u < kChunk; ++u) {
                        if (k0 + u < n_steps) {
                            wait_hot(tempty_s + u * 8, (q >> u) & 1u, c, a.status, 3u);
                            q ^= 1u << u;
                            tc_fence_after();
                            if (elect_one()) {
                                mma_f8(d + u * kStripN, desc_of(a_at + u * (kStripABlk >> 4)), desc_of(m_lo), kIdescStrip);
                                mma_f8(d + u * kStripN, desc_of(a_at + u * (kStripABlk >> 4)), desc_of(b_at + u * (kStripBBlk >> 4)), kIdescStrip, 1u);
                                mma_commit(tfull_s + u * 8);
                            }
                            __syncwarp();
                        }
                    }
                    if (elect_one()) mma_commit(empty_s + s * 8);
                    __syncwarp();
                    a_at += kStripABytes >> 4;
                    if (++s == n_stages) { s = 0; ph ^= 1; }
                }
                if (++nt == a.tiles_n) { nt = 0; ac.next(n_bufs); }
            }
        } else {
            // ------------------------------------------------------------ output stores, channel constants
            // Half a staged tile is two boxes of 32 columns x 128 rows; the copy engine clips them at the edges of y.  A phase of
            // sfree says that the engine has read the half before it and that the constants are in place.
            float* wsb = reinterpret_cast<float*>(smem_raw + (wsb_s - sm_s) + (uint32_t)h * kStripConsts);
            auto fetch = [&](int nt) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int64_t col = (int64_t)nt * kBN + h * kStripN + 32 * i + lane;
                    wsb[32 * i + lane] = col < a.O ? __fmul_rn(__ldg(a.wscale + col), a.out_scale) : 0.f;
                    wsb[kStripN + 32 * i + lane] = (a.bias && col < a.O) ? __ldg(a.bias + col) : 0.f;
                }
                __syncwarp();
            };
            uint32_t sph = 0;
            int mt = mt0, nt = nt0;
            fetch(nt);
            mbar_arrive_lane0(&g->sfree[h], lane);
            for (int tile = t0; tile < t1; ++tile) {
                wait_hot(smem_u32(&g->sfull[h]), sph, c, a.status, 8u);
                if (c->abort_flag) break;
                sph ^= 1u;
                if (lane == 0) {
                    const int64_t n0 = (int64_t)nt * kBN + h * kStripN;
#pragma unroll
                    for (int cb = 0; cb < 2; ++cb)
                        if (n0 + 32 * cb < a.O)
                            tma_store_2d(&ymap, stage_s + (uint32_t)(2 * h + cb) * kBox, (int32_t)n0 + 32 * cb, mt * kBM);
                    bulk_commit_group();
                }
                if (++nt == a.tiles_n) { nt = 0; ++mt; }
                if (tile + 1 < t1) fetch(nt);
                if (lane == 0) bulk_wait_group_read0();
                __syncwarp();
                mbar_arrive_lane0(&g->sfree[h], lane);
            }
            if (lane == 0) bulk_wait_group0();   // no store may still be reading this CTA's shared memory at exit
        }
    } else if (warp < kStripCtlWarps + kStripExpWarps) {
        setmaxnreg_dec<kRegsStripExp>();
        // ------------------------------------------------------------ operands from the packed codes
        // A thread's K-step is its lane index modulo four, so that a warp reads 64 bytes of each of eight rows; the next stage's
        // codes of B are under way while this one's are written.
        const int h = (warp - kStripCtlWarps) >> 2, r = (t & 127) >> 2, ks = t & 3;
        const uint32_t full_s = smem_u32(&g->full[h][0]), empty_s = smem_u32(&g->empty[h][0]);
        const uint4* wrow = reinterpret_cast<const uint4*>(a.wcodes + (int64_t)r * a.row_bytes) + ks;
        const int64_t pitch = 2 * (int64_t)a.row_bytes;      // 32 rows, in units of 16 bytes
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        // row r + 32 j is 1024 j bytes on
        const uint32_t at = (uint32_t)((r >> 3) * 256 + (r & 7) * 16);
        const uint32_t at_a = a_s + (uint32_t)ks * kStripABlk + at;
        const uint32_t at_b = b_s + (uint32_t)h * n_stages * kStripBBytes + (uint32_t)ks * kStripBBlk + at;
        int i = 0, tile = t0, mt = mt0, nt = nt0;
        AChunks ac;
        uint32_t s = 0, ph = 1;
        uint4 pb[2];
        auto load_b = [&](int j) {
            const int64_t o = (int64_t)nt * kBN + h * kStripN + r + 32 * j;
            pb[j] = tile < t1 && i * kChunk + ks < n_steps && o < a.O ? __ldg(wrow + (4 * (int64_t)nt + 2 * h + j) * pitch + i * kChunk) : zero;
        };
        load_b(0);
        load_b(1);
        while (tile < t1 && !c->abort_flag) {
            if ((nt == 0 || tile == t0) && (i & 1) == h) {   // a new row block: every other chunk of it
                const int64_t m = (int64_t)mt * kBM + r;
                const uint4* sa = reinterpret_cast<const uint4*>(a.xcodes + m * a.row_bytes) + i * kChunk + ks;
                const float* sx = a.xscale + m * a.Kg + i * kChunk + ks;
                const uint32_t slot = ac.buf * (uint32_t)chunks + (uint32_t)i, dst = slot * kStripABytes;
                uint4 pa[kChunk];
                float d[kChunk];
#pragma unroll
                for (int j = 0; j < kChunk; ++j) {
                    const bool on = i * kChunk + ks < n_steps && m + 32 * j < a.M;
                    pa[j] = on ? __ldg(sa + j * pitch) : zero;
                    d[j] = on ? __ldg(sx + (int64_t)(32 * j) * a.Kg) : 0.0f;
                }
                wait_hot(aempty_s + slot * 8, ac.use ^ 1u, c, a.status, 5u);
#pragma unroll
                for (int j = 0; j < kChunk; ++j) {
                    put_acts(at_a + dst + j * 1024, pa[j]);
                    sts32(a_s + dst + kStripSteps + (uint32_t)ks * kScaleBlock + (uint32_t)(r + 32 * j) * 4, __float_as_uint(d[j]));
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // written through the generic proxy, read by the tensor core
                __syncwarp();
                mbar_arrive_lane0_s(afull_s + slot * 8, lane);
            }
            wait_hot(empty_s + s * 8, ph, c, a.status, 5u);
            if (++i == chunks) {
                i = 0;
                ++tile;
                if (++nt == a.tiles_n) { nt = 0; ++mt; ac.next(n_bufs); }
            }
            const uint32_t dst = at_b + s * kStripBBytes;
            put_weights(dst, pb[0]);
            load_b(0);
            put_weights(dst + 1024, pb[1]);
            load_b(1);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            mbar_arrive_lane0_s(full_s + s * 8, lane);
            if (++s == n_stages) { s = 0; ph ^= 1; }
        }
    } else {
        setmaxnreg_inc<kRegsStripPromo>();
        // ------------------------------------------------------------ promotion + epilogue
        const int quarter = warp & 3;                 // TMEM lanes 32 * quarter .. + 31
        const int h = (warp - kStripCtlWarps - kStripExpWarps) >> 2;
        const int row = quarter * 32 + lane;
        uint64_t yacc[kStripN / 2];                   // 64 sums, packed in pairs
        uint32_t va[32], vb[32];                      // landing buffers: columns 0-31 and 32-63 of a slot
#pragma unroll
        for (int q = 0; q < 32; ++q) { va[q] = 0u; vb[q] = 0u; yacc[q] = 0ull; }
        uint32_t tfull_s = smem_u32(&g->tfull[h][0]), tempty_s = smem_u32(&g->tempty[h][0]);
        uint32_t tmem_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)h * (kChunk * kStripN);
        const uint32_t my_row = stage_s + (uint32_t)(2 * h) * kBox + (uint32_t)row * (Y16 ? 64u : 128u);
        const uint32_t swz = Y16 ? ((uint32_t)lane >> 1) & 3u : (uint32_t)lane & 7u;
        const uint32_t wsb_h = wsb_s + (uint32_t)h * kStripConsts;
        // opaque to the compiler: kept in registers instead of being recomputed from the thread index at every use
        asm volatile("" : "+r"(tfull_s), "+r"(tempty_s), "+r"(tmem_row));
        uint32_t par = 0u, sf_par = 0u;               // bit i: parity to wait for on tfull[i]; on sfree
        uint32_t dnext = 0u;                          // the step of the group whose load is in flight
        const uint32_t step0 = a_s + kStripSteps + (uint32_t)row * 4;
        uint32_t scale_q = step0;                     // steps of the chunk

        auto fold = [&](uint64_t* y, const uint32_t* v, uint64_t d2) {
#pragma unroll
            for (int q = 0; q < 16; ++q) fma2(y[q], pack2(v[2 * q], v[2 * q + 1]), d2);
        };
        // One group (slot U) whose first half is on its way into va: start the second half, fold the first in, hand the slot back
        // once the second has landed, start the next group's first half, fold the second in.  LAST: the group is the chunk's
        // last, the next one is slot 0 of the next chunk, if there is one (`more`).  A barrier test answers about a hundred
        // clocks after it is issued and a shared-memory load after about thirty, so both are issued well before they are needed.
        auto group = [&](auto u_tag, auto last_tag, bool more, uint32_t next_step, uint32_t a_wait, uint32_t a_par, uint32_t a_done) {
            constexpr uint32_t U = decltype(u_tag)::value;
            constexpr bool LAST = decltype(last_tag)::value != 0;
            constexpr uint32_t N = LAST ? 0 : U + 1;
            const bool on = !LAST || more;
            // U == N: its next phase, otherwise the one that is still to come
            const uint32_t np = ((par >> N) & 1u) ^ (LAST ? 1u : 0u);
            const bool rn = on ? mbar_test_s(tfull_s + N * 8, np) : true;
            const uint64_t d2 = pack2(dnext, dnext);
            tmem_ld_wait_on(va);
            tmem_ld32(tmem_row + U * kStripN + 32, vb);
            fold(yacc, va, d2);
            if (LAST && a_wait) wait_hot(a_wait, a_par, c, a.status, 7u);   // the next chunk's steps have only just been written
            if (on) dnext = lds32(next_step);
            tmem_ld_wait_on(vb);
            tc_fence_before();                            // the slot is drained
            __syncwarp();
            mbar_arrive_lane0_s(tempty_s + U * 8, lane);
            if (LAST && a_done) mbar_arrive_lane0_s(a_done, lane);          // and so is the chunk of A
            if (on) {
                if (!rn) wait_cold(tfull_s + N * 8, np, c, a.status, 2u);
                tc_fence_after();
                tmem_ld32(tmem_row + N * kStripN, va);
            }
            fold(yacc + 16, vb, d2);
        };
        const std::integral_constant<int, 0> i0{};
        const std::integral_constant<int, 1> i1{};
        const std::integral_constant<int, 2> i2{};
        const std::integral_constant<int, 3> i3{};
        int tile = t0, nt = nt0;
        AChunks ac;
        wait_hot(afull_s, 0u, c, a.status, 7u);
        dnext = lds32(scale_q);
        wait_hot(tfull_s, 0u, c, a.status, 2u);
        tc_fence_after();
        tmem_ld32(tmem_row, va);
#pragma unroll 1
        while (!c->abort_flag) {
            // one tile, its first group's load in flight
            const bool more = tile + 1 < t1, row_end = nt + 1 == a.tiles_n || !more;   // the row block's last tile in this block
            const uint32_t slot = ac.buf * (uint32_t)chunks;
            uint32_t a_done = row_end ? aempty_s + slot * 8 : 0u;
            uint32_t a_wait = nt == 0 || tile == t0 ? afull_s + slot * 8 : 0u;         // a new row block's chunks
#pragma unroll 1
            for (int ci = 1; ci < chunks; ++ci) {                 // the chunks before the last one
                if (a_wait) a_wait += 8;
                group(i0, i0, true, scale_q + kScaleBlock, 0u, 0u, 0u);
                group(i1, i0, true, scale_q + 2 * kScaleBlock, 0u, 0u, 0u);
                group(i2, i0, true, scale_q + 3 * kScaleBlock, 0u, 0u, 0u);
                scale_q += kStripABytes;
                group(i3, i1, true, scale_q, a_wait, ac.use, a_done);
                par ^= 15u;
                if (a_done) a_done += 8;
            }
            const int cnt = n_steps - (chunks - 1) * kChunk;
            const bool fresh = nt + 1 == a.tiles_n;
            if (++nt == a.tiles_n) { nt = 0; ac.next(n_bufs); }
            const uint32_t slot_n = ac.buf * (uint32_t)chunks, scale_n = step0 + slot_n * kStripABytes;
            a_wait = fresh && more ? afull_s + slot_n * 8 : 0u;
            if (cnt == 1) {
                group(i0, i1, more, scale_n, a_wait, ac.use, a_done);
            } else {
                group(i0, i0, true, scale_q + kScaleBlock, 0u, 0u, 0u);
                if (cnt == 2) {
                    group(i1, i1, more, scale_n, a_wait, ac.use, a_done);
                } else {
                    group(i1, i0, true, scale_q + 2 * kScaleBlock, 0u, 0u, 0u);
                    if (cnt == 3) {
                        group(i2, i1, more, scale_n, a_wait, ac.use, a_done);
                    } else {
                        group(i2, i0, true, scale_q + 3 * kScaleBlock, 0u, 0u, 0u);
                        group(i3, i1, more, scale_n, a_wait, ac.use, a_done);
                    }
                }
            }
            par ^= (1u << cnt) - 1u;
            scale_q = scale_n;
            // y = (s_o * 2^18) * sum + bias, parked as the source of the bulk tensor stores: box cb = columns 32 cb .. + 31 of this half
            // of all 128 rows, rows of 128 bytes whose 16-byte chunk j sits at j ^ (row & 7) (fp32), or rows of 64 bytes with
            // chunk j at j ^ ((row >> 1) & 3) (16-bit types).
            wait_hot(smem_u32(&g->sfree[h]), sf_par, c, a.status, 9u);
            sf_par ^= 1u;
            uint64_t cs[2][4], cb[2][4];                  // eight columns' constants, read eight columns ahead
            auto fetch = [&](int i) {
                const uint32_t from = wsb_h + 32 * i;
                lds128(from, cs[i & 1][0], cs[i & 1][1]);
                lds128(from + 16, cs[i & 1][2], cs[i & 1][3]);
                lds128(from + kStripN * 4, cb[i & 1][0], cb[i & 1][1]);
                lds128(from + kStripN * 4 + 16, cb[i & 1][2], cb[i & 1][3]);
            };
            fetch(0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {                 // eight columns
                if (i < 7) fetch(i + 1);
                float f[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    fma2(cb[i & 1][q], yacc[4 * i + q], cs[i & 1][q]);
                    unpack2(cb[i & 1][q], f[2 * q], f[2 * q + 1]);
                    yacc[4 * i + q] = 0ull;
                }
                const uint32_t to = my_row + (uint32_t)(i >> 2) * kBox, w = (uint32_t)(i & 3);
                if (!Y16) {
                    sts128(to + (((2 * w) ^ swz) << 4), __float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
                    sts128(to + (((2 * w + 1) ^ swz) << 4), __float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]), __float_as_uint(f[7]));
                } else {
                    sts128(to + ((w ^ swz) << 4), pack16(f[0], f[1], a.y_f16), pack16(f[2], f[3], a.y_f16), pack16(f[4], f[5], a.y_f16), pack16(f[6], f[7], a.y_f16));
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the engine's reads
            __syncwarp();
            mbar_arrive_lane0(&g->sfull[h], lane);
            ++tile;
            if (!more) break;
        }
        tmem_ld_wait();            // nothing may still be landing when TMEM is released
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        // all MMAs this CTA issued have completed unless a wait gave up; in that case give the
        // tensor core a moment before the columns are handed back
        if (c->abort_flag) __nanosleep(1000000);
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * kChunk * kStripN) : "memory");
    }
}

struct StripPlan { int32_t bufs, stages; uint32_t smem; };
// Six chunks of A where they fit (several short row blocks, so that the next one is ready in time) and two or three stages of B
// for each half.
bool strip_plan(bool y16, int32_t n_steps, StripPlan& p) {
    const int64_t chunks = (n_steps + kChunk - 1) / kChunk;
    if (chunks > kStripMaxChunks) return false;
    p.bufs = (int32_t)(chunks < 6 ? 6 / chunks : 1);
    const int64_t fixed = kStripCtrl + kStripN * 32 + 1024 + 4 * (y16 ? kStripBox16 : kStripBoxF32) + 2 * kStripConsts + p.bufs * chunks * kStripABytes;
    const int64_t stages = (kSmemLimit - fixed) / (2 * kStripBBytes);
    if (stages < 2) return false;
    p.stages = (int32_t)(stages < kStripMaxStages ? stages : kStripMaxStages);
    p.smem = (uint32_t)(fixed + p.stages * 2 * kStripBBytes);
    return true;
}

}  // namespace

bool linear_strip_fits(bool y16, int32_t n_steps) {
    StripPlan p;
    return strip_plan(y16, n_steps, p);
}

tdq_status launch_linear_strip(LinArgs a, const CUtensorMap& ymap, int n_sm, int dev, bool ybf, cudaStream_t stream) {
    constexpr int kInst = 2;
    void (*const kernels[kInst])(LinArgs, CUtensorMap) = {w4a4_strip_kernel<false>, w4a4_strip_kernel<true>};
    StripPlan p;
    if (!a.tma_ok || a.steps_per_grp != 1 || !strip_plan(ybf, a.n_steps, p)) return TDQ_ERR_UNSUPPORTED;
    a.n_ibuf = p.bufs;
    a.n_stages = p.stages;
    a.out_scale = 262144.0f;     // operands q 2^-9 and q 2^-9
    static std::atomic<uint64_t> smem_done[kInst];
    if (allow_smem(kernels[ybf ? 1 : 0], kSmemLimit, smem_done[ybf ? 1 : 0], dev) != cudaSuccess) return TDQ_ERR_CUDA;
    const int64_t tiles = (int64_t)a.tiles_m * a.tiles_n;
    if (launch_pdl(kernels[ybf ? 1 : 0], dim3((unsigned)(tiles < n_sm ? tiles : n_sm)), dim3(kStripThreads), p.smem, stream, a, ymap) != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

}  // namespace tdq
