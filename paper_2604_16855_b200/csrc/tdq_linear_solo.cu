// The W4A4 linear layer (Algorithm S1 step 10 with Eq. 9 and Eq. 4 substituted) where there are no more 128 x 64 tiles than
// SMs, from the packed codes in one launch:
//
//   acc[m,o,k] = sum_{i in group k} q_x[m,i] q_w[o,i]      tcgen05.mma, exact
//   y[m,o]     = s_o * sum_k Delta[m,k] * acc[m,o,k] + b_o  fp32 in registers ("promotion")
//
// bit for bit what the other kernels of the layer compute.
//
// What bounds it.  A block has an SM to itself and one tile to do, so everything is latency: the launch of an expansion kernel
// in front (about 3 us), the hand-over of a TMEM slot (about 900 clocks, with four slots of 128 columns 225 a group), the
// epilogue.  So: the operands come from the packed codes in the kernel itself, TMEM holds eight slots of 64 columns, and eight
// promotion warps have 32 columns each.  What is left per K-step is shared memory: at g = 32 about 220 clocks (the operand
// writes, two instructions' reads, the codes through L1), at wider groups about 130.
//
//   warps 0-3    MMA issue; group k goes to TMEM slot k & 7
//   warps 4-15   operands: three teams of four warps take the ring's stages (four K-steps) in turn
//   warps 16-23  promotion and epilogue: 32 rows x 32 columns each, two landing buffers
//
// Operand bytes.  The channels of a group may be summed in any order, so the two nibbles of a byte stay apart (even channels in
// one half of a K-step, odd ones in the other) in both operands.  Groups of one K-step go as E4M3 into fp32 accumulators, which
// need no conversion before their multiply-add.  The E4M3 byte n is the number n 2^-9 for n = 0..15, so an activation
// code takes one bit operation as q + 8, and a second instruction with a constant block of -8 takes 8 sum q_w off again
// (exact: everything is below 2^12 in units of 2^-18); the sign-and-magnitude bytes that the weights get cost five times
// as much.  Wider groups go as int8: 16 q is a mask or a shift away from the codes, and a group's conversion to float is
// spread over several K-steps.  The promotion works in the units of the kernels that take these groups elsewhere (E4M3's 2^-18 up
// to 128 codes a group), so a sum is finite here exactly where it is finite there.
//
// Measured (B200, from a graph), us, against the expansion and the kernels behind it: 1152 x 512 -> 512 fp32 at g = 32 8.1 -> 7.6,
// at g = 64 8.0 -> 5.9; 576 x 320 -> 960 at g = 32 6.8 -> 6.0; 200 x 768 -> 768 bf16 at g = 768 7.8 -> 5.7; 128 x 1312 -> 56 fp16 at
// g = 1312 12.3 -> 7.3; 97 x 256 -> 2047 fp32 (y off the 16-byte grid) 8.1 -> 5.9.  Both sides at more sizes are beside the rule in
// tdq_linear.cu.  Not kept: a row of A per lane (every load then touches 32 rows: 144 x 2048 -> 512 22.5 us, now 14.8), two teams of
// operand warps (15.8), eight MMA warps (14.5, but 576 x 320 -> 960 6.0 -> 6.6), loads that bypass L1 (no difference).
#include "tdq_tc.cuh"

namespace tdq {
namespace {

constexpr int kSoloN = 64, kSoloSlots = 8;                  // columns per tile = one TMEM slot; all of TMEM is this block's
constexpr int kSoloMmaWarps = 4, kSoloTeams = 3, kSoloExpWarps = 4 * kSoloTeams, kSoloPromoWarps = 8;
constexpr int kSoloThreads = (kSoloMmaWarps + kSoloExpWarps + kSoloPromoWarps) * 32;   // 768
constexpr int kRegsSoloMma = 32, kRegsSoloExp = 64, kRegsSoloPromo = 128;              // 128 * 32 + 384 * 64 + 256 * 128 = 768 * 80
constexpr int kSoloStages = 7;
// K-steps inside a stage are 32 bytes off a multiple of 128 bytes apart, so that the four lanes that write a row's four K-steps
// meet different banks
constexpr uint32_t kSoloABlk = kBlock + 32, kSoloBBlk = kSoloN * 32 + 32;
constexpr uint32_t kSoloB = kChunk * kSoloABlk, kSoloSteps = kSoloB + kChunk * kSoloBBlk;   // offsets inside a stage: B, the steps Delta
constexpr uint32_t kSoloStageBytes = kSoloSteps + kChunk * kScaleBlock;
constexpr uint32_t kSoloCtrl = 1024;
constexpr uint32_t kSoloBoxF32 = 128 * 128, kSoloBox16 = 128 * 64;   // one 32-column box of 128 rows in the staging area
constexpr uint32_t kSoloSmem = kSoloCtrl + kBlock + kSoloStages * kSoloStageBytes + 1024 + 2 * kSoloBoxF32 + 2 * kSoloN * 4;
static_assert(kSoloSmem <= kSmemLimit, "shared memory");
constexpr uint32_t kIdescSoloShape = ((uint32_t)(kSoloN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
constexpr uint32_t kIdescSoloF8 = (1u << 4) | kIdescSoloShape;

struct SoloCtrl {
    uint64_t full[kSoloStages], empty[kSoloStages];
    uint64_t tfull[kSoloSlots], tempty[kSoloSlots];
};
static_assert(sizeof(Ctrl) + sizeof(SoloCtrl) <= kSoloCtrl, "control block outgrew its reservation");

// `n` (one to four) int8 instructions on consecutive K-steps of the same accumulator; the descriptors are built once and move by an add
__device__ __forceinline__ void mma_i8_steps(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate_first, uint32_t n) {
    asm volatile(
        "{\n\t.reg .pred p, q, t;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\tmov.b64 da, %1;\n\tmov.b64 db, %2;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %3, p;\n\t"
        "add.s64 da, da, %6;\n\tadd.s64 db, db, %7;\n\tsetp.gt.u32 q, %5, 1;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %3, t;\n\t"
        "add.s64 da, da, %6;\n\tadd.s64 db, db, %7;\n\tsetp.gt.u32 q, %5, 2;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %3, t;\n\t"
        "add.s64 da, da, %6;\n\tadd.s64 db, db, %7;\n\tsetp.gt.u32 q, %5, 3;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %3, t;\n\t}"
        ::"r"(d), "l"(adesc), "l"(bdesc), "r"((2u << 4) | (1u << 7) | (1u << 10) | kIdescSoloShape), "r"(accumulate_first), "r"(n),
          "n"(kSoloABlk >> 4), "n"(kSoloBBlk >> 4)
        : "memory");
}

// 32 packed codes of an activation row -> operand bytes (even channels, then odd ones): 16 q for int8; for E4M3 q + 8, as the
// bytes 0..15 are the numbers 0..15 in units of 2^-9
template <bool I8>
__device__ __forceinline__ void act_bytes(const uint4& p, uint4& ev, uint4& od) {
    const uint32_t w[4] = {p.x, p.y, p.z, p.w};
    uint32_t e[4], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        e[i] = I8 ? (w[i] << 4) & 0xF0F0F0F0u : (w[i] & 0x0F0F0F0Fu) ^ 0x08080808u;
        o[i] = I8 ? w[i] & 0xF0F0F0F0u : ((w[i] >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
    }
    ev = make_uint4(e[0], e[1], e[2], e[3]);
    od = make_uint4(o[0], o[1], o[2], o[3]);
}
// 32 packed weight codes -> operand bytes in the same order: sign and magnitude (E4M3, units of 2^-9) or 16 q (int8)
template <bool I8>
__device__ __forceinline__ void weight_bytes(const uint4& p, uint4& ev, uint4& od) {
    const uint32_t w[4] = {p.x, p.y, p.z, p.w};
    uint32_t e[4], o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        e[i] = (w[i] << 4) & 0xF0F0F0F0u;
        o[i] = w[i] & 0xF0F0F0F0u;
        if (!I8) {
            e[i] = to_sign_magnitude(e[i]);
            o[i] = to_sign_magnitude(o[i]);
        }
    }
    ev = make_uint4(e[0], e[1], e[2], e[3]);
    od = make_uint4(o[0], o[1], o[2], o[3]);
}

// K-steps per group: one (E4M3), up to four or more (int8, a.steps_per_grp of them; the units of the sums differ, see below)
enum SoloKind { kSoloOne, kSoloFew, kSoloMany };
template <bool YBF16, SoloKind KIND>
__global__ void __launch_bounds__(kSoloThreads, 1) w4a4_solo_kernel(const LinArgs a, const __grid_constant__ CUtensorMap ymap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];
    constexpr bool SPG1 = KIND == kSoloOne, I8 = !SPG1;
    constexpr uint32_t kBox = YBF16 ? kSoloBox16 : kSoloBoxF32;
    Ctrl* c = reinterpret_cast<Ctrl*>(smem_raw);             // its abort flag and TMEM address; the barriers are g's
    SoloCtrl* g = reinterpret_cast<SoloCtrl*>(smem_raw + sizeof(Ctrl));
    const uint32_t sm_s = smem_u32(smem_raw);
    const uint32_t minus_s = sm_s + kSoloCtrl;               // an operand block of -8
    const uint32_t ring_s = minus_s + kBlock;
    const uint32_t stage_s = (ring_s + kSoloStages * kSoloStageBytes + 1023u) & ~1023u;   // the swizzle patterns repeat every 1024 bytes
    const uint32_t wsb_s = stage_s + 2 * kBox;               // [64] channel scales, [64] biases
    const int t = threadIdx.x, warp = uniform_warp(), lane = t & 31;

    // the MMA warps take the groups in turn where a stage holds whole groups, else the first one takes all
    const bool spread = !SPG1 && (a.steps_per_grp == 2 || a.steps_per_grp == 4);

    if (t == 0) {
        for (int i = 0; i < kSoloStages; ++i) { mbar_init(&g->full[i], 4); mbar_init(&g->empty[i], SPG1 ? kSoloPromoWarps : spread ? kSoloMmaWarps : 1); }
        for (int i = 0; i < kSoloSlots; ++i) { mbar_init(&g->tfull[i], 1); mbar_init(&g->tempty[i], kSoloPromoWarps); }
        c->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&c->tmem_base)), "r"(kSoloSlots * kSoloN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (SPG1 && t >= 128 && t < 128 + kBlock / 16) {
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
    const int mt = (int)blockIdx.x / a.tiles_n, nt = (int)blockIdx.x - mt * a.tiles_n;
    const int n_steps = a.n_steps, chunks = (n_steps + kChunk - 1) / kChunk;
    const uint32_t full_s = smem_u32(&g->full[0]), empty_s = smem_u32(&g->empty[0]);

    if (warp < kSoloMmaWarps) {
        setmaxnreg_dec<kRegsSoloMma>();
        // ------------------------------------------------------------ MMA issue: group k in slot k & 7
        // SPG1: the activations' operand bytes are q + 8, and an instruction with the block of -8 takes 8 sum q_w off again.
        const uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        const uint32_t m_lo = desc_lo(minus_s);
        uint32_t s = 0, ph = 0;
        if (SPG1) {
            // this warp takes K-step `warp` of every stage
            const uint32_t a_lo = desc_lo(ring_s) + (uint32_t)warp * (kSoloABlk >> 4);
            const uint32_t b_lo = desc_lo(ring_s + kSoloB) + (uint32_t)warp * (kSoloBBlk >> 4);
            for (int k = warp; k < n_steps && !c->abort_flag; k += kChunk) {
                const uint32_t slot = (uint32_t)k & (kSoloSlots - 1), par = (((uint32_t)k / kSoloSlots) & 1u) ^ 1u;
                const uint32_t so = s * (kSoloStageBytes >> 4);
                const bool rf = mbar_test_s(full_s + s * 8, ph);   // the two tests are in flight together
                const bool rt = mbar_test_s(tempty_s + slot * 8, par);
                if (!rf) wait_cold(full_s + s * 8, ph, c, a.status, 4u);
                if (!rt) wait_cold(tempty_s + slot * 8, par, c, a.status, 3u);
                tc_fence_after();
                if (elect_one()) {
                    mma_f8(tmem_base + slot * kSoloN, desc_of(m_lo), desc_of(b_lo + so), kIdescSoloF8);
                    mma_f8(tmem_base + slot * kSoloN, desc_of(a_lo + so), desc_of(b_lo + so), kIdescSoloF8, 1u);
                    mma_commit(tfull_s + slot * 8);
                }
                __syncwarp();
                if (++s == kSoloStages) { s = 0; ph ^= 1; }
            }
        } else if (spread) {
            // group k is this warp's if k & 3 is its index; every warp hands every stage back
            const uint32_t a_lo = desc_lo(ring_s), b_lo = desc_lo(ring_s + kSoloB);
            const int spg = a.steps_per_grp, per = kChunk / spg;
            for (int k0 = 0; k0 < a.Kg && !c->abort_flag; k0 += per) {
                // the stage's group that may be this warp's: the first, or with two per stage the one of its parity
                const int k = per == 2 ? k0 + (warp & 1) : k0;
                const bool mine = (k & 3) == warp && k < a.Kg;
                const uint32_t slot = (uint32_t)k & (kSoloSlots - 1), par = (((uint32_t)k / kSoloSlots) & 1u) ^ 1u;
                const bool rf = mbar_test_s(full_s + s * 8, ph);   // the two tests are in flight together
                const bool rt = mine ? mbar_test_s(tempty_s + slot * 8, par) : true;
                if (!rf) wait_cold(full_s + s * 8, ph, c, a.status, 4u);
                if (!rt) wait_cold(tempty_s + slot * 8, par, c, a.status, 3u);
                tc_fence_after();
                if (elect_one()) {
                    if (mine) {
                        const uint32_t so = s * (kSoloStageBytes >> 4), first = (uint32_t)((k - k0) * spg);
                        mma_i8_steps(tmem_base + slot * kSoloN, desc_of(a_lo + so + first * (kSoloABlk >> 4)), desc_of(b_lo + so + first * (kSoloBBlk >> 4)), 0u, (uint32_t)spg);
                        mma_commit(tfull_s + slot * 8);
                    }
                    mma_commit(empty_s + s * 8);
                }
                __syncwarp();
                if (++s == kSoloStages) { s = 0; ph ^= 1; }
            }
        } else if (warp == 0) {
            const uint32_t a_lo = desc_lo(ring_s), b_lo = desc_lo(ring_s + kSoloB);
            int in_stage = 0;
            for (int k = 0; k < a.Kg && !c->abort_flag; ++k) {
                const uint32_t slot = (uint32_t)k & (kSoloSlots - 1);
                const uint32_t d = tmem_base + slot * kSoloN;
                wait_hot(tempty_s + slot * 8, (((uint32_t)k / kSoloSlots) & 1u) ^ 1u, c, a.status, 3u);
                for (int i = 0; i < a.steps_per_grp;) {
                    // the K-steps of this stage that belong to the group
                    if (in_stage == 0) wait_hot(full_s + s * 8, ph, c, a.status, 4u);
                    const int n = min(kChunk - in_stage, a.steps_per_grp - i);
                    const uint32_t so = s * (kSoloStageBytes >> 4);
                    const bool stage_end = in_stage + n == kChunk, group_end = i + n == a.steps_per_grp;
                    tc_fence_after();
                    if (elect_one()) {
                        mma_i8_steps(d, desc_of(a_lo + so + (uint32_t)in_stage * (kSoloABlk >> 4)), desc_of(b_lo + so + (uint32_t)in_stage * (kSoloBBlk >> 4)),
                                     i ? 1u : 0u, (uint32_t)n);
                        if (group_end) mma_commit(tfull_s + slot * 8);
                        if (stage_end) mma_commit(empty_s + s * 8);
                    }
                    __syncwarp();
                    i += n;
                    in_stage += n;
                    if (stage_end) {
                        in_stage = 0;
                        if (++s == kSoloStages) { s = 0; ph ^= 1; }
                    }
                }
            }
        }
    } else if (warp < kSoloMmaWarps + kSoloExpWarps) {
        setmaxnreg_dec<kRegsSoloExp>();
        // ------------------------------------------------------------ operands from the packed codes
        // Three teams of four warps take the stages in turn.  A thread's K-step is its lane index modulo four, so that a warp
        // reads 64 bytes of each of eight rows; a team's next stage is loaded while the other teams write theirs.
        const int team = (warp - kSoloMmaWarps) >> 2, r = (t & 127) >> 2, ks = t & 3;
        const int64_t m0 = (int64_t)mt * kBM + r, o0 = (int64_t)nt * kSoloN + r;
        const uint4* sa = reinterpret_cast<const uint4*>(a.xcodes + m0 * a.row_bytes) + ks;
        const uint4* sb = reinterpret_cast<const uint4*>(a.wcodes + o0 * a.row_bytes) + ks;
        const float* sx = a.xscale + m0 * a.Kg + ks;
        const int64_t pitch = 2 * (int64_t)a.row_bytes;      // 32 rows, in units of 16 bytes
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        uint4 pa[kChunk], pb[2];
        float d[kChunk];
        auto load_a = [&](int n, int j) {
            const bool on = n * kChunk + ks < n_steps && m0 + 32 * j < a.M;
            pa[j] = on ? __ldg(sa + j * pitch + n * kChunk) : zero;
            if (SPG1) d[j] = on ? __ldg(sx + (int64_t)(32 * j) * a.Kg + n * kChunk) : 0.0f;
        };
        auto load_b = [&](int n, int j) { pb[j] = n * kChunk + ks < n_steps && o0 + 32 * j < a.O ? __ldg(sb + j * pitch + n * kChunk) : zero; };
        // row r + 32 j is 1024 j bytes on
        const uint32_t at = (uint32_t)((r >> 3) * 256 + (r & 7) * 16), at_a = (uint32_t)ks * kSoloABlk + at, at_b = kSoloB + (uint32_t)ks * kSoloBBlk + at;
        uint32_t s = (uint32_t)team, ph = 1;
#pragma unroll
        for (int j = 0; j < kChunk; ++j) load_a(team, j);
#pragma unroll
        for (int j = 0; j < 2; ++j) load_b(team, j);
        for (int n = team; n < chunks && !c->abort_flag; n += kSoloTeams) {
            wait_hot(empty_s + s * 8, ph, c, a.status, 5u);
            const uint32_t st = ring_s + s * kSoloStageBytes;
            uint4 ev, od;
#pragma unroll
            for (int j = 0; j < kChunk; ++j) {
                act_bytes<I8>(pa[j], ev, od);
                sts128(st + at_a + j * 1024, ev.x, ev.y, ev.z, ev.w);
                sts128(st + at_a + j * 1024 + 128, od.x, od.y, od.z, od.w);
                if (SPG1) sts32(st + kSoloSteps + (uint32_t)ks * kScaleBlock + (uint32_t)(r + 32 * j) * 4, __float_as_uint(d[j]));
                load_a(n + kSoloTeams, j);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                weight_bytes<I8>(pb[j], ev, od);
                sts128(st + at_b + j * 1024, ev.x, ev.y, ev.z, ev.w);
                sts128(st + at_b + j * 1024 + 128, od.x, od.y, od.z, od.w);
                load_b(n + kSoloTeams, j);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // written through the generic proxy, read by the tensor core
            __syncwarp();
            mbar_arrive_lane0_s(full_s + s * 8, lane);
            s += kSoloTeams;
            if (s >= kSoloStages) { s -= kSoloStages; ph ^= 1; }
        }
    } else {
        setmaxnreg_inc<kRegsSoloPromo>();
        // ------------------------------------------------------------ promotion + epilogue
        const int quarter = warp & 3;                 // TMEM lanes 32 * quarter .. + 31
        const int half = (warp - kSoloMmaWarps - kSoloExpWarps) >> 2;   // columns 32 * half .. + 31 of the tile
        const int row = quarter * 32 + lane, pt = t - (kSoloMmaWarps + kSoloExpWarps) * 32;
        float* wsb = reinterpret_cast<float*>(smem_raw + (wsb_s - sm_s));
        if (pt < kSoloN) {
            const int64_t col = (int64_t)nt * kSoloN + pt;
            wsb[pt] = col < a.O ? __fmul_rn(__ldg(a.wscale + col), a.out_scale) : 0.f;
            wsb[kSoloN + pt] = (a.bias && col < a.O) ? __ldg(a.bias + col) : 0.f;
        }
        uint64_t yacc[16];
        uint32_t va[32], vb[32];                      // landing buffers of even and of odd groups
#pragma unroll
        for (int q = 0; q < 32; ++q) { va[q] = 0u; vb[q] = 0u; }
#pragma unroll
        for (int q = 0; q < 16; ++q) yacc[q] = 0ull;
        uint32_t tfull_s = smem_u32(&g->tfull[0]), tempty_s = smem_u32(&g->tempty[0]);
        uint32_t tmem_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 32);
        const uint32_t steps_s = ring_s + kSoloSteps + (uint32_t)row * 4;
        uint32_t scale_q = steps_s, rs = 0, rph = 0;  // SPG1: the stage's steps, its index and phase
        // opaque to the compiler: kept in registers instead of being recomputed from the thread index at every use
        asm volatile("" : "+r"(tfull_s), "+r"(tempty_s), "+r"(tmem_row));
        const int64_t m_row = (int64_t)mt * kBM + row;
        const float* gx = a.xscale + (m_row < a.M ? m_row : 0) * a.Kg;   // otherwise the steps come from memory, a group ahead
        // int8 sums are 256 times the group's.  Up to 128 codes a group the other kernels add sums in units of 2^-18 (E4M3), beyond
        // that 256 times the sums; the same units here, or a product near the ends of binary32's range would be rounded or
        // overflow in one kernel and not in the other.  (Exact: a power of two, and the sums are whole numbers below 2^22.)  The
        // multiplication is up to 4 % of such a layer (1152 x 1024 -> 512 at g = 128 6.25 -> 6.51 us).  Dearer: the step scaled instead
        // where that is exact, and a vote on it, 12 %; a scan of the warp's steps in front and a second loop 6 %; a conversion by way
        // of a float with the sum in its last bits 13 %.
        constexpr uint32_t kUnit = 0x32800000u;       // 2^-26
        const uint64_t unit2 = pack2(kUnit, kUnit);
        uint32_t par = 0u;                            // parity of the slots' completions in this turn of eight groups
        uint32_t dnext = 0u;
        bool ready = true;                            // the barrier of the group after the one whose load is in flight
        bool stage_ready = true;                      // SPG1: the next stage's barrier, asked a group before it is needed

        // One group (slot U) whose load is in flight: when it has landed start the next group's, hand the slot back, fold.  A
        // barrier test answers about a hundred clocks after it is issued, so it is issued a group ahead.  left: groups from this one on.
        auto group = [&](auto u_tag, int k, int left) {
            constexpr uint32_t U = decltype(u_tag)::value, N = (U + 1) & (kSoloSlots - 1), F = (U + 2) & (kSoloSlots - 1);
            const bool more = left > 1;
            uint32_t (&v)[32] = U & 1 ? vb : va;
            uint32_t (&w)[32] = U & 1 ? va : vb;
            const uint32_t npar = N ? par : par ^ 1u;
            const uint64_t d2 = pack2(dnext, dnext);
            if (!SPG1 && more) dnext = __float_as_uint(__ldg(gx + k + 1));
            tmem_ld_wait_on(v);
            if (more) {
                if (!ready) wait_cold(tfull_s + N * 8, npar, c, a.status, 2u);
                tc_fence_after();
                tmem_ld32(tmem_row + N * kSoloN, w);
                ready = left > 2 ? mbar_test_s(tfull_s + F * 8, F > U ? par : par ^ 1u) : true;
            }
            tc_fence_before();                            // this slot is drained
            __syncwarp();
            mbar_arrive_lane0_s(tempty_s + U * 8, lane);
            if (SPG1) {
                if ((U & 3) == 3) {
                    // all groups of the stage have been seen complete and their steps read: it may be filled again
                    mbar_arrive_lane0_s(empty_s + rs * 8, lane);
                    if (++rs == kSoloStages) { rs = 0; rph ^= 1; }
                    scale_q = steps_s + rs * kSoloStageBytes;
                    if (more && !stage_ready) wait_cold(full_s + rs * 8, rph, c, a.status, 7u);
                }
                dnext = lds32(scale_q + ((U + 1) & 3) * kScaleBlock);   // past the tile's last group: not used
                if ((U & 3) == 2) {
                    const bool wrap = rs + 1 == kSoloStages;
                    stage_ready = mbar_test_s(wrap ? full_s : full_s + (rs + 1) * 8, rph ^ (wrap ? 1u : 0u));
                }
            }
            if (I8) {
#pragma unroll
                for (int q = 0; q < 32; ++q) v[q] = __float_as_uint((float)(int32_t)v[q]);
            }
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                uint64_t f = pack2(v[2 * q], v[2 * q + 1]);
                if (KIND == kSoloFew) asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(f) : "l"(unit2));
                fma2(yacc[q], f, d2);
            }
        };
        const std::integral_constant<int, 0> u0{};
        const std::integral_constant<int, 1> u1{};
        const std::integral_constant<int, 2> u2{};
        const std::integral_constant<int, 3> u3{};
        const std::integral_constant<int, 4> u4{};
        const std::integral_constant<int, 5> u5{};
        const std::integral_constant<int, 6> u6{};
        const std::integral_constant<int, 7> u7{};
        const int Kg = a.Kg;
        if (SPG1) {
            wait_hot(full_s, 0u, c, a.status, 7u);
            dnext = lds32(scale_q);
        } else {
            dnext = __float_as_uint(__ldg(gx));
        }
        wait_hot(tfull_s, 0u, c, a.status, 2u);
        tc_fence_after();
        tmem_ld32(tmem_row, va);
        if (Kg > 1) ready = mbar_test_s(tfull_s + 8, 0u);
        int k = 0;
#pragma unroll 1
        for (; k + 8 < Kg && !c->abort_flag; k += 8) {       // eight groups, and more behind them
            group(u0, k, 8);
            group(u1, k + 1, 8);
            group(u2, k + 2, 8);
            group(u3, k + 3, 8);
            group(u4, k + 4, 8);
            group(u5, k + 5, 8);
            group(u6, k + 6, 8);
            group(u7, k + 7, 8);
            par ^= 1u;
        }
        const int rem = Kg - k;                              // the last one to eight groups
        group(u0, k, rem);
        if (rem > 1) group(u1, k + 1, rem - 1);
        if (rem > 2) group(u2, k + 2, rem - 2);
        if (rem > 3) group(u3, k + 3, rem - 3);
        if (rem > 4) group(u4, k + 4, rem - 4);
        if (rem > 5) group(u5, k + 5, rem - 5);
        if (rem > 6) group(u6, k + 6, rem - 6);
        if (rem > 7) group(u7, k + 7, 1);

        // y = (s_o * 2^n) * sum + bias, parked as the source of the bulk tensor stores: box `half` = 32 columns of all 128 rows, rows of
        // 128 bytes whose 16-byte chunk j sits at j ^ (row & 7) (fp32), or rows of 64 bytes with chunk j at j ^ ((row >> 1) & 3).
        asm volatile("bar.sync 1, 256;" ::: "memory");       // the channel constants are there
        const float4* wsb4 = reinterpret_cast<const float4*>(wsb) + 8 * half;
        const uint32_t row_s = stage_s + (uint32_t)half * kBox + (uint32_t)row * (YBF16 ? 64u : 128u);
#pragma unroll
        for (int j = 0; j < 4; ++j) {                        // eight columns
            const float4 ca = wsb4[2 * j], cb = wsb4[2 * j + 1], ba = wsb4[kSoloN / 4 + 2 * j], bb = wsb4[kSoloN / 4 + 2 * j + 1];
            float o[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) unpack2(yacc[4 * j + q], o[2 * q], o[2 * q + 1]);
            o[0] = __fmaf_rn(ca.x, o[0], ba.x); o[1] = __fmaf_rn(ca.y, o[1], ba.y);
            o[2] = __fmaf_rn(ca.z, o[2], ba.z); o[3] = __fmaf_rn(ca.w, o[3], ba.w);
            o[4] = __fmaf_rn(cb.x, o[4], bb.x); o[5] = __fmaf_rn(cb.y, o[5], bb.y);
            o[6] = __fmaf_rn(cb.z, o[6], bb.z); o[7] = __fmaf_rn(cb.w, o[7], bb.w);
            if (!YBF16) {
                const uint32_t x7 = (uint32_t)lane & 7u;
                sts128(row_s + (((uint32_t)(2 * j) ^ x7) << 4), __float_as_uint(o[0]), __float_as_uint(o[1]), __float_as_uint(o[2]), __float_as_uint(o[3]));
                sts128(row_s + (((uint32_t)(2 * j + 1) ^ x7) << 4), __float_as_uint(o[4]), __float_as_uint(o[5]), __float_as_uint(o[6]), __float_as_uint(o[7]));
            } else {
                sts128(row_s + (((uint32_t)j ^ (((uint32_t)lane >> 1) & 3u)) << 4), pack16(o[0], o[1], a.y_f16), pack16(o[2], o[3], a.y_f16),
                       pack16(o[4], o[5], a.y_f16), pack16(o[6], o[7], a.y_f16));
            }
        }
        const int64_t n0 = (int64_t)nt * kSoloN + 32 * half;
        if (a.tma_ok) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes before the engine's reads
            asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory");  // the box's four warps
            if ((pt & 127) == 0) {
                if (n0 < a.O) tma_store_2d(&ymap, stage_s + (uint32_t)half * kBox, (int32_t)n0, mt * kBM);
                bulk_commit_group();
                bulk_wait_group0();                          // no store may still be reading this CTA's shared memory at exit
            }
        } else {
            // y off the 16-byte grid: the warp writes its own 32 rows, a row's columns side by side, eight rows at a time
            __syncwarp();
            const int64_t r0 = (int64_t)mt * kBM + quarter * 32;
            const int rows = (int)min((int64_t)32, a.M - r0), cols = (int)min((int64_t)32, a.O - n0);
            const uint8_t* tile_sm = smem_raw + (stage_s - sm_s) + (uint32_t)half * kBox + (uint32_t)(quarter * 32) * (YBF16 ? 64u : 128u);
            constexpr int kBatch = 8;
#pragma unroll 1
            for (int b0 = 0; b0 < rows; b0 += kBatch) {
                uint32_t v[kBatch];
#pragma unroll
                for (int i = 0; i < kBatch; ++i) {
                    const uint32_t r = (uint32_t)(b0 + i);
                    if (!YBF16) v[i] = *reinterpret_cast<const uint32_t*>(tile_sm + r * 128u + ((((uint32_t)lane >> 2) ^ (r & 7u)) << 4) + ((uint32_t)lane & 3u) * 4u);
                    else v[i] = *reinterpret_cast<const uint16_t*>(tile_sm + r * 64u + ((((uint32_t)lane >> 3) ^ ((r >> 1) & 3u)) << 4) + ((uint32_t)lane & 7u) * 2u);
                }
#pragma unroll
                for (int i = 0; i < kBatch; ++i) {
                    if (b0 + i >= rows || lane >= cols) break;
                    const int64_t to = (r0 + b0 + i) * a.y_stride + n0 + lane;
                    if (!YBF16) reinterpret_cast<uint32_t*>(a.y)[to] = v[i];
                    else reinterpret_cast<uint16_t*>(a.y)[to] = (uint16_t)v[i];
                }
            }
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
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kSoloSlots * kSoloN) : "memory");
    }
}

}  // namespace

// a.tiles_n is in units of 64 columns here.
tdq_status launch_linear_solo(LinArgs a, const CUtensorMap& ymap, int dev, bool ybf, cudaStream_t stream) {
    constexpr int kInst = 6;
    void (*const kernels[kInst])(LinArgs, CUtensorMap) = {
        w4a4_solo_kernel<false, kSoloOne>, w4a4_solo_kernel<true, kSoloOne>, w4a4_solo_kernel<false, kSoloFew>,
        w4a4_solo_kernel<true, kSoloFew>, w4a4_solo_kernel<false, kSoloMany>, w4a4_solo_kernel<true, kSoloMany>};
    const int inst = (ybf ? 1 : 0) + 2 * (a.steps_per_grp == 1 ? kSoloOne : a.steps_per_grp <= 4 ? kSoloFew : kSoloMany);
    a.out_scale = a.steps_per_grp > 4 ? 0.00390625f : 262144.0f;     // the units of the sums that the promotion adds: 2^8 or 2^-18
    static std::atomic<uint64_t> smem_done[kInst];
    if (allow_smem(kernels[inst], (int)kSoloSmem, smem_done[inst], dev) != cudaSuccess) return TDQ_ERR_CUDA;
    if (launch_pdl(kernels[inst], dim3((unsigned)(a.tiles_m * a.tiles_n)), dim3(kSoloThreads), kSoloSmem, stream, a, ymap) != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

}  // namespace tdq
