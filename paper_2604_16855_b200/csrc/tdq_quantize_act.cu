// tdq_quantize_act: token-group dual-constraint activation quantizer (Algorithm S1 steps 1-7).
//
// Six kernels:
//   * act_g32_kernel   the fast path: g = 32, C % 32 == 0, 16-byte aligned rows.  A thread owns one
//     whole group in registers: max, sums, a pruned sorting network for the rank-k magnitude, the DCRP
//     projection, an exact quotient, round-half-even, and one 128-bit store of 32 nibbles (the
//     per-group arithmetic is in tdq_act_group.cuh).
//     One pass over HBM: 2 (bf16) or 4 (fp32) bytes in, 0.5 + 0.125 bytes out per element.
//   * act_g32_ragged_kernel   g = 32 on any other rows: staged element by element.
//   * act_g32_nchw_kernel   channel-major input [B, C, H*W]: each thread loads one position's 32
//     channels (tdq_quantize_act_nchw).
//   * act_fixed_kernel   the fixed-radius control: no reductions, 8 channels per thread
//     (tdq_quantize_act_fixed).
//   * act_wide_kernel   (tdq_quantize_act_wide.cu) groups of a multiple of 8, any C, any alignment.
//   * act_generic_kernel   the rest, that is groups that are not a multiple of 8: one warp per group,
//     rank selection by bisection on the bit patterns of |x|, IEEE division.
//
// Exactness.  Codes must equal clip(rint(fl(fl(clip(x)) / Delta))) in binary32.  The fast
// kernel replaces the division by y = RN(1/Delta), q0 = RN(x y), e = x - q0 Delta (one FMA,
// exact), q1 = RN(q0 + e y).  q0 + e y differs from x / Delta by less than 2^-23 ulp, so q1
// is the correctly rounded quotient unless x / Delta lies within that distance of a midpoint
// between two floats; a quotient that is exactly a multiple of 0.5 is reproduced exactly.
// The group standard deviation only matters when the C1 bound can be the minimum; a cheap
// binary32 test with a 1 % margin on the squared radius (a bf16 one with a wider margin on bf16 input at g = 32) proves
// it cannot for almost every zero-mean group, and the other groups recompute it in binary64: at g = 32, and for groups
// that one lane holds, in the sequential order of the definition; where several lanes share a group (act_wide_kernel,
// act_generic_kernel) lane by lane and then across the lanes.  The two orders differ by at most g 2^-53 relative, which
// moves the binary32 deviation by one unit in its last place in fewer than one group in 2^29 / g.
#include <cmath>

#include "tdq_act_group.cuh"
#include "tdq_common.cuh"
#include "tdq_tc.cuh"

namespace tdq {

std::atomic<uint64_t> g_launch_count{0};

namespace {

// ------------------------------------------------------------------------------------------
// generic kernel: one warp per group

constexpr int kGenericWarps = 4;

template <bool BF16>
__device__ __forceinline__ float load_elem(const void* x, int64_t idx) {
    if (BF16) return bf16_bits_to_float(reinterpret_cast<const uint16_t*>(x)[idx]);
    return reinterpret_cast<const float*>(x)[idx];
}

// k-th smallest (1-indexed) key of the warp's group by bisection over the key space:
// the smallest v with #{key <= v} >= k.  Keys are bit patterns of non-negative floats.
__device__ __forceinline__ uint32_t warp_kth_key(const float* sm, int g, int lane, int k, uint32_t key_max) {
    uint32_t lo = 0, hi = key_max;
    while (lo < hi) {   // at most 32 rounds: hi - lo halves each time
        uint32_t mid = lo + ((hi - lo) >> 1);
        int cnt = 0;
        for (int i = lane; i < g; i += 32) cnt += (__float_as_uint(fabsf(sm[i])) <= mid) ? 1 : 0;
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (cnt >= k) hi = mid; else lo = mid + 1;
    }
    return lo;
}

template <bool BF16>
__global__ void __launch_bounds__(kGenericWarps * 32) act_generic_kernel(ActArgs a) {
    extern __shared__ float smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* sm = smem + (size_t)warp * a.g;
    const int g = a.g;
    const int64_t C_pad = (int64_t)a.K * g;
    for (int64_t gi = (int64_t)blockIdx.x * kGenericWarps + warp; gi < a.total_groups;
         gi += (int64_t)gridDim.x * kGenericWarps) {
        const int64_t m = gi / a.K;
        const int k = (int)(gi - m * a.K);
        uint32_t kmax = 0;
        double s = 0.0;
        for (int i = lane; i < g; i += 32) {
            int64_t ch = (int64_t)k * g + i;
            float v = (ch < a.C) ? load_elem<BF16>(a.x, m * a.row_stride + ch) : 0.0f;
            sm[i] = v;
            kmax = max(kmax, __float_as_uint(fabsf(v)));
            s += (double)v;
        }
        __syncwarp();
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        float c_base = __uint_as_float(kmax);
        if (a.k_base < g) c_base = __uint_as_float(warp_kth_key(sm, g, lane, a.k_base, kmax));
        float thr = 0.0f, sigma = 0.0f;
        if (a.flags & TDQ_ENABLE_C2) thr = __uint_as_float(warp_kth_key(sm, g, lane, a.k_zr, kmax));
        if (a.flags & TDQ_ENABLE_C1) {
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const double mu = s / (double)g;
            double ss = 0.0;
            for (int i = lane; i < g; i += 32) {
                double d = (double)sm[i] - mu;
                ss = __dadd_rn(ss, __dmul_rn(d, d));
            }
            for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            sigma = __fadd_rn(__double2float_rn(sqrt(ss / (double)g)), kStdEps);
        }
        float c, delta;
        dcrp_project(c_base, sigma, thr, a.seven_tau, a.flags, c, delta);
        uint8_t* row_codes = a.codes + (m * C_pad + (int64_t)k * g) / 2;
        for (int j = lane; j < g / 2; j += 32) {
            int q0 = quantize_ieee(sm[2 * j], c, delta);
            int q1 = quantize_ieee(sm[2 * j + 1], c, delta);
            row_codes[j] = (uint8_t)((q0 & 0xF) | ((q1 & 0xF) << 4));
        }
        if (lane == 0) {
            a.scale[gi] = delta;
            if (a.offset) a.offset[gi] = 0.0f;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------
// fast kernel: g = 32, one thread per group

// Threads, and so groups, of a block of the fast kernels.  Small blocks: ten of them fill an SM's registers without the remainder
// that two of 256 threads leave, and no warp waits for more than one other.
constexpr int kFastThreads = 64, kFastBlocks = 16;

// The instances of the fast kernels differ in the registers that they may take, by the blocks per SM of the launch.
enum Length { kFew, kShort, kLong };

// The launch bound of an instance (0: none).
constexpr int resident_blocks(Length len, int long_blocks) { return len == kLong ? long_blocks : len == kFew ? 1 : 0; }

// Blocks per SM up to which fp32 inputs and maps are few.  A bound of one block lets the compiler take 106 to 108 registers (without a bound 87 to
// 96), and the group is done sooner (it may keep more of a group's loads in flight; not shown).  Four such warps fit a scheduler, eight blocks an SM, so beyond
// eight a second round would start that ten or eleven blocks of the other instances do not need.  Quantizer and layer behind it, bound of one
// over none at 1, 3, 5, 7, 8, 8.4 and 9 blocks per SM: fp32 rows of 320 -> 320 1.02, 0.95, 0.97, 0.97, 0.98, 1.01, 1.02, rows of 64 -> 64 1.0, 0.94,
// 0.95, 0.95, 0.96, 1.02, 1.03; maps of 64 -> 64 bf16 0.98, 0.96, 0.95, 0.96, 0.96, 1.04, 1.05, of 768 -> 768 fp32 1.0, 1.0, 0.97, 0.96, 0.98, 0.98,
// 1.04; images of 10 x 10 positions, 256 -> 256 bf16, as launched: 2.6 1.0, 3.8 0.96, 7.7 0.97, 9 1.05.  (Quantizers alone, one behind the
// other, overlap less with it at four to five: 320 channels fp32 3.3 and 3.8 us at 4.9, 4.4 and 4.1 at 5.8.)  bf16 rows take 90 or 92 registers either way.
constexpr int kFewBlocks = 8;

bool few_blocks(int64_t blocks) {
    const int n_sm = current_device_sm_count();
    return blocks <= kFewBlocks * (int64_t)(n_sm > 0 ? n_sm : 148);
}

// Whether a bf16 input is long: at least 40 blocks per SM.  Its instances are held to 64 registers (72 channel-major; they spill 8 and 12
// bytes), with the rare paths out of line, so that 32 warps instead of 20 hide each other's latencies: issue slots 0.54 -> 0.59 busy.  us from a
// graph, the other instances (ten blocks per SM) and these: 16384 x 4096 44.3 and 38.6, 73728 x 256 14.6 and 13.2, 18464 x 768 11.4 and 10.4, the
// same with a mean of 30 (every group takes a rare path) 14.3 and 13.4, map [16, 512, 60, 60] 28.3 and 26.3.  Short inputs lose: where all blocks
// are resident at once the SMs get uneven shares of them, and the kernel behind finds no room to set itself up in; quantizer and layer behind it,
// 9216 x 320 -> 960 (9.7 blocks per SM) 22.4 and 23.9, 18432 x 128 -> 128 (7.8) 10.1 and 11.5, 73728 x 64 -> 64 (15.6) 15.6 and 16.4, 4608 x 1280 ->
// 320 (19.5) 20.1 and 20.8, but 18432 x 512 -> 128 (31) 18.3 and 17.7, 73728 x 256 -> 64 (62) 30.4 and 29.6.  The ratio of the two with a
// layer behind, over 16 layers of 64 to 768 channels in a graph and in a stream, worst and best: at 25 blocks per SM 1.028 and 0.97, 28 1.015 and
// 0.976, 32 1.013 and 0.96, 40 1.005 and 0.94, 64 0.997 and 0.95; maps, 8 layers: at 26 1.013 and 0.988, 34 1.002 and 0.964, 50 1.000 and 0.95.
// Behind a layer with a large output they gain less: of two layers C -> 4 C -> C with their quantizers, C 64 to 768, at 31 blocks per SM 1.023 and
// 0.975, 42 1.012 and 0.98, 64 1.005 and 0.97, 100 0.996 and 0.97 (worst at C = 64 with a binary32 output, which loses up to 80).  Twenty blocks (48 registers)
// are 2 % faster alone (not timed with a layer); two or four groups a thread, the next one's loads in flight: level.
// The ranks of the paper's sweep with the maximum as base radius have them; percentile radii, other ranks and maps taken across the images keep
// the other instances at every length (not timed).
// fp32 has no such instances: with 64 registers it is up to 6 % faster alone (18464 x 768 15.4 and 15.3, 16384 x 4096 62.2 and 58.7), but slower
// with the layer behind it (36864 x 320 -> 320 39.6 and 42.9, 73728 x 256 -> 64 38.8 and 41.9, 18464 x 768 -> 768 52.9 and 55.8, map
// [16, 512, 33, 35] -> 512 34.1 and 35.4), on rows with a pitch (18464 x 768 16.8 and 18.0) and with a mean of 30 (17.8 and 19.8).
bool many_blocks(int64_t blocks) {
    const int n_sm = current_device_sm_count();
    return blocks >= 40 * (int64_t)(n_sm > 0 ? n_sm : 148);
}

// One group: quantize it in registers, write its 16 code bytes and its scale.
template <bool BF16, int KZR, int KB = 32, Length LEN = kShort>
__device__ __forceinline__ void process_group(const uint32_t (&w)[BF16 ? 16 : 32], const ActArgs& a, int64_t gi) {
    uint32_t out[4];
    float delta;
    quantize_group32<BF16, KZR, KB, LEN == kLong>(w, a.seven_tau, a.flags, out, delta, a.k_zr, a.k_base);
    reinterpret_cast<uint4*>(a.codes)[gi] = make_uint4(out[0], out[1], out[2], out[3]);
    a.scale[gi] = delta;
    if (a.offset) a.offset[gi] = 0.0f;
}

// Bound by the instructions of the groups (about 435 a thread, of which the ALU pipe takes 205 at two clocks each; 456 and 235 before
// the clip was one instruction, the maximum came from the network's first layer and the network took signed numbers).  Warps that depend on
// nothing but their own loads keep the pipes fed better than a persistent block with a ring of bulk copies, whose first and last
// tiles cost a latency each and whose number of tiles is rarely a multiple of the blocks; us, that ring (two blocks of eight working
// warps per SM) and this: bf16 18464 x 768 13.7 and 11.8, 73728 x 256 17.0 and 14.9, 9216 x 320 5.9 and 3.8, 1152 x 512 2.4 and 1.75, 16384 x
// 4096 50.4 and 46.3; fp32 18464 x 768 22.6 and 16.2, 9216 x 320 8.8 and 4.9, 256 x 64 3.3 and 1.7.
// A bf16 group is four 16-byte loads of its own thread, whose sectors the neighbours share.  An fp32 group is eight, too far apart
// for that, so a warp loads its 32 groups in order and passes them on through its own part of shared memory (18464 x 768 17.2
// against 16.2 us, 9216 x 320 6.2 and 4.9; bf16 11.8 against 12.0); rows with a pitch, which cost a division a group, are loaded
// directly in either type (the staging kernel that had them before and this, pitch 8 longer: 18464 x 768 bf16 21.6 and 12.8, 9216 x
// 320 6.0 and 3.75; fp32 2304 x 768 8.4 and 5.25, 1152 x 512 4.8 and 2.4).  Blocks of 128 threads: level, long bf16 inputs 1 to 2 % slower.
template <bool BF16, int KZR, int KB, Length LEN>
__global__ void __launch_bounds__(kFastThreads, resident_blocks(LEN, kFastBlocks)) act_g32_kernel(ActArgs a) {
    constexpr int kGroupBytes = BF16 ? 64 : 128;
    constexpr int kChunks = kGroupBytes / 16;          // 16-byte chunks per group
    const int t = threadIdx.x;
    const int64_t gi = (int64_t)blockIdx.x * kFastThreads + t;
    const char* xb = reinterpret_cast<const char*>(a.x);
    const bool flat = a.row_stride == a.C;
    uint32_t w[kChunks * 4];                           // this thread's group: 16 packed bf16 pairs or 32 floats
    pdl_wait();
    pdl_trigger();
    if (BF16 || !flat) {
        if (gi >= a.total_groups) return;
        int64_t off = gi * kGroupBytes;
        if (!flat) {
            int64_t m, k;
            if (a.total_groups <= 0x7fffffff) {
                m = (uint32_t)gi / (uint32_t)a.K;
                k = (uint32_t)gi - (uint32_t)m * (uint32_t)a.K;
            } else {
                m = gi / a.K;
                k = gi - m * a.K;
            }
            off = m * a.row_stride * (BF16 ? 2 : 4) + k * kGroupBytes;
        }
        const uint4* src = reinterpret_cast<const uint4*>(xb + off);
#pragma unroll
        for (int p = 0; p < kChunks; ++p) {
            const uint4 v = __ldg(src + p);
            w[4 * p + 0] = v.x; w[4 * p + 1] = v.y; w[4 * p + 2] = v.z; w[4 * p + 3] = v.w;
        }
    } else {
        // chunk p of the warp's group l lands at l * kChunks + (p ^ l % kChunks): conflict-free both ways
        __shared__ __align__(16) uint4 tile[BF16 ? 1 : kFastThreads * kChunks];
        const int lane = t & 31, w0 = t & ~31;
        const int64_t g0 = gi - lane;
        const uint4* src = reinterpret_cast<const uint4*>(xb + g0 * kGroupBytes) + lane;
        uint4 v[kChunks];
#pragma unroll
        for (int j = 0; j < kChunks; ++j) {
            v[j] = make_uint4(0u, 0u, 0u, 0u);
            if (g0 + (lane + 32 * j) / kChunks < a.total_groups) v[j] = __ldg(src + 32 * j);
        }
#pragma unroll
        for (int j = 0; j < kChunks; ++j) {
            const int ch = lane + 32 * j, l = ch / kChunks, p = ch % kChunks;
            tile[(w0 + l) * kChunks + (p ^ (l % kChunks))] = v[j];
        }
        __syncwarp();
        if (gi >= a.total_groups) return;
#pragma unroll
        for (int p = 0; p < kChunks; ++p) {
            const uint4 u = tile[t * kChunks + (p ^ (t % kChunks))];
            w[4 * p + 0] = u.x; w[4 * p + 1] = u.y; w[4 * p + 2] = u.z; w[4 * p + 3] = u.w;
        }
    }
    process_group<BF16, KZR, KB, LEN>(w, a, gi);
}

// every zero-bin rank of a group of 32 has its instance of the row-major kernel
#define TDQ_ALL_RANKS \
    TDQ_CASE(1) TDQ_CASE(2) TDQ_CASE(3) TDQ_CASE(4) TDQ_CASE(5) TDQ_CASE(6) TDQ_CASE(7) TDQ_CASE(8) \
    TDQ_CASE(9) TDQ_CASE(10) TDQ_CASE(11) TDQ_CASE(12) TDQ_CASE(13) TDQ_CASE(14) TDQ_CASE(15) TDQ_CASE(16) \
    TDQ_CASE(17) TDQ_CASE(18) TDQ_CASE(19) TDQ_CASE(20) TDQ_CASE(21) TDQ_CASE(22) TDQ_CASE(23) TDQ_CASE(24) \
    TDQ_CASE(25) TDQ_CASE(26) TDQ_CASE(27) TDQ_CASE(28) TDQ_CASE(29) TDQ_CASE(30) TDQ_CASE(31) TDQ_CASE(32)
template <bool BF16, Length LEN>
cudaError_t launch_ranks(const ActArgs& a, dim3 grid, cudaStream_t st) {
    const dim3 block(kFastThreads);
    if (a.k_base != 32 && (a.k_base < 29 || a.k_zr != 7)) {
        // any other pair of ranks: the instance that takes both at run time
        return launch_pdl(act_g32_kernel<BF16, 0, 0, LEN>, grid, block, 0, st, a);
    }
    if (a.k_base != 32) {        // percentile base radius: ranks 29..31 beside the default zero-bin rank
        switch (a.k_base) {
#define TDQ_CASE(KB_) case KB_: return launch_pdl(act_g32_kernel<BF16, 7, KB_, LEN>, grid, block, 0, st, a);
            TDQ_CASE(29) TDQ_CASE(30) TDQ_CASE(31)
#undef TDQ_CASE
            default: return cudaErrorInvalidValue;
        }
    }
    switch (a.k_zr) {
#define TDQ_CASE(KZ) case KZ: return launch_pdl(act_g32_kernel<BF16, KZ, 32, LEN>, grid, block, 0, st, a);
        TDQ_ALL_RANKS
#undef TDQ_CASE
        default: return cudaErrorInvalidValue;
    }
}
template <bool BF16>
cudaError_t launch_fast(const ActArgs& a, cudaStream_t st) {
    const int64_t blocks = (a.total_groups + kFastThreads - 1) / kFastThreads;
    const dim3 grid((unsigned)blocks);
    if constexpr (BF16) {
        if (a.k_base == 32 && many_blocks(blocks)) {
            switch (a.k_zr) {
#define TDQ_CASE(KZ) case KZ: return launch_pdl(act_g32_kernel<true, KZ, 32, kLong>, grid, dim3(kFastThreads), 0, st, a);
                TDQ_CASE(4) TDQ_CASE(7) TDQ_CASE(10) TDQ_CASE(13) TDQ_CASE(16) TDQ_CASE(32)
#undef TDQ_CASE
                default: break;
            }
        }
    } else if (few_blocks(blocks)) {
        return launch_ranks<false, kFew>(a, grid, st);
    }
    return launch_ranks<BF16, kShort>(a, grid, st);
}

// ------------------------------------------------------------------------------------------
// g = 32 on rows that 16-byte loads cannot read (a channel count that is not a multiple of 32, a base or pitch off the
// 16-byte grid): the same per-group code behind a staging pass that reads element by element.  A warp stages whole
// groups, lane = channel (or channel pair of bf16), so every load instruction still reads up to 128 contiguous bytes;
// channels past the end of the row are zeros.  The staging costs about as many instructions as the groups themselves.
// Measured, 9217 x 147 fp32: 89 us in the bisection kernel that served these rows before, 7.0 us with batches of eight loads, 6.3
// with all 32 of a warp in flight (20000 x 1000 fp32 47.8 -> 38.9; bf16, 16 at a time, 20689 x 161 12.6 -> 12.0).

// Blocks of 256 threads: with 64 the kernel alone is up to a microsecond faster (9217 x 147 fp32 5.9 -> 4.8), but all SMs then finish
// together and the layer behind it has none to set itself up on: 9217 x 147 -> 63 as a pair 11.9 -> 12.6.
constexpr int kRaggedThreads = 256;
template <bool BF16, int KZR, int KB>
__global__ void __launch_bounds__(kRaggedThreads) act_g32_ragged_kernel(ActArgs a, int32_t pairs_ok) {
    constexpr int kGroupBytes = BF16 ? 64 : 128;
    constexpr int kChunks = kGroupBytes / 16;
    constexpr int kSwzMask = kChunks - 1;
    __shared__ __align__(16) uint4 tile[kRaggedThreads * kChunks];
    pdl_wait();
    pdl_trigger();
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t g0 = (int64_t)blockIdx.x * kRaggedThreads;
    uint8_t* tb = reinterpret_cast<uint8_t*>(tile);
    // channel `e` of local group `l`: the group's 16-byte pieces are swizzled so that a warp reads its groups without bank conflicts
    auto slot = [&](int l, int e) -> uint8_t* {
        const int byte = e * (BF16 ? 2 : 4), swz = BF16 ? ((l >> 1) & kSwzMask) : (l & kSwzMask);
        return tb + (l * kChunks + ((byte >> 4) ^ swz)) * 16 + (byte & 15);
    };
    // The warp's first group; the others follow by stepping through the groups of a token, without a division.  A batch
    // of loads is in flight before the first of them is stored (one dependent load after the other took 21 us instead).
    int64_t gi = g0 + warp * 32;
    int64_t m;
    int32_t k;
    if (a.total_groups <= 0x7fffffff) {
        m = (uint32_t)gi / (uint32_t)a.K;
        k = (int32_t)((uint32_t)gi - (uint32_t)m * (uint32_t)a.K);
    } else {
        m = gi / a.K;
        k = (int32_t)(gi - m * a.K);
    }
    const bool pairs = BF16 && pairs_ok;
    const int e = pairs ? 2 * (lane & 15) : lane;         // this lane's channel; pairs: half-warps take even and odd groups
    const int per = pairs ? 2 : 1;
    const uint8_t* row = reinterpret_cast<const uint8_t*>(a.x) + m * a.row_stride * (BF16 ? 2 : 4);
    const int64_t pitch = a.row_stride * (BF16 ? 2 : 4);
    auto step = [&]() {
        ++gi;
        if (++k == a.K) { k = 0; row += pitch; }
    };
    if (pairs && lane >= 16) step();
    constexpr int kBatch = BF16 ? 16 : 32;                // with pairs a batch is 32 groups, all that a warp stages
    static_assert((BF16 ? 2 : 1) * kBatch <= 32, "a warp's groups");
#pragma unroll 1
    for (int j0 = 0; j0 < 32; j0 += kBatch * per) {
        uint32_t v[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int left = gi < a.total_groups ? (int)min((int64_t)32, a.C - (int64_t)k * 32) : 0;   // channels that exist
            const uint8_t* src = row + ((int64_t)k * 32 + e) * (BF16 ? 2 : 4);
            v[j] = 0u;
            if (!BF16) { if (e < left) v[j] = __ldg(reinterpret_cast<const uint32_t*>(src)); }
            else if (pairs && e + 1 < left) v[j] = __ldg(reinterpret_cast<const uint32_t*>(src));
            else if (e < left) v[j] = __ldg(reinterpret_cast<const uint16_t*>(src));
            step();
            if (pairs) step();
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int l = warp * 32 + j0 + j * per + (pairs ? lane >> 4 : 0);
            if (BF16 && !pairs) *reinterpret_cast<uint16_t*>(slot(l, e)) = (uint16_t)v[j];
            else *reinterpret_cast<uint32_t*>(slot(l, e)) = v[j];
        }
    }
    __syncwarp();                                         // a warp reads back only what it staged
    gi = g0 + t;
    if (gi >= a.total_groups) return;
    uint32_t w[kChunks * 4];
    const int swz = BF16 ? ((t >> 1) & kSwzMask) : (t & kSwzMask);
#pragma unroll
    for (int p = 0; p < kChunks; ++p) {
        const uint4 v = tile[t * kChunks + (p ^ swz)];
        w[4 * p + 0] = v.x; w[4 * p + 1] = v.y; w[4 * p + 2] = v.z; w[4 * p + 3] = v.w;
    }
    process_group<BF16, KZR, KB>(w, a, gi);
}

template <bool BF16>
cudaError_t launch_ragged(const ActArgs& a, cudaStream_t st) {
    const dim3 grid((unsigned)((a.total_groups + kRaggedThreads - 1) / kRaggedThreads)), block(kRaggedThreads);
    const int32_t pairs_ok = reinterpret_cast<uintptr_t>(a.x) % 4 == 0 && a.row_stride % 2 == 0;
    // the zero-bin ranks of the paper's sweep have an instance of their own, every other pair shares the one with run-time ranks
    if (a.k_base == 32) {
        switch (a.k_zr) {
#define TDQ_CASE(KZ) case KZ: return launch_pdl(act_g32_ragged_kernel<BF16, KZ, 32>, grid, block, 0, st, a, pairs_ok);
            TDQ_CASE(4) TDQ_CASE(7) TDQ_CASE(10) TDQ_CASE(13) TDQ_CASE(16) TDQ_CASE(32)
#undef TDQ_CASE
        }
    }
    return launch_pdl(act_g32_ragged_kernel<BF16, 0, 0>, grid, block, 0, st, a, pairs_ok);
}

// ------------------------------------------------------------------------------------------
// channel-major input: x is [B][C][H*W] (a convolutional feature map) and is quantized along C
// without a permuted copy.  A thread takes one group: it loads its position's 32 channels, all in flight together and next to
// its neighbours', and quantizes them like any other group.  Codes and scales come out token-major, [B*H*W, C/2] and
// [B*H*W, C/32].
// A programmatic dependent like the other quantizers: its blocks are in place when the kernel before it ends, and the linear
// layer behind it sets up under its tail ([8, 256, 48, 48] bf16 6.36 -> 5.97 us, [1, 64, 56, 56] fp32 3.17 -> 2.76).
// Bound by the instructions of the groups.  64 positions a block: ten blocks fill an SM's registers without the remainder that two
// of 256 threads leave, and a row's last block wastes less.  us, before (blocks of 256 positions behind a tile in shared memory,
// element-wise loads four at a time where rows are off the 16-byte grid) and now, bf16: [16, 320, 24, 24] 6.4 -> 5.0, [16, 768, 24, 24]
// 12.2 -> 8.0, [16, 512, 60, 60] 39.1 -> 25.2, [16, 512, 33, 35] 33.5 -> 10.1, [2, 320, 7, 7] 3.1 -> 1.75; fp32: [16, 320, 24, 24] 7.2 -> 5.7,
// [16, 256, 31, 31] 15.3 -> 7.0, [16, 768, 12, 12] 4.9 -> 5.4.  A tile in shared memory on 16-byte loads is level or up to 4 %
// slower at 64 positions, 128 positions up to 11 %, 32 up to 5 %.
constexpr int kNchwThreads = 64, kNchwBlocks = 14;

// ACROSS: the positions of all images in one row, a division a thread, instead of blocks of their own for each image, whose last one
// is a quarter full at 144 positions and a sixth at 72.  The time goes in steps of about five blocks per SM (2.5 warps per scheduler), so
// this is taken where it saves one; us, blocks per image and across, the 256-position blocks before them in brackets: bf16 [16, 512,
// 12, 12] (5.2 and 3.9 blocks per SM) 3.42 and 2.63 (2.86), [32, 256, 12, 12] 3.37 and 2.54 (2.83), fp32 [16, 768, 10, 10] (5.2 and 4.05)
// 3.91 and 3.01 (3.47), [64, 512, 12, 12] (20.8 and 15.6) 8.58 and 7.84 (9.79); without a step saved [16, 768, 12, 12] (7.8 and 5.8) 4.43 and 4.69
// (4.55), bf16 [16, 64, 18, 18] 1.91 and 2.03.
struct NchwArgs {
    ActArgs a;          // x, M (positions of all images), K, k_zr, seven_tau, flags, codes, scale, offset
    int64_t HW;         // positions per image
};

template <bool BF16, int KZR, bool ACROSS, Length LEN>
__global__ void __launch_bounds__(kNchwThreads, resident_blocks(LEN, kNchwBlocks)) act_g32_nchw_kernel(NchwArgs n) {
    constexpr int esz = BF16 ? 2 : 4;
    const ActArgs& a = n.a;
    const int t = threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.x * kNchwThreads;    // first position of the block
    const int k = blockIdx.y;                                  // channel group
    int64_t b = blockIdx.z, s = s0 + t;                        // image and position in it
    pdl_wait();
    pdl_trigger();
    if (t >= (ACROSS ? a.M : n.HW) - s0) return;
    if (ACROSS) {
        b = (uint32_t)s / (uint32_t)n.HW;
        s -= b * n.HW;
    }
    const int64_t row = n.HW * esz;
    const uint8_t* src = reinterpret_cast<const uint8_t*>(a.x) + (b * a.C + (int64_t)k * 32) * row + s * esz;
    uint32_t w[BF16 ? 16 : 32];
    if (BF16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t lo = __ldg(reinterpret_cast<const uint16_t*>(src + (2 * i) * row));
            const uint32_t hi = __ldg(reinterpret_cast<const uint16_t*>(src + (2 * i + 1) * row));
            w[i] = lo | (hi << 16);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = __ldg(reinterpret_cast<const uint32_t*>(src + i * row));
    }
    process_group<BF16, KZR, 32, LEN>(w, a, ((b * n.HW + s) * a.K) + k);
}

template <bool BF16, bool ACROSS, Length LEN>
cudaError_t launch_nchw_ranks(const NchwArgs& n, dim3 grid, cudaStream_t st) {
    switch (n.a.k_zr) {
#define TDQ_CASE(KZ) case KZ: return launch_pdl(act_g32_nchw_kernel<BF16, KZ, ACROSS, LEN>, grid, dim3(kNchwThreads), 0, st, n);
        TDQ_CASE(4) TDQ_CASE(7) TDQ_CASE(10) TDQ_CASE(13) TDQ_CASE(16) TDQ_CASE(32)
#undef TDQ_CASE
        default: return cudaErrorInvalidValue;
    }
}
template <bool BF16, bool ACROSS>
cudaError_t launch_nchw(const NchwArgs& n, int64_t B, cudaStream_t st) {
    const int64_t per_row = ((ACROSS ? n.a.M : n.HW) + kNchwThreads - 1) / kNchwThreads, blocks = per_row * n.a.K * (ACROSS ? 1 : B);
    const dim3 grid((unsigned)per_row, (unsigned)n.a.K, ACROSS ? 1u : (unsigned)B);
    if (few_blocks(blocks)) return launch_nchw_ranks<BF16, ACROSS, kFew>(n, grid, st);
    if constexpr (BF16 && !ACROSS) {
        if (many_blocks(blocks)) return launch_nchw_ranks<true, false, kLong>(n, grid, st);
    }
    return launch_nchw_ranks<BF16, ACROSS, kShort>(n, grid, st);
}

// ------------------------------------------------------------------------------------------
// fixed-radius control: no reductions at all.  A thread takes 8 consecutive channels of a row:
// one or two 16-byte loads, eight exact quotients, one 4-byte store of codes.

struct FixedArgs {
    const void* x;
    int64_t M, C, row_stride;   // elements
    int64_t chunks_per_row;     // C / 8
    int32_t g, K;
    float c, delta;
    uint8_t* codes;
    float* scale;
    float* offset;
};

template <bool BF16>
__global__ void __launch_bounds__(256) act_fixed_kernel(FixedArgs f) {
    const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= f.M * f.chunks_per_row) return;
    int64_t m, ch8;
    if (f.M * f.chunks_per_row <= 0xffffffffll) {   // the usual case: 32-bit division
        const uint32_t q32 = (uint32_t)idx / (uint32_t)f.chunks_per_row;
        m = q32;
        ch8 = (uint32_t)idx - q32 * (uint32_t)f.chunks_per_row;
    } else {
        m = idx / f.chunks_per_row;
        ch8 = idx - m * f.chunks_per_row;
    }
    float v[8];
    if (BF16) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(f.x) + m * f.row_stride + ch8 * 8));
        const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    } else {
        const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(f.x) + m * f.row_stride + ch8 * 8);
        const uint4 t0 = __ldg(src), t1 = __ldg(src + 1);
        v[0] = __uint_as_float(t0.x); v[1] = __uint_as_float(t0.y); v[2] = __uint_as_float(t0.z); v[3] = __uint_as_float(t0.w);
        v[4] = __uint_as_float(t1.x); v[5] = __uint_as_float(t1.y); v[6] = __uint_as_float(t1.z); v[7] = __uint_as_float(t1.w);
    }
    uint32_t word = 0u;
    if (f.delta <= 1e30f) {   // two channels at a time, as in the token-group kernels
        const float rcp = __frcp_rn(f.delta);
        const uint64_t rcp2 = f2_pack(rcp, rcp), neg_delta2 = f2_pack(-f.delta, -f.delta);
        const uint64_t magic2 = f2_pack(kRoundMagic8, kRoundMagic8);
        uint32_t acc = 0u;
#pragma unroll
        for (int n = 6; n >= 0; n -= 2)
            nibbles_fast2(f2_pack(clip_f32(v[n], f.c), clip_f32(v[n + 1], f.c)), neg_delta2, rcp2, magic2, acc);
        word = pack_word(acc);
    } else {                  // 1 / Delta would be subnormal: take the IEEE division
#pragma unroll
        for (int n = 0; n < 8; ++n) word |= nibble_ieee(v[n], f.c, f.delta) << (4 * n);
    }
    reinterpret_cast<uint32_t*>(f.codes)[idx] = word;
    const int64_t ch = ch8 * 8;
    if (ch % f.g == 0) {
        const int64_t gi = m * f.K + ch / f.g;
        f.scale[gi] = f.delta;
        if (f.offset) f.offset[gi] = 0.0f;
    }
}

// the zero-bin ranks the channel-major kernel is instantiated for (those of the paper's sweep over zr)
bool fast_rank(int k) { return k == 4 || k == 7 || k == 10 || k == 13 || k == 16 || k == 32; }
// base radius: any rank (the maximum and ranks 29-31 with the default zero-bin rank have instances of their own, the
// other pairs share the instance that takes its ranks at run time)
bool fast_base_rank(const tdq_act_params*) { return true; }

}  // namespace

// Argument checks shared with the fused entry point.
tdq_status check_act_args(const void* x, tdq_dtype dt, int64_t B, int64_t N, int64_t C, int64_t stride,
                          const tdq_act_params* p) {
    if (!x || !p) return TDQ_ERR_INVALID_ARG;
    if (dt != TDQ_F32 && dt != TDQ_BF16) return TDQ_ERR_INVALID_ARG;
    if (B < 0 || N < 0 || C <= 0 || stride < C) return TDQ_ERR_INVALID_ARG;
    if (p->group_size < 2 || p->group_size > 4096 || (p->group_size & 1)) return TDQ_ERR_INVALID_ARG;
    if (!(p->tau > 0.0f) || !(p->zr > 0.0f && p->zr <= 1.0f)) return TDQ_ERR_INVALID_ARG;
    if (!(p->base_percentile > 0.0f && p->base_percentile <= 1.0f)) return TDQ_ERR_INVALID_ARG;
    if (p->flags & ~(TDQ_ENABLE_C1 | TDQ_ENABLE_C2 | TDQ_POW2_STEP)) return TDQ_ERR_INVALID_ARG;
    return TDQ_OK;
}

bool act_fast_path_ok(const void* x, tdq_dtype dt, int64_t C, int64_t stride, const tdq_act_params* p) {
    const int32_t g = p->group_size;
    const int64_t esize = dt == TDQ_BF16 ? 2 : 4;
    return g == 32 && C % 32 == 0 && (reinterpret_cast<uintptr_t>(x) % 16 == 0) &&
           (stride * esize) % 16 == 0 && fast_base_rank(p);   // every zero-bin rank has its instance
}

}  // namespace tdq

using namespace tdq;

extern "C" void tdq_default_act_params(tdq_act_params* p) {
    if (!p) return;
    p->group_size = 32;
    p->tau = 1.0f;
    p->zr = 0.2f;
    p->base_percentile = 1.0f;
    p->flags = TDQ_ENABLE_C1 | TDQ_ENABLE_C2;
}

extern "C" tdq_status tdq_quantize_act(const void* x, tdq_dtype x_dtype, int64_t B, int64_t N, int64_t C,
                                       int64_t row_stride_elems, const tdq_act_params* p, uint8_t* codes,
                                       float* scale, float* offset, void* cuda_stream) {
    tdq_status st = check_act_args(x, x_dtype, B, N, C, row_stride_elems, p);
    if (st != TDQ_OK) return st;
    if (!codes || !scale) return TDQ_ERR_INVALID_ARG;
    const int64_t M = B * N;
    if (M == 0) return TDQ_OK;
    const int32_t g = p->group_size;
    ActArgs a;
    a.x = x;
    a.M = M;
    a.C = C;
    a.row_stride = row_stride_elems;
    a.g = g;
    const int64_t K = (C + g - 1) / g;
    if (K > INT32_MAX) return TDQ_ERR_INVALID_ARG;
    a.K = (int32_t)K;
    a.total_groups = M * K;
    a.k_zr = rank_of(p->zr, g);
    a.k_base = rank_of(p->base_percentile, g);
    a.seven_tau = 7.0f * p->tau;
    a.flags = p->flags;
    a.codes = codes;
    a.scale = scale;
    a.offset = offset;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    cudaError_t e;
    const bool out_aligned = reinterpret_cast<uintptr_t>(codes) % 16 == 0;
    if (out_aligned && g == 32 && a.total_groups / kFastThreads < INT32_MAX) {
        if (!(a.flags & TDQ_ENABLE_C2)) a.k_zr = 7;   // rank unused; pick an instantiated kernel
        if (act_fast_path_ok(x, x_dtype, C, row_stride_elems, p))
            e = (x_dtype == TDQ_BF16) ? launch_fast<true>(a, stream) : launch_fast<false>(a, stream);
        else
            e = (x_dtype == TDQ_BF16) ? launch_ragged<true>(a, stream) : launch_ragged<false>(a, stream);
    } else if (act_wide_ok(a)) {
        e = launch_act_wide(a, x_dtype == TDQ_BF16, stream);
    } else {
        const size_t smem = (size_t)kGenericWarps * g * sizeof(float);
        int64_t blocks = (a.total_groups + kGenericWarps - 1) / kGenericWarps;
        if (blocks > 148 * 64) blocks = 148 * 64;
        if (smem > 48 * 1024) {
            cudaFuncSetAttribute(act_generic_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            cudaFuncSetAttribute(act_generic_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        }
        if (x_dtype == TDQ_BF16)
            act_generic_kernel<true><<<(unsigned)blocks, kGenericWarps * 32, smem, stream>>>(a);
        else
            act_generic_kernel<false><<<(unsigned)blocks, kGenericWarps * 32, smem, stream>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

extern "C" tdq_status tdq_quantize_act_nchw(const void* x, tdq_dtype x_dtype, int64_t B, int64_t C, int64_t H, int64_t W,
                                            const tdq_act_params* p, uint8_t* codes, float* scale, float* offset,
                                            void* cuda_stream) {
    if (H < 0 || W < 0) return TDQ_ERR_INVALID_ARG;
    const int64_t HW = H * W;
    if (B >= 0 && C > 0 && p && B * HW == 0) return TDQ_OK;   // an empty map: nothing to read, x may be null
    tdq_status st = check_act_args(x, x_dtype, B, HW, C, C, p);
    if (st != TDQ_OK) return st;
    if (!codes || !scale) return TDQ_ERR_INVALID_ARG;
    if (B * HW == 0) return TDQ_OK;
    const int32_t g = p->group_size;
    // the channel-major kernel is the fast path only: 32-channel groups, max-abs base radius, a rank it has
    if (g != 32 || C % 32 != 0 || rank_of(p->base_percentile, g) != g || reinterpret_cast<uintptr_t>(codes) % 16 ||
        ((p->flags & TDQ_ENABLE_C2) && !fast_rank(rank_of(p->zr, g))))
        return TDQ_ERR_UNSUPPORTED;
    if (C / 32 > 65535 || B > 65535 || (HW + kNchwThreads - 1) / kNchwThreads > INT32_MAX) return TDQ_ERR_UNSUPPORTED;
    NchwArgs n;
    n.a.x = x;
    n.a.M = B * HW;
    n.a.C = C;
    n.a.row_stride = C;
    n.a.g = g;
    n.a.K = (int32_t)(C / 32);
    n.a.total_groups = n.a.M * n.a.K;
    n.a.k_zr = (p->flags & TDQ_ENABLE_C2) ? rank_of(p->zr, g) : 7;   // rank unused without C2; pick an instantiated kernel
    n.a.k_base = g;
    n.a.seven_tau = 7.0f * p->tau;
    n.a.flags = p->flags;
    n.a.codes = codes;
    n.a.scale = scale;
    n.a.offset = offset;
    n.HW = HW;
    const int64_t apart = B * ((HW + kNchwThreads - 1) / kNchwThreads) * n.a.K, together = (n.a.M + kNchwThreads - 1) / kNchwThreads * n.a.K;
    bool across = false;
    if (together < apart && n.a.M <= INT32_MAX) {
        const int n_sm = current_device_sm_count();
        const int64_t step = 5 * (int64_t)(n_sm > 0 ? n_sm : 148);
        across = (together + step - 1) / step < (apart + step - 1) / step;
    }
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    const bool bf16 = x_dtype == TDQ_BF16;
    const cudaError_t e = across ? (bf16 ? launch_nchw<true, true>(n, B, stream) : launch_nchw<false, true>(n, B, stream))
                                 : (bf16 ? launch_nchw<true, false>(n, B, stream) : launch_nchw<false, false>(n, B, stream));
    if (e != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

extern "C" tdq_status tdq_quantize_act_fixed(const void* x, tdq_dtype x_dtype, int64_t B, int64_t N, int64_t C,
                                             int64_t row_stride_elems, int32_t group_size, float radius, uint8_t* codes,
                                             float* scale, float* offset, void* cuda_stream) {
    if (!x || !codes || !scale) return TDQ_ERR_INVALID_ARG;
    if (x_dtype != TDQ_F32 && x_dtype != TDQ_BF16) return TDQ_ERR_INVALID_ARG;
    if (B < 0 || N < 0 || C <= 0 || row_stride_elems < C) return TDQ_ERR_INVALID_ARG;
    if (group_size < 2 || group_size > 4096 || (group_size & 1) || !(radius > 0.0f)) return TDQ_ERR_INVALID_ARG;
    const int64_t M = B * N;
    if (M == 0) return TDQ_OK;
    const int64_t esz = x_dtype == TDQ_BF16 ? 2 : 4;
    if (group_size % 8 || C % group_size || reinterpret_cast<uintptr_t>(x) % 16 || (row_stride_elems * esz) % 16 ||
        reinterpret_cast<uintptr_t>(codes) % 4)
        return TDQ_ERR_UNSUPPORTED;
    FixedArgs f;
    f.x = x; f.M = M; f.C = C; f.row_stride = row_stride_elems; f.chunks_per_row = C / 8;
    f.g = group_size; f.K = (int32_t)(C / group_size);
    f.c = fmaxf(radius, kClipFloor);
    f.delta = fmaxf(f.c / kQmax, kStepFloor);      // binary32 division on the host: the same IEEE operation
    f.codes = codes; f.scale = scale; f.offset = offset;
    const int64_t blocks = (M * f.chunks_per_row + 255) / 256;
    if (blocks > INT32_MAX) return TDQ_ERR_UNSUPPORTED;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    if (x_dtype == TDQ_BF16)
        act_fixed_kernel<true><<<(unsigned)blocks, 256, 0, stream>>>(f);
    else
        act_fixed_kernel<false><<<(unsigned)blocks, 256, 0, stream>>>(f);
    if (cudaGetLastError() != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}

// ------------------------------------------------------------------------------------------
// tdq_quantize_status and its self-test.  No quantizer kernel waits on a barrier at present, so only the self-test writes the word.

namespace tdq {
namespace {
// Bits 0-7 name the wait that ran out (14 the self-test), bits 8-31 the CTA.  One word per device, read and cleared by
// tdq_quantize_status().
__device__ uint32_t g_act_wait_status = 0u;

// One warp: a fresh barrier with one expected arrival that never comes, waited on with the linear layer's
// routine and a short limit.  Nothing is in flight when the warp leaves.
__global__ void __launch_bounds__(32) act_wait_selftest_kernel(long long limit) {
    __shared__ Ctrl c;
    if (threadIdx.x == 0) {
        mbar_init(&c.full[0], 1);
        c.abort_flag = 0;
    }
    __syncwarp();
    mbar_wait_warp(&c.full[0], 0u, &c, &g_act_wait_status, 14u, limit);
}
}  // namespace

tdq_status act_wait_selftest(long long limit_cycles, cudaStream_t stream) {
    act_wait_selftest_kernel<<<1, 32, 0, stream>>>(limit_cycles);
    if (cudaGetLastError() != cudaSuccess) return TDQ_ERR_CUDA;
    g_launch_count.fetch_add(1, std::memory_order_relaxed);
    return TDQ_OK;
}
}  // namespace tdq

extern "C" tdq_status tdq_quantize_status(void* cuda_stream, uint32_t* detail) {
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    uint32_t word = 0;
    const uint32_t zero = 0;
    if (cudaMemcpyFromSymbolAsync(&word, g_act_wait_status, sizeof word, 0, cudaMemcpyDeviceToHost, stream) != cudaSuccess)
        return TDQ_ERR_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return TDQ_ERR_CUDA;
    if (word != 0 &&
        (cudaMemcpyToSymbolAsync(g_act_wait_status, &zero, sizeof zero, 0, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
         cudaStreamSynchronize(stream) != cudaSuccess))
        return TDQ_ERR_CUDA;
    if (detail) *detail = word;
    return word == 0 ? TDQ_OK : TDQ_ERR_DEVICE_TIMEOUT;
}
