// The token-group quantizer for every group size that is a multiple of 8 and any row layout: wide groups (64 up to a
// whole token of 4096 channels), channel counts that are not a multiple of the group, rows without 16-byte alignment.
// (g = 32 on aligned rows has kernels of its own in tdq_quantize_act.cu.)
//
// L lanes of a warp (1 to 32), or all of two or four warps, own a group and hold it in registers: chunk n of 8
// channels belongs to lane n % (lanes), so a warp reads and writes contiguous pieces.  One pass over memory: 2 or 4 bytes in, 0.5 out per channel.
//
// What bounds it is instruction issue, and of that the rank selection.  It is a search for the k-th smallest magnitude
// over the ordered bit patterns of |x|: count the elements <= a probe (bf16: two per packed compare and add), narrow the
// bracket, repeat.  A plain bisection needs 15 (bf16) or 31 (fp32) counting passes.  Three things keep their number down:
//   * the zero-bin rank only matters where 14 thr < c_base, so the search ends once the bracket lies above c_base / 14, and
//     the first probe is that or the Gaussian quantile of the group's rms, whichever is less (for a Gaussian group of 128 the
//     20 % quantile is 3.5 sigma / 14 and the maximum 2.8 sigma: one probe);
//   * the probes then follow straight lines of the counting function (it is nearly flat near zero, where the rank lies), and
//     an end of the bracket that stays while the other moves twice counts for half (the Illinois rule), which is what a steep or
//     curved piece needs: the percentile radius, heavy tails;
//   * the third probe asks for the zeros, of which padding and rectified inputs have more than the rank: the lines approach
//     that jump from above a bit at a time (36 probes for bf16, 70 for fp32, for every group of such a warp).
// A bisection step every eighth probe is the guarantee (it halves the bit patterns, so it is of little use while the lower end is
// near zero: every sixth costs heavy tails 2 % of the time and a 0.9 percentile 7 %); the search ends when the bracket's upper end has
// exactly k elements at or below it or its lower end k - 1.  1.2 to 1.5 probes on average at g = 128 and zr = 0.2, three for the slowest
// of the eight groups of a warp.  On heavy tails (a Gaussian over another's magnitude) nothing stops early, and what a probe does
// besides counting shows: fp32 16384 x 1536 at g = 768 44 us in the plain search, 49 in this one.
//
// Lanes per group and chunks per lane (NC): as few lanes as keep a lane at four chunks (32 channels), because the
// probe's bookkeeping and the reduction over the group are paid per lane.  Past 1024 channels two or four warps share a
// group: a lane with more chunks has the same instruction count, but the straight-line code for 16 chunks ran at 0.47
// instructions per clock with the instruction cache as its main stall.  Groups of up to 32 channels follow the same rule,
// one lane each: 18464 x 768 bf16 at g = 8 143 -> 39 us against four lanes with one chunk each, at g = 16 81 -> 30, at
// g = 24 56 -> 25, at g = 32 (codes off the 16-byte grid) 43 -> 24.
//
// Measured (B200, from a graph), us, before the search had the last two rules, the first one and rough moments, and now:
// bf16 18464 x 768 at g = 128 24.8 -> 19.5 (zr = 0.3 24.8 -> 16.8, rectified 47.2 -> 17.6, p = 0.9 48.7 -> 33.2, with a mean
// of 30 39.3 -> 22.9), at g = 64 25.0 -> 20.7; 46005 x 608 at g = 128 (a quarter of a row's last group is padding) 129.4 ->
// 36.9, with p = 0.9 175.0 -> 69.1; 16384 x 4096 at g = 4096 76.8 -> 64.6 (of it eight chunks a lane 8.4); fp32 18464 x 768 at
// g = 128 26.2 -> 22.8, rectified 76.1 -> 18.6.  The bisection kernel that served these cases at first: 978 us on the long groups.
// Since then the maximum and both moments take one exchange, the element next to the last probe is found in one pass for either side of it,
// and the clip is one instruction: 16384 x 4096 at g = 4096 64.2 -> 56.0; with the layer behind it 222.5 -> 213.1 from a graph, 245.8 -> 238.5 in a
// stream (3 %).
#include <climits>

#include "tdq_act_group.cuh"
#include "tdq_common.cuh"

namespace tdq {
namespace {

constexpr int kWideThreads = 128;

struct WideArgs {
    ActArgs a;
    int32_t load_mode;     // 0: 16-byte loads, 1: 4-byte loads (pairs of bf16), 2: element by element
    float guess_zr, guess_base;   // Gaussian quantile of the two ranks, in units of the rms
};

// Reductions over the lanes of a group: L lanes of one warp, or (W > 1) all W warps of the block, which then exchange
// their results through shared memory.  `turn` alternates between two sets of slots, so that one barrier per
// reduction is enough.
template <int L, int W, typename T, typename F>
__device__ __forceinline__ T group_reduce(T v, F f, uint32_t& turn) {
#pragma unroll
    for (int o = L / 2; o; o >>= 1) v = f(v, __shfl_xor_sync(0xffffffffu, v, o));
    if constexpr (W > 1) {
        __shared__ double slots[2][W];
        T* mine = reinterpret_cast<T*>(&slots[turn & 1u][threadIdx.x >> 5]);
        if ((threadIdx.x & 31) == 0) *mine = v;
        __syncthreads();
        v = *reinterpret_cast<T*>(&slots[turn & 1u][0]);
#pragma unroll
        for (int w = 1; w < W; ++w) v = f(v, *reinterpret_cast<T*>(&slots[turn & 1u][w]));
        ++turn;
    }
    return v;
}

// Largest bit pattern of the group: over a full warp one instruction instead of five shuffles.
template <int L, int W>
__device__ __forceinline__ uint32_t group_max(uint32_t v, uint32_t& turn) {
    auto f = [](uint32_t p, uint32_t q) { return max(p, q); };
    if constexpr (L < 32) return group_reduce<L, W>(v, f, turn);
    v = __reduce_max_sync(0xffffffffu, v);
    return W > 1 ? group_reduce<1, W>(v, f, turn) : v;
}
// The group's largest magnitude and its two moments, with one exchange between the warps.  The lanes of a group halve the moments between
// them first, so that a shuffle after the first carries one of the two for each half.
template <int L, int W>
__device__ __forceinline__ void group_stats(uint32_t& kmax, float& s1, float& s2, uint32_t& turn) {
    kmax = group_max<L, 1>(kmax, turn);
    if constexpr (L > 1) {
        const bool up = (threadIdx.x & (L / 2)) != 0;
        float v = (up ? s2 : s1) + __shfl_xor_sync(0xffffffffu, up ? s1 : s2, L / 2);
#pragma unroll
        for (int o = L / 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const float w = __shfl_xor_sync(0xffffffffu, v, L / 2);
        s1 = up ? w : v;
        s2 = up ? v : w;
    }
    if constexpr (W > 1) {
        __shared__ float4 slots[W];
        if ((threadIdx.x & 31) == 0) slots[threadIdx.x >> 5] = make_float4(__uint_as_float(kmax), s1, s2, 0.0f);
        __syncthreads();
        const float4 v = slots[0];
        kmax = __float_as_uint(v.x);
        s1 = v.y;
        s2 = v.z;
#pragma unroll
        for (int w = 1; w < W; ++w) {
            const float4 u = slots[w];
            kmax = max(kmax, __float_as_uint(u.x));
            s1 += u.y;
            s2 += u.z;
        }
    }
}

// The same for a sum of small whole numbers held in floats.  Over a full warp it is one integer reduction of the floats'
// bits above 2^23 (whose low bits are the number) instead of five shuffles and adds.
template <int L, int W>
__device__ __forceinline__ float group_sum_count(float v, uint32_t& turn) {
    auto add = [](float p, float q) { return p + q; };
    if constexpr (L < 32) {
        return group_reduce<L, 1>(v, add, turn);
    } else {
        constexpr float kMagic = 8388608.0f;             // 2^23 = 0x4b000000; 32 of them add up to 0x60000000 mod 2^32
        const uint32_t sum = __reduce_add_sync(0xffffffffu, __float_as_uint(v + kMagic)) - 0x60000000u;
        v = __uint_as_float(sum | 0x4b000000u) - kMagic;
        return W > 1 ? group_reduce<1, W>(v, add, turn) : v;
    }
}

// A lane's share of a group: NC chunks of 8 channels; bf16 as packed pairs.  Chunks past the group are zero.
template <bool BF16, int NC>
struct Share {
    static constexpr int kWords = BF16 ? 4 : 8;
    uint32_t w[NC * kWords];
    __device__ __forceinline__ float get(int i) const {
        if (BF16) return (i & 1) ? __uint_as_float(w[i >> 1] & 0xffff0000u) : __uint_as_float(w[i >> 1] << 16);
        return __uint_as_float(w[i]);
    }
    // The phases of the kernel each unpack what they need: without this the compiler keeps the unpacked floats of the
    // whole share alive from one phase to the next (twice the registers, half the warps).
    __device__ __forceinline__ void opaque() {
#pragma unroll
        for (int i = 0; i < NC * kWords; ++i) asm volatile("" : "+r"(w[i]));
    }
    // Elements of this share whose magnitude is at most the float with bit pattern `key`, as a float: counts stay exact
    // and never pass through the conversion unit.  bf16: `mag` holds |x| packed (taking the
    // signs off in every compare is slower), probes are whole bf16 keys, the packed
    // compare yields 1.0 or 0.0 and a bf16 holds counts up to 256.
    __device__ __forceinline__ float count_le(const uint32_t (&mag)[NC * kWords], uint32_t key) const {
        if (BF16) {
            const uint32_t m = __byte_perm(key, 0u, 0x3232u);
            const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162*>(&m);
            __nv_bfloat162 n[2];
            n[0] = n[1] = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll
            for (int i = 0; i < NC * kWords; ++i) n[i & 1] = __hadd2(n[i & 1], __hle2(*reinterpret_cast<const __nv_bfloat162*>(&mag[i]), m2));
            const __nv_bfloat162 s2 = __hadd2(n[0], n[1]);
            const uint32_t s = *reinterpret_cast<const uint32_t*>(&s2);
            return __uint_as_float(s << 16) + __uint_as_float(s & 0xffff0000u);
        }
        const float m = __uint_as_float(key);
        float n0 = 0.0f, n1 = 0.0f;
#pragma unroll
        for (int i = 0; i < NC * kWords; i += 2) {
            n0 += fabsf(__uint_as_float(w[i])) <= m ? 1.0f : 0.0f;
            n1 += fabsf(__uint_as_float(w[i + 1])) <= m ? 1.0f : 0.0f;
        }
        return n0 + n1;
    }
    // The magnitude of this share that is nearest to `key` from below (at most it) or from above, as a number that is larger the nearer it is;
    // magnitude() takes the group's largest such number back.  Setting the sign bit and taking key + 1 off leaves 0x8000 + |x| - key - 1,
    // which as a signed number is largest for the one and smallest for the other, with those on the wrong side beyond zero.
    __device__ __forceinline__ uint32_t nearest(int key, bool below) const {
        if constexpr (BF16) {
            const uint32_t m = ((uint32_t)key + 1u) * 0x00010001u;
            uint32_t hi = 0x80008000u, lo = 0x7fff7fffu;
#pragma unroll
            for (int i = 0; i < NC * kWords; i += 2) {
                const uint32_t t0 = (w[i] | 0x80008000u) - m, t1 = (w[i + 1] | 0x80008000u) - m;   // no borrow: key + 1 <= 0x8000
                hi = __vimax3_s16x2(hi, t0, t1);
                lo = __vimin3_s16x2(lo, t0, t1);
            }
            const int a = max((int)(int16_t)hi, (int)hi >> 16), b = min((int)(int16_t)lo, (int)lo >> 16);
            return (uint32_t)(below ? a : ~b) ^ 0x80000000u;
        } else {
            const uint32_t m = (uint32_t)key + 1u;
            int hi = INT_MIN, lo = INT_MAX;
#pragma unroll
            for (int i = 0; i < NC * kWords; i += 2) {
                const int t0 = (int)((w[i] | 0x80000000u) - m), t1 = (int)((w[i + 1] | 0x80000000u) - m);
                hi = __vimax3_s32(hi, t0, t1);
                lo = __vimin3_s32(lo, t0, t1);
            }
            return (uint32_t)(below ? hi : ~lo) ^ 0x80000000u;
        }
    }
    static __device__ __forceinline__ uint32_t magnitude(uint32_t n, int key, bool below) {   // bit pattern
        n ^= 0x80000000u;
        const uint32_t t = (below ? n : ~n) + (uint32_t)key + 1u;
        return BF16 ? (t & 0x7fffu) << 16 : t & 0x7fffffffu;
    }
};

// The k-th smallest magnitude (bit pattern) of the group; k counts the zeros that stand for absent elements too.
// kmax is the group's largest magnitude, guess the first probe.  limit: a magnitude above which the caller does not need to
// know the result; what is returned then is some magnitude above it.
template <bool BF16, int NC, int L, int W>
__device__ __forceinline__ uint32_t group_kth(const Share<BF16, NC>& x, int k, int absent, uint32_t kmax, float guess, float limit, uint32_t& turn) {
    constexpr int kStep = BF16 ? 16 : 0;             // keys are compared as key >> kStep
    constexpr float n = (float)(L * W * NC * 8);
    if (BF16) kmax >>= kStep;
    uint32_t mag[NC * Share<BF16, NC>::kWords];
#pragma unroll
    for (int i = 0; i < NC * Share<BF16, NC>::kWords; ++i) mag[i] = BF16 ? x.w[i] & 0x7fff7fffu : 0u;
    int lo = -1, hi = (int)kmax;                     // count(lo) < k <= count(hi)
    const int enough = (int)(__float_as_uint(limit) >> kStep);
    // counts without the absent elements' zeros (a count below them stands for none)
    const float kf = (float)k, af = (float)absent;
    float c_lo = 0.0f, c_hi = n;
    float probe_v = fminf(guess, limit);
    const float aim = kf - af - 0.5f;                // between the k-th element and the one before it
    float w_lo = 1.0f, w_hi = 1.0f;                  // an end that stays while the other moves twice counts for half (Illinois rule)
    int last = 0;
    int round = 0;
#pragma unroll 1
    for (;;) {
        const bool done = hi - lo <= 1 || c_hi == kf || c_lo + 1.0f == kf || lo >= enough;
        if (L == 32 ? done : __all_sync(0xffffffffu, done)) break;
        int p = (int)(__float_as_uint(probe_v) >> kStep);
        ++round;
        if (round == 3 && lo < 0) p = 0;             // as many zeros as that: padding, rectified inputs
        if (round == 8) { p = lo + ((hi - lo) >> 1); round = 0; }   // the guarantee
        p = max(lo + 1, min(hi - 1, p));
        const float c = group_sum_count<L, W>(x.count_le(mag, (uint32_t)p << kStep), turn);
        if (!done) {
            const bool up = c >= kf;
            if (up) { hi = p; c_hi = c; w_lo = last > 0 ? 0.5f * w_lo : 1.0f; w_hi = 1.0f; last = 1; }
            else { lo = p; c_lo = c; w_hi = last < 0 ? 0.5f * w_hi : 1.0f; w_lo = 1.0f; last = -1; }
            const float v_lo = __uint_as_float((uint32_t)max(lo, 0) << kStep), v_hi = __uint_as_float((uint32_t)hi << kStep);
            const float n_lo = fmaxf(c_lo - af, 0.0f);
            // no upper end but the maximum yet: the line through the origin; else the line between the ends
            const bool open = c_hi == n && n_lo > 0.0f;
            const float below = (aim - n_lo) * w_lo, above = (c_hi - af - aim) * w_hi;
            const float slope = __fdividef(open ? v_lo : v_hi - v_lo, open ? n_lo : below + above);
            probe_v = open ? slope * aim : fmaf(slope, below, v_lo);
        }
    }
    // exactly k elements at or below hi: the largest of them; exactly k - 1 at or below lo: the smallest of the rest
    // (all lanes of the warp take part in the reductions)
    const bool wide = hi - lo > 1 && lo < enough, below = wide && c_hi == kf;
    uint32_t r = (uint32_t)hi << kStep;
    if (__any_sync(0xffffffffu, wide)) {
        const int key = below ? hi : lo;
        const uint32_t n = group_max<L, W>(x.nearest(key, below), turn);
        if (wide) r = x.magnitude(n, key, below);
    }
    return r;
}

// Resident blocks the registers are allocated for: the share (4 or 8 words a chunk) and about fifty more.  No instance spills.  us from a
// graph, bf16, with a block less, so many and one more: 16384 x 4096 at g = 4096 59.6, 56.0 and 55.8 (with p = 0.9 96.2, 96.7 and 100.0), 16384 x
// 1536 at 512 29.1, 28.1 and 28.0, 18464 x 768 at 128 19.1, 18.6 and 18.9 (p = 0.9 30.5, 30.3 and 31.4); inputs of one round or less like fewer:
// 1024 x 4096 at 4096 7.4, 8.0 and 8.7, 4616 x 768 at 128 7.5, 8.1 and 8.8.  fp32 takes the same registers either way.
constexpr int wide_blocks(bool bf16, int nc) {
    const int regs = bf16 ? 4 * nc + 48 : 8 * nc + 64;
    return 512 / (regs < 64 ? 64 : regs);
}

// Eight codes by IEEE division, out of line: 1 / Delta is subnormal in hardly any group.
__device__ __noinline__ uint32_t word_ieee(float4 a, float4 b, float c, float delta) {
    return nibble_ieee(a.x, c, delta) | nibble_ieee(a.y, c, delta) << 4 | nibble_ieee(a.z, c, delta) << 8 | nibble_ieee(a.w, c, delta) << 12 |
           nibble_ieee(b.x, c, delta) << 16 | nibble_ieee(b.y, c, delta) << 20 | nibble_ieee(b.z, c, delta) << 24 | nibble_ieee(b.w, c, delta) << 28;
}

template <bool BF16, int NC, int L, int W>
__global__ void __launch_bounds__(W > 1 ? W * 32 : kWideThreads, wide_blocks(BF16, NC) * (W == 2 ? 2 : 1)) act_wide_kernel(const WideArgs wa) {
    const ActArgs& a = wa.a;
    constexpr int kPerWarp = 32 / L;
    constexpr int kLanes = L * W;                     // of a group
    const int lane = threadIdx.x & 31, sub = W > 1 ? (int)threadIdx.x : lane & (L - 1);
    const int64_t gw = W > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * (kWideThreads / 32) + (threadIdx.x >> 5);
    uint32_t turn = 0u;
    pdl_wait();
    pdl_trigger();
    if (gw * kPerWarp >= a.total_groups) return;      // the whole warp
    const int64_t gi_raw = gw * kPerWarp + lane / L;
    const bool live = gi_raw < a.total_groups;        // the last warp's lanes past the end repeat its last group
    const int64_t gi = live ? gi_raw : a.total_groups - 1;
    int64_t m, k;
    if (a.total_groups <= 0x7fffffff) {
        const uint32_t q = (uint32_t)gi / (uint32_t)a.K;
        m = q;
        k = (uint32_t)gi - q * (uint32_t)a.K;
    } else {
        m = gi / a.K;
        k = gi - m * a.K;
    }
    const int g = a.g;
    const int64_t ch0 = k * g;                        // first channel of the group
    const int in_row = (int)min((int64_t)g, a.C - ch0);   // channels that exist; the rest of the group is zero
    Share<BF16, NC> x;
    constexpr int kW = Share<BF16, NC>::kWords;
    const uint8_t* src = reinterpret_cast<const uint8_t*>(a.x) + (m * a.row_stride + ch0) * (BF16 ? 2 : 4);
#pragma unroll
    for (int j = 0; j < NC * kW; ++j) x.w[j] = 0u;
    if (wa.load_mode == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int e = (sub + c * kLanes) * 8;
            if (e + 8 <= in_row) {
#pragma unroll
                for (int h = 0; h < kW / 4; ++h) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + e * (BF16 ? 2 : 4)) + h);
                    x.w[c * kW + 4 * h] = v.x; x.w[c * kW + 4 * h + 1] = v.y;
                    x.w[c * kW + 4 * h + 2] = v.z; x.w[c * kW + 4 * h + 3] = v.w;
                }
            }
        }
    } else if (wa.load_mode == 1) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int e = (sub + c * kLanes) * 8;
            if (e + 8 <= in_row) {
#pragma unroll
                for (int j = 0; j < kW; ++j) x.w[c * kW + j] = __ldg(reinterpret_cast<const uint32_t*>(src + e * (BF16 ? 2 : 4)) + j);
            }
        }
    }
    // the chunk that the end of the row cuts (all chunks where elements are not even 4-byte aligned)
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int e = (sub + c * kLanes) * 8;
        if (e < in_row && (wa.load_mode == 2 || e + 8 > in_row)) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (e + j < in_row) {
                    if (BF16) x.w[c * kW + j / 2] |= (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(src) + e + j) << (16 * (j & 1));
                    else x.w[c * kW + j] = __ldg(reinterpret_cast<const uint32_t*>(src) + e + j);
                }
            }
        }
    }

    // largest magnitude and the moments
    uint32_t kmax = 0u;
    float s1 = 0.0f, s2 = 0.0f;
    if (BF16) {
#pragma unroll
        for (int j = 0; j < NC * kW; ++j) kmax = max_mag2(kmax, x.w[j]);
        kmax = __float_as_uint(larger_half(kmax));
    } else {
#pragma unroll
        for (int j = 0; j < NC * kW; ++j) kmax = max(kmax, x.w[j] & 0x7fffffffu);
    }
    // Moments: for bf16 rough ones, two channels per instruction, at most 16 additions in a sum (see c1_cannot_bind_rough)
    if (BF16) {
#pragma unroll
        for (int h = 0; h < NC * kW; h += 16) {
            __nv_bfloat162 s1b = *reinterpret_cast<const __nv_bfloat162*>(&x.w[h]);
            __nv_bfloat162 s2b = __hmul2(s1b, s1b);
#pragma unroll
            for (int j = h + 1; j < (h + 16 < NC * kW ? h + 16 : NC * kW); ++j) {
                const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&x.w[j]);
                s1b = __hadd2(s1b, v);
                s2b = __hfma2(v, v, s2b);
            }
            s1 += __low2float(s1b) + __high2float(s1b);
            s2 += __low2float(s2b) + __high2float(s2b);
        }
    } else {
#pragma unroll
        for (int j = 0; j < NC * 8; ++j) {
            const float v = x.get(j);
            s1 += v;
            s2 = fmaf(v, v, s2);
        }
    }
    x.opaque();
    group_stats<L, W>(kmax, s1, s2, turn);

    const int absent = kLanes * NC * 8 - g;
    const float rms = sqrtf(s2 / (float)g);
    float c_base = __uint_as_float(kmax), thr = 0.0f;
    if (a.k_base < g) c_base = __uint_as_float(group_kth<BF16, NC, L, W>(x, a.k_base + absent, absent, kmax, rms * wa.guess_base, INFINITY, turn));
    // C2 only acts if 14 thr < c_base: a threshold above c_base / 14 (rounded up a little) need not be known
    if (a.flags & TDQ_ENABLE_C2)
        thr = __uint_as_float(group_kth<BF16, NC, L, W>(x, a.k_zr + absent, absent, kmax, rms * wa.guess_zr, c_base * (1.000001f / 14.0f), turn));
    float sigma = INFINITY;                           // an idle C1 bound
    if (a.flags & TDQ_ENABLE_C1) {
        float cmin = c_base;
        if (a.flags & TDQ_ENABLE_C2) cmin = fminf(cmin, __fmul_rn(14.0f, thr));
        bool idle = BF16 ? c1_cannot_bind_rough(s1, s2, a.seven_tau, cmin, 1.0f / (float)g) : c1_cannot_bind(s1, s2, a.seven_tau, cmin, 1.0f / (float)g);
        if (BF16 && !__all_sync(0xffffffffu, idle)) {     // the rough moments do not decide: binary32 ones
            x.opaque();
            s1 = 0.0f;
            s2 = 0.0f;
#pragma unroll
            for (int j = 0; j < NC * 8; ++j) {
                const float v = x.get(j);
                s1 += v;
                s2 = fmaf(v, v, s2);
            }
            s1 = group_reduce<L, W>(s1, [](float p, float q) { return p + q; }, turn);
            s2 = group_reduce<L, W>(s2, [](float p, float q) { return p + q; }, turn);
            idle = c1_cannot_bind(s1, s2, a.seven_tau, cmin, 1.0f / (float)g);
        }
        if (!__all_sync(0xffffffffu, idle)) {
            x.opaque();
            // binary64, per lane and then across the lanes; the absent chunks are left out of the second sum
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < NC * 8; ++j) s = __dadd_rn(s, (double)x.get(j));
            x.opaque();
            const double mu = group_reduce<L, W>(s, [](double p, double q) { return p + q; }, turn) / (double)g;
            double ss = 0.0;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if ((sub + c * kLanes) * 8 < g) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const double d = __dsub_rn((double)x.get(c * 8 + j), mu);
                        ss = __dadd_rn(ss, __dmul_rn(d, d));
                    }
                }
            }
            ss = group_reduce<L, W>(ss, [](double p, double q) { return p + q; }, turn);
            const float exact = __fadd_rn(__double2float_rn(sqrt(ss / (double)g)), kStdEps);
            if (!idle) sigma = exact;
        }
    }
    x.opaque();
    float c, delta;
    dcrp_project(c_base, sigma, thr, a.seven_tau, a.flags, c, delta);

    if (live) {
        uint32_t* codes = reinterpret_cast<uint32_t*>(a.codes) + gi * (g / 8);
        const bool fast = delta <= 1e30f;             // otherwise 1 / Delta would be subnormal: take the IEEE division
        const float rcp = fast ? __frcp_rn(delta) : 0.0f;
        const uint32_t cup = (__float_as_uint(c) + 0xffffu) >> 16, c2 = cup | (cup << 16);
        const uint64_t rcp2 = f2_pack(rcp, rcp), neg_delta2 = f2_pack(-delta, -delta), magic2 = f2_pack(kRoundMagic8, kRoundMagic8);
#pragma unroll
        for (int ch = 0; ch < NC; ++ch) {
            const int n = sub + ch * kLanes;
            if (n * 8 >= g) continue;
            uint32_t acc = 0u;
            if (fast) {
#pragma unroll
                for (int j = 6; j >= 0; j -= 2) {
                    uint64_t xt;
                    if (BF16) {                       // two channels at a time against c rounded up to a bf16 (see quantize_group32)
                        const uint32_t u = min_mag2(x.w[ch * 4 + j / 2], c2);
                        xt = f2_pack(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
                    } else {
                        const float v0 = x.get(ch * 8 + j), v1 = x.get(ch * 8 + j + 1);
                        xt = f2_pack(clip_f32(v0, c), clip_f32(v1, c));
                    }
                    nibbles_fast2(xt, neg_delta2, rcp2, magic2, acc);
                }
                acc = pack_word(acc);
            } else {
                acc = word_ieee(make_float4(x.get(ch * 8), x.get(ch * 8 + 1), x.get(ch * 8 + 2), x.get(ch * 8 + 3)),
                                make_float4(x.get(ch * 8 + 4), x.get(ch * 8 + 5), x.get(ch * 8 + 6), x.get(ch * 8 + 7)), c, delta);
            }
            codes[n] = acc;
        }
        if (sub == 0) {
            a.scale[gi] = delta;
            if (a.offset) a.offset[gi] = 0.0f;
        }
    }
}

template <bool BF16, int NC, int L, int W = 1>
cudaError_t launch(const WideArgs& w, cudaStream_t st) {
    const int64_t per_block = W > 1 ? 1 : (int64_t)(kWideThreads / 32) * (32 / L);
    const int64_t blocks = (w.a.total_groups + per_block - 1) / per_block;
    return launch_pdl(act_wide_kernel<BF16, NC, L, W>, dim3((unsigned)blocks), dim3(W > 1 ? W * 32 : kWideThreads), 0, st, w);
}

template <bool BF16>
cudaError_t pick(const WideArgs& w, cudaStream_t st) {
    const int chunks = w.a.g / 8;
    if (chunks <= 1) return launch<BF16, 1, 1>(w, st);
    if (chunks <= 2) return launch<BF16, 2, 1>(w, st);
    if (chunks <= 3) return launch<BF16, 3, 1>(w, st);
    if (chunks <= 4) return launch<BF16, 4, 1>(w, st);
    if (chunks <= 6) return launch<BF16, 3, 2>(w, st);
    if (chunks <= 8) return launch<BF16, 4, 2>(w, st);
    if (chunks <= 12) return launch<BF16, 3, 4>(w, st);
    if (chunks <= 16) return launch<BF16, 4, 4>(w, st);
    if (chunks <= 24) return launch<BF16, 3, 8>(w, st);
    if (chunks <= 32) return launch<BF16, 4, 8>(w, st);
    if (chunks <= 48) return launch<BF16, 3, 16>(w, st);
    if (chunks <= 64) return launch<BF16, 4, 16>(w, st);
    if (chunks <= 96) return launch<BF16, 3, 32>(w, st);
    if (chunks <= 128) return launch<BF16, 4, 32>(w, st);
    if constexpr (BF16) {
        // From 8 M channels on, long groups of bf16 take half the lanes: what a lane does besides its channels (reductions,
        // barriers, the probes' bookkeeping) weighs as much as they do.  us, four chunks a lane and eight: 16384 x 4096 73.0 and
        // 64.6, 16384 x 3072 64.2 and 48.8, 4096 x 2048 11.7 and 10.7, 2048 x 4096 12.0 and 11.1; 2048 x 2048 7.7 and 8.4, 1024 x
        // 4096 7.8 and 8.8 (too few warps); groups of up to 1024 gain nothing (18464 x 768 at 128 19.5 and 20.9, at 768 17.8 and 17.5).
        if (w.a.total_groups * w.a.g >= ((int64_t)1 << 23)) {
            if (chunks <= 192) return launch<BF16, 6, 32>(w, st);
            if (chunks <= 256) return launch<BF16, 8, 32>(w, st);
            if (chunks <= 384) return launch<BF16, 6, 32, 2>(w, st);
            return launch<BF16, 8, 32, 2>(w, st);
        }
    }
    if (chunks <= 192) return launch<BF16, 3, 32, 2>(w, st);
    if (chunks <= 256) return launch<BF16, 4, 32, 2>(w, st);
    if (chunks <= 384) return launch<BF16, 3, 32, 4>(w, st);
    return launch<BF16, 4, 32, 4>(w, st);
}

// Where the k-th smallest of g standard normal magnitudes lies (only the first probe of the search: any value is right).
float gaussian_quantile(int k, int g) {
    const float f = ((float)k - 0.5f) / (float)g;
    return 1.2533f * f * (1.0f + 0.26f * f * f) / (1.0f - 0.45f * f * f * f * f);
}

}  // namespace

bool act_wide_ok(const ActArgs& a) {
    return a.g % 8 == 0 && a.g <= 4096 && reinterpret_cast<uintptr_t>(a.codes) % 4 == 0 && a.total_groups < ((int64_t)1 << 32);
}

cudaError_t launch_act_wide(const ActArgs& a, bool bf16, cudaStream_t st) {
    WideArgs w;
    w.a = a;
    const int64_t esz = bf16 ? 2 : 4;
    const uintptr_t base = reinterpret_cast<uintptr_t>(a.x);
    const int64_t pitch = a.row_stride * esz;
    w.load_mode = (base % 16 == 0 && pitch % 16 == 0) ? 0 : (base % 4 == 0 && pitch % 4 == 0) ? 1 : 2;
    w.guess_zr = gaussian_quantile(a.k_zr, a.g);
    w.guess_base = gaussian_quantile(a.k_base, a.g);
    return bf16 ? pick<true>(w, st) : pick<false>(w, st);
}

}  // namespace tdq
