// Device-side building blocks shared by the GranQ kernels: ordered keys for min/max,
// the per-element quantizer arithmetic, 128-bit element packs, fast integer division and
// the warp-level run accumulator of the range reduction.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace granq {

// ---------------------------------------------------------------------------------------
// Ordered keys.  enc() maps a float to an unsigned integer with the same ordering, so an
// unsigned max over enc(x) is the float max and an unsigned max over ~enc(x) is the float
// min.  0 is the identity of both reductions (no finite float encodes to 0 or ~0).
// ---------------------------------------------------------------------------------------
__host__ __device__ __forceinline__ uint32_t enc_bits(uint32_t b) {
    return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ uint32_t enc(float f) { return enc_bits(__float_as_uint(f)); }
__device__ __forceinline__ float dec(uint32_t k) {
    uint32_t b = (k & 0x80000000u) ? (k ^ 0x80000000u) : ~k;
    return __uint_as_float(b);
}
// key pair -> (lo, hi), with -0 canonicalised to +0
__device__ __forceinline__ void keys_to_range(uint32_t kmin, uint32_t kmax, float& lo, float& hi) {
    lo = __fadd_rn(dec(~kmin), 0.0f);
    hi = __fadd_rn(dec(kmax), 0.0f);
}

// ---------------------------------------------------------------------------------------
// Quantizer arithmetic (Eq. 1, 2, 5, 6).  Every operation is an explicitly rounded fp32
// intrinsic, so the compiler can neither contract multiply-adds nor replace the divisions.
// ---------------------------------------------------------------------------------------
struct QParam {
    float s, z;
};

__device__ __forceinline__ QParam make_qparam(float lo, float hi, float qmax) {
    QParam p;
    float s = __fdiv_rn(__fsub_rn(hi, lo), qmax);
    p.s = fmaxf(s, 1e-8f);
    p.z = __fadd_rn(rintf(__fdiv_rn(-lo, p.s)), 0.0f);
    return p;
}

// Given t = x / s: rounds u = t + z to the nearest integer (ties to even) and clamps it to
// [0, qmax].  The value is first clamped to [-1, qmax + 1]: rounding is monotone and the
// bounds are integers, so this changes neither the clamped code nor whether the clamp was
// active, and it makes the add/subtract of 1.5 * 2^23 an exact round-half-to-even
// (|u| < 2^22) that never yields -0.
__device__ __forceinline__ float quant_from_quotient(float t, float s, float z, float qmax, float& y, bool& inside) {
    const float kMagic = 12582912.0f;  // 1.5 * 2^23
    float u = __fadd_rn(t, z);
    float uc = fminf(fmaxf(u, -1.0f), __fadd_rn(qmax, 1.0f));
    float r = __fsub_rn(__fadd_rn(uc, kMagic), kMagic);
    float q = fminf(fmaxf(r, 0.0f), qmax);
    inside = (r == q);
    y = __fmul_rn(s, __fsub_rn(q, z));
    return q;
}

__device__ __forceinline__ float quant_one(float x, QParam p, float qmax, float& y, bool& inside) {
    return quant_from_quotient(__fdiv_rn(x, p.s), p.s, p.z, qmax, y, inside);
}

// Correctly rounded x / s from the correctly rounded reciprocal rcp = RN(1 / s): a product
// and two residual corrections, each residual x - q * s being exact in one fused
// multiply-add.  After the first correction q is a faithful rounding of x / s; a further
// correction of a faithful quotient with a correctly rounded reciprocal gives RN(x / s)
// (Markstein's division theorem), provided nothing over- or underflows on the way.
// div_is_safe() states the range for which that holds; groups outside it use __fdiv_rn.
__device__ __forceinline__ float div_by_scale(float x, float s, float rcp) {
    float q = __fmul_rn(x, rcp);
    float e = __fmaf_rn(-q, s, x);
    q = __fmaf_rn(e, rcp, q);
    e = __fmaf_rn(-q, s, x);
    return __fmaf_rn(e, rcp, q);
}
// s and every |x| of the group within [2^-60, 2^60] (x may also be tiny or zero: a quotient
// below 2^-120 cannot move u = x / s + z across a rounding boundary).
__device__ __forceinline__ bool div_is_safe(float s, float lo, float hi) {
    const float kBig = 1152921504606846976.0f;       // 2^60
    const float kSmall = 8.67361737988403547e-19f;   // 2^-60
    return s >= kSmall && s <= kBig && fmaxf(fabsf(lo), fabsf(hi)) <= kBig;
}

// ---------------------------------------------------------------------------------------
// 16-byte packs of elements.
// ---------------------------------------------------------------------------------------
template <typename T>
struct Pack;

template <>
struct Pack<float> {
    static constexpr int V = 4;
    uint4 raw;
    __device__ __forceinline__ float get(int i) const { return __uint_as_float((&raw.x)[i]); }
    __device__ __forceinline__ void set(int i, float v) { (&raw.x)[i] = __float_as_uint(v); }
    __device__ __forceinline__ void set_all(const float (&v)[4]) {
        raw = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
    }
    // element i of g where bit i of `keep` is set, +0 elsewhere (the straight-through gradient)
    __device__ __forceinline__ void select(const Pack& g, uint32_t keep) {
        raw.x = (keep & 1u) ? g.raw.x : 0u;
        raw.y = (keep & 2u) ? g.raw.y : 0u;
        raw.z = (keep & 4u) ? g.raw.z : 0u;
        raw.w = (keep & 8u) ? g.raw.w : 0u;
    }
};

template <>
struct Pack<__nv_bfloat16> {
    static constexpr int V = 8;
    uint4 raw;
    __device__ __forceinline__ float get(int i) const {
        uint32_t w = (&raw.x)[i >> 1];
        uint32_t b = (i & 1) ? (w & 0xFFFF0000u) : (w << 16);
        return __uint_as_float(b);
    }
    __device__ __forceinline__ void set(int i, float v) {
        uint32_t h = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v));
        uint32_t& w = (&raw.x)[i >> 1];
        w = (i & 1) ? ((w & 0x0000FFFFu) | (h << 16)) : ((w & 0xFFFF0000u) | h);
    }
    // eight floats -> eight bf16 (round to nearest even), two per conversion instruction
    __device__ __forceinline__ void set_all(const float (&v)[8]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);      // .x, the low half, = the first
            (&raw.x)[k] = *reinterpret_cast<const uint32_t*>(&h);
        }
    }
    // element i of g where bit i of `keep` is set, +0 elsewhere: on the raw halves, nothing is converted
    __device__ __forceinline__ void select(const Pack& g, uint32_t keep) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t m = ((keep >> (2 * k)) & 1u ? 0x0000FFFFu : 0u) | ((keep >> (2 * k + 1)) & 1u ? 0xFFFF0000u : 0u);
            (&raw.x)[k] = (&g.raw.x)[k] & m;
        }
    }
};

__device__ __forceinline__ float load_scalar(const float* p) { return __ldg(p); }
__device__ __forceinline__ float load_scalar(const __nv_bfloat16* p) {
    return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p)) << 16);
}
__device__ __forceinline__ void store_scalar(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_scalar(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// streaming 128-bit global accesses: data that is touched once should not displace anything
__device__ __forceinline__ uint4 ld_stream_16(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream_16(void* p, uint4 v) {
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// ---------------------------------------------------------------------------------------
// Division of n < 2^31 by a run-time constant d (1 <= d < 2^31): q = (n * M) >> (31 + l)
// with l = ceil(log2 d), M = floor(2^(31+l) / d) + 1.
// ---------------------------------------------------------------------------------------
struct FastDiv {
    uint32_t d, M, sh;
    __host__ __device__ __forceinline__ uint32_t div(uint32_t n) const {
        return (uint32_t)(((uint64_t)n * (uint64_t)M) >> sh);
    }
    __host__ __device__ __forceinline__ void divmod(uint32_t n, uint32_t& q, uint32_t& r) const {
        q = div(n);
        r = n - q * d;
    }
};

inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f;
    f.d = d;
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    f.M = (uint32_t)(((1ull << (31 + l)) / d) + 1ull);
    f.sh = 31 + l;
    return f;
}

constexpr uint32_t kNoGroup = 0xFFFFFFFFu;
constexpr uint32_t kFullMask = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------------------
// Warp-level run accumulator for per-group min/max (Eq. 4).
// A warp walks memory in order, so the group of its elements changes rarely.  While all
// lanes see the same group the partial min/max stay in registers; a change of group (or
// a warp that straddles several groups) is resolved with warp reductions on the ordered
// keys and one pair of atomics per group.
// ---------------------------------------------------------------------------------------
struct WarpRun {
    uint32_t g, kmn, kmx;
};

__device__ __forceinline__ void run_flush(WarpRun& r, uint32_t* kmin, uint32_t* kmax) {
    if (r.g != kNoGroup) {
        uint32_t a = __reduce_max_sync(kFullMask, r.kmn);
        uint32_t b = __reduce_max_sync(kFullMask, r.kmx);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(kmin + r.g, a);
            atomicMax(kmax + r.g, b);
        }
    }
    r.g = kNoGroup;
    r.kmn = 0;
    r.kmx = 0;
}

// must be called by all 32 lanes of a warp
__device__ __forceinline__ void run_add(WarpRun& r, bool valid, uint32_t g, uint32_t mn, uint32_t mx,
                                        uint32_t* kmin, uint32_t* kmax) {
    uint32_t pending = __ballot_sync(kFullMask, valid);
    if (!pending) return;
    const int lane = threadIdx.x & 31;
    uint32_t first = __shfl_sync(kFullMask, g, __ffs(pending) - 1);
    bool uniform = __all_sync(kFullMask, !valid || g == first);
    if (!valid) {
        mn = 0;
        mx = 0;
    }
    if (uniform) {
        if (first != r.g) {
            run_flush(r, kmin, kmax);
            r.g = first;
        }
        r.kmn = max(r.kmn, mn);
        r.kmx = max(r.kmx, mx);
        return;
    }
    run_flush(r, kmin, kmax);
    while (pending) {
        int src = __ffs(pending) - 1;
        uint32_t cur = __shfl_sync(kFullMask, g, src);
        bool mine = valid && g == cur;
        uint32_t a = __reduce_max_sync(kFullMask, mine ? mn : 0u);
        uint32_t b = __reduce_max_sync(kFullMask, mine ? mx : 0u);
        if (lane == src) {
            atomicMax(kmin + cur, a);
            atomicMax(kmax + cur, b);
        }
        pending &= ~__ballot_sync(kFullMask, mine);
    }
}

// A 16-byte unit from global to shared memory (both aligned), past the L1, without waiting; without an L2 policy, which is worth nothing
// here and is under suspicion on this instruction (granq_colteam.cu).
__device__ __forceinline__ void cp_async_16(void* dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src)
                 : "memory");
}
// a word that another CTA released
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The kernel behind this one in the stream may be set up; it waits for this one's end, memory included, by itself.
__device__ __forceinline__ void let_the_kernel_behind_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The kernel ahead in the stream has completed and its memory is there.
__device__ __forceinline__ void wait_for_the_kernel_ahead() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// First thing in a kernel launched by launch_after(): the kernel ahead of it in the stream has completed and its memory is
// there; the kernel behind it may be set up (it waits in the same way).
__device__ __forceinline__ void after_the_kernel_ahead() {
    wait_for_the_kernel_ahead();
    let_the_kernel_behind_start();
}

// ---------------------------------------------------------------------------------------
// Per-group parameters, and the arithmetic of one pack.
// ---------------------------------------------------------------------------------------
struct GroupParam {
    float s, z, r;   // scale, zero-point, RN(1 / s) or 0 when the group must use IEEE division
    float thr;       // tie threshold of the single-multiply-add rounding below: positive where no element can be
                     // clamped, negative where the clamp is needed, 0: the sequence as defined
};

constexpr float kRoundMagic = 12582912.0f;               // 1.5 * 2^23: adding it rounds to an integer, ties to even
constexpr uint32_t kRoundMagicBits = 0x4B400000u;

// The rounded value r = round(x / s + z) from ONE fused multiply-add, where that is provably the same integer.
// Only r enters the results (code = clamp(r), y = s * (code - z), mask = (r == code)); the quotient and the sum
// are intermediates.  z is an integer, so with |z| <= 2^20 the constant mz = 1.5 * 2^23 + z is exact, and
//     m = fma(x, RN(1 / s), mz)
// is 1.5 * 2^23 + (x * RN(1 / s) + z rounded to an integer, ties to even): its low mantissa bits are the code, and
// t = m - mz = code - z is exact, so that y = s * t.  Bound: let w = x * RN(1 / s), v = x / s,
// u = RN(RN(v) + z) the sum as defined.  |w - v| and |RN(v) - v| are at most 2^-24 |v|, |u - (RN(v) + z)| at most
// 2^-24 (|u| + 1), and where the clamp does not decide, |v| <= |z| + qmax + 2 and |u| <= qmax + 2: u and w + z differ
// by at most 2^-24 (2 |z| + 3 qmax + 7).  d = fma(x, RN(1 / s), -t) is w - t up to 2^-26.  So |d| below
//     thr = 0.5 - 2^-23 (|z| + 1.5 qmax + 4)
// puts u less than 0.5 away from the integer t + z: round(u) = t + z.  An element that fails the test takes the
// sequence as defined (one in 3e5 at 4 bits, one in 1e4 at 8).  Values beyond [-2, qmax + 2] clamp alike either way.
__device__ __forceinline__ float tie_threshold(float rcp, float z, float qmax) {
    if (rcp == 0.0f || !(fabsf(z) <= 1048576.0f)) return 0.0f;
    return __fmaf_rn(-1.1920928955078125e-07f, __fadd_rn(fabsf(z), __fmaf_rn(1.5f, qmax, 4.0f)), 0.5f);
}

// the larger of two values, NaN if either is (fmaxf drops it)
__device__ __forceinline__ float max_or_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// u = x / s + z as defined, rounded: 1.5 * 2^23 + clamp(round(u), -1, qmax + 1), given the quotient t = RN(x / s)
__device__ __forceinline__ float exact_round_magic(float t, float z, float qmax) {
    const float u = __fadd_rn(t, z);
    return __fadd_rn(fminf(fmaxf(u, -1.0f), __fadd_rn(qmax, 1.0f)), kRoundMagic);
}

// Parameters of a group whose range (lo, hi) is that of the tensor itself.  thr is positive only where no element
// of the group is clamped: rounding is monotone in x, so it is enough that neither lo nor hi is.  (lo never is:
// z = round(RN(-lo / s)), so u(lo) lies within [-0.5, 0.5] and rounds to 0; hi is where u(hi) reaches qmax + 0.5,
// a tie of lo / s, as in a range with lo = -hi.)  In such a group every mask bit is set and gx = gy.
__device__ __forceinline__ GroupParam group_param_from_range(float lo, float hi, float qmax) {
    const QParam p = make_qparam(lo, hi, qmax);
    GroupParam gp;
    gp.s = p.s;
    gp.z = p.z;
    gp.r = div_is_safe(p.s, lo, hi) ? __frcp_rn(p.s) : 0.0f;
    gp.thr = tie_threshold(gp.r, gp.z, qmax);
    const float rl = exact_round_magic(div_by_scale(lo, gp.s, gp.r), gp.z, qmax);
    const float rh = exact_round_magic(div_by_scale(hi, gp.s, gp.r), gp.z, qmax);
    if (!(rl >= kRoundMagic && rh <= __fadd_rn(kRoundMagic, qmax))) gp.thr = -gp.thr;
    return gp;
}
__device__ __forceinline__ GroupParam group_param_from_keys(const uint32_t* kmin, const uint32_t* kmax, uint32_t g,
                                                            float qmax, float& lo, float& hi) {
    keys_to_range(__ldcg(kmin + g), __ldcg(kmax + g), lo, hi);
    return group_param_from_range(lo, hi, qmax);
}

template <int H>
struct PartAt {
    static constexpr int value = H;
};

// Clamp the rounded values m[H .. H + W) = 1.5 * 2^23 + r to codes.  The bits of `in` of elements that were beyond: taken
// out (where a clamp is the exception, `in` starts full), or the others put in (where it is the rule, from none).
template <int H, int W, bool RULE, int V>
__device__ __forceinline__ void clamp_codes(float (&m)[V], float top, uint32_t& in) {
#pragma unroll
    for (int i = H; i < H + W; ++i) {
        const float c = fminf(fmaxf(m[i], kRoundMagic), top);
        if (RULE) in |= (m[i] == c) ? (1u << i) : 0u;
        else in &= (m[i] == c) ? 0xFFFFFFFFu : ~(1u << i);
        m[i] = c;
    }
}

// What the extra outputs of one pack are made of (EXTRAS as in quantize_pack): bytes of codes and mask (1), mask
// bits (2), strings of code_bits per code (3).  m: 1.5 * 2^23 + code of element i, in: the clamp was inactive.
template <int V, int EXTRAS>
__device__ __forceinline__ void pack_extras(const float (&m)[V], uint32_t in, uint32_t (&cb)[V / 4],
                                            uint32_t (&mb)[V / 4], int code_bits) {
#pragma unroll
    for (int h = 0; h < V / 4; ++h) {
        cb[h] = 0;
        mb[h] = 0;
    }
    if constexpr (EXTRAS == 1 || EXTRAS == 3) {
        // sum of (magic bits + code) << shift, less the magic bits' share: one multiply-add per code
        const uint32_t b = EXTRAS == 3 ? (uint32_t)code_bits : 8u;
        const uint32_t m1 = 1u << b, m2 = 1u << (2 * b), m3 = 1u << (3 * b);
        const uint32_t off = kRoundMagicBits * (1u + m1 + m2 + m3);
#pragma unroll
        for (int h = 0; h < V / 4; ++h)
            cb[h] = __float_as_uint(m[4 * h]) + __float_as_uint(m[4 * h + 1]) * m1 + __float_as_uint(m[4 * h + 2]) * m2 +
                    __float_as_uint(m[4 * h + 3]) * m3 - off;
    }
    if constexpr (EXTRAS == 1) {
#pragma unroll
        for (int i = 0; i < V; ++i) mb[i / 4] |= ((in >> i) & 1u) << (8 * (i % 4));
    } else if constexpr (EXTRAS == 2) {
        mb[0] = in;
    }
}

// Quantize one pack: elements [0, n1) belong to the group with parameters g1, the rest to
// g2 (n1 = V when the pack lies in one group).  EXTRAS = 1 also packs the codes and the mask
// (one byte per element); EXTRAS = 2 leaves the codes out and returns the mask as V bits in mb[0]
// (bit i: the clamp was inactive for element i), which is all the packed mask needs; EXTRAS = 3 returns
// only the codes, code_bits each (cb[h] = the four codes of half h as a string of 4 * code_bits bits; bytes for
// the default of 8), taken from the low mantissa bits of code + 1.5 * 2^23 instead of a float-to-integer
// conversion (packed-code output); EXTRAS = 4 returns neither (the caller adds up the distortion).  SELF: the range is
// that of the tensor itself and thr comes from group_param_from_range(), so where it is positive nothing is clamped and the
// gradient passes whole; without SELF it comes from tie_threshold() alone and x may lie anywhere.  A NaN element takes the
// clamp - without SELF it always does, with it the tie test fails - and becomes code 0 without a gradient, as in the
// sequence as defined, whatever its neighbours are.  PARTS: see W.
// Instructions per element, bf16 or fp32 alike: two multiply-adds, one add, half a three-way maximum and one
// product (SELF), where rounding by add and subtract, clamp, compare and select took eleven.  Measured against that
// form: forward-only bf16 [256,512,28,28] at 8 bits 127.6 -> 119.6 us (issue slots bind where an element is two
// bytes), packed codes of fp32 [128,144,56,56] 150 -> 142 us, packed mask of [128,64,56,56] 63.0 -> 60.6 us.
template <typename T, bool BWD, bool SPLIT, int EXTRAS, bool SELF = false, bool PARTS = true>
__device__ __forceinline__ void quantize_pack(const Pack<T>& px, const Pack<T>& pg, const GroupParam& g1,
                                              const GroupParam& g2, int n1, float qmax, Pack<T>& py, Pack<T>& pgx,
                                              uint32_t (&cb)[Pack<T>::V / 4], uint32_t (&mb)[Pack<T>::V / 4],
                                              int code_bits = 8) {
    constexpr int V = Pack<T>::V;
    // Elements worked on together.  Eight at a time, with the two sets of parameters of a pack that straddles groups or
    // with the clamp in the main line, take 74 to 99 registers in kernels that want 64: bf16 then takes four at a time.
    constexpr int W = (V == 8 && PARTS && (SPLIT || !SELF)) ? 4 : V;
    // ... and the elements that miss the shortcut share their branch with the groups that have none
    constexpr bool kOneBranch = !SELF && W < V;
    float m[V], yv[V];
    uint32_t in = SELF ? (1u << V) - 1u : 0u;                   // bit i: the clamp was inactive for element i
    const float thr = SPLIT ? fminf(fabsf(g1.thr), fabsf(g2.thr)) : fabsf(g1.thr);
    const float top = __fadd_rn(kRoundMagic, qmax);
    if (kOneBranch || thr > 0.0f) {
        const float mz1 = __fadd_rn(kRoundMagic, g1.z), mz2 = SPLIT ? __fadd_rn(kRoundMagic, g2.z) : mz1;
        auto part = [&](auto at) {
            constexpr int H = decltype(at)::value;
            float worst = 0.0f;
#pragma unroll
            for (int i = H; i < H + W; ++i) {
                const bool first = !SPLIT || i < n1;
                const float rc = first ? g1.r : g2.r, mz = first ? mz1 : mz2;
                const float x = px.get(i);
                m[i] = __fmaf_rn(x, rc, mz);
                const float d = fabsf(__fmaf_rn(x, rc, __fsub_rn(mz, m[i])));
                worst = SELF ? max_or_nan(worst, d) : fmaxf(worst, d);
            }
            bool clamp = !SELF || g1.thr < 0.0f || (SPLIT && g2.thr < 0.0f);
            if (!(worst < thr)) {                               // rare: too close to a tie for the shortcut, or NaN
#pragma unroll
                for (int i = H; i < H + W; ++i) {
                    const bool first = !SPLIT || i < n1;
                    const float s = first ? g1.s : g2.s, z = first ? g1.z : g2.z, rc = first ? g1.r : g2.r;
                    const float mz = first ? mz1 : mz2, x = px.get(i);
                    if (!(fabsf(__fmaf_rn(x, rc, __fsub_rn(mz, m[i]))) < thr))
                        m[i] = exact_round_magic(SELF ? div_by_scale(x, s, rc) : __fdiv_rn(x, s), z, qmax);
                }
                // NaN: in a place of its own, so that the condition below stays one that the walk around this need not look
                // at again ([256,960,7,7] fp32 with a gradient 50.9 -> 47.0 us); beside byte codes it is the other way
                // round (54.9 / 61.2)
                if constexpr (SELF && W == V && EXTRAS != 1) {
                    if (worst != worst) clamp_codes<H, W, !SELF>(m, top, in);
                } else if constexpr (SELF) {
                    clamp = clamp || worst != worst;
                }
            }
            if (clamp) clamp_codes<H, W, !SELF>(m, top, in);
            if (!kOneBranch || thr > 0.0f) {
#pragma unroll
                for (int i = H; i < H + W; ++i) {
                    const bool first = !SPLIT || i < n1;
                    yv[i] = __fmul_rn(first ? g1.s : g2.s, __fsub_rn(m[i], first ? mz1 : mz2));
                }
            } else {                                            // the zero-point may be too large for mz
#pragma unroll
                for (int i = H; i < H + W; ++i) {
                    const bool first = !SPLIT || i < n1;
                    yv[i] = __fmul_rn(first ? g1.s : g2.s, __fsub_rn(__fsub_rn(m[i], kRoundMagic), first ? g1.z : g2.z));
                }
            }
        };
        part(PartAt<0>{});
        if constexpr (W < V) part(PartAt<W>{});
    } else {                                                    // the sequence as defined, element by element
        in = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const bool first = !SPLIT || i < n1;
            const float s = first ? g1.s : g2.s, z = first ? g1.z : g2.z;
            const float r = exact_round_magic(__fdiv_rn(px.get(i), s), z, qmax);
            m[i] = fminf(fmaxf(r, kRoundMagic), top);
            in |= (m[i] == r) ? (1u << i) : 0u;
            yv[i] = __fmul_rn(s, __fsub_rn(__fsub_rn(m[i], kRoundMagic), z));
        }
    }
    if constexpr (BWD) pgx.select(pg, in);
    pack_extras<V, EXTRAS>(m, in, cb, mb, code_bits);
    py.set_all(yv);
}

// Two floats side by side: the fp32 pipe takes both with one instruction (fma, add, multiply; each rounded as its scalar
// form), which is half the issue slots.
struct F2 {
    uint64_t v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_split(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// Quantize one fp32 pack of one group whose range is that of the tensor itself (thr from group_param_from_range()); bf16 goes
// on to quantize_pack(), which also says what the outputs are.  In the main line nothing is clamped and the gradient passes
// whole: w = fma(x, 1 / s, mz) rounds, e = mz - w = -(code - z) exactly, fma(x, 1 / s, e) is the distance from the integer,
// and y = s * (code - z) is fma(-s, e, +0), whose +0 keeps a zero from coming out as -0: four packed instructions for two
// elements.  A pack with an element too close to a tie or a NaN (which becomes code 0 without a gradient, as in the sequence
// as defined), or of a group without a shortcut, is worked out again element by element; groups that may be clamped clamp.
// Against the scalar form, geometric mean over 26 shapes: forward 0.98, with sums 0.98, weights 0.96 of the time.  bf16, whose
// elements have to be moved into pairs of registers first, is 3 to 10 % slower this way.
template <typename T, bool BWD, int EXTRAS>
__device__ __forceinline__ void quantize_own(const Pack<T>& px, const Pack<T>& pg, const GroupParam& g, float qmax, Pack<T>& py,
                                             Pack<T>& pgx, uint32_t (&cb)[Pack<T>::V / 4], uint32_t (&mb)[Pack<T>::V / 4],
                                             int code_bits = 8) {
    constexpr int V = Pack<T>::V;
    if constexpr (V == 8) {
        quantize_pack<T, BWD, false, EXTRAS, true>(px, pg, g, g, V, qmax, py, pgx, cb, mb, code_bits);
    } else {
        const float mz = __fadd_rn(kRoundMagic, g.z), top = __fadd_rn(kRoundMagic, qmax);
        const F2 r2 = f2(g.r, g.r), mz2 = f2(mz, mz), ns2 = f2(-g.s, -g.s), zero = {0};
        float m[V], yv[V], worst = 0.0f;
        uint32_t in = (1u << V) - 1u;
#pragma unroll
        for (int k = 0; k < V; k += 2) {
            const F2 x = f2(px.get(k), px.get(k + 1)), w = f2_fma(x, r2, mz2), e = f2_sub(mz2, w);
            float d0, d1;
            f2_split(f2_fma(x, r2, e), d0, d1);
            worst = max_or_nan(max_or_nan(worst, fabsf(d0)), fabsf(d1));
            f2_split(f2_fma(ns2, e, zero), yv[k], yv[k + 1]);
            f2_split(w, m[k], m[k + 1]);
        }
        if constexpr (BWD) pgx.raw = pg.raw;
        if (!(worst < fabsf(g.thr))) {
            in = 0;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const float x = px.get(i);
                float r = __fmaf_rn(x, g.r, mz);
                if (g.thr == 0.0f) r = exact_round_magic(__fdiv_rn(x, g.s), g.z, qmax);
                else if (!(fabsf(__fmaf_rn(x, g.r, __fsub_rn(mz, r))) < fabsf(g.thr))) r = exact_round_magic(div_by_scale(x, g.s, g.r), g.z, qmax);
                m[i] = fminf(fmaxf(r, kRoundMagic), top);
                in |= (m[i] == r) ? (1u << i) : 0u;
                yv[i] = __fmul_rn(g.s, __fsub_rn(__fsub_rn(m[i], kRoundMagic), g.z));
            }
            if constexpr (BWD) pgx.select(pg, in);
        } else if (g.thr < 0.0f) {
            clamp_codes<0, V, false>(m, top, in);
#pragma unroll
            for (int k = 0; k < V; k += 2)
                f2_split(f2_fma(ns2, f2_sub(mz2, f2(m[k], m[k + 1])), zero), yv[k], yv[k + 1]);
            if constexpr (BWD) pgx.select(pg, in);
        }
        pack_extras<V, EXTRAS>(m, in, cb, mb, code_bits);
        py.set_all(yv);
    }
}

// Quantize one pack whose V elements belong to V different groups (channels-last rows), the range being the
// tensor's own: element i takes scale s[i], reciprocal r[i] and mz[i] = 1.5 * 2^23 + z; thr is the smallest of the
// V groups' thresholds in magnitude, negative when one of them is, and where it is 0 the parameters are read again
// from `par` (the zero-point may then be too large for mz).  Same arithmetic as quantize_pack<SELF>.
template <typename T, bool BWD, bool EXTRAS>
__device__ __forceinline__ void quantize_pack_each(const Pack<T>& px, const Pack<T>& pg, const float (&s)[Pack<T>::V],
                                                   const float (&r)[Pack<T>::V], const float (&mz)[Pack<T>::V],
                                                   float thr, const GroupParam* par, float qmax, Pack<T>& py,
                                                   Pack<T>& pgx, uint32_t (&cb)[Pack<T>::V / 4],
                                                   uint32_t (&mb)[Pack<T>::V / 4]) {
    constexpr int V = Pack<T>::V;
    float m[V], yv[V];
    uint32_t in = (1u << V) - 1u;
    const float bound = fabsf(thr), top = __fadd_rn(kRoundMagic, qmax);
    if (bound > 0.0f) {
        float worst = 0.0f;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const float x = px.get(i);
            m[i] = __fmaf_rn(x, r[i], mz[i]);
            worst = max_or_nan(worst, fabsf(__fmaf_rn(x, r[i], __fsub_rn(mz[i], m[i]))));
        }
        bool clamp = thr < 0.0f;
        if (!(worst < bound)) {                                   // rare: too close to a tie for the shortcut, or NaN
            clamp = clamp || worst != worst;                      // which the clamp turns into code 0 without a gradient
#pragma unroll
            for (int i = 0; i < V; ++i) {
                const float x = px.get(i);
                if (!(fabsf(__fmaf_rn(x, r[i], __fsub_rn(mz[i], m[i]))) < bound))
                    m[i] = exact_round_magic(div_by_scale(x, s[i], r[i]), __fsub_rn(mz[i], kRoundMagic), qmax);
            }
        }
        if (clamp) clamp_codes<0, V, false>(m, top, in);
#pragma unroll
        for (int i = 0; i < V; ++i) yv[i] = __fmul_rn(s[i], __fsub_rn(m[i], mz[i]));
    } else {                                                    // the sequence as defined, element by element
        in = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const GroupParam g = par[i];
            const float q = exact_round_magic(__fdiv_rn(px.get(i), g.s), g.z, qmax);
            m[i] = fminf(fmaxf(q, kRoundMagic), top);
            in |= (m[i] == q) ? (1u << i) : 0u;
            yv[i] = __fmul_rn(g.s, __fsub_rn(__fsub_rn(m[i], kRoundMagic), g.z));
        }
    }
    if constexpr (BWD) pgx.select(pg, in);
    pack_extras<V, EXTRAS ? 1 : 0>(m, in, cb, mb, 8);
    py.set_all(yv);
}

// Smallest and largest of any number of packs (NaN left out, as by fminf / fmaxf); two independent chains.
template <typename T>
struct RangeFold;
template <>
struct RangeFold<float> {
    float mn[2] = {INFINITY, INFINITY}, mx[2] = {-INFINITY, -INFINITY};
    __device__ __forceinline__ void add(const Pack<float>& p) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            mn[e & 1] = fminf(mn[e & 1], p.get(e));
            mx[e & 1] = fmaxf(mx[e & 1], p.get(e));
        }
    }
    __device__ __forceinline__ void result(float& lo, float& hi) const {
        lo = fminf(mn[0], mn[1]);
        hi = fmaxf(mx[0], mx[1]);
    }
};
// bf16 two at a time as they are stored: half an instruction per element and side, nothing to widen
template <>
struct RangeFold<__nv_bfloat16> {
    uint32_t mn[2] = {0x7F807F80u, 0x7F807F80u}, mx[2] = {0xFF80FF80u, 0xFF80FF80u};
    __device__ __forceinline__ static void min2(uint32_t& a, uint32_t b) { asm("min.bf16x2 %0, %0, %1;" : "+r"(a) : "r"(b)); }
    __device__ __forceinline__ static void max2(uint32_t& a, uint32_t b) { asm("max.bf16x2 %0, %0, %1;" : "+r"(a) : "r"(b)); }
    __device__ __forceinline__ void add(const Pack<__nv_bfloat16>& p) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            min2(mn[k & 1], (&p.raw.x)[k]);
            max2(mx[k & 1], (&p.raw.x)[k]);
        }
    }
    __device__ __forceinline__ void result(float& lo, float& hi) const {
        uint32_t a = mn[0], b = mx[0];
        min2(a, mn[1]);
        max2(b, mx[1]);
        lo = fminf(__uint_as_float(a << 16), __uint_as_float(a & 0xFFFF0000u));
        hi = fmaxf(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u));
    }
};

// Smallest and largest per element of a pack, over any number of packs: a unit column, whose element i belongs to the same
// channel all the way down.
template <typename T>
struct RangeColumn;
template <>
struct RangeColumn<float> {
    float mn[4], mx[4];
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mn[i] = INFINITY;
            mx[i] = -INFINITY;
        }
    }
    __device__ __forceinline__ void add(const Pack<float>& p) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mn[i] = fminf(mn[i], p.get(i));
            mx[i] = fmaxf(mx[i], p.get(i));
        }
    }
    __device__ __forceinline__ float lo(int i) const { return mn[i]; }
    __device__ __forceinline__ float hi(int i) const { return mx[i]; }
};
template <>
struct RangeColumn<__nv_bfloat16> {
    Pack<__nv_bfloat16> mn, mx;         // as they are stored, two to a word (RangeFold)
    __device__ __forceinline__ void reset() {
        mn.raw = make_uint4(0x7F807F80u, 0x7F807F80u, 0x7F807F80u, 0x7F807F80u);
        mx.raw = make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u);
    }
    __device__ __forceinline__ void add(const Pack<__nv_bfloat16>& p) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            RangeFold<__nv_bfloat16>::min2((&mn.raw.x)[k], (&p.raw.x)[k]);
            RangeFold<__nv_bfloat16>::max2((&mx.raw.x)[k], (&p.raw.x)[k]);
        }
    }
    __device__ __forceinline__ float lo(int i) const { return mn.get(i); }
    __device__ __forceinline__ float hi(int i) const { return mx.get(i); }
};
// ordered keys of elements [first, last) of a column; (0, 0) when that range is empty or nothing was added
template <typename T>
__device__ __forceinline__ void column_keys(const RangeColumn<T>& c, int first, int last, uint32_t& kmn, uint32_t& kmx) {
    float a = INFINITY, b = -INFINITY;
#pragma unroll
    for (int i = 0; i < Pack<T>::V; ++i) {
        if (i >= first && i < last) {
            a = fminf(a, c.lo(i));
            b = fmaxf(b, c.hi(i));
        }
    }
    kmn = (a <= b) ? ~enc(a) : 0u;
    kmx = (a <= b) ? enc(b) : 0u;
}

// per-lane min / max of elements [first, last) of one pack
template <typename T>
__device__ __forceinline__ void pack_minmax(const Pack<T>& p, int first, int last, float& mn, float& mx) {
#pragma unroll
    for (int i = 0; i < Pack<T>::V; ++i) {
        if (i >= first && i < last) {
            float v = p.get(i);
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
        }
    }
}

// The V mask bits of one pack, from the mask bytes of quantize_pack<EXTRAS = 1> or the bits of <EXTRAS = 2>.
template <int V, int EXTRAS>
__device__ __forceinline__ uint32_t mask_bits_of(const uint32_t (&mb)[V / 4]) {
    if constexpr (EXTRAS == 2) {
        return mb[0];
    } else {
        uint32_t bits = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) bits |= ((mb[i / 4] >> (8 * (i % 4))) & 1u) << i;
        return bits;
    }
}

// Masks and codes are written 8 elements at a time, which takes two neighbouring lanes of fp32 packs, and words of codes
// eight.  `lanes` are the lanes of the warp that are here, whole groups of them, and the same value in every lane: with a mask
// per group the warp goes through a shuffle group by group: 61 % of the time of the unit that takes it on, packed mask of
// [128,64,56,56] (the kernel alone, with what else follows here: 51.3 -> 41.9 us; 5-bit codes of [128,144,56,56] 83.9 -> 65.9, 4-bit codes of
// [128,256,14,14] 21.8 -> 18.0).
__device__ __forceinline__ uint32_t from_lane(uint32_t lanes, uint32_t v, uint32_t src) {
    return lanes == kFullMask ? __shfl_sync(kFullMask, v, (int)src) : __shfl_sync(lanes, v, (int)src);
}

// Store the packed mask one byte (8 elements) at a time: `bits` are the V mask bits of the pack that starts at
// element `first` (a multiple of V; for V = 4 the even lane of a pair holds the low half of a byte, and both
// lanes of the pair must call this together with neighbouring packs).
template <int V>
__device__ __forceinline__ void store_mask_byte(uint32_t* pmask, size_t first, uint32_t bits, uint32_t lane, uint32_t lanes) {
    if constexpr (V == 4) {
        const uint32_t other = from_lane(lanes, bits, lane ^ 1u);
        if (!(lane & 1)) reinterpret_cast<uint8_t*>(pmask)[first >> 3] = (uint8_t)(bits | (other << 4));
    } else {
        static_assert(V == 8, "a pack is 4 or 8 elements");
        reinterpret_cast<uint8_t*>(pmask)[first >> 3] = (uint8_t)bits;
    }
}

// The codes of one pack as a string of V * b bits, from the half strings of quantize_pack<EXTRAS = 3>(.., code_bits).
template <int V>
__device__ __forceinline__ uint64_t code_string_of(const uint32_t (&cb)[V / 4], int code_bits) {
    uint64_t str = cb[0];
    if constexpr (V == 8) str |= (uint64_t)cb[1] << (4 * code_bits);
    return str;
}

// b bytes: the codes of the elements 8 * eight ... of the bit string.  The buffer is only known to be 4-byte aligned.
__device__ __forceinline__ void store_eight_codes(uint32_t* pcodes, size_t eight, uint64_t str, int code_bits) {
    uint8_t* dst = reinterpret_cast<uint8_t*>(pcodes) + eight * (size_t)code_bits;
    switch (code_bits) {
        case 8:
            reinterpret_cast<uint32_t*>(dst)[0] = (uint32_t)str;
            reinterpret_cast<uint32_t*>(dst)[1] = (uint32_t)(str >> 32);
            break;
        case 4: *reinterpret_cast<uint32_t*>(dst) = (uint32_t)str; break;
        case 2: *reinterpret_cast<uint16_t*>(dst) = (uint16_t)str; break;
        case 6:
            reinterpret_cast<uint16_t*>(dst)[0] = (uint16_t)str;
            reinterpret_cast<uint16_t*>(dst)[1] = (uint16_t)(str >> 16);
            reinterpret_cast<uint16_t*>(dst)[2] = (uint16_t)(str >> 32);
            break;
        default:
            for (int t = 0; t < code_bits; ++t) dst[t] = (uint8_t)(str >> (8 * t));
            break;
    }
}

// Store the packed codes 8 codes = b bytes at a time: `str` is the code string of the pack that starts at element
// `first` (a multiple of V).  For V = 4 the even lane of a pair holds the first half and stores; both lanes of the pair must
// call this together with neighbouring packs.
template <int V>
__device__ __forceinline__ void store_code_bytes(uint32_t* pcodes, size_t first, uint64_t str, int code_bits, uint32_t lane, uint32_t lanes) {
    uint64_t eight = str;
    if constexpr (V == 4) {
        const uint32_t other = from_lane(lanes, (uint32_t)str, lane ^ 1u);
        if (lane & 1) return;
        eight |= (uint64_t)other << (4 * code_bits);
    }
    store_eight_codes(pcodes, first >> 3, eight, code_bits);
}

// Two fp32 packs of every lane of a warp at once: the strings s0 and s1 (4 * b bits) of this lane's packs, the lane beside it
// holding their neighbours.  The even lane of a pair leaves with the eight codes of the first, the odd lane with those of the
// second: one shuffle and, behind it, one store for two packs of a lane.
__device__ __forceinline__ uint64_t pair_up_codes(uint32_t s0, uint32_t s1, int code_bits, uint32_t lane) {
    const bool odd = lane & 1u;
    const uint32_t got = __shfl_xor_sync(kFullMask, odd ? s0 : s1, 1);
    return (odd ? got : s0) | ((uint64_t)(odd ? s1 : got) << (4 * code_bits));
}
// The same for the mask: 4 bits of each of U packs, U / 2 bytes of every lane for one shuffle, byte k that of pack 2 k (even lane)
// or 2 k + 1 (odd lane).
template <int U>
__device__ __forceinline__ uint32_t pair_up_mask(const uint32_t (&bits)[U], uint32_t lane) {
    static_assert(U == 2 || U == 4, "one byte or two of every lane");
    const uint32_t a = U == 4 ? bits[0] | (bits[U - 2] << 8) : bits[0], b = U == 4 ? bits[1] | (bits[U - 1] << 8) : bits[1];
    const bool odd = lane & 1u;
    const uint32_t got = __shfl_xor_sync(kFullMask, odd ? a : b, 1);
    return (odd ? got : a) | ((odd ? b : got) << 4);
}

// Store the codes of 8 elements per lane as whole words: four lanes, STRIDE apart, hold 32 consecutive codes = BITS whole words
// of the bit string, the first of them an element whose index is a multiple of 32 (q: which of the four this lane is).  Strings
// of 3 bytes: word q is this lane's string and the next one's; of 5 to 7 bytes: a lane completes the word its string begins in with
// the end of the string before, and adds the word that its own string may hold besides.  One shuffle and one or two coalesced
// stores in place of BITS single bytes, each of which rewrote part of a sector in the L2.  The whole warp must call.  Codes and their
// expansion, us: fp32 [128,144,56,56] at 3, 5, 8 bits 135 -> 109, 125 -> 109, 125 -> 115; bf16, whose bytes were no slower, 72 / 72, 85 / 83.
template <int BITS, int STRIDE>
__device__ __forceinline__ void store_code_words(uint32_t* pcodes, size_t eight, uint64_t str, uint32_t q, uint32_t lane) {
    uint32_t* dst = pcodes + (eight >> 2) * (size_t)BITS;
    if constexpr (BITS == 3) {
        const uint32_t next = __shfl_sync(kFullMask, (uint32_t)str, (int)((lane + STRIDE) & 31u));
        if (q < 3) dst[q] = __funnelshift_r((uint32_t)str | (next << 24), next >> 8, 8 * q);
    } else if constexpr (BITS > 4 && BITS < 8) {
        const uint32_t before = __shfl_sync(kFullMask, (uint32_t)(str >> (8 * BITS - 32)), (int)((lane - STRIDE) & 31u));
        const uint32_t at = (8 * BITS * q) & 31u, k = (BITS * q) >> 2;      // where the string begins
        dst[k] = __funnelshift_l(before, (uint32_t)str, at);
        if (8 * BITS - 32 + at >= 32) dst[k + 1] = (uint32_t)(str >> (32u - at));
    } else {
        store_eight_codes(pcodes, eight, str, BITS);
    }
}

// ---------------------------------------------------------------------------------------
// Distortion statistics of a quantization (Section 4.1, Table 2): sum x^2, sum q^2, sum x*q,
// sum (x - q)^2.  The terms of one pack are summed in fp32 (fused multiply-adds), everything
// beyond a pack in fp64, so a sum differs from the exact one by at most a few fp32 roundings
// of a pack-sized partial sum.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float as_stored(float v, const float*) { return v; }
__device__ __forceinline__ float as_stored(float v, const __nv_bfloat16*) {
    return __bfloat162float(__float2bfloat16_rn(v));
}

struct DistAcc {
    double xx, qq, xq, dd;
    __device__ __forceinline__ void reset() { xx = qq = xq = dd = 0.0; }
    __device__ __forceinline__ void add_one(float x, float q) {
        const float d = __fsub_rn(x, q);
        xx += (double)__fmul_rn(x, x);
        qq += (double)__fmul_rn(q, q);
        xq += (double)__fmul_rn(x, q);
        dd += (double)__fmul_rn(d, d);
    }
    template <typename T>
    __device__ __forceinline__ void add(const Pack<T>& px, const Pack<T>& pq) {
        float a = 0.0f, b = 0.0f, c = 0.0f, e = 0.0f;
#pragma unroll
        for (int i = 0; i < Pack<T>::V; ++i) {
            const float x = px.get(i), q = pq.get(i), d = __fsub_rn(x, q);
            a = __fmaf_rn(x, x, a);
            b = __fmaf_rn(q, q, b);
            c = __fmaf_rn(x, q, c);
            e = __fmaf_rn(d, d, e);
        }
        xx += (double)a;
        qq += (double)b;
        xq += (double)c;
        dd += (double)e;
    }
    // must be called by every thread of the block, once: one atomic per block and sum.  The four sums share a sector,
    // and atomics on one sector are served one after the other, about 1.4 ns each: with one per warp they took
    // longer than everything else (layer-wise [128,128,28,28]: 69.6 us of kernel for 38 000 of them, now 21 us).
    __device__ __forceinline__ void flush(double* out) {
        __shared__ double part[32][4];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            xx += __shfl_xor_sync(kFullMask, xx, d);
            qq += __shfl_xor_sync(kFullMask, qq, d);
            xq += __shfl_xor_sync(kFullMask, xq, d);
            dd += __shfl_xor_sync(kFullMask, dd, d);
        }
        const uint32_t warp = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            part[warp][0] = xx;
            part[warp][1] = qq;
            part[warp][2] = xq;
            part[warp][3] = dd;
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            double sum = 0.0;
            for (uint32_t w = 0; w < (blockDim.x >> 5); ++w) sum += part[w][threadIdx.x];
            atomicAdd(out + threadIdx.x, sum);
        }
    }
};

// 128-bit global accesses with an L2 eviction policy (createpolicy.fractional.L2::evict_*)
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// `bytes` from p, both of whole 16-byte units and bytes > 0, on their way to the L2
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint4 ld_hint_16(const void* p, uint64_t policy) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(policy)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_hint_16(void* p, uint4 v, uint64_t policy) {
    asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w), "l"(policy)
                 : "memory");
}

}  // namespace granq
