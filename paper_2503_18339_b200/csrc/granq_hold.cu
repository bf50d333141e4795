// Range and quantization in one launch for what has no run of channels to stage by itself: planes that are not whole 16-byte
// units in slabs that are not either, and one group over the whole tensor.
//
// One cooperative launch, two CTAs per SM.  A CTA takes an equal, contiguous piece of the tensor, whatever planes it cuts
// through, copies it to shared memory (33 MB over the GPU), folds it into one pair of keys per plane (Eq. 4) and those into the
// groups' keys with atomics; the grid hands over once (bounded), every CTA works out the parameters of its planes (Eq. 5) and
// quantizes its piece from shared memory (Eq. 1, clamp, Eq. 6, STE).  Of one group over a larger tensor what does not stay is
// read again, the last of it first, most of it from the L2.
// Bound by the chain copy, fold, hand-over, quantize; of the kept piece gy is brought into the L2 during the hand-over, when memory
// is idle: with gradient, [200,33,33,33] fp32, 29 MB, 22.8 -> 21.2, one group [128,64,28,28] fp32 20.5 -> 18.7, [128,192,28,28] bf16
// 30.6 -> 28.9 us.  Before that, against range pass and quantize pass (us, with gradient / forward / with
// sums): [100,75,27,27] fp32, 21.9 MB, 37.9 / 31.6 / 36.7 -> 25.0 / 18.7 / 21.4; [200,301,7,7] bf16 38.5 / 34.0 / 37.9 -> 17.6 /
// 16.6 / 19.8; one group: [128,128,28,28] fp32, 51 MB, sums 39.9 -> 29.2; [128,64,28,28] bf16, 13 MB, sums 24.5 -> 17.5.  Packed mask,
// 4-bit and 5-bit codes of one group: [128,128,28,28] fp32, a third of it read again, 33.9 / 37.0 / 38.7 -> 32.3 / 32.9 / 33.6; [96,128,28,28]
// fp32 27.0 / 28.8 / 29.9 -> 26.6 / 26.5 / 27.2; bf16 20.8 / 22.3 / 22.6 -> 16.6 / 20.7 / 20.8.  Against the L2-resident waves, one group:
// bf16 [128,192,28,28], 38.5 MB, 38.9 / 30.8 -> 35.4 / 24.7; fp32 [128,64,28,28] 26.6 / 18.8 -> 26.2 / 18.0.  What is left
// behind the last whole unit, and the last word of a mask or of codes, is one thread's: two passes with scalar loads there (with gradient)
// [60,301,7,7] bf16 41.2 -> 10.4, [150,75,27,27] bf16 138 -> 18.7, [5,75,27,27] fp32 30.5 -> 8.9.  There is no smallest size: a tensor
// of 80 KB, [8,75,5,7], takes 5.8 us from a graph and 11.9 eagerly where two passes took 23.1 and 25.4, one group of 0.5 MB 6.0 and 9.9 where the
// waves took 12.4 and 9.8.
#include "granq_internal.h"

#include <algorithm>

namespace granq {

namespace {

constexpr int kHThreads = 512;
constexpr uint32_t kHWarps = kHThreads / 32;
constexpr uint32_t kHSpinLimit = 1u << 24;              // bounded wait for the grid (x ~32 ns)
constexpr uint32_t kHStatusTimeout = 5;                 // GRANQ_ERR_TIMEOUT
constexpr uint32_t kHSmemBytes = 111u * 1024;           // two CTAs per SM
constexpr uint32_t kHFetchUnits = 1024;                 // gy of a kept piece of 16 KB and more is sent for during the hand-over,
constexpr uint32_t kHFetchPlane = 256;                  // of bf16 in planes of this many elements
constexpr uint32_t kHPlaneBytes = 2 * sizeof(uint32_t) + sizeof(GroupParam);      // keys and parameters of one plane

enum : int { H_ONE = 0, H_PLANES = 1, H_RAGGED = 2 };   // one group; planes of whole units; planes that are not

struct HArgs {
    const void* x;
    const void* gy;
    void* y;
    void* gx;
    uint32_t* pmask;       // the STE mask at one bit per element, or null
    uint32_t* pcodes;      // the codes as a bit string of code_bits each, or null (y is then not written)
    int code_bits;
    double* dist;          // four running sums of Table 2's statistics, or null
    uint32_t* status;
    uint32_t* kmin;
    uint32_t* kmax;
    uint32_t* counters;
    float* lo;
    float* hi;
    float* s_out;
    float* z_out;
    float qmax;
    uint32_t units;        // whole 16-byte units of the tensor (with a mask or codes, an even number of fp32 ones)
    uint32_t tail;         // elements behind them
    uint32_t share;        // of one CTA
    uint32_t held;         // of those, kept in shared memory
    uint32_t planes;       // room in the tables
    uint32_t inner;        // elements of one plane
    uint32_t groups;
    uint32_t spin_limit, expected;
    uint32_t early;        // x may be read before the kernel ahead has completed: it only clears the workspace
    FastDiv div_inner, div_groups;
};

// END: elements are left behind the last whole unit, or mask or codes end inside a 32-bit word (a form of its own: the code for it
// cost the others 0.3 us of 10).  U = units a thread handles together in the quantize walk
template <typename T, int MODE, int EXTRAS, int KIND, bool END, int U>
__global__ void __launch_bounds__(kHThreads, 2) hold_kernel(const HArgs a) {
    constexpr int V = Pack<T>::V;
    constexpr bool kBwd = (MODE & MODE_BWD) != 0;
    extern __shared__ __align__(16) unsigned char h_smem[];
    __shared__ uint32_t s_one[2][kHWarps];
    __shared__ uint32_t s_ok;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t u0 = blockIdx.x * a.share, n = min(a.share, a.units - u0), held = min(n, a.held);      // no CTA without units
    uint4* tile = reinterpret_cast<uint4*>(h_smem);
    GroupParam* s_par = reinterpret_cast<GroupParam*>(tile + a.held);
    uint32_t* s_kmn = reinterpret_cast<uint32_t*>(s_par + a.planes);
    uint32_t* s_kmx = s_kmn + a.planes;
    const uint4* xg = reinterpret_cast<const uint4*>(a.x) + u0;
    const uint4* gyg = reinterpret_cast<const uint4*>(a.gy) + u0;
    uint4* yg = reinterpret_cast<uint4*>(a.y) + u0;
    uint4* gxg = reinterpret_cast<uint4*>(a.gx) + u0;
    const float qmax = a.qmax;
    // elements behind the last whole unit, all of the last plane: the last CTA's, one thread handles them
    const uint32_t tail = END && blockIdx.x == gridDim.x - 1 ? a.tail : 0u;
    const T* xt = reinterpret_cast<const T*>(a.x) + (size_t)a.units * V;
    // planes of this piece: p0, p0 + 1, ..., the first of them from element rem0 on
    uint32_t p0 = 0, rem0 = 0, np = 1;
    if constexpr (KIND != H_ONE) {
        a.div_inner.divmod(u0 * V, p0, rem0);
        np = a.div_inner.div((u0 + n) * V - 1) - p0 + 1;
    }

    if (!a.early) after_the_kernel_ahead();
    for (uint32_t i = tid; i < held; i += kHThreads) cp_async_16(tile + i, xg + i);
    if constexpr (KIND != H_ONE) {
        for (uint32_t p = tid; p < np; p += kHThreads) s_kmn[p] = s_kmx[p] = 0;
    }

    // ---- Eq. 4 ----
    if constexpr (KIND == H_ONE) {
        RangeFold<T> fold;
        constexpr int UR = 4;
        for (uint32_t i = held + tid; i < n; i += UR * kHThreads) {        // what does not stay
            Pack<T> v[UR];
#pragma unroll
            for (int k = 0; k < UR; ++k)
                if (i + k * kHThreads < n) v[k].raw = __ldg(xg + i + k * kHThreads);
#pragma unroll
            for (int k = 0; k < UR; ++k)
                if (i + k * kHThreads < n) fold.add(v[k]);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        for (uint32_t i = tid; i < held; i += kHThreads) {                 // its own copies
            Pack<T> v;
            v.raw = tile[i];
            fold.add(v);
        }
        float m0, m1;
        fold.result(m0, m1);
        if constexpr (END) {
            for (uint32_t i = 0; tid == kHThreads - 1 && i < tail; ++i) {
                const float v = load_scalar(xt + i);
                m0 = fminf(m0, v);
                m1 = fmaxf(m1, v);
            }
        }
        uint32_t ka = m0 <= m1 ? ~enc(m0) : 0u, kb = m0 <= m1 ? enc(m1) : 0u;
        ka = __reduce_max_sync(kFullMask, ka);
        kb = __reduce_max_sync(kFullMask, kb);
        if (lane == 0) {
            s_one[0][tid >> 5] = ka;
            s_one[1][tid >> 5] = kb;
        }
        if (a.early) after_the_kernel_ahead();
        __syncthreads();
        if (tid < 32) {
            ka = __reduce_max_sync(kFullMask, lane < kHWarps ? s_one[0][lane] : 0u);
            kb = __reduce_max_sync(kFullMask, lane < kHWarps ? s_one[1][lane] : 0u);
            if (lane == 0) {
                atomicMax(a.kmin, ka);
                atomicMax(a.kmax, kb);
            }
        }
    } else {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // a run of neighbouring units per thread (an odd number of them: no bank conflicts), so that the plane seldom changes
        const uint32_t run = ((n + kHThreads - 1) / kHThreads) | 1u, first = tid * run, last = min(n, first + run);
        if (first < last) {
            uint32_t p, rem;
            a.div_inner.divmod(rem0 + first * V, p, rem);
            uint32_t left = a.inner - rem;                                 // elements of the plane from here on
            float mn = INFINITY, mx = -INFINITY;
            auto flush = [&] {
                if (mn <= mx) {
                    atomicMax(s_kmn + p, ~enc(mn));
                    atomicMax(s_kmx + p, enc(mx));
                }
                mn = INFINITY;
                mx = -INFINITY;
                ++p;
            };
            for (uint32_t i = first; i < last; ++i) {
                Pack<T> v;
                v.raw = tile[i];
                if (left >= (uint32_t)V) {
                    pack_minmax(v, 0, V, mn, mx);
                    left -= V;
                    if (left == 0) {
                        flush();
                        left = a.inner;
                    }
                } else {                                                   // ragged: the plane ends inside
                    pack_minmax(v, 0, (int)left, mn, mx);
                    flush();
                    pack_minmax(v, (int)left, V, mn, mx);
                    left += a.inner - V;
                }
            }
            flush();
        }
        if constexpr (END) {
            for (uint32_t i = 0; tid == kHThreads - 1 && i < tail; ++i) {
                const float v = load_scalar(xt + i);
                if (v == v) {
                    atomicMax(s_kmn + np - 1, ~enc(v));
                    atomicMax(s_kmx + np - 1, enc(v));
                }
            }
        }
        if (a.early) after_the_kernel_ahead();
        __syncthreads();
        for (uint32_t t = tid; t < np; t += kHThreads) {
            const uint32_t c = p0 + t - a.div_groups.div(p0 + t) * a.groups, k1 = s_kmn[t], k2 = s_kmx[t];
            if (k1 | k2) {
                atomicMax(a.kmin + c, k1);
                atomicMax(a.kmax + c, k2);
            }
        }
    }
    // ---- the grid's hand-over (bounded) ----
    if constexpr (kBwd) {
        // what the kept piece meets is on its way to the L2 while the grid waits for its last CTA (half of it gives half as much); a
        // smaller one is most often still there ([20,75,27,27] fp32 10.1 -> 10.5), and CTAs that fold short planes of bf16 leave memory no idle
        // time to use ([789,75,13,13] 31.3 -> 32.2, [5333,75,5,5] 81.2 -> 81.8, of 17 x 17 on 38.6 -> 37.5; fp32 [1361,75,7,7] 36.4 -> 34.0)
        if (tid == 0 && held >= kHFetchUnits && (V == 4 || a.inner >= kHFetchPlane)) prefetch_l2(gyg, held * 16u);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        atomicAdd(a.counters, 1u);
        uint32_t ready = 0;
        for (uint32_t i = 0; i < a.spin_limit; ++i) {
            if (ld_acquire(a.counters) >= a.expected) {
                ready = 1;
                break;
            }
            __nanosleep(32);
        }
        s_ok = ready;
        if (!ready) atomicExch(a.status, kHStatusTimeout);
    }
    __syncthreads();
    if (!s_ok) return;
    for (uint32_t t = tid; t < np; t += kHThreads) {
        const uint32_t c = KIND == H_ONE ? 0u : p0 + t - a.div_groups.div(p0 + t) * a.groups;
        float lo, hi;
        const GroupParam gp = group_param_from_keys(a.kmin, a.kmax, c, qmax, lo, hi);
        s_par[t] = gp;
        if (p0 + t == c && (t > 0 || rem0 == 0)) {                         // where the group's first plane begins
            a.lo[c] = lo;
            a.hi[c] = hi;
            if (a.s_out) a.s_out[c] = gp.s;
            if (a.z_out) a.z_out[c] = gp.z;
        }
    }
    __syncthreads();
    if (tid == 0) {          // the keys have been read; the last CTA to say so leaves the workspace zero (below)
        __threadfence();
        s_ok = (atomicAdd(a.counters + 1, 1u) == gridDim.x - 1) ? 1u : 0u;
    }

    // ---- Eq. 1, clamp, Eq. 6, STE ----
    DistAcc dacc;               // Table 2's sums over everything this thread quantizes (EXTRAS = 4)
    dacc.reset();
    const GroupParam one = s_par[0];
    constexpr bool kPairs = V == 4 && (EXTRAS == 2 || EXTRAS == 3);      // written by neighbouring lanes together
    auto emit = [&](const Pack<T>& px, const Pack<T>& pg, uint32_t i, uint32_t lanes) {
        Pack<T> py, pgx;
        uint32_t cb[V / 4], mb[V / 4];
        const int code_bits = EXTRAS == 3 ? a.code_bits : 8;
        if constexpr (KIND == H_ONE) {
            quantize_own<T, kBwd, EXTRAS>(px, pg, one, qmax, py, pgx, cb, mb, code_bits);
        } else {
            uint32_t p, rem;
            a.div_inner.divmod(rem0 + i * V, p, rem);
            if constexpr (KIND == H_PLANES) {
                quantize_own<T, kBwd, EXTRAS>(px, pg, s_par[p], qmax, py, pgx, cb, mb, code_bits);
            } else {
                const int n1 = (int)min((uint32_t)V, a.inner - rem);
                const GroupParam g1 = s_par[p];
                if (n1 == V) quantize_own<T, kBwd, EXTRAS>(px, pg, g1, qmax, py, pgx, cb, mb, code_bits);
                else quantize_pack<T, kBwd, true, EXTRAS, true>(px, pg, g1, s_par[p + 1], n1, qmax, py, pgx, cb, mb, code_bits);
            }
        }
        // masks and codes 8 elements at a time, a pair of fp32 units by the two lanes of a pair, the first of them by the even one: the
        // whole units are a multiple of 8 elements, a piece begins on a multiple of 8 units, and both walks give an even lane an even unit
        if constexpr (EXTRAS == 3) {
            store_code_bytes<V>(a.pcodes, (size_t)(u0 + i) * V, code_string_of<V>(cb, code_bits), code_bits, lane, lanes);
            return;
        }
        st_stream_16(yg + i, py.raw);
        if constexpr (kBwd) st_stream_16(gxg + i, pgx.raw);
        if constexpr (EXTRAS == 2) store_mask_byte<V>(a.pmask, (size_t)(u0 + i) * V, mask_bits_of<V, EXTRAS>(mb), lane, lanes);
        if constexpr (EXTRAS == 4) dacc.add(px, py);
    };
    if constexpr (END) {
        if (tid == kHThreads - 1 && blockIdx.x == gridDim.x - 1) {
            const size_t e0 = (size_t)a.units * V;
            const GroupParam gp = s_par[np - 1];
            uint64_t str = 0;                   // masks and codes: of the tail, a whole number of bytes before it
            for (uint32_t off = 0; off < tail; off += V) {
                Pack<T> px, pg, py, pgx;
                uint32_t cb[V / 4], mb[V / 4];
                px.raw = pg.raw = make_uint4(0, 0, 0, 0);
                for (uint32_t i = 0; i < (uint32_t)V; ++i)
                    if (off + i < tail) {
                        px.set(i, load_scalar(xt + off + i));
                        if constexpr (kBwd) pg.set(i, load_scalar(reinterpret_cast<const T*>(a.gy) + e0 + off + i));
                    }
                quantize_own<T, kBwd, EXTRAS>(px, pg, gp, qmax, py, pgx, cb, mb, EXTRAS == 3 ? a.code_bits : 8);
                for (uint32_t i = 0; i < (uint32_t)V; ++i)
                    if (off + i < tail) {
                        if constexpr (EXTRAS != 3) store_scalar(reinterpret_cast<T*>(a.y) + e0 + off + i, py.get(i));
                        if constexpr (kBwd) store_scalar(reinterpret_cast<T*>(a.gx) + e0 + off + i, pgx.get(i));
                        if constexpr (EXTRAS == 4) dacc.add_one(px.get(i), py.get(i));
                    }
                if constexpr (EXTRAS == 2) str |= (uint64_t)mask_bits_of<V, EXTRAS>(mb) << off;
                if constexpr (EXTRAS == 3) str |= code_string_of<V>(cb, a.code_bits) << (off * a.code_bits);
            }
            if constexpr (EXTRAS == 2 || EXTRAS == 3) {                        // up to the end of the last word
                const uint32_t width = EXTRAS == 3 ? a.code_bits : 1;
                uint8_t* dst = reinterpret_cast<uint8_t*>(EXTRAS == 3 ? a.pcodes : a.pmask) + e0 / 8 * width;
                const size_t bytes = ((e0 + tail) * width + 31) / 32 * 4 - e0 / 8 * width;
                str &= (1ull << (tail * width)) - 1;                           // at most 7 codes: 56 bits
                for (size_t i = 0; i < bytes; ++i) dst[i] = i < 8 ? (uint8_t)(str >> (8 * i)) : (uint8_t)0;
            }
        }
    }
    // what did not stay, a block of units at a time from the end back; inside a block forward from an even unit (masks and codes:
    // n and held are even), so that the even lane of a pair has its first unit there too
    if constexpr (KIND == H_ONE) {
        for (uint32_t end = n; end > held;) {
            const uint32_t len = min((uint32_t)(U * kHThreads), end - held), start = end - len;
            Pack<T> px[U], pg[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t i = k * kHThreads + tid;
                if (i < len) {
                    px[k].raw = ld_stream_16(xg + start + i);
                    if constexpr (kBwd) pg[k].raw = ld_stream_16(gyg + start + i);
                }
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t i = k * kHThreads + tid;
                const uint32_t lanes = kPairs ? __ballot_sync(kFullMask, i < len) : 0u;
                if (i < len) emit(px[k], pg[k], start + i, lanes);
            }
            end = start;
        }
    }
    for (uint32_t b = 0; b < held; b += U * kHThreads) {
        Pack<T> px[U], pg[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const uint32_t i = b + k * kHThreads + tid;
            if (i < held) {
                if constexpr (kBwd) pg[k].raw = ld_stream_16(gyg + i);
                px[k].raw = tile[i];
            }
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const uint32_t i = b + k * kHThreads + tid;
            const uint32_t lanes = kPairs ? __ballot_sync(kFullMask, i < held) : 0u;
            if (i < held) emit(px[k], pg[k], i, lanes);
        }
    }
    if constexpr (EXTRAS == 4) dacc.flush(a.dist);
    __syncthreads();
    if (s_ok) {
        for (uint32_t t = tid; t < a.groups; t += kHThreads) {
            a.kmin[t] = 0;
            a.kmax[t] = 0;
        }
        if (tid < 2) a.counters[tid] = 0;
    }
}

bool h_aligned16(const void* p) { return p == nullptr || ((uintptr_t)p & 15) == 0; }

template <typename T, int MODE, int EXTRAS>
cudaError_t h_launch(const HArgs& a, const HoldPlan& p, int kind, const StagedTuning& tune, cudaStream_t st) {
    constexpr int U = MODE == MODE_FWD ? 4 : 2;
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kHSmemBytes);
        if (e != cudaSuccess) return e;
        void* params[] = {(void*)&a};
        return launch_cooperative((const void*)kern, p.ctas, kHThreads, params, p.held * 16 + p.planes * kHPlaneBytes, tune, st);
    };
    if (kind == H_ONE) return p.whole ? go(hold_kernel<T, MODE, EXTRAS, H_ONE, false, U>) : go(hold_kernel<T, MODE, EXTRAS, H_ONE, true, U>);
    if (kind == H_RAGGED) return p.whole ? go(hold_kernel<T, MODE, EXTRAS, H_RAGGED, false, U>) : go(hold_kernel<T, MODE, EXTRAS, H_RAGGED, true, U>);
    // planes of whole units leave nothing behind the last of them but for a mask or codes
    if constexpr (EXTRAS == 2 || EXTRAS == 3)
        if (!p.whole) return go(hold_kernel<T, MODE, EXTRAS, H_PLANES, true, U>);
    return go(hold_kernel<T, MODE, EXTRAS, H_PLANES, false, U>);
}

}  // namespace

// All of the tensor stays on chip; of one group up to as much again is read twice, but not in fp32 with a gradient, where the
// waves are faster ([128,128,28,28], 51 MB, 43.5 / 45.5 us).
HoldPlan plan_hold(int dtype, const Geom& g, const QuantIO& io, int sm_count) {
    HoldPlan p{};
    p.ok = false;
    const int64_t V = dtype == 0 ? 4 : 8;
    if (io.codes || io.mask) return p;
    const bool packed = io.pmask || io.pcodes;
    if (packed && io.gy) return p;
    const int64_t step = packed ? 8 : V;                  // the whole units: masks and codes whole bytes of them
    p.tail = (uint32_t)(g.E % step);
    p.whole = p.tail == 0 && !(packed && g.E % 32 != 0);
    if (g.E < step || g.inner < V || (p.tail && g.inner < step) || g.E >= (1ll << 31) || g.C >= (1ll << 28)) return p;
    if (!h_aligned16(io.x) || !h_aligned16(io.gy) || !h_aligned16(io.y) || !h_aligned16(io.gx)) return p;
    const uint64_t units = (uint64_t)((g.E - p.tail) / V), most = 2ull * (uint64_t)sm_count;
    p.share = (uint32_t)((std::max<uint64_t>((units + most - 1) / most, 64) + 7) / 8 * 8);
    p.ctas = (uint32_t)((units + p.share - 1) / p.share);
    const bool one = g.C == 1 && g.outer == 1;
    const uint64_t planes = one ? 1 : (uint64_t)p.share * V / (uint64_t)g.inner + 2;
    if (planes * kHPlaneBytes >= kHSmemBytes / 2) return p;
    p.planes = (uint32_t)planes;
    const uint32_t room = (kHSmemBytes - (p.planes * kHPlaneBytes + 15) / 16 * 16) / 16;
    p.held = std::min(p.share, room / 2 * 2);             // whole pairs of fp32 units, which lanes write masks and codes of together
    if (p.held < p.share && !(one && p.share <= 2 * room && (dtype == 1 || !io.gy))) return p;
    p.ok = true;
    return p;
}

cudaError_t launch_hold(const HoldPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                        const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt, const StagedTuning& tune,
                        cudaStream_t st) {
    const uint32_t V = dtype == 0 ? 4 : 8;
    HArgs a{};
    a.x = io.x;
    a.gy = io.gy;
    a.y = io.y;
    a.gx = io.gx;
    a.pmask = io.pmask;
    a.pcodes = io.pcodes;
    a.code_bits = io.code_bits;
    a.dist = io.dist;
    a.status = ws.status;
    a.kmin = ws.kmin;
    a.kmax = ws.kmax;
    a.counters = ws.counters;
    a.lo = lo;
    a.hi = hi;
    a.s_out = s_opt;
    a.z_out = z_opt;
    a.qmax = (float)((1 << bits) - 1);
    a.units = (uint32_t)((g.E - plan.tail) / V);
    a.tail = plan.tail;
    a.share = plan.share;
    a.held = plan.held;
    a.planes = plan.planes;
    a.inner = (uint32_t)g.inner;
    a.groups = (uint32_t)g.C;
    a.spin_limit = tune.spin_limit > 0 ? (uint32_t)tune.spin_limit : kHSpinLimit;
    a.expected = plan.ctas + (uint32_t)(tune.extra_arrivals > 0 ? tune.extra_arrivals : 0);
    a.early = ws.cleared ? 1u : 0u;
    a.div_inner = make_fastdiv(a.inner);
    a.div_groups = make_fastdiv(a.groups);
    const int kind = g.C == 1 && g.outer == 1 ? H_ONE : g.inner % V == 0 ? H_PLANES : H_RAGGED;
    auto go = [&](auto zero) -> cudaError_t {
        using T = decltype(zero);
        if (mode != MODE_FWD) return h_launch<T, MODE_BOTH, 0>(a, plan, kind, tune, st);
        if (io.dist) return h_launch<T, MODE_FWD, 4>(a, plan, kind, tune, st);
        if (io.pmask) return h_launch<T, MODE_FWD, 2>(a, plan, kind, tune, st);
        if (io.pcodes) return h_launch<T, MODE_FWD, 3>(a, plan, kind, tune, st);
        return h_launch<T, MODE_FWD, 0>(a, plan, kind, tune, st);
    };
    return dtype == 0 ? go(0.0f) : go(__nv_bfloat16());
}

}  // namespace granq
