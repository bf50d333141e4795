// Resident column walk: every activation of a large channel group is read from HBM once.
//
// A channel of a large plane (1.6 MB for 56 x 56 planes at batch 128, 6.4 MB for 112 x 112) fits neither one SM nor
// one thread-block cluster, but it fits the shared memory of a TEAM of CTAs of one cooperative launch, and the
// whole GPU holds 18 teams of 16 such CTAs.  Each team takes one channel at a time:
//   - its units (16 bytes each, all slabs laid end to end) are dealt out evenly over the team's CTAs; a CTA copies
//     its share to shared memory with per-thread asynchronous copies, every thread copying exactly the units it will
//     read, so no barrier stands between a copy and its use;
//   - each CTA reduces its share (Eq. 4), publishes one pair of ordered keys with atomics, arrives on the channel's
//     counter and waits (bounded) for the rest of its team - not for the grid;
//   - scale and zero-point (Eq. 5) are worked out once per CTA and the share is quantized from shared memory (Eq. 1,
//     clamp, Eq. 6, STE).  A unit's place in shared memory is free as soon as its thread has read it, so the same
//     loop sends the copy of the team's NEXT channel after it: reads stay in flight through the whole write phase.
// With a gradient gy is staged the same way as far as shared memory goes and read in place beyond that; where a team then
// has several rounds of channels, colteam_lag_kernel below holds two of them at a time instead.
//
// Why not the L2-resident waves of colwalk_kernel: the L2 does not keep a wave (forward-only calls read x 1.4
// times from HBM, ncu: 9-15 % L2 hits), and its phases alternate.  Why teams and not clusters of 16 CTAs: a
// cluster must sit in one GPC, which leaves an SM in ten without one.  Measured against the waves (fp32 / bf16, us):
// forward [128,64,56,56] 55.8 -> 45.7 / 34.7 -> 30.3, [128,96,112,112] 309 -> 264 / 174 -> 139, [256,512,28,28]
// 219 -> 156 / 123 -> 92; with a gradient 87.5 -> 81.9 / 47.4 -> 45.6, 472 -> 469 / 258 -> 234, 332 -> 298 / 183 -> 153;
// [256,16,32,32] 16.7 -> 14.9 and 21.9 -> 19.4.  Bound by the chain of copy, hand-over and quantize when a team has one
// channel.  With several it moves 4.5 to 5.7 TB/s where plain copies in blocks that come in order move 6.7: 66 (with a
// packed mask) to 106 (with a gradient) instructions per unit, sixteen wavefronts for an asynchronous copy of a warp, and
// equal shares, of which half of the SMs move 21 KB/us and the other half 37 when nothing holds them together.  Chunks dealt
// out by a counter even the SMs out but publish, poll and fetch keys per chunk: 10 us of residence against the 10 us that
// 33 MB last at full rate; with a gradient they reached 425 us where two channels side by side take 433, forward 183 where
// this form takes 151.
//
// Two CTAs of 512 threads per SM, 113 KB of shared memory each: one transfers while the other waits for its team.
// The kernel expects zeroed keys and counters and, when no wait ran out, leaves them zeroed (slot C of the
// counters counts the CTAs that have finished; the last one clears).
#include "granq_internal.h"

#include <algorithm>
#include <atomic>

namespace granq {

namespace {

constexpr int kTThreads = 512;
constexpr uint32_t kTWarps = kTThreads / 32;
constexpr uint32_t kTSpinLimit = 1u << 24;   // bounded wait on a channel's counter (x ~32 ns)
constexpr uint32_t kTStatusTimeout = 5;      // GRANQ_ERR_TIMEOUT
constexpr uint32_t kTSmemUnits = 111u * 1024 / 16;      // staged units per CTA: two CTAs per SM, 228 KB between them
constexpr uint32_t kTLagUnits = 1700;                   // smallest share of each of two channels side by side

struct TArgs {
    const void* x;
    const void* gy;
    void* y;
    void* gx;
    uint32_t* pmask;       // the STE mask at one bit per element, or null
    uint32_t* pcodes;      // the codes as a bit string of code_bits each, or null (y is then not written)
    int code_bits;
    uint32_t code_words;   // planes are whole runs of 32 codes: they are written as words
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
    uint32_t C;            // channels
    uint32_t plane_units;  // units of one plane
    uint32_t units;        // units of one channel over all slabs
    uint32_t R, teams;     // CTAs per team, teams
    uint32_t tile_units;   // room for x in shared memory
    uint32_t gy_units;     // of a CTA's share of gy, this many units are staged behind it
    uint32_t spin_limit, expected;
    uint32_t early;        // x and gy may be read before the kernel ahead has completed: it only clears the workspace
    uint32_t slab_units;   // units of one slab (where there is more than one)
    FastDiv div_plane;     // units per plane
};

__device__ __forceinline__ void t_arrive_release(uint32_t* p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
// No L2 policy operand here, nor on any access of this kernel: a form that gave the copies sent from the quantize walk one
// ended in an illegal instruction on [128,64,56,56], forward.  The cause was not found: operand widths, the policy's
// lifetime, addresses, sizes and trip counts were in order, and the same instruction in loops of unequal trip counts ran
// elsewhere without fault.  Without the operand, with streaming loads and stores: the same times.
__device__ __forceinline__ void t_cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// U = units a thread handles together in the quantize walk
// BITS = bits of a code (EXTRAS = 3 only: shifts and lanes of the code string are then constants)
// At = index of a unit of the tensor: 32 bits below 64 GB
template <typename T, int MODE, int EXTRAS, int U, int BITS, typename At, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) colteam_kernel(const TArgs a) {
    constexpr int V = Pack<T>::V;
    constexpr bool kBwd = (MODE & MODE_BWD) != 0;
    extern __shared__ __align__(16) uint4 t_smem[];
    __shared__ uint32_t s_kmn[(NT / 32)], s_kmx[(NT / 32)];
    __shared__ GroupParam s_par;
    __shared__ uint32_t s_ok;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t team = blockIdx.x / a.R, rank = blockIdx.x - team * a.R;
    // this CTA's share: whole runs of 8 units (128 bytes) of the channel's units laid end to end
    const uint32_t runs = (a.units + 7) / 8;
    const uint32_t q0 = 8 * (uint32_t)(((uint64_t)rank * runs) / a.R);
    const uint32_t q1 = min(a.units, 8 * (uint32_t)(((uint64_t)(rank + 1) * runs) / a.R));
    const uint32_t n = q1 - q0;
    const uint32_t cnt = tid < n ? (n - tid + NT - 1) / NT : 0u;      // units of this thread
    // where they are: unit q lies in slab q / plane_units, and the next one of this thread is NT units on
    uint32_t slab0, off0;
    a.div_plane.divmod(q0 + min(tid, n), slab0, off0);
    const At first = (At)slab0 * a.slab_units + off0;
    uint32_t dslab, doff;
    a.div_plane.divmod((uint32_t)NT, dslab, doff);
    const At dstep = (At)dslab * a.slab_units + doff, dwrap = a.slab_units - a.plane_units;
    auto advance = [&](At& at, uint32_t& off) {
        at += dstep;
        off += doff;
        if (off >= a.plane_units) {
            off -= a.plane_units;
            at += dwrap;
        }
    };
    // words of codes and fp32 masks take neighbouring lanes together: units that every lane of the warp has (the first lanes may have one more)
    constexpr bool kPairs = EXTRAS == 3 || (EXTRAS == 2 && V == 4);
    const uint32_t whole = kPairs ? __shfl_sync(kFullMask, cnt, 31) : cnt;
    uint4* tile = t_smem + tid;
    uint4* tileg = t_smem + a.tile_units + tid;
    const uint32_t gcnt = kBwd ? (tid < a.gy_units ? min(cnt, (a.gy_units - tid + NT - 1) / NT) : 0u) : 0u;
    const uint4* xg = reinterpret_cast<const uint4*>(a.x);
    const uint4* gyg = reinterpret_cast<const uint4*>(a.gy);
    uint4* yg = reinterpret_cast<uint4*>(a.y);
    uint4* gxg = reinterpret_cast<uint4*>(a.gx);
    const float qmax = a.qmax;
    DistAcc dacc;               // Table 2's sums over everything this thread quantizes (EXTRAS = 4)
    dacc.reset();
    if (!a.early) after_the_kernel_ahead();

    // the first channel's copies; those of the later ones are sent from the quantize walk
    {
        At at = first + (At)team * a.plane_units;
        uint32_t off = off0;
        for (uint32_t i = 0; i < cnt; ++i) {
            cp_async_16(tile + i * NT, xg + at);
            if (kBwd && i < gcnt) cp_async_16(tileg + i * NT, gyg + at);
            advance(at, off);
        }
    }
    if (a.early) after_the_kernel_ahead();
    for (uint32_t c = team; c < a.C; c += a.teams) {
        t_cp_async_wait_all();
        // ---- Eq. 4: range of this CTA's share ----
        RangeFold<T> fold;
        for (uint32_t i = 0; i < cnt; ++i) {
            Pack<T> p;
            p.raw = tile[i * NT];
            fold.add(p);
        }
        float m0, m1;
        fold.result(m0, m1);
        uint32_t ka = m0 <= m1 ? ~enc(m0) : 0u, kb = m0 <= m1 ? enc(m1) : 0u;
        ka = __reduce_max_sync(kFullMask, ka);
        kb = __reduce_max_sync(kFullMask, kb);
        if (lane == 0) {
            s_kmn[tid >> 5] = ka;
            s_kmx[tid >> 5] = kb;
        }
        __syncthreads();
        if (tid < 32) {
            ka = __reduce_max_sync(kFullMask, lane < (NT / 32) ? s_kmn[lane] : 0u);
            kb = __reduce_max_sync(kFullMask, lane < (NT / 32) ? s_kmx[lane] : 0u);
            if (lane == 0) {
                atomicMax(a.kmin + c, ka);
                atomicMax(a.kmax + c, kb);
                t_arrive_release(a.counters + c);
                // ---- wait (bounded) until the whole team has published the channel; Eq. 5 ----
                uint32_t ready = 0;
                for (uint32_t i = 0; i < a.spin_limit; ++i) {
                    if (ld_acquire(a.counters + c) >= a.expected) {
                        ready = 1;
                        break;
                    }
                    __nanosleep(32);
                }
                s_ok = ready;
                if (ready) {
                    float lo, hi;
                    const GroupParam gp = group_param_from_keys(a.kmin, a.kmax, c, qmax, lo, hi);
                    s_par = gp;
                    if (rank == 0) {
                        a.lo[c] = lo;
                        a.hi[c] = hi;
                        if (a.s_out) a.s_out[c] = gp.s;
                        if (a.z_out) a.z_out[c] = gp.z;
                    }
                } else {
                    atomicExch(a.status, kTStatusTimeout);
                }
            }
        }
        __syncthreads();
        if (!s_ok) return;      // nothing is in flight: the copies of this channel have landed, the next ones are not sent
        const GroupParam g = s_par;

        // ---- Eq. 1, clamp, Eq. 6, STE from shared memory; the next channel's copies follow on the heels ----
        const bool more = c + a.teams < a.C;
        const At ahead = (At)a.teams * a.plane_units;
        auto quantize = [&](const Pack<T>& px, const Pack<T>& pg, At at, uint32_t (&cb)[V / 4], uint32_t (&mb)[V / 4]) {
            Pack<T> py, pgx;
            // with a gradient the scalar form: f32 [190,4,96,97] 28.0 us, in packed pairs 29.5; [112,126,56,56] 132.7 / 137.3
            if constexpr (kBwd) quantize_pack<T, kBwd, false, EXTRAS, true>(px, pg, g, g, V, qmax, py, pgx, cb, mb);
            else quantize_own<T, kBwd, EXTRAS>(px, pg, g, qmax, py, pgx, cb, mb, BITS);
            if constexpr (EXTRAS != 3) st_stream_16(yg + at, py.raw);
            if constexpr (kBwd) st_stream_16(gxg + at, pgx.raw);
            if constexpr (EXTRAS == 4) dacc.add(px, py);
        };
        At at = first + (At)c * a.plane_units;
        uint32_t off = off0, i = 0;
        // N units of every lane of the warp
        auto together = [&](auto number) {
            constexpr int N = decltype(number)::value;
            Pack<T> px[N], pg[N];
            At w[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                w[j] = at;
                if constexpr (kBwd) {
                    if (i + j < gcnt) pg[j].raw = tileg[(i + j) * NT];
                    else pg[j].raw = ld_stream_16(gyg + at);
                }
                px[j].raw = tile[(i + j) * NT];
                advance(at, off);
            }
            if (more) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    cp_async_16(tile + (i + j) * NT, xg + (w[j] + ahead));
                    if (kBwd && i + j < gcnt) cp_async_16(tileg + (i + j) * NT, gyg + (w[j] + ahead));
                }
            }
            i += N;
            uint32_t cb[N][V / 4], mb[N][V / 4];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                quantize(px[j], pg[j], w[j], cb[j], mb[j]);
                if constexpr (EXTRAS == 2 && V == 8) reinterpret_cast<uint8_t*>(a.pmask)[w[j]] = (uint8_t)mb[j][0];
                if constexpr (EXTRAS == 3 && V == 8) {
                    const uint64_t str = code_string_of<V>(cb[j], BITS);
                    if (a.code_words) store_code_words<BITS, 1>(a.pcodes, w[j], str, lane & 3u, lane);
                    else store_eight_codes(a.pcodes, w[j], str, BITS);
                }
            }
            if constexpr (EXTRAS == 2 && V == 4) {
                uint32_t bits[N];
#pragma unroll
                for (int j = 0; j < N; ++j) bits[j] = mb[j][0];
                const uint32_t bytes = pair_up_mask<N>(bits, lane);
#pragma unroll
                for (int j = 0; j < N; j += 2)
                    reinterpret_cast<uint8_t*>(a.pmask)[(lane & 1 ? w[j + 1] : w[j]) >> 1] = (uint8_t)(bytes >> (4 * j));
            } else if constexpr (EXTRAS == 3 && V == 4) {
#pragma unroll
                for (int j = 0; j < N; j += 2) {
                    const uint64_t str = pair_up_codes(cb[j][0], cb[j + 1][0], BITS, lane);
                    const At eight = (lane & 1 ? w[j + 1] : w[j]) >> 1;
                    if (a.code_words) store_code_words<BITS, 2>(a.pcodes, eight, str, (lane >> 1) & 3u, lane);
                    else store_eight_codes(a.pcodes, eight, str, BITS);
                }
            }
        };
        auto alone = [&](uint32_t lanes) {
            Pack<T> px, pg;
            if constexpr (kBwd) {
                if (i < gcnt) pg.raw = tileg[i * NT];
                else pg.raw = ld_stream_16(gyg + at);
            }
            px.raw = tile[i * NT];
            if (more) {
                cp_async_16(tile + i * NT, xg + (at + ahead));
                if (kBwd && i < gcnt) cp_async_16(tileg + i * NT, gyg + (at + ahead));
            }
            uint32_t cb[V / 4], mb[V / 4];
            quantize(px, pg, at, cb, mb);
            if constexpr (EXTRAS == 2) store_mask_byte<V>(a.pmask, (size_t)at * V, mask_bits_of<V, EXTRAS>(mb), lane, lanes);
            if constexpr (EXTRAS == 3) store_code_bytes<V>(a.pcodes, (size_t)at * V, code_string_of<V>(cb, BITS), BITS, lane, lanes);
            advance(at, off);
            ++i;
        };
        while (i + U <= whole) together(PartAt<U>{});
        if constexpr (kPairs && U > 2) {
            if (i + 2 <= whole) together(PartAt<2>{});
        }
        while (i < whole) alone(kFullMask);
        if constexpr (kPairs) {
            const uint32_t lanes = __ballot_sync(kFullMask, i < cnt);
            if (i < cnt) alone(lanes);
        }
    }
    if constexpr (EXTRAS == 4) dacc.flush(a.dist);

    // ---- leave the workspace as it was found: the last CTA to finish clears keys and counters ----
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_ok = (atomicAdd(a.counters + a.C, 1u) == gridDim.x - 1) ? 1u : 0u;
    }
    __syncthreads();
    if (s_ok) {
        for (uint32_t i = tid; i < a.C; i += NT) {
            a.kmin[i] = 0;
            a.kmax[i] = 0;
        }
        for (uint32_t i = tid; i <= a.C; i += NT) a.counters[i] = 0;
    }
}

// The same with a gradient where a team has several rounds of channels: two channels side by side in shared memory, gy read in
// place.  The range of channel t is taken and handed to the team before channel t - 1 is quantized, so that the hand-over has
// that whole walk to complete in; a warp that holds no units does it.  (Forward calls lose by it: their walk is half as long,
// and twice the rounds cost more than the hand-over: [256,512,28,28] 151 / 163 us.)
// The channels may be those of a list of tensors of the same dims that share no memory: they follow one another without a
// launch or a wait between them (fp32, seven of [256,16,32,32] 143.9 -> 90.6 us, six of [128,64,56,56] 475.7 -> 418.6).
constexpr uint32_t kTWork = kTThreads - 32;

struct TTensor {
    const void* x;
    const void* gy;
    void* y;
    void* gx;
    uint32_t* status;
    uint32_t* kmin;
    uint32_t* kmax;
    uint32_t* counters;
    float* lo;
    float* hi;
    float* s_out;
    float* z_out;
    float qmax;
};
struct TList {
    uint32_t n;
    FastDiv div_C;
    TTensor t[kTeamListMax];
};

template <typename T, int U, bool LIST>
__global__ void __launch_bounds__(kTThreads, 2) colteam_lag_kernel(const TArgs a, const __grid_constant__ TList list) {
    constexpr int V = Pack<T>::V;
    constexpr uint32_t depth = 2;
    extern __shared__ __align__(16) uint4 t_smem[];
    __shared__ uint32_t s_kmn[2][kTWarps], s_kmx[2][kTWarps];
    __shared__ GroupParam s_par[2];
    __shared__ uint32_t s_bad, s_last;      // the job whose hand-over ran out of its wait; is this the last CTA?
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t team = blockIdx.x / a.R, rank = blockIdx.x - team * a.R;
    // channels of this team: team, team + teams, ... of all tensors' channels one after the other
    const uint32_t total = LIST ? list.n * a.C : a.C, jobs = team < total ? (total - team + a.teams - 1) / a.teams : 0u;
    // this CTA's share: whole runs of 8 units (128 bytes) of the channel's units laid end to end
    const uint32_t runs = (a.units + 7) / 8;
    const uint32_t q0 = 8 * (uint32_t)(((uint64_t)rank * runs) / a.R);
    const uint32_t q1 = min(a.units, 8 * (uint32_t)(((uint64_t)(rank + 1) * runs) / a.R));
    const uint32_t n = q1 - q0;
    const uint32_t cnt = tid < min(n, (uint32_t)kTWork) ? (n - tid + kTWork - 1) / kTWork : 0u;      // units of this thread
    // where they are: unit q lies in slab q / plane_units, and the next one of this thread is kTWork units on
    uint32_t slab0, off0;
    a.div_plane.divmod(q0 + min(tid, n), slab0, off0);
    const uint32_t first = slab0 * a.slab_units + off0;
    uint32_t dslab, doff;
    a.div_plane.divmod((uint32_t)kTWork, dslab, doff);
    const uint32_t dstep = dslab * a.slab_units + doff, dwrap = a.slab_units - a.plane_units;
    auto advance = [&](uint32_t& at, uint32_t& off) {
        at += dstep;
        off += doff;
        if (off >= a.plane_units) {
            off -= a.plane_units;
            at += dwrap;
        }
    };
    auto job = [&](uint32_t j, uint32_t& t, uint32_t& c) {
        t = 0;
        c = team + j * a.teams;
        if constexpr (LIST) list.div_C.divmod(c, t, c);
    };

    // ---- Eq. 4: range of this CTA's share of job j, from its tile to the warps' keys ----
    auto reduce = [&](uint32_t j, const uint4* tile) {
        RangeFold<T> fold;
        for (uint32_t i = 0; i < cnt; ++i) {
            Pack<T> p;
            p.raw = tile[i * kTWork];
            fold.add(p);
        }
        float m0, m1;
        fold.result(m0, m1);
        uint32_t ka = m0 <= m1 ? ~enc(m0) : 0u, kb = m0 <= m1 ? enc(m1) : 0u;
        ka = __reduce_max_sync(kFullMask, ka);
        kb = __reduce_max_sync(kFullMask, kb);
        if (lane == 0) {
            s_kmn[j & 1][warp] = ka;
            s_kmx[j & 1][warp] = kb;
        }
    };
    // ---- the last warp: publish job j's keys, wait (bounded) until the whole team has; Eq. 5 ----
    auto hand_over = [&](uint32_t j) {
        uint32_t ti, c;
        job(j, ti, c);
        const TTensor& t = list.t[ti];
        const uint32_t ka = __reduce_max_sync(kFullMask, lane < kTWork / 32 ? s_kmn[j & 1][lane] : 0u);
        const uint32_t kb = __reduce_max_sync(kFullMask, lane < kTWork / 32 ? s_kmx[j & 1][lane] : 0u);
        if (lane != 0) return;
        atomicMax(t.kmin + c, ka);
        atomicMax(t.kmax + c, kb);
        t_arrive_release(t.counters + c);
        uint32_t ready = 0;
        for (uint32_t i = 0; i < a.spin_limit; ++i) {
            if (ld_acquire(t.counters + c) >= a.expected) {
                ready = 1;
                break;
            }
            __nanosleep(32);
        }
        if (!ready) {
            s_bad = j;
            for (uint32_t k = 0; k < list.n; ++k) atomicExch(list.t[k].status, kTStatusTimeout);
            return;
        }
        float lo, hi;
        const GroupParam gp = group_param_from_keys(t.kmin, t.kmax, c, t.qmax, lo, hi);
        s_par[j & 1] = gp;
        if (rank == 0) {
            t.lo[c] = lo;
            t.hi[c] = hi;
            if (t.s_out) t.s_out[c] = gp.s;
            if (t.z_out) t.z_out[c] = gp.z;
        }
    };
    // ---- Eq. 1, clamp, Eq. 6, STE of job j from its tile; the copies of job j + depth follow on the heels ----
    auto quantize = [&](uint32_t j, uint4* tile) {
        const GroupParam g = s_par[j & 1];
        const bool more = j + depth < jobs;
        uint32_t ti, c;
        job(more ? j + depth : j, ti, c);
        const uint4* xn = reinterpret_cast<const uint4*>(list.t[ti].x) + (size_t)c * a.plane_units;
        job(j, ti, c);
        const size_t base = (size_t)c * a.plane_units;
        const uint4* gyg = reinterpret_cast<const uint4*>(list.t[ti].gy) + base;
        uint4* yg = reinterpret_cast<uint4*>(list.t[ti].y) + base;
        uint4* gxg = reinterpret_cast<uint4*>(list.t[ti].gx) + base;
        const float qmax = list.t[ti].qmax;
        auto emit = [&](const Pack<T>& px, const Pack<T>& pg, uint32_t at) {
            Pack<T> py, pgx;
            uint32_t cb[V / 4], mb[V / 4];
            quantize_own<T, true, 0>(px, pg, g, qmax, py, pgx, cb, mb);
            st_stream_16(yg + at, py.raw);
            st_stream_16(gxg + at, pgx.raw);
        };
        uint32_t at = first, off = off0, i = 0;
        for (; i + U <= cnt; i += U) {
            Pack<T> px[U], pg[U];
            uint32_t w[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                w[k] = at;
                pg[k].raw = ld_stream_16(gyg + at);
                px[k].raw = tile[(i + k) * kTWork];
                advance(at, off);
            }
            if (more) {
#pragma unroll
                for (int k = 0; k < U; ++k) cp_async_16(tile + (i + k) * kTWork, xn + w[k]);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) emit(px[k], pg[k], w[k]);
        }
        for (; i < cnt; ++i) {
            Pack<T> px, pg;
            pg.raw = ld_stream_16(gyg + at);
            px.raw = tile[i * kTWork];
            if (more) cp_async_16(tile + i * kTWork, xn + at);
            emit(px, pg, at);
            advance(at, off);
        }
    };

    if (tid == 0) s_bad = 0xFFFFFFFFu;
    if (!a.early) after_the_kernel_ahead();
    // the first copies; those of the later jobs are sent from the quantize walk
    for (uint32_t j = 0; j < depth && j < jobs; ++j) {
        uint32_t ti, c;
        job(j, ti, c);
        const uint4* xg = reinterpret_cast<const uint4*>(list.t[ti].x) + (size_t)c * a.plane_units;
        uint4* tile = t_smem + j * a.tile_units + tid;
        uint32_t at = first, off = off0;
        for (uint32_t i = 0; i < cnt; ++i) {
            cp_async_16(tile + i * kTWork, xg + at);
            advance(at, off);
        }
    }
    if (a.early) after_the_kernel_ahead();
    for (uint32_t t = 0; t <= jobs; ++t) {
        if (t < jobs) {
            t_cp_async_wait_all();
            if (warp < kTWork / 32) reduce(t, t_smem + (t & 1) * a.tile_units + tid);
        }
        __syncthreads();
        // job t's wait may run out while a slow warp is still here: it looks at the jobs before
        if (t > 0 && *(volatile uint32_t*)&s_bad < t) break;
        if (t < jobs && warp == kTWork / 32) hand_over(t);
        if (t > 0) quantize(t - 1, t_smem + ((t - 1) & 1) * a.tile_units + tid);
    }
    if (*(volatile uint32_t*)&s_bad < jobs) {      // a wait has run out: nothing may be in flight when the CTA leaves
        t_cp_async_wait_all();
        return;
    }

    // ---- leave the workspaces as they were found: the last CTA to finish clears keys and counters ----
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = (atomicAdd(list.t[0].counters + a.C, 1u) == gridDim.x - 1) ? 1u : 0u;
    }
    __syncthreads();
    if (s_last) {
        for (uint32_t t = 0; t < list.n; ++t)
            for (uint32_t i = tid; i <= a.C; i += kTThreads) {
                if (i < a.C) list.t[t].kmin[i] = list.t[t].kmax[i] = 0;
                list.t[t].counters[i] = 0;
            }
    }
}

template <typename T, int MODE, int EXTRAS, int BITS = 8>
cudaError_t t_launch(const TArgs& args, const TeamPlan& p, const StagedTuning& tune, cudaStream_t st) {
    constexpr int U = MODE == MODE_FWD ? 4 : 2;
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kTSmemUnits * 16);
        if (e != cudaSuccess) return e;
        void* params[] = {(void*)&args};
        return launch_cooperative((const void*)kern, args.R * args.teams, p.threads, params, p.smem_bytes, tune, st);
    };
    if constexpr (MODE == MODE_FWD) {
        if (p.threads == kTThreads / 2) return go(colteam_kernel<T, MODE, EXTRAS, U, BITS, uint32_t, kTThreads / 2>);
    }
    return (uint64_t)args.units * args.C < (1ull << 32) ? go(colteam_kernel<T, MODE, EXTRAS, U, BITS, uint32_t, kTThreads>)
                                                        : go(colteam_kernel<T, MODE, EXTRAS, U, BITS, uint64_t, kTThreads>);
}

template <typename T>
cudaError_t t_launch_lag(const TArgs& args, const TList& list, const TeamPlan& p, const StagedTuning& tune, cudaStream_t st) {
    auto launch = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kTSmemUnits * 16);
        if (e != cudaSuccess) return e;
        void* params[] = {(void*)&args, (void*)&list};
        return launch_cooperative((const void*)kern, args.R * args.teams, kTThreads, params, p.smem_bytes, tune, st);
    };
    if constexpr (sizeof(T) == 4) {
        if (list.n > 1) return launch(colteam_lag_kernel<T, 2, true>);
    }
    return list.n == 1 ? launch(colteam_lag_kernel<T, 2, false>) : cudaErrorInvalidValue;      // lists are fp32
}

template <typename T>
cudaError_t t_launch_mode(const TArgs& a, int mode, int extras, const TeamPlan& p, const StagedTuning& tune, cudaStream_t st) {
    if (mode == MODE_BOTH) return t_launch<T, MODE_BOTH, 0>(a, p, tune, st);
    switch (extras) {
        case 2: return t_launch<T, MODE_FWD, 2>(a, p, tune, st);
        case 3:
            switch (a.code_bits) {
                case 1: return t_launch<T, MODE_FWD, 3, 1>(a, p, tune, st);
                case 2: return t_launch<T, MODE_FWD, 3, 2>(a, p, tune, st);
                case 3: return t_launch<T, MODE_FWD, 3, 3>(a, p, tune, st);
                case 4: return t_launch<T, MODE_FWD, 3, 4>(a, p, tune, st);
                case 5: return t_launch<T, MODE_FWD, 3, 5>(a, p, tune, st);
                case 6: return t_launch<T, MODE_FWD, 3, 6>(a, p, tune, st);
                case 7: return t_launch<T, MODE_FWD, 3, 7>(a, p, tune, st);
                default: return t_launch<T, MODE_FWD, 3, 8>(a, p, tune, st);
            }
        case 4: return t_launch<T, MODE_FWD, 4>(a, p, tune, st);
        default: return t_launch<T, MODE_FWD, 0>(a, p, tune, st);
    }
}

}  // namespace

// Team size: the number of CTAs R for which rounds x (share of one CTA + what a hand-over costs) is smallest, the
// share fitting the shared memory of one of two CTAs per SM.
TeamPlan plan_colteam(int dtype, const Geom& g, const QuantIO& io, bool backward, int sm_count, const StagedTuning& tune,
                      uint32_t tensors) {
    TeamPlan p{};
    p.ok = false;
    const uint32_t V = dtype == 0 ? 4 : 8;
    // whole units; codes and masks are written 8 elements at a time
    if (g.inner % V != 0 || g.C * tensors >= (1ll << 28) || g.inner >= (1ll << 28)) return p;
    if ((io.pmask || io.pcodes) && g.inner % 8 != 0) return p;
    if (io.codes || io.mask) return p;
    const uint64_t units = (uint64_t)g.outer * (uint64_t)(g.inner / V);
    if (g.outer > 1 && (uint64_t)g.C * (uint64_t)(g.inner / V) >= (1ull << 32)) return p;      // the stride of slabs is 32 bits
    const uint32_t ctas = 2u * (uint32_t)sm_count;
    if (units >= (1ull << 30) || units > (uint64_t)ctas * (kTSmemUnits - 8)) return p;
    // What a hand-over costs, in units that one CTA moves meanwhile: about 3 us, from sweeps over R (forward
    // [128,64,56,56]: 4 rounds of 5576 units 47 us, 8 of 2720 60 us, 16 of 1360 85 us; with gradient 84, 90, 115 us).  With a
    // gradient and several rounds, two channels side by side hide most of it: [256,512,28,28] 32 rounds of 2792 units 283 us, 29
    // of 3136 291, 43 of 2096 293, one channel at a time 14 of 6272 300; [128,96,112,112] 48 of 2720 433, 24 of 5432 476;
    // [128,64,56,56] 8 of 2720 78, 4 of 6272 84; bf16 [128,96,112,112] 24 of 2720 218, 20 of 3408 222, 12 of 5432 242, but
    // [256,512,28,28] 16 of 2792 163, one channel at a time 7 of 6272 158.
    // Two channels side by side halve the share, and many short rounds lose all the same: from 1700 units each on (one / two channels /
    // waves, us: f32 [140,7,96,97] at 1104 units 36 / 42 / 40, [92,11,128,127] at 1264 58 / 66 / 65, [11,90,96,96] at 1584 33.1 / 35.1 /
    // 35.3, then [166,31,40,40] at 1800 32.7 / 32.0 / 34.7, [212,366,40,40] at 2296 346 / 341 / 400, [112,111,56,56] at 2376 120 / 112 /
    // 131; bf16 [91,31,112,112] at 1936 63 / 59 / 70).  Where that leaves none it is one channel, or the waves.  For a list the
    // other side is separate calls, and whoever plans it weighs those.
    const uint32_t runs = (uint32_t)((units + 7) / 8), C = tensors * (uint32_t)g.C;
    const uint32_t least = tensors > 1 || tune.col_team == 1 ? 0u : kTLagUnits;
    uint64_t best = ~0ull;
    bool one_round = false;
    const int most = backward && units * (uint64_t)g.C < (1ull << 32) ? 2 : 1;      // two channels: 32-bit unit indexes
    for (int depth = 1; depth <= most && !one_round; ++depth) {
        const uint32_t hand_over = depth == 2 ? (dtype == 0 ? 250 : 340) : backward ? 700 : 2000;
        for (uint32_t R = 1; R <= ctas && R <= runs; ++R) {
            const uint32_t share = 8 * ((runs + R - 1) / R);
            if (depth * share > kTSmemUnits || (depth == 2 && share < least)) continue;
            const uint32_t teams = std::min(ctas / R, C), rounds = (C + teams - 1) / teams;
            one_round |= rounds == 1;
            const uint64_t cost = (uint64_t)rounds * (share + hand_over);
            if (cost < best) {
                best = cost;
                p.R = R;
                p.teams = teams;
                p.tile_units = share;
                p.lag = depth == 2;
            }
        }
    }
    if (best == ~0ull) return p;
    p.threads = kTThreads;
    p.sm_count = (uint32_t)sm_count;
    p.gy_units = backward && !p.lag ? std::min(p.tile_units, kTSmemUnits - p.tile_units) : 0u;
    p.smem_bytes = 16u * ((p.lag ? 2 : 1) * p.tile_units + p.gy_units);
    p.ok = true;
    return p;
}

namespace {

// Forward, four CTAs of half the threads and half the shared memory per SM: a finer cut, which is worth having where it saves a round
// or more of several (two / four, us: fp32 [87,240,56,56], 10 / 9 rounds, 111 / 102, with sums 109 / 103, codes 123 / 120.5; [60,200,48,48], 5 / 4,
// 51.6 / 47.3; [49,608,56,56], 13 / 12, 141 / 137; bf16 [128,96,112,112], 12 / 10, 139 / 135; but fp32 [150,60,56,56], 4 / 4, 49.9 / 53.1, codes of
// [64,64,112,112], 8 / 8, 103.6 / 107.0, and anything of one or two rounds), and of y alone or with a packed mask in bf16 also at the same rounds in
// teams of up to 16 CTAs: [200,300,40,40], teams of 13, 85.7 / 82.9 and 88.2 / 85.1; [87,240,56,56], 12, 63.0 / 62.1 and 67.0 / 64.5; [26,393,88,88],
// 10, 72.4 / 70.9 and 75.0 / 73.7; [90,700,32,32], 4, 59.9 / 57.5 and 63.7 / 63.8; [256,512,28,28], 8, 87.6 / 87.6 and 93.0 / 94.1.  Larger teams
// wait for the last of more CTAs: [300,200,44,44], 23, 101.0 / 102.4; [156,102,68,68], 28, 68.2 / 69.7 and 69.4 / 70.5; [246,99,52,52], 29, 62.4 /
// 64.0; [247,25,104,104], 98, packed mask 68.5 / 71.2.  The plan that was asked about stays that of two CTAs per SM.
TeamPlan finer_cut(const TeamPlan& plan, const QuantIO& io, int dtype, const Geom& g, const StagedTuning& tune) {
    const uint32_t C = (uint32_t)g.C, rounds = (C + plan.teams - 1) / plan.teams;
    const uint64_t units = (uint64_t)g.outer * (uint64_t)(g.inner / (dtype == 0 ? 4 : 8));
    if (rounds < 5 || tune.col_team == 1 || units * C >= (1ull << 32)) return plan;
    const uint32_t ctas = 4u * plan.sm_count, runs = (uint32_t)((units + 7) / 8);
    uint64_t best = ~0ull;
    TeamPlan f = plan;
    for (uint32_t R = 1; R <= ctas && R <= runs; ++R) {
        const uint32_t share = 8 * ((runs + R - 1) / R);
        if (share > kTSmemUnits / 2) continue;
        const uint32_t teams = std::min(ctas / R, C);
        const uint64_t cost = (uint64_t)((C + teams - 1) / teams) * (share + 1000);
        if (cost < best) {
            best = cost;
            f.R = R;
            f.teams = teams;
            f.tile_units = share;
        }
    }
    const uint32_t finer = (C + f.teams - 1) / f.teams;
    if (best == ~0ull || f.tile_units < 2500 || !(finer < rounds || (finer == rounds && dtype == 1 && f.R <= 16 && !io.dist && !io.pcodes))) return plan;
    f.smem_bytes = 16u * f.tile_units;
    f.threads = kTThreads / 2;
    return f;
}

}  // namespace

cudaError_t launch_colteam_list(const TeamPlan& plan, const TeamTensor* tensors, uint32_t n, int dtype, const Geom& g,
                                const StagedTuning& tune, cudaStream_t st) {
    TArgs a{};
    a.C = (uint32_t)g.C;
    a.plane_units = (uint32_t)(g.inner / (dtype == 0 ? 4 : 8));
    a.units = (uint32_t)((uint64_t)g.outer * a.plane_units);
    a.slab_units = (uint32_t)((uint64_t)a.C * a.plane_units);
    a.R = plan.R;
    a.teams = plan.teams;
    a.tile_units = plan.tile_units;
    a.spin_limit = tune.spin_limit > 0 ? (uint32_t)tune.spin_limit : kTSpinLimit;
    a.expected = plan.R + (uint32_t)(tune.extra_arrivals > 0 ? tune.extra_arrivals : 0);
    a.early = n == 1 && tensors[0].ws.cleared ? 1u : 0u;
    a.div_plane = make_fastdiv(a.plane_units);
    TList list{};
    list.n = n;
    list.div_C = make_fastdiv(a.C);
    for (uint32_t i = 0; i < n; ++i) {
        const TeamTensor& t = tensors[i];
        list.t[i] = {t.io.x, t.io.gy, t.io.y, t.io.gx, t.ws.status, t.ws.kmin, t.ws.kmax, t.ws.counters, t.lo, t.hi,
                     t.s_opt, t.z_opt, (float)((1 << t.bits) - 1)};
    }
    return dtype == 0 ? t_launch_lag<float>(a, list, plan, tune, st) : t_launch_lag<__nv_bfloat16>(a, list, plan, tune, st);
}

cudaError_t launch_colteam(const TeamPlan& asked, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                           const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                           const StagedTuning& tune, cudaStream_t st) {
    const uint32_t V = dtype == 0 ? 4 : 8;
    if (asked.lag) {
        const TeamTensor one{io, bits, ws, lo, hi, s_opt, z_opt};
        return launch_colteam_list(asked, &one, 1, dtype, g, tune, st);
    }
    TArgs a{};
    a.x = io.x;
    a.gy = io.gy;
    a.y = io.y;
    a.gx = io.gx;
    a.pmask = io.pmask;
    a.pcodes = io.pcodes;
    a.code_bits = io.code_bits;
    a.code_words = g.inner % 32 == 0 ? 1u : 0u;
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
    a.C = (uint32_t)g.C;
    a.plane_units = (uint32_t)(g.inner / V);
    a.units = (uint32_t)((uint64_t)g.outer * a.plane_units);
    a.slab_units = (uint32_t)((uint64_t)a.C * a.plane_units);
    a.spin_limit = tune.spin_limit > 0 ? (uint32_t)tune.spin_limit : kTSpinLimit;
    a.early = ws.cleared ? 1u : 0u;
    a.div_plane = make_fastdiv(a.plane_units);
    const int extras = io.dist ? 4 : io.pmask ? 2 : io.pcodes ? 3 : 0;
    auto go = [&](const TeamPlan& plan) -> cudaError_t {
        a.R = plan.R;
        a.teams = plan.teams;
        a.tile_units = plan.tile_units;
        a.gy_units = plan.gy_units;
        a.expected = plan.R + (uint32_t)(tune.extra_arrivals > 0 ? tune.extra_arrivals : 0);
        return dtype == 0 ? t_launch_mode<float>(a, mode, extras, plan, tune, st)
                          : t_launch_mode<__nv_bfloat16>(a, mode, extras, plan, tune, st);
    };
    const TeamPlan plan = mode == MODE_FWD ? finer_cut(asked, io, dtype, g, tune) : asked;
    const cudaError_t e = go(plan);
    // where the GPU does not hold the finer cut's CTAs at once it may hold those asked for
    return e == cudaErrorCooperativeLaunchTooLarge && plan.threads != asked.threads ? go(asked) : e;
}

}  // namespace granq
