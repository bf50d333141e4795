// Channels-last GranQ kernel: geometries whose channel is the innermost axis ([N, H, W, C] with the
// channel axis last, or [N, C, 1, 1]), i.e. a row-major matrix [rows, C] with one group per column.
//
// Every channel is spread over the whole tensor, so nothing can be quantized before all of it has been read.  One
// cooperative launch, two CTAs per SM.  The matrix is cut into slices of 16 .. 64 unit columns (a 16-byte unit holds V
// consecutive channels), and a team of CTAs owns a slice: channels of different slices have nothing to do with each
// other, so what a CTA does per channel (keys, atomics, parameters) stays small however wide the rows are, and nobody
// waits for another slice.  The CTAs of a team take turns at blocks of rows; each keeps its blocks in shared memory
// between the two halves of the work where all of them fit (33 MB over the GPU):
//   range (Eq. 4):  rows that will be kept are sent for with per-thread asynchronous copies, others are read
//                   directly; a thread keeps ONE unit column, its running min / max per channel are folded
//                   in shared memory and reach global memory as one pair of atomics per channel and CTA;
//   hand-over:      one arrival per CTA and a bounded wait for the team;
//   quantize (Eq. 5, 1, 6, STE): the CTA turns the slice's keys into a table of parameters once; a thread loads the V
//                   sets of its column and streams, from shared memory or, rows that were not kept, from memory again: the
//                   last read first, as the likeliest to still be in the L2.
// Neither half divides an index or looks anything up inside the walk.
// Bound by HBM for the streams of the second half, by the hand-over (about 3 us) for small tensors.  Against a
// range launch and a quantize launch that spread every channel over all CTAs (us, forward / with gradient): bf16
// [128,28,28,192] 42 / 49 -> 31 / 42, [17,14,14,2048] 30 / 36 -> 19 / 23; fp32 [15,22,22,784] 30 / 38 -> 19 / 28,
// [31,28,28,2048] 134 / 179 -> 101 / 162, [16,32,32,16] 17 / 18 -> 10 / 10; [128,112,112,64] 243 / 327 -> 208 / 336.
#include "granq_internal.h"

#include <algorithm>

namespace granq {

namespace {

// Threads of a CTA at most: two CTAs leave 72 registers per thread to fp32 and 80 to bf16 (V sets of parameters each).
template <typename T>
constexpr int kRMaxThreads = Pack<T>::V == 4 ? 448 : 384;
constexpr uint32_t kRMaxChannels = 4096;      // 64 slices at most
constexpr uint32_t kRSmemBytes = 111u * 1024; // of one of two CTAs on an SM
// From here on gy is sent for during the hand-over; a smaller one is most often still in the L2, and asking for it again costs
// what it takes.  With gradient, us, gy in memory | gy in the L2: [32,28,28,128] fp32, 13 MB, 23.5 -> 21.4 | 14.8 -> 15.4;
// [61,35,34,56] fp32, 16 MB, 25.6 -> 23.5 | 16.1 -> 16.6; [134,71,70,8] fp32, 21 MB, 28.4 -> 25.5 | 18.9 -> 18.8; [64,14,14,512]
// fp32, 26 MB, 31.2 -> 29.7 | 22.4 -> 20.7; [17,14,14,2048] fp32, 27 MB, 31.7 -> 29.7 | 22.8 -> 20.9.
constexpr uint64_t kRFetchBytes = 20ull << 20;
constexpr uint32_t kRSpinLimit = 1u << 24;    // bounded wait on the grid (x ~32 ns)
constexpr uint32_t kRStatusTimeout = 5;       // GRANQ_ERR_TIMEOUT

struct RArgs {
    const void* x;
    const void* gy;
    void* y;
    void* gx;
    uint8_t* codes;
    uint8_t* mask;
    uint32_t* status;
    uint32_t* kmin;
    uint32_t* kmax;
    uint32_t* counters;
    float* lo;
    float* hi;
    float* s_out;
    float* z_out;
    float qmax;
    uint32_t C;          // channels
    uint32_t ncol;       // 16-byte units per row
    uint32_t P;          // unit columns of a slice
    uint32_t slices;
    uint32_t team;       // CTAs per slice
    uint32_t lanes;      // rows of threads: the rows of one block
    uint32_t hold;       // blocks of rows a CTA keeps in shared memory
    uint32_t lost;       // of the others, those before this one are not expected to be in the L2 when they are read again
    uint32_t spin_limit, expected;
    uint32_t fetch;      // what the kept blocks meet of gy is sent for during the hand-over
    uint32_t early;      // x may be read before the kernel ahead has completed: it only clears the workspace
    uint64_t rows;
};

// U1 / U2 = rows a thread has in flight in the range / quantize walk
template <typename T, int MODE, bool EXTRAS, int U1, int U2>
__global__ void __launch_bounds__(kRMaxThreads<T>, 2) rows_kernel(const RArgs a) {
    constexpr int V = Pack<T>::V;
    constexpr bool kBwd = (MODE & MODE_BWD) != 0;
    extern __shared__ __align__(16) unsigned char r_smem[];
    // first the keys (min, max: element i of unit column c at i * P + c), later the parameter table, then the rows
    uint32_t* s_kmn = reinterpret_cast<uint32_t*>(r_smem);
    uint32_t* s_kmx = s_kmn + a.P * V;
    GroupParam* s_par = reinterpret_cast<GroupParam*>(r_smem);
    __shared__ uint32_t s_ok;
    const uint32_t tid = threadIdx.x, NT = blockDim.x, P = a.P, L = a.lanes;
    const uint32_t slice = blockIdx.x / a.team, rank = blockIdx.x - slice * a.team;
    const uint32_t col0 = slice * P, width = min(P, a.ncol - col0), ch0 = col0 * V, chans = width * V;
    const uint32_t r0 = tid / P, cin = tid - r0 * P;
    // this thread's rows: row first + k * stride, k < n; the first `held` of them stay in shared memory
    const uint64_t first = (uint64_t)rank * L + r0, stride = (uint64_t)a.team * L;
    const uint32_t n = (r0 < L && cin < width && first < a.rows) ? (uint32_t)((a.rows - 1 - first) / stride) + 1 : 0u;
    const uint32_t held = min(n, a.hold);
    const uint64_t origin = first * a.ncol + col0 + cin;
    const size_t step = (size_t)stride * a.ncol;
    const uint4* xg = reinterpret_cast<const uint4*>(a.x) + origin;
    const uint4* gyg = reinterpret_cast<const uint4*>(a.gy) + origin;
    uint4* yg = reinterpret_cast<uint4*>(a.y) + origin;
    uint4* gxg = reinterpret_cast<uint4*>(a.gx) + origin;
    uint4* tile = reinterpret_cast<uint4*>(r_smem + (size_t)P * V * sizeof(GroupParam)) + r0 * P + cin;
    const uint32_t tstep = L * P;
    const float qmax = a.qmax;
    const uint64_t drop = l2_policy_evict_first();

    if (!a.early) after_the_kernel_ahead();
    for (uint32_t k = 0; k < held; ++k) cp_async_16(tile + k * tstep, xg + k * step);
    for (uint32_t t = tid; t < 2 * P * V; t += NT) s_kmn[t] = 0;
    __syncthreads();

    // ---- Eq. 4: rows beyond the kept ones straight from memory, then the kept ones ----
    {
        RangeColumn<T> acc;
        acc.reset();
        const uint4* src = xg + held * step;
        for (uint32_t k = held; k < n; k += U1, src += U1 * step) {
            Pack<T> v[U1];
#pragma unroll
            for (int j = 0; j < U1; ++j)
                if (k + j < n) v[j].raw = k < a.lost ? ld_hint_16(src + j * step, drop) : __ldg(src + j * step);
#pragma unroll
            for (int j = 0; j < U1; ++j)
                if (k + j < n) acc.add(v[j]);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        for (uint32_t k = 0; k < held; ++k) {
            Pack<T> v;
            v.raw = tile[k * tstep];
            acc.add(v);
        }
        if (n > 0) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                uint32_t ka, kb;
                column_keys(acc, i, i + 1, ka, kb);
                atomicMax(s_kmn + i * P + cin, ka);
                atomicMax(s_kmx + i * P + cin, kb);
            }
        }
    }
    if (a.early) after_the_kernel_ahead();
    __syncthreads();
    for (uint32_t t = tid; t < chans; t += NT) {           // channel t of the slice: element t % V of unit column t / V
        const uint32_t at = (t % V) * P + t / V, k1 = s_kmn[at], k2 = s_kmx[at];
        if (k1 | k2) {
            atomicMax(a.kmin + ch0 + t, k1);
            atomicMax(a.kmax + ch0 + t, k2);
        }
    }
    // ---- the team's hand-over (bounded) ----
    if constexpr (kBwd) {
        if (a.fetch) {
            if (a.slices == 1) {                           // a block of rows is one piece
                const uint64_t row0 = ((uint64_t)rank + (uint64_t)tid * a.team) * L;
                if (tid < a.hold && row0 < a.rows) prefetch_l2(reinterpret_cast<const uint4*>(a.gy) + row0 * a.ncol, (uint32_t)min((uint64_t)L, a.rows - row0) * a.ncol * 16u);
            } else if (cin == 0) {
                for (uint32_t k = 0; k < held; ++k) prefetch_l2(gyg + k * step, width * 16u);
            }
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        atomicAdd(a.counters + slice, 1u);
        uint32_t ready = 0;
        for (uint32_t i = 0; i < a.spin_limit; ++i) {
            if (ld_acquire(a.counters + slice) >= a.expected) {
                ready = 1;
                break;
            }
            __nanosleep(32);
        }
        s_ok = ready;
        if (!ready) atomicExch(a.status, kRStatusTimeout);
    }
    __syncthreads();
    if (!s_ok) return;
    for (uint32_t t = tid; t < chans; t += NT) {
        float lo, hi;
        const GroupParam gp = group_param_from_keys(a.kmin, a.kmax, ch0 + t, qmax, lo, hi);
        s_par[t] = gp;
        if (rank == 0) {
            a.lo[ch0 + t] = lo;
            a.hi[ch0 + t] = hi;
            if (a.s_out) a.s_out[ch0 + t] = gp.s;
            if (a.z_out) a.z_out[ch0 + t] = gp.z;
        }
    }
    __syncthreads();
    if (tid == 0) {          // the keys have been read; the last CTA to say so leaves the workspace zero (below)
        __threadfence();
        s_ok = (atomicAdd(a.counters + a.slices, 1u) == gridDim.x - 1) ? 1u : 0u;
    }

    // ---- Eq. 1, clamp, Eq. 6, STE ----
    if (n > 0) {
        const GroupParam* par = s_par + cin * V;
        float s[V], rc[V], mz[V], thr = 1.0f;
        bool clamped = false;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const GroupParam g = par[i];
            s[i] = g.s;
            rc[i] = g.r;
            mz[i] = __fadd_rn(kRoundMagic, g.z);
            thr = fminf(thr, fabsf(g.thr));
            clamped |= g.thr < 0.0f;
        }
        if (clamped) thr = -thr;
        auto emit = [&](const Pack<T>& px, const Pack<T>& pg, size_t at) {
            Pack<T> py, pgx;
            uint32_t cb[V / 4], mb[V / 4];
            quantize_pack_each<T, kBwd, EXTRAS>(px, pg, s, rc, mz, thr, par, qmax, py, pgx, cb, mb);
            st_stream_16(yg + at, py.raw);
            if constexpr (kBwd) st_stream_16(gxg + at, pgx.raw);
            if constexpr (EXTRAS) {
                const size_t w = (origin + at) * (V / 4);
                if (a.codes) {
#pragma unroll
                    for (int i = 0; i < V / 4; ++i) reinterpret_cast<uint32_t*>(a.codes)[w + i] = cb[i];
                }
                if (kBwd && a.mask) {
#pragma unroll
                    for (int i = 0; i < V / 4; ++i) reinterpret_cast<uint32_t*>(a.mask)[w + i] = mb[i];
                }
            }
        };
        // rows that were not kept, from the last one back
        {
            uint32_t left = n - held;
            size_t at = (size_t)(n - 1) * step;
            for (; left >= (uint32_t)U2; left -= U2, at -= U2 * step) {
                Pack<T> px[U2], pg[U2];
#pragma unroll
                for (int j = 0; j < U2; ++j) {
                    px[j].raw = ld_stream_16(xg + (at - j * step));
                    if constexpr (kBwd) pg[j].raw = ld_stream_16(gyg + (at - j * step));
                }
#pragma unroll
                for (int j = 0; j < U2; ++j) emit(px[j], pg[j], at - j * step);
            }
            for (; left > 0; --left, at -= step) {
                Pack<T> px, pg;
                px.raw = ld_stream_16(xg + at);
                if constexpr (kBwd) pg.raw = ld_stream_16(gyg + at);
                emit(px, pg, at);
            }
        }
        // the kept ones
        size_t at = 0;
        uint32_t k = 0;
        for (; k + U2 <= held; k += U2, at += U2 * step) {
            Pack<T> px[U2], pg[U2];
#pragma unroll
            for (int j = 0; j < U2; ++j)
                if constexpr (kBwd) pg[j].raw = ld_stream_16(gyg + at + j * step);
#pragma unroll
            for (int j = 0; j < U2; ++j) px[j].raw = tile[(k + j) * tstep];
#pragma unroll
            for (int j = 0; j < U2; ++j) emit(px[j], pg[j], at + j * step);
        }
        for (; k < held; ++k, at += step) {
            Pack<T> px, pg;
            if constexpr (kBwd) pg.raw = ld_stream_16(gyg + at);
            px.raw = tile[k * tstep];
            emit(px, pg, at);
        }
    }
    __syncthreads();
    if (s_ok) {
        for (uint32_t t = tid; t < a.C; t += NT) {
            a.kmin[t] = 0;
            a.kmax[t] = 0;
        }
        for (uint32_t t = tid; t <= a.slices; t += NT) a.counters[t] = 0;
    }
}

bool r_aligned16(const void* p) { return p == nullptr || ((uintptr_t)p & 15) == 0; }

template <typename T, int MODE>
cudaError_t r_launch(const RArgs& a, bool extras, int grid, int threads, size_t smem, const StagedTuning& tune, cudaStream_t st) {
    auto go = [&](auto kern) -> cudaError_t {
        const cudaError_t e = allow_smem(kern, kRSmemBytes);
        if (e != cudaSuccess) return e;
        void* params[] = {(void*)&a};
        return launch_cooperative((const void*)kern, (uint32_t)grid, (uint32_t)threads, params, smem, tune, st);
    };
    constexpr int U1 = Pack<T>::V == 4 ? 8 : 6;
    return extras ? go(rows_kernel<T, MODE, true, U1, 2>) : go(rows_kernel<T, MODE, false, U1, 2>);
}

}  // namespace

// inner == 1 (the channel is the innermost axis), rows of whole 16-byte units, everything 16-byte aligned
bool plan_rows(int dtype, const Geom& g, const QuantIO& io) {
    const int64_t V = dtype == 0 ? 4 : 8;
    if (io.pmask || io.dist || io.pcodes) return false;
    if (g.inner != 1 || g.C < V || g.C % V != 0 || g.C > (int64_t)kRMaxChannels || g.outer < 1) return false;
    if (!r_aligned16(io.x) || !r_aligned16(io.gy) || !r_aligned16(io.y) || !r_aligned16(io.gx)) return false;
    if (((uintptr_t)io.codes & 3) || ((uintptr_t)io.mask & 3)) return false;
    return true;
}

// The cut of a row into slices that leaves the fewest threads and CTAs without work (196 unit columns: 7 slices of 28,
// 16 rows of threads each); slices of 64 unit columns at most, of 16 at least where there are several.
// Where a slice ends inside a 32-byte sector or a 128-byte line, two CTAs write the two parts of it at different times.
// A tensor that stays on chip is small enough for the L2 to join the sectors up; of a larger one they go to memory in
// pieces, so its slices are whole lines.  fp32 with a gradient (us): [40,100,100,200] two slices of 25 columns 315, of 26
// 279, one slice of 50 257; [64,56,56,264] 33 columns 192, 24 columns 181; [20,56,56,784] 49 columns 183, 40 columns 169;
// bf16 [40,100,100,400] 324, one slice 297.  On chip: [8,30,30,520] 26 columns 21.0, 48 columns 21.6; bf16 [16,28,28,408]
// 17 columns 21.7, one slice of 51 23.0.
// Threads: all that fit, 448 or 384; with an fp32 gradient beyond 200 MB 400, which is what loads in flight of two
// streams take there ([128,112,112,64] 334 / 327 us, [128,112,112,96] 503 / 491, [64,112,112,128] 333 / 326; 320 threads
// 325, 522, 325; but [128,28,28,192], 77 MB, 63.6 / 64.8).
bool cut_rows(int dtype, const Geom& g, bool backward, uint32_t ctas, RowsCut& cut) {
    const uint32_t V = dtype == 0 ? 4 : 8, ncol = (uint32_t)(g.C / V);
    const uint64_t bytes = (uint64_t)g.outer * ncol * 16;
    const uint32_t most = dtype == 0 ? kRMaxThreads<float> : kRMaxThreads<__nv_bfloat16>;
    const uint32_t top = dtype == 0 && backward && bytes > (200ull << 20) ? 400 : most;
    const uint32_t whole = bytes > (uint64_t)ctas * kRSmemBytes ? 8 : ncol % 2 == 0 ? 2 : 1;      // unit columns
    double best = 0.0;
    for (uint32_t slices = (ncol + 63) / 64; slices <= std::max<uint32_t>(1, ncol / 16); ++slices) {
        const uint32_t share = (ncol + slices - 1) / slices, P = slices > 1 ? (share + whole - 1) / whole * whole : share;
        const uint32_t lanes = top / P, used = (ncol + P - 1) / P;
        const double eff = (double)ncol / (double)(used * P) * (double)(P * lanes) / top * (double)(ctas / used * used) / ctas;
        if (eff > best + (whole == 8 ? 0.05 : 0.02)) {
            best = eff;
            cut.P = P;
            cut.slices = used;
            cut.lanes = lanes;
        }
    }
    if (best == 0.0) return false;
    const uint64_t blocks = ((uint64_t)g.outer + cut.lanes - 1) / cut.lanes;      // no more CTAs than there are blocks of rows
    cut.team = (uint32_t)std::min<uint64_t>(blocks, ctas / cut.slices);
    return true;
}

cudaError_t launch_rows(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, const Workspace& ws,
                        float* lo, float* hi, float* s_opt, float* z_opt, const StagedTuning& tune, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint32_t V = dtype == 0 ? 4 : 8;
    RArgs a{};
    a.x = io.x;
    a.gy = io.gy;
    a.y = io.y;
    a.gx = io.gx;
    a.codes = io.codes;
    a.mask = io.mask;
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
    a.ncol = (uint32_t)(g.C / V);
    a.rows = (uint64_t)g.outer;
    RowsCut cut{};
    if (!cut_rows(dtype, g, mode != MODE_FWD, 2u * (uint32_t)sms, cut)) return cudaErrorCooperativeLaunchTooLarge;
    a.P = cut.P;
    a.slices = cut.slices;
    a.lanes = cut.lanes;
    a.team = cut.team;
    const uint64_t blocks = (a.rows + a.lanes - 1) / a.lanes;
    const int grid = (int)(a.team * a.slices), threads = (int)((a.P * a.lanes + 31) / 32 * 32);
    const size_t table = (size_t)a.P * V * sizeof(GroupParam), block = (size_t)a.P * a.lanes * 16;
    // all of a CTA's blocks or none: loads in flight need L1, which is what shared memory leaves of 256 KB (keeping a
    // part: fp32 [128,112,112,64] with gradient 363 us, none 343; bf16 [128,28,28,192] 38.5 MB, 85 % kept, 33.4 / 31.3)
    const uint64_t per_cta = (blocks + a.team - 1) / a.team;
    a.hold = per_cta <= (kRSmemBytes - table) / block ? (uint32_t)per_cta : 0u;
    const size_t smem = table + a.hold * block;
    // of a tensor that is read twice, the last 64 MB have a chance to still be in the L2: the rest makes way for them
    // ([128,112,112,64] fp32 forward 217 -> 208 us)
    const double tail = 64e6 / ((double)a.rows * a.ncol * 16);
    a.lost = tail < 1.0 ? (uint32_t)((1.0 - tail) * (double)per_cta) : 0u;
    a.fetch = (uint64_t)a.rows * a.ncol * 16 >= kRFetchBytes ? 1u : 0u;
    a.spin_limit = tune.spin_limit > 0 ? (uint32_t)tune.spin_limit : kRSpinLimit;
    a.expected = a.team + (uint32_t)(tune.extra_arrivals > 0 ? tune.extra_arrivals : 0);
    a.early = ws.cleared ? 1u : 0u;
    const bool extras = io.codes != nullptr || io.mask != nullptr;
    if (dtype == 0) {
        if (mode == MODE_FWD) return r_launch<float, MODE_FWD>(a, extras, grid, threads, smem, tune, st);
        return r_launch<float, MODE_BOTH>(a, extras, grid, threads, smem, tune, st);
    }
    if (mode == MODE_FWD) return r_launch<__nv_bfloat16, MODE_FWD>(a, extras, grid, threads, smem, tune, st);
    return r_launch<__nv_bfloat16, MODE_BOTH>(a, extras, grid, threads, smem, tune, st);
}

}  // namespace granq
