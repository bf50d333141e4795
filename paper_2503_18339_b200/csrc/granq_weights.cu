// Channel-wise fake-quantization of many small tensors in one launch (Section 5.1: every weight
// tensor is quantized per output channel).  A weight tensor [channels, group_elems] has one group
// per leading index and each group is a short contiguous run (27 .. a few thousand values).
//
// A group is read once: a team of 1, 2, 4 or 8 warps holds it in registers (kWHold 16-byte units, or single
// elements where groups are not whole units, per lane), reduces it to its range (Eq. 4: warp shuffles, and shared
// memory where the team is more than a warp), works out scale and zero-point (Eq. 5) and quantizes, clamps,
// dequantizes and masks from registers (Eq. 1, 6, STE).  Only what a team of 8 warps cannot hold (beyond 5120 fp32
// elements) is read a second time.  The team is the smallest that holds the group: 3 x 3 kernels of 64 .. 512 input
// channels all come to 4.5 units per lane, so every block moves about 18 KB whatever the tensor, and the block
// scheduler evens out the batch.  The descriptors travel in the kernel's parameters: no copy ahead of the launch,
// and the search for a block's tensor runs over the constant bank.
// Bound by the latency of one read, one reduction and one write per block, four blocks to an SM in turn.  All
// weights of ResNet-18 (11.7 M fp32 elements, 93 MB moved): 40.2 -> 21.5 us a call (a warp per group that read it
// twice took 37 us of kernel, this one 20.6 = 4.5 TB/s).
#include "../../include/granq.h"

#include "granq_internal.h"

#include <vector>

namespace granq {

namespace {

constexpr int kWThreads = 256;
constexpr uint32_t kWWarps = kWThreads / 32;
constexpr int kWHold = 5;               // units (or elements) of a group one lane holds at most
constexpr int kWTail = 4;               // units in flight per lane where a group is more than its team holds

struct WDesc {
    const void* x;
    const void* gy;
    void* y;
    void* gx;
    float* lo;
    float* hi;
    float* s;
    float* z;
    uint32_t channels;
    uint32_t group_elems;
    uint32_t first_block;   // index of this tensor's first block in the launch
    uint32_t team;          // warps per group: 1, 2, 4 or 8
    float qmax;
    uint32_t vec;           // groups start on 16-byte boundaries and are whole packs
};

template <int N>
struct WTable {
    WDesc d[N];
};

// HOLD = units (or elements) of a group one lane holds
template <typename T, bool GRAD, int N, int HOLD>
__global__ void __launch_bounds__(kWThreads, HOLD == 1 ? (GRAD ? 5 : 6) : GRAD ? 3 : 4) weights_kernel(const __grid_constant__ WTable<N> tab, uint32_t n) {
    constexpr int V = Pack<T>::V;
    __shared__ float s_mn[kWWarps], s_mx[kWWarps];
    // the tensor of this block: last descriptor with first_block <= blockIdx.x
    uint32_t a = 0, b = n - 1;
    while (a < b) {
        const uint32_t m = (a + b + 1) >> 1;
        if (tab.d[m].first_block <= blockIdx.x) a = m;
        else b = m - 1;
    }
    const WDesc& d = tab.d[a];
    after_the_kernel_ahead();
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, team = d.team;
    const uint32_t c = (blockIdx.x - d.first_block) * (kWWarps / team) + warp / team;      // this team's group
    const bool valid = c < d.channels;
    const uint32_t ge = d.group_elems, stride = team * 32, tl = (warp % team) * 32 + lane;
    const size_t at = (size_t)(valid ? c : 0) * ge;
    const T* x = reinterpret_cast<const T*>(d.x) + at;
    const T* gy = reinterpret_cast<const T*>(d.gy) + at;
    T* y = reinterpret_cast<T*>(d.y) + at;
    T* gx = reinterpret_cast<T*>(d.gx) + at;
    const bool grad = GRAD && d.gy != nullptr;
    const uint32_t units = valid ? (d.vec ? ge / V : ge) : 0;
    const uint32_t held = HOLD * stride;          // with one unit a lane: the whole group

    // ---- Eq. 4: the group's range; the group stays in registers ----
    Pack<T> px[HOLD], pg[GRAD ? HOLD : 1];
    float sx[HOLD], sg[GRAD ? HOLD : 1];
    float mn = INFINITY, mx = -INFINITY;
    if (d.vec) {
#pragma unroll
        for (int j = 0; j < HOLD; ++j) {
            const uint32_t u = tl + j * stride;
            if (u < units) px[j].raw = ld_stream_16(x + (size_t)u * V);
        }
        if constexpr (GRAD) {
            if (grad) {
#pragma unroll
                for (int j = 0; j < HOLD; ++j) {
                    const uint32_t u = tl + j * stride;
                    if (u < units) pg[j].raw = ld_stream_16(gy + (size_t)u * V);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < HOLD; ++j)
            if (tl + j * stride < units) pack_minmax(px[j], 0, V, mn, mx);
        if constexpr (HOLD > 1)
            for (uint32_t u = held + tl; u < units; u += kWTail * stride) {
                Pack<T> p[kWTail];
#pragma unroll
                for (int j = 0; j < kWTail; ++j)
                    if (u + j * stride < units) p[j].raw = *reinterpret_cast<const uint4*>(x + (size_t)(u + j * stride) * V);
#pragma unroll
                for (int j = 0; j < kWTail; ++j)
                    if (u + j * stride < units) pack_minmax(p[j], 0, V, mn, mx);
            }
    } else {
#pragma unroll
        for (int j = 0; j < HOLD; ++j) {
            const uint32_t e = tl + j * stride;
            if (e < units) {
                sx[j] = load_scalar(x + e);
                if constexpr (GRAD) {
                    if (grad) sg[j] = load_scalar(gy + e);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < HOLD; ++j)
            if (tl + j * stride < units) {
                mn = fminf(mn, sx[j]);
                mx = fmaxf(mx, sx[j]);
            }
        if constexpr (HOLD > 1)
            for (uint32_t e = held + tl; e < units; e += stride) {
                const float v = load_scalar(x + e);
                mn = fminf(mn, v);
                mx = fmaxf(mx, v);
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(kFullMask, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, o));
    }
    if (team > 1) {                                  // the same for every thread of the block
        if (lane == 0) {
            s_mn[warp] = mn;
            s_mx[warp] = mx;
        }
        __syncthreads();
        const uint32_t first = warp - warp % team;
        for (uint32_t w = 0; w < team; ++w) {
            mn = fminf(mn, s_mn[first + w]);
            mx = fmaxf(mx, s_mx[first + w]);
        }
    }
    if (!valid) return;
    const float lo = __fadd_rn(mn, 0.0f), hi = __fadd_rn(mx, 0.0f), qmax = d.qmax;      // -0 -> +0
    const GroupParam gp = group_param_from_range(lo, hi, qmax);                         // Eq. 5
    if (tl == 0) {
        d.lo[c] = lo;
        d.hi[c] = hi;
        if (d.s) d.s[c] = gp.s;
        if (d.z) d.z[c] = gp.z;
    }

    // ---- Eq. 1, clamp, Eq. 6, STE ----
    if (d.vec) {
        auto emit = [&](const Pack<T>& p, const Pack<T>& g, uint32_t u) {
            Pack<T> py, pgx;
            uint32_t cb[V / 4], mb[V / 4];
            if constexpr (GRAD) quantize_pack<T, GRAD, false, 0, true>(p, g, gp, gp, V, qmax, py, pgx, cb, mb);
            else quantize_own<T, GRAD, 0>(p, g, gp, qmax, py, pgx, cb, mb);
            st_stream_16(y + (size_t)u * V, py.raw);
            if constexpr (GRAD) {
                if (grad) st_stream_16(gx + (size_t)u * V, pgx.raw);
            }
        };
#pragma unroll
        for (int j = 0; j < HOLD; ++j) {
            const uint32_t u = tl + j * stride;
            if (u < units) emit(px[j], pg[GRAD ? j : 0], u);
        }
        if constexpr (HOLD > 1)
            for (uint32_t u = held + tl; u < units; u += 2 * stride) {
                const bool two = u + stride < units;
                Pack<T> p[2], g[2];
                p[0].raw = *reinterpret_cast<const uint4*>(x + (size_t)u * V);
                if (two) p[1].raw = *reinterpret_cast<const uint4*>(x + (size_t)(u + stride) * V);
                if constexpr (GRAD) {
                    if (grad) {
                        g[0].raw = *reinterpret_cast<const uint4*>(gy + (size_t)u * V);
                        if (two) g[1].raw = *reinterpret_cast<const uint4*>(gy + (size_t)(u + stride) * V);
                    }
                }
                emit(p[0], g[0], u);
                if (two) emit(p[1], g[1], u + stride);
            }
    } else {
        const QParam qp{gp.s, gp.z};
        auto emit = [&](float v, float g, uint32_t e) {
            float yv;
            bool in;
            quant_one(v, qp, qmax, yv, in);
            store_scalar(y + e, yv);
            if constexpr (GRAD) {
                if (grad) store_scalar(gx + e, in ? g : 0.0f);
            }
        };
#pragma unroll
        for (int j = 0; j < HOLD; ++j) {
            const uint32_t e = tl + j * stride;
            if (e < units) emit(sx[j], sg[GRAD ? j : 0], e);
        }
        if constexpr (HOLD > 1)
            for (uint32_t e = held + tl; e < units; e += stride)
                emit(load_scalar(x + e), grad ? load_scalar(gy + e) : 0.0f, e);
    }
}

constexpr int kWSmallTable = 32, kWTable = 256;      // descriptors of one launch (2.9 KB / 23 KB of parameters)

// Launches whose groups are at most a warp's lanes (depthwise kernels, small first layers) hold one unit per lane: fewer
// registers and twice the blocks per SM, which is all such groups are bound by.
template <typename T, bool GRAD, int N>
cudaError_t w_launch_n(const WDesc* descs, int n, uint32_t blocks, cudaStream_t st) {
    constexpr uint32_t V = Pack<T>::V;
    WTable<N> tab;
    bool small = true;
    uint64_t bytes = 0;
    for (int i = 0; i < n; ++i) {
        tab.d[i] = descs[i];
        bytes += (uint64_t)descs[i].channels * descs[i].group_elems * sizeof(T);
        small = small && (descs[i].vec ? descs[i].group_elems / V : descs[i].group_elems) <= 32;
    }
    const int layout = sm_layout(0, bytes);
    if (small) return launch_after(layout, weights_kernel<T, GRAD, N, 1>, blocks, kWThreads, 0, st, tab, (uint32_t)n);
    return launch_after(layout, weights_kernel<T, GRAD, N, kWHold>, blocks, kWThreads, 0, st, tab, (uint32_t)n);
}

template <typename T>
cudaError_t w_launch(const WDesc* descs, int n, uint32_t blocks, bool grad, cudaStream_t st) {
    if (n <= kWSmallTable)
        return grad ? w_launch_n<T, true, kWSmallTable>(descs, n, blocks, st) : w_launch_n<T, false, kWSmallTable>(descs, n, blocks, st);
    return grad ? w_launch_n<T, true, kWTable>(descs, n, blocks, st) : w_launch_n<T, false, kWTable>(descs, n, blocks, st);
}

size_t table_bytes(int n) { return (((size_t)n * sizeof(WDesc)) + 255) & ~(size_t)255; }

}  // namespace

}  // namespace granq

using namespace granq;

extern "C" {

size_t granq_weights_workspace_bytes(int n_tensors) { return n_tensors > 0 ? table_bytes(n_tensors) : 0; }

int granq_fakequant_weights(const granq_weight_desc* descs, int n_tensors, int dtype, void* workspace,
                            size_t workspace_bytes, uint32_t flags, void* cuda_stream) {
    (void)flags;
    if (!descs || n_tensors <= 0 || (dtype != GRANQ_F32 && dtype != GRANQ_BF16)) return GRANQ_ERR_INVALID_ARG;
    if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < table_bytes(n_tensors)) return GRANQ_ERR_WORKSPACE;
    const size_t esz = dtype == GRANQ_F32 ? 4 : 2;
    const uint32_t V = dtype == GRANQ_F32 ? 4 : 8;
    std::vector<WDesc> table((size_t)n_tensors);
    uint64_t total = 0;
    for (int i = 0; i < n_tensors; ++i) {
        const granq_weight_desc& s = descs[i];
        if (!s.x || !s.y || !s.min_out || !s.max_out || s.bits < 1 || s.bits > 8 || s.channels <= 0 ||
            s.group_elems <= 0 || (s.gy_opt == nullptr) != (s.gx_opt == nullptr))
            return GRANQ_ERR_INVALID_ARG;
        if (s.channels >= (1ll << 31) || s.group_elems >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
        const size_t nb = (size_t)s.channels * (size_t)s.group_elems * esz;
        const char *px = (const char*)s.x, *py = (const char*)s.y, *pgy = (const char*)s.gy_opt,
                   *pgx = (const char*)s.gx_opt;
        auto hit = [nb](const char* a, const char* b) { return a && b && a < b + nb && b < a + nb; };
        if (hit(px, py) || hit(px, pgx) || hit(pgy, py) || hit(pgy, pgx) || hit(py, pgx)) return GRANQ_ERR_INVALID_ARG;
        WDesc& d = table[(size_t)i];
        d.x = s.x;
        d.gy = s.gy_opt;
        d.y = s.y;
        d.gx = s.gx_opt;
        d.lo = s.min_out;
        d.hi = s.max_out;
        d.s = s.scale_opt;
        d.z = s.zp_opt;
        d.channels = (uint32_t)s.channels;
        d.group_elems = (uint32_t)s.group_elems;
        d.qmax = (float)((1 << s.bits) - 1);
        const uintptr_t all = (uintptr_t)s.x | (uintptr_t)s.y | (uintptr_t)s.gy_opt | (uintptr_t)s.gx_opt;
        d.vec = ((all & 15) == 0 && s.group_elems % V == 0) ? 1u : 0u;
        const uint64_t units = d.vec ? d.group_elems / V : d.group_elems;
        d.team = 1;
        while (d.team < kWWarps && units > (uint64_t)d.team * 32 * kWHold) d.team *= 2;
        total += (uint64_t)s.channels;
        if (total >= (1ull << 31)) return GRANQ_ERR_UNSUPPORTED;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // documented as not capturable, and kept that way: a caller may rely on the refusal
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capturing) != cudaSuccess) return GRANQ_ERR_CUDA;
    if (capturing != cudaStreamCaptureStatusNone) return GRANQ_ERR_UNSUPPORTED;
    for (int i = 0; i < n_tensors; i += kWTable) {
        const int n = n_tensors - i < kWTable ? n_tensors - i : kWTable;
        uint64_t blocks = 0;
        bool grad = false;
        for (int k = i; k < i + n; ++k) {
            WDesc& d = table[(size_t)k];
            const uint32_t groups = kWWarps / d.team;          // groups of one block
            d.first_block = (uint32_t)blocks;
            blocks += (d.channels + groups - 1) / groups;
            grad = grad || d.gy != nullptr;
        }
        const cudaError_t e = dtype == GRANQ_F32 ? w_launch<float>(&table[(size_t)i], n, (uint32_t)blocks, grad, st)
                                                 : w_launch<__nv_bfloat16>(&table[(size_t)i], n, (uint32_t)blocks, grad, st);
        if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    }
    return GRANQ_OK;
}

}  // extern "C"
