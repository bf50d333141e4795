// Host-side declarations shared by the translation units of the GranQ library.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "granq_device.cuh"

namespace granq {

// A tensor reduced to channel-group form: element e lies in plane p = e / inner and in
// group p % C.  Sample-channel grouping is (outer = 1, C = outer * C); tensor grouping is
// (outer = 1, C = 1, inner = E).
struct Geom {
    int64_t E;      // elements
    int64_t outer;  // slabs
    int64_t C;      // groups (< 2^31)
    int64_t inner;  // contiguous elements of one (slab, group) plane
};

// (dims, channel axis, group mode) -> channel-group form and the number of groups; false when the
// arguments are invalid (null dims, axis or mode out of range, a non-positive dim, more than 2^40 elements).
constexpr int64_t kMaxElements = 1ll << 40;
inline bool make_geom(const int64_t dims[4], int axis, int group, Geom& g, int64_t& G) {
    if (!dims || axis < 0 || axis > 3 || group < 0 || group > 2) return false;
    int64_t E = 1;
    for (int d = 0; d < 4; ++d) {
        if (dims[d] <= 0 || dims[d] > kMaxElements) return false;
        if (E > kMaxElements / dims[d]) return false;
        E *= dims[d];
    }
    if (E > kMaxElements) return false;
    int64_t outer = 1, inner = 1;
    for (int d = 0; d < axis; ++d) outer *= dims[d];
    for (int d = axis + 1; d < 4; ++d) inner *= dims[d];
    const int64_t C = dims[axis];
    g.E = E;
    if (group == 0) {            // GRANQ_GROUP_CHANNEL
        g.outer = outer; g.C = C; g.inner = inner;
    } else if (group == 1) {     // GRANQ_GROUP_SAMPLE_CHANNEL
        g.outer = 1; g.C = outer * C; g.inner = inner;
    } else {                     // GRANQ_GROUP_TENSOR
        g.outer = 1; g.C = 1; g.inner = E;
    }
    G = g.C;
    return true;
}

// Workspace layout (all plans): a 256-byte header whose first word is the device status,
// then G min-keys, G max-keys, then G + 1 wave arrival counters.
constexpr size_t kWsHeaderBytes = 256;
struct Workspace {
    uint32_t* status;
    uint32_t* kmin;
    uint32_t* kmax;
    uint32_t* counters;
    size_t clear_bytes;  // bytes from the start that must be zero before a launch
    bool cleared;        // the kernel ahead of the launch is launch_clear()'s
};
inline size_t workspace_bytes_for(int64_t G) {
    size_t b = kWsHeaderBytes + (size_t)G * 8 + ((size_t)G + 1) * 4;
    return (b + 255) & ~(size_t)255;
}
inline Workspace carve_workspace(void* ws, int64_t G) {
    Workspace w;
    char* p = (char*)ws;
    w.status = (uint32_t*)p;
    w.kmin = (uint32_t*)(p + kWsHeaderBytes);
    w.kmax = w.kmin + G;
    w.counters = w.kmax + G;
    w.clear_bytes = kWsHeaderBytes + (size_t)G * 8 + ((size_t)G + 1) * 4;
    w.cleared = false;
    return w;
}

enum { MODE_FWD = 1, MODE_BWD = 2, MODE_BOTH = 3 };

struct QuantIO {
    const void* x;
    const void* gy;   // MODE_BWD / MODE_BOTH
    void* y;          // MODE_FWD / MODE_BOTH
    void* gx;         // MODE_BWD / MODE_BOTH
    uint8_t* codes;   // optional
    uint8_t* mask;    // optional
    uint32_t* pmask;  // optional: the mask at one bit per element (forward plans that support it)
    double* dist;     // optional: 4 running sums of Table 2's statistics, zero on entry (same plans)
    uint32_t* pcodes; // optional: the integer codes as a bit string, code_bits each (flat forward kernel; y may then be null)
    int code_bits;
    bool behind_range;  // the flat kernels: the kernel ahead on the stream is this call's range
};

// Room for dynamic shared memory.  The attribute belongs to the kernel, not to the launch: every call states the same
// value, the most the kernel's plans ask for, so that calls of different sizes from several threads cannot take it
// from one another between stating it and launching.  (What a launch really takes of an SM is its own size.)
template <typename K>
inline cudaError_t allow_smem(K kern, size_t most) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// Launch of a kernel that begins with after_the_kernel_ahead(): its grid is set up while the kernel ahead of it in the stream
// drains, which hides a launch's latency: weights of a network 20.5 -> 17.6 us, range, forward and backward of [128,960,7,7]
// 41.0 -> 37.1, codes and back of [128,144,56,56] 128.7 -> 123.9.
// smem_kb: the shared memory that an SM full of its blocks takes, or kAnyLayout.  Stating it keeps blocks off an SM that is still laid
// out for the shared memory of the kernel ahead; once on it, one after the other would read through what that layout leaves of
// the L1 until the last is done.  Worth it from 16 MB on (sm_layout()); below, starting early on any SM is worth more.  Stated / not, us:
// packed mask and backward of fp32 [128,144,56,56] 173.1 / 184.9 and [41,1896,15,16] 60.7 / 64.8, fused call and backward from x of
// [116,1240,16,15] 110.7 / 125.3, fused call and weights of a network 113.0 / 114.9; bf16 [212,568,7,8], 13 MB, fused call and backward 25.2 /
// 23.9.
// kAlone: not before the kernel ahead has ended.
constexpr int kAnyLayout = -1, kAlone = -2;
inline int sm_layout(int smem_kb, uint64_t bytes) { return bytes >= (16ull << 20) ? smem_kb : kAnyLayout; }
template <typename... P, typename... A>
inline cudaError_t launch_after(int smem_kb, void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                                A&&... args) {
    constexpr int kSmemKB = 228;           // of an SM; the attribute is a percentage of it
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = smem_kb < 0 ? 0u : (unsigned)(smem_kb * 100 / kSmemKB);
    cfg.attrs = attr;
    cfg.numAttrs = smem_kb == kAlone ? 0 : smem_kb == kAnyLayout ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Zero `bytes` of a workspace (a multiple of 4) and, where given, four sums: a kernel in place of one memset or two, which a
// cooperative launch behind it need not wait for to read its inputs (a memset and the launch behind it 7.2 us, this 4.7).
cudaError_t launch_clear(void* workspace, size_t bytes, double* sums_opt, cudaStream_t st);

// ---- generic ("flat") kernels: any geometry, any alignment --------------------------------
// Range of every group (Eq. 4) into lo / hi, and s / z when bits > 0 and the pointers are given (Eq. 5).  The keys and,
// where one is given, the counter must be zero on entry; with a counter the range launch finishes by itself.
// behind_clear: the kernel ahead is launch_clear()'s.  The range launch is set up beside that one only: beside another its blocks, about
// a wave of them, crowd on the SMs that have room first (fused call on a zeroed workspace and forward, [33,41,51,51] 64 us / 68).
cudaError_t launch_range(const void* x, int dtype, const Geom& g, uint32_t* kmin, uint32_t* kmax, uint32_t* counter,
                         float* lo, float* hi, int bits, float* s_opt, float* z_opt, bool behind_clear, cudaStream_t st);
// lo / hi -> s / z
cudaError_t launch_params(const float* lo, const float* hi, int64_t G, int bits, float* s_opt, float* z_opt,
                          cudaStream_t st);
// elementwise quantize / backward with a per-group range in lo / hi
cudaError_t launch_quant_flat(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, const float* lo,
                              const float* hi, cudaStream_t st);
// STE backward from the mask at one bit per element (bit e % 32 of word e / 32)
cudaError_t launch_bwd_packmask(const void* gy, const uint32_t* pmask, void* gx, int dtype, int64_t E,
                                cudaStream_t st);
// sums[0..3] += sum x^2, sum q^2, sum x*q, sum (x-q)^2 over E elements (Table 2's raw material)
cudaError_t launch_distortion(const void* x, const void* q, int dtype, int64_t E, double* sums, cudaStream_t st);
// Eq. 6 from the packed integer codes (element e in bits [e*b, (e+1)*b) of the bit string)
cudaError_t launch_dequant_packed(const uint32_t* pcodes, void* y, int dtype, const Geom& g, int bits, const float* s,
                                  const float* z, cudaStream_t st);
// the "conventional" scheme: a host loop over groups with three launches each
cudaError_t launch_naive(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, uint32_t* kmin,
                         uint32_t* kmax, float* lo, float* hi, cudaStream_t st, int* launches);

// ---- on-chip staged persistent kernel ------------------------------------------------------
struct StagedPlan {
    bool ok;
    int grid, threads, depth;      // CTAs, threads per CTA, buffers per CTA
    uint32_t smem_bytes;           // dynamic shared memory per CTA
    uint32_t buf_units;            // 16-byte units per buffer
    uint32_t cw;                   // channels per wave
    uint32_t cu;                   // units per chunk
    uint32_t nwaves;
};
// Test / tuning overrides of the planner (0 = automatic).
struct StagedTuning {
    int depth;            // force the number of buffers per CTA (1..3)
    int max_buf_units;    // cap on 16-byte units per buffer (forces many small waves)
    int grid;             // cap on the number of CTAs
    int spin_limit;       // iteration limit of the wait on a wave's arrival count
    int extra_arrivals;   // test hook: arrivals a wave waits for beyond the grid size (never come)
    int ctas_per_sm;      // CTAs sharing one SM (1 or 2); they split its threads and shared memory
    int l2_wave_kb;       // L2-wave plan: target x bytes of one wave, in KiB
    int l2_upl;           // L2-wave plan: 16-byte units per lane and step (2 or 4)
    int l2_ctas_per_sm;   // L2-wave and column-walk plans: cap on resident CTAs per SM
    int l2_lag;           // column-walk plan: waves of phase 1 running ahead of phase 2 (1..3)
    int cl_tile_kb;       // cluster plan: limit on the staged tile of one CTA, in KiB
    int cl_r;             // cluster plan: CTAs per cluster (1, 2, 4, 8)
    int cl_threads;       // cluster plan: threads per CTA
    int cl_load;          // cluster plan: 1 = bulk copies for x, 2 = plain loads that reduce on the way, 3 = bulk copies for x and gy
    int cl_prefetch;      // cluster plan: 1 = ask the L2 for gy while x is loading, 2 = do not
    int cl_kmul;          // cluster plan: multiplier of the minimal channel count of a run
    int cl_pdl;           // cluster plan: 2 = no programmatic dependent launch
    int col_team;         // column-walk plan: 1 = resident form wherever it can, 2 = L2 waves only
    int coop_ctas;        // test hook: launch_cooperative() refuses more CTAs than this
};
extern StagedTuning g_tune;      // what granq_tune() sets
// A cooperative launch that may be refused: every CTA has to be resident at once, and where the GPU is shared out (a
// partition, a limit on the SMs of a process) fewer are than its attributes say.  cudaErrorCooperativeLaunchTooLarge,
// with nothing enqueued and no error left behind, tells the caller to take a plan that needs no such launch.
// The grid is set up while the kernel ahead drains; the kernel waits for that one's memory itself: before it reads anything, or,
// where the kernel ahead only clears its workspace (Workspace::cleared; that one has waited for all before it), between
// reading its inputs and touching anything else.
inline cudaError_t launch_cooperative(const void* kern, uint32_t grid, uint32_t threads, void** params, size_t smem,
                                      const StagedTuning& tune, cudaStream_t st) {
    if (tune.coop_ctas > 0 && grid > (uint32_t)tune.coop_ctas) return cudaErrorCooperativeLaunchTooLarge;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, kern, params);
    if (e == cudaErrorCooperativeLaunchTooLarge) (void)cudaGetLastError();
    return e;
}
StagedPlan plan_staged(int dtype, const Geom& g, const QuantIO& io, int device, const StagedTuning& tune);
StagedPlan plan_staged_on(int dtype, const Geom& g, const QuantIO& io, int sm_count, int smem_optin,
                          const StagedTuning& tune);
cudaError_t launch_staged(const StagedPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                          const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                          const StagedTuning& tune, cudaStream_t st);

// ---- L2-resident-wave persistent kernel ---------------------------------------------------
struct L2Plan {
    bool ok;
    int upl;                 // 16-byte units per lane and step
    uint32_t smem_bytes;     // dynamic shared memory per CTA
    uint32_t cw;             // channels per wave
    uint32_t nwaves;
};
L2Plan plan_l2wave(int dtype, const Geom& g, const QuantIO& io, const StagedTuning& tune);
cudaError_t launch_l2wave(const L2Plan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                          const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                          const StagedTuning& tune, cudaStream_t st);

// ---- column-walk persistent kernel (L2-resident waves, one unit column per thread) ----------
// Where a channel fits the shared memory of a team of CTAs the walk keeps it there (granq_colteam.cu).
struct TeamPlan {
    bool ok;
    uint32_t R, teams;       // CTAs per team, teams
    bool lag;                // two channels side by side, the hand-over of one behind the quantize walk of the other
    uint32_t tile_units;     // 16-byte units of x one CTA holds of each
    uint32_t gy_units;       // units of gy it holds beside them
    uint32_t smem_bytes;     // dynamic shared memory per CTA
    uint32_t threads;        // of a CTA
    uint32_t sm_count;       // planned for
};
// tensors: that many of these dims in one launch
TeamPlan plan_colteam(int dtype, const Geom& g, const QuantIO& io, bool backward, int sm_count, const StagedTuning& tune,
                      uint32_t tensors = 1);
// does the column walk take this form rather than the waves?
bool team_over_waves(const TeamPlan& plan, const Geom& g, const StagedTuning& tune);
// may be refused: launch_cooperative()
cudaError_t launch_colteam(const TeamPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                           const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                           const StagedTuning& tune, cudaStream_t st);
// a list of fp32 tensors of the same dims that share no memory, with a gradient (or one tensor of either type); the plan has to
// be one with `lag`
constexpr uint32_t kTeamListMax = 16;
struct TeamTensor {
    QuantIO io;
    int bits;
    Workspace ws;
    float *lo, *hi, *s_opt, *z_opt;
};
cudaError_t launch_colteam_list(const TeamPlan& plan, const TeamTensor* tensors, uint32_t n, int dtype, const Geom& g,
                                const StagedTuning& tune, cudaStream_t st);
struct ColPlan {
    bool ok;
    uint32_t cw;             // channels per wave
    uint32_t nwaves;
    uint32_t lag;            // waves of phase 1 running ahead of phase 2
};
ColPlan plan_colwalk(int dtype, const Geom& g, const QuantIO& io, const StagedTuning& tune);
cudaError_t launch_colwalk(const ColPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                           const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                           const StagedTuning& tune, cudaStream_t st);

// forward with a given range by columns (granq_flat.cu)
struct ColsCut {
    uint32_t side;                   // slabs side by side in a row
    uint32_t row_units, last_units;  // 16-byte units of a row, of the last row
    uint32_t ncol;                   // blocks across a row
    uint32_t rows, walk;             // rows, those a block walks
};
bool cut_cols(int dtype, const Geom& g, bool packed_mask, int sms, ColsCut& cut);

// ---- range and quantization of a tensor held in shared memory piece by piece (granq_hold.cu) ----
struct HoldPlan {
    bool ok;
    uint32_t ctas, share;    // CTAs, 16-byte units of one
    uint32_t held, planes;   // of those, kept in shared memory; planes it can cut through
    uint32_t tail;           // elements behind the last whole unit (masks and codes: behind the last whole byte)
    bool whole;              // nothing is left behind the units, or in the last word of a mask or of codes
};
HoldPlan plan_hold(int dtype, const Geom& g, const QuantIO& io, int sm_count);
// may be refused: launch_cooperative()
cudaError_t launch_hold(const HoldPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                        const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt, const StagedTuning& tune,
                        cudaStream_t st);

// ---- channels-last kernels (the channel is the innermost axis: one 16-byte unit holds V channels of a row) ----
bool plan_rows(int dtype, const Geom& g, const QuantIO& io);
struct RowsCut {
    uint32_t P, slices;      // unit columns of a slice, slices
    uint32_t lanes;          // rows of threads: the rows of one block
    uint32_t team;           // CTAs per slice
};
// false where the GPU holds too few CTAs at once for any cut (ctas: how many)
bool cut_rows(int dtype, const Geom& g, bool backward, uint32_t ctas, RowsCut& cut);
// may be refused: launch_cooperative()
cudaError_t launch_rows(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, const Workspace& ws,
                        float* lo, float* hi, float* s_opt, float* z_opt, const StagedTuning& tune, cudaStream_t st);

// ---- cluster-local kernel (a run of channels staged once in the shared memory of one cluster) ----
struct ClusterPlan {
    bool ok;
    uint32_t k;              // channels per run
    uint32_t R;              // CTAs per cluster
    uint32_t threads;        // threads per CTA
    uint32_t tile_bytes;     // staged tile of one CTA
    uint32_t smem_bytes;     // dynamic shared memory per CTA (tile + keys + parameters)
    int load;                // 0 = plain loads, 1 = x staged by bulk copies, 2 = x and gy staged by bulk copies
    bool prefetch_gy;
    bool early_launch;       // programmatic dependent launch: set the grid up while the kernel ahead drains
    bool clears_status;      // the kernel can write status 0 itself (no wait in it can run out)
    bool zero_status;        // and is to do so: not where the caller vouched for a zero workspace (set by the caller)
    bool late_wait;          // it shares no memory with the kernels ahead of it that may still run: it need not wait for
                             // them before it starts, only before it ends
};
ClusterPlan plan_cluster(int dtype, const Geom& g, const QuantIO& io, bool backward, const StagedTuning& tune);
cudaError_t launch_cluster(const ClusterPlan& plan, const QuantIO& io, int mode, int dtype, const Geom& g, int bits,
                           const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt,
                           const StagedTuning& tune, cudaStream_t st);

}  // namespace granq
