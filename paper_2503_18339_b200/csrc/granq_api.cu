// C ABI of the GranQ library: argument validation, reduction of (dims, channel axis, group
// mode) to channel-group geometry, plan selection and launches.  See include/granq.h.
#include "../../include/granq.h"

#include "granq_internal.h"

#include <math.h>

using namespace granq;

StagedTuning granq::g_tune = {};

namespace {

bool dtype_ok(int dtype) { return dtype == GRANQ_F32 || dtype == GRANQ_BF16; }
size_t elt_size(int dtype) { return dtype == GRANQ_F32 ? 4 : 2; }

bool overlaps(const void* a, size_t na, const void* b, size_t nb) {
    if (!a || !b) return false;
    const char* pa = (const char*)a;
    const char* pb = (const char*)b;
    return pa < pb + nb && pb < pa + na;
}

int check_workspace(const void* ws, size_t bytes, int64_t G) {
    if (!ws || ((uintptr_t)ws & 255) != 0) return GRANQ_ERR_WORKSPACE;
    if (bytes < workspace_bytes_for(G)) return GRANQ_ERR_WORKSPACE;
    return GRANQ_OK;
}

int cuda_status(cudaError_t e) { return e == cudaSuccess ? GRANQ_OK : GRANQ_ERR_CUDA; }

enum { PLAN_TWO_PASS = 0, PLAN_NAIVE = 1, PLAN_STAGED = 2, PLAN_L2WAVE = 3, PLAN_COLWALK = 4, PLAN_CLUSTER = 5, PLAN_ROWS = 6 };

// plan of the fused entry point; `plan_out` is filled when the staged plan is taken
int choose_plan(int dtype, const Geom& g, const QuantIO& io, bool backward, uint32_t flags, StagedPlan* plan_out,
                L2Plan* l2_out, ColPlan* col_out, ClusterPlan* cl_out) {
    if (flags & GRANQ_FLAG_FORCE_NAIVE) return PLAN_NAIVE;
    if (flags & GRANQ_FLAG_FORCE_TWO_PASS) return PLAN_TWO_PASS;
    if (flags & GRANQ_FLAG_FORCE_CLUSTER) {
        ClusterPlan kp = plan_cluster(dtype, g, io, backward, g_tune);
        if (!kp.ok) return -GRANQ_ERR_UNSUPPORTED;
        if (cl_out) *cl_out = kp;
        return PLAN_CLUSTER;
    }
    if (flags & GRANQ_FLAG_FORCE_COLWALK) {
        ColPlan cp = plan_colwalk(dtype, g, io, g_tune);
        if (!cp.ok) return -GRANQ_ERR_UNSUPPORTED;
        if (col_out) *col_out = cp;
        return PLAN_COLWALK;
    }
    if (flags & GRANQ_FLAG_FORCE_L2WAVE) {
        L2Plan lp = plan_l2wave(dtype, g, io, g_tune);
        if (!lp.ok) return -GRANQ_ERR_UNSUPPORTED;
        if (l2_out) *l2_out = lp;
        return PLAN_L2WAVE;
    }
    if (flags & GRANQ_FLAG_FORCE_STAGED) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return -GRANQ_ERR_CUDA;
        StagedPlan p = plan_staged(dtype, g, io, dev, g_tune);
        if (!p.ok) return -GRANQ_ERR_UNSUPPORTED;
        if (plan_out) *plan_out = p;
        return PLAN_STAGED;
    }
    // channels-last geometries (the channel is the innermost axis) have plans of their own: the cluster-local
    // kernel cannot stage them (a run of channels is a few bytes per row) and there are no planes to walk
    if (g.inner == 1 && plan_rows(dtype, g, io)) return PLAN_ROWS;
    // default: the cluster-local kernel where a run of channels fits the shared memory of one cluster
    // (x is then read once and nothing waits on the grid), else the column-walk kernel where there are
    // slabs to walk, else the L2-resident-wave kernel
    ClusterPlan kp = plan_cluster(dtype, g, io, backward, g_tune);
    ColPlan cp{};
    cp.ok = false;
    // Measured exception: forward-only bf16 tensors of 48 MB and more (a 100 KB tile then holds 51 200 elements
    // and a CTA's chain of copy, fold and quantize is twice as long as for fp32) run faster on the column walk in
    // its resident form ([256,512,28,28] 104 / 92 us); with a gradient, and for fp32, see prefer_team() below.
    const bool long_chain = dtype == 1 && !backward && !(io.codes || io.mask || io.pmask || io.dist) &&
                            (uint64_t)g.E * 2 >= (48ull << 20);
    if (kp.ok && long_chain) {
        cp = plan_colwalk(dtype, g, io, g_tune);
        if (cp.ok) {
            if (col_out) *col_out = cp;
            return PLAN_COLWALK;
        }
    }
    if (kp.ok) {
        if (cl_out) *cl_out = kp;
        return PLAN_CLUSTER;
    }
    cp = plan_colwalk(dtype, g, io, g_tune);
    if (cp.ok) {
        if (col_out) *col_out = cp;
        return PLAN_COLWALK;
    }
    L2Plan lp = plan_l2wave(dtype, g, io, g_tune);
    if (lp.ok) {
        if (l2_out) *l2_out = lp;
        return PLAN_L2WAVE;
    }
    return PLAN_TWO_PASS;
}

// Where the cluster-local plan takes a call by default, the form in which its channels are held: one cluster per
// channel, or (this returns a plan) teams of CTAs of one cooperative launch.  Both read x once; the cluster starts
// sooner (its launch overlaps the kernel ahead) and hands over faster, the team is dealt out evenly, keeps reads in
// flight while it writes and needs no GPC with eight free CTAs.  Measured (cluster / team, us): the team from 96 MB
// of x and 256 KB per channel on - fp32 [256,512,28,28] forward 169 / 156, with gradient 319 / 298, packed mask
// 227 / 174, codes 276 / 202; [64,256,56,56] 89 / 81, 157 / 150, 125 / 91, codes 155 / 106; bf16 63 / 56, 86 / 84 -
// and the cluster below: [128,192,28,28] 37 / 38, 62 / 62; [256,256,16,16] 33 / 40; [32,64,56,56] 17 / 19, and with
// small channels: [256,1024,14,14] 87 / 88, 159 / 163.  fp32 with a gradient crosses later ([128,256,28,28], 98 MB:
// 80 / 83).
TeamPlan prefer_team(int dtype, const Geom& g, const QuantIO& io, bool backward, uint32_t flags) {
    TeamPlan none{};
    if (flags & GRANQ_FLAG_FORCE_CLUSTER) return none;
    const StagedTuning& t = g_tune;
    if (t.cl_tile_kb || t.cl_r || t.cl_threads || t.cl_load || t.cl_prefetch || t.cl_kmul || t.cl_pdl || t.col_team == 2) return none;
    const uint64_t bytes = (uint64_t)g.E * elt_size(dtype);
    const uint64_t from = (backward && dtype == GRANQ_F32 ? 128ull : 96ull) << 20;
    if (bytes < from || bytes / (uint64_t)g.C < (256ull << 10)) return none;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return none;
    return plan_colteam(dtype, g, io, backward, sms, g_tune);
}

// The call with its channels held on chip, in the form chosen; where the GPU does not hold that many CTAs at once, by
// the cluster, which needs no cooperative launch.
cudaError_t launch_held(const TeamPlan& tp, const ClusterPlan& kp, const QuantIO& io, int mode, int dtype, const Geom& g,
                        int bits, const Workspace& ws, float* lo, float* hi, float* s_opt, float* z_opt, cudaStream_t st) {
    if (tp.ok) {
        const cudaError_t e = launch_colteam(tp, io, mode, dtype, g, bits, ws, lo, hi, s_opt, z_opt, g_tune, st);
        if (e != cudaErrorCooperativeLaunchTooLarge) return e;
    }
    return launch_cluster(kp, io, mode, dtype, g, bits, ws, lo, hi, s_opt, z_opt, g_tune, st);
}

// Where a call would take two passes or the L2-resident waves, not because it or a knob of the waves asked for them: one launch that
// holds the tensor on chip (what it gains stands at the kernel).
bool hold_allowed(uint32_t flags) {
    return !(flags & (GRANQ_FLAG_FORCE_TWO_PASS | GRANQ_FLAG_FORCE_L2WAVE)) && !g_tune.l2_wave_kb && !g_tune.l2_upl && !g_tune.l2_ctas_per_sm;
}
// Whether it pays for a tensor that leaves something behind its whole units, or whose codes end inside a 32-bit word.  A group's keys come together
// by atomics, one per plane: two passes are faster for codes of many short planes of whole packs (of planes that are none they cost more: 4-bit codes
// of fp32 [5656,11,9,9] 39 / 33), and where planes are groups, some hundred thousand of them.  Two passes / held, us: 5-bit codes of fp32
// [3473,18,2,2] 17 / 23, [27779,18,2,4] 32 / 135, [701,150,2,4] 16 / 19, [601,301,2,4] 17 / 18.5, but [415,301,2,4] 17 / 14.5, [1501,18,2,2] 15 /
// 14.5; bf16 [3473,18,2,4] 15 / 23, [701,150,2,4] 12 / 18, [415,301,4,4] 13.7 / 14.7, [301,301,4,4] 12.3 / 12.7, but [209,301,2,4] 12 / 10; a group
// per plane, forward, fp32 [118,3767,3,3] 75 / 92, but [67,2133,7,7] 52 / 49; bf16 [117,3761,5,5] 88 / 103, [67,2132,7,7] 39 / 48, but [83,2677,3,3]
// 48 / 49, from a graph 53 / 46, [71,2254,5,5] 44 / 43.
bool remainder_held(int dtype, const Geom& g, const QuantIO& io) {
    if (g.outer == 1) return g.C <= (dtype == GRANQ_F32 || g.E <= 5'000'000 ? 250'000 : 100'000);
    if (!io.pcodes || g.inner % (dtype == GRANQ_F32 ? 4 : 8) != 0) return true;
    return g.outer * g.C + 110 * g.outer <= (dtype == GRANQ_F32 ? 180'000 : 88'000);
}
HoldPlan prefer_hold(int dtype, const Geom& g, const QuantIO& io, uint32_t flags) {
    HoldPlan none{};
    if (!hold_allowed(flags)) return none;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return none;
    const HoldPlan p = plan_hold(dtype, g, io, sms);
    return p.ok && !p.whole && !remainder_held(dtype, g, io) ? none : p;
}

// In place of the cluster-local plan, where every group is one plane (a group per sample and channel, or a batch of one): a cluster then
// has one slab to walk, and a thread that keeps a unit column works out its parameters for a single unit; pieces of equal size have tables of
// them.  Against that stand a clearing launch and a cooperative one instead of a plain launch, one after another 2 us of every call, and atomics of
// every plane.  A wave of clusters holds 9 MB, up to where their time hardly grows and the pieces' does; a second one takes half as long
// again.  Cluster / piece by piece, us, calls one after another:
// bf16 whose planes are not whole units, forward [64,256,3,3] 49.0 / 13.4, [8,64,7,7] 19.5 / 10.3, [64,64,13,13] 15.4 / 10.3, with gradient
// [16,784,14,14] 18.6 / 14.7, but [8,8,7,7], 3136 elements, 6.3 / 8.5, packed mask [8,64,7,7] 22.5 / 23.7; of many groups [79,2536,5,5] 51 / 49,
// [44,1408,9,9] 31 / 27, but [132,4216,3,3] 63 / 99, [100,3200,5,5] 52 / 72, and beyond the wave [33,1080,15,15] 27 / 28, [31,984,19,19] 39 / 35, but
// [56,1764,9,9] 33 / 40, [44,1414,15,15] 40 / 46. Of whole units with gradient [16,64,112,112] 36 / 25, [10,73,64,64] 13.3 / 12.4; forward
// [12,102,64,64], 10 MB, 15.4 / 14.4, [17,144,64,64] 23.6 / 20.1, [4,40,112,112] 12.6 / 10.3, but [11,89,64,64], 8 MB, 10.7 / 12.5, [8,61,64,64] 9.4
// / 10.3, [16,64,56,56] 10.6 / 11.1. With the sums [22,178,16,16] 12.1 / 10.4, [16,122,32,32] 12.4 / 11.7, [12,102,64,64] 20.1 / 16.5, but
// [19,154,32,32], 6 MB, 13.0 / 13.9, [11,89,64,64] 13.5 / 14.5, [61,480,16,16] 20.8 / 23.1; fp32 [31,242,20,20], 12 MB, 15.7 / 14.6, [40,312,20,20]
// 23.6 / 18.9, but [13,108,56,56], 18 MB, 16.0 / 16.5, [37,297,20,20] 16.7 / 18.5, [64,300,14,14] 15.4 / 16.4; fp32 without sums a third slower or
// more.  From a graph the pieces are 2 us better throughout. Not in a list, whose cluster-local kernels run beside one another: eight bf16
// [16,256,14,14] 34 / 82, [8,16,112,112] 39 / 82.
HoldPlan hold_over_cluster(int dtype, const Geom& g, const QuantIO& io, uint32_t flags) {
    HoldPlan none{};
    const StagedTuning& t = g_tune;
    if ((flags & (GRANQ_FLAG_FORCE_CLUSTER | GRANQ_FLAG_FORCE_COLWALK)) || t.cl_tile_kb || t.cl_r || t.cl_threads || t.cl_load || t.cl_prefetch ||
        t.cl_kmul || t.cl_pdl || g.outer != 1 || g.C == 1)
        return none;
    const bool bf16 = dtype == GRANQ_BF16, sums = io.dist != nullptr, beyond = g.E >= 4'800'000, long_planes = g.inner >= 8192;
    bool pays;
    if (bf16 && g.inner % 8 != 0)
        pays = g.E >= (io.pmask || io.pcodes ? 1 << 16 : 8192) && g.C <= (g.E <= 6'000'000 ? 200'000 : 32'000);
    else if (sums)
        pays = g.inner >= (bf16 ? 256 : 400) && (bf16 || g.E >= 3'000'000) &&
               (long_planes || g.E <= (bf16 ? 2'500'000 : 3'500'000) || (beyond && g.inner >= 400));
    else
        pays = bf16 && g.inner >= 4096 && g.E >= 1 << 20 && (io.gy || long_planes || beyond);
    return pays ? prefer_hold(dtype, g, io, flags) : none;
}

// The workspace set to zero ahead of one cooperative launch, or of range launches.  On the device the clearing kernel, which the launch
// behind it need not wait for to read on, is 3 us shorter than a memset (with the launch behind it, from a graph, 1.1 / 4.1), but it
// costs the host 1.5 us more (2.4 / 0.85).  So a call whose kernels take less time than the host needs to make it, and which is not
// being captured, takes the memset: up to `host_bound` elements, where the two cross for a call with everything to allocate, through the
// binding's native calls.  Kernel / memset, us: range of 0.26 M elements 8.8 / 8.4, 1 M 8.7 / 8.4, 1.5 M 8.65 / 8.5, 2 M fp32 8.7 / 10.0; ahead of a
// cooperative launch, fp32, channels-last of 0.12 M elements 11.5 / 10.8, 0.26 M 11.4 / 10.6, 1.5 M 11.2 / 12.4, bf16 0.5 M 12.4 / 12.7, 1 M 12.5 /
// 14.1, one group with gradient of 0.26 M 12.6 / 12.0.  A call with its buffers at hand makes the host no match for the GPU and would be better off
// with the kernel: range 5.6 / 7.4, 1 M 5.6 / 8.3, channels-last of 0.12 M 8.2 / 8.8, 0.26 M 8.4 / 9.6.
constexpr int64_t kHostBoundHeld = 1 << 18, kHostBoundRange = 1'500'000;
cudaError_t clear_workspace(Workspace& ws, const Geom& g, int64_t host_bound, cudaStream_t st) {
    if (g.E <= host_bound) {
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        const cudaError_t e = cudaStreamIsCapturing(st, &capturing);
        if (e != cudaSuccess) return e;
        if (capturing == cudaStreamCaptureStatusNone) return cudaMemsetAsync(ws.status, 0, ws.clear_bytes, st);
    }
    ws.cleared = true;
    return launch_clear(ws.status, ws.clear_bytes, nullptr, st);
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

extern "C" {

const char* granq_status_string(int status) {
    switch (status) {
        case GRANQ_OK: return "ok";
        case GRANQ_ERR_INVALID_ARG: return "invalid argument";
        case GRANQ_ERR_UNSUPPORTED: return "unsupported geometry or plan";
        case GRANQ_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case GRANQ_ERR_CUDA: return "CUDA error";
        case GRANQ_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        default: return "unknown status";
    }
}

int64_t granq_num_groups(const int64_t dims[4], int channel_axis, int group) {
    Geom g;
    int64_t G;
    if (!make_geom(dims, channel_axis, group, g, G)) return -1;
    return G;
}

size_t granq_workspace_bytes(int dtype, const int64_t dims[4], int channel_axis, int group) {
    Geom g;
    int64_t G;
    if (!dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return 0;
    return workspace_bytes_for(G);
}

int granq_range(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group, float* min_out,
                float* max_out, void* workspace, size_t workspace_bytes, uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!x || !min_out || !max_out || !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    if (int rc = check_workspace(workspace, workspace_bytes, G)) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Workspace ws = carve_workspace(workspace, G);
    // (tensors that are no whole 16-byte units keep the GPU longer than the host, with everything to allocate too: [7,33,33,33] 8.8 by the
    // kernel, 10.4 by a memset, [19,133,7,7] 12.7 / 15.4)
    cudaError_t e = clear_workspace(ws, g, g.E * (int64_t)elt_size(dtype) % 16 == 0 ? kHostBoundRange : 0, st);
    if (e == cudaSuccess)
        e = launch_range(x, dtype, g, ws.kmin, ws.kmax, ws.counters, min_out, max_out, 0, nullptr, nullptr, ws.cleared, st);
    return cuda_status(e);
}

int granq_fakequant_fwd(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group, int bits,
                        const float* min_in, const float* max_in, void* y, uint8_t* codes_opt, float* scale_opt,
                        float* zp_opt, uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!x || !y || !min_in || !max_in || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype);
    if (overlaps(x, nb, y, nb)) return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, y, nullptr, codes_opt, nullptr};
    cudaError_t e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_in, max_in, st);
    if (e == cudaSuccess && (scale_opt || zp_opt)) e = launch_params(min_in, max_in, G, bits, scale_opt, zp_opt, st);
    return cuda_status(e);
}

int granq_fakequant_bwd(const void* gy, const void* x, int dtype, const int64_t dims[4], int channel_axis, int group,
                        int bits, const float* min_in, const float* max_in, void* gx, uint8_t* mask_opt,
                        uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!gy || !x || !gx || !min_in || !max_in || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype);
    if (overlaps(x, nb, gx, nb) || overlaps(gy, nb, gx, nb)) return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, gy, nullptr, gx, nullptr, mask_opt};
    return cuda_status(launch_quant_flat(io, MODE_BWD, dtype, g, bits, min_in, max_in, st));
}

// granq_fakequant_fused(); independent: the call shares no memory with those ahead of it on the stream that were made
// since one that was not (a cluster-local kernel then need not wait for theirs before it starts); listed: one of several
static int fused_call(const void* x, const void* gy_opt, int dtype, const int64_t dims[4], int channel_axis, int group,
                      int bits, void* y, void* gx_opt, float* min_out, float* max_out, uint8_t* codes_opt,
                      uint8_t* mask_opt, float* scale_opt, float* zp_opt, void* workspace, size_t workspace_bytes,
                      uint32_t flags, void* cuda_stream, bool independent, bool listed) {
    Geom g;
    int64_t G;
    if (!x || !y || !min_out || !max_out || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    if ((gy_opt == nullptr) != (gx_opt == nullptr)) return GRANQ_ERR_INVALID_ARG;
    if (mask_opt && !gy_opt) return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype);
    if (overlaps(x, nb, y, nb) || overlaps(x, nb, gx_opt, nb) || overlaps(gy_opt, nb, y, nb) ||
        overlaps(gy_opt, nb, gx_opt, nb) || overlaps(y, nb, gx_opt, nb))
        return GRANQ_ERR_INVALID_ARG;
    if (int rc = check_workspace(workspace, workspace_bytes, G)) return rc;

    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int mode = gy_opt ? MODE_BOTH : MODE_FWD;
    QuantIO io{x, gy_opt, y, gx_opt, codes_opt, mask_opt};
    StagedPlan sp{};
    L2Plan lp{};
    ColPlan cp{};
    ClusterPlan kp{};
    const int plan = choose_plan(dtype, g, io, gy_opt != nullptr, flags, &sp, &lp, &cp, &kp);
    if (plan < 0) return -plan;
    kp.late_wait = independent && kp.clears_status;

    Workspace ws = carve_workspace(workspace, G);
    // The column-walk and channels-last kernels leave a zeroed workspace zeroed and the cluster-local kernel writes
    // nothing but the status word (0 where the caller did not vouch for it, or that a wait on its bulk copies ran
    // out); with the caller's word that the workspace is zero on entry nothing has to be cleared.  The other plans, to keep that word
    // true for the next call, clear after themselves.
    const bool zeroed = (flags & GRANQ_FLAG_WORKSPACE_ZEROED) != 0;
    kp.zero_status = !zeroed && kp.clears_status;
    HoldPlan hp{};
    if (plan == PLAN_TWO_PASS || plan == PLAN_L2WAVE) hp = prefer_hold(dtype, g, io, flags);
    if (plan == PLAN_CLUSTER && !listed) hp = hold_over_cluster(dtype, g, io, flags);
    bool keeps_zero = plan == PLAN_COLWALK || plan == PLAN_CLUSTER || plan == PLAN_ROWS || hp.ok;
    TeamPlan tp{};
    if (plan == PLAN_CLUSTER && !hp.ok) tp = prefer_team(dtype, g, io, gy_opt != nullptr, flags);
    cudaError_t e = cudaSuccess;
    if (plan == PLAN_CLUSTER && !tp.ok && !hp.ok) {
        if (!zeroed && !kp.clears_status) e = cudaMemsetAsync(workspace, 0, sizeof(uint32_t), st);      // the status word
    } else if (!zeroed) {
        e = clear_workspace(ws, g, plan == PLAN_ROWS || hp.ok ? kHostBoundHeld : 0, st);
    }
    if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    // two passes over x by ordinary launches: any geometry, any GPU
    auto two_pass = [&]() -> cudaError_t {
        cudaError_t r = launch_range(x, dtype, g, ws.kmin, ws.kmax, ws.counters, min_out, max_out, bits, scale_opt, zp_opt, ws.cleared, st);
        io.behind_range = true;
        return r == cudaSuccess ? launch_quant_flat(io, mode, dtype, g, bits, min_out, max_out, st) : r;
    };
    if (hp.ok && (e = launch_hold(hp, io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st)) !=
                     cudaErrorCooperativeLaunchTooLarge) {
        // done
    } else if (plan == PLAN_CLUSTER) {
        e = launch_held(tp, kp, io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, st);
    } else if (plan == PLAN_ROWS) {
        e = launch_rows(io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
        if (e == cudaErrorCooperativeLaunchTooLarge) {
            keeps_zero = false;
            e = two_pass();
        }
    } else if (plan == PLAN_STAGED) {
        e = launch_staged(sp, io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
    } else if (plan == PLAN_L2WAVE) {
        keeps_zero = false;
        e = launch_l2wave(lp, io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
    } else if (plan == PLAN_COLWALK) {
        e = launch_colwalk(cp, io, mode, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
    } else if (plan == PLAN_NAIVE) {
        e = launch_naive(io, mode, dtype, g, bits, ws.kmin, ws.kmax, min_out, max_out, st, nullptr);
        if (e == cudaSuccess && (scale_opt || zp_opt))
            e = launch_params(min_out, max_out, G, bits, scale_opt, zp_opt, st);
    } else {
        keeps_zero = false;
        e = two_pass();
    }
    if (e == cudaSuccess && zeroed && !keeps_zero)
        e = cudaMemsetAsync((char*)workspace + sizeof(uint32_t), 0, ws.clear_bytes - sizeof(uint32_t), st);
    return cuda_status(e);
}

int granq_fakequant_fused(const void* x, const void* gy_opt, int dtype, const int64_t dims[4], int channel_axis,
                          int group, int bits, void* y, void* gx_opt, float* min_out, float* max_out,
                          uint8_t* codes_opt, uint8_t* mask_opt, float* scale_opt, float* zp_opt, void* workspace,
                          size_t workspace_bytes, uint32_t flags, void* cuda_stream) {
    return fused_call(x, gy_opt, dtype, dims, channel_axis, group, bits, y, gx_opt, min_out, max_out, codes_opt, mask_opt,
                      scale_opt, zp_opt, workspace, workspace_bytes, flags, cuda_stream, false, false);
}

size_t granq_packmask_bytes(const int64_t dims[4]) {
    Geom g;
    int64_t G;
    if (!make_geom(dims, 1, GRANQ_GROUP_TENSOR, g, G)) return 0;
    return (size_t)((g.E + 31) / 32) * 4;
}

int granq_fakequant_fwd_packmask(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group,
                                 int bits, const float* min_in, const float* max_in, void* y,
                                 uint32_t* packed_mask, float* scale_opt, float* zp_opt, uint32_t flags,
                                 void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!x || !y || !packed_mask || !min_in || !max_in || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)packed_mask & 3))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype), mb = (size_t)((g.E + 31) / 32) * 4;
    if (overlaps(x, nb, y, nb) || overlaps(x, nb, packed_mask, mb) || overlaps(y, nb, packed_mask, mb))
        return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, y, nullptr, nullptr, nullptr, packed_mask};
    cudaError_t e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_in, max_in, st);
    if (e == cudaSuccess && (scale_opt || zp_opt)) e = launch_params(min_in, max_in, G, bits, scale_opt, zp_opt, st);
    return cuda_status(e);
}

int granq_fakequant_bwd_packmask(const void* gy, const uint32_t* packed_mask, int dtype, const int64_t dims[4],
                                 void* gx, uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!gy || !gx || !packed_mask || !dtype_ok(dtype) || !make_geom(dims, 1, GRANQ_GROUP_TENSOR, g, G) ||
        ((uintptr_t)packed_mask & 3))
        return GRANQ_ERR_INVALID_ARG;
    const size_t nb = (size_t)g.E * elt_size(dtype), mb = (size_t)((g.E + 31) / 32) * 4;
    if (overlaps(gy, nb, gx, nb) || overlaps(packed_mask, mb, gx, nb)) return GRANQ_ERR_INVALID_ARG;
    return cuda_status(launch_bwd_packmask(gy, packed_mask, gx, dtype, g.E, (cudaStream_t)cuda_stream));
}

int granq_fakequant_fused_fwd_packmask(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group,
                                       int bits, void* y, uint32_t* packed_mask, float* min_out, float* max_out,
                                       float* scale_opt, float* zp_opt, void* workspace, size_t workspace_bytes,
                                       uint32_t flags, void* cuda_stream) {
    Geom g;
    int64_t G;
    if (!x || !y || !packed_mask || !min_out || !max_out || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)packed_mask & 3))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype), mb = (size_t)((g.E + 31) / 32) * 4;
    if (overlaps(x, nb, y, nb) || overlaps(x, nb, packed_mask, mb) || overlaps(y, nb, packed_mask, mb))
        return GRANQ_ERR_INVALID_ARG;
    if (int rc = check_workspace(workspace, workspace_bytes, G)) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, y, nullptr, nullptr, nullptr, packed_mask};
    // the cluster-local kernel where a run of whole mask words fits one cluster, else the column-walk kernel
    // where the geometry allows whole mask words per wave, else range pass + flat pass
    ColPlan cp{};
    ClusterPlan kp{};
    const bool two_pass = (flags & GRANQ_FLAG_FORCE_TWO_PASS) != 0;
    if (!two_pass && !(flags & GRANQ_FLAG_FORCE_COLWALK)) kp = plan_cluster(dtype, g, io, false, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_CLUSTER) && !kp.ok) return GRANQ_ERR_UNSUPPORTED;
    if (!two_pass && !kp.ok) cp = plan_colwalk(dtype, g, io, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_COLWALK) && !cp.ok) return GRANQ_ERR_UNSUPPORTED;
    Workspace ws = carve_workspace(workspace, G);
    const bool zeroed = (flags & GRANQ_FLAG_WORKSPACE_ZEROED) != 0;
    kp.zero_status = !zeroed && kp.clears_status;
    cudaError_t e = cudaSuccess;
    HoldPlan hp{};
    if (kp.ok) hp = hold_over_cluster(dtype, g, io, flags);
    else if (!cp.ok) hp = prefer_hold(dtype, g, io, flags);
    const TeamPlan tp = kp.ok && !hp.ok ? prefer_team(dtype, g, io, false, flags) : TeamPlan{};
    if (hp.ok) {
        if (!zeroed) e = clear_workspace(ws, g, kHostBoundHeld, st);
        if (e != cudaSuccess) return GRANQ_ERR_CUDA;
        e = launch_hold(hp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
        if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_status(e);
        e = cudaSuccess;
    }
    if (kp.ok) {
        // the team form needs zeroed keys and counters; of the cluster kernel, the status word where it does not write it
        if (!zeroed && (tp.ok || !kp.clears_status))
            e = launch_clear(workspace, tp.ok ? ws.clear_bytes : sizeof(uint32_t), nullptr, st);
        ws.cleared = !zeroed && tp.ok;
        // the kernel writes the mask byte by byte: the padding bits of a last, partial word are cleared here
        if (e == cudaSuccess && g.E % 32 != 0) e = cudaMemsetAsync(packed_mask + g.E / 32, 0, sizeof(uint32_t), st);
        if (e != cudaSuccess) return GRANQ_ERR_CUDA;
        return cuda_status(launch_held(tp, kp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, st));
    }
    if (!zeroed && !hp.ok) e = clear_workspace(ws, g, 0, st);
    if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    if (cp.ok) {
        e = launch_colwalk(cp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
    } else {
        e = launch_range(x, dtype, g, ws.kmin, ws.kmax, ws.counters, min_out, max_out, bits, scale_opt, zp_opt, ws.cleared, st);
        io.behind_range = true;
        if (e == cudaSuccess) e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_out, max_out, st);
        if (e == cudaSuccess && zeroed)
            e = cudaMemsetAsync((char*)workspace + sizeof(uint32_t), 0, ws.clear_bytes - sizeof(uint32_t), st);
    }
    return cuda_status(e);
}

// Do two calls of a list touch common memory, at least one of them writing it?
static bool batch_conflict(const granq_fused_desc& a, const granq_fused_desc& b, int dtype, int channel_axis, int group) {
    struct Range {
        const void* p;
        size_t n;
    };
    auto ranges = [&](const granq_fused_desc& d, Range (&r)[2], Range (&w)[7]) -> bool {
        Geom g;
        int64_t G;
        if (!make_geom(d.dims, channel_axis, group, g, G)) return false;      // refused by its own call
        const size_t nb = (size_t)g.E * elt_size(dtype), gb = (size_t)G * sizeof(float);
        r[0] = {d.x, nb};
        r[1] = {d.gy_opt, nb};
        w[0] = {d.y, nb};
        w[1] = {d.gx_opt, nb};
        w[2] = {d.min_out, gb};
        w[3] = {d.max_out, gb};
        w[4] = {d.scale_opt, gb};
        w[5] = {d.zp_opt, gb};
        w[6] = {d.workspace, d.workspace_bytes};
        return true;
    };
    Range ra[2], wa[7], rb[2], wb[7];
    if (!ranges(a, ra, wa) || !ranges(b, rb, wb)) return true;
    for (const Range& u : wa) {
        for (const Range& v : rb)
            if (overlaps(u.p, u.n, v.p, v.n)) return true;
        for (const Range& v : wb)
            if (overlaps(u.p, u.n, v.p, v.n)) return true;
    }
    for (const Range& u : wb)
        for (const Range& v : ra)
            if (overlaps(u.p, u.n, v.p, v.n)) return true;
    return false;
}

// How many of the first tensors of a list of `count` of these dims, each with a gradient and sharing no memory, one launch of the
// resident walk takes together; 0: none, each is a call of its own.  bf16 gains nothing (seven of [256,16,32,32] 51.9 / 56.1 us, three
// of [16,64,56,56] 21.1 / 21.3).  Where no cluster holds a channel, the separate calls are resident walks one after the other and
// together takes 0.53 to 0.97 of their time (two to sixteen tensors of 6 to 40 MB).  Where one does, they are cluster-local kernels that
// run beside one another, and together pays only for many CTAs: of channels of 220 KB and more, whose tiles leave a cluster few
// neighbours, or of few slabs, which a cluster cannot share out evenly.  Of 1400 lists, separate / together, us: six of
// [232,32,16,16] 46 / 42, but of [214,32,16,16] 33 / 39, and four of [256,32,16,16] 33 / 33; six of [160,16,32,32] 51 / 55; three of
// [8,72,80,80] 72 / 40; two of [70,256,14,14] 25 / 31.  Those that pass: 0.52 to 1.02, mean 0.85.  Of the others many would be up to
// 1.5 times as slow; some long lists would gain a fifth.
static int list_takes(int dtype, const Geom& g, int count, int sms, TeamPlan& plan) {
    count = count < (int)kTeamListMax ? count : (int)kTeamListMax;
    const bool large = g.E / g.C >= (220 << 10) / 4;
    // most lists go no further: of small channels, and more slabs than a cluster of eight has too few of
    if (dtype != GRANQ_F32 || count < 2 || (!large && g.outer > 24) || g.C >= (1ll << 28)) return 0;
    const ClusterPlan kp = plan_cluster(dtype, g, QuantIO{}, true, g_tune);      // null pointers: alignment is assumed
    if (kp.ok) {
        const int64_t ctas = count * ((g.C + kp.k - 1) / kp.k * kp.R);
        const bool few_slabs = g.outer <= 3 * (int64_t)kp.R;
        if (!(large && ctas >= 9ll * sms) && !(few_slabs && ctas >= 5ll * sms)) return 0;
    }
    plan = plan_colteam(dtype, g, QuantIO{}, true, sms, g_tune, (uint32_t)count);
    return plan.ok && plan.lag ? count : 0;
}

// Tensors of a list from `first` on that are launched together (list_takes()): on workspaces handed over as zero.  0: none; -1: the
// launch failed.
static int batch_together(const granq_fused_desc* descs, int first, int n_tensors, int dtype, int channel_axis, int group,
                          uint32_t flags, void* cuda_stream) {
    const StagedTuning& t = g_tune;
    if (flags != GRANQ_FLAG_WORKSPACE_ZEROED || !dtype_ok(dtype) || t.cl_tile_kb || t.cl_r || t.cl_threads || t.cl_load ||
        t.cl_prefetch || t.cl_kmul || t.cl_pdl || t.col_team == 2)
        return 0;
    Geom g;
    int64_t G;
    if (!make_geom(descs[first].dims, channel_axis, group, g, G)) return 0;
    auto like_first = [&](int k) {
        for (int i = 0; i < 4; ++i)
            if (descs[first + k].dims[i] != descs[first].dims[i]) return false;
        return true;
    };
    int alike = 1;
    while (first + alike < n_tensors && alike < (int)kTeamListMax && like_first(alike)) ++alike;
    int dev = 0, sms = 0;
    TeamPlan plan{};
    if (alike < 2 || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || list_takes(dtype, g, alike, sms, plan) == 0)
        return 0;
    const size_t nb = (size_t)g.E * elt_size(dtype);
    TeamTensor tensors[kTeamListMax];
    int n = 0;
    for (; n < alike; ++n) {
        const granq_fused_desc& d = descs[first + n];
        bool fits = d.x && d.gy_opt && d.y && d.gx_opt && d.min_out && d.max_out && d.bits >= 1 && d.bits <= 8 &&
                    !(((uintptr_t)d.x | (uintptr_t)d.gy_opt | (uintptr_t)d.y | (uintptr_t)d.gx_opt) & 15) &&
                    check_workspace(d.workspace, d.workspace_bytes, G) == GRANQ_OK &&
                    !(overlaps(d.x, nb, d.y, nb) || overlaps(d.x, nb, d.gx_opt, nb) || overlaps(d.gy_opt, nb, d.y, nb) ||
                      overlaps(d.gy_opt, nb, d.gx_opt, nb) || overlaps(d.y, nb, d.gx_opt, nb));
        for (int k = 0; fits && k < n; ++k) fits = !batch_conflict(descs[first + k], d, dtype, channel_axis, group);
        if (!fits) break;
        tensors[n] = {QuantIO{d.x, d.gy_opt, d.y, d.gx_opt}, d.bits, carve_workspace(d.workspace, G), d.min_out, d.max_out,
                      d.scale_opt, d.zp_opt};
    }
    if (n < alike && list_takes(dtype, g, n, sms, plan) == 0) return 0;
    const cudaError_t e = launch_colteam_list(plan, tensors, (uint32_t)n, dtype, g, g_tune, (cudaStream_t)cuda_stream);
    if (e == cudaErrorCooperativeLaunchTooLarge) return 0;
    return e == cudaSuccess ? n : -1;
}

// Calls that share no memory may run beside one another (their kernels are chained so that the last one's completion is
// everyone's): a kernel of a few MB is a chain of latencies that leaves most of the chip idle.  Every eighth call, and
// one that shares memory with a call since, waits for those ahead of it as a call of its own would.  The 19 activations
// of the small network at batch 256: 238 -> 217 us; with the seven of 17 MB and the six of 8 MB taken together 157.
int granq_fakequant_fused_batch(const granq_fused_desc* descs, int n_tensors, int dtype, int channel_axis, int group,
                                uint32_t flags, void* cuda_stream, int* failed_opt) {
    constexpr int kTogether = 8;
    if (failed_opt) *failed_opt = -1;
    if (!descs || n_tensors < 0) return GRANQ_ERR_INVALID_ARG;
    int first = 0;                 // the calls since the last one that waited, itself included, are [first, i)
    for (int i = 0; i < n_tensors; ++i) {
        const granq_fused_desc& d = descs[i];
        const int together = batch_together(descs, i, n_tensors, dtype, channel_axis, group, flags, cuda_stream);
        if (together) {
            if (together < 0) {
                if (failed_opt) *failed_opt = i;
                return GRANQ_ERR_CUDA;
            }
            i += together - 1;
            first = i + 1;
            continue;
        }
        bool independent = i > first && i - first < kTogether && dtype_ok(dtype);
        for (int k = first; independent && k < i; ++k)
            if (batch_conflict(descs[k], d, dtype, channel_axis, group)) independent = false;
        if (!independent) first = i;
        const int rc = fused_call(d.x, d.gy_opt, dtype, d.dims, channel_axis, group, d.bits, d.y, d.gx_opt, d.min_out,
                                  d.max_out, nullptr, nullptr, d.scale_opt, d.zp_opt, d.workspace, d.workspace_bytes, flags,
                                  cuda_stream, independent, n_tensors > 1);
        if (rc != GRANQ_OK) {
            if (failed_opt) *failed_opt = i;
            return rc;
        }
    }
    return GRANQ_OK;
}

int granq_distortion(const void* x, const void* q, int dtype, const int64_t dims[4], double* sums_out,
                     uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!x || !q || !sums_out || !dtype_ok(dtype) || !make_geom(dims, 1, GRANQ_GROUP_TENSOR, g, G) ||
        ((uintptr_t)sums_out & 7))
        return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    cudaError_t e = launch_clear(nullptr, 0, sums_out, st);
    if (e == cudaSuccess) e = launch_distortion(x, q, dtype, g.E, sums_out, st);
    return cuda_status(e);
}

int granq_distortion_stats(const double sums[4], double* cosine_out, double* rel_error_out) {
    if (!sums) return GRANQ_ERR_INVALID_ARG;
    const double sxx = sums[0], sqq = sums[1], sxq = sums[2], sdd = sums[3];
    const double den = sqrt(sxx) * sqrt(sqq);
    if (cosine_out) *cosine_out = den > 0.0 ? sxq / den : 0.0;
    if (rel_error_out) *rel_error_out = sxx > 0.0 ? sqrt(sdd) / sqrt(sxx) : 0.0;
    return GRANQ_OK;
}

int granq_fakequant_fused_stats(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group,
                                int bits, void* y, float* min_out, float* max_out, float* scale_opt, float* zp_opt,
                                double* sums_out, void* workspace, size_t workspace_bytes, uint32_t flags,
                                void* cuda_stream) {
    Geom g;
    int64_t G;
    if (!x || !y || !sums_out || !min_out || !max_out || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)sums_out & 7))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype);
    if (overlaps(x, nb, y, nb) || overlaps(x, nb, sums_out, 32) || overlaps(y, nb, sums_out, 32))
        return GRANQ_ERR_INVALID_ARG;
    if (int rc = check_workspace(workspace, workspace_bytes, G)) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, y, nullptr, nullptr, nullptr, nullptr, sums_out};
    // the column-walk kernel where there are slabs to walk, else range pass + flat pass (layer-wise and
    // per-sample groups): the statistics are gathered in the pass that writes y either way
    ColPlan cp{};
    ClusterPlan kp{};
    const bool two_pass = (flags & GRANQ_FLAG_FORCE_TWO_PASS) != 0;
    if (!two_pass && !(flags & GRANQ_FLAG_FORCE_COLWALK)) kp = plan_cluster(dtype, g, io, false, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_CLUSTER) && !kp.ok) return GRANQ_ERR_UNSUPPORTED;
    if (!two_pass && !kp.ok) cp = plan_colwalk(dtype, g, io, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_COLWALK) && !cp.ok) return GRANQ_ERR_UNSUPPORTED;
    Workspace ws = carve_workspace(workspace, G);
    const bool zeroed = (flags & GRANQ_FLAG_WORKSPACE_ZEROED) != 0;
    kp.zero_status = !zeroed && kp.clears_status;
    HoldPlan hp{};
    if (kp.ok) hp = hold_over_cluster(dtype, g, io, flags);
    else if (!cp.ok) hp = prefer_hold(dtype, g, io, flags);
    const TeamPlan tp = kp.ok && !hp.ok ? prefer_team(dtype, g, io, false, flags) : TeamPlan{};
    // the team form needs zeroed keys and counters; of the cluster kernel, the status word where it does not write it
    const size_t clear = zeroed ? 0 : !kp.ok || tp.ok || hp.ok ? ws.clear_bytes : kp.clears_status ? 0 : sizeof(uint32_t);
    cudaError_t e = launch_clear(workspace, clear, sums_out, st);
    ws.cleared = true;
    if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    if (hp.ok) {
        e = launch_hold(hp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
        if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_status(e);
        e = cudaSuccess;
    }
    if (kp.ok)
        return cuda_status(launch_held(tp, kp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, st));
    if (cp.ok) {
        e = launch_colwalk(cp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_opt, zp_opt, g_tune, st);
    } else {
        e = launch_range(x, dtype, g, ws.kmin, ws.kmax, ws.counters, min_out, max_out, bits, scale_opt, zp_opt, ws.cleared, st);
        io.behind_range = true;
        if (e == cudaSuccess) e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_out, max_out, st);
        if (e == cudaSuccess && zeroed)
            e = cudaMemsetAsync((char*)workspace + sizeof(uint32_t), 0, ws.clear_bytes - sizeof(uint32_t), st);
    }
    return cuda_status(e);
}

size_t granq_packed_codes_bytes(const int64_t dims[4], int bits) {
    Geom g;
    int64_t G;
    if (bits < 1 || bits > 8 || !make_geom(dims, 1, GRANQ_GROUP_TENSOR, g, G)) return 0;
    return (size_t)((g.E * bits + 31) / 32) * 4;
}

int granq_quantize_packed(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group, int bits,
                          const float* min_in, const float* max_in, uint32_t* packed_codes, void* y_opt,
                          float* scale_out, float* zp_out, uint32_t flags, void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!x || !packed_codes || !min_in || !max_in || !scale_out || !zp_out || bits < 1 || bits > 8 ||
        !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)packed_codes & 3))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype), cbytes = (size_t)((g.E * bits + 31) / 32) * 4;
    if (overlaps(x, nb, y_opt, nb) || overlaps(x, nb, packed_codes, cbytes) || overlaps(y_opt, nb, packed_codes, cbytes))
        return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, y_opt, nullptr, nullptr, nullptr, nullptr, nullptr, packed_codes, bits};
    cudaError_t e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_in, max_in, st);
    if (e == cudaSuccess) e = launch_params(min_in, max_in, G, bits, scale_out, zp_out, st);
    return cuda_status(e);
}

int granq_quantize_packed_fused(const void* x, int dtype, const int64_t dims[4], int channel_axis, int group, int bits,
                                uint32_t* packed_codes, float* min_out, float* max_out, float* scale_out, float* zp_out,
                                void* workspace, size_t workspace_bytes, uint32_t flags, void* cuda_stream) {
    Geom g;
    int64_t G;
    if (!x || !packed_codes || !min_out || !max_out || !scale_out || !zp_out || bits < 1 || bits > 8 ||
        !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)packed_codes & 3))
        return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const size_t nb = (size_t)g.E * elt_size(dtype), cbytes = (size_t)((g.E * bits + 31) / 32) * 4;
    if (overlaps(x, nb, packed_codes, cbytes)) return GRANQ_ERR_INVALID_ARG;
    if (int rc = check_workspace(workspace, workspace_bytes, G)) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    QuantIO io{x, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, packed_codes, bits};
    // the cluster-local kernel where a run of whole groups of 8 codes fits one cluster, the column walk where
    // slabs and waves are such groups, else range pass, parameters, elementwise pass
    ColPlan cp{};
    ClusterPlan kp{};
    const bool two_pass = (flags & GRANQ_FLAG_FORCE_TWO_PASS) != 0;
    if (!two_pass && !(flags & GRANQ_FLAG_FORCE_COLWALK)) kp = plan_cluster(dtype, g, io, false, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_CLUSTER) && !kp.ok) return GRANQ_ERR_UNSUPPORTED;
    if (!two_pass && !kp.ok) cp = plan_colwalk(dtype, g, io, g_tune);
    if ((flags & GRANQ_FLAG_FORCE_COLWALK) && !cp.ok) return GRANQ_ERR_UNSUPPORTED;
    Workspace ws = carve_workspace(workspace, G);
    const bool zeroed = (flags & GRANQ_FLAG_WORKSPACE_ZEROED) != 0;
    kp.zero_status = !zeroed && kp.clears_status;
    cudaError_t e = cudaSuccess;
    HoldPlan hp{};
    if (kp.ok) hp = hold_over_cluster(dtype, g, io, flags);
    else if (!cp.ok) hp = prefer_hold(dtype, g, io, flags);
    const TeamPlan tp = kp.ok && !hp.ok ? prefer_team(dtype, g, io, false, flags) : TeamPlan{};
    if (hp.ok) {
        if (!zeroed) e = clear_workspace(ws, g, kHostBoundHeld, st);
        if (e != cudaSuccess) return GRANQ_ERR_CUDA;
        e = launch_hold(hp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_out, zp_out, g_tune, st);
        if (e != cudaErrorCooperativeLaunchTooLarge) return cuda_status(e);
        e = cudaSuccess;
    }
    if (kp.ok) {
        // the team form needs zeroed keys and counters; of the cluster kernel, the status word where it does not write it
        if (!zeroed && (tp.ok || !kp.clears_status))
            e = launch_clear(workspace, tp.ok ? ws.clear_bytes : sizeof(uint32_t), nullptr, st);
        ws.cleared = !zeroed && tp.ok;
        if (e != cudaSuccess) return GRANQ_ERR_CUDA;
        return cuda_status(launch_held(tp, kp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_out, zp_out, st));
    }
    if (!zeroed && !hp.ok) e = clear_workspace(ws, g, 0, st);
    if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    if (cp.ok) {
        e = launch_colwalk(cp, io, MODE_FWD, dtype, g, bits, ws, min_out, max_out, scale_out, zp_out, g_tune, st);
    } else {
        e = launch_range(x, dtype, g, ws.kmin, ws.kmax, ws.counters, min_out, max_out, bits, scale_out, zp_out, ws.cleared, st);
        io.behind_range = true;
        if (e == cudaSuccess) e = launch_quant_flat(io, MODE_FWD, dtype, g, bits, min_out, max_out, st);
        if (e == cudaSuccess && zeroed)
            e = cudaMemsetAsync((char*)workspace + sizeof(uint32_t), 0, ws.clear_bytes - sizeof(uint32_t), st);
    }
    return cuda_status(e);
}

int granq_dequantize_packed(const uint32_t* packed_codes, int dtype, const int64_t dims[4], int channel_axis,
                            int group, int bits, const float* scale_in, const float* zp_in, void* y, uint32_t flags,
                            void* cuda_stream) {
    (void)flags;
    Geom g;
    int64_t G;
    if (!packed_codes || !scale_in || !zp_in || !y || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G) || ((uintptr_t)packed_codes & 3))
        return GRANQ_ERR_INVALID_ARG;
    const size_t nb = (size_t)g.E * elt_size(dtype), cbytes = (size_t)((g.E * bits + 31) / 32) * 4;
    if (overlaps(y, nb, packed_codes, cbytes)) return GRANQ_ERR_INVALID_ARG;
    return cuda_status(launch_dequant_packed(packed_codes, y, dtype, g, bits, scale_in, zp_in, (cudaStream_t)cuda_stream));
}

int granq_workspace_status(const void* workspace, void* cuda_stream) {
    if (!workspace) return GRANQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    uint32_t word = 0;
    if (cudaMemcpyAsync(&word, workspace, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return GRANQ_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return GRANQ_ERR_CUDA;
    return word == 0 ? GRANQ_OK : (word == GRANQ_ERR_TIMEOUT ? GRANQ_ERR_TIMEOUT : GRANQ_ERR_CUDA);
}

// arena layout: x | gy | y | gx | lo | hi | s | z | workspace, each piece 256-byte aligned
size_t granq_host_arena_bytes(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward) {
    Geom g;
    int64_t G;
    if (!dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return 0;
    const size_t nb = align256((size_t)g.E * elt_size(dtype));
    return nb * (with_backward ? 4 : 2) + 4 * align256((size_t)G * 4) + workspace_bytes_for(G);
}

int granq_fakequant_fused_host(const void* x_host, const void* gy_host_opt, int dtype, const int64_t dims[4],
                               int channel_axis, int group, int bits, void* y_host, void* gx_host_opt,
                               float* min_host, float* max_host, float* scale_host_opt, float* zp_host_opt,
                               void* device_arena, size_t arena_bytes, uint32_t flags, void* cuda_stream) {
    Geom g;
    int64_t G;
    if (!x_host || !y_host || !min_host || !max_host || bits < 1 || bits > 8 || !dtype_ok(dtype) ||
        !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    if ((gy_host_opt == nullptr) != (gx_host_opt == nullptr)) return GRANQ_ERR_INVALID_ARG;
    if (G >= (1ll << 31)) return GRANQ_ERR_UNSUPPORTED;
    const int bwd = gy_host_opt ? 1 : 0;
    if (!device_arena || ((uintptr_t)device_arena & 255) ||
        arena_bytes < granq_host_arena_bytes(dtype, dims, channel_axis, group, bwd))
        return GRANQ_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const size_t raw = (size_t)g.E * elt_size(dtype), nb = align256(raw), gb = align256((size_t)G * 4);
    char* p = (char*)device_arena;
    char* dx = p; p += nb;
    char* dgy = nullptr; if (bwd) { dgy = p; p += nb; }
    char* dy = p; p += nb;
    char* dgx = nullptr; if (bwd) { dgx = p; p += nb; }
    float* dlo = (float*)p; p += gb;
    float* dhi = (float*)p; p += gb;
    float* ds = (float*)p; p += gb;
    float* dz = (float*)p; p += gb;
    void* ws = p;
    if (cudaMemcpyAsync(dx, x_host, raw, cudaMemcpyHostToDevice, st) != cudaSuccess) return GRANQ_ERR_CUDA;
    if (bwd && cudaMemcpyAsync(dgy, gy_host_opt, raw, cudaMemcpyHostToDevice, st) != cudaSuccess)
        return GRANQ_ERR_CUDA;
    int rc = granq_fakequant_fused(dx, dgy, dtype, dims, channel_axis, group, bits, dy, dgx, dlo, dhi, nullptr,
                                   nullptr, scale_host_opt ? ds : nullptr, zp_host_opt ? dz : nullptr, ws,
                                   workspace_bytes_for(G), flags, cuda_stream);
    if (rc != GRANQ_OK) return rc;
    cudaError_t e = cudaMemcpyAsync(y_host, dy, raw, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && bwd) e = cudaMemcpyAsync(gx_host_opt, dgx, raw, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(min_host, dlo, (size_t)G * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(max_host, dhi, (size_t)G * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && scale_host_opt)
        e = cudaMemcpyAsync(scale_host_opt, ds, (size_t)G * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && zp_host_opt) e = cudaMemcpyAsync(zp_host_opt, dz, (size_t)G * 4, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return GRANQ_ERR_CUDA;
    if (flags & GRANQ_FLAG_HOST_ASYNC) return GRANQ_OK;
    return granq_workspace_status(ws, cuda_stream);
}

int granq_host_arena_status(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward,
                            const void* device_arena, void* cuda_stream) {
    Geom g;
    int64_t G;
    if (!device_arena || !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    const size_t nb = align256((size_t)g.E * elt_size(dtype)), gb = align256((size_t)G * 4);
    const char* ws = (const char*)device_arena + nb * (with_backward ? 4 : 2) + 4 * gb;
    return granq_workspace_status(ws, cuda_stream);
}

// Stand-ins for a call's arrays, 16-byte aligned, for what a query asks of a plan.
static QuantIO aligned_io(bool backward, bool packed) {
    QuantIO io{};
    void* const some = (void*)256;
    io.x = io.y = some;
    if (backward) io.gy = io.gx = some;
    if (packed) io.pmask = (uint32_t*)some;
    return io;
}

int granq_fused_plan(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward,
                     uint32_t flags, int* launches_out) {
    Geom g;
    int64_t G;
    if (!dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return -GRANQ_ERR_INVALID_ARG;
    const QuantIO io = aligned_io(with_backward != 0, false);
    const int plan = choose_plan(dtype, g, io, with_backward != 0, flags, nullptr, nullptr, nullptr, nullptr);
    if (launches_out) {
        const bool held = plan == PLAN_TWO_PASS && prefer_hold(dtype, g, io, flags).ok;
        if (held || plan == PLAN_STAGED || plan == PLAN_L2WAVE || plan == PLAN_COLWALK || plan == PLAN_CLUSTER || plan == PLAN_ROWS) *launches_out = 1;
        else if (plan == PLAN_NAIVE) *launches_out = (int)(3 * g.C);
        else if (plan == PLAN_TWO_PASS) *launches_out = g.C <= 4096 ? 2 : 3;
    }
    return plan;
}

int granq_staged_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int sm_count,
                          int smem_bytes, int64_t out[8]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    QuantIO io{};
    StagedPlan p = plan_staged_on(dtype, g, io, sm_count, smem_bytes, g_tune);
    if (!p.ok) return GRANQ_ERR_UNSUPPORTED;
    out[0] = p.grid; out[1] = p.threads; out[2] = p.depth; out[3] = p.smem_bytes;
    out[4] = p.buf_units; out[5] = p.cw; out[6] = p.cu; out[7] = p.nwaves;
    return GRANQ_OK;
}

int granq_cluster_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward,
                           int64_t out[8]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    QuantIO io{};
    ClusterPlan p = plan_cluster(dtype, g, io, with_backward != 0, g_tune);
    if (!p.ok) return GRANQ_ERR_UNSUPPORTED;
    out[0] = (int64_t)((g.C + p.k - 1) / p.k) * p.R; out[1] = p.threads; out[2] = p.R; out[3] = p.smem_bytes;
    out[4] = p.tile_bytes; out[5] = p.k; out[6] = p.load; out[7] = p.prefetch_gy ? 1 : 0;
    return GRANQ_OK;
}

int granq_rows_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward, int sm_count,
                        int64_t out[4]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || sm_count < 1 || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    const QuantIO io{};
    RowsCut cut{};
    if (!plan_rows(dtype, g, io) || !cut_rows(dtype, g, with_backward != 0, 2u * (uint32_t)sm_count, cut)) return GRANQ_ERR_UNSUPPORTED;
    const int64_t v[4] = {cut.P, cut.slices, cut.lanes, cut.team};
    for (int i = 0; i < 4; ++i) out[i] = v[i];
    return GRANQ_OK;
}

int granq_team_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward, int sm_count,
                        int64_t out[5]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || sm_count < 1 || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    const TeamPlan p = plan_colteam(dtype, g, QuantIO{}, with_backward != 0, sm_count, g_tune);
    if (!p.ok) return GRANQ_ERR_UNSUPPORTED;
    const int64_t v[5] = {p.R, p.teams, (p.lag ? 2 : 1) * p.tile_units, (g.C + p.teams - 1) / p.teams, team_over_waves(p, g, g_tune) ? 1 : 0};
    for (int i = 0; i < 5; ++i) out[i] = v[i];
    return GRANQ_OK;
}

int granq_forward_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int packed_mask, int sm_count, int64_t out[4]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || sm_count < 1 || !make_geom(dims, channel_axis, group, g, G)) return GRANQ_ERR_INVALID_ARG;
    ColsCut cut{};
    if (!cut_cols(dtype, g, packed_mask != 0, sm_count, cut)) return GRANQ_ERR_UNSUPPORTED;
    const int64_t v[4] = {cut.side, cut.ncol, cut.rows, cut.walk};
    for (int i = 0; i < 4; ++i) out[i] = v[i];
    return GRANQ_OK;
}

int granq_hold_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int with_backward, int packed, int sm_count,
                        int64_t out[4]) {
    Geom g;
    int64_t G;
    if (!out || !dtype_ok(dtype) || sm_count < 1 || (with_backward && packed) || !make_geom(dims, channel_axis, group, g, G))
        return GRANQ_ERR_INVALID_ARG;
    const bool backward = with_backward != 0;
    const QuantIO io = aligned_io(backward, packed != 0);
    const HoldPlan p = plan_hold(dtype, g, io, sm_count);
    if (!p.ok || !p.whole) return GRANQ_ERR_UNSUPPORTED;
    const int plan = packed ? (plan_cluster(dtype, g, io, false, g_tune).ok ? PLAN_CLUSTER : plan_colwalk(dtype, g, io, g_tune).ok ? PLAN_COLWALK : PLAN_TWO_PASS)
                            : choose_plan(dtype, g, io, backward, 0, nullptr, nullptr, nullptr, nullptr);
    const bool taken = ((plan == PLAN_TWO_PASS || plan == PLAN_L2WAVE) && hold_allowed(0)) || (plan == PLAN_CLUSTER && hold_over_cluster(dtype, g, io, 0).ok);
    const int64_t v[4] = {p.ctas, p.share, p.held, taken ? 1 : 0};
    for (int i = 0; i < 4; ++i) out[i] = v[i];
    return GRANQ_OK;
}

int granq_batch_geometry(int dtype, const int64_t dims[4], int channel_axis, int group, int n_tensors, int sm_count) {
    Geom g;
    int64_t G;
    if (!dtype_ok(dtype) || n_tensors < 0 || sm_count < 1 || !make_geom(dims, channel_axis, group, g, G)) return -GRANQ_ERR_INVALID_ARG;
    TeamPlan plan{};
    return list_takes(dtype, g, n_tensors, sm_count, plan);
}

int granq_tune(int knob, int value) {
    switch (knob) {
        case GRANQ_KNOB_STAGED_DEPTH: g_tune.depth = value; return GRANQ_OK;
        case GRANQ_KNOB_STAGED_MAX_BUF_UNITS: g_tune.max_buf_units = value; return GRANQ_OK;
        case GRANQ_KNOB_STAGED_GRID: g_tune.grid = value; return GRANQ_OK;
        case GRANQ_KNOB_SPIN_LIMIT: g_tune.spin_limit = value; return GRANQ_OK;
        case GRANQ_KNOB_TEST_EXTRA_ARRIVALS: g_tune.extra_arrivals = value; return GRANQ_OK;
        case GRANQ_KNOB_STAGED_CTAS_PER_SM: g_tune.ctas_per_sm = value; return GRANQ_OK;
        case GRANQ_KNOB_L2_WAVE_KB: g_tune.l2_wave_kb = value; return GRANQ_OK;
        case GRANQ_KNOB_L2_UPL: g_tune.l2_upl = value; return GRANQ_OK;
        case GRANQ_KNOB_L2_CTAS_PER_SM: g_tune.l2_ctas_per_sm = value; return GRANQ_OK;
        case GRANQ_KNOB_L2_LAG: g_tune.l2_lag = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_TILE_KB: g_tune.cl_tile_kb = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_CTAS: g_tune.cl_r = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_THREADS: g_tune.cl_threads = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_LOAD: g_tune.cl_load = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_PREFETCH: g_tune.cl_prefetch = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_KMUL: g_tune.cl_kmul = value; return GRANQ_OK;
        case GRANQ_KNOB_CLUSTER_EARLY_LAUNCH: g_tune.cl_pdl = value; return GRANQ_OK;
        case GRANQ_KNOB_COLWALK_TEAM: g_tune.col_team = value; return GRANQ_OK;
        case GRANQ_KNOB_TEST_COOP_CTAS: g_tune.coop_ctas = value; return GRANQ_OK;
        default: return GRANQ_ERR_INVALID_ARG;
    }
}

}  // extern "C"
