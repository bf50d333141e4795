// Generic GranQ kernels: they accept any geometry and any pointer alignment and make no
// assumption about what fits on chip.  The fused two-pass plan is
//   range_flat_kernel (Eq. 4)  ->  finalize_range_kernel (Eq. 5)  ->  quant_flat_kernel (Eq. 1, 6, STE)
// and the stand-alone entry points (range / forward / backward) use the same kernels.
// Also here: the "conventional" per-channel loop the paper measures against (Section 5.3.2).
#include "granq_internal.h"

#include <algorithm>

namespace granq {

namespace {

constexpr int kThreads = 256;
constexpr uint32_t kTile = 8192;          // elements per CTA tile
constexpr int kUnroll = 4;                // 16-byte loads in flight per thread
constexpr uint32_t kTableMax = 1026;      // planes of one tile whose (s, z) are tabled in shared memory

struct FlatGeom {
    int64_t E, inner, C, ntiles;
    FastDiv div_inner, div_C;   // valid when the divisor is < 2^30
    int inner_big, C_big;       // divisor >= 2^30: at most one wrap inside a tile
};

FlatGeom make_flat(const Geom& g) {
    FlatGeom f;
    f.E = g.E;
    f.inner = g.inner;
    f.C = g.C;
    f.ntiles = (g.E + kTile - 1) / kTile;
    f.inner_big = g.inner >= (1ll << 30);
    f.C_big = g.C >= (1ll << 30);
    f.div_inner = make_fastdiv(f.inner_big ? 1u : (uint32_t)g.inner);
    f.div_C = make_fastdiv(f.C_big ? 1u : (uint32_t)g.C);
    return f;
}

// Position of a tile's first element: plane remainder and group of its first plane.
struct TileBase {
    int64_t rem;      // e0 % inner
    uint32_t c;       // (e0 / inner) % C
};

__device__ __forceinline__ TileBase tile_base(const FlatGeom& g, int64_t e0) {
    TileBase b;
    int64_t p = e0 / g.inner;
    b.rem = e0 - p * g.inner;
    b.c = (uint32_t)(p % g.C);
    return b;
}

// plane offset (relative to the tile's first plane) of the element k elements into the tile
__device__ __forceinline__ uint32_t plane_offset(const FlatGeom& g, const TileBase& b, uint32_t k) {
    if (g.inner_big) return (b.rem + (int64_t)k >= g.inner) ? 1u : 0u;
    return g.div_inner.div((uint32_t)b.rem + k);
}
// group of the plane `q` planes after the tile's first plane
__device__ __forceinline__ uint32_t group_at(const FlatGeom& g, const TileBase& b, uint32_t q) {
    if (g.C_big) {
        int64_t v = (int64_t)b.c + q;
        return (uint32_t)(v >= g.C ? v - g.C : v);
    }
    uint32_t v = b.c + q, quo, r;
    g.div_C.divmod(v, quo, r);
    return r;
}

// What the last block of a range launch turns the keys into (Eq. 4, Eq. 5); without a counter the keys stay keys.
struct RangeEnd {
    uint32_t* counter;      // zero on entry; blocks that have published
    const uint32_t* kmin;
    const uint32_t* kmax;
    float* lo;
    float* hi;
    float* s_opt;
    float* z_opt;
    uint32_t G;
    int bits;               // 0: lo and hi alone
};

__device__ __forceinline__ void finalize_group(const uint32_t* kmin, const uint32_t* kmax, int64_t i, float* lo, float* hi,
                                               int bits, float* s_opt, float* z_opt) {
    float l, h;
    keys_to_range(__ldcg(kmin + i), __ldcg(kmax + i), l, h);
    lo[i] = l;
    hi[i] = h;
    if (bits > 0) {
        const QParam p = make_qparam(l, h, (float)((1 << bits) - 1));
        if (s_opt) s_opt[i] = p.s;
        if (z_opt) z_opt[i] = p.z;
    }
}

// Must be called by every thread of the block, after its last atomic on the keys.  Saves a launch per range call; the
// host gives no counter where the groups are so many that one block would take longer than a launch.
__device__ __forceinline__ void finish_range(const RangeEnd& e) {
    if (!e.counter) return;
    __shared__ uint32_t s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(e.counter, 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (uint32_t i = threadIdx.x; i < e.G; i += kThreads) finalize_group(e.kmin, e.kmax, i, e.lo, e.hi, e.bits, e.s_opt, e.z_opt);
}

// ---- Eq. 4: range ------------------------------------------------------------------------------
// V = elements per load: a 16-byte pack when planes and pointers allow it, else 1.
template <typename T, int V>
__global__ void __launch_bounds__(kThreads, 8) range_flat_kernel(const T* __restrict__ x, FlatGeom g,
                                                              uint32_t* __restrict__ kmin,
                                                              uint32_t* __restrict__ kmax, RangeEnd end) {
    after_the_kernel_ahead();
    __shared__ TileBase s_base;
    WarpRun run{kNoGroup, 0u, 0u};
    for (int64_t tile = blockIdx.x; tile < g.ntiles; tile += gridDim.x) {
        const int64_t e0 = tile * (int64_t)kTile;
        const uint32_t ne = (uint32_t)min((int64_t)kTile, g.E - e0);
        __syncthreads();
        if (threadIdx.x == 0) s_base = tile_base(g, e0);
        __syncthreads();
        const TileBase base = s_base;
        for (uint32_t k0 = 0; k0 < ne; k0 += kThreads * V * kUnroll) {
            uint32_t mn[kUnroll], mx[kUnroll], k[kUnroll];
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                k[j] = k0 + (j * kThreads + threadIdx.x) * V;
                mn[j] = 0;
                mx[j] = 0;
                if (k[j] < ne) {
                    if constexpr (V == 1) {
                        uint32_t e = enc(load_scalar(x + e0 + k[j]));
                        mn[j] = ~e;
                        mx[j] = e;
                    } else {
                        Pack<T> p;
                        p.raw = *reinterpret_cast<const uint4*>(x + e0 + k[j]);
                        float lo = INFINITY, hi = -INFINITY;
                        pack_minmax(p, 0, V, lo, hi);
                        mn[j] = ~enc(lo);
                        mx[j] = enc(hi);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                bool valid = k[j] < ne;
                uint32_t grp = valid ? group_at(g, base, plane_offset(g, base, k[j])) : kNoGroup;
                run_add(run, valid, grp, mn[j], mx[j], kmin, kmax);
            }
        }
    }
    run_flush(run, kmin, kmax);
    finish_range(end);
}

// ---- Eq. 4: range, vector path -----------------------------------------------------------------
// Planes made of whole 16-byte packs, fewer than 2^31 packs: a warp takes rows of 128 consecutive
// packs (two rows in flight), a row that lies in one plane costs one run update, and the CTA
// combines its warps' keys in shared memory before touching the global keys.
constexpr uint32_t kRangeSmemGroups = 1024;

// ALIGNED: planes are whole packs (div_plane divides pack indices); otherwise a pack may straddle two
// planes (div_plane divides element indices, `inner` >= V elements per plane), and `tail` elements may be left behind
// the last whole pack, all of them of the last plane.
template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(kThreads) range_rows_kernel(const uint4* __restrict__ x, uint32_t n_units, uint32_t tail,
                                                              uint32_t inner, FastDiv div_plane, FastDiv div_C,
                                                              uint32_t groups, uint32_t* __restrict__ kmin,
                                                              uint32_t* __restrict__ kmax, RangeEnd end) {
    after_the_kernel_ahead();
    constexpr int V = Pack<T>::V;
    __shared__ uint32_t s_kmn[kRangeSmemGroups], s_kmx[kRangeSmemGroups];
    const bool combine = groups <= kRangeSmemGroups;       // else: straight to the global keys
    if (combine) {
        for (uint32_t i = threadIdx.x; i < groups; i += kThreads) {
            s_kmn[i] = 0;
            s_kmx[i] = 0;
        }
        __syncthreads();
    }
    uint32_t* dmn = combine ? s_kmn : kmin;
    uint32_t* dmx = combine ? s_kmx : kmax;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t nwarps = gridDim.x * (kThreads / 32), gw = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    const uint32_t nrows = (n_units + 127u) / 128u;
    WarpRun run{kNoGroup, 0u, 0u}, run2{kNoGroup, 0u, 0u};
    auto fetch = [&](uint32_t row, Pack<T> (&p)[4]) {
        if (row >= nrows) return;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t u = row * 128u + j * 32 + lane;
            if (u < n_units) p[j].raw = ld_stream_16(x + u);
        }
    };
    auto reduce = [&](uint32_t row, const Pack<T> (&p)[4]) {
        if (row >= nrows) return;
        const uint32_t r0 = row * 128u;
        bool v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = r0 + j * 32 + lane < n_units;
        if constexpr (ALIGNED) {
            float mn[4], mx[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mn[j] = INFINITY;
                mx[j] = -INFINITY;
                if (v[j]) pack_minmax(p[j], 0, V, mn[j], mx[j]);
            }
            const uint32_t pl_first = div_plane.div(r0), pl_last = div_plane.div(min(r0 + 128u, n_units) - 1);
            if (pl_first == pl_last) {
                uint32_t q, g;
                div_C.divmod(pl_first, q, g);
                const float m0 = fminf(fminf(mn[0], mn[1]), fminf(mn[2], mn[3]));
                const float m1 = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                run_add(run, v[0], g, ~enc(m0), enc(m1), dmn, dmx);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t q, g;
                    div_C.divmod(div_plane.div(v[j] ? r0 + j * 32 + lane : r0), q, g);
                    run_add(run, v[j], g, ~enc(mn[j]), enc(mx[j]), dmn, dmx);
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t pl, rem, q, g1, g2;
                div_plane.divmod((v[j] ? r0 + j * 32 + lane : r0) * V, pl, rem);
                const int n1 = (int)min((uint32_t)V, inner - rem);          // elements of the first plane
                div_C.divmod(pl, q, g1);
                div_C.divmod(pl + 1, q, g2);
                float mn1 = INFINITY, mx1 = -INFINITY, mn2 = INFINITY, mx2 = -INFINITY;
                if (v[j]) {
                    pack_minmax(p[j], 0, n1, mn1, mx1);
                    pack_minmax(p[j], n1, V, mn2, mx2);
                }
                run_add(run, v[j], g1, ~enc(mn1), enc(mx1), dmn, dmx);
                run_add(run2, v[j] && n1 < V, g2, ~enc(mn2), enc(mx2), dmn, dmx);
            }
        }
    };
    for (uint32_t row = gw; row < nrows; row += 2 * nwarps) {
        Pack<T> pa[4], pb[4];
        fetch(row, pa);
        fetch(row + nwarps, pb);
        reduce(row, pa);
        reduce(row + nwarps, pb);
    }
    run_flush(run, dmn, dmx);
    if constexpr (!ALIGNED) {
        run_flush(run2, dmn, dmx);
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x < tail) {
            const float v = load_scalar(reinterpret_cast<const T*>(x + n_units) + threadIdx.x);
            if (v == v) {
                atomicMax(dmn + groups - 1, ~enc(v));
                atomicMax(dmx + groups - 1, enc(v));
            }
        }
    }
    if (combine) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < groups; i += kThreads) {
            const uint32_t k1 = s_kmn[i], k2 = s_kmx[i];
            if (k1 | k2) {
                atomicMax(kmin + i, k1);
                atomicMax(kmax + i, k2);
            }
        }
    }
    finish_range(end);
}

// ---- Eq. 4: range, column path -----------------------------------------------------------------
// Slabs made of whole 16-byte units, planes of any size from a unit on: the unit at offset u of a slab belongs to the
// same channel (or pair of channels) in every slab, so a thread keeps one unit column, walks it down a run of slabs
// with its running min / max per element in registers, and folds them once at the end.  A block takes 256 adjacent
// columns (at most 258 channels) of a chunk of the slabs.  For planes shorter than a row of the vector path, or not
// whole units: there every load costs divisions and a change of channel costs a warp reduction.  Bound by HBM and one
// walk's latency.  With one launch less per range (finish_range), a data-parallel layer of [128,960,7,7]: 59.8 -> 41.5 us a
// pass; the range kernel took 26 us of it before.
constexpr uint32_t kColTab = 264;

template <typename T, bool ALIGNED, int U>
__global__ void __launch_bounds__(kThreads) range_cols_kernel(const uint4* __restrict__ x, uint32_t slab_units,
                                                              uint32_t outer, uint32_t chunks, FastDiv div_ncol,
                                                              FastDiv div_plane, uint32_t* __restrict__ kmin,
                                                              uint32_t* __restrict__ kmax, RangeEnd end) {
    after_the_kernel_ahead();
    constexpr int V = Pack<T>::V;
    __shared__ uint32_t s_kmn[kColTab], s_kmx[kColTab];
    for (uint32_t t = threadIdx.x; t < kColTab; t += kThreads) {
        s_kmn[t] = 0;
        s_kmx[t] = 0;
    }
    __syncthreads();
    uint32_t chunk, col;
    div_ncol.divmod(blockIdx.x, chunk, col);
    const uint32_t n0 = (uint32_t)(((uint64_t)chunk * outer) / chunks);
    const uint32_t n1 = (uint32_t)(((uint64_t)(chunk + 1) * outer) / chunks);
    const uint32_t u = col * kThreads + threadIdx.x;
    const bool valid = u < slab_units && n0 < n1;
    float mn[V], mx[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
        mn[i] = INFINITY;
        mx[i] = -INFINITY;
    }
    if (valid) {
        const uint4* p = x + ((size_t)n0 * slab_units + u);
        for (uint32_t n = n0; n < n1; n += U, p += (size_t)U * slab_units) {
            Pack<T> v[U];
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (n + j < n1) v[j].raw = ld_stream_16(p + (size_t)j * slab_units);
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (n + j < n1) {
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        mn[i] = fminf(mn[i], v[j].get(i));
                        mx[i] = fmaxf(mx[i], v[j].get(i));
                    }
                }
        }
    }
    // the channel of this column, of its first `ne` elements where a unit straddles two planes
    const uint32_t uu = valid ? u : col * kThreads;
    uint32_t ch, base;
    int ne = V;
    if constexpr (ALIGNED) {
        ch = div_plane.div(uu);
        base = div_plane.div(col * kThreads);
    } else {
        uint32_t rem;
        div_plane.divmod(uu * V, ch, rem);
        ne = (int)min((uint32_t)V, div_plane.d - rem);
        base = div_plane.div(col * kThreads * V);
    }
    auto keys = [&](int first, int last, uint32_t& ka, uint32_t& kb) {
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (i >= first && i < last) {
                lo = fminf(lo, mn[i]);
                hi = fmaxf(hi, mx[i]);
            }
        ka = lo <= hi ? ~enc(lo) : 0u;
        kb = lo <= hi ? enc(hi) : 0u;
    };
    uint32_t ka, kb;
    keys(0, ne, ka, kb);
    const uint32_t rel = ch - base, rel0 = __shfl_sync(kFullMask, rel, 0);
    if (__all_sync(kFullMask, rel == rel0 && ne == V)) {             // the warp lies in one channel
        ka = __reduce_max_sync(kFullMask, ka);
        kb = __reduce_max_sync(kFullMask, kb);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(s_kmn + rel0, ka);
            atomicMax(s_kmx + rel0, kb);
        }
    } else if (valid) {
        atomicMax(s_kmn + rel, ka);
        atomicMax(s_kmx + rel, kb);
        if (ne < V) {
            keys(ne, V, ka, kb);
            atomicMax(s_kmn + rel + 1, ka);
            atomicMax(s_kmx + rel + 1, kb);
        }
    }
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < kColTab; t += kThreads) {
        const uint32_t k1 = s_kmn[t], k2 = s_kmx[t];
        if (k1 | k2) {
            atomicMax(kmin + base + t, k1);
            atomicMax(kmax + base + t, k2);
        }
    }
    finish_range(end);
}

__global__ void finalize_range_kernel(const uint32_t* __restrict__ kmin, const uint32_t* __restrict__ kmax,
                                      int64_t G, float* __restrict__ lo, float* __restrict__ hi, int bits,
                                      float* __restrict__ s_opt, float* __restrict__ z_opt) {
    after_the_kernel_ahead();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < G) finalize_group(kmin, kmax, i, lo, hi, bits, s_opt, z_opt);
}

__global__ void __launch_bounds__(kThreads) clear_kernel(uint32_t* __restrict__ p, uint32_t words, double* __restrict__ sums) {
    after_the_kernel_ahead();
    for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < words; i += gridDim.x * kThreads) p[i] = 0;
    if (sums && blockIdx.x == 0 && threadIdx.x < 4) sums[threadIdx.x] = 0.0;
}

__global__ void params_kernel(const float* __restrict__ lo, const float* __restrict__ hi, int64_t G, int bits,
                              float* __restrict__ s_opt, float* __restrict__ z_opt) {
    after_the_kernel_ahead();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G) return;
    QParam p = make_qparam(__fadd_rn(lo[i], 0.0f), __fadd_rn(hi[i], 0.0f), (float)((1 << bits) - 1));
    if (s_opt) s_opt[i] = p.s;
    if (z_opt) z_opt[i] = p.z;
}

// Packing a warp's row of integer codes into a bit string.  Every lane holds `nb` bits (its V codes
// of b bits, nb = V * b <= 64): lane i owns bits [i * nb, (i + 1) * nb) of a row of nb 32-bit words.
// Lane k returns word k of the row in out[0] and word k + 32 in out[1] (0 where the row has no such
// word); all 32 lanes must call.
__device__ __forceinline__ void warp_pack_row(uint64_t mine, uint32_t nb, uint32_t lane, uint32_t first0,
                                              uint32_t first1, uint32_t (&out)[2]) {
    // first0 / first1 = (32 * lane) / nb and (32 * (lane + 32)) / nb: the first lane that reaches into the
    // word(s) this lane assembles (lane constants, worked out once per kernel)
    out[0] = 0;
    out[1] = 0;
    if ((nb & (nb - 1)) == 0 && nb <= 32) {              // 32 / nb lanes make up one word exactly
        const uint32_t lpw = 32 / nb;
        uint32_t w = (uint32_t)mine << (nb * (lane & (lpw - 1)));
        for (uint32_t d = 1; d < lpw; d <<= 1) w |= __shfl_xor_sync(kFullMask, w, d);
        out[0] = __shfl_sync(kFullMask, w, (lane * lpw) & 31);      // word k sits in lanes k * lpw ...
        return;
    }
    const uint32_t nsrc = 32 / nb + 2;                   // lanes whose bits can fall into one word
    if (nb <= 32) {                                      // one word per lane at most, 32-bit shuffles
        const uint32_t lo = (uint32_t)mine;
        uint32_t acc = 0;
        for (uint32_t j = 0; j < nsrc; ++j) {
            const uint32_t src = first0 + j;
            const uint32_t v = __shfl_sync(kFullMask, lo, src & 31);
            const int off = (int)(src * nb) - (int)(32 * lane);     // where src's bits start, relative to the word
            if (src < 32 && off < 32 && lane < nb) acc |= off >= 0 ? (v << off) : (v >> (-off));
        }
        out[0] = acc;
        return;
    }
    for (int h = 0; h < 2; ++h) {
        const uint32_t wk = lane + 32 * h;               // word of the row this lane assembles
        const uint32_t first = h ? first1 : first0;
        uint32_t acc = 0;
        for (uint32_t j = 0; j < nsrc; ++j) {
            const uint32_t src = first + j;
            const uint64_t v = __shfl_sync(kFullMask, mine, src & 31);
            const int off = (int)(src * nb) - (int)(32 * wk);
            if (src < 32 && off < 32 && wk < nb) acc |= (uint32_t)(off >= 0 ? (v << off) : (v >> (-off)));
        }
        out[h] = acc;
    }
}

// bf16 where a pack straddles planes, and wherever there is a gradient: four elements of a pack at a time, compiled for
// four blocks per SM; eight at a time take 73 to 99 registers, which costs one or two of them.  Backward [256,512,28,28]
// 147 -> 118 us, range and both directions there 207 -> 188; on ragged planes [256,1024,14,14] forward 82 -> 66, backward
// 92 -> 70, range and both 147 -> 129.  Forward on whole packs is faster the other way (138 / 144).
template <int V, int MODE, int EXTRAS, bool RAGGED>
constexpr bool kFlatParts = V == 8 && (MODE == MODE_BOTH ? EXTRAS == 0 : RAGGED || MODE == MODE_BWD);
// blocks per SM the kernel is compiled for; 0: left to the compiler
template <int V, int MODE, int EXTRAS, bool PACKONLY, bool RAGGED>
constexpr int kFlatBlocks = !kFlatParts<V, MODE, EXTRAS, RAGGED> ? 0 : MODE == MODE_FWD && EXTRAS == 1 ? (PACKONLY ? 3 : 0) : 4;

// ---- Eq. 1, clamp, Eq. 6, STE: elementwise pass with a given per-group range ----------------------
// EXTRAS = 1: the optional codes / mask / packed-mask / sums outputs are compiled in; 2: the packed mask alone; 4: the
// distortion sums alone.  The packed mask holds
// one bit per element (bit e % 32 of word e / 32): a warp's lanes own consecutive elements or packs
// starting at a multiple of 32 elements, so whole words are assembled with warp shuffles.
// PACKONLY: the packed integer codes are the only output (everything else is compiled out).  With EXTRAS = 3
// (tensors of a multiple of 32 elements) the bit string is written 8 codes = b bytes at a time by every second
// fp32 lane (every bf16 lane) with plain stores: no word assembly across the warp.
// RAGGED: planes are not whole 16-byte packs (7x7 planes), so a pack may straddle two planes and takes the
// parameters of both (planes of at least one pack: never more than two).
// END (RAGGED): the last pack is not whole; it is read and written element by element, the rest of it is +0 and says nothing.
// Calls against the scalar form, us: bf16 forward of [31,1509,29,29], 79 MB, range and quantize 236 -> 105; fp32 with gradient
// [51,79,69,69] 142 -> 93, sums [207,77,34,35] 121 -> 73; range, mask and the way back of bf16 [61,225,18,17] 82.5 -> 23.9, fp32
// [22,193,95,95] 323 -> 188; codes and back of [31,157,23,22] bf16 22.8 -> 17.3 (the way back alone).
template <typename T, int V, int MODE, int EXTRAS, bool PACKONLY = false, bool RAGGED = false, bool END = false>
__global__ void __launch_bounds__(kThreads, (kFlatBlocks<V, MODE, EXTRAS, PACKONLY, RAGGED>))
                                            quant_flat_kernel(const T* __restrict__ x, const T* __restrict__ gy,
                                                              T* __restrict__ y, T* __restrict__ gx,
                                                              uint8_t* __restrict__ codes,
                                                              uint8_t* __restrict__ mask,
                                                              uint32_t* __restrict__ pmask,
                                                              double* __restrict__ dist,
                                                              uint32_t* __restrict__ pcodes, int code_bits,
                                                              FlatGeom g, float qmax,
                                                              const float* __restrict__ lo,
                                                              const float* __restrict__ hi) {
    after_the_kernel_ahead();
    __shared__ TileBase s_base;
    __shared__ float s_tab_s[kTableMax], s_tab_z[kTableMax], s_tab_r[kTableMax];
    constexpr bool kParts = kFlatParts<V, MODE, EXTRAS, RAGGED>;
    // The first loads before the parameters, not where their registers cost a block per SM or are spilled, nor in the
    // backward pass on ragged planes ([256,960,7,7] bf16 21.4 -> 22.6 us).
    constexpr bool kEarly = EXTRAS != 1 && !(V == 8 && MODE == MODE_BOTH) && !(RAGGED && MODE == MODE_BWD);
    constexpr bool kFwd = (MODE & MODE_FWD) != 0, kBwd = (MODE & MODE_BWD) != 0;
    DistAcc dacc;
    dacc.reset();
    const uint32_t pk_nb = (uint32_t)(V * (code_bits > 0 ? code_bits : 1));
    const uint32_t pk_first0 = (32 * (threadIdx.x & 31)) / pk_nb, pk_first1 = (32 * ((threadIdx.x & 31) + 32)) / pk_nb;
    for (int64_t tile = blockIdx.x; tile < g.ntiles; tile += gridDim.x) {
        const int64_t e0 = tile * (int64_t)kTile;
        const uint32_t ne = (uint32_t)min((int64_t)kTile, g.E - e0);
        uint32_t k[kUnroll];
        Pack<T> px[kUnroll], pg[kUnroll];
        float sx[kUnroll], sg[kUnroll];
        auto fetch = [&](uint32_t k0) {
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                k[j] = k0 + (j * kThreads + threadIdx.x) * V;
                if (k[j] < ne) {
                    if constexpr (V == 1) {
                        sx[j] = load_scalar(x + e0 + k[j]);
                        if constexpr (kBwd) sg[j] = load_scalar(gy + e0 + k[j]);
                    } else if (END && k[j] + V > ne) {
                        px[j].raw = make_uint4(0, 0, 0, 0);
                        if constexpr (kBwd) pg[j].raw = make_uint4(0, 0, 0, 0);
#pragma unroll
                        for (int i = 0; i < V; ++i)
                            if (k[j] + i < ne) {
                                px[j].set(i, load_scalar(x + e0 + k[j] + i));
                                if constexpr (kBwd) pg[j].set(i, load_scalar(gy + e0 + k[j] + i));
                            }
                    } else {
                        px[j].raw = ld_stream_16(x + e0 + k[j]);
                        if constexpr (kBwd) pg[j].raw = ld_stream_16(gy + e0 + k[j]);
                    }
                }
            }
        };
        if constexpr (kEarly) fetch(0);            // under way while the table is made
        __syncthreads();
        if (threadIdx.x == 0) s_base = tile_base(g, e0);
        __syncthreads();
        const TileBase base = s_base;
        const uint32_t nplanes = plane_offset(g, base, ne - 1) + 1;
        const bool tabled = nplanes <= kTableMax;
        if (tabled) {
            for (uint32_t q = threadIdx.x; q < nplanes; q += kThreads) {
                uint32_t grp = group_at(g, base, q);
                const QParam qp = make_qparam(__fadd_rn(lo[grp], 0.0f), __fadd_rn(hi[grp], 0.0f), qmax);
                s_tab_s[q] = qp.s;
                s_tab_z[q] = qp.z;
                s_tab_r[q] = div_is_safe(qp.s, 0.0f, 0.0f) ? __frcp_rn(qp.s) : 0.0f;
            }
            __syncthreads();
        }
        for (uint32_t k0 = 0; k0 < ne; k0 += kThreads * V * kUnroll) {
            if (!kEarly || k0 > 0) fetch(k0);
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const bool valid = k[j] < ne;
                uint32_t inside_bits = 0;            // bit i: the clamp was inactive for this thread's element i
                uint64_t code_string = 0;            // this thread's V codes, b bits each, first element lowest
                if (valid) {
                const uint32_t q = plane_offset(g, base, k[j]);
                QParam p;
                float rcp = 0.0f;            // reciprocal of the scale when the short division applies
                if (tabled) {
                    p.s = s_tab_s[q];
                    p.z = s_tab_z[q];
                    rcp = s_tab_r[q];
                } else {
                    uint32_t grp = group_at(g, base, q);
                    p = make_qparam(__fadd_rn(lo[grp], 0.0f), __fadd_rn(hi[grp], 0.0f), qmax);
                }
                const int64_t e = e0 + k[j];
                if constexpr (V == 1) {
                    float yv;
                    bool in;
                    float code = quant_one(sx[j], p, qmax, yv, in);
                    inside_bits = in ? 1u : 0u;
                    code_string = (uint64_t)code;
                    if constexpr (kFwd) {
                        if (dist) dacc.add_one(sx[j], as_stored(yv, y));
                        if (y) store_scalar(y + e, yv);
                        if (codes) codes[e] = (uint8_t)code;
                    }
                    if constexpr (kBwd) {
                        store_scalar(gx + e, in ? sg[j] : 0.0f);
                        if (mask) mask[e] = in ? 1 : 0;
                    }
                } else {
                    Pack<T> py, pgx;
                    uint32_t cb[V / 4 > 0 ? V / 4 : 1], mb[V / 4 > 0 ? V / 4 : 1];
                    GroupParam gp{p.s, p.z, rcp, tie_threshold(rcp, p.z, qmax)};
                    GroupParam gp2 = gp;
                    int n1 = V;
                    const bool whole = !END || k[j] + V <= ne;
                    if constexpr (RAGGED) {
                        const uint32_t rem = (uint32_t)base.rem + k[j] - q * (uint32_t)g.inner;      // position inside plane q
                        n1 = whole ? (int)min((uint32_t)V, (uint32_t)g.inner - rem) : V;
                        if (n1 < V) {                                                           // the rest lies in plane q + 1
                            if (tabled) {
                                gp2.s = s_tab_s[q + 1];
                                gp2.z = s_tab_z[q + 1];
                                gp2.r = s_tab_r[q + 1];
                                gp2.thr = tie_threshold(gp2.r, gp2.z, qmax);
                            } else {
                                const uint32_t grp2 = group_at(g, base, q + 1);
                                const QParam p2 = make_qparam(__fadd_rn(lo[grp2], 0.0f), __fadd_rn(hi[grp2], 0.0f), qmax);
                                gp2.s = p2.s;
                                gp2.z = p2.z;
                                gp2.r = 0.0f;
                                gp2.thr = 0.0f;
                            }
                        }
                    }
                    quantize_pack<T, kBwd, RAGGED, EXTRAS, false, kParts>(px[j], pg[j], gp, gp2, n1, qmax, py, pgx, cb, mb, EXTRAS == 3 ? code_bits : 8);
                    if constexpr (END) {
                        if (!whole) {
#pragma unroll
                            for (int i = 0; i < V; ++i)
                                if (k[j] + i < ne) {
                                    if constexpr (kFwd && !PACKONLY) store_scalar(y + e + i, py.get(i));
                                    if constexpr (kBwd) store_scalar(gx + e + i, pgx.get(i));
                                } else {
                                    py.set(i, 0.0f);
                                    if constexpr (EXTRAS == 1) cb[i / 4] &= ~(0xFFu << (8 * (i % 4)));
                                    if constexpr (EXTRAS == 2) mb[0] &= ~(1u << i);
                                }
                        }
                    }
                    if constexpr (EXTRAS == 3) {
                        code_string = code_string_of<V>(cb, code_bits);
                    } else if constexpr (EXTRAS != 0) {
                        if constexpr (!PACKONLY && EXTRAS != 4) inside_bits = mask_bits_of<V, EXTRAS>(mb);
                        if constexpr (EXTRAS == 4) dacc.add(px[j], py);
                        if constexpr (kFwd && EXTRAS == 1) {
                            if (PACKONLY || pcodes) {
#pragma unroll
                                for (int i = 0; i < V; ++i)
                                    code_string |= (uint64_t)((cb[i / 4] >> (8 * (i % 4))) & 0xFFu) << (i * code_bits);
                            }
                        }
                    }
                    if constexpr (kFwd && !PACKONLY) {
                        if ((EXTRAS != 1 || y) && whole) st_stream_16(y + e, py.raw);
                        if constexpr (EXTRAS == 1) {
                            if (codes) {
#pragma unroll
                                for (int i = 0; i < V / 4; ++i) reinterpret_cast<uint32_t*>(codes + e)[i] = cb[i];
                            }
                        }
                    }
                    if constexpr (kBwd) {
                        if (whole) st_stream_16(gx + e, pgx.raw);
                        if constexpr (EXTRAS == 1) {
                            if (mask) {
#pragma unroll
                                for (int i = 0; i < V / 4; ++i) reinterpret_cast<uint32_t*>(mask + e)[i] = mb[i];
                            }
                        }
                    }
                }
                }
                if constexpr (EXTRAS != 0 && EXTRAS != 4 && kFwd) {
                    if (!PACKONLY && pmask) {          // every lane of the warp is here: assemble whole 32-bit words
                        const uint32_t lane = threadIdx.x & 31;
                        const int64_t word = (e0 + k[j]) >> 5;
                        if constexpr (V == 1) {
                            const uint32_t w = __ballot_sync(kFullMask, inside_bits != 0);
                            if (lane == 0 && valid) pmask[word] = w;
                        } else {
                            constexpr uint32_t kLanes = 32 / V;             // lanes that share one word
                            uint32_t w = inside_bits << (V * (lane & (kLanes - 1)));
#pragma unroll
                            for (uint32_t d = 1; d < kLanes; d <<= 1) w |= __shfl_xor_sync(kFullMask, w, d);
                            if ((lane & (kLanes - 1)) == 0 && valid) pmask[word] = w;
                        }
                    }
                    if constexpr (EXTRAS == 3) {
                        // 8 consecutive codes are b whole bytes of the bit string (the tensor is a multiple of 32
                        // elements, so the lanes of a pair are valid or not together, and a lane without a pack has
                        // nothing to say)
                        if constexpr (V > 1) {
                            const uint32_t lanes = V == 4 ? __ballot_sync(kFullMask, valid) : 0u;
                            if (valid) store_code_bytes<V>(pcodes, (size_t)(e0 + k[j]), code_string, code_bits, threadIdx.x & 31, lanes);
                        }
                    } else if (EXTRAS == 1 && (PACKONLY || pcodes)) {      // the warp's 32 * V codes are V * b whole words of the bit string
                        const uint32_t lane = threadIdx.x & 31;
                        const uint32_t nb = (uint32_t)(V * code_bits);
                        const int64_t row_e = e0 + k0 + (int64_t)(j * kThreads + (threadIdx.x & ~31u)) * V;
                        const int64_t word0 = (row_e >> 5) * code_bits, nwords = (g.E * code_bits + 31) >> 5;
                        uint32_t out[2];
                        warp_pack_row(code_string, nb, lane, pk_first0, pk_first1, out);
                        if (lane < nb && word0 + lane < nwords) pcodes[word0 + lane] = out[0];
                        if (lane + 32 < nb && word0 + lane + 32 < nwords) pcodes[word0 + lane + 32] = out[1];
                    }
                }
            }
        }
    }
    if constexpr (EXTRAS == 4 || (V == 1 && EXTRAS == 1 && kFwd)) {      // the scalar form keeps all extras in one
        if (dist) dacc.flush(dist);
    }
}

// ---- Eq. 1, clamp, Eq. 6 with a given range, column path -------------------------------------------
// As range_cols_kernel: a thread keeps one unit column of the slabs (of rows of several short ones) and with it the parameters of its channel, or
// of the two that its unit straddles, in registers, and walks a few of them; y and, PMASK, the packed mask.  In the tile kernel above every pack of a
// short or ragged plane costs a division, two table rows and a choice of parameters per element: 180 instructions a unit at [128,960,7,7] with a
// mask, here about 50.  Tiles / columns, us, without and with a mask: fp32 [128,960,7,7] 9.6 / 7.7, 11.8 / 8.5; [128,256,14,14] 9.5 / 6.3, 11.8 /
// 6.6; [32,64,56,56] 8.7 / 5.7, 11.1 / 6.0; [256,512,28,28], 411 MB, 122 / 123, 134 / 127; bf16 [128,96,33,33] 17.3 / 14.1, 21.0 / 16.5,
// [256,1024,14,14] 60.8 / 46.3, 72.3 / 52.3.  Bound by the instructions of 16 bytes up to a few times the L2, then by HBM.  Eight of bf16 that
// straddle planes keep two units in flight and four blocks per SM (four and three: small tensors 4 to 15 % slower).
template <typename T, bool ALIGNED, bool PMASK>
__global__ void __launch_bounds__(kThreads, 4) quant_cols_kernel(const uint4* __restrict__ x, uint4* __restrict__ y, uint8_t* __restrict__ pmask,
                                                                 ColsCut cut, FastDiv div_ncol, FastDiv div_plane, FastDiv div_C, float qmax,
                                                                 const float* __restrict__ lo, const float* __restrict__ hi) {
    after_the_kernel_ahead();
    constexpr int V = Pack<T>::V, U = V == 8 && !ALIGNED ? 2 : 4, EXTRAS = PMASK ? 2 : 0;
    const uint32_t row_units = cut.row_units;
    uint32_t chunk, col;
    div_ncol.divmod(blockIdx.x, chunk, col);
    const uint32_t n0 = chunk * cut.walk, n1 = min(cut.rows, n0 + cut.walk), lane = threadIdx.x & 31;
    const uint32_t u = col * kThreads + threadIdx.x;
    // the rows this thread has a unit in: none beyond the last column, where lanes walk along for the shuffles, and the tensor may
    // end inside the last row
    const uint32_t end = u >= row_units ? n0 : n1 == cut.rows && u >= cut.last_units ? n1 - 1 : n1;
    const uint4* p = x + ((size_t)n0 * row_units + u);
    Pack<T> px[U];
    auto fetch = [&](uint32_t n) {
#pragma unroll
        for (int j = 0; j < U; ++j)
            if (n + j < end) px[j].raw = ld_stream_16(p + (size_t)j * row_units);
    };
    fetch(n0);                                                // under way while the parameters are made
    const uint32_t own = min(u, row_units - 1);
    uint32_t ch;
    int ne = V;
    if constexpr (ALIGNED) {
        ch = div_plane.div(own);
    } else {
        uint32_t rem;
        div_plane.divmod(own * V, ch, rem);
        ne = (int)min((uint32_t)V, div_plane.d - rem);
    }
    if (cut.side > 1) ch -= div_C.div(ch) * div_C.d;          // (a unit that straddles planes lies in one slab)
    auto params = [&](uint32_t c) {
        const QParam q = make_qparam(__fadd_rn(lo[c], 0.0f), __fadd_rn(hi[c], 0.0f), qmax);
        const float r = div_is_safe(q.s, 0.0f, 0.0f) ? __frcp_rn(q.s) : 0.0f;
        return GroupParam{q.s, q.z, r, tie_threshold(r, q.z, qmax)};
    };
    const GroupParam g1 = params(ch);
    GroupParam g2 = g1;
    if constexpr (!ALIGNED) {
        if (ne < V) g2 = params(ch + 1);
    }
    // fp32: two elements to an instruction where nothing of a pack is clamped or close to a tie
    const float thr = fminf(g1.thr, g2.thr), top = __fadd_rn(kRoundMagic, qmax);
    const float mza = __fadd_rn(kRoundMagic, g1.z), mzb = __fadd_rn(kRoundMagic, g2.z);
    F2 r2[2], mz2[2], ns2[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool a = ALIGNED || 2 * k < ne, b = ALIGNED || 2 * k + 1 < ne;
        r2[k] = f2(a ? g1.r : g2.r, b ? g1.r : g2.r);
        mz2[k] = f2(a ? mza : mzb, b ? mza : mzb);
        ns2[k] = f2(a ? -g1.s : -g2.s, b ? -g1.s : -g2.s);
    }
    auto quantize = [&](const Pack<T>& q, Pack<T>& py, uint32_t& bits) {
        uint32_t cb[V / 4], mb[V / 4];
        if constexpr (V == 4) {
            float m[4], yv[4], worst = 0.0f;
            const F2 zero = {0};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const F2 v = f2(q.get(2 * k), q.get(2 * k + 1)), w = f2_fma(v, r2[k], mz2[k]), e = f2_sub(mz2[k], w);
                float d0, d1;
                f2_split(f2_fma(v, r2[k], e), d0, d1);
                worst = max_or_nan(max_or_nan(worst, fabsf(d0)), fabsf(d1));
                f2_split(f2_fma(ns2[k], e, zero), yv[2 * k], yv[2 * k + 1]);
                f2_split(w, m[2 * k], m[2 * k + 1]);
            }
            const float least = fminf(fminf(m[0], m[1]), fminf(m[2], m[3])), most = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
            if (worst < thr && least >= kRoundMagic && most <= top) {
                py.set_all(yv);
                bits = 15;
                return;
            }
        }
        quantize_pack<T, false, !ALIGNED, EXTRAS, false, true>(q, q, g1, g2, ne, qmax, py, py, cb, mb, 8);
        if constexpr (PMASK) bits = mb[0];
    };
    uint4* out = y + ((size_t)n0 * row_units + u);
    uint32_t at = n0 * row_units + u;                        // of the units of the tensor
    for (uint32_t n = n0; n < n1; n += U) {
        if (n > n0) fetch(n);
        uint32_t bits[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            bits[j] = 0;
            if (n + j < end) {
                Pack<T> py;
                quantize(px[j], py, bits[j]);
                st_stream_16(out + (size_t)j * row_units, py.raw);
                if constexpr (PMASK && V == 8) pmask[at + j * row_units] = (uint8_t)bits[j];
            }
        }
        if constexpr (PMASK && V == 4) {
            const uint32_t bytes = pair_up_mask<U>(bits, lane);
#pragma unroll
            for (int j = 0; j < U; j += 2)
                if (n + j + (lane & 1u) < end) pmask[(at + (j + (lane & 1u)) * row_units) >> 1] = (uint8_t)(bytes >> (4 * j));
        }
        p += (size_t)U * row_units;
        out += (size_t)U * row_units;
        at += U * row_units;
    }
}

// ---- the "conventional" per-channel scheme (Section 5.3.2): one group per launch ------------------
template <typename T, bool IS_MAX>
__global__ void __launch_bounds__(kThreads) naive_extreme_kernel(const T* __restrict__ x, Geom g, int64_t c,
                                                                 uint32_t* __restrict__ key) {
    uint32_t acc = 0;
    for (int64_t o = blockIdx.x; o < g.outer; o += gridDim.x) {
        const T* plane = x + (o * g.C + c) * g.inner;
        for (int64_t i = threadIdx.x; i < g.inner; i += kThreads) {
            uint32_t e = enc(load_scalar(plane + i));
            acc = max(acc, IS_MAX ? e : ~e);
        }
    }
    acc = __reduce_max_sync(kFullMask, acc);
    if ((threadIdx.x & 31) == 0) atomicMax(key, acc);
}

template <typename T, int MODE>
__global__ void __launch_bounds__(kThreads) naive_quant_kernel(const T* __restrict__ x, const T* __restrict__ gy,
                                                               T* __restrict__ y, T* __restrict__ gx,
                                                               uint8_t* __restrict__ codes,
                                                               uint8_t* __restrict__ mask, Geom g, int64_t c,
                                                               float qmax, const uint32_t* __restrict__ kmin,
                                                               const uint32_t* __restrict__ kmax,
                                                               float* __restrict__ lo_out,
                                                               float* __restrict__ hi_out) {
    constexpr bool kFwd = (MODE & MODE_FWD) != 0, kBwd = (MODE & MODE_BWD) != 0;
    float lo, hi;
    keys_to_range(kmin[c], kmax[c], lo, hi);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        lo_out[c] = lo;
        hi_out[c] = hi;
    }
    const QParam p = make_qparam(lo, hi, qmax);
    for (int64_t o = blockIdx.x; o < g.outer; o += gridDim.x) {
        const int64_t b = (o * g.C + c) * g.inner;
        for (int64_t i = threadIdx.x; i < g.inner; i += kThreads) {
            float yv;
            bool in;
            float code = quant_one(load_scalar(x + b + i), p, qmax, yv, in);
            if constexpr (kFwd) {
                store_scalar(y + b + i, yv);
                if (codes) codes[b + i] = (uint8_t)code;
            }
            if constexpr (kBwd) {
                store_scalar(gx + b + i, in ? load_scalar(gy + b + i) : 0.0f);
                if (mask) mask[b + i] = in ? 1 : 0;
            }
        }
    }
}

// ---- STE backward from the packed mask alone (Section 2.1): gx = gy where the element's bit is set ----
// A stream, bound by HBM: a block per 1024 units, in the order of memory ([128,96,112,112] 200 -> 185 us against a
// persistent grid).  The kernel behind is not let start beside it: that is mostly one that takes an SM's shared memory (the next
// layer's), which a stream of a wave or two is slower beside (packed mask and backward, us, with / without: bf16 [128,960,7,7] 26.0 / 21.2,
// fp32 [25,856,14,14] 21.6 / 19.2, [41,1896,15,16] 60.8 / 60.3; 26 shapes 0.98).
// V = elements per thread and step: a 16-byte pack when the pointers allow it, else 1.  What is left behind the whole packs
// is the first threads' of the last block, in a form of its own (END: the test for it took 0.1 us of 2.7).  Four arguments of
// 8 bytes: with a fifth a launch cost the host 0.35 us more (calls one after another, 16 KB tensors: 2.73 -> 2.38 us).
template <typename T, int V, bool END>
__global__ void __launch_bounds__(kThreads) bwd_packmask_kernel(const T* __restrict__ gy,
                                                                const uint32_t* __restrict__ pmask,
                                                                T* __restrict__ gx, int64_t all) {
    wait_for_the_kernel_ahead();      // and no word to the kernel behind
    const int64_t E = END ? all - all % V : all;
    if (END && blockIdx.x == gridDim.x - 1 && threadIdx.x < (uint32_t)(all - E)) {
        const int64_t at = E + threadIdx.x;
        store_scalar(gx + at, (__ldg(pmask + (at >> 5)) >> (uint32_t)(at & 31)) & 1u ? load_scalar(gy + at) : 0.0f);
    }
    const int64_t u0 = (int64_t)blockIdx.x * kThreads * kUnroll;
    int64_t e[kUnroll];
    Pack<T> pg[kUnroll];
    float sg[kUnroll];
    uint32_t w[kUnroll];
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
        e[j] = (u0 + j * kThreads + threadIdx.x) * V;
        if (e[j] < E) {
            if constexpr (V == 1) sg[j] = load_scalar(gy + e[j]);
            else pg[j].raw = ld_stream_16(gy + e[j]);
            w[j] = __ldg(pmask + (e[j] >> 5));
        }
    }
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
        if (e[j] >= E) continue;
        const uint32_t bits = w[j] >> (uint32_t)(e[j] & 31);
        if constexpr (V == 1) {
            store_scalar(gx + e[j], (bits & 1u) ? sg[j] : 0.0f);
        } else {
            Pack<T> out;
            out.select(pg[j], bits);
            st_stream_16(gx + e[j], out.raw);
        }
    }
}

// ---- Table 2's raw material for an existing pair (x, q): four fp64 sums -----------------------------
template <typename T, int V>
__global__ void __launch_bounds__(kThreads) distortion_kernel(const T* __restrict__ x, const T* __restrict__ q,
                                                              int64_t E, double* __restrict__ sums) {
    after_the_kernel_ahead();
    DistAcc acc;
    acc.reset();
    const int64_t nunits = E / V;
    const int64_t stride = (int64_t)gridDim.x * kThreads * 2;
    for (int64_t u0 = (int64_t)blockIdx.x * kThreads * 2; u0 < nunits; u0 += stride) {
        int64_t e[2];
        Pack<T> px[2], pq[2];
        float sx[2], sq[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            e[j] = (u0 + j * kThreads + threadIdx.x) * V;
            if (e[j] < E) {
                if constexpr (V == 1) {
                    sx[j] = load_scalar(x + e[j]);
                    sq[j] = load_scalar(q + e[j]);
                } else {
                    px[j].raw = ld_stream_16(x + e[j]);
                    pq[j].raw = ld_stream_16(q + e[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (e[j] >= E) continue;
            if constexpr (V == 1) acc.add_one(sx[j], sq[j]);
            else acc.add(px[j], pq[j]);
        }
    }
    acc.flush(sums);
}

// ---- Eq. 6 from the packed integer codes: y = s * (code - z) --------------------------------------
// Eight codes (BITS bytes of the bit string) per thread and step, two such strings in flight: two or three words of
// codes, one pair of divisions for the channel, shifts that are constants, and 32 bytes of fp32 (16 of bf16) stored at
// once.  Planes of at least 8 elements; where they are no multiple of 8 (RAGGED) a string may reach into the next
// plane.  `tail` codes behind the last whole string, all of the last plane, are the first threads' of the last block.
// Bound by the stores: [128,144,56,56], 231 MB written from 36 MB of 5-bit codes, 92 -> 45 us
// (5.9 TB/s; a thread per 16 bytes with two 32-bit divisions took 171 instructions for 4 elements).  A block per 512
// strings rather than a persistent grid, so that the stores go out in the order of memory: [128,96,112,112] 133 -> 110 us.
// END: there is such a tail (in a form of its own: bf16 [26,920,45,44], 6 bits, 31.1 without, 31.8 with the test for it).
template <typename T, int BITS, bool RAGGED, bool END>
__global__ void __launch_bounds__(kThreads) dequant_strings_kernel(const uint32_t* __restrict__ pcodes, T* __restrict__ y,
                                                                   uint32_t nstrings, uint32_t tail, uint32_t last_word, uint32_t inner,
                                                                   FastDiv div_inner, FastDiv div_C,
                                                                   const float* __restrict__ s, const float* __restrict__ z) {
    after_the_kernel_ahead();
    constexpr uint32_t kField = (1u << BITS) - 1u;
    constexpr int kFly = 2;
    if (END && blockIdx.x == gridDim.x - 1 && threadIdx.x < tail) {
        const uint64_t bit = ((uint64_t)nstrings * 8 + threadIdx.x) * BITS;
        const uint32_t w0 = (uint32_t)(bit >> 5), c = __funnelshift_r(__ldg(pcodes + w0), __ldg(pcodes + min(w0 + 1, last_word)), (uint32_t)bit & 31);
        store_scalar(y + (size_t)nstrings * 8 + threadIdx.x, __fmul_rn(__ldg(s + div_C.d - 1), __fsub_rn((float)(c & kField), __ldg(z + div_C.d - 1))));
    }
    const uint32_t t0 = blockIdx.x * (kThreads * kFly) + threadIdx.x;
    uint32_t w[kFly][3];
#pragma unroll
    for (int f = 0; f < kFly; ++f) {
        const uint32_t t = t0 + f * kThreads;
        if (t >= nstrings) break;
        const uint32_t w0 = (uint32_t)(((uint64_t)t * BITS) >> 2);              // 8 * BITS bits per string
        w[f][0] = __ldg(pcodes + w0);
        if constexpr (BITS > 1) w[f][1] = __ldg(pcodes + min(w0 + 1, last_word));
        if constexpr (BITS == 6 || BITS == 7) w[f][2] = __ldg(pcodes + min(w0 + 2, last_word));
    }
#pragma unroll
    for (int f = 0; f < kFly; ++f) {
        const uint32_t t = t0 + f * kThreads;
        if (t >= nstrings) break;
        const uint32_t sh = (t * (8u * BITS)) & 31u;                            // 0, 8, 16 or 24
        uint32_t lo, hi = 0;
        if constexpr (BITS == 1) lo = w[f][0] >> sh;
        else lo = __funnelshift_r(w[f][0], w[f][1], sh);
        if constexpr (BITS == 8) hi = w[f][1];
        else if constexpr (BITS == 6 || BITS == 7) hi = __funnelshift_r(w[f][1], w[f][2], sh);
        else if constexpr (BITS == 5) hi = w[f][1] >> sh;
        uint32_t plane, rem, q, g1;
        div_inner.divmod(t * 8u, plane, rem);
        div_C.divmod(plane, q, g1);
        const float s1 = __ldg(s + g1), z1 = __ldg(z + g1);
        float s2 = s1, z2 = z1;
        const uint32_t n1 = inner - rem;                                        // elements left in this plane
        if constexpr (RAGGED) {
            if (n1 < 8) {
                const uint32_t g2 = g1 + 1 == div_C.d ? 0u : g1 + 1;
                s2 = __ldg(s + g2);
                z2 = __ldg(z + g2);
            }
        }
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            constexpr uint32_t kTwo23 = 0x4B000000u;                            // 2^23: the code becomes the low mantissa
            const int pos = i * BITS;
            uint32_t c;
            if (pos + BITS <= 32) c = lo >> pos;
            else if (pos >= 32) c = hi >> (pos - 32);
            else c = __funnelshift_r(lo, hi, pos);
            const float code = __fsub_rn(__uint_as_float((c & kField) | kTwo23), 8388608.0f);
            const bool first = !RAGGED || (uint32_t)i < n1;
            v[i] = __fmul_rn(first ? s1 : s2, __fsub_rn(code, first ? z1 : z2));
        }
        T* out = y + (size_t)t * 8;
        if constexpr (Pack<T>::V == 8) {
            Pack<T> p;
            p.set_all(v);
            st_stream_16(out, p.raw);
        } else {
            asm volatile("st.global.L1::no_allocate.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(out), "f"(v[0]), "f"(v[1]),
                         "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                         : "memory");
        }
    }
}

// Any geometry: V = elements per thread and step (a 16-byte pack of y when E and the pointer allow it, else 1).
template <typename T, int V>
__global__ void __launch_bounds__(kThreads) dequant_packed_kernel(const uint32_t* __restrict__ pcodes,
                                                                  T* __restrict__ y, int64_t E, int64_t inner,
                                                                  int64_t C, int bits,
                                                                  const float* __restrict__ s,
                                                                  const float* __restrict__ z) {
    after_the_kernel_ahead();
    const int64_t nunits = E / V;
    const uint32_t field = (1u << bits) - 1u;
    for (int64_t u = (int64_t)blockIdx.x * kThreads + threadIdx.x; u < nunits; u += (int64_t)gridDim.x * kThreads) {
        const int64_t e = u * V;
        int64_t rem, grp;
        if (E < (1ll << 31)) {                       // 32-bit divisions are several times cheaper
            const uint32_t plane = (uint32_t)e / (uint32_t)inner;
            rem = (uint32_t)e - plane * (uint32_t)inner;
            grp = plane % (uint32_t)C;
        } else {
            const int64_t plane = e / inner;
            rem = e - plane * inner;
            grp = plane % C;
        }
        float sg = __ldg(s + grp), zg = __ldg(z + grp);
        Pack<T> out;
        // the thread's V * b <= 64 bits lie in at most three consecutive words
        const int64_t first_bit = e * bits, last_word = (E * bits - 1) >> 5;
        const uint32_t bit0 = (uint32_t)(first_bit & 31);
        const int64_t w0 = first_bit >> 5;
        const uint32_t q0 = __ldg(pcodes + w0);
        const uint32_t q1 = w0 + 1 <= last_word ? __ldg(pcodes + w0 + 1) : 0u;
        const uint32_t q2 = (V * 8 > 32 && w0 + 2 <= last_word) ? __ldg(pcodes + w0 + 2) : 0u;
        const uint64_t lo64 = ((uint64_t)q1 << 32) | q0, hi64 = ((uint64_t)q2 << 32) | q1;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const uint32_t pos = bit0 + (uint32_t)(i * bits);               // < 96
            const uint32_t v = pos < 32u ? (uint32_t)(lo64 >> pos) : (uint32_t)(hi64 >> (pos - 32u));
            const float yv = __fmul_rn(sg, __fsub_rn((float)(v & field), zg));
            if constexpr (V == 1) store_scalar(y + e, yv);
            else out.set(i, yv);
            if (V > 1 && ++rem == inner) {          // the next element starts the next plane
                rem = 0;
                grp = (grp + 1 == C) ? 0 : grp + 1;
                sg = __ldg(s + grp);
                zg = __ldg(z + grp);
            }
        }
        if constexpr (V > 1) st_stream_16(y + e, out.raw);
    }
}

bool aligned16(const void* p) { return p == nullptr || ((uintptr_t)p & 15) == 0; }

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

int flat_grid(const FlatGeom& f) {
    const int64_t cap = (int64_t)sm_count() * 8;
    return (int)(f.ntiles < cap ? f.ntiles : cap);
}

int range_rows_ctas() {
    return sm_count() * 4;
}

// With elements behind the last whole pack: where scalar loads are faster than packs.  In planes of a few packs every pack of the
// vector path straddles two planes, each lane of a warp with a group of its own, two updates a pack; scalars have one update an element,
// and wait for one another's atomics when a group's elements are many.  Scalar / packs, us: bf16 [301,33,3,3] 29 / 60, 1101 of them 58 / 61,
// 1684 86 / 61, [301,501,3,3] 38 / 62, [1746,509,3,3] 198 / 134; planes of 15 [451,33,3,5] 31 / 41, [701,33,3,5] 45 / 40, of 25 [301,33,5,5]
// 25 / 27, [451,33,5,5] 37 / 28, of 49 no more; fp32 [301,33,1,5] 39 / 52, [1101,33,1,5] 61 / 52, [451,33,3,3] 30 / 32, [701,33,3,3] 42 / 32, of 15
// 25 / 23. Of a few channels the lanes of a warp share groups again: bf16 [407,5,3,3] 27 / 16, [301,9,3,3] 29 / 25, [301,13,3,3] 29 / 33; fp32 29 /
// 17, 27 / 23, 27 / 29. Of a group per plane, whose atomics meet nobody: bf16 [1001,901,3,3] 82 / 137, fp32 83 / 117, planes of 25 125 / 134 and 126
// / 153, but 126 K groups fp32 of 15 to 25 as fast.  Of a few thousand elements in short planes [7,5,5,5] 5.2 / 9.5, [7,61,3,5] fp32 18 / 21.
template <typename T>
bool scalar_range(const Geom& g) {
    const int64_t channel = g.outer * g.inner * (int64_t)sizeof(T);      // its bytes
    const bool few = g.inner < (sizeof(T) == 4 ? 12 : 32);
    if (g.E < (g.C < 12 ? 4096 : 8192) && g.inner < 64) return true;
    if (g.outer == 1) return few || (g.inner < 32 && g.C > 200'000);
    return few && g.C >= 12 && channel <= 18'432 && channel * g.C <= 1 << 22;
}

template <typename T>
cudaError_t range_flat_t(const void* x, const Geom& g, uint32_t* kmin, uint32_t* kmax, const RangeEnd& end, int layout, cudaStream_t st) {
    FlatGeom f = make_flat(g);
    constexpr int VF = Pack<T>::V;
    bool vec = aligned16(x) && (g.inner % VF == 0);
    int grid = flat_grid(f);
    const bool rows_ok = aligned16(x) && g.inner >= VF && g.E < (1ll << 31) &&
                         g.C < (1ll << 30) && g.inner < (1ll << 30) && (g.E % VF == 0 || !scalar_range<T>(g));
    // columns: slabs of whole units, at least a batch of them to walk, planes shorter than a row of the vector path or
    // not whole units
    if (rows_ok && (g.C * g.inner) % VF == 0 && g.outer >= 8 && (!vec || g.inner / VF < 128)) {
        const uint32_t slab_units = (uint32_t)(g.C * g.inner / VF), ncol = (slab_units + kThreads - 1) / kThreads;
        const uint32_t cap = (uint32_t)range_rows_ctas(), outer = (uint32_t)g.outer;
        // chunks of slabs: enough blocks to fill the chip twice over, walks of at least 4 slabs
        const uint32_t chunks = std::max<uint32_t>(1, std::min<uint32_t>((2 * cap + ncol - 1) / ncol, outer / 4));
        constexpr int U = VF == 4 ? 8 : 4;
        auto cols = [&](auto kern, uint32_t plane) {
            return launch_after(layout, kern, ncol * chunks, kThreads, 0, st, (const uint4*)x, slab_units, outer, chunks,
                                make_fastdiv(ncol), make_fastdiv(plane), kmin, kmax, end);
        };
        return vec ? cols(range_cols_kernel<T, true, U>, (uint32_t)(g.inner / VF)) : cols(range_cols_kernel<T, false, U>, (uint32_t)g.inner);
    }
    if (rows_ok) {
        const uint32_t n_units = (uint32_t)(g.E / VF);
        int64_t rows = ((int64_t)n_units + 127) / 128, ctas = (rows + 2 * (kThreads / 32) - 1) / (2 * (kThreads / 32));
        const int64_t cap = (int64_t)range_rows_ctas();                 // 4 resident CTAs per SM at 64 registers
        int rgrid = (int)(ctas < cap ? ctas : cap);
        auto by_rows = [&](auto kern, uint32_t plane) {
            return launch_after(layout, kern, rgrid, kThreads, 0, st, (const uint4*)x, n_units, (uint32_t)(g.E % VF), (uint32_t)g.inner, make_fastdiv(plane),
                                make_fastdiv((uint32_t)g.C), (uint32_t)g.C, kmin, kmax, end);
        };
        return vec ? by_rows(range_rows_kernel<T, true>, (uint32_t)(g.inner / VF)) : by_rows(range_rows_kernel<T, false>, (uint32_t)g.inner);
    }
    return vec ? launch_after(layout, range_flat_kernel<T, VF>, grid, kThreads, 0, st, (const T*)x, f, kmin, kmax, end)
               : launch_after(layout, range_flat_kernel<T, 1>, grid, kThreads, 0, st, (const T*)x, f, kmin, kmax, end);
}

template <typename T, int MODE>
cudaError_t quant_flat_t(const QuantIO& io, const Geom& g, int bits, const float* lo, const float* hi,
                         cudaStream_t st) {
    FlatGeom f = make_flat(g);
    constexpr int VF = Pack<T>::V;
    bool vec = (g.inner % VF == 0) && aligned16(io.x) && aligned16(io.gy) && aligned16(io.y) && aligned16(io.gx) &&
               ((uintptr_t)io.codes % 4 == 0) && ((uintptr_t)io.mask % 4 == 0);
    // A block per tile: blocks are then started in the order of memory, while the blocks of a persistent grid drift apart and
    // DRAM sees more open pages (two reads and two writes of 617 MB: 5.9 to 6.3 TB/s persistent, 6.9 in order).  Given range,
    // us: forward [128,96,112,112] 207 -> 182, [256,512,28,28] 138 -> 121, bf16 97 -> 90; backward from x, channels-last
    // bf16 [40,100,100,200] 348 -> 281.  With the distortion sums a few tiles each, as every block ends in atomics on one
    // sector, and so the scalar form below four rounds of blocks ([32,56,56,256] channels-last 115 / 119).
    const int few = flat_grid(f);
    const unsigned grid = io.dist || (!vec && f.ntiles < 4 * (int64_t)few) ? (unsigned)few : (unsigned)f.ntiles;
    float qmax = (float)((1 << bits) - 1);
    const bool extras = io.codes != nullptr || io.mask != nullptr || io.pmask != nullptr || io.dist != nullptr ||
                        io.pcodes != nullptr;
    // forward with y and the packed mask as the only outputs: a leaner instantiation
    const bool pmask_only = io.pmask != nullptr && io.y != nullptr && io.codes == nullptr && io.mask == nullptr &&
                            io.dist == nullptr && io.pcodes == nullptr;
    const bool dist_only = io.dist != nullptr && io.y != nullptr && io.codes == nullptr && io.mask == nullptr &&
                           io.pmask == nullptr && io.pcodes == nullptr;
    const bool pack_only = io.pcodes != nullptr && io.y == nullptr && io.codes == nullptr && io.mask == nullptr &&
                           io.pmask == nullptr && io.dist == nullptr;
    // planes that are not whole packs, everything else in place for 16-byte accesses: the vector kernel with
    // packs that may straddle two planes
    const bool planes = !vec && g.inner >= VF && g.inner % VF != 0 && !f.inner_big && aligned16(io.x) &&
                        aligned16(io.gy) && aligned16(io.y) && aligned16(io.gx) && ((uintptr_t)io.codes % 4 == 0) &&
                        ((uintptr_t)io.mask % 4 == 0);
    // ... and of those, where the last pack is not whole either: all outputs but codes and masks by the byte
    const bool ragged = planes && g.E % VF == 0, end = planes && g.E % VF != 0 && (!extras || pmask_only || pack_only || dist_only);
    // Five blocks of a table each fill an SM.  The scalar form is bound by its instructions, and its grids of up to a wave are spread evenly
    // only over an empty GPU: blocks that start before the kernel ahead has ended crowd on the SMs that have room first, unless two grids
    // leave SMs free.  Alone / set up early, us, by blocks: backward (seven to an SM) channels-last [60,30,30,75], 494, 22.7 / 28.3, bf16
    // 24.8 / 31.8, [120,30,30,35], 461, 22.7 / 28.3, but [4001,201,1,3], 295, 16.7 / 15.3, [64,14,14,51], 79, 12.8 / 11.8; behind the range of the
    // same call (four to an SM), whose last block ends late, both directions [4001,201,1,3] 381 / 387, bf16 [9001,50,2,2], 220, 377 / 382, codes
    // [1916,672,2,1], 314, 222 / 227; forward with a given range 16.2 / 13.8 at 79 blocks, 24.8 / 23.4 at 494.
    const int64_t sms = sm_count();
    const bool scalar = !vec && !ragged && !end;
    const bool crowded = scalar && (io.behind_range ? 2 * f.ntiles > sms && f.ntiles <= 4 * sms
                                                    : MODE == MODE_BWD && f.ntiles > 3 * sms && f.ntiles <= 7 * sms);
    const int layout = crowded ? kAlone : sm_layout(100, (uint64_t)g.E * sizeof(T));
    auto go = [&](auto kern) {
        return launch_after(layout, kern, grid, kThreads, 0, st, (const T*)io.x, (const T*)io.gy, (T*)io.y, (T*)io.gx, io.codes, io.mask,
                            io.pmask, io.dist, io.pcodes, io.code_bits, f, qmax, lo, hi);
    };
    if constexpr (MODE == MODE_FWD) {
        // columns: slabs of whole units (with a mask whole bytes of it, and whole words in all), at least a batch of them: faster for
        // all planes, see the kernel
        const bool plain = !io.codes && !io.mask && !io.dist && !io.pcodes && io.y;
        ColsCut cut{};
        if (plain && (vec || ragged) && cut_cols(VF == 4 ? 0 : 1, g, io.pmask != nullptr, (int)sms, cut)) {
            auto cols = [&](auto kern, uint32_t plane) {
                return launch_after(sm_layout(0, (uint64_t)g.E * sizeof(T)), kern, cut.ncol * ((cut.rows + cut.walk - 1) / cut.walk), kThreads, 0, st,
                                    (const uint4*)io.x, (uint4*)io.y, (uint8_t*)io.pmask, cut, make_fastdiv(cut.ncol), make_fastdiv(plane),
                                    make_fastdiv((uint32_t)g.C), qmax, lo, hi);
            };
            const uint32_t plane = (uint32_t)(vec ? g.inner / VF : g.inner);
            if (io.pmask) return vec ? cols(quant_cols_kernel<T, true, true>, plane) : cols(quant_cols_kernel<T, false, true>, plane);
            return vec ? cols(quant_cols_kernel<T, true, false>, plane) : cols(quant_cols_kernel<T, false, false>, plane);
        }
        if ((vec || ragged) && pack_only && g.E % 32 == 0)         // whole words of codes: the byte-wise writer
            return vec ? go(quant_flat_kernel<T, VF, MODE, 3, true>) : go(quant_flat_kernel<T, VF, MODE, 3, true, true>);
        if ((vec || ragged) && pack_only)
            return vec ? go(quant_flat_kernel<T, VF, MODE, 1, true>) : go(quant_flat_kernel<T, VF, MODE, 1, true, true>);
        if ((vec || ragged) && dist_only)
            return vec ? go(quant_flat_kernel<T, VF, MODE, 4>) : go(quant_flat_kernel<T, VF, MODE, 4, false, true>);
        if ((vec || ragged) && pmask_only)
            return vec ? go(quant_flat_kernel<T, VF, MODE, 2>) : go(quant_flat_kernel<T, VF, MODE, 2, false, true>);
    }
    if (end) {
        if constexpr (MODE == MODE_FWD) {
            if (pack_only) return go(quant_flat_kernel<T, VF, MODE, 1, true, true, true>);
            if (dist_only) return go(quant_flat_kernel<T, VF, MODE, 4, false, true, true>);
            if (pmask_only) return go(quant_flat_kernel<T, VF, MODE, 2, false, true, true>);
        }
        return go(quant_flat_kernel<T, VF, MODE, 0, false, true, true>);
    }
    if (ragged) return extras ? go(quant_flat_kernel<T, VF, MODE, 1, false, true>) : go(quant_flat_kernel<T, VF, MODE, 0, false, true>);
    if (vec) return extras ? go(quant_flat_kernel<T, VF, MODE, 1>) : go(quant_flat_kernel<T, VF, MODE, 0>);
    return go(quant_flat_kernel<T, 1, MODE, 1>);
}

template <typename T, int MODE>
cudaError_t naive_t(const QuantIO& io, const Geom& g, int bits, uint32_t* kmin, uint32_t* kmax, float* lo,
                    float* hi, cudaStream_t st, int* launches) {
    int grid = (int)(g.outer < 1024 ? g.outer : 1024);
    float qmax = (float)((1 << bits) - 1);
    int n = 0;
    for (int64_t c = 0; c < g.C; ++c) {
        naive_extreme_kernel<T, false><<<grid, kThreads, 0, st>>>((const T*)io.x, g, c, kmin + c);
        naive_extreme_kernel<T, true><<<grid, kThreads, 0, st>>>((const T*)io.x, g, c, kmax + c);
        naive_quant_kernel<T, MODE><<<grid, kThreads, 0, st>>>((const T*)io.x, (const T*)io.gy, (T*)io.y,
                                                               (T*)io.gx, io.codes, io.mask, g, c, qmax, kmin,
                                                               kmax, lo, hi);
        n += 3;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (launches) *launches = n;
    return cudaSuccess;
}

template <typename T, int BITS>
cudaError_t dequant_strings_bits(const uint32_t* pcodes, T* y, const Geom& g, const float* s, const float* z,
                                 cudaStream_t st) {
    const uint32_t n = (uint32_t)(g.E / 8), last = (uint32_t)((g.E * BITS - 1) >> 5);
    const uint32_t per_cta = kThreads * 2, grid = (n + per_cta - 1) / per_cta;
    const FastDiv di = make_fastdiv((uint32_t)g.inner), dc = make_fastdiv((uint32_t)g.C);
    auto go = [&](auto kern) {
        return launch_after(sm_layout(0, (uint64_t)g.E * sizeof(T)), kern, grid, kThreads, 0, st, pcodes, y, n, (uint32_t)(g.E % 8), last, (uint32_t)g.inner,
                            di, dc, s, z);
    };
    if (g.inner % 8 == 0) return go(dequant_strings_kernel<T, BITS, false, false>);
    return g.E % 8 == 0 ? go(dequant_strings_kernel<T, BITS, true, false>) : go(dequant_strings_kernel<T, BITS, true, true>);
}

template <typename T>
cudaError_t dequant_strings(const uint32_t* pcodes, T* y, const Geom& g, int bits, const float* s, const float* z, cudaStream_t st) {
    switch (bits) {
        case 1: return dequant_strings_bits<T, 1>(pcodes, y, g, s, z, st);
        case 2: return dequant_strings_bits<T, 2>(pcodes, y, g, s, z, st);
        case 3: return dequant_strings_bits<T, 3>(pcodes, y, g, s, z, st);
        case 4: return dequant_strings_bits<T, 4>(pcodes, y, g, s, z, st);
        case 5: return dequant_strings_bits<T, 5>(pcodes, y, g, s, z, st);
        case 6: return dequant_strings_bits<T, 6>(pcodes, y, g, s, z, st);
        case 7: return dequant_strings_bits<T, 7>(pcodes, y, g, s, z, st);
        default: return dequant_strings_bits<T, 8>(pcodes, y, g, s, z, st);
    }
}

}  // namespace

cudaError_t launch_range(const void* x, int dtype, const Geom& g, uint32_t* kmin, uint32_t* kmax, uint32_t* counter,
                         float* lo, float* hi, int bits, float* s_opt, float* z_opt, bool behind_clear, cudaStream_t st) {
    const bool fused = counter != nullptr && g.C <= 4096;       // the last block's share: 16 groups per thread
    const RangeEnd end{fused ? counter : nullptr, kmin, kmax, lo, hi, s_opt, z_opt, (uint32_t)g.C, bits};
    const int layout = behind_clear ? kAnyLayout : kAlone;
    const cudaError_t e = dtype == 0 ? range_flat_t<float>(x, g, kmin, kmax, end, layout, st)
                                     : range_flat_t<__nv_bfloat16>(x, g, kmin, kmax, end, layout, st);
    if (e != cudaSuccess || fused) return e;
    const int grid = (int)((g.C + 255) / 256);
    return launch_after(kAnyLayout, finalize_range_kernel, grid, 256, 0, st, kmin, kmax, g.C, lo, hi, bits, s_opt, z_opt);
}

cudaError_t launch_clear(void* workspace, size_t bytes, double* sums_opt, cudaStream_t st) {
    const size_t words = bytes / 4, blocks = (words + 4 * kThreads - 1) / (4 * kThreads);
    return launch_after(kAnyLayout, clear_kernel, (unsigned)std::max<size_t>(1, std::min<size_t>(blocks, 256)), kThreads, 0, st,
                        (uint32_t*)workspace, (uint32_t)words, sums_opt);
}

cudaError_t launch_params(const float* lo, const float* hi, int64_t G, int bits, float* s_opt, float* z_opt,
                          cudaStream_t st) {
    int grid = (int)((G + 255) / 256);
    return launch_after(kAnyLayout, params_kernel, grid, 256, 0, st, lo, hi, G, bits, s_opt, z_opt);
}

cudaError_t launch_quant_flat(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, const float* lo,
                              const float* hi, cudaStream_t st) {
    if (dtype == 0) {
        if (mode == MODE_FWD) return quant_flat_t<float, MODE_FWD>(io, g, bits, lo, hi, st);
        if (mode == MODE_BWD) return quant_flat_t<float, MODE_BWD>(io, g, bits, lo, hi, st);
        return quant_flat_t<float, MODE_BOTH>(io, g, bits, lo, hi, st);
    }
    if (mode == MODE_FWD) return quant_flat_t<__nv_bfloat16, MODE_FWD>(io, g, bits, lo, hi, st);
    if (mode == MODE_BWD) return quant_flat_t<__nv_bfloat16, MODE_BWD>(io, g, bits, lo, hi, st);
    return quant_flat_t<__nv_bfloat16, MODE_BOTH>(io, g, bits, lo, hi, st);
}

cudaError_t launch_naive(const QuantIO& io, int mode, int dtype, const Geom& g, int bits, uint32_t* kmin,
                         uint32_t* kmax, float* lo, float* hi, cudaStream_t st, int* launches) {
    if (dtype == 0) {
        if (mode == MODE_FWD) return naive_t<float, MODE_FWD>(io, g, bits, kmin, kmax, lo, hi, st, launches);
        return naive_t<float, MODE_BOTH>(io, g, bits, kmin, kmax, lo, hi, st, launches);
    }
    if (mode == MODE_FWD) return naive_t<__nv_bfloat16, MODE_FWD>(io, g, bits, kmin, kmax, lo, hi, st, launches);
    return naive_t<__nv_bfloat16, MODE_BOTH>(io, g, bits, kmin, kmax, lo, hi, st, launches);
}

// Of a forward with a given range by columns (quant_cols_kernel).  A row is as many slabs side by side as fill the blocks across it to
// 15/16, of 8192 units at most: with a slab to a row the lanes beyond a slab of 64 units were three of four ([65536,4,4,4] fp32
// 22.3, by tiles 8.8, slabs side by side 7.2 us; bf16 34.7, 7.6, 7.0).  Four to sixteen rows to a block, so that blocks start in the order of
// memory: as many as leave a small tensor one wave of blocks, and a larger one whole waves (bf16 [1178,11,40,40], a wave and an
// eighth of 16 rows 22.2, by tiles 20.3, two waves of 9 19.2 us).
bool cut_cols(int dtype, const Geom& g, bool packed_mask, int sms, ColsCut& cut) {
    const int64_t V = dtype == 0 ? 4 : 8, slab = g.C * g.inner;
    if (g.outer < 8 || g.inner < V || slab % V != 0 || g.E >= (1ll << 31) || g.C >= (1ll << 30)) return false;
    if (packed_mask && (slab % 8 != 0 || g.E % 32 != 0)) return false;
    const uint32_t units = (uint32_t)(slab / V), outer = (uint32_t)g.outer;
    auto lanes = [&](uint32_t side) { return ((uint64_t)side * units + kThreads - 1) / kThreads * kThreads; };
    cut.side = 1;
    for (uint32_t side = 1; side <= outer && (side == 1 || (uint64_t)side * units <= 8192); ++side) {
        if (lanes(side) * cut.side < lanes(cut.side) * side) cut.side = side;
        if (15 * lanes(side) <= 16ull * side * units) break;
    }
    cut.row_units = cut.side * units;
    cut.ncol = (cut.row_units + kThreads - 1) / kThreads;
    cut.rows = (outer + cut.side - 1) / cut.side;
    cut.last_units = (outer - (cut.rows - 1) * cut.side) * units;
    const uint64_t slots = (uint64_t)sms * 4, each = ((uint64_t)cut.rows * cut.ncol + slots - 1) / slots, waves = (each + 15) / 16;
    cut.walk = (uint32_t)std::max<uint64_t>(4, (each + waves - 1) / waves);
    return true;
}

// With elements behind the last whole pack, scalar loads up to here: a small call ends sooner with more blocks of less each.
// Scalar / packs, us from a graph: [3,31,25,25] 1.0 / 1.35; fp32 [9,301,15,15], 0.6 M, 1.5 / 1.7, [21,251,15,15], 1.2 M, 1.94 / 2.02,
// [33,301,15,15], 2.2 M, 3.45 / 3.25; bf16 1.5 / 1.4, 1.9 / 1.6, 2.9 / 2.0.
constexpr int64_t kTailElements[2] = {1'500'000, 500'000};

cudaError_t launch_bwd_packmask(const void* gy, const uint32_t* pmask, void* gx, int dtype, int64_t E,
                                cudaStream_t st) {
    const int VF = dtype == 0 ? 4 : 8;
    const bool tail = E % VF != 0, vec = aligned16(gy) && aligned16(gx) && (!tail || E >= kTailElements[dtype == 0 ? 0 : 1]);
    const int64_t units = vec ? E / VF : E;
    const int64_t per_cta = (int64_t)kThreads * kUnroll;
    const unsigned grid = (unsigned)((units + per_cta - 1) / per_cta);
    auto go = [&](auto kern, auto zero) {
        using T = decltype(zero);
        return launch_after(sm_layout(0, (uint64_t)E * sizeof(T)), kern, grid, kThreads, 0, st, (const T*)gy, pmask, (T*)gx, E);
    };
    auto by_type = [&](auto zero) {
        using T = decltype(zero);
        if (!vec) return go(bwd_packmask_kernel<T, 1, false>, zero);
        return tail ? go(bwd_packmask_kernel<T, Pack<T>::V, true>, zero) : go(bwd_packmask_kernel<T, Pack<T>::V, false>, zero);
    };
    return dtype == 0 ? by_type(0.0f) : by_type(__nv_bfloat16{});
}

cudaError_t launch_distortion(const void* x, const void* q, int dtype, int64_t E, double* sums, cudaStream_t st) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int VF = dtype == 0 ? 4 : 8;
    const bool vec = aligned16(x) && aligned16(q) && (E % VF == 0);
    const int64_t units = vec ? E / VF : E;
    const int64_t per_cta = (int64_t)kThreads * 2;
    const int64_t ctas = (units + per_cta - 1) / per_cta, cap = (int64_t)sms * 8;
    const int grid = (int)(ctas < 1 ? 1 : (ctas < cap ? ctas : cap));
    auto go = [&](auto kern, auto zero) {
        using T = decltype(zero);
        return launch_after(sm_layout(16, (uint64_t)E * sizeof(T)), kern, grid, kThreads, 0, st, (const T*)x, (const T*)q, E, sums);
    };
    if (dtype == 0) return vec ? go(distortion_kernel<float, 4>, 0.0f) : go(distortion_kernel<float, 1>, 0.0f);
    const __nv_bfloat16 zero{};
    return vec ? go(distortion_kernel<__nv_bfloat16, 8>, zero) : go(distortion_kernel<__nv_bfloat16, 1>, zero);
}

cudaError_t launch_dequant_packed(const uint32_t* pcodes, void* y, int dtype, const Geom& g, int bits,
                                  const float* s, const float* z, cudaStream_t st) {
    // strings of 8 codes: planes of at least 8 elements, 32-byte (fp32) stores; with codes behind the last whole string from 64 K on, fp32
    // 128 K (one by one / strings, us from a graph: [7,373,4,5], 52 K, bf16 1.5 / 1.6, fp32 1.5 / 1.7, [165,52,3,3], 77 K, 1.75 / 1.5, a group per
    // plane fp32 1.5 / 1.75)
    if ((g.E % 8 == 0 || g.E >= (dtype == 0 ? 1 << 17 : 1 << 16)) && g.E < (1ll << 31) && g.inner >= 8 && g.inner < (1ll << 30) && g.C < (1ll << 30) &&
        ((uintptr_t)y & (dtype == 0 ? 31 : 15)) == 0)
        return dtype == 0 ? dequant_strings<float>(pcodes, (float*)y, g, bits, s, z, st)
                          : dequant_strings<__nv_bfloat16>(pcodes, (__nv_bfloat16*)y, g, bits, s, z, st);
    const int VF = dtype == 0 ? 4 : 8;
    const bool vec = aligned16(y) && (g.E % VF == 0);
    const int64_t units = vec ? g.E / VF : g.E;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ctas = (units + kThreads - 1) / kThreads, cap = (int64_t)sms * 16;
    const int grid = (int)(ctas < 1 ? 1 : (ctas < cap ? ctas : cap));
    auto go = [&](auto kern, auto zero) {
        using T = decltype(zero);
        return launch_after(sm_layout(0, (uint64_t)g.E * sizeof(T)), kern, grid, kThreads, 0, st, pcodes, (T*)y, g.E, g.inner, g.C, bits, s, z);
    };
    if (dtype == 0) return vec ? go(dequant_packed_kernel<float, 4>, 0.0f) : go(dequant_packed_kernel<float, 1>, 0.0f);
    const __nv_bfloat16 zero{};
    return vec ? go(dequant_packed_kernel<__nv_bfloat16, 8>, zero) : go(dequant_packed_kernel<__nv_bfloat16, 1>, zero);
}

}  // namespace granq
