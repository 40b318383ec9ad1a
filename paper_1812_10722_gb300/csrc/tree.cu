// Treecode structures (Sec. II.D): the octree over the Gauss-node sources with at
// most N_crit sources per leaf, and per block of 64 collocation targets the list of
// boxes accepted by the multipole-acceptance criterion r_b < theta * r (Taylor
// expansion, M2P) and of leaves summed directly (P2P).
//
// Device pipeline: bounding cube -> 30-bit Morton keys (10 bits per axis) ->
// LSD radix sort (8-bit digits, stable) of sources and targets -> permuted
// work-order arrays -> octree, level by level in one CTA (deterministic box
// numbering) -> box centres (centre of the sources' bounding box) and radii
// r_b = max |y - c| -> target-block bounding boxes -> interaction lists (count,
// scan, fill; one thread per target block walks the tree depth first).
#include <algorithm>
#include <cstdlib>
#include <cmath>

#include "lspr_internal.cuh"
#include "tc_lists.h"

namespace lspr {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kDigitBits = 8;
constexpr int kDigits = 1 << kDigitBits;
constexpr int kSortWarps = kSortThreads / 32;
static_assert(kDigits == kSortThreads, "one thread per digit");
constexpr int kP2PChunk = 256;      // sources per P2P work item (upper bound)
constexpr int kM2PSeg = 16;         // boxes per M2P work item
constexpr int kP2MChunk = 512;      // sources per P2M work item
constexpr int kStack = 96;
constexpr int kGeomThreads = 256;

// ------------------------------------------------------------ bounding cube
// two stages: kBoxBlocks blocks reduce slices of the points into part[block][6], then one
// block reduces the partials into out = (lo[3], hi[3])
__global__ void bbox_partial_kernel(const dbl4 *__restrict__ a, int64_t na, const dbl4 *__restrict__ b, int64_t nb,
                                    double *part) {
    __shared__ double red[6][256];
    const int t = threadIdx.x;
    double l[3] = {1e300, 1e300, 1e300}, h[3] = {-1e300, -1e300, -1e300};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + t; i < na + nb; i += (int64_t)gridDim.x * blockDim.x) {
        const dbl4 p = i < na ? a[i] : b[i - na];
        l[0] = fmin(l[0], p.x); l[1] = fmin(l[1], p.y); l[2] = fmin(l[2], p.z);
        h[0] = fmax(h[0], p.x); h[1] = fmax(h[1], p.y); h[2] = fmax(h[2], p.z);
    }
    for (int d = 0; d < 3; ++d) { red[d][t] = l[d]; red[3 + d][t] = h[d]; }
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (t < s)
            for (int d = 0; d < 3; ++d) {
                red[d][t] = fmin(red[d][t], red[d][t + s]);
                red[3 + d][t] = fmax(red[3 + d][t], red[3 + d][t + s]);
            }
        __syncthreads();
    }
    if (t == 0)
        for (int q = 0; q < 6; ++q) part[blockIdx.x * 6 + q] = red[q][0];
}

// one warp per component
__global__ void bbox_final_kernel(const double *part, int nparts, double *out) {
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = q < 3 ? 1e300 : -1e300;
    for (int k = lane; k < nparts; k += 32) v = q < 3 ? fmin(v, part[k * 6 + q]) : fmax(v, part[k * 6 + q]);
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_xor_sync(0xffffffffu, v, o);
        v = q < 3 ? fmin(v, w) : fmax(v, w);
    }
    if (lane == 0) out[q] = v;
}

int launch_bbox(lspr_ctx *ctx, const dbl4 *a, int64_t na, const dbl4 *b, int64_t nb, double *part, double *out) {
    ctx->n_launches += 2;
    bbox_partial_kernel<<<kBoxBlocks, 256, 0, ctx->stream>>>(a, na, b, nb, part);
    bbox_final_kernel<<<1, 6 * 32, 0, ctx->stream>>>(part, kBoxBlocks, out);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// key bit 3l+2 / 3l+1 / 3l = x / y / z bit l, so the top triple selects the octant
__global__ void morton_kernel(const dbl4 *__restrict__ p, int64_t n, const double *cube /* lo[3], size */,
                              unsigned *keys, int *vals) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const dbl4 q = p[i];
    const double inv = 1024.0 / cube[3];
    unsigned ix = (unsigned)min(1023.0, fmax(0.0, floor((q.x - cube[0]) * inv)));
    unsigned iy = (unsigned)min(1023.0, fmax(0.0, floor((q.y - cube[1]) * inv)));
    unsigned iz = (unsigned)min(1023.0, fmax(0.0, floor((q.z - cube[2]) * inv)));
    keys[i] = (spread10(ix) << 2) | (spread10(iy) << 1) | spread10(iz);
    vals[i] = (int)i;
}

// ----------------------------------------------------------------- radix sort
// Stable LSD sort by 8-bit digits (four passes for the 30-bit keys): tile histograms, one scan
// block per digit over the tiles, and a scatter whose warps rank equal digits with match.any in key
// order.  Latency-bound (a pass moves 5 MB): halving the passes and launches of the 4-bit form took
// the sorts of a new geometry (81920, 81920 and 327680 pairs) from 495 to 241 us.
__global__ void __launch_bounds__(kSortThreads) radix_hist_kernel(const unsigned *__restrict__ keys, int64_t n,
                                                                  int shift, int nblocks, int *hist) {
    __shared__ int cnt[kDigits];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int64_t i = base + k * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & (kDigits - 1)], 1);
    }
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = cnt[threadIdx.x];
}

__device__ __forceinline__ int warp_inclusive(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int w = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w;
    }
    return v;
}

// exclusive scan of each digit's tile counts in place, and the digit's total
__global__ void radix_scan_kernel(int *hist, int nblocks, int *total) {
    const int lane = threadIdx.x & 31, d = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int *h = hist + (int64_t)d * nblocks;
    int run = 0;
    for (int base = 0; base < nblocks; base += 32) {
        const int i = base + lane;
        const int v = i < nblocks ? h[i] : 0;
        const int inc = warp_inclusive(v, lane);
        if (i < nblocks) h[i] = run + inc - v;
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) total[d] = run;
}

// exclusive scan over a block of kDigits threads
__device__ __forceinline__ int block_exclusive(int v, int *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int inc = warp_inclusive(v, lane);
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    int add = 0;
    for (int w = 0; w < warp; ++w) add += sh[w];
    return add + inc - v;
}

__global__ void __launch_bounds__(kSortThreads) radix_scatter_kernel(const unsigned *__restrict__ kin,
                                                                     const int *__restrict__ vin, int64_t n, int shift,
                                                                     int nblocks, const int *__restrict__ offs,
                                                                     const int *__restrict__ total, unsigned *kout,
                                                                     int *vout) {
    __shared__ int cnt[kSortWarps][kDigits];   // a warp's count per digit, then its first position
    __shared__ int sh[kSortWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int w = 0; w < kSortWarps; ++w) cnt[w][t] = 0;
    __syncthreads();
    // a warp takes 32 kSortItems consecutive keys, 32 at a time
    const int64_t base = (int64_t)blockIdx.x * kSortTile + warp * (32 * kSortItems) + lane;
    unsigned k[kSortItems];
    int rank[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int64_t i = base + 32 * j;
        const bool live = i < n;
        k[j] = live ? kin[i] : 0u;
        const int d = (k[j] >> shift) & (kDigits - 1);
        const unsigned same = __match_any_sync(0xffffffffu, live ? d : kDigits);
        const int before = __popc(same & ((1u << lane) - 1u));
        int c = 0;
        if (live) c = cnt[warp][d];
        __syncwarp();
        if (live && before == 0) cnt[warp][d] = c + __popc(same);
        __syncwarp();
        rank[j] = c + before;
    }
    __syncthreads();
    // first output position of every (digit, warp)
    const int first = block_exclusive(total[t], sh) + offs[t * nblocks + blockIdx.x];
    int run = first;
    for (int w = 0; w < kSortWarps; ++w) {
        const int c = cnt[w][t];
        cnt[w][t] = run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int64_t i = base + 32 * j;
        if (i >= n) continue;
        const int pos = cnt[warp][(k[j] >> shift) & (kDigits - 1)] + rank[j];
        kout[pos] = k[j];
        vout[pos] = vin[i];
    }
}

// sorts (keys, vals) of length n in place using the given scratch
int64_t radix_sort_scratch_ints(int64_t n) { return kDigits * ((n + kSortTile - 1) / kSortTile); }

int radix_sort(lspr_ctx *ctx, unsigned *keys, int *vals, unsigned *ktmp, int *vtmp, int64_t n, int bits,
                      int *hist, int *total) {
    const int nblocks = (int)((n + kSortTile - 1) / kSortTile);
    cudaStream_t st = ctx->stream;
    unsigned *ka = keys, *kb = ktmp;
    int *va = vals, *vb = vtmp;
    const int passes = (bits + kDigitBits - 1) / kDigitBits;
    for (int p = 0; p < passes; ++p) {
        const int shift = p * kDigitBits;
        ctx->n_launches += 3;
        radix_hist_kernel<<<nblocks, kSortThreads, 0, st>>>(ka, n, shift, nblocks, hist);
        radix_scan_kernel<<<kDigits / 8, 256, 0, st>>>(hist, nblocks, total);
        radix_scatter_kernel<<<nblocks, kSortThreads, 0, st>>>(ka, va, n, shift, nblocks, hist, total, kb, vb);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    LSPR_TRY(ctx, cudaGetLastError());
    if (ka != keys) {
        LSPR_TRY(ctx, cudaMemcpyAsync(keys, ka, sizeof(unsigned) * n, cudaMemcpyDeviceToDevice, st));
        LSPR_TRY(ctx, cudaMemcpyAsync(vals, va, sizeof(int) * n, cudaMemcpyDeviceToDevice, st));
    }
    return LSPR_OK;
}

__global__ void permute_sources_kernel(int64_t Ns, const int *__restrict__ perm, const dbl4 *__restrict__ pos,
                                       const dbl4 *__restrict__ nrm, dbl4 *spos64, dbl4 *snrm64,
                                       float4 *spos32, float4 *snrm32, int *src_panel) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= Ns) return;
    const int o = perm[s];
    const dbl4 p = pos[o], n = nrm[o];
    const int pid = (int)n.w;
    spos64[s] = p;
    snrm64[s] = n;
    spos32[s] = make_float4((float)p.x, (float)p.y, (float)p.z, (float)p.w);
    snrm32[s] = make_float4((float)n.x, (float)n.y, (float)n.z, __int_as_float(pid));
    src_panel[s] = pid;
}

__global__ void permute_targets_kernel(int64_t N, const int *__restrict__ perm, const dbl4 *__restrict__ tgt,
                                       dbl4 *tgt64, float4 *tgt32, int *tgt_panel, int *tgt_pos) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int o = perm[i];
    const dbl4 t = tgt[o];
    tgt64[i] = t;
    tgt32[i] = make_float4((float)t.x, (float)t.y, (float)t.z, __int_as_float(o));
    tgt_panel[i] = o;
    tgt_pos[o] = (int)i;
}

__global__ void src_tblock_kernel(int64_t Ns, const int *__restrict__ src_panel, const int *__restrict__ tgt_pos,
                                  int *src_tblock) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= Ns) return;
    src_tblock[s] = tgt_pos[src_panel[s]] / kTargetBlock;
}

// --------------------------------------------------------------------- octree
__device__ int lower_bound_key(const unsigned *keys, int lo, int hi, unsigned v) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (keys[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// block-wide exclusive scan of n ints in place (blockDim.x == 1024); returns the total
__device__ int block_scan_inplace(int *a, int n, int *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < n; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const int v = i < n ? a[i] : 0;
        const int inc = warp_inclusive(v, lane);
        if (lane == 31) sh[warp] = inc;
        __syncthreads();
        if (warp == 0) sh[lane] = warp_inclusive(sh[lane], lane);
        __syncthreads();
        if (i < n) a[i] = carry + (warp ? sh[warp - 1] : 0) + inc - v;
        carry += sh[31];
        __syncthreads();
    }
    return carry;
}

// One CTA, level by level.  Box b covers keys [beg, end) sharing the top 3*level
// bits; it is split into its non-empty octants while it holds more than ncrit
// sources and is above the maximum depth.  Children of a box are contiguous and
// ordered by octant; boxes are numbered level by level (deterministic).  Eight lanes take a box,
// one octant boundary each (a binary search over its keys, kept for the fill): a chain of searches
// eight times shorter than one thread per box (69 us at 81920 panels after 480).  At the end the boxes' sources are cut into slices
// of kSliceSrc, the work items of the box geometry.
constexpr int kSliceSrc = 2048;
__global__ void __launch_bounds__(1024) octree_kernel(const unsigned *__restrict__ keys, int Ns, int ncrit, int cap,
                                                      int *beg, int *end, int *child, int *nchild, int *level,
                                                      int *parent, unsigned *bkey, int *scratch, int *bound,
                                                      int2 *slices, int slice_cap, int *out /* boxes, slices */) {
    __shared__ int sh[32];
    __shared__ int s_lb, s_le, s_overflow;
    const int oct = threadIdx.x & 7, grp = threadIdx.x >> 3, ngrp = blockDim.x >> 3;
    if (threadIdx.x == 0) {
        beg[0] = 0; end[0] = Ns; level[0] = 0; bkey[0] = 0u; child[0] = -1; nchild[0] = 0; parent[0] = -1;
        s_lb = 0; s_le = 1; s_overflow = 0;
    }
    __syncthreads();
    for (int l = 0; l < kMaxDepth; ++l) {
        const int lb = s_lb, le = s_le;
        if (lb == le) break;
        const int shift = 3 * (kMaxDepth - 1 - l);
        // octant boundaries and the number of non-empty children
        for (int b0 = lb; b0 < le; b0 += ngrp) {
            const int b = b0 + grp;
            int s0 = 0, s1 = 0;
            bool split = false;
            if (b < le) {
                const int bb = beg[b], be = end[b];
                split = be - bb > ncrit;
                if (split) s0 = oct ? lower_bound_key(keys, bb, be, ((bkey[b] << 3) | oct) << shift) : bb;
                s1 = be;
            }
            const int nx = __shfl_down_sync(0xffffffffu, s0, 1, 8);
            if (oct < 7) s1 = nx;
            const unsigned m = __ballot_sync(0xffffffffu, split && s1 > s0);
            if (b < le) {
                if (split) bound[8 * (b - lb) + oct] = s0;
                if (oct == 0) scratch[b - lb] = __popc((m >> (threadIdx.x & 24)) & 0xffu);
            }
        }
        __syncthreads();
        const int total = block_scan_inplace(scratch, le - lb, sh);
        if (le + total > cap) {
            if (threadIdx.x == 0) s_overflow = 1;
            __syncthreads();
            break;
        }
        for (int b0 = lb; b0 < le; b0 += ngrp) {
            const int b = b0 + grp;
            int s0 = 0, s1 = 0;
            bool split = false;
            if (b < le) {
                const int bb = beg[b], be = end[b];
                split = be - bb > ncrit;
                if (split) s0 = bound[8 * (b - lb) + oct];
                s1 = be;
            }
            const int nx = __shfl_down_sync(0xffffffffu, s0, 1, 8);
            if (oct < 7) s1 = nx;
            const bool full = split && s1 > s0;
            const unsigned m = (__ballot_sync(0xffffffffu, full) >> (threadIdx.x & 24)) & 0xffu;
            if (b < le) {
                const int first = le + scratch[b - lb];
                if (full) {
                    const int pos = first + __popc(m & ((1u << oct) - 1u));
                    beg[pos] = s0; end[pos] = s1; level[pos] = l + 1; bkey[pos] = (bkey[b] << 3) | oct;
                    child[pos] = -1; nchild[pos] = 0; parent[pos] = b;
                }
                if (oct == 0) {
                    child[b] = split ? first : -1;
                    nchild[b] = __popc(m);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) { s_lb = le; s_le = le + total; }
        __syncthreads();
    }
    const int nb = s_le;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) scratch[b] = (end[b] - beg[b] + kSliceSrc - 1) / kSliceSrc;
    __syncthreads();
    const int ns = block_scan_inplace(scratch, nb, sh);
    if (ns > slice_cap) s_overflow = 1;   // cannot happen: slice_cap bounds the slices of a full tree
    __syncthreads();
    if (!s_overflow)
        for (int b = threadIdx.x; b < nb; b += blockDim.x) {
            const int n = (end[b] - beg[b] + kSliceSrc - 1) / kSliceSrc, o = scratch[b];
            for (int q = 0; q < n; ++q) slices[o + q] = make_int2(b, q);
        }
    if (threadIdx.x == 0) {
        out[0] = s_overflow ? -1 : nb;
        out[1] = ns;
    }
}

// Centre of the bounding box of the box's sources and r_b = max distance to it, from
// the FP32 source copies (FP64 min/max would run on the narrow FP64 pipe).  The radius is enlarged
// to cover the FP32 rounding of the coordinates (<= 2^-24 |y| each) and of the distance itself, so
// it bounds the true one.  One block per slice of a box (the root alone holds every source);
// slices meet in integer atomics on order-preserving images of the floats, so the result does not
// depend on their order.  Latency-bound: 24 us for 81920 panels, 439 with one block per box.
__device__ __forceinline__ int ford(float f) {   // order-preserving int image of a float
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ford_inv(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__global__ void box_init_kernel(int n, int *ext /* [n][8] lo, hi, r^2, |y| */) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 8 * n) return;
    const int q = i & 7;
    ext[i] = q < 3 ? 0x7fffffff : (q < 6 ? (int)0x80000000 : 0);
}

__global__ void __launch_bounds__(kGeomThreads) box_extent_kernel(const int2 *__restrict__ slices, const int *beg,
                                                                  const int *end, const float4 *__restrict__ spos,
                                                                  int *ext) {
    __shared__ int red[6];
    const int2 sl = slices[blockIdx.x];
    const int t = threadIdx.x;
    if (t < 6) red[t] = t < 3 ? 0x7fffffff : (int)0x80000000;
    __syncthreads();
    const int s0 = beg[sl.x] + sl.y * kSliceSrc, s1 = min(end[sl.x], s0 + kSliceSrc);
    float l[3] = {3e38f, 3e38f, 3e38f}, h[3] = {-3e38f, -3e38f, -3e38f};
    for (int s = s0 + t; s < s1; s += kGeomThreads) {
        const float4 p = spos[s];
        l[0] = fminf(l[0], p.x); l[1] = fminf(l[1], p.y); l[2] = fminf(l[2], p.z);
        h[0] = fmaxf(h[0], p.x); h[1] = fmaxf(h[1], p.y); h[2] = fmaxf(h[2], p.z);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int lo = __reduce_min_sync(0xffffffffu, ford(l[d])), hi = __reduce_max_sync(0xffffffffu, ford(h[d]));
        if ((t & 31) == 0) {
            atomicMin(&red[d], lo);
            atomicMax(&red[3 + d], hi);
        }
    }
    __syncthreads();
    if (t < 3) atomicMin(&ext[8 * sl.x + t], red[t]);
    else if (t < 6) atomicMax(&ext[8 * sl.x + t], red[t]);
}

__device__ __forceinline__ void box_centre(const int *ext, int b, float (&c)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d] = 0.5f * (ford_inv(ext[8 * b + d]) + ford_inv(ext[8 * b + 3 + d]));
}

__global__ void __launch_bounds__(kGeomThreads) box_radius_kernel(const int2 *__restrict__ slices, const int *beg,
                                                                  const int *end, const float4 *__restrict__ spos,
                                                                  int *ext) {
    __shared__ int red[2];
    const int2 sl = slices[blockIdx.x];
    const int t = threadIdx.x;
    if (t < 2) red[t] = 0;
    float cen[3];
    box_centre(ext, sl.x, cen);
    __syncthreads();
    const int s0 = beg[sl.x] + sl.y * kSliceSrc, s1 = min(end[sl.x], s0 + kSliceSrc);
    float r2 = 0.f, ymax = 0.f;
    for (int s = s0 + t; s < s1; s += kGeomThreads) {
        const float4 p = spos[s];
        const float dx = p.x - cen[0], dy = p.y - cen[1], dz = p.z - cen[2];
        r2 = fmaxf(r2, dx * dx + dy * dy + dz * dz);
        ymax = fmaxf(ymax, fmaxf(fabsf(p.x), fmaxf(fabsf(p.y), fabsf(p.z))));
    }
    const int a = __reduce_max_sync(0xffffffffu, __float_as_int(r2));       // both are non-negative
    const int y = __reduce_max_sync(0xffffffffu, __float_as_int(ymax));
    if ((t & 31) == 0) {
        atomicMax(&red[0], a);
        atomicMax(&red[1], y);
    }
    __syncthreads();
    if (t < 2) atomicMax(&ext[8 * sl.x + 6 + t], red[t]);
}

__global__ void box_final_kernel(int nboxes, const int *ext, dbl4 *c64, float4 *c32) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nboxes) return;
    float cen[3];
    box_centre(ext, b, cen);
    const double rb = (double)sqrtf(__int_as_float(ext[8 * b + 6])) * (1.0 + 1e-6) +
                      4e-7 * (double)__int_as_float(ext[8 * b + 7]);
    c64[b] = make_dbl4(cen[0], cen[1], cen[2], rb);
    c32[b] = make_float4(cen[0], cen[1], cen[2], (float)(rb * (1.0 + 1e-6)));
}

// mask of the surfaces of each box's sources (several surfaces), one block per slice
__global__ void __launch_bounds__(kGeomThreads) box_surf_kernel(const int2 *__restrict__ slices, const int *beg,
                                                                const int *end, const int *__restrict__ src_panel,
                                                                const int *__restrict__ surf, int *box_surf) {
    const int2 sl = slices[blockIdx.x];
    const int s0 = beg[sl.x] + sl.y * kSliceSrc, s1 = min(end[sl.x], s0 + kSliceSrc);
    unsigned m = 0;
    for (int s = s0 + threadIdx.x; s < s1; s += kGeomThreads) m |= 1u << surf[src_panel[s]];
    m = __reduce_or_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicOr(&box_surf[sl.x], (int)m);
}

// the surface masks of the tensor-core work lists: M2P entries from their boxes, one warp per P2P
// source range
__global__ void tc_list_surf_kernel(int64_t n, int2 *list, const int *__restrict__ box_surf) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) list[i].y |= (box_surf ? box_surf[list[i].x] : 1) << kTcSurf;
}
__global__ void tc_ivl_surf_kernel(int64_t n, int4 *ivl, int S, const int *__restrict__ src_panel,
                                   const int *__restrict__ surf, int *mask, int per) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    unsigned m = S > 1 ? 0u : 1u;
    if (S > 1)
        for (int s = ivl[i].x + lane; s < ivl[i].y; s += 32) m |= 1u << surf[src_panel[s]];
    m = __reduce_or_sync(0xffffffffu, m);
    if (lane == 0) ivl[i].w = (int)m;
    if (S > 1)
        for (int g = ivl[i].x / per + lane; g * per < ivl[i].y; g += 32) atomicOr(&mask[g], (int)m);
}

// stat[0], stat[1]: smallest and largest squared distance (FP32 bits) between a target and a source of
// another panel over the P2P items, one warp per item (stat[0] starts at the largest int)
__global__ void __launch_bounds__(128)
    pair_range_kernel(int64_t nitems, const int4 *__restrict__ items, int64_t N, const float4 *__restrict__ tgt,
                      const float4 *__restrict__ spos, const int *__restrict__ src_panel, int *stat) {
    const int64_t it = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (it >= nitems) return;
    const int4 item = items[it];
    const int64_t t0 = (int64_t)item.x * kTargetBlock + lane;
    const float4 q0 = tgt[min(t0, N - 1)], q1 = tgt[min(t0 + 32, N - 1)];
    float lo = 3e38f, hi = 0.f;
#pragma unroll 4
    for (int s = item.y; s < item.z; ++s) {
        const float4 p = __ldg(spos + s);
        const int id = __ldg(src_panel + s);
        const float ax = q0.x - p.x, ay = q0.y - p.y, az = q0.z - p.z;
        const float bx = q1.x - p.x, by = q1.y - p.y, bz = q1.z - p.z;
        const float ra = ax * ax + ay * ay + az * az, rb = bx * bx + by * by + bz * bz;
        if (id != __float_as_int(q0.w)) { lo = fminf(lo, ra); hi = fmaxf(hi, ra); }
        if (id != __float_as_int(q1.w)) { lo = fminf(lo, rb); hi = fmaxf(hi, rb); }
    }
    const int l = __reduce_min_sync(0xffffffffu, __float_as_int(lo)), h = __reduce_max_sync(0xffffffffu, __float_as_int(hi));
    if (lane == 0) {
        if (l < __ldcg(stat)) atomicMin(stat, l);
        if (h > __ldcg(stat + 1)) atomicMax(stat + 1, h);
    }
}

// geometry of the sources of every stage (n of them), one row per component, in the layout that the
// tensor-core P2P reads: positions negated and divided by gs, normals times ts / gs^2 (the scales of G
// and dG/dn, see p2p_tc.cu); sources past the end repeat the last one.  stat[2]: the largest weight.
__global__ void tc_src_kernel(int64_t Ns, int n, float gs, float ts, const float4 *__restrict__ spos,
                              const float4 *__restrict__ snrm, float *src, int *stat) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t s = min(i, Ns - 1);
    const float4 p = spos[s], v = snrm[s];
    const int w = __reduce_max_sync(0xffffffffu, __float_as_int(fabsf(p.w * (float)kInv4Pi)));
    if ((threadIdx.x & 31) == 0) atomicMax(stat + 2, w);
    if (i >= (Ns + n - 1) / n * n) return;
    const float ig = 1.f / gs, f = ts * ig * ig;
    float *o = src + i / n * (kTcSrcRows * n) + i % n;
    o[0] = -p.x * ig;
    o[n] = -p.y * ig;
    o[2 * n] = -p.z * ig;
    o[3 * n] = v.x * f;
    o[4 * n] = v.y * f;
    o[5 * n] = v.z * f;
    o[6 * n] = v.w;
    o[7 * n] = 0.f;
}

// box node of the list walk: (first child or -1, children, source begin, source end)
__global__ void box_nodes_kernel(int nboxes, const int *beg, const int *end, const int *child, const int *nchild,
                                 int4 *node) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nboxes) node[b] = make_int4(child[b], nchild[b], beg[b], end[b]);
}

// one warp per target block
__global__ void tblock_bbox_kernel(int64_t ntb, int64_t N, const dbl4 *__restrict__ tgt, dbl4 *lo, dbl4 *hi) {
    const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= ntb) return;
    double l[3] = {1e300, 1e300, 1e300}, h[3] = {-1e300, -1e300, -1e300};
    for (int64_t i = b * kTargetBlock + lane; i < min(N, (b + 1) * kTargetBlock); i += 32) {
        const dbl4 p = tgt[i];
        l[0] = fmin(l[0], p.x); l[1] = fmin(l[1], p.y); l[2] = fmin(l[2], p.z);
        h[0] = fmax(h[0], p.x); h[1] = fmax(h[1], p.y); h[2] = fmax(h[2], p.z);
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int d = 0; d < 3; ++d) {
            l[d] = fmin(l[d], __shfl_xor_sync(0xffffffffu, l[d], o));
            h[d] = fmax(h[d], __shfl_xor_sync(0xffffffffu, h[d], o));
        }
    if (lane == 0) {
        lo[b] = make_dbl4(l[0], l[1], l[2], 0);
        hi[b] = make_dbl4(h[0], h[1], h[2], 0);
    }
}

// Multipole-acceptance test of box (c, r_b) against a target block's bounding box:
// r = distance from c to the nearest point of the block.  Accepted iff
// r_b < theta * r and the box keeps clear of every target's own panel and of its
// near-singular panels (r - r_b > clear), so that those stay in direct sums.
__device__ __forceinline__ bool mac_accept(const dbl4 &c, const dbl4 &lo, const dbl4 &hi, double theta,
                                           double clear) {
    const double dx = fmax(0.0, fmax(lo.x - c.x, c.x - hi.x));
    const double dy = fmax(0.0, fmax(lo.y - c.y, c.y - hi.y));
    const double dz = fmax(0.0, fmax(lo.z - c.z, c.z - hi.z));
    const double r = sqrt(dx * dx + dy * dy + dz * dz);
    return c.w < theta * r && r - c.w > clear;
}

// The same decision from FP32 copies where they settle it (the box centres are FP32 values, the
// block's bounds are rounded), else in FP64: margin bounds the difference of both sides of each
// comparison, from 2^-24 of the coordinates (at most cmax), the radius's 1e-6 enlargement and the
// arithmetic, twice over.  The FP64 test alone made the list walk FP64-bound.
__device__ __forceinline__ bool mac_decide(const float4 &c, const float4 &lo, const float4 &hi, float cmax, float theta,
                                           float clear, const dbl4 *c64, const dbl4 &lo64, const dbl4 &hi64,
                                           double theta64, double clear64) {
    const float dx = fmaxf(0.f, fmaxf(lo.x - c.x, c.x - hi.x));
    const float dy = fmaxf(0.f, fmaxf(lo.y - c.y, c.y - hi.y));
    const float dz = fmaxf(0.f, fmaxf(lo.z - c.z, c.z - hi.z));
    const float r = sqrtf(dx * dx + dy * dy + dz * dz);
    const float margin = 1e-6f * cmax + 3e-6f * r + 6e-6f * c.w + 1e-6f * clear;
    const float a = fminf(theta * r - c.w, r - c.w - clear);
    if (a > margin) return true;
    if (a < -margin) return false;
    return mac_accept(*c64, lo64, hi64, theta64, clear64);
}

// One warp per target block walks the tree depth first.  A popped box is known to be
// rejected by the MAC: a leaf becomes a direct (P2P) source range, merged with the
// previous range when contiguous; for an internal box the lanes test its children in
// parallel, accepted children join the block's M2P list and rejected ones are pushed in
// reverse octant order, so leaves come out in Morton order.
// The stack holds the boxes' nodes, loaded together with their acceptance test, so that a pop costs
// one dependent load (the children's centres and nodes) instead of three.  81920 panels:
// 63 us (counting) and 98 us (filling) a walk, 245 with the acceptance test in FP64, 283 before that.
// FILL = false: count P2P items, M2P boxes and M2P items per target block.
// FILL = true: write them at the scanned offsets and mark accepted boxes as used.
constexpr int kListWarps = 4;
template <bool FILL>
__global__ void __launch_bounds__(kListWarps * 32) lists_kernel(
    int64_t ntb, int64_t N, const dbl4 *lo, const dbl4 *hi, const dbl4 *__restrict__ bc,
    const float4 *__restrict__ bc32, const int4 *__restrict__ node, double theta, double clear, int *n_p2p, int *n_m2p, int *n_m2pi,
    const int *o_p2p, const int *o_m2p, const int *o_m2pi, int4 *p2p_items, int *m2p_list, int4 *m2p_items,
    int *used, unsigned long long *pairs, int *overflow) {
    __shared__ int4 stk[kListWarps][kStack];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t tb = (int64_t)blockIdx.x * kListWarps + warp;
    if (tb >= ntb) return;
    int4 *stack = stk[warp];
    const dbl4 l = lo[tb], h = hi[tb];
    const float4 lf = make_float4((float)l.x, (float)l.y, (float)l.z, 0.f);
    const float4 hf = make_float4((float)h.x, (float)h.y, (float)h.z, 0.f);
    const float cmax = fmaxf(fmaxf(fmaxf(fabsf(lf.x), fabsf(hf.x)), fmaxf(fabsf(lf.y), fabsf(hf.y))),
                             fmaxf(fabsf(lf.z), fabsf(hf.z)));
    const float thf = (float)theta, clf = (float)clear;
    const int ntgt = (int)min((int64_t)kTargetBlock, N - tb * kTargetBlock);
    if (lane == 0) stack[0] = node[0];
    __syncwarp();
    int sp = 1;
    int np = 0, nm = 0;
    int cur_b = -1, cur_e = -1;   // pending merged P2P range
    int p_out = FILL ? o_p2p[tb] : 0, m_out = FILL ? o_m2p[tb] : 0;
    unsigned long long pp = 0;
    auto flush = [&](int b0, int e0) {
        const int n = e0 - b0;
        const int k = (n + kP2PChunk - 1) / kP2PChunk;
        for (int q = 0; q < k; ++q) {
            const int s0 = b0 + (int)((int64_t)n * q / k), s1 = b0 + (int)((int64_t)n * (q + 1) / k);
            if (FILL && lane == 0) p2p_items[p_out] = make_int4((int)tb, s0, s1, 0);
            ++p_out;
        }
        np += k;
        pp += (unsigned long long)n * ntgt;
    };
    bool ovf = false;
    while (sp > 0) {
        const int4 bn = stack[--sp];
        __syncwarp();
        const int nc = bn.y;
        if (nc == 0) {
            if (cur_e == bn.z) {
                cur_e = bn.w;
            } else {
                if (cur_b >= 0) flush(cur_b, cur_e);
                cur_b = bn.z;
                cur_e = bn.w;
            }
            continue;
        }
        int ch = -1;
        int4 cn = make_int4(0, 0, 0, 0);
        bool acc = false, push = false;
        if (lane < nc) {
            ch = bn.x + lane;
            cn = node[ch];
            acc = mac_decide(bc32[ch], lf, hf, cmax, thf, clf, bc + ch, l, h, theta, clear);
            push = !acc;
        }
        const unsigned am = __ballot_sync(0xffffffffu, acc), pm = __ballot_sync(0xffffffffu, push);
        const unsigned below = (1u << lane) - 1u;
        if (FILL && acc) {
            m2p_list[m_out + __popc(am & below)] = ch;
            used[ch] = 1;
        }
        m_out += __popc(am);
        nm += __popc(am);
        const int npush = __popc(pm);
        if (sp + npush > kStack) {
            ovf = true;
            break;
        }
        if (push) stack[sp + npush - 1 - __popc(pm & below)] = cn;
        __syncwarp();
        sp += npush;
    }
    if (ovf) {
        if (lane == 0) atomicOr(overflow, 1);
        return;
    }
    if (cur_b >= 0) flush(cur_b, cur_e);
    const int nmi = (nm + kM2PSeg - 1) / kM2PSeg;
    if (lane != 0) return;
    if (!FILL) {
        n_p2p[tb] = np;
        n_m2p[tb] = nm;
        n_m2pi[tb] = nmi;
        atomicAdd(pairs, pp);
    } else {
        const int base = o_m2p[tb];
        for (int q = 0; q < nmi; ++q) {
            const int s0 = base + q * kM2PSeg, s1 = min(base + nm, s0 + kM2PSeg);
            m2p_items[o_m2pi[tb] + q] = make_int4((int)tb, s0, s1, 0);
        }
    }
}

// exclusive scans of the int arrays in + q n (one block of 1024 threads each), totals to total[q]
__global__ void __launch_bounds__(1024) scan_int_kernel(const int *in, int64_t n, int *out, int64_t *total) {
    __shared__ int64_t sh[33];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    in += blockIdx.x * n;
    out += blockIdx.x * n;
    int64_t run = 0;
    for (int64_t base = 0; base < n; base += 1024) {
        const int64_t i = base + t;
        const int v = i < n ? in[i] : 0;
        int64_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t w = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += w;
        }
        if (lane == 31) sh[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            int64_t x = sh[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t w = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += w;
            }
            sh[lane] = x;
        }
        __syncthreads();
        if (i < n) out[i] = (int)(run + (warp ? sh[warp - 1] : 0) + inc - v);
        run += sh[31];
        __syncthreads();
    }
    if (t == 0) total[blockIdx.x] = run;
}

// P2M work items (leaf, source begin, source end): the leaves with an accepted box among
// themselves or their ancestors, in pieces of kP2MChunk sources, in any order
__global__ void p2m_items_kernel(int nboxes, const int4 *__restrict__ node, const int *__restrict__ parent,
                                 const int *__restrict__ used, int4 *items, int *count) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nboxes) return;
    const int4 nd = node[b];
    if (nd.y != 0) return;
    bool under = false;
    for (int A = b; A >= 0 && !under; A = parent[A]) under = used[A] != 0;
    if (!under) return;
    const int n = (nd.w - nd.z + kP2MChunk - 1) / kP2MChunk;
    int o = atomicAdd(count, n);
    for (int s0 = nd.z; s0 < nd.w; s0 += kP2MChunk) items[o++] = make_int4(b, s0, min(nd.w, s0 + kP2MChunk), 0);
}

// --------------------------------------------------------------------- driver
int tree_build(lspr_ctx *ctx, double theta, int P, int Ncrit) {
    Mesh &m = ctx->mesh;
    Tree &tr = ctx->tree;
    WorkOrder &w = ctx->wo;
    cudaStream_t st = ctx->stream;
    tr.ready = false;
    tr.theta = theta;
    tr.P = P;
    tr.Ncrit = Ncrit;
    tr.NT = n_terms(P);
    const int64_t Ns = m.Ns, N = m.N;
    cudaEvent_t ev;
    timer_begin(ctx, T_TREE, &ev);

    Tmp<double> cube(ctx->scratch[0]);
    LSPR_TRY(ctx, cube.ensure(8 + 6 * kBoxBlocks));
    LSPR_TRY_ST(launch_bbox(ctx, m.src_pos64.p, Ns, m.tgt64.p, N, cube.p + 8, cube.p));
    double hb[6];
    LSPR_TRY(ctx, cudaMemcpyAsync(hb, cube.p, sizeof(hb), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    double size = std::max(hb[3] - hb[0], std::max(hb[4] - hb[1], hb[5] - hb[2]));
    size = size * (1.0 + 1e-6) + 1e-12;
    double hc[4] = {hb[0] - 1e-7 * size, hb[1] - 1e-7 * size, hb[2] - 1e-7 * size, size * (1.0 + 2e-7)};
    LSPR_TRY(ctx, cudaMemcpyAsync(cube.p, hc, sizeof(hc), cudaMemcpyHostToDevice, st));

    // keys and sort
    Tmp<unsigned> keys(ctx->scratch[1]), ktmp(ctx->scratch[2]);
    Tmp<int> vals(ctx->scratch[3]), vtmp(ctx->scratch[4]), hist(ctx->scratch[5]), offs(ctx->scratch[6]);
    const int64_t nmax = std::max(Ns, N);
    LSPR_TRY(ctx, keys.ensure(nmax));
    LSPR_TRY(ctx, ktmp.ensure(nmax));
    LSPR_TRY(ctx, vals.ensure(nmax));
    LSPR_TRY(ctx, vtmp.ensure(nmax));
    LSPR_TRY(ctx, hist.ensure(radix_sort_scratch_ints(nmax)));
    LSPR_TRY(ctx, offs.ensure(kDigits));
    LSPR_TRY(ctx, w.spos64.ensure(Ns));
    LSPR_TRY(ctx, w.snrm64.ensure(Ns));
    LSPR_TRY(ctx, w.spos32.ensure(Ns));
    LSPR_TRY(ctx, w.snrm32.ensure(Ns));
    LSPR_TRY(ctx, w.src_panel.ensure(Ns));
    LSPR_TRY(ctx, w.tgt64.ensure(N));
    LSPR_TRY(ctx, w.tgt32.ensure(N));
    LSPR_TRY(ctx, w.tgt_panel.ensure(N));
    LSPR_TRY(ctx, w.tgt_pos.ensure(N));
    LSPR_TRY(ctx, w.src_tblock.ensure(Ns));

    // targets first (their sorted keys are not kept)
    ++ctx->n_launches;
    morton_kernel<<<grid_for(N, 256), 256, 0, st>>>(m.tgt64.p, N, cube.p, keys.p, vals.p);
    LSPR_TRY_ST(radix_sort(ctx, keys.p, vals.p, ktmp.p, vtmp.p, N, 30, hist.p, offs.p));
    ++ctx->n_launches;
    permute_targets_kernel<<<grid_for(N, 256), 256, 0, st>>>(N, vals.p, m.tgt64.p, w.tgt64.p, w.tgt32.p, w.tgt_panel.p,
                                                              w.tgt_pos.p);
    // sources
    ++ctx->n_launches;
    morton_kernel<<<grid_for(Ns, 256), 256, 0, st>>>(m.src_pos64.p, Ns, cube.p, keys.p, vals.p);
    LSPR_TRY_ST(radix_sort(ctx, keys.p, vals.p, ktmp.p, vtmp.p, Ns, 30, hist.p, offs.p));
    ++ctx->n_launches;
    permute_sources_kernel<<<grid_for(Ns, 256), 256, 0, st>>>(Ns, vals.p, m.src_pos64.p, m.src_nrm64.p, w.spos64.p,
                                                              w.snrm64.p, w.spos32.p, w.snrm32.p, w.src_panel.p);
    ++ctx->n_launches;
    src_tblock_kernel<<<grid_for(Ns, 256), 256, 0, st>>>(Ns, w.src_panel.p, w.tgt_pos.p, w.src_tblock.p);
    LSPR_TRY(ctx, cudaGetLastError());
    // the direct-mode items now address the Morton work order: refresh their own-panel flags
    LSPR_TRY_ST(launch_direct_flags(ctx));
    LSPR_TRY_ST(launch_ff_geometry(ctx));

    // octree
    const int64_t cap64 = 1 + 8LL * kMaxDepth * (Ns / (Ncrit + 1) + 1);
    const int cap = (int)std::min<int64_t>(cap64, 1 << 30);
    for (DArr<int> *a : {&tr.box_beg, &tr.box_end, &tr.box_child, &tr.box_nchild, &tr.box_level, &tr.box_used})
        LSPR_TRY(ctx, a->ensure(cap));
    LSPR_TRY(ctx, tr.box_key.ensure(cap));
    LSPR_TRY(ctx, tr.box_parent.ensure(cap));
    // a split box holds more than Ncrit sources, so a level has at most 8 (Ns / (Ncrit + 1)) boxes
    Tmp<int> scratch(ctx->scratch[7]), nbox_d(ctx->scratch[8]), bound(ctx->scratch[9]);
    LSPR_TRY(ctx, scratch.ensure(cap));
    LSPR_TRY(ctx, bound.ensure(8 + 64 * (size_t)(Ns / (Ncrit + 1) + 1)));
    LSPR_TRY(ctx, nbox_d.ensure(2));
    // a level's boxes hold Ns sources in all, so it has at most Ns / kSliceSrc slices and one per box
    const int slice_cap = cap + (kMaxDepth + 1) * (int)(Ns / kSliceSrc + 1);
    Tmp<int2> slices(ctx->scratch[10]);
    LSPR_TRY(ctx, slices.ensure(slice_cap));
    ++ctx->n_launches;
    octree_kernel<<<1, 1024, 0, st>>>(keys.p, (int)Ns, Ncrit, cap, tr.box_beg.p, tr.box_end.p, tr.box_child.p,
                                      tr.box_nchild.p, tr.box_level.p, tr.box_parent.p, tr.box_key.p, scratch.p,
                                      bound.p, slices.p, slice_cap, nbox_d.p);
    LSPR_TRY(ctx, cudaGetLastError());
    int nbs[2] = {0, 0};
    LSPR_TRY(ctx, cudaMemcpyAsync(nbs, nbox_d.p, sizeof(nbs), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    const int nboxes = nbs[0];
    if (nboxes <= 0) {
        ctx->last_error = "octree capacity exceeded";
        return LSPR_E_OOM;
    }
    tr.nboxes = nboxes;
    LSPR_TRY(ctx, tr.box_c64.ensure(nboxes));
    LSPR_TRY(ctx, tr.box_c32.ensure(nboxes));
    LSPR_TRY(ctx, tr.box_node.ensure(nboxes));
    Tmp<int> ext(ctx->scratch[11]);
    LSPR_TRY(ctx, ext.ensure(8 * (size_t)nboxes));
    ctx->n_launches += 5;
    box_init_kernel<<<grid_for(8 * nboxes, 256), 256, 0, st>>>(nboxes, ext.p);
    box_extent_kernel<<<nbs[1], kGeomThreads, 0, st>>>(slices.p, tr.box_beg.p, tr.box_end.p, w.spos32.p, ext.p);
    box_radius_kernel<<<nbs[1], kGeomThreads, 0, st>>>(slices.p, tr.box_beg.p, tr.box_end.p, w.spos32.p, ext.p);
    box_final_kernel<<<grid_for(nboxes, 256), 256, 0, st>>>(nboxes, ext.p, tr.box_c64.p, tr.box_c32.p);
    box_nodes_kernel<<<grid_for(nboxes, 256), 256, 0, st>>>(nboxes, tr.box_beg.p, tr.box_end.p, tr.box_child.p,
                                                            tr.box_nchild.p, tr.box_node.p);
    if (m.S > 1) {
        LSPR_TRY(ctx, tr.box_surf.ensure(nboxes));
        LSPR_TRY(ctx, cudaMemsetAsync(tr.box_surf.p, 0, sizeof(int) * nboxes, st));
        ++ctx->n_launches;
        box_surf_kernel<<<nbs[1], kGeomThreads, 0, st>>>(slices.p, tr.box_beg.p, tr.box_end.p, w.src_panel.p, m.surf.p,
                                                         tr.box_surf.p);
    }
    LSPR_TRY_ST(launch_ff_boxes(ctx));

    // target blocks
    const int64_t ntb = (N + kTargetBlock - 1) / kTargetBlock;
    tr.ntblocks = ntb;
    Tmp<dbl4> tlo(ctx->scratch[5]), thi(ctx->scratch[6]);
    LSPR_TRY(ctx, tlo.ensure(ntb));
    LSPR_TRY(ctx, thi.ensure(ntb));
    ++ctx->n_launches;
    tblock_bbox_kernel<<<grid_for(ntb * 32, 128), 128, 0, st>>>(ntb, N, w.tgt64.p, tlo.p, thi.p);

    // lists: count
    const double clear = m.Lmax / m.thr + m.rho_max;
    // an accepted box is at least clear away; a power of two, since recorded graphs are told apart by it
    tr.rho_min = (float)std::exp2(std::floor(std::log2(theta * clear)));
    Tmp<int> cnt3(ctx->scratch[11]), off3(ctx->scratch[12]);
    Tmp<int64_t> tot3(ctx->scratch[13]);
    Tmp<unsigned long long> pairs(ctx->scratch[14]);
    Tmp<int> ovf(ctx->scratch[15]);
    LSPR_TRY(ctx, cnt3.ensure(3 * ntb));
    LSPR_TRY(ctx, off3.ensure(3 * ntb));
    LSPR_TRY(ctx, tot3.ensure(3));
    LSPR_TRY(ctx, pairs.ensure(1));
    LSPR_TRY(ctx, ovf.ensure(1));
    LSPR_TRY(ctx, cudaMemsetAsync(pairs.p, 0, sizeof(unsigned long long), st));
    LSPR_TRY(ctx, cudaMemsetAsync(ovf.p, 0, sizeof(int), st));
    LSPR_TRY(ctx, cudaMemsetAsync(tr.box_used.p, 0, sizeof(int) * nboxes, st));
    ++ctx->n_launches;
    lists_kernel<false><<<grid_for(ntb, kListWarps), kListWarps * 32, 0, st>>>(
        ntb, N, tlo.p, thi.p, tr.box_c64.p, tr.box_c32.p, tr.box_node.p, theta, clear,
        cnt3.p, cnt3.p + ntb, cnt3.p + 2 * ntb, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
        pairs.p, ovf.p);
    ++ctx->n_launches;
    scan_int_kernel<<<3, 1024, 0, st>>>(cnt3.p, ntb, off3.p, tot3.p);
    LSPR_TRY(ctx, cudaGetLastError());
    int64_t tot[3];
    unsigned long long hp = 0;
    int hovf = 0;
    LSPR_TRY(ctx, cudaMemcpyAsync(tot, tot3.p, sizeof(tot), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaMemcpyAsync(&hp, pairs.p, sizeof(hp), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaMemcpyAsync(&hovf, ovf.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    if (hovf) {
        ctx->last_error = "tree traversal stack overflow";
        return LSPR_E_ARG;
    }
    tr.n_p2p_items = tot[0];
    tr.n_m2p_pairs = tot[1];
    tr.n_m2p_items = tot[2];
    tr.p2p_pairs = (int64_t)hp;
    LSPR_TRY(ctx, tr.p2p_items.ensure(std::max<int64_t>(1, tot[0])));
    LSPR_TRY(ctx, tr.m2p_list.ensure(std::max<int64_t>(1, tot[1])));
    LSPR_TRY(ctx, tr.m2p_items.ensure(std::max<int64_t>(1, tot[2])));
    ++ctx->n_launches;
    lists_kernel<true><<<grid_for(ntb, kListWarps), kListWarps * 32, 0, st>>>(
        ntb, N, tlo.p, thi.p, tr.box_c64.p, tr.box_c32.p, tr.box_node.p, theta, clear,
        nullptr, nullptr, nullptr, off3.p, off3.p + ntb, off3.p + 2 * ntb, tr.p2p_items.p, tr.m2p_list.p,
        tr.m2p_items.p, tr.box_used.p, pairs.p, ovf.p);
    LSPR_TRY(ctx, cudaGetLastError());
    LSPR_TRY_ST(launch_item_flags(ctx, tr.p2p_items.p, tr.n_p2p_items));

    // P2M work; each leaf chunk's moments are shifted into every accepted ancestor inside the P2M kernel
    LSPR_TRY(ctx, tr.p2m_items.ensure((size_t)nboxes + Ns / kP2MChunk + 1));
    LSPR_TRY(ctx, cudaMemsetAsync(ovf.p, 0, sizeof(int), st));
    ++ctx->n_launches;
    p2m_items_kernel<<<grid_for(nboxes, 128), 128, 0, st>>>(nboxes, tr.box_node.p, tr.box_parent.p, tr.box_used.p,
                                                            tr.p2m_items.p, ovf.p);
    int np2m = 0;
    LSPR_TRY(ctx, cudaMemcpyAsync(&np2m, ovf.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    // the group lists of the tensor-core far field are formed on first use (tree_tc_lists)
    tr.tc_built = tr.tcp_built = tr.tcp_f16 = false;
    tr.tcp_gs = tr.tcp_ts = 1.f;
    tr.n_tc_items = tr.n_tc_pairs = tr.n_tcp_items = tr.n_tcp_ivl = tr.n_tcp_sources = tr.n_tcp_stages = 0;
    timer_end(ctx, T_TREE, ev);
    LSPR_TRY(ctx, cudaGetLastError());
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    tr.n_p2m_items = np2m;
    tr.ready = true;
    return LSPR_OK;
}


// Group lists of the tensor-core far field (groups of kTcGroup consecutive target blocks), formed
// on the host from the tree's lists on first use after a tree build: the M2P lists always, the
// P2P source ranges when p2p is set.  Host copies and a synchronisation: not to be called while
// a stream is being captured (solves form them before their first product).
int tree_tc_lists(lspr_ctx *ctx, bool p2p) {
    Tree &tr = ctx->tree;
    cudaStream_t st = ctx->stream;
    const int64_t ntb = tr.ntblocks;
    if (!tr.ready) return LSPR_E_STATE;
    if (!tr.tc_built) {
        // M2P lists of the groups
        std::vector<int> hlist((size_t)tr.n_m2p_pairs);
        std::vector<int4> hitems((size_t)tr.n_m2p_items);
        if (tr.n_m2p_pairs > 0) {
            LSPR_TRY(ctx, cudaMemcpyAsync(hlist.data(), tr.m2p_list.p, sizeof(int) * tr.n_m2p_pairs, cudaMemcpyDeviceToHost, st));
            LSPR_TRY(ctx, cudaMemcpyAsync(hitems.data(), tr.m2p_items.p, sizeof(int4) * tr.n_m2p_items, cudaMemcpyDeviceToHost, st));
            LSPR_TRY(ctx, cudaStreamSynchronize(st));
        }
        std::vector<TcEntry> glist;
        std::vector<TcItem> gitems;
        tc_union_m2p(ntb, kTcGroup, hlist.data(), (const int *)hitems.data(), tr.n_m2p_items, glist, gitems);
        tr.n_tc_pairs = (int64_t)glist.size();
        tc_cut_m2p(tc_unit(tr.n_tc_pairs, ctx->num_sms, kTcSegMin, kTcSegMax), gitems);
        tr.n_tc_items = (int64_t)gitems.size();
        LSPR_TRY(ctx, tr.tc_list.ensure(std::max<size_t>(1, glist.size())));
        LSPR_TRY(ctx, tr.tc_items.ensure(std::max<size_t>(1, gitems.size())));
        if (!glist.empty()) {
            static_assert(sizeof(TcEntry) == sizeof(int2) && sizeof(TcItem) == sizeof(int4), "device layouts");
            LSPR_TRY(ctx, cudaMemcpyAsync(tr.tc_list.p, glist.data(), sizeof(int2) * glist.size(), cudaMemcpyHostToDevice, st));
            LSPR_TRY(ctx, cudaMemcpyAsync(tr.tc_items.p, gitems.data(), sizeof(int4) * gitems.size(), cudaMemcpyHostToDevice, st));
            ++ctx->n_launches;
            tc_list_surf_kernel<<<grid_for(glist.size(), 256), 256, 0, st>>>(
                (int64_t)glist.size(), tr.tc_list.p, ctx->mesh.S > 1 ? tr.box_surf.p : nullptr);
            LSPR_TRY(ctx, cudaGetLastError());
        }
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
        tr.tc_built = true;
    }
    if (p2p && !tr.tcp_built) {
        // P2P source ranges of the same groups
        std::vector<int4> hp2p((size_t)tr.n_p2p_items);
        if (tr.n_p2p_items > 0) {
            LSPR_TRY(ctx, cudaMemcpyAsync(hp2p.data(), tr.p2p_items.p, sizeof(int4) * tr.n_p2p_items,
                                          cudaMemcpyDeviceToHost, st));
            LSPR_TRY(ctx, cudaStreamSynchronize(st));
        }
        std::vector<TcRange> pivl;
        std::vector<TcItem> pitems;
        static_assert(sizeof(TcRange) == sizeof(int4), "device layout");
        const int64_t psrc = tc_union_p2p(ntb, kTcGroup, (const int *)hp2p.data(), tr.n_p2p_items, pivl, pitems);
        tr.n_tcp_sources = psrc;
        tr.n_tcp_stages = 0;
        // the range of distances chooses the operand parts and their scales
        const int64_t Ns = ctx->mesh.Ns;
        int stat[3] = {0x7fffffff, 0, 0};
        LSPR_TRY(ctx, tr.tcp_stat.ensure(3));
        LSPR_TRY(ctx, cudaMemcpyAsync(tr.tcp_stat.p, stat, sizeof(stat), cudaMemcpyHostToDevice, st));
        if (tr.n_p2p_items > 0) {
            ++ctx->n_launches;
            pair_range_kernel<<<grid_for(tr.n_p2p_items * 32, 128), 128, 0, st>>>(
                tr.n_p2p_items, tr.p2p_items.p, ctx->mesh.N, ctx->wo.tgt32.p, ctx->wo.spos32.p, ctx->wo.src_panel.p,
                tr.tcp_stat.p);
            LSPR_TRY(ctx, cudaGetLastError());
            LSPR_TRY(ctx, cudaMemcpyAsync(stat, tr.tcp_stat.p, sizeof(stat), cudaMemcpyDeviceToHost, st));
            LSPR_TRY(ctx, cudaStreamSynchronize(st));
        }
        float r2lo, r2hi;
        std::memcpy(&r2lo, &stat[0], sizeof(float));
        std::memcpy(&r2hi, &stat[1], sizeof(float));
        // moderate lengths only, so that no scale leaves the FP32 range
        tr.tcp_f16 = r2lo > 1e-12f && r2hi < 1e12f && r2hi <= kTcP2PRange * kTcP2PRange * r2lo;
        tr.tcp_gs = tr.tcp_f16 ? std::exp2(std::floor(std::log2(32768.f * std::sqrt(r2lo)))) : 1.f;
        tr.tcp_ts = tr.tcp_f16 ? std::exp2(std::floor(std::log2(32768.f * r2lo))) : 1.f;
        const int per = tr.tcp_f16 ? 16 : 8;   // sources per stage
        tc_cut_p2p(tc_unit(psrc, ctx->num_sms, kTcSrcMin, tr.tcp_f16 ? kTcSrcMax : kTcSrcMaxTf32), pivl, pitems);
        tr.n_tcp_items = (int64_t)pitems.size();
        tr.n_tcp_ivl = (int64_t)pivl.size();
        for (const TcRange &r : pivl) tr.n_tcp_stages += (r.s1 + per - 1) / per - r.s0 / per;
        LSPR_TRY(ctx, tr.tcp_items.ensure(std::max<size_t>(1, pitems.size())));
        const int64_t ng = (Ns + per - 1) / per;
        if (ctx->mesh.S > 1) {
            LSPR_TRY(ctx, tr.tcp_mask.ensure((size_t)ng));
            LSPR_TRY(ctx, cudaMemsetAsync(tr.tcp_mask.p, 0, sizeof(int) * ng, st));
        }
        LSPR_TRY(ctx, tr.tcp_src.ensure((size_t)ng * (kTcSrcRows * per)));
        ++ctx->n_launches;
        tc_src_kernel<<<grid_for(ng * per, 256), 256, 0, st>>>(Ns, per, tr.tcp_gs, tr.tcp_ts, ctx->wo.spos32.p,
                                                               ctx->wo.snrm32.p, tr.tcp_src.p, tr.tcp_stat.p);
        LSPR_TRY(ctx, tr.tcp_ivl.ensure(std::max<size_t>(1, pivl.size())));
        if (!pitems.empty()) {
            LSPR_TRY(ctx, cudaMemcpyAsync(tr.tcp_items.p, pitems.data(), sizeof(int4) * pitems.size(),
                                          cudaMemcpyHostToDevice, st));
            LSPR_TRY(ctx, cudaMemcpyAsync(tr.tcp_ivl.p, pivl.data(), sizeof(int4) * pivl.size(), cudaMemcpyHostToDevice, st));
            ++ctx->n_launches;
            tc_ivl_surf_kernel<<<grid_for(pivl.size() * 32, 256), 256, 0, st>>>(
                (int64_t)pivl.size(), tr.tcp_ivl.p, ctx->mesh.S, ctx->wo.src_panel.p, ctx->mesh.surf.p, tr.tcp_mask.p, per);
            LSPR_TRY(ctx, cudaGetLastError());
        }
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
        tr.tcp_built = true;
    }
    return LSPR_OK;
}

}  // namespace lspr
