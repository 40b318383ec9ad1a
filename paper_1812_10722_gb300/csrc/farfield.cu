// Far-field kernels of the matrix-vector product (Sec. II.D, Eq. summation):
// sources are the far-rule Gauss nodes y_j with weights q_j = w_j A_j dphi_j / (4 pi)
// (single layer) and mu_j = w_j A_j phi_j / (4 pi) (double layer); targets are the
// panel centroids x_i.  For every target
//     Vd_i = sum_j q_j / |x_i - y_j|,   Kp_i = sum_j mu_j (x_i - y_j).n_j / |x_i - y_j|^3
// over all sources except those of panel i itself (its singular integral is
// added exactly by the near-field correction).  Complex weights are carried as
// two real channels (the paper's real/imaginary split of the treecode work).
//
// Several right-hand sides (wavelengths) share one geometry: the kernels generate G,
// dG/dn (P2P), the monomials (P2M) or the Taylor coefficients (M2P) once per pair,
// source or (target, box) and apply them to a chunk of NB right-hand sides.
// Layouts for B right-hand sides: weights [source][B], accumulators [panel][B][4],
// moments [box][term][B].
//
//   p2p_kernel  direct sums of a 64-target block against a contiguous source range
//   p2m_kernel  moments of a leaf about its centre c in the harmonic basis g_k (the terms k with
//               k_3 <= 1, see farfield.cuh), shifted into every accepted ancestor box:
//                 M^V_k = sum_j q_j g_k(c - y_j)
//                 M^K_k = -sum_j mu_j n_j . grad g_k(c - y_j)
//   m2p_kernel  Vd_i += sum_{|k|<=P} a_k(x_i - c) k_1! k_2! M^V_k (same for K), with
//               a_k(R) = D^k (1/|R|) / k! from the recurrence
//               n |R|^2 a_k + (2n-1) sum_d R_d a_(k-e_d) + (n-1) sum_d a_(k-2e_d) = 0,
//               n = |k|, a_0 = 1/|R|.
// Partial sums are formed in the kernel's precision (FP32 or FP64) per work
// item and accumulated in FP64 with atomics.
#include <algorithm>

#include "farfield.cuh"

namespace lspr {

// ----------------------------------------------------------------- weights
// w[s][slot] = w_s A_s / (4 pi) * (dphi_b, phi_b) at the source's panel, b = map[slot]
// (identity without a map; only the first *nact slots are formed when nact is given);
// x is [B][2N] complex
// The kernels also clear the product's sums (accumulators and counters, moments): zero.p[0..n).
struct ZeroRanges {
    float4 *p[2];
    int64_t n[2];
};
__device__ __forceinline__ void clear_ranges(const ZeroRanges &z, int64_t g) {
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
    for (int q = 0; q < 2; ++q)
        for (int64_t i = g; i < z.n[q]; i += step) z.p[q][i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <typename T4>
// Several surfaces (S > 1): channel set slot = t K + k (surface t of the k-th of K running systems)
// carries the weights of the sources of surface t only (zero elsewhere), so that each surface's
// layer potentials come out separately; BS = B * S sets per source.
__global__ void weights_kernel(int64_t Ns, int64_t N, int B, int S, const dbl4 *__restrict__ spos64,
                               const int *__restrict__ src_panel, const int *__restrict__ surf,
                               const double2 *__restrict__ x, const double2 *__restrict__ xt, T4 *__restrict__ w,
                               const int *map, const int *nact, ZeroRanges zero) {
    const int BS = B * S;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    clear_ranges(zero, g);
    if (g >= Ns * BS) return;
    const int64_t s = g / BS;
    const int slot = (int)(g - s * BS);
    if (nact && slot >= *nact) return;
    const int p = src_panel[s];
    // set slot = t K + k: surface t of the k-th running system (map: k -> system)
    const int K = nact ? *nact / S : B, t = slot / K, k = slot - t * K;
    const int b = map ? map[k] : k;
    if (S > 1 && surf[p] != t) {
        w[g] = zero4<T4>();
        return;
    }
    const double wa = spos64[s].w * kInv4Pi;
    // x [B][2N], or its transposed copy xt [2N][B] when given
    const double2 phi = xt ? xt[(int64_t)p * B + b] : x[(int64_t)b * 2 * N + p];
    const double2 dphi = xt ? xt[(N + p) * B + b] : x[(int64_t)b * 2 * N + N + p];
    T4 o;
    o.x = wa * dphi.x;
    o.y = wa * dphi.y;
    o.z = wa * phi.x;
    o.w = wa * phi.y;
    w[g] = o;
}

// The same for FP32 products of several right-hand sides from the FP32 transposed copy
// xt [2N][B], in FP32 arithmetic (the weights feed FP32 kernels; FP64 arithmetic would run
// at 1/64 of the FP32 rate on this GPU)
__global__ void weights_f32t_kernel(int64_t Ns, int64_t N, int B, int S, const float4 *__restrict__ spos32,
                                    const int *__restrict__ src_panel, const int *__restrict__ surf,
                                    const float2 *__restrict__ xt, float4 *__restrict__ w, const int *map,
                                    const int *nact, ZeroRanges zero) {
    const int BS = B * S;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    clear_ranges(zero, g);
    if (g >= Ns * BS) return;
    const int64_t s = g / BS;
    const int slot = (int)(g - s * BS);
    if (nact && slot >= *nact) return;
    const int p = src_panel[s];
    const int K = nact ? *nact / S : B, t = slot / K, k = slot - t * K;
    const int b = map ? map[k] : k;
    if (S > 1 && surf[p] != t) {
        w[g] = zero4<float4>();
        return;
    }
    const float wa = spos32[s].w * (float)kInv4Pi;
    const float2 phi = xt[(int64_t)p * B + b], dphi = xt[(N + p) * B + b];
    w[g] = make_float4(wa * dphi.x, wa * dphi.y, wa * phi.x, wa * phi.y);
}

// item.w: bit 0 set iff some source of [item.y, item.z) belongs to a panel of the item's target block;
// from bit kItemSurf the mask of the sources' surfaces (several surfaces)
__global__ void item_flags_kernel(int4 *items, int64_t nitems, const int *__restrict__ src_tblock, int S,
                                  const int *__restrict__ src_panel, const int *__restrict__ surf) {
    const int64_t it = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (it >= nitems) return;
    int4 item = items[it];
    unsigned w = S > 1 ? 0u : 1u << kItemSurf;
    for (int s = item.y + lane; s < item.z; s += 32) {
        w |= src_tblock[s] == item.x;
        if (S > 1) w |= 1u << (kItemSurf + surf[src_panel[s]]);
    }
    w = __reduce_or_sync(0xffffffffu, w);
    if (lane == 0) items[it].w = (int)w;
}

// first and last target block that a chunk of sources belongs to (one warp per chunk)
__global__ void chunk_range_kernel(int64_t nch, int64_t chunk, int64_t Ns, const int *__restrict__ src_tblock,
                                   int2 *range) {
    const int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (c >= nch) return;
    int lo = 0x7fffffff, hi = -1;
    for (int64_t s = c * chunk + lane; s < min(Ns, (c + 1) * chunk); s += 32) {
        lo = min(lo, src_tblock[s]);
        hi = max(hi, src_tblock[s]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) range[c] = make_int2(lo, hi);
}

// direct-mode items i = (target block i mod ntb, source chunk i / ntb), consecutive warps sharing a
// chunk; item.w = 1 where the chunk may hold sources of the block's own panels (the flag only turns
// the own-panel test on)
__global__ void direct_items_kernel(int4 *items, int64_t ntb, int64_t nch, int64_t chunk, int64_t Ns,
                                    const int2 *__restrict__ range) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ntb * nch) return;
    const int64_t c = i / ntb, tb = i - c * ntb;
    const int2 r = range[c];
    items[i] = make_int4((int)tb, (int)(c * chunk), (int)min(Ns, (c + 1) * chunk),
                          (tb >= r.x && tb <= r.y) | kAllSurf << kItemSurf);
}

// FP64 -> float-float copies (moments accumulated in FP64, geometry)
__global__ void to_ff_kernel(int64_t n, const dbl4 *__restrict__ a, ff4 *__restrict__ b, int id_in_w) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const dbl4 v = a[i];
    ff4 o;
    o.x = ffloat(v.x);
    o.y = ffloat(v.y);
    o.z = ffloat(v.z);
    o.w = id_in_w ? ffloat(__int_as_float((int)v.w), 0.f) : ffloat(v.w);
    b[i] = o;
}

// --------------------------------------------------------------- launchers
int launch_weights(lspr_ctx *ctx, int prec, const double2 *x, const double2 *xt, int64_t N, int B, int S,
                   const float2 *xtf, bool tree) {
    const int64_t Ns = ctx->mesh.Ns;
    const int BS = B * S;
    ZeroRanges z = {{(float4 *)ctx->acc.p, nullptr}, {(int64_t)(4 * N * BS * sizeof(double) + acc_tail_ints(BS) * sizeof(int)) / 16, 0}};
    if (tree) {
        Tree &tr = ctx->tree;
        const int64_t nm = tr.nboxes * tr.NT * BS;
        if (prec == PREC_F32) {
            LSPR_TRY(ctx, tr.mom32.ensure(nm));
            z.p[1] = tr.mom32.p;
            z.n[1] = nm;
        } else {
            LSPR_TRY(ctx, tr.mom64.ensure(nm));
            z.p[1] = (float4 *)tr.mom64.p;
            z.n[1] = 2 * nm;
        }
    }
    const unsigned grid = grid_for(Ns * BS, 256);
    cudaEvent_t ev;
    timer_begin(ctx, T_WEIGHTS, &ev);
    ++ctx->n_launches;
    if (prec == PREC_F64) {
        LSPR_TRY(ctx, ctx->w64.ensure(Ns * BS));
        weights_kernel<dbl4><<<grid, 256, 0, ctx->stream>>>(Ns, N, B, S, ctx->wo.spos64.p, ctx->wo.src_panel.p, ctx->mesh.surf.p, x, xt,
                                                            ctx->w64.p, ctx->rhs_map, ctx->rhs_nact, z);
    } else if (prec == PREC_FF) {
        LSPR_TRY(ctx, ctx->w_ff.ensure(Ns * BS));
        weights_kernel<ff4><<<grid, 256, 0, ctx->stream>>>(Ns, N, B, S, ctx->wo.spos64.p, ctx->wo.src_panel.p, ctx->mesh.surf.p, x, xt,
                                                           ctx->w_ff.p, ctx->rhs_map, ctx->rhs_nact, z);
    } else if (xtf) {
        LSPR_TRY(ctx, ctx->w32.ensure(Ns * BS));
        weights_f32t_kernel<<<grid, 256, 0, ctx->stream>>>(Ns, N, B, S, ctx->wo.spos32.p, ctx->wo.src_panel.p,
                                                           ctx->mesh.surf.p, xtf, ctx->w32.p, ctx->rhs_map,
                                                           ctx->rhs_nact, z);
    } else {
        LSPR_TRY(ctx, ctx->w32.ensure(Ns * BS));
        weights_kernel<float4><<<grid, 256, 0, ctx->stream>>>(Ns, N, B, S, ctx->wo.spos64.p, ctx->wo.src_panel.p, ctx->mesh.surf.p, x, xt,
                                                              ctx->w32.p, ctx->rhs_map, ctx->rhs_nact, z);
    }
    timer_end(ctx, T_WEIGHTS, ev);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// float-float copies of the work-order geometry (after every change of work order)
int launch_ff_geometry(lspr_ctx *ctx) {
    const Mesh &m = ctx->mesh;
    WorkOrder &w = ctx->wo;
    LSPR_TRY(ctx, w.spos_ff.ensure(m.Ns));
    LSPR_TRY(ctx, w.snrm_ff.ensure(m.Ns));
    LSPR_TRY(ctx, w.tgt_ff.ensure(m.N));
    ctx->n_launches += 3;
    to_ff_kernel<<<grid_for(m.Ns, 256), 256, 0, ctx->stream>>>(m.Ns, w.spos64.p, w.spos_ff.p, 0);
    to_ff_kernel<<<grid_for(m.Ns, 256), 256, 0, ctx->stream>>>(m.Ns, w.snrm64.p, w.snrm_ff.p, 1);
    to_ff_kernel<<<grid_for(m.N, 256), 256, 0, ctx->stream>>>(m.N, w.tgt64.p, w.tgt_ff.p, 1);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

int launch_ff_boxes(lspr_ctx *ctx) {
    Tree &tr = ctx->tree;
    LSPR_TRY(ctx, tr.box_c_ff.ensure(tr.nboxes));
    ++ctx->n_launches;
    to_ff_kernel<<<grid_for(tr.nboxes, 256), 256, 0, ctx->stream>>>(tr.nboxes, tr.box_c64.p, tr.box_c_ff.p, 0);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// ---------------------------------------------- P2P, several right-hand sides in FP32
// Per tile of kPgTile sources, a block of 64 threads forms G and dG/dn of the 64-target block in shared
// memory (one target per thread, two sources at a time in packed f32x2 arithmetic) and multiplies them
// with the tile's weights as two small matrix products, V += G W_V and K += dG/dn W_K: a thread holds
// 8 targets x RB/2 channels of one layer (RB right-hand sides per chunk: 16, or 8 or 4 where no more are
// left, as in a solve whose number in use falls), so four shared-memory reads feed 64 multiply-adds.
// The FP32 pipe's share is 12 + 4 RB operations per pair.  A tile's weights are copied asynchronously
// while its kernel values are formed, the next tile's geometry behind the products.  20480 panels (86 M pairs), 16 right-hand sides: 326 us; 377 with
// both loaded through registers when the tile begins (FP32 pipe 52 % busy), 476 with two targets per lane
// and the weights read by broadcast (bound by the shared-memory reads, ten 16-byte reads per 32 packed
// multiply-adds); four targets per lane and 8 right-hand sides took 453 (217 registers, two warps per
// scheduler).  81920 panels, P 7: 12 right-hand sides 2.47 -> 2.19 ms, 20: 3.92 -> 3.43.
constexpr int kPgTile = 32, kPgThreads = 64, kPgRB = 16;
struct PgSmem {
    float G[kPgTile][kTargetBlock], T[kPgTile][kTargetBlock];
    float4 w[kPgTile][kPgRB];                               // weights, (re, im) of both layers per right-hand side
    float src[6][kPgTile];                                  // -x, -y, -z, normal
    float4 raw[2][kPgTile];                                 // the next tile's positions and normals
    int pid[kPgTile], tpid[kTargetBlock];
};
// 16 bytes into shared memory without a register; zeros where !on
__device__ __forceinline__ void copy16(float4 *dst, const float4 *src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(on ? 16 : 0)
                 : "memory");
}

template <int RB, bool CHECK>
__device__ __forceinline__ void pg_unit(const int4 &item, int B, int b0, int nb, PgSmem &sm, const float4 &q, int64_t t0,
                                        int64_t ntgt, const float4 *__restrict__ spos,
                                        const float4 *__restrict__ snrm, const float4 *__restrict__ sw,
                                        double *__restrict__ acc) {
    constexpr int NP = RB / 4;   // right-hand sides per thread
    const int tid = threadIdx.x, tx = tid & 7, layer = tid >> 5, cg = (tid >> 3) & 3;
    const int tp = panel_of(q.w);
    const float2 qx = make_float2(q.x, q.x), qy = make_float2(q.y, q.y), qz = make_float2(q.z, q.z);
    float2 a[8][NP];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int p = 0; p < NP; ++p) a[i][p] = make_float2(0.f, 0.f);
    auto fetch = [&](int base) {   // a tile's geometry; past the end: the first source again, with zero weights
        if (tid < kPgTile && base < item.z) {
            const int s = base + (tid < item.z - base ? tid : 0);
            copy16(&sm.raw[0][tid], spos + s, true);
            copy16(&sm.raw[1][tid], snrm + s, true);
        }
    };
    fetch(item.y);
    for (int base = item.y; base < item.z; base += kPgTile) {
        const int cnt = min(kPgTile, item.z - base);
        asm volatile("cp.async.wait_all;" ::: "memory");   // the geometry, behind the previous tile's products
        __syncthreads();   // the previous tile has been read
        // the weights arrive while G and dG/dn are formed
#pragma unroll 4
        for (int e = tid; e < kPgTile * RB; e += kPgThreads) {
            const int s = e / RB, j = e - s * RB;
            const bool on = s < cnt && j < nb;
            copy16(&sm.w[s][j], sw + (on ? (int64_t)(base + s) * B + b0 + j : 0), on);
        }
        if (tid < kPgTile) {
            const float4 gp = sm.raw[0][tid], gn = sm.raw[1][tid];   // this thread's own copies
            sm.src[0][tid] = -gp.x; sm.src[1][tid] = -gp.y; sm.src[2][tid] = -gp.z;
            sm.src[3][tid] = gn.x; sm.src[4][tid] = gn.y; sm.src[5][tid] = gn.z;
            sm.pid[tid] = panel_of(gn.w);
        }
        __syncthreads();
#pragma unroll 4
        for (int s = 0; s < kPgTile; s += 2) {
            const float2 dx = __fadd2_rn(qx, *(const float2 *)&sm.src[0][s]);
            const float2 dy = __fadd2_rn(qy, *(const float2 *)&sm.src[1][s]);
            const float2 dz = __fadd2_rn(qz, *(const float2 *)&sm.src[2][s]);
            const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
            float2 r = make_float2(rsq(r2.x), rsq(r2.y));
            if (CHECK) {   // the far-rule terms of the target's own panel are skipped
                r.x = sm.pid[s] == tp ? 0.f : r.x;
                r.y = sm.pid[s + 1] == tp ? 0.f : r.y;
            }
            const float2 dn = __ffma2_rn(dz, *(const float2 *)&sm.src[5][s],
                              __ffma2_rn(dy, *(const float2 *)&sm.src[4][s],
                              __fmul2_rn(dx, *(const float2 *)&sm.src[3][s])));
            const float2 t = __fmul2_rn(__fmul2_rn(dn, __fmul2_rn(r, r)), r);
            sm.G[s][tid] = r.x;
            sm.G[s + 1][tid] = r.y;
            sm.T[s][tid] = t.x;
            sm.T[s + 1][tid] = t.y;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        fetch(base + kPgTile);
        const float (*m)[kTargetBlock] = layer ? sm.T : sm.G;
#pragma unroll 4
        for (int s = 0; s < kPgTile; ++s) {
            const float4 g0 = *(const float4 *)&m[s][4 * tx], g1 = *(const float4 *)&m[s][32 + 4 * tx];
            const float g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 wp = *((const float2 *)&sm.w[s][cg + 4 * p] + layer);
#pragma unroll
                for (int i = 0; i < 8; ++i) a[i][p] = __ffma2_rn(make_float2(g[i], g[i]), wp, a[i][p]);
            }
        }
    }
    // target (i < 4: 4 tx + i, else 28 + 4 tx + i), right-hand side cg + 4 p, components 2 layer, + 1
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int t = (i < 4 ? 0 : 28) + 4 * tx + i;
        if (t0 + t >= ntgt) continue;
        double *o = acc + 4 * ((int64_t)sm.tpid[t] * B + b0) + 2 * layer;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const int j = cg + 4 * p;
            if (j < nb) {
                atomicAdd(o + 4 * j, (double)a[i][p].x);
                atomicAdd(o + 4 * j + 1, (double)a[i][p].y);
            }
        }
    }
}

template <int RB, class... A>
__device__ __forceinline__ void pg_check(const int4 &item, A &&...a) {
    if (item.w & 1) pg_unit<RB, true>(item, a...);
    else pg_unit<RB, false>(item, a...);
}

// Work units (item, chunk of kPgRB right-hand sides) from an atomic counter; nothing is done when at
// least skip_from right-hand sides are in use (the tensor-core P2P then takes the product)
__global__ void __launch_bounds__(kPgThreads, 7)
    p2p_multi_kernel(const int4 *__restrict__ items, int64_t nitems, int B, const float4 *__restrict__ tgt, int64_t ntgt,
                     const float4 *__restrict__ spos, const float4 *__restrict__ snrm, const float4 *__restrict__ sw,
                     double *__restrict__ acc, int *counter, const int *nact, int skip_from, int S) {
    __shared__ __align__(16) PgSmem sm;
    __shared__ int64_t unit_s;
    const int tid = threadIdx.x;
    const int Bact = nact ? *nact : B;   // right-hand sides in use (the first Bact slots)
    if (Bact >= skip_from) return;
    const int nbc = (Bact + kPgRB - 1) / kPgRB;
    const int64_t units = nitems * nbc;
    while (true) {
        __syncthreads();   // the previous unit's readers are done with unit_s and tpid
        if (tid == 0) unit_s = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t it = unit_s;
        if (it >= units) return;
        const int64_t ii = it / nbc;
        const int b0 = (int)(it - ii * nbc) * kPgRB, nb = min(kPgRB, Bact - b0);
        const int4 item = __ldg(items + ii);
        if (S > 1 && !((item.w >> kItemSurf) & set_surfaces(b0, nb, Bact, S))) continue;
        const int64_t t0 = (int64_t)item.x * kTargetBlock, ti = t0 + tid;
        const float4 q = ti < ntgt ? tgt[ti] : tgt[0];
        sm.tpid[tid] = panel_of(q.w);   // read after the tile's barriers
        if (nb > 8) pg_check<16>(item, B, b0, nb, sm, q, t0, ntgt, spos, snrm, sw, acc);
        else if (nb > 4) pg_check<8>(item, B, b0, nb, sm, q, t0, ntgt, spos, snrm, sw, acc);
        else pg_check<4>(item, B, b0, nb, sm, q, t0, ntgt, spos, snrm, sw, acc);
    }
}

static int p2p_multi_launch(lspr_ctx *ctx, const int4 *items, int64_t nitems, int B, double *acc, cudaStream_t st,
                            int *counter, int skip_from = 1 << 30) {
    static int occ = 0;
    const int64_t units = nitems * ((B + kPgRB - 1) / kPgRB);
    const unsigned grid =
        (unsigned)std::min<int64_t>(units, persistent_grid(ctx, p2p_multi_kernel, kPgThreads, &occ));
    p2p_multi_kernel<<<grid, kPgThreads, 0, st>>>(items, nitems, B, Views<float>::tgt(ctx), ctx->mesh.N,
                                                  Views<float>::spos(ctx), Views<float>::snrm(ctx),
                                                  Views<float>::w(ctx), acc, counter, ctx->rhs_nact, skip_from,
                                                  ctx->mesh.S);
    return LSPR_OK;
}

static int slot_of(int prec, int f32, int f64, int ff) { return prec == PREC_F64 ? f64 : (prec == PREC_FF ? ff : f32); }

int launch_p2p(lspr_ctx *ctx, int prec, const int4 *items, int64_t nitems, double *acc, cudaStream_t st,
               int *counter, int B) {
    if (nitems == 0) return LSPR_OK;
    cudaEvent_t ev;
    const int slot = slot_of(prec, T_P2P, T_P2P64, T_P2PFF);
    timer_begin_on(ctx, slot, &ev, st);
    ++ctx->n_launches;
    if (prec == PREC_F64) {
        if (B == 1) p2p_launch<double, 1>(ctx, items, nitems, B, acc, st, counter);
        else p2p_launch<double, batch_chunk<double>(2)>(ctx, items, nitems, B, acc, st, counter);
    } else if (prec == PREC_FF) {
        if (B == 1) p2p_launch<ffloat, 1>(ctx, items, nitems, B, acc, st, counter);
        else LSPR_TRY_ST(p2p_ff_multi(ctx, items, nitems, B, acc, st, counter));
    } else if (B > 1 && (ctx->tensor_cores & 2) && items == ctx->tree.p2p_items.p) {
        // the tensor-core P2P for products of at least kTcP2PMinSets right-hand sides in use, the
        // FP32 pipe below: decided on the host when every slot is in use, else on the device from
        // the count of running systems (both kernels are launched; the one not chosen returns at once)
        const int mn = kTcP2PMinSets;
        if (!ctx->rhs_nact) {
            if (B >= mn) LSPR_TRY_ST(p2p_tc_launch(ctx, acc, st, counter, B, 0));
            else LSPR_TRY_ST(p2p_multi_launch(ctx, items, nitems, B, acc, st, counter));
        } else {
            if (B >= mn) LSPR_TRY_ST(p2p_tc_launch(ctx, acc, st, counter, B, mn));
            LSPR_TRY_ST(p2p_multi_launch(ctx, items, nitems, B, acc, st, counter, mn));
        }
    } else {
        if (B == 1) p2p1_launch(ctx, items, nitems, acc, st, counter);
        else LSPR_TRY_ST(p2p_multi_launch(ctx, items, nitems, B, acc, st, counter));
    }
    timer_end_on(ctx, slot, ev, st);
    timer_rhs(ctx, slot, B);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

int launch_item_flags(lspr_ctx *ctx, int4 *items, int64_t nitems) {
    if (nitems == 0) return LSPR_OK;
    ++ctx->n_launches;
    item_flags_kernel<<<grid_for(nitems * 32, 256), 256, 0, ctx->stream>>>(items, nitems, ctx->wo.src_tblock.p, ctx->mesh.S,
                                                                          ctx->wo.src_panel.p, ctx->mesh.surf.p);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

int launch_direct_flags(lspr_ctx *ctx) {
    const int64_t ntb = (ctx->mesh.N + kTargetBlock - 1) / kTargetBlock, Ns = ctx->mesh.Ns;
    for (DirectItems *d : {&ctx->direct, &ctx->direct_multi}) {
        if (d->n == 0) continue;
        const int64_t nch = d->n / ntb;
        LSPR_TRY(ctx, d->range.ensure(nch));
        ctx->n_launches += 2;
        chunk_range_kernel<<<grid_for(nch * 32, 128), 128, 0, ctx->stream>>>(nch, d->chunk, Ns, ctx->wo.src_tblock.p,
                                                                             d->range.p);
        direct_items_kernel<<<grid_for(d->n, 256), 256, 0, ctx->stream>>>(d->items.p, ntb, nch, d->chunk, Ns,
                                                                          d->range.p);
    }
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

int launch_p2m(lspr_ctx *ctx, int prec, int B) {
    Tree &tr = ctx->tree;
    if (tr.n_p2m_items == 0) return LSPR_OK;
    const int64_t nm = tr.nboxes * tr.NT * B;
    cudaEvent_t ev;
    const int slot = slot_of(prec, T_P2M, T_P2M64, T_P2MFF);
    timer_begin(ctx, slot, &ev);
    ++ctx->n_launches;
    if (prec == PREC_F32) {
        LSPR_TRY_ST(p2m_orders_f32(ctx, B));
    } else {
        if (prec == PREC_F64) {
            LSPR_TRY_ST(p2m_orders_f64(ctx, B));
        } else {
            LSPR_TRY_ST(p2m_orders_ff(ctx, B));
            LSPR_TRY(ctx, tr.mom_ff.ensure(nm));
            ++ctx->n_launches;
            to_ff_kernel<<<grid_for(nm, 256), 256, 0, ctx->stream>>>(nm, tr.mom64.p, tr.mom_ff.p, 0);
        }
    }
    timer_end(ctx, slot, ev);
    timer_rhs(ctx, slot, B);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

int launch_m2p(lspr_ctx *ctx, int prec, double *acc, int *counter, int B) {
    Tree &tr = ctx->tree;
    if (tr.n_m2p_items == 0) return LSPR_OK;
    cudaEvent_t ev;
    const int slot = slot_of(prec, T_M2P, T_M2P64, T_M2PFF);
    timer_begin(ctx, slot, &ev);
    ++ctx->n_launches;
    if (prec == PREC_F64) {
        LSPR_TRY_ST(m2p_orders_f64(ctx, acc, counter, B));
    } else if (prec == PREC_FF) {
        LSPR_TRY_ST(m2p_orders_ff(ctx, acc, counter, B));
    } else {
        LSPR_TRY_ST(m2p_orders_f32(ctx, acc, counter, B));
    }
    timer_end(ctx, slot, ev);
    timer_rhs(ctx, slot, B);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// Launchers on explicit buffers (no context-owned scratch), one right-hand side: used
// by the allocation-free matvec entry point.
int launch_weights_fp32_raw(cudaStream_t st, int64_t Ns, int64_t N, const dbl4 *spos64, const int *src_panel,
                            const double2 *x, float4 *w) {
    weights_kernel<float4><<<grid_for(Ns, 256), 256, 0, st>>>(Ns, N, 1, 1, spos64, src_panel, nullptr, x, nullptr, w, nullptr,
                                                               nullptr, ZeroRanges{});
    return cudaGetLastError() == cudaSuccess ? LSPR_OK : LSPR_E_CUDA;
}

int launch_p2p_fp32_raw(cudaStream_t st, const int4 *items, int64_t nitems, const float4 *tgt, int64_t ntgt,
                        const float4 *spos, const float4 *snrm, const float4 *w, double *acc) {
    if (nitems == 0) return LSPR_OK;
    p2p_kernel<float, 1, false><<<grid_for(nitems, p2p_warps(1)), p2p_warps(1) * 32, 0, st>>>(
        items, nitems, 1, 1, tgt, ntgt, spos, snrm, w, acc, nullptr, nullptr, 1);
    return cudaGetLastError() == cudaSuccess ? LSPR_OK : LSPR_E_CUDA;
}

}  // namespace lspr