// P2M and M2P launches of every compiled Taylor order, float-float arithmetic.
//
// The float-float M2P evaluates the same recurrence as the FP32/FP64 kernels,
//   n |R|^2 a_k + (2n-1) sum_d R_d a_(k-e_d) + (n-1) sum_d a_(k-2e_d) = 0,  a_0 = 1/|R|,
// but rolled: one code path serves every order P <= kMaxP, walking a table of the terms
// (degree-ordered, so the terms of order P are a prefix of the table) and keeping each
// lane's coefficients a_k in shared memory.  Fully unrolled, the float-float recurrence
// is ~10^4 instructions per (target, box) and overflows the instruction cache.
#include "farfield.cuh"

namespace lspr {

namespace {

// right-hand sides per float-float P2P work unit: 95.9 ms per 64-right-hand-side product on the
// 81920-panel sphere's tree (theta 0.4, P 7, Ncrit 512) against 120.6 ms for chunks of 4 and
// 281.6 ms for the two-targets-per-lane kernel with chunks of 2; chunks of 16 spill (162
// registers at 8 before the channels were packed)
constexpr int kFfP2PChunk = 8;

// one term k of the table: distances u - index(k - e_d) and u - index(k - 2 e_d) to the term's
// own index u (0: absent); and per degree the recurrence weight kappa_n as a float-float pair
struct FfTerm {
    unsigned char d1[3], d2[2];
    unsigned char pad[3];
};
struct FfTermTable {
    FfTerm t[n_terms(kMaxP)];
    float kh[kMaxP + 1], kl[kMaxP + 1];
};

constexpr FfTermTable make_ff_terms() {
    FfTermTable tab{};
    constexpr MultiIndex<kMaxP> mi{};
    for (int u = 0; u < n_terms(kMaxP); ++u)
        for (int d = 0; d < 3; ++d) {
            tab.t[u].d1[d] = (unsigned char)(mi.m1[u][d] >= 0 ? u - mi.m1[u][d] : 0);
            if (d < 2) tab.t[u].d2[d] = (unsigned char)(mi.m2[u][d] >= 0 ? u - mi.m2[u][d] : 0);   // k_3 <= 1
        }
    for (int n = 0; n <= kMaxP; ++n) {
        tab.kh[n] = (float)mi_kappa(n);
        tab.kl[n] = (float)(mi_kappa(n) - (double)(float)mi_kappa(n));
    }
    return tab;
}
static_assert(n_terms(kMaxP) - n_terms(kMaxP - 3) <= 255, "term distances must fit the table's bytes");

__constant__ FfTermTable c_ff_terms = make_ff_terms();

// The recurrence of a degree-n term reads terms of degrees n-1 and n-2 only, so each lane keeps
// its coefficients in a ring of W slots (term u in slot u mod W), W = the terms of the three
// highest degrees P-2, P-1, P (39 instead of 64 at P = 7): every term read is among the W
// written last.
__host__ __device__ inline int ff_ring(int P) {
    return P < 2 ? n_terms(P) : n_terms(P) - n_terms(P - 3);
}

// Shared memory of a block: one part (TP terms) of a box's staged moments for its chunk of
// right-hand sides (TP x NB, shared by the block's two warps) and each warp's coefficient ring
// (2 x W x 32)
__host__ __device__ inline size_t ff_m2p_smem(int TP, int W, int NB) {
    return (size_t)TP * NB * sizeof(ff4) + 2 * (size_t)W * 32 * sizeof(ffloat);
}

// a ff4 with its parts grouped for ff_mac2: (x.hi, y.hi, x.lo, y.lo), (z.hi, w.hi, z.lo, w.lo)
struct __align__(16) ff4p {
    float4 xy, zw;
};
__device__ __forceinline__ ff4p packed(const ff4 &m) {
    return {make_float4(m.x.hi, m.y.hi, m.x.lo, m.y.lo), make_float4(m.z.hi, m.w.hi, m.z.lo, m.w.lo)};
}
// the two channels of each layer of one right-hand side += f m
__device__ __forceinline__ void mac4(ff2 (&a)[2], float2 fh, float2 nfh, float2 fl, const ff4p &m) {
    ff_mac2(a[0], fh, nfh, fl, make_float2(m.xy.x, m.xy.y), make_float2(m.xy.z, m.xy.w));
    ff_mac2(a[1], fh, nfh, fl, make_float2(m.zw.x, m.zw.y), make_float2(m.zw.z, m.zw.w));
}
__device__ __forceinline__ double ff2_x(const ff2 &a) { return (double)a.hi.x + (double)a.lo.x; }
__device__ __forceinline__ double ff2_y(const ff2 &a) { return (double)a.hi.y + (double)a.lo.y; }

// One work unit for up to NB right-hand sides; see m2p_ff_kernel
template <int NB>
__device__ __forceinline__ void m2p_ff_unit(const int4 &item, int B, int b0, int nb, int um, int NT,
                                            const ff4 *__restrict__ tgt, int64_t ntgt, const int *__restrict__ list,
                                            const ff4 *__restrict__ box_c, const ff4 *__restrict__ mom,
                                            double *__restrict__ acc, int W, int TP,
                                            const int *__restrict__ box_surf, int S, ff4p *sm, ffloat *sa) {
    const int h = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ti = (int64_t)item.x * kTargetBlock + lane + 32 * h;
    const ff4 q = ti < ntgt ? tgt[ti] : tgt[0];
    ff2 a[NB][2];
#pragma unroll
    for (int j = 0; j < NB; ++j)
#pragma unroll
        for (int c = 0; c < 2; ++c) a[j][c].hi = a[j][c].lo = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int l = item.y; l < item.z; ++l) {
        const int b = __ldg(list + l);
        if (S > 1 && !(box_surf[b] & um)) continue;
        const ff4 c = box_c[b];
        // terms t0 .. t0 + TP - 1 of the box's moments into sm (the whole block, at the same t)
        auto stage = [&](int t0) {
            __syncthreads();   // the previous part's moments are no longer read
            const int nq = min(TP, NT - t0) * NB;
            for (int q2 = threadIdx.x; q2 < nq; q2 += 64) {
                const int t = q2 / NB, j = q2 - t * NB;
                sm[q2] = packed(j < nb ? mom[((int64_t)b * NT + t0 + t) * B + b0 + j] : zero4<ff4>());
            }
            __syncthreads();
        };
        stage(0);
        const ffloat d[3] = {q.x - c.x, q.y - c.y, q.z - c.z};
        const ffloat r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        const ffloat a0 = rsq(r2);
        const ffloat ir2 = a0 * a0;
        const ffloat R[3] = {d[0] * ir2, d[1] * ir2, d[2] * ir2};
        ffloat kap(0.f, 0.f);   // kappa_n / |R|^2 of the current degree n
        int n = 0, tn = 1;      // degree, first term of the next one
        sa[lane] = a0;
        int su = 0;      // slot of term t
        int tpart = 0;   // first term of the staged part
        {
            const float2 fh = both(a0.hi), nfh = both(-a0.hi), fl = both(a0.lo);
#pragma unroll
            for (int j = 0; j < NB; ++j) mac4(a[j], fh, nfh, fl, sm[j]);
        }
#pragma unroll 1
        for (int t = 1; t < NT; ++t) {
            if (t == tpart + TP) stage(tpart = t);
            if (t == tn) {
                ++n;
                tn = (n + 1) * (n + 1);
                kap = ffloat(c_ff_terms.kh[n], c_ff_terms.kl[n]) * ir2;
            }
            const FfTerm &e = c_ff_terms.t[t];
            su = su + 1 == W ? 0 : su + 1;
            ffloat at(0.f, 0.f);
            if (e.d2[0] | e.d2[1]) {
                ffloat s2(0.f, 0.f);
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    if (e.d2[x]) {
                        const int sl = su - e.d2[x];
                        s2 += sa[(sl < 0 ? sl + W : sl) * 32 + lane];
                    }
                at = kap * s2;
            }
#pragma unroll
            for (int x = 0; x < 3; ++x)
                if (e.d1[x]) {
                    const int sl = su - e.d1[x];
                    at += R[x] * sa[(sl < 0 ? sl + W : sl) * 32 + lane];
                }
            sa[su * 32 + lane] = at;
            const float2 fh = both(at.hi), nfh = both(-at.hi), fl = both(at.lo);
#pragma unroll
            for (int j = 0; j < NB; ++j) mac4(a[j], fh, nfh, fl, sm[(t - tpart) * NB + j]);
        }
    }
    if (ti < ntgt) {
        const int64_t tp = panel_of(q.w);
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (j < nb)
                atomic_add4(acc + 4 * (tp * B + b0 + j), ff2_x(a[j][0]), ff2_y(a[j][0]), ff2_x(a[j][1]),
                            ff2_y(a[j][1]));
    }
}

// Work units and accumulation as in m2p_kernel; NT = n_terms(P) at run time.  A block of two
// warps takes a unit: warp h the targets 32 h .. 32 h + 31 of the 64-target block, both on the
// same boxes, so each box's moments are staged once for the two, in parts of TP terms (the
// launcher picks TP so that more blocks fit per SM).  The recurrence is rolled (each lane's
// coefficients live in its column of the warp's ring), and the contraction accumulates with
// ff_mac2, the real and imaginary channel at once.  A unit takes the narrowest of NB, NB / 2 and
// NB / 4 that holds its right-hand sides (the contraction is 9/10 of the work).  Issue-bound.
// 40500 panels, 12 right-hand sides: 10.5 ms (11.7 with 12 operations per product, 15.0 with units of
// eight and scalar parts).
template <int NB>
__global__ void __launch_bounds__(64)
    m2p_ff_kernel(const int4 *__restrict__ items, int64_t nitems, int nbc, int B, int NT,
                  const ff4 *__restrict__ tgt, int64_t ntgt, const int *__restrict__ list,
                  const ff4 *__restrict__ box_c, const ff4 *__restrict__ mom, double *__restrict__ acc, int *counter,
                  const int *nact, int W, int TP, const int *__restrict__ box_surf, int S) {
    extern __shared__ __align__(16) unsigned char ff_smem[];
    __shared__ int64_t unit;
    ff4p *sm = (ff4p *)ff_smem;
    ffloat *sa = (ffloat *)(sm + TP * NB) + (size_t)(threadIdx.x >> 5) * W * 32;   // sa[(t mod W) * 32 + lane]
    const int Bact = nact ? *nact : B;   // right-hand sides in use (the first Bact slots)
    nbc = (Bact + NB - 1) / NB;
    const int64_t units = nitems * nbc;
    while (true) {
        if (threadIdx.x == 0) unit = atomicAdd(counter, 1);
        __syncthreads();
        const int64_t it = unit;
        __syncthreads();   // every thread has read the unit before thread 0 takes the next one
        if (it >= units) return;
        const int64_t ii = it / nbc;
        const int b0 = (int)(it - ii * nbc) * NB, nb = min(NB, Bact - b0);
        const int um = set_surfaces(b0, nb, Bact, S);
        const int4 item = __ldg(items + ii);
        if (NB < 4 || nb > NB / 2)
            m2p_ff_unit<NB>(item, B, b0, nb, um, NT, tgt, ntgt, list, box_c, mom, acc, W, TP, box_surf, S, sm, sa);
        else if (nb > NB / 4)
            m2p_ff_unit<(NB < 4 ? 1 : NB / 2)>(item, B, b0, nb, um, NT, tgt, ntgt, list, box_c, mom, acc, W, TP, box_surf, S,
                                              sm, sa);
        else
            m2p_ff_unit<(NB < 4 ? 1 : NB / 4)>(item, B, b0, nb, um, NT, tgt, ntgt, list, box_c, mom, acc, W, TP, box_surf, S,
                                              sm, sa);
    }
}

template <int NB>
int m2p_ff_launch(lspr_ctx *ctx, double *acc, int *counter, int B) {
    static int occ = 0, occ_nt = -1, tp_sel = 0;
    static int smem_set[kSmemDevices] = {};
    Tree &tr = ctx->tree;
    const int NT = n_terms(tr.P), W = ff_ring(tr.P);
    LSPR_TRY(ctx, allow_smem(m2p_ff_kernel<NB>, (int)ff_m2p_smem(NT, W, NB), ctx->device, smem_set));
    if (occ_nt != NT) {
        // the fewest parts (1 to 3) of a box's moments that give the most resident blocks per SM (P 7,
        // 8 right-hand sides: whole, 36 KB, which leaves room for the six blocks that the registers allow)
        occ = 0;
        tp_sel = NT;
        for (int parts = 1; parts <= 3; ++parts) {
            const int tp = (NT + parts - 1) / parts;
            int per_sm = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, m2p_ff_kernel<NB>, 64,
                                                              ff_m2p_smem(tp, W, NB)) != cudaSuccess) {
                (void)cudaGetLastError();
                per_sm = 0;
            }
            if (per_sm > occ) {
                occ = per_sm;
                tp_sel = tp;
            }
        }
        if (occ < 1) {
            occ = 1;
            tp_sel = NT;
        }
        occ_nt = NT;
    }
    const size_t smem = ff_m2p_smem(tp_sel, W, NB);
    const int nbc = (B + NB - 1) / NB;
    const unsigned grid =
        (unsigned)std::min<int64_t>(tr.n_m2p_items * nbc, (int64_t)occ * std::max(1, ctx->num_sms));
    m2p_ff_kernel<NB><<<grid, 64, smem, ctx->stream>>>(
        tr.m2p_items.p, tr.n_m2p_items, nbc, B, NT, Views<ffloat>::tgt(ctx), ctx->mesh.N, tr.m2p_list.p,
        Views<ffloat>::bc(ctx), Views<ffloat>::mom(ctx), acc, counter, ctx->rhs_nact, W, tp_sel, tr.box_surf.p,
        ctx->mesh.S);
    return LSPR_OK;
}

// Float-float P2P of several right-hand sides, one target per lane: a warp takes (item, half
// of its 64-target block, chunk of NB right-hand sides), so G and dG/dn of a pair (~170 FP32
// instructions in float-float) serve NB right-hand sides (4 ff_mac each) instead of the two of
// the two-targets-per-lane kernel.  Sources are staged per warp in chunks of 32 and read by
// broadcast; sums and the own-panel rule are those of p2p_kernel.
constexpr int kFfP2PWarps = 4;
template <int NBW, int NB>
__device__ __forceinline__ void p2p_ff1_unit(const int4 &item, int B, int b0, int nb, int64_t t,
                                             const ff4 *__restrict__ tgt, int64_t ntgt, const ff4 *__restrict__ spos,
                                             const ff4 *__restrict__ snrm, const ff4 *__restrict__ sw,
                                             double *__restrict__ acc, ff4 (*sh)[32], ff4p (*shw)[NB]) {
    const int lane = threadIdx.x & 31;
    const ff4 q = t < ntgt ? tgt[t] : tgt[0];
    const int tp = panel_of(q.w);
    ff2 a[NBW][2];
#pragma unroll
    for (int k = 0; k < NBW; ++k)
#pragma unroll
        for (int c = 0; c < 2; ++c) a[k][c].hi = a[k][c].lo = make_float2(0.f, 0.f);
    for (int base = item.y; base < item.z; base += 32) {
        const int s = base + lane;
        if (s < item.z) {
            sh[0][lane] = spos[s];
            sh[1][lane] = snrm[s];
#pragma unroll
            for (int k = 0; k < NBW; ++k)
                shw[lane][k] = packed(k < nb ? sw[(int64_t)s * B + b0 + k] : zero4<ff4>());
        }
        __syncwarp();
        const int cnt = min(32, item.z - base);
#pragma unroll 2
        for (int kk = 0; kk < cnt; ++kk) {
            const ff4 p = sh[0][kk], n = sh[1][kk];
            const ffloat dx = ff_diff(q.x, p.x), dy = ff_diff(q.y, p.y), dz = ff_diff(q.z, p.z);
            ffloat r = rsq(dx * dx + dy * dy + dz * dz);
            if ((item.w & 1) && panel_of(n.w) == tp) r = ffloat(0.f, 0.f);
            const ffloat tk = (dx * n.x + dy * n.y + dz * n.z) * (r * r) * r;
            const float2 rh = both(r.hi), nrh = both(-r.hi), rl = both(r.lo);
            const float2 th = both(tk.hi), nth = both(-tk.hi), tl = both(tk.lo);
#pragma unroll
            for (int k = 0; k < NBW; ++k) {
                const ff4p w = shw[kk][k];
                ff_mac2(a[k][0], rh, nrh, rl, make_float2(w.xy.x, w.xy.y), make_float2(w.xy.z, w.xy.w));
                ff_mac2(a[k][1], th, nth, tl, make_float2(w.zw.x, w.zw.y), make_float2(w.zw.z, w.zw.w));
            }
        }
        __syncwarp();
    }
    if (t < ntgt) {
#pragma unroll
        for (int k = 0; k < NBW; ++k)
            if (k < nb)
                atomic_add4(acc + 4 * ((int64_t)tp * B + b0 + k), ff2_x(a[k][0]), ff2_y(a[k][0]), ff2_x(a[k][1]),
                            ff2_y(a[k][1]));
    }
}

// 40500 panels, 12 right-hand sides: 7.1 ms (7.88 with 12 operations per product, 9.52 with units of eight
// and scalar parts).
template <int NB>
__global__ void __launch_bounds__(kFfP2PWarps * 32)
    p2p_ff1_kernel(const int4 *__restrict__ items, int64_t nitems, int B, const ff4 *__restrict__ tgt, int64_t ntgt,
                   const ff4 *__restrict__ spos, const ff4 *__restrict__ snrm, const ff4 *__restrict__ sw,
                   double *__restrict__ acc, int *counter, const int *nact, int S) {
    __shared__ ff4 sh[kFfP2PWarps][2][32];
    __shared__ ff4p shw[kFfP2PWarps][32][NB];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int Bact = nact ? *nact : B;
    const int nbc = (Bact + NB - 1) / NB;
    const int64_t units = nitems * 2 * nbc;
    while (true) {
        int v = 0;
        if (lane == 0) v = atomicAdd(counter, 1);
        const int64_t it = __shfl_sync(0xffffffffu, v, 0);
        if (it >= units) return;
        const int64_t ii = it / (2 * nbc);
        const int rem = (int)(it - ii * 2 * nbc), h = rem / nbc;
        const int b0 = (rem - h * nbc) * NB, nb = min(NB, Bact - b0);
        const int4 item = __ldg(items + ii);
        if (S > 1 && !((item.w >> kItemSurf) & set_surfaces(b0, nb, Bact, S))) continue;
        const int64_t t = (int64_t)item.x * kTargetBlock + 32 * h + lane;
        // the narrowest of NB and NB / 2 that holds the unit's right-hand sides
        if (nb > NB / 2)
            p2p_ff1_unit<NB, NB>(item, B, b0, nb, t, tgt, ntgt, spos, snrm, sw, acc, sh[warp], shw[warp]);
        else
            p2p_ff1_unit<NB / 2, NB>(item, B, b0, nb, t, tgt, ntgt, spos, snrm, sw, acc, sh[warp], shw[warp]);
    }
}

template <int NB>
int p2p_ff1_launch(lspr_ctx *ctx, const int4 *items, int64_t nitems, int B, double *acc, cudaStream_t st,
                   int *counter) {
    static int occ = 0;
    const int nbc = (B + NB - 1) / NB;
    const unsigned grid = std::min<unsigned>(grid_for(nitems * 2 * nbc, kFfP2PWarps),
                                             persistent_grid(ctx, p2p_ff1_kernel<NB>, kFfP2PWarps * 32, &occ));
    p2p_ff1_kernel<NB><<<grid, kFfP2PWarps * 32, 0, st>>>(items, nitems, B, Views<ffloat>::tgt(ctx), ctx->mesh.N,
                                                          Views<ffloat>::spos(ctx), Views<ffloat>::snrm(ctx),
                                                          Views<ffloat>::w(ctx), acc, counter, ctx->rhs_nact, ctx->mesh.S);
    return LSPR_OK;
}

}  // namespace

int p2p_ff_multi(lspr_ctx *ctx, const int4 *items, int64_t nitems, int B, double *acc, cudaStream_t st, int *counter) {
    return p2p_ff1_launch<kFfP2PChunk>(ctx, items, nitems, B, acc, st, counter);
}

int p2m_orders_ff(lspr_ctx *ctx, int B) {
    LSPR_DISPATCH_P(p2m_launch, ffloat, B, ctx, B);
    return LSPR_OK;
}

int m2p_orders_ff(lspr_ctx *ctx, double *acc, int *counter, int B) {
    if (ctx->tree.P < 1 || ctx->tree.P > kMaxP) return LSPR_E_ARG;
    // chunks of 8 right-hand sides: the recurrence is shared by more of them (24.8 / 29.5 / 28.5 ms
    // for chunks of 8 / 4 / 16 at 16 right-hand sides, 20480 panels, P = 7)
    return B == 1 ? m2p_ff_launch<1>(ctx, acc, counter, B) : m2p_ff_launch<8>(ctx, acc, counter, B);
}

}  // namespace lspr
