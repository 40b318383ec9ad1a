// Restarted GMRES(m) (Sec. II.D-E: complex GMRES) for B systems in lockstep.
//
// One Arnoldi cycle:
//   init        v_0 = r / beta, g = beta e_1
//   loop        (the body is one Arnoldi step; its last kernel decides, on the device,
//               whether another step follows)
//                 z = M^-1 v_j                      (v_j = w / ||w|| formed here, j > 0)
//                 w = A z                           (the far field, near SpMV and block rows)
//                 classical Gram-Schmidt h = V^H w, w -= V h, repeated once for the systems
//                 whose w lost more than a factor 1/sqrt(2) of its norm in the first pass
//                 (the Daniel-Gragg-Kaufman-Stewart criterion: one repetition restores
//                 orthogonality to working precision, and a pass that removes little
//                 needs none)
//                 ||w||, Givens rotation of the new Hessenberg column, residual
//                 estimate |g_{j+1}|, per-system stop test
//   back substitution R y = g, x += M^-1 V y
// The cycle is recorded once as a CUDA graph whose loop is a conditional WHILE node, so the
// host only takes part once per cycle (explicit residual and stop decision).  Without graphs
// (or with per-kernel timing) the host launches the same kernels itself and reads the loop
// condition after every step.  Inner products reduce over blocks with a last-block ticket
// instead of a second launch.
//
// Precision.  The Krylov basis, the Gram-Schmidt coefficients and the vector being
// orthogonalised are float-float (hi + lo FP32 pairs, ~48 significant bits): on this GPU the
// FP64 pipe runs at 1/64 of the FP32 rate, and the Gram-Schmidt passes (8 FP64 multiply-adds
// per basis entry and pass) would be bound by it at ~3x the time of reading the basis from
// memory.  In float-float they are bound by the basis traffic.  A basis entry takes 16 bytes
// as in FP64.  The rotations, the small triangular solve, norms' final sums, the residual and
// the solution stay FP64.
#include <algorithm>
#include <cmath>
#include <vector>

#include "cplx.cuh"
#include "ffloat.cuh"
#include "lspr_internal.cuh"

namespace lspr {
namespace {

constexpr int kT = 256;                 // threads per block of the vector kernels
constexpr double kReorthEta = 0.70710678118654752;   // second pass when ||w_1|| < eta ||w_0||
constexpr int kDotPart = 256;           // entries of a part of a chunk: a warp's task is four vectors on one part
constexpr int kAxpyPer = 2;             // entries per thread of the update
constexpr int kUpdChunk = 512;          // entries per block of the update with the second inner products

// one complex entry in float-float: re = rh + rl, im = ih + il
struct __align__(16) cff {
    float rh, ih, rl, il;
};
static_assert(sizeof(cff) == sizeof(float4), "a basis entry is one 16-byte word");

__device__ __forceinline__ cff to_cff(double2 v) {
    const float rh = (float)v.x, ih = (float)v.y;
    return {rh, ih, (float)(v.x - (double)rh), (float)(v.y - (double)ih)};
}
__device__ __forceinline__ double2 to_d2(const cff &v) {
    return make_double2((double)v.rh + (double)v.rl, (double)v.ih + (double)v.il);
}
__device__ __forceinline__ ffloat re_of(const cff &v) { return ffloat(v.rh, v.rl); }
__device__ __forceinline__ ffloat im_of(const cff &v) { return ffloat(v.ih, v.il); }

// hi + lo renormalised (|lo| <= ulp(hi)/2) after unnormalised accumulation
__device__ __forceinline__ ffloat ff_norm(const ffloat &x) {
    ffloat r;
    ff_two_sum(x.hi, x.lo, r.hi, r.lo);
    return r;
}
__device__ __forceinline__ cff pack(const ffloat &re, const ffloat &im) {
    const ffloat r = ff_norm(re), i = ff_norm(im);
    return {r.hi, i.hi, r.lo, i.lo};
}

// Packed products of a complex factor f with v: a += f_re (v_re, v_im), b += f_im (v_re, v_im), so that
// f v = (a.x - b.y, a.y + b.x) and f conj(v) = (a.x + b.y, b.x - a.y).  f's parts come in both halves of
// a pair, the leading ones with their negatives (ff_mac2).
struct CPair {
    ff2 a, b;
};
struct __align__(16) CFactor {
    float2 rh, nrh, rl, ih, nih, il;
};
__device__ __forceinline__ CFactor factor(const cff &f) {
    return {both(f.rh), both(-f.rh), both(f.rl), both(f.ih), both(-f.ih), both(f.il)};
}
__device__ __forceinline__ void cff_mac2(CPair &p, const CFactor &f, const float4 &v) {
    const float2 vh = make_float2(v.x, v.y), vl = make_float2(v.z, v.w);
    ff_mac2(p.a, f.rh, f.nrh, f.rl, vh, vl);
    ff_mac2(p.b, f.ih, f.nih, f.il, vh, vl);
}
// (ar, ai) += v h
__device__ __forceinline__ void cff_mac(ffloat &ar, ffloat &ai, const cff &v, const cff &h) {
    const ffloat vr = re_of(v), vi = im_of(v);
    const ffloat hr = re_of(h), hi = im_of(h);
    ff_mac(ar, vr, hr);
    ff_mac(ar, -vi, hi);
    ff_mac(ai, vr, hi);
    ff_mac(ai, vi, hr);
}
// |v|^2 added to s
__device__ __forceinline__ void cff_abs2_mac(ffloat &s, const ffloat &re, const ffloat &im) {
    ff_mac(s, re, re);
    ff_mac(s, im, im);
}

struct Arn {
    int B, m, nch, nblk, chunk;   // chunk: entries per inner-product block, nch of them
    int64_t N, n2, vstride;
    cff *V;              // [B][m+1][2N] Krylov basis
    double2 *w;          // [B][2N] A z (FP64 from the operator; float-float in place once the
                         // first Gram-Schmidt pass has read it)
    double2 *z, *x;
    const double2 *b, *s;
    const double *vinv;  // [N] 1 / V_ii (preconditioner)
    const double2 *pq;   // [B][S] 1 / (1 + s) (preconditioner)
    const ffloat *vinvf; // [N] the same three in float-float: 1 / V_ii,
    const cff *pqf, *sf; // [B] 1 / (1 + s), s (one surface)
    float2 *xtf;         // [2N][B] preconditioned vectors in FP32 (null: z)
    const int *surf;     // surface of each panel; s is [B][S]
    int S;
    double2 *h, *hcol, *part, *H, *sn, *g, *y;
    cff *hff, *yff;      // [B][m+1] Gram-Schmidt coefficients, [B][m] update coefficients
    ffloat *ninv;        // [B] 1 / ||w||
    double *npart, *nrm, *cs, *res, *npart0;
    int *reorth;
    const double *bn, *par;
    unsigned *tick;      // [2B + 1] last-block tickets
    int *jdev, *active, *jb, *iters;
    int *rmap;   // [2B + 2]: slot -> system, system -> slot (-1: not running), running count,
                 // channel sets in use (running count x surfaces)
    int *go;     // host-driven cycles: the loop condition (nullptr inside a graph)
    unsigned long long *stats;   // [4] sum (j+1), system-steps, the same over second passes
    cudaGraphConditionalHandle cond;
};

__device__ __forceinline__ cff *wff(const Arn &a, int b) { return (cff *)(a.w + (int64_t)b * a.n2); }

// packs the running systems into the first slots (one whole warp); returns their number
__device__ __forceinline__ int pack_running(const Arn &a) {
    const int lane = threadIdx.x & 31;
    int n = 0;
    for (int b0 = 0; b0 < a.B; b0 += 32) {
        const int b = b0 + lane;
        const bool on = b < a.B && __ldcg(a.active + b);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        const int slot = n + __popc(m & ((1u << lane) - 1));
        if (on) a.rmap[slot] = b;
        if (b < a.B) a.rmap[a.B + b] = on ? slot : -1;
        n += __popc(m);
    }
    for (int q = n + lane; q < a.B; q += 32) a.rmap[q] = 0;
    if (lane == 0) {
        a.rmap[2 * a.B] = n;
        a.rmap[2 * a.B + 1] = n * a.S;
    }
    return n;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double2 warp_sum2(double2 v) { return make_double2(warp_sum(v.x), warp_sum(v.y)); }

__device__ __forceinline__ ffloat shfl_xor(const ffloat &v, int o) {
    return ffloat(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
__device__ __forceinline__ ffloat ff_warp_sum(ffloat v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = v + shfl_xor(v, o);
    return v;
}

// sum over a block of kT threads, valid in warp 0
__device__ __forceinline__ double block_sum(double v, double *sh) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) t = warp_sum(threadIdx.x < kT / 32 ? sh[threadIdx.x] : 0.0);
    return t;
}
// float-float partial sums of a block: warps reduce in float-float, warp 0 sums the kT/32
// warp results in FP64 (valid in thread 0)
__device__ __forceinline__ double block_sum_ff(const ffloat &v, double *sh) {
    const ffloat s = ff_warp_sum(ff_norm(v));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = (double)s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int q = 0; q < kT / 32; ++q) t += sh[q];
    return t;
}

// true in every thread of the block that arrives last among `count` blocks on ticket *t
// (the partial results written before the call are visible to it)
__device__ __forceinline__ bool last_block(unsigned *t, unsigned count) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(t, 1u) == count - 1;
    __syncthreads();
    return last;
}

// final sum of the squared-norm partials of system b into nrm[b] and 1/nrm[b] (last block
// only); decide: the first Gram-Schmidt pass decides whether the second runs
__device__ __forceinline__ void norm_final(const Arn &a, int b, int nblk, double *sh) {
    double t = 0.0;
    for (int c = threadIdx.x; c < nblk; c += kT) t += __ldcg(a.npart + (int64_t)b * a.nblk + c);
    t = block_sum(t, sh);
    if (threadIdx.x == 0) {
        const double r = sqrt(t);
        a.nrm[b] = r;
        a.ninv[b] = ffloat(r > 0 ? 1.0 / r : 0.0);
        a.tick[a.B + b] = 0;
    }
}

// Right preconditioner of panel i (inverse of the diagonal 2x2 block of the operator,
// [[1/2 + K_ii, -V_ii], [1/2 - K_ii, s V_ii]] with K_ii = 0):
//   o0 = 2 (s u0 + u1) / (1 + s),  o1 = (u1 - u0) / (V_ii (1 + s))
// with pq = 1 / (1 + s) and vinv = 1 / V_ii formed once per solve (no division per entry)
__device__ __forceinline__ void precond(double vinv, double2 q, double2 s, double2 u0, double2 u1, double2 &o0,
                                        double2 &o1) {
    o0 = cscale(cmul(q, cadd(cmul(s, u0), u1)), 2.0);
    o1 = cscale(cmul(q, csub(u1, u0)), vinv);
}

// w = A x - b (w holds A x on entry; x_zero: x = 0 and w = -b), nrm[b] = ||w||
__global__ void __launch_bounds__(kT) arn_resid_kernel(Arn a, int x_zero) {
    __shared__ double sh[kT / 32];
    const int b = blockIdx.y;
    const int64_t k = blockIdx.x * (int64_t)kT + threadIdx.x;
    double q = 0.0;
    if (k < a.n2) {
        const int64_t o = (int64_t)b * a.n2 + k;
        const double2 bb = a.b[o];
        const double2 v = x_zero ? make_double2(-bb.x, -bb.y) : csub(a.w[o], bb);
        a.w[o] = v;
        q = cabs2(v);
    }
    q = block_sum(q, sh);
    if (threadIdx.x == 0) a.npart[(int64_t)b * a.nblk + blockIdx.x] = q;
    if (last_block(a.tick + a.B + b, a.nblk)) norm_final(a, b, a.nblk, sh);
}

// v_0 = -w / beta for the running systems (w = A x - b); cycle state reset
__global__ void __launch_bounds__(kT) arn_init_kernel(Arn a) {
    const int b = blockIdx.y;
    const int64_t k = blockIdx.x * (int64_t)kT + threadIdx.x;
    const bool act = a.active[b] != 0;
    if (act && k < a.n2) a.V[(int64_t)b * a.vstride + k] = to_cff(cscale(a.w[(int64_t)b * a.n2 + k], -1.0 / a.nrm[b]));
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i <= a.m; i += kT)
            a.g[(int64_t)b * (a.m + 1) + i] = make_double2(i == 0 && act ? a.nrm[b] : 0.0, 0.0);
        if (threadIdx.x == 0) {
            a.jb[b] = 0;
            a.tick[b] = 0;
            a.tick[a.B + b] = 0;
            if (b == 0) {
                *a.jdev = 0;
                a.tick[2 * a.B] = 0;
            }
        }
        if (b == 0 && threadIdx.x < 32) pack_running(a);
    }
}

// v_j = w / ||w|| (j > 0, w float-float; v_0 comes from the init kernel), z = M^-1 v_j
__global__ void __launch_bounds__(kT) arn_precond_kernel(Arn a) {
    const int b = blockIdx.y;
    const int64_t t = blockIdx.x * (int64_t)kT + threadIdx.x;
    if (t >= a.N || !a.active[b]) return;
    const int j = *a.jdev;
    cff *Vj = a.V + (int64_t)b * a.vstride + (int64_t)j * a.n2;
    cff v0, v1;
    if (j == 0) {
        v0 = Vj[t];
        v1 = Vj[a.N + t];
    } else {
        const ffloat inv = a.ninv[b];
        const cff *wb = wff(a, b);
        const cff w0 = wb[t], w1 = wb[a.N + t];
        v0 = pack(re_of(w0) * inv, im_of(w0) * inv);
        v1 = pack(re_of(w1) * inv, im_of(w1) * inv);
        Vj[t] = v0;
        Vj[a.N + t] = v1;
    }
    double2 o0, o1;
    precond(a.vinv[t], a.pq[b * a.S + a.surf[t]], a.s[b * a.S + a.surf[t]], to_d2(v0), to_d2(v1), o0, o1);
    a.z[(int64_t)b * a.n2 + t] = o0;
    a.z[(int64_t)b * a.n2 + a.N + t] = o1;
}

// The same for FP32 products of several right-hand sides (one surface), which read their vectors
// transposed and in FP32: formed in float-float (the FP64 form above is bound by the FP64 pipe,
// some 34 operations per panel) and written transposed, 32 panels x 32 systems per block, instead of
// going through z and a transposing kernel.  20480 panels, 16 systems: solve 64.6 -> 63.4 ms; 81920
// panels, 64: 976 -> 948.
__global__ void __launch_bounds__(256) arn_precond_t_kernel(Arn a) {
    __shared__ float2 tile[2][32][33];
    const int64_t t0 = (int64_t)blockIdx.x * 32;
    const int b0 = blockIdx.y * 32, tx = threadIdx.x;
    const int j = *a.jdev;
    const int64_t t = t0 + tx;
    const ffloat vi = t < a.N ? a.vinvf[t] : ffloat(0.f, 0.f);
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int b = b0 + r;
        if (b >= a.B || t >= a.N || !a.active[b]) continue;
        cff *Vj = a.V + (int64_t)b * a.vstride + (int64_t)j * a.n2;
        cff v0, v1;
        if (j == 0) {
            v0 = Vj[t];
            v1 = Vj[a.N + t];
        } else {
            const ffloat inv = a.ninv[b];
            const cff *wb = wff(a, b);
            const cff w0 = wb[t], w1 = wb[a.N + t];
            v0 = pack(re_of(w0) * inv, im_of(w0) * inv);
            v1 = pack(re_of(w1) * inv, im_of(w1) * inv);
            Vj[t] = v0;
            Vj[a.N + t] = v1;
        }
        const cff s = a.sf[b], q = a.pqf[b];
        ffloat cr = re_of(v1), ci = im_of(v1), r0(0.f, 0.f), i0(0.f, 0.f), r1(0.f, 0.f), i1(0.f, 0.f);
        cff_mac(cr, ci, v0, s);   // s u0 + u1
        cff_mac(r0, i0, pack(cr, ci), q);
        cff_mac(r1, i1, pack(re_of(v1) - re_of(v0), im_of(v1) - im_of(v0)), q);
        tile[0][r][tx] = make_float2(2.f * ff_norm(r0).hi, 2.f * ff_norm(i0).hi);
        tile[1][r][tx] = make_float2((ff_norm(r1) * vi).hi, (ff_norm(i1) * vi).hi);
    }
    __syncthreads();
    const int b = b0 + tx;
    if (b >= a.B || !a.active[b]) return;
    for (int r = threadIdx.y; r < 32 && t0 + r < a.N; r += 8) {
        a.xtf[(t0 + r) * a.B + b] = tile[0][tx][r];
        a.xtf[(a.N + t0 + r) * a.B + b] = tile[1][tx][r];
    }
}

// Inner products of a Gram-Schmidt pass, h_i = <v_i, w> for i <= j.  A block takes a chunk of CH
// entries of one system: its threads stage the chunk of w in shared memory, then a warp takes
// tasks of four basis vectors on a part of the chunk, so that an entry of w read from shared
// memory serves four products and eight or sixteen loads per lane are in flight.  The 8 sums of a
// task are reduced over the warp by halves (9 exchanges instead of 40).  The last block of the
// system sums the chunks into h (FP64 and float-float) and into the Hessenberg column (hcol = h on
// pass 0, hcol += h on pass 1).
//   pass 0 converts w to float-float in place and forms ||w||^2; its last block decides from
//     ||w||^2 - ||h||^2, the squared norm left, whether the second pass runs (reorth[b]).
//   pass 1 (UPDATE) first does the update w -= sum_i v_i h_i of pass 0 on its chunk, for every
//     system; the second inner products then find the chunk of the basis in the L2 (512 entries:
//     some 50 MB over the blocks in flight at 20 vectors), so that the basis is read three times
//     from memory per step instead of four (vector kernels of a solve, 81920 panels, 64 systems: 194 ->
//     175 ms; 20480, 16: 14.1 -> 12.3).  A system without a second pass stops at its norm.
// 20480 panels, 16 systems, mid-cycle, cold caches: 51 us for pass 0 (81 with one vector per warp,
// chunks of 2048 and unpacked products, whose 320 blocks left SMs idle).
constexpr int kDotVec = 4;
// 2048 entries per block (one reduction over the warp per 16 entries of a lane) where that gives every SM
// eight blocks, else 1024.  81920 panels, 64 systems: vector kernels of a solve 195 ms, 201 with 1024
// throughout; 20480 panels, 16 systems: 14.3 ms with 1024, 14.7 with 2048.
inline int dot_chunk(int64_t n2, int B, int num_sms) {
    return (n2 + 2047) / 2048 * B >= 8 * (int64_t)num_sms ? 2048 : 1024;
}
inline size_t dot_smem(int chunk, int m, bool update) {   // w, the sums of the parts, the update's coefficients
    return chunk * sizeof(cff) + (size_t)(m + 1) * (chunk / kDotPart * sizeof(double2) + (update ? sizeof(CFactor) : 0));
}
template <int NV, int U>
__device__ __forceinline__ void dot_task(const cff *__restrict__ v, int64_t stride, const cff *ws, int e0, int len,
                                         double2 *red) {
    const int lane = threadIdx.x & 31;
    CPair p[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k)
        p[k].a.hi = p[k].a.lo = p[k].b.hi = p[k].b.lo = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int e = e0 + lane; e < e0 + kDotPart; e += 32 * U) {
        float4 x[U][NV];   // entries loaded together
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < NV; ++k)
                x[u][k] = e + 32 * u < len ? __ldg((const float4 *)(v + k * stride + e + 32 * u))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const CFactor f = factor(ws[e + 32 * u]);
#pragma unroll
            for (int k = 0; k < NV; ++k) cff_mac2(p[k], f, x[u][k]);
        }
    }
    // w conj(v): (a.x + b.y, b.x - a.y)
    ffloat t[2 * NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        t[2 * k] = ff_norm(ffloat(p[k].a.hi.x, p[k].a.lo.x)) + ff_norm(ffloat(p[k].b.hi.y, p[k].b.lo.y));
        t[2 * k + 1] = ff_norm(ffloat(p[k].b.hi.x, p[k].b.lo.x)) - ff_norm(ffloat(p[k].a.hi.y, p[k].a.lo.y));
    }
    if (NV == 4) {   // each exchange halves the values a lane holds: lanes with the same lane >> 2 end with one
#pragma unroll
        for (int o = 16, n = NV; o >= 4; o >>= 1, n >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int q = 0; q < n; ++q) {
                const ffloat send = up ? t[q] : t[q + n], keep = up ? t[q + n] : t[q];
                t[q] = keep + shfl_xor(send, o);
            }
        }
        ffloat s = t[0] + shfl_xor(t[0], 2);
        s = s + shfl_xor(s, 1);
        if ((lane & 3) == 0) {   // value 4 (bit 4) + 2 (bit 3) + (bit 2) of the lane
            const int q = ((lane & 16) >> 2) | ((lane & 8) >> 2) | ((lane & 4) >> 2);
            ((double *)red)[q] = (double)s;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 2 * NV; ++q) {
            const ffloat s = ff_warp_sum(t[q]);
            if (lane == 0) ((double *)red)[q] = (double)s;
        }
    }
}

// this thread's entries k0 + u kT of w -= sum_{i < nv} v_i h_i (hs: -h), those below n; f(u, entry) takes
// the results (an entry past the end reads the basis at the last one, and is dropped by f)
template <class F>
__device__ __forceinline__ void update_w(const cff *__restrict__ Vb, const cff *wb, int64_t n2, int nv,
                                         const CFactor *hs, int64_t k0, int64_t n, F &&f) {
    CPair p[kAxpyPer];
    int64_t k[kAxpyPer];
#pragma unroll
    for (int u = 0; u < kAxpyPer; ++u) {
        const bool on = k0 + u * kT < n;
        k[u] = on ? k0 + u * kT : n - 1;
        const cff w0 = on ? wb[k[u]] : cff{0.f, 0.f, 0.f, 0.f};
        p[u].a.hi = make_float2(w0.rh, w0.ih);
        p[u].a.lo = make_float2(w0.rl, w0.il);
        p[u].b.hi = p[u].b.lo = make_float2(0.f, 0.f);
    }
#pragma unroll 4
    for (int i = 0; i < nv; ++i) {
        const CFactor h = hs[i];
#pragma unroll
        for (int u = 0; u < kAxpyPer; ++u) cff_mac2(p[u], h, *(const float4 *)(Vb + (int64_t)i * n2 + k[u]));
    }
    // w - h v: (a.x - b.y, a.y + b.x)
#pragma unroll
    for (int u = 0; u < kAxpyPer; ++u)
        f(u, pack(ff_norm(ffloat(p[u].a.hi.x, p[u].a.lo.x)) - ff_norm(ffloat(p[u].b.hi.y, p[u].b.lo.y)),
                  ff_norm(ffloat(p[u].a.hi.y, p[u].a.lo.y)) + ff_norm(ffloat(p[u].b.hi.x, p[u].b.lo.x))));
}
__device__ __forceinline__ void load_factors(const Arn &a, int b, int nv, CFactor *hs) {
    for (int i = threadIdx.x; i < nv; i += kT) {
        const cff h = a.hff[(int64_t)b * (a.m + 1) + i];
        hs[i] = factor({-h.rh, -h.ih, -h.rl, -h.il});
    }
}

template <int CH, bool UPDATE>
__global__ void __launch_bounds__(kT, 2) arn_dot_kernel(Arn a) {
    static_assert(CH % (kT * kAxpyPer) == 0 && CH % kDotPart == 0, "whole tasks");
    constexpr int kSub = CH / kDotPart;
    extern __shared__ double2 dsm[];
    cff *ws = (cff *)dsm;
    double2 *red = dsm + CH;   // [kSub][m + 1]
    CFactor *hs = (CFactor *)(red + kSub * (a.m + 1));
    __shared__ double shn[kT / 32];
    const int b = blockIdx.y, chunk = blockIdx.x, nch = gridDim.x;
    if (!a.active[b]) return;
    const int nv = *a.jdev + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c0 = (int64_t)chunk * CH;
    const int len = (int)min((int64_t)CH, a.n2 - c0);
    cff *wb = wff(a, b) + c0;
    const cff *Vb = a.V + (int64_t)b * a.vstride + c0;
    ffloat w2(0.f, 0.f);
    if (UPDATE) {
        load_factors(a, b, nv, hs);
        __syncthreads();
        for (int e0 = threadIdx.x; e0 < CH; e0 += kT * kAxpyPer) {
            update_w(Vb, wb, a.n2, nv, hs, e0, len, [&](int u, cff v) {
                const int e = e0 + u * kT;
                if (e < len) {
                    wb[e] = v;
                    cff_abs2_mac(w2, re_of(v), im_of(v));
                } else {
                    v = {0.f, 0.f, 0.f, 0.f};
                }
                ws[e] = v;
            });
        }
        __syncthreads();
        if (!a.reorth[b]) {   // one pass is enough: its norm
            const double t = block_sum_ff(w2, shn);
            if (threadIdx.x == 0) a.npart[(int64_t)b * a.nblk + chunk] = t;
            if (last_block(a.tick + a.B + b, nch)) norm_final(a, b, nch, shn);
            return;
        }
    } else {
        for (int e = threadIdx.x; e < CH; e += kT) {
            cff v = {0.f, 0.f, 0.f, 0.f};
            if (e < len) {
                v = to_cff(a.w[(int64_t)b * a.n2 + c0 + e]);
                wb[e] = v;
            }
            ws[e] = v;
            cff_abs2_mac(w2, re_of(v), im_of(v));
        }
        // ||A z||^2 of this chunk, for the second-pass criterion
        const double t = block_sum_ff(w2, shn);
        if (threadIdx.x == 0) a.npart0[(int64_t)b * nch + chunk] = t;
        __syncthreads();
    }
    constexpr int kU = CH == 2048 ? 4 : 2;
    const int tasks = kSub * ((nv + kDotVec - 1) / kDotVec);
    for (int q = warp; q < tasks; q += kT / 32) {
        const int sub = q % kSub, i = q / kSub * kDotVec;
        const cff *v = Vb + (int64_t)i * a.n2;
        double2 *r = red + sub * (a.m + 1) + i;
        switch (min(kDotVec, nv - i)) {
            case 4: dot_task<4, kU>(v, a.n2, ws, sub * kDotPart, len, r); break;
            case 3: dot_task<3, kU>(v, a.n2, ws, sub * kDotPart, len, r); break;
            case 2: dot_task<2, kU>(v, a.n2, ws, sub * kDotPart, len, r); break;
            default: dot_task<1, kU>(v, a.n2, ws, sub * kDotPart, len, r); break;
        }
    }
    __syncthreads();
    double2 *pb = a.part + (int64_t)b * (a.m + 1) * nch;
    for (int i = threadIdx.x; i < nv; i += kT) {
        double2 t = red[i];
#pragma unroll
        for (int s = 1; s < kSub; ++s) t = cadd(t, red[s * (a.m + 1) + i]);
        pb[(int64_t)i * nch + chunk] = t;
    }
    if (!last_block(a.tick + b, nch)) return;
    double n0 = 0.0, hh = 0.0;   // ||A z||^2 (thread 0), this warp's share of ||h||^2 (lane 0)
    if (!UPDATE) {
        for (int c = threadIdx.x; c < nch; c += kT) n0 += __ldcg(a.npart0 + (int64_t)b * nch + c);
        n0 = block_sum(n0, shn);
    }
    // rows i = warp + 8 u: lanes stride over the chunks
    for (int i0 = warp; i0 < nv; i0 += 4 * (kT / 32)) {
        double2 t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            t[u] = make_double2(0.0, 0.0);
            const int i = i0 + u * (kT / 32);
            if (i < nv)
                for (int c = lane; c < nch; c += 32) t[u] = cadd(t[u], __ldcg(pb + (int64_t)i * nch + c));
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * (kT / 32);
            const double2 sum = warp_sum2(t[u]);
            if (lane == 0 && i < nv) {
                a.h[(int64_t)b * (a.m + 1) + i] = sum;
                a.hff[(int64_t)b * (a.m + 1) + i] = to_cff(sum);
                double2 &e = a.hcol[(int64_t)b * (a.m + 1) + i];
                e = UPDATE ? cadd(e, sum) : sum;
                hh += cabs2(sum);
            }
        }
    }
    if (!UPDATE) {
        __syncthreads();   // shn has been read
        if (lane == 0) shn[warp] = hh;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < kT / 32; ++q) hh += shn[q];
            a.reorth[b] = !(n0 - hh >= kReorthEta * kReorthEta * n0);
        }
    }
    if (threadIdx.x == 0) a.tick[b] = 0;
}

// The second pass's update w -= sum_{i <= j} v_i h_i, then ||w|| into nrm[b] (partials per block, the
// last block sums them)
__global__ void __launch_bounds__(kT) arn_axpy_kernel(Arn a) {
    __shared__ double sh[kT / 32];
    __shared__ CFactor hs[kMaxRestart + 1];
    const int b = blockIdx.y;
    if (!a.active[b] || !a.reorth[b]) return;
    const int nv = *a.jdev + 1;
    load_factors(a, b, nv, hs);
    __syncthreads();
    const int64_t k0 = blockIdx.x * (int64_t)(kT * kAxpyPer) + threadIdx.x;
    cff *wb = wff(a, b);
    ffloat q(0.f, 0.f);
    update_w(a.V + (int64_t)b * a.vstride, wb, a.n2, nv, hs, k0, a.n2, [&](int u, const cff &w1) {
        if (k0 + u * kT >= a.n2) return;
        wb[k0 + u * kT] = w1;
        cff_abs2_mac(q, re_of(w1), im_of(w1));
    });
    const double t = block_sum_ff(q, sh);
    if (threadIdx.x == 0) a.npart[(int64_t)b * a.nblk + blockIdx.x] = t;
    if (last_block(a.tick + a.B + b, gridDim.x)) norm_final(a, b, gridDim.x, sh);
}

// shared memory of the rotation kernel: column (m+1), sines (m), cosines (m)
inline size_t tail_smem(int m) { return (size_t)(3 * m + 1) * sizeof(double2); }

// End of an Arnoldi step, one warp (and block) per system: the new Hessenberg column (hcol, ||w||)
// is rotated by the previous Givens rotations, a new rotation zeroes its subdiagonal,
// g is rotated, |g_{j+1}| is the residual estimate and decides whether the system keeps
// running.  The last block then advances j and sets the loop condition (the graph's, or the flag
// the host reads): another step runs while a system is running and j < m.
// An FP64 instruction of a single lane holds the SM's FP64 pipe as long as one of 32, so the systems'
// warps are spread over SMs and the rotations composed by a scan.  16 systems, 30 rotations: 31 us with
// the systems on 16 warps of one block, 18 spread, less with the scan.
__global__ void __launch_bounds__(32) arn_tail_kernel(Arn a) {
    extern __shared__ double2 dsm[];
    const int lane = threadIdx.x, b = blockIdx.x;
    const int m = a.m, j = *a.jdev;
    if (__ldcg(a.active + b)) {
        double2 *col = dsm, *snw = col + m + 1, *csw = snw + m;
        const double2 *hc = a.hcol + (int64_t)b * (m + 1);
        for (int i = lane; i <= j; i += 32) col[i] = hc[i];
        for (int i = lane; i < j; i += 32) {
            snw[i] = a.sn[(int64_t)b * m + i];
            csw[i] = make_double2(a.cs[(int64_t)b * m + i], 0.0);
        }
        __syncwarp();
        // The previous rotations carry row i + 1: a_0 = col_0, row i gets c a_i + s d, d = col_(i+1), and
        // a_(i+1) = c d - conj(s) a_i.  Each is an affine map of a_i, so a scan over the lanes composes 32
        // of them in five steps (the factors conj(s) are at most 1 in magnitude).
        double2 *Hb = a.H + (int64_t)b * (m + 1) * m;
        double2 a0 = col[0];
        for (int i0 = 0; i0 < j; i0 += 32) {
            const int i = i0 + lane;
            const bool on = i < j;
            const double c = on ? csw[i].x : 0.0;
            const double2 sg = on ? snw[i] : make_double2(0.0, 0.0), d0 = on ? col[i + 1] : make_double2(0.0, 0.0);
            double2 A = on ? make_double2(-sg.x, sg.y) : make_double2(1.0, 0.0), Bc = cscale(d0, c);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {   // maps composed with those of the lanes before
                const double2 pA = make_double2(__shfl_up_sync(0xffffffffu, A.x, o), __shfl_up_sync(0xffffffffu, A.y, o));
                const double2 pB = make_double2(__shfl_up_sync(0xffffffffu, Bc.x, o), __shfl_up_sync(0xffffffffu, Bc.y, o));
                if (lane >= o) {
                    Bc = cadd(Bc, cmul(A, pB));
                    A = cmul(A, pA);
                }
            }
            const double2 nx = cadd(Bc, cmul(A, a0));   // a_(i+1)
            double2 ai = make_double2(__shfl_up_sync(0xffffffffu, nx.x, 1), __shfl_up_sync(0xffffffffu, nx.y, 1));
            if (lane == 0) ai = a0;
            if (on) Hb[(int64_t)i * m + j] = cadd(cscale(ai, c), cmul(sg, d0));
            a0 = make_double2(__shfl_sync(0xffffffffu, nx.x, 31), __shfl_sync(0xffffffffu, nx.y, 31));
        }
        if (lane == 0) {
            const double hn = a.nrm[b];   // subdiagonal entry ||w||, real
            const double aa = sqrt(cabs2(a0)), t = sqrt(aa * aa + hn * hn);
            double c;
            double2 sg;
            if (aa == 0.0) {
                c = 0.0;
                sg = make_double2(1.0, 0.0);
            } else {
                c = aa / t;
                sg = cscale(a0, hn / (aa * t));
            }
            Hb[(int64_t)j * m + j] = cadd(cscale(a0, c), cscale(sg, hn));
            a.cs[(int64_t)b * m + j] = c;
            a.sn[(int64_t)b * m + j] = sg;
            double2 *gb = a.g + (int64_t)b * (m + 1);
            const double2 gj = gb[j];
            gb[j + 1] = cmul(make_double2(-sg.x, sg.y), gj);   // -conj(s) g_j
            gb[j] = cscale(gj, c);
            const double r = sqrt(cabs2(gb[j + 1]));
            a.res[b] = r;
            a.jb[b] = j + 1;
            atomicAdd(a.stats + 0, (unsigned long long)(j + 1));
            atomicAdd(a.stats + 1, 1ull);
            if (a.reorth[b]) {
                atomicAdd(a.stats + 2, (unsigned long long)(j + 1));
                atomicAdd(a.stats + 3, 1ull);
            }
            const int it = ++a.iters[b];
            a.active[b] = (r / a.bn[b] > a.par[0]) && it < (int)a.par[1] && isfinite(r);
        }
    }
    if (!last_block(a.tick + 2 * a.B, gridDim.x)) return;
    const int n = pack_running(a);
    if (lane == 0) {
        a.tick[2 * a.B] = 0;
        *a.jdev = j + 1;
        const unsigned more = (n && j + 1 < m) ? 1u : 0u;
        if (a.go)
            *a.go = (int)more;
        else
            cudaGraphSetConditional(a.cond, more);
    }
}

// R y = g by back substitution (one warp and block per system), y into a.y (FP64) and a.yff
__global__ void __launch_bounds__(32) arn_backsub_kernel(Arn a) {
    extern __shared__ double2 ys[];
    const int lane = threadIdx.x, b = blockIdx.x;
    const int m = a.m, n = a.jb[b];
    const double2 *Hb = a.H + (int64_t)b * (m + 1) * m, *gb = a.g + (int64_t)b * (m + 1);
    for (int i = n - 1; i >= 0; --i) {
        double2 s = make_double2(0.0, 0.0);
        for (int k = i + 1 + lane; k < n; k += 32) s = cadd(s, cmul(Hb[(int64_t)i * m + k], ys[k]));
        s = warp_sum2(s);
        if (lane == 0) ys[i] = cdiv(csub(gb[i], s), Hb[(int64_t)i * m + i]);
        __syncwarp();
    }
    for (int i = lane; i < n; i += 32) {
        a.y[(int64_t)b * m + i] = ys[i];
        a.yff[(int64_t)b * m + i] = to_cff(ys[i]);
    }
}

// x += M^-1 sum_{i < jb} v_i y_i (the sum in float-float)
__global__ void __launch_bounds__(kT) arn_update_kernel(Arn a) {
    const int b = blockIdx.y;
    const int64_t t = blockIdx.x * (int64_t)kT + threadIdx.x;
    const int n = a.jb[b];
    if (t >= a.N || n == 0) return;
    const cff *Vb = a.V + (int64_t)b * a.vstride;
    const cff *yb = a.yff + (int64_t)b * a.m;
    ffloat r0(0.f, 0.f), i0(0.f, 0.f), r1(0.f, 0.f), i1(0.f, 0.f);
    for (int i = 0; i < n; ++i) {
        const cff yi = yb[i];
        cff_mac(r0, i0, Vb[(int64_t)i * a.n2 + t], yi);
        cff_mac(r1, i1, Vb[(int64_t)i * a.n2 + a.N + t], yi);
    }
    const double2 u0 = make_double2((double)r0, (double)i0), u1 = make_double2((double)r1, (double)i1);
    double2 o0, o1;
    const int q = b * a.S + a.surf[t];
    precond(a.vinv[t], a.pq[q], a.s[q], u0, u1, o0, o1);
    double2 *xb = a.x + (int64_t)b * a.n2;
    xb[t] = cadd(xb[t], o0);
    xb[a.N + t] = cadd(xb[a.N + t], o1);
}

// preconditioner constants of a solve: vinv = 1 / V_ii, pq = 1 / (1 + s)
__global__ void arn_precond_setup_kernel(int64_t N, int BS, const double *Vself, const double2 *s, double *vinv,
                                         double2 *pq, ffloat *vinvf, cff *pqf, cff *sf) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < N) {
        vinv[t] = 1.0 / Vself[t];
        vinvf[t] = ffloat(vinv[t]);
    }
    if (t < BS) {
        pq[t] = cdiv(make_double2(1.0, 0.0), make_double2(1.0 + s[t].x, s[t].y));
        pqf[t] = to_cff(pq[t]);
        sf[t] = to_cff(s[t]);
    }
}

// the scales that the tensor-core launches carry by value (powers of two) and their operand parts
uint64_t tc_scales(const Tree &tr) {
    uint64_t k = tr.tcp_f16 ? 1 : 0;
    for (const float f : {tr.rho_min, tr.tcp_gs, tr.tcp_ts}) {
        uint32_t b;
        std::memcpy(&b, &f, sizeof(b));
        k = k << 9 | b >> 23;
    }
    return k;
}

// the start of an Arnoldi step: v_j and M^-1 v_j, which the product takes from z or (null) xtf
int launch_precond(lspr_ctx *ctx, const Arn &a, cudaStream_t st) {
    ++ctx->n_launches;
    if (a.xtf)
        arn_precond_t_kernel<<<dim3(grid_for(a.N, 32), grid_for(a.B, 32)), dim3(32, 8), 0, st>>>(a);
    else
        arn_precond_kernel<<<dim3(grid_for(a.N, kT), a.B), kT, 0, st>>>(a);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// the two Gram-Schmidt passes and the end of an Arnoldi step
int launch_orthogonalise(lspr_ctx *ctx, const Arn &a, cudaStream_t st) {
    static int set0[kSmemDevices] = {}, set1[kSmemDevices] = {}, setu[kSmemDevices] = {};
    const bool wide = a.chunk == 2048;
    const size_t smem = dot_smem(a.chunk, a.m, false), smem_u = dot_smem(kUpdChunk, a.m, true);
    LSPR_TRY(ctx, wide ? allow_smem(arn_dot_kernel<2048, false>, (int)smem, ctx->device, set1)
                       : allow_smem(arn_dot_kernel<1024, false>, (int)smem, ctx->device, set0));
    LSPR_TRY(ctx, allow_smem(arn_dot_kernel<kUpdChunk, true>, (int)smem_u, ctx->device, setu));
    const dim3 g0(a.nch, a.B);
    if (wide) arn_dot_kernel<2048, false><<<g0, kT, smem, st>>>(a);
    else arn_dot_kernel<1024, false><<<g0, kT, smem, st>>>(a);
    arn_dot_kernel<kUpdChunk, true><<<dim3(grid_for(a.n2, kUpdChunk), a.B), kT, smem_u, st>>>(a);
    arn_axpy_kernel<<<dim3(grid_for(a.n2, kT * kAxpyPer), a.B), kT, 0, st>>>(a);
    ctx->n_launches += 3;
    arn_tail_kernel<<<a.B, 32, tail_smem(a.m), st>>>(a);
    ++ctx->n_launches;
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

// Records one Arnoldi cycle into gc: [init] -> while{step} -> [back substitution, update].
// Launches go to ctx->gstream (ctx->stream is redirected there while recording so that
// the operator's launchers record into the graph too).  Kernel counts of the recording
// are kept in gc and removed from the context's counters.
int capture_cycle(lspr_ctx *ctx, int mode, const Arn &a0, GraphCache &gc) {
    gc.reset();
    cudaStream_t cs = ctx->gstream, saved = ctx->stream;
    const int64_t l0 = ctx->n_launches, mv0 = ctx->matvec_count;
    const dim3 gv(grid_for(a0.n2, kT), a0.B), gN(grid_for(a0.N, kT), a0.B);
    cudaGraph_t g = nullptr;
    bool capturing = false;
    auto fail = [&](int code) {
        if (capturing) {
            cudaGraph_t tmp = nullptr;
            cudaStreamEndCapture(cs, &tmp);
        }
        cudaGetLastError();
        ctx->stream = saved;
        ctx->n_launches = l0;
        ctx->matvec_count = mv0;
        if (g) cudaGraphDestroy(g);
        return code;
    };
#define CAP_TRY(expr)                                                      \
    do {                                                                   \
        cudaError_t e__ = (expr);                                          \
        if (e__ != cudaSuccess) return fail(cuda_status(ctx, e__, #expr)); \
    } while (0)
    CAP_TRY(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h;
    CAP_TRY(cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault));
    Arn a = a0;
    a.cond = h;
    a.go = nullptr;
    ctx->stream = cs;
    // head: v_0 and the cycle state
    CAP_TRY(cudaStreamBeginCaptureToGraph(cs, g, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    capturing = true;
    arn_init_kernel<<<gv, kT, 0, cs>>>(a);
    CAP_TRY(cudaGetLastError());
    CAP_TRY(cudaStreamEndCapture(cs, &g));
    capturing = false;
    cudaGraphNode_t head = nullptr;
    size_t nn = 1;
    CAP_TRY(cudaGraphGetNodes(g, &head, &nn));
    // the loop over Arnoldi steps
    cudaGraphNodeParams p = {};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeWhile;
    p.conditional.size = 1;
    cudaGraphNode_t loop = nullptr;
    CAP_TRY(cudaGraphAddNode(&loop, g, &head, nullptr, 1, &p));
    cudaGraph_t body = p.conditional.phGraph_out[0];
    const int64_t l1 = ctx->n_launches;
    CAP_TRY(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    capturing = true;
    const int rp = launch_precond(ctx, a, cs);
    if (rp != LSPR_OK) return fail(rp);
    // the product works on the running systems only, packed into the first slots (with
    // several surfaces, set t K + k is surface t of the k-th of the K running systems)
    ctx->rhs_map = a.rmap;
    ctx->rhs_inv = a.rmap + a.B;
    ctx->rhs_nact = a.rmap + 2 * a.B + 1;
    const int rc = apply_operator(ctx, mode, a.xtf ? nullptr : a.z, a.w, a.s, a.B);
    ctx->rhs_map = ctx->rhs_inv = ctx->rhs_nact = nullptr;
    if (rc != LSPR_OK) return fail(rc);
    const int rt = launch_orthogonalise(ctx, a, cs);
    if (rt != LSPR_OK) return fail(rt);
    CAP_TRY(cudaStreamEndCapture(cs, &body));
    capturing = false;
    const int64_t l2 = ctx->n_launches;
    // tail: x += M^-1 V y
    CAP_TRY(cudaStreamBeginCaptureToGraph(cs, g, &loop, nullptr, 1, cudaStreamCaptureModeRelaxed));
    capturing = true;
    arn_backsub_kernel<<<a.B, 32, a.m * sizeof(double2), cs>>>(a);
    arn_update_kernel<<<gN, kT, 0, cs>>>(a);
    CAP_TRY(cudaGetLastError());
    CAP_TRY(cudaStreamEndCapture(cs, &g));
    capturing = false;
    cudaGraphExec_t exec = nullptr;
    CAP_TRY(cudaGraphInstantiate(&exec, g, 0));
#undef CAP_TRY
    ctx->stream = saved;
    ctx->n_launches = l0;
    ctx->matvec_count = mv0;
    gc.graph = g;
    gc.exec = exec;
    gc.per_step = l2 - l1;
    gc.outer = 3;   // init, back substitution, update
    return LSPR_OK;
}

// One Arnoldi cycle launched from the host, without a graph: the kernels of the recorded
// cycle in the same order, the loop condition read back after every step.  With per-kernel
// timing the vector kernels are timed under T_GMRES (the operator's under their own slots).
// Launches are counted as they happen; products are counted by the caller per running
// system, as for a recorded cycle.
int host_cycle(lspr_ctx *ctx, int mode, const Arn &a0, int *go_d) {
    cudaStream_t st = ctx->stream;
    Arn a = a0;
    a.go = go_d;
    a.cond = 0;
    const int64_t mv0 = ctx->matvec_count;
    const dim3 gv(grid_for(a.n2, kT), a.B), gN(grid_for(a.N, kT), a.B);
    cudaEvent_t ev;
    timer_begin(ctx, T_GMRES, &ev);
    arn_init_kernel<<<gv, kT, 0, st>>>(a);
    ++ctx->n_launches;
    timer_end(ctx, T_GMRES, ev);
    int more = 1, sets = a.B * a.S;
    const bool count = ctx->timing.enabled;   // channel sets of each product, for the timing counts
    if (count) {
        LSPR_TRY(ctx, cudaMemcpyAsync(&sets, a.rmap + 2 * a.B + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
    }
    while (more) {
        timer_begin(ctx, T_GMRES, &ev);
        LSPR_TRY_ST(launch_precond(ctx, a, st));
        timer_end(ctx, T_GMRES, ev);
        ctx->rhs_map = a.rmap;
        ctx->rhs_inv = a.rmap + a.B;
        ctx->rhs_nact = a.rmap + 2 * a.B + 1;
        ctx->timing_sets = count ? sets : -1;
        const int rc = apply_operator(ctx, mode, a.xtf ? nullptr : a.z, a.w, a.s, a.B);
        ctx->rhs_map = ctx->rhs_inv = ctx->rhs_nact = nullptr;
        ctx->timing_sets = -1;
        LSPR_TRY_ST(rc);
        timer_begin(ctx, T_GMRES, &ev);
        LSPR_TRY_ST(launch_orthogonalise(ctx, a, st));
        timer_end(ctx, T_GMRES, ev);
        LSPR_TRY(ctx, cudaMemcpyAsync(&more, go_d, sizeof(int), cudaMemcpyDeviceToHost, st));
        if (count)
            LSPR_TRY(ctx, cudaMemcpyAsync(&sets, a.rmap + 2 * a.B + 1, sizeof(int), cudaMemcpyDeviceToHost, st));
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
    }
    timer_begin(ctx, T_GMRES, &ev);
    arn_backsub_kernel<<<a.B, 32, a.m * sizeof(double2), st>>>(a);
    arn_update_kernel<<<gN, kT, 0, st>>>(a);
    ctx->n_launches += 2;
    timer_end(ctx, T_GMRES, ev);
    LSPR_TRY(ctx, cudaGetLastError());
    ctx->matvec_count = mv0;
    return LSPR_OK;
}

}  // namespace

int gmres_graph_solve(lspr_ctx *ctx, int mode, int B, int m, int maxiter, double tol, const double2 *s_d,
                      const double2 *b_d, double2 *x_d, bool x_zero, bool trust_estimate, std::vector<int> &iters,
                      std::vector<double> &relres, const std::vector<double> &bnorm) {
    if (B < 1 || m < 1 || m > kMaxRestart) return LSPR_E_ARG;
    const Mesh &me = ctx->mesh;
    const int64_t N = me.N, n2 = 2 * N;
    cudaStream_t st = ctx->stream;
    if (ctx->use_graphs && !ctx->timing.enabled && !ctx->gstream) {
        LSPR_TRY(ctx, cudaStreamCreateWithFlags(&ctx->gstream, cudaStreamNonBlocking));
        LSPR_TRY(ctx, cudaEventCreateWithFlags(&ctx->ev_g0, cudaEventDisableTiming));
        LSPR_TRY(ctx, cudaEventCreateWithFlags(&ctx->ev_g1, cudaEventDisableTiming));
    }
    ArnoldiBufs &ab = ctx->arn;
    const int chunk = dot_chunk(n2, B, std::max(1, ctx->num_sms));
    const int nch = (int)((n2 + chunk - 1) / chunk), nblk = (int)grid_for(n2, kT);
    const int64_t vstride = (int64_t)(m + 1) * n2;
    LSPR_TRY(ctx, ctx->gm_V.ensure((size_t)B * vstride));
    LSPR_TRY(ctx, ctx->gm_w.ensure((size_t)B * n2));
    LSPR_TRY(ctx, ctx->gm_z.ensure((size_t)B * n2));
    LSPR_TRY(ctx, ab.h.ensure((size_t)B * (m + 1)));
    LSPR_TRY(ctx, ab.hcol.ensure((size_t)B * (m + 1)));
    LSPR_TRY(ctx, ab.part.ensure((size_t)B * (m + 1) * std::max<int64_t>(nch, grid_for(n2, kUpdChunk))));
    LSPR_TRY(ctx, ab.npart.ensure((size_t)B * nblk));
    LSPR_TRY(ctx, ab.nrm.ensure(B));
    LSPR_TRY(ctx, ab.npart0.ensure((size_t)B * nch));
    LSPR_TRY(ctx, ab.reorth.ensure(B));
    LSPR_TRY(ctx, ab.H.ensure((size_t)B * (m + 1) * m));
    LSPR_TRY(ctx, ab.cs.ensure((size_t)B * m));
    LSPR_TRY(ctx, ab.sn.ensure((size_t)B * m));
    LSPR_TRY(ctx, ab.g.ensure((size_t)B * (m + 1)));
    LSPR_TRY(ctx, ab.y.ensure((size_t)B * m));
    LSPR_TRY(ctx, ab.res.ensure(B));
    LSPR_TRY(ctx, ab.bn.ensure(B));
    LSPR_TRY(ctx, ab.par.ensure(2));
    LSPR_TRY(ctx, ab.tick.ensure(2 * (size_t)B + 1));
    LSPR_TRY(ctx, ab.ctl.ensure(1 + 3 * (size_t)B));
    LSPR_TRY(ctx, ab.rmap.ensure(2 * (size_t)B + 2));
    LSPR_TRY(ctx, ab.hff.ensure((size_t)B * (m + 1)));
    LSPR_TRY(ctx, ab.yff.ensure((size_t)B * m));
    LSPR_TRY(ctx, ab.ninv.ensure(B));
    LSPR_TRY(ctx, ab.vinv.ensure(N));
    LSPR_TRY(ctx, ab.pq.ensure((size_t)B * me.S));
    LSPR_TRY(ctx, ab.vinvf.ensure(N));
    LSPR_TRY(ctx, ab.pqf.ensure(2 * (size_t)B * me.S));
    const bool transposed = mode_prec(mode) == PREC_F32 && B > 1 && me.S == 1;
    if (transposed) LSPR_TRY(ctx, ctx->xtf.ensure((size_t)B * n2));
    LSPR_TRY(ctx, ab.go.ensure(1));
    if (!ab.stats.p) {
        LSPR_TRY(ctx, ab.stats.ensure(4));
        LSPR_TRY(ctx, cudaMemsetAsync(ab.stats.p, 0, 4 * sizeof(unsigned long long), st));
    }
    Arn a;
    a.B = B;
    a.m = m;
    a.nch = nch;
    a.chunk = chunk;
    a.nblk = nblk;
    a.N = N;
    a.n2 = n2;
    a.vstride = vstride;
    a.V = (cff *)ctx->gm_V.p;
    a.w = ctx->gm_w.p;
    a.z = ctx->gm_z.p;
    a.x = x_d;
    a.b = b_d;
    a.s = s_d;
    a.vinv = ab.vinv.p;
    a.pq = ab.pq.p;
    a.vinvf = (const ffloat *)ab.vinvf.p;
    a.pqf = (const cff *)ab.pqf.p;
    a.sf = a.pqf + (size_t)B * me.S;
    a.xtf = transposed ? ctx->xtf.p : nullptr;
    a.surf = me.surf.p;
    a.S = me.S;
    a.h = ab.h.p;
    a.hcol = ab.hcol.p;
    a.part = ab.part.p;
    a.H = ab.H.p;
    a.sn = ab.sn.p;
    a.g = ab.g.p;
    a.y = ab.y.p;
    a.npart = ab.npart.p;
    a.nrm = ab.nrm.p;
    a.npart0 = ab.npart0.p;
    a.reorth = ab.reorth.p;
    a.cs = ab.cs.p;
    a.res = ab.res.p;
    a.bn = ab.bn.p;
    a.par = ab.par.p;
    a.tick = ab.tick.p;
    a.jdev = ab.ctl.p;
    a.active = ab.ctl.p + 1;
    a.jb = ab.ctl.p + 1 + B;
    a.iters = ab.ctl.p + 1 + 2 * B;
    a.rmap = ab.rmap.p;
    a.hff = (cff *)ab.hff.p;
    a.yff = (cff *)ab.yff.p;
    a.ninv = (ffloat *)ab.ninv.p;
    a.go = nullptr;
    a.stats = ab.stats.p;
    a.cond = 0;
    // per-call parameters live in device memory, so one recorded graph serves every call
    const double par[2] = {tol, (double)std::max(1, maxiter)};
    LSPR_TRY(ctx, cudaMemcpyAsync(ab.bn.p, bnorm.data(), sizeof(double) * B, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyAsync(ab.par.p, par, sizeof(par), cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemsetAsync(ab.ctl.p, 0, sizeof(int) * (1 + 3 * (size_t)B), st));
    LSPR_TRY(ctx, cudaMemsetAsync(ab.tick.p, 0, sizeof(unsigned) * (2 * (size_t)B + 1), st));
    ++ctx->n_launches;
    arn_precond_setup_kernel<<<grid_for(std::max<int64_t>(N, (int64_t)B * me.S), kT), kT, 0, st>>>(
        N, B * me.S, me.Vself.p, s_d, ab.vinv.p, ab.pq.p, (ffloat *)ab.vinvf.p, (cff *)ab.pqf.p,
        (cff *)ab.pqf.p + (size_t)B * me.S);
    for (int b = 0; b < B; ++b) {
        iters[b] = 0;
        relres[b] = 1.0;
    }
    std::vector<int> act(B), ctl(1 + 3 * (size_t)B);
    std::vector<double> est(B), beta(B);
    const dim3 gv(grid_for(n2, kT), B);
    static uint64_t clock = 0;
    bool first = true;
    while (true) {
        // explicit residual w = A x - b and beta = ||w|| (x = 0 on entry: w = -b)
        const bool skip_mv = first && x_zero;
        if (!skip_mv) LSPR_TRY_ST(apply_operator(ctx, mode, x_d, a.w, s_d, B));
        ++ctx->n_launches;
        arn_resid_kernel<<<gv, kT, 0, st>>>(a, skip_mv ? 1 : 0);
        LSPR_TRY(ctx, cudaGetLastError());
        LSPR_TRY(ctx, cudaMemcpyAsync(beta.data(), a.nrm, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
        first = false;
        bool any = false;
        for (int b = 0; b < B; ++b) {
            relres[b] = beta[b] / bnorm[b];
            act[b] = relres[b] > tol && iters[b] < maxiter && std::isfinite(relres[b]);
            any = any || act[b];
        }
        if (!any) break;
        LSPR_TRY(ctx, cudaMemcpyAsync(a.active, act.data(), sizeof(int) * B, cudaMemcpyHostToDevice, st));
        // The graph recorded for this configuration.  Recorded launches hold buffer
        // addresses (unchanged while no buffer is reallocated: the allocation count) and
        // sizes that set grids and loop bounds (the counts below); a geometry or tree
        // rebuilt with the same sizes reuses the graph, since the kernels read the new
        // contents from the same buffers.
        const Tree &tr = ctx->tree;
        uint64_t key[24] = {g_alloc_generation.load(), (uint64_t)mode, (uint64_t)B, (uint64_t)m,
                            (uint64_t)(uintptr_t)x_d, (uint64_t)(uintptr_t)b_d, (uint64_t)(uintptr_t)s_d,
                            (uint64_t)N, (uint64_t)me.Ns, (uint64_t)me.nnz, (uint64_t)tr.ready, (uint64_t)tr.P,
                            (uint64_t)tr.NT, (uint64_t)tr.nboxes, (uint64_t)tr.n_p2p_items,
                            (uint64_t)tr.n_m2p_items, (uint64_t)tr.n_p2m_items,
                            (uint64_t)direct_items(ctx, (int64_t)B * me.S).n,
                            (uint64_t)(uintptr_t)ctx->gm_V.p, (uint64_t)ctx->num_sms, (uint64_t)me.S,
                            (uint64_t)ctx->tensor_cores | tc_scales(tr) << 8, (uint64_t)tr.n_tc_items,
                            (uint64_t)tr.n_tcp_items};
        GraphCache *gc = nullptr;
        const bool graphs = ctx->use_graphs && !ctx->timing.enabled;
        for (GraphCache &c : ctx->gcache)
            if (graphs && c.exec && std::equal(key, key + 24, c.key)) gc = &c;
        if (graphs && !gc) {
            gc = &ctx->gcache[0];
            for (GraphCache &c : ctx->gcache)
                if (c.use < gc->use) gc = &c;
            // the operator's buffers must exist before recording (no allocation inside a graph)
            if (skip_mv) LSPR_TRY_ST(apply_operator(ctx, mode, b_d, a.z, s_d, B));
            LSPR_TRY(ctx, cudaStreamSynchronize(st));
            if (capture_cycle(ctx, mode, a, *gc) != LSPR_OK) {
                ctx->use_graphs = false;   // host-driven cycles from now on
                gc = nullptr;
            }
            if (gc) {
                ++ctx->graph_recordings;
                key[0] = g_alloc_generation.load();   // buffers the recording itself sized
                std::copy(key, key + 24, gc->key);
            }
        }
        if (gc) {
            gc->use = ++clock;
            LSPR_TRY(ctx, cudaEventRecord(ctx->ev_g0, st));
            LSPR_TRY(ctx, cudaStreamWaitEvent(ctx->gstream, ctx->ev_g0, 0));
            LSPR_TRY(ctx, cudaGraphLaunch(gc->exec, ctx->gstream));
            LSPR_TRY(ctx, cudaEventRecord(ctx->ev_g1, ctx->gstream));
            LSPR_TRY(ctx, cudaStreamWaitEvent(st, ctx->ev_g1, 0));
        }
        if (!gc) LSPR_TRY_ST(host_cycle(ctx, mode, a, ab.go.p));
        LSPR_TRY(ctx, cudaMemcpyAsync(ctl.data(), ab.ctl.p, sizeof(int) * ctl.size(), cudaMemcpyDeviceToHost, st));
        LSPR_TRY(ctx, cudaMemcpyAsync(est.data(), a.res, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
        LSPR_TRY(ctx, cudaStreamSynchronize(st));
        const int steps = ctl[0];
        if (gc) {
            ++ctx->graph_cycles;
            ctx->n_launches += gc->outer + gc->per_step * steps;
        }
        bool all_met = true;
        for (int b = 0; b < B; ++b) {
            ctx->matvec_count += ctl[1 + 2 * B + b] - iters[b];   // products of the running systems only
            iters[b] = ctl[1 + 2 * B + b];
            if (act[b]) {
                const double r = est[b] / bnorm[b];
                if (!(r <= tol) && iters[b] < maxiter) all_met = false;
                relres[b] = r;
            }
        }
        if (trust_estimate && all_met) break;
    }
    return LSPR_OK;
}

}  // namespace lspr
