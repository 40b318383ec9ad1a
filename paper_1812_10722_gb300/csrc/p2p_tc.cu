// P2P of several right-hand sides on the fifth-generation tensor cores (tcgen05).
//
// The direct far-rule sums of Eq. summation for a target x over sources y_s,
//   V_j(x) = sum_s G(x, y_s) q_s[j],   K_j(x) = sum_s dG/dn(x, y_s) mu_s[j],
// (q, mu complex per right-hand side j) are two matrix products once the kernel values of a
// tile are laid out as operands:
//   D_V[channel][target] += W_V[channel][source] G[source][target]
//   D_K[channel][target] += W_K[channel][source] dG/dn[source][target]
// with the channels (re and im of each of up to 64 right-hand sides: 128 rows) as the MMA's M,
// the 256 targets of a group of four consecutive 64-target blocks as its N, and the sources of a
// pipeline stage as its K.  W_V holds only single-layer weights and W_K only double-layer ones,
// so no operand carries structural zeros, and one kernel tile serves 64 right-hand sides.
// The group walks the union of its blocks' P2P source ranges; a target whose block does not sum
// a range gets zero kernel values there, and a target's own panel is skipped (its exact integral
// is in the near correction), as in p2p_kernel.  Both operands are split into high and low
// parts (each rounded to nearest) with FP32 accumulation in tensor memory: with more than 32
// right-hand sides in the unit, three MMAs per operand pair give W_hi G_hi + W_hi G_lo +
// W_lo G_hi; with at most 32,
// W_hi and W_lo are the two halves of one 128-row operand and two MMAs give all four products
// (the epilogue adds both halves).
//
// The parts are FP16 (16 sources per stage) where the kernel values' range allows it, else TF32 (8
// sources; FP16 parts hold the same 22 bits at twice the rate, but for the smallest values, see below).  The smallest and the largest distance
// of a P2P pair (pair_range_kernel, once per tree) set powers of two that bring G and dG/dn (at most
// 1/r and 1/r^2) below 2^15.  With their ratio at most kTcP2PRange = 4096, G stays above 2^3 and loses
// nothing; dG/dn falls to 2^-9 at the largest distances, where its parts keep 2^-25 absolute: summed
// over the sources of a P2P region of area a that is below 2^-40 a / r_min^2 of a potential of order 2 pi
// (2^-27 at a = 10 nm^2, r_min = 0.04 nm), less than the accumulation rounds off.  The weights of one
// right-hand side, layer and part (re, im) are scaled by a bound of their largest magnitude.  All scales are powers of
// two: those of G and dG/dn are folded into the positions and normals, all are undone as the
// accumulators are drained.
//
// The split weights are formed once per product in operand layout (p2p_image_kernel: 16 KB per stage's
// sources and 64 right-hand sides), so that staging them is one bulk copy; stages are
// therefore aligned to multiples of their sources, and a range that begins or ends inside one gets
// zero kernel values for the rest.
//
// Roles (persistent, one CTA per SM, both accumulators in the SM's 512 tensor-memory columns):
//   warp 16 (one lane) fetches work units into a small ring and bulk-copies every stage's inputs
//     (the weight operands, and the positions and normals of its sources);
//   warps 0-15 (two threads per target of the group, half of the stage's sources each)
//     generate G and dG/dn of every stage in registers, two sources at a time in packed f32x2
//     arithmetic, split them and write the B operands; after the first
//     stage of the next unit they drain the finished unit's accumulators (tcgen05.ld) into the
//     FP64 accumulators;
//   warp 17 (one lane) issues the MMAs of each stage once it is written, commits to the stage's
//     "empty" barrier and, at the end of a unit, to the accumulator barrier.
// While a unit's accumulators are drained no MMA runs, so units are long (tc_unit) and the drain adds
// whole 32-byte sectors: rows 2 j and 2 j + 1 of an operand are re and im of right-hand side j, and a
// warp exchanges halves of D_V and D_K so that one instruction adds all four components of eight.
// 81920 panels, 64 right-hand sides, with the preparing kernels: 1.84 ms; 1.76 with units of 4096 sources,
// whose error was too large (lspr_internal.cuh); at that length 1.92 with the sectors
// touched by two instructions each and every range's bounds loaded when it begins instead of one range
// ahead, and 2.19 in that form with units of 2048 sources; 3.44 with TF32 parts (a stage
// of 8 sources took 0.86 us, 0.48 of it the MMAs and as much its 121 KB of shared-memory traffic; FP16
// halves both per source); 4.24 with the weights split by four of the generating warps (which every
// stage waited for) and a barrier arrival per thread.  Error of the product of 28 right-hand sides
// against the float-float operator: 2.3e-6 with FP16 parts, 4.4e-6 with TF32 (half as many
// accumulation steps).
// Every wait is bounded (about a second): one that runs out raises an abort flag that the
// other roles see, the block drains its bulk copies and MMAs in flight, frees its tensor memory
// and returns,
// and the context's device error count (error[0]) records it.  With error[1] set, thread 0
// first waits on a barrier that nothing arrives on, so that the wait runs out before any work
// is issued (the host's check of this failure path).
#include "farfield.cuh"
#include "tcgen05.cuh"

namespace lspr {

namespace {

using namespace tc;

constexpr int kRC = 64;                        // right-hand sides per work unit
constexpr int kTcN = kTcGroup * kTargetBlock;  // targets per work unit (the MMA's N)
constexpr int kSBO = 256;                      // bytes per 8-row group of a stage operand (two 16-byte columns)
constexpr int kGenSplit = 2;                   // generating threads per target (one column each)
constexpr int kGenThreads = kGenSplit * kTcN;
constexpr int kGenWarps = kGenThreads / 32;
constexpr int kProdWarp = kGenWarps, kMmaWarp = kGenWarps + 1;
constexpr int kTcThreads = 32 * (kGenWarps + 2);
constexpr int kUnitRing = 4;
constexpr int kRingConsumers = kGenWarps + 1;  // lane 0 of each consumer warp
constexpr uint32_t kTmemCols = 2 * kTcN;       // D_V in columns [0, 256), D_K in [256, 512)
constexpr int kAPart = (128 / 8) * kSBO;       // one split part of a weight operand (128 rows)
constexpr int kBPart = (kTcN / 8) * kSBO;      // one split part of a kernel operand (256 rows)
// stage: the weight operands as bulk-copied from the image (W_V hi | W_V lo | W_K hi | W_K lo, or
// stacked W_V | W_K) | G hi | G lo | dG hi | dG lo | the geometry of the stage's sources (kTcSrcRows
// rows of a float per source)
constexpr int kOffG = 4 * kAPart, kOffD = 4 * kAPart + 2 * kBPart;
constexpr int kOffSrc = 4 * kAPart + 4 * kBPart;
constexpr int kImgBlock = 4 * kAPart;          // image bytes per stage's sources and 64 right-hand sides
constexpr int kStage = kOffSrc + kTcSrcRows * 16 * 4;
constexpr int kStages = 4;
constexpr int kSmem = kStages * kStage;
static_assert(kSmem + 1024 <= 232448, "the stages and the static shared memory fit one SM");
// operand parts: FP16 with 16 sources per stage, or TF32 with 8
template <bool F16>
struct P2PShape {
    static constexpr int SRC = F16 ? 16 : 8;           // sources per stage (the MMA's K)
    static constexpr int PART = SRC / kGenSplit;       // sources per generating thread and 16-byte column
    static constexpr uint32_t SRC_BYTES = kTcSrcRows * SRC * 4;
    static constexpr uint32_t IDESC = F16 ? idesc_f16(128, kTcN) : idesc_tf32(128, kTcN);
    static __device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
        if (F16) tc_mma_f16(d, a, b, IDESC, acc);
        else tc_mma(d, a, b, IDESC, acc);
    }
    // the high and low parts of PART values to their columns
    static __device__ __forceinline__ void split(const float (&v)[PART], unsigned char *hi, unsigned char *lo) {
        if constexpr (F16) {
            const HalfPair p = f16_split(v);
            *(uint4 *)hi = p.hi;
            *(uint4 *)lo = p.lo;
        } else {
            const TfPair p = tf32_split(make_float4(v[0], v[1], v[2], v[3]));
            *(float4 *)hi = p.hi;
            *(float4 *)lo = p.lo;
        }
    }
};
static_assert(kTmemCols <= 512 && kTcN <= 256, "both accumulators fit the tensor memory");
static_assert(kStages >= 2, "at least two stages");
static_assert(kRC * 2 == 128, "re and im of the unit's right-hand sides fill the MMA's M");

// byte offset of (row r, 16-byte column c) inside one split part of a stage operand (K-major 8 x
// 16-byte core matrices, no swizzle)
__device__ __forceinline__ int core_off(int r, int c) { return (r >> 3) * kSBO + c * 128 + (r & 7) * 16; }

// largest magnitude per layer, part (re, im) and system of the right-hand sides xt [2N][B], times the
// largest source weight: a bound of the weights of the system's sets, as the bits of non-negative floats
// in mx[4 set + c], c = re and im of the single layer, then of the double layer
constexpr int kMaxSets = 512;   // right-hand sides per block column
__global__ void __launch_bounds__(256)
    p2p_max_kernel(int64_t N, int B, int S, const float2 *__restrict__ xt, const int *__restrict__ stat, int *mx,
                   const int *inv, const int *nact, int min_rhs) {
    __shared__ int smax[4 * kMaxSets];
    const int sets = nact ? *nact : B * S;
    if (sets < min_rhs) return;
    const int j0 = blockIdx.y * kMaxSets, nj = min(kMaxSets, B - j0), K = sets / S;
    for (int j = threadIdx.x; j < 4 * nj; j += blockDim.x) smax[j] = 0;
    __syncthreads();
    const float wa = __int_as_float(stat[2]);
    const int64_t rows = (2 * N + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = blockIdx.x * rows, r1 = min(2 * N, r0 + rows);
    for (int64_t q = threadIdx.x; q < (r1 - r0) * nj; q += blockDim.x) {
        const int64_t r = r0 + q / nj;
        const int j = (int)(q % nj);
        int *const s = smax + 4 * j + (r < N ? 2 : 0);
        const float2 v = __ldg(xt + r * B + j0 + j);
        const int re = __float_as_int(fabsf(v.x) * wa), im = __float_as_int(fabsf(v.y) * wa);
        if (re > s[0]) atomicMax(s, re);
        if (im > s[1]) atomicMax(s + 1, im);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < 4 * nj; j += blockDim.x) {
        const int b = j0 + (j >> 2), k = inv ? inv[b] : b;
        if (k < 0 || smax[j] == 0) continue;
        for (int t = 0; t < S; ++t) atomicMax(&mx[4 * (t * K + k) + (j & 3)], smax[j]);
    }
}

// The split weights of every stage's sources in operand layout.  One thread per (sources of a
// stage, unit chunk, half of them, right-hand side).  Sources past the end have zero weights;
// rows of right-hand sides not in use are not written (their accumulator rows are not read).
template <bool F16>
__global__ void __launch_bounds__(128)
    p2p_image_kernel(int64_t Ns, int B, int nrc, const float4 *__restrict__ sw, unsigned char *__restrict__ img,
                     const int *nact, int min_rhs, int nsurf, const int *__restrict__ mask, const int *__restrict__ mx) {
    using H = P2PShape<F16>;
    const int Bact = nact ? *nact : B;
    if (Bact < min_rhs) return;
    const int64_t blk = blockIdx.x;   // (sources of a stage, chunk)
    const int64_t g = blk / nrc;
    const int rc = (int)(blk - g * nrc), b0 = rc * kRC, nb = min(kRC, Bact - b0);
    if (nb <= 0) return;
    const int q = threadIdx.x >> 6, j = threadIdx.x & 63;
    const int64_t s0 = g * H::SRC + H::PART * q;
    // no range that holds these sources has one of the chunk's surfaces: no unit reads the block
    if (nsurf > 1 && !(mask[g] & set_surfaces(b0, nb, Bact, nsurf))) return;
    if (j >= nb) return;
    float f[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) f[c] = F16 ? f16_scale(__ldg(mx + 4 * (b0 + j) + c)) : 1.f;
    float w[4][H::PART];
#pragma unroll
    for (int i = 0; i < H::PART; ++i) {
        const float4 v = s0 + i < Ns ? __ldg(sw + (s0 + i) * B + b0 + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        w[0][i] = v.x * f[0];
        w[1][i] = v.y * f[1];
        w[2][i] = v.z * f[2];
        w[3][i] = v.w * f[3];
    }
    const bool stacked = nb <= kRC / 2;
    // rows: 2 j + (0: re, 1: im), the high part, then the low part; stacked: the low rows are 64 + 2 j + ..
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        unsigned char *o = img + blk * kImgBlock + (c >> 1) * (stacked ? kAPart : 2 * kAPart);
        unsigned char *hi = o + core_off(2 * j + (c & 1), q);
        H::split(w[c], hi, stacked ? o + core_off(64 + 2 * j + (c & 1), q) : hi + kAPart);
    }
}

template <bool F16>
__global__ void __launch_bounds__(kTcThreads, 1)
    p2p_tc_kernel(const int4 *__restrict__ items, int64_t nitems, const int4 *__restrict__ ivl, int B,
                  const float4 *__restrict__ tgt, int64_t ntgt, const float *__restrict__ srcs,
                  const unsigned char *__restrict__ img, int nrc, double *__restrict__ acc,
                  int *counter, int *error, const int *nact, int min_rhs, int nsurf, float gs, float ts,
                  const int *__restrict__ mx) {
    using H = P2PShape<F16>;
    constexpr int kSrc = H::SRC;
    // fewer right-hand sides in use than min_rhs: the FP32-pipe P2P takes this product
    if ((nact ? *nact : B) < min_rhs) return;
    extern __shared__ __align__(128) unsigned char tc_smem[];
    __shared__ __align__(8) uint64_t full_s[kStages], empty_s[kStages], raw_s[kStages];
    __shared__ __align__(8) uint64_t acc_full, acc_empty, ring_full[kUnitRing], ring_empty[kUnitRing], drain, gate;
    __shared__ int64_t ring[kUnitRing];
    __shared__ uint32_t tslot;
    __shared__ volatile int abort_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = smem_addr(tc_smem);
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            bar_init(smem_addr(&full_s[s]), kGenWarps);   // one arrival per generating warp
            bar_init(smem_addr(&empty_s[s]), 1);     // the MMAs' commit
            bar_init(smem_addr(&raw_s[s]), 1);       // the producer's expect_tx (+ the copies' bytes)
        }
        bar_init(smem_addr(&acc_full), 1);
        bar_init(smem_addr(&acc_empty), kGenWarps);
        for (int r = 0; r < kUnitRing; ++r) {
            bar_init(smem_addr(&ring_full[r]), 1);
            bar_init(smem_addr(&ring_empty[r]), kRingConsumers);
        }
        bar_init(smem_addr(&drain), 1);
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // failure-path check (error[1] set by the host): a bounded wait on a barrier that nothing
        // arrives on runs out before any work is issued, and the block returns without work
        if (__ldcg(error + 1)) {
            bar_init(smem_addr(&gate), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            bar_wait(smem_addr(&gate), 0u, &abort_s);   // phase 0 never completes: no arrival
        }
    }
    if (warp == 0) {
        __syncwarp();   // lane 0 may come from the set-up above (and its bounded check wait)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tslot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    const int Bact = nact ? *nact : B;   // right-hand sides in use (the first Bact slots)
    const int nbc = (Bact + kRC - 1) / kRC;
    const int64_t units = nitems * nbc;

    if (warp == kProdWarp) {
        // ---- work units, and the inputs of every stage by bulk copies: positions and normals
        // of the stage's sources, their weights for the unit's right-hand sides
        if (lane == 0) {
            int64_t seq = 0;   // stages armed so far
            for (int uc = 0;; ++uc) {
                const int slot = uc % kUnitRing;
                if (uc >= kUnitRing &&
                    !bar_wait(smem_addr(&ring_empty[slot]), (uint32_t)((uc / kUnitRing) - 1) & 1u, &abort_s))
                    break;
                const int64_t u = abort_s ? units : (int64_t)atomicAdd(counter, 1);
                ring[slot] = u;
                bar_arrive(smem_addr(&ring_full[slot]));
                if (u >= units) break;
                const int64_t ii = u / nbc;
                const int rc = (int)(u - ii * nbc), b0 = rc * kRC, nb = min(kRC, Bact - b0);
                const uint32_t abytes = nb <= kRC / 2 ? 2 * kAPart : 4 * kAPart;
                const int4 item = __ldg(items + ii);
                bool ok = true;
                const int um = set_surfaces(b0, nb, Bact, nsurf);
                int4 e_nx = item.y < item.z ? __ldg(ivl + item.y) : make_int4(0, 0, 0, 0);   // one range ahead
                for (int iv = item.y; iv < item.z && ok; ++iv) {
                    const int4 e = e_nx;
                    if (iv + 1 < item.z) e_nx = __ldg(ivl + iv + 1);
                    if (!(e.w & um)) continue;   // no source of the unit's surfaces (all roles agree)
                    for (int g = e.x / kSrc; g * kSrc < e.y; ++g, ++seq) {
                        const int s = (int)(seq % kStages);
                        if (seq >= kStages &&
                            !bar_wait(smem_addr(&empty_s[s]), (uint32_t)((seq / kStages) - 1) & 1u, &abort_s)) {
                            ok = false;
                            break;
                        }
                        const uint32_t rb = smem_addr(&raw_s[s]), dst = sbase + (uint32_t)(s * kStage);
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(rb),
                                     "r"((uint32_t)(abytes + H::SRC_BYTES))
                                     : "memory");
                        asm volatile(
                            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                dst + kOffSrc),
                            "l"(srcs + (int64_t)g * (kTcSrcRows * kSrc)), "r"(H::SRC_BYTES), "r"(rb)
                            : "memory");
                        asm volatile(
                            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                                dst),
                            "l"(img + ((int64_t)g * nrc + rc) * kImgBlock), "r"(abytes), "r"(rb)
                            : "memory");
                    }
                }
                if (!ok) break;
            }
            // the copies of the last armed stages may still be in flight
            for (int64_t k = seq > kStages ? seq - kStages : 0; k < seq; ++k)
                drain_wait(smem_addr(&raw_s[k % kStages]), (uint32_t)(k / kStages) & 1u);
        }
    } else if (warp == kMmaWarp) {
        // ---- MMA issue: one lane
        if (lane == 0) {
            int64_t seq = 0;
            int nu = 0;   // units with stages so far
            for (int uc = 0;; ++uc) {
                const int slot = uc % kUnitRing;
                if (!bar_wait(smem_addr(&ring_full[slot]), (uint32_t)(uc / kUnitRing) & 1u, &abort_s)) break;
                const int64_t u = ring[slot];
                if (u >= units) break;
                const int64_t ii = u / nbc;
                const int b0 = (int)(u - ii * nbc) * kRC, nb = min(kRC, Bact - b0);
                const bool stacked = nb <= kRC / 2;
                const int um = set_surfaces(b0, nb, Bact, nsurf);
                const int4 item = __ldg(items + ii);
                {
                    const uint32_t dv = tmem, dk = tmem + (uint32_t)kTcN;
                    bool ok = true, first = true;
                    int4 e_nx = item.y < item.z ? __ldg(ivl + item.y) : make_int4(0, 0, 0, 0);
                    for (int iv = item.y; iv < item.z && ok; ++iv) {
                        const int4 e = e_nx;
                        if (iv + 1 < item.z) e_nx = __ldg(ivl + iv + 1);
                        if (!(e.w & um)) continue;
                        // the accumulators are free once the previous unit is drained
                        if (first && nu >= 1) {
                            if (!bar_wait(smem_addr(&acc_empty), (uint32_t)((nu - 1) & 1), &abort_s)) {
                                ok = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;");
                        }
                        for (int g = e.x / kSrc; g * kSrc < e.y; ++g, ++seq) {
                            const int s = (int)(seq % kStages);
                            const uint32_t par = (uint32_t)(seq / kStages) & 1u;
                            if (!bar_wait(smem_addr(&raw_s[s]), par, &abort_s) ||
                                !bar_wait(smem_addr(&full_s[s]), par, &abort_s)) {
                                ok = false;
                                break;
                            }
                            asm volatile("tcgen05.fence::after_thread_sync;");
                            const uint32_t st = sbase + (uint32_t)(s * kStage);
                            const uint32_t koff = stacked ? kAPart : 2 * kAPart;
                            const uint64_t wvh = umma_desc(st, 128, kSBO);
                            const uint64_t wvl = umma_desc(st + kAPart, 128, kSBO);
                            const uint64_t wkh = umma_desc(st + koff, 128, kSBO);
                            const uint64_t wkl = umma_desc(st + koff + kAPart, 128, kSBO);
                            const uint64_t gh = umma_desc(st + kOffG, 128, kSBO);
                            const uint64_t gl = umma_desc(st + kOffG + kBPart, 128, kSBO);
                            const uint64_t hh = umma_desc(st + kOffD, 128, kSBO);
                            const uint64_t hl = umma_desc(st + kOffD + kBPart, 128, kSBO);
                            const uint32_t on = first ? 0u : 1u;
                            first = false;
                            H::mma(dv, wvh, gh, on);
                            H::mma(dv, wvh, gl, 1u);
                            H::mma(dk, wkh, hh, on);
                            H::mma(dk, wkh, hl, 1u);
                            if (!stacked) {
                                H::mma(dv, wvl, gh, 1u);
                                H::mma(dk, wkl, hh, 1u);
                            }
                            tc_commit(smem_addr(&empty_s[s]));
                        }
                    }
                    if (!ok) break;
                    if (!first) {
                        tc_commit(smem_addr(&acc_full));
                        ++nu;
                    }
                }
                bar_arrive(smem_addr(&ring_empty[slot]));
            }
            // the MMAs in flight complete before the block frees the tensor memory
            tc_commit(smem_addr(&drain));
            drain_wait(smem_addr(&drain), 0u);
        }
    } else {
        // ---- generators: thread tid owns target tt = tid mod 256 of the group (row tt of the
        // kernel operands) for the sources of 16-byte column hf of each stage, hf = tid / 256
        const int tt = tid & (kTcN - 1), hf = tid / kTcN;
        const int blk = tt / kTargetBlock;
        int64_t seq = 0;
        int nu = 0;
        bool pend = false;
        int p_nb = 0, p_b0 = 0;
        bool p_stacked = false;
        int64_t p_tbase = 0;
        // epilogue: warp w reads tensor-memory lanes 32 (w % 4).. (channel rows) and the 64
        // targets from column 64 (w / 4) of both accumulators; false: a wait ran out
        auto drain_acc = [&]() -> bool {
            const int qd = warp & 3, part = warp >> 2;
            const int64_t tc0 = p_tbase + part * (kTcN / 4) + lane;   // the targets of this lane's columns
            const int pc0 = tc0 < ntgt ? panel_of(tgt[tc0].w) : -1;
            const int pc1 = tc0 + 32 < ntgt ? panel_of(tgt[tc0 + 32].w) : -1;
            // row m: 2 j + (0: re, 1: im) of right-hand side j; stacked: of the high (m < 64) or the low half
            const int m = (32 * qd + lane) & (p_stacked ? 63 : 127), j = m >> 1;
            // the scales undone: of the kernel values and of the weights
            float undo_v = 1.f, undo_k = 1.f;
            if (F16 && j < p_nb) {
                undo_v = 1.f / gs * (1.f / f16_scale(__ldg(mx + 4 * (p_b0 + j) + (m & 1))));
                undo_k = 1.f / ts * (1.f / f16_scale(__ldg(mx + 4 * (p_b0 + j) + 2 + (m & 1))));
            }
            if (!warp_wait(smem_addr(&acc_full), (uint32_t)((nu - 1) & 1), &abort_s)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;");
            // The 16 right-hand sides of the warp's rows are added eight at a time, all four components of
            // each by one instruction (whole 32-byte sectors; a warp per accumulator would touch every
            // sector twice): lanes 0-15 take D_V, lanes 16-31 D_K, after one exchange between the halves.
            const bool dk = lane >= 16;
            const int jw = (m - lane) >> 1, ja = jw + ((lane & 15) >> 1), jb = ja + 8;   // the lane's right-hand sides
            double *const dst = acc + 4 * (p_b0 + ja) + 2 * (int)dk + (lane & 1);
            if (jw < p_nb) {
#pragma unroll 1
                for (int c0 = 0; c0 < kTcN / 4; c0 += 16) {
                    uint32_t v[16], k[16];
                    const uint32_t addr = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(part * (kTcN / 4) + c0);
                    tc_ld16(addr, v);
                    tc_ld16(addr + kTcN, k);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const int pc = c0 < 32 ? pc0 : pc1;
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const int p = __shfl_sync(0xffffffffu, pc, (c0 & 16) + x);
                        float fv = __uint_as_float(v[x]), fk = __uint_as_float(k[x]);
                        if (F16) fv *= undo_v, fk *= undo_k;
                        const float y = __shfl_xor_sync(0xffffffffu, dk ? fv : fk, 16);
                        if (p >= 0) {
                            double *const o = dst + 4 * (int64_t)p * B;
                            if (ja < p_nb) atomicAdd(o, (double)(dk ? y : fv));
                            if (jb < p_nb) atomicAdd(o + 32, (double)(dk ? fk : y));
                        }
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) bar_arrive(smem_addr(&acc_empty));
            pend = false;
            return true;
        };
        bool ok = true;
        for (int uc = 0; ok; ++uc) {
            const int slot = uc % kUnitRing;
            if (!warp_wait(smem_addr(&ring_full[slot]), (uint32_t)(uc / kUnitRing) & 1u, &abort_s)) {
                ok = false;
                break;
            }
            const int64_t u = ring[slot];
            if (u >= units) break;
            const int64_t ii = u / nbc;
            const int b0 = (int)(u - ii * nbc) * kRC, nb = min(kRC, Bact - b0);
            const bool stacked = nb <= kRC / 2;
            const int4 item = __ldg(items + ii);
            const int64_t tbase = (int64_t)item.x * kTcN;   // first target of the group
            const int64_t ti = tbase + tt;
            const bool live = ti < ntgt;
            const float4 q = live ? tgt[ti] : tgt[0];
            const int tp = live ? panel_of(q.w) : -1;
            // lengths are taken in units of gs (1 for TF32): r, then, is gs / |x - y|
            const float ig = F16 ? 1.f / gs : 1.f;
            const float2 qx = make_float2(q.x * ig, q.x * ig), qy = make_float2(q.y * ig, q.y * ig);
            const float2 qz = make_float2(q.z * ig, q.z * ig);
            const int um = set_surfaces(b0, nb, Bact, nsurf);
            bool begun = false;
            int4 e_nx = item.y < item.z ? __ldg(ivl + item.y) : make_int4(0, 0, 0, 0);
            for (int iv = item.y; iv < item.z && ok; ++iv) {
                const int4 e = e_nx;
                if (iv + 1 < item.z) e_nx = __ldg(ivl + iv + 1);
                if (!(e.w & um)) continue;
                begun = true;
                const bool on = live && ((e.z >> blk) & 1);   // uniform over the warp but for the tail
                for (int g8 = e.x / kSrc; g8 * kSrc < e.y && ok; ++g8) {
                    // the stage's inputs have landed (and its operands are free: the producer
                    // armed the copies after the stage's previous MMAs completed)
                    const int s = (int)(seq % kStages);
                    if (!warp_wait(smem_addr(&raw_s[s]), (uint32_t)(seq / kStages) & 1u, &abort_s)) {
                        ok = false;
                        break;
                    }
                    unsigned char *stg = tc_smem + s * kStage;
                    // row r of this thread's sources: src[r * kSrc / 4 + quad] (positions are stored
                    // negated; the normals carry dG/dn's scale)
                    constexpr int kPart = H::PART, kRow = kSrc / 4;
                    const float4 *src = (const float4 *)(stg + kOffSrc) + hf * (kPart / 4);
                    float g[kPart], h[kPart];
                    if (on) {
#pragma unroll
                        for (int k4 = 0; k4 < kPart / 4; ++k4) {
                            const float4 px = src[k4], py = src[kRow + k4], pz = src[2 * kRow + k4];
                            const float4 nx = src[3 * kRow + k4], ny = src[4 * kRow + k4], nz = src[5 * kRow + k4];
                            const float4 id = src[6 * kRow + k4];
                            const int pid[4] = {__float_as_int(id.x), __float_as_int(id.y), __float_as_int(id.z),
                                                __float_as_int(id.w)};
#pragma unroll
                            for (int p = 0; p < 2; ++p) {
                                const float2 dx = __fadd2_rn(qx, p ? make_float2(px.z, px.w) : make_float2(px.x, px.y));
                                const float2 dy = __fadd2_rn(qy, p ? make_float2(py.z, py.w) : make_float2(py.x, py.y));
                                const float2 dz = __fadd2_rn(qz, p ? make_float2(pz.z, pz.w) : make_float2(pz.x, pz.y));
                                const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
                                // zero for the target's own panel and for sources outside the range
                                const int k = g8 * kSrc + kPart * hf + 4 * k4 + 2 * p;
                                const float r0 = pid[2 * p] == tp || k < e.x || k >= e.y ? 0.f : rsq(r2.x);
                                const float r1 = pid[2 * p + 1] == tp || k + 1 < e.x || k + 1 >= e.y ? 0.f : rsq(r2.y);
                                const float2 r = make_float2(r0, r1);
                                const float2 dn = __ffma2_rn(dz, p ? make_float2(nz.z, nz.w) : make_float2(nz.x, nz.y),
                                                  __ffma2_rn(dy, p ? make_float2(ny.z, ny.w) : make_float2(ny.x, ny.y),
                                                  __fmul2_rn(dx, p ? make_float2(nx.z, nx.w) : make_float2(nx.x, nx.y))));
                                const float2 t = __fmul2_rn(__fmul2_rn(dn, __fmul2_rn(r, r)), r);
                                g[4 * k4 + 2 * p] = r.x;
                                g[4 * k4 + 2 * p + 1] = r.y;
                                h[4 * k4 + 2 * p] = t.x;
                                h[4 * k4 + 2 * p + 1] = t.y;
                            }
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < kPart; ++k) g[k] = h[k] = 0.f;
                    }
                    unsigned char *bg = stg + kOffG, *bd = stg + kOffD;
                    H::split(g, bg + core_off(tt, hf), bg + kBPart + core_off(tt, hf));
                    H::split(h, bd + core_off(tt, hf), bd + kBPart + core_off(tt, hf));
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();   // one arrival per warp: a thread each would serialise on the barrier
                    if (lane == 0) bar_arrive(smem_addr(&full_s[s]));
                    ++seq;
                    if (pend) ok = drain_acc();   // the previous unit, behind this unit's first stage
                }
            }
            if (ok && pend) ok = drain_acc();     // the previous unit, if this one had no source
            if (!ok) break;
            if (begun) {
                pend = true;
                p_tbase = tbase;
                p_b0 = b0;
                p_nb = nb;
                p_stacked = stacked;
                ++nu;
            }
            __syncwarp();
            if (lane == 0) bar_arrive(smem_addr(&ring_empty[slot]));
        }
        if (ok && pend) drain_acc();
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    if (tid == 0 && abort_s) atomicAdd(error, 1);
}

template <bool F16>
int launch_parts(lspr_ctx *ctx, double *acc, cudaStream_t st, int *counter, int B, int min_rhs) {
    static int smem_set[kSmemDevices] = {};
    using H = P2PShape<F16>;
    Tree &tr = ctx->tree;
    LSPR_TRY(ctx, allow_smem(p2p_tc_kernel<F16>, kSmem, ctx->device, smem_set));
    const int nrc = (B + kRC - 1) / kRC;
    const int64_t Ns = ctx->mesh.Ns, N = ctx->mesh.N, ng = (Ns + H::SRC - 1) / H::SRC;
    LSPR_TRY(ctx, ctx->tcp_img.ensure((size_t)(ng * nrc) * kImgBlock));
    int *mx = (int *)(acc + 4 * N * B) + kCounters + 4 * B;   // cleared with the accumulators
    if (F16) {
        const int S = ctx->mesh.S, nsys = B / S;
        ++ctx->n_launches;
        p2p_max_kernel<<<dim3(4 * std::max(1, ctx->num_sms), (nsys + kMaxSets - 1) / kMaxSets), 256, 0, st>>>(
            N, nsys, S, ctx->xtf.p, tr.tcp_stat.p, mx, ctx->rhs_inv, ctx->rhs_nact, min_rhs);
    }
    ++ctx->n_launches;   // the image; the caller counts the P2P launch
    p2p_image_kernel<F16><<<(unsigned)(ng * nrc), 128, 0, st>>>(Ns, B, nrc, Views<float>::w(ctx), ctx->tcp_img.p,
                                                               ctx->rhs_nact, min_rhs, ctx->mesh.S, tr.tcp_mask.p, mx);
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>(tr.n_tcp_items * nrc, std::max(1, ctx->num_sms)));
    p2p_tc_kernel<F16><<<grid, kTcThreads, kSmem, st>>>(tr.tcp_items.p, tr.n_tcp_items, tr.tcp_ivl.p, B,
                                                       Views<float>::tgt(ctx), N, tr.tcp_src.p, ctx->tcp_img.p, nrc, acc,
                                                       counter, ctx->dev_err.p, ctx->rhs_nact, min_rhs, ctx->mesh.S,
                                                       tr.tcp_gs, tr.tcp_ts, mx);
    LSPR_TRY(ctx, cudaGetLastError());
    return LSPR_OK;
}

}  // namespace

// FP32 tree P2P of B >= 2 right-hand sides on the tensor cores
int p2p_tc_launch(lspr_ctx *ctx, double *acc, cudaStream_t st, int *counter, int B, int min_rhs) {
    Tree &tr = ctx->tree;
    if (!tr.tcp_built) LSPR_TRY_ST(tree_tc_lists(ctx, true));
    if (tr.n_tcp_items == 0) return LSPR_OK;
    if (!ctx->dev_err.p) return LSPR_E_STATE;
    ctx->tc_launched = true;
    return tr.tcp_f16 ? launch_parts<true>(ctx, acc, st, counter, B, min_rhs)
                      : launch_parts<false>(ctx, acc, st, counter, B, min_rhs);
}

}  // namespace lspr
