// Internal declarations of the sm_103a LSPR boundary-element library.
// Layout of device data (all owned by one lspr_ctx):
//   panels    FP64 structure-of-arrays in input order (centroid, normal, area, L, V_ii)
//   sources   Gauss nodes of the far rule, "work order" (input order until a tree
//             is built, Morton order afterwards): position+weight (x,y,z,w_g*A),
//             normal (nx,ny,nz,panel id as int bits) in FP64 and FP32 copies
//   targets   collocation points in work order (x,y,z,panel id as int bits)
//   near CSR  per panel row: the self entry first, then every near-singular panel,
//             with FP64 corrections dV, dK (fine rule minus far rule; self: V_ii, 0)
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "ffloat.cuh"
#include "lspr.h"

// 32-byte aligned four-double vector (CUDA's double4 is deprecated)
struct __align__(32) dbl4 {
    double x, y, z, w;
};
__host__ __device__ inline dbl4 make_dbl4(double x, double y, double z, double w) { return dbl4{x, y, z, w}; }

namespace lspr {

// arithmetic of the far-field kernels
enum Prec { PREC_F32 = 0, PREC_F64 = 1, PREC_FF = 2 };
inline int mode_prec(int mode) {
    return (mode == LSPR_DIRECT_FP64 || mode == LSPR_TREE_FP64) ? PREC_F64
           : (mode == LSPR_DIRECT_FF || mode == LSPR_TREE_FF)   ? PREC_FF
                                                                : PREC_F32;
}
inline bool mode_tree(int mode) { return mode == LSPR_TREE_FP64 || mode == LSPR_TREE_FP32 || mode == LSPR_TREE_FF; }

constexpr double kInv4Pi = 0.079577471545947667884;   // 1 / (4 pi)
constexpr int kTargetBlock = 64;                       // targets per interaction block (2 per lane)
constexpr int kTcGroup = 4;        // target blocks per tensor-core M2P group (256 targets)
// Boxes per tensor-core M2P work unit and sources per P2P unit, at most (tc_unit).  A unit ends with its
// accumulators added in FP64, which no MMA overlaps, so units are long; but a sum of one sign loses a part
// of its last place at every step added in FP32, and the upper limits keep the error of products of smooth
// vectors below that of TF32 parts in units of 32 boxes and 2048 sources (256 stages of 8, still the limit
// with TF32 parts).  81920 panels, P 7, 64 right-hand sides, smooth vectors, M2P on the tensor cores / P2P
// / both: 3.3e-6, 1.7e-6, 4.8e-6 in 4.14 ms; 5.7e-6, 2.6e-6, 8.1e-6 in 4.01 ms with limits of 112 and 4096;
// 4.7e-6, 2.1e-6, 6.6e-6 with TF32 parts.  3072 sources: above TF32 parts at P 8 (1.01 times); 2048: 4.22 ms.
constexpr int kTcSegMin = 32, kTcSegMax = 64;
constexpr int kTcSrcMin = 1024, kTcSrcMax = 2560, kTcSrcMaxTf32 = 2048;
constexpr int kTcSrcRows = 8;      // tensor-core P2P source geometry per stage: rows -x, -y, -z, normal, panel, -
constexpr float kTcP2PRange = 4096.f;   // largest ratio of P2P distances for FP16 parts
constexpr int kTcSurf = 8;         // tensor-core M2P list entry.y: block mask, from this bit the box's surfaces
constexpr int kMaxP = 8;                               // highest Taylor order compiled
constexpr int kMaxDepth = 10;                          // octree levels below the root (10 bits per axis)
constexpr int kMaxNk = 32;
constexpr int kMaxSurfaces = 16;                       // particle + analyte surfaces
// The tensor-core P2P takes products of at least this many right-hand sides (channel sets) in use; fewer
// take the FP32-pipe P2P.  It bounds the weights from the transposed FP32 vectors, which products of one
// system do not form, so it must never take one system's surfaces.
constexpr int kTcP2PMinSets = 24;
static_assert(kTcP2PMinSets > kMaxSurfaces, "the tensor-core P2P needs two systems or more");

// terms of an expansion of order P in the harmonic basis: the multi-indices |k| <= P with k_3 <= 1
__host__ __device__ constexpr int n_terms(int P) { return (P + 1) * (P + 1); }

// Channel sets of a product of K running systems and S surfaces are numbered t K + k (surface t of
// system k), so that the sets of one surface are neighbours: a source or box whose surfaces have no
// set in a chunk of sets contributes zeros to it and is skipped.  A sensor of 145920 panels on three
// surfaces, 32 wavelengths: M2P 10.4 -> 6.15 ms, P2P 14.3 -> 7.3, P2M 2.7 -> 1.08 (the sets of a
// system next to each other put every surface into every chunk).  The mask of the surfaces with a
// set in [b0, b0 + nb) of nsets = K S:
__host__ __device__ inline int set_surfaces(int b0, int nb, int nsets, int S) {
    if (S == 1) return 1;
    const int K = nsets / S, t0 = b0 / K, t1 = (b0 + nb - 1) / K;
    return (2 << t1) - (1 << t0);
}
constexpr int kItemSurf = 8;                 // P2P item.w: bit 0 the own-panel flag, from here on
constexpr int kAllSurf = 0xffff;             // the mask of the surfaces of the item's sources

// ---------------------------------------------------------------- device arrays
// Counts device allocations made through DArr: captured CUDA graphs embed buffer
// addresses and are re-recorded when this number has changed since their recording.
inline std::atomic<uint64_t> g_alloc_generation{0};

template <class T>
struct DArr {
    T *p = nullptr;
    size_t n = 0;      // elements allocated
    DArr() = default;
    DArr(const DArr &) = delete;
    DArr &operator=(const DArr &) = delete;
    ~DArr() { release(); }
    cudaError_t ensure(size_t count) {
        if (count <= n && p) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
        size_t c = count ? count : 1;
        cudaError_t e = cudaMalloc((void **)&p, c * sizeof(T));
        if (e == cudaSuccess) n = c;
        ++g_alloc_generation;
        return e;
    }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        n = 0;
    }
};

// Typed view of a context-owned scratch buffer: the temporaries of the mesh and tree
// builds reuse device memory from call to call instead of allocating and freeing it
// (cudaFree synchronises the device).  Temporaries that are live at the same time use
// different slots.
template <class T>
struct Tmp {
    DArr<unsigned char> *buf;
    T *p = nullptr;
    size_t n = 0;
    explicit Tmp(DArr<unsigned char> &b) : buf(&b) {}
    cudaError_t ensure(size_t count) {
        const cudaError_t e = buf->ensure((count ? count : 1) * sizeof(T));
        if (e == cudaSuccess) {
            p = (T *)buf->p;
            n = count;
        }
        return e;
    }
};
constexpr int kScratchSlots = 16;

struct Mesh {
    bool ready = false;
    int64_t N = 0, nv = 0, Ns = 0;
    int K = 4, Kf = 19, Nk = 9;
    double thr = 0.5;
    double Lmax = 0, rho_max = 0;         // largest L and largest centroid-to-node distance
    DArr<double> verts;                   // [nv*3]
    DArr<int> tris;                       // [N*3]
    DArr<double> cx, cy, cz, nx, ny, nz, area, L, Vself;   // [N]
    int S = 1;                            // surfaces (surface 0: the particle)
    DArr<int> surf;                       // [N] surface of each panel
    // natural-order sources (s = K*i + g) and targets (i)
    DArr<dbl4> src_pos64, src_nrm64;
    DArr<dbl4> tgt64;
    // near CSR
    DArr<int64_t> near_ptr;               // [N+1]
    DArr<int> near_col;                   // [nnz]
    DArr<double> near_dV, near_dK;        // [nnz]
    DArr<float2> near_f32;                // [nnz] (dV, dK) in FP32, for FP32 products
    int64_t nnz = 0;
};

struct WorkOrder {   // sources/targets in the order the far-field kernels walk them
    DArr<dbl4> spos64, snrm64;
    DArr<float4> spos32, snrm32;
    DArr<dbl4> tgt64;
    DArr<float4> tgt32;
    DArr<int> src_panel;   // [Ns]
    DArr<int> tgt_panel;   // [N]
    DArr<ff4> spos_ff, snrm_ff, tgt_ff;   // float-float copies
    DArr<int> tgt_pos;     // [N] work-order position of each panel's target
    DArr<int> src_tblock;  // [Ns] target block holding the source's own panel
};

struct Tree {
    bool ready = false;
    double theta = 0.5;
    int P = 6, Ncrit = 300, NT = 49;
    int64_t nboxes = 0, ntblocks = 0;
    int64_t n_p2p_items = 0, n_m2p_items = 0, n_m2p_pairs = 0, n_p2m_items = 0;
    int64_t p2p_pairs = 0;
    // boxes
    DArr<int> box_beg, box_end, box_child, box_nchild, box_level, box_used;
    DArr<unsigned> box_key;
    DArr<int4> box_node;     // (first child, children, source begin, source end)
    DArr<int> box_surf;      // several surfaces: mask of the surfaces of the box's sources
    DArr<dbl4> box_c64;   // centre (x,y,z), radius r_b
    DArr<float4> box_c32;
    float rho_min = 0.f;     // least scale length of a box's expansion (box_scale)
    // lists
    DArr<int4> p2p_items;    // (target block, source begin, source end, 0)
    DArr<int4> m2p_items;    // (target block, list begin, list end, 0)
    DArr<int> m2p_list;      // box ids
    // the M2P lists of groups of kTcGroup consecutive target blocks (tensor-core M2P): the
    // union of the blocks' lists, sorted by box, with a mask of the blocks that accepted each
    // box, cut into segments
    DArr<int4> tc_items;     // (group, list begin, list end, 0)
    DArr<int2> tc_list;      // (box id, block mask)
    int64_t n_tc_items = 0, n_tc_pairs = 0;
    // the P2P source ranges of the same groups (tensor-core P2P): the union of the blocks'
    // ranges cut at every range end, each piece with the mask of the blocks that sum it
    DArr<int4> tcp_items;    // (group, interval begin, interval end, 0)
    DArr<int4> tcp_ivl;      // (source begin, source end, block mask, surface mask)
    DArr<int> tcp_mask;      // several surfaces: [stage's sources] the surface masks of the ranges that hold them
    DArr<float> tcp_src;     // [stage's sources][kTcSrcRows][sources] their geometry, scaled
    DArr<int> tcp_stat;      // bits of the smallest and largest squared P2P distance, the largest source weight
    bool tcp_f16 = false;    // FP16 parts (16 sources per stage) rather than TF32 (8)
    float tcp_gs = 1.f, tcp_ts = 1.f;   // scales of G and dG/dn
    int64_t n_tcp_items = 0, n_tcp_ivl = 0, n_tcp_sources = 0, n_tcp_stages = 0;   // stages of 16 (TF32: 8) sources
    bool tc_built = false, tcp_built = false;   // the group lists above match the tree
    DArr<int4> p2m_items;    // (leaf, source begin, source end, 0): leaves under an accepted box
    DArr<int> box_parent;    // parent box (-1 for the root)
    // moments [box][NT] x (Vre, Vim, Kre, Kim)
    DArr<float4> mom32;
    DArr<dbl4> mom64;        // FP64 moments; also the accumulation buffer of the float-float ones
    DArr<ff4> mom_ff, box_c_ff;
};

struct DirectItems {
    int64_t n = 0, chunk = 0;   // items, sources per item
    DArr<int2> range;           // per source chunk: first and last target block of its sources' panels
    DArr<int4> items;
};

// An instantiated Arnoldi-cycle graph and what it was recorded for
struct GraphCache {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint64_t key[24] = {0};
    uint64_t use = 0;        // last use, for replacement
    int64_t per_step = 0;    // kernels launched per Arnoldi step (body of the loop)
    int64_t outer = 0;       // kernels launched once per cycle
    void reset() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
        use = 0;
    }
    ~GraphCache() { reset(); }
};

// device state of the Arnoldi cycles of B systems with restart length m
struct ArnoldiBufs {
    DArr<double2> h;        // [B][m+1]  coefficients of one Gram-Schmidt pass
    DArr<double2> hcol;     // [B][m+1]  Hessenberg column being built
    DArr<double2> part;     // [B][m+1][chunks] partial inner products
    DArr<double> npart;     // [B][blocks] partial squared norms
    DArr<double> nrm;       // [B] norm of the new basis vector / of the residual
    DArr<double> npart0;    // [B][chunks] partial squared norms of A z before orthogonalisation
    DArr<int> reorth;       // [B] 1: the step takes the second Gram-Schmidt pass
    DArr<double2> H;        // [B][m+1][m] rotated Hessenberg matrix (R)
    DArr<double> cs;        // [B][m] Givens cosines
    DArr<double2> sn;       // [B][m] Givens sines
    DArr<double2> g;        // [B][m+1] rotated right-hand side beta e_1
    DArr<double2> y;        // [B][m] update coefficients
    DArr<double> res;       // [B] residual estimate |g_{j+1}|
    DArr<double> bn;        // [B] reference norm of the relative residual
    DArr<double> par;       // [2] tolerance, iteration limit
    DArr<unsigned> tick;    // [2B + 1] last-block tickets
    DArr<int> ctl;          // [1 + 3B] current column j, active[B], jb[B], iters[B]
    DArr<int> rmap;         // [2B + 2] running systems packed first: slot -> b, b -> slot, count, sets
    DArr<float4> hff;       // [B][m+1]  h in float-float (re.hi, im.hi, re.lo, im.lo)
    DArr<float4> yff;       // [B][m]    update coefficients in float-float
    DArr<float2> ninv;      // [B] 1 / ||w|| in float-float
    DArr<double> vinv;      // [N] 1 / V_ii (preconditioner)
    DArr<double2> pq;       // [B][S] 1 / (1 + s) (preconditioner)
    DArr<float2> vinvf;     // [N] vinv in float-float
    DArr<float4> pqf;       // [2][B][S] pq and s in float-float
    DArr<int> go;           // host-driven cycles: the loop condition
    DArr<unsigned long long> stats;   // [4] work counters (lspr_get_arnoldi_stats)
};

constexpr int kTimerSlots = 16;

struct Timing {
    bool enabled = false;
    double ms[kTimerSlots] = {0};
    int64_t launches[kTimerSlots] = {0};
    int64_t rhs[kTimerSlots] = {0};    // right-hand sides (channel sets) summed over the launches
    std::vector<cudaEvent_t> pool;
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> pending;
    size_t used = 0;
};

enum TimerSlot {
    T_P2P = 0, T_M2P = 1, T_P2M = 2, T_NEAR = 3, T_GMRES = 4, T_TREE = 5, T_MESH = 6, T_OTHER = 7,
    T_P2P64 = 8, T_M2P64 = 9, T_P2M64 = 10, T_WEIGHTS = 11, T_P2PFF = 12, T_M2PFF = 13, T_P2MFF = 14
};

}  // namespace lspr

struct lspr_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t side = nullptr;       // second stream: P2P overlaps P2M -> M2P
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    lspr::DArr<int> counters;          // selftest results
    int num_sms = 0;
    lspr::Mesh mesh;
    lspr::WorkOrder wo;
    lspr::Tree tree;
    lspr::DirectItems direct;          // one right-hand side
    lspr::DirectItems direct_multi;    // several: fewer, longer items (n = 0: those of direct)
    lspr::Timing timing;
    // per-matvec scratch
    lspr::DArr<double> acc;            // [N][B][4]: V re/im, K re/im (far part), then the work-item counters
    lspr::DArr<float4> w32;            // [Ns] source weights
    lspr::DArr<dbl4> w64;
    lspr::DArr<ff4> w_ff;
    lspr::DArr<double2> xbuf, ybuf;    // staging for host matvec
    lspr::DArr<double2> xt;            // [2N][B] transposed right-hand sides of a product
    lspr::DArr<float2> xtf;            // [2N][B] the same in FP32 (FP32 products)
    lspr::DArr<double2> sbuf;
    // solver scratch
    lspr::DArr<float4> gm_V;   // Krylov basis, float-float complex entries
    lspr::DArr<double2> gm_w, gm_z, gm_x, gm_b, gm_r;
    lspr::DArr<double> gm_bnorm, gm_dpart;
    lspr::DArr<double2> gm_s, gm_vinc, gm_eps;
    lspr::DArr<double> gm_out;         // dipole + sigma results
    lspr::DArr<double2> gm_dx;         // refinement correction
    lspr::DArr<int> gm_rmap;           // [2B + 2] systems of a refinement product (packing map)
    lspr::DArr<double> gm_dippart, gm_lambda;
    lspr::DArr<unsigned char> scratch[lspr::kScratchSlots];   // see lspr::Tmp
    // device-driven Arnoldi cycles (a CUDA graph per configuration, gmres_graph.cu)
    bool use_graphs = true;
    int tensor_cores = 1;              // tcgen05 for B >= 2 in FP32: bit 0 M2P, bit 1 P2P
    lspr::DArr<unsigned char> tc_img;  // split moments in tensor-core operand layout
    lspr::DArr<unsigned char> tcp_img; // split source weights in tensor-core operand layout
    lspr::DArr<int> dev_err;           // [0] bounded device waits that ran out (never reset);
                                       // [1] failure-path check: tensor-core kernels give up at once
    int dev_err_seen = 0;              // [0] as last reported by a status (LSPR_E_TIMEOUT)
    int *host_err = nullptr;           // pinned copy of [0]
    bool tc_launched = false;          // a tensor-core kernel was launched since [0] was last read
    // point charges inside the surfaces (lspr_set_charges): (x, y, z, q) and the surface of each
    lspr::DArr<dbl4> charges;
    lspr::DArr<int> charge_surf;
    int64_t nq = 0;
    int max_charge_surf = -1;
    lspr::DArr<double> coul;           // [N] sum_k q_k / |c_i - r_k| over the charges of i's surface
    cudaStream_t gstream = nullptr;    // private recording/launch stream
    cudaEvent_t ev_g0 = nullptr, ev_g1 = nullptr;
    lspr::GraphCache gcache[2];
    lspr::ArnoldiBufs arn;
    // right-hand sides in use while recording an Arnoldi step (null: all B): slot -> system
    // map, system -> slot map (-1: converged), and the number of channel sets in use (running
    // systems x surfaces); the far-field kernels work on the first *rhs_nact sets only
    const int *rhs_map = nullptr, *rhs_inv = nullptr, *rhs_nact = nullptr;
    int timing_sets = -1;   // host copy of *rhs_nact for the per-launch work count of timing
    int64_t graph_cycles = 0, graph_recordings = 0;
    // last error text
    std::string last_error;
    int64_t matvec_count = 0;
    int64_t n_launches = 0;            // kernels launched by this context
};

namespace lspr {

// the direct-mode items of a product of BS channel sets
inline const DirectItems &direct_items(const lspr_ctx *c, int64_t BS) {
    return BS > 1 && c->direct_multi.n ? c->direct_multi : c->direct;
}

// -------------------------------------------------------------- error helpers
int cuda_status(lspr_ctx *ctx, cudaError_t e, const char *what);
// LSPR_E_TIMEOUT in place of rc (LSPR_OK or LSPR_E_NOT_CONVERGED) when a bounded device wait ran
// out since the last status that reported one; call with the context's stream synchronised
int timeout_status(lspr_ctx *ctx, int rc);
// the same for a product whose stream is not synchronised yet: the count is fetched behind the
// product's kernels (only when a kernel with bounded waits was launched) and the stream synchronised
int finish_status(lspr_ctx *ctx);
#define LSPR_TRY(ctx, expr)                                              \
    do {                                                                 \
        cudaError_t e__ = (expr);                                        \
        if (e__ != cudaSuccess) return ::lspr::cuda_status(ctx, e__, #expr); \
    } while (0)
#define LSPR_TRY_ST(expr)             \
    do {                              \
        int s__ = (expr);             \
        if (s__ != LSPR_OK) return s__; \
    } while (0)

// timing helpers (no-ops unless enabled)
void timer_begin(lspr_ctx *ctx, int slot, cudaEvent_t *ev);
void timer_end(lspr_ctx *ctx, int slot, cudaEvent_t ev);
void timer_begin_on(lspr_ctx *ctx, int slot, cudaEvent_t *ev, cudaStream_t st);
void timer_end_on(lspr_ctx *ctx, int slot, cudaEvent_t ev, cudaStream_t st);
void timer_collect(lspr_ctx *ctx);
// channel sets a timed far-field launch works on: the packed count when the host knows it
// (timing_sets >= 0: host-driven Arnoldi steps and refinement products), else all B
inline void timer_rhs(lspr_ctx *ctx, int slot, int64_t B) {
    if (ctx->timing.enabled) ctx->timing.rhs[slot] += ctx->timing_sets >= 0 ? std::min<int64_t>(ctx->timing_sets, B) : B;
}

inline unsigned grid_for(int64_t n, int block) { return (unsigned)((n + block - 1) / block); }

// ------------------------------------------------------------ mesh.cu
// surf: [ntri] surface index of each panel in [0, nsurf) (null: one surface)
int mesh_build(lspr_ctx *ctx, const double *verts, int64_t nv, const int *tris, int64_t ntri, const int *surf,
               int nsurf, int on_device,
               const lspr_quad_opts &q);
// natural-order work arrays (direct mode)
int workorder_natural(lspr_ctx *ctx);

// ------------------------------------------------------------ tree.cu
// A kernel's dynamic shared memory above 48 KB is opted into on every device it runs on:
// set[d] holds the size already allowed on device d (devices past the table set it each call).
constexpr int kSmemDevices = 64;
template <class K>
inline cudaError_t allow_smem(K kernel, int bytes, int device, int *set) {
    const bool tracked = device >= 0 && device < kSmemDevices;
    if (tracked && set[device] >= bytes) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && tracked) set[device] = bytes;
    return e;
}

int tree_build(lspr_ctx *ctx, double theta, int P, int Ncrit);
// out = (lo[3], hi[3]) of the points a and b; part: 6 kBoxBlocks doubles of scratch
constexpr int kBoxBlocks = 128;
int launch_bbox(lspr_ctx *ctx, const dbl4 *a, int64_t na, const dbl4 *b, int64_t nb, double *part, double *out);
int tree_tc_lists(lspr_ctx *ctx, bool p2p);
int selftest_wait_timeout(lspr_ctx *ctx, int32_t *result);
// stable LSD radix sort of (keys, vals) on the context's stream (bits: key width)
// total: 256 ints
int radix_sort(lspr_ctx *ctx, unsigned *keys, int *vals, unsigned *ktmp, int *vals_tmp, int64_t n, int bits, int *hist,
               int *total);
int64_t radix_sort_scratch_ints(int64_t n);   // ints needed by hist
// 10-bit coordinate -> every third bit (Morton interleave helper)
__device__ __forceinline__ unsigned spread10(unsigned v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// ------------------------------------------------------------ farfield.cu
// accumulate far parts (coarse rule everywhere except own panel) into acc[N][4]
// B right-hand sides: weights [source][B], accumulators acc [panel][B][4]
int launch_p2p(lspr_ctx *ctx, int prec, const int4 *items, int64_t nitems, double *acc, cudaStream_t st,
               int *counter, int B);
// the moments are zero on entry (launch_weights clears them)
int launch_p2m(lspr_ctx *ctx, int prec, int B);
// behind the accumulators of a product, cleared with them: the work-item counters, then per channel set
// and component (re and im of both layers) the largest magnitudes that scale the tensor-core operands
constexpr int kCounters = 8;
inline int64_t acc_tail_ints(int64_t BS) { return kCounters + 8 * BS; }   // M2P's, then P2P's
int launch_m2p(lspr_ctx *ctx, int prec, double *acc, int *counter, int B);
// float-float copies of the work-order geometry / box centres
int launch_ff_geometry(lspr_ctx *ctx);
int launch_ff_boxes(lspr_ctx *ctx);
// item.w = 1 where a P2P item may contain sources of its own target block's panels: exactly, or for
// the direct-mode lists from the range of target blocks that each chunk of sources belongs to
int launch_item_flags(lspr_ctx *ctx, int4 *items, int64_t nitems);
int launch_direct_flags(lspr_ctx *ctx);
// xt: x transposed to [2N][B] (B > 1), or null
// S > 1 surfaces: B x S channel sets, weights of set (b, t) masked to the sources of surface t
// x [B][2N]; xt: its transposed FP64 copy [2N][B] or null; xtf: its transposed FP32 copy
// (FP32 products of several right-hand sides) or null.  Clears the accumulators and counters of the
// product and, with tree set, its moments.
int launch_weights(lspr_ctx *ctx, int prec, const double2 *x, const double2 *xt, int64_t N, int B, int S,
                   const float2 *xtf, bool tree);
int launch_weights_fp32_raw(cudaStream_t st, int64_t Ns, int64_t N, const dbl4 *spos64, const int *src_panel,
                            const double2 *x, float4 *w);
int launch_p2p_fp32_raw(cudaStream_t st, const int4 *items, int64_t nitems, const float4 *tgt, int64_t ntgt,
                        const float4 *spos, const float4 *snrm, const float4 *w, double *acc);

// ------------------------------------------------------------ solve.cu
// y = A(s) x for B right-hand sides, x and y device [B][2N] complex; x null: an FP32 product of several
// right-hand sides on one surface whose transposed vectors are in xtf already
int apply_operator(lspr_ctx *ctx, int mode, const double2 *x, double2 *y, const double2 *s, int B);
// layer potentials without the block assembly: out[i] = (V dphi)_i, (K phi)_i
// per source surface t (S of them): Vd[t * N + i] = (V dphi)_t, Kp[t * N + i] = (K phi)_t
int layer_potentials(lspr_ctx *ctx, int mode, const double2 *x, double2 *Vd, double2 *Kp);
int solve_impl(lspr_ctx *ctx, const double *eps_in, double eps_out_re, double eps_out_im, const double *E0,
               const double *lambda_nm, int B, const lspr_solve_opts &o, double *dipole_out, double *sigma_out,
               lspr_solve_stats *st);

// ------------------------------------------------------------ gmres_graph.cu
constexpr int kMaxRestart = 512;   // longest Arnoldi cycle (restart length m)
// Restarted GMRES(m) for B systems A(s_b) x_b = b_b whose Arnoldi cycles each run as one
// CUDA graph launch (a device-side loop over the steps), or host-driven launches of the
// same kernels without graphs or with per-kernel timing.  x_zero: x holds zeros on entry
// (the first residual is b without a matrix-vector product).  trust_estimate: return
// after a cycle whose recurrence residual estimates meet tol, without the explicit
// residual (for inner solves whose caller forms the residual itself).  iters/relres
// receive the steps taken and the last relative residual (explicit or estimated) per
// system.
int gmres_graph_solve(lspr_ctx *ctx, int mode, int B, int m, int maxiter, double tol, const double2 *s_d,
                      const double2 *b_d, double2 *x_d, bool x_zero, bool trust_estimate, std::vector<int> &iters,
                      std::vector<double> &relres, const std::vector<double> &bnorm);

}  // namespace lspr
