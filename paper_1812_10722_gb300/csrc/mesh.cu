// Geometry and quadrature precompute (Sec. II.C of the paper):
//   panel centroids / normals / areas / L = sqrt(2A), Gauss-node sources of the
//   far rule, semi-analytical self integrals, the near-singular pair list and
//   its FP64 corrections.  Everything here depends only on the mesh and the
//   quadrature options, so it runs once per geometry.
#include <algorithm>
#include <cmath>

#include "lspr_internal.cuh"
#include "rsq.cuh"

namespace lspr {

// ----------------------------------------------------------------------------
// Dunavant's symmetric triangle rules (Dunavant 1985), barycentric points and
// weights normalised to sum 1.  Orbit form: type 0 centroid, type 1 (a,b,b)
// with b = (1-a)/2, type 2 all permutations of (a, b, 1-a-b).
// ----------------------------------------------------------------------------
struct Orbit {
    int type;
    double a, b, w;
};
static const Orbit kR1[] = {{0, 0., 0., 1.0}};
static const Orbit kR3[] = {{1, 0.666666666666667, 0., 0.333333333333333}};
static const Orbit kR4[] = {{0, 0., 0., -0.5625}, {1, 0.6, 0., 0.520833333333333}};
static const Orbit kR19[] = {{0, 0., 0., 0.097135796282799},
                             {1, 0.020634961602525, 0., 0.031334700227139},
                             {1, 0.125820817014127, 0., 0.077827541004774},
                             {1, 0.623592928761935, 0., 0.079647738927210},
                             {1, 0.910540973211095, 0., 0.025577675658698},
                             {2, 0.036838412054736, 0.221962989160766, 0.043283539377289}};
static const Orbit kR25[] = {{0, 0., 0., 0.090817990382754},
                             {1, 0.028844733232685, 0., 0.036725957756467},
                             {1, 0.781036849029926, 0., 0.045321059435528},
                             {2, 0.141707219414880, 0.307939838764121, 0.072757916845420},
                             {2, 0.025003534762686, 0.246672560639903, 0.028327242531057},
                             {2, 0.009540815400299, 0.066803251012200, 0.009421666963733}};
static const Orbit kR37[] = {{0, 0., 0., 0.052520923400802},
                             {1, 0.009903630120591, 0., 0.011280145209330},
                             {1, 0.062566729780852, 0., 0.031423518362454},
                             {1, 0.170957326397447, 0., 0.047072502504194},
                             {1, 0.541200855914337, 0., 0.047363586536355},
                             {1, 0.771151009607340, 0., 0.031167529045794},
                             {1, 0.950377217273082, 0., 0.007975771465074},
                             {2, 0.094853828379579, 0.268794997058761, 0.036848402728732},
                             {2, 0.018100773278807, 0.291730066734288, 0.017401463303822},
                             {2, 0.022233076674090, 0.126357385491669, 0.015521786839045}};

// fills bary[3*K], w[K]; returns the point count or -1
static int expand_rule(int K, double *bary, double *w) {
    const Orbit *o = nullptr;
    int no = 0;
    if (K == 1) { o = kR1; no = 1; }
    else if (K == 3) { o = kR3; no = 1; }
    else if (K == 4) { o = kR4; no = 2; }
    else if (K == 19) { o = kR19; no = 6; }
    else if (K == 25) { o = kR25; no = 6; }
    else if (K == 37) { o = kR37; no = 10; }
    else return -1;
    int k = 0;
    for (int r = 0; r < no; ++r) {
        const double a = o[r].a;
        if (o[r].type == 0) {
            bary[3 * k] = bary[3 * k + 1] = bary[3 * k + 2] = 1.0 / 3.0;
            w[k++] = o[r].w;
        } else if (o[r].type == 1) {
            const double b = 0.5 * (1.0 - a);
            const double pts[3][3] = {{a, b, b}, {b, a, b}, {b, b, a}};
            for (auto &p : pts) {
                bary[3 * k] = p[0]; bary[3 * k + 1] = p[1]; bary[3 * k + 2] = p[2];
                w[k++] = o[r].w;
            }
        } else {
            const double b = o[r].b, c = 1.0 - a - b;
            const double pts[6][3] = {{a, b, c}, {a, c, b}, {b, a, c}, {b, c, a}, {c, a, b}, {c, b, a}};
            for (auto &p : pts) {
                bary[3 * k] = p[0]; bary[3 * k + 1] = p[1]; bary[3 * k + 2] = p[2];
                w[k++] = o[r].w;
            }
        }
    }
    return k;
}

// Gauss-Legendre nodes/weights on [-1, 1] by Newton iteration on P_n.
static void gauss_legendre(int n, double *x, double *w) {
    for (int i = 0; i < n; ++i) {
        double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        double pp = 0;
        for (int it = 0; it < 100; ++it) {
            double p1 = 1.0, p2 = 0.0;
            for (int j = 1; j <= n; ++j) {
                double p3 = p2;
                p2 = p1;
                p1 = ((2.0 * j - 1.0) * z * p2 - (j - 1.0) * p3) / j;
            }
            pp = n * (z * p1 - p2) / (z * z - 1.0);
            double dz = p1 / pp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * pp * pp);
    }
}

__constant__ double c_far_bary[37 * 3];
__constant__ double c_far_w[37];
__constant__ double c_fine_bary[37 * 3];
__constant__ double c_fine_w[37];
__constant__ double c_gl_x[kMaxNk];
__constant__ double c_gl_w[kMaxNk];

// ----------------------------------------------------------------------------
// Panel geometry with every FP64 operation rounded on its own (no contraction),
// so centroids, areas and L are reproducible bit for bit on any IEEE machine;
// the near-singular classification depends on them.
// ----------------------------------------------------------------------------
__global__ void panel_kernel(const double *__restrict__ verts, const int *__restrict__ tris, int64_t N, int64_t nv,
                             double *cx, double *cy, double *cz, double *nx, double *ny, double *nz, double *area,
                             double *L, int *bad) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    int i0 = tris[3 * i], i1 = tris[3 * i + 1], i2 = tris[3 * i + 2];
    if (i0 < 0 || i1 < 0 || i2 < 0 || i0 >= nv || i1 >= nv || i2 >= nv) {
        atomicOr(bad, 1);
        return;
    }
    double v[3][3];
    for (int d = 0; d < 3; ++d) {
        v[0][d] = verts[3 * (int64_t)i0 + d];
        v[1][d] = verts[3 * (int64_t)i1 + d];
        v[2][d] = verts[3 * (int64_t)i2 + d];
    }
    double e1[3], e2[3];
    for (int d = 0; d < 3; ++d) {
        e1[d] = __dsub_rn(v[1][d], v[0][d]);
        e2[d] = __dsub_rn(v[2][d], v[0][d]);
    }
    double c0 = __dsub_rn(__dmul_rn(e1[1], e2[2]), __dmul_rn(e1[2], e2[1]));
    double c1 = __dsub_rn(__dmul_rn(e1[2], e2[0]), __dmul_rn(e1[0], e2[2]));
    double c2 = __dsub_rn(__dmul_rn(e1[0], e2[1]), __dmul_rn(e1[1], e2[0]));
    double nc = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(c0, c0), __dmul_rn(c1, c1)), __dmul_rn(c2, c2)));
    if (!(nc > 0.0) || !isfinite(nc)) {
        atomicOr(bad, 2);
        nc = 1.0;
    }
    nx[i] = __ddiv_rn(c0, nc);
    ny[i] = __ddiv_rn(c1, nc);
    nz[i] = __ddiv_rn(c2, nc);
    cx[i] = __ddiv_rn(__dadd_rn(__dadd_rn(v[0][0], v[1][0]), v[2][0]), 3.0);
    cy[i] = __ddiv_rn(__dadd_rn(__dadd_rn(v[0][1], v[1][1]), v[2][1]), 3.0);
    cz[i] = __ddiv_rn(__dadd_rn(__dadd_rn(v[0][2], v[1][2]), v[2][2]), 3.0);
    double A = __dmul_rn(0.5, nc);
    area[i] = A;
    L[i] = __dsqrt_rn(__dmul_rn(2.0, A));
}

__device__ __forceinline__ void atomic_max_pos(double *addr, double v) {
    // non-negative doubles order like their bit patterns
    atomicMax((unsigned long long *)addr, (unsigned long long)__double_as_longlong(v));
}

// the warp's largest v (every lane of the block takes part)
__device__ __forceinline__ void warp_max_pos(double *addr, double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) atomic_max_pos(addr, v);
}

// Far-rule Gauss nodes in natural order s = K*i + g: position, w_g*A_i, normal, panel id.
__global__ void sources_kernel(const double *__restrict__ verts, const int *__restrict__ tris, int64_t N, int K,
                               const double *area, const double *nx, const double *ny, const double *nz,
                               const double *cx, const double *cy, const double *cz, dbl4 *pos, dbl4 *nrm,
                               dbl4 *tgt, double *rho_max, double *L_max, const double *L, const int *bad) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (*bad & 1) return;   // a vertex index out of range (the panel kernel found it)
    const bool live = s < N * K;
    if (!live) s = N * K - 1;   // repeats the last node, which changes no maximum
    int64_t i = s / K;
    int g = (int)(s - i * K);
    double y[3];
    const int *t = tris + 3 * i;
    for (int d = 0; d < 3; ++d)
        y[d] = c_far_bary[3 * g] * verts[3 * (int64_t)t[0] + d] + c_far_bary[3 * g + 1] * verts[3 * (int64_t)t[1] + d] +
               c_far_bary[3 * g + 2] * verts[3 * (int64_t)t[2] + d];
    if (live) {
        pos[s] = make_dbl4(y[0], y[1], y[2], c_far_w[g] * area[i]);
        nrm[s] = make_dbl4(nx[i], ny[i], nz[i], (double)i);
        if (g == 0) tgt[i] = make_dbl4(cx[i], cy[i], cz[i], (double)i);
    }
    const double dx = y[0] - cx[i], dy = y[1] - cy[i], dz = y[2] - cz[i];
    // one atomic per warp and maximum (one per node: 327 us at 327680 nodes, all on one address)
    warp_max_pos(rho_max, sqrt(dx * dx + dy * dy + dz * dz));
    warp_max_pos(L_max, L[i]);
}

// Semi-analytical singular integral: for x = centroid of panel i, the panel
// is split at x into three triangles over its edges.  In polar coordinates about
// x the radial integral of 1/rho * rho is exact (the distance to the edge,
// h / cos(phi)); the angle from phi_a to phi_b is integrated by N_k-point
// Gauss-Legendre, i.e. N_k nodes on each edge.
__global__ void self_kernel(const double *__restrict__ verts, const int *__restrict__ tris, int64_t N, int Nk,
                            const double *cx, const double *cy, const double *cz, double *Vself, const int *bad) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N || (*bad & 1)) return;
    const double x[3] = {cx[i], cy[i], cz[i]};
    double v[3][3];
    for (int k = 0; k < 3; ++k)
        for (int d = 0; d < 3; ++d) v[k][d] = verts[3 * (int64_t)tris[3 * i + k] + d];
    double sum = 0.0;
    for (int e = 0; e < 3; ++e) {
        const double *a = v[e], *b = v[(e + 1) % 3];
        double t[3], ax[3];
        double len = 0;
        for (int d = 0; d < 3; ++d) {
            t[d] = b[d] - a[d];
            len += t[d] * t[d];
        }
        len = sqrt(len);
        double sa = 0, sb = 0;
        for (int d = 0; d < 3; ++d) {
            t[d] /= len;
            ax[d] = a[d] - x[d];
            sa += ax[d] * t[d];
            sb += (b[d] - x[d]) * t[d];
        }
        double h2 = 0;
        for (int d = 0; d < 3; ++d) {
            double p = ax[d] - sa * t[d];
            h2 += p * p;
        }
        double h = sqrt(h2);
        if (!(h > 0)) continue;
        double pa = atan2(sa, h), pb = atan2(sb, h);
        double mid = 0.5 * (pa + pb), half = 0.5 * (pb - pa);
        double q = 0;
        for (int k = 0; k < Nk; ++k) q += c_gl_w[k] / cos(mid + half * c_gl_x[k]);
        sum += h * half * q;
    }
    Vself[i] = sum * kInv4Pi;
}

// ----------------------------------------------------------------------------
// Near-singular decision: the FP64 test L_j / |c_i - c_j| >= threshold with every
// operation rounded separately (reproducible on any IEEE machine).
// ----------------------------------------------------------------------------
__device__ __forceinline__ bool near_exact(double xi, double yi, double zi, double xj, double yj, double zj,
                                           double Lj, double thr) {
    double dx = __dsub_rn(xi, xj), dy = __dsub_rn(yi, yj), dz = __dsub_rn(zi, zj);
    double dist = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
    return __ddiv_rn(Lj, dist) >= thr;
}

// ----------------------------------------------------------------------------
// Cell list for the near-singular search: cubic cells of edge h >= L_max/threshold,
// panels sorted by the Morton key of the cell holding their centroid.  Every panel
// j with L_j/|c_i - c_j| >= threshold lies within L_max/threshold of c_i, hence in
// one of the 27 cells around c_i's cell.  Cell coordinates come from the same FP64
// expression for keys and queries.
// ----------------------------------------------------------------------------
__device__ __forceinline__ int cell_coord(double c, double lo, double inv_h) {
    const double u = floor((c - lo) * inv_h);
    return (int)fmin(1023.0, fmax(0.0, u));
}

__device__ __forceinline__ unsigned cell_key(int ix, int iy, int iz) {
    return (spread10((unsigned)ix) << 2) | (spread10((unsigned)iy) << 1) | spread10((unsigned)iz);
}

__global__ void cell_key_kernel(int64_t N, const double *__restrict__ cx, const double *__restrict__ cy,
                                const double *__restrict__ cz, const double *__restrict__ L, double thr,
                                const double *grid /* lo[3], 1/h */, unsigned *keys, int *vals, float4 *cf) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    cf[i] = make_float4((float)cx[i], (float)cy[i], (float)cz[i], (float)(L[i] / thr));
    keys[i] = cell_key(cell_coord(cx[i], grid[0], grid[3]), cell_coord(cy[i], grid[1], grid[3]),
                       cell_coord(cz[i], grid[2], grid[3]));
    vals[i] = (int)i;
}

__device__ __forceinline__ int lower_bound_u(const unsigned *a, int n, unsigned v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Near decision from FP32 copies when the FP32 distance is clearly inside or outside
// L_j/threshold, else the exact FP64 test.  band bounds |d32 - d| + |r32 - r|: FP32
// rounding of the coordinates (2^-24 |c| each) and of the arithmetic.
__device__ __forceinline__ bool near_decide(const float4 &fi, const float4 &fj, float band, double xi, double yi,
                                            double zi, int j, const double *__restrict__ cx,
                                            const double *__restrict__ cy, const double *__restrict__ cz,
                                            const double *__restrict__ L, double thr) {
    const float dx = fi.x - fj.x, dy = fi.y - fj.y, dz = fi.z - fj.z;
    const float d2 = dx * dx + dy * dy + dz * dz;
    const float r = fj.w, lo = fmaxf(r - band, 0.f), hi = r + band;
    if (d2 < lo * lo) return true;
    if (d2 > hi * hi) return false;
    return near_exact(xi, yi, zi, cx[j], cy[j], cz[j], L[j], thr);
}

// One warp per slice of up to kCellTargets panels of an occupied cell: lane c < 27 searches neighbour
// cell c once for all the slice's targets; the neighbours' panels, in cell order, are the candidates.
// Each lane holds one candidate of a chunk of 32 and tests it against the targets in turn, a ballot
// counts the hits.  A row is laid out as the self entry, then the hits of cell 0, 1, ... in sorted order.
// Bound by the searches' latency where cells hold few panels: 140 us for both passes at 81920 panels,
// 317 with a warp (and its searches) per target.  Cells are sized by the largest panel, so beside a few
// large panels, or at a small threshold, thousands of panels share a cell and a slice's chain of tests
// sets the time.  Whole uploads of 20480 panels beside 20 large ones: 5.7 ms in slices of 16, 8.2 of
// 32, 15.4 of 64, 3630 with a warp per cell, 58.7 with a warp per target; 5120 panels at threshold 0.1:
// 3.6, 4.2, 5.4, 12.0, 4.6; a uniform mesh of 81920 2.40 in all three.
constexpr int kCellTargets = 16;   // targets of a slice
constexpr int kCellWarps = 4;
template <bool FILL>
__global__ void __launch_bounds__(kCellWarps * 32)
    near_cells_kernel(int64_t N, const double *__restrict__ cx, const double *__restrict__ cy,
                      const double *__restrict__ cz, const double *__restrict__ L, double thr, const double *grid,
                      const unsigned *__restrict__ skeys, const int *__restrict__ sidx, const float4 *__restrict__ cf,
                      int64_t *count, const int64_t *ptr, int *col, int *row) {
    __shared__ int hits[kCellWarps][kCellTargets];
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    int *hit = hits[threadIdx.x >> 5];
    if (k >= N) return;
    const unsigned mykey = skeys[k];
    // the first panel of a slice of its cell?
    int t0 = 0;
    if (k > 0 && skeys[k - 1] == mykey) {
        if (k < kCellTargets || skeys[k - kCellTargets] != mykey) return;
        t0 = (int)k - lower_bound_u(skeys, (int)k, mykey);
        if (t0 % kCellTargets) return;
    }
    const float cmax = (float)grid[4];
    const int i0 = sidx[k];
    const int ix = cell_coord(cx[i0], grid[0], grid[3]), iy = cell_coord(cy[i0], grid[1], grid[3]),
              iz = cell_coord(cz[i0], grid[2], grid[3]);
    int k0 = 0, len = 0;
    if (lane < 27) {
        const int qx = ix + lane % 3 - 1, qy = iy + (lane / 3) % 3 - 1, qz = iz + lane / 9 - 1;
        if (qx >= 0 && qy >= 0 && qz >= 0 && qx <= 1023 && qy <= 1023 && qz <= 1023) {
            const unsigned key = cell_key(qx, qy, qz);
            k0 = lower_bound_u(skeys, (int)N, key);
            if (k0 < N && skeys[k0] == key) len = lower_bound_u(skeys, (int)N, key + 1) - k0;
        }
    }
    int pre = len;   // inclusive scan: candidates up to and including this lane's cell
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, pre, o);
        if (lane >= o) pre += v;
    }
    const int total = __shfl_sync(0xffffffffu, pre, 31);
    const int mine = __shfl_sync(0xffffffffu, len, 13);   // the cell itself (offsets 0, 0, 0)
    const int nt = min(kCellTargets, mine - t0);
    for (int t = lane; t < nt; t += 32) hit[t] = 0;
    __syncwarp();
    for (int c0 = 0; c0 < total; c0 += 32) {
        const int c = c0 + lane;
        // the cell that holds candidate c: the first lane whose inclusive count exceeds it
        int lo = 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int v = __shfl_sync(0xffffffffu, pre, lo + o - 1);
            if (v <= c) lo += o;
        }
        lo = min(lo, 31);
        const int cb = __shfl_sync(0xffffffffu, k0, lo), cp = __shfl_sync(0xffffffffu, pre - len, lo);
        int j = -1;
        float4 fj = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < total) {
            j = sidx[cb + (c - cp)];
            fj = cf[j];
        }
        for (int t = 0; t < nt; ++t) {
            const int i = sidx[k + t];
            bool near = false;
            if (j >= 0 && j != i)
                near = near_decide(cf[i], fj, 1e-6f * fj.w + 5e-7f * cmax, cx[i], cy[i], cz[i], j, cx, cy, cz, L, thr);
            const unsigned m = __ballot_sync(0xffffffffu, near);
            const int run = hit[t];
            if (FILL && near) {
                const int64_t out = ptr[i] + 1 + run + __popc(m & ((1u << lane) - 1u));
                col[out] = j;
                row[out] = i;
            }
            __syncwarp();
            if (lane == 0) hit[t] = run + __popc(m);
            __syncwarp();
        }
    }
    for (int t = lane; t < nt; t += 32) {
        const int i = sidx[k + t];
        if (FILL) {
            col[ptr[i]] = i;   // self entry first
            row[ptr[i]] = i;
        } else {
            count[i] = hit[t] + 1;
        }
    }
}

// exclusive scan of n int64 counts into ptr[0..n], single block, four counts per thread and step
__global__ void __launch_bounds__(1024) scan_kernel(const int64_t *__restrict__ in, int64_t n, int64_t *out) {
    __shared__ int64_t sh[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int64_t run = 0;
    for (int64_t base = 0; base < n; base += 4096) {
        const int64_t i = base + 4 * t;
        int64_t v[4], s = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = i + q < n ? in[i + q] : 0;
            s += v[q];
        }
        int64_t inc = s;
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
        int64_t e = run + (warp ? sh[warp - 1] : 0) + inc - s;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (i + q < n) out[i + q] = e;
            e += v[q];
        }
        run += sh[31];
        __syncthreads();
    }
    if (t == 0) out[n] = run;
}

// FP32 copies (dV, dK) of the near-field corrections, read by the FP32 products of several
// right-hand sides
__global__ void near_f32_kernel(int64_t nnz, const double *__restrict__ dV, const double *__restrict__ dK,
                                float2 *__restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < nnz) out[e] = make_float2((float)dV[e], (float)dK[e]);
}

// Per near pair: dV, dK = (K_fine rule - far rule) over panel j seen from c_i,
// and for the self entry V_ii (the far-field kernels skip a panel's own nodes).
// FP64-pipe bound (23 nodes per pair): the node's offset is taken from the panel's edges (d = w -
// b_1 e_1 - b_2 e_2 with w = x - v_0), (x - y).n = w.n is the same at every node of a flat panel,
// and 1/r is rsq (five operations), so a node takes 18 FP64 operations.  81920 panels (2.05 M
// pairs): 1.63 ms, 2.36 with the nodes formed from the vertices and the library's rsqrt.
__global__ void near_values_kernel(int64_t nnz, const int *row, const int *col, const double *__restrict__ verts,
                                   const int *__restrict__ tris, const double *cx, const double *cy, const double *cz,
                                   const double *nx, const double *ny, const double *nz, const double *area,
                                   const double *Vself, int K, int Kf, double *dV, double *dK) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= nnz) return;
    const int i = row[e], j = col[e];
    if (i == j) {
        dV[e] = Vself[i];
        dK[e] = 0.0;
        return;
    }
    const double x[3] = {cx[i], cy[i], cz[i]};
    const double n[3] = {nx[j], ny[j], nz[j]};
    double w[3], e1[3], e2[3];
    const int *t = tris + 3 * (int64_t)j;
    for (int q = 0; q < 3; ++q) {
        const double v0 = verts[3 * (int64_t)t[0] + q];
        w[q] = x[q] - v0;
        e1[q] = verts[3 * (int64_t)t[1] + q] - v0;
        e2[q] = verts[3 * (int64_t)t[2] + q] - v0;
    }
    const double dn = w[0] * n[0] + w[1] * n[1] + w[2] * n[2];
    auto node = [&](double b1, double b2, double wt, double &sv, double &sk) {
        const double d0 = fma(-b2, e2[0], fma(-b1, e1[0], w[0]));
        const double d1 = fma(-b2, e2[1], fma(-b1, e1[1], w[1]));
        const double d2 = fma(-b2, e2[2], fma(-b1, e1[2], w[2]));
        const double r = rsq(d0 * d0 + d1 * d1 + d2 * d2);
        const double wr = wt * r;
        sv += wr;
        sk = fma(wr, r * r, sk);
    };
    double fv = 0, fk = 0, cv = 0, ck = 0;
    for (int g = 0; g < Kf; ++g) node(c_fine_bary[3 * g + 1], c_fine_bary[3 * g + 2], c_fine_w[g], fv, fk);
    for (int g = 0; g < K; ++g) node(c_far_bary[3 * g + 1], c_far_bary[3 * g + 2], c_far_w[g], cv, ck);
    const double A = area[j] * kInv4Pi;
    dV[e] = (fv - cv) * A;
    dK[e] = (fk - ck) * dn * A;
}

__global__ void natural_order_kernel(int64_t N, int K, const dbl4 *pos, const dbl4 *nrm, const dbl4 *tgt,
                                     dbl4 *spos64, dbl4 *snrm64, float4 *spos32, float4 *snrm32,
                                     dbl4 *tgt64, float4 *tgt32, int *src_panel, int *tgt_panel, int *tgt_pos,
                                     int *src_tblock) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N * K) return;
    dbl4 p = pos[s], n = nrm[s];
    int pid = (int)(s / K);
    spos64[s] = p;
    snrm64[s] = n;
    spos32[s] = make_float4((float)p.x, (float)p.y, (float)p.z, (float)p.w);
    snrm32[s] = make_float4((float)n.x, (float)n.y, (float)n.z, __int_as_float(pid));
    src_panel[s] = pid;
    src_tblock[s] = pid / kTargetBlock;
    if (s % K == 0) {
        dbl4 t = tgt[pid];
        tgt64[pid] = t;
        tgt32[pid] = make_float4((float)t.x, (float)t.y, (float)t.z, __int_as_float(pid));
        tgt_panel[pid] = pid;
        tgt_pos[pid] = pid;
    }
}

// ----------------------------------------------------------------------------
int cuda_status(lspr_ctx *ctx, cudaError_t e, const char *what) {
    ctx->last_error = std::string(what) + ": " + cudaGetErrorString(e);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return LSPR_E_OOM;
    }
    return LSPR_E_CUDA;
}

// flags[0] |= 1 for a surface index outside [0, S)
__global__ void surf_check_kernel(int64_t N, int S, const int *__restrict__ surf, int *flag) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < N && (surf[i] < 0 || surf[i] >= S)) atomicOr(flag, 1);
}

int mesh_build(lspr_ctx *ctx, const double *verts, int64_t nv, const int *tris, int64_t N, const int *surf,
               int nsurf, int on_device, const lspr_quad_opts &q) {
    Mesh &m = ctx->mesh;
    cudaStream_t st = ctx->stream;
    m.ready = false;
    ctx->tree.ready = false;
    double fb[37 * 3], fw[37], gb[37 * 3], gw[37], glx[kMaxNk], glw[kMaxNk];
    if (expand_rule(q.K, fb, fw) != q.K || (q.K != 1 && q.K != 3 && q.K != 4)) return LSPR_E_ARG;
    if (expand_rule(q.K_fine, gb, gw) != q.K_fine || q.K_fine < 19) return LSPR_E_ARG;
    if (q.N_k < 1 || q.N_k > kMaxNk || !(q.threshold > 0)) return LSPR_E_ARG;
    gauss_legendre(q.N_k, glx, glw);
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_far_bary, fb, sizeof(double) * 3 * q.K, 0, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_far_w, fw, sizeof(double) * q.K, 0, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_fine_bary, gb, sizeof(double) * 3 * q.K_fine, 0, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_fine_w, gw, sizeof(double) * q.K_fine, 0, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_gl_x, glx, sizeof(double) * q.N_k, 0, cudaMemcpyHostToDevice, st));
    LSPR_TRY(ctx, cudaMemcpyToSymbolAsync(c_gl_w, glw, sizeof(double) * q.N_k, 0, cudaMemcpyHostToDevice, st));

    m.N = N;
    m.nv = nv;
    m.K = q.K;
    m.Kf = q.K_fine;
    m.Nk = q.N_k;
    m.thr = q.threshold;
    m.Ns = N * q.K;
    LSPR_TRY(ctx, m.verts.ensure(3 * nv));
    LSPR_TRY(ctx, m.tris.ensure(3 * N));
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    LSPR_TRY(ctx, cudaMemcpyAsync(m.verts.p, verts, sizeof(double) * 3 * nv, kind, st));
    LSPR_TRY(ctx, cudaMemcpyAsync(m.tris.p, tris, sizeof(int) * 3 * N, kind, st));
    for (DArr<double> *a : {&m.cx, &m.cy, &m.cz, &m.nx, &m.ny, &m.nz, &m.area, &m.L, &m.Vself})
        LSPR_TRY(ctx, a->ensure(N));
    LSPR_TRY(ctx, m.src_pos64.ensure(m.Ns));
    LSPR_TRY(ctx, m.src_nrm64.ensure(m.Ns));
    LSPR_TRY(ctx, m.tgt64.ensure(N));

    // scratch: [0] bad flag (int), [1] rho_max, [2] L_max, [4..9] bounding box of the centroids
    Tmp<double> flags(ctx->scratch[0]);
    LSPR_TRY(ctx, flags.ensure(10 + 6 * kBoxBlocks));
    LSPR_TRY(ctx, cudaMemsetAsync(flags.p, 0, 4 * sizeof(double), st));
    m.S = nsurf;
    LSPR_TRY(ctx, m.surf.ensure(N));
    if (surf) {
        LSPR_TRY(ctx, cudaMemcpyAsync(m.surf.p, surf, sizeof(int) * N, kind, st));
        ++ctx->n_launches;
        surf_check_kernel<<<grid_for(N, 256), 256, 0, st>>>(N, nsurf, m.surf.p, (int *)flags.p);
    } else {
        LSPR_TRY(ctx, cudaMemsetAsync(m.surf.p, 0, sizeof(int) * N, st));
    }
    cudaEvent_t ev;
    timer_begin(ctx, T_MESH, &ev);
    ++ctx->n_launches;
    panel_kernel<<<grid_for(N, 256), 256, 0, st>>>(m.verts.p, m.tris.p, N, nv, m.cx.p, m.cy.p, m.cz.p, m.nx.p, m.ny.p,
                                                   m.nz.p, m.area.p, m.L.p, (int *)flags.p);
    ++ctx->n_launches;
    sources_kernel<<<grid_for(m.Ns, 256), 256, 0, st>>>(m.verts.p, m.tris.p, N, m.K, m.area.p, m.nx.p, m.ny.p,
                                                        m.nz.p, m.cx.p, m.cy.p, m.cz.p, m.src_pos64.p,
                                                        m.src_nrm64.p, m.tgt64.p, flags.p + 1, flags.p + 2, m.L.p,
                                                        (const int *)flags.p);
    ++ctx->n_launches;
    self_kernel<<<grid_for(N, 128), 128, 0, st>>>(m.verts.p, m.tris.p, N, m.Nk, m.cx.p, m.cy.p, m.cz.p, m.Vself.p,
                                                (const int *)flags.p);
    LSPR_TRY_ST(launch_bbox(ctx, m.tgt64.p, N, nullptr, 0, flags.p + 10, flags.p + 4));
    double hflags[10];
    LSPR_TRY(ctx, cudaMemcpyAsync(hflags, flags.p, sizeof(hflags), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    int bad;
    std::memcpy(&bad, &hflags[0], sizeof(int));
    m.rho_max = hflags[1];
    m.Lmax = hflags[2];
    if (bad & 1) return LSPR_E_ARG;
    if (bad & 2) return LSPR_E_MESH;

    // near-singular list from a cell list (cell edge >= L_max / threshold)
    Tmp<int64_t> cnt(ctx->scratch[1]);
    LSPR_TRY(ctx, cnt.ensure(N));
    LSPR_TRY(ctx, m.near_ptr.ensure(N + 1));
    double hgrid[5];
    {
        const double *lo = hflags + 4, *hi = hflags + 7;
        const double ext = std::max(hi[0] - lo[0], std::max(hi[1] - lo[1], hi[2] - lo[2]));
        const double h = std::max(m.Lmax / m.thr * (1.0 + 1e-9), ext / 1023.0) * (1.0 + 1e-12) + 1e-300;
        hgrid[0] = lo[0];
        hgrid[1] = lo[1];
        hgrid[2] = lo[2];
        hgrid[3] = 1.0 / h;
        hgrid[4] = std::max(std::max(std::fabs(lo[0]), std::fabs(hi[0])),
                            std::max(std::max(std::fabs(lo[1]), std::fabs(hi[1])),
                                     std::max(std::fabs(lo[2]), std::fabs(hi[2]))));
    }
    Tmp<double> grid(ctx->scratch[2]);
    Tmp<unsigned> keys(ctx->scratch[3]), ktmp(ctx->scratch[4]);
    Tmp<int> vals(ctx->scratch[5]), vtmp(ctx->scratch[6]), hist(ctx->scratch[7]), offs(ctx->scratch[8]);
    LSPR_TRY(ctx, grid.ensure(5));
    Tmp<float4> cf(ctx->scratch[9]);
    LSPR_TRY(ctx, cf.ensure(N));
    LSPR_TRY(ctx, keys.ensure(N));
    LSPR_TRY(ctx, ktmp.ensure(N));
    LSPR_TRY(ctx, vals.ensure(N));
    LSPR_TRY(ctx, vtmp.ensure(N));
    LSPR_TRY(ctx, hist.ensure(radix_sort_scratch_ints(N)));
    LSPR_TRY(ctx, offs.ensure(256));
    LSPR_TRY(ctx, cudaMemcpyAsync(grid.p, hgrid, sizeof(hgrid), cudaMemcpyHostToDevice, st));
    ++ctx->n_launches;
    cell_key_kernel<<<grid_for(N, 256), 256, 0, st>>>(N, m.cx.p, m.cy.p, m.cz.p, m.L.p, m.thr, grid.p, keys.p,
                                                      vals.p, cf.p);
    LSPR_TRY_ST(radix_sort(ctx, keys.p, vals.p, ktmp.p, vtmp.p, N, 30, hist.p, offs.p));
    ++ctx->n_launches;
    near_cells_kernel<false><<<grid_for(N * 32, 128), 128, 0, st>>>(N, m.cx.p, m.cy.p, m.cz.p, m.L.p, m.thr, grid.p,
                                                               keys.p, vals.p, cf.p, cnt.p, nullptr, nullptr, nullptr);
    ++ctx->n_launches;
    scan_kernel<<<1, 1024, 0, st>>>(cnt.p, N, m.near_ptr.p);
    LSPR_TRY(ctx, cudaGetLastError());
    LSPR_TRY(ctx, cudaMemcpyAsync(&m.nnz, m.near_ptr.p + N, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    LSPR_TRY(ctx, m.near_col.ensure(m.nnz));
    LSPR_TRY(ctx, m.near_dV.ensure(m.nnz));
    LSPR_TRY(ctx, m.near_dK.ensure(m.nnz));
    Tmp<int> rowidx(ctx->scratch[10]);
    LSPR_TRY(ctx, rowidx.ensure(m.nnz));
    ++ctx->n_launches;
    near_cells_kernel<true><<<grid_for(N * 32, 128), 128, 0, st>>>(N, m.cx.p, m.cy.p, m.cz.p, m.L.p, m.thr, grid.p,
                                                              keys.p, vals.p, cf.p, nullptr, m.near_ptr.p, m.near_col.p,
                                                              rowidx.p);
    ++ctx->n_launches;
    near_values_kernel<<<grid_for(m.nnz, 128), 128, 0, st>>>(m.nnz, rowidx.p, m.near_col.p, m.verts.p, m.tris.p,
                                                             m.cx.p, m.cy.p, m.cz.p, m.nx.p, m.ny.p, m.nz.p, m.area.p,
                                                             m.Vself.p, m.K, m.Kf, m.near_dV.p, m.near_dK.p);
    LSPR_TRY(ctx, m.near_f32.ensure(m.nnz));
    ++ctx->n_launches;
    near_f32_kernel<<<grid_for(m.nnz, 256), 256, 0, st>>>(m.nnz, m.near_dV.p, m.near_dK.p, m.near_f32.p);
    LSPR_TRY(ctx, cudaGetLastError());
    timer_end(ctx, T_MESH, ev);
    LSPR_TRY(ctx, cudaStreamSynchronize(st));
    m.ready = true;
    return workorder_natural(ctx);
}

// Direct-mode work items: every target block against source chunks.  An item is one warp's work, so
// a small mesh is cut finer, up to the point where adding an item's sums (4 FP64 atomics per target
// and right-hand side) costs more than the warps in flight gain: at least 12288 items of 32 to 512
// sources for one right-hand side, 3072 of 64 to 512 for several.  1280 panels in FP64: 305 us
// with 3200 items of 32 sources, 1609 with the 200 of 512; 5120 panels in FP32: 80 us after 86.
static int direct_lists(lspr_ctx *ctx, DirectItems &d, int64_t target, int64_t least) {
    const Mesh &m = ctx->mesh;
    const int64_t ntb = (m.N + kTargetBlock - 1) / kTargetBlock;
    const int64_t chunk = std::max(least, std::min<int64_t>(512, ntb * m.Ns / target / 32 * 32));
    if (&d == &ctx->direct_multi && chunk == ctx->direct.chunk) {   // the same list: not formed twice
        d.n = 0;
        return LSPR_OK;
    }
    d.chunk = chunk;
    d.n = ntb * ((m.Ns + chunk - 1) / chunk);
    LSPR_TRY(ctx, d.items.ensure(d.n));
    return LSPR_OK;
}

int workorder_natural(lspr_ctx *ctx) {
    Mesh &m = ctx->mesh;
    WorkOrder &w = ctx->wo;
    cudaStream_t st = ctx->stream;
    LSPR_TRY(ctx, w.spos64.ensure(m.Ns));
    LSPR_TRY(ctx, w.snrm64.ensure(m.Ns));
    LSPR_TRY(ctx, w.spos32.ensure(m.Ns));
    LSPR_TRY(ctx, w.snrm32.ensure(m.Ns));
    LSPR_TRY(ctx, w.tgt64.ensure(m.N));
    LSPR_TRY(ctx, w.tgt32.ensure(m.N));
    LSPR_TRY(ctx, w.src_panel.ensure(m.Ns));
    LSPR_TRY(ctx, w.tgt_panel.ensure(m.N));
    LSPR_TRY(ctx, w.tgt_pos.ensure(m.N));
    LSPR_TRY(ctx, w.src_tblock.ensure(m.Ns));
    ++ctx->n_launches;
    natural_order_kernel<<<grid_for(m.Ns, 256), 256, 0, st>>>(m.N, m.K, m.src_pos64.p, m.src_nrm64.p, m.tgt64.p,
                                                              w.spos64.p, w.snrm64.p, w.spos32.p, w.snrm32.p,
                                                              w.tgt64.p, w.tgt32.p, w.src_panel.p, w.tgt_panel.p,
                                                              w.tgt_pos.p, w.src_tblock.p);
    LSPR_TRY(ctx, cudaGetLastError());
    LSPR_TRY_ST(direct_lists(ctx, ctx->direct, 12288, 32));
    LSPR_TRY_ST(direct_lists(ctx, ctx->direct_multi, 3072, 64));
    LSPR_TRY_ST(launch_direct_flags(ctx));
    LSPR_TRY_ST(launch_ff_geometry(ctx));
    LSPR_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    return LSPR_OK;
}

}  // namespace lspr
