// indexing.cu -- step (a6): the look-up table and Eq. 3 matching, and step
// (a7): Gauss-Newton orientation refinement on a bilinear elevation-azimuth
// reference image, with forward and backward kernels for automatic
// differentiation.
//
// Supplement "Indexing algorithm": the reference signature of a candidate is
// normalised, its n_hat strongest nodes are kept, every test orientation g
// rotates them, and the look-up table holds the measured-image node nearest
// to each rotated reference node; Eq. 3 scores g by the sum of squared
// differences of the image values there.  Rotations map crystal to lab.
#include <math.h>

#include "common.cuh"

namespace aptidx {

namespace {

// ---- rotations (FP64, fixed operation order, no contraction) ----------------

struct M3 {
    double a[9];
};

__device__ __forceinline__ M3 quat_to_matrix(double w, double x, double y, double z) {
    const double xx = __dmul_rn(x, x), yy = __dmul_rn(y, y), zz = __dmul_rn(z, z);
    const double xy = __dmul_rn(x, y), xz = __dmul_rn(x, z), yz = __dmul_rn(y, z);
    const double wx = __dmul_rn(w, x), wy = __dmul_rn(w, y), wz = __dmul_rn(w, z);
    M3 m;
    m.a[0] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(yy, zz)));
    m.a[1] = __dmul_rn(2.0, __dsub_rn(xy, wz));
    m.a[2] = __dmul_rn(2.0, __dadd_rn(xz, wy));
    m.a[3] = __dmul_rn(2.0, __dadd_rn(xy, wz));
    m.a[4] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(xx, zz)));
    m.a[5] = __dmul_rn(2.0, __dsub_rn(yz, wx));
    m.a[6] = __dmul_rn(2.0, __dsub_rn(xz, wy));
    m.a[7] = __dmul_rn(2.0, __dadd_rn(yz, wx));
    m.a[8] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(xx, yy)));
    return m;
}

__device__ __forceinline__ void quat_mul(const double* a, const double* b, double* o) {
    const double r0 = a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
    const double r1 = a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2];
    const double r2 = a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1];
    const double r3 = a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0];
    o[0] = r0;
    o[1] = r1;
    o[2] = r2;
    o[3] = r3;
}

__device__ __forceinline__ void exp_quat(const double* d, double* q) {
    const double th = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    if (th < 1e-300) {
        q[0] = 1.0;
        q[1] = q[2] = q[3] = 0.0;
        return;
    }
    const double s = sin(0.5 * th) / th;
    q[0] = cos(0.5 * th);
    q[1] = s * d[0];
    q[2] = s * d[1];
    q[3] = s * d[2];
}

// ---- strongest reference nodes (bitonic sort of packed keys, one block) -----

__device__ __forceinline__ uint32_t ordered_f32(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// key = (descending value, ascending index); padding sorts last
__global__ void __launch_bounds__(1024) k_top_nodes(const float* __restrict__ sig, int32_t nv, int32_t npow2,
                                                    uint64_t* keys, int32_t n_hat, int32_t* top, float* top_val) {
    for (int i = threadIdx.x; i < npow2; i += blockDim.x)
        keys[i] = i < nv ? ((uint64_t)(~ordered_f32(sig[i])) << 32) | (uint32_t)i : ~0ull;
    __syncthreads();
    for (int k = 2; k <= npow2; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < npow2; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i) {
                    const uint64_t a = keys[i], b = keys[l];
                    const bool up = (i & k) == 0;
                    if ((a > b) == up) {
                        keys[i] = b;
                        keys[l] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < n_hat; i += blockDim.x) {
        const int32_t idx = (int32_t)(keys[i] & 0xFFFFFFFFu);
        top[i] = idx;
        top_val[i] = sig[idx];
    }
}

// The same for n_hat <= kSelMax: the n_hat-th smallest 32-bit key (descending
// value) by a radix select over four 8-bit digits, then the keys below it and
// the lowest-index ones equal to it, sorted in shared memory.  The full sort
// above walks 136 passes of 65536 keys in global memory at 40962 directions
// (2.16 ms in one CTA); four counting passes and a sort of 1024 keys take
// 0.04 ms.  Where the sort is no longer for all keys, and up to kSortAll directions, it
// takes them all: the four passes, with a walk over 256 counts each, cost 12 us more
// (aptidx_set_reference of 162 directions 50 us, now 37; of 1025 and all of them 75, 54).
constexpr int kSelMax = 4096;
constexpr int kSortAll = 1024;

__global__ void __launch_bounds__(1024) k_top_select(const float* __restrict__ sig, int32_t nv, int32_t n_hat,
                                                     int32_t* top, float* top_val) {
    __shared__ uint64_t sel[kSelMax];
    __shared__ uint32_t hist[256], wcnt[32];
    __shared__ uint32_t s_prefix, s_rem, s_count;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_prefix = 0;
        s_rem = (uint32_t)n_hat;
        s_count = 0;
    }
    int kp = 1;
    while (kp < (nv <= kSortAll ? nv : n_hat)) kp <<= 1;
    for (int i = tid; i < kp; i += 1024) sel[i] = ~0ull;
    __syncthreads();
    if (nv <= kp) {
        for (int i = tid; i < nv; i += 1024) sel[i] = ((uint64_t)(~ordered_f32(sig[i])) << 32) | (uint32_t)i;
    } else {
        for (int pass = 3; pass >= 0; --pass) {
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            const uint32_t prefix = s_prefix, hmask = pass == 3 ? 0u : 0xFFFFFFFFu << (8 * (pass + 1));
            for (int i = tid; i < nv; i += 1024) {
                const uint32_t k = ~ordered_f32(sig[i]);
                if ((k & hmask) == (prefix & hmask)) atomicAdd(&hist[(k >> (8 * pass)) & 255u], 1u);
            }
            __syncthreads();
            if (tid == 0) {
                uint32_t rem = s_rem, d = 0;
                while (hist[d] < rem) rem -= hist[d++];
                s_rem = rem;
                s_prefix = prefix | (d << (8 * pass));
            }
            __syncthreads();
        }
        const uint32_t kth = s_prefix, need_eq = s_rem, n_less = (uint32_t)n_hat - need_eq;
        for (int i = tid; i < nv; i += 1024) {
            const uint32_t k = ~ordered_f32(sig[i]);
            if (k < kth) sel[atomicAdd(&s_count, 1u)] = ((uint64_t)k << 32) | (uint32_t)i;
        }
        uint32_t taken = 0;
        for (int i0 = 0; i0 < nv && taken < need_eq; i0 += 1024) {
            const int i = i0 + tid;
            const bool eq = i < nv && ~ordered_f32(sig[i]) == kth;
            const uint32_t bal = __ballot_sync(0xffffffffu, eq);
            __syncthreads();
            if (lane == 0) wcnt[warp] = __popc(bal);
            __syncthreads();
            uint32_t before = 0, total = 0;
            for (int w = 0; w < 32; ++w) {
                if (w < warp) before += wcnt[w];
                total += wcnt[w];
            }
            const uint32_t rank = taken + before + __popc(bal & ((1u << lane) - 1u));
            if (eq && rank < need_eq) sel[n_less + rank] = ((uint64_t)kth << 32) | (uint32_t)i;
            taken += total;
        }
    }
    __syncthreads();
    for (int k = 2; k <= kp; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < kp; i += 1024) {
                const int l = i ^ j;
                if (l > i) {
                    const uint64_t x = sel[i], y = sel[l];
                    if ((x > y) == ((i & k) == 0)) {
                        sel[i] = y;
                        sel[l] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < n_hat; i += 1024) {
        const int32_t idx = (int32_t)(sel[i] & 0xFFFFFFFFu);
        top[i] = idx;
        top_val[i] = sig[idx];
    }
}

// ---- look-up table ---------------------------------------------------------------

constexpr int kLutThreads = 256;
constexpr int kLutPer = 4;                       // queries per thread
constexpr int kLutTile = 2048;                   // nodes per shared-memory tile

// The rotated node r = (float)(R(q) n), FP64 products summed left to right.
__device__ __forceinline__ float3 rotate_node(const M3& R, float4 n) {
    const double nx = n.x, ny = n.y, nz = n.z;
    float3 r;
    r.x = __double2float_rn(__dadd_rn(__dadd_rn(__dmul_rn(R.a[0], nx), __dmul_rn(R.a[1], ny)), __dmul_rn(R.a[2], nz)));
    r.y = __double2float_rn(__dadd_rn(__dadd_rn(__dmul_rn(R.a[3], nx), __dmul_rn(R.a[4], ny)), __dmul_rn(R.a[5], nz)));
    r.z = __double2float_rn(__dadd_rn(__dadd_rn(__dmul_rn(R.a[6], nx), __dmul_rn(R.a[7], ny)), __dmul_rn(R.a[8], nz)));
    return r;
}

__device__ __forceinline__ float node_dot(float4 u, float3 r) {
    return __fmaf_rn(u.z, r.z, __fmaf_rn(u.y, r.y, __fmul_rn(u.x, r.x)));
}

// lut_t[k * ng_pad + g] = argmax_p u_p . r with r = R(q_g) n_top[k], the dot
// product by the FP32 contract fma(u_z, r_z, fma(u_y, r_y, u_x r_x)); ties
// resolve to the lowest index.  IdxT is uint16_t when every node index fits
// (nv <= 65536), else int32_t.
//
// The nodes lie in a cubic grid of cells of edge h (about one and a half node
// spacings of an even covering).  A query scans the 3 x 3 x 3 cells around r, nine
// runs of consecutive nodes.  A node outside them is at least h away, so its exact dot
// product is at most (max |u|^2 + |r|^2 - h^2) / 2: when the best found exceeds
// that by more than the FP32 errors it is the answer of a scan over all nodes.
// Queries it does not settle (r in a gap of the direction set), and those with more
// than kLutRun nodes in their cells (clustered directions: a thread that walked
// thousands of nodes by itself took up to 54 ms for 10^6 queries on 40000 directions
// within one degree, the scan 9.1), are listed and left to k_lut_scan.
// Scanning all 40962 nodes for every query took 29.1 ms for 3419 x 1000 queries
// (1.4e11 dot products); this reads about 20 nodes per query, bound by the L2 latency
// of the run bounds and nodes: 0.4 ms.
constexpr int kLutRun = 512;
constexpr int kLutK = 8;   // nodes per thread (one rotation matrix, kLutK of its columns of the table)

struct NodeGrid {
    const int32_t* start;   // [dim^3 + 1]
    const float4* nodes;    // in cell order, in any order inside a cell; w = index bits
    int dim;
    float org, inv_h, far2;   // cell = (x - org) * inv_h; far2 = max |u|^2 - (0.999 h)^2
};

__device__ __forceinline__ int node_cell(float x, const NodeGrid& g) {
    return min(max((int)((x - g.org) * g.inv_h), 0), g.dim - 1);
}

__device__ __forceinline__ int node_cell3(float4 u, const NodeGrid& g) {
    return node_cell(u.x, g) + g.dim * (node_cell(u.y, g) + g.dim * node_cell(u.z, g));
}

__global__ void __launch_bounds__(256) k_node_count(const float4* __restrict__ dirs, int32_t nv, NodeGrid g,
                                                    unsigned long long* counts) {
    const int v = blockIdx.x * 256 + threadIdx.x;
    if (v < nv) atomicAdd(&counts[node_cell3(dirs[v], g)], 1ull);
}

// every node into its cell (in any order: queries resolve ties by index), counting the
// cells down, and the cells' first nodes in 32 bits
__global__ void __launch_bounds__(256) k_node_fill(const float4* __restrict__ dirs, int32_t nv, NodeGrid g, int n_cells,
                                                   const int64_t* __restrict__ off, unsigned long long* counts,
                                                   int32_t* start, float4* nodes) {
    for (int i = blockIdx.x * 256 + threadIdx.x; i <= n_cells; i += gridDim.x * 256) start[i] = (int32_t)off[i];
    for (int v = blockIdx.x * 256 + threadIdx.x; v < nv; v += gridDim.x * 256) {
        const float4 u = dirs[v];
        const int c = node_cell3(u, g);
        const int64_t k = off[c] + (int64_t)atomicAdd(&counts[c], ~0ull) - 1;
        nodes[k] = make_float4(u.x, u.y, u.z, __int_as_float(v));
    }
}

template <typename IdxT>
__global__ void __launch_bounds__(kLutThreads) k_build_lut(NodeGrid grid, const float4* __restrict__ dirs,
                                                           const int32_t* __restrict__ top, int32_t n_hat,
                                                           const double* __restrict__ quats, int64_t ng,
                                                           int64_t ng_pad, IdxT* lut_t, int32_t k0, int32_t k1,
                                                           uint32_t* open, uint32_t* n_open) {
    const int64_t g = (int64_t)blockIdx.x * kLutThreads + threadIdx.x;
    const int kb = k0 + (int)blockIdx.y * kLutK;
    if (g >= ng) return;
    const M3 R = quat_to_matrix(quats[4 * g], quats[4 * g + 1], quats[4 * g + 2], quats[4 * g + 3]);
    for (int k = kb; k < min(kb + kLutK, k1); ++k) {
        const float3 r = rotate_node(R, dirs[top[k]]);
        const int ix = node_cell(r.x, grid), iy = node_cell(r.y, grid), iz = node_cell(r.z, grid);
        const int xa = max(ix - 1, 0), xb = min(ix + 2, grid.dim);
        float best = -INFINITY;
        int32_t bi = 0x7FFFFFFF;
        int32_t beg[9], end[9], run = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const int y = iy + j % 3 - 1, z = iz + j / 3 - 1;
            const bool in = y >= 0 && y < grid.dim && z >= 0 && z < grid.dim;
            const int c = in ? grid.dim * (y + grid.dim * z) : 0;
            beg[j] = in ? __ldg(grid.start + c + xa) : 0;
            end[j] = in ? __ldg(grid.start + c + xb) : 0;
            run += end[j] - beg[j];
        }
#pragma unroll
        for (int j = 0; j < 9; ++j)
            for (int i = beg[j]; i < end[j] && run <= kLutRun; ++i) {
                const float4 u = __ldg(grid.nodes + i);
                const float d = node_dot(u, r);
                const int32_t idx = __float_as_int(u.w);
                if (d > best || (d == best && idx < bi)) {
                    best = d;
                    bi = idx;
                }
            }
        const float r2 = r.x * r.x + r.y * r.y + r.z * r.z;
        if (run <= kLutRun && best > 0.5f * (grid.far2 + r2) + 2e-6f) {
            lut_t[(int64_t)k * ng_pad + g] = (IdxT)bi;
        } else {
            open[atomicAdd(n_open, 1u)] = (uint32_t)((int64_t)(k - k0) * ng + g);
        }
    }
}

// The listed queries (open == nullptr: all n_all of them) against every node, staged
// through shared memory, four queries per thread.
template <typename IdxT>
__global__ void __launch_bounds__(kLutThreads) k_lut_scan(const float4* __restrict__ dirs, int32_t nv,
                                                          const int32_t* __restrict__ top,
                                                          const double* __restrict__ quats, int64_t ng,
                                                          int64_t ng_pad, IdxT* lut_t, int32_t k0, uint32_t n_all,
                                                          const uint32_t* __restrict__ open,
                                                          const uint32_t* __restrict__ n_open) {
    __shared__ float4 tile[kLutTile];
    const uint32_t n = open ? *n_open : n_all;
    for (uint32_t q0 = blockIdx.x * (uint32_t)(kLutThreads * kLutPer); q0 < n;
         q0 += gridDim.x * (uint32_t)(kLutThreads * kLutPer)) {
        float3 r[kLutPer];
        float best[kLutPer];
        int32_t bi[kLutPer];
#pragma unroll
        for (int j = 0; j < kLutPer; ++j) {
            const uint32_t i = q0 + (uint32_t)j * kLutThreads + threadIdx.x;
            best[j] = -INFINITY;
            bi[j] = 0;
            r[j] = make_float3(0.f, 0.f, 0.f);
            if (i < n) {
                const uint32_t q = open ? open[i] : i;
                const int64_t g = q % ng;
                const M3 R = quat_to_matrix(quats[4 * g], quats[4 * g + 1], quats[4 * g + 2], quats[4 * g + 3]);
                r[j] = rotate_node(R, dirs[top[k0 + (int)(q / ng)]]);
            }
        }
        for (int p0 = 0; p0 < nv; p0 += kLutTile) {
            const int cnt = min(kLutTile, nv - p0);
            __syncthreads();
            for (int i = threadIdx.x; i < cnt; i += kLutThreads) tile[i] = dirs[p0 + i];
            __syncthreads();
            for (int i = 0; i < cnt; ++i) {
                const float4 u = tile[i];
#pragma unroll
                for (int j = 0; j < kLutPer; ++j) {
                    const float d = node_dot(u, r[j]);
                    if (d > best[j]) {
                        best[j] = d;
                        bi[j] = p0 + i;
                    }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kLutPer; ++j) {
            const uint32_t i = q0 + (uint32_t)j * kLutThreads + threadIdx.x;
            if (i < n) {
                const uint32_t q = open ? open[i] : i;
                lut_t[(k0 + (int64_t)(q / ng)) * ng_pad + q % ng] = (IdxT)bi[j];
            }
        }
    }
}

// ---- Eq. 3 -----------------------------------------------------------------------

// One CTA per ROI (persistent): the ROI's signature row in shared memory,
// Delta(g) = sum_k (S[lut[k, g]] - ref[k])^2 accumulated in FP32 in k order,
// argmin with ties to the lowest g.  The table streams from L2 once per ROI:
// each thread reads 16 bytes of a table row per k (G = 16 / sizeof(IdxT)
// consecutive orientations) and keeps kMatchDepth rows in flight.
constexpr int kMatchDepth = 8;   // table rows in flight per thread

template <typename IdxT>
__device__ __forceinline__ uint4 lut_load(const IdxT* p) {
    uint4 v;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

template <typename IdxT>
__device__ __forceinline__ void lut_accumulate(const uint4 w, const float* row, float rk, float* acc) {
    if (sizeof(IdxT) == 2) {
        const float d0 = row[w.x & 0xFFFFu] - rk, d1 = row[w.x >> 16] - rk;
        const float d2 = row[w.y & 0xFFFFu] - rk, d3 = row[w.y >> 16] - rk;
        const float d4 = row[w.z & 0xFFFFu] - rk, d5 = row[w.z >> 16] - rk;
        const float d6 = row[w.w & 0xFFFFu] - rk, d7 = row[w.w >> 16] - rk;
        acc[0] = fmaf(d0, d0, acc[0]);
        acc[1] = fmaf(d1, d1, acc[1]);
        acc[2] = fmaf(d2, d2, acc[2]);
        acc[3] = fmaf(d3, d3, acc[3]);
        acc[4] = fmaf(d4, d4, acc[4]);
        acc[5] = fmaf(d5, d5, acc[5]);
        acc[6] = fmaf(d6, d6, acc[6]);
        acc[7] = fmaf(d7, d7, acc[7]);
    } else {
        const float d0 = row[w.x] - rk, d1 = row[w.y] - rk, d2 = row[w.z] - rk, d3 = row[w.w] - rk;
        acc[0] = fmaf(d0, d0, acc[0]);
        acc[1] = fmaf(d1, d1, acc[1]);
        acc[2] = fmaf(d2, d2, acc[2]);
        acc[3] = fmaf(d3, d3, acc[3]);
    }
}

// The signature row into shared memory (all threads, closing barrier); whether all
// its values are equal.
__device__ __forceinline__ bool stage_row(float* row, const float* __restrict__ src, int32_t nv) {
    const float first = src[0];
    bool flat = true;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
        const float v = src[i];
        row[i] = v;
        flat &= v == first;
    }
    return __syncthreads_and(flat) != 0;
}

// Delta of every orientation for a row of the value v, in k order
__device__ __forceinline__ float flat_score(float v, const float* ref, int32_t n_hat) {
    float acc = 0.f;
    for (int k = 0; k < n_hat; ++k) {
        const float d = v - ref[k];
        acc = fmaf(d, d, acc);
    }
    return acc;
}

// With scores_out, weight x Delta(g) of ROI r also goes to scores_out[r * ng
// + g] (accumulate: added to the value there, for sums over signature
// channels).  kListed: the ROIs list[1 .. list[0]] instead of all nroi; a row of
// one value (a ROI without atoms, or with one), whose orientations all tie, takes
// one sum.
template <typename IdxT, bool kListed = false>
__global__ void __launch_bounds__(1024, 1) k_match(const float* __restrict__ S, int64_t nroi, int32_t nv,
                                                const IdxT* __restrict__ lut_t, int64_t ng, int64_t ng_pad,
                                                const float* __restrict__ top_val, int32_t n_hat, int32_t* best,
                                                float* score, float* scores_out, bool accumulate, float weight,
                                                const uint32_t* list) {
    constexpr int G = 16 / (int)sizeof(IdxT);
    extern __shared__ float sm[];
    float* row = sm;                     // nv
    float* ref = sm + nv;                // n_hat
    __shared__ float red_v[32];
    __shared__ int32_t red_g[32];
    const int nwarps = blockDim.x >> 5;
    if (kListed) asm volatile("griddepcontrol.wait;" ::: "memory");   // the list is written
    const int64_t n = kListed ? (int64_t)list[0] : nroi;
    if (kListed && blockIdx.x >= n) return;
    for (int i = threadIdx.x; i < n_hat; i += blockDim.x) ref[i] = top_val[i];
    for (int64_t item = blockIdx.x; item < n; item += gridDim.x) {
        const int64_t r = kListed ? (int64_t)list[1 + item] : item;
        __syncthreads();
        const float* src = S + r * (int64_t)nv;
        if (kListed) {
            if (stage_row(row, src, nv)) {
                if (threadIdx.x == 0) {
                    const float v = flat_score(row[0], ref, n_hat);
                    if (best) best[r] = v < INFINITY ? 0 : 0x7FFFFFFF;
                    if (score) score[r] = v < INFINITY ? v : INFINITY;
                }
                continue;
            }
        } else {
            for (int i = threadIdx.x; i < nv; i += blockDim.x) row[i] = src[i];
            __syncthreads();
        }
        float bv = INFINITY;
        int32_t bg = 0x7FFFFFFF;
        for (int64_t g0 = (int64_t)threadIdx.x * G; g0 < ng; g0 += (int64_t)blockDim.x * G) {
            float acc[G];
#pragma unroll
            for (int e = 0; e < G; ++e) acc[e] = 0.f;
            const IdxT* lp = lut_t + g0;
            int k = 0;
            for (; k + kMatchDepth <= n_hat; k += kMatchDepth) {
                uint4 w[kMatchDepth];
#pragma unroll
                for (int j = 0; j < kMatchDepth; ++j) w[j] = lut_load(lp + (int64_t)(k + j) * ng_pad);
#pragma unroll
                for (int j = 0; j < kMatchDepth; ++j) lut_accumulate<IdxT>(w[j], row, ref[k + j], acc);
            }
            for (; k < n_hat; ++k) lut_accumulate<IdxT>(lut_load(lp + (int64_t)k * ng_pad), row, ref[k], acc);
#pragma unroll
            for (int e = 0; e < G; ++e)
                if (g0 + e < ng && acc[e] < bv) {
                    bv = acc[e];
                    bg = (int32_t)(g0 + e);
                }
            if (scores_out) {
#pragma unroll
                for (int e = 0; e < G; ++e)
                    if (g0 + e < ng) {
                        float* o = scores_out + r * ng + g0 + e;
                        *o = accumulate ? fmaf(weight, acc[e], *o) : weight * acc[e];
                    }
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int32_t og = __shfl_xor_sync(0xffffffffu, bg, o);
            if (ov < bv || (ov == bv && og < bg)) {
                bv = ov;
                bg = og;
            }
        }
        if ((threadIdx.x & 31) == 0) {
            red_v[threadIdx.x >> 5] = bv;
            red_g[threadIdx.x >> 5] = bg;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < nwarps; ++w)
                if (red_v[w] < bv || (red_v[w] == bv && red_g[w] < bg)) {
                    bv = red_v[w];
                    bg = red_g[w];
                }
            if (best) best[r] = bg;
            if (score) score[r] = bv;
        }
    }
}

// ---- Eq. 3 for many ROIs -----------------------------------------------------------
//
// k_match gathers 32 random words of one signature row per instruction: 3.5
// shared-memory wavefronts on average, which bounds it (7.2 ms for 4096 ROIs,
// 3419 orientations, 1000 nodes: 6.2 look-ups per SM cycle).  Here a lane is a
// pair of ROIs: a CTA holds the values of 64 ROIs at a tile of nodes,
// [node][ROI] in shared memory, and walks the table entries whose node lies in
// its tile, so that a look-up of 64 ROIs is two wavefronts and the entry, which
// every lane needs (a broadcast costs its bytes times 32 lanes), is one: 4
// bytes, the reference value rounded to 22 bits and the node's row in the other
// ten.  Entries are stored per (tile, orientation) in lists padded to four with
// entries that read a row of zeros.  The tiles' partial sums of an orientation
// add up in global memory, in any order.
//
// The sums serve as estimates only.  With every reference off by at most
// delta = 2^-14 max |ref|, the root of an estimate is within eta = sqrt(n_hat)
// delta of the root of the exact sum (triangle inequality), and any FP32 order
// of summation is within eps = (n_hat + 64) 2^-24 of it: every orientation
// whose estimate is at most (sqrt(m) + 2 eta)^2 (1 + 5 eps), m the smallest (or
// the topk-th smallest) estimate, is summed again in k order, and these decide.
// Results are those of k_match bit for bit.
// 4096 ROIs, 3419 orientations, 1000 nodes: 7.2 ms before, 2.9 now (k_tm_sum 2.75,
// k_tm_best 0.14); top 1000 of 50000 orientations for 192 ROIs: 6.8 ms before,
// 3.0 now (sums 1.9, exact sums 0.65, selections 0.4).
constexpr int kTmRois = 64;
constexpr int kTmPitch = 66;          // words per node row (8-byte aligned, written by columns)
constexpr int kTmTileMax = 879;       // nodes per tile: (879 + 1) x 264 bytes of shared memory, < 1024 rows
constexpr int kTmThreads = 1024;
constexpr uint32_t kTmRowBits = 0x3FFu;

__device__ __forceinline__ uint32_t tm_entry(float ref, int row) {
    const uint32_t b = __float_as_uint(ref);   // round to nearest at 13 mantissa bits (finite)
    return ((b + 0x200u) & ~kTmRowBits) | (uint32_t)row;
}

__global__ void __launch_bounds__(256) k_tm_count(const uint16_t* __restrict__ lut_t, int64_t ng, int64_t ng_pad, int T,
                                                  int32_t* counts) {
    const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (g < ng) atomicAdd(&counts[(int64_t)((int)lut_t[(int64_t)blockIdx.y * ng_pad + g] / T) * ng + g], 1);
}

__global__ void __launch_bounds__(256) k_tm_pad(const int32_t* __restrict__ counts, int64_t n, int64_t* padded) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < n) padded[i] = (counts[i] + 3) & ~3;
}

// 32-bit offsets, the padding entries, and the counts zeroed (they become the
// lists' cursors)
__global__ void __launch_bounds__(256) k_tm_off(const int64_t* __restrict__ off64, int32_t* counts, int64_t n, int T,
                                                uint32_t* off, uint32_t* ent) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i <= n) off[i] = (uint32_t)off64[i];
    if (i >= n) return;
    const int32_t c = counts[i];
    for (int k = c; k < ((c + 3) & ~3); ++k) ent[off64[i] + k] = (uint32_t)T;
    counts[i] = 0;
}

__global__ void __launch_bounds__(256) k_tm_fill(const uint16_t* __restrict__ lut_t, int64_t ng, int64_t ng_pad,
                                                 const float* __restrict__ top_val, int T,
                                                 const uint32_t* __restrict__ off, int32_t* cursor, uint32_t* ent) {
    const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (g >= ng) return;
    const int node = (int)lut_t[(int64_t)blockIdx.y * ng_pad + g];
    const int p = node / T;
    const int64_t l = (int64_t)p * ng + g;
    ent[(size_t)off[l] + (uint32_t)atomicAdd(&cursor[l], 1)] = tm_entry(top_val[blockIdx.y], node - p * T);
}

// k-major table to rows per orientation, lut_g[g * pitch + k] (32 x 32 tiles)
__global__ void __launch_bounds__(256) k_tm_rowmajor(const uint16_t* __restrict__ lut_t, int64_t ng, int64_t ng_pad,
                                                     int32_t n_hat, int pitch, uint16_t* lut_g) {
    __shared__ uint16_t t[32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t g0 = (int64_t)blockIdx.x * 32;
    const int k0 = (int)blockIdx.y * 32;
    for (int i = w; i < 32; i += 8)
        t[i][lane] = k0 + i < n_hat && g0 + lane < ng ? lut_t[(int64_t)(k0 + i) * ng_pad + g0 + lane] : (uint16_t)0;
    __syncthreads();
    for (int i = w; i < 32; i += 8)
        if (g0 + i < ng && k0 + lane < pitch) lut_g[(g0 + i) * pitch + k0 + lane] = t[lane][i];
}

// CTA (tile, part of the orientations; group of 64 ROIs); D[group][g][2][32],
// ROI 2 l + i of the group at [i][l]
__global__ void __launch_bounds__(kTmThreads, 1) k_tm_sum(const float* __restrict__ S, int64_t nroi, int32_t nv,
                                                          const uint32_t* __restrict__ ent,
                                                          const uint32_t* __restrict__ off, int64_t ng, int T,
                                                          int gsplit, float* D) {
    extern __shared__ float st[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = (int)blockIdx.x / gsplit, gs = (int)blockIdx.x % gsplit;
    const int n0 = p * T, cnt = min(T, nv - n0);
    for (int i = warp; i < kTmRois; i += kTmThreads / 32) {
        const int64_t roi = (int64_t)blockIdx.y * kTmRois + i;
        for (int n = lane; n < cnt; n += 32) st[n * kTmPitch + i] = roi < nroi ? S[roi * (int64_t)nv + n0 + n] : 0.f;
    }
    if (threadIdx.x < kTmPitch) st[T * kTmPitch + threadIdx.x] = 0.f;
    __syncthreads();
    const uint32_t sb = smem_u32(st) + 8u * (uint32_t)lane;
    const int64_t per = (ng + gsplit - 1) / gsplit;
    const int64_t g1 = tmin<int64_t>(ng, (gs + 1) * per);
    const uint32_t* o = off + (int64_t)p * ng;
    auto term = [&](uint32_t e, float& a, float& b) {
        float x, y;
        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(sb + (e & kTmRowBits) * (kTmPitch * 4u)));
        const float ref = __uint_as_float(e & ~kTmRowBits);
        x -= ref;
        y -= ref;
        a = fmaf(x, x, a);
        b = fmaf(y, y, b);
    };
    int64_t g = gs * per + warp;
    uint32_t b = g < g1 ? o[g] : 0, e = g < g1 ? o[g + 1] : 0;
    for (; g < g1; g += kTmThreads / 32) {
        const uint4* q = reinterpret_cast<const uint4*>(ent + b);
        const int n = (int)((e - b) >> 2);
        const int64_t gn = g + kTmThreads / 32;
        if (gn < g1) {
            b = o[gn];
            e = o[gn + 1];
        }
        if (n > 0) {
            float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
            uint4 x = __ldg(q);
            for (int i = 1; i < n; ++i) {
                const uint4 nx = __ldg(q + i);
                term(x.x, a0, b0);
                term(x.y, a1, b1);
                term(x.z, a0, b0);
                term(x.w, a1, b1);
                x = nx;
            }
            term(x.x, a0, b0);
            term(x.y, a1, b1);
            term(x.z, a0, b0);
            term(x.w, a1, b1);
            float* d = D + ((int64_t)blockIdx.y * ng + g) * kTmRois + lane;
            atomicAdd(d, a0 + a1);
            atomicAdd(d + 32, b0 + b1);
        }
    }
}

// largest estimate whose exact sum can be the smallest: see above (and the
// smallest normal number for sums of terms that underflow)
struct TmMargin {
    float eta2, rel;   // 2 eta, 1 + 5 eps
};
__device__ __forceinline__ float tm_threshold(float estimate, TmMargin m) {
    const float r = sqrtf(estimate) + m.eta2;
    return r * r * m.rel + 1.1754944e-38f;
}

// The best orientation of 32 ROIs (half a group per CTA, lane = ROI): the smallest
// estimate, then the sums in k order of every orientation near it, a warp per
// (ROI, orientation): the lanes read 32 terms, which are added in turn.  A ROI with
// more than kTmNear orientations near its best (a row of one or few values) is left
// to k_match, which sums all of a ROI's orientations in the time this form takes for
// some 60: heavy[1 ..] lists such ROIs, heavy[0] (zero before) counts them.  Summed
// here, 200 rows of zeros among 4096 (3419 orientations, 1000 nodes) took 90 ms; now
// 3.0, as any other rows (2.9).
constexpr int kTmNear = 64;

__global__ void __launch_bounds__(kTmThreads, 1) k_tm_best(const float* __restrict__ S, int64_t nroi, int32_t nv,
                                                        const uint16_t* __restrict__ lut_g, int64_t ng, int pitch,
                                                        const float* __restrict__ top_val, int32_t n_hat,
                                                        TmMargin margin, const float* __restrict__ D, int32_t* best,
                                                        float* score, uint32_t* heavy) {
    __shared__ float red[32][33];
    __shared__ float thr[32];
    __shared__ unsigned long long key[32];
    __shared__ uint32_t near_g[32][kTmNear];
    __shared__ uint32_t n_near[32];    // orientations near the best, then their inclusive sums
    __shared__ uint32_t s_heavy;       // lanes left to k_match
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t roi0 = (int64_t)(blockIdx.x >> 1) * kTmRois + (blockIdx.x & 1);   // ROI of lane l: roi0 + 2 l
    const float* d = D + (int64_t)(blockIdx.x >> 1) * ng * kTmRois + (blockIdx.x & 1) * 32 + lane;
    float m = INFINITY;
#pragma unroll 4
    for (int64_t g = warp; g < ng; g += 32) m = fminf(m, d[g * kTmRois]);
    red[warp][lane] = m;
    if (warp == 0) {
        key[lane] = 0x7F8000007FFFFFFFull;   // (+inf, no orientation)
        n_near[lane] = 0;
    }
    __syncthreads();
    if (warp == 0) {
        for (int w = 1; w < 32; ++w) m = fminf(m, red[w][lane]);
        thr[lane] = tm_threshold(m, margin);
    }
    __syncthreads();
    const float t = thr[lane];
    const bool valid = roi0 + 2 * lane < nroi;
    volatile uint32_t* seen = n_near;
#pragma unroll 4
    for (int64_t g = warp; g < ng; g += 32)
        if (valid && d[g * kTmRois] <= t && seen[lane] <= kTmNear) {
            const uint32_t i = atomicAdd(&n_near[lane], 1u);
            if (i < kTmNear) near_g[lane][i] = (uint32_t)g;
        }
    __syncthreads();
    if (warp == 0) {
        const bool many = n_near[lane] > kTmNear;
        const uint32_t bal = __ballot_sync(0xffffffffu, many);
        if (many) heavy[1 + atomicAdd(heavy, 1u)] = (uint32_t)(roi0 + 2 * lane);
        if (lane == 0) s_heavy = bal;
        uint32_t x = many ? 0 : n_near[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        n_near[lane] = x;
    }
    __syncthreads();
    const uint32_t upto = n_near[lane], total = n_near[31];
    for (uint32_t i = warp; i < total; i += 32) {
        // pair i: ROI r, the first whose inclusive sum exceeds i
        const int r = __popc(__ballot_sync(0xffffffffu, upto <= i));
        const int64_t cg = near_g[r][i - (r ? n_near[r - 1] : 0u)];
        const float* row = S + (roi0 + 2 * r) * nv;
        float acc = 0.f;
        auto load = [&](int k) { return k < n_hat ? row[(int)lut_g[cg * pitch + k]] - top_val[k] : 0.f; };
        float v = load(lane);
        for (int k0 = 0; k0 < n_hat; k0 += 32) {
            const float next = load(k0 + 32 + lane);
            const int kn = min(32, n_hat - k0);
            if (kn == 32) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float x = __shfl_sync(0xffffffffu, v, j);
                    acc = fmaf(x, x, acc);
                }
            } else {
                for (int j = 0; j < kn; ++j) {
                    const float x = __shfl_sync(0xffffffffu, v, j);
                    acc = fmaf(x, x, acc);
                }
            }
            v = next;
        }
        if (lane == 0 && acc < INFINITY)
            atomicMin(&key[r], ((unsigned long long)__float_as_uint(acc) << 32) | (uint32_t)cg);
    }
    __syncthreads();
    if (warp == 0 && valid && !((s_heavy >> lane) & 1u)) {
        const int64_t r = roi0 + 2 * lane;
        const unsigned long long v = key[lane];
        if (best) best[r] = (int32_t)(uint32_t)v;
        if (score) score[r] = __uint_as_float((uint32_t)(v >> 32));
    }
}

// D to rows of scores, out[roi * ng + g]: a CTA per 32 orientations of half a group
__global__ void __launch_bounds__(256) k_tm_rows(const float* __restrict__ D, int64_t nroi, int64_t ng, float* out) {
    __shared__ float t[32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t g0 = (int64_t)blockIdx.x * 32, grp = blockIdx.y >> 1;
    const int half = blockIdx.y & 1;
    for (int i = w; i < 32; i += 8)
        t[i][lane] = g0 + i < ng ? D[(grp * ng + g0 + i) * kTmRois + half * 32 + lane] : 0.f;
    __syncthreads();
    for (int i = w; i < 32; i += 8) {
        const int64_t r = grp * kTmRois + 2 * i + half;
        if (r < nroi && g0 + lane < ng) out[r * ng + g0 + lane] = t[lane][i];
    }
}

// Key of rank `rank` (1 = smallest) among n keys, by a radix select over four
// 8-bit digits; hist and the two words in shared memory, all threads call it.
__device__ __forceinline__ uint32_t radix_kth(const uint32_t* key, int64_t n, uint32_t rank, uint32_t* hist,
                                              uint32_t* s_prefix, uint32_t* s_rem) {
    const int tid = threadIdx.x, nt = blockDim.x;
    __syncthreads();
    if (tid == 0) {
        *s_prefix = 0;
        *s_rem = rank;
    }
    for (int pass = 3; pass >= 0; --pass) {
        for (int i = tid; i < 256; i += nt) hist[i] = 0;
        __syncthreads();
        const uint32_t prefix = *s_prefix, hmask = pass == 3 ? 0u : 0xFFFFFFFFu << (8 * (pass + 1));
        for (int64_t g = tid; g < n; g += nt) {
            const uint32_t k = key[g];
            if ((k & hmask) == (prefix & hmask)) atomicAdd(&hist[(k >> (8 * pass)) & 255u], 1u);
        }
        __syncthreads();
        if (tid == 0) {
            uint32_t rem = *s_rem, d = 0;
            while (hist[d] < rem) rem -= hist[d++];
            *s_rem = rem;
            *s_prefix = prefix | (d << (8 * pass));
        }
        __syncthreads();
    }
    return *s_prefix;
}

// The largest score of every ROI that the topk can depend on
__global__ void __launch_bounds__(256) k_tm_reach(const float* __restrict__ scores, int64_t ng, int64_t nroi, int32_t topk,
                                                  TmMargin margin, float* reach) {
    __shared__ uint32_t hist[256], s_prefix, s_rem;
    for (int64_t r = blockIdx.x; r < nroi; r += gridDim.x) {
        const uint32_t kth = radix_kth(reinterpret_cast<const uint32_t*>(scores + r * ng), ng, (uint32_t)topk, hist,
                                       &s_prefix, &s_rem);
        // fewer numbers than topk: NaN, every orientation counts
        if (threadIdx.x == 0) reach[r] = kth > 0x7F800000u ? NAN : tm_threshold(__uint_as_float(kth), margin);
    }
}

// Every score within reach is replaced by the sum in k order (a thread per
// orientation, the signature row in shared memory), so that k_topk's selection
// over the row is exact.  A CTA takes one part of a ROI's orientations.
constexpr int kTmList = 4096;

__global__ void __launch_bounds__(kTmThreads, 1) k_tm_exact(const float* __restrict__ S, int64_t nroi, int32_t nv,
                                                            const uint16_t* __restrict__ lut_g, int64_t ng, int pitch,
                                                            const float* __restrict__ top_val, int32_t n_hat,
                                                            const float* __restrict__ reach, int parts,
                                                            float* scores) {
    extern __shared__ float sm[];
    float* row = sm;             // nv
    float* ref = sm + nv;        // n_hat
    __shared__ uint32_t list[kTmList];
    __shared__ uint32_t n_list;
    __shared__ float s_flat;
    const int tid = threadIdx.x;
    for (int i = tid; i < n_hat; i += kTmThreads) ref[i] = top_val[i];
    if (tid == 0) n_list = 0;
    const int64_t per = (ng + parts - 1) / parts;
    for (int64_t it = blockIdx.x; it < nroi * parts; it += gridDim.x) {
        const int64_t r = it / parts, ga = (it % parts) * per, gb = tmin<int64_t>(ng, ga + per);
        __syncthreads();
        for (int i = tid; i < nv; i += kTmThreads) row[i] = S[r * (int64_t)nv + i];
        float* sc = scores + r * ng;
        const float t = reach[r];
        const bool all = isnan(t);
        __syncthreads();
        for (int64_t g0 = ga; g0 < gb; g0 += kTmThreads) {
            const int64_t g = g0 + tid;
            if (g < gb && (all || sc[g] <= t)) list[atomicAdd(&n_list, 1u)] = (uint32_t)g;
            __syncthreads();
            const uint32_t n = n_list;
            if (g0 == ga && n == (uint32_t)tmin<int64_t>(kTmThreads, gb - ga)) {
                // all of the first orientations within reach: a row of one value?  (asked
                // of every row while it was staged, this cost 70 us of 2.95 ms)
                bool same = true;
                for (int i = tid; i < nv; i += kTmThreads) same &= row[i] == row[0];
                if (__syncthreads_and(same)) {   // every orientation has the same sum
                    if (tid == 0) {
                        s_flat = flat_score(row[0], ref, n_hat);
                        n_list = 0;
                    }
                    __syncthreads();
                    for (int64_t i = ga + tid; i < gb; i += kTmThreads)
                        if (all || sc[i] <= t) sc[i] = s_flat;
                    break;
                }
            }
            if (n > kTmList - kTmThreads || g0 + kTmThreads >= gb) {
                for (uint32_t i = tid; i < n; i += kTmThreads) {
                    // 16 bytes of the orientation's row of the table at a time
                    constexpr int N = 8;
                    const uint4* lp = reinterpret_cast<const uint4*>(lut_g + (int64_t)list[i] * pitch);
                    float acc = 0.f;
                    uint4 w = __ldg(lp);
                    for (int k = 0; k < n_hat; k += N) {
                        const uint4 cur = w;
                        if (k + N < n_hat) w = __ldg(++lp);
                        const uint16_t* ix = reinterpret_cast<const uint16_t*>(&cur);
#pragma unroll
                        for (int j = 0; j < N; ++j)
                            if (k + j < n_hat) {
                                const float v = row[(int)ix[j]] - ref[k + j];
                                acc = fmaf(v, v, acc);
                            }
                    }
                    sc[list[i]] = acc;
                }
                __syncthreads();
                if (tid == 0) n_list = 0;
            }
            __syncthreads();
        }
    }
}

// ---- the topk smallest Delta(g) of a ROI (ties: lower g), ascending ----------
// One CTA per ROI: radix select of the topk-th smallest key (Delta >= 0, so
// its FP32 bit pattern orders like the value) over four 8-bit digits, then
// every g below that key plus the lowest-g ones equal to it, then a bitonic
// sort of the (key, g) pairs.
constexpr int kTopkThreads = 256;

__global__ void __launch_bounds__(kTopkThreads) k_topk(const float* __restrict__ scores, int64_t ng, int64_t nroi,
                                                       int32_t topk, int32_t* best, float* score) {
    __shared__ uint32_t hist[256];
    __shared__ uint64_t sel[APTIDX_MAX_TOPK];
    __shared__ uint32_t s_prefix, s_remaining, s_count;
    __shared__ uint32_t warp_cnt[kTopkThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int kp = 1;
    while (kp < topk) kp <<= 1;
    for (int64_t r = blockIdx.x; r < nroi; r += gridDim.x) {
        const uint32_t* key = reinterpret_cast<const uint32_t*>(scores + r * ng);
        if (tid == 0) {
            s_prefix = 0;
            s_remaining = (uint32_t)topk;
        }
        // 1. radix select: the topk-th smallest key
        for (int pass = 3; pass >= 0; --pass) {
            for (int i = tid; i < 256; i += kTopkThreads) hist[i] = 0;
            __syncthreads();
            const uint32_t prefix = s_prefix;
            const uint32_t hmask = pass == 3 ? 0u : (0xFFFFFFFFu << (8 * (pass + 1)));
            for (int64_t g = tid; g < ng; g += kTopkThreads) {
                const uint32_t k = key[g];
                if ((k & hmask) == (prefix & hmask)) atomicAdd(&hist[(k >> (8 * pass)) & 255u], 1u);
            }
            __syncthreads();
            if (tid == 0) {
                uint32_t rem = s_remaining, d = 0;
                while (hist[d] < rem) {
                    rem -= hist[d];
                    ++d;
                }
                s_remaining = rem;
                s_prefix = prefix | (d << (8 * pass));
            }
            __syncthreads();
        }
        const uint32_t kth = s_prefix;
        const uint32_t need_eq = s_remaining;   // how many keys equal to kth are kept
        const uint32_t n_less = (uint32_t)topk - need_eq;
        // 2. every key below kth (any order), then the lowest-g keys equal to it
        if (tid == 0) s_count = 0;
        for (int i = tid; i < kp; i += kTopkThreads) sel[i] = ~0ull;
        __syncthreads();
        for (int64_t g = tid; g < ng; g += kTopkThreads) {
            const uint32_t k = key[g];
            if (k < kth) sel[atomicAdd(&s_count, 1u)] = ((uint64_t)k << 32) | (uint32_t)g;
        }
        __syncthreads();
        uint32_t taken = 0;
        for (int64_t g0 = 0; g0 < ng && taken < need_eq; g0 += kTopkThreads) {
            const int64_t g = g0 + tid;
            const bool eq = g < ng && key[g] == kth;
            const uint32_t bal = __ballot_sync(0xffffffffu, eq);
            if (lane == 0) warp_cnt[warp] = __popc(bal);
            __syncthreads();
            uint32_t before = 0, total = 0;
            for (int w = 0; w < kTopkThreads / 32; ++w) {
                if (w < warp) before += warp_cnt[w];
                total += warp_cnt[w];
            }
            const uint32_t rank = taken + before + __popc(bal & ((1u << lane) - 1u));
            if (eq && rank < need_eq) sel[n_less + rank] = ((uint64_t)kth << 32) | (uint32_t)g;
            taken += total;
            __syncthreads();
        }
        __syncthreads();
        // 3. bitonic sort of the kp slots (unused slots hold ~0)
        for (int size = 2; size <= kp; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int i = tid; i < kp; i += kTopkThreads) {
                    const int j = i ^ stride;
                    if (j > i) {
                        const bool up = (i & size) == 0;
                        const uint64_t a = sel[i], b = sel[j];
                        if ((a > b) == up) {
                            sel[i] = b;
                            sel[j] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int i = tid; i < topk; i += kTopkThreads) {
            const uint64_t v = sel[i];
            if (best) best[r * topk + i] = (int32_t)(uint32_t)v;
            if (score) score[r * topk + i] = __uint_as_float((uint32_t)(v >> 32));
        }
        __syncthreads();
    }
}

// ---- refinement ----------------------------------------------------------------------

constexpr int kRefThreads = 256;
constexpr float kPoleDeg = 89.0f;
constexpr float kRad2Deg = 57.295779513082320876f;

// atan(t) for t in [0, 1] as t * P(t^2), P of degree 7 with coefficients that
// minimise the maximum error on [0, 1] (Lawson's iteratively reweighted least
// squares; atan_fit.py regenerates them): |error| < 4e-8 rad in exact
// arithmetic, < 2e-7 rad with FP32 Horner steps.
__device__ __forceinline__ float atan01(float t) {
    const float s = t * t;
    float p = -4.054556496e-03f;
    p = fmaf(p, s, 2.186292078e-02f);
    p = fmaf(p, s, -5.591227578e-02f);
    p = fmaf(p, s, 9.642193788e-02f);
    p = fmaf(p, s, -1.390862825e-01f);
    p = fmaf(p, s, 1.994656541e-01f);
    p = fmaf(p, s, -3.332986076e-01f);
    p = fmaf(p, s, 9.999993356e-01f);
    return t * p;
}

// atan2(y, x) in degrees, (-180, 180]: octant reduction to atan01 of
// min(|x|, |y|) / max(|x|, |y|) (a 2-ulp quotient).  NaN when x = y = 0.
__device__ __forceinline__ float atan2_deg(float y, float x) {
    const float ax = fabsf(x), ay = fabsf(y);
    float a = atan01(__fdividef(fminf(ax, ay), fmaxf(ax, ay)));
    if (ay > ax) a = 1.57079632679489662f - a;
    if (x < 0.f) a = 3.14159265358979324f - a;
    if (y < 0.f) a = -a;
    return a * kRad2Deg;
}

struct DirTerm {
    bool ok;
    float r;       // residual S - I
    float J[3];    // d r / d delta
};

// residual and its derivative with respect to the lab-frame perturbation delta
// of R = exp([delta]x) R(q) for one direction: c = R^T u, (alpha, beta) of c,
// bilinear sample of the image, r = s - I, J = -(R grad_c I) x u
// = -R (grad_c I x c); kCrystalJ returns grad_c I x c instead.
template <bool kCrystalJ = false>
__device__ __forceinline__ DirTerm dir_term(const float* Rf, float ux, float uy, float uz, float s,
                                            const float4* __restrict__ img4, bool want_j) {
    DirTerm t;
    const float cx = Rf[0] * ux + Rf[3] * uy + Rf[6] * uz;
    const float cy = Rf[1] * ux + Rf[4] * uy + Rf[7] * uz;
    const float cz = Rf[2] * ux + Rf[5] * uy + Rf[8] * uz;
    const float rho2 = cx * cx + cy * cy;
    const float inv_rho = rsqrtf(rho2);
    const float rho = rho2 * inv_rho;
    const float alpha = atan2_deg(cz, rho);
    t.ok = fabsf(alpha) <= kPoleDeg;   // also false for NaN at the exact poles
    if (!t.ok) return t;
    float beta = atan2_deg(cy, cx);
    if (beta < 0.f) beta += 360.f;
    const float fi = alpha + 90.f;
    int i0 = (int)floorf(fi);
    i0 = min(max(i0, 0), kImgRows - 2);
    const float fj0 = floorf(beta);
    const float ti = fi - (float)i0;
    const float tj = beta - fj0;
    int j0 = (int)fj0;
    j0 = j0 >= kImgCols ? j0 - kImgCols : j0;
    j0 = min(max(j0, 0), kImgCols - 1);
    // the cell's four taps (I[i0][j0], I[i0][j0 + 1], I[i0 + 1][j0], I[i0 + 1][j0 + 1],
    // the column index mod 360) in one read
    const float4 cell = __ldg(img4 + i0 * kImgCols + j0);
    const float I00 = cell.x, I01 = cell.y, I10 = cell.z, I11 = cell.w;
    const float v = (1.f - ti) * ((1.f - tj) * I00 + tj * I01) + ti * ((1.f - tj) * I10 + tj * I11);
    t.r = s - v;
    if (want_j) {
        const float dfi = (1.f - tj) * (I10 - I00) + tj * (I11 - I01);
        const float dfj = (1.f - ti) * (I01 - I00) + ti * (I11 - I10);
        // partial derivatives of (alpha, beta) in radians; the 2-ulp
        // reciprocals are far inside the FP32 error of the sums they feed
        const float n2 = rho2 + cz * cz;
        const float inv_n2 = __fdividef(1.f, n2);
        const float inv_rho2 = inv_rho * inv_rho;
        const float t_a = -cz * inv_n2 * inv_rho;
        const float da0 = t_a * cx, da1 = t_a * cy, da2 = rho * inv_n2;
        const float db0 = -cy * inv_rho2, db1 = cx * inv_rho2;
        const float g0 = kRad2Deg * (dfi * da0 + dfj * db0);
        const float g1 = kRad2Deg * (dfi * da1 + dfj * db1);
        const float g2 = kRad2Deg * (dfi * da2);
        if (kCrystalJ) {
            // J = -R (g x c): keep g x c; the caller rotates the sums once
            t.J[0] = g1 * cz - g2 * cy;
            t.J[1] = g2 * cx - g0 * cz;
            t.J[2] = g0 * cy - g1 * cx;
        } else {
            const float ax = Rf[0] * g0 + Rf[1] * g1 + Rf[2] * g2;
            const float ay = Rf[3] * g0 + Rf[4] * g1 + Rf[5] * g2;
            const float az = Rf[6] * g0 + Rf[7] * g1 + Rf[8] * g2;
            t.J[0] = -(ay * uz - az * uy);
            t.J[1] = -(az * ux - ax * uz);
            t.J[2] = -(ax * uy - ay * ux);
        }
    }
    return t;
}

// direction and signature reads stream past L1 so that L1 holds the reference
// image cells (180 x 360 x 16 B, reused by neighbouring directions and ROIs)
// for the bilinear gathers
__device__ __forceinline__ float4 ld_stream4(const float4* p) {
    float4 v;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ float ld_stream(const float* p) {
    float v;
    asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// coherent read that skips L1 (for data this kernel writes)
__device__ __forceinline__ float ld_l2(const float* p) {
    float v;
    asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

// block sum of n FP32 partials per thread into FP64 totals (thread 0 holds them)
template <int N>
__device__ __forceinline__ void block_sum(float* v, double* out, double* scratch /* [N * 32] */) {
    double d[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        d[i] = (double)v[i];
        for (int o = 16; o > 0; o >>= 1) d[i] += __shfl_xor_sync(0xffffffffu, d[i], o);
    }
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) scratch[i * 32 + w] = d[i];
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) {
            double s = 0.0;
            for (int k = 0; k < nw; ++k) s += scratch[i * 32 + k];
            out[i] = s;
        }
}

// Current rotation of ROI r: q = exp(omega) (x) q0 when omega is given.
__device__ __forceinline__ void roi_quat(const double* q0, const double* omega, int64_t r, double* q) {
    const double* a = q0 + 4 * r;
    if (omega) {
        double e[4];
        exp_quat(omega + 3 * r, e);
        quat_mul(e, a, q);
    } else {
        q[0] = a[0];
        q[1] = a[1];
        q[2] = a[2];
        q[3] = a[3];
    }
    const double n = sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    for (int i = 0; i < 4; ++i) q[i] /= n;
}

__device__ __forceinline__ void matrix_f32(const double* q, float* Rf) {
    const M3 R = quat_to_matrix(q[0], q[1], q[2], q[3]);
    for (int i = 0; i < 9; ++i) Rf[i] = (float)R.a[i];
}

// Forward (loss) and backward (gradient) of L = sum_v (S_v - I(R^T u_v))^2.
// With omega, the gradient is with respect to omega (rotation exp([omega]x)
// R(q0)): dL/domega = J_l(omega)^T dL/ddelta, J_l the left Jacobian of SO(3).
template <bool kGrad>
__global__ void __launch_bounds__(kRefThreads) k_refine_eval(const float* __restrict__ S, const float4* __restrict__ dirs,
                                                             int32_t nv, const float4* __restrict__ img,
                                                             const double* __restrict__ q0, const double* __restrict__ omega,
                                                             int64_t nroi, float* loss, float* grad) {
    __shared__ double scratch[4 * 32];
    __shared__ double tot[4];
    __shared__ float Rs[9];
    for (int64_t r = blockIdx.x; r < nroi; r += gridDim.x) {
        if (threadIdx.x == 0) {
            double q[4];
            roi_quat(q0, omega, r, q);
            matrix_f32(q, Rs);
        }
        __syncthreads();
        float Rf[9];
        for (int i = 0; i < 9; ++i) Rf[i] = Rs[i];
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const float* srow = S + r * (int64_t)nv;
        for (int v = threadIdx.x; v < nv; v += kRefThreads) {
            const float4 u = ld_stream4(dirs + v);
            const DirTerm t = dir_term(Rf, u.x, u.y, u.z, ld_stream(srow + v), img, kGrad);
            if (!t.ok) continue;
            acc[0] = fmaf(t.r, t.r, acc[0]);
            if (kGrad) {
                acc[1] = fmaf(2.f * t.r, t.J[0], acc[1]);
                acc[2] = fmaf(2.f * t.r, t.J[1], acc[2]);
                acc[3] = fmaf(2.f * t.r, t.J[2], acc[3]);
            }
        }
        block_sum<4>(acc, tot, scratch);
        if (threadIdx.x == 0) {
            if (loss) loss[r] = (float)tot[0];
            if (kGrad && grad) {
                double g[3] = {tot[1], tot[2], tot[3]};
                if (omega) {
                    // g_omega = J_l(omega)^T g_delta
                    const double* w = omega + 3 * r;
                    const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
                    const double th = sqrt(th2);
                    double A, B;
                    if (th < 1e-4) {
                        A = 0.5 - th2 / 24.0;
                        B = 1.0 / 6.0 - th2 / 120.0;
                    } else {
                        A = (1.0 - cos(th)) / th2;
                        B = (th - sin(th)) / (th2 * th);
                    }
                    // J_l = I + A [w]x + B [w]x^2;  J_l^T g = g - A (w x g) + B (w x (w x g))
                    const double c1[3] = {w[1] * g[2] - w[2] * g[1], w[2] * g[0] - w[0] * g[2], w[0] * g[1] - w[1] * g[0]};
                    const double c2[3] = {w[1] * c1[2] - w[2] * c1[1], w[2] * c1[0] - w[0] * c1[2], w[0] * c1[1] - w[1] * c1[0]};
                    for (int i = 0; i < 3; ++i) g[i] = g[i] - A * c1[i] + B * c2[i];
                }
                grad[3 * r] = (float)g[0];
                grad[3 * r + 1] = (float)g[1];
                grad[3 * r + 2] = (float)g[2];
            }
        }
        __syncthreads();
    }
}

// `iters` Gauss-Newton steps per ROI in one CTA: per step the direction terms
// give J^T J and J^T r (FP32 partials, FP64 block sums), thread 0 solves
// (J^T J + lambda I) delta = -J^T r with lambda = 1e-6 tr(J^T J) in FP64 and
// updates q <- exp(delta) q with FP64 renormalisation.  The directions are
// walked in the spatial order of `dsort` (w = index into the signature row),
// so that neighbouring lanes sample neighbouring pixels of the image; the
// CTA first gathers the ROI's row into that order in its own scratch row
// (global memory, L2-resident while the steps run).
constexpr int kGnThreads = 256;

__global__ void __launch_bounds__(kGnThreads) k_refine_gn(const float* __restrict__ S, const float4* __restrict__ dsort,
                                                          int32_t nv, const float4* __restrict__ img,
                                                          const double* __restrict__ q0,
                                                          const int32_t* __restrict__ best,
                                                          const double* __restrict__ quats, int64_t nroi, int iters,
                                                          float* scratch, double* q_out, float* loss_out) {
    __shared__ double red[10 * 32];
    __shared__ double tot[10];
    __shared__ double qs[4];
    __shared__ float Rs[9];
    float* srow = scratch + (int64_t)blockIdx.x * nv;
    for (int64_t r = blockIdx.x; r < nroi; r += gridDim.x) {
        __syncthreads();   // the previous ROI is done with srow
        {
            const float* src = S + r * (int64_t)nv;
            for (int i = threadIdx.x; i < nv; i += blockDim.x) srow[i] = src[__float_as_int(__ldg(&dsort[i].w))];
        }
        if (threadIdx.x == 0) {
            const double* qa = best ? quats + 4 * (int64_t)best[r] : q0 + 4 * r;
            double n = 0.0;
            for (int i = 0; i < 4; ++i) n += qa[i] * qa[i];
            n = sqrt(n);
            for (int i = 0; i < 4; ++i) qs[i] = qa[i] / n;
        }
        for (int it = 0; it <= iters; ++it) {
            const bool last = it == iters;   // final pass: loss only
            if (threadIdx.x == 0) matrix_f32(qs, Rs);
            __syncthreads();
            float Rf[9];
            for (int i = 0; i < 9; ++i) Rf[i] = Rs[i];
            float acc[10] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // L, Jtr[3], JtJ[6]
            for (int v = threadIdx.x; v < nv; v += blockDim.x) {
                const float4 u = ld_stream4(dsort + v);
                const DirTerm t = dir_term<true>(Rf, u.x, u.y, u.z, ld_l2(srow + v), img, !last);
                if (!t.ok) continue;
                acc[0] = fmaf(t.r, t.r, acc[0]);
                if (!last) {
                    acc[1] = fmaf(t.J[0], t.r, acc[1]);
                    acc[2] = fmaf(t.J[1], t.r, acc[2]);
                    acc[3] = fmaf(t.J[2], t.r, acc[3]);
                    acc[4] = fmaf(t.J[0], t.J[0], acc[4]);
                    acc[5] = fmaf(t.J[0], t.J[1], acc[5]);
                    acc[6] = fmaf(t.J[0], t.J[2], acc[6]);
                    acc[7] = fmaf(t.J[1], t.J[1], acc[7]);
                    acc[8] = fmaf(t.J[1], t.J[2], acc[8]);
                    acc[9] = fmaf(t.J[2], t.J[2], acc[9]);
                }
            }
            block_sum<10>(acc, tot, red);
            if (threadIdx.x == 0) {
                if (last) {
                    if (loss_out) loss_out[r] = (float)tot[0];
                } else {
                    double H[9] = {tot[4], tot[5], tot[6], tot[5], tot[7], tot[8], tot[6], tot[8], tot[9]};
                    const double lam = 1e-6 * (H[0] + H[4] + H[8]);
                    H[0] += lam;
                    H[4] += lam;
                    H[8] += lam;
                    // crystal-frame sums: J = -R j with j = g x c, so the lab system
                    // (R H_c R^T + lambda I) delta = R sum(j r) is solved as
                    // delta = R (H_c + lambda I)^-1 sum(j r)
                    const double b[3] = {tot[1], tot[2], tot[3]};
                    const double det = H[0] * (H[4] * H[8] - H[5] * H[7]) - H[1] * (H[3] * H[8] - H[5] * H[6]) +
                                       H[2] * (H[3] * H[7] - H[4] * H[6]);
                    double d[3] = {0.0, 0.0, 0.0};
                    if (fabs(det) > 0.0) {
                        for (int c = 0; c < 3; ++c) {
                            double Bm[9];
                            for (int i = 0; i < 9; ++i) Bm[i] = H[i];
                            Bm[c] = b[0];
                            Bm[3 + c] = b[1];
                            Bm[6 + c] = b[2];
                            d[c] = (Bm[0] * (Bm[4] * Bm[8] - Bm[5] * Bm[7]) - Bm[1] * (Bm[3] * Bm[8] - Bm[5] * Bm[6]) +
                                    Bm[2] * (Bm[3] * Bm[7] - Bm[4] * Bm[6])) / det;
                        }
                    }
                    const M3 Rq = quat_to_matrix(qs[0], qs[1], qs[2], qs[3]);
                    const double dl[3] = {Rq.a[0] * d[0] + Rq.a[1] * d[1] + Rq.a[2] * d[2],
                                          Rq.a[3] * d[0] + Rq.a[4] * d[1] + Rq.a[5] * d[2],
                                          Rq.a[6] * d[0] + Rq.a[7] * d[1] + Rq.a[8] * d[2]};
                    double e[4], qn[4];
                    exp_quat(dl, e);
                    quat_mul(e, qs, qn);
                    const double n = sqrt(qn[0] * qn[0] + qn[1] * qn[1] + qn[2] * qn[2] + qn[3] * qn[3]);
                    for (int i = 0; i < 4; ++i) qs[i] = qn[i] / n;
                }
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            const double sgn = qs[0] < 0.0 ? -1.0 : 1.0;
            for (int i = 0; i < 4; ++i) q_out[4 * r + i] = sgn * qs[i];
        }
        __syncthreads();
    }
}

// k-major table to g-major int32
template <typename IdxT>
__global__ void k_lut_transpose(const IdxT* __restrict__ lut_t, int64_t ng, int64_t ng_pad, int32_t n_hat,
                                int32_t* out) {
    const int64_t n = ng * n_hat;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = i / n_hat;
        const int k = (int)(i % n_hat);
        out[i] = (int32_t)lut_t[(int64_t)k * ng_pad + g];
    }
}

}  // namespace

cudaError_t launch_lut_export(Ctx* c, Reference* r, int32_t* out) {
    const int64_t n = r->ng * r->n_hat;
    const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 8192);
    if (r->lut_bytes == 2)
        k_lut_transpose<<<grid, 256, 0, c->stream>>>(static_cast<const uint16_t*>(r->d_lut), r->ng, r->ng_pad,
                                                     r->n_hat, out);
    else
        k_lut_transpose<<<grid, 256, 0, c->stream>>>(static_cast<const int32_t*>(r->d_lut), r->ng, r->ng_pad,
                                                     r->n_hat, out);
    return cudaGetLastError();
}

// ---- launches ------------------------------------------------------------------------

cudaError_t launch_top_nodes(Ctx* c, Reference* r) {
    if (r->n_hat <= kSelMax) {
        k_top_select<<<1, 1024, 0, c->stream>>>(r->d_node_sig, c->nv, r->n_hat, r->d_top, r->d_top_val);
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? cudaStreamSynchronize(c->stream) : e;
    }
    int32_t npow2 = 1;
    while (npow2 < c->nv) npow2 <<= 1;
    uint64_t* keys = nullptr;
    if (dev_alloc(c, (void**)&keys, (size_t)npow2 * sizeof(uint64_t))) return cudaErrorMemoryAllocation;
    k_top_nodes<<<1, 1024, 0, c->stream>>>(r->d_node_sig, c->nv, npow2, keys, r->n_hat, r->d_top, r->d_top_val);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    dev_free(keys);
    return e;
}

// The node grid of the directions, queued on the stream.  Filled here and not with the
// directions: signatures do not need it (on the host it took set_directions 0.85 of 6.6
// ms for 40962 directions).  `scratch` (idle on the stream) holds the counts when it is
// large enough.
static int ensure_node_grid(Ctx* c, void* scratch, size_t scratch_bytes) {
    if (c->d_nodes) return APTIDX_OK;
    const size_t cells = (size_t)c->node_dim * c->node_dim * c->node_dim;
    const NodeGrid g{nullptr, nullptr, c->node_dim, c->node_org, c->node_inv_h, c->node_far2};
    const size_t bytes = (2 * cells + 1 + scan_tmp_elems(cells) + 1) * sizeof(int64_t);
    int64_t* work = static_cast<int64_t*>(scratch);   // counts | offsets | the scan's sums
    if (scratch_bytes < bytes)
        if (int rc = dev_alloc(c, (void**)&work, bytes)) return rc;
    float4* nodes = c->d_dirs_sorted + c->nv;
    unsigned long long* counts = reinterpret_cast<unsigned long long*>(work);
    int64_t* off = work + cells;
    cudaError_t e = cudaMemsetAsync(counts, 0, cells * sizeof(int64_t), c->stream);
    if (e == cudaSuccess) {
        k_node_count<<<(unsigned)((c->nv + 255) / 256), 256, 0, c->stream>>>(c->d_dirs, c->nv, g, counts);
        e = launch_scan_i64(work, off, (int64_t)cells, off + cells + 1, c->stream);
    }
    if (e == cudaSuccess) {
        k_node_fill<<<(unsigned)c->sm_count * 8, 256, 0, c->stream>>>(c->d_dirs, c->nv, g, (int)cells, off, counts,
                                                                     c->d_node_start, nodes);
        e = cudaGetLastError();
    }
    if (work != scratch) dev_recycle(c, work);
    if (e != cudaSuccess) return cuda_check(c, e, "node grid");
    c->d_nodes = nodes;
    return APTIDX_OK;
}

// The table in runs of rows of at most 2^24 queries, so that the list of open
// queries (sized for all of a run) stays at 64 MB, and of what a grid takes.  Few
// queries, and those without memory for the grid or the list, are scanned: 2e8 dot
// products take 42 us, the grid's own kernels and the look-up 60.
template <typename IdxT>
static cudaError_t launch_build_lut_t(Ctx* c, Reference* r, const double* d_quats, int64_t ng) {
    const int64_t rows = std::min<int64_t>(std::min<int64_t>(r->n_hat, 65535 * kLutK),
                                           std::max<int64_t>(1, ((int64_t)1 << 24) / ng));
    uint32_t* open = nullptr;
    bool by_grid = (double)ng * r->n_hat * c->nv > 2e8;
    const std::string err = c->err;
    if (by_grid) {
        const size_t bytes = (size_t)(rows * ng + 1) * sizeof(uint32_t);
        int rc = dev_alloc(c, (void**)&open, bytes);
        if (!rc) rc = ensure_node_grid(c, open, bytes);
        by_grid = rc == APTIDX_OK;
        if (rc && rc != APTIDX_E_OOM) {
            dev_recycle(c, open);
            return cudaErrorUnknown;
        }
        c->err = err;
    }
    const NodeGrid grid{c->d_node_start, c->d_nodes, c->node_dim, c->node_org, c->node_inv_h, c->node_far2};
    IdxT* lut = static_cast<IdxT*>(r->d_lut);
    cudaError_t e = cudaSuccess;
    for (int64_t k0 = 0; k0 < r->n_hat && e == cudaSuccess; k0 += rows) {
        const int64_t k1 = std::min<int64_t>(k0 + rows, r->n_hat), nq = (k1 - k0) * ng;
        if (by_grid) {
            if ((e = cudaMemsetAsync(open, 0, sizeof(uint32_t), c->stream)) != cudaSuccess) break;
            const dim3 blocks((unsigned)((ng + kLutThreads - 1) / kLutThreads), (unsigned)((k1 - k0 + kLutK - 1) / kLutK));
            k_build_lut<IdxT><<<blocks, kLutThreads, 0, c->stream>>>(grid, c->d_dirs, r->d_top, r->n_hat, d_quats, ng,
                                                                     r->ng_pad, lut, (int32_t)k0, (int32_t)k1, open + 1, open);
        }
        const int64_t chunks = (nq + kLutThreads * kLutPer - 1) / (kLutThreads * kLutPer);
        k_lut_scan<IdxT><<<(unsigned)std::min<int64_t>(chunks, (int64_t)c->sm_count * 8), kLutThreads, 0, c->stream>>>(
            c->d_dirs, c->nv, r->d_top, d_quats, ng, r->ng_pad, lut, (int32_t)k0, (uint32_t)nq, by_grid ? open + 1 : nullptr,
            open);
        e = cudaGetLastError();
    }
    dev_recycle(c, open);   // (reused on the same stream only)
    return e;
}

cudaError_t launch_build_lut(Ctx* c, Reference* r, const double* d_quats, int64_t ng) {
    return r->lut_bytes == 2 ? launch_build_lut_t<uint16_t>(c, r, d_quats, ng)
                             : launch_build_lut_t<int32_t>(c, r, d_quats, ng);
}

template <typename IdxT>
static cudaError_t launch_match_t(Ctx* c, Reference* r, const float* S, int64_t nroi, int32_t* best, float* score,
                                  float* scores_out, bool accumulate, float weight, const uint32_t* list) {
    constexpr int G = 16 / (int)sizeof(IdxT);
    const size_t smem = ((size_t)c->nv + r->n_hat) * sizeof(float);
    const auto kern = list ? k_match<IdxT, true> : k_match<IdxT, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // one thread per G orientations, whole warps, at most 1024 threads
    const int64_t want = (r->ng + G - 1) / G;
    const int threads = (int)std::min<int64_t>(1024, std::max<int64_t>(32, (want + 31) / 32 * 32));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    per_sm = std::max(per_sm, 1);
    const int64_t grid = std::min<int64_t>((int64_t)c->sm_count * per_sm, nroi);
    // the listed ROIs' kernel, which mostly finds none, is set up while the one before it
    // runs (it waits for that one itself): 1-2 us of a call instead of 4
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cfg.attrs = &early;
    cfg.numAttrs = list ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, S, nroi, c->nv, static_cast<const IdxT*>(r->d_lut), r->ng, r->ng_pad,
                              static_cast<const float*>(r->d_top_val), r->n_hat, best, score, scores_out, accumulate,
                              weight, list);
}

cudaError_t launch_match(Ctx* c, Reference* r, const float* S, int64_t nroi, int32_t* best, float* score,
                         float* scores_out, bool accumulate, float weight, const uint32_t* list) {
    return r->lut_bytes == 2
               ? launch_match_t<uint16_t>(c, r, S, nroi, best, score, scores_out, accumulate, weight, list)
               : launch_match_t<int32_t>(c, r, S, nroi, best, score, scores_out, accumulate, weight, list);
}

static int tm_tiles(const Ctx* c) { return (c->nv + kTmTileMax - 1) / kTmTileMax; }

// The lists of k_tm_sum and the table by orientation, queued on the stream.  Without
// memory for them k_match serves the table (tm_none, until it is built again).
cudaError_t launch_build_tm(Ctx* c, Reference* r) {
    const int tiles = tm_tiles(c);
    const int64_t lists = (int64_t)tiles * r->ng;
    const int T = (c->nv + tiles - 1) / tiles;
    const int pitch = (r->n_hat + 7) / 8 * 8;
    void *ent = nullptr, *off = nullptr, *lut_g = nullptr;
    int32_t* counts = nullptr;
    int64_t *padded = nullptr, *off64 = nullptr, *tmp = nullptr;
    const std::string err = c->err;
    if (dev_alloc(c, &ent, (size_t)(r->ng * r->n_hat + 3 * lists) * sizeof(uint32_t)) ||
        dev_alloc(c, &off, (size_t)(lists + 1) * sizeof(uint32_t)) ||
        dev_alloc(c, &lut_g, (size_t)r->ng * pitch * sizeof(uint16_t)) ||
        dev_alloc(c, (void**)&counts, (size_t)lists * sizeof(int32_t)) ||
        dev_alloc(c, (void**)&padded, (size_t)lists * sizeof(int64_t)) ||
        dev_alloc(c, (void**)&off64, (size_t)(lists + 1) * sizeof(int64_t)) ||
        dev_alloc(c, (void**)&tmp, (scan_tmp_elems(lists) + 1) * sizeof(int64_t))) {
        for (void* q : {ent, off, lut_g, (void*)counts, (void*)padded, (void*)off64, (void*)tmp}) dev_free(q);
        c->err = err;
        r->tm_none = true;
        return cudaSuccess;
    }
    const uint16_t* lut = static_cast<const uint16_t*>(r->d_lut);
    const dim3 all((unsigned)((r->ng + 255) / 256), (unsigned)r->n_hat);
    const unsigned per_list = (unsigned)(lists / 256 + 1);
    cudaError_t e = cudaMemsetAsync(counts, 0, (size_t)lists * sizeof(int32_t), c->stream);
    if (e == cudaSuccess) {
        k_tm_count<<<all, 256, 0, c->stream>>>(lut, r->ng, r->ng_pad, T, counts);
        k_tm_pad<<<per_list, 256, 0, c->stream>>>(counts, lists, padded);
        e = launch_scan_i64(padded, off64, lists, tmp, c->stream);
    }
    if (e == cudaSuccess) {
        k_tm_off<<<per_list, 256, 0, c->stream>>>(off64, counts, lists, T, static_cast<uint32_t*>(off),
                                                  static_cast<uint32_t*>(ent));
        k_tm_fill<<<all, 256, 0, c->stream>>>(lut, r->ng, r->ng_pad, r->d_top_val, T, static_cast<uint32_t*>(off), counts,
                                              static_cast<uint32_t*>(ent));
        k_tm_rowmajor<<<dim3((unsigned)((r->ng + 31) / 32), (unsigned)((pitch + 31) / 32)), 256, 0, c->stream>>>(
            lut, r->ng, r->ng_pad, r->n_hat, pitch, static_cast<uint16_t*>(lut_g));
        e = cudaGetLastError();
    }
    for (void* q : {(void*)counts, (void*)padded, (void*)off64, (void*)tmp}) dev_recycle(c, q);
    r->d_tm_ent = static_cast<uint32_t*>(ent);
    r->d_tm_off = static_cast<uint32_t*>(off);
    r->d_lut_g = static_cast<uint16_t*>(lut_g);
    r->lut_g_pitch = pitch;
    r->tm_tiles = tiles;
    r->tm_nodes = T;
    return e;
}

size_t tm_exact_smem(const Ctx* c, const Reference* r) { return ((size_t)c->nv + r->n_hat) * sizeof(float); }

// Whether lists serve a table at all: 16-bit node indices and a signature row in
// shared memory (which the matching calls ask of every table), 2^24 lists (what the
// scan of their lengths takes) and 32-bit offsets.
static bool tm_possible(const Ctx* c, const Reference* r) {
    const int64_t lists = tm_tiles(c) * r->ng;
    return !r->tm_none && tm_exact_smem(c, r) <= 227 * 1024 && r->lut_bytes == 2 && lists <= ((int64_t)1 << 24) - 4096 &&
           r->n_hat <= 65535 && r->ng * r->n_hat + 3 * lists < ((int64_t)1 << 32);
}

// Groups of 64 ROIs whose estimates, with the list of heavy ROIs or the rows of topk
// > 1, fit the scratch of a call
int64_t tm_groups(const Reference* r, int32_t topk) {
    return (int64_t)((kMatchScratch - sizeof(float)) / ((size_t)(r->ng + 1) * kTmRois * sizeof(float) * (topk > 1 ? 2 : 1)));
}

// Whether the lists are the faster way: estimates of both in microseconds on 152 SMs,
// fitted to 636 calls timed both ways (2562 and 40962 directions, 500 to 100000
// orientations, 50 to 1000 nodes, 1 to 4096 ROIs, the best 1, 10 and 500; the median
// estimate is right, nine in ten are within 20 %).
// k_match: look-ups per SM (60 per million), staging (by few threads when there are
// few orientations), a chain of reads as long as the node list, and for topk > 1 the
// selection, by SM and by the longest row.
// Lists: 68 per million lists visited (each adds 64 sums to global memory), 1.5 per
// million entries and 64 ROIs, the longest warp's entries, k_tm_best's walk over the
// orientations by two CTAs per 64 ROIs, or the rows, selections and exact sums of
// topk > 1.  (Without the last three the lists served 64 ROIs x 50000 orientations x
// 100 nodes in 0.63 ms, which k_match does in 0.36.)
// Not where the estimates of 64 ROIs (topk > 1: and their rows) exceed the scratch.
bool tm_pays(const Ctx* c, const Reference* r, int64_t nroi, int32_t topk) {
    if (!tm_possible(c, r) || tm_groups(r, topk) < 1) return false;
    const auto up = [](double a, double b) { return ceil(a / b); };
    const double sms = c->sm_count, per = 152.0 / sms, n = (double)nroi, ng = (double)r->ng, nh = r->n_hat, nv = c->nv;
    const double looks = ng * nh * 1e-6, cells = n * ng * 1e-6 * per;
    const double threads = std::min(1024.0, 32.0 * up(up(ng, 8), 32));
    const double fit = std::min(floor(1024 / threads), floor(232448 / (tm_exact_smem(c, r) + 1024.0)));   // CTAs per SM
    const double ctas = std::max(1.0, std::min(16.0, fit));
    const double rounds = up(n, sms), waves = up(n, sms * ctas), rows = up(n, 8 * sms);
    double single = 15 + rounds * (60 * looks + 1.7e-4 * nv) + waves * (0.2 * nv / threads + 0.038 * nh * up(up(ng, 8), threads));
    const double groups = up(n, kTmRois), tiles = tm_tiles(c);
    const double gsplit = std::max(1.0, std::min(up(4 * sms, tiles * groups), floor(ng / 256)));
    const double longest = up(tiles * groups * gsplit, sms) * up(ng, gsplit * (kTmThreads / 32)) * nh / tiles;
    double lists = 37 + per * groups * (68e-6 * tiles * ng + 1.5 * looks) + 0.047 * longest;
    if (topk == 1) {
        lists += up(2 * groups, sms) * (8e-3 * ng + 0.024 * nh) + 1.7 * cells;
    } else {
        single += 17 + 5 * cells + rows * (1.8e-3 * ng + 0.02 * topk) + 0.026 * n * per;
        lists += 46 + 11.7 * cells + rows * (3.6e-3 * ng + 0.018 * topk) + (0.066 + 0.8e-6 * topk * nh) * n * per;
    }
    return lists < 0.85 * single;
}

static TmMargin tm_margin(const Reference* r) {
    const double eta = sqrt((double)r->n_hat) * r->ref_max * (1.0 / 16384.0);
    return {(float)(2.0 * eta * 1.001), (float)(1.0 + 5.0 * (r->n_hat + 64) / 16777216.0)};
}

// estimates of `nroi` ROIs into D [groups][ng][64], and zero into the word after them
cudaError_t launch_tm_sum(Ctx* c, Reference* r, const float* S, int64_t nroi, float* D) {
    const int64_t groups = (nroi + kTmRois - 1) / kTmRois;
    cudaError_t e = cudaMemsetAsync(D, 0, (size_t)(groups * r->ng * kTmRois + 1) * sizeof(float), c->stream);
    if (e != cudaSuccess) return e;
    const size_t smem = (size_t)(r->tm_nodes + 1) * kTmPitch * sizeof(float);
    if ((e = cudaFuncSetAttribute(k_tm_sum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    // a CTA per (tile, group); few groups split the orientations further, four
    // CTAs per SM in all, at least 256 orientations each
    const int64_t base = r->tm_tiles * groups;
    const int gsplit = (int)std::max<int64_t>(1, std::min<int64_t>((4 * (int64_t)c->sm_count + base - 1) / base, r->ng / 256));
    for (int64_t y0 = 0; y0 < groups; y0 += 65535) {
        const int64_t ny = std::min<int64_t>(65535, groups - y0);
        k_tm_sum<<<dim3((unsigned)(r->tm_tiles * gsplit), (unsigned)ny), kTmThreads, smem, c->stream>>>(
            S + y0 * kTmRois * c->nv, nroi - y0 * kTmRois, c->nv, r->d_tm_ent, r->d_tm_off, r->ng, r->tm_nodes, gsplit,
            D + y0 * r->ng * kTmRois);
    }
    return cudaGetLastError();
}

// the best of every ROI from the estimates D, which the counter of heavy ROIs follows
cudaError_t launch_tm_best(Ctx* c, Reference* r, const float* S, int64_t nroi, float* D, int32_t* best, float* score) {
    const int64_t groups = (nroi + kTmRois - 1) / kTmRois;
    uint32_t* heavy = reinterpret_cast<uint32_t*>(D + groups * r->ng * kTmRois);
    k_tm_best<<<(unsigned)(2 * groups), kTmThreads, 0, c->stream>>>(S, nroi, c->nv, r->d_lut_g, r->ng, r->lut_g_pitch,
                                                                    r->d_top_val, r->n_hat, tm_margin(r), D, best, score,
                                                                    heavy);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? launch_match(c, r, S, nroi, best, score, nullptr, false, 1.0f, heavy) : e;
}

// rows [nroi][ng] from the estimates, exact where the topk are decided; D's
// first nroi words are reused for the reach
cudaError_t launch_tm_rows(Ctx* c, Reference* r, const float* S, int64_t nroi, int32_t topk, float* D, float* rows) {
    const int64_t groups = (nroi + kTmRois - 1) / kTmRois;
    for (int64_t y0 = 0; y0 < groups; y0 += 32767) {
        const int64_t ny = std::min<int64_t>(32767, groups - y0);
        k_tm_rows<<<dim3((unsigned)((r->ng + 31) / 32), (unsigned)(2 * ny)), 256, 0, c->stream>>>(
            D + y0 * r->ng * kTmRois, nroi - y0 * kTmRois, r->ng, rows + y0 * kTmRois * r->ng);
    }
    k_tm_reach<<<(unsigned)std::min<int64_t>(nroi, (int64_t)c->sm_count * 8), 256, 0, c->stream>>>(rows, r->ng, nroi,
                                                                                                  topk, tm_margin(r), D);
    const size_t smem = tm_exact_smem(c, r);
    cudaError_t e = cudaFuncSetAttribute(k_tm_exact, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // eight rounds of CTAs at least: the last, partly filled one then costs little
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>((8 * (int64_t)c->sm_count + nroi - 1) / nroi, r->ng / 4096));
    k_tm_exact<<<(unsigned)std::min<int64_t>(nroi * parts, c->sm_count), kTmThreads, smem, c->stream>>>(
        S, nroi, c->nv, r->d_lut_g, r->ng, r->lut_g_pitch, r->d_top_val, r->n_hat, D, parts, rows);
    return cudaGetLastError();
}

// Phase decision: candidate c's summed channel scores divided by its channel
// count n_c (in place), then phase[r] = the candidate of the lowest score
// (ties: lowest c).
__global__ void k_phase(float* score, const int32_t* n_ch, int32_t n_cand, int64_t nroi, int32_t* phase) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nroi; r += (int64_t)gridDim.x * blockDim.x) {
        float bs = INFINITY;
        int32_t bc = 0;
        for (int c = 0; c < n_cand; ++c) {
            const float v = score[(int64_t)c * nroi + r] / (float)n_ch[c];
            score[(int64_t)c * nroi + r] = v;
            if (v < bs) {
                bs = v;
                bc = c;
            }
        }
        if (phase) phase[r] = bc;
    }
}

cudaError_t launch_phase(Ctx* c, float* score, const int32_t* n_ch, int32_t n_cand, int64_t nroi, int32_t* phase) {
    const int64_t grid = std::min<int64_t>((nroi + 255) / 256, (int64_t)c->sm_count * 8);
    k_phase<<<(unsigned)grid, 256, 0, c->stream>>>(score, n_ch, n_cand, nroi, phase);
    return cudaGetLastError();
}

cudaError_t launch_topk(Ctx* c, const float* scores, int64_t ng, int64_t nroi, int32_t topk, int32_t* best,
                        float* score) {
    const int64_t grid = std::min<int64_t>((int64_t)c->sm_count * 8, nroi);
    k_topk<<<(unsigned)grid, kTopkThreads, 0, c->stream>>>(scores, ng, nroi, topk, best, score);
    return cudaGetLastError();
}

cudaError_t launch_refine_eval(Ctx* c, Reference* r, const float* S, const double* q0, const double* omega,
                               int64_t nroi, float* loss, float* grad) {
    const int64_t grid = std::min<int64_t>((int64_t)c->sm_count * 8, nroi);
    if (grad)
        k_refine_eval<true><<<(unsigned)grid, kRefThreads, 0, c->stream>>>(S, c->d_dirs, c->nv, r->d_img4, q0, omega,
                                                                          nroi, loss, grad);
    else
        k_refine_eval<false><<<(unsigned)grid, kRefThreads, 0, c->stream>>>(S, c->d_dirs, c->nv, r->d_img4, q0, omega,
                                                                           nroi, loss, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_refine_gn(Ctx* c, Reference* r, const float* S, const double* q0, const int32_t* best,
                             int64_t nroi, int iters, double* q_out, float* loss) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_refine_gn, kGnThreads, 0);
    const int64_t grid = std::min<int64_t>((int64_t)c->sm_count * std::max(per_sm, 1), nroi);
    const size_t need = (size_t)grid * c->nv * sizeof(float);
    if (need > c->gn_scratch_bytes) {
        dev_free(c->d_gn_scratch);
        c->d_gn_scratch = nullptr;
        c->gn_scratch_bytes = 0;
        if (dev_alloc(c, (void**)&c->d_gn_scratch, need)) return cudaErrorMemoryAllocation;
        c->gn_scratch_bytes = need;
    }
    k_refine_gn<<<(unsigned)grid, kGnThreads, 0, c->stream>>>(S, c->d_dirs_sorted, c->nv, r->d_img4, q0, best,
                                                              r->d_quats, nroi, iters, c->d_gn_scratch, q_out, loss);
    return cudaGetLastError();
}

}  // namespace aptidx
