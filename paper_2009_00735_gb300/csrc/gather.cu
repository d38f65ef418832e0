// gather.cu -- step (a1): ROI atom query and centring on the GPU.
//
// The paper queries the atoms of each ROI with a tree (supplement, cost term
// N_roi f R^3 rho log(V rho)).  Here the positions are bucketed once into a
// uniform cell grid (counting sort, cells ordered by atom index so results
// are deterministic), and one CTA per ROI walks the rows of cells that its
// sphere touches.  Membership is the FP64 closed-ball test
// (dx*dx + dy*dy) + dz*dz <= R*R without fused multiply-add, decided in FP32 where
// that is certain to agree, and the centred coordinates x_i - p_c are formed in FP64
// and rounded once to FP32 (Eq. 1: p_i - p_c).
#include <float.h>

#include "common.cuh"

namespace aptidx {

// -----------------------------------------------------------------------------
// bounding box
// -----------------------------------------------------------------------------
__device__ __forceinline__ int f2ord(float f) {
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7FFFFFFF;
}

__global__ void k_bbox_init(int* mm) {
    if (threadIdx.x < 3) mm[threadIdx.x] = 0x7FFFFFFF;
    else if (threadIdx.x < 6) mm[threadIdx.x] = (int)0x80000000;
}

__global__ void k_bbox(const float* __restrict__ pos, int64_t n, int* mm) {
    int lo[3] = {0x7FFFFFFF, 0x7FFFFFFF, 0x7FFFFFFF};
    int hi[3] = {(int)0x80000000, (int)0x80000000, (int)0x80000000};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int o = f2ord(pos[3 * i + d]);
            lo[d] = min(lo[d], o);
            hi[d] = max(hi[d], o);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int off = 16; off > 0; off >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
        }
    }
    if ((threadIdx.x & 31) == 0) {
        for (int d = 0; d < 3; ++d) {
            atomicMin(&mm[d], lo[d]);
            atomicMax(&mm[3 + d], hi[d]);
        }
    }
}

__global__ void k_bbox_decode(const int* mm, float* out) {
    int t = threadIdx.x;
    if (t < 6) {
        int i = mm[t];
        i = i >= 0 ? i : i ^ 0x7FFFFFFF;
        out[t] = __int_as_float(i);
    }
}

cudaError_t launch_bbox(const float* pos, int64_t n, float* d_minmax, cudaStream_t s) {
    int* mm = reinterpret_cast<int*>(d_minmax) + 6;   // caller provides 12 floats
    k_bbox_init<<<1, 32, 0, s>>>(mm);
    int blocks = (int)tmin<int64_t>((n + 255) / 256, 4096);
    k_bbox<<<blocks, 256, 0, s>>>(pos, n, mm);
    k_bbox_decode<<<1, 32, 0, s>>>(mm, d_minmax);
    return cudaGetLastError();
}

// -----------------------------------------------------------------------------
// exclusive scan of int64 (out[n] = total), up to 4096 * 4096 elements
// -----------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;
constexpr int kScanBlock = kScanThreads * kScanPer;

size_t scan_tmp_elems(int64_t n) { return (size_t)((n + kScanBlock - 1) / kScanBlock) + 1; }

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t* warp_sums, int64_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
        for (int off = 1; off < 32; off <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        warp_sums[lane] = w;   // inclusive
    }
    __syncthreads();
    int64_t before = warp == 0 ? 0 : warp_sums[warp - 1];
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    return before + x - v;
}

__global__ void k_scan_blocks(const int64_t* __restrict__ in, int64_t* out, int64_t n, int64_t* sums) {
    __shared__ int64_t ws[32];
    __shared__ int64_t tot;
    int64_t base = (int64_t)blockIdx.x * kScanBlock + threadIdx.x * kScanPer;
    int64_t v[kScanPer];
    int64_t local = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        v[i] = base + i < n ? in[base + i] : 0;
        local += v[i];
    }
    int64_t ex = block_exclusive_scan(local, ws, &tot);
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        if (base + i < n) out[base + i] = ex;
        ex += v[i];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(int64_t* sums, int64_t nb) {
    __shared__ int64_t ws[32];
    __shared__ int64_t tot;
    int64_t base = threadIdx.x * kScanPer;
    int64_t v[kScanPer];
    int64_t local = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        v[i] = base + i < nb ? sums[base + i] : 0;
        local += v[i];
    }
    int64_t ex = block_exclusive_scan(local, ws, &tot);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        if (base + i < nb) sums[base + i] = ex;
        ex += v[i];
    }
    if (threadIdx.x == 0) sums[nb] = tot;
}

__global__ void k_scan_add(int64_t* out, int64_t n, const int64_t* sums, int64_t nb) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += sums[i / kScanBlock];
    if (i == 0) out[n] = sums[nb];
}

cudaError_t launch_scan_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t s) {
    int64_t nb = (n + kScanBlock - 1) / kScanBlock;
    if (nb > kScanBlock) return cudaErrorInvalidValue;
    if (nb == 0) {
        return cudaMemsetAsync(out, 0, sizeof(int64_t), s);
    }
    k_scan_blocks<<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, tmp);
    k_scan_sums<<<1, kScanThreads, 0, s>>>(tmp, nb);
    k_scan_add<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(out, n, tmp, nb);
    return cudaGetLastError();
}

// -----------------------------------------------------------------------------
// cell grid
// -----------------------------------------------------------------------------
struct GridDesc {
    double lo[3];
    double inv_h;
    double h;
    int dims[3];
};

__device__ __forceinline__ int cell_coord(double x, double lo, double inv_h, int dim) {
    int i = (int)floor((x - lo) * inv_h);
    return min(max(i, 0), dim - 1);
}

__global__ void k_cell_of(const float* __restrict__ pos, int64_t n, GridDesc g, int32_t* cell_of,
                          unsigned long long* counts) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int ix = cell_coord((double)pos[3 * i + 0], g.lo[0], g.inv_h, g.dims[0]);
        int iy = cell_coord((double)pos[3 * i + 1], g.lo[1], g.inv_h, g.dims[1]);
        int iz = cell_coord((double)pos[3 * i + 2], g.lo[2], g.inv_h, g.dims[2]);
        int c = ix + g.dims[0] * (iy + g.dims[1] * iz);
        cell_of[i] = c;
        atomicAdd(&counts[c], 1ull);
    }
}

// Atom indices in cell order, ascending inside every cell: a stable
// least-significant-digit radix sort of the cell ids (8 bits per pass) with
// the atom index as value, starting from ascending indices.  A pass splits the
// keys into tiles of kRsTile; k_rs_count counts each tile's digits,
// an exclusive scan of the counts (digit-major) gives every (digit, tile) its
// output offset, and k_rs_scatter writes each tile's keys in order: within a
// chunk of 256 keys a key's position is its digit's running offset plus the
// same-digit keys of lower lanes (warp match) and of lower warps.
constexpr int kRsThreads = 256;
constexpr int kRsChunks = 16;
constexpr int kRsTile = kRsThreads * kRsChunks;
constexpr int kRsWarps = kRsThreads / 32;

__global__ void __launch_bounds__(kRsThreads) k_rs_count(const int32_t* __restrict__ keys, int64_t n, int shift,
                                                         int64_t ntiles, int64_t* hist) {
    __shared__ int32_t h[256];
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        h[threadIdx.x] = 0;
        __syncthreads();
        const int64_t t0 = tile * kRsTile;
        for (int i = threadIdx.x; i < kRsTile; i += kRsThreads) {
            const int64_t k = t0 + i;
            if (k < n) atomicAdd(&h[(keys[k] >> shift) & 255], 1);
        }
        __syncthreads();
        hist[(int64_t)threadIdx.x * ntiles + tile] = h[threadIdx.x];
        __syncthreads();
    }
}

// vin == nullptr: the values are the key positions (atom indices)
__global__ void __launch_bounds__(kRsThreads) k_rs_scatter(const int32_t* __restrict__ kin,
                                                           const int32_t* __restrict__ vin, int64_t n, int shift,
                                                           int64_t ntiles, const int64_t* __restrict__ offs,
                                                           int32_t* kout, int32_t* vout) {
    __shared__ unsigned long long base[256];
    __shared__ int32_t wcnt[kRsWarps][257];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < kRsWarps * 257; i += kRsThreads) (&wcnt[0][0])[i] = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        __syncthreads();
        base[tid] = (unsigned long long)offs[(int64_t)tid * ntiles + tile];
        for (int ch = 0; ch < kRsChunks; ++ch) {
            const int64_t k = tile * kRsTile + (int64_t)ch * kRsThreads + tid;
            const bool valid = k < n;
            const int32_t key = valid ? kin[k] : 0;
            const int32_t val = valid ? (vin ? vin[k] : (int32_t)k) : 0;
            const int d = valid ? ((key >> shift) & 255) : 256;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const bool leader = lane == __ffs(peers) - 1;
            const int rank = __popc(peers & ((1u << lane) - 1u));
            if (leader) wcnt[warp][d] = __popc(peers);
            __syncthreads();
            if (valid) {
                long long pos = (long long)base[d] + rank;
                for (int w = 0; w < warp; ++w) pos += wcnt[w][d];
                kout[pos] = key;
                vout[pos] = val;
            }
            __syncthreads();
            if (leader) {
                if (valid) atomicAdd(&base[d], (unsigned long long)__popc(peers));
                wcnt[warp][d] = 0;
            }
            __syncthreads();
        }
    }
}

__global__ void k_cell_fill(const float* __restrict__ pos, const uint8_t* __restrict__ types,
                            const int32_t* __restrict__ idx, int64_t n, float4* cell_pos) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = idx[k];
        float t = types ? (float)types[i] : 0.0f;
        cell_pos[k] = make_float4(pos[3 * (int64_t)i], pos[3 * (int64_t)i + 1], pos[3 * (int64_t)i + 2], t);
    }
}

static GridDesc grid_desc(const Ctx* c) {
    GridDesc g;
    for (int d = 0; d < 3; ++d) {
        g.lo[d] = c->lo[d];
        g.dims[d] = c->dims[d];
    }
    g.h = c->cell_h;
    g.inv_h = 1.0 / c->cell_h;
    return g;
}

// Build the cell grid of the loaded positions for the cell size c->cell_h.
// Scratch (caller-owned): cell_of, k2, idx, v2 [n] int32, counts [n_cells]
// int64, hist and offs [256 * ceil(n / kRsTile) + 1] int64.
size_t cell_sort_hist_elems(int64_t n) { return (size_t)256 * (size_t)((n + kRsTile - 1) / kRsTile) + 1; }

cudaError_t launch_cell_build(Ctx* c, int32_t* d_cell_of, int32_t* d_k2, int32_t* d_idx, int32_t* d_v2,
                              int64_t* d_counts, int64_t* d_hist, int64_t* d_offs) {
    cudaStream_t s = c->stream;
    GridDesc g = grid_desc(c);
    const int64_t n = c->n_atoms;
    int blocks = (int)tmin<int64_t>((n + 255) / 256, 8192);
    cudaError_t e;
    if ((e = cudaMemsetAsync(d_counts, 0, sizeof(int64_t) * c->n_cells, s)) != cudaSuccess) return e;
    k_cell_of<<<blocks, 256, 0, s>>>(c->d_pos, n, g, d_cell_of, reinterpret_cast<unsigned long long*>(d_counts));
    if ((e = launch_scan_i64(d_counts, c->d_cell_start, c->n_cells, c->d_scan_tmp, s)) != cudaSuccess) return e;
    // radix passes over the bits of the largest cell id
    int bits = 0;
    while (bits < 31 && ((int64_t)1 << bits) < c->n_cells) ++bits;
    const int passes = tmax(1, (bits + 7) / 8);
    const int64_t ntiles = (n + kRsTile - 1) / kRsTile;
    const unsigned rblocks = (unsigned)tmin<int64_t>(tmax<int64_t>(ntiles, 1), (int64_t)c->sm_count * 8);
    const int32_t* kin = d_cell_of;
    const int32_t* vin = nullptr;
    int32_t* kbuf[2] = {d_k2, d_cell_of};
    int32_t* vbuf[2] = {d_idx, d_v2};
    for (int pass = 0; pass < passes && ntiles > 0; ++pass) {
        k_rs_count<<<rblocks, kRsThreads, 0, s>>>(kin, n, 8 * pass, ntiles, d_hist);
        if ((e = launch_scan_i64(d_hist, d_offs, 256 * ntiles, c->d_scan_tmp, s)) != cudaSuccess) return e;
        k_rs_scatter<<<rblocks, kRsThreads, 0, s>>>(kin, vin, n, 8 * pass, ntiles, d_offs, kbuf[pass & 1],
                                                    vbuf[pass & 1]);
        kin = kbuf[pass & 1];
        vin = vbuf[pass & 1];
    }
    k_cell_fill<<<blocks, 256, 0, s>>>(c->d_pos, c->d_types, vin, n, c->d_cell_pos);
    return cudaGetLastError();
}

// -----------------------------------------------------------------------------
// ROI gather: one CTA per ROI.  The cells of a grid row (fixed iy, iz) are
// consecutive, so the atoms a row contributes are one contiguous run of
// cell_pos: a thread per row clips the row against the sphere, then warps walk
// the rows in chunks of 32 candidates (four loads in flight) and keep each
// chunk's member mask in shared memory; a prefix sum over the row counts gives
// every row its output offset and the members are written in (z, y, x) cell
// order, ascending atom index inside a cell.
//
// What bounds it: FP64, which this GPU issues at 1/64 of the FP32 rate.  The
// membership of Eq. 1's ROI is an FP64 comparison, so it is decided in FP32
// wherever the FP32 distance is clear of the sphere by more than its own error
// and in FP64 only in the shell between; only members pay the FP64 subtraction
// of the centre.  One warp per ROI with an FP64 test per cell and per candidate
// took 1.69 ms to count and 1.90 ms to write for 8192 ROIs of 1133 atoms; this
// takes 0.09 and 0.42 ms (512 such ROIs: 0.30 ms to write before, 0.04 now; 61
// ROIs of 9077 atoms: 1.16 ms before, 0.07 now).
// -----------------------------------------------------------------------------
constexpr int kGaRows = 128;      // grid rows handled at once
constexpr int kGaMasks = 2048;    // member masks kept (a batch of rows with more chunks tests membership twice)

struct GatherParams {
    GridDesc g;
    const int64_t* cell_start;
    const float4* cell_pos;
    const double* centres;
    const double* radii;
    int64_t nroi;
    uint32_t type_mask;
    int32_t* nw;           // atoms per ROI (both passes)
    const int64_t* off;    // fill pass: slot of ROI r is [off[r], off[r + 1])
    float4* atoms;         // fill pass output
    int* status;
};

// The ROI's sphere for the FP32 decision: the centre as a float pair and the
// squared radii below which an FP32 distance is certainly inside and above
// which it is certainly outside.  (a - ch) - cl carries two roundings of at
// most 2^-24 of its terms and the pair drops at most 2^-48 of the centre, so
// the FP32 square sum is within 1e-6 R^2 plus 1e-12 R |c| of the exact one for
// any distance near R.  NaN fails both comparisons and goes to FP64.
struct RoiSphere {
    float ch[3], cl[3], in2, out2;
};

// cd: the centre and R^2 (shared memory; read only by lanes in the shell)
__device__ __forceinline__ bool roi_member(const RoiSphere& s, const double* cd, float4 a, uint32_t type_mask) {
    const unsigned t = (unsigned)a.w;
    if (!(t < 32u && ((type_mask >> t) & 1u))) return false;
    const float dx = (a.x - s.ch[0]) - s.cl[0], dy = (a.y - s.ch[1]) - s.cl[1], dz = (a.z - s.ch[2]) - s.cl[2];
    const float q = dx * dx + dy * dy + dz * dz;
    if (q > s.out2) return false;
    if (q < s.in2) return true;
    const double ex = __dsub_rn((double)a.x, cd[0]), ey = __dsub_rn((double)a.y, cd[1]),
                 ez = __dsub_rn((double)a.z, cd[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) <= cd[3];
}

template <bool kFill>
__global__ void __launch_bounds__(512, 2) k_gather(GatherParams p) {
    __shared__ int64_t row_beg[kGaRows];
    __shared__ int32_t row_len[kGaRows];     // candidates of the row
    __shared__ int32_t row_mask[kGaRows];    // first entry of masks
    __shared__ int32_t row_cnt[kGaRows];     // members, then their exclusive prefix
    __shared__ uint32_t masks[kGaMasks];
    __shared__ int32_t s_chunks, s_members;
    __shared__ double cd[4];                 // centre, R^2
    __shared__ RoiSphere s_sphere;
    __shared__ int32_t lo3[3], hi3[3];       // cells the ROI's bounding box touches
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    for (int64_t r = blockIdx.x; r < p.nroi; r += gridDim.x) {
        __syncthreads();   // the ROI before is done with the shared state
        if (tid < 4) {
            const double R = p.radii[r];
            const double c0 = p.centres[3 * r], c1 = p.centres[3 * r + 1], c2 = p.centres[3 * r + 2];
            if (tid < 3) {
                const double c = tid == 0 ? c0 : tid == 1 ? c1 : c2;
                const float ch = (float)c;
                cd[tid] = c;
                s_sphere.ch[tid] = ch;
                s_sphere.cl[tid] = (float)(c - (double)ch);
                const double top = (double)(p.g.dims[tid] - 1);
                const double a = (c - R - p.g.lo[tid]) * p.g.inv_h - 1e-9;
                const double b = (c + R - p.g.lo[tid]) * p.g.inv_h + 1e-9;
                lo3[tid] = (int)fmin(fmax(floor(a), 0.0), top);
                hi3[tid] = (int)fmax(fmin(floor(b), top), -1.0);
            } else {
                const double R2 = __dmul_rn(R, R);
                const double m = 2e-6 * R2 + 1e-11 * (1.0 + fabs(c0) + fabs(c1) + fabs(c2)) * R;
                cd[3] = R2;
                s_sphere.in2 = __double2float_rd(R2 - m);
                s_sphere.out2 = __double2float_ru(R2 + m);
            }
        }
        __syncthreads();
        const RoiSphere s = s_sphere;
        const int ny = hi3[1] - lo3[1] + 1;
        const int64_t nrows = ny > 0 && hi3[2] >= lo3[2] && hi3[0] >= lo3[0] ? (int64_t)ny * (hi3[2] - lo3[2] + 1) : 0;
        const int64_t base = kFill ? p.off[r] : 0;
        const int64_t slot = kFill ? p.off[r + 1] - base : 0;
        int64_t count = 0;
        for (int64_t row0 = 0; row0 < nrows; row0 += kGaRows) {
            const int nb = (int)tmin<int64_t>(kGaRows, nrows - row0);
            __syncthreads();   // the batch before has been written out
            for (int i = tid; i < nb; i += blockDim.x) {
                const int64_t row = row0 + i;
                const int iy = lo3[1] + (int)(row % ny), iz = lo3[2] + (int)(row / ny);
                // distance of the row's (y, z) rectangle from the centre; cells
                // on the grid's faces hold atoms clamped into them and are
                // taken whole
                const double ylo = p.g.lo[1] + iy * p.g.h, zlo = p.g.lo[2] + iz * p.g.h;
                const double ty = fmax(fmax(ylo - cd[1], cd[1] - (ylo + p.g.h)), 0.0);
                const double tz = fmax(fmax(zlo - cd[2], cd[2] - (zlo + p.g.h)), 0.0);
                const double w2 = cd[3] * (1.0 + 1e-9) + 1e-12 - (ty * ty + tz * tz);
                const bool face = iy == 0 || iz == 0 || iy == p.g.dims[1] - 1 || iz == p.g.dims[2] - 1;
                int xa = lo3[0], xb = hi3[0];
                if (!face) {
                    if (w2 < 0.0) {
                        xb = xa - 1;
                    } else {
                        // half chord, rounded up (FP32 root)
                        const double w = (double)__fsqrt_ru(__double2float_ru(w2)) + 1e-9;
                        const double a = (cd[0] - w - p.g.lo[0]) * p.g.inv_h - 1e-9;
                        const double b = (cd[0] + w - p.g.lo[0]) * p.g.inv_h + 1e-9;
                        if (xa > 0) xa = tmax(xa, (int)fmin(floor(a), (double)xb));
                        if (xb < p.g.dims[0] - 1) xb = tmin(xb, (int)fmax(floor(b), (double)xa));
                    }
                }
                const int64_t cell = (int64_t)p.g.dims[0] * (iy + (int64_t)p.g.dims[1] * iz);
                int64_t beg = 0, end = 0;
                if (xb >= xa) {
                    beg = p.cell_start[cell + xa];
                    end = p.cell_start[cell + xb + 1];
                }
                row_beg[i] = beg;
                row_len[i] = (int32_t)(end - beg);
            }
            __syncthreads();
            if (warp == 0) {
                // exclusive prefix of the rows' chunk counts
                int32_t run = 0;
                for (int i0 = 0; i0 < nb; i0 += 32) {
                    const int i = i0 + lane;
                    const int32_t v = i < nb ? (row_len[i] >> 5) + ((row_len[i] & 31) != 0) : 0;
                    int32_t x = v;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    if (i < nb) row_mask[i] = run + x - v;
                    run += __shfl_sync(0xffffffffu, x, 31);
                }
                if (lane == 0) s_chunks = run;
            }
            __syncthreads();
            const bool keep = kFill && s_chunks <= kGaMasks;
            for (int i = warp; i < nb; i += nwarps) {
                const float4* src = p.cell_pos + row_beg[i];
                const uint32_t len = (uint32_t)row_len[i];
                int32_t n = 0;
                for (uint32_t j0 = 0; j0 < len; j0 += 128) {
                    float4 a[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t j = j0 + 32 * u + lane;
                        a[u] = j < len ? src[j] : make_float4(0.f, 0.f, 0.f, -1.f);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t j = j0 + 32 * u + lane;
                        const unsigned bal = __ballot_sync(0xffffffffu, j < len && roi_member(s, cd, a[u], p.type_mask));
                        if (keep && lane == 0 && j0 + 32 * u < len) masks[row_mask[i] + (j0 >> 5) + u] = bal;
                        n += __popc(bal);
                    }
                }
                if (lane == 0) row_cnt[i] = n;
            }
            __syncthreads();
            if (warp == 0) {
                int32_t run = 0;
                for (int i0 = 0; i0 < nb; i0 += 32) {
                    const int i = i0 + lane;
                    const int32_t v = i < nb ? row_cnt[i] : 0;
                    int32_t x = v;
                    for (int o = 1; o < 32; o <<= 1) {
                        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    if (i < nb) row_cnt[i] = run + x - v;
                    run += __shfl_sync(0xffffffffu, x, 31);
                }
                if (lane == 0) s_members = run;
            }
            __syncthreads();
            if (kFill) {
                for (int i = warp; i < nb; i += nwarps) {
                    const float4* src = p.cell_pos + row_beg[i];
                    const uint32_t len = (uint32_t)row_len[i];
                    int64_t o = count + row_cnt[i];
                    for (uint32_t j0 = 0; j0 < len; j0 += 32) {
                        const uint32_t j = j0 + lane;
                        bool in;
                        unsigned bal;
                        float4 a;
                        if (keep) {
                            bal = masks[row_mask[i] + (j0 >> 5)];
                            in = (bal >> lane) & 1u;
                            if (in) a = src[j];
                        } else {
                            a = j < len ? src[j] : make_float4(0.f, 0.f, 0.f, -1.f);
                            in = j < len && roi_member(s, cd, a, p.type_mask);
                            bal = __ballot_sync(0xffffffffu, in);
                        }
                        if (in) {
                            const int64_t k = o + __popc(bal & lt_mask);
                            if (k < slot)
                                p.atoms[base + k] = make_float4(__double2float_rn(__dsub_rn((double)a.x, cd[0])),
                                                                __double2float_rn(__dsub_rn((double)a.y, cd[1])),
                                                                __double2float_rn(__dsub_rn((double)a.z, cd[2])), 0.0f);
                            else
                                raise_status(p.status, kStatusOverflow);
                        }
                        o += __popc(bal);
                    }
                }
            }
            count += s_members;
        }
        if (tid == 0) {
            if (!kFill && count > APTIDX_MAX_ATOMS_PER_ROI) raise_status(p.status, kStatusOverflow);
            p.nw[r] = (int32_t)tmin<int64_t>(kFill ? tmin<int64_t>(count, slot) : count, 0x7FFFFFFF);
        }
    }
}

static GatherParams gather_params(Ctx* c) {
    GatherParams p;
    p.g = grid_desc(c);
    p.cell_start = c->d_cell_start;
    p.cell_pos = c->d_cell_pos;
    p.centres = c->d_centres;
    p.radii = c->d_radii;
    p.nroi = c->nroi;
    p.type_mask = c->type_mask;
    p.nw = c->d_nw;
    p.off = c->d_off;
    p.atoms = c->d_atoms;
    p.status = c->d_status;
    return p;
}

// one CTA per ROI: 512 threads while there are fewer ROIs than two per SM,
// whose walks are then the latency of the call, else 128, which keeps eight ROIs in
// flight per SM
static cudaError_t launch_gather(Ctx* c, bool fill) {
    const GatherParams p = gather_params(c);
    const int threads = c->nroi < 2 * (int64_t)c->sm_count ? 512 : 128;
    const unsigned blocks = (unsigned)tmin<int64_t>(c->nroi, (int64_t)1 << 30);
    if (fill)
        k_gather<true><<<blocks, threads, 0, c->stream>>>(p);
    else
        k_gather<false><<<blocks, threads, 0, c->stream>>>(p);
    return cudaGetLastError();
}

__global__ void k_widen(const int32_t* __restrict__ nw, int64_t n, int64_t* out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = nw[i];
}

// The slots of the gather buffer for the type mask: N_w into d_nw, their
// exclusive sum into d_off.  The slots hold the atoms of that mask and of any
// narrower one.
cudaError_t launch_gather_layout(Ctx* c) {
    cudaError_t e = launch_gather(c, false);
    if (e != cudaSuccess) return e;
    k_widen<<<(unsigned)((c->nroi + 255) / 256), 256, 0, c->stream>>>(c->d_nw, c->nroi, c->d_nw64);
    return launch_scan_i64(c->d_nw64, c->d_off, c->nroi, c->d_scan_tmp, c->stream);
}

// The centred atoms of every ROI into its slot, and N_w.  The slots were laid
// out when the ROIs were set, so a call runs this pass alone (it ran the count,
// five small kernels of the offsets and this).
cudaError_t launch_gather_fill(Ctx* c) { return launch_gather(c, true); }

// -----------------------------------------------------------------------------
// ROI order for the persistent kernels: large N_w first (longest processing
// time first).  One CTA sorts by counting on the leading bits of (float)N_w
// (seven mantissa bits: ROIs within 0.8 % of each other share a bin), and
// zeroes the work counters of the kernels that follow.  A counting sort on all
// 65536 values of N_w took four launches and 106 us in its scan, whatever the
// number of ROIs.
// -----------------------------------------------------------------------------
constexpr int kOrdThreads = 1024;
constexpr int kOrdBins = 4096;   // 32 octaves x 128

__device__ __forceinline__ int order_bin(int32_t nw) {
    // 0 for the largest: N_w < 2^31 has its exponent in [127, 158)
    return nw > 0 ? kOrdBins - 1 - (int)((__float_as_uint((float)nw) >> 16) - (127u << 7)) : kOrdBins - 1;
}

__global__ void __launch_bounds__(kOrdThreads) k_order(const int32_t* __restrict__ nw, int64_t n, int32_t* order,
                                                       int32_t* counters) {
    __shared__ int32_t h[kOrdBins];
    __shared__ int32_t ws[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = t; i < kOrdBins; i += kOrdThreads) h[i] = 0;
    if (t < 4) counters[t] = 0;
    __syncthreads();
    for (int64_t i = t; i < n; i += kOrdThreads) atomicAdd(&h[order_bin(nw[i])], 1);
    __syncthreads();
    constexpr int per = kOrdBins / kOrdThreads;
    int32_t v[per], sum = 0;
#pragma unroll
    for (int k = 0; k < per; ++k) {
        v[k] = h[t * per + k];
        sum += v[k];
    }
    int32_t x = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    int32_t ex = x - sum;
    for (int w = 0; w < warp; ++w) ex += ws[w];
#pragma unroll
    for (int k = 0; k < per; ++k) {
        h[t * per + k] = ex;
        ex += v[k];
    }
    __syncthreads();
    for (int64_t i = t; i < n; i += kOrdThreads) order[atomicAdd(&h[order_bin(nw[i])], 1)] = (int32_t)i;
}

cudaError_t launch_roi_order(Ctx* c) {
    k_order<<<1, kOrdThreads, 0, c->stream>>>(c->d_nw, c->nroi, c->d_order, c->d_counter);
    c->counters_zero = true;
    return cudaGetLastError();
}

cudaError_t zero_counters(Ctx* c) {
    if (c->counters_zero) {
        c->counters_zero = false;
        return cudaSuccess;
    }
    return cudaMemsetAsync(c->d_counter, 0, 4 * sizeof(int32_t), c->stream);
}

// -----------------------------------------------------------------------------
// twiddle table (cos, sin)(pi j / 2^m), j < 2 x 2^m, in FP32, from FP64 sincospi
// with the angle index reduced exactly in integers (half steps of the DFT's
// angle: the folded sum takes its phase from the middle of the histogram)
// -----------------------------------------------------------------------------
__global__ void k_twiddles(float2* tw, int m) {
    int nb = 1 << m;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < 2 * nb; j += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi((double)j / (double)nb, &sn, &cs);
        tw[j] = make_float2((float)cs, (float)sn);
    }
}

cudaError_t launch_twiddles(float2* tw, int m, cudaStream_t s) {
    k_twiddles<<<((2 << m) + 255) / 256, 256, 0, s>>>(tw, m);
    return cudaGetLastError();
}

// -----------------------------------------------------------------------------
// local refinement of a cubic ROI grid (Section 3.4, aluminium bicrystal): a
// ROI qualifies when its peak signature value reaches kappa times the largest
// value over all ROIs; its grid cell is split into split^3 cells with a new
// ROI at every cell centre
// -----------------------------------------------------------------------------
namespace {

__global__ void __launch_bounds__(256) k_roi_peak(const float* __restrict__ S, int64_t nroi, int32_t nv, float* peak,
                                                  unsigned* gmax_bits) {
    __shared__ float red[8];
    for (int64_t r = blockIdx.x; r < nroi; r += gridDim.x) {
        const float* row = S + r * (int64_t)nv;
        float mx = 0.f;
        for (int v = threadIdx.x; v < nv; v += 256) mx = fmaxf(mx, row[v]);
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) mx = fmaxf(mx, red[w]);
            peak[r] = mx;
            atomicMax(gmax_bits, __float_as_uint(mx));   // non-negative floats order like their bits
        }
        __syncthreads();
    }
}

__global__ void k_roi_qualify(const float* __restrict__ peak, int64_t nroi, float kappa,
                              const unsigned* __restrict__ gmax_bits, int64_t* flag) {
    const float g = __uint_as_float(*gmax_bits);
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nroi; r += (int64_t)gridDim.x * blockDim.x)
        flag[r] = (g > 0.f && peak[r] >= __fmul_rn(kappa, g)) ? 1 : 0;
}

// new ROI k = off[r] * split^3 + j, sub-cell j = ix + split (iy + split iz):
// centre = c + (i - (split - 1) / 2) * (spacing / split) per axis
__global__ void k_roi_split(const double* __restrict__ centres, const int64_t* __restrict__ flag,
                            const int64_t* __restrict__ off, int64_t nroi, double spacing, int split, double* out,
                            int32_t* parent, int64_t cap) {
    const int s3 = split * split * split;
    const double hh = __ddiv_rn(spacing, (double)split);
    const double mid = (double)(split - 1) * 0.5;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nroi * s3;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / s3;
        const int j = (int)(t % s3);
        if (!flag[r]) continue;
        const int64_t k = off[r] * s3 + j;
        if (k >= cap) continue;
        const int ix = j % split, iy = (j / split) % split, iz = j / (split * split);
        const int ii[3] = {ix, iy, iz};
        for (int d = 0; d < 3; ++d)
            out[3 * k + d] = __dadd_rn(centres[3 * r + d], __dmul_rn(__dadd_rn((double)ii[d], -mid), hh));
        if (parent) parent[k] = (int32_t)r;
    }
}

}  // namespace

cudaError_t launch_roi_refine(Ctx* c, const float* S, float kappa, double spacing, int split, double* out,
                              int32_t* parent, int64_t cap, int64_t* n_qualified) {
    const int64_t nroi = c->nroi;
    float* peak = nullptr;
    unsigned* gmax = nullptr;
    int64_t *flag = nullptr, *off = nullptr;
    cudaError_t e = cudaSuccess;
    if (dev_alloc(c, (void**)&peak, (size_t)nroi * sizeof(float)) ||
        dev_alloc(c, (void**)&gmax, sizeof(unsigned)) || dev_alloc(c, (void**)&flag, (size_t)nroi * sizeof(int64_t)) ||
        dev_alloc(c, (void**)&off, (size_t)(nroi + 1) * sizeof(int64_t)))
        e = cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = cudaMemsetAsync(gmax, 0, sizeof(unsigned), c->stream);
    if (e == cudaSuccess) {
        k_roi_peak<<<(unsigned)tmin<int64_t>(nroi, (int64_t)c->sm_count * 16), 256, 0, c->stream>>>(S, nroi, c->nv,
                                                                                                     peak, gmax);
        k_roi_qualify<<<(unsigned)tmin<int64_t>((nroi + 255) / 256, 4096), 256, 0, c->stream>>>(peak, nroi, kappa,
                                                                                                gmax, flag);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = launch_scan_i64(flag, off, nroi, c->d_scan_tmp, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(n_qualified, off + nroi, sizeof(int64_t), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess && cap > 0 && out) {
        const int64_t s3 = (int64_t)split * split * split;
        k_roi_split<<<(unsigned)tmin<int64_t>((nroi * s3 + 255) / 256, 65535), 256, 0, c->stream>>>(
            c->d_centres, flag, off, nroi, spacing, split, out, parent, cap);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    dev_free(peak);
    dev_free(gmax);
    dev_free(flag);
    dev_free(off);
    return e;
}

}  // namespace aptidx
