// common.cuh -- device helpers shared by the aptidx kernels: the binning
// contract of Eq. 1, bounded mbarrier waits, bulk (TMA) copies.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace aptidx {

template <typename T>
__host__ __device__ __forceinline__ T tmin(T a, T b) { return a < b ? a : b; }
template <typename T>
__host__ __device__ __forceinline__ T tmax(T a, T b) { return a > b ? a : b; }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// -----------------------------------------------------------------------------
// Eq. 1, the bin of a projected atom.  With dR = R / (2^(m-1) - 1) (Fig. 2
// caption) Eq. 1 is b = floor(2^(m-1) + s (2^(m-1) - 1) / R).  The library
// evaluates s in FP32 with a fixed fma order and takes the floor of the exact
// product s * scale: one fma rounding toward -inf onto the integer grid of
// [2^23, 2^24), whose bit pattern is 0x4B000000 + integer part.
// -----------------------------------------------------------------------------
__device__ __forceinline__ float project_f32(float ux, float uy, float uz, float4 a) {
    return __fmaf_rn(uz, a.z, __fmaf_rn(uy, a.y, __fmul_rn(ux, a.x)));
}

// magic = 2^23 + 2^(m-1) as float
__host__ __device__ __forceinline__ float bin_magic(int m) {
    return 8388608.0f + (float)(1 << (m - 1));
}

// exact small non-negative integer (< 2^23) to float with one integer op and
// one FP32 add (no conversion-pipe instruction)
__device__ __forceinline__ float u23_to_float(uint32_t c) {
    return __int_as_float(0x4B000000 | c) - 8388608.0f;
}

// One atom into the histograms of a 64-direction tile: lane l owns
// directions 2l (low 16 bits) and 2l + 1 (high 16 bits) of the word
// H[b * 32 + l].  The word of a lane lies in bank l for every bin b, so the
// 32 atomics of one warp instruction never share a bank.  `hbase` is the
// shared address of H plus 4 * lane.  The low m bits of the bin fma's pattern are
// the bin (for inputs the library accepts the clamp of the contract never acts:
// |u| within 1e-5 of 1 and |x| <= R give |s * scale| < 2^(m-1) - 1 + 0.01); the mask
// keeps every address in range whatever the input.
__device__ __forceinline__ void hist_add_atom(uint32_t hbase, float4 a, float4 d0, float4 d1, float scale,
                                              float magic, int nbm1) {
    const float s0 = project_f32(d0.x, d0.y, d0.z, a);
    const float s1 = project_f32(d1.x, d1.y, d1.z, a);
    const uint32_t t0 = __float_as_uint(__fmaf_rd(s0, scale, magic));
    const uint32_t t1 = __float_as_uint(__fmaf_rd(s1, scale, magic));
    const uint32_t w0 = hbase + ((t0 & (uint32_t)nbm1) << 7);
    const uint32_t w1 = hbase + ((t1 & (uint32_t)nbm1) << 7);
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(w0), "r"(1u) : "memory");
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(w1), "r"(0x10000u) : "memory");
}

// Histograms of one 64-direction tile over `cn` staged atoms; warp w takes
// atoms w, w + W, w + 2W, ...
template <int W>
__device__ __forceinline__ void hist_tile(uint32_t* H, const float4* A, int cn, int warp, int lane, float4 d0,
                                          float4 d1, float scale, float magic, int nbm1) {
    const uint32_t hbase = smem_u32(H) + 4u * (uint32_t)lane;
    int j = warp;
    if (j + 3 * W < cn) {
        // groups of four atoms, the next group's loads issued before the
        // current group's increments
        float4 a0 = A[j], a1 = A[j + W], a2 = A[j + 2 * W], a3 = A[j + 3 * W];
        for (; j + 7 * W < cn; j += 4 * W) {
            const float4 b0 = A[j + 4 * W], b1 = A[j + 5 * W], b2 = A[j + 6 * W], b3 = A[j + 7 * W];
            hist_add_atom(hbase, a0, d0, d1, scale, magic, nbm1);
            hist_add_atom(hbase, a1, d0, d1, scale, magic, nbm1);
            hist_add_atom(hbase, a2, d0, d1, scale, magic, nbm1);
            hist_add_atom(hbase, a3, d0, d1, scale, magic, nbm1);
            a0 = b0;
            a1 = b1;
            a2 = b2;
            a3 = b3;
        }
        hist_add_atom(hbase, a0, d0, d1, scale, magic, nbm1);
        hist_add_atom(hbase, a1, d0, d1, scale, magic, nbm1);
        hist_add_atom(hbase, a2, d0, d1, scale, magic, nbm1);
        hist_add_atom(hbase, a3, d0, d1, scale, magic, nbm1);
        j += 4 * W;
    }
    for (; j < cn; j += W) hist_add_atom(hbase, A[j], d0, d1, scale, magic, nbm1);
}

// Packed FP32 pairs (f32x2): each half is one IEEE FP32 operation with the
// stated rounding, so a pair gives bit for bit the two scalar results.
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma_rd(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma_ru(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float f2_lo(uint64_t x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float f2_hi(uint64_t x) { return __uint_as_float((uint32_t)(x >> 32)); }
// min(|a|, |b|, |c|), one instruction
__device__ __forceinline__ float fmin3_abs(float a, float b, float c) {
    float d;
    asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint64_t f2_dup(float v) {
    return ((uint64_t)__float_as_uint(v) << 32) | (uint64_t)__float_as_uint(v);
}

// Whether, along any direction of norm <= 1 + 1e-5, a projection s of an atom
// with |x|^2 <= r2max can make s * scale an exact nonzero integer.  With
// scale = J 2^E (J odd) and s = j 2^e (j odd), s * scale = j J 2^(e + E) is an
// integer only if e >= -E, i.e. |s| >= 2^-E.  |s| <= |u| |x| (1 + 4 2^-24)
// and r2max carries at most ~2e-7 relative rounding, so |s| stays below 2^-E
// when r2max (1 + 5e-5) < 2^-2E.  Otherwise only s = 0 gives an integer product.
__device__ __forceinline__ bool nonzero_integer_products_possible(float scale, float r2max) {
    const uint32_t bits = __float_as_uint(scale);
    const int ex = (int)((bits >> 23) & 0xFFu);
    if (ex == 0 || ex == 0xFF) return true;   // subnormal or not finite: no claim
    const uint32_t mant = (bits & 0x7FFFFFu) | 0x800000u;
    const int E = ex - 150 + (__ffs((int)mant) - 1);
    if (-2 * E >= 126) return false;
    return !(r2max * 1.00005f < ldexpf(1.0f, -2 * E));
}

// Antipodal directions: along -u the projection is exactly -s (round to
// nearest is symmetric), so the bin of -u is 2^m - 1 - b(u) whenever the exact
// product x = s * scale is not an integer, and 2^m - b(u) when it is.  With the
// product rounded down (t_rd) and up (t_ru) onto the integer grid, t_ru - t_rd is
// one unit for a non-integer x and 0 for an integer x; a lane sums it over its atoms
// (kCount == 1), so the histogram of -u is the mirror image of the histogram of u
// exactly when that sum equals the lane's atom count.

// -----------------------------------------------------------------------------
// Histogram pass of the signature kernels.  Atoms lie in 64-byte
// blocks of four (x of the four | y | z | unused), three 16-byte loads that are
// the FP32 pairs of two packed steps.  The bin fma runs at 1024 times the scale
// on the integer grid of [2^33, 2^34) (spacing 1024): its bit pattern is
// 0x50000000 + row, and shifting that left by 7 (5 for tiles of 16 directions, whose
// rows are a quarter as long) drops every exponent bit -- the grid of [2^25, 2^26),
// 0x4C000000, would keep one --, so one funnel shift with the lane's byte offset in the
// top bits of the low word gives row * 128 + 4 lane, the shared address itself when the
// magic number carries the histogram's base / 128.  That keeps the address off the
// FMA pipe, which a multiply-add of the pattern loads as much as four packed
// FMAs do per atom pair.
// -----------------------------------------------------------------------------
__device__ __forceinline__ void quad_atoms(float4* A, int n, int tid, int nthreads, unsigned* r2max = nullptr) {
    float m = 0.f;
    for (int q = tid; q < (n >> 2); q += nthreads) {
        float4* B = A + 4 * q;
        const float4 a = B[0], b = B[1], c = B[2], d = B[3];
        B[0] = make_float4(a.x, b.x, c.x, d.x);
        B[1] = make_float4(a.y, b.y, c.y, d.y);
        B[2] = make_float4(a.z, b.z, c.z, d.z);
        m = fmaxf(fmaxf(m, fmaxf(a.x * a.x + a.y * a.y + a.z * a.z, b.x * b.x + b.y * b.y + b.z * b.z)),
                  fmaxf(c.x * c.x + c.y * c.y + c.z * c.z, d.x * d.x + d.y * d.y + d.z * d.z));
    }
    if (r2max) {
        if (tid < (n & 3)) {
            const float4 a = A[(n & ~3) + tid];
            m = fmaxf(m, a.x * a.x + a.y * a.y + a.z * a.z);
        }
        atomicMax(r2max, __float_as_uint(m));
    }
}

constexpr uint32_t kQuadBits = 0x50000000u;   // bit pattern of 2^33

// 1024 (2^23 + 2^(m-1) + base row): the magic number of the pass whose histogram
// starts at shared row `row0` (its byte address / row pitch)
__device__ __forceinline__ float quad_magic(int m, uint32_t row0) {
    return 1024.0f * (8388608.0f + (float)((1 << (m - 1)) + (int)row0));
}

// Per-lane state of the pass.
struct QuadDirs {
    uint64_t x0, y0, z0, x1, y1, z1, sc, mg;
    uint32_t lane_top;   // the lane's byte offset in its row, in the top bits
    uint32_t t_lo;       // chunked: bit pattern of the chunk's first bin
    uint32_t h_lane;     // chunked: H + 4 lane
};

// word: the lane's word of the row; rows of 32 >> split words
__device__ __forceinline__ QuadDirs quad_dirs(float4 d0, float4 d1, float scale, float magic, int word, int split = 0) {
    QuadDirs q;
    q.x0 = f2_dup(d0.x);
    q.y0 = f2_dup(d0.y);
    q.z0 = f2_dup(d0.z);
    q.x1 = f2_dup(d1.x);
    q.y1 = f2_dup(d1.y);
    q.z1 = f2_dup(d1.z);
    q.sc = f2_dup(1024.0f * scale);
    q.mg = f2_dup(magic);
    q.lane_top = (uint32_t)word << (27 + split);
    q.t_lo = q.h_lane = 0;
    return q;
}

template <bool kChunked, int kSplit = 0>
__device__ __forceinline__ void quad_inc(uint32_t t, uint32_t one, const QuadDirs& q) {
    if (kChunked) {
        const uint32_t v = t - q.t_lo;   // bin - first bin of the chunk
        if (v < 1024u) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(v * 128u + q.h_lane), "r"(one) : "memory");
    } else {
        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(__funnelshift_l(q.lane_top, t, 7 - kSplit)), "r"(one) : "memory");
    }
}

// kCount == 1: c0, c1 accumulate the lane's non-integer counts of its two
// directions.  kCount == 2 (only s = 0 can give an integer product): the smallest
// |s s'| of the lane's two directions, 0 when some projection is exactly zero (or a
// product underflows, which would only cost the tile a second pass).
template <int kCount, bool kChunked, int kSplit = 0>
__device__ __forceinline__ void quad_add_pair(uint64_t x, uint64_t y, uint64_t z, const QuadDirs& q, uint32_t& c0,
                                              uint32_t& c1, float& zmin) {
    const uint64_t s0 = f2_fma(z, q.z0, f2_fma(y, q.y0, f2_mul(x, q.x0)));
    const uint64_t s1 = f2_fma(z, q.z1, f2_fma(y, q.y1, f2_mul(x, q.x1)));
    const uint64_t t0 = f2_fma_rd(s0, q.sc, q.mg);
    const uint64_t t1 = f2_fma_rd(s1, q.sc, q.mg);
    if (kCount == 2) {
        const uint64_t pr = f2_mul(s0, s1);
        zmin = fmin3_abs(zmin, f2_lo(pr), f2_hi(pr));
    } else if (kCount == 1) {
        const uint64_t u0 = f2_fma_ru(s0, q.sc, q.mg);
        const uint64_t u1 = f2_fma_ru(s1, q.sc, q.mg);
        c0 += ((uint32_t)u0 - (uint32_t)t0) + ((uint32_t)(u0 >> 32) - (uint32_t)(t0 >> 32));
        c1 += ((uint32_t)u1 - (uint32_t)t1) + ((uint32_t)(u1 >> 32) - (uint32_t)(t1 >> 32));
    }
    quad_inc<kChunked, kSplit>((uint32_t)t0, 1u, q);
    quad_inc<kChunked, kSplit>((uint32_t)(t0 >> 32), 1u, q);
    quad_inc<kChunked, kSplit>((uint32_t)t1, 0x10000u, q);
    quad_inc<kChunked, kSplit>((uint32_t)(t1 >> 32), 0x10000u, q);
}

// Histograms of one tile over `cn` atoms staged by quad_atoms; group g of G
// (warps, or the parts of a warp that hold a whole row of words each) takes
// blocks g, g + G, ..., two at a time with their loads first; the up to three
// trailing atoms go to group (cn / 4) % G.  Returns the number of atoms this
// group handled.
template <int kCount, bool kChunked, int kSplit = 0>
__device__ __forceinline__ int hist_tile_quads(const float4* A, int cn, int warp, int W, const QuadDirs& q, uint32_t& c0,
                                               uint32_t& c1, float& zmin) {
    const int nq = cn >> 2;
    auto ld = [&](int i, int k) { return *reinterpret_cast<const ulonglong2*>(A + 4 * i + k); };
    int j = warp;
    for (; j + W < nq; j += 2 * W) {
        const ulonglong2 xa = ld(j, 0), ya = ld(j, 1), za = ld(j, 2);
        const ulonglong2 xb = ld(j + W, 0), yb = ld(j + W, 1), zb = ld(j + W, 2);
        quad_add_pair<kCount, kChunked, kSplit>(xa.x, ya.x, za.x, q, c0, c1, zmin);
        quad_add_pair<kCount, kChunked, kSplit>(xa.y, ya.y, za.y, q, c0, c1, zmin);
        quad_add_pair<kCount, kChunked, kSplit>(xb.x, yb.x, zb.x, q, c0, c1, zmin);
        quad_add_pair<kCount, kChunked, kSplit>(xb.y, yb.y, zb.y, q, c0, c1, zmin);
    }
    if (j < nq) {
        const ulonglong2 xa = ld(j, 0), ya = ld(j, 1), za = ld(j, 2);
        quad_add_pair<kCount, kChunked, kSplit>(xa.x, ya.x, za.x, q, c0, c1, zmin);
        quad_add_pair<kCount, kChunked, kSplit>(xa.y, ya.y, za.y, q, c0, c1, zmin);
    }
    int handled = warp < nq ? 4 * ((nq - warp + W - 1) / W) : 0;
    if (warp == nq % W) {
        for (int i = nq * 4; i < cn; ++i) {
            const float4 a = A[i];
            const float sc = f2_lo(q.sc), mg = f2_lo(q.mg);
            const float s0 = project_f32(f2_lo(q.x0), f2_lo(q.y0), f2_lo(q.z0), a);
            const float s1 = project_f32(f2_lo(q.x1), f2_lo(q.y1), f2_lo(q.z1), a);
            const uint32_t t0 = __float_as_uint(__fmaf_rd(s0, sc, mg));
            const uint32_t t1 = __float_as_uint(__fmaf_rd(s1, sc, mg));
            if (kCount == 2) {
                zmin = fminf(zmin, fminf(fabsf(s0), fabsf(s1)));
            } else if (kCount == 1) {
                c0 += __float_as_uint(__fmaf_ru(s0, sc, mg)) - t0;
                c1 += __float_as_uint(__fmaf_ru(s1, sc, mg)) - t1;
            }
            quad_inc<kChunked, kSplit>(t0, 1u, q);
            quad_inc<kChunked, kSplit>(t1, 0x10000u, q);
            ++handled;
        }
    }
    return handled;
}

// Band maxima of one direction: frequency f with amplitude a updates every
// band holding f (strictly greater, so with f ascending ties keep the lowest
// f).  bs.n == 0: the single band [klo, khi] of the ROI.
__device__ __forceinline__ int band_count(const BandSet& bs) { return bs.n == 0 ? 1 : bs.n; }

__device__ __forceinline__ void band_init(const BandSet& bs, int klo, float* best, int* bk) {
#pragma unroll
    for (int b = 0; b < APTIDX_MAX_BANDS; ++b) {
        best[b] = -1.f;
        bk[b] = bs.n == 0 ? klo : bs.lo[b];
    }
}

__device__ __forceinline__ void band_update(const BandSet& bs, int klo, int khi, int f, float a, float* best,
                                            int* bk) {
    const int nb = band_count(bs);
#pragma unroll
    for (int b = 0; b < APTIDX_MAX_BANDS; ++b) {
        const int lo = bs.n == 0 ? klo : bs.lo[b], hi = bs.n == 0 ? khi : bs.hi[b];
        if (b < nb && f >= lo && f <= hi && a > best[b]) {
            best[b] = a;
            bk[b] = f;
        }
    }
}

// The same with the slot count fixed at compile time: kNB == 1 is the
// single-band kernel (the ROI's band [klo, khi]; the BandSet is not read).
template <int kNB>
__device__ __forceinline__ void band_init_t(const BandSet& bs, int klo, float* best, int* bk) {
    if (kNB == 1) {
        best[0] = -1.f;
        bk[0] = klo;
    } else {
        band_init(bs, klo, best, bk);
    }
}

template <int kNB>
__device__ __forceinline__ void band_update_t(const BandSet& bs, int klo, int khi, int f, float a, float* best,
                                              int* bk) {
    if (kNB == 1) {
        if (f >= klo && f <= khi && a > best[0]) {
            best[0] = a;
            bk[0] = f;
        }
    } else {
        band_update(bs, klo, khi, f, a, best, bk);
    }
}

template <int kNB>
__device__ __forceinline__ int band_count_t(const BandSet& bs) { return kNB == 1 ? 1 : band_count(bs); }

template <int kNB>
__device__ __forceinline__ int64_t band_off_t(const BandSet& bs, int b) { return kNB == 1 ? 0 : bs.off[b]; }

constexpr int kTcMaxAtoms = 2048;  // fp16 carries every count <= 2048 exactly

// -----------------------------------------------------------------------------
// status word
// -----------------------------------------------------------------------------
__device__ __forceinline__ void raise_status(int* status, int bit) {
    atomicOr(status, bit);
}

// -----------------------------------------------------------------------------
// shared-memory addresses, mbarriers and bulk copies (inline PTX)
// -----------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of an mbarrier, at most `limit` polls.  Returns
// false (and raises the timeout status bit) if the phase never completed.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, int* status,
                                                  uint32_t limit = (1u << 22)) {
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    raise_status(status, kStatusTimeout);
    return false;
}

// 1-D bulk copy global -> shared (TMA engine), completion counted in bytes on
// `bar`.  dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 16-byte asynchronous copy global -> shared (no L1 allocation); completion
// by cp_async_wait_all of the issuing thread.  Both addresses 16-byte aligned.
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Stage `n` float4 atoms from global into shared memory with one bulk copy
// issued by thread 0, then make them visible to the whole CTA.  `phase` is
// the barrier's parity bit, toggled per use.  Returns false on a timeout
// (every thread of the CTA returns the same value).
__device__ __forceinline__ bool stage_atoms(float4* dst, const float4* src, int n, uint64_t* bar,
                                            uint32_t& phase, int* status, int* flag_smem) {
    if (threadIdx.x == 0) {
        int ok = 1;
        if (n > 0) {
            fence_proxy_async_smem();   // earlier generic reads of dst before the async write
            mbar_arrive_expect_tx(bar, (uint32_t)n * 16u);
            bulk_g2s(dst, src, (uint32_t)n * 16u, bar);
            ok = mbar_wait_bounded(bar, phase, status) ? 1 : 0;
            if (!ok) mbar_wait_bounded(bar, phase, status, 1u << 20);   // let an in-flight copy land
            phase ^= 1u;
        }
        *flag_smem = ok;
    }
    __syncthreads();
    int ok = *flag_smem;
    if (threadIdx.x != 0 && n > 0) phase ^= 1u;
    __syncthreads();   // flag_smem is rewritten by the next call
    return ok != 0;
}

}  // namespace aptidx
