// signature_plain.cu -- steps (a2)-(a5) on CUDA cores, FP32: projection (Eq. 1
// dot product), binning into 2^m-bin histograms, the band of the DFT
// amplitude spectrum (Section 2.2), and the per-direction band maximum (the
// signature value, supplement "Al bicrystal").
//
// Work item = (ROI, group of 64-direction tiles).  A persistent grid claims
// items from a global counter, ROIs in longest-first order.  Per item the
// ROI's centred atoms are copied into shared memory once (bulk copy on the
// TMA engine).  Per tile every warp walks a strided subset of the atoms; lane
// l owns directions 2l and 2l+1 and adds 1 to 16-bit halves of the word
// H[b * 32 + l].  A lane's words sit in bank l whatever the bin, so the
// shared-memory atomics of one warp instruction never conflict.
//
// The band spectrum takes the phase from the middle of the histogram: with
// bins n and N - 1 - n folded into their sum e and difference o,
//   |X(k)|^2 = (sum_n e_n cos t_n)^2 + (sum_n o_n sin t_n)^2,
// t_n = 2 pi k (j + 1/2) / N at the j-th bin from the middle, and the bins j
// and N / 2 - 1 - j share one cosine and sine up to the sign (-1)^k.  The folds
// are exact (small integers), so four bins cost two FMAs per frequency (a
// complex sum over all bins costs eight), and the value of the mirrored
// histogram, that of the direction -u, is the same bit for bit.  Antipodal
// pairs are therefore projected once (as on the tensor-core path, with the same
// exact check for atoms whose mirror image falls into another bin).
// 512 ROIs of 1133 atoms x 40962 directions, 2^10 bins, four frequencies:
// 24.9 ms with every direction projected and the complex sum, 8.6 ms now.
#include <mutex>

#include "common.cuh"

namespace aptidx {

namespace {

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kDirs = kTileDirs;        // 64 directions per tile
constexpr int kWords = kDirs / 2;       // u32 words per bin
constexpr int kKpw = 4;                 // frequencies per warp unit
constexpr int kPartBytes = kWarps * kKpw * kDirs * 8;
constexpr int kChunkBins = 1024;        // bins per histogram chunk (128 KB of words)
constexpr int kBlockAtoms = 65535;      // atoms per block: every 16-bit count of a block is exact

// Histograms of one tile for bin chunk bc over `cn` staged atoms (the
// multi-pass path: 2^m > 1024 bins, or a ROI above kBlockAtoms atoms): the bin
// is masked to m bits and only bins of [1024 bc, 1024 bc + 1024) are added,
// at row b - 1024 bc.
template <int W>
__device__ __forceinline__ void hist_tile_chunk(uint32_t* H, const float4* A, int cn, int warp, int lane, float4 d0,
                                                float4 d1, float scale, float magic, uint32_t nbm1, uint32_t bc) {
    const uint32_t hb = smem_u32(H) + 4u * (uint32_t)lane;
    for (int j = warp; j < cn; j += W) {
        const float4 a = A[j];
        const uint32_t b0 = __float_as_uint(__fmaf_rd(project_f32(d0.x, d0.y, d0.z, a), scale, magic)) & nbm1;
        const uint32_t b1 = __float_as_uint(__fmaf_rd(project_f32(d1.x, d1.y, d1.z, a), scale, magic)) & nbm1;
        if ((b0 >> 10) == bc)
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(hb + ((b0 & 1023u) << 7)), "r"(1u) : "memory");
        if ((b1 >> 10) == bc)
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(hb + ((b1 & 1023u) << 7)), "r"(0x10000u) : "memory");
    }
}

// Debug export of one pass: adds the counts of rows [0, nbc) to
// h_out[v * 2^m + bc * nbc + row] (the caller zeroes h_out).
__device__ __forceinline__ void hist_export_add_p(const uint32_t* H, int nbc, int NB, int bc, int tile, int nv,
                                                  uint16_t* h_out, int tid, int nthreads) {
    for (int i = tid; i < nbc * 32; i += nthreads) {
        const int b = i >> 5, l = i & 31;
        const uint32_t w = H[i];
        const int64_t v0 = (int64_t)tile * 64 + 2 * l;
        const int64_t col = (int64_t)bc * nbc + b;
        if (v0 < nv) h_out[v0 * NB + col] = (uint16_t)(h_out[v0 * NB + col] + (w & 0xFFFFu));
        if (v0 + 1 < nv) h_out[(v0 + 1) * NB + col] = (uint16_t)(h_out[(v0 + 1) * NB + col] + (w >> 16));
    }
}

struct SigParams {
    const float4* atoms;
    const int64_t* off;
    const int32_t* nw;
    const int32_t* order;
    const float4* dirs;      // direction slots, padded to whole tiles with (1, 0, 0)
    const int2* slot_idx;    // per slot: (output direction, antipodal partner or -1); NULL: slot = direction
    int32_t nv;
    int32_t tiles_per_roi;
    int32_t tiles_per_item;
    int32_t items_per_roi;
    int64_t n_items;
    const float* scale;
    const int32_t* band;
    int m;
    const float2* tw;
    float* S;
    uint16_t* argk;
    uint16_t* hist_out;
    int64_t single_roi;
    int32_t* counter;
    int* status;
    int atom_cap;
    int64_t nroi;
    BandSet bands;
};

// Folded partial spectrum of kKpw frequencies from k0 over the bins j0 .. j0 +
// span - 1 from the middle (and their three images), for the lane's two
// directions: re = sum e cos, im = sum o sin.  TW2[i] = (cos, sin)(pi i / N),
// i < 2 N; kOdd = k0 & 1.  Bound by issue; kUnroll bins a step: 8 where the bins are
// split among warps (512 ROIs x 40962 directions, four frequencies: 8.65 ms by 2, 8.44),
// 3 where a warp walks them all (100 ROIs x 10242, k = 8..100: 4.65, 4.41).
template <int kOdd, int kUnroll>
__device__ __forceinline__ void fold_dft(const uint32_t* H, const float2* TW2, int NB, int lane, int j0, int span,
                                         int k0, float (&re)[kKpw][2], float (&im)[kKpw][2]) {
    const unsigned mask = 2u * (unsigned)NB - 1u;
    unsigned idx[kKpw];
#pragma unroll
    for (int q = 0; q < kKpw; ++q) idx[q] = ((unsigned)(k0 + q) * (2u * (unsigned)j0 + 1u)) & mask;
    const uint32_t* ha = H + (NB / 2 - 1 - j0) * kWords + lane;   // a: below the middle, descending
    const uint32_t* hb = H + (NB / 2 + j0) * kWords + lane;       // b: above the middle
    const uint32_t* hc = H + j0 * kWords + lane;                  // c: from the first bin
    const uint32_t* hd = H + (NB - 1 - j0) * kWords + lane;       // d: from the last bin
#pragma unroll kUnroll
    for (int j = 0; j < span; ++j) {
        const uint32_t wa = *ha, wc = *hc;
        const uint32_t s1 = wa + *hb, s2 = wc + *hd;   // 16-bit halves: no carry, a histogram holds at most 65535 atoms
        ha -= kWords;
        hb += kWords;
        hc += kWords;
        hd -= kWords;
        float ee[2], eo[2], oe[2], oo[2];   // e and o of even and odd frequencies
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            const float f1 = u23_to_float(d ? s1 >> 16 : s1 & 0xFFFFu), f2 = u23_to_float(d ? s2 >> 16 : s2 & 0xFFFFu);
            const float fa = u23_to_float(d ? wa >> 16 : wa & 0xFFFFu), fc = u23_to_float(d ? wc >> 16 : wc & 0xFFFFu);
            const float p = fmaf(2.f, fa, -f1), r = fmaf(2.f, fc, -f2);   // a - b, c - d
            ee[d] = f1 + f2;
            eo[d] = f1 - f2;
            oe[d] = p - r;
            oo[d] = p + r;
        }
#pragma unroll
        for (int q = 0; q < kKpw; ++q) {
            const float2 t = TW2[idx[q]];
            idx[q] = (idx[q] + 2u * (unsigned)(k0 + q)) & mask;
            const bool odd = ((q + kOdd) & 1) != 0;
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                re[q][d] = fmaf(odd ? eo[d] : ee[d], t.x, re[q][d]);
                im[q][d] = fmaf(odd ? oo[d] : oe[d], t.y, im[q][d]);
            }
        }
    }
}

// kNB: band slots of the epilogue (1: the ROI's own band; APTIDX_MAX_BANDS:
// the pass's BandSet).  kSafe: atoms and directions come from the caller
// unchecked, so bins are masked to m bits (memory-safe for any input).  kMode: which
// ROIs of a launch take the passes over bin chunks and atom blocks (all above 2^10
// bins, those above kBlockAtoms atoms, none); registers are short, and each loop is
// faster in an instance without the other (by 2 to 5 %).
enum { kSinglePass, kMixed, kAllPasses };

template <int kNB, bool kSafe, int kMode>
__global__ void __launch_bounds__(kThreads, 1) k_sig_plain(SigParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int NB = 1 << p.m;
    const int nbm1 = NB - 1;
    const int NBc = NB < kChunkBins ? NB : kChunkBins;   // histogram rows held at once
    const int nchunk = kMode == kSinglePass ? 1 : NB / NBc;
    const int ntw = nchunk == 1 ? 2 * NB : NB;   // half-step angles for the folded sum
    uint32_t* H = reinterpret_cast<uint32_t*>(smem);
    float2* TW = reinterpret_cast<float2*>(smem + (size_t)NBc * kWords * 4);
    float4* A = reinterpret_cast<float4*>(smem + (size_t)NBc * kWords * 4 + (size_t)ntw * 8);
    float2* PART = reinterpret_cast<float2*>(A + p.atom_cap);
    uint64_t* bar = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(PART) + kPartBytes);
    int* flag = reinterpret_cast<int*>(bar + 1);
    int64_t* item_s = reinterpret_cast<int64_t*>(bar + 2);
    unsigned* r2max_s = reinterpret_cast<unsigned*>(bar + 3);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int j = tid; j < ntw; j += kThreads) TW[j] = p.tw[nchunk == 1 ? j : 2 * j];
    auto zero_h = [&](int t0) {   // threads t0 .. kThreads - 1
        for (int i = tid - t0; i < NBc * kWords / 4; i += kThreads - t0)
            reinterpret_cast<uint4*>(H)[i] = make_uint4(0, 0, 0, 0);
    };
    zero_h(0);   // every pass finds the histogram zero
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_barrier_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    const uint32_t h_addr = smem_u32(H);
    const float magic = kSafe ? bin_magic(p.m) : quad_magic(p.m, h_addr >> 7);
    const bool sym = !kSafe && p.slot_idx != nullptr;
    const int64_t n_items = p.n_items;

    for (;;) {
        if (tid == 0) *item_s = atomicAdd(p.counter, 1);
        __syncthreads();
        const int64_t item = *item_s;
        __syncthreads();
        if (item >= n_items) break;
        const int64_t roi_rank = item / p.items_per_roi;
        const int grp = (int)(item % p.items_per_roi);
        const int64_t roi = p.single_roi >= 0 ? p.single_roi : (int64_t)p.order[roi_rank];
        const int nw = p.nw[roi];
        const int64_t abase = p.off[roi];
        const float scale = p.scale[roi];
        const int klo = p.band[2 * roi], khi = p.band[2 * roi + 1];
        const int K = khi - klo + 1;
        const int G = (K + kKpw - 1) / kKpw;   // frequency groups of kKpw
        const int t0 = grp * p.tiles_per_item;
        const int t1 = min(t0 + p.tiles_per_item, p.tiles_per_roi);
        const bool one_chunk = nw <= p.atom_cap;
        const int64_t out_base = (p.single_roi >= 0 ? 0 : roi) * (int64_t)p.nv;
        // stage n atoms, in blocks of four unless the checked loops read them
        auto stage = [&](const float4* src, int n, unsigned* r2) -> bool {
            if (r2 && tid == 0) *r2 = 0u;
            if (!stage_atoms(A, src, n, bar, phase, p.status, flag)) return false;
            if (!kSafe) {
                quad_atoms(A, n, tid, kThreads, r2);
                __syncthreads();
            }
            return true;
        };
        if (one_chunk && !stage(p.atoms + abase, nw, r2max_s)) return;
        const bool zero_check =
            sym && one_chunk && !nonzero_integer_products_possible(scale, __uint_as_float(*r2max_s));
        // one pass of the histogram over bn atoms from a0 (bin chunk bc); the
        // counts of the antipodal check go to c0, c1, zmin, handled
        QuadDirs q;
        float4 d0, d1;
        uint32_t c0 = 0, c1 = 0;
        float zmin = 1.f;
        int handled = 0;
        auto histogram = [&](const float4* src, int bn, int bc, bool count) -> bool {
            for (int s0 = 0; s0 < bn || s0 == 0; s0 += p.atom_cap) {
                const int cn = min(p.atom_cap, bn - s0);
                if (!one_chunk && !stage(src + s0, cn, nullptr)) return false;
                if (kSafe) {
                    if (nchunk == 1)
                        hist_tile<kWarps>(H, A, cn, warp, lane, d0, d1, scale, magic, nbm1);
                    else
                        hist_tile_chunk<kWarps>(H, A, cn, warp, lane, d0, d1, scale, magic, (uint32_t)nbm1, (uint32_t)bc);
                } else if (nchunk == 1) {
                    if (count && zero_check)
                        handled += hist_tile_quads<2, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                    else if (count)
                        handled += hist_tile_quads<1, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                    else
                        hist_tile_quads<0, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                } else {
                    q.t_lo = kQuadBits + (h_addr >> 7) + (uint32_t)bc * kChunkBins;
                    q.h_lane = h_addr + 4u * (uint32_t)lane;
                    hist_tile_quads<0, true>(A, cn, warp, kWarps, q, c0, c1, zmin);
                }
                if (!one_chunk) __syncthreads();
            }
            return true;
        };
        // where direction `at` of the tile goes: pass 0 the slot's direction (and
        // its partner when `mirror`), pass 1 the partner
        auto write_out = [&](int tile, int at, int pass, bool mirror, int b, float value, int k) {
            const int slot = tile * kDirs + at;
            int v0 = slot < p.nv ? slot : -1, v1 = -1;
            if (sym) {
                const int2 si = p.slot_idx[slot];
                v0 = pass ? si.y : si.x;
                v1 = mirror ? si.y : -1;
            }
            const int64_t ob = band_off_t<kNB>(p.bands, b) + out_base;
            if (v0 >= 0) {
                p.S[ob + v0] = value;
                if (p.argk) p.argk[ob + v0] = (uint16_t)k;
            }
            if (v1 >= 0) {
                p.S[ob + v1] = value;
                if (p.argk) p.argk[ob + v1] = (uint16_t)k;
            }
        };

        const bool multi_pass = kMode == kAllPasses || (kMode == kMixed && (nchunk > 1 || nw > kBlockAtoms));
        for (int tile = t0; tile < t1; ++tile) {
            bool partners = sym && multi_pass;   // a partner pass is due
            for (int pass = 0; pass < 2; ++pass) {
                if (pass == 1 && !partners) break;
                d0 = p.dirs[(int64_t)tile * kDirs + 2 * lane];
                d1 = p.dirs[(int64_t)tile * kDirs + 2 * lane + 1];
                const bool pt0 = d0.w != 0.f, pt1 = d1.w != 0.f;
                if (pass == 1) {
                    d0 = make_float4(-d0.x, -d0.y, -d0.z, d0.w);
                    d1 = make_float4(-d1.x, -d1.y, -d1.z, d1.w);
                }
                if (!kSafe) q = quad_dirs(d0, d1, scale, magic, lane);
                if (multi_pass) {
                    // ---- multi-pass path: the histogram of a tile in passes over atom
                    // blocks of at most kBlockAtoms and bin chunks of 1024; each warp
                    // unit (4 frequencies x a span of the chunk's bins) accumulates its
                    // partial DFT in registers across the passes.  Bands of more than
                    // kWarps groups of frequencies run in rounds of kWarps groups.
                    const int nblk = (nw + kBlockAtoms - 1) / kBlockAtoms;
                    // full-step angles: with half steps in the table the index runs in
                    // twos.  Bound by issue: the index scaled at every look-up and no
                    // unrolling cost 10 % each (60 ROIs, 10242 directions, 2^12 bins,
                    // k = 8..60: 34.8 ms, now 26.5)
                    const unsigned tws = nchunk == 1 ? 2u : 1u, tmask = tws * (unsigned)NB - 1u;
                    float best[kNB];
                    int bk[kNB];
                    if (tid < kDirs) band_init_t<kNB>(p.bands, klo, best, bk);
                    for (int g_lo = 0; g_lo < G; g_lo += kWarps) {
                        const int Gr = min(kWarps, G - g_lo);
                        int nsplit = 1;
                        while (Gr * nsplit * 2 <= kWarps && nsplit * 2 <= NBc / 32) nsplit *= 2;
                        const int span = NBc / nsplit;
                        const bool unit = warp < Gr * nsplit;
                        const int g = g_lo + warp / nsplit, sp = warp % nsplit;
                        const int k0 = klo + g * kKpw;
                        float re[kKpw][2], im[kKpw][2];
#pragma unroll
                        for (int i = 0; i < kKpw; ++i) re[i][0] = re[i][1] = im[i][0] = im[i][1] = 0.f;
                        for (int blk = 0; blk < max(nblk, 1); ++blk) {
                            const int b0 = blk * kBlockAtoms, bn = max(0, min(kBlockAtoms, nw - b0));
                            for (int bc = 0; bc < nchunk; ++bc) {
                                if (!histogram(p.atoms + abase + b0, bn, bc, false)) return;
                                __syncthreads();
                                if (p.hist_out && g_lo == 0) {
                                    hist_export_add_p(H, NBc, NB, bc, tile, p.nv, p.hist_out, tid, kThreads);
                                    __syncthreads();
                                }
                                if (unit) {
                                    const int n0 = bc * NBc + sp * span;
                                    unsigned idx[kKpw], step[kKpw];
#pragma unroll
                                    for (int i = 0; i < kKpw; ++i) {
                                        step[i] = tws * (unsigned)(k0 + i);
                                        idx[i] = step[i] * (unsigned)n0 & tmask;
                                    }
                                    const uint32_t* hp = H + sp * span * kWords + lane;
#pragma unroll 4
                                    for (int n = 0; n < span; ++n) {
                                        const uint32_t w = hp[n * kWords];
                                        const float f0 = u23_to_float(w & 0xFFFFu), f1 = u23_to_float(w >> 16);
#pragma unroll
                                        for (int i = 0; i < kKpw; ++i) {
                                            const float2 t = TW[idx[i]];
                                            re[i][0] = fmaf(f0, t.x, re[i][0]);
                                            im[i][0] = fmaf(f0, t.y, im[i][0]);
                                            re[i][1] = fmaf(f1, t.x, re[i][1]);
                                            im[i][1] = fmaf(f1, t.y, im[i][1]);
                                            idx[i] = (idx[i] + step[i]) & tmask;
                                        }
                                    }
                                }
                                __syncthreads();   // H has been read
                                zero_h(0);
                                __syncthreads();
                            }
                        }
                        if (unit) {
#pragma unroll
                            for (int i = 0; i < kKpw; ++i) {
                                PART[((size_t)warp * kKpw + i) * kDirs + 2 * lane] = make_float2(re[i][0], im[i][0]);
                                PART[((size_t)warp * kKpw + i) * kDirs + 2 * lane + 1] = make_float2(re[i][1], im[i][1]);
                            }
                        }
                        __syncthreads();
                        if (tid < kDirs) {
                            for (int kk = g_lo * kKpw; kk < min(K, (g_lo + Gr) * kKpw); ++kk) {
                                const int gg = kk / kKpw - g_lo, i = kk % kKpw;
                                float sr = 0.f, si = 0.f;
                                for (int s2 = 0; s2 < nsplit; ++s2) {
                                    const float2 t = PART[((size_t)(gg * nsplit + s2) * kKpw + i) * kDirs + tid];
                                    sr += t.x;
                                    si += t.y;
                                }
                                band_update_t<kNB>(p.bands, klo, khi, klo + kk, sqrtf(sr * sr + si * si), best, bk);
                            }
                        }
                        __syncthreads();
                    }
                    if (tid < kDirs)
#pragma unroll
                        for (int b = 0; b < kNB; ++b)
                            if (b < band_count_t<kNB>(p.bands)) write_out(tile, tid, pass, false, b, best[b], bk[b]);
                    continue;
                }

                const bool count = sym && pass == 0;
                c0 = c1 = 0;
                zmin = 1.f;
                handled = 0;
                if (!histogram(p.atoms + abase, nw, 0, count)) return;
                const int bad = count && (zero_check ? (pt0 || pt1) && zmin == 0.f
                                                     : (pt0 && c0 != (uint32_t)handled) || (pt1 && c1 != (uint32_t)handled));
                const bool any_bad = __syncthreads_or(bad) != 0;
                if (pass == 0) partners = any_bad;
                const bool mirror = count && !any_bad;

                if (p.hist_out) hist_export_add_p(H, NB, NB, 0, tile, p.nv, p.hist_out, tid, kThreads);

                // ---- band spectrum (FP32) and band maximum ----
                if (G <= kWarps) {
                    int nsplit = 1;
                    while (G * nsplit * 2 <= kWarps && nsplit * 2 <= NB / 32) nsplit *= 2;
                    const int span = NB / 4 / nsplit;
                    if (warp < G * nsplit) {
                        const int g = warp / nsplit, sp = warp % nsplit;
                        const int k0 = klo + g * kKpw;
                        float re[kKpw][2], im[kKpw][2];
#pragma unroll
                        for (int i = 0; i < kKpw; ++i) re[i][0] = re[i][1] = im[i][0] = im[i][1] = 0.f;
                        if (k0 & 1)
                            fold_dft<1, 8>(H, TW, NB, lane, sp * span, span, k0, re, im);
                        else
                            fold_dft<0, 8>(H, TW, NB, lane, sp * span, span, k0, re, im);
#pragma unroll
                        for (int i = 0; i < kKpw; ++i) {
                            PART[((size_t)warp * kKpw + i) * kDirs + 2 * lane] = make_float2(re[i][0], im[i][0]);
                            PART[((size_t)warp * kKpw + i) * kDirs + 2 * lane + 1] = make_float2(re[i][1], im[i][1]);
                        }
                    }
                    __syncthreads();
                    if (tid < kDirs) {
                        float best[kNB];
                        int bk[kNB];
                        band_init_t<kNB>(p.bands, klo, best, bk);
                        for (int kk = 0; kk < K; ++kk) {
                            const int g = kk / kKpw, i = kk % kKpw;
                            float sr = 0.f, si = 0.f;
                            for (int sp = 0; sp < nsplit; ++sp) {
                                const float2 t = PART[((size_t)(g * nsplit + sp) * kKpw + i) * kDirs + tid];
                                sr += t.x;
                                si += t.y;
                            }
                            band_update_t<kNB>(p.bands, klo, khi, klo + kk, sqrtf(sr * sr + si * si), best, bk);
                        }
#pragma unroll
                        for (int b = 0; b < kNB; ++b)
                            if (b < band_count_t<kNB>(p.bands)) write_out(tile, tid, pass, mirror, b, best[b], bk[b]);
                    } else {
                        zero_h(kDirs);
                    }
                } else {
                    float b0[kNB], b1[kNB];
                    int bk0[kNB], bk1[kNB];
                    band_init_t<kNB>(p.bands, klo, b0, bk0);
                    band_init_t<kNB>(p.bands, klo, b1, bk1);
                    for (int g = warp; g < G; g += kWarps) {
                        const int k0 = klo + g * kKpw;
                        float re[kKpw][2], im[kKpw][2];
#pragma unroll
                        for (int i = 0; i < kKpw; ++i) re[i][0] = re[i][1] = im[i][0] = im[i][1] = 0.f;
                        if (k0 & 1)
                            fold_dft<1, 3>(H, TW, NB, lane, 0, NB / 4, k0, re, im);
                        else
                            fold_dft<0, 3>(H, TW, NB, lane, 0, NB / 4, k0, re, im);
#pragma unroll
                        for (int i = 0; i < kKpw; ++i) {
                            if (k0 + i > khi) break;
                            const float a0 = sqrtf(re[i][0] * re[i][0] + im[i][0] * im[i][0]);
                            const float a1 = sqrtf(re[i][1] * re[i][1] + im[i][1] * im[i][1]);
                            band_update_t<kNB>(p.bands, klo, khi, k0 + i, a0, b0, bk0);
                            band_update_t<kNB>(p.bands, klo, khi, k0 + i, a1, b1, bk1);
                        }
                    }
                    // per band, each warp's best over its frequency groups; the
                    // band's slab of PART holds kWarps x kDirs (value, k) pairs
#pragma unroll
                    for (int b = 0; b < kNB; ++b) {
                        if (b < band_count_t<kNB>(p.bands)) {
                            PART[((size_t)b * kWarps + warp) * kDirs + 2 * lane] = make_float2(b0[b], __int_as_float(bk0[b]));
                            PART[((size_t)b * kWarps + warp) * kDirs + 2 * lane + 1] =
                                make_float2(b1[b], __int_as_float(bk1[b]));
                        }
                    }
                    __syncthreads();
                    if (tid < kDirs) {
                        for (int b = 0; b < band_count_t<kNB>(p.bands); ++b) {
                            float best = -1.f;
                            int bk = kNB == 1 ? klo : p.bands.lo[b];
                            for (int w = 0; w < kWarps; ++w) {
                                const float2 t = PART[((size_t)b * kWarps + w) * kDirs + tid];
                                const int k = __float_as_int(t.y);
                                if (t.x > best || (t.x == best && k < bk)) {
                                    best = t.x;
                                    bk = k;
                                }
                            }
                            write_out(tile, tid, pass, mirror, b, best, bk);
                        }
                    } else {
                        zero_h(kDirs);
                    }
                }
                __syncthreads();
            }
        }
    }
}

// per-ROI normalisation (supplement "Indexing algorithm", step 1): S / max_v S.  A
// CTA holds its row in shared memory between the maximum and the scaling, so the row is
// read once, all its reads in flight (256-thread CTAs that read it twice had 200 MB of
// rows in flight, more than L2 holds); only what lies beyond kNormHeld values is read
// again.  A thread reads back only the words it copied.  Bound by HBM: 8192 rows of 40962
// values (2.7 GB) 1.09 ms before, 0.55 now.
constexpr int kNormHeld = 48 * 1024;

__global__ void __launch_bounds__(1024, 1) k_normalise(float* S, int32_t nv) {
    extern __shared__ float held[];
    __shared__ float red[32];
    const int T = blockDim.x, tid = threadIdx.x, nh = min(nv, kNormHeld);
    float* row = S + (int64_t)blockIdx.x * nv;
    const uint32_t dst = smem_u32(held);
    for (int v = tid; v < nh; v += T)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * (uint32_t)v), "l"(row + v) : "memory");
    cp_async_wait_all();
    float mx = 0.f;
    for (int v = tid; v < nh; v += T) mx = fmaxf(mx, held[v]);
    for (int v = kNormHeld + tid; v < nv; v += T) mx = fmaxf(mx, row[v]);
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    __syncthreads();
    mx = (tid & 31) < (T >> 5) ? red[tid & 31] : 0.f;
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const float inv = mx > 0.f ? 1.0f / mx : 0.f;
    for (int v = tid; v < nh; v += T) row[v] = mx > 0.f ? held[v] * inv : 0.f;
    for (int v = kNormHeld + tid; v < nv; v += T) row[v] = mx > 0.f ? row[v] * inv : 0.f;
}

}  // namespace

cudaError_t launch_normalise(Ctx* c, float* S, int64_t rows) {
    if (rows < 0) rows = c->nroi;
    if (rows <= 0) return cudaSuccess;
    // some 40 values per thread; short rows leave room for several CTAs per SM
    const int threads = 32 * std::min(32, (c->nv + 1279) / 1280);
    const int smem = std::min(c->nv, kNormHeld) * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_normalise, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kNormHeld * (int)sizeof(float));   // the same whatever the call: threads may race
    if (e != cudaSuccess) return e;
    k_normalise<<<(unsigned)rows, threads, smem, c->stream>>>(S, c->nv);
    return cudaGetLastError();
}

size_t plain_smem_bytes(int m, int atom_cap) {
    const size_t NB = (size_t)1 << m;
    const size_t NBc = NB < (size_t)kChunkBins ? NB : (size_t)kChunkBins;
    const size_t ntw = NB == NBc ? 2 * NB : NB;   // as in the kernel
    return NBc * kWords * 4 + ntw * 8 + (size_t)atom_cap * 16 + kPartBytes + 64;
}

cudaError_t launch_signatures_plain(Ctx* c, float* S, uint16_t* argk, uint16_t* hist_out, int64_t hist_roi) {
    static int max_optin = -1;
    if (max_optin < 0) {
        cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
    }
    const size_t base = plain_smem_bytes(c->m, 0);
    int cap = (int)(((size_t)max_optin - base) / 16);
    cap = min(cap, 4096) & ~15;
    if (cap < 256) return cudaErrorInvalidConfiguration;
    const size_t smem = plain_smem_bytes(c->m, cap);
    const bool multi = !hist_out && c->multi.n > 0;
    const int mode = c->m > 10 ? kAllPasses : c->nw_max > kBlockAtoms ? kMixed : kSinglePass;
    void (*const kerns[2][3])(SigParams) = {
        {k_sig_plain<1, false, kSinglePass>, k_sig_plain<1, false, kMixed>, k_sig_plain<1, false, kAllPasses>},
        {k_sig_plain<APTIDX_MAX_BANDS, false, kSinglePass>, k_sig_plain<APTIDX_MAX_BANDS, false, kMixed>,
         k_sig_plain<APTIDX_MAX_BANDS, false, kAllPasses>}};
    void (*const kern)(SigParams) = kerns[multi][mode];
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;

    SigParams p;
    p.atoms = c->d_atoms;
    p.off = c->d_off;
    p.nw = c->d_nw;
    p.order = c->d_order;
    // antipodal pairs (one projection per pair) unless switched off, exporting,
    // or in passes over bin chunks (whose spectrum is not folded)
    const bool pairs = !hist_out && c->use_pairs && c->d_slot_idx && c->m <= 10;
    p.dirs = pairs ? c->d_slot_dirs : c->d_dirs;
    p.slot_idx = pairs ? c->d_slot_idx : nullptr;
    p.nv = c->nv;
    p.tiles_per_roi = (pairs ? c->nslot_pad : c->nv_pad) / kDirs;
    p.tiles_per_item = min(max(c->tune_tpi[0], 1), p.tiles_per_roi);
    p.items_per_roi = (p.tiles_per_roi + p.tiles_per_item - 1) / p.tiles_per_item;
    const int64_t nroi_lim = c->rank_limit > 0 ? tmin<int64_t>(c->nroi, c->rank_limit) : c->nroi;
    const int64_t nroi_eff = hist_out ? 1 : nroi_lim;
    p.n_items = nroi_eff * p.items_per_roi;
    p.scale = c->d_scale;
    p.band = c->d_band;
    p.m = c->m;
    p.tw = c->d_tw;
    p.S = S;
    p.argk = argk;
    p.hist_out = hist_out;
    p.single_roi = hist_out ? hist_roi : -1;
    p.counter = c->d_counter;
    p.status = c->d_status;
    p.atom_cap = cap;
    p.nroi = nroi_lim;
    p.bands = hist_out ? BandSet() : c->multi;
    if ((e = zero_counters(c)) != cudaSuccess) return e;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
    per_sm = max(per_sm, 1);
    const int64_t grid = tmin<int64_t>((int64_t)c->sm_count * per_sm, p.n_items);
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, kThreads, smem, c->stream>>>(p);
    return cudaGetLastError();
}

// -----------------------------------------------------------------------------
// No-allocation variant (aptidx_signatures_noalloc).  Everything a call derives
// from its inputs -- padded directions, per-ROI scale, band, atom count and
// order, the twiddle table, the work counter -- lives in one fixed scratch
// array in device memory, so the call allocates nothing.  Every GPU that loads
// the library holds the array until the process exits; all calls share it.
// -----------------------------------------------------------------------------
namespace {

constexpr int64_t kNaMaxRoi = APTIDX_NOALLOC_MAX_ROIS;
constexpr int64_t kNaMaxDirs = APTIDX_NOALLOC_MAX_DIRS;
// byte offsets inside the scratch array
constexpr size_t kNaDirs = 0;                                        // float4 [kNaMaxDirs]
constexpr size_t kNaTw = kNaDirs + 16 * (size_t)kNaMaxDirs;          // float2 [2 x 2^APTIDX_MAX_M]
constexpr size_t kNaScale = kNaTw + 16 * ((size_t)1 << APTIDX_MAX_M);  // float  [kNaMaxRoi]
constexpr size_t kNaBand = kNaScale + 4 * (size_t)kNaMaxRoi;         // int32  [2 kNaMaxRoi]
constexpr size_t kNaNw = kNaBand + 8 * (size_t)kNaMaxRoi;            // int32  [kNaMaxRoi]
constexpr size_t kNaOrder = kNaNw + 4 * (size_t)kNaMaxRoi;           // int32  [kNaMaxRoi]
constexpr size_t kNaCounter = kNaOrder + 4 * (size_t)kNaMaxRoi;      // int32  [4]
constexpr size_t kNaStatus = kNaCounter + 16;                        // int    [1]
constexpr size_t kNaEnd = kNaStatus + 16;
static_assert(kNaEnd <= APTIDX_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds the declared size");

static __device__ __align__(256) unsigned char g_noalloc_scratch[APTIDX_NOALLOC_SCRATCH_BYTES];

// Per-call set-up: counts, scales, bands and identity order per ROI; padded
// float4 directions; the twiddle table.  Flags ROIs above 65535 atoms
// (overflow), radii outside [1e-6, 1e6] nm and directions that are not unit
// vectors (invalid input); a flagged ROI gets zero atoms, so its row of S is
// zero.
__global__ void k_noalloc_setup(unsigned char* scr, const int64_t* __restrict__ off, const double* __restrict__ radii,
                                int64_t nroi, const float* __restrict__ u, int32_t nv, int32_t nv_pad, int m,
                                int32_t k_lo, int32_t k_hi, int* status) {
    float4* dirs = reinterpret_cast<float4*>(scr + kNaDirs);
    float2* tw = reinterpret_cast<float2*>(scr + kNaTw);
    float* scale = reinterpret_cast<float*>(scr + kNaScale);
    int32_t* band = reinterpret_cast<int32_t*>(scr + kNaBand);
    int32_t* nw = reinterpret_cast<int32_t*>(scr + kNaNw);
    int32_t* order = reinterpret_cast<int32_t*>(scr + kNaOrder);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int half = 1 << (m - 1);
    for (int64_t r = t0; r < nroi; r += stride) {
        int64_t n = off[r + 1] - off[r];
        if (n < 0 || n > APTIDX_MAX_ATOMS_PER_ROI) {
            atomicOr(status, kStatusOverflow);
            n = 0;
        }
        const double R = radii[r];
        if (!(R >= 1e-6 && R <= 1e6)) {   // also false for NaN
            atomicOr(status, kStatusInvalid);
            n = 0;
        }
        nw[r] = (int32_t)n;
        scale[r] = n > 0 ? __double2float_rn((double)(half - 1) / R) : 0.f;
        band[2 * r] = k_lo;
        band[2 * r + 1] = k_hi;
        order[r] = (int32_t)r;
    }
    for (int64_t v = t0; v < nv_pad; v += stride) {
        float4 d = make_float4(1.f, 0.f, 0.f, 0.f);
        if (v < nv) {
            d = make_float4(u[3 * v], u[3 * v + 1], u[3 * v + 2], 0.f);
            const double n2 = (double)d.x * d.x + (double)d.y * d.y + (double)d.z * d.z;
            if (!(fabs(sqrt(n2) - 1.0) <= 1e-5)) atomicOr(status, kStatusInvalid);
        }
        dirs[v] = d;
    }
    for (int64_t j = t0; j < (int64_t)(2 << m); j += stride) {
        double sn, cs;
        sincospi((double)j / (double)(1 << m), &sn, &cs);
        tw[j] = make_float2((float)cs, (float)sn);
    }
}

std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64] = {};

}  // namespace

}  // namespace aptidx

extern "C" int aptidx_signatures_noalloc(const float* xc4, const int64_t* off, const double* radii, int64_t nroi,
                                         const float* u, int32_t nv, int m, int32_t k_lo, int32_t k_hi, float* S,
                                         int* status, void* cuda_stream) {
    using namespace aptidx;
    if (nroi < 0 || nroi > kNaMaxRoi || nv <= 0 || nv > kNaMaxDirs) return APTIDX_E_INVALID_ARG;
    if (m < APTIDX_MIN_M || m > APTIDX_MAX_M) return APTIDX_E_INVALID_ARG;
    if (k_lo < 0 || k_hi < k_lo || k_hi > (1 << (m - 1))) return APTIDX_E_INVALID_ARG;
    if (nroi == 0) return APTIDX_OK;
    if (!xc4 || !off || !radii || !u || !S) return APTIDX_E_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(xc4) & 15u) != 0) return APTIDX_E_INVALID_ARG;   // bulk copies need 16-byte rows
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return APTIDX_E_CUDA;
    }
    void* scr = nullptr;
    {
        // set-up, once per device, with that device current: the host-side
        // name of the array is not a device address
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
                cudaGetLastError();
                return APTIDX_E_CUDA;
            }
            g_noalloc_ptr[dev] = ptr;
        }
        scr = g_noalloc_ptr[dev];
    }
    unsigned char* base = static_cast<unsigned char*>(scr);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int* st = status ? status : reinterpret_cast<int*>(base + kNaStatus);
    int32_t* counter = reinterpret_cast<int32_t*>(base + kNaCounter);
    const int32_t nv_pad = (nv + kTileDirs - 1) / kTileDirs * kTileDirs;
    int sm_count = 0, max_optin = 0;
    if (cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return APTIDX_E_CUDA;
    }
    // the work counter must start at zero; the rest is rewritten by the set-up kernel
    if (cudaMemsetAsync(counter, 0, 16, s) != cudaSuccess) return APTIDX_E_CUDA;
    const int64_t work = std::max<int64_t>(nroi, (int64_t)nv_pad);
    k_noalloc_setup<<<(unsigned)std::min<int64_t>((work + 255) / 256, 1024), 256, 0, s>>>(base, off, radii, nroi, u, nv,
                                                                                       nv_pad, m, k_lo, k_hi, st);
    if (cudaGetLastError() != cudaSuccess) return APTIDX_E_CUDA;
    const size_t smem_base = plain_smem_bytes(m, 0);
    int cap = (int)(((size_t)max_optin - smem_base) / 16);
    cap = std::min(cap, 4096) & ~15;
    if (cap < 256) return APTIDX_E_CUDA;
    const size_t smem = plain_smem_bytes(m, cap);
    if (cudaFuncSetAttribute(k_sig_plain<1, true, kMixed>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return APTIDX_E_CUDA;
    }
    SigParams p;
    p.atoms = reinterpret_cast<const float4*>(xc4);
    p.off = off;
    p.nw = reinterpret_cast<const int32_t*>(base + kNaNw);
    p.order = reinterpret_cast<const int32_t*>(base + kNaOrder);
    p.dirs = reinterpret_cast<const float4*>(base + kNaDirs);
    p.slot_idx = nullptr;
    p.nv = nv;
    p.tiles_per_roi = nv_pad / kDirs;
    p.tiles_per_item = std::min(16, p.tiles_per_roi);
    p.items_per_roi = (p.tiles_per_roi + p.tiles_per_item - 1) / p.tiles_per_item;
    p.n_items = nroi * p.items_per_roi;
    p.scale = reinterpret_cast<const float*>(base + kNaScale);
    p.band = reinterpret_cast<const int32_t*>(base + kNaBand);
    p.m = m;
    p.tw = reinterpret_cast<const float2*>(base + kNaTw);
    p.S = S;
    p.argk = nullptr;
    p.hist_out = nullptr;
    p.single_roi = -1;
    p.counter = counter;
    p.status = st;
    p.atom_cap = cap;
    p.nroi = nroi;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sig_plain<1, true, kMixed>, kThreads, smem);
    per_sm = std::max(per_sm, 1);
    const int64_t grid = std::min<int64_t>((int64_t)sm_count * per_sm, p.n_items);
    k_sig_plain<1, true, kMixed><<<(unsigned)grid, kThreads, smem, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? APTIDX_OK : APTIDX_E_CUDA;
}
