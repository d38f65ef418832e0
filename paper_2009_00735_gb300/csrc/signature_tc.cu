// signature_tc.cu -- steps (a2)-(a5) with the band spectrum on the tcgen05
// tensor cores: X = H x T, H the [64 directions x bins] histogram tile and T
// the [bins x band columns] DFT matrix (cos and sin of 2 pi k n / 2^m),
// accumulated in FP32 in tensor memory (Section 2.2: the Fourier amplitude
// spectrum of every SDM; the paper notes that the SDMs of a ROI share one
// bin count, which permits batching their transforms).
//
// The histogram of a tile covers all bins (tiles of 64 directions up to 2^10 bins,
// of 32 and 16 at 2^11 and 2^12) over blocks of at most 2048 atoms, so that every
// count of a block is exact in fp16; all blocks are contracted into the same
// tensor-memory accumulators.  The bins split into four parts (eight of 2^12 bins):
// the rows of the contraction (M = 128) are (part, direction), all parts use the
// twiddles of the first, since w^(k (n + h)) = w^(k h) w^(k n) for
// w = exp(-2 pi i / 2^m), and the epilogue adds the parts with their factors
// w^(k h), fourth or eighth roots of one.
//
// Antipodal pairs: when the direction set holds u and -u, only u is projected;
// -u gets the same signature value and frequency bin (its histogram is the
// mirror image of u's, whose spectrum has the same amplitudes), provided no
// atom's bin product along u is an exact integer, which the histogram pass
// checks exactly (common.cuh).  A tile with such an atom runs a second pass
// over the negated directions and writes their signatures from their own
// histograms.
//
// Per tile and atom block:
//   1. 16 warps histogram by shared-memory atomics (bank-private columns, as in the
//      FP32 path); counts c <= 2048, so the u16 bit pattern of c is the fp16 value
//      c * 2^-24 exactly (fp16 is linear through its subnormal range up to 0x0800);
//   2. the same warps exchange every word with zero and store the counts to tensor
//      memory, pairs of bins to a column: that is the A operand, and the histogram is
//      ready for the next tile;
//   3. four more warps issue the tcgen05.mma (A in tensor memory, K = 16, N = 16 per
//      group of 4 frequencies: 8 hi columns, then 8 lo columns, where T = T_hi + T_lo
//      with both parts fp16; the twiddles stay in shared memory) and
//   4. read the accumulators (tcgen05.ld) of the tile before, add the partials, hi and
//      lo parts and the bin parts (one exchange in shared memory), scale by 2^24 and
//      keep the band maximum of |X(k)|.
// 3 and 4 run under the next tile's 1.  Wide bands (more groups than shared memory
// holds twiddles for) take k_sig_wide, below.
//
// What bounds it (2^10 bins, 1133 atoms, per 64-direction tile, cycles): the
// histogram takes 5.2-5.6 K and the transfer 1.4 K, with 1.1 K to set up a tile and
// 0.5 K of barriers; MMAs and epilogue (3.7 K) hide behind them.  The histogram is
// bound by issue and the shared-memory pipe together: 8 packed FMAs of two slots each,
// 4 shifts, 3 slots of the zero check and about four slots per increment for every two
// atoms and two directions; 2.26 K increments and 1.7 K atom-load wavefronts
// (neither unrolling, software pipelining, 8 to 24 warps, halved atom loads nor
// stores in place of the atomics change it).  Over the whole kernel 60 % of the issue
// slots, 65 % of the shared-memory cycles.  One CTA per SM ran these phases one
// after the other with the counts in shared memory: 13.5 K cycles, 116.5 ms for 8192
// ROIs x 40962 directions; now 73.9 ms.
#include <cuda_fp16.h>

#include "tcgen05.cuh"

namespace aptidx {

namespace {

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kDirs = kTileDirs;     // 64 directions per tile
constexpr int kRows = 2 * kDirs;     // MMA M of wide bands: (direction, bin half)
constexpr int kBtBytes = 32 * 1024;  // shared-memory budget of the B operand (narrow bands)
constexpr int kWideStage = 16 * 1024;   // wide bands: one of four twiddle stream stages
constexpr int kExBytes = kDirs * 8 * 4;   // epilogue exchange: one group's (re, im) x 4 per direction
constexpr int kChunkBins = 1024;     // bins per histogram chunk (128 KB of words)

struct TcParams {
    const float4* atoms;
    const int64_t* off;
    const int32_t* nw;
    const int32_t* order;
    const float4* dirs;     // direction slots, padded to whole tiles with (1, 0, 0)
    const int2* slot_idx;   // per slot: (output direction, antipodal partner or -1); NULL: slot = direction
    int32_t nv;
    int32_t tiles_per_roi;
    int32_t tiles_per_item;
    int32_t items_per_roi;
    int64_t nroi;
    const float* scale;
    const int32_t* band;
    int m;
    int32_t kbase;          // frequency of column group 0
    const uint8_t* twb;     // global B: [chunk][hi|lo][group][k-block] x 1 KB
    const uint8_t* twk;     // global B, streamed layout: [chunk][32-bin block of the first quarter][hi|lo]
                            // [group] x 512 B, 64-byte swizzle (wide bands), ng_total + 1 groups per run,
                            // the last one zero
    int32_t bt_bytes;       // shared-memory bytes of the B region (kBtBytes, or 4 kWideStage)
    int32_t ng_total;
    uint32_t tmem_cols;     // wide bands
    float* S;
    uint16_t* argk;
    uint16_t* hist_out;
    int64_t single_roi;
    int32_t* counter;
    int* status;
    int atom_cap;           // atoms per block (<= 2048)
    int n_iss;              // MMA issuer warps of narrow bands (2 or 4)
    BandSet bands;
};

__device__ __forceinline__ void cp_async8(void* dst_smem, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}

// Debug export of one (block, chunk) pass: adds the counts of rows
// [0, nbc) to h_out[v * 2^m + bc * nbc + row] (the caller zeroes h_out).
__device__ __forceinline__ void hist_export_add(const uint32_t* H, int nbc, int NB, int bc, int tile, int nv,
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

// v += (-i)^(R0 + q) u for the n complex pairs (re, im) of v and u, where a
// pair (r, i) stands for r - i i: multiplying by -i maps it to (-i, r), by -1
// to (-r, -i), by i to (i, -r)
template <int R0>
__device__ __forceinline__ void quarter_rot(float* v, const float* u, int n) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        if (q < n) {
            const int ph = (R0 + q) & 3;   // constant once unrolled
            const float ur = u[2 * q], ui = u[2 * q + 1];
            v[2 * q] += ph == 0 ? ur : ph == 1 ? -ui : ph == 2 ? -ur : ui;
            v[2 * q + 1] += ph == 0 ? ui : ph == 1 ? ur : ph == 2 ? -ui : -ur;
        }
    }
}

// ---- the kernel ----------------------------------------------------------------

constexpr int kHistWarps = 16;                       // warps 0-15: projection, histogram, transfer
constexpr int kHistThreads = kHistWarps * 32;
constexpr int kAuxThreads = 128;                     // warps 16-19: MMA issue, epilogue, output
constexpr int kTpThreads = kHistThreads + kAuxThreads;
constexpr int kExFloats = 4 * 2 * 8 * 32;            // epilogue exchange: 4 bin quarters x 2 x 8 values x 32 lanes
constexpr int kTmemA = 0;                            // A operand: even directions, odd directions 128 columns on
constexpr int kTmemD = 256;                          // accumulators
constexpr int kTmemCols = 512;

// (cos, sin)(pi j / 4)
__constant__ float2 kRoots[8] = {{1.f, 0.f},  {0.70710678118654752f, 0.70710678118654752f},
                                 {0.f, 1.f},  {-0.70710678118654752f, 0.70710678118654752f},
                                 {-1.f, 0.f}, {-0.70710678118654752f, -0.70710678118654752f},
                                 {0.f, -1.f}, {0.70710678118654752f, -0.70710678118654752f}};

// what a pass hands from the histogram warps to the others
struct TpPass {
    int64_t roi;
    int32_t tile, flags;
    int32_t g0, ng, klo, khi;   // first frequency group, groups, the ROI's band
};
constexpr int kPassStop = 1, kPassFirst = 2, kPassLast = 4, kPassBad = 8, kPassPartner = 16;

__device__ __forceinline__ void hist_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kHistThreads) : "memory"); }
__device__ __forceinline__ void aux_sync() { asm volatile("bar.sync 3, 128;" ::: "memory"); }
__device__ __forceinline__ bool hist_sync_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 2, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(v ? 1u : 0u), "n"(kHistThreads)
        : "memory");
    return r != 0;
}

// K rows of the B operand: the bins of one part (a quarter of up to 2^11, an
// eighth of 2^12)
__host__ __device__ __forceinline__ int tp_k_rows(int m) { return m <= 11 ? 1 << (m - 2) : 1 << (m - 3); }

// Debug export of one pass: adds the counts to h_out[v * 2^m + bin] (the caller
// zeroes h_out); rows of 32 >> split words
__device__ __forceinline__ void hist_export_rows(const uint32_t* H, int m, int split, int tile, int nv, uint16_t* h_out,
                                                 int tid, int nthreads) {
    const int64_t NB = (int64_t)1 << m;
    for (int i = tid; i < (1 << m) * (32 >> split); i += nthreads) {
        const int b = i >> (5 - split), l = i & ((32 >> split) - 1);
        const uint32_t w = H[i];
        const int64_t v0 = (int64_t)tile * (kDirs >> split) + 2 * l;
        if (v0 < nv) h_out[v0 * NB + b] = (uint16_t)(h_out[v0 * NB + b] + (w & 0xFFFFu));
        if (v0 + 1 < nv) h_out[(v0 + 1) * NB + b] = (uint16_t)(h_out[(v0 + 1) * NB + b] + (w >> 16));
    }
}

// kNB: band slots of the epilogue (1: the ROI's own band; APTIDX_MAX_BANDS:
// the pass's BandSet, aptidx_compute_signatures_multi)
// split: 2^11 and 2^12 bins run tiles of 32 and 16 directions, rows of 16 and 8
// words, so that a tile's histogram stays at 128 KB and no atom is projected twice
// (passes over chunks of 1024 bins projected each atom two or four times, with
// predicated increments: 18 K cycles for 1815 atoms, 10 per atom, against 5).  A
// template argument: as a variable of one kernel it cost the 2^10-bin pass 20 %.
template <int kNB, int split>
__global__ void __launch_bounds__(kTpThreads, 1) k_sig_tp(TcParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int DT = kDirs >> split;      // directions per tile
    const int NB = 1 << p.m;
    constexpr int pitch = 128 >> split;     // bytes of a histogram row (one bin)
    const int K = tp_k_rows(p.m);           // bins per part (a quarter, of 2^12 an eighth)
    const int KB = K / 64;                  // 64-row K blocks of the B operand
    uint32_t* H = reinterpret_cast<uint32_t*>(smem);
    unsigned char* BT = smem + (size_t)NB * pitch;
    float* EX = reinterpret_cast<float*>(BT + p.bt_bytes);   // [2][kExFloats]
    float4* A = reinterpret_cast<float4*>(EX + 2 * kExFloats);
    float4* DB = A + p.atom_cap;   // [2][parity][32]: this tile's directions and the next tile's
    TpPass* pass_s = reinterpret_cast<TpPass*>(DB + 2 * kDirs);   // [2]
    uint64_t* bars = reinterpret_cast<uint64_t*>(pass_s + 2);
    uint64_t* bar_atoms = bars;
    uint64_t* bar_b = bars + 1;
    uint64_t* bar_full = bars + 2;    // A operand of a pass written (16 histogram warps)
    uint64_t* bar_mma = bars + 3;     // [2] its MMAs done (4 auxiliary warps), by pass parity
    int* item_s = reinterpret_cast<int*>(bars + 5);
    uint32_t* tmem_s = reinterpret_cast<uint32_t*>(bars + 6);
    unsigned* r2max_s = tmem_s + 1;   // largest |x|^2 of the item's atoms
    volatile int* hist_fail = reinterpret_cast<volatile int*>(bars + 7);
    volatile int* aux_fail = hist_fail + 1;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(bar_atoms, 1);
        mbar_init(bar_b, 1);
        mbar_init(bar_full, kHistWarps);
        mbar_init(&bar_mma[0], 4);
        mbar_init(&bar_mma[1], 4);
        *hist_fail = 0;
        *aux_fail = 0;
        fence_barrier_init();
    }
    for (int i = tid; i < NB * pitch / 16; i += kTpThreads) reinterpret_cast<uint4*>(H)[i] = make_uint4(0, 0, 0, 0);
    if (warp == kHistWarps) tmem_alloc(tmem_s, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_s;
    const uint32_t h_addr = smem_u32(H);
    const bool sym = p.slot_idx != nullptr;

    if (warp < kHistWarps) {
        // ================= histogram warps =================
        const float magic = quad_magic(p.m, h_addr / (uint32_t)pitch);
        // the lane's word of a row, and its group of lanes (warps hold 1, 2 or 4
        // whole rows, each group walks its own atoms)
        const int word = lane & ((32 >> split) - 1);
        const int group = (warp << split) + (lane >> (5 - split)), ngroups = kHistWarps << split;
        const int n_items = (int)((p.single_roi >= 0 ? 1 : p.nroi) * p.items_per_roi);   // < 2^31 (launch)
        uint32_t ph_atoms = 0, t = 0;   // t: passes handed over
        // this warp's share of the transfer: the bins of quarter warp & 3 (the
        // tensor-memory lanes it may write), a quarter of its 128-byte lines
        const int tr_lines = NB * pitch / 128 / 16;
        const uint32_t tr_addr =
            h_addr + ((uint32_t)((warp & 3) * 4 * tr_lines) << 7) + 4u * (uint32_t)lane;
        const uint32_t tr_tmem = tmem + kTmemA + ((uint32_t)((warp & 3) * 32) << 16);
        bool failed = false;
        if (tid == 0) *item_s = atomicAdd(p.counter, 1);
        hist_sync();
        int item = *item_s;
        // atoms [0, n) from src into A by one bulk copy, arranged in blocks of four
        auto stage = [&](const float4* src, int n, unsigned* r2) -> bool {
            if (tid == 0) {
                if (r2) *r2 = 0u;
                if (n > 0) {
                    fence_proxy_async_smem();   // earlier generic accesses of A before the async write
                    mbar_arrive_expect_tx(bar_atoms, (uint32_t)n * 16u);
                    bulk_g2s(A, src, (uint32_t)n * 16u, bar_atoms);
                    if (!mbar_wait_bounded(bar_atoms, ph_atoms, p.status)) {
                        mbar_wait_bounded(bar_atoms, ph_atoms, p.status, 1u << 20);   // let the copy land
                        *hist_fail = 1;
                    }
                }
            }
            if (n > 0) ph_atoms ^= 1u;
            hist_sync();
            if (*hist_fail) return false;
            quad_atoms(A, n, tid, kHistThreads, r2);
            hist_sync();
            return true;
        };
        while (item < n_items && !failed) {
            // the next item, published when this one is done: claimed ahead while many are
            // left (a claim takes 0.7 us), but none of the last, which a CTA that starts
            // early would hold while another has nothing to do (152 items of 21 ROIs on
            // 152 SMs took 0.64 ms or 1.2, from one launch to the next)
            int next = -1;
            if (tid == 0 && item + 2 * (int)gridDim.x < n_items) next = atomicAdd(p.counter, 1);
            const int roi = p.single_roi >= 0 ? (int)p.single_roi : p.order[item / p.items_per_roi];
            const int grp = item % p.items_per_roi;
            const int nw = p.nw[roi];
            const float scale = p.scale[roi];
            const int klo = p.band[2 * roi], khi = p.band[2 * roi + 1];
            const int t0 = grp * p.tiles_per_item;
            const int t1 = min(t0 + p.tiles_per_item, p.tiles_per_roi);
            const int nblk = max(1, (nw + p.atom_cap - 1) / p.atom_cap);   // atom blocks
            // the first tile's directions (later tiles' arrive while the tile before
            // them runs; held in shared memory: in registers the loop spilled them,
            // 1.6 K cycles per tile)
            // slot 2 l + i of a tile at [i][l]: a warp reads 512 consecutive bytes
            const int db_slot = (tid & 1) * 32 + (tid >> 1);
            if (tid < DT) cp_async16(DB + (t0 & 1) * kDirs + db_slot, p.dirs + (int64_t)t0 * DT + tid);
            cp_async_wait_all();
            if (nblk > 1) {
                hist_sync();
            } else if (!stage(p.atoms + p.off[roi], nw, r2max_s)) {
                failed = true;
                break;
            }
            // with one atom block and no nonzero integer product possible, the
            // antipodal check only looks for s = 0
            const bool zero_check =
                sym && nblk == 1 && !nonzero_integer_products_possible(scale, __uint_as_float(*r2max_s));
            for (int tile = t0; tile < t1 && !failed; ++tile) {
                float4 d0 = DB[(tile & 1) * kDirs + word], d1 = DB[(tile & 1) * kDirs + 32 + word];
                if (tile + 1 < t1 && tid < DT)
                    cp_async16(DB + ((tile + 1) & 1) * kDirs + db_slot, p.dirs + (int64_t)(tile + 1) * DT + tid);
                const bool pt0 = d0.w != 0.f, pt1 = d1.w != 0.f;   // the slot has an antipodal partner
                bool tile_bad = false;
                for (int pass = 0; pass < 2 && !failed; ++pass) {
                    if (pass == 1) {
                        if (!tile_bad) break;
                        // the partners -u of this tile's directions, from their own histograms
                        d0 = make_float4(-d0.x, -d0.y, -d0.z, d0.w);
                        d1 = make_float4(-d1.x, -d1.y, -d1.z, d1.w);
                    }
                    const bool count = sym && pass == 0;
                    const QuadDirs q = quad_dirs(d0, d1, scale, magic, word, split);
                    uint32_t c0 = 0, c1 = 0;
                    float zmin = 1.f;
                    int handled = 0;
                    for (int blk = 0; blk < nblk; ++blk, ++t) {
                        const int cn = min(p.atom_cap, nw - blk * p.atom_cap);
                        const bool last = blk == nblk - 1;
                        if (nblk > 1 && !stage(p.atoms + p.off[roi] + (int64_t)blk * p.atom_cap, cn, nullptr)) {
                            failed = true;
                            break;
                        }
                        // ---- 1. histograms (H is zero here) ----
                        if (count && zero_check)
                            handled += hist_tile_quads<2, false, split>(A, cn, group, ngroups, q, c0, c1, zmin);
                        else if (count)
                            handled += hist_tile_quads<1, false, split>(A, cn, group, ngroups, q, c0, c1, zmin);
                        else
                            hist_tile_quads<0, false, split>(A, cn, group, ngroups, q, c0, c1, zmin);
                        // the non-integer counts are complete once the last pass's
                        // histogram is in: a partner whose count falls short of the
                        // atoms this group handled needs its own histogram
                        const bool bad = count && last &&
                                         (zero_check ? (pt0 || pt1) && zmin == 0.f
                                                     : (pt0 && c0 != (uint32_t)handled) || (pt1 && c1 != (uint32_t)handled));
                        // the A operand of the pass before has been read (asked by the
                        // last warp, which never has more atoms than the others)
                        if (tid == kHistThreads - 1) {
                            if (t > 0 && !mbar_wait_bounded(&bar_mma[(t - 1) & 1], ((t - 1) >> 1) & 1u, p.status))
                                *hist_fail = 1;
                            if (*aux_fail) *hist_fail = 1;
                        }
                        const bool any_bad = hist_sync_or(bad);
                        if (last && pass == 0) tile_bad = any_bad;
                        if (*hist_fail) {
                            failed = true;
                            break;
                        }
                        tc_fence_after();
                        if (p.hist_out) {
                            hist_export_rows(H, p.m, split, tile, p.nv, p.hist_out, tid, kHistThreads);
                            hist_sync();   // every row is read before the transfer zeroes it
                        }
                        if (tid == 0) {
                            TpPass m;
                            m.roi = roi;
                            m.tile = tile;
                            m.flags = (blk == 0 ? kPassFirst : 0) | (last ? kPassLast : 0) | (tile_bad ? kPassBad : 0) |
                                      (pass ? kPassPartner : 0);
                            m.g0 = (klo - p.kbase) >> 2;
                            m.ng = ((khi - p.kbase) >> 2) - m.g0 + 1;
                            m.klo = klo;
                            m.khi = khi;
                            pass_s[t & 1] = m;
                        }
                        // ---- 2. transfer: counts into tensor memory, the histogram
                        // zeroed behind them by exchanging each word with 0 (a load
                        // and a store pass over the rows took twice the shared-memory
                        // cycles).  Word (bin, lane) holds directions 2 lane and
                        // 2 lane + 1; two bins' words make a K pair of either ----
                        for (int r = 0; r < tr_lines; r += 16) {
                            // split 2 takes eight lines of either eighth of its quarter
                            const int l0 = (warp >> 2) * tr_lines + r;
                            uint32_t w[16];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int line = split < 2 ? l0 + i : l0 / 2 + (i >> 1) + (i & 1) * 2 * tr_lines;
                                asm volatile("atom.shared.exch.b32 %0, [%1], 0;"
                                             : "=r"(w[i])
                                             : "r"(tr_addr + 128u * (uint32_t)line)
                                             : "memory");
                            }
                            if (split == 0) {
                                // a line is a bin: pairs of lines make K pairs of the even
                                // directions (columns 0..) and of the odd ones (128..)
                                uint32_t e[8], o[8];
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    e[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
                                    o[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
                                }
                                tmem_st8(tr_tmem + (uint32_t)(l0 / 2), e);
                                tmem_st8(tr_tmem + 128u + (uint32_t)(l0 / 2), o);
                            } else if (split == 1) {
                                // a line is two bins, one K pair: lanes 0-15 take the even
                                // directions, 16-31 the odd ones
                                const bool odd = lane >= 16;
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    const uint32_t x = __shfl_xor_sync(0xffffffffu, w[i], 16);
                                    w[i] = odd ? __byte_perm(x, w[i], 0x7632) : __byte_perm(w[i], x, 0x5410);
                                }
                                tmem_st8(tr_tmem + (uint32_t)l0, w);
                                tmem_st8(tr_tmem + (uint32_t)l0 + 8u, w + 8);
                            } else {
                                // a line is four bins, two K pairs; a line of the quarter's
                                // first eighth (lanes 0-15) and one of its second (16-31)
                                // make two columns, even directions in the lower eight lanes
                                const bool odd = (lane & 8) != 0, hi = lane >= 16;
#pragma unroll
                                for (int i = 0; i < 16; i += 2) {
                                    const uint32_t xa = __shfl_xor_sync(0xffffffffu, w[i], 8);
                                    const uint32_t xb = __shfl_xor_sync(0xffffffffu, w[i + 1], 8);
                                    const uint32_t va = odd ? __byte_perm(xa, w[i], 0x7632) : __byte_perm(w[i], xa, 0x5410);
                                    const uint32_t vb = odd ? __byte_perm(xb, w[i + 1], 0x7632) : __byte_perm(w[i + 1], xb, 0x5410);
                                    const uint32_t x = __shfl_xor_sync(0xffffffffu, hi ? va : vb, 16);
                                    w[i] = hi ? x : va;
                                    w[i + 1] = hi ? vb : x;
                                }
                                tmem_st8(tr_tmem + (uint32_t)l0, w);
                                tmem_st8(tr_tmem + (uint32_t)l0 + 8u, w + 8);
                            }
                        }
                        tmem_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_full);
                        cp_async_wait_all();
                        hist_sync();   // the histogram is zero, the next directions are in
                    }
                }
            }
            if (tid == 0) *item_s = next >= 0 ? next : atomicAdd(p.counter, 1);
            hist_sync();
            item = *item_s;
            // (the next write of item_s comes after the barriers of an item)
        }
        // the auxiliary warps leave at a pass marked stop, handed over (like any
        // other) only once the pass before has been taken: bar_full never runs two
        // phases ahead of its reader
        if (tid == 0) {
            if (!failed && t > 0) mbar_wait_bounded(&bar_mma[(t - 1) & 1], ((t - 1) >> 1) & 1u, p.status);
            pass_s[t & 1].flags = kPassStop;
        }
        hist_sync();
        if (lane == 0) mbar_arrive(bar_full);
    } else {
        // ================= auxiliary warps =================
        const int at = tid - kHistThreads, aw = at >> 5;   // warp aw: tensor-memory lanes 32 aw .., bin quarter aw
        const uint32_t bt_addr = smem_u32(BT);
        constexpr int blocks = split == 0 ? 2 : 1;   // A operands of a tile: even and odd directions, or all
        const int nh = p.n_iss / blocks;         // accumulators per block (parts of K)
        uint32_t ph_b = 0, exb = 0;
        int cur_g0 = -1, cur_ng = -1;   // B operand in shared memory
        // accumulators: two buffers of 128 columns in turn when a tile's fit one,
        // else one of 256
        bool pending = false;
        TpPass pend;
        uint32_t pend_t = 0, pend_d = 0, dbuf = 0;

        // wait for the MMAs of pass `u` (thread 0 of the group) and publish the outcome
        auto done = [&](uint32_t u) -> bool {
            if (at == 0 && !mbar_wait_bounded(&bar_mma[u & 1], (u >> 1) & 1u, p.status)) *aux_fail = 1;
            aux_sync();
            return *aux_fail == 0;
        };
        // |X(k)| and the band maximum of one tile: every warp sums its quarter's
        // partials of a frequency group, threads 0-63 (one per direction) add the
        // four quarters with their factors w^(f q NBc / 4)
        auto epilogue = [&](const TpPass& m, uint32_t u, uint32_t dsel) -> bool {
            if (!done(u)) return false;
            tc_fence_after();
            const uint32_t cols = (uint32_t)(16 * m.ng);
            const uint32_t dcol = tmem + ((uint32_t)(aw * 32) << 16) + kTmemD + dsel;
            float best[kNB];
            int bk[kNB];
            band_init_t<kNB>(p.bands, m.klo, best, bk);
            for (int j = 0; j < m.ng; ++j) {
                float* ex = EX + (exb & 1) * kExFloats;
                ++exb;
#pragma unroll
                for (int b = 0; b < blocks; ++b) {
                    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                    for (int h = 0; h < nh; ++h) {
                        float hi[8], lo[8];
                        const uint32_t c = dcol + (uint32_t)(h * blocks + b) * cols + (uint32_t)(8 * j);
                        tmem_ld8(c, hi);
                        tmem_ld8(c + (uint32_t)(8 * m.ng), lo);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] += hi[i] + lo[i];
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) ex[((aw * blocks + b) * 8 + i) * 32 + lane] = v[i];
                }
                tc_fence_before();
                aux_sync();
                if (at < DT) {
                    const int f0 = p.kbase + 4 * (m.g0 + j);
                    // direction at: parity at & 1, word at >> 1; part q of the bins at + q * step
                    const int pos = split == 0 ? (at & 1) * 256 + (at >> 1) : (at & 1) * (16 >> (split - 1)) + (at >> 1);
                    const float* x = ex + pos;
                    float xr[4] = {0.f, 0.f, 0.f, 0.f}, xi[4] = {0.f, 0.f, 0.f, 0.f};
                    constexpr int parts = split == 2 ? 8 : 4;
                    // 2^12 bins: 16 threads add eight parts, unrolled and with the factors
                    // read from a table (formed by selects in a loop this took 6.9 K
                    // cycles per tile and bounded small ROIs: 700 of 31 atoms x 9001
                    // directions 11.5 ms, now 8.2; the other tiles hide it)
#pragma unroll
                    for (int q = 0; q < parts; ++q) {
                        const float* y = split == 0 ? x + q * 512 : split == 1 ? x + q * 256 : x + (q >> 1) * 256 + (q & 1) * 16;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            // w^(f q NB / parts) = fc - i fs, an eighth root of one
                            const int ph = ((f0 + i) * q * (8 / parts)) & 7;
                            const float root = 0.70710678118654752f;
                            float fc, fs;
                            if constexpr (split == 2) {
                                fc = kRoots[ph].x;
                                fs = kRoots[ph].y;
                            } else {
                                fc = (ph & 3) == 2 ? 0.f : ((ph & 1) ? root : 1.f) * (ph > 2 && ph < 6 ? -1.f : 1.f);
                                fs = (ph & 3) == 0 ? 0.f : ((ph & 1) ? root : 1.f) * (ph > 4 ? -1.f : 1.f);
                            }
                            const float r = y[(2 * i) * 32], s = y[(2 * i + 1) * 32];
                            xr[i] += fc * r - fs * s;
                            xi[i] += fs * r + fc * s;
                        }
                    }
                    // the band maximum on |X|^2 (its root is the maximum amplitude)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        band_update_t<kNB>(p.bands, m.klo, m.khi, f0 + i, xr[i] * xr[i] + xi[i] * xi[i], best, bk);
                }
            }
            if (at < DT) {
                const int slot = m.tile * DT + at;
                int v0 = slot < p.nv ? slot : -1, v1 = -1;
                if (sym) {
                    // the slot's direction, and its partner when the tile's mirror
                    // images are exact; a partner pass writes the partners
                    const int2 si = p.slot_idx[slot];
                    v0 = (m.flags & kPassPartner) ? si.y : si.x;
                    v1 = (m.flags & (kPassPartner | kPassBad)) ? -1 : si.y;
                }
                const int64_t rb = (p.single_roi >= 0 ? 0 : m.roi) * (int64_t)p.nv;
#pragma unroll
                for (int b = 0; b < kNB; ++b) {
                    if (b < band_count_t<kNB>(p.bands)) {
                        const float a = best[b] >= 0.f ? sqrtf(best[b]) * 16777216.0f : best[b];
                        const int64_t ob = band_off_t<kNB>(p.bands, b) + rb;
                        if (v0 >= 0) {
                            p.S[ob + v0] = a;
                            if (p.argk) p.argk[ob + v0] = (uint16_t)bk[b];
                        }
                        if (v1 >= 0) {
                            p.S[ob + v1] = a;
                            if (p.argk) p.argk[ob + v1] = (uint16_t)bk[b];
                        }
                    }
                }
            }
            return true;
        };

        bool ok = true;
        for (uint32_t t = 0; ok; ++t) {
            if (at == 0 && !mbar_wait_bounded(bar_full, t & 1u, p.status)) *aux_fail = 1;
            aux_sync();
            if (*aux_fail) break;
            tc_fence_after();
            const TpPass m = pass_s[t & 1];
            if (m.flags & kPassStop) break;
            // ---- B operand of the band ----
            const uint32_t part = (uint32_t)m.ng * KB * 1024u;
            if (m.g0 != cur_g0 || m.ng != cur_ng) {
                if (t > 0 && !done(t - 1)) break;   // its MMAs read the operand held so far
                if (at == 0) {
                    fence_proxy_async_smem();
                    mbar_arrive_expect_tx(bar_b, 2u * part);
                    for (int i = 0; i < 2; ++i)
                        bulk_g2s(BT + (size_t)i * part, p.twb + ((size_t)i * p.ng_total + m.g0) * KB * 1024, part, bar_b);
                    if (!mbar_wait_bounded(bar_b, ph_b, p.status)) {
                        mbar_wait_bounded(bar_b, ph_b, p.status, 1u << 20);
                        *aux_fail = 1;
                    }
                }
                ph_b ^= 1u;
                aux_sync();
                if (*aux_fail) break;
                cur_g0 = m.g0;
                cur_ng = m.ng;
            }
            // ---- 3. contraction: issuer aw takes block aw % blocks (directions of
            // one parity, or all) and part aw / blocks of K ----
            const uint32_t cols = (uint32_t)(16 * m.ng);
            const bool dbl = p.n_iss * (int)cols <= 128;
            if (m.flags & kPassFirst) dbuf = dbl ? dbuf ^ 128u : 0u;
            if (pending && !dbl) {   // the columns about to be written hold the tile before
                pending = false;
                if (!epilogue(pend, pend_t, pend_d)) break;
            }
            if (lane == 0) {
                if (aw < p.n_iss) {
                    const int nk = K / 16 / nh;   // K = 16 steps of this issuer
                    const int k0 = (aw / blocks) * nk;
                    const uint32_t idesc = idesc_f16_mk(128, (int)cols, false);
                    const uint32_t d = tmem + kTmemD + dbuf + (uint32_t)aw * cols;
                    const uint32_t a = tmem + kTmemA + (uint32_t)(aw % blocks) * 128u;
                    const uint64_t b = sdesc_sw128(bt_addr, 16u, (uint32_t)KB * 1024u);
                    for (int k = k0; k < k0 + nk; ++k)
                        mma_f16_ta(d, a + (uint32_t)(8 * k), b + (uint64_t)((k >> 2) * 64 + (k & 3) * 2), idesc,
                                   k > k0 || !(m.flags & kPassFirst) ? 1u : 0u);
                    mma_commit(&bar_mma[t & 1]);
                } else {
                    mbar_arrive(&bar_mma[t & 1]);
                }
            }
            __syncwarp();
            // ---- 4. epilogue: of the tile before while these MMAs run when the
            // accumulators are double buffered ----
            if (pending) {
                pending = false;
                ok = epilogue(pend, pend_t, pend_d);
            }
            if (ok && (m.flags & kPassLast)) {
                if (dbl) {
                    pending = true;
                    pend = m;
                    pend_t = t;
                    pend_d = dbuf;
                } else {
                    ok = epilogue(m, t, dbuf);
                }
            }
        }
        if (pending && *aux_fail == 0) epilogue(pend, pend_t, pend_d);
    }
    // teardown
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kHistWarps) tmem_dealloc(tmem, kTmemCols);
}

// ---- wide bands ----------------------------------------------------------------

// Bands of more frequency groups than shared memory holds twiddles for.  A tile is 64
// directions over chunks of at most 1024 bins (2^m <= 1024: one chunk; m = 11, 12: two
// or four) and blocks of at most 2048 atoms; every (block, chunk) pass is contracted
// into the same tensor-memory accumulators.  Per pass:
//   1. histograms by shared-memory atomics, as above;
//   2. an in-place permutation of 16-byte chunks gives the MN-major 128-byte swizzled
//      layout (chunk c of bin row k moves to c ^ (k & 7)): the A operand, M = 128 rows
//      of (64 directions, bin half);
//   3. the chunk's bins split into quarters; the first quarter's twiddles stream from L2
//      through four shared-memory stages, and each stage feeds two MMAs per K step (bin
//      quarters 0 | 2 and 1 | 3);
//   4. after the last pass, warps 0-7 read the accumulators and form X(k) = sum over the
//      quarters with their factors w^(k q NBc / 4), while warps 8-15 zero the histogram.
// The phases run one after the other (7.0, 2.6, 12.7 and 5.4 K cycles at 31 groups, 1133
// atoms and 2^10 bins; 15.0 -> 14.9 ms with the atoms in blocks of four).  The
// pipeline above, with the twiddles streamed under the next tile's histogram, is no
// faster: 16.4-24 ms against 14.9 for 512 ROIs x 40962 directions, k = 8 .. 128.  The
// counts in tensor memory leave 48 KB of shared memory for stages beside the next
// histogram, and every wait of the issuing thread between such small batches of MMAs
// costs 250-500 cycles, with 32 or more of them per tile.
// kNB: band slots of the epilogue (1: the ROI's own band; APTIDX_MAX_BANDS: the pass's
// BandSet, aptidx_compute_signatures_multi)
template <int kNB>
__global__ void __launch_bounds__(kThreads, 1) k_sig_wide(TcParams p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment for the swizzled operands; offset arithmetic on the
    // shared array keeps the pointers in the shared address space
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int NB = 1 << p.m;
    const int NBc = NB < kChunkBins ? NB : kChunkBins;   // bins per chunk
    const int nchunk = NB / NBc;
    uint32_t* H = reinterpret_cast<uint32_t*>(smem);
    unsigned char* BT = smem + (size_t)NBc * 128;
    float* EX = reinterpret_cast<float*>(BT + p.bt_bytes);   // [kDirs][8]
    float4* A = reinterpret_cast<float4*>(BT + p.bt_bytes + kExBytes);
    float4* DB = A + p.atom_cap;   // [2][kDirs]: this tile's directions and the next tile's
    int2* DI = reinterpret_cast<int2*>(DB + 2 * kDirs);   // [2][kDirs]: (output, partner) of those slots
    float* EX2 = reinterpret_cast<float*>(DI + 2 * kDirs);   // [128][8]
    // barriers: [0] atoms, then four stage loads and four stage MMA completions
    constexpr int kBars = 1 + 8;
    uint64_t* bars = reinterpret_cast<uint64_t*>(EX2 + 128 * 8);
    uint64_t* wbar = bars + 1;
    int* flag = reinterpret_cast<int*>(bars + kBars);
    int64_t* item_s = reinterpret_cast<int64_t*>(bars + kBars + 1);
    uint32_t* tmem_s = reinterpret_cast<uint32_t*>(bars + kBars + 2);
    int* iss_ok = reinterpret_cast<int*>(bars + kBars + 3);
    int* prod_ok = iss_ok + 1;
    unsigned* r2max_s = reinterpret_cast<unsigned*>(iss_ok + 2);   // largest |x|^2 of the item's atoms

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int i = 0; i < kBars; ++i) mbar_init(&bars[i], 1);
        fence_barrier_init();
    }
    for (int i = tid; i < NBc * 8; i += kThreads) reinterpret_cast<uint4*>(H)[i] = make_uint4(0, 0, 0, 0);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_s)),
                     "r"(p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_s;
    const uint32_t h_addr = smem_u32(H);
    const uint32_t bt_addr = smem_u32(BT);

    uint32_t ph_atoms = 0;
    uint32_t wph = 0u, wdph = 0u;   // stream parity bits (bit i: buffer i): stage loads (thread 0), stage MMAs (thread 32)
    const float magic = quad_magic(p.m, h_addr >> 7);
    const bool sym = p.slot_idx != nullptr;
    const int64_t n_items = (p.single_roi >= 0 ? 1 : p.nroi) * (int64_t)p.items_per_roi;
    bool failed = false;

    for (;;) {
        if (tid == 0) *item_s = atomicAdd(p.counter, 1);
        __syncthreads();
        const int64_t item = *item_s;
        __syncthreads();
        if (item >= n_items) break;
        const int64_t roi = p.single_roi >= 0 ? p.single_roi : (int64_t)p.order[item / p.items_per_roi];
        const int grp = (int)(item % p.items_per_roi);
        const int nw = p.nw[roi];
        const int64_t abase = p.off[roi];
        const float scale = p.scale[roi];
        const int klo = p.band[2 * roi], khi = p.band[2 * roi + 1];
        const int fg0 = (klo - p.kbase) >> 2, fg1 = (khi - p.kbase) >> 2;
        const int ng = fg1 - fg0 + 1;
        const int t0 = grp * p.tiles_per_item;
        const int t1 = min(t0 + p.tiles_per_item, p.tiles_per_roi);
        const int nblk = max(1, (nw + p.atom_cap - 1) / p.atom_cap);   // atom blocks
        if (nblk == 1) {
            if (tid == 0) *r2max_s = 0u;
            if (!stage_atoms(A, p.atoms + abase, nw, &bars[0], ph_atoms, p.status, flag)) {
                failed = true;
                break;
            }
            quad_atoms(A, nw, tid, kThreads, r2max_s);
        }
        // the first tile's directions (later tiles' arrive while the tile
        // before them runs)
        if (tid < kDirs) {
            cp_async16(DB + (t0 & 1) * kDirs + tid, p.dirs + (int64_t)t0 * kDirs + tid);
            if (sym) cp_async8(DI + (t0 & 1) * kDirs + tid, p.slot_idx + (int64_t)t0 * kDirs + tid);
        }
        cp_async_wait_all();
        __syncthreads();
        // with one atom block and no nonzero integer product possible, the
        // antipodal check only looks for s = 0 (a product per lane instead of
        // an exact count)
        const bool zero_check = sym && nblk == 1 && !nonzero_integer_products_possible(scale, __uint_as_float(*r2max_s));

        for (int tile = t0; tile < t1 && !failed; ++tile) {
            const int cur = tile & 1;
            float4 d0 = DB[cur * kDirs + 2 * lane];
            float4 d1 = DB[cur * kDirs + 2 * lane + 1];
            const int pt0 = sym ? DI[cur * kDirs + 2 * lane].y : -1;
            const int pt1 = sym ? DI[cur * kDirs + 2 * lane + 1].y : -1;
            if (tile + 1 < t1 && tid < kDirs) {
                cp_async16(DB + (cur ^ 1) * kDirs + tid, p.dirs + (int64_t)(tile + 1) * kDirs + tid);
                if (sym) cp_async8(DI + (cur ^ 1) * kDirs + tid, p.slot_idx + (int64_t)(tile + 1) * kDirs + tid);
            }
            int tile_bad = 0;
            for (int pass = 0; pass < 2 && !failed; ++pass) {
                if (pass == 1) {
                    if (!tile_bad) break;
                    // the partners -u of this tile's directions, from their own histograms
                    d0 = make_float4(-d0.x, -d0.y, -d0.z, d0.w);
                    d1 = make_float4(-d1.x, -d1.y, -d1.z, d1.w);
                }
                const bool count = sym && pass == 0;
                uint32_t c0 = 0, c1 = 0;
                float zmin = 1.f;
                QuadDirs q = quad_dirs(d0, d1, scale, magic, lane);
                int handled = 0;
                const int n_sub = nblk * nchunk;
                for (int sub = 0; sub < n_sub && !failed; ++sub) {
                    const int blk = sub / nchunk, bc = sub % nchunk;
                    const int cn = min(p.atom_cap, nw - blk * p.atom_cap);
                    const bool last = sub == n_sub - 1;
                    if (nblk > 1 && bc == 0) {
                        if (!stage_atoms(A, p.atoms + abase + (int64_t)blk * p.atom_cap, cn, &bars[0], ph_atoms,
                                         p.status, flag)) {
                            failed = true;
                            break;
                        }
                        quad_atoms(A, cn, tid, kThreads);
                        __syncthreads();
                    }
                    // ---- 1. histograms (H is zero here) ----
                    if (nchunk == 1) {
                        if (count && zero_check)
                            handled += hist_tile_quads<2, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                        else if (count)
                            handled += hist_tile_quads<1, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                        else
                            hist_tile_quads<0, false>(A, cn, warp, kWarps, q, c0, c1, zmin);
                    } else {
                        q.t_lo = kQuadBits + (h_addr >> 7) + (uint32_t)bc * kChunkBins;
                        q.h_lane = h_addr + 4u * (uint32_t)lane;
                        if (count && bc == 0 && zero_check)
                            handled += hist_tile_quads<2, true>(A, cn, warp, kWarps, q, c0, c1, zmin);
                        else if (count && bc == 0)
                            handled += hist_tile_quads<1, true>(A, cn, warp, kWarps, q, c0, c1, zmin);
                        else
                            hist_tile_quads<0, true>(A, cn, warp, kWarps, q, c0, c1, zmin);
                    }
                    __syncthreads();
                    if (p.hist_out) {
                        hist_export_add(H, NBc, NB, bc, tile, p.nv, p.hist_out, tid, kThreads);
                        __syncthreads();   // every row is read before the permutation moves it
                    }

                    // ---- 2. swizzle: every warp brings bin rows into the MN-major
                    // 128-byte swizzled layout in place (a warp holds four rows, 512
                    // contiguous bytes, one 16-byte chunk per lane, and writes chunk c
                    // of row k to chunk c ^ (k & 7); rows with k & 7 == 0 stay).  The
                    // pass runs at the shared-memory bandwidth; interleaving it with
                    // the MMAs below slows both, so the two run one after the other.
                    // ---- 3. contraction: the twiddles of the first quarter of the
                    // chunk's bins, all the ROI's groups, stream through four
                    // 16 KB shared-memory stages, one per (32-bin K block, hi|lo
                    // part), in the 64-byte-swizzled K-major layout.  Each stage
                    // feeds two M = 128 MMAs per K step: block 0 (rows 0-63 the first
                    // quarter's bins, rows 64-127 the third's) into tensor-memory
                    // columns 8 g .. 8 g + 7 of group g, block 1 (second and fourth
                    // quarters) into the same columns from bo1 on; hi and lo products
                    // accumulate into the same columns, one MMA of N = 8 x groups per
                    // block and K step.  Twiddle row n serves bin n + j NBc / 4 of
                    // quarter j up to the factor w^(f j NBc / 4) the epilogue applies,
                    // so a stage's bytes feed twice the tensor work of the bin-half
                    // split alone.  Thread 0 issues the MMAs as stages land; thread 32
                    // refills a stage once its MMAs are done, three stages ahead.
                    const uint32_t acc0 = sub > 0 ? 1u : 0u;
                    // N = 8 x groups must be a multiple of 16 (M = 128): an odd group
                    // count takes one more group of twiddles (zeros past the last
                    // group), whose columns are never read
                    const int ngw = (ng + 1) & ~1;
                    const uint32_t bo1 = (uint32_t)((8 * ngw + 31) & ~31);   // block 1's first column
                    const uint32_t wbytes = (uint32_t)ngw * 512u;
                    const int KB4 = NBc / 128;      // 32-bin K blocks of the chunk's first quarter
                    const int S = 2 * KB4;          // stages: (block, part)
                    auto wide_load = [&](int s) {   // stage s = 2 x block + part, into buffer s & 3
                        const int kb = s >> 1, part = s & 1, bf = s & 3;
                        mbar_arrive_expect_tx(&wbar[bf], wbytes);
                        bulk_g2s(BT + (size_t)bf * kWideStage,
                                 p.twk + ((((size_t)bc * KB4 + kb) * 2 + part) * (p.ng_total + 1) + fg0) * 512, wbytes,
                                 &wbar[bf]);
                    };
                    if (tid == 0) {
                        // the first stages load while the histogram is swizzled
                        // (the epilogue before wrote the B region through the
                        // generic proxy)
                        fence_proxy_async_smem();
                        for (int st = 0; st < 4; ++st) wide_load(st);
                        *prod_ok = 1;
                    }
                    // two groups of four rows per pass, 64 rows apart (same k & 7;
                    // the chunk's rows are a multiple of 128)
                    for (int r0 = warp * 4; r0 < NBc; r0 += kWarps * 8) {
                        const int k = r0 + (lane >> 3), c = lane & 7, sw = k & 7;
                        uint4* row = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(H) + (size_t)k * 128);
                        uint4* row2 = row + kWarps * 4 * 8;   // row k + 64
                        uint4 x, x2;
                        if (sw) {
                            x = row[c];
                            x2 = row2[c];
                        }
                        __syncwarp();
                        if (sw) {
                            row[c ^ sw] = x;
                            row2[c ^ sw] = x2;
                        }
                    }
                    fence_proxy_async_smem();
                    tc_fence_before();
                    __syncthreads();
                    // A: rows 64-127 (second bin half) one swizzle atom along M
                    // away, NBc / 2 bin rows of 128 bytes
                    const uint64_t a0 = sdesc_sw128(h_addr, (uint32_t)NBc * 64u, 1024u);
                    if (tid == 0) {
                        int ok = 1;
                        // the consumer: MMAs of each stage as it lands
                        tc_fence_after();
                        const uint32_t idw = idesc_f16_mk(kRows, 8 * ngw, true);
                        for (int s = 0; s < S && ok; ++s) {
                            const int kb = s >> 1, bf = s & 3;
                            if (!mbar_wait_bounded(&wbar[bf], (wph >> bf) & 1u, p.status)) {
                                mbar_wait_bounded(&wbar[bf], (wph >> bf) & 1u, p.status, 1u << 20);
                                ok = 0;
                            }
                            wph ^= 1u << bf;
                            if (!ok) break;
                            tc_fence_after();
                            // B: 8 x groups rows (4 frequencies x cos, sin per group) of
                            // 32 bins, 512 bytes per 8 rows; 32 bytes per K step.  A:
                            // block 0 from bin 0, block 1 from bin NBc / 4 (NBc x 32
                            // bytes on), the other half NBc / 2 bins away in both
                            const uint64_t b0 = sdesc_sw64(bt_addr + (uint32_t)bf * kWideStage, 16u, 512u);
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                const uint64_t ad = a0 + (uint64_t)((2 * kb + kk) * 128);
                                const uint64_t bd = b0 + (uint64_t)(kk * 2);
                                const uint32_t acc = (s > 0 || kk > 0) ? 1u : acc0;
                                mma_f16(tmem, ad, bd, idw, acc);
                                mma_f16(tmem + bo1, ad + (uint64_t)(NBc * 2), bd, idw, acc);
                            }
                            mma_commit(&wbar[4 + bf]);
                        }
                        *iss_ok = ok;
                    } else if (tid == 32) {
                        // the producer: a stage's buffer takes the stage four later
                        // once its MMAs are done; then the last four stages' MMAs
                        int pok = 1;
                        for (int s = 4; s < S + 4 && pok; ++s) {
                            const int bf = s & 3;
                            if (!mbar_wait_bounded(&wbar[4 + bf], (wdph >> bf) & 1u, p.status)) {
                                mbar_wait_bounded(&wbar[4 + bf], (wdph >> bf) & 1u, p.status, 1u << 20);
                                pok = 0;
                            }
                            wdph ^= 1u << bf;
                            if (pok && s < S) wide_load(s);
                        }
                        *prod_ok = pok;
                    }
                    // the non-integer counts are complete once the last pass's
                    // histogram is in: a partner whose count falls short of the
                    // atoms this warp handled needs its own histogram
                    const int bad = count && last &&
                                    (zero_check ? (pt0 >= 0 || pt1 >= 0) && zmin == 0.f
                                                : ((pt0 >= 0 && c0 != (uint32_t)handled) ||
                                                   (pt1 >= 0 && c1 != (uint32_t)handled)));
                    const int any_bad = __syncthreads_or(bad);
                    if (last) tile_bad = any_bad;
                    if (!*prod_ok || !*iss_ok) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    if (!last) {
                        // H is read by the MMAs above; zero it for the next pass
                        for (int i = tid; i < NBc * 8; i += kThreads)
                            reinterpret_cast<uint4*>(H)[i] = make_uint4(0, 0, 0, 0);
                        __syncthreads();
                    }
                }
                if (failed) break;

                // ---- 4. epilogue: |X(k)| and the band maximum, warps 0-7; the others
                // zero H for the next tile meanwhile ----
                // pass 0 writes the slot's direction (and its partner
                // when the tile's mirror images are exact); pass 1 the partners
                auto write_out = [&](const float* best, const int* bk, int dir) {
                    const int slot = tile * kDirs + dir;
                    int v0, v1;
                    if (sym) {
                        const int2 si = DI[cur * kDirs + dir];
                        v0 = pass == 0 ? si.x : si.y;
                        v1 = (pass == 0 && !tile_bad) ? si.y : -1;
                    } else {
                        v0 = slot < p.nv ? slot : -1;
                        v1 = -1;
                    }
                    const int64_t rb = (p.single_roi >= 0 ? 0 : roi) * (int64_t)p.nv;
#pragma unroll
                    for (int b = 0; b < kNB; ++b) {
                        if (b < band_count_t<kNB>(p.bands)) {
                            const int64_t ob = band_off_t<kNB>(p.bands, b) + rb;
                            if (v0 >= 0) {
                                p.S[ob + v0] = best[b];
                                if (p.argk) p.argk[ob + v0] = (uint16_t)bk[b];
                            }
                            if (v1 >= 0) {
                                p.S[ob + v1] = best[b];
                                if (p.argk) p.argk[ob + v1] = (uint16_t)bk[b];
                            }
                        }
                    }
                };
                if (warp >= 8) {
                    for (int i = tid - 256; i < NBc * 8; i += kThreads - 256)
                        reinterpret_cast<uint4*>(H)[i] = make_uint4(0, 0, 0, 0);
                } else {
                    // the 64 directions form two groups
                    // (32 p .. 32 p + 31, p = warp & 1); a group's first-half rows are
                    // lane quadrant p (warps p, p + 4), its second-half rows quadrant
                    // 2 + p (warps p + 2, p + 6).  The 4-group column batches split
                    // into four frequency quarters, one per warp of the group
                    // (quarter 0: warp p, 1: p + 4, 2: p + 2, 3: p + 6).  Each warp
                    // first hands the warp of quarter qi ^ 2 (the other bin half)
                    // its own rows of that quarter through the (now idle) B region
                    // as [column][direction], then forms X = D_lo + w^(f h) D_hi over
                    // its quarter and keeps the band maximum of |X|^2 (its root is
                    // the maximum amplitude); quarters 1-3 pass their maxima to
                    // quarter 0 through EX and EX2, which keeps a higher quarter's
                    // value only when strictly greater (lowest-k ties).
                    float best[kNB];
                    int bk[kNB];
                    band_init_t<kNB>(p.bands, klo, best, bk);
                    const int q4 = warp & 3;
                    const uint32_t lane_base = tmem + ((uint32_t)(q4 * 32) << 16);
                    const int dir = (warp & 1) * 32 + lane;
                    const bool first = q4 < 2;                       // first bin half
                    const int qi = (first ? 0 : 2) + (warp >> 2);    // frequency quarter
                    float* xw = reinterpret_cast<float*>(BT);        // [8 x 32 groups][kDirs]
                    const int nb32 = (ng + 3) >> 2;
                    auto qb = [&](int j) { return (j * nb32 + 3) >> 2; };   // quarter j = batches [qb(j), qb(j + 1))
                    const uint32_t bo1 = (uint32_t)((8 * ((ng + 1) & ~1) + 31) & ~31);
                    // columns [c, c + 2 n) of batch b (n frequencies from f0, cos and
                    // sin) over this lane quadrant's bin half: D = D_a + w^(f NBc / 4)
                    // D_b from blocks 0 and 1; w^(f N / 4) = (-i)^f for one chunk,
                    // whose exponent mod 4 follows from kbase mod 4 (a permutation
                    // with signs, fixed per unrolled frequency)
                    auto quarter_add = [&](float* v, const float* u, int n, int f0) {
                        if (nchunk == 1) {
                            switch (p.kbase & 3) {
                                case 0: quarter_rot<0>(v, u, n); break;
                                case 1: quarter_rot<1>(v, u, n); break;
                                case 2: quarter_rot<2>(v, u, n); break;
                                default: quarter_rot<3>(v, u, n); break;
                            }
                        } else {
                            for (int q = 0; q < n; ++q) {
                                float fs, fc;   // w^(f NBc / 4) = fc - i fs
                                sincospif((float)(f0 + q) * (float)NBc / (float)(2 * NB), &fs, &fc);
                                const float ur = u[2 * q], ui = u[2 * q + 1];
                                v[2 * q] += fc * ur - fs * ui;
                                v[2 * q + 1] += fs * ur + fc * ui;
                            }
                        }
                    };
                    for (int b = qb(qi ^ 2); b < qb((qi ^ 2) + 1); ++b) {
                        float v[32], u[32];
                        const uint32_t col = lane_base + (uint32_t)(32 * b);
                        tmem_ld16(col, v);
                        tmem_ld16(col + 16u, v + 16);
                        tmem_ld16(col + bo1, u);
                        tmem_ld16(col + bo1 + 16u, u + 16);
                        tmem_wait_ld();
                        quarter_add(v, u, 16, p.kbase + 4 * (fg0 + 4 * b));
#pragma unroll
                        for (int i = 0; i < 32; ++i) xw[(32 * b + i) * kDirs + dir] = v[i];
                    }
                    asm volatile("bar.sync 1, 256;" ::: "memory");
                    for (int b = qb(qi); b < qb(qi + 1); ++b) {
                        float v[32];
                        {
                            float u[32];
                            const uint32_t col = lane_base + (uint32_t)(32 * b);
                            tmem_ld16(col, v);
                            tmem_ld16(col + 16u, v + 16);
                            tmem_ld16(col + bo1, u);
                            tmem_ld16(col + bo1 + 16u, u + 16);
                            tmem_wait_ld();
                            quarter_add(v, u, 16, p.kbase + 4 * (fg0 + 4 * b));
                        }
                        const int f0 = p.kbase + 4 * (fg0 + 4 * b);
                        const float* xo = xw + 32 * b * kDirs + dir;
                        // the second half's factor w^(f h): (-1)^f for one chunk (a
                        // branch outside the frequency loop, so that the loop carries
                        // no predicated sincos), else cos and sin of pi f h 2 / 2^m
                        if (nchunk == 1) {
                            const float sg0 = (f0 & 1) ? -1.f : 1.f;
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const float orr = xo[(2 * q) * kDirs], ori = xo[(2 * q + 1) * kDirs];
                                const float lr = first ? v[2 * q] : orr, li = first ? v[2 * q + 1] : ori;
                                const float hr = first ? orr : v[2 * q], hs = first ? ori : v[2 * q + 1];
                                const float sg = (q & 1) ? -sg0 : sg0;
                                const float xr = lr + sg * hr, xi = li + sg * hs;
                                band_update_t<kNB>(p.bands, klo, khi, f0 + q, xr * xr + xi * xi, best, bk);
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                const int f = f0 + q;
                                const float orr = xo[(2 * q) * kDirs], ori = xo[(2 * q + 1) * kDirs];
                                const float lr = first ? v[2 * q] : orr, li = first ? v[2 * q + 1] : ori;
                                const float hr = first ? orr : v[2 * q], hs = first ? ori : v[2 * q + 1];
                                float fs, fc;   // w^(f h) = fc - i fs, h = 512
                                sincospif((float)f * (float)NBc / (float)NB, &fs, &fc);
                                const float xr = lr + fc * hr - fs * hs, xi = li + fs * hr + fc * hs;
                                band_update_t<kNB>(p.bands, klo, khi, f, xr * xr + xi * xi, best, bk);
                            }
                        }
                    }
                    // maxima of quarters 1-3: slot ((qi - 1) x 64 + dir) x 8 of EX
                    // (first 512 floats) and EX2
                    auto mx = [&](int qq, int k) -> float& {
                        const int f = ((qq - 1) * kDirs + dir) * 8 + k;
                        return f < kDirs * 8 ? EX[f] : EX2[f - kDirs * 8];
                    };
                    if (qi > 0) {
#pragma unroll
                        for (int b = 0; b < kNB; ++b) {
                            mx(qi, 2 * b) = best[b];
                            mx(qi, 2 * b + 1) = __int_as_float(bk[b]);
                        }
                    }
                    asm volatile("bar.sync 1, 256;" ::: "memory");
                    if (qi == 0) {
#pragma unroll
                        for (int b = 0; b < kNB; ++b) {
                            for (int qq = 1; qq < 4; ++qq) {
                                const float ob = mx(qq, 2 * b);
                                if (ob > best[b]) {
                                    best[b] = ob;
                                    bk[b] = __float_as_int(mx(qq, 2 * b + 1));
                                }
                            }
                            if (best[b] >= 0.f) best[b] = sqrtf(best[b]) * 16777216.0f;
                        }
                        write_out(best, bk, dir);
                    }
                }
                tc_fence_before();
                // the next tile's directions have landed (this thread's copies;
                // the barrier publishes them), H is zero and the accumulators
                // are read before the next pass or tile
                cp_async_wait_all();
                __syncthreads();
                tc_fence_after();
            }
        }
        if (failed) break;
    }
    // teardown: warp 0 frees the tensor memory
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
    }
}

// ---- the global B operand: DFT matrix columns, fp16 hi + lo, K-major SW128 ----

// Narrow bands: the first part's bins n < K (tp_k_rows), layout [hi|lo][group]
// [64-row K block] x 1 KB, 128-byte swizzle (a run of groups is contiguous per
// part).  With `streamed` (wide bands), chunk bc covers bins [bc nbc, bc nbc +
// nbc) with nbc = min(2^m, 1024), the first nbc / 4 of them as K rows: [chunk]
// [32-row K block][hi|lo][group] x 512 B, 64-byte swizzle, with ng + 1 groups per
// run, the last left as the caller's zeros (one K block of one part over a run of
// groups is contiguous).
__global__ void k_build_twb(uint8_t* twb, int m, int kbase, int ng, bool streamed) {
    const int NB = 1 << m;
    const int NBc = NB < kChunkBins ? NB : kChunkBins;
    const int nchunk = NB / NBc;
    const int NK = streamed ? NBc / 4 : tp_k_rows(m);
    const int KB = NK / 64, KBs = NBc / 128;
    const int64_t total = (int64_t)(streamed ? nchunk : 1) * 2 * ng * NK * 8;   // chunks x [hi|lo] x groups x K rows x 8 columns
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(i & 7);
        const int64_t t = i >> 3;
        const int k = (int)(t % NK);
        const int64_t t2 = t / NK;
        const int g = (int)(t2 % ng);
        const int64_t t3 = t2 / ng;
        const int part = (int)(t3 % 2);   // 0 hi, 1 lo
        const int bc = (int)(t3 / 2);
        const int f = kbase + 4 * g + (r >> 1);
        const int64_t n = (int64_t)bc * NBc + k;
        const int jn = (int)(((int64_t)f * n) % NB);
        double sn, cs;
        sincospi(2.0 * (double)jn / (double)NB, &sn, &cs);
        const double v = (r & 1) ? sn : cs;
        const __half hi = __double2half(v);
        const __half lo = __double2half(v - (double)__half2float(hi));
        size_t off;
        if (streamed) {
            const int kb = k >> 5, kin = k & 31;
            const size_t blk = ((size_t)(bc * KBs + kb) * 2 + part) * (ng + 1) + g;
            off = blk * 512 + (size_t)r * 64 + (size_t)(((kin >> 3) ^ ((r >> 1) & 3)) << 4) + (size_t)(kin & 7) * 2;
        } else {
            const int kb = k >> 6, kin = k & 63;
            const size_t blk = (size_t)(part * ng + g) * KB + kb;
            off = blk * 1024 + (size_t)r * 128 + (size_t)(((kin >> 3) ^ r) << 4) + (size_t)(kin & 7) * 2;
        }
        *reinterpret_cast<__half*>(twb + off) = part ? lo : hi;
    }
}

}  // namespace

bool tc_supported(Ctx* c) {
    int major = 0, minor = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, c->device);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, c->device);
    return major == 10 && minor == 3;
}

static size_t tc_smem_bytes(int m, int atom_cap, size_t bt_bytes) {
    const size_t nbc = std::min<size_t>((size_t)1 << m, kChunkBins);
    return 1024 + nbc * 128 + bt_bytes + kExBytes + (size_t)atom_cap * 16 + 2 * kDirs * 16 + 2 * kDirs * 8 +
           128 * 8 * 4 + 256;
}

static size_t tp_smem_bytes(int m, int atom_cap, size_t bt_bytes) {
    const size_t nbc = std::min<size_t>((size_t)1 << m, kChunkBins);
    return 1024 + nbc * 128 + bt_bytes + 2 * kExFloats * 4 + (size_t)atom_cap * 16 + 2 * kDirs * 16 + 2 * sizeof(TpPass) + 128;
}

// Build the B operand for the current ROI bands and pick the TMEM size.
int prepare_tc(Ctx* c) {
    if (!tc_supported(c)) return set_error(c, APTIDX_E_INVALID_ARG, "tensor-core path needs an sm_103 device");
    const int NB = 1 << c->m;
    const int NBc = std::min(NB, kChunkBins);
    const int nchunk = NB / NBc;
    const int KB = tp_k_rows(c->m) / 64;   // 1 KB blocks of 64 K rows
    const int kbase = c->band_min;
    const int ng = (c->band_max - kbase) / 4 + 1;
    // groups whose B operand shared memory holds beside the histogram (32 KB, above
    // 2^10 bins 64 KB) and whose accumulators tensor memory holds for two issuers
    const int gb = std::min(8, (c->m > 10 ? 2 : 1) * kBtBytes / (2 * KB * 1024));
    int ng_roi_max = 1;
    for (int64_t r = 0; r < c->nroi; ++r) {
        const int g0 = (c->h_band[2 * r] - kbase) >> 2, g1 = (c->h_band[2 * r + 1] - kbase) >> 2;
        ng_roi_max = std::max(ng_roi_max, g1 - g0 + 1);
    }
    // wider bands stream their twiddles and accumulate 8 columns per
    // group in each of two blocks (bin quarters 0 and 2, 1 and 3), all groups in
    // one MMA of N = 8 x groups <= 256 per block
    const bool wide = ng_roi_max > gb;
    if (wide && ng_roi_max > 32)
        return set_error(c, APTIDX_E_INVALID_ARG,
                         "tensor-core path: a ROI band spans %d frequency groups (4 frequencies each); at most 32",
                         ng_roi_max);
    // (wide: two blocks of 8 x groups columns, the second from a multiple of 32)
    const int wcols = 8 * ((ng_roi_max + 1) & ~1);
    const uint32_t need = (uint32_t)(((wcols + 31) & ~31) + wcols);
    uint32_t cols = 32;
    while (cols < need) cols <<= 1;
    if (c->twb_key[0] != c->m || c->twb_key[1] != kbase || c->twb_key[2] != ng) {
        dev_free(c->d_twb);
        c->d_twb = nullptr;
        c->twb_key[0] = c->twb_key[1] = c->twb_key[2] = -1;
        // both layouts of the same twiddles: [narrow | streamed (one zero group more per run)]
        const size_t bytes = (size_t)2 * ng * KB * 1024;
        const size_t sbytes = (size_t)nchunk * 2 * (ng + 1) * (NBc / 128) * 512;
        int rc = dev_alloc(c, &c->d_twb, bytes + sbytes);
        if (rc) return rc;
        cudaError_t e0 = cudaMemsetAsync((uint8_t*)c->d_twb + bytes, 0, sbytes, c->stream);
        if (e0 != cudaSuccess) return cuda_check(c, e0, "twiddle operand");
        for (int streamed = 0; streamed < 2; ++streamed) {
            k_build_twb<<<(unsigned)std::min<int64_t>(((int64_t)nchunk * ng * NBc * 8 + 255) / 256, 4096), 256, 0,
                          c->stream>>>((uint8_t*)c->d_twb + streamed * bytes, c->m, kbase, ng, streamed != 0);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_check(c, e, "twiddle operand");
            c->launches += 1;
        }
        c->twb_bytes = bytes;
        c->twb_key[0] = c->m;
        c->twb_key[1] = kbase;
        c->twb_key[2] = ng;
    }
    c->tc_ng = ng;
    c->tc_tmem_cols = cols;
    c->tc_wide = wide;
    c->tc_ng_roi = ng_roi_max;
    return APTIDX_OK;
}

static int tp_tile_dirs(int m) { return kDirs >> std::max(0, m - 10); }

// Tiles per work item when none was tuned: the split of a ROI into items that
// ends first if every CTA takes the same number of items, a set-up (staging and
// arranging the ROI's atoms) counted as a few tiles of a small ROI; at most 64
// tiles.  Few ROIs then spread over every SM (16 ROIs of 81 tiles: 9 tiles per
// item, one wave), many ROIs get long items.
static int tiles_per_item_rule(const Ctx* c, int tiles, int64_t nroi) {
    const double mean = nroi > 0 ? (double)c->atoms_total / (double)c->nroi : 0.0;
    const double setup = 0.3 + 300.0 / (mean + 150.0);   // in tiles
    int best = 1;
    double best_t = 1e300;
    for (int tpi = 1; tpi <= std::min(tiles, 64); ++tpi) {
        const int64_t items = nroi * ((tiles + tpi - 1) / tpi);
        const double t = (double)((items + c->sm_count - 1) / c->sm_count) * (tpi + setup);
        if (t < best_t * 0.999) {
            best_t = t;
            best = tpi;
        }
    }
    return best;
}

int tuned_tiles_per_item(const Ctx* c, int path) {
    if (c->tune_tpi[path] > 0) return c->tune_tpi[path];
    if (path == 0 || c->nroi <= 0) return 16;
    const bool pairs = c->use_pairs && c->d_slot_idx;
    return tiles_per_item_rule(c, (pairs ? c->nslot_pad : c->nv_pad) / (c->tc_wide ? kDirs : tp_tile_dirs(c->m)), c->nroi);
}

cudaError_t launch_signatures_tc(Ctx* c, float* S, uint16_t* argk, uint16_t* hist_out, int64_t hist_roi) {
    cudaError_t e;
    static int max_optin = -1;
    if (max_optin < 0) cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
    const size_t bt_bytes = c->tc_wide ? 4 * (size_t)kWideStage : 32 * (size_t)c->tc_ng_roi * tp_k_rows(c->m);
    const size_t base = c->tc_wide ? tc_smem_bytes(c->m, 0, bt_bytes) : tp_smem_bytes(c->m, 0, bt_bytes);
    int cap = (int)(((size_t)max_optin - base) / 16);
    cap = std::min(cap, kTcMaxAtoms) & ~15;
    if (cap < 256) return cudaErrorInvalidConfiguration;
    const size_t smem = base + (size_t)cap * 16;
    const bool multi = !hist_out && c->multi.n > 0;
    void (*kern)(TcParams);
    if (c->tc_wide)
        kern = multi ? k_sig_wide<APTIDX_MAX_BANDS> : k_sig_wide<1>;
    else if (c->m <= 10)
        kern = multi ? k_sig_tp<APTIDX_MAX_BANDS, 0> : k_sig_tp<1, 0>;
    else if (c->m == 11)
        kern = multi ? k_sig_tp<APTIDX_MAX_BANDS, 1> : k_sig_tp<1, 1>;
    else
        kern = multi ? k_sig_tp<APTIDX_MAX_BANDS, 2> : k_sig_tp<1, 2>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    // antipodal pairs (one projection per pair) unless switched off or exporting
    const bool pairs = !hist_out && c->use_pairs && c->d_slot_idx;
    TcParams p;
    p.atoms = c->d_atoms;
    p.off = c->d_off;
    p.nw = c->d_nw;
    p.order = c->d_order;
    p.dirs = pairs ? c->d_slot_dirs : c->d_dirs;
    p.slot_idx = pairs ? c->d_slot_idx : nullptr;
    p.nv = c->nv;
    p.tiles_per_roi = (pairs ? c->nslot_pad : c->nv_pad) / (c->tc_wide ? kDirs : tp_tile_dirs(c->m));
    p.nroi = c->rank_limit > 0 ? std::min<int64_t>(c->nroi, c->rank_limit) : c->nroi;
    p.tiles_per_item = std::min(c->tune_tpi[1] > 0 ? c->tune_tpi[1]
                                                   : tiles_per_item_rule(c, p.tiles_per_roi, hist_out ? 1 : p.nroi),
                                p.tiles_per_roi);
    p.items_per_roi = (p.tiles_per_roi + p.tiles_per_item - 1) / p.tiles_per_item;
    p.scale = c->d_scale;
    p.band = c->d_band;
    p.m = c->m;
    p.kbase = c->band_min;
    p.twb = (const uint8_t*)c->d_twb;
    p.twk = (const uint8_t*)c->d_twb + c->twb_bytes;
    p.bt_bytes = (int32_t)bt_bytes;
    p.ng_total = c->tc_ng;
    p.tmem_cols = c->tc_tmem_cols;
    p.S = S;
    p.argk = argk;
    p.hist_out = hist_out;
    p.single_roi = hist_out ? hist_roi : -1;
    p.counter = c->d_counter + 2;
    p.status = c->d_status;
    p.atom_cap = cap;
    // four issuers while their accumulators fit (16 columns per group and
    // issuer, 256 in all), else two
    p.n_iss = c->tune_iss >= 4 && c->tc_ng_roi <= 4 ? 4 : 2;
    p.bands = hist_out ? BandSet() : c->multi;
    if ((e = zero_counters(c)) != cudaSuccess) return e;
    // one CTA per SM (registers; the pipelined kernel takes all tensor memory)
    const int64_t items = (hist_out ? 1 : p.nroi) * (int64_t)p.items_per_roi;
    if (items >= ((int64_t)1 << 31) - 4096) return cudaErrorInvalidConfiguration;   // the work counter is 32 bits
    const int64_t grid = std::min<int64_t>((int64_t)c->sm_count, items);
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, c->tc_wide ? kThreads : kTpThreads, smem, c->stream>>>(p);
    c->launches += hist_out ? 0 : 1;
    return cudaGetLastError();
}

}  // namespace aptidx
