// Pair-separation histogram kernels (templates; instantiated per binning
// mode in pairs_*.cu).
//
// Work decomposition of the FP32 kernel (grid traversal of Sect. 2.1 with the
// half-shell duplicate removal of Sect. 3.1): every warp works on its own,
// with no barrier among the warps of a CTA, which share only the histogram.
// A warp takes up to 64 consecutive points of one cell (the i-points, in
// registers: a lane holds one of either half) and walks the candidate j-points of the neighbouring
// cells.  Neighbours are visited row by row: for a stencil row (dy, dz) the
// cells (ax + xlo .. ax + xhi, ay + dy, az + dz) are contiguous in the
// cell-sorted arrays, so each row is one index range (split at most in three
// by periodic wrapping).  Periodic images are handled by shifting whole cells
// (Sect. 3.1), never by testing each pair.  The build stores the bounding box
// of every run of eight points (an oct); the warp tests 32 octs at a time
// against the boxes of its two halves and keeps three lists, octs that reach
// both or only one, staged a batch at a time in its own slice of shared memory.
// Batches of one list need no test in the loop; one half's run with one i-point
// a lane, at half the instructions.
//
// FP32 arithmetic: the j-point is staged as its offset from the i-cell centre,
// rel_j + delta * c, so a pair costs three subtractions and three
// multiply-adds, two j-points per packed instruction.  In-range pairs are
// binned by floors of scaled values (evenly spaced or logarithmic s, evenly
// spaced mu, sigma and pi; Sect. 3.2.2) or through lookup tables for other
// edges (Sect. 3.2.3), each table entry holding the single bin edge near that
// table cell.  The floor paths form a counter's address in FP32 as well and
// send every pair outside the histogram to a discarded entry with one integer
// minimum, so the loop has no branch and no range test.  A pair whose value
// lies within the proven FP32 error band of an edge is checked with the exact
// binary64 definition and its counter corrected if the FP32 bin was another
// one, so the integer counts equal the binary64 definition exactly.
//
// What bounds it (2M clustered points, (s, mu) 40 x 100, 6.70e10 pairs in
// range): issue slots (75 % of the cycles issue; the FMA and integer pipes at 51 and
// 54 %, the shared-memory pipe at 61 %).  1.52 pairs are evaluated for each in range,
// against 1.70 with one list for the 64 points along a Morton curve; 113 of 147 warp
// instructions per 64 x 4 pairs are the loop itself.  Weighted counts of many bins wait
// for bank conflicts of their additions: survey (sigma, pi) with binary64 weights, 86 %
// of the shared-memory pipe, 67 % of its wavefronts conflicts.  65.4 ms against 154.7 ms for
// CTAs of 128 threads that staged every candidate tile behind a barrier and queued
// near-edge pairs for a second kernel (138 instructions per 64 x 2 pairs, issued
// on 60 % of the cycles).
//
// The warps of an SM are spread over all of this code, so its size counts: with a
// second loop body (two quads unrolled) for one half, unrolled staging and an
// unrolled near-edge check, warps waited for instructions longer than for anything
// else (stall 0.1 -> 5.5 an instruction, 312k points 3.2 -> 4.6 ms).  Loops that
// run rarely are rolled.
#pragma once

#include "pc_internal.cuh"

namespace pc {

constexpr unsigned long long FLUSH_LIMIT = 1ull << 30;
// integer weight path: most products (each at most 2^48) in one lane copy's
// record: each of its three u32 piece sums then adds at most 65,535 pieces of
// 16 bits (the top one at most 2^16, with binary64 weights), and the record's
// recombined sum stays below 2^64.
constexpr unsigned WINT_LIMIT = 65535;

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---------------------------------------------------------------------------
// FP32 kernel: shared memory
// ---------------------------------------------------------------------------
constexpr int BI = 64;        // i-points per warp: two halves of 32, one point of each a lane
// j-points per staged batch: 128 (64 is 4 % slower), or 64 where the range of the
// weights' records bounds a batch (bytes: LAY_BYTES) and in the FP64 kernel
__host__ __device__ constexpr int batch_points(int w, bool bytes) { return w == 0 || (w == 2 && bytes) ? 128 : 64; }
constexpr int QCAP = 64;      // near-edge quads kept by a warp before it checks them
constexpr int SEG_G = 97;     // j-segments of a chunk: 32 stencil rows, <= 3 each, and the own cell
constexpr int SEG_T = 33;     // 32 listed tree nodes and the own node

// Byte offsets of a warp's slice: segments, their offsets (tree), the staged
// batch (FP64: coordinates and weight, and the images' shifts), its weights, the
// near-edge queue, the octs to stage, the halves' boxes and the octs before each
// segment.
template <bool TREE, bool WEIGHTED, bool F64, int JB>
struct WarpOff {
    enum {
        jb = JB,
        jo = jb / 8,
        list = jo + 32,                                      // octs kept per class: jo - 1 and a round
        nseg = TREE ? SEG_T : SEG_G,
        soff = nseg * 16,                                    // int4[nseg] before it
        tile = soff + (TREE ? SEG_T * 16 : 0),               // float4[nseg]
        tw = tile + (F64 ? jb * 7 * 8 : 3 * jb * 4),         // x, y, z (+ w, shifts)
        queue = tw + (WEIGHTED && !F64 ? jb * 8 : 0),        // 8 B a point
        ring = (queue + (F64 ? 0 : QCAP * 8) + 15) / 16 * 16,   // uint2[QCAP]
        ibox = ring + 3 * list * 8,                          // uint2[3][list]
        pref = ibox + 64,                                    // IBox[2]
        total = (pref + (nseg + 1) * 4 + 15) / 16 * 16       // int[nseg + 1]
    };
};
inline size_t warp_slice(const PairParams &p) {
    const bool wide = batch_points(!p.weighted ? 0 : (p.wint ? 2 + p.wcorr : 1), p.layout == LAY_BYTES) == 128;
    int n = 0;
    if (p.f64) n = (int)WarpOff<false, false, true, 64>::total;
    else if (!p.weighted) n = p.tree ? (int)WarpOff<true, false, false, 128>::total : (int)WarpOff<false, false, false, 128>::total;
    else if (wide) n = p.tree ? (int)WarpOff<true, true, false, 128>::total : (int)WarpOff<false, true, false, 128>::total;
    else n = p.tree ? (int)WarpOff<true, true, false, 64>::total : (int)WarpOff<false, true, false, 64>::total;
    return (size_t)n;
}

// Histogram layouts (word = 4 bytes; entry (n, m), lane copy k of hist_k):
// (n counts a discarded row first when p.row0 is 1)
//  LAY_ROWS   word (n hs + m) hist_k + k; weights: binary64 sums at the same
//             index, or records of three u32 at 3 x the word
//  LAY_SKEW   word w + w / 32, w = 256 n + m: the bytes of the two fixed-point
//             floors side by side; the skew puts rows 8 banks apart (counts only)
//  LAY_BYTES  word 64 n + k, 32 copies (one axis); weights: the count and a
//             product's lowest piece share that word (the count in its upper 12
//             bits), the next 20 bits add up at + 32 words and the top ones past
//             the last row

__host__ __device__ inline int hist_words(const PairParams &p) {
    if (p.layout == LAY_SKEW) {
        const int w = 256 * (p.n_a + p.row0) + 255;
        return w + w / 32 + 1;
    }
    if (p.layout == LAY_BYTES) return 64 * (p.n_a + p.row0 + 1);
    return p.nent * p.hist_k;
}

// Fill in the layout of a CTA of nw warps: histograms, weight sums, tables (FP64:
// squared edges, and their FP32 roundings when sm_guess says so), the warps'
// slices.  Returns the bytes.
inline size_t cta_layout(PairParams &p, int nw) {
    size_t o = 0;
    if (p.smem_hist_ok) o = align_up(o + (size_t)hist_words(p) * sizeof(int), 16);
    p.sm_whist = (int)o;
    if (p.smem_hist_ok && p.weighted) {   // piece sums, or binary64 sums
        if (p.layout == LAY_BYTES) o += (size_t)hist_words(p) * sizeof(unsigned);
        else o = align_up(o + (size_t)hist_words(p) * (p.wint ? 3 * sizeof(unsigned) : sizeof(double)), 16);
    }
    p.sm_lut = (int)o;
    if (p.f64) {
        const size_t ne = (size_t)(p.n_a + 1) + (size_t)(p.n_b + 1);
        o = align_up(o + ne * (sizeof(double) + (p.sm_guess ? sizeof(float) : 0)), 16);
    } else {
        o = align_up(o + (size_t)p.lut_total * sizeof(float2), 16);
    }
    p.sm_warp = (int)o;
    p.nwarps = nw;
    return o + (size_t)nw * warp_slice(p);
}

// ---------------------------------------------------------------------------
// warp helpers
// ---------------------------------------------------------------------------
constexpr unsigned FULL = 0xffffffffu;

// Order-preserving map of binary32 onto int32 (its own inverse): a < b as
// floats iff fkey(a) < fkey(b) as signed integers.
__device__ __forceinline__ int fkey(float f) {
    const int b = __float_as_int(f);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float fkey_inv(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }
__device__ __forceinline__ float warp_minf(float v) { return fkey_inv(__reduce_min_sync(FULL, fkey(v))); }
__device__ __forceinline__ float warp_maxf(float v) { return fkey_inv(__reduce_max_sync(FULL, fkey(v))); }
__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += t;
    }
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// ---------------------------------------------------------------------------
// shared histogram -> global
// ---------------------------------------------------------------------------
// The counters of an entry's lane copies are read by hist_k consecutive lanes
// and summed with shuffles; the entries (the rows' discarded columns among them,
// the discarded row not) are dealt to warps first, first + nw, ...  A counter is
// taken by an exchange, so a warp can flush what has been added so far while
// others keep adding.
__device__ __forceinline__ int hist_entries(const PairParams &p) {
    return p.layout == LAY_ROWS ? p.n_a * p.hs : p.nbins;
}
__device__ __forceinline__ int hist_word(const PairParams &p, int e, int k, int &bin) {
    bin = e;
    if (p.layout == LAY_SKEW) {
        const int n = e / p.n_b, w = 256 * (n + p.row0) + (e - n * p.n_b);
        return w + (w >> 5);
    }
    if (p.layout == LAY_BYTES) return 64 * (e + p.row0) + k;
    if (p.hs != p.n_b) {
        const int n = e / p.hs, m = e - n * p.hs;
        bin = m < p.n_b ? n * p.n_b + m : -1;
    }
    return (e + p.row0 * p.hs) * p.hist_k + k;
}

static __device__ __noinline__ void flush_counts(const PairParams &p, int first, int nw, int h) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, K = p.hist_k, words = hist_entries(p) * K;
    int *hist = reinterpret_cast<int *>(smem);
    for (int w0 = first * 32; w0 < words; w0 += nw * 32) {
        const int idx = w0 + lane;
        int v = 0, b = -1;
        if (idx < words) {
            const int word = hist_word(p, idx / K, idx & (K - 1), b);
            v = atomicExch(&hist[word], 0);
        }
        for (int o = 1; o < K; o <<= 1) v += __shfl_xor_sync(FULL, v, o);
        if (b >= 0 && (lane & (K - 1)) == 0 && v)
            atomicAdd(&p.hist[(size_t)h * p.nbins + b], (unsigned long long)(long long)v);
    }
}

// Integer weights: a CTA's exact sums of its products by bin (PairParams::wsums),
// two words of value low + high 2^32, both signed, so that additions need no carry
// and return nothing.  A flush adds less than 2^32 to the low word: 2^31 flushes of
// tens of thousands of products fit.  They are converted and scaled once, when the
// CTA is done with a histogram: adding every flush's sum to the binary64 totals
// instead cost 3.9e-12 where 2e10 pairs of equal weights fall in one bin (their
// partial sums round alike), against 3e-16.
__device__ __forceinline__ void add_exact(const PairParams &p, int b, unsigned long long lo, unsigned long long hi) {
    unsigned long long *f = p.wsums + ((size_t)blockIdx.x * p.nbins + b) * 2;
    atomicAdd(&f[0], lo & 0xffffffffull);
    hi += lo >> 32;
    if (hi) atomicAdd(&f[1], hi);
}

// A product that this CTA has added is taken off again.  (Taken off the binary64
// totals, it left their rounding behind: up to 4e-10 in a bin without pairs, for
// 90,000 products of about 0.6 just below its edge.)
__device__ __forceinline__ void sub_exact(const PairParams &p, int b, unsigned long long v) {
    unsigned long long *f = p.wsums + ((size_t)blockIdx.x * p.nbins + b) * 2;
    atomicAdd(&f[0], 0ull - (v & 0xffffffffull));
    atomicAdd(&f[1], 0ull - (v >> 32));
}

// The CTA's exact sums into the global histogram (after a barrier that follows the
// last flush).
__device__ __forceinline__ void flush_exact(const PairParams &p, int h, double wscale) {
    for (int b = threadIdx.x; b < p.nbins; b += blockDim.x) {
        unsigned long long *f = p.wsums + ((size_t)blockIdx.x * p.nbins + b) * 2;
        const long long lo = (long long)atomicExch(&f[0], 0ull);
        const long long hi = (long long)atomicExch(&f[1], 0ull) + (lo >> 32);
        const double w = fma((double)hi, 4294967296.0, (double)(lo & 0xffffffffll));
        if (w != 0.0) atomicAdd(&p.whist[(size_t)h * p.nbins + b], w * wscale);
    }
}

// LAY_BYTES with weights: counts and products of the bins whose fullest record
// holds more than `above` of them (-1: all), four bins a step dealt to warps first,
// first + nw, ...  A lane's records fill unevenly (128 neighbouring j-points are at
// much the same distance): flushing all bins for the fullest of 1,280 records took
// 50 of 340 ms.  Pieces are summed as integers (FP64 shuffles are slow here).
static __device__ __noinline__ void flush_bytes(const PairParams &p, int above, int first, int nw, int h) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    unsigned *hist = reinterpret_cast<unsigned *>(smem) + 64 * p.row0;
    unsigned *top = reinterpret_cast<unsigned *>(smem + p.sm_whist) + 64 * p.row0;
    for (int g = first; 4 * g < p.n_a; g += nw) {
        const int bin = 4 * g + (lane >> 3);
        bool full = false;
        if (bin < p.n_a) {
            const uint4 v = reinterpret_cast<const uint4 *>(hist + 64 * bin)[lane & 7];
            full = (int)(max(max(v.x, v.y), max(v.z, v.w)) >> 20) > above;
        }
        unsigned who = __ballot_sync(FULL, full);
        while (who) {
            const int k = (__ffs(who) - 1) >> 3;
            who &= ~(0xffu << (8 * k));
            const int b = 4 * g + k, word = 64 * b + lane;
            const unsigned v = atomicExch(&hist[word], 0u), mid = atomicExch(&hist[word + 32], 0u),
                           hi = atomicExch(&top[word], 0u);
            const unsigned cnt = __reduce_add_sync(FULL, v >> 20), lo = __reduce_add_sync(FULL, v & 0xFFFFFu);
            const unsigned m0 = __reduce_add_sync(FULL, mid & 0xFFFFu), m1 = __reduce_add_sync(FULL, mid >> 16);
            const unsigned h0 = __reduce_add_sync(FULL, hi & 0xFFFFu), h1 = __reduce_add_sync(FULL, hi >> 16);
            if (lane == 0 && (cnt | lo | m0 | m1 | h0 | h1)) {
                if (cnt) atomicAdd(&p.hist[(size_t)h * p.nbins + b], (unsigned long long)cnt);
                const int sh = 8 + p.wcorr;   // bits of the lowest piece
                const unsigned long long m = m0 + ((unsigned long long)m1 << 16),
                                         t = h0 + ((unsigned long long)h1 << 16);
                // m 2^sh + lo (below 2^47) + t 2^(20 + sh)
                add_exact(p, b, ((m << sh) + lo) + ((t << (20 + sh)) & 0xffffffffull), t >> (12 - sh));
            }
        }
    }
}

// LAY_ROWS with integer weights: every entry's counter and record of products.
//
// Other warps keep adding meanwhile, and may look for full records or flush them
// as well.  A counter must never say less than its record holds (but for the quad
// that each warp is in): it is marked by CLAIM, the record is taken, and only then
// are the mark and the counts that stood there taken off.  Of several warps at an
// entry the first takes the counts; each takes the record, which is thus empty for
// whoever has flushed.  (Taking all counters first and the records after them left
// full records beside counters of zero: a warp that looked then added another
// share, and the sums could wrap.)
constexpr int CLAIM = 1 << 24;   // above any count between flushes
static __device__ __noinline__ void flush_records(const PairParams &p, int first, int nw, int h) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, K = p.hist_k, words = hist_entries(p) * K;
    int *hist = reinterpret_cast<int *>(smem);
    for (int w0 = first * 32; w0 < words; w0 += nw * 32) {
        const int idx = w0 + lane;
        unsigned long long lo = 0ull, hi = 0ull;   // of the record's sum: lower 32 bits and upper
        int b = -1, n = 0;
        if (idx < words) {
            const int word = hist_word(p, idx / K, idx & (K - 1), b);
            unsigned *r = reinterpret_cast<unsigned *>(smem + p.sm_whist) + 3 * (size_t)word;
            // (a record may hold the products of a quad whose counts an earlier flush took)
            volatile const unsigned *v = r;
            if (b >= 0 && (*reinterpret_cast<volatile int *>(hist + word) || (v[0] | v[1] | v[2]))) {
                n = atomicAdd(&hist[word], CLAIM);
                if (n >= CLAIM) n = 0;   // another warp's
                __threadfence_block();
                const unsigned long long r0 = atomicExch(r, 0u), r1 = atomicExch(r + 1, 0u),
                                         r2 = atomicExch(r + 2, 0u);
                lo = r0 + ((r1 & 0xffffull) << 16);
                hi = r2 + (r1 >> 16);
                __threadfence_block();
                atomicSub(&hist[word], CLAIM + n);
            }
        }
        for (int o = 1; o < K; o <<= 1) {
            n += __shfl_xor_sync(FULL, n, o);
            lo += __shfl_xor_sync(FULL, lo, o);
            hi += __shfl_xor_sync(FULL, hi, o);
        }
        if (b >= 0 && (lane & (K - 1)) == 0) {
            if (n) atomicAdd(&p.hist[(size_t)h * p.nbins + b], (unsigned long long)n);
            if (lo | hi) add_exact(p, b, lo, hi);
        }
    }
}

// Binary64 weighted sums.
static __device__ __noinline__ void flush_weights(const PairParams &p, int first, int nw, int h) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, K = p.hist_k, words = hist_entries(p) * K;
    unsigned long long *sums = reinterpret_cast<unsigned long long *>(smem + p.sm_whist);
    for (int w0 = first * 32; w0 < words; w0 += nw * 32) {
        const int idx = w0 + lane;
        double w = 0.0;
        int b = -1;
        if (idx < words) {
            const int word = hist_word(p, idx / K, idx & (K - 1), b);
            w = __longlong_as_double((long long)atomicExch(&sums[word], 0ull));
        }
        for (int o = 1; o < K; o <<= 1) w += __shfl_xor_sync(FULL, w, o);
        if (b >= 0 && (lane & (K - 1)) == 0 && w != 0.0) atomicAdd(&p.whist[(size_t)h * p.nbins + b], w);
    }
}

// Everything a CTA has added, by warps first, first + nw, ...  W as in the kernels.
template <int W>
__device__ __forceinline__ void flush_all(const PairParams &p, int first, int nw, int h) {
    if (W >= 2) {
        if (p.layout == LAY_BYTES) flush_bytes(p, -1, first, nw, h);
        else flush_records(p, first, nw, h);
    } else {
        flush_counts(p, first, nw, h);
        if (W) flush_weights(p, first, nw, h);
    }
}

// Largest counter of a LAY_ROWS histogram with integer weights: no record holds
// more products (but for the quads in flight, flush_records).
static __device__ __noinline__ int most_counted(const PairParams &p) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, rows = p.n_a + p.row0;
    const int words = rows * p.hs * p.hist_k, n4 = words / 4;
    int *hist = reinterpret_cast<int *>(smem);
    // the discarded columns and the discarded first row fill fastest: nobody reads them
    if (p.hs != p.n_b)
        for (int k = lane; k < rows * p.hist_k; k += 32)
            hist[((k / p.hist_k) * p.hs + p.n_b) * p.hist_k + (k & (p.hist_k - 1))] = 0;
    for (int k = lane; k < p.row0 * p.hs * p.hist_k; k += 32) hist[k] = 0;
    constexpr int counts = CLAIM - 1;   // without the marks of warps that flush
    int m = 0;
    for (int k = lane; k < n4; k += 32) {
        const int4 v = reinterpret_cast<const int4 *>(hist)[k];
        m = max(max(m, max(v.x & counts, v.y & counts)), max(v.z & counts, v.w & counts));
    }
    if (4 * n4 + lane < words) m = max(m, hist[4 * n4 + lane] & counts);
    return __reduce_max_sync(FULL, m);
}

// ---------------------------------------------------------------------------
// FP32 binning of one in-range candidate
// ---------------------------------------------------------------------------
// Reciprocal square root: one MUFU.RSQ (PTX rsqrt.approx.ftz.f32, documented
// maximum relative error 2^-22.9; the rescue bands budget 2^-22).  +0 gives
// +inf, so coincident points produce NaN separations and are rescued.
// Base-2 logarithm: one MUFU.LG2 (PTX lg2.approx.ftz.f32).  Its error, at
// most 2.3e-7 max(1, |log2 x|) over every positive normal binary32 input
// (measured exhaustively; the log-bin bands budget 2^-21 max(1, |log2 x|)),
// is checked on the device by the test suite.  +0 gives -inf.
__device__ __forceinline__ float lg2_fast(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rsqrt_fast(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Binning scalars, read from the kernel parameters once and kept in registers.
struct BinCtx {
    const float2 *lutA, *lutB;   // tables in shared memory
    float invA, invB;            // table cells per unit
    unsigned TA1, TB1;           // index of each table's sentinel cell
    float epsA, epsB;            // rescue bands of the two binned quantities
    float muA, muB, muW;         // mu band = muA / s + muB, table window muW
    unsigned nA, nB;
};

struct Bin32 {
    int k, j;    // bin on each axis, valid only if ok
    bool ok;     // falls inside the histogram
    bool near;   // within an error band: needs the binary64 definition
};

__device__ __forceinline__ void lut_locate(const float2 *lut, float inv, unsigned t1, float v,
                                           int &k, float &edge) {
    // v >= 0 by construction; the unsigned clamp also sends any negative
    // index to the always-rescue sentinel cell
    unsigned t = min((unsigned)lut_index(v, inv), t1);
    float2 e = lut[t];
    edge = e.x;
    k = __float_as_int(e.y) + (v >= e.x ? 1 : 0);
}

// Within eps of the table edge (a NaN edge -- several edges in the cell's
// window -- always counts as near).
__device__ __forceinline__ bool is_near(float v, float e, float eps) {
    return !(fabsf(v - e) >= eps);
}

template <int MODE, int LOS>
__device__ __forceinline__ Bin32 bin_f32(const BinCtx &c, float dx, float dy, float dz,
                                         float qxy, float s2, float ax_, float ay_, float az_) {
    Bin32 r;
    if (MODE == MODE_S) {
        float rs = rsqrt_fast(s2);
        float s = s2 * rs;
        int k; float e;
        lut_locate(c.lutA, c.invA, c.TA1, s, k, e);
        r.near = is_near(s, e, c.epsA);
        r.ok = (unsigned)k < c.nA;
        r.k = k;
        r.j = 0;
        return r;
    }
    if (LOS == LOS_Z) {
        if (MODE == MODE_SMU) {
            float rs = rsqrt_fast(s2);
            float s = s2 * rs;
            float mu = fabsf(dz) * rs;
            int k, j; float e, em;
            lut_locate(c.lutA, c.invA, c.TA1, s, k, e);
            lut_locate(c.lutB, c.invB, c.TB1, mu, j, em);
            float epsm = fmaf(c.muA, rs, c.muB);
            r.near = is_near(s, e, c.epsA) || is_near(mu, em, epsm) || (epsm > c.muW);
            r.ok = (unsigned)k < c.nA;
            r.k = k;
            r.j = j;
            return r;
        }
        // (sigma, pi) along z
        float sg = qxy * rsqrt_fast(qxy);
        float pz = fabsf(dz);
        int k, j; float e, ep;
        lut_locate(c.lutA, c.invA, c.TA1, sg, k, e);
        lut_locate(c.lutB, c.invB, c.TB1, pz, j, ep);
        r.near = is_near(sg, e, c.epsA) || is_near(pz, ep, c.epsB);
        r.ok = ((unsigned)k < c.nA) && ((unsigned)j < c.nB);
        r.k = k;
        r.j = j;
        return r;
    }
    // midpoint line of sight: l = 2 x_i + d (ax_ holds 2 x_i)
    float lx = ax_ + dx, ly = ay_ + dy, lz = az_ + dz;
    float sl = fmaf(dz, lz, fmaf(dy, ly, dx * lx));
    float ll = fmaf(lz, lz, fmaf(ly, ly, lx * lx));
    float rl = rsqrt_fast(ll);
    float pi = fabsf(sl) * rl;
    if (MODE == MODE_SMU) {
        float rs = rsqrt_fast(s2);
        float s = s2 * rs;
        float mu = pi * rs;
        int k, j; float e, em;
        lut_locate(c.lutA, c.invA, c.TA1, s, k, e);
        lut_locate(c.lutB, c.invB, c.TB1, mu, j, em);
        float epsm = fmaf(c.muA, rs, c.muB);
        r.near = is_near(s, e, c.epsA) || is_near(mu, em, epsm) || (epsm > c.muW);
        r.ok = (unsigned)k < c.nA;
        r.k = k;
        r.j = j;
        return r;
    }
    // sigma = |d x l| / |l|
    float cxp = fmaf(dy, lz, -dz * ly);
    float cyp = fmaf(dz, lx, -dx * lz);
    float czp = fmaf(dx, ly, -dy * lx);
    float cc = fmaf(czp, czp, fmaf(cyp, cyp, cxp * cxp));
    float sg = cc * rsqrt_fast(cc) * rl;
    int k, j; float e, ep;
    lut_locate(c.lutA, c.invA, c.TA1, sg, k, e);
    lut_locate(c.lutB, c.invB, c.TB1, pi, j, ep);
    r.near = is_near(sg, e, c.epsA) || is_near(pi, ep, c.epsB);
    r.ok = ((unsigned)k < c.nA) && ((unsigned)j < c.nB);
    r.k = k;
    r.j = j;
    return r;
}

// Shared-memory reductions of the weighted sums.
//
// The three 16-bit pieces of an integer weight product p = P >> 16 into one
// lane copy's record {lo, mid, hi} (immediate offsets from one address),
// taken from the 64-bit product P itself: bits 16-31, 32-47 and 48-63.
__device__ __forceinline__ void red_shared_pieces(unsigned addr, unsigned long long P) {
    const unsigned lo = (unsigned)P, hi = (unsigned)(P >> 32);
    asm volatile(
        "red.shared.add.u32 [%0], %1;\n\t"
        "red.shared.add.u32 [%0+4], %2;\n\t"
        "red.shared.add.u32 [%0+8], %3;" ::"r"(addr),
        "r"(lo >> 16), "r"(hi & 0xFFFFu), "r"(hi >> 16));
}
// Integer weight product of a pair with binary64 weights (W == 3), in units of
// the task's wscale: a weight is A + B 2^-31 in units of its grid's scale (A the
// packed 32 bits, B the next 31), the i-point's halved: A' + B' 2^-31.  P = A' A_j
// + 2 t, t = (A' B_j + B' A_j) 2^-32 from the products' high words, is the exact
// product / 2 but for less than 5 (the two truncated high words, the dropped
// B' B_j and the bit B' lost), and V = round(P 2^-15) is non-negative and at most
// 2^48.  All integer: the binary32 remainders this replaces took a conversion
// each way on the slow pipe.
__device__ __forceinline__ unsigned long long corrected_product(unsigned wi, unsigned bi, unsigned wj,
                                                                unsigned bj) {
    const unsigned t = __umulhi(wi, bj) + __umulhi(bi, wj) + 0x2000u;   // below 2^32
    const unsigned long long P = (unsigned long long)t * 2u + (unsigned long long)wi * wj;
    return P >> 15;
}
// The three pieces of V (bits 0-15, 16-31 and 32-48) into one lane copy's
// record, as red_shared_pieces does for P >> 16.
__device__ __forceinline__ void red_shared_pieces_v(unsigned addr, unsigned long long V) {
    const unsigned lo = (unsigned)V, hi = (unsigned)(V >> 32);
    asm volatile(
        "red.shared.add.u32 [%0], %1;\n\t"
        "red.shared.add.u32 [%0+4], %2;\n\t"
        "red.shared.add.u32 [%0+8], %3;" ::"r"(addr),
        "r"(lo & 0xFFFFu), "r"(lo >> 16), "r"(hi));
}
__device__ __forceinline__ void red_shared_f64_if(unsigned addr, double v, bool on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.shared.add.f64 [%0], %1;\n\t}"
        ::"r"(addr), "d"(v), "r"((unsigned)on));
}

__host__ __device__ constexpr bool is_fix(int path) { return path >= PATH_FIX; }

// Two pairs' outcome: byte offset of the counter in the shared histogram
// (PATH_GLOBAL: bin, or ~0u for none), and whether the pair lies within an
// error band of an edge.  A floor path's near pair still gets the counter of
// its FP32 bin (or the discarded one); a table path's gets the discarded one.
struct Pair2 {
    unsigned a0, a1;
    bool n0, n1;
};

// Binning state of a thread (the floor paths' other constants are in the
// kernel parameters).
template <int MODE, int LOS, int PATH>
struct Ctx {
    BinCtx bc;                    // tables
    float2 kA;                    // floor paths: counter address constant, lane copy included
    unsigned trash;               // this thread's discarded counter
    unsigned hk4, copy;           // bytes between counters of consecutive entries; lane copy

    // cp: byte offset of this thread's lane copy
    __device__ __forceinline__ void init(const PairParams &p, const float2 *s_lut, unsigned cp) {
        hk4 = 4u * (unsigned)p.hist_k;
        copy = cp;
        trash = PATH == PATH_GLOBAL ? 0xffffffffu : hk4 * (unsigned)(p.n_a * p.hs) + cp;
        if (PATH == PATH_LUT || PATH == PATH_GLOBAL) {
            bc.lutA = s_lut + p.la.off;
            bc.lutB = s_lut + p.lb.off;
            bc.invA = p.la.inv_w;
            bc.invB = p.lb.inv_w;
            bc.TA1 = (unsigned)(p.la.T + 1);
            bc.TB1 = (unsigned)(p.lb.T + 1);
            bc.epsA = p.eps_a;
            bc.epsB = p.eps_b;
            bc.muA = p.mu_A;
            bc.muB = p.mu_B;
            bc.muW = p.mu_W;
            bc.nA = (unsigned)p.n_a;
            bc.nB = (unsigned)p.n_b;
            return;
        }
        // address of entry (n, m): row n + col m + copy, with g_A = -(n' + 1/2),
        // n' = n (+ 1 with an offset: t carries + 1), g_B = -(m + 1/2): FP32
        // integers below 2^24, so every step is exact
        kA = make_float2(p.c_kA + (float)cp, p.c_kA + (float)cp);
    }
};

// Counter offsets from the floors: n' and m as g = -(floor + 1/2); the FP32
// sum 2^23 + offset holds the offset in its low bits.  Offsets past the last
// row, below the first (they wrap as unsigned) and NaN become the discarded
// counter with one add-and-minimum.
template <class C>
__device__ __forceinline__ void addr2(const C &c, float2 A, Pair2 &o) {
    o.a0 = __viaddmin_u32(__float_as_uint(A.x), 0xB5000000u, c.trash);
    o.a1 = __viaddmin_u32(__float_as_uint(A.y), 0xB5000000u, c.trash);
}

// Bin of entry e of a LAY_ROWS histogram, -1 for a discarded one.
__device__ __forceinline__ int entry_bin(const PairParams &p, int e) {
    if (e >= p.n_a * p.hs) return -1;
    const int row = e / p.hs, col = e - row * p.hs;
    return col < p.n_b ? row * p.n_b + col : -1;
}

// Bins of two pairs (x and y lanes) from their FP32 separations.
//
// Floor of the first axis, t = (s - e_0) / D evaluated as s2 (rsqrt(s2) / D):
// adding 2^23 rounded down leaves floor(t) in the low bits; g = -(floor + 1/2)
// and d = t + g = frac(t) - 1/2 in one fused step, and the pair is near an
// edge unless |d| < 1/2 - band.  With an offset (first edge above zero, and
// logarithmic s) t carries + 1: below 2^23 the FP32 spacing is 1/2, so floors
// are exact only for t >= 0, and everything below -1 is out of range whatever
// its floor.  NaN (s2 = 0) compares false: near.
template <int MODE, int LOS, int PATH>
__device__ __forceinline__ Pair2 bin2(const PairParams &p, const Ctx<MODE, LOS, PATH> &c, float2 dx, float2 dy, float2 dz,
                                      float2 q, float2 s2, float xa, float ya, float za) {
    Pair2 o;
    if (PATH == PATH_LUT || PATH == PATH_GLOBAL) {
        const Bin32 b0 = bin_f32<MODE, LOS>(c.bc, dx.x, dy.x, dz.x, q.x, s2.x, xa, ya, za);
        const Bin32 b1 = bin_f32<MODE, LOS>(c.bc, dx.y, dy.y, dz.y, q.y, s2.y, xa, ya, za);
        const bool in0 = s2.x < p.r2cut, in1 = s2.y < p.r2cut;
        o.n0 = in0 && b0.near;
        o.n1 = in1 && b1.near;
        const bool u0 = in0 && b0.ok && !b0.near, u1 = in1 && b1.ok && !b1.near;
        if (PATH == PATH_GLOBAL) {
            o.a0 = u0 ? (unsigned)(b0.k * (int)c.bc.nB + b0.j) : c.trash;
            o.a1 = u1 ? (unsigned)(b1.k * (int)c.bc.nB + b1.j) : c.trash;
        } else {
            o.a0 = u0 ? c.hk4 * (unsigned)(b0.k * p.hs + b0.j) + c.copy : c.trash;
            o.a1 = u1 ? c.hk4 * (unsigned)(b1.k * p.hs + b1.j) + c.copy : c.trash;
        }
        return o;
    }
    const float2 C23 = p.c_23, CP = p.c_p, M1 = p.c_m1;
    // line-of-sight components (midpoint: l = 2 x_i + d; xa holds 2 x_i)
    float2 pz, rl, lx, ly, lz;
    if (LOS == LOS_MID && MODE != MODE_S) {
        lx = __fadd2_rn(make_float2(xa, xa), dx);
        ly = __fadd2_rn(make_float2(ya, ya), dy);
        lz = __fadd2_rn(make_float2(za, za), dz);
        const float2 sl = __ffma2_rn(dz, lz, __ffma2_rn(dy, ly, __fmul2_rn(dx, lx)));
        const float2 ll = __ffma2_rn(lz, lz, __ffma2_rn(ly, ly, __fmul2_rn(lx, lx)));
        rl = make_float2(rsqrt_fast(ll.x), rsqrt_fast(ll.y));
        pz = make_float2(fabsf(sl.x), fabsf(sl.y));
    } else if (MODE != MODE_S) {
        pz = make_float2(fabsf(dz.x), fabsf(dz.y));
    }
    if (MODE == MODE_SIGPI) {
        // sigma = q rsqrt(q) along z, |d x l| / |l| along the midpoint
        float2 v, rv;
        if (LOS == LOS_Z) {
            v = q;
            rv = __fmul2_rn(make_float2(rsqrt_fast(q.x), rsqrt_fast(q.y)), p.c_invA);
        } else {
            const float2 ndx = __fmul2_rn(dx, M1), ndy = __fmul2_rn(dy, M1), ndz = __fmul2_rn(dz, M1);
            const float2 cx = __ffma2_rn(dy, lz, __fmul2_rn(ndz, ly));
            const float2 cy = __ffma2_rn(dz, lx, __fmul2_rn(ndx, lz));
            const float2 cz = __ffma2_rn(dx, ly, __fmul2_rn(ndy, lx));
            v = __ffma2_rn(cz, cz, __ffma2_rn(cy, cy, __fmul2_rn(cx, cx)));
            const float2 rla = __fmul2_rn(rl, p.c_invA);
            rv = __fmul2_rn(make_float2(rsqrt_fast(v.x), rsqrt_fast(v.y)), rla);
        }
        const float2 rp = LOS == LOS_Z ? p.c_invB : __fmul2_rn(rl, p.c_invB);
        const float2 fa = __ffma2_rd(v, rv, C23), fb = __ffma2_rd(pz, rp, C23);
        const float2 ga = __ffma2_rn(fa, M1, CP), gb = __ffma2_rn(fb, M1, CP);
        const float2 da = __ffma2_rn(v, rv, ga), db = __ffma2_rn(pz, rp, gb);
        o.n0 = !(fabsf(da.x) < p.c_thrA.x) | !(fabsf(db.x) < p.c_cB.x);
        o.n1 = !(fabsf(da.y) < p.c_thrA.y) | !(fabsf(db.y) < p.c_cB.y);
        // pi past its last bin: the discarded column n_b of the row (pi may
        // exceed pi_max while s is still below sqrt(sigma_max^2 + pi_max^2))
        const float lim = 0.5f - (float)p.hs;
        const float2 gc = make_float2(fmaxf(gb.x, lim), fmaxf(gb.y, lim));
        addr2(c, __ffma2_rn(gc, p.c_ncol, __ffma2_rn(ga, p.c_nrow, c.kA)), o);
        return o;
    }
    const float2 rs = make_float2(rsqrt_fast(s2.x), rsqrt_fast(s2.y));
    float2 ga, da;
    if (PATH == PATH_LIN) {
        const float2 ra = __fmul2_rn(rs, p.c_invA);
        const float2 f = __ffma2_rd(s2, ra, C23);
        ga = __ffma2_rn(f, M1, CP);
        da = __ffma2_rn(s2, ra, ga);
    } else {
        const float2 ts = PATH == PATH_LOG
                              ? __ffma2_rn(make_float2(lg2_fast(s2.x), lg2_fast(s2.y)), p.c_invA, p.c_offA)
                              : __ffma2_rn(s2, __fmul2_rn(rs, p.c_invA), p.c_offA);
        const float2 f = __fadd2_rd(ts, C23);
        ga = __ffma2_rn(f, M1, CP);
        da = __fadd2_rn(ts, ga);
    }
    const float2 th = PATH == PATH_LOG ? __ffma2_rn(p.c_nmS, rs, p.c_thrA) : p.c_thrA;
    o.n0 = !(fabsf(da.x) < th.x);
    o.n1 = !(fabsf(da.y) < th.y);
    float2 A = __ffma2_rn(ga, p.c_nrow, c.kA);
    if (MODE == MODE_SMU) {
        // t_mu = mu n_mu, scaled just below n_mu: mu = 1 is in the last bin
        const float2 rm = LOS == LOS_Z ? __fmul2_rn(rs, p.c_invB) : __fmul2_rn(__fmul2_rn(rl, rs), p.c_invB);
        const float2 f = __ffma2_rd(pz, rm, C23);
        const float2 gm = __ffma2_rn(f, M1, CP);
        const float2 dm = __ffma2_rn(pz, rm, gm);
        const float2 tm = __ffma2_rn(p.c_nmB, rs, p.c_cB);
        o.n0 = o.n0 | !(fabsf(dm.x) < tm.x);
        o.n1 = o.n1 | !(fabsf(dm.y) < tm.y);
        A = __ffma2_rn(gm, p.c_ncol, A);
    }
    addr2(c, A, o);
    return o;
}

// A warp's i-points: lane l holds point l of either half of the block.
template <int LOS, int W>
struct IPts {
    float x[2], y[2], z[2];        // offsets from the i-cell centre (far away if unused)
    float xa[2], ya[2], za[2];     // twice the absolute positions (midpoint line of sight)
    double w[2];                   // W == 1
    unsigned wm[2];                // W >= 2: packed integer weight
    unsigned wb[2];                // W == 3: wm halved and the next 31 bits
};

// The second half's points where the first's are (batches of that half alone).
template <int MODE, int LOS, int W>
__device__ __forceinline__ IPts<LOS, W> half_points(const IPts<LOS, W> &I, bool second) {
    IPts<LOS, W> o = I;
    if (second) {
        o.x[0] = I.x[1]; o.y[0] = I.y[1]; o.z[0] = I.z[1];
        if (LOS == LOS_MID && MODE != MODE_S) { o.xa[0] = I.xa[1]; o.ya[0] = I.ya[1]; o.za[0] = I.za[1]; }
        if (W == 1) o.w[0] = I.w[1];
        if (W >= 2) o.wm[0] = I.wm[1];
        if (W == 3) o.wb[0] = I.wb[1];
    }
    return o;
}

// One i-point's registers from its record (the midpoint sums start from 2 x_i:
// doubling is exact, so 2 x_i + d rounds once, as a fused multiply-add would).
template <int MODE, int LOS, int W>
__device__ __forceinline__ void load_i(const GridDev &g, int i, IPts<LOS, W> &I, int r) {
    const float4 q = g.rel[i];
    I.x[r] = q.x; I.y[r] = q.y; I.z[r] = q.z;
    if (W >= 2) I.wm[r] = __float_as_uint(q.w);
    if (W == 3) {
        const unsigned B = g.wlo ? g.wlo[i] : 0u;
        I.wb[r] = (I.wm[r] & 1u) << 30 | B >> 1;
        I.wm[r] >>= 1;
    }
    if ((LOS == LOS_MID && MODE != MODE_S) || W == 1) {
        const double4_32a a = g.xw[i];
        I.xa[r] = 2.0f * (float)a.x; I.ya[r] = 2.0f * (float)a.y; I.za[r] = 2.0f * (float)a.z;
        if (W == 1) I.w[r] = a.w;
    }
}

// A j-point in the i-cell's frame: grid, rel_j + delta c (delta the offset of
// the cells, periodic image included); tree, rel_j + o (o the offset of the
// two node centres).
__device__ __forceinline__ float3 stage_grid(const PairParams &p, float4 q, int cx, int ax, int meta, int img) {
    const int dxc = cx - ax + (img / 9 - 1) * p.g.ng[0];
    const int dyc = (int)(short)(meta & 0xFFFF), dzc = meta >> 16;
    return make_float3(fmaf((float)dxc, p.g.c32[0], q.x), fmaf((float)dyc, p.g.c32[1], q.y),
                       fmaf((float)dzc, p.g.c32[2], q.z));
}
__device__ __forceinline__ float4 tree_offset(const PairParams &p, int inode, int jnode, int img) {
    const double *ci = p.tcen_i + 3 * (size_t)inode, *cj = p.tcen_j + 3 * (size_t)jnode;
    const double sx = (double)(img / 9 - 1), sy = (double)((img / 3) % 3 - 1), sz = (double)(img % 3 - 1);
    return make_float4(__double2float_rn(__dsub_rn(__dadd_rn(cj[0], __dmul_rn(sx, p.g.L[0])), ci[0])),
                       __double2float_rn(__dsub_rn(__dadd_rn(cj[1], __dmul_rn(sy, p.g.L[1])), ci[1])),
                       __double2float_rn(__dsub_rn(__dadd_rn(cj[2], __dmul_rn(sz, p.g.L[2])), ci[2])), 0.f);
}

// The staged batch of j-points in a warp's slice.
struct Tile {
    const float *x, *y, *z;
    const double *w;               // W == 1
    const unsigned *wm;            // W >= 2 (same storage)
    const unsigned *wl;            // W == 3: the next 31 bits, after wm
};

// All pairs of the warp's i-points with nq quads of staged j-points: per
// iteration four j-points x R i-points a lane, in packed FP32, every
// counter updated by the full warp (pairs outside the histogram go to the
// discarded counter).  Returns a bit per quad: some pair of this lane is near
// an edge.  MASK: the tile holds points jbase, jbase + 1, ... of the i-block
// itself and only pairs j > i count.
template <int MODE, int LOS, int W, int PATH, bool MASK, int R>
__device__ __forceinline__ unsigned pair_quads(const PairParams &p, const Tile &t, int nq,
                                               const IPts<LOS, W> &I, const Ctx<MODE, LOS, PATH> &c,
                                               unsigned char *hist, unsigned wbase, int jbase, int me,
                                               size_t hbase) {
    const int lane = threadIdx.x & 31;
    unsigned near = 0u;
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
        const float4 X = reinterpret_cast<const float4 *>(t.x)[q];
        const float4 Y = reinterpret_cast<const float4 *>(t.y)[q];
        const float4 Z = reinterpret_cast<const float4 *>(t.z)[q];
        bool any = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 Xh = h ? make_float2(X.z, X.w) : make_float2(X.x, X.y);
            const float2 Yh = h ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y);
            const float2 Zh = h ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float2 dx = __fadd2_rn(Xh, make_float2(-I.x[r], -I.x[r]));
                const float2 dy = __fadd2_rn(Yh, make_float2(-I.y[r], -I.y[r]));
                const float2 dz = __fadd2_rn(Zh, make_float2(-I.z[r], -I.z[r]));
                if (MASK) {   // masked pairs: far out of range
                    const int jj = jbase + 4 * q + 2 * h;
                    if (jj <= me) dx.x = p.far;
                    if (jj + 1 <= me) dx.y = p.far;
                }
                const float2 qq = __ffma2_rn(dy, dy, __fmul2_rn(dx, dx));
                const float2 s2 = __ffma2_rn(dz, dz, qq);
                const Pair2 b = bin2<MODE, LOS, PATH>(p, c, dx, dy, dz, qq, s2, I.xa[r], I.ya[r], I.za[r]);
                any = any | b.n0 | b.n1;
                if (PATH == PATH_GLOBAL) {
                    if (b.a0 != c.trash) atomicAdd(p.hist + hbase + b.a0, 1ull);
                    if (b.a1 != c.trash) atomicAdd(p.hist + hbase + b.a1, 1ull);
                    if (W == 1) {
                        if (b.a0 != c.trash)
                            atomicAdd(p.whist + hbase + b.a0, __dmul_rn(I.w[r], t.w[4 * q + 2 * h]));
                        if (b.a1 != c.trash)
                            atomicAdd(p.whist + hbase + b.a1, __dmul_rn(I.w[r], t.w[4 * q + 2 * h + 1]));
                    }
                    continue;
                }
                atomicAdd(reinterpret_cast<unsigned *>(hist + b.a0), 1u);
                atomicAdd(reinterpret_cast<unsigned *>(hist + b.a1), 1u);
                if (W == 1) {   // near pairs are added by their binary64 check
                    const double2 wj = *reinterpret_cast<const double2 *>(t.w + 4 * q + 2 * h);
                    red_shared_f64_if(wbase + 2u * b.a0, __dmul_rn(I.w[r], wj.x), b.a0 < c.trash && !b.n0);
                    red_shared_f64_if(wbase + 2u * b.a1, __dmul_rn(I.w[r], wj.y), b.a1 < c.trash && !b.n1);
                } else if (W == 2) {
                    // (M_i M_j) >> (k_i + k_j), k = emax - e the exponent offset:
                    // the packed M 2^(8 - k) multiplied exactly in 64 bits is
                    // P = M_i M_j 2^(16 - k_i - k_j), and the product is P >> 16
                    // (truncation < 2^(k_i + k_j - 46) relative, below 2^48).  A
                    // record is 12 bytes and has the count's place among them
                    const uint2 wj = *reinterpret_cast<const uint2 *>(t.wm + 4 * q + 2 * h);
                    red_shared_pieces(wbase + 3u * b.a0, (unsigned long long)I.wm[r] * wj.x);
                    red_shared_pieces(wbase + 3u * b.a1, (unsigned long long)I.wm[r] * wj.y);
                } else if (W == 3) {
                    const uint2 wj = *reinterpret_cast<const uint2 *>(t.wm + 4 * q + 2 * h);
                    const uint2 lj = *reinterpret_cast<const uint2 *>(t.wl + 4 * q + 2 * h);
                    red_shared_pieces_v(wbase + 3u * b.a0,
                                        corrected_product(I.wm[r], I.wb[r], wj.x, lj.x));
                    red_shared_pieces_v(wbase + 3u * b.a1,
                                        corrected_product(I.wm[r], I.wb[r], wj.y, lj.y));
                }
            }
        }
        near |= (any ? 1u : 0u) << q;
    }
    return near;
}

// ---------------------------------------------------------------------------
// fixed-point floors (PATH_FIX)
// ---------------------------------------------------------------------------
// For at most FIX_TOP bins an axis, a scaled value t (s / D, log_q(s / e_0), mu
// n_mu, sigma / D, pi / D) is added to 128 + B 2^-16 in one fused multiply-add.
// FP32 numbers in [128, 256) are multiples of 2^-16: byte 2 of the sum is
// floor(t + B 2^-16) and its low half the 16-bit fraction.  B is the error band
// in these units (the arithmetic's bound and the sum's own rounding, rounded
// up), so the pair is near an edge iff the fraction is below 2 B, and otherwise
// the byte is its bin.  One three-input minimum of 16-bit halves covers two
// values of the near test (the upper halves ride along unused), one byte
// permutation puts the two bins side by side as the counter's index, and values
// past the last bin are clamped to half a bin past it: the discarded row (pi:
// column), never near.  With a first edge above zero (PATH_FIXOFF, PATH_FIXLOG) t
// carries + 1 and is clamped below to half a bin, another discarded row.  mu n_mu
// has no shrunken scale: mu = 1 lands in column n_mu, is near, and is put right
// by its binary64 check.  A tiny constant added to the squares keeps coincident
// points finite.  Bands that grow as 1 / s (mu, logarithms) are taken at the
// batch's smallest separation, from the boxes' gap.  Every index stays inside
// the histogram: coordinates are finite and below 1e16 (others count as absent;
// the host limits the extents to 1e15, so no square overflows), hence 128 <= T <
// n_a + 130 and 128 <= M < 256.
//
// Against the packed floors of bin2 this leaves 40 of 68 packed FP32
// instructions a quad (their three-register forms cost three register-read
// cycles each); measured on the loop alone, (s, mu) 40 x 100: 161 against 224
// cycles a quad and scheduler, one axis 121 against 147.
// Whole kernel: 300,001 points, 40 logarithmic s bins x 100 mu bins 4.44 -> 3.40
// ms against the packed floors; 10^6 points, 20 logarithmic sigma x 60 pi bins
// 4.58 -> 2.70 ms against the tables.
__device__ __forceinline__ unsigned prmt(unsigned a, unsigned b, unsigned s) {
    unsigned d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(s));
    return d;
}

// The three 16-bit pieces of P >> 16, taken from P; of V (the top one 17 bits).
__device__ __forceinline__ uint3 pieces(unsigned long long P) {
    const unsigned lo = (unsigned)P, hi = (unsigned)(P >> 32);
    return make_uint3(lo >> 16, hi & 0xFFFFu, hi >> 16);
}
__device__ __forceinline__ uint3 pieces_v(unsigned long long V) {
    const unsigned lo = (unsigned)V;
    return make_uint3(lo & 0xFFFFu, lo >> 16, (unsigned)(V >> 32));
}
__device__ __forceinline__ void add_pieces(unsigned char *a0, unsigned char *a1, unsigned char *a2, uint3 v) {
    atomicAdd(reinterpret_cast<unsigned *>(a0), v.x);
    atomicAdd(reinterpret_cast<unsigned *>(a1), v.y);
    atomicAdd(reinterpret_cast<unsigned *>(a2), v.z);
}

// The words of a LAY_BYTES record that a product adds to: 1 << 20 | its lowest 8
// bits (of P >> 16; 9 of V), the next 20 bits, the top 20.  Three shared additions
// a pair instead of four, for 4,095 products a record between flushes (2,047).
__device__ __forceinline__ uint3 packed_p(unsigned long long P) {
    const unsigned lo = (unsigned)P, hi = (unsigned)(P >> 32);
    return make_uint3(prmt(lo, 0x00100000u, 0x7642), __funnelshift_r(lo, hi, 24) & 0xFFFFFu, hi >> 12);
}
__device__ __forceinline__ uint3 packed_v(unsigned long long V) {
    const unsigned lo = (unsigned)V, hi = (unsigned)(V >> 32);
    return make_uint3((lo & 0x1FFu) | 0x100000u, __funnelshift_r(lo, hi, 9) & 0xFFFFFu, __funnelshift_r(lo, hi, 29));
}

// A batch's constants, from a 16-bit lower bound of its separations' square (the
// upper half of the FP32 number; 0: none).
struct Bands {
    float2 cfs;          // first axis: 128 (+ 1 - offset) + band
    float cfm;           // second axis
    unsigned ts2, tm2;   // twice the bands, in units
    float close;         // (s, mu): below it a pair is near whatever its mu
};
template <int MODE, int PATH>
__device__ __forceinline__ Bands fix_bands(const PairParams &p, unsigned key) {
    Bands b;
    const float s2m = __uint_as_float(key << 16);
    b.cfs = p.f_cfs;
    b.ts2 = p.f_ts2;
    b.cfm = p.f_cfp;
    b.tm2 = p.f_tp2;
    if (PATH == PATH_FIXLOG) {
        const unsigned n = __float2uint_ru(fmaf(p.f_sA, rsqrt_fast(fmaxf(s2m, p.f_se2)), p.f_sC));
        const float c = fmaf((float)n, 1.0f / 65536.0f, p.f_cfs.x);
        b.cfs = make_float2(c, c);
        b.ts2 = 2u * n;
    }
    if (MODE == MODE_SMU) {
        const unsigned n = __float2uint_ru(fmaf(p.f_mA, rsqrt_fast(fmaxf(s2m, p.f_sf2)), p.f_mB));
        b.cfm = fmaf((float)n, 1.0f / 65536.0f, 128.0f);
        b.tm2 = 2u * n;
    }
    b.close = fmaf((float)b.ts2, 1.0f / 65536.0f, p.f_close);
    return b;
}

struct Fix2 {
    float2 T, M;   // first axis (clamped) and second axis, in fixed point
};

template <int MODE, int LOS, int PATH>
__device__ __forceinline__ Fix2 fix2(const PairParams &p, float2 dx, float2 dy, float2 dz, float2 cfs, float2 cfm,
                                     float xa, float ya, float za, float2 &s2) {
    Fix2 o;
    float2 pz, rl, lx, ly, lz;
    const float2 q = __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, p.f_tiny));
    s2 = __ffma2_rn(dz, dz, q);
    if (LOS == LOS_MID && MODE != MODE_S) {   // l = 2 x_i + d
        lx = __fadd2_rn(make_float2(xa, xa), dx);
        ly = __fadd2_rn(make_float2(ya, ya), dy);
        lz = __fadd2_rn(make_float2(za, za), dz);
        const float2 sl = __ffma2_rn(dz, lz, __ffma2_rn(dy, ly, __fmul2_rn(dx, lx)));
        const float2 ll = __ffma2_rn(lz, lz, __ffma2_rn(ly, ly, __ffma2_rn(lx, lx, p.f_tiny)));
        rl = make_float2(rsqrt_fast(ll.x), rsqrt_fast(ll.y));
        pz = make_float2(fabsf(sl.x), fabsf(sl.y));
    } else if (MODE != MODE_S) {
        pz = make_float2(fabsf(dz.x), fabsf(dz.y));
    }
    float2 T;
    if (MODE == MODE_SIGPI) {
        float2 v = q;
        if (LOS == LOS_MID) {   // sigma = |d x l| / |l|
            const float2 M1 = p.c_m1;
            const float2 ndx = __fmul2_rn(dx, M1), ndy = __fmul2_rn(dy, M1), ndz = __fmul2_rn(dz, M1);
            const float2 cx = __ffma2_rn(dy, lz, __fmul2_rn(ndz, ly));
            const float2 cy = __ffma2_rn(dz, lx, __fmul2_rn(ndx, lz));
            const float2 cz = __ffma2_rn(dx, ly, __fmul2_rn(ndy, lx));
            v = __ffma2_rn(cz, cz, __ffma2_rn(cy, cy, __ffma2_rn(cx, cx, p.f_tiny)));
        }
        if (PATH == PATH_FIXLOG) {
            if (LOS == LOS_MID) v = __fmul2_rn(__fmul2_rn(v, rl), rl);
            T = __ffma2_rn(make_float2(lg2_fast(v.x), lg2_fast(v.y)), p.c_invA, cfs);
        } else {
            float2 rv = make_float2(rsqrt_fast(v.x), rsqrt_fast(v.y));
            rv = __fmul2_rn(rv, LOS == LOS_Z ? p.c_invA : __fmul2_rn(rl, p.c_invA));
            T = __ffma2_rn(v, rv, cfs);
        }
        const float2 M = __ffma2_rn(pz, LOS == LOS_Z ? p.c_invB : __fmul2_rn(rl, p.c_invB), cfm);
        o.M = make_float2(fminf(M.x, p.f_limB), fminf(M.y, p.f_limB));
    } else {
        float2 rs;
        if (PATH != PATH_FIXLOG || MODE == MODE_SMU) rs = make_float2(rsqrt_fast(s2.x), rsqrt_fast(s2.y));
        if (PATH == PATH_FIXLOG)
            T = __ffma2_rn(make_float2(lg2_fast(s2.x), lg2_fast(s2.y)), p.c_invA, cfs);
        else
            T = __ffma2_rn(s2, __fmul2_rn(rs, p.c_invA), cfs);
        if (MODE == MODE_SMU)
            o.M = __ffma2_rn(pz, LOS == LOS_Z ? __fmul2_rn(rs, p.c_invB)
                                              : __fmul2_rn(__fmul2_rn(rl, rs), p.c_invB), cfm);
    }
    if (PATH != PATH_FIX) T = make_float2(fmaxf(T.x, 128.5f), fmaxf(T.y, 128.5f));
    o.T = make_float2(fminf(T.x, p.f_lim), fminf(T.y, p.f_lim));
    return o;
}

// All pairs of the warp's i-points with nq quads of staged j-points, as
// pair_quads.  SLOW: batches that may hold pairs closer than the separation the
// mu band is taken at (T below f_close: near), and the block's own points (the
// tile holds its points from jbase on, pairs j <= i are masked; jbase past any
// i: none is).
template <int MODE, int LOS, int W, int PATH, bool SLOW, int R>
__device__ __forceinline__ unsigned quads_fix(const PairParams &p, const Tile &t, int nq, const IPts<LOS, W> &I,
                                              unsigned char *smem, const Bands &bd, int jbase, int me) {
    const int lane = threadIdx.x & 31;
    const float2 cfm = make_float2(bd.cfm, bd.cfm);
    const unsigned copy = 4u * (unsigned)lane;                 // LAY_BYTES
    const unsigned kc = (unsigned)(lane & (p.hist_k - 1));    // LAY_ROWS
    unsigned *hist = reinterpret_cast<unsigned *>(smem);
    unsigned near = 0u;
    // two quads an iteration only where the code stays small (instruction cache)
    constexpr int UNROLL = R == 1 || W || (LOS == LOS_MID && MODE != MODE_S) ? 1 : 2;
#pragma unroll UNROLL
    for (int q = 0; q < nq; ++q) {
        const float4 X = reinterpret_cast<const float4 *>(t.x)[q];
        const float4 Y = reinterpret_cast<const float4 *>(t.y)[q];
        const float4 Z = reinterpret_cast<const float4 *>(t.z)[q];
        unsigned accT = 0xffffffffu, accM = 0xffffffffu;
        bool close = false;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 Xh = h ? make_float2(X.z, X.w) : make_float2(X.x, X.y);
            const float2 Yh = h ? make_float2(Y.z, Y.w) : make_float2(Y.x, Y.y);
            const float2 Zh = h ? make_float2(Z.z, Z.w) : make_float2(Z.x, Z.y);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float2 dx = __fadd2_rn(Xh, make_float2(-I.x[r], -I.x[r]));
                const float2 dy = __fadd2_rn(Yh, make_float2(-I.y[r], -I.y[r]));
                const float2 dz = __fadd2_rn(Zh, make_float2(-I.z[r], -I.z[r]));
                if (SLOW) {   // masked pairs: far out of range
                    const int jj = jbase + 4 * q + 2 * h;
                    if (jj <= me) dx.x = p.far;
                    if (jj + 1 <= me) dx.y = p.far;
                }
                float2 s2;
                const Fix2 f = fix2<MODE, LOS, PATH>(p, dx, dy, dz, bd.cfs, cfm, I.xa[r], I.ya[r], I.za[r], s2);
                const unsigned t0 = __float_as_uint(f.T.x), t1 = __float_as_uint(f.T.y);
                accT = __vimin3_u16x2(accT, t0, t1);
                if (SLOW && MODE == MODE_SMU) close = close | (f.T.x < bd.close) | (f.T.y < bd.close);
                unsigned P0 = 0u, P1 = 0u;   // W >= 2: addresses of the pieces' records
                if (MODE == MODE_S) {
                    // byte 1: the bin, byte 0: this lane's copy
                    const unsigned a0 = prmt(t0, copy, 0x5524), a1 = prmt(t1, copy, 0x5524);
                    if (W == 0) {
                        atomicAdd(reinterpret_cast<unsigned *>(smem + a0), 1u);
                        atomicAdd(reinterpret_cast<unsigned *>(smem + a1), 1u);
                    }
                    P0 = a0;
                    P1 = a1;
                } else {
                    const unsigned m0 = __float_as_uint(f.M.x), m1 = __float_as_uint(f.M.y);
                    accM = __vimin3_u16x2(accM, m0, m1);
                    // 256 n + m from the two bytes (the sign bit of byte 2 is 0)
                    const unsigned w0 = prmt(m0, t0, 0xAA62), w1 = prmt(m1, t1, 0xAA62);
                    if (W == 0) {
                        atomicAdd(&hist[w0 + (w0 >> 5)], 1u);
                        atomicAdd(&hist[w1 + (w1 >> 5)], 1u);
                    } else {   // LAY_ROWS
                        P0 = __dp4a(w0, p.f_coef, kc);   // (n hs + m) hist_k + copy
                        P1 = __dp4a(w1, p.f_coef, kc);
                        atomicAdd(&hist[P0], 1u);
                        atomicAdd(&hist[P1], 1u);
                    }
                }
                if (W >= 2) {
                    // (M_i M_j) >> (k_i + k_j), k = emax - e the exponent offset:
                    // the packed M 2^(8 - k) multiplied exactly in 64 bits is
                    // P = M_i M_j 2^(16 - k_i - k_j), and the product is P >> 16
                    // (truncation < 2^(k_i + k_j - 46) relative, below 2^48)
                    const uint2 wj = *reinterpret_cast<const uint2 *>(t.wm + 4 * q + 2 * h);
                    uint3 v0, v1;   // pieces, lowest first
                    if (W == 2) {
                        const unsigned long long p0 = (unsigned long long)I.wm[r] * wj.x,
                                                 p1 = (unsigned long long)I.wm[r] * wj.y;
                        v0 = MODE == MODE_S ? packed_p(p0) : pieces(p0);
                        v1 = MODE == MODE_S ? packed_p(p1) : pieces(p1);
                    } else {
                        const uint2 lj = *reinterpret_cast<const uint2 *>(t.wl + 4 * q + 2 * h);
                        const unsigned long long p0 = corrected_product(I.wm[r], I.wb[r], wj.x, lj.x),
                                                 p1 = corrected_product(I.wm[r], I.wb[r], wj.y, lj.y);
                        v0 = MODE == MODE_S ? packed_v(p0) : pieces_v(p0);
                        v1 = MODE == MODE_S ? packed_v(p1) : pieces_v(p1);
                    }
                    if (MODE == MODE_S) {
                        add_pieces(smem + P0, smem + P0 + 128, smem + P0 + p.sm_whist, v0);
                        add_pieces(smem + P1, smem + P1 + 128, smem + P1 + p.sm_whist, v1);
                    } else {
                        unsigned char *r0 = smem + p.sm_whist + 12 * P0, *r1 = smem + p.sm_whist + 12 * P1;
                        add_pieces(r0, r0 + 4, r0 + 8, v0);
                        add_pieces(r1, r1 + 4, r1 + 8, v1);
                    }
                }
            }
        }
        bool any = (accT & 0xffffu) < bd.ts2;
        if (MODE != MODE_S) any = any | ((accM & 0xffffu) < bd.tm2);
        if (SLOW) any = any | close;
        near |= (any ? 1u : 0u) << q;
    }
    return near;
}

// Two pairs' bins and near flags from their fixed-point values (the near-edge
// check repeats the loop's arithmetic with them); bin -1: discarded.
template <int MODE, int PATH>
__device__ __forceinline__ int fix_bin(const PairParams &p, float T, float M, const Bands &b, bool &near) {
    const unsigned t = __float_as_uint(T), m = MODE == MODE_S ? 0u : __float_as_uint(M);
    near = (t & 0xffffu) < b.ts2;
    if (MODE != MODE_S) near = near || (m & 0xffffu) < b.tm2;
    if (MODE == MODE_SMU) near = near || T < b.close;
    const int n = (int)((t >> 16) & 0x7f) - (PATH == PATH_FIX ? 0 : 1), k = (int)((m >> 16) & 0x7f);
    return n >= 0 && n < p.n_a && k < p.n_b ? n * p.n_b + k : -1;
}

// Weighted product of a pair as the fast path added it (integer paths).
template <int LOS, int W>
__device__ __forceinline__ unsigned long long fast_product(const IPts<LOS, W> &I, int r, unsigned wj, unsigned lj) {
    if (W == 3) return corrected_product(I.wm[r], I.wb[r], wj, lj);
    return ((unsigned long long)I.wm[r] * wj) >> 16;
}

// Check n queued near-edge quads with the binary64 definition, one per lane.
// An entry is {first of its four j-points, source lane | own block << 5 |
// segment << 6 | the batch's bound (fix_bands) << 13}.  The lane repeats the quad's FP32 arithmetic
// on the same operands, so it sees the same bins and the same near pairs, and
// corrects the global histogram (integer weights: the CTA's exact sums) where the
// binary64 bin differs from the one counted.  (Pairs of a half that the batch left out are repeated too: they are
// beyond the last edge by more than the error bands, bin -1 both ways.)  With a
// rescue queue (pc_opts.rescue_capacity > 0) the fast count is
// undone instead and the pair queued while there is room.
template <int MODE, int LOS, int W, int PATH, bool TREE>
__device__ __noinline__ void check_near(const PairParams &p, const uint2 *queue, const int4 *seg, int n, int task,
                                        int cell, int start, int count, int half, unsigned copy, const float2 *s_lut) {
    const int lane = threadIdx.x & 31;
    const TaskDev &T = p.tasks[task];
    Ctx<MODE, LOS, is_fix(PATH) ? PATH_LIN : PATH> c;
    if (!is_fix(PATH)) c.init(p, s_lut, copy);
    // The lane's quad: segment, image, i-points and the batch's bands.
    int i0 = 0, j0 = 0, img = 13, meta = 0;
    unsigned vm = 0u, key = 0u;   // its j-points that are there; fix_bands
    bool own = false;
    if (lane < n) {
        const uint2 e = queue[lane];
        const int src = (int)(e.y & 31u);
        own = (e.y >> 5) & 1u;
        key = e.y >> 13;
        j0 = (int)e.x;
        i0 = start + src;
        int4 sg = make_int4(start, start + count, TREE ? -1 : 0, 13);
        if (!own) sg = seg[(e.y >> 6) & 127u];
        meta = sg.z;
        img = sg.w;
#pragma unroll
        for (int j = 0; j < 4; ++j) vm |= (j0 + j >= sg.x && j0 + j < sg.y) ? 1u << j : 0u;
        vm |= (src < half ? 1u << 8 : 0u) | (src < count - half ? 1u << 9 : 0u);
    }
    const Bands bd = fix_bands<MODE, PATH>(p, key);
    const float2 cfm = make_float2(bd.cfm, bd.cfm);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (TREE && meta >= 0 && !own && lane < n) o = tree_offset(p, cell, meta, img);
    const int ax = TREE ? 0 : cell % p.g.ng[0];
    auto stage = [&](int j) -> float3 {
        const float4 q = T.gj.rel[j];
        if (own) return make_float3(q.x, q.y, q.z);
        if (TREE) return make_float3(o.x + q.x, o.y + q.y, o.z + q.z);
        return stage_grid(p, q, T.gj.cx[j], ax, meta, img);
    };
    // Pass 1, a pair of j-points and an i-point at a time (rolled: this function
    // runs once in thousands of quads and shares the instruction cache with the
    // loops): which are near (bit 4 r + j), and the bins they were counted in,
    // two 16-bit words each (0xffff: none)
    unsigned m8 = 0u;
    unsigned b0 = 0u, b1 = 0u, b2 = 0u, b3 = 0u;
#pragma unroll 1
    for (int u = 0; u < 4; ++u) {
        const int r = u >> 1, j = j0 + 2 * (u & 1), i = i0 + r * half;
        const unsigned v = (vm >> 8 >> r & 1u) ? vm >> (2 * (u & 1)) & 3u : 0u;
        if (!v) continue;
        const float3 s0 = (v & 1u) ? stage(j) : make_float3(0.f, 0.f, 0.f);
        const float3 s1 = (v & 2u) ? stage(j + 1) : make_float3(0.f, 0.f, 0.f);
        IPts<LOS, W> I;
        I.xa[0] = I.ya[0] = I.za[0] = 0.f;
        load_i<MODE, LOS, W>(T.gi, i, I, 0);
        const float2 dx = __fadd2_rn(make_float2(s0.x, s1.x), make_float2(-I.x[0], -I.x[0]));
        const float2 dy = __fadd2_rn(make_float2(s0.y, s1.y), make_float2(-I.y[0], -I.y[0]));
        const float2 dz = __fadd2_rn(make_float2(s0.z, s1.z), make_float2(-I.z[0], -I.z[0]));
        float2 s2;
        bool n0, n1;
        int f0 = -1, f1 = -1;   // tables: near pairs are not counted
        if (is_fix(PATH)) {
            const Fix2 f = fix2<MODE, LOS, PATH>(p, dx, dy, dz, bd.cfs, cfm, I.xa[0], I.ya[0], I.za[0], s2);
            f0 = fix_bin<MODE, PATH>(p, f.T.x, f.M.x, bd, n0);
            f1 = fix_bin<MODE, PATH>(p, f.T.y, f.M.y, bd, n1);
        } else {
            const float2 qq = __ffma2_rn(dy, dy, __fmul2_rn(dx, dx));
            s2 = __ffma2_rn(dz, dz, qq);
            const Pair2 b = bin2<MODE, LOS, is_fix(PATH) ? PATH_LIN : PATH>(p, c, dx, dy, dz, qq, s2, I.xa[0],
                                                                           I.ya[0], I.za[0]);
            n0 = b.n0;
            n1 = b.n1;
            if (PATH != PATH_LUT && PATH != PATH_GLOBAL) {
                if (b.a0 < c.trash) f0 = entry_bin(p, (int)((b.a0 - copy) / c.hk4));
                if (b.a1 < c.trash) f1 = entry_bin(p, (int)((b.a1 - copy) / c.hk4));
            }
        }
        if ((v & 1u) && !(own && j <= i) && n0 && s2.x < p.r2cut) m8 |= 1u << (2 * u);
        if ((v & 2u) && !(own && j + 1 <= i) && n1 && s2.y < p.r2cut) m8 |= 2u << (2 * u);
        const unsigned w = (unsigned)f0 & 0xffffu | (unsigned)f1 << 16;
        b0 = u == 0 ? w : b0;
        b1 = u == 1 ? w : b1;
        b2 = u == 2 ? w : b2;
        b3 = u == 3 ? w : b3;
    }
    // Pass 2: the near pairs, one a lane
    unsigned done = 0u;
    while (__any_sync(FULL, m8 != 0u)) {
        if (m8) {
            const int k = __ffs(m8) - 1;
            m8 &= m8 - 1;
            const unsigned w = k < 4 ? (k < 2 ? b0 : b1) : (k < 6 ? b2 : b3);
            const unsigned fb = (k & 1) ? w >> 16 : w & 0xffffu;   // below 2^16 - 1: 4 bytes each fit shared memory
            const int fast = fb == 0xffffu ? -1 : (int)fb;
            const int i = i0 + half * (k >> 2), j = j0 + (k & 3);
            const size_t hb = (size_t)T.hist * p.nbins;
            unsigned long long slot = ~0ull;
            if (p.qcap) slot = atomicAdd(p.qcount, 1ull);
            int bin = -1;
            double wp = 0.0;
            if (slot < p.qcap) {
                p.queue[slot] = make_uint3((unsigned)i, (unsigned)j, (unsigned)img | ((unsigned)task << 5));
            } else {
                const double4_32a A = T.gi.xw[i], B = T.gj.xw[j];
                bin = max(f64_pair_bin<MODE, LOS>(A, B, img, p.g, p.Ea, p.n_a, p.Eb, p.n_b), -1);
                wp = __dmul_rn(A.w, B.w);
                ++done;
            }
            if (bin != fast) {
                if (fast >= 0) {
                    atomicAdd(&p.hist[hb + (size_t)fast], 0xffffffffffffffffull);   // - 1
                    if (W >= 2) {
                        IPts<LOS, W> I;
                        load_i<MODE, LOS, W>(T.gi, i, I, 0);
                        const unsigned wj = __float_as_uint(T.gj.rel[j].w);
                        const unsigned lj = (W == 3 && T.gj.wlo) ? T.gj.wlo[j] : 0u;
                        sub_exact(p, fast, fast_product<LOS, W>(I, 0, wj, lj));
                    }
                }
                if (bin >= 0) {
                    atomicAdd(&p.hist[hb + (size_t)bin], 1ull);
                    if (W >= 1) atomicAdd(&p.whist[hb + (size_t)bin], wp);
                }
            } else if (W == 1 && bin >= 0) {   // near pairs' binary64 weights are added here only
                atomicAdd(&p.whist[hb + (size_t)bin], wp);
            }
        }
        __syncwarp();
    }
    const unsigned tot = __reduce_add_sync(FULL, done);
    if (lane == 0 && tot) atomicAdd(&p.counters[1], (unsigned long long)tot);
}

// ---------------------------------------------------------------------------
// work items, candidate segments and box tests (both precisions)
// ---------------------------------------------------------------------------
// Work items: (block, 64-point part of the block, slice of its octs).  Slices
// (S > 1) split the i-points' candidates among warps, for about 12 items a
// warp of the grid, so that the last items do not leave the chip half empty (24:
// a warp starts over too often, 312k points 2.97 -> 3.32 ms; 6: within 2 %, but
// 3 to 4 % slower where a batch of items takes long).
// One histogram: each warp takes items from the global counter until none are
// left.  Several (batches): the CTA takes ranges of items of one histogram and
// flushes between them.
struct RangeShared {
    int cur, end, next, lim, task;
};
struct Items {
    int per_block, S, chunk;
    long long n;
    __device__ __forceinline__ void init(const PairParams &p, int nw) {
        const int nblocks = *p.nblocks;
        const long long units = max((long long)nblocks, p.npts_i / BI + 1);
        const long long want = 12ll * gridDim.x * nw;
        S = 1;
        if (units < want) S = (int)min(32ll, (want + units - 1) / units);
        per_block = p.nsub * S;
        n = (long long)nblocks * per_block;
        chunk = (int)max((long long)nw, min((long long)nw * 32 * S, n / (6ll * gridDim.x)));
    }
};

// Next item of this warp, -1 when none is left.  flush(task): every warp of the
// CTA, between barriers, after the last item of `task` (batches).
template <class F>
__device__ __forceinline__ long long next_item(const PairParams &p, const Items &W, RangeShared &R, F flush) {
    const int lane = threadIdx.x & 31;
    if (!p.multi) {
        unsigned v = 0u;
        if (lane == 0) v = (unsigned)atomicAdd(p.work_counter, 1);
        const long long it = __shfl_sync(FULL, v, 0);
        return it < W.n ? it : -1;
    }
    for (;;) {
        int v = 0;
        if (lane == 0) v = atomicAdd(&R.cur, 1);
        v = __shfl_sync(FULL, v, 0);
        if (v < R.end) return v;
        // range used up: every warp arrives here; the next one of a single
        // task is fetched, the histograms flushed on a change
        __syncthreads();
        const int old = R.task;
        __syncthreads();
        if (threadIdx.x == 0) {
            int b = R.next;
            if (b >= R.lim) {
                b = (int)min((long long)atomicAdd(p.work_counter, W.chunk), W.n);
                R.lim = (int)min((long long)b + W.chunk, W.n);
            }
            int e = b;
            if (b < R.lim) {
                const int task = p.blocks[b / W.per_block].task;
                int lo = b + 1, hi = R.lim;   // items [b, e) belong to `task`
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (p.blocks[mid / W.per_block].task == task) lo = mid + 1; else hi = mid;
                }
                e = lo;
                R.task = task;
            } else {
                R.task = -2;
            }
            R.cur = b;
            R.end = e;
            R.next = e;
        }
        __syncthreads();
        if (R.task != old && old >= 0) flush(old);
        if (R.task == -2) return -1;
    }
}

// The i-points of an item: [start, start + count) of block B, slice `part`.
struct Item {
    Block B;
    int start, count, part;
    int half;                // points of the first half: lane l holds points l and half + l
    int ax, ay, az;          // grid: the i-cell
    int ts0, ntl, own_end;   // list (tree) or stencil rows; end of the own cell (auto)
};
template <bool TREE>
__device__ __forceinline__ bool open_item(const PairParams &p, const Items &W, long long it, Item &I) {
    const unsigned blk = (unsigned)it / (unsigned)W.per_block;   // (the counter of the items is an int)
    I.B = p.blocks[blk];
    const int rem = (int)((unsigned)it - blk * (unsigned)W.per_block), sub = rem / W.S;
    I.part = rem - sub * W.S;
    const int k = (I.B.count + BI - 1) / BI;
    if (sub >= k) return false;
    if (TREE) {   // equal parts: close to the k-d tree's own cuts
        I.start = I.B.start + (int)((long long)I.B.count * sub / k);
        I.count = I.B.start + (int)((long long)I.B.count * (sub + 1) / k) - I.start;
        I.half = (I.count + 1) / 2;
    } else {      // full parts: a rest of up to 32 points leaves the second half out
        I.start = I.B.start + BI * sub;
        I.count = min(BI, I.B.count - BI * sub);
        I.half = min(32, I.count);
    }
    const TaskDev &T = p.tasks[I.B.task];
    const int nx = p.g.ng[0], ny = p.g.ng[1];
    I.ax = TREE ? 0 : I.B.cell % nx;
    I.ay = TREE ? 0 : (I.B.cell / nx) % ny;
    I.az = TREE ? 0 : I.B.cell / (nx * ny);
    I.ts0 = 0;
    I.own_end = 0;
    if (TREE) {
        I.ts0 = p.tseg_off[I.B.cell];
        I.ntl = p.tseg_off[I.B.cell + 1] - I.ts0;
        if (T.is_auto) {
            const int2 r = p.tblk_j[I.B.cell];
            I.own_end = r.x + r.y;
        }
    } else {
        I.ntl = p.nrows;
        if (T.is_auto) I.own_end = T.gi.cell_start[I.B.cell + 1];
    }
    return true;
}

// Bounding box of a half of the warp's i-points, relative to the j-grid's origin
// (no points: infinitely far from everything).
struct IBox {
    float lx, ly, lz, hx, hy, hz;
    __device__ __forceinline__ void clear() {
        lx = ly = lz = INFINITY;
        hx = hy = hz = -INFINITY;
    }
    __device__ __forceinline__ void add(const GridDev &g, const double4_32a &a) {
        const double ox = a.x - g.org[0], oy = a.y - g.org[1], oz = a.z - g.org[2];
        lx = fminf(lx, __double2float_rd(ox)); hx = fmaxf(hx, __double2float_ru(ox));
        ly = fminf(ly, __double2float_rd(oy)); hy = fmaxf(hy, __double2float_ru(oy));
        lz = fminf(lz, __double2float_rd(oz)); hz = fmaxf(hz, __double2float_ru(oz));
    }
    __device__ __forceinline__ void finish(const TaskDev &T) {
        const float ogx = (float)(T.gj.org[0] - T.gi.org[0]), ogy = (float)(T.gj.org[1] - T.gi.org[1]),
                    ogz = (float)(T.gj.org[2] - T.gi.org[2]);
        lx = warp_minf(lx) - ogx; ly = warp_minf(ly) - ogy; lz = warp_minf(lz) - ogz;
        hx = warp_maxf(hx) - ogx; hy = warp_maxf(hy) - ogy; hz = warp_maxf(hz) - ogz;
    }
    __device__ __forceinline__ void store(float4 *b) const {
        if ((threadIdx.x & 31) == 0) {
            b[0] = make_float4(lx, ly, lz, 0.f);
            b[1] = make_float4(hx, hy, hz, 0.f);
        }
    }
};

// Segments of chunk `ch` (32 stencil rows or listed nodes; the rest of the own
// cell with the first): seg = {first point, end, dy | dz << 16 (tree: j-node),
// image code}, pref the octs before each.  Returns their octs.
template <bool TREE>
__device__ __forceinline__ int build_chunk(const PairParams &p, const TaskDev &T, const Item &I, int ch, int4 *seg,
                                           float4 *soff, int *pref, int &nseg) {
    const int lane = threadIdx.x & 31;
    const int nx = p.g.ng[0], ny = p.g.ng[1], nz = p.g.ng[2];
    int noct = 0;
    nseg = 0;
    if (ch == 0 && I.own_end > I.start + I.count) {   // rest of the own cell: j > i for all
        const int a0 = I.start + I.count;
        if (lane == 0) {
            seg[0] = make_int4(a0, I.own_end, TREE ? -1 : 0, 13);
            pref[0] = 0;
            if (TREE) soff[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        nseg = 1;
        noct = ((I.own_end + 7) >> 3) - (a0 >> 3);
    }
    const int row = ch * 32 + lane;
    int a0[3], a1[3], im[3], np = 0, no = 0, meta = 0;
    if (row < I.ntl) {
        if (TREE) {
            const int2 e = p.tseg[I.ts0 + row];
            const int2 r = p.tblk_j[e.x];
            a0[0] = r.x; a1[0] = r.x + r.y; im[0] = e.y;
            meta = e.x;
            np = r.y > 0 ? 1 : 0;
            no = np ? ((a1[0] + 7) >> 3) - (a0[0] >> 3) : 0;
        } else {
            const int4 sr = p.stencil[row];
            const int dy = sr.x, dz = sr.y;
            int y = I.ay + dy, z = I.az + dz, wy = 0, wz = 0;
            bool in = true;
            if (y < 0) { in = in && p.g.periodic; y += ny; wy = -1; }
            else if (y >= ny) { in = in && p.g.periodic; y -= ny; wy = 1; }
            if (z < 0) { in = in && p.g.periodic; z += nz; wz = -1; }
            else if (z >= nz) { in = in && p.g.periodic; z -= nz; wz = 1; }
            meta = (dy & 0xFFFF) | (dz << 16);
            const int rowbase = (z * ny + y) * nx;
            const int x0 = I.ax + sr.z, x1 = I.ax + sr.w;
#pragma unroll
            for (int q = 0; q < 3; ++q) {   // the part left of the box, inside, right of it
                int c0, c1;
                if (q == 0) { c0 = x0 + nx; c1 = min(x1, -1) + nx; }
                else if (q == 1) { c0 = max(x0, 0); c1 = min(x1, nx - 1); }
                else { c0 = max(x0, nx) - nx; c1 = x1 - nx; }
                const bool use = in && c0 <= c1 && (q == 1 || p.g.periodic) && (q != 0 || x0 < 0) &&
                                 (q != 2 || x1 >= nx);
                a0[q] = a1[q] = 0;
                im[q] = q * 9 + (wy + 1) * 3 + (wz + 1);
                if (use) {
                    a0[q] = T.gj.cell_start[rowbase + c0];
                    a1[q] = T.gj.cell_start[rowbase + c1 + 1];
                }
                if (a1[q] > a0[q]) {
                    ++np;
                    no += ((a1[q] + 7) >> 3) - (a0[q] >> 3);
                }
            }
        }
    }
    const int is = warp_incl_scan(np), io = warp_incl_scan(no);
    int slot = nseg + is - np, o = noct + io - no;
#pragma unroll
    for (int q = 0; q < (TREE ? 1 : 3); ++q)
        if (np && a1[q] > a0[q]) {
            seg[slot] = make_int4(a0[q], a1[q], meta, im[q]);
            if (TREE) soff[slot] = tree_offset(p, I.B.cell, meta, im[q]);
            pref[slot] = o;
            o += ((a1[q] + 7) >> 3) - (a0[q] >> 3);
            ++slot;
        }
    nseg += __shfl_sync(FULL, is, 31);
    noct += __shfl_sync(FULL, io, 31);
    return noct;
}

// One round: octs 32 rd .. 32 rd + 31 of the chunk.  Those whose box can reach
// both halves of the i-points, or only the first or the second, are appended to
// that class's list {first point, segment | upper half of the squared gap << 16}
// and its length n[] grows.  Boxes are rounded outward, and r2prune carries the
// rounding of this test (host side), so a dropped pair is at least rcut apart.
template <int MODE, int LOS, class O>
__device__ __forceinline__ void ring_round(const PairParams &p, const TaskDev &T, int rd, int noct, int nseg,
                                           const int4 *seg, const int *pref, const float4 *ibox, int count, int half,
                                           uint2 *ring, int (&n)[3], unsigned long long &cand,
                                           unsigned long long &pruned) {
    const int lane = threadIdx.x & 31;
    const int f = rd * 32 + lane;
    bool keep[2] = {false, false};
    int lo = 0, p0 = 0;
    float g2 = INFINITY;
    if (f < noct) {
        int hi = nseg;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pref[mid] <= f) lo = mid; else hi = mid;
        }
        const int4 sg = seg[lo];
        const int oct = (sg.x >> 3) + (f - pref[lo]);
        p0 = oct << 3;
        float4 bl = T.gj.obox[2 * (size_t)oct], bh = T.gj.obox[2 * (size_t)oct + 1];
        if (p.g.periodic) {
            const float sx = (float)(sg.w / 9 - 1) * p.L32[0];
            const float sy = (float)((sg.w / 3) % 3 - 1) * p.L32[1];
            const float sz = (float)(sg.w % 3 - 1) * p.L32[2];
            bl.x += sx; bl.y += sy; bl.z += sz;
            bh.x += sx; bh.y += sy; bh.z += sz;
        }
        const unsigned nj = (unsigned)(min(sg.y, p0 + 8) - max(sg.x, p0));
        cand += (unsigned long long)(nj * (unsigned)count);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float4 l = ibox[2 * r], h = ibox[2 * r + 1];
            const float gx = fmaxf(fmaxf(bl.x - h.x, l.x - bh.x), 0.f);
            const float gy = fmaxf(fmaxf(bl.y - h.y, l.y - bh.y), 0.f);
            const float gz = fmaxf(fmaxf(bl.z - h.z, l.z - bh.z), 0.f);
            const float gq = fmaf(gy, gy, gx * gx), g = fmaf(gz, gz, gq);
            keep[r] = g <= p.r2prune;                 // (an infinite limit keeps gaps that overflow)
            if (MODE == MODE_SIGPI && LOS == LOS_Z)   // the reach is a cylinder
                keep[r] = keep[r] && gq <= p.q2prune && gz <= p.zprune;
            // (sigma, pi): the gap across the line of sight
            if (keep[r]) g2 = fminf(g2, MODE != MODE_SIGPI ? g : (LOS == LOS_Z ? gq : 0.f));
            else pruned += (unsigned long long)(nj * (unsigned)(r ? count - half : half));
        }
    }
    const uint2 e = make_uint2((unsigned)p0, (unsigned)lo | (__float_as_uint(g2) & 0xffff0000u));
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const bool in = c == 0 ? keep[0] && keep[1] : (c == 1 ? keep[0] && !keep[1] : !keep[0] && keep[1]);
        const unsigned who = __ballot_sync(FULL, in);
        if (in) ring[c * O::list + n[c] + __popc(who & below)] = e;
        n[c] += __popc(who);
    }
    __syncwarp();
}

// The class of the next batch: one with a full batch, else (rounds over) any with
// octs left; the batch takes the last of its list.  -1: none.
template <class O>
__device__ __forceinline__ int next_class(const int (&n)[3], bool over) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (n[c] >= O::jo) return c;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (over && n[c] > 0) return c;
    return -1;
}

// ---------------------------------------------------------------------------
// FP32 kernel
// ---------------------------------------------------------------------------
// W: 0 unweighted, 1 binary64 weighted sums, 2 integer weight products, 3 the
// same with binary64 remainders.  TREE: blocks are k-d tree nodes and their
// j-segments come from the list of the dual-tree traversal instead of the
// stencil rows.
//
// Registers: the loops need 50 to 80; with the rest of a warp's state 80 (96 with
// more operands a pair) give 24 (20) resident warps.  80 to 128 measured within
// 2 %, the loop alone loses 5 % at 12 warps.
template <int MODE, int LOS, int W, int PATH, bool TREE>
__global__ void __maxnreg__((LOS == LOS_MID && MODE != MODE_S) || W == 1 || PATH == PATH_LUT ? 96 : 80)
    k_pairs_f32(const __grid_constant__ PairParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RangeShared s_range;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    constexpr bool BYTES = is_fix(PATH) && MODE == MODE_S;   // LAY_BYTES
    using O = WarpOff<TREE, W != 0, false, batch_points(W, BYTES)>;
    unsigned char *ws = smem + p.sm_warp + (size_t)warp * O::total;
    int4 *seg = reinterpret_cast<int4 *>(ws);
    float4 *soff = reinterpret_cast<float4 *>(ws + O::soff);
    float *tx = reinterpret_cast<float *>(ws + O::tile);
    float *ty = tx + O::jb, *tz = ty + O::jb;
    double *tw = reinterpret_cast<double *>(ws + O::tw);
    unsigned *twm = reinterpret_cast<unsigned *>(tw);
    unsigned *twl = twm + O::jb;
    uint2 *queue = reinterpret_cast<uint2 *>(ws + O::queue);
    uint2 *ring = reinterpret_cast<uint2 *>(ws + O::ring);
    float4 *ibox = reinterpret_cast<float4 *>(ws + O::ibox);
    int *pref = reinterpret_cast<int *>(ws + O::pref);
    const Tile tile{tx, ty, tz, tw, twm, twl};
    const float2 *s_lut = reinterpret_cast<const float2 *>(smem + p.sm_lut);

    // clear the histograms, stage the tables
    for (int k = threadIdx.x; k < p.sm_lut / 4; k += blockDim.x) reinterpret_cast<unsigned *>(smem)[k] = 0u;
    for (int k = threadIdx.x; k < p.lut_total; k += blockDim.x)
        reinterpret_cast<float2 *>(smem + p.sm_lut)[k] = p.lut[k];
    if (W >= 2)
        for (int b = threadIdx.x; b < 2 * p.nbins; b += blockDim.x)
            p.wsums[(size_t)blockIdx.x * p.nbins * 2 + b] = 0ull;
    if (threadIdx.x == 0) s_range = RangeShared{0, 0, 0, 0, -1};
    const unsigned copy = 4u * (unsigned)(lane & (p.hist_k - 1));
    Ctx<MODE, LOS, is_fix(PATH) ? PATH_LIN : PATH> c;
    if (!is_fix(PATH)) c.init(p, s_lut, copy);
    const unsigned wbase = (unsigned)__cvta_generic_to_shared(smem + p.sm_whist);
    const float far = p.far;

    Items items;
    items.init(p, nw);
    unsigned long long cand = 0, pruned = 0;   // per lane
    unsigned since = 0, wterms = 0;            // quads, products per copy since this warp's flushes
    const unsigned flush_quads = (unsigned)(FLUSH_LIMIT / 256 / nw);
    // Integer weights: no record may hold more than `wmax` products.  Each warp adds
    // at most `wlimit` to any (a batch or more), then looks for the largest counter,
    // and flushes (counts with the weights) only past a quarter of the bound
    // (LAY_BYTES: bin by bin, past half).  After the latest look of any warp a record
    // holds at most what that look leaves, wkeep: the counter and the quad (eight
    // pairs a lane, taken as 16) that each warp is in; and each warp has added at most
    // wlimit since, so wkeep + nwarps wlimit <= wmax is the bound
    constexpr unsigned wmax = BYTES ? (W == 3 ? 2047u : 4095u) : WINT_LIMIT;
    // one loop body for both halves in turn where a body of two i-points a lane is
    // too large to share the instruction cache with the rest: (s, mu) along the
    // midpoint with binary64 weights (500k survey randoms 15.9 -> 12.1 ms; (sigma, pi)
    // there takes the two-point body, 100k x 2M points 32.1 -> 30.8)
    constexpr bool TWO = !(W == 3 && LOS == LOS_MID && MODE == MODE_SMU);
    constexpr unsigned wkeep = BYTES ? wmax / 2 : wmax / 4;   // what a look may leave in a record
    constexpr unsigned wbatch = 8u * (BYTES ? 1u : 32u) * O::jb / 4u;   // largest batch to one record
    static_assert(W < 2 || 8u * wbatch <= wmax - wkeep, "a batch of each of 8 warps fits");
    static_assert(W < 2 || wkeep > 16u * 8u * (BYTES ? 1u : 32u), "the quads in flight fit");
    const unsigned wlimit = (wmax - wkeep) / (unsigned)nw;
    const int wfull = (int)wkeep - 16 * nw * (32 / p.hist_k);
    const unsigned wper = W >= 2 ? 8u * (unsigned)(32 / p.hist_k) : 0u;   // products per copy and quad
    __syncthreads();

    for (;;) {
        auto flush = [&](int old) {
            const int h = p.tasks[old].hist;
            if (PATH != PATH_GLOBAL) flush_all<W>(p, warp, nw, h);
            __syncthreads();
            if (W >= 2) flush_exact(p, h, p.tasks[old].wscale);
            since = wterms = 0;
            __syncthreads();
        };
        const long long id = next_item(p, items, s_range, flush);
        if (id < 0) break;
        Item it;
        if (!open_item<TREE>(p, items, id, it)) continue;
        const TaskDev &T = p.tasks[it.B.task];

        IPts<LOS, W> I;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            IBox box;
            box.clear();
            I.x[r] = -far;      // unused: out of range of every j-point
            I.y[r] = I.z[r] = 0.f;
            // (midpoint: l = 2 x_i + d across d, else mu = 1 and sigma = 0 are near an
            // edge and every quad of such a lane is queued)
            I.xa[r] = I.za[r] = 0.f;
            I.ya[r] = LOS == LOS_MID ? far : 0.f;
            I.w[r] = 0.0;
            I.wm[r] = 0u;
            I.wb[r] = 0u;
            if (lane < (r ? it.count - it.half : it.half)) {
                const int i = it.start + lane + r * it.half;
                load_i<MODE, LOS, W>(T.gi, i, I, r);
                if (is_fix(PATH) && !(fabsf(I.x[r]) + fabsf(I.y[r]) + fabsf(I.z[r]) < 1e16f)) {
                    I.x[r] = -far;      // not a number: no pair
                    I.y[r] = I.z[r] = 0.f;
                }
                box.add(T.gi, T.gi.xw[i]);
            }
            box.finish(T);
            box.store(ibox + 2 * r);
        }

        // pairs inside the block (j > i) first
        bool own = T.is_auto && it.part == 0;
        if (own && lane == 0) cand += (unsigned long long)it.count * (unsigned)(it.count - 1) / 2;
        const int nchunk = max(1, (it.ntl + 31) / 32);
        int round0 = 0;      // rounds of 32 octs before this chunk
        int qn = 0;          // queued near-edge quads
        for (int ch = 0; ch < nchunk; ++ch) {
            __syncwarp();
            int nseg;
            const int noct = build_chunk<TREE>(p, T, it, ch, seg, soff, pref, nseg);
            __syncwarp();
            const int nround = (noct + 31) / 32;
            // this slice's rounds: global round number = part (mod S)
            int rd = (it.part - round0 % items.S + items.S) % items.S;
            round0 += nround;
            int left[3] = {0, 0, 0};   // octs to stage: for both halves, the first, the second
            for (;;) {
                while (!own && next_class<O>(left, false) < 0 && rd < nround) {
                    ring_round<MODE, LOS, O>(p, T, rd, noct, nseg, seg, pref, ibox, it.count, it.half, ring, left, cand,
                                             pruned);
                    rd += items.S;
                }
                // one batch: the block's own points, or up to eight octs of a class
                const int cls = own ? 0 : next_class<O>(left, true);
                int m = (it.count + 7) >> 3;
                if (!own) {
                    const int nc = cls == 1 ? left[1] : (cls == 2 ? left[2] : left[0]);
                    m = cls < 0 ? 0 : min((int)O::jo, nc);
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (c == cls) left[c] -= m;
                }
                const uint2 *list = ring + (cls == 1 ? O::list + left[1] : (cls == 2 ? 2 * O::list + left[2] : left[0]));
                unsigned near = 0u;
                unsigned key = 0u;   // bound of the batch's separations (fix_bands)
                if (m > 0) {
                    unsigned kmin = 0x7f80u;
#pragma unroll 2
                    for (int h = 0; h < (m + 3) >> 2; ++h) {
                        const int sl = lane + 32 * h, oc = sl >> 3;
                        float3 s = make_float3(far, 0.f, 0.f);
                        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                        int pj = it.start + sl;
                        bool v = own && sl < it.count;
                        if (v) {
                            q = T.gj.rel[pj];
                            s = make_float3(q.x, q.y, q.z);
                        } else if (!own && oc < m) {
                            const uint2 e = list[oc];
                            const unsigned es = e.y & 0xffffu;
                            const int4 sg = seg[es];
                            kmin = min(kmin, e.y >> 16);
                            pj = (int)e.x + (lane & 7);
                            v = pj >= sg.x && pj < sg.y;
                            if (v) {
                                q = T.gj.rel[pj];
                                if (TREE) {
                                    const float4 o = soff[es];
                                    s = make_float3(o.x + q.x, o.y + q.y, o.z + q.z);
                                } else {
                                    s = stage_grid(p, q, T.gj.cx[pj], it.ax, sg.z, sg.w);
                                }
                            }
                        }
                        if (is_fix(PATH) && !(fabsf(s.x) + fabsf(s.y) + fabsf(s.z) < 1e16f))
                            s = make_float3(far, 0.f, 0.f);   // not a number: no pair
                        tx[sl] = s.x; ty[sl] = s.y; tz[sl] = s.z;
                        if (W == 1) tw[sl] = v ? T.gj.xw[pj].w : 0.0;
                        if (W >= 2) twm[sl] = __float_as_uint(q.w);
                        if (W == 3) twl[sl] = (v && T.gj.wlo) ? T.gj.wlo[pj] : 0u;
                    }
                    __syncwarp();
                    const int nq = 2 * m;
                    since += nq;
                    if (since > flush_quads && PATH != PATH_GLOBAL) {
                        if (W >= 2) flush_all<W>(p, 0, 1, T.hist);
                        else flush_counts(p, 0, 1, T.hist);
                        since = nq;
                    }
                    if (W >= 2) {
                        wterms += wper * (unsigned)nq;
                        if (wterms > wlimit) {
                            if (BYTES) flush_bytes(p, wfull, 0, 1, T.hist);
                            else if (most_counted(p) > wfull) flush_records(p, 0, 1, T.hist);
                            wterms = wper * (unsigned)nq;
                        }
                    }
                    if constexpr (is_fix(PATH)) {
                        bool slow = own;
                        if (MODE == MODE_SMU || PATH == PATH_FIXLOG) {
                            // the batch's smallest separation: the smallest gap less the
                            // box tests' rounding
                            const float g2 = own ? 0.f : __uint_as_float(__reduce_min_sync(FULL, kmin) << 16);
                            const float g = fmaxf(g2 * rsqrt_fast(fmaxf(g2, 1e-30f)) - p.f_gm, 0.f);
                            key = __float_as_uint(g * g) >> 16;
                            slow = own || (MODE == MODE_SMU && __uint_as_float(key << 16) < p.f_sf2);
                        }
                        const Bands bd = fix_bands<MODE, PATH>(p, key);
                        if (slow) {
#pragma unroll 1
                            for (int r = cls == 2; r < (cls == 1 ? 1 : 2); ++r)
                                near |= quads_fix<MODE, LOS, W, PATH, true, 1>(
                                    p, tile, nq, half_points<MODE, LOS, W>(I, r), smem, bd, own ? 0 : BI,
                                    lane + r * it.half);
                        } else if (TWO && cls == 0) {
                            near = quads_fix<MODE, LOS, W, PATH, false, TWO ? 2 : 1>(p, tile, nq, I, smem, bd, 0, 0);
                        } else {
#pragma unroll 1
                            for (int r = cls == 2; r < (TWO || cls == 1 ? 1 + (cls == 2) : 2); ++r)
                                near |= quads_fix<MODE, LOS, W, PATH, false, 1>(
                                    p, tile, nq, half_points<MODE, LOS, W>(I, r), smem, bd, 0, 0);
                        }
                    } else {
                        const size_t hbase = (size_t)T.hist * p.nbins;
                        if (own) {
#pragma unroll 1
                            for (int r = 0; r < 2; ++r)
                                near |= pair_quads<MODE, LOS, W, PATH, true, 1>(
                                    p, tile, nq, half_points<MODE, LOS, W>(I, r), c, smem, wbase, 0,
                                    lane + r * it.half, hbase);
                        } else if (cls == 0) {
                            near = pair_quads<MODE, LOS, W, PATH, false, 2>(p, tile, nq, I, c, smem, wbase, 0, 0, hbase);
                        } else {
                            near = pair_quads<MODE, LOS, W, PATH, false, 1>(
                                p, tile, nq, half_points<MODE, LOS, W>(I, cls == 2), c, smem, wbase, 0, 0, hbase);
                        }
                    }
                }
                // queue the near quads, check them 32 at a time (and, before the
                // segments change, the rest)
                const bool last = rd >= nround && left[0] + left[1] + left[2] == 0 && !(own && nround > 0);
                for (;;) {
                    const unsigned who = __ballot_sync(FULL, near != 0u);
                    if (near) {
                        const int q = __ffs(near) - 1;
                        near &= near - 1;
                        uint2 e = make_uint2((unsigned)(it.start + 4 * q), (unsigned)lane | 32u | key << 13);
                        if (!own) {
                            const uint2 o = list[q >> 1];
                            e = make_uint2(o.x + 4u * (unsigned)(q & 1),
                                           (unsigned)lane | (o.y & 0xffffu) << 6 | key << 13);
                        }
                        queue[qn + __popc(who & ((1u << lane) - 1u))] = e;
                    }
                    qn += __popc(who);
                    const bool rest = last && !__any_sync(FULL, near != 0u);
                    if (qn >= 32 || (rest && qn > 0)) {
                        const int n = min(qn, 32);
                        __syncwarp();
                        check_near<MODE, LOS, W, PATH, TREE>(p, queue, seg, n, it.B.task, it.B.cell, it.start, it.count, it.half, copy,
                                                             s_lut);
                        __syncwarp();
                        qn -= n;
                        uint2 e = make_uint2(0u, 0u);
                        if (lane < qn) e = queue[n + lane];
                        __syncwarp();
                        if (lane < qn) queue[lane] = e;
                    }
                    __syncwarp();
                    if (who == 0u && qn < 32 && !(last && qn > 0)) break;
                }
                own = false;
                if (last) break;
            }
        }
    }
    __syncthreads();
    if (!p.multi) {   // batches have flushed after their last range
        if (PATH != PATH_GLOBAL) flush_all<W>(p, warp, nw, 0);
        if (W >= 2) {
            __syncthreads();
            flush_exact(p, 0, p.tasks[0].wscale);
        }
    }
    cand = warp_sum_u64(cand);
    pruned = warp_sum_u64(pruned);
    if (lane == 0 && cand) atomicAdd(&p.counters[0], cand);
    if (lane == 0 && pruned) atomicAdd(&p.counters[3], pruned);
}

// ---------------------------------------------------------------------------
// plain FP64 kernel: the binary64 definition for every pair of a box in reach
// ---------------------------------------------------------------------------
// Items, segments and box tests as the FP32 kernel's; the staged j-points and
// the i-points are the canonical binary64 coordinates.  This GPU issues about
// 1.7 binary64 operations per SM clock, so the kernel is bound by their number:
// eight a pair in reach (eleven with a periodic image) and two to four for the
// bin, which a search over the edges' FP32 roundings only proposes and binary64
// comparisons decide.  The definition's wrap rule needs no test: a pair in range
// under the visited image is one the rule gives that image, since the reach
// stays below L / 2 by more than the roundings.  Before: every candidate of the
// stencil, with six comparisons for the wrap rule and a binary64 search; 50,001
// uniform points in 40 s bins took 115 ms as a whole call, now 5.45 ms.
struct F64Edges {
    const double *Ea, *Eb;
    const float *Fa, *Fb;    // FP32 roundings, or null
};

// Largest k with v >= E[k] (v >= E[0] holds), from a guess by the FP32 edges.
__device__ __forceinline__ int locate64(double v, const double *E, const float *F, int n) {
    if (!F) return f64_locate(v, E, n);
    const float f = (float)v;
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (f >= F[mid]) lo = mid; else hi = mid;
    }
    while (lo > 0 && v < E[lo]) --lo;
    while (lo + 1 < n && v >= E[lo + 1]) ++lo;
    return lo;
}
// Largest j < n with p2 >= M[j] s2 (the product rounded once).
__device__ __forceinline__ int locate64_mu(double p2, double s2, const double *M, const float *F, int n) {
    if (!F) return f64_locate_mu(p2, s2, M, n);
    const float f = __fdividef((float)p2, (float)s2);
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (f >= F[mid]) lo = mid; else hi = mid;
    }
    while (lo > 0 && !(p2 >= __dmul_rn(M[lo], s2))) --lo;
    while (lo + 1 < n && p2 >= __dmul_rn(M[lo + 1], s2)) ++lo;
    return lo;
}

// Bin of an in-reach pair from its separation d (a, b: the positions, for the
// midpoint line of sight); -1 outside.
template <int MODE, int LOS>
__device__ __forceinline__ int bin64(double d0, double d1, double d2, double s2, const double *a, const double *b,
                                     const F64Edges &E, int na, int nb) {
    if (MODE == MODE_S) {
        if (!(s2 >= E.Ea[0] && s2 < E.Ea[na])) return -1;
        return locate64(s2, E.Ea, E.Fa, na);
    }
    double p2;
    if (LOS == LOS_Z) {
        p2 = __dmul_rn(d2, d2);
    } else {
        const double l0 = __dadd_rn(a[0], b[0]), l1 = __dadd_rn(a[1], b[1]), l2 = __dadd_rn(a[2], b[2]);
        const double sl = __dadd_rn(__dadd_rn(__dmul_rn(d0, l0), __dmul_rn(d1, l1)), __dmul_rn(d2, l2));
        const double ll = __dadd_rn(__dadd_rn(__dmul_rn(l0, l0), __dmul_rn(l1, l1)), __dmul_rn(l2, l2));
        p2 = (ll > 0.0) ? __ddiv_rn(__dmul_rn(sl, sl), ll) : 0.0;
    }
    if (MODE == MODE_SMU) {
        if (!(s2 >= E.Ea[0] && s2 < E.Ea[na])) return -1;
        const int k = locate64(s2, E.Ea, E.Fa, na);
        const int j = (s2 > 0.0) ? locate64_mu(p2, s2, E.Eb, E.Fb, nb) : 0;
        return k * nb + j;
    }
    double q2 = __dsub_rn(s2, p2);
    if (q2 < 0.0) q2 = 0.0;
    if (!(q2 >= E.Ea[0] && q2 < E.Ea[na])) return -1;
    if (!(p2 >= E.Eb[0] && p2 < E.Eb[nb])) return -1;
    return locate64(q2, E.Ea, E.Fa, na) * nb + locate64(p2, E.Eb, E.Fb, nb);
}

template <int MODE, int LOS, bool W>
__global__ void __maxnreg__(96) k_pairs_f64(const __grid_constant__ PairParams p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RangeShared s_range;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    using O = WarpOff<false, false, true, 64>;
    unsigned char *ws = smem + p.sm_warp + (size_t)warp * O::total;
    int4 *seg = reinterpret_cast<int4 *>(ws);
    double *tile = reinterpret_cast<double *>(ws + O::tile);   // {x, y, z, w, shift x, y, z} by point
    uint2 *ring = reinterpret_cast<uint2 *>(ws + O::ring);
    float4 *ibox = reinterpret_cast<float4 *>(ws + O::ibox);
    int *pref = reinterpret_cast<int *>(ws + O::pref);
    double *sEa = reinterpret_cast<double *>(smem + p.sm_lut), *sEb = sEa + p.n_a + 1;
    float *sF = reinterpret_cast<float *>(sEb + p.n_b + 1);
    F64Edges E{sEa, sEb, p.sm_guess ? sF : nullptr, p.sm_guess ? sF + p.n_a + 1 : nullptr};

    for (int k = threadIdx.x; k < p.sm_lut / 4; k += blockDim.x) reinterpret_cast<unsigned *>(smem)[k] = 0u;
    for (int k = threadIdx.x; k <= p.n_a; k += blockDim.x) {
        sEa[k] = p.Ea[k];
        if (p.sm_guess) sF[k] = (float)p.Ea[k];
    }
    for (int k = threadIdx.x; k <= p.n_b; k += blockDim.x) {
        sEb[k] = p.Eb[k];
        if (p.sm_guess) sF[p.n_a + 1 + k] = (float)p.Eb[k];
    }
    if (threadIdx.x == 0) s_range = RangeShared{0, 0, 0, 0, -1};
    int *hist = reinterpret_cast<int *>(smem);
    double *whist = reinterpret_cast<double *>(smem + p.sm_whist);
    const int K = p.hist_k, kc = lane & (K - 1);
    Items items;
    items.init(p, nw);
    unsigned long long cand = 0, pruned = 0;
    unsigned since = 0;                              // j-points since this warp's last flush
    const unsigned flush_j = (unsigned)(FLUSH_LIMIT / BI / nw);
    __syncthreads();
    // squared reach, with the rounding of the squares (sigma^2 + pi^2 for both)
    const double reach2 = (MODE == MODE_SIGPI ? sEa[p.n_a] + sEb[p.n_b] : sEa[p.n_a]) * (1.0 + 1e-12);

    for (;;) {
        auto flush = [&](int old) {
            if (p.smem_hist_ok) flush_all<W ? 1 : 0>(p, warp, nw, p.tasks[old].hist);
            since = 0;
            __syncthreads();
        };
        const long long id = next_item(p, items, s_range, flush);
        if (id < 0) break;
        Item it;
        if (!open_item<false>(p, items, id, it)) continue;
        const TaskDev &T = p.tasks[it.B.task];
        const size_t hbase = (size_t)T.hist * p.nbins;
        double a[2][3], wi[2];
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            IBox box;
            box.clear();
            a[r][0] = a[r][1] = a[r][2] = __longlong_as_double(0x7ff8000000000000ll);   // no point: not a number
            wi[r] = 0.0;
            if (lane < (r ? it.count - it.half : it.half)) {
                const double4_32a q = T.gi.xw[it.start + lane + r * it.half];
                a[r][0] = q.x; a[r][1] = q.y; a[r][2] = q.z;
                wi[r] = q.w;
                box.add(T.gi, q);
            }
            box.finish(T);
            box.store(ibox + 2 * r);
        }
        bool own = T.is_auto && it.part == 0;
        if (own && lane == 0) cand += (unsigned long long)it.count * (unsigned)(it.count - 1) / 2;
        const int nchunk = max(1, (it.ntl + 31) / 32);
        int round0 = 0;
        for (int ch = 0; ch < nchunk; ++ch) {
            __syncwarp();
            int nseg;
            const int noct = build_chunk<false>(p, T, it, ch, seg, nullptr, pref, nseg);
            __syncwarp();
            const int nround = (noct + 31) / 32;
            int rd = (it.part - round0 % items.S + items.S) % items.S;
            round0 += nround;
            int left[3] = {0, 0, 0};   // octs to stage: for both halves, the first, the second
            for (;;) {
                while (!own && next_class<O>(left, false) < 0 && rd < nround) {
                    ring_round<MODE, LOS, O>(p, T, rd, noct, nseg, seg, pref, ibox, it.count, it.half, ring, left, cand,
                                             pruned);
                    rd += items.S;
                }
                const int cls = own ? 0 : next_class<O>(left, true);
                int m = (it.count + 7) >> 3;
                if (!own) {
                    const int nc = cls == 1 ? left[1] : (cls == 2 ? left[2] : left[0]);
                    m = cls < 0 ? 0 : min((int)O::jo, nc);
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (c == cls) left[c] -= m;
                }
                if (m == 0) break;
                const uint2 *list = ring + (cls == 1 ? O::list + left[1] : (cls == 2 ? 2 * O::list + left[2] : left[0]));
                bool shifted = false;
#pragma unroll
                for (int h = 0; h < O::jb / 32; ++h) {
                    const int sl = lane + 32 * h, oc = sl >> 3;
                    int pj = it.start + sl, img = 13;
                    bool v = own && sl < it.count;
                    if (!own && oc < m) {
                        const uint2 e = list[oc];
                        const int4 sg = seg[e.y & 0xffffu];
                        pj = (int)e.x + (lane & 7);
                        v = pj >= sg.x && pj < sg.y;
                        img = sg.w;
                    }
                    double4_32a q = make_double4_32a(0.0, 0.0, 0.0, 0.0);
                    q.x = __longlong_as_double(0x7ff8000000000000ll);
                    if (v) q = T.gj.xw[pj];
                    double *t = tile + 7 * sl;
                    t[0] = q.x; t[1] = q.y; t[2] = q.z; t[3] = q.w;
                    // d - L is d + (-L), and d + 0 is d
                    t[4] = (double)(img / 9 - 1) * p.g.L[0];
                    t[5] = (double)((img / 3) % 3 - 1) * p.g.L[1];
                    t[6] = (double)(img % 3 - 1) * p.g.L[2];
                    shifted = shifted || (p.g.periodic && img != 13);
                }
                shifted = __any_sync(FULL, shifted);
                __syncwarp();
                since += 8 * m;
                if (since > flush_j && p.smem_hist_ok) {
                    flush_counts(p, 0, 1, T.hist);
                    since = 8 * m;
                }
                for (int j = 0; j < 8 * m; ++j) {
                    const double *t = tile + 7 * j;
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        if (cls == 2 - r) continue;   // the other half's batch
                        double d0 = __dsub_rn(t[0], a[r][0]), d1 = __dsub_rn(t[1], a[r][1]),
                               d2 = __dsub_rn(t[2], a[r][2]);
                        if (shifted) {
                            d0 = __dadd_rn(d0, t[4]);
                            d1 = __dadd_rn(d1, t[5]);
                            d2 = __dadd_rn(d2, t[6]);
                        }
                        const double s2 =
                            __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
                        bool in = s2 < reach2;
                        if (own) in = in && j > lane + r * it.half;
                        if (in) {
                            const int b = bin64<MODE, LOS>(d0, d1, d2, s2, a[r], t, E, p.n_a, p.n_b);
                            if (b >= 0) {
                                if (p.smem_hist_ok) {
                                    atomicAdd(&hist[b * K + kc], 1);
                                    if (W) atomicAdd(&whist[b * K + kc], __dmul_rn(wi[r], t[3]));
                                } else {
                                    atomicAdd(&p.hist[hbase + b], 1ull);
                                    if (W) atomicAdd(&p.whist[hbase + b], __dmul_rn(wi[r], t[3]));
                                }
                            }
                        }
                    }
                }
                own = false;
                __syncwarp();
            }
        }
    }
    __syncthreads();
    if (!p.multi && p.smem_hist_ok) flush_all<W ? 1 : 0>(p, warp, nw, 0);
    cand = warp_sum_u64(cand);
    pruned = warp_sum_u64(pruned);
    if (lane == 0 && cand) atomicAdd(&p.counters[0], cand);
    if (lane == 0 && pruned) atomicAdd(&p.counters[3], pruned);
}

// ---------------------------------------------------------------------------
// rescue kernel: binary64 definition for every queued pair
// ---------------------------------------------------------------------------
template <int MODE, int LOS>
__global__ void __launch_bounds__(256) k_rescue(const __grid_constant__ PairParams p) {
    const unsigned long long n = min(*p.qcount, p.qcap);
    for (unsigned long long k = blockIdx.x * 256ull + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * 256ull) {
        uint3 e = p.queue[k];
        const int task = (int)(e.z >> 5), img = (int)(e.z & 31);
        const TaskDev &T = p.tasks[task];
        double4_32a a = T.gi.xw[e.x];
        double4_32a b = T.gj.xw[e.y];
        int bin = f64_pair_bin<MODE, LOS>(a, b, img, p.g, p.Ea, p.n_a, p.Eb, p.n_b);
        if (bin >= 0) {
            size_t h = (size_t)T.hist * p.nbins + bin;
            atomicAdd(&p.hist[h], 1ull);
            if (p.weighted) atomicAdd(&p.whist[h], __dmul_rn(a.w, b.w));
        }
    }
}

// ---------------------------------------------------------------------------
// instantiation helpers
// ---------------------------------------------------------------------------
template <int MODE, int LOS>
using PairKernel = void (*)(PairParams);

template <int MODE, int LOS, int PATH, bool TREE>
PairKernel<MODE, LOS> pick_w(const PairParams &p) {
    if (!p.weighted) return k_pairs_f32<MODE, LOS, 0, PATH, TREE>;
    if constexpr (is_fix(PATH))   // integer weight products only
        return p.wcorr ? k_pairs_f32<MODE, LOS, 3, PATH, TREE> : k_pairs_f32<MODE, LOS, 2, PATH, TREE>;
    else {
    if constexpr (PATH != PATH_LUT && PATH != PATH_GLOBAL) {
        if (p.wint && p.wcorr) return k_pairs_f32<MODE, LOS, 3, PATH, TREE>;
        if (p.wint) return k_pairs_f32<MODE, LOS, 2, PATH, TREE>;
    }
    return k_pairs_f32<MODE, LOS, 1, PATH, TREE>;
    }
}

// Kernel variant for the weights and the way the bins are found; (sigma, pi)
// floors exist for edges from zero only.
template <int MODE, int LOS, bool TREE>
PairKernel<MODE, LOS> pick_f32(const PairParams &p) {
    if (!p.smem_hist_ok) return pick_w<MODE, LOS, PATH_GLOBAL, TREE>(p);
    if constexpr (MODE != MODE_SIGPI) {
        if (p.path == PATH_LINOFF) return pick_w<MODE, LOS, PATH_LINOFF, TREE>(p);
        if (p.path == PATH_FIXOFF) return pick_w<MODE, LOS, PATH_FIXOFF, TREE>(p);
        if (p.path == PATH_LOG) return pick_w<MODE, LOS, PATH_LOG, TREE>(p);
    }
    if (p.path == PATH_FIX) return pick_w<MODE, LOS, PATH_FIX, TREE>(p);
    if (p.path == PATH_FIXLOG) return pick_w<MODE, LOS, PATH_FIXLOG, TREE>(p);
    if (p.path == PATH_LIN) return pick_w<MODE, LOS, PATH_LIN, TREE>(p);
    return pick_w<MODE, LOS, PATH_LUT, TREE>(p);
}

template <int MODE, int LOS, bool TREE>
cudaError_t launch_mode_f32(const PairParams &p, int grid, size_t smem, cudaStream_t st) {
    PairKernel<MODE, LOS> k = pick_f32<MODE, LOS, TREE>(p);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (grid <= 0) return cudaSuccess;
    k<<<grid, 32 * p.nwarps, smem, st>>>(p);
    note_launch();
    return cudaGetLastError();
}

template <int MODE, int LOS, bool TREE>
int occupancy_mode_f32(const PairParams &p, size_t smem) {
    PairKernel<MODE, LOS> k = pick_f32<MODE, LOS, TREE>(p);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, 32 * p.nwarps, smem) != cudaSuccess) return 0;
    return nb;
}

template <int MODE, int LOS>
cudaError_t launch_mode_f64(const PairParams &p, int grid, size_t smem, cudaStream_t st) {
    void (*k)(PairParams) = p.weighted ? k_pairs_f64<MODE, LOS, true> : k_pairs_f64<MODE, LOS, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (grid <= 0) return cudaSuccess;
    k<<<grid, 32 * p.nwarps, smem, st>>>(p);
    note_launch();
    return cudaGetLastError();
}

template <int MODE, int LOS>
int occupancy_mode_f64(const PairParams &p, size_t smem) {
    void (*k)(PairParams) = p.weighted ? k_pairs_f64<MODE, LOS, true> : k_pairs_f64<MODE, LOS, false>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, 32 * p.nwarps, smem) != cudaSuccess) return 0;
    return nb;
}

template <int MODE, int LOS>
cudaError_t launch_mode_rescue(const PairParams &p, int grid, cudaStream_t st) {
    k_rescue<MODE, LOS><<<grid, 256, 0, st>>>(p);
    note_launch();
    return cudaGetLastError();
}

}  // namespace pc
