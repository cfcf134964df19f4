// Row statistics for truncated sampling distributions (top-k / top-p; rules in cut.cuh).
//
// The nucleus of a row is a few dozen to a few thousand tokens out of 10^5, and its cut is a VALUE, so the
// selection need not keep the row.  One CTA per row; the row is streamed once from HBM through a ring of
// asynchronous copies, and while it passes every logit at or above a running BOUND that is known to lie below
// the cut is set aside as a CANDIDATE:
//   top-k        bound = the k-th largest of the units' maxima in the first slice (each is a logit of the row, so
//                at least k logits lie at or above it), tightened to the k-th largest candidate so far a few times;
//   top-p alone  the mass of the whole row, which fixes the target, is summed in the same pass; bf16: bound = the cut
//                that the first slice alone would have at a larger top-p (a guess: the end of the row tells whether
//                the nucleus stayed above it); fp32: WINDOW_OCTAVES below the row's running maximum.
// One packed maximum per 16-byte unit finds the units that hold a candidate; a warp lists those of its share of a
// slice and then looks at their logits, a logit per lane, in the ring.  bf16 candidates become counts in a histogram over logit VALUES (a bf16 logit has 16 bits: 20 octaves of
// magnitude, both signs, are 5120 bins), from which both cuts and all kept sums follow: the mass of a bin is
// its count times the mass of its value, and no number of candidates overflows it.  fp32 candidates become a
// list of keys (4096 entries) for a radix selection.  Where the first slice says that more than DENSE of the row are
// candidates (T near 1 with top-p near 1: a quarter of it) every logit is compared and counted on the spot.
// A bf16 nucleus that reaches below the bound is counted again from L2, down to one that the row's mass guarantees.
// What is left over (fp32 nuclei beyond the list, k above 1024 (fp32: 256), values outside the 20 octaves) runs an adaptive
// radix selection over the row in L2, in the same CTA.
//
// Bound by HBM for large batches.  The ring runs ahead across rows, so the copies of the next row are in flight
// while the selection of the current one (a few microseconds of block-wide scans) runs.
#pragma once
#include "common.cuh"
#include "cut.cuh"
#include "stream.cuh"

namespace specv {
namespace trunc {

constexpr int NT = 256;
constexpr int NW = NT / 32;
constexpr int UN = 4;                // 16-byte units per thread and slice
constexpr int DEPTH = 3;             // stages of the ring, one slice each
constexpr int NB = cut::NB;          // bins of a radix level
constexpr int PER = NB / NT;
constexpr int CAP = 4096;            // fp32: candidate keys per row
constexpr float WINDOW_OCTAVES = 14.f;
constexpr float SAMPLE_OCTAVES = 24.f;   // bf16 top-p: how far below its maximum the first slice is counted
constexpr float SAMPLE_REST = 0.7f;      // safety factor of the bound it gives (mass_bound)
constexpr float DENSE = 0.008f;           // share of candidates above which a list of units costs more than counting all
constexpr float LOWEST = -3.3e38f;   // a bound that every finite logit passes and -inf does not
template <int DT> constexpr int K_FAST = DT == SPEC_BF16 ? UN * NT : NT;      // largest top-k the first slice can bound

// bf16 value bins, largest value first: TB positive magnitudes, then TB negative ones; magnitudes below 2^-11
// share the two bins in the middle (0 itself in the first of them), those of 2^9 and more the outermost ones
constexpr int TB = 20 * 128;
constexpr int M0 = (127 - 11) << 7;
constexpr float HIGH = 508.f;                 // below the outermost bin's value
constexpr int ODD_LOW = 1, ODD_HIGH = 2;      // a candidate in such a shared bin (other than 0) was seen

struct RParams {
    int B, N, V, top_k;
    float top_p;
    const void *zp, *zq;
    long long seq_stride, node_stride, topo_stride;
    const int *parent;         // NULL: every row of `zp` only (spec_tree_probs)
    float T;
    const float *T_seq;
    RowPart *part;             // [B*N*2] the rows' statistics
    float *cut;                // [B*N*2] smallest kept logit of every row (for spec_tree_probs)
    stream::NodeInit init;     // per-call words of the workspace to set (every-node verification)
};

// the scale factors of a temperature
struct Scale {
    float T, sf, s_hi, s_lo, window;
    double s_d;
};
struct __align__(16) Shared {
    Scale sc;
    unsigned long long warp_tot[NW];
    double red[NW][2];
    int verdict;               // bf16: what the selecting warp found (below)
    float bound;               // top-k: the bound it set
    double total;              // mass of the row in units of its largest e
    uint32_t runmax;           // key of the largest logit seen by the row so far
    int count;                 // fp32: candidates appended (may exceed CAP: overflow)
    int odd;
    int sel_bin;
    unsigned long long sel_before;
};
template <int DT> struct Layout {
    static constexpr int RING = DEPTH * UN * NT * 16;
    static constexpr int HITS = NW * UN * 32;            // a byte per unit of a warp's share of a slice
    // bf16: counts of 2 TB values; fp32: a radix histogram (64-bit bins as two words) and the candidate keys
    static constexpr int BINS = DT == SPEC_BF16 ? 2 * TB * 4 : NB * 8 + CAP * 4;
    static constexpr int BYTES = RING + HITS + BINS + (int)sizeof(Shared);
};
static_assert(2 * TB * 4 >= NB * 8, "the radix histogram of the slow path fits in the value bins");
template <int DT> constexpr int CTAS = DT == SPEC_BF16 ? 3 : 2;       // per SM
static_assert(Layout<SPEC_BF16>::BYTES <= (227 * 1024) / 3 - 1024 && Layout<SPEC_F32>::BYTES <= 113 * 1024, "CTAs per SM");

// e 2^44 truncated to an integer, for e = 2^x in [0, 2): integer arithmetic on the bits of the float
// (the same value as casting the exact product (double)e * 2^44 to an unsigned integer)
__device__ __forceinline__ unsigned long long fix44(float e)
{
    const uint32_t u = __float_as_uint(e);
    const int ex = (int)(u >> 23) & 0xFF;
    if (ex == 0) return 0ull;                                    // zero (subnormals are flushed by ex2.approx.ftz)
    const unsigned long long mant = (unsigned long long)((u & 0x7FFFFFu) | 0x800000u);
    const int sh = ex - 127 - 23 + 44;                           // e = mant 2^(ex - 127 - 23)
    return sh >= 0 ? mant << sh : (sh > -64 ? mant >> (-sh) : 0ull);
}

__device__ __forceinline__ int bin_of(uint32_t u16, int &t)
{
    const int mag = (int)(u16 & 0x7FFFu);
    t = min(max(mag, M0) - M0, TB - 1);
    return u16 > 0x8000u ? TB + t : TB - 1 - t;
}
__device__ __forceinline__ int bin_of(float z)
{
    int t;
    return bin_of(__float_as_uint(z) >> 16, t);
}
__device__ __forceinline__ float value_of_bin(int b)
{
    const int t = b < TB ? TB - 1 - b : b - TB;
    const uint32_t mag = t == 0 ? 0u : (uint32_t)(t + M0) << 16;
    return __uint_as_float(b < TB ? mag : mag | 0x80000000u);
}
// the last bin of which every value is at or above `bound`
__device__ __forceinline__ int last_bin_above(float bound)
{
    const int b = bin_of(bound);
    if (b == TB || b == TB - 1) return bound <= 0.f ? b : b - 1;
    return (bound > 0.f && value_of_bin(b) < bound) ? b - 1 : b;
}
__device__ __forceinline__ void count_value(uint32_t *cnt, int *odd, uint32_t u16)
{
    int t;
    const int b = bin_of(u16, t);
    if ((unsigned)(t - 1) >= (unsigned)(TB - 2) && (u16 & 0x7FFFu)) atomicOr(odd, t ? ODD_HIGH : ODD_LOW);
    atomicAdd(&cnt[b], 1u);
}
// The 8 logits of a bf16 unit that are at or above the bound.  zmax: none is larger.
__device__ __forceinline__ void count_unit(uint32_t *cnt, int *odd, const uint4 &r, float bound, float zmax)
{
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
    const int b16 = (int)(__float_as_uint(bound) >> 16) + ((__float_as_uint(bound) & 0xFFFFu) ? 1 : 0);
    if (bound > 0.f && b16 >= M0 && zmax < HIGH) {
        // Positive values order like their bits and none of these falls into a shared bin: four instructions a logit
        // (written out: the compiler makes a branch of the predicated addition, twice as many).
        const uint32_t base = smem_u32(cnt) + (uint32_t)(TB - 1 + M0) * 4u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int v = (k & 1) ? (int)w[k >> 1] >> 16 : (int)(short)w[k >> 1];
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %0, %1;\n\t@p red.shared.add.u32 [%2], 1;\n\t}" ::"r"(v), "r"(b16),
                         "r"(base - 4u * (uint32_t)v)
                         : "memory");
        }
    } else {
        float z[8];
        stream::unpack_unit<SPEC_BF16>(r, z);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (z[k] >= bound) count_value(cnt, odd, __float_as_uint(z[k]) >> 16);
    }
}

// The first of the bins b0 .. b1 at which the running sum of weight(bin) reaches `target`, by one warp, 128 bins per
// step; -1 when the total stays below.
template <typename T, typename F>
__device__ __forceinline__ int warp_find(int b0, int b1, double target, F weight)
{
    const int lane = threadIdx.x & 31;
    T carry = 0;
    for (int base = b0; base <= b1; base += 128) {
        T loc[4], lsum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int b = base + lane * 4 + k;
            loc[k] = b <= b1 ? weight(b) : (T)0;
            lsum += loc[k];
        }
        T incl = lsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        T run = carry + incl - lsum;
        int hit = -1;
        if ((double)run < target && (double)(run + lsum) >= target) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (hit < 0 && (double)(run + loc[k]) >= target) hit = base + lane * 4 + k;
                run += loc[k];
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit >= 0);
        if (m) return __shfl_sync(0xffffffffu, hit, __ffs(m) - 1);
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    return -1;
}

// The first of the bins b0 .. b1 at which the running sum of weight(bin) reaches `target`; -1 when the total
// stays below.  before: the sum of the bins ahead of it.  All threads of the block call it and get the answer.
template <typename F>
__device__ __forceinline__ int find_bin(Shared &S, int b0, int b1, double target, unsigned long long &before, F weight)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    unsigned long long carry = 0;
    int found = -1;
    before = 0;
    for (int base = b0; base <= b1 && found < 0; base += NT * PER) {
        unsigned long long loc[PER], lsum = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int b = base + tid * PER + k;
            loc[k] = b <= b1 ? weight(b) : 0ull;
            lsum += loc[k];
        }
        unsigned long long incl = lsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        __syncthreads();
        if (lane == 31) S.warp_tot[w] = incl;
        if (tid == 0) S.sel_bin = -1;
        __syncthreads();
        unsigned long long ahead = carry;
        for (int k = 0; k < NW; ++k) { const unsigned long long t = S.warp_tot[k]; carry += t; if (k < w) ahead += t; }
        unsigned long long run = ahead + incl - lsum;
        if ((double)run < target && (double)(run + lsum) >= target) {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                if ((double)run < target && (double)(run + loc[k]) >= target) { S.sel_bin = base + tid * PER + k; S.sel_before = run; }
                run += loc[k];
            }
        }
        __syncthreads();
        found = S.sel_bin;
        before = S.sel_before;
    }
    return found;
}

__device__ __forceinline__ unsigned long long block_sum(Shared &S, unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) S.warp_tot[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
    for (int k = 0; k < NW; ++k) v += S.warp_tot[k];
    return v;
}

// 64-bit bins as two words: a shared-memory addition of 32 bits is one instruction, one of 64 is a loop
__device__ __forceinline__ void bin_add(uint32_t *lo, uint32_t *hi, int b, unsigned long long v)
{
    const uint32_t l = (uint32_t)v, old = atomicAdd(&lo[b], l);
    const uint32_t h = (uint32_t)(v >> 32) + (old + l < old ? 1u : 0u);
    if (h) atomicAdd(&hi[b], h);
}

// Selection over keys by radix levels of at most NB bins, the levels fitted to the range [klo, khi] that is still
// open.  MASS false: the key of the need-th largest element (need counts elements); MASS true: the key at
// which the fixed-point mass, taken in descending key order, first reaches `need`.  visit(f) calls f(key) for
// every element of the block's set.  False when the elements do not reach `need`.
template <bool MASS, typename V>
__device__ __forceinline__ bool radix_select(Shared &S, uint32_t *lo, uint32_t *hi, double need, uint32_t klo, uint32_t khi,
                                             float m, float sf, uint32_t &key_out, V visit)
{
    double above = 0.0;
    for (;;) {
        const uint32_t range = khi - klo;
        const int sh = range < (uint32_t)NB ? 0 : 32 - __clz(range) - cut::NBITS;
        __syncthreads();
        for (int i = threadIdx.x; i < NB; i += NT) { lo[i] = 0; hi[i] = 0; }
        __syncthreads();
        visit([&](uint32_t key) {
            if (key < klo || key > khi) return;
            const int b = (int)((khi - key) >> sh);
            if (MASS) bin_add(lo, hi, b, fix44(ex2_approx((cut::value_of(key) - m) * sf)));
            else atomicAdd(&lo[b], 1u);
        });
        __syncthreads();
        unsigned long long before;
        const int bin = find_bin(S, 0, (int)(range >> sh), need - above, before,
                                 [&](int b) { return ((unsigned long long)hi[b] << 32) | lo[b]; });
        if (bin < 0) return false;
        above += (double)before;
        khi -= (uint32_t)bin << sh;
        if (sh == 0) { key_out = khi; return true; }
        const uint32_t width = (1u << sh) - 1u;
        klo = khi - klo > width ? khi - width : klo;
    }
}

// f(unit) for every 16-byte unit of a row, read again (from L2 for most rows); logits beyond the row: -inf
template <int DT, typename F>
__device__ __forceinline__ void visit_units(const stream::RowSpan &row, F f)
{
    const uint4 *src = reinterpret_cast<const uint4 *>(row.base);
    for (int u0 = threadIdx.x; u0 < row.units; u0 += NT * 4) {
        uint4 raw[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (u0 + c * NT < row.units) raw[c] = __ldg(src + u0 + c * NT);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int u = u0 + c * NT;
            if (u >= row.units) break;
            if (u == 0 || u == row.units - 1) stream::mask_unit<DT>(raw[c], u, row);
            f(raw[c]);
        }
    }
}
// f(z) for every logit of a row
template <int DT, typename F>
__device__ __forceinline__ void visit_row(const stream::RowSpan &row, F f)
{
    constexpr int E = DT == SPEC_BF16 ? 8 : 4;
    const uint4 *src = reinterpret_cast<const uint4 *>(row.base);
    for (int u = threadIdx.x; u < row.units; u += NT) {
        const uint4 raw = __ldg(src + u);
        const int e0 = u == 0 ? row.head : 0, e1 = u == row.units - 1 ? row.last : E;
        float z[E];
        stream::unpack_unit<DT>(raw, z);
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (k >= e0 && k < e1) f(z[k]);
    }
}

struct Kept {
    uint32_t key;      // key of the cut (0: nothing is cut)
    double Z, X;       // sum over the kept tokens of e and e x
};

// Selection and kept sums of a row the one pass could not settle: radix levels over the row in L2.  total: mass
// of the row in units of its largest e (top-p alone; it only narrows the first range).  Out of line: rare.
template <int DT>
__device__ __noinline__ Kept settle_from_row(Shared &S, uint32_t *bins, const stream::RowSpan row, int V, int top_k,
                                             float top_p, float m, float sf, float s_hi, float s_lo, float of, double total)
{
    uint32_t *lo = bins, *hi = bins + NB;
    const bool use_k = top_k > 0 && top_k < V, use_p = top_p < 1.f;
    const uint32_t key_m = cut::key_of(m);
    const auto visit = [&](auto g) { visit_row<DT>(row, [&](float z) { g(cut::key_of(z)); }); };
    Kept r = {0u, 0.0, 0.0};
    if (use_k && !radix_select<false>(S, lo, hi, (double)top_k, 0u, key_m, m, sf, r.key, visit)) r.key = 0u;
    if (use_p) {
        const uint32_t key_k = r.key;
        unsigned long long part = 0;
        visit_row<DT>(row, [&](float z) { if (cut::key_of(z) >= key_k) part += fix44(ex2_approx((z - m) * sf)); });
        const double target = (double)top_p * (double)block_sum(S, part);
        // no cut lies so far below the maximum that all tokens below it together could not make up 1 - top_p
        uint32_t from = key_k, key_p = 0u;
        if (total > 0.0 && top_p < 1.f) {
            const float w = log2f((float)V / ((1.f - top_p) * (float)total)) + 0.5f;
            from = max(key_k, cut::key_of(m - w / sf));
        }
        if (radix_select<true>(S, lo, hi, target, from, key_m, m, sf, key_p, visit) ||
            (from > key_k && radix_select<true>(S, lo, hi, target, key_k, key_m, m, sf, key_p, visit)))
            r.key = key_p;
        // (the set itself stays below the target by a rounding: the whole set is kept)
    }
    const float cutv = r.key == 0u ? -CUDART_INF_F : cut::value_of(r.key);
    double Z = 0.0, X = 0.0;
    visit_row<DT>(row, [&](float z) {
        if (z >= cutv) {
            const float x = fmaxf(fmaf(z, s_lo, fmaf(z, s_hi, -of)), -200.f);
            const float e = ex2_approx(x);
            Z += (double)e;
            X += (double)e * (double)x;
        }
    });
    Z = warp_sum(Z);
    X = warp_sum(X);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) { S.red[threadIdx.x >> 5][0] = Z; S.red[threadIdx.x >> 5][1] = X; }
    __syncthreads();
    for (int k = 0; k < NW; ++k) { r.Z += S.red[k][0]; r.X += S.red[k][1]; }
    __syncthreads();
    return r;
}

// The pieces of the kernel below that run once per row or now and then stay out of line: the loop over the slices then
// has its registers to itself (inlined, they made it spill, and with the ring in shared memory there is next to no
// first-level cache left to spill to: 1.9 against 1.3 ms on 12000 rows of 128256 logits).

// shared memory of the kernel
template <int DT> struct Smem {
    uint4 *ring;
    unsigned char *hits;         // the thread's warp's
    uint32_t *bins, *keys;       // keys: fp32 only
    Shared &S;
    __device__ __forceinline__ Smem()
        : ring(reinterpret_cast<uint4 *>(dyn_smem)), hits(dyn_smem + Layout<DT>::RING + (threadIdx.x >> 5) * UN * 32),
          bins(reinterpret_cast<uint32_t *>(dyn_smem + Layout<DT>::RING + Layout<DT>::HITS)), keys(bins + 2 * NB),
          S(*reinterpret_cast<Shared *>(dyn_smem + Layout<DT>::RING + Layout<DT>::HITS + Layout<DT>::BINS)) {}
};

// The first item from `id` on, in steps of the grid, whose row is read: every target row, the draft rows of nodes with
// children (every warp finds out by itself).
__device__ __noinline__ int next_read(const RParams &P, int id, int items)
{
    for (; id < items; id += gridDim.x) {
        if ((id & 1) == 0) break;
        const int row = id >> 1;
        if (P.parent && stream::has_children(P.parent + (row / P.N) * P.topo_stride, P.N, row % P.N, threadIdx.x & 31)) break;
    }
    return id;
}
template <int DT>
__device__ __forceinline__ stream::RowSpan span_of(const RParams &P, int id)
{
    const int row = id >> 1;
    return stream::row_span<DT>((id & 1) ? P.zq : P.zp, (row / P.N) * P.seq_stride + (row % P.N) * P.node_stride, P.V);
}

// top-k: a bound from the first slice (the k-th largest of its units' maxima mu; fp32: of the threads' maxima), or
// from the candidates so far.  All threads of the block.
template <int DT>
__device__ __noinline__ float first_bound(int top_k, const uint4 mu)
{
    const Smem<DT> M;
    if (DT == SPEC_BF16) {
        const uint32_t m[4] = {mu.x, mu.y, mu.z, mu.w};
        int at[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float v = stream::fold_max<DT>(m[c]);
            at[c] = v > LOWEST ? bin_of(v) : -1;
            if (at[c] >= 0) atomicAdd(&M.bins[at[c]], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            const int kb = top_k <= K_FAST<DT> ? warp_find<uint32_t>(bin_of(cut::value_of(M.S.runmax)), 2 * TB - 1, (double)top_k,
                                                                     [&](int i) { return M.bins[i]; }) : -1;
            if (threadIdx.x == 0) M.S.bound = kb > 0 && kb < 2 * TB - 1 && kb != TB && kb != TB - 1 ? value_of_bin(kb) : LOWEST;
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (at[c] >= 0) M.bins[at[c]] = 0u;
        __syncthreads();
        return M.S.bound;
    }
    // the k-th largest of the threads' maxima, to 16 bits of its key (a lower bound)
    const float ms = stream::fold_max<DT>(stream::max_raw<DT>(stream::max_raw<DT>(mu.x, mu.y), stream::max_raw<DT>(mu.z, mu.w)));
    const uint32_t k16 = cut::key_of(ms) >> 16;
    uint32_t t16 = 0;
    if (top_k <= K_FAST<DT>)
        for (int bit = 15; bit >= 0; --bit) {
            const uint32_t t = t16 | (1u << bit);
            if (__syncthreads_count(k16 >= t) >= top_k) t16 = t;
        }
    const float v = cut::value_of(t16 << 16);
    return t16 && v > LOWEST ? v : LOWEST;           // (false for the NaN of a row that will be reported)
}
template <int DT, bool TOTAL>
__device__ __noinline__ float tighter_bound(int top_k, float bound)
{
    const Smem<DT> M;
    Shared &S = M.S;
    const int tid = threadIdx.x;
    __syncthreads();                                  // all candidates of the slices so far are in
    if (DT == SPEC_BF16) {
        if (tid < 32) {
            const int kb = warp_find<uint32_t>(bin_of(cut::value_of(S.runmax)), 2 * TB - 1, (double)top_k, [&](int i) { return M.bins[i]; });
            if (tid == 0) S.bound = kb > 0 && kb < 2 * TB - 1 && kb != TB && kb != TB - 1 ? value_of_bin(kb) : LOWEST;
        }
        __syncthreads();
        return fmaxf(bound, S.bound);
    }
    // fp32: the list of keys is then compacted to what the bound still admits
    const int n = S.count;
    if (tid == 0) S.bound = bound;
    __syncthreads();
    bound = S.bound;
    if (n > CAP) return bound;
    uint32_t key = 0u;
    if (!TOTAL && n >= top_k &&
        radix_select<false>(S, M.bins, M.bins + NB, (double)top_k, 0u, 0xFFFFFFFFu, 0.f, 1.f, key, [&](auto g) {
            for (int i = tid; i < n; i += NT) g(M.keys[i]);
        }))
        bound = fmaxf(bound, cut::value_of(key));
    uint32_t keep[CAP / NT];
    const uint32_t kb = cut::key_of(bound);
#pragma unroll
    for (int j = 0; j < CAP / NT; ++j) keep[j] = tid + j * NT < n ? M.keys[tid + j * NT] : 0u;
    __syncthreads();
    if (tid == 0) S.count = 0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < CAP / NT; ++j)
        if (keep[j] >= kb) M.keys[atomicAdd(&S.count, 1)] = keep[j];
    __syncthreads();
    return bound;
}

// bf16 top-p: a bound from the n logits seen so far, whose candidates are in the bins down to `loose` (all threads
// have put theirs there): the cut these alone would have at a larger top-p.  m: their maximum; set / of / Sd: the
// thread's reference and sum of e.  Returns the bound; S.verdict: whether to count densely from it.
__device__ __noinline__ float mass_bound(float m, float loose, bool set, float of_t, double Sd, float top_p, float sf, double s_d, int n, int V)
{
    const Smem<SPEC_BF16> M;
    Shared &S = M.S;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int o_t = set ? (int)of_t : ROWPART_EMPTY;
    const int O_w = __reduce_max_sync(0xffffffffu, o_t);
    const double Sw = warp_sum(Sd * (double)pow2i(max(o_t - O_w, -127)));
    if (lane == 0) { S.red[w][0] = Sw; S.red[w][1] = (double)O_w; }
    __syncthreads();
    if (w == 0) {
        const int Ok = lane < NW ? (int)S.red[lane][1] : ROWPART_EMPTY;
        const int Om = __reduce_max_sync(0xffffffffu, Ok);
        double total = warp_sum(lane < NW ? S.red[lane][0] * (double)pow2i(max(Ok - Om, -127)) : 0.0);
        total *= (double)exp2f((float)((double)Om - (double)m * s_d));
        const int b_max = bin_of(m), b_lo = last_bin_above(loose);
        const int kb = warp_find<unsigned long long>(b_max, b_lo, (1.0 - (double)(SAMPLE_REST * (float)n / (float)V) * (1.0 - (double)top_p)) * total * cut::FIX, [&](int i) {
            const unsigned long long c = M.bins[i];
            return c ? c * fix44(ex2_approx((value_of_bin(i) - m) * sf)) : 0ull;
        });
        uint32_t c = 0;
        for (int i = b_max + lane; i <= (kb >= 0 ? kb : b_lo); i += 32) c += M.bins[i];
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) {
            S.bound = kb >= 0 && kb != TB && kb != TB - 1 ? value_of_bin(kb) : loose;
            S.verdict = (float)c > DENSE * (float)n ? 1 : 0;
        }
    }
    __syncthreads();
    return S.bound;
}
// the maximum of the block's logits so far, from the threads' maxima
__device__ __forceinline__ float block_max(Shared &S, float ms)
{
    const uint32_t km = __reduce_max_sync(0xffffffffu, cut::key_of(ms));
    if ((threadIdx.x & 31) == 0) atomicMax(&S.runmax, km);
    __syncthreads();
    return cut::value_of(S.runmax);
}
// the first slice (r0 .. r3, beyond the row: -inf) into the bins, and the first bound from it
__device__ __noinline__ float sample_bound(const uint4 r0, const uint4 r1, const uint4 r2, const uint4 r3, float ms, bool set,
                                           float of_t, double Sd, float top_p, int n, int V)
{
    const Smem<SPEC_BF16> M;
    Shared &S = M.S;
    const float m = block_max(S, ms);
    const float sf = S.sc.sf;
    const double s_d = S.sc.s_d;
    if (!(m > -CUDART_INF_F && m < CUDART_INF_F)) {       // nothing finite so far, or a row that will be reported
        if (threadIdx.x == 0) S.verdict = 1;
        __syncthreads();
        return LOWEST;
    }
    const float loose = fmaxf(m - SAMPLE_OCTAVES / sf, LOWEST);
    count_unit(M.bins, &S.odd, r0, loose, ms);
    count_unit(M.bins, &S.odd, r1, loose, ms);
    count_unit(M.bins, &S.odd, r2, loose, ms);
    count_unit(M.bins, &S.odd, r3, loose, ms);
    return mass_bound(m, loose, set, of_t, Sd, top_p, sf, s_d, n, V);
}

// what the pass over a row leaves in a thread
struct Pass {
    float tmax;                // the thread's maximum (NaN if it saw one)
    float of;                  // its integer reference, and its sum of e in units of 2^of (TOTAL)
    double Sd;
    bool set;
    float bound;               // the row is complete from it upwards (fp32 top-p: from the window upwards)
};

// The row's statistics from what the pass has set aside; leaves bins and counters as the next row wants them.
template <int DT, bool TOTAL>
__device__ __noinline__ void finish_row(const RParams &P, int id, const Pass ps)
{
    const Smem<DT> M;
    Shared &S = M.S;
    const Scale sc = S.sc;
    uint32_t *const bins = M.bins, *const keys = M.keys;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const bool use_k = P.top_k > 0 && P.top_k < P.V, use_p = P.top_p < 1.f;
    const float sf = sc.sf, s_hi = sc.s_hi, s_lo = sc.s_lo, window = sc.window;
    const double s_d = sc.s_d;
    RowPart *out = P.part + id;
    auto clear = [&]() {
        if (DT == SPEC_BF16)
            for (int i = tid; i < 2 * TB / 4; i += NT) reinterpret_cast<uint4 *>(bins)[i] = make_uint4(0, 0, 0, 0);
    };
    // ---- the row's maximum and mass; NaN / +inf ------------------------------------------------------------------
    float m;
    double total = 0.0;                // sum over the row of 2^((z - m) s)
    {
        const bool nan = ps.tmax != ps.tmax;
        float wm = ps.tmax;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
        int O_w = 0;
        double Sw = 0.0;
        if (TOTAL) {
            const int o_t = ps.set ? (int)ps.of : ROWPART_EMPTY;
            O_w = __reduce_max_sync(0xffffffffu, o_t);
            Sw = warp_sum(ps.Sd * (double)pow2i(max(o_t - O_w, -127)));
        }
        // (maximum and reference share a word pair: both are exact in fp32)
        if (lane == 0) { S.red[w][0] = Sw; S.red[w][1] = __hiloint2double(__float_as_int(wm), O_w); }
        const int any_nan = __syncthreads_or((int)nan);
        const double part = lane < NW ? S.red[lane][1] : __hiloint2double(__float_as_int(-CUDART_INF_F), ROWPART_EMPTY);
        const int Ok = __double2loint(part);
        m = __int_as_float(__double2hiint(part));
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        m = __shfl_sync(0xffffffffu, m, 0);
        if (any_nan || !(m > -CUDART_INF_F) || m == CUDART_INF_F) {
            if (tid == 0) {
                RowPart r = {};
                r.cut = -CUDART_INF_F; r.O = ROWPART_EMPTY; r.bad = 1;
                *out = r;
                P.cut[id] = -CUDART_INF_F;
            }
            __syncthreads();
            clear();
            if (tid == 0) { S.runmax = 0u; S.count = 0; S.odd = 0; }
            __syncthreads();
            return;
        }
        if (TOTAL && (DT == SPEC_F32 || w == 0)) {
            const int Om = __reduce_max_sync(0xffffffffu, Ok);
            total = warp_sum(lane < NW ? S.red[lane][0] * pow2d(max(Ok - Om, -1000)) : 0.0);
            // from units of 2^Om to units of the row maximum: 2^(Om - m s), Om - m s in [0, 1]
            const double d = (double)Om - (double)m * s_d;
            total *= 1.4142135623730951 * exp2_frac(fmin(fmax(d, 0.0), 1.0) - 0.5);
            if (lane == 0) S.total = total;
        }
    }
    const double Od = ceil((double)m * s_d);
    const float of = (float)fmin(fmax(Od, -1.0e9), 1.0e9);
    auto write = [&](double Z, double X, float cutv) {
        RowPart r;
        r.S = Z; r.X = X; r.O = (int)of; r.cut = cutv;
        r.xmax = (float)((double)m * s_d - (double)of);
        r.bad = 0;
        *out = r;
        P.cut[id] = cutv;
    };
    bool settled = false;
    if (DT == SPEC_BF16) {
        const int b_max = bin_of(m);
        // selection, kept sums and record by one warp, from bins that are complete down to b_lo; says whether it
        // could settle the row
        auto select = [&](int b_lo) {
            auto count = [&](int i) { return bins[i]; };
            auto mass = [&](int i) {
                const unsigned long long c = bins[i];
                return c ? c * fix44(ex2_approx((value_of_bin(i) - m) * sf)) : 0ull;
            };
            int b_cut = -1;
            if (TOTAL) {
                b_cut = warp_find<unsigned long long>(b_max, b_lo, (double)P.top_p * total * cut::FIX, mass);
            } else if (P.top_k <= K_FAST<DT>) {
                b_cut = warp_find<uint32_t>(b_max, b_lo, (double)P.top_k, count);
                if (use_p && b_cut >= 0) {
                    // the set's mass, exactly: its tokens are all in the bins
                    unsigned long long part = 0;
                    for (int i = b_max + lane; i <= b_cut; i += 32) part += mass(i);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
                    const int b_p = warp_find<unsigned long long>(b_max, b_cut, (double)P.top_p * (double)part, mass);
                    if (b_p >= 0) b_cut = b_p;       // (else the set itself stays below the target: rounding)
                }
            }
            if (b_cut < 0) return false;
            // (a shared bin among the kept ones holds values that the bins cannot tell apart)
            if (fabsf(m) >= HIGH || (S.odd & ODD_HIGH) || ((S.odd & ODD_LOW) && b_cut >= TB - 1)) return false;
            double Z = 0.0, X = 0.0;
            for (int i = b_max + lane; i <= b_cut; i += 32) {
                const uint32_t c = bins[i];
                if (c) {
                    const float z = value_of_bin(i);
                    const float x = fmaxf(fmaf(z, s_lo, fmaf(z, s_hi, -of)), -200.f);
                    const double e = (double)ex2_approx(x) * (double)c;
                    Z += e;
                    X += e * (double)x;
                }
            }
            Z = warp_sum(Z);
            X = warp_sum(X);
            if (lane == 0) write(Z, X, value_of_bin(b_cut));
            return true;
        };
        if (w == 0) {
            const bool ok = select(last_bin_above(ps.bound));
            if (lane == 0) S.verdict = ok ? 1 : 0;
        }
        __syncthreads();
        settled = S.verdict != 0;
        if (TOTAL && !settled) {
            total = S.total;
            // The nucleus reaches below the bound.  All tokens more than log2(V / ((1 - top_p) total)) octaves
            // below the maximum together have no more than 1 - top_p of the mass: counted again, from L2, down
            // to there.
            const float wide = log2f((float)P.V / ((1.f - P.top_p) * (float)total)) + 0.01f;
            const float bound2 = fmaxf(m - wide / sf, LOWEST);
            clear();
            __syncthreads();
            visit_units<DT>(span_of<DT>(P, id), [&](const uint4 &r) { count_unit(bins, &S.odd, r, bound2, m); });
            __syncthreads();
            if (w == 0) {
                const bool ok = select(last_bin_above(bound2));
                if (lane == 0) S.verdict = ok ? 1 : 0;
            }
            __syncthreads();
            settled = S.verdict != 0;
        }
    } else {
        // ---- fp32: radix selection on the list of candidates --------------------------------------------------
        const int n = S.count;
        auto visit = [&](auto g) { for (int i = tid; i < n; i += NT) g(keys[i]); };
        uint32_t key = 0u;
        float cutv = -CUDART_INF_F;
        double Z = 0.0, X = 0.0;
        settled = n <= CAP && (TOTAL || P.top_k <= K_FAST<DT>);
        // (at least k logits lie at or above the bound, so the k-th largest is in the list)
        if (settled && use_k) settled = radix_select<false>(S, bins, bins + NB, (double)P.top_k, 0u, cut::key_of(m), m, sf, key, visit);
        if (settled && use_p) {
            const uint32_t key_k = key;        // the set: key >= key_k (0: the whole row)
            double target = (double)P.top_p * total * cut::FIX;
            if (!TOTAL) {
                unsigned long long part = 0;
                visit([&](uint32_t k) { if (k >= key_k) part += fix44(ex2_approx((cut::value_of(k) - m) * sf)); });
                target = (double)P.top_p * (double)block_sum(S, part);
            }
            // complete from the final bound upwards only
            const uint32_t from = TOTAL ? cut::key_of(m - window) : key_k;
            uint32_t key_p = 0u;
            if (radix_select<true>(S, bins, bins + NB, target, from, cut::key_of(m), m, sf, key_p, visit)) key = key_p;
            else settled = !TOTAL;             // TOTAL: the nucleus reaches below the window; else: the whole set (rounding)
        }
        settled = settled && key != 0u;
        if (settled) {
            cutv = cut::value_of(key);
            for (int i = tid; i < n; i += NT)
                if (keys[i] >= key) {
                    const float z = cut::value_of(keys[i]);
                    const float x = fmaxf(fmaf(z, s_lo, fmaf(z, s_hi, -of)), -200.f);
                    const double e = (double)ex2_approx(x);
                    Z += e;
                    X += e * (double)x;
                }
        }
        if (settled) {
            Z = warp_sum(Z);
            X = warp_sum(X);
            __syncthreads();
            if (lane == 0) { S.red[w][0] = Z; S.red[w][1] = X; }
            __syncthreads();
            Z = X = 0.0;
            if (tid == 0) {
                for (int k = 0; k < NW; ++k) { Z += S.red[k][0]; X += S.red[k][1]; }
                write(Z, X, cutv);
            }
        }
    }
    if (!settled) {
        const Kept kp = settle_from_row<DT>(S, bins, span_of<DT>(P, id), P.V, P.top_k, P.top_p, m, sf, s_hi, s_lo, of, total);
        if (tid == 0) write(kp.Z, kp.X, kp.key ? cut::value_of(kp.key) : -CUDART_INF_F);
    }
    clear();
    if (tid == 0) { S.runmax = 0u; S.count = 0; S.odd = 0; }
    __syncthreads();             // the bins, counters and partials are free for the next row
}

// TOTAL: top-p without top-k (the pass also sums the mass of the whole row)
template <int DT, bool TOTAL>
__global__ void __launch_bounds__(NT, CTAS<DT>) spec_row_trunc_kernel(const __grid_constant__ RParams P)
{
    constexpr int E = DT == SPEC_BF16 ? 8 : 4;           // logits of a unit
    const Smem<DT> M;
    Shared &S = M.S;
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t ring_s = smem_u32(M.ring) + tid * 16u;
    const unsigned lt = (1u << lane) - 1u;
    const int items = 2 * P.B * P.N;           // (at most 2^25: the host checks B N)
    grid_launch_dependents();

    if (DT == SPEC_BF16) for (int i = tid; i < 2 * TB; i += NT) M.bins[i] = 0;
    if (tid == 0) { S.runmax = 0u; S.count = 0; S.odd = 0; }
    __syncthreads();

    // ---- the copying side of the ring: DEPTH - 1 slices ahead, across rows ----------------------------------
    int i_id = (int)blockIdx.x - (int)gridDim.x;
    const unsigned char *i_src = nullptr;
    int i_left = -tid, i_stage = 0;       // units of the row from the thread's next one on; the stage it goes to
    bool i_more = true;
    auto issue = [&]() {
        if (i_more && i_left + tid <= 0) {
            i_id = next_read(P, i_id + gridDim.x, items);
            i_more = i_id < items;
            if (i_more) {
                const stream::RowSpan r = span_of<DT>(P, i_id);
                i_src = r.base + (size_t)tid * 16;
                i_left = r.units - tid;
            }
        }
        if (i_more) {
            const uint32_t dst = ring_s + (uint32_t)(i_stage * UN * NT) * 16u;
#pragma unroll
            for (int c = 0; c < UN; ++c)
                if (c * NT < i_left) stream::cp_async16(dst + (uint32_t)(c * NT) * 16u, i_src + (size_t)(c * NT) * 16, 16);
            i_src += (size_t)UN * NT * 16;
            i_left -= UN * NT;
            i_stage = i_stage + 1 == DEPTH ? 0 : i_stage + 1;
        }
        stream::cp_async_commit();
    };
    for (int k = 0; k < DEPTH - 1; ++k) issue();

    int c_stage = 0;
    float T_now = 0.f, s_hi = 0.f, s_lo = 0.f, window = 0.f;      // of the current temperature
    for (int id = blockIdx.x; id < items; id += gridDim.x) {
        // ---- rows that are not read, up to the next one that is --------------------------------------------------
        const int to = next_read(P, id, items);
        for (; id < min(to + 1, items); id += gridDim.x) {
            if (tid == 0) {
                const int node = id >> 1;
                if ((id & 1) == 0) P.init.set(node, node / P.N, node % P.N);
                if (id < to) {
                    RowPart r = {};
                    r.cut = -CUDART_INF_F; r.O = ROWPART_EMPTY; r.bad = -1;
                    P.part[id] = r;
                    P.cut[id] = -CUDART_INF_F;
                }
            }
            if (id == to) break;
        }
        if (id >= items) break;
        const stream::RowSpan row = span_of<DT>(P, id);
        const float T = P.T_seq ? __ldg(P.T_seq + (id >> 1) / P.N) : P.T;
        if (T != T_now) {                      // (the block agrees; the scale factors are next read after a barrier)
            T_now = T;
            const double s_d = 1.4426950408889634 / (double)T;
            stream::split_scale(s_d, s_hi, s_lo);
            if (tid == 0) {
                const float sf = 1.4426950408889634f / T;
                S.sc = Scale{T, sf, s_hi, s_lo, WINDOW_OCTAVES / sf, s_d};
            }
            window = WINDOW_OCTAVES / (1.4426950408889634f / T);
        }
        // ---- the pass ------------------------------------------------------------------------------------------
        Pass ps = {-CUDART_INF_F, 0.f, 0.0, false, LOWEST};
        bool dense = false;                // bf16 top-p: count every logit on the spot
        const int nsl = (row.units + NT * UN - 1) / (NT * UN);
        for (int sl = 0; sl < nsl; ++sl) {
            if (!(DT == SPEC_BF16 && TOTAL) && nsl > sl + 2 && (sl == 2 || sl == 6 || (DT == SPEC_F32 && sl == 16))) {
                // a better bound, from the slices so far
                ps.bound = tighter_bound<DT, TOTAL>(P.top_k, ps.bound);
            }
            stream::cp_async_wait<DEPTH - 2>();
            issue();                                    // into the stage of the previous iteration
            uint4 *const stage = M.ring + c_stage * UN * NT + (tid & ~31);      // the warp's share of the slice
            c_stage = c_stage + 1 == DEPTH ? 0 : c_stage + 1;
            uint4 raw[UN];
#pragma unroll
            for (int c = 0; c < UN; ++c) raw[c] = stage[c * NT + lane];
            if (sl == 0 || sl == nsl - 1) {
#pragma unroll
                for (int c = 0; c < UN; ++c) {
                    stream::mask_unit<DT>(raw[c], (sl * UN + c) * NT + tid, row);
                    stage[c * NT + lane] = raw[c];
                }
            }
            // the units' maxima (bf16: still as pairs) and the thread's maximum of the slice; a NaN stays
            uint32_t mu[UN];
#pragma unroll
            for (int c = 0; c < UN; ++c) mu[c] = stream::unit_max_raw<DT>(raw[c]);
            const float ms = stream::fold_max<DT>(stream::max_raw<DT>(stream::max_raw<DT>(mu[0], mu[1]), stream::max_raw<DT>(mu[2], mu[3])));
            static_assert(UN == 4, "slice maximum of four units");
            if (TOTAL && ms > -CUDART_INF_F && ms < CUDART_INF_F) {
                // the row's mass, as in the streaming statistics kernel: a running integer reference per
                // thread, fp32 sums of a slice's logits, fp64 above
                const float onew = fminf(fmaxf(ceilf(ms * s_hi), -1.0e9f), 1.0e9f);
                if (!ps.set) { ps.of = onew; ps.set = true; }
                else if (onew > ps.of) { ps.Sd *= (double)pow2i((int)fmaxf(ps.of - onew, -127.f)); ps.of = onew; }
                unsigned long long acc[2] = {0ull, 0ull};
                const unsigned long long sh2 = pack_f32x2(s_hi, s_hi), sl2 = pack_f32x2(s_lo, s_lo), no2 = pack_f32x2(-ps.of, -ps.of);
#pragma unroll
                for (int c = 0; c < UN; ++c) {
                    float z[E];
                    stream::unpack_unit<DT>(raw[c], z);
#pragma unroll
                    for (int k = 0; k < E; k += 2) {
                        const unsigned long long z2 = pack_f32x2(z[k], z[k + 1]);
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(z2, sl2, fma_f32x2(z2, sh2, no2)), x0, x1);
                        acc[c & 1] = add_f32x2(acc[c & 1], pack_f32x2(ex2_approx(x0), ex2_approx(x1)));
                    }
                }
                float a0, a1;
                unpack_f32x2(add_f32x2(acc[0], acc[1]), a0, a1);
                ps.Sd += (double)(a0 + a1);
            }
            // ---- the running maximum and the bound ----------------------------------------------------------------
            if (DT == SPEC_BF16 && TOTAL) {
                if (sl == 0) {
                    ps.tmax = ms;
                    ps.bound = sample_bound(raw[0], raw[1], raw[2], raw[3], ms, ps.set, ps.of, ps.Sd, P.top_p, min(P.V, UN * NT * E), P.V);
                    dense = S.verdict != 0;
                    continue;                           // (the first slice is in the bins)
                }
            } else {
                if (sl == 0) {
                    const uint32_t km = __reduce_max_sync(0xffffffffu, cut::key_of(ms));
                    if (lane == 0) atomicMax(&S.runmax, km);
                    if (TOTAL) __syncthreads();
                    else ps.bound = first_bound<DT>(P.top_k, make_uint4(mu[0], mu[1], mu[2], mu[3]));
                } else if (ms > ps.tmax && ms > cut::value_of(*(volatile uint32_t *)&S.runmax)) {
                    atomicMax(&S.runmax, cut::key_of(ms));
                }
                if (TOTAL) ps.bound = fmaxf(cut::value_of(*(volatile uint32_t *)&S.runmax) - window, LOWEST);
            }
            ps.tmax = stream::max_nan(ps.tmax, ms);
            // ---- candidates ----------------------------------------------------------------------------------
            if (DT == SPEC_BF16 && TOTAL && dense) {
#pragma unroll
                for (int c = 0; c < UN; ++c) count_unit(M.bins, &S.odd, raw[c], ps.bound, ms);
            } else if (__any_sync(0xffffffffu, ms >= ps.bound)) {
                int n = 0;
#pragma unroll
                for (int c = 0; c < UN; ++c) {
                    const bool in = stream::fold_max<DT>(mu[c]) >= ps.bound;
                    const unsigned bal = __ballot_sync(0xffffffffu, in);
                    if (in) M.hits[n + __popc(bal & lt)] = (unsigned char)(c * 32 + lane);
                    n += __popc(bal);
                }
                __syncwarp();
                for (int i0 = 0; i0 < n * E; i0 += 32) {          // a logit per lane
                    const int i = i0 + lane;
                    const bool on = i < n * E;
                    const int u = on ? M.hits[i / E] : 0;
                    const uint4 *unit = stage + (u >> 5) * NT + (u & 31);
                    if (DT == SPEC_BF16) {
                        const uint32_t u16 = on ? reinterpret_cast<const unsigned short *>(unit)[i % E] : 0xFF80u;
                        if (__uint_as_float(u16 << 16) >= ps.bound) count_value(M.bins, &S.odd, u16);
                    } else {
                        const float z = on ? reinterpret_cast<const float *>(unit)[i % E] : -CUDART_INF_F;
                        const bool in = z >= ps.bound;
                        const unsigned bal = __ballot_sync(0xffffffffu, in);
                        if (!bal) continue;
                        int base = 0;
                        if (lane == 0) base = atomicAdd(&S.count, __popc(bal));
                        const int pos = __shfl_sync(0xffffffffu, base, 0) + __popc(bal & lt);
                        if (in && pos < CAP) M.keys[pos] = cut::key_of(z);
                    }
                }
                __syncwarp();
            }
        }
        finish_row<DT, TOTAL>(P, id, ps);
    }
    stream::cp_async_wait<0>();
}

}  // namespace trunc
}  // namespace specv
