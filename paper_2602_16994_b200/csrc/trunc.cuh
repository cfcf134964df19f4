// Row statistics for truncated sampling distributions (top-k / top-p; rules in cut.cuh).
//
// The nucleus of a row is a few dozen to a few thousand tokens out of 10^5, and its cut is a VALUE, so the
// selection need not keep the row.  One CTA per row; the row is streamed once from HBM through a ring of
// asynchronous copies, and while it passes every logit at or above a running BOUND that is known to lie below
// the cut is set aside as a CANDIDATE:
//   top-k        bound = the k-th largest of the units' maxima in the first slice (each is a logit of the row, so
//                at least k logits lie at or above it), tightened to the k-th largest candidate so far a few times;
//   top-p alone  the mass of the whole row, which fixes the target, is summed in the same pass; bf16: bound = the cut that the first
//                slices alone would have at a larger top-p, after 1, 4 and 16 of them (a guess: the end of the row tells
//                whether the nucleus stayed above it); fp32: WINDOW_OCTAVES below the row's running maximum.
// bf16 candidates become counts in a histogram over logit VALUES (a bf16 logit has 16 bits: 20 octaves of
// magnitude, both signs, are 5120 bins), from which both cuts and all kept sums follow: the mass of a bin is
// its count times the mass of its value, and no number of candidates overflows it.  fp32 candidates become a
// list of keys (4096 entries) for a radix selection.
// How candidates are found: top-k (a few hundred per row) and fp32: one packed maximum per 16-byte unit finds the units that hold one;
// a warp lists those of its share of a slice and then looks at their logits, a logit per lane, in the ring.  bf16 top-p, with a
// few per cent of candidates or (T near 1 with top-p near 1) a quarter of the row: all logits of a unit that holds
// one anywhere in the warp are counted, without a branch (count_unit).
// A bf16 nucleus that reaches below the bound is counted again from L2, down to one that the row's mass guarantees.
// What is left over (fp32 nuclei beyond the list, k above 1024 (fp32: 256), values outside the 20 octaves) runs an adaptive
// radix selection over the row in L2, in the same CTA.
//
// top-k is bound by HBM for large batches; the ring runs ahead across rows, so the copies of the next row are in flight
// while the selection of the current one (a few microseconds of scans) runs.  top-p is bound by instructions: per logit 4.4 for its mass,
// 2.5 where it is counted, about 5 for ring, maxima and tests.  Row statistics of 2368 rows of 151936 (T 0.6, top-p 0.95): 341 -> 286 us;
// 272 rows of 128256 (T 1, top-p 0.99, nuclei of 30000): 97 -> 51 us, since every logit of a slice is counted by
// multiply-adds and not by branches, and the bound rises as the row goes by.
#pragma once
#include <cuda_bf16.h>

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
constexpr int CAP = 4096;            // fp32: candidate keys per row
constexpr float WINDOW_OCTAVES = 14.f;
constexpr float SAMPLE_OCTAVES = 24.f;   // bf16 top-p: how far below its maximum the first slice is counted
constexpr float SAMPLE_REST = 0.7f;      // safety factor of the bounds from a part of the row (mass_bound)
constexpr float UNSET = -2.0e9f;
// a bound that every finite logit passes but the lowest values of both types (masks: a row that keeps some of them is settled from L2)
constexpr float LOWEST = -3.3e38f;
template <int DT> constexpr int K_FAST = DT == SPEC_BF16 ? UN * NT : NT;      // largest top-k the first slice can bound

// bf16 value bins, largest value first: TB positive magnitudes, then TB negative ones; magnitudes below 2^-11
// share the two bins in the middle (0 itself in the first of them), those of 2^9 and more the outermost ones
constexpr int TB = 20 * 128;
constexpr int M0 = (127 - 11) << 7;
constexpr float HIGH = 508.f;                 // below the outermost bin's value
constexpr int PLAIN_KEY = M0 + 33;            // the smallest value that has 32 values with bins of their own below it, as bits
constexpr int PLAIN_NEG = M0 + TB - 2 - 32;   // ... and, of negative ones, the largest magnitude
constexpr float NEGATIVE = -4.8828125e-4f;    // -2^-11: the negative values below have bins of their own
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
    int *kept;                 // spec_tree_probs: number of kept tokens of every row and its largest logit as bits [B*N][2]; else NULL
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
    int verdict;               // bf16: what a selecting warp found, or see mass_bound
    float bound;               // fp32 top-p: the block's bound
    unsigned inner[SPEC_MAX_NODES / 32];       // one tree for all: its nodes with children
    uint32_t runmax;           // key of the largest logit seen by the row so far
    int count;                 // fp32: candidates appended (may exceed CAP: overflow)
    int odd;
    int sel_bin;
    unsigned long long sel_before;
};
template <int DT> struct Layout {
    static constexpr int RING = DEPTH * UN * NT * 16;
    // a byte per unit of a warp's share of a slice; bf16 top-p: a word per lane (count_unit)
    static constexpr int HITS = NW * UN * 32;
    // bf16: counts of 2 TB values; fp32: a radix histogram (64-bit bins as two words) and the candidate keys
    static constexpr int BINS = DT == SPEC_BF16 ? 2 * TB * 4 : NB * 8 + CAP * 4;
    static constexpr int BYTES = RING + HITS + BINS + (int)sizeof(Shared);
};
static_assert(2 * TB * 4 >= NB * 8, "the radix histogram of the slow path fits in the value bins");
template <int DT> constexpr int CTAS = DT == SPEC_BF16 ? 3 : 2;       // per SM
static_assert(Layout<SPEC_BF16>::BYTES <= (228 * 1024) / 3 - 1024 && Layout<SPEC_F32>::BYTES <= 113 * 1024, "CTAs per SM");

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
// bf16 values as integers in their order, -0 and +0 alike: the smallest that is at or above `bound` (one above -inf)
__device__ __forceinline__ int bound_key(float bound)
{
    const uint32_t u = __float_as_uint(bound);
    const int mag = (int)(u >> 16) & 0x7FFF;
    if (!(u >> 31)) return mag + ((u & 0xFFFFu) ? 1 : 0);
    return mag ? -1 - mag : 0;
}
// What the counting of bf16 logits needs to know about a bound.
struct Counter {
    int kb;                    // the bound as a key
    // Logits below this one are counted the plain way (count_unit): the bound and the 32 keys below it are values of one sign with
    // bins of their own, and so are the candidates: positive ones below HIGH, or, where the bound is negative, negative ones.
    __device__ __forceinline__ bool positive() const { return kb >= PLAIN_KEY; }
    __device__ __forceinline__ float plain_below() const
    {
        return positive() ? HIGH : kb < -1 - M0 && kb >= -1 - PLAIN_NEG ? NEGATIVE : -CUDART_INF_F;
    }
    // whether a unit with these maxima holds a candidate
    __device__ __forceinline__ bool reaches(uint32_t max_pair) const
    {
        const uint32_t pair = (uint32_t)(kb >= 0 ? kb : 0x8000 | (-1 - kb)) * 0x10001u;
        return __hge2_mask(reinterpret_cast<const __nv_bfloat162 &>(max_pair), reinterpret_cast<const __nv_bfloat162 &>(pair)) != 0u;
    }
};
// Counts the 8 logits of a bf16 unit that are at or above the bound.  Every lane adds to some word for each of its logits: an
// addition under a predicate is a branch to the compiler, and a slice of 8192 logits then takes 1310 cycles with no candidate
// and 2150 with 9 to 49 % of them (one CTA of 8 warps on an SM); without, 675 and 760 to 900.
// plain (no logit of the unit reaches plain_below): values of one sign order like their bits, or the other way round, so a logit below the
// bound is raised to one of the 32 keys below it, whose bins nobody reads any more (bounds only rise), and a pair of
// logits takes one maximum (negative: minimum), two multiply-adds and the two additions.  Logits that are all negative (log-probabilities),
// counted one by one: 272 rows of 128256 shifted by -20, T 1, top-p 0.99: 124 us, 76 rows (T 0.8, top-p 0.9): 72; now 78 and 39.
__device__ __forceinline__ void count_unit(const Counter &C, uint32_t bins, uint32_t dump, int *odd, const uint4 &r, bool plain)
{
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
    if (plain && C.kb < 0) {
        // bits 0x8000 + magnitude, as a 16-bit integer magnitude - 0x8000
        const int base = (int)bins + (TB - M0 + 0x8000) * 4;
        const uint32_t ceiling = (uint32_t)(0x8000 - C.kb + (int)(threadIdx.x & 31)) * 0x10001u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t v;
            asm("min.s16x2 %0, %1, %2;" : "=r"(v) : "r"(w[k]), "r"(ceiling));
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(__dp2a_lo((int)v, 0x0004, base)) : "memory");     // base + 4 low half
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(__dp2a_lo((int)v, 0x0400, base)) : "memory");     // base + 4 high half
        }
    } else if (plain) {
        const int base = (int)bins + (TB - 1 + M0) * 4;
        const uint32_t floor = (uint32_t)(C.kb - 1 - (int)(threadIdx.x & 31)) * 0x10001u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t v;
            asm("max.s16x2 %0, %1, %2;" : "=r"(v) : "r"(w[k]), "r"(floor));
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(__dp2a_lo((int)v, 0x00FC, base)) : "memory");     // base - 4 low half
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(__dp2a_lo((int)v, 0xFC00, base)) : "memory");     // base - 4 high half
        }
    } else {
        int seen = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int v = (k & 1) ? (int)w[k >> 1] >> 16 : (int)(short)w[k >> 1];
            int key = v ^ ((v >> 31) & 0x7FFF);
            key += key == -1 ? 1 : 0;
            const int mag = key < 0 ? -1 - key : key;
            const int b = key >= 0 ? max(min(TB - 1 + M0 - key, TB - 1), 0) : min(max(TB - M0 + mag, TB), 2 * TB - 1);
            if (key >= C.kb) seen |= (mag - 1 < M0 && mag > 0 ? ODD_LOW : 0) | (mag >= M0 + TB - 1 ? ODD_HIGH : 0);
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(key >= C.kb ? bins + 4u * (uint32_t)b : dump) : "memory");
        }
        if (seen) atomicOr(odd, seen);
    }
}

__device__ __forceinline__ void count_value(uint32_t *cnt, int *odd, uint32_t u16)
{
    int t;
    const int b = bin_of(u16, t);
    if ((unsigned)(t - 1) >= (unsigned)(TB - 2) && (u16 & 0x7FFFu)) atomicOr(odd, t ? ODD_HIGH : ODD_LOW);
    atomicAdd(&cnt[b], 1u);
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
// stays below.  before: the sum of the bins ahead of it.  All threads of the block call it and get the answer.  Every thread takes a run
// of an odd number of bins (consecutive lanes then read different banks) and goes through it a second time where the target lies in it.
template <typename T, typename F>
__device__ __forceinline__ int find_bin(Shared &S, int b0, int b1, double target, T &before, F weight)
{
    static_assert(sizeof(T) <= 8, "fits the slot");
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int per = ((b1 - b0) / NT + 1) | 1, i0 = b0 + tid * per, i1 = min(i0 + per - 1, b1);
    T sum = 0;
    for (int i = i0; i <= i1; ++i) sum += weight(i);
    T incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    T *tot = reinterpret_cast<T *>(S.warp_tot), *sel = reinterpret_cast<T *>(&S.sel_before);
    __syncthreads();
    if (lane == 31) tot[w] = incl;
    if (tid == 0) { S.sel_bin = -1; *sel = 0; }
    __syncthreads();
    T run = incl - sum;
    for (int k = 0; k < w; ++k) run += tot[k];
    if ((double)run < target && (double)(run + sum) >= target) {
        for (int i = i0; i <= i1; ++i) {
            const T x = weight(i);
            if ((double)(run + x) >= target) { S.sel_bin = i; *sel = run; break; }
            run += x;
        }
    }
    __syncthreads();
    before = *sel;
    return S.sel_bin;
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
        const int bin = find_bin<unsigned long long>(S, 0, (int)(range >> sh), need - above, before,
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
// f(z) for every logit of a row.  fp32, whose wide nuclei are settled this way: the load of the unit after next is under way while a unit is
// gone through; one at a time, a pass waited for L2 at every unit (T 1, top-p 0.99, 76 rows of 50257: 225 us, now 207; 272
// rows of 128256: 1099, now 1000).  (For bf16, where it is rare, the registers that this takes are missing in the loop over the slices: 541
// instead of 511 us on 2368 rows.)
template <int DT, typename F>
__device__ __forceinline__ void visit_row(const stream::RowSpan &row, F f)
{
    constexpr int E = DT == SPEC_BF16 ? 8 : 4;
    constexpr bool AHEAD = DT == SPEC_F32;
    const uint4 *src = reinterpret_cast<const uint4 *>(row.base);
    int u = threadIdx.x;
    uint4 raw = {}, next = {};
    if (AHEAD && u < row.units) raw = __ldg(src + u);
    if (AHEAD && u + NT < row.units) next = __ldg(src + u + NT);
#pragma unroll 1
    for (; u < row.units; u += NT) {
        uint4 far = {};
        if (!AHEAD) raw = __ldg(src + u);
        else if (u + 2 * NT < row.units) far = __ldg(src + u + 2 * NT);
        const int e0 = u == 0 ? row.head : 0, e1 = u == row.units - 1 ? row.last : E;
        float z[E];
        stream::unpack_unit<DT>(raw, z);
#pragma unroll
        for (int k = 0; k < E; ++k)
            if (k >= e0 && k < e1) f(z[k]);
        if (AHEAD) { raw = next; next = far; }
    }
}

// adds c tokens of logit z to a row's kept sums, in fp64: the sums are shared by all that is made of the row
__device__ __forceinline__ void add_kept(double z, double c, double s_d, double O, double &Z, double &X)
{
    const double x = fmax(z * s_d - O, -200.0), n = rint(x), e = c * exp2_frac_once(x - n) * pow2d((int)n);
    Z += e;
    X += e * x;
}
// a row's reference: an integer within 1e9 that is a float as well, because the verification kernels take it for one
__device__ __forceinline__ double reference(double largest) { return (double)(float)fmin(fmax(ceil(largest), -1.0e9), 1.0e9); }

struct Kept {
    uint32_t key;      // key of the cut (0: nothing is cut)
    double Z, X;       // sum over the kept tokens of e and e x
    int n;             // their number
};

// Selection and kept sums of a row the one pass could not settle: radix levels over the row in L2.  total: mass
// of the row in units of its largest e (top-p alone; it only narrows the first range; 0: not known).  own: the sums' unit is the largest
// e as well.  Out of line: rare.
template <int DT>
__device__ __noinline__ Kept settle_from_row(Shared &S, uint32_t *bins, const stream::RowSpan row, int V, int top_k,
                                             float top_p, float m, float sf, float s_hi, float s_lo, double s_d, bool own, double total)
{
    uint32_t *lo = bins, *hi = bins + NB;
    const bool use_k = top_k > 0 && top_k < V, use_p = top_p < 1.f;
    const uint32_t key_m = cut::key_of(m);
    const auto visit = [&](auto g) { visit_row<DT>(row, [&](float z) { g(cut::key_of(z)); }); };
    Kept r = {0u, 0.0, 0.0, 0};
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
    int n = 0;
    const double base = own ? (double)m : 0.0, O = own ? 0.0 : reference((double)m * s_d);
    const bool far = own || fabs(O) > FAR_EXPONENT;
    const float of = (float)O;
    visit_row<DT>(row, [&](float z) {
        if (z >= cutv) {
            const float x = fmaxf(fmaf(z, s_lo, fmaf(z, s_hi, -of)), -200.f);
            ++n;
            if (far || x > -4.f) {                     // (there may be as many tokens as the row has: only the largest in fp64)
                add_kept((double)z - base, 1.0, s_d, O, Z, X);
            } else {
                const float e = exp2_fine(z, s_hi, s_lo, (int)of);
                Z += (double)e;
                X += (double)e * (double)x;
            }
        }
    });
    r.n = (int)block_sum(S, (unsigned long long)n);
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
        : ring(reinterpret_cast<uint4 *>(dyn_smem)),
          hits(dyn_smem + Layout<DT>::RING + (threadIdx.x >> 5) * UN * 32),
          bins(reinterpret_cast<uint32_t *>(dyn_smem + Layout<DT>::RING + Layout<DT>::HITS)), keys(bins + 2 * NB),
          S(*reinterpret_cast<Shared *>(dyn_smem + Layout<DT>::RING + Layout<DT>::HITS + Layout<DT>::BINS)) {}
    __device__ __forceinline__ void count(const Counter &c, const uint4 &r, bool plain) const
    {
        count_unit(c, smem_u32(bins), smem_u32(hits) + (threadIdx.x & 31) * 4, &S.odd, r, plain);
    }
};

// row / N and row % N for row < 2^24
struct Split {
    int b, a;
    __device__ __forceinline__ Split(int row, int N, float inv)
    {
        b = (int)((float)row * inv);                 // (off by one at most)
        a = row - b * N;
        if (a < 0) { --b; a += N; }
        if (a >= N) { ++b; a -= N; }
    }
};
// The first item from `id` on, in steps of the grid, whose row is read: every target row, the draft rows of nodes with
// children (one tree for all: from the block's list; else every warp finds out by itself).
__device__ __noinline__ int next_read(const RParams &P, int id, int items, const unsigned *inner)
{
    const float inv = 1.f / (float)P.N;
    for (; id < items; id += gridDim.x) {
        if ((id & 1) == 0) break;
        if (!P.parent) continue;
        const Split r(id >> 1, P.N, inv);
        if (P.topo_stride == 0 ? (inner[r.a >> 5] >> (r.a & 31)) & 1u
                               : stream::has_children(P.parent + r.b * P.topo_stride, P.N, r.a, threadIdx.x & 31)) break;
    }
    return id;
}
template <int DT>
__device__ __forceinline__ stream::RowSpan span_of(const RParams &P, int id)
{
    const Split r(id >> 1, P.N, 1.f / (float)P.N);
    return stream::row_span<DT>((id & 1) ? P.zq : P.zp, r.b * P.seq_stride + r.a * P.node_stride, P.V);
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

// bf16 top-p: a bound from the n logits seen so far, whose candidates are in the bins down to `bound`: where the tokens below it, taken
// for the whole row, would together fall short of 1 - top_p of the mass seen so far (SAMPLE_REST of it).  That mass only
// grows, so the guess fails only where the first part of a row holds fewer of its light tokens than the rest; it
// gets better as V / n goes to 1, hence it is made again after 4 and 16 slices.  All threads of the block; tmax, of, Sd: what the
// thread has seen (Pass).  S.verdict = 1: the bins hold so little of the mass seen so far that the cut can't be expected above `bound`.
__device__ __noinline__ float mass_bound(float tmax, float bound, float of, double Sd, float top_p, int n, int V)
{
    const Smem<SPEC_BF16> M;
    Shared &S = M.S;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float sf = S.sc.sf;
    const int o_t = of > UNSET ? (int)of : ROWPART_EMPTY;
    const int O_w = __reduce_max_sync(0xffffffffu, o_t);
    const double Sw = warp_sum(Sd * (double)pow2i(max(o_t - O_w, -127)));
    const uint32_t km = __reduce_max_sync(0xffffffffu, cut::key_of(tmax));
    if (lane == 0) { S.red[w][0] = Sw; S.red[w][1] = __hiloint2double((int)km, O_w); }
    __syncthreads();                                  // all candidates so far are in
    const double part = S.red[lane & (NW - 1)][1];
    const float m = cut::value_of(__reduce_max_sync(0xffffffffu, (uint32_t)__double2hiint(part)));
    if (!(m > -CUDART_INF_F && m < CUDART_INF_F)) {       // nothing finite so far, or a row that will be reported
        __syncthreads();                              // (the partials may be written again)
        if (threadIdx.x == 0) S.verdict = 1;
        __syncthreads();
        return bound;
    }
    const int Ok = __double2loint(part), Om = __reduce_max_sync(0xffffffffu, Ok);
    double total = lane < NW ? S.red[lane][0] * (double)pow2i(max(Ok - Om, -127)) : 0.0;
    total = warp_sum(total) * (double)exp2f((float)((double)Om - (double)m * S.sc.s_d));
    const double need = (1.0 - (double)(SAMPLE_REST * (float)n / (float)V) * (1.0 - (double)top_p)) * total;
    const auto mass = [&](int i) {
        const uint32_t c = M.bins[i];
        return c ? (double)((float)c * ex2_approx((value_of_bin(i) - m) * sf)) : 0.0;
    };
    double before;
    const int b1 = last_bin_above(bound);
    const int kb = find_bin<double>(S, bin_of(m), b1, need, before, mass);
    if (kb < 0) {
        const int enough = find_bin<double>(S, bin_of(m), b1, (1.0 - 0.5 * (1.0 - (double)top_p)) * total, before, mass);
        if (threadIdx.x == 0) S.verdict = enough < 0 ? 1 : 0;
        __syncthreads();
    }
    return kb > 0 && kb < 2 * TB - 1 && kb != TB && kb != TB - 1 ? fmaxf(bound, value_of_bin(kb)) : bound;
}
// How far down the first slice matters.
__device__ __forceinline__ float sample_floor()
{
    const Smem<SPEC_BF16> M;
    const float m = cut::value_of(M.S.runmax);
    return m > -CUDART_INF_F && m < CUDART_INF_F ? fmaxf(m - SAMPLE_OCTAVES / M.S.sc.sf, LOWEST) : LOWEST;
}
// Starts a row's state (runmax, verdict) from the threads' maxima of the first slice, ms; returns how far down that slice matters.
__device__ __noinline__ float sample_bound(float ms)
{
    const Smem<SPEC_BF16> M;
    const uint32_t km = __reduce_max_sync(0xffffffffu, cut::key_of(ms));
    if ((threadIdx.x & 31) == 0) atomicMax(&M.S.runmax, km);
    if (threadIdx.x == 0) M.S.verdict = 0;
    __syncthreads();
    return sample_floor();
}
// The first bound, from the first slice alone.  Of a row of several slices with a positive logit in the first only positive ones have been
// counted: a cut below zero keeps more than half of a row of logits around zero.  Where they hold too little of the mass, the
// slice is counted again, from the ring (stage: the warp's share), all of it that matters.
__device__ __noinline__ float first_mass_bound(float tmax, float bound, float of, double Sd, float top_p, int n, int V, const uint4 *stage)
{
    const Smem<SPEC_BF16> M;
    const float b = mass_bound(tmax, bound, of, Sd, top_p, n, V);
    if (!M.S.verdict) return b;
    const float loose = sample_floor();
    const Counter cnt{bound_key(loose)};
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * TB / 4; i += NT) reinterpret_cast<uint4 *>(M.bins)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (int c = 0; c < UN; ++c) M.count(cnt, stage[c * NT + (threadIdx.x & 31)], false);
    return mass_bound(tmax, loose, of, Sd, top_p, n, V);
}

// Units of which some logits may be negative, or have no bins of their own; ms: the lane's maximum.  (Out of line: with the
// negative bounds' way of counting in the loop over the slices as well, rows of both signs took 3 % longer.)
__device__ __noinline__ void count_pair(const Counter cnt, const uint4 r0, const uint4 r1, float ms)
{
    const Smem<SPEC_BF16> M;
    const bool plain = !__any_sync(0xffffffffu, !(ms < cnt.plain_below()));
    M.count(cnt, r0, plain);
    M.count(cnt, r1, plain);
}

// what the pass over a row leaves in a thread (UNSET: no reference yet)
struct Pass {
    float tmax;                // the thread's maximum (NaN if it saw one)
    float of;                  // its integer reference, and its sum of e in units of 2^of (TOTAL)
    double Sd;
    float bound;               // the row is complete from it upwards (fp32 top-p: from the window upwards)
};

// Adds n units to the row's mass, as in the streaming statistics kernel: a running integer reference per thread, fp32 sums (a chain of
// additions per unit), fp64 above.  ms: the units' maximum.
template <int DT, int NU>
__device__ __forceinline__ void add_mass(const uint4 (&raw)[NU], float ms, float s_hi, float s_lo, Pass &ps)
{
    constexpr int E = DT == SPEC_BF16 ? 8 : 4;
    if (!(ms > -CUDART_INF_F && ms < CUDART_INF_F)) return;
    const float onew = fminf(fmaxf(ceilf(ms * s_hi), -1.0e9f), 1.0e9f);
    if (onew > ps.of) { ps.Sd *= (double)pow2i((int)fmaxf(ps.of - onew, -127.f)); ps.of = onew; }
    const unsigned long long sh2 = pack_f32x2(s_hi, s_hi), sl2 = pack_f32x2(s_lo, s_lo), no2 = pack_f32x2(-ps.of, -ps.of);
    unsigned long long sum = 0ull;
#pragma unroll
    for (int c = 0; c < NU; ++c) {
        float z[E];
        stream::unpack_unit<DT>(raw[c], z);
        unsigned long long acc = 0ull;
#pragma unroll
        for (int k = 0; k < E; k += 2) {
            const unsigned long long z2 = pack_f32x2(z[k], z[k + 1]);
            float x0, x1;
            unpack_f32x2(fma_f32x2(z2, sl2, fma_f32x2(z2, sh2, no2)), x0, x1);
            const unsigned long long e2 = pack_f32x2(ex2_approx(x0), ex2_approx(x1));
            acc = k == 0 ? e2 : add_f32x2(acc, e2);
        }
        sum = c == 0 ? acc : add_f32x2(sum, acc);
    }
    float a0, a1;
    unpack_f32x2(sum, a0, a1);
    ps.Sd += (double)(a0 + a1);
}

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
    double total = 0.0;                // sum over the row of 2^((z - m) s); 0: not known
    {
        const bool nan = ps.tmax != ps.tmax;
        float wm = ps.tmax;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
        int O_w = 0;
        double Sw = 0.0;
        if (TOTAL) {
            const int o_t = ps.of > UNSET ? (int)ps.of : ROWPART_EMPTY;
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
            }
            __syncthreads();
            clear();
            if (tid == 0) { S.runmax = 0u; S.count = 0; S.odd = 0; }
            __syncthreads();
            return;
        }
        if (TOTAL) {
            const int Om = __reduce_max_sync(0xffffffffu, Ok);
            total = warp_sum(lane < NW ? S.red[lane][0] * pow2d(max(Ok - Om, -1000)) : 0.0);
            // From units of 2^Om to units of the row maximum: 2^(Om - m s).  Om - m s lies in [0, 1] but for exponents beyond 2^24, where
            // a reference is rounded to a float.  Beyond 1e9 references end and the sums overflow or vanish: such a mass is not known (0),
            // and the row is settled without it.
            const double d = (double)Om - (double)m * s_d, n = rint(d);
            total *= exp2_frac(d - n) * pow2d((int)n);
            if (!(total > 0.0 && total < CUDART_INF)) total = 0.0;
        }
    }
    // The exponents of a row beyond the range of references fit no fp32 e; its sum is recorded as infinite, for which a verification reports
    // its sequence.  A distribution with far exponents is referenced to the largest logit itself, before anything is rounded (and settled
    // from the row).
    const double ms = (double)m * s_d, Od = reference(ms);
    const bool own = P.kept && fabs(ms) > FAR_EXPONENT;
    auto write = [&](double Z, double X, float cutv, int kept) {
        RowPart r;
        r.S = own || fabs(ms - Od) < 126.0 ? Z : CUDART_INF; r.X = X; r.O = (int)Od; r.cut = cutv;
        r.xmax = own ? 0.f : (float)(ms - Od);
        r.bad = own ? ROW_FAR : 0;
        *out = r;
        if (P.kept) { P.kept[id] = kept; P.kept[id + 1] = __float_as_int(m); }
    };
    bool settled = false;
    if (DT == SPEC_BF16) {
        const int b_max = bin_of(m);
        // Selection, kept sums and record from bins that are complete down to b_lo; says whether that settles the row.  By one warp: the
        // other CTAs of the SM make better use of the issue slots (by the block: 165 against 151 us on 3008 rows of top-k at V = 128256,
        // and within 1 us on few rows with wide nuclei).
        auto mass = [&](int i) {
            const unsigned long long c = bins[i];
            return c ? c * fix44(ex2_approx((value_of_bin(i) - m) * sf)) : 0ull;
        };
        // (a shared bin among the kept ones holds values that the bins cannot tell apart)
        auto sound = [&](int b_cut) {
            return b_cut >= 0 && !(fabsf(m) >= HIGH || (S.odd & ODD_HIGH) || ((S.odd & ODD_LOW) && b_cut >= TB - 1));
        };
        auto keep = [&](int b_cut) {
            double Z = 0.0, X = 0.0;
            int n = 0;
            for (int i = b_max + lane; i <= b_cut; i += 32) {
                const uint32_t c = bins[i];
                if (c) add_kept(value_of_bin(i), (double)c, s_d, Od, Z, X);
                n += (int)c;
            }
            Z = warp_sum(Z);
            X = warp_sum(X);
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) write(Z, X, value_of_bin(b_cut), n);
        };
        auto select = [&](int b_lo) {
            __syncthreads();
            if (w == 0) {
                int b_cut = -1;
                if (TOTAL) {
                    b_cut = warp_find<unsigned long long>(b_max, b_lo, (double)P.top_p * total * cut::FIX, mass);
                } else if (P.top_k <= K_FAST<DT>) {
                    b_cut = warp_find<uint32_t>(b_max, b_lo, (double)P.top_k, [&](int i) { return bins[i]; });
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
                const bool ok = sound(b_cut);
                if (ok) keep(b_cut);
                if (lane == 0) S.verdict = ok ? 1 : 0;
            }
            __syncthreads();
            return S.verdict != 0;
        };
        settled = !own && select(last_bin_above(ps.bound));
        if (TOTAL && !own && !settled && total > 0.0) {
            // The nucleus reaches below the bound.  All tokens more than log2(V / ((1 - top_p) total)) octaves
            // below the maximum together have no more than 1 - top_p of the mass: counted again, from L2, down
            // to there.
            const float wide = log2f((float)P.V / ((1.f - P.top_p) * (float)total)) + 0.01f;
            // (never above the maximum, whatever `wide` is: count_unit raises lower logits to the keys just below the bound, which
            // have bins because the maximum has one)
            const float bound2 = fminf(m, fmaxf(m - wide / sf, LOWEST));
            const Counter C{bound_key(bound2)};
            const bool plain = m < C.plain_below();
            __syncthreads();
            clear();
            __syncthreads();
            visit_units<DT>(span_of<DT>(P, id), [&](const uint4 &r) { M.count(C, r, plain); });
            __syncthreads();
            settled = select(last_bin_above(bound2));
        }
    } else {
        // ---- fp32: radix selection on the list of candidates --------------------------------------------------
        const int n = S.count;
        auto visit = [&](auto g) { for (int i = tid; i < n; i += NT) g(keys[i]); };
        uint32_t key = 0u;
        float cutv = -CUDART_INF_F;
        double Z = 0.0, X = 0.0;
        int kept = 0;
        settled = !own && n <= CAP && (TOTAL || P.top_k <= K_FAST<DT>);
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
                if (keys[i] >= key) { add_kept(cut::value_of(keys[i]), 1.0, s_d, Od, Z, X); ++kept; }
        }
        if (P.kept) kept = (int)block_sum(S, (unsigned long long)kept);
        if (settled) {
            Z = warp_sum(Z);
            X = warp_sum(X);
            __syncthreads();
            if (lane == 0) { S.red[w][0] = Z; S.red[w][1] = X; }
            __syncthreads();
            Z = X = 0.0;
            if (tid == 0) {
                for (int k = 0; k < NW; ++k) { Z += S.red[k][0]; X += S.red[k][1]; }
                write(Z, X, cutv, kept);
            }
        }
    }
    if (!settled) {
        __syncthreads();
        const Kept kp = settle_from_row<DT>(S, bins, span_of<DT>(P, id), P.V, P.top_k, P.top_p, m, sf, s_hi, s_lo, s_d, own, total);
        if (tid == 0) write(kp.Z, kp.X, kp.key ? cut::value_of(kp.key) : -CUDART_INF_F, kp.n);
    }
    if (DT == SPEC_BF16) __syncthreads();                // the bins have been read
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
    grid_dependency_wait();       // (what the call was given may come from the kernel before)
    grid_launch_dependents();

    if (DT == SPEC_BF16) for (int i = tid; i < 2 * TB; i += NT) M.bins[i] = 0;
    if (tid == 0) { S.runmax = 0u; S.count = 0; S.odd = 0; }
    if (P.parent && P.topo_stride == 0) {
        for (int i = tid; i < (P.N + 31) / 32; i += NT) S.inner[i] = 0u;
        __syncthreads();
        for (int c = 1 + tid; c < P.N; c += NT) {
            const int pa = __ldg(P.parent + c);
            if (pa >= 0 && pa < c) atomicOr(&S.inner[pa >> 5], 1u << (pa & 31));
        }
    }
    __syncthreads();

    // ---- the copying side of the ring: DEPTH - 1 slices ahead, across rows ----------------------------------
    int i_id = (int)blockIdx.x - (int)gridDim.x;
    const unsigned char *i_src = nullptr;
    int i_left = -tid, i_stage = 0;       // units of the row from the thread's next one on; the stage it goes to
    bool i_more = true;
    auto issue = [&]() {
        if (i_more && i_left + tid <= 0) {
            i_id = next_read(P, i_id + gridDim.x, items, S.inner);
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
    float T_now = 0.f, s_hi = 0.f, s_lo = 0.f;      // of the current temperature
    for (int id = blockIdx.x; id < items; id += gridDim.x) {
        // ---- rows that are not read, up to the next one that is --------------------------------------------------
        const int to = next_read(P, id, items, S.inner);
        for (; id < min(to + 1, items); id += gridDim.x) {
            if (tid == 0) {
                const int node = id >> 1;
                if ((id & 1) == 0) { const Split r(node, P.N, 1.f / (float)P.N); P.init.set(node, r.b, r.a); }
                if (id < to) {
                    RowPart r = {};
                    r.cut = -CUDART_INF_F; r.O = ROWPART_EMPTY; r.bad = -1;
                    P.part[id] = r;
                }
            }
            if (id == to) break;
        }
        if (id >= items) break;
        const stream::RowSpan row = span_of<DT>(P, id);
        const float T = P.T_seq ? __ldg(P.T_seq + Split(id >> 1, P.N, 1.f / (float)P.N).b) : P.T;
        if (T != T_now) {                      // (the block agrees; the scale factors are next read after a barrier)
            T_now = T;
            const double s_d = 1.4426950408889634 / (double)T;
            stream::split_scale(s_d, s_hi, s_lo);
            if (tid == 0) {
                const float sf = 1.4426950408889634f / T;
                S.sc = Scale{T, sf, s_hi, s_lo, WINDOW_OCTAVES / sf, s_d};
            }
        }
        // ---- the pass ------------------------------------------------------------------------------------------
        Pass ps = {-CUDART_INF_F, UNSET, 0.0, LOWEST};
        Counter cnt{0};
        int sure = 0;                      // slices for which the warp takes all its units to hold candidates
        const int nsl = (row.units + NT * UN - 1) / (NT * UN);
        for (int sl = 0; sl < nsl; ++sl) {
            // a better bound, from the slices so far
            if (DT == SPEC_BF16 && TOTAL) {
                if ((sl == 4 || sl == 16) && nsl > sl + 2) {
                    ps.bound = mass_bound(ps.tmax, ps.bound, ps.of, ps.Sd, P.top_p, min(P.V, sl * UN * NT * E), P.V);
                    cnt.kb = bound_key(ps.bound);
                    sure = 0;
                }
            } else if (nsl > sl + 2 && (sl == 2 || sl == 6 || (DT == SPEC_F32 && sl == 16))) {
                ps.bound = tighter_bound<DT, TOTAL>(P.top_k, ps.bound);
            }
            stream::cp_async_wait<DEPTH - 2>();
            issue();                                    // into the stage of the previous iteration
            uint4 *const stage = M.ring + c_stage * UN * NT + (tid & ~31);      // the warp's share of the slice
            c_stage = c_stage + 1 == DEPTH ? 0 : c_stage + 1;
            if (sl == 0 || sl == nsl - 1) {
#pragma unroll
                for (int c = 0; c < UN; ++c) {
                    uint4 r = stage[c * NT + lane];
                    stream::mask_unit<DT>(r, (sl * UN + c) * NT + tid, row);
                    stage[c * NT + lane] = r;
                }
            }
            if (DT == SPEC_BF16 && TOTAL) {
                if (sl == 0) {
                    uint32_t m = 0xFF80FF80u;
#pragma unroll
                    for (int c = 0; c < UN; ++c) m = stream::max_raw<DT>(m, stream::unit_max_raw<DT>(stage[c * NT + lane]));
                    ps.bound = sample_bound(stream::fold_max<DT>(m));
                    if (nsl > 1 && cut::value_of(S.runmax) > 0.f) ps.bound = fmaxf(ps.bound, __uint_as_float((uint32_t)PLAIN_KEY << 16));
                    cnt.kb = bound_key(ps.bound);
                }
                // two units at a time: what a step needs fits the registers
                bool all = true;
#pragma unroll 1
                for (int c = 0; c < UN; c += 2) {
                    uint4 raw[2] = {stage[c * NT + lane], stage[(c + 1) * NT + lane]};
                    const uint32_t mu[2] = {stream::unit_max_raw<DT>(raw[0]), stream::unit_max_raw<DT>(raw[1])};
                    const float ms = stream::fold_max<DT>(stream::max_raw<DT>(mu[0], mu[1]));      // (a NaN stays)
                    ps.tmax = stream::max_nan(ps.tmax, ms);
                    add_mass<DT, 2>(raw, ms, s_hi, s_lo, ps);
                    // A unit that holds a candidate anywhere in the warp is counted by all lanes.  Where all units of a slice did, those
                    // of the next three are not asked.
                    if (!cnt.positive() || __any_sync(0xffffffffu, !(ms < HIGH))) {
                        if (__any_sync(0xffffffffu, ms >= ps.bound)) count_pair(cnt, raw[0], raw[1], ms);
                    } else {
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            if (sure > 0 || __any_sync(0xffffffffu, cnt.reaches(mu[k]))) M.count(cnt, raw[k], true);
                            else all = false;
                        }
                    }
                }
                sure = sure > 0 ? sure - 1 : all ? 3 : 0;
                if (sl == 0 && nsl > 1) {
                    ps.bound = first_mass_bound(ps.tmax, ps.bound, ps.of, ps.Sd, P.top_p, min(P.V, UN * NT * E), P.V, stage);
                    cnt.kb = bound_key(ps.bound);
                    sure = 0;
                }
            } else {
                uint4 raw[UN];
#pragma unroll
                for (int c = 0; c < UN; ++c) raw[c] = stage[c * NT + lane];
                // the units' maxima (bf16: still as pairs) and the thread's maximum of the slice; a NaN stays
                uint32_t mu[UN];
#pragma unroll
                for (int c = 0; c < UN; ++c) mu[c] = stream::unit_max_raw<DT>(raw[c]);
                const float ms = stream::fold_max<DT>(stream::max_raw<DT>(stream::max_raw<DT>(mu[0], mu[1]), stream::max_raw<DT>(mu[2], mu[3])));
                static_assert(UN == 4, "slice maximum of four units");
                if (TOTAL) add_mass<DT, UN>(raw, ms, s_hi, s_lo, ps);
                // ---- the running maximum and the bound ----------------------------------------------------------------
                if (sl == 0) {
                    const uint32_t km = __reduce_max_sync(0xffffffffu, cut::key_of(ms));
                    if (lane == 0) atomicMax(&S.runmax, km);
                    if (TOTAL) __syncthreads();
                    else ps.bound = first_bound<DT>(P.top_k, make_uint4(mu[0], mu[1], mu[2], mu[3]));
                } else if (ms > ps.tmax && ms > cut::value_of(*(volatile uint32_t *)&S.runmax)) {
                    atomicMax(&S.runmax, cut::key_of(ms));
                }
                if (TOTAL) ps.bound = fmaxf(cut::value_of(*(volatile uint32_t *)&S.runmax) - S.sc.window, LOWEST);
                ps.tmax = stream::max_nan(ps.tmax, ms);
                // ---- candidates ----------------------------------------------------------------------------------
                if (__any_sync(0xffffffffu, ms >= ps.bound)) {
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
        }
        finish_row<DT, TOTAL>(P, id, ps);
    }
    stream::cp_async_wait<0>();
}

}  // namespace trunc
}  // namespace specv
