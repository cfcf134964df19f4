// Streaming row statistics (no truncation): every logit row the verifiers may touch is read once from
// HBM, straight into registers, and reduced to per-slice partial sums of the row's softmax normaliser.
// No residency: a CTA streams a row (or a part of it) in slices of 8192 logits, 32 per thread,
// the asynchronous copies of the next slices in flight while the current one is exponentiated.
//
// A thread turns its logits into e = 2^(z s - o) (s = log2(e)/T, o = ceil of its own largest z s, an
// integer, so partial sums combine by exact powers of two) and the CTA writes, for its row or part of one,
//     O = largest o, S = sum e 2^(o - O), X = sum e x 2^(o - O) with x = z s - O, the largest exponent.
// Rows in parts (batches with fewer rows than half the places) are a cluster each, and its first CTA merges them.
#pragma once
#include "common.cuh"

namespace specv {

// one slice of one row (stream kernel) or a whole row (row-statistics kernel, one slice per row)
struct __align__(16) RowPart {
    double S;          // sum over kept tokens of 2^(z s - O)
    double X;          // sum over kept tokens of e x, x = z s - O
    int O;             // reference (integer); ROWPART_EMPTY when the slice has no finite logit
    float xmax;        // largest exponent relative to O
    float cut;         // smallest kept logit of the row (-inf: nothing cut)
    int bad;           // 1: NaN or +inf seen; -1: row not read (draft row of a node without children)
};
constexpr int ROWPART_EMPTY = -(1 << 30);
// exponents z s beyond which the fp32 product no longer has an integer part exact to 1/16: kept sums and distributions go by fp64 there
constexpr double FAR_EXPONENT = 1048576.0;
constexpr int ROW_FAR = 2;         // RowPart::bad of such a row for which a distribution is wanted: S and X are in units of its largest e

namespace stream {

constexpr int MAX_PARTS = 4;             // of a row
constexpr int NT = 256;
constexpr int PER = 32;                  // logits per thread
constexpr int SLICE = NT * PER;          // logits per CTA and slice

// Per-call words of the workspace that an every-node verification wants set (w_pub NULL: none): the published
// weights, first-child ratios and accepted nodes to pending, counters to zero.  The
// statistics kernels set them, which saves the memset nodes of a call.
struct NodeInit {
    unsigned long long *w_pub;   // [B*N]
    unsigned int *done;          // [B]
    int *fin;                    // [B]
    unsigned int *ticket;        // [1]
    ulonglong2 *chain;           // [B*N]
    __device__ __forceinline__ void set(long long node, int b, int a) const
    {
        if (!w_pub) return;
        w_pub[node] = W_PENDING;
        chain[node] = make_ulonglong2(W_PENDING, 0ull);
        if (a == 0) { done[b] = 0u; fin[b] = -1; }
        if (node == 0) *ticket = 0u;
    }
};

struct SParams {
    int B, N, V, NSL;        // NSL: parts a row is split into (more CTAs than rows), a cluster of as many CTAs
    const void *zp, *zq;
    long long seq_stride, node_stride, topo_stride;
    const int *parent;
    float T;
    const float *T_seq;
    RowPart *part;           // [B*N*2]
    NodeInit init;
};

// A row as whole 16-byte units of memory: wherever the row starts, its logits are in the units from the one that
// holds its first byte to the one that holds its last, and the statistics do not care about positions inside
// the row -- so every row takes the 16-byte path, and only its first and last units are masked.
struct RowSpan {
    const unsigned char *base;   // 16-byte aligned
    int units;
    short head, last;            // first logit of the first unit; logits of the last unit, counted from its start
};
template <int DT>
__device__ __forceinline__ RowSpan row_span(const void *z, long long first, int V)
{
    constexpr int ESZ = DT == SPEC_BF16 ? 2 : 4, E = 16 / ESZ;
    const uintptr_t at = (uintptr_t)z + (uintptr_t)(first * ESZ);
    RowSpan r;
    r.base = (const unsigned char *)(at & ~(uintptr_t)15);
    r.head = (short)((at & 15) / ESZ);
    r.units = (r.head + V + E - 1) / E;
    r.last = (short)(r.head + V - (r.units - 1) * E);
    return r;
}
// the logits of unit u that are not the row's become -inf (all of them beyond the last unit)
template <int DT>
__device__ __forceinline__ void mask_unit(uint4 &r, int u, const RowSpan &row)
{
    constexpr int E = DT == SPEC_BF16 ? 8 : 4;
    const int e0 = u == 0 ? row.head : 0, e1 = u < row.units - 1 ? E : (u == row.units - 1 ? row.last : 0);
    if (e0 == 0 && e1 == E) return;
    uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int k = 0; k < E; ++k) {
        const bool out = k < e0 || k >= e1;
        if (DT == SPEC_BF16) {
            if (out) w[k >> 1] = (k & 1) ? (w[k >> 1] & 0xFFFFu) | 0xFF800000u : (w[k >> 1] & 0xFFFF0000u) | 0xFF80u;
        } else {
            if (out) w[k] = 0xFF800000u;
        }
    }
    r = make_uint4(w[0], w[1], w[2], w[3]);
}
// the logits of a unit (8 bf16 or 4 fp32)
template <int DT>
__device__ __forceinline__ void unpack_unit(const uint4 &r, float (&z)[DT == SPEC_BF16 ? 8 : 4])
{
    if (DT == SPEC_BF16) {
        z[0] = bf16_lo(r.x); z[1] = bf16_hi(r.x); z[2] = bf16_lo(r.y); z[3] = bf16_hi(r.y);
        z[4 % (DT == SPEC_BF16 ? 8 : 4)] = bf16_lo(r.z); z[5 % (DT == SPEC_BF16 ? 8 : 4)] = bf16_hi(r.z);
        z[6 % (DT == SPEC_BF16 ? 8 : 4)] = bf16_lo(r.w); z[7 % (DT == SPEC_BF16 ? 8 : 4)] = bf16_hi(r.w);
    } else {
        z[0] = __uint_as_float(r.x); z[1] = __uint_as_float(r.y); z[2] = __uint_as_float(r.z); z[3] = __uint_as_float(r.w);
    }
}
// maxima that a NaN operand makes NaN
__device__ __forceinline__ float max_nan(float a, float b)
{
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ uint32_t max_nan_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// maximum of a unit, as the bits of an fp32 value or of a pair of bf16 values (fold_max: the larger of the pair)
template <int DT>
__device__ __forceinline__ uint32_t max_raw(uint32_t a, uint32_t b)
{
    return DT == SPEC_BF16 ? max_nan_bf16x2(a, b) : __float_as_uint(max_nan(__uint_as_float(a), __uint_as_float(b)));
}
template <int DT>
__device__ __forceinline__ uint32_t unit_max_raw(const uint4 &r)
{
    return max_raw<DT>(max_raw<DT>(r.x, r.y), max_raw<DT>(r.z, r.w));
}
template <int DT>
__device__ __forceinline__ float fold_max(uint32_t m)
{
    return DT == SPEC_BF16 ? max_nan(bf16_lo(m), bf16_hi(m)) : __uint_as_float(m);
}
// s = s_hi + s_lo in two floats, s_lo > 0 (so that a -inf logit gives an exponent of -inf, never NaN)
__device__ __forceinline__ void split_scale(double s_d, float &s_hi, float &s_lo)
{
    s_hi = (float)s_d;
    if ((double)s_hi > s_d) s_hi = __uint_as_float(__float_as_uint(s_hi) - 1u);
    s_lo = (float)(s_d - (double)s_hi);
    if (!(s_lo > 0.f)) s_lo = 1.0e-30f;
}
// whether node a of a tree has children (warp-collective)
__device__ __forceinline__ bool has_children(const int *parent, int N, int a, int lane)
{
    for (int c0 = a + 1; c0 < N; c0 += 32) {
        const int c = c0 + lane;
        if (__any_sync(0xffffffffu, c < N && __ldg(parent + c) == a)) return true;
    }
    return false;
}

// depth of the per-thread staging ring and its size
template <int DT> struct Ring {
    static constexpr int NV = DT == SPEC_BF16 ? 1 : 2;         // 16-byte units per 8 logits
    static constexpr int UNITS = (PER / 8) * NV;               // 16-byte units per thread and slice
    static constexpr int DEPTH = DT == SPEC_BF16 ? 5 : 3;
    static constexpr int BYTES = DEPTH * UNITS * NT * 16;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One CTA per (row, part of the row).  The part's slices of 8192 logits are streamed one after the
// other; every thread stages its own 32 logits of the next DEPTH - 1 slices in shared memory with
// asynchronous 16-byte copies (a thread reads back only what it copied itself, so the ring needs no
// barrier) and keeps a running (reference, sum) pair, rescaled by an exact power of two when a later
// slice raises its reference.  The CTA reduces once per part.
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));     // a NaN operand yields the other one
    return d;
}

// a part of a row into the same place of the cluster's first CTA
__device__ __forceinline__ void store_part(RowPart *slot, const RowPart &r)
{
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"(smem_u32(slot)));
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(at), "d"(r.S), "d"(r.X) : "memory");
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + 16u), "r"(r.O), "r"(__float_as_int(r.xmax)), "r"(__float_as_int(r.cut)), "r"(r.bad) : "memory");
}
// the parts of a row as one record, by one warp
__device__ __forceinline__ RowPart merge_parts(const RowPart *p, int n, bool feat)
{
    const int lane = threadIdx.x & 31;
    const bool has = lane < n;
    const int Ok = has ? p[lane].O : ROWPART_EMPTY, O = __reduce_max_sync(0xffffffffu, Ok);
    const int bad = __any_sync(0xffffffffu, has && p[lane].bad == 1);
    double S = 0.0, X = 0.0, best = -1.0e300;
    if (Ok > ROWPART_EMPTY) {
        const int d = max(Ok - O, -100000);
        const double f = pow2d(d);
        S = p[lane].S * f;
        X = f * (p[lane].X + (double)d * p[lane].S);
        best = (double)Ok + (double)p[lane].xmax;
    }
    S = warp_sum(S);
    X = warp_sum(X);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    RowPart r;
    r.S = S; r.X = X; r.O = O; r.xmax = feat && O > ROWPART_EMPTY ? (float)(best - (double)O) : 0.f;
    r.cut = -CUDART_INF_F;
    r.bad = bad || !(S > 0.0) || !(S < CUDART_INF) ? 1 : 0;
    return r;
}

// FEAT: also accumulate X (needed only by the entropy features).  Without it a NaN or +inf logit is
// found from the sum itself (such a logit makes its e, and so the thread's sum, non-finite), which
// keeps comparisons out of the inner loop.
template <int DT, bool FEAT>
__global__ void __launch_bounds__(NT, 2) spec_row_partial_kernel(const SParams P)
{
    constexpr int NV = Ring<DT>::NV, UNITS = Ring<DT>::UNITS, DEPTH = Ring<DT>::DEPTH;
    __shared__ double sS[NT / 32], sX[NT / 32], sB[NT / 32];
    __shared__ int sO[NT / 32], sBad[NT / 32];
    __shared__ RowPart sPart[MAX_PARTS];                          // of the cluster's row, in its first CTA
    uint4 *ring = reinterpret_cast<uint4 *>(dyn_smem);            // [DEPTH][UNITS][NT]
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long items = 2ll * P.B * P.N * P.NSL;
    grid_dependency_wait();       // (what the call was given may come from the kernel before)
    grid_launch_dependents();     // a dependent verifier's CTAs may take the places of CTAs that have finished
    if (P.NSL > 1) cluster_sync_all();       // the first CTA's shared memory is there to be written

    for (long long id = blockIdx.x; id < items; id += gridDim.x) {
        const int h = (int)(id % P.NSL);
        const long long row2 = id / P.NSL;
        const int which = (int)(row2 & 1);
        const long long row = row2 >> 1;
        const int b = (int)(row / P.N), a = (int)(row % P.N);
        RowPart *out = P.part + row2;
        if (which == 0 && h == 0 && tid == 0) P.init.set(row, b, a);
        // a draft row is read only for nodes that have children (every warp finds out by itself)
        if (which == 1 && !has_children(P.parent + (long long)b * P.topo_stride, P.N, a, lane)) {
            if (tid == 0 && h == 0) { RowPart r = {}; r.O = ROWPART_EMPTY; r.cut = -CUDART_INF_F; r.bad = -1; *out = r; }
            continue;
        }
        const RowSpan span = row_span<DT>(which ? P.zq : P.zp, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V);
        const int slices_row = (span.units + NT * UNITS - 1) / (NT * UNITS);
        const int slices_part = (slices_row + P.NSL - 1) / P.NSL;
        const int s_begin = h * slices_part, s_end = min(slices_row, s_begin + slices_part);
        const double s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
        float s_hi, s_lo;
        split_scale(s_d, s_hi, s_lo);

        // the thread's running state
        float of = 0.f, S_t = 0.f, X_t = 0.f, xm_t = -CUDART_INF_F;
        bool set = false;
        int bad = 0;

        // a slice's maximum moves the thread's reference up by an exact power of two
        auto new_reference = [&](float zm) {
            bad |= zm == CUDART_INF_F;
            if (zm > -CUDART_INF_F) {
                const float onew = fminf(fmaxf(ceilf(zm * s_hi), -1.0e9f), 1.0e9f);
                if (!set) { of = onew; set = true; }
                else if (onew > of) {
                    const float dlt = of - onew;
                    const float f = pow2i((int)fmaxf(dlt, -127.f));
                    X_t = f * fmaf(dlt, S_t, X_t);
                    S_t *= f;
                    xm_t += dlt;
                    of = onew;
                }
                if (FEAT) xm_t = fmaxf(xm_t, fmaf(zm, s_lo, fmaf(zm, s_hi, -of)));
            }
        };
        // 8 logits into the sums
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, b0 = 0.f, b1 = 0.f;
        auto add8 = [&](const float (&z)[8]) {
            if (FEAT) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float x = fmaxf(fmaf(z[k], s_lo, fmaf(z[k], s_hi, -of)), -200.f);
                    bad |= z[k] != z[k];
                    const float e = ex2_approx(x);
                    if (k & 1) { a1 += e; b1 = fmaf(e, x, b1); } else { a0 += e; b0 = fmaf(e, x, b0); }
                }
            } else {
                // two logits per instruction: the exponents z s - of and the running sums as fp32 pairs
                // (each half is the same IEEE operation as the scalar form)
                const unsigned long long sh2 = pack_f32x2(s_hi, s_hi), sl2 = pack_f32x2(s_lo, s_lo), no2 = pack_f32x2(-of, -of);
                unsigned long long acc01 = pack_f32x2(a0, a1), acc23 = pack_f32x2(a2, a3);
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    const unsigned long long z2 = pack_f32x2(z[k], z[k + 1]);
                    const unsigned long long x2 = fma_f32x2(z2, sl2, fma_f32x2(z2, sh2, no2));
                    float x0, x1;
                    unpack_f32x2(x2, x0, x1);
                    const unsigned long long e2 = pack_f32x2(ex2_approx(x0), ex2_approx(x1));
                    if (k & 2) acc23 = add_f32x2(acc23, e2); else acc01 = add_f32x2(acc01, e2);
                }
                unpack_f32x2(acc01, a0, a1);
                unpack_f32x2(acc23, a2, a3);
            }
        };
        auto flush = [&]() {
            S_t += (a0 + a1) + (a2 + a3);
            X_t += b0 + b1;
            a0 = a1 = a2 = a3 = b0 = b1 = 0.f;
        };

        // ---- the part's slices through the ring; the units at the ends of the row are masked ----------------------
        {
            const unsigned char *src = span.base + ((size_t)s_begin * NT * UNITS + tid) * 16;
            const uint32_t dst0 = ring_s + (uint32_t)tid * 16u;
            int isl = s_begin, ist = 0, cst = 0;
            auto issue = [&]() {
                if (isl < s_end) {
                    const int u0 = isl * NT * UNITS + tid;
#pragma unroll
                    for (int u = 0; u < UNITS; ++u)
                        if (u0 + u * NT < span.units)
                            cp_async16(dst0 + (uint32_t)((ist * UNITS + u) * NT) * 16u, src + (size_t)u * NT * 16, 16);
                    src += (size_t)NT * UNITS * 16;
                    ++isl;
                    ist = ist + 1 == DEPTH ? 0 : ist + 1;
                }
                cp_async_commit();
            };
#pragma unroll
            for (int k = 0; k < DEPTH - 1; ++k) issue();
            for (int sl = s_begin; sl < s_end; ++sl) {
                cp_async_wait<DEPTH - 2>();
                const uint4 *st = ring + (size_t)cst * UNITS * NT + tid;
                uint4 raw[UNITS];
#pragma unroll
                for (int u = 0; u < UNITS; ++u) raw[u] = st[u * NT];
                cst = cst + 1 == DEPTH ? 0 : cst + 1;
                issue();                                  // the stage read in the previous iteration is free again
                if (sl == 0 || sl == slices_row - 1) {
#pragma unroll
                    for (int u = 0; u < UNITS; ++u) mask_unit<DT>(raw[u], (sl * UNITS + u) * NT + tid, span);
                }
                float zm;
                if (DT == SPEC_BF16) {
                    uint32_t m2 = 0xFF80FF80u;            // the slice maximum on packed pairs
#pragma unroll
                    for (int u = 0; u < UNITS; ++u)
                        m2 = max_bf16x2(m2, max_bf16x2(max_bf16x2(raw[u].x, raw[u].y), max_bf16x2(raw[u].z, raw[u].w)));
                    zm = fmaxf(bf16_lo(m2), bf16_hi(m2));
                } else {
                    zm = -CUDART_INF_F;
#pragma unroll
                    for (int u = 0; u < UNITS; ++u)
                        zm = fmaxf(zm, fmaxf(fmaxf(__uint_as_float(raw[u].x), __uint_as_float(raw[u].y)),
                                             fmaxf(__uint_as_float(raw[u].z), __uint_as_float(raw[u].w))));
                }
                new_reference(zm);
#pragma unroll
                for (int c = 0; c < PER / 8; ++c) {
                    float z[8];
                    if (DT == SPEC_BF16) {
                        const uint4 r = raw[c];
                        z[0] = bf16_lo(r.x); z[1] = bf16_hi(r.x); z[2] = bf16_lo(r.y); z[3] = bf16_hi(r.y);
                        z[4] = bf16_lo(r.z); z[5] = bf16_hi(r.z); z[6] = bf16_lo(r.w); z[7] = bf16_hi(r.w);
                    } else {
                        const uint4 r0 = raw[c * NV], r1 = raw[c * NV + NV - 1];
                        z[0] = __uint_as_float(r0.x); z[1] = __uint_as_float(r0.y); z[2] = __uint_as_float(r0.z); z[3] = __uint_as_float(r0.w);
                        z[4] = __uint_as_float(r1.x); z[5] = __uint_as_float(r1.y); z[6] = __uint_as_float(r1.z); z[7] = __uint_as_float(r1.w);
                    }
                    add8(z);
                }
                flush();
            }
            cp_async_wait<0>();
        }
        // a NaN logit leaves a NaN in the sum; +inf was seen in the maximum
        bad |= !(fabsf(S_t) <= 3.0e38f);
        const int o_t = set ? (int)of : ROWPART_EMPTY;

        // ---- warp, then CTA: merge (reference, sums) pairs by exact powers of two --------------------------------
        const int O_w = __reduce_max_sync(0xffffffffu, o_t);
        const int d = max(o_t - O_w, -100000);
        const double f = (double)pow2i(max(d, -127));
        const double Sw = warp_sum((double)S_t * f);
        double Xw = 0.0, best = -1.0e300;
        if (FEAT) {
            Xw = warp_sum(f * ((double)X_t + (double)d * (double)S_t));
            best = set ? (double)o_t + (double)xm_t : -1.0e300;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
        }
        bad = __any_sync(0xffffffffu, bad);
        __syncthreads();             // the previous item's partials have been read
        if (lane == 0) { sS[w] = Sw; sX[w] = Xw; sB[w] = best; sO[w] = O_w; sBad[w] = bad; }
        __syncthreads();
        if (w == 0) {
            // the warps' partials, one per lane
            const bool has = lane < NT / 32;
            const int Ok = has ? sO[lane] : ROWPART_EMPTY;
            const int O = __reduce_max_sync(0xffffffffu, Ok);
            const int dk = max(Ok - O, -100000);
            const double fk = pow2d(dk), Sk = has ? sS[lane] : 0.0;
            double S = Sk * fk, X = has ? fk * (sX[lane] + (double)dk * Sk) : 0.0, bst = has ? sB[lane] : -1.0e300;
#pragma unroll
            for (int o = (NT / 64); o > 0; o >>= 1) {
                S += __shfl_xor_sync(0xffffffffu, S, o);
                X += __shfl_xor_sync(0xffffffffu, X, o);
                bst = fmax(bst, __shfl_xor_sync(0xffffffffu, bst, o));
            }
            const int bd = __any_sync(0xffffffffu, has && sBad[lane]);
            if (lane == 0) {
                RowPart r;
                r.S = S; r.X = X; r.O = O; r.xmax = (FEAT && O > ROWPART_EMPTY) ? (float)(bst - (double)O) : 0.f;
                r.cut = -CUDART_INF_F; r.bad = bd;
                if (P.NSL == 1) *out = r;
                else store_part(&sPart[h], r);
            }
        }
        if (P.NSL > 1) {
            cluster_sync_all();
            if (h == 0 && w == 0) {
                const RowPart r = merge_parts(sPart, P.NSL, FEAT);
                if (lane == 0) *out = r;
            }
            cluster_sync_all();          // the parts have been read
        }
    }
}

// Selector features of every row from its record: entropy (nats) and largest probability, [nodes][4]: H_p, H_q, top1_p, top1_q (those of
// a row that is not read are 0).  A thread per row.  (In the statistics kernels, by the thread that writes the record, they hold
// up the next row of the CTA: 760 instead of 710 us for a top-k call with 12000 rows.)
struct FParams {
    long long rows;          // 2 B N
    const RowPart *part;
    float *features;
};

__global__ void __launch_bounds__(128) spec_features_kernel(const FParams P)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= P.rows) return;
    const RowPart r = P.part[row];
    float H = 0.f, top = 0.f;
    if (r.bad != -1) {
        const bool ok = r.bad == 0 && r.S > 0.0 && r.S < CUDART_INF;
        H = ok ? (float)(log(r.S) - 0.6931471805599453 * r.X / r.S) : CUDART_NAN_F;
        top = ok ? (float)(exp2((double)r.xmax) / r.S) : CUDART_NAN_F;
    }
    float *f = P.features + (row >> 1) * 4 + (row & 1);
    f[0] = H;
    f[2] = top;
}

}  // namespace stream
}  // namespace specv
