// Row kernels of libspecverify: materialised sampling distributions (spec_tree_probs) and the
// stand-alone inverse-CDF draw (spec_sample_bonus).  These are utility entry points; the verification path proper is
// verify.cuh.
//   distributions  without truncation: one cluster per row, each CTA stages its vocabulary slice with bulk asynchronous copies and the
//                  CTAs combine through distributed shared memory (spec_probs_kernel); with top-k / top-p: the selection kernel of
//                  trunc.cuh, then one pass that writes (spec_probs_kept_kernel);
//   draw           a cluster per row, nothing staged (spec_bonus_kernel).
#pragma once
#include <cooperative_groups.h>
#include <type_traits>

#include "common.cuh"
#include "stream.cuh"

namespace specv {
namespace rowops {
namespace cg = cooperative_groups;

constexpr int NT = 512;              // threads per CTA
constexpr int NWARP = NT / 32;
constexpr int CMAX = 16;             // CTAs per cluster (16 needs the non-portable attribute)
constexpr int NX = 10;               // doubles per CTA per exchange
constexpr uint32_t BULK_CHUNK = 16384;

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) { mbar_arrive_expect_tx(bar, bytes); }
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// exp2((z - m) * s) with s = s_hi + s_lo: the product is formed in two parts so that the rounding of
// the exponent (|x| up to ~100) does not cost relative accuracy in e.
__device__ __forceinline__ float exp_scaled(float z, float m, float s_hi, float s_lo, float &x_out)
{
    float d = z - m;
    float x = d * s_hi;
    float lo = fmaf(d, s_lo, fmaf(d, s_hi, -x));
    x_out = x;
    if (!(x > -150.f)) { x_out = 0.f; return 0.f; }
    float e = ex2_approx(x);
    return fmaf(e, lo * 0.6931471805599453f, e);
}

// ------------------------------------------------------------------------------------------------
// shared state of one CTA
// ------------------------------------------------------------------------------------------------
struct Shared {
    double warp_part[NWARP][NX];
    double xchg[2][CMAX][NX];
    double scale_p[CMAX], scale_q[CMAX];   // exp((m_r - m)/T) per cluster rank
    double ctl_d[4];
    int ctl_i[4];
    int kc, err;
    uint64_t mbar;
};

// Thread 0 holds v[0..nv); copies them into slot [parity][my_rank] of every CTA of the cluster, then
// the cluster barrier makes all slots visible everywhere.
__device__ __forceinline__ void cluster_allgather(cg::cluster_group &cluster, Shared &S, int parity,
                                                  const double *v, int nv)
{
    if (threadIdx.x == 0) {
        unsigned C = cluster.num_blocks(), me = cluster.block_rank();
        for (unsigned r = 0; r < C; ++r) {
            double *dst = cluster.map_shared_rank(&S.xchg[parity][me][0], r);
            for (int i = 0; i < nv; ++i) dst[i] = v[i];
        }
    }
    cluster.sync();
}

// block-wide sum of nv doubles per thread; result valid in thread 0.  Uses S.warp_part; the caller
// must pass a block or cluster barrier before the next use.
template <int NV>
__device__ __forceinline__ void block_sum(Shared &S, double (&v)[NV])
{
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) S.warp_part[w][i] = v[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            double t = 0.0;
            for (int k = 0; k < NWARP; ++k) t += S.warp_part[k][i];
            v[i] = t;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// row staging: global -> shared (raw dtype), placed so that the in-place widening to fp32 is safe
// ------------------------------------------------------------------------------------------------
// region: SL floats.  fp32 raw data sits at the start; bf16 raw data in the upper half.
__device__ __forceinline__ unsigned char *raw_ptr(float *region, int SL, int dtype)
{
    return (unsigned char *)region + (dtype == SPEC_BF16 ? 2 * (size_t)SL : 0);
}

// Issue the copy of `n` elements starting at element `g0` of the row at `row` into `region`.
// Thread 0 enqueues bulk copies for the 16-byte aligned body; everything else (a misaligned row,
// the last partial 16 bytes) is fetched with ordinary loads by all threads.
// Returns the number of bytes that will complete on the mbarrier (valid in thread 0).
__device__ __forceinline__ uint32_t stage_row(float *region, int SL, int dtype, const void *row,
                                              long long g0, int n, uint64_t *bar, bool count_only)
{
    const int esz = dtype == SPEC_BF16 ? 2 : 4;
    const unsigned char *src = (const unsigned char *)row + g0 * esz;
    unsigned char *dst = raw_ptr(region, SL, dtype);
    bool aligned = (((uintptr_t)src) & 15) == 0;
    uint32_t body = aligned ? (((uint32_t)n * esz) & ~15u) : 0u;
    if (count_only) return body;
    if (threadIdx.x == 0) {
        for (uint32_t off = 0; off < body; off += BULK_CHUNK) {
            uint32_t sz = body - off < BULK_CHUNK ? body - off : BULK_CHUNK;
            bulk_g2s(dst + off, src + off, sz, bar);
        }
    }
    int first = body / esz;               // elements not covered by the bulk copies
    if (dtype == SPEC_BF16) {
        const unsigned short *s = (const unsigned short *)src;
        unsigned short *d = (unsigned short *)dst;
        for (int i = first + threadIdx.x; i < n; i += NT) d[i] = __ldg(s + i);
    } else {
        const float *s = (const float *)src;
        float *d = (float *)dst;
        for (int i = first + threadIdx.x; i < n; i += NT) d[i] = __ldg(s + i);
    }
    return body;
}

// max over the raw slice (ignoring NaN, which is reported through `nan`)
__device__ __forceinline__ float raw_max(const float *region, int SL, int dtype, int n, bool &nan)
{
    float m = -CUDART_INF_F;
    bool bad = false;
    const unsigned char *raw = raw_ptr(const_cast<float *>(region), SL, dtype);
    if (dtype == SPEC_BF16) {
        const uint4 *v = (const uint4 *)raw;
        int nv = n >> 3;
        for (int i = threadIdx.x; i < nv; i += NT) {
            uint4 q = v[i];
            uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float a = bf16_lo(w[k]), b = bf16_hi(w[k]);
                bad |= (a != a) | (b != b);
                m = fmaxf(m, fmaxf(a, b));
            }
        }
        const unsigned short *h = (const unsigned short *)raw;
        for (int i = (nv << 3) + threadIdx.x; i < n; i += NT) {
            float a = __uint_as_float((uint32_t)h[i] << 16);
            bad |= (a != a);
            m = fmaxf(m, a);
        }
    } else {
        const float4 *v = (const float4 *)raw;
        int nv = n >> 2;
        for (int i = threadIdx.x; i < nv; i += NT) {
            float4 q = v[i];
            bad |= (q.x != q.x) | (q.y != q.y) | (q.z != q.z) | (q.w != q.w);
            m = fmaxf(m, fmaxf(fmaxf(q.x, q.y), fmaxf(q.z, q.w)));
        }
        const float *h = (const float *)raw;
        for (int i = (nv << 2) + threadIdx.x; i < n; i += NT) {
            float a = h[i];
            bad |= (a != a);
            m = fmaxf(m, a);
        }
    }
    nan = bad;
    return m;
}

// In-place widening raw -> e = exp((z - m)/T) for z >= cut (0 otherwise, and 0 in the padding up to
// SL).  Accumulates sum e and sum e*log2(e).  bf16: a step reads 8 values per thread, a block
// barrier, then writes 8 floats; step s writes bytes [16384 s, 16384 (s+1)) of the region while the
// unread raw data starts at 2 SL + 8192 (s+1) >= 16384 (s+1) as long as a later step exists.
__device__ __forceinline__ void widen_exp(float *region, int SL, int dtype, int n, float m, float cut,
                                          float s_hi, float s_lo, double &sum_e, double &sum_ex, int &kept)
{
    double acc_e = 0.0, acc_x = 0.0;
    int nk = 0;
    if (dtype == SPEC_BF16) {
        const unsigned char *raw = raw_ptr(region, SL, dtype);
        int steps = (SL + NT * 8 - 1) / (NT * 8);
        for (int s = 0; s < steps; ++s) {
            int t0 = (s * NT + threadIdx.x) * 8;
            bool act = t0 < SL;
            uint4 q = make_uint4(0, 0, 0, 0);
            if (act) q = *(const uint4 *)(raw + (size_t)t0 * 2);
            __syncthreads();
            if (act) {
                uint32_t w[4] = {q.x, q.y, q.z, q.w};
                float e[8];
                float pe = 0.f, px = 0.f;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    float z = (k & 1) ? bf16_hi(w[k >> 1]) : bf16_lo(w[k >> 1]);
                    bool keep = (t0 + k < n) && (z >= cut);
                    nk += keep ? 1 : 0;
                    float x;
                    float v = exp_scaled(keep ? z : -CUDART_INF_F, m, s_hi, s_lo, x);
                    e[k] = v;
                    pe += v;
                    px = fmaf(v, x, px);
                }
                acc_e += (double)pe;
                acc_x += (double)px;
                float4 *o = (float4 *)(region + t0);
                o[0] = make_float4(e[0], e[1], e[2], e[3]);
                o[1] = make_float4(e[4], e[5], e[6], e[7]);
            }
        }
    } else {
        int nv = SL >> 2;
        float4 *v = (float4 *)region;
        for (int i = threadIdx.x; i < nv; i += NT) {
            float4 q = v[i];
            float zz[4] = {q.x, q.y, q.z, q.w};
            float e[4];
            float pe = 0.f, px = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float x;
                bool keep = ((i * 4 + k) < n) && (zz[k] >= cut);
                nk += keep ? 1 : 0;
                float val = exp_scaled(keep ? zz[k] : -CUDART_INF_F, m, s_hi, s_lo, x);
                e[k] = val;
                pe += val;
                px = fmaf(val, x, px);
            }
            acc_e += (double)pe;
            acc_x += (double)px;
            v[i] = make_float4(e[0], e[1], e[2], e[3]);
        }
    }
    sum_e = acc_e;
    sum_ex = acc_x;
    kept = nk;
}

// ------------------------------------------------------------------------------------------------
// spec_tree_probs: materialise the sampling distribution of every row
// ------------------------------------------------------------------------------------------------
struct TParams {
    int rows, N, V, dtype, SL;
    const void *z;
    long long seq_stride, node_stride;
    float T;
    const float *T_seq;
    float *probs, *stats;
};

__global__ void __launch_bounds__(NT, 2) spec_probs_kernel(const TParams P)
{
    cg::cluster_group cluster = cg::this_cluster();
    grid_dependency_wait();
    const int C = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int row_id = blockIdx.x / C;
    const int b = row_id / P.N, a = row_id % P.N;
    const int tid = threadIdx.x;
    const int SL = P.SL;
    __shared__ Shared S;
    float *ep = (float *)dyn_smem;
    const long long tok0 = (long long)rank * SL;
    const int n = (int)max(0ll, min((long long)SL, (long long)P.V - tok0));
    const double T = (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
    if (tid == 0) { mbar_init(&S.mbar, 1); mbar_fence_init(); }
    __syncthreads();
    const void *row = (const unsigned char *)P.z +
                      ((long long)b * P.seq_stride + (long long)a * P.node_stride) * (P.dtype == SPEC_BF16 ? 2 : 4);
    uint32_t tx = stage_row(ep, SL, P.dtype, row, tok0, n, &S.mbar, true);
    if (tid == 0 && tx) mbar_expect_tx(&S.mbar, tx);
    stage_row(ep, SL, P.dtype, row, tok0, n, &S.mbar, false);
    bool gave_up = false;
    if (tx) gave_up = !mbar_wait(&S.mbar, 0);
    __syncthreads();
    bool nan = gave_up;          // a copy that was given up on: the row comes out as a non-finite one
    bool nan2 = false;
    float m = warp_max(raw_max(ep, SL, P.dtype, n, nan2));
    nan = nan || nan2;
    if ((tid & 31) == 0) S.warp_part[tid >> 5][0] = (double)m;
    int any_nan = __syncthreads_or((int)nan);
    m = -CUDART_INF_F;
    for (int k = 0; k < NWARP; ++k) m = fmaxf(m, (float)S.warp_part[k][0]);
    __syncthreads();
    float s_hi, s_lo;
    split_float(1.4426950408889634 / T, s_hi, s_lo);
    const float ref = (m > -CUDART_INF_F && m < CUDART_INF_F) ? m : 0.f;
    double v[NX];
#pragma unroll
    for (int i = 0; i < NX; ++i) v[i] = 0.0;
    int kept = 0;
    widen_exp(ep, SL, P.dtype, n, ref, -CUDART_INF_F, s_hi, s_lo, v[1], v[2], kept);
    {
        double red[3] = {v[1], v[2], (double)kept};
        block_sum<3>(S, red);
        v[1] = red[0]; v[2] = red[1]; v[3] = red[2];
    }
    v[0] = (double)m; v[6] = any_nan ? 1.0 : 0.0;
    cluster.sync();                      // peers must be running before their shared memory is written
    cluster_allgather(cluster, S, 0, v, NX);
    double (*X)[NX] = S.xchg[0];
    double mg = -CUDART_INF;
    bool bad = false;
    for (int r = 0; r < C; ++r) { mg = fmax(mg, X[r][0]); bad |= X[r][6] != 0.0; }
    bad |= !(mg > -CUDART_INF && mg < CUDART_INF);
    if (tid < C) {
        double mr = X[tid][0];
        S.scale_p[tid] = (!bad && mr > -CUDART_INF) ? exp((mr - mg) / T) : 0.0;
    }
    __syncthreads();
    double Z = 0.0;
    for (int r = 0; r < C; ++r) Z += S.scale_p[r] * X[r][1];
    const float mul = bad ? 0.f : (float)(S.scale_p[rank] / Z);
    if (P.probs) {
        float *out = P.probs + (long long)row_id * P.V + tok0;
        for (int i = tid; i < n; i += NT) out[i] = ep[i] * mul;
    }
    if (P.stats && rank == 0 && tid == 0) {
        float *st = P.stats + (long long)row_id * 6;
        if (bad) {
            for (int i = 0; i < 6; ++i) st[i] = CUDART_NAN_F;
        } else {
            double h = 0.0;
            for (int r = 0; r < C; ++r) {
                double sp = S.scale_p[r];
                if (sp > 0.0) h -= (sp / Z) * (0.6931471805599453 * X[r][2] + (log(sp) - log(Z)) * X[r][1]);
            }
            double nkept = 0.0;
            for (int r = 0; r < C; ++r) nkept += X[r][3];
            st[0] = (float)(mg / T); st[1] = (float)Z; st[2] = (float)nkept;
            st[3] = (float)h; st[4] = (float)(1.0 / Z); st[5] = -CUDART_INF_F;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// spec_tree_probs under top-k / top-p: the kept tokens of a row are known by value (its record), so that its distribution is written
// in one pass without shared memory or barriers
// ------------------------------------------------------------------------------------------------
// A CTA writes parts of KEPT_PART tokens, four consecutive tokens per thread and step; all its loads are issued first.  Bound by
// the writes.
// 76 rows of 128256, bf16 (58 MB): 37 us with the row staged in shared memory and widened there, 14 now.
constexpr int KEPT_NT = 256, KEPT_STEPS = 4, KEPT_PART = KEPT_NT * 4 * KEPT_STEPS;
struct KParams {
    int N, V, parts;
    long long items;         // rows * parts
    const void *z;
    long long seq_stride, node_stride;
    float T;
    const float *T_seq;
    const RowPart *part;     // [rows][2], the first of each pair
    const int *kept;         // [rows][2]: kept tokens, largest logit as bits
    float *probs, *stats;
};
// of a token that is no less than 2^-4 of the unit of the row's sum
__device__ __noinline__ float heavy_prob(float z, double s_d, int O, double S) { return (float)(exp2_exact((double)z, s_d, (double)O) / S); }
// tokens t0 .. t1 - 1 of a row with far exponents, whose unit is its largest logit m
__device__ __noinline__ void write_far(const void *z, int dtype, float *out, int t0, int t1, float cut, float m, double s_d, double S)
{
    for (int t = t0 + (int)threadIdx.x; t < t1; t += KEPT_NT) {
        const float v = load_logit(z, dtype, t);
        out[t] = v >= cut ? (float)(exp2_exact((double)v - (double)m, s_d, 0.0) / S) : 0.f;
    }
}

template <int DT>
__global__ void __launch_bounds__(KEPT_NT, 4) spec_probs_kept_kernel(const KParams P)
{
    constexpr int ESZ = DT == SPEC_BF16 ? 2 : 4;
    const int tid = threadIdx.x;
    grid_dependency_wait();
    for (long long it = blockIdx.x; it < P.items; it += gridDim.x) {
        const int row = (int)(it / P.parts), part = (int)(it % P.parts), b = row / P.N;
        const RowPart *rp = P.part + 2ll * row;
        const double T = (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T), S = rp->S, s_d = 1.4426950408889634 / T;
        const int O = rp->O, bad = rp->bad;
        const float cut = rp->cut;
        if (P.stats && part == 0 && tid == 0) {
            float *st = P.stats + 6ll * row;
            if (bad == 1) {
                for (int i = 0; i < 6; ++i) st[i] = CUDART_NAN_F;
            } else {
                // in units of the largest e, 2^xmax
                const double x = (double)rp->xmax, Z = S * exp2(-x);
                st[0] = (float)((double)__int_as_float(P.kept[2ll * row + 1]) / T); st[1] = (float)Z; st[2] = (float)P.kept[2ll * row];
                st[3] = (float)(log(S) - 0.6931471805599453 * rp->X / S); st[4] = (float)(1.0 / Z); st[5] = cut;
            }
        }
        if (!P.probs) continue;
        float s_hi, s_lo, inv_hi, inv_lo;
        stream::split_scale(s_d, s_hi, s_lo);
        split_float(bad ? 0.0 : 1.0 / S, inv_hi, inv_lo);
        const unsigned char *z = (const unsigned char *)P.z + ((long long)b * P.seq_stride + (long long)(row % P.N) * P.node_stride) * ESZ;
        float *out = P.probs + (long long)row * P.V;
        const int t0 = part * KEPT_PART, t1 = min(P.V, t0 + KEPT_PART);
        if (bad == ROW_FAR) {
            write_far(z, DT, out, t0, t1, cut, __int_as_float(P.kept[2ll * row + 1]), s_d, S);
            continue;
        }
        const float near = (float)(((double)O - 4.0) / s_d);
        const auto prob = [&](float v) {
            if (!(v >= cut) || bad) return 0.f;
            if (v >= near) return heavy_prob(v, s_d, O, S);
            const float e = exp2_fine(v, s_hi, s_lo, O);
            return fmaf(e, inv_lo, e * inv_hi);
        };
        // (t0 is a multiple of 4; a row whose logits or probabilities start elsewhere goes token by token)
        if (((uintptr_t)z & (4 * ESZ - 1)) == 0 && ((uintptr_t)out & 15) == 0) {
            using Four = std::conditional_t<DT == SPEC_BF16, uint2, uint4>;
            Four raw[KEPT_STEPS];
#pragma unroll
            for (int k = 0; k < KEPT_STEPS; ++k) {
                const int t = t0 + (k * KEPT_NT + tid) * 4;
                if (t + 3 < t1) raw[k] = __ldg(reinterpret_cast<const Four *>(z + (size_t)t * ESZ));
            }
#pragma unroll
            for (int k = 0; k < KEPT_STEPS; ++k) {
                const int t = t0 + (k * KEPT_NT + tid) * 4;
                if (t + 3 < t1) {
                    float v[4];
                    if constexpr (DT == SPEC_BF16) {
                        v[0] = bf16_lo(raw[k].x); v[1] = bf16_hi(raw[k].x); v[2] = bf16_lo(raw[k].y); v[3] = bf16_hi(raw[k].y);
                    } else {
                        v[0] = __uint_as_float(raw[k].x); v[1] = __uint_as_float(raw[k].y); v[2] = __uint_as_float(raw[k].z); v[3] = __uint_as_float(raw[k].w);
                    }
                    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])) >= cut) o = make_float4(prob(v[0]), prob(v[1]), prob(v[2]), prob(v[3]));
                    *reinterpret_cast<float4 *>(out + t) = o;
                } else {
                    for (int i = t; i < t1; ++i) out[i] = prob(load_logit(z, DT, i));
                }
            }
        } else {
#pragma unroll 4
            for (int t = t0 + tid; t < t1; t += KEPT_NT) out[t] = prob(load_logit(z, DT, t));
        }
    }
}

// ------------------------------------------------------------------------------------------------
// spec_sample_bonus: inverse CDF over rows of fp32 weights
// ------------------------------------------------------------------------------------------------
// A cluster per row, a slice per CTA, a tile of 128 weights per warp and step.  The sums of the tiles stay in shared memory; the cluster
// exchanges the slices' sums, and the CTA that owns the target finds the tile by one scan and reads that tile once more.  Nothing else is
// kept, so an SM holds eight CTAs with four tiles per warp in flight.  76 rows of 128256 (39 MB, written just before): 20 us with
// the slices staged in shared memory, one CTA per SM; 12 now.
constexpr int BN_NT = 256, BN_TILE = 128, BN_TILES = 1024;      // tiles of a slice at most
constexpr int BN_CMAX = 8;
struct BParams {
    int R, V, SL;            // SL: weights of a slice, a multiple of BN_TILE
    const float *w, *u;
    int *token;
    float *margin;
};
// first lane with running sum > tau (and weight); else the last with weight and rest = inf; -1 where there is none.  (The sum ahead of the
// lane is a difference: it may exceed tau by a rounding, and what is left of tau is then 0.)
__device__ __forceinline__ int first_above(double v, double tau, double &rest)
{
    const int lane = threadIdx.x & 31;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, v > 0.0 && incl > tau), pos = __ballot_sync(0xffffffffu, v > 0.0);
    const int at = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
    const double before = __shfl_sync(0xffffffffu, incl - v, at < 0 ? 0 : at);
    rest = hit ? fmax(tau - before, 0.0) : CUDART_INF;
    return pos ? at : -1;
}
// the lane's four consecutive weights of a tile; beyond the slice: 0
__device__ __forceinline__ float4 tile_weights(const float *row, int t, int end, bool vec)
{
    if (vec && t + 3 < end) return __ldg(reinterpret_cast<const float4 *>(row + t));
    return make_float4(t < end ? __ldg(row + t) : 0.f, t + 1 < end ? __ldg(row + t + 1) : 0.f, t + 2 < end ? __ldg(row + t + 2) : 0.f,
                       t + 3 < end ? __ldg(row + t + 3) : 0.f);
}

__global__ void __launch_bounds__(BN_NT) spec_bonus_kernel(const BParams P)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int r_id = blockIdx.x / C, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ double tile[BN_TILES], total[BN_CMAX];
    grid_dependency_wait();
    const float *row = P.w + (long long)r_id * P.V;
    const bool vec = ((uintptr_t)row & 15) == 0;
    const int t0 = rank * P.SL, end = min(P.V, t0 + P.SL), tiles = max(0, (end - t0 + BN_TILE - 1) / BN_TILE);
    constexpr int AHEAD = 4, WARPS = BN_NT / 32;
    for (int i0 = warp; i0 < tiles; i0 += WARPS * AHEAD) {
        float4 x[AHEAD];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) x[k] = tile_weights(row, t0 + (i0 + k * WARPS) * BN_TILE + lane * 4, end, vec);
        double s[AHEAD];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) s[k] = ((double)x[k].x + (double)x[k].y) + ((double)x[k].z + (double)x[k].w);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < AHEAD; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        }
        if (lane < AHEAD) {
            const int i = i0 + lane * WARPS;
            const double mine = lane == 0 ? s[0] : lane == 1 ? s[1] : lane == 2 ? s[2] : s[3];
            if (i < tiles) tile[i] = mine;
        }
    }
    __syncthreads();
    // a run of tiles per lane (of every warp alike: the slice's sum is needed by all)
    const int per = ((tiles + 31) / 32) | 1, i0 = lane * per, i1 = min(tiles, i0 + per);
    double mine = 0.0;
    for (int i = i0; i < i1; ++i) mine += tile[i];
    const double slice = warp_sum(mine);
    if (C > 1) {
        cluster.sync();                  // peers must be running before their shared memory is written
        if (tid < C) *cluster.map_shared_rank(&total[rank], tid) = slice;
        cluster.sync();
    } else {
        if (tid == 0) total[0] = slice;
        __syncthreads();
    }
    const double share = lane < C ? total[lane] : 0.0;
    double all = 0.0;
    for (int r = 0; r < C; ++r) all += total[r];
    double tau, tau2, tau3;
    const int owner = first_above(share, (double)__ldg(P.u + r_id) * all, tau);
    if (owner < 0) {
        if (rank == 0 && tid == 0) { P.token[r_id] = -1; if (P.margin) P.margin[r_id] = 0.f; }
        return;
    }
    if (owner != rank || warp != 0) return;
    const int l = first_above(mine, tau, tau2);
    // the tile inside the lane's run, by that lane
    int ti = -1;
    double rest = tau2;
    if (lane == l) {
        int last = -1;
        double run = 0.0, upto = 0.0;
        for (int i = i0; i < i1; ++i) {
            const double x = tile[i];
            if (x > 0.0) last = i;
            if (x > 0.0 && run + x > tau2) { ti = i; upto = run; break; }
            run += x;
        }
        if (ti >= 0) rest = tau2 - upto;
        else { ti = last; rest = CUDART_INF; }
    }
    ti = __shfl_sync(0xffffffffu, ti, l < 0 ? 0 : l);
    rest = __shfl_sync(0xffffffffu, rest, l < 0 ? 0 : l);
    const int at = t0 + ti * BN_TILE + lane * 4;
    const float4 x = tile_weights(row, at, end, vec);
    const float v[4] = {x.x, x.y, x.z, x.w};
    const int who = first_above(((double)v[0] + (double)v[1]) + ((double)v[2] + (double)v[3]), rest, tau3);
    if (lane != who) return;
    int found = -1, last = -1;
    double run = 0.0, lo = 0.0, hi = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double before = run;
        run += (double)v[k];
        if (v[k] > 0.f) last = k;
        if (found < 0 && v[k] > 0.f && run > tau3) { found = k; lo = tau3 - before; hi = run - tau3; }
    }
    P.token[r_id] = at + (found >= 0 ? found : last);
    if (P.margin) P.margin[r_id] = found >= 0 ? (float)(fmin(lo, hi) / all) : 0.f;
}

}  // namespace rowops
}  // namespace specv
