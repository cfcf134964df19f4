// Pieces shared by the verification kernels (walk.cuh: SpecInfer along the accepted path, Algorithm 4
// composed top-down, Section 3.2; nodes.cuh: every node, Traversal Verification of Section 3.2 with the
// block-verification weights of Section 3.1): constants and shared-memory layouts, the handling of
// one chunk of 8 logits (load, mask, exponentiate), the residual pass over resident e, prefix picks,
// the inverse-CDF search for the bonus token, and the writing of a sequence's outputs from the node
// records.
//
// Common ground of the kernels.  A row is cut into chunks of 8 logits that start on 16-byte boundaries (the first
// chunk holds fewer where the row starts on none); each CTA of a cluster owns a contiguous range of chunks, each
// consumer thread every NCONS-th chunk of that range.  A logit becomes e = 2^(z s - O) with s = log2(e)/T and O the
// row's integer reference, so every scale factor is an exact power of two.  The e of a thread's first RC chunks stay
// in registers, the others in shared memory; nothing is written back to HBM.
//
// A node on chip is a chain of short dependent phases (load, exponentials, a few sweeps, each ended by a sum over the
// cluster), so it is bound by latency, not by bandwidth or arithmetic.  Hence every consumer thread loads its own
// logits, three chunks ahead of the one it works on (a ring filled by a producer warp kept 3 of 9 tiles in flight and cost a
// wait and a hand-back per tile: 5 us for the first pass at V = 128256, 2 us now).  All kernels have 8 warps: 8 consumers, or
// 7 and a helper warp (spec_recursion_kernel).
//
// The recursion is the paper's own, step by step.  A node's state after j rejected children is the
// residual law P_j with P_0 = p, held as u_j(t) = kappa_j P_j(t) in place of the resident e_p:
//     u_j(t) = (g_j u_{j-1}(t) - e_q(t))+ ,   g_j = w_{j-1} Z_q / kappa_{j-1} ,   kappa_j = sum_t u_j(t) ,
// which is Z_q (w_{j-1} P_{j-1} - q)+, so kappa_j = Z_q S_j with S_j the step's residual mass
// (SpecInfer: w = 1 throughout and child j is accepted with min(1, P_{j-1}(x) / q(x)); Traversal
// Verification: w_j = S_j / (S_j + 1 - w_{j-1}) and child j is handed min(1, w_{j-1} P_{j-1}(x) / q(x))).
// One sibling step is one sweep over the resident data (subtract, clamp, store, sum) plus one scalar
// exchange through distributed shared memory.  Every step renormalises, as the paper's
// P <- norm((P - q)+) does, so a state that is reached with probability 1e-15 is as well conditioned
// as the first one; a closed form in the original units, (w P_0 - c_j q)+ with accumulated c_j, is
// not: its difference cancels to the rounding of fp64 once the accumulated mass drops below 1e-11.
// The children's tokens follow the same recursion as scalars in fp64.
//
// Precision.  The e are fp32 (one ex2.approx each, relative error about 2^-22), which is not enough
// where a residual mass E_j is small against the probabilities it is the difference of (two peaked
// laws on the same token: near-greedy temperatures, top-k / top-p): w_in P0(x) - c_j q(x) then cancels
// to a few 1e-7 of its terms.  The few tokens that carry a row's mass are therefore kept exactly: every
// consumer warp owns a short list of DOMINANT tokens of its part of the slice (above 2^-DOM_A of the
// row's mass always; above 2^-DOM_B while the list has room), whose exponentials are evaluated in fp64
// and whose fp32 copies are set to zero.  Every sum over the vocabulary is then (fp32 over the tail,
// accumulated in fp64 above a thread) + (fp64 over the lists), and so are the rows' normalisers, which
// the cluster recomputes from the resident e instead of taking them from the statistics pass.
//
// Sums over the cluster.  Every consumer warp leaves its partial sum in its CTA's shared memory; one warp adds them up
// and sends the CTA's sum into the shared memory of all CTAs (st.async, which counts the bytes on the receiver's
// mbarrier); every warp waits on its own CTA's mbarrier and reduces the C sums itself.  One fixed order everywhere,
// so all warps of the cluster hold bit-identical totals and take identical decisions.
#pragma once
#include "common.cuh"
#include "stream.cuh"

namespace specv {

constexpr int CHMAX = 24;    // chunks per thread, in registers (RC of them) and shared memory
constexpr int CMAX = 16;     // CTAs per cluster (above 8: non-portable size)
constexpr int NWMAX = 8;     // consumer warps
constexpr int NVMAX = 6;     // doubles per sum over the cluster
constexpr int FAST_N = 32;   // trees up to this size are finished warp-parallel
constexpr int FIN_PENDING = -1;     // VParams::fin of a sequence whose nodes are not all done
constexpr int FIN_FAULTY = -2;      // ... of a sequence with a device-detected fault: no bonus draw
constexpr int FIN_LEN_SHIFT = 12;   // a selected node is published as node | (accepted length << FIN_LEN_SHIFT)
static_assert(SPEC_MAX_NODES <= (1 << FIN_LEN_SHIFT) && SPEC_MAX_NODES < (1 << (30 - FIN_LEN_SHIFT)), "packing of the published node");
// A residual step whose mass is below this fraction of the mass before it is treated as S = 0: where P
// equals q (the same row twice, two one-token nuclei on the same token) the exact difference is 0 and
// the computed one a few 1e-16 of the mass (the rounding of the coefficient g).
constexpr double RESIDUAL_FLOOR = 1.0e-13;
// Traversal: a handed-down weight this close to 1 is 1 (a ratio that is exactly 1 may come out one
// rounding below; the step after it is discontinuous at w = 1 when S = 0)
constexpr double WEIGHT_SNAP = 1.0e-12;

// exact list of dominant tokens, one per consumer warp
constexpr int MW = 32;       // entries (one per lane in a pass)
constexpr int MW_RES = 8;    // entries kept free for tokens above 2^-DOM_A of a row's mass
constexpr int DOM_A = 6;     // such a token is always listed: at most 64 per row, and they are what bounds the tail's error
constexpr int DOM_B = 34;    // tokens above 2^-DOM_B of a row's mass are listed while the list has room

enum Mode { MODE_SPECINFER = 0, MODE_TRAVERSAL = 1 };

// Traversal: a node of weight w hands its first child min(1, w ratio), with ratio = p(x) / q(x) of the unmodified rows
struct __align__(16) ChainRec {
    unsigned long long ratio;    // bits of the double; W_PENDING: not known; NO_CHILD
    int child;
    int parts;                   // of a peaked node's normalisers, while they are being summed (0 at launch)
};

struct VParams {
    int B, N, V, C, mode, all_thr;
    int early;                // let the next call's statistics take the places that are free (finish kernel)
    int off_es;               // byte offset of the resident e inside dynamic shared memory
    const void *zp, *zq;
    long long seq_stride, node_stride, topo_stride;
    const int *parent, *token;
    float T;
    const float *T_seq;
    const float *u_accept, *u_bonus;
    NodeRec *rec;
    unsigned long long *w_pub;   // [B*N] weight handed to a node by its parent (Traversal), W_PENDING until known
    unsigned int *done;          // [B] arrivals per sequence (one per node); the last one selects the accepted node
    int *fin;                    // [B] the accepted node once it is selected (FIN_PENDING before, FIN_FAULTY for a faulty sequence)
    ChainRec *chain;             // [B*N] the node's first child and its ratio
    SpecOut out;
};

struct __align__(16) WarpList {
    double ep[MW], eq[MW];         // exact 2^(z s - O) of the token in the target / draft row (0: cut, or no draft row)
    int pos[MW];                   // (chunk of the thread << 8) | (lane << 3) | position in the chunk
};

// the e of the RC register chunks of a thread
template <int RC> struct Resident {
    float p[RC > 0 ? RC : 1][8], q[RC > 0 ? RC : 1][8];
};

// shared memory of the consumer warps' common work
struct __align__(16) Common {
    uint64_t xbar[2], cbar;
    double part[2][NVMAX][NWMAX];  // the warps' partial sums, by parity of the sum
    double xsum[2][NVMAX][CMAX];   // the CTAs' sums
    double wtile[NWMAX + 1][CHMAX];
    WarpList list[NWMAX];
    int poison;
};
// a consumer warp's view of it
struct Team {
    Common &M;
    int C, warp, lane, n;          // n: sums so far
    unsigned rank;
    uint32_t cph;                  // phase of the consumers' barrier
};
__device__ __forceinline__ void common_init(Common &M, int nw)
{
    mbar_init(&M.xbar[0], 1);
    mbar_init(&M.xbar[1], 1);
    mbar_init(&M.cbar, nw);
    M.poison = 0;
}

// ------------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------------
// the CTA's chunks of a node's two rows
struct Slice {
    const unsigned char *p, *q;    // 16-byte boundaries at which chunk 0 of the rows starts
    int u0, nu;                    // first chunk and number of chunks of this CTA
    int h, V;                      // chunk u holds the row's logits 8 u - h .. 8 u - h + 7
    bool vec;                      // both rows start at the same offset from a 16-byte boundary
};
template <int DT>
__device__ __forceinline__ Slice make_slice(const void *zp, const void *zq, long long first, int V, int C, unsigned rank)
{
    constexpr int ESZ = DT == SPEC_BF16 ? 2 : 4;
    const uintptr_t ap = (uintptr_t)zp + (uintptr_t)(first * ESZ), aq = (uintptr_t)zq + (uintptr_t)(first * ESZ);
    Slice s;
    s.vec = ((ap ^ aq) & 15) == 0 && (ap & (ESZ - 1)) == 0;
    const int off = s.vec ? (int)(ap & 15) : 0;
    s.h = off / ESZ;
    s.p = (const unsigned char *)(ap - off);
    s.q = (const unsigned char *)(aq - off);
    s.V = V;
    const int units = (s.h + V + 7) >> 3, per = (units + C - 1) / C;
    s.u0 = (int)rank * per;
    s.nu = max(0, min(per, units - s.u0));
    return s;
}
// the 8 logits of a chunk as they sit in memory
template <int DT>
struct RawChunk {
    uint4 a, b;      // bf16: a only
};
// chunk u of one row; what lies outside the row may be anything (mask_chunk).  Rows at different offsets from a 16-byte
// boundary (two tensors of their own odd alignment) are read logit by logit, out of line.
template <int DT>
__device__ __noinline__ RawChunk<DT> load_raw_scalar(const unsigned char *row, int u, int V)
{
    RawChunk<DT> r;
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int t = min(u * 8 + k, V - 1);
        w[k] = DT == SPEC_BF16 ? (uint32_t)__ldg((const unsigned short *)row + t) : __ldg((const uint32_t *)row + t);
    }
    if (DT == SPEC_BF16) r.a = make_uint4(w[0] | w[1] << 16, w[2] | w[3] << 16, w[4] | w[5] << 16, w[6] | w[7] << 16);
    else { r.a = make_uint4(w[0], w[1], w[2], w[3]); r.b = make_uint4(w[4], w[5], w[6], w[7]); }
    return r;
}
template <int DT>
__device__ __forceinline__ RawChunk<DT> load_raw(const unsigned char *row, int u, const Slice &s)
{
    RawChunk<DT> r;
    const uint4 *src = reinterpret_cast<const uint4 *>(row) + (size_t)u * (DT == SPEC_BF16 ? 1 : 2);
    r.a = __ldg(src);
    if (DT == SPEC_F32) r.b = u * 8 - s.h + 4 < s.V ? __ldg(src + 1) : r.a;
    return r;
}
template <int DT>
__device__ __forceinline__ void unpack_chunk(const RawChunk<DT> &r, float (&z)[8])
{
    if (DT == SPEC_BF16) {
        z[0] = bf16_lo(r.a.x); z[1] = bf16_hi(r.a.x); z[2] = bf16_lo(r.a.y); z[3] = bf16_hi(r.a.y);
        z[4] = bf16_lo(r.a.z); z[5] = bf16_hi(r.a.z); z[6] = bf16_lo(r.a.w); z[7] = bf16_hi(r.a.w);
    } else {
        z[0] = __uint_as_float(r.a.x); z[1] = __uint_as_float(r.a.y); z[2] = __uint_as_float(r.a.z); z[3] = __uint_as_float(r.a.w);
        z[4] = __uint_as_float(r.b.x); z[5] = __uint_as_float(r.b.y); z[6] = __uint_as_float(r.b.z); z[7] = __uint_as_float(r.b.w);
    }
}
// logits outside the row (positions of the chunk outside lo .. hi - 1) or below the row's cut become -inf
__device__ __forceinline__ void mask_chunk(float (&z)[8], int lo, int hi, bool has_cut, float cut)
{
    if (lo > 0 || hi < 8) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < lo || k >= hi) z[k] = -CUDART_INF_F;
    }
    if (has_cut) {
#pragma unroll
        for (int k = 0; k < 8; ++k) z[k] = z[k] >= cut ? z[k] : -CUDART_INF_F;
    }
}

// e[k] = 2^(z[k] s - of) for the 8 logits of a chunk (the large product z s_hi - of is formed first, in
// one rounding, so that the exponent's error is relative to the exponent and not to of), of the thread's reference for this row (an
// integer-valued float); returns sum e.  FEAT: also sx += sum e x with x the exponent.
template <bool FEAT>
__device__ __forceinline__ float exp_chunk(const float (&z)[8], float s_hi, float s_lo, float of, float (&e)[8],
                                           float &sx)
{
    float sum = 0.f;
    if (FEAT) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float x = fmaxf(fmaf(z[k], s_lo, fmaf(z[k], s_hi, -of)), -200.f);
            e[k] = ex2_approx(x);
            sum += e[k];
            sx = fmaf(e[k], x, sx);
        }
    } else {
        // two exponents per instruction (fp32 pairs; each half is the scalar operation)
        const unsigned long long sh2 = pack_f32x2(s_hi, s_hi), sl2 = pack_f32x2(s_lo, s_lo), no2 = pack_f32x2(-of, -of);
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            const unsigned long long z2 = pack_f32x2(z[k], z[k + 1]);
            float x0, x1;
            unpack_f32x2(fma_f32x2(z2, sl2, fma_f32x2(z2, sh2, no2)), x0, x1);
            e[k] = ex2_approx(x0);
            e[k + 1] = ex2_approx(x1);
            sum += e[k] + e[k + 1];
        }
    }
    return sum;
}
__device__ __forceinline__ void load_e8(const float4 *d, int stride, float (&e)[8])
{
    const float4 lo = d[0], hi = d[stride];
    e[0] = lo.x; e[1] = lo.y; e[2] = lo.z; e[3] = lo.w; e[4] = hi.x; e[5] = hi.y; e[6] = hi.z; e[7] = hi.w;
}

// first lane whose running sum of v exceeds tau (v >= 0 in every lane); if rounding leaves none, the
// last lane with v > 0 and tau_res = +inf; -1 if no lane has weight.  All lanes get the same answer.
// Not inlined on purpose: it runs a handful of times per sequence, and one copy that is already in the
// instruction cache after its first call is faster than several cold ones.
__device__ __noinline__ int pick_lane(double v, double tau, double &tau_res)
{
    const int lane = threadIdx.x & 31;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const double excl = incl - v;
    const unsigned hit = __ballot_sync(0xffffffffu, incl > tau && v > 0.0);
    if (hit) {
        const int idx = __ffs(hit) - 1;
        tau_res = tau - __shfl_sync(0xffffffffu, excl, idx);
        return idx;
    }
    const unsigned pos = __ballot_sync(0xffffffffu, v > 0.0);
    tau_res = CUDART_INF;
    return pos ? 31 - __clz(pos) : -1;
}

// ------------------------------------------------------------------------------------------------
// pass 1: a node's rows into resident e, its dominant tokens into the warp's exact list
// ------------------------------------------------------------------------------------------------
// what pass 1 has to know about the two rows of a node
struct NodeRows {
    bool hq;                  // the node has children: its draft row is read too
    float cut_p, cut_q;       // smallest kept logit (-inf: nothing cut)
    int O_p, O_q;             // integer references of the rows
    float s_hi, s_lo;         // log2(e) / T = s_hi + s_lo
    double s_d;
    float thrA_p, thrA_q;     // e above this: always listed (2^-DOM_A of the row's mass)
    float thrB_p, thrB_q;     // e above this: listed while the list has room (2^-DOM_B)
};
// Z: the row's normaliser from the statistics pass (fp32 exponentials: good enough for a threshold).
// The second tier pays only where it can hold nearly all of a row's mass, that is on laws that are
// peaked (near-greedy temperatures, short nuclei), and it is needed only where a residual mass is small
// against the weight, which takes two laws that nearly agree on their heavy tokens: both rows peaked.
// The largest e of a row lies in (1/2, 1], so Z > LIST_FLAT_Z means that no token holds more than
// 1/LIST_FLAT_Z of the row's mass.  On such a row the tier would fill with the first tokens it meets and
// buy nothing, so it is left out; a node without a draft row (nothing is subtracted there) has no use
// for it either.
constexpr double LIST_FLAT_Z = 4.0;
__device__ __forceinline__ void set_list_thresholds(NodeRows &nr, double Z_p, double Z_q)
{
    const double a = 1.0 / (double)(1ull << DOM_A), b = 1.0 / (double)(1ull << DOM_B);
    const bool flat = !nr.hq || Z_p > LIST_FLAT_Z || Z_q > LIST_FLAT_Z;
    nr.thrA_p = (float)(Z_p * a);
    nr.thrB_p = flat ? nr.thrA_p : (float)(Z_p * b);
    nr.thrA_q = nr.hq ? (float)(Z_q * a) : CUDART_INF_F;
    nr.thrB_q = nr.hq ? (flat ? nr.thrA_q : (float)(Z_q * b)) : CUDART_INF_F;
}
// the e of the 8 tokens a thread owns in one chunk, both rows (passed by value to list_append)
struct Chunk16 {
    float p[8], q[8];
};

// logit k of a chunk
template <int DT>
__device__ __forceinline__ float raw_logit(const RawChunk<DT> &r, int k)
{
    const int j = DT == SPEC_BF16 ? k >> 1 : k & 3;
    const uint32_t x = (DT == SPEC_F32 && k >= 4) ? r.b.x : r.a.x, y = (DT == SPEC_F32 && k >= 4) ? r.b.y : r.a.y;
    const uint32_t z = (DT == SPEC_F32 && k >= 4) ? r.b.z : r.a.z, w = (DT == SPEC_F32 && k >= 4) ? r.b.w : r.a.w;
    const uint32_t v = j & 2 ? (j & 1 ? w : z) : (j & 1 ? y : x);
    return DT == SPEC_BF16 ? ((k & 1) ? bf16_hi(v) : bf16_lo(v)) : __uint_as_float(v);
}

// Warp-collective, and out of line on purpose (it runs on a few per cent of the chunks, and the kernels
// are short of instruction cache): the tokens of the lane's chunk whose e exceeds the always-listed
// threshold (thrA), or the while-there-is-room threshold (tp, tq), are appended to the warp's list while
// it has room, as raw logits (pass1 evaluates the exponentials in fp64 once all chunks are in).  Places are dealt by
// one scan over the lanes (position by position, with its ballots, it was the longest part of pass 1: 4 of 8.7
// thousand cycles at V = 1000).  n is the list's fill, the same in every lane.  Returns (new fill << 8) | the lane's
// mask of appended tokens (the caller zeroes their fp32 copies).
template <int DT>
__device__ __noinline__ unsigned list_append(WarpList &L, int n, const RawChunk<DT> raw_p, const RawChunk<DT> raw_q,
                                             const Chunk16 e, float thrA_p, float thrA_q, float tp, float tq, int lo, int hi,
                                             float cut_p, float cut_q, bool hq, int slot)
{
    const int lane = threadIdx.x & 31;
    unsigned m_a = 0, m_b = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (e.p[k] > thrA_p || e.q[k] > thrA_q) m_a |= 1u << k;
        if (e.p[k] > tp || e.q[k] > tq) m_b |= 1u << k;
    }
    m_b &= ~m_a;
    const unsigned mine = (unsigned)__popc(m_a) | (unsigned)__popc(m_b) << 16;
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned tot = __shfl_sync(0xffffffffu, incl, 31), before = incl - mine;
    const int capB = MW - MW_RES, nA = min(n + (int)(tot & 0xFFFFu), MW);
    int iA = n + (int)(before & 0xFFFFu), iB = nA + (int)(before >> 16);
    unsigned adm = 0;
    for (unsigned m = m_a | m_b; m; m &= m - 1u) {
        const int k = __ffs(m) - 1;
        const bool a = (m_a >> k) & 1u;
        const int idx = a ? iA++ : iB++;
        if (idx >= (a ? MW : capB)) continue;
        const float z0 = raw_logit<DT>(raw_p, k), z1 = raw_logit<DT>(raw_q, k);
        const bool valid = k >= lo && k < hi;
        L.ep[idx] = (valid && z0 >= cut_p) ? (double)z0 : -CUDART_INF;      // (-inf: cut, or no draft row)
        L.eq[idx] = (valid && hq && z1 >= cut_q) ? (double)z1 : -CUDART_INF;
        L.pos[idx] = (slot << 8) | (lane << 3) | k;
        adm |= 1u << k;
    }
    __syncwarp();
    return (unsigned)max(nA, min(nA + (int)(tot >> 16), capB)) << 8 | adm;
}

// cross sums of the two rows for the Kullback-Leibler divergences (analysis instantiation only):
// sum e_p x_p, sum e_p x_q, sum e_q x_p, sum e_q x_q with x = z s - O the exponents (a token cut from one row
// has x = -inf there, which makes the divergence from the other row infinite, as it is)
struct KlSums {
    float pp, pq, qp, qq;
};

// chunk i of the CTA in both rows (zeros beyond the CTA's chunks)
template <int DT>
__device__ __forceinline__ void fetch_pair(const Slice &sl, bool hq, int i, RawChunk<DT> &p, RawChunk<DT> &q)
{
    p.a = q.a = make_uint4(0, 0, 0, 0);
    if (DT == SPEC_F32) p.b = q.b = make_uint4(0, 0, 0, 0);
    if (i >= sl.nu) return;
    if (sl.vec) {
        p = load_raw<DT>(sl.p, sl.u0 + i, sl);
        if (hq) q = load_raw<DT>(sl.q, sl.u0 + i, sl);
    } else {
        p = load_raw_scalar<DT>(sl.p, sl.u0 + i, sl.V);
        if (hq) q = load_raw_scalar<DT>(sl.q, sl.u0 + i, sl.V);
    }
}

// One chunk: its 8 logits of both rows into e (EP, EQ), dominant tokens to the list.  The thread's tail sums of e go to
// zs_p / zs_q.  c: the chunk's index in the thread.
template <int DT, int NW, bool KLS = false>
__device__ __forceinline__ void pass1_chunk(const Slice &sl, const NodeRows &nr, const RawChunk<DT> &raw_p, const RawChunk<DT> &raw_q,
                                            int c, int tid, float (&EP)[8], float (&EQ)[8], WarpList &L, int &nl, float &zs_p,
                                            float &zs_q, KlSums *kl = nullptr)
{
    const int i = c * NW * 32 + tid, t0 = (sl.u0 + i) * 8 - sl.h;
    const int lo = -t0, hi = i < sl.nu ? sl.V - t0 : 0;          // positions that are the row's
    float z[8], dsx = 0.f;
    float sum_p, sum_q = 0.f;
    if (KLS) {
        // the exponents themselves are needed: scalar form
        float xp[8], xq[8];
        unpack_chunk<DT>(raw_p, z);
        mask_chunk(z, lo, hi, nr.cut_p > -CUDART_INF_F, nr.cut_p);
        sum_p = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) { xp[k] = fmaf(z[k], nr.s_lo, fmaf(z[k], nr.s_hi, -(float)nr.O_p)); EP[k] = ex2_approx(xp[k]); sum_p += EP[k]; }
        unpack_chunk<DT>(raw_q, z);
        mask_chunk(z, lo, hi, nr.cut_q > -CUDART_INF_F, nr.cut_q);
#pragma unroll
        for (int k = 0; k < 8; ++k) { xq[k] = fmaf(z[k], nr.s_lo, fmaf(z[k], nr.s_hi, -(float)nr.O_q)); EQ[k] = ex2_approx(xq[k]); sum_q += EQ[k]; }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (EP[k] > 0.f) { kl->pp = fmaf(EP[k], xp[k], kl->pp); kl->pq = fmaf(EP[k], xq[k], kl->pq); }
            if (EQ[k] > 0.f) { kl->qp = fmaf(EQ[k], xp[k], kl->qp); kl->qq = fmaf(EQ[k], xq[k], kl->qq); }
        }
    } else {
        unpack_chunk<DT>(raw_p, z);
        mask_chunk(z, lo, hi, nr.cut_p > -CUDART_INF_F, nr.cut_p);
        sum_p = exp_chunk<false>(z, nr.s_hi, nr.s_lo, (float)nr.O_p, EP, dsx);
        if (nr.hq) {
            unpack_chunk<DT>(raw_q, z);
            mask_chunk(z, lo, hi, nr.cut_q > -CUDART_INF_F, nr.cut_q);
            sum_q = exp_chunk<false>(z, nr.s_hi, nr.s_lo, (float)nr.O_q, EQ, dsx);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) EQ[k] = 0.f;
        }
    }
    // dominant tokens: a chunk whose sum stays below the threshold holds none (e >= 0)
    const bool room = nl < MW - MW_RES;
    const float tp = room ? nr.thrB_p : nr.thrA_p, tq = room ? nr.thrB_q : nr.thrA_q;
    if (__any_sync(0xffffffffu, sum_p > tp || sum_q > tq)) {
        Chunk16 e;
#pragma unroll
        for (int k = 0; k < 8; ++k) { e.p[k] = EP[k]; e.q[k] = EQ[k]; }
        const unsigned r = list_append<DT>(L, nl, raw_p, raw_q, e, nr.thrA_p, nr.thrA_q, tp, tq, lo, hi, nr.cut_p,
                                           nr.cut_q, nr.hq, c);
        nl = (int)(r >> 8);
        const unsigned adm = r & 255u;
        if (adm) {
            sum_p = 0.f; sum_q = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if ((adm >> k) & 1u) { EP[k] = 0.f; EQ[k] = 0.f; }
                sum_p += EP[k]; sum_q += EQ[k];
            }
        }
    }
    zs_p += sum_p;
    zs_q += sum_q;
}

// the listed tokens' exponentials in fp64, an entry per lane (list_append left the raw logits)
__device__ __forceinline__ void list_exact(WarpList &L, int nl, const NodeRows &nr)
{
    __syncwarp();
    const int i = threadIdx.x & 31;
    if (i < nl) {
        const double zp = L.ep[i], zq = L.eq[i];
        L.ep[i] = zp > -CUDART_INF ? exp2_exact((float)zp, nr.s_d, nr.O_p) : 0.0;
        L.eq[i] = zq > -CUDART_INF ? exp2_exact((float)zq, nr.s_d, nr.O_q) : 0.0;
    }
    __syncwarp();
}

// Pass 1 of a node.  es: [chunk - RC][p lo, p hi, q lo, q hi][NCONS].  On return nl is the fill of the warp's list and
// zs_p / zs_q the thread's sums of the fp32 e it keeps (listed tokens excluded).
template <int DT, int NW, int RC, bool KLS = false>
__device__ __forceinline__ void pass1(const Slice &sl, const NodeRows &nr, float4 *es, int tid, Resident<RC> &R, WarpList &L,
                                      int &nl, float &zs_p, float &zs_q, KlSums *kl = nullptr)
{
    constexpr int NCONS = NW * 32;
    nl = 0; zs_p = 0.f; zs_q = 0.f;
    if (RC > 0) {
        // every load of the register chunks is issued before the first is used
        RawChunk<DT> rp[RC > 0 ? RC : 1], rq[RC > 0 ? RC : 1];
#pragma unroll
        for (int c = 0; c < RC; ++c) fetch_pair<DT>(sl, nr.hq, c * NCONS + tid, rp[c], rq[c]);
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            if (c * NCONS < sl.nu) {
                pass1_chunk<DT, NW, KLS>(sl, nr, rp[c], rq[c], c, tid, R.p[c], R.q[c], L, nl, zs_p, zs_q, kl);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) { R.p[c][k] = 0.f; R.q[c][k] = 0.f; }
            }
        }
    }
    // the others, one piece of code for all of them, three chunks' loads ahead
    RawChunk<DT> ap, aq, bp, bq, cp, cq;
    fetch_pair<DT>(sl, nr.hq, RC * NCONS + tid, ap, aq);
    fetch_pair<DT>(sl, nr.hq, (RC + 1) * NCONS + tid, bp, bq);
    fetch_pair<DT>(sl, nr.hq, (RC + 2) * NCONS + tid, cp, cq);
#pragma unroll 1
    for (int c = RC; c * NCONS < sl.nu; ++c) {
        const RawChunk<DT> xp = ap, xq = aq;
        ap = bp; aq = bq; bp = cp; bq = cq;
        fetch_pair<DT>(sl, nr.hq, (c + 3) * NCONS + tid, cp, cq);
        float ep[8], eq[8];
        pass1_chunk<DT, NW, KLS>(sl, nr, xp, xq, c, tid, ep, eq, L, nl, zs_p, zs_q, kl);
        float4 *d = es + (size_t)((c - RC) * 4) * NCONS + tid;
        d[0] = make_float4(ep[0], ep[1], ep[2], ep[3]);
        d[NCONS] = make_float4(ep[4], ep[5], ep[6], ep[7]);
        d[2 * NCONS] = make_float4(eq[0], eq[1], eq[2], eq[3]);
        d[3 * NCONS] = make_float4(eq[4], eq[5], eq[6], eq[7]);
    }
    list_exact(L, nl, nr);
}

// One step on a chunk: u <- (g u - q)+ for its 8 tokens, g = gh + gl; returns the sum of the new u
// (two tokens per fused multiply-add; q - g u is formed and its negation clamped)
__device__ __forceinline__ float step_chunk(float (&u)[8], const float (&q)[8], float gh, float gl)
{
    const unsigned long long ngh2 = pack_f32x2(-gh, -gh), ngl2 = pack_f32x2(-gl, -gl);
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        const unsigned long long u2 = pack_f32x2(u[k], u[k + 1]);
        float d0, d1;
        unpack_f32x2(fma_f32x2(ngl2, u2, fma_f32x2(ngh2, u2, pack_f32x2(q[k], q[k + 1]))), d0, d1);
        u[k] = fmaxf(-d0, 0.f);
        u[k + 1] = fmaxf(-d1, 0.f);
        acc += u[k] + u[k + 1];
    }
    return acc;
}
__device__ __forceinline__ float sum_chunk(const float (&u)[8])
{
    return ((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + (u[6] + u[7]));
}

// One sibling step over the thread's share of the resident node (nu: the CTA's chunks), in place: u <- (g u - e_q)+ for its
// fp32 tail tokens and for the entry of the warp's exact list that falls to its lane.  Returns the
// thread's sum of the new u.
template <int NW, int RC>
__device__ __forceinline__ double step_sweep(float4 *es, int nu, int tid, Resident<RC> &R, WarpList &L, int nl, double g)
{
    constexpr int NCONS = NW * 32;
    float g_hi, g_lo;
    split_float(g, g_hi, g_lo);
    float tot = 0.f;
#pragma unroll 1
    for (int c = RC; c * NCONS < nu; ++c) {
        float u[8], q[8];
        float4 *d = es + (size_t)((c - RC) * 4) * NCONS + tid;
        load_e8(d, NCONS, u);
        load_e8(d + 2 * NCONS, NCONS, q);
        tot += step_chunk(u, q, g_hi, g_lo);
        d[0] = make_float4(u[0], u[1], u[2], u[3]);
        d[NCONS] = make_float4(u[4], u[5], u[6], u[7]);
    }
    float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < RC; ++c) part[c & 3] += step_chunk(R.p[c], R.q[c], g_hi, g_lo);
    tot += (part[0] + part[1]) + (part[2] + part[3]);
    double d = (double)tot;
    const int lane = tid & 31;
    if (lane < nl) {
        const double v = fmax(fma(g, L.ep[lane], -L.eq[lane]), 0.0);
        L.ep[lane] = v;
        d += v;
    }
    return d;
}

// SpecTr's residual (Algorithm 3) in place, in the units of the resident e_p: u <- (u - gm min(u ir, e_q r))+
// with ir = 1 / rho, r = Z_p / Z_q, gm = gamma, for the thread's fp32 tail tokens and for the entry of the
// warp's exact list that falls to its lane.  Returns the thread's sum of the new u.
template <int NW, int RC>
__device__ __forceinline__ double spectr_sweep(float4 *es, int nu, int tid, Resident<RC> &R, WarpList &L, int nl, double gm,
                                               double ir, double r)
{
    constexpr int NCONS = NW * 32;
    const float gf = (float)gm, irf = (float)ir, rf = (float)r;
    float tot = 0.f;
#pragma unroll 1
    for (int c = RC; c * NCONS < nu; ++c) {
        float u[8], q[8];
        float4 *d = es + (size_t)((c - RC) * 4) * NCONS + tid;
        load_e8(d, NCONS, u);
        load_e8(d + 2 * NCONS, NCONS, q);
#pragma unroll
        for (int k = 0; k < 8; ++k) { u[k] = fmaxf(u[k] - gf * fminf(u[k] * irf, q[k] * rf), 0.f); tot += u[k]; }
        d[0] = make_float4(u[0], u[1], u[2], u[3]);
        d[NCONS] = make_float4(u[4], u[5], u[6], u[7]);
    }
#pragma unroll
    for (int j = 0; j < RC; ++j) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            R.p[j][k] = fmaxf(R.p[j][k] - gf * fminf(R.p[j][k] * irf, R.q[j][k] * rf), 0.f);
            tot += R.p[j][k];
        }
    }
    double d = (double)tot;
    const int lane = tid & 31;
    if (lane < nl) {
        const double v = fmax(L.ep[lane] - gm * fmin(L.ep[lane] * ir, L.eq[lane] * r), 0.0);
        L.ep[lane] = v;
        d += v;
    }
    return d;
}

// A read-only sweep over the thread's share of the resident node: f.tail8(e_p, e_q, a) on every 8 fp32 tokens (f's running
// sums), f.exact(...) in fp64 on the entry of the warp's exact list that falls to the lane.  Listed tokens are zero
// in the fp32 arrays; every f maps (0, 0) to nothing.
template <int NW, int RC, int NO, typename F>
__device__ __forceinline__ void reduce_sweep(const float4 *es, int nu, int tid, const Resident<RC> &R, const WarpList &L, int nl,
                                             const F &f, double (&o)[NO])
{
    constexpr int NCONS = NW * 32;
    float a[NO];
#pragma unroll
    for (int i = 0; i < NO; ++i) a[i] = 0.f;
#pragma unroll 1
    for (int c = RC; c * NCONS < nu; ++c) {
        float p[8], q[8];
        const float4 *d = es + (size_t)((c - RC) * 4) * NCONS + tid;
        load_e8(d, NCONS, p);
        load_e8(d + 2 * NCONS, NCONS, q);
        f.tail8(p, q, a);
    }
#pragma unroll
    for (int j = 0; j < RC; ++j) f.tail8(R.p[j], R.q[j], a);
#pragma unroll
    for (int i = 0; i < NO; ++i) o[i] = (double)a[i];
    if ((tid & 31) < nl) f.exact(L.ep[tid & 31], L.eq[tid & 31], o);
}

// barrier of the consumer warps of a CTA on an mbarrier (one arrival per warp), with a bounded wait
__device__ __forceinline__ void consumer_sync(Team &T)
{
    __syncwarp();
    if (T.lane == 0) mbar_arrive(&T.M.cbar);
    if (!*(volatile int *)&T.M.poison && !mbar_wait(&T.M.cbar, T.cph)) T.M.poison = 1;
    T.cph ^= 1u;
}

// Sums of NV doubles per consumer thread over the cluster: tot[i] over everything (bit-identical in all warps of all
// CTAs: one fixed order), mine[i] in lane r < C the sum over CTA r.
template <int NW, int NV>
__device__ __forceinline__ void cluster_sum(Team &T, const double (&v)[NV], double (&tot)[NV], double (&mine)[NV])
{
    static_assert(NV <= NVMAX, "room for the partial sums");
    Common &M = T.M;
    const int par = T.n & 1;
    double s[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] = v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int i = 0; i < NV; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
    }
    if (T.lane < NV) {
        double x = s[0];
#pragma unroll
        for (int i = 1; i < NV; ++i) x = T.lane == i ? s[i] : x;
        M.part[par][T.lane][T.warp] = x;
    }
    if (T.C > 1 && T.warp == 0 && T.lane == 0) mbar_arrive_expect_tx(&M.xbar[par], (uint32_t)(T.C * 8 * NV));
    consumer_sync(T);
    if (T.C == 1 || T.warp == 0) {
        // every lane adds up all partial sums by itself: broadcast reads and a tree of additions, no shuffles
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            double x[8];
#pragma unroll
            for (int w = 0; w < 8; ++w) x[w] = w < NW ? M.part[par][i][w] : 0.0;
#pragma unroll
            for (int h = 4; h > 0; h >>= 1) {
#pragma unroll
                for (int w = 0; w < h; ++w) x[w] += x[w + h];
            }
            tot[i] = x[0];
            mine[i] = T.lane == 0 ? x[0] : 0.0;
            if (T.C > 1 && T.lane < T.C) st_async_f64(&M.xsum[par][i][T.rank], &M.xbar[par], (uint32_t)T.lane, x[0]);
        }
    }
    if (T.C > 1) {
        if (!*(volatile int *)&M.poison && !mbar_wait_cluster(&M.xbar[par], (uint32_t)((T.n >> 1) & 1))) M.poison = 1;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            double x[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] = r < T.C ? M.xsum[par][i][r] : 0.0;
            if (T.C > 8) {
#pragma unroll
                for (int r = 0; r < 8; ++r) x[r] += M.xsum[par][i][r + 8];
            }
            tot[i] = ((x[0] + x[4]) + (x[2] + x[6])) + ((x[1] + x[5]) + (x[3] + x[7]));
            mine[i] = T.lane < T.C ? M.xsum[par][i][T.lane] : 0.0;
        }
    }
    ++T.n;
}

// Inverse-CDF search over one CTA's share of the node's current state u (from_q: of the draft row e_q
// instead, for a state that equals q), run by all consumer warps of the CTA that owns the target
// (tau_rel, in units of e).  Token order is (chunk of the thread, warp, lane, position in the chunk): that is also how
// the search descends.  The per-chunk totals of a warp are reduced together, so that their shuffles overlap.  Listed
// tokens enter with their exact values.
// role: 1 = this thread found the token (index in the row in `token`, distance to the nearer
// CDF edge in `edge`, in units of e); 2 = this thread reports that no token carries weight;
// 3 = this thread reports that a bounded wait ran out; 0 = nothing to do. 
struct BonusFind {
    int role, token;
    double edge;
};
template <int NW, int RC>
__device__ __forceinline__ BonusFind bonus_search(Team &T, const Slice &sl, const float4 *es, int tid, const Resident<RC> &R,
                                                  const WarpList &L, int nl, bool from_q, double tau_rel)
{
    constexpr int NCONS = NW * 32;
    const int warp = T.warp, lane = T.lane;
    double (*wtile)[CHMAX] = T.M.wtile;
    const int qoff = from_q ? 2 * NCONS : 0;
    BonusFind out = {0, -1, 0.0};
    // the warp's total of every chunk: fp32 sums of 8 in a lane, its listed tokens exactly, fp64 across lanes
    const double lr = lane < nl ? (from_q ? L.eq[lane] : L.ep[lane]) : 0.0;
    const int lpos = lane < nl ? L.pos[lane] : -1;
    double r[RC > 0 ? RC : 1], mine = 0.0;
#pragma unroll
    for (int c = 0; c < RC; ++c) r[c] = (double)(from_q ? sum_chunk(R.q[c]) : sum_chunk(R.p[c])) + ((lpos >> 8) == c ? lr : 0.0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int c = 0; c < RC; ++c) r[c] += __shfl_xor_sync(0xffffffffu, r[c], o);
    }
#pragma unroll
    for (int c = 0; c < RC; ++c)
        if (lane == c) mine = r[c];
#pragma unroll 1
    for (int c = RC; c * NCONS < sl.nu; ++c) {
        float p[8];
        load_e8(es + (size_t)((c - RC) * 4) * NCONS + tid + qoff, NCONS, p);
        const double x = warp_sum_once((double)sum_chunk(p) + ((lpos >> 8) == c ? lr : 0.0));
        if (lane == c) mine = x;
    }
    if (lane < CHMAX) wtile[warp][lane] = mine;
    consumer_sync(T);
    // every warp picks the chunk and the warp inside it for itself; the one that is picked goes on
    if (*(volatile int *)&T.M.poison) {
        if (tid == 0) out.role = 3;
        return out;
    }
    double Ti = 0.0;
    if (lane < CHMAX) {
        double x[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) x[w] = wtile[w][lane];
#pragma unroll
        for (int w = 1; w < NW; ++w) x[0] += x[w];
        Ti = x[0];
    }
    double tau2, tau3 = 0.0, tau4;
    const int s_star = pick_lane(Ti, tau_rel, tau2);
    const int w_star = s_star >= 0 ? pick_lane(lane < NW ? wtile[lane][s_star] : 0.0, tau2, tau3) : -1;
    if (w_star < 0) {
        if (tid == 0) out.role = 2;
        return out;
    }
    if (warp != w_star) return out;
    float p[8];
    if (s_star >= RC) {
        load_e8(es + (size_t)((s_star - RC) * 4) * NCONS + tid + qoff, NCONS, p);
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) p[k] = 0.f;
#pragma unroll
        for (int c = 0; c < RC; ++c)
            if (c == s_star) {
#pragma unroll
                for (int k = 0; k < 8; ++k) p[k] = from_q ? R.q[c][k] : R.p[c][k];
            }
    }
    double wk[8], v = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) wk[k] = (double)p[k];
    // the listed tokens of this chunk: each goes to the lane and position it was taken from
    for (unsigned m = __ballot_sync(0xffffffffu, lpos >= 0 && (lpos >> 8) == s_star); m; m &= m - 1u) {
        const int i = __ffs(m) - 1;
        const int ps = __shfl_sync(0xffffffffu, lpos, i);
        const double rv = __shfl_sync(0xffffffffu, lr, i);
        if (((ps >> 3) & 31) == lane) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if ((ps & 7) == k) wk[k] = rv;
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) v += wk[k];
    const int l_star = pick_lane(v, tau3, tau4);
    if (l_star < 0) {
        if (lane == 0) out.role = 2;
        return out;
    }
    if (lane == l_star) {
        double run = 0.0, dlo = 0.0, dhi = 0.0;
        int found = -1, last_pos = -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double before = run;
            run += wk[k];
            if (wk[k] > 0.0) last_pos = k;
            if (found < 0 && run > tau4) { found = k; dlo = tau4 - before; dhi = run - tau4; }
        }
        if (found < 0) { found = last_pos; dlo = 0.0; dhi = 0.0; }
        out.role = found >= 0 ? 1 : 2;
        out.token = found >= 0 ? (sl.u0 + s_star * NCONS + tid) * 8 - sl.h + found : -1;
        out.edge = fmin(dlo, dhi);
    }
    return out;
}

// ------------------------------------------------------------------------------------------------
// selecting the accepted node of one sequence: run by the whole warp whose lane made the last arrival
// ------------------------------------------------------------------------------------------------
// Writes every output of the sequence except the bonus token (accepted node, length, path tokens, status,
// the per-node diagnostics) and publishes the accepted node in P.fin for the sequence's finish kernel.
__device__ __noinline__ void finalize_sequence(const VParams &P, int b)
{
    const int lane = threadIdx.x & 31;
    const int N = P.N;
    const int *parent = P.parent + (long long)b * P.topo_stride;
    const int *token = P.token + (long long)b * N;
    const NodeRec *rec = P.rec + (long long)b * N;
    const float *ua = P.u_accept + (long long)b * N;
    int acc = -1, len = 0;
    const bool fast = N <= FAST_N;
    // a lane's own node, everything the selection needs of it fetched in one round of loads
    const bool own = fast && lane < N;
    const int par = own ? __ldg(parent + lane) : -2;
    const int tok = own ? __ldg(token + lane) : -1;
    const int nx = own ? __ldcg(&rec[lane].next_child) : -1;
    const double thr_l = own ? __ldcg(&rec[lane].thr) : 0.0;
    const float ua_l = own ? __ldg(ua + lane) : 0.f;
    int status = 0;
    for (int i = lane; i < N; i += 32) status = max(status, __ldcg(&rec[i].status));
    status = __reduce_max_sync(0xffffffffu, status);
    // (fast path) the ancestors of the lane's node, itself included, as a bit mask: pointer doubling, five
    // rounds for up to 32 levels; on a tree whose parents come first (checked by the nodes: status)
    unsigned anc = own ? 1u << lane : 0u;
    if (fast) {
        int jump = own ? par : -1;
#pragma unroll
        for (int it = 0; it < 5; ++it) {
            const int src = jump < 0 ? lane : jump;
            const unsigned up = __shfl_sync(0xffffffffu, anc, src);
            const int jj = __shfl_sync(0xffffffffu, jump, src);
            if (jump >= 0) { anc |= up; jump = jj; }
        }
    }
    if (!status) {
        if (fast) {
            if (P.mode == MODE_SPECINFER) {
                acc = 0;
                for (int hop = 0; hop < N; ++hop) {
                    const int n = __shfl_sync(0xffffffffu, nx, acc);
                    if (n < 0 || n >= N) break;
                    acc = n;
                }
            } else {
                // Depth-first post-order; the first node with u < w_fin (the root always) is accepted.  With H the
                // set of nodes whose subtree holds such a node: from the root, step to the first child in H
                // while there is one (the subtrees of the children before it are rejected as a whole).
                const bool hit = own && (lane == 0 || (double)ua_l < thr_l);
                const unsigned H = __reduce_or_sync(0xffffffffu, hit ? anc : 0u);
                int cur = 0;
                for (int d = 0; d < N; ++d) {
                    const unsigned m = __ballot_sync(0xffffffffu, own && par == cur && ((H >> lane) & 1u));
                    if (!m) break;
                    cur = __ffs(m) - 1;
                }
                acc = cur;
            }
            // the path's length is the accepted node's depth
            len = __popc(__shfl_sync(0xffffffffu, anc, acc)) - 1;
        } else {
            if (lane == 0) {
                if (P.mode == MODE_SPECINFER) {
                    acc = 0;
                    for (int hop = 0; hop < N; ++hop) {
                        int nx = __ldcg(&rec[acc].next_child);
                        if (nx < 0) break;
                        acc = nx;
                    }
                } else {
                    int cur = 0;
                    for (int guard = 0; guard < 4 * N + 4 && acc < 0; ++guard) {
                        for (;;) {
                            int fc = -1;
                            for (int c = cur + 1; c < N; ++c)
                                if (parent[c] == cur) { fc = c; break; }
                            if (fc < 0) break;
                            cur = fc;
                        }
                        for (;;) {
                            if (cur == 0 || (double)ua[cur] < __ldcg(&rec[cur].thr)) { acc = cur; break; }
                            const int p = parent[cur];
                            int sib = -1;
                            for (int d = cur + 1; d < N; ++d)
                                if (parent[d] == p) { sib = d; break; }
                            if (sib >= 0) { cur = sib; break; }
                            cur = p;
                        }
                    }
                }
                if (acc >= 0)
                    for (int x = acc; x != 0; x = parent[x]) ++len;
            }
            acc = __shfl_sync(0xffffffffu, acc, 0);
            len = __shfl_sync(0xffffffffu, len, 0);
        }
        if (acc < 0) status = SPEC_DEV_TOPOLOGY;
    }
    if (status) { acc = -1; len = -1; }
    int *ot = P.out.out_tokens + (long long)b * N;
    if (fast) {
        // a node on the accepted path (an ancestor of the accepted node, or that node; not the root) puts its
        // token at its depth - 1
        const unsigned path = acc >= 0 ? __shfl_sync(0xffffffffu, anc, acc) : 0u;
        const int mine = (own && lane > 0 && ((path >> lane) & 1u)) ? __popc(anc) - 1 : 0;
        for (int j = lane; j < N; j += 32) ot[j] = -1;
        __syncwarp();
        if (mine > 0) ot[mine - 1] = tok;
    } else {
        for (int i = lane; i < N; i += 32) ot[i] = -1;
        __syncwarp();
        if (lane == 0 && acc >= 0) {
            int i = len;
            for (int x = acc; x != 0 && i > 0; x = parent[x]) ot[--i] = token[x];
        }
    }
    if (lane == 0) {
        P.out.accepted_node[b] = acc;
        P.out.accept_len[b] = len;
        P.out.bonus_token[b] = -1;         // the finish kernel draws it
        P.out.status[b] = status;
        if (P.out.margin) P.out.margin[(long long)b * (N + 1) + N] = CUDART_NAN_F;   // (the finish kernel's slot)
    }
    // publication: the outputs above are visible to whoever sees the accepted node (the diagnostics below
    // are read by nobody on the device)
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        *(volatile int *)(P.fin + b) = status ? FIN_FAULTY : (acc | (len << FIN_LEN_SHIFT));
    }
    if (P.out.node_thr)
        for (int i = lane; i < N; i += 32) P.out.node_thr[(long long)b * N + i] = (float)__ldcg(&rec[i].thr);
    if (P.out.node_w_in && P.mode == MODE_TRAVERSAL)
        for (int i = lane; i < N; i += 32) P.out.node_w_in[(long long)b * N + i] = (float)__ldcg(&rec[i].w_in);
    if (P.out.margin) {
        float *mg = P.out.margin + (long long)b * (N + 1);
        for (int i = lane; i < N; i += 32)
            mg[i] = i == 0 ? CUDART_NAN_F : (float)fabs((double)ua[i] - __ldcg(&rec[i].thr));
    }
}

// The arrival of `count` nodes at their sequence (a node and the childless children it finished), made
// by lane 0 of a converged warp; the warp that makes the last of the N arrivals selects the accepted node.
__device__ __forceinline__ void arrive_sequence(const VParams &P, int b, unsigned count = 1u)
{
    int last = 0;
    if ((threadIdx.x & 31) == 0) {
        // release: the node's record (written by this warp, ordered before by __syncwarp where another
        // lane wrote it) is visible to whoever sees the count; acquire: the last arrival sees all records
        unsigned prev;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(prev) : "l"(P.done + b), "r"(count) : "memory");
        last = (prev + count == (unsigned)P.N) ? 1 : 0;
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    if (last) finalize_sequence(P, b);
}

}  // namespace specv
