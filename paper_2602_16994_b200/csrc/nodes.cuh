// Whole-tree verification on top of the row statistics (stream.cuh / trunc.cuh): Traversal Verification, whose weights are
// defined for every node, top-down (Section 3.2), SpecInfer's diagnostic outputs (the threshold of every node,
// Algorithm 4), and the offline analysis.
//
// What a node needs depends on its children:
//   none          its weight is the one it is handed: finished with its parent;
//   one           its child's weight is two logits and two normalisers, its own the residual mass of one step: one sum over
//                 the two rows, nothing resident (spec_single_kernel, a CTA or a small cluster per node);
//   two or more   the residual recursion of verify.cuh, step by step, over resident rows (spec_recursion_kernel, a cluster per
//                 node; in the analysis every node with children).
// Weights flow down without waiting for rows: a node hands its first child min(1, w ratio) with ratio the quotient of two
// probabilities of the unmodified rows, and a kernel of their own writes all ratios (spec_ratio_kernel).  Whoever
// publishes a node's weight publishes those of its whole line of first children (publish_weight), so the only chain of
// dependent vocabulary-wide work is from branching node to branching node.  The accepted node of a sequence is selected by
// whoever makes its last arrival, and one more kernel (spec_finish_kernel, a cluster per sequence) brings that node on chip,
// takes its recorded steps and draws the bonus token.
//
// Order of the kernels: ratios (Traversal only), recursion, single, finish.  They overlap (programmatic dependent launch): a
// kernel's CTAs take the places that the one before leaves free and poll, with a limit, for what is published.  A kernel
// starts only when all CTAs of the one before have started, and polls only for words that its own smaller items or
// EARLIER kernels write:
//   ratio      polls for nothing;
//   recursion  ratios: from the ratio kernel; weights: from it, or from a smaller item of its own (drawn before it, hence
//              running);
//   single     ratios (exact normalisers come with them): from the ratio kernel; weights: from it or the recursion, never
//              from its own kind;
//   finish     accepted nodes: from the recursion or the single kernel.
// So the calls of a stream come out the same when nothing overlaps (kernels run one at a time by a profiler, a debugger or
// CUDA_LAUNCH_BLOCKING), and when kernels of other streams hold any part of the chip.  A kernel ends only after the
// one before it has ended.
//
// Measured at V = 128256, bf16, batch 8, trunk of 2 and 4 branches of 4 (one branching node per sequence): see the
// kernels.  A single kernel in which every node was an item of a cluster took 74 to 80 us here: its items cost 7 us
// each on 15 to 33 clusters, and a chain of first children was a chain of items.
#pragma once
#include "analysis.cuh"
#include "stream.cuh"
#include "verify.cuh"

namespace specv {

struct NParams {
    VParams v;                // shapes, inputs, records, published weights, arrival counters, outputs
    const RowPart *part;      // [B*N*2] statistics of every row the verifier reads
    double *gseq;             // [B*N][KMAX]: the step coefficients g_j of every branching node
    unsigned int *ticket;     // item counter of the branch kernel (0 at launch)
    // analysis only (SpecInfer mode, every threshold evaluated)
    AnRec *an;                // [B*N] per-node scalars for the branching probabilities
    float *an_acc;            // [B,N,4] acceptance rates: NSS, Naive, SpecTr written here (SpecInfer by spec_branch_kernel)
    float *an_div;            // [B,N,3] L1, KL(p||q), KL(q||p)
};

// A sum of fp32 exponentials, fp64 above a thread's chunk of 8, is off by at most 2^-22 + 3 2^-24 = 4.2e-7 of the mass.  Measured
// against fp64 (V = 6080 to 262144): 2.9e-7 where one token may hold most of it, 8.6e-8 where none holds more than a
// quarter (LIST_FLAT_Z).  A node's weight S / (S + 1 - w) is off by that over S + 1 - w.  So fp32 sums are used on
// flat rows only, and only while S + 1 - w is above this (bound 8.4e-6 in the weight).
constexpr double SMALL_STEP = 0.05;
__device__ __forceinline__ bool flat_rows(double Z_p, double Z_q) { return Z_p > LIST_FLAT_Z && Z_q > LIST_FLAT_Z; }
constexpr int FEW_SEQS = 2048;        // nodes whose child counts a cluster looks at in one go
// sequences that are gone through node by node, window after window (all of them where they share one tree)
__device__ __forceinline__ int window_seqs(const VParams &P)
{
    return P.topo_stride == 0 ? P.B : min(P.B, max(1, FEW_SEQS / P.N));
}

constexpr unsigned long long NO_CHILD = W_PENDING - 1;        // a childless node's ratio
__device__ __forceinline__ double token_ratio(double Pp, double Pq)
{
    return !(Pp > 0.0) ? 0.0 : (!(Pq > 0.0) ? CUDART_INF : Pp / Pq);
}
// Traversal's weight for a child from its parent's state, min(1, w P / q).  A weight within a rounding of 1 is 1: the step after it
// is discontinuous at w = 1 when P = q (S = 0 gives weight 1 for w = 1 and weight 0 for any w < 1).
__device__ __forceinline__ double handed_weight(double w, double ratio)
{
    const double thr = w > 0.0 ? fmin(1.0, w * ratio) : 0.0;
    return thr > 1.0 - WEIGHT_SNAP ? 1.0 : thr;
}

// the statistics of one row, and whether they are usable
struct RowStat {
    double Z;
    int O;
    float cut;
    int bad;
    __device__ __forceinline__ bool ok() const { return bad == 0 && O > ROWPART_EMPTY && Z > 0.0 && Z < CUDART_INF; }
};
__device__ __forceinline__ RowStat load_stat(const RowPart *p)
{
    const double Z = __ldcg(&p->S);
    const int4 r = __ldcg(reinterpret_cast<const int4 *>(p) + 1);       // O, xmax, cut, bad
    return RowStat{Z, r.x, __int_as_float(r.z), r.w};
}
// unnormalised probability of a token in a row, in units of 2^O
__device__ __forceinline__ double token_e(float z, const RowStat &r, double s_d) { return z >= r.cut ? exp2_exact(z, s_d, r.O) : 0.0; }

// The ratio record of a node, written and read in one piece.
__device__ __forceinline__ void put_chain(const VParams &P, long long node, unsigned long long ratio, int child)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(P.chain + node), "l"(ratio),
                 "l"((unsigned long long)(unsigned)child)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 get_chain(const VParams &P, long long node)
{
    ulonglong2 e;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}" : "=l"(e.x), "=l"(e.y) : "l"(P.chain + node) : "memory");
    return e;
}
// Publishes weight thr of node c (warp-collective), and with it the weights of c's line of first children, down to the childless end
// or to a node whose ratio is not known yet (only while the ratio kernel runs): there whoever writes that ratio goes
// on.  Both write before they look (put_ratio), so one of them sees the other; if both do, they write the same weights.
// A line is mostly consecutive nodes, so one load brings 32 ratios.
__device__ __noinline__ void publish_weight(const VParams &P, int b, int c, double thr)
{
    const int lane = threadIdx.x & 31;
    int base = c;
    ulonglong2 e = make_ulonglong2(W_PENDING, 0ull);
    bool have = false;
    for (int hop = 0; hop < P.N; ++hop) {
        const long long at = (long long)b * P.N + c;
        if ((int)at == c_hold_slot) return;               // (a test may ask for one slot to stay pending)
        // (the slot carries all there is to know: nothing to fence for its readers)
        if (lane == 0) *(volatile unsigned long long *)(P.w_pub + at) = (unsigned long long)__double_as_longlong(thr);
        if (!have || c - base > 31) {
            base = c;
            have = true;
            if (c + lane < P.N) e = get_chain(P, at + lane);
        }
        unsigned long long ratio = __shfl_sync(0xffffffffu, e.x, c - base), child = __shfl_sync(0xffffffffu, e.y, c - base);
        if (ratio == W_PENDING) {
            __syncwarp();
            __threadfence();
            const ulonglong2 again = get_chain(P, at);
            ratio = again.x;
            child = again.y;
        }
        ratio = __shfl_sync(0xffffffffu, ratio, 0);       // (one answer for all lanes)
        child = __shfl_sync(0xffffffffu, child, 0);
        if (ratio == W_PENDING || ratio == NO_CHILD) return;
        c = (int)(unsigned)child;
        thr = handed_weight(thr, __longlong_as_double((long long)ratio));
    }
}
// bounded poll of a published weight; W_PENDING when the limit ran out
__device__ __forceinline__ unsigned long long poll_weight(const unsigned long long *slot_, const int *poison)
{
    volatile const unsigned long long *slot = slot_;
    unsigned long long bits = *slot;
    if (bits != W_PENDING) return bits;
    const long long t0 = clock64();
    for (;;) {
        bits = *slot;
        if (bits != W_PENDING || clock64() - t0 > WAIT_CYCLES || *(volatile const int *)poison) break;
        __nanosleep(32);
    }
    return bits;
}

// The record of a childless node, finished by whoever hands it its weight thr (lane 0 of a converged warp writes; the node's
// arrival is counted by the caller).
__device__ __noinline__ void leaf_record(const VParams &P, const RowPart *part, int b, int c, double thr)
{
    if ((threadIdx.x & 31) != 0) return;
    NodeRec &R = P.rec[(long long)b * P.N + c];
    const RowStat p = load_stat(part + ((long long)b * P.N + c) * 2);
    R.O_p = (double)p.O; R.Z_p = p.Z; R.O_q = 0.0; R.Z_q = 0.0;
    R.kappa = p.Z; R.nsteps = 0;
    R.cut_p = p.cut; R.cut_q = -CUDART_INF_F;
    R.next_child = -1;
    R.status = p.ok() ? 0 : SPEC_DEV_NONFINITE;
    R.bonus = -1; R.bonus_margin = 0.f;
    R.w_in = P.mode == MODE_TRAVERSAL ? thr : 1.0;
    R.thr = thr;
}

// ------------------------------------------------------------------------------------------------
// nodes with one child
// ------------------------------------------------------------------------------------------------
// Sums of NT threads (a CTA, or a warp) over their share of a node's two rows, which come through a ring in shared memory:
// every thread copies and reads its own chunks, NS - 1 of them ahead (one chunk ahead in registers, a pass of one CTA over
// V = 128256 took 33 us, nearly all of it the latency of L2).
// Kinds of sums: SUM_STEP o[0] = sum (g e_p - e_q)+ in fp32; SUM_STEP_HEAVY the same and SUM_NORM the rows' normalisers (o[0],
// o[1]) with the tokens above 2^-DOM_S of a row's mass (at most 1024 per row, about 120 on the synthetic logits) in fp64
// and the others in fp32.  Each of those is good to 2^-22 of itself, so their sum to 2.4e-7 of their share of the mass; they are at
// least as many as 1024 times that share and round by themselves, so 2^-22 / 32 = 7e-9 is its usual size.  The heavy ones
// are collected per warp and evaluated 32 at a time.
enum SumKind { SUM_STEP, SUM_STEP_HEAVY, SUM_NORM };
constexpr int DOM_S = 10;
template <int DT> constexpr int NS = DT == SPEC_BF16 ? 4 : 3;                                  // stages of the ring
template <int DT> constexpr int SUMS_RING = NS<DT> * (DT == SPEC_BF16 ? 2 : 4) * 256 * 16;     // bytes of it
// (out of line: its registers would be spilled around every chunk of the loop below)
template <int KIND>
__device__ __noinline__ double2 heavy_terms(float2 z, float cut_p, float cut_q, int O_p, int O_q, double s_d, double g)
{
    const double xp = z.x >= cut_p ? exp2_exact(z.x, s_d, O_p) : 0.0, xq = z.y >= cut_q ? exp2_exact(z.y, s_d, O_q) : 0.0;
    return KIND == SUM_NORM ? make_double2(xp, xq) : make_double2(fmax(fma(g, xp, -xq), 0.0), 0.0);
}
__device__ __forceinline__ void set_sum_rows(NodeRows &nr, const RowStat &p, const RowStat &q, double s_d)
{
    nr.s_d = s_d;
    stream::split_scale(s_d, nr.s_hi, nr.s_lo);
    nr.hq = true;
    nr.cut_p = p.cut; nr.cut_q = q.cut; nr.O_p = p.O; nr.O_q = q.O;
    nr.thrB_p = (float)(p.Z / (double)(1 << DOM_S));
    nr.thrB_q = (float)(q.Z / (double)(1 << DOM_S));
}
template <int DT, int KIND, int NT = 256>
__device__ __noinline__ void node_sums(const Slice &sl, const NodeRows &nr, double g, uint4 *ring, float2 *heavy, double (&o)[2])
{
    constexpr int U = DT == SPEC_BF16 ? 1 : 2;         // 16-byte units of a chunk
    const int tid = threadIdx.x & (NT - 1), lane = tid & 31, nu = sl.nu, V = sl.V;
    constexpr bool HEAVY = KIND != SUM_STEP;
    const bool vec = sl.vec;
    const float s_hi = nr.s_hi, s_lo = nr.s_lo, O_p = (float)nr.O_p, O_q = (float)nr.O_q, cut_p = nr.cut_p, cut_q = nr.cut_q;
    const float thr_p = nr.thrB_p, thr_q = nr.thrB_q;
    float g_hi, g_lo, dsx = 0.f;
    split_float(g, g_hi, g_lo);
    double o0 = 0.0, o1 = 0.0;
    int n = 0;                             // entries of the warp's list (below 32 between chunks)
    ring += tid;
    auto issue = [&](int c) {
        const int i = c * NT + tid;
        if (vec && i < nu) {
            const size_t u = (size_t)(sl.u0 + i) * U;
            const uint4 *p = reinterpret_cast<const uint4 *>(sl.p) + u, *q = reinterpret_cast<const uint4 *>(sl.q) + u;
            const uint32_t dst = smem_u32(ring + (c % NS<DT>) * 2 * U * NT);
            stream::cp_async16(dst, p, 16);
            stream::cp_async16(dst + U * NT * 16, q, 16);
            if (U == 2 && (sl.u0 + i) * 8 - sl.h + 4 < V) {
                stream::cp_async16(dst + NT * 16, p + 1, 16);
                stream::cp_async16(dst + 3 * NT * 16, q + 1, 16);
            }
        }
        stream::cp_async_commit();
    };
#pragma unroll 1
    for (int c = 0; c < NS<DT> - 1; ++c) issue(c);
#pragma unroll 1
    for (int c = 0; c * NT < nu; ++c) {
        const int i = c * NT + tid, t0 = (sl.u0 + i) * 8 - sl.h, lo = -t0, hi = i < nu ? V - t0 : 0;
        RawChunk<DT> rp, rq;
        stream::cp_async_wait<NS<DT> - 2>();
        const uint4 *st = ring + (c % NS<DT>) * 2 * U * NT;
        rp.a = st[0];
        rq.a = st[U * NT];
        if (U == 2) { rp.b = st[NT]; rq.b = st[3 * NT]; }
        if (!vec && i < nu) {
            rp = load_raw_scalar<DT>(sl.p, sl.u0 + i, V);
            rq = load_raw_scalar<DT>(sl.q, sl.u0 + i, V);
        }
        issue(c + NS<DT> - 1);             // into the stage read in the previous iteration
        float z[8], ep[8], eq[8];
        unpack_chunk<DT>(rp, z);
        mask_chunk(z, lo, hi, cut_p > -CUDART_INF_F, cut_p);
        exp_chunk<false>(z, s_hi, s_lo, O_p, ep, dsx);
        unpack_chunk<DT>(rq, z);
        mask_chunk(z, lo, hi, cut_q > -CUDART_INF_F, cut_q);
        exp_chunk<false>(z, s_hi, s_lo, O_q, eq, dsx);
        if (HEAVY) {
            unsigned m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (ep[k] > thr_p || eq[k] > thr_q) { m |= 1u << k; ep[k] = eq[k] = 0.f; }
            for (;;) {
                const unsigned bal = __ballot_sync(0xffffffffu, m != 0);
                if (!bal) break;
                if (m) {
                    const int k = __ffs(m) - 1;           // (inside the row: the others' e are 0)
                    heavy[n + __popc(bal & ((1u << lane) - 1u))] = make_float2(raw_logit<DT>(rp, k), raw_logit<DT>(rq, k));
                    m &= m - 1u;
                }
                n += __popc(bal);
                __syncwarp();
                if (n >= 32) {
                    n -= 32;
                    const double2 x = heavy_terms<KIND>(heavy[n + lane], cut_p, cut_q, nr.O_p, nr.O_q, nr.s_d, g);
                    o0 += x.x;
                    o1 += x.y;
                    __syncwarp();
                }
            }
        }
        // (a thread's sums over its chunks in fp64: in fp32 each of up to hundreds of additions would round)
        if (KIND == SUM_NORM) { o0 += (double)sum_chunk(ep); o1 += (double)sum_chunk(eq); }
        else o0 += (double)step_chunk(ep, eq, g_hi, g_lo);
    }
    stream::cp_async_wait<0>();
    if (HEAVY && lane < n) {
        const double2 x = heavy_terms<KIND>(heavy[lane], cut_p, cut_q, nr.O_p, nr.O_q, nr.s_d, g);
        o0 += x.x;
        o1 += x.y;
    }
    __syncwarp();
    o[0] = o0;
    o[1] = o1;
}

// What a node hands its first child depends on: that child, its logits in the node's rows, and whether anything is wrong with
// the node's own arguments (what spec_single_kernel and spec_recursion_kernel look at too).  Warp-collective.
struct __align__(16) FirstChild {
    int child;
    unsigned short kc, err;
    float zp, zq;
};
template <int DT>
__device__ __noinline__ FirstChild first_child(const VParams &P, int b, int a)
{
    const int lane = threadIdx.x & 31;
    const int *parent = P.parent + (long long)b * P.topo_stride, *token = P.token + (long long)b * P.N;
    FirstChild f = {0, 0, 0, 0.f, 0.f};
    for (int c0 = a + 1; c0 < P.N; c0 += 32) {
        const int c = c0 + lane;
        const bool is = c < P.N && __ldg(parent + c) == a;
        const unsigned bal = __ballot_sync(0xffffffffu, is);
        if (bal && !f.kc) f.child = c0 + __ffs(bal) - 1;
        f.kc += __popc(bal);
        if (is) { const int x = __ldg(token + c); f.err |= x < 0 || x >= P.V; }
    }
    if (!f.kc) return f;
    const int pa = __ldg(parent + a), xa = __ldg(token + a), x = __ldg(token + f.child);
    f.err |= f.kc > KMAX || (a == 0 ? pa != -1 : (pa < 0 || pa >= a || xa < 0 || xa >= P.V));
    f.err = __any_sync(0xffffffffu, f.err);
    if (!f.err) {
        const long long at = (long long)b * P.seq_stride + (long long)a * P.node_stride + x;
        f.zp = load_logit(P.zp, DT, at);
        f.zq = load_logit(P.zq, DT, at);
    }
    return f;
}

// A node's ratio is known (in lane 0; warp-collective): written down, and the line below the node published if the node's weight has
// been (the root's is 1, that of a node without a parent to hand it one is 0).
__device__ __noinline__ void put_ratio(const VParams &P, int b, int a, double ratio, int child)
{
    const long long node = (long long)b * P.N + a;
    ratio = __shfl_sync(0xffffffffu, ratio, 0);
    unsigned long long bits = (unsigned long long)__double_as_longlong(1.0);
    if ((threadIdx.x & 31) == 0) {
        put_chain(P, node, (unsigned long long)__double_as_longlong(ratio), child);
        __threadfence();
        const int pa = a == 0 ? 0 : __ldg(P.parent + (long long)b * P.topo_stride + a);
        if (a > 0) bits = pa < 0 || pa >= a ? 0ull : *(volatile unsigned long long *)(P.w_pub + node);
    }
    bits = __shfl_sync(0xffffffffu, bits, 0);
    if (bits != W_PENDING) publish_weight(P, b, child, handed_weight(__longlong_as_double((long long)bits), ratio));
}

// Traversal: the ratio of every first child, and the line of first children below each root, so that the kernels below ask for no
// weight that a kernel after them would have to hand on.  A node with a fault of any kind hands on 0 and reports it itself.
//   flat rows    two logits over the normalisers of the statistics pass, a warp per node (from the last CTA on, so that the
//                first ones are free for the others);
//   peaked rows  (flat_rows) both rows are summed again, heavy tokens in fp64.
//     few    every CTA makes the same list of these nodes from the statistics, and as many CTAs take one as there are for each
//            (up to SPLIT_MAX).  They and the node's warp leave what they have in the node's record, unused until the
//            node's ratio is known, and the last of them writes the ratio;
//     many   the node's warp does it by itself (many: see there).
//   A node with one child keeps the exact normalisers in its record.
// Bound by latency: what the call was given is read while the statistics kernel's last rows are on their way, a warp's ratio
// is then one round of loads, one store and one look at the node's weight; a peaked node at V = 128256 on 5 CTAs is 13
// rounds of its ring (9 us, 2.5 before it for the list and 2 after it).
struct __align__(16) PeakedNode {
    static constexpr int MOST = 5;
    double2 part[MOST];          // the rows' sums of each CTA
    FirstChild f;
};
static_assert(sizeof(PeakedNode) <= sizeof(NodeRec), "a node's record holds its partial sums");
constexpr int SPLIT_MAX = PeakedNode::MOST;
constexpr int PEAKED_LIST = 4096;                    // nodes that every CTA goes through (beyond: many)

// One of the C + 1 who contribute to a peaked node has written its part (lane 0 of a converged warp): the last one writes the
// ratio.
__device__ __noinline__ void arrive_peaked(const VParams &P, const RowPart *part, long long node, int C)
{
    const int lane = threadIdx.x & 31;
    int prev = 0;
    if (lane == 0) asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(prev) : "l"(&P.chain[node].parts) : "memory");
    if (__shfl_sync(0xffffffffu, prev, 0) != C) return;
    const int b = (int)(node / P.N);
    double ratio = 0.0;
    int child = 0;
    if (lane == 0) {
        PeakedNode *R = reinterpret_cast<PeakedNode *>(P.rec + node);
        double Z_p = 0.0, Z_q = 0.0;
        double2 x[SPLIT_MAX];
#pragma unroll
        for (int k = 0; k < SPLIT_MAX; ++k) x[k] = k < C ? __ldcg(R->part + k) : make_double2(0.0, 0.0);
        const uint4 f4 = __ldcg(reinterpret_cast<const uint4 *>(&R->f));
        const RowStat p = load_stat(part + node * 2), q = load_stat(part + node * 2 + 1);
#pragma unroll
        for (int k = 0; k < SPLIT_MAX; ++k) { Z_p += x[k].x; Z_q += x[k].y; }
        const double s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
        const int kc = (int)(f4.y & 0xFFFFu), err = (int)(f4.y >> 16);
        const double e_p = token_e(__uint_as_float(f4.z), p, s_d), e_q = token_e(__uint_as_float(f4.w), q, s_d);
        if (kc == 1) { __stcg(&P.rec[node].Z_p, Z_p); __stcg(&P.rec[node].Z_q, Z_q); __threadfence(); }
        if (!err) ratio = token_ratio(e_p / Z_p, e_q / Z_q);
        child = (int)f4.x;
    }
    put_ratio(P, b, (int)(node % P.N), ratio, __shfl_sync(0xffffffffu, child, 0));
}

template <int DT>
__global__ void __launch_bounds__(256, 3) spec_ratio_kernel(const NParams NP)
{
    constexpr int NW = 8;
    const VParams &P = NP.v;
    __shared__ float2 s_heavy[NW][64];
    __shared__ double s_sum[NW][2];
    __shared__ int s_cnt[NW];
    __shared__ unsigned short s_list[PEAKED_LIST];
    uint4 *ring = reinterpret_cast<uint4 *>(dyn_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ctas = (int)gridDim.x;
    const long long nodes = (long long)P.B * P.N, step = (long long)ctas * NW;
    const auto scale = [&](int b) { return 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T); };
    const auto peaked_node = [&](long long node) {
        // (a childless node's draft row has not been read: not ok)
        const RowStat p = load_stat(NP.part + node * 2), q = load_stat(NP.part + node * 2 + 1);
        return p.ok() && q.ok() && !flat_rows(p.Z, q.Z);
    };

    long long id = (long long)(ctas - 1 - (int)blockIdx.x) * NW + warp;
    FirstChild f = {};
    if (id < nodes) f = first_child<DT>(P, (int)(id / P.N), (int)(id % P.N));
    grid_dependency_wait();
    grid_launch_dependents();     // (from here on: the recursion finds the statistics complete)

    // ---- the list of peaked nodes -----------------------------------------------------------------------------------------
    int n = 0, C = 1;
    bool many = nodes > PEAKED_LIST;
    if (!many) {
        for (int i0 = 0; i0 < (int)nodes; i0 += 256) {
            const int i = i0 + tid;
            const bool peaked = i < (int)nodes && peaked_node(i);
            const unsigned bal = __ballot_sync(0xffffffffu, peaked);
            __syncthreads();
            if (lane == 0) s_cnt[warp] = __popc(bal);
            __syncthreads();
            int at = n;
#pragma unroll
            for (int w = 0; w < NW; ++w) { if (w < warp) at += s_cnt[w]; n += s_cnt[w]; }
            if (peaked) s_list[at + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)i;
        }
        __syncthreads();
        // A node costs about as much as 30 rounds of a CTA's ring besides its rows: loads that wait for each other, a barrier, the
        // handing over.  A warp takes eight times the rounds and overlaps seven others.
        const int rounds = (P.V + 2047) >> 11;
        many = (n + ctas - 1) / ctas * (30 + rounds) > (n + ctas * NW - 1) / (ctas * NW) * (30 + NW * rounds);
    }
    if (!many) {
        C = max(1, min(min(SPLIT_MAX, ctas / max(n, 1)), P.V >> 12));        // (a part of a row is at least 4096 logits)
        for (int it = (int)blockIdx.x; it < n * C; it += ctas) {
            const long long node = s_list[it / C];
            const int r = it % C, b = (int)(node / P.N), a = (int)(node % P.N);
            const RowStat p = load_stat(NP.part + node * 2), q = load_stat(NP.part + node * 2 + 1);
            NodeRows nr;
            set_sum_rows(nr, p, q, scale(b));
            const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, (unsigned)r);
            double v[2];
            node_sums<DT, SUM_NORM>(sl, nr, 0.0, ring, s_heavy[warp], v);
            v[0] = warp_sum(v[0]);
            v[1] = warp_sum(v[1]);
            if (lane == 0) { s_sum[warp][0] = v[0]; s_sum[warp][1] = v[1]; }
            __syncthreads();
            if (warp == 0) {
                double2 z = make_double2(0.0, 0.0);
                for (int w = 0; w < NW; ++w) { z.x += s_sum[w][0]; z.y += s_sum[w][1]; }
                if (lane == 0) __stcg(reinterpret_cast<PeakedNode *>(P.rec + node)->part + r, z);
                arrive_peaked(P, NP.part, node, C);
            }
            __syncthreads();
        }
    }

    // ---- a warp per node ------------------------------------------------------------------------------------------------
    while (id < nodes) {
        const int b = (int)(id / P.N);
        if (f.kc && !many && peaked_node(id)) {
            if (lane == 0)
                __stcg(reinterpret_cast<uint4 *>(&reinterpret_cast<PeakedNode *>(P.rec + id)->f),
                       make_uint4((unsigned)f.child, (unsigned)f.kc | (unsigned)f.err << 16, __float_as_uint(f.zp), __float_as_uint(f.zq)));
            arrive_peaked(P, NP.part, id, C);
        } else if (f.kc) {
            const int a = (int)(id % P.N);
            const RowStat p = load_stat(NP.part + id * 2), q = load_stat(NP.part + id * 2 + 1);
            const double s_d = scale(b);
            double ratio = 0.0;
            if (!f.err && p.ok() && q.ok()) {
                double Z_p = p.Z, Z_q = q.Z;
                if (!flat_rows(Z_p, Z_q)) {
                    NodeRows nr;
                    set_sum_rows(nr, p, q, s_d);
                    const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, 1, 0u);
                    double v[2];
                    node_sums<DT, SUM_NORM, 32>(sl, nr, 0.0, ring + warp * (SUMS_RING<DT> / (16 * NW)), s_heavy[warp], v);
                    Z_p = warp_sum(v[0]);
                    Z_q = warp_sum(v[1]);
                    if (f.kc == 1 && lane == 0) { __stcg(&P.rec[id].Z_p, Z_p); __stcg(&P.rec[id].Z_q, Z_q); __threadfence(); }
                }
                ratio = token_ratio(token_e(f.zp, p, s_d) / Z_p, token_e(f.zq, q, s_d) / Z_q);
            }
            put_ratio(P, b, a, ratio, f.child);
        } else if (lane == 0) {
            put_chain(P, id, NO_CHILD, 0);
        }
        id += step;
        if (id < nodes) f = first_child<DT>(P, (int)(id / P.N), (int)(id % P.N));
    }
}

// One cluster of P.C CTAs (one where the batch fills the chip) per node, node-major; nodes of other kinds leave at once, except
// those nobody else finishes: a tree of one node, and a childless node whose parent index is no parent.  Bound by the
// special-function unit (two exponentials per token and row pair) once it runs, by the poll for its weight before.
template <int DT>
__global__ void __launch_bounds__(256, 3) spec_single_kernel(const NParams NP)
{
    constexpr int NW = 8;
    const VParams &P = NP.v;
    __shared__ Common M;
    __shared__ int s_first, s_count, s_nonleaf;
    __shared__ unsigned long long s_w;
    uint4 *ring = reinterpret_cast<uint4 *>(dyn_smem);
    __shared__ float2 s_heavy[NW][64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, C = P.C;
    const unsigned rank = C > 1 ? cluster_ctarank() : 0u;
    // the same order as the items of spec_recursion_kernel: windows of sequences, node by node
    const int id = (int)(blockIdx.x / (unsigned)C), G = window_seqs(P), b0 = id / (G * P.N) * G, in_w = id - b0 * P.N;
    const int Gw = min(G, P.B - b0), a = in_w / Gw, b = b0 + in_w % Gw;
    const int *parent = P.parent + (long long)b * P.topo_stride;
    const int *token = P.token + (long long)b * P.N;
    const bool trav = P.mode == MODE_TRAVERSAL;
    grid_launch_dependents();
    if (tid == 0) { s_first = P.N; s_count = 0; s_nonleaf = 0; }
    __syncthreads();
    for (int c = a + 1 + tid; c < P.N; c += 256)
        if (__ldg(parent + c) == a) { atomicMin(&s_first, c); atomicAdd(&s_count, 1); }
    __syncthreads();
    const int kc = s_count, c = s_first, pa = __ldg(parent + a);
    const bool orphan = a == 0 ? pa != -1 : (pa < 0 || pa >= a);
    if (kc == 1 || (kc == 0 && (a == 0 || orphan))) {
        int err = orphan ? SPEC_DEV_TOPOLOGY : 0;
        if (a > 0) { const int x = __ldg(token + a); if (x < 0 || x >= P.V) err = max(err, SPEC_DEV_TOKEN); }
        const RowPart *rp = NP.part + ((long long)b * P.N + a) * 2;
        const RowStat p = load_stat(rp), q = kc ? load_stat(rp + 1) : p;
        if (kc) for (int d = c + 1 + tid; d < P.N; d += 256) if (__ldg(parent + d) == c) s_nonleaf = 1;
        NodeRows nr;
        set_sum_rows(nr, p, q, 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T));
        double e_p = 0.0, e_q = 0.0;
        if (kc) {
            const int x = __ldg(token + c);
            if (x < 0 || x >= P.V) err = max(err, SPEC_DEV_TOKEN);
            else {
                const long long at = (long long)b * P.seq_stride + (long long)a * P.node_stride + x;
                const float zp = load_logit(P.zp, DT, at), zq = load_logit(P.zq, DT, at);
                e_p = token_e(zp, p, nr.s_d);
                e_q = token_e(zq, q, nr.s_d);
            }
        }
        if (!err && (!p.ok() || !q.ok())) err = SPEC_DEV_NONFINITE;
        if (tid == 0) { common_init(M, NW); mbar_fence_init(); }
        __syncthreads();
        if (C > 1) cluster_sync_all();
        Team T = {M, C, warp, lane, 0, rank, 0u};
        const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
        double Z_p = p.Z, Z_q = q.Z;
        if (trav && kc && p.ok() && q.ok() && !flat_rows(Z_p, Z_q)) {
            // left in the record by the ratio kernel, with its ratio (a faulty node waits as well: partial sums may be there)
            const long long node = (long long)b * P.N + a;
            if (tid == 0) s_w = poll_weight(&P.chain[node].ratio, &M.poison);
            __syncthreads();
            if (s_w == W_PENDING) err = SPEC_DEV_TIMEOUT;
            __threadfence();
            Z_p = __ldcg(&P.rec[node].Z_p);
            Z_q = __ldcg(&P.rec[node].Z_q);
            __syncthreads();
        }
        const double ratio = token_ratio(e_p / Z_p, e_q / Z_q);
        if (tid == 0) {
            s_w = (trav && a > 0 && !err) ? poll_weight(P.w_pub + (long long)b * P.N + a, &M.poison) : (unsigned long long)__double_as_longlong(1.0);
        }
        __syncthreads();
        double w = __longlong_as_double((long long)s_w);
        if (s_w == W_PENDING || err == SPEC_DEV_TIMEOUT) { err = SPEC_DEV_TIMEOUT; M.poison = 1; }
        if (err) w = 0.0;
        const double thr = err ? 0.0 : (trav ? handed_weight(w, ratio) : fmin(1.0, ratio));
        // (the child's weight has been published with this node's; after a wait that ran out, those below need not wait as well)
        if (err == SPEC_DEV_TIMEOUT && kc && s_nonleaf && rank == 0 && warp == 0) publish_weight(P, b, c, 0.0);
        double w_fin = w;
        if (trav && kc && w > 0.0) {
            double tot[1], mine[1];
            double Sm = 0.0;
            bool careful = !flat_rows(p.Z, q.Z);
            if (!careful) {
                double v[2];
                node_sums<DT, SUM_STEP>(sl, nr, w * Z_q / Z_p, ring, s_heavy[warp], v);
                const double v1[1] = {v[0]};
                cluster_sum<NW, 1>(T, v1, tot, mine);
                Sm = tot[0] / Z_q;
                if (!(Sm + (1.0 - w) > SMALL_STEP)) {
                    double t2[2], m2[2];
                    careful = true;
                    node_sums<DT, SUM_NORM>(sl, nr, 0.0, ring, s_heavy[warp], v);
                    cluster_sum<NW, 2>(T, v, t2, m2);
                    Z_p = t2[0]; Z_q = t2[1];
                }
            }
            if (careful) {
                double v[2];
                node_sums<DT, SUM_STEP_HEAVY>(sl, nr, w * Z_q / Z_p, ring, s_heavy[warp], v);
                const double v1[1] = {v[0]};
                cluster_sum<NW, 1>(T, v1, tot, mine);
                Sm = tot[0] / Z_q;
                if (!(Sm > RESIDUAL_FLOOR * w)) Sm = 0.0;         // P = q, and what is left is the rounding of g
            }
            if (*(volatile int *)&M.poison) err = SPEC_DEV_TIMEOUT;
            // S = 0 at weight 1: the state equals q and the weight stays; at a weight below 1 it drops to 0
            w_fin = w < 1.0 ? Sm / (Sm + (1.0 - w)) : 1.0;
        }
        if (err) w_fin = 0.0;
        if (rank == 0 && warp == 0) {
            // (in the order that keeps the atomic's wait short: nothing but the record's own stores before it)
            NodeRec *rec = P.rec + (long long)b * P.N;
            unsigned narr = 1u;
            if (kc) {
                if (!s_nonleaf) { leaf_record(P, NP.part, b, c, thr); ++narr; }
                else if (!trav && lane == 0) rec[c].thr = thr;
            }
            if (lane == 0) {
                NodeRec &R = rec[a];
                R.O_p = (double)p.O; R.Z_p = p.Z; R.O_q = (double)q.O; R.Z_q = kc ? q.Z : 0.0;
                R.kappa = p.Z;
                R.nsteps = kc && w > 0.0 ? STATE_FIRST : 0;
                R.cut_p = p.cut; R.cut_q = kc ? q.cut : -CUDART_INF_F;
                R.next_child = kc && !trav && !err && (double)__ldg(P.u_accept + (long long)b * P.N + c) < thr ? c : -1;
                R.status = err;
                R.bonus = -1; R.bonus_margin = 0.f;
                R.w_in = trav && a > 0 ? w : 1.0;
                if (trav) R.thr = a == 0 ? 1.0 : w_fin;
                else if (a == 0) R.thr = 1.0;
            }
            __syncwarp();
            arrive_sequence(P, b, narr);
        }
        if (C > 1) cluster_sync_all();         // nobody leaves while a peer may still write to its shared memory
    }
    if (blockIdx.x == 0) grid_dependency_wait();      // this kernel ends only after the one before it
}

// ---- the analysis of nodes with one child -----------------------------------------------------------------------------------
// Everything Algorithms 6-9 and the divergences ask of such a node are sums over its two rows (SpecTr's division factor is 1, its
// beta and acceptance are sum min(p, q)): two passes of the ring, nothing resident.  Tokens above 2^-DOM_S of a row's mass in fp64,
// the others in fp32, fp64 above a chunk.
// NORM: o = Z_p, Z_q and the cross sums of KlSums (pp, pq, qq, qp); else |p - q|, min(p, q), p min(q, 1) and (p - q)+.
struct AnTerms {
    double o[6];
};
template <bool NORM>
__device__ __noinline__ AnTerms an_heavy(float2 z, float cut_p, float cut_q, int O_p, int O_q, double s_d, double ip, double iq)
{
    AnTerms t = {};
    const double ep = z.x >= cut_p ? exp2_exact(z.x, s_d, O_p) : 0.0, eq = z.y >= cut_q ? exp2_exact(z.y, s_d, O_q) : 0.0;
    if (NORM) {
        const double xp = z.x >= cut_p ? (double)z.x * s_d - (double)O_p : -CUDART_INF, xq = z.y >= cut_q ? (double)z.y * s_d - (double)O_q : -CUDART_INF;
        t.o[0] = ep; t.o[1] = eq;
        if (ep > 0.0) { t.o[2] = ep * xp; t.o[3] = ep * xq; }
        if (eq > 0.0) { t.o[4] = eq * xq; t.o[5] = eq * xp; }
    } else {
        const double p = ep * ip, q = eq * iq;
        t.o[0] = fabs(p - q); t.o[1] = fmin(p, q); t.o[2] = p * fmin(q, 1.0); t.o[3] = fmax(p - q, 0.0);
    }
    return t;
}
template <int DT, bool NORM>
__device__ __noinline__ AnTerms an_sums(const Slice sl, const NodeRows nr, double ip, double iq, uint4 *ring, float2 *heavy)
{
    constexpr int U = DT == SPEC_BF16 ? 1 : 2, NT = 256, NO = NORM ? 6 : 4;
    const int tid = threadIdx.x, lane = tid & 31;
    const float s_hi = nr.s_hi, s_lo = nr.s_lo, O_p = (float)nr.O_p, O_q = (float)nr.O_q, ipf = (float)ip, iqf = (float)iq;
    AnTerms sum = {};
    int n = 0;                             // entries of the warp's list (below 32 between chunks)
    ring += tid;
    const auto take = [&](int at, bool on) {
        const AnTerms t = an_heavy<NORM>(on ? heavy[at] : make_float2(-CUDART_INF_F, -CUDART_INF_F), nr.cut_p, nr.cut_q, nr.O_p, nr.O_q, nr.s_d, ip, iq);
#pragma unroll
        for (int i = 0; i < NO; ++i) sum.o[i] += on ? t.o[i] : 0.0;
    };
    auto issue = [&](int c) {
        const int i = c * NT + tid;
        if (sl.vec && i < sl.nu) {
            const size_t u = (size_t)(sl.u0 + i) * U;
            const uint4 *p = reinterpret_cast<const uint4 *>(sl.p) + u, *q = reinterpret_cast<const uint4 *>(sl.q) + u;
            const uint32_t dst = smem_u32(ring + (c % NS<DT>) * 2 * U * NT);
            stream::cp_async16(dst, p, 16);
            stream::cp_async16(dst + U * NT * 16, q, 16);
            if (U == 2 && (sl.u0 + i) * 8 - sl.h + 4 < sl.V) {
                stream::cp_async16(dst + NT * 16, p + 1, 16);
                stream::cp_async16(dst + 3 * NT * 16, q + 1, 16);
            }
        }
        stream::cp_async_commit();
    };
#pragma unroll 1
    for (int c = 0; c < NS<DT> - 1; ++c) issue(c);
#pragma unroll 1
    for (int c = 0; c * NT < sl.nu; ++c) {
        const int i = c * NT + tid, t0 = (sl.u0 + i) * 8 - sl.h, lo = -t0, hi = i < sl.nu ? sl.V - t0 : 0;
        RawChunk<DT> rp, rq;
        stream::cp_async_wait<NS<DT> - 2>();
        const uint4 *st = ring + (c % NS<DT>) * 2 * U * NT;
        rp.a = st[0];
        rq.a = st[U * NT];
        if (U == 2) { rp.b = st[NT]; rq.b = st[3 * NT]; }
        if (!sl.vec && i < sl.nu) {
            rp = load_raw_scalar<DT>(sl.p, sl.u0 + i, sl.V);
            rq = load_raw_scalar<DT>(sl.q, sl.u0 + i, sl.V);
        }
        issue(c + NS<DT> - 1);             // into the stage read in the previous iteration
        float xp[8], xq[8], ep[8], eq[8];
        unpack_chunk<DT>(rp, xp);
        mask_chunk(xp, lo, hi, nr.cut_p > -CUDART_INF_F, nr.cut_p);
        unpack_chunk<DT>(rq, xq);
        mask_chunk(xq, lo, hi, nr.cut_q > -CUDART_INF_F, nr.cut_q);
        unsigned m = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            xp[k] = fmaf(xp[k], s_lo, fmaf(xp[k], s_hi, -O_p));
            xq[k] = fmaf(xq[k], s_lo, fmaf(xq[k], s_hi, -O_q));
            ep[k] = ex2_approx(xp[k]);
            eq[k] = ex2_approx(xq[k]);
            if (ep[k] > nr.thrB_p || eq[k] > nr.thrB_q) { m |= 1u << k; ep[k] = eq[k] = 0.f; }
        }
        for (;;) {
            const unsigned bal = __ballot_sync(0xffffffffu, m != 0);
            if (!bal) break;
            if (m) {
                const int k = __ffs(m) - 1;           // (inside the row: the others' e are 0)
                heavy[n + __popc(bal & ((1u << lane) - 1u))] = make_float2(raw_logit<DT>(rp, k), raw_logit<DT>(rq, k));
                m &= m - 1u;
            }
            n += __popc(bal);
            __syncwarp();
            if (n >= 32) {
                n -= 32;
                take(n + lane, true);
                __syncwarp();
            }
        }
        float a[NO];
#pragma unroll
        for (int i2 = 0; i2 < NO; ++i2) a[i2] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (NORM) {
                a[0] += ep[k];
                a[1] += eq[k];
                if (ep[k] > 0.f) { a[2] = fmaf(ep[k], xp[k], a[2]); a[3] = fmaf(ep[k], xq[k], a[3]); }
                if (eq[k] > 0.f) { a[NO - 2] = fmaf(eq[k], xq[k], a[NO - 2]); a[NO - 1] = fmaf(eq[k], xp[k], a[NO - 1]); }
            } else {
                const float p = ep[k] * ipf, q = eq[k] * iqf, d = p - q;
                a[0] += fabsf(d);
                a[1] += fminf(p, q);
                a[2] = fmaf(p, fminf(q, 1.f), a[2]);
                a[3] += fmaxf(d, 0.f);
            }
        }
#pragma unroll
        for (int i2 = 0; i2 < NO; ++i2) sum.o[i2] += (double)a[i2];
    }
    stream::cp_async_wait<0>();
    if (n > 0) take(lane, lane < n);
    __syncwarp();
    return sum;
}

// A cluster of P.C CTAs per node, as spec_single_kernel; nodes of other kinds leave at once.  As items of the recursion kernel, rows
// resident, 112 such nodes at V = 128256 were 7 rounds of 26 us on its clusters; here a call takes 153 us in place of 260 (with
// two CTAs per SM, and no spills, 162).
template <int DT>
__global__ void __launch_bounds__(256, 3) spec_single_analysis_kernel(const NParams NP)
{
    constexpr int NW = 8;
    const VParams &P = NP.v;
    __shared__ Common M;
    __shared__ float2 s_heavy[NW][64];
    __shared__ FirstChild s_f;
    uint4 *ring = reinterpret_cast<uint4 *>(dyn_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, C = P.C;
    const unsigned rank = C > 1 ? cluster_ctarank() : 0u;
    const int id = (int)(blockIdx.x / (unsigned)C), b = id / P.N, a = id % P.N;
    const long long node = id;
    grid_launch_dependents();
    if (warp == 0) {
        const FirstChild f = first_child<DT>(P, b, a);
        if (lane == 0) s_f = f;
    }
    if (tid == 0) { common_init(M, NW); mbar_fence_init(); }
    __syncthreads();
    const FirstChild f = s_f;
    const RowStat p = load_stat(NP.part + node * 2), q = load_stat(NP.part + node * 2 + 1);
    // (what is wrong with a node is wrong for all CTAs of its cluster; its outputs stay NaN)
    if (f.kc == 1 && !f.err && p.ok() && q.ok()) {
        if (C > 1) cluster_sync_all();
        Team T = {M, C, warp, lane, 0, rank, 0u};
        NodeRows nr;
        set_sum_rows(nr, p, q, 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T));
        const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
        double v[6], t[6], mine[6];
        AnTerms o = an_sums<DT, true>(sl, nr, 0.0, 0.0, ring, s_heavy[warp]);
#pragma unroll
        for (int i = 0; i < 6; ++i) v[i] = o.o[i];
        cluster_sum<NW, 6>(T, v, t, mine);
        const double Z_p = t[0], Z_q = t[1];
        if (Z_p > 0.0 && Z_q > 0.0) {
            const double ip = 1.0 / Z_p, iq = 1.0 / Z_q;
            o = an_sums<DT, false>(sl, nr, ip, iq, ring, s_heavy[warp]);
            double v4[4], t4[4], m4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v4[i] = o.o[i];
            cluster_sum<NW, 4>(T, v4, t4, m4);
            if (rank == 0 && tid == 0 && !*(volatile int *)&M.poison) {
                const double l1 = t4[0], smin = t4[1], nss = t4[2], spos = t4[3];
                // KL(p||q) = ln 2 (sum e_p x_p - sum e_p x_q) / Z_p - ln Z_p + ln Z_q, and the mirror image
                const double lz = log(Z_p) - log(Z_q);
                float *ao = NP.an_acc + node * 4, *dv = NP.an_div + node * 3;
                ao[0] = (float)nss; ao[1] = (float)smin; ao[2] = (float)smin;
                dv[0] = (float)l1;
                dv[1] = (float)(0.6931471805599453 * (t[2] - t[3]) * ip - lz);
                dv[2] = (float)(0.6931471805599453 * (t[4] - t[5]) * iq + lz);
                const double px = token_e(f.zp, p, nr.s_d) * ip, qx = token_e(f.zq, q, nr.s_d) * iq;
                const double S = spos > RESIDUAL_FLOOR ? spos : 0.0;
                AnRec &A = NP.an[node];
                A.A[0][0] = fmin(1.0, token_ratio(px, qx));
                A.A[1][0] = S > 0.0 ? fmax(px - qx, 0.0) / S : qx;            // p_1(x); S = 0: the state equals q
                A.S[0] = S;
                A.px[0] = px; A.qx[0] = qx;
                A.rho = 1.0; A.beta = smin; A.pacc = smin; A.s_res = spos;
                A.k = 1; A.valid = 1;
            }
        }
        if (C > 1) cluster_sync_all();         // nobody leaves while a peer may still write to its shared memory
    }
    if (blockIdx.x == 0) grid_dependency_wait();      // this kernel ends only after the one before it
}

// ------------------------------------------------------------------------------------------------
// nodes with several children
// ------------------------------------------------------------------------------------------------
// what the consumers need to know about a node besides its rows
struct __align__(16) NodeScalars {
    double cpm[KMAX], cqm[KMAX];   // exact 2^(z s - O) of the children's tokens in the node's target and draft rows
    float cu[KMAX];                // the children's acceptance uniforms
    int child[KMAX];
    double Z_p, Z_q;
    int kc, a, b, more, O_p, O_q;
    float cut_p, cut_q;
    unsigned leaf_mask;            // bit j: child j has no children
};
// the node's outcome, for the warp that writes it down
struct __align__(16) Outcome {
    double thr[KMAX];              // what child j is handed
    double w_in, w_fin, kappa, Z_p, Z_q;
    int nsteps, acc, err;
};
struct __align__(16) BHdr {
    Common M;
    uint64_t sfull[2], sempty[2], tbar[2], abar[2], mb[2][KMAX], mend[2];
    unsigned long long item[2];    // ticket | (weight already 0) << 32, written by the first CTA's helper
    NodeScalars sc[2];             // by parity of the item
    Outcome out[2];
    int cnt[FEW_SEQS];             // children per node
    unsigned short list[FEW_SEQS]; // the nodes that are items
};

__device__ __forceinline__ void st_async_u64(unsigned long long *slot, uint64_t *bar, uint32_t rank, unsigned long long v)
{
    asm volatile(
        "{\n\t.reg .b32 ra, rb;\n\tmapa.shared::cluster.u32 ra, %0, %2;\n\tmapa.shared::cluster.u32 rb, %1, %2;\n\t"
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [ra], %3, [rb];\n\t}" ::"r"(smem_u32(slot)),
        "r"(smem_u32(bar)), "r"(rank), "l"(v)
        : "memory");
}
// one arrival on the mbarrier at the same offset in CTA `rank` of the cluster
__device__ __forceinline__ void mbar_arrive_remote(uint64_t *bar, uint32_t rank)
{
    asm volatile(
        "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t}" ::"r"(smem_u32(bar)), "r"(rank)
        : "memory");
}

// The nodes with at least `least` children among sequences b0 .. b0 + G - 1, node-major (one tree: G = 1 stands for all).  By one
// warp; returns their number.
__device__ __noinline__ int list_nodes(BHdr &S, const VParams &P, int b0, int G, int least)
{
    const int lane = threadIdx.x & 31, n = G * P.N;
    for (int i = lane; i < n; i += 32) S.cnt[i] = 0;
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
        const int g = i / P.N, a = i % P.N;
        const int pa = __ldg(P.parent + (long long)(b0 + g) * P.topo_stride + a);
        if (pa >= 0 && pa < P.N && pa < a) atomicAdd(&S.cnt[pa * G + g], 1);
    }
    __syncwarp();
    int m = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const bool is = i0 + lane < n && S.cnt[i0 + lane] >= least;
        const unsigned bal = __ballot_sync(0xffffffffu, is);
        if (is) S.list[m + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)(i0 + lane);
        m += __popc(bal);
    }
    __syncwarp();
    return m;
}

// One cluster per item, items drawn from a counter by the first CTA's helper warp and passed to the others through distributed
// shared memory (an item waits only for weights that the ratio kernel or smaller items publish, and an item that is drawn
// runs, so whatever share of the grid is resident, the smallest unfinished one never waits on anything unfinished).
//   helper warp     draws items; gathers an item's scalars while the one before runs; in the first CTA publishes what the
//                   children are handed, writes the record and makes the arrivals -- so that none of this holds up
//                   the consumers, whose sums over the cluster wait for their slowest warp
//   consumer warps  pass 1; the rows' normalisers again, from the resident e and the lists (one sum: the statistics pass
//                   gives them to fp32 accuracy only, too coarse for the differences below); the weight (Traversal);
//                   the recursion, a sweep and a sum over the cluster per rejected child
template <int DT, int NW, int RC, bool AN>
__global__ void __launch_bounds__((NW + 1) * 32, 1) spec_recursion_kernel(const NParams NP)
{
    const VParams &P = NP.v;
    BHdr &S = *reinterpret_cast<BHdr *>(dyn_smem);
    float4 *es = reinterpret_cast<float4 *>(dyn_smem + P.off_es);    // [chunk - RC][p lo, p hi, q lo, q hi][NCONS]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, C = P.C;
    const unsigned rank = cluster_ctarank();
    const bool trav = P.mode == MODE_TRAVERSAL;
    grid_launch_dependents();
    if (tid == 0) {
        common_init(S.M, NW);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&S.sfull[i], 1);
            mbar_init(&S.sempty[i], NW);
            mbar_init(&S.tbar[i], 1);
            mbar_init(&S.abar[i], C);
        }
        for (int i = 0; i < 2; ++i) {
            for (int j = 0; j < KMAX; ++j) mbar_init(&S.mb[i][j], 1);
            mbar_init(&S.mend[i], 1);
        }
        mbar_fence_init();
    }
    __syncthreads();
    cluster_sync_all();

    if (warp == NW) {
        // ================================ helper warp ===================================================
        const bool shared_tree = P.topo_stride == 0;
        const int G = shared_tree ? 1 : window_seqs(P), per = shared_tree ? P.B : 1;
        int b0 = 0, sidx = 0;
        int count = list_nodes(S, P, 0, G, 2);
        long long base = 0;
        uint32_t mph[2] = {0u, 0u}, eph = 0;      // phases of the mailboxes
        int prev = -1;                       // scalars block of the item the consumers are at
        bool going = true;
        // Analysis: where there is a cluster for every item, none draws a second one while it is at its first (50 us).
        const int clusters = (int)(gridDim.x / (unsigned)C);
        const bool ahead = !AN || (shared_tree ? (long long)count * per > clusters : G < P.B || count > clusters);
        // A node's record is written once its ratio is known: until then it may hold partial sums of the ratio kernel's.
        auto after_ratio = [&](int b, int a) {
            int w = 1;
            __syncwarp();
            if (trav && lane == 0) w = poll_weight(&P.chain[(long long)b * P.N + a].ratio, &S.M.poison) != W_PENDING;
            if (!__shfl_sync(0xffffffffu, w, 0)) S.M.poison = 1;
        };

        // rank 0: what the children of an item are handed, published as the consumers find it (the first child's has been, with the
        // item's own); the record; the arrivals
        auto serve = [&](int sb) {
            const NodeScalars &W = S.sc[sb];
            const Outcome &O = S.out[sb];
            NodeRec *rec = P.rec + (long long)W.b * P.N;
            unsigned narr = 1u;
            after_ratio(W.b, W.a);
            for (int j = 0; j < W.kc; ++j) {
                if (!*(volatile int *)&S.M.poison && !mbar_wait(&S.mb[sb][j], (mph[sb] >> j) & 1u)) S.M.poison = 1;
                mph[sb] ^= 1u << j;
                const double thr = *(volatile int *)&S.M.poison ? 0.0 : *(volatile double *)&S.out[sb].thr[j];
                const int c = W.child[j];
                if ((W.leaf_mask >> j) & 1u) { leaf_record(P, NP.part, W.b, c, thr); ++narr; }
                else if (trav) { if (j > 0 || *(volatile int *)&S.M.poison) publish_weight(P, W.b, c, thr); }
                else if (lane == 0) rec[c].thr = thr;
            }
            if (!*(volatile int *)&S.M.poison && !mbar_wait(&S.mend[sb], (eph >> sb) & 1u)) S.M.poison = 1;
            eph ^= 1u << sb;
            const bool lost = *(volatile int *)&S.M.poison != 0;
            if (lane == 0) {
                NodeRec &R = rec[W.a];
                R.O_p = (double)W.O_p; R.Z_p = O.Z_p; R.O_q = (double)W.O_q; R.Z_q = O.Z_q;
                R.kappa = O.kappa; R.nsteps = O.nsteps;
                R.cut_p = W.cut_p; R.cut_q = W.cut_q;
                R.next_child = O.acc;
                R.status = lost ? SPEC_DEV_TIMEOUT : O.err;
                R.bonus = -1; R.bonus_margin = 0.f;
                R.w_in = trav && W.a > 0 ? O.w_in : 1.0;
                if (trav) R.thr = W.a == 0 ? 1.0 : O.w_fin;
                else if (W.a == 0) R.thr = 1.0;
            }
            __syncwarp();
            arrive_sequence(P, W.b, narr);
        };

        // ticket t as a node; false: there is no such item
        auto node_of = [&](long long t, int &a, int &b) {
            while (t >= base + (long long)count * per && !shared_tree && b0 + G < P.B) {
                base += count;
                b0 += G;
                count = list_nodes(S, P, b0, min(G, P.B - b0), 2);
            }
            const int Gn = shared_tree ? 1 : min(G, P.B - b0);
            const long long k = t - base;
            if (k >= (long long)count * per) return false;
            const int li = S.list[(int)(k / per)];
            a = li / Gn;
            b = shared_tree ? (int)(k % per) : b0 + li % Gn;
            return true;
        };
        for (int kidx = 0; going; ++kidx) {
            const int buf = kidx & 1;
            int a = 0, b = 0;
            if (!ahead && rank == 0 && sidx > 0) {
                if (lane == 0 && !mbar_wait(&S.sempty[(sidx - 1) & 1], (uint32_t)(((sidx - 1) >> 1) & 1))) S.M.poison = 1;
                __syncwarp();
            }
            // ---- the item: drawn by the first CTA's helper, passed on to the others --------------------------------
            if (rank == 0) {
                int w = 1;
                unsigned t = 0;
                if (lane == 0) {
                    // every helper has read the item that used this slot before
                    if (kidx >= 2) w = mbar_wait_cluster(&S.abar[buf], (uint32_t)(((kidx >> 1) - 1) & 1)) ? 1 : 0;
                    t = atomicAdd(NP.ticket, 1u);
                }
                w = __shfl_sync(0xffffffffu, w, 0);
                t = __shfl_sync(0xffffffffu, t, 0);
                unsigned long long val = 0xFFFFFFFFull;
                if (!w) S.M.poison = 1;                            // gave up: everybody leaves
                else if (node_of((long long)t, a, b)) {
                    // a node whose weight is already known to be 0 needs no rows
                    const bool zero = trav && a > 0 && *(volatile unsigned long long *)(P.w_pub + (long long)b * P.N + a) == 0ull;
                    val = (unsigned long long)t | (zero ? 1ull << 32 : 0ull);
                }
                if (lane < C) st_async_u64(&S.item[buf], &S.tbar[buf], (uint32_t)lane, val);
            }
            unsigned long long item = 0;
            {
                int w = 1;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&S.tbar[buf], 8u);
                    w = mbar_wait_cluster(&S.tbar[buf], (uint32_t)((kidx >> 1) & 1)) ? 1 : 0;
                    item = *(volatile unsigned long long *)&S.item[buf];
                    mbar_arrive_remote(&S.abar[buf], 0u);
                }
                w = __shfl_sync(0xffffffffu, w, 0);
                item = __shfl_sync(0xffffffffu, item, 0);
                if (!w) { S.M.poison = 1; item = 0xFFFFFFFFull; }
            }
            going = (item & 0xFFFFFFFFull) != 0xFFFFFFFFull && !*(volatile int *)&S.M.poison;
            const bool zero = (item >> 32) != 0;
            if (going && rank != 0) node_of((long long)(item & 0xFFFFFFFFull), a, b);
            // ---- its scalars -----------------------------------------------------------------------------------------------
            const int sb = sidx & 1;
            if (sidx >= 2) {
                int w = 1;
                if (lane == 0) w = mbar_wait(&S.sempty[sb], (uint32_t)(((sidx >> 1) - 1) & 1)) ? 1 : 0;
                w = __shfl_sync(0xffffffffu, w, 0);
                if (!w) S.M.poison = 1;
            }
            NodeScalars &N = S.sc[sb];
            int err = 0;
            if (going) {
                const int *parent = P.parent + (long long)b * P.topo_stride;
                const int *token = P.token + (long long)b * P.N;
                const double s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
                const RowPart *rp = NP.part + ((long long)b * P.N + a) * 2;
                const RowStat p = load_stat(rp), q = load_stat(rp + 1);
                if (lane == 0) {
                    const int pa = __ldg(parent + a);
                    if (a == 0 ? (pa != -1) : (pa < 0 || pa >= a)) err = SPEC_DEV_TOPOLOGY;
                    if (a > 0) { const int x = __ldg(token + a); if (x < 0 || x >= P.V) err = SPEC_DEV_TOKEN; }
                }
                int kc = 0;
                for (int c0 = a + 1; c0 < P.N; c0 += 32) {
                    const int c = c0 + lane;
                    const bool is = c < P.N && __ldg(parent + c) == a;
                    const unsigned bal = __ballot_sync(0xffffffffu, is);
                    const int pos = kc + __popc(bal & ((1u << lane) - 1u));
                    if (is && pos < KMAX) N.child[pos] = c;
                    kc += __popc(bal);
                }
                if (kc > KMAX) err = SPEC_DEV_TOPOLOGY;
                __syncwarp();
                // lanes 0 .. 15: child j in the target row, 16 .. 31: in the draft row
                const int j = lane & 15, kce = min(kc, KMAX);
                double pr = 0.0;
                if (j < kce) {
                    const int x = __ldg(token + N.child[j]);
                    if (x < 0 || x >= P.V) err = SPEC_DEV_TOKEN;
                    else {
                        const float z = load_logit(lane < 16 ? P.zp : P.zq, DT, (long long)b * P.seq_stride + (long long)a * P.node_stride + x);
                        pr = token_e(z, lane < 16 ? p : q, s_d);
                    }
                    if (lane < 16) N.cu[j] = __ldg(P.u_accept + (long long)b * P.N + N.child[j]);
                }
                if (lane < 16) N.cpm[j] = pr; else N.cqm[j] = pr;
                // which children are childless (their grandchildren name them as parent)
                unsigned nonleaf = 0;
                for (int d0 = a + 2; d0 < P.N; d0 += 32) {
                    const int d = d0 + lane;
                    const int pd = d < P.N ? __ldg(parent + d) : -1;
                    for (int i = 0; i < kce; ++i)
                        if (pd == N.child[i]) nonleaf |= 1u << i;
                }
                nonleaf = __reduce_or_sync(0xffffffffu, nonleaf);
                err = __reduce_max_sync(0xffffffffu, err);
                if (!err && (!p.ok() || !q.ok())) err = SPEC_DEV_NONFINITE;
                if (lane == 0) {
                    N.Z_p = p.Z; N.Z_q = q.Z; N.O_p = p.O; N.O_q = q.O; N.cut_p = p.cut; N.cut_q = q.cut;
                    N.kc = kce; N.a = a; N.b = b; N.leaf_mask = ~nonleaf;
                }
                if ((err || zero) && rank == 0 && !AN) {
                    // A faulty node, or one of weight 0, is finished here: every child gets weight / threshold 0.
                    after_ratio(b, a);
                    NodeRec *rec = P.rec + (long long)b * P.N;
                    unsigned narr = 1u;
                    for (int c = a + 1; c < P.N; ++c) {
                        if (__ldg(parent + c) != a) continue;
                        if (!stream::has_children(parent, P.N, c, lane)) { leaf_record(P, NP.part, b, c, 0.0); ++narr; }
                        else if (trav) publish_weight(P, b, c, 0.0);
                        else if (lane == 0) rec[c].thr = 0.0;
                    }
                    if (lane == 0) {
                        NodeRec &R = rec[a];
                        R.O_p = (double)p.O; R.Z_p = p.Z; R.O_q = (double)q.O; R.Z_q = q.Z;
                        R.kappa = 0.0; R.nsteps = 0; R.cut_p = p.cut; R.cut_q = q.cut;
                        R.next_child = -1; R.status = err; R.bonus = -1; R.bonus_margin = 0.f;
                        R.w_in = trav && a > 0 ? 0.0 : 1.0;
                        if (trav) R.thr = a == 0 ? 1.0 : 0.0;
                        else if (a == 0) R.thr = 1.0;
                    }
                    __syncwarp();
                    arrive_sequence(P, b, narr);
                }
            }
            const bool done = err || (zero && !AN);
            if (!done) {
                if (lane == 0) N.more = going ? 1 : 0;
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.sfull[sb]);
                ++sidx;
            }
            // ---- the item before, at which the consumers have been meanwhile ---------------------------------------------
            if (!AN && rank == 0 && prev >= 0) {
                serve(prev);
                prev = -1;
            }
            if (!done && going) prev = sb;
        }
    } else {
        // ================================ consumer warps ================================================
        const bool scribe = rank == 0 && warp == 0;     // the one warp that hands results to the helper
        WarpList &L = S.M.list[warp];
        Team T = {S.M, C, warp, lane, 0, rank, 0u};
        Resident<RC> R;
        for (int kidx = 0;; ++kidx) {
            const int sb = kidx & 1;
            if (!*(volatile int *)&S.M.poison && !mbar_wait(&S.sfull[sb], (uint32_t)((kidx >> 1) & 1))) S.M.poison = 1;
            const NodeScalars &W = S.sc[sb];
            Outcome &O = S.out[sb];
            if (*(volatile int *)&S.M.poison || !W.more) break;
            const int a = W.a, b = W.b, kc = W.kc;
            int err = 0;
            NodeRows nr;
            nr.s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
            stream::split_scale(nr.s_d, nr.s_hi, nr.s_lo);
            nr.hq = true;
            nr.cut_p = W.cut_p; nr.cut_q = W.cut_q; nr.O_p = W.O_p; nr.O_q = W.O_q;
            set_list_thresholds(nr, W.Z_p, W.Z_q);
            unsigned long long bits = (unsigned long long)__double_as_longlong(1.0);
            if (trav && a > 0) bits = *(volatile unsigned long long *)(P.w_pub + (long long)b * P.N + a);    // (on its way during pass 1)
            const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
            int nl;
            float zs_p, zs_q;
            KlSums kls = {0.f, 0.f, 0.f, 0.f};
            pass1<DT, NW, RC, AN>(sl, nr, es, tid, R, L, nl, zs_p, zs_q, &kls);

            // ---- the rows' normalisers from what is resident -------------------------------------------------------------
            double Z_p = W.Z_p, Z_q = W.Z_q;
            {
                const double v[2] = {(double)zs_p + (lane < nl ? L.ep[lane] : 0.0), (double)zs_q + (lane < nl ? L.eq[lane] : 0.0)};
                double tot[2], mine[2];
                cluster_sum<NW, 2>(T, v, tot, mine);
                if (*(volatile int *)&S.M.poison) err = SPEC_DEV_TIMEOUT;
                else if (!(tot[0] > 0.0) || !(tot[1] > 0.0)) err = SPEC_DEV_NONFINITE;
                else { Z_p = tot[0]; Z_q = tot[1]; }
            }
            const double invZq = err ? 0.0 : __drcp_rn(Z_q);
            // ---- Traversal: the weight handed down by the parent (every warp for itself) --------------------------------
            double w_in = 1.0;
            if (trav && a > 0 && !err) {
                if (lane == 0 && bits == W_PENDING) bits = poll_weight(P.w_pub + (long long)b * P.N + a, &S.M.poison);
                bits = __shfl_sync(0xffffffffu, bits, 0);
                if (bits == W_PENDING) { err = SPEC_DEV_TIMEOUT; S.M.poison = 1; w_in = 0.0; }
                else w_in = __longlong_as_double((long long)bits);
            }
            // ---- offline analysis on the untouched rows (read-only sweeps, totals identical in every warp) ----------
            double an_rho = 1.0, an_beta = 0.0, an_pacc = 0.0, an_sres = 0.0;
            if (AN && !err) {
                const double ip = __drcp_rn(Z_p), iq = invZq;
                const double kd = (double)kc;
                auto sweep2 = [&](auto f, double &t0, double &t1) {
                    double v[2], tot[2], mine[2];
                    reduce_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, f, v);
                    cluster_sum<NW, 2>(T, v, tot, mine);
                    t0 = tot[0]; t1 = tot[1];
                };
                // one sweep and one sum for everything that does not depend on rho
                double v6[6], t6[6], m6[6];
                {
                    double v4[4];
                    reduce_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, FnFirst{(float)ip, (float)iq, ip, iq, kc}, v4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) v6[i] = v4[i];
                    v6[4] = (double)kls.pp - (double)kls.pq; v6[5] = (double)kls.qq - (double)kls.qp;
                    cluster_sum<NW, 6>(T, v6, t6, m6);
                }
                const double l1 = t6[0], smin = t6[1], nss = t6[2], naive2 = t6[3];
                // KL(p||q) = ln 2 (sum e_p x_p - sum e_p x_q) / Z_p - ln Z_p + ln Z_q, and the mirror image
                const double lz = log(Z_p) - log(Z_q);
                const double klpq = 0.6931471805599453 * t6[4] * ip - lz;
                const double klqp = 0.6931471805599453 * t6[5] * iq + lz;
                double sacc = 0.0;
                {
                    double dummy;
                    const auto beta = [&](double r) {
                        const double ipr = ip / r;
                        double bt;
                        sweep2(FnBeta{(float)ipr, (float)iq, ipr, iq}, bt, dummy);
                        return bt;
                    };
                    an_rho = spectr_root(kd, beta);
                    an_beta = beta(an_rho);
                    an_pacc = 1.0 - pow(1.0 - an_beta, kd);
                    const double gamma = an_beta > 0.0 ? an_pacc / an_beta : 0.0;
                    const double ib = an_beta < 1.0 ? 1.0 / (1.0 - an_beta) : 0.0;
                    sweep2(FnSpecTrRes{(float)ip, (float)iq, (float)(1.0 / an_rho), (float)gamma, (float)ib,
                                       ip, iq, 1.0 / an_rho, gamma, ib, kc}, an_sres, sacc);
                }
                if (*(volatile int *)&S.M.poison) err = SPEC_DEV_TIMEOUT;
                if (scribe && lane == 0 && !err) {
                    float *ao = NP.an_acc + ((long long)b * P.N + a) * 4, *dv = NP.an_div + ((long long)b * P.N + a) * 3;
                    ao[0] = (float)nss;
                    ao[1] = (float)(smin + naive2);
                    ao[2] = (float)(an_pacc + (1.0 - an_pacc) * (an_sres > 0.0 ? sacc / an_sres : 0.0));
                    dv[0] = (float)l1; dv[1] = (float)klpq; dv[2] = (float)klqp;
                }
            }

            // ---- the recursion, step by step (identical in every warp of the cluster) ---------------------------------------
            // state: the resident u (total kappa), the node's weight w, and in lane j < kc the value of u at
            // child j's token with its e_q (fp64, the same recursion as the vocabulary)
            const bool live = !err && w_in > 0.0;
            double w = live ? w_in : 0.0, kappa = Z_p;
            bool dead = !live, is_q = false;      // is_q: a step with S = 0 at weight 1 showed that the state equals q
            int nsteps = 0, acc = -1;
            double ux = (lane < kc) ? W.cpm[lane] : 0.0;
            const double eqx = (lane < kc) ? W.cqm[lane] : 0.0;
            double *gs = NP.gseq + ((long long)b * P.N + a) * KMAX;
            auto hand = [&](int j, double thr) {
                if (!AN && scribe && lane == 0) { *(volatile double *)&O.thr[j] = thr; mbar_arrive(&S.mb[sb][j]); }
            };
            for (int j = 0; j < kc; ++j) {
                if (err || acc >= 0 && !P.all_thr) { hand(j, err ? 0.0 : CUDART_NAN); continue; }
                // child j from the current state: P(x) = u(x) / kappa, q(x) = e_q(x) / Z_q
                const double uxj = __shfl_sync(0xffffffffu, ux, j), eqj = __shfl_sync(0xffffffffu, eqx, j);
                const double Pq = eqj * invZq;
                const double Pp = is_q ? Pq : uxj / kappa;
                if (AN && scribe && lane < kc) {
                    // round j's acceptance probability of every child's token: min(1, p_j(x_t) / q(x_t))
                    const double q_t = eqx * invZq, p_t = is_q ? q_t : ux / kappa;
                    NP.an[(long long)b * P.N + a].A[j][lane] = fmin(1.0, token_ratio(p_t, q_t));
                }
                const double thr = dead ? 0.0 : (trav ? handed_weight(w, token_ratio(Pp, Pq)) : fmin(1.0, token_ratio(Pp, Pq)));
                hand(j, thr);
                if (!trav && acc < 0 && (double)W.cu[j] < thr) {
                    acc = W.child[j];
                    if (!P.all_thr) continue;
                }
                if (AN && scribe && lane == 0 && (dead || is_q)) NP.an[(long long)b * P.N + a].S[j] = 0.0;
                if (dead || is_q) continue;       // weight 0, or P = q (every further step has S = 0 again)
                // the step after rejecting child j: u <- (g u - e_q)+ , g = w Z_q / kappa
                const double g = __ddiv_rn(w * Z_q, kappa);
                const double v[1] = {step_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, g)};
                double tot[1], mine[1];
                cluster_sum<NW, 1>(T, v, tot, mine);
                if (*(volatile int *)&S.M.poison) { err = SPEC_DEV_TIMEOUT; continue; }
                ux = fmax(fma(g, ux, -eqx), 0.0);
                const double Sj = tot[0] * invZq;
                if (AN && scribe && lane == 0) NP.an[(long long)b * P.N + a].S[j] = Sj > RESIDUAL_FLOOR * w ? Sj : 0.0;
                // A step whose mass is below 1e-13 of the weight before it counts as S = 0: P equals q, and what
                // is left is the rounding of g.
                if (Sj > RESIDUAL_FLOOR * w) {
                    kappa = tot[0];
                    if (trav) w = Sj / (Sj + (1.0 - w));
                    if (scribe && lane == 0) gs[nsteps] = g;
                    ++nsteps;
                } else if (w >= 1.0) {
                    is_q = true;       // S = 0 with w = 1: the state is q itself (the stored u is no longer used)
                    kappa = Z_q;
                } else {
                    dead = true;       // S = 0 with w < 1: the weight drops to 0 (Traversal only)
                    w = 0.0;
                }
            }
            if (AN && scribe) {
                AnRec &Ar = NP.an[(long long)b * P.N + a];
                if (lane < kc) {
                    const double q_t = eqx * invZq;
                    Ar.A[kc][lane] = err ? 0.0 : (is_q ? q_t : ux / kappa);      // p_k(x_t)
                    Ar.px[lane] = W.cpm[lane] / Z_p;
                    Ar.qx[lane] = q_t;
                }
                if (lane == 0) {
                    Ar.rho = an_rho; Ar.beta = an_beta; Ar.pacc = an_pacc; Ar.s_res = an_sres;
                    Ar.k = kc; Ar.valid = err ? 0 : 1;
                }
            }
            if (!AN && scribe && lane == 0) {
                O.w_in = w_in;
                O.w_fin = (dead || err) ? 0.0 : w;
                O.kappa = (dead || err) ? 0.0 : kappa;
                O.Z_p = Z_p; O.Z_q = Z_q;
                O.nsteps = is_q ? STATE_IS_Q : nsteps;
                O.acc = acc; O.err = err;
                mbar_arrive(&S.mend[sb]);
            }
            // the scalars block may be rewritten
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.sempty[sb]);
        }
    }
    __syncthreads();
    cluster_sync_all();        // nobody leaves while a peer may still write to its shared memory
    if (blockIdx.x == 0) grid_dependency_wait();      // this kernel ends only after the one before it
}

// ------------------------------------------------------------------------------------------------
// the bonus draw
// ------------------------------------------------------------------------------------------------
struct __align__(16) FHdr {
    Common M;
};

// One cluster per sequence: waits (bounded) until the accepted node is selected, brings its rows on chip, takes its recorded steps
// (the step of a node with one child, which was left out, from the rows' exact normalisers) and draws the bonus token.
template <int DT, int NW, int RC>
__global__ void __launch_bounds__(NW * 32, 1) spec_finish_kernel(const NParams NP)
{
    const VParams &P = NP.v;
    FHdr &S = *reinterpret_cast<FHdr *>(dyn_smem);
    float4 *es = reinterpret_cast<float4 *>(dyn_smem + P.off_es);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, C = P.C;
    const unsigned rank = C > 1 ? cluster_ctarank() : 0u;
    if (P.early) grid_launch_dependents();
    if (tid == 0) {
        common_init(S.M, NW);
        mbar_fence_init();
    }
    __syncthreads();
    if (C > 1) cluster_sync_all();
    WarpList &L = S.M.list[warp];
    Team T = {S.M, C, warp, lane, 0, rank, 0u};
    Resident<RC> R;
    for (int b = (int)(blockIdx.x / (unsigned)C); b < P.B; b += (int)(gridDim.x / (unsigned)C)) {
        int acc = FIN_PENDING;
        if (lane == 0) {
            volatile int *slot = P.fin + b;
            const long long t0 = clock64();
            for (;;) {
                acc = *slot;
                if (acc != FIN_PENDING || clock64() - t0 > WAIT_CYCLES || *(volatile int *)&S.M.poison) break;
                __nanosleep(64);
            }
            __threadfence();       // the records written before the publication are read below
        }
        acc = __shfl_sync(0xffffffffu, acc, 0);
        if (acc == FIN_PENDING) S.M.poison = 1;
        if (acc == FIN_FAULTY) continue;           // a faulty sequence has no bonus draw: its status says why
        const int len = acc < 0 ? 0 : acc >> FIN_LEN_SHIFT, a = acc < 0 ? 0 : acc & ((1 << FIN_LEN_SHIFT) - 1);
        NodeRec *rc = P.rec + (long long)b * P.N + a;
        // (all coefficients are fetched in the same round of loads as the step count: only the first nsteps are used)
        const double gj = lane < KMAX ? __ldcg(NP.gseq + ((long long)b * P.N + a) * KMAX + lane) : 0.0;
        const int nsteps = __ldcg(&rc->nsteps);
        const double w = __ldcg(&rc->w_in), Zs_p = __ldcg(&rc->Z_p), Zs_q = __ldcg(&rc->Z_q);
        NodeRows nr;
        nr.s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
        stream::split_scale(nr.s_d, nr.s_hi, nr.s_lo);
        nr.hq = nsteps != 0;                       // (the draft row only if the node's state is not its target row)
        nr.O_p = (int)__ldcg(&rc->O_p); nr.O_q = (int)__ldcg(&rc->O_q);
        nr.cut_p = __ldcg(&rc->cut_p); nr.cut_q = __ldcg(&rc->cut_q);
        set_list_thresholds(nr, Zs_p, Zs_q);
        const double ub = (double)__ldg(P.u_bonus + (long long)b * P.N + a);
        const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
        int nl;
        float zs_p, zs_q;
        pass1<DT, NW, RC>(sl, nr, es, tid, R, L, nl, zs_p, zs_q);
        bool is_q = nsteps == STATE_IS_Q;
        double part = (double)zs_p + (lane < nl ? L.ep[lane] : 0.0);
        const double part_q = (double)zs_q + (lane < nl ? L.eq[lane] : 0.0);
        double tot[1], mine[1];
        if (nsteps == STATE_FIRST) {
            const double v2[2] = {part, part_q};
            double t2[2], m2[2];
            cluster_sum<NW, 2>(T, v2, t2, m2);
            const double g = t2[0] > 0.0 ? __ddiv_rn(w * t2[1], t2[0]) : 0.0;
            const double v[1] = {step_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, g)};
            cluster_sum<NW, 1>(T, v, tot, mine);
            is_q = !(tot[0] > RESIDUAL_FLOOR * w * t2[1]);
            if (P.out.residual && rank == 0 && tid == 0) {
                // (the residual output replays the recorded steps)
                NP.gseq[((long long)b * P.N + a) * KMAX] = g;
                rc->kappa = is_q ? t2[1] : tot[0];
                rc->nsteps = is_q ? STATE_IS_Q : 1;
            }
            if (is_q) { tot[0] = t2[1]; mine[0] = m2[1]; }     // S = 0: the state equals q
        } else {
            if (is_q) part = part_q;
            for (int j = 0; j < nsteps; ++j) part = step_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, __shfl_sync(0xffffffffu, gj, j));
            const double v[1] = {part};
            cluster_sum<NW, 1>(T, v, tot, mine);
        }
        int ferr = *(volatile int *)&S.M.poison ? SPEC_DEV_TIMEOUT : 0;
        double tau = 0.0;
        int owner = -1;
        if (!ferr) {
            owner = pick_lane(lane < C ? mine[0] : 0.0, ub * tot[0], tau);
            if (owner < 0) ferr = SPEC_DEV_NONFINITE;
        }
        int role = 0, tokn = -1;
        float mg = 0.f;
        if (ferr) {
            role = (rank == 0 && tid == 0) ? (ferr == SPEC_DEV_TIMEOUT ? 3 : 2) : 0;
        } else if (owner == (int)rank) {
            const BonusFind bf = bonus_search<NW, RC>(T, sl, es, tid, R, L, nl, is_q, tau);
            role = bf.role;
            tokn = bf.token;
            mg = (float)(bf.edge / tot[0]);
        }
        if (role == 1) {
            P.out.bonus_token[b] = tokn;
            P.out.out_tokens[(long long)b * P.N + len] = tokn;
            if (P.out.margin) P.out.margin[(long long)b * (P.N + 1) + P.N] = mg;
        } else if (role >= 2) {
            P.out.status[b] = role == 3 ? SPEC_DEV_TIMEOUT : SPEC_DEV_NONFINITE;
            P.out.accepted_node[b] = -1; P.out.accept_len[b] = -1; P.out.bonus_token[b] = -1;
            int *ot = P.out.out_tokens + (long long)b * P.N;
            for (int i = 0; i < P.N; ++i) ot[i] = -1;
        }
    }
    __syncthreads();
    if (C > 1) cluster_sync_all();        // nobody leaves while a peer may still write to its shared memory
    if (blockIdx.x == 0) grid_dependency_wait();      // this kernel ends only after the ones before it
}

}  // namespace specv
