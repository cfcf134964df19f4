// Offline analysis of a draft tree on the resident node data of the recursion kernel (nodes.cuh in its
// analysis instantiation): acceptance rates (Definition 5.1, Algorithms 6-9), the divergences between
// target and draft (Section 5's L1, the selector's KL features of Section 6), branching probabilities
// (Definition 5.3, Algorithms 11-14) and the block-efficiency sum of equation (3); and the forward-time
// model of equation (8).
//
// Division of work.  The recursion kernel holds a node's e_p, e_q on chip with its dominant tokens
// exact; in analysis mode it runs, before the SpecInfer recursion, read-only sweeps for the vocabulary-wide
// sums (the functors below) and the search for SpecTr's rho*, and dumps per node the scalars everything
// else follows from (AnRec).  spec_branch_kernel (one warp per node) turns them into branching
// probabilities -- for SpecInfer with uniformly picked children the dynamic programme of Algorithm 14 over
// the sets of remaining children -- and spec_reach_kernel multiplies them down the tree.
//
// Algorithm 9's last term vanishes identically: a token with positive final residual p_k(t) was above
// q(t) in every round, so its m(t) stayed 1 and p_k(t) (1 - m(t)) = 0; SpecInfer's acceptance rate is
// 1 - prod_i S_i with S_i the residual mass of round i, which the recursion already has.
#pragma once
#include "common.cuh"

namespace specv {

constexpr int AN_KDP = 10;            // uniform-order SpecInfer: the DP covers up to 2^AN_KDP sets of children

// per node, dumped by the recursion kernel in analysis mode
struct __align__(16) AnRec {
    double A[KMAX + 1][KMAX];   // A[i][t] = min(1, p_i(x_t) / q(x_t)) for round i < k; row k: p_k(x_t)
    double S[KMAX];             // residual mass of round i (0 once the state equals q)
    double px[KMAX], qx[KMAX];  // p(x_t), q(x_t)
    double rho, beta, pacc, s_res;   // SpecTr: division factor, beta(rho*), p_acc, sum (p - min(p/rho, q) gamma)+
    int k, valid, pad[2];
};

// ---- functors of the read-only sweeps: tail in fp32, listed tokens in fp64 -----------------------------------
// x (1 + r + ... + r^(k-1)) with r = 1 - x, that is 1 - (1 - x)^k without its cancellation (all terms positive)
template <typename F>
__device__ __forceinline__ F one_minus_power(F x, int k)
{
    const F r = (F)1 - x;
    F s = (F)1;
    for (int i = 1; i < k; ++i) s = s * r + (F)1;
    return k > 0 ? x * s : (F)0;
}
struct FnFirst {        // sum |p - q|, sum min(p, q), sum p (1 - (1-q)^k)  (Algorithm 6), sum (p-q)+ (1 - (1-q)^(k-1))
                        // (Algorithm 7)
    float ipf, iqf; double ip, iq; int k;
    template <typename F> __device__ __forceinline__ void add(F p, F q, F (&a)[4]) const
    {
        const F d = p - q, dp = d > (F)0 ? d : (F)0, qc = q < (F)1 ? q : (F)1;
        a[0] += d > (F)0 ? d : -d;
        a[1] += p < q ? p : q;
        a[2] += p * one_minus_power(qc, k);
        a[3] += dp * one_minus_power(qc, k - 1);
    }
    // (eight tokens side by side in the loop over k)
    __device__ __forceinline__ void tail8(const float (&ep)[8], const float (&eq)[8], float (&a)[4]) const
    {
        float p[8], q[8], r[8], s[8], before[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) { p[t] = ep[t] * ipf; q[t] = eq[t] * iqf; r[t] = 1.f - fminf(q[t], 1.f); s[t] = 1.f; before[t] = 0.f; }
#pragma unroll 1
        for (int i = 1; i < k; ++i) {
#pragma unroll
            for (int t = 0; t < 8; ++t) { before[t] = s[t]; s[t] = fmaf(s[t], r[t], 1.f); }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const float d = p[t] - q[t], dp = fmaxf(d, 0.f), qc = fminf(q[t], 1.f);
            a[0] += fabsf(d);
            a[1] += fminf(p[t], q[t]);
            a[2] = fmaf(p[t], qc * s[t], a[2]);
            a[3] = fmaf(dp, qc * before[t], a[3]);
        }
    }
    __device__ __forceinline__ void exact(double ep, double eq, double (&a)[4]) const { add(ep * ip, eq * iq, a); }
};
struct FnBeta {         // beta(rho) = sum min(p / rho, q)   (Appendix B, above Algorithm 3)
    float ipf, iqf; double ip, iq;   // ip already divided by rho
    __device__ __forceinline__ void tail8(const float (&ep)[8], const float (&eq)[8], float (&a)[2]) const
    {
        float u = 0.f, v = 0.f;                 // (two chains of additions)
#pragma unroll
        for (int t = 0; t < 8; t += 2) { u += fminf(ep[t] * ipf, eq[t] * iqf); v += fminf(ep[t + 1] * ipf, eq[t + 1] * iqf); }
        a[0] += u + v;
    }
    __device__ __forceinline__ void exact(double ep, double eq, double (&a)[2]) const { a[0] += fmin(ep * ip, eq * iq); }
};
struct FnSpecTrRes {    // sum d, sum d (1 - (1-r)^k), d = (p - min(p/rho, q) gamma)+, r = (q - p/rho)+ / (1-beta)
    float ipf, iqf, irf, gf, ibf; double ip, iq, ir, g, ib; int k;     // ir = 1/rho, ib = 1/(1-beta) (0 when beta = 1)
    __device__ __forceinline__ void tail8(const float (&ep)[8], const float (&eq)[8], float (&a)[2]) const
    {
        float d[8], x[8], s[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const float p = ep[t] * ipf, q = eq[t] * iqf, pr = p * irf;
            d[t] = fmaxf(p - fminf(pr, q) * gf, 0.f);
            x[t] = fminf(fmaxf(q - pr, 0.f) * ibf, 1.f);
            s[t] = 1.f;
        }
#pragma unroll 1
        for (int i = 1; i < k; ++i) {
#pragma unroll
            for (int t = 0; t < 8; ++t) s[t] = fmaf(s[t], 1.f - x[t], 1.f);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) { a[0] += d[t]; a[1] = fmaf(d[t], x[t] * s[t], a[1]); }
    }
    __device__ __forceinline__ void exact(double ep, double eq, double (&a)[2]) const
    {
        const double p = ep * ip, q = eq * iq, pr = p * ir;
        const double d = fmax(p - fmin(pr, q) * g, 0.0);
        const double r = fmin(fmax(q - pr, 0.0) * ib, 1.0);
        a[0] += d;
        a[1] += d * one_minus_power(r, k);
    }
};

// SpecTr's division factor: the root of f(rho) = 1 - (1 - beta)^k - rho beta on [1, k] (Appendix B), f(1) >= 0 >= f(k).
// Regula falsi with the Illinois rule (the value at an end that stays is halved), and the middle whenever two steps
// have not halved the bracket -- so never more than about twice the steps of a bisection, and about ten where f is
// smooth (40 halvings of [1, k], the accuracy that is asked for here, are 40 sweeps over the node and sums over the cluster).
// (on the host too, for its test)
#pragma nv_exec_check_disable
template <typename F>
__host__ __device__ __forceinline__ double spectr_root(double k, F beta)
{
    const auto f = [&](double r) { const double b = beta(r); return (1.0 - pow(1.0 - b, k)) - r * b; };
    double lo = 1.0, hi = k, flo = f(lo), fhi = f(hi);
    if (!(flo > 0.0)) return 1.0;
    const double close = (k - 1.0) * 9.094947017729282e-13;       // 2^-40
    double was = hi - lo;
    int side = 0;
    for (int it = 0; it < 96 && hi - lo > close; ++it) {
        double x = fhi < 0.0 ? (lo * fhi - hi * flo) / (fhi - flo) : hi;
        if ((it & 1) && hi - lo > 0.5 * was) x = 0.5 * (lo + hi);
        if (it & 1) was = hi - lo;
        if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
        const double fx = f(x);
        if (fx > 0.0) {
            lo = x; flo = fx;
            if (side > 0) fhi *= 0.5;
            side = 1;
        } else {
            hi = x; fhi = fx;
            if (side < 0) flo *= 0.5;
            side = -1;
        }
    }
    return 0.5 * (lo + hi);
}

namespace analysis {

enum Solver { NSS = 0, NAIVE = 1, SPECTR = 2, SPECINFER = 3, SPECINFER_UNIFORM = 4, NSOLVER = 5 };

struct BParams {
    int B, N;
    const int *parent, *token;
    long long topo_stride;
    const AnRec *an;         // [B*N]
    float *acc;              // [B,N,4]: entry 3 (SpecInfer) is written here; NaN at childless nodes
    float *branch;           // [NSOLVER][B,N]: probability of moving from the parent into the node (root: 1)
};

__device__ __forceinline__ double clip1(double r) { return r < 1.0 ? r : 1.0; }
__device__ __forceinline__ double ratio(double P, double Q) { return !(P > 0.0) ? 0.0 : (!(Q > 0.0) ? CUDART_INF : P / Q); }

// One warp per node with children: branching probabilities of the five solvers into each child.
// A child whose token an earlier sibling carries is never moved to (the walk takes the first): 0.
__global__ void __launch_bounds__(128) spec_branch_kernel(const BParams P)
{
    __shared__ double dp[4][1 << AN_KDP];
    grid_dependency_wait();
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long node = (long long)blockIdx.x * 4 + wib;
    if (node >= (long long)P.B * P.N) return;
    const int b = (int)(node / P.N), a = (int)(node % P.N);
    const long long BN = (long long)P.B * P.N;
    if (a == 0 && lane < NSOLVER) P.branch[(long long)lane * BN + node] = 1.f;
    const AnRec &R = P.an[node];
    const int k = R.k;
    if (k <= 0 || !R.valid) {
        if (lane == 0) P.acc[node * 4 + 3] = CUDART_NAN_F;
        return;
    }
    const int *parent = P.parent + (long long)b * P.topo_stride;
    const int *token = P.token + (long long)b * P.N;
    // the children (list order) and their tokens: lane j holds child j
    int child = -1, tok = -1;
    {
        int seen = 0;
        for (int c0 = a + 1; c0 < P.N && seen < k; c0 += 32) {
            const int c = c0 + lane;
            const bool is = c < P.N && __ldg(parent + c) == a;
            const unsigned bal = __ballot_sync(0xffffffffu, is);
            // child number pos sits in lane pos
            for (int l = 0; l < 32; ++l) {
                if (!((bal >> l) & 1u)) continue;
                const int pos = seen + __popc(bal & ((1u << l) - 1u));
                const int cc = c0 + l;
                if (lane == pos) { child = cc; tok = __ldg(token + cc); }
            }
            seen += __popc(bal);
        }
    }
    // SpecInfer acceptance (Algorithm 9): 1 - prod S_i
    if (lane == 0) {
        double prej = 1.0;
        for (int i = 0; i < k; ++i) prej *= R.S[i];
        P.acc[node * 4 + 3] = (float)(1.0 - prej);
    }
    const bool mine = lane < k;
    bool dup = false;
    for (int l = 0; l < k; ++l) {
        const int tl = __shfl_sync(0xffffffffu, tok, l);
        if (mine && l < lane && tl == tok) dup = true;
    }
    const double pj = mine ? R.px[lane] : 0.0, qj = mine ? R.qx[lane] : 0.0;
    double out[NSOLVER] = {0.0, 0.0, 0.0, 0.0, 0.0};
    // NSS (Algorithm 11)
    out[NSS] = pj;
    // Naive (Algorithm 12): a = min(1, p(X_1)/q(X_1)); residual (p - q)+ / S_1
    {
        const double a1 = clip1(ratio(R.px[0], R.qx[0]));
        const double S1 = R.S[0];
        const double res = S1 > 0.0 ? fmax(pj - qj, 0.0) / S1 : pj;
        const int t0 = __shfl_sync(0xffffffffu, tok, 0);
        out[NAIVE] = (1.0 - a1) * res + (tok == t0 ? a1 : 0.0);
    }
    // SpecTr (Algorithm 13)
    {
        const double rho = R.rho;
        const double gamma = R.beta > 0.0 ? R.pacc / R.beta : 0.0;
        const double aj = mine ? clip1(ratio(pj, qj) / rho) : 0.0;
        double pre = 1.0, s = 0.0;
        for (int l = 0; l < k; ++l) {
            const double al = __shfl_sync(0xffffffffu, aj, l);
            const int tl = __shfl_sync(0xffffffffu, tok, l);
            if (tl == tok) s += al * pre;
            pre *= 1.0 - al;
        }
        const double res = R.s_res > 0.0 ? fmax(pj - fmin(pj / rho, qj) * gamma, 0.0) / R.s_res : pj;
        out[SPECTR] = s + res * pre;
    }
    // SpecInfer, children tried in list order: child l is tested in round l with A[l][l]
    {
        double pre = 1.0, s = 0.0;
        for (int l = 0; l < k; ++l) {
            const double al = R.A[l][l];
            const int tl = __shfl_sync(0xffffffffu, tok, l);
            if (tl == tok) s += al * pre;
            pre *= 1.0 - al;
        }
        out[SPECINFER] = s + (mine ? R.A[k][lane] : 0.0) * pre;
    }
    // SpecInfer, the next child picked uniformly (Algorithm 14): dynamic programme over the sets of children
    // still in S (bit t of the mask: child t), sets visited in increasing order, 32 per step
    if (k <= AN_KDP) {
        double *Bt = dp[wib];
        int toks[AN_KDP];
#pragma unroll
        for (int t = 0; t < AN_KDP; ++t) toks[t] = __shfl_sync(0xffffffffu, tok, t);
        for (int xi = 0; xi < k; ++xi) {
            const int tx = __shfl_sync(0xffffffffu, tok, xi);
            const double pkx = R.A[k][xi];
            const int nS = 1 << k;
            if (lane == 0) Bt[0] = pkx;
            __syncwarp();
            // all sets with cnt members depend only on sets with cnt - 1 members
            for (int cnt = 1; cnt <= k; ++cnt) {
                for (int S0 = 0; S0 < nS; S0 += 32) {
                    const int Sm = S0 + lane;
                    if (Sm < nS && __popc(Sm) == cnt) {
                        const int i = k - cnt;
                        double s = 0.0;
#pragma unroll
                        for (int t = 0; t < AN_KDP; ++t)
                            if (t < k && ((Sm >> t) & 1)) {
                                const double at = R.A[i][t];
                                s += at * (toks[t] == tx ? 1.0 : 0.0) + (1.0 - at) * Bt[Sm & ~(1 << t)];
                            }
                        Bt[Sm] = s / (double)cnt;
                    }
                }
                __syncwarp();
            }
            const double v = Bt[nS - 1];
            if (lane == xi) out[SPECINFER_UNIFORM] = v;
            __syncwarp();
        }
    } else {
        out[SPECINFER_UNIFORM] = CUDART_NAN;
    }
    if (mine) {
#pragma unroll
        for (int s = 0; s < NSOLVER; ++s) P.branch[(long long)s * BN + (long long)b * P.N + child] = dup ? 0.f : (float)out[s];
    }
}

struct RParams {
    int B, N;
    const int *parent;
    long long topo_stride;
    const float *branch;     // [NSOLVER][B,N]
    float *reach;            // [NSOLVER][B,N]: product of the branching probabilities along the node's path
    float *block_eff;        // [NSOLVER][B]: sum of reach over the nodes = E[tau + 1 | tree]  (equation (3))
};

// one thread per (solver, sequence): parents come before their children
__global__ void spec_reach_kernel(const RParams P)
{
    grid_dependency_wait();
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= NSOLVER * P.B) return;
    const int s = id / P.B, b = id % P.B;
    const int *parent = P.parent + (long long)b * P.topo_stride;
    const float *br = P.branch + ((long long)s * P.B + b) * P.N;
    float *re = P.reach + ((long long)s * P.B + b) * P.N;
    double total = 0.0;
    for (int a = 0; a < P.N; ++a) {
        const int pa = parent[a];
        const double r = a == 0 ? 1.0 : ((pa >= 0 && pa < a) ? (double)re[pa] * (double)br[a] : CUDART_NAN);
        re[a] = (float)r;
        total += r;
    }
    P.block_eff[(long long)s * P.B + b] = (float)total;
}

// Equation (8): forward-pass time of every action (K, L1, L2) at context length ctx from the measured
// tables t_q, t_p (a length beyond a table uses its last entry); one thread per action.
struct LParams {
    const double *t_q, *t_p;
    int n_len, ctx, A;
    const int *actions;      // [A,3]
    double *T_hat;           // [A]
};
__global__ void spec_latency_kernel(const LParams P)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= P.A) return;
    const int K = P.actions[3 * a], L1 = P.actions[3 * a + 1], L2 = P.actions[3 * a + 2];
    auto tab = [&](const double *t, int l) { return t[l < 0 ? 0 : (l >= P.n_len ? P.n_len - 1 : l)]; };
    double s = 0.0;
    for (int j = 0; j < L1; ++j) s += tab(P.t_q, P.ctx + j);
    for (int j = 0; j < L2; ++j) s += tab(P.t_q, P.ctx + L1 + j * K);
    s += tab(P.t_p, P.ctx + L1 + K * L2);
    P.T_hat[a] = s;
}

}  // namespace analysis
}  // namespace specv
