// SpecInfer verification as a walk (Algorithm 4 composed top-down, Section 3.2), one thread-block
// cluster per sequence, on top of the row statistics (stream.cuh / trunc.cuh).
//
// With every row's normaliser known, the decision about a node's FIRST child needs no vocabulary-wide
// work: its threshold is min(1, p(x)/q(x)), two logits and two normalisers.  The cluster therefore walks
// down the tree with scalar arithmetic only, and brings a node's rows on chip (verify.cuh) only
// where Algorithm 4 needs a residual: at a node whose first child was rejected, and at the stop node
// for the bonus draw.  That is one or two resident nodes per sequence instead of every node of the tree.
//
// The prologue brings the sequence's scalars into shared memory: topology, tokens and uniforms with, for every
// non-root node, the two logits at its token in its parent's rows (inputs, so the first sequence's are fetched while
// the statistics kernel is still running), then the row records, then the exponentials of those logits in fp64.
// After that a step down the tree is a few shared-memory reads.  The first child's test uses the
// normalisers of the statistics pass (fp32 exponentials: its threshold is good to a few 1e-7); a node
// that comes on chip gets its normalisers again from the resident e and the exact lists of verify.cuh.
//
// Every warp of the cluster runs the same walk on the same numbers (the sums over the cluster are
// bit-identical in all of them), so control flow agrees across the cluster without barriers.
// The thread that finds the bonus token writes all outputs of the sequence.
#pragma once
#include "analysis.cuh"
#include "stream.cuh"
#include "verify.cuh"

namespace specv {

constexpr int NWALK = 128;        // nodes per sequence the walk keeps in shared memory

struct WParams {
    int B, N, V, C;
    int off_es;
    const void *zp, *zq;
    long long seq_stride, node_stride, topo_stride;
    const int *parent, *token;
    float T;
    const float *T_seq;
    const RowPart *part;      // [B*N*2]
    const float *u_accept, *u_bonus;
    SpecOut out;
    int solver;               // OT instantiation: 0 NSS (Algorithm 1), 1 NaiveTree (Algorithm 2), 2 SpecTr (Algorithm 3)
};

// per warp: the children of the current node
struct __align__(16) WarpArea {
    double cpm[KMAX], cqm[KMAX];   // exact 2^(z s - O) of the children's tokens in the node's target and draft rows
    float cu[KMAX];
    int child[KMAX];
};

struct __align__(16) WHdr {
    Common M;
    WarpArea wa[NWMAX];
    // the sequence's scalars (written by the prologue of every sequence)
    int t_parent[NWALK], t_token[NWALK], t_fc[NWALK], t_kc[NWALK];
    float t_u[NWALK], t_ub[NWALK];
    float t_zp[NWALK], t_zq[NWALK];    // the logits of the node's token in its parent's rows
    double t_Z[2 * NWALK];        // normaliser of row (node, target / draft), in units of 2^O
    int t_O[2 * NWALK];
    float t_cut[2 * NWALK];
    double t_cp[NWALK], t_cq[NWALK];   // exact 2^(z s - O) of the node's token in its parent's target and draft rows
    int t_status;
};

// statistics of one row: normaliser, reference, cut
struct RowSum {
    double Z;
    int O;
    float cut;
};

// NW consumer warps (8 in all variants).  RC chunks of a thread in registers and MINB CTAs per SM: 0 and 1 where a CTA
// has an SM to itself, 4 and 2 (bf16 only) where two share one, 8 and 1 for vocabularies beyond the shared memory of 16 CTAs.
// OT: the walk with one of the other OTLP solvers of Appendix B instead of SpecInfer (Section 3.2: move to the
// child whose token the solver put out, stop when the output is no child's token).  Every draw is then
// made known to the whole cluster (one more sum), because the walk may go on from it.
template <int DT, int NW, int RC, int MINB, bool OT>
__global__ void __launch_bounds__(NW * 32, MINB) spec_walk_kernel(const WParams P)
{
    constexpr int NCONS = NW * 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    WHdr &S = *reinterpret_cast<WHdr *>(dyn_smem);
    float4 *es = reinterpret_cast<float4 *>(dyn_smem + P.off_es);    // [chunk - RC][p lo, p hi, q lo, q hi][NCONS]
    const int C = P.C;
    const unsigned rank = cluster_ctarank();
    const int cid = blockIdx.x / C, NC = gridDim.x / C;

    if (tid == 0) {
        common_init(S.M, NW);
        mbar_fence_init();
    }
    __syncthreads();
    if (C > 1) cluster_sync_all();

    {
        WarpArea &W = S.wa[warp];
        WarpList &L = S.M.list[warp];
        Team T = {S.M, C, warp, lane, 0, rank, 0u};
        Resident<RC> R;

        for (int b = cid; b < P.B; b += NC) {
            const int *parent = P.parent + (long long)b * P.topo_stride;
            const int *token = P.token + (long long)b * P.N;
            NodeRows nr;
            nr.s_d = 1.4426950408889634 / (double)(P.T_seq ? __ldg(P.T_seq + b) : P.T);
            stream::split_scale(nr.s_d, nr.s_hi, nr.s_lo);
            const double s_d = nr.s_d;

            // ---- the inputs' scalars; the whole tree is checked -------------------------------------------------------
            bar_sync(1, NCONS);                      // the previous sequence's scalars are no longer read
            if (tid == 0) S.t_status = 0;
            bar_sync(1, NCONS);
            {
                int st1 = 0;
                for (int i = tid; i < P.N; i += NCONS) {
                    const int pa = __ldg(parent + i);
                    const bool bad_pa = i == 0 ? (pa != -1) : (pa < 0 || pa >= i);
                    if (bad_pa) st1 = max(st1, SPEC_DEV_TOPOLOGY);
                    int x = 0;
                    if (i > 0) {
                        x = __ldg(token + i);
                        const bool bad_x = x < 0 || x >= P.V;
                        if (bad_x) st1 = max(st1, SPEC_DEV_TOKEN);
                        if (!bad_pa && !bad_x) {
                            const long long at = (long long)b * P.seq_stride + (long long)pa * P.node_stride + x;
                            S.t_zp[i] = load_logit(P.zp, DT, at);
                            S.t_zq[i] = load_logit(P.zq, DT, at);
                        }
                    }
                    S.t_parent[i] = pa; S.t_token[i] = x; S.t_fc[i] = P.N; S.t_kc[i] = 0;
                    S.t_u[i] = __ldg(P.u_accept + (long long)b * P.N + i);
                    S.t_ub[i] = __ldg(P.u_bonus + (long long)b * P.N + i);
                }
                if (b == cid) grid_dependency_wait();       // the row statistics come from the kernel before
                for (int r2 = tid; r2 < 2 * P.N; r2 += NCONS) {
                    const RowPart *p = P.part + ((long long)b * 2 * P.N + r2);
                    const double Zr = __ldcg(&p->S);
                    const int4 rest = __ldcg(reinterpret_cast<const int4 *>(p) + 1);     // O, xmax, cut, bad
                    const int Or = rest.x, bd = rest.w;
                    // a row is not finite if it holds NaN / +inf, or no finite logit at all
                    if (bd != -1 && (bd == 1 || !(Or > ROWPART_EMPTY) || !(Zr > 0.0) || !(Zr < CUDART_INF)))
                        st1 = max(st1, SPEC_DEV_NONFINITE);
                    S.t_Z[r2] = Zr; S.t_O[r2] = Or; S.t_cut[r2] = __int_as_float(rest.z);
                }
                if (st1) atomicMax(&S.t_status, st1);
            }
            bar_sync(1, NCONS);
            // ---- children, and the exponential of every node's token in its parent's rows -----------------------------
            if (S.t_status == 0) {
                int st2 = 0;
                for (int c2 = 2 + tid; c2 < 2 * P.N; c2 += NCONS) {        // (node, target / draft)
                    const int c = c2 >> 1, h = c2 & 1, a = S.t_parent[c];
                    if (h == 0) {
                        atomicMin(&S.t_fc[a], c);
                        if (atomicAdd(&S.t_kc[a], 1) >= KMAX) st2 = SPEC_DEV_TOPOLOGY;
                    }
                    const float z = h ? S.t_zq[c] : S.t_zp[c];
                    const double xd = (double)z * s_d - (double)S.t_O[2 * a + h];
                    double pr = 0.0;
                    if (z >= S.t_cut[2 * a + h] && xd > -1000.0) {
                        const double nd = rint(xd);
                        pr = exp2_frac_once(xd - nd) * pow2d((int)nd);
                    }
                    (h ? S.t_cq : S.t_cp)[c] = pr;
                }
                if (st2) atomicMax(&S.t_status, st2);
            }
            bar_sync(1, NCONS);
            int status = S.t_status;
            int cur = 0, len = 0;
            int bonus = -1;
            bool writer = false;          // this lane writes the sequence's outputs
            bool done = status != 0;
            if (done && rank == 0 && warp == 0 && lane == 0) { writer = true; cur = -1; len = -1; }

            while (!done) {
                const int a = cur;
                const int c_first = S.t_fc[a];
                const bool hq = c_first < P.N;
                const int kc = S.t_kc[a];
                RowSum rp, rq;
                rp.Z = S.t_Z[2 * a]; rp.O = S.t_O[2 * a]; rp.cut = S.t_cut[2 * a];
                rq = rp;
                if (hq) { rq.Z = S.t_Z[2 * a + 1]; rq.O = S.t_O[2 * a + 1]; rq.cut = S.t_cut[2 * a + 1]; }
                if (OT) {
                    // ================= Algorithms 1-3 at node a =================================================
                    const int solver = P.solver;
                    const bool use_q = hq && solver != 0;            // Algorithm 1 ignores the drafts
                    // Algorithm 2 tests the first child only; Algorithm 3 with one child has rho = 1 and is the same
                    const bool one_test = use_q && (solver == 1 || kc == 1);
                    int acc = -1;
                    if (one_test) {
                        const double ep = S.t_cp[c_first], eq = S.t_cq[c_first];
                        const bool zero = !(ep > 0.0), one = !zero && !(eq > 0.0);
                        if (!zero && (one || (double)S.t_u[c_first] * eq * rp.Z < ep * rq.Z)) acc = c_first;
                    }
                    if (acc < 0) {
                        if (kc > 1) {
                            __syncwarp();
                            int seen = 0;
                            for (int c0 = a + 1; c0 < P.N && seen < kc; c0 += 32) {
                                const int c = c0 + lane;
                                const bool is = c < P.N && S.t_parent[c] == a;
                                const unsigned bal = __ballot_sync(0xffffffffu, is);
                                if (is) {
                                    const int pos = seen + __popc(bal & ((1u << lane) - 1u));
                                    W.child[pos] = c; W.cpm[pos] = S.t_cp[c]; W.cqm[pos] = S.t_cq[c]; W.cu[pos] = S.t_u[c];
                                }
                                seen += __popc(bal);
                            }
                            __syncwarp();
                        }
                        const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
                        nr.hq = use_q; nr.cut_p = rp.cut; nr.cut_q = rq.cut; nr.O_p = rp.O; nr.O_q = rq.O;
                        set_list_thresholds(nr, rp.Z, rq.Z);
                        int nl;
                        float zs_p, zs_q;
                        pass1<DT, NW, RC>(sl, nr, es, tid, R, L, nl, zs_p, zs_q);
                        double Z_q = rq.Z, kappa, tot_r, Zr_q = 0.0;
                        {
                            const double v[2] = {(double)zs_p + (lane < nl ? L.ep[lane] : 0.0), (double)zs_q + (lane < nl ? L.eq[lane] : 0.0)};
                            double tot[2], mine[2];
                            cluster_sum<NW, 2>(T, v, tot, mine);
                            kappa = tot[0]; tot_r = mine[0];
                            if (use_q && tot[1] > 0.0) { Z_q = tot[1]; Zr_q = mine[1]; }
                        }
                        if (*(volatile int *)&S.M.poison) status = SPEC_DEV_TIMEOUT;
                        else if (!(kappa > 0.0)) status = SPEC_DEV_NONFINITE;
                        const double invZq = use_q ? __drcp_rn(Z_q) : 0.0;
                        bool is_q = false;
                        if (!status && one_test) {
                            // the first child was rejected: Y ~ norm((p - q)+), one step of the recursion of verify.cuh
                            const double g = __ddiv_rn(Z_q, kappa);
                            const double v[1] = {step_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, g)};
                            double tot[1], mine[1];
                            cluster_sum<NW, 1>(T, v, tot, mine);
                            if (*(volatile int *)&S.M.poison) status = SPEC_DEV_TIMEOUT;
                            else if (tot[0] * invZq > RESIDUAL_FLOOR) { kappa = tot[0]; tot_r = mine[0]; }
                            else { is_q = true; kappa = Z_q; tot_r = Zr_q; }      // S = 0: p = q, drawn from q's row
                        } else if (!status && use_q) {
                            // ---- Algorithm 3 with k >= 2 children: the division factor (Appendix B) ----
                            const double ip = __drcp_rn(kappa), kd = (double)kc;
                            auto sweep2 = [&](auto f, double &t0, double &t1) {
                                double v[2], tot[2], mine[2];
                                reduce_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, f, v);
                                cluster_sum<NW, 2>(T, v, tot, mine);
                                t0 = tot[0]; t1 = tot[1];
                            };
                            double dummy, beta;
                            const double rho = spectr_root(kd, [&](double r) {
                                const double ipr = ip / r;
                                double bt;
                                sweep2(FnBeta{(float)ipr, (float)invZq, ipr, invZq}, bt, dummy);
                                return bt;
                            });
                            {
                                const double ipr = ip / rho;
                                sweep2(FnBeta{(float)ipr, (float)invZq, ipr, invZq}, beta, dummy);
                            }
                            const double pacc = 1.0 - pow(1.0 - beta, kd);
                            const double gamma = beta > 0.0 ? pacc / beta : 0.0;
                            // the children in list order, each against min(1, p(x) / (rho q(x)))
                            const double ux = lane < kc ? W.cpm[lane] : 0.0, eqx = lane < kc ? W.cqm[lane] : 0.0;
                            for (int j = 0; j < kc; ++j) {
                                const double Pp = __shfl_sync(0xffffffffu, ux, j) * ip;
                                const double Pq = __shfl_sync(0xffffffffu, eqx, j) * invZq;
                                double thr;
                                if (!(Pp > 0.0)) thr = 0.0;
                                else if (!(Pq > 0.0)) thr = 1.0;
                                else thr = fmin(1.0, (Pp / Pq) / rho);
                                if ((double)W.cu[j] < thr) {
                                    // the solver's output is the child's TOKEN: the walk moves to the first child,
                                    // in list order, that carries it (duplicates stay separate nodes)
                                    const int y = S.t_token[W.child[j]];
                                    for (int i = 0; i <= j && acc < 0; ++i)
                                        if (S.t_token[W.child[i]] == y) acc = W.child[i];
                                    break;
                                }
                            }
                            if (acc < 0) {
                                // all rejected: Y ~ norm((p - min(p / rho, q) gamma)+); p itself where that is empty
                                const double ib = beta < 1.0 ? 1.0 / (1.0 - beta) : 0.0;
                                double sres, sacc;
                                sweep2(FnSpecTrRes{(float)ip, (float)invZq, (float)(1.0 / rho), (float)gamma, (float)ib,
                                                   ip, invZq, 1.0 / rho, gamma, ib, kc}, sres, sacc);
                                if (sres > 0.0) {
                                    const double v[1] = {spectr_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, gamma, 1.0 / rho, kappa * invZq)};
                                    double tot[1], mine[1];
                                    cluster_sum<NW, 1>(T, v, tot, mine);
                                    kappa = tot[0]; tot_r = mine[0];
                                    if (!(kappa > 0.0)) status = SPEC_DEV_NONFINITE;
                                }
                            }
                            if (*(volatile int *)&S.M.poison) status = SPEC_DEV_TIMEOUT;
                        }
                        if (!status && acc < 0) {
                            // ---- the draw, and its token made known to every warp of the cluster ---------------------
                            const double target = (double)S.t_ub[a] * kappa;
                            double tau;
                            const int owner = pick_lane(lane < C ? tot_r : 0.0, target, tau);
                            double say = 0.0;             // token + 1 from the one thread that found it; -role on a failure
                            if (owner < 0) {
                                status = SPEC_DEV_NONFINITE;
                            } else {
                                if (owner == (int)rank) {
                                    const BonusFind bf = bonus_search<NW, RC>(T, sl, es, tid, R, L, nl, is_q, tau);
                                    if (bf.role == 1) say = (double)bf.token + 1.0;
                                    else if (bf.role >= 2) say = -(double)bf.role;
                                }
                                const double v[1] = {say};
                                double tot[1], mine[1];
                                cluster_sum<NW, 1>(T, v, tot, mine);
                                if (*(volatile int *)&S.M.poison || tot[0] == -3.0) status = SPEC_DEV_TIMEOUT;
                                else if (!(tot[0] >= 1.0)) status = SPEC_DEV_NONFINITE;
                                else {
                                    const int y = (int)(tot[0] - 1.0);
                                    // the first child, in list order, that carries the token
                                    if (hq) {
                                        if (kc == 1) { if (S.t_token[c_first] == y) acc = c_first; }
                                        else
                                            for (int j = 0; j < kc && acc < 0; ++j)
                                                if (S.t_token[W.child[j]] == y) acc = W.child[j];
                                    }
                                    if (acc < 0) {
                                        done = true;
                                        bonus = y;
                                        if (rank == 0 && warp == 0 && lane == 0) writer = true;
                                    }
                                }
                            }
                        }
                        if (status) {
                            done = true;
                            if (rank == 0 && warp == 0 && lane == 0) { writer = true; cur = -1; len = -1; }
                        }
                    }
                    if (acc >= 0 && !done) { cur = acc; ++len; }
                    continue;
                }
                // ---- first child: needs no residual -------------------------------------------------------------------
                int acc = -1;
                int j0 = 0;
                if (hq) {
                    // p(x) / q(x) = (e_p / Z_p) / (e_q / Z_q), written without a division
                    const double ep = S.t_cp[c_first], eq = S.t_cq[c_first];
                    const bool zero = !(ep > 0.0), one = !zero && !(eq > 0.0);
                    if (!zero && (one || (double)S.t_u[c_first] * eq * rp.Z < ep * rq.Z)) acc = c_first;
                    j0 = 1;
                }
                if (acc < 0) {
                    // ---- the node comes on chip: e = 2^(z s - O) of both rows ----------------------------------------
                    // the warp's list of the node's children, in index order
                    if (kc > 1) {
                        __syncwarp();
                        int seen = 0;
                        for (int c0 = a + 1; c0 < P.N && seen < kc; c0 += 32) {
                            const int c = c0 + lane;
                            const bool is = c < P.N && S.t_parent[c] == a;
                            const unsigned bal = __ballot_sync(0xffffffffu, is);
                            if (is) {
                                const int pos = seen + __popc(bal & ((1u << lane) - 1u));
                                W.child[pos] = c; W.cpm[pos] = S.t_cp[c]; W.cqm[pos] = S.t_cq[c]; W.cu[pos] = S.t_u[c];
                            }
                            seen += __popc(bal);
                        }
                        __syncwarp();
                    }
                    const Slice sl = make_slice<DT>(P.zp, P.zq, (long long)b * P.seq_stride + (long long)a * P.node_stride, P.V, C, rank);
                    nr.hq = hq; nr.cut_p = rp.cut; nr.cut_q = rq.cut; nr.O_p = rp.O; nr.O_q = rq.O;
                    set_list_thresholds(nr, rp.Z, rq.Z);
                    int nl;
                    float zs_p, zs_q;
                    pass1<DT, NW, RC>(sl, nr, es, tid, R, L, nl, zs_p, zs_q);
                    // ---- the rows' totals from what is resident: the normalisers, and each rank's share of u_0 = e_p
                    double Z_q = rq.Z, kappa, tot_r, Zr_q = 0.0;
                    {
                        const double v[2] = {(double)zs_p + (lane < nl ? L.ep[lane] : 0.0), (double)zs_q + (lane < nl ? L.eq[lane] : 0.0)};
                        double tot[2], mine[2];
                        cluster_sum<NW, 2>(T, v, tot, mine);
                        kappa = tot[0]; tot_r = mine[0];
                        if (hq && tot[1] > 0.0) { Z_q = tot[1]; Zr_q = mine[1]; }
                    }
                    if (*(volatile int *)&S.M.poison) status = SPEC_DEV_TIMEOUT;
                    else if (!(kappa > 0.0)) status = SPEC_DEV_NONFINITE;
                    const double invZq = hq ? __drcp_rn(Z_q) : 0.0;
                    // ---- the recursion of verify.cuh, step by step (the first child, if any, is already rejected);
                    // lane j < kc follows child j's token in fp64
                    double ux = 0.0, eqx = 0.0;
                    if (lane < kc) {
                        ux = kc > 1 ? W.cpm[lane] : S.t_cp[c_first];
                        eqx = kc > 1 ? W.cqm[lane] : S.t_cq[c_first];
                    }
                    bool is_q = false;
                    for (int j = 0; j < kc && !status; ++j) {
                        if (j >= j0) {
                            // child j from the current state
                            const double uxj = __shfl_sync(0xffffffffu, ux, j), eqj = __shfl_sync(0xffffffffu, eqx, j);
                            const double Pq = eqj * invZq;
                            const double Pp = is_q ? Pq : uxj / kappa;
                            double thr;
                            if (!(Pp > 0.0)) thr = 0.0;
                            else if (!(Pq > 0.0)) thr = 1.0;
                            else thr = fmin(1.0, Pp / Pq);
                            if ((double)W.cu[j] < thr) { acc = W.child[j]; break; }
                        }
                        if (is_q) continue;
                        // the step after rejecting child j: u <- (g u - e_q)+ , g = Z_q / kappa
                        const double g = __ddiv_rn(Z_q, kappa);
                        const double v[1] = {step_sweep<NW, RC>(es, sl.nu, tid, R, L, nl, g)};
                        double tot[1], mine[1];
                        cluster_sum<NW, 1>(T, v, tot, mine);
                        if (*(volatile int *)&S.M.poison) { status = SPEC_DEV_TIMEOUT; break; }
                        ux = fmax(fma(g, ux, -eqx), 0.0);
                        if (tot[0] * invZq > RESIDUAL_FLOOR) { kappa = tot[0]; tot_r = mine[0]; }
                        else { is_q = true; kappa = Z_q; tot_r = Zr_q; }      // S = 0: the state equals q
                    }
                    if (status) { done = true; if (rank == 0 && warp == 0 && lane == 0) { writer = true; cur = -1; len = -1; } break; }
                    if (acc < 0) {
                        // ---- stop here: the bonus token from the final state ----------------------------------------------
                        done = true;
                        const double target = (double)S.t_ub[a] * kappa;
                        double tau;
                        const int owner = pick_lane(lane < C ? tot_r : 0.0, target, tau);
                        if (owner < 0) {
                            status = SPEC_DEV_NONFINITE;
                            if (rank == 0 && warp == 0 && lane == 0) { writer = true; cur = -1; len = -1; }
                        } else if (owner == (int)rank) {
                            const BonusFind bf = bonus_search<NW, RC>(T, sl, es, tid, R, L, nl, is_q, tau);
                            if (bf.role == 1) {
                                bonus = bf.token;
                                writer = true;
                            } else if (bf.role >= 2) {
                                status = bf.role == 3 ? SPEC_DEV_TIMEOUT : SPEC_DEV_NONFINITE;
                                writer = true; cur = -1; len = -1;
                            }
                        }
                    }
                }
                if (acc >= 0) { cur = acc; ++len; continue; }
            }

            // ---- outputs of the sequence: by the warp that holds the writer -----------------------------------------------
            __syncwarp();
            const unsigned wm = __ballot_sync(0xffffffffu, writer);
            if (wm) {
                const int src = __ffs(wm) - 1;
                const int st = __shfl_sync(0xffffffffu, status, src);
                const int accn = st ? -1 : __shfl_sync(0xffffffffu, cur, src), ln = st ? -1 : __shfl_sync(0xffffffffu, len, src);
                const int bn = st ? -1 : __shfl_sync(0xffffffffu, bonus, src);
                if (lane == 0) {
                    P.out.accepted_node[b] = accn;
                    P.out.accept_len[b] = ln;
                    P.out.bonus_token[b] = bn;
                    P.out.status[b] = st;
                }
                int *ot = P.out.out_tokens + (long long)b * P.N;
                for (int i0 = 0; i0 < P.N; i0 += 32) {
                    const int i = i0 + lane;
                    int v = i == ln ? bn : -1;
                    int x = accn;
                    for (int d = ln - 1; d >= 0; --d) {          // the path, from its end
                        if (d == i) v = S.t_token[x];
                        x = S.t_parent[x];
                    }
                    if (i < P.N) ot[i] = v;
                }
            }
        }
    }
    __syncthreads();
    if (C > 1) cluster_sync_all();       // nobody leaves while a peer may still write to its shared memory
}

}  // namespace specv
