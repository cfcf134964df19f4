// libspecverify: batched draft-tree verification for sm_100a -- host side of the C ABI.
//
// Kernels: stream.cuh (row statistics, the one pass over HBM), trunc.cuh (the same for top-k / top-p
// rows), walk.cuh (SpecInfer along the accepted path), nodes.cuh (every node: Traversal Verification,
// diagnostic outputs, analysis), rowops.cuh (materialised row distributions, stand-alone inverse CDF), and the
// residual kernel below.  This file validates
// arguments, chooses the launch plan and enqueues; it never allocates and, except for the
// host-buffer entry point, never synchronises.
#include <algorithm>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "analysis.cuh"
#include "common.cuh"
#include "cut.cuh"
#include "nodes.cuh"
#include "rowops.cuh"
#include "trunc.cuh"
#include "specverify.h"
#include "verify.cuh"
#include "walk.cuh"

namespace specv {
namespace {

// ------------------------------------------------------------------------------------------------
// residual output: the law the bonus was drawn from, for the accepted node of each sequence
// ------------------------------------------------------------------------------------------------
struct RParams {
    int B, N, V, dtype;
    const void *zp, *zq;
    long long seq_stride, node_stride;
    float T;
    const float *T_seq;
    const NodeRec *rec;
    const double *gseq;        // [B*N][KMAX] step coefficients of every node
    const int *accepted;
    float *residual;
};

// The accepted node's final law, token by token: the recursion of verify.cuh replayed in fp64 with the
// node's recorded coefficients, u <- (g_j u - e_q)+ from u = e_p, divided by the recorded total.
__global__ void spec_residual_kernel(const RParams P)
{
    grid_dependency_wait();
    const int b = blockIdx.y;
    const int acc = P.accepted[b];
    float *out = P.residual + (long long)b * P.V;
    if (acc < 0) {
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < P.V; t += gridDim.x * blockDim.x) out[t] = 0.f;
        return;
    }
    const NodeRec R = P.rec[(long long)b * P.N + acc];
    const double *g = P.gseq + ((long long)b * P.N + acc) * KMAX;
    const double s = 1.4426950408889634 / (double)(P.T_seq ? P.T_seq[b] : P.T);
    const long long row = (long long)b * P.seq_stride + (long long)acc * P.node_stride;
    const int nsteps = R.nsteps;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < P.V; t += gridDim.x * blockDim.x) {
        double u = 0.0;
        if (nsteps == STATE_IS_Q) {
            const float zq = load_logit(P.zq, P.dtype, row + t);
            if (zq >= R.cut_q) u = exp2((double)zq * s - R.O_q);
        } else {
            const float zp = load_logit(P.zp, P.dtype, row + t);
            if (zp >= R.cut_p) u = exp2((double)zp * s - R.O_p);
            if (nsteps > 0) {
                const float zq = load_logit(P.zq, P.dtype, row + t);
                const double eq = zq >= R.cut_q ? exp2((double)zq * s - R.O_q) : 0.0;
                for (int j = 0; j < nsteps; ++j) u = fmax(fma(g[j], u, -eq), 0.0);
            }
        }
        out[t] = (float)(R.kappa > 0.0 ? u / R.kappa : 0.0);
    }
}

// ------------------------------------------------------------------------------------------------
// launch plans
// ------------------------------------------------------------------------------------------------
struct VPlan {
    int C, slice_len, off_es, smem;
};

constexpr int SMEM_1CTA = 227 * 1024;          // opt-in limit per CTA
constexpr int SMEM_2CTA = 113 * 1024;          // so that two CTAs share an SM

inline int up(int x, int m) { return (x + m - 1) / m * m; }

// Launch shape of the cluster kernels (walk, tree) with NW consumer warps of RC register chunks per thread: the smallest
// cluster in which a thread has at most `want` chunks, those beyond RC in shared memory; eight CTAs with as many as fit
// before sixteen (a non-portable size, and fewer clusters fit the chip).  Dynamic shared memory: header | resident e
// of the chunks that do not fit in registers.
bool make_vplan(int V, int NW, int RC, int budget, int want, int hdr_bytes, VPlan *p)
{
    const int chunk_bytes = NW * 32 * 64, off_es = up(hdr_bytes, 128);
    const int most = RC + (budget - off_es) / chunk_bytes, cap = most < CHMAX ? most : CHMAX;
    const int units = (int)(((long long)V + 14) / 8);          // chunks of a row, wherever it starts
    for (int C = 1; C <= CMAX; C <<= 1) {
        const int per = (units + C - 1) / C, nch = (per + NW * 32 - 1) / (NW * 32);
        if (nch > (C < 8 ? (want < cap ? want : cap) : cap)) continue;
        p->C = C; p->slice_len = per * 8; p->off_es = off_es;
        p->smem = off_es + (nch > RC ? nch - RC : 0) * chunk_bytes;
        return true;
    }
    return false;
}
// The kernels keep a node's e in shared memory and go through it in loops: their code runs a few times per sequence, and its first
// run costs about 80 cycles per 128 bytes of instructions (unrolled over eight chunks in registers, a first pass took 7000
// cycles and the analysis' sweeps ten times that).  Registers as well (big: RC = 8) only for vocabularies beyond
// what the shared memory of 16 CTAs holds; the walk of a batch that fills the chip puts two CTAs on an SM (RC = 4).
bool one_cta_plan(int V, int NW, int hdr_bytes, VPlan *p, bool *big)
{
    *big = false;
    if (make_vplan(V, NW, 0, SMEM_1CTA, 9, hdr_bytes, p)) return true;
    *big = true;
    return make_vplan(V, NW, 8, SMEM_1CTA, 9, hdr_bytes, p);
}
bool two_cta_plan(int V, int hdr_bytes, VPlan *p) { return make_vplan(V, 8, 4, SMEM_2CTA, 8, hdr_bytes, p); }

struct RowPlan {
    int C, SL, smem;
};
constexpr int ROW_SMEM_BUDGET = 227 * 1024 - (int)sizeof(rowops::Shared) - 1024;

// `rows` rows of fp32 values, each in the shared memory of a cluster: two CTAs per SM where eight CTAs are enough for that, but one
// where all CTAs of clusters of four, and not of clusters of eight, have an SM to themselves (19 rows of 128256: 16.5 and 18.5 us; one CTA
// against two does not pay: 76 rows of 32000 17.6 and 15.3).
bool make_row_plan(int V, long long rows, int sms, RowPlan *p)
{
    const auto plan = [&](int budget, int most) {
        for (int C = 1; C <= most; C <<= 1) {
            const long long sl = (((long long)V + C - 1) / C + 63) / 64 * 64, need = sl * 4;
            if (need > budget) continue;
            *p = RowPlan{C, (int)sl, (int)need};
            return true;
        }
        return false;
    };
    if (!plan(ROW_SMEM_BUDGET / 2 - 4096, 8)) return plan(ROW_SMEM_BUDGET, rowops::CMAX);
    const RowPlan two = *p;
    if (two.C == 8 && rows * two.C > sms && plan(ROW_SMEM_BUDGET, rowops::CMAX) && rows * p->C > sms) *p = two;
    return true;
}

int check_in(const SpecIn *in, bool need_tree)
{
    if (!in) return SPEC_ERR_NULL;
    if (in->B <= 0 || in->N <= 0 || in->V <= 0 || in->N > SPEC_MAX_NODES) return SPEC_ERR_SHAPE;
    if ((long long)in->B * in->N > (1ll << 24)) return SPEC_ERR_SHAPE;
    if (in->logits_dtype != SPEC_F32 && in->logits_dtype != SPEC_BF16) return SPEC_ERR_DTYPE;
    if (in->node_stride < in->V || in->seq_stride < 0) return SPEC_ERR_SHAPE;
    if (in->topo_seq_stride != 0 && in->topo_seq_stride < in->N) return SPEC_ERR_SHAPE;
    if (!(in->temperature > 0.f) || !(in->temperature < 3.0e38f)) {
        if (!in->temperature_per_seq) return SPEC_ERR_PARAM;
    }
    if (in->top_k < 0 || !(in->top_p > 0.f) || in->top_p > 1.f) return SPEC_ERR_PARAM;
    if (need_tree) {
        if (!in->target_logits || !in->draft_logits || !in->parent || !in->token || !in->u_accept || !in->u_bonus)
            return SPEC_ERR_NULL;
    }
    return SPEC_OK;
}

inline int64_t up256(int64_t x) { return (x + 255) / 256 * 256; }

// workspace layout: node records | published weights + arrival counters (cleared per call) | kept counts
struct WsLayout {
    int64_t rec, pub, fin, done, ticket, chain, kept, stat, gseq, total;
};
WsLayout ws_layout(const SpecIn *in)
{
    WsLayout L;
    const int64_t nodes = (int64_t)in->B * in->N;
    int64_t o = 0;
    L.rec = o; o += up256(nodes * (int64_t)sizeof(NodeRec));
    // set per call by the statistics kernels (NodeInit)
    L.pub = o; o += nodes * 8;
    L.fin = o; o += (int64_t)in->B * 4;
    L.done = o; o += (int64_t)in->B * 4;
    L.ticket = o; o += 4;
    o = up256(o);
    L.chain = o; o += up256(nodes * (int64_t)sizeof(ChainRec));
    L.kept = o; o += up256(nodes * 8);
    L.stat = o; o += up256(nodes * 2 * (int64_t)sizeof(RowPart));
    L.gseq = o; o += up256(nodes * KMAX * 8);       // step coefficients of every node
    L.total = o;
    return L;
}

// kernels enqueued by the library in this process (benchmarks report it)
std::atomic<long long> g_kernel_launches{0};

template <typename K>
int launch_clustered(K kernel, int ctas, int C, int threads, int smem, cudaStream_t st, void *params_ptr,
                     bool dependent = false)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    // (C = 0: a kernel that knows no clusters; the recursion kernel uses cluster instructions in a cluster of one as well)
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (C > 0) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = C;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    // dependent: the kernel waits by itself (grid_dependency_wait) for the kernel before it in the stream, so
    // its CTAs may be placed, and run their set-up, while that kernel's last CTAs still work
    if (dependent) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    void *args[1] = {params_ptr};
    cudaError_t e = cudaLaunchKernelExC(&cfg, (const void *)kernel, args);
    if (e != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
    return SPEC_OK;
}

// a kernel without clusters or dynamic shared memory that waits by itself for the kernel before it
template <typename K, typename A>
int launch_after(K kernel, dim3 grid, int threads, cudaStream_t st, A *params)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[1] = {params};
    if (cudaLaunchKernelExC(&cfg, (const void *)kernel, args) != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
    return SPEC_OK;
}

std::mutex g_cache_mutex;

int sm_count()
{
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 148; }
    if (!cached[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) { cudaGetLastError(); n = 148; }
        cached[dev] = n;
    }
    return cached[dev];
}

// Kernel attributes are set once per (device, kernel): the largest dynamic shared memory asked for
// so far and the permission for clusters above 8 CTAs.  Later calls only launch.
template <typename K>
int prepare_kernel(K kernel, int C, int smem, bool overlap = false)
{
    struct Entry { const void *k; int dev, smem, big; };
    static Entry cache[256];
    static int used = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    std::lock_guard<std::mutex> lock(g_cache_mutex);
    Entry *ent = nullptr;
    for (int i = 0; i < used; ++i)
        if (cache[i].k == (const void *)kernel && cache[i].dev == dev) ent = &cache[i];
    if (!ent) {
        if (used >= 256) return SPEC_ERR_CUDA;
        ent = &cache[used++];
        *ent = Entry{(const void *)kernel, dev, -1, 0};
        // overlap: as much of an SM's L1 as can be is shared memory, so that CTAs of the kernels that run at the same time
        // find room beside this one
        if (overlap && cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            cudaGetLastError();
    }
    if (smem > ent->smem) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_CUDA; }
        ent->smem = smem;
    }
    if (C > 8 && !ent->big) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_UNSUPPORTED; }
        ent->big = 1;
    }
    return SPEC_OK;
}

// number of clusters of this shape that can be resident at once (cached per device / kernel / shape)
template <typename K>
int resident_clusters(K kernel, int C, int threads, int smem)
{
    struct Entry { const void *k; int dev, C, smem, n; };
    static Entry cache[256];
    static int used = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    std::lock_guard<std::mutex> lock(g_cache_mutex);
    for (int i = 0; i < used; ++i)
        if (cache[i].k == (const void *)kernel && cache[i].dev == dev && cache[i].C == C && cache[i].smem == smem)
            return cache[i].n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(C * 1024), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, (const void *)kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    if (used < 256) cache[used++] = Entry{(const void *)kernel, dev, C, smem, n};
    return n;
}

// nodes with several children (AN: with any): a cluster each
template <int DT, int RC, bool AN>
int launch_branch(VPlan pl, NParams &np, cudaStream_t st)
{
    // An SM's shared memory comes in configurations of ..., 132, 164, 196 and 228 KB (1 KB a CTA is the system's).  A CTA that nearly fills
    // the 164 KB one leaves the CTAs of the kernels beside it no place until it is done; asking for more than that, it runs in a larger one.
    // Traversal, V = 262144 (164 KB), us: B = 16 218 and 204, B = 8 134 and 128.
    if (pl.smem > 160 * 1024 && pl.smem <= 163 * 1024) pl.smem = 163 * 1024 + 64;
    auto kernel = spec_recursion_kernel<DT, 7, RC, AN>;
    const int rc = prepare_kernel(kernel, pl.C, pl.smem, true);
    if (rc) return rc;
    int nc = resident_clusters(kernel, pl.C, 256, pl.smem);
    if (nc <= 0) return SPEC_ERR_UNSUPPORTED;
    const long long items = (long long)np.v.B * np.v.N;
    if (nc > items) nc = (int)items;
    np.v.C = pl.C; np.v.off_es = pl.off_es;
    return launch_clustered(kernel, nc * pl.C, pl.C, 256, pl.smem, st, &np, np.v.mode == MODE_TRAVERSAL);
}
template <int DT, int RC>
int launch_finish(const VPlan &pl, NParams &np, cudaStream_t st)
{
    auto kernel = spec_finish_kernel<DT, 8, RC>;
    const int rc = prepare_kernel(kernel, pl.C, pl.smem, true);
    if (rc) return rc;
    int nc = resident_clusters(kernel, pl.C, 256, pl.smem);
    if (nc <= 0) return SPEC_ERR_UNSUPPORTED;
    if (nc > np.v.B) nc = np.v.B;
    np.v.C = pl.C; np.v.off_es = pl.off_es;
    return launch_clustered(kernel, nc * pl.C, pl.C, 256, pl.smem, st, &np, true);
}

// row statistics (cut, reference, normaliser) of every row the verifiers read, or of every row of `zp` when no
// tree is given, under top-k / top-p
int launch_trunc(const SpecIn *in, const void *zp, const void *zq, const int *parent, unsigned char *ws,
                 const WsLayout &L, const stream::NodeInit &init, cudaStream_t st)
{
    trunc::RParams rp = {};
    rp.B = in->B; rp.N = in->N; rp.V = in->V; rp.top_k = in->top_k; rp.top_p = in->top_p;
    rp.zp = zp; rp.zq = zq; rp.seq_stride = in->seq_stride; rp.node_stride = in->node_stride;
    rp.topo_stride = in->topo_seq_stride; rp.parent = parent; rp.T = in->temperature; rp.T_seq = in->temperature_per_seq;
    rp.part = (RowPart *)(ws + L.stat); rp.init = init;
    rp.kept = parent ? nullptr : (int *)(ws + L.kept);
    const bool bf = in->logits_dtype == SPEC_BF16;
    const long long items = 2ll * in->B * in->N;
    const long long want = (long long)sm_count() * (bf ? trunc::CTAS<SPEC_BF16> : trunc::CTAS<SPEC_F32>);
    const unsigned grid = (unsigned)(items < want ? items : want);
    const bool total = in->top_p < 1.f && !(in->top_k > 0 && in->top_k < in->V);
    auto go = [&](auto kernel, int smem) {
        const int rc = prepare_kernel(kernel, 1, smem);
        if (rc) return rc;
        return launch_clustered(kernel, (int)grid, 0, trunc::NT, smem, st, &rp, true);
    };
    if (bf)
        return total ? go(trunc::spec_row_trunc_kernel<SPEC_BF16, true>, trunc::Layout<SPEC_BF16>::BYTES)
                     : go(trunc::spec_row_trunc_kernel<SPEC_BF16, false>, trunc::Layout<SPEC_BF16>::BYTES);
    return total ? go(trunc::spec_row_trunc_kernel<SPEC_F32, true>, trunc::Layout<SPEC_F32>::BYTES)
                 : go(trunc::spec_row_trunc_kernel<SPEC_F32, false>, trunc::Layout<SPEC_F32>::BYTES);
}

// SpecInfer without diagnostic outputs: row statistics of every row, then one walk per sequence
template <int DT, int NW, int RC, int MINB, bool OT>
int launch_walk(const VPlan &pl, WParams &wp, cudaStream_t st)
{
    auto kernel = spec_walk_kernel<DT, NW, RC, MINB, OT>;
    int rc = prepare_kernel(kernel, pl.C, pl.smem);
    if (rc) return rc;
    const int threads = NW * 32;
    int nc = resident_clusters(kernel, pl.C, threads, pl.smem);
    if (nc <= 0) return SPEC_ERR_UNSUPPORTED;
    if (nc > wp.B) nc = wp.B;
    return launch_clustered(kernel, nc * pl.C, pl.C, threads, pl.smem, st, &wp, true);
}

// Statistics of every row the verifiers read (reference, normaliser, cut), and the entropy features when asked for.
int row_statistics(const SpecIn *in, const SpecOut *out, unsigned char *w, const WsLayout &L, bool trunc, cudaStream_t st,
                   bool init_nodes = false)
{
    stream::NodeInit init = {};
    if (init_nodes)
        init = {(unsigned long long *)(w + L.pub), (unsigned int *)(w + L.done), (int *)(w + L.fin),
                (unsigned int *)(w + L.ticket), (ulonglong2 *)(w + L.chain)};
    const bool feat = out->node_features != nullptr;
    const auto features = [&]() {
        if (!feat) return (int)SPEC_OK;
        stream::FParams fp = {2ll * in->B * in->N, (const RowPart *)(w + L.stat), out->node_features};
        return launch_after(stream::spec_features_kernel, dim3((unsigned)((fp.rows + 127) / 128)), 128, st, &fp);
    };
    if (trunc) {
        const int rc = launch_trunc(in, in->target_logits, in->draft_logits, in->parent, w, L, init, st);
        return rc ? rc : features();
    }
    // rows are split into parts only when there are fewer rows than resident CTAs
    const long long rows2 = 2ll * in->B * in->N;
    const int slices_row = (in->V + stream::SLICE - 1) / stream::SLICE;
    int NSL = 1;
    while (NSL < stream::MAX_PARTS && NSL < slices_row && rows2 * NSL < 2 * sm_count()) NSL *= 2;
    stream::SParams sp = {};
    sp.B = in->B; sp.N = in->N; sp.V = in->V; sp.NSL = NSL;
    sp.zp = in->target_logits; sp.zq = in->draft_logits;
    sp.seq_stride = in->seq_stride; sp.node_stride = in->node_stride; sp.topo_stride = in->topo_seq_stride;
    sp.parent = in->parent; sp.T = in->temperature; sp.T_seq = in->temperature_per_seq;
    sp.part = (RowPart *)(w + L.stat); sp.init = init;
    // one CTA per item: those of unread rows retire at once
    const long long items = rows2 * NSL;
    const int grid = (int)(items < (1ll << 20) ? items : (1ll << 20));
    const auto go = [&](auto kernel, int smem) {
        int rc = prepare_kernel(kernel, 1, smem);
        if (!rc) rc = launch_clustered(kernel, grid, NSL > 1 ? NSL : 0, stream::NT, smem, st, &sp, true);
        return rc ? rc : features();
    };
    if (in->logits_dtype == SPEC_BF16)
        return feat ? go(stream::spec_row_partial_kernel<SPEC_BF16, true>, stream::Ring<SPEC_BF16>::BYTES)
                    : go(stream::spec_row_partial_kernel<SPEC_BF16, false>, stream::Ring<SPEC_BF16>::BYTES);
    return feat ? go(stream::spec_row_partial_kernel<SPEC_F32, true>, stream::Ring<SPEC_F32>::BYTES)
                : go(stream::spec_row_partial_kernel<SPEC_F32, false>, stream::Ring<SPEC_F32>::BYTES);
}

// The launch shape of the walk.
// The walk keeps one cluster per sequence busy.  While all of them fit on the chip with one CTA per SM, a CTA has an SM to itself.
// Larger batches run in rounds that way, and two CTAs on an SM (half of the registers, the first chunks in them) pay only
// where a thread has few chunks of 16-bit logits and the clusters are no larger for it.  Calls with three nodes per path, us,
// two CTAs against one: V = 50257 (7 chunks) B = 40 33.5 / 36.6, V = 100352 (7) B = 80 88 / 99, 128 127 / 148; but V = 128256 (8) B = 32
// 57.7 / 53.0, 64 102 / 91, 128 180 / 167, V = 151936 (10) B = 32 73 / 62, V = 262144 B = 64 195 / 175, V = 65536 (cluster of 8 against
// 4) B = 80 73 / 64, and fp32 V = 50257 B = 90 124 / 102.  With 8 chunks (up to V = 131072 on clusters of 8) also for large batches under
// top-k, which leaves few tokens to evaluate: V = 114688 / 120064 / 128256 / 131072, two against one, B = 56 115 114 / 134 128 / 134 128 / 124
// 122, B = 64 130 131 / 138 141 / 141 146 / 128 142, B = 96 181 181 / 187 197 / 191 199 / 182 196, B = 128 233 237 / 236 249 / 243 256 / 240
// 248.  Under top-p alone neither is better throughout (T 0.6, 0.95: B = 80 225 221 / 233 236 / 242 222 / 240 226, B = 96 246 251 / 268 267 / 269
// 270 / 276 271, B = 128 348 329 / 334 352 / 371 364 / 376 362): two from four CTAs per SM on, up to slices of 16384.
struct WalkPlan {
    VPlan pl;
    bool two, big;       // two CTAs on an SM; chunks in registers as well
};
bool walk_plan(int V, int dtype, long long B, bool top_k, bool top_p, int sms, WalkPlan *w)
{
    VPlan one;
    if (!one_cta_plan(V, 8, (int)sizeof(WHdr), &one, &w->big)) return false;
    w->two = B * one.C > sms && dtype == SPEC_BF16 && two_cta_plan(V, (int)sizeof(WHdr), &w->pl) && w->pl.C == one.C &&
             (w->pl.slice_len <= 7 * 256 * 8 || (top_k && 5 * B * one.C >= 17ll * sms && V <= 8 * 256 * 8 * one.C) ||
              (top_p && B * one.C >= 4ll * sms && w->pl.slice_len <= 8 * 256 * 8));
    if (!w->two) w->pl = one;
    return true;
}

// solver: -1 SpecInfer, otherwise the OTLP solver of spec_verify_otlp
int verify_walk(const SpecIn *in, const SpecOut *out, unsigned char *w, const WsLayout &L, bool trunc, cudaStream_t st, int solver = -1)
{
    WalkPlan plan;
    if (!walk_plan(in->V, in->logits_dtype, in->B, in->top_k > 0 && in->top_k < in->V, in->top_p < 1.f, sm_count(), &plan)) return SPEC_ERR_UNSUPPORTED;
    const VPlan &pl = plan.pl;
    int rc = row_statistics(in, out, w, L, trunc, st);
    if (rc) return rc;
    WParams wp = {};
    wp.B = in->B; wp.N = in->N; wp.V = in->V; wp.C = pl.C; wp.off_es = pl.off_es;
    wp.zp = in->target_logits; wp.zq = in->draft_logits;
    wp.seq_stride = in->seq_stride; wp.node_stride = in->node_stride; wp.topo_stride = in->topo_seq_stride;
    wp.parent = in->parent; wp.token = in->token; wp.T = in->temperature; wp.T_seq = in->temperature_per_seq;
    wp.part = (RowPart *)(w + L.stat); wp.u_accept = in->u_accept; wp.u_bonus = in->u_bonus; wp.out = *out;
    wp.solver = solver;
    const bool bf = in->logits_dtype == SPEC_BF16;
    auto go = [&](auto ot) {
        constexpr bool OT = decltype(ot)::value;
        if (plan.two) return launch_walk<SPEC_BF16, 8, 4, 2, OT>(pl, wp, st);
        if (plan.big) return bf ? launch_walk<SPEC_BF16, 8, 8, 1, OT>(pl, wp, st) : launch_walk<SPEC_F32, 8, 8, 1, OT>(pl, wp, st);
        return bf ? launch_walk<SPEC_BF16, 8, 0, 1, OT>(pl, wp, st) : launch_walk<SPEC_F32, 8, 0, 1, OT>(pl, wp, st);
    };
    return solver >= 0 ? go(std::true_type{}) : go(std::false_type{});
}

void fill_params(const SpecIn *in, const SpecOut *out, unsigned char *w, const WsLayout &L, int mode, NParams &tp)
{
    VParams &vp = tp.v;
    vp.B = in->B; vp.N = in->N; vp.V = in->V; vp.mode = mode;
    vp.all_thr = (out->node_thr != nullptr || out->margin != nullptr) ? 1 : 0;
    // Whether the finish kernel, a cluster per sequence for 15 us, lets the first kernel of the next call in while it runs (that kernel then
    // waits for its end; it helps where calls of this library follow each other, and changes nothing for any other kernel that comes
    // next): where such a call's rows fill the chip (Traversal B = 8 92 -> 86 us, V = 262144 B = 16 219 -> 201).  Fewer CTAs
    // would crowd onto the SMs that are free at that moment and leave the others idle, and so would the selection's
    // (wide nuclei, B = 8: 121 -> 127); nothing is gained after a walk (SpecInfer B = 8; top-k, B = 128: 708 -> 741).
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    vp.early = !trunc && 2ll * in->B * in->N >= 2ll * sm_count();
    vp.zp = in->target_logits; vp.zq = in->draft_logits;
    vp.seq_stride = in->seq_stride; vp.node_stride = in->node_stride; vp.topo_stride = in->topo_seq_stride;
    vp.parent = in->parent; vp.token = in->token;
    vp.T = in->temperature; vp.T_seq = in->temperature_per_seq;
    vp.u_accept = in->u_accept; vp.u_bonus = in->u_bonus;
    vp.rec = (NodeRec *)(w + L.rec);
    vp.w_pub = (unsigned long long *)(w + L.pub);
    vp.done = (unsigned int *)(w + L.done);
    vp.fin = (int *)(w + L.fin);
    vp.chain = (ChainRec *)(w + L.chain);
    vp.out = *out;
    tp.part = (const RowPart *)(w + L.stat);
    tp.gseq = (double *)(w + L.gseq);
    tp.ticket = (unsigned int *)(w + L.ticket);
}

// every node of every sequence, on top of the row statistics
int launch_nodes(const SpecIn *in, NParams &np, bool analysis, cudaStream_t st)
{
    const bool bf = in->logits_dtype == SPEC_BF16;
    VPlan br, fi;
    bool big, bigf;
    if (!one_cta_plan(in->V, 7, (int)sizeof(BHdr), &br, &big) || !one_cta_plan(in->V, 8, (int)sizeof(FHdr), &fi, &bigf)) return SPEC_ERR_UNSUPPORTED;
    const long long nodes = (long long)in->B * in->N;
    const int smem = bf ? SUMS_RING<SPEC_BF16> : SUMS_RING<SPEC_F32>;
    int rc;
    if (np.v.mode == MODE_TRAVERSAL) {
        // A CTA per SM, so that the recursion's clusters, which wait for its results, find their places beside it; as many as fit (3)
        // where there are the nodes for them.
        const int ctas = nodes < 2 * sm_count() ? sm_count() : 3 * sm_count();
        const auto go = [&](auto kernel) {
            const int e = prepare_kernel(kernel, 1, smem, true);
            return e ? e : launch_clustered(kernel, ctas, 1, 256, smem, st, &np, true);
        };
        rc = bf ? go(spec_ratio_kernel<SPEC_BF16>) : go(spec_ratio_kernel<SPEC_F32>);
        if (rc) return rc;
    }
    const auto branch = [&](auto an) {
        constexpr bool AN = decltype(an)::value;
        if (big) return bf ? launch_branch<SPEC_BF16, 8, AN>(br, np, st) : launch_branch<SPEC_F32, 8, AN>(br, np, st);
        return bf ? launch_branch<SPEC_BF16, 0, AN>(br, np, st) : launch_branch<SPEC_F32, 0, AN>(br, np, st);
    };
    rc = analysis ? branch(std::true_type{}) : branch(std::false_type{});
    if (rc) return rc;
    {
        // nodes with one child: more CTAs per node while few waves hold them all (with one CTA a node its passes, not their sum, are the
        // latency: traversal, batch 8, V = 128256, 152 nodes: 131 us with 1, 109 with 2, 94 with 4)
        int C = 1, bytes = smem;
        while (C < 8 && nodes * C * 2 <= 8 * sm_count() && in->V >= C * 8192) C <<= 1;
        if (analysis) {
            // The analysis' passes are arithmetic, and left alone three CTAs share an SM while others idle: with few nodes a CTA asks for so
            // much shared memory that they spread, and clusters of 16 are taken where each of their CTAs finds an SM and 24 KB of the row.
            // Paths of six nodes, us, packed and spread: fp32 V = 262144 B = 1 123 and 64 (78 in clusters of 8), B = 2 129 and 78, B = 4 (two a SM) 136 and 110,
            // V = 128256 B = 2 89 and 62, bf16 V = 262144 B = 1 70 and 57, V = 128256 B = 4 68 and 61; from three a SM on, packed is as it was
            // (spread all the same, B = 8: 76 and 85).  Clusters of 16 for smaller rows: bf16 V = 128256 B = 1 46 and 48.
            if (C == 8 && nodes * 16 <= sm_count() && (long long)in->V * (bf ? 2 : 4) >= 16 * 24 * 1024) C = 16;
            const long long per_sm = (nodes * C + sm_count() - 1) / sm_count();
            // (with 14 KB of its own, one or two of them fit the 228 KB of an SM)
            if (per_sm <= 2) bytes = per_sm == 1 ? 104 * 1024 : 66 * 1024;
        }
        np.v.C = C;
        const auto go = [&](auto kernel) {
            const int e = prepare_kernel(kernel, C, bytes, true);
            return e ? e : launch_clustered(kernel, (int)nodes * C, C, 256, bytes, st, &np, true);
        };
        if (analysis) return bf ? go(spec_single_analysis_kernel<SPEC_BF16>) : go(spec_single_analysis_kernel<SPEC_F32>);
        rc = bf ? go(spec_single_kernel<SPEC_BF16>) : go(spec_single_kernel<SPEC_F32>);
        if (rc) return rc;
    }
    if (bigf) return bf ? launch_finish<SPEC_BF16, 8>(fi, np, st) : launch_finish<SPEC_F32, 8>(fi, np, st);
    return bf ? launch_finish<SPEC_BF16, 0>(fi, np, st) : launch_finish<SPEC_F32, 0>(fi, np, st);
}

int verify_common(const SpecIn *in, const SpecOut *out, void *ws, int64_t ws_bytes, void *stream, int mode)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    if (!out || !out->accepted_node || !out->accept_len || !out->out_tokens || !out->bonus_token || !out->status)
        return SPEC_ERR_NULL;
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    const WsLayout L = ws_layout(in);
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < L.total) return SPEC_ERR_WORKSPACE;
    VPlan pl;
    bool big;
    if (!one_cta_plan(in->V, 7, (int)sizeof(BHdr), &pl, &big)) return SPEC_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char *w = (unsigned char *)ws;
    const bool diagnostics = out->residual || out->node_thr || out->node_w_in || out->margin;
    if (mode == MODE_SPECINFER && !diagnostics && in->N <= NWALK) return verify_walk(in, out, w, L, trunc, st);
    // every node of every sequence on chip once, on top of the row statistics (which also set the
    // published-weight slots to pending and the arrival counters to zero)
    rc = row_statistics(in, out, w, L, trunc, st, true);
    if (rc) return rc;
    NParams tp = {};
    fill_params(in, out, w, L, mode, tp);
    VParams &vp = tp.v;
    rc = launch_nodes(in, tp, false, st);
    if (rc) return rc;
    if (out->residual) {
        RParams rp = {};
        rp.B = in->B; rp.N = in->N; rp.V = in->V; rp.dtype = in->logits_dtype;
        rp.zp = in->target_logits; rp.zq = in->draft_logits;
        rp.seq_stride = in->seq_stride; rp.node_stride = in->node_stride;
        rp.T = in->temperature; rp.T_seq = in->temperature_per_seq;
        rp.rec = vp.rec; rp.gseq = tp.gseq; rp.accepted = out->accepted_node; rp.residual = out->residual;
        int gx = (in->V + 255) / 256;
        if (gx > 296) gx = 296;
        rc = launch_after(spec_residual_kernel, dim3(gx, in->B), 256, st, &rp);
        if (rc) return rc;
    }
    return SPEC_OK;
}

// ------------------------------------------------------------------------------------------------
// host-buffer entry point: staging layout inside the caller's device buffer
// ------------------------------------------------------------------------------------------------
struct HostLayout {
    int64_t zp, zq, parent, token, ua, ub, acc, len, toks, bonus, status, ws, total;
    int64_t logit_bytes, parent_bytes, bn4, b4;
};

HostLayout host_layout(const SpecIn *in)
{
    HostLayout L = {};
    const int64_t esz = in->logits_dtype == SPEC_BF16 ? 2 : 4;
    L.logit_bytes = (int64_t)in->B * in->N * in->V * esz;
    L.parent_bytes = (in->topo_seq_stride ? (int64_t)in->B : 1) * in->N * 4;
    L.bn4 = (int64_t)in->B * in->N * 4;
    L.b4 = (int64_t)in->B * 4;
    int64_t o = 0;
    L.zp = o; o += up256(L.logit_bytes);
    L.zq = o; o += up256(L.logit_bytes);
    L.parent = o; o += up256(L.parent_bytes);
    L.token = o; o += up256(L.bn4);
    L.ua = o; o += up256(L.bn4);
    L.ub = o; o += up256(L.bn4);
    L.acc = o; o += up256(L.b4);
    L.len = o; o += up256(L.b4);
    L.toks = o; o += up256(L.bn4);
    L.bonus = o; o += up256(L.b4);
    L.status = o; o += up256(L.b4);
    L.ws = o; o += up256(ws_layout(in).total);
    L.total = o;
    return L;
}

// The draft rows to the device: those of childless nodes stay behind (a tree of 4 branches: 1 row in 5; B = 8, V = 128256: 1.51 ->
// 1.38 ms a call, which is bound by the PCIe copies).  A gap is left out where its bytes take longer than the
// copy that it makes necessary (a few us, 256 KB).  Work that the stream still has may yet write the tree: it is waited for
// before the tree is read (the copies would have waited for it as well, and the call ends with a wait).
constexpr int64_t GAP_BYTES = 256 << 10, GAP_ROW_BYTES = 64 << 10;
cudaError_t wait_for_earlier_work(cudaStream_t st)
{
    cudaEvent_t e;                    // (an event, so that the default stream's order with other streams counts)
    cudaError_t rc = cudaEventCreateWithFlags(&e, cudaEventDisableTiming);
    if (rc != cudaSuccess) return rc;
    rc = cudaEventRecord(e, st);
    if (rc == cudaSuccess) rc = cudaEventSynchronize(e);
    cudaEventDestroy(e);
    return rc;
}
cudaError_t copy_draft_rows(const SpecIn *in, const HostLayout &L, unsigned char *dst, cudaStream_t st)
{
    const unsigned char *src = (const unsigned char *)in->draft_logits;
    const int64_t row = L.logit_bytes / ((int64_t)in->B * in->N), seq = row * in->N;
    if (row < GAP_ROW_BYTES) return cudaMemcpyAsync(dst, src, (size_t)L.logit_bytes, cudaMemcpyHostToDevice, st);
    const cudaError_t waited = wait_for_earlier_work(st);
    if (waited != cudaSuccess) return waited;
    // one tree for all: a strided copy per run of nodes; a tree per sequence: copies per sequence
    const int trees = in->topo_seq_stride ? in->B : 1, N = in->N;
    const int64_t height = in->topo_seq_stride ? 1 : in->B;
    char inner[SPEC_MAX_NODES];
    for (int t = 0; t < trees; ++t) {
        std::fill(inner, inner + N, 0);
        for (int c = 0; c < N; ++c) {
            const int pa = in->parent[(int64_t)t * in->topo_seq_stride + c];
            if (pa >= 0 && pa < N) inner[pa] = 1;
        }
        for (int a = 0; a < N;) {
            if (!inner[a]) { ++a; continue; }
            int end = a + 1;                                  // the run a .. end - 1, short gaps included
            for (int c = end; c < N && (c - end) * row * height < GAP_BYTES; ++c)
                if (inner[c]) end = c + 1;
            const int64_t off = t * seq + a * row;
            const cudaError_t e = height > 1
                ? cudaMemcpy2DAsync(dst + off, (size_t)seq, src + off, (size_t)seq, (size_t)((end - a) * row), (size_t)height, cudaMemcpyHostToDevice, st)
                : cudaMemcpyAsync(dst + off, src + off, (size_t)((end - a) * row), cudaMemcpyHostToDevice, st);
            if (e != cudaSuccess) return e;
            a = end;
        }
    }
    return cudaSuccess;
}

// ------------------------------------------------------------------------------------------------
// scratch that lives inside the library image, for spec_verify_specinfer_static
// ------------------------------------------------------------------------------------------------
constexpr int64_t STATIC_WS_BYTES = SPEC_STATIC_WS_BYTES;
static __device__ __align__(256) unsigned char g_static_ws[STATIC_WS_BYTES];

// Device address of g_static_ws on the current device.  In host code the array's name is only a
// handle for the runtime, never a device pointer, so the address is asked for once per device (with
// that device current) and remembered.
int static_ws_address(void **ptr)
{
    static void *addr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    std::lock_guard<std::mutex> lock(g_cache_mutex);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_ws) != cudaSuccess || !p) { cudaGetLastError(); return SPEC_ERR_CUDA; }
        addr[dev] = p;
    }
    *ptr = addr[dev];
    return SPEC_OK;
}

}  // namespace
}  // namespace specv

using namespace specv;

extern "C" {

int32_t spec_workspace_bytes(const SpecIn *in, int64_t *bytes)
{
    if (!in || !bytes) return SPEC_ERR_NULL;
    if (in->B <= 0 || in->N <= 0 || in->N > SPEC_MAX_NODES || (long long)in->B * in->N > (1ll << 24))
        return SPEC_ERR_SHAPE;
    *bytes = ws_layout(in).total;
    return SPEC_OK;
}

int32_t spec_query_plan(int32_t V, int32_t logits_dtype, int32_t *cluster_size, int32_t *slice_len,
                        int32_t *smem_bytes, int32_t *threads)
{
    if (V <= 0) return SPEC_ERR_SHAPE;
    if (logits_dtype != SPEC_F32 && logits_dtype != SPEC_BF16) return SPEC_ERR_DTYPE;
    WalkPlan plan;
    if (!walk_plan(V, logits_dtype, 1 << 20, true, false, 148, &plan)) return SPEC_ERR_UNSUPPORTED;
    const VPlan &pl = plan.pl;
    if (cluster_size) *cluster_size = pl.C;
    if (slice_len) *slice_len = pl.slice_len;
    if (smem_bytes) *smem_bytes = pl.smem;
    if (threads) *threads = 256;
    return SPEC_OK;
}

int64_t spec_kernel_launches(void) { return (int64_t)g_kernel_launches.load(std::memory_order_relaxed); }

int32_t spec_test_hooks(int64_t wait_cycles, int32_t hold_slot)
{
    const long long wc = wait_cycles > 0 ? (long long)wait_cycles : WAIT_CYCLES_DEFAULT;
    const int hs = hold_slot;
    if (cudaMemcpyToSymbol(c_wait_cycles, &wc, sizeof(wc)) != cudaSuccess ||
        cudaMemcpyToSymbol(c_hold_slot, &hs, sizeof(hs)) != cudaSuccess) {
        cudaGetLastError();
        return SPEC_ERR_CUDA;
    }
    return SPEC_OK;
}

int32_t spec_row_statistics(const SpecIn *in, void *ws, int64_t ws_bytes, void *stream)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    const WsLayout L = ws_layout(in);
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < L.total) return SPEC_ERR_WORKSPACE;
    SpecOut none = {};
    return row_statistics(in, &none, (unsigned char *)ws, L, trunc, (cudaStream_t)stream, true);
}

int32_t spec_verify_specinfer(const SpecIn *in, const SpecOut *out, void *ws, int64_t ws_bytes, void *stream)
{
    return verify_common(in, out, ws, ws_bytes, stream, MODE_SPECINFER);
}

int32_t spec_verify_traversal(const SpecIn *in, const SpecOut *out, void *ws, int64_t ws_bytes, void *stream)
{
    return verify_common(in, out, ws, ws_bytes, stream, MODE_TRAVERSAL);
}

int32_t spec_verify_otlp(const SpecIn *in, const SpecOut *out, int32_t solver, void *ws, int64_t ws_bytes, void *stream)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    if (!out || !out->accepted_node || !out->accept_len || !out->out_tokens || !out->bonus_token || !out->status)
        return SPEC_ERR_NULL;
    if (solver < 0 || solver > 2) return SPEC_ERR_PARAM;
    if (out->residual || out->node_thr || out->node_w_in || out->margin || out->node_features || in->N > NWALK)
        return SPEC_ERR_UNSUPPORTED;
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    const WsLayout L = ws_layout(in);
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < L.total) return SPEC_ERR_WORKSPACE;
    return verify_walk(in, out, (unsigned char *)ws, L, trunc, (cudaStream_t)stream, solver);
}

int32_t spec_verify_specinfer_static(const SpecIn *in, const SpecOut *out, void *stream)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    if ((int64_t)in->B * in->N > SPEC_STATIC_MAX_NODES || ws_layout(in).total > STATIC_WS_BYTES) return SPEC_ERR_WORKSPACE;
    void *ws = nullptr;
    rc = static_ws_address(&ws);
    if (rc) return rc;
    return verify_common(in, out, ws, STATIC_WS_BYTES, stream, MODE_SPECINFER);
}

// analysis workspace: the verifiers' layout | per-node scalars | scratch for the decision outputs nobody reads
struct AnLayout {
    int64_t an, acc, len, toks, bonus, status, total;
};
static AnLayout an_layout(const SpecIn *in)
{
    AnLayout A;
    const int64_t nodes = (int64_t)in->B * in->N;
    int64_t o = up256(ws_layout(in).total);
    A.an = o; o += up256(nodes * (int64_t)sizeof(AnRec));
    A.acc = o; o += up256((int64_t)in->B * 4);
    A.len = o; o += up256((int64_t)in->B * 4);
    A.toks = o; o += up256(nodes * 4);
    A.bonus = o; o += up256((int64_t)in->B * 4);
    A.status = o; o += up256((int64_t)in->B * 4);
    A.total = o;
    return A;
}

int32_t spec_analysis_workspace_bytes(const SpecIn *in, int64_t *bytes)
{
    if (!in || !bytes) return SPEC_ERR_NULL;
    if (in->B <= 0 || in->N <= 0 || in->N > SPEC_MAX_NODES || (long long)in->B * in->N > (1ll << 24))
        return SPEC_ERR_SHAPE;
    *bytes = an_layout(in).total;
    return SPEC_OK;
}

int32_t spec_tree_analysis(const SpecIn *in, const SpecAnalysisOut *out, void *ws, int64_t ws_bytes, void *stream)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    if (!out || !out->acceptance || !out->divergence || !out->branch || !out->reach || !out->block_eff) return SPEC_ERR_NULL;
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    const WsLayout L = ws_layout(in);
    const AnLayout A = an_layout(in);
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < A.total) return SPEC_ERR_WORKSPACE;
    VPlan pl;
    bool big;
    if (!one_cta_plan(in->V, 7, (int)sizeof(BHdr), &pl, &big)) return SPEC_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char *w = (unsigned char *)ws;
    const int64_t nodes = (int64_t)in->B * in->N;
    // outputs start as NaN (all-ones), the per-node scalars as "no children"
    bool ok = true;
    ok &= cudaMemsetAsync(out->acceptance, 0xFF, (size_t)nodes * 16, st) == cudaSuccess;
    ok &= cudaMemsetAsync(out->divergence, 0xFF, (size_t)nodes * 12, st) == cudaSuccess;
    ok &= cudaMemsetAsync(out->branch, 0xFF, (size_t)nodes * 4 * analysis::NSOLVER, st) == cudaSuccess;
    ok &= cudaMemsetAsync(w + A.an, 0, (size_t)nodes * sizeof(AnRec), st) == cudaSuccess;
    if (!ok) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    SpecOut so = {};
    so.accepted_node = (int32_t *)(w + A.acc); so.accept_len = (int32_t *)(w + A.len);
    so.out_tokens = (int32_t *)(w + A.toks); so.bonus_token = (int32_t *)(w + A.bonus);
    so.status = (int32_t *)(w + A.status);
    rc = row_statistics(in, &so, w, L, trunc, st, true);
    if (rc) return rc;
    NParams tp = {};
    fill_params(in, &so, w, L, MODE_SPECINFER, tp);
    tp.v.all_thr = 1;
    tp.an = (AnRec *)(w + A.an); tp.an_acc = out->acceptance; tp.an_div = out->divergence;
    rc = launch_nodes(in, tp, true, st);
    if (rc) return rc;
    analysis::BParams bp = {in->B, in->N, in->parent, in->token, in->topo_seq_stride, tp.an, out->acceptance, out->branch};
    rc = launch_after(analysis::spec_branch_kernel, dim3((unsigned)((nodes + 3) / 4)), 128, st, &bp);
    if (rc) return rc;
    analysis::RParams rp = {in->B, in->N, in->parent, in->topo_seq_stride, out->branch, out->reach, out->block_eff};
    return launch_after(analysis::spec_reach_kernel, dim3((unsigned)((analysis::NSOLVER * in->B + 127) / 128)), 128, st, &rp);
}

int32_t spec_latency_model(const double *t_q, const double *t_p, int32_t n_len, int32_t ctx, const int32_t *actions,
                           int32_t n_actions, double *T_hat, void *stream)
{
    if (!t_q || !t_p || !actions || !T_hat) return SPEC_ERR_NULL;
    if (n_len <= 0 || n_actions <= 0 || ctx < 0) return SPEC_ERR_SHAPE;
    analysis::LParams lp = {t_q, t_p, n_len, ctx, n_actions, actions, T_hat};
    analysis::spec_latency_kernel<<<(unsigned)((n_actions + 127) / 128), 128, 0, (cudaStream_t)stream>>>(lp);
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
    if (cudaGetLastError() != cudaSuccess) return SPEC_ERR_CUDA;
    return SPEC_OK;
}

int32_t spec_tree_probs(const SpecIn *in, int32_t which, float *probs, float *row_stats, void *ws,
                        int64_t ws_bytes, void *stream)
{
    int rc = check_in(in, false);
    if (rc) return rc;
    if (which != 0 && which != 1) return SPEC_ERR_PARAM;
    const void *z = which ? in->draft_logits : in->target_logits;
    if (!z || (!probs && !row_stats)) return SPEC_ERR_NULL;
    const bool trunc = (in->top_k > 0 && in->top_k < in->V) || in->top_p < 1.f;
    RowPlan pl;
    if (!make_row_plan(in->V, (long long)in->B * in->N, sm_count(), &pl)) return SPEC_ERR_UNSUPPORTED;
    if (trunc) {
        // the record of every row of the chosen side goes to the first of its pair in the workspace
        const WsLayout L = ws_layout(in);
        if (!ws || ((uintptr_t)ws & 255) || ws_bytes < L.total) return SPEC_ERR_WORKSPACE;
        rc = launch_trunc(in, z, z, nullptr, (unsigned char *)ws, L, stream::NodeInit{}, (cudaStream_t)stream);
        if (rc) return rc;
        rowops::KParams kp = {};
        kp.N = in->N; kp.V = in->V; kp.z = z; kp.seq_stride = in->seq_stride; kp.node_stride = in->node_stride;
        kp.T = in->temperature; kp.T_seq = in->temperature_per_seq;
        kp.part = (const RowPart *)((unsigned char *)ws + L.stat); kp.kept = (const int *)((unsigned char *)ws + L.kept);
        kp.probs = probs; kp.stats = row_stats;
        kp.parts = probs ? (in->V + rowops::KEPT_PART - 1) / rowops::KEPT_PART : 1;
        kp.items = (long long)in->B * in->N * kp.parts;
        const int grid = (int)std::min(kp.items, 1ll << 20);
        const auto go = [&](auto kernel) { return launch_clustered(kernel, grid, 0, rowops::KEPT_NT, 0, (cudaStream_t)stream, &kp, true); };
        return in->logits_dtype == SPEC_BF16 ? go(rowops::spec_probs_kept_kernel<SPEC_BF16>) : go(rowops::spec_probs_kept_kernel<SPEC_F32>);
    }
    rowops::TParams tp = {};
    tp.rows = in->B * in->N; tp.N = in->N; tp.V = in->V; tp.dtype = in->logits_dtype; tp.SL = pl.SL;
    tp.z = z; tp.seq_stride = in->seq_stride; tp.node_stride = in->node_stride;
    tp.T = in->temperature; tp.T_seq = in->temperature_per_seq; tp.probs = probs; tp.stats = row_stats;
    rc = prepare_kernel(rowops::spec_probs_kernel, pl.C, pl.smem);
    if (rc) return rc;
    return launch_clustered(rowops::spec_probs_kernel, tp.rows * pl.C, pl.C, rowops::NT, pl.smem, (cudaStream_t)stream, &tp, true);
}

int32_t spec_sample_bonus(const float *weights, int32_t R, int32_t V, const float *u, int32_t *token,
                          float *margin, void *ws, int64_t ws_bytes, void *stream)
{
    (void)ws; (void)ws_bytes;
    if (!weights || !u || !token) return SPEC_ERR_NULL;
    if (R <= 0 || V <= 0) return SPEC_ERR_SHAPE;
    RowPlan pl;
    if (!make_row_plan(V, R, sm_count(), &pl)) return SPEC_ERR_UNSUPPORTED;
    // CTAs for about four per SM, a slice of at least 4096 weights each, as many as the tiles' sums of a slice ask for
    int C = 1;
    while (C < rowops::BN_CMAX && (((long long)R * C < 4ll * sm_count() && V >= C * 8192) || (V + C - 1) / C > (rowops::BN_TILES - 1) * rowops::BN_TILE)) C <<= 1;
    rowops::BParams bp = {R, V, up((V + C - 1) / C, rowops::BN_TILE), weights, u, token, margin};
    return launch_clustered(rowops::spec_bonus_kernel, R * C, C, rowops::BN_NT, 0, (cudaStream_t)stream, &bp, true);
}

int32_t spec_host_staging_bytes(const SpecIn *in, int64_t *bytes)
{
    if (!in || !bytes) return SPEC_ERR_NULL;
    int rc = check_in(in, false);
    if (rc) return rc;
    *bytes = host_layout(in).total;
    return SPEC_OK;
}

int32_t spec_verify_host(const SpecIn *in, const SpecOut *out, int32_t algorithm, void *dev_buf,
                         int64_t dev_bytes, void *stream)
{
    int rc = check_in(in, true);
    if (rc) return rc;
    if (!out || !out->accepted_node || !out->accept_len || !out->out_tokens || !out->bonus_token || !out->status)
        return SPEC_ERR_NULL;
    if (out->residual || out->node_thr || out->node_w_in || out->node_features || out->margin)
        return SPEC_ERR_UNSUPPORTED;
    if (algorithm != 0 && algorithm != 1) return SPEC_ERR_PARAM;
    if (in->temperature_per_seq) return SPEC_ERR_UNSUPPORTED;
    if (in->node_stride != in->V || in->seq_stride != (int64_t)in->N * in->V) return SPEC_ERR_SHAPE;
    if (in->topo_seq_stride != 0 && in->topo_seq_stride != in->N) return SPEC_ERR_SHAPE;
    const HostLayout L = host_layout(in);
    if (!dev_buf || ((uintptr_t)dev_buf & 255) || dev_bytes < L.total) return SPEC_ERR_WORKSPACE;
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char *d = (unsigned char *)dev_buf;
    bool ok = true;
    ok &= copy_draft_rows(in, L, d + L.zq, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(d + L.zp, in->target_logits, (size_t)L.logit_bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(d + L.parent, in->parent, (size_t)L.parent_bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(d + L.token, in->token, (size_t)L.bn4, cudaMemcpyHostToDevice, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(d + L.ua, in->u_accept, (size_t)L.bn4, cudaMemcpyHostToDevice, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(d + L.ub, in->u_bonus, (size_t)L.bn4, cudaMemcpyHostToDevice, st) == cudaSuccess;
    if (!ok) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    SpecIn din = *in;
    din.target_logits = d + L.zp; din.draft_logits = d + L.zq;
    din.parent = (const int32_t *)(d + L.parent); din.token = (const int32_t *)(d + L.token);
    din.u_accept = (const float *)(d + L.ua); din.u_bonus = (const float *)(d + L.ub);
    SpecOut dout = {};
    dout.accepted_node = (int32_t *)(d + L.acc); dout.accept_len = (int32_t *)(d + L.len);
    dout.out_tokens = (int32_t *)(d + L.toks); dout.bonus_token = (int32_t *)(d + L.bonus);
    dout.status = (int32_t *)(d + L.status);
    rc = verify_common(&din, &dout, d + L.ws, L.total - L.ws, stream, algorithm == 0 ? MODE_SPECINFER : MODE_TRAVERSAL);
    if (rc) return rc;
    ok &= cudaMemcpyAsync(out->accepted_node, dout.accepted_node, (size_t)L.b4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(out->accept_len, dout.accept_len, (size_t)L.b4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(out->out_tokens, dout.out_tokens, (size_t)L.bn4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(out->bonus_token, dout.bonus_token, (size_t)L.b4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok &= cudaMemcpyAsync(out->status, dout.status, (size_t)L.b4, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    if (!ok || cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return SPEC_ERR_CUDA; }
    return SPEC_OK;
}

}  // extern "C"
