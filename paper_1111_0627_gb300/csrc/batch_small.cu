// batch_small.cu -- the batched form's persistent per-graph solver.
//
// The regions of Sec. 3.3 are independent; for the small ones a whole Howard
// iteration (Alg. 1: evaluate the policy, improve it, stop when stable) fits
// one team, a thread block or a cluster of four (team.cuh).  A persistent grid
// of teams pops graph tasks from a queue ordered by decreasing size (a log2
// bucket per size class, the largest first, so the longest tasks start first),
// and every team runs all iterations of its graph with barriers of its own: no
// grid barrier and no launch per iteration.  Each graph converges on its own
// (the paper's per-region "work" flag becomes the end of the team's loop) and
// leaves its answer in the per-graph records of the batch; the larger graphs go
// through the disjoint-union path of batch.cu / evaluate.cu / sweep.cu, which
// skips the graphs solved here.
//
// Bound: the latency of gathers from L2, 32 warps per SM, and the longest task.
// 1,024 graphs of up to 200,000 vertices (27 million in all): the largest, 200,000
// vertices through 47 iterations, took 158 ms in one block, longer than the
// others together; with clusters of four from 2^15 vertices the batch takes 72 ms
// (2: 94, 8: 85, 16: 108 ms), and 178 ms before the teams walked.  4,096 graphs
// of up to 20,000, none above a sixth of the vertices per block: 24 ms (32 before
// the walks), and 27 with the largest in clusters.
#include <climits>

#include "common.cuh"
#include "grid_sync.cuh"
#include "team.cuh"

namespace ocm {

constexpr int kSmallBuckets = 32;

// Size buckets of the queue: floor(log2(n_g)), largest first.
static __device__ __forceinline__ int size_bucket(int n) { return 31 - __clz(n); }

static __device__ __forceinline__ bool small_eligible(const BatchState &bs,
                                                      const int *__restrict__ row_ptr, int g,
                                                      int max_n, int *n_out) {
    const int a = bs.vptr[g], b = bs.vptr[g + 1];
    const int n = b - a;
    const long long m = (long long)row_ptr[b] - row_ptr[a];
    *n_out = n;
    return n <= max_n && m <= 16LL * max_n;
}

__global__ void __launch_bounds__(kThreads)
small_count_kernel(const int *__restrict__ row_ptr, BatchState bs, int max_n, Ctrl *c) {
    __shared__ int s_cnt[kSmallBuckets];
    if (threadIdx.x < kSmallBuckets) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < bs.G; g += gridDim.x * blockDim.x) {
        int n;
        if (small_eligible(bs, row_ptr, g, max_n, &n)) atomicAdd(&s_cnt[size_bucket(n)], 1);
    }
    __syncthreads();
    if (threadIdx.x < kSmallBuckets && s_cnt[threadIdx.x])
        atomicAdd(&c->small_bucket[threadIdx.x], s_cnt[threadIdx.x]);
}

// Queue positions: bucket b (larger b first) starts after all larger buckets;
// within a bucket the order is that of the atomics (it decides only which
// block solves which graph, never a result).
__global__ void __launch_bounds__(kThreads)
small_fill_kernel(const int *__restrict__ row_ptr, BatchState bs, int max_n, int big_bucket,
                  Ctrl *c, int *queue) {
    __shared__ int s_start[kSmallBuckets];
    if (threadIdx.x == 0) {
        int run = 0;
        for (int b = kSmallBuckets - 1; b >= 0; --b) {
            s_start[b] = run;
            run += c->small_bucket[b];
            if (blockIdx.x == 0 && b == big_bucket) c->small_big = run;
        }
        if (blockIdx.x == 0) c->small_total = run;
    }
    __syncthreads();
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < bs.G; g += gridDim.x * blockDim.x) {
        int n;
        if (small_eligible(bs, row_ptr, g, max_n, &n)) {
            const int b = size_bucket(n);
            queue[s_start[b] + atomicAdd(&c->small_cursor[b], 1)] = g;
        }
    }
}

// One graph after the other from the queue, each by one team (team.cuh).
template <int C>
__global__ void __launch_bounds__(kTeamThreads, 1)
small_graph_kernel(const int *__restrict__ row_ptr, const int *__restrict__ col,
                   const int *__restrict__ w, int sign, const int *__restrict__ queue,
                   long long max_iters, int warm, Workspace ws, BatchState bs) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ TeamShared s_team;
    Ctrl *c = ws.ctrl;
    // (the blocks of the other instance may fill the SMs these clusters leave)
    if (C > 1) asm volatile("griddepcontrol.launch_dependents;");
    Team<C> tm;
    tm.init(&s_team);
    // the cluster instance takes the queue's first small_big graphs
    const int first = C > 1 ? 0 : c->small_big;
    const int total = (C > 1 ? c->small_big : c->small_total) - first;
    int *head = C > 1 ? &c->big_head : &c->small_head;
    for (;;) {
        if (tm.tid == 0) {
            // an error anywhere fails the whole call: stop
            const bool stop = load_volatile(&c->err) != 0 || load_volatile(&c->not_converged);
            tm.sh->task = stop ? INT_MAX : atomicAdd(head, 1);
        }
        tm.sync();
        const int qi = *reinterpret_cast<volatile int *>(&tm.sh->task);
        if (qi >= total) break;   // (the same decision in every thread of the team)
        const int g = queue[first + qi];
        const int v0 = bs.vptr[g], n = bs.vptr[g + 1] - v0;
        bool in_shared;
        const TeamGraph tg = team_place<C>(s_dyn, row_ptr, col, w, sign, v0, n, ws,
                                              C > 1 ? 0 : kTeamBytes, &in_shared);
        int it = 0;
        long long switched = 0;
        bool capped = false;
        const bool ok = C == 1 && in_shared
                            ? team_iterate<C, true>(tm, tg, warm, max_iters, &it, &switched, &capped)
                            : team_iterate<C, false>(tm, tg, warm, max_iters, &it, &switched, &capped);
        if (tm.tid == 0) {
            if (capped) c->not_converged = 1;
            if (ok) {
                const unsigned long long packed =
                    *reinterpret_cast<volatile unsigned long long *>(tg.best);
                const int root = INT_MAX - (int)(unsigned)(packed & 0xffffffffu);
                const int i = ws.cid_of_root[root];
                bs.gbest[g] = packed;
                bs.groot[g] = root;
                bs.glen[g] = ws.cyc_L[i];
                bs.gp[g] = ws.cyc_p[i];
                bs.gq[g] = ws.cyc_q[i];
                bs.gconv[g] = 1;
                atomicMax(&c->small_iters, it);
            }
        }
        tm.sync();
    }
    tm.sync();   // (the first block's shared memory stays until all are done)
    // (what follows in the stream waits for this instance, so this one for the other)
    if (C == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

constexpr int kBigCluster = 4;       // blocks that solve a big graph together
constexpr int kBigMinBucket = 12;    // 4,096 vertices: smaller graphs do not fill them

// Builds the queue of graphs with at most max_n vertices (and at most 16 max_n
// edges) and solves them, each by a block, or by a cluster of kBigCluster
// blocks where it holds more than about a sixth of the batch's vertices
// per resident block; returns the number of kernel launches, or -1.  max_n == 0
// picks the size limit from the batch: a graph stays out of the queue (for the
// whole-grid path) when it holds more than four times the batch's vertices per
// resident block (a few huge graphs are faster on the whole grid, the rest of
// the batch is not worth a launch per iteration), and never below
// kBatchSmallDefault.
int launch_batch_small(const int *row_ptr, const int *col, const int *w, int sign, int max_n,
                       long long N, int max_ng, long long max_iters, int warm, int *queue,
                       Workspace ws, BatchState bs, cudaStream_t st) {
    static int cached_dev = -1, cached_blocks = 0, cached_clusters = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    cudaLaunchConfig_t big = {};
    big.gridDim = dim3(kBigCluster);
    big.blockDim = dim3(kTeamThreads);
    big.stream = st;
    cudaLaunchAttribute cluster[1];
    cluster[0].id = cudaLaunchAttributeClusterDimension;
    cluster[0].val.clusterDim.x = kBigCluster;
    cluster[0].val.clusterDim.y = 1;
    cluster[0].val.clusterDim.z = 1;
    big.attrs = cluster;
    big.numAttrs = 1;
    if (dev != cached_dev) {
        int sms = 0, per_sm = 0, clusters = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return -1;
        if (cudaFuncSetAttribute(small_graph_kernel<1>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kTeamBytes) != cudaSuccess)
            return -1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, small_graph_kernel<1>,
                                                          kTeamThreads, kTeamBytes) != cudaSuccess ||
            per_sm < 1)
            return -1;
        // (a device that cannot place the cluster solves those graphs in blocks)
        if (cudaOccupancyMaxActiveClusters(&clusters, small_graph_kernel<kBigCluster>, &big) !=
            cudaSuccess) {
            cudaGetLastError();
            clusters = 0;
        }
        cached_blocks = sms * per_sm;
        cached_clusters = clusters;
        cached_dev = dev;
    }
    if (max_n == 0) {
        const long long auto_n = 4 * N / cached_blocks;
        max_n = (int)(auto_n > INT_MAX / 16 ? INT_MAX / 16
                                            : (auto_n < kBatchSmallDefault ? kBatchSmallDefault
                                                                           : auto_n));
    }
    int big_bucket = kBigMinBucket;
    while (big_bucket < 31 && (1LL << big_bucket) < N / (6LL * cached_blocks)) ++big_bucket;
    const bool has_big = cached_clusters > 0 && big_bucket < 31 && max_ng >= (1 << big_bucket) &&
                         max_n >= (1 << big_bucket);
    int gb = (bs.G + kThreads - 1) / kThreads;
    if (gb > 1024) gb = 1024;
    prof_begin(kProfEvaluate, st);
    small_count_kernel<<<gb, kThreads, 0, st>>>(row_ptr, bs, max_n, ws.ctrl);
    small_fill_kernel<<<gb, kThreads, 0, st>>>(row_ptr, bs, max_n, has_big ? big_bucket : -1,
                                               ws.ctrl, queue);
    cudaError_t e = cudaSuccess;
    if (has_big) {
        big.gridDim = dim3((bs.G < cached_clusters ? bs.G : cached_clusters) * kBigCluster);
        e = cudaLaunchKernelEx(&big, small_graph_kernel<kBigCluster>, row_ptr, col, w, sign,
                               (const int *)queue, max_iters, warm, ws, bs);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cached_blocks);
    cfg.blockDim = dim3(kTeamThreads);
    cfg.dynamicSmemBytes = kTeamBytes;
    cfg.stream = st;
    cudaLaunchAttribute along[1];
    along[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    along[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = along;
    cfg.numAttrs = has_big ? 1 : 0;
    if (e == cudaSuccess)
        e = cudaLaunchKernelEx(&cfg, small_graph_kernel<1>, row_ptr, col, w, sign,
                               (const int *)queue, max_iters, warm, ws, bs);
    prof_end(kProfEvaluate, st);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? (has_big ? 4 : 3) : -1;
}

}  // namespace ocm
