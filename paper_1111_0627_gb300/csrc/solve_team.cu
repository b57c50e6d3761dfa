// solve_team.cu -- the whole solve of a small graph in one launch: validation,
// initial policy, every iteration and the critical cycle, by one block or one
// cluster (team.cuh).
//
// A small solve is bound by launches and host round trips: 25 launches besides
// the loop, five kernels and a grid barrier or two per iteration, each a few
// microseconds whatever the size.  One team needs a barrier of its own between
// steps (under a microsecond) and a single launch and read-back.  Measured, ring
// plus 0-4 extra edges a vertex, four graphs a size, against the launch per
// step: n = 257 152 against 457 us, 1,100 347 / 644, 4,500 591 / 899, 10,000
// 733 / 957, 16,000 944 / 1,167; at 25,000 16 blocks no longer suffice (1,464 /
// 1,462).
#include <climits>

#include "common.cuh"
#include "grid_sync.cuh"
#include "team.cuh"

namespace ocm {

// Graphs solved by one team: up to kTeamSolveN vertices with 8 edges each on
// average (the sweep gives a vertex of up to 32 edges one thread), by one block
// up to kTeamBlockN.
constexpr int kTeamSolveN = 16384;
constexpr int kTeamBlockN = 1024;
static_assert(2LL * kTeamSolveN * kTeamSolveN < (1LL << 62 >> 31), "values and keys stay exact");
static_assert(kTeamBlockN <= kTeamSharedN, "one block's states fit in its shared memory");

// The checks of check_row_ptr_kernel; also notes vertices of more than
// kHeavyEdges edges (Ctrl::team_off).
template <int C>
static __device__ bool team_check(Team<C> &tm, const int *row_ptr, int n, int m, Ctrl *ctrl) {
    int err = 0, heavy = 0;
    for (int v = tm.tid; v <= n; v += tm.W) {
        const int a = row_ptr[v];
        if (v == 0 && a != 0) err |= kErrRowPtr;
        if (v == n) {
            if (a != m) err |= kErrRowPtr;
        } else {
            const int b = row_ptr[v + 1];
            if (b < a || a < 0 || b > m) err |= kErrRowPtr;
            else if (b == a) err |= kErrNoOutEdge;
            else if (b - a > kHeavyEdges) heavy = 1;
        }
    }
    if (err) atomicOr(&ctrl->err, err);
    if (heavy) ctrl->team_off = 1;
    return tm.sum((err != 0) + heavy) == 0;
}

// The initial policy and the checks of init_policy_kernel: the heaviest
// out-edge in the s*w sense, ties to the smallest edge index, or the caller's
// edge.  A thread per vertex of out-degree <= 32, a warp per vertex with more.
template <int C>
static __device__ bool team_init(Team<C> &tm, const int *row_ptr, const int *col, const int *w,
                                 int sign, int n, const int *init, const Workspace &ws) {
    Ctrl *ctrl = ws.ctrl;
    const int lane = threadIdx.x & 31;
    int err = 0, maxabs = 0;
    for (int base = tm.tid - lane; base < n; base += tm.W) {
        const int v = base + lane;
        const int a = v < n ? row_ptr[v] : 0, b = v < n ? row_ptr[v + 1] : 0;
        int best_k = INT_MIN, best_e = INT_MAX;
        auto take = [&](int e, int &bk, int &be) {
            const int t = col[e];
            int x = w[e];
            if ((unsigned)t >= (unsigned)n) err |= kErrCol;
            if (x == INT_MIN) {
                err |= kErrWeightMin;
                x = 0;
            }
            maxabs = max(maxabs, x < 0 ? -x : x);
            const int k = sign * x;   // (edges in increasing order)
            if (be == INT_MAX || k > bk) {
                bk = k;
                be = e;
            }
        };
        const bool wide = b - a > 32;
        if (!wide) {
#pragma unroll 4
            for (int e = a; e < b; ++e) take(e, best_k, best_e);
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, wide); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const int ea = __shfl_sync(0xffffffffu, a, src), eb = __shfl_sync(0xffffffffu, b, src);
            int bk = INT_MIN, be = INT_MAX;
            for (int e = ea + lane; e < eb; e += 32) take(e, bk, be);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                const int oe = __shfl_xor_sync(0xffffffffu, be, o);
                if (oe != INT_MAX && (be == INT_MAX || ok > bk || (ok == bk && oe < be))) {
                    bk = ok;
                    be = oe;
                }
            }
            if (lane == src) {
                best_k = bk;
                best_e = be;
            }
        }
        if (v < n) {
            int be = best_e;
            if (init) {
                const int e = init[v];
                if (e >= a && e < b) be = e;
                else err |= kErrInitPolicy;
            }
            const int t = col[be], x = w[be];
            ws.pi[v] = be;
            ws.succ[v] = (unsigned)t < (unsigned)n ? t : 0;
            ws.wpi[v] = sign * (x == INT_MIN ? 0 : x);
            ws.root_mark[v] = 0;
            ws.cyc_tag[v] = 0;
        }
    }
    maxabs = __reduce_max_sync(0xffffffffu, maxabs);
    if (lane == 0 && maxabs) atomicMax(&ctrl->maxabsw, maxabs);
    if (err) atomicOr(&ctrl->err, err);
    return tm.sum(err != 0) == 0;
}

// The critical cycle from its root: a short one by one thread, a longer one by
// binary lifting over the vertices (v is on it iff its root is r and
// succ^L(v) = v, at position (L - len(v)) mod L).
template <int C>
static __device__ void team_extract(Team<C> &tm, const TeamGraph &g, int r, int L, int *cycle_out) {
    const Workspace &ws = g.ws;
    const int n = g.n;
    if (L <= kChainLen) {
        if (tm.tid == 0) follow_cycle(ws, r, L, cycle_out);
        return;
    }
    int *cur = ws.aprev, *J = reinterpret_cast<int *>(ws.jm[0]), *J2 = reinterpret_cast<int *>(ws.jm[1]);
    for (int v = tm.tid; v < n; v += tm.W) {
        cur[v] = v;
        J[v] = ws.succ[v];
    }
    tm.sync();
    for (int b = 0; (L >> b) != 0; ++b) {
        for (int v = tm.tid; v < n; v += tm.W) {
            if ((L >> b) & 1) cur[v] = J[cur[v]];
            J2[v] = J[J[v]];
        }
        tm.sync();
        int *t = J;
        J = J2;
        J2 = t;
    }
    int found = 0;
    for (int v = tm.tid; v < n; v += tm.W) {
        const JLS s = ws.jls[0][v];
        if (~s.J == r && s.len < L && cur[v] == v) {
            cycle_out[s.len == 0 ? 0 : L - s.len] = ws.pi[v];
            ++found;
        }
    }
    found = tm.sum(found);
    if (tm.tid == 0) ws.ctrl->cnt[0] = found;
}

template <int C>
__global__ void __launch_bounds__(kTeamThreads, 1)
solve_team_kernel(const int *__restrict__ row_ptr, const int *__restrict__ col,
                  const int *__restrict__ w, int sign, int n, int m, const int *init,
                  long long max_iters, int *cycle_out, int room, Workspace ws) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ TeamShared s_team;
    Ctrl *c = ws.ctrl;
    Team<C> tm;
    for (int i = threadIdx.x; i < (int)(sizeof(Ctrl) / 4); i += blockDim.x)
        if (C == 1 || cluster_rank() == 0) reinterpret_cast<int *>(c)[i] = 0;
    tm.init(&s_team);
    if (!team_check<C>(tm, row_ptr, n, m, c) ||
        !team_init<C>(tm, row_ptr, col, w, sign, n, init, ws)) {
        tm.sync();   // (the first block's shared memory stays until all are done)
        return;
    }
    // (the exactness bound, 2 n^2 max|w| < 2^62, holds up to kTeamSolveN vertices;
    // one block's states are in shared memory, see launch_solve_team)
    bool in_shared;
    const TeamGraph g = team_place<C>(s_dyn, row_ptr, col, w, sign, 0, n, ws, room, &in_shared);
    int it = 0;
    long long switched = 0;
    bool capped = false;
    const bool ok =
        team_iterate<C, C == 1>(tm, g, init != nullptr, max_iters, &it, &switched, &capped);
    if (tm.tid == 0 && capped) c->not_converged = 1;
    if (ok) {
        const unsigned long long packed = *reinterpret_cast<volatile unsigned long long *>(g.best);
        const int r = INT_MAX - (int)(unsigned)(packed & 0xffffffffu);
        const int i = ws.cid_of_root[r];
        const int L = ws.cyc_L[i];
        if (tm.tid == 0) {
            c->res_root = r;
            c->res_len = L;
            c->res_num = ws.cyc_p[i];
            c->res_den = ws.cyc_q[i];
            c->res_cycles = tm.sh->nrep;
            c->iter = it;
            c->switched_total = switched;
            c->rounds_detect = it + 1;
            c->items_detect = (long long)n * (it + 1);
        }
        team_extract<C>(tm, g, r, L, cycle_out);
    }
    tm.sync();
}

bool team_solves(int n, int m) { return n <= kTeamSolveN && m <= 8LL * n + 1024; }

namespace {

template <int C>
int launch_team(int threads, int room, const int *row_ptr, const int *col, const int *w, int sign,
                int n, int m, const int *init, long long max_iters, int *cycle_out,
                const Workspace &ws, cudaStream_t st) {
    if (cudaFuncSetAttribute(solve_team_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kTeamBytes) != cudaSuccess ||
        (C > 8 && cudaFuncSetAttribute(solve_team_kernel<C>,
                                       cudaFuncAttributeNonPortableClusterSizeAllowed,
                                       1) != cudaSuccess))
        return -1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = room;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, solve_team_kernel<C>, row_ptr, col, w, sign, n, m, init,
                              max_iters, cycle_out, room, ws) == cudaSuccess ? 1 : -1;
}

}  // namespace

int launch_solve_team(const int *row_ptr, const int *col, const int *w, int sign, int n, int m,
                      const int *init, long long max_iters, int *cycle_out, Workspace ws,
                      cudaStream_t st) {
    // (the states of one block's graph in shared memory: see team_place).  The
    // teams were the fastest of 1 to 16 blocks of 128 to 1,024 threads at their
    // sizes: below 512 vertices more warps only wait for each other (257: 155 us
    // with 256 threads, 164 with 1,024), from 1,100 vertices on one block takes
    // longer than eight (351 against 325), from 4,500 on eight than 16 (684 / 622).
    if (n <= 512)
        return launch_team<1>(256, kTeamBytes, row_ptr, col, w, sign, n, m, init, max_iters,
                              cycle_out, ws, st);
    if (n <= kTeamBlockN)
        return launch_team<1>(1024, kTeamBytes, row_ptr, col, w, sign, n, m, init, max_iters,
                              cycle_out, ws, st);
    if (n <= 4096)
        return launch_team<8>(512, 0, row_ptr, col, w, sign, n, m, init, max_iters, cycle_out, ws,
                              st);
    return launch_team<16>(n <= 8192 ? 512 : 1024, 0, row_ptr, col, w, sign, n, m, init, max_iters,
                           cycle_out, ws, st);
}

}  // namespace ocm
