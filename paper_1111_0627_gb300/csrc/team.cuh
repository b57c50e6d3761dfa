// team.cuh -- a whole Howard iteration (Alg. 1: evaluate the policy, improve
// it, stop when stable) of one graph by one team of threads: a block (C == 1)
// or a cluster of C blocks, with block or cluster barriers only -- no grid
// barrier and no launch per iteration.  Every step computes what the
// whole-grid kernels compute (evaluate.cu, sweep.cu), with the same order and
// tie rules (cycle root = smallest vertex, V = q*S - p*len, key q_t*s*w(e) +
// V(t) compared within equal mean rank, strict switching, ties to the smaller
// edge index), so the policies are the ones the oracle goes through.
//
// State lives in the workspace at the graph's own vertex range [v0, v1), or,
// for graphs that fit, in the block's shared memory.
#pragma once

#include <climits>

#include "common.cuh"
#include "grid_sync.cuh"

namespace ocm {

constexpr int kTeamThreads = 1024;   // largest block
constexpr int kSU = 4;   // vertices per thread per pass of a jump round (64 registers)
// Dynamic shared memory of a team's block: the frontier bitmap, then the policy
// states and in their place, once the cycles are known, the records (16 bytes a
// vertex), or the bitmaps of the jump rounds.
constexpr int kTeamBytes = 196608;
constexpr int team_bitmap_bytes(int n) { return ((n + 31) / 32 * 4 + 15) / 16 * 16; }
constexpr int kTeamSharedN = 12192;   // largest graph whose states fit beside the bitmap
static_assert(team_bitmap_bytes(kTeamSharedN) + 16 * kTeamSharedN <= kTeamBytes &&
                  team_bitmap_bytes(kTeamSharedN + 1) + 16 * (kTeamSharedN + 1) > kTeamBytes,
              "kTeamSharedN");

// Evaluation by walks (team_walk): steps between two published parts and between
// two looks for a new cycle, the most steps of a walk and of a sample, new cycles
// a warp looks for, and the number of detection rounds up to which the policy
// counts as shallow enough.
constexpr int kTeamPart = 8;
constexpr int kTeamTight = 32;
// (states in shared memory: jump rounds take 40-80 us there, and so does a walk of
// some 100 steps with its looks; 1,024 graphs of up to 200,000 vertices, whose
// states are in global memory, took 79 ms with the smaller limits, 72 with these)
constexpr int team_steps(bool sm) { return sm ? 128 : 256; }
constexpr int team_seed_steps(bool sm) { return sm ? 256 : 512; }
constexpr int kTeamCycles = 8;
constexpr int kTeamPublish = 1 << 22;   // longest published part (times team_steps: an int)
constexpr int kTeamWalkRounds = 9;
constexpr int kTeamFirstRounds = 12;   // (before any was dropped)
constexpr int kTeamMarkLen = 256;   // longest cycle whose vertices are tagged
constexpr int kTeamRankSplit = 512;  // cycles from which several threads rank one

static __device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// What the team's blocks share, in the shared memory of its first block.
struct TeamShared {
    int sum[3];
    int nrep;
    int quit;
    int task;
};

template <int C>
struct Team {
    TeamShared *sh;   // the first block's
    int tid;          // in the team
    int round;        // sums taken so far
    int W;            // its threads

    __device__ __forceinline__ void init(TeamShared *own) {
        tid = threadIdx.x;
        W = C * (int)blockDim.x;
        sh = own;
        if (threadIdx.x < 3) own->sum[threadIdx.x] = 0;
        if (C > 1) {
            tid += (int)(cluster_rank() * blockDim.x);
            unsigned long long p;
            asm volatile("mapa.u64 %0, %1, 0;" : "=l"(p) : "l"((unsigned long long)own));
            sh = reinterpret_cast<TeamShared *>(p);
        }
        round = 0;
        sync();
    }
    __device__ __forceinline__ void sync() const {
        if (C == 1) {
            __syncthreads();
        } else {
            asm volatile("barrier.cluster.arrive.release.aligned;\n"
                         "barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
    // Sum of x over the team, and a barrier.  Three slots in turn: the slot of
    // the next sum is cleared here, after everybody has read it (two barriers
    // ago) and before anybody adds to it (after this one).
    __device__ __forceinline__ int sum(int x) {
        const int k = round % 3;
        round = (round + 1) % 3;
        x = __reduce_add_sync(0xffffffffu, x);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(&sh->sum[k], x);
        if (tid == 0) sh->sum[round] = 0;
        sync();
        return *reinterpret_cast<volatile int *>(&sh->sum[k]);
    }
};

// The graph a team works on.  st, rec and old are indexed by vertex - v0.
struct TeamGraph {
    const int *row_ptr, *col, *w;
    int sign;
    int v0, n;
    JLS *st;
    Rec *rec;             // the records the sweep gathers (in shared memory: st's place)
    Rec *old;             // the records kept until the next evaluation
    unsigned *dirty;      // n bits: records the last evaluation changed (nullptr: no room)
    unsigned *bits;       // bitmaps of the jump rounds (nullptr: no trimming)
    // the best cycle's (rank, INT_MAX - root).  In global memory: a 64-bit maximum
    // in another block's shared memory lost updates (32-bit counts there do not).
    unsigned long long *best;
    Workspace ws;
};

// Inclusive sum over the block (all threads call it).
static __device__ __forceinline__ int block_scan_incl(int x, int *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int wv = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wv, o);
            if (lane >= o) wv += y;
        }
        s_warp[lane] = wv;
    }
    __syncthreads();
    const int r = x + (warp > 0 ? s_warp[warp - 1] : 0);
    __syncthreads();
    return r;
}

// The root's cycle is a policy cycle: tag its vertices, so that the sweep can
// tell when one of them switches (team_switch).  Returns whether it is short
// enough to be tagged.
static __device__ __forceinline__ bool team_tag_cycle(const Workspace &ws, int r) {
    int y = r, k = 0;
    do {
        ws.cyc_tag[y] = r + 1;
        y = ws.succ[y];
    } while (y != r && ++k < kTeamMarkLen);
    return y == r;
}

// root_mark of a vertex.  Settled before the walks: kRootOld, root of a tagged
// cycle; kRootSeed, the same of a cycle too long to be tagged (known to this
// evaluation only).  Found and settled while others walk: kRootNew, kRootLong.
enum : int { kRootOld = 1, kRootNew = 2, kRootLong = 4, kRootSeed = 5 };

// cur lies on a policy cycle: its smallest vertex, which the first to come
// lists as a root (*first); -1 if the cycle is longer than limit.
template <int C>
static __device__ __forceinline__ int team_list_cycle(const Team<C> &tm, const TeamGraph &g,
                                                      int cur, int limit, bool *first) {
    const Workspace &ws = g.ws;
    int r = cur, k = 0;
    for (int y = ws.succ[cur]; y != cur && k < limit; y = ws.succ[y], ++k) r = min(r, y);
    *first = false;
    if (k >= limit) return -1;
    if (atomicCAS(&ws.root_mark[r], 0, kRootNew) == 0) {
        *first = true;
        const int pos = g.v0 + atomicAdd(&tm.sh->nrep, 1);
        ws.cyc_root[pos] = r;
        ws.cid_of_root[r] = pos;
    }
    return r;
}

// Evaluation by walks: every vertex follows its policy path to a settled vertex
// (state {~root, len, S}) and settles itself, as in walk_kernel of evaluate.cu.
// States hold one step each, or the settled root of a cycle no switch broke,
// when it starts.
//   seed: first a sample of the vertices, one per thread, walks, every lane
// looking for a cycle as it goes (Brent: keep the vertex passed after 2^k - 1
// steps and notice when it comes back).  The samples meet every cycle with more
// than a few vertices behind it, and their roots are settled before the rest
// starts.  (A walk that passes a root before it is settled goes round once too
// often and has to add its steps up again: with a thread for 10 to 200
// vertices, and settled vertices all around, that took five times the walk
// itself.)
//   rest: what remains walks to the settled vertices, 4 steps on average.  A
// walk still open after kTeamPart steps publishes the part it has walked, so that
// those behind it take it in one step; after kTeamTight (and twice, four times as
// many) one lane of its warp looks for a cycle the samples missed, and a vertex
// that ends at such a root adds its steps up again, to the first time its path
// meets it.
//   giving up: one vertex left open sends all to the jump rounds, so the first
// warp to leave one tells the others.  A cycle of 2,852 in 3,000 vertices, solved
// by one block: 1.75 ms with every warp walking to the end and looking eight
// times, 0.59 now, 0.53 with jump rounds alone.

// The seed phase, after which `kept` old roots and the new ones are listed;
// returns their number, the same in every thread (the shared counter may be
// raised by those already walking), or -1 where an eighth of the samples met
// neither a settled vertex nor a cycle: too deep to walk.
template <int C, bool SM>
static __device__ __forceinline__ int team_seed(Team<C> &tm, const TeamGraph &g, JLS *st,
                                                int kept) {
    const Workspace &ws = g.ws;
    const int i = g.n <= tm.W ? tm.tid : (int)((long long)tm.tid * g.n / tm.W);
    const int v = g.v0 + min(i, g.n - 1);
    int cur = v, tort = v, lam = 0, power = 1, len = 0;
    long long S = 0;
    bool cycle = false, first = false;
    JLS s = load_state<SM>(&st[cur]);
    for (int k = 0; k < team_seed_steps(SM) && s.J >= 0; ++k) {
        len += s.len;
        S += s.S;
        cur = s.J;
        if (cur == tort) {
            cycle = true;
            break;
        }
        if (++lam == power) {
            tort = cur;
            power <<= 1;
            lam = 0;
        }
        s = load_state<SM>(&st[cur]);
    }
    if (cycle) team_list_cycle<C>(tm, g, cur, team_seed_steps(SM), &first);
    else if (s.J < 0 && len > 0) store_state<SM>(&st[v], JLS{s.J, len + s.len, S + s.S});
    // (both counts are at most the team's 16,384 threads)
    const int both = tm.sum((int)first + ((tm.tid < g.n && !cycle && s.J >= 0) << 16));
    const int fresh = both & 0xffff;
    if ((both >> 16) > tm.W >> 3) return -1;
    const int seeded = kept + fresh;
    if (fresh) {
        for (int k = kept + tm.tid; k < seeded; k += tm.W) {
            const int r = ws.cyc_root[g.v0 + k];
            store_state<SM>(&st[r], JLS{~r, 0, 0});
            ws.root_mark[r] = kRootOld;
        }
        tm.sync();
        // (tagged while the others go on)
        for (int k = kept + tm.tid; k < seeded; k += tm.W) {
            const int r = ws.cyc_root[g.v0 + k];
            if (!team_tag_cycle(ws, r)) ws.root_mark[r] = kRootSeed;
        }
    }
    return seeded;
}

// Both phases on one copy of the states, the first `kept` roots being listed
// and settled; returns the vertices left open.
template <int C, bool SM>
static __device__ __forceinline__ int team_walk(Team<C> &tm, const TeamGraph &g, int kept) {
    const Workspace &ws = g.ws;
    const int lane = threadIdx.x & 31;
    JLS *st = g.st - g.v0;
    const int v1 = g.v0 + g.n;
    bool first = false;
    volatile int *quit = &tm.sh->quit;   // a warp gave up
    const int seeded = team_seed<C, SM>(tm, g, st, kept);
    if (seeded < 0) return g.n;
    const int root0 = seeded > 0 ? ws.cyc_root[g.v0] : -1;
    int left = 0;
    for (int base = g.v0 + tm.tid - lane; base < v1; base += tm.W) {
        const int v = base + lane;
        const bool on = v < v1;
        JLS s{-1, 0, 0};
        if (on) s = load_state<SM>(&st[v]);
        int cur = v, len = 0;
        long long S = 0;
        int total = 0, found = 0;
        unsigned open;   // lanes still walking
        for (;;) {
#pragma unroll 1
            for (int k = 0; k < kTeamPart && __any_sync(0xffffffffu, s.J >= 0); ++k) {
                if (s.J >= 0) {
                    len += s.len;
                    S += s.S;
                    cur = s.J;
                    s = load_state<SM>(&st[cur]);
                }
            }
            open = __ballot_sync(0xffffffffu, s.J >= 0);
            if (!open) break;
            total += kTeamPart;
            if (total >= team_steps(SM)) break;
            if (s.J >= 0 && len <= kTeamPublish) store_state<SM>(&st[v], JLS{cur, len, S});
            if (total < kTeamTight || (total & (total - 1))) continue;   // (looks after 32, 64, 128)
            if (__any_sync(0xffffffffu, *quit)) break;   // (the whole warp or none of it)
            int r = -1;
            if (lane == __ffs(open) - 1) {
                // (policy edges, not states: those may skip ahead)
                int y = cur, tort = cur, lam = 0, power = 1;
                bool cycle = false;
                for (int k = 0; k < 2 * total; ++k) {
                    y = ws.succ[y];
                    if (y == tort) {
                        cycle = true;
                        break;
                    }
                    if (++lam == power) {
                        tort = y;
                        power <<= 1;
                        lam = 0;
                    }
                    if (load_state<SM>(&st[y]).J < 0) break;
                }
                if (cycle) r = team_list_cycle<C>(tm, g, y, 2 * total, &first);
                if (r >= 0 && first) {
                    if (!team_tag_cycle(ws, r)) ws.root_mark[r] = kRootLong;
                    // (its vertices take single steps again: a published part
                    // may go round the cycle without ever stopping at the root;
                    // nothing is settled by it before the root is, here)
                    for (y = ws.succ[r]; y != r; y = ws.succ[y])
                        store_state<SM>(&st[y], JLS{ws.succ[y], 1, (long long)ws.wpi[y]});
                    __threadfence();   // (before anything that follows from the root)
                    store_state<SM>(&st[r], JLS{~r, 0, 0});
                }
            }
            r = __reduce_max_sync(0xffffffffu, r);
            if (r >= 0) {
                if (++found > kTeamCycles) break;
                if (s.J >= 0) {   // from the start, the root being settled now
                    cur = v;
                    len = 0;
                    S = 0;
                    s = JLS{ws.succ[v], 1, (long long)ws.wpi[v]};
                }
            }
        }
        if (on && s.J < 0) {
            const int root = ~s.J;
            JLS f{s.J, len + s.len, S + s.S};
            if (root == v) {
                f = JLS{~v, 0, 0};
            } else if (root != root0 && !(ws.root_mark[root] & 1)) {
                // found on the way: passed before it was settled?
                int y = v, k = 0;
                long long Sy = 0;
                while (k < f.len && y != root) {
                    Sy += ws.wpi[y];
                    y = ws.succ[y];
                    ++k;
                }
                if (y == root) f = JLS{~root, k, Sy};
                __threadfence();   // (after the cycle's states were put back, above)
            }
            store_state<SM>(&st[v], f);
        }
        left += on && s.J >= 0;
        if (open) {   // (what one leaves open sends all to the jump rounds)
            *quit = 1;
            break;
        }
    }
    return tm.sum(left);
}

// Evaluation by jump rounds, the steps of evaluate_kernel over every vertex
// that is no leaf in every round: cycle detection by doubling with window
// minima, resolved vertices holding J = ~root; then value propagation with
// (len, S) until the root.  States are final in g.st, roots listed in cyc_root
// from v0.  Returns the detection rounds, or -1 on an error.
template <int C>
static __device__ int team_jump(Team<C> &tm, const TeamGraph &g) {
    const int n = g.n, v0 = g.v0, v1 = g.v0 + g.n;
    const Workspace &ws = g.ws;
    int lg = 0;
    while ((1 << lg) < n) ++lg;
    Ctrl *c = ws.ctrl;
    const int Wt = tm.W;
    // Vertices nobody points to (leaves), and those whose predecessors are
    // all leaves, lie on no cycle and no other vertex jumps to them: when the
    // graph's bitmaps fit in shared memory the others are renumbered densely
    // (rank in the "has a predecessor that is no leaf" bitmap) and the jump
    // rounds run on that dense space; the leaves take their successor's final
    // state at the end.
    const int nw = (n + 31) / 32;
    const bool trim = C == 1 && g.bits != nullptr;
    unsigned *bits = g.bits, *keepb = bits + nw, *pref = bits + 2 * nw;
    int nk = n;
    if (trim) {
        for (int i = threadIdx.x; i < 2 * nw; i += Wt) bits[i] = 0u;
        __syncthreads();
        for (int v = v0 + (int)threadIdx.x; v < v1; v += Wt) {
            const int l = ws.succ[v] - v0;
            atomicOr(&bits[l >> 5], 1u << (l & 31));
        }
        __syncthreads();
        for (int v = v0 + (int)threadIdx.x; v < v1; v += Wt) {
            const int lv = v - v0;
            if ((bits[lv >> 5] >> (lv & 31)) & 1u) {
                const int l = ws.succ[v] - v0;
                atomicOr(&keepb[l >> 5], 1u << (l & 31));
            }
        }
        __syncthreads();
        const int per = (nw + Wt - 1) / Wt;
        const int w0 = min(nw, (int)threadIdx.x * per), w1 = min(nw, w0 + per);
        int sum = 0;
        for (int i = w0; i < w1; ++i) sum += __popc(keepb[i]);
        __shared__ int s_warp[32];
        __shared__ int s_total;
        const int incl = block_scan_incl(sum, s_warp);
        int run = incl - sum;
        for (int i = w0; i < w1; ++i) {
            pref[i] = (unsigned)run;
            run += __popc(keepb[i]);
        }
        if (threadIdx.x == Wt - 1) s_total = incl;
        __syncthreads();
        nk = s_total;
    }
    auto dense = [&](int v) -> int {
        const int l = v - v0;
        return trim ? (int)pref[l >> 5] + __popc(keepb[l >> 5] & ((1u << (l & 31)) - 1u)) : l;
    };
    auto kept = [&](int v) -> bool {
        const int l = v - v0;
        return !trim || ((keepb[l >> 5] >> (l & 31)) & 1u);
    };
    auto leaf1 = [&](int v) -> bool {
        const int l = v - v0;
        return trim && !((bits[l >> 5] >> (l & 31)) & 1u);
    };
    int *orig = ws.aprev + v0;    // dense index -> vertex
    int *ap = ws.list[0] + v0;    // previous window minimum, per dense index
    // ---- cycle detection on the dense space (window minima of vertex ids)
    JM *X = ws.jm[0] + v0, *Y = ws.jm[1] + v0;
    for (int v = v0 + tm.tid; v < v1; v += Wt) {
        if (!kept(v)) continue;
        const int d = dense(v);
        orig[d] = v;
        X[d] = JM{dense(ws.succ[v]), v};
    }
    tm.sync();
    int rounds = 0;
    for (int r = 0;; ++r) {
        int pend = 0;
        for (int base = tm.tid; base < nk; base += kSU * Wt) {
            JM sj[kSU], tj[kSU];
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int d = base + u * Wt;
                sj[u] = d < nk ? X[d] : JM{-1, 0};
            }
#pragma unroll
            for (int u = 0; u < kSU; ++u)
                if (sj[u].J >= 0) tj[u] = X[sj[u].J];
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int d = base + u * Wt;
                if (d >= nk) continue;
                if (sj[u].J < 0) { Y[d] = sj[u]; continue; }
                int root = -1;
                if (tj[u].J < 0) root = ~tj[u].J;
                else if (r > 0 && tj[u].M == ap[d]) root = tj[u].M;
                if (root >= 0) { Y[d] = JM{~root, 0}; ws.rep[orig[d]] = root; }
                else { Y[d] = JM{tj[u].J, min(sj[u].M, tj[u].M)}; ap[d] = tj[u].M; ++pend; }
            }
        }
        JM *tmp = X; X = Y; Y = tmp;
        rounds = r + 1;
        if (tm.sum(pend) == 0) break;
        if (r + 1 > lg + 4) { if (tm.tid == 0) atomicOr(&c->err, kErrDetect); return -1; }
    }
    // ---- values on the dense space, the root terminal (final J = ~root)
    JLS *A = ws.jls[1] + v0, *B = reinterpret_cast<JLS *>(ws.scratch16) + v0;
    for (int d = tm.tid; d < nk; d += Wt) {
        const int v = orig[d];
        const int root = ws.rep[v];
        JLS st;
        if (root == v) {
            st = JLS{~v, 0, 0};
            const int i = v0 + atomicAdd(&tm.sh->nrep, 1);
            ws.cyc_root[i] = v;
            ws.cid_of_root[v] = i;
        } else {
            const int sv = ws.succ[v];
            st = ws.rep[sv] == sv ? JLS{~sv, 1, (long long)ws.wpi[v]}
                                  : JLS{dense(sv), 1, (long long)ws.wpi[v]};
        }
        A[d] = st;
    }
    tm.sync();
    for (int r = 0;; ++r) {
        int pend = 0;
        for (int base = tm.tid; base < nk; base += kSU * Wt) {
            JLS sj[kSU], tj[kSU];
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int d = base + u * Wt;
                sj[u] = d < nk ? A[d] : JLS{-1, 0, 0};
            }
#pragma unroll
            for (int u = 0; u < kSU; ++u) if (sj[u].J >= 0) tj[u] = A[sj[u].J];
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int d = base + u * Wt;
                if (d >= nk) continue;
                if (sj[u].J < 0) { B[d] = sj[u]; continue; }
                const JLS nu{tj[u].J, sj[u].len + tj[u].len, sj[u].S + tj[u].S};
                B[d] = nu; pend += nu.J >= 0;
            }
        }
        JLS *tmp = A; A = B; B = tmp;
        if (tm.sum(pend) == 0) break;
        if (r + 1 > lg + 3) { if (tm.tid == 0) atomicOr(&c->err, kErrValue); return -1; }
    }
    // the leaves' bitmaps lie where g.st begins when that is in shared memory:
    // final states first in jls[0]
    JLS *fin = ws.jls[0] + v0;
    for (int d = tm.tid; d < nk; d += Wt) fin[orig[d] - v0] = A[d];
    tm.sync();
    // then the leaves: second level first, from their successors
    for (int pass = 0; pass < 2 && trim; ++pass) {
        for (int v = v0 + tm.tid; v < v1; v += Wt) {
            if (kept(v) || leaf1(v) != (pass == 1)) continue;
            const JLS f = fin[ws.succ[v] - v0];
            fin[v - v0] = JLS{f.J, f.len + 1, f.S + (long long)ws.wpi[v]};
        }
        tm.sync();
    }
    if (g.st != fin) {
        for (int i = tm.tid; i < n; i += Wt) g.st[i] = fin[i];
        tm.sync();
    }
    return rounds;
}

// Whether the next evaluation walks (else jump rounds): not for 0, 1, 3, 7 ..
// evaluations after walks that were dropped, counted from the last that were not.
struct TeamMode {
    bool walk;
    int tries, pause;
};

// Policy evaluation: states, cycle table, records {V, rank, q} (with mark: the
// bits of those that change; *n_dirty counts them).  The cycle records sit at
// [v0, v0 + K); the best (rank, INT_MAX - root) is in *g.best.  Returns
// false on an error (recorded in the control block).  tm.sh->nrep is 0 and
// every team thread is past a barrier when it is called.
template <int C, bool SM>
static __device__ bool team_evaluate(Team<C> &tm, const TeamGraph &g, TeamMode &mode, bool mark,
                                     int *n_dirty) {
    const Workspace &ws = g.ws;
    const int n = g.n, v0 = g.v0;
    const int W = tm.W;
    bool walked = false;
    if (mode.walk) {
        int kept = 0;   // roots whose cycle no switch broke
        for (int base = tm.tid; base < n; base += kSU * W) {
            int m[kSU], sv[kSU], wv[kSU];   // (loads of kSU vertices in flight)
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int i = base + u * W;
                m[u] = i < n ? ws.root_mark[v0 + i] : 0;
                sv[u] = i < n ? ws.succ[v0 + i] : 0;
                wv[u] = i < n ? ws.wpi[v0 + i] : 0;
            }
#pragma unroll
            for (int u = 0; u < kSU; ++u) {
                const int i = base + u * W, v = v0 + i;
                if (i >= n) continue;
                JLS s{sv[u], 1, (long long)wv[u]};
                const bool keep = m[u] == kRootOld || m[u] == kRootNew;
                if (keep) {   // its cycle still is one
                    const int pos = v0 + atomicAdd(&tm.sh->nrep, 1);
                    ws.cyc_root[pos] = v;
                    ws.cid_of_root[v] = pos;
                    s = JLS{~v, 0, 0};
                    ++kept;
                }
                if (m[u]) ws.root_mark[v] = keep ? kRootOld : 0;
                g.st[i] = s;
            }
        }
        if (tm.tid == 0) tm.sh->quit = 0;
        walked = team_walk<C, SM>(tm, g, tm.sum(kept)) == 0;
        if (!walked) mode.pause = (1 << mode.tries) - 1;
        mode.tries = walked ? 0 : min(mode.tries + 1, 20);
        if (!walked) {
            if (tm.tid == 0) tm.sh->nrep = 0;
            tm.sync();
        }
    } else if (mode.pause > 0) {
        --mode.pause;
    }
    if (!walked) {
        for (int i = tm.tid; i < n; i += W) ws.root_mark[v0 + i] = 0;
        const int rounds = team_jump<C>(tm, g);
        if (rounds < 0) return false;
        mode.walk = mode.pause == 0 && rounds <= (mode.tries ? kTeamWalkRounds : kTeamFirstRounds);
        // (the next evaluation walks from these cycles' roots)
        if (mode.walk) {
            const int K = *reinterpret_cast<volatile int *>(&tm.sh->nrep);
            for (int i = tm.tid; i < K; i += W) {
                const int r = ws.cyc_root[v0 + i];
                if (team_tag_cycle(ws, r)) ws.root_mark[r] = kRootNew;
            }
        }
    }
    // ---- cycles: mean W/L reduced, exact key, rank among this graph's cycles
    const int K = *reinterpret_cast<volatile int *>(&tm.sh->nrep);
    const long long N2 = (long long)n * n;
    for (int i = v0 + tm.tid; i < v0 + K; i += W) {
        const int r = ws.cyc_root[i];
        const JLS s = g.st[ws.succ[r] - v0];
        const long long Wc = (long long)ws.wpi[r] + s.S;
        const long long L = 1 + (long long)s.len;
        const long long d = gcd_ll(Wc, L);
        ws.cyc_p[i] = Wc / d;
        ws.cyc_q[i] = (int)(L / d);
        ws.cyc_L[i] = (int)L;
        ws.cyc_rank[i] = 0;
        if (K > 1) ws.cyc_key[i] = mean_key(Wc / d, L / d, N2);
        else *g.best = (unsigned)(INT_MAX - r);
    }
    if (mark)
        for (int i = tm.tid; i < (n + 31) / 32; i += W) g.dirty[i] = 0u;
    if (K > 1 && tm.tid == 0) *g.best = 0;
    tm.sync();
    // ranks: number of smaller keys.  Many cycles but at most half the threads:
    // several threads a cycle, each with a part of the keys (4,000 cycles in
    // 16,000 vertices, 16 blocks: 1.10 ms a solve, 2.31 with one thread each)
    const int parts = K >= kTeamRankSplit ? W / K : 1;
    if (parts > 1) {
        const int part = tm.tid / K, i = v0 + tm.tid % K;
        if (part < parts) {
            const long long key = ws.cyc_key[i];
            const int j1 = v0 + (int)((long long)(part + 1) * K / parts);
            int cnt = 0;
#pragma unroll 4
            for (int j = v0 + (int)((long long)part * K / parts); j < j1; ++j)
                cnt += ws.cyc_key[j] < key;
            if (cnt) atomicAdd(&ws.cyc_rank[i], cnt);
        }
        tm.sync();
    }
    if (K > 1) {
        unsigned long long top = 0;
        for (int i = v0 + tm.tid; i < v0 + K; i += W) {
            int rank = 0;
            if (parts > 1) {
                rank = ws.cyc_rank[i];
            } else {
                const long long key = ws.cyc_key[i];
                for (int j = v0; j < v0 + K; ++j) rank += ws.cyc_key[j] < key;
                ws.cyc_rank[i] = rank;
            }
            top = max(top, ((unsigned long long)(unsigned)rank << 32) |
                               (unsigned)(INT_MAX - ws.cyc_root[i]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if ((threadIdx.x & 31) == 0 && top) atomicMax(g.best, top);
        tm.sync();
    }
    // ---- materialise the records the sweep gathers
    const long long p1 = ws.cyc_p[v0];
    const int q1 = ws.cyc_q[v0];
    int changed = 0;
    for (int base = tm.tid; base < n; base += kSU * W) {
        JLS s[kSU];
        Rec old[kSU];
        int k[kSU];
#pragma unroll
        for (int u = 0; u < kSU; ++u) {
            const int i = base + u * W;
            if (i < n) {
                s[u] = g.st[i];
                if (mark) old[u] = g.old[i];
            }
        }
#pragma unroll
        for (int u = 0; u < kSU; ++u)
            k[u] = K > 1 && base + u * W < n ? ws.cid_of_root[~s[u].J] : v0;
#pragma unroll
        for (int u = 0; u < kSU; ++u) {
            const int i = base + u * W;
            if (i >= n) continue;
            const long long p = K > 1 ? ws.cyc_p[k[u]] : p1;
            const int q = K > 1 ? ws.cyc_q[k[u]] : q1;
            Rec rec;
            rec.V = (long long)q * s[u].S - p * (long long)s[u].len;
            rec.rank = K > 1 ? ws.cyc_rank[k[u]] : 0;
            rec.q = q;
            if (mark && (old[u].V != rec.V || old[u].rank != rec.rank || old[u].q != rec.q)) {
                atomicOr(&g.dirty[i >> 5], 1u << (i & 31));
                ++changed;
            }
            if (SM) {
                ws.jls[0][v0 + i] = s[u];   // (kept for the extraction)
                g.rec[i] = rec;
            }
            g.old[i] = rec;
        }
    }
    if (mark) *n_dirty = tm.sum(changed);   // (its barrier ends the pass)
    else tm.sync();
    return true;
}

// Switch decision of vertex v given the best candidate and the candidate of
// its current policy edge (strict improvement, Alg. 1).
static __device__ __forceinline__ int team_switch(const TeamGraph &g, int v, const Cand &best,
                                                  const Cand &own) {
    const Workspace &ws = g.ws;
    if (own.e == INT_MAX) {
        atomicOr(&ws.ctrl->err, kErrSweep);
        return 0;
    }
    if (best.rank > own.rank || (best.rank == own.rank && best.key > own.key)) {
        ws.pi[v] = best.e;
        ws.succ[v] = g.col[best.e];
        ws.wpi[v] = g.sign * g.w[best.e];
        // on a tagged cycle: that is no cycle any more (a tag left from an
        // earlier one may unmark a cycle that is; it is then found anew)
        const int t = ws.cyc_tag[v];
        if (t) ws.root_mark[t - 1] = 0;
        return 1;
    }
    return 0;
}

static __device__ __forceinline__ bool target_changed(const TeamGraph &g, int t) {
    const int l = t - g.v0;
    return (g.dirty[l >> 5] >> (l & 31)) & 1u;
}

static __device__ __forceinline__ Cand team_cand(const TeamGraph &g, int e, int t, int x) {
    const Rec r = g.rec[t - g.v0];
    return Cand{r.rank, e, (long long)r.q * (long long)(g.sign * x) + r.V};
}

// One improvement sweep (the candidate order of improve_kernel): a thread per
// vertex of out-degree <= 32, four edges in flight; a warp per vertex with
// more (lanes stride its edges, shuffles combine); returns the number of
// switches.  frontier: a vertex none of whose targets' records changed in the
// last evaluation would choose as in the last sweep, and is skipped.
template <int C>
static __device__ int team_sweep(Team<C> &tm, const TeamGraph &g, bool frontier) {
    int sw = 0;
    bool heavy = false;
    const int v1 = g.v0 + g.n;
    const int *__restrict__ row_ptr = g.row_ptr;
    const int *__restrict__ col = g.col;
    const int *__restrict__ w = g.w;
    for (int v = g.v0 + tm.tid; v < v1; v += tm.W) {
        const int a = row_ptr[v], b = row_ptr[v + 1];
        if (b - a > 32) {
            heavy = true;
            continue;
        }
        if (frontier) {
            bool any = false;
            for (int e = a; e < b && !any; ++e) any = target_changed(g, col[e]);
            if (!any) continue;
        }
        const int pv = g.ws.pi[v];
        Cand best{INT_MIN, INT_MAX, LLONG_MIN};
        Cand own{INT_MIN, INT_MAX, LLONG_MIN};
        for (int e0 = a; e0 < b; e0 += 4) {
            int t[4], x[4];
            Cand cd[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                t[u] = e0 + u < b ? col[e0 + u] : -1;
                x[u] = e0 + u < b ? w[e0 + u] : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                cd[u] = t[u] >= 0 ? team_cand(g, e0 + u, t[u], x[u])
                                  : Cand{INT_MIN, INT_MAX, LLONG_MIN};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (cd[u].e == pv) own = cd[u];
                if (better(cd[u], best)) best = cd[u];
            }
        }
        sw += team_switch(g, v, best, own);
    }
    if (__syncthreads_or(heavy)) {   // (each block its own vertices)
        const int lane = threadIdx.x & 31;
        for (int base = g.v0 + tm.tid - lane; base < v1; base += tm.W) {
            const int mine = base + lane;
            unsigned todo = __ballot_sync(0xffffffffu,
                                          mine < v1 && row_ptr[mine + 1] - row_ptr[mine] > 32);
            for (; todo; todo &= todo - 1u) {
                const int v = base + __ffs(todo) - 1;
                const int a = row_ptr[v], b = row_ptr[v + 1];
                if (frontier) {
                    bool any = false;
                    for (int e = a + lane; e < b && !any; e += 32) any = target_changed(g, col[e]);
                    if (!__any_sync(0xffffffffu, any)) continue;
                }
                const int pv = g.ws.pi[v];
                Cand best{INT_MIN, INT_MAX, LLONG_MIN};
                Cand own{INT_MIN, INT_MAX, LLONG_MIN};
                for (int e = a + lane; e < b; e += 32) {
                    const Cand x = team_cand(g, e, col[e], w[e]);
                    if (e == pv) own = x;
                    if (better(x, best)) best = x;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    Cand y;
                    y.rank = __shfl_xor_sync(0xffffffffu, best.rank, o);
                    y.e = __shfl_xor_sync(0xffffffffu, best.e, o);
                    y.key = __shfl_xor_sync(0xffffffffu, best.key, o);
                    if (better(y, best)) best = y;
                    Cand z;
                    z.rank = __shfl_xor_sync(0xffffffffu, own.rank, o);
                    z.e = __shfl_xor_sync(0xffffffffu, own.e, o);
                    z.key = __shfl_xor_sync(0xffffffffu, own.key, o);
                    if (z.e != INT_MAX) own = z;   // one lane met the policy edge
                }
                if (lane == 0) sw += team_switch(g, v, best, own);
            }
        }
    }
    return tm.sum(sw);
}

// Places states, records and bitmaps in `room` bytes of dynamic shared memory
// (see kTeamBytes): *in_shared tells whether the states are in shared memory.
template <int C>
static __device__ __forceinline__ TeamGraph team_place(unsigned char *dyn, const int *row_ptr,
                                                       const int *col, const int *w, int sign,
                                                       int v0, int n, const Workspace &ws,
                                                       int room, bool *in_shared) {
    TeamGraph g{row_ptr, col, w, sign, v0, n, ws.jls[0] + v0, ws.rec + v0, ws.rec + v0,
                nullptr, nullptr, reinterpret_cast<unsigned long long *>(ws.recp + v0), ws};
    *in_shared = false;
    const long long nw = (n + 31) / 32;
    const long long d = team_bitmap_bytes(n);   // the frontier bitmap
    if (C > 1) {
        g.dirty = reinterpret_cast<unsigned *>(ws.list[1] + v0);
    } else if (d <= room) {
        g.dirty = reinterpret_cast<unsigned *>(dyn);
        if (d + 12 * nw <= room) g.bits = reinterpret_cast<unsigned *>(dyn + d);
        if (n <= kTeamSharedN) {
            *in_shared = true;
            g.st = reinterpret_cast<JLS *>(dyn + d);
            g.rec = reinterpret_cast<Rec *>(g.st);
        }
    }
    return g;
}

// All iterations of the graph.  Returns false on an error, or when the
// iteration cap was reached (*capped); *iters counts the improving sweeps.
// On success the final states are in jls[0] at the vertices' own indices.
template <int C, bool SM>
static __device__ bool team_iterate(Team<C> &tm, const TeamGraph &g, bool warm,
                                    long long max_iters, int *iters, long long *switched,
                                    bool *capped) {
    const int n = g.n;
    TeamMode mode{warm, 0, 0};
    int last_sw = n;
    long long it = 0, total = 0;
    *capped = false;
    if (tm.tid == 0) tm.sh->nrep = 0;
    tm.sync();
    for (;;) {
        // the frontier form: once the last sweep switched fewer than n/8
        // vertices, the record pass marks the records it changes, and the
        // sweep looks only at vertices with a changed target when fewer than
        // n/4 changed
        const bool mark = g.dirty != nullptr && it > 0 && last_sw < (n >> 3);
        int n_dirty = n;
        if (!team_evaluate<C, SM>(tm, g, mode, mark, &n_dirty)) return false;
        last_sw = team_sweep<C>(tm, g, mark && n_dirty < (n >> 2));
        total += last_sw;
        if (last_sw == 0) break;
        if (++it >= max_iters) {
            *capped = true;
            return false;
        }
        if (tm.tid == 0) tm.sh->nrep = 0;
        tm.sync();
    }
    *iters = (int)it;
    *switched = total;
    return true;
}

}  // namespace ocm
