// Pieces of steps 2-4: the per-file disagreement masks, the warp-wide
// maximum-clique search and the copy chosen for a file.
#pragma once

#include "aspis_internal.cuh"

namespace aspis {

constexpr uint32_t kDefaultNodeBudget = 1u << 20;   // per lane

// The workers of the pairs that differ in file word w disagree: their bits
// are set in the shared masks dis[] (one word per worker).
__device__ __forceinline__ void add_disagreements(uint32_t w, const uint8_t *fw_i, int r, uint32_t *dis)
{
    while (w) {
        int rem = __ffs(w) - 1;
        w &= w - 1;
        int s = 0;
        while (rem >= r - 1 - s) {
            rem -= r - 1 - s;
            ++s;
        }
        const int t = s + 1 + rem;
        const int a = fw_i[s], b = fw_i[t];
        // most pairs of colluders are seen many times: read before the atomic
        if (!((((volatile uint32_t *)dis)[a] >> b) & 1u)) atomicOr(&dis[a], 1u << b);
        if (!((((volatile uint32_t *)dis)[b] >> a) & 1u)) atomicOr(&dis[b], 1u << a);
    }
}

struct Frame {
    uint32_t R, P, X, cand;
};

struct CliqueResult {
    int omega;
    uint32_t n_max, first, nodes;
    bool over;
};

// All maximum cliques of the graph adj[0..K) (shared memory, bits >= K and
// self loops clear), by one full warp; the result is the same in all lanes.
// Lane v explores the cliques whose smallest vertex is v (R = {v}, P = later
// neighbours, X = earlier neighbours), so every maximal clique is reported by
// exactly one lane: Bron-Kerbosch with Tomita pivoting over 32-bit masks, an
// explicit stack in shared memory, pruning against the largest clique any
// lane has found, and a node budget per lane.
//
// CLOSE (symmetric graphs): vertices of P adjacent to all the rest of P lie
// in every maximal clique of the branch, so the pivot scan, which counts
// every vertex's neighbours in P anyway, moves them to R at once and keeps in
// X only their common neighbours.  The agreement graphs of attacks are nearly
// complete: a branch that took one node per clique member (up to K dependent
// pivot scans) is settled in one or two.  A round of 455 files and 36,928
// coordinates under the optimal attack went from 81.6 to 74.6 us.
template <bool CLOSE>
__device__ __forceinline__ CliqueResult max_cliques_warp(const uint32_t *adj, int K, uint32_t budget,
                                                         Frame (*stack)[32], int *shared_best)
{
    const int v = threadIdx.x & 31;
    int best = 0;
    uint32_t count = 0, first = 0xffffffffu, nodes = 0;
    bool over = false;
    if (v < K) {
        int sp = 0;
        auto report = [&](uint32_t R) {
            const int sz = __popc(R);
            if (sz > best) {
                best = sz;
                count = 1;
                first = R;
                atomicMax(shared_best, sz);
            } else if (sz == best) {
                ++count;
                if (R < first) first = R;
            }
        };
        // a child node: report it if maximal, else push it unless it cannot
        // reach the best size known to any lane
        auto visit = [&](uint32_t R, uint32_t P, uint32_t X) {
            while (true) {
                if (P == 0u) {
                    if (X == 0u) report(R);
                    return;
                }
                const int bound = max(best, *(volatile int *)shared_best);
                if (__popc(R) + __popc(P) < bound) return;
                // pivot: the vertex of P u X with most neighbours in P
                const int np1 = __popc(P) - 1;
                uint32_t PX = P | X, uni = 0u, common = 0xffffffffu;
                int piv = __ffs(PX) - 1, most = -1;
                while (PX) {
                    const int u = __ffs(PX) - 1;
                    PX &= PX - 1;
                    const uint32_t au = adj[u];
                    const int c = __popc(P & au);
                    if (c > most) {
                        most = c;
                        piv = u;
                    }
                    if (CLOSE && c == np1 && ((P >> u) & 1u)) {
                        uni |= 1u << u;
                        common &= au;
                    }
                }
                if (CLOSE && uni) {
                    R |= uni;
                    P &= ~uni;
                    X &= common;
                    continue;
                }
                stack[sp][v] = Frame{R, P, X, P & ~adj[piv]};
                ++sp;
                return;
            }
        };
        const uint32_t bit = 1u << v;
        visit(bit, adj[v] & ~(bit | (bit - 1u)), adj[v] & (bit - 1u));
        while (sp > 0) {
            Frame &fr = stack[sp - 1][v];
            if (fr.cand == 0u) {
                --sp;
                continue;
            }
            if (++nodes > budget) {
                over = true;
                break;
            }
            const int u = __ffs(fr.cand) - 1;
            const uint32_t ub = 1u << u;
            fr.cand &= ~ub;
            const uint32_t R = fr.R | ub, P = fr.P & adj[u], X = fr.X & adj[u];
            fr.P &= ~ub;
            fr.X |= ub;
            visit(R, P, X);
        }
    }
    __syncwarp();
    const unsigned full = 0xffffffffu;
    CliqueResult res;
    res.omega = __reduce_max_sync(full, best);
    res.n_max = __reduce_add_sync(full, best == res.omega ? count : 0u);
    res.first = __reduce_min_sync(full, (best == res.omega && count) ? first : 0xffffffffu);
    res.nodes = __reduce_add_sync(full, nodes);
    res.over = __any_sync(full, over);
    return res;
}

// Case 2: the lowest slot of the largest class of equal copies (ties to the
// class holding the lower slot); the class of slot s has 1 + the number of
// slots equal to it.
template <int R>
__device__ __forceinline__ int majority_slot(uint32_t w)
{
    int pick = 0, best = 0;
#pragma unroll
    for (int s = 0; s < R; ++s) {
        int size = 1, p = 0;
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
            for (int b = a + 1; b < R; ++b, ++p)
                if ((a == s || b == s) && !((w >> p) & 1u)) ++size;
        if (size > best) {
            best = size;
            pick = s;
        }
    }
    return pick;
}

// Step 4 for one file: the slot of its chosen copy, -1 if it is dropped.
template <int R>
__device__ __forceinline__ int chosen_slot(bool success, uint32_t clique, const uint8_t *fw_i, uint32_t w)
{
    int pick = -1;
    if (success) {
#pragma unroll
        for (int s = R - 1; s >= 0; --s)
            if ((clique >> fw_i[s]) & 1u) pick = s;
    } else {
        pick = majority_slot<R>(w);
    }
    return pick;
}

}  // namespace aspis
