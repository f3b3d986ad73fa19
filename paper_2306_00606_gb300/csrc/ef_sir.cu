// SIR epidemic simulation of libef (Section 3.1's model; Section 3.2's
// measurements: final size, global outbreaks, epidemic length, time to
// peak, and the spreading power of order k from the infection tree).
//
// Discrete time, synchronous steps t = 0, 1, ... on the states at the start
// of the step:
//   - every node u infected at the start of step t tries once each neighbour
//     x susceptible at that time, with success when the draw
//     R(sim, t, u, x) < floor(beta 2^32); x becomes infected at the end of
//     the step when any try succeeds, its infector being the smallest such u;
//   - u recovers at the end of step t when R(sim, t, u, 2^32 - 1) <
//     floor(gamma 2^32);
//   - the epidemic ends at the first t with no infected node (its length).
// R is Philox4x32-10 (Salmon et al., SC 2011) with counter (sim, t, u, x)
// and key = the 64-bit seed, first output word: a simulation's course
// depends on its id and the seed only, not on the batch or the launch.
//
// Layout, node-major: a batch of B <= SIR_BATCH simulations runs together,
// and each node keeps WB = ceil(B / 32) words of one bit per simulation:
// susceptible, infected at the start of the step (inf[cur]), infected at the
// start of the next (inf[nxt]), and infected during this step (newinf).  A
// node infected in any simulation is in the step's frontier once; its
// neighbour list is read once for all simulations, and for a neighbour x
// the words inf[cur][u] & susc[x] say which simulations try the edge, the
// words read by consecutive lanes.  cand (node-major, x * B + s) holds the
// smallest successful infector of the step, parent (simulation-major, the
// output layout) the infection tree.
//
// A step works in one of two directions, chosen on the device from the rows
// of its frontier (sir_dense); both make the same draws and the same choices.
//   push   (few infected nodes) every frontier node tries its neighbours:
//     k_sir_step        a warp per frontier node: recovery draws (slot 0),
//                       then (slot, word) lanes over the neighbours; nodes of
//                       degree > SIR_HEAVY are listed for
//     k_sir_step_hub    a CTA per listed node over its neighbours
//     k_sir_commit      per node with a success: new infections, parents
//   pull   (dense frontier) every node looks at its own neighbours, so it
//     alone writes its words and its parents: no atomics on global memory, no
//     cand.  k_sir_step takes a warp per node, k_sir_step_hub a CTA per hub.
// then
//   k_sir_clear       zeroes the frontier's inf[cur] words for reuse
//   k_sir_stats       per simulation: peak, its step, length
// Lists are deduplicated by per-node step stamps, per-simulation counts are
// summed in shared memory per block, and the host reads whether any
// simulation is still running every SIR_CHECK steps.
#include "ef_internal.cuh"

#include <algorithm>

namespace ef {

constexpr int32_t NO_CAND = 0x7fffffff;
constexpr uint32_t RECOVER_WORD = 0xffffffffu;
constexpr int SIR_HEAVY = 256;   // frontier nodes of higher degree take a CTA each
constexpr int SIR_WARPS = 8;     // warps per block of the step kernels
constexpr int SIR_NODES = 8;     // consecutive nodes per warp step (pull)

// Direction of step t: pull once the frontier's nodes hold half of all row
// entries, a third from eight words of simulations on (flen: its length, and
// those entries).  A pull step reads every node's row and a word row per entry
// whatever the frontier holds; a push step reads those of the frontier and
// costs a round trip to memory per successful try.  The entries, not the
// nodes, say what a push costs: where degrees are uneven, few nodes hold most of
// them.  Whole calls, gamma = 1/3, R0 = 1.3, in ms, push only / a half / a third /
// a quarter, and by the number of nodes (one in 8 from 8 words on, else one in
// 2): BA 500k with 512 simulations 82.1 / 36.2 / 35.9 / 36.0 and 36.6; ER 500k
// with 250 42.5 / 41.4 / 40.5 / 42.1 and 45.4, with 130 24.9 / 25.1 / 25.1 / 28.4
// and 24.8; ER 100k with 250 12.6 / 12.7 / 13.2 / 13.7 and 14.4; a half / a third:
// ER 300k of degree 10 with 211 26.0 / 26.9 and 25.8, BA 300k with 260 20.3 /
// 20.2 and 20.5, with 40 7.7 / 7.4 and 8.0.
__device__ __forceinline__ bool sir_dense(const SirState &st, int t) {
    return (int64_t)(uint32_t)st.flen[t & 1].y * (st.WB >= 8 ? 3 : 2) > st.m;
}

// Room for len nodes with the given row entries in all in the frontier nx, for
// one lane: their first position.  One atomic on the pair.
__device__ __forceinline__ int front_room(const SirState &st, int nx, int len, int entries) {
    return (int)(uint32_t)atomicAdd(reinterpret_cast<unsigned long long *>(st.flen + nx),
                                    (unsigned long long)(uint32_t)entries << 32 | (uint32_t)len);
}

// Philox4x32-10, first output word only.
__device__ __forceinline__ uint32_t philox_w0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint64_t key) {
    uint32_t k0 = (uint32_t)key, k1 = (uint32_t)(key >> 32);
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    return c0;
}

// Lane geometry of a warp over (slot, word) pairs: wbp = WB rounded up to a
// power of two, 32 / wbp slots (nodes or neighbours) per warp.
struct SirLanes {
    int wbp, slots, slot, w;
    bool wv;
    __device__ __forceinline__ explicit SirLanes(int WB) {
        wbp = 1;
        while (wbp < WB) wbp <<= 1;
        slots = 32 / wbp;
        const int lane = threadIdx.x & 31;
        slot = lane / wbp;
        w = lane % wbp;
        wv = w < WB;
    }
};

// Append v, of D row entries, to the frontier nx unless it is there (stamp);
// the lanes that get here together share an atomic (one each: 5% of a call
// whose steps push).
__device__ __forceinline__ void front_append(const SirState &st, int nx, int v, int D, int stamp) {
    if (atomicExch(st.fmark + v, stamp) == stamp) return;
    const unsigned act = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(act) - 1;
    const int entries = __reduce_add_sync(act, D);
    int pos = 0;
    if (lane == leader) pos = front_room(st, nx, __popc(act), entries);
    pos = __shfl_sync(act, pos, leader);
    st.front[nx][pos + __popc(act & ((1u << lane) - 1u))] = v;
}

__global__ void k_sir_fill(int32_t *__restrict__ a, int64_t len, int32_t value) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = value;
}

// Susceptibility words: every simulation but those whose immune set holds v.
__global__ void k_sir_init_susc(int32_t n, const uint8_t *__restrict__ immune, int32_t num_sets,
                                const int32_t *__restrict__ imm_set, SirState st) {
    const int64_t words = (int64_t)n * st.WB;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (int64_t)gridDim.x * blockDim.x) {
        const int v = (int)(i / st.WB), w = (int)(i - (int64_t)v * st.WB);
        uint32_t word = 0;
        for (int b = 0; b < 32; ++b) {
            const int s = w * 32 + b;
            if (s >= st.B) break;
            int set = imm_set ? imm_set[s] : -1;
            if (set >= num_sets) {
                atomicOr(st.err, ERRB_SIR_ARG);
                set = -1;
            }
            if (set < 0 || !immune[(int64_t)set * n + v]) word |= 1u << b;
        }
        st.susc[i] = word;
    }
}

// The index cases and the first frontier (an immune index case is an error).
__global__ void k_sir_seed(const int32_t *__restrict__ rp, const int32_t *__restrict__ index_cases, int32_t n,
                           SirState st) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < st.B; s += gridDim.x * blockDim.x) {
        const int u = index_cases[s];
        st.peak[s] = 1;
        st.peak_step[s] = 0;
        st.length[s] = 0;
        st.count[s] = 1;
        st.fsize[s] = 1;
        st.done[s] = 0;
        const uint32_t bit = 1u << (s & 31);
        if (u < 0 || u >= n || !(st.susc[(int64_t)u * st.WB + (s >> 5)] & bit)) {
            atomicOr(st.err, ERRB_SIR_ARG);
            st.done[s] = 1;
            st.count[s] = 0;
            st.fsize[s] = 0;
            continue;
        }
        atomicAnd(st.susc + (int64_t)u * st.WB + (s >> 5), ~bit);   // index cases may share a node
        atomicOr(st.inf[0] + (int64_t)u * st.WB + (s >> 5), bit);
        st.parent[(int64_t)s * n + u] = u;
        front_append(st, 0, u, rp[u + 1] - rp[u], -1);
    }
}

// Tries of u's infected simulations (its inf[cur] words iw) over the
// neighbours k_first, k_first + stride, ... (the warp's slots taking
// consecutive neighbours).
// The loads of SIR_UNROLL neighbours are issued before any of their tries.
constexpr int SIR_UNROLL = 4;
__device__ __forceinline__ void sir_tries(const int32_t *__restrict__ ci, int a, int D, int u, int t, uint32_t iw,
                                          const SirLanes &L, int k_first, int stride, const SirStep &p,
                                          const SirState &st) {
    for (int k0 = k_first; k0 < D; k0 += SIR_UNROLL * stride) {
        int x[SIR_UNROLL];
        uint32_t act[SIR_UNROLL];
#pragma unroll
        for (int q = 0; q < SIR_UNROLL; ++q) {
            const int k = k0 + q * stride + L.slot;
            x[q] = k < D ? ci[a + k] : -1;
        }
#pragma unroll
        for (int q = 0; q < SIR_UNROLL; ++q)
            act[q] = x[q] >= 0 && L.wv ? iw & st.susc[(int64_t)x[q] * st.WB + L.w] : 0u;
#pragma unroll
        for (int q = 0; q < SIR_UNROLL; ++q) {
            uint32_t m = act[q];
            while (m) {
                const int b = __ffs(m) - 1;
                m &= m - 1;
                const int s = L.w * 32 + b;
                const uint32_t r =
                    philox_w0((uint32_t)(p.sim_base + s), (uint32_t)t, (uint32_t)u, (uint32_t)x[q], p.seed);
                if ((uint64_t)r < p.beta_thr && atomicMin(st.cand + (int64_t)x[q] * st.B + s, u) == NO_CAND) {
                    atomicOr(st.newinf + (int64_t)x[q] * st.WB + L.w, 1u << b);
                    if (atomicExch(st.tmark + x[q], t + 1) != t + 1) st.touched[atomicAdd(st.counts, 1)] = x[q];
                }
            }
        }
    }
}

// ------------------------------------------------------------------- pull
// The draws of a warp's nodes, tries and recoveries, queued in shared memory
// so that a Philox evaluation has a draw in every lane (a lane's own bits one
// after the other left five of six lanes idle): lanes append one of their
// bits a round, and every 32 queued draws are evaluated together.
struct SirQueue {
    int32_t u[64], x[64], e[64];   // infector; node; slot of SirNode | SIR_RECOVER
};
constexpr int SIR_RECOVER = 1 << 30;

// What the draws brought, per (node of the warp step, simulation): new
// infections and recoveries, and the smallest infector (NO_CAND when none).
struct SirNode {
    int32_t best[SIR_BATCH];
    uint32_t newb[SIR_BATCH / 32], recb[SIR_BATCH / 32];
};

struct SirDraw {
    SirQueue &Q;
    SirNode &N;
    const SirStep &p;
    int t, smask, len;   // smask: simulations per node, rounded up to a power of two, minus 1

    // Evaluates the first cnt (<= 32) queued draws and drops them.
    __device__ __forceinline__ void evaluate(int cnt) {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        if (lane < cnt) {
            const int u = Q.u[lane], e = Q.e[lane], i = e & (SIR_BATCH - 1);
            const bool rec = (e & SIR_RECOVER) != 0;
            const uint32_t r = philox_w0((uint32_t)(p.sim_base + (i & smask)), (uint32_t)t, (uint32_t)u,
                                         rec ? RECOVER_WORD : (uint32_t)Q.x[lane], p.seed);
            if ((uint64_t)r < (rec ? p.gamma_thr : p.beta_thr)) {
                atomicOr((rec ? N.recb : N.newb) + (i >> 5), 1u << (i & 31));
                if (!rec) atomicMin(N.best + i, u);
            }
        }
        len -= cnt;
        int u = 0, x = 0, e = 0;
        if (lane < len) {
            u = Q.u[lane + cnt];
            x = Q.x[lane + cnt];
            e = Q.e[lane + cnt];
        }
        __syncwarp();
        if (lane < len) {
            Q.u[lane] = u;
            Q.x[lane] = x;
            Q.e[lane] = e;
        }
    }
    // Queues a draw for every bit of every lane's word (word i of SirNode, infector u, node x).
    __device__ __forceinline__ void add(uint32_t word, int i, int u, int x, int flag) {
        const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
        for (;;) {
            const unsigned has = __ballot_sync(FULL, word != 0u);
            if (!has) break;
            if (word) {
                const int k = len + __popc(has & lt);   // len < 32, so k < 64
                Q.u[k] = u;
                Q.x[k] = x;
                Q.e[k] = (i * 32 + __ffs(word) - 1) | flag;
                word &= word - 1u;
            }
            len += __popc(has);
            if (len >= 32) evaluate(32);
        }
    }
    __device__ __forceinline__ void flush() {
        if (len) evaluate(len);
        __syncwarp();
    }
};

// Lane geometry of a pull step: (node, slot, word), slots taking a node's
// neighbours; few words leave room for several nodes per warp.
struct PullLanes {
    int wbp, slots, nodes;   // powers of two with wbp * slots * nodes = 32
    int node, slot, w, i;    // i: the lane's word of SirNode
    bool wv;
    __device__ __forceinline__ PullLanes(int WB, int max_slots) {
        wbp = 1;
        while (wbp < WB) wbp <<= 1;
        slots = min(32 / wbp, max_slots);
        nodes = 32 / (wbp * slots);
        const int lane = threadIdx.x & 31;
        w = lane % wbp;
        slot = lane / wbp % slots;
        node = lane / (wbp * slots);
        i = node * wbp + w;
        wv = w < WB;
    }
};

// Neighbours a lane loads together.
constexpr int PULL_UNROLL = 4;

// The words and the first neighbours of the lane's node, loaded ahead.
struct PullNode {
    int x, a, D;
    uint32_t iw, sx;
    int u[PULL_UNROLL];
    uint32_t act[PULL_UNROLL];
    // own words and neighbour ids from entry k0 on (D = 0: none)
    __device__ __forceinline__ void ids(const int32_t *__restrict__ ci, const PullLanes &L, int k0, int stride) {
#pragma unroll
        for (int q = 0; q < PULL_UNROLL; ++q) {
            const int k = k0 + q * stride + L.slot;
            u[q] = k < D ? ci[a + k] : -1;
        }
    }
    __device__ __forceinline__ void own(const PullLanes &L, int c, const SirState &st) {
        const bool v = D >= 0 && L.wv;
        const int64_t j = (int64_t)x * st.WB + L.w;
        iw = v ? st.inf[c][j] : 0u;
        sx = v ? st.susc[j] : 0u;
    }
    __device__ __forceinline__ void words(const PullLanes &L, int c, const SirState &st) {
#pragma unroll
        for (int q = 0; q < PULL_UNROLL; ++q)
            act[q] = u[q] >= 0 && L.wv ? st.inf[c][(int64_t)u[q] * st.WB + L.w] : 0u;
    }
    __device__ __forceinline__ void tries(const PullLanes &L, SirDraw &W) const {
#pragma unroll
        for (int q = 0; q < PULL_UNROLL; ++q) W.add(act[q] & sx, L.i, u[q], x, 0);
    }
};

// Writes a node's words and parents after its draws; the lanes of slot 0 hold
// (node, word).  True in lanes whose node is infected in one of the word's
// simulations at the start of the next step.
__device__ __forceinline__ bool sir_pull_commit(const PullNode &P, int32_t n, int nx, const PullLanes &L,
                                                const SirState &st, SirNode &N, int32_t *s_new, int32_t *s_rec) {
    uint32_t next = 0;
    if (L.slot == 0 && L.wv && P.D >= 0) {
        const uint32_t nb = N.newb[L.i], rb = N.recb[L.i];
        N.newb[L.i] = 0;
        N.recb[L.i] = 0;
        const int64_t j = (int64_t)P.x * st.WB + L.w;
        if (nb) st.susc[j] = P.sx & ~nb;
        next = (P.iw & ~rb) | nb;
        if (next) st.inf[nx][j] = next;
        for (uint32_t m = nb; m; m &= m - 1u) {
            const int b = __ffs(m) - 1, s = L.w * 32 + b;
            st.parent[(int64_t)s * n + P.x] = N.best[L.i * 32 + b];
            N.best[L.i * 32 + b] = NO_CAND;
            atomicAdd(s_new + s, 1);
        }
        for (uint32_t m = rb; m; m &= m - 1u) atomicAdd(s_rec + L.w * 32 + __ffs(m) - 1, 1);
    }
    __syncwarp();
    return next != 0u;
}

// Adds a block's per-simulation counts (all threads).
__device__ __forceinline__ void sir_counts(const SirState &st, const int32_t *s_new, const int32_t *s_rec) {
    __syncthreads();
    for (int s = threadIdx.x; s < st.B; s += blockDim.x) {
        const int a = s_new ? s_new[s] : 0, r = s_rec[s];
        if (a != r) atomicAdd(st.count + s, a - r);
        if (a) atomicAdd(st.fsize + s, a);
    }
}

// Neighbours beside each other in a warp's lanes in a pull step, and the nodes
// that this leaves room for (as PullLanes).
constexpr int PULL_SLOTS = 8;
static int pull_nodes(int WB) {
    int wbp = 1;
    while (wbp < WB) wbp <<= 1;
    return 32 / (wbp * std::min(32 / wbp, PULL_SLOTS));
}

// One step.  Push: recoveries of the frontier front[cur], survivors into
// inf[nxt] and front[nxt], tries of the nodes of degree <= SIR_HEAVY.  Pull:
// the nodes of degree <= SMALL_MAX in node order, a software pipeline of
// three stages per warp: a node's row and words, its neighbours' words, its draws.
__global__ void __launch_bounds__(SIR_WARPS * 32, 4) k_sir_step(const int32_t *__restrict__ rp,
                                                                const int32_t *__restrict__ ci, int32_t n,
                                                                int32_t t, int steps, SirStep p, SirState st,
                                                                const int32_t *__restrict__ bins,
                                                                const int32_t *__restrict__ cnt) {
    __shared__ int32_t s_rec[SIR_BATCH], s_new[SIR_BATCH];
    extern __shared__ unsigned char sir_smem[];
    SirNode *s_node = reinterpret_cast<SirNode *>(sir_smem);   // per warp
    SirQueue *s_q = reinterpret_cast<SirQueue *>(s_node + SIR_WARPS);
    const int c = t & 1, nx = c ^ 1, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int total = st.flen[c].x;
    const int64_t nwarps = (int64_t)gridDim.x * SIR_WARPS, warp = (int64_t)blockIdx.x * SIR_WARPS + wid;
    if (total == 0) return;
    for (int i = threadIdx.x; i < st.B; i += blockDim.x) s_rec[i] = s_new[i] = 0;
    const bool pull = sir_dense(st, t);
    if (pull) {
        for (int i = lane; i < SIR_BATCH; i += 32) s_node[wid].best[i] = NO_CAND;
        s_node[wid].newb[lane] = s_node[wid].recb[lane] = 0;
    }
    __syncthreads();
    if (!pull) {
        const SirLanes L(st.WB);
        for (int64_t i = warp; i < total; i += nwarps) {
            const int u = st.front[c][i];
            const int a = rp[u], D = rp[u + 1] - a;
            const uint32_t iw = L.wv ? st.inf[c][(int64_t)u * st.WB + L.w] : 0u;
            uint32_t sv = iw;
            if (L.slot == 0 && L.wv) {
                uint32_t m = iw;
                while (m) {
                    const int b = __ffs(m) - 1;
                    m &= m - 1;
                    const int s = L.w * 32 + b;
                    const uint32_t r =
                        philox_w0((uint32_t)(p.sim_base + s), (uint32_t)t, (uint32_t)u, RECOVER_WORD, p.seed);
                    if ((uint64_t)r < p.gamma_thr) {
                        sv &= ~(1u << b);
                        atomicAdd(s_rec + s, 1);
                    }
                }
                st.inf[nx][(int64_t)u * st.WB + L.w] = sv;
            }
            const bool survives = __any_sync(FULL, L.slot == 0 && sv != 0u);
            if (survives && lane == 0) front_append(st, nx, u, D, t + 1);
            if (D > SIR_HEAVY) {
                if (lane == 0) st.heavy[atomicAdd(st.counts + 1, 1)] = u;
                continue;
            }
            sir_tries(ci, a, D, u, t, iw, L, 0, L.slots, p, st);
        }
        sir_counts(st, nullptr, s_rec);
        return;
    }
    const PullLanes L(st.WB, PULL_SLOTS);
    SirDraw W{s_q[wid], s_node[wid], p, t, L.wbp * 32 - 1, 0};
    const int per = steps * L.nodes;   // consecutive nodes of a warp step, L.nodes at a time
    const unsigned mine = (L.wbp * L.slots == 32 ? FULL : (1u << L.wbp * L.slots) - 1u) << L.node * L.wbp * L.slots;
    for (int64_t base = warp * per; base < n; base += nwarps * per) {
        const int64_t v = base + lane;
        const int r0 = lane < per && v < n ? rp[v] : 0, r1 = lane < per && v < n ? rp[v + 1] : 0;
        const int groups = (int)min((int64_t)steps, (n - base + L.nodes - 1) / L.nodes);
        // row and own words of group g (D = -1: no node, or one of the lists below)
        auto start = [&](int g) {
            PullNode P;
            const int k = min(g, steps - 1) * L.nodes + L.node;
            P.a = __shfl_sync(FULL, r0, k);
            P.D = __shfl_sync(FULL, r1, k) - P.a;
            P.x = (int)base + k;
            if (g >= groups || base + k >= n || P.D > SMALL_MAX) P.D = -1;
            P.own(L, c, st);
            P.ids(ci, L, 0, L.slots);
            return P;
        };
        unsigned ahead = 0;   // nodes of the next frontier, by position in the warp step
        PullNode P0 = start(0);
        P0.words(L, c, st);
        PullNode P1 = start(1);
        for (int g = 0; g < groups; ++g) {
            P1.words(L, c, st);
            PullNode P2 = start(g + 2);
            W.add(L.slot == 0 ? P0.iw : 0u, L.i, P0.x, P0.x, SIR_RECOVER);
            P0.tries(L, W);
            // rows longer than the words loaded ahead
            const int longest = __reduce_max_sync(FULL, P0.D);
            for (int k0 = PULL_UNROLL * L.slots; k0 < longest; k0 += PULL_UNROLL * L.slots) {
                P0.ids(ci, L, k0, L.slots);
                P0.words(L, c, st);
                P0.tries(L, W);
            }
            W.flush();
            const unsigned inf = __ballot_sync(FULL, sir_pull_commit(P0, n, nx, L, st, s_node[wid], s_new, s_rec));
            const unsigned node = __ballot_sync(FULL, L.slot == 0 && L.w == 0 && (inf & mine) != 0u);
            // first lanes of the group's infected nodes -> positions in the warp step
            for (int i = 0; i < L.nodes; ++i)
                if (node >> (i * L.wbp * L.slots) & 1u) ahead |= 1u << (g * L.nodes + i);
            P0 = P1;
            P1 = P2;
        }
        if (ahead) {
            const int entries = __reduce_add_sync(FULL, ahead >> lane & 1u ? r1 - r0 : 0);
            int pos = 0;
            if (lane == 0) pos = front_room(st, nx, __popc(ahead), entries);
            pos = __shfl_sync(FULL, pos, 0);
            if (ahead >> lane & 1u) st.front[nx][pos + __popc(ahead & ((1u << lane) - 1u))] = (int)base + lane;
        }
    }
    // rows of degree 33 .. hub_min - 1, a warp each, from the degree pass's
    // list (in node order a run of them falls to one warp: preferential
    // attachment numbers its large nodes together, 0.5 ms a step)
    const PullLanes L1(st.WB, 32);
    W.smask = L1.wbp * 32 - 1;
    const int mids = mid_total(cnt);
    for (int64_t it = warp; it < mids; it += nwarps) {
        PullNode P;
        P.x = mid_node(bins, n, cnt, (int)it);
        P.a = rp[P.x];
        P.D = rp[P.x + 1] - P.a;
        P.own(L1, c, st);
        W.add(L1.slot == 0 ? P.iw : 0u, L1.i, P.x, P.x, SIR_RECOVER);
        if (__any_sync(FULL, P.sx != 0u))
            for (int k0 = 0; k0 < P.D; k0 += PULL_UNROLL * L1.slots) {
                P.ids(ci, L1, k0, L1.slots);
                P.words(L1, c, st);
                P.tries(L1, W);
            }
        W.flush();
        const bool inf = sir_pull_commit(P, n, nx, L1, st, s_node[wid], s_new, s_rec);
        if (__any_sync(FULL, inf) && lane == 0) st.front[nx][front_room(st, nx, 1, P.D)] = P.x;
    }
    sir_counts(st, s_new, s_rec);
}

// Push: the listed frontier nodes' tries; pull: the hubs (degree >= hub_min,
// from the degree pass's lists).  A CTA per node.
constexpr int SIR_HUB_WARPS = 32;
__global__ void __launch_bounds__(SIR_HUB_WARPS * 32) k_sir_step_hub(const int32_t *__restrict__ rp,
                                                                     const int32_t *__restrict__ ci, int32_t n,
                                                                     int32_t t, SirStep p, SirState st,
                                                                     const int32_t *__restrict__ bins,
                                                                     const int32_t *__restrict__ cnt) {
    const int c = t & 1, nx = c ^ 1, wid = threadIdx.x >> 5;
    if (st.flen[c].x == 0) return;
    if (!sir_dense(st, t)) {
        const SirLanes L(st.WB);
        const int total = st.counts[1];
        for (int i = blockIdx.x; i < total; i += gridDim.x) {
            const int u = st.heavy[i];
            const int a = rp[u], D = rp[u + 1] - a;
            const uint32_t iw = L.wv ? st.inf[c][(int64_t)u * st.WB + L.w] : 0u;
            sir_tries(ci, a, D, u, t, iw, L, wid * L.slots, SIR_HUB_WARPS * L.slots, p, st);
        }
        return;
    }
    const int total = hub_total(cnt);
    if ((int)blockIdx.x >= total) return;
    __shared__ int32_t s_rec[SIR_BATCH], s_new[SIR_BATCH];
    __shared__ SirQueue s_q[SIR_HUB_WARPS];
    __shared__ SirNode s_node;
    const PullLanes L(st.WB, 32);   // one node per warp
    for (int i = threadIdx.x; i < SIR_BATCH; i += blockDim.x) {
        s_rec[i] = s_new[i] = 0;
        s_node.best[i] = NO_CAND;
    }
    if (threadIdx.x < 32) s_node.newb[threadIdx.x] = s_node.recb[threadIdx.x] = 0;
    SirDraw W{s_q[wid], s_node, p, t, L.wbp * 32 - 1, 0};
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        __syncthreads();
        PullNode P;
        P.x = hub_row(bins, n, cnt, it);
        P.a = rp[P.x];
        P.D = rp[P.x + 1] - P.a;
        P.own(L, c, st);
        if (wid == 0) W.add(L.slot == 0 ? P.iw : 0u, L.i, P.x, P.x, SIR_RECOVER);
        if (__any_sync(FULL, P.sx != 0u))
            for (int k0 = wid * L.slots; k0 < P.D; k0 += PULL_UNROLL * SIR_HUB_WARPS * L.slots) {
                P.ids(ci, L, k0, SIR_HUB_WARPS * L.slots);
                P.words(L, c, st);
                P.tries(L, W);
            }
        W.flush();
        __syncthreads();
        if (wid == 0) {
            const bool inf = sir_pull_commit(P, n, nx, L, st, s_node, s_new, s_rec);
            if (__any_sync(FULL, inf) && threadIdx.x == 0) st.front[nx][front_room(st, nx, 1, P.D)] = P.x;
        }
    }
    sir_counts(st, s_new, s_rec);
}

// New infections of the step: per node with a success, its newinf words.
__global__ void __launch_bounds__(256) k_sir_commit(const int32_t *__restrict__ D, int32_t n, int32_t t,
                                                    SirState st) {
    __shared__ int s_new[SIR_BATCH];
    if (st.counts[0] == 0) return;   // also every pull step
    for (int i = threadIdx.x; i < st.B; i += blockDim.x) s_new[i] = 0;
    __syncthreads();
    const int nx = (t & 1) ^ 1;
    const SirLanes L(st.WB);
    const int total = st.counts[0];
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const unsigned mine = (L.wbp == 32 ? FULL : (1u << L.wbp) - 1u) << (L.slot * L.wbp);
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * L.slots; base < total;
         base += nwarps * L.slots) {
        const int64_t i = base + L.slot;
        const int x = i < total ? st.touched[i] : -1;
        const int Dx = x >= 0 && L.w == 0 ? D[x] : 0;
        uint32_t nb = 0;
        if (x >= 0 && L.wv) {
            const int64_t j = (int64_t)x * st.WB + L.w;
            nb = st.newinf[j];
            if (nb) {
                st.newinf[j] = 0;
                st.susc[j] &= ~nb;
                st.inf[nx][j] |= nb;
                uint32_t m = nb;
                while (m) {
                    const int b = __ffs(m) - 1;
                    m &= m - 1;
                    const int s = L.w * 32 + b;
                    int32_t *cs = st.cand + (int64_t)x * st.B + s;
                    st.parent[(int64_t)s * n + x] = *cs;
                    *cs = NO_CAND;
                    atomicAdd(s_new + s, 1);
                }
            }
        }
        // the node joins the next frontier once (it may already be there as a survivor)
        const unsigned any = __ballot_sync(FULL, nb != 0u);
        if (L.w == 0 && (any & mine)) front_append(st, nx, x, Dx, t + 1);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < st.B; s += blockDim.x)
        if (s_new[s]) {
            atomicAdd(st.count + s, s_new[s]);
            atomicAdd(st.fsize + s, s_new[s]);
        }
}

// The frontier's words of inf[cur], zeroed: the buffer is the next step's inf[nxt].
__global__ void k_sir_clear(int32_t t, SirState st) {
    const int c = t & 1;
    const int64_t total = (int64_t)st.flen[c].x * st.WB;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int v = st.front[c][i / st.WB];
        st.inf[c][(int64_t)v * st.WB + (i % st.WB)] = 0u;
    }
}

// After step t: count[s] = infected at the start of step t + 1.  active[t & 1]
// counts warps with a simulation still running; the emptied lists and
// active[(t + 1) & 1] are cleared for the next step.
__global__ void k_sir_stats(int32_t t, SirState st, int64_t *__restrict__ active) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st.flen[t & 1] = make_int2(0, 0);
        st.counts[0] = st.counts[1] = 0;
        active[(t + 1) & 1] = 0;
    }
    int act = 0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < st.B; s += gridDim.x * blockDim.x) {
        if (st.done[s]) continue;
        const int cnt = st.count[s];
        if (cnt > st.peak[s]) {
            st.peak[s] = cnt;
            st.peak_step[s] = t + 1;
        }
        if (cnt == 0) {
            st.length[s] = t + 1;
            st.done[s] = 1;
        } else {
            act = 1;
        }
    }
    act = __reduce_or_sync(FULL, act);
    if ((threadIdx.x & 31) == 0 && act) atomicAdd((unsigned long long *)(active + (t & 1)), 1ull);
}

// Simulations still running after the last step: truncated at `steps`.
__global__ void k_sir_close(int32_t steps, SirState st, uint8_t *__restrict__ truncated) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < st.B; s += gridDim.x * blockDim.x) {
        const bool tr = !st.done[s];
        if (tr) st.length[s] = steps;
        if (truncated) truncated[s] = tr;
    }
}

// Spreading power: an infected non-root node v is a descendant of its g-th
// ancestor at generation g; exact[g-1][anc] counts those, over simulations
// with final size >= min_size.  infected[v] counts those simulations in
// which v was infected.
__global__ void k_sir_tree(int32_t n, int32_t depth, int32_t min_size, SirState st,
                           unsigned long long *__restrict__ exact, unsigned long long *__restrict__ infected) {
    const int s = blockIdx.y;
    if (st.fsize[s] < min_size) return;
    const int32_t *par = st.parent + (int64_t)s * n;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        if (par[v] < 0) continue;
        if (infected) atomicAdd(infected + v, 1ull);
        if (!exact) continue;
        int anc = v;
        for (int g = 0; g < depth; ++g) {
            const int p = par[anc];
            if (p == anc) break;
            atomicAdd(exact + (int64_t)g * n + p, 1ull);
            anc = p;
        }
    }
}

// spread[k-1][v] = sum over g <= k of exact[g-1][v], in place.
__global__ void k_sir_cumulate(int32_t n, int32_t depth, int64_t *__restrict__ spread) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        int64_t acc = 0;
        for (int g = 0; g < depth; ++g) {
            acc += spread[(int64_t)g * n + v];
            spread[(int64_t)g * n + v] = acc;
        }
    }
}

static inline unsigned grid_for(int64_t work, int per_block, int64_t cap) {
    int64_t g = (work + per_block - 1) / per_block;
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

int launch_sir_init(const int32_t *rp, const int32_t *index_cases, int32_t n, const uint8_t *immune, int32_t num_sets,
                    const int32_t *imm_set, const SirState &st, const Tune &t, cudaStream_t s) {
    const int64_t cap = (int64_t)t.num_sms * 32, nb = (int64_t)n * st.B;
    k_sir_fill<<<grid_for(nb, 256, cap), 256, 0, s>>>(st.cand, nb, NO_CAND);
    k_sir_fill<<<grid_for(nb, 256, cap), 256, 0, s>>>(st.parent, nb, -1);
    k_sir_init_susc<<<grid_for((int64_t)n * st.WB, 256, cap), 256, 0, s>>>(n, immune, num_sets, imm_set, st);
    k_sir_seed<<<grid_for(st.B, 256, cap), 256, 0, s>>>(rp, index_cases, n, st);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

constexpr size_t SIR_STEP_SMEM = SIR_WARPS * (sizeof(SirNode) + sizeof(SirQueue));
// Opt the step kernel in to its dynamic shared memory on the current device.
int prepare_sir() {
    return cudaFuncSetAttribute(k_sir_step, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)SIR_STEP_SMEM) == cudaSuccess
               ? 0
               : -1;
}

int launch_sir_step(const int32_t *rp, const int32_t *ci, int32_t n, int32_t step, const SirStep &p,
                    const SirState &st, int64_t *active, const Scratch &sc, const Tune &t, cudaStream_t s) {
    const unsigned g = (unsigned)t.num_sms * 8;
    // groups of nodes of a warp step of a pull: fewer than SIR_NODES where warps
    // would be left without one (a group waits for the one before; ER 2000 with
    // 512 simulations 6.0 -> 5.0 ms, BA 2000 4.6 -> 3.3)
    const int64_t warps = (int64_t)t.num_sms * 4 * SIR_WARPS, per = pull_nodes(st.WB);
    const int steps = (int)std::min<int64_t>(SIR_NODES, (n + warps * per - 1) / (warps * per));
    k_sir_step<<<(unsigned)t.num_sms * 4, SIR_WARPS * 32, SIR_STEP_SMEM, s>>>(rp, ci, n, step, steps, p, st, sc.bins,
                                                                             sc.counters);
    k_sir_step_hub<<<(unsigned)t.num_sms * 2, SIR_HUB_WARPS * 32, 0, s>>>(rp, ci, n, step, p, st, sc.bins, sc.counters);
    k_sir_commit<<<g, 256, 0, s>>>(sc.D, n, step, st);
    k_sir_clear<<<g, 256, 0, s>>>(step, st);
    k_sir_stats<<<grid_for(st.B, 256, (int64_t)t.num_sms * 4), 256, 0, s>>>(step, st, active);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_sir_close(int32_t steps, const SirState &st, uint8_t *truncated, const Tune &t, cudaStream_t s) {
    k_sir_close<<<grid_for(st.B, 256, (int64_t)t.num_sms * 4), 256, 0, s>>>(steps, st, truncated);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_sir_tree(int32_t n, int32_t depth, int32_t min_size, const SirState &st, int64_t *exact,
                    int64_t *infected, const Tune &t, cudaStream_t s) {
    const dim3 grid(grid_for(n, 256 * 4, 1 << 16), (unsigned)st.B);
    k_sir_tree<<<grid, 256, 0, s>>>(
        n, depth, min_size, st, reinterpret_cast<unsigned long long *>(exact),
        reinterpret_cast<unsigned long long *>(infected));
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_sir_cumulate(int32_t n, int32_t depth, int64_t *spread, const Tune &t, cudaStream_t s) {
    k_sir_cumulate<<<grid_for(n, 256, (int64_t)t.num_sms * 32), 256, 0, s>>>(n, depth, spread);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace ef
