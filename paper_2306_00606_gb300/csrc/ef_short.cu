// Short-row path of libef: graphs (or batches) in which no node has more than
// SMALL_MAX = 32 neighbours -- lattices, small-world ensembles, sparse random
// graphs.  One kernel takes the place of the orientation, the small wedge
// kernels and the pair tests, reads the graph once more and writes 8 bytes
// per node.
//
// A warp takes 32 consecutive nodes and packs their rows, whole, into its
// lanes (a row's lanes are consecutive, so the column reads are coalesced).
// Wedges: lane k of a middle node u owns u's neighbour x_k; the lanes' sums
// R_u(x_k) are those of k_wedge_small, term for term.  Triangles: packed again
// with the entries above u only, a suffix of the row (its position is in the
// node's word, left by the row pass); a triangle u < x < z is found once, by
// u's lane of x, as an entry z of x's suffix (held in registers) among u's.
// It brings each of its nodes 4 (f(s-6) - f(s-4)), an integer in units of
// 2^-F as in the pair tests, added to T in FP64, and one count.
//
// Why not the oriented pair tests: they need an oriented copy of the graph
// with hash tables (20 bytes per entry written, read again) and issue about
// 300 instructions per 32 tests to find each pair's lower end and list.  Here
// the order is the node id, so the lists are the CSR's own rows, and on rows
// this short a suffix is 4-6 entries in one or two sectors.
//
// Both phases are bound by instruction issue (77% of cycles).  Measured on
// the WS batch (4096 graphs, 4.1e7 nodes, 3.3e8 entries), FP32C: orientation +
// small wedges + pair tests 11.4 ms; this kernel 7.0 ms (8.4 ms
// a call, 13.4 before).
// Left out: membership in N(u) through a shared-memory hash table per row,
// triangles found at each of their nodes (10.1 ms); found at each of their
// nodes by comparing all neighbours with the suffix in the wedge loop (8.0 ms).
#include "ef_internal.cuh"

namespace ef {

constexpr int SH_WARPS = 8;
constexpr int SH_SUMS = 3 * SMALL_MAX + 1;
constexpr int SH_Z = 8;            // suffix entries held in registers at most

struct ShortArgs {
    const int32_t *ci;
    const int2 *info;              // {row start, short_word}
    int32_t n;
    int32_t per;                   // nodes per warp step (at most 32)
    double *Tacc;
    int32_t *tri;
    uint64_t *stat;
    double qscale;
};

template <bool F64>
struct ShortSmem {
    int64_t tq[SH_SUMS];           // corrections, and in natural units (FP64 stays out of the loops)
    double tqd[SH_SUMS];
    float2 f[F64 ? SH_SUMS : 1];
    int4 node[SH_WARPS][32];       // the warp's nodes with entries: {node, word, column index - position}
};

// One lane of a pack: entry x of node u's list (its first lane: first; cnt
// entries, 0 in an idle lane).
struct Pack {
    int u, uword, first, cnt, x;
    int cmin, cmax;                // shortest and longest list of the pack
};

// The warp's lists (lane v's: cnt entries at column index start), in shared
// memory, and their positions one after the other.
struct PackList {
    int cnt, pre, total;
    template <bool F64>
    __device__ __forceinline__ void load(ShortSmem<F64> &S, int v, int word, int start, int count) {
        const int lane = threadIdx.x & 31;
        cnt = count;
        int inc = count;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += y;
        }
        pre = inc - count;
        total = __shfl_sync(FULL, inc, 31);
        const unsigned some = __ballot_sync(FULL, count > 0);
        __syncwarp();   // the previous lists have been read
        if (count > 0)
            S.node[threadIdx.x >> 5][__popc(some & ((1u << lane) - 1u))] = make_int4(v, word, start - pre, 0);
        __syncwarp();
    }
    // The pack: the lists from position t0 on that fit into 32 lanes (at
    // least one: no list exceeds 32 entries); t0 and taken move past them.
    template <bool F64>
    __device__ __forceinline__ Pack next(const ShortSmem<F64> &S, const int32_t *ci, int &t0, int &taken) const {
        const int lane = threadIdx.x & 31;
        const unsigned le = 2u * (1u << lane) - 1u;
        Pack P;
        const int rel = pre - t0;
        const bool fits = cnt > 0 && rel >= 0 && rel + cnt <= 32;
        const unsigned heads = __reduce_or_sync(FULL, fits ? 1u << rel : 0u);
        const int used = __reduce_max_sync(FULL, fits ? rel + cnt : 0);
        P.cmax = __reduce_max_sync(FULL, fits ? cnt : 0);
        P.cmin = __reduce_min_sync(FULL, fits ? cnt : 32);
        const bool act = lane < used;
        const int4 nd = act ? S.node[threadIdx.x >> 5][taken + __popc(heads & le) - 1] : make_int4(0, 0, 0, 0);
        P.u = nd.x;
        P.uword = nd.y;
        P.x = act ? ci[nd.z + t0 + lane] : -1;
        P.first = act ? 31 - __clz(heads & le) : lane;
        const unsigned after = heads & ~le;   // the next list's first lane
        P.cnt = act ? (after ? __ffs(after) - 1 : used) - P.first : 0;
        t0 += used;
        taken += __popc(heads);
        return P;
    }
};

// Sum over the lanes of a list, in its lane k = 0 (strides 16 .. 1, the tree
// order of group_sum).
template <typename T>
__device__ __forceinline__ T list_sum(T v, int k, const Pack &P) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (o >= P.cmax) continue;
        const T y = __shfl_down_sync(FULL, v, o);
        if (k + o < P.cnt) v += y;
    }
    return v;
}

// Wedge sums of a pack of whole rows.
template <bool F64>
__device__ __forceinline__ void short_wedges(const ShortArgs &A, const ShortSmem<F64> &S, const Pack &P) {
    using Acc = AccT<F64>;
    const int k = (threadIdx.x & 31) - P.first, Du = P.cnt;
    const bool own = Du > 0;
    const int word = own ? A.info[P.x].y : 0;
    const int ak = word & 0xff;
    const int b0 = Du - 4 + ak;
    Acc acc = 0;
    if constexpr (F64) {
        F2Sum a2;
#pragma unroll 4
        for (int j = 0; j < P.cmax; ++j) {
            const int aj = __shfl_sync(FULL, ak, P.first + j);
            if (j < Du && j != k) a2.add(S.f[b0 + aj]);
        }
        acc = a2.value();
    } else {
        // one FMA per term; up to the shortest row every lane's terms are
        // real, beyond it they add under j < D_u.  Both include the lane's
        // own term j = k once, removed at the end.  d >= 1 needs the guard
        // (0 log2 0) only in rows of degree <= 4
        const float akf = (float)ak, b0f = (float)b0;
        float sum = 0.0f;
        int j = 0;
#pragma unroll 4
        for (; j < P.cmin; ++j) {
            const float d = fmaxf(b0f + __shfl_sync(FULL, akf, P.first + j), 1.0f);
            sum = fmaf(d, lg2(d), sum);
        }
        for (; j < P.cmax; ++j) {
            const float d = fmaxf(b0f + __shfl_sync(FULL, akf, P.first + j), 1.0f);
            const float t = lg2(d);
            if (j < Du) sum = fmaf(d, t, sum);
        }
        acc = sum - dlog2d(fmaxf(b0f + akf, 1.0f));
    }
    const Acc rs = own ? (F64 ? acc : acc * (Acc)LN2) : (Acc)0;
    if (own) credit_end(A.Tacc, P.x, (double)rs);
    const Acc c = list_sum(rs, k, P);
    const uint32_t st = list_sum((uint32_t)(ak * ak) | (uint32_t)word >> 16 << 16, k, P);
    if (own && k == 0) {
        // (a node of degree 1 is the middle of no cluster: its c is rounding residue)
        if (Du >= 2) credit_end(A.Tacc, P.u, (double)c);
        A.stat[P.u] = (uint64_t)st << 32 | (uint32_t)P.uword;
    }
}

// The bits j of the list's entries x_j among NZ entries of x's suffix.
template <int NZ>
__device__ __forceinline__ unsigned short_hits(const Pack &P, const int32_t *zp, int len) {
    int z[NZ];
#pragma unroll
    for (int c = 0; c < NZ; ++c) z[c] = c < len ? zp[c] : -2;
    unsigned found = 0, bit = 2;
#pragma unroll 2
    for (int j = 1; j < P.cmax; ++j) {
        const int y = __shfl_sync(FULL, P.x, P.first + j);
        bool m = false;
#pragma unroll
        for (int c = 0; c < NZ; ++c) m |= z[c] == y;
        if (m) found |= bit;
        bit += bit;
    }
    // lanes past their list's end compared with other lists' entries
    return found & (P.cnt < 32 ? (1u << P.cnt) - 1u : FULL);
}

// Triangles whose lowest node is u, a pack of the nodes' entries above them.
template <bool F64>
__device__ __forceinline__ void short_triangles(const ShortArgs &A, const ShortSmem<F64> &S, const Pack &P) {
    const int k = (threadIdx.x & 31) - P.first;
    const int2 ix = P.cnt > 0 ? A.info[P.x] : make_int2(0, 0);
    const int ax = ix.y & 0xff, lo = ix.y >> 8 & 0xff;
    // the list's last entry has no later one to pair with
    const int len = k + 1 < P.cnt ? ax - lo : 0;
    const int32_t *zp = A.ci + ix.x + lo;
    const int longest = __reduce_max_sync(FULL, len);
    unsigned hits = 0;
    for (int e = 0; e < longest; e += SH_Z)
        hits |= longest - e <= 4 ? short_hits<4>(P, zp + e, len - e) : short_hits<SH_Z>(P, zp + e, len - e);
    if (!__any_sync(FULL, hits != 0u)) return;
    int64_t q = 0;
    int t = __popc(hits);
    const int sum0 = (P.uword & 0xff) + ax;
    for (unsigned left = hits; __any_sync(FULL, left != 0u); left &= left - 1u) {
        const int src = P.first + __ffs(left) - 1;
        const int z = __shfl_sync(FULL, P.x, src), az = __shfl_sync(FULL, ax, src);
        if (left) {
            q += S.tq[sum0 + az];
            credit_end(A.Tacc, z, S.tqd[sum0 + az]);
            atomicAdd(A.tri + z, 1);
        }
    }
    if (t) {
        credit_end(A.Tacc, P.x, (double)q * A.qscale);
        atomicAdd(A.tri + P.x, t);
    }
    q = list_sum(q, k, P);
    t = list_sum(t, k, P);
    if (k == 0 && t) {
        credit_end(A.Tacc, P.u, (double)q * A.qscale);
        atomicAdd(A.tri + P.u, t);
    }
}

template <bool F64>
__global__ void __launch_bounds__(SH_WARPS * 32, 5) k_short(ShortArgs A, const int32_t *__restrict__ cnt,
                                                            const float2 *__restrict__ ftab,
                                                            const int64_t *__restrict__ tq, bool chosen) {
    if (short_closed(cnt, chosen)) return;
    __shared__ ShortSmem<F64> S;
    A.qscale = ldexp(1.0, -cnt[CNT_TRIFRAC]);
    const int sums = min(3 * cnt[CNT_MAXDEG] + 1, SH_SUMS);
    for (int i = threadIdx.x; i < sums; i += blockDim.x) {
        S.tq[i] = tq[i];
        S.tqd[i] = (double)tq[i] * A.qscale;
        if (F64) S.f[i] = ftab[i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t step = (int64_t)gridDim.x * SH_WARPS * A.per;
    for (int64_t base = ((int64_t)blockIdx.x * SH_WARPS + w) * A.per; base < A.n; base += step) {
        const int64_t v = base + lane;
        const int2 iv = lane < A.per && v < A.n ? A.info[v] : make_int2(0, 0);
        const int Dv = iv.y & 0xff, lo = iv.y >> 8 & 0xff;
        PackList L{};
        L.load(S, (int)v, iv.y, iv.x, Dv);
        for (int t0 = 0, taken = 0; t0 < L.total;) short_wedges<F64>(A, S, L.next(S, A.ci, t0, taken));
        // a node with one entry above it opens no pair
        L.load(S, (int)v, iv.y, iv.x + lo, Dv - lo >= 2 ? Dv - lo : 0);
        for (int t0 = 0, taken = 0; t0 < L.total;) short_triangles<F64>(A, S, L.next(S, A.ci, t0, taken));
    }
}

int launch_short(const int32_t *ci, const Scratch &s, int precision, int32_t n, const Tune &t, bool chosen,
                 cudaStream_t st) {
    // fewer nodes per step while that leaves warp slots of the GPU empty (ER
    // 2000: 8 nodes, five packs one after the other, 15 us in FP32C and
    // 18 in FP64; 2 nodes, 9.8 and 11.0)
    const int32_t slots = t.num_sms * 32;
    const int32_t per = n >= slots * 32 ? 32 : n >= slots * 8 ? 8 : 2;
    const ShortArgs A{ci, reinterpret_cast<const int2 *>(s.info), n, per, s.Tacc, s.outdeg,
                      reinterpret_cast<uint64_t *>(s.sig1), 0.0};
    const int64_t g = ((int64_t)n + per * SH_WARPS - 1) / (per * SH_WARPS), cap = (int64_t)t.num_sms * 16;
    const unsigned grid = (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
    if (precision == EF_PREC_FP64)
        k_short<true><<<grid, SH_WARPS * 32, 0, st>>>(A, s.counters, s.ftab, s.tq, chosen);
    else
        k_short<false><<<grid, SH_WARPS * 32, 0, st>>>(A, s.counters, s.ftab, s.tq, chosen);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace ef
