// Triangle pass of libef (Algorithm 1, Phase 2: the "i in Adj(j)" test).
//
// The wedge pass credits every cluster with its open degree; clusters whose
// ends are adjacent (triangles) need d - 2 instead.  Edges are oriented from
// lower to higher (degree, id); each triangle is found exactly once, at its
// lowest-ranked node a, as an adjacent pair {b, c} of a's out-neighbours
// N+(a) (b before c in N+(a)'s id order).  Its three nodes each hold 4
// credits of degree sum-6 that the wedge pass counted at sum-4
// (sum = D_a + D_b + D_c), so each receives g = 4 (f(sum-6) - f(sum-4)) and
// one triangle count.
//
// Pair tests: b and c are adjacent iff the higher-ranked of the two is in the
// lower-ranked one's out-list.  That is sum_a C(|N+(a)|, 2) independent tests
// -- 1.1e8 on the 4M-node power-law workload, against 1.15e9 dependent steps
// for merging the two out-lists of every edge.  A warp takes 64 consecutive
// oriented edges, cuts each edge's candidates c into units of TRI_UNIT and
// spreads the units evenly over its lanes.
//
// The pass is bound by L2 latency, so every membership test is one round of
// two independent 16-byte loads, the same instructions for every lane: an
// out-list of at most SHORT_MAX entries is read whole (it spans at most two
// aligned quads); of a longer one the key's bucket of its hash table (8 slots
// in one sector, out_table), which settles the test but for rare full
// buckets.  The oriented CSR carries, for each out-neighbour, the probe
// descriptor of its own list (which quads to load and how to read them, fixed
// once per node by the orientation), so no test waits for an out_ptr load or
// recomputes a table's geometry.  Owners of more than TRI_LONG
// out-neighbours have their own kernel (k_tri_long).
//
// Measured and left out (4M-node power-law graph): L2 eviction hints
// (evict_last on probes, evict_first on the candidate stream) changed
// nothing; staging each tile's candidates in shared memory was slower
// (2.00 against 1.84 ms, and again 1.74 against 1.65 ms with a warp step's
// 128 entries staged by coalesced loads); loading each test's correction
// tq[sum] with its probes, to save the second round trip of a hit, was
// slower too (1.85 against 1.65 ms; the per-unit binary search replaced by
// a shared-memory unit map changed nothing).  Short owners of the 2M-node
// power-law graph: the kernel issues in 48% of its cycles and waits 9.0 cycles
// per instruction on its loads, with 45% of the warp slots filled (64
// registers allow half); DRAM 17%, L2 26% of their throughput.
//
// The pass is integer-only: g comes from a table in fixed point (units of
// 2^-F, F chosen per call from the maximum degree), so the sums are exact and
// independent of the order of the atomics, and no FP64 instruction (one lane
// per clock per SM sub-partition on this GPU) sits in a divergent branch.
// Corrections and counts go to per-node accumulators (qacc, tcnt) by L2
// reductions: c's at once, b's once per unit, a's merged per lane over
// consecutive units of the same owner.
//
// A shard of the pass lists the triangles whose lowest-ranked node lies in
// its node range (a node id range: the oriented layout's list order comes
// from atomics and differs between calls, node ids and ranks do not).
#include "ef_internal.cuh"

namespace ef {

constexpr int TRI_WARPS = 8;
// Kernel variants: candidate pairs per lane step (TRI_UNIT), resident blocks
// per SM the registers are sized for, and oriented edges per warp step (EW).
// Measured on the 4M-node power-law graph with EW = 32: (2, 4) 1.80 ms,
// (2, 3) 1.98, (2, 5) 2.06, (4, 3) 2.28, (4, 4) 2.51 (register spills).
// EW = 64 fills the last round of a step better where out-lists are short:
// WS batch 6.13 -> 5.65 ms, BA 1M 0.174 -> 0.154, power-law 1.665 -> 1.653.
// Variant 0 = (2, 4, 64), 1 = (4, 3, 32).

__device__ __forceinline__ unsigned match4(int4 v, int key) {
    return (unsigned)(v.x == key) | (unsigned)(v.y == key) << 1 | (unsigned)(v.z == key) << 2 |
           (unsigned)(v.w == key) << 3;
}

// One membership test "key in the out-list of probe descriptor pd", split so
// that a lane issues the loads of all its tests before it waits for any: the
// quads p0 and p0 + 1, and which of their entries count (info bits 0-3 and
// 4-7) and the kind of list (bits 8-9, the descriptor's kind).
struct Probe {
    const int4 *p0;
    unsigned info;
};

__device__ __forceinline__ Probe probe_of(const int32_t *out_col, const int32_t *out_hash, int2 pd, int key) {
    Probe r;
    const unsigned kind = (unsigned)pd.y >> DESC_KIND_SHIFT;
    if (kind == 1) {
        const int nb = pd.y & DESC_MASK;
        const int b0 = bucket_of(key, nb);
        r.p0 = reinterpret_cast<const int4 *>(out_hash) + ((int64_t)pd.x + 2 * b0);
        r.info = 0xffu | 1u << 8;
    } else if (kind == 0) {
        r.p0 = reinterpret_cast<const int4 *>(out_col) + pd.x;
        r.info = (unsigned)pd.y & 0xffu;
    } else {
        r.p0 = reinterpret_cast<const int4 *>(out_col) + (pd.x >> 2);
        r.info = 2u << 8;
    }
    return r;
}

// Resolve a probe from its two loaded quads.  The rare ends -- a full home
// bucket without the key (continue with the next ones), a long list without
// a table (malformed input only: binary search) -- reload what they need.
__device__ __forceinline__ bool probe_more(const int4 *p0, const int32_t *out_col, const int32_t *out_hash, int2 pd,
                                           int key) {
    if ((unsigned)pd.y >> DESC_KIND_SHIFT == 1u) {
        const int nb = pd.y & DESC_MASK;
        const int4 *t = reinterpret_cast<const int4 *>(out_hash) + pd.x;
        int b = (int)(p0 - t) >> 1;
        for (int tries = 1; tries < nb; ++tries) {
            b = b + 1 == nb ? 0 : b + 1;
            const int4 x = __ldg(t + 2 * b), y = __ldg(t + 2 * b + 1);
            if (match4(x, key) | match4(y, key)) return true;
            if (y.w < 0) return false;
        }
        return false;
    }
    const int ls = pd.x, le = pd.y & DESC_MASK;
    const int pos = ls + lower_bound_i32(out_col + ls, le - ls, key);
    return pos < le && out_col[pos] == key;
}

__device__ __forceinline__ bool probe_done(const Probe &r, int4 x, int4 y, const int32_t *out_col,
                                           const int32_t *out_hash, int2 pd, int key) {
    if ((match4(x, key) & r.info) | (match4(y, key) & (r.info >> 4) & 0xfu)) return true;
    const unsigned kind = (r.info >> 8) & 3u;
    if (kind == 0 || (kind == 1 && y.w < 0)) return false;
    return probe_more(r.p0, out_col, out_hash, pd, key);
}

__device__ __forceinline__ void credit_tri(int64_t *qacc, int64_t *tcnt, int v, int64_t q, int cnt) {
    atomicAdd((unsigned long long *)(qacc + v), (unsigned long long)q);
    atomicAdd((unsigned long long *)(tcnt + v), (unsigned long long)cnt);
}

template <int TRI_UNIT, int TRI_BLOCKS, int EW>
__global__ void __launch_bounds__(TRI_WARPS * 32, TRI_BLOCKS) k_tri_pairs(
    const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_col, const int32_t *__restrict__ out_D,
    const int2 *__restrict__ out_pd, const int32_t *__restrict__ out_src, const int32_t *__restrict__ out_hash,
    const int32_t *__restrict__ outdeg, const int32_t *__restrict__ D, int32_t n,
    const int32_t *__restrict__ owner_range, const int64_t *__restrict__ tq,
    int64_t *__restrict__ qacc, int64_t *__restrict__ tcnt, const int32_t *__restrict__ cnt) {
    static_assert(EW == 32 || EW == 64, "a warp step takes 32 or 64 edges");
    __shared__ int s_ex[TRI_WARPS][EW];   // exclusive prefix of unit counts
    __shared__ int s_kend[TRI_WARPS][EW], s_b[TRI_WARPS][EW], s_Db[TRI_WARPS][EW], s_Dab[TRI_WARPS][EW];
    __shared__ int s_a[TRI_WARPS][EW];
    __shared__ int2 s_bpd[TRI_WARPS][EW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t total = gate_closed(cnt) ? 0 : out_ptr[n];   // no pairs when the device check failed
    const int64_t stride = (int64_t)gridDim.x * TRI_WARPS * EW;
    // owners a in [a_lo, a_hi) open their pairs (all nodes, or one shard's range)
    const int a_lo = owner_range ? owner_range[0] : 0, a_hi = owner_range ? owner_range[1] : n;
    for (int64_t K0 = ((int64_t)blockIdx.x * TRI_WARPS + w) * EW; K0 < total; K0 += stride) {
        int U = 0;
#pragma unroll
        for (int h = 0; h < EW / 32; ++h) {
            const int e = h * 32 + lane;
            const int64_t k = K0 + e;
            int nu = 0;
            if (k < total) {
                const int a = out_src[k];
                const int kend = out_ptr[a] + outdeg[a];
                // (the long owners' pairs are k_tri_long's)
                const int np = a >= a_lo && a < a_hi && kend - out_ptr[a] <= TRI_LONG ? kend - (int)k - 1 : 0;
                if (np > 0) {
                    const int b = out_col[k];
                    const int Db = out_D[k];
                    s_kend[w][e] = kend;
                    s_b[w][e] = b;
                    s_Db[w][e] = Db;
                    s_bpd[w][e] = out_pd[k];
                    s_Dab[w][e] = D[a] + Db;
                    s_a[w][e] = a;
                    nu = (np + TRI_UNIT - 1) / TRI_UNIT;
                }
            }
            int inc = nu;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += y;
            }
            s_ex[w][e] = U + inc - nu;
            U += __shfl_sync(FULL, inc, 31);
        }
        __syncwarp();
        int cur_a = -1, hit_a = 0;
        int64_t acc_a = 0;
        int i = -1, kend = 0, exi = 0, b = 0, Db = 0, Dab = 0, ai = 0;
        int2 bpd = make_int2(0, 0);
        for (int t = lane; t < U; t += 32) {
            // the warp edge owning unit t: the last i with s_ex[i] <= t (s_ex is
            // non-decreasing; i + step <= EW - 1 at every step)
            int ni = 0;
#pragma unroll
            for (int step = EW / 2; step > 0; step >>= 1)
                if (s_ex[w][ni + step] <= t) ni += step;
            if (ni != i) {
                i = ni;
                kend = s_kend[w][i];
                exi = s_ex[w][i];
                b = s_b[w][i];
                Db = s_Db[w][i];
                bpd = s_bpd[w][i];
                Dab = s_Dab[w][i];
                ai = s_a[w][i];
            }
            const int64_t j0 = K0 + i + 1 + TRI_UNIT * (t - exi);
            const int jn = (int)min((int64_t)TRI_UNIT, kend - j0);
            int c[TRI_UNIT], Dc[TRI_UNIT];
            int2 rc[TRI_UNIT];
#pragma unroll
            for (int q = 0; q < TRI_UNIT; ++q) {
                if (q < jn) {
                    c[q] = __ldg(out_col + j0 + q);
                    Dc[q] = __ldg(out_D + j0 + q);
                    rc[q] = __ldg(out_pd + j0 + q);
                }
            }
            Probe pr[TRI_UNIT];
            int4 x[TRI_UNIT], y[TRI_UNIT];
#pragma unroll
            for (int q = 0; q < TRI_UNIT; ++q) {
                if (q < jn) {
                    const bool b_low = rank_less(Db, b, Dc[q], c[q]);
                    pr[q] = probe_of(out_col, out_hash, b_low ? bpd : rc[q], b_low ? c[q] : b);
                    pr[q].info |= (unsigned)b_low << 10;
                    x[q] = __ldg(pr[q].p0);
                    y[q] = __ldg(pr[q].p0 + 1);
                }
            }
            int hits = 0;
            int64_t gsum = 0;
#pragma unroll
            for (int q = 0; q < TRI_UNIT; ++q) {
                if (q < jn) {
                    const bool b_low = (pr[q].info >> 10) & 1u;
                    if (probe_done(pr[q], x[q], y[q], out_col, out_hash, b_low ? bpd : rc[q], b_low ? c[q] : b)) {
                        const int64_t g = __ldg(tq + Dab + Dc[q]);
                        credit_tri(qacc, tcnt, c[q], g, 1);
                        gsum += g;
                        ++hits;
                    }
                }
            }
            if (hits) {
                credit_tri(qacc, tcnt, b, gsum, hits);
                if (ai != cur_a) {
                    if (hit_a) credit_tri(qacc, tcnt, cur_a, acc_a, hit_a);
                    cur_a = ai;
                    acc_a = 0;
                    hit_a = 0;
                }
                acc_a += gsum;
                hit_a += hits;
            }
        }
        if (hit_a) credit_tri(qacc, tcnt, cur_a, acc_a, hit_a);
        __syncwarp();
    }
}

// ------------------------------------------------------------- long owners
// Owners a of more than TRI_LONG out-neighbours.  Their out-lists are first
// sorted by rank (k_sort_long), so that of a pair b before c the lower end is
// always b.  Then a warp per 32 candidates (k_tri_long): lane l holds c =
// N+(a)[32 k + l] and the warp walks the earlier entries b, whose table is
// the same for all lanes: a test is a hash, one 32-byte load (of a short list
// two of 16) and its compares, with nothing to decide per lane.  The hits of 32 b are kept as a
// bit matrix (a word per lane); its rows give c's credits, its transpose b's,
// so a correction is looked up only where a triangle is, and the credits go
// out once per (a, c) and per (a, b, item) instead of once per hit.  (Where
// most tests close a triangle, as in R-MAT, the hits' reductions to a few
// large c had bound the pass.)
//
// Pair tests of a call, all owners in k_tri_pairs / with the long owners
// here: R-MAT 2^16 (955k entries) 0.74 / 0.21 ms (0.18 with shared items),
// R-MAT 2^18 1.9 / 0.62, power-law 4M 1.60 / 1.36, its 87M-entry variant 5.8 /
// 4.7.  The kernel issues in 54% of its cycles on both (L1 wavefronts 53%,
// loads waited for 5.4 and 5.8 cycles per instruction).  TRI_LONG = 16:
// R-MAT 2^16 0.17 but power-law 4M 1.42 and 0.40 against 0.38 at 1M (lanes
// past the list idle); four entries b together: 1.42.  Without the sort, the
// lower end of each pair decided per lane and b's credits reduced by warp
// sums per b: R-MAT 0.24, power-law 1.54.
constexpr int TL_WARPS = 8;

// Entry e of every 32 of a long list: its position by rank is the number of
// entries below it.  A warp per item.
__global__ void __launch_bounds__(256) k_sort_long(const int32_t *__restrict__ out_ptr,
                                                   const int32_t *__restrict__ out_col,
                                                   const int32_t *__restrict__ out_D,
                                                   const int2 *__restrict__ out_pd,
                                                   const int32_t *__restrict__ outdeg,
                                                   const int2 *__restrict__ items, const int32_t *__restrict__ cnt,
                                                   int4 *__restrict__ rec) {
    if (gate_closed(cnt)) return;
    const int lane = threadIdx.x & 31;
    const int total = cnt[CNT_TRILONG];
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t it = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < total; it += nwarps) {
        const int2 item = items[it];
        const int ls = out_ptr[item.x], p = outdeg[item.x], e = item.y * 32 + lane;
        const bool own = e < p;
        const int x = own ? out_col[ls + e] : 0, Dx = own ? out_D[ls + e] : 0;
        int pos = 0;
        for (int i0 = 0; i0 < p; i0 += 32) {
            const bool in = i0 + lane < p;
            const int y = in ? out_col[ls + i0 + lane] : 0, Dy = in ? out_D[ls + i0 + lane] : 0x7fffffff;
#pragma unroll 8
            for (int i = 0; i < 32; ++i)   // entries past the list rank above all
                pos += rank_less(__shfl_sync(FULL, Dy, i), __shfl_sync(FULL, y, i), Dx, x);
        }
        if (own) {
            const int2 pd = out_pd[ls + e];
            rec[ls + pos] = make_int4(x, Dx, pd.x, pd.y);
        }
    }
}

// One 32-byte sector in one load (p 32-byte aligned).
__device__ __forceinline__ void load_sector(const int4 *p, int4 &x, int4 &y) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w), "=r"(y.x), "=r"(y.y), "=r"(y.z), "=r"(y.w)
        : "l"(p));
}

// Lane i's word of the transpose of the 32 x 32 bit matrix whose rows are the
// lanes' words.
__device__ __forceinline__ unsigned transpose32(unsigned v) {
    const int lane = threadIdx.x & 31;
    unsigned m = 0x0000ffffu;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const unsigned o = __shfl_xor_sync(FULL, v, s);
        v = lane & s ? (v & ~m) | (o >> s & m) : (v & m) | (o << s & ~m);
        m ^= m << (s >> 1);
    }
    return v;
}

constexpr int TL_STEP = 2;   // entries b tested together
// Small graphs: an item is shared among warps while that leaves each of them at
// most TL_ROUNDS shares on average, by up to eight chunks of b, then (at most
// TL_PART_ROUNDS) by up to four parts of a chunk.  A pair of b takes the
// latency of one L2 load, so the longest list decides there: power-law 100k
// 31 -> 20 us, 20k 23 -> 10, R-MAT 2^16 100 -> 75; larger graphs have the items.
constexpr int TL_ROUNDS = 16, TL_PART_ROUNDS = 6;

__global__ void __launch_bounds__(TL_WARPS * 32, 4) k_tri_long(
    const int32_t *__restrict__ out_ptr, const int32_t *__restrict__ out_col, const int32_t *__restrict__ out_hash,
    const int32_t *__restrict__ outdeg, const int32_t *__restrict__ D, int32_t n,
    const int32_t *__restrict__ owner_range, const int64_t *__restrict__ tq, const int2 *__restrict__ items,
    const int4 *__restrict__ rec, int64_t *__restrict__ qacc, int64_t *__restrict__ tcnt, int32_t *__restrict__ cnt) {
    if (gate_closed(cnt)) return;
    __shared__ int4 s_b[TL_WARPS][32];   // {b, D_b, its descriptor}
    __shared__ int s_Dc[TL_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int total = cnt[CNT_TRILONG];
    const int a_lo = owner_range ? owner_range[0] : 0, a_hi = owner_range ? owner_range[1] : n;
    const int4 *cols = reinterpret_cast<const int4 *>(out_col), *table = reinterpret_cast<const int4 *>(out_hash);
    // the first item by position, the others from the counter (an atomic by every
    // warp before its first item cost a graph without long owners 3 us a call)
    const int nwarps = gridDim.x * TL_WARPS;
    // few items: 2^chunks warps share an item's entries b by chunks of 32, then
    // 2^parts a chunk
    int chunks = 0, parts = 0;
    while (chunks < 3 && ((int64_t)total << (chunks + 1)) <= (int64_t)TL_ROUNDS * nwarps) ++chunks;
    while (chunks == 3 && parts < 2 && ((int64_t)total << (parts + 4)) <= (int64_t)TL_PART_ROUNDS * nwarps) ++parts;
    const int split = chunks + parts, width = 32 >> parts;
    auto take = [&]() {
        int it = 0;
        if (lane == 0) it = nwarps + atomicAdd(cnt + CNT_TRINEXT, 1);
        return __shfl_sync(FULL, it, 0);
    };
    for (int it = blockIdx.x * TL_WARPS + w; it >> split < total; it = take()) {
        const int2 item = items[total - 1 - (it >> split)];
        const int first = 32 * (it & ((1 << chunks) - 1)), lo = width * ((it & ((1 << split) - 1)) >> chunks);
        if (first > item.y * 32) continue;   // (no entries before its candidates there)
        const int a = item.x;
        if (a < a_lo || a >= a_hi) continue;
        const int ls = out_ptr[a], p = outdeg[a], Da = D[a];
        const int j = item.y * 32 + lane;
        const bool own = j < p;
        const int4 rc = own ? rec[ls + j] : make_int4(-2, 0, 0, 0);   // -2: no key
        const int c = rc.x;
        const uint32_t hc = (uint32_t)c * 0x9E3779B1u;                // bucket_of's hash
        const int sum_c = Da + rc.y;
        const int last = min(item.y * 32 + 31, p - 1);   // b runs over the entries below this one
        s_Dc[w][lane] = rc.y;
        int64_t qc = 0;
        int tc = 0;
        for (int i0 = first; i0 < last; i0 += 32 << chunks) {
            __syncwarp();
            const int4 rb = i0 + lane < last ? rec[ls + i0 + lane] : make_int4(0, 0, 0, 0);
            s_b[w][lane] = rb;
            __syncwarp();
            const int nb = min(lo + width, last - i0);
            unsigned found = 0;   // bit i: {b_i, c} adjacent
            for (int i = lo; i < nb; i += TL_STEP) {
                int4 x[TL_STEP], y[TL_STEP];
                const int4 *p0[TL_STEP];
                unsigned mask[TL_STEP];   // entries of the two quads that count
                int2 pd[TL_STEP];
#pragma unroll
                for (int q = 0; q < TL_STEP; ++q) {
                    // past the chunk's end: an empty list
                    const int4 b = s_b[w][min(i + q, nb - 1)];
                    pd[q] = i + q < nb ? make_int2(b.z, b.w) : make_int2(0, 0);
                    const unsigned kind = (unsigned)pd[q].y >> DESC_KIND_SHIFT;
                    if (kind == 1) {
                        p0[q] = table + (pd[q].x + 2 * (int)(((uint64_t)hc * (uint32_t)(pd[q].y & DESC_MASK)) >> 32));
                        mask[q] = 0xff;
                        load_sector(p0[q], x[q], y[q]);
                    } else {
                        // a short list's quads, or (kind 2) none: resolved below
                        p0[q] = cols + (kind == 0 ? pd[q].x : 0);
                        mask[q] = kind == 0 ? (unsigned)pd[q].y & 0xffu : 0u;
                        x[q] = __ldg(p0[q]);
                        y[q] = __ldg(p0[q] + 1);
                    }
                }
#pragma unroll
                for (int q = 0; q < TL_STEP; ++q) {
                    const unsigned kind = (unsigned)pd[q].y >> DESC_KIND_SHIFT;
                    bool hit = ((match4(x[q], c) | match4(y[q], c) << 4) & mask[q]) != 0u;
                    // a full bucket without the key, or a list without a table
                    if (own && !hit && (kind == 2 || (kind == 1 && y[q].w >= 0)))
                        hit = probe_more(p0[q], out_col, out_hash, pd[q], c);
                    if (hit) found |= 1u << (i + q);
                }
            }
            // only entries before c (c = -2 matches no key)
            if (i0 + 31 >= j) found &= j > i0 ? (1u << (j - i0)) - 1u : 0u;
            const unsigned col = transpose32(found);   // lane i: the c adjacent to b_i
            tc += __popc(found);
            for (unsigned f = found; f; f &= f - 1u) qc += __ldg(tq + sum_c + s_b[w][__ffs(f) - 1].y);
            if (col) {
                int64_t qb = 0;
                for (unsigned f = col; f; f &= f - 1u) qb += __ldg(tq + Da + rb.y + s_Dc[w][__ffs(f) - 1]);
                credit_tri(qacc, tcnt, rb.x, qb, __popc(col));
            }
        }
        if (tc) credit_tri(qacc, tcnt, c, qc, tc);
        const int64_t qa = warp_sum(qc);
        const int ta = __reduce_add_sync(FULL, tc);
        if (lane == 0 && ta) credit_tri(qacc, tcnt, a, qa, ta);
        __syncwarp();
    }
}

static inline unsigned grid_of(int64_t work, int per_block, int64_t cap) {
    int64_t g = (work + per_block - 1) / per_block;
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

int launch_tri_pairs(const Scratch &s, int32_t n, int64_t m, const Tune &t, cudaStream_t st,
                     const int32_t *owner_range, bool long_lists) {
    const unsigned grid = grid_of(m / 2, TRI_WARPS * 32, (int64_t)t.num_sms * 16);
    if (t.tri_variant == 1)
        k_tri_pairs<4, 3, 32><<<grid, TRI_WARPS * 32, 0, st>>>(s.out_ptr, s.out_col, s.out_D, s.out_pd, s.out_src,
                                                            s.out_hash, s.outdeg, s.D, n, owner_range, s.tq, s.qacc,
                                                            s.tcnt, s.counters);
    else
        k_tri_pairs<2, 4, 64><<<grid, TRI_WARPS * 32, 0, st>>>(s.out_ptr, s.out_col, s.out_D, s.out_pd, s.out_src,
                                                            s.out_hash, s.outdeg, s.D, n, owner_range, s.tq, s.qacc,
                                                            s.tcnt, s.counters);
    if (!long_lists) return cudaGetLastError() == cudaSuccess ? 0 : -1;
    k_sort_long<<<(unsigned)t.num_sms * 8, 256, 0, st>>>(s.out_ptr, s.out_col, s.out_D, s.out_pd, s.outdeg,
                                                        s.tri_items, s.counters, s.tri_rec);
    k_tri_long<<<(unsigned)t.num_sms * 4, TL_WARPS * 32, 0, st>>>(s.out_ptr, s.out_col, s.out_hash, s.outdeg, s.D, n,
                                                                 owner_range, s.tq, s.tri_items, s.tri_rec, s.qacc,
                                                                 s.tcnt, s.counters);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace ef
