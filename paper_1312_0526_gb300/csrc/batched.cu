// batched.cu -- many independent bucket hypergraphs in one persistent launch.
//
// The key set is cut into buckets (the HEM layout of sec. 3 "Practical
// workarounds": one small hypergraph per bucket); bucket b hashes its keys
// with seed b into a 3-partite hypergraph of m_b = 3 ceil(ceil(gamma n_b)/3)
// vertices and is peeled on its own.  One CTA takes one bucket at a time
// from a shared counter (work stealing over a largest-first schedule, one
// launch per size class unless the caller gives a shape) and runs the whole
// path for it, block-synchronous:
//   hash + AddEdge (sec. 3, 4.1), round 0 scan, rounds with the claims of
//   round t+1 made by the deletions of round t (sec. 4.2; same scheme as the
//   single-graph path), the canonical order (layers ascending by round, edge
//   ids ascending inside a layer, 2-core edges last) by a stable counting pass,
//   and optionally the MWHC g values (sec. 3, layers last to first).
// A bucket's state lives in shared memory when it fits: vertex records of 32
// bits (degree in the low 16, sum of incident local edge ids mod 2^16 in the
// high 16; a bucket in shared memory has far fewer than 2^16 edges, so the
// degree never carries into the sum), claim words, the layers as 16-bit local
// edge ids, the layer table and the g values, about 9 bytes per key; when 6
// more fit, the edges' vertices too (2,000-key buckets: 128 -> 172 keys per us
// and SM, with the order pass on all warps), else an edge's vertices are hashed
// again from its key (read through the cache) when a round or the assignment
// needs them.  Larger buckets use a per-CTA region of the workspace,
// with 32-bit records too unless the bucket has 2^16 - 1 edges or more.  No
// block waits on another; the only cross-block state is the bucket counter.
#include <algorithm>

#include "cluster.cuh"
#include "kernels.cuh"

namespace hp {

constexpr uint32_t kBatchMaxEdges = 65536;        // per bucket
constexpr uint32_t kBatchMaxVertices = (1u << 17) - 1;  // packed 17-bit local ids
// Claim words: (round << 2) | hinge, all ones while unclaimed.  16 bits in
// shared memory and in the 32-bit global path (layer tables of at most
// kClaim16Rounds entries, fewer if the tuning says so), 32 bits in the
// 64-bit path.
constexpr uint32_t kClaim16Rounds = 16383;

template <typename C>
__device__ __forceinline__ uint32_t unclaimed() { return (uint32_t)(C)~(C)0; }

// A claim is (round << 2) | code, code 0, 1, 3 for hinge position 0, 1, 2: the
// bitwise and of a round's claims of an edge is its smallest one, so a claim in
// a 16-bit word is one atomicAnd on the 32-bit word around it, with no
// compare-and-swap loop.  (All ones is no claim: a 16-bit round stays below
// kClaim16Rounds.)  It must not touch an edge claimed in an earlier round, so
// the word is read first: such a claim was there before the round's barrier.
__device__ __forceinline__ uint32_t hinge_code(uint32_t j) { return j + (j >> 1); }
__device__ __forceinline__ uint32_t hinge_of(uint32_t claim) { return (claim & 3u) - ((claim >> 1) & 1u); }
__device__ __forceinline__ bool claim_open(const uint32_t *, uint32_t) { return true; }
__device__ __forceinline__ bool claim_open(const uint16_t *p, uint32_t tag) {
    const uint32_t c = *reinterpret_cast<const volatile uint16_t *>(p);
    return c == 0xFFFFu || (c >> 2) == (tag >> 2);
}
// the claim before this one (call for an open claim word)
__device__ __forceinline__ uint32_t claim_put(uint32_t *p, uint32_t tag) { return atomicMin(p, tag); }
__device__ __forceinline__ uint32_t claim_put(uint16_t *p, uint32_t tag) {
    uint32_t *w = reinterpret_cast<uint32_t *>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3);
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 2u) * 8u;
    return (atomicAnd(w, ~((0xFFFFu ^ tag) << sh)) >> sh) & 0xFFFFu;
}

__device__ __forceinline__ uint32_t bucket_vertices(uint32_t n, uint32_t gamma_milli) {
    const uint64_t gn = ((uint64_t)n * gamma_milli + 999u) / 1000u;
    return (uint32_t)((gn + 2) / 3 * 3);
}

// The three vertices of a bucket's edge: its key hashed with the bucket's
// seed into the three parts (the same hash as the single-graph path).
__device__ __forceinline__ void bucket_edge(uint64_t k, uint64_t seed, const FastMod &fm,
                                            uint32_t P, uint32_t (&v)[3]) {
#pragma unroll
    for (int j = 0; j < 3; j++)
        v[j] = (uint32_t)fastmod(mix64(k ^ (seed + (uint64_t)j)), fm) + (uint32_t)j * P;
}

// Vertex record arithmetic: degree in the low W bits, id sum in the rest.
template <typename T>
struct VRec;
template <>
struct VRec<uint32_t> {
    static constexpr int W = 16;
    __device__ static uint32_t deg(uint32_t r) { return r & 0xFFFFu; }
    __device__ static uint32_t sum(uint32_t r) { return r >> 16; }
    __device__ static uint32_t unit(uint32_t e) { return (e << 16) + 1u; }
    __device__ static uint32_t mask() { return 0xFFFFu; }
};
template <>
struct VRec<unsigned long long> {
    static constexpr int W = 32;
    __device__ static uint32_t deg(unsigned long long r) { return (uint32_t)r; }
    __device__ static uint32_t sum(unsigned long long r) { return (uint32_t)(r >> 32); }
    __device__ static unsigned long long unit(uint32_t e) {
        return ((unsigned long long)e << 32) + 1ull;
    }
    __device__ static uint32_t mask() { return 0xFFFFFFFFu; }
};

// Where one bucket's state lives (shared memory or the CTA's global region).
template <typename T, typename C>
struct BucketState {
    T *rec;          // [m]
    C *claim;        // [n] (round << 2) | hinge
    uint16_t *L;     // [n] layers appended (local edge ids < 2^16)
    uint32_t *loff;  // [rcap + 2] layer starts
    uint32_t *cnt;   // [rcap + 2] running starts of the order pass
    uint32_t *G;     // [ceil(m / 16)] 2-bit g values (MPHF)
    uint16_t *V;     // [3][n] the edges' vertices, each in its part, or null (hashed again)
    uint32_t rcap;   // rounds the loff table holds
};

struct BatchArgs {
    const uint64_t *keys;
    const uint64_t *off;  // [B + 1]
    uint32_t B;
    uint32_t gamma_milli;
    const uint32_t *sched;    // processing order of the buckets
    const uint32_t *range;    // this launch's first and end place in sched, or null (all B)
    uint32_t *next;           // work-stealing counter
    uint32_t *late;           // null, or where a bucket goes that does not fit this launch's
    uint32_t *late_count;     //   shared memory (a class launch has no global regions)
    uint32_t *order;          // [total] per-bucket canonical order (local ids)
    uint32_t *rounds;         // [B] or null
    uint32_t *status;         // [B] or null: 0 peeled, 1 2-core left, 2 too large
    uint64_t *G;              // or null
    const uint64_t *G_off;    // [B + 1] word offsets of the buckets' g arrays
    char *scratch;            // per-CTA global regions
    size_t scratch_bytes;     // bytes per CTA region
    uint32_t smem_bytes;      // dynamic shared memory per CTA
    uint32_t smem_rounds;     // layer-table entries of a bucket in shared memory
    uint32_t global16_rounds; // layer-table entries on the 32-bit global path
    uint32_t wait;            // 1: reads what the launch before it wrote
};

__host__ __device__ inline size_t a16(size_t x) { return (x + 15) & ~(size_t)15; }

// Bytes of one bucket's state with records of rec_bytes and a loff table of
// rcap + 2 entries.
__host__ __device__ inline size_t bucket_bytes(uint32_t n, uint32_t m, uint32_t rec_bytes,
                                               uint32_t claim_bytes, uint32_t rcap,
                                               bool verts = false) {
    return a16((size_t)m * rec_bytes) + a16((size_t)n * claim_bytes) + a16((size_t)n * 2) +
           2 * a16(((size_t)rcap + 2) * 4) + a16(((size_t)m + 15) / 16 * 4) +
           (verts ? a16((size_t)n * 6) : 0);
}

template <typename T, typename C>
__device__ BucketState<T, C> carve(char *base, uint32_t n, uint32_t m, uint32_t rcap,
                                   bool verts = false) {
    BucketState<T, C> s;
    size_t o = 0;
    s.rec = reinterpret_cast<T *>(base + o);
    o += a16((size_t)m * sizeof(T));
    s.claim = reinterpret_cast<C *>(base + o);
    o += a16((size_t)n * sizeof(C));
    s.L = reinterpret_cast<uint16_t *>(base + o);
    o += a16((size_t)n * 2);
    s.loff = reinterpret_cast<uint32_t *>(base + o);
    o += a16(((size_t)rcap + 2) * 4);
    s.cnt = reinterpret_cast<uint32_t *>(base + o);
    o += a16(((size_t)rcap + 2) * 4);
    s.G = reinterpret_cast<uint32_t *>(base + o);
    o += a16(((size_t)m + 15) / 16 * 4);
    s.V = verts ? reinterpret_cast<uint16_t *>(base + o) : nullptr;
    s.rcap = rcap;
    return s;
}

// Warp-aggregated append to a block-local list (slot list_base + the value of a
// shared counter): two candidates per lane, one reservation.
__device__ __forceinline__ void cta_append2(uint32_t *cursor, uint16_t *list, uint32_t list_base,
                                            const bool (&pred)[2], const uint32_t (&v)[2]) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t b0 = __ballot_sync(0xFFFFFFFFu, pred[0]);
    const uint32_t b1 = __ballot_sync(0xFFFFFFFFu, pred[1]);
    if (!(b0 | b1)) return;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(cursor, (uint32_t)(__popc(b0) + __popc(b1)));
    base = list_base + __shfl_sync(0xFFFFFFFFu, base, 0);
    const uint32_t lt = (1u << lane) - 1u;
    if (pred[0]) list[base + __popc(b0 & lt)] = (uint16_t)v[0];
    if (pred[1]) list[base + __popc(b0) + __popc(b1 & lt)] = (uint16_t)v[1];
}

// Edges of a layer that one warp takes: one per lane (65,536 lognormal buckets,
// 8.28 ms; layers of up to 48 8.48, 64 8.63, none 8.60).
constexpr uint32_t kWarpLayer = 32;

// The whole path for one bucket.  Every thread of the block calls it.
// Returns false (writing nothing) when the bucket needs more rounds than its
// layer table holds; the caller reruns it with a larger table.
template <typename T, typename C, bool VERTS>
__device__ bool run_bucket(const BatchArgs &a, uint32_t b, BucketState<T, C> s, uint32_t n,
                           uint32_t m, uint32_t *sh) {
    const uint32_t kUnc = unclaimed<C>();
    using V = VRec<T>;
    const uint32_t T_ = blockDim.x;
    const uint32_t tid = threadIdx.x;
    const uint32_t P = m / 3;
    const uint64_t key0 = a.off[b];
    uint32_t &lcur = sh[0];
    uint64_t &magic = *reinterpret_cast<uint64_t *>(sh + 2);
    if (tid == 0) {
        lcur = 0;
        magic = ~0ull / P;  // reciprocal for the remainder by P
    }
    for (uint32_t v = tid; v < m; v += T_) s.rec[v] = 0;
    for (uint32_t e = tid; e < n; e += T_) s.claim[e] = (C)kUnc;
    __syncthreads();
    const FastMod fm{P, magic};
    const uint64_t seed = b;
    // the bucket's keys, read through the cache: hashed here and again
    // whenever an edge's vertices are needed
    const uint64_t *keys = a.keys + key0;
    // hash + AddEdge
    for (uint32_t e = tid; e < n; e += T_) {
        uint32_t v[3];
        bucket_edge(__ldg(keys + e), seed, fm, P, v);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            atomicAdd(s.rec + v[j], V::unit(e));
            if (VERTS) s.V[(uint32_t)j * n + e] = (uint16_t)(v[j] - (uint32_t)j * P);
        }
    }
    __syncthreads();
    // round 0: four records per thread and append (one record: 9,300 cycles of
    // a 2,000-key bucket's 103,000)
    for (uint32_t v0 = 0; v0 < m; v0 += 4u * T_) {
        const uint32_t v = v0 + 4u * tid;
        T r[4] = {0, 0, 0, 0};
        if constexpr (sizeof(T) == 4) {
            // the records' space is a multiple of 16 bytes
            if (v < m) {
                const uint4 q = *reinterpret_cast<const uint4 *>(s.rec + v);
                r[0] = q.x;
                r[1] = q.y;
                r[2] = q.z;
                r[3] = q.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (v + q < m) r[q] = s.rec[v + q];
        }
        uint32_t who[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t e = V::sum(r[q]), x = v + (uint32_t)q;
            bool take = x < m && V::deg(r[q]) == 1u && e < n;
            if (take) {
                const uint32_t tag = hinge_code((x >= P) + (x >= 2 * P));
                take = claim_open(s.claim + e, tag) && claim_put(s.claim + e, tag) == kUnc;
            }
            who[q] = __ballot_sync(0xFFFFFFFFu, take);
        }
        const uint32_t lane = tid & 31u;
        uint32_t at = 0;
        if (lane == 0)
            at = atomicAdd(&lcur, (uint32_t)(__popc(who[0]) + __popc(who[1]) + __popc(who[2]) +
                                             __popc(who[3])));
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if ((who[q] >> lane) & 1u)
                s.L[at + __popc(who[q] & ((1u << lane) - 1u))] = (uint16_t)V::sum(r[q]);
            at += __popc(who[q]);
        }
    }
    // DeleteEdge of the i-th listed edge in round t: take[k] when the vertex
    // that loses it is the first to claim its last edge f[k]
    auto delete_edge = [&](uint32_t i, uint32_t t, bool(&take)[2], uint32_t(&f)[2]) {
        const uint32_t e = s.L[i];
        const uint32_t h = hinge_of(s.claim[e]);
        const uint32_t j0 = h == 0 ? 1u : 0u, j1 = h == 2 ? 1u : 2u;
        uint32_t x[2];
        if (VERTS) {
            x[0] = s.V[j0 * n + e] + j0 * P;
            x[1] = s.V[j1 * n + e] + j1 * P;
        } else {
            uint32_t v[3];
            bucket_edge(__ldg(keys + e), seed, fm, P, v);
            x[0] = h == 0 ? v[1] : v[0];
            x[1] = h == 2 ? v[1] : v[2];
        }
        T old[2];
#pragma unroll
        for (int k = 0; k < 2; k++) old[k] = atomicAdd(s.rec + x[k], (T)(0) - V::unit(e));
        // both claim words are read before either is claimed
#pragma unroll
        for (int k = 0; k < 2; k++) {
            f[k] = (V::sum(old[k]) - e) & V::mask();
            take[k] = V::deg(old[k]) == 2u && f[k] < n &&
                      claim_open(s.claim + f[k], (t + 1) << 2);
        }
#pragma unroll
        for (int k = 0; k < 2; k++)
            if (take[k])
                take[k] = claim_put(s.claim + f[k], ((t + 1) << 2) | hinge_code(k ? j1 : j0)) == kUnc;
    };
    // Rounds, one block barrier each: round t appends layer t + 1 from its
    // start le through counter t mod 3.  Every thread reads that counter just
    // after the round's barrier; the counter round t + 1 will use was last
    // read before the previous barrier, so thread 0 clears it during round t.
    // A layer of at most kWarpLayer edges, and those after it while they stay
    // as small, are run by one warp, with no block barrier and no counter: a
    // bucket of 2,000 keys has 37 rounds, 33 of them on 64 edges or fewer, and
    // a round of the block took 2,900 cycles (47 % of the warps' time at its
    // barrier) whatever its layer held.  With the claims by one atomicAnd and
    // the vector scan of round 0: 9.33 -> 8.02 ms for 65,536 lognormal buckets.
    uint32_t *cnt3 = sh + 4;  // sh[4..6]
    __syncthreads();
    if (tid == 0) {
        s.loff[0] = 0;
        s.loff[1] = lcur;
        cnt3[0] = cnt3[1] = cnt3[2] = 0;
    }
    __syncthreads();
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t t = 0, lb = 0, le = s.loff[1];
    bool too_many = false;
    while (le > lb) {
        if (t + 2 > s.rcap) {  // more rounds than the table holds (block-uniform)
            too_many = true;
            break;
        }
        if (le - lb <= kWarpLayer) {
            __syncthreads();  // every thread has read the last round's counter
            if (warp == 0) {
                do {
                    uint32_t next = le;
                    for (uint32_t i0 = lb; i0 < le; i0 += 32u) {
                        bool take[2] = {false, false};
                        uint32_t f[2] = {0, 0};
                        if (i0 + lane < le) delete_edge(i0 + lane, t, take, f);
                        const uint32_t b0 = __ballot_sync(0xFFFFFFFFu, take[0]);
                        const uint32_t b1 = __ballot_sync(0xFFFFFFFFu, take[1]);
                        if (take[0]) s.L[next + __popc(b0 & lt)] = (uint16_t)f[0];
                        next += __popc(b0);
                        if (take[1]) s.L[next + __popc(b1 & lt)] = (uint16_t)f[1];
                        next += __popc(b1);
                    }
                    if (lane == 0) s.loff[t + 2] = next;
                    __syncwarp();
                    lb = le;
                    le = next;
                    t++;
                } while (le > lb && le - lb <= kWarpLayer && t + 2 <= s.rcap);
                if (lane == 0) {
                    cnt3[0] = cnt3[1] = cnt3[2] = 0;
                    sh[0] = t;
                }
            }
            __syncthreads();
            t = *(volatile uint32_t *)(sh + 0);
            lb = s.loff[t];
            le = s.loff[t + 1];
            continue;
        }
        uint32_t *cur = cnt3 + t % 3;
        if (tid == 0) cnt3[(t + 1) % 3] = 0;
        for (uint32_t i0 = lb; i0 < le; i0 += T_) {
            const uint32_t i = i0 + tid;
            bool take[2] = {false, false};
            uint32_t f[2] = {0, 0};
            if (i < le) delete_edge(i, t, take, f);
            cta_append2(cur, s.L, le, take, f);
        }
        __syncthreads();
        const uint32_t next = le + *(volatile uint32_t *)cur;
        if (tid == 0) s.loff[t + 2] = next;
        lb = le;
        le = next;
        t++;
    }
    const uint32_t R = t;
    const uint32_t peeled = lb;  // loff[R]: the empty layer R starts where L ends
    __syncthreads();
    uint32_t *out = a.order + key0;
    if (too_many) return false;  // block-uniform
    // canonical order.  Every warp takes a run of consecutive edges: counts
    // per layer, the layers' starts and the counts of the lower warps give
    // where its edges of a layer go, and a second walk places them in id order
    // (the vertex records are dead: their space holds the counts).
    const uint32_t nw = T_ / 32u;
    auto key_of = [&](uint32_t e) {
        const uint32_t c = s.claim[e];
        return c == kUnc ? R : c >> 2;
    };
    if ((size_t)nw * (R + 1) * 4 <= (size_t)m * sizeof(T)) {
        uint32_t *wh = reinterpret_cast<uint32_t *>(s.rec) + warp * (R + 1);
        for (uint32_t r = lane; r <= R; r += 32) wh[r] = 0;
        __syncwarp();
        const uint32_t run = ((n + nw - 1) / nw + 31u) & ~31u;
        const uint32_t e_lo = min(warp * run, n), e_hi = min(e_lo + run, n);
        for (uint32_t e0 = e_lo; e0 < e_hi; e0 += 32) {
            const uint32_t e = e0 + lane;
            if (e < e_hi) atomicAdd(wh + key_of(e), 1u);
        }
        __syncthreads();
        for (uint32_t r = tid; r <= R; r += T_) {
            uint32_t at = r < R ? s.loff[r] : peeled;
            uint32_t *p = reinterpret_cast<uint32_t *>(s.rec) + r;
            for (uint32_t w = 0; w < nw; w++, p += R + 1) {
                const uint32_t c = *p;
                *p = at;
                at += c;
            }
        }
        __syncthreads();
        for (uint32_t e0 = e_lo; e0 < e_hi; e0 += 32) {
            const uint32_t e = e0 + lane;
            const bool valid = e < e_hi;
            const uint32_t key = valid ? key_of(e) : 0xFFFFFFFFu;
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, key);
            const uint32_t below = __popc(peers & lt);
            uint32_t at = 0;
            if (valid) {
                at = wh[key];
                out[at + below] = e;
            }
            __syncwarp();
            if (valid && below == 0) wh[key] = at + __popc(peers);
            __syncwarp();
        }
    } else if (warp == 0) {
        // more layers than the records' space holds: one warp walks all edges,
        // the running start of every layer in cnt[0..R]
        uint32_t *cnt = s.cnt;
        for (uint32_t r = lane; r <= R; r += 32) cnt[r] = r < R ? s.loff[r] : peeled;
        __syncwarp();
        for (uint32_t e0 = 0; e0 < n; e0 += 32) {
            const uint32_t e = e0 + lane;
            const bool valid = e < n;
            const uint32_t key = valid ? key_of(e) : 0xFFFFFFFFu;
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, key);
            if (valid) out[cnt[key] + __popc(peers & lt)] = e;
            __syncwarp();
            if (valid && lane == (uint32_t)(__ffs(peers) - 1)) cnt[key] += __popc(peers);
            __syncwarp();
        }
    }
    if (tid == 0) {
        if (a.status) a.status[b] = peeled < n ? 1u : 0u;
        if (a.rounds) a.rounds[b] = R;
    }
    __syncthreads();
    // MWHC g values (sec. 3), last layer first: layer r is L[loff[r],
    // loff[r + 1]).
    if (a.G && peeled == n) {
        const uint32_t words = (m + 15) / 16;
        for (uint32_t w = tid; w < words; w += T_) s.G[w] = 0;
        __syncthreads();
        auto solve = [&](uint32_t i) {
            const uint32_t e = s.L[i];
            const uint32_t h = hinge_of(s.claim[e]);
            uint32_t v[3];
            if (VERTS) {
#pragma unroll
                for (int j = 0; j < 3; j++) v[j] = s.V[(uint32_t)j * n + e] + (uint32_t)j * P;
            } else {
                bucket_edge(__ldg(keys + e), seed, fm, P, v);
            }
            uint32_t sum = 0;
#pragma unroll
            for (int j = 0; j < 3; j++)
                if ((uint32_t)j != h)
                    sum += (((volatile uint32_t *)s.G)[v[j] >> 4] >> (2 * (v[j] & 15))) & 3u;
            const uint32_t val = (h + 6u - sum) % 3u;
            const uint32_t vh = h == 0 ? v[0] : (h == 1 ? v[1] : v[2]);
            atomicOr(s.G + (vh >> 4), (val ? val : 3u) << (2 * (vh & 15)));
        };
        for (int32_t r = (int32_t)R - 1; r >= 0; r--) {
            const uint32_t lo = s.loff[r], hi = s.loff[r + 1];
            if (hi - lo <= kWarpLayer) {  // a run of small layers: one warp (see the rounds)
                int32_t q = r;
                uint32_t top = hi;
                for (; q >= 0; q--) {
                    const uint32_t bot = s.loff[q];
                    if (top - bot > kWarpLayer) break;
                    if (warp == 0) {
                        for (uint32_t i = bot + lane; i < top; i += 32u) solve(i);
                        __syncwarp();
                    }
                    top = bot;
                }
                r = q + 1;
            } else {
                for (uint32_t i = lo + tid; i < hi; i += T_) solve(i);
            }
            __syncthreads();
        }
        uint64_t *dst = a.G + a.G_off[b];
        const uint32_t words64 = (m + 31) / 32;
        for (uint32_t w = tid; w < words64; w += T_) {
            const uint64_t lo32 = s.G[2 * w];
            const uint64_t hi32 = (2 * w + 1 < words) ? s.G[2 * w + 1] : 0u;
            dst[w] = lo32 | (hi32 << 32);
        }
    } else if (a.G) {
        uint64_t *dst = a.G + a.G_off[b];
        const uint32_t words64 = (m + 31) / 32;
        for (uint32_t w = tid; w < words64; w += T_) dst[w] = 0;
    }
    __syncthreads();
    return true;
}


// 32 registers and so 2,048 threads per SM (9.57 ms for 65,536 lognormal
// buckets; with 56 registers 9.84, with 40 by __maxnreg__ 11.06).
__global__ void __launch_bounds__(1024, 2) k_batched(BatchArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ __align__(16) uint32_t sh[8];  // sh[2..3] hold a 64-bit value
    __shared__ uint32_t s_b;
    if (a.wait) asm volatile("griddepcontrol.wait;" ::: "memory");
    // the next class's blocks may start as this one's leave (see launch_batched)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    char *region = a.scratch + (size_t)blockIdx.x * a.scratch_bytes;
    const uint32_t lo = a.range ? __ldcg(a.range) : 0u, hi = a.range ? __ldcg(a.range + 1) : a.B;
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t k = lo < hi ? lo + atomicAdd(a.next, 1u) : hi;
            s_b = k < hi ? __ldcg(a.sched + k) : 0xFFFFFFFFu;
        }
        __syncthreads();
        const uint32_t b = s_b;
        __syncthreads();
        if (b == 0xFFFFFFFFu) break;
        const uint64_t n64 = a.off[b + 1] - a.off[b];
        if (n64 == 0 || n64 > kBatchMaxEdges) {
            if (threadIdx.x == 0) {
                if (a.status) a.status[b] = n64 == 0 ? 0u : 2u;
                if (a.rounds) a.rounds[b] = 0;
            }
            if (a.G && n64 == 0) {
                // nothing to write: an empty bucket has no g words
            }
            continue;
        }
        const uint32_t n = (uint32_t)n64;
        const uint32_t m = bucket_vertices(n, a.gamma_milli);
        const uint32_t rcap_s = min(n + 1, a.smem_rounds);
        bool done = false;
        if (n < 0xFFFFu) {
            if (bucket_bytes(n, m, 4, 2, rcap_s, true) <= a.smem_bytes)
                done = run_bucket<uint32_t, uint16_t, true>(
                    a, b, carve<uint32_t, uint16_t>(smem, n, m, rcap_s, true), n, m, sh);
            else if (bucket_bytes(n, m, 4, 2, rcap_s) <= a.smem_bytes)
                done = run_bucket<uint32_t, uint16_t, false>(
                    a, b, carve<uint32_t, uint16_t>(smem, n, m, rcap_s), n, m, sh);
        }
        if (!done && a.late) {
            if (threadIdx.x == 0) a.late[atomicAdd(a.late_count, 1u)] = b;
            continue;
        }
        // the global region: 32-bit records and 16-bit claims when the
        // 16-bit fields hold the bucket (fewer than 2^16 - 1 edges, at most
        // global16_rounds <= kClaim16Rounds rounds), as in shared memory;
        // else 64-bit records and 32-bit claims with room for every round
        // (n + 1 layer starts)
        if (!done && n < 0xFFFFu)
            done = run_bucket<uint32_t, uint16_t, false>(
                a, b, carve<uint32_t, uint16_t>(region, n, m, min(n + 1, a.global16_rounds)), n,
                m, sh);
        if (!done)
            run_bucket<unsigned long long, uint32_t, false>(
                a, b, carve<unsigned long long, uint32_t>(region, n, m, n + 1), n, m, sh);
    }
    // a launch ends only after the one before it
    if (blockIdx.x == 0 && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Word offsets of the buckets' g arrays: G_off[b] = sum of ceil(m_c / 32)
// over c < b (the scan kernel turns counts into offsets).
__global__ void k_batch_g_words(const uint64_t *off, uint32_t B, uint32_t gamma_milli,
                                uint32_t *words) {
    for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
        const uint64_t n = off[b + 1] - off[b];
        words[b] = n <= kBatchMaxEdges ? (bucket_vertices((uint32_t)n, gamma_milli) + 31) / 32 : 0u;
    }
}

__global__ void k_widen_u32(const uint32_t *in, const uint32_t *cnt, uint32_t B, uint64_t *out) {
    for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b <= B; b += gridDim.x * blockDim.x)
        out[b] = b < B ? (uint64_t)in[b] : (B ? (uint64_t)in[B - 1] + cnt[B - 1] : 0ull);
}

void launch_batch_g_offsets(const Launch &L, const uint64_t *off, uint32_t B, uint32_t gamma_milli,
                            uint32_t *words, uint32_t *scanned, uint32_t *tmp, uint64_t *G_off) {
    count_launch();
    k_batch_g_words<<<grid_for(L, B ? B : 1, 1, 4), kThreads, 0, L.stream>>>(off, B, gamma_milli,
                                                                             words);
    launch_scan_u32(L, words, scanned, B, tmp);
    count_launch();
    k_widen_u32<<<grid_for(L, (uint64_t)B + 1, 1, 4), kThreads, 0, L.stream>>>(scanned, words, B,
                                                                               G_off);
}

// Launch classes: buckets of one size range in one launch, with the blocks per
// SM (and so the shared memory per block) and the threads that suit them.  One
// shape for all sizes leaves half the keys of a lognormal workload in the
// global regions (2.01e8 keys in 65,536 buckets: 14.9 ms at 256 threads x 6
// blocks, the best single shape).  Rates of uniform buckets (keys per us and
// SM, with g values) at the class's shape and at the best other of 24: 200 keys
// 140 / 154 (128 threads x 16), 500 191 / 211 (128 x 16), 1000 189 / 226 (128 x
// 12), 1500 197 / 200, 2000 188 / 174, 3500 177 / 174, 4000 160 / 156, 6000 143 /
// 140, 8000 120 / 120, 12000 114 / 113, 24000 101 / 102.  (The classes were chosen
// before one warp took the small layers, when each was the best at its sizes.)
struct BatchClass {
    uint32_t threads, ctas;
    bool verts;   // takes buckets whose vertices fit beside their state, or
    int launch;   // any that fit; index of the launch (largest buckets first)
};
constexpr int kBatchLaunches = 9;  // 0: the global regions
constexpr int kBatchClasses = 11;
struct BatchShapes {
    uint32_t smem[kBatchClasses];  // dynamic shared memory of a class's block
    uint32_t launch[kBatchClasses];
    bool verts[kBatchClasses];
    uint32_t smem_rounds, gamma_milli;
};
// tried in this order, the first that holds the bucket takes it
constexpr BatchClass kBatchClass[kBatchClasses] = {
    {64, 24, true, 8},  {128, 12, true, 7}, {128, 8, true, 6},  {256, 6, true, 5},
    {384, 4, true, 4},  {384, 3, true, 3},  {384, 4, false, 4}, {512, 2, true, 2},
    {384, 3, false, 3}, {512, 2, false, 2}, {768, 1, false, 1}};

__device__ __forceinline__ uint32_t batch_launch(const BatchShapes &s, uint32_t n) {
    const uint32_t m = bucket_vertices(n, s.gamma_milli), rcap = min(n + 1, s.smem_rounds);
    const size_t plain = bucket_bytes(n, m, 4, 2, rcap), verts = bucket_bytes(n, m, 4, 2, rcap, true);
    if (n >= 0xFFFFu) return 0;
#pragma unroll
    for (int c = 0; c < kBatchClasses; c++)
        if ((s.verts[c] ? verts : plain) <= s.smem[c]) return s.launch[c];
    return 0;
}

// Schedule: buckets by launch, largest first inside a launch (quarters of an
// octave), by one cluster.  ctl: [0 .. kBatchLaunches] the launches' starts
// (and end), from 16 on their counters, then the late list's count and counter.
// plain: one launch of all buckets, largest first.
constexpr uint32_t kBatchSizes = 4 * 17 + 1;  // quarter octaves up to 2^17
constexpr uint32_t kBatchBins = kBatchLaunches * kBatchSizes;
constexpr uint32_t kBatchCtlNext = 16, kBatchCtlLate = 32, kBatchCtlWords = 34;
__global__ void __launch_bounds__(1024)
k_batch_schedule(const uint64_t *off, uint32_t B, BatchShapes shapes, uint32_t plain, uint32_t *sched,
                 uint32_t *ctl) {
    __shared__ uint32_t cnt[kBatchBins], total[kBatchBins], low[kBatchBins];
    const uint32_t tid = threadIdx.x, rank = cl_rank(), blocks = gridDim.x;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto bin_of = [&](uint32_t b) {
        const uint64_t n64 = off[b + 1] - off[b];
        const uint32_t n = (uint32_t)(n64 < 131071u ? n64 : 131071u);
        // larger sizes in lower bins; a bucket past the limit is only reported
        const uint32_t lg = n ? 31u - __clz(n) : 0u;
        const uint32_t q = n ? 4u * lg + (lg >= 2 ? (n >> (lg - 2)) & 3u : 0u) + 1u : 0u;
        const uint32_t launch = plain ? 0u : (n64 > kBatchMaxEdges ? 0u : batch_launch(shapes, n));
        return launch * kBatchSizes + (kBatchSizes - 1u - q);
    };
    for (uint32_t i = tid; i < kBatchBins; i += 1024) cnt[i] = 0;
    cl_sync<false>();
    const uint32_t stride = blocks * 1024u, first = rank * 1024u + tid;
    for (uint64_t b = first; b < B; b += stride) atomicAdd(&cnt[bin_of((uint32_t)b)], 1u);
    cl_sync<false>();
    for (uint32_t i = tid; i < kBatchBins; i += 1024) {
        uint32_t s = 0, l = 0;
        for (uint32_t c = 0; c < blocks; c++) {
            if (c == rank) l = s;
            s += cl_load<false>(cl_map<false>(smem_u32(cnt + i), c));
        }
        total[i] = s;
        low[i] = l;
    }
    cl_sync<false>();  // the counts are read: they become cursors
    block_scan_counts<1024>(total, cnt, kBatchBins);
    if (rank == 0) {
        if (tid < kBatchLaunches) ctl[tid] = cnt[tid * kBatchSizes];
        if (tid == kBatchLaunches) ctl[tid] = B;
        if (tid >= kBatchCtlNext && tid < kBatchCtlWords) ctl[tid] = 0;
    }
    __syncthreads();
    for (uint32_t i = tid; i < kBatchBins; i += 1024) cnt[i] += low[i];
    __syncthreads();
    for (uint64_t b = first; b < B; b += stride)
        sched[atomicAdd(&cnt[bin_of((uint32_t)b)], 1u)] = (uint32_t)b;
}

// Per-CTA global region: the largest bucket at this sparsity.
size_t batched_scratch_bytes(uint32_t gamma_milli) {
    const uint64_t gn = ((uint64_t)kBatchMaxEdges * gamma_milli + 999u) / 1000u;
    const uint32_t mmax = (uint32_t)((gn + 2) / 3 * 3);
    return (bucket_bytes(kBatchMaxEdges, mmax, 8, 4, kBatchMaxEdges + 1) + 255) & ~(size_t)255;
}

uint32_t batched_claim16_rounds() { return kClaim16Rounds; }

uint32_t batched_max_gamma_milli() {
    // largest gamma whose biggest bucket keeps its vertex ids within 17 bits
    uint32_t g = 1000;
    while (true) {
        const uint64_t gn = ((uint64_t)kBatchMaxEdges * (g + 1) + 999u) / 1000u;
        if ((gn + 2) / 3 * 3 > kBatchMaxVertices) return g;
        g++;
    }
}

void launch_batched(const Launch &L, const uint64_t *keys, const uint64_t *off, uint32_t B,
                    uint32_t gamma_milli, uint32_t *order, uint32_t *rounds, uint32_t *status,
                    uint64_t *G, const uint64_t *G_off, uint32_t threads, uint32_t ctas,
                    uint32_t smem_bytes, uint32_t smem_rounds, uint32_t global16_rounds,
                    uint32_t smem_per_sm, uint32_t *sched, uint32_t *ctl, uint32_t *late,
                    char *scratch) {
    const bool classes = smem_per_sm != 0;
    // Few buckets: a class with more blocks per SM than hold them all at once is
    // left out (its buckets run in the next larger one), and no launch has more
    // blocks than there are buckets.  An empty launch of a full grid costs
    // 4 us, of few blocks 1.6.  Per call, buckets of one size; one launch of the
    // default shape / all classes on full grids / this: 1 bucket of 64 keys
    // 23 / 54 / 20 us, of 2,000 66 / 66 / 32, 16 of 64 28 / 54 / 22, 256 of 64
    // 36 / 62 / 35, 256 of 2,000 154 / 100 / 75, 1,024 of 64 65 / 67 / 51.
    uint32_t most = 0;
    for (int c = kBatchClasses - 1; c >= 0; c--)
        if (most == 0 || (uint64_t)L.sms * most < B) most = std::max(most, kBatchClass[c].ctas);
    BatchShapes sh{};
    sh.smem_rounds = smem_rounds;
    sh.gamma_milli = gamma_milli;
    smem_optin((const void *)k_batched);
    // what a block may ask for, and what the SM holds of them (1 KB per block
    // is reserved, 64 B static)
    for (int c = 0; c < kBatchClasses; c++) {
        sh.launch[c] = (uint32_t)kBatchClass[c].launch;
        sh.verts[c] = kBatchClass[c].verts;
        sh.smem[c] = classes && kBatchClass[c].ctas <= most
                         ? std::min(smem_bytes, (smem_per_sm / kBatchClass[c].ctas - 1024 - 64) & ~15u)
                         : 0u;
    }
    {
        uint32_t plain = classes ? 0u : 1u;
        uint32_t blocks = max_cluster((const void *)k_batch_schedule, 1024, 0);
        if (blocks == 0) blocks = 1;
        while (blocks > 1 && (uint64_t)(blocks / 2) * 1024u >= B) blocks /= 2;
        void *args[] = {(void *)&off, (void *)&B, (void *)&sh, (void *)&plain, (void *)&sched,
                        (void *)&ctl};
        count_launch();
        launch_cluster((const void *)k_batch_schedule, blocks, 1024, 0, L.stream, args);
    }
    BatchArgs a{keys, off, B, gamma_milli, sched, nullptr, ctl + kBatchCtlNext, nullptr, nullptr,
                order, rounds, status, G, G_off, scratch, batched_scratch_bytes(gamma_milli),
                smem_bytes, smem_rounds, global16_rounds, 0u};
    if (!classes) {
        count_launch();
        k_batched<<<ctas, threads, smem_bytes, L.stream>>>(a);
        return;
    }
    // The launches overlap: each lets the next one's blocks start as its own
    // leave (programmatic dependent launch; they share nothing but the
    // outputs, bucket by bucket), and ends only after the one before it.  The
    // first waits for the schedule before it lets any other start.  The
    // last takes the buckets that needed more rounds than their class's shared
    // memory holds; it shares the global regions with the first, so it waits
    // until all others have ended.
    for (int l = 0; l <= kBatchLaunches; l++) {
        const bool global = l == 0 || l == kBatchLaunches;
        BatchArgs x = a;
        uint32_t th = 1024, per = global ? 2 : 0;
        for (int c = 0; c < kBatchClasses && !global; c++)
            if (kBatchClass[c].launch == l && sh.smem[c]) {
                th = kBatchClass[c].threads;
                per = kBatchClass[c].ctas;
                x.smem_bytes = sh.smem[c];
            }
        if (per == 0) continue;
        if (l < kBatchLaunches) {
            x.range = ctl + l;
            x.next = ctl + kBatchCtlNext + l;
        } else {
            x.sched = late;
            x.range = ctl + kBatchCtlLate - 1;  // 0, the late buckets' count
            x.next = ctl + kBatchCtlLate + 1;
        }
        x.wait = global ? 1u : 0u;
        if (global) {
            x.smem_bytes = 0;
        } else {
            x.late = late;
            x.late_count = ctl + kBatchCtlLate;
        }
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(std::min((unsigned)L.sms * per, B));
        cfg.blockDim = dim3(th);
        cfg.dynamicSmemBytes = x.smem_bytes;
        cfg.stream = L.stream;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        void *args[] = {(void *)&x};
        count_launch();
        cudaLaunchKernelExC(&cfg, (const void *)k_batched, args);
    }
}

}  // namespace hp
