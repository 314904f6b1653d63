// small.cu -- small graphs: the whole path in one launch, one thread-block
// cluster, the graph spread over the cluster's shared memory.
//
// A peel of up to 2^17 edges fits the shared memory of at most 16 SMs, and
// its cost is the latency of its rounds, not the work in them: sec. 4.2's
// rounds are a chain, 40-70 of them whatever n is.  The general path pays a
// kernel launch and four to eight trips to L2 per round (12 us on a GB300,
// measured at n = 1e3 and n = 1e5 alike).  Here a round is one pass over the
// cluster's own edges, one shared-memory atomic per deleted incidence and one
// hardware barrier (barrier.cluster between blocks: no spinning, and the
// hardware starts the blocks of a cluster together): 0.35 us per round at
// n = 1e3, 0.9 us at 12,000, 1.9 us at 1e5.  MPHF build of 1009 keys 810-1000 ->
// 56-63 us (kernel 31 us where the first seed peels), hash and peel of 1e5 edges
// 830-910 -> 183-198 us (kernel of the peel 168 us).
//
// Layout.  Block c of the cluster owns epc consecutive edges (their vertices
// and claim words) and every vertex whose 512-vertex group is c modulo the
// cluster size, so a vertex group's words of G and of the rank directory come
// from one block.  A vertex record is 32 bits: degree in the low 15, sum of
// incident edge ids modulo 2^17 above (sec. 4.1's packed list, with addition
// instead of XOR as in peel.cu).  A degree of 2^15 or more would carry into
// the sum; it shows as a total of the degrees other than r n after the build,
// and the attempt is then run again with 64-bit records in the workspace.
//
// Rounds.  Layer t is the set of edges whose claim word holds round t.  There
// is no layer list: the atomic that takes a vertex from degree 2 to 1 names
// its last edge f (old sum - e), and the vertex's claim is a minimum on f's claim
// word in its owner's shared memory that nothing waits for; the owner finds its
// part of the next layer in its own claim words.  All claims of a round are
// in before the barrier, so the claim word names the hinge when the edge is
// deleted.  Three forms, by size:
//   EPT = 1, 4  one block of up to 1024 threads, each with 1 or 4 edges whose
//               record addresses stay in registers: a round is one load of
//               the claim words, two atomics, one minimum, one block barrier;
//   EPT = 16    16 edges per thread; a claim also sets its edge's bit in a
//               bitmap, so a round reads one 16-bit word per thread instead
//               of 16 claim words.  In one block while the graph fits its
//               shared memory (a local atomic takes 78 cycles and a block
//               barrier 21-78, a remote atomic 335 and a cluster barrier
//               370-600; one SM serves 7.6 local atomics a cycle, a remote one
//               0.3), else over a cluster of up to 16 blocks.  There the end
//               shows two rounds late: one warp per block gathers the blocks'
//               "deleted something" flags of round t during round t + 1, and
//               everyone reads the outcome in round t + 2.
#include "cluster.cuh"
#include "kernels.cuh"

namespace hp {

namespace {

constexpr uint32_t kSmThreads = 1024;
constexpr uint32_t kSmScan = 4;                    // rounds whose layer is read off the claim words
constexpr uint32_t kSmMaxGroups = 384;             // vertex groups of an MPHF (parts below 2^16)
constexpr uint32_t kSmMaxEdges = 1u << 17;         // 17-bit id sums
constexpr uint32_t kSmDegBits = 15;
constexpr uint32_t kSmDegMask = (1u << kSmDegBits) - 1u;
constexpr uint32_t kSmSumMask = (1u << (32 - kSmDegBits)) - 1u;
constexpr uint32_t kSmBins = 256;                  // layers per pass of the order
constexpr uint32_t kSmWarpGroups = 16;             // groups of 32 edges per warp at most
constexpr uint32_t kSmGroup = 9;                   // log2 of the vertices per group
constexpr size_t kSmMaxSmem = 224u << 10;          // dynamic shared memory of a block

// ------------------------------------------------------------ one block --
struct SmallShared {
    uint32_t any[4];   // this block deleted an edge in round t, slot t mod 4
    uint32_t all[4];   // the same over the cluster
    uint32_t deg;      // sum of the degrees of this block's vertices
    uint32_t bad;      // an input edge of this block is invalid
    uint32_t cross;    // vertices that fell from degree 2 to 1
    uint32_t moves;    // this block's edges with two claims or more in their round
    uint32_t err;      // device error code of this block
    uint32_t peeled;   // peeled edges of this block
    uint32_t first;    // those of layer 0
    uint32_t base;     // order: edges in the layers before this pass
    uint32_t listed;   // edges in this block's list
    uint32_t gcnt[kSmMaxGroups];  // assigned vertices per group (block 0)
};

// Stored vertex of an edge: its place in its part (16 bits); a general
// graph's ids keep 32.
template <bool GEN>
struct SmallVertex {
    using type = uint16_t;
};
template <>
struct SmallVertex<true> {
    using type = uint32_t;
};

// This block's view: its arrays and their shared addresses (the same in
// every block).
template <bool GEN>
struct SmallView {
    using V = typename SmallVertex<GEN>::type;
    uint32_t rank, blocks, lc;  // cluster rank, size and its log2
    uint32_t e0, ne;            // first edge and edges of this block
    uint32_t vslots;            // vertex slots of a block
    uint32_t *claim, *rec;      // [epc], [vslots]
    uint32_t *hits;             // claims of this block's edges beyond the first (small_claim)
    uint32_t *bits;             // EPT = 16: [2][epc / 32], claims of even and odd rounds
    uint16_t *list;             // EPT = 16: [epc] this block's edges in the order they go
    V *vert;                    // [R][epc] (EPT = 16, or a general graph)
    uint32_t s_claim, s_rec, s_hits, s_bits, s_vert;
};

template <bool SOLO>
__device__ __forceinline__ uint32_t edge_owner(const SmallArgs &a, uint32_t e) {
    return SOLO ? 0u : __umulhi(e, a.epc_magic);  // e / epc, exact for e < 2^17
}
template <bool SOLO, bool GEN>
__device__ __forceinline__ uint32_t rec_addr(const SmallView<GEN> &w, uint32_t v) {
    if (SOLO) return w.s_rec + 4u * v;
    const uint32_t g = v >> kSmGroup;
    const uint32_t slot = ((g >> w.lc) << kSmGroup) | (v & ((1u << kSmGroup) - 1u));
    return cl_map<SOLO>(w.s_rec + 4u * slot, g & (w.blocks - 1u));
}
// vertex id of this block's slot
template <bool GEN>
__device__ __forceinline__ uint32_t slot_vertex(const SmallView<GEN> &w, uint32_t slot) {
    return ((((slot >> kSmGroup) << w.lc) | w.rank) << kSmGroup) | (slot & ((1u << kSmGroup) - 1u));
}
// vertex j of this block's edge i
template <bool GEN>
__device__ __forceinline__ uint32_t edge_vertex(const SmallArgs &a, const SmallView<GEN> &w,
                                                uint32_t i, uint32_t j) {
    return (uint32_t)w.vert[j * a.epc + i] + (GEN ? 0u : j * a.P);
}

// A cluster's claims of one thread for one round, whose outcomes have not been
// looked at: the claim words they found (all ones: none, or the edge's first
// claim) and their edges.
template <int N>
struct SmallPending {
    uint32_t old[N], edge[N], t;
};

// Claim of edge f for round t by vertex x at position j of
// its edges (in a general graph: at the first slot of f's row that holds x).
// Edges with two claims or more are counted.  In one block each edge has a byte,
// 4 bits for the claims of even rounds and 4 for those of odd ones: an edge
// deleted in round t has claims for t, and late ones for t + 1, which do not
// count (one more local addition; looking at the minimum's result takes 1 us
// more of 12.6 for a peel of 1009 edges).  In a cluster a second remote atomic
// takes 8 us more of 148 for a peel of 1e5 edges, the minimum's result (`old`),
// looked at later, 3.
template <int R, bool GEN, bool SOLO, bool BITS>
__device__ __forceinline__ void small_claim(const SmallArgs &a, const SmallView<GEN> &w, uint32_t f,
                                            uint32_t x, uint32_t j, uint32_t t, uint32_t &old) {
    const uint32_t o = edge_owner<SOLO>(a, f), i = f - o * a.epc;
    if (GEN) {
        j = R - 1;
#pragma unroll
        for (int k = R - 2; k >= 0; k--)
            j = cl_load<SOLO>(cl_map<SOLO>(w.s_vert + 4u * ((uint32_t)k * a.epc + i), o)) == x
                    ? (uint32_t)k
                    : j;
    }
    const uint32_t at = cl_map<SOLO>(w.s_claim + 4u * i, o);
    if (SOLO) {
        cl_red_min<SOLO>(at, (t << 2) | j);
        cl_red_add<SOLO>(w.s_hits + (i & ~3u), 1u << (8u * (i & 3u) + 4u * (t & 1u)));
    } else {
        old = cl_min<SOLO>(at, (t << 2) | j);
    }
    if (BITS && t >= kSmScan)
        cl_red_or<SOLO>(cl_map<SOLO>(w.s_bits + 4u * ((t & 1u) * (a.epc >> 5) + (i >> 5)), o),
                        1u << (i & 31u));
}

// Looks at a thread's last claims: an edge that had a claim for the same round gets
// its bit in its owner's `hits`.  The order does not matter, so this is done
// while the thread waits for the vertices of the next edge it deletes, and
// nothing in it is waited for.
template <bool GEN, int N>
__device__ __forceinline__ void small_settle(const SmallArgs &a, const SmallView<GEN> &w,
                                             SmallPending<N> &p) {
    uint32_t all = kUnclaimed;
#pragma unroll
    for (int q = 0; q < N; q++) all &= p.old[q];
    if (all == kUnclaimed) return;
#pragma unroll
    for (int q = 0; q < N; q++) {
        if ((p.old[q] >> 2) == p.t) {
            const uint32_t o = edge_owner<false>(a, p.edge[q]), i = p.edge[q] - o * a.epc;
            cl_red_or<false>(cl_map<false>(w.s_hits + 4u * (i >> 5), o), 1u << (i & 31u));
        }
        p.old[q] = kUnclaimed;
    }
}

struct SmallPeel {
    uint32_t rounds, peeled, first_layer;
};

// Vertices of edge e: hashed from its key, or read from its row (false: a
// vertex lies outside its part).
template <int R, bool GEN, bool KEYS>
__device__ __forceinline__ bool small_edge(const SmallArgs &a, uint64_t seed, uint64_t key,
                                           uint32_t e, uint32_t (&v)[R]) {
    bool ok = true;
    if (KEYS) {
#pragma unroll
        for (int j = 0; j < R; j++)
            v[j] = (uint32_t)fastmod(mix64(key ^ (seed + (uint64_t)j)), a.fm) + (uint32_t)j * a.P;
    } else {
#pragma unroll
        for (int j = 0; j < R; j++) {
            v[j] = a.edges[(uint64_t)e * R + j];
            ok &= (v[j] - (GEN ? 0u : (uint32_t)j * a.P)) < a.P;
        }
    }
    return ok;
}

// DeleteEdge of edge e with hinge position h in round t: its other vertices
// lose it, and one that falls to degree 1 claims its last edge for round t + 1.
// pend: a cluster thread's last claims, then those made here.
// at(q): record address of the q-th vertex that is not the hinge, id(q) its id
// (called for WIDE and general graphs only).
template <int R, bool GEN, bool SOLO, bool BITS, bool WIDE, typename At, typename Id>
__device__ __forceinline__ void small_delete(const SmallArgs &a, const SmallView<GEN> &w,
                                             SmallShared &sh, uint32_t e, uint32_t h, uint32_t t,
                                             At at, Id id, uint32_t &cross,
                                             SmallPending<R - 1> &pend) {
    uint32_t deg[R - 1], f[R - 1];
#pragma unroll
    for (int q = 0; q < R - 1; q++) {
        if (WIDE) {
            const unsigned long long old =
                atomicAdd(a.wide + id(q), 0ull - (((unsigned long long)e << 32) | 1ull));
            deg[q] = (uint32_t)old;
            f[q] = (uint32_t)(old >> 32) - e;
        } else {
            deg[q] = cl_add<SOLO>(at(q), 0u - ((e << kSmDegBits) + 1u));
        }
    }
    if (!SOLO) {
        small_settle(a, w, pend);
        pend.t = t + 1u;
    }
    if (!WIDE) {
#pragma unroll
        for (int q = 0; q < R - 1; q++) {
            f[q] = ((deg[q] >> kSmDegBits) - e) & kSmSumMask;
            deg[q] &= kSmDegMask;
        }
    }
#pragma unroll
    for (int q = 0; q < R - 1; q++) {
        if (deg[q] != 2u) continue;
        cross++;
        if (f[q] < a.n) {
            small_claim<R, GEN, SOLO, BITS>(a, w, f[q], GEN ? id(q) : 0u,
                                            (uint32_t)q + ((uint32_t)q >= h ? 1u : 0u), t + 1u,
                                            pend.old[q]);
            pend.edge[q] = f[q];
        } else {
            sh.err = kDevBadEdge;
        }
    }
}
// The same for this block's edge i, from its stored vertices.
template <int R, bool GEN, bool SOLO, bool WIDE>
__device__ __forceinline__ void small_delete_at(const SmallArgs &a, const SmallView<GEN> &w,
                                                SmallShared &sh, uint32_t i, uint32_t t,
                                                uint32_t &cross, SmallPending<R - 1> &pend) {
    const uint32_t h = w.claim[i] & 3u;
    uint32_t x[R - 1];
#pragma unroll
    for (int q = 0; q < R - 1; q++)
        x[q] = edge_vertex(a, w, i, (uint32_t)q + ((uint32_t)q >= h ? 1u : 0u));
    small_delete<R, GEN, SOLO, true, WIDE>(
        a, w, sh, w.e0 + i, h, t, [&](int q) { return rec_addr<SOLO>(w, x[q]); },
        [&](int q) { return x[q]; }, cross, pend);
}

// One peel: records, round 0 and the rounds.  Every thread of the cluster
// calls it; all return the same value: 0 done, kDevBadVertex an invalid edge,
// kDevCapacity the 32-bit records overflowed (WIDE = false only).
// addr: EPT < 16: shared addresses of the records of this thread's edges
// EPT tid .. EPT tid + EPT - 1.
template <int R, bool GEN, bool KEYS, bool SOLO, int EPT, bool WIDE>
__device__ uint32_t small_peel(const SmallArgs &a, const SmallView<GEN> &w, SmallShared &sh,
                               uint64_t seed, uint32_t (&addr)[EPT < 16 ? EPT : 1][R],
                               SmallPeel &out) {
    using V = typename SmallVertex<GEN>::type;
    constexpr bool BITS = EPT == 16, LIST = KEYS;  // the assignment reads the list
    static_assert(SOLO || BITS, "a cluster takes the bitmap form");
    const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t n = a.n, m = a.m;
    for (uint32_t i = tid; i < w.vslots; i += T) {
        w.rec[i] = 0;
        if (WIDE && slot_vertex(w, i) < m) a.wide[slot_vertex(w, i)] = 0ull;
    }
    for (uint32_t i = tid; i < a.epc; i += T) w.claim[i] = kUnclaimed;
    for (uint32_t i = tid; i < (SOLO ? a.epc >> 2 : a.epc >> 5); i += T) w.hits[i] = 0;
    if (BITS)
        for (uint32_t i = tid; i < (a.epc >> 4); i += T) w.bits[i] = 0;
    if (tid < 4) sh.any[tid] = sh.all[tid] = 0;
    if (tid == 4)
        sh.deg = sh.bad = sh.cross = sh.moves = sh.err = sh.peeled = sh.first = sh.listed = 0;
    cl_sync<SOLO>();
    // AddEdge of this block's edges, four keys in flight per thread
    constexpr int kU = BITS ? 4 : EPT;
    for (uint32_t i0 = tid; i0 < w.ne; i0 += kU * T) {
        uint64_t key[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const uint32_t i = BITS ? i0 + (uint32_t)u * T : tid * EPT + (uint32_t)u;
            key[u] = KEYS && i < w.ne ? a.keys[w.e0 + i] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const uint32_t i = BITS ? i0 + (uint32_t)u * T : tid * EPT + (uint32_t)u;
            if (!BITS) {
#pragma unroll
                for (int j = 0; j < R; j++) addr[u % (EPT < 16 ? EPT : 1)][j] = w.s_rec;
            }
            if (i >= w.ne) continue;
            const uint32_t e = w.e0 + i;
            uint32_t v[R];
            const bool ok = small_edge<R, GEN, KEYS>(a, seed, key[u], e, v);
            if (!ok) sh.bad = 1;
#pragma unroll
            for (int j = 0; j < R; j++) {
                if (BITS || GEN)
                    w.vert[(uint32_t)j * a.epc + i] =
                        (V)(ok ? v[j] - (GEN ? 0u : (uint32_t)j * a.P) : 0u);
                if (!ok) continue;
                if (WIDE) {
                    atomicAdd(a.wide + v[j], ((unsigned long long)e << 32) | 1ull);
                } else {
                    const uint32_t at = rec_addr<SOLO>(w, v[j]);
                    cl_red_add<SOLO>(at, (e << kSmDegBits) + 1u);
                    if (!BITS) addr[u % (EPT < 16 ? EPT : 1)][j] = at;
                }
            }
        }
    }
    cl_sync<SOLO>();
    // round 0: every vertex of degree 1 claims its edge
    {
        constexpr int kV = SOLO ? 1 : 4;  // a cluster's claims in flight per thread
        uint32_t degs = 0;
        for (uint32_t i0 = tid; i0 < w.vslots; i0 += kV * T) {
            SmallPending<kV> pend;
            pend.t = 0;
#pragma unroll
            for (int u = 0; u < kV; u++) {
                pend.old[u] = kUnclaimed;
                const uint32_t i = i0 + (uint32_t)u * T;
                if (i >= w.vslots) continue;
                const uint32_t v = slot_vertex(w, i);
                uint32_t deg, f;
                if (WIDE) {
                    const unsigned long long r = v < m ? __ldcg(a.wide + v) : 0ull;
                    deg = (uint32_t)r;
                    f = (uint32_t)(r >> 32);
                } else {
                    const uint32_t r = w.rec[i];
                    deg = r & kSmDegMask;
                    f = r >> kSmDegBits;
                }
                degs += deg;
                pend.edge[u] = f;
                if (deg == 1u && f < n)
                    small_claim<R, GEN, SOLO, BITS>(a, w, f, v, GEN ? 0u : part_of<R>(v, a.P), 0u,
                                                    pend.old[u]);
            }
            if (!SOLO) small_settle(a, w, pend);
        }
        if (BITS && !WIDE) {  // EPT < 16: at most 4096 edges, no degree can overflow
            degs = __reduce_add_sync(0xFFFFFFFFu, degs);
            if (lane == 0 && degs) atomicAdd(&sh.deg, degs);
        }
    }
    cl_sync<SOLO>();
    {
        uint32_t degs = 0, bad = 0;
        if (lane < w.blocks) {
            degs = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.deg), lane));
            bad = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.bad), lane));
        }
        if (__any_sync(0xFFFFFFFFu, bad != 0u)) return kDevBadVertex;
        if (BITS && !WIDE && __reduce_add_sync(0xFFFFFFFFu, degs) != (uint32_t)R * n)
            return kDevCapacity;
    }
    uint32_t cross = 0, t = 0;
    SmallPending<R - 1> pend;
    pend.t = 0;
#pragma unroll
    for (int q = 0; q < R - 1; q++) {
        pend.old[q] = kUnclaimed;
        pend.edge[q] = 0;
    }
    if constexpr (!BITS) {
        for (;; t++) {
            uint32_t c[EPT];
            if constexpr (EPT == 4) {
                const uint4 q = tid * 4u < a.epc ? *reinterpret_cast<const uint4 *>(w.claim + 4u * tid)
                                                 : make_uint4(~0u, ~0u, ~0u, ~0u);
                c[0] = q.x; c[1] = q.y; c[2] = q.z; c[3] = q.w;
            } else {
                c[0] = tid < a.epc ? *(volatile uint32_t *)(w.claim + tid) : 0xFFFFFFFFu;
            }
            bool hit = false;
#pragma unroll
            for (int k = 0; k < EPT; k++) {
                if ((c[k] >> 2) != t) continue;
                hit = true;
                const uint32_t h = c[k] & 3u;
                auto at = [&](int q) { return (uint32_t)q >= h ? addr[k][q + 1] : addr[k][q]; };
                small_delete<R, GEN, SOLO, BITS, WIDE>(
                    a, w, sh, tid * EPT + (uint32_t)k, h, t, at,
                    [&](int q) { return (at(q) - w.s_rec) >> 2; }, cross, pend);
            }
            if (!__syncthreads_or(hit)) break;
        }
    } else {
        // this thread's 16 edges, 16 tid ..; a cluster's last warp has none
        const uint32_t slices = a.epc >> 4, row = a.epc >> 5;
        const bool clerk = !SOLO && warp == T / 32u - 1u;
        for (;; t++) {
            uint32_t mask = 0;
            if (tid < slices) {
                if (t < kSmScan) {
#pragma unroll
                    for (uint32_t q = 0; q < 4; q++) {
                        const uint4 c = *reinterpret_cast<const uint4 *>(w.claim + 16u * tid + 4u * q);
                        mask |= ((c.x >> 2) == t ? 1u << (4 * q) : 0u) |
                                ((c.y >> 2) == t ? 2u << (4 * q) : 0u) |
                                ((c.z >> 2) == t ? 4u << (4 * q) : 0u) |
                                ((c.w >> 2) == t ? 8u << (4 * q) : 0u);
                    }
                } else {
                    uint16_t *slice = reinterpret_cast<uint16_t *>(w.bits + (t & 1u) * row) + tid;
                    uint32_t m16 = *(volatile uint16_t *)slice;
                    if (m16) *(volatile uint16_t *)slice = 0;
                    for (; m16; m16 &= m16 - 1u) {
                        // not one claimed while it was being deleted
                        const uint32_t k = __ffs(m16) - 1u;
                        if ((w.claim[16u * tid + k] >> 2) == t) mask |= 1u << k;
                    }
                }
            }
            if (!SOLO) {
                if (t >= 2 && *(volatile uint32_t *)&sh.all[(t - 2) & 3u] == 0u) break;
                if (clerk) {
                    if (t >= 1) {
                        const uint32_t f = lane < w.blocks
                                               ? cl_load<SOLO>(cl_map<SOLO>(
                                                     smem_u32(&sh.any[(t - 1) & 3u]), lane))
                                               : 0u;
                        const bool s = __any_sync(0xFFFFFFFFu, f != 0u);
                        if (lane == 0) sh.all[(t - 1) & 3u] = s ? 1u : 0u;
                    }
                    if (lane == 0) sh.any[(t + 2) & 3u] = 0;
                }
            }
            // With at most one edge per lane each lane deletes its own; more are
            // shared out evenly through the list (two or three in turn per
            // lane: 184 us instead of 166 at n = 1e5).
            const uint32_t mine = __popc(mask);
            const uint32_t who = __ballot_sync(0xFFFFFFFFu, mine != 0u);
            const bool hit = who != 0u;
            if (hit && !__any_sync(0xFFFFFFFFu, mine > 1u)) {
                const uint32_t i = 16u * tid + __ffs(mask) - 1u;
                uint32_t base = 0;
                if (LIST && lane == 0) base = atomicAdd(&sh.listed, __popc(who));
                if (mask) small_delete_at<R, GEN, SOLO, WIDE>(a, w, sh, i, t, cross, pend);
                if (LIST) {
                    base = __shfl_sync(0xFFFFFFFFu, base, 0);
                    if (mask) w.list[base + __popc(who & ((1u << lane) - 1u))] = (uint16_t)i;
                }
            } else if (hit) {
                uint32_t x = mine;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
                    if (lane >= (uint32_t)d) x += y;
                }
                const uint32_t total = __shfl_sync(0xFFFFFFFFu, x, 31);
                uint32_t base = 0;
                if (lane == 0) base = atomicAdd(&sh.listed, total);
                base = __shfl_sync(0xFFFFFFFFu, base, 0);
                for (uint32_t at = base + x - mine; mask; mask &= mask - 1u, at++)
                    w.list[at] = (uint16_t)(16u * tid + __ffs(mask) - 1u);
                __syncwarp();
                for (uint32_t k = lane; k < total; k += 32u)
                    small_delete_at<R, GEN, SOLO, WIDE>(a, w, sh, w.list[base + k], t, cross, pend);
            }
            if (SOLO) {
                if (!__syncthreads_or(hit)) break;
            } else {
                if (hit && lane == 0) *(volatile uint32_t *)&sh.any[t & 3u] = 1u;
                cl_sync<SOLO>();
            }
        }
    }
    out.rounds = SOLO ? t : t - 2u;
    if (!SOLO) small_settle(a, w, pend);
    // what was peeled: counted off the claim words
    uint32_t peeled = 0, first = 0, moves = 0;
    for (uint32_t i = tid; i < w.ne; i += T) {
        const uint32_t c = w.claim[i];
        // (an edge that is not peeled has no claims)
        if (SOLO)
            moves += ((reinterpret_cast<const uint8_t *>(w.hits)[i] >> (c & 4u)) & 15u) > 1u ? 1u : 0u;
        peeled += c != kUnclaimed ? 1u : 0u;
        first += c < 4u ? 1u : 0u;
    }
    cross = __reduce_add_sync(0xFFFFFFFFu, cross);
    peeled = __reduce_add_sync(0xFFFFFFFFu, peeled);
    first = __reduce_add_sync(0xFFFFFFFFu, first);
    if (lane == 0) {
        if (cross) atomicAdd(&sh.cross, cross);
        if (peeled) atomicAdd(&sh.peeled, peeled);
        if (first) atomicAdd(&sh.first, first);
    }
    cl_sync<SOLO>();
    peeled = first = 0;
    if (lane < w.blocks) {
        peeled = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.peeled), lane));
        first = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.first), lane));
    }
    // (added to sh.moves, which is read after other barriers)
    if (!SOLO)
        for (uint32_t i = tid; i < (a.epc >> 5); i += T) moves += __popc(w.hits[i]);
    moves = __reduce_add_sync(0xFFFFFFFFu, moves);
    if (lane == 0 && moves) atomicAdd(&sh.moves, moves);
    out.peeled = __reduce_add_sync(0xFFFFFFFFu, peeled);
    out.first_layer = __reduce_add_sync(0xFFFFFFFFu, first);
    return 0u;
}

// Spread the 32 bits of x over the even bits of a 64-bit word.
__device__ __forceinline__ uint64_t spread_bits(uint32_t x) {
    uint64_t v = x;
    v = (v | (v << 16)) & 0x0000FFFF0000FFFFull;
    v = (v | (v << 8)) & 0x00FF00FF00FF00FFull;
    v = (v | (v << 4)) & 0x0F0F0F0F0F0F0F0Full;
    v = (v | (v << 2)) & 0x3333333333333333ull;
    v = (v | (v << 1)) & 0x5555555555555555ull;
    return v;
}

// The canonical order (layers by round, ascending ids, the 2-core last): for
// kSmBins keys at a time, each warp ranks its consecutive edges of a key, and
// a key's edges start after the smaller keys' and the lower blocks' and warps'.
// `area`: this block's scratch, past the claim words.
template <bool SOLO, bool GEN>
__device__ void small_order(const SmallArgs &a, const SmallView<GEN> &w, uint32_t *area,
                            SmallShared &sh, const SmallPeel &pe) {
    const uint32_t tid = threadIdx.x, T = blockDim.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t nw = T / 32u;
    uint32_t *tb = area;              // [kSmBins] counts of this block
    uint32_t *gb = tb + kSmBins;      // [kSmBins] counts of the lower blocks, then first place
    uint32_t *tl = gb + kSmBins;      // [kSmBins] counts of the cluster
    uint32_t *wh = tl + kSmBins;      // [nw][kSmBins] counts, then starts, of the warps
    uint32_t *mywh = wh + warp * kSmBins;
    const uint32_t groups = (w.ne + 31u) / 32u, gpw = (groups + nw - 1u) / nw;  // <= kSmWarpGroups
    const bool offs = a.layer_off && pe.rounds <= a.max_layers && w.rank == 0;
    if (tid == 0) sh.base = 0;
    for (uint32_t b0 = 0; b0 <= pe.rounds; b0 += kSmBins) {
        const uint32_t nb = min(kSmBins, pe.rounds + 1u - b0);
        for (uint32_t b = lane; b < nb; b += 32u) mywh[b] = 0;
        __syncwarp();
        uint32_t br[kSmWarpGroups];  // (bin << 16) | rank in the warp (below 512)
#pragma unroll
        for (uint32_t g = 0; g < kSmWarpGroups; g++) {
            br[g] = 0xFFFFFFFFu;
            if (g >= gpw) continue;
            uint32_t bin = 0xFFFFFFFFu;
            const uint32_t i = (warp * gpw + g) * 32u + lane;
            if (i < w.ne) {
                const uint32_t c = w.claim[i], d = (c == kUnclaimed ? pe.rounds : c >> 2) - b0;
                if (d < nb) bin = d;
            }
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, bin);
            const uint32_t below = __popc(peers & ((1u << lane) - 1u));
            const bool in = bin != 0xFFFFFFFFu;
            if (in) br[g] = (bin << 16) | (mywh[bin] + below);
            __syncwarp();
            if (in && below == 0u) mywh[bin] += __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        for (uint32_t b = tid; b < nb; b += T) {
            uint32_t s = 0;
            for (uint32_t q = 0; q < nw; q++) {
                const uint32_t c = wh[q * kSmBins + b];
                wh[q * kSmBins + b] = s;
                s += c;
            }
            tb[b] = s;
        }
        cl_sync<SOLO>();
        for (uint32_t b = tid; b < nb; b += T) {
            uint32_t s = 0, low = 0, n_c[SOLO ? 1 : 16];
#pragma unroll
            for (uint32_t c = 0; c < (SOLO ? 1u : 16u); c++)
                n_c[c] = c < w.blocks ? cl_load<SOLO>(cl_map<SOLO>(smem_u32(tb + b), c)) : 0u;
#pragma unroll
            for (uint32_t c = 0; c < (SOLO ? 1u : 16u); c++) {
                if (c < w.rank) low += n_c[c];
                s += n_c[c];
            }
            gb[b] = low;
            tl[b] = s;
        }
        __syncthreads();
        if (warp == 0) {  // the layers' starts
            uint32_t run = sh.base;
            for (uint32_t c0 = 0; c0 < nb; c0 += 32u) {
                const uint32_t b = c0 + lane, v = b < nb ? tl[b] : 0u;
                uint32_t x = v;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
                    if (lane >= (uint32_t)d) x += y;
                }
                if (b < nb) {
                    gb[b] += run + x - v;
                    if (offs) a.layer_off[b0 + b] = run + x - v;
                }
                run += __shfl_sync(0xFFFFFFFFu, x, 31);
            }
            if (lane == 0) sh.base = run;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t g = 0; g < kSmWarpGroups; g++)
            if (br[g] != 0xFFFFFFFFu)
                a.order[gb[br[g] >> 16] + mywh[br[g] >> 16] + (br[g] & 0xFFFFu)] =
                    w.e0 + (warp * gpw + g) * 32u + lane;
        cl_sync<SOLO>();  // the counts are read by other blocks; the next pass rewrites them
    }
}

// MWHC back substitution (sec. 3, sec. 4.3), last layer first: the vertex
// records' space now holds one value per vertex.  SF: values mod sigma, else
// the MPHF's codes (1, 2, 3 for 0).
// Value of an edge's hinge, given the sum of its other vertices' values.
template <bool SF>
__device__ __forceinline__ bool small_value(const SmallArgs &a, SmallShared &sh, uint32_t e,
                                            uint32_t h, uint32_t ua, uint32_t ub, uint32_t &val) {
    if (SF) {
        const uint32_t f = __ldg(a.values + e);
        if (f >= a.fs.P) {
            sh.err = kDevBadValue;
            return false;
        }
        const uint64_t other = fastmod((uint64_t)ua + ub, a.fs);
        val = (uint32_t)fastmod((uint64_t)f + a.fs.P - other, a.fs);
    } else {
        const uint32_t g = (h + 6u - ua - ub) % 3u;  // ua, ub <= 3
        val = g ? g : 3u;
    }
    return true;
}

template <bool SF, bool SOLO, int EPT>
__device__ void small_assign(const SmallArgs &a, const SmallView<false> &w, SmallShared &sh,
                             const uint32_t (&addr)[EPT < 16 ? EPT : 1][3], uint32_t rounds) {
    const uint32_t tid = threadIdx.x;
    for (uint32_t i = tid; i < w.vslots; i += blockDim.x) w.rec[i] = 0;
    cl_sync<SOLO>();
    // layer of each of this thread's edges, ~0 for none
    if constexpr (EPT < 16) {
        uint32_t c[EPT];
#pragma unroll
        for (int k = 0; k < EPT; k++)
            c[k] = tid * EPT + (uint32_t)k < w.ne ? w.claim[tid * EPT + (uint32_t)k] : 0xFFFFFFFFu;
        for (uint32_t t = rounds; t-- > 0;) {
#pragma unroll
            for (int k = 0; k < EPT; k++) {
                if ((c[k] >> 2) != t) continue;
                const uint32_t h = c[k] & 3u;
                const uint32_t u0 = h != 0 ? cl_load<SOLO>(addr[k][0]) : 0u;
                const uint32_t u1 = h != 1 ? cl_load<SOLO>(addr[k][1]) : 0u;
                const uint32_t u2 = h != 2 ? cl_load<SOLO>(addr[k][2]) : 0u;
                uint32_t val;
                if (small_value<SF>(a, sh, tid * EPT + (uint32_t)k, h, h == 0 ? u1 : u0,
                                    h == 2 ? u1 : u2, val))
                    cl_store<SOLO>(h == 0 ? addr[k][0] : (h == 1 ? addr[k][1] : addr[k][2]), val);
            }
            cl_sync<SOLO>();
        }
    } else {
        // the block's list ends with its edges of layer t
        uint32_t left = sh.listed;
        for (uint32_t t = rounds; t-- > 0;) {
            uint32_t got;
            do {
                bool mine = false;
                if (tid < left) {
                    const uint32_t i = w.list[left - 1u - tid], c = w.claim[i], h = c & 3u;
                    mine = (c >> 2) == t;
                    if (mine) {
                        const uint32_t ua = cl_load<SOLO>(
                            rec_addr<SOLO>(w, edge_vertex(a, w, i, h == 0 ? 1u : 0u)));
                        const uint32_t ub = cl_load<SOLO>(
                            rec_addr<SOLO>(w, edge_vertex(a, w, i, h == 2 ? 1u : 2u)));
                        uint32_t val;
                        if (small_value<SF>(a, sh, w.e0 + i, h, ua, ub, val))
                            cl_store<SOLO>(rec_addr<SOLO>(w, edge_vertex(a, w, i, h)), val);
                    }
                }
                got = __syncthreads_count(mine);
                left -= got;
            } while (got == blockDim.x);
            if (!SOLO) cl_sync<SOLO>();
        }
    }
}

// G words and rank counts of this block's vertex groups, then the directory.
template <bool SOLO>
__device__ void small_pack_g(const SmallArgs &a, const SmallView<false> &w, SmallShared &sh) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x / 32u;
    const uint32_t words = (a.m + 31u) / 32u, groups = (a.m + 511u) / 512u;
    for (uint32_t g = threadIdx.x; g < groups; g += blockDim.x) sh.gcnt[g] = 0;
    cl_sync<SOLO>();
    // four words at a time
    for (uint32_t u = warp; u < (w.vslots >> 7); u += nw) {
        const uint32_t g = ((u >> 2) << w.lc) | w.rank;
        if (g >= groups) break;
        uint64_t mine = 0;
        uint32_t cnt = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4; q++) {
            const uint32_t x = w.rec[(u << 7) + q * 32u + lane];
            const uint32_t lo = __ballot_sync(0xFFFFFFFFu, x & 1u);
            const uint32_t hi = __ballot_sync(0xFFFFFFFFu, x & 2u);
            cnt += __popc(lo | hi);
            if (lane == q) mine = spread_bits(lo) | (spread_bits(hi) << 1);
        }
        const uint32_t word = g * 16u + (u & 3u) * 4u + lane;
        if (lane < 4u && word < words) a.G[word] = mine;
        if (lane == 0) cl_red_add<SOLO>(cl_map<SOLO>(smem_u32(sh.gcnt + g), 0u), cnt);
    }
    cl_sync<SOLO>();
    if (w.rank == 0 && warp == 0) {
        const uint32_t per = (groups + 31u) / 32u, b0 = lane * per;
        uint32_t s = 0;
        for (uint32_t q = 0; q < per; q++)
            if (b0 + q < groups) s += sh.gcnt[b0 + q];
        uint32_t x = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
            if (lane >= (uint32_t)d) x += y;
        }
        uint32_t run = x - s;
        for (uint32_t q = 0; q < per; q++)
            if (b0 + q < groups) {
                a.D[b0 + q] = run;
                run += sh.gcnt[b0 + q];
            }
        if (lane == 31u) a.D[groups] = x;
    }
}

// The bit string of a static function: a group of 512 vertices is 8 b words.
__device__ void small_pack_u(const SmallArgs &a, const SmallView<false> &w) {
    const uint32_t b = a.bits, gw = 8u * b;
    const uint64_t words = ((uint64_t)a.m * b + 63u) / 64u;
    const uint32_t total = (w.vslots >> kSmGroup) * gw;
    for (uint32_t i = threadIdx.x; i < total; i += blockDim.x) {
        const uint32_t lg = i / gw, q = i - lg * gw;
        const uint64_t word = (uint64_t)((lg << w.lc) | w.rank) * gw + q;
        if (word >= words) continue;
        uint64_t x = 0;
        for (uint32_t v = 64u * q / b; v * b < 64u * q + 64u; v++) {
            const uint64_t u = w.rec[(lg << kSmGroup) + v];
            const int sh = (int)(v * b) - (int)(64u * q);
            x |= sh >= 0 ? u << sh : u >> -sh;
        }
        a.U[word] = x;
    }
}

}  // namespace

// MODE 0: peel of an edge list; 1: MPHF from keys; 2: static function.
template <int R, bool GEN, int MODE, bool SOLO, int EPT>
__global__ void __launch_bounds__(kSmThreads, 1) k_small(const SmallArgs a) {
    extern __shared__ __align__(16) uint32_t small_smem[];
    __shared__ SmallShared sh;
    SmallView<GEN> w;
    w.rank = SOLO ? 0u : cl_rank();
    w.blocks = SOLO ? 1u : gridDim.x;
    w.lc = SOLO ? 0u : 31u - __clz(w.blocks);
    w.e0 = w.rank * a.epc;
    w.ne = w.e0 < a.n ? min(a.epc, a.n - w.e0) : 0u;
    w.vslots = a.vslots;
    w.claim = small_smem;
    w.rec = w.claim + a.epc;
    w.hits = w.rec + a.vslots;
    w.bits = w.hits + (SOLO ? a.epc >> 2 : a.epc >> 5);
    w.list = reinterpret_cast<uint16_t *>(w.bits + (EPT == 16 ? a.epc >> 4 : 0u));
    w.vert = reinterpret_cast<typename SmallView<GEN>::V *>(w.list + (EPT == 16 ? a.epc : 0u));
    w.s_hits = smem_u32(w.hits);
    w.s_bits = smem_u32(w.bits);
    w.s_claim = smem_u32(w.claim);
    w.s_rec = smem_u32(w.rec);
    w.s_vert = smem_u32(w.vert);
    constexpr bool KEYS = MODE != 0;
    SmallPeel pe{0, 0, 0};
    uint32_t addr[EPT < 16 ? EPT : 1][R];
    uint32_t code = 0, attempt = 0;
    for (;; attempt++) {  // the same decision in every thread
        if (attempt) cl_sync<SOLO>();  // the last attempt's counters are read and done with
        code = small_peel<R, GEN, KEYS, SOLO, EPT, false>(a, w, sh, a.seed + attempt, addr, pe);
        if constexpr (EPT == 16) {
            if (code == kDevCapacity) {
                cl_sync<SOLO>();  // the totals just read are cleared by the next attempt
                code = small_peel<R, GEN, KEYS, SOLO, EPT, true>(a, w, sh, a.seed + attempt, addr,
                                                                 pe);
            }
        }
        if (!KEYS || code || pe.peeled == a.n || attempt + 1 >= a.max_tries) break;
    }
    const bool done = code == 0 && (!KEYS || pe.peeled == a.n);
    if (done) {
        if (MODE == 0 && a.claim)
            for (uint32_t i = threadIdx.x; i < w.ne; i += blockDim.x) a.claim[w.e0 + i] = w.claim[i];
        if constexpr (MODE != 0) small_assign<MODE == 2, SOLO, EPT>(a, w, sh, addr, pe.rounds);
        if constexpr (MODE == 1) small_pack_g<SOLO>(a, w, sh);
        if constexpr (MODE == 2) small_pack_u(a, w);
        if (a.order) {
            cl_sync<SOLO>();  // the vertices' space is free
            small_order<SOLO>(a, w, w.rec, sh, pe);
        }
    }
    cl_sync<SOLO>();
    if (w.rank == 0 && threadIdx.x < 32u) {
        uint32_t cross = 0, moves = 0, err = 0;
        if (threadIdx.x < w.blocks) {
            cross = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.cross), threadIdx.x));
            moves = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.moves), threadIdx.x));
            err = cl_load<SOLO>(cl_map<SOLO>(smem_u32(&sh.err), threadIdx.x));
        }
        cross = __reduce_add_sync(0xFFFFFFFFu, cross);
        moves = __reduce_add_sync(0xFFFFFFFFu, moves);
        err = code ? code : __reduce_max_sync(0xFFFFFFFFu, err);
        if (threadIdx.x == 0) {
            hpeel_stats st{};
            st.n_peeled = pe.peeled;
            st.rounds = pe.rounds;
            st.attempts = attempt + 1;
            st.device_err = err;
            st.first_layer = pe.first_layer;
            st.frontier = cross;
            st.hinge_moves = moves;
            if (MODE == 0) {
                st.core_nonempty = pe.peeled < a.n ? 1u : 0u;
                st.async_status = err ? 3u : (a.layer_off && pe.rounds > a.max_layers ? 4u : 1u);
            } else {
                st.async_status = err ? (uint32_t)kAsyncDeviceError
                                      : (done ? (uint32_t)kAsyncPeeled
                                              : (uint32_t)kAsyncRetriesExhausted);
                st.core_nonempty = st.async_status == kAsyncRetriesExhausted ? 1u : 0u;
                st.seed_used = st.async_status == kAsyncPeeled ? a.seed + attempt : 0ull;
            }
            *a.stats = st;
        }
    }
    cl_sync<SOLO>();  // no block leaves while another reads its shared memory
}

namespace {

template <bool SOLO, int EPT>
const void *small_fn_t(int mode, uint32_t r, bool gen) {
    if (mode == 1) return (const void *)k_small<3, false, 1, SOLO, EPT>;
    if (mode == 2) return (const void *)k_small<3, false, 2, SOLO, EPT>;
    if (r == 2)
        return gen ? (const void *)k_small<2, true, 0, SOLO, EPT>
                   : (const void *)k_small<2, false, 0, SOLO, EPT>;
    if (r == 3)
        return gen ? (const void *)k_small<3, true, 0, SOLO, EPT>
                   : (const void *)k_small<3, false, 0, SOLO, EPT>;
    return gen ? (const void *)k_small<4, true, 0, SOLO, EPT>
               : (const void *)k_small<4, false, 0, SOLO, EPT>;
}
const void *small_fn(int mode, uint32_t r, bool gen, bool solo, uint32_t ept) {
    if (!solo) return small_fn_t<false, 16>(mode, r, gen);
    if (ept == 1) return small_fn_t<true, 1>(mode, r, gen);
    return ept == 4 ? small_fn_t<true, 4>(mode, r, gen) : small_fn_t<true, 16>(mode, r, gen);
}

// Edges per thread of the one-block forms (kernel time per peel / MPHF build):
// n = 1009 with one edge per thread 18.6 / 27.8 us, with four 32.9 / 55; n =
// 4000 with four 45 / 82 us, with sixteen 60 / 74 (before claims were counted,
// which takes 1-4 % more).
constexpr uint32_t kSmOnePer = 1024, kSmFourPer = 4096;
// Shape of a launch: blocks (a power of two), edges per thread, edges and
// vertex slots per block, threads, dynamic shared memory.
struct SmallShape {
    uint32_t blocks, ept, epc, vslots, threads;
    size_t smem;
};
SmallShape small_shape(uint32_t n, uint32_t m, uint32_t r, bool gen, uint32_t blocks) {
    SmallShape s{};
    s.blocks = blocks;
    s.epc = ((n + blocks - 1) / blocks + 31u) & ~31u;
    s.ept = blocks > 1 || s.epc > kSmFourPer ? 16u : (s.epc > kSmOnePer ? 4u : 1u);
    const uint32_t groups = (m + 511u) / 512u;
    s.vslots = ((groups + blocks - 1) / blocks) << kSmGroup;
    // a cluster has one more warp for the bookkeeping
    const uint32_t want = ((s.epc / s.ept + 31u) & ~31u) + (blocks > 1 ? 32u : 0u);
    s.threads = want > kSmThreads ? kSmThreads : (want < 128u ? 128u : want);
    size_t graph = 4 * ((size_t)s.epc + s.vslots) + (blocks > 1 ? s.epc / 8 : s.epc);
    if (s.ept == 16) graph += s.epc / 4 + 2 * (size_t)s.epc;
    if (s.ept == 16 || gen) graph += (gen ? 4 : 2) * (size_t)s.epc * r;
    const size_t order = 4 * ((size_t)s.epc + kSmBins * (3 + s.threads / 32u));
    s.smem = graph > order ? graph : order;
    return s;
}
bool shape_ok(const SmallShape &s) {
    return s.smem <= kSmMaxSmem && s.epc <= s.ept * (s.threads - (s.blocks > 1 ? 32u : 0u));
}

}  // namespace

bool small_plan(int mode, uint64_t n, uint64_t m, uint32_t r, bool gen, SmallArgs *a,
                SmallLaunch *out) {
    const uint64_t P = gen ? m : m / r;
    if (n == 0 || n > kSmMaxEdges || m == 0 || m > (1ull << 24) || (!gen && P > 65536)) return false;
    static_assert(kSmMaxGroups * 512u >= 3u * 65536u, "group counts of the largest MPHF");
    // one block when the graph fits it (n = 12,000: 92 us per peel), else the
    // largest cluster (n = 16,000: 107 us; of 8 blocks 122)
    SmallShape s = small_shape((uint32_t)n, (uint32_t)m, r, gen, 1);
    const void *fn = small_fn(mode, r, gen, true, s.ept);
    if (shape_ok(s)) {
        smem_optin(fn);
    } else {
        fn = small_fn(mode, r, gen, false, 16);
        const uint32_t most = max_cluster(fn, kSmThreads, kSmMaxSmem);
        if (most < 2) return false;
        s = small_shape((uint32_t)n, (uint32_t)m, r, gen, most);
        if (!shape_ok(s)) return false;
    }
    a->n = (uint32_t)n;
    a->m = (uint32_t)m;
    a->P = (uint32_t)P;
    a->epc = s.epc;
    a->epc_magic = (uint32_t)((1ull << 32) / s.epc) + 1u;
    a->vslots = s.vslots;
    out->fn = fn;
    out->blocks = s.blocks;
    out->threads = s.threads;
    out->smem = s.smem;
    return true;
}

void launch_small(const Launch &L, const SmallLaunch &k, const SmallArgs &a) {
    void *args[] = {(void *)&a};
    count_launch();
    launch_cluster(k.fn, k.blocks, k.threads, k.smem, L.stream, args);
}

}  // namespace hp
