// mphf.cu -- MWHC assignment and rank directory (r = 3).
//
// sec. 3: find u with u[h_0(x)] + u[h_1(x)] + u[h_2(x)] = f(x) (mod 3), where
// f(x) = i for the hinge h_i(x) of x's edge; then h_{f(x)} is a perfect hash
// and a rank over the non-zero u makes it minimal.  sec. 4.3 ("Avoiding
// backward scans"): layers are solved from the last to the first, and the
// order inside a layer is free.  Inside one layer no edge reads a 2-bit
// value another edge of the layer writes (a hinge has degree 1 in its round,
// so it belongs to no other edge alive then), so one launch per layer solves
// the whole layer in parallel; edges that share a 64-bit word of G combine
// their bits with atomicOr.
// sec. 5: the rank counts non-zero 2-bit pairs of a word with a broadword
// expression instead of a bit loop.
#include "cluster.cuh"
#include "kernels.cuh"

namespace hp {

// ------------------------------------------------------ static functions --
// sec. 3: any f: S -> [sigma] is stored as u with f(x) = u[h0] + u[h1] +
// u[h2] mod sigma, b = ceil(log2 sigma) bits per vertex in one bit string
// (vertex v at bits [v b, (v + 1) b), bit i in word i / 64): a value may
// straddle two words, so it is read from one or two words and set with one
// or two atomicOr.  The MPHF is the case sigma = 3, f = hinge.
__device__ __forceinline__ uint64_t u_get(const uint64_t *U, uint32_t v, uint32_t b) {
    const uint64_t bit = (uint64_t)v * b;
    const uint64_t w = bit >> 6;
    const uint32_t sh = (uint32_t)(bit & 63u);
    uint64_t x = __ldcg(U + w) >> sh;
    if (sh + b > 64) x |= __ldcg(U + w + 1) << (64 - sh);
    return x & ((1ull << b) - 1ull);  // b <= 32
}

__device__ __forceinline__ void u_or(uint64_t *U, uint32_t v, uint32_t b, uint64_t x) {
    const uint64_t bit = (uint64_t)v * b;
    const uint64_t w = bit >> 6;
    const uint32_t sh = (uint32_t)(bit & 63u);
    atomicOr((unsigned long long *)(U + w), (unsigned long long)(x << sh));
    if (sh + b > 64) atomicOr((unsigned long long *)(U + w + 1), (unsigned long long)(x >> (64 - sh)));
}


// ------------------------------------------------------------ assignment --
// One list entry {v_hinge, v_a, v_b, e} (the hinge position is the part of
// v_hinge) in three steps, so that a thread has several in flight and the
// first step, which reads nothing an earlier layer wrote, can run ahead:
// load (entry, and its key's value for a static function), read (values of
// v_a and v_b), solve: MPHF g[v_hinge] = hinge - g[v_a] - g[v_b] mod 3 (0
// stored as 3), static function u[v_hinge] = value - u[v_a] - u[v_b] mod
// sigma (a value >= sigma raises kDevBadValue).
template <bool SF>
struct AssignItem {
    uint4 s;
    uint32_t f;
    uint64_t wa, wb;

    __device__ __forceinline__ void load(const AssignArgs &a, bool ok, uint64_t i) {
        s = ok ? __ldcs(a.Lst + i) : make_uint4(0u, 0u, 0u, 0u);
        if (SF) f = ok ? __ldg(a.values + s.w) : 0u;
    }
    __device__ __forceinline__ void read(const AssignArgs &a, bool ok) {
        if (SF) {
            wa = ok ? u_get(a.G, s.y, a.b) : 0ull;
            wb = ok ? u_get(a.G, s.z, a.b) : 0ull;
        } else {
            wa = ok ? __ldcg(a.G + (s.y >> 5)) : 0ull;
            wb = ok ? __ldcg(a.G + (s.z >> 5)) : 0ull;
        }
    }
    __device__ __forceinline__ void solve(const AssignArgs &a) const {
        if (SF) {
            const uint64_t sigma = a.fs.P;
            if (f >= sigma) {
                raise_err(a.ctl, kDevBadValue);
                return;
            }
            const uint64_t val = fastmod((uint64_t)f + sigma - fastmod(wa + wb, a.fs), a.fs);
            if (val) u_or(a.G, s.x, a.b, val);
        } else {
            const uint32_t h = part_of<3>(s.x, a.P);
            const uint32_t sum = (uint32_t)(wa >> (2u * (s.y & 31u)) & 3u) +
                                 (uint32_t)(wb >> (2u * (s.z & 31u)) & 3u);
            const uint32_t val = (h + 6u - sum) % 3u;  // sum <= 6
            const uint64_t code = val ? val : 3u;
            atomicOr((unsigned long long *)(a.G + (s.x >> 5)),
                     (unsigned long long)(code << (2u * (s.x & 31u))));
        }
    }
};

// Entries [lb, le) by the whole grid.  wait: the first entries are loaded
// before the kernel ahead in the stream (the layer after this one) is waited
// for.
template <bool SF>
__device__ __forceinline__ void assign_range(const AssignArgs &a, uint32_t lb, uint32_t le,
                                             bool wait) {
    constexpr int kU = SF ? 2 : 4;
    const uint64_t stride = (uint64_t)gridDim.x * kThreads * kU;
    for (uint64_t i0 = lb + (uint64_t)blockIdx.x * kThreads * kU + threadIdx.x;; i0 += stride) {
        AssignItem<SF> x[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const uint64_t i = i0 + (uint64_t)u * kThreads;
            x[u].load(a, i < le, i);
        }
        if (wait) asm volatile("griddepcontrol.wait;" ::: "memory");
        wait = false;
        if (i0 >= le) break;
#pragma unroll
        for (int u = 0; u < kU; u++) x[u].read(a, i0 + (uint64_t)u * kThreads < le);
#pragma unroll
        for (int u = 0; u < kU; u++)
            if (i0 + (uint64_t)u * kThreads < le) x[u].solve(a);
    }
}

// One layer, launched from the host, which knows where it lies.  Layers
// follow each other by programmatic dependent launch: the next layer's blocks
// start and load their entries while this one's finish.
// With the runs of small layers below: static function of 1e7 keys (10 bits)
// 880 -> 430 us of assignment, MPHF build of 1e8 keys -0.2 ms.
template <bool SF>
__global__ void __launch_bounds__(kThreads)
k_assign(const AssignArgs a, uint32_t lb, uint32_t le) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    assign_range<SF>(a, lb, le, true);
}

// The layer whose index the device holds (the assignment loop of a
// device-driven build), when it is larger than small.
template <bool SF>
__global__ void __launch_bounds__(kThreads)
k_assign_at(const AssignArgs a, const int32_t *t, uint32_t small) {
    const uint32_t tt = (uint32_t)*(volatile const int32_t *)t;
    const uint32_t lb = __ldcg(a.loff + tt), le = __ldcg(a.loff + tt + 1);
    if (le - lb > small) assign_range<SF>(a, lb, le, false);
}

// Layers thi, thi - 1, .. while they hold at most kAssignTail entries (and
// down to tlo), in one launch of one cluster: a layer waits for the one before
// only in the cluster barrier, and its entries are loaded ahead of it.  A
// launch per layer costs 6-14 us, one after the other, for about 1 us here.
// Device-driven build of 1e6 keys: 1021 -> 667 us.  At 32,768 entries and
// two per thread a layer still takes less than a grid's launch; larger ones
// are better off with all SMs.
// state: the device holds the layer (s->t); a layer that is too large at the
// start has just been solved by k_assign_at and is skipped.
constexpr uint32_t kAssignTail = 32768;  // 16 blocks x 1024 threads x 2 entries
template <bool SF>
__global__ void __launch_bounds__(1024, 1)
k_assign_tail(const AssignArgs a, int32_t thi, int32_t tlo, AsyncState *state,
              cudaGraphConditionalHandle cond) {
    constexpr int kU = 2;
    const uint32_t lanes = gridDim.x * 1024u, g = cl_rank() * 1024u + threadIdx.x;
    int32_t t = state ? (int32_t)__ldcg(reinterpret_cast<const uint32_t *>(&state->t)) : thi;
    uint32_t le = __ldcg(a.loff + t + 1), lb = __ldcg(a.loff + t);
    cl_sync<false>();  // every block has read the state
    if (state && le - lb > kAssignTail) {
        t--;
        le = lb;
        if (t >= tlo) lb = __ldcg(a.loff + t);
    }
    AssignItem<SF> x[kU];
    auto load = [&](uint32_t b, uint32_t e) {
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const uint32_t i = b + (uint32_t)u * lanes + g;
            x[u].load(a, i < e, i);
        }
    };
    if (t >= tlo && le - lb <= kAssignTail) load(lb, le);
    while (t >= tlo && le - lb <= kAssignTail) {
        bool ok[kU];
        AssignItem<SF> now[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
            ok[u] = lb + (uint32_t)u * lanes + g < le;
            now[u] = x[u];
        }
#pragma unroll
        for (int u = 0; u < kU; u++) now[u].read(a, ok[u]);
        // the next layer's entries come while this one is solved
        t--;
        le = lb;
        if (t >= tlo) {
            lb = __ldcg(a.loff + t);
            if (le - lb <= kAssignTail) load(lb, le);
        }
#pragma unroll
        for (int u = 0; u < kU; u++)
            if (ok[u]) now[u].solve(a);
        cl_sync<false>();
    }
    if (state && g == 0) {
        state->t = t;
        cudaGraphSetConditional(cond, t >= 0 ? 1u : 0u);
    }
}

uint32_t assign_tail_blocks(bool sf) {
    const void *fn = sf ? (const void *)k_assign_tail<true> : (const void *)k_assign_tail<false>;
    const uint32_t b = max_cluster(fn, 1024, 0);
    return b == 16 ? b : 0;  // kAssignTail entries need all sixteen
}

// Reverse layer order (sec. 4.3 "Avoiding backward scans") with the layer
// starts in host memory: runs of small layers in one cluster launch, the
// others by one grid each.
void launch_assign(const Launch &L, bool sf, const AssignArgs &a, const uint32_t *loff_h,
                   uint32_t rounds) {
    const uint32_t tail = assign_tail_blocks(sf);
    for (int64_t t = (int64_t)rounds - 1; t >= 0;) {
        int64_t lo = t;  // layers lo + 1 .. t are small
        while (tail && lo >= 0 && loff_h[lo + 1] - loff_h[lo] <= kAssignTail) lo--;
        if (t - lo >= 2) {
            int32_t thi = (int32_t)t, tlo = (int32_t)lo + 1;
            AsyncState *none = nullptr;
            cudaGraphConditionalHandle c0 = 0;
            void *args[] = {(void *)&a, &thi, &tlo, &none, &c0};
            count_launch();
            launch_cluster(sf ? (const void *)k_assign_tail<true> : (const void *)k_assign_tail<false>,
                           tail, 1024, 0, L.stream, args);
            t = lo;
            continue;
        }
        uint32_t lb = loff_h[t], le = loff_h[t + 1];
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid_for(L, le - lb, sf ? 2 : 4, 8));
        cfg.blockDim = dim3(kThreads);
        cfg.stream = L.stream;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        void *args[] = {(void *)&a, &lb, &le};
        count_launch();
        cudaLaunchKernelExC(&cfg, sf ? (const void *)k_assign<true> : (const void *)k_assign<false>,
                            args);
        t--;
    }
}

// Body of the device-driven assignment loop: the layer s->t when it is large,
// then the run of small layers after it (every layer by the grid, one per
// turn, where the device runs no cluster of sixteen).
void launch_assign_body(const Launch &L, bool sf, const AssignArgs &a, AsyncState *s,
                        cudaGraphConditionalHandle h) {
    const uint32_t tail = assign_tail_blocks(sf);
    const uint32_t small = tail ? kAssignTail : 0u;
    count_launch(2);
    if (sf)
        k_assign_at<true><<<grid_fixed(L, 8), kThreads, 0, L.stream>>>(a, &s->t, small);
    else
        k_assign_at<false><<<grid_fixed(L, 8), kThreads, 0, L.stream>>>(a, &s->t, small);
    if (!tail) {
        launch_async_assign_step(L, s, h);
        return;
    }
    int32_t thi = 0, tlo = 0;
    void *args[] = {(void *)&a, &thi, &tlo, &s, &h};
    launch_cluster(sf ? (const void *)k_assign_tail<true> : (const void *)k_assign_tail<false>, tail,
                   1024, 0, L.stream, args);
}

// Non-zero 2-bit values of a word: a pair is non-zero when either bit is set.
__device__ __forceinline__ uint32_t nonzero_pairs(uint64_t w) {
    return (uint32_t)__popcll((w | (w >> 1)) & 0x5555555555555555ull);
}

// One thread per 512 vertices (16 words of G, 32 vertices per word).
__global__ void k_rank_counts(const uint64_t *__restrict__ G, uint64_t words, uint64_t blocks,
                              uint32_t *__restrict__ cnt) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < blocks; b += stride) {
        uint32_t c = 0;
        const uint64_t w0 = b * 16;
        if (w0 + 16 <= words && ((((uintptr_t)G) & 15u) == 0)) {
            const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(G + w0);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const ulonglong2 x = p[q];
                c += nonzero_pairs(x.x) + nonzero_pairs(x.y);
            }
        } else {
            for (uint64_t w = w0; w < words && w < w0 + 16; w++) c += nonzero_pairs(G[w]);
        }
        cnt[b] = c;
    }
}

void launch_rank_counts(const Launch &L, const uint64_t *G, uint64_t m, uint32_t *cnt) {
    const uint64_t words = (m + 31) / 32, blocks = (m + 511) / 512;
    if (blocks == 0) return;
    count_launch();
    k_rank_counts<<<grid_for(L, blocks, 1, 8), kThreads, 0, L.stream>>>(G, words, blocks, cnt);
}

__global__ void k_widen_dir(const uint32_t *__restrict__ scanned, const uint32_t *__restrict__ cnt,
                            uint64_t blocks, uint64_t *__restrict__ dir) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= blocks; b += stride) {
        if (b < blocks)
            dir[b] = scanned[b];
        else
            dir[b] = blocks ? (uint64_t)scanned[blocks - 1] + cnt[blocks - 1] : 0ull;
    }
}

void launch_widen_dir(const Launch &L, const uint32_t *scanned, const uint32_t *cnt,
                      uint64_t blocks, uint64_t *dir) {
    count_launch();
    k_widen_dir<<<grid_for(L, blocks + 1, 1, 8), kThreads, 0, L.stream>>>(scanned, cnt, blocks,
                                                                          dir);
}

// f(key) = (u[h0] + u[h1] + u[h2]) mod sigma.
__global__ void __launch_bounds__(kThreads)
k_sf_lookup(const uint64_t *__restrict__ keys, uint64_t nq, FastMod fm, uint64_t seed,
            FastMod fs, uint32_t b, const uint64_t *__restrict__ U, uint32_t *__restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * kThreads;
    const uint32_t P = (uint32_t)fm.P;
    for (uint64_t q = (uint64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += stride) {
        const uint64_t k = __ldcs(keys + q);
        uint64_t s = 0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const uint32_t v =
                (uint32_t)fastmod(mix64(k ^ (seed + (uint64_t)j)), fm) + (uint32_t)j * P;
            s += u_get(U, v, b);
        }
        out[q] = (uint32_t)fastmod(s, fs);
    }
}

void launch_sf_lookup(const Launch &L, const uint64_t *keys, uint64_t nq, FastMod fm,
                      uint64_t seed, uint64_t sigma, uint32_t b, const uint64_t *U,
                      uint32_t *out) {
    if (nq == 0) return;
    count_launch();
    k_sf_lookup<<<grid_for(L, nq, 1, 8), kThreads, 0, L.stream>>>(keys, nq, fm, seed,
                                                                  make_fastmod(sigma), b, U, out);
}

// ---------------------------------------------------------------- lookup --
// MPHF value of a key (sec. 3 and sec. 5): hash to h_0..h_2, i = (g[h_0] +
// g[h_1] + g[h_2]) mod 3 (a stored 3 counts as 0), v = h_i, and the value is
// the rank of v among the assigned vertices: the directory entry of v's
// 512-vertex block plus the non-zero pairs before v inside the block,
// counted a word at a time with the broadword expression.
__device__ __forceinline__ uint32_t lookup_vertex(const uint32_t (&v)[3], uint32_t g) {
    const uint32_t i = g % 3u;
    return i == 0 ? v[0] : (i == 1 ? v[1] : v[2]);
}
__device__ __forceinline__ uint32_t lookup_words(const uint64_t *__restrict__ G,
                                                 const uint64_t *__restrict__ dir,
                                                 const uint32_t (&v)[3]) {
    uint32_t g = 0;
#pragma unroll
    for (int j = 0; j < 3; j++) g += (uint32_t)(__ldg(G + (v[j] >> 5)) >> (2u * (v[j] & 31u))) & 3u;
    const uint32_t x = lookup_vertex(v, g);
    const uint32_t blk = x >> 9, w_end = x >> 5;
    uint64_t rank = __ldg(dir + blk);
    for (uint32_t w = blk << 4; w < w_end; w++) rank += nonzero_pairs(__ldg(G + w));
    const uint32_t sh = 2u * (x & 31u);
    if (sh) rank += nonzero_pairs(__ldg(G + w_end) & ((1ull << sh) - 1ull));
    return (uint32_t)rank;
}

// Four consecutive words (128 vertices), 32-byte aligned: one load.
struct Words4 {
    uint64_t w[4];
};
__device__ __forceinline__ Words4 load_words4(const uint64_t *p) {
    Words4 x;
    asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
        : "=l"(x.w[0]), "=l"(x.w[1]), "=l"(x.w[2]), "=l"(x.w[3])
        : "l"(p));
    return x;
}
// Non-zero pairs among pairs [0, k) of the 128 (up), or [k, 128) (not up).
// Two words' flags share one population count.
__device__ __forceinline__ uint64_t pair_flags(uint64_t w) {
    return (w | (w >> 1)) & 0x5555555555555555ull;
}
__device__ __forceinline__ uint32_t pairs_side(const Words4 &x, uint32_t k, bool up) {
    uint64_t f[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const int left = (int)k - 32 * q;  // pairs of word q before k
        const uint64_t mask =
            left <= 0 ? 0ull : (left >= 32 ? ~0ull : (1ull << (2 * left)) - 1ull);
        f[q] = pair_flags(x.w[q]) & (up ? mask : ~mask);
    }
    return (uint32_t)(__popcll(f[0] | (f[1] << 1)) + __popcll(f[2] | (f[3] << 1)));
}
__device__ __forceinline__ uint32_t pairs_all(const Words4 &x) {
    return (uint32_t)(__popcll(pair_flags(x.w[0]) | (pair_flags(x.w[1]) << 1)) +
                      __popcll(pair_flags(x.w[2]) | (pair_flags(x.w[3]) << 1)));
}

// The L1 serves about one lane's request per cycle, so a query is bound by
// its loads, not their width, and by the arithmetic of three hashes: three
// 32-byte sectors of G (the words that hold the three values), one directory
// entry, and half the time one more sector.  The rank is counted from the
// nearer end of the 512-vertex block: up from dir[block] in its lower half,
// down from dir[block + 1] in its upper one, and the vertex's own sector is
// already in registers.  A word at a time from the block's start a query took
// 12 loads: 1e8 queries of a 1e8-key function 2.97 -> 1.64 ms (8-byte loads of
// the three values and the chosen sector again: 1.90 ms; two queries per
// thread: 2.4 against 2.2 ms before the arithmetic was cut).
__global__ void __launch_bounds__(kThreads, 6)
k_lookup(const uint64_t *__restrict__ keys, uint64_t nq, FastMod fm, uint64_t seed,
         const uint64_t *__restrict__ G, uint32_t words, const uint64_t *__restrict__ dir,
         uint32_t *__restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * kThreads;
    const uint32_t P = (uint32_t)fm.P;
    for (uint64_t q = (uint64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += stride) {
        const uint64_t k = __ldcs(keys + q);
        uint32_t v[3];
        bool whole = true;  // none of the sectors reaches past the last word
#pragma unroll
        for (int j = 0; j < 3; j++) {
            v[j] = (uint32_t)fastmod(mix64(k ^ (seed + (uint64_t)j)), fm) + (uint32_t)j * P;
            whole &= ((v[j] >> 5) | 3u) < words;
        }
        const uint32_t last = ((v[2] >> 9) << 4) + 16u;  // the outer sector of the last block
        if (!whole || last > words) {
            out[q] = lookup_words(G, dir, v);
            continue;
        }
        Words4 s[3];
#pragma unroll
        for (int j = 0; j < 3; j++) s[j] = load_words4(G + ((v[j] >> 7) << 2));
        uint32_t g = 0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const uint32_t w = (v[j] >> 5) & 3u;
            const uint64_t word = w < 2 ? (w == 0 ? s[j].w[0] : s[j].w[1])
                                        : (w == 2 ? s[j].w[2] : s[j].w[3]);
            g += (uint32_t)(word >> (2u * (v[j] & 31u))) & 3u;
        }
        const uint32_t x = lookup_vertex(v, g);
        const Words4 own = x == v[0] ? s[0] : (x == v[1] ? s[1] : s[2]);
        // sector 0 or 1 of the block: up from dir[block]; 2 or 3: down from
        // the next entry; 1 and 2 need the outer sector as well
        const uint32_t sec = (x >> 7) & 3u;
        const bool up = sec < 2u;
        uint32_t rank = (uint32_t)__ldg(dir + (x >> 9) + (up ? 0u : 1u));
        uint32_t c = 0;
        if (sec == 1u || sec == 2u) c = pairs_all(load_words4(G + ((x >> 9) << 4) + (up ? 0u : 12u)));
        c += pairs_side(own, x & 127u, up);
        out[q] = up ? rank + c : rank - c;
    }
}

// The same a word at a time, for a G that is not 32-byte aligned.
__global__ void __launch_bounds__(kThreads)
k_lookup_words(const uint64_t *__restrict__ keys, uint64_t nq, FastMod fm, uint64_t seed,
               const uint64_t *__restrict__ G, const uint64_t *__restrict__ dir,
               uint32_t *__restrict__ out) {
    const uint64_t stride = (uint64_t)gridDim.x * kThreads;
    for (uint64_t q = (uint64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += stride) {
        const uint64_t k = __ldcs(keys + q);
        uint32_t v[3];
#pragma unroll
        for (int j = 0; j < 3; j++)
            v[j] = (uint32_t)fastmod(mix64(k ^ (seed + (uint64_t)j)), fm) + (uint32_t)j * (uint32_t)fm.P;
        out[q] = lookup_words(G, dir, v);
    }
}

void launch_lookup(const Launch &L, const uint64_t *keys, uint64_t nq, FastMod fm, uint64_t seed,
                   const uint64_t *G, const uint64_t *dir, uint32_t *out) {
    if (nq == 0) return;
    count_launch();
    if (((uintptr_t)G & 31u) == 0)
        k_lookup<<<grid_for(L, nq, 1, 16), kThreads, 0, L.stream>>>(
            keys, nq, fm, seed, G, (uint32_t)((3 * fm.P + 31) / 32), dir, out);
    else
        k_lookup_words<<<grid_for(L, nq, 1, 8), kThreads, 0, L.stream>>>(keys, nq, fm, seed, G, dir,
                                                                         out);
}

}  // namespace hp
