// Shortest paths to a few targets at a time, by relaxation over edge lists
// sorted by weight (relax.cu describes the method; the batched launch uses the
// same pieces).
//
// Lists.  Row v's list holds its edges (v, k), lightest first, 4 to a 16-byte
// chunk, each edge as (w << 16) | k with w saturated at 0x7FFF, and the same
// edges' full weights in a second array.  Chunk c of rows 32 r .. 32 r + 31 is
// contiguous, so a warp that reads chunk c of 32 rows reads 512 bytes.  A list
// shorter than the capacity ends with chunks of pads (w = 0x7FFF, INF).  A row
// with more edges than the capacity keeps its lightest ones; next[v] is then a
// lower bound of the weights left out (INF: none).
#pragma once

#include <type_traits>

#include "common.cuh"

namespace btas {
namespace relax {

constexpr int kCap = 512;          // most edges a list holds
__host__ __device__ constexpr int list_chunks(long long n) { return (int)((n < kCap ? n : kCap) + 3) / 4; }
__host__ __device__ constexpr size_t list_words(long long n) {  // of Lists::edges, and of Lists::wide
    return (size_t)((n + 31) / 32) * 32 * list_chunks(n) * 4;
}
constexpr int kTruncTarget = 256;  // a longer row keeps at most about this many
constexpr int kPadChunks = 2;      // chunks of pads after a list: one per lane that reads it (solve's G)
constexpr int kEarlySweeps = 2, kEarlyChunks = 2;  // solve's first sweeps
constexpr int kSample = 1024;      // entries the first guess of a long row's cutoff is taken from

// When a block gives its solve up.  Random graphs, of any density and any
// weights, are solved in 10 to 23 sweeps (n = 49 ... 8192).  Shortest paths of
// many edges take more, and there are two kinds of graphs with such paths.
// - Distances are still missing after 8 sweeps (chains, rings, grids, lattices,
//   and the sparsest random graphs).  They are found at an even pace or a growing
//   one until all are, so the share found, or what the last 8 sweeps added to it,
//   says how long that still takes.  From kSettle sweeps on the solve goes on while
//   that is less than what solving otherwise is worth, up to twice its worth; up to
//   `cycles` in 16 bits that do not hold all weights, where a longer edge counts as
//   missing.
// - All are known by then and some still improve: nothing tells for how long,
//   and `cycles` end it.
struct Patience {
    bool by_share;     // false: `cycles` alone counts (tests)
    long long cycles;  // about twice what the slowest random graphs take
    long long worth16, worth32;  // a block's share of what solving otherwise takes, where 16 bits do and where not
};
constexpr int kSettle = 24;

struct Lists {
    uint4 *edges;  // [ceil(n / 32)][chunks][32]
    int4 *wide;    // the weights in 32 bits, same places
    int *next;     // n words
    int *len;      // optional: edges in each list
    int chunks;    // capacity / 4
    Patience patience;
    // > 0: only lists of whole rows are of use, of at most `whole` edges, none
    // heavier than `top`; other rows are counted and no more
    int whole, top;
};

// What building the lists of some rows finds out.
struct RowStats {
    int bad;    // entries outside the domain
    int maxw;   // largest weight
    int minw;   // smallest off-diagonal weight (INF: no edge)
    int deg;    // most edges of a row
    int far;    // 1: some row's lightest edge does not fit 16 bits
    float light;  // sum of the rows' lightest weights
    int cut;      // 1: some list holds less than its row
    int edges;    // of all rows
};

// Clock cycles a block of 8 targets is worth: about twice what the slowest
// random graphs take (n = 256 ... 8192, edge probability 0.01 ... 1).
__host__ __device__ constexpr long long budget_cycles(long long n) {
    return 30000 + 200 * n + (n / 8 < 300 ? n / 8 : 300) * n;
}

// Whether 16 bits are likely to be too few: the largest distance of a random
// graph is about 3 ln n times the mean of its rows' lightest weights.
__device__ __forceinline__ bool expects_wide(int n, float light) {
    return 3.0f * __logf((float)n) * light >= (float)n * BTAS_INF_U16;
}

__device__ __forceinline__ size_t chunk_at(const Lists &l, int row, int c) {
    return ((size_t)(row >> 5) * l.chunks + c) * 32 + (row & 31);
}

// --------------------------------------------------------------- sorting
template <class Key>
__device__ __forceinline__ void order(Key &a, Key &b, bool up) {
    const Key lo = min(a, b), hi = max(a, b);
    a = up ? lo : hi;
    b = up ? hi : lo;
}

// The stages of a bitonic merge inside one lane's E consecutive elements.
template <class Key, int E>
__device__ __forceinline__ void merge_lane(Key (&key)[E], int first, bool up) {
#pragma unroll
    for (int j = E / 2; j > 0; j >>= 1)
        if (j <= first) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((e & j) == 0) order(key[e], key[e | j], up);
        }
}

// Ascending bitonic sort of 32 E keys, element lane * E + e in key[e]: the
// short exchanges stay in registers, the others are one shuffle per key.
template <class Key, int E>
__device__ __forceinline__ void sort_warp(Key (&key)[E], int lane) {
#pragma unroll
    for (int k = 2; k < E; k <<= 1)  // runs of k inside the lane, alternating directions
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((e & j) == 0) order(key[e], key[e | j], (e & k) == 0);
    for (int k = E; k <= 32 * E; k <<= 1) {
        const bool up = ((lane * E) & k) == 0;
        for (int j = k >> 1; j >= E; j >>= 1) {
            const int d = j / E;
            const bool low = ((lane & d) == 0) == up;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const Key o = __shfl_xor_sync(0xffffffffu, key[e], d);
                key[e] = low ? min(key[e], o) : max(key[e], o);
            }
        }
        merge_lane<Key, E>(key, k >> 1, up);
    }
}

// cnt <= 32 E keys (w << 32 | k) in `buf` -> the row's chunks, lightest first.
// Key32: (w - base) << 16 | k, where the weights span less than 2^16 - 1.
template <bool Key32, int E>
__device__ __forceinline__ void sort_and_store(const unsigned long long *buf, int cnt, int row, int base,
                                               const Lists &l, int lane) {
    using Key = typename std::conditional<Key32, unsigned, unsigned long long>::type;
    Key key[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = lane * E + e;
        if (Key32) {
            const unsigned long long b = i < cnt ? buf[i] : 0;
            key[e] = i < cnt ? (Key)((((unsigned)(b >> 32) - (unsigned)base) << 16) | (unsigned)b) : ~(Key)0;
        } else {
            key[e] = i < cnt ? (Key)buf[i] : ~(Key)0;
        }
    }
    sort_warp<Key, E>(key, lane);
    // the list's chunks and its pads; a full list has none
    const int chunks = min(l.chunks, (cnt + 3) / 4 + kPadChunks);
#pragma unroll
    for (int q = 0; q < E / 4; ++q) {
        const int c = lane * (E / 4) + q;
        if (c >= chunks) continue;
        unsigned p[4];
        int w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const Key kk = key[4 * q + e];
            const bool edge = 4 * c + e < cnt;
            w[e] = !edge ? kInfI32 : Key32 ? (int)((unsigned)kk >> 16) + base : (int)((unsigned long long)kk >> 32);
            p[e] = ((unsigned)min(w[e], BTAS_INF_U16) << 16) | (edge ? (unsigned)kk & 0xFFFFu : (unsigned)row);
        }
        l.edges[chunk_at(l, row, c)] = make_uint4(p[0], p[1], p[2], p[3]);
        l.wide[chunk_at(l, row, c)] = make_int4(w[0], w[1], w[2], w[3]);
    }
    // pads beyond the sorted block (cnt close to 32 E)
    const int c = 8 * E + lane;
    if (c < chunks) {
        const unsigned p = ((unsigned)BTAS_INF_U16 << 16) | (unsigned)row;
        l.edges[chunk_at(l, row, c)] = make_uint4(p, p, p, p);
        l.wide[chunk_at(l, row, c)] = make_int4(kInfI32, kInfI32, kInfI32, kInfI32);
    }
}

// A weight such that about `target` of the edges among the row's first m
// entries are lighter (at most `target`; at least half of it unless weights
// repeat too often: then ties is set and edges at the cutoff weight itself
// may fill up the list).  `below`: how many are lighter.  Histograms of 256 equal
// bins of [lo, hi], refined around the bin that does not fit.  `hist`: 256
// words of the warp's own.
__device__ __forceinline__ int select_cut(const int *wr, int row, int m, int target, int lo, int hi, int *hist,
                                          int lane, bool &ties, int &below) {
    below = 0;  // edges lighter than lo
    ties = false;
    for (;;) {
        const int sh = max(0, 24 - __clz(max(hi - lo, 1)));  // (hi - lo) >> sh <= 255
        for (int b = lane; b < 256; b += 32) hist[b] = 0;
        __syncwarp();
        for (int j0 = 0; j0 < m; j0 += 128) {
            int v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + 32 * u + lane;
                v[u] = j < m && j != row ? __ldg(wr + j) : kInfI32;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (v[u] >= lo && v[u] <= hi) atomicAdd(hist + ((v[u] - lo) >> sh), 1);
        }
        __syncwarp();
        int h[8], tot = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            h[b] = hist[lane * 8 + b];
            tot += h[b];
        }
        int pre = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o) pre += x;
        }
        pre -= tot;  // edges in the bins of the lanes before this one
        int fit = 0, kept = 0;  // bins, from the first, that fit together
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            pre += h[b];
            if (below + pre <= target) {
                ++fit;
                kept = pre;
            }
        }
        fit = __reduce_add_sync(0xffffffffu, fit);
        kept = __reduce_max_sync(0xffffffffu, kept);
        __syncwarp();
        below += kept;
        if (fit == 256) return hi + 1;
        const int cut = lo + (fit << sh);
        if (2 * below >= target) return cut;
        if (sh == 0) {
            ties = true;
            return cut;
        }
        lo = cut;
        hi = min(hi, cut + (1 << sh) - 1);
    }
}

// One pass over row `row` of W by one warp: the domain check, the statistics,
// and the edges lighter than `cut`, with the first `room` of those as light as
// it, to buf, kCap of them at most.  Returns how many there are; deg: all of
// the row's edges.
__device__ __forceinline__ int scan_row(const int *wr, int n, int row, int cut, int room, unsigned long long *buf,
                                        int lane, RowStats &st, int &mn, int &mx, int &deg) {
    constexpr int U = 8;
    const unsigned lt = (1u << lane) - 1u;
    int cnt = 0, tied = 0;
    deg = 0;
    mn = kInfI32;
    mx = 0;
    int bad = 0;
    for (int c0 = 0; c0 < n; c0 += 32 * U) {
        int v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = c0 + 32 * u + lane;
            v[u] = j < n ? __ldg(wr + j) : kInfI32;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = c0 + 32 * u + lane;
            const bool fin = (unsigned)v[u] <= (unsigned)BTAS_I32_FINITE_MAX;
            bad += (!fin && v[u] != kInfI32) || (j == row && v[u] != 0);
            const bool edge = fin && j != row;
            deg += edge;
            mx = max(mx, edge ? v[u] : 0);
            mn = min(mn, edge ? v[u] : kInfI32);
            bool keep = edge && v[u] < cut;
            if (room > 0) {
                const bool tie = edge && v[u] == cut;
                const unsigned m = __ballot_sync(0xffffffffu, tie);
                keep = keep || (tie && tied + __popc(m & lt) < room);
                tied += __popc(m);
            }
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            const int q = cnt + __popc(m & lt);
            if (keep && q < kCap) buf[q] = ((unsigned long long)(unsigned)v[u] << 32) | (unsigned)j;
            cnt += __popc(m);
        }
    }
    st.bad = __reduce_add_sync(0xffffffffu, bad);
    deg = __reduce_add_sync(0xffffffffu, deg);
    mx = __reduce_max_sync(0xffffffffu, mx);
    mn = __reduce_min_sync(0xffffffffu, mn);
    __syncwarp();
    return cnt;
}

// Row `row`'s list, by one warp.  buf: kCap keys, hist: 256 words, both the
// warp's own shared memory.
__device__ __forceinline__ RowStats build_row(const int *W, long long ldw, int n, int row, const Lists &l,
                                              unsigned long long *buf, int *hist, int lane) {
    const int *wr = W + (long long)row * ldw;
    const int cap = min(kCap, 4 * l.chunks);
    RowStats st{};
    int cut = kInfI32;
    bool ties = false;
    int below;
    // A long row is read once: its first entries say whether it will overflow
    // and, if so, about where to cut.
    if (n >= 2 * kSample && l.whole == 0) {
        int d = 0, mn = kInfI32, mx = 0;
#pragma unroll 8
        for (int j = lane; j < kSample; j += 32) {
            const int v = __ldg(wr + j);
            if ((unsigned)v <= (unsigned)BTAS_I32_FINITE_MAX && j != row) {
                ++d;
                mn = min(mn, v);
                mx = max(mx, v);
            }
        }
        d = __reduce_add_sync(0xffffffffu, d);
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((long long)d * n > (long long)cap * kSample * 9 / 10)
            cut = select_cut(wr, row, kSample, max(4, (int)((long long)kTruncTarget * kSample / n)), mn, mx, hist,
                             lane, ties, below);
        if (ties) cut = kInfI32;
    }
    int mn, mx, deg;
    int cnt = scan_row(wr, n, row, cut, 0, buf, lane, st, mn, mx, deg);
    if (l.whole > 0 && (deg > l.whole || mx > l.top)) {
        st.maxw = mx;
        st.minw = mn;
        st.deg = deg;
        st.cut = 1;
        st.edges = deg;
        return st;
    }
    if (cnt > cap || (cnt < deg && cnt < 64)) {
        // every lighter edge (at most kTruncTarget) and as many at the cutoff as fit
        cut = select_cut(wr, row, n, kTruncTarget, mn, mx, hist, lane, ties, below);
        cnt = scan_row(wr, n, row, cut, ties ? cap - below : 0, buf, lane, st, mn, mx, deg);
    }
    if (lane == 0) {
        l.next[row] = cnt < deg ? cut : kInfI32;
        if (l.len != nullptr) l.len[row] = cnt;
    }
    const bool k32 = (cnt < deg ? cut : mx) - mn < 0xFFFF;
    if (cnt <= 128) {
        if (k32) sort_and_store<true, 4>(buf, cnt, row, mn, l, lane);
        else sort_and_store<false, 4>(buf, cnt, row, mn, l, lane);
    } else {
        if (k32) sort_and_store<true, 16>(buf, cnt, row, mn, l, lane);
        else sort_and_store<false, 16>(buf, cnt, row, mn, l, lane);
    }
    st.maxw = mx;
    st.minw = mn;
    st.deg = deg;
    st.far = deg > 0 && mn >= BTAS_INF_U16;
    st.light = deg > 0 ? (float)mn : 0.0f;
    st.cut = cnt < deg;
    st.edges = deg;
    return st;
}

// -------------------------------------------------------------- relaxing
// Y in shared memory: a row of R vectors of NV words per vertex v, the distances
// from v to 2 NV R targets in 16 bits (0x7FFF: none known) or to NV R in 32.  Each
// vector has its own lane.  Only v's own lanes write its row, and a stale read
// costs a further sweep and no more, so the accesses of a sweep are relaxed ones.
template <int NV>
struct __align__(4 * NV) Vec {
    unsigned w[NV];
};

template <int NV>
__device__ __forceinline__ Vec<NV> lds_relaxed(const Vec<NV> *p) {
    Vec<NV> v;
    if constexpr (NV == 4)
        asm volatile("ld.relaxed.cta.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3])
                     : "r"(smem_u32(p))
                     : "memory");
    else if constexpr (NV == 2)
        asm volatile("ld.relaxed.cta.shared.v2.b32 {%0, %1}, [%2];"
                     : "=r"(v.w[0]), "=r"(v.w[1])
                     : "r"(smem_u32(p))
                     : "memory");
    else
        asm volatile("ld.relaxed.cta.shared.b32 %0, [%1];" : "=r"(v.w[0]) : "r"(smem_u32(p)) : "memory");
    return v;
}
template <int NV>
__device__ __forceinline__ void sts_relaxed(Vec<NV> *p, const Vec<NV> &v) {
    if constexpr (NV == 4)
        asm volatile("st.relaxed.cta.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(smem_u32(p)), "r"(v.w[0]),
                     "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3])
                     : "memory");
    else if constexpr (NV == 2)
        asm volatile("st.relaxed.cta.shared.v2.b32 [%0], {%1, %2};" ::"r"(smem_u32(p)), "r"(v.w[0]), "r"(v.w[1])
                     : "memory");
    else
        asm volatile("st.relaxed.cta.shared.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v.w[0]) : "memory");
}
template <bool U16, int NV>
__device__ __forceinline__ int top(const Vec<NV> &y) {
    unsigned m = y.w[0];
    if (U16) {
#pragma unroll
        for (int q = 1; q < NV; ++q) m = __vmaxu2(m, y.w[q]);
        return (int)max(m >> 16, m & 0xFFFFu);
    }
#pragma unroll
    for (int q = 1; q < NV; ++q) m = (unsigned)max((int)m, (int)y.w[q]);
    return (int)m;
}
// acc = min(acc, y + w); w: the weight in both halves with U16
template <bool U16, int NV>
__device__ __forceinline__ void relax_edge(Vec<NV> &acc, const Vec<NV> &y, unsigned w) {
#pragma unroll
    for (int q = 0; q < NV; ++q)
        acc.w[q] = U16 ? u16x2_addmin(y.w[q], w, acc.w[q])
                       : (unsigned)__viaddmin_s32((int)y.w[q], (int)w, (int)acc.w[q]);
}
// acc = min(acc, the same vector of lane ^ o)
template <bool U16, int NV>
__device__ __forceinline__ void min_with_lane(Vec<NV> &acc, int o) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const unsigned b = __shfl_xor_sync(0xffffffffu, acc.w[q], o);
        acc.w[q] = U16 ? __vminu2(acc.w[q], b) : (unsigned)min((int)acc.w[q], (int)b);
    }
}
template <int NV>
__device__ __forceinline__ void clamp(Vec<NV> &v) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v.w[q] = (unsigned)clamp_i32<kMin>((int)v.w[q]);
}
template <int NV>
__device__ __forceinline__ bool differ(const Vec<NV> &a, const Vec<NV> &b) {
    unsigned d = 0;
#pragma unroll
    for (int q = 0; q < NV; ++q) d |= a.w[q] ^ b.w[q];
    return d != 0;
}

template <bool U16, int R, int NV>
constexpr int targets() { return (U16 ? 2 : 1) * NV * R; }

// Columns [j0, j0 + targets) of W -> Y: the paths of one edge.
template <bool U16, int R, int NV>
__device__ __forceinline__ void load_columns(const int *W, long long ldw, int n, Vec<NV> *Y, int j0) {
    constexpr int S = targets<U16, 1, NV>();
    const bool vec = S % 4 == 0 && (ldw & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
    for (int i = threadIdx.x; i < n * R; i += blockDim.x) {
        const int j = j0 + (i % R) * S;
        int x[S];
        const int *p = W + (long long)(i / R) * ldw + j;
        if (vec && j + S <= n) {
#pragma unroll
            for (int s = 0; s + 4 <= S; s += 4) {
                const int4 q = __ldg(reinterpret_cast<const int4 *>(p + s));
                x[s] = q.x, x[s + 1] = q.y, x[s + 2] = q.z, x[s + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int s = 0; s < S; ++s) x[s] = j + s < n ? __ldg(p + s) : 0;  // an absent target: nothing to lower
        }
        Vec<NV> y;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if constexpr (U16) y.w[q] = min(x[2 * q], BTAS_INF_U16) | min(x[2 * q + 1], BTAS_INF_U16) << 16;
            else y.w[q] = (unsigned)x[q];
        }
        Y[i] = y;
    }
}

// Y -> columns [j0, j0 + targets) of D.
template <bool U16, int R, int NV>
__device__ __forceinline__ void store_columns(int *D, long long ldd, int n, const Vec<NV> *Y, int j0) {
    constexpr int S = targets<U16, 1, NV>();
    const bool vec = S % 4 == 0 && (ldd & 3) == 0 && (reinterpret_cast<uintptr_t>(D) & 15) == 0;
    for (int i = threadIdx.x; i < n * R; i += blockDim.x) {
        const int j = j0 + (i % R) * S;
        const Vec<NV> y = Y[i];
        int x[S];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if constexpr (U16) {
                x[2 * q] = (int)(y.w[q] & 0xFFFFu);
                x[2 * q + 1] = (int)(y.w[q] >> 16);
                if (x[2 * q] == BTAS_INF_U16) x[2 * q] = kInfI32;
                if (x[2 * q + 1] == BTAS_INF_U16) x[2 * q + 1] = kInfI32;
            } else {
                x[q] = (int)y.w[q];
            }
        }
        int *p = D + (long long)(i / R) * ldd + j;
        if (vec && j + S <= n) {
#pragma unroll
            for (int s = 0; s + 4 <= S; s += 4)
                *reinterpret_cast<int4 *>(p + s) = make_int4(x[s], x[s + 1], x[s + 2], x[s + 3]);
        } else {
#pragma unroll
            for (int s = 0; s < S; ++s)
                if (j + s < n) p[s] = x[s];
        }
    }
}

struct Looks {  // in shared memory, set by thread 0 before a solve's first sweep
    int found;    // entries
    float last_found, last_t;
};

// Whether a tenth of the vertices still misses a path to some target; the same in every
// thread.  Called by the whole block.
template <bool U16, int R, int NV>
__device__ __forceinline__ bool some_missing(const Vec<NV> *Y, int n) {
    const int rows = n * R, looked = min(rows, (int)blockDim.x);
    const int i = rows > looked ? (int)((long long)threadIdx.x * rows / looked) : threadIdx.x;
    const bool missing = i < rows && top<U16, NV>(lds_relaxed(Y + i)) >= (U16 ? BTAS_INF_U16 : kInfI32);
    return 10 * __syncthreads_count(missing) > looked;
}

// Whether the patience of a block with distances missing is at its end, asked after
// every 8 sweeps from 16 on; valid in thread 0.  t0: the clock when the solve began.
// Called by the whole block; random graphs do not get here, whose smallest batches would
// pay for fetching these instructions (32 graphs of n = 128: 10 of 90 us).
template <bool U16, int R, int NV>
__device__ __forceinline__ bool late(const Patience &p, const Vec<NV> *Y, int n, int sweeps, long long t0, Looks &k) {
    int c = 0;
    for (int i = threadIdx.x; i < n * R; i += blockDim.x) {
        const Vec<NV> y = lds_relaxed(Y + i);
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if (U16) c += ((y.w[q] & 0xFFFFu) != BTAS_INF_U16) + ((y.w[q] >> 16) != BTAS_INF_U16);
            else c += (int)y.w[q] < kInfI32;
        }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) atomicAdd(&k.found, c);
    __syncthreads();
    if (threadIdx.x != 0) return false;
    const float found = (float)k.found / ((float)n * (float)targets<U16, R, NV>());
    k.found = 0;  // for the next look, some barriers from here
    const float t = (float)(clock64() - t0), worth = (float)(U16 ? p.worth16 : p.worth32);
    const float more = (1.0f - found) * (t - k.last_t) / fmaxf(found - k.last_found, 1e-6f);
    k.last_found = found;
    k.last_t = t;
    if (found >= 0.9f) return t > 1.5f * worth;  // near its end
    return sweeps < kSettle ? t > worth : t > 2.0f * worth || fminf(t / found - t, more) > worth;
}

// The same out of the way of the sweeps' registers, for rows of 4 words.  Smaller rows
// take it in line: a kernel without calls needs no stack, and small graphs show it (n =
// 49 ... 304: 1 to 2 %).
template <bool U16, int R, int NV>
__device__ __noinline__ bool late_apart(const Patience &p, const Vec<NV> *Y, int n, int sweeps, long long t0,
                                        Looks &k) {
    return late<U16, R, NV>(p, Y, n, sweeps, t0, k);
}

// Sweeps over all vertices until Y is the closure's columns.  A sweep lowers
// every Y[v] through v's edges, R lanes to a vertex's row and G sets of them to
// a vertex (set g takes chunks g, g + G, ...).  A path of two or more edges that
// improves Y[v] starts with an edge of weight w and goes on for at least minw,
// so w + minw < max(Y[v]): the list is sorted, and the first chunk with w >=
// max(Y[v]) - minw ends it, for each lane by its own targets.
// A row whose list was cut short of that bound at the fixpoint is then relaxed
// from W itself, and the sweeps go on if that lowered anything.  In the end
// every edge that could lower an entry has been tried against final values.
//
// One thread asks give_up(late) from time to time, late: this block's patience
// is at its end; returns false if it said so.  start: the clock when the block
// began, earlier solves included.  Called by the whole block.
template <bool U16, int G, int R, int NV, class GiveUp>
__device__ __forceinline__ bool solve(const int *W, long long ldw, int n, const Lists &l, Vec<NV> *Y, int minw, int maxw,
                                      long long start, GiveUp give_up) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    constexpr int VW = 32 / (G * R);  // vertices of a warp
    static_assert(G <= kPadChunks, "every lane's share of a list ends with a pad chunk");
    const int sub = lane % R, g = (lane / R) % G;
    const Vec<NV> *Ys = Y + sub;  // Ys[v * R]: this lane's part of v's row
    int sweeps = 0;
    const long long t0 = clock64();
    __shared__ Looks looks;
    if (tid == 0) looks = Looks{0, 0.0f, 0.0f};
    // the same in every thread: distances were missing after 8 sweeps, and the budget
    // of cycles does not hold then, unless 16 bits are too few for some weight
    bool finding = false;
    const bool heavy = U16 && maxw >= BTAS_INF_U16;
    for (;;) {
        for (;;) {
            bool ch = false, cut = false;
            ++sweeps;
            const int early_c = sweeps <= kEarlySweeps ? kEarlyChunks : l.chunks;
            for (int v0 = warp * VW; v0 < n; v0 += nwarps * VW) {
                const int v = v0 + lane / (G * R);
                if (G == 1 && v >= n) break;
                const int vc = G == 1 ? v : min(v, n - 1);
                const Vec<NV> old = lds_relaxed(Ys + vc * R);
                Vec<NV> acc = old;
                int lim = top<U16, NV>(acc) - minw;
                const uint4 *pe = l.edges + chunk_at(l, vc, g);
                const int4 *pw = l.wide + chunk_at(l, vc, g);
                uint4 e = *pe;
                int4 w = make_int4(0, 0, 0, 0);
                if (!U16) w = *pw;
                const int heavy = 4 * (U16 ? (int)(e.x >> 16) : w.x);
                for (int c = g;;) {
                    if ((U16 ? (int)(e.x >> 16) : w.x) >= lim) break;
                    const Vec<NV> y0 = lds_relaxed(Ys + (e.x & 0xFFFFu) * R), y1 = lds_relaxed(Ys + (e.y & 0xFFFFu) * R);
                    const Vec<NV> y2 = lds_relaxed(Ys + (e.z & 0xFFFFu) * R), y3 = lds_relaxed(Ys + (e.w & 0xFFFFu) * R);
                    const unsigned w0 = U16 ? __byte_perm(e.x, 0, 0x3232) : (unsigned)w.x;
                    const unsigned w1 = U16 ? __byte_perm(e.y, 0, 0x3232) : (unsigned)w.y;
                    const unsigned w2 = U16 ? __byte_perm(e.z, 0, 0x3232) : (unsigned)w.z;
                    const unsigned w3 = U16 ? __byte_perm(e.w, 0, 0x3232) : (unsigned)w.w;
                    c += G;
                    const bool more = c < l.chunks;
                    if (more) {  // the next chunk, while this one is relaxed
                        pe += 32 * G;
                        e = *pe;
                        if (!U16) {
                            pw += 32 * G;
                            w = *pw;
                        }
                    }
                    relax_edge<U16, NV>(acc, y0, w0);
                    relax_edge<U16, NV>(acc, y1, w1);
                    relax_edge<U16, NV>(acc, y2, w2);
                    relax_edge<U16, NV>(acc, y3, w3);
                    if (!more) break;
                    lim = top<U16, NV>(acc) - minw;
                    // an early sweep leaves the heavier edges for later
                    if (c >= early_c && (U16 ? (int)(e.x >> 16) : w.x) >= heavy) {
                        cut = true;
                        break;
                    }
                }
                if (G > 1) {
                    __syncwarp();
#pragma unroll
                    for (int o = G * R / 2; o >= R; o >>= 1) min_with_lane<U16, NV>(acc, o);
                }
                if (!U16) clamp(acc);
                if (differ(acc, old) && (G == 1 || (g == 0 && v < n))) {
                    sts_relaxed(Y + v * R + sub, acc);
                    ch = true;
                }
            }
            if (!__syncthreads_or(ch || cut)) break;
            if ((sweeps & 7) == 0) {
                if (sweeps == 8) finding = l.patience.by_share && some_missing<U16, R, NV>(Y, n);
                bool at_end = (!finding || heavy) && clock64() - start > (U16 ? 1 : 2) * l.patience.cycles;
                if (finding && sweeps > 8) {
                    if constexpr (NV == 4) at_end |= late_apart<U16, R, NV>(l.patience, Y, n, sweeps, t0, looks);
                    else at_end |= late<U16, R, NV>(l.patience, Y, n, sweeps, t0, looks);
                }
                if (__syncthreads_or(tid == 0 && give_up(at_end))) return false;
            }
        }
        bool ch = false;
        for (int v0 = warp * VW; v0 < n; v0 += nwarps * VW) {
            const int vv = min(v0 + lane / (G * R), n - 1);
            const bool need = l.next[vv] < top<U16, NV>(lds_relaxed(Ys + vv * R)) - minw;
            for (unsigned m = __ballot_sync(0xffffffffu, need); m;) {
                const int first = (__ffs(m) - 1) / (G * R);  // the row's number in the warp
                m &= ~(((1u << (G * R)) - 1u) << (first * G * R));
                const int v = min(v0 + first, n - 1);
                const Vec<NV> old = lds_relaxed(Ys + v * R);
                Vec<NV> acc = old;
                const int *wr = W + (long long)v * ldw;
                for (int k = lane / R; k < n; k += 32 / R) {
                    const int w = __ldg(wr + k);
                    if (w < (U16 ? BTAS_INF_U16 : kInfI32))
                        relax_edge<U16, NV>(acc, lds_relaxed(Ys + k * R),
                                            U16 ? (unsigned)w * 0x10001u : (unsigned)w);
                }
                __syncwarp();
#pragma unroll
                for (int o = 16; o >= R; o >>= 1) min_with_lane<U16, NV>(acc, o);
                if (!U16) clamp(acc);
                if (differ(acc, old)) {
                    if (lane < R) sts_relaxed(Y + v * R + sub, acc);
                    ch = true;
                }
            }
        }
        if (!__syncthreads_or(ch)) return true;
        // (reading whole rows takes many sweeps' time)
        if (__syncthreads_or(tid == 0 && give_up(clock64() - start > (U16 ? 1 : 2) * l.patience.cycles))) return false;
    }
}

// Whether 16 bits were enough.  Saturating sums commute with the minimum, so
// Y = min(distance, 0x7FFF); an entry at 0x7FFF is a missing path when no
// finite distance plus one edge, and no path of n - 1 edges, reaches 0x7FFF.
template <int R, int NV>
__device__ __forceinline__ bool fits16(const Vec<NV> *Y, int n, int maxw) {
    int inf = 0, fin = 0;
    for (int i = threadIdx.x; i < n * R; i += blockDim.x) {
        const Vec<NV> y = Y[i];
#pragma unroll
        for (int s = 0; s < 2 * NV; ++s) {
            const int x = (int)((y.w[s >> 1] >> (16 * (s & 1))) & 0xFFFFu);
            if (x == BTAS_INF_U16) inf = 1;
            else fin = max(fin, x);
        }
    }
    const bool some_inf = __syncthreads_or(inf) != 0;
    const bool some_far = __syncthreads_or((long long)fin + maxw >= BTAS_INF_U16) != 0;
    return !some_inf || !some_far || (long long)(n - 1) * maxw < BTAS_INF_U16;
}

}  // namespace relax
}  // namespace btas
