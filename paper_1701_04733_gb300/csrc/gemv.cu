// Level 2: tropical matrix-vector products, and single-source shortest paths
// by repeated vector-matrix products (Bellman-Ford in min-plus form).
//
//   trans == 0: y[i] = (+)_j A[i][j] (.) x[j]   one warp per row, 128-bit
//               loads along the row, warp-shuffle (+)-reduction
//   trans == 1: y[j] = (+)_i x[i] (.) A[i][j]   one thread per 4 columns,
//               row chunks spread over the grid, partial results combined
//               with atomic min/max (order-independent, so exact)
// Both stream A once: HBM-bound (4 bytes of A per term).
#include <algorithm>
#include <cstdint>
#include <mutex>

#include "common.cuh"
#include "grid_sync.cuh"
#include "kernels.h"

namespace btas {

namespace {

template <typename T, int SR>
__device__ __forceinline__ T op_plus(T a, T b) {
    return SR == kMin ? (b < a ? b : a) : (b > a ? b : a);
}
template <int SR>
__device__ __forceinline__ int op_times(int a, int b) {
    return clamp_i32<SR>(a + b);
}
template <int SR>
__device__ __forceinline__ float op_times(float a, float b) {
    return __fadd_rn(a, b);
}

// (+)-combine v into *addr atomically; returns true if *addr changed.
template <int SR>
__device__ __forceinline__ bool atomic_oplus(int *addr, int v) {
    const int old = SR == kMin ? atomicMin(addr, v) : atomicMax(addr, v);
    return SR == kMin ? v < old : v > old;
}
// Float min/max through integer atomics: non-negative floats order like
// their bit patterns as signed ints, negative floats in reverse as unsigned.
template <int SR>
__device__ __forceinline__ bool atomic_oplus(float *addr, float v) {
    if (SR == kMin) {
        if (__float_as_int(v) >= 0) return v < __int_as_float(atomicMin(reinterpret_cast<int *>(addr), __float_as_int(v)));
        return v < __uint_as_float(atomicMax(reinterpret_cast<unsigned *>(addr), __float_as_uint(v)));
    }
    if (__float_as_int(v) >= 0) return v > __int_as_float(atomicMax(reinterpret_cast<int *>(addr), __float_as_int(v)));
    return v > __uint_as_float(atomicMin(reinterpret_cast<unsigned *>(addr), __float_as_uint(v)));
}

template <typename T, int SR>
__global__ void gemv_rows_kernel(int m, int n, const T *__restrict__ A, long long lda, const T *__restrict__ x,
                                 T *__restrict__ y, int accumulate, int vec) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= m) return;
    const T *row = A + (long long)warp * lda;
    T acc = Ident<T, SR>::v();
    if (vec) {
        int j = lane * 4;
        // four independent 128-bit loads in flight per lane
        for (; j + 384 + 4 <= n; j += 512) {
            uint4 a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = __ldg(reinterpret_cast<const uint4 *>(row + j + 128 * u));
                b[u] = __ldg(reinterpret_cast<const uint4 *>(x + j + 128 * u));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t av[4] = {a[u].x, a[u].y, a[u].z, a[u].w}, bv[4] = {b[u].x, b[u].y, b[u].z, b[u].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    T ae, be;
                    memcpy(&ae, &av[q], 4);
                    memcpy(&be, &bv[q], 4);
                    acc = op_plus<T, SR>(acc, op_times<SR>(ae, be));
                }
            }
        }
        for (; j < n; j += 128) {
            if (j + 4 <= n) {
                const uint4 a = __ldg(reinterpret_cast<const uint4 *>(row + j));
                const uint4 b = __ldg(reinterpret_cast<const uint4 *>(x + j));
                const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    T ae, be;
                    memcpy(&ae, &av[q], 4);
                    memcpy(&be, &bv[q], 4);
                    acc = op_plus<T, SR>(acc, op_times<SR>(ae, be));
                }
            } else {
                for (int q = j; q < n; ++q) acc = op_plus<T, SR>(acc, op_times<SR>(row[q], x[q]));
            }
        }
    } else {
        for (int j = lane; j < n; j += 32) acc = op_plus<T, SR>(acc, op_times<SR>(row[j], x[j]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = op_plus<T, SR>(acc, __shfl_xor_sync(0xffffffffu, acc, o));
    if (lane == 0) y[warp] = accumulate ? op_plus<T, SR>(y[warp], acc) : acc;
}

constexpr int kColThreads = 256, kRowChunk = 64;

// y[j] (+)= (+)_{i in chunk} x[i] (.) A[i][j]; y must hold the (+)-identity
// or the accumulate start values.  *changed is set if some y entry changed.
template <typename T, int SR>
__global__ void gemv_cols_kernel(int m, int n, const T *__restrict__ A, long long lda, const T *__restrict__ x,
                                 T *y, int *changed, const int *skip, int vec) {
    if (skip != nullptr && __ldcg(skip) == 0) return;  // the previous relaxation changed nothing
    const int j0 = (blockIdx.x * kColThreads + threadIdx.x) * 4;
    const int i0 = blockIdx.y * kRowChunk, i1 = min(m, i0 + kRowChunk);
    if (j0 >= n) return;
    T acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = Ident<T, SR>::v();
    const bool full = vec && j0 + 4 <= n;
#pragma unroll 8
    for (int i = i0; i < i1; ++i) {
        const T xi = __ldg(x + i);
        const T *row = A + (long long)i * lda;
        if (full) {
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(row + j0));
            const uint32_t av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                T ae;
                memcpy(&ae, &av[q], 4);
                acc[q] = op_plus<T, SR>(acc[q], op_times<SR>(xi, ae));
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (j0 + q < n) acc[q] = op_plus<T, SR>(acc[q], op_times<SR>(xi, row[j0 + q]));
        }
    }
    bool ch = false;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (j0 + q < n && acc[q] != Ident<T, SR>::v()) ch |= atomic_oplus<SR>(y + j0 + q, acc[q]);
    if (changed != nullptr && ch) atomicOr(changed, 1);
}

template <typename T>
__global__ void fill_kernel(T *y, int n, T v) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = v;
}

template <typename T, int SR>
cudaError_t gemv_t(int trans, int m, int n, const void *A, long long lda, const void *x, void *y, int accumulate,
                   int *changed, const int *skip, cudaStream_t st) {
    const T *a = static_cast<const T *>(A);
    const T *xx = static_cast<const T *>(x);
    T *yy = static_cast<T *>(y);
    if (trans == 0) {
        const int vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(xx)) & 15) == 0 && (lda & 3) == 0;
        const int blocks = (m + 7) / 8;
        gemv_rows_kernel<T, SR><<<blocks, 256, 0, st>>>(m, n, a, lda, xx, yy, accumulate, vec);
        note_launch();
    } else {
        if (!accumulate) {
            int b = (n + 255) / 256;
            b = b > 1216 ? 1216 : (b < 1 ? 1 : b);
            fill_kernel<T><<<b, 256, 0, st>>>(yy, n, Ident<T, SR>::v());
            note_launch();
        }
        const int vec = (reinterpret_cast<uintptr_t>(a) & 15) == 0 && (lda & 3) == 0;
        dim3 grid((n + 4 * kColThreads - 1) / (4 * kColThreads), (m + kRowChunk - 1) / kRowChunk);
        gemv_cols_kernel<T, SR><<<grid, kColThreads, 0, st>>>(m, n, a, lda, xx, yy, changed, skip, vec);
        note_launch();
    }
    return cudaGetLastError();
}

// ---- Bellman-Ford SSSP (repeated vector-matrix products) in ONE
// cooperative launch.  d_0 = e_src; d_{t+1}[j] = min_i d_t[i] + W[i][j] until
// d stops changing (at most n - 1 products).
//
// Only a vertex that product t lowered can lower anything in product t + 1, so
// a product relaxes the edges of those vertices and nothing else.  The first
// pass reads W once, for the domain check, the first product (row src) and the
// edge lists of all rows; a row with more edges than its list holds is relaxed
// from W.  W is thus read once and not once per product:
// 1105 -> 203 us per call at n = 8192 (p = 0.01, 19 products), 1141 -> 615 us on a
// complete graph (21 products), 216 -> 151 us on one of n = 2048.
//
// Three buffers rotate.  Product t reads d_{t-1} and d_{t-2}, whose difference is
// the set of vertices to relax, and lowers the third, which holds d_{t-3}, by
// d_{t-1} and by its candidates, in any order (min commutes): that makes it d_t.
// No entry that is read changes meanwhile, so the products, and the number of
// them that change d, are those of the definition.  A product is one grid barrier
// and three dependent L2 round trips.  Each vertex with a list belongs to a warp;
// long rows are shared out by 32 rows x 128 columns, so that a warp merges the
// changed ones among its rows in registers.
constexpr int kSsspThreads = 1024;
constexpr int kSsspSeg = 1024;  // entries of a row that one warp takes at a time

struct SsspArgs {
    const int *W;
    long long ldw;
    int n;
    int src;
    int vec;         // W rows 16-byte aligned (int4 loads)
    int *d;          // three buffers of ld ints
    long long ld;
    int *any_long;   // some row is longer than its list.  Zero first
    int *deg;        // edges of each row.  Zero first
    int2 *lists;     // cap edges (column, weight) per row, in no particular order
    int cap;
    int *dist;
    GridSync sync;   // status: info[1]
    int *info;       // [0] products that changed d, [1] status, [2] entries of W outside the domain
};

// s = d_t[u] + w for edge (u, j): lowers out[j] where it is below in[j].
__device__ __forceinline__ bool sssp_relax(const int *in, int *out, int s, int j) {
    if (s >= kClampI32 || s >= __ldcg(in + j)) return false;
    atomicMin(out + j, s);
    return true;
}

// Row i's entries [c0, c1), kSsspSeg at most: edges to the row's list.  Each
// lane keeps its 32 entries in registers, and one atomicAdd reserves the
// warp's places.  Returns the entries outside the domain.
__device__ __forceinline__ int sssp_list(const SsspArgs &a, int i, int c0, int c1, int lane) {
    const int *row = a.W + (long long)i * a.ldw;
    constexpr int U = kSsspSeg / 128;
    int x[4 * U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int j = c0 + 128 * u + 4 * lane;
        int4 v = make_int4(kInfI32, kInfI32, kInfI32, kInfI32);
        if (a.vec) {
            if (j < c1) v = __ldg(reinterpret_cast<const int4 *>(row + j));
        } else {
            if (j < c1) v.x = __ldg(row + j);
            if (j + 1 < c1) v.y = __ldg(row + j + 1);
            if (j + 2 < c1) v.z = __ldg(row + j + 2);
            if (j + 3 < c1) v.w = __ldg(row + j + 3);
        }
        x[4 * u] = v.x, x[4 * u + 1] = v.y, x[4 * u + 2] = v.z, x[4 * u + 3] = v.w;
    }
    unsigned edges = 0;
    int bad = 0;
#pragma unroll
    for (int e = 0; e < 4 * U; ++e) {
        const bool fin = (unsigned)x[e] <= (unsigned)BTAS_I32_FINITE_MAX;
        bad += !fin && x[e] != kInfI32;
        edges |= (fin ? 1u : 0u) << e;
    }
    const int self = i - c0 - 4 * lane;  // i's place in this lane's entries, if it is one
    if (self >= 0 && i < c1 && (self & 127) < 4) {
        const int e = (self >> 7) * 4 + (self & 3);
        if (!((edges >> e) & 1u)) bad += row[i] == kInfI32;  // any other value was counted
        else bad += row[i] != 0;
        edges &= ~(1u << e);
    }
    const int own = __popc(edges);
    int at = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    const int tot = __shfl_sync(0xffffffffu, at, 31);
    if (tot == 0) return bad;
    int base = 0;
    if (lane == 0) {
        base = atomicAdd(a.deg + i, tot);
        if (base + tot > a.cap) *a.any_long = 1;
    }
    at += __shfl_sync(0xffffffffu, base, 0) - own;
    int2 *L = a.lists + (long long)i * a.cap;
#pragma unroll
    for (int e = 0; e < 4 * U; ++e)
        if ((edges >> e) & 1u) {
            if (at < a.cap) L[at] = make_int2(c0 + 128 * (e >> 2) + 4 * lane + (e & 3), x[e]);
            ++at;
        }
    return bad;
}

__global__ void __launch_bounds__(kSsspThreads, 1) sssp_coop_kernel(const SsspArgs a) {
    const int n = a.n, lane = threadIdx.x & 31;
    const long long gthreads = (long long)gridDim.x * blockDim.x;
    const long long gtid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    // consecutive numbers on different SMs
    const int nw = (int)(gthreads >> 5), gw = (int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    unsigned gen = 0;
    // d_0, d_1, and the buffer of d_2
    bool ch = false;
    for (long long j = gtid; j < n; j += gthreads) {
        const int w = a.W[(long long)a.src * a.ldw + j];
        const bool edge = j != a.src && (unsigned)w <= (unsigned)BTAS_I32_FINITE_MAX;
        const int d0 = j == a.src ? 0 : kInfI32;
        a.d[j] = d0;
        a.d[a.ld + j] = edge ? w : d0;
        a.d[2 * a.ld + j] = kInfI32;
        ch |= edge;
    }
    const int segs = (n + kSsspSeg - 1) / kSsspSeg;
    int bad = 0;
    for (long long it = gw; it < (long long)n * segs; it += nw) {
        const int i = (int)(it / segs), c0 = (int)(it % segs) * kSsspSeg;
        bad += sssp_list(a, i, c0, min(n, c0 + kSsspSeg), lane);
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0 && bad) atomicAdd(a.info + 2, bad);
    int changed = 0, v1 = 0;
    if (!grid_barrier_fn(
            a.sync, gen, ch,
            [&]() -> unsigned {
                return (gsync::ld_relaxed_i32(a.info + 2) ? 1u : 0u) | (gsync::ld_relaxed_i32(a.any_long) ? 2u : 0u);
            },
            changed, v1))
        return;
    if (v1 & 1) return;  // W outside the domain: dist untouched
    const bool long_rows = (v1 & 2) != 0;
    // vertices [w0, w1) are this warp's
    const int per = (n + nw - 1) / nw;
    const int w0 = (int)min((long long)gw * per, (long long)n), w1 = min(w0 + per, n);
    int done = 0;
    const int *in = a.d + a.ld;
    for (int t = 2; changed; ++t) {
        ++done;
        if (t > n - 1) break;
        const int *prev = a.d + (t - 2) % 3 * a.ld;
        int *out = a.d + t % 3 * a.ld;
        ch = false;
        for (int b = w0; b < w1; b += 32) {
            const int v = b + lane;
            int x = kInfI32, d = 0;
            bool go = false;
            if (v < w1) {
                x = __ldcg(in + v);
                d = __ldcg(a.deg + v);
                go = x != __ldcg(prev + v) && d <= a.cap;
                atomicMin(out + v, x);
            }
            for (unsigned m = __ballot_sync(0xffffffffu, go); m; m &= m - 1) {
                const int src = __ffs(m) - 1, xu = __shfl_sync(0xffffffffu, x, src);
                const int du = __shfl_sync(0xffffffffu, d, src);
                const int2 *L = a.lists + (long long)(b + src) * a.cap;
                for (int q0 = 0; q0 < du; q0 += 128) {
                    int2 e[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int k = q0 + 32 * q + lane;
                        e[q] = k < du ? __ldcg(L + k) : make_int2(0, kInfI32);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) ch |= sssp_relax(in, out, xu + e[q].y, e[q].x);
                }
            }
        }
        if (long_rows) {
            const int cblocks = (n + 127) / 128;
            for (long long it = gw; it < (long long)((n + 31) / 32) * cblocks; it += nw) {
                const int r = (int)(it / cblocks) * 32 + lane, j0 = (int)(it % cblocks) * 128 + 4 * lane;
                const int x = r < n ? __ldcg(in + r) : kInfI32;
                unsigned m = __ballot_sync(0xffffffffu, r < n && x != __ldcg(prev + min(r, n - 1)) &&
                                                            __ldcg(a.deg + min(r, n - 1)) > a.cap);
                if (m == 0) continue;
                int acc[4] = {kInfI32, kInfI32, kInfI32, kInfI32};
                while (m) {  // 8 rows at a time
                    int4 w[8];
                    int xq[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int src = m ? __ffs(m) - 1 : 0;
                        const int *p = a.W + (long long)(r - lane + src) * a.ldw + j0;
                        xq[q] = __shfl_sync(0xffffffffu, x, src);
                        w[q] = make_int4(kInfI32, kInfI32, kInfI32, kInfI32);
                        if (m == 0) continue;
                        m &= m - 1;
                        if (a.vec) {
                            if (j0 < n) w[q] = __ldg(reinterpret_cast<const int4 *>(p));
                        } else {
                            if (j0 < n) w[q].x = __ldg(p);
                            if (j0 + 1 < n) w[q].y = __ldg(p + 1);
                            if (j0 + 2 < n) w[q].z = __ldg(p + 2);
                            if (j0 + 3 < n) w[q].w = __ldg(p + 3);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        acc[0] = __viaddmin_s32(xq[q], w[q].x, acc[0]);
                        acc[1] = __viaddmin_s32(xq[q], w[q].y, acc[1]);
                        acc[2] = __viaddmin_s32(xq[q], w[q].z, acc[2]);
                        acc[3] = __viaddmin_s32(xq[q], w[q].w, acc[3]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (j0 + c < n) ch |= sssp_relax(in, out, acc[c], j0 + c);
            }
        }
        if (!grid_barrier(a.sync, gen, ch, nullptr, changed, v1)) return;
        in = out;
    }
    for (long long j = gtid; j < n; j += gthreads) a.dist[j] = __ldcg(in + j);
    if (gtid == 0) a.info[0] = done;
}

}  // namespace

cudaError_t launch_gemv(int sr, int dtype, int trans, int m, int n, const void *A, long long lda, const void *x,
                        void *y, int accumulate, int *changed, cudaStream_t st, const int *skip) {
    if (dtype == BTAS_I32)
        return sr == kMin ? gemv_t<int, kMin>(trans, m, n, A, lda, x, y, accumulate, changed, skip, st)
                          : gemv_t<int, kMax>(trans, m, n, A, lda, x, y, accumulate, changed, skip, st);
    return sr == kMin ? gemv_t<float, kMin>(trans, m, n, A, lda, x, y, accumulate, changed, skip, st)
                      : gemv_t<float, kMax>(trans, m, n, A, lda, x, y, accumulate, changed, skip, st);
}

namespace {
// Edges a row's list holds: an eighth of the row, 64 at least and 1024 at most.
// A longer row is relaxed from W, whose read is then not much longer than the
// list's.
int sssp_cap(long long n) { return (int)std::min(1024LL, std::max(64LL, n / 8)); }
size_t sssp_vec(long long n) { return ((size_t)n * 4 + 255) & ~size_t(255); }
}  // namespace

// barrier words, info words and row degrees (one memset), then the three
// buffers and the lists
size_t sssp_coop_workspace(long long n) {
    return 512 + 4 * sssp_vec(n) + (size_t)n * sssp_cap(n) * 8;
}

int *sssp_coop_info(void *ws) { return reinterpret_cast<int *>(static_cast<char *>(ws) + 256 + 64); }

cudaError_t launch_sssp_coop(const int *W, long long n, int src, int *dist, void *ws, cudaStream_t st) {
    DeviceInfo di{};
    if (!current_device_info(&di)) return cudaErrorInvalidDevice;
    const size_t vb = sssp_vec(n);
    char *p = static_cast<char *>(ws);
    SsspArgs a{};
    a.W = W;
    a.ldw = n;
    a.n = (int)n;
    a.src = src;
    a.vec = ((reinterpret_cast<uintptr_t>(W) & 15) == 0) && (n & 3) == 0;
    a.sync.bar = reinterpret_cast<unsigned *>(p);
    a.any_long = reinterpret_cast<int *>(p + 256);
    a.deg = reinterpret_cast<int *>(p + 512);
    p += 512 + vb;
    a.d = reinterpret_cast<int *>(p);
    a.ld = (long long)(vb / 4);
    a.lists = reinterpret_cast<int2 *>(p + 3 * vb);
    a.cap = sssp_cap(n);
    a.dist = dist;
    a.info = sssp_coop_info(ws);
    a.sync.status = a.info + 1;
    a.sync.timeout_cycles = (long long)(2.0 * (di.clock_khz > 0 ? di.clock_khz : 2000000) * 1e3);  // about 2 s
    cudaError_t e = cudaMemsetAsync(ws, 0, 512 + vb, st);
    if (e != cudaSuccess) return e;
    // one block per SM: fewer arrivals at the barriers, which are most of a product
    const long long segs = (n + kSsspSeg - 1) / kSsspSeg;
    const int grid = (int)std::max(1LL, std::min((n * segs + 31) / 32, (long long)di.sms));
    void *args[] = {&a};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(sssp_coop_kernel), dim3(grid), dim3(kSsspThreads),
                                    args, 0, st);
    note_launch();
    return e;
}

}  // namespace btas
