// APSP by relaxation over sorted edge lists, many targets at a time: what
// btas_apsp runs when the caller wants the distances alone.
//
// Squaring (Sec. III) computes n^3 terms several times over, and nearly all of
// them are sums of two long paths that a third one undercuts.  Bellman-Ford
// over W's edges computes far fewer, and every block can solve a few targets by
// itself, without a grid barrier: 16 bytes per vertex hold the distances to 8
// targets in 16 bits (or 4 in 32), which fits shared memory up to n = 14400.
// (Smaller graphs take 2 or 4 targets per block: launch_relax.)
// One edge is then one 16-byte load and 4 DPX add-mins for 8 terms.
//
// What makes it short is the order of the edges.  Each row's list is sorted by
// weight, and an edge of weight w cannot start a better path of two or more
// edges unless w plus the lightest weight of all stays below the largest of the
// vertex's current distances; so a sweep reads a row's list up to that bound
// only, about 3 chunks of 4 edges on random graphs, whatever their density.
// The same bound makes a list of the lightest edges enough on dense graphs; the
// rare row that needs more is read from W.  The first two sweeps also leave
// edges of 4 or more times the row's lightest weight for later (n = 8192, p =
// 0.01: 3.93 -> 3.32 ms; the same at p = 1).
//
// Sums of non-negative weights reach one fixpoint in any order, so the result is
// that of the squarings bit for bit; only the number of squarings is not known.
//
// Measured (GB300, us per call with its synchronisation, squarings -> relaxation):
//   n = 128 (complete), 256 (p = 0.1):              51 -> 34, 59 -> 39
//   n = 512, 1024 (p = 0.1, w <= 100):              94 -> 63, 290 -> 89
//   n = 2048 (p = 0.1 / complete, w <= 10^6):       1668 -> 187 / 3278 -> 250
//   n = 2999 (p = 0.5, w <= 10^6):                  11060 -> 570
//   n = 4096 (p = 0.05, w <= 7 / p = 0.01, w <= 10^6): 5840 -> 608 / 16790 -> 1514
//   n = 8192 (p = 0.01, w <= 1000 / complete, w <= 100): 93670 -> 3450 / 47010 -> 4045
// The sweeps are bound by shared memory: ncu at n = 4096 (p = 0.05, w <= 7) has the L1
// pipe 89 % busy while SMs are active, 35 % of its wavefronts bank conflicts of the
// random 16-byte rows (8 lanes on 8 bank groups).  Wider rows conflict less but do not
// fit; ordering a chunk's 4 edges by bank gains 5 %.
// The last wave costs 15-30 % where n / 8 blocks are few per SM.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "relax.cuh"

namespace btas {
namespace {

using relax::Lists;
using relax::RowStats;

constexpr int kListWarps = 8;               // rows of a block of the list kernel
constexpr int kSolveSmem = 225 * 1024;       // most dynamic shared memory of the solve kernel
constexpr int kTwoBlocksMaxN = 7000;         // 16 n bytes, twice, with what each block takes besides
static_assert(2 * (16 * kTwoBlocksMaxN + 2048) <= 228 * 1024, "two blocks per SM");
enum Ctl { kAbort = 0, kWide = 1, kDone = 2 };  // control words, cleared by the list kernel

struct RelaxArgs {
    const int *W;
    long long ldw;
    int n;
    Lists lists;
    RowStats *stats;  // one per block of the list kernel
    int *ctl;
    int *D;
    long long ldd;
    int *out;  // host-mapped words (see kernels.h)
    int *found;  // optional: four words, zero before, to take entries outside the domain, the largest weight, the
                 // most edges of a row (INT_MAX: some list does not hold its row) and all edges; then no stats
    int halves;  // 2: a second block takes half of each block's targets where 32 bits are needed from the start
};

__global__ void __launch_bounds__(kListWarps * 32) relax_lists_kernel(const RelaxArgs a) {
    __shared__ unsigned long long buf[kListWarps][relax::kCap];
    __shared__ int hist[kListWarps][256];
    __shared__ RowStats s_st[kListWarps];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x * kListWarps + warp;
    if (blockIdx.x == 0 && threadIdx.x < 3) a.ctl[threadIdx.x] = 0;
    RowStats st{0, 0, kInfI32, 0, 0, 0.0f};
    if (row < a.n) st = relax::build_row(a.W, a.ldw, a.n, row, a.lists, buf[warp], hist[warp], lane);
    if (lane == 0) s_st[warp] = st;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kListWarps; ++i) {
            const RowStats &o = s_st[i];
            st.bad += o.bad;
            st.maxw = max(st.maxw, o.maxw);
            st.minw = min(st.minw, o.minw);
            st.deg = max(st.deg, o.deg);
            st.far |= o.far;
            st.light += o.light;
            st.cut |= o.cut;
            st.edges += o.edges;
        }
        if (a.found != nullptr) {
            if (st.bad) atomicAdd(a.found, st.bad);
            atomicMax(a.found + 1, st.maxw);
            atomicMax(a.found + 2, st.cut ? 0x7FFFFFFF : st.deg);
            atomicAdd(a.found + 3, st.edges);
        } else {
            a.stats[blockIdx.x] = st;
        }
    }
}

template <int G, int NV, int MAXT>
__global__ void __launch_bounds__(MAXT) relax_solve_kernel(const RelaxArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto *Y = reinterpret_cast<relax::Vec<NV> *>(smem_raw);
    __shared__ int s_abort, s_wide;
    __shared__ RowStats s_st;
    const long long t0 = clock64();
    const int n = a.n, tid = threadIdx.x;
    constexpr int R = 1, T = relax::targets<true, R, NV>();  // targets of a block, in 16 bits
    const int groups = (n + T - 1) / T, part = blockIdx.x >= groups ? 1 : 0;  // the second parts on SMs of their own
    const int j0 = (blockIdx.x - part * groups) * T;
    if (tid == 0) s_st = RowStats{0, 0, kInfI32, 0, 0, 0.0f};
    if (part == 0) relax::load_columns<true, R, NV>(a.W, a.ldw, n, Y, j0);  // needs no lists
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    const int nst = (n + kListWarps - 1) / kListWarps;
    RowStats st{0, 0, kInfI32, 0, 0, 0.0f};
    for (int i = tid; i < nst; i += blockDim.x) {
        const RowStats o = a.stats[i];
        st.bad += o.bad;
        st.maxw = max(st.maxw, o.maxw);
        st.minw = min(st.minw, o.minw);
        st.deg = max(st.deg, o.deg);
        st.far |= o.far;
        st.light += o.light;
    }
    if (tid < nst) {
        if (st.bad) atomicAdd(&s_st.bad, st.bad);
        atomicMax(&s_st.maxw, st.maxw);
        atomicMin(&s_st.minw, st.minw);
        atomicMax(&s_st.deg, st.deg);
        if (st.far) atomicOr(&s_st.far, 1);
        atomicAdd(&s_st.light, st.light);
    }
    if (tid == 0) {
        s_abort = *(volatile int *)(a.ctl + kAbort);
        s_wide = *(volatile int *)(a.ctl + kWide);
    }
    __syncthreads();
    st = s_st;
    const bool wide_first = st.far != 0 || relax::expects_wide(n, st.light);  // the same in every block
    if (st.bad == 0 && s_abort == 0) {
        bool wide = wide_first || s_wide != 0;
        auto give_up = [&](bool late) {
            if (*(volatile int *)(a.ctl + kAbort) != 0) return true;
            if (late) a.ctl[kAbort] = 1;
            return late;
        };
        if (part == 0 && !wide && relax::solve<true, G, R, NV>(a.W, a.ldw, n, a.lists, Y, st.minw, st.maxw, t0, give_up)) {
            wide = !relax::fits16<R, NV>(Y, n, st.maxw);
            if (!wide) relax::store_columns<true, R, NV>(a.D, a.ldd, n, Y, j0);
            else if (tid == 0) a.ctl[kWide] = 1;
        }
        // in 32 bits, half of the targets at a time
        const bool split = wide_first && a.halves == 2;
        if (wide && (part == 0 || split)) {
            for (int h = part * T / 2; h < (split ? (part + 1) * T / 2 : T) && j0 + h < n; h += T / 2) {
                __syncthreads();
                relax::load_columns<false, R, NV>(a.W, a.ldw, n, Y, j0 + h);
                __syncthreads();
                if (!relax::solve<false, G, R, NV>(a.W, a.ldw, n, a.lists, Y, st.minw, st.maxw, t0, give_up)) break;
                relax::store_columns<false, R, NV>(a.D, a.ldd, n, Y, j0 + h);
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(a.ctl + kDone, 1) == (int)gridDim.x - 1) {  // the last block tells the host
            __threadfence();
            a.out[1] = st.bad;
            a.out[2] = st.deg;
            a.out[3] = *(volatile int *)(a.ctl + kWide) | st.far;
            __threadfence_system();  // the host may watch out[0]
            a.out[0] = st.bad ? kRelaxBad : *(volatile int *)(a.ctl + kAbort) ? kRelaxGaveUp : kRelaxDone;
            __threadfence_system();
        }
    }
}

// The first squaring of W with smallest minimising k, as keys (value << shift) |
// k, from the lists: row i of K in shared memory starts with the terms k = i and k
// = j, both W[i][j], and takes the terms of every pair of edges (i, k), (k, j).
// One block per row; its warps take row i's edges in turn and read row k's list
// along their lanes.
__global__ void __launch_bounds__(256) sparse_key_kernel(const int *W, int n, Lists l, int shift, int *K) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *key = reinterpret_cast<int *>(smem_raw);
    const int i = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int w = W[(long long)i * n + j];
        key[j] = w < kInfI32 ? (w << shift) | min(i, j) : kInfI32;
    }
    __syncthreads();
    const int own = l.len[i];
    for (int e = warp; e < own; e += warps) {
        const size_t at = relax::chunk_at(l, i, e >> 2) * 4 + (e & 3);
        const int k = (int)(reinterpret_cast<const unsigned *>(l.edges)[at] & 0xFFFFu);
        const int w1 = reinterpret_cast<const int *>(l.wide)[at], len = l.len[k];
        for (int c = lane; 4 * c < len; c += 32) {
            const uint4 to = l.edges[relax::chunk_at(l, k, c)];
            const int4 w2 = l.wide[relax::chunk_at(l, k, c)];
            const unsigned j[4] = {to.x & 0xFFFFu, to.y & 0xFFFFu, to.z & 0xFFFFu, to.w & 0xFFFFu};
            const int w[4] = {w2.x, w2.y, w2.z, w2.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (4 * c + q < len) atomicMin(key + j[q], ((w1 + w[q]) << shift) | k);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) K[(long long)i * n + j] = key[j];
}

size_t align256(size_t v) { return (v + 255) & ~size_t(255); }
}  // namespace

int relax_max_n() { return kSolveSmem / 16; }

size_t relax_workspace(long long n) {
    const size_t rows = (size_t)((n + 31) & ~31LL);
    return 256 + align256((size_t)((n + kListWarps - 1) / kListWarps) * sizeof(RowStats)) + align256(rows * 4) +
           relax::list_words(n) * 8;
}

namespace {
// Places in a workspace of relax_workspace(n) bytes.
void place(void *ws, int n, int **ctl, RowStats **stats, Lists *lists) {
    const size_t rows = (size_t)((n + 31) & ~31);
    char *p = static_cast<char *>(ws);
    *ctl = reinterpret_cast<int *>(p);
    *stats = reinterpret_cast<RowStats *>(p += 256);
    lists->next = reinterpret_cast<int *>(p += align256((n + kListWarps - 1) / kListWarps * sizeof(RowStats)));
    lists->edges = reinterpret_cast<uint4 *>(p += align256(rows * 4));
    lists->wide = reinterpret_cast<int4 *>(p + relax::list_words(n) * 4);
    lists->chunks = relax::list_chunks(n);
}
}  // namespace

size_t edge_lists_workspace(long long n) { return relax_workspace(n) + align256((size_t)n * 4); }

// The most edges that a row's list is kept for, and the most edges of all with
// which the pairs of edges (all d^2 of a row, on average) pay.  us per call, dense
// first squaring / over the lists, all rows with n / 8, n / 7, n / 6 and n / 5 edges: n =
// 300 284/270, 274/261, 278/270, 273/263; n = 600 410/385, 406/394, 410/403, 408/415; n =
// 1000 725/708, 726/721, 726/761, 725/801; n = 2048 3492/3465, 4049/4192, 3490/3866,
// 3487/4252; n = 3000 10009/9987, 11671/12095, 10019/11165.
static int sparse_row(long long n) { return (int)std::max(1LL, std::min<long long>(relax::kCap, n / 6)); }

bool sparse_keys_pay(long long n, int most_edges, int edges) {
    return most_edges <= sparse_row(n) && (n < 800 || 8LL * edges <= n * n);
}

// A row too full or too heavy decides against sparse_keys_pay, so its list is
// not sorted or stored: with every list built a whole call on n = 519, p = 0.35
// took 9 us longer than with a plain scan of W (453 against 444), so it takes 6
// us less (388 against 394).
cudaError_t launch_edge_lists(const int *W, int n, int max_weight, void *ws, int *found, cudaStream_t st) {
    const int blocks = (n + kListWarps - 1) / kListWarps;
    RelaxArgs a{};
    a.W = W;
    a.ldw = n;
    a.n = n;
    place(ws, n, &a.ctl, &a.stats, &a.lists);
    a.lists.len = reinterpret_cast<int *>(static_cast<char *>(ws) + relax_workspace(n));
    a.lists.whole = sparse_row(n);
    a.lists.top = max_weight;
    a.found = found;
    relax_lists_kernel<<<blocks, kListWarps * 32, 0, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_sparse_keys(const int *W, int n, void *ws, int shift, int *K, cudaStream_t st) {
    Lists l{};
    int *ctl;
    RowStats *stats;
    place(ws, n, &ctl, &stats, &l);
    l.len = reinterpret_cast<int *>(static_cast<char *>(ws) + relax_workspace(n));
    sparse_key_kernel<<<n, 256, (size_t)n * 4, st>>>(W, n, l, shift, K);
    note_launch();
    return cudaGetLastError();
}

// A block's patience in a call of its own: `blocks` with all targets, `resident`
// of them at once; split: in 32 bits twice as many with half of them each, else one
// half after the other.  What a call takes where its relaxation is given up, in
// cycles (chains, GB300): below n = 2048 the squarings, 68 us at n = 128, 148 at 512,
// 555 at 1024, 3280 at 2047 in 16 bits and 73, 180, 805, 5300 in 32; from there on
// blocked Floyd-Warshall, 2.1 ms at n = 2048, 5.4 at 4096.
static relax::Patience relax_patience(long long n, int blocks, int resident, bool split) {
    relax::Patience p{};
    if (const char *e = getenv("BTAS_RELAX_BUDGET"); e && *e) {
        p.cycles = atoll(e);
        return p;
    }
    p.by_share = true;
    p.cycles = relax::budget_cycles(n);
    const double n3 = (double)n * n * n, fw = 1730.0 * n + n3 / 20000;
    const double worth16 = n < 2048 ? 110e3 + 120.0 * n + n3 / 1500 : fw;
    const double worth32 = n < 2048 ? 110e3 + 120.0 * n + n3 / 900 : fw;
    p.worth16 = (long long)(worth16 * std::min(1.0, (double)resident / blocks));
    p.worth32 = (long long)(worth32 * (split ? std::min(1.0, 0.5 * resident / blocks)
                                             : 0.5 * std::min(1.0, (double)resident / blocks)));
    return p;
}

cudaError_t launch_relax(const int *W, long long ldw, int n, int *D, long long ldd, void *ws, int *out,
                         cudaStream_t st) {
    const int blocks = (n + kListWarps - 1) / kListWarps;
    RelaxArgs a{};
    a.W = W;
    a.ldw = ldw;
    a.n = n;
    a.D = D;
    a.ldd = ldd;
    a.out = out;
    place(ws, n, &a.ctl, &a.stats, &a.lists);
    DeviceInfo di{};
    const int sms = current_device_info(&di) ? di.sms : 152;
    // Two blocks share a block's targets in 32 bits while one wave holds them all (n =
    // 1024, w <= 10^6, p = 0.5: 283 -> 158 us per call).
    a.halves = n <= 8 * sms ? 2 : 1;
    relax_lists_kernel<<<blocks, kListWarps * 32, 0, st>>>(a);
    note_launch();
    // Small graphs take fewer targets per block, so that more SMs share the
    // sweeps' shared-memory loads: 2 while that makes at most a block per SM (n <= 304
    // on 152 SMs; 46 -> 41 us per call at n = 256, p = 0.1) and 4 likewise (n <= 608; 60
    // -> 55 us at n = 512); two lanes per vertex while one would leave warps idle.
    // From there on 8 targets, with 1024 threads where one block per SM holds all
    // targets (n = 1024, p = 0.1: 93 us, 112 with 512 threads) or fills shared memory (n
    // = 8192: 3662 us against 3779), 512 and two blocks per SM between (n = 4096, p =
    // 0.01: 1060 us against 1118).  Rows of 16 or 32 targets, which pay in the batched
    // launch, lose more to their fewer blocks than they gain (n = 2048: 265 and 377 us
    // against 249).  (These figures compare the shapes; the calls were 4 to 40 us longer
    // then than above.)
    const int words = n <= 2 * sms ? 1 : n <= 4 * sms ? 2 : 4, lanes = words == 1 ? 2 : 1;
    const int maxt = (words == 4 && n <= 8 * sms) || n > kTwoBlocksMaxN ? 1024 : 512;
    void (*kern)(const RelaxArgs) = words == 1 ? relax_solve_kernel<2, 1, 512>
                                    : words == 2 ? relax_solve_kernel<1, 2, 512>
                                    : maxt == 512 ? relax_solve_kernel<1, 4, 512> : relax_solve_kernel<1, 4, 1024>;
    cudaError_t e = set_smem_once(reinterpret_cast<const void *>(kern), kSolveSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((n + 2 * words - 1) / (2 * words) * a.halves);
    cfg.blockDim = dim3(std::min(maxt, (n * lanes + 31) / 32 * 32));
    cfg.dynamicSmemBytes = (size_t)n * 4 * words;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    a.lists.patience = relax_patience(n, cfg.gridDim.x / a.halves, (maxt == 1024 ? 1 : 2) * sms, a.halves == 2);
    e = cudaLaunchKernelEx(&cfg, kern, a);
    if (e == cudaSuccess) note_launch();
    return e;
}

}  // namespace btas
