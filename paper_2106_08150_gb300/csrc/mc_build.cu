// Database build kernels (Section 4.1 build phase, Section 5.1 GPU hash
// tables, Section 5.2 build pipeline) for sm_103a.
//
// GB300 design.  The paper inserts each (feature, location) pair into a
// multi-bucket hash table with warp-aggregated atomics.  Here the build is
// organised around streaming HBM passes instead of random-sector updates:
//   1. sketch + emit: a warp sketches 32 windows at a time, one per lane
//      (shared with the query path, mc_sketch.cuh), and writes (h2(feature)
//      << 32 | global window) pairs in window order;
//   2. a stable LSD radix sort (4 single-pass digits of 8 bits over the
//      upper word) groups the pairs by feature while keeping them in window order,
//      which is (target, window) order, so every bucket comes out sorted;
//   3. finalize keeps the first `cap` pairs of each feature (Section 4.1:
//      at most 254 locations per feature; the smallest are kept, as in the
//      CPU version that inserts in ascending order), converts global windows
//      to (target, window) locations, and lays out the condensed layout of
//      Section 5.1: one contiguous location array plus a feature table;
//   4. the feature table is an ordered linear-probing table built without
//      atomics: features arrive sorted by h2, so slot(k) = max(home(k),
//      slot(k-1)+1) = k + max_{k'<=k}(home(k') - k'), a max-scan.
// Every step reads and writes HBM in coalesced streams; the only random
// accesses of the whole database life are the lookups of the query path.
#include <atomic>
#include <cstdio>
#include <vector>

#include "mc_internal.h"
#include "mc_sketch.cuh"

namespace mc {

namespace {

constexpr int BT = 256;  // threads of the streaming kernels
constexpr int NWARP = BT / 32;

inline uint32_t grid_for(uint64_t tiles, uint32_t per_sm = 8) {
    uint64_t g = (uint64_t)NUM_SMS_HINT * per_sm;
    if (tiles < g) g = tiles;
    return (uint32_t)(g ? g : 1);
}

struct OpSum {
    __device__ __forceinline__ uint64_t operator()(uint64_t a, uint64_t b) const { return a + b; }
};
struct OpMaxI {
    __device__ __forceinline__ int64_t operator()(int64_t a, int64_t b) const { return a > b ? a : b; }
};

template <class T, class Op>
__device__ __forceinline__ T warp_inclusive(T v, Op op) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T o = __shfl_up_sync(FULL_MASK, v, d);
        if ((int)lane_id() >= d) v = op(v, o);
    }
    return v;
}

// Block-wide exclusive scan of one value per thread (BT threads).  Returns
// the exclusive prefix; *total receives the block aggregate.  `sm` needs
// NWARP entries.  Contains two __syncthreads.
template <class T, class Op>
__device__ __forceinline__ T block_exclusive(T v, T identity, Op op, T* sm, T* total) {
    T inc = warp_inclusive(v, op);
    const int w = threadIdx.x >> 5;
    const int l = lane_id();
    if (l == 31) sm[w] = inc;
    __syncthreads();
    T warp_pre = identity, tot = identity;
#pragma unroll
    for (int i = 0; i < NWARP; ++i) {
        T x = sm[i];
        if (i < w) warp_pre = op(warp_pre, x);
        tot = op(tot, x);
    }
    T ex = __shfl_up_sync(FULL_MASK, inc, 1);
    if (l == 0) ex = identity;
    *total = tot;
    __syncthreads();
    return op(warp_pre, ex);
}

template <class T, class Op>
__device__ __forceinline__ T block_reduce(T v, T identity, Op op, T* sm) {
    T tot;
    block_exclusive(v, identity, op, sm, &tot);
    return tot;
}

// ------------------------------------------------------------------ scan
constexpr int SCAN_ITEMS = 8;
constexpr uint64_t SCAN_TILE = (uint64_t)BT * SCAN_ITEMS;

__global__ void __launch_bounds__(BT) k_scan_tile_sums(const uint64_t* __restrict__ in, uint64_t n,
                                                       uint64_t* __restrict__ sums, uint64_t n_tiles) {
    __shared__ uint64_t sm[NWARP];
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        uint64_t base = tile * SCAN_TILE, acc = 0;
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) {
            uint64_t e = base + (uint64_t)i * BT + threadIdx.x;
            if (e < n) acc += in[e];
        }
        uint64_t tot = block_reduce(acc, (uint64_t)0, OpSum(), sm);
        if (threadIdx.x == 0) sums[tile] = tot;
    }
}

// Exclusive scan of each tile with its prefix (tile_pre, or 0 if null).
// The element of round i, thread t is base + i*BT + t (sequential order).
__global__ void __launch_bounds__(BT) k_scan_downsweep(const uint64_t* in, uint64_t* out, uint64_t n,
                                                       const uint64_t* __restrict__ tile_pre, uint64_t n_tiles,
                                                       uint64_t* total) {
    __shared__ uint64_t sm[NWARP];
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        uint64_t base = tile * SCAN_TILE;
        uint64_t carry = tile_pre ? tile_pre[tile] : 0;
        for (int i = 0; i < SCAN_ITEMS; ++i) {
            uint64_t e = base + (uint64_t)i * BT + threadIdx.x;
            uint64_t v = e < n ? in[e] : 0;
            uint64_t tot;
            uint64_t ex = block_exclusive(v, (uint64_t)0, OpSum(), sm, &tot);
            if (e < n) out[e] = carry + ex;
            carry += tot;
        }
        if (tile == n_tiles - 1 && threadIdx.x == 0 && total) *total = carry;
    }
}

}  // namespace

cudaError_t scan_exclusive_sum(const Mem& mem, const uint64_t* in, uint64_t* out, uint64_t n, cudaStream_t s) {
    if (n == 0) return cudaMemsetAsync(out, 0, sizeof(uint64_t), s);
    uint64_t n_tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (n_tiles == 1) {
        MC_LAUNCH("scan_downsweep", s, k_scan_downsweep<<<1, BT, 0, s>>>(in, out, n, nullptr, 1, out + n));
        return cudaGetLastError();
    }
    Tmp<uint64_t> sums(mem, n_tiles + 1, s);
    if (!sums.ok()) return cudaErrorMemoryAllocation;
    MC_LAUNCH("scan_tile_sums", s, k_scan_tile_sums<<<grid_for(n_tiles), BT, 0, s>>>(in, n, sums.ptr, n_tiles));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = scan_exclusive_sum(mem, sums.ptr, sums.ptr, n_tiles, s);
    if (e != cudaSuccess) return e;
    MC_LAUNCH("scan_downsweep", s, k_scan_downsweep<<<grid_for(n_tiles), BT, 0, s>>>(in, out, n, sums.ptr, n_tiles, out + n));
    return cudaGetLastError();
}

// ------------------------------------------------------ window offsets
namespace {
__global__ void k_window_counts(const uint64_t* __restrict__ offs, uint32_t n, uint32_t k, uint32_t stride,
                                uint64_t* __restrict__ cnt, uint32_t* bad) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t a = offs[i], b = offs[i + 1];
        if (b < a) {
            atomicMax(bad, 1u);
            cnt[i] = 0;
        } else {
            cnt[i] = num_windows(b - a, k, stride);
        }
    }
}
}  // namespace

cudaError_t window_offsets(const Mem& mem, const SketchParams& p, uint32_t n_seq, const uint64_t* offs,
                           uint64_t* win_offs, uint32_t* bad_offs, cudaStream_t s) {
    if (n_seq > 0) {
        MC_LAUNCH("window_counts", s, k_window_counts<<<grid_for((n_seq + BT - 1) / BT), BT, 0, s>>>(offs, n_seq, p.k, p.stride, win_offs,
                                                                         bad_offs));
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return scan_exclusive_sum(mem, win_offs, win_offs, n_seq, s);
}

// ---------------------------------------------------------------- sketch
namespace {
constexpr uint32_t WINDOWS_PER_TASK = 16;
constexpr int SK_NW = 2;  // windows sketched together by a warp

// One warp per window (sketch sizes above 16, which lane_sketch does not
// take, and k-mers so short that they repeat); a warp takes
// WINDOWS_PER_TASK consecutive windows and walks the sequences they belong
// to.  EMIT = build pairs, else the debug sketch export.  Five resident
// blocks per SM (48 registers).
template <int R, int KC, bool EMIT>
__global__ void __launch_bounds__(BT, 5) k_sketch(SketchParams p, uint32_t n_seq, const uint8_t* __restrict__ seq,
                                               const uint64_t* __restrict__ offs,
                                               const uint64_t* __restrict__ win_offs, uint64_t n_windows,
                                               uint32_t gw_base, uint64_t* __restrict__ pairs,
                                               uint32_t* __restrict__ sketch, uint32_t* __restrict__ counts,
                                               unsigned long long* real_pairs) {
    __shared__ uint32_t cand_sm[NWARP][SK_NW * 32];
    const uint32_t lane = lane_id();
    uint32_t* cand = cand_sm[threadIdx.x >> 5];
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t n_tasks = (n_windows + WINDOWS_PER_TASK - 1) / WINDOWS_PER_TASK;
    unsigned long long real = 0;
    for (uint64_t task = warp; task < n_tasks; task += n_warps) {
        uint64_t w0 = task * WINDOWS_PER_TASK;
        uint64_t w1 = min(w0 + WINDOWS_PER_TASK, n_windows);
        // sequence of w0: last i with win_offs[i] <= w0
        uint32_t lo = 0, hi = n_seq;  // invariant: win_offs[lo] <= w0 < win_offs[hi]
        while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (win_offs[mid] <= w0) lo = mid; else hi = mid;
        }
        uint32_t t = lo;
        for (uint64_t lw = w0; lw < w1; lw += SK_NW) {
            const uint8_t* sq[SK_NW];
            uint64_t Ls[SK_NW], wss[SK_NW];
            bool act[SK_NW];
#pragma unroll
            for (int i = 0; i < SK_NW; ++i) {
                const uint64_t x = lw + i;
                act[i] = x < w1;
                if (act[i]) {
                    while (win_offs[t + 1] <= x) ++t;
                    sq[i] = seq + offs[t];
                    Ls[i] = offs[t + 1] - offs[t];
                    wss[i] = (x - win_offs[t]) * p.stride;
                } else {
                    sq[i] = seq;
                    Ls[i] = 0;
                    wss[i] = 0;
                }
            }
            uint32_t f[SK_NW], cnt[SK_NW];
            warp_sketch_multi<R, SK_NW, KC>(sq, Ls, wss, act, p, cand, f, cnt);
#pragma unroll
            for (int i = 0; i < SK_NW; ++i) {
                if (!act[i]) continue;
                const uint64_t x = lw + i;
                if (EMIT) {
                    if (lane < p.s) {
                        uint64_t v = lane < cnt[i] ? (((uint64_t)hash_h2(f[i]) << 32) | (uint32_t)(gw_base + x))
                                                   : SENTINEL_PAIR;
                        pairs[x * p.s + lane] = v;
                    }
                    real += cnt[i];
                } else {
                    if (lane < p.s) sketch[x * p.s + lane] = lane < cnt[i] ? f[i] : 0u;
                    if (lane == 0) counts[x] = cnt[i];
                }
            }
        }
    }
    if (EMIT && lane == 0 && real) atomicAdd(real_pairs, real);
}

// The same work with one window per lane (lane_sketch, sketch sizes up to
// 16): a warp takes 32 consecutive windows at a time, stages the bases they
// cover as 2-bit codes in shared memory (each base loaded and encoded once,
// 16 bytes a lane), sketches them together and writes their pairs, which are
// consecutive in memory, through shared memory with whole-line stores.
// Windows of consecutive targets are in memory order too; should targets too
// short for a window lie between them and spread the 32 windows over more
// bytes than the staging area holds, the windows that fit are taken first.
// A window that lane_sketch does not settle is sketched by the whole warp, and
// where more than EMIT_LANE_EXACT of the 32 are left, those by their lanes
// (lane_sketch_exact).
// Bound by the integer ALU (74-80% busy, half the issue rate; 118 warp
// instructions per window): 14.3 Gbp of the large workload take 20.5 ms (127 M
// windows of 113 k-mers), against 64.5 ms with one warp per window.  Six CTAs
// per SM: 5% and 15% faster than five and four.
constexpr uint32_t EMIT_CAP = 48;  // candidates per lane
constexpr int EMIT_LANE_EXACT = 12;  // (by their lanes, 32 cost what 8 to 17 do one by one)
__host__ __device__ constexpr uint32_t emit_stage_words(const SketchParams& p) {
    return (31 * p.stride + p.w + 30) / 16 + 2;
}
__host__ __device__ constexpr size_t emit_warp_bytes(const SketchParams& p) {
    const size_t words = emit_stage_words(p);
    return words * 4 + ((words * 2 + 3) & ~(size_t)3) + ls_cand_words(EMIT_CAP) * 4;
}
// The parameters that need most: windows of 512 bases without overlap.
constexpr SketchParams EMIT_LARGEST{1, LS_MAX_S, 512, 512};
constexpr int EMIT_WARPS = 4;
constexpr int EMIT_CTAS = 6;  // resident per SM: 80 registers, 34 KB of shared memory each

template <int R, int KC, bool EMIT>
__global__ void __launch_bounds__(EMIT_WARPS * 32, EMIT_CTAS)
    k_sketch_lanes(SketchParams p, uint32_t n_seq, const uint8_t* __restrict__ seq, const uint64_t* __restrict__ offs,
                   const uint64_t* __restrict__ win_offs, uint64_t n_windows, uint32_t task_windows, uint32_t gw_base,
                   uint64_t* __restrict__ pairs, uint32_t* __restrict__ sketch, uint32_t* __restrict__ counts,
                   unsigned long long* real_pairs) {
    extern __shared__ __align__(16) unsigned char emit_smem[];
    const uint32_t lane = lane_id();
    const uint32_t n_words = emit_stage_words(p);
    uint32_t* code = reinterpret_cast<uint32_t*>(emit_smem + (threadIdx.x >> 5) * emit_warp_bytes(p));
    uint32_t* cand = code + n_words;  // candidates, then the features
    uint16_t* inv = reinterpret_cast<uint16_t*>(cand + ls_cand_words(EMIT_CAP));
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t k = KC ? (uint32_t)KC : p.k;
    unsigned long long real = 0;
    for (uint64_t w0 = warp * task_windows; w0 < n_windows; w0 += n_warps * task_windows) {
        const uint64_t w1 = min(w0 + task_windows, n_windows);
        uint32_t t = 0;  // last target with win_offs[t] <= the round's first window
        {
            uint32_t hi = n_seq;
            while (hi - t > 1) {
                const uint32_t mid = (t + hi) >> 1;
                if (win_offs[mid] <= w0) t = mid; else hi = mid;
            }
        }
        for (uint64_t x0 = w0; x0 < w1; x0 += 32) {
            const uint64_t x = min(x0 + lane, w1 - 1);
            const bool act = x0 + lane < w1;
            uint32_t tl = t;
            if (win_offs[t + 1] <= min(x0 + 31, w1 - 1)) {  // the round leaves target t
                uint32_t hi = n_seq;
                while (hi - tl > 1) {
                    const uint32_t mid = (tl + hi) >> 1;
                    if (win_offs[mid] <= x) tl = mid; else hi = mid;
                }
            }
            t = __shfl_sync(FULL_MASK, tl, 31);  // a later target or the same for the next round
            const uint64_t L = offs[tl + 1] - offs[tl];
            const uint64_t ws = (x - win_offs[tl]) * p.stride;
            const uint32_t n_k = window_kmers(L, ws, p);
            const uintptr_t first = reinterpret_cast<uintptr_t>(seq) + offs[tl] + ws;
            const uintptr_t end = first + n_k + k - 1;
            uint32_t todo = __ballot_sync(FULL_MASK, act);
            while (todo) {
                // the run of windows from the first one left whose bases fit
                const uint32_t lead = __ffs(todo) - 1;
                const uintptr_t f0 = __shfl_sync(FULL_MASK, first, lead);
                const uintptr_t a0 = f0 & ~(uintptr_t)15;
                const uint32_t fits = __ballot_sync(FULL_MASK, ((todo >> lane) & 1u) && first >= f0 &&
                                                                   end <= a0 + (uintptr_t)(n_words - 1) * 16);
                const uint32_t run = fits >> lead;  // bit 0 is set: one window always fits
                const uint32_t n_now = run == FULL_MASK ? 32u : __ffs(~run) - 1;
                const bool in = lane - lead < n_now;
                todo &= ~((n_now == 32 ? FULL_MASK : (1u << n_now) - 1u) << lead);
                const uint32_t n_ch = (__reduce_max_sync(FULL_MASK, in ? (uint32_t)(end - a0) : 0u) + 15) / 16;
                // bytes outside the targets of these windows are not read
                const uintptr_t lo = reinterpret_cast<uintptr_t>(seq) + __shfl_sync(FULL_MASK, offs[tl], lead);
                const uintptr_t t_end = reinterpret_cast<uintptr_t>(seq) + offs[tl + 1];
                const uintptr_t hi =
                    a0 + __reduce_max_sync(FULL_MASK, in ? (uint32_t)min(t_end - a0, (uintptr_t)0x7FFFFFFF) : 0u);
                __syncwarp();
                uint32_t bad = 0;
                if (a0 >= lo && a0 + 16 * (uintptr_t)n_ch <= hi) {
                    for (uint32_t c = lane; c < n_ch; c += 32) {
                        uint32_t iv;
                        code[c] = encode16(__ldg(reinterpret_cast<const uint4*>(a0) + c), iv);
                        inv[c] = (uint16_t)iv;
                        bad |= iv;
                    }
                } else {
                    for (uint32_t c = lane; c < n_ch; c += 32) {
                        uint32_t iv;
                        code[c] = encode16(load_chunk(a0 + 16 * (uintptr_t)c, lo, hi), iv);
                        inv[c] = (uint16_t)iv;
                        bad |= iv;
                    }
                }
                const bool any_inv = __any_sync(FULL_MASK, bad != 0);
                __syncwarp();
                uint32_t v[16], cnt;
                const bool ok = lane_sketch<KC, EMIT_CAP>(code, inv, n_ch, any_inv, in ? (uint32_t)(first - a0) : 0u,
                                                in ? n_k : 0u, p, cand, v, cnt);
                uint32_t again = __ballot_sync(FULL_MASK, in && !ok);
                __syncwarp();  // the candidates are read: the buffer now takes the features
                uint32_t* feat = cand;
#pragma unroll
                for (int i = 0; i < 16; ++i) feat[i * LS_FEAT_STRIDE + lane] = v[i];
                if (__popc(again) > EMIT_LANE_EXACT) {
                    const bool mine = (again >> lane) & 1u;
                    const uint32_t c = lane_sketch_exact<KC>(code, inv, n_ch, in ? (uint32_t)(first - a0) : 0u,
                                                             mine ? n_k : 0u, k, p.s, feat);
                    if (mine) cnt = c;
                    again = 0;
                }
                while (again) {  // exact selection by the whole warp
                    const uint32_t l = __ffs(again) - 1;
                    again &= again - 1;
                    const uint32_t ta = __shfl_sync(FULL_MASK, tl, l);
                    const uint8_t* const sq[1] = {seq + offs[ta]};
                    const uint64_t Ls[1] = {__shfl_sync(FULL_MASK, L, l)}, wss[1] = {__shfl_sync(FULL_MASK, ws, l)};
                    const bool on[1] = {true};
                    uint32_t f[1], c1[1];
                    __syncwarp();
                    warp_sketch_multi<R, 1, KC>(sq, Ls, wss, on, p, feat + 16 * LS_FEAT_STRIDE, f, c1);
                    if (lane < c1[0]) feat[lane * LS_FEAT_STRIDE + l] = f[0];
                    if (lane == l) cnt = c1[0];
                }
                __syncwarp();
                if (!in) cnt = 0;
                real += cnt;
                if (!EMIT && in) counts[x] = cnt;
                // entry e of the round's n_now * s outputs: feature e % s of window e / s
                const uint64_t out0 = (x0 + lead) * p.s;
                for (uint32_t e0 = 0; e0 < n_now * p.s; e0 += 32) {
                    const uint32_t e = e0 + lane;
                    const uint32_t wl = p.s == 16 ? e >> 4 : e / p.s;
                    const uint32_t i = e - wl * p.s;
                    const uint32_t src = (lead + wl) & 31u;
                    const uint32_t c = __shfl_sync(FULL_MASK, cnt, src);
                    if (wl < n_now) {
                        const uint32_t fv = feat[i * LS_FEAT_STRIDE + src];
                        if (EMIT)
                            pairs[out0 + e] = i < c ? (((uint64_t)hash_h2(fv) << 32) |
                                                       (uint32_t)(gw_base + x0 + lead + wl))
                                                    : SENTINEL_PAIR;
                        else
                            sketch[out0 + e] = i < c ? fv : 0u;
                    }
                }
                __syncwarp();
            }
        }
    }
    if (EMIT) {
        for (int o = 16; o >= 1; o >>= 1) real += __shfl_xor_sync(FULL_MASK, real, o);
        if (lane == 0 && real) atomicAdd(real_pairs, real);
    }
}

template <bool EMIT>
cudaError_t launch_sketch(const SketchParams& p, uint32_t n_seq, const uint8_t* seq, const uint64_t* offs,
                          const uint64_t* win_offs, uint64_t n_windows, uint32_t gw_base, uint64_t* pairs,
                          uint32_t* sketch, uint32_t* counts, unsigned long long* real, cudaStream_t s) {
    if (n_windows == 0) return cudaSuccess;
    const int r = sketch_r_for(p.w);
    const char* name = EMIT ? "sketch_emit" : "sketch";
    // Where a window's smallest hashes mostly repeat, as of 4^k / 2 canonical
    // k-mers a window of n holds s n / (4^k / 2) repeats of one of its s
    // smallest, most windows need the exact selection, and the kernel that
    // makes no other is faster (k = 4, 64 Mbp: 339 us, 410 with lanes).
    const bool repeats = 4ull * p.s * (p.w - p.k + 1) > 1ull << (2 * p.k);
    if (p.s <= LS_MAX_S && !repeats) {
        using Kernel = void (*)(SketchParams, uint32_t, const uint8_t*, const uint64_t*, const uint64_t*, uint64_t,
                                uint32_t, uint32_t, uint64_t*, uint32_t*, uint32_t*, unsigned long long*);
        const bool k16 = p.k == 16;
        const Kernel kern = r == 4   ? (k16 ? k_sketch_lanes<4, 16, EMIT> : k_sketch_lanes<4, 0, EMIT>)
                            : r == 8 ? (k16 ? k_sketch_lanes<8, 16, EMIT> : k_sketch_lanes<8, 0, EMIT>)
                                     : (k16 ? k_sketch_lanes<16, 16, EMIT> : k_sketch_lanes<16, 0, EMIT>);
        const size_t smem = EMIT_WARPS * emit_warp_bytes(p);
        cudaError_t e = allow_smem(kern, EMIT_WARPS * emit_warp_bytes(EMIT_LARGEST));
        if (e != cudaSuccess) return e;
        // rounds of 32 windows per task: 16 where there are windows enough
        // for every resident warp, fewer in small calls
        const uint64_t warps = (uint64_t)NUM_SMS_HINT * EMIT_CTAS * EMIT_WARPS;
        const uint64_t rounds = (n_windows + 32 * warps - 1) / (32 * warps);
        const uint32_t task_windows = 32u * (uint32_t)(rounds < 16 ? rounds : 16);
        const uint64_t tasks = (n_windows + task_windows - 1) / task_windows;
        const uint32_t g = grid_for((tasks + EMIT_WARPS - 1) / EMIT_WARPS, 20);
        MC_LAUNCH(name, s,
                  kern<<<g, EMIT_WARPS * 32, smem, s>>>(p, n_seq, seq, offs, win_offs, n_windows, task_windows,
                                                        gw_base, pairs, sketch, counts, real));
        return cudaGetLastError();
    }
    uint64_t tasks = (n_windows + WINDOWS_PER_TASK - 1) / WINDOWS_PER_TASK;
    uint64_t blocks = (tasks + NWARP - 1) / NWARP;
    uint32_t g = grid_for(blocks, 16);
#define MC_SK(RR, KK) \
    MC_LAUNCH(name, s, k_sketch<RR, KK, EMIT><<<g, BT, 0, s>>>(p, n_seq, seq, offs, win_offs, n_windows, gw_base, pairs, sketch, counts, real))
    if (r == 4) {
        if (p.k == 16) MC_SK(4, 16); else MC_SK(4, 0);
    } else if (r == 8) {
        if (p.k == 16) MC_SK(8, 16); else MC_SK(8, 0);
    } else {
        if (p.k == 16) MC_SK(16, 16); else MC_SK(16, 0);
    }
#undef MC_SK
    return cudaGetLastError();
}
}  // namespace

cudaError_t sketch_windows(const SketchParams& p, uint32_t n_seq, const uint8_t* seq, const uint64_t* offs,
                           const uint64_t* win_offs, uint64_t n_windows, uint32_t* sketch, uint32_t* counts,
                           cudaStream_t s) {
    return launch_sketch<false>(p, n_seq, seq, offs, win_offs, n_windows, 0, nullptr, sketch, counts, nullptr, s);
}

cudaError_t emit_pairs(const SketchParams& p, uint32_t n_targets, const uint8_t* seq, const uint64_t* offs,
                       const uint64_t* win_offs, uint64_t n_windows, uint32_t gw_base, uint64_t* pairs,
                       unsigned long long* real_pairs, cudaStream_t s) {
    return launch_sketch<true>(p, n_targets, seq, offs, win_offs, n_windows, gw_base, pairs, nullptr, nullptr,
                               real_pairs, s);
}

// ------------------------------------------------------------ radix sort
// Single-pass LSD radix sort (one kernel per 8-bit digit; Merrill and
// Garland's decoupled look-back, as in "Onesweep", Adinets and Merrill
// 2022).  One streaming read computes the digit totals of all four passes;
// then every pass reads each pair once and writes it once.  A tile
// (4,096 pairs) ranks its pairs by digit, publishes its per-digit counts,
// looks back over earlier tiles' published counts for its global offsets,
// and writes each digit's run with consecutive threads on consecutive
// addresses.
namespace {
constexpr int RS_ITEMS = 16;
constexpr uint64_t RS_TILE = (uint64_t)BT * RS_ITEMS;  // 4096 pairs
constexpr int RS_BLOCKS_PER_SM = 3;
constexpr int RS_LOOKBACK = 4;  // earlier tiles read per look-back step
// element of (warp w, round i, lane l) in a tile: w*32*RS_ITEMS + i*32 + l

// Look-back status word of (tile, digit): kind (2 bits: 1 = this tile's
// count, 2 = inclusive prefix over tiles 0..tile), pass tag (4 bits: pass +
// 1, so that one zeroing serves all four passes), value (58 bits).
constexpr uint64_t ST_COUNT = 1ull << 62;
constexpr uint64_t ST_PREFIX = 2ull << 62;
constexpr uint64_t ST_VALUE = (1ull << 58) - 1;
constexpr uint64_t LOOKBACK_LIMIT_NS = 2000000000ull;  // a wait longer than this is an error

__device__ __forceinline__ uint64_t ld_relaxed_gpu(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_gpu(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Digit totals of the four passes (sentinels excluded): totals[pass][digit].
__global__ void __launch_bounds__(BT) k_radix_totals(const uint64_t* __restrict__ in, uint64_t n,
                                                     unsigned long long* __restrict__ totals) {
    __shared__ uint32_t sh[NWARP][4][256];
    for (int i = threadIdx.x; i < NWARP * 1024; i += BT) (&sh[0][0][0])[i] = 0;
    __syncthreads();
    const int w = threadIdx.x >> 5;
    const uint64_t stride = (uint64_t)gridDim.x * BT * 4;
    for (uint64_t e0 = (uint64_t)blockIdx.x * BT * 4 + threadIdx.x; e0 < n; e0 += stride) {
        uint64_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint64_t e = e0 + (uint64_t)i * BT;
            v[i] = e < n ? in[e] : SENTINEL_PAIR;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (v[i] == SENTINEL_PAIR) continue;
            const uint32_t k = (uint32_t)(v[i] >> 32);
            atomicAdd(&sh[w][0][k & 255u], 1u);
            atomicAdd(&sh[w][1][(k >> 8) & 255u], 1u);
            atomicAdd(&sh[w][2][(k >> 16) & 255u], 1u);
            atomicAdd(&sh[w][3][k >> 24], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 1024; i += BT) {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < NWARP; ++j) c += (&sh[j][0][0])[i];
        if (c) atomicAdd(totals + i, (unsigned long long)c);
    }
}

// Rank of round i of a warp's 32 pairs: the lanes holding the same digit
// (each lane sets its bit in the digit's word of a per-warp mask table in
// shared memory, then reads the word back; two tables alternate so that a
// table's reset is ordered before its next use by the warp barriers of the
// round in between) and the warp's running count of that digit.  Invalid
// lanes carry digit 256, which is neither counted nor reset.  Bound by shared
// memory (L1 77% busy, issue 51%); peers from eight ballots (60.8 ms for the
// four passes of the large workload, then bound by the ALU) or match.any
// (55.9 ms) are slower than this (45.3 ms).
__device__ __forceinline__ uint32_t rank_round(int i, bool valid, uint32_t d, uint32_t lane, uint32_t lt,
                                               uint32_t* wcount, uint32_t* mask0, uint32_t* mask1) {
    uint32_t* mask = (i & 1) ? mask1 : mask0;
    atomicOr(&mask[d], 1u << lane);
    __syncwarp();
    const uint32_t peers = mask[d];
    __syncwarp();
    const uint32_t rank = __popc(peers & lt);
    const uint32_t leader = (__ffs(peers) - 1) & 31u;
    uint32_t before = 0;
    if (valid && rank == 0) {
        before = atomicAdd(&wcount[d], (uint32_t)__popc(peers));
        mask[d] = 0;
    }
    return __shfl_sync(FULL_MASK, before, leader) + rank;
}

// One pass over digit `pass` (bits 32 + 8 pass ..).  Persistent blocks take
// tiles in order from *tile_ctr, so a tile only ever waits for tiles that
// running blocks hold.  FILTER drops sentinel pairs (first pass).
template <bool FILTER>
__global__ void __launch_bounds__(BT, RS_BLOCKS_PER_SM)
    k_radix_pass(const uint64_t* __restrict__ in, uint64_t* __restrict__ out, uint64_t n, uint32_t pass,
                 const unsigned long long* __restrict__ totals, uint64_t* status, uint32_t* tile_ctr,
                 uint64_t n_tiles, uint64_t limit_ns, uint32_t* err) {
    __shared__ uint32_t wc[NWARP][257];       // per-warp digit counts, then tile offsets
    __shared__ uint32_t peer_mask[2][NWARP][257];
    __shared__ uint64_t gdelta[256];          // global position of a digit's run minus its tile offset
    __shared__ uint64_t staged[RS_TILE];
    __shared__ uint64_t sm[NWARP];
    __shared__ uint32_t s_tile;
    const int w = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    const uint32_t sel = 0x4440u + pass;  // __byte_perm selector of byte `pass` of the key
    const uint64_t tag = (uint64_t)(pass + 1) << 58;
    for (int i = threadIdx.x; i < 2 * NWARP * 257; i += BT) (&peer_mask[0][0][0])[i] = 0;
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1u);
    uint64_t all;
    const uint64_t dbase = block_exclusive((uint64_t)totals[threadIdx.x], (uint64_t)0, OpSum(), sm, &all);
    uint64_t tile = s_tile;
    while (tile < n_tiles) {
        for (int i = threadIdx.x; i < NWARP * 257; i += BT) (&wc[0][0])[i] = 0;
        __syncthreads();
        uint64_t v[RS_ITEMS];
        uint32_t dr[RS_ITEMS];  // digit << 16 | rank within the warp's pairs of that digit
        const uint64_t base = tile * RS_TILE + (uint64_t)w * 32 * RS_ITEMS + lane;
        if ((tile + 1) * RS_TILE <= n) {
#pragma unroll
            for (int i = 0; i < RS_ITEMS; ++i) v[i] = in[base + (uint64_t)i * 32];
#pragma unroll
            for (int i = 0; i < RS_ITEMS; ++i) {
                const bool valid = !FILTER || v[i] != SENTINEL_PAIR;
                const uint32_t d = valid ? __byte_perm((uint32_t)(v[i] >> 32), 0, sel) : 256u;
                dr[i] = (d << 16) | rank_round(i, valid, d, lane, lt, wc[w], peer_mask[0][w], peer_mask[1][w]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < RS_ITEMS; ++i) {
                const uint64_t e = base + (uint64_t)i * 32;
                v[i] = e < n ? in[e] : SENTINEL_PAIR;
            }
#pragma unroll
            for (int i = 0; i < RS_ITEMS; ++i) {
                const bool valid = base + (uint64_t)i * 32 < n && (!FILTER || v[i] != SENTINEL_PAIR);
                const uint32_t d = valid ? __byte_perm((uint32_t)(v[i] >> 32), 0, sel) : 256u;
                dr[i] = (d << 16) | rank_round(i, valid, d, lane, lt, wc[w], peer_mask[0][w], peer_mask[1][w]);
            }
        }
        __syncthreads();
        // thread d: exclusive offsets of digit d over the warps, tile count
        uint32_t run = 0;
#pragma unroll
        for (int i = 0; i < NWARP; ++i) {
            const uint32_t c = wc[i][threadIdx.x];
            wc[i][threadIdx.x] = run;
            run += c;
        }
        // publish, then look back for the count of digit d in earlier tiles
        uint64_t excl = 0;
        uint64_t* mine = status + tile * 256 + threadIdx.x;
        if (tile == 0) {
            st_relaxed_gpu(mine, ST_PREFIX | tag | run);
        } else {
            st_relaxed_gpu(mine, ST_COUNT | tag | run);
            int64_t t = (int64_t)tile - 1;
            uint64_t t0 = 0;
            uint32_t polls = 0;
            while (true) {
                uint64_t st[RS_LOOKBACK];
#pragma unroll
                for (int k = 0; k < RS_LOOKBACK; ++k)
                    st[k] = t - k >= 0 ? ld_relaxed_gpu(status + (uint64_t)(t - k) * 256 + threadIdx.x)
                                       : ST_PREFIX | tag;
                uint32_t used = 0;
                bool stop = false, done = false;
#pragma unroll
                for (int k = 0; k < RS_LOOKBACK; ++k) {
                    if (!stop) {
                        if ((st[k] & (15ull << 58)) != tag || (st[k] >> 62) == 0) {
                            stop = true;  // not published in this pass yet
                        } else {
                            excl += st[k] & ST_VALUE;
                            ++used;
                            if ((st[k] >> 62) == 2) stop = done = true;
                        }
                    }
                }
                if (done) break;
                t -= used;
                if (used == 0 && (++polls & 255u) == 0) {
                    const uint64_t now = globaltimer_ns();
                    if (t0 == 0) {
                        t0 = now;
                    } else if (now - t0 > limit_ns) {
                        atomicMax(err, 1u);
                        break;
                    }
                }
            }
            st_relaxed_gpu(mine, ST_PREFIX | tag | (excl + run));
        }
        uint64_t tot;
        const uint32_t ds = (uint32_t)block_exclusive((uint64_t)run, (uint64_t)0, OpSum(), sm, &tot);
        gdelta[threadIdx.x] = dbase + excl - ds;
#pragma unroll
        for (int i = 0; i < NWARP; ++i) wc[i][threadIdx.x] += ds;
        __syncthreads();
        // stage in digit order, then write each digit's run
#pragma unroll
        for (int i = 0; i < RS_ITEMS; ++i) {
            const uint32_t d = dr[i] >> 16;
            if (d < 256u) staged[wc[w][d] + (dr[i] & 0xFFFFu)] = v[i];
        }
        __syncthreads();
        const uint32_t count = (uint32_t)tot;
        for (uint32_t j = threadIdx.x; j < count; j += BT) {
            const uint64_t x = staged[j];
            out[gdelta[__byte_perm((uint32_t)(x >> 32), 0, sel)] + j] = x;
        }
        if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1u);
        __syncthreads();
        tile = s_tile;
    }
}
// One-shot stall of the next sort's last pass (mc_debug_stall_next_sort):
// the wait limit of that pass in ns, 0 = not armed.
std::atomic<uint64_t> g_stall_limit_ns{0};
}  // namespace

void arm_sort_stall(uint64_t limit_ns) { g_stall_limit_ns.store(limit_ns); }

cudaError_t sort_pairs(const Mem& mem, uint64_t* a, uint64_t* b, uint64_t n_total, uint64_t n_real, cudaStream_t s) {
    if (n_total == 0) return cudaSuccess;
    // An armed stall makes the last pass start at tile 1: tile 0's counts are
    // never published, so tile 1's look-back wait gives up after the armed
    // limit.  Every look-back sum stays a sum over a subset of earlier tiles'
    // counts, so every write stays inside the pass's output; only the last
    // pass is disturbed, because an earlier one would hand the next pass
    // data whose digits disagree with the digit totals.
    const uint64_t stall_ns = g_stall_limit_ns.exchange(0);
    const uint64_t max_tiles = (n_total + RS_TILE - 1) / RS_TILE;
    // control block: totals[4][256], tile counters[4], error word
    constexpr size_t CTRL_WORDS = 4 * 256 + 3;
    Tmp<uint64_t> ctrl(mem, CTRL_WORDS, s);
    Tmp<uint64_t> status(mem, max_tiles * 256, s);
    if (!ctrl.ok() || !status.ok()) return cudaErrorMemoryAllocation;
    unsigned long long* totals = (unsigned long long*)ctrl.ptr;
    uint32_t* tile_ctr = (uint32_t*)(ctrl.ptr + 4 * 256);
    uint32_t* err = tile_ctr + 4;
    cudaError_t e = cudaMemsetAsync(ctrl.ptr, 0, CTRL_WORDS * 8, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(status.ptr, 0, max_tiles * 256 * 8, s);
    if (e != cudaSuccess) return e;
    MC_LAUNCH("radix_totals", s,
              k_radix_totals<<<grid_for((n_total + 4 * BT - 1) / (4 * BT), 4), BT, 0, s>>>(a, n_total, totals));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    uint64_t* src = a;
    uint64_t* dst = b;
    for (uint32_t pass = 0; pass < 4; ++pass) {
        const uint64_t n = pass == 0 ? n_total : n_real;
        if (n == 0) break;
        const uint64_t tiles = (n + RS_TILE - 1) / RS_TILE;
        const uint32_t g = grid_for(tiles, RS_BLOCKS_PER_SM);
        const unsigned long long* tp = totals + 256 * pass;
        uint64_t limit = LOOKBACK_LIMIT_NS;
        if (stall_ns && pass == 3 && tiles >= 2) {
            limit = stall_ns;
            e = cudaMemsetAsync(tile_ctr + pass, 1, 1, s);  // the counter's low byte: tiles are taken from 1
            if (e != cudaSuccess) return e;
        }
        if (pass == 0)
            MC_LAUNCH("radix_pass", s,
                      k_radix_pass<true><<<g, BT, 0, s>>>(src, dst, n, pass, tp, status.ptr, tile_ctr + pass, tiles,
                                                          limit, err));
        else
            MC_LAUNCH("radix_pass", s,
                      k_radix_pass<false><<<g, BT, 0, s>>>(src, dst, n, pass, tp, status.ptr, tile_ctr + pass, tiles,
                                                           limit, err));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        uint64_t* t = src;
        src = dst;
        dst = t;
    }
    // after 4 passes the data is back in `a`; a look-back that gave up
    // leaves a wrong order, which is reported as a timeout
    uint32_t h_err = 0;
    e = cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    return h_err ? cudaErrorTimeout : cudaSuccess;
}

// --------------------------------------------------------------- finalize
namespace {
constexpr int FIN_ITEMS = 8;
constexpr uint64_t FIN_TILE = (uint64_t)BT * FIN_ITEMS;  // warp w: [base + 256 w, base + 256 (w+1))
constexpr uint32_t FIN_BUCKETS = 4096;  // window ranges of the target lookup table
constexpr uint32_t FIN_WB_SMEM_MAX = 12288;  // window bases k_fin_emit keeps in shared memory (48 KiB)

__device__ __forceinline__ uint32_t hk_of(uint64_t v) { return (uint32_t)(v >> 32); }

// In the sorted pair array, e starts a feature's run if its predecessor has
// another feature; e is kept (rank in its run < cap) unless the pair cap
// places earlier has the same feature (runs are contiguous).  Sentinel
// pairs may end a run (the part a sharded build gives up to earlier
// shards, finalize_after): they are neither kept nor starts, and a pair
// after one starts a new run.
__device__ __forceinline__ bool same_feature(uint64_t x, uint32_t hk) {
    return x != SENTINEL_PAIR && hk_of(x) == hk;
}

// The pair, its predecessor and the pair cap places earlier are loaded
// together (each only bounded by the array), so that the loads of all the
// items a thread handles are in flight at once.
__device__ __forceinline__ void fin_flags(const uint64_t* __restrict__ a, uint64_t n, uint32_t cap, uint64_t e,
                                          uint64_t& v, bool& st, bool& kept, bool& over) {
    st = kept = over = false;
    const bool in = e < n;
    v = in ? a[e] : SENTINEL_PAIR;
    const uint64_t prev = (in && e > 0) ? a[e - 1] : SENTINEL_PAIR;
    const uint64_t back = (in && e >= cap) ? a[e - cap] : SENTINEL_PAIR;
    if (!in || v == SENTINEL_PAIR) return;
    const uint32_t hk = hk_of(v);
    st = e == 0 || !same_feature(prev, hk);
    const bool dropped = e >= cap && same_feature(back, hk);
    kept = !dropped;
    // the first dropped pair of an overflowing run: the pair cap earlier starts the run
    over = dropped && (e == cap || !same_feature(a[e - cap - 1], hk));
}

// Tile sums of kept pairs and run starts.
__global__ void __launch_bounds__(BT) k_fin_count(const uint64_t* __restrict__ a, uint64_t n, uint32_t cap,
                                                  uint64_t* __restrict__ tkept, uint64_t* __restrict__ tkeys,
                                                  uint64_t n_tiles) {
    __shared__ uint64_t sm[NWARP];
    const int w = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint64_t base = tile * FIN_TILE + (uint64_t)w * 32 * FIN_ITEMS + lane;
        uint32_t nk = 0, ns = 0;
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            uint64_t v;
            bool st, kept, over;
            fin_flags(a, n, cap, base + (uint64_t)i * 32, v, st, kept, over);
            nk += kept;
            ns += st;
        }
        const uint64_t both = block_reduce(((uint64_t)ns << 32) | nk, (uint64_t)0, OpSum(), sm);
        if (threadIdx.x == 0) {
            tkept[tile] = both & 0xFFFFFFFFull;
            tkeys[tile] = both >> 32;
        }
    }
}

// Writes the condensed outputs at the scanned positions: locations of kept
// pairs (global window -> (target, window), 32-bit target << jbits | window
// when jbits > 0, else 64-bit target << 32 | window), and per feature its h2
// value and the position of its first location.
// The target of a global window gw is the last t with wbase[t] <= gw; a
// block first tabulates that target for the first window of each of
// FIN_BUCKETS equal window ranges, which narrows every search to the
// targets that overlap gw's range (a few for genome-sized targets).  WB:
// wbase (n_targets + 1 words) is copied to shared memory too.
// A thread's items are searched four at a time, one step of each per round,
// so that their reads overlap, and a pair's predecessor comes from the lane
// before it.  Bound by the ALU (70%) and issue (69%), about 130 instructions
// per 32 pairs: large workload 12.9 ms (16.0 with one search after the other
// and whole pairs compared instead of keys), where its bytes, 28 GB, take 4.
template <bool WB>
__global__ void __launch_bounds__(BT, 4) k_fin_emit(const uint64_t* __restrict__ a, uint64_t n, uint32_t cap,
                                                    const uint64_t* __restrict__ tkept, const uint64_t* __restrict__ tkeys,
                                                    uint64_t n_tiles, const uint32_t* __restrict__ wbase,
                                                    uint32_t n_targets, uint32_t jbits, void* __restrict__ locs,
                                                    uint32_t* __restrict__ khk, uint64_t* __restrict__ koff,
                                                    unsigned long long* overflow) {
    extern __shared__ uint32_t fin_smem[];
    uint32_t* first_target = fin_smem;  // FIN_BUCKETS + 1 words
    uint32_t* copy = fin_smem + FIN_BUCKETS + 1;
    __shared__ uint32_t wk[NWARP], wsx[NWARP];
    const int w = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    if (WB) {
        for (uint32_t t = threadIdx.x; t <= n_targets; t += BT) copy[t] = wbase[t];
        __syncthreads();
    }
    const auto wb = [&](uint32_t t) { return WB ? copy[t] : __ldg(wbase + t); };
    const uint64_t n_win = wb(n_targets);
    uint32_t bshift = 0;
    while ((n_win >> bshift) >= FIN_BUCKETS) ++bshift;
    for (uint32_t b = threadIdx.x; b <= FIN_BUCKETS; b += BT) {
        const uint64_t x = (uint64_t)b << bshift;
        uint32_t lo = 0, hi = n_targets;  // last t with wb[t] <= x
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (wb(mid) <= x) lo = mid; else hi = mid;
        }
        first_target[b] = lo;
    }
    __syncthreads();
    uint32_t n_over = 0;
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint64_t base = tile * FIN_TILE + (uint64_t)w * 32 * FIN_ITEMS + lane;
        uint64_t v[FIN_ITEMS];
        uint32_t back[FIN_ITEMS];  // key of the pair cap places earlier
        const uint32_t* keys = reinterpret_cast<const uint32_t*>(a) + 1;  // key of pair e at keys[2 e]
        const uint64_t lead = base - lane;
        const bool deep = lead >= cap;  // every item has a pair cap places earlier
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            const uint64_t e = base + (uint64_t)i * 32;
            v[i] = e < n ? a[e] : SENTINEL_PAIR;
            back[i] = e < n && (deep || e >= cap) ? keys[2 * (e - cap)] : 0u;
        }
        // As fin_flags, on the keys alone (32 bits), with the predecessor from
        // the neighbouring lane.  A sentinel's key is all ones, which a
        // feature may have too: those look at the whole pair.
        uint32_t before = lead > 0 && lead - 1 < n ? keys[2 * (lead - 1)] : 0u;
        uint32_t bk[FIN_ITEMS], bs[FIN_ITEMS];  // ballots: kept, run start
        uint32_t nk = 0, ns = 0;
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            const uint64_t e = base + (uint64_t)i * 32;
            const uint32_t hk = hk_of(v[i]);
            uint32_t prev = __shfl_up_sync(FULL_MASK, hk, 1);
            if (lane == 0) prev = before;
            before = __shfl_sync(FULL_MASK, hk, 31);
            bool real = true, st = e == 0 || prev != hk, dropped = (deep || e >= cap) && back[i] == hk;
            if (hk == 0xFFFFFFFFu) {
                real = v[i] != SENTINEL_PAIR;
                st = real && (e == 0 || !same_feature(a[e - 1], hk));
                dropped = real && e >= cap && same_feature(a[e - cap], hk);
            }
            // the first dropped pair of an overflowing run: the pair cap earlier starts the run
            if (dropped && (e == cap || !same_feature(a[e - cap - 1], hk))) ++n_over;
            bk[i] = __ballot_sync(FULL_MASK, real && !dropped);
            bs[i] = __ballot_sync(FULL_MASK, st);
            nk += __popc(bk[i]);
            ns += __popc(bs[i]);
        }
        if (lane == 0) {
            wk[w] = nk;
            wsx[w] = ns;
        }
        __syncthreads();
        uint64_t kpos = tkept[tile], kidx = tkeys[tile];
        for (int i = 0; i < w; ++i) {
            kpos += wk[i];
            kidx += wsx[i];
        }
        __syncthreads();
        uint32_t n_k = 0, n_s = 0;
#pragma unroll
        for (int i0 = 0; i0 < FIN_ITEMS; i0 += 4) {
            uint32_t lo[4], hi[4];
            bool open = false;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // (a sentinel or dropped pair searches too, in bounds; its result is not used)
                const uint32_t rng = min((uint32_t)v[i0 + u] >> bshift, FIN_BUCKETS - 1);
                lo[u] = first_target[rng];  // last t with wb[t] <= gw lies in [lo, hi)
                hi[u] = min(first_target[rng + 1] + 1, n_targets);
                open |= hi[u] - lo[u] > 1;
            }
            while (__any_sync(FULL_MASK, open)) {
                open = false;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (hi[u] - lo[u] > 1) {
                        const uint32_t mid = (lo[u] + hi[u]) >> 1;
                        if (wb(mid) <= (uint32_t)v[i0 + u]) lo[u] = mid; else hi[u] = mid;
                        open |= hi[u] - lo[u] > 1;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u;
                const uint32_t my_k = n_k + __popc(bk[i] & lt);  // within the warp's pairs
                if ((bk[i] >> lane) & 1u) {
                    const uint32_t off = (uint32_t)v[i] - wb(lo[u]);
                    if (jbits)
                        (static_cast<uint32_t*>(locs) + kpos)[my_k] = (lo[u] << jbits) | off;
                    else
                        (static_cast<uint64_t*>(locs) + kpos)[my_k] = ((uint64_t)lo[u] << 32) | off;
                }
                if ((bs[i] >> lane) & 1u) {
                    const uint32_t my_s = n_s + __popc(bs[i] & lt);
                    (khk + kidx)[my_s] = hk_of(v[i]);
                    (koff + kidx)[my_s] = kpos + my_k;
                }
                n_k += __popc(bk[i]);
                n_s += __popc(bs[i]);
            }
        }
    }
    n_over = __reduce_add_sync(FULL_MASK, n_over);
    if (lane == 0 && n_over) atomicAdd(overflow, (unsigned long long)n_over);
}

// Pairs (h2 << 32 | global window) of a finalized layout, in layout order:
// the input of the next finalize after an extension.
__global__ void k_reconstruct_pairs(const uint64_t* __restrict__ table, uint64_t table_len, TableFmt fmt,
                                    const void* __restrict__ locs, uint32_t jbits,
                                    const uint32_t* __restrict__ wbase, uint64_t* __restrict__ out) {
    const uint32_t jmask = jbits ? (1u << jbits) - 1u : 0u;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < table_len;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t e = table[i];
        if (e == 0) continue;
        const uint64_t off = fmt.offset(e);
        const uint32_t cnt = fmt.count(e);
        const uint64_t hk = (uint64_t)fmt.key(e, i) << 32;
        for (uint32_t j = 0; j < cnt; ++j) {
            uint32_t t, w;
            if (jbits) {
                const uint32_t x = static_cast<const uint32_t*>(locs)[off + j];
                t = x >> jbits;
                w = x & jmask;
            } else {
                const uint64_t x = static_cast<const uint64_t*>(locs)[off + j];
                t = (uint32_t)(x >> 32);
                w = (uint32_t)x;
            }
            out[off + j] = hk | (uint32_t)(wbase[t] + w);
        }
    }
}

// Exclusive max-scan of the tile maxima (one block; the tiles are few).
__global__ void __launch_bounds__(BT) k_exclusive_max_i64(const int64_t* __restrict__ in, int64_t* __restrict__ out,
                                                          uint64_t n, int64_t* total) {
    __shared__ int64_t sm[NWARP];
    int64_t carry = INT64_MIN;
    for (uint64_t base = 0; base < n; base += BT * 8) {
        const uint64_t e0 = base + threadIdx.x * 8;
        int64_t v[8], m = INT64_MIN;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] = e0 + i < n ? in[e0 + i] : INT64_MIN;
            m = max(m, v[i]);
        }
        int64_t tot;
        int64_t ex = max(carry, block_exclusive(m, (int64_t)INT64_MIN, OpMaxI(), sm, &tot));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (e0 + i < n) out[e0 + i] = ex;
            ex = max(ex, v[i]);
        }
        carry = max(carry, tot);
    }
    if (threadIdx.x == 0) *total = carry;
}

__device__ __forceinline__ uint64_t home_slot(uint32_t hk, uint32_t log_t) {
    return log_t >= 32 ? hk : (hk >> (32 - log_t));
}

// Tile maxima of home(k) - k.
__global__ void __launch_bounds__(BT) k_tab_dispmax(const uint32_t* __restrict__ khk, uint64_t n, uint32_t log_t,
                                                    int64_t* __restrict__ tmax, uint64_t n_tiles) {
    __shared__ int64_t sm[NWARP];
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        uint64_t base = tile * FIN_TILE;
        int64_t m = INT64_MIN;
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            uint64_t e = base + (uint64_t)i * BT + threadIdx.x;
            if (e < n) m = max(m, (int64_t)home_slot(khk[e], log_t) - (int64_t)e);
        }
        int64_t tot = block_reduce(m, (int64_t)INT64_MIN, OpMaxI(), sm);
        if (threadIdx.x == 0) tmax[tile] = tot;
    }
}

// slot(k) = k + max(prefix, inclusive max of home - k): packs the words
// (count = kept locations, koff[k + 1] - koff[k]) and writes the table.  A
// thread takes eight consecutive keys, so a tile needs one block-wide scan;
// the tile's keys take consecutive slots up to the next tile's first one, and
// the block writes that whole range, empty words included, through shared
// memory with consecutive threads on consecutive words (the table is not
// cleared before): 2.36 ms for the 2^30 slots of the large database, where
// clearing (1.3 ms) and single words in their places took 5.2.  A displacement beyond the word's field sets *too_far (the
// host then retries with a larger table).
constexpr uint32_t TAB_CHUNK = 4096;  // slots staged at a time

__global__ void __launch_bounds__(BT, 3) k_tab_emit(const uint32_t* __restrict__ khk, const uint64_t* __restrict__ koff,
                                                 uint64_t n, TableFmt fmt, const int64_t* __restrict__ tpre, uint64_t n_tiles,
                                                 uint64_t* __restrict__ table, uint64_t table_len,
                                                 unsigned int* max_disp, unsigned int* too_far) {
    __shared__ int64_t sm[NWARP];
    __shared__ __align__(16) uint64_t out[TAB_CHUNK];
    static_assert(FIN_ITEMS == 8, "eight keys per thread");
    uint32_t most = 0;
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint64_t first = tile * FIN_TILE;
        const uint64_t e0 = first + threadIdx.x * FIN_ITEMS;
        uint32_t hk[FIN_ITEMS];
        uint64_t off[FIN_ITEMS + 1];
        if (e0 + FIN_ITEMS <= n) {
            const uint4 x = __ldg(reinterpret_cast<const uint4*>(khk + e0));
            const uint4 y = __ldg(reinterpret_cast<const uint4*>(khk + e0) + 1);
            hk[0] = x.x, hk[1] = x.y, hk[2] = x.z, hk[3] = x.w;
            hk[4] = y.x, hk[5] = y.y, hk[6] = y.z, hk[7] = y.w;
#pragma unroll
            for (int i = 0; i < FIN_ITEMS; i += 2) {
                const ulonglong2 z = __ldg(reinterpret_cast<const ulonglong2*>(koff + e0 + i));
                off[i] = z.x;
                off[i + 1] = z.y;
            }
            off[FIN_ITEMS] = koff[e0 + FIN_ITEMS];
        } else {
#pragma unroll
            for (int i = 0; i < FIN_ITEMS; ++i) hk[i] = e0 + i < n ? khk[e0 + i] : 0u;
#pragma unroll
            for (int i = 0; i <= FIN_ITEMS; ++i) off[i] = e0 + i <= n ? koff[e0 + i] : 0u;
        }
        int64_t m = INT64_MIN;
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i)
            if (e0 + i < n) m = max(m, (int64_t)fmt.home(hk[i]) - (int64_t)(e0 + i));
        int64_t tot;
        int64_t run = max(tpre[tile], block_exclusive(m, (int64_t)INT64_MIN, OpMaxI(), sm, &tot));
        uint64_t slot[FIN_ITEMS], word[FIN_ITEMS];
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            const uint64_t home = fmt.home(hk[i]);
            const bool in = e0 + i < n;
            if (in) run = max(run, (int64_t)home - (int64_t)(e0 + i));
            slot[i] = in ? (uint64_t)((int64_t)(e0 + i) + run) : ~0ull;
            const uint64_t disp = in ? slot[i] - home : 0;
            if (disp > TAB_MAX_DISP) atomicMax(too_far, 1u);
            most = max(most, (uint32_t)min(disp, (uint64_t)0xFFFFFFFFu));
            word[i] = fmt.pack(off[i], hk[i], (uint32_t)(disp & TAB_MAX_DISP), (uint32_t)(off[i + 1] - off[i]));
        }
        // the tile's slots: from its first key's (or 0) to the next tile's first key's
        const auto first_slot = [&](uint64_t t) -> uint64_t {
            if (t == 0) return 0;
            if (t >= n_tiles) return table_len;
            const uint64_t e = t * FIN_TILE;
            return (uint64_t)((int64_t)e + max(tpre[t], (int64_t)fmt.home(khk[e]) - (int64_t)e));
        };
        const uint64_t s1 = first_slot(tile + 1);
        for (uint64_t s0 = first_slot(tile); s0 < s1; s0 += TAB_CHUNK) {
            for (uint32_t i = threadIdx.x; i < TAB_CHUNK / 2; i += BT)
                reinterpret_cast<ulonglong2*>(out)[i] = make_ulonglong2(0, 0);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < FIN_ITEMS; ++i)
                if (slot[i] - s0 < TAB_CHUNK) out[slot[i] - s0] = word[i];
            __syncthreads();
            const uint32_t len = (uint32_t)min(s1 - s0, (uint64_t)TAB_CHUNK);
            for (uint32_t i = threadIdx.x; i < len; i += BT) table[s0 + i] = out[i];
            __syncthreads();
        }
    }
    most = __reduce_max_sync(FULL_MASK, most);
    if (lane_id() == 0 && most) atomicMax(max_disp, most);
}
}  // namespace

cudaError_t reconstruct_pairs(const uint64_t* table, uint64_t table_len, TableFmt fmt, const void* locs, uint32_t jbits,
                              const uint32_t* wbase, uint64_t* out, cudaStream_t s) {
    if (table_len == 0) return cudaSuccess;
    MC_LAUNCH("reconstruct_pairs", s,
              k_reconstruct_pairs<<<grid_for((table_len + BT - 1) / BT), BT, 0, s>>>(table, table_len, fmt, locs, jbits,
                                                                                     wbase, out));
    return cudaGetLastError();
}

cudaError_t finalize_pairs(const Mem& mem, const uint64_t* sorted, uint64_t n, uint32_t cap, const uint32_t* wbase,
                           uint32_t n_targets, uint32_t jbits, FinalizeOut* out, cudaStream_t s) {
    cudaError_t e;
    *out = FinalizeOut();
    const uint64_t tiles = (n + FIN_TILE - 1) / FIN_TILE;
    const uint32_t g = grid_for(tiles ? tiles : 1);
    // counters: [0] overflow keys, [1] max displacement (u32 in low word),
    // [2] displacement beyond the word's field
    Tmp<unsigned long long> ctr(mem, 4, s);
    if (!ctr.ok()) return cudaErrorMemoryAllocation;
    if ((e = cudaMemsetAsync(ctr.ptr, 0, 4 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    uint64_t host_tot[2] = {0, 0};
    Tmp<uint64_t> tkept(mem, tiles + 1, s), tkeys(mem, tiles + 1, s);
    if (!tkept.ok() || !tkeys.ok()) return cudaErrorMemoryAllocation;
    if (n > 0) {
        MC_LAUNCH("fin_count", s, k_fin_count<<<g, BT, 0, s>>>(sorted, n, cap, tkept.ptr, tkeys.ptr, tiles));
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = scan_exclusive_sum(mem, tkept.ptr, tkept.ptr, tiles, s)) != cudaSuccess) return e;
        if ((e = scan_exclusive_sum(mem, tkeys.ptr, tkeys.ptr, tiles, s)) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&host_tot[0], tkept.ptr + tiles, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(&host_tot[1], tkeys.ptr + tiles, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    }
    const uint64_t n_kept = host_tot[0], n_keys = host_tot[1];
    // table format: slots = 2^log_t >= 2 n_keys (load factor <= 1/2), and
    // enough offset bits for every location; a larger table is taken when
    // a displacement does not fit the word's field
    TableFmt fmt{1, count_bits(cap)};
    while ((1ull << fmt.log_t) < 2 * n_keys) ++fmt.log_t;
    while (fmt.log_t <= 32 && fmt.obits() < 64 && (n_kept >> fmt.obits()) != 0) ++fmt.log_t;
    if (fmt.log_t > 32) {
        out->table_full = true;
        return cudaSuccess;
    }
    Tmp<unsigned char> locs(mem, n_kept * loc_bytes(jbits), s);
    Tmp<uint64_t> koff(mem, n_keys + 1, s);
    Tmp<uint32_t> khk(mem, n_keys, s);
    if (!locs.ok() || !koff.ok() || !khk.ok()) return cudaErrorMemoryAllocation;
    if (n > 0) {
        // wbase in shared memory when it fits next to the range table
        const bool wb_smem = n_targets + 1 <= FIN_WB_SMEM_MAX;
        const size_t smem = (size_t)(FIN_BUCKETS + 1 + (wb_smem ? n_targets + 1 : 0)) * 4;
        const auto kern = wb_smem ? k_fin_emit<true> : k_fin_emit<false>;
        if ((e = allow_smem(kern, (size_t)(FIN_BUCKETS + 1 + (wb_smem ? FIN_WB_SMEM_MAX : 0)) * 4)) != cudaSuccess) return e;
        MC_LAUNCH("fin_emit", s,
                  kern<<<g, BT, smem, s>>>(sorted, n, cap, tkept.ptr, tkeys.ptr, tiles, wbase, n_targets, jbits,
                                           locs.ptr, khk.ptr, koff.ptr, ctr.ptr));
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = cudaMemcpyAsync(koff.ptr + n_keys, &n_kept, 8, cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    }
    const uint64_t ktiles = (n_keys + FIN_TILE - 1) / FIN_TILE;
    Tmp<int64_t> kt_max(mem, ktiles + 1, s), kt_pre(mem, ktiles + 1, s);
    if (!kt_max.ok() || !kt_pre.ok()) return cudaErrorMemoryAllocation;
    unsigned long long host_ctr[3] = {0, 0, 0};
    for (;;) {
        const uint64_t T = 1ull << fmt.log_t;
        int64_t host_maxa = INT64_MIN;
        if (n_keys > 0) {
            MC_LAUNCH("tab_dispmax", s,
                      k_tab_dispmax<<<grid_for(ktiles), BT, 0, s>>>(khk.ptr, n_keys, fmt.log_t, kt_max.ptr, ktiles));
            MC_LAUNCH("exclusive_max_i64", s,
                      k_exclusive_max_i64<<<1, BT, 0, s>>>(kt_max.ptr, kt_pre.ptr, ktiles, kt_pre.ptr + ktiles));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            if ((e = cudaMemcpyAsync(&host_maxa, kt_pre.ptr + ktiles, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
                return e;
            if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        }
        const uint64_t last_slot = n_keys ? (uint64_t)((int64_t)(n_keys - 1) + host_maxa) : 0;
        // two empty words past the last key or the home slots, rounded to whole 32-byte sectors
        const uint64_t table_len = (((last_slot + 1 > T ? last_slot + 1 : T) + 2) + 3) & ~3ull;
        Tmp<uint64_t> table(mem, table_len, s);
        if (!table.ok()) return cudaErrorMemoryAllocation;
        if (n_keys == 0 && (e = cudaMemsetAsync(table.ptr, 0, table_len * sizeof(uint64_t), s)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(ctr.ptr + 1, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
        if (n_keys > 0) {
            MC_LAUNCH("tab_emit", s,
                      k_tab_emit<<<grid_for(ktiles), BT, 0, s>>>(khk.ptr, koff.ptr, n_keys, fmt, kt_pre.ptr, ktiles,
                                                                 table.ptr, table_len,
                                                                 (unsigned int*)(ctr.ptr + 1),
                                                                 (unsigned int*)(ctr.ptr + 2)));
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        if ((e = cudaMemcpyAsync(host_ctr, ctr.ptr, 24, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        if (host_ctr[2]) {  // a displacement beyond the word's field: twice the slots
            if (++fmt.log_t > 32) {
                out->table_full = true;
                return cudaSuccess;
            }
            continue;
        }
        out->table_len = table_len;
        out->table_bytes = table_len * sizeof(uint64_t);
        out->table = table.release();
        break;
    }
    out->n_keys = n_keys;
    out->n_kept = n_kept;
    out->overflow_keys = host_ctr[0];
    out->max_probe = (uint32_t)(host_ctr[1] & 0xFFFFFFFFull);
    out->fmt = fmt;
    out->locs = locs.release();
    return cudaSuccess;
}

// ------------------------------------------------------------ merge path
// Live extension (Section 4.1: new targets get the next ids): the stored
// pairs (reconstructed in layout order) and the sorted pairs of the new
// targets are two sorted runs; merging them gives the sorted pairs of the
// whole database without sorting the stored ones again.  Merge path
// (Odeh, Green, Mwassi, Shmueli, Birk 2012): a block takes 2,048
// consecutive outputs, takes where that output range starts and ends in
// both inputs (a binary search along the diagonals, k_merge_splits), stages the two input
// slices in shared memory, and each thread merges eight outputs.
namespace {
constexpr int MP_ITEMS = 8;
constexpr uint64_t MP_TILE = (uint64_t)BT * MP_ITEMS;

// Number of elements of a in the first d outputs of merge(a, b), ties
// taken from a first.
__device__ __forceinline__ uint64_t merge_split(const uint64_t* a, uint64_t na, const uint64_t* b, uint64_t nb,
                                                uint64_t d) {
    uint64_t lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (a[mid] <= b[d - mid - 1]) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// split[i] = elements of a in the first min(i * MP_TILE, na + nb) outputs.  A
// kernel of its own, a thread per tile: searched by the merging blocks, a
// tile waited for about 27 dependent reads before it could start (four
// merges of 300 M pairs in all: 3.75 ms, now 0.15 + 1.71).
__global__ void __launch_bounds__(BT) k_merge_splits(const uint64_t* __restrict__ a, uint64_t na,
                                                     const uint64_t* __restrict__ b, uint64_t nb,
                                                     uint64_t* __restrict__ split, uint64_t n_split) {
    for (uint64_t i = blockIdx.x * (uint64_t)BT + threadIdx.x; i < n_split; i += (uint64_t)gridDim.x * BT)
        split[i] = merge_split(a, na, b, nb, min(i * MP_TILE, na + nb));
}

__global__ void __launch_bounds__(BT) k_merge_path(const uint64_t* __restrict__ a, uint64_t na,
                                                   const uint64_t* __restrict__ b, uint64_t nb,
                                                   const uint64_t* __restrict__ splits, uint64_t* __restrict__ c) {
    __shared__ uint64_t in[MP_TILE];
    __shared__ uint64_t out[MP_TILE];
    const uint64_t n = na + nb;
    for (uint64_t d0 = (uint64_t)blockIdx.x * MP_TILE; d0 < n; d0 += (uint64_t)gridDim.x * MP_TILE) {
        const uint64_t d1 = min(d0 + MP_TILE, n);
        const uint64_t i0 = splits[d0 / MP_TILE], i1 = splits[d0 / MP_TILE + 1];
        const uint32_t ta = (uint32_t)(i1 - i0), tb = (uint32_t)((d1 - d0) - ta);
        for (uint32_t k = threadIdx.x; k < ta + tb; k += BT) in[k] = k < ta ? a[i0 + k] : b[(d0 - i0) + (k - ta)];
        __syncthreads();
        const uint64_t* sa = in;
        const uint64_t* sb = in + ta;
        const uint32_t dl = threadIdx.x * MP_ITEMS;
        if (dl < ta + tb) {
            uint32_t lo = dl > tb ? dl - tb : 0, hi = dl < ta ? dl : ta;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (sa[mid] <= sb[dl - mid - 1]) lo = mid + 1; else hi = mid;
            }
            uint32_t ia = lo, ib = dl - lo;
            for (uint32_t k = 0; k < MP_ITEMS && dl + k < ta + tb; ++k) {
                const bool take_a = ib >= tb || (ia < ta && sa[ia] <= sb[ib]);
                out[dl + k] = take_a ? sa[ia++] : sb[ib++];
            }
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < ta + tb; k += BT) c[d0 + k] = out[k];
        __syncthreads();
    }
}
}  // namespace

cudaError_t merge_sorted_pairs(const Mem& mem, const uint64_t* a, uint64_t na, const uint64_t* b, uint64_t nb,
                               uint64_t* c, cudaStream_t s) {
    const uint64_t n = na + nb;
    if (n == 0) return cudaSuccess;
    const uint64_t tiles = (n + MP_TILE - 1) / MP_TILE;
    Tmp<uint64_t> splits(mem, tiles + 1, s);
    if (!splits.ok()) return cudaErrorMemoryAllocation;
    MC_LAUNCH("merge_splits", s,
              k_merge_splits<<<grid_for((tiles + BT) / BT), BT, 0, s>>>(a, na, b, nb, splits.ptr, tiles + 1));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    MC_LAUNCH("merge_path", s, k_merge_path<<<grid_for(tiles, 6), BT, 0, s>>>(a, na, b, nb, splits.ptr, c));
    return cudaGetLastError();
}

// ------------------------------------------------------- sharded builds
// Section 4.3 partitions the reference targets over GPUs.  A shard holds a
// contiguous range of target ids, so every location of an earlier shard is
// smaller than every location of a later one, and the cap smallest
// locations of a feature over all shards are: those of the earlier shards
// first.  A shard therefore keeps at most cap - prior(f) of its own
// locations of feature f, prior(f) = f's locations in the earlier shards
// (clamped to cap), and the union of the shards equals the database of all
// targets.
namespace {

// Run starts of sorted pairs: keys and start indices at the scanned
// positions tkeys (exclusive prefix of each tile's run starts).
__global__ void __launch_bounds__(BT) k_run_emit(const uint64_t* __restrict__ a, uint64_t n,
                                                 const uint64_t* __restrict__ tkeys, uint64_t n_tiles,
                                                 uint32_t* __restrict__ khk, uint64_t* __restrict__ kstart) {
    __shared__ uint32_t wsx[NWARP];
    const int w = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const uint64_t base = tile * FIN_TILE + (uint64_t)w * 32 * FIN_ITEMS + lane;
        uint32_t smask = 0, ns = 0;
        uint64_t v[FIN_ITEMS];
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            bool st, kept, over;
            fin_flags(a, n, 0xFFFFFFFFu, base + (uint64_t)i * 32, v[i], st, kept, over);
            smask |= (st ? 1u : 0u) << i;
            ns += __popc(__ballot_sync(FULL_MASK, st));
        }
        if (lane == 0) wsx[w] = ns;
        __syncthreads();
        uint64_t kidx = tkeys[tile];
        for (int i = 0; i < w; ++i) kidx += wsx[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < FIN_ITEMS; ++i) {
            const bool st = (smask >> i) & 1u;
            const uint32_t bs = __ballot_sync(FULL_MASK, st);
            if (st) {
                const uint64_t my_s = kidx + __popc(bs & lt);
                khk[my_s] = hk_of(v[i]);
                kstart[my_s] = base + (uint64_t)i * 32;
            }
            kidx += __popc(bs);
        }
    }
}

// counts[i] = min(cap, length of run i); kstart has n_runs + 1 entries.
__global__ void k_run_counts(const uint64_t* __restrict__ kstart, uint64_t n_runs, uint32_t cap,
                             uint32_t* __restrict__ counts) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n_runs;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t len = kstart[i + 1] - kstart[i];
        counts[i] = (uint32_t)(len < cap ? len : cap);
    }
}

// One list of earlier shards' feature counts (keys ascending).
struct PriorList {
    const uint32_t* keys;
    const uint32_t* counts;
    uint64_t n;
};

// Per run (thread per run): prior = the run's feature counts in the prior
// lists (binary search in each), limit = max(0, cap - prior); pairs of the
// run beyond the limit become sentinels.  Counts features whose locations
// together with the prior ones exceed cap.
__global__ void k_prior_limits(uint64_t* __restrict__ a, const uint32_t* __restrict__ khk,
                               const uint64_t* __restrict__ kstart, uint64_t n_runs, uint32_t cap,
                               const PriorList* __restrict__ lists, uint32_t n_lists,
                               unsigned long long* overflow) {
    unsigned long long n_over = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n_runs;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t key = khk[i];
        uint64_t prior = 0;
        for (uint32_t l = 0; l < n_lists; ++l) {
            const PriorList L = lists[l];
            uint64_t lo = 0, hi = L.n;  // first index with keys >= key
            while (lo < hi) {
                const uint64_t mid = (lo + hi) >> 1;
                if (L.keys[mid] < key) lo = mid + 1; else hi = mid;
            }
            if (lo < L.n && L.keys[lo] == key) prior += L.counts[lo];
        }
        if (prior == 0) continue;  // the plain cap applies
        const uint64_t len = kstart[i + 1] - kstart[i];
        const uint64_t limit = prior >= cap ? 0 : cap - prior;
        if (prior + len > cap) ++n_over;
        for (uint64_t e = kstart[i] + limit; e < kstart[i] + len; ++e) a[e] = SENTINEL_PAIR;
    }
    for (int o = 16; o >= 1; o >>= 1) n_over += __shfl_xor_sync(FULL_MASK, n_over, o);
    if (lane_id() == 0 && n_over) atomicAdd(overflow, n_over);
}

// Run starts of sorted pairs a[0..n): *n_runs, and (when keys != null and
// the runs fit max) keys[i], kstart[i] (n_runs + 1 entries, kstart[n_runs]
// = n) allocated by the caller.
cudaError_t sorted_runs(const Mem& mem, const uint64_t* a, uint64_t n, uint64_t max, uint32_t* keys,
                        uint64_t* kstart, uint64_t* n_runs, cudaStream_t s) {
    cudaError_t e;
    *n_runs = 0;
    if (n == 0) return cudaSuccess;
    const uint64_t tiles = (n + FIN_TILE - 1) / FIN_TILE;
    Tmp<uint64_t> tkept(mem, tiles + 1, s), tkeys(mem, tiles + 1, s);
    if (!tkept.ok() || !tkeys.ok()) return cudaErrorMemoryAllocation;
    MC_LAUNCH("fin_count", s, k_fin_count<<<grid_for(tiles), BT, 0, s>>>(a, n, 0xFFFFFFFFu, tkept.ptr, tkeys.ptr, tiles));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = scan_exclusive_sum(mem, tkeys.ptr, tkeys.ptr, tiles, s)) != cudaSuccess) return e;
    uint64_t total = 0;
    if ((e = cudaMemcpyAsync(&total, tkeys.ptr + tiles, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    *n_runs = total;
    if (!keys || total > max) return cudaSuccess;
    MC_LAUNCH("run_emit", s, k_run_emit<<<grid_for(tiles), BT, 0, s>>>(a, n, tkeys.ptr, tiles, keys, kstart));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaMemcpyAsync(kstart + total, &n, 8, cudaMemcpyHostToDevice, s);
}
}  // namespace

cudaError_t feature_counts(const Mem& mem, const uint64_t* a, uint64_t n, uint32_t cap, uint64_t max, uint32_t* keys,
                           uint32_t* counts, uint64_t* n_keys, cudaStream_t s) {
    uint64_t runs = 0;
    cudaError_t e = sorted_runs(mem, a, n, 0, nullptr, nullptr, &runs, s);
    *n_keys = runs;
    if (e != cudaSuccess || runs == 0 || runs > max || !keys || !counts) return e;
    Tmp<uint64_t> kstart(mem, runs + 1, s);
    if (!kstart.ok()) return cudaErrorMemoryAllocation;
    uint64_t again = 0;
    if ((e = sorted_runs(mem, a, n, runs, keys, kstart.ptr, &again, s)) != cudaSuccess) return e;
    MC_LAUNCH("run_counts", s,
              k_run_counts<<<grid_for((runs + BT - 1) / BT), BT, 0, s>>>(kstart.ptr, runs, cap, counts));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

cudaError_t apply_prior(const Mem& mem, uint64_t* a, uint64_t n, uint32_t cap, uint32_t n_lists,
                        const uint32_t* const* keys, const uint32_t* const* counts, const uint64_t* list_n,
                        uint64_t* overflow, cudaStream_t s) {
    cudaError_t e;
    *overflow = 0;
    if (n == 0 || n_lists == 0) return cudaSuccess;
    uint64_t runs = 0;
    if ((e = sorted_runs(mem, a, n, 0, nullptr, nullptr, &runs, s)) != cudaSuccess) return e;
    Tmp<uint32_t> khk(mem, runs, s);
    Tmp<uint64_t> kstart(mem, runs + 1, s);
    Tmp<PriorList> dl(mem, n_lists, s);
    Tmp<unsigned long long> ctr(mem, 1, s);
    if (!khk.ok() || !kstart.ok() || !dl.ok() || !ctr.ok()) return cudaErrorMemoryAllocation;
    std::vector<PriorList> hl(n_lists);
    for (uint32_t l = 0; l < n_lists; ++l) hl[l] = PriorList{keys[l], counts[l], list_n[l]};
    uint64_t again = 0;
    if ((e = sorted_runs(mem, a, n, runs, khk.ptr, kstart.ptr, &again, s)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(dl.ptr, hl.data(), n_lists * sizeof(PriorList), cudaMemcpyHostToDevice, s)) !=
        cudaSuccess)
        return e;
    if ((e = cudaMemsetAsync(ctr.ptr, 0, 8, s)) != cudaSuccess) return e;
    MC_LAUNCH("prior_limits", s,
              k_prior_limits<<<grid_for((runs + BT - 1) / BT), BT, 0, s>>>(a, khk.ptr, kstart.ptr, runs, cap, dl.ptr,
                                                                           n_lists, ctr.ptr));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    unsigned long long h = 0;
    if ((e = cudaMemcpyAsync(&h, ctr.ptr, 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    *overflow = h;
    return cudaSuccess;
}

// -------------------------------------------------------------- taxonomy
namespace {
__global__ void k_tax_depth(const uint32_t* __restrict__ parent, uint32_t n, uint32_t* __restrict__ depth,
                            uint32_t* max_depth, uint32_t* cycle) {
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        uint32_t d = 0, y = x;
        while (parent[y] != y) {
            y = parent[y];
            if (++d > n) {
                atomicMax(cycle, 1u);
                d = 0;
                break;
            }
        }
        depth[x] = d;
        atomicMax(max_depth, d);
    }
}

__global__ void k_tax_lineage(const uint32_t* __restrict__ parent, uint32_t n, const uint32_t* __restrict__ depth,
                              uint32_t* __restrict__ lin, uint32_t stride) {
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        uint32_t y = x;
        for (int64_t d = depth[x]; d >= 0; --d) {
            lin[(uint64_t)x * stride + d] = y;
            y = parent[y];
        }
    }
}
}  // namespace

cudaError_t taxonomy_depths(const uint32_t* parent, uint32_t n_taxa, uint32_t* depth, uint32_t* max_depth,
                            uint32_t* cycle_flag, cudaStream_t s) {
    MC_LAUNCH("tax_depth", s, k_tax_depth<<<grid_for((n_taxa + BT - 1) / BT), BT, 0, s>>>(parent, n_taxa, depth, max_depth, cycle_flag));
    return cudaGetLastError();
}

cudaError_t taxonomy_lineage(const uint32_t* parent, uint32_t n_taxa, const uint32_t* depth, uint32_t* lin,
                             uint32_t stride, cudaStream_t s) {
    MC_LAUNCH("tax_lineage", s, k_tax_lineage<<<grid_for((n_taxa + BT - 1) / BT), BT, 0, s>>>(parent, n_taxa, depth, lin, stride));
    return cudaGetLastError();
}

// ------------------------------------------------------------------ dump
namespace {
__global__ void k_dump_select(const uint64_t* __restrict__ table, uint64_t len, TableFmt fmt, uint64_t lo,
                              uint64_t hi, uint32_t* keys, uint64_t* offs, uint32_t* counts, uint64_t cap,
                              unsigned long long* n_sel) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < len; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t e = table[i];
        if (e == 0) continue;
        uint64_t key = hash_h2_inverse(fmt.key(e, i));
        if (key < lo || key >= hi) continue;
        unsigned long long idx = atomicAdd(n_sel, 1ull);
        if (idx < cap) {
            keys[idx] = (uint32_t)key;
            offs[idx] = fmt.offset(e);
            counts[idx] = fmt.count(e);
        }
    }
}

__global__ void k_dump_gather(const void* __restrict__ locs, uint32_t jbits, const uint64_t* __restrict__ src_off,
                              const uint32_t* __restrict__ counts, const uint64_t* __restrict__ dst_off, uint64_t n,
                              uint64_t* __restrict__ out) {
    for (uint64_t i = blockIdx.x; i < n; i += gridDim.x)
        for (uint32_t j = threadIdx.x; j < counts[i]; j += blockDim.x) {
            uint64_t v;
            if (jbits) {
                const uint32_t x = static_cast<const uint32_t*>(locs)[src_off[i] + j];
                v = ((uint64_t)(x >> jbits) << 32) | (x & ((1u << jbits) - 1u));
            } else {
                v = static_cast<const uint64_t*>(locs)[src_off[i] + j];
            }
            out[dst_off[i] + j] = v;
        }
}
}  // namespace

cudaError_t dump_select(const uint64_t* table, uint64_t table_len, TableFmt fmt, uint64_t lo, uint64_t hi,
                        uint32_t* keys, uint64_t* offs, uint32_t* counts, uint64_t cap, unsigned long long* n_sel,
                        cudaStream_t s) {
    if (table_len == 0) return cudaSuccess;
    MC_LAUNCH("dump_select", s,
              k_dump_select<<<grid_for((table_len + BT - 1) / BT), BT, 0, s>>>(table, table_len, fmt, lo, hi, keys,
                                                                               offs, counts, cap, n_sel));
    return cudaGetLastError();
}

cudaError_t dump_gather(const void* locs, uint32_t jbits, const uint64_t* src_off, const uint32_t* counts,
                        const uint64_t* dst_off, uint64_t n, uint64_t* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    MC_LAUNCH("dump_gather", s,
              k_dump_gather<<<grid_for(n, 32), 128, 0, s>>>(locs, jbits, src_off, counts, dst_off, n, out));
    return cudaGetLastError();
}

}  // namespace mc
