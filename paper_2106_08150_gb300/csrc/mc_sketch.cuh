// Warp-cooperative minhash sketch of one window (Section 2, Section 5.2
// steps 1-3, Section 5.3).
//
// One warp computes the sketch of one window of up to 32*R bases:
//  1. lane l loads the R bases at window offsets R*l .. R*l+R-1 and encodes
//     them into 2-bit codes plus an invalid-base mask (Section 5.3: "3-bit"
//     A,C,G,T,N representation);
//  2. the codes of the next E = ceil((k-1)/R) lanes arrive by warp
//     shuffles, so lane l holds the R + E*R bases its k-mers need and forms
//     the k-mers starting at R*l .. R*l+R-1 (Section 5.3 does the same with
//     4-base loads and sub-warp shuffles; here the window start is any base,
//     the stride need not be a multiple of 4);
//  3. canonical code = min(forward, reverse complement), hashed by h1
//     (the reverse complement of all the lane's bases is formed once);
//  4. the s smallest distinct hashes (Section 2: repeated k-mers count
//     once) are selected by a cutoff + warp bitonic sort, with an exact
//     min-reduction fallback (see warp_sketch_multi).
// Lane i (< count) ends up holding the i-th smallest feature.  Several
// windows can be sketched together so that their dependency chains overlap.
#pragma once

#include <type_traits>
#include <utility>

#include "mc_common.cuh"

namespace mc {

template <int R>
__device__ __forceinline__ void sort_small(uint32_t (&h)[R]) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
#pragma unroll
        for (int j = 0; j < R - 1 - i; ++j) {
            uint32_t a = h[j], b = h[j + 1];
            h[j] = min(a, b);
            h[j + 1] = max(a, b);
        }
    }
}

// Number of k-mer starts of the window that starts at `ws` in a sequence
// of length L (the window exists, i.e. ws + k <= L).
__device__ __forceinline__ uint32_t window_kmers(uint64_t L, uint64_t ws, const SketchParams& p) {
    uint64_t last = ws + p.w - p.k;
    if (last > L - p.k) last = L - p.k;
    return (uint32_t)(last - ws + 1);
}

// Encodes 4 bases packed little-endian in x (byte 0 = first base): code8 =
// their 2-bit codes, first base most significant; inv4 = 1 bit per invalid
// base, first base most significant.  A byte is a base iff (byte | 0x20)
// is one of a, c, g, t; each check is done on all four bytes at once.
__device__ __forceinline__ void encode4(uint32_t x, uint32_t& code8, uint32_t& inv4) {
    const uint32_t c = ((x >> 1) ^ (x >> 2)) & 0x03030303u;  // code of every byte
    code8 = (c * 0x40100401u) >> 24;                        // b0<<6 | b1<<4 | b2<<2 | b3
    // the only letter (lower case) with code c: 'a' + {0, 2, 6, 19}[c]
    const uint32_t hi = (c >> 1) & 0x01010101u;
    const uint32_t both = c & (c >> 1) & 0x01010101u;
    const uint32_t expect = 0x61616161u + (c << 1) + (hi << 1) + both * 11u;
    const uint32_t d = (x | 0x20202020u) ^ expect;            // zero byte <=> valid base
    uint32_t z = (d & 0x7F7F7F7Fu) + 0x7F7F7F7Fu;
    z = ~(z | d | 0x7F7F7F7Fu);                               // bit 7 of each zero byte
    const uint32_t valid = (((z >> 7) & 0x01010101u) * 0x08040201u) >> 24;  // b0<<3 | ... | b3
    inv4 = ~valid & 0xFu;
}

// Bitonic sort of one value per lane across the warp (ascending by lane),
// in mirror form: each merge stage of size k first pairs lane i with lane
// i ^ (k - 1), then with i ^ j for j = k/4 .. 1, and the lower lane of a
// pair always keeps the minimum (five lane-bit predicates in all).
__device__ __forceinline__ uint32_t warp_sort32(uint32_t v) {
    const uint32_t lane = lane_id();
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
        {
            const uint32_t u = __shfl_xor_sync(FULL_MASK, v, k - 1);
            v = (lane & (uint32_t)(k >> 1)) == 0 ? min(v, u) : max(v, u);
        }
#pragma unroll
        for (int j = k >> 2; j > 0; j >>= 1) {
            const uint32_t u = __shfl_xor_sync(FULL_MASK, v, j);
            v = (lane & (uint32_t)j) == 0 ? min(v, u) : max(v, u);
        }
    }
    return v;
}

// Computes the sketches of NW windows at once (independent dependency
// chains interleave).  Window w starts at base ws[w] of seq[w] (length
// L[w]; global memory, or shared memory when GLOBAL_SEQ is false); inactive
// windows yield count 0.  count[w] is warp-uniform; lane i < count[w] holds
// feature i of window w (ascending) in feature[w].  Requires 32*R >= w.
// cand: per-warp shared scratch of NW*32 words.
//
// Selection of the s smallest distinct hashes: a cutoff tau is chosen so
// that about 24 of the window's n_k hashes fall below it (all of them when
// n_k <= 32).  The hashes <= tau (at most 32 of them) are gathered one per
// lane, sorted by a warp bitonic network and de-duplicated.  If that gives
// at least s distinct values, or no valid hash lies above tau, they are
// exactly the s smallest distinct hashes.  Otherwise (a few percent of
// windows, and low-complexity windows) the exact fallback runs: s rounds of
// a warp min-reduction over locally sorted, de-duplicated lane lists.
template <int R, int NW, int KC = 0, bool GLOBAL_SEQ = true>
__device__ __forceinline__ void warp_sketch_multi(const uint8_t* const (&seq)[NW], const uint64_t (&L)[NW],
                                                  const uint64_t (&ws)[NW], const bool (&active)[NW],
                                                  const SketchParams& p, uint32_t* cand, uint32_t (&feature)[NW],
                                                  uint32_t (&count)[NW]) {
    constexpr int E_MAX = (15 + R - 1) / R;  // neighbours for k <= 16
    constexpr int T = R * (1 + E_MAX);       // bases held by a lane
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    const uint32_t k = KC ? (uint32_t)KC : p.k;  // k-mer length (compile-time when KC != 0)
    const uint32_t kmask_bits = 2 * k;
    const uint64_t cmask = (kmask_bits == 32) ? 0xFFFFFFFFull : ((1ull << kmask_bits) - 1);
    const uint64_t imask = (1ull << k) - 1;
    uint32_t h[NW][R];
    uint32_t vmask[NW];  // bit r: h[w][r] is a valid k-mer's hash
    bool fast[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const uint32_t n_k = active[w] ? window_kmers(L[w], ws[w], p) : 0u;
        uint64_t lim = ws[w] + p.w;
        if (lim > L[w]) lim = L[w];
        if (!active[w]) lim = 0;
        // 1. load and encode R bases (bytes past the window's end read as 0,
        // an invalid base), four at a time
        uint32_t code = 0, inv = 0;
        const uint64_t b0 = ws[w] + (uint64_t)R * lane;
#pragma unroll
        for (int g = 0; g < R / 4; ++g) {
            uint32_t x = 0;
            if (GLOBAL_SEQ) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint64_t b = b0 + 4 * g + i;
                    const uint32_t c = b < lim ? (uint32_t)__ldg(seq[w] + b) : 0u;
                    x |= c << (8 * i);
                }
            } else {
                // staged bases: the aligned words holding bases bg .. bg+3 and a
                // funnel shift; a word is read only if it holds a base before
                // lim, so every read stays inside the staged range
                const uint64_t bg = b0 + 4 * g;
                if (bg < lim) {
                    const uintptr_t a = reinterpret_cast<uintptr_t>(seq[w] + bg);
                    const uint32_t sh = (uint32_t)(a & 3u);
                    const uint32_t* wp = reinterpret_cast<const uint32_t*>(a - sh);
                    const uint32_t lo = wp[0];
                    const uint32_t hi = (sh != 0 && bg + (4 - sh) < lim) ? wp[1] : 0u;
                    x = __funnelshift_r(lo, hi, 8 * sh);
                    const uint64_t nb = lim - bg;
                    if (nb < 4) x &= (1u << (8 * (uint32_t)nb)) - 1u;
                }
            }
            uint32_t c8, i4;
            encode4(x, c8, i4);
            code = (code << 8) | c8;
            inv = (inv << 4) | i4;
        }
        // 2. bases of the following lanes
        uint64_t comb = code, combinv = inv;
#pragma unroll
        for (int e = 1; e <= E_MAX; ++e) {
            comb = (comb << (2 * R)) | __shfl_down_sync(FULL_MASK, code, e);
            combinv = (combinv << R) | __shfl_down_sync(FULL_MASK, inv, e);
        }
        // 3. canonical k-mers and h1; the reverse complement of the lane's T
        // bases is formed once (reverse the 2-bit digits, complement), and
        // the k-mer starting at base r reads as its digits 2r .. 2r + 2k - 1
        vmask[w] = 0;
        uint64_t rcomb = __brevll(comb);
        rcomb = ((rcomb >> 1) & 0x5555555555555555ull) | ((rcomb & 0x5555555555555555ull) << 1);
        rcomb = ~rcomb >> (64 - 2 * T);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t shift = (uint32_t)(T - r) - k;  // >= 0 since T >= R + k - 1
            const uint32_t fwd = (uint32_t)((comb >> (2 * shift)) & cmask);
            const bool bad = ((combinv >> shift) & imask) != 0;
            const bool ok = ((uint32_t)R * lane + r < n_k) && !bad;
            const uint32_t rc = (uint32_t)((rcomb >> (2 * r)) & cmask);
            h[w][r] = ok ? hash_h1(fwd < rc ? fwd : rc) : 0xFFFFFFFFu;
            vmask[w] |= (ok ? 1u : 0u) << r;
        }
        // 4. candidates below the cutoff, one per lane in cand[]
        // (any cutoff is correct; a fast reciprocal is plenty for aiming at ~24)
        const uint32_t tau = n_k <= 32 ? 0xFFFFFFFFu : __float2uint_rz(__fdividef(24.0f, (float)n_k) * 4294967296.0f);
        uint32_t cmine = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) cmine += (((vmask[w] >> r) & 1u) && h[w][r] <= tau) ? 1u : 0u;
        uint32_t pre = cmine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t x = __shfl_up_sync(FULL_MASK, pre, d);
            if ((int)lane >= d) pre += x;
        }
        const uint32_t C = __shfl_sync(FULL_MASK, pre, 31);
        const uint32_t Nv = __reduce_add_sync(FULL_MASK, (uint32_t)__popc(vmask[w]));
        pre -= cmine;
        fast[w] = C <= 32;
        if (fast[w]) {
            uint32_t o = pre;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (((vmask[w] >> r) & 1u) && h[w][r] <= tau) cand[w * 32 + o++] = h[w][r];
        }
        __syncwarp();
        if (fast[w]) {
            uint32_t v = lane < C ? cand[w * 32 + lane] : 0xFFFFFFFFu;
            v = warp_sort32(v);
            const uint32_t prev = __shfl_up_sync(FULL_MASK, v, 1);
            const bool fresh = lane < C && (lane == 0 || v != prev);
            const uint32_t nd = __ballot_sync(FULL_MASK, fresh);
            const uint32_t D = __popc(nd);
            fast[w] = D >= p.s || C == Nv;
            if (fast[w]) {
                if (D != C) {  // duplicates: compact the distinct values
                    __syncwarp();
                    if (fresh) cand[w * 32 + __popc(nd & lt)] = v;
                    __syncwarp();
                    v = cand[w * 32 + lane];
                }
                count[w] = D < p.s ? D : p.s;
                feature[w] = lane < count[w] ? v : 0u;
            }
        }
    }

    // exact fallback for the windows the cutoff did not settle
    uint32_t need = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) need |= (fast[w] ? 0u : 1u) << w;
    if (need == 0) return;
    int nv[NW];
    bool any_dup = false;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        nv[w] = 0;
        if (fast[w]) continue;
        // local sort + local de-duplication (valid entries become the first nv)
        nv[w] = __popc(vmask[w]);
        sort_small<R>(h[w]);
#pragma unroll
        for (int r = R - 1; r >= 1; --r) {
            if ((r < nv[w]) && (h[w][r] == h[w][r - 1])) {
                h[w][r] = 0xFFFFFFFFu;
                nv[w] -= 1;
                any_dup = true;
            }
        }
        count[w] = 0;
        feature[w] = 0;
    }
    if (__any_sync(FULL_MASK, any_dup)) {
#pragma unroll
        for (int w = 0; w < NW; ++w)
            if (!fast[w]) sort_small<R>(h[w]);
    }
    for (uint32_t it = 0; it < p.s; ++it) {
        uint32_t mine = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) mine |= (nv[w] > 0 ? 1u : 0u) << w;
        const uint32_t live = __reduce_or_sync(FULL_MASK, mine);
        if (live == 0) break;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (!((live >> w) & 1u)) continue;
            const bool has = nv[w] > 0;
            const uint32_t m = __reduce_min_sync(FULL_MASK, has ? h[w][0] : 0xFFFFFFFFu);
            const bool pop = has && (h[w][0] == m);
#pragma unroll
            for (int r = 0; r < R - 1; ++r) h[w][r] = pop ? h[w][r + 1] : h[w][r];
            h[w][R - 1] = pop ? 0xFFFFFFFFu : h[w][R - 1];
            nv[w] -= pop ? 1 : 0;
            if (lane == it) feature[w] = m;
            count[w] += 1;
        }
    }
}


// ------------------------------------------------------ lane-wide sketches
// The same sketch with one window per lane: a warp sketches 32 windows at
// once, each lane walking its own window over bases staged in shared memory
// as 2-bit codes.  What it saves over one warp per window: a k-mer is one
// funnel shift of two 32-bit words (16 bases) and its reverse complement
// another (no shuffles, no 64-bit arithmetic), and the selection sorts in
// registers without cross-lane steps, so that a window costs about 120 warp
// instructions instead of about 500.  What it needs: 32 windows to fill the
// warp, and s <= 16.

constexpr uint32_t LS_MAX_S = 16;      // largest sketch size of the lane path
// words of the candidate buffer for at most cap candidates per lane (eight
// more rows: the count is checked every 8 k-mers)
__host__ __device__ constexpr uint32_t ls_cand_words(uint32_t cap) { return (cap + 8) * 32; }
constexpr uint32_t LS_FEAT_STRIDE = 33;  // feat[i * 33 + lane]: rows and columns without bank conflicts
constexpr uint32_t LS_MARGIN = 12;     // the cutoff aims at s + 12 candidates

// 16 bases (byte 0 of x = the first) as a 32-bit word of 2-bit codes, first
// base in the top digit; inv = one bit per invalid base, first base in bit
// 15.  c is the code of every byte; the letter of a code comes from a byte
// permute, so a byte is a base iff it equals its own code's letter with bit
// 5 set.  The invalid bits are only formed when there are some.
__device__ __forceinline__ uint32_t encode16(const uint4& x, uint32_t& inv) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
    uint32_t code = 0, d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t c = ((w[i] >> 1) ^ (w[i] >> 2)) & 0x03030303u;
        code = (code << 8) | ((c * 0x40100401u) >> 24);
        const uint32_t n = __byte_perm(c | (c >> 4), 0, 0x4420);  // the four codes as nibbles
        d[i] = (w[i] | 0x20202020u) ^ __byte_perm(0x74676361u, 0, n);  // 'a' 'c' 'g' 't'
    }
    inv = 0;
    if (d[0] | d[1] | d[2] | d[3]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t z = ((d[i] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | d[i];  // bit 7 of each nonzero byte
            inv = (inv << 4) | (((((z >> 7) & 0x01010101u) * 0x08040201u) >> 24) & 0xFu);
        }
    }
    return code;
}

// Reverse complement of 16 bases.
__device__ __forceinline__ uint32_t revcomp16(uint32_t a) {
    const uint32_t r = __brev(a);
    return ~(((r >> 1) & 0x55555555u) | ((r & 0x55555555u) << 1));
}

// The 16-byte aligned chunk at address c, with bytes outside [lo, hi) left
// unread (0, an invalid base).
__device__ __forceinline__ uint4 load_chunk(uintptr_t c, uintptr_t lo, uintptr_t hi) {
    if (c >= lo && c + 16 <= hi) return __ldg(reinterpret_cast<const uint4*>(c));
    uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (c + i >= lo && c + i < hi)
            w[i >> 2] |= (uint32_t)__ldg(reinterpret_cast<const uint8_t*>(c + i)) << (8 * (i & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Batcher's odd-even merge sort of 16 registers: its 63 comparators as a
// table, applied through a fold so that every register index is a constant
// (left to loop unrolling, the compiler may give up and move the registers
// to local memory).
struct SortNet16 {
    int a[63] = {}, b[63] = {};
};
constexpr SortNet16 make_sort_net16() {
    SortNet16 n{};
    int c = 0;
    for (int p = 1; p < 16; p *= 2)
        for (int k = p; k >= 1; k /= 2)
            for (int j = k % p; j + k < 16; j += 2 * k)
                for (int i = 0; i < k; ++i)
                    if (i + j + k < 16 && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
                        n.a[c] = i + j;
                        n.b[c++] = i + j + k;
                    }
    return n;
}

__device__ __forceinline__ void compare_exchange(uint32_t& x, uint32_t& y) {
    const uint32_t a = x, b = y;
    x = min(a, b);
    y = max(a, b);
}

template <size_t... I>
__device__ __forceinline__ void sort16_steps(uint32_t (&v)[16], std::index_sequence<I...>) {
    constexpr SortNet16 net = make_sort_net16();
    (compare_exchange(v[std::integral_constant<int, net.a[I]>::value], v[std::integral_constant<int, net.b[I]>::value]),
     ...);
}

__device__ __forceinline__ void sort16(uint32_t (&v)[16]) { sort16_steps(v, std::make_index_sequence<63>()); }

// v = the 16 smallest of the sorted v and u, sorted.
__device__ __forceinline__ void keep_smallest16(uint32_t (&v)[16], const uint32_t (&u)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = min(v[i], u[15 - i]);  // bitonic
#pragma unroll
    for (int j = 8; j > 0; j >>= 1) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if ((i & j) == 0) {
                const uint32_t a = v[i], b = v[i | j];
                v[i] = min(a, b);
                v[i | j] = max(a, b);
            }
        }
    }
}

// Keeps y (h1 before its last step) as a candidate if it is at most tau:
// stored at shared address at, which moves on by one row.
__device__ __forceinline__ void lane_candidate(uint32_t y, uint32_t tau, uint32_t& at) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.le.u32 p, %1, %2;\n\t"
        "@p st.shared.u32 [%0], %1;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(at)
        : "r"(y), "r"(tau)
        : "memory");
}

// The same if on is not 0.
__device__ __forceinline__ void lane_candidate_if(uint32_t on, uint32_t y, uint32_t tau, uint32_t& at) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %3, 0;\n\t"
        "setp.le.and.u32 p, %1, %2, q;\n\t"
        "@p st.shared.u32 [%0], %1;\n\t"
        "@p add.u32 %0, %0, 128;\n\t}"
        : "+r"(at)
        : "r"(y), "r"(tau), "r"(on)
        : "memory");
}

// Sketches one window per lane (all lanes of the warp call together).
//  code, inv : the staged bases (encode16), n_words entries each;
//  any_inv   : warp-uniform, false if every staged base is valid;
//  pos, n_k  : this lane's window: staged index of its first base and its
//              number of k-mers (0 = no window);
//  cand      : ls_cand_words(CAP) words of the warp's shared memory, for at
//              most CAP candidates per lane.
// Returns true if v[0 .. cnt) are the window's features, ascending; false if
// this lane's window has to be sketched by the exact warp-wide selection:
// fewer than s candidates below the cutoff, more than CAP, or a repeated
// value among the s smallest (of random sequence 0.3% of the windows with
// CAP = 48, 0.7% with CAP = 40).
// Every word index is clamped to the staged words, so that a lane whose
// window is shorter than its neighbours' stays inside them.
template <int KC, uint32_t CAP>
__device__ __forceinline__ bool lane_sketch(const uint32_t* code, const uint16_t* inv, uint32_t n_words, bool any_inv,
                                            uint32_t pos, uint32_t n_k, const SketchParams& p, uint32_t* cand,
                                            uint32_t (&v)[16], uint32_t& cnt) {
    const uint32_t lane = lane_id();
    const uint32_t k = KC ? (uint32_t)KC : p.k;
    const uint32_t aim = p.s + LS_MARGIN;
    // Any cutoff is correct; a fast reciprocal is plenty for aiming.  Its low
    // 16 bits are ones: h1's last step y ^= y >> 16 keeps the top 16 bits, so
    // h1 <= tau iff y <= tau, and only the candidates take that step.
    const uint32_t tau =
        n_k <= aim ? 0xFFFFFFFFu : __float2uint_rz(__fdividef((float)aim, (float)n_k) * 4294967296.0f) | 0xFFFFu;
    const uint32_t n_max = __reduce_max_sync(FULL_MASK, n_k);
    const uint32_t last = n_words - 1;
    const uint32_t boff = pos & 15u, sh = 2 * boff;
    uint32_t wi = pos >> 4;
    uint32_t w1 = code[min(wi + 1, last)];
    uint32_t a0 = __funnelshift_l(w1, code[min(wi, last)], sh);
    uint32_t r0 = revcomp16(a0);
    // Candidates go to row C of the lane's column: a predicated store and
    // add each (a branch per k-mer costs more than the k-mer).
    const uint32_t col = (uint32_t)__cvta_generic_to_shared(cand + lane);
    const uint32_t col_cap = col + CAP * 128;
    uint32_t at = col;
    bool over = false;
    __syncwarp();  // the candidate buffer may still be read by its previous use
    for (uint32_t base = 0; base < n_max; base += 16, ++wi) {
        const uint32_t w2 = code[min(wi + 2, last)];
        const uint32_t a1 = __funnelshift_l(w2, w1, sh);
        const uint32_t r1 = revcomp16(a1);
        // bit 15 - r: k-mer base + r exists and holds no invalid base
        const uint32_t rem = n_k > base ? n_k - base : 0u;
        uint32_t ok = rem >= 16 ? 0xFFFFu : (0xFFFF0000u >> rem) & 0xFFFFu;
        if (any_inv) {
            const uint32_t hi = ((uint32_t)inv[min(wi, last)] << 16) | inv[min(wi + 1, last)];
            uint32_t z = __funnelshift_l((uint32_t)inv[min(wi + 2, last)] << 16, hi, boff);
            uint32_t c = 1;
            for (; 2 * c <= k; c *= 2) z |= z << c;
            z |= z << (k - c);
            ok &= ~(z >> 16);
        }
        if (__all_sync(FULL_MASK, ok == 0xFFFFu)) {
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                uint32_t f = __funnelshift_l(a1, a0, 2 * r);
                uint32_t g = __funnelshift_r(r0, r1, 2 * r);
                if (KC == 0) {
                    f >>= 32 - 2 * k;
                    g &= 0xFFFFFFFFu >> (32 - 2 * k);
                }
                lane_candidate(hash_h1_head(min(f, g)), tau, at);
                if ((r & 7) == 7 && at > col_cap) {
                    over = true;
                    at = col;
                }
            }
        } else {  // ends of sequences and windows, invalid bases
            const uint32_t r_max = n_max - base;
#pragma unroll
            for (int r4 = 0; r4 < 16; r4 += 4) {
                if ((uint32_t)r4 < r_max) {
#pragma unroll
                    for (int r = r4; r < r4 + 4; ++r) {
                        uint32_t f = __funnelshift_l(a1, a0, 2 * r);
                        uint32_t g = __funnelshift_r(r0, r1, 2 * r);
                        if (KC == 0) {
                            f >>= 32 - 2 * k;
                            g &= 0xFFFFFFFFu >> (32 - 2 * k);
                        }
                        lane_candidate_if(ok & (1u << (15 - r)), hash_h1_head(min(f, g)), tau, at);
                    }
                    if (r4 == 4 && at > col_cap) {
                        over = true;
                        at = col;
                    }
                }
            }
            if (at > col_cap) {
                over = true;
                at = col;
            }
        }
        a0 = a1;
        r0 = r1;
        w1 = w2;
    }
    const uint32_t C = (at - col) >> 7;
    const uint32_t c_max = __reduce_max_sync(FULL_MASK, C);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0xFFFFFFFFu;
#pragma unroll 1
    for (uint32_t b = 0; b < c_max; b += 16) {
        uint32_t u[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) u[i] = b + i < C ? hash_h1_tail(cand[(b + i) * 32 + lane]) : 0xFFFFFFFFu;
        sort16(u);
        keep_smallest16(v, u);
    }
    cnt = min(C, p.s);
    bool dup = false;
#pragma unroll
    for (int i = 0; i < 15; ++i) dup |= (uint32_t)(i + 1) < cnt && v[i] == v[i + 1];
    return !over && !dup && (C >= p.s || tau == 0xFFFFFFFFu);
}

// The exact selection with one window per lane, for the windows that
// lane_sketch leaves (n_k = 0: not this lane's; all lanes call together): a
// lane keeps its 16 smallest distinct hashes sorted in registers.  A k-mer
// that is new to no lane costs the hash, 16 compares and a vote, one that is
// another 32 minimum and maximum steps.  Writes the features to the lane's
// column of feat (stride LS_FEAT_STRIDE) and returns their number.
// Sequence without variety leaves most windows of a warp, and the exact
// selection by the whole warp takes them one by one: 64 Mbp of a repeat of six
// bases 527 us that way, 271 this way, of N 336 and 107.
template <int KC>
__device__ __forceinline__ uint32_t lane_sketch_exact(const uint32_t* code, const uint16_t* inv, uint32_t n_words,
                                                   uint32_t pos, uint32_t n_k, uint32_t k_any, uint32_t s,
                                                   uint32_t* feat) {
    const uint32_t lane = lane_id();
    const uint32_t k = KC ? (uint32_t)KC : k_any;
    const uint32_t n_max = __reduce_max_sync(FULL_MASK, n_k);
    const uint32_t last = n_words - 1;
    const uint32_t boff = pos & 15u, sh = 2 * boff;
    uint32_t wi = pos >> 4;
    uint32_t w1 = code[min(wi + 1, last)];
    uint32_t a0 = __funnelshift_l(w1, code[min(wi, last)], sh);
    uint32_t r0 = revcomp16(a0);
    uint32_t v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0xFFFFFFFFu;
    bool ones = false;  // the hash of all ones, which marks a free place too, was met
    for (uint32_t base = 0; base < n_max; base += 16, ++wi) {
        const uint32_t w2 = code[min(wi + 2, last)];
        const uint32_t a1 = __funnelshift_l(w2, w1, sh);
        const uint32_t r1 = revcomp16(a1);
        // bit 15 - r: k-mer base + r exists and holds no invalid base
        const uint32_t rem = n_k > base ? n_k - base : 0u;
        uint32_t ok = rem >= 16 ? 0xFFFFu : (0xFFFF0000u >> rem) & 0xFFFFu;
        const uint32_t hi = ((uint32_t)inv[min(wi, last)] << 16) | inv[min(wi + 1, last)];
        uint32_t z = __funnelshift_l((uint32_t)inv[min(wi + 2, last)] << 16, hi, boff);
        uint32_t c = 1;
        for (; 2 * c <= k; c *= 2) z |= z << c;
        z |= z << (k - c);
        ok &= ~(z >> 16);
        if (__any_sync(FULL_MASK, ok != 0)) {
#pragma unroll 1
            for (uint32_t r = 0; r < 16; ++r) {
                uint32_t f = __funnelshift_l(a1, a0, 2 * r);
                uint32_t g = __funnelshift_r(r0, r1, 2 * r);
                if (KC == 0) {
                    f >>= 32 - 2 * k;
                    g &= 0xFFFFFFFFu >> (32 - 2 * k);
                }
                uint32_t y = hash_h1(min(f, g));
                bool in = (ok >> (15 - r)) & 1u;
                ones |= in && y == 0xFFFFFFFFu;
                in = in && y < v[15];
#pragma unroll
                for (int i = 0; i < 15; ++i) in = in && y != v[i];
                if (__any_sync(FULL_MASK, in)) {
                    if (!in) y = 0xFFFFFFFFu;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const uint32_t x = v[i];
                        v[i] = min(x, y);
                        y = max(x, y);
                    }
                }
            }
        }
        a0 = a1;
        r0 = r1;
        w1 = w2;
    }
    uint32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) cnt += (uint32_t)i < s && v[i] != 0xFFFFFFFFu;
    cnt = min(cnt + (ones ? 1u : 0u), s);
    if (n_k) {
#pragma unroll
        for (int i = 0; i < 16; ++i) feat[i * LS_FEAT_STRIDE + lane] = v[i];
    }
    return cnt;
}

// R for a window length: the warp covers 32*R >= w bases.
__host__ __device__ inline int sketch_r_for(uint32_t w) { return w <= 128 ? 4 : (w <= 256 ? 8 : 16); }

}  // namespace mc
