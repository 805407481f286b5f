// Read classification kernels (Section 4.2 query phase, Section 5.2 query
// steps 1-8, Sections 5.3-5.6) for sm_103a.
//
// GB300 design.  The paper runs the query as a pipeline of kernels with
// global-memory hand-offs: sketch+lookup, compaction, a segmented sort
// (about half of its query time, Section 6.4) and a top-candidate kernel.
// Here a launch set has a lookup kernel and scoring kernels:
//   1. lookup: every window of every mate is sketched (mc_sketch.cuh; one
//      window per lane in large launches, one per warp in small ones) and
//      each feature looked up in the feature table (one 16-byte probe,
//      Section 5.3); a query's found buckets go to its list;
//   2. sort path, one warp per query, in size classes: the bucket locations
//      are gathered, those that cannot reach the label's threshold dropped by
//      a count per (target, window block), the rest sorted in registers; runs
//      of equal locations give the window count statistic (Section 4.2),
//      index differences the sliding-window scores (Section 5.6), warp
//      arg-max rounds the top candidates, labelled by the top target or the
//      LCA of the close candidates via the lineage table;
//   3. medium and large paths, one CTA per query, for more locations, windows
//      or bases; launches of a few queries go straight to the large path.
// The hash path (a tuning choice) counts locations in a per-warp shared-memory
// histogram instead of sorting them.  Every path gives the same results.
#include <algorithm>
#include <type_traits>

#include "mc_internal.h"
#include "mc_sketch.cuh"

namespace mc {

namespace {

constexpr int CLS_WARPS = 4;                 // warps per CTA (score path)
constexpr int LK_WARPS = 8;                  // warps per CTA (lookup path)
constexpr int WIN_A = 8;                     // windows per query on the shared-memory path
constexpr uint32_t KB_SLOTS = 1u << 16;      // large-path histogram slots per CTA
constexpr uint32_t LIST_B = MC_MAX_QUERY_WINDOWS * MAX_S;
constexpr uint32_t LIST_CAP_MAX = WIN_A * MAX_S;  // bucket list of a query of the lookup kernels, any sketch size
constexpr uint32_t MED_DISTINCT = 1536;      // distinct locations of a query on the medium path
constexpr int SK_NW = 2;  // windows sketched together

struct Cand {
    uint32_t score, t, j0, j1;
};

// Order of candidates: higher score first, then smaller target, then
// smaller first window (Section 4.2 top hits; ties are our reading).
__device__ __forceinline__ bool better(const Cand& a, const Cand& b) {
    if (a.score != b.score) return a.score > b.score;
    if (a.t != b.t) return a.t < b.t;
    return a.j0 < b.j0;
}

__device__ __forceinline__ uint32_t loc_slot(uint64_t loc, uint32_t mask) {
    uint64_t h = (loc ^ (loc >> 29)) * 0x9E3779B97F4A7C15ull;
    return (uint32_t)(h >> 32) & mask;
}
__device__ __forceinline__ uint32_t loc_slot(uint32_t key, uint32_t mask) {
    uint32_t h = key * 0x9E3779B1u;
    return (h ^ (h >> 15)) & mask;
}

// Histogram keys.  A database stores its locations as 32-bit words target
// << jbits | window when every id fits, else as 64-bit words target << 32 |
// window (LocT).  The histogram keys a location by the stored word itself
// (KeyT == LocT), or, for 32-bit words, optionally by the 64-bit form (the
// wide-key launch shape).
template <class KeyT, class LocT = KeyT>
struct KeyCodec {
    static_assert(sizeof(KeyT) >= sizeof(LocT), "keys are at least as wide as locations");
    uint32_t jbits;
    __device__ __forceinline__ KeyT encode(LocT loc) const {
        if (sizeof(KeyT) == sizeof(LocT)) return (KeyT)loc;
        const uint32_t x = (uint32_t)loc;
        return (KeyT)(((uint64_t)(x >> jbits) << 32) | (x & ((1u << jbits) - 1u)));
    }
    __device__ __forceinline__ uint32_t target(KeyT k) const {
        return sizeof(KeyT) == 8 ? (uint32_t)((uint64_t)k >> 32) : (uint32_t)k >> jbits;
    }
    __device__ __forceinline__ uint32_t window(KeyT k) const {
        return sizeof(KeyT) == 8 ? (uint32_t)k : (uint32_t)k & ((1u << jbits) - 1u);
    }
    // windows after this key's window before the id field would overflow
    __device__ __forceinline__ uint32_t room(KeyT k) const {
        return sizeof(KeyT) == 8 ? 0xFFFFFFFFu - (uint32_t)k : ((1u << jbits) - 1u) - window(k);
    }
    static constexpr KeyT empty() { return (KeyT)~(KeyT)0; }
};

__device__ __forceinline__ uint64_t key_cas(uint64_t* p, uint64_t cmp, uint64_t val) {
    return atomicCAS((unsigned long long*)p, (unsigned long long)cmp, (unsigned long long)val);
}
__device__ __forceinline__ uint32_t key_cas(uint32_t* p, uint32_t cmp, uint32_t val) { return atomicCAS(p, cmp, val); }

// Histogram count increment: 32-bit counts use atomicAdd directly; 16-bit
// counts add 1 << 16*(slot&1) to the aligned 32-bit word holding them (a
// count never passes 65535 there, so the neighbour is not disturbed).
__device__ __forceinline__ void count_inc(uint32_t* cnts, uint32_t slot) { atomicAdd(cnts + slot, 1u); }
__device__ __forceinline__ void count_inc(uint16_t* cnts, uint32_t slot) {
    atomicAdd(reinterpret_cast<uint32_t*>(cnts) + (slot >> 1), 1u << ((slot & 1u) * 16));
}

// Histogram insert (count + 1).  `fresh_slot` receives the slot if the
// location was new, else stays -1.  Returns false if the table is full.
template <class CntT, class KeyT>
__device__ __forceinline__ bool hist_insert(KeyT* keys, CntT* cnts, uint32_t mask, KeyT key, int& fresh_slot) {
    constexpr KeyT EMPTY = KeyCodec<KeyT>::empty();
    uint32_t slot = loc_slot(key, mask);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        KeyT k = *(volatile KeyT*)(keys + slot);
        if (k == key) {
            count_inc(cnts, slot);
            return true;
        }
        if (k == EMPTY) {
            const KeyT prev = key_cas(keys + slot, EMPTY, key);
            if (prev == EMPTY || prev == key) {
                count_inc(cnts, slot);
                if (prev == EMPTY) fresh_slot = (int)slot;
                return true;
            }
        }
        slot = (slot + 1) & mask;
    }
    return false;
}

template <class CntT, class KeyT>
__device__ __forceinline__ uint32_t hist_count(const KeyT* keys, const CntT* cnts, uint32_t mask, KeyT key) {
    constexpr KeyT EMPTY = KeyCodec<KeyT>::empty();
    uint32_t slot = loc_slot(key, mask);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        const KeyT k = keys[slot];
        if (k == key) return cnts[slot];
        if (k == EMPTY) return 0;
        slot = (slot + 1) & mask;
    }
    return 0;
}

__device__ __forceinline__ uint32_t lca2(const ClassifyDb& db, uint32_t a, uint32_t b) {
    if (a >= db.n_taxa || b >= db.n_taxa) return NO_TAXON;
    uint32_t da = db.depth[a], dbb = db.depth[b];
    int64_t d = da < dbb ? da : dbb;
    const uint32_t* la = db.lineage + (uint64_t)a * db.lin_stride;
    const uint32_t* lb = db.lineage + (uint64_t)b * db.lin_stride;
    for (; d >= 0; --d)
        if (la[d] == lb[d]) return la[d];
    return NO_TAXON;
}

enum { Q_DONE = 0, Q_ESCALATE = 1, Q_TOO_LARGE = 2 };

constexpr uint32_t MAX_MATES = MC_MAX_QUERY_MATES;  // mates per query (lane i holds mate i)
constexpr int LB_DEFAULT = 4;       // feature-table probes in flight per lane
constexpr int GB_DEFAULT = 8;       // bucket loads in flight per lane

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Per-warp working memory (shared memory on the main path, global scratch
// on the large path).  CntT is the histogram count type: 16 bits on the
// shared-memory path (whose queries gather at most 65,535 locations), 32
// bits on the large path.  Unused regions have size 0.
template <class CntT, class KeyT = uint64_t>
struct Scratch {
    KeyT* keys;        // histogram keys (location), kcap
    CntT* cnts;        // histogram counts, kcap
    CntT* score;       // sliding-window scores of the dense entries, kcap
    uint16_t* dense;   // slots of the distinct locations, kcap
    uint32_t kcap;     // power of two, <= 65536
    uint64_t* list;    // found buckets, offset << 16 | size, list_cap
    uint32_t* l_pre;   // exclusive prefix of bucket sizes, list_cap + 1
    uint32_t list_cap;
    uint32_t* feat;    // features of all windows, feat_cap
    uint32_t* cand;    // sketch selection scratch, SK_NW * 32
    uint8_t* buf;      // the query's bases, buf_cap
    uint32_t buf_cap;
    uint32_t win_cap;  // windows per query
    uint32_t max_locs; // locations per query
};

template <class CntT, class KeyT = uint64_t>
__host__ __device__ constexpr size_t scratch_bytes(uint32_t kcap, uint32_t list_cap, uint32_t feat_cap,
                                                   uint32_t buf_cap) {
    return align16((size_t)kcap * sizeof(KeyT)) + 2 * align16((size_t)kcap * sizeof(CntT)) + align16((size_t)kcap * 2) +
           align16((size_t)list_cap * 8) + align16(((size_t)list_cap + 4) * 4) + align16((size_t)feat_cap * 4) +
           (feat_cap ? align16(4 * 32 * SK_NW) : 0) + (buf_cap ? align16(buf_cap + 16) : 0);
}

// Carves a Scratch out of `base` (16-byte aligned), in scratch_bytes order.
template <class CntT, class KeyT = uint64_t>
__device__ __forceinline__ Scratch<CntT, KeyT> carve(unsigned char* base, uint32_t kcap, uint32_t list_cap,
                                                     uint32_t feat_cap, uint32_t buf_cap, uint32_t win_cap) {
    Scratch<CntT, KeyT> S;
    unsigned char* p = base;
    S.keys = reinterpret_cast<KeyT*>(p);
    p += align16((size_t)kcap * sizeof(KeyT));
    S.cnts = reinterpret_cast<CntT*>(p);
    p += align16((size_t)kcap * sizeof(CntT));
    S.score = reinterpret_cast<CntT*>(p);
    p += align16((size_t)kcap * sizeof(CntT));
    S.dense = reinterpret_cast<uint16_t*>(p);
    p += align16((size_t)kcap * 2);
    S.list = reinterpret_cast<uint64_t*>(p);
    p += align16((size_t)list_cap * 8);
    S.l_pre = reinterpret_cast<uint32_t*>(p);
    p += align16(((size_t)list_cap + 4) * 4);
    S.feat = reinterpret_cast<uint32_t*>(p);
    p += align16((size_t)feat_cap * 4);
    S.cand = reinterpret_cast<uint32_t*>(p);
    p += feat_cap ? align16(4 * 32 * SK_NW) : 0;
    S.buf = p;
    S.kcap = kcap;
    S.list_cap = list_cap;
    S.buf_cap = buf_cap;
    S.win_cap = win_cap;
    S.max_locs = sizeof(CntT) == 2 ? 0xFFFFu : 0xFFFFFFFFu;
    return S;
}

struct Counters {
    unsigned long long features = 0, locations = 0, distinct = 0, found = 0, sectors = 0, queries = 0;
};

// Per-kernel counter block of mc_classify_debug: kernel k (0 hash score,
// 1-3 sort path 256/512/1024, 4 medium path, 5 large path, 6 sort path
// 2048) adds the queries it finished, their found buckets and their
// 32-byte sectors at counters[7 + 3k ...].
constexpr int KC_SCORE = 0, KC_MEDIUM = 4, KC_LARGE = 5;

// Batch holding query q of a multi-batch launch: the last batch whose
// first query is <= q (empty batches share their first query number with
// the next batch, so they are never chosen).
__device__ __forceinline__ uint32_t find_batch(const ClassifyQuery& Q, uint32_t q) {
    const uint32_t* pre = Q.bhdr + 2;
    uint32_t lo = 0, hi = Q.bhdr[0];
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (pre[mid] <= q) lo = mid; else hi = mid;
    }
    return lo;
}

// Number of queries of the launch (read on the device in the multi-batch
// form, so that a captured launch serves any batch set within capacity).
__device__ __forceinline__ uint32_t total_queries(const ClassifyQuery& Q) {
    return Q.batches ? Q.bhdr[1] : Q.n_q;
}

// Input of query q: its sequences and its mates' range.
struct QueryIn {
    const uint8_t* seq;
    const uint64_t* offs;
    uint32_t m0, m1;
};

__device__ __forceinline__ QueryIn query_in(const ClassifyQuery& Q, uint32_t q) {
    if (!Q.batches) return QueryIn{Q.seq, Q.offs, Q.qoffs[q], Q.qoffs[q + 1]};
    const uint32_t b = find_batch(Q, q);
    const BatchDesc& B = Q.batches[b];
    const uint32_t lq = q - Q.bhdr[2 + b];
    return QueryIn{B.seq, B.offs, B.qoffs[lq], B.qoffs[lq + 1]};
}

// Lane i (< m) writes candidate slot i; `mine` is the lane's candidate.
__device__ __forceinline__ void write_result(const ClassifyQuery& Q, uint32_t q, uint32_t label, uint32_t hits,
                                             uint32_t top, const Cand& mine) {
    const uint32_t lane = lane_id();
    if (lane == 0) {
        uint32_t* lab = Q.label;
        uint32_t* hit = Q.hits;
        uint32_t* tt = Q.top_target;
        uint32_t lq = q;
        if (Q.batches) {
            const uint32_t b = find_batch(Q, q);
            lab = Q.batches[b].label;
            hit = Q.batches[b].hits;
            tt = Q.batches[b].top_target;
            lq = q - Q.bhdr[2 + b];
        }
        lab[lq] = label;
        hit[lq] = hits;
        if (tt) tt[lq] = top;
    }
    if (Q.cands && lane < Q.m) {
        uint32_t* o = Q.cands + ((uint64_t)q * Q.m + lane) * 4;
        o[0] = mine.score;
        o[1] = mine.t;
        o[2] = mine.j0;
        o[3] = mine.j1;
    }
}

__device__ __forceinline__ void write_unclassified(const ClassifyQuery& Q, uint32_t q) {
    write_result(Q, q, NO_TAXON, 0, 0xFFFFFFFFu, Cand{0, 0xFFFFFFFFu, 0, 0});
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

// 16-byte asynchronous copy global -> shared (completion: cp_async_wait_all).
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// A query whose bases are (being) staged in working memory.  Per lane: the
// length, window count and staging offset of mate `lane`; the rest is
// warp-uniform.
struct Staged {
    int status;  // Q_DONE, Q_ESCALATE or Q_TOO_LARGE
    uint32_t nm, shift, span, n_win;
    uint32_t L, nw, boff;
};

// Query step 1a: reads the query's mates and stages its bases in buf (the
// mates of a query are consecutive sequences, so this is one contiguous
// range), placed at the same offset mod 16 as in memory.  ASYNC: every
// 16-byte aligned chunk that holds a base of the query is copied with
// cp.async (completion: cp_async_wait_all + __syncwarp; bytes of those
// chunks outside the query are copied too and never read).  Otherwise the
// aligned chunks inside the range are vector loads and the partial chunks
// at both ends are copied byte by byte.
template <bool ASYNC>
__device__ __forceinline__ Staged stage_query(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q, uint8_t* buf,
                                              uint32_t buf_cap, uint32_t win_cap) {
    const uint32_t lane = lane_id();
    const SketchParams& p = db.sp;
    Staged st{};
    const QueryIn in = query_in(Q, q);
    const uint32_t m0 = in.m0, m1 = in.m1;
    if (m1 < m0 || m1 - m0 > MAX_MATES) {
        st.status = Q_TOO_LARGE;
        return st;
    }
    const uint32_t nm = m1 - m0;
    // mates: lane i holds mate i's offset, length and window count
    const uint64_t o = lane <= nm ? in.offs[m0 + lane] : 0;
    const uint64_t o_next = __shfl_down_sync(FULL_MASK, o, 1);
    const uint64_t L = (lane < nm && o_next > o) ? o_next - o : 0;
    const uint64_t nw = lane < nm ? num_windows(L, p.k, p.stride) : 0;
    const uint64_t span_sum = warp_sum_u64(L);
    const uint64_t n_win = warp_sum_u64(nw);
    if (n_win > MC_MAX_QUERY_WINDOWS) {
        st.status = Q_TOO_LARGE;
        return st;
    }
    if (n_win > win_cap || span_sum > buf_cap) {
        st.status = Q_ESCALATE;
        return st;
    }
    uint64_t boff = L;  // exclusive prefix of mate lengths
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint64_t x = __shfl_up_sync(FULL_MASK, boff, d);
        if ((int)lane >= d) boff += x;
    }
    boff -= L;
    const uint64_t start = __shfl_sync(FULL_MASK, o, 0);
    const uintptr_t first = (uintptr_t)(in.seq + start);
    const uint32_t shift = (uint32_t)(first & 15u);
    const uintptr_t a0 = first - shift;
    const uint64_t n_chunks = (shift + span_sum + 15) / 16;
    if (ASYNC) {
        for (uint64_t c = lane; c < n_chunks; c += 32)
            cp_async16(buf + 16 * c, reinterpret_cast<const void*>(a0 + 16 * c));
        cp_async_commit();
    } else {
        for (uint64_t c = lane; c < n_chunks; c += 32) {
            const uintptr_t cs = a0 + 16 * c;
            if (cs >= first && cs + 16 <= first + span_sum) {
                *reinterpret_cast<uint4*>(buf + 16 * c) = __ldg(reinterpret_cast<const uint4*>(cs));
            } else {
                const uintptr_t lo = cs > first ? cs : first;
                const uintptr_t hi = cs + 16 < first + span_sum ? cs + 16 : first + span_sum;
                for (uintptr_t b = lo; b < hi; ++b) buf[b - a0] = __ldg(reinterpret_cast<const uint8_t*>(b));
            }
        }
        __syncwarp();
    }
    st.status = Q_DONE;
    st.nm = nm;
    st.shift = shift;
    st.span = (uint32_t)span_sum;
    st.n_win = (uint32_t)n_win;
    st.L = (uint32_t)L;
    st.nw = (uint32_t)nw;
    st.boff = (uint32_t)boff;
    return st;
}

// Query steps 1b-4 of Section 5.2 on one warp, for a query staged in buf:
// sketch every window of every mate, look every feature up; the found
// buckets are written to `list` (working memory or global scratch), packed
// as offset << 16 | size.  Also returns the sliding-window size, the number
// of features and the 32-byte sectors of the found buckets (warp totals).
template <int R, int KC, int LB, class CntT>
__device__ __forceinline__ void sketch_probe(const ClassifyDb& db, const ClassifyQuery& Q, const Scratch<CntT>& S,
                                             const uint8_t* buf, const Staged& sq, uint64_t* __restrict__ list,
                                             uint32_t& n_list_out, uint32_t& sws_out, uint32_t& n_feat_out,
                                             uint32_t& n_sect_out, uint32_t& n_locs_out) {
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    const SketchParams& p = db.sp;
    const uint32_t nm = sq.nm, shift = sq.shift;
    const uint64_t L = sq.L, nw = sq.nw, boff = sq.boff, n_win = sq.n_win, span_sum = sq.span;

    // 1b. sketch every window of every mate (Section 4.2: reads are windowed
    // like the targets), SK_NW windows at a time; feat[] gets the features
    // in window order
    uint32_t F = 0;
    {
        uint32_t mi = 0;          // mate of the next window
        uint64_t jn = 0;          // its window index
        uint64_t nw_mi = __shfl_sync(FULL_MASK, nw, 0);
        for (uint64_t done = 0; done < n_win; done += SK_NW) {
            const uint8_t* sqp[SK_NW];
            uint64_t Ls[SK_NW], wss[SK_NW];
            bool act[SK_NW];
#pragma unroll
            for (int i = 0; i < SK_NW; ++i) {
                act[i] = done + i < n_win;
                while (act[i] && jn >= nw_mi) {  // skip to the mate of this window
                    ++mi;
                    jn = 0;
                    nw_mi = __shfl_sync(FULL_MASK, nw, mi & 31);
                }
                sqp[i] = buf + shift + __shfl_sync(FULL_MASK, boff, mi & 31);
                Ls[i] = act[i] ? __shfl_sync(FULL_MASK, L, mi & 31) : 0;
                wss[i] = jn * p.stride;
                if (act[i]) ++jn;
            }
            uint32_t f[SK_NW], cnt[SK_NW];
            warp_sketch_multi<R, SK_NW, KC, false>(sqp, Ls, wss, act, p, S.cand, f, cnt);
#pragma unroll
            for (int i = 0; i < SK_NW; ++i) {
                if (lane < cnt[i]) S.feat[F + lane] = f[i];
                F += cnt[i];
            }
        }
    }
    __syncwarp();

    // 1c. feature table probes, LB per lane in flight.  A probe reads the
    // aligned 16-byte pair of table words holding the home slot, then
    // follows the ordered probe sequence (stop at an empty slot or a key >=
    // h) one word at a time; the longest sequence is the table's largest
    // displacement.
    const TableFmt fmt = db.fmt;
    const uint32_t lsz = db.jbits ? 4u : 8u;  // bytes per stored location
    uint32_t n_list = 0;
    unsigned long long n_sect = 0, n_locs = 0;
    for (uint32_t base = 0; base < F; base += 32 * LB) {
        uint32_t hk[LB];
        uint64_t pos[LB];
        ulonglong2 pr[LB];
#pragma unroll
        for (int b = 0; b < LB; ++b) {
            const uint32_t idx = base + b * 32 + lane;
            hk[b] = idx < F ? hash_h2(S.feat[idx]) : 0u;
            pos[b] = fmt.home(hk[b]);
            pr[b] = idx < F ? __ldg(reinterpret_cast<const ulonglong2*>(db.table + (pos[b] & ~1ull)))
                            : make_ulonglong2(0, 0);
        }
#pragma unroll
        for (int b = 0; b < LB; ++b) {
            const uint32_t idx = base + b * 32 + lane;
            uint32_t c = 0;
            uint64_t off = 0;
            if (idx < F) {
                uint64_t slot = pos[b];
                uint64_t e = (slot & 1) ? pr[b].y : pr[b].x;
                for (uint32_t d = 0; e != 0; ) {
                    const uint32_t k = fmt.key(e, slot);
                    if (k >= hk[b]) {
                        if (k == hk[b]) {
                            c = fmt.count(e);
                            off = fmt.offset(e);
                        }
                        break;
                    }
                    if (++d > db.max_probe) break;
                    ++slot;
                    e = (slot == (pos[b] | 1ull)) ? pr[b].y : __ldg(db.table + slot);
                }
            }
            const uint32_t found = __ballot_sync(FULL_MASK, c > 0);
            if (c > 0) {
                list[n_list + __popc(found & lt)] = (off << 16) | c;
                n_sect += ((off * lsz + (uint64_t)c * lsz - 1) >> 5) - ((off * lsz) >> 5) + 1;
                n_locs += c;
            }
            n_list += __popc(found);
        }
    }
    __syncwarp();
    n_feat_out = F;
    n_sect_out = (uint32_t)warp_sum_u64(n_sect);
    n_locs_out = (uint32_t)warp_sum_u64(n_locs);  // <= 2048 features x 65535
    const uint64_t span = (nm <= 1) ? span_sum : (span_sum > Q.max_insert ? span_sum : (uint64_t)Q.max_insert);
    sws_out = span >= p.k ? (uint32_t)((span - p.k + p.stride - 1) / p.stride + 1) : 0;
    n_list_out = n_list;
}

// Query steps 1-4 on one warp (staging, sketch, lookup), synchronously.
// Returns Q_DONE, Q_ESCALATE (needs the large path) or Q_TOO_LARGE.
template <int R, int KC, int LB, class CntT>
__device__ __forceinline__ int query_lookup(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                            const Scratch<CntT>& S, uint64_t* __restrict__ list, uint32_t& n_list_out,
                                            uint32_t& sws_out, uint32_t& n_feat_out, uint32_t& n_sect_out) {
    const Staged st = stage_query<false>(db, Q, q, S.buf, S.buf_cap, S.win_cap);
    if (st.status != Q_DONE) return st.status;
    uint32_t n_locs = 0;
    sketch_probe<R, KC, LB>(db, Q, S, S.buf, st, list, n_list_out, sws_out, n_feat_out, n_sect_out, n_locs);
    return Q_DONE;
}

// Query steps 5-8 of Section 5.2 on one warp, from the bucket list in
// working memory: gather, window count statistic, sliding-window scores,
// top m, label.  Writes the outputs and returns Q_DONE, or Q_ESCALATE if the
// histogram does not fit the working memory.
template <int GB, class LocT, class CntT, class KeyT>
__device__ __forceinline__ int query_score(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                           const Scratch<CntT, KeyT>& S, uint32_t n_list, uint32_t sws,
                                           Counters& ctr) {
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    const KeyCodec<KeyT, LocT> kc{db.jbits};
    constexpr KeyT EMPTY = KeyCodec<KeyT>::empty();
    constexpr LocT NO_LOC = (LocT)~(LocT)0;  // never a stored location
    const LocT* __restrict__ locs = static_cast<const LocT*>(db.locs);

    // 2. exclusive prefix of bucket sizes; H = locations to gather
    uint32_t H = 0;
    for (uint32_t base = 0; base < n_list; base += 32) {
        const uint32_t idx = base + lane;
        const uint32_t c = idx < n_list ? (uint32_t)(S.list[idx] & 0xFFFFu) : 0;
        uint32_t inc = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            uint32_t x = __shfl_up_sync(FULL_MASK, inc, d);
            if ((int)lane >= d) inc += x;
        }
        if (idx < n_list) S.l_pre[idx] = H + inc - c;
        H += __shfl_sync(FULL_MASK, inc, 31);
    }
    if (lane == 0) S.l_pre[n_list] = H;
    if (H > S.max_locs) return Q_ESCALATE;
    uint32_t kq = 32;
    while (kq < 2 * H && kq < S.kcap) kq <<= 1;
    const uint32_t mask = kq - 1;
    for (uint32_t s = lane; s < kq; s += 32) {
        S.keys[s] = EMPTY;
        S.cnts[s] = 0;
    }
    __syncwarp();

    // 3. gather the buckets into the hit histogram (window count statistic,
    // Section 4.2): each lane loads GB consecutive locations of the flat
    // list (all in flight), then inserts them; the slots of new locations
    // are appended to a dense list
    // at most 3/4 of the slots in use: linear probing stays short (an absent
    // key costs about 8.5 probes at 3/4, 32 at 7/8)
    const uint32_t limit = kq - kq / 4;
    uint32_t D = 0;
    for (uint32_t base = 0; base < H; base += 32 * GB) {
        const uint32_t x0 = base + lane * GB;
        // bucket of x0: last b with l_pre[b] <= x0
        uint32_t lo = 0, hi = n_list;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (S.l_pre[mid] <= x0) lo = mid; else hi = mid;
        }
        uint32_t bkt = lo;
        LocT v[GB];
#pragma unroll
        for (int g = 0; g < GB; ++g) {
            const uint32_t x = x0 + g;
            v[g] = NO_LOC;
            if (x < H) {
                while (S.l_pre[bkt + 1] <= x) ++bkt;
                v[g] = __ldg(locs + (S.list[bkt] >> 16) + (x - S.l_pre[bkt]));
            }
        }
        bool ok = true;
#pragma unroll
        for (int g = 0; g < GB; ++g) {
            int slot = -1;
            if (v[g] != NO_LOC) ok &= hist_insert(S.keys, S.cnts, mask, kc.encode(v[g]), slot);
            const uint32_t fresh = __ballot_sync(FULL_MASK, slot >= 0);
            if (slot >= 0) S.dense[D + __popc(fresh & lt)] = (uint16_t)slot;
            D += __popc(fresh);
            // checked after every round, so the table never passes limit + 32
            // entries: inserts stay cheap and a query that will not fit is
            // handed on as soon as it is known
            if (D > limit) return Q_ESCALATE;
        }
        if (__any_sync(FULL_MASK, !ok)) return Q_ESCALATE;
    }
    __syncwarp();
    ctr.locations += H;
    ctr.distinct += D;

    // 4. sliding-window scores (Section 5.6): score(t, j0) = sum of the
    // counts of (t, j0 .. j0+sws-1), for the distinct locations
    for (uint32_t i = lane; i < D; i += 32) {
        const uint32_t slot = S.dense[i];
        const KeyT key = S.keys[slot];
        uint32_t sc = S.cnts[slot];
        const uint32_t room = kc.room(key);  // windows left before the id wraps
        for (uint32_t d = 1; d < sws && d <= room; ++d) sc += hist_count(S.keys, S.cnts, mask, (KeyT)(key + d));
        S.score[i] = (CntT)sc;
    }
    __syncwarp();

    // 5. top m with one candidate per target (Section 4.2 / 5.6): rounds of
    // warp arg-max; the winner's target is excluded from later rounds by
    // zeroing the scores of its entries.  The label is folded as the
    // candidates come (hit threshold of Section 6.5, LCA of the close
    // candidates of Section 4.2).  Later rounds only give lower scores, so
    // unless the full top-m list is requested the rounds stop once the
    // query is unclassified or the best remaining score is not close.
    const int m = (int)Q.m;
    Cand mine = Cand{0, 0xFFFFFFFFu, 0, 0};
    uint32_t label = NO_TAXON, hits = 0, top = 0xFFFFFFFFu;
    uint64_t bar = 0;
    uint32_t prev_t = 0xFFFFFFFFu;
    for (int r = 0; r < m; ++r) {
        Cand best = Cand{0, 0xFFFFFFFFu, 0xFFFFFFFFu, 0};
        for (uint32_t i = lane; i < D; i += 32) {
            uint32_t sc = S.score[i];
            if (sc == 0) continue;
            const KeyT key = S.keys[S.dense[i]];
            const uint32_t t = kc.target(key);
            if (t == prev_t) {
                S.score[i] = 0;
                continue;
            }
            const Cand c = Cand{sc, t, kc.window(key), 0};
            if (better(c, best)) best = c;
        }
        // warp arg-max in the candidate order: highest score, then smallest
        // target, then smallest first window
        {
            const uint32_t ms = __reduce_max_sync(FULL_MASK, best.score);
            const uint32_t mt = __reduce_min_sync(FULL_MASK, best.score == ms ? best.t : 0xFFFFFFFFu);
            const uint32_t mj =
                __reduce_min_sync(FULL_MASK, (best.score == ms && best.t == mt) ? best.j0 : 0xFFFFFFFFu);
            best = Cand{ms, mt, mj, 0};
        }
        if (best.score == 0) break;
        prev_t = best.t;
        if (Q.cands) {
            // last window of the range present in the histogram
            uint32_t j1 = best.j0;
            for (uint32_t i = lane; i < D; i += 32) {
                const KeyT key = S.keys[S.dense[i]];
                const uint32_t j = kc.window(key);
                if (kc.target(key) == best.t && j >= best.j0 && (uint64_t)j < (uint64_t)best.j0 + sws && j > j1)
                    j1 = j;
            }
            best.j1 = __reduce_max_sync(FULL_MASK, j1);
        }
        if ((int)lane == r) mine = best;
        if (r == 0) {
            hits = best.score;
            top = best.t;
            bar = (uint64_t)(100 - Q.band) * hits;
            if (hits >= Q.hits_min) label = top < db.n_targets ? db.taxon_of_target[top] : NO_TAXON;
            else if (!Q.cands) break;
        } else if (hits >= Q.hits_min && 100ull * best.score >= bar) {
            const uint32_t tx = best.t < db.n_targets ? db.taxon_of_target[best.t] : NO_TAXON;
            label = lca2(db, label, tx);
        } else if (!Q.cands) {
            break;
        }
        __syncwarp();
    }
    write_result(Q, q, label, hits, top, mine);
    return Q_DONE;
}

// Whole query on one warp with the bucket list in working memory.
template <int R, int KC, class LocT, class CntT>
__device__ __noinline__ int process_query(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                             const Scratch<CntT>& S, Counters& ctr) {
    uint32_t n_list = 0, sws = 0, n_feat = 0, n_sect = 0;
    int r = query_lookup<R, KC, LB_DEFAULT>(db, Q, q, S, S.list, n_list, sws, n_feat, n_sect);
    if (r != Q_DONE) return r;
    r = query_score<GB_DEFAULT, LocT>(db, Q, q, S, n_list, sws, ctr);
    if (r == Q_DONE) {
        ctr.features += n_feat;
        ctr.found += n_list;
        ctr.sectors += n_sect;
        ++ctr.queries;
    }
    return r;
}

// counters: [0] features looked up, [1] locations gathered, [2] distinct
// locations, [3] queries on the large path, [4] features found, [5] 32-byte
// sectors of the gathered buckets, [6] queries finished on the medium path.
__device__ __forceinline__ void flush_counters(const ClassifyQuery& Q, const Counters& c, int kidx) {
    const unsigned long long sect = c.sectors;
    if (Q.counters && lane_id() == 0) {
        atomicAdd(Q.counters + 0, c.features);
        atomicAdd(Q.counters + 1, c.locations);
        atomicAdd(Q.counters + 2, c.distinct);
        atomicAdd(Q.counters + 4, c.found);
        atomicAdd(Q.counters + 5, sect);
        atomicAdd(Q.counters + 7 + 3 * kidx, c.queries);
        atomicAdd(Q.counters + 8 + 3 * kidx, c.found);
        atomicAdd(Q.counters + 9 + 3 * kidx, sect);
    }
}

// The counters of a warp's queries in a counting call (COUNTING kernels), kept
// in shared memory by its lane 0 and added up once: added per query, on eight
// addresses, they took longer than the sort (10^6 pairs, smallest class: 5.4
// ms that way, 1.6 this way).
__device__ __forceinline__ void flush_tally(const ClassifyQuery& Q, const unsigned long long* tally, int kidx) {
    if (lane_id()) return;
    Counters c;
    c.features = tally[0];
    c.locations = tally[1];
    c.distinct = tally[2];
    c.found = tally[3];
    c.sectors = tally[4];
    c.queries = tally[5];
    flush_counters(Q, c, kidx);
}

constexpr uint32_t BUF_A = 1024;   // bases per query on the shared-memory path
constexpr uint32_t BUF_B = 16384;  // bases per query on the large path

constexpr uint32_t ESCALATED = 0xFFFFFFFFu;

// A Staged query kept in shared memory (per lane: L, nw, boff; then the
// warp-uniform fields).
constexpr size_t STAGED_BYTES = 3 * 32 * 4 + 8 * 4;

__device__ __forceinline__ void save_staged(unsigned char* rec, const Staged& st) {
    uint32_t* r = reinterpret_cast<uint32_t*>(rec);
    const uint32_t lane = lane_id();
    r[lane] = st.L;
    r[32 + lane] = st.nw;
    r[64 + lane] = st.boff;
    if (lane == 0) {
        r[96] = (uint32_t)st.status;
        r[97] = st.nm;
        r[98] = st.shift;
        r[99] = st.span;
        r[100] = st.n_win;
    }
}

__device__ __forceinline__ Staged load_staged(const unsigned char* rec) {
    const uint32_t* r = reinterpret_cast<const uint32_t*>(rec);
    const uint32_t lane = lane_id();
    Staged st;
    st.L = r[lane];
    st.nw = r[32 + lane];
    st.boff = r[64 + lane];
    st.status = (int)r[96];
    st.nm = r[97];
    st.shift = r[98];
    st.span = r[99];
    st.n_win = r[100];
    return st;
}

// Shared memory of one lookup warp: working memory, a second staging buffer
// and two staged-query records.
__host__ __device__ constexpr size_t lookup_warp_bytes(uint32_t list_cap) {
    return scratch_bytes<uint16_t>(0, 0, list_cap, BUF_A) + align16(BUF_A + 16) + 2 * STAGED_BYTES;
}

// Counters of a launch set, behind the large-path queue.  The first two words
// count over all chunks, those up to QC_WIDEST over one chunk's score
// kernels; QC_WIDEST belongs to a chunk's lookup.
enum {
    QC_LARGE = 0,       // large-path queue length
    QC_LARGE_WORK = 1,  // its next entry
    QC_MID = 2,         // medium-path queue length
    QC_MID_WORK = 3,    // its next entry
    QC_GROUP = 4,       // next group of sort-path class c: QC_GROUP + c
    QC_QUEUED_WORK = 8, // next entry of the queue that warps take
    QC_REST = 9,        // length of the queue of what they leave
    QC_WIDEST = 10,     // most locations of a query, as far as the classes tell them apart
    QC_END = 11,
    QC_SAVED = 15       // large-path queue length after the lookup (autotuner)
};

// The lookup's warps note the size class of their largest query, so that the
// kernels of classes without a query end at once: handing out groups of
// queries to find none took each 8 us in launches of 8,000 queries and 20 us
// from 20,000 on (one counter serves about 10^9 groups/s).  widest holds a
// number of locations of the highest class that a query is in, or 0 if none
// is beyond the first.  seen: the warp's own highest so far (a warp writes at
// most once per class).
constexpr uint32_t CLASS_0_MAX = 256;
__device__ __forceinline__ void note_widest(uint32_t* widest, uint32_t locations, uint32_t& seen) {
    if (locations > max(seen, CLASS_0_MAX)) {
        atomicMax(widest, locations);
        // the next class's edge, or no further
        seen = locations <= 512 ? 512u : (locations <= 1024 ? 1024u : (locations <= 2048 ? 2048u : 0xFFFFFFFFu));
    }
}

// Per-query metadata written by the lookup kernel: {found buckets, sliding
// window size | features << META_FEAT_SHIFT, locations to gather, 32-byte
// sectors of those locations}, or x = ESCALATED.  On this path a query has
// at most WIN_A * MAX_S = 256 features and a sliding window below 2^17.
constexpr uint32_t META_FEAT_SHIFT = 20;
__device__ __forceinline__ uint32_t meta_sws(const uint4& m) { return m.y & ((1u << META_FEAT_SHIFT) - 1u); }
__device__ __forceinline__ uint32_t meta_feat(const uint4& m) { return m.y >> META_FEAT_SHIFT; }

__device__ __forceinline__ void tally_query(unsigned long long* tally, const uint4& mt, uint32_t distinct) {
    __syncwarp();
    if (lane_id()) return;
    tally[0] += meta_feat(mt);
    tally[1] += mt.z;
    tally[2] += distinct;
    tally[3] += mt.x;
    tally[4] += mt.w;
    tally[5] += 1;
}

// Main path, part 1 (sketch + lookup): one warp per query of the chunk
// [q0, q0 + nq), shared memory for the query's bases and features only, so
// many warps fit on an SM.  Software-pipelined: the bases of the warp's
// next query are copied (cp.async) into the other staging buffer while the
// current query is sketched and looked up.  Writes each query's bucket list
// to glist[(q - q0) * list_cap ...] and {list size, sliding-window size} to
// meta; queries that need the large path are queued.
template <int R, int KC, int LB>
__global__ void __launch_bounds__(LK_WARPS * 32, 4) k_classify_lookup(ClassifyDb db, ClassifyQuery Q, uint32_t q0,
                                                                  uint32_t chunk, uint32_t list_cap,
                                                                  uint64_t* __restrict__ glist,
                                                                  uint4* __restrict__ meta,
                                                                  uint32_t* __restrict__ ovf_list,
                                                                  uint32_t* __restrict__ ovf_n) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t w = threadIdx.x >> 5;
    unsigned char* mine = smem + w * lookup_warp_bytes(list_cap);
    const Scratch<uint16_t> S = carve<uint16_t>(mine, 0, 0, list_cap, BUF_A, WIN_A);
    uint8_t* const buf0 = S.buf;
    uint8_t* const buf1 = mine + scratch_bytes<uint16_t>(0, 0, list_cap, BUF_A);
    unsigned char* recs = buf1 + align16(BUF_A + 16);
    const uint32_t total = total_queries(Q);
    if (q0 >= total) return;
    const uint32_t nq = min(chunk, total - q0);
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarp = (gridDim.x * blockDim.x) >> 5;
    uint32_t cur = 0, seen = 0;
    if (gw < nq) save_staged(recs, stage_query<true>(db, Q, q0 + gw, buf0, BUF_A, WIN_A));
    for (uint32_t i = gw; i < nq; i += nwarp) {
        cp_async_wait_all();
        __syncwarp();
        const uint32_t nx = i + nwarp;
        if (nx < nq)
            save_staged(recs + (cur ^ 1) * STAGED_BYTES,
                        stage_query<true>(db, Q, q0 + nx, cur ? buf0 : buf1, BUF_A, WIN_A));
        const Staged st = load_staged(recs + cur * STAGED_BYTES);
        const uint32_t q = q0 + i;
        uint32_t n_list = 0, sws = 0, n_feat = 0, n_sect = 0, n_locs = 0;
        int r = st.status;
        if (r == Q_DONE)
            sketch_probe<R, KC, LB>(db, Q, S, cur ? buf1 : buf0, st, glist + (uint64_t)i * list_cap, n_list, sws, n_feat,
                                    n_sect, n_locs);
        if (r == Q_ESCALATE) {
            if (lane_id() == 0) {
                ovf_list[atomicAdd(ovf_n, 1u)] = q;
                meta[i] = make_uint4(ESCALATED, 0, 0, 0);
            }
        } else if (r == Q_TOO_LARGE) {
            write_unclassified(Q, q);
            if (lane_id() == 0) {
                atomicMax(Q.status, DEV_ERR_CAPACITY);
                meta[i] = make_uint4(ESCALATED, 0, 0, 0);
            }
        } else if (lane_id() == 0) {
            meta[i] = make_uint4(n_list, sws | (n_feat << META_FEAT_SHIFT), n_locs, n_sect);
            note_widest(ovf_n + QC_WIDEST, n_locs, seen);
        }
        __syncwarp();
        cur ^= 1;
    }
    cp_async_wait_all();
}

// Main path, part 1 with one window per lane (lane_sketch, sketch sizes up
// to 16).  A warp takes 2^batch_shift <= 32 consecutive queries, one lane
// each for their metadata, and works through them in groups that fill its
// 32 lanes with windows: as many queries as LKL_CHUNKS 16-base chunks and
// LKL_ITEMS windows hold (16 pairs of 150).  For a group it
//   - stages the bases as 2-bit codes, a chunk per lane and step;
//   - lists the windows, whole ones first, so that the lanes of a round
//     walk windows of like length (a read of 150 has one of 113 k-mers and
//     one of 22);
//   - per round of 32 windows sketches them and probes the feature table,
//     each lane for its own window's features, LB probes in flight.
// The order of a query's bucket list is of no consequence.
// Bound by the random reads of the table: 2 M pairs of 150 against the large
// database (128 M probes of 8.6 GB) take 4.59 ms, 28 G probes/s, against 5.89
// with one window per warp, which was bound by the sketching; without the
// probes this kernel takes 1.22 ms.  Entries written one by one instead of
// through shared memory: 4.87 ms; four or eight probes in flight instead of
// two: 4.9 and 5.5 ms.
constexpr uint32_t LKL_CHUNKS = 336;
constexpr uint32_t LKL_ITEMS = 64;
constexpr uint32_t LKL_CAP = 40;  // candidates per lane
constexpr uint32_t LKL_WORDS = (LKL_CHUNKS + 31) / 32 + 1;  // bitmap of chunk starts

struct LookupLanesMem {
    uint32_t code[LKL_CHUNKS];
    union {
        uint32_t cand[ls_cand_words(LKL_CAP)];
        struct {
            uint32_t hash[16 * 32];  // [i * 32 + lane]: h2 of a round's features
            uint32_t exact[32];      // scratch of the exact selection
            uint16_t more[16 * 32];  // probes to go on with
            uint64_t found[8 * 32];  // [i * 32 + lane]: buckets found with eight features
            uint32_t out_start[8];   // bitmap of the lanes' first entries in the output of those
            uint8_t out_lane[32];    // the lanes that have some, in order
        };
        struct {
            uint64_t base[32];  // chunk c of the group is at base[its query's rank] + 16 c
            uint32_t starts[LKL_WORDS];
        } stage;
    };
    uint32_t item[LKL_ITEMS];  // staged position | k-mers << 13 | query lane << 23
    uint32_t q_list[32];       // per query lane: found buckets | features << 16
    uint32_t q_locs[32];       // locations
    uint32_t q_sect[32];       // 32-byte sectors
    uint32_t seen;             // (note_widest)
    uint16_t inv[LKL_CHUNKS];
};
static_assert(LKL_CHUNKS * 16 <= 1u << 13, "staged positions take 13 bits");

template <int R, int KC, int LB>
__global__ void __launch_bounds__(LK_WARPS * 32, 3)
    k_lookup_lanes(ClassifyDb db, ClassifyQuery Q, uint32_t q0, uint32_t chunk, uint32_t list_cap,
                   uint64_t* __restrict__ glist, uint4* __restrict__ meta, uint32_t* __restrict__ ovf_list,
                   uint32_t* __restrict__ ovf_n, uint32_t batch_shift) {
    extern __shared__ __align__(16) unsigned char smem[];
    LookupLanesMem& M = reinterpret_cast<LookupLanesMem*>(smem)[threadIdx.x >> 5];
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    const uint32_t le = lt | (1u << lane);
    const SketchParams& p = db.sp;
    const uint32_t k = KC ? (uint32_t)KC : p.k;
    const uint32_t total = total_queries(Q);
    if (q0 >= total) return;
    const uint32_t nq = min(chunk, total - q0);
    const uint64_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarp = (gridDim.x * blockDim.x) >> 5;
    const TableProbe tp(db.fmt);
    const uint32_t lsz = db.jbits ? 4u : 8u;  // bytes per stored location
    if (lane == 0) M.seen = 0;

    for (uint64_t i0 = gw << batch_shift; i0 < nq; i0 += nwarp << batch_shift) {
        // one lane per query: size, status, sliding window
        const uint64_t i = i0 + lane;
        const bool mine = (lane >> batch_shift) == 0 && i < nq;
        const uint32_t q = q0 + (uint32_t)i;
        QueryIn in{};
        int status = Q_DONE;
        uint32_t n_win = 0, n_whole = 0, span = 0;
        uint64_t start = 0;
        if (mine) {
            in = query_in(Q, q);
            if (in.m1 < in.m0 || in.m1 - in.m0 > MAX_MATES) {
                status = Q_TOO_LARGE;
            } else {
                start = in.offs[in.m0];
                uint64_t o = start, sum = 0, wins = 0;
                for (uint32_t m = in.m0; m < in.m1; ++m) {
                    const uint64_t o2 = in.offs[m + 1];
                    const uint64_t L = o2 > o ? o2 - o : 0;
                    const uint32_t l = (uint32_t)min(L, (uint64_t)0x7FFFFFFF);  // more is too large anyway
                    sum += L;
                    wins += l < k ? 0u : (l - k + p.stride) / p.stride;
                    n_whole += l < p.w ? 0u : (l - p.w) / p.stride + 1;
                    o = o2;
                }
                if (wins > MC_MAX_QUERY_WINDOWS) status = Q_TOO_LARGE;
                else if (wins > WIN_A || sum > BUF_A) status = Q_ESCALATE;
                n_win = (uint32_t)wins;
                span = (uint32_t)min(sum, (uint64_t)0xFFFFFFFF);
            }
            if (status != Q_DONE) {
                meta[i] = make_uint4(ESCALATED, 0, 0, 0);
                if (status == Q_ESCALATE) ovf_list[atomicAdd(ovf_n, 1u)] = q;
                else atomicMax(Q.status, DEV_ERR_CAPACITY);
            }
        }
        for (uint32_t big = __ballot_sync(FULL_MASK, status == Q_TOO_LARGE); big; big &= big - 1)
            write_unclassified(Q, q0 + (uint32_t)i0 + __ffs(big) - 1);
        const uintptr_t first = reinterpret_cast<uintptr_t>(in.seq + start);
        const uint32_t shift = (uint32_t)(first & 15u);
        const bool active = mine && status == Q_DONE;
        const uint32_t n_ch = active && n_win ? (shift + span + 15) / 16 : 0u;
        const uint32_t n_it = active ? n_win : 0u;
        if (!active) n_whole = 0;
        M.q_list[lane] = M.q_locs[lane] = M.q_sect[lane] = 0;

        uint32_t todo = __ballot_sync(FULL_MASK, n_it > 0);
        while (todo) {
            // the group: queries from the first one left that fit together
            const bool left = (todo >> lane) & 1u;
            uint32_t s1 = left ? n_ch | (n_it << 16) : 0u;  // <= 32 * 66 chunks, 32 * 8 windows
            uint32_t inc = s1;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t x = __shfl_up_sync(FULL_MASK, inc, d);
                if ((int)lane >= d) inc += x;
            }
            const bool in_g = left && (inc & 0xFFFFu) <= LKL_CHUNKS && (inc >> 16) <= LKL_ITEMS;
            const uint32_t group = __ballot_sync(FULL_MASK, in_g);
            todo &= ~group;
            const uint32_t c0 = (inc - s1) & 0xFFFFu;  // first chunk (the group's lanes precede the others left)
            uint32_t wh = in_g ? n_whole : 0u;
            uint32_t wh_inc = wh;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t x = __shfl_up_sync(FULL_MASK, wh_inc, d);
                if ((int)lane >= d) wh_inc += x;
            }
            const uint32_t all_whole = __shfl_sync(FULL_MASK, wh_inc, 31);
            const uint32_t g_last = 31 - __clz(group);
            const uint32_t n_chunks = __shfl_sync(FULL_MASK, inc, g_last) & 0xFFFFu;
            const uint32_t n_items = __shfl_sync(FULL_MASK, inc, g_last) >> 16;
            const uint32_t rank = __popc(group & lt);

            __syncwarp();
            if (lane < LKL_WORDS) M.stage.starts[lane] = 0;
            __syncwarp();
            if (in_g) {
                M.stage.base[rank] = (uint64_t)(first - shift) - 16 * (uint64_t)c0;
                atomicOr(&M.stage.starts[c0 >> 5], 1u << (c0 & 31u));
                // its windows, whole ones first
                uint32_t whole_at = wh_inc - wh;
                uint32_t part_at = all_whole + ((inc - s1) >> 16) - (wh_inc - wh);
                uint32_t pos = c0 * 16 + shift;
                uint64_t o = start;
                for (uint32_t m = in.m0; m < in.m1; ++m) {
                    const uint64_t o2 = in.offs[m + 1];
                    const uint32_t L = o2 > o ? (uint32_t)(o2 - o) : 0u;  // <= BUF_A
                    for (uint32_t ws = 0; ws + k <= L; ws += p.stride) {
                        const uint32_t n_k = min(p.w, L - ws) - k + 1;
                        const uint32_t at = L - ws >= p.w ? whole_at++ : part_at++;
                        M.item[at] = (pos + ws) | (n_k << 13) | (lane << 23);
                    }
                    pos += L;
                    o = o2;
                }
            }
            __syncwarp();
            uint32_t bad = 0, ranks = 0;
#pragma unroll 1
            for (uint32_t r = 0; r * 32 < n_chunks; r += 4) {
                uint4 x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t w = M.stage.starts[min(r + u, LKL_WORDS - 1)];
                    const uint32_t c = (r + u) * 32 + lane;
                    if (c < n_chunks)
                        x[u] = __ldg(reinterpret_cast<const uint4*>(M.stage.base[ranks + __popc(w & le) - 1] +
                                                                    16 * (uint64_t)c));
                    ranks += __popc(w);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t c = (r + u) * 32 + lane;
                    if (c < n_chunks) {
                        uint32_t iv;
                        M.code[c] = encode16(x[u], iv);
                        M.inv[c] = (uint16_t)iv;
                        bad |= iv;
                    }
                }
            }
            const bool any_inv = __any_sync(FULL_MASK, bad != 0);
            __syncwarp();

            for (uint32_t r0 = 0; r0 < n_items; r0 += 32) {
                const uint32_t it = r0 + lane < n_items ? M.item[r0 + lane] : 0u;
                const uint32_t pos = it & 0x1FFFu, n_k = (it >> 13) & 0x3FFu, owner = it >> 23;
                uint32_t v[16], cnt;
                const bool ok = lane_sketch<KC, LKL_CAP>(M.code, M.inv, n_chunks, any_inv, pos, n_k, p, M.cand, v, cnt);
                uint32_t again = __ballot_sync(FULL_MASK, !ok);
                __syncwarp();
                // (the candidate buffer now takes the features' hashes)
#pragma unroll
                for (int x = 0; x < 16; ++x) M.hash[x * 32 + lane] = hash_h2(v[x]);
                while (again) {  // exact selection by the whole warp
                    const uint32_t l = __ffs(again) - 1;
                    again &= again - 1;
                    const uint32_t lpos = __shfl_sync(FULL_MASK, pos, l), lnk = __shfl_sync(FULL_MASK, n_k, l);
                    // address of staged position 0 of the lane's query
                    const uint64_t q_first = (uint64_t)(first - shift) - 16 * (uint64_t)c0;
                    const uint64_t a = __shfl_sync(FULL_MASK, q_first, __shfl_sync(FULL_MASK, owner, l)) + lpos;
                    const uint8_t* const sq[1] = {reinterpret_cast<const uint8_t*>(a)};
                    const uint64_t Ls[1] = {lnk + k - 1}, wss[1] = {0};
                    const bool on[1] = {true};
                    uint32_t f[1], c1[1];
                    warp_sketch_multi<R, 1, KC>(sq, Ls, wss, on, p, M.exact, f, c1);
                    if (lane < c1[0]) M.hash[lane * 32 + l] = hash_h2(f[0]);
                    if (lane == l) cnt = c1[0];
                    __syncwarp();
                }
                // Feature table probes: the aligned 16-byte pair of words
                // holding the home slot; the ordered probe stops at an empty
                // slot or a key >= h.  The probes that go on beyond their
                // pair (one in eight) are queued and shared out over the
                // lanes afterwards, so that a step waits for one load and
                // not for the longest probe of 32.
                uint32_t n_more = 0;
                const auto sectors = [&](uint64_t b) {
                    const uint64_t lo = (b >> 16) * lsz, hi = lo + (b & 0xFFFFu) * lsz - 1;
                    return (uint32_t)((hi >> 5) - (lo >> 5) + 1);
                };
                const auto queue = [&](bool on, uint32_t entry) {
                    const uint32_t b = __ballot_sync(FULL_MASK, on);
                    if (on) M.more[n_more + __popc(b & lt)] = (uint16_t)entry;
                    n_more += __popc(b);
                };
                if (cnt) atomicAdd(&M.q_list[owner], cnt << 16);
                const uint32_t most = __reduce_max_sync(FULL_MASK, cnt);
                uint32_t locs = 0, sect = 0;
#pragma unroll 1
                for (uint32_t h0 = 0; h0 < most; h0 += 8) {
                    uint32_t n_f = 0;
#pragma unroll 1
                    for (uint32_t b0 = h0; b0 < h0 + 8; b0 += LB) {
                        ulonglong2 pr[LB];
#pragma unroll
                        for (int b = 0; b < LB; ++b) {
                            const uint32_t home = tp.home(M.hash[(b0 + b) * 32 + lane]);
                            pr[b] = b0 + b < cnt ? __ldcg(reinterpret_cast<const ulonglong2*>(db.table) + (home >> 1))
                                                 : make_ulonglong2(0, 0);
                        }
#pragma unroll
                        for (int b = 0; b < LB; ++b) {
                            const uint32_t h = M.hash[(b0 + b) * 32 + lane];
                            const uint32_t odd = tp.home(h) & 1u;
                            uint64_t e = pr[b].x;
                            uint32_t what = odd ? 2u : tp.step(e, 0, h);
                            if (what == 2) {
                                e = pr[b].y;
                                what = tp.step(e, 1 - odd, h);
                            }
                            if (what == 1) {
                                const uint64_t bk = tp.bucket(e);
                                M.found[n_f * 32 + lane] = bk;
                                ++n_f;
                                locs += (uint32_t)bk & 0xFFFFu;
                                if (Q.counters) sect += sectors(bk);
                            }
                            queue(what == 2, lane | ((b0 + b) << 5));
                        }
                    }
                    // the lanes' entries take the next places of their
                    // queries' lists; consecutive lanes write consecutive
                    // entries
                    uint32_t inc = n_f;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const uint32_t x = __shfl_up_sync(FULL_MASK, inc, d);
                        if ((int)lane >= d) inc += x;
                    }
                    const uint32_t n_out = __shfl_sync(FULL_MASK, inc, 31), e_first = inc - n_f;
                    const uint32_t has = __ballot_sync(FULL_MASK, n_f > 0);
                    if (lane < 8) M.out_start[lane] = 0;
                    __syncwarp();
                    uint32_t to = 0;  // place of entry e of the output in the chunk's lists, minus e
                    if (n_f) {
                        const uint32_t at = atomicAdd(&M.q_list[owner], n_f) & 0xFFFFu;
                        to = (uint32_t)(i0 + owner) * list_cap + at - e_first;
                        atomicOr(&M.out_start[e_first >> 5], 1u << (e_first & 31u));
                        M.out_lane[__popc(has & lt)] = (uint8_t)lane;
                    }
                    __syncwarp();
                    uint32_t before = 0;
                    for (uint32_t r = 0; r * 32 < n_out; ++r) {
                        const uint32_t w = M.out_start[r];
                        const uint32_t e = r * 32 + lane;
                        const uint32_t src = M.out_lane[before + __popc(w & le) - 1];
                        const uint32_t ef = __shfl_sync(FULL_MASK, e_first, src), d0 = __shfl_sync(FULL_MASK, to, src);
                        if (e < n_out) glist[d0 + e] = M.found[(e - ef) * 32 + src];
                        before += __popc(w);
                    }
                    __syncwarp();
                }
                if (locs) atomicAdd(&M.q_locs[owner], locs);
                if (sect) atomicAdd(&M.q_sect[owner], sect);
                // entry: lane | feature << 5; the step is the pair after home's
                for (uint32_t step = 1; n_more; ++step) {
                    __syncwarp();
                    const uint32_t n_now = n_more;
                    n_more = 0;
                    for (uint32_t j0 = 0; j0 < n_now; j0 += 32) {
                        const uint32_t en = j0 + lane < n_now ? M.more[j0 + lane] : 0u;
                        bool over = true;
                        const uint32_t h = M.hash[en];  // [feature * 32 + lane]
                        const uint32_t home = tp.home(h);
                        const uint32_t d = 2 * step - (home & 1u);  // of the pair's first word
                        if (j0 + lane < n_now && d <= db.max_probe) {
                            const uint32_t qi = M.item[r0 + (en & 31u)] >> 23;
                            const ulonglong2 w =
                                __ldcg(reinterpret_cast<const ulonglong2*>(db.table) + ((uint64_t)(home >> 1) + step));
                            uint64_t e = w.x;
                            uint32_t what = tp.step(e, d, h);
                            if (what == 2 && d + 1 <= db.max_probe) {
                                e = w.y;
                                what = tp.step(e, d + 1, h);
                            }
                            if (what == 1) {
                                const uint64_t bk = tp.bucket(e);
                                const uint32_t at = atomicAdd(&M.q_list[qi], 1u) & 0xFFFFu;
                                glist[(uint32_t)(i0 + qi) * list_cap + at] = bk;
                                atomicAdd(&M.q_locs[qi], (uint32_t)bk & 0xFFFFu);
                                if (Q.counters) atomicAdd(&M.q_sect[qi], sectors(bk));
                            }
                            over = what != 2;
                        }
                        __syncwarp();  // the entries are read before their places are taken again
                        queue(!over, en);
                    }
                }
                __syncwarp();
            }
        }
        __syncwarp();
        if (active) {
            const uint32_t nm = in.m1 - in.m0;
            const uint32_t sp = nm <= 1 ? span : max(span, Q.max_insert);
            const uint32_t sws = sp >= k ? (sp - k + p.stride - 1) / p.stride + 1 : 0u;
            const uint32_t lf = M.q_list[lane];
            meta[i] = make_uint4(lf & 0xFFFFu, sws | ((lf >> 16) << META_FEAT_SHIFT), M.q_locs[lane], M.q_sect[lane]);
        }
        {
            const uint32_t most = __reduce_max_sync(FULL_MASK, active ? M.q_locs[lane] : 0u);
            if (lane == 0) note_widest(ovf_n + QC_WIDEST, most, M.seen);
        }
        __syncwarp();
    }
}

// Main path, part 2 (gather + score + label): one warp per query of the
// chunk, KA histogram slots per warp in shared memory.  Queries whose
// histogram does not fit are queued (chunk index) for the medium path.
template <int KA, int GB, class KeyT, class LocT>
__global__ void __launch_bounds__(CLS_WARPS * 32, 8) k_classify_score(ClassifyDb db, ClassifyQuery Q, uint32_t q0,
                                                                     uint32_t chunk, uint32_t list_cap,
                                                                     const uint64_t* __restrict__ glist,
                                                                     const uint4* __restrict__ meta,
                                                                     uint32_t* __restrict__ mid_list,
                                                                     uint32_t* __restrict__ mid_n) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t w = threadIdx.x >> 5;
    const uint32_t lane = lane_id();
    const size_t per_warp = scratch_bytes<uint16_t, KeyT>(KA, list_cap, 0, 0);
    const Scratch<uint16_t, KeyT> S = carve<uint16_t, KeyT>(smem + w * per_warp, KA, list_cap, 0, 0, WIN_A);
    Counters ctr;
    const uint32_t total = total_queries(Q);
    if (q0 >= total) return;
    const uint32_t nq = min(chunk, total - q0);
    const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarp = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i = gw; i < nq; i += nwarp) {
        const uint4 mt = meta[i];
        if (mt.x == ESCALATED) continue;
        // more locations than histogram slots: almost surely more distinct
        // locations than the histogram holds, so straight to the medium path
        if (mt.z > (uint32_t)KA) {
            if (lane == 0) mid_list[atomicAdd(mid_n, 1u)] = i;
            continue;
        }
        const uint64_t* src = glist + (uint64_t)i * list_cap;
        for (uint32_t j = lane; j < mt.x; j += 32) S.list[j] = __ldg(src + j);
        __syncwarp();
        const uint32_t q = q0 + i;
        if (query_score<GB, LocT>(db, Q, q, S, mt.x, meta_sws(mt), ctr) == Q_ESCALATE) {
            if (lane == 0) mid_list[atomicAdd(mid_n, 1u)] = i;
        } else {
            ctr.features += meta_feat(mt);
            ctr.found += mt.x;
            ctr.sectors += mt.w;
            ++ctr.queries;
        }
        __syncwarp();
    }
    flush_counters(Q, ctr, KC_SCORE);
}

// Queries of the chunk with h_lo < H <= h_hi gathered locations (h_lo = 0:
// no lower bound), not escalated: a warp takes groups of 2^shift <= 32
// consecutive queries from a counter (*ctr, zero before the launch), reads
// their metadata at once and takes those in range by ballot, so that warps
// that start late take fewer groups.  With mid_list, the queries beyond h_hi
// are queued there (chunk index) as they are met.
struct ChunkScan {
    uint32_t base, nq;  // first query of the current group, chunk size
    uint32_t shift;     // log2 of the queries per group
    uint32_t* ctr;      // next group
    uint4 mt;           // this lane's query of the group
    uint32_t todo;      // lanes of the group still to be processed
};

__device__ __forceinline__ ChunkScan chunk_scan(uint32_t nq, uint32_t shift, uint32_t* ctr) {
    ChunkScan it;
    it.nq = nq;
    it.shift = shift;
    it.ctr = ctr;
    it.base = 0;
    it.todo = 0;
    return it;
}

__device__ __forceinline__ bool next_chunk_query(ChunkScan& it, const uint4* __restrict__ meta, uint32_t h_lo,
                                                uint32_t h_hi, uint32_t* __restrict__ mid_list,
                                                uint32_t* __restrict__ mid_n, uint32_t& i, uint4& mt) {
    const uint32_t lane = lane_id();
    while (it.todo == 0) {
        uint32_t g = 0;
        if (lane == 0) g = atomicAdd(it.ctr, 1u);
        g = __shfl_sync(FULL_MASK, g, 0);
        const uint64_t first = (uint64_t)g << it.shift;
        if (first >= it.nq) return false;
        it.base = (uint32_t)first;
        const uint64_t qi = first + lane;
        it.mt = (lane >> it.shift) == 0 && qi < it.nq ? meta[qi] : make_uint4(ESCALATED, 0, 0, 0);
        const bool in = it.mt.x != ESCALATED && !(h_lo && it.mt.z <= h_lo);
        if (mid_list && in && it.mt.z > h_hi) mid_list[atomicAdd(mid_n, 1u)] = (uint32_t)qi;
        it.todo = __ballot_sync(FULL_MASK, in && it.mt.z <= h_hi);
    }
    const int l = __ffs(it.todo) - 1;
    it.todo &= it.todo - 1;
    i = it.base + (uint32_t)l;
    mt.x = __shfl_sync(FULL_MASK, it.mt.x, l);
    mt.y = __shfl_sync(FULL_MASK, it.mt.y, l);
    mt.z = __shfl_sync(FULL_MASK, it.mt.z, l);
    mt.w = __shfl_sync(FULL_MASK, it.mt.w, l);
    return true;
}

// ------------------------------------------------------------------
// Sort path: query steps 5-8 of Section 5.2 for a query of at most 32*E
// gathered locations, on one warp.  The paper compacts the gathered
// locations and sorts each read's segment (Sections 5.4-5.5); here one warp
// gathers the query's locations straight into registers (E per lane, all
// loads in flight at once), drops those that cannot matter, and sorts the
// rest with an in-register bitonic network to read off the window count
// statistic (runs of equal locations) and the sliding-window scores
// (Section 5.6: elements in [x, x + sws) of the sorted array).  Same outputs
// as query_score.
//
// Dropping locations.  Windows are grouped into blocks of 2^b >= sws, so a
// candidate's window range lies in its first window's block and the next
// one.  Counting the locations per (target, block) in a small table
// (colliding blocks share a counter, so a counter is never too low) bounds
// the score of every candidate whose range can hold location X from above by
// c(block of X) + max(c(block before), c(block after)).  With a threshold T,
// every location that counts towards a candidate of score >= T has a bound
// >= T; the others are dropped, and the scores of the candidates of score
// >= T stay exact while all others stay below T.  T is guessed from the
// largest bound; the guess is right if the top score s1 found this way puts
// the close threshold (the smallest score that matters for the label) at T
// or above, else the query is done once more with T = close(s1), which is
// then right because the top score is at least s1.  With the full top-m list
// requested the m-th score takes the place of the close threshold.
//
// What it saves, on 2 M pairs against the large database: of 495 locations
// per query 96 are sorted (one query in 2,000 is done twice); the 512 and
// 1024 classes take 3.30 and 3.23 ms against 4.96 and 7.28 ms with every
// location sorted.  Half of that is the gather (about 45 G sectors/s, the
// rate of random reads), the rest issue: about 1,500 warp instructions per
// query.  More resident warps help more than the next query's gather in
// flight behind the current one's sort (3.55 and 4.83 ms: its second buffer
// costs a quarter of the warps).

// Bitonic sort of 32*E keys held E per lane, element i = lane*E + r, into
// ascending order of i.  Mirror form of the network: each merge stage of
// block size K starts by comparing i with its mirror i ^ (K - 1) and goes on
// with half-cleaners i ^ J, J = K/4 .. 1, and every comparator puts the
// smaller key at the smaller index, so the steps within a lane's registers
// need no direction select.  Stages up to K = E stay in the lane's
// registers; the stages beyond run as a loop whose body holds one mirror
// step, the cross-lane half-cleaners (each guarded by the stage) and the
// E/2 .. 1 in-register half-cleaners, which keeps the code small.
template <int E, class T>
__device__ __forceinline__ void sort_in_lane_halves(T (&k)[E]) {
#pragma unroll
    for (int J = E >> 1; J > 0; J >>= 1) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
            if ((r & J) == 0) {
                const T a = k[r], b = k[r | J];
                k[r] = min(a, b);
                k[r | J] = max(a, b);
            }
        }
    }
}

template <int E, class T>
__device__ __forceinline__ void warp_bitonic_sort(T (&k)[E]) {
    const uint32_t lane = lane_id();
#pragma unroll
    for (int K = 2; K <= E; K <<= 1) {
#pragma unroll
        for (int r = 0; r < E; ++r) {
            if ((r & (K >> 1)) == 0) {
                const int o = r ^ (K - 1);
                const T a = k[r], b = k[o];
                k[r] = min(a, b);
                k[o] = max(a, b);
            }
        }
#pragma unroll
        for (int J = K >> 2; J > 0; J >>= 1) {
#pragma unroll
            for (int r = 0; r < E; ++r) {
                if ((r & J) == 0) {
                    const T a = k[r], b = k[r | J];
                    k[r] = min(a, b);
                    k[r | J] = max(a, b);
                }
            }
        }
    }
#pragma unroll 1
    for (uint32_t kl = 2; kl <= 32; kl <<= 1) {  // K = kl * E
        {
            // mirror partner of element (lane, r): lane ^ (kl - 1), register
            // E-1-r; the lower lane keeps the minimum.  As a mirror pair
            // (r, E-1-r) of this lane meets the pair (E-1-r, r) of the
            // partner, each register takes the partner's value first.
            const T up = (lane & (kl >> 1)) ? ~(T)0 : (T)0;  // the upper lane keeps the max
            const uint32_t lm = kl - 1;
            if (E == 1) {
                const T o = __shfl_xor_sync(FULL_MASK, k[0], lm);
                k[0] = up ? max(k[0], o) : min(k[0], o);
            }
#pragma unroll
            for (int r = 0; r < E / 2; ++r) {
                const T a = k[r], b = k[E - 1 - r];
                const T pa = __shfl_xor_sync(FULL_MASK, b, lm);  // partner's E-1-r
                const T pb = __shfl_xor_sync(FULL_MASK, a, lm);  // partner's r
                const T na = min(a, pa), nb = min(b, pb);
                k[r] = na ^ ((na ^ max(a, pa)) & up);
                k[E - 1 - r] = nb ^ ((nb ^ max(b, pb)) & up);
            }
        }
#pragma unroll
        for (int t = 3; t >= 0; --t) {  // lane distances kl/4 .. 1 (warp-uniform guard)
            const uint32_t lj = 1u << t;
            if (lj <= (kl >> 2)) {
                const T up = (lane & lj) ? ~(T)0 : (T)0;
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const T o = __shfl_xor_sync(FULL_MASK, k[r], lj);
                    const T n = min(k[r], o);
                    k[r] = n ^ ((n ^ max(k[r], o)) & up);
                }
            }
        }
        sort_in_lane_halves<E>(k);
    }
}

constexpr int SORT_WARPS = 4;           // warps per CTA of the sort path
constexpr int GU = 4;                   // gather steps unrolled together
constexpr uint32_t SMALL_SORT = 256;    // survivors that are sorted eight per lane
constexpr uint32_t QUEUED_MAX = 1024;   // locations of a queued query that a warp sorts
constexpr uint32_t NO_FILTER = 64;      // locations that are sorted without a look at the counts

// Per-warp shared memory of the sort path: the buckets' location indices,
// the bitmap of bucket starts in the flat list, the gathered locations, and
// three regions used in turn: `a` holds the
// block counters (16 bits), then the sorted survivors and their runs'
// locations; `b` the surviving locations, then the runs' first sorted indices
// (rs); `c` the counter slots, then the bounds, then the runs' scores.  When
// all the locations have to be sorted, they are so in place (raw) and `a`
// takes rs.  The gathered locations stay here rather than in registers: the
// loops over them then take H / 32 steps of a small body (unrolled over
// registers, a query missed the instruction cache all the way).
template <int E, class LocT>
struct SortMem {
    static constexpr uint32_t CAP = 32 * E;
    static constexpr uint32_t SURV = CAP < SMALL_SORT ? CAP : SMALL_SORT;
    static constexpr size_t BM_BYTES = align16((E + GU) * 4);
    static constexpr size_t RAW_BYTES = align16((CAP + 4) * sizeof(LocT));
    static constexpr size_t SURV_BYTES = align16(SURV * sizeof(LocT));
    static constexpr size_t U16_BYTES = align16((CAP + 4) * 2);
    static constexpr size_t A_BYTES = SURV_BYTES > U16_BYTES ? SURV_BYTES : U16_BYTES;
    static constexpr size_t B_BYTES = align16((SURV + 4) * 2) > SURV_BYTES ? align16((SURV + 4) * 2) : SURV_BYTES;
    uint64_t* adj;  // bucket b's first location minus its place in the flat list
    uint32_t* bm;   // bit i of word r: element 32 r + i of the flat list starts a bucket
    LocT* raw;      // the gathered locations, in the order of the flat list
    unsigned char *a, *b;
    uint16_t* c;
    __host__ __device__ static constexpr size_t bytes(uint32_t list_cap) {
        return align16((size_t)list_cap * 8) + BM_BYTES + RAW_BYTES + A_BYTES + B_BYTES + U16_BYTES;
    }
    __device__ __forceinline__ SortMem(unsigned char* p, uint32_t list_cap) {
        adj = reinterpret_cast<uint64_t*>(p);
        p += align16((size_t)list_cap * 8);
        bm = reinterpret_cast<uint32_t*>(p);
        p += BM_BYTES;
        raw = reinterpret_cast<LocT*>(p);
        p += RAW_BYTES;
        a = p;
        p += A_BYTES;
        b = p;
        p += B_BYTES;
        c = reinterpret_cast<uint16_t*>(p);
    }
    // adds one to counter s; a counter never passes 32 E < 65,536
    __device__ __forceinline__ void count(uint32_t s) const {
        atomicAdd(reinterpret_cast<uint32_t*>(a) + (s >> 1), 1u << ((s & 1u) * 16));
    }
};

// The block counters' view of a location: 2^b >= sws windows per block, the
// counters of a target's consecutive blocks next to each other.
template <class LocT>
struct BlockSlot {
    uint32_t jb, jmask, b;
    __device__ __forceinline__ uint32_t operator()(LocT x, uint32_t mask) const {
        const uint32_t t = (uint32_t)(x >> jb);
        return ((((uint32_t)x & jmask) >> b) + ((t * 0x9E3779B1u) >> 16)) & mask;
    }
};

// Starts gathering a query's H <= 32*E locations into M.raw: asynchronous
// copies of one location each, so that all of them are in flight at once
// without a register each (completion: cp_async_wait_all).  The bucket of an
// element is the number of bucket starts up to it, read off the bitmap.
template <int E, class LocT>
__device__ __forceinline__ void sort_gather(const ClassifyDb& db, const SortMem<E, LocT>& M, const uint64_t* src,
                                           uint32_t n_list, uint32_t H) {
    const uint32_t lane = lane_id();
    const LocT* __restrict__ locs = static_cast<const LocT*>(db.locs);
    __syncwarp();  // the last query is done with the working memory
#pragma unroll
    for (int r = 0; r < E + GU; r += 32)
        if (r + lane < E + GU) M.bm[r + lane] = 0;
    __syncwarp();
    uint32_t tot = 0;
    for (uint32_t base = 0; base < n_list; base += 32) {
        const uint32_t idx = base + lane;
        const uint64_t e = idx < n_list ? __ldg(src + idx) : 0;
        const uint32_t c = (uint32_t)e & 0xFFFFu;
        uint32_t inc = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t x = __shfl_up_sync(FULL_MASK, inc, d);
            if ((int)lane >= d) inc += x;
        }
        if (idx < n_list) {
            const uint32_t pre = tot + inc - c;
            M.adj[idx] = (e >> 16) - pre;
            atomicOr(&M.bm[pre >> 5], 1u << (pre & 31u));
        }
        tot += __shfl_sync(FULL_MASK, inc, 31);
    }
    __syncwarp();
    const uint32_t le = lanemask_lt() | (1u << lane);
    uint32_t before = 0;
#pragma unroll 1
    for (uint32_t x0 = lane, r = 0; r * 32 < H; r += GU, x0 += 32 * GU) {
#pragma unroll
        for (int u = 0; u < GU; ++u) {
            const uint32_t w = M.bm[r + u];
            const uint32_t x = x0 + 32 * u;
            if (x < H) {
                const LocT* g = locs + (M.adj[before + __popc(w & le) - 1] + x);
                const unsigned d = (unsigned)__cvta_generic_to_shared(M.raw + x);
                if (sizeof(LocT) == 4)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(g) : "memory");
                else
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(g) : "memory");
            }
            before += __popc(w);
        }
    }
    cp_async_commit();
}

// Sorts the n <= 32*EE locations src and leaves them ascending in dst.  A
// function of its own for every size: a query runs one of them, and the
// others do not lie between the steps before and after.
template <int EE, class LocT>
__device__ __noinline__ void sort_to(LocT* dst, const LocT* src, uint32_t n) {
    const uint32_t lane = lane_id();
    LocT k[EE];
#pragma unroll
    for (int r = 0; r < EE; ++r) {
        const uint32_t x = (uint32_t)r * 32 + lane;
        k[r] = x < n ? src[x] : ~(LocT)0;
    }
    warp_bitonic_sort<EE>(k);
    __syncwarp();  // (dst may still be read as counters)
    LocT* o = dst + lane * EE;
#pragma unroll
    for (int r = 0; r < EE; r += 2) {  // vector stores
        if (EE == 1)
            o[r] = k[r];
        else if (sizeof(LocT) == 8)
            *reinterpret_cast<ulonglong2*>(o + r) = make_ulonglong2((uint64_t)k[r], (uint64_t)k[(r + 1) % EE]);
        else
            *reinterpret_cast<uint2*>(o + r) = make_uint2((uint32_t)k[r], (uint32_t)k[(r + 1) % EE]);
    }
}

// Steps 6-8 of a query from its D distinct locations, ascending in loc, with
// rs[j] = number of gathered locations below loc[j] (D + 1 entries): scores,
// top m, label.  Locations may have been dropped with threshold T (see
// above).  Returns 0 with the outputs written, or, if T turns out too high,
// the threshold to use instead.  score: working memory of D entries.
template <class LocT, class IdxT>
__device__ __forceinline__ uint32_t score_runs(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                               const LocT* loc, const IdxT* rs, IdxT* score, uint32_t sws, uint32_t D,
                                               uint32_t T) {
    const uint32_t lane = lane_id();
    const uint32_t jb = sizeof(LocT) == 8 ? 32u : db.jbits;
    const uint32_t jmask = sizeof(LocT) == 8 ? 0xFFFFFFFFu : (1u << jb) - 1u;
    // Sliding-window scores (Section 5.6): the score of run j is the number
    // of sorted locations in [loc[j], hi], hi = loc[j] + sws - 1 cut at the
    // last window id of the target.  Runs have distinct locations, so at most
    // sws - 1 runs after j lie in that range; e is the first run beyond it
    // and the score is rs[e] - rs[j].  Four runs are checked per step (the
    // locations ascend, so the count of those <= hi is the advance).  The
    // first top-m round is folded in.
    const uint32_t w1 = sws ? sws - 1 : 0u;  // no wrap: stays in the run's target
    Cand best = Cand{0, 0xFFFFFFFFu, 0xFFFFFFFFu, 0};
    for (uint32_t j = lane; j < D; j += 32) {
        const LocT x = loc[j];
        const uint32_t win = (uint32_t)x & jmask;
        const LocT hi = x + min(w1, jmask - win);
        uint32_t e = j + 1;
        for (;;) {
            uint32_t adv = 0;
#pragma unroll
            for (int d = 0; d < 4; ++d) adv += (e + d < D && loc[e + d] <= hi) ? 1u : 0u;
            e += adv;
            if (adv < 4) break;
        }
        const uint32_t sc = (uint32_t)rs[e] - (uint32_t)rs[j];
        score[j] = (IdxT)sc;
        const Cand c = Cand{sc, (uint32_t)(x >> jb), win, 0};
        if (better(c, best)) best = c;
    }
    __syncwarp();

    // top m with one candidate per target (Section 4.2 / 5.6): rounds of
    // warp arg-max; the winner's target is excluded from later rounds by
    // zeroing the scores of its runs; the label is folded as in
    // query_score.  Unless the full top-m list is requested, later rounds
    // only matter for "close" candidates, so after the first round every
    // score below the close threshold is cleared at once.
    const int m = (int)Q.m;
    Cand mine = Cand{0, 0xFFFFFFFFu, 0, 0};
    uint32_t label = NO_TAXON, hits = 0, top = 0xFFFFFFFFu;
    uint64_t bar = 0;
    uint32_t prev_t = 0xFFFFFFFFu;
    for (int rd = 0; rd < m; ++rd) {
        if (rd) {
            best = Cand{0, 0xFFFFFFFFu, 0xFFFFFFFFu, 0};
            for (uint32_t j = lane; j < D; j += 32) {
                const uint32_t sc = score[j];
                if (sc == 0) continue;
                const LocT x = loc[j];
                const uint32_t t = (uint32_t)(x >> jb);
                if (t == prev_t) {
                    score[j] = 0;
                    continue;
                }
                const Cand c = Cand{sc, t, (uint32_t)x & jmask, 0};
                if (better(c, best)) best = c;
            }
        }
        {
            const uint32_t ms = __reduce_max_sync(FULL_MASK, best.score);
            const uint32_t mt = __reduce_min_sync(FULL_MASK, best.score == ms ? best.t : 0xFFFFFFFFu);
            const uint32_t mj =
                __reduce_min_sync(FULL_MASK, (best.score == ms && best.t == mt) ? best.j0 : 0xFFFFFFFFu);
            best = Cand{ms, mt, mj, 0};
        }
        if (Q.cands && best.score < T && T > 1) return 1;  // the full list needs every location
        if (best.score == 0) break;
        prev_t = best.t;
        if (Q.cands) {
            // last window of the range present: the location of the last run <= hi
            const LocT x0 = ((LocT)best.t << jb) | best.j0;
            const LocT hi = x0 + min(w1, jmask - best.j0);
            uint32_t lo = 0, up = D;  // first run beyond hi
            while (lo < up) {
                const uint32_t mid = (lo + up) >> 1;
                if (loc[mid] <= hi) lo = mid + 1; else up = mid;
            }
            best.j1 = (uint32_t)loc[lo - 1] & jmask;
        }
        if ((int)lane == rd) mine = best;
        if (rd == 0) {
            hits = best.score;
            top = best.t;
            bar = (uint64_t)(100 - Q.band) * hits;
            const uint32_t s_min = (uint32_t)((bar + 99) / 100);  // smallest score s with 100 s >= bar
            if (!Q.cands && s_min < T && T > 1) return max(s_min, 1u);
            if (hits >= Q.hits_min) label = top < db.n_targets ? db.taxon_of_target[top] : NO_TAXON;
            else if (!Q.cands) break;
            if (!Q.cands) {
                for (uint32_t j = lane; j < D; j += 32)
                    if (score[j] < s_min) score[j] = 0;
            }
        } else if (hits >= Q.hits_min && 100ull * best.score >= bar) {
            const uint32_t tx = best.t < db.n_targets ? db.taxon_of_target[best.t] : NO_TAXON;
            label = lca2(db, label, tx);
        } else if (!Q.cands) {
            break;
        }
        __syncwarp();
    }
    write_result(Q, q, label, hits, top, mine);
    return 0;
}

// Steps 5-8 of a query from its n locations, sorted in loc: runs of equal
// locations (the window count statistic of Section 5.6), then score_runs.
// Run j has location loc[j] and covers sorted indices [rs[j], rs[j+1]); the
// runs are written over the sorted locations: a run's index is at most its
// first element's, and a round's elements are read before its runs are
// written.  rs and score: working memory of n + 1 and n entries.
template <class LocT>
__device__ __forceinline__ uint32_t score_sorted(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q, LocT* loc,
                                                 uint16_t* rs, uint16_t* score, uint32_t sws, uint32_t n, uint32_t T,
                                                 uint32_t& distinct) {
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    uint32_t D = 0;
    LocT carry = 0;  // the element before the round's first
    for (uint32_t base = 0; base < n; base += 32) {
        const uint32_t i = base + lane;
        const LocT x = i < n ? loc[i] : (LocT)0;
        LocT prev = __shfl_up_sync(FULL_MASK, x, 1);
        if (lane == 0) prev = carry;
        carry = __shfl_sync(FULL_MASK, x, 31);
        const bool start = i < n && (i == 0 || x != prev);
        const uint32_t b = __ballot_sync(FULL_MASK, start);
        if (start) {
            const uint32_t pos = D + __popc(b & lt);
            loc[pos] = x;
            rs[pos] = (uint16_t)i;
        }
        D += __popc(b);
        __syncwarp();
    }
    if (lane == 0) rs[D] = (uint16_t)n;
    __syncwarp();
    distinct = D;
    return score_runs<LocT, uint16_t>(db, Q, q, loc, rs, score, sws, D, T);
}

// One query of H <= 32*E locations, gathered in M.raw.  Returns false if its
// survivors do not fit the small sorts and there is no sort of all the
// locations (64-bit locations): the query goes to the medium path.
template <int E, class LocT>
__device__ __forceinline__ bool query_sort(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                          const SortMem<E, LocT>& M, uint32_t sws, uint32_t H, bool counting,
                                          uint32_t& distinct) {
    using Mem = SortMem<E, LocT>;
    constexpr uint32_t MASK = Mem::CAP - 1;  // block counters
    const uint32_t lane = lane_id();
    const uint32_t lt = lanemask_lt();
    BlockSlot<LocT> bs;
    bs.jb = sizeof(LocT) == 8 ? 32u : db.jbits;
    bs.jmask = sizeof(LocT) == 8 ? 0xFFFFFFFFu : (1u << bs.jb) - 1u;
    bs.b = sws > 1 ? 32u - (uint32_t)__clz(sws - 1) : 0u;  // 2^b >= sws (sws < 2^17)
    const uint16_t* cnt = reinterpret_cast<const uint16_t*>(M.a);
    LocT* const raw = M.raw;
    LocT* surv = reinterpret_cast<LocT*>(M.b);
    // the counters of mc_classify_debug count all distinct locations
    uint32_t T = (H <= NO_FILTER || counting) ? 1u : 0u;
    do {
        const LocT* from = raw;
        uint32_t n = H;
        if (T != 1) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < E / 8; ++i) reinterpret_cast<uint4*>(M.a)[i * 32 + lane] = make_uint4(0, 0, 0, 0);
            __syncwarp();
#pragma unroll 2
            for (uint32_t x = lane; x < H; x += 32) {
                const uint32_t s = bs(raw[x], MASK);
                M.c[x] = (uint16_t)s;
                M.count(s);
            }
            __syncwarp();
            uint32_t most = 0;
#pragma unroll 2
            for (uint32_t x = lane; x < H; x += 32) {
                const uint32_t s = M.c[x];
                const uint32_t u = (uint32_t)cnt[s] + max(cnt[(s - 1) & MASK], cnt[(s + 1) & MASK]);
                most = max(most, u);
                M.c[x] = (uint16_t)u;
            }
            if (T == 0) {
                // aim a little below the close threshold of the largest
                // bound (for a full list, at a quarter of it), as the top
                // score may be lower than its bound
                most = __reduce_max_sync(FULL_MASK, most);
                const uint32_t close = ((100 - Q.band) * most + 99) / 100;
                T = max(Q.cands ? most / 4 : close - close / 8, 1u);
            }
            n = 0;
#pragma unroll 2
            for (uint32_t x0 = 0; x0 < H; x0 += 32) {
                const uint32_t x = x0 + lane;
                const bool in = x < H && M.c[x] >= T;
                const uint32_t v = __ballot_sync(FULL_MASK, in);
                const uint32_t at = n + __popc(v & lt);
                if (in && at < Mem::SURV) surv[at] = raw[x];
                n += __popc(v);
            }
            from = surv;
        }
        __syncwarp();
        LocT* loc = reinterpret_cast<LocT*>(M.a);
        uint16_t* rs = reinterpret_cast<uint16_t*>(M.b);
        if (n <= 32) {
            sort_to<1>(loc, from, n);
        } else if (n <= 64) {
            sort_to<2>(loc, from, n);
        } else if (n <= 128) {
            sort_to<4>(loc, from, n);
        } else if (E <= 8 || n <= SMALL_SORT) {
            sort_to<8>(loc, from, n);
        } else if (sizeof(LocT) == 4) {
            n = H;  // too many left: sort them all, in place
            T = 1;
            loc = raw;
            rs = reinterpret_cast<uint16_t*>(M.a);
            sort_to<E>(loc, (const LocT*)raw, n);
        } else {
            return false;
        }
        __syncwarp();
        T = score_sorted<LocT>(db, Q, q, loc, rs, M.c, sws, n, T, distinct);
    } while (T != 0);
    return true;
}

// A query of H <= 32 locations, one per lane: gather, sort, runs, scores and
// top m stay in registers (through the shared memory of the larger ones it
// takes twice the instructions).
template <class LocT>
__device__ __forceinline__ void query_small(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                            const uint64_t* src, uint32_t n_list, uint32_t sws, uint32_t H,
                                            uint32_t& distinct) {
    const uint32_t lane = lane_id();
    const uint32_t le = lanemask_lt() | (1u << lane);
    const uint32_t jb = sizeof(LocT) == 8 ? 32u : db.jbits;
    const uint32_t jmask = sizeof(LocT) == 8 ? 0xFFFFFFFFu : (1u << jb) - 1u;
    const uint64_t e = lane < n_list ? __ldg(src + lane) : 0;  // n_list <= H: no bucket is empty
    const uint32_t c = (uint32_t)e & 0xFFFFu;
    uint32_t pre = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(FULL_MASK, pre, d);
        if ((int)lane >= d) pre += x;
    }
    pre -= c;
    const uint32_t starts = __reduce_or_sync(FULL_MASK, lane < n_list ? 1u << (pre & 31u) : 0u);
    const uint64_t adj = __shfl_sync(FULL_MASK, (e >> 16) - pre, (__popc(starts & le) - 1) & 31);
    LocT k[1] = {~(LocT)0};
    if (lane < H) k[0] = __ldg(static_cast<const LocT*>(db.locs) + (adj + lane));
    warp_bitonic_sort<1>(k);
    const LocT x = k[0];
    const LocT prev = __shfl_up_sync(FULL_MASK, x, 1);
    const bool start = lane < H && (lane == 0 || x != prev);
    distinct = __popc(__ballot_sync(FULL_MASK, start));
    const uint32_t t = (uint32_t)(x >> jb), win = (uint32_t)x & jmask;
    const LocT hi = x + min(sws ? sws - 1 : 0u, jmask - win);
    uint32_t ub = 0;  // locations <= hi
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const LocT v = __shfl_sync(FULL_MASK, x, ub + s - 1);
        if (v <= hi) ub += s;
    }
    if (__shfl_sync(FULL_MASK, x, ub & 31u) <= hi) ++ub;
    ub = min(ub, H);
    uint32_t sc = start ? ub - lane : 0u;

    const int m = (int)Q.m;
    Cand mine = Cand{0, 0xFFFFFFFFu, 0, 0};
    uint32_t label = NO_TAXON, hits = 0, top = 0xFFFFFFFFu;
    uint64_t bar = 0;
    for (int rd = 0; rd < m; ++rd) {
        const uint32_t ms = __reduce_max_sync(FULL_MASK, sc);
        if (ms == 0) break;
        const uint32_t mt = __reduce_min_sync(FULL_MASK, sc == ms ? t : 0xFFFFFFFFu);
        if (Q.cands) {
            const uint32_t mj = __reduce_min_sync(FULL_MASK, sc == ms && t == mt ? win : 0xFFFFFFFFu);
            const uint32_t l = __ffs(__ballot_sync(FULL_MASK, sc == ms && t == mt && win == mj)) - 1;
            const uint32_t j1 = __shfl_sync(FULL_MASK, win, __shfl_sync(FULL_MASK, ub, l) - 1);
            if ((int)lane == rd) mine = Cand{ms, mt, mj, j1};
        }
        if (t == mt) sc = 0;  // one candidate per target
        if (rd == 0) {
            hits = ms;
            top = mt;
            bar = (uint64_t)(100 - Q.band) * hits;
            if (hits >= Q.hits_min) label = top < db.n_targets ? db.taxon_of_target[top] : NO_TAXON;
            else if (!Q.cands) break;
        } else if (hits >= Q.hits_min && 100ull * ms >= bar) {
            label = lca2(db, label, mt < db.n_targets ? db.taxon_of_target[mt] : NO_TAXON);
        } else if (!Q.cands) {
            break;
        }
    }
    write_result(Q, q, label, hits, top, mine);
}

// Resident CTAs per SM that the register budget of a sort-path kernel is
// sized for.  The classes are bound by issue and by the latency of the
// gather, and more warps help up to where registers spill in the loops
// (sort256: 319 us at 8, 300 at 10 CTAs, 64-bit locations 381 at 5, 336 at 7;
// sort512: 3.28 ms at 8, 3.33 at 9).
template <int E, class LocT>
constexpr int sort_min_ctas() {
    return sizeof(LocT) == 8 ? (E == 8 ? 7 : (E == 16 ? 4 : 2)) : (E == 8 ? 10 : (E == 16 ? 8 : (E == 32 ? 5 : 3)));
}

// Sort path over the chunk's queries with h_lo < H <= 32*E gathered
// locations; with last (the largest class), larger ones are queued for the
// medium path.
template <int E, class LocT, bool COUNTING>
__global__ void __launch_bounds__(SORT_WARPS * 32, sort_min_ctas<E, LocT>())
    k_classify_sort(ClassifyDb db, ClassifyQuery Q, uint32_t q0, uint32_t chunk, uint32_t list_cap,
                    const uint64_t* __restrict__ glist, const uint4* __restrict__ meta, uint32_t h_lo, bool last,
                    uint32_t group_shift, uint32_t* __restrict__ mid_list, uint32_t* __restrict__ mid_n,
                    uint32_t* __restrict__ group_ctr, const uint32_t* __restrict__ widest) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t w = threadIdx.x >> 5;
    const SortMem<E, LocT> M(smem + w * SortMem<E, LocT>::bytes(list_cap), list_cap);
    __shared__ unsigned long long tally[COUNTING ? SORT_WARPS : 1][6];
    if (COUNTING && lane_id() < 6) tally[w][lane_id()] = 0;
    // the next size class, which shares no data with this one, may start
    // while this one's last queries finish
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t total = total_queries(Q);
    if (q0 < total && (h_lo == 0 || *widest > h_lo)) {
        ChunkScan it = chunk_scan(min(chunk, total - q0), group_shift, group_ctr);
        uint32_t i;
        uint4 mt;
        while (next_chunk_query(it, meta, h_lo, 32u * E, last ? mid_list : nullptr, mid_n, i, mt)) {
            const uint64_t* src = glist + (uint64_t)i * list_cap;
            uint32_t distinct;
            bool done = true;
            if ((E == 8 || (E == 32 && sizeof(LocT) == 8)) && mt.z <= 32) {
                query_small<LocT>(db, Q, q0 + i, src, mt.x, meta_sws(mt), mt.z, distinct);
            } else {
                sort_gather<E>(db, M, src, mt.x, mt.z);
                cp_async_wait_all();
                __syncwarp();
                done = query_sort<E>(db, Q, q0 + i, M, meta_sws(mt), mt.z, COUNTING, distinct);
            }
            if (!done) {
                if (lane_id() == 0) mid_list[atomicAdd(mid_n, 1u)] = i;
            } else if (COUNTING) {
                tally_query(tally[w], mt, distinct);
            }
        }
        if (COUNTING) flush_tally(Q, tally[w], E == 8 ? 1 : (E == 16 ? 2 : (E == 32 ? 3 : 6)));
    }
    // Launched as a programmatic dependent of the medium path or of another
    // size class, this kernel may run alongside it; waiting for that grid
    // before exiting makes this kernel's completion imply the other's, so
    // that later work in the stream or graph never overtakes it.  A no-op
    // for an ordinary launch.
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Queries that the hash path's score kernel or a small sort_max leaves, as
// far as a warp can sort them: up to 1,024 locations, a warp each, off the
// queue mid_list; the rest go on to the medium path's CTAs (rest_list).
// There are many of them where the tuning draws the line low, and a CTA for
// each is slow (200,000 mixed reads, 1,000 genomes, sort_max 256: 4.66 ms, here
// 0.98; score_mode 2 with 256 slots: 4.87 ms, here 1.22).  Lines of 1,024 leave
// few that a warp could take, and the kernel is not launched.
template <class LocT, bool COUNTING>
__global__ void __launch_bounds__(SORT_WARPS * 32, sort_min_ctas<32, LocT>())
    k_sort_queued(ClassifyDb db, ClassifyQuery Q, uint32_t q0, uint32_t list_cap, const uint64_t* __restrict__ glist,
                  const uint4* __restrict__ meta, const uint32_t* __restrict__ mid_list,
                  const uint32_t* __restrict__ mid_n, uint32_t* __restrict__ work, uint32_t* __restrict__ rest_list,
                  uint32_t* __restrict__ rest_n) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5;
    const SortMem<32, LocT> M(smem + w * SortMem<32, LocT>::bytes(list_cap), list_cap);
    __shared__ unsigned long long tally[COUNTING ? SORT_WARPS : 1][6];
    if (COUNTING && lane < 6) tally[w][lane] = 0;
    const uint32_t n = *mid_n;
    for (;;) {
        uint32_t k = 0;
        if (lane == 0) k = atomicAdd(work, 1u);
        k = __shfl_sync(FULL_MASK, k, 0);
        if (k >= n) break;
        const uint32_t i = mid_list[k];
        const uint4 mt = meta[i];
        uint32_t distinct = 0;
        bool done = false;
        if (mt.z <= QUEUED_MAX) {
            sort_gather<32>(db, M, glist + (uint64_t)i * list_cap, mt.x, mt.z);
            cp_async_wait_all();
            __syncwarp();
            done = query_sort<32>(db, Q, q0 + i, M, meta_sws(mt), mt.z, COUNTING, distinct);
        }
        if (!done) {
            if (lane == 0) rest_list[atomicAdd(rest_n, 1u)] = i;
        } else if (COUNTING) {
            tally_query(tally[w], mt, distinct);
        }
    }
    if (COUNTING) {
        flush_tally(Q, tally[w], KC_MEDIUM);
        if (lane == 0) atomicAdd(Q.counters + 6, tally[w][5]);
    }
}

// ------------------------------------------------------------------
// Queries beyond the sort path's size classes: one CTA per query.  All its
// threads gather, count by block and drop locations as in query_sort, with
// the two passes over the locations both reading them from global memory
// (there may be any number); one warp then sorts and scores the survivors.
// More than BLK_DISTINCT distinct survivors (which takes hundreds of equally
// good targets) are left to the histogram code of one warp.
//
// One warp per query with a histogram took 0.6 ms for the slowest of a
// launch of 2^20 pairs, whatever the others did (large database, 2 launches
// 1.24 ms, here 0.71), and 5,000 reads of 1 to 6 kbp took 9.05 ms on
// global-memory histograms, here 0.72.
constexpr int BLK_THREADS = 256;
constexpr int BLK_WARPS = BLK_THREADS / 32;
constexpr uint32_t BLK_LIST = MC_MAX_QUERY_WINDOWS * MAX_S;  // buckets of one query
constexpr uint32_t BLK_CNT = 4096;                           // block counters
constexpr uint32_t BLK_HASH = 4096;                          // slots of the distinct survivors,
constexpr uint32_t BLK_DISTINCT = 2048;                      // of which as many are used (what a warp sorts)
constexpr int BLK_CTAS = 2;                                  // resident per SM
constexpr int BLK_STEP = 8;                                  // consecutive locations per thread and step

// The block counters and the sorted distinct survivors.  With 64-bit locations
// the survivors take the counters' place, without which two CTAs do not fit
// an SM (a query that is done again then counts again: 2 to 6 us).
template <class LocT>
struct BlockCounters {
    uint32_t cnt[BLK_CNT];
    LocT loc[BLK_DISTINCT];
};
template <>
struct BlockCounters<uint64_t> {
    union {
        uint32_t cnt[BLK_CNT];
        uint64_t loc[BLK_DISTINCT];
    };
};

template <class LocT>
struct BlockMem : BlockCounters<LocT> {
    uint64_t list[BLK_LIST];      // found buckets, offset << 16 | size
    uint32_t pre[BLK_LIST + 4];   // exclusive prefix of their sizes
    union {
        LocT key[BLK_HASH];       // the distinct survivors, hashed (times: how often each was gathered)
        struct {                  // (before them) the lookup's windows:
            uint64_t waddr[MC_MAX_QUERY_WINDOWS];  // address of the first base,
            uint32_t wnk[MC_MAX_QUERY_WINDOWS];    // k-mers, features
            uint32_t wcnt[MC_MAX_QUERY_WINDOWS];
            uint32_t cand[BLK_WARPS][32];
        };
    };
    uint32_t times[BLK_HASH];
    uint32_t rs[BLK_DISTINCT + 4];
    union {
        uint32_t score[BLK_DISTINCT + 4];
        uint32_t feat[BLK_LIST];  // (before the scores) the windows' features
    };
    uint32_t part[BLK_WARPS];     // block-wide scan and maximum
    uint32_t n_list, sect, n, T, n_win, sws, n_feat, work;
    int status;
};

// Two CTAs within 196 KB, the largest shared memory of an SM but one, leave it
// 60 KB of L1 instead of 28 (5,000 reads of 1 to 6 kbp: 0.72 ms instead of
// 0.87).
static_assert(BLK_CTAS * (sizeof(BlockMem<uint32_t>) + 1024) <= 196 * 1024, "shared memory of an SM");
static_assert(BLK_CTAS * (sizeof(BlockMem<uint64_t>) + 1024) <= 228 * 1024, "shared memory of an SM");

// f(location) for every location of the query's n_list buckets (H in all).
template <class LocT, class F>
__device__ __forceinline__ void block_for_each(const ClassifyDb& db, const BlockMem<LocT>& B, uint32_t n_list,
                                               uint32_t H, F f) {
    const LocT* __restrict__ locs = static_cast<const LocT*>(db.locs);
    for (uint32_t x0 = threadIdx.x * BLK_STEP; x0 < H; x0 += BLK_THREADS * BLK_STEP) {
        uint32_t lo = 0, hi = n_list;  // last bucket with pre <= x0
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (B.pre[mid] <= x0) lo = mid; else hi = mid;
        }
        LocT v[BLK_STEP];
#pragma unroll
        for (int u = 0; u < BLK_STEP; ++u) {
            const uint32_t x = x0 + u;
            v[u] = 0;
            if (x < H) {
                while (B.pre[lo + 1] <= x) ++lo;
                v[u] = __ldcg(locs + (B.list[lo] >> 16) + (x - B.pre[lo]));
            }
        }
#pragma unroll
        for (int u = 0; u < BLK_STEP; ++u)
            if (x0 + u < H) f(v[u]);
    }
}

// The block counters once more, for a query that is done again (out of line:
// one in thousands).  Between barriers, ends with one.
template <class LocT>
__device__ __noinline__ void block_count_again(const ClassifyDb& db, BlockMem<LocT>& B, uint32_t n_list, uint32_t H,
                                               const BlockSlot<LocT>& bs) {
    for (uint32_t i = threadIdx.x; i < BLK_CNT; i += BLK_THREADS) B.cnt[i] = 0;
    __syncthreads();
    block_for_each(db, B, n_list, H, [&](LocT x) { atomicAdd(&B.cnt[bs(x, BLK_CNT - 1)], 1u); });
    __syncthreads();
}

// Steps 5-8 of the query whose n_list buckets are in B.list, by the whole
// CTA (called between barriers; ends with one).  The surviving locations are
// made distinct by a hash table before they are sorted: repeats and long
// queries gather the same ones many times.  False: more than d_max of them.
template <class LocT>
__device__ __forceinline__ bool block_score(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                            BlockMem<LocT>& B, uint32_t n_list, uint32_t sws, uint32_t d_max,
                                            uint32_t& H_out, uint32_t& distinct) {
    constexpr uint32_t MASK = BLK_CNT - 1;
    const uint32_t tid = threadIdx.x, lane = lane_id(), w = tid >> 5;
    BlockSlot<LocT> bs;
    bs.jb = sizeof(LocT) == 8 ? 32u : db.jbits;
    bs.jmask = sizeof(LocT) == 8 ? 0xFFFFFFFFu : (1u << bs.jb) - 1u;
    bs.b = sws > 1 ? 32u - (uint32_t)__clz(sws - 1) : 0u;
    // exclusive prefix of the bucket sizes: eight buckets per thread
    constexpr uint32_t PER = BLK_LIST / BLK_THREADS;
    uint32_t sum = 0;
    for (uint32_t i = tid * PER; i < min((tid + 1) * PER, n_list); ++i) sum += (uint32_t)B.list[i] & 0xFFFFu;
    uint32_t inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(FULL_MASK, inc, d);
        if ((int)lane >= d) inc += x;
    }
    if (lane == 31) B.part[w] = inc;
    for (uint32_t i = tid; i < BLK_CNT; i += BLK_THREADS) B.cnt[i] = 0;
    __syncthreads();
    uint32_t H = 0, at = inc - sum;
    for (uint32_t i = 0; i < BLK_WARPS; ++i) {
        if (i < w) at += B.part[i];
        H += B.part[i];
    }
    for (uint32_t i = tid * PER; i < min((tid + 1) * PER, n_list); ++i) {
        B.pre[i] = at;
        at += (uint32_t)B.list[i] & 0xFFFFu;
    }
    if (tid == 0) B.pre[n_list] = H;
    H_out = H;
    __syncthreads();
    uint32_t T = Q.counters ? 1u : 0u;
    if (T == 0) {
        block_for_each(db, B, n_list, H, [&](LocT x) { atomicAdd(&B.cnt[bs(x, MASK)], 1u); });
        __syncthreads();
        uint32_t most = 0;
        for (uint32_t s = tid; s < BLK_CNT; s += BLK_THREADS)
            if (B.cnt[s]) most = max(most, B.cnt[s] + max(B.cnt[(s - 1) & MASK], B.cnt[(s + 1) & MASK]));
        most = __reduce_max_sync(FULL_MASK, most);
        if (lane == 0) B.part[w] = most;
        __syncthreads();
        for (uint32_t i = 0; i < BLK_WARPS; ++i) most = max(most, B.part[i]);
        const uint64_t close = ((uint64_t)(100 - Q.band) * most + 99) / 100;
        T = max(Q.cands ? most / 4 : (uint32_t)(close - close / 8), 1u);
    }
    constexpr LocT EMPTY = KeyCodec<LocT>::empty();
    for (;;) {
        for (uint32_t i = tid; i < BLK_HASH; i += BLK_THREADS) {
            B.key[i] = EMPTY;
            B.times[i] = 0;
        }
        if (tid == 0) B.n = 0;
        __syncthreads();
        block_for_each(db, B, n_list, H, [&](LocT x) {
            if (T > 1) {
                const uint32_t s = bs(x, MASK);
                if (B.cnt[s] + max(B.cnt[(s - 1) & MASK], B.cnt[(s + 1) & MASK]) < T) return;
            }
            // (the threads together pass the limit by at most one each, so
            // the table never fills)
            if (*(volatile uint32_t*)&B.n > d_max) return;
            int fresh = -1;
            hist_insert(B.key, B.times, BLK_HASH - 1, x, fresh);
            if (fresh >= 0) atomicAdd(&B.n, 1u);
        });
        __syncthreads();
        const uint32_t D = B.n;
        __syncthreads();
        if (D > d_max) return false;
        if (tid == 0) B.n = 0;
        __syncthreads();
        for (uint32_t i = tid; i < BLK_HASH; i += BLK_THREADS)
            if (B.key[i] != EMPTY) B.loc[atomicAdd(&B.n, 1u)] = B.key[i];
        __syncthreads();
        if (w == 0) {
            const LocT* from = B.loc;  // sorted in place
            if (D <= 32) sort_to<1>(B.loc, from, D);
            else if (D <= 64) sort_to<2>(B.loc, from, D);
            else if (D <= 256) sort_to<8>(B.loc, from, D);
            else if (D <= 512) sort_to<16>(B.loc, from, D);
            else if (D <= 1024) sort_to<32>(B.loc, from, D);
            else sort_to<64>(B.loc, from, D);
            __syncwarp();
            uint32_t before = 0;
            for (uint32_t j0 = 0; j0 < D; j0 += 32) {
                const uint32_t j = j0 + lane;
                uint32_t c = j < D ? hist_count(B.key, B.times, BLK_HASH - 1, B.loc[j]) : 0u;
                uint32_t pre = c;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t x = __shfl_up_sync(FULL_MASK, pre, d);
                    if ((int)lane >= d) pre += x;
                }
                if (j < D) B.rs[j] = before + pre - c;
                before += __shfl_sync(FULL_MASK, pre, 31);
            }
            if (lane == 0) B.rs[D] = before;
            __syncwarp();
            const uint32_t t2 = score_runs<LocT, uint32_t>(db, Q, q, B.loc, B.rs, B.score, sws, D, T);
            if (lane == 0) B.T = t2;
        }
        __syncthreads();
        T = B.T;
        distinct = D;
        if (T == 0) return true;
        if (sizeof(LocT) == 8 && T > 1) block_count_again<LocT>(db, B, n_list, H, bs);
    }
}

// Medium path: the queries queued by the hash path's score kernel or the
// sort path's classes, less those that k_sort_queued took; one CTA each (work
// queue), the bucket list taken
// over from the lookup; queries of more than MED_DISTINCT distinct locations
// go to the large path.
template <class LocT>
__global__ void __launch_bounds__(BLK_THREADS, BLK_CTAS) k_classify_medium(ClassifyDb db, ClassifyQuery Q, uint32_t q0,
                                                                   uint32_t list_cap,
                                                                   const uint64_t* __restrict__ glist,
                                                                   const uint4* __restrict__ meta,
                                                                   const uint32_t* __restrict__ mid_list,
                                                                   const uint32_t* __restrict__ mid_n,
                                                                   uint32_t* __restrict__ mid_work,
                                                                   uint32_t* __restrict__ ovf_list,
                                                                   uint32_t* __restrict__ ovf_n) {
    extern __shared__ __align__(16) unsigned char smem[];
    BlockMem<LocT>& B = *reinterpret_cast<BlockMem<LocT>*>(smem);
    // a kernel launched after this one with programmatic stream
    // serialization (a sort-path class, which shares no data with this one)
    // may start while this one's few long queries finish
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t n = *mid_n;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) B.work = atomicAdd(mid_work, 1u);
        __syncthreads();
        const uint32_t k = B.work;
        if (k >= n) break;
        const uint32_t i = mid_list[k];
        const uint4 mt = meta[i];
        const uint64_t* src = glist + (uint64_t)i * list_cap;
        for (uint32_t j = threadIdx.x; j < mt.x; j += BLK_THREADS) B.list[j] = __ldg(src + j);
        __syncthreads();
        uint32_t H = 0;
        uint32_t distinct = 0;
        const bool done = block_score<LocT>(db, Q, q0 + i, B, mt.x, meta_sws(mt), MED_DISTINCT, H, distinct);
        if (!done && threadIdx.x == 0) ovf_list[atomicAdd(ovf_n, 1u)] = q0 + i;
        if (Q.counters && done && threadIdx.x < 32) {
            Counters ctr;
            ctr.locations = H;
            ctr.distinct = distinct;
            ctr.features = meta_feat(mt);
            ctr.found = mt.x;
            ctr.sectors = mt.w;
            ctr.queries = 1;
            flush_counters(Q, ctr, KC_MEDIUM);
            if (threadIdx.x == 0) atomicAdd(Q.counters + 6, 1ull);
        }
    }
}

// Windows, sketches and table probes of a query of the large path by the
// whole CTA: fills B.list, B.n_list, B.sws, B.n_feat, B.sect; B.status is
// Q_DONE, or else the query is beyond the large path's limits.  Ends with a
// barrier.
template <int R, int KC, class LocT>
__device__ __forceinline__ void block_lookup(const ClassifyDb& db, const ClassifyQuery& Q, uint32_t q,
                                             BlockMem<LocT>& B) {
    const SketchParams& p = db.sp;
    const uint32_t tid = threadIdx.x, lane = lane_id(), w = tid >> 5;
    const uint32_t k = KC ? (uint32_t)KC : p.k;
    if (w == 0) {  // lane i holds mate i
        const QueryIn in = query_in(Q, q);
        const bool mates_ok = in.m1 >= in.m0 && in.m1 - in.m0 <= MAX_MATES;
        const uint32_t nm = mates_ok ? in.m1 - in.m0 : 0u;
        const uint64_t o = mates_ok && lane <= nm ? in.offs[in.m0 + lane] : 0;
        const uint64_t o_next = __shfl_down_sync(FULL_MASK, o, 1);
        const uint64_t L = (lane < nm && o_next > o) ? o_next - o : 0;
        const uint64_t nw = num_windows(L, k, p.stride);
        const uint64_t span = warp_sum_u64(L), n_win = warp_sum_u64(nw);
        const bool fits = mates_ok && n_win <= MC_MAX_QUERY_WINDOWS && span <= BUF_B;
        if (fits) {
            uint32_t off = (uint32_t)L, wat = (uint32_t)nw;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t x = __shfl_up_sync(FULL_MASK, off, d), y = __shfl_up_sync(FULL_MASK, wat, d);
                if ((int)lane >= d) {
                    off += x;
                    wat += y;
                }
            }
            off -= (uint32_t)L;
            wat -= (uint32_t)nw;
            const uint64_t base = (uint64_t)(uintptr_t)in.seq + __shfl_sync(FULL_MASK, o, 0) + off;
            for (uint32_t j = 0; j < (uint32_t)nw; ++j) {
                const uint32_t ws = j * p.stride;
                B.waddr[wat + j] = base + ws;
                B.wnk[wat + j] = min(p.w, (uint32_t)L - ws) - k + 1;
            }
        }
        if (lane == 0) {
            const uint64_t sp = nm <= 1 ? span : (span > Q.max_insert ? span : (uint64_t)Q.max_insert);
            B.status = fits ? Q_DONE : Q_TOO_LARGE;
            B.n_win = fits ? (uint32_t)n_win : 0u;
            B.sws = fits && sp >= k ? (uint32_t)((sp - k + p.stride - 1) / p.stride + 1) : 0u;
            B.n_list = B.n_feat = B.sect = 0;
        }
    }
    __syncthreads();
    const uint32_t n_win = B.n_win;
    for (uint32_t j = w; j < n_win; j += BLK_WARPS) {
        const uint8_t* const sq[1] = {reinterpret_cast<const uint8_t*>(B.waddr[j])};
        const uint64_t Ls[1] = {B.wnk[j] + k - 1}, wss[1] = {0};
        const bool on[1] = {true};
        uint32_t f[1], c[1];
        warp_sketch_multi<R, 1, KC>(sq, Ls, wss, on, p, B.cand[w], f, c);
        if (lane < c[0]) B.feat[j * p.s + lane] = f[0];
        if (lane == 0) {
            B.wcnt[j] = c[0];
            atomicAdd(&B.n_feat, c[0]);
        }
        __syncwarp();
    }
    __syncthreads();
    const TableProbe tp(db.fmt);
    const uint32_t lsz = sizeof(LocT);
    for (uint32_t x = tid; x < n_win * p.s; x += BLK_THREADS) {
        const uint32_t j = x / p.s;
        if (x - j * p.s >= B.wcnt[j]) continue;
        const uint32_t h = hash_h2(B.feat[x]);
        const uint64_t home = tp.home(h);
        const uint64_t* t = db.table + home;
        for (uint32_t d = 0; d <= db.max_probe; ++d) {
            const uint64_t e = __ldcg(t + d);
            const uint32_t what = tp.step(e, d, h);
            if (what == 2) continue;
            if (what == 1) {
                const uint64_t bk = tp.bucket(e);
                B.list[atomicAdd(&B.n_list, 1u)] = bk;
                const uint64_t lo = (bk >> 16) * lsz, hi = lo + (bk & 0xFFFFu) * lsz - 1;
                atomicAdd(&B.sect, (uint32_t)((hi >> 5) - (lo >> 5) + 1));
            }
            break;
        }
    }
    __syncthreads();
}

// Large path: queries with too many windows or bases for the lookup kernels
// and those that the medium path does not hold (the queue ovf_list), or, in a
// launch of few queries (ovf_list null), all of them; one CTA each; what does not
// fit the CTA's memory is processed by one warp with working memory in
// global scratch (one piece per CTA).
template <int R, int KC, class LocT>
__global__ void __launch_bounds__(BLK_THREADS, BLK_CTAS) k_classify_large(ClassifyDb db, ClassifyQuery Q,
                                                                   const uint32_t* __restrict__ ovf_list,
                                                                   const uint32_t* __restrict__ ovf_n,
                                                                   uint32_t* __restrict__ work,
                                                                   unsigned char* __restrict__ scratch,
                                                                   size_t per_cta) {
    extern __shared__ __align__(16) unsigned char smem[];
    BlockMem<LocT>& B = *reinterpret_cast<BlockMem<LocT>*>(smem);
    const uint32_t n = ovf_list ? *ovf_n : total_queries(Q);
    for (uint32_t turn = 0;; ++turn) {
        __syncthreads();
        if (threadIdx.x == 0) B.work = ovf_list ? atomicAdd(work, 1u) : turn * gridDim.x + blockIdx.x;
        __syncthreads();
        const uint32_t i = B.work;
        if (i >= n) break;
        const uint32_t q = ovf_list ? ovf_list[i] : i;
        block_lookup<R, KC, LocT>(db, Q, q, B);
        bool done = false;
        uint32_t H = 0, distinct = 0;
        if (B.status == Q_DONE) done = block_score<LocT>(db, Q, q, B, B.n_list, B.sws, BLK_DISTINCT, H, distinct);
        if (threadIdx.x < 32) {
            Counters ctr;
            if (done) {
                ctr.features = B.n_feat;
                ctr.locations = H;
                ctr.distinct = distinct;
                ctr.found = B.n_list;
                ctr.sectors = B.sect;
                ctr.queries = 1;
            } else {
                const Scratch<uint32_t> S = carve<uint32_t>(scratch + blockIdx.x * per_cta, KB_SLOTS, LIST_B, LIST_B,
                                                            BUF_B, MC_MAX_QUERY_WINDOWS);
                if (process_query<R, KC, LocT>(db, Q, q, S, ctr) != Q_DONE) {
                    write_unclassified(Q, q);
                    if (threadIdx.x == 0) atomicMax(Q.status, DEV_ERR_CAPACITY);
                }
            }
            if (Q.counters) {
                flush_counters(Q, ctr, KC_LARGE);
                if (threadIdx.x == 0) atomicAdd(Q.counters + 3, 1ull);
            }
        }
    }
}


constexpr uint32_t CHUNK = CLASSIFY_CHUNK;

using QueuedKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, const uint64_t*, const uint4*,
                              const uint32_t*, const uint32_t*, uint32_t*, uint32_t*, uint32_t*);

using LookupKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, uint32_t, uint64_t*, uint4*, uint32_t*,
                              uint32_t*);
using ScoreKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, uint32_t, const uint64_t*, const uint4*,
                             uint32_t*, uint32_t*);
using LargeKernel = void (*)(ClassifyDb, ClassifyQuery, const uint32_t*, const uint32_t*, uint32_t*, unsigned char*,
                             size_t);
using MediumKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, const uint64_t*, const uint4*,
                              const uint32_t*, const uint32_t*, uint32_t*, uint32_t*, uint32_t*);

using LookupLanesKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, uint32_t, uint64_t*, uint4*,
                                   uint32_t*, uint32_t*, uint32_t);

template <int R, int KC>
LookupLanesKernel lookup_lanes_for_lb(uint32_t lb) {
    if (lb == 2) return k_lookup_lanes<R, KC, 2>;
    if (lb == 8) return k_lookup_lanes<R, KC, 8>;
    return k_lookup_lanes<R, KC, 4>;
}

// One window per lane (sketch sizes up to 16), or nullptr.
LookupLanesKernel pick_lookup_lanes(const SketchParams& sp, uint32_t lb) {
    if (sp.s > LS_MAX_S) return nullptr;
    const int r = sketch_r_for(sp.w);
    const bool k16 = sp.k == 16;
    if (r == 4) return k16 ? lookup_lanes_for_lb<4, 16>(lb) : lookup_lanes_for_lb<4, 0>(lb);
    if (r == 8) return k16 ? lookup_lanes_for_lb<8, 16>(lb) : lookup_lanes_for_lb<8, 0>(lb);
    return k16 ? lookup_lanes_for_lb<16, 16>(lb) : lookup_lanes_for_lb<16, 0>(lb);
}

template <int R, int KC>
LookupKernel lookup_for_lb(uint32_t lb) {
    if (lb == 2) return k_classify_lookup<R, KC, 2>;
    if (lb == 8) return k_classify_lookup<R, KC, 8>;
    return k_classify_lookup<R, KC, 4>;
}

LookupKernel pick_lookup(const SketchParams& sp, uint32_t lb) {
    const int r = sketch_r_for(sp.w);
    const bool k16 = sp.k == 16;
    if (r == 4) return k16 ? lookup_for_lb<4, 16>(lb) : lookup_for_lb<4, 0>(lb);
    if (r == 8) return k16 ? lookup_for_lb<8, 16>(lb) : lookup_for_lb<8, 0>(lb);
    return k16 ? lookup_for_lb<16, 16>(lb) : lookup_for_lb<16, 0>(lb);
}

template <int KA, class KeyT, class LocT>
ScoreKernel score_for_gb(uint32_t gb) {
    if (gb == 4) return k_classify_score<KA, 4, KeyT, LocT>;
    if (gb == 16) return k_classify_score<KA, 16, KeyT, LocT>;
    return k_classify_score<KA, 8, KeyT, LocT>;
}

template <class KeyT, class LocT>
ScoreKernel score_for_ka(uint32_t ka, uint32_t gb) {
    if (ka == 256) return score_for_gb<256, KeyT, LocT>(gb);
    if (ka == 1024) return score_for_gb<1024, KeyT, LocT>(gb);
    return score_for_gb<512, KeyT, LocT>(gb);
}

// Histogram key / location types of a launch: compact = 32-bit keys of
// 32-bit locations; wide = 64-bit keys of 32-bit locations; otherwise both
// 64-bit.
enum class KeyMode { compact, wide32, wide64 };

KeyMode key_mode(const ClassifyDb& db, const Tuning& t) {
    if (!db.jbits) return KeyMode::wide64;
    return t.wide_keys ? KeyMode::wide32 : KeyMode::compact;
}

ScoreKernel pick_score(uint32_t ka, uint32_t gb, KeyMode km) {
    if (km == KeyMode::compact) return score_for_ka<uint32_t, uint32_t>(ka, gb);
    if (km == KeyMode::wide32) return score_for_ka<uint64_t, uint32_t>(ka, gb);
    return score_for_ka<uint64_t, uint64_t>(ka, gb);
}

MediumKernel pick_medium(KeyMode km) {
    return km == KeyMode::wide64 ? k_classify_medium<uint64_t> : k_classify_medium<uint32_t>;
}

template <class LocT>
LargeKernel pick_large_t(const SketchParams& sp) {
    const int r = sketch_r_for(sp.w);
    const bool k16 = sp.k == 16;
    if (r == 4) return k16 ? k_classify_large<4, 16, LocT> : k_classify_large<4, 0, LocT>;
    if (r == 8) return k16 ? k_classify_large<8, 16, LocT> : k_classify_large<8, 0, LocT>;
    return k16 ? k_classify_large<16, 16, LocT> : k_classify_large<16, 0, LocT>;
}

LargeKernel pick_large(const ClassifyDb& db) {
    return db.jbits ? pick_large_t<uint32_t>(db.sp) : pick_large_t<uint64_t>(db.sp);
}

// Kernels and launch shapes of one launch set.
using SortKernel = void (*)(ClassifyDb, ClassifyQuery, uint32_t, uint32_t, uint32_t, const uint64_t*, const uint4*,
                            uint32_t, bool, uint32_t, uint32_t*, uint32_t*, uint32_t*, const uint32_t*);

// The sort path's size classes: queries of up to 256, 512, 1024 and 2048
// gathered locations, each with its own kernel (E = 8, 16, 32, 64 per lane).
constexpr int N_SORT_CLASSES = 4;
constexpr uint32_t SORT_CLASS_MAX[N_SORT_CLASSES] = {CLASS_0_MAX, 512, 1024, 2048};
static_assert(QC_QUEUED_WORK - QC_GROUP == N_SORT_CLASSES, "a group counter per class");

// Launches of at least this many queries look up with one window per lane:
// four to five for each of the 3,648 resident warps; with fewer, lanes stay
// empty and one warp per query is faster.  Measured (us, per query / per
// lane): single reads of 100, 8,000 queries 23 / 29, 20,000 42 / 38, 100,000
// 168 / 68; half pairs, lengths 50-300, 8,000 queries 38 / 39, 20,000 73 / 65,
// 100,000 276 / 180.
constexpr uint32_t LANES_MIN_QUERIES = 16384;

// Launches of at most this many queries for each resident warp of the largest
// sort class leave them all to that class, with 64-bit locations: its warps
// have the room, and the other classes' kernels, of 2 us each with nothing to
// do, are not launched (1,000 pairs of 100, draft assemblies: 34.5 us, here 32.4).
// With 32-bit locations the largest class runs before the medium path and the
// others beside it, which is worth more where that path has queries (1,000
// pairs, repeat-rich genomes: 122 us, 129 in one class).
constexpr uint32_t ONE_CLASS_ROUNDS = 2;

struct Geometry {
    LookupKernel kl;         // one window per warp
    LookupLanesKernel kll;   // one window per lane
    uint32_t batch_shift;    // log2 of the queries a lookup warp takes at a time (kll)
    ScoreKernel ks;
    MediumKernel km;
    QueuedKernel kq;  // queued queries of up to QUEUED_MAX locations, or nullptr
    LargeKernel kb;
    SortKernel kt[N_SORT_CLASSES];
    bool sort;           // score by the sort path (else the hash path)
    int n_sort;          // sort classes in use
    bool one_class;      // the largest takes them all
    uint32_t list_cap;
    size_t smem_l, smem_s, smem_m, smem_b, smem_q, per_warp_b, smem_t[N_SORT_CLASSES];
    uint32_t threads_l, threads_s, grid_l, grid_s, grid_m, grid_q, blocks_b, grid_t[N_SORT_CLASSES];
    uint32_t group_shift;  // log2 of the queries a sort-path warp takes at a time
};

// Resident CTAs per SM of a kernel, remembered per thread: the query takes
// several microseconds, and a call that classifies a handful of queries makes
// five of them.  A function of the kernel, the launch shape and the device.
// (A fixed array: nothing is allocated, and a thread that uses more shapes
// than it holds asks again for the others.)
cudaError_t resident_ctas(const void* kernel, uint32_t threads, size_t smem, int dev, int* out) {
    struct Known {
        const void* kernel;
        size_t smem;
        uint32_t threads;
        int dev, ctas;
    };
    constexpr int MOST = 64;
    thread_local Known known[MOST];
    thread_local int n_known = 0;
    for (int i = 0; i < n_known; ++i) {
        const Known& k = known[i];
        if (k.kernel == kernel && k.smem == smem && k.threads == threads && k.dev == dev) {
            *out = k.ctas;
            return cudaSuccess;
        }
    }
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kernel, (int)threads, smem);
    if (e == cudaSuccess && n_known < MOST) known[n_known++] = Known{kernel, smem, threads, dev, *out};
    return e;
}

// counting: a call with counters, which drops no location before the sort;
// then 64-bit locations, of which no class sorts more than 256, take the hash
// path.
cudaError_t geometry(const ClassifyDb& db, const Tuning& t, const ClassifyScratch& sc, bool counting, Geometry* g) {
    cudaError_t e;
    int dev = 0, sms = NUM_SMS_HINT;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    g->list_cap = WIN_A * db.sp.s;
    g->kll = sc.chunk >= LANES_MIN_QUERIES ? pick_lookup_lanes(db.sp, t.probe_batch) : nullptr;
    g->kl = g->kll ? nullptr : pick_lookup(db.sp, t.probe_batch);
    const void* const kl_any = g->kll ? (const void*)g->kll : (const void*)g->kl;
    const KeyMode km = key_mode(db, t);
    const bool compact = km == KeyMode::compact;
    g->ks = pick_score(t.hist_slots, t.gather_batch, km);
    g->kb = pick_large(db);
    g->km = pick_medium(km);
    const size_t blk = db.jbits ? sizeof(BlockMem<uint32_t>) : sizeof(BlockMem<uint64_t>);
    g->smem_b = blk;
    g->smem_m = blk;
    if ((e = allow_smem(g->km, g->smem_m)) != cudaSuccess) return e;
    if ((e = allow_smem(g->kb, g->smem_b)) != cudaSuccess) return e;
    g->grid_m = std::min<uint32_t>((uint32_t)sms * BLK_CTAS, std::max<uint32_t>(sc.chunk, 1));
    g->threads_l = t.lookup_warps * 32;
    g->threads_s = t.score_warps * 32;
    const auto lookup_bytes = [&](uint32_t lc) { return g->kll ? sizeof(LookupLanesMem) : lookup_warp_bytes(lc); };
    const auto score_bytes = [&](uint32_t lc) {
        return compact ? scratch_bytes<uint16_t, uint32_t>(t.hist_slots, lc, 0, 0)
                       : scratch_bytes<uint16_t, uint64_t>(t.hist_slots, lc, 0, 0);
    };
    g->smem_l = t.lookup_warps * lookup_bytes(g->list_cap);
    g->smem_s = t.score_warps * score_bytes(g->list_cap);
    if ((e = allow_smem(kl_any, LK_WARPS * lookup_bytes(LIST_CAP_MAX))) != cudaSuccess) return e;
    if ((e = allow_smem(g->ks, CLS_WARPS * score_bytes(LIST_CAP_MAX))) != cudaSuccess) return e;
    int occ_l = 1, occ_s = 1;
    if ((e = resident_ctas(kl_any, g->threads_l, g->smem_l, dev, &occ_l)) != cudaSuccess)
        return e;
    if ((e = resident_ctas((const void*)g->ks, g->threads_s, g->smem_s, dev, &occ_s)) != cudaSuccess)
        return e;
    occ_l = std::max(occ_l, 1);
    occ_s = std::max(occ_s, 1);
    const uint64_t c = std::max<uint32_t>(sc.chunk, 1);
    g->grid_l = (uint32_t)std::min<uint64_t>((c + t.lookup_warps - 1) / t.lookup_warps, (uint64_t)sms * occ_l);
    g->batch_shift = 0;
    if (g->kll) {
        // as few queries per warp as one wave of resident warps needs, up to
        // a lane per query (half as many, in two waves: 100,000 queries 223
        // us instead of 180)
        const uint64_t warps = (uint64_t)sms * occ_l * t.lookup_warps;
        while (g->batch_shift < 5 && ((c + (1u << g->batch_shift) - 1) >> g->batch_shift) > warps) ++g->batch_shift;
        const uint64_t batches = (c + (1u << g->batch_shift) - 1) >> g->batch_shift;
        g->grid_l = (uint32_t)std::min<uint64_t>((batches + t.lookup_warps - 1) / t.lookup_warps, (uint64_t)sms * occ_l);
    }
    g->grid_s = (uint32_t)std::min<uint64_t>((c + t.score_warps - 1) / t.score_warps, (uint64_t)sms * occ_s);
    g->per_warp_b = scratch_bytes<uint32_t>(KB_SLOTS, LIST_B, LIST_B, BUF_B);
    g->blocks_b = std::max<uint32_t>(1, std::min(sc.large_warps, sc.n_q_cap));  // one piece of global scratch each
    // sort path: locations sorted as they are stored (not with wide keys of 32-bit ones)
    g->sort = km != KeyMode::wide32 && t.score_mode != SCORE_HASH && !(counting && km == KeyMode::wide64);
    g->n_sort = 0;
    g->one_class = false;
    g->group_shift = 0;
    if (g->sort) {
        const SortKernel kts[N_SORT_CLASSES] = {
            !compact ? k_classify_sort<8, uint64_t, false>
                     : (counting ? k_classify_sort<8, uint32_t, true> : k_classify_sort<8, uint32_t, false>),
            !compact ? k_classify_sort<16, uint64_t, false>
                     : (counting ? k_classify_sort<16, uint32_t, true> : k_classify_sort<16, uint32_t, false>),
            !compact ? k_classify_sort<32, uint64_t, false>
                     : (counting ? k_classify_sort<32, uint32_t, true> : k_classify_sort<32, uint32_t, false>),
            !compact ? nullptr
                     : (counting ? k_classify_sort<64, uint32_t, true> : k_classify_sort<64, uint32_t, false>)};
        const auto bytes = [&](int c2, uint32_t lc) {
            const size_t b[N_SORT_CLASSES] = {
                compact ? SortMem<8, uint32_t>::bytes(lc) : SortMem<8, uint64_t>::bytes(lc),
                compact ? SortMem<16, uint32_t>::bytes(lc) : SortMem<16, uint64_t>::bytes(lc),
                compact ? SortMem<32, uint32_t>::bytes(lc) : SortMem<32, uint64_t>::bytes(lc),
                compact ? SortMem<64, uint32_t>::bytes(lc) : 0};
            return SORT_WARPS * b[c2];
        };
        const uint32_t largest = compact ? t.sort_max : std::min(t.sort_max, 1024u);  // 64-bit: registers
        // groups of 32 queries where every resident warp gets several,
        // smaller ones in small launches, down to one query per warp
        const uint64_t warps = (uint64_t)sms * 28;
        while (g->group_shift < 5 && (c >> (g->group_shift + 1)) >= 4 * warps) ++g->group_shift;
        for (int c2 = 0; c2 < N_SORT_CLASSES && SORT_CLASS_MAX[c2] <= largest; ++c2) {
            g->kt[c2] = kts[c2];
            g->smem_t[c2] = bytes(c2, g->list_cap);
            if ((e = allow_smem(kts[c2], bytes(c2, LIST_CAP_MAX))) != cudaSuccess) return e;
            int occ_t = 1;
            if ((e = resident_ctas((const void*)kts[c2], SORT_WARPS * 32, g->smem_t[c2], dev, &occ_t)) !=
                cudaSuccess)
                return e;
            g->grid_t[c2] = (uint32_t)std::min<uint64_t>((c + SORT_WARPS - 1) / SORT_WARPS,
                                                         (uint64_t)sms * std::max(occ_t, 1));
            g->n_sort = c2 + 1;
        }
        const uint64_t last_warps = (uint64_t)g->grid_t[g->n_sort - 1] * SORT_WARPS;
        g->one_class = !compact && !counting && c <= ONE_CLASS_ROUNDS * last_warps;
    }
    g->kq = nullptr;
    // (queries beyond this many locations are queued)
    const uint32_t line = g->sort ? SORT_CLASS_MAX[g->n_sort - 1] : t.hist_slots;
    if (line < QUEUED_MAX) {
        const auto bytes = [&](uint32_t lc) {
            return SORT_WARPS * (db.jbits ? SortMem<32, uint32_t>::bytes(lc) : SortMem<32, uint64_t>::bytes(lc));
        };
        g->kq = db.jbits ? (counting ? k_sort_queued<uint32_t, true> : k_sort_queued<uint32_t, false>)
                         : (counting ? k_sort_queued<uint64_t, true> : k_sort_queued<uint64_t, false>);
        g->smem_q = bytes(g->list_cap);
        if ((e = allow_smem(g->kq, bytes(LIST_CAP_MAX))) != cudaSuccess) return e;
        int occ_q = 1;
        if ((e = resident_ctas((const void*)g->kq, SORT_WARPS * 32, g->smem_q, dev, &occ_q)) != cudaSuccess) return e;
        g->grid_q = (uint32_t)std::min<uint64_t>((c + SORT_WARPS - 1) / SORT_WARPS, (uint64_t)sms * std::max(occ_q, 1));
    }
    return cudaSuccess;
}

__host__ __device__ constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch layout: escalation queue + counters, chunk metadata, medium-path
// queue and the queue of what warps leave of it, chunk bucket lists,
// large-path working memory.
struct ScratchLayout {
    size_t ovf, meta, mid, glist, large, total;
    uint32_t chunk;
};

constexpr ScratchLayout scratch_layout(uint32_t n_q_cap, uint32_t sketch_size, uint32_t large_warps) {
    ScratchLayout L{};
    const size_t list_cap = (size_t)WIN_A * sketch_size;
    const size_t per_warp_b = scratch_bytes<uint32_t>(KB_SLOTS, LIST_B, LIST_B, BUF_B);
    L.chunk = n_q_cap < CHUNK ? n_q_cap : CHUNK;
    L.ovf = 0;
    L.meta = align256(L.ovf + ((size_t)n_q_cap + 16) * 4);
    L.mid = align256(L.meta + (size_t)L.chunk * sizeof(uint4));
    L.glist = align256(L.mid + (size_t)L.chunk * 4 * 2);
    L.large = align256(L.glist + (size_t)L.chunk * list_cap * 8);
    L.total = align256(L.large + (size_t)large_warps * per_warp_b);
    return L;
}

uint32_t* queue_counters(const ClassifyScratch& sc) { return sc.ovf + sc.n_q_cap; }

cudaError_t launch_lookup(const Geometry& g, const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc,
                          uint32_t q0, cudaStream_t s) {
    if (g.kll)
        MC_LAUNCH("classify_lookup", s,
                  g.kll<<<g.grid_l, g.threads_l, g.smem_l, s>>>(db, Q, q0, sc.chunk, g.list_cap, sc.glist, sc.meta,
                                                               sc.ovf, queue_counters(sc), g.batch_shift));
    else
        MC_LAUNCH("classify_lookup", s,
              g.kl<<<g.grid_l, g.threads_l, g.smem_l, s>>>(db, Q, q0, sc.chunk, g.list_cap, sc.glist, sc.meta, sc.ovf,
                                                          queue_counters(sc)));
    return cudaGetLastError();
}

// Medium path of the chunk at q0 (its queue).
cudaError_t launch_medium(const Geometry& g, const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc,
                          uint32_t q0, cudaStream_t s) {
    uint32_t* qc = queue_counters(sc);
    const uint32_t* queue = sc.mid;
    uint32_t* queue_n = qc + QC_MID;
    if (g.kq) {
        uint32_t* rest = sc.mid + sc.chunk;
        MC_LAUNCH("classify_queued", s,
                  g.kq<<<g.grid_q, SORT_WARPS * 32, g.smem_q, s>>>(db, Q, q0, g.list_cap, sc.glist, sc.meta, sc.mid,
                                                                 qc + QC_MID, qc + QC_QUEUED_WORK, rest,
                                                                 qc + QC_REST));
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        queue = rest;
        queue_n = qc + QC_REST;
    }
    MC_LAUNCH("classify_medium", s,
              g.km<<<g.grid_m, BLK_THREADS, g.smem_m, s>>>(db, Q, q0, g.list_cap, sc.glist, sc.meta, queue, queue_n,
                                                         qc + QC_MID_WORK, sc.ovf, qc + QC_LARGE));
    return cudaGetLastError();
}

// A launch of few queries: all of them straight to the large path's kernel.
// One launch instead of the six kernels and a memset of a launch set,
// whose latency is what such a call takes: 16 pairs 23 us on the device
// against some 40.  One wave of CTAs (two per SM) holds 304 queries; a second
// is faster or slower than the launch set by the reads (512 queries this way,
// 600 the other: mixed reads, related genomes 46 and 55 us, repeat-rich genomes
// 99 and 113, reads of 100 40 and 35), and the line lies within it.
// With 64-bit locations a launch set is shorter (one size class), and the line
// is one wave: pairs of 100, draft assemblies, 200 queries 23 us this way and
// 30 the other, 400 queries 38 and 31 (54 and 37 with candidate lists).
constexpr uint32_t DIRECT_MAX_QUERIES = 512;

// (a CTA per piece of global scratch, and at most two queries each, or one
// with 64-bit locations: an allocation-free launch has eight)
uint32_t direct_max(const ClassifyDb& db, const ClassifyScratch& sc) {
    return std::min(DIRECT_MAX_QUERIES, (db.jbits ? 2 : 1) * sc.large_warps);
}

cudaError_t launch_direct(const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc, cudaStream_t s) {
    const LargeKernel kb = pick_large(db);
    const size_t smem = db.jbits ? sizeof(BlockMem<uint32_t>) : sizeof(BlockMem<uint64_t>);
    cudaError_t e = allow_smem(kb, smem);
    if (e != cudaSuccess) return e;
    const uint32_t grid = std::max<uint32_t>(1, std::min(sc.large_warps, Q.n_q));
    MC_LAUNCH("classify_large", s,
              kb<<<grid, BLK_THREADS, smem, s>>>(db, Q, nullptr, nullptr, nullptr, sc.large,
                                                scratch_bytes<uint32_t>(KB_SLOTS, LIST_B, LIST_B, BUF_B)));
    return cudaGetLastError();
}

// Zeroes the counters from..to of a launch set.
cudaError_t reset_counters(const ClassifyScratch& sc, int from, int to, cudaStream_t s) {
    return cudaMemsetAsync(queue_counters(sc) + from, 0, (to - from) * sizeof(uint32_t), s);
}

// Score of the chunk at q0, whose counters from QC_MID up to QC_WIDEST are zero
// (each launch appends up to a chunk's queries to the queues).  Sort path,
// 32-bit locations: the largest size
// class first (it queues the queries beyond it), then the medium path, then
// the other classes, the most populous one (512) first.  Each of those is
// launched with programmatic stream serialization, so that it fills the SMs
// that the last queries of the kernel before leave idle (they share no data:
// the sort kernels read the lookup's outputs and write other queries'
// results; their groups of queries come from a counter, so the CTAs that
// start late take fewer).  64-bit locations: every class may queue queries,
// so the medium path comes last.  Hash path: the score kernel, then the
// medium path for the queries whose histogram did not fit.
cudaError_t launch_score(const Geometry& g, const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc,
                         uint32_t q0, cudaStream_t s) {
    uint32_t* qc = queue_counters(sc);
    cudaError_t e = cudaSuccess;
    if (!g.sort) {
        MC_LAUNCH("classify_score", s,
                  g.ks<<<g.grid_s, g.threads_s, g.smem_s, s>>>(db, Q, q0, sc.chunk, g.list_cap, sc.glist, sc.meta,
                                                              sc.mid, qc + QC_MID));
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        return launch_medium(g, db, Q, sc, q0, s);
    }
    static const char* const names[N_SORT_CLASSES] = {"classify_sort256", "classify_sort512", "classify_sort1024",
                                                      "classify_sort2048"};
    const int last = g.n_sort - 1;
    const bool narrow = db.jbits != 0;
    int order[N_SORT_CLASSES + 1], n = 0;
    order[n++] = last;
    if (narrow) order[n++] = -1;  // medium path
    if (last >= 2 && !g.one_class) order[n++] = 1;
    for (int c = 0; c < last && !g.one_class; ++c)
        if (c != 1 || last < 2) order[n++] = c;
    if (!narrow) order[n++] = -1;
    for (int k = 0; k < n; ++k) {
        const int c = order[k];
        if (c < 0) {
            if ((e = launch_medium(g, db, Q, sc, q0, s)) != cudaSuccess) return e;
            continue;
        }
        const uint32_t h_lo = c && !g.one_class ? SORT_CLASS_MAX[c - 1] : 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g.grid_t[c]);
        cfg.blockDim = dim3(SORT_WARPS * 32);
        cfg.dynamicSmemBytes = g.smem_t[c];
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = k > 0 ? 1 : 0;  // after the medium path or another class
        MC_LAUNCH(names[c], s,
                  e = cudaLaunchKernelEx(&cfg, g.kt[c], db, Q, q0, (uint32_t)sc.chunk, g.list_cap,
                                         (const uint64_t*)sc.glist, (const uint4*)sc.meta, h_lo, c == last, g.group_shift,
                                         sc.mid, qc + QC_MID, qc + QC_GROUP + c,
                                         (const uint32_t*)qc + QC_WIDEST));
        if (e != cudaSuccess) return e;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_large(const Geometry& g, const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc,
                         cudaStream_t s) {
    uint32_t* qc = queue_counters(sc);
    MC_LAUNCH("classify_large", s,
              g.kb<<<g.blocks_b, BLK_THREADS, g.smem_b, s>>>(db, Q, sc.ovf, qc + QC_LARGE, qc + QC_LARGE_WORK, sc.large,
                                                        g.per_warp_b));
    return cudaGetLastError();
}

}  // namespace

// ------------------------------------------------------------ shard merge
// Sharded classification (Section 4.2: with the database partitioned over
// GPUs, the top candidates of every partition are merged).  One thread per
// query merges the per-shard top-m lists into the global top m (score
// descending, global target ascending; a target lives in one shard, so no
// candidate spans lists) and labels it as query_score does.
namespace {
__global__ void k_merge_candidates(ClassifyDb db, const uint32_t* __restrict__ taxon, uint32_t n_targets,
                                   const MergeList* __restrict__ lists, uint32_t n_lists, uint32_t n_q, uint32_t m,
                                   uint32_t hits_min, uint32_t band, uint32_t* __restrict__ label,
                                   uint32_t* __restrict__ hits, uint32_t* __restrict__ top_target,
                                   uint32_t* __restrict__ cands_out) {
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n_q; q += gridDim.x * blockDim.x) {
        uint32_t ts[MAX_M], tt[MAX_M], tj0[MAX_M], tj1[MAX_M];
#pragma unroll
        for (int a = 0; a < MAX_M; ++a) {
            ts[a] = 0;
            tt[a] = 0xFFFFFFFFu;
            tj0[a] = tj1[a] = 0;
        }
        for (uint32_t l = 0; l < n_lists; ++l) {
            const MergeList L = lists[l];
            for (uint32_t i = 0; i < m; ++i) {
                const uint4 c = *reinterpret_cast<const uint4*>(L.cands + ((uint64_t)q * m + i) * 4);
                if (c.x == 0) break;  // the rest of this list is empty
                uint32_t cs = c.x, ct = L.base + c.y, c0 = c.z, c1 = c.w;
                // one bubbling insertion pass (score descending, target ascending)
#pragma unroll
                for (int a = 0; a < MAX_M; ++a) {
                    if ((uint32_t)a < m && (cs > ts[a] || (cs == ts[a] && ct < tt[a]))) {
                        const uint32_t xs = ts[a], xt = tt[a], x0 = tj0[a], x1 = tj1[a];
                        ts[a] = cs;
                        tt[a] = ct;
                        tj0[a] = c0;
                        tj1[a] = c1;
                        cs = xs;
                        ct = xt;
                        c0 = x0;
                        c1 = x1;
                    }
                }
            }
        }
        uint32_t lab = NO_TAXON;
        const uint32_t h = ts[0];
        if (h > 0 && h >= hits_min) {
            lab = tt[0] < n_targets ? taxon[tt[0]] : NO_TAXON;
            const uint64_t bar = (uint64_t)(100 - band) * h;
#pragma unroll
            for (int a = 1; a < MAX_M; ++a) {
                if ((uint32_t)a >= m || ts[a] == 0 || 100ull * ts[a] < bar) break;
                lab = lca2(db, lab, tt[a] < n_targets ? taxon[tt[a]] : NO_TAXON);
            }
        }
        label[q] = lab;
        hits[q] = h;
        if (top_target) top_target[q] = h ? tt[0] : 0xFFFFFFFFu;
        if (cands_out) {
#pragma unroll
            for (int a = 0; a < MAX_M; ++a)
                if ((uint32_t)a < m)
                    *reinterpret_cast<uint4*>(cands_out + ((uint64_t)q * m + a) * 4) =
                        make_uint4(ts[a], ts[a] ? tt[a] : 0xFFFFFFFFu, ts[a] ? tj0[a] : 0, ts[a] ? tj1[a] : 0);
        }
    }
}
}  // namespace

cudaError_t merge_candidates(const Mem& mem, const ClassifyDb& db, const uint32_t* taxon, uint32_t n_targets,
                             const MergeList* lists, uint32_t n_lists, uint32_t n_q, uint32_t m, uint32_t hits_min,
                             uint32_t band, uint32_t* label, uint32_t* hits, uint32_t* top_target, uint32_t* cands_out,
                             cudaStream_t s) {
    if (n_q == 0) return cudaSuccess;
    Tmp<MergeList> dl(mem, std::max<uint32_t>(n_lists, 1), s);
    if (!dl.ok()) return cudaErrorMemoryAllocation;
    cudaError_t e;
    if (n_lists &&
        (e = cudaMemcpyAsync(dl.ptr, lists, n_lists * sizeof(MergeList), cudaMemcpyHostToDevice, s)) != cudaSuccess)
        return e;
    const uint32_t grid = (uint32_t)std::min<uint64_t>((n_q + 255) / 256, (uint64_t)NUM_SMS_HINT * 8);
    MC_LAUNCH("merge_candidates", s,
              k_merge_candidates<<<grid, 256, 0, s>>>(db, taxon, n_targets, dl.ptr, n_lists, n_q, m, hits_min, band,
                                                      label, hits, top_target, cands_out));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // the host list array is read by the copy above: wait for it before returning
    return cudaStreamSynchronize(s);
}

uint32_t compact_key_bits(uint64_t n_targets, uint64_t max_windows) {
    auto bits = [](uint64_t x) { return x ? 64u - (uint32_t)__builtin_clzll(x) : 0u; };
    if (n_targets == 0 || max_windows == 0) return 0;
    const uint32_t jb = std::max(1u, bits(max_windows - 1));
    const uint32_t tb = bits(n_targets - 1);
    if (jb >= 32) return 0;  // one target of more than 2^31 windows: 64-bit locations
    if (jb + tb < 32) return jb;
    // 32 bits: usable unless the all-ones key (the empty-slot marker) is a
    // location; a sliding-window lookup of that key only ever meets empty
    // slots and counts 0
    if (jb + tb == 32 && !(n_targets == (1ull << tb) && max_windows == (1ull << jb))) return jb;
    return 0;
}

bool tuning_valid(const Tuning& t) {
    auto in = [](uint32_t v, std::initializer_list<uint32_t> set) {
        for (uint32_t x : set)
            if (v == x) return true;
        return false;
    };
    return in(t.hist_slots, {256, 512, 1024}) && in(t.probe_batch, {2, 4, 8}) && in(t.gather_batch, {4, 8, 16}) &&
           in(t.lookup_warps, {4, 8}) && in(t.score_warps, {2, 4}) && t.wide_keys <= 1 &&
           in(t.score_mode, {SCORE_SORT, SCORE_HASH}) && in(t.sort_max, {256, 512, 1024, 2048});
}

uint32_t classify_default_large_warps() {
    int dev = 0, sms = NUM_SMS_HINT;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        sms = NUM_SMS_HINT;
    }
    return (uint32_t)(sms * BLK_CTAS);
}

size_t classify_scratch_bytes(uint32_t n_q_cap, uint32_t sketch_size, uint32_t large_warps) {
    return scratch_layout(n_q_cap, sketch_size, large_warps).total;
}

ClassifyScratch classify_scratch_carve(unsigned char* base, uint32_t n_q_cap, uint32_t sketch_size,
                                       uint32_t large_warps) {
    const ScratchLayout L = scratch_layout(n_q_cap, sketch_size, large_warps);
    ClassifyScratch sc;
    sc.ovf = reinterpret_cast<uint32_t*>(base + L.ovf);
    sc.meta = reinterpret_cast<uint4*>(base + L.meta);
    sc.mid = reinterpret_cast<uint32_t*>(base + L.mid);
    sc.glist = reinterpret_cast<uint64_t*>(base + L.glist);
    sc.large = base + L.large;
    sc.n_q_cap = n_q_cap;
    sc.chunk = L.chunk;
    sc.large_warps = large_warps;
    return sc;
}

int classify_set_sizes(const ClassifyDb& db, const ClassifyScratch& sc, uint32_t sizes[CLASSIFY_MAX_SIZES]) {
    int n = 0;
    const auto add = [&](uint32_t most) {
        if (most < sc.n_q_cap) sizes[n++] = most;
    };
    add(direct_max(db, sc));
    add(LANES_MIN_QUERIES - 1);
    // from there on shapes change every doubling: the lookup's queries per warp
    // at 8 and 16 times its 3,648 resident warps (the sizes lie just under
    // those), the sort path's up to 32 queries per group at half a million
    for (uint32_t most = 28 << 10; most < CHUNK; most *= 2) add(most);
    sizes[n++] = sc.n_q_cap;
    return n;
}

cudaError_t classify_enqueue(const ClassifyDb& db, const ClassifyQuery& Q, const Tuning& t,
                             const ClassifyScratch& scratch, cudaStream_t s, int* n_kernels) {
    cudaError_t e;
    int n = 0;
    if (n_kernels) *n_kernels = 0;
    if (Q.n_q == 0) return cudaSuccess;
    if (Q.n_q > scratch.n_q_cap) return cudaErrorInvalidValue;
    ClassifyScratch sc = scratch;
    sc.chunk = std::min(sc.chunk, Q.n_q);  // the launch's shape follows its queries, not its scratch
    if (Q.n_q <= direct_max(db, sc) && !Q.counters) {
        if ((e = launch_direct(db, Q, sc, s)) != cudaSuccess) return e;
        if (n_kernels) *n_kernels = 1;
        return cudaSuccess;
    }
    Geometry g;
    if ((e = geometry(db, t, sc, Q.counters != nullptr, &g)) != cudaSuccess) return e;
    for (uint32_t q0 = 0; q0 < Q.n_q; q0 += sc.chunk) {
        // only the counters must start at zero
        if ((e = reset_counters(sc, q0 ? QC_MID : QC_LARGE, QC_END, s)) != cudaSuccess) return e;
        if ((e = launch_lookup(g, db, Q, sc, q0, s)) != cudaSuccess) return e;
        if ((e = launch_score(g, db, Q, sc, q0, s)) != cudaSuccess) return e;
        n += 2 + (g.sort && !g.one_class ? g.n_sort : 1) + (g.kq ? 1 : 0);
        if (sc.chunk == 0) break;
    }
    if ((e = launch_large(g, db, Q, sc, s)) != cudaSuccess) return e;
    if (n_kernels) *n_kernels = n + 1;
    return cudaSuccess;
}

cudaError_t classify_launch(const Mem& mem, const ClassifyDb& db, const ClassifyQuery& Q, const Tuning& t,
                            cudaStream_t s) {
    if (Q.n_q == 0) return cudaSuccess;
    const uint32_t lw = classify_default_large_warps();
    Tmp<unsigned char> buf(mem, classify_scratch_bytes(Q.n_q, db.sp.s, lw), s);
    if (!buf.ok()) return cudaErrorMemoryAllocation;
    const ClassifyScratch sc = classify_scratch_carve(buf.ptr, Q.n_q, db.sp.s, lw);
    return classify_enqueue(db, Q, t, sc, s, nullptr);
}

// Number of large-path CTAs of the allocation-free launch.
constexpr uint32_t NOALLOC_LARGE_WARPS = 8;
// The documented per-call maximum of the allocation-free entry point must
// fit its fixed scratch array at the largest sketch size.
static_assert(scratch_layout(MC_NOALLOC_MAX_QUERIES, MC_MAX_SKETCH, NOALLOC_LARGE_WARPS).total <=
                  MC_NOALLOC_SCRATCH_BYTES,
              "MC_NOALLOC_MAX_QUERIES queries at MC_MAX_SKETCH do not fit MC_NOALLOC_SCRATCH_BYTES");

size_t classify_noalloc_bytes(uint32_t n_q, uint32_t sketch_size) {
    return classify_scratch_bytes(n_q, sketch_size, NOALLOC_LARGE_WARPS);
}

cudaError_t classify_launch_noalloc(const ClassifyDb& db, const ClassifyQuery& Q, const Tuning& t,
                                   unsigned char* scratch, size_t scratch_len, cudaStream_t s) {
    if (Q.n_q == 0) return cudaSuccess;
    if (classify_noalloc_bytes(Q.n_q, db.sp.s) > scratch_len) return cudaErrorInvalidValue;
    const ClassifyScratch sc = classify_scratch_carve(scratch, Q.n_q, db.sp.s, NOALLOC_LARGE_WARPS);
    return classify_enqueue(db, Q, t, sc, s, nullptr);
}

cudaError_t classify_autotune(const ClassifyDb& db, const ClassifyQuery& Q, const ClassifyScratch& sc, uint32_t reps,
                              cudaStream_t s, Tuning* best, std::vector<TuneRecord>* records) {
    cudaError_t e = cudaSuccess;
    if (Q.n_q == 0 || Q.n_q > sc.chunk || reps == 0) return cudaErrorInvalidValue;
    cudaEvent_t a = nullptr, b = nullptr;
    if ((e = cudaEventCreate(&a)) != cudaSuccess) return e;
    if ((e = cudaEventCreate(&b)) != cudaSuccess) {
        cudaEventDestroy(a);
        return e;
    }
    uint32_t* qc = queue_counters(sc);
    Tuning cur = DEFAULT_TUNING;
    float best_ms = 0;
    auto timed = [&](auto&& body, float* ms) -> cudaError_t {
        cudaError_t err;
        float total = 0;
        for (uint32_t r = 0; r <= reps; ++r) {  // run 0 warms up
            if ((err = cudaEventRecord(a, s)) != cudaSuccess) return err;
            if ((err = body()) != cudaSuccess) return err;
            if ((err = cudaEventRecord(b, s)) != cudaSuccess) return err;
            if ((err = cudaEventSynchronize(b)) != cudaSuccess) return err;
            float x = 0;
            if ((err = cudaEventElapsedTime(&x, a, b)) != cudaSuccess) return err;
            if (r) total += x;
        }
        *ms = total / reps;
        return cudaSuccess;
    };
    // stage 0: lookup settings
    {
        bool first = true;
        Tuning bl = cur;
        for (uint32_t lb : {2u, 4u, 8u}) {
            for (uint32_t lw : {4u, 8u}) {
                Tuning t = cur;
                t.probe_batch = lb;
                t.lookup_warps = lw;
                Geometry g;
                if ((e = geometry(db, t, sc, Q.counters != nullptr, &g)) != cudaSuccess) goto done;
                float ms = 0;
                e = timed(
                    [&]() -> cudaError_t {
                        cudaError_t err = reset_counters(sc, QC_LARGE, QC_END, s);
                        return err != cudaSuccess ? err : launch_lookup(g, db, Q, sc, 0, s);
                    },
                    &ms);
                if (e != cudaSuccess) goto done;
                if (records) records->push_back(TuneRecord{t, 0, ms});
                if (first || ms < best_ms) {
                    best_ms = ms;
                    bl = t;
                    first = false;
                }
            }
        }
        cur = bl;
    }
    // lookup output of the chosen setting, and its queue length, for stage 1
    {
        Geometry g;
        if ((e = geometry(db, cur, sc, Q.counters != nullptr, &g)) != cudaSuccess) goto done;
        if ((e = reset_counters(sc, QC_LARGE, QC_END, s)) != cudaSuccess) goto done;
        if ((e = launch_lookup(g, db, Q, sc, 0, s)) != cudaSuccess) goto done;
        if ((e = cudaMemcpyAsync(qc + QC_SAVED, qc + QC_LARGE, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s)) !=
            cudaSuccess)
            goto done;
    }
    // stage 1: score settings (with the large path they leave), each from the
    // lookup's output and its counters as the lookup left them
    {
        const auto score_again = [&](const Geometry& g) -> cudaError_t {
            cudaError_t err;
            if ((err = cudaMemcpyAsync(qc + QC_LARGE, qc + QC_SAVED, sizeof(uint32_t), cudaMemcpyDeviceToDevice, s)) !=
                cudaSuccess)
                return err;
            if ((err = reset_counters(sc, QC_LARGE_WORK, QC_WIDEST, s)) != cudaSuccess) return err;
            if ((err = launch_score(g, db, Q, sc, 0, s)) != cudaSuccess) return err;
            return launch_large(g, db, Q, sc, s);
        };
        bool first = true;
        Tuning bs = cur;
        for (uint32_t ka : {256u, 512u, 1024u}) {
            for (uint32_t gb : {4u, 8u, 16u}) {
                for (uint32_t sw : {2u, 4u}) {
                    Tuning t = cur;
                    t.score_mode = SCORE_HASH;
                    t.hist_slots = ka;
                    t.gather_batch = gb;
                    t.score_warps = sw;
                    Geometry g;
                    if ((e = geometry(db, t, sc, Q.counters != nullptr, &g)) != cudaSuccess) goto done;
                    float ms = 0;
                    e = timed([&]() -> cudaError_t { return score_again(g); }, &ms);
                    if (e != cudaSuccess) goto done;
                    if (records) records->push_back(TuneRecord{t, 1, ms});
                    if (first || ms < best_ms) {
                        best_ms = ms;
                        bs = t;
                        first = false;
                    }
                }
            }
        }
        // the sort path, for each largest size class (64-bit locations have
        // no larger one than 1,024: 2,048 would be timed twice)
        {
            for (uint32_t smax : {256u, 512u, 1024u, 2048u}) {
                if (smax > 1024 && !db.jbits) break;
                Tuning t = cur;
                t.score_mode = SCORE_SORT;
                t.sort_max = smax;
                t.wide_keys = 0;
                Geometry g;
                if ((e = geometry(db, t, sc, Q.counters != nullptr, &g)) != cudaSuccess) goto done;
                float ms = 0;
                e = timed([&]() -> cudaError_t { return score_again(g); }, &ms);
                if (e != cudaSuccess) goto done;
                if (records) records->push_back(TuneRecord{t, 1, ms});
                if (ms < best_ms) {
                    best_ms = ms;
                    bs = t;
                }
            }
        }
        cur = bs;
    }
    *best = cur;
done:
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return e;
}

}  // namespace mc
