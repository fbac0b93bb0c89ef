// lpa_sweep_lane.cu -- synchronous sweep for mid-degree vertices
// (small_max < d <= warp_max): one lane per frontier vertex, its row sorted in
// registers.
//
// Eq. 2 (Section 3.3) sums the weights of a row per label.  A whole warp on
// one row of a few dozen entries pays for every step of that once per row:
// grouping 32 lanes with distinct labels by __match_any_sync costs 64 cycles
// of an SM and summing the groups' weights 129 more (measured on GB300), and
// a shared table with atomics still takes about 450 instructions per row.
// Here an instruction serves 32 rows.  A lane takes its row 32 slots at a
// time: 16-byte loads of the ids, all labels gathered at once (32 gathers in
// flight per lane), each label packed with its weight into one 32-bit key and
// the keys sorted in registers with a Batcher network (191 comparators of two
// instructions).  Of a row of up to 64 slots the first half waits in the
// lane's column of shared memory (slot i of lane l in word 32 i + l: no
// conflicts) and the two sorted halves are merged (32 comparators across, then
// a bitonic merge of each half).  In the sorted keys equal labels meet, and one
// pass takes the largest run sum; labels ascend, so the first of the largest
// runs is the smallest label of the tie.  One network serves every row, each
// part of the code appears once and is looped over: with a network per length
// (up to 64 keys, 543 comparators) the straight-line code outgrew the
// instruction caches and warps waited for instructions two thirds of the time.
//
// Measured on a batch of 64 planted partitions (54 M entries, weights 1..4, a
// dense sweep): a warp per row with match groups 1.6 ms, with table atomics
// 0.81, a lane per row with a hash table of its own 0.96 (8 warps per SM), with
// all pairs compared 0.75, this kernel 0.39 (141 G entries/s; the gathers alone
// take 0.18 at the 296 G/s of L2).  It is bound by instructions and their
// latency at 16 to 20 warps per SM; 24 warps at 85 registers spill (0.46).
//
// Keys (chosen at the launch from the number of vertices and the largest
// weight): the label alone for unit weights; label and weight where both fit
// 32 bits; else label and place in the row (6 bits), the weights waiting in
// shared memory -- also for fp32 weights, whose sums are so taken in the row's
// entry order.  Longer rows (more than 64 slots) and the few rows at the very end
// of the index array (a 16-byte load would pass it) are taken by a whole warp
// each (lpa_warp_row.cuh): within k_sweep_lane where the key is the label or
// holds the weight, else by a kernel of their own, k_sweep_long (see there), which
// also takes every row of graphs whose labels leave no room for a key.
//
// The 32 rows of a step cost as much as the longest of them, so each warp
// sorts the vertices of its part of the frontier into queues by row length and
// takes a step when a queue holds 32 rows; what is left in the queues at the
// end of the pass is taken in as few steps as possible, longest rows first.
//
// Self-loops are skipped (Algorithm 1); ties go to the smallest label id
// (Section 4.1.5).  A lane whose vertex changes walks the row again to mark
// the neighbours unprocessed (Section 4.1.4).
#include <utility>
#include <vector>

#include "lpa_warp_row.cuh"

namespace lpa {

constexpr int kSortSlots = 32;          // row slots sorted at a time
constexpr int kLaneMax = 64;            // row slots a lane can take
constexpr int kPosBits = 6;             // log2(kLaneMax)
static_assert(kLaneEntries + 3 == kLaneMax, "a row may start up to 3 slots past a 16-byte boundary");
constexpr int kLaneQueues = 3;          // rows of up to 32 slots, of up to 64, longer ones
constexpr int kLong = kLaneQueues - 1;
constexpr int kLaneQueueCap = 64;       // a queue is drained before it can pass 31 + 32
constexpr int kLaneWarps = 4;           // per block
constexpr uint32_t kNoKey = 0xffffffffu;    // sorts last; no real key has all bits set

enum LaneKey : int {
    KEY_LABEL = 0,      // label (unit weights)
    KEY_PACKED = 1,     // label << weight_bits | weight
    KEY_PLACE = 2,      // label << kPosBits | place in the row
};

// ---- Batcher's odd-even merge sorting network for N keys -------------------
template <typename F>
constexpr int sort_net(int n, F&& comparator) {
    int count = 0;
    for (int p = 1; p < n; p += p)
        for (int k = p; k > 0; k /= 2)
            for (int j = k % p; j + k < n; j += 2 * k)
                for (int i = 0; i < k && i + j + k < n; ++i)
                    if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) comparator(count++, i + j, i + j + k);
    return count;
}

constexpr int sort_net_size(int n) {
    return sort_net(n, [](int, int, int) {});
}

template <int N>
struct SortNet {
    static constexpr int kSize = sort_net_size(N);
    struct Table {
        unsigned char lo[kSize], hi[kSize];
    };
    static constexpr Table make() {
        Table t{};
        sort_net(N, [&t](int c, int x, int y) {
            t.lo[c] = (unsigned char)x;
            t.hi[c] = (unsigned char)y;
        });
        return t;
    }
};
template <int N>
constexpr typename SortNet<N>::Table kSortNet = SortNet<N>::make();

template <int A, int B, int N>
__device__ __forceinline__ void compare_exchange(uint32_t (&k)[N]) {
    const uint32_t lo = min(k[A], k[B]), hi = max(k[A], k[B]);
    k[A] = lo;
    k[B] = hi;
}

template <int N, size_t... I>
__device__ __forceinline__ void sort_keys(uint32_t (&k)[N], std::index_sequence<I...>) {
    (compare_exchange<kSortNet<N>.lo[I], kSortNet<N>.hi[I]>(k), ...);
}

// Sorts a bitonic sequence (N a power of two).
template <int N>
__device__ __forceinline__ void bitonic_merge(uint32_t (&k)[N]) {
#pragma unroll
    for (int o = N / 2; o > 0; o /= 2)
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((i & o) == 0) {
                const uint32_t lo = min(k[i], k[i + o]), hi = max(k[i], k[i + o]);
                k[i] = lo;
                k[i + o] = hi;
            }
}

// A queued vertex: its slot in the frontier list, its row.
struct LaneRow {
    uint32_t k;
    int32_t v, d;
    int64_t st;
};
__device__ __forceinline__ uint4 pack_row(const LaneRow& r) {      // st < 2^48, d <= warp_max <= 256
    return make_uint4(r.k, (uint32_t)r.v, (uint32_t)r.st, (uint32_t)((uint64_t)r.st >> 32) | ((uint32_t)r.d << 16));
}
__device__ __forceinline__ LaneRow unpack_row(const uint4& q) {
    LaneRow r;
    r.k = q.x;
    r.v = (int32_t)q.y;
    r.st = (int64_t)(((uint64_t)(q.w & 0xffffu) << 32) | q.z);
    r.d = (int32_t)(q.w >> 16);
    return r;
}

template <int KM, int WK>
struct LaneShape {
    static constexpr size_t QUEUES = kLaneQueues * kLaneQueueCap * sizeof(uint4);
    static constexpr size_t COLUMNS = (size_t)kSortSlots * 32 * 4;
    static constexpr size_t WEIGHTS = KM == KEY_PLACE ? (size_t)kLaneMax * 32 * 4 : 0;
    static constexpr size_t TABLE = (size_t)512 * 4 * kTableWords<WK>;     // of a longer row, in the columns' place
    static constexpr size_t WARP_BYTES = QUEUES + (COLUMNS + WEIGHTS > TABLE ? COLUMNS + WEIGHTS : TABLE);
};

// Entries [a, a + 4) of row [st, en) of vertex v (a a multiple of 4): ids, v
// outside the row, and weights.  16-byte loads below E_al.
template <int WK>
__device__ __forceinline__ void load_row4(const DevState& s, int64_t a, int64_t st, int64_t en, int64_t E_al, int32_t v,
                                          int32_t (&j)[4], typename Acc<WK>::T (&w)[4]) {
    using T = typename Acc<WK>::T;
    if (a + 4 <= E_al) {
        const int4 x = __ldg(reinterpret_cast<const int4*>(s.idx + a));
        const int32_t z[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) j[c] = a + c >= st && a + c < en ? z[c] : v;
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) j[c] = a + c >= st && a + c < en ? __ldg(s.idx + a + c) : v;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) w[c] = WK != W_UNIT && j[c] != v ? load_weight<WK>(s.w, a + c) : (T)1;
}

// Keys of slots [0, 32) of a row whose slot 0 is entry a0 (a multiple of 4)
// and whose entries are slots [lo, hi).  `place0` is the place of slot 0 among
// the row's slots (0 or 32).
template <int KM, int WK>
__device__ __forceinline__ void load_keys(const DevState& s, const int32_t* C, int32_t v, int64_t a0, int lo, int hi,
                                          int place0, uint32_t (&key)[kSortSlots],
                                          [[maybe_unused]] typename Acc<WK>::T* wts) {
    constexpr int S = kSortSlots;
    int4 x[S / 4];
    [[maybe_unused]] uint32_t wb[S / 4];
#pragma unroll
    for (int t = 0; t < S / 4; ++t) {
        x[t] = make_int4(v, v, v, v);
        if (4 * t < hi) x[t] = __ldcs(reinterpret_cast<const int4*>(s.idx + a0) + t);
        if constexpr (WK == W_U8) {
            wb[t] = 0u;
            if (4 * t < hi) wb[t] = __ldcs(reinterpret_cast<const uint32_t*>(static_cast<const unsigned char*>(s.w) + a0) + t);
        }
    }
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const int4& q = x[i / 4];
        const int32_t j = (i & 3) == 0 ? q.x : (i & 3) == 1 ? q.y : (i & 3) == 2 ? q.z : q.w;
        key[i] = i >= lo && i < hi && j != v ? (uint32_t)load_label<false>(C, j) : kNoKey;
    }
    if constexpr (KM == KEY_PLACE && WK != W_U8) {
#pragma unroll
        for (int t = 0; t < S / 4; ++t) {
            if (4 * t < hi) {
                const uint4 q = __ldcs(reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(s.w) + a0) + t);
                const uint32_t z[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if constexpr (WK == W_F32) wts[(place0 + 4 * t + c) * 32] = __uint_as_float(z[c]);
                    else wts[(place0 + 4 * t + c) * 32] = z[c];
                }
            }
        }
    }
    if constexpr (KM != KEY_LABEL) {
        const int shift = KM == KEY_PACKED ? s.weight_bits : kPosBits;
#pragma unroll
        for (int i = 0; i < S; ++i) {
            uint32_t add = (uint32_t)(place0 + i);
            if constexpr (KM == KEY_PACKED) {
                if constexpr (WK == W_U8) {
                    add = (wb[i / 4] >> (8 * (i & 3))) & 0xffu;
                } else {
                    add = 4 * (i / 4) < hi ? __ldcs(static_cast<const uint32_t*>(s.w) + a0 + i) : 0u;
                }
            } else if constexpr (WK == W_U8) {
                wts[(place0 + i) * 32] = (wb[i / 4] >> (8 * (i & 3))) & 0xffu;
            }
            if (key[i] != kNoKey) key[i] = (key[i] << shift) | add;
        }
    }
}

// Scans one vertex in each lane whose row of d entries from st spans at most
// 32 * halves slots (halves 1 or 2, the same in every lane) from the 4-entry
// boundary before it.  Returns the winning label or -1.
template <int KM, int WK, bool NS>
__device__ __forceinline__ int32_t lane_pick(const DevState& s, const int32_t* C, int32_t v, int64_t st, int d,
                                             const TieRule& tr, int halves, uint32_t* col,
                                             [[maybe_unused]] typename Acc<WK>::T* wts) {
    using T = typename Acc<WK>::T;
    constexpr int S = kSortSlots;
    const int64_t a0 = st & ~(int64_t)3;
    const int lo = (int)(st - a0), hi = d > 0 ? lo + d : 0;
    uint32_t key[S];
#pragma unroll 1
    for (int h = 0; h < halves; ++h) {
        if (h > 0) {
#pragma unroll
            for (int i = 0; i < S; ++i) col[i * 32] = key[i];
        }
        load_keys<KM, WK>(s, C, v, a0 + S * h, lo - S * h, min(hi - S * h, S), S * h, key, wts);
        sort_keys<S>(key, std::make_index_sequence<SortNet<S>::kSize>{});
    }
    if (halves > 1) {
        // the smaller half of both stays in registers, the larger one in the column
#pragma unroll
        for (int i = 0; i < S / 2; ++i) {
            const int r = S - 1 - i;
            const uint32_t x = col[i * 32], y = col[r * 32], p = key[r], q = key[i];
            key[i] = min(x, p);
            key[r] = min(y, q);
            col[i * 32] = max(x, p);
            col[r * 32] = max(y, q);
        }
    }
    // runs of one label: the largest sum, then the first (strict: smallest
    // label) or the smallest tie key (non-strict)
    const int shift = KM == KEY_PACKED ? s.weight_bits : KM == KEY_PLACE ? kPosBits : 0;
    const uint32_t low = (1u << shift) - 1u;
    uint32_t prev = kNoKey, best_lab = kNoKey;
    [[maybe_unused]] uint32_t best_tie = 0xffffffffu;
    T run = (T)0, best = (T)0;
#pragma unroll 1
    for (int h = 0; h < halves; ++h) {
        if (h > 0) {
#pragma unroll
            for (int i = 0; i < S; ++i) key[i] = col[i * 32];
        }
        if (halves > 1) bitonic_merge<S>(key);
#pragma unroll
        for (int i = 0; i < S; ++i) {
            const uint32_t k = key[i];
            const uint32_t lab = KM == KEY_LABEL ? k : k >> shift;
            T w = (T)1;
            if constexpr (KM == KEY_PACKED) w = (T)(k & low);
            if constexpr (KM == KEY_PLACE) w = wts[(k & low) * 32];
            run = lab == prev ? run + w : w;
            prev = lab;
            bool better = best_lab == kNoKey || run > best;
            if constexpr (NS) {
                const uint32_t t = tr.key((int32_t)lab);
                better = better || (run == best && t < best_tie);
                if (k != kNoKey && better) best_tie = t;
            }
            if (k != kNoKey && better) {
                best = run;
                best_lab = lab;
            }
        }
    }
    return (int32_t)best_lab;
}

// First sweep of a repeat-free graph: every label is still its vertex's id and
// occurs once in a row, so the pick is the row's heaviest entry.  A lane per row,
// straight from the list.  All threads of the block must call, once, as the last
// step of the kernel.
template <int WK, bool NS>
__device__ __forceinline__ void identity_rows(const DevState& s, const Labels& L, const BinView& bv, bool marks,
                                              uint32_t sweep, int64_t E_al) {
    using T = typename Acc<WK>::T;
    const unsigned cnt = bv.cnt;
    unsigned long long my_changed = 0, my_changed_entries = 0;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += gridDim.x * blockDim.x) {
        const int32_t v = bv.list[k];
        const int64_t st = s.off[v], en = s.off_end[v];
        const int32_t own = L.C[v];
        int32_t best = -1;
        if (WK == W_UNIT && !NS) {
            // equal weights and ascending neighbours: the first entry that
            // is not v itself
            for (int64_t e = st; e < en && best < 0; ++e) {
                const int32_t j = __ldg(s.idx + e);
                if (j != v) best = initial_label(s, j);
            }
        } else {
            const TieRule tr = tie_rule(s, NS, sweep, v);
            uint32_t key = 0, tie = 0xffffffffu;
            for (int64_t a = st & ~(int64_t)3; a < en; a += 4) {
                int32_t j[4];
                T w[4];
                load_row4<WK>(s, a, st, en, E_al, v, j, w);
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (j[c] != v) offer_candidate<T>(tr, w[c], initial_label(s, j[c]), key, tie);
            }
            if (key != 0u) best = tr.label(tie);
        }
        const bool changed = best >= 0 && best != own;
        record_label<false>(L, bv.chg + k, v, own, best, changed);
        if (changed) {
            ++my_changed;
            my_changed_entries += (unsigned)(en - st);
            if (marks)
                for (int64_t e = st; e < en; ++e) {
                    const int32_t j = __ldg(s.idx + e);
                    if (j != v) mark_unprocessed(s.flags, j);
                }
        }
    }
    flush_bin_counts(s, 1, my_changed, my_changed_entries);
}

// A row that a lane cannot take.
__device__ __forceinline__ bool is_long(int64_t st, int64_t en, int64_t E_al) {
    return en - (st & ~(int64_t)3) > kLaneMax || en > E_al;
}

// Row of frontier entry `at`; true if it is a longer one (or `all`) of a graph
// that still runs.
__device__ __forceinline__ bool load_long(const DevState& s, const Labels& L, const BinView& bv, bool batch, unsigned at,
                                          int64_t E_al, LaneRow& r, bool all = false) {
    r.k = bv.slot(at);
    r.v = bv.list[r.k];
    r.st = s.off[r.v];
    const int64_t en = s.off_end[r.v];
    r.d = (int)(en - r.st);
    if (!all && !is_long(r.st, en, E_al)) return false;
    if (batch && s.done[s.gid[r.v]]) {
        const int32_t own = L.C[r.v];               // a done graph's vertex keeps its label
        record_label<false>(L, bv.chg + r.k, r.v, own, own, false);
        return false;
    }
    return true;
}

// After a warp scanned vertex v of row [st, en) (frontier slot k): its label, the
// counts, and its neighbours' marks.  All 32 lanes must call.
__device__ __forceinline__ void finish_long(const DevState& s, const Labels& L, const BinView& bv, bool batch, bool marks,
                                            unsigned k, int32_t v, int64_t st, int64_t en, int32_t own, int32_t best,
                                            unsigned long long& my_changed, unsigned long long& my_changed_entries) {
    const unsigned lane = lane_id();
    const bool changed = best >= 0 && best != own;      // warp-uniform
    if (lane == 0) {
        record_label<false>(L, bv.chg + k, v, own, best, changed);
        if (changed) {
            ++my_changed;
            my_changed_entries += (unsigned long long)(en - st);
            if (batch) atomicAdd(&s.dN[s.gid[v]], 1ull);
        }
    }
    if (changed && marks) {
        for (int64_t e0 = st + lane; e0 < en; e0 += 128) {
            int32_t jj[4];
            uint8_t f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) jj[u] = e0 + 32 * u < en ? s.idx[e0 + 32 * u] : v;
#pragma unroll
            for (int u = 0; u < 4; ++u) f[u] = jj[u] != v ? __ldcg(s.flags + jj[u]) : (uint8_t)1;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (f[u] == 0) s.flags[jj[u]] = 1;
        }
    }
}

// Blocks per SM that the registers are to allow.  Rows are sorted faster by 16
// warps with 128 registers each than by 20 with 96 (one sort after another: planted
// partitions of 130,000 vertices, unit weights 389 -> 352 us a run, weights 1..4
// 578 -> 542; 256 of them in a batch 20.18 -> 19.87 ms), except where the weight
// columns leave room for 12 warps only (fp32, 1 M vertices: 8.94 ms at up to 168
// registers, 8.82 at 128, 8.69 at 96) and where longer rows, a warp each, want 20
// (200,000 vertices of mean degree 120, unit weights: 1.96 ms with 16, 1.72).
template <int KM, bool SHARE>
constexpr int kLaneBlocks = KM == KEY_PLACE || SHARE ? 5 : 4;

// Rows that no lane can take are left to k_sweep_long (take_long 0) or scanned by
// the warp that meets them; SHARE: shared out where warps are to spare (compiled
// in for graphs without such rows, that takes 2% of a sweep of short ones).
template <int KM, int WK, bool NS, bool SHARE>
__global__ void __launch_bounds__(kLaneWarps * 32, kLaneBlocks<KM, SHARE>) k_sweep_lane(DevState s, int flag_neighbours, int take_long) {
    using T = typename Acc<WK>::T;
    using Sh = LaneShape<KM, WK>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned lane = lane_id();
    const int wib = threadIdx.x >> 5;
    const bool batch = s.G > 1;
    uint4* queue = reinterpret_cast<uint4*>(smem_raw + (size_t)wib * Sh::WARP_BYTES);    // pack_row()
    unsigned char* mem = reinterpret_cast<unsigned char*>(queue) + Sh::QUEUES;
    uint32_t* col = reinterpret_cast<uint32_t*>(mem) + lane;                             // sorted keys, entry i at [32 i]
    [[maybe_unused]] T* wts = reinterpret_cast<T*>(mem + Sh::COLUMNS) + lane;            // place i at [32 i]

    const BinView bv = bin_view(s, 1);
    const Labels L = labels_of(s);
    const bool marks = marks_on(s, flag_neighbours);
    const uint32_t sweep = NS ? (uint32_t)s.ctrl->iter + 1u : 0u;   // non-strict tie-break (Section 4.1.5)
    const unsigned cnt = bv.cnt;
    const int64_t E_al = s.E & ~(int64_t)3;                                // 16-byte loads end here
    unsigned long long my_changed = 0, my_changed_entries = 0;

    // Each active lane scans the vertex of its queue entry.
    auto step = [&](bool act, const LaneRow& r, int halves) {
        const unsigned k = r.k;
        const int32_t v = r.v;
        const int64_t st = r.st, en = st + r.d;
        const int d = act ? r.d : 0;
        const int32_t own = act ? L.C[v] : 0;
        const TieRule tr = tie_rule(s, NS && act, sweep, v);
        int32_t best = -1;
        best = lane_pick<KM, WK, NS>(s, L.C, v, st, d, tr, halves, col, wts);
        const bool changed = act && best >= 0 && best != own;
        if (act) record_label<false>(L, bv.chg + k, v, own, best, changed);
        if (changed) {
            ++my_changed;
            my_changed_entries += (unsigned)d;
            if (marks) {
                for (int64_t a = st & ~(int64_t)3; a < en; a += 8) {
                    int32_t j[8];
                    uint8_t f[8];
                    const int4 x = __ldg(reinterpret_cast<const int4*>(s.idx + a));
                    const int4 y = a + 4 < en ? __ldg(reinterpret_cast<const int4*>(s.idx + a + 4)) : make_int4(v, v, v, v);
                    const int32_t z[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int c = 0; c < 8; ++c) j[c] = a + c >= st && a + c < en ? z[c] : v;
#pragma unroll
                    for (int c = 0; c < 8; ++c) f[c] = j[c] != v ? __ldcg(s.flags + j[c]) : (uint8_t)1;
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (f[c] == 0) s.flags[j[c]] = 1;
                }
            }
        }
        __syncwarp();
        if (batch) count_graph_changes<true>(s, changed, v);
    };

    // The whole warp scans the vertex of one queue entry.
    auto long_step = [&](const LaneRow& r) {
        const int32_t v = r.v;
        const int64_t st = r.st, en = st + r.d;
        const int32_t own = L.C[v];
        const TieRule tr = tie_rule(s, NS, sweep, v);
        uint32_t key = 0, tie = 0xffffffffu;
        const int32_t j = (int)lane < r.d ? load_index_keep(s.idx, st + lane) : v;
        const bool ok = j != v;
        const int32_t lab[1] = {ok ? load_label<false>(L.C, j) : kEmptyKey};
        const T w[1] = {ok ? load_weight<WK>(s.w, st + lane) : (T)0};
        int32_t* keys = reinterpret_cast<int32_t*>(mem);
        T* vals = reinterpret_cast<T*>(keys + 512);
        warp_long_row<false, WK>(s, L, keys, vals, reinterpret_cast<unsigned*>(vals + 512), 9, tr, st, en, v, lab, w, key,
                                 tie);
        const uint32_t best_key = warp_argmax_tie(key, tie);
        const int32_t best = best_key == 0xffffffffu ? -1 : tr.label(best_key);
        finish_long(s, L, bv, batch, marks, r.k, v, st, en, own, best, my_changed, my_changed_entries);
    };

    if (!batch && identity_sweep<false, false>(s)) {
        identity_rows<WK, NS>(s, L, bv, marks, sweep, E_al);
        return;
    }

    // Consecutive chunks of 32 frontier entries go to different blocks, so a
    // small frontier spreads over the chip.  The vertices and rows of the next
    // chunk are loaded while this one is scanned.
    const unsigned nchunks = (cnt + 31u) / 32u;
    const unsigned nwarps = gridDim.x * kLaneWarps;
    unsigned chunk = (unsigned)wib * gridDim.x + blockIdx.x;
    unsigned n[kLaneQueues];
#pragma unroll
    for (int q = 0; q < kLaneQueues; ++q) n[q] = 0u;
    // Where at least half of the warps have no chunk, these read the frontier a
    // second time and take its longer rows, one part of at most 32 entries each
    // (otherwise the rows of a chunk are scanned one after another: 2,000 vertices
    // of degree 90, unit weights, 5 sweeps: 320 us, so 110).
    const bool shared_out = SHARE && nchunks * 2u <= nwarps;
    if (shared_out && chunk >= nchunks) {
        const unsigned others = nwarps - nchunks, width = (cnt + others - 1u) / others;     // <= 32
        const unsigned k = (chunk - nchunks) * width + lane;
        LaneRow r{};
        const bool mine = lane < width && k < cnt && load_long(s, L, bv, batch, k, E_al, r);
        const unsigned m = __ballot_sync(kFull, mine);
        if (mine) queue[kLong * kLaneQueueCap + __popc(m & lanes_below())] = pack_row(r);
        n[kLong] = __popc(m);
        __syncwarp();
    }
    const bool longs = take_long && !shared_out;
    unsigned k_c = 0, k_n = 0;                      // their slots in the frontier list
    auto vertex_of = [&](unsigned c, unsigned& slot) -> int32_t {
        const unsigned k = c * 32u + lane;
        if (c >= nchunks || k >= cnt) return -1;
        slot = bv.slot(k);
        return bv.list[slot];
    };
    int32_t v_c = vertex_of(chunk, k_c), v_n = vertex_of(chunk + nwarps, k_n);
    int64_t st_c = 0, en_c = 0;
    int32_t done_c = 0;
    auto load_row = [&]() {
        if (v_c >= 0) {
            st_c = s.off[v_c];
            en_c = s.off_end[v_c];
            if (batch) done_c = s.done[s.gid[v_c]];
        }
    };
    load_row();
    for (;;) {
        bool full = false;
#pragma unroll
        for (int q = 0; q < kLaneQueues; ++q) full = full || n[q] >= 32u;
        if (!full && chunk < nchunks) {
            // sort the chunk's vertices into the queues
            LaneRow r;
            r.k = k_c;
            r.v = v_c;
            r.st = st_c;
            r.d = (int)(en_c - st_c);
            int cls = -1;
            if (v_c >= 0) {
                cls = is_long(st_c, en_c, E_al) ? kLong : en_c - (st_c & ~(int64_t)3) <= kSortSlots ? 0 : 1;
                if (cls == kLong && !longs) cls = -1;               // other warps take it
                if (batch && done_c && cls >= 0) {
                    cls = -1;                       // a done graph's vertex keeps its label
                    const int32_t own = L.C[v_c];
                    record_label<false>(L, bv.chg + r.k, v_c, own, own, false);
                }
            }
#pragma unroll
            for (int q = 0; q < kLaneQueues; ++q) {
                const unsigned m = __ballot_sync(kFull, cls == q);
                if (cls == q) queue[q * kLaneQueueCap + n[q] + __popc(m & lanes_below())] = pack_row(r);
                n[q] += __popc(m);
            }
            __syncwarp();
            chunk += nwarps;
            v_c = v_n;
            k_c = k_n;
            v_n = vertex_of(chunk + nwarps, k_n);
            load_row();
            continue;
        }
        if (n[kLong] >= 32u || (!full && n[kLong] > 0u)) {
            // the table is cleared here once; each row leaves it clear
            uint32_t* table = reinterpret_cast<uint32_t*>(mem);
            for (int q = lane; q < 512 * kTableWords<WK>; q += 32) table[q] = q < 512 ? (uint32_t)kEmptyKey : 0u;
            __syncwarp();
            while (n[kLong] > 0u) long_step(unpack_row(queue[kLong * kLaneQueueCap + --n[kLong]]));
            __syncwarp();
            continue;
        }
        // up to 32 rows: one full queue, or at the end of the pass what is
        // left in the queues, the longest rows first
        unsigned left = 32u, first = 0u;
        int halves = 0;
        uint4 at = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int q = kLong - 1; q >= 0; --q) {
            const bool from = full ? (n[q] >= 32u && left == 32u) : true;
            const unsigned take = from ? min(n[q], left) : 0u;
            left -= take;
            n[q] -= take;
            if (take && halves == 0) halves = q + 1;
            if (lane >= first && lane < first + take) at = queue[q * kLaneQueueCap + n[q] + lane - first];
            first += take;
        }
        if (first == 0u) break;                     // nothing left
        __syncwarp();
        step(lane < first, unpack_row(at), halves);
    }
    flush_bin_counts(s, 1, my_changed, my_changed_entries);
}

// ---- longer rows, a warp per row -------------------------------------------
// The rows that no lane can take, or (`all`) every row of the bin.  Each warp
// goes through chunks of the frontier, as small as gives every warp one, and
// collects their longer rows in a queue; while one row is scanned, the labels and
// weights of the next one's first kAhead x 32 entries and the ids of the one after
// that are on their way (labels do not change during a synchronous sweep).
//
// fp32 rows spend their time in the table (a claim, a lane mask and ordered sums
// per chunk of 32 entries), one row's steps waiting for each other, so it takes
// warps to hide them: inside k_sweep_lane, whose weight columns leave room for 12
// warps per SM, planted partitions of 200,000 vertices and mean degree 80 took
// 4.23 ms a run, here 2.51 (a warp per row with table atomics for every row of the
// bin, before k_sweep_lane came: 2.86).
constexpr int kLongWarps = 8;           // per block
constexpr int kAhead = 4;

template <int WK, bool NS>
__global__ void __launch_bounds__(kLongWarps * 32, 3) k_sweep_long(DevState s, int flag_neighbours, int all) {
    using T = typename Acc<WK>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned lane = lane_id();
    const int wib = threadIdx.x >> 5;
    const bool batch = s.G > 1;
    const bool ident = !batch && identity_sweep<false, false>(s);
    if (ident && !all) return;                      // k_sweep_lane took every row
    const unsigned slots = (unsigned)s.warp_slots;
    const int log_slots = ceil_log2(slots);
    const size_t warp_bytes = kLaneQueueCap * sizeof(uint4) + (size_t)slots * 4 * kTableWords<WK>;
    uint4* queue = reinterpret_cast<uint4*>(smem_raw + (size_t)wib * warp_bytes);
    int32_t* keys = reinterpret_cast<int32_t*>(queue + kLaneQueueCap);
    T* vals = reinterpret_cast<T*>(keys + slots);
    unsigned* peers_of = reinterpret_cast<unsigned*>(vals + slots);
    for (unsigned q = lane; q < slots * kTableWords<WK>; q += 32) keys[q] = q < slots ? kEmptyKey : 0;

    const BinView bv = bin_view(s, 1);
    const Labels L = labels_of(s);
    const bool marks = marks_on(s, flag_neighbours);
    const uint32_t sweep = NS ? (uint32_t)s.ctrl->iter + 1u : 0u;   // non-strict tie-break (Section 4.1.5)
    const unsigned cnt = bv.cnt;
    const int64_t E_al = s.E & ~(int64_t)3;
    if (ident) {
        identity_rows<WK, NS>(s, L, bv, marks, sweep, E_al);
        return;
    }
    unsigned long long my_changed = 0, my_changed_entries = 0;

    auto load_ids = [&](const LaneRow& r, int32_t (&j)[kAhead]) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            j[u] = 32 * u + (int)lane < r.d ? load_index_keep(s.idx, r.st + 32 * u + lane) : r.v;
    };
    auto load_labels = [&](const LaneRow& r, const int32_t (&j)[kAhead], int32_t& own, int32_t (&lab)[kAhead],
                           T (&w)[kAhead]) {
        own = L.C[r.v];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const bool ok = j[u] != r.v;
            lab[u] = ok ? load_label<false>(L.C, j[u]) : kEmptyKey;
            w[u] = ok ? load_weight<WK>(s.w, r.st + 32 * u + lane) : (T)0;
        }
    };
    // the queue's `rows` vertices, one after another
    auto scan_queue = [&](unsigned rows) {
        LaneRow now = unpack_row(queue[0]), next = unpack_row(queue[rows > 1u ? 1 : 0]);
        int32_t ids[kAhead], lab[kAhead], own = 0;
        T w[kAhead];
        load_ids(now, ids);
        load_labels(now, ids, own, lab, w);
        load_ids(next, ids);
#pragma unroll 1
        for (unsigned i = 0; i < rows; ++i) {
            int32_t next_lab[kAhead], next_own = 0;
            T next_w[kAhead];
            load_labels(next, ids, next_own, next_lab, next_w);
            const LaneRow after = unpack_row(queue[min(i + 2u, rows - 1u)]);
            load_ids(after, ids);
            const TieRule tr = tie_rule(s, NS, sweep, now.v);
            uint32_t key = 0, tie = 0xffffffffu;
            const int64_t en = now.st + now.d;
            warp_long_row<false, WK>(s, L, keys, vals, peers_of, log_slots, tr, now.st, en, now.v, lab, w, key, tie);
            const uint32_t best_key = warp_argmax_tie(key, tie);
            const int32_t best = best_key == 0xffffffffu ? -1 : tr.label(best_key);
            finish_long(s, L, bv, batch, marks, now.k, now.v, now.st, en, own, best, my_changed, my_changed_entries);
            now = next;
            next = after;
            own = next_own;
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                lab[u] = next_lab[u];
                w[u] = next_w[u];
            }
        }
        __syncwarp();
    };

    const unsigned nwarps = gridDim.x * kLongWarps;
    const unsigned width = max(1u, min(32u, (cnt + nwarps - 1u) / nwarps));
    const unsigned nchunks = (cnt + width - 1u) / width;
    unsigned n = 0;                                 // rows in the queue
    for (unsigned chunk = (unsigned)wib * gridDim.x + blockIdx.x; chunk < nchunks; chunk += nwarps) {
        const unsigned at = chunk * width + lane;
        LaneRow r{};
        const bool mine = lane < width && at < cnt && load_long(s, L, bv, batch, at, E_al, r, all != 0);
        const unsigned m = __ballot_sync(kFull, mine);
        if (mine) queue[n + __popc(m & lanes_below())] = pack_row(r);
        n += __popc(m);
        __syncwarp();
        if (n >= 32u) {
            scan_queue(n);
            n = 0;
        }
    }
    if (n > 0u) scan_queue(n);
    flush_bin_counts(s, 1, my_changed, my_changed_entries);
}

template <int WK, bool NS>
static cudaError_t launch_long_k(const DevState& s, int flag, int all, cudaStream_t st, int sms) {
    constexpr int threads = kLongWarps * 32;
    const size_t smem = kLongWarps * (kLaneQueueCap * sizeof(uint4) + (size_t)s.warp_slots * 4 * kTableWords<WK>);
    auto kern = k_sweep_long<WK, NS>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    kern<<<sms * per_sm, threads, smem, st>>>(s, flag, all);
    return cudaGetLastError();
}

// Appends the nodes that the next launch captured from st would depend on (none
// outside a capture, or at the beginning of one).
static cudaError_t captured_deps(cudaStream_t st, std::vector<cudaGraphNode_t>& deps) {
    cudaStreamCaptureStatus status;
    cudaGraph_t graph = nullptr;
    const cudaGraphNode_t* d = nullptr;
    size_t n = 0;
    const cudaError_t err = cudaStreamGetCaptureInfo(st, &status, nullptr, &graph, &d, nullptr, &n);
    if (err == cudaSuccess && status == cudaStreamCaptureStatusActive) deps.insert(deps.end(), d, d + n);
    return err;
}

static cudaError_t set_deps(cudaStream_t st, std::vector<cudaGraphNode_t>& deps) {
    return cudaStreamUpdateCaptureDependencies(st, deps.data(), nullptr, deps.size(), cudaStreamSetCaptureDependencies);
}

template <int KM, int WK, bool NS, bool SHARE>
static cudaError_t launch_lane_k(const DevState& s, int flag, cudaStream_t st, int sms) {
    constexpr int threads = kLaneWarps * 32;
    const bool apart = KM == KEY_PLACE && s.long_rows == 2;
    const size_t smem = kLaneWarps * LaneShape<KM, WK>::WARP_BYTES;
    auto kern = k_sweep_lane<KM, WK, NS, SHARE>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    // The two kernels write different vertices, so a captured sweep runs them side
    // by side: the second takes the first one's dependencies, what follows waits
    // for both (one after the other, a batch of 64 planted partitions, 3.2 M
    // entries, fp32 weights, lost 4 of 32 us a sweep).
    std::vector<cudaGraphNode_t> before, both;
    if (apart && (err = captured_deps(st, before)) != cudaSuccess) return err;
    kern<<<sms * per_sm, threads, smem, st>>>(s, flag, apart ? 0 : 1);
    err = cudaGetLastError();
    if constexpr (KM == KEY_PLACE) {
        if (err != cudaSuccess || !apart) return err;
        if (before.empty()) return launch_long_k<WK, NS>(s, flag, 0, st, sms);
        if ((err = captured_deps(st, both)) != cudaSuccess) return err;
        if ((err = set_deps(st, before)) != cudaSuccess) return err;
        if ((err = launch_long_k<WK, NS>(s, flag, 0, st, sms)) != cudaSuccess) return err;
        if ((err = captured_deps(st, both)) != cudaSuccess) return err;
        err = set_deps(st, both);
    }
    return err;
}

template <int KM, int WK, bool NS>
static cudaError_t launch_lane_s(const DevState& s, int flag, cudaStream_t st, int sms) {
    if constexpr (KM != KEY_PLACE) {
        if (s.long_rows) return launch_lane_k<KM, WK, NS, true>(s, flag, st, sms);
    }
    return launch_lane_k<KM, WK, NS, false>(s, flag, st, sms);
}

template <int KM, int WK>
static cudaError_t launch_lane_t(const DevState& s, int flag, int ns, cudaStream_t st, int sms) {
    return ns ? launch_lane_s<KM, WK, true>(s, flag, st, sms) : launch_lane_s<KM, WK, false>(s, flag, st, sms);
}

// The key layout of the graph's rows, -1 if none fits.
static int key_of(const DevState& s) {
    if (s.weight_kind == W_UNIT) return KEY_LABEL;
    if (s.weight_kind != W_F32 && s.weight_bits > 0 && s.weight_bits < 32 && s.N < (1ll << (32 - s.weight_bits)))
        return KEY_PACKED;
    // 16-byte loads of 4-byte weights (the caller's own array may start anywhere)
    const bool aligned = s.weight_kind == W_U8 || (reinterpret_cast<uintptr_t>(s.w) & 15u) == 0;
    return aligned && s.N < (1ll << (32 - kPosBits)) ? KEY_PLACE : -1;
}

int lane_long_rows(const DevState& s, int64_t max_degree) {
    if (max_degree <= kLaneEntries || s.warp_max <= kLaneEntries) return 0;
    return key_of(s) == KEY_PLACE ? 2 : 1;
}

template <int WK>
static cudaError_t launch_lane_w(const DevState& s, int flag, int ns, cudaStream_t st, int sms) {
    if constexpr (WK == W_UNIT) {
        return launch_lane_t<KEY_LABEL, WK>(s, flag, ns, st, sms);
    } else {
        const int key = key_of(s);
        if constexpr (WK != W_F32) {
            if (key == KEY_PACKED) return launch_lane_t<KEY_PACKED, WK>(s, flag, ns, st, sms);
        }
        if (key == KEY_PLACE) return launch_lane_t<KEY_PLACE, WK>(s, flag, ns, st, sms);
        return ns ? launch_long_k<WK, true>(s, flag, 1, st, sms) : launch_long_k<WK, false>(s, flag, 1, st, sms);
    }
}

cudaError_t launch_sweep_lane(const DevState& s, int mode, cudaStream_t st, int sms) {
    const int ns = (mode & kModeNonstrict) != 0;
    const int flag = (mode & ~kModeNonstrict) != MODE_SYNC_FULL;
    switch (s.weight_kind) {
        case W_UNIT: return launch_lane_w<W_UNIT>(s, flag, ns, st, sms);
        case W_U32: return launch_lane_w<W_U32>(s, flag, ns, st, sms);
        case W_U8: return launch_lane_w<W_U8>(s, flag, ns, st, sms);
        default: return launch_lane_w<W_F32>(s, flag, ns, st, sms);
    }
}

}  // namespace lpa
