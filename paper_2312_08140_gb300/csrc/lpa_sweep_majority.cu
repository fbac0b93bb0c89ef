// lpa_sweep_majority.cu -- sweeps that one label dominates.
//
// On graphs with hubs (web and social graphs) a label takes nearly every edge
// end within a sweep or two, and each later sweep spends its time finding out
// that row after row still has that label as its heaviest: one random 4-byte
// gather per entry, which costs a 32-byte sector and, once the label array
// outgrows L2, a DRAM access (measured on GB300: 296 G gathers/s from L2, 77
// G/s at random over 256 MB).  If a label's weight in a row exceeds the weight
// of all other entries together it is the row's pick (Eq. 2, Section 3.3) under
// either tie-break, whatever the others are.  So, before the ordinary kernels
// of a sweep's main pass:
//
//   k_dom_pick    samples 4096 entries' labels and finds the label, if any, that
//                 holds 5/8 of them (in the first asynchronous sweep, whose hubs
//                 and low-degree vertices have their new labels by then, also
//                 before the 128- and the 256-thread bin);
//   k_dom_bits    sets bit v for each vertex v that carries it: 32 vertices per
//                 word, so the array that the rows read is 1/32 of the labels
//                 (8 MB for 67 M vertices, and largely L1 hits);
//   k_majority_*  walk the rows, adding up the weight of entries whose bit is
//                 set, and stop as soon as the label's weight exceeds the rest
//                 of the row, read or not -- about half of an agreeing row.
//                 The row is then settled; other rows are listed and left to the
//                 bin's ordinary kernel.
//
// A frontier of fewer than kMajorityEntries entries (lpa_internal.h) is left to
// the ordinary kernels without a search.  A synchronous sweep takes the rows of
// all bins in one launch, where a block that runs out of rows of one bin goes on
// with the next; an asynchronous pass takes each bin before its ordinary kernel,
// as rows of one bin may read the new labels of the bins before.  R-MAT 22,
// synchronous: 1358 -> 1134 us a run by that; a long tail (R-MAT 20, edge factor
// 8, tolerance 0, 100 sweeps) 8.6 -> 5.4 ms (6.6 without majority kernels, by the
// ordinary kernels of the time).
//
// Measured on R-MAT 26 (1.84 G entries, asynchronous): the three row bins of the
// second and third sweep 20.5 -> 5.4 ms, the warp bin there 4.3 -> 0.95, the 128-
// and 256-thread bins of the first sweep 9.7 -> 3.5.
//
// In the asynchronous mode a vertex that leaves the label clears its bit
// (write_label in lpa_device.cuh); the words are read through L1, so a row may
// still see a label that its neighbour had earlier in the same pass, as it may
// through the ordinary kernels' prefetch.  fp32 weights ask for a margin above
// the rounding of any summation order of the row.
#include "lpa_warp_row.cuh"

namespace lpa {

constexpr int kPickThreads = 1024;
constexpr int kPickSamples = 4;             // per thread
constexpr int kMajThreads = 256;
constexpr int kMajVec = 2;                  // 4-entry vectors per lane and step

// `mid`: between two bins of the first asynchronous sweep, where the bins before
// have just left their own labels; otherwise before a later sweep.  The label
// must hold `need` / 16 of the samples.
__global__ void __launch_bounds__(kPickThreads) k_dom_pick(DevState s, int mid, int need) {
    __shared__ int ones[31], same;
    Ctrl* c = s.ctrl;
    if ((c->iter == 0) != (mid != 0)) return;
    // a frontier of a few rows is not worth the search (the label stays off)
    unsigned long long entries = 0;
#pragma unroll
    for (int b = 1; b < kBins; ++b) entries += c->bin_entries[c->rd][b];
    if (entries < (unsigned long long)kMajorityEntries) return;
    if (threadIdx.x < 31) ones[threadIdx.x] = 0;
    if (threadIdx.x == 31) same = 0;
    __syncthreads();
    const int32_t* C = s.lab[c->cbuf];
    const uint64_t seed = ((uint64_t)c->iter << 32) + ((uint64_t)need << 48);
    int32_t lab[kPickSamples];
#pragma unroll
    for (int q = 0; q < kPickSamples; ++q) {
        const uint64_t e = splitmix64(seed + (uint64_t)(q * kPickThreads) + threadIdx.x) % (uint64_t)s.E;
        lab[q] = __ldcg(C + __ldg(s.idx + e));
    }
    // a label that holds more than half of the samples has the majority's value
    // in every bit (and most often one that holds a good part of them); the
    // count below decides
    const unsigned lane = lane_id();
    for (int b = 0; b < 31; ++b) {
        int n = 0;
#pragma unroll
        for (int q = 0; q < kPickSamples; ++q) n += __popc(__ballot_sync(kFull, (lab[q] >> b) & 1));
        if (lane == 0) atomicAdd(&ones[b], n);
    }
    __syncthreads();
    int32_t label = 0;
    for (int b = 0; b < 31; ++b)
        if (2 * ones[b] > kPickThreads * kPickSamples) label |= 1 << b;
    int n = 0;
#pragma unroll
    for (int q = 0; q < kPickSamples; ++q) n += __popc(__ballot_sync(kFull, lab[q] == label));
    if (lane == 0) atomicAdd(&same, n);
    __syncthreads();
    if (threadIdx.x < kBins) {
        c->dom_next[threadIdx.x] = 0;
        c->defer_cnt[threadIdx.x] = 0;
    }
    if (threadIdx.x == 0) {
        c->dom_label = label;
        c->dom_on = 16 * same >= need * kPickThreads * kPickSamples ? 1 : 0;
    }
}

__global__ void __launch_bounds__(256) k_dom_bits(DevState s, int mid) {
    const Ctrl* c = s.ctrl;
    if (!c->dom_on || (c->iter == 0) != (mid != 0)) return;
    const int32_t* C = s.lab[c->cbuf];
    const int32_t label = c->dom_label;
    const unsigned lane = lane_id();
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    constexpr int U = 8;                    // words per warp and step
    for (int64_t w0 = warp * U; w0 * 32 < s.N; w0 += nwarps * U) {
        int32_t x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t v = (w0 + u) * 32 + lane;
            x[u] = v < s.N ? __ldcs(C + v) : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned m = __ballot_sync(kFull, x[u] == label);
            if (lane == (unsigned)u && (w0 + u) * 32 < s.N) s.dom_bits[w0 + u] = m;
        }
    }
}

// Before a sweep the label must hold 5/8 of the entries, before a row bin of the
// first asynchronous sweep 3/8: the ordinary kernels gather at the rate of DRAM
// sectors there, several times the cost of a bit that settles nothing.
cudaError_t launch_dominant(const DevState& s, int before_bin, cudaStream_t st, int sms) {
    const int mid = before_bin > 0;
    const int need = mid ? 6 : 10;
    k_dom_pick<<<1, kPickThreads, 0, st>>>(s, mid, need);
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    k_dom_bits<<<sms * 8, 256, 0, st>>>(s, mid);
    return cudaGetLastError();
}

// Weight of the label (in) and of the other entries (out) read so far; `rest`
// entries of the row are unread.
template <int WK>
struct MajSum {
    using A = typename std::conditional<WK == W_F32, float, unsigned long long>::type;
    A in, out;
};

// The label's weight exceeds everything else the row can hold.
template <int WK>
__device__ __forceinline__ bool settled(const DevState& s, const MajSum<WK>& m, int64_t rest, int64_t d) {
    if constexpr (WK == W_F32) {
        const float other = m.out + (float)rest * s.weight_max;
        // fp32 sums of d terms: relative error below d / 2^24 each, in any order
        const float slack = (m.in + other) * ((float)d * 2.4e-7f);
        return m.in > other + slack;
    } else if constexpr (WK == W_UNIT) {
        return m.in > m.out + (unsigned long long)rest;
    } else {
        return m.in > m.out + (unsigned long long)rest * (unsigned long long)s.weight_max;
    }
}

// The label can no longer exceed the others, or is unlikely to.
template <int WK>
__device__ __forceinline__ bool hopeless(const DevState& s, const MajSum<WK>& m, int64_t rest) {
    if constexpr (WK == W_F32) {
        return rest == 0 || 3.0f * m.in < m.out || m.in + (float)rest * s.weight_max <= m.out;
    } else {
        const unsigned long long w = WK == W_UNIT ? 1ull : (unsigned long long)s.weight_max;
        return rest == 0 || 3ull * m.in < m.out || m.in + (unsigned long long)rest * w <= m.out;
    }
}


// One step over a row: this thread's share of entries [e0, ...) added to
// in / out.  Threads 0..GROUP-1 take 4-entry vectors in turn.
template <int WK, int GROUP>
__device__ __forceinline__ void count_step(const DevState& s, int64_t e0, int64_t st, int64_t en, int32_t v,
                                           unsigned rank, typename Acc<WK>::T& in, typename Acc<WK>::T& out) {
    using T = typename Acc<WK>::T;
    int32_t j[kMajVec][4];
    uint32_t word[kMajVec][4];
#pragma unroll
    for (int u = 0; u < kMajVec; ++u) {
        const int64_t e = e0 + 4 * ((int64_t)GROUP * u + rank);
        if (e < en) {
            load_idx4(s.idx, e, st, en, v, j[u]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) j[u][c] = v;
        }
    }
#pragma unroll
    for (int u = 0; u < kMajVec; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) word[u][c] = j[u][c] != v ? __ldca(s.dom_bits + (j[u][c] >> 5)) : 0u;
#pragma unroll
    for (int u = 0; u < kMajVec; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (j[u][c] != v) {
                const int64_t e = e0 + 4 * ((int64_t)GROUP * u + rank) + c;
                const T w = load_weight<WK>(s.w, e);
                if ((word[u][c] >> (j[u][c] & 31)) & 1u) in += w;
                else out += w;
            }
        }
}

template <int WK, typename T>
__device__ __forceinline__ T warp_add(T x) {
    if constexpr (WK == W_F32) {
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        return x;
    } else {
        return __reduce_add_sync(kFull, x);
    }
}

// Appends the frontier slots of the lanes with `left` set to the bin's list.
__device__ __forceinline__ void leave_rows(const DevState& s, int bin, bool left, unsigned slot) {
    const unsigned m = __ballot_sync(kFull, left);
    if (m == 0u) return;
    unsigned base = 0;
    if (lane_id() == 0) base = atomicAdd(&s.ctrl->defer_cnt[bin], (unsigned)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (left) s.defer[s.bin_base[bin] + base + __popc(m & lanes_below())] = (int32_t)slot;
}

// Bin 1: a thread per row, 8 entries at a time.
template <bool ASYNC, int WK>
__device__ __forceinline__ void majority_lane(const DevState& s, int flag_neighbours) {
    using T = typename Acc<WK>::T;
    const Ctrl* c = s.ctrl;
    const int rd = c->rd;
    const Labels L = labels_of(s);
    const int32_t* list = (L.dense ? s.slist : s.flist) + s.bin_base[1];
    int32_t* chg = s.chg + s.bin_base[1];
    const unsigned cnt = c->bin_cnt[rd][1];
    const int32_t label = c->dom_label;
    const bool marks = marks_on(s, flag_neighbours);
    const bool po = ASYNC && c->prune_other != 0;
    unsigned long long my_changed = 0, my_changed_entries = 0;
    for (unsigned k0 = blockIdx.x * blockDim.x; k0 < cnt; k0 += gridDim.x * blockDim.x) {
        const unsigned k = k0 + threadIdx.x;
        const bool act = k < cnt;
        bool ok = false;
        if (act) {
            const int32_t v = list[k];
            const int64_t st = s.off[v], en = s.off_end[v];
            const int32_t own = ASYNC ? __ldcg(L.C + v) : L.C[v];
            MajSum<WK> m{};
            for (int64_t e = st & ~(int64_t)3; e < en; e += 4 * kMajVec) {
                T in = (T)0, out = (T)0;
                count_step<WK, 1>(s, e, st, en, v, 0u, in, out);
                m.in += in;
                m.out += out;
                const int64_t rest = max((int64_t)0, en - (e + 4 * kMajVec));
                ok = settled<WK>(s, m, rest, en - st);
                if (ok || hopeless<WK>(s, m, rest)) break;
            }
            if (ok) {
                const bool changed = own != label;
                record_label<ASYNC>(L, chg + k, v, own, label, changed);
                if (changed) {
                    ++my_changed;
                    my_changed_entries += (unsigned long long)(en - st);
                    if (marks)
                        for (int64_t e = st; e < en; ++e) {
                            const int32_t j = __ldg(s.idx + e);
                            if (j != v && !(po && load_label<ASYNC>(L.C, j) == label)) mark_unprocessed(s.flags, j);
                        }
                }
            }
        }
        __syncwarp();
        leave_rows(s, 1, act && !ok, k);
    }
    flush_bin_counts(s, 1, my_changed, my_changed_entries);
}

// Bins 2 and 3: a warp per row, 32 rows taken at a time.
template <bool ASYNC, int WK>
__device__ __forceinline__ void majority_rows(const DevState& s, int bin, int flag_neighbours) {
    using T = typename Acc<WK>::T;
    Ctrl* c = s.ctrl;
    const int rd = c->rd;
    const Labels L = labels_of(s);
    const int32_t* list = (L.dense ? s.slist : s.flist) + s.bin_base[bin];
    int32_t* chg = s.chg + s.bin_base[bin];
    const unsigned cnt = c->bin_cnt[rd][bin];
    const int32_t label = c->dom_label;
    const bool marks = marks_on(s, flag_neighbours);
    const bool po = ASYNC && c->prune_other != 0;
    const unsigned lane = lane_id();
    unsigned long long my_changed = 0, my_changed_entries = 0;
    for (;;) {
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&c->dom_next[bin], 32u);
        base = __shfl_sync(kFull, base, 0);
        if (base >= cnt) break;
        const unsigned k = base + lane;
        const bool act = k < cnt;
        const int32_t vl = act ? list[k] : 0;
        int64_t stl = 0, enl = 0;
        int32_t ownl = 0;
        if (act) {
            stl = s.off[vl];
            enl = s.off_end[vl];
            ownl = ASYNC ? __ldcg(L.C + vl) : L.C[vl];
        }
        const unsigned rows = min(32u, cnt - base);
        unsigned okm = 0u;                              // settled rows of the batch
        for (unsigned i = 0; i < rows; ++i) {
            const int32_t v = __shfl_sync(kFull, vl, i);
            const int64_t st = __shfl_sync(kFull, stl, i), en = __shfl_sync(kFull, enl, i);
            MajSum<WK> m{};
            bool ok = false;
            for (int64_t e = st & ~(int64_t)3; e < en; e += 128 * kMajVec) {
                T in = (T)0, out = (T)0;
                count_step<WK, 32>(s, e, st, en, v, lane, in, out);
                m.in += warp_add<WK>(in);
                m.out += warp_add<WK>(out);
                const int64_t rest = max((int64_t)0, en - (e + 128 * kMajVec));
                ok = settled<WK>(s, m, rest, en - st);  // warp-uniform
                if (ok || hopeless<WK>(s, m, rest)) break;
            }
            if (ok) {
                okm |= 1u << i;
                const bool changed = __any_sync(kFull, lane == i && ownl != label);
                if (changed && marks) mark_row<ASYNC, 32, 1>(s, L, st, en, v, lane, po, label);
            }
        }
        const bool ok = (okm >> lane) & 1u;
        if (act && ok) {
            const bool changed = ownl != label;
            record_label<ASYNC>(L, chg + k, vl, ownl, label, changed);
            if (changed) {
                ++my_changed;
                my_changed_entries += (unsigned long long)(enl - stl);
            }
        }
        leave_rows(s, bin, act && !ok, k);
    }
    flush_bin_counts(s, bin, my_changed, my_changed_entries);
}

// Last bin: a block per row.  The block's running sums are taken through three
// shared accumulators in turn, so one barrier per step suffices: step t adds
// into slot t % 3 before its barrier and every thread reads it after; the slot
// of step t + 1 was last read before the barrier of step t - 1 and is cleared
// during step t.
template <bool ASYNC, int WK>
__device__ __forceinline__ void majority_block(const DevState& s, int bin, int flag_neighbours) {
    using T = typename Acc<WK>::T;
    using A = typename MajSum<WK>::A;
    __shared__ A acc[3][2];
    __shared__ unsigned next_row;
    Ctrl* c = s.ctrl;
    const int rd = c->rd;
    const Labels L = labels_of(s);
    const int32_t* list = (L.dense ? s.slist : s.flist) + s.bin_base[bin];
    int32_t* chg = s.chg + s.bin_base[bin];
    const unsigned cnt = c->bin_cnt[rd][bin];
    const int32_t label = c->dom_label;
    const bool marks = marks_on(s, flag_neighbours);
    const bool po = ASYNC && c->prune_other != 0;
    const unsigned lane = lane_id();
    unsigned long long my_changed = 0, my_changed_entries = 0;
    if (threadIdx.x < 6) acc[threadIdx.x >> 1][threadIdx.x & 1] = (A)0;
    unsigned t = 0;
    for (;;) {
        if (threadIdx.x == 0) next_row = atomicAdd(&c->dom_next[bin], 1u);
        __syncthreads();
        const unsigned k = next_row;
        if (k >= cnt) break;                            // block-uniform
        const int32_t v = list[k];
        const int64_t st = s.off[v], en = s.off_end[v];
        const int32_t own = ASYNC ? __ldcg(L.C + v) : L.C[v];
        MajSum<WK> m{};
        bool ok = false;
        for (int64_t e = st & ~(int64_t)3; e < en; e += (int64_t)4 * kMajThreads * kMajVec, ++t) {
            T in = (T)0, out = (T)0;
            count_step<WK, kMajThreads>(s, e, st, en, v, threadIdx.x, in, out);
            in = warp_add<WK>(in);
            out = warp_add<WK>(out);
            if (lane == 0) {
                atomicAdd(&acc[t % 3][0], (A)in);
                atomicAdd(&acc[t % 3][1], (A)out);
            }
            if (threadIdx.x < 2) acc[(t + 1) % 3][threadIdx.x] = (A)0;
            __syncthreads();
            m.in += acc[t % 3][0];
            m.out += acc[t % 3][1];
            const int64_t rest = max((int64_t)0, en - (e + (int64_t)4 * kMajThreads * kMajVec));
            ok = settled<WK>(s, m, rest, en - st);      // block-uniform
            if (ok || hopeless<WK>(s, m, rest)) {
                ++t;
                break;
            }
        }
        if (ok) {
            const bool changed = own != label;
            if (threadIdx.x == 0) {
                record_label<ASYNC>(L, chg + k, v, own, label, changed);
                if (changed) {
                    ++my_changed;
                    my_changed_entries += (unsigned long long)(en - st);
                }
            }
            if (changed && marks) mark_row<ASYNC, kMajThreads, 2>(s, L, st, en, v, threadIdx.x, po, label);
        } else if (threadIdx.x == 0) {
            s.defer[s.bin_base[bin] + atomicAdd(&c->defer_cnt[bin], 1u)] = (int32_t)k;
        }
        __syncthreads();                                // next_row was read
    }
    flush_bin_counts(s, bin, my_changed, my_changed_entries);
}

// Asynchronous passes: one bin, before its ordinary kernel.  (`flag` is always 1;
// as a constant it cost k_majority_block 7% on R-MAT 26, 1640 -> 1755 us.)
template <int WK>
__global__ void __launch_bounds__(kMajThreads) k_majority_lane(DevState s, int flag) {
    if (!s.ctrl->dom_on) return;
    majority_lane<true, WK>(s, flag);
}
template <int WK>
__global__ void __launch_bounds__(kMajThreads) k_majority_rows(DevState s, int bin, int flag) {
    if (!s.ctrl->dom_on) return;
    majority_rows<true, WK>(s, bin, flag);
}
template <int WK>
__global__ void __launch_bounds__(kMajThreads) k_majority_block(DevState s, int bin, int flag) {
    if (!s.ctrl->dom_on) return;
    majority_block<true, WK>(s, bin, flag);
}

// Synchronous sweeps: every bin, as no row's pick depends on another's.
template <int WK>
__global__ void __launch_bounds__(kMajThreads) k_majority_all(DevState s, int flag_neighbours) {
    if (!s.ctrl->dom_on) return;
    majority_block<false, WK>(s, kBins - 1, flag_neighbours);
    for (int bin = kBins - 2; bin > 1; --bin) {
        __syncthreads();                                // flush_bin_counts' sums were read
        majority_rows<false, WK>(s, bin, flag_neighbours);
    }
    __syncthreads();
    majority_lane<false, WK>(s, flag_neighbours);
}

template <typename K>
static cudaError_t wave_of(K kern, int threads, int sms, int* blocks) {
    int per_sm = 0;
    const cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0);
    *blocks = sms * (per_sm > 0 ? per_sm : 1);
    return err;
}

template <int WK>
static cudaError_t launch_majority_w(const DevState& s, int mode, int bin, cudaStream_t st, int sms) {
    int blocks = 0;
    cudaError_t err;
    if (mode == MODE_ASYNC && bin == 1) {
        if ((err = wave_of(k_majority_lane<WK>, kMajThreads, sms, &blocks)) != cudaSuccess) return err;
        k_majority_lane<WK><<<blocks, kMajThreads, 0, st>>>(s, 1);
    } else if (mode == MODE_ASYNC && bin < kBins - 1) {
        if ((err = wave_of(k_majority_rows<WK>, kMajThreads, sms, &blocks)) != cudaSuccess) return err;
        k_majority_rows<WK><<<blocks, kMajThreads, 0, st>>>(s, bin, 1);
    } else if (mode == MODE_ASYNC) {
        if ((err = wave_of(k_majority_block<WK>, kMajThreads, sms, &blocks)) != cudaSuccess) return err;
        k_majority_block<WK><<<blocks, kMajThreads, 0, st>>>(s, bin, 1);
    } else {
        if ((err = wave_of(k_majority_all<WK>, kMajThreads, sms, &blocks)) != cudaSuccess) return err;
        k_majority_all<WK><<<blocks, kMajThreads, 0, st>>>(s, mode != MODE_SYNC_FULL);
    }
    return cudaGetLastError();
}

cudaError_t launch_majority(const DevState& s, int mode, int bin, cudaStream_t st, int sms) {
    const int base = mode & ~kModeNonstrict;
    switch (s.weight_kind) {
        case W_UNIT: return launch_majority_w<W_UNIT>(s, base, bin, st, sms);
        case W_U32: return launch_majority_w<W_U32>(s, base, bin, st, sms);
        case W_U8: return launch_majority_w<W_U8>(s, base, bin, st, sms);
        default: return launch_majority_w<W_F32>(s, base, bin, st, sms);
    }
}

}  // namespace lpa
