// lpa_warp_row.cuh -- a whole warp (or block) on one row: 16-byte reads of a
// row's ids and its neighbours' marks (row and majority kernels), per-label
// sums by lane groups and a per-warp open-addressing table in shared memory
// (warp kernel), and the label sums of a row that no lane sorts (lane kernels).
#pragma once

#include "lpa_device.cuh"

namespace lpa {

constexpr int kWarpUnroll = 3;      // chunks of 32 entries in flight per warp beyond the first

// Entries [e, e + 4) of idx (e a multiple of 4, e < en; idx starts at a
// 16-byte aligned address): one 16-byte load where the vector lies inside the
// row [st, en), else entry by entry; entries outside the row read as `fill`.
__device__ __forceinline__ void load_idx4(const int32_t* idx, int64_t e, int64_t st, int64_t en, int32_t fill,
                                          int32_t (&j)[4]) {
    if (e >= st && e + 4 <= en) {
        const int4 x = __ldg(reinterpret_cast<const int4*>(idx + e));
        j[0] = x.x;
        j[1] = x.y;
        j[2] = x.z;
        j[3] = x.w;
    } else {
        // the first or last vector of the row
#pragma unroll
        for (int c = 0; c < 4; ++c) j[c] = (e + c >= st && e + c < en) ? __ldg(idx + e + c) : fill;
    }
}

// Marks the neighbours of changed vertex v unprocessed (Section 4.1.4): the
// GROUP threads of rank 0..GROUP-1 walk row [st, en) in 4-entry vectors,
// VEC vectors per thread in flight (their ids, then their flags, then the
// stores).  FLPA's rule (po) leaves a neighbour already carrying `best`.
template <bool ASYNC, int GROUP, int VEC>
__device__ __forceinline__ void mark_row(const DevState& s, const Labels& L, int64_t st, int64_t en, int32_t v,
                                         unsigned rank, bool po, int32_t best) {
    for (int64_t e0 = (st & ~(int64_t)3) + 4 * (int64_t)rank; e0 < en; e0 += 4 * GROUP * VEC) {
        int32_t j[VEC][4];
        uint8_t f[VEC][4];
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            const int64_t e = e0 + 4 * GROUP * u;
            if (e < en) {
                load_idx4(s.idx, e, st, en, v, j[u]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) j[u][c] = v;
            }
        }
#pragma unroll
        for (int u = 0; u < VEC; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) f[u][c] = j[u][c] != v ? __ldcg(s.flags + j[u][c]) : (uint8_t)1;
#pragma unroll
        for (int u = 0; u < VEC; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (f[u][c] == 0 && !(po && load_label<ASYNC>(L.C, j[u][c]) == best)) s.flags[j[u][c]] = 1;
    }
}

// Words of a table slot: label, sum, and the lane mask of fp32 sums.
template <int WK>
constexpr int kTableWords = WK == W_F32 ? 3 : 2;

// Sum of the weights of the lanes in `peers` (a lane's own group, itself
// included), the same value in every lane of the group.  fp32: added in lane
// order, one shuffle per member of the largest group in the warp, so the
// result does not depend on the schedule.  All 32 lanes must call.
__device__ __forceinline__ float ordered_group_sum(unsigned peers, float w) {
    const int most = (int)__reduce_max_sync(kFull, (unsigned)__popc(peers));
    float sum = 0.f;
    for (int q = 0; q < most; ++q) {
        const float wq = __shfl_sync(kFull, w, peers ? __ffs(peers) - 1 : 0);
        if (peers) sum += wq;
        peers &= peers - 1u;
    }
    return sum;
}

// Slot of `label` in the warp's table, claimed if the label is not there yet
// (free slots hold kEmptyKey; the table has at least twice as many slots as a
// row has entries, so a free one is always found; the probe is bounded by the
// table all the same).  Returns -1 when the bound was reached.
__device__ __forceinline__ int claim_slot(int32_t* keys, int log_slots, int32_t label) {
    const unsigned mask = (1u << log_slots) - 1u;
    unsigned h = slot_of(label, log_slots);
    for (unsigned p = 0; p <= mask; ++p) {
        const int32_t old = atomicCAS(keys + h, kEmptyKey, label);
        if (old == kEmptyKey || old == label) return (int)h;
        h = (h + 1u) & mask;
    }
    return -1;
}

// Offers (sum, label) as this lane's candidate: the larger sum key (0 = none),
// then the smaller tie key.
template <typename T>
__device__ __forceinline__ void offer_candidate(const TieRule& tr, T sum, int32_t lab, uint32_t& key, uint32_t& tie) {
    const uint32_t k = sum_key(sum), t = tr.key(lab);
    if (k > key || (k == key && t < tie)) {
        key = k;
        tie = t;
    }
}

// Row [st, en) of vertex v (en - st at most half the table's slots, and 256):
// this lane's best (sum key, tie key).  lab0[c] and w0[c] are the label and
// weight of entry 32 c + lane (kEmptyKey: none), loaded by the caller.  The table
// is all free slots before and after.  All 32 lanes must call.
//
// The label of the row's first entry is summed apart, by votes: once
// communities form it is most often the label of nearly the whole row, and its
// lanes would all meet in one slot (33 cycles of an SM for 32 lanes adding to
// one word, against 2 for distinct words).  Entries of other labels go into
// the table; each lane remembers the slots of its entries (16 bits per chunk
// of 32 entries) and reads their sums when the row is complete.
template <bool ASYNC, int WK, int K>
__device__ __forceinline__ void warp_long_row(const DevState& s, const Labels& L, int32_t* keys,
                                              typename Acc<WK>::T* vals, [[maybe_unused]] unsigned* peers_of,
                                              int log_slots, const TieRule& tr, int64_t st, int64_t en, int32_t v,
                                              const int32_t (&lab0)[K], const typename Acc<WK>::T (&w0)[K],
                                              uint32_t& key, uint32_t& tie) {
    using T = typename Acc<WK>::T;
    const unsigned lane = lane_id();
    const unsigned okm = __ballot_sync(kFull, lab0[0] != kEmptyKey);
    const int32_t lead = __shfl_sync(kFull, lab0[0], okm ? __ffs(okm) - 1 : 0);
    T lead_sum = (T)0;
    uint64_t mine[2] = {~0ull, ~0ull};
    auto add_chunk = [&](int32_t lab, T w, int c) {
        const bool ok = lab != kEmptyKey;
        const bool is_lead = ok && lab == lead;
        const unsigned lm = __ballot_sync(kFull, is_lead);
        if constexpr (WK == W_UNIT) lead_sum += (T)__popc(lm);
        else lead_sum += is_lead ? w : (T)0;                // per lane until the row is complete
        int slot = -1;
        if (ok && !is_lead) {
            slot = claim_slot(keys, log_slots, lab);
            if (slot < 0) atomicExch(&s.ctrl->error, 2);
            else if constexpr (WK != W_F32) atomicAdd(vals + slot, w);
        }
        if constexpr (WK == W_F32) {
            // the lanes of one slot add up in lane order and the
            // first of them adds their sum
            if (slot >= 0) atomicOr(peers_of + slot, 1u << lane);
            __syncwarp();
            const unsigned peers = slot >= 0 ? peers_of[slot] : 0u;
            const float sum = ordered_group_sum(peers, w);
            if (peers && lane == (unsigned)(__ffs(peers) - 1)) {
                peers_of[slot] = 0u;
                vals[slot] += sum;
            }
            __syncwarp();
        }
        if (slot >= 0) {
            const int sh = 16 * (c & 3);
            const uint64_t put = ~(0xffffull << sh) | ((uint64_t)slot << sh);
            if (c < 4) mine[0] &= put;
            else mine[1] &= put;
        }
    };
    int c = 0;
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (st + 32 * u < en) add_chunk(lab0[u], w0[u], c++);       // warp-uniform
    for (int64_t e0 = st + 32 * K; e0 < en; e0 += 32 * kWarpUnroll) {
        int32_t jj[kWarpUnroll], ll[kWarpUnroll];
        T wq[kWarpUnroll];
#pragma unroll
        for (int u = 0; u < kWarpUnroll; ++u) {
            const int64_t e = e0 + 32 * u + lane;
            jj[u] = e < en ? load_index_keep(s.idx, e) : v;
        }
#pragma unroll
        for (int u = 0; u < kWarpUnroll; ++u) {
            const bool ok = jj[u] != v;
            ll[u] = ok ? load_label<ASYNC>(L.C, jj[u]) : kEmptyKey;
            wq[u] = ok ? load_weight<WK>(s.w, e0 + 32 * u + lane) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < kWarpUnroll; ++u) {
            if (e0 + 32 * u >= en) break;      // warp-uniform
            add_chunk(ll[u], wq[u], c++);
        }
    }
    if constexpr (WK == W_U32 || WK == W_U8) lead_sum = __reduce_add_sync(kFull, lead_sum);
    if constexpr (WK == W_F32)
        for (int o = 16; o > 0; o >>= 1) lead_sum += __shfl_xor_sync(kFull, lead_sum, o);
    if (okm) offer_candidate<T>(tr, lead_sum, lead, key, tie);
    __syncwarp();
    for (int q = 0; q < c; ++q) {
        const unsigned slot = (unsigned)((q < 4 ? mine[0] : mine[1]) >> (16 * (q & 3))) & 0xffffu;
        if (slot != 0xffffu) offer_candidate<T>(tr, vals[slot], keys[slot], key, tie);
    }
    __syncwarp();
    for (int q = 0; q < c; ++q) {
        const unsigned slot = (unsigned)((q < 4 ? mine[0] : mine[1]) >> (16 * (q & 3))) & 0xffffu;
        if (slot != 0xffffu) {
            keys[slot] = kEmptyKey;
            vals[slot] = (T)0;
        }
    }
    __syncwarp();
}

}  // namespace lpa
