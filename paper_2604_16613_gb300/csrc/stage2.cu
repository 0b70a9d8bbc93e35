// stage2.cu -- probability aggregation (Sec. 3.2) and the adjoint.
//
// Stage 1 leaves records in a pool: a noise row, a word column that sees it and
// the X / Z planes of the row's qubits, an entry each (every entry handed out
// belongs to a record or is marked empty).
// Stage 2:
//   scatter    per record: a slot of its row by one atomic add, the column and
//              the planes into it (kRowSlots slots a row, then an overflow list)
//   group      one thread per mechanism: its mask words are XORs of the row's
//              planes, formed in registers; the key is the word count and the
//              sum of the words' hashes (equal masks give equal keys in any
//              order of the columns).  It claims or joins a slot
//              of an open-addressing table whose claims are verified on the
//              whole mask (word count and every (column, word) pair), so the
//              grouping is exact whatever the hash does; keep the smallest
//              member and add t_i = -log(1 - 2 q_i) to the class sum as an
//              exact 128-bit fixed-point integer: 1 - 2P = prod(1 - 2 q_i) =
//              exp(-sum t_i) (Eq. pmerge), and integer addition makes the sum
//              independent of the order in which the atomics land
//   compact    classes are numbered by their smallest member: a two-pass scan
//              whose input is read straight from the table (1 and the class's
//              detector count for the smallest member of a class, else 0)
//              lists the leaders in edge order with their detector offsets;
//              then one thread per hyperedge writes it: ascending detector
//              ids, observable word, P = -expm1(-T) / 2 and
//              w = log1p(-P) - log(P)
//   finalize   per-mechanism class ids; used table slots are cleared for the
//              next compile; the status goes to the host
//   backward   dP/dp_i = (1 - 2P) / 2 * dt_i/dp and dw/dP = -1 / (P (1 - P)),
//              summed per noise location in fixed point
// Every grid is fixed by the driver's bounds, so the whole sequence can be
// captured once and replayed.
#include <algorithm>

#include "common.cuh"

namespace gpdem {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;                          // elements per thread
constexpr uint32_t kScanBlock = kScanThreads * kScanPer;

__device__ __forceinline__ uint2 add2(uint2 a, uint2 b) { return make_uint2(a.x + b.x, a.y + b.y); }

// block-wide exclusive scan of two channels
__device__ __forceinline__ uint2 block_scan2(uint2 v, uint32_t *tmp, uint2 &total) {
    uint32_t tx, ty;
    const uint32_t ex = block_exclusive_scan<kScanThreads>(v.x, tmp, tx);
    const uint32_t ey = block_exclusive_scan<kScanThreads>(v.y, tmp, ty);
    total = make_uint2(tx, ty);
    return make_uint2(ex, ey);
}

// ---- rows' word columns ---------------------------------------------------------
// Each record's column and planes into its row's next slot (or overflow list),
// by the thread of its first entry.  Each thread takes kScatterILP entries per
// round, with every load and atomic of the round in flight before the first
// store (the kernel is bound by their latency).
constexpr int kScatterILP = 2;

__global__ void __launch_bounds__(512, 2) scatter_kernel(Buffers B) {
    if (B.status->code != 0u) return;
    const Params &P = *B.params;
    const uint32_t n = min(B.status->rec_count, P.rec_cap);
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i0 = blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kScatterILP * stride) {
        uint2 h[kScatterILP];
        ulonglong2 a[kScatterILP], b[kScatterILP];
        uint32_t k[kScatterILP];
#pragma unroll
        for (int u = 0; u < kScatterILP; u++) {
            const uint32_t i = i0 + u * stride;
            h[u] = make_uint2(kNone, 0u);
            if (i < n) {
                h[u] = B.rec_hdr[i];
                a[u] = B.rec_pl[i];
            }
        }
#pragma unroll
        for (int u = 0; u < kScatterILP; u++)
            if (h[u].x != kNone) {
                k[u] = atomicAdd(&B.row_cnt[h[u].x], 1u);
                b[u] = make_ulonglong2(0ull, 0ull);
                // (the lane beside loads this entry, too)
                if (h[u].y & kRecTwo) b[u] = B.rec_pl[i0 + u * stride + 1u];
            }
#pragma unroll
        for (int u = 0; u < kScatterILP; u++) {
            if (h[u].x == kNone) continue;
            h[u].y &= ~kRecTwo;
            if (k[u] < (uint32_t)kRowSlots) {
                const size_t x = (size_t)kRowSlots * h[u].x + k[u];
                B.row_col[x] = h[u].y;
                B.row_pl[2u * x] = a[u];
                B.row_pl[2u * x + 1u] = b[u];
            } else {
                const uint32_t j = atomicAdd(&B.status->rov_count, 1u);
                if (j < P.rov_cap) {
                    RowOverflow o;
                    o.pl[0] = a[u].x;
                    o.pl[1] = a[u].y;
                    o.pl[2] = b[u].x;
                    o.pl[3] = b[u].y;
                    o.col = h[u].y;
                    o.next = atomicExch(&B.row_ov[h[u].x], j);     // the list ends by its count
                    B.rov[j] = o;
                } else {
                    report(B.status, GP_ERR_CAPACITY, 11u, j, P.rov_cap);
                }
            }
        }
    }
}

// ---- a mechanism's mask words ------------------------------------------------
// Hash of one (column, word) pair; a mask's key adds these up (mod 2^64, low
// byte masked off for the word count), so equal masks give equal keys in any
// order of their columns.
__device__ __forceinline__ unsigned long long word_hash(uint32_t col, unsigned long long w) {
    return mix64(w ^ (0x9E3779B97F4A7C15ull * (col + 1ull)));
}

// XOR of the planes a component's Pauli names (code: comp_planes), p -> {X, Z}
// of the row's first qubit, {X, Z} of its second (read only when named: a
// one-qubit row has none)
__device__ __forceinline__ unsigned long long comp_word(uint32_t code, const ulonglong2 *p) {
    unsigned long long w = 0ull;
    if (code & 3u) {
        const ulonglong2 a = p[0];
        w = ((code & 1u) ? a.x : 0ull) ^ ((code & 2u) ? a.y : 0ull);
    }
    if (code & 12u) {
        const ulonglong2 b = p[1];
        w ^= ((code & 4u) ? b.x : 0ull) ^ ((code & 8u) ? b.y : 0ull);
    }
    return w;
}

// Row g's column count and first kRowSlots column ids.
struct RowHdr {
    uint32_t cnt, col[kRowSlots];
};
__device__ __forceinline__ RowHdr row_hdr(const Buffers &B, uint32_t g) {
    const uint4 *p = reinterpret_cast<const uint4 *>(B.row_col) + 2u * (size_t)g;
    static_assert(kRowSlots == 8, "two 16-byte loads");
    const uint32_t n = B.row_cnt[g];
    const uint4 a = p[0], b = p[1];
    return RowHdr{n, {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// f(column, word) for each non-zero mask word of a component (code) of row g
// with header h: the row's slots, then its overflow list.
template <class F>
__device__ __forceinline__ void for_words(const Buffers &B, uint32_t g, const RowHdr &h, uint32_t code, F f) {
    const ulonglong2 *pp = &B.row_pl[2u * (size_t)kRowSlots * g];
#pragma unroll
    for (int i = 0; i < kRowSlots; i++) {
        if ((uint32_t)i >= h.cnt) break;
        const unsigned long long w = comp_word(code, pp + 2 * i);
        if (w != 0ull) f(h.col[i], w);
    }
    if (h.cnt > (uint32_t)kRowSlots) {
        uint32_t j = B.row_ov[g];
        for (uint32_t i = kRowSlots; i < h.cnt; i++) {
            const RowOverflow &o = B.rov[j];
            const ulonglong2 p[2] = {make_ulonglong2(o.pl[0], o.pl[1]), make_ulonglong2(o.pl[2], o.pl[3])};
            const unsigned long long w = comp_word(code, p);
            if (w != 0ull) f(o.col, w);
            j = o.next;
        }
    }
}

// Words of a mechanism as the grouping holds them: N (column, word) slots,
// a zero word for an empty one.
template <int N>
struct Words {
    uint32_t col[N];
    unsigned long long w[N];
    uint32_t cnt, dets;
    unsigned long long key;

    __device__ __forceinline__ void finish() {
        cnt = 0;
        dets = 0;
        key = 0ull;
#pragma unroll
        for (int i = 0; i < N; i++)
            if (w[i] != 0ull) {
                cnt++;
                if (!(col[i] & kObsColFlag)) dets += (uint32_t)__popcll(w[i]);
                key += word_hash(col[i], w[i]) & ~0xFFull;
            }
        key |= cnt;
    }
    __device__ __forceinline__ bool has(uint32_t c, unsigned long long x) const {
        bool found = false;
#pragma unroll
        for (int i = 0; i < N; i++) found |= col[i] == c && w[i] == x;
        return found;
    }
    // exact comparison with the mask of the mechanism of an entry: as many
    // words, each at its column here (columns are distinct within a mask).
    // The claimant's words are formed from its row's planes again, which the
    // stage before this kernel wrote, so a claim publishes nothing.
    __device__ __forceinline__ bool same(const Buffers &B, unsigned long long e) const {
        const uint32_t g = (uint32_t)(e >> 4);
        uint32_t n = 0;
        bool ok = true;
        for_words(B, g, row_hdr(B, g), (uint32_t)e & 0xFu, [&](uint32_t c, unsigned long long x) {
            n++;
            ok = ok && has(c, x);
        });
        return ok && n == cnt;
    }
};

// Claim or join the class of mechanism m (hash h, the planes `code` of row g)
// in the open-addressing table; a slot with the same tag is joined when its
// claimant's mask is equal.  Mechanisms are numbered in row order, so a
// claimant of an earlier row already keeps m from being the smallest member,
// and most joins leave `min` alone.
// Returns the slot, or kNone when the table is full.
template <int N>
__device__ __forceinline__ uint32_t claim_or_join(const Buffers &B, const Words<N> &words, unsigned long long h,
                                                  uint32_t m, uint32_t g, uint32_t code, uint32_t first,
                                                  uint32_t cap_mask) {
    const unsigned long long mine = (h >> 36 << 36) | ((unsigned long long)g << 4) | code;
    uint32_t pos = first;
    for (uint32_t probe = 0; probe <= cap_mask; probe++) {
        unsigned long long e = __ldcg(&B.table[pos].entry);
        if (e == kEmpty) {
            e = atomicCAS(&B.table[pos].entry, kEmpty, mine);
            if (e == kEmpty) {
                B.table[pos].cls = words.dets;    // the claim records the class's detector count
                atomicMin(&B.table[pos].min, m);
                return pos;
            }
        }
        if ((e ^ mine) >> 36 == 0ull && words.same(B, e)) {
            if (g <= (uint32_t)(e >> 4)) atomicMin(&B.table[pos].min, m);
            return pos;
        }
        pos = (pos + 1u) & cap_mask;
    }
    report(B.status, GP_ERR_CAPACITY, 6u, m, cap_mask + 1u);
    return kNone;
}

// Where hash h starts probing for a mechanism of circuit b.  Classes never
// span circuits, so each circuit has its own stretch of the table, as large as
// its share of the mechanisms (1.5 to 3 slots a mechanism): the slots in use at
// a time lie together, and a small compile on a large driver uses a small part.
// per: table slots per mechanism, 16 fraction bits (slots_per_mech).
__device__ __forceinline__ unsigned long long slots_per_mech(const Params &P, uint32_t n_mech) {
    return min(((1ull << P.table_log2) << 16) / max(n_mech, 1u), 3ull << 16);
}
__device__ __forceinline__ uint32_t probe_start(const Buffers &B, unsigned long long per, uint32_t b,
                                                unsigned long long h) {
    const CircuitDev &C = B.circ[b];
    const uint32_t base = (uint32_t)((C.mech_base * per) >> 16), size = (uint32_t)((C.n_mech * per) >> 16);
    return base + __umulhi((uint32_t)h, size);
}

// What the grouping does with one mechanism once its words are known; returns
// its slot or kNone.
template <int N>
__device__ __forceinline__ uint32_t group_words(const Buffers &B, const Params &P, Words<N> &words, uint32_t m,
                                                uint32_t g, uint32_t kind, uint32_t code, uint32_t b,
                                                unsigned long long per) {
    words.finish();
    if (words.cnt == 0u) return kNone;
    if (words.cnt > P.mask_words) {
        report(B.status, GP_ERR_CAPACITY, 4u, m, words.cnt);
        return kNone;
    }
    const uint32_t loc = B.row_loc[g];
    const float p = P.noise[loc];
    if (!(p >= 0.0f && p <= channel_pmax(kind))) {
        report(B.status, GP_ERR_INVALID, 5u, loc, __float_as_uint(p));
        return kNone;
    }
    if (p == 0.0f) return kNone;
    float c, k;
    channel_ck(kind, c, k);
    float t = -log1pf(-c * p) / k;
    if (!(t < 1048576.0f)) t = 1048576.0f;     // q = 1/2 saturates P at 1/2
    // collisions cost probes, never correctness (claims are verified on
    // the whole mask)
    const unsigned long long h = weaken_hash(mix64(words.key ^ 0x243F6A8885A308D3ull), P.weak_hash);
    const uint32_t slot = claim_or_join<N>(B, words, h, m, g, code, probe_start(B, per, b, h),
                                           (1u << P.table_log2) - 1u);
    if (slot == kNone) return kNone;
    unsigned long long lo, hi;
    to_fixed(t, kProbShift, lo, hi);
    acc128_add(&B.table[slot].acc_lo, lo, hi);
    return slot;
}

// a mechanism of a row that more than kRowSlots word columns see
__device__ __noinline__ uint32_t group_many(const Buffers &B, uint32_t m, uint32_t g, uint32_t kind, uint32_t code,
                                            uint32_t b, unsigned long long per) {
    Words<kMaxMaskWords> words;
    for (int i = 0; i < kMaxMaskWords; i++) { words.col[i] = kNone; words.w[i] = 0ull; }
    uint32_t n = 0;
    for_words(B, g, row_hdr(B, g), code, [&](uint32_t c, unsigned long long w) {
        if (n < (uint32_t)kMaxMaskWords) { words.col[n] = c; words.w[n] = w; }
        n++;
    });
    if (n > (uint32_t)kMaxMaskWords) {
        report(B.status, GP_ERR_CAPACITY, 4u, m, n);
        return kNone;
    }
    return group_words<kMaxMaskWords>(B, *B.params, words, m, g, kind, code, b, per);
}

__global__ void __launch_bounds__(512, 2) group_kernel(Buffers B) {
    const Params &P = *B.params;
    if (B.status->code != 0u) return;
    const uint32_t N = B.status->n_mech;
    const unsigned long long per = slots_per_mech(P, N);
    for (uint32_t m = blockIdx.x * blockDim.x + threadIdx.x; m < N; m += gridDim.x * blockDim.x) {
        const unsigned long long info = B.mech_info[m];
        const uint32_t g = (uint32_t)info;
        const uint32_t kind = (uint32_t)(info >> 32) & 0xFFu;
        const uint32_t code = comp_planes(kind, (uint32_t)(info >> 40) & 0xFFu);
        const RowHdr h = row_hdr(B, g);
        uint32_t slot = kNone;
        if (h.cnt > (uint32_t)kRowSlots) {
            slot = group_many(B, m, g, kind, code, (uint32_t)(info >> 48), per);
        } else if (h.cnt != 0u) {
            Words<kRowSlots> words;
            const ulonglong2 *pp = &B.row_pl[2u * (size_t)kRowSlots * g];
#pragma unroll
            for (int i = 0; i < kRowSlots; i++) {
                words.col[i] = h.col[i];
                words.w[i] = 0ull;
                if ((uint32_t)i < h.cnt) words.w[i] = comp_word(code, pp + 2 * i);
            }
            slot = group_words<kRowSlots>(B, P, words, m, g, kind, code, (uint32_t)(info >> 48), per);
        }
        B.slot_of[m] = slot;
    }
}

// ---- compaction scan: classes numbered by their smallest member ------------
// Input of mechanism i: (1, the detector count its class's claim left in the
// slot) when i is the smallest member of its class, else (0, 0).
__device__ __forceinline__ uint2 leader_in(const Buffers &B, uint32_t i) {
    const uint32_t slot = B.slot_of[i];
    if (slot == kNone) return make_uint2(0u, 0u);
    const uint2 mc = *reinterpret_cast<const uint2 *>(&B.table[slot].min);
    return mc.x == i ? make_uint2(1u, mc.y) : make_uint2(0u, 0u);
}

__global__ void __launch_bounds__(kScanThreads) leader_reduce_kernel(Buffers B) {
    if (B.status->code != 0u) return;
    const uint32_t n = B.status->n_mech;
    const uint32_t nb = (n + kScanBlock - 1) / kScanBlock;
    __shared__ uint32_t tmp[kScanThreads / 32];
    for (uint32_t c = blockIdx.x; c < nb; c += gridDim.x) {
        const uint32_t b0 = c * kScanBlock;
        uint2 v[kScanPer];
#pragma unroll
        for (int k = 0; k < kScanPer; k++) {
            const uint32_t i = b0 + threadIdx.x * kScanPer + k;
            v[k] = i < n ? leader_in(B, i) : make_uint2(0u, 0u);
        }
        uint2 acc = make_uint2(0u, 0u);
#pragma unroll
        for (int k = 0; k < kScanPer; k++) acc = add2(acc, v[k]);
        // the inputs, once, for the second pass (coalesced 8-byte writes)
#pragma unroll
        for (int k = 0; k < kScanPer; k++) {
            const uint32_t i = b0 + threadIdx.x * kScanPer + k;
            if (i < n) B.scan_val[i] = v[k];
        }
        uint2 tot;
        block_scan2(acc, tmp, tot);
        if (threadIdx.x == 0) B.scan_bsum[c] = tot;
    }
}

// Each chunk adds up the sums of the chunks before it itself; every leader
// gets its edge index (its rank) and detector offset: edge_mech[e] = leader,
// det_off[e] = offset.  Block 0 writes the totals (edge count, detector
// entries, det_off[E]) and checks them against the bounds.
__global__ void __launch_bounds__(kScanThreads) leader_down_kernel(Buffers B) {
    if (B.status->code != 0u) return;
    const uint32_t n = B.status->n_mech;
    const uint32_t nb = (n + kScanBlock - 1) / kScanBlock;
    __shared__ uint32_t tmp[kScanThreads / 32];
    if (blockIdx.x == 0) {
        uint2 all = make_uint2(0, 0);
        for (uint32_t i = threadIdx.x; i < nb; i += kScanThreads) all = add2(all, B.scan_bsum[i]);
        uint2 tot;
        block_scan2(all, tmp, tot);
        if (threadIdx.x == 0) {
            if ((unsigned long long)tot.y > B.params->max_det_entries) {
                report(B.status, GP_ERR_CAPACITY, 7u, tot.y,
                       (uint32_t)(B.params->max_det_entries > 0xFFFFFFFFull ? 0xFFFFFFFFull
                                                                            : B.params->max_det_entries));
            } else {
                B.status->n_edges = tot.x;
                B.status->n_det_entries = tot.y;
                B.det_off[tot.x] = tot.y;
            }
        }
    }
    for (uint32_t c = blockIdx.x; c < nb; c += gridDim.x) {
        const uint32_t b0 = c * kScanBlock;
        uint2 before = make_uint2(0, 0);
        for (uint32_t i = threadIdx.x; i < c; i += kScanThreads) before = add2(before, B.scan_bsum[i]);
        uint2 prefix;
        block_scan2(before, tmp, prefix);
        uint2 v[kScanPer];
        uint2 acc = make_uint2(0, 0);
#pragma unroll
        for (int k = 0; k < kScanPer; k++) {
            const uint32_t i = b0 + threadIdx.x * kScanPer + k;
            v[k] = i < n ? B.scan_val[i] : make_uint2(0u, 0u);
            acc = add2(acc, v[k]);
        }
        uint2 tot;
        uint2 run = add2(block_scan2(acc, tmp, tot), prefix);
#pragma unroll
        for (int k = 0; k < kScanPer; k++) {
            if (v[k].x) {
                B.edge_mech[run.x] = b0 + threadIdx.x * kScanPer + k;
                B.det_off[run.x] = run.y;
            }
            run = add2(run, v[k]);
        }
    }
}

__global__ void compact_write_kernel(Buffers B) {
    if (B.status->code != 0u) return;
    const uint32_t E = B.status->n_edges;
    const uint32_t lane = threadIdx.x & 31u;
    // host output (when set): the same arrays, written into host memory too
    const Params &P = *B.params;
    uint32_t *const h_off = reinterpret_cast<uint32_t *>(P.h_det_off);
    uint32_t *const h_idx = reinterpret_cast<uint32_t *>(P.h_det_idx);
    unsigned long long *const h_obs = reinterpret_cast<unsigned long long *>(P.h_obs);
    float *const h_prob = reinterpret_cast<float *>(P.h_prob);
    float *const h_lo = reinterpret_cast<float *>(P.h_logodds);
    const uint64_t h_ecap = P.h_edges_cap, h_dcap = P.h_det_cap;
    if (h_off && E == 0u && blockIdx.x == 0 && threadIdx.x == 0) h_off[0] = 0u;
    for (uint32_t base = blockIdx.x * blockDim.x; base < E; base += gridDim.x * blockDim.x) {
        const uint32_t e = base + threadIdx.x;
        uint32_t b = 0xFFFFFFFFu;
        uint32_t d0 = 0u, d1 = 0u;          // this edge's detector ids [d0, d1)
        if (e < E) {
            const uint32_t m = B.edge_mech[e];
            uint32_t d = B.det_off[e];
            d0 = d;
            const uint32_t slot = B.slot_of[m];
            const unsigned long long info = B.mech_info[m];
            b = (uint32_t)(info >> 48);
            const uint32_t col_base = B.circ[b].col_base;
            uint32_t col[kMaxMaskWords];
            unsigned long long w[kMaxMaskWords];
            uint32_t cnt = 0;
            const uint32_t g = (uint32_t)info, kind = (uint32_t)(info >> 32) & 0xFFu;
            for_words(B, g, row_hdr(B, g), comp_planes(kind, (uint32_t)(info >> 40) & 0xFFu),
                      [&](uint32_t c, unsigned long long x) {
                          col[cnt] = c;
                          w[cnt++] = x;
                      });
            unsigned long long obs = 0ull;
            // words in ascending column order (selection), so the detector
            // ids come out ascending
            uint32_t prev = 0u;
            for (uint32_t k = 0; k < cnt; k++) {
                uint32_t cmin = 0xFFFFFFFFu, jmin = 0u;
                for (uint32_t j = 0; j < cnt; j++) {
                    const uint32_t c = col[j];
                    if ((k == 0u || c > prev) && c < cmin) { cmin = c; jmin = j; }
                }
                prev = cmin;
                unsigned long long x = w[jmin];
                if (cmin & kObsColFlag) { obs ^= x; continue; }
                const uint32_t base_id = (cmin - col_base) * 64u;
                while (x) {
                    const int bit = __ffsll((long long)x) - 1;
                    B.det_idx[d++] = base_id + (uint32_t)bit;
                    x &= x - 1ull;
                }
            }
            d1 = d;
            const TabSlot &ts = B.table[slot];
            const float T = fixed_to_float(ts.acc_lo, ts.acc_hi, kProbShift);
            const float Pc = -0.5f * expm1f(-T);
            const float lo = log1pf(-Pc) - logf(Pc);
            B.obs_mask[e] = obs;
            B.prob[e] = Pc;
            B.logodds[e] = lo;
            B.class_slot[e] = slot;
            B.edge_circ[e] = b;
            B.table[slot].cls = e;
            if (h_off && e < h_ecap) {
                h_off[e] = d0;
                h_obs[e] = obs;
                h_prob[e] = Pc;
                h_lo[e] = lo;
                if (e + 1u == E && E <= h_ecap) h_off[E] = d1;
            }
        }
        if (h_off) {
            // the warp's edges are consecutive, so their detector ids are one
            // range: copied to the host lane by lane (coalesced stores)
            __syncwarp();
            const uint32_t lo_w = __shfl_sync(0xFFFFFFFFu, d0, 0);
            const unsigned has = __ballot_sync(0xFFFFFFFFu, e < E);
            const uint32_t hi_w = has ? __shfl_sync(0xFFFFFFFFu, d1, 31 - __clz(has)) : lo_w;
            for (uint32_t i = lo_w + lane; i < hi_w && i < h_dcap; i += 32u) h_idx[i] = B.det_idx[i];
        }
        // edges per circuit: one atomic per circuit present in the warp
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, b);
        if (e < E && (uint32_t)(__ffs(peers) - 1) == lane) atomicAdd(&B.circ_edges[b], (uint32_t)__popc(peers));
    }
}

// per-mechanism class ids (four consecutive mechanisms per thread: one 16-byte
// load of their slots, one 16-byte store of their ids) and used table slots
// cleared (one edge per thread): disjoint fields, one pass
__global__ void finalize_kernel(Buffers B) {
    if (blockIdx.x == 0) {
        // nothing below reports or counts, so the status and the counts are
        // final: written to the host here, the compile needs no copy after its
        // last kernel
        const Params &P = *B.params;
        uint32_t *hs = reinterpret_cast<uint32_t *>(P.h_status), *he = reinterpret_cast<uint32_t *>(P.h_circ_edges);
        const uint32_t *st = reinterpret_cast<const uint32_t *>(B.status);
        for (uint32_t i = threadIdx.x; i < sizeof(Status) / 4u; i += blockDim.x) hs[i] = st[i];
        for (uint32_t i = threadIdx.x; i < P.n_circuits; i += blockDim.x) he[i] = B.circ_edges[i];
    }
    if (B.status->code != 0u) return;
    const uint32_t N = B.status->n_mech, E = B.status->n_edges;
    const uint32_t N4 = (N + 3u) / 4u;
    const uint32_t M = max(N4, E);
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += stride) {
        const uint32_t cs = i < E ? B.class_slot[i] : kNone;
        if (i < N4) {
            const bool full = 4u * i + 3u < N;
            uint32_t sl[4];
            if (full) {
                const uint4 v = *reinterpret_cast<const uint4 *>(&B.slot_of[4u * i]);
                sl[0] = v.x; sl[1] = v.y; sl[2] = v.z; sl[3] = v.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; u++) sl[u] = 4u * i + u < N ? B.slot_of[4u * i + u] : kNone;
            }
            int32_t cl[4];
#pragma unroll
            for (int u = 0; u < 4; u++) cl[u] = sl[u] == kNone ? -1 : (int32_t)B.table[sl[u]].cls;
            if (full) {
                *reinterpret_cast<int4 *>(&B.mech_class[4u * i]) = make_int4(cl[0], cl[1], cl[2], cl[3]);
            } else {
#pragma unroll
                for (int u = 0; u < 4; u++)
                    if (4u * i + u < N) B.mech_class[4u * i + u] = cl[u];
            }
        }
        // cls is left alone: other threads may still be reading it (a claim
        // overwrites it in the next compile)
        if (cs != kNone) {
            TabSlot &ts = B.table[cs];
            ts.entry = kEmpty;
            ts.min = kNone;
            *reinterpret_cast<uint4 *>(&ts.acc_lo) = make_uint4(0u, 0u, 0u, 0u);   // acc_lo, acc_hi
        }
    }
}

__global__ void backward_mech_kernel(Buffers B, const float *g_prob, const float *g_logodds, uint32_t N) {
    const float *noise = B.params->noise;
    for (uint32_t m = blockIdx.x * blockDim.x + threadIdx.x; m < N; m += gridDim.x * blockDim.x) {
        const int32_t e = B.mech_class[m];
        if (e < 0) continue;
        const unsigned long long info = B.mech_info[m];
        const uint32_t loc = B.row_loc[(uint32_t)info];
        const uint32_t kind = (uint32_t)(info >> 32) & 0xFFu;
        const float p = noise[loc];
        const float Pc = B.prob[e];
        const float one_m_2P = 1.0f - 2.0f * Pc;
        if (one_m_2P <= 0.0f) continue;            // saturated class: P = 1/2
        const float gp = g_prob ? g_prob[e] : 0.0f;
        const float gw = g_logodds ? g_logodds[e] : 0.0f;
        const float gbar = gp - gw / (Pc * (1.0f - Pc));
        float c, k;
        channel_ck(kind, c, k);
        const float dtdp = (c / k) / (1.0f - c * p);
        const float g = gbar * 0.5f * one_m_2P * dtdp;
        acc128_add_signed(&B.gacc[2 * (size_t)loc], g, kGradShift);
    }
}

__global__ void backward_loc_kernel(Buffers B, float *g_noise, uint32_t n_loc) {
    for (uint32_t l = blockIdx.x * blockDim.x + threadIdx.x; l < n_loc; l += gridDim.x * blockDim.x) {
        const unsigned long long lo = B.gacc[2 * (size_t)l], hi = B.gacc[2 * (size_t)l + 1];
        g_noise[l] = fixed_to_float_signed(lo, hi, kGradShift);
        B.gacc[2 * (size_t)l] = 0ull;
        B.gacc[2 * (size_t)l + 1] = 0ull;
    }
}

__global__ void init_table_kernel(TabSlot *t, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        t[i].entry = kEmpty;
        t[i].min = kNone;
        t[i].cls = 0;
        t[i].acc_lo = 0ull;
        t[i].acc_hi = 0ull;
    }
}

}  // namespace

static uint32_t scan_grid(uint32_t max_n, uint32_t n_sms) {
    const uint32_t chunks = (max_n + kScanBlock - 1) / kScanBlock;
    return std::max(1u, std::min(chunks, 8u * std::max(n_sms, 1u)));
}

void launch_group(const Buffers &b, uint32_t grid, uint32_t threads, uint32_t max_mech, cudaStream_t s,
                  uint32_t *launches) {
    (void)max_mech;
    scatter_kernel<<<grid, threads, 0, s>>>(b);
    group_kernel<<<grid, threads, 0, s>>>(b);
    *launches += 2;
}

void launch_compact(const Buffers &b, uint32_t grid, uint32_t threads, uint32_t max_mech, uint32_t n_sms,
                    cudaStream_t s, uint32_t *launches) {
    const uint32_t grid1 = scan_grid(max_mech, n_sms);
    leader_reduce_kernel<<<grid1, kScanThreads, 0, s>>>(b);
    leader_down_kernel<<<grid1, kScanThreads, 0, s>>>(b);
    compact_write_kernel<<<grid, threads, 0, s>>>(b);
    finalize_kernel<<<grid, threads, 0, s>>>(b);
    *launches += 4;
}

void launch_backward(const Buffers &b, const float *g_prob, const float *g_logodds, float *g_noise,
                     uint32_t n_mech, uint32_t n_loc, uint32_t grid, uint32_t threads, cudaStream_t s,
                     uint32_t *launches) {
    backward_mech_kernel<<<grid, threads, 0, s>>>(b, g_prob, g_logodds, n_mech);
    backward_loc_kernel<<<grid, threads, 0, s>>>(b, g_noise, n_loc);
    *launches += 2;
}

void launch_init_table(TabSlot *t, size_t n, cudaStream_t s) {
    init_table_kernel<<<1024, 256, 0, s>>>(t, n);
}

}  // namespace gpdem
