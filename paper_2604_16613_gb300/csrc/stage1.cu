// stage1.cu -- error-equivalence-class generation (Sec. 3.1).
//
// The straight-line program of Eq. slp is linear over GF(2), so every 64
// detectors (one "word column") can be propagated on their own.  A thread
// block takes word columns from a work queue and keeps, in shared memory, two
// 64-bit bit-planes per qubit of the column:
//   x[q] bit j = detector j flips under an X error on q at the current time
//   z[q] bit j = the same for a Z error.
// It walks the TICK layers backward from the latest measurement of the
// column's detectors (Eq. init-slp sets the bits there) and stops once every
// plane is zero and no earlier measurement of the column remains.
//
// A step at layer L reads the planes of one buffer and writes the other's:
//   emit   the noise rows touching an active qubit (non-zero planes) after the
//          gates of L and before the gates of L + 1 (the planes hold the state
//          between the two), one (qubit, row) pair per thread: a record with
//          the planes of the row's qubits.  A two-qubit row is listed under
//          both of its qubits and taken by the first one that is active.
//   undo   the gates of L, each thread its own qubits from their old planes
//          and their partners': H swaps the planes, S: x ^= z, CX(c,t):
//          x_c ^= x_t and z_t ^= z_c, CZ(a,b): x_a ^= z_b and x_b ^= z_a;
//          resets clear the planes after checking that the detectors commute
//          with them.  The qubits left with non-zero planes are listed for
//          the next step's emission.  On the layers that measure for the
//          column its bits are XORed in afterwards.
// The walk is a chain of such steps, so a step is made short: every qubit is
// read and written whether active or not (one select chain without branches,
// no dependent list lookups), its gate is in a register before the step
// begins, and one barrier ends the step.
//
// An observable's walk spans the whole circuit.  It is done twice: a pass that
// only undoes gates (no noise rows, no lists) leaves the planes of every
// kSegLayers-th step in memory, and each stretch of kSegLayers steps is a work
// item of its own, which any block walks and emits once its starting planes
// are there.
//
// What a step at L reads -- the gates of L as seen from each qubit, the
// after-gate list offsets of L, the before-gate list offsets of L+1 and the
// list entries between them -- is contiguous in the lowering's layer index.
// One further warp of the block (the service warp, outside the steps'
// barrier) stages it into shared memory by two 1-D bulk copies (TMA) issued
// several steps ahead into a ring of window buffers, each tracked by an
// mbarrier, and publishes the pass's checkpoints.  Windows too large for a
// buffer are read from global memory.
#include <algorithm>

#include "common.cuh"

namespace gpdem {

namespace {

constexpr int kMaxBufs = 8;         // window ring slots at most
constexpr uint32_t kFlagDone = 0x80000000u;   // checkpoint flag: no more follow
constexpr int kStepDone = -1000;    // progress: the walk is over

struct Smem {
    ulonglong2 *pl0, *pl1;          // per qubit: {X plane, Z plane}, two buffers
    uint2 *ent;                     // entries {layer, qubit | x-basis << 15 | column bit << 16}
    uint16_t *act0, *act1;          // active qubits of a step
    unsigned char *win;             // window buffers
};

__host__ __device__ inline uint32_t round8(uint32_t x) { return (x + 7u) & ~7u; }

// bytes of the fixed part of the layout (everything but the windows)
__host__ __device__ inline size_t smem_base_bytes(uint32_t maxq, bool listed) {
    const size_t q8 = round8(maxq);
    const size_t b = (listed ? 20 : 36) * q8 + sizeof(uint2) * (size_t)kMaxEntries;
    return (b + 127) & ~(size_t)127;
}

// bytes of the index part of a window buffer
__host__ __device__ inline uint32_t window_index_bytes(uint32_t maxq) {
    const uint32_t b = layer_geo(maxq).bytes;
    return (b + 127u) & ~127u;
}

__device__ __forceinline__ Smem carve(unsigned char *base, uint32_t maxq, bool listed) {
    const uint32_t q8 = round8(maxq);
    Smem s;
    s.pl0 = reinterpret_cast<ulonglong2 *>(base);
    s.pl1 = listed ? s.pl0 : s.pl0 + q8;
    s.ent = reinterpret_cast<uint2 *>(s.pl1 + q8);
    s.act0 = reinterpret_cast<uint16_t *>(s.ent + kMaxEntries);
    s.act1 = s.act0 + q8;
    s.win = base + smem_base_bytes(maxq, listed);
    return s;
}

// the noise rows of a walk step, published by the service warp with the window
struct RowWindow {
    const uint16_t *aoff;       // after-gate list offsets of L
    const uint16_t *boff;       // before-gate list offsets of L + 1
    const uint2 *lists;         // after-gate lists of L, then before-gate
                                // lists of L + 1
    uint32_t n_after;           // entries of the after-gate lists
};

struct Shared {
    unsigned long long mbar[kMaxBufs];
    RowWindow desc[kMaxBufs];
    uint32_t item, bail, nent, lmax;
    uint32_t tmo[2];        // a wait of a step (of a slot, in the gates-only pass) of
                            // this parity gave up (never cleared: the block leaves).
                            // Only walking threads write it, before the step's
                            // barrier, so every thread reads the same value after
                            // it, while a faster warp may already be in the next
                            // wait, which writes the other one
    uint32_t next_ent[2];   // 1 + latest layer with an entry still to come
    uint32_t n_act[3];      // active qubits: of this step, of the next, being cleared
    uint32_t flag;          // checkpoint flag read by the first thread
    uint32_t post_par;      // parity of the posts per ring slot when the item began
    int progress;           // last step whose barrier was passed, or kStepDone
};

__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t load_acquire(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_release(uint32_t *p, uint32_t v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// the walk's progress, from its first thread to the service warp: what was
// written before the step's barrier is visible to who reads it
__device__ __forceinline__ void set_progress(int *p, int v) {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int get_progress(int *p) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
    return v;
}
// barrier of the NT walking threads (the service warp stays out of it)
template <int NT>
__device__ __forceinline__ void step_sync() {
    asm volatile("barrier.cta.sync 1, %0;" ::"n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ bool step_sync_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(NT)
        : "memory");
    return r != 0u;
}

// The entries of one word column (Eq. init-slp): each measurement that a
// detector of the column (or an observable of an observable word) reads, as
// {layer, qubit | x-basis << 15 | column bit << 16}.  Every walking thread
// calls it, with nent and lmax (1 + the latest layer of an entry) zeroed, and
// meets a barrier before reading them.
template <int NT>
__device__ __forceinline__ void column_entries(const Buffers &B, const CircuitDev &C, uint32_t cidx, uint32_t local,
                                               bool is_obs, uint2 *ent, uint32_t *nent, uint32_t *lmax) {
    auto add = [&](uint32_t meas, uint32_t bit) {
        const uint2 lq = B.meas_lq[C.meas_base + meas];
        const uint32_t e = atomicAdd(nent, 1u);
        if (e >= (uint32_t)kMaxEntries) return;
        ent[e] = make_uint2(lq.x, (lq.y & 0x7FFFu) | (lq.y >> 31 << 15) | (bit << 16));
        atomicMax(lmax, lq.x + 1u);
    };
    if (!is_obs) {
        // several threads per detector: its records' lookups run side by side
        constexpr uint32_t G = NT >= 960 ? 8 : 4;
        static_assert(NT % G == 0, "whole groups");
        const uint32_t j0 = local * 64u, j1 = min(j0 + 64u, C.n_det);
        for (uint32_t j = j0 + threadIdx.x / G; j < j1; j += NT / G) {
            const uint32_t row = B.det_row[C.det_base + j];
            const uint4 op = C.ops[row];
            const uint32_t mb = B.aux[C.op_base + row];
            for (uint32_t i = threadIdx.x % G; i < op.z; i += G) add(mb - C.recs[op.y + i], j & 63u);
        }
    } else {
        // observable word k holds observables k * obs_per .. (bit = observable);
        // one warp per row, its records over the lanes (a logical reads many)
        const uint32_t o0 = (local - (C.n_cols - C.n_ocols)) * C.obs_per, o1 = o0 + C.obs_per;
        const uint32_t n_rows = B.obs_count[cidx];
        for (uint32_t i0 = threadIdx.x >> 5; i0 < n_rows; i0 += NT / 32u) {
            const uint32_t row = B.obs_rows[C.op_base + i0];
            const uint4 op = C.ops[row];
            if (op.w < o0 || op.w >= o1) continue;
            const uint32_t mb = B.aux[C.op_base + row];
            for (uint32_t i = threadIdx.x & 31u; i < op.z; i += 32u) add(mb - C.recs[op.y + i], op.w);
        }
    }
}

// A warp's share of the record pool.  A record is one word column's planes of
// a noise row: {X, Z} of its qubit in one pool entry, of its second qubit in the
// next (kRecTwo).  A row has few columns (1 to 4, at most 10 in the codes here),
// so the planes of a row are 5 to 6 times fewer records than the words of its up
// to 15 mechanisms, which the grouping forms from them in registers.  Entries
// go to chunks of the pool that a warp takes by one atomic, the next one asked
// for while half of the last is left, so a step never waits for global memory;
// every entry handed out belongs to a record or is marked empty.  Emission is
// bound by issue slots and registers: one 40-byte record a row would save 3 to
// 5 % of stage 1 (us: 16 adaptive branches 706 against 731, BB 4 rounds 104
// against 109, d = 25 135 against 135) for a pool of 170 instead of 102 bytes a
// mechanism; an entry for every non-zero plane costs more than it saves (872,
// BB 12 rounds 145 against 131).

// (out of line, for its registers)
__device__ __noinline__ void pool_full(Status *st, uint32_t at, uint32_t cap) {
    report(st, GP_ERR_CAPACITY, 8u, at, cap);
}

struct Chunk {
    uint32_t pos = 0, end = 0, next = 0;
    bool has_next = false;

    // warp-uniform: positions [a, b) marked empty
    __device__ __forceinline__ void fill(const Buffers &B, uint32_t a, uint32_t b, uint32_t lane) const {
        for (uint32_t i = a + lane; i < b; i += 32u) B.rec_hdr[i] = make_uint2(kNone, 0u);
    }
    __device__ __forceinline__ void prefetch(const Buffers &B, uint32_t lane) {
        if (!has_next && end - pos < kChunk / 2u) {
            if (lane == 0u) next = atomicAdd(&B.status->rec_count, kChunk);
            has_next = true;
        }
    }
    // the warp's records (a lane's row, word column and planes a, b; two: of a
    // two-qubit row) appended
    __device__ __forceinline__ void emit(const Buffers &B, uint32_t rec_cap, bool have, bool two, uint32_t row,
                                         uint32_t col, ulonglong2 a, ulonglong2 b, uint32_t lane) {
        const unsigned m = __ballot_sync(0xFFFFFFFFu, have), m2 = __ballot_sync(0xFFFFFFFFu, have && two);
        const unsigned lt = (1u << lane) - 1u;
        const uint32_t n = (uint32_t)(__popc(m) + __popc(m2)), room = end - pos;
        uint32_t at = pos + (uint32_t)(__popc(m & lt) + __popc(m2 & lt));
        if (n > room) {
            // the rest of this chunk, then the next one
            if (!has_next && lane == 0u) next = atomicAdd(&B.status->rec_count, kChunk);
            has_next = false;
            const uint32_t nb = __shfl_sync(0xFFFFFFFFu, next, 0);
            if (nb >= rec_cap || rec_cap - nb < kChunk) {
                // (the compile fails, and nothing reads the pool)
                if (lane == 0u) pool_full(B.status, nb, rec_cap);
                pos = end = 0;
                return;
            }
            // a record with one entry's room left goes to the next chunk whole
            const bool split = have && two && at + 1u == end;
            const uint32_t hole = __any_sync(0xFFFFFFFFu, split) ? 1u : 0u;
            if (split) B.rec_hdr[at] = make_uint2(kNone, 0u);
            if (at >= end || split) at = nb + (at - end + hole);
            pos = nb + (n - room + hole);
            end = nb + kChunk;
        } else {
            pos += n;
        }
        if (have) {
            B.rec_hdr[at] = make_uint2(row, two ? col | kRecTwo : col);
            B.rec_pl[at] = a;
            if (two) {
                B.rec_hdr[at + 1u] = make_uint2(kNone, 0u);
                B.rec_pl[at + 1u] = b;
            }
        }
    }
    // at the end: the unused rest of the chunk and the chunk asked for
    __device__ __forceinline__ void flush(const Buffers &B, uint32_t rec_cap, uint32_t lane) {
        fill(B, pos, end, lane);
        pos = end;
        if (has_next) {
            const uint32_t nb = __shfl_sync(0xFFFFFFFFu, next, 0);
            if (nb < rec_cap) fill(B, nb, min(nb + kChunk, rec_cap), lane);
            has_next = false;
        }
    }
};

// The noise rows of the active qubits act[0 .. n_act) of a step, four threads a
// qubit, by warps starting at thread w0 of every `stride` (whole warps call
// it).  planes(q): a qubit's planes in this step; anti(): a detector
// anticommutes with the initial state (checked when `after` is false, step -1).
template <class Planes, class Anti>
__device__ __forceinline__ void emit_rows(const Buffers &B, uint32_t rec_cap, Chunk &chunk, const uint16_t *aoff,
                                          const uint16_t *boff, const uint2 *lists, uint32_t n_after, bool after,
                                          const uint16_t *act, uint32_t n_act, uint32_t w0, uint32_t stride,
                                          uint32_t lane, uint32_t col_tag, Planes planes, Anti anti) {
    const ulonglong2 none = make_ulonglong2(0ull, 0ull);
    for (uint32_t w = w0; w < 4u * n_act; w += stride) {
        const uint32_t a = w + lane;
        ulonglong2 p = none;
        uint32_t q = 0;
        if (a < 4u * n_act) {
            q = act[a >> 2];
            p = planes(q);
        }
        uint32_t a0 = 0, na = 0, b0 = 0, n = 0;
        if ((p.x | p.y) != 0ull) {
            if (after) {
                a0 = aoff[q];
                na = aoff[q + 1u] - a0;
            } else if (p.y != 0ull) {
                anti();
            }
            b0 = boff[q];
            n = na + boff[q + 1u] - b0;
        }
        for (uint32_t i = a & 3u; __any_sync(0xFFFFFFFFu, i < n); i += 4u) {
            ulonglong2 pa = none, pb = none;
            uint32_t row = 0;
            bool two = false;
            if (i < n) {
                const uint2 r = lists[i < na ? a0 + i : n_after + b0 + (i - na)];
                const uint32_t kind = row_kind(r);
                row = r.y;
                two = kind == K_DEP2;
                if (two) {
                    const uint32_t ra = row_a(r);
                    const ulonglong2 o = planes(ra == q ? row_b(r) : ra);
                    if (ra == q) {
                        pa = p;
                        pb = o;
                    } else if ((o.x | o.y) == 0ull) {     // else taken by its first qubit
                        pb = p;
                    }
                } else {
                    // a plane that no component of the kind reads is dropped
                    pa = make_ulonglong2(kind == K_ZERR ? 0ull : p.x, kind == K_XERR ? 0ull : p.y);
                }
            }
            chunk.emit(B, rec_cap, (pa.x | pa.y | pb.x | pb.y) != 0ull, two, row, col_tag, pa, pb, lane);
        }
    }
}

// planes of a qubit before its gate (a gate view), from its planes p and its
// partner's r after it; bad collects planes a measurement or reset anticommutes with
__device__ __forceinline__ ulonglong2 undo_gate(uint32_t g, ulonglong2 p, ulonglong2 r, unsigned long long &bad) {
    auto bit = [&](uint32_t f) { return (unsigned long long)(long long)((int)(g << __clz(f)) >> 31); };
    const unsigned long long d = (p.x ^ p.y) & bit(kGateSwap);
    bad |= (p.y & bit(kGateCheckZ)) | (p.x & bit(kGateCheckX));
    const unsigned long long keep = ~bit(kGateClear);
    return make_ulonglong2((p.x ^ d ^ (r.x & bit(kGateXX)) ^ (r.y & bit(kGateXZ))) & keep,
                           (p.y ^ d ^ (r.y & bit(kGateZZ))) & keep);
}

// Kinds of work items: a detector column's walk, the gates-only pass of an
// observable column, one stretch of an observable column's walk.
enum ItemMode : uint32_t { kWalk = 0, kPass = 1, kStretch = 2 };

// NT walking threads and the service warp, for circuits of up to NT * QPT
// qubits.  LISTED: for circuits too wide to read every qubit in a step (and
// for two plane buffers) only the active qubits' gates are undone, one thread
// an active qubit; an inactive partner has one active neighbour, whose thread
// gives it its planes.  The new planes wait in registers for a second barrier,
// after which they are stored and the next list is made of them.
constexpr int min_blocks(int nt) { return nt > 480 ? 1 : (nt > 256 ? 2 : 3); }

template <int NT, int QPT, bool LISTED>
__global__ void __launch_bounds__(NT + 32, min_blocks(NT)) stage1_kernel(Buffers B, uint32_t maxq, Stage1Shape shape) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Smem s = carve(smem_raw, maxq, LISTED);
    __shared__ Shared sh;
    const Params &P = *B.params;
    const uint32_t rec_cap = P.rec_cap;
    const uint32_t wlim = P.wait_limit;            // polls of a bounded wait
    const bool stall = P.stall_windows != 0u;      // test knob: no window is staged
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const bool service = tid >= (uint32_t)NT;
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t n_items = P.n_items, n_all = n_items + B.status->n_segs;
    const uint32_t windex = window_index_bytes(maxq);

    if (tid == 0) {
        for (int i = 0; i < kMaxBufs; i++) mbar_init(&sh.mbar[i], 1);
        fence_mbar_init();
        sh.tmo[0] = sh.tmo[1] = 0;
    }
    bool timed_out = false;
    uint32_t post_par = 0, posted_any = 0;   // service: parity of the posts per ring slot; slots ever posted to
    Chunk chunk;

    for (;;) {
        if (tid == 0) {
            sh.item = atomicAdd(&B.status->queue_head, 1u);
            sh.bail = (*(volatile uint32_t *)&B.status->code) != 0u;
            sh.nent = 0;
            sh.lmax = 0;
            sh.next_ent[0] = sh.next_ent[1] = 0;
            sh.n_act[0] = sh.n_act[1] = sh.n_act[2] = 0;
            sh.progress = 1 << 30;
        }
        if (service && lane == 0u) sh.post_par = post_par;
        __syncthreads();
        const uint32_t item = sh.item;
        if (item >= n_all || sh.bail || timed_out) break;
        // ---- which column, and which part of its walk --------------------
        uint32_t b, gcol, mode, seg = 0;
        if (item < n_items) {
            gcol = B.items[item];
            b = B.col_circ[gcol];
            mode = item < P.n_ocols_total ? kPass : kWalk;
        } else {
            const uint32_t si = item - n_items;
            uint32_t lo = 0, hi = P.n_circuits;       // circuits are laid out in stretch order
            while (hi - lo > 1u) {
                const uint32_t mid = (lo + hi) >> 1;
                if (B.circ[mid].seg_base <= si) lo = mid; else hi = mid;
            }
            b = lo;
            const CircuitDev &C = B.circ[b];
            const uint32_t r = si - C.seg_base;       // the latest stretch of every column first
            seg = r / C.n_ocols;
            gcol = C.col_base + C.n_cols - C.n_ocols + r % C.n_ocols;
            mode = kStretch;
        }
        const CircuitDev &C = B.circ[b];
        const uint32_t n_seg = C.n_seg;
        if (mode == kPass && n_seg <= 1u) { __syncthreads(); continue; }   // its one stretch starts from nothing
        const uint32_t local = gcol - C.col_base;
        const bool is_obs = mode != kWalk;
        const uint32_t col_tag = gcol | (is_obs ? kObsColFlag : 0u);
        const uint32_t nq = C.n_qubits, op_base = C.op_base;
        const uint32_t ocol = is_obs ? local - (C.n_cols - C.n_ocols) : 0u;
        uint32_t *const flag = B.seg_flag + C.ocol_base + ocol;
        ulonglong2 *const ckpt = B.ckpt + (size_t)(C.seg_base + ocol * n_seg) * maxq;
        if (!service) {
            for (uint32_t q = tid; q < nq; q += NT) s.pl0[q] = s.pl1[q] = make_ulonglong2(0ull, 0ull);
            column_entries<NT>(B, C, b, local, is_obs, s.ent, &sh.nent, &sh.lmax);
        }
        __syncthreads();
        const uint32_t n_ent = sh.nent;
        if (n_ent == 0u || n_ent > (uint32_t)kMaxEntries) {
            // nothing to walk, or over capacity
            if (n_ent && tid == 0) report(B.status, GP_ERR_CAPACITY, 5u, gcol, n_ent);
            __syncthreads();
            continue;
        }
        const int lmax = (int)sh.lmax - 1;
        // steps L .. L_lo of the walk (lmax .. -1 in all)
        int L = lmax, L_lo = -1;
        bool any = false;                 // some plane is non-zero
        if (mode == kStretch) {
            L = lmax - (int)(seg * kSegLayers);
            if (n_seg > 1u) L_lo = max(L - (int)kSegLayers + 1, -1);
            if (L < -1) { __syncthreads(); continue; }
            if (seg > 0u) {
                // the planes the gates-only pass left before step L
                if (tid == 0) {
                    uint32_t f = 0, it = 0;
                    for (; it < wlim; it++) {
                        f = load_acquire(flag);
                        if ((f & kFlagDone) || (f & ~kFlagDone) > seg) break;
                        if (*(volatile uint32_t *)&B.status->code != 0u) { f = kFlagDone; break; }
                        __nanosleep(64);
                    }
                    sh.flag = it == wlim ? kNone : f;
                }
                __syncthreads();
                if (sh.flag == kNone) {
                    if (tid == 0) report(B.status, GP_ERR_TIMEOUT, 1u, gcol, (uint32_t)L);
                    timed_out = true;
                    __syncthreads();
                    continue;
                }
                if ((sh.flag & ~kFlagDone) <= seg) { __syncthreads(); continue; }   // the walk ended above
                any = true;
            }
        } else if (mode == kPass) {
            L_lo = lmax - (int)(((uint32_t)lmax + 1u) / kSegLayers * kSegLayers);   // the last stretch's first step
        }

        // ---- layer index geometry of this circuit --------------------------
        const LayerGeo geo = layer_geo(nq);
        const unsigned char *qbase = B.qidx + (size_t)C.qidx_off * 16u;
        const bool gates_only = mode == kPass;
        // ring of window slots, in posting order from slot 0.  The gates-only
        // pass stages only the gates, gbatch layers to a slot.
        const uint32_t wbytes = gates_only ? shape.gbatch * shape.gbytes : shape.wbytes;
        const bool staged = (gates_only ? shape.ngbuf : shape.nbuf) >= 2u;
        const uint32_t nring = staged ? (gates_only ? shape.ngbuf : shape.nbuf) : 2u;
        const int w_lo = gates_only ? L_lo + 1 : L_lo;     // lowest window the walk can need

        if (service) {
            // ---- service warp (one lane): windows L, L - 1, ... into the ring,
            // each once the step that used its slot is over; the pass's
            // checkpoints once the step that stored them is over
            if (lane == 0u) {
                const uint2 *lbase = B.lists + 2ull * op_base;
                const uint4 *seg_g = B.layer_seg + C.layer_base;
                uint32_t slot = 0, n_ck = 1;
                int w = L;                                // next window to post
                int next_ck = L - (int)kSegLayers;        // next checkpoint's step
                uint4 s1 = make_uint4(0u, 0u, 0u, 0u);
                if (!gates_only && w >= w_lo) s1 = seg_g[w + 1];
                uint32_t idle = 0;
                for (;;) {
                    const int p = get_progress(&sh.progress);
                    if (gates_only && p <= next_ck && p != kStepDone) {
                        // the planes before step next_ck were stored during
                        // that step, whose barrier orders them before this
                        __threadfence();
                        store_release(flag, ++n_ck);
                        next_ck -= (int)kSegLayers;
                        continue;
                    }
                    if (p == kStepDone) break;
                    // steps a slot serves
                    const int per = gates_only ? (int)shape.gbatch : 1;
                    if (w < w_lo || stall || (L - w >= (int)nring * per && p > w + ((int)nring - 1) * per + 1)) {
                        // giving up: no further window is posted, and the
                        // step that needs the next one gives up in its own
                        // wait, before its barrier (a flag written from here
                        // would reach the walking warps at different steps,
                        // and their barrier waits for all of them)
                        if (++idle >= wlim && !stall && w >= w_lo) break;
                        __nanosleep(32);
                        continue;
                    }
                    idle = 0;
                    unsigned char *dst = s.win + (size_t)slot * wbytes;
                    if (gates_only) {
                        const int n = min(per, w - w_lo + 1);
                        if (staged) {
                            mbar_expect_tx(&sh.mbar[slot], (uint32_t)n * 4u * geo.nq4);
                            for (int i = 0; i < n; i++)
                                bulk_load(dst + (uint32_t)i * shape.gbytes, qbase + (size_t)(w - i) * geo.bytes + 2u * geo.qb,
                                          4u * geo.nq4, &sh.mbar[slot]);
                        } else {
                            mbar_arrive(&sh.mbar[slot]);
                        }
                    } else {
                        const uint4 s0 = w >= 0 ? seg_g[w] : make_uint4(0u, 0u, 0u, 0u);
                        const uint32_t n_after = s0.y;
                        const uint32_t list_start = 2u * s1.x - n_after;
                        const uint32_t list_n = n_after + s1.z;
                        s1 = s0;
                        // the index part and the lists, each staged when it fits
                        const unsigned char *qsrc = w >= 0 ? qbase + (size_t)w * geo.bytes + 2u * geo.qb : qbase;
                        const uint32_t qbytes = w >= 0 ? 4u * geo.nq4 + 4u * geo.qb : 2u * geo.qb;
                        const uint32_t delta = list_start & 1u;
                        const bool lists_in = staged && list_n + 1u <= shape.list_cap;
                        const uint32_t lbytes = lists_in && list_n ? ((list_n + delta) * 8u + 15u) & ~15u : 0u;
                        const unsigned char *qp = staged ? dst : qsrc;
                        RowWindow &d = sh.desc[slot];
                        d.n_after = n_after;
                        d.lists = lists_in ? reinterpret_cast<const uint2 *>(dst + windex) + delta : lbase + list_start;
                        d.aoff = w >= 0 ? reinterpret_cast<const uint16_t *>(qp + 4u * geo.nq4) : nullptr;
                        d.boff = w >= 0 ? d.aoff + geo.qb : reinterpret_cast<const uint16_t *>(qp);
                        if (staged) {
                            mbar_expect_tx(&sh.mbar[slot], qbytes + lbytes);
                            bulk_load(dst, qsrc, qbytes, &sh.mbar[slot]);
                            if (lbytes) bulk_load(dst + windex, lbase + list_start - delta, lbytes, &sh.mbar[slot]);
                        } else {
                            mbar_arrive(&sh.mbar[slot]);
                        }
                    }
                    post_par ^= 1u << slot;
                    posted_any |= 1u << slot;
                    slot = slot + 1u == nring ? 0u : slot + 1u;
                    w -= per;
                }
                // windows published ahead of the walk's end land before their
                // slots are reused (the walk waited for the others)
                for (uint32_t i = 0; i < nring && !stall; i++)
                    if ((posted_any >> i) & 1u) mbar_wait_bounded(&sh.mbar[i], ((post_par >> i) & 1u) ^ 1u);
            }
        } else {
            // ---- walking threads
            uint32_t phase = sh.post_par;         // parity of the next post per slot
            uint32_t slot = 0;
            bool landed = true;
            // waits for the window of the step (parity of the step: l)
            auto wait = [&](uint32_t sl, int l) {
                if (!mbar_try_wait(&sh.mbar[sl], (phase >> sl) & 1u)) {
                    landed = mbar_wait_bounded(&sh.mbar[sl], (phase >> sl) & 1u, wlim);
                    if (!landed) sh.tmo[l & 1] = 1u;
                }
                phase ^= 1u << sl;
            };
            // the gates of layer l for this thread's qubits
            uint32_t g[QPT];
            const uint32_t *gp = nullptr;
            auto load_gates = [&](uint32_t sl, uint32_t at, int l) {
                gp = reinterpret_cast<const uint32_t *>(
                    staged ? s.win + sl * wbytes + at * shape.gbytes : qbase + (size_t)l * geo.bytes + 2u * geo.qb);
                if (LISTED) return;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const uint32_t q = tid + i * NT;
                    g[i] = q < nq && landed && l >= 0 ? gp[q] : 0u;
                }
            };
            uint32_t cur = 0;                     // plane buffer of this step
            auto planes = [&](uint32_t c) { return c ? s.pl1 : s.pl0; };
            auto list = [&](uint32_t c) { return c ? s.act1 : s.act0; };
            // this thread's qubits in mask m (bit i: qubit i) appended to a list
            auto append = [&](uint16_t *dst, uint32_t *n, uint32_t m) {
                uint32_t mine[QPT], tot = 0;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const unsigned v = __ballot_sync(0xFFFFFFFFu, (m >> i) & 1u);
                    mine[i] = tot + (uint32_t)__popc(v & lt_mask);
                    tot += (uint32_t)__popc(v);
                }
                if (tot == 0u) return;
                uint32_t at = 0;
                if (lane == 0u) at = atomicAdd(n, tot);
                at = __shfl_sync(0xFFFFFFFFu, at, 0);
#pragma unroll
                for (int i = 0; i < QPT; i++)
                    if ((m >> i) & 1u) dst[at + mine[i]] = (uint16_t)(tid + i * NT);
            };
            uint32_t k3 = 0;                      // n_act counter of this step
            // own qubits that are non-zero, one step ago (what the buffer to be
            // written holds) and now
            uint32_t old = 0, now = 0;
            ulonglong2 p[QPT];                    // own qubits' planes
#pragma unroll
            for (int i = 0; i < QPT; i++) p[i] = make_ulonglong2(0ull, 0ull);
            if (any) {
                const ulonglong2 *const c = ckpt + (size_t)seg * maxq;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const uint32_t q = tid + i * NT;
                    if (q < nq) {
                        p[i] = __ldcg(&c[q]);
                        s.pl0[q] = p[i];
                        if ((p[i].x | p[i].y) != 0ull) now |= 1u << i;
                    }
                }
                append(list(0), &sh.n_act[0], now);
            }
            // 1 + the latest layer <= L holding an entry
            for (uint32_t i = tid; i < n_ent; i += NT)
                if ((int)s.ent[i].x <= L) atomicMax(&sh.next_ent[0], s.ent[i].x + 1u);
            uint32_t np = 0;                      // next_ent slot in use
            step_sync<NT>();                      // planes, lists and next_ent in place
            uint32_t ne = sh.next_ent[0];         // 1 + the latest layer with an entry <= L
            if (w_lo <= L) {
                wait(slot, L);
                load_gates(slot, 0u, L);
            }
            // qubits a (when add_a) and c (when add_c) appended to a list, by whole warps
            auto append2 = [&](uint16_t *dst, uint32_t *n, bool add_a, uint32_t a, bool add_c, uint32_t c) {
                const unsigned ma = __ballot_sync(0xFFFFFFFFu, add_a), mc = __ballot_sync(0xFFFFFFFFu, add_c);
                if ((ma | mc) == 0u) return;
                uint32_t at = 0;
                if (lane == 0u) at = atomicAdd(n, (uint32_t)(__popc(ma) + __popc(mc)));
                at = __shfl_sync(0xFFFFFFFFu, at, 0);
                if (add_a) dst[at + __popc(ma & lt_mask)] = (uint16_t)a;
                if (add_c) dst[at + __popc(ma) + __popc(mc & lt_mask)] = (uint16_t)c;
            };
            // LISTED: the gates of L undone on the n_act listed qubits; unless
            // the column measures at L, the next list is made as well
            auto undo_listed = [&](uint32_t n_act, uint32_t *n, bool words) {
                ulonglong2 r[QPT];
                uint32_t qp[QPT];                 // qubit | partner << 16, kNone: none
                unsigned long long bad = 0ull;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const uint32_t a = tid + i * NT;
                    qp[i] = kNone;
                    p[i] = r[i] = make_ulonglong2(0ull, 0ull);
                    if (a < n_act && landed) {
                        const uint32_t q = list(cur)[a], gq = gp[q], pay = gq & kGatePartner;
                        const ulonglong2 o = s.pl0[q], f = s.pl0[pay];
                        qp[i] = q | (pay << 16);
                        p[i] = undo_gate(gq, o, f, bad);
                        if ((f.x | f.y) == 0ull)
                            r[i] = make_ulonglong2((gq & kGateZZ ? o.x : 0ull) ^ (gq & kGateXZ ? o.y : 0ull),
                                                   gq & kGateXX ? o.y : 0ull);
                    }
                }
                if (bad != 0ull) report(B.status, GP_ERR_NONDETERMINISTIC, b, (uint32_t)L, gcol);
                step_sync<NT>();                  // every plane read before one is written
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    if (tid - lane + i * NT >= n_act) break;
                    const bool add = (r[i].x | r[i].y) != 0ull;
                    const uint32_t q = qp[i] & 0xFFFFu, pay = qp[i] >> 16;
                    if (qp[i] != kNone) s.pl0[q] = p[i];
                    if (add) s.pl0[pay] = r[i];
                    if (!words) append2(list(cur ^ 1u), n, (p[i].x | p[i].y) != 0ull, q, add, pay);
                }
            };
            // the gates of L undone on this thread's qubits, from the planes of
            // buffer cur into the other's (skipped where both stay zero)
            auto undo = [&]() {
                const ulonglong2 *const src = planes(cur);
                ulonglong2 *const dst = planes(cur ^ 1u);
                uint32_t m = 0;
                unsigned long long bad = 0ull;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const uint32_t q = tid + i * NT;
                    if (q >= nq) continue;
                    const ulonglong2 r = src[g[i] & kGatePartner];
                    if ((p[i].x | p[i].y | r.x | r.y) != 0ull) {
                        p[i] = undo_gate(g[i], p[i], r, bad);
                        if ((p[i].x | p[i].y) != 0ull) m |= 1u << i;
                        dst[q] = p[i];
                    } else if ((old >> i) & 1u) {
                        dst[q] = r;
                    }
                }
                if (bad != 0ull) report(B.status, GP_ERR_NONDETERMINISTIC, b, (uint32_t)L, gcol);
                old = now;
                now = m;
            };
            // the column's measurements at L: their bits into the new planes
            // (between two barriers), and the next layer that has any
            auto measure = [&]() {
                step_sync<NT>();
                unsigned long long *const dst = reinterpret_cast<unsigned long long *>(planes(cur ^ 1u));
                for (uint32_t i = tid; i < n_ent; i += NT) {
                    const uint2 e = s.ent[i];
                    if ((int)e.x == L)
                        atomicXor(&dst[2u * (e.y & 0x7FFFu) + ((e.y >> 15) & 1u)], 1ull << (e.y >> 16));
                    else if ((int)e.x < L)
                        atomicMax(&sh.next_ent[np ^ 1u], e.x + 1u);
                }
                step_sync<NT>();
                if (tid == 0) sh.next_ent[np] = 0;
                np ^= 1u;
                ne = sh.next_ent[np];
                const ulonglong2 *const pl = planes(cur ^ 1u);
                now = 0;
#pragma unroll
                for (int i = 0; i < QPT; i++) {
                    const uint32_t q = tid + i * NT;
                    if (q >= nq) continue;
                    p[i] = pl[q];
                    if ((p[i].x | p[i].y) != 0ull) now |= 1u << i;
                }
            };
            // after a step's last barrier
            auto advance = [&]() {
                if (tid == 0) set_progress(&sh.progress, L);
                slot = slot + 1u == nring ? 0u : slot + 1u;
                cur ^= 1u;
                L--;
            };

            // ---- backward wave over the layers -----------------------------
            if (gates_only) {
                uint32_t to_ck = kSegLayers, n_ck = 1, in_slot = 0;
                int batch = 0;                // parity of the slot waited for
                for (; L > L_lo; to_ck--) {
                    if (to_ck == 0u) {
                        // the planes before step L (the service warp publishes them)
                        to_ck = kSegLayers;
                        ulonglong2 *const c = ckpt + (size_t)n_ck++ * maxq;
#pragma unroll
                        for (int i = 0; i < QPT; i++)
                            if (tid + i * NT < nq) __stcg(&c[tid + i * NT], LISTED ? s.pl0[tid + i * NT] : p[i]);
                    }
                    const bool words = ne == (uint32_t)L + 1u;
                    const uint32_t k3n = k3 == 2u ? 0u : k3 + 1u;
                    if (LISTED) {
                        if (tid == 0) sh.n_act[k3n == 2u ? 0u : k3n + 1u] = 0;
                        undo_listed(sh.n_act[k3], &sh.n_act[k3n], words);
                    } else {
                        undo();
                    }
                    if (words) {
                        measure();
                        if (LISTED) append(list(cur ^ 1u), &sh.n_act[k3n], now);
                    }
                    if (LISTED) k3 = k3n;
                    if (++in_slot < shape.gbatch && L - 1 > L_lo) {
                        load_gates(slot, in_slot, L - 1);
                        step_sync<NT>();
                        cur ^= 1u;
                        L--;
                        continue;
                    }
                    // the last step of a slot: the next one's wait, and the ends
                    in_slot = 0;
                    slot = slot + 1u == nring ? 0u : slot + 1u;
                    batch ^= 1;
                    if (L - 1 >= w_lo) {
                        wait(slot, batch);
                        load_gates(slot, 0u, L - 1);
                    }
                    any = step_sync_or<NT>(LISTED || now != 0u || words);
                    if (LISTED) any = sh.n_act[k3] != 0u;
                    timed_out = sh.tmo[batch] != 0u;
                    if (tid == 0) set_progress(&sh.progress, L);
                    cur ^= 1u;
                    L--;
                    if (timed_out || (!any && ne == 0u)) break;
                }
                const bool last = !timed_out && L == L_lo && L < lmax && (any || ne != 0u);
                if (last) {
                    ulonglong2 *const c = ckpt + (size_t)n_ck++ * maxq;
#pragma unroll
                    for (int i = 0; i < QPT; i++)
                        if (tid + i * NT < nq) __stcg(&c[tid + i * NT], LISTED ? s.pl0[tid + i * NT] : p[i]);
                }
                step_sync<NT>();
                if (tid == 0) {
                    set_progress(&sh.progress, kStepDone);
                    __threadfence();
                    sh.flag = n_ck | kFlagDone;
                }
            } else {
                for (;;) {
                    // emission: one (active qubit, row) pair per thread, four
                    // threads per qubit
                    const uint32_t n_act = sh.n_act[k3];
                    const uint32_t k3n = k3 == 2u ? 0u : k3 + 1u;
                    if (tid == 0) sh.n_act[k3n == 2u ? 0u : k3n + 1u] = 0;
                    if (n_act != 0u && __all_sync(0xFFFFFFFFu, landed)) {
                        const RowWindow v = sh.desc[slot];
                        const ulonglong2 *const pl = planes(cur);
                        const uint16_t *const al = list(cur);
                        emit_rows(B, rec_cap, chunk, v.aoff, v.boff, v.lists, v.n_after, L >= 0, al, n_act,
                                  tid - lane, (uint32_t)NT, lane, col_tag, [&](uint32_t q) { return pl[q]; },
                                  [&]() { report(B.status, GP_ERR_NONDETERMINISTIC, b, 0xFFFFFFFFu, gcol); });
                        chunk.prefetch(B, lane);
                    }
                    if (L == L_lo) break;
                    const bool words = ne == (uint32_t)(L + 1);
                    if (LISTED) undo_listed(n_act, &sh.n_act[k3n], words);
                    else undo();
                    if (words) measure();
                    if (!LISTED || words) append(list(cur ^ 1u), &sh.n_act[k3n], now);
                    {
                        const uint32_t nx = slot + 1u == nring ? 0u : slot + 1u;
                        wait(nx, L);
                        load_gates(nx, 0u, L - 1);
                    }
                    step_sync<NT>();
                    timed_out = sh.tmo[L & 1] != 0u;
                    any = sh.n_act[k3n] != 0u;
                    k3 = k3n;
                    advance();
                    if (timed_out || (!any && (ne == 0u || (int)ne - 1 < L_lo))) break;
                }
                if (tid == 0) set_progress(&sh.progress, kStepDone);
            }
        }
        __syncthreads();
        timed_out = (sh.tmo[0] | sh.tmo[1]) != 0u;
        if (gates_only && tid == 0) store_release(flag, timed_out ? kFlagDone : sh.flag);
        if (timed_out) {
            if (tid == 0) report(B.status, GP_ERR_TIMEOUT, 1u, gcol, (uint32_t)L);
            break;
        }
    }
    if (!service) chunk.flush(B, rec_cap, lane);
    // after a wait gave up, copies may still be in flight: the last one posted
    // to each slot lands before the block exits (full limit)
    if (service && lane == 0u) {
        for (uint32_t i = 0; i < (uint32_t)kMaxBufs; i++)
            if ((posted_any >> i) & 1u) mbar_wait_bounded(&sh.mbar[i], ((post_par >> i) & 1u) ^ 1u);
    }
}

// ---------------------------------------------------------------------------
// Circuits of many qubits (and the smallest ones).  With many, most qubits are
// inactive in a column (a detector column of the distance-25 surface code has
// about 190 of 1,249 active, its observable 25 to 45), and reading every qubit
// in every step, as the walk above does, costs more than keeping candidate
// lists.
// ---------------------------------------------------------------------------
constexpr int kSplitSegCache = 256; // layer segments cached for the producer
constexpr int kSplitBufs = 4;       // window ring slots at most
constexpr uint32_t kSplitMinLayers = 64;   // observable walks this long are split in two (twice: three)
constexpr uint32_t kRankSortMax = 256;     // column entries sorted in one rank pass (else bitonic)
constexpr unsigned char kAdded = 1, kActive = 2;

// what one walk step reads (shared or global memory), published by the
// producer with the window
struct SplitWindow {
    const uint32_t *gate;       // gate of each qubit in L (step L >= 0)
    const uint16_t *aoff;       // after-gate list offsets of L
    const uint16_t *boff;       // before-gate list offsets of L + 1
    const uint2 *lists;         // after-gate lists of L, then before-gate
                                // lists of L + 1
    uint32_t n_after;           // entries of the after-gate lists
};

// The (measurement, word) entries of one word column (Eq. init-slp): each
// measurement a detector of the column (or an observable of an observable
// word) reads, with the column bit it sets, sorted by measurement, each run merged into its first
// entry, and each entry's layer and qubit.  Every thread of the block calls
// it, with nent_sh and lmax_sh zeroed.  Returns the entry count, or 0 when
// the column has nothing to walk (no entries, every word cancelled, or over
// capacity: reported); then lmax_sh - 1 is the latest layer holding a
// non-zero word and ent_l[0] the earliest layer of an entry.
template <int NT>
__device__ uint32_t sorted_entries(const Buffers &B, const CircuitDev &C, uint32_t cidx, uint32_t local, bool is_obs,
                                   uint32_t gcol, uint32_t *ent_m, unsigned long long *ent_w, uint32_t *ent_l,
                                   uint32_t *ent_q, uint32_t &nent_sh, uint32_t &lmax_sh) {
    // (measurement, word) entries of this column (Eq. init-slp)
    if (!is_obs) {
        const uint32_t j0 = local * 64u, j1 = min(j0 + 64u, C.n_det);
        for (uint32_t j = j0 + threadIdx.x; j < j1; j += NT) {
            const uint32_t row = B.det_row[C.det_base + j];
            const uint4 op = C.ops[row];
            const uint32_t mb = B.aux[C.op_base + row];
            for (uint32_t i = 0; i < op.z; i++) {
                const uint32_t e = atomicAdd(&nent_sh, 1u);
                if (e < (uint32_t)kMaxEntries) {
                    ent_m[e] = mb - C.recs[op.y + i];
                    ent_w[e] = 1ull << (j & 63u);
                }
            }
        }
    } else {
        // observable word k holds observables k * obs_per .. (bit = observable)
        const uint32_t o0 = (local - (C.n_cols - C.n_ocols)) * C.obs_per, o1 = o0 + C.obs_per;
        // one warp per row, its records over the lanes (a logical reads
        // many records)
        const uint32_t n_rows = B.obs_count[cidx];
        const uint32_t lane = threadIdx.x & 31u;
        for (uint32_t i0 = threadIdx.x >> 5; i0 < n_rows; i0 += NT / 32u) {
            const uint32_t row = B.obs_rows[C.op_base + i0];
            const uint4 op = C.ops[row];
            if (op.w < o0 || op.w >= o1) continue;
            const uint32_t mb = B.aux[C.op_base + row];
            for (uint32_t i = lane; i < op.z; i += 32u) {
                const uint32_t e = atomicAdd(&nent_sh, 1u);
                if (e < (uint32_t)kMaxEntries) {
                    ent_m[e] = mb - C.recs[op.y + i];
                    ent_w[e] = 1ull << op.w;
                }
            }
        }
    }
    __syncthreads();
    const uint32_t n_ent = nent_sh;
    if (n_ent > (uint32_t)kMaxEntries) {
        if (threadIdx.x == 0) report(B.status, GP_ERR_CAPACITY, 5u, gcol, n_ent);
        return 0u;
    }
    if (n_ent == 0u) return 0u;
    if (n_ent <= kRankSortMax) {
        // few entries: each one's place is the number of entries before it
        // in (measurement, position) order -- one pass instead of the
        // bitonic network's barriers.  The sorted copies go to the layer and
        // qubit arrays (free until the merge below), then back.
        unsigned long long *sw = reinterpret_cast<unsigned long long *>(ent_l);     // n_ent words
        uint32_t *sm = ent_q + kMaxEntries / 2u;                                   // n_ent measurements
        static_assert(2 * kRankSortMax <= kMaxEntries / 2, "rank-sort scratch inside ent_l / ent_q");
        for (uint32_t i = threadIdx.x; i < n_ent; i += NT) {
            const uint32_t m = ent_m[i];
            uint32_t r = 0;
            for (uint32_t j = 0; j < n_ent; j++) {
                const uint32_t mj = ent_m[j];
                r += (mj < m || (mj == m && j < i)) ? 1u : 0u;
            }
            sm[r] = m;
            sw[r] = ent_w[i];
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n_ent; i += NT) {
            ent_m[i] = sm[i];
            ent_w[i] = sw[i];
        }
        __syncthreads();
    } else {
    // bitonic sort of the entries by measurement index
    uint32_t npow = 1;
    while (npow < n_ent) npow <<= 1;
    for (uint32_t i = n_ent + threadIdx.x; i < npow; i += NT) { ent_m[i] = 0xFFFFFFFFu; ent_w[i] = 0ull; }
    __syncthreads();
    for (uint32_t k2 = 2; k2 <= npow; k2 <<= 1) {
        for (uint32_t j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
            for (uint32_t i = threadIdx.x; i < npow; i += NT) {
                const uint32_t ixj = i ^ j2;
                if (ixj > i) {
                    const bool asc = (i & k2) == 0u;
                    const uint32_t mi = ent_m[i], mj = ent_m[ixj];
                    if ((mi > mj) == asc) {
                        ent_m[i] = mj; ent_m[ixj] = mi;
                        const unsigned long long wi = ent_w[i];
                        ent_w[i] = ent_w[ixj]; ent_w[ixj] = wi;
                    }
                }
            }
            __syncthreads();
        }
    }
    }
    // merge the entries of one measurement: the first of a run holds the
    // XOR of the run, the rest hold zero (the layer array holds the merged
    // words meanwhile)
    unsigned long long *merged = reinterpret_cast<unsigned long long *>(ent_l);
    static_assert(kMaxEntries % 2 == 0, "ent_l and ent_q hold one 64-bit word per entry");
    for (uint32_t i = threadIdx.x; i < n_ent; i += NT) {
        unsigned long long w = 0ull;
        if (i == 0u || ent_m[i] != ent_m[i - 1u]) {
            for (uint32_t j = i; j < n_ent && ent_m[j] == ent_m[i]; j++) w ^= ent_w[j];
        }
        merged[i] = w;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_ent; i += NT) {
        const unsigned long long w = merged[i];
        ent_w[i] = w;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_ent; i += NT) {
        const uint2 lq = B.meas_lq[C.meas_base + ent_m[i]];
        ent_l[i] = lq.x;
        ent_q[i] = lq.y;
        if (ent_w[i] != 0ull) atomicMax(&lmax_sh, lq.x + 1u);
    }
    __syncthreads();
    if (lmax_sh == 0u) return 0u;   // every word cancelled
    return n_ent;
}

// ---------------------------------------------------------------------------
// Role-split walk.  The walk of a column is a chain over its layers; the
// noise rows of a layer only read the planes of that layer.  So one warp (the
// walker) advances the planes layer by layer with warp-level syncs only, and
// publishes for each step a snapshot of its active qubits' planes; the other
// warps (emitters) evaluate the noise rows of a step from that snapshot while
// the walker is already on the next one; the last warp stages the layer
// windows.  From 512 threads a second walker warp (four from 1024) waits on a
// named barrier and joins only the steps of more than 64 candidates, which
// warp 0 hands to it: the long chain of small steps (an observable's walk)
// keeps its single-warp latency, and the wide steps of detector columns are
// undone in parallel.  The snapshot tables are double-buffered by step parity and
// tagged with the step that wrote an entry (a qubit whose tag differs is not
// active in that step), so they are never cleared.  mbarriers order the
// roles: window full (producer -> walker), window free (walker, emitters ->
// producer), table full (walker -> emitters: it also carries the window,
// which the walker saw land before publishing), table free (emitters ->
// walker); every wait is bounded.
// ---------------------------------------------------------------------------
struct SplitSmem {
    ulonglong2 *pl;                 // walker: per qubit {X plane, Z plane}
    ulonglong2 *tab0, *tab1;        // snapshot planes per step parity
    uint4 *segc;                    // producer: layer segments
    unsigned long long *ent_w;      // entry words
    uint32_t *tag0, *tag1;          // step that wrote a snapshot entry
    uint32_t *ent_m, *ent_l, *ent_q;
    uint16_t *act0, *act1;          // active qubits of a step
    uint16_t *add;                  // qubits the walker adds to the next step's candidates
    unsigned char *bits;            // walker: kActive / kAdded / 0 per qubit
    unsigned char *win;             // window buffers
};

// Warps of a block: the first warps walk (two from 512 threads, four from
// 1024), the last warp stages windows, the rest emit.
__host__ __device__ constexpr uint32_t split_walkers(uint32_t nt) { return nt >= 1024u ? 4u : (nt >= 512u ? 2u : 1u); }
__host__ __device__ constexpr uint32_t split_emitters(uint32_t nt) { return nt / 32u - 1u - split_walkers(nt); }

__host__ __device__ inline size_t split_base_bytes(uint32_t maxq) {
    const size_t q8 = round8(maxq);
    size_t b = 16 * q8 * 3                          // pl, tab[2]
               + 16 * (size_t)kSplitSegCache             // segc
               + 8 * (size_t)kMaxEntries            // ent_w
               + 4 * q8 * 2                         // tag[2]
               + 12 * (size_t)kMaxEntries           // ent_m, ent_l, ent_q
               + 2 * q8 * 3                         // act[2], add
               + q8;                                // bits
    return (b + 127) & ~(size_t)127;
}

__device__ __forceinline__ SplitSmem split_carve(unsigned char *base, uint32_t maxq) {
    const uint32_t q8 = round8(maxq);
    SplitSmem s;
    s.pl = reinterpret_cast<ulonglong2 *>(base);
    s.tab0 = s.pl + q8;
    s.tab1 = s.tab0 + q8;
    s.segc = reinterpret_cast<uint4 *>(s.tab1 + q8);
    s.ent_w = reinterpret_cast<unsigned long long *>(s.segc + kSplitSegCache);
    s.tag0 = reinterpret_cast<uint32_t *>(s.ent_w + kMaxEntries);
    s.tag1 = s.tag0 + q8;
    s.ent_m = s.tag1 + q8;
    s.ent_l = s.ent_m + kMaxEntries;
    s.ent_q = s.ent_l + kMaxEntries;
    s.act0 = reinterpret_cast<uint16_t *>(s.ent_q + kMaxEntries);
    s.act1 = s.act0 + q8;
    s.add = s.act1 + q8;
    s.bits = reinterpret_cast<unsigned char *>(s.add + q8);
    s.win = base + split_base_bytes(maxq);
    return s;
}
// the parity-b copies (selects, not an indexed array: no stack frame)
__device__ __forceinline__ ulonglong2 *tab_of(const SplitSmem &s, uint32_t b) { return b ? s.tab1 : s.tab0; }
__device__ __forceinline__ uint32_t *tag_of(const SplitSmem &s, uint32_t b) { return b ? s.tag1 : s.tag0; }
__device__ __forceinline__ uint16_t *act_of(const SplitSmem &s, uint32_t b) { return b ? s.act1 : s.act0; }

// what the walker publishes with a step's snapshot
struct StepDesc {
    int layer;          // L (-1: the before-gate noise of layer 0)
    uint32_t n_act;     // active qubits (act list of the step's parity)
    uint32_t slot;      // window slot of L
    uint32_t end;       // 1: no step; the column is done
};

// a large step of the walk, as warp 0 hands it to the helper walker warps
struct WalkStep {
    int L;
    uint32_t n_prev, n_cand, slot;
    uint16_t *ab;
    const uint16_t *prev;
    uint32_t b, snap, stamp, cmd;     // cmd 0: the walk is over
};

struct SplitShared {
    unsigned long long win_full[kSplitBufs], win_free[kSplitBufs];
    unsigned long long tab_full[2], tab_free[2];
    SplitWindow desc[kSplitBufs];
    StepDesc step[2];
    uint32_t item, bail, nent, lmax;
    uint32_t tmo;           // a wait gave up (every role leaves)
    uint32_t walk_done;     // the walker left the column (the producer stops)
    int stop_layer;         // last layer the walker stepped through
    int posted_lo;          // lowest window the producer posted
    WalkStep wstep;         // warp 0 -> helper walker warps: the large step
    uint32_t wcnt[2];       // large step: {active, added}
};

template <int NT>
__global__ void __launch_bounds__(NT, 1) stage1_split_kernel(Buffers B, uint32_t maxq, Stage1Shape shape) {
    const uint32_t nbuf = shape.nbuf, list_cap = shape.list_cap, wbytes = shape.wbytes;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const SplitSmem s = split_carve(smem_raw, maxq);
    __shared__ SplitShared sh;
    constexpr uint32_t NW = NT / 32;
    constexpr uint32_t WW = split_walkers(NT);      // walker warps
    constexpr uint32_t NE = split_emitters(NT);     // emitter warps
    static_assert(NE >= 1, "walkers, emitters and producer");
    const Params &P = *B.params;
    const uint32_t rec_cap = P.rec_cap;
    const uint32_t wlim = P.wait_limit;            // polls of a bounded wait
    const bool stall = P.stall_windows != 0u;      // test knob: no window is staged
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    const bool walker = warp < WW, producer = warp == NW - 1u;
    const uint32_t ew = warp - WW;                  // emitter index
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t windex = window_index_bytes(maxq);
    const uint32_t nring = nbuf >= 2u ? nbuf : 2u;
    volatile uint32_t *const tmo_v = &sh.tmo;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kSplitBufs; i++) {
            mbar_init(&sh.win_full[i], 1);
            mbar_init(&sh.win_free[i], NE + 1u);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&sh.tab_full[i], 1);
            mbar_init(&sh.tab_free[i], NE);
        }
        fence_mbar_init();
        sh.tmo = 0;
    }
    for (uint32_t q = threadIdx.x; q < round8(maxq); q += NT) s.tag0[q] = s.tag1[q] = kNone;
    __syncthreads();

    // per-thread barrier phases (bit i: slot or buffer i)
    uint32_t full_par = 0;                  // walker: window full
    uint32_t free_par = 0, free_pend = 0;   // producer: window free; slots awaiting a release
    uint32_t post_par = 0, posted_any = 0;  // producer: parity of the posts per slot
    uint32_t tfull_par = 0;                 // emitters: table full
    uint32_t tfree_par = 0, tfree_pend = 0; // walker: table free; buffers awaiting a release
    uint32_t st = 0;                        // steps taken by this block (snapshot tags)
    Chunk chunk;
    uint32_t seg_lo = 0xFFFFFFFFu;

    // bounded wait; gives up early once another role has given up
    auto wait_bar = [&](unsigned long long *bar, uint32_t parity) -> bool {
        for (uint32_t it = 0; it < wlim; it++) {
            if (mbar_try_wait(bar, parity)) return true;
            if ((it & 31u) == 31u && *tmo_v) return false;
        }
        *tmo_v = 1u;
        return false;
    };
    // the same, by every lane of a warp with one outcome for all (the loops
    // around it use warp-wide votes)
    auto wait_warp = [&](unsigned long long *bar, uint32_t parity) -> bool {
        if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;     // usually done already
        return __all_sync(0xFFFFFFFFu, wait_bar(bar, parity));
    };
    for (;;) {
        if (threadIdx.x == 0) {
            sh.item = atomicAdd(&B.status->queue_head, 1u);
            sh.bail = (*(volatile uint32_t *)&B.status->code) != 0u;
            sh.nent = 0;
            sh.lmax = 0;
            sh.walk_done = 0;
            sh.stop_layer = 0;
            sh.posted_lo = 0;
            sh.wcnt[0] = sh.wcnt[1] = 0;
        }
        __syncthreads();
        const uint32_t item = sh.item;
        if (item >= P.n_items || sh.bail || sh.tmo) break;
        const uint32_t item_word = B.items[item];
        const uint32_t seg = item_word >> kSegShift;      // segment of a split walk
        const uint32_t gcol = item_word & kColMask;
        const uint32_t cidx = B.col_circ[gcol];
        const CircuitDev &C = B.circ[cidx];
        const uint32_t local = gcol - C.col_base;
        const bool is_obs = local >= C.n_cols - C.n_ocols;
        const uint32_t col_tag = gcol | (is_obs ? kObsColFlag : 0u);
        const uint32_t nq = C.n_qubits;
        const uint32_t op_base = C.op_base;
        seg_lo = 0xFFFFFFFFu;
        for (uint32_t q = threadIdx.x; q < nq; q += NT) {
            s.pl[q] = make_ulonglong2(0ull, 0ull);
            s.bits[q] = 0;
        }
        const uint32_t n_ent = sorted_entries<NT>(B, C, cidx, local, is_obs, gcol, s.ent_m, s.ent_w, s.ent_l,
                                                  s.ent_q, sh.nent, sh.lmax);
        if (n_ent == 0u) { __syncthreads(); continue; }
        const uint32_t lmax = sh.lmax - 1u;
        const uint32_t lmin = s.ent_l[0];
        // a long observable walk is shared by up to three blocks (one work
        // item each): segment k emits the steps emit_hi .. emit_lo and
        // fast-forwards through the steps above emit_hi first (gates undone,
        // nothing emitted or published).  A fast-forward step costs about
        // 0.73 of an emitting one, so segments of equal time emit, from the
        // top: 79 % / 21 % of the walk (two segments), 74.5 % / 20 % / 5.5 %
        // (three).
        const uint32_t n_seg = !is_obs ? 1u
                                       : min(P.obs_segments,
                                             lmax >= 2u * kSplitMinLayers ? 3u : (lmax >= kSplitMinLayers ? 2u : 1u));
        if (seg >= n_seg) { __syncthreads(); continue; }
        int b1 = -1, b2 = -1;                             // segment boundaries
        if (n_seg == 2u) b1 = max(1, (int)(3u * lmax / 14u));
        if (n_seg == 3u) {
            b1 = max(2, (int)(51u * lmax / 200u));
            b2 = min(b1 - 1, max(1, (int)(11u * lmax / 200u)));
        }
        const int emit_hi = seg == 0u ? (int)lmax : (seg == 1u ? b1 - 1 : b2 - 1);
        const int emit_lo = seg + 1u == n_seg ? -1 : (seg == 0u ? b1 : b2);
        const LayerGeo geo = layer_geo(nq);
        const unsigned char *qbase = B.qidx + (size_t)C.qidx_off * 16u;
        const uint2 *lbase = B.lists + 2ull * C.op_base;
        const uint4 *seg_g = B.layer_seg + C.layer_base;
        auto slot_of = [&](int L) -> uint32_t { return (uint32_t)(L + 1) % nring; };

        // ---- walker warps.  Warp 0 walks; a step of more than 64 candidates
        // is split over all walker warps (the helpers wait on a named barrier
        // in between): the activity pass over the candidates, a barrier, the
        // gates undone over the active list, a barrier.  The owner rule
        // leaves every plane a single writer, so the warps need no other
        // synchronisation; list positions come from shared counters.
        auto wsync = [&]() {
            if (WW == 1u) __syncwarp();
            else asm volatile("bar.sync 1, %0;" ::"n"(WW * 32u) : "memory");
        };
        // a position for n entries of this warp's ballot (one shared atomic)
        auto take = [&](uint32_t *ctr, uint32_t n) -> uint32_t {
            uint32_t o = 0;
            if (lane == 0u && n) o = atomicAdd(ctr, n);
            return __shfl_sync(0xFFFFFFFFu, o, 0);
        };
        auto large_activity = [&](uint32_t wid, int Lc, uint32_t np, uint32_t nc, const uint16_t *prv, uint16_t *abl,
                                  ulonglong2 *tbl, uint32_t *tgl, bool snp, uint32_t stamp) {
            for (uint32_t base = 64u * wid; base < nc; base += 64u * WW) {
                const uint32_t i0 = base + lane, i1 = base + lane + 32u;
                uint32_t q0 = 0, q1 = 0;
                if (i0 < nc) q0 = i0 < np ? prv[i0] : s.add[i0 - np];
                if (i1 < nc) q1 = i1 < np ? prv[i1] : s.add[i1 - np];
                const ulonglong2 p0 = s.pl[q0], p1 = s.pl[q1];
                const bool a0 = i0 < nc && (p0.x | p0.y) != 0ull;
                const bool a1 = i1 < nc && (p1.x | p1.y) != 0ull;
                if (i0 < nc) s.bits[q0] = a0 ? kActive : (unsigned char)0;
                if (i1 < nc) s.bits[q1] = a1 ? kActive : (unsigned char)0;
                if (a0 && snp) { tbl[q0] = p0; tgl[q0] = stamp; }
                if (a1 && snp) { tbl[q1] = p1; tgl[q1] = stamp; }
                if (Lc < 0 && ((a0 && p0.y != 0ull) || (a1 && p1.y != 0ull)))
                    report(B.status, GP_ERR_NONDETERMINISTIC, cidx, 0xFFFFFFFFu, gcol);
                const unsigned m0 = __ballot_sync(0xFFFFFFFFu, a0), m1 = __ballot_sync(0xFFFFFFFFu, a1);
                const uint32_t o = take(&sh.wcnt[0], (uint32_t)(__popc(m0) + __popc(m1)));
                if (a0) abl[o + __popc(m0 & lt_mask)] = (uint16_t)q0;
                if (a1) abl[o + __popc(m0) + __popc(m1 & lt_mask)] = (uint16_t)q1;
            }
        };
        // the gates of L undone for one candidate: the owner of a two-qubit
        // gate (its active qubit, or its control / first qubit when both are
        // active) updates both planes; returns the partner it touched
        auto undo = [&](uint32_t q, ulonglong2 P, uint32_t g, bool act, int Lc) -> uint32_t {
            if (!act) return kNone;
            const uint32_t pay = g & kGatePartner;
            if (pay != q) {
                const bool cxc = g & kGateXX, cxt = g & kGateZZ, cz = g & kGateXZ;
                const bool pact = s.bits[pay] == kActive;
                // both active: the control's or the lower qubit's thread undoes it
                if (pact && (cxt || (cz && q > pay))) return kNone;
                const ulonglong2 Q = s.pl[pay];
                // CX(c,t): x_c ^= x_t, z_t ^= z_c; CZ(a,b): x_a ^= z_b, x_b ^= z_a
                const unsigned long long ox = P.x ^ (cxc ? Q.x : 0ull) ^ (cz ? Q.y : 0ull);
                const unsigned long long oz = P.y ^ (cxt ? Q.y : 0ull);
                const unsigned long long px = Q.x ^ (cxt ? P.x : 0ull) ^ (cz ? P.y : 0ull);
                const unsigned long long pz = Q.y ^ (cxc ? P.y : 0ull);
                s.pl[q] = make_ulonglong2(ox, oz);
                s.pl[pay] = make_ulonglong2(px, pz);
                return pay;
            }
            if (g == q) return kNone;                   // no gate
            unsigned long long bad = 0ull;
            const ulonglong2 t = undo_gate(g, P, P, bad);
            if (bad != 0ull) report(B.status, GP_ERR_NONDETERMINISTIC, cidx, (uint32_t)Lc, gcol);
            s.pl[q] = t;
            return kNone;
        };
        auto large_undo = [&](uint32_t wid, int Lc, uint32_t na, const uint16_t *abl, const SplitWindow &vw) {
            for (uint32_t base = 32u * wid; base < na; base += 32u * WW) {
                const uint32_t i = base + lane;
                const uint32_t q = i < na ? abl[i] : 0u;
                const ulonglong2 P = s.pl[q];
                const uint32_t partner = undo(q, P, i < na ? vw.gate[q] : q, i < na, Lc);
                const bool add = partner != kNone && s.bits[partner] == 0;
                if (add) s.bits[partner] = kAdded;
                const unsigned m = __ballot_sync(0xFFFFFFFFu, add);
                const uint32_t o = take(&sh.wcnt[1], (uint32_t)__popc(m));
                if (add) s.add[o + __popc(m & lt_mask)] = (uint16_t)partner;
            }
        };
        if (walker && warp != 0u) {
            // ---- helper walker warps: large steps of warp 0's walk
            for (;;) {
                wsync();
                const WalkStep ws = sh.wstep;
                if (ws.cmd == 0u) break;
                const SplitWindow vw = sh.desc[ws.slot];
                large_activity(warp, ws.L, ws.n_prev, ws.n_cand, ws.prev, ws.ab, tab_of(s, ws.b), tag_of(s, ws.b),
                               ws.snap != 0u, ws.stamp);
                wsync();
                if (ws.L >= 0) large_undo(warp, ws.L, sh.wcnt[0], ws.ab, vw);
                wsync();
            }
        } else if (walker && warp == 0u) {
            // ---- walker: candidates of a step = the active qubits of the
            // last step, then the qubits the last step added
            uint32_t n_prev = 0, n_add = 0, cur = n_ent;
            int L = (int)lmax;
            bool ok = true;
            uint32_t slot = slot_of(L);
            // fast-forward steps (L > emit_hi) keep their active lists in the
            // two act buffers alternately, arranged so that the last one lands
            // where the first emitting step reads its predecessor's
            uint32_t ff_buf = 0u;
            if (emit_hi < (int)lmax) {
                const uint32_t n_ff = lmax - (uint32_t)emit_hi;
                ff_buf = ((st & 1u) ^ 1u) ^ ((n_ff - 1u) & 1u);
            }
            for (;;) {
                const bool ff = L > emit_hi;
                const bool snap = !ff;            // a snapshot is published for the emitters
                const uint32_t b = st & 1u;
                if (!wait_warp(&sh.win_full[slot], (full_par >> slot) & 1u)) { ok = false; break; }
                full_par ^= 1u << slot;
                const SplitWindow v = sh.desc[slot];
                if (snap) {
                    if ((tfree_pend >> b) & 1u) {
                        if (!wait_warp(&sh.tab_free[b], (tfree_par >> b) & 1u)) { ok = false; break; }
                        tfree_par ^= 1u << b;
                    }
                    tfree_pend |= 1u << b;
                }
                const uint16_t *prev = ff ? act_of(s, ff_buf ^ 1u) : act_of(s, b ^ 1u);
                ulonglong2 *const tb = tab_of(s, b);
                uint32_t *const tg = tag_of(s, b);
                uint16_t *const ab = ff ? act_of(s, ff_buf) : act_of(s, b);
                const uint32_t n_cand = n_prev + n_add;
                uint32_t n_act = 0, n_new = 0;
                // activity and snapshot of candidates c0, c1 (one lane's pair)
                auto activity = [&](uint32_t i0, uint32_t i1, uint32_t &q0, uint32_t &q1, ulonglong2 &p0, ulonglong2 &p1,
                                    uint32_t &g0, uint32_t &g1, bool &a0, bool &a1) {
                    q0 = q1 = 0;
                    if (i0 < n_cand) q0 = i0 < n_prev ? prev[i0] : s.add[i0 - n_prev];
                    if (i1 < n_cand) q1 = i1 < n_prev ? prev[i1] : s.add[i1 - n_prev];
                    p0 = s.pl[q0];
                    p1 = s.pl[q1];
                    g0 = L >= 0 ? v.gate[q0] : q0;
                    g1 = L >= 0 ? v.gate[q1] : q1;
                    a0 = i0 < n_cand && (p0.x | p0.y) != 0ull;
                    a1 = i1 < n_cand && (p1.x | p1.y) != 0ull;
                    if (i0 < n_cand) s.bits[q0] = a0 ? kActive : (unsigned char)0;
                    if (i1 < n_cand) s.bits[q1] = a1 ? kActive : (unsigned char)0;
                    if (a0 && snap) { tb[q0] = p0; tg[q0] = st; }
                    if (a1 && snap) { tb[q1] = p1; tg[q1] = st; }
                    if (L < 0 && ((a0 && p0.y != 0ull) || (a1 && p1.y != 0ull)))
                        report(B.status, GP_ERR_NONDETERMINISTIC, cidx, 0xFFFFFFFFu, gcol);
                    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, a0), m1 = __ballot_sync(0xFFFFFFFFu, a1);
                    if (a0) ab[n_act + __popc(m0 & lt_mask)] = (uint16_t)q0;
                    n_act += __popc(m0);
                    if (a1) ab[n_act + __popc(m1 & lt_mask)] = (uint16_t)q1;
                    n_act += __popc(m1);
                };
                auto append = [&](uint32_t partner) {
                    const bool add = partner != kNone && s.bits[partner] == 0;
                    if (add) s.bits[partner] = kAdded;
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, add);
                    if (add) s.add[n_new + __popc(m & lt_mask)] = (uint16_t)partner;
                    n_new += __popc(m);
                };
                auto publish = [&]() {
                    if (!snap) {
                        __syncwarp();
                        return;
                    }
                    if (lane == 0u) sh.step[b] = StepDesc{L, n_act, slot, 0u};
                    __syncwarp();
                    if (lane == 0u) mbar_arrive(&sh.tab_full[b]);
                };
                if (n_cand <= 32u) {
                    // the step's candidates stay in registers (one per lane)
                    uint32_t q0 = 0;
                    if (lane < n_cand) q0 = lane < n_prev ? prev[lane] : s.add[lane - n_prev];
                    const ulonglong2 p0 = s.pl[q0];
                    const uint32_t g0 = L >= 0 ? v.gate[q0] : q0;
                    const bool a0 = lane < n_cand && (p0.x | p0.y) != 0ull;
                    if (lane < n_cand) s.bits[q0] = a0 ? kActive : (unsigned char)0;
                    if (a0 && snap) { tb[q0] = p0; tg[q0] = st; }
                    if (L < 0 && a0 && p0.y != 0ull) report(B.status, GP_ERR_NONDETERMINISTIC, cidx, 0xFFFFFFFFu, gcol);
                    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, a0);
                    if (a0) ab[__popc(m0 & lt_mask)] = (uint16_t)q0;
                    n_act = __popc(m0);
                    publish();
                    if (L >= 0) append(undo(q0, p0, g0, a0, L));
                } else if (n_cand <= 64u) {
                    // two per lane
                    uint32_t q0, q1, g0, g1;
                    ulonglong2 p0, p1;
                    bool a0, a1;
                    activity(lane, lane + 32u, q0, q1, p0, p1, g0, g1, a0, a1);
                    publish();
                    if (L >= 0) {
                        append(undo(q0, p0, g0, a0, L));
                        append(undo(q1, p1, g1, a1, L));
                    }
                } else {
                    // more than 64 candidates: the helper walker warps join in
                    if (lane == 0u) {
                        sh.wcnt[0] = sh.wcnt[1] = 0u;
                        sh.wstep = WalkStep{L, n_prev, n_cand, slot, ab, prev, b, snap ? 1u : 0u, st, 1u};
                    }
                    wsync();                                // the helpers wake
                    large_activity(0u, L, n_prev, n_cand, prev, ab, tb, tg, snap, st);
                    wsync();                                // every candidate classified
                    n_act = sh.wcnt[0];
                    publish();
                    if (L >= 0) large_undo(0u, L, n_act, ab, v);
                    wsync();                                // the helpers are done
                    n_new = sh.wcnt[1];
                }
                if (L >= 0) {
                // the column's measurements at L: their bits into the planes
                    if (cur > 0u && s.ent_l[cur - 1u] == (uint32_t)L) {
                        uint32_t l0 = 0, h0 = cur;
                        while (l0 < h0) {
                            const uint32_t mid = (l0 + h0) >> 1;
                            if (s.ent_l[mid] < (uint32_t)L) l0 = mid + 1; else h0 = mid;
                        }
                        __syncwarp();                       // the gates of L are undone
                        for (uint32_t base = l0; base < cur; base += 32u) {
                            const uint32_t i = base + lane;
                            bool add = false;
                            uint32_t q = 0;
                            if (i < cur) {
                                const unsigned long long w = s.ent_w[i];
                                const uint32_t qv = s.ent_q[i];
                                q = qv & 0x7FFFFFFFu;
                                if (w != 0ull) {
                                    if (qv >> 31) s.pl[q].y ^= w; else s.pl[q].x ^= w;
                                    add = s.bits[q] == 0;        // else on the next list already
                                    if (add) s.bits[q] = kAdded;
                                }
                            }
                            const unsigned m = __ballot_sync(0xFFFFFFFFu, add);
                            if (add) s.add[n_new + __popc(m & lt_mask)] = (uint16_t)q;
                            n_new += __popc(m);
                        }
                        cur = l0;
                    }
                }
                __syncwarp();
                // the emitters see no fast-forward step: the walker releases
                // its window for them too
                if (lane == 0u) {
                    if (ff) mbar_arrive_count(&sh.win_free[slot], NE + 1u);
                    else mbar_arrive(&sh.win_free[slot]);
                }
                if (ff) ff_buf ^= 1u;
                else st++;
                slot = slot == 0u ? nring - 1u : slot - 1u;   // window L - 1
                n_prev = n_act;
                n_add = n_new;
                if (L < 0) break;
                if (emit_lo >= 0 && L == emit_lo) break;        // the segment's last step
                if (L == 0) { L = -1; continue; }
                if (n_prev + n_add == 0u && (uint32_t)(L - 1) < lmin) break;
                L--;
            }
            // the helpers leave
            if (WW > 1u) {
                if (lane == 0u) sh.wstep.cmd = 0u;
                wsync();
            }
            if (ok) {
                // the end-of-column step: the emitters leave on it
                const uint32_t b = st & 1u;
                if ((tfree_pend >> b) & 1u) {
                    if (!wait_warp(&sh.tab_free[b], (tfree_par >> b) & 1u)) ok = false;
                    else tfree_par ^= 1u << b;
                }
                if (ok) {
                    tfree_pend |= 1u << b;
                    if (lane == 0u) {
                        sh.step[b] = StepDesc{0, 0u, 0u, 1u};
                        sh.stop_layer = L;
                    }
                    __syncwarp();
                    if (lane == 0u) mbar_arrive(&sh.tab_full[b]);
                    st++;
                }
            }
            if (lane == 0u) *(volatile uint32_t *)&sh.walk_done = 1u;
        } else if (!producer) {
            // ---- emitters: the noise rows of each published step, a record
            // (the planes of the row's qubits) each
            for (;;) {
                const uint32_t b = st & 1u;
                if (!wait_warp(&sh.tab_full[b], (tfull_par >> b) & 1u)) break;
                tfull_par ^= 1u << b;
                const StepDesc sd = sh.step[b];
                if (sd.end) {
                    __syncwarp();
                    if (lane == 0u) mbar_arrive(&sh.tab_free[b]);
                    st++;
                    break;
                }
                // the walker waited for the window before it published the
                // step, so the window's contents are visible here through the
                // step's release and acquire
                const uint32_t slot = sd.slot;
                const SplitWindow v = sh.desc[slot];
                const ulonglong2 *const tb = tab_of(s, b);
                const uint32_t *const tg = tag_of(s, b);
                const uint16_t *const ab = act_of(s, b);
                const uint32_t n_act = sd.n_act;
                const bool after = sd.layer >= 0;
                const uint32_t stamp = st;
                // planes of qubit x in this step (0 unless x is active)
                auto planes = [&](uint32_t x) -> ulonglong2 {
                    const uint32_t t = tg[x];
                    const ulonglong2 p = tb[x];
                    return t == stamp ? p : make_ulonglong2(0ull, 0ull);
                };
                // (the walker checks the initial state)
                emit_rows(B, rec_cap, chunk, v.aoff, v.boff, v.lists, v.n_after, after, ab, n_act, 32u * ew, 32u * NE,
                          lane, col_tag, planes, []() {});
                chunk.prefetch(B, lane);
                __syncwarp();
                if (lane == 0u) {
                    mbar_arrive(&sh.tab_free[b]);
                    mbar_arrive(&sh.win_free[slot]);
                }
                st++;
            }
        } else {
            // ---- producer: windows lmax, lmax - 1, ..., -1 until the walker
            // leaves the column, each into a slot its last window released
            auto post = [&](int L) {
                const uint32_t need = L > 0 ? (uint32_t)L : 0u;
                if (seg_lo == 0xFFFFFFFFu || need < seg_lo || (uint32_t)L + 1u >= seg_lo + (uint32_t)kSplitSegCache) {
                    seg_lo = (uint32_t)L + 2u > (uint32_t)kSplitSegCache ? (uint32_t)L + 2u - (uint32_t)kSplitSegCache : 0u;
                    const uint32_t n = min((uint32_t)kSplitSegCache, C.n_layers + 1u - seg_lo);
                    __syncwarp();
                    for (uint32_t i = lane; i < n; i += 32u) s.segc[i] = seg_g[seg_lo + i];
                    __syncwarp();
                }
                if (lane != 0u) return;
                const uint4 s1 = s.segc[L + 1 - (int)seg_lo];
                const uint32_t n_after = L >= 0 ? s.segc[L - (int)seg_lo].y : 0u;
                const uint32_t list_start = 2u * s1.x - n_after;
                const uint32_t list_n = n_after + s1.z;
                const uint32_t slot = slot_of(L);
                SplitWindow &d = sh.desc[slot];
                d.n_after = n_after;
                if (nbuf >= 2u && list_n + 1u <= list_cap) {
                    unsigned char *dst = s.win + (size_t)slot * wbytes;
                    const unsigned char *qsrc = L >= 0 ? qbase + (size_t)L * geo.bytes + 2u * geo.qb : qbase;
                    const uint32_t qbytes = L >= 0 ? 4u * geo.nq4 + 4u * geo.qb : 2u * geo.qb;
                    const uint32_t delta = list_start & 1u;
                    const uint32_t lbytes = list_n ? ((list_n + delta) * 8u + 15u) & ~15u : 0u;
                    d.lists = reinterpret_cast<const uint2 *>(dst + windex) + delta;
                    if (L >= 0) {
                        d.gate = reinterpret_cast<const uint32_t *>(dst);
                        d.aoff = reinterpret_cast<const uint16_t *>(dst + 4u * geo.nq4);
                        d.boff = d.aoff + geo.qb;
                    } else {
                        d.gate = nullptr;
                        d.aoff = nullptr;
                        d.boff = reinterpret_cast<const uint16_t *>(dst);
                    }
                    mbar_expect_tx(&sh.win_full[slot], qbytes + lbytes);
                    bulk_load(dst, qsrc, qbytes, &sh.win_full[slot]);
                    if (lbytes) bulk_load(dst + windex, lbase + list_start - delta, lbytes, &sh.win_full[slot]);
                } else {
                    d.lists = lbase + list_start;
                    if (L >= 0) {
                        const unsigned char *p = qbase + (size_t)L * geo.bytes + 2u * geo.qb;
                        d.gate = reinterpret_cast<const uint32_t *>(p);
                        d.aoff = reinterpret_cast<const uint16_t *>(p + 4u * geo.nq4);
                        d.boff = d.aoff + geo.qb;
                    } else {
                        d.gate = nullptr;
                        d.aoff = nullptr;
                        d.boff = reinterpret_cast<const uint16_t *>(qbase);
                    }
                    mbar_arrive(&sh.win_full[slot]);
                }
            };
            volatile uint32_t *const done_v = &sh.walk_done;
            int Lp = (int)lmax;
            while (Lp >= -1) {
                const uint32_t slot = slot_of(Lp);
                if ((free_pend >> slot) & 1u) {
                    uint32_t got = 0;
                    if (lane == 0u) {
                        uint32_t it = 0;
                        for (; it < wlim; it++) {
                            if (mbar_try_wait(&sh.win_free[slot], (free_par >> slot) & 1u)) { got = 1u; break; }
                            if ((it & 15u) == 15u && (*done_v || *tmo_v)) break;
                        }
                        if (it == wlim) *tmo_v = 1u;
                    }
                    if (!__shfl_sync(0xFFFFFFFFu, got, 0)) break;
                    free_par ^= 1u << slot;
                    free_pend &= ~(1u << slot);
                }
                const uint32_t stop = lane == 0u ? (*done_v | *tmo_v) : 0u;
                if (__shfl_sync(0xFFFFFFFFu, stop, 0)) break;
                if (!stall) {
                    post(Lp);
                    post_par ^= 1u << slot;
                    posted_any |= 1u << slot;
                }
                free_pend |= 1u << slot;
                Lp--;
            }
            if (lane == 0u) sh.posted_lo = Lp + 1;
        }
        __syncthreads();
        if (!sh.tmo) {
            // windows posted below the walk's last layer were never used:
            // their copies land (consumers absorb the phase), and no release
            // comes for them
            const int stop_layer = sh.stop_layer, posted_lo = sh.posted_lo;
            for (int k2 = stop_layer - 1; k2 >= posted_lo; k2--) {
                const uint32_t slot = slot_of(k2);
                if (producer) {
                    free_pend &= ~(1u << slot);
                } else if (warp == 0u) {
                    // the walker warp that tracks the window phases
                    if (!wait_bar(&sh.win_full[slot], (full_par >> slot) & 1u)) break;
                    full_par ^= 1u << slot;
                }
            }
        }
        __syncthreads();
        if (sh.tmo) {
            if (threadIdx.x == 0) report(B.status, GP_ERR_TIMEOUT, 1u, gcol, 0u);
            break;
        }
    }
    if (!walker && !producer) chunk.flush(B, rec_cap, lane);
    // copies still in flight (after a timeout) land before the block exits
    if (producer && lane == 0u) {
        for (uint32_t i = 0; i < nring; i++)
            if ((posted_any >> i) & 1u) mbar_wait_bounded(&sh.win_full[i], ((post_par >> i) & 1u) ^ 1u);
    }
}

// instances: walking threads, most qubits, LISTED.  A narrow circuit gets more
// threads than qubits: its active qubits' rows are emitted by four threads each.
struct Instance {
    uint32_t threads, maxq;
    bool listed;
    void (*fn)(Buffers, uint32_t, Stage1Shape);
};
const Instance kInstances[] = {
    {256, 64, false, stage1_kernel<256, 1, false>},
    {480, 480, false, stage1_kernel<480, 1, false>},
    {960, 2880, true, stage1_kernel<960, 3, true>},
    {960, 3840, true, stage1_kernel<960, 4, true>},
    {960, 4800, true, stage1_kernel<960, 5, true>},
    {960, 8640, true, stage1_kernel<960, 9, true>},
};
// the role-split walk, by its threads
const Instance kSplit[] = {
    {128, 0, false, stage1_split_kernel<128>}, {256, 0, false, stage1_split_kernel<256>},
    {512, 0, false, stage1_split_kernel<512>}, {1024, 0, false, stage1_split_kernel<1024>},
};
constexpr uint32_t kNumSplit = 4;
constexpr uint32_t kDenseMin = 32, kDenseMax = 480;   // qubits of the circuits walked one qubit a thread
constexpr uint32_t kNumInstances = sizeof(kInstances) / sizeof(kInstances[0]);

const Instance &instance(uint32_t i) { return i < kNumInstances ? kInstances[i] : kSplit[i - kNumInstances]; }

}  // namespace

cudaError_t stage1_setup(int device, size_t *limit) {
    int optin = 0;
    cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    size_t stat = 0;
    for (uint32_t i = 0; i < kNumInstances + kNumSplit; i++) {
        cudaFuncAttributes fa{};
        if ((e = cudaFuncGetAttributes(&fa, (const void *)instance(i).fn)) != cudaSuccess) return e;
        stat = std::max(stat, fa.sharedSizeBytes);
    }
    *limit = (size_t)optin > stat ? (size_t)optin - stat : 0;
    for (uint32_t i = 0; i < kNumInstances + kNumSplit; i++)
        if ((e = cudaFuncSetAttribute((const void *)instance(i).fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)*limit)) != cudaSuccess)
            return e;
    return cudaSuccess;
}

int stage1_occupancy(const Stage1Shape &sh) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void *)instance(sh.instance).fn,
                                                      (int)sh.threads, sh.smem) != cudaSuccess)
        return 0;
    return occ;
}

// Kernel instance, resident blocks and window ring for circuits of up to maxq
// qubits.  Which walk (stage 1 alone, us, role-split against the walk of every
// qubit): BB [[144,12,12]] (288 qubits, 12 rounds) 268 against 128, 16 adaptive
// branches (399) 1,552 against 693, repetition 25 x 100 rounds (49) 240 against
// 175, surface d = 11 (241) 71 against 61, d = 15 (449) 83 against 74; but
// surface d = 3 (17) 30 against 47, whose two short columns gain nothing from
// stretches, and d = 25 (1,249) 132 against 187, where most of a step's qubits
// are inactive.  Neither line is pinned down: between 480 and 1,249 qubits, and
// for long memories of fewer than 32, only the role-split walk was measured.
// Above 2,520 qubits the role-split tables and two windows no longer fit, and
// the listed walk takes over, with as few qubits a thread as maxq allows (they
// are registers) and at least three windows (stage 1, us, five qubits a thread
// up to 4,800 and two windows / these / candidate lists kept by the whole block:
// d = 36, 6 rounds 125 / 88 / 104, d = 38, 6 rounds 137 / 94 / 109, d = 40, 12
// rounds 240 / 157 / 246; d = 45, 9 rounds 186 / 184 / 211).
// A step is a chain of shared-memory reads and a barrier, so as many blocks as
// fit walk side by side on an SM.  A window buffer holds a whole layer where that fits (about
// two list entries a qubit: every noise row after the gates of L and before
// those of L + 1, two-qubit rows twice), otherwise the index part alone, with
// the lists read from global memory.
Stage1Shape stage1_shape(uint32_t maxq, uint32_t threads, uint32_t blocks_per_sm, size_t limit) {
    Stage1Shape sh{};
    const size_t per_sm = limit + 1024;
    const uint32_t wi = window_index_bytes(maxq);
    if (maxq > kDenseMax || maxq < kDenseMin) {
        // the role-split walk when its tables and at least two windows fit (in
        // as many of the blocks asked for as there is room for); the deepest
        // ring whose windows hold a whole layer is preferred
        const size_t base = split_base_bytes(maxq);
        for (uint32_t k = std::max(blocks_per_sm, 1u); k >= 1u; k--)
        for (size_t want : {2 * (size_t)maxq + 64, (size_t)512})
            for (uint32_t nbuf = kSplitBufs; nbuf >= 2u; nbuf--) {
                const size_t budget = k > 1u ? std::min(limit, per_sm / k - 1024) : limit;
                if (budget < base + (size_t)nbuf * (wi + want * 8)) continue;
                const size_t cap = std::min<size_t>(((budget - base) / nbuf - wi) / 8, 4096) & ~(size_t)15;
                sh.split = 1;
                sh.instance = kNumInstances;
                while (instance(sh.instance).threads < threads) sh.instance++;
                sh.threads = threads;
                sh.blocks = k;
                sh.nbuf = nbuf;
                sh.list_cap = (uint32_t)cap;
                sh.wbytes = wi + (uint32_t)cap * 8;
                sh.smem = base + (size_t)nbuf * sh.wbytes;
                return sh;
            }
    }
    uint32_t i = 0;
    while (i + 1u < kNumInstances && kInstances[i].maxq < maxq) i++;
    const Instance &in = kInstances[i];
    sh.instance = i;
    sh.threads = in.threads + 32u;
    const size_t base = smem_base_bytes(maxq, in.listed);
    const size_t full = wi + 8 * (((size_t)2 * maxq + 64 + 15) & ~(size_t)15);
    const uint32_t most = (uint32_t)min_blocks((int)in.threads);
    const uint32_t first = blocks_per_sm ? std::min(blocks_per_sm, most) : most;
    // whole layers before more blocks, more blocks before a deeper ring; but
    // the listed walk waits less on three windows without their lists than on
    // two with them (d = 38, 6 rounds: 137 -> 117 us)
    for (size_t list_bytes : {full - wi, (size_t)0})
        for (uint32_t k = first; k >= 1u; k--) {
            const size_t budget = k > 1u ? std::min(limit, per_sm / k - 1024) : limit;
            const size_t slot = (wi + list_bytes + 127) & ~(size_t)127;
            if (budget < base + (in.listed && list_bytes ? 3 : 2) * slot) continue;
            const uint32_t nbuf = (uint32_t)std::min<size_t>((budget - base) / slot, 4);
            sh.blocks = k;
            sh.nbuf = nbuf;
            sh.wbytes = (uint32_t)slot;
            sh.list_cap = (uint32_t)((slot - wi) / 8);
            sh.smem = base + nbuf * slot;
            sh.gbytes = (4u * ((maxq + 3u) & ~3u) + 127u) & ~127u;
            // two layers' gates are a window's index part, so two slots fit
            sh.gbatch = std::min<uint32_t>((uint32_t)((sh.smem - base) / sh.gbytes / 2u), 4u);
            sh.ngbuf = std::min<uint32_t>((uint32_t)((sh.smem - base) / ((size_t)sh.gbatch * sh.gbytes)),
                                          (uint32_t)kMaxBufs);
            return sh;
        }
    // no room for window buffers: every window is read from global memory
    sh.blocks = 1;
    sh.gbatch = 1;
    sh.smem = base;
    return sh;
}

void launch_stage1(const Buffers &b, uint32_t grid, uint32_t maxq, const Stage1Shape &sh, cudaStream_t s,
                   uint32_t *launches) {
    instance(sh.instance).fn<<<grid, sh.threads, sh.smem, s>>>(b, maxq, sh);
    *launches += 1;
}

}  // namespace gpdem
