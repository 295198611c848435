// ccpm_kernels.cu -- sm_103a kernels of the constraint-checking pipeline and
// the C ABI that drives them.
//
// Device state of one prune (the paper's vertex state, Alg. 3):
//   omega[2][n]  uint32  omega(v) for rounds k and k+1 (snapshot/Jacobi LCC)
//   ebits[W]     uint32  1 bit per CSR entry: the active edge map epsilon(v)
// A vertex is active exactly when omega(v) != 0.
//
// Edge bits are kept exact for rows of active vertices only.  A bit in the row
// of an active v that points to a vertex u eliminated in the previous round is
// cleared lazily: the next round sees omega(u) = 0, treats the entry as
// inactive and clears the bit.  Rows of eliminated vertices, and of vertices
// that never become active, keep bits that no round reads; they are zeroed when
// the edge bitmap is handed back without the final search.  Once the rows are
// compacted (K4) the rounds read the compacted rows and their own bitmap; the
// full bitmap is then frozen and handed back in its fixpoint form (bit, both
// ends live, compatible omegas).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>


#include <atomic>
#include <climits>
#include <cmath>
#include <chrono>
#include <mutex>
#include <thread>

#include "ccpm_internal.h"

namespace ccpm {

#define FULL_MASK 0xFFFFFFFFu

// -------------------------------------------------------------------------
// device-side bookkeeping
// -------------------------------------------------------------------------

struct RoundStats {
    unsigned long long scanned;   // active CSR entries read this round
    unsigned long long windows;   // CSR entries examined by searches
    unsigned long long expanded;  // ... and while their items were listed
    unsigned long long matches;   // final search: matches found
    unsigned long long tokens;    // NLCC: (vertex, head) searches issued
    unsigned long long row_entries;   // CSR entries in rows of active vertices
    unsigned long long alive;         // active vertices processed
    unsigned long long kept;          // entries still active after the round (rows of survivors)
    unsigned long long rows_next;     // CSR entries in the rows of the survivors
    unsigned int changed;         // any omega or edge changed
    unsigned int n_small, n_med, n_chunk;   // next frontier sizes
    unsigned int n_hub_slots;
    unsigned int n_roots;
    unsigned int n_items;         // (root, head, first candidate) search items
    unsigned int overflow;        // a search hit its budget
    unsigned int skipped;         // LCC round queued after the fixpoint: did nothing
    // changes of omega waiting to be passed on to the neighbours (Change list,
    // and the pieces of their long rows); for a delta round also what its
    // vertices had before: entries active after their last evaluation, and the
    // vertices it eliminates with the entries in their rows
    unsigned int n_chg, n_chg_piece;
    unsigned int died;            // full rounds: survivors are alive - died
    unsigned long long old_kept, died_rows;
};

// Counters of one pass of a search over its items: the next item to take, the
// items handed on by searches that ran long (reserved), and the complement of
// the index below which that list is valid (see spill; zero: all of it).
struct PassCtl {
    unsigned long long next;
    unsigned int n_out, stop_inv;
    __device__ __host__ unsigned int handed_on() const { return n_out < ~stop_inv ? n_out : ~stop_inv; }
};

// A vertex whose omega a round (or a non-local check) has changed, and its new
// omega; a piece of its row if that is long.
struct Change { int32_t v; uint32_t w; };
struct ChangePiece { int32_t v, c; };

struct HubAcc {                   // partial LCC state of one split row
    uint32_t U, nN, flags, done;
    uint32_t cnt[kMaxCls];
    uint32_t pbase;               // index of the row's first piece when the pieces were made
};

struct ChunkItem {                // one piece of a long row
    int32_t v, c, slot, nchunks;
};

struct SmemTmpl {
    uint32_t adj[kMaxT];
    uint32_t cls_mask[kMaxCls];
    uint32_t cls_need[kMaxCls];
    uint32_t cls_q[kMaxCls];
    int n_cls;
};

// Per warp: the rows of one batch of the short-row path.
struct ShortRows {
    int64_t off[32];      // row i's entry k of the batch stream is CSR entry off[i] + k
    uint32_t nbr[32];     // template neighbours of omega(v_i)
    int row[32];          // row whose piece of the current step starts at this lane
};

__device__ __forceinline__ void load_tmpl(SmemTmpl &s, const DevTmpl &t) {
    for (int i = threadIdx.x; i < kMaxT; i += blockDim.x) s.adj[i] = t.adj[i];
    for (int i = threadIdx.x; i < kMaxCls; i += blockDim.x) {
        s.cls_mask[i] = t.cls_mask[i];
        s.cls_need[i] = t.cls_need[i];
        s.cls_q[i] = t.cls_q[i];
    }
    if (threadIdx.x == 0) s.n_cls = t.n_cls;
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Per-warp staging buffer for frontier appends: one global atomic per 32 items.
template <typename T>
struct WarpBuf {
    T *buf;          // 32 slots in shared memory
    int *cnt;        // shared counter
    T *out;          // global list
    unsigned int *gcount;
    unsigned long long cap = ~0ull;   // items past this index are counted, not stored

    __device__ __forceinline__ void flush() {
        int c = *cnt;
        if (c == 0) return;
        unsigned int base = 0;
        if (lane_id() == 0) base = atomicAdd(gcount, (unsigned int)c);
        base = __shfl_sync(FULL_MASK, base, 0);
        if ((int)lane_id() < c && (unsigned long long)base + lane_id() < cap) out[base + lane_id()] = buf[lane_id()];
        __syncwarp();
        if (lane_id() == 0) *cnt = 0;
        __syncwarp();
    }
    // warp-uniform call; lanes with pred push val
    __device__ __forceinline__ void push(bool pred, const T &val) {
        uint32_t m = __ballot_sync(FULL_MASK, pred);
        if (!m) return;
        int n = __popc(m);
        if (*cnt + n > 32) flush();
        int c = *cnt;
        if (pred) buf[c + __popc(m & ((1u << lane_id()) - 1u))] = val;
        __syncwarp();
        if (lane_id() == 0) *cnt = c + n;
        __syncwarp();
    }
};

// The leftovers of a block's warp buffers (at most 32 items each, counts in
// cnt[0..8)): appended with one atomic for the block.  Called by every thread
// after a __syncthreads.
template <typename T>
__device__ __forceinline__ void block_flush(const WarpBuf<T> &b, const int *cnt, int wib) {
    __shared__ unsigned int base;
    int before = 0, total = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
        if (w < wib) before += cnt[w];
        total += cnt[w];
    }
    if (total == 0) return;                          // block-uniform
    if (threadIdx.x == 0) base = atomicAdd(b.gcount, (unsigned int)total);
    __syncthreads();
    if ((int)lane_id() < cnt[wib]) b.out[base + before + lane_id()] = b.buf[lane_id()];
    __syncthreads();                                 // base is reused by the next list
}

__device__ __forceinline__ unsigned long long warp_total(unsigned long long x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL_MASK, x, o);
    return x;
}

// Zero the bits of CSR entries [beg, end); `G` lanes cooperate.  Words fully
// inside the range belong to this row alone and are stored; the two boundary
// words are shared with neighbouring rows and are cleared atomically.
template <int G>
__device__ __forceinline__ void clear_row(uint32_t *ebits, int64_t beg, int64_t end, int lane_g) {
    if (beg >= end) return;
    int64_t w0 = beg >> 5, w1 = (end - 1) >> 5;
    for (int64_t w = w0 + lane_g; w <= w1; w += G) {
        int64_t lo = w << 5;
        uint32_t keep = 0;
        if (beg > lo) keep |= (1u << (uint32_t)(beg - lo)) - 1u;
        if (end < lo + 32) keep |= ~((1u << (uint32_t)(end - lo)) - 1u);
        if (keep) atomicAnd(&ebits[w], keep);
        else ebits[w] = 0u;
    }
}

// OR / sum over aligned groups of G lanes (whole warp: one redux instruction)
template <int G>
__device__ __forceinline__ uint32_t grp_or(uint32_t x) {
    if constexpr (G == 32) {
        return __reduce_or_sync(FULL_MASK, x);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) x |= __shfl_xor_sync(FULL_MASK, x, o);
        return x;
    }
}
template <int G>
__device__ __forceinline__ uint32_t grp_sum(uint32_t x) {
    if constexpr (G == 32) {
        return __reduce_add_sync(FULL_MASK, x);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(FULL_MASK, x, o);
        return x;
    }
}

// -------------------------------------------------------------------------
// K1: INIT_VERTEX_STATE (Alg. 3) and the first frontier
// -------------------------------------------------------------------------

struct LabelMask { uint32_t m[256]; };

// The narrow copy of omega the LCC gathers read (1 or 2 bytes per vertex; 0: none).
__device__ __forceinline__ void store_narrow(void *nw, int bytes, int64_t v, uint32_t w) {
    if (bytes == 1) ((uint8_t *)nw)[v] = (uint8_t)w;
    else if (bytes == 2) ((uint16_t *)nw)[v] = (uint16_t)w;
}

__global__ void __launch_bounds__(256)
k_init(int64_t n, const int64_t *__restrict__ rp, const uint8_t *__restrict__ lab, LabelMask lm,
       const uint32_t *__restrict__ om_in, uint32_t *om0, uint32_t *om1, void *nw0, void *nw1, int nw_bytes,
       int32_t *small_out, int32_t *med_out, ChunkItem *chunk_out, HubAcc *acc, RoundStats *st, int hub_deg,
       int short_max, unsigned int set_changed, const RoundStats *only_if, uint32_t *ebits, int64_t m) {
    if (only_if && only_if->changed == 0u) return;
    if (ebits && blockIdx.x == 0 && threadIdx.x == 0) {
        // no entries past m: the padding bits of the last word and the guard word stay 0
        if (m & 31) ebits[m >> 5] &= (1u << (uint32_t)(m & 31)) - 1u;
        ebits[(m + 31) >> 5] = 0u;
    }
    __shared__ uint32_t slm[256];
    __shared__ int32_t sbuf[2][8][32];
    __shared__ int scnt[2][8];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) slm[i] = lm.m[i];
    const int wib = threadIdx.x >> 5;
    if (lane_id() == 0) { scnt[0][wib] = 0; scnt[1][wib] = 0; }
    __syncthreads();
    WarpBuf<int32_t> bs{sbuf[0][wib], &scnt[0][wib], small_out, &st->n_small};
    WarpBuf<int32_t> bm{sbuf[1][wib], &scnt[1][wib], med_out, &st->n_med};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_pad = (n + 31) & ~(int64_t)31;
    unsigned long long rows = 0;          // entries in the rows of the active vertices
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_pad; v += stride) {
        uint32_t w = 0;
        int64_t deg = 0;
        if (v < n) {
            w = slm[lab[v]];
            if (om_in) w &= om_in[v];     // resumed state, kept inside the initial one
            om0[v] = w;
            om1[v] = w;
            store_narrow(nw0, nw_bytes, v, w);
            store_narrow(nw1, nw_bytes, v, w);
            if (w) deg = rp[v + 1] - rp[v];
        }
        rows += (unsigned long long)deg;
        // buckets: short rows (4 lanes each), medium rows (a warp each), long
        // rows (split into pieces of hub_deg entries); every active vertex is
        // in exactly one of them
        const int64_t small_max = hub_deg < short_max ? hub_deg : short_max;
        bs.push(w && deg <= small_max, (int32_t)v);
        bm.push(w && deg > small_max && deg <= hub_deg, (int32_t)v);
        if (w && deg > hub_deg) {
            int nch = (int)((deg + hub_deg - 1) / hub_deg);
            int slot = (int)atomicAdd(&st->n_hub_slots, 1u);
            unsigned int base = atomicAdd(&st->n_chunk, (unsigned int)nch);
            acc[slot].pbase = base;
            for (int c = 0; c < nch; c++) chunk_out[base + c] = ChunkItem{(int32_t)v, c, slot, nch};
        }
    }
    bs.flush();
    bm.flush();
    for (int o = 16; o > 0; o >>= 1) rows += __shfl_xor_sync(FULL_MASK, rows, o);
    if (lane_id() == 0 && rows) atomicAdd(&st->row_entries, rows);
    // the first round reads these counters as those of a round before it
    if (blockIdx.x == 0 && threadIdx.x == 0 && set_changed) st->changed = 1u;
}

// -------------------------------------------------------------------------
// K2/K3: one LCC round (Alg. 4 with Alg. 5), snapshot form
// -------------------------------------------------------------------------

struct LccArgs {
    const int64_t *rp;
    const int32_t *col;
    const uint32_t *om_cur;
    uint32_t *om_next;
    uint32_t *ebits;
    const int32_t *small_in;
    const int32_t *med_in;
    const ChunkItem *chunk_in;
    int64_t n_small, n_med, n_chunk;
    int32_t *small_out;
    int32_t *med_out;
    ChunkItem *chunk_out;
    HubAcc *acc;
    RoundStats *st;
    int hub_deg;
    uint32_t *deg;                // entries each evaluated vertex keeps (0 if it dies), or nullptr
    // delta rounds (kDelta): the lists hold the vertices to look at again (their
    // bit in `dirty` is set), omega is read and not written: what changes goes
    // to the Change list
    uint32_t *dirty;
    Change *chg;
    ChangePiece *chg_piece;
    int med_chunk;                // medium vertices a warp prefetches together (1..16)
    // first round after a fresh init: omega(u) is the initial mask of u's
    // label, so the neighbour gather reads the 1-byte label instead of the
    // 4-byte omega word (lab0 = labels, lmask = label -> initial omega)
    const uint8_t *lab0;
    LabelMask lmask;
    // with lab0: the neighbours' labels in CSR entry order (one byte per
    // entry, built once per graph), so the first round reads neither the
    // column index nor the neighbour's label: omega(u) = lmask[elab[e]]
    const uint8_t *elab;
    // later rounds over the full rows: warp-per-row paths visit only the set
    // bits (most entries of a live row are inactive by then)
    int sparse;
    // rounds queued without a host round trip: the list sizes come from the
    // previous round's counters, and a round after the fixpoint does nothing
    const RoundStats *prev;       // nullable: sizes are the fields above
    const RoundStats *gate;       // nullable: the round runs only if these counters say `changed`
    int resident_warps;           // warps of one resident wave (medium prefetch unit)
    uint32_t eta_off;             // ~0: ablation without edge elimination (every live
                                  // neighbour passes eta); 0: the method
    // a narrow copy of omega for the neighbour gathers (templates of at most
    // 8 / 16 vertices: 1 / 2 bytes per vertex, 4x / 2x fewer bytes than the
    // 32-bit words, so it stays in L2 at scale 25): read nw_cur, written to
    // nw_next beside om_next; nw_bytes 0 = no copy (gather om_cur)
    const void *nw_cur;
    void *nw_next;
    int nw_bytes;
};

// A neighbour's omega for the LCC gathers: from the narrow copy when there is one.
__device__ __forceinline__ uint32_t gather_om(const uint32_t *__restrict__ om, const void *nw, int nwb, int32_t u) {
    if (nwb == 1) return __ldg((const uint8_t *)nw + u);
    if (nwb == 2) return __ldg((const uint16_t *)nw + u);
    return __ldg(om + u);
}

// omega'(v) of the next round, and its narrow copy.
__device__ __forceinline__ void store_om(const LccArgs &a, int32_t v, uint32_t w) {
    a.om_next[v] = w;
    store_narrow(a.nw_next, a.nw_bytes, v, w);
}

// Rounds: the first after init (every edge bit of its rows set), over every
// active vertex, and over the vertices near a change only.
constexpr int kDense = 0, kFull = 1, kDelta = 2;

template <int MAXC>
struct Partial {
    uint32_t U = 0, nN = 0, achg = 0;
    uint32_t cnt[MAXC > 0 ? MAXC : 1];
    __device__ __forceinline__ Partial() {
#pragma unroll
        for (int c = 0; c < (MAXC > 0 ? MAXC : 1); c++) cnt[c] = 0;
    }
};

// Position of the r-th (0-based) set bit of x (x has more than r set bits):
// halve the range, keeping the half that holds it.
__device__ __forceinline__ uint32_t select_bit(uint32_t x, uint32_t r) {
    uint32_t pos = 0;
#pragma unroll
    for (uint32_t w = 16; w > 0; w >>= 1) {
        const uint32_t low = __popc(x & ((1u << w) - 1u));
        if (low <= r) { r -= low; x >>= w; pos += w; }
    }
    return pos;
}

template <int MAXC>
__device__ __forceinline__ void tally_entry(uint32_t w, uint32_t nbr_v, const SmemTmpl &s, const uint32_t (&cm)[4],
                                            Partial<MAXC> &p, uint32_t &scanned, bool &keep) {
    keep = (w & nbr_v) != 0u;
    scanned += w != 0u;
    if (w != 0u && !keep) p.achg = 1u;  // eta eliminates the entry
    if (keep) {
        p.U |= w;
        p.nN++;
        if constexpr (MAXC > 0 && MAXC <= 4) {
#pragma unroll
            for (int c = 0; c < MAXC; c++) p.cnt[c] += (w & cm[c]) ? 1u : 0u;
        } else {
#pragma unroll
            for (int c = 0; c < MAXC; c++)
                if (c < s.n_cls) p.cnt[c] += (w & s.cls_mask[c]) ? 1u : 0u;
        }
    }
}

// Visit the entries of [beg, end) whose bit is set, 32 at a time and in
// ascending order: f(e, valid) is called by all lanes, lane i with the i-th
// set entry of the batch (valid) or none.  The bits are read 32 words
// (1024 entries) per load, so long runs of inactive entries cost little.
template <typename F>
__device__ __forceinline__ void for_set_bits(const uint32_t *bits, int64_t beg, int64_t end, F &&f) {
    const int lane = (int)lane_id();
    const int64_t wb = beg >> 5, we = (end + 31) >> 5;
    for (int64_t w0 = wb; w0 < we; w0 += 32) {
        const int64_t wi = w0 + lane;
        uint32_t word = 0u;
        if (wi < we) {
            word = bits[wi];
            const int64_t e0 = wi << 5;
            if (e0 < beg) word &= ~0u << (uint32_t)(beg - e0);
            if (end - e0 < 32) word &= (1u << (uint32_t)(end - e0)) - 1u;
        }
        const uint32_t c = __popc(word);
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t total = __shfl_sync(FULL_MASK, incl, 31);
        const uint32_t excl = incl - c;
        for (uint32_t k0 = 0; k0 < total; k0 += 32) {
            const uint32_t k = k0 + (uint32_t)lane;
            int i = 0;                                // last word whose prefix is <= k
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const uint32_t ex = __shfl_sync(FULL_MASK, excl, i + step);
                if (ex <= k) i += step;
            }
            const uint32_t wd = __shfl_sync(FULL_MASK, word, i);
            const uint32_t ex_i = __shfl_sync(FULL_MASK, excl, i);
            const bool valid = k < total;
            int64_t e = -1;
            if (valid) e = ((w0 + i) << 5) + (int64_t)select_bit(wd, k - ex_i);
            f(e, valid);
        }
    }
}

// Later rounds over the full rows, where most entries of a live row are
// already inactive: only the entries whose bit is set are visited, 32 per
// step (one per lane).  The bits of up to 1024 entries are read per load (one
// word per lane); lane k takes the k-th set bit of the group by a search over
// the words' prefix counts.  The next step's entries are located and their
// column indices loaded while the current step's neighbour omegas are
// gathered.  A failing entry's bit is cleared with an atomic (the words at
// the ends of the range are shared with other rows).
template <int MAXC>
__device__ __forceinline__ void scan_row_sparse(int64_t beg, int64_t end, uint32_t nbr_v,
                                                const int32_t *__restrict__ col, const uint32_t *__restrict__ om,
                                                uint32_t *ebits, const SmemTmpl &s, Partial<MAXC> &p,
                                                uint32_t &scanned, const uint32_t (&cm)[4], const void *nw, int nwb) {
    const int lane = (int)lane_id();
    const int64_t wb = beg >> 5, we = (end + 31) >> 5;
    for (int64_t g0 = wb; g0 < we; g0 += 32) {
        const int64_t wi = g0 + lane;
        uint32_t word = 0u;
        if (wi < we) {
            word = ebits[wi];
            const int64_t e0 = wi << 5;
            if (e0 < beg) word &= ~0u << (uint32_t)(beg - e0);
            if (end - e0 < 32) word &= (1u << (uint32_t)(end - e0)) - 1u;
        }
        const uint32_t c = __popc(word);
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t total = __shfl_sync(FULL_MASK, incl, 31);
        const uint32_t excl = incl - c;
        // lane k of a step: the (k0 + k)-th set entry of the group, and its column
        auto locate = [&](uint32_t k0, int64_t &e, int32_t &u) {
            const uint32_t k = k0 + (uint32_t)lane;
            int i = 0;                                  // last word whose prefix is <= k
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const uint32_t ex = __shfl_sync(FULL_MASK, excl, i + step);
                if (ex <= k) i += step;
            }
            const uint32_t wd = __shfl_sync(FULL_MASK, word, i);
            const uint32_t ex_i = __shfl_sync(FULL_MASK, excl, i);
            e = -1;
            u = 0;
            if (k < total) {
                e = ((g0 + i) << 5) + (int64_t)select_bit(wd, k - ex_i);
                u = __ldcs(col + e);
            }
        };
        int64_t e_c = -1;
        int32_t u_c = 0;
        if (total) locate(0, e_c, u_c);
        for (uint32_t k0 = 0; k0 < total; k0 += 32) {
            const uint32_t w = e_c >= 0 ? gather_om(om, nw, nwb, u_c) : 0u;
            int64_t e_n = -1;
            int32_t u_n = 0;
            if (k0 + 32 < total) locate(k0 + 32, e_n, u_n);
            bool keep;
            tally_entry<MAXC>(w, nbr_v, s, cm, p, scanned, keep);
            if (e_c >= 0 && !keep) atomicAnd(&ebits[e_c >> 5], ~(1u << (uint32_t)(e_c & 31)));
            e_c = e_n;
            u_c = u_n;
        }
    }
}

// Stream the CSR entries [beg, end) of an active vertex: edge elimination by
// eta (entry kept iff the neighbour's omega contains a template neighbour of
// some q in omega(v)), the union omega' of Alg. 4 and the per-class counts of
// distinct compatible neighbours.
//
// Warp form: all 32 lanes walk the row together in windows aligned to the
// 32-entry words of the edge bitmap, so lane i of a window always owns bit i
// of one word: the bits of a window are one broadcast load and its failing
// entries are cleared with one ballot and one atomic.  Entry offsets are kept
// relative to the first window (32-bit), so the loads of a step use one base
// pointer with constant offsets.
// DENSE: every edge bit of the rows read is still set (the first round after
// init), so the bits are not loaded; otherwise a column index is only loaded
// for entries whose bit is set.
template <int MAXC, bool DENSE>
__device__ __forceinline__ void scan_row_warp(int64_t beg, int64_t end, uint32_t nbr_v,
                                              const int32_t *__restrict__ col,
                                              const uint32_t *__restrict__ om, uint32_t *ebits,
                                              const SmemTmpl &s, Partial<MAXC> &p,
                                              uint32_t &scanned, const uint8_t *__restrict__ lab0,
                                              const uint32_t *slm, const uint32_t (&cm)[4], const void *nw,
                                              int nwb, const uint8_t *__restrict__ elab, bool sparse) {
    if constexpr (!DENSE) {
        if (sparse) {
            scan_row_sparse<MAXC>(beg, end, nbr_v, col, om, ebits, s, p, scanned, cm, nw, nwb);
            return;
        }
    }
    constexpr int UNR = 4;   // windows per step
    const int lane = (int)lane_id();
    const int64_t w0 = beg >> 5;
    const int nwin = (int)(((end + 31) >> 5) - w0);
    const int lo = (int)(beg - (w0 << 5));          // entries before lo belong to the previous row
    const int hi = (int)(end - (w0 << 5));          // entries from hi on belong to the next row
    const int32_t *cb = col + (w0 << 5) + lane;
    const uint8_t *lb = (DENSE && elab) ? elab + (w0 << 5) + lane : nullptr;   // first round only
    uint32_t *eb = ebits + w0;
    // the column indices of the next step are loaded while the neighbour
    // omegas of the current step are gathered
    bool act[UNR];
    int32_t u[UNR];
    auto load_step = [&](int k0) {
        const int rel0 = k0 * 32 + lane;
        const int32_t *c0 = cb + k0 * 32;
        uint32_t word[UNR];
#pragma unroll
        for (int j = 0; j < UNR; j++) {
            word[j] = ~0u;
            if (!DENSE) word[j] = (k0 + j < nwin) ? eb[k0 + j] : 0u;
        }
#pragma unroll
        for (int j = 0; j < UNR; j++) {
            const int rel = rel0 + j * 32;
            act[j] = rel >= lo && rel < hi && ((word[j] >> lane) & 1u);
            // the column index, or the neighbour's label when the entry labels are given
            if (lb) u[j] = act[j] ? (int32_t)__ldcs(lb + k0 * 32 + j * 32) : 0;
            else u[j] = act[j] ? __ldcs(c0 + j * 32) : 0;
        }
    };
    load_step(0);
    for (int k0 = 0; k0 < nwin; k0 += UNR) {
        uint32_t wu[UNR];
        bool was[UNR];
#pragma unroll
        for (int j = 0; j < UNR; j++) {
            was[j] = act[j];
            if (lb) wu[j] = act[j] ? slm[u[j]] : 0u;
            else if (lab0) wu[j] = act[j] ? slm[__ldg(lab0 + u[j])] : 0u;
            else wu[j] = act[j] ? gather_om(om, nw, nwb, u[j]) : 0u;
        }
        if (k0 + UNR < nwin) load_step(k0 + UNR);
#pragma unroll
        for (int j = 0; j < UNR; j++) {
            if (k0 + j >= nwin) break;          // past the row's last window (warp-uniform)
            const uint32_t w = wu[j];
            const bool keep = (w & nbr_v) != 0u;
            scanned += w != 0u;
            if (w != 0u && !keep) p.achg = 1u;  // eta eliminates the entry
            if (keep) {
                p.U |= w;
                p.nN++;
                if constexpr (MAXC > 0 && MAXC <= 4) {
#pragma unroll
                    for (int c = 0; c < MAXC; c++) p.cnt[c] += (w & cm[c]) ? 1u : 0u;
                } else {
#pragma unroll
                    for (int c = 0; c < MAXC; c++)
                        if (c < s.n_cls) p.cnt[c] += (w & s.cls_mask[c]) ? 1u : 0u;
                }
            }
            // the bit goes with the failing entries and with those whose other
            // end is already inactive (no change of the state A: that entry is
            // inactive already), so later rounds and compaction see only live
            // compatible entries
            const uint32_t drop = __ballot_sync(FULL_MASK, was[j] && !keep);
            if (drop) {
                const int k = k0 + j;
                if (k * 32 >= lo && k * 32 + 32 <= hi) {
                    // the word holds entries of this row only
                    const uint32_t kept = __ballot_sync(FULL_MASK, keep);
                    if (lane == 0) eb[k] = kept;
                } else if (lane == 0) {
                    atomicAnd(&eb[k], ~drop);
                }
            }
        }
    }
}

// Clear the entries of a row (at most 32 long) given by a row-relative mask.
__device__ __forceinline__ void clear_rel(uint32_t *ebits, int64_t beg, uint32_t clr) {
    if (!clr) return;
    const uint32_t sh = (uint32_t)(beg & 31);
    atomicAnd(&ebits[beg >> 5], ~(clr << sh));
    if (sh && (clr >> (32 - sh))) atomicAnd(&ebits[(beg >> 5) + 1], ~(clr >> (32 - sh)));
}

// The vertex-elimination rule of Alg. 4 plus the multiplicity rule of
// Section 4.1: q survives iff adj(q) is inside omega' and every class of q
// has enough distinct neighbours; no surviving edge eliminates the vertex.
template <int MAXC>
__device__ __forceinline__ uint32_t decide(uint32_t wv, const Partial<MAXC> &p, const SmemTmpl &s) {
    uint32_t keep = 0;
    for (uint32_t m = wv; m; m &= m - 1u) {
        int q = __ffs(m) - 1;
        if ((s.adj[q] & ~p.U) == 0u) keep |= 1u << q;
    }
#pragma unroll
    for (int c = 0; c < MAXC; c++)
        if (c < s.n_cls && p.cnt[c] < s.cls_need[c]) keep &= ~s.cls_q[c];
    if (p.nN == 0u) keep = 0u;
    return keep;
}

__device__ __forceinline__ uint32_t nbr_mask(uint32_t wv, const SmemTmpl &s) {
    uint32_t m = 0;
    for (uint32_t x = wv; x; x &= x - 1u) m |= s.adj[__ffs(x) - 1];
    return m;
}

// Round counters one warp accumulates (summed once at the end of the kernel).
struct LccTally {
    uint32_t scanned = 0;          // per lane
    unsigned long long rows = 0, alive = 0, kept = 0, rows_next = 0;   // lane 0 (or the row lanes)
    unsigned long long old_kept = 0, died_rows = 0;                    // delta rounds
    uint32_t changed = 0, died = 0;
};

// The round counters of a block's warps, one atomic per counter and block:
// with a warp each, the thousands of atomics on one address lasted longer than
// the round itself on small frontiers.  totals: 9 zeroed words of shared memory.
__device__ __forceinline__ void add_totals(const LccTally &tl, unsigned long long *totals, RoundStats *st) {
    auto add = [&](int i, unsigned long long x) {
        x = warp_total(x);
        if (lane_id() == 0 && x) atomicAdd(&totals[i], x);
    };
    add(0, tl.scanned);
    add(1, tl.rows);
    add(2, tl.alive);
    add(3, tl.kept);
    add(4, tl.rows_next);
    add(5, tl.changed);
    add(6, tl.died);
    add(7, tl.old_kept);
    add(8, tl.died_rows);
    __syncthreads();
    const unsigned long long sum = threadIdx.x < 9 ? totals[threadIdx.x] : 0ull;
    if (sum) {
        switch (threadIdx.x) {
            case 0: atomicAdd(&st->scanned, sum); break;
            case 1: atomicAdd(&st->row_entries, sum); break;
            case 2: atomicAdd(&st->alive, sum); break;
            case 3: atomicAdd(&st->kept, sum); break;
            case 4: atomicAdd(&st->rows_next, sum); break;
            case 5: atomicOr(&st->changed, 1u); break;
            case 6: atomicAdd(&st->died, (unsigned int)sum); break;
            case 7: atomicAdd(&st->old_kept, sum); break;
            default: atomicAdd(&st->died_rows, sum); break;
        }
    }
}

// What a round decided for vertex v (one lane): its omega was wv and is now
// `keep`, `kept` of the `len` entries of its row stay active.  A full round
// writes omega'; a delta round lists the change (long: the row is longer than
// hub_deg, its pieces are listed too).
template <int MODE>
__device__ __forceinline__ void settle(const LccArgs &a, int32_t v, uint32_t wv, uint32_t keep, uint32_t kept,
                                       int64_t len, bool is_long, LccTally &tl) {
    if (keep) { tl.kept += kept; tl.rows_next += (unsigned long long)len; }
    else tl.died++;
    if (MODE == kDelta) {
        tl.old_kept += a.deg[v];
        if (keep == 0u) tl.died_rows += (unsigned long long)len;
        if (keep != wv && is_long) {
            const unsigned int np = (unsigned int)((len + a.hub_deg - 1) / a.hub_deg);
            const unsigned int b = atomicAdd(&a.st->n_chg_piece, np);
            for (unsigned int c = 0; c < np; c++)
                a.chg_piece[b + c] = ChangePiece{v, (int32_t)c};
        }
    } else {
        store_om(a, v, keep);
    }
    if (a.deg) a.deg[v] = keep ? kept : 0u;
}

// A listed vertex that died in an earlier round.
template <int MODE>
__device__ __forceinline__ void settle_dead(const LccArgs &a, int32_t v) {
    if (MODE == kDelta) return;
    store_om(a, v, 0u);
    if (a.deg) a.deg[v] = 0u;
}

__device__ __forceinline__ void clear_dirty(const LccArgs &a, int32_t v) {
    atomicAnd(&a.dirty[v >> 5], ~(1u << (v & 31)));
}


// Short rows, up to 32 per warp batch (lane i owns row i of the batch).  The rows'
// entries are walked as one stream, 32 per step with one entry per lane, so
// lanes stay busy whatever the row lengths.  A step holds pieces of several
// rows: every lane finds its row from the piece starts, and per-row sums are
// segmented warp reductions whose result each row's lane collects.
//
// The walk is software-pipelined: while the neighbour omegas (or labels) of
// one step are gathered, the next step's rows are located and its edge bits
// and column indices are loaded, and the next batch's list entries, omegas
// and row offsets are loaded during the current batch.  The column loads
// stream past the caches (read once per round).

// Where the entries of one step lie: lane k holds stream entry k0 + k.
struct ShortStep {
    uint32_t seg;        // lanes of this lane's row piece
    int seg_lo;          // first lane of the piece
    int64_t e;           // CSR entry
    uint32_t nb;         // template neighbours of its row's omega
    bool act;            // a live entry (in range, bit set)
    int32_t u;           // its column index (valid when act)
    bool ov;             // row lane: its row has a piece in this step ...
    int lo;              // ... starting at this lane
};

template <bool DENSE>
__device__ __forceinline__ void short_locate(const LccArgs &a, ShortRows &sr, int k0, int T, int start, int d,
                                             ShortStep &st) {
    const int lane = (int)lane_id();
    const int lo = max(start, k0) - k0, hi = min(start + d, k0 + 32) - k0;
    st.ov = lo < hi;
    st.lo = lo;
    if (st.ov) sr.row[lo] = lane;
    const uint32_t H = __reduce_or_sync(FULL_MASK, st.ov ? (1u << lo) : 0u);   // piece starts (bit 0 always)
    __syncwarp();
    const uint32_t upto = lane == 31 ? FULL_MASK : ((2u << lane) - 1u);
    st.seg_lo = 31 - __clz(H & upto);
    const uint32_t above = H & ~upto;
    const int seg_hi = above ? __ffs(above) - 1 : 32;
    st.seg = (seg_hi == 32 ? FULL_MASK : ((1u << seg_hi) - 1u)) & ~((1u << st.seg_lo) - 1u);
    const int r = sr.row[st.seg_lo];
    const int k = k0 + lane;
    const bool valid = k < T;
    st.e = sr.off[r] + k;
    st.nb = sr.nbr[r];
    st.act = valid;
    if (!DENSE && valid) st.act = (__ldg(a.ebits + (st.e >> 5)) >> (uint32_t)(st.e & 31)) & 1u;
    if (DENSE && a.elab) st.u = st.act ? (int32_t)__ldcs(a.elab + st.e) : 0;   // the neighbour's label
    else st.u = st.act ? __ldcs(a.col + st.e) : 0;
    __syncwarp();                                // sr.row is rewritten by the next step
}

template <int MAXC, int MODE>
__device__ __forceinline__ void short_rows(const LccArgs &a, const SmemTmpl &s, const uint32_t *slm,
                                           const uint32_t (&cm)[4], ShortRows &sr, int64_t first, int64_t stride,
                                           int64_t n_small, WarpBuf<int32_t> &bs, WarpBuf<Change> &bg, LccTally &tl) {
    constexpr bool DENSE = MODE == kDense;
    const int lane = (int)lane_id();
    // A batch is one serial walk over its rows' entries: 32 rows of 50 entries
    // take 50 steps of a microsecond each.  A frontier that gives the resident
    // warps less than 32 rows each is dealt out in smaller batches (a round over
    // 3000 such rows of an 8192-vertex graph: 55 us with 32 rows to a warp, 10 us
    // with one).
    const int per = (int)max((int64_t)1, min((int64_t)32, n_small / stride));
    const int64_t n_batch = (n_small + per - 1) / per;
    auto load_v = [&](int64_t ch) -> int32_t {
        const int64_t idx = ch * per + lane;
        return (ch < n_batch && lane < per && idx < n_small) ? a.small_in[idx] : -1;
    };
    int32_t v_nx = load_v(first);
    uint32_t wv_nx = 0u;
    int64_t b_nx = 0;
    int d_nx = 0;
    auto load_row = [&]() {
        wv_nx = 0u; b_nx = 0; d_nx = 0;
        if (v_nx >= 0) {
            wv_nx = __ldg(a.om_cur + v_nx);
            if (wv_nx) {
                b_nx = a.rp[v_nx];
                d_nx = (int)(a.rp[v_nx + 1] - b_nx);
            }
        }
    };
    load_row();
    for (int64_t ch = first; ch < n_batch; ch += stride) {
        const int32_t v = v_nx;
        const uint32_t wv = wv_nx;
        const int64_t b = b_nx;
        const int d = d_nx;
        v_nx = load_v(ch + stride);              // in flight during this batch
        const uint32_t nbr = wv ? (nbr_mask(wv, s) | a.eta_off) : 0u;
        int S = d;                               // inclusive prefix of the row lengths
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL_MASK, S, o);
            if (lane >= o) S += t;
        }
        const int T = __shfl_sync(FULL_MASK, S, 31);
        const int start = S - d;
        sr.off[lane] = b - start;
        sr.nbr[lane] = nbr;
        uint32_t U = 0u, N = 0u;
        uint32_t cnt[MAXC > 0 ? MAXC : 1];
#pragma unroll
        for (int c = 0; c < (MAXC > 0 ? MAXC : 1); c++) cnt[c] = 0u;
        __syncwarp();
        ShortStep cur;
        if (T > 0) short_locate<DENSE>(a, sr, 0, T, start, d, cur);
        load_row();                              // the next batch's omegas and offsets
        for (int k0 = 0; k0 < T; k0 += 32) {
            uint32_t w = 0u;
            if (cur.act)
                w = (DENSE && a.elab) ? slm[cur.u]
                           : (a.lab0 ? slm[__ldg(a.lab0 + cur.u)] : gather_om(a.om_cur, a.nw_cur, a.nw_bytes, cur.u));
            ShortStep nx;
            if (k0 + 32 < T) short_locate<DENSE>(a, sr, k0 + 32, T, start, d, nx);
            const bool keep = (w & cur.nb) != 0u;
            tl.scanned += w != 0u;
            if (w != 0u && !keep) tl.changed = 1u;       // eta eliminates a live entry
            // entries whose other end is already inactive lose their bit too (no
            // change of the state: such an entry is inactive already)
            const uint32_t dm = __ballot_sync(FULL_MASK, cur.act && !keep) & cur.seg;
            uint32_t gk[MAXC > 4 ? MAXC : 1];
            uint32_t rk;
            const uint32_t ru = __reduce_or_sync(cur.seg, keep ? w : 0u);
            if constexpr (MAXC <= 4) {
                // the kept count and up to four class counts of a piece (each at
                // most 32) packed in 6-bit fields
                uint32_t pk = keep ? 1u : 0u;
#pragma unroll
                for (int c = 0; c < MAXC; c++)
                    if (keep && (w & cm[c])) pk += 1u << (6 * (c + 1));
                rk = __reduce_add_sync(cur.seg, pk);
            } else {
                rk = __reduce_add_sync(cur.seg, keep ? 1u : 0u);
#pragma unroll
                for (int c = 0; c < MAXC; c++)
                    gk[c] = c < s.n_cls ? __reduce_add_sync(cur.seg, (keep && (w & s.cls_mask[c])) ? 1u : 0u) : 0u;
            }
            if (lane == cur.seg_lo && dm) {
                // the piece's entries are consecutive from e: at most two words
                const uint32_t bits = dm >> cur.seg_lo;
                const uint32_t sh = (uint32_t)(cur.e & 31);
                atomicAnd(&a.ebits[cur.e >> 5], ~(bits << sh));
                if (sh && (bits >> (32 - sh))) atomicAnd(&a.ebits[(cur.e >> 5) + 1], ~(bits >> (32 - sh)));
            }
            // each row's lane takes the sums of its piece
            const int src = cur.ov ? cur.lo : 0;
            const uint32_t gu = __shfl_sync(FULL_MASK, ru, src);
            const uint32_t gr = __shfl_sync(FULL_MASK, rk, src);
            if constexpr (MAXC <= 4) {
                if (cur.ov) {
                    U |= gu;
                    N += gr & 63u;
#pragma unroll
                    for (int c = 0; c < MAXC; c++) cnt[c] += (gr >> (6 * (c + 1))) & 63u;
                }
            } else {
                uint32_t gc[MAXC];
#pragma unroll
                for (int c = 0; c < MAXC; c++) gc[c] = __shfl_sync(FULL_MASK, gk[c], src);
                if (cur.ov) {
                    U |= gu;
                    N += gr;
#pragma unroll
                    for (int c = 0; c < MAXC; c++) cnt[c] += gc[c];
                }
            }
            cur = nx;
        }
        uint32_t keep = 0u;
        if (v >= 0) {
            if (wv) {
                Partial<MAXC> p;
                p.U = U;
                p.nN = N;
#pragma unroll
                for (int c = 0; c < (MAXC > 0 ? MAXC : 1); c++) p.cnt[c] = cnt[c];
                keep = decide<MAXC>(wv, p, s);
                tl.rows += (unsigned long long)d;
                tl.alive++;
                if (keep != wv) tl.changed = 1u;
                settle<MODE>(a, v, wv, keep, N, d, d > a.hub_deg, tl);
            } else {
                settle_dead<MODE>(a, v);
            }
            if (MODE == kDelta) clear_dirty(a, v);
        }
        // the batch's vertices that were active at the start of the round (delta:
        // those whose omega changes)
        if (MODE == kDelta) bg.push(v >= 0 && keep != wv, Change{v, keep});
        else bs.push(v >= 0 && wv != 0u, v);
        __syncwarp();                            // sr.off / sr.nbr are rewritten by the next batch
    }
}

template <int MAXC, int MODE>
__global__ void __launch_bounds__(256, 4)
k_lcc_round(LccArgs a, DevTmpl t) {
    constexpr bool DENSE = MODE == kDense;
    int64_t n_small = a.n_small, n_med = a.n_med, n_chunk = a.n_chunk;
    int MB = a.med_chunk;
    const RoundStats *gate = a.prev ? a.prev : a.gate;
    if (gate && gate->changed == 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.st->skipped = 1u;
        return;
    }
    if (a.prev) {
        // a full round's lists were written by the round before, a delta
        // round's by k_push into its own counters
        const RoundStats *sizes = MODE == kDelta ? a.st : a.prev;
        n_small = sizes->n_small;
        n_med = sizes->n_med;
        n_chunk = sizes->n_chunk;
        MB = (int)max((int64_t)1, min((int64_t)16, n_med / (4 * (int64_t)a.resident_warps)));
    }
    __shared__ SmemTmpl s;
    __shared__ uint32_t slm[256];
    __shared__ int32_t sbuf[2][8][32];
    __shared__ ChunkItem cbuf[8][32];
    __shared__ ShortRows srows[8];
    __shared__ Change gbuf[MODE == kDelta ? 8 : 1][32];
    __shared__ int scnt[4][8];
    __shared__ unsigned long long totals[9];
    if (threadIdx.x < 9) totals[threadIdx.x] = 0ull;
    load_tmpl(s, t);
    if (a.lab0)
        for (int i = threadIdx.x; i < 256; i += blockDim.x) slm[i] = a.lmask.m[i];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane == 0) { scnt[0][wib] = 0; scnt[1][wib] = 0; scnt[2][wib] = 0; scnt[3][wib] = 0; }
    __syncthreads();
    WarpBuf<Change> bg{gbuf[MODE == kDelta ? wib : 0], &scnt[3][wib], a.chg, &a.st->n_chg};
    WarpBuf<int32_t> bs{sbuf[0][wib], &scnt[0][wib], a.small_out, &a.st->n_small};
    WarpBuf<int32_t> bm{sbuf[1][wib], &scnt[1][wib], a.med_out, &a.st->n_med};
    WarpBuf<ChunkItem> bc{cbuf[wib], &scnt[2][wib], a.chunk_out, &a.st->n_chunk};
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    LccTally tl;
    // masks of the first four label-multiplicity classes in registers (0 for
    // classes the template does not have: they never count)
    uint32_t cm[4];
#pragma unroll
    for (int c = 0; c < 4; c++) cm[c] = s.cls_mask[c];

    // (1) pieces of long rows: one warp per piece, combined through HubAcc;
    // the last piece to finish decides for the vertex.
    for (int64_t it = gwarp; it < n_chunk; it += nwarps) {
        ChunkItem ci = a.chunk_in[it];
        const uint32_t wv = __ldg(a.om_cur + ci.v);
        if (wv == 0u) {
            if (ci.c == 0 && lane == 0) {
                settle_dead<MODE>(a, ci.v);
                if (MODE == kDelta) clear_dirty(a, ci.v);
            }
            continue;
        }
        const int64_t rbeg = a.rp[ci.v], rend = a.rp[ci.v + 1];
        const int64_t beg = rbeg + (int64_t)ci.c * a.hub_deg;
        const int64_t end = min(rend, beg + (int64_t)a.hub_deg);
        if (lane == 0) { tl.rows += (unsigned long long)(end - beg); tl.alive += ci.c == 0; }
        Partial<MAXC> p;
        scan_row_warp<MAXC, DENSE>(beg, end, nbr_mask(wv, s) | a.eta_off, a.col, a.om_cur, a.ebits, s, p, tl.scanned, a.lab0,
                                   slm, cm, a.nw_cur, a.nw_bytes, a.elab, a.sparse != 0);
        p.U = grp_or<32>(p.U);
        p.nN = grp_sum<32>(p.nN);
        p.achg = grp_or<32>(p.achg);
#pragma unroll
        for (int c = 0; c < MAXC; c++) p.cnt[c] = grp_sum<32>(p.cnt[c]);
        HubAcc *h = a.acc + ci.slot;
        Change change{ci.v, wv};
        unsigned int ticket = 0;
        if (lane == 0) {
            if (p.U) atomicOr(&h->U, p.U);
            if (p.nN) atomicAdd(&h->nN, p.nN);
            if (p.achg) atomicOr(&h->flags, 1u);
#pragma unroll
            for (int c = 0; c < MAXC; c++)
                if (p.cnt[c]) atomicAdd(&h->cnt[c], p.cnt[c]);
            __threadfence();
            ticket = atomicAdd(&h->done, 1u);
        }
        ticket = __shfl_sync(FULL_MASK, ticket, 0);
        if (ticket == (unsigned int)(ci.nchunks - 1)) {
            __threadfence();
            Partial<MAXC> tot;
            tot.U = atomicOr(&h->U, 0u);
            tot.nN = atomicAdd(&h->nN, 0u);
            tot.achg = atomicOr(&h->flags, 0u);
#pragma unroll
            for (int c = 0; c < MAXC; c++) tot.cnt[c] = atomicAdd(&h->cnt[c], 0u);
            uint32_t keep = decide<MAXC>(wv, tot, s);
            if (lane == 0) {
                settle<MODE>(a, ci.v, wv, keep, tot.nN, rend - rbeg, true, tl);
                if (MODE == kDelta) clear_dirty(a, ci.v);
            }
            change.w = keep;
            if (keep != wv || tot.achg) tl.changed = 1u;
            __syncwarp();
            if (lane == 0) {
                h->U = 0u; h->nN = 0u; h->flags = 0u; h->done = 0u;
                for (int c = 0; c < MAXC; c++) h->cnt[c] = 0u;
            }
        }
        if (MODE == kDelta) bg.push(lane == 0 && change.w != wv, change);
        else bc.push(lane == 0, ci);
    }

    // (2) medium rows: one warp per vertex, taken 16 at a time: the list
    // entries, omega and row offsets of the next 16 vertices are loaded by 16
    // lanes at once, so each row walk starts from registers
    const int64_t n_mchunks = (n_med + MB - 1) / MB;
    for (int64_t ch = gwarp; ch < n_mchunks; ch += nwarps) {
        const int64_t idx = ch * MB + lane;
        int32_t vl = -1;
        uint32_t wl = 0u;
        int64_t bl = 0, el = 0;
        if (lane < MB && idx < n_med) {
            vl = a.med_in[idx];
            wl = __ldg(a.om_cur + vl);
            if (wl) { bl = a.rp[vl]; el = a.rp[vl + 1]; }
        }
        uint32_t wnew = wl;
        for (int j = 0; j < MB; j++) {
            const int32_t v = __shfl_sync(FULL_MASK, vl, j);
            if (v < 0) break;
            const uint32_t wv = __shfl_sync(FULL_MASK, wl, j);
            const int64_t beg = __shfl_sync(FULL_MASK, bl, j), end = __shfl_sync(FULL_MASK, el, j);
            if (wv) {
                if (lane == 0) { tl.rows += (unsigned long long)(end - beg); tl.alive++; }
                Partial<MAXC> p;
                scan_row_warp<MAXC, DENSE>(beg, end, nbr_mask(wv, s) | a.eta_off, a.col, a.om_cur, a.ebits, s, p, tl.scanned,
                                           a.lab0, slm, cm, a.nw_cur, a.nw_bytes, a.elab, a.sparse != 0);
                p.U = grp_or<32>(p.U);
                p.nN = grp_sum<32>(p.nN);
                p.achg = grp_or<32>(p.achg);
#pragma unroll
                for (int c = 0; c < MAXC; c++) p.cnt[c] = grp_sum<32>(p.cnt[c]);
                const uint32_t keep = decide<MAXC>(wv, p, s);
                if (keep != wv || p.achg) tl.changed = 1u;
                if (lane == 0) settle<MODE>(a, v, wv, keep, p.nN, end - beg, end - beg > a.hub_deg, tl);
                if (lane == j) wnew = keep;
            } else if (lane == 0) {
                settle_dead<MODE>(a, v);
            }
        }
        // the chunk's vertices that were active at the start of the round (delta:
        // those whose omega changes), in one push
        if (MODE == kDelta) {
            if (vl >= 0) clear_dirty(a, vl);
            bg.push(vl >= 0 && wnew != wl, Change{vl, wnew});
        } else {
            bm.push(vl >= 0 && wl != 0u, vl);
        }
    }

    // (3) short rows: 32 vertices per warp batch, entries streamed flat
    short_rows<MAXC, MODE>(a, s, slm, cm, srows[wib], gwarp, nwarps, n_small, bs, bg, tl);

    // what is left in the warps' buffers goes out once per block
    __syncthreads();
    if (MODE == kDelta) {
        block_flush(bg, &scnt[3][0], wib);
    } else {
        block_flush(bs, &scnt[0][0], wib);
        block_flush(bm, &scnt[1][0], wib);
        block_flush(bc, &scnt[2][0], wib);
    }
    add_totals(tl, totals, a.st);
}

// -------------------------------------------------------------------------
// The first round of templates with at most four multiplicity classes, and their
// later ones where the rows are huge and omega fits a byte (kHugeRows);
// k_lcc_round above serves the others.
//
// A lane takes four consecutive entries per step: their edge bits are a nibble
// of a bitmap word, their columns one 16-byte load, and the four gathers that
// follow are in flight together.  A neighbour's omega arrives as a byte (its
// label in the first round, its narrow omega later) that indexes a table of
// (omega, one byte per class it meets), so class counts are one addition.
// Rows are walked by as many lanes as they fill: up to 16 entries by their own
// lane, up to 64 by 8 lanes (four rows side by side), longer ones by the warp.
//
// The rounds are bound by the latency of dependent loads (list entry, omega and
// offsets, bits, columns, neighbours), not by bytes: a warp that walked one row
// after the other, 32 entries a step, spent 3 to 4 us on a row of 200 entries.
// long_rows keeps the bits of the next two stretches, the columns of the next
// step and the gathers of the current one in flight, across rows.
//
// The first round of a fresh prune needs labels only (omega_0 is the mask of a
// vertex's label), so it is one with the initialisation (Alg. 3): k_first_round
// takes the vertices in id order, with no list written and read back, decides
// short rows and lists the longer ones for k_rows.  It writes omega as the
// round leaves it, in both buffers, and lists survivors only.
// -------------------------------------------------------------------------

// Where a neighbour's omega comes from: its label in entry order (first round,
// graphs that have the entry labels), its label (first round), its 1-byte
// omega, or omega itself (allocation-free LCC, which keeps no narrow copy).
constexpr int kByEntry = 0, kByLabel = 1, kByByte = 2, kByWord = 3;
constexpr int kFirst = 3;                    // a round's MODE, beside kFull and kDelta

// Entries in the initially active rows from which k_rows takes the rounds after
// the first, where omega fits a byte (templates of up to 8 vertices).  ms of
// these rounds with k_rows and with k_lcc_round, Zipf labels, 30 entries a vertex:
//   vertices               8M (142M entries)   32M (570M entries)
//   8, two classes         1.09   1.41         4.12   5.13
//   8, three classes       0.81   1.05         2.83   3.85
//   7, three classes       0.92   1.00         3.22   3.52
//   5, no class            0.66   0.68         2.54   2.44
//   9, two classes         1.36   1.27         5.62   5.00
//   12, three classes      1.57   1.50         6.77   5.71
// 13 templates of up to 8 vertices at 32M: 0.92 to 1.36 times as fast, 1.12 on
// average.  A wider omega leaves k_rows without its table by bytes: slower at
// every size.  The line itself is not sharp: at 36M entries (2M vertices) 0.45 against 0.52
// with two classes and 0.21 against 0.17 without (8M entries); degree labels, 3M
// vertices (40M entries), 0.18 against 0.16; on 64K vertices a round takes 7.6
// against 6.3 us (one chain of latencies, which k_lcc_round keeps shorter).
constexpr int64_t kHugeRows = (int64_t)1 << 28;
// ... below which k_first_round walks the longer rows too, with no second
// kernel over a list of them (64K vertices: 31 against 41 us; 3M: 216 against
// 197).
constexpr int64_t kInlineRows = (int64_t)1 << 22;
// Entries in the live rows from which later rounds evaluate changes only
// (Pipeline::use_deltas).
constexpr int64_t kDeltaRows = (int64_t)1 << 22;

struct RowArgs {
    int64_t n, m;                 // m: columns that may be read four at a time
    const int64_t *rp;
    const int32_t *col;
    int col_vec;                  // col is 16-byte aligned
    const uint8_t *lab;
    const uint8_t *elab;          // readable up to entry m + 15
    const uint32_t *om;           // omega the round reads (kFull, kDelta), and its narrow copy
    const void *nw;
    int nw_bytes;
    uint32_t *om_out[2];          // omega the round writes: [0] (kFull), both (kFirst)
    void *nw_out[2];
    uint32_t *ebits;
    int guard;                    // kFirst: a word follows the bitmap's last
    int inline_long;              // kFirst: k_first_round walks rows of up to 1024 entries itself
    uint32_t *deg;                // entries each evaluated vertex keeps (nullable)
    uint32_t *dirty;
    Change *chg;
    ChangePiece *chg_piece;
    const int32_t *small_in, *med_in;
    const ChunkItem *chunk_in;
    const RoundStats *sizes;      // sizes of these lists (NULL: the next three)
    int64_t n_small, n_med, n_chunk;
    const RoundStats *gate;       // the round runs only if these counters say `changed` (nullable)
    int32_t *small_out, *med_out;
    ChunkItem *chunk_out;
    int32_t *first_med;           // kFirst: the rows k_first_round leaves to k_rows, sizes in first_sizes
    ChunkItem *first_chunk;
    RoundStats *first_sizes;
    HubAcc *acc;
    RoundStats *st;
    int hub_deg, short_max;
    uint32_t eta_off;
    LabelMask lm;
};

constexpr int kLaneRow = 16, kGroupRow = 64, kWarpRow = 1024;   // row lengths of the three paths

struct RowAcc { uint32_t U = 0, cp = 0, nN = 0; };   // union, class counts (four bytes), kept entries

// byte -> (omega, 1 in the byte of every class it meets)
template <int F>
__device__ __forceinline__ void make_table(uint2 *lut, const SmemTmpl &s, const LabelMask &lm) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        const uint32_t w = (F == kByEntry || F == kByLabel) ? lm.m[i] : (uint32_t)i;
        uint32_t pack = 0;
        for (int c = 0; c < 4 && c < s.n_cls; c++) pack |= (w & s.cls_mask[c]) ? 1u << (8 * c) : 0u;
        lut[i] = make_uint2(w, pack);
    }
}

// Columns of the entries e + j with bit j of nib set (e a multiple of 4).
__device__ __forceinline__ void quad_cols(const RowArgs &a, int64_t e, uint32_t nib, int32_t (&u)[4]) {
    u[0] = u[1] = u[2] = u[3] = 0;
    if (!nib) return;
    if (a.col_vec && e + 4 <= a.m) {
        const int4 c = __ldcs((const int4 *)(a.col + e));
        u[0] = c.x; u[1] = c.y; u[2] = c.z; u[3] = c.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; j++)
            if ((nib >> j) & 1u) u[j] = __ldcs(a.col + e + j);
    }
}

// What the four entries' neighbours hold: four bytes, or four words.
template <int F> struct Quad { uint32_t v[F == kByWord ? 4 : 1]; };

template <int F>
__device__ __forceinline__ Quad<F> quad_gather(const RowArgs &a, uint32_t nib, const int32_t (&u)[4]) {
    Quad<F> q;
    uint32_t x[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        x[j] = 0u;
        if ((nib >> j) & 1u) {
            if (F == kByLabel) x[j] = __ldg(a.lab + u[j]);
            else if (F == kByByte) x[j] = __ldg((const uint8_t *)a.nw + u[j]);
            else x[j] = gather_om(a.om, a.nw, a.nw_bytes, u[j]);
        }
    }
    if constexpr (F == kByWord) {
#pragma unroll
        for (int j = 0; j < 4; j++) q.v[j] = x[j];
    } else {
        q.v[0] = x[0] | (x[1] << 8) | (x[2] << 16) | (x[3] << 24);
    }
    return q;
}

// Four entries (those of nib): the kept ones as a nibble.  Entries without a
// bit hold an empty omega, except where labels come from a stream (kByEntry).
template <int MAXC, int F>
__device__ __forceinline__ uint32_t quad_take(const Quad<F> &q, uint32_t nib, uint32_t nbr, const uint2 *lut,
                                              const uint32_t (&cm)[4], RowAcc &A, LccTally &tl) {
    uint32_t keep = 0, live = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        uint32_t w, pack = 0u;
        if constexpr (F == kByWord) {
            w = q.v[j];
#pragma unroll
            for (int c = 0; c < MAXC; c++) pack |= (w & cm[c]) ? 1u << (8 * c) : 0u;
        } else {
            const uint2 x = lut[(q.v[0] >> (8 * j)) & 255u];
            w = x.x;
            pack = x.y;
            if ((F == kByEntry || F == kByLabel) && !((nib >> j) & 1u)) w = 0u;
        }
        if (F != kByByte) live += w != 0u;
        if (w & nbr) {
            A.U |= w;
            if (MAXC > 0) A.cp += pack;
            keep |= 1u << j;
        }
    }
    if (F == kByByte)                        // bytes that are not zero
        live = __popc((((q.v[0] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | q.v[0]) & 0x80808080u);
    const uint32_t k = __popc(keep);
    A.nN += k;
    tl.scanned += live;
    if (k != live) tl.changed = 1u;          // eta eliminates a live entry
    return keep;
}

// Bits of the word wi that belong to the row [beg, end).
__device__ __forceinline__ uint32_t word_range(int64_t wi, int64_t beg, int64_t end) {
    const int64_t e0 = wi << 5;
    if (e0 >= end || e0 + 32 <= beg) return 0u;
    uint32_t in = ~0u;
    if (e0 < beg) in &= ~0u << (uint32_t)(beg - e0);
    if (end - e0 < 32) in &= (1u << (uint32_t)(end - e0)) - 1u;
    return in;
}

// The row's bits `had` of word wi shrink to `kept`.  The bit goes with failing
// entries and with those whose other end is inactive already.
__device__ __forceinline__ void store_bits(uint32_t *ebits, int64_t wi, uint32_t in, uint32_t had, uint32_t kept) {
    if (!(had & ~kept)) return;
    if (in == ~0u) ebits[wi] = kept;
    else atomicAnd(&ebits[wi], ~(had & ~kept));          // shared with a neighbouring row
}

// The row's active bits in word wi.
template <int MODE>
__device__ __forceinline__ uint32_t row_word(const RowArgs &a, int64_t wi, int64_t beg, int64_t end) {
    const uint32_t in = word_range(wi, beg, end);
    if (MODE == kFirst) return in;
    return in ? a.ebits[wi] & in : 0u;
}

template <int MAXC>
__device__ __forceinline__ void unpack_classes(uint32_t cp, Partial<MAXC> &p) {
#pragma unroll
    for (int c = 0; c < MAXC; c++) p.cnt[c] += (cp >> (8 * c)) & 255u;
}

// Rows of up to 64 entries, one vertex per lane (wv = 0: none): omega' and the
// number of entries kept.  All lanes call.
template <int MAXC, int MODE, int F>
__device__ __forceinline__ void short_batch(const RowArgs &a, const SmemTmpl &s, const uint2 *lut,
                                            const uint32_t (&cm)[4], uint32_t wv, uint32_t nbr, int64_t beg, int64_t end,
                                            uint32_t &keep, uint32_t &kept, LccTally &tl) {
    const int lane = (int)lane_id();
    const int64_t len = end - beg;
    // (1) up to 16 entries, by the lane itself
    if (wv && len > 0 && len <= kLaneRow) {
        RowAcc A;
        const int64_t wi = beg >> 5;
        const uint32_t sh = (uint32_t)(beg & 31), in = (1u << (int)len) - 1u;
        uint32_t had = in;                               // active entries, relative to beg
        if (MODE != kFirst) {
            had = a.ebits[wi] >> sh;
            if (sh + (uint32_t)len > 32u) had |= a.ebits[wi + 1] << (32 - sh);
            had &= in;
        }
        uint32_t kb = 0;
        const int64_t e0 = beg & ~(int64_t)3;
        const int lead = (int)(beg - e0);
        const uint32_t nibs = had << lead;               // by groups of four entries from e0
        if (F == kByEntry) {
            uint32_t labs[5];
#pragma unroll
            for (int i = 0; i < 5; i++)
                labs[i] = e0 + 4 * i < end ? __ldcs((const unsigned int *)(a.elab + e0 + 4 * i)) : 0u;
#pragma unroll
            for (int i = 0; i < 5; i++) {
                Quad<F> q;
                q.v[0] = labs[i];
                const uint32_t nib = (nibs >> (4 * i)) & 15u;
                if (nib) kb |= quad_take<MAXC, F>(q, nib, nbr, lut, cm, A, tl) << (4 * i);
            }
        } else {
            int32_t u[4], nx[4];
            quad_cols(a, e0, nibs & 15u, u);
            for (int i = 0; (nibs >> (4 * i)) != 0u; i++) {
                const uint32_t nib = (nibs >> (4 * i)) & 15u;
                const Quad<F> q = quad_gather<F>(a, nib, u);
                quad_cols(a, e0 + 4 * (i + 1), (nibs >> (4 * i + 4)) & 15u, nx);
                kb |= quad_take<MAXC, F>(q, nib, nbr, lut, cm, A, tl) << (4 * i);
#pragma unroll
                for (int j = 0; j < 4; j++) u[j] = nx[j];
            }
        }
        kb >>= lead;
        Partial<MAXC> p;
        p.U = A.U;
        p.nN = A.nN;
        unpack_classes<MAXC>(A.cp, p);
        keep = decide<MAXC>(wv, p, s);
        kept = A.nN;
        // the bits of a vertex that dies: no round reads them again
        if (keep) clear_rel(a.ebits, beg, had & ~kb);
    }
    // (2) up to 64, four rows at a time, eight lanes each
    for (uint32_t todo = __ballot_sync(FULL_MASK, wv && len > kLaneRow && len <= kGroupRow); todo;) {
        int src[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            src[i] = todo ? __ffs(todo) - 1 : -1;
            todo &= todo - 1u;
        }
        const int g = lane >> 3, j = lane & 7;
        const int from = g == 0 ? src[0] : g == 1 ? src[1] : g == 2 ? src[2] : src[3];
        const int f = from < 0 ? 0 : from;
        const int64_t gb = __shfl_sync(FULL_MASK, beg, f), ge0 = __shfl_sync(FULL_MASK, end, f);
        const int64_t ge = from < 0 ? gb : ge0;          // an empty group: no entry is in range
        const uint32_t gn = __shfl_sync(FULL_MASK, nbr, f), gw = __shfl_sync(FULL_MASK, wv, f);
        const int64_t w0 = gb >> 5;
        uint32_t had[3], word[3];
        Quad<F> q[3];
        RowAcc A;
#pragma unroll
        for (int k = 0; k < 3; k++) had[k] = row_word<MODE>(a, w0 + k, gb, ge);
        if (F == kByEntry) {
#pragma unroll
            for (int k = 0; k < 3; k++)
                q[k].v[0] = (had[k] >> (4 * j)) & 15u
                                ? __ldcs((const unsigned int *)(a.elab + ((w0 + k) << 5) + 4 * j)) : 0u;
        } else {
            int32_t u[3][4];
#pragma unroll
            for (int k = 0; k < 3; k++) quad_cols(a, ((w0 + k) << 5) + 4 * j, (had[k] >> (4 * j)) & 15u, u[k]);
#pragma unroll
            for (int k = 0; k < 3; k++) q[k] = quad_gather<F>(a, (had[k] >> (4 * j)) & 15u, u[k]);
        }
#pragma unroll
        for (int k = 0; k < 3; k++)
            word[k] = quad_take<MAXC, F>(q[k], (had[k] >> (4 * j)) & 15u, gn, lut, cm, A, tl) << (4 * j);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
            for (int k = 0; k < 3; k++) word[k] |= __shfl_xor_sync(FULL_MASK, word[k], o);
            A.U |= __shfl_xor_sync(FULL_MASK, A.U, o);
            A.nN += __shfl_xor_sync(FULL_MASK, A.nN, o);
            if (MAXC > 0) A.cp += __shfl_xor_sync(FULL_MASK, A.cp, o);   // at most 64 per byte
        }
        Partial<MAXC> p;
        p.U = A.U;
        p.nN = A.nN;
        unpack_classes<MAXC>(A.cp, p);
        const uint32_t gk = decide<MAXC>(gw, p, s);
        if (gk && from >= 0 && j < 3)
            store_bits(a.ebits, w0 + j, word_range(w0 + j, gb, ge), j == 0 ? had[0] : j == 1 ? had[1] : had[2],
                       j == 0 ? word[0] : j == 1 ? word[1] : word[2]);
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const uint32_t k = __shfl_sync(FULL_MASK, gk, 8 * i), c = __shfl_sync(FULL_MASK, A.nN, 8 * i);
            if (lane == src[i]) { keep = k; kept = c; }
        }
    }
}

// Row sums over the warp.
template <int MAXC>
__device__ __forceinline__ void reduce_row(const RowAcc &A, Partial<MAXC> &p, int n_cls) {
    p.U = __reduce_or_sync(FULL_MASK, A.U);
    p.nN = __reduce_add_sync(FULL_MASK, A.nN);
#pragma unroll
    for (int c = 0; c < MAXC; c++)
        if (c < n_cls) p.cnt[c] = __reduce_add_sync(FULL_MASK, p.cnt[c] + ((A.cp >> (8 * c)) & 255u));
}

// Rows (or pieces of rows) of any length, one per lane of `rows`, walked by the
// warp one after the other; done(j, sums) is called by all lanes after the row
// of lane j.  Stretches of 1024 entries (a bitmap word per lane), steps of 128
// entries that hold an active one.
template <int MAXC, int MODE, int F, typename D>
__device__ __forceinline__ void long_rows(const RowArgs &a, int n_cls, const uint2 *lut, const uint32_t (&cm)[4],
                                          uint32_t rows,
                                          int64_t beg, int64_t end, uint32_t nbr, LccTally &tl, D &&done) {
    if (!rows) return;
    const int lane = (int)lane_id();
    const int first = __ffs(rows) - 1;
    auto next_row = [&](int j) {                     // the lane after j that has a row (32: none)
        const uint32_t rest = j < 31 ? rows >> (j + 1) << (j + 1) : 0u;
        return rest ? __ffs(rest) - 1 : 32;
    };
    RowAcc A;
    Partial<MAXC> p;
    int since = 0;                                   // steps since the class bytes were emptied
    auto finish = [&](int j) {
        Partial<MAXC> sum = p;
        reduce_row<MAXC>(A, sum, n_cls);
        done(j, sum);
        A = RowAcc();
        p = Partial<MAXC>();
        since = 0;
    };
    auto spill_classes = [&](int steps, int most) {
        since += steps;
        if (MAXC > 0 && since >= most) {             // before a byte can overflow
            unpack_classes<MAXC>(A.cp, p);
            A.cp = 0;
            since = 0;
        }
    };
    if constexpr (F == kByEntry) {
        // the labels are one contiguous stream: 16 per lane and step
        int j = first;
        int64_t b = __shfl_sync(FULL_MASK, beg, j), e = __shfl_sync(FULL_MASK, end, j);
        int64_t base = b & ~(int64_t)31;
        auto load = [&](int64_t at, int64_t rb, int64_t re) {
            const int64_t x = at + 16 * lane;
            return x < re && x + 16 > rb ? __ldcs((const uint4 *)(a.elab + x)) : make_uint4(0, 0, 0, 0);
        };
        uint4 nx = load(base, b, e);
        while (j < 32) {
            const uint4 cur = nx;
            const int64_t cb = b, ce = e, at = base;
            const int cj = j;
            base += 512;
            if (base >= e) {
                j = next_row(j);
                if (j < 32) {
                    b = __shfl_sync(FULL_MASK, beg, j);
                    e = __shfl_sync(FULL_MASK, end, j);
                    base = b & ~(int64_t)31;
                }
            }
            if (j < 32) nx = load(base, b, e);
            const uint32_t rn = __shfl_sync(FULL_MASK, nbr, cj);
            const int64_t wi = (at >> 5) + (lane >> 1);
            const uint32_t in = word_range(wi, cb, ce);
            const uint32_t half = (in >> (16 * (lane & 1))) & 0xFFFFu;
            uint32_t kept = 0;
            if (half) {
                const uint32_t x[4] = {cur.x, cur.y, cur.z, cur.w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    Quad<F> q;
                    q.v[0] = x[i];
                    kept |= quad_take<MAXC, F>(q, (half >> (4 * i)) & 15u, rn, lut, cm, A, tl) << (4 * i);
                }
            }
            kept <<= 16 * (lane & 1);
            kept |= __shfl_xor_sync(FULL_MASK, kept, 1);
            if (!(lane & 1)) store_bits(a.ebits, wi, in, in, kept);
            spill_classes(1, 15);
            if (j != cj) finish(cj);
        }
        return;
    } else {
        // offsets inside a row count from its first bitmap word whose index is a
        // multiple of 4, so that they fit 32 bits and a lane's four columns
        // are 16-byte aligned
        const int64_t my_w0 = (beg >> 7) << 2;
        const int my_lo = (int)(beg - (my_w0 << 5)), my_hi = (int)(end - (my_w0 << 5));
        struct Seg { int j, at, hi; uint32_t word; };        // row, first entry of the stretch, row end
        auto read = [&](Seg &g) {
            g.word = 0u;
            if (g.j >= 32) return;
            g.hi = __shfl_sync(FULL_MASK, my_hi, g.j);
            const int lo = __shfl_sync(FULL_MASK, my_lo, g.j);
            const int64_t w0 = __shfl_sync(FULL_MASK, my_w0, g.j);
            const int e = g.at + 32 * lane;
            if (e >= g.hi || e + 32 <= lo) return;
            uint32_t in = ~0u;
            if (e < lo) in &= ~0u << (lo - e);
            if (g.hi - e < 32) in &= (1u << (g.hi - e)) - 1u;
            g.word = MODE == kFirst ? in : a.ebits[w0 + (e >> 5)] & in;
        };
        auto after = [&](const Seg &g) {
            Seg n{g.j, g.at + 1024, g.hi, 0u};
            if (n.at >= g.hi) { n.j = next_row(g.j); n.at = 0; }
            return n;
        };
        auto steps = [&](const Seg &g) {             // bit 4k: step k holds an active entry
            uint32_t b = __ballot_sync(FULL_MASK, g.word != 0u);
            b |= b >> 1;
            b |= b >> 2;
            return b & 0x11111111u;
        };
        Seg cur{first, 0, 0, 0u};
        read(cur);
        Seg n1 = after(cur);
        read(n1);
        uint32_t u_nib = 0;                          // the step whose columns are loaded
        int32_t u[4];
        bool have = false;
        auto columns = [&](const Seg &g, int k4) {
            const uint32_t wd = __shfl_sync(FULL_MASK, g.word, k4 + (lane >> 3));
            const int64_t w0 = __shfl_sync(FULL_MASK, my_w0, g.j);
            u_nib = (wd >> (4 * (lane & 7))) & 15u;
            quad_cols(a, (w0 << 5) + (g.at + 32 * k4 + 4 * lane), u_nib, u);
            have = true;
        };
        for (;;) {
            Seg n2 = after(n1);
            read(n2);
            const uint32_t rn = __shfl_sync(FULL_MASK, nbr, cur.j);
            for (uint32_t t = steps(cur); t;) {
                const int k4 = __ffs(t) - 1;
                t &= t - 1u;
                if (!have) columns(cur, k4);
                const uint32_t nib = u_nib;
                const Quad<F> q = quad_gather<F>(a, nib, u);
                have = false;
                if (t) {
                    columns(cur, __ffs(t) - 1);
                } else {
                    const uint32_t tn = steps(n1);
                    if (tn) columns(n1, __ffs(tn) - 1);
                }
                const uint32_t keep = quad_take<MAXC, F>(q, nib, rn, lut, cm, A, tl);
                if (__any_sync(FULL_MASK, keep != nib)) {
                    uint32_t kept = keep << (4 * (lane & 7));
                    kept |= __shfl_xor_sync(FULL_MASK, kept, 1);
                    kept |= __shfl_xor_sync(FULL_MASK, kept, 2);
                    kept |= __shfl_xor_sync(FULL_MASK, kept, 4);
                    const uint32_t had = __shfl_sync(FULL_MASK, cur.word, k4 + (lane >> 3));
                    const int lo = __shfl_sync(FULL_MASK, my_lo, cur.j);
                    const int64_t w0 = __shfl_sync(FULL_MASK, my_w0, cur.j);
                    if ((lane & 7) == 0 && (had & ~kept)) {
                        const int e = cur.at + 32 * (k4 + (lane >> 3));
                        uint32_t *p_word = a.ebits + w0 + (e >> 5);
                        if (e >= lo && e + 32 <= cur.hi) *p_word = kept;
                        else atomicAnd(p_word, ~(had & ~kept));          // shared with a neighbouring row
                    }
                }
                spill_classes(1, 60);
            }
            if (n1.j != cur.j) finish(cur.j);
            if (n1.j >= 32) break;
            cur = n1;
            n1 = n2;
        }
    }
}

// What a round decided for the lane's vertex v: its omega was wv and is now
// `keep`, `kept` of the `len` entries of its row stay active.
template <int MODE>
__device__ __forceinline__ void settle_row(const RowArgs &a, int32_t v, uint32_t wv, uint32_t keep, uint32_t kept,
                                           int64_t len, LccTally &tl) {
    tl.alive++;
    tl.rows += (unsigned long long)len;
    if (keep) { tl.kept += kept; tl.rows_next += (unsigned long long)len; }
    else tl.died++;
    if (keep != wv) tl.changed = 1u;
    if (MODE == kDelta) {
        tl.old_kept += a.deg[v];
        if (keep == 0u) tl.died_rows += (unsigned long long)len;
        if (keep != wv && len > a.hub_deg) {
            const unsigned int np = (unsigned int)((len + a.hub_deg - 1) / a.hub_deg);
            const unsigned int b = atomicAdd(&a.st->n_chg_piece, np);
            for (unsigned int c = 0; c < np; c++) a.chg_piece[b + c] = ChangePiece{v, (int32_t)c};
        }
    }
    if (a.deg) a.deg[v] = keep ? kept : 0u;
}

// omega' of the lane's vertex (a vertex that was inactive gets its 0 again: the
// buffer may still hold what it had before it died).
template <int MODE>
__device__ __forceinline__ void write_omega(const RowArgs &a, int64_t v, uint32_t keep) {
    if (MODE == kDelta) return;
    a.om_out[0][v] = keep;
    store_narrow(a.nw_out[0], a.nw_bytes, v, keep);
    if (MODE == kFirst) {
        a.om_out[1][v] = keep;
        store_narrow(a.nw_out[1], a.nw_bytes, v, keep);
    }
}

// List a vertex for the next round by its row length (all lanes call).
__device__ __forceinline__ void list_row(const RowArgs &a, bool want, int32_t v, int64_t len, WarpBuf<int32_t> &bs,
                                         WarpBuf<int32_t> &bm) {
    const int64_t small_max = a.hub_deg < a.short_max ? a.hub_deg : a.short_max;
    bs.push(want && len <= small_max, v);
    bm.push(want && len > small_max && len <= a.hub_deg, v);
    if (want && len > a.hub_deg) {
        const int nch = (int)((len + a.hub_deg - 1) / a.hub_deg);
        const int slot = (int)atomicAdd(&a.st->n_hub_slots, 1u);
        const unsigned int base = atomicAdd(&a.st->n_chunk, (unsigned int)nch);
        for (int c = 0; c < nch; c++) a.chunk_out[base + c] = ChunkItem{v, c, slot, nch};
    }
}

// The first round: every vertex in id order.  Rows of more than 64 entries are
// left to k_rows (those past max(hub_deg, 1024) in pieces of hub_deg).
template <int MAXC, int F>
__global__ void __launch_bounds__(256, 4)
k_first_round(RowArgs a, DevTmpl t) {
    __shared__ SmemTmpl s;
    __shared__ uint2 lut[256];
    __shared__ int32_t sbuf[3][8][32];
    __shared__ int scnt[3][8];
    __shared__ unsigned long long totals[9];
    if (threadIdx.x < 9) totals[threadIdx.x] = 0ull;
    load_tmpl(s, t);
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane < 3) scnt[lane][wib] = 0;
    __syncthreads();
    make_table<F>(lut, s, a.lm);
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // no entries past m: the padding bits of the last word (and a guard word
        // after it, where the bitmap has one) stay 0
        if (a.m & 31) atomicAnd(&a.ebits[a.m >> 5], (1u << (uint32_t)(a.m & 31)) - 1u);
        if (a.guard) a.ebits[(a.m + 31) >> 5] = 0u;
    }
    WarpBuf<int32_t> bs{sbuf[0][wib], &scnt[0][wib], a.small_out, &a.st->n_small};
    WarpBuf<int32_t> bm{sbuf[1][wib], &scnt[1][wib], a.med_out, &a.st->n_med};
    WarpBuf<int32_t> bl{sbuf[2][wib], &scnt[2][wib], a.first_med, &a.first_sizes->n_med};
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // small graphs: fewer than 32 vertices per warp, so that every warp has some
    const int per = (int)max((int64_t)1, min((int64_t)32, a.n / nwarps));
    const int64_t in_warp = max((int64_t)kWarpRow, (int64_t)a.hub_deg), stride = nwarps * per;
    uint32_t cm[4];
#pragma unroll
    for (int c = 0; c < 4; c++) cm[c] = s.cls_mask[c];
    LccTally tl;
    // the labels of the next batch but one and the offsets of the next one are
    // loaded while a batch is walked
    auto label_mask = [&](int64_t v) { return lane < per && v < a.n ? lut[a.lab[v]].x : 0u; };
    auto offsets = [&](int64_t v, uint32_t w, int64_t &b, int64_t &e) {
        b = e = 0;
        if (w) { b = a.rp[v]; e = a.rp[v + 1]; }
    };
    int64_t v = gwarp * per + lane;
    uint32_t w1 = label_mask(v), w2 = label_mask(v + stride);
    int64_t b1, e1;
    offsets(v, w1, b1, e1);
    for (int64_t v0 = gwarp * per; v0 < a.n; v0 += stride, v += stride) {
        const uint32_t wv = w1;
        const int64_t beg = b1, end = e1, len = end - beg;
        w1 = w2;
        offsets(v + stride, w1, b1, e1);
        w2 = label_mask(v + 2 * stride);
        uint32_t keep = 0u, kept = 0u;
        const uint32_t nbr = wv ? nbr_mask(wv, s) | a.eta_off : 0u;
        short_batch<MAXC, kFirst, F>(a, s, lut, cm, wv, nbr, beg, end, keep, kept, tl);
        const bool later = a.inline_long ? len > in_warp : len > kGroupRow;
        if (a.inline_long) {
            Partial<MAXC> sums;
            const bool longer = len > kGroupRow && !later;
            long_rows<MAXC, kFirst, F>(a, s.n_cls, lut, cm, __ballot_sync(FULL_MASK, longer), beg, end, nbr, tl,
                                       [&](int j, const Partial<MAXC> &p) { if (lane == j) sums = p; });
            if (longer) {
                keep = decide<MAXC>(wv, sums, s);
                kept = sums.nN;
            }
        }
        bl.push(later && len <= in_warp, (int32_t)v);
        if (len > in_warp) {
            const int nch = (int)((len + a.hub_deg - 1) / a.hub_deg);
            const int slot = (int)atomicAdd(&a.first_sizes->n_hub_slots, 1u);
            const unsigned int base = atomicAdd(&a.first_sizes->n_chunk, (unsigned int)nch);
            for (int c = 0; c < nch; c++) a.first_chunk[base + c] = ChunkItem{(int32_t)v, c, slot, nch};
        }
        if (!later && lane < per && v < a.n) {
            if (wv) settle_row<kFirst>(a, (int32_t)v, wv, keep, kept, len, tl);
            write_omega<kFirst>(a, v, keep);
        }
        list_row(a, keep != 0u, (int32_t)v, len, bs, bm);
    }
    __syncthreads();
    block_flush(bs, &scnt[0][0], wib);
    block_flush(bm, &scnt[1][0], wib);
    block_flush(bl, &scnt[2][0], wib);
    add_totals(tl, totals, a.st);
}

// A round over lists: all active vertices (kFull), those near a change
// (kDelta), or the long rows of the first round (kFirst).
template <int MAXC, int MODE, int F>
__global__ void __launch_bounds__(256, 4)
k_rows(RowArgs a, DevTmpl t) {
    if (a.gate && a.gate->changed == 0u) {
        if (blockIdx.x == 0 && threadIdx.x == 0) a.st->skipped = 1u;
        return;
    }
    const int64_t n_small = MODE == kFirst ? 0 : (a.sizes ? (int64_t)a.sizes->n_small : a.n_small);
    const int64_t n_med = a.sizes ? (int64_t)a.sizes->n_med : a.n_med;
    const int64_t n_chunk = a.sizes ? (int64_t)a.sizes->n_chunk : a.n_chunk;
    if (n_small + n_med + n_chunk == 0) return;
    __shared__ SmemTmpl s;
    __shared__ uint2 lut[F == kByWord ? 1 : 256];
    __shared__ int32_t sbuf[2][8][32];
    __shared__ ChunkItem cbuf[MODE == kFull ? 8 : 1][32];
    __shared__ Change gbuf[MODE == kDelta ? 8 : 1][32];
    __shared__ int scnt[4][8];
    __shared__ unsigned long long totals[9];
    if (threadIdx.x < 9) totals[threadIdx.x] = 0ull;
    load_tmpl(s, t);
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane < 4) scnt[lane][wib] = 0;
    __syncthreads();
    if (F != kByWord) make_table<F>(lut, s, a.lm);
    __syncthreads();
    WarpBuf<int32_t> bs{sbuf[0][wib], &scnt[0][wib], a.small_out, &a.st->n_small};
    WarpBuf<int32_t> bm{sbuf[1][wib], &scnt[1][wib], a.med_out, &a.st->n_med};
    WarpBuf<ChunkItem> bc{cbuf[MODE == kFull ? wib : 0], &scnt[2][wib], a.chunk_out, &a.st->n_chunk};
    WarpBuf<Change> bg{gbuf[MODE == kDelta ? wib : 0], &scnt[3][wib], a.chg, &a.st->n_chg};
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    uint32_t cm[4];
#pragma unroll
    for (int c = 0; c < 4; c++) cm[c] = s.cls_mask[c];
    LccTally tl;
    auto omega_of = [&](int32_t v) { return MODE == kFirst ? lut[a.lab[v]].x : __ldg(a.om + v); };
    auto clear = [&](int32_t v) { atomicAnd(&a.dirty[v >> 5], ~(1u << (v & 31))); };
    // few rows: fewer per warp and batch, so that every warp has some
    auto batch = [&](int64_t rows, int64_t share) { return (int)max((int64_t)1, min((int64_t)32, rows / (share * nwarps))); };

    // (1) pieces of long rows, combined through HubAcc; a row's last piece decides
    const int pc = batch(n_chunk, 4);
    for (int64_t b0 = gwarp * pc; b0 < n_chunk; b0 += nwarps * pc) {
        const int cnt = (int)min((int64_t)pc, n_chunk - b0);
        ChunkItem ci{0, 0, 0, 0};
        uint32_t wv = 0u;
        int64_t rb = 0, re = 0, beg = 0, end = 0;
        if (lane < cnt) {
            ci = a.chunk_in[b0 + lane];
            wv = omega_of(ci.v);
            rb = a.rp[ci.v];
            re = a.rp[ci.v + 1];
            if (wv) {
                beg = rb + (int64_t)ci.c * a.hub_deg;
                end = min(re, beg + (int64_t)a.hub_deg);
            } else if (ci.c == 0) {
                write_omega<MODE>(a, ci.v, 0u);
                if (MODE == kFull && a.deg) a.deg[ci.v] = 0u;
                if (MODE == kDelta) clear(ci.v);
            }
        }
        const uint32_t nbr = wv ? nbr_mask(wv, s) | a.eta_off : 0u;
        // the lanes keep their pieces' sums and combine them side by side: one
        // fence and ticket after the other cost more than the rows
        Partial<MAXC> mine;
        long_rows<MAXC, MODE, F>(a, s.n_cls, lut, cm, __ballot_sync(FULL_MASK, wv != 0u), beg, end, nbr, tl,
                                 [&](int j, const Partial<MAXC> &p) { if (lane == j) mine = p; });
        uint32_t now = wv;                            // omega', if the lane's piece was the row's last
        if (wv) {
            HubAcc *h = a.acc + ci.slot;
            if (mine.U) atomicOr(&h->U, mine.U);
            if (mine.nN) atomicAdd(&h->nN, mine.nN);
#pragma unroll
            for (int c = 0; c < MAXC; c++)
                if (mine.cnt[c]) atomicAdd(&h->cnt[c], mine.cnt[c]);
            __threadfence();
            if (atomicAdd(&h->done, 1u) == (unsigned int)(ci.nchunks - 1)) {
                __threadfence();
                Partial<MAXC> tot;
                tot.U = atomicOr(&h->U, 0u);
                tot.nN = atomicAdd(&h->nN, 0u);
#pragma unroll
                for (int c = 0; c < MAXC; c++) tot.cnt[c] = atomicAdd(&h->cnt[c], 0u);
                now = decide<MAXC>(wv, tot, s);
                settle_row<MODE>(a, ci.v, wv, now, tot.nN, re - rb, tl);
                write_omega<MODE>(a, ci.v, now);
                if (MODE == kDelta) clear(ci.v);
                h->U = 0u; h->nN = 0u; h->flags = 0u; h->done = 0u;
                for (int c = 0; c < MAXC; c++) h->cnt[c] = 0u;
                if (MODE == kFirst && now) ci.nchunks = -ci.nchunks;      // listed below
            }
        }
        if (MODE == kFirst) list_row(a, ci.nchunks < 0, ci.v, re - rb, bs, bm);
        else if (MODE == kFull) bc.push(lane < cnt && wv != 0u, ci);
        else bg.push(lane < cnt && now != wv, Change{ci.v, now});
    }

    // (2) whole rows, the warp together
    const int mc = batch(n_med, 4);
    for (int64_t b0 = gwarp * mc; b0 < n_med; b0 += nwarps * mc) {
        const int cnt = (int)min((int64_t)mc, n_med - b0);
        int32_t v = -1;
        uint32_t wv = 0u, keep = 0u, kept = 0u;
        int64_t beg = 0, end = 0;
        if (lane < cnt) {
            v = a.med_in[b0 + lane];
            wv = omega_of(v);
            if (wv) {
                beg = a.rp[v];
                end = a.rp[v + 1];
            }
        }
        const uint32_t nbr = wv ? nbr_mask(wv, s) | a.eta_off : 0u;
        Partial<MAXC> mine;
        long_rows<MAXC, MODE, F>(a, s.n_cls, lut, cm, __ballot_sync(FULL_MASK, wv != 0u), beg, end, nbr, tl,
                                 [&](int j, const Partial<MAXC> &p) { if (lane == j) mine = p; });
        if (wv) {
            keep = decide<MAXC>(wv, mine, s);
            kept = mine.nN;
        }
        if (v >= 0) {
            if (wv) settle_row<MODE>(a, v, wv, keep, kept, end - beg, tl);
            else if (MODE == kFull && a.deg) a.deg[v] = 0u;
            write_omega<MODE>(a, v, keep);
            if (MODE == kDelta) clear(v);
        }
        if (MODE == kFirst) list_row(a, keep != 0u, v, end - beg, bs, bm);
        else if (MODE == kFull) bm.push(wv != 0u, v);
        else bg.push(v >= 0 && keep != wv, Change{v, keep});
    }

    // (3) short rows, 32 per batch; rows of more than 64 entries among them
    // (options.short_rows) by the warp
    const int sc = batch(n_small, 1);
    for (int64_t b0 = gwarp * sc; b0 < n_small; b0 += nwarps * sc) {
        int32_t v = -1;
        uint32_t wv = 0u, keep = 0u, kept = 0u;
        int64_t beg = 0, end = 0;
        if (lane < sc && b0 + lane < n_small) {
            v = a.small_in[b0 + lane];
            wv = omega_of(v);
            if (wv) {
                beg = a.rp[v];
                end = a.rp[v + 1];
            }
        }
        const uint32_t nbr = wv ? nbr_mask(wv, s) | a.eta_off : 0u;
        short_batch<MAXC, MODE, F>(a, s, lut, cm, wv, nbr, beg, end, keep, kept, tl);
        long_rows<MAXC, MODE, F>(a, s.n_cls, lut, cm, __ballot_sync(FULL_MASK, wv && end - beg > kGroupRow), beg, end,
                                 nbr, tl, [&](int j, const Partial<MAXC> &p) {
            if (lane == j) {
                keep = decide<MAXC>(wv, p, s);
                kept = p.nN;
            }
        });
        if (v >= 0) {
            if (wv) settle_row<MODE>(a, v, wv, keep, kept, end - beg, tl);
            else if (MODE == kFull && a.deg) a.deg[v] = 0u;
            write_omega<MODE>(a, v, keep);
            if (MODE == kDelta) clear(v);
        }
        if (MODE == kFull) bs.push(wv != 0u, v);
        else if (MODE == kDelta) bg.push(v >= 0 && keep != wv, Change{v, keep});
    }

    __syncthreads();
    if (MODE == kDelta) {
        block_flush(bg, &scnt[3][0], wib);
    } else {
        block_flush(bs, &scnt[0][0], wib);
        block_flush(bm, &scnt[1][0], wib);
        if (MODE == kFull) block_flush(bc, &scnt[2][0], wib);
    }
    add_totals(tl, totals, a.st);
}

// -------------------------------------------------------------------------
// Delta rounds.  What a round decides for a vertex depends on its own omega,
// its neighbours' and the bits of its row, so a vertex can only be decided
// otherwise than in the round before if its omega or a neighbour's changed
// there.  k_push writes the changes (Jacobi: after the round that found them)
// and lists the vertices to look at again: the changed ones and every
// neighbour over an entry that was still active (a vertex that died keeps its
// bits; no round reads them again).  k_lcc_round<., kDelta> evaluates these.  All
// other active vertices would find what they found before: the entries they
// scan are the entries they kept, so the counts of a round follow from the
// totals and the evaluated vertices alone (Pipeline::lcc).
//
// An 8-vertex template over frequent labels on 32M vertices (10^9 entries)
// eliminates 16M vertices in its first round and changes few after the second:
// its rounds three to six took 3.2 ms each, nearly all of it gathers of
// neighbours that had not changed, and take 1.6 ms together as delta rounds with
// 0.3 ms of k_push (the LCC phase 22.7 -> 11.7 ms).
// -------------------------------------------------------------------------

struct PushArgs {
    const int64_t *rp;
    const int32_t *col;
    const uint32_t *bits;
    uint32_t *om;                 // the current omega and its narrow copy
    void *nw;
    int nw_bytes;
    const uint32_t *om_old;       // after a full round: omega before it
    const int32_t *small_in, *med_in;
    const ChunkItem *chunk_in;
    const Change *chg;
    const ChangePiece *chg_piece;
    const RoundStats *prev;       // the counters of the round (or check) that made the changes
    uint32_t *dirty;
    int32_t *small_out, *med_out;
    ChunkItem *chunk_out;
    RoundStats *st;               // list sizes of the round to come
    int hub_deg, short_max;
};

// List the vertices u of the lanes with `want` that are not listed yet.
__device__ __forceinline__ void list_dirty(const PushArgs &a, bool want, int32_t u, WarpBuf<int32_t> &bs,
                                           WarpBuf<int32_t> &bm) {
    if (want) {
        const uint32_t m = 1u << (u & 31);
        want = !(a.dirty[u >> 5] & m) && !(atomicOr(&a.dirty[u >> 5], m) & m);
    }
    int64_t deg = 0;
    if (want) deg = a.rp[u + 1] - a.rp[u];
    const int64_t small_max = a.hub_deg < a.short_max ? a.hub_deg : a.short_max;
    bs.push(want && deg <= small_max, u);
    bm.push(want && deg > small_max && deg <= a.hub_deg, u);
    if (want && deg > a.hub_deg) {
        const int nch = (int)((deg + a.hub_deg - 1) / a.hub_deg);
        const int slot = (int)atomicAdd(&a.st->n_hub_slots, 1u);
        const unsigned int base = atomicAdd(&a.st->n_chunk, (unsigned int)nch);
        for (int c = 0; c < nch; c++) a.chunk_out[base + c] = ChunkItem{u, c, slot, nch};
    }
}

// The neighbours over the active entries of [beg, end) in a changed vertex's row.
__device__ __forceinline__ void push_row(const PushArgs &a, int64_t beg, int64_t end, WarpBuf<int32_t> &bs,
                                         WarpBuf<int32_t> &bm) {
    for_set_bits(a.bits, beg, end, [&](int64_t e, bool valid) {
        int32_t u = 0;
        if (valid) {
            u = __ldg(a.col + e);
            valid = a.om[u] != 0u;
        }
        list_dirty(a, valid, u, bs, bm);
    });
}

// LISTS: the changes are those between om_old and om over the lists of a full
// round; else they come from the Change list and are written to omega here.
template <bool LISTS>
__global__ void __launch_bounds__(256)
k_push(PushArgs a) {
    if (a.prev->changed == 0u) return;
    __shared__ int32_t sbuf[2][8][32];
    __shared__ int scnt[2][8];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane == 0) { scnt[0][wib] = 0; scnt[1][wib] = 0; }
    __syncthreads();
    WarpBuf<int32_t> bs{sbuf[0][wib], &scnt[0][wib], a.small_out, &a.st->n_small};
    WarpBuf<int32_t> bm{sbuf[1][wib], &scnt[1][wib], a.med_out, &a.st->n_med};
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // (1) pieces of long rows, one warp each
    const int64_t n_piece = LISTS ? a.prev->n_chunk : a.prev->n_chg_piece;
    for (int64_t it = gwarp; it < n_piece; it += nwarps) {
        int32_t v, c;
        if (LISTS) {
            const ChunkItem ci = a.chunk_in[it];
            v = ci.v;
            c = ci.c;
            const uint32_t w = a.om[v];
            if (w == a.om_old[v]) continue;
            if (c == 0) list_dirty(a, lane == 0 && w != 0u, v, bs, bm);
        } else {
            const ChangePiece cp = a.chg_piece[it];
            v = cp.v;
            c = cp.c;
        }
        const int64_t rend = a.rp[v + 1], beg = a.rp[v] + (int64_t)c * a.hub_deg;
        push_row(a, beg, min(rend, beg + (int64_t)a.hub_deg), bs, bm);
    }
    // (2) the other rows, 32 vertices per warp step, each changed one walked by the warp
    const int64_t n_small = LISTS ? a.prev->n_small : 0;
    const int64_t n_rows = LISTS ? n_small + a.prev->n_med : a.prev->n_chg;
    // few changes: fewer per warp, so that every warp gets some
    const int per = (int)max((int64_t)1, min((int64_t)32, n_rows / nwarps));
    for (int64_t b = gwarp * per; b < n_rows; b += nwarps * per) {
        const int64_t idx = b + lane;
        int32_t v = -1;
        uint32_t w = 0u;
        int64_t beg = 0, end = 0;
        if (lane < per && idx < n_rows) {
            if (LISTS) {
                v = idx < n_small ? a.small_in[idx] : a.med_in[idx - n_small];
                w = a.om[v];
                if (w == a.om_old[v]) v = -1;
            } else {
                const Change ch = a.chg[idx];
                v = ch.v;
                w = ch.w;
                a.om[v] = w;
                store_narrow(a.nw, a.nw_bytes, v, w);
            }
            if (v >= 0) {
                beg = a.rp[v];
                end = a.rp[v + 1];
            }
        }
        list_dirty(a, v >= 0 && w != 0u, v, bs, bm);
        const bool walk = v >= 0 && (LISTS || end - beg <= a.hub_deg);   // long rows: (1)
        for (uint32_t todo = __ballot_sync(FULL_MASK, walk); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            push_row(a, __shfl_sync(FULL_MASK, beg, src), __shfl_sync(FULL_MASK, end, src), bs, bm);
        }
    }
    __syncthreads();
    block_flush(bs, &scnt[0][0], wib);
    block_flush(bm, &scnt[1][0], wib);
}

// -------------------------------------------------------------------------
// K4: row compaction between LCC rounds (frontier and edge-bitmap compaction)
//
// Later rounds touch only the survivors, but the rows of the survivors still
// hold every neighbour they started with; once most of those entries are
// inactive a round spends its time skipping them.  Compaction writes a new
// CSR whose rows keep, in the same (ascending id) order, only the entries
// whose bit is set and whose other end point is still active: exactly the
// entries the next round would examine.  Ids stay the original vertex ids;
// the new bitmap starts with every bit set.  Entries left out are inactive
// for good (bits are only ever cleared and omega only shrinks), so every
// later round, and every search at a fixpoint, sees the same active entries
// as on the full rows.
//
// The frontier is rebuilt first (k_init over the live vertices) so that the
// pieces of a long row are consecutive in the piece list, in piece order:
// piece c's output offset is then the row's offset plus the counts of pieces
// 0..c-1.
// -------------------------------------------------------------------------

struct CompactArgs {
    const int64_t *rp;            // rows being compacted
    const int32_t *col;
    const uint32_t *bits;         // set exactly for the entries to keep
    const uint8_t *lab;
    const uint32_t *om;           // omega after the last round
    const int32_t *small_in;
    const int32_t *med_in;
    const ChunkItem *chunk_in;
    const HubAcc *acc;            // first-piece index of each long row (pbase)
    const RoundStats *lists;      // sizes of the three lists (written by the rebuild before)
    int hub_deg;
    int n_rank;                   // distinct labels of the template
    uint8_t lab_rank[256];        // rank of a template label among them
    uint8_t rank_label[kMaxT];
    uint32_t *piece_cnt;          // kept entries per (piece, rank) of long rows
    const int64_t *sub_rp;        // offsets of the new rows
    int32_t *sub_col;             // the new rows, grouped by label, ids ascending
    uint8_t *sub_nlab;            // inside a group, and their labels
    int32_t *dslot;               // per live vertex: its slot in gdir
    int64_t *gdir;                // per slot: start of each label group, then the row end
    unsigned int *n_slots;        // slot counter (zeroed before)
};

__device__ __forceinline__ uint32_t lane_rank_count(int r, int n_rank) {
    uint32_t rc = 0;
    for (int rr = 0; rr < n_rank; rr++) {
        const uint32_t m = __ballot_sync(FULL_MASK, r == rr);
        if ((int)lane_id() == rr) rc = __popc(m);
    }
    return rc;
}

// Kept entries of [beg, end) per label rank, summed into lane r (r < n_rank).
__device__ __forceinline__ uint32_t rank_counts(const CompactArgs &a, int64_t beg, int64_t end) {
    uint32_t rc = 0;
    for_set_bits(a.bits, beg, end, [&](int64_t e, bool valid) {
        int r = valid ? (int)a.lab_rank[__ldg(a.lab + __ldg(a.col + e))] : -1;
        if (r >= a.n_rank) r = -1;           // never: kept entries have template labels
        rc += lane_rank_count(r, a.n_rank);
    });
    return rc;
}

// Write the kept entries of [beg, end): lane r holds the next output index of
// label rank r.  Order inside a rank is the visiting order (ascending).
__device__ __forceinline__ void place_ranked(const CompactArgs &a, int64_t beg, int64_t end, int64_t cur) {
    const int lane = (int)lane_id();
    const uint32_t below = (1u << lane) - 1u;
    for_set_bits(a.bits, beg, end, [&](int64_t e, bool valid) {
        int32_t u = -1;
        int r = -1;
        if (valid) {
            u = __ldg(a.col + e);
            r = (int)a.lab_rank[__ldg(a.lab + u)];
            if (r >= a.n_rank) r = -1;
        }
        int64_t pos = -1;
        for (int rr = 0; rr < a.n_rank; rr++) {
            const uint32_t m = __ballot_sync(FULL_MASK, r == rr);
            const int64_t base = __shfl_sync(FULL_MASK, cur, rr);
            if (r == rr) pos = base + __popc(m & below);
            if (lane == rr) cur += __popc(m);
        }
        if (r >= 0) {
            a.sub_col[pos] = u;
            a.sub_nlab[pos] = a.rank_label[r];
        }
    });
}

// Exclusive prefix over lanes.
__device__ __forceinline__ uint32_t lane_excl(uint32_t x) {
    const int lane = (int)lane_id();
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += t;
    }
    return incl - x;
}

// Per-(piece, rank) kept entries of the pieces of long rows.
__global__ void __launch_bounds__(256)
k_compact_count(CompactArgs a) {
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    const int64_t n_chunk = a.lists->n_chunk;
    for (int64_t it = gwarp; it < n_chunk; it += nwarps) {
        const ChunkItem ci = a.chunk_in[it];
        if (__ldg(a.om + ci.v) == 0u) continue;
        const int64_t rbeg = a.rp[ci.v], rend = a.rp[ci.v + 1];
        const int64_t beg = rbeg + (int64_t)ci.c * a.hub_deg;
        const int64_t end = min(rend, beg + (int64_t)a.hub_deg);
        const uint32_t rc = rank_counts(a, beg, end);
        const int64_t p = (int64_t)a.acc[ci.slot].pbase + ci.c;
        if (lane < a.n_rank) a.piece_cnt[p * a.n_rank + lane] = rc;
    }
}

// Write the new rows and their label-group directory.  Pieces of long rows:
// rank r's group starts after the lower ranks of the whole row, and a piece's
// entries of rank r follow those of the row's earlier pieces.  Whole rows:
// by one lane when the row keeps at most 16 entries, else by the warp.
__global__ void __launch_bounds__(256)
k_compact_fill(CompactArgs a) {
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    const int64_t n_chunk = a.lists->n_chunk, n_med = a.lists->n_med, n_small = a.lists->n_small;
    for (int64_t it = gwarp; it < n_chunk; it += nwarps) {
        const ChunkItem ci = a.chunk_in[it];
        if (__ldg(a.om + ci.v) == 0u) continue;
        const int64_t rbeg = a.rp[ci.v], rend = a.rp[ci.v + 1];
        const int64_t beg = rbeg + (int64_t)ci.c * a.hub_deg;
        const int64_t end = min(rend, beg + (int64_t)a.hub_deg);
        const int64_t p0 = (int64_t)a.acc[ci.slot].pbase;
        // per rank, the row's total and the part in pieces before this one
        // (lanes stride over the pieces; lane r keeps rank r's sums)
        uint32_t tot = 0, before = 0;
        for (int r = 0; r < a.n_rank; r++) {
            uint32_t t = 0, b = 0;
            for (int c2 = lane; c2 < ci.nchunks; c2 += 32) {
                const uint32_t x = a.piece_cnt[(p0 + c2) * a.n_rank + r];
                t += x;
                if (c2 < ci.c) b += x;
            }
            t = __reduce_add_sync(FULL_MASK, t);
            b = __reduce_add_sync(FULL_MASK, b);
            if (lane == r) { tot = t; before = b; }
        }
        const int64_t gstart = a.sub_rp[ci.v] + (int64_t)lane_excl(tot);
        if (ci.c == 0) {
            unsigned int slot = 0;
            if (lane == 0) {
                slot = atomicAdd(a.n_slots, 1u);
                a.dslot[ci.v] = (int32_t)slot;
            }
            slot = __shfl_sync(FULL_MASK, slot, 0);
            if (lane <= a.n_rank) a.gdir[(int64_t)slot * (a.n_rank + 1) + lane] = gstart;
        }
        place_ranked(a, beg, end, gstart + before);
    }
    // whole rows, up to 32 list entries per warp step.  A row keeping at most 16
    // entries (most of them, once the first round has run) is written by its
    // own lane, one pass per label rank; the others by the whole warp in turn.
    // Short lists are dealt out over more warps, down to four rows each (and one
    // slot atomic): 1000 rows, 630 of them long, took 72 us at 32 a step.
    const int64_t n_rows = n_med + n_small;
    const int per = (int)max((int64_t)4, min((int64_t)32, n_rows / nwarps));
    for (int64_t b = gwarp * per; b < n_rows; b += nwarps * per) {
        const int64_t idx = b + lane;
        int32_t vl = -1;
        int64_t beg = 0, end = 0, out = 0, k = 0;
        if (lane < per && idx < n_rows) {
            vl = idx < n_med ? a.med_in[idx] : a.small_in[idx - n_med];
            if (__ldg(a.om + vl) == 0u) vl = -1;
        }
        if (vl >= 0) {
            beg = a.rp[vl];
            end = a.rp[vl + 1];
            out = a.sub_rp[vl];
            k = a.sub_rp[vl + 1] - out;
        }
        // one directory slot per live row, one atomic per warp step
        const uint32_t live = __ballot_sync(FULL_MASK, vl >= 0);
        unsigned int slot0 = 0;
        if (lane == 0 && live) slot0 = atomicAdd(a.n_slots, (unsigned int)__popc(live));
        const unsigned int slot = __shfl_sync(FULL_MASK, slot0, 0) + (unsigned int)__popc(live & ((1u << lane) - 1u));
        if (vl >= 0) a.dslot[vl] = (int32_t)slot;
        if (vl >= 0 && k <= 16) {
            const int64_t stop = out + k;
            int64_t *dir = a.gdir + (int64_t)slot * (a.n_rank + 1);
            // the row's kept entries (at most 16): positions from the bit words
            // (four words per step), then their columns, then their labels, each
            // as independent loads; then placed label by label
            int32_t eu[16];
            uint8_t er[16];
            int n = 0;
            for (int64_t wi = beg >> 5; (wi << 5) < end && n < 16; wi += 4) {
                uint32_t wd[4];
#pragma unroll
                for (int j = 0; j < 4; j++) wd[j] = ((wi + j) << 5) < end ? a.bits[wi + j] : 0u;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    uint32_t word = wd[j];
                    const int64_t e0 = (wi + j) << 5;
                    if (e0 < beg) word &= ~0u << (uint32_t)(beg - e0);
                    if (end - e0 < 32) word &= end > e0 ? (1u << (uint32_t)(end - e0)) - 1u : 0u;
                    for (; word && n < 16; word &= word - 1u) eu[n++] = (int32_t)(e0 + __ffs(word) - 1 - beg);
                }
            }
#pragma unroll
            for (int i = 0; i < 16; i++)
                if (i < n) eu[i] = __ldg(a.col + beg + eu[i]);
#pragma unroll
            for (int i = 0; i < 16; i++)
                er[i] = i < n ? a.lab_rank[__ldg(a.lab + eu[i])] : (uint8_t)0xFF;
            for (int r = 0; r < a.n_rank; r++) {
                dir[r] = out;
                const uint8_t L = a.rank_label[r];
#pragma unroll
                for (int i = 0; i < 16; i++) {
                    if (er[i] == r && out < stop) {
                        a.sub_col[out] = eu[i];
                        a.sub_nlab[out] = L;
                        out++;
                    }
                }
            }
            dir[a.n_rank] = stop;
        }
        for (uint32_t big = __ballot_sync(FULL_MASK, vl >= 0 && k > 16); big; big &= big - 1u) {
            const int src = __ffs(big) - 1;
            const int64_t rb = __shfl_sync(FULL_MASK, beg, src), re = __shfl_sync(FULL_MASK, end, src);
            const int64_t ro = __shfl_sync(FULL_MASK, out, src);
            const unsigned int rslot = __shfl_sync(FULL_MASK, slot, src);
            const uint32_t rc = rank_counts(a, rb, re);
            const int64_t gstart = ro + (int64_t)lane_excl(lane < a.n_rank ? rc : 0u);
            if (lane <= a.n_rank) a.gdir[(int64_t)rslot * (a.n_rank + 1) + lane] = gstart;
            place_ranked(a, rb, re, gstart);
        }
    }
}

// The entries of a result's edge map that join two live vertices, as the
// bitmap `out` (zeroed before) and as counts per vertex and in all: the rows a
// listing search reads.  A warp takes 32 vertices, one per lane, and walks the
// rows of the live ones together, so a state that keeps few of the vertices
// costs one pass over omega.
__global__ void __launch_bounds__(256)
k_live_entries(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
               const uint32_t *__restrict__ om, const uint32_t *__restrict__ bits, uint32_t *out, uint32_t *deg,
               RoundStats *st) {
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    unsigned long long total = 0;
    for (int64_t b = gwarp * 32; b < n; b += nwarps * 32) {
        const int64_t v = b + lane;
        int64_t beg = 0, end = 0;
        uint32_t mine = 0;
        const bool live = v < n && om[v] != 0u;
        if (live) { beg = rp[v]; end = rp[v + 1]; }
        for (uint32_t todo = __ballot_sync(FULL_MASK, live); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const int64_t rb = __shfl_sync(FULL_MASK, beg, src), re = __shfl_sync(FULL_MASK, end, src);
            uint32_t c = 0;
            for_set_bits(bits, rb, re, [&](int64_t e, bool valid) {
                const bool keep = valid && __ldg(om + __ldg(col + e)) != 0u;
                if (keep) atomicOr(&out[e >> 5], 1u << (uint32_t)(e & 31));
                c += (uint32_t)__popc(__ballot_sync(FULL_MASK, keep));
            });
            if (lane == src) mine = c;
        }
        if (live) deg[v] = mine;
        total += (unsigned long long)mine;
    }
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(FULL_MASK, total, o);
    if (lane == 0 && total) atomicAdd(&st->kept, total);
}

// Bits of the compacted rows: every entry active, nothing past the last one.
__global__ void k_compact_bits(uint32_t *bits, const int64_t *total) {
    const int64_t m2 = *total;
    const int64_t words = (m2 + 31) / 32;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= words; i += stride) {
        uint32_t v = 0u;
        if (i < words) v = (i == words - 1 && (m2 & 31)) ? (1u << (uint32_t)(m2 & 31)) - 1u : ~0u;
        bits[i] = v;
    }
}

// Edge map of the final state when it is handed back without the final
// search: at an LCC fixpoint an entry between two active vertices is active
// iff their omegas are compatible (eta); entries cleared earlier stay
// cleared.  One warp per vertex, over the full rows.
__global__ void __launch_bounds__(256)
k_materialize_fix(int64_t n, const uint32_t *__restrict__ om, const int64_t *__restrict__ rp,
                  const int32_t *__restrict__ col, uint32_t *ebits, DevTmpl t) {
    __shared__ uint32_t sadj[kMaxT];
    for (int i = threadIdx.x; i < kMaxT; i += blockDim.x) sadj[i] = t.adj[i];
    __syncthreads();
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    for (int64_t v = gwarp; v < n; v += nwarps) {
        const int64_t beg = rp[v], end = rp[v + 1];
        if (beg == end) continue;
        const uint32_t wv = om[v];
        if (wv == 0u) {
            clear_row<32>(ebits, beg, end, lane);
            continue;
        }
        uint32_t nb = 0;
        for (uint32_t x = wv; x; x &= x - 1u) nb |= sadj[__ffs(x) - 1];
        for (int64_t w0 = beg >> 5; (w0 << 5) < end; w0++) {
            const int64_t e = (w0 << 5) + lane;
            const uint32_t word = ebits[w0];
            bool drop = false;
            if (e >= beg && e < end && ((word >> lane) & 1u)) drop = (__ldg(om + __ldg(col + e)) & nb) == 0u;
            const uint32_t dm = __ballot_sync(FULL_MASK, drop);
            if (dm && lane == 0) atomicAnd(&ebits[w0], ~dm);
        }
    }
}

// Hand-back of the edge map when the live rows are exact: their bits, into a
// zeroed bitmap.  A warp takes 32 vertices and copies the live rows together:
// most vertices are dead by then, and clearing their rows instead cost two
// atomics each (1.15 ms over 32M vertices with 3.6M live; this 0.40).
__global__ void __launch_bounds__(256)
k_copy_live_rows(int64_t n, const uint32_t *__restrict__ om, const int64_t *__restrict__ rp,
                 const uint32_t *__restrict__ bits, uint32_t *out) {
    const int lane = (int)lane_id();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; b < n; b += stride) {
        const int64_t v = b + lane;
        const bool live = v < n && om[v] != 0u;
        int64_t beg = 0, end = 0;
        if (live) { beg = rp[v]; end = rp[v + 1]; }
        const bool shrt = end - beg <= 64;               // at most three words: by the lane itself
        if (live && shrt) {
            for (int64_t wi = beg >> 5; (wi << 5) < end; wi++) {
                const uint32_t in = word_range(wi, beg, end), x = bits[wi] & in;
                if (in == ~0u) out[wi] = x;
                else if (x) atomicOr(&out[wi], x);
            }
        }
        for (uint32_t todo = __ballot_sync(FULL_MASK, live && !shrt); todo; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            const int64_t rb = __shfl_sync(FULL_MASK, beg, src), re = __shfl_sync(FULL_MASK, end, src);
            for (int64_t wi = (rb >> 5) + lane; (wi << 5) < re; wi += 32) {
                const uint32_t in = word_range(wi, rb, re), x = bits[wi] & in;
                if (in == ~0u) out[wi] = x;
                else if (x) atomicOr(&out[wi], x);
            }
        }
    }
}

// -------------------------------------------------------------------------
// Rooted injective embedding search (NLCC token walk, Alg. 6/7, and the
// final template-driven search, Remark 1).  One warp per root vertex, roots
// handed out dynamically; the warp walks the plan depth first, testing 32
// candidates at a time in parallel.
//
// Searches run only at LCC fixpoints.  There an entry (x, u) is active
// exactly when some template edge joins omega(x) and omega(u) (edge
// elimination has removed every other entry and keeps every such one), so a
// search needs adjacency and omega only: a candidate u for template vertex q
// next to a placed x with q_x in omega(x) is joined to x by an active entry
// iff u is a neighbour of x with q in omega(u).  Candidates are read from a
// copy of every row grouped by neighbour label (label, then id), so only the
// neighbours that carry label(q) are ever scanned.
// -------------------------------------------------------------------------

// A partial embedding of a search plan: positions 0..depth-1 placed.  An item
// handed on by a long search may hold a part of the next position's candidates
// only: entries [lo, hi) of the label group its level scans, counted from the
// group's start (hi = 0: all of them).
constexpr int kItemMaxDepth = 10;
struct __align__(16) SearchItem {
    int32_t psi[kItemMaxDepth];
    int64_t entry;            // edge pass: CSR entry (psi[0], psi[1]) the item asks about
    uint32_t lo, hi;
    int32_t hd;               // head | depth << 8
};

struct SearchArgs {
    const int64_t *rp;
    const int32_t *col;       // id-sorted rows (edge-bitmap indexing)
    const int32_t *dslot;     // compacted rows: slot of a live vertex in gdir
    const int64_t *gdir;      // per slot: start of each label group, then the row end
    int n_rank;               // distinct template labels (groups per compacted row)
    uint8_t lab_rank[256];    // rank of a template label among them
    const int64_t *rl;        // offsets of the rows the searches scan:
    const int32_t *lcol;      // the full rows grouped by neighbour label, ids ascending
    const uint8_t *nlab;      // inside a group, with nlab = label of lcol[e]; or
                              // compacted rows (ids ascending) with nlab = nullptr
    const uint32_t *om;
    const int32_t *roots;
    int64_t n_roots;          // -1: st->n_roots
    PassCtl *ctl;             // this pass
    const PassCtl *ctl_prev;  // nullable: the items are those that pass handed on
    const DevPlan *plans;     // plans[h] for each head h (NLCC) or plans[0] (final)
    uint32_t heads;           // NLCC: heads of the constraint; final: 1 << plans[0].q[0]
    uint32_t *sat;            // NLCC output: satisfied heads per vertex
    uint32_t *om_out;         // final: omega*
    uint32_t *eb_out;         // final: edge bitmap of E*
    RoundStats *st;
    uint64_t budget;          // windows per (root, head)
    uint64_t cap;             // final: stop past this many matches
    SearchItem *items;        // split search work: partial embeddings
    int64_t n_items;          // -1: st->n_items (none of them if they are more than items_cap)
    int64_t items_cap;
    SearchItem *spill;        // a search that has scanned spill_after windows hands its
    int64_t spill_cap;        // untried candidates on here as new items (0: never)
    uint64_t spill_after;
    int starve;               // also hand on when the item list has run dry (idle warps)
    int enum_heads;           // k_expand: 1 = final search (one head), 0 = NLCC
    const uint32_t *sat_seed; // existence passes: heads already known satisfied (nullable)
    // listing (mode kList): every match found gets an index from list_count;
    // the first list_cap are written as n0 vertex ids in template order; vcnt
    // and ecnt (nullable) count the matches per vertex and per CSR entry
    int32_t *list_out;
    uint64_t list_cap;
    int list_n0;
    unsigned long long *list_count;
    unsigned long long *vcnt;
    unsigned long long *ecnt;
};

constexpr int kMaxBack = 4;  // joins per level whose label group is kept in shared memory

struct WarpSearch {
    int32_t psi[kMaxT];
    int64_t pos[kMaxT];       // next window start inside the chosen label range
    int64_t end[kMaxT];
    int64_t base[kMaxT];      // start of the scanned label group
    int64_t wbase[kMaxT];     // start of the window the mask refers to
    uint32_t mask[kMaxT];     // untried valid candidates of that window
    uint32_t chk[kMaxT];      // further joins, looked up from scratch per candidate
    int nb[kMaxT];            // joins with a stored label group
    int64_t blo[kMaxT][kMaxBack], bhi[kMaxT][kMaxBack];
    const uint32_t *done_word;  // existence: the answer is known once this bit is set
    uint32_t done_bit;          // (by another warp's embedding); nullptr: never
    int head;                   // plan slot of the running item (spilled items keep it)
    int64_t entry;              // edge pass: the running item's CSR entry
    int64_t n_items;            // items of this pass
    // the first kJoinCache stored join groups of one level in shared memory:
    // whole when they hold at most kJoinCacheLen ids, else every jc_step-th
    // id, which leaves a join test the search of one stretch of jc_step ids
    int jc_level;
    int jc_n[2], jc_step[2];
    int32_t jc[2][128];
    // the last match this warp marked (by plan position) and its plan: a
    // match found next in depth-first order usually differs from it only at
    // its last positions, and only what differs needs marking
    const DevPlan *last_plan;
    int32_t last[kMaxT];
    unsigned long long pub;     // matches of this warp already added to the global count
};
constexpr int kJoinCache = 2, kJoinCacheLen = 128;

// [lo, hi) of the label-L group in the label-grouped row of x: read from the
// group directory of the compacted rows, else found by binary search in the
// full rows.
__device__ __forceinline__ void label_range(const SearchArgs &a, int32_t x, uint32_t L, int64_t &lo, int64_t &hi) {
    if (a.gdir) {
        const int64_t *d = a.gdir + (int64_t)__ldg(a.dslot + x) * (a.n_rank + 1) + a.lab_rank[L];
        lo = __ldg(d);
        hi = __ldg(d + 1);
        return;
    }
    const int64_t b0 = a.rl[x], b1 = a.rl[x + 1];
    int64_t l = b0, h = b1;
    while (l < h) {
        int64_t m = (l + h) >> 1;
        if ((uint32_t)__ldg(a.nlab + m) < L) l = m + 1; else h = m;
    }
    lo = l;
    h = b1;
    while (l < h) {
        int64_t m = (l + h) >> 1;
        if ((uint32_t)__ldg(a.nlab + m) <= L) l = m + 1; else h = m;
    }
    hi = l;
}

// Is u (label L) a neighbour of x?  Binary search inside x's label-L group.
__device__ __forceinline__ bool adjacent(const SearchArgs &a, int32_t x, int32_t u, uint32_t L) {
    int64_t lo, hi;
    label_range(a, x, L, lo, hi);
    const int64_t stop = hi;
    while (lo < hi) {
        int64_t m = (lo + hi) >> 1;
        if (__ldg(a.lcol + m) < u) lo = m + 1; else hi = m;
    }
    return lo < stop && __ldg(a.lcol + lo) == u;
}

// CSR entries e1 of (x, y) and e2 of (y, x) in the id-sorted rows, or -1.  The
// two binary searches run side by side, so their loads overlap.
__device__ __forceinline__ void find_entries(const int64_t *rp, const int32_t *col, int32_t x, int32_t y, int64_t &e1,
                                             int64_t &e2) {
    int64_t l1 = rp[x], h1 = rp[x + 1], l2 = rp[y], h2 = rp[y + 1];
    const int64_t s1 = h1, s2 = h2;
    while (l1 < h1 || l2 < h2) {
        const int64_t m1 = (l1 + h1) >> 1, m2 = (l2 + h2) >> 1;
        const int32_t c1 = l1 < h1 ? __ldg(col + m1) : 0;
        const int32_t c2 = l2 < h2 ? __ldg(col + m2) : 0;
        if (l1 < h1) { if (c1 < y) l1 = m1 + 1; else h1 = m1; }
        if (l2 < h2) { if (c2 < x) l2 = m2 + 1; else h2 = m2; }
    }
    e1 = (l1 < s1 && __ldg(col + l1) == y) ? l1 : -1;
    e2 = (l2 < s2 && __ldg(col + l2) == x) ? l2 : -1;
}

__device__ __forceinline__ void set_bit(uint32_t *bits, int64_t e) {
    const uint32_t b = 1u << (uint32_t)(e & 31);
    if (!(bits[e >> 5] & b)) atomicOr(&bits[e >> 5], b);
}

// Both entries of the edge (x, y) get their bit in the output edge map.
__device__ __forceinline__ void mark_edge(const SearchArgs &a, int32_t x, int32_t y) {
    int64_t e1, e2;
    find_entries(a.rp, a.col, x, y, e1, e2);
    if (e1 >= 0) set_bit(a.eb_out, e1);
    if (e2 >= 0) set_bit(a.eb_out, e2);
}

// Open level d: among the placed neighbours of position d pick the one whose
// label group is shortest; scan that group, look the others up.
__device__ __forceinline__ void open_level(const SearchArgs &a, const DevPlan &P, WarpSearch &W, int d) {
    const int lane = (int)lane_id();
    // level d gets new groups: a join cache of this or a deeper level is stale
    if (lane == 0 && W.jc_level >= d) W.jc_level = -1;
    const uint32_t cm = P.nbr[d];
    const int cnt = __popc(cm);
    int64_t lo = 0, hi = 0, len = INT64_MAX;
    int j = -1;
    if (lane < cnt) {
        uint32_t m = cm;
        for (int i = 0; i < lane; i++) m &= m - 1u;
        j = __ffs(m) - 1;
        label_range(a, W.psi[j], P.lab[d], lo, hi);
        len = hi - lo;
    }
    int best = lane;
    for (int o = 16; o > 0; o >>= 1) {
        int64_t ol = __shfl_xor_sync(FULL_MASK, len, o);
        int ob = __shfl_xor_sync(FULL_MASK, best, o);
        if (ol < len || (ol == len && ob < best)) { len = ol; best = ob; }
    }
    // the other placed neighbours are joins: keep their label groups
    const int slot = lane < best ? lane : lane - 1;
    const bool join = lane < cnt && lane != best;
    if (join && slot < kMaxBack) {
        W.blo[d][slot] = lo;
        W.bhi[d][slot] = hi;
    }
    const uint32_t extra = __reduce_or_sync(FULL_MASK, (join && slot >= kMaxBack) ? (1u << j) : 0u);
    if (lane == best) {
        W.base[d] = lo;
        W.pos[d] = lo;
        W.end[d] = hi;
        W.mask[d] = 0u;
        W.chk[d] = extra;
        W.nb[d] = min(cnt - 1, kMaxBack);
    }
    __syncwarp();
}

// Both directions of every template edge of the embedding in W.psi get their
// bit in the output edge map (id-sorted entry indices).
__device__ __forceinline__ void mark_edges(const SearchArgs &a, const DevPlan &P, const WarpSearch &W) {
    for (int t = (int)lane_id(); t < P.n_marks; t += 32) mark_edge(a, W.psi[P.mark_a[t]], W.psi[P.mark_b[t]]);
    __syncwarp();
}

// `n` matches use the edge (x, y): counted on both of its entries.
__device__ __forceinline__ void count_edge(const SearchArgs &a, int32_t x, int32_t y, unsigned long long n) {
    int64_t e1, e2;
    find_entries(a.rp, a.col, x, y, e1, e2);
    if (e1 >= 0) atomicAdd(&a.ecnt[e1], n);
    if (e2 >= 0) atomicAdd(&a.ecnt[e2], n);
}

// Matches found by a listing search: positions 0..k-2 in W.psi, and in the
// lanes of vm one image u each of the last position.  Every match is stored
// (if its index is below the cap) and counted on every vertex and on both
// entries of every edge it uses; what the matches share is counted once for
// all of them.
__device__ __forceinline__ void list_window(const SearchArgs &a, const DevPlan &P, const WarpSearch &W, uint32_t vm,
                                            int32_t u) {
    const int lane = (int)lane_id(), last = P.k - 1;
    const unsigned long long n = (unsigned long long)__popc(vm);
    const bool ok = (vm >> lane) & 1u;
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(a.list_count, n);
    idx = __shfl_sync(FULL_MASK, idx, 0) + (unsigned long long)__popc(vm & ((1u << lane) - 1u));
    if (ok && idx < a.list_cap) {
        int32_t *row = a.list_out + idx * (unsigned long long)a.list_n0;
        for (int j = 0; j < last; j++) row[P.q[j]] = W.psi[j];
        row[P.q[last]] = u;
    }
    if (a.vcnt) {
        if (lane < last) atomicAdd(&a.vcnt[W.psi[lane]], n);
        if (ok) atomicAdd(&a.vcnt[u], 1ull);
    }
    if (a.ecnt) {
        for (int t = lane; t < P.n_marks; t += 32) {
            const int pa = P.mark_a[t], pb = P.mark_b[t];
            if (pa != last && pb != last) count_edge(a, W.psi[pa], W.psi[pb], n);
        }
        for (int t = 0; t < P.n_marks; t++) {
            const int pa = P.mark_a[t], pb = P.mark_b[t];
            if ((pa == last || pb == last) && ok) count_edge(a, W.psi[pa == last ? pb : pa], u, 1ull);
        }
    }
    __syncwarp();
}

// Warp-uniform: make the join cache hold level d's first stored groups.
__device__ __forceinline__ void join_cache(const SearchArgs &a, WarpSearch &W, int d) {
    if (W.jc_level == d) return;
    const int lane = (int)lane_id();
    const int nb = min(W.nb[d], kJoinCache);
    for (int b = 0; b < nb; b++) {
        const int64_t lo = W.blo[d][b], len = W.bhi[d][b] - lo;
        const int64_t step = len <= kJoinCacheLen ? 1 : (len + kJoinCacheLen - 1) / kJoinCacheLen;
        const int n = (int)((len + step - 1) / step);
        for (int i = lane; i < n; i += 32) W.jc[b][i] = __ldg(a.lcol + lo + i * step);
        if (lane == 0) { W.jc_n[b] = n; W.jc_step[b] = (int)step; }
    }
    if (lane == 0) W.jc_level = d;
    __syncwarp();
}

// Is the entry e of the scanned label group a valid image u for position d?
// Its omega must hold q_d, it must differ from earlier same-label images, and
// it must be joined to every other placed neighbour of position d.
__device__ __forceinline__ bool test_candidate(const SearchArgs &a, const DevPlan &P, WarpSearch &W,
                                               int d, int64_t e, int64_t end, int32_t &u) {
    if (W.nb[d] > 0) join_cache(a, W, d);
    u = -1;
    if (e >= end) return false;
    u = __ldg(a.lcol + e);
    if (!((__ldg(a.om + u) >> P.q[d]) & 1u)) return false;
    for (uint32_t sm = P.same[d]; sm; sm &= sm - 1u)
        if (W.psi[__ffs(sm) - 1] == u) return false;
    for (int b = 0; b < W.nb[d]; b++) {
        int64_t lo = W.blo[d][b], hi = W.bhi[d][b];
        if (b < kJoinCache) {
            int i = 0, h = W.jc_n[b];                // i: ids of the cache that are <= u
            while (i < h) {
                const int m2 = (i + h) >> 1;
                if (W.jc[b][m2] <= u) i = m2 + 1; else h = m2;
            }
            if (i == 0) return false;
            if (W.jc[b][i - 1] == u) continue;
            const int step = W.jc_step[b];
            if (step == 1) return false;
            hi = min(hi, lo + (int64_t)i * step);
            lo += (int64_t)(i - 1) * step + 1;
        }
        const int64_t stop = hi;
        while (lo < hi) {
            int64_t m2 = (lo + hi) >> 1;
            if (__ldg(a.lcol + m2) < u) lo = m2 + 1; else hi = m2;
        }
        if (!(lo < stop && __ldg(a.lcol + lo) == u)) return false;
    }
    for (uint32_t bm = W.chk[d]; bm; bm &= bm - 1u)
        if (!adjacent(a, W.psi[__ffs(bm) - 1], u, P.lab[d])) return false;
    return true;
}

// Mark the matches found by a marking enumeration (positions 0..k-2 in W.psi,
// the images u of the last position in the lanes of vm): every (vertex,
// template vertex) pair and both entries of every template edge.  What the
// matches of a window share is marked by one lane each, and only where it
// differs from what the warp marked last (same plan): marks are only ever set,
// and a pair or an edge whose positions hold the same vertices as then is
// marked already.  What hangs on the last position is marked by the match's
// own lane: each edge costs two binary searches of up to 17 dependent loads, so
// marking match by match kept 31 of 32 lanes idle (a marking pass of up to 2^16
// matches took 18.7 ms on one template over 4M vertices, 0.7 ms now).
__device__ __forceinline__ void mark_window(const SearchArgs &a, const DevPlan &P, WarpSearch &W, uint32_t vm,
                                            int32_t u) {
    const int lane = (int)lane_id(), last = P.k - 1;
    const bool same_plan = W.last_plan == &P;
    if (lane < last) {
        const int32_t x = W.psi[lane];
        if (!(same_plan && W.last[lane] == x)) {
            const uint32_t bit = 1u << P.q[lane];
            if (!(a.om_out[x] & bit)) atomicOr(&a.om_out[x], bit);
        }
    }
    for (int t = lane; t < P.n_marks; t += 32) {
        const int pa = P.mark_a[t], pb = P.mark_b[t];
        if (pa == last || pb == last) continue;
        const int32_t x = W.psi[pa], y = W.psi[pb];
        if (!(same_plan && W.last[pa] == x && W.last[pb] == y)) mark_edge(a, x, y);
    }
    if ((vm >> lane) & 1u) {
        const uint32_t bit = 1u << P.q[last];
        if (!(a.om_out[u] & bit)) atomicOr(&a.om_out[u], bit);
        for (int t = 0; t < P.n_marks; t++) {
            const int pa = P.mark_a[t], pb = P.mark_b[t];
            if (pa == last || pb == last) mark_edge(a, W.psi[pa == last ? pb : pa], u);
        }
    }
    __syncwarp();
    if (lane < last) W.last[lane] = W.psi[lane];
    if (lane == 0) W.last_plan = &P;
    __syncwarp();
}

// Search modes: does an embedding exist / count the embeddings / count them
// and mark the vertices and edges of every one / count them and list them.
constexpr int kExist = 0, kCount = 1, kMark = 2, kList = 3;

// Windows between a search's looks at what the other warps do, and so at least
// before it hands work on to idle ones.  A window that marks takes up to 8 us
// (every match's edges are looked up), one that only asks or counts 1 us, but all
// warps look at the same two words.  us of a prune with a 6-vertex tree on 5785
// vertices, of one with a 5-cycle on 16M, and of a listing on 1M, at 16, 8, 4 and
// 2 windows in every mode: 754, 542, 422, 440; 7917, 7281, 7363, 8018; 1791, 1821,
// 2085, 2629.  With 4 where marks are made, else 8: 415, 7040 and 1800.  A listing
// over fewer than kFewItems items hands on at once, the quickest way to more items
// (9*10^6 entries, 3 roots: 470 -> 370 us); pruning lost by it (415 -> 455 us).
__host__ __device__ constexpr uint64_t look_windows(int mode) { return mode == kMark ? 4 : 8; }
constexpr int64_t kFewItems = 1024;
constexpr int kSpillParts = 32;      // items one open level's untested candidates become, at most

// Hand the rest of a long search to other warps.  Every open level L (d0..d)
// gives one item (psi[0..L-1], c) of depth L+1 per tested and untried
// candidate c, and up to kSpillParts items of depth L that each hold a stretch
// of its untested candidates.  No candidate is tested here: handing on costs a
// few dozen stores, so a search can do it as soon as other warps are idle.
// That is what bounds these kernels: a window is a chain of dependent loads (a
// microsecond or more), so a pass lasts as long as its longest search.  Handing
// on only after 2048 windows, 16M vertices / 5*10^8 entries / 5-cycle template:
// 50 ms in 10 passes of k_nlcc_items and 18.6 ms in 3 of k_edge_search; handing
// on when the list is empty: 2.0 ms in 40 passes and 0.5 ms in 8 (the whole
// prune 78.6 -> 5.9 ms; a batch of 24 templates on 4M vertices 105 -> 23 ms).
// Returns false (the search goes on where it is) when the list is full.
// Reservations only ever add to the counter: the successful ones are exactly
// those ending at or below the capacity, and they fill the list up to the
// lowest start of a failed one (PassCtl::handed_on).
__device__ bool spill(const SearchArgs &a, const WarpSearch &W, int d0, int d) {
    const int lane = (int)lane_id();
    unsigned int total = 0;
    for (int L = d0; L <= d; L++) {
        const int64_t wins = (W.end[L] - W.pos[L] + 31) >> 5;
        total += (unsigned int)__popc(W.mask[L]) + (unsigned int)max((int64_t)0, min(wins, (int64_t)kSpillParts));
    }
    unsigned int base = 0, fits = 1;
    if (lane == 0 && total) {
        if ((int64_t)*(volatile const unsigned int *)&a.ctl->n_out >= a.spill_cap) {
            fits = 0;                               // full already: do not grow the counter
        } else {
            base = atomicAdd(&a.ctl->n_out, total);
            if ((int64_t)base + total > a.spill_cap) {
                atomicMax(&a.ctl->stop_inv, ~base);
                fits = 0;
            }
        }
    }
    if (!__shfl_sync(FULL_MASK, fits, 0)) return false;
    base = __shfl_sync(FULL_MASK, base, 0);
    for (int L = d0; L <= d; L++) {
        SearchItem si;
#pragma unroll
        for (int j = 0; j < kItemMaxDepth; j++) si.psi[j] = j < L ? W.psi[j] : 0;
        si.entry = W.entry;
        si.lo = si.hi = 0u;
        const uint32_t m = W.mask[L];
        if ((m >> lane) & 1u) {
            const int32_t c = __ldg(a.lcol + W.wbase[L] + lane);
#pragma unroll
            for (int j = 0; j < kItemMaxDepth; j++)
                if (j == L) si.psi[j] = c;
            si.hd = W.head | ((L + 1) << 8);
            a.spill[base + __popc(m & ((1u << lane) - 1u))] = si;
#pragma unroll
            for (int j = 0; j < kItemMaxDepth; j++)
                if (j == L) si.psi[j] = 0;
        }
        base += (unsigned int)__popc(m);
        const int64_t from = W.pos[L] - W.base[L], to = W.end[L] - W.base[L], wins = (to - from + 31) >> 5;
        if (wins <= 0) continue;
        const int parts = (int)min(wins, (int64_t)kSpillParts);
        if (lane < parts) {
            si.lo = (uint32_t)(from + 32 * (wins * lane / parts));
            si.hi = (uint32_t)min(to, from + 32 * (wins * (lane + 1) / parts));
            si.hd = W.head | (L << 8);
            a.spill[base + lane] = si;
        }
        base += (unsigned int)parts;
    }
    __syncwarp();
    return true;
}

// Depth-first search from positions 0..d0-1 already placed in W.psi (part_hi:
// over entries [part_lo, part_hi) of position d0's label group only).  kExist:
// true if an embedding exists; the other modes enumerate every embedding.
// `over` is set when the window budget ran out; for existence the root is then
// reported as satisfied, which keeps the result a superset of the exact answer.
template <int MODE>
__device__ bool search_from(const SearchArgs &a, const DevPlan &P, int d0, WarpSearch &W,
                            unsigned long long &entries, unsigned long long &matches, bool &over,
                            uint32_t part_lo = 0u, uint32_t part_hi = 0u) {
    const int lane = (int)lane_id();
    const int k = P.k;
    const uint64_t look_every = MODE == kList && a.starve && W.n_items < kFewItems ? 1 : look_windows(MODE);
    bool pending = false;
    unsigned int was_stop = 0;
    unsigned long long was_next = 0;
    uint64_t used = 0;
    unsigned long long pub = (MODE == kCount || MODE == kMark) ? W.pub : 0;   // matches published so far
    if (d0 >= k) {                                  // the placed prefix is already a full map
        if (MODE == kExist) return true;
        matches++;
        const int32_t x = W.psi[k - 1];
        if (MODE == kMark) mark_window(a, P, W, 1u, x);
        if (MODE == kList) list_window(a, P, W, 1u, x);
        return false;
    }
    open_level(a, P, W, d0);
    if (part_hi) {
        if (lane == 0) {
            W.end[d0] = W.base[d0] + part_hi;
            W.pos[d0] = W.base[d0] + part_lo;
        }
        __syncwarp();
    }
    int d = d0;
    while (d >= d0) {
        const uint32_t m = W.mask[d];
        if (m == 0u) {
            const int64_t pos = W.pos[d], end = W.end[d];
            if (pos >= end) { d--; continue; }
            if (++used > a.budget) { over = true; return MODE == kExist; }
            // every few windows (marking: and every 128 matches): has another
            // warp answered this existence question already, has the count run
            // past its cap, are other warps out of work?
            bool look = (used & (look_every - 1)) == 0u || (MODE == kMark && matches - pub >= 128u);
            if (MODE == kExist || MODE == kList) {
                // loaded here, looked at a window later
                const bool due = pending;
                pending = look;
                look = due;
            }
            unsigned int seen_stop = was_stop;
            unsigned long long seen_next = was_next;
            if ((MODE == kExist || MODE == kList) && pending && lane == 0) {
                if (MODE == kList) was_stop = *(volatile const unsigned int *)&a.st->overflow;
                else was_stop = W.done_word ? *(volatile const uint32_t *)W.done_word & W.done_bit : 0u;
                if (a.starve) was_next = *(volatile const unsigned long long *)&a.ctl->next;
            }
            if (look) {
                unsigned int stop = 0, hand = 0;
                if (lane == 0) {
                    if (MODE == kExist) {
                        stop = seen_stop;
                    } else if (MODE == kCount || MODE == kMark) {
                        // counting (and marking) stops as soon as the total passes
                        // the cap: publish this warp's new matches and read the
                        // total, so that no warp runs on to the cap by itself
                        const unsigned long long dm = matches - pub;
                        const unsigned long long tot =
                            dm ? atomicAdd(&a.st->matches, dm) + dm : *(volatile const unsigned long long *)&a.st->matches;
                        W.pub = matches;
                        stop = tot > a.cap || *(volatile const unsigned int *)&a.st->overflow;
                    } else {
                        stop = matches > a.cap || seen_stop;
                    }
                    if (MODE == kCount || MODE == kMark)
                        seen_next = a.starve && used >= look_every ? *(volatile const unsigned long long *)&a.ctl->next : 0ull;
                    hand = a.starve && seen_next >= (unsigned long long)W.n_items;
                }
                pub = matches;
                if (__shfl_sync(FULL_MASK, stop, 0)) {
                    // past the cap (the matches are published already, so the
                    // caller's batch-end check would not see it)
                    if (MODE == kCount || MODE == kMark) over = true;
                    return false;
                }
                hand = __shfl_sync(FULL_MASK, hand, 0);
                if (hand && d < kItemMaxDepth && spill(a, W, d0, d)) return false;
            }
            if (a.spill_after && used > a.spill_after && d < kItemMaxDepth && spill(a, W, d0, d))
                return false;                       // the rest runs as new items
            entries += (unsigned long long)min((int64_t)32, end - pos);
            int32_t u;
            const bool ok = test_candidate(a, P, W, d, pos + lane, end, u);
            const uint32_t vm = __ballot_sync(FULL_MASK, ok);
            if (d == k - 1) {
                // every valid image of the last position completes a match
                if (MODE == kExist) {
                    if (vm) {
                        if (lane == __ffs(vm) - 1) W.psi[d] = u;
                        __syncwarp();
                        return true;
                    }
                } else if (vm) {
                    matches += (unsigned long long)__popc(vm);
                    if (MODE == kMark) mark_window(a, P, W, vm, u);
                    if (MODE == kList) list_window(a, P, W, vm, u);
                }
                __syncwarp();
                if (lane == 0) W.pos[d] = pos + 32;
                __syncwarp();
                continue;
            }
            __syncwarp();
            if (lane == 0) { W.mask[d] = vm; W.wbase[d] = pos; W.pos[d] = pos + 32; }
            __syncwarp();
            continue;
        }
        const int b = __ffs(m) - 1;
        __syncwarp();
        if (lane == 0) { W.mask[d] = m & (m - 1u); W.psi[d] = __ldg(a.lcol + W.wbase[d] + b); }
        __syncwarp();
        d++;
        open_level(a, P, W, d);
    }
    return false;
}

__device__ __forceinline__ int64_t grab_root(const SearchArgs &a) {
    unsigned long long r = 0;
    if (lane_id() == 0) r = atomicAdd(&a.ctl->next, 1ull);
    return (int64_t)__shfl_sync(FULL_MASK, r, 0);
}

__global__ void __launch_bounds__(128)
k_nlcc_search(SearchArgs a) {
    __shared__ WarpSearch ws[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    unsigned long long entries = 0, matches = 0;
    bool over = false;
    for (int64_t it = grab_root(a); it < a.n_roots; it = grab_root(a)) {
        const int32_t v = a.roots[it];
        const uint32_t seed = a.sat_seed ? __ldg(a.sat_seed + v) : 0u;
        const uint32_t hv = __ldg(a.om + v) & a.heads & ~seed;
        uint32_t sat = seed;
        for (uint32_t hm = hv; hm; hm &= hm - 1u) {
            const int h = __ffs(hm) - 1;
            if (lane == 0) { W.psi[0] = v; W.done_word = nullptr; }
            __syncwarp();
            if (search_from<kExist>(a, a.plans[h], 1, W, entries, matches, over)) sat |= 1u << h;
            __syncwarp();
        }
        if (lane == 0) a.sat[v] = sat;
    }
    // entries, tokens and over are identical in every lane of the warp
    if (lane == 0) {
        if (entries) atomicAdd(&a.st->windows, entries);
        if (over) atomicOr(&a.st->overflow, 1u);
    }
}

template <int MODE>
__global__ void __launch_bounds__(128)
k_final_search(SearchArgs a) {
    __shared__ WarpSearch ws[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    if (lane == 0) { W.last_plan = nullptr; W.pub = 0; }
    __syncwarp();
    unsigned long long entries = 0, matches = 0;
    bool over = false;
    for (int64_t it = grab_root(a); it < a.n_roots; it = grab_root(a)) {
        unsigned int stop = 0;
        if (lane == 0) stop = *(volatile unsigned int *)&a.st->overflow;
        if (__shfl_sync(FULL_MASK, stop, 0)) break;
        const int32_t v = a.roots[it];
        if (lane == 0) { W.psi[0] = v; W.done_word = nullptr; }
        __syncwarp();
        search_from<MODE>(a, a.plans[0], 1, W, entries, matches, over);
        __syncwarp();
        const unsigned long long pub = W.pub;     // read by every lane before lane 0 moves it
        __syncwarp();
        if (matches != pub) {
            unsigned long long tot = 0;
            if (lane == 0) {
                tot = atomicAdd(&a.st->matches, matches - pub) + (matches - pub);
                W.pub = matches;
            }
            tot = __shfl_sync(FULL_MASK, tot, 0);
            __syncwarp();
            if (tot > a.cap) over = true;
        }
        if (over) {
            if (lane == 0) atomicOr(&a.st->overflow, 1u);
            break;
        }
    }
    if (lane == 0 && entries) atomicAdd(&a.st->windows, entries);
}

// Split search work by the first level: every (root, head) becomes one item per
// candidate for position 1, so expensive roots spread over many warps.
__global__ void __launch_bounds__(256)
k_expand(SearchArgs a) {
    __shared__ SearchItem sbuf[8][32];
    __shared__ int scnt[8];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane == 0) scnt[wib] = 0;
    __syncthreads();
    WarpBuf<SearchItem> b{sbuf[wib], &scnt[wib], a.items, &a.st->n_items};
    b.cap = (unsigned long long)a.items_cap;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long entries = 0, tokens = 0;
    const int64_t n_roots = a.n_roots >= 0 ? a.n_roots : (int64_t)a.st->n_roots;
    for (int64_t it = gwarp; it < n_roots; it += nwarps) {
        const int32_t v = a.roots[it];
        const uint32_t seed = (!a.enum_heads && a.sat_seed) ? __ldg(a.sat_seed + v) : 0u;
        const uint32_t hv = a.enum_heads ? a.heads : (__ldg(a.om + v) & a.heads & ~seed);
        if (!a.enum_heads && lane == 0) a.sat[v] = seed;
        tokens += (unsigned long long)__popc(hv);
        for (uint32_t hm = hv; hm; hm &= hm - 1u) {
            const int h = __ffs(hm) - 1;
            const DevPlan &P = a.plans[a.enum_heads ? 0 : h];
            const int q1 = P.q[1];
            int64_t lo, hi;
            label_range(a, v, P.lab[1], lo, hi);
            entries += (unsigned long long)(hi - lo);
            for (int64_t base = lo; base < hi; base += 32) {
                const int64_t e = base + lane;
                bool ok = false;
                int32_t u = -1;
                if (e < hi) {
                    u = __ldg(a.lcol + e);
                    ok = ((__ldg(a.om + u) >> q1) & 1u) && !((P.same[1] & 1u) && u == v);
                }
                SearchItem si;
#pragma unroll
                for (int j = 2; j < kItemMaxDepth; j++) si.psi[j] = 0;
                si.psi[0] = v;
                si.psi[1] = u;
                si.entry = 0;
                si.lo = si.hi = 0u;
                si.hd = h | (2 << 8);
                b.push(ok, si);
            }
        }
    }
    b.flush();
    if (lane == 0) {
        if (entries) atomicAdd(&a.st->expanded, entries);
        if (tokens) atomicAdd(&a.st->tokens, tokens);
    }
}

// When there are too few items to fill the GPU, place one more position:
// every input item of depth D becomes one item per valid image of position D.
// Items that already place every position pass through.
__global__ void __launch_bounds__(128)
k_expand_next(SearchArgs a, const SearchItem *in, int64_t n_in) {
    __shared__ WarpSearch ws[4];
    __shared__ SearchItem sbuf[4][32];
    __shared__ int scnt[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    if (lane == 0) scnt[wib] = 0;
    __syncthreads();
    WarpBuf<SearchItem> b{sbuf[wib], &scnt[wib], a.items, &a.st->n_items};
    b.cap = (unsigned long long)a.items_cap;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long entries = 0;
    for (int64_t it = gwarp; it < n_in; it += nwarps) {
        const SearchItem item = in[it];
        const int h = item.hd & 0xff, depth = item.hd >> 8;
        const DevPlan &P = a.plans[a.enum_heads ? 0 : h];
        if (depth >= P.k || depth >= kItemMaxDepth) {
            b.push(lane == 0, item);
            continue;
        }
        if (lane < depth) W.psi[lane] = item.psi[lane];
        __syncwarp();
        open_level(a, P, W, depth);
        const int64_t lo = W.pos[depth], hi = W.end[depth];
        entries += (unsigned long long)(hi - lo);
        for (int64_t base = lo; base < hi; base += 32) {
            int32_t u;
            const bool ok = test_candidate(a, P, W, depth, base + lane, hi, u);
            SearchItem si = item;
#pragma unroll
            for (int j = 0; j < kItemMaxDepth; j++)
                if (j == depth) si.psi[j] = u;
            si.hd = h | ((depth + 1) << 8);
            b.push(ok, si);
        }
    }
    b.flush();
    if (lane == 0 && entries) atomicAdd(&a.st->expanded, entries);
}

__device__ __forceinline__ int64_t grab_items(const SearchArgs &a, int batch) {
    unsigned long long r = 0;
    if (lane_id() == 0) r = atomicAdd(&a.ctl->next, (unsigned long long)batch);
    return (int64_t)__shfl_sync(FULL_MASK, r, 0);
}

// Items of this pass, and how many of them a warp takes at a time: one where
// there are few, so that none waits behind a long one.
__device__ __forceinline__ int64_t pass_items(const SearchArgs &a, int &batch) {
    int64_t n = a.n_items;
    if (a.ctl_prev) n = a.ctl_prev->handed_on();
    else if (n < 0) n = a.st->n_items <= a.items_cap ? (int64_t)a.st->n_items : 0;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    batch = (int)max((int64_t)1, min((int64_t)16, n / (8 * warps)));
    return n;
}

constexpr int kMaxPlans = 64;      // plan slots (heads, or oriented template edges)
constexpr uint64_t kMarkCap = 1ull << 20;   // matches one marking enumeration handles
constexpr uint64_t kFewMatches = 1ull << 16;   // marked during the first enumeration itself
// Below this many first-level items the searches place position 2 as well.
constexpr int64_t kExpandBelow = 16384;

__global__ void __launch_bounds__(128)
k_nlcc_items(SearchArgs a) {
    int batch;
    const int64_t n_items = pass_items(a, batch);
    if (n_items == 0) return;                        // a pass queued after the last one
    __shared__ WarpSearch ws[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    if (lane == 0) W.n_items = n_items;
    __syncwarp();
    unsigned long long entries = 0, matches = 0;
    bool over = false;
    for (int64_t it0 = grab_items(a, batch); it0 < n_items; it0 = grab_items(a, batch)) {
        const int64_t it1 = min(n_items, it0 + batch);
        for (int64_t it = it0; it < it1; it++) {
            const SearchItem item = a.items[it];
            const int h = item.hd & 0xff, depth = item.hd >> 8;
            const uint32_t bit = 1u << h;
            uint32_t done = 0;                                       // satisfied by another item?
            if (lane == 0) done = *(volatile uint32_t *)&a.sat[item.psi[0]] & bit;
            if (__shfl_sync(FULL_MASK, done, 0)) continue;
            if (lane < depth) W.psi[lane] = item.psi[lane];
            if (lane == 0) { W.done_word = &a.sat[item.psi[0]]; W.done_bit = bit; W.head = h; W.entry = 0; }
            __syncwarp();
            bool ran_out = false;
            if (search_from<kExist>(a, a.plans[h], depth, W, entries, matches, ran_out, item.lo, item.hi)) {
                const DevPlan &P = a.plans[h];
                if (ran_out) {
                    // budget exhausted: keep the head (a superset of the exact answer)
                    if (lane == 0) atomicOr(&a.sat[item.psi[0]], bit);
                } else {
                    // the embedding found satisfies every head it places, not only h
                    if (lane < P.k) {
                        const int q = P.q[lane];
                        if ((a.heads >> q) & 1u) atomicOr(&a.sat[W.psi[lane]], 1u << q);
                    }
                    if (a.eb_out) mark_edges(a, P, W);
                }
            }
            over = over || ran_out;
            __syncwarp();
        }
    }
    if (lane == 0) {
        if (entries) atomicAdd(&a.st->windows, entries);
        if (over) atomicOr(&a.st->overflow, 1u);
    }
}

template <int MODE>
__global__ void __launch_bounds__(128)
k_final_items(SearchArgs a) {
    int batch;
    const int64_t n_items = pass_items(a, batch);
    if (n_items == 0) return;                        // a pass queued after the last one
    __shared__ WarpSearch ws[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    if (lane == 0) W.n_items = n_items;
    __syncwarp();
    if (lane == 0) { W.last_plan = nullptr; W.pub = 0; }
    __syncwarp();
    unsigned long long entries = 0, matches = 0;
    bool over = false;
    for (int64_t it0 = grab_items(a, batch); it0 < n_items; it0 = grab_items(a, batch)) {
        unsigned int stop = 0;
        if (lane == 0) stop = *(volatile unsigned int *)&a.st->overflow;
        if (__shfl_sync(FULL_MASK, stop, 0)) break;
        const int64_t it1 = min(n_items, it0 + batch);
        for (int64_t it = it0; it < it1 && !over; it++) {
            const SearchItem item = a.items[it];
            const int depth = item.hd >> 8;
            if (lane < depth) W.psi[lane] = item.psi[lane];
            if (lane == 0) { W.done_word = nullptr; W.head = item.hd & 0xff; W.entry = 0; }
            __syncwarp();
            search_from<MODE>(a, a.plans[0], depth, W, entries, matches, over, item.lo, item.hi);
            __syncwarp();
        }
        const unsigned long long pub = W.pub;     // read by every lane before lane 0 moves it
        __syncwarp();
        if (matches != pub) {
            unsigned long long tot = 0;
            if (lane == 0) {
                tot = atomicAdd(&a.st->matches, matches - pub) + (matches - pub);
                W.pub = matches;
            }
            tot = __shfl_sync(FULL_MASK, tot, 0);
            __syncwarp();
            if (tot > a.cap) over = true;
        }
        if (over) {
            if (lane == 0) atomicOr(&a.st->overflow, 1u);
            break;
        }
    }
    if (lane == 0 && entries) atomicAdd(&a.st->windows, entries);
}

// Edge pass of the final step: every entry (x, y), x < y, whose ends hold
// omega* sets joined by some template edge and that no embedding found so far
// has marked becomes one item per orientation (a, b) of a template edge with
// a in omega*(x), b in omega*(y); plans[o] is rooted at that oriented edge.
struct EdgeTab {
    int n;                       // oriented template edges in this pass
    int8_t a[32], b[32];
};

__global__ void __launch_bounds__(256)
k_edge_items(SearchArgs a, EdgeTab tab) {
    __shared__ SearchItem sbuf[8][32];
    __shared__ int scnt[8];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    if (lane == 0) scnt[wib] = 0;
    __syncthreads();
    WarpBuf<SearchItem> b{sbuf[wib], &scnt[wib], a.items, &a.st->n_items};
    b.cap = (unsigned long long)a.items_cap;
    // one block per root: its warps take every (blockDim/32)-th window of the
    // root's row, so the rows of hubs are split across the block
    const int nwb = (int)(blockDim.x >> 5);
    const int64_t n_roots = a.n_roots >= 0 ? a.n_roots : (int64_t)a.st->n_roots;
    for (int64_t it = blockIdx.x; it < n_roots; it += gridDim.x) {
        const int32_t x = a.roots[it];
        const uint32_t wx = __ldg(a.om + x);
        const int64_t beg = a.rp[x], end = a.rp[x + 1];
        for (int64_t base = beg + (int64_t)wib * 32; base < end; base += (int64_t)nwb * 32) {
            const int64_t e = base + lane;
            int32_t y = -1;
            uint32_t wy = 0u;
            if (e < end) {
                y = __ldg(a.col + e);
                if (y > x && !((a.eb_out[e >> 5] >> (uint32_t)(e & 31)) & 1u)) wy = __ldg(a.om + y);
            }
            // most neighbours of a hub are outside omega*: nothing to push
            if (!__any_sync(FULL_MASK, wy != 0u)) continue;
            for (int o = 0; o < tab.n; o++) {
                const bool ok = wy && ((wx >> tab.a[o]) & 1u) && ((wy >> tab.b[o]) & 1u);
                SearchItem si;
#pragma unroll
                for (int j = 2; j < kItemMaxDepth; j++) si.psi[j] = 0;
                si.psi[0] = x;
                si.psi[1] = y;
                si.entry = e;
                si.lo = si.hi = 0u;
                si.hd = o | (2 << 8);
                b.push(ok, si);
            }
        }
    }
    b.flush();
}

__global__ void __launch_bounds__(128)
k_edge_search(SearchArgs a) {
    int batch;
    const int64_t n_items = pass_items(a, batch);
    if (n_items == 0) return;                        // a pass queued after the last one
    __shared__ WarpSearch ws[4];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    WarpSearch &W = ws[wib];
    if (lane == 0) W.n_items = n_items;
    __syncwarp();
    unsigned long long entries = 0, matches = 0;
    bool over = false;
    for (int64_t it0 = grab_items(a, batch); it0 < n_items; it0 = grab_items(a, batch)) {
        const int64_t it1 = min(n_items, it0 + batch);
        for (int64_t it = it0; it < it1; it++) {
            const SearchItem item = a.items[it];
            const int o = item.hd & 0xff, depth = item.hd >> 8;
            // the entry of the item's template edge (items handed on by long
            // searches keep it)
            const int64_t e = item.entry;
            uint32_t done = 0;                          // marked by an embedding found meanwhile?
            if (lane == 0) done = (*(volatile uint32_t *)&a.eb_out[e >> 5] >> (uint32_t)(e & 31)) & 1u;
            if (__shfl_sync(FULL_MASK, done, 0)) continue;
            if (lane < depth) W.psi[lane] = item.psi[lane];
            if (lane == 0) {
                W.done_word = &a.eb_out[e >> 5];
                W.done_bit = 1u << (uint32_t)(e & 31);
                W.head = o;
                W.entry = e;
            }
            __syncwarp();
            const DevPlan &P = a.plans[o];
            bool ran_out = false;
            if (search_from<kExist>(a, P, depth, W, entries, matches, ran_out, item.lo, item.hi)) {
                if (!ran_out) {
                    mark_edges(a, P, W);
                } else if (lane == 0) {
                    // budget exhausted: keep the edge (a superset of the exact answer)
                    mark_edge(a, item.psi[0], item.psi[1]);
                }
            }
            over = over || ran_out;
        }
    }
    if (lane == 0) {
        if (entries) atomicAdd(&a.st->windows, entries);
        if (over) atomicOr(&a.st->overflow, 1u);
    }
}

// omega* of the roots from their satisfied bits.
__global__ void k_sat_to_omega(const int32_t *roots, const RoundStats *st, const uint32_t *sat, const uint32_t *om,
                               uint32_t *om_out) {
    const int64_t n_roots = st->n_roots;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_roots; i += stride) {
        const int32_t v = roots[i];
        om_out[v] = sat[v] & om[v];
    }
}

// Label of the neighbour at every CSR entry (sort keys for the grouped rows).
__global__ void __launch_bounds__(256)
k_gather_labels(int64_t m, const int32_t *__restrict__ col, const uint8_t *__restrict__ lab, uint8_t *out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride)
        out[e] = __ldg(lab + __ldg(col + e));
}

// Label-grouped rows (once per graph): every row's entries stably sorted by
// their neighbour's label, by a counting sort per row.  One warp per row: a
// histogram of the row's labels in shared memory (256 bins), its exclusive
// scan, then the entries in order, 32 at a time, each placed at its label's
// next slot (lanes with equal labels are ranked by lane order, so equal
// labels keep their order).  keys: the labels in entry order, or NULL to
// gather them.
__device__ __forceinline__ uint32_t row_label(const uint8_t *keys, const int32_t *col, const uint8_t *lab,
                                              int64_t e, int64_t end) {
    if (e >= end) return 256u;                    // no entry: a value no label has
    return keys ? (uint32_t)keys[e] : (uint32_t)__ldg(lab + __ldg(col + e));
}

__global__ void __launch_bounds__(256)
k_label_sort(int64_t n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
             const uint8_t *__restrict__ lab, const uint8_t *__restrict__ keys, uint8_t *nlab, int32_t *lcol) {
    __shared__ uint32_t bins[8][256];
    const int wib = threadIdx.x >> 5;
    const int lane = (int)lane_id();
    uint32_t *h = bins[wib];
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = gw; v < n; v += nw) {
        const int64_t beg = rp[v], end = rp[v + 1];
        if (end <= beg) continue;
#pragma unroll
        for (int k = 0; k < 8; k++) h[lane * 8 + k] = 0u;
        __syncwarp();
        for (int64_t c = beg; c < end; c += 32) {
            const uint32_t L = row_label(keys, col, lab, c + lane, end);
            const uint32_t grp = __match_any_sync(FULL_MASK, L);
            if (L < 256u && lane == __ffs(grp) - 1) h[L] += (uint32_t)__popc(grp);
            __syncwarp();
        }
        // exclusive scan of the 256 bins: 8 per lane, then across lanes
        uint32_t loc[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; k++) { loc[k] = sum; sum += h[lane * 8 + k]; }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL_MASK, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t excl = incl - sum;
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; k++) h[lane * 8 + k] = excl + loc[k];
        __syncwarp();
        for (int64_t c = beg; c < end; c += 32) {
            const int64_t e = c + lane;
            const uint32_t L = row_label(keys, col, lab, e, end);
            const uint32_t grp = __match_any_sync(FULL_MASK, L);
            if (L < 256u) {
                const uint32_t below = grp & ((1u << lane) - 1u);
                const int64_t pos = beg + (int64_t)h[L] + __popc(below);
                nlab[pos] = (uint8_t)L;
                lcol[pos] = __ldg(col + e);
            }
            __syncwarp();
            if (L < 256u && lane == __ffs(grp) - 1) h[L] += (uint32_t)__popc(grp);
            __syncwarp();
        }
    }
}

// Row offsets of a compaction: exclusive prefix sum, over vertices 0..n (one
// value past the last), of the entries each live vertex keeps (deg; vertices
// whose omega is empty keep none), in three passes: each block scans
// a tile of kScanTile values and writes its total, one block scans the tile
// totals (in tiles of its own, carrying the running sum), and each tile adds
// its offset.
constexpr int kScanTile = 2048;                 // 256 threads x 8 values

__device__ __forceinline__ int64_t block_excl_scan(int64_t x, int64_t &total) {
    __shared__ int64_t warp_tot[8];
    const int lane = (int)lane_id(), wib = threadIdx.x >> 5;
    int64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[wib] = incl;
    __syncthreads();
    int64_t before = 0;
    total = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
        if (w < wib) before += warp_tot[w];
        total += warp_tot[w];
    }
    __syncthreads();
    return before + incl - x;
}

__global__ void __launch_bounds__(256)
k_scan_tiles(int64_t n, const uint32_t *__restrict__ deg, const uint32_t *__restrict__ om, int64_t *out,
             int64_t *tile_sum) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * 8;
    int64_t v[8], s = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        v[k] = base + k < n && om[base + k] ? (int64_t)deg[base + k] : 0;
        s += v[k];
    }
    int64_t total;
    int64_t run = block_excl_scan(s, total);
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (base + k <= n) out[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = total;
}

__global__ void __launch_bounds__(256)
k_scan_sums(int64_t tiles, int64_t *tile_sum) {
    int64_t carry = 0;
    for (int64_t t0 = 0; t0 < tiles; t0 += kScanTile) {
        const int64_t base = t0 + (int64_t)threadIdx.x * 8;
        int64_t v[8], s = 0;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            v[k] = base + k < tiles ? tile_sum[base + k] : 0;
            s += v[k];
        }
        int64_t total;
        int64_t run = carry + block_excl_scan(s, total);
#pragma unroll
        for (int k = 0; k < 8; k++) {
            if (base + k < tiles) tile_sum[base + k] = run;
            run += v[k];
        }
        carry += total;
    }
}

__global__ void __launch_bounds__(256)
k_scan_add(int64_t n, int64_t *out, const int64_t *__restrict__ tile_off) {
    const int64_t off = tile_off[blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    for (int i = threadIdx.x; i < kScanTile; i += blockDim.x)
        if (base + i <= n) out[base + i] += off;
}

// Roots of a search: every vertex whose omega meets `heads`.
__global__ void __launch_bounds__(256)
k_collect_roots(int64_t n, const uint32_t *__restrict__ om, uint32_t heads, int32_t *roots, RoundStats *st) {
    __shared__ int32_t sbuf[8][32];
    __shared__ int scnt[8];
    const int wib = threadIdx.x >> 5;
    if (lane_id() == 0) scnt[wib] = 0;
    __syncthreads();
    WarpBuf<int32_t> b{sbuf[wib], &scnt[wib], roots, &st->n_roots};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_pad = (n + 31) & ~(int64_t)31;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_pad; v += stride) {
        bool p = v < n && (__ldg(om + v) & heads);
        b.push(p, (int32_t)v);
    }
    b.flush();
}

// Alg. 6 lines 5-11: issuers whose token failed lose the head; a vertex whose
// omega empties is eliminated with its edges.  The changes are listed for the
// LCC rounds that follow, and the totals of the state (entries kept, rows) lose
// what the eliminated vertices held.  Both omega buffers are written: which
// one the rounds continue from is the caller's matter.  last: the last queued
// pass of the search (NULL: the search is known to be complete).
__global__ void __launch_bounds__(256)
k_nlcc_apply(const int32_t *__restrict__ roots, const PassCtl *last, int64_t items_cap, uint32_t heads,
             const uint32_t *__restrict__ sat, const uint32_t *om, uint32_t *om0, uint32_t *om1, void *nw0, void *nw1,
             int nw_bytes, const int64_t *__restrict__ rp, uint32_t *deg, Change *chg,
             ChangePiece *chg_piece, int hub_deg, RoundStats *st) {
    // queued behind the search's passes: does nothing if they did not finish it
    if (last && (st->n_items > items_cap || last->handed_on())) return;
    const int64_t n_roots = st->n_roots;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint32_t changed = 0, died = 0;
    unsigned long long old_kept = 0, died_rows = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_roots; i += stride) {
        const int32_t v = roots[i];
        const uint32_t w = om[v];
        const uint32_t nw = w & ~(heads & ~sat[v]);
        if (nw != w) {
            om0[v] = nw;
            om1[v] = nw;
            store_narrow(nw0, nw_bytes, v, nw);
            store_narrow(nw1, nw_bytes, v, nw);
            changed = 1u;
            const int64_t beg = rp[v], len = rp[v + 1] - beg;
            if (nw == 0u) {
                old_kept += deg[v];
                deg[v] = 0u;
                died_rows += (unsigned long long)len;
                died++;
            }
            if (!chg) continue;                      // no delta rounds follow
            chg[atomicAdd(&st->n_chg, 1u)] = Change{v, nw};
            if (len > hub_deg) {
                const unsigned int np = (unsigned int)((len + hub_deg - 1) / hub_deg);
                const unsigned int b = atomicAdd(&st->n_chg_piece, np);
                for (unsigned int c = 0; c < np; c++) chg_piece[b + c] = ChangePiece{v, (int32_t)c};
            }
        }
    }
    changed = __any_sync(FULL_MASK, changed);
    died = __reduce_add_sync(FULL_MASK, died);
    old_kept = warp_total(old_kept);
    died_rows = warp_total(died_rows);
    if (lane_id() == 0 && changed) {
        atomicOr(&st->changed, 1u);
        if (died) {
            atomicAdd(&st->died, died);
            atomicAdd(&st->old_kept, old_kept);
            atomicAdd(&st->died_rows, died_rows);
        }
    }
}

__device__ __forceinline__ bool ebit(const uint32_t *eb, int64_t e) {
    return (eb[e >> 5] >> (uint32_t)(e & 31)) & 1u;
}

// Make the edge map exact everywhere (used when it is handed back without the
// final search): rows of inactive vertices are zeroed, and in live rows the
// bits of entries whose other end is inactive are cleared.  One warp per vertex.
__global__ void __launch_bounds__(256)
k_materialize(int64_t n, const uint32_t *__restrict__ om, const int64_t *__restrict__ rp,
              const int32_t *__restrict__ col, uint32_t *ebits) {
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = (int)lane_id();
    for (int64_t v = gwarp; v < n; v += nwarps) {
        const int64_t beg = rp[v], end = rp[v + 1];
        if (beg == end) continue;
        if (om[v] == 0u) {
            clear_row<32>(ebits, beg, end, lane);
            continue;
        }
        for (int64_t e = beg + lane; e < end; e += 32) {
            if (ebit(ebits, e) && om[col[e]] == 0u)
                atomicAnd(&ebits[e >> 5], ~(1u << (uint32_t)(e & 31)));
        }
    }
}

__global__ void k_set_word(uint32_t *p, uint32_t v) { *p = v; }

// Per template vertex q: number of vertices with q in omega(v); slot 32: the
// total of |omega(v)|.  Inputs of the ordering features and the logs, and what
// says that a check has no root.  One pass over omega: lane q counts template
// vertex q, and 32 empty words (most of them, once LCC has run) cost a load and
// a vote (all 32 counters of every lane used to be added up for every word: 85
// us over 16M vertices, 18 us now).
__global__ void __launch_bounds__(256)
k_omega_hist(int64_t n, const uint32_t *__restrict__ om, int n0, unsigned long long *hist) {
    __shared__ unsigned int sh[kMaxT];
    if (threadIdx.x < kMaxT) sh[threadIdx.x] = 0u;
    __syncthreads();
    const int lane = (int)lane_id();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned int mine = 0;
    constexpr int U = 4;                             // words in flight per lane
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) - lane; b < n; b += stride * U) {
        uint32_t w[U];
#pragma unroll
        for (int j = 0; j < U; j++) {
            const int64_t v = b + j * stride + lane;
            w[j] = v < n ? __ldg(om + v) : 0u;
        }
#pragma unroll
        for (int j = 0; j < U; j++) {
            for (uint32_t any = __reduce_or_sync(FULL_MASK, w[j]); any; any &= any - 1u) {
                const int q = __ffs(any) - 1;
                const uint32_t m = __ballot_sync(FULL_MASK, (w[j] >> q) & 1u);
                if (lane == q) mine += __popc(m);
            }
        }
    }
    if (mine) atomicAdd(&sh[lane], mine);
    __syncthreads();
    if ((int)threadIdx.x < n0 && sh[threadIdx.x]) {
        atomicAdd(&hist[threadIdx.x], (unsigned long long)sh[threadIdx.x]);
        atomicAdd(&hist[kMaxT], (unsigned long long)sh[threadIdx.x]);
    }
}

// Per label: vertices (out[0..255]) and the entries in their rows (out[256..511]).
__global__ void __launch_bounds__(256)
k_label_hist(int64_t n, const int64_t *__restrict__ rp, const uint8_t *__restrict__ lab, unsigned long long *out) {
    __shared__ unsigned int cnt[256];
    __shared__ unsigned long long rows[256];
    cnt[threadIdx.x] = 0u;
    rows[threadIdx.x] = 0ull;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        atomicAdd(&cnt[lab[v]], 1u);
        atomicAdd(&rows[lab[v]], (unsigned long long)(rp[v + 1] - rp[v]));
    }
    __syncthreads();
    if (cnt[threadIdx.x]) atomicAdd(&out[threadIdx.x], (unsigned long long)cnt[threadIdx.x]);
    if (rows[threadIdx.x]) atomicAdd(&out[256 + threadIdx.x], rows[threadIdx.x]);
}

// Population counts for the result summary.
__global__ void __launch_bounds__(256)
k_count(int64_t n, const uint32_t *__restrict__ om, int64_t words, const uint32_t *__restrict__ eb,
        unsigned long long *out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long av = 0, ae = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) av += om[i] != 0u;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += stride) ae += __popc(eb[i]);
    for (int o = 16; o > 0; o >>= 1) {
        av += __shfl_xor_sync(FULL_MASK, av, o);
        ae += __shfl_xor_sync(FULL_MASK, ae, o);
    }
    if (lane_id() == 0) {
        if (av) atomicAdd(&out[0], av);
        if (ae) atomicAdd(&out[1], ae);
    }
}

}  // namespace ccpm

// ===========================================================================
// C ABI
// ===========================================================================

using namespace ccpm;

// LCC rounds queued per host round trip: the first group of a prune, and the
// later ones.  A round queued past the fixpoint costs two launches that return
// at once (3 us), a host round trip 20 us or more.
constexpr int kLccFirstGroup = 6, kLccGroup = 4;

// Passes of a search queued per host round trip (even: each batch of passes
// starts with the same of the two item buffers).  A search rarely needs more
// where the graph is small; a pass without items costs 3 us.
constexpr int kChain = 4;

// Device counters with a pinned host mirror, copied in one piece.
struct RoundGroup {
    RoundStats ring[kLccFirstGroup];
    unsigned long long hist[kMaxT + 1];
};
struct Control {
    RoundGroup grp[2];            // two groups of queued LCC rounds, and omega's histogram after each
    RoundStats init;              // k_init: sizes of the lists it makes
    RoundStats st;                // searches and checks
    PassCtl pass[kChain];
    unsigned long long cnt[2];    // population counts of the result
};

struct Workspace {
    bool ready = false;              // everything below that ws_make allocates is there
    bool lean = false;               // made without what a call can do without (ws_ensure)
    int64_t n = 0, m = 0, words = 0;
    int hub_deg = 0;
    uint32_t *om[2] = {nullptr, nullptr};
    uint16_t *nw[2] = {nullptr, nullptr};   // narrow copies of omega (up to 16 template vertices)
    uint32_t *ebits = nullptr;
    int32_t *small[2] = {nullptr, nullptr};
    int32_t *med[2] = {nullptr, nullptr};
    ChunkItem *chunk[2] = {nullptr, nullptr};
    int64_t chunk_cap = 0;
    HubAcc *acc = nullptr;
    int64_t acc_cap = 0;
    int32_t *roots = nullptr;
    uint32_t *sat = nullptr;
    SearchItem *items = nullptr;     // split search work
    int64_t items_cap = 0;
    SearchItem *items2 = nullptr;    // input of a further expansion
    SearchItem *spill_items = nullptr;   // items handed on by long searches
    int64_t spill_cap = 0;
    DevPlan *plans = nullptr;
    Control *ctl = nullptr, *ctl_h = nullptr;     // device, pinned host mirror
    RoundStats *st = nullptr, *st_h = nullptr;    // their search counters
    unsigned long long *cnt = nullptr, *cnt_h = nullptr;
    unsigned long long hist_h[kMaxT + 1] = {};    // the latest omega histogram
    // delta rounds (NULL where memory is short: no such rounds)
    uint32_t *dirty = nullptr;       // one bit per listed vertex, all zero between rounds
    int32_t *dsmall = nullptr, *dmed = nullptr;   // their lists
    ChunkItem *dchunk = nullptr;
    Change *chg = nullptr;           // changes of omega not passed on yet
    ChangePiece *chg_piece = nullptr;
    DevPlan *plans_h = nullptr;      // pinned staging for plan uploads
    cudaEvent_t ev[13] = {};
    // compacted rows (K4), two generations; allocated at the first compaction
    int64_t *sub_rp[2] = {nullptr, nullptr};
    int32_t *sub_col[2] = {nullptr, nullptr};
    uint32_t *sub_bits[2] = {nullptr, nullptr};
    int64_t sub_cap[2] = {0, 0};     // entries sub_col / sub_bits can hold
    uint32_t *deg = nullptr;         // entries each live vertex kept in its last evaluation
    uint8_t *sub_nlab[2] = {nullptr, nullptr};
    int32_t *sub_dslot[2] = {nullptr, nullptr};   // live vertex -> label-group directory slot
    int64_t *sub_gdir[2] = {nullptr, nullptr};
    int64_t gdir_cap[2] = {0, 0};
    unsigned int *slot_ctr = nullptr;
    uint32_t *piece_cnt = nullptr;   // kept entries per (piece, label rank) of long rows
    int64_t piece_cap = 0;
    void *scan_tmp = nullptr;
    size_t scan_tmp_bytes = 0;
    MlpScratch mlp;                  // scoring scratch of the learned order
};

struct ccpm_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int num_sms = 0;                      // SMs this context sizes its grids for
    int sm_total = 0;                     // SMs of the device
    std::string err;
    Workspace ws;                         // scratch of prunes issued on this context
    std::vector<ccpm_ctx *> workers;      // contexts of concurrent batch workers
    // row entries from which the LCC rounds go another way; tests lower them
    int64_t huge_rows = kHugeRows, inline_rows = kInlineRows, delta_rows = kDeltaRows;
    unsigned long long *label_hist = nullptr;   // counters of a graph load (borrowed arrays)
    cudaEvent_t load_ev = nullptr;        // ... and the default stream's state before it
    cudaEvent_t wait_ev = nullptr;        // batch workers: waits poll this event and yield
    // batch workers: grids are sized for sm_total / min(batch_share, workers
    // busy right now), so the last templates of a batch get the whole GPU back
    const std::atomic<int> *batch_busy = nullptr;
    int batch_share = 1;
};

// SMs a launch of this context sizes its grid for.
int grid_sms(const ccpm_ctx *ctx) {
    if (!ctx->batch_busy) return ctx->num_sms;
    const int busy = std::max(1, std::min(ctx->batch_share, ctx->batch_busy->load(std::memory_order_relaxed)));
    return std::max(1, ctx->sm_total / busy);
}

struct ccpm_graph {
    ccpm_ctx *ctx = nullptr;
    int64_t n = 0, m = 0;
    int64_t *rp = nullptr;
    int32_t *col = nullptr;
    uint8_t *lab = nullptr;
    bool borrowed = false;
    int64_t label_freq[256] = {};
    int64_t label_rows[256] = {};   // entries in the rows of each label's vertices
    int32_t *lcol = nullptr;      // rows grouped by neighbour label (built on first search)
    uint8_t *nlab = nullptr;
    std::mutex lrow_mu;           // concurrent batch workers build the grouped rows once
    int tuned_workers = 0;        // batch settings chosen by the autotuner (0: not tuned yet)
    int tuned_split = 0, tuned_short = 0, tuned_hub = 0, tuned_share = 0;
    double tuned_ms = 0.0;        // the chosen setting's time on the tuning slice
    std::atomic<int> prunes{0};   // prunes started on this graph
    std::atomic<int> listings{0};
    std::atomic<bool> lrows_ready{false};   // lcol/nlab built (read without the lock)
    uint8_t *elab = nullptr;      // label of each entry's neighbour, CSR order (built on first use)
    uint8_t *edge_lab = nullptr;  // edge label of each entry (ccpm_graph_set_edge_labels), or none
    bool edge_lab_borrowed = false;
};

struct ccpm_tmpl {
    ccpm_ctx *ctx = nullptr;
    Template t;
};

struct ccpm_result {
    ccpm_graph *g = nullptr;
    uint64_t tmpl_fp = 0;           // fingerprint of the template it was made for
    uint32_t *om = nullptr;
    uint32_t *eb = nullptr;
    ccpm_counts counts{};
    std::vector<int32_t> phase_rounds;
    std::vector<ccpm_constraint_log> logs;
};

namespace {

// Every CUDA failure is reported through here, so the runtime's record of it is
// cleared here: left standing, the next call would find it after its first
// launch and fail for it.
int set_err(ccpm_ctx *ctx, int code, const std::string &msg) {
    if (code == CCPM_ENOMEM || code == CCPM_ECUDA) cudaGetLastError();
    if (ctx) ctx->err = msg;
    return code;
}

// Wait for the work queued on the context's stream.  A batch worker polls an
// event and yields its core between polls: the runtime's own wait spins, and
// a dozen workers spinning at once would hold the host cores that the other
// workers need to launch their next kernels (a worker whose GPU work is done
// could then wait a scheduler time slice for a core).
cudaError_t ctx_sync(ccpm_ctx *ctx) {
    if (!ctx->wait_ev) return cudaStreamSynchronize(ctx->stream);
    cudaError_t e = cudaEventRecord(ctx->wait_ev, ctx->stream);
    if (e != cudaSuccess) return e;
    while ((e = cudaEventQuery(ctx->wait_ev)) == cudaErrorNotReady) std::this_thread::yield();
    return e;
}

// FNV-1a 64 over a byte range (fingerprints and the checksum of saved states)
uint64_t fnv1a(const void *p, size_t len, uint64_t h = 0xcbf29ce484222325ull) {
    const unsigned char *b = (const unsigned char *)p;
    for (size_t i = 0; i < len; i++) { h ^= b[i]; h *= 0x100000001b3ull; }
    return h;
}

// the template as labels and sorted edge list: equal for the same template
// however its edges were listed
uint64_t tmpl_fingerprint(const Template &t) {
    std::vector<std::pair<int, int>> e = t.edges;
    std::sort(e.begin(), e.end());
    uint64_t h = fnv1a(&t.n0, sizeof(t.n0));
    h = fnv1a(t.labels, (size_t)t.n0, h);
    for (auto &x : e) { int32_t ab[2] = {x.first, x.second}; h = fnv1a(ab, sizeof(ab), h); }
    return h;
}

uint64_t graph_fingerprint(const ccpm_graph &g) {
    uint64_t h = fnv1a(&g.n, sizeof(g.n));
    h = fnv1a(&g.m, sizeof(g.m), h);
    return fnv1a(g.label_freq, sizeof(g.label_freq), h);
}

#define CU(ctx, call)                                                                 \
    do {                                                                              \
        cudaError_t e_ = (call);                                                      \
        if (e_ != cudaSuccess)                                                        \
            return set_err((ctx), e_ == cudaErrorMemoryAllocation ? CCPM_ENOMEM : CCPM_ECUDA, \
                           std::string(#call) + ": " + cudaGetErrorString(e_));       \
    } while (0)

template <typename T>
int dalloc(ccpm_ctx *ctx, T **p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    cudaError_t e = cudaMalloc((void **)p, sizeof(T) * count);
    if (e != cudaSuccess) {
        *p = nullptr;
        return set_err(ctx, CCPM_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    }
    return CCPM_OK;
}

void ws_free(Workspace &w) {
    cudaFree(w.om[0]); cudaFree(w.om[1]); cudaFree(w.nw[0]); cudaFree(w.nw[1]); cudaFree(w.ebits);
    cudaFree(w.small[0]); cudaFree(w.small[1]); cudaFree(w.med[0]); cudaFree(w.med[1]);
    cudaFree(w.chunk[0]); cudaFree(w.chunk[1]); cudaFree(w.acc); cudaFree(w.roots);
    cudaFree(w.sat); cudaFree(w.items); cudaFree(w.items2); cudaFree(w.spill_items); cudaFree(w.plans); cudaFree(w.ctl);
    if (w.ctl_h) cudaFreeHost(w.ctl_h);
    cudaFree(w.dirty); cudaFree(w.dsmall); cudaFree(w.dmed); cudaFree(w.dchunk); cudaFree(w.chg); cudaFree(w.chg_piece);
    if (w.plans_h) cudaFreeHost(w.plans_h);
    for (auto &e : w.ev) if (e) cudaEventDestroy(e);
    for (int i = 0; i < 2; i++) { cudaFree(w.sub_rp[i]); cudaFree(w.sub_col[i]); cudaFree(w.sub_bits[i]); }
    for (int i = 0; i < 2; i++) { cudaFree(w.sub_nlab[i]); cudaFree(w.sub_dslot[i]); cudaFree(w.sub_gdir[i]); }
    cudaFree(w.slot_ctr);
    cudaFree(w.deg); cudaFree(w.piece_cnt); cudaFree(w.scan_tmp);
    mlp_scratch_free(w.mlp);
    w = Workspace{};
}

int ws_make(ccpm_ctx *ctx, ccpm_graph *g, int hub_deg, bool lean) {
    Workspace &w = ctx->ws;
    w.lean = lean;
    w.n = g->n;
    w.m = g->m;
    w.words = (g->m + 31) / 32;
    w.hub_deg = hub_deg;
    w.chunk_cap = 2 * (g->m / hub_deg) + 16;
    w.acc_cap = g->m / hub_deg + 16;
    int rc;
    if ((rc = dalloc(ctx, &w.om[0], (size_t)g->n))) return rc;
    if ((rc = dalloc(ctx, &w.om[1], (size_t)g->n))) return rc;
    if ((rc = dalloc(ctx, &w.nw[0], (size_t)g->n))) return rc;
    if ((rc = dalloc(ctx, &w.nw[1], (size_t)g->n))) return rc;
    if ((rc = dalloc(ctx, &w.ebits, (size_t)w.words + 1))) return rc;
    for (int i = 0; i < 2; i++) {
        if ((rc = dalloc(ctx, &w.small[i], (size_t)g->n))) return rc;
        if ((rc = dalloc(ctx, &w.med[i], (size_t)g->n))) return rc;
        if ((rc = dalloc(ctx, &w.chunk[i], (size_t)w.chunk_cap))) return rc;
    }
    if ((rc = dalloc(ctx, &w.acc, (size_t)w.acc_cap))) return rc;
    if ((rc = dalloc(ctx, &w.roots, (size_t)g->n))) return rc;
    if ((rc = dalloc(ctx, &w.sat, (size_t)g->n))) return rc;
    w.items_cap = std::min<int64_t>(std::max<int64_t>(g->m, (int64_t)1 << 22), (int64_t)1 << 24) >> (lean ? 1 : 0);
    if ((rc = dalloc(ctx, &w.items, (size_t)w.items_cap))) return rc;
    if ((rc = dalloc(ctx, &w.items2, (size_t)kExpandBelow))) return rc;
    w.spill_cap = std::max<int64_t>(w.items_cap / 4, (int64_t)1 << (lean ? 19 : 20));
    if ((rc = dalloc(ctx, &w.spill_items, (size_t)w.spill_cap))) return rc;
    if ((rc = dalloc(ctx, &w.plans, (size_t)kMaxPlans))) return rc;
    if ((rc = dalloc(ctx, &w.ctl, 1))) return rc;
    CU(ctx, cudaMallocHost((void **)&w.ctl_h, sizeof(Control)));
    w.st = &w.ctl->st;
    w.st_h = &w.ctl_h->st;
    w.cnt = w.ctl->cnt;
    w.cnt_h = w.ctl_h->cnt;
    if (!lean) {
        if ((rc = dalloc(ctx, &w.dirty, (size_t)g->n / 32 + 1))) return rc;
        if ((rc = dalloc(ctx, &w.dsmall, (size_t)g->n))) return rc;
        if ((rc = dalloc(ctx, &w.dmed, (size_t)g->n))) return rc;
        if ((rc = dalloc(ctx, &w.dchunk, (size_t)w.chunk_cap))) return rc;
        if ((rc = dalloc(ctx, &w.chg, (size_t)g->n))) return rc;
        if ((rc = dalloc(ctx, &w.chg_piece, (size_t)w.chunk_cap))) return rc;
    }
    if ((rc = dalloc(ctx, &w.deg, (size_t)g->n))) return rc;
    CU(ctx, cudaMallocHost((void **)&w.plans_h, kMaxPlans * sizeof(DevPlan)));
    CU(ctx, cudaMemsetAsync(w.acc, 0, sizeof(HubAcc) * (size_t)w.acc_cap, ctx->stream));
    for (auto &e : w.ev) CU(ctx, cudaEventCreate(&e));
    w.ready = true;
    return CCPM_OK;
}

// The context's workspace for this graph: all of it, or, if something could not
// be had, nothing.  What a call can do without is left out where memory is short
// (lean): half of the item lists (searches with more items run one warp per root),
// and the lists of delta rounds (every round is a full one).  That is 16 B a
// vertex and up to 0.7 GB less.
int ws_ensure(ccpm_ctx *ctx, ccpm_graph *g, int hub_deg, bool lean = false) {
    Workspace &w = ctx->ws;
    if (w.ready && (w.lean || !lean) && w.hub_deg == hub_deg && w.n == g->n && w.m == g->m) return CCPM_OK;
    ws_free(w);
    int rc = ws_make(ctx, g, hub_deg, lean);
    if (rc) ws_free(w);
    if (rc == CCPM_ENOMEM && !lean) return ws_ensure(ctx, g, hub_deg, true);
    return rc;
}

// Something beside the workspace did not fit: true if a smaller workspace has
// taken its place, so that the caller can try again.
bool ws_shrink(ccpm_ctx *ctx, ccpm_graph *g) {
    return ctx->ws.ready && !ctx->ws.lean && ws_ensure(ctx, g, ctx->ws.hub_deg, true) == CCPM_OK;
}

// Label-grouped copy of the rows: a stable segmented sort of every row by the
// neighbours' labels keeps ids ascending inside each label group.  Built once
// per graph, the first time a search needs it.
int ensure_label_rows(ccpm_ctx *ctx, ccpm_graph *g) {
    std::lock_guard<std::mutex> lock(g->lrow_mu);
    if (g->lcol || g->m == 0) return CCPM_OK;
    int rc;
    if ((rc = dalloc(ctx, &g->lcol, (size_t)g->m))) return rc;
    if ((rc = dalloc(ctx, &g->nlab, (size_t)g->m))) {
        cudaFree(g->lcol);
        g->lcol = nullptr;
        return rc;
    }
    // a counting sort of every row by neighbour label; its keys are the entry
    // labels (gathered here into a temporary array when they are not built:
    // the sort reads them twice)
    uint8_t *keys = g->elab;
    if (!keys) {
        if ((rc = dalloc(ctx, &keys, (size_t)g->m))) {
            cudaFree(g->lcol); cudaFree(g->nlab);
            g->lcol = nullptr; g->nlab = nullptr;
            return rc;
        }
        const int gg = (int)std::min<int64_t>((g->m + 255) / 256, (int64_t)ctx->num_sms * 8);
        k_gather_labels<<<gg, 256, 0, ctx->stream>>>(g->m, g->col, g->lab, keys);
    }
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((g->n + 7) / 8, (int64_t)grid_sms(ctx) * 8));
    k_label_sort<<<grid, 256, 0, ctx->stream>>>(g->n, g->rp, g->col, g->lab, keys, g->nlab, g->lcol);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (keys != g->elab) cudaFree(keys);
    if (e != cudaSuccess) {
        cudaFree(g->lcol); cudaFree(g->nlab);
        g->lcol = nullptr; g->nlab = nullptr;
        return set_err(ctx, CCPM_ECUDA, std::string("label-grouped rows: ") + cudaGetErrorString(e));
    }
    g->lrows_ready.store(true);
    return CCPM_OK;
}

// The label of every entry's neighbour in CSR order (one byte per entry):
// the first LCC round after init reads it instead of the column index and the
// neighbour's label.  Built once per graph, the first time a first round
// covers a large share of the entries.
int ensure_entry_labels(ccpm_ctx *ctx, ccpm_graph *g) {
    std::lock_guard<std::mutex> lock(g->lrow_mu);
    if (g->elab || g->m == 0) return CCPM_OK;
    uint8_t *el = nullptr;
    int rc;
    if ((rc = dalloc(ctx, &el, (size_t)g->m + 16))) return rc;    // read 16 at a time
    int grid = (int)std::min<int64_t>((g->m + 255) / 256, (int64_t)ctx->num_sms * 8);
    k_gather_labels<<<grid, 256, 0, ctx->stream>>>(g->m, g->col, g->lab, el);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) {
        cudaFree(el);
        return set_err(ctx, CCPM_ECUDA, std::string("entry labels: ") + cudaGetErrorString(e));
    }
    g->elab = el;
    return CCPM_OK;
}

// For searches that do not hand work on to idle warps (a caller's own budget,
// search_split < 0): split the work level by level while there is too little to fill
// the GPU (and the items still leave positions to place).
int expand_more(ccpm_ctx *ctx, Workspace &w, SearchArgs &a, int max_depth, int64_t &launches) {
    for (int depth = 2; depth < max_depth && depth < kItemMaxDepth; depth++) {
        if (a.n_items <= 0 || a.n_items >= kExpandBelow) return CCPM_OK;
        CU(ctx, cudaMemcpyAsync(w.items2, w.items, sizeof(SearchItem) * (size_t)a.n_items, cudaMemcpyDeviceToDevice,
                                ctx->stream));
        CU(ctx, cudaMemsetAsync(&w.st->n_items, 0, sizeof(unsigned int), ctx->stream));
        launches++;
        int grid = (int)std::max<int64_t>(1, std::min<int64_t>((a.n_items + 3) / 4, (int64_t)grid_sms(ctx) * 16));
        k_expand_next<<<grid, 128, 0, ctx->stream>>>(a, w.items2, a.n_items);
        CU(ctx, cudaGetLastError());
        CU(ctx, cudaMemcpyAsync(w.st_h, w.st, sizeof(RoundStats), cudaMemcpyDeviceToHost, ctx->stream));
        CU(ctx, ctx_sync(ctx));
        const unsigned int n2 = w.st_h->n_items;
        if ((int64_t)n2 > w.items_cap) {
            // more than fit: the items stay at the level they were at
            w.st_h->n_items = (unsigned int)a.n_items;
            CU(ctx, cudaMemcpyAsync(w.items, w.items2, sizeof(SearchItem) * (size_t)a.n_items, cudaMemcpyDeviceToDevice,
                                    ctx->stream));
            CU(ctx, cudaMemcpyAsync(&w.st->n_items, &w.st_h->n_items, sizeof(unsigned int), cudaMemcpyHostToDevice,
                                    ctx->stream));
            return CCPM_OK;
        }
        a.n_items = n2;
    }
    return CCPM_OK;
}

// Grid of one resident wave for a 256-thread grid-stride kernel.
template <typename K>
int lcc_grid(ccpm_ctx *ctx, K kernel, int64_t warps) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0) != cudaSuccess || per_sm < 1)
        per_sm = 4;
    int64_t need = (warps + 7) / 8;
    return (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)grid_sms(ctx) * per_sm));
}

int grid_for(ccpm_ctx *ctx, int64_t work_items, int per_block, int blocks_per_sm) {
    int64_t need = (work_items + per_block - 1) / per_block;
    int64_t cap = (int64_t)grid_sms(ctx) * blocks_per_sm;
    if (need < 1) need = 1;
    return (int)std::min(need, cap);
}

// Windows a search scans before it hands the rest of its work to other warps.
constexpr uint64_t kSpillAfter = 2048;

// Read all counters.
int read_control(ccpm_ctx *ctx, Workspace &w) {
    CU(ctx, cudaMemcpyAsync(w.ctl_h, w.ctl, sizeof(Control), cudaMemcpyDeviceToHost, ctx->stream));
    CU(ctx, ctx_sync(ctx));
    return CCPM_OK;
}

// Zero the counters of a search.
int clear_search(ccpm_ctx *ctx, Workspace &w) {
    CU(ctx, cudaMemsetAsync(w.st, 0, sizeof(RoundStats) + sizeof(PassCtl) * kChain, ctx->stream));
    return CCPM_OK;
}
static_assert(offsetof(Control, pass) == offsetof(Control, st) + sizeof(RoundStats), "cleared together");

// How a search runs.  kind 0: NLCC existence (k_nlcc_items), 1: final count, 2:
// final count and mark, 3: count and list, 4: per-entry existence
// (k_edge_search).  split: windows a search scans before it hands its rest on
// in any case (0: never); starve: it also does when other warps are idle.
struct SearchMode {
    int kind;
    uint64_t split;
    bool starve;
};

// Queue kChain passes over the items in a.items (a.n_items, or on the device):
// each but the first runs over what the one before handed on.
int queue_passes(ccpm_ctx *ctx, Workspace &w, SearchArgs &a, const SearchMode &m, int64_t &launches) {
    SearchItem *bufs[2] = {w.items, w.spill_items};
    const int64_t caps[2] = {w.items_cap, w.spill_cap};
    a.spill_after = m.split;
    a.starve = m.starve ? 1 : 0;
    // known item counts: no more warps than items
    const int gi = a.n_items >= 0 ? grid_for(ctx, a.n_items * 32, 128, 16) : grid_sms(ctx) * 16;
    for (int p = 0; p < kChain; p++) {
        a.items = bufs[p & 1];
        a.spill = bufs[(p & 1) ^ 1];
        a.spill_cap = caps[(p & 1) ^ 1];
        a.ctl = w.ctl->pass + p;
        a.ctl_prev = p ? a.ctl - 1 : nullptr;
        const int grid = p ? grid_sms(ctx) * 16 : gi;
        launches++;
        if (m.kind == 0) k_nlcc_items<<<grid, 128, 0, ctx->stream>>>(a);
        else if (m.kind == 1) k_final_items<kCount><<<grid, 128, 0, ctx->stream>>>(a);
        else if (m.kind == 2) k_final_items<kMark><<<grid, 128, 0, ctx->stream>>>(a);
        else if (m.kind == 3) k_final_items<kList><<<grid, 128, 0, ctx->stream>>>(a);
        else k_edge_search<<<grid, 128, 0, ctx->stream>>>(a);
        CU(ctx, cudaGetLastError());
    }
    a.items = w.items;
    a.spill = nullptr;
    a.spill_after = 0;
    a.starve = 0;
    a.ctl = w.ctl->pass;
    a.ctl_prev = nullptr;
    return CCPM_OK;
}

// Queue the item list of a search over a.roots and its first passes, with no
// host round trip (searches that do not hand on to idle warps: one per level
// of the expansion).  The counters were cleared before.
int queue_search(ccpm_ctx *ctx, Workspace &w, SearchArgs &a, const SearchMode &m, int max_depth, int64_t &launches) {
    a.ctl = w.ctl->pass;
    a.ctl_prev = nullptr;
    launches++;
    const int64_t most = a.n_roots >= 0 ? a.n_roots : (int64_t)1 << 40;
    k_expand<<<grid_for(ctx, most * 32, 256, 8), 256, 0, ctx->stream>>>(a);
    CU(ctx, cudaGetLastError());
    a.n_items = -1;
    if (!m.starve) {
        int rc = read_control(ctx, w);
        if (rc) return rc;
        a.n_items = w.st_h->n_items;
        if (a.n_items > w.items_cap) a.n_items = -1;         // more than fit: the passes do nothing
        else if ((rc = expand_more(ctx, w, a, max_depth, launches))) return rc;
    }
    return queue_passes(ctx, w, a, m, launches);
}

// Was a queued search complete?  (Its counters have been read.)
bool search_complete(const Workspace &w, const SearchMode &m) {
    if (w.st_h->n_items > w.items_cap) return false;
    if (m.kind >= 1 && m.kind <= 3 && w.st_h->overflow) return true;    // past the cap (or out of budget): stopped
    return w.ctl_h->pass[kChain - 1].handed_on() == 0;
}

// Complete a queued search whose counters have been read: further passes over
// what was handed on (an item handed on is deeper, or holds fewer candidates
// of the same position, than the one it came from, so the passes end), or, if
// its items did not fit, one warp per root.
int finish_search(ccpm_ctx *ctx, Workspace &w, SearchArgs &a, const SearchMode &m, int64_t &launches) {
    int rc;
    if (w.st_h->n_items > w.items_cap && m.kind != 4) {
        CU(ctx, cudaMemsetAsync(w.ctl->pass, 0, sizeof(PassCtl), ctx->stream));
        launches++;
        a.n_roots = w.st_h->n_roots;
        a.ctl = w.ctl->pass;
        const int grid = grid_for(ctx, a.n_roots * 32, 128, 16);
        if (m.kind == 0) k_nlcc_search<<<grid, 128, 0, ctx->stream>>>(a);
        else if (m.kind == 1) k_final_search<kCount><<<grid, 128, 0, ctx->stream>>>(a);
        else if (m.kind == 2) k_final_search<kMark><<<grid, 128, 0, ctx->stream>>>(a);
        else k_final_search<kList><<<grid, 128, 0, ctx->stream>>>(a);
        CU(ctx, cudaGetLastError());
        return read_control(ctx, w);
    }
    while (!search_complete(w, m)) {
        a.n_items = w.ctl_h->pass[kChain - 1].handed_on();
        CU(ctx, cudaMemsetAsync(w.ctl->pass, 0, sizeof(PassCtl) * kChain, ctx->stream));
        if ((rc = queue_passes(ctx, w, a, m, launches))) return rc;
        if ((rc = read_control(ctx, w))) return rc;
    }
    return CCPM_OK;
}

// Ordering features of one constraint in the current state (alive[q] =
// vertices with q in omega, total = sum of |omega|), step = constraints run.
void constraint_features(const Template &t, const HostConstraint &c, const unsigned long long *alive,
                         unsigned long long total, int step, int n_constraints, float *f) {
    for (int i = 0; i < CCPM_MLP_IN; i++) f[i] = 0.f;
    f[c.kind] = 1.f;
    const int nv = __builtin_popcount(c.vmask), ne = (int)c.edges.size(), nh = __builtin_popcount(c.hmask);
    f[5] = nv / 8.f;
    f[6] = ne / 8.f;
    f[7] = nh / 8.f;
    double sh = 0, sv = 0, mn = 1e300, mx = 0;
    for (int q = 0; q < t.n0; q++) {
        if ((c.hmask >> q) & 1u) sh += (double)alive[q];
        if ((c.vmask >> q) & 1u) {
            sv += (double)alive[q];
            mn = std::min(mn, (double)alive[q]);
            mx = std::max(mx, (double)alive[q]);
        }
    }
    if (mn > 1e299) mn = 0;
    f[8] = (float)(std::log2(1.0 + sh) / 32.0);
    f[9] = (float)(std::log2(1.0 + mn) / 32.0);
    f[10] = (float)(std::log2(1.0 + mx) / 32.0);
    f[11] = (float)(std::log2(1.0 + sv) / 32.0);
    f[12] = (float)nv / (float)t.n0;
    f[13] = (float)(ne - nv + 1) / 4.f;
    f[14] = n_constraints ? (float)step / (float)n_constraints : 0.f;
    f[15] = (float)(std::log2(1.0 + (double)total) / 32.0);
}

struct Pipeline {
    ccpm_ctx *ctx;
    ccpm_graph *g;
    const Template *t;
    DevTmpl dt;
    int cur = 0;            // omega buffer holding round-k state
    bool dense = true;      // next round is the first after init: all edge bits set
    bool from_labels = false;  // next round is the first after a fresh init: omega = initial label mask
    LabelMask lm0{};        // label -> initial omega (Alg. 3)
    int li = 0;             // frontier list parity
    int64_t n_small = 0, n_med = 0, n_chunk = 0;
    int64_t scanned = 0;
    int64_t windows = 0;
    int64_t rows = 0, alive = 0, launches = 0, lcc_launches = 0;
    int64_t alg_bytes = 0, kernel_bytes = 0, first_entries = 0, lcc_rounds_run = 0;
    double ms_first = 0.0;
    double ms_lcc_kernel = 0.0;
    double ms_search_kernel = 0.0;
    int64_t search_launches = 0, nlcc_entries = 0;
    int maxc = 0;
    int short_max = kSmallDeg;      // rows up to this length take the flat short-row path
    bool eta_off = false;           // ablation: no edge elimination
    int nw_bytes = 0;               // width of the narrow copy of omega (0: none)
    const uint8_t *elab = nullptr;  // the graph's entry labels for the first round (or none)
    int64_t first_rows = 0;         // entries in the rows of the initially active vertices
    // rows the LCC rounds read: the graph's, or the latest compacted ones (K4)
    const int64_t *lrp = nullptr;
    const int32_t *lcol = nullptr;
    uint32_t *lbits = nullptr;
    int gen = -1;                   // compacted generation in use, -1 = full rows
    int compact_mode = 0;           // options.compact
    int searches_ahead = 0;         // non-local constraints not yet checked
    int64_t compactions = 0;
    const uint8_t *lnlab = nullptr; // labels of lcol (compacted rows are label-grouped)
    const int32_t *ldslot = nullptr;  // their label-group directory
    const int64_t *lgdir = nullptr;
    int lnrank = 0;
    uint8_t llab_rank[256] = {};
    // the state after the latest round: entries still active, entries in the
    // rows of the active vertices, active vertices
    int64_t last_kept = -1, last_rows = -1, last_alive = 0;
    bool synced = true;             // the lists hold every live vertex, both omega buffers are equal

    int read_stats() { return read_control(ctx, ctx->ws); }

    // One LCC round.  slot: its counters; prev (nullable): the counters of the
    // round before, from which the round reads its list sizes and whether there
    // is anything to do on the device (without: the host's sizes, and the round
    // runs only if the counters `gate` (nullable) say that something changed).  c, l: the
    // omega and list buffers it reads (the host flips cur / li only once a
    // group of queued rounds is done, by the number of rounds that ran).
    int launch_round(RoundStats *slot, const RoundStats *prev, const RoundStats *gate, int c, int l, bool delta) {
        launches++;
        lcc_launches++;
        if (maxc > 4 || nw_bytes != 1 || first_rows < ctx->huge_rows)
            return launch_small(slot, prev, gate, c, l, delta);
        Workspace &w = ctx->ws;
        RowArgs a = row_args(slot);
        a.om = w.om[c];
        a.nw = w.nw[c];
        a.om_out[0] = w.om[c ^ 1];
        a.nw_out[0] = w.nw[c ^ 1];
        a.small_in = delta ? w.dsmall : w.small[l];
        a.med_in = delta ? w.dmed : w.med[l];
        a.chunk_in = delta ? w.dchunk : w.chunk[l];
        // a full round's lists were written by the round before, a delta
        // round's by k_push into its own counters
        a.sizes = delta ? slot : prev;
        a.n_small = n_small;
        a.n_med = n_med;
        a.n_chunk = n_chunk;
        a.gate = prev ? prev : gate;
        a.small_out = w.small[l ^ 1];
        a.med_out = w.med[l ^ 1];
        a.chunk_out = w.chunk[l ^ 1];
        // a queued round does not know its sizes: one full resident wave
        const int64_t warps = a.sizes ? (int64_t)1 << 40 : n_small + n_med + n_chunk;
        from_labels = dense = false;
#define CCPM_ROWS(C, M) \
    k_rows<C, M, kByByte><<<lcc_grid(ctx, k_rows<C, M, kByByte>, warps), 256, 0, ctx->stream>>>(a, dt)
        if (maxc == 0) { if (delta) CCPM_ROWS(0, kDelta); else CCPM_ROWS(0, kFull); }
        else { if (delta) CCPM_ROWS(4, kDelta); else CCPM_ROWS(4, kFull); }
#undef CCPM_ROWS
        CU(ctx, cudaGetLastError());
        return CCPM_OK;
    }

    RowArgs row_args(RoundStats *slot) const {
        Workspace &w = ctx->ws;
        RowArgs a{};
        a.n = g->n;
        a.m = gen < 0 ? g->m : INT64_MAX;            // compacted rows: room past their end
        a.rp = lrp;
        a.col = lcol;
        a.col_vec = ((uintptr_t)lcol & 15) == 0;
        a.lab = g->lab;
        a.elab = elab;
        a.nw_bytes = nw_bytes;
        a.ebits = lbits;
        a.deg = w.deg;
        a.dirty = w.dirty;
        a.chg = w.chg;
        a.chg_piece = w.chg_piece;
        a.acc = w.acc;
        a.st = slot;
        a.hub_deg = w.hub_deg;
        a.short_max = short_max;
        a.eta_off = eta_off ? ~0u : 0u;
        a.lm = lm0;
        return a;
    }

    // A round of a template with more than eight vertices or four multiplicity
    // classes, or of one that starts from fewer than kHugeRows entries.
    int launch_small(RoundStats *slot, const RoundStats *prev, const RoundStats *gate, int c, int l, bool delta) {
        Workspace &w = ctx->ws;
        LccArgs a;
        a.rp = lrp;
        a.col = lcol;
        a.om_cur = w.om[c];
        a.om_next = w.om[c ^ 1];
        a.ebits = lbits;
        a.small_in = delta ? w.dsmall : w.small[l];
        a.med_in = delta ? w.dmed : w.med[l];
        a.chunk_in = delta ? w.dchunk : w.chunk[l];
        a.n_small = n_small;
        a.n_med = n_med;
        a.n_chunk = n_chunk;
        a.small_out = w.small[l ^ 1];
        a.med_out = w.med[l ^ 1];
        a.chunk_out = w.chunk[l ^ 1];
        a.acc = w.acc;
        a.st = slot;
        a.prev = prev;
        a.gate = gate;
        a.resident_warps = grid_sms(ctx) * 32;
        a.hub_deg = w.hub_deg;
        a.deg = w.deg;
        a.dirty = w.dirty;
        a.chg = w.chg;
        a.chg_piece = w.chg_piece;
        a.lab0 = from_labels ? g->lab : nullptr;
        a.elab = from_labels ? elab : nullptr;
        a.sparse = (!dense && gen < 0) ? 1 : 0;
        a.lmask = lm0;
        a.eta_off = eta_off ? ~0u : 0u;
        a.nw_bytes = nw_bytes;
        a.nw_cur = w.nw[c];
        a.nw_next = w.nw[c ^ 1];
        from_labels = false;
        // prefetch units: large enough to hide the per-vertex loads, small
        // enough that every resident warp gets several of them
        const int64_t resident = (int64_t)grid_sms(ctx) * 32;
        a.med_chunk = (int)std::max<int64_t>(1, std::min<int64_t>(16, n_med / (4 * resident)));
        // a queued round does not know its sizes: one full resident wave
        const int64_t warps = prev ? ((int64_t)1 << 40)
                                   : n_chunk + (n_med + a.med_chunk - 1) / a.med_chunk + n_small;
        // one resident wave: grid-stride work is split evenly over warps that all run at once
#define CCPM_LAUNCH_LCC(C, M) k_lcc_round<C, M><<<lcc_grid(ctx, k_lcc_round<C, M>, warps), 256, 0, ctx->stream>>>(a, dt)
        if (maxc == 0 && delta) CCPM_LAUNCH_LCC(0, kDelta);
        else if (maxc == 0) CCPM_LAUNCH_LCC(0, kFull);
        else if (maxc <= 4 && delta) CCPM_LAUNCH_LCC(4, kDelta);
        else if (maxc <= 4) CCPM_LAUNCH_LCC(4, kFull);
        else if (delta) CCPM_LAUNCH_LCC(kMaxCls, kDelta);
        else if (dense) CCPM_LAUNCH_LCC(kMaxCls, kDense);
        else CCPM_LAUNCH_LCC(kMaxCls, kFull);
#undef CCPM_LAUNCH_LCC
        dense = false;      // only the first round after init sees every bit set
        CU(ctx, cudaGetLastError());
        return CCPM_OK;
    }

    // Fresh prunes start with k_first_round unless the template has more
    // multiplicity classes than its packed counts hold.
    bool first_kernel() const { return dense && from_labels && gen < 0 && maxc <= 4; }

    // The first round of a fresh prune (no initialisation runs before it).
    int launch_first(RoundStats *slot) {
        Workspace &w = ctx->ws;
        RowArgs a = row_args(slot);
        a.guard = 1;
        a.inline_long = first_rows < ctx->inline_rows ? 1 : 0;
        for (int i = 0; i < 2; i++) {
            a.om_out[i] = w.om[i];
            a.nw_out[i] = w.nw[i];
        }
        a.small_out = w.small[li ^ 1];
        a.med_out = w.med[li ^ 1];
        a.chunk_out = w.chunk[li ^ 1];
        a.first_med = w.med[li];
        a.first_chunk = w.chunk[li];
        a.first_sizes = &w.ctl->init;
        a.med_in = w.med[li];
        a.chunk_in = w.chunk[li];
        a.sizes = &w.ctl->init;
        launches += 2;
        lcc_launches++;
        from_labels = dense = false;
#define CCPM_LAUNCH_FIRST(C, F)                                                                              \
    do {                                                                                                     \
        k_first_round<C, F><<<lcc_grid(ctx, k_first_round<C, F>, g->n), 256, 0, ctx->stream>>>(a, dt);       \
        k_rows<C, kFirst, F><<<lcc_grid(ctx, k_rows<C, kFirst, F>,                                           \
                                        first_rows / (a.inline_long ? kWarpRow : kGroupRow) + 1), 256, 0,    \
                               ctx->stream>>>(a, dt);                                                        \
    } while (0)
        if (elab) {
            if (maxc == 0) CCPM_LAUNCH_FIRST(0, kByEntry); else CCPM_LAUNCH_FIRST(4, kByEntry);
        } else {
            if (maxc == 0) CCPM_LAUNCH_FIRST(0, kByLabel); else CCPM_LAUNCH_FIRST(4, kByLabel);
        }
#undef CCPM_LAUNCH_FIRST
        CU(ctx, cudaGetLastError());
        return CCPM_OK;
    }

    // Pass the changes of a round (prev) on: the lists of the delta round whose
    // counters are `slot`.  lists: the round was a full one that read the omega
    // buffer c ^ 1 and left its vertices in the lists l.
    int launch_push(RoundStats *slot, const RoundStats *prev, int c, int l, bool lists) {
        Workspace &w = ctx->ws;
        PushArgs a;
        a.rp = lrp;
        a.col = lcol;
        a.bits = lbits;
        a.om = w.om[c];
        a.nw = w.nw[c];
        a.nw_bytes = nw_bytes;
        a.om_old = w.om[c ^ 1];
        a.small_in = w.small[l];
        a.med_in = w.med[l];
        a.chunk_in = w.chunk[l];
        a.chg = w.chg;
        a.chg_piece = w.chg_piece;
        a.prev = prev;
        a.dirty = w.dirty;
        a.small_out = w.dsmall;
        a.med_out = w.dmed;
        a.chunk_out = w.dchunk;
        a.st = slot;
        a.hub_deg = w.hub_deg;
        a.short_max = short_max;
        launches++;
        const int grid = grid_for(ctx, (int64_t)1 << 40, 256, 8);
        if (lists) k_push<true><<<grid, 256, 0, ctx->stream>>>(a);
        else k_push<false><<<grid, 256, 0, ctx->stream>>>(a);
        CU(ctx, cudaGetLastError());
        return CCPM_OK;
    }

    // LCC to fixpoint; returns rounds via *rounds.  Rounds are queued in groups
    // with one host round trip per group: each reads what it needs from the
    // counters of the round before (the first: of the initialisation, or of the
    // non-local check queued before it, whose changes are in the Change list),
    // and rounds queued after the fixpoint, or after a check that changed
    // nothing, return at once.  After each group omega's histogram is taken if
    // asked for (w.hist_h).  A prune's first rounds (two, or one
    // from a saved state) evaluate every active vertex, as nearly all of them
    // change; where the rows are large (use_deltas) the later ones are delta
    // rounds.  With options.compact > 0 every round is a full one and the rows
    // may be compacted between groups.
    int lcc(int64_t *rounds, bool initial, bool want_hist) {
        Workspace &w = ctx->ws;
        int64_t r = 0;
        const bool deltas = use_deltas(initial ? first_rows : last_rows);
        int full_left = initial ? (dense ? 2 : 1) : 0;
        const RoundStats *src = initial ? &w.ctl->init : (deltas ? w.st : nullptr);
        const RoundStats *gate = initial ? nullptr : w.st;
        const bool was_synced = synced;
        if (!initial && !deltas && !synced) {
            // earlier delta rounds left the lists and the other omega buffer
            // behind: rebuild them if the check changed anything (k_init then
            // marks its counters as changed)
            int rc = rebucket(lrp, false, w.st);
            if (rc) return rc;
            src = &w.ctl->init;
        }
        bool seed = false;                // the next delta round follows a full one
        for (int group = 0;; group++) {
            const bool first = initial && group == 0;
            const int G = first ? (compact_mode > 0 ? 1 : kLccFirstGroup) : kLccGroup;
            RoundGroup *grp = w.ctl->grp + (group & 1);
            RoundStats *ring = grp->ring;
            CU(ctx, cudaMemsetAsync(grp, 0, sizeof(RoundGroup), ctx->stream));
            CU(ctx, cudaEventRecord(w.ev[4], ctx->stream));
            int n_full = 0, c = cur, l = li, rc;
            for (int i = 0; i < G; i++) {
                const RoundStats *prev = i ? ring + i - 1 : src;
                if (!deltas || full_left > 0) {
                    if (full_left > 0) full_left--;
                    if (first && i == 0 && first_kernel()) rc = launch_first(ring);
                    else rc = launch_round(ring + i, prev, i ? nullptr : gate, c, l, false);
                    if (rc) return rc;
                    n_full++;
                    c ^= 1;
                    l ^= 1;
                    seed = true;
                    synced = true;
                } else {
                    if ((rc = launch_push(ring + i, prev, c, l, seed))) return rc;
                    if ((rc = launch_round(ring + i, prev, nullptr, c, l, true))) return rc;
                    seed = false;
                    synced = false;
                }
                if (first && i == 0) CU(ctx, cudaEventRecord(w.ev[12], ctx->stream));
            }
            CU(ctx, cudaEventRecord(w.ev[5], ctx->stream));
            if (want_hist) {
                // the omega buffer the state is in if every queued round ran; any
                // that did not leaves the two buffers equal (a fixpoint)
                launches++;
                k_omega_hist<<<grid_for(ctx, g->n, 256, 8), 256, 0, ctx->stream>>>(g->n, w.om[c], t->n0, grp->hist);
                CU(ctx, cudaGetLastError());
            }
            if ((rc = read_control(ctx, w))) return rc;
            if (group == 0 && !initial) after_check();
            const RoundGroup &grp_h = w.ctl_h->grp[group & 1];
            if (want_hist) std::memcpy(w.hist_h, grp_h.hist, sizeof(w.hist_h));
            if (first && (w.ctl_h->init.n_hub_slots > (unsigned)w.acc_cap ||
                          (int64_t)w.ctl_h->init.n_chunk > w.chunk_cap))
                return set_err(ctx, CCPM_EOVERFLOW, "hub bookkeeping overflow");
            if (!initial && group == 0 && !w.st_h->changed) {
                synced = was_synced;                      // the check changed nothing: no round ran
                lcc_launches -= G;
                break;
            }
            gate = nullptr;
            float ms = 0.f;
            CU(ctx, cudaEventElapsedTime(&ms, w.ev[4], w.ev[5]));
            ms_lcc_kernel += ms;
            if (first) {
                CU(ctx, cudaEventElapsedTime(&ms, w.ev[4], w.ev[12]));
                ms_first = ms;
            }
            bool done = false;
            int ran = 0;
            for (int i = 0; i < G && !done; i++) {
                const RoundStats &h = grp_h.ring[i];
                if (h.skipped) break;
                ran++;
                r++;
                int64_t sc, n_rows, n_alive;
                if (i < n_full) {
                    sc = (int64_t)h.scanned;
                    n_rows = (int64_t)h.row_entries;
                    n_alive = (int64_t)h.alive;
                    last_kept = (int64_t)h.kept;
                    last_rows = (int64_t)h.rows_next;
                    last_alive = n_alive - (int64_t)h.died;
                    n_small = h.n_small;
                    n_med = h.n_med;
                    n_chunk = h.n_chunk;
                    li ^= 1;
                    cur ^= 1;
                } else {
                    // the vertices not evaluated scan what they kept
                    sc = last_kept - (int64_t)h.old_kept + (int64_t)h.scanned;
                    n_rows = last_rows;
                    n_alive = last_alive;
                    last_kept += (int64_t)h.kept - (int64_t)h.old_kept;
                    last_rows -= (int64_t)h.died_rows;
                    last_alive -= (int64_t)h.died;
                }
                scanned += sc;
                rows += n_rows;
                alive += n_alive;
                alg_bytes += (33 * sc) / 4 + 16 * n_alive;
                // what the round itself reads: the vertices it evaluates
                kernel_bytes += 24 * (int64_t)h.alive + (33 * (int64_t)h.row_entries) / 8 + 4 * (int64_t)h.scanned;
                if (lcc_rounds_run == 0) first_entries = sc;
                lcc_rounds_run++;
                done = !h.changed;
            }
            // launches that returned at once are not rounds
            lcc_launches -= G - ran;
            if (done) break;
            if (r > (int64_t)4 * (g->m + g->n) + 8)
                return set_err(ctx, CCPM_ETIMEOUT, "LCC did not converge");
            src = ring + G - 1;
            if (compact_mode > 0 && want_compact()) {
                if ((rc = compact())) return rc;
                src = nullptr;            // rebuilt lists: their sizes are the host's
            }
        }
        *rounds = r;
        return CCPM_OK;
    }

    // The totals after a non-local check (its counters in w.st_h): the vertices
    // it eliminated, and the entries they held, are gone.
    void after_check() {
        const RoundStats &h = *ctx->ws.st_h;
        last_kept -= (int64_t)h.old_kept;
        last_rows -= (int64_t)h.died_rows;
        last_alive -= (int64_t)h.died;
    }

    // Label-group directory of the compacted rows for the searches (none on
    // the full rows: they find groups by binary search).
    void directory(SearchArgs &a) const {
        a.dslot = gen >= 0 ? ldslot : nullptr;
        a.gdir = gen >= 0 ? lgdir : nullptr;
        a.n_rank = lnrank;
        std::memcpy(a.lab_rank, llab_rank, sizeof(llab_rank));
    }

    // Compact when most entries of the live rows are inactive: the next round
    // (or search) would mostly skip them.
    // Automatic mode compacts for searches: while non-local constraints are
    // still to run, and before the final search.  The LCC rounds alone barely
    // pay for the copy (measured on the scale-22 tree template), so an
    // LCC-only template is not compacted between its rounds.
    bool want_compact(bool final_search = false) const {
        if (compact_mode < 0 || last_rows <= 0) return false;
        if (compact_mode > 0) return last_kept < last_rows;
        return (final_search || searches_ahead > 0) && last_rows >= ((int64_t)1 << 21) &&
               last_kept * 8 < last_rows;
    }

    // A search needs label-grouped rows.  The grouped copy of the full rows
    // (a sort of every row, once per graph) pays off over many prunes of a
    // resident graph; for a graph's first prunes compacting the live rows is
    // far cheaper.
    bool cheaper_than_label_rows() const {
        return compact_mode >= 0 && gen < 0 && !g->lrows_ready.load() && g->prunes < 2 && last_rows > 0 &&
               last_kept < last_rows;
    }

    // Delta rounds pay for their second kernel (5 us) once a full round has more
    // than a few million entries to look over: exploring a clique on 8192
    // vertices took 154 ms with full rounds and 177 with delta rounds, the LCC
    // phase of 32M vertices with 350M entries in the live rows 22.7 and 11.7.
    bool use_deltas(int64_t rows_now) const {
        return compact_mode <= 0 && rows_now >= ctx->delta_rows && !ctx->ws.lean;
    }

    // Frontier of the live vertices over rows rp (the pieces of a long row
    // consecutive and in order); also makes both omega buffers equal.
    // only_if (nullable): on the device, only if these counters say `changed`.
    int rebucket(const int64_t *rp, bool sync = true, const RoundStats *only_if = nullptr) {
        synced = true;
        Workspace &w = ctx->ws;
        LabelMask all;
        std::memset(&all, 0xFF, sizeof(all));
        CU(ctx, cudaMemsetAsync(&w.ctl->init, 0, sizeof(RoundStats), ctx->stream));
        launches++;
        k_init<<<grid_for(ctx, g->n, 256, 8), 256, 0, ctx->stream>>>(g->n, rp, g->lab, all, w.om[cur], w.om[cur],
                                                                     w.om[cur ^ 1], w.nw[cur], w.nw[cur ^ 1], nw_bytes,
                                                                     w.small[li], w.med[li], w.chunk[li], w.acc,
                                                                     &w.ctl->init, w.hub_deg, short_max,
                                                                     only_if ? 1u : 0u, only_if, nullptr, 0);
        CU(ctx, cudaGetLastError());
        if (!sync) return CCPM_OK;
        int rc = read_stats();
        if (rc) return rc;
        const RoundStats &h = w.ctl_h->init;
        n_small = h.n_small;
        n_med = h.n_med;
        n_chunk = h.n_chunk;
        if (h.n_hub_slots > (unsigned)w.acc_cap || n_chunk > w.chunk_cap)
            return set_err(ctx, CCPM_EOVERFLOW, "hub bookkeeping overflow");
        return CCPM_OK;
    }

    // K4: new rows holding only the entries the next round would examine,
    // grouped by label (the searches scan label groups).  The kept entries
    // are a subset of those the last round found compatible (last_kept), so
    // the new arrays are sized before anything runs; one host sync at the end
    // reads the new frontier sizes.
    int compact() {
        Workspace &w = ctx->ws;
        cudaStream_t s = ctx->stream;
        const int nb = gen < 0 ? 0 : (gen ^ 1);
        int rc;
        // label ranks of the template vertices
        uint8_t labs[kMaxT];
        int nl = 0;
        for (int q = 0; q < t->n0; q++) labs[nl++] = t->labels[q];
        std::sort(labs, labs + nl);
        nl = (int)(std::unique(labs, labs + nl) - labs);
        if (w.piece_cap < w.chunk_cap * nl) {
            cudaFree(w.piece_cnt);
            w.piece_cnt = nullptr;
            w.piece_cap = 0;
            if ((rc = dalloc(ctx, &w.piece_cnt, (size_t)(w.chunk_cap * kMaxT)))) return rc;
            w.piece_cap = w.chunk_cap * kMaxT;
        }
        if (!w.sub_rp[nb] && (rc = dalloc(ctx, &w.sub_rp[nb], (size_t)g->n + 1))) return rc;
        if (!w.sub_dslot[nb] && (rc = dalloc(ctx, &w.sub_dslot[nb], (size_t)g->n))) return rc;
        if (!w.slot_ctr && (rc = dalloc(ctx, &w.slot_ctr, 1))) return rc;
        // buffers grow to twice what is needed (a cudaFree waits for the whole
        // device, which would stall every other worker of a batch)
        const int64_t dir_need = (n_small + n_med + n_chunk + 1) * (int64_t)(nl + 1);
        if (dir_need > w.gdir_cap[nb]) {
            cudaFree(w.sub_gdir[nb]);
            w.sub_gdir[nb] = nullptr;
            w.gdir_cap[nb] = 0;
            const int64_t cap = std::max<int64_t>(2 * dir_need, w.gdir_cap[nb ^ 1]);
            if ((rc = dalloc(ctx, &w.sub_gdir[nb], (size_t)cap))) return rc;
            w.gdir_cap[nb] = cap;
        }
        const int64_t need = last_kept + 64;
        if (need > w.sub_cap[nb]) {
            cudaFree(w.sub_col[nb]);
            cudaFree(w.sub_nlab[nb]);
            cudaFree(w.sub_bits[nb]);
            w.sub_col[nb] = nullptr;
            w.sub_nlab[nb] = nullptr;
            w.sub_bits[nb] = nullptr;
            w.sub_cap[nb] = 0;
            const int64_t cap = std::max<int64_t>(std::min<int64_t>(2 * need, g->m + 64), w.sub_cap[nb ^ 1]);
            if ((rc = dalloc(ctx, &w.sub_col[nb], (size_t)cap))) return rc;
            if ((rc = dalloc(ctx, &w.sub_nlab[nb], (size_t)cap))) return rc;
            if ((rc = dalloc(ctx, &w.sub_bits[nb], (size_t)(cap / 32 + 2)))) return rc;
            w.sub_cap[nb] = cap;
        }
        // the lists name every vertex live at the start of the last round; the
        // rows to copy are those of the vertices live now: list only those (the
        // kernels read the new sizes on the device, no host sync)
        const int64_t listed = n_small + n_med + n_chunk;
        if ((rc = rebucket(lrp, false))) return rc;
        CompactArgs ca{};
        ca.rp = lrp;
        ca.col = lcol;
        ca.bits = lbits;
        ca.lab = g->lab;
        ca.om = w.om[cur];
        ca.small_in = w.small[li];
        ca.med_in = w.med[li];
        ca.chunk_in = w.chunk[li];
        ca.acc = w.acc;
        ca.lists = &w.ctl->init;
        ca.hub_deg = w.hub_deg;
        ca.n_rank = nl;
        std::memset(ca.lab_rank, 0xFF, sizeof(ca.lab_rank));
        for (int r = 0; r < nl; r++) {
            ca.lab_rank[labs[r]] = (uint8_t)r;
            ca.rank_label[r] = labs[r];
        }
        ca.piece_cnt = w.piece_cnt;
        // offsets of the new rows from the entries each vertex kept in the last
        // round (0 for every vertex that is not live): exclusive prefix sum of
        // the kept counts (tile scans, a scan of the tile totals, the tile
        // offsets added)
        const int64_t tiles = g->n / kScanTile + 1;
        const size_t tmp = sizeof(int64_t) * (size_t)tiles;
        if (tmp > w.scan_tmp_bytes) {
            cudaFree(w.scan_tmp);
            w.scan_tmp = nullptr;
            w.scan_tmp_bytes = 0;
            CU(ctx, cudaMalloc(&w.scan_tmp, tmp));
            w.scan_tmp_bytes = tmp;
        }
        int64_t *tile_sum = (int64_t *)w.scan_tmp;
        launches += 3;
        k_scan_tiles<<<(unsigned)tiles, 256, 0, s>>>(g->n, w.deg, w.om[cur], w.sub_rp[nb], tile_sum);
        k_scan_sums<<<1, 256, 0, s>>>(tiles, tile_sum);
        k_scan_add<<<(unsigned)tiles, 256, 0, s>>>(g->n, w.sub_rp[nb], tile_sum);
        CU(ctx, cudaGetLastError());
        if (n_chunk > 0) {
            launches++;
            k_compact_count<<<grid_for(ctx, n_chunk * 32, 256, 8), 256, 0, s>>>(ca);
            CU(ctx, cudaGetLastError());
        }
        ca.sub_rp = w.sub_rp[nb];
        ca.sub_col = w.sub_col[nb];
        ca.sub_nlab = w.sub_nlab[nb];
        ca.dslot = w.sub_dslot[nb];
        ca.gdir = w.sub_gdir[nb];
        ca.n_slots = w.slot_ctr;
        CU(ctx, cudaMemsetAsync(w.slot_ctr, 0, sizeof(unsigned int), s));
        launches++;
        k_compact_fill<<<grid_for(ctx, listed * 32, 256, 8), 256, 0, s>>>(ca);
        CU(ctx, cudaGetLastError());
        launches++;
        k_compact_bits<<<grid_for(ctx, last_kept / 32 + 2, 256, 8), 256, 0, s>>>(w.sub_bits[nb], w.sub_rp[nb] + g->n);
        CU(ctx, cudaGetLastError());
        lrp = w.sub_rp[nb];
        lcol = w.sub_col[nb];
        lnlab = w.sub_nlab[nb];
        lbits = w.sub_bits[nb];
        ldslot = w.sub_dslot[nb];
        lgdir = w.sub_gdir[nb];
        lnrank = nl;
        std::memcpy(llab_rank, ca.lab_rank, sizeof(llab_rank));
        gen = nb;
        dense = true;
        compactions++;
        if ((rc = rebucket(lrp))) return rc;
        last_rows = last_kept;          // at most; every entry is now active
        return CCPM_OK;
    }
};

}  // namespace

namespace ccpm {
int ctx_device(ccpm_ctx *ctx) { return ctx->device; }
void *ctx_stream_ptr(ccpm_ctx *ctx) { return (void *)ctx->stream; }
int ctx_num_sms(ccpm_ctx *ctx) { return ctx->num_sms; }
int ctx_set_err(ccpm_ctx *ctx, int code, const char *msg) { return set_err(ctx, code, msg); }
GraphView graph_view(ccpm_graph *g) {
    GraphView v;
    v.n = g->n;
    v.m = g->m;
    v.rp = g->rp;
    v.col = g->col;
    v.lab = g->lab;
    v.el = g->edge_lab;
    v.ctx = g->ctx;
    return v;
}
}  // namespace ccpm

extern "C" {

void ccpm_options_default(ccpm_options *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->order_mode = CCPM_ORDER_FIXED;
    o->run_final = 1;
    o->max_embeddings = 1ull << 32;
    o->search_budget = 0;
    o->hub_degree = 0;
    o->batch_workers = 0;
}

int ccpm_ctx_create(int device, void *stream, ccpm_ctx_t *out) {
    if (!out) return CCPM_EINVAL;
    *out = nullptr;
    ccpm_ctx *c = new (std::nothrow) ccpm_ctx();
    if (!c) return CCPM_ENOMEM;
    c->device = device;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device);
    c->sm_total = c->num_sms;
    if (e == cudaSuccess) {
        if (stream) {
            c->stream = (cudaStream_t)stream;
        } else {
            e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
            c->own_stream = true;
        }
    }
    if (e != cudaSuccess) {
        delete c;
        return CCPM_ECUDA;
    }
    *out = c;
    return CCPM_OK;
}

void ccpm_test_round_limits(ccpm_ctx_t c, int64_t huge_rows, int64_t inline_rows, int64_t delta_rows) {
    c->huge_rows = huge_rows;
    c->inline_rows = inline_rows;
    c->delta_rows = delta_rows;
}

void ccpm_ctx_destroy(ccpm_ctx_t c) {
    if (!c) return;
    cudaSetDevice(c->device);
    for (ccpm_ctx *wk : c->workers) ccpm_ctx_destroy(wk);
    ws_free(c->ws);
    cudaFree(c->label_hist);
    if (c->load_ev) cudaEventDestroy(c->load_ev);
    if (c->wait_ev) cudaEventDestroy(c->wait_ev);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
    delete c;
}

const char *ccpm_last_error(ccpm_ctx_t c) { return c ? c->err.c_str() : "null context"; }

int ccpm_graph_load_csr(ccpm_ctx_t ctx, int64_t n, int64_t m, const int64_t *row_ptr, const int32_t *col,
                        const uint8_t *labels, int flags, ccpm_graph_t *out) {
    if (!ctx || !out) return CCPM_EINVAL;
    *out = nullptr;
    if (n < 1 || n >= (int64_t)1 << 31 || m < 0 || !row_ptr || !labels || (m > 0 && !col))
        return set_err(ctx, CCPM_EINVAL, "graph: need 1 <= n < 2^31, m >= 0 and non-NULL arrays");
    CU(ctx, cudaSetDevice(ctx->device));
    const bool dev = (flags & CCPM_DEVICE_PTRS) != 0;
    if (!dev) {
        if (row_ptr[0] != 0 || row_ptr[n] != m)
            return set_err(ctx, CCPM_EINVAL, "graph: row_ptr[0] must be 0 and row_ptr[n] == m_dir");
        if (flags & CCPM_VALIDATE) {
            for (int64_t v = 0; v < n; v++)
                if (row_ptr[v + 1] < row_ptr[v]) return set_err(ctx, CCPM_EINVAL, "graph: row_ptr not monotone");
            for (int64_t v = 0; v < n; v++) {
                for (int64_t e = row_ptr[v]; e < row_ptr[v + 1]; e++) {
                    int32_t u = col[e];
                    if (u < 0 || u >= n) return set_err(ctx, CCPM_EINVAL, "graph: column index out of range");
                    if (u == v) return set_err(ctx, CCPM_EINVAL, "graph: self loop");
                    if (e > row_ptr[v] && col[e - 1] >= u)
                        return set_err(ctx, CCPM_EINVAL, "graph: row not sorted or duplicate entry");
                    // reverse entry must exist
                    const int32_t *lo = col + row_ptr[u], *hi = col + row_ptr[u + 1];
                    const int32_t *f = std::lower_bound(lo, hi, (int32_t)v);
                    if (f == hi || *f != v) return set_err(ctx, CCPM_EINVAL, "graph: missing reverse entry");
                }
            }
        }
    } else if (flags & CCPM_VALIDATE) {
        return set_err(ctx, CCPM_EINVAL, "graph: CCPM_VALIDATE needs host pointers");
    }
    ccpm_graph *g = new (std::nothrow) ccpm_graph();
    if (!g) return set_err(ctx, CCPM_ENOMEM, "graph: host allocation");
    g->ctx = ctx;
    g->n = n;
    g->m = m;
    g->borrowed = dev;
    if (dev) {
        g->rp = const_cast<int64_t *>(row_ptr);
        g->col = const_cast<int32_t *>(col);
        g->lab = const_cast<uint8_t *>(labels);
        // label counts on the device.  The arrays may still be in the making on the
        // default stream (or one that waits for it): the count waits for these, and
        // for no other stream's work.  Event and counters stay with the context,
        // since giving memory back waits for the whole device.
        unsigned long long h[512];
        cudaError_t e = cudaSuccess;
        if (!ctx->load_ev) e = cudaEventCreateWithFlags(&ctx->load_ev, cudaEventDisableTiming);
        if (e == cudaSuccess && !ctx->label_hist) e = cudaMalloc((void **)&ctx->label_hist, sizeof(h));
        if (e == cudaSuccess) e = cudaEventRecord(ctx->load_ev, nullptr);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ctx->stream, ctx->load_ev, 0);
        if (e == cudaSuccess) e = cudaMemsetAsync(ctx->label_hist, 0, sizeof(h), ctx->stream);
        if (e == cudaSuccess) {
            k_label_hist<<<grid_for(ctx, n, 256, 8), 256, 0, ctx->stream>>>(n, row_ptr, labels, ctx->label_hist);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, ctx->label_hist, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) {
            delete g;
            return set_err(ctx, e == cudaErrorMemoryAllocation ? CCPM_ENOMEM : CCPM_ECUDA, "graph: label counts");
        }
        for (int L = 0; L < 256; L++) {
            g->label_freq[L] = (int64_t)h[L];
            g->label_rows[L] = (int64_t)h[256 + L];
        }
    } else {
        int rc;
        if ((rc = dalloc(ctx, &g->rp, (size_t)n + 1)) || (rc = dalloc(ctx, &g->col, (size_t)m)) ||
            (rc = dalloc(ctx, &g->lab, (size_t)n))) {
            cudaFree(g->rp); cudaFree(g->col); cudaFree(g->lab);
            delete g;
            return rc;
        }
        cudaError_t e = cudaMemcpyAsync(g->rp, row_ptr, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess && m > 0)
            e = cudaMemcpyAsync(g->col, col, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(g->lab, labels, (size_t)n, cudaMemcpyHostToDevice, ctx->stream);
        // the offsets' check and the label histogram run while the copies do
        bool monotone = true;
        for (int64_t v = 0; v < n && monotone; v++) monotone = row_ptr[v + 1] >= row_ptr[v];
        for (int64_t v = 0; v < n; v++) {
            g->label_freq[labels[v]]++;
            g->label_rows[labels[v]] += row_ptr[v + 1] - row_ptr[v];
        }
        const cudaError_t e2 = cudaStreamSynchronize(ctx->stream);
        if (e == cudaSuccess) e = e2;
        if (e != cudaSuccess || !monotone) {
            cudaFree(g->rp); cudaFree(g->col); cudaFree(g->lab);
            delete g;
            if (!monotone) return set_err(ctx, CCPM_EINVAL, "graph: row_ptr not monotone");
            return set_err(ctx, CCPM_ECUDA, std::string("graph upload: ") + cudaGetErrorString(e));
        }
    }
    *out = g;
    return CCPM_OK;
}

void ccpm_graph_destroy(ccpm_graph_t g) {
    if (!g) return;
    cudaSetDevice(g->ctx->device);
    if (!g->borrowed) { cudaFree(g->rp); cudaFree(g->col); cudaFree(g->lab); }
    cudaFree(g->lcol);
    cudaFree(g->nlab);
    cudaFree(g->elab);
    if (!g->edge_lab_borrowed) cudaFree(g->edge_lab);
    delete g;
}

int ccpm_graph_set_edge_labels(ccpm_graph_t g, const uint8_t *edge_labels, int flags) {
    if (!g) return CCPM_EINVAL;
    ccpm_ctx *ctx = g->ctx;
    CU(ctx, cudaSetDevice(ctx->device));
    const bool dev = (flags & CCPM_DEVICE_PTRS) != 0;
    if (edge_labels && (flags & CCPM_VALIDATE)) {
        if (dev) return set_err(ctx, CCPM_EINVAL, "edge labels: CCPM_VALIDATE needs host pointers");
        // both entries of every edge carry the same label
        std::vector<int64_t> rp((size_t)g->n + 1);
        std::vector<int32_t> col((size_t)g->m);
        CU(ctx, cudaMemcpy(rp.data(), g->rp, sizeof(int64_t) * rp.size(), cudaMemcpyDeviceToHost));
        if (g->m > 0) CU(ctx, cudaMemcpy(col.data(), g->col, sizeof(int32_t) * col.size(), cudaMemcpyDeviceToHost));
        for (int64_t v = 0; v < g->n; v++)
            for (int64_t e = rp[(size_t)v]; e < rp[(size_t)v + 1]; e++) {
                const int32_t u = col[(size_t)e];
                const int32_t *lo = col.data() + rp[(size_t)u], *hi = col.data() + rp[(size_t)u + 1];
                const int32_t *f = std::lower_bound(lo, hi, (int32_t)v);
                if (f == hi || *f != v) return set_err(ctx, CCPM_EINVAL, "edge labels: missing reverse entry");
                if (edge_labels[(size_t)(f - col.data())] != edge_labels[(size_t)e])
                    return set_err(ctx, CCPM_EINVAL, "edge labels: the two entries of an edge differ");
            }
    }
    if (!g->edge_lab_borrowed) cudaFree(g->edge_lab);
    g->edge_lab = nullptr;
    g->edge_lab_borrowed = false;
    if (!edge_labels) return CCPM_OK;
    if (dev) {
        g->edge_lab = const_cast<uint8_t *>(edge_labels);
        g->edge_lab_borrowed = true;
        return CCPM_OK;
    }
    int rc = dalloc(ctx, &g->edge_lab, (size_t)std::max<int64_t>(g->m, 1));
    if (rc) return rc;
    if (g->m > 0) CU(ctx, cudaMemcpyAsync(g->edge_lab, edge_labels, (size_t)g->m, cudaMemcpyHostToDevice, ctx->stream));
    CU(ctx, cudaStreamSynchronize(ctx->stream));
    return CCPM_OK;
}

int ccpm_tmpl_load(ccpm_ctx_t ctx, int n0, const uint8_t *labels, int m0, const int32_t *edges, ccpm_tmpl_t *out) {
    if (!out) return CCPM_EINVAL;
    *out = nullptr;
    ccpm_tmpl *t = new (std::nothrow) ccpm_tmpl();
    if (!t) return CCPM_ENOMEM;
    t->ctx = ctx;
    int rc = template_build(t->t, n0, labels, m0, edges);
    if (rc) {
        if (ctx) ctx->err = t->t.err;
        delete t;
        return rc;
    }
    *out = t;
    return CCPM_OK;
}

void ccpm_tmpl_destroy(ccpm_tmpl_t t) { delete t; }

int ccpm_constraints_generate(ccpm_tmpl_t t, ccpm_graph_t g, int *n) {
    (void)g;
    if (!t) return CCPM_EINVAL;
    std::string err;
    int rc = constraints_generate(t->t, err);
    if (rc) {
        t->t.err = err;
        if (t->ctx) t->ctx->err = err;
        return rc;
    }
    if (n) *n = (int)t->t.k0.size();
    return CCPM_OK;
}

int ccpm_constraints_describe(ccpm_tmpl_t t, int i, ccpm_constraint_info *out) {
    if (!t || !out || !t->t.generated) return CCPM_ESTATE;
    if (i < 0 || i >= (int)t->t.order.size()) return CCPM_EINVAL;
    const HostConstraint &c = t->t.k0[(size_t)t->t.order[(size_t)i]];
    std::memset(out, 0, sizeof(*out));
    out->kind = c.kind;
    out->vert_mask = c.vmask;
    out->head_mask = c.hmask;
    out->n_verts = __builtin_popcount(c.vmask);
    out->n_edges = (int)c.edges.size();
    for (size_t k = 0; k < c.edges.size(); k++) {
        out->edges[k][0] = c.edges[k].first;
        out->edges[k][1] = c.edges[k].second;
    }
    return CCPM_OK;
}

int ccpm_tmpl_set_order(ccpm_tmpl_t t, int n, const int32_t *order) {
    if (!t || !t->t.generated) return CCPM_ESTATE;
    if (n != (int)t->t.k0.size() || (n > 0 && !order)) return CCPM_EINVAL;
    std::vector<int> seen((size_t)n, 0), ord((size_t)n);
    for (int i = 0; i < n; i++) {
        if (order[i] < 0 || order[i] >= n || seen[(size_t)order[i]]) return CCPM_EINVAL;
        seen[(size_t)order[i]] = 1;
        ord[(size_t)i] = order[i];
    }
    t->t.order = ord;
    return CCPM_OK;
}

static int prune(ccpm_ctx_t ctx, ccpm_graph_t g, ccpm_tmpl_t tm, const ccpm_options *opt_in, ccpm_result_t *out) {
    if (!ctx || !g || !tm || !out) return CCPM_EINVAL;
    if (g->ctx->device != ctx->device) return set_err(ctx, CCPM_EINVAL, "graph lives on another device");
    ccpm_options opt;
    if (opt_in) opt = *opt_in; else ccpm_options_default(&opt);
    CU(ctx, cudaSetDevice(ctx->device));
    Template &t = tm->t;
    if (!t.generated) {
        std::string err;
        int rc = constraints_generate(t, err);
        if (rc) return set_err(ctx, rc, err);
    }
    const int hub_deg = opt.hub_degree > 0 ? std::min(opt.hub_degree, kMaxHubDeg) : kDefaultHubDeg;
    const uint64_t budget = opt.search_budget ? opt.search_budget : kDefaultSearchBudget;
    const uint64_t split = opt.search_split < 0 ? 0 : (opt.search_split == 0 ? kSpillAfter : (uint64_t)opt.search_split);
    // a caller's own budget counts windows as one search scans them: no handing
    // on to idle warps, which would restart its count.  Those searches are
    // spread up front instead (expand_more: a kernel and a host round trip per
    // level) and handed on after `split` windows only, which is slower where both
    // work: a prune with the 5-cycle template over 16M vertices 43.6 against 5.8
    // ms, a batch of 24 templates over 4M 35 against 20
    const bool starve = opt.search_split >= 0 && opt.search_budget == 0;
    int rc = ws_ensure(ctx, g, hub_deg);
    if (rc) return rc;
    Workspace &w = ctx->ws;
    ccpm_result *r = *out;
    if (r && r->g != g) return set_err(ctx, CCPM_EINVAL, "result was made for another graph");
    const uint64_t tfp = tmpl_fingerprint(t);
    const bool resume = opt.resume != 0;
    if (resume && (!r || r->tmpl_fp != tfp))
        return set_err(ctx, CCPM_EINVAL, "options.resume needs *out to hold a state of this graph and template");
    bool fresh = false;
    if (!r) {
        r = new (std::nothrow) ccpm_result();
        if (!r) return set_err(ctx, CCPM_ENOMEM, "result: host allocation");
        r->g = g;
        if ((rc = dalloc(ctx, &r->om, (size_t)g->n)) || (rc = dalloc(ctx, &r->eb, (size_t)w.words + 1))) {
            cudaFree(r->om); cudaFree(r->eb);
            delete r;
            return rc;
        }
        fresh = true;
    }
    auto fail = [&](int code) {
        if (fresh) { cudaFree(r->om); cudaFree(r->eb); delete r; }
        return code;
    };
    std::memset(&r->counts, 0, sizeof(r->counts));
    r->phase_rounds.clear();
    r->tmpl_fp = tfp;

    Pipeline P;
    P.ctx = ctx;
    P.g = g;
    P.t = &t;
    build_dev_tmpl(t, P.dt);
    P.maxc = P.dt.n_cls;
    P.lrp = g->rp;
    P.lcol = g->col;
    P.lbits = w.ebits;
    P.short_max = opt.short_rows > 0 ? std::min(opt.short_rows, kMaxHubDeg) : kSmallDeg;
    P.eta_off = opt.no_edge_elimination != 0;
    P.nw_bytes = t.n0 <= 8 ? 1 : (t.n0 <= 16 ? 2 : 0);
    g->prunes++;
    P.compact_mode = opt.compact;
    cudaStream_t s = ctx->stream;

#define CUF(call)                                                                       \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            set_err(ctx, CCPM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
            return fail(CCPM_ECUDA);                                                    \
        }                                                                               \
    } while (0)
#define RCF(expr)                     \
    do {                              \
        int rc_ = (expr);             \
        if (rc_) return fail(rc_);    \
    } while (0)

    if (!w.lean) CUF(cudaMemsetAsync(w.dirty, 0, sizeof(uint32_t) * (size_t)(g->n / 32 + 1), s));
    CUF(cudaEventRecord(w.ev[0], s));
    // ---- init (Alg. 3)
    LabelMask lm;
    std::memset(&lm, 0, sizeof(lm));
    for (int q = 0; q < t.n0; q++) lm.m[t.labels[q]] |= 1u << q;
    P.lm0 = lm;
    P.from_labels = !resume;
    if (resume) {
        // a saved state: its edge bits, then (below) its omega inside the initial one
        CUF(cudaMemcpyAsync(w.ebits, r->eb, sizeof(uint32_t) * (size_t)w.words, cudaMemcpyDeviceToDevice, s));
    } else {
        CUF(cudaMemsetAsync(w.ebits, 0xFF, sizeof(uint32_t) * (size_t)w.words, s));
    }
    CUF(cudaMemsetAsync(&w.ctl->init, 0, sizeof(RoundStats), s));
    if (!P.first_kernel() || resume) {
        int grid = grid_for(ctx, g->n, 256, 8);
        P.launches++;
        k_init<<<grid, 256, 0, s>>>(g->n, g->rp, g->lab, lm, resume ? r->om : nullptr, w.om[0], w.om[1], w.nw[0],
                                    w.nw[1], P.nw_bytes, w.small[0], w.med[0], w.chunk[0], w.acc, &w.ctl->init,
                                    hub_deg, P.short_max, 1u, nullptr, w.ebits, g->m);
        CUF(cudaGetLastError());
    }
    if (resume) {
        // entries with a dead end point carry no bit; the first round reads the bits
        P.launches++;
        k_materialize<<<grid_for(ctx, g->n * 32, 256, 8), 256, 0, s>>>(g->n, w.om[0], g->rp, g->col, w.ebits);
        CUF(cudaGetLastError());
        P.dense = false;
    }
    P.cur = 0;
    P.li = 0;
    for (int L = 0; L < 256; L++)
        if (lm.m[L]) P.first_rows += g->label_rows[L];
    // the first round reads the entry labels when its rows cover a large
    // share of the graph (building them is one pass over the entries)
    if (P.dense && (opt.entry_labels > 0 ||
                    (opt.entry_labels == 0 && P.first_rows >= kEntryLabelRows && P.first_rows * 8 >= g->m))) {
        RCF(ensure_entry_labels(ctx, g));
        P.elab = g->elab;
    }

    // ---- LCC to fixpoint (Alg. 4)
    P.searches_ahead = opt.lcc_only ? 0 : (int)t.order.size();
    int64_t rounds = 0;
    RCF(P.lcc(&rounds, true, P.searches_ahead > 0));
    r->phase_rounds.push_back((int32_t)rounds);
    int64_t total_rounds = rounds;
    CUF(cudaEventRecord(w.ev[1], s));

    // ---- non-local constraints, one at a time (Alg. 1, Alg. 6/7)
    int64_t tokens = 0;
    bool over = false;
    int nl_run = 0;
    std::vector<int> remaining = t.order;
    if (opt.lcc_only) {
        remaining.clear();
        opt.run_final = 0;
    }
    const int n_constraints = (int)remaining.size();
    const bool learned = opt.order_mode == CCPM_ORDER_LEARNED && opt.mlp;
    if (opt.order_mode == CCPM_ORDER_LEARNED && !opt.mlp)
        return fail(set_err(ctx, CCPM_EINVAL, "CCPM_ORDER_LEARNED needs options.mlp"));
    r->logs.clear();
    for (int step = 0; step < n_constraints; step++) {
        // features of every remaining constraint in the current state
        std::vector<float> feats(remaining.size() * CCPM_MLP_IN);
        for (size_t i = 0; i < remaining.size(); i++)
            constraint_features(t, t.k0[(size_t)remaining[i]], w.hist_h, w.hist_h[kMaxT], step, n_constraints,
                                &feats[i * CCPM_MLP_IN]);
        // a constraint none of whose heads is matched by a live vertex issues no
        // token and changes nothing: it is checked without launching anything
        auto is_noop = [&](size_t i) {
            const uint32_t hm = t.k0[(size_t)remaining[i]].hmask;
            for (int q = 0; q < t.n0; q++)
                if (((hm >> q) & 1u) && w.hist_h[q]) return false;
            return true;
        };
        size_t pick = 0;
        if (learned && remaining.size() > 1) {
            size_t first_noop = remaining.size();
            for (size_t i = 0; i < remaining.size() && first_noop == remaining.size(); i++)
                if (is_noop(i)) first_noop = i;
            if (first_noop < remaining.size()) {
                pick = first_noop;
            } else {
                // the network predicts -log2(1 + microseconds) of running each
                // constraint now; a later constraint of the fixed order runs
                // first if it is predicted more than twice as cheap as the fixed
                // order's next one (the one predicted cheapest among those), so
                // expensive checks wait for a state that cheaper ones have shrunk
                std::vector<float> score(remaining.size());
                P.launches++;
                RCF(mlp_score(opt.mlp, (int)remaining.size(), feats.data(), score.data(), (void *)s, w.mlp,
                               (void *)ctx->wait_ev));
                for (size_t i = 1; i < remaining.size(); i++)
                    if (score[i] > score[0] + 1.f && score[i] > score[pick]) pick = i;
            }
        }
        const bool noop = is_noop(pick);
        const int chosen = remaining[pick];
        ccpm_constraint_log lg;
        std::memset(&lg, 0, sizeof(lg));
        lg.constraint = chosen;
        lg.position = step;
        std::memcpy(lg.features, &feats[pick * CCPM_MLP_IN], sizeof(lg.features));
        lg.bits_before = (int64_t)w.hist_h[kMaxT];
        remaining.erase(remaining.begin() + (long)pick);
        P.searches_ahead = (int)remaining.size() + 1;
        const HostConstraint &c = t.k0[(size_t)chosen];
        nl_run++;
        if (noop) {
            lg.bits_after = lg.bits_before;
            r->logs.push_back(lg);
            r->phase_rounds.push_back(0);
            continue;
        }
        CUF(cudaEventRecord(w.ev[6], s));
        const int64_t tokens_before = tokens;
        uint32_t sadj[kMaxT] = {};
        for (auto &e : c.edges) { sadj[e.first] |= 1u << e.second; sadj[e.second] |= 1u << e.first; }
        for (int h = 0; h < kMaxT; h++)
            if ((c.hmask >> h) & 1u) build_plan(t, c.vmask, sadj, h, g->label_freq, false, w.plans_h[h], -1, w.hist_h);
        CUF(cudaMemcpyAsync(w.plans, w.plans_h, sizeof(DevPlan) * kMaxT, cudaMemcpyHostToDevice, s));
        // not a no-op: some live vertex is a root, so rows to search are needed
        if (P.want_compact() || P.cheaper_than_label_rows()) RCF(P.compact());
        if (P.gen < 0) RCF(ensure_label_rows(ctx, g));
        RCF(clear_search(ctx, w));
        P.launches++;
        k_collect_roots<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, w.om[P.cur], c.hmask, w.roots, w.st);
        CUF(cudaGetLastError());
        SearchArgs a{};
        a.rp = g->rp;
        a.col = g->col;
        a.rl = P.gen >= 0 ? P.lrp : g->rp;
        a.lcol = P.gen >= 0 ? P.lcol : g->lcol;
        a.nlab = P.gen >= 0 ? P.lnlab : g->nlab;
        P.directory(a);
        a.om = w.om[P.cur];
        a.roots = w.roots;
        a.n_roots = -1;
        a.plans = w.plans;
        a.heads = c.hmask;
        a.sat = w.sat;
        a.st = w.st;
        a.budget = budget;
        a.items = w.items;
        a.items_cap = w.items_cap;
        a.enum_heads = 0;
        const SearchMode mode{0, split, starve};
        P.search_launches++;
        // one item per (root, head, candidate for position 1); the search, the
        // elimination of the issuers that failed and the LCC rounds after it are
        // queued together, and one host round trip reads what became of them
        CUF(cudaEventRecord(w.ev[10], s));
        RCF(queue_search(ctx, w, a, mode, __builtin_popcount(c.vmask), P.launches));
        CUF(cudaEventRecord(w.ev[11], s));
        auto apply = [&](const PassCtl *last) {
            P.launches++;
            k_nlcc_apply<<<grid_for(ctx, g->n, 256, 4), 256, 0, s>>>(
                w.roots, last, w.items_cap, c.hmask, w.sat, w.om[P.cur], w.om[0], w.om[1], w.nw[0], w.nw[1], P.nw_bytes,
                P.lrp, w.deg, w.chg, w.chg_piece, hub_deg, w.st);
            return cudaGetLastError();
        };
        CUF(apply(w.ctl->pass + kChain - 1));
        CUF(cudaEventRecord(w.ev[7], s));
        P.searches_ahead = (int)remaining.size();
        int64_t rr = 0;
        RCF(P.lcc(&rr, false, true));
        if (!search_complete(w, mode)) {
            // more passes than were queued: the elimination has not run yet
            RCF(finish_search(ctx, w, a, mode, P.launches));
            CUF(cudaEventRecord(w.ev[11], s));
            CUF(apply(nullptr));
            CUF(cudaEventRecord(w.ev[7], s));
            RCF(P.lcc(&rr, false, true));
        }
        if (w.st_h->overflow) over = true;
        P.windows += (int64_t)(w.st_h->windows + w.st_h->expanded);
        P.nlcc_entries += (int64_t)w.st_h->windows;
        tokens += (int64_t)w.st_h->tokens;
        float ms_k = 0.f;
        CUF(cudaEventElapsedTime(&ms_k, w.ev[10], w.ev[11]));
        P.ms_search_kernel += ms_k;
        r->phase_rounds.push_back((int32_t)rr);
        total_rounds += rr;
        float ms_a = 0.f, ms_b = 0.f;
        cudaEventElapsedTime(&ms_a, w.ev[6], w.ev[7]);
        cudaEventElapsedTime(&ms_b, w.ev[7], w.ev[5]);
        lg.ms_search = ms_a;
        lg.ms_lcc = rr ? ms_b : 0.0;
        lg.lcc_rounds = (int32_t)rr;
        lg.tokens = (int32_t)std::min<int64_t>(tokens - tokens_before, INT32_MAX);
        lg.bits_after = (int64_t)w.hist_h[kMaxT];
        r->logs.push_back(lg);
    }
    CUF(cudaEventRecord(w.ev[2], s));

    // ---- final template-driven search and match count (Remark 1, Sec. 4.7)
    // omega* and E* are existence questions answered exactly by searches over
    // the whole template; the number of matches is counted separately.
    bool count_valid = false;
    uint64_t matches = 0;
    bool final_done = false;
    float ms_fc = 0.f, ms_fv = 0.f, ms_fe = 0.f;
    bool summary_done = false, existence = false;
    // the end of the result's making, then its active vertices and entries
    auto queue_summary = [&]() -> int {
        CU(ctx, cudaEventRecord(w.ev[3], s));
        CU(ctx, cudaMemsetAsync(w.cnt, 0, 2 * sizeof(unsigned long long), s));
        P.launches++;
        k_count<<<grid_for(ctx, std::max<int64_t>(g->n, w.words), 256, 8), 256, 0, s>>>(g->n, r->om, w.words, r->eb, w.cnt);
        CU(ctx, cudaGetLastError());
        return CCPM_OK;
    };
    cudaEvent_t fev[4] = {w.ev[6], w.ev[7], w.ev[8], w.ev[9]};
    if (opt.run_final) {
        const uint32_t all = t.n0 == 32 ? 0xFFFFFFFFu : ((1u << t.n0) - 1u);
        if (P.want_compact(true) || P.cheaper_than_label_rows()) RCF(P.compact());
        if (P.gen < 0) RCF(ensure_label_rows(ctx, g));
        CUF(cudaMemsetAsync(r->om, 0, sizeof(uint32_t) * (size_t)g->n, s));
        CUF(cudaMemsetAsync(r->eb, 0, sizeof(uint32_t) * (size_t)(w.words + 1), s));
        SearchArgs a{};
        a.rp = g->rp;
        a.col = g->col;
        a.rl = P.gen >= 0 ? P.lrp : g->rp;
        a.lcol = P.gen >= 0 ? P.lcol : g->lcol;
        a.nlab = P.gen >= 0 ? P.lnlab : g->nlab;
        P.directory(a);
        a.roots = w.roots;
        a.plans = w.plans;
        a.sat = w.sat;
        a.eb_out = r->eb;
        a.st = w.st;
        a.budget = budget;
        a.items = w.items;
        a.items_cap = w.items_cap;
        // the final enumeration keeps the background label frequencies (measured
        // faster than ordering by live candidates there)
        int root = 0;
        for (int q = 1; q < t.n0; q++)
            if (g->label_freq[t.labels[q]] < g->label_freq[t.labels[root]]) root = q;
        // one pass over every match from roots of `root`: count (mode kCount) or
        // count and mark (kMark); returns overflow of the cap
        auto count_pass = [&](int mode, const uint32_t *om_src, uint64_t cap, uint64_t &found, bool &capped) -> int {
            build_plan(t, all, t.adj, root, g->label_freq, true, w.plans_h[0]);
            CU(ctx, cudaMemcpyAsync(w.plans, w.plans_h, sizeof(DevPlan), cudaMemcpyHostToDevice, s));
            int rc2 = clear_search(ctx, w);
            if (rc2) return rc2;
            P.launches++;
            k_collect_roots<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, om_src, 1u << root, w.roots, w.st);
            CU(ctx, cudaGetLastError());
            a.om = om_src;
            a.n_roots = -1;
            a.heads = 1u << root;
            a.cap = cap;
            a.enum_heads = 1;
            a.om_out = r->om;
            a.eb_out = r->eb;
            const SearchMode sm{mode == kMark ? 2 : 1, split, starve};
            if ((rc2 = queue_search(ctx, w, a, sm, t.n0, P.launches))) return rc2;
            CU(ctx, cudaEventRecord(fev[1], s));
            // most often the enumeration is over by then and marked everything:
            // the summary needs no round trip of its own
            if (mode == kMark && (rc2 = queue_summary())) return rc2;
            if ((rc2 = read_control(ctx, w))) return rc2;
            summary_done = mode == kMark && search_complete(w, sm) && w.st_h->n_items <= w.items_cap && !w.st_h->overflow;
            if (!search_complete(w, sm) && (rc2 = finish_search(ctx, w, a, sm, P.launches))) return rc2;
            P.windows += (int64_t)(w.st_h->windows + w.st_h->expanded);
            found = w.st_h->matches;
            capped = w.st_h->overflow != 0;
            return CCPM_OK;
        };
        // count the matches (every match lies inside the pruned state); with
        // few of them one more enumeration that marks each gives omega* and E*
        // few matches (at most kFewMatches): one enumeration counts and marks
        // them.  More: a counting enumeration up to the cap; then, up to
        // kMarkCap matches, one more enumeration marks them, and past that the
        // existence passes answer omega* and E*.
        bool capped = false;
        CUF(cudaEventRecord(fev[0], s));
        RCF(count_pass(kMark, w.om[P.cur], std::min<uint64_t>(opt.max_embeddings, kFewMatches), matches, capped));
        if (!capped) {
            count_valid = true;
            final_done = true;
        } else if (opt.max_embeddings > kFewMatches) {
            RCF(count_pass(kCount, w.om[P.cur], opt.max_embeddings, matches, capped));
            count_valid = !capped;
            if (!capped && matches <= kMarkCap) {
                uint64_t again = 0;
                CUF(cudaMemsetAsync(r->om, 0, sizeof(uint32_t) * (size_t)g->n, s));
                CUF(cudaMemsetAsync(r->eb, 0, sizeof(uint32_t) * (size_t)(w.words + 1), s));
                RCF(count_pass(kMark, w.om[P.cur], opt.max_embeddings, again, capped));
                final_done = true;
            }
        } else {
            count_valid = false;
        }
        if (!final_done || !summary_done) CUF(cudaEventRecord(fev[1], s));
        if (!final_done) {
            // the capped enumeration's marks stay: every one belongs to a match
            // found, so the existence searches below skip those (vertex,
            // template vertex) pairs and entries
            a.om_out = nullptr;
            a.eb_out = r->eb;
            a.sat_seed = r->om;
        }
        if (!final_done) {
            // (A) every (v, q): some match has phi(q) = v?  Found embeddings also
            // satisfy the other (vertex, template vertex) pairs they place and mark
            // their edges.
            for (int q = 0; q < t.n0; q++) build_plan(t, all, t.adj, q, g->label_freq, true, w.plans_h[q]);
            CUF(cudaMemcpyAsync(w.plans, w.plans_h, sizeof(DevPlan) * (size_t)t.n0, cudaMemcpyHostToDevice, s));
            RCF(clear_search(ctx, w));
            P.launches++;
            k_collect_roots<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, w.om[P.cur], all, w.roots, w.st);
            CUF(cudaGetLastError());
            a.om = w.om[P.cur];
            a.n_roots = -1;
            a.heads = all;
            a.enum_heads = 0;
            const SearchMode vm{0, split, starve};
            RCF(queue_search(ctx, w, a, vm, t.n0, P.launches));
            RCF(read_control(ctx, w));
            if (!search_complete(w, vm)) RCF(finish_search(ctx, w, a, vm, P.launches));
            if (w.st_h->overflow) over = true;
            P.windows += (int64_t)(w.st_h->windows + w.st_h->expanded);
            P.launches++;
            k_sat_to_omega<<<grid_for(ctx, w.st_h->n_roots, 256, 8), 256, 0, s>>>(w.roots, w.st, w.sat, w.om[P.cur], r->om);
            CUF(cudaGetLastError());
            a.sat_seed = nullptr;
            CUF(cudaEventRecord(fev[2], s));
            // (B) every entry between omega* vertices that no embedding has marked
            // yet: some match maps a template edge onto it?
            std::vector<std::pair<int, int>> oriented;
            for (auto &e : t.edges) { oriented.push_back(e); oriented.push_back({e.second, e.first}); }
            // (the roots are collected with the first edges; -1: the host does not
            // know their number yet)
            int64_t n_roots = -1;
            for (size_t o0 = 0; n_roots != 0 && o0 < oriented.size(); o0 += 32) {
                EdgeTab tab;
                std::memset(&tab, 0, sizeof(tab));
                tab.n = (int)std::min<size_t>(32, oriented.size() - o0);
                for (int o = 0; o < tab.n; o++) {
                    tab.a[o] = (int8_t)oriented[o0 + (size_t)o].first;
                    tab.b[o] = (int8_t)oriented[o0 + (size_t)o].second;
                    build_plan(t, all, t.adj, tab.a[o], g->label_freq, true, w.plans_h[o], tab.b[o]);
                }
                CUF(cudaMemcpyAsync(w.plans, w.plans_h, sizeof(DevPlan) * (size_t)tab.n, cudaMemcpyHostToDevice, s));
                a.om = r->om;
                // the candidate entries of a range of roots become items; a range
                // whose items do not fit is halved and made again (the bits marked
                // so far stay: every one of them is a found match's edge)
                const SearchMode em{4, split, starve};
                int64_t span = n_roots, r0 = 0;
                while (n_roots < 0 || r0 < n_roots) {
                    const int64_t r1 = n_roots < 0 ? -1 : std::min(n_roots, r0 + span);
                    RCF(clear_search(ctx, w));
                    a.roots = w.roots + r0;
                    a.n_roots = n_roots < 0 ? -1 : r1 - r0;
                    if (n_roots < 0) {
                        P.launches++;
                        k_collect_roots<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, r->om, all, w.roots, w.st);
                        CUF(cudaGetLastError());
                    }
                    P.launches++;
                    k_edge_items<<<grid_sms(ctx) * 8, 256, 0, s>>>(a, tab);
                    CUF(cudaGetLastError());
                    a.n_items = -1;
                    RCF(queue_passes(ctx, w, a, em, P.launches));
                    RCF(read_control(ctx, w));
                    if (n_roots < 0) span = n_roots = w.st_h->n_roots;
                    const int64_t done_to = r1 < 0 ? n_roots : r1;
                    if (w.st_h->n_items > w.items_cap) {
                        if (done_to - r0 == 1)
                            return fail(set_err(ctx, CCPM_EOVERFLOW, "edge pass: one vertex has too many candidate edges"));
                        span = std::max<int64_t>(1, (done_to - r0) / 2);
                        continue;
                    }
                    RCF(finish_search(ctx, w, a, em, P.launches));
                    if (w.st_h->overflow) over = true;
                    P.windows += (int64_t)w.st_h->windows;
                    r0 = done_to;
                }
                a.roots = w.roots;
            }
            CUF(cudaEventRecord(fev[3], s));
            existence = true;
        }
        final_done = true;
    }
    if (!final_done) {
        // hand back the pruned state: exact edge map for live rows, dead rows
        // zeroed.  When every round ran on the full rows with edge
        // elimination, the last (quiescent) round has already left the live
        // rows exact, and they are copied out.
        P.launches++;
        if (P.gen < 0 && !P.eta_off) {
            CUF(cudaMemsetAsync(r->eb, 0, sizeof(uint32_t) * (size_t)(w.words + 1), s));
            k_copy_live_rows<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, w.om[P.cur], g->rp, w.ebits, r->eb);
            CUF(cudaGetLastError());
        } else {
            k_materialize_fix<<<grid_for(ctx, g->n * 32, 256, 8), 256, 0, s>>>(g->n, w.om[P.cur], g->rp, g->col,
                                                                               w.ebits, P.dt);
            CUF(cudaGetLastError());
            CUF(cudaMemcpyAsync(r->eb, w.ebits, sizeof(uint32_t) * (size_t)w.words, cudaMemcpyDeviceToDevice, s));
        }
        CUF(cudaMemcpyAsync(r->om, w.om[P.cur], sizeof(uint32_t) * (size_t)g->n, cudaMemcpyDeviceToDevice, s));
    }
    if (!summary_done) {
        RCF(queue_summary());
        RCF(read_control(ctx, w));
    }
    if (opt.run_final) {
        cudaEventElapsedTime(&ms_fc, fev[0], fev[1]);
        if (existence) {
            cudaEventElapsedTime(&ms_fv, fev[1], fev[2]);
            cudaEventElapsedTime(&ms_fe, fev[2], fev[3]);
        }
    }
    float ms_lcc = 0, ms_nlcc = 0, ms_final = 0;
    cudaEventElapsedTime(&ms_lcc, w.ev[0], w.ev[1]);
    cudaEventElapsedTime(&ms_nlcc, w.ev[1], w.ev[2]);
    cudaEventElapsedTime(&ms_final, w.ev[2], w.ev[3]);

    ccpm_counts &cn = r->counts;
    cn.active_v = (int64_t)w.cnt_h[0];
    cn.active_e_dir = (int64_t)w.cnt_h[1];
    cn.lcc_rounds_total = total_rounds;
    cn.n_phases = (int32_t)r->phase_rounds.size();
    cn.nlcc_constraints_run = nl_run;
    cn.count_valid = count_valid ? 1 : 0;
    cn.match_embeddings = count_valid ? matches : 0;
    cn.automorphisms = t.automorphisms;
    cn.match_subgraphs = (count_valid && t.automorphisms) ? matches / t.automorphisms : 0;
    cn.tokens = tokens;
    cn.edges_scanned_lcc = P.scanned;
    cn.edges_scanned_search = P.windows;
    cn.ms_lcc = ms_lcc;
    cn.ms_nlcc = ms_nlcc;
    cn.ms_final = ms_final;
    cn.ms_total = (double)ms_lcc + ms_nlcc + ms_final;
    cn.lcc_launches = P.lcc_launches;
    cn.ms_lcc_kernel = P.ms_lcc_kernel;
    cn.lcc_row_entries = P.rows;
    cn.lcc_active_vertices = P.alive;
    cn.lcc_alg_bytes = P.alg_bytes;
    cn.lcc_kernel_bytes = P.kernel_bytes;
    cn.lcc_first_entries = P.first_entries;
    cn.ms_lcc_first = P.ms_first;
    cn.ms_final_count = ms_fc;
    cn.ms_final_vertex = ms_fv;
    cn.ms_final_edge = ms_fe;
    cn.kernel_launches = P.launches;
    cn.lcc_compactions = P.compactions;
    cn.ms_search_kernel = P.ms_search_kernel;
    cn.search_launches = P.search_launches;
    cn.search_entries_nlcc = P.nlcc_entries;
    int status = CCPM_OK;
    if (over || (opt.run_final && !count_valid)) status = CCPM_EBUDGET;
    cn.status = status;
    *out = r;
    if (status == CCPM_EBUDGET) set_err(ctx, CCPM_EBUDGET, "a search budget was exceeded");
    return status;
#undef CUF
#undef RCF
}

int ccpm_prune(ccpm_ctx_t ctx, ccpm_graph_t g, ccpm_tmpl_t tm, const ccpm_options *opt_in, ccpm_result_t *out) {
    const int rc = prune(ctx, g, tm, opt_in, out);
    // every allocation comes before the result is written: a saved state is still
    // there to resume from
    if (rc != CCPM_ENOMEM || !ws_shrink(ctx, g)) return rc;
    g->prunes--;                                     // one prune
    return prune(ctx, g, tm, opt_in, out);
}

// Run the templates tmpls[order[0..)] of a batch on `W` worker contexts, one
// host thread each, taking templates from a shared counter in that order.
// Returns the first error.
static int run_batch(ccpm_ctx *ctx, ccpm_graph *g, const std::vector<int> &order, const ccpm_tmpl_t *tmpls,
                     const ccpm_options *opt, ccpm_result_t *outs, int W, int *budget_hit) {
    const int hi = (int)order.size();
    W = std::max(1, std::min(W, hi));
    while ((int)ctx->workers.size() < W) {
        ccpm_ctx *wk = nullptr;
        int rc = ccpm_ctx_create(ctx->device, nullptr, &wk);
        if (rc) return set_err(ctx, rc, "batch: worker context");
        ctx->workers.push_back(wk);
        if (cudaEventCreateWithFlags(&wk->wait_ev, cudaEventDisableTiming) != cudaSuccess)
            return set_err(ctx, CCPM_ECUDA, "batch: worker event");
    }
    // grid share: while k workers are busy a worker sizes its grids for
    // 1/min(share, k) of the SMs (the persistent-style search kernels would
    // otherwise hold every SM until they finish, and the small kernels of
    // other templates would wait behind them); the last templates of the
    // batch get the whole GPU back
    const int share = std::max(1, opt->grid_share);
    std::atomic<int> busy(0);
    // workers start after everything already queued on the caller's stream
    cudaEvent_t ready;
    CU(ctx, cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    if (cudaEventRecord(ready, ctx->stream) != cudaSuccess) {
        cudaEventDestroy(ready);
        return set_err(ctx, CCPM_ECUDA, "batch: event record");
    }
    for (int i = 0; i < W; i++)
        if (cudaStreamWaitEvent(ctx->workers[(size_t)i]->stream, ready, 0) != cudaSuccess) {
            cudaEventDestroy(ready);
            return set_err(ctx, CCPM_ECUDA, "batch: stream wait");
        }
    // the counter lives on this call's stack: the workers see it only
    // while their threads run
    for (int i = 0; i < W; i++) {
        ccpm_ctx *wk = ctx->workers[(size_t)i];
        wk->batch_busy = &busy;
        wk->batch_share = share;
    }
    std::atomic<int> next(0);
    std::atomic<int> first_err(0);
    std::atomic<int> budget(0);
    std::mutex err_mu;
    std::string err_msg;
    std::vector<std::thread> pool;
    for (int i = 0; i < W; i++) {
        ccpm_ctx *wk = ctx->workers[(size_t)i];
        pool.emplace_back([&, wk]() {
            cudaSetDevice(wk->device);
            for (int i = next.fetch_add(1); i < hi; i = next.fetch_add(1)) {
                if (first_err.load()) break;
                const int k = order[(size_t)i];
                busy.fetch_add(1);
                int rc = ccpm_prune(wk, g, tmpls[k], opt, &outs[k]);
                busy.fetch_sub(1);
                if (rc == CCPM_EBUDGET) {
                    budget.store(1);
                } else if (rc) {
                    int zero = 0;
                    if (first_err.compare_exchange_strong(zero, rc)) {
                        std::lock_guard<std::mutex> lk(err_mu);
                        err_msg = wk->err;
                    }
                }
            }
        });
    }
    for (auto &t : pool) t.join();
    for (int i = 0; i < W; i++) ctx->workers[(size_t)i]->batch_busy = nullptr;
    cudaEventDestroy(ready);
    if (budget.load()) *budget_hit = 1;
    if (first_err.load()) return set_err(ctx, first_err.load(), "batch: " + err_msg);
    return CCPM_OK;
}

int ccpm_prune_batch(ccpm_ctx_t ctx, ccpm_graph_t g, int T, const ccpm_tmpl_t *tmpls, const ccpm_options *opt_in,
                     ccpm_result_t *outs) {
    if (!ctx || !g || T < 0 || (T > 0 && (!tmpls || !outs))) return CCPM_EINVAL;
    for (int i = 0; i < T; i++)
        if (!tmpls[i]) return set_err(ctx, CCPM_EINVAL, "batch: NULL template");
    ccpm_options opt;
    if (opt_in) opt = *opt_in; else ccpm_options_default(&opt);
    CU(ctx, cudaSetDevice(ctx->device));
    // constraint generation is host work: do it here, not inside the workers
    for (int i = 0; i < T; i++) {
        if (!tmpls[i]->t.generated) {
            std::string err;
            int rc = constraints_generate(tmpls[i]->t, err);
            if (rc) return set_err(ctx, rc, err);
        }
    }
    int rc = ensure_label_rows(ctx, g);
    if (rc) return rc;
    int budget_hit = 0;
    const bool tune = opt.batch_workers <= 0 && g->tuned_workers <= 0;
    if (tune) {
        // autotune on one slice of this batch, the same templates for every
        // candidate (results are the same whatever the setting, so the slice's
        // results are simply made again): first the worker count, then the
        // windows a search scans before it hands work on, then the row length
        // of the flat short-row path, then the piece length of long rows.  The
        // choice is kept on the graph.
        // the slice: 32 templates spread evenly over the batch (long enough
        // for workers to queue, as they do on the whole batch)
        const int slice = std::max(1, std::min(T, 32));
        std::vector<int> sl;
        for (int i = 0; i < slice; i++) sl.push_back((int)((int64_t)i * T / slice));
        ccpm_options cand = opt;
        cand.search_split = 0;
        cand.short_rows = 0;
        cand.hub_degree = 0;
        cand.grid_share = 1;
        int best_w = 8;
        double best = 1e300;
        auto time_slice = [&](const ccpm_options &o, int W, double &ms) -> int {
            auto t0 = std::chrono::steady_clock::now();
            int rc2 = run_batch(ctx, g, sl, tmpls, &o, outs, W, &budget_hit);
            ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
            return rc2;
        };
        double ms = 0;
        int rc;
        for (int Wc : {1, 2, 4, 8, 16}) {
            if ((rc = time_slice(cand, Wc, ms))) return rc;
            if (ms < best) { best = ms; best_w = Wc; }
        }
        for (int gs : {2, 4}) {
            ccpm_options o = cand;
            o.grid_share = gs;
            if ((rc = time_slice(o, best_w, ms))) return rc;
            if (ms < best) { best = ms; cand.grid_share = gs; }
        }
        for (int sp : {512, 8192}) {
            ccpm_options o = cand;
            o.search_split = sp;
            if ((rc = time_slice(o, best_w, ms))) return rc;
            if (ms < best) { best = ms; cand.search_split = sp; }
        }
        for (int sr : {32, 256}) {
            ccpm_options o = cand;
            o.short_rows = sr;
            if ((rc = time_slice(o, best_w, ms))) return rc;
            if (ms < best) { best = ms; cand.short_rows = sr; }
        }
        for (int hd : {4096}) {
            ccpm_options o = cand;
            o.hub_degree = hd;
            if ((rc = time_slice(o, best_w, ms))) return rc;
            if (ms < best) { best = ms; cand.hub_degree = hd; }
        }
        g->tuned_workers = best_w;
        g->tuned_split = cand.search_split;
        g->tuned_short = cand.short_rows;
        g->tuned_hub = cand.hub_degree;
        g->tuned_share = cand.grid_share;
        g->tuned_ms = best;
    }
    int W = opt.batch_workers > 0 ? opt.batch_workers : g->tuned_workers;
    if (opt.batch_workers <= 0) {
        // the tuned settings apply where the caller left the library default
        if (opt.search_split == 0) opt.search_split = g->tuned_split;
        if (opt.short_rows == 0) opt.short_rows = g->tuned_short;
        if (opt.hub_degree == 0) opt.hub_degree = g->tuned_hub;
        if (opt.grid_share == 0) opt.grid_share = g->tuned_share;
    }
    if (T > 0) {
        // longest first when the results of an earlier call give each
        // template's time (the tail of the batch is then short templates)
        std::vector<int> order(T);
        for (int i = 0; i < T; i++) order[(size_t)i] = i;
        bool timed = true;
        for (int i = 0; i < T && timed; i++) timed = outs[i] && outs[i]->counts.ms_total > 0.0;
        if (timed)
            std::stable_sort(order.begin(), order.end(),
                             [&](int x, int y) { return outs[x]->counts.ms_total > outs[y]->counts.ms_total; });
        int rc = run_batch(ctx, g, order, tmpls, &opt, outs, W, &budget_hit);
        if (rc) return rc;
    }
    if (budget_hit) return set_err(ctx, CCPM_EBUDGET, "a search budget was exceeded in the batch");
    return CCPM_OK;
}

}  // extern "C"

namespace {

__global__ void k_or_words(uint32_t *dst, const uint32_t *src, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) dst[i] |= src[i];
}

// Arrays of a state, between two prunes (the workspace is idle).
int state_arrays(ccpm_ctx *ctx, ccpm_graph *g, int64_t words, uint32_t **om, uint32_t **eb) {
    for (;;) {
        int rc = dalloc(ctx, om, (size_t)g->n);
        if (!rc && (rc = dalloc(ctx, eb, (size_t)words + 1))) {
            cudaFree(*om);
            *om = nullptr;
        }
        if (rc != CCPM_ENOMEM || !ws_shrink(ctx, g)) return rc;
    }
}

// A result on graph g for template t holding (om, eb) copied from `src`
// arrays (the candidate set), ready for a resumed prune.
int result_from(ccpm_ctx *ctx, ccpm_graph *g, const Template &t, const uint32_t *om, const uint32_t *eb,
                int64_t words, ccpm_result **out) {
    ccpm_result *r = new (std::nothrow) ccpm_result();
    if (!r) return set_err(ctx, CCPM_ENOMEM, "result: host allocation");
    r->g = g;
    const int rc = state_arrays(ctx, g, words, &r->om, &r->eb);
    if (rc) {
        delete r;
        return rc;
    }
    r->tmpl_fp = tmpl_fingerprint(t);
    cudaError_t e = cudaMemcpyAsync(r->om, om, sizeof(uint32_t) * (size_t)g->n, cudaMemcpyDeviceToDevice, ctx->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(r->eb, eb, sizeof(uint32_t) * (size_t)(words + 1), cudaMemcpyDeviceToDevice, ctx->stream);
    if (e != cudaSuccess) {
        cudaFree(r->om); cudaFree(r->eb);
        delete r;
        return set_err(ctx, CCPM_ECUDA, std::string("result copy: ") + cudaGetErrorString(e));
    }
    *out = r;
    return CCPM_OK;
}

}  // namespace

extern "C" {

int ccpm_explore(ccpm_ctx_t ctx, ccpm_graph_t g, ccpm_tmpl_t base, int max_removed, const ccpm_options *opt_in,
                 ccpm_explore_variant *variants, int variants_cap, int *n_variants, int *level_found,
                 double *ms_candidates, ccpm_result_t *out) {
    if (!ctx || !g || !base || !out || max_removed < 0 || (variants_cap > 0 && !variants)) return CCPM_EINVAL;
    if (g->ctx->device != ctx->device) return set_err(ctx, CCPM_EINVAL, "graph lives on another device");
    const Template &B = base->t;
    const int m0 = (int)B.edges.size();
    if (m0 > 64) return set_err(ctx, CCPM_EINVAL, "explore: the base template may have at most 64 edges");
    ccpm_options opt;
    if (opt_in) opt = *opt_in; else ccpm_options_default(&opt);
    opt.resume = 0;
    CU(ctx, cudaSetDevice(ctx->device));
    if (n_variants) *n_variants = 0;
    if (level_found) *level_found = -1;
    if (ms_candidates) *ms_candidates = 0.0;
    cudaStream_t s = ctx->stream;
    const int64_t words = (g->m + 31) / 32;
    // connected variants by level: every set of `k` template edges whose
    // removal leaves the template connected (vertices are never removed, so
    // template vertex q means the same in every variant)
    struct Variant { int level; uint64_t removed; Template t; };
    std::vector<Variant> vs;
    for (int k = 0; k <= std::min(max_removed, m0 - 1); k++) {
        std::vector<int> pick(k);
        for (int i = 0; i < k; i++) pick[i] = i;
        for (;;) {
            uint64_t mask = 0;
            for (int i : pick) mask |= 1ull << i;
            std::vector<int32_t> ed;
            for (int e = 0; e < m0; e++)
                if (!((mask >> e) & 1ull)) { ed.push_back(B.edges[(size_t)e].first); ed.push_back(B.edges[(size_t)e].second); }
            Variant v{k, mask, Template{}};
            if (template_build(v.t, B.n0, B.labels, (int)ed.size() / 2, ed.data()) == CCPM_OK) vs.push_back(std::move(v));
            int i = k - 1;
            while (i >= 0 && pick[(size_t)i] == m0 - k + i) i--;
            if (i < 0) break;
            pick[(size_t)i]++;
            for (int j = i + 1; j < k; j++) pick[(size_t)j] = pick[(size_t)j - 1] + 1;
        }
    }
    // the candidate set: the union of the LCC fixpoints of every variant (local
    // constraints only, so each costs one LCC to fixpoint); it holds every
    // match of every variant
    uint32_t *c_om = nullptr, *c_eb = nullptr;
    int rc;
    if ((rc = state_arrays(ctx, g, words, &c_om, &c_eb))) return rc;
    ccpm_result *made = nullptr;         // the union, if this call made it
    auto cleanup = [&]() { cudaFree(c_om); cudaFree(c_eb); };
    auto fail_c = [&](int code) { cleanup(); ccpm_result_destroy(made); return code; };
    if (cudaMemsetAsync(c_om, 0, sizeof(uint32_t) * (size_t)g->n, s) != cudaSuccess ||
        cudaMemsetAsync(c_eb, 0, sizeof(uint32_t) * (size_t)(words + 1), s) != cudaSuccess)
        return fail_c(set_err(ctx, CCPM_ECUDA, "explore: memset"));
    ccpm_options lcc_only = opt;
    lcc_only.run_final = 0;
    lcc_only.order_mode = CCPM_ORDER_FIXED;
    auto t_start = std::chrono::steady_clock::now();
    for (auto &v : vs) {
        ccpm_tmpl tl;
        tl.ctx = ctx;
        tl.t = v.t;
        tl.t.generated = true;          // no non-local constraint: LCC only
        tl.t.k0.clear();
        tl.t.order.clear();
        ccpm_result *r = nullptr;
        rc = ccpm_prune(ctx, g, &tl, &lcc_only, &r);
        if (rc && rc != CCPM_EBUDGET) return fail_c(rc);
        const int gr = grid_for(ctx, std::max<int64_t>(g->n, words), 256, 8);
        k_or_words<<<gr, 256, 0, s>>>(c_om, r->om, g->n);
        k_or_words<<<gr, 256, 0, s>>>(c_eb, r->eb, words);
        ccpm_result_destroy(r);
        if (cudaGetLastError() != cudaSuccess) return fail_c(set_err(ctx, CCPM_ECUDA, "explore: union"));
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail_c(set_err(ctx, CCPM_ECUDA, "explore: sync"));
    if (ms_candidates)
        *ms_candidates = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t_start).count();
    // the union of the matching variants' omega* and E* at the first level
    // with a match
    ccpm_result *u = *out;
    if (u && u->g != g) return fail_c(set_err(ctx, CCPM_EINVAL, "explore: result was made for another graph"));
    if (!u) {
        if ((rc = result_from(ctx, g, B, c_om, c_eb, words, &made))) return fail_c(rc);
        u = made;
    }
    u->tmpl_fp = tmpl_fingerprint(B);
    u->phase_rounds.clear();
    u->logs.clear();
    std::memset(&u->counts, 0, sizeof(u->counts));
    cudaMemsetAsync(u->om, 0, sizeof(uint32_t) * (size_t)g->n, s);
    cudaMemsetAsync(u->eb, 0, sizeof(uint32_t) * (size_t)(words + 1), s);
    int found = -1, nv = 0;
    bool budget = false;
    ccpm_options resumed = opt;
    resumed.resume = 1;
    for (int k = 0; k <= max_removed && found < 0; k++) {
        bool any = false;
        for (auto &v : vs) {
            if (v.level != k) continue;
            ccpm_tmpl tv;
            tv.ctx = ctx;
            tv.t = v.t;
            ccpm_result *r = nullptr;
            if ((rc = result_from(ctx, g, tv.t, c_om, c_eb, words, &r))) return fail_c(rc);
            rc = ccpm_prune(ctx, g, &tv, &resumed, &r);
            if (rc == CCPM_EBUDGET) budget = true;
            else if (rc) { ccpm_result_destroy(r); return fail_c(rc); }
            const ccpm_counts &c = r->counts;
            if (c.active_v > 0) {
                any = true;
                const int gr = grid_for(ctx, std::max<int64_t>(g->n, words), 256, 8);
                k_or_words<<<gr, 256, 0, s>>>(u->om, r->om, g->n);
                k_or_words<<<gr, 256, 0, s>>>(u->eb, r->eb, words);
            }
            if (nv < variants_cap) {
                ccpm_explore_variant &o = variants[nv];
                o.level = k;
                o.n_edges = (int32_t)v.t.edges.size();
                o.removed = v.removed;
                o.active_v = c.active_v;
                o.active_e_dir = c.active_e_dir;
                o.match_embeddings = c.match_embeddings;
                o.count_valid = c.count_valid;
                o.status = c.status;
                o.ms_total = c.ms_total;
            }
            nv++;
            ccpm_result_destroy(r);
        }
        if (any) found = k;
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail_c(set_err(ctx, CCPM_ECUDA, "explore: sync"));
    cleanup();
    if (n_variants) *n_variants = nv;
    if (level_found) *level_found = found;
    *out = u;
    // counts of the union
    CU(ctx, cudaMemsetAsync(ctx->ws.cnt, 0, 2 * sizeof(unsigned long long), s));
    k_count<<<grid_for(ctx, std::max<int64_t>(g->n, words), 256, 8), 256, 0, s>>>(g->n, u->om, words, u->eb, ctx->ws.cnt);
    CU(ctx, cudaGetLastError());
    CU(ctx, cudaMemcpyAsync(ctx->ws.cnt_h, ctx->ws.cnt, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    CU(ctx, cudaStreamSynchronize(s));
    u->counts.active_v = (int64_t)ctx->ws.cnt_h[0];
    u->counts.active_e_dir = (int64_t)ctx->ws.cnt_h[1];
    if (budget) return set_err(ctx, CCPM_EBUDGET, "explore: a search budget was exceeded");
    return CCPM_OK;
}

int ccpm_result_omega(ccpm_result_t r, uint32_t *dst, int64_t n, int dst_on_device) {
    if (!r || !dst || n != r->g->n) return CCPM_EINVAL;
    ccpm_ctx *ctx = r->g->ctx;
    CU(ctx, cudaSetDevice(ctx->device));
    CU(ctx, cudaMemcpyAsync(dst, r->om, sizeof(uint32_t) * (size_t)n,
                            dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream));
    CU(ctx, cudaStreamSynchronize(ctx->stream));
    return CCPM_OK;
}

int ccpm_result_edge_bitmap(ccpm_result_t r, uint32_t *dst, int64_t words, int dst_on_device) {
    if (!r || !dst || words != (r->g->m + 31) / 32) return CCPM_EINVAL;
    ccpm_ctx *ctx = r->g->ctx;
    CU(ctx, cudaSetDevice(ctx->device));
    CU(ctx, cudaMemcpyAsync(dst, r->eb, sizeof(uint32_t) * (size_t)words,
                            dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream));
    CU(ctx, cudaStreamSynchronize(ctx->stream));
    return CCPM_OK;
}

int ccpm_result_constraint_log(ccpm_result_t r, int i, ccpm_constraint_log *out) {
    if (!r || !out || i < 0 || i >= (int)r->logs.size()) return CCPM_EINVAL;
    *out = r->logs[(size_t)i];
    return CCPM_OK;
}

int ccpm_result_counts(ccpm_result_t r, ccpm_counts *out) {
    if (!r || !out) return CCPM_EINVAL;
    *out = r->counts;
    return CCPM_OK;
}

int ccpm_result_phase_rounds(ccpm_result_t r, int32_t *dst, int cap) {
    if (!r || (!dst && cap > 0)) return CCPM_EINVAL;
    int k = std::min(cap, (int)r->phase_rounds.size());
    for (int i = 0; i < k; i++) dst[i] = r->phase_rounds[(size_t)i];
    return CCPM_OK;
}

// Does a listing copy the result's entries into rows of their own (K4) before it
// searches?  Otherwise it reads the label-grouped copy of the graph's rows.  The
// copy costs some 0.1 ms and several passes over all vertices; on the graph's rows
// a label group holds entries outside the result, and partial maps run over edges
// outside it.  us without / with the copy (list of 1000, no counts):
//   result entries, template, graph                      without     with
//      17,300  triangle, Zipf labels, 32M vertices           224    1,396
//     179,272  triangle, Zipf labels, 32M                    366    1,601
//     117,340  triangle, Zipf labels, 16M                    268      976
//      26,920  5-cycle, Zipf labels, 1M                      724      767
//     149,792  4-cycle, Zipf labels, 4M                    1,099    1,388
//      14,130  two 4-cycles sharing a path, 100 labels, 1M 3,738    2,401
//       2,284  4-cycle + triangle, degree labels, 1M         172      278
//      10,294  the same, 22K                                 598      688
//      22,478  the same, 26K                               2,085    1,372
//     117,320  the same, 80K                              14,683    2,963
//     879,814  the same, 1M                              266,655    1,716
//     486,850  tree, degree labels, 1M                     2,098    2,338
// What makes the difference is the length of the groups: past a window (32
// entries) on average, as under hubs that carry their degree as label, every step
// of a search reads several.  With shorter ones the copy was worse in 207 of 231
// results of 2 to 940,000 entries and at most 1.6 times as fast, with three
// template vertices always worse.  Results that no final search made may hold many
// entries that no match uses; they are copied, unless they are small.  The first
// listing of a graph whose rows are not grouped yet copies, too: grouping them
// pays off from the second on.
constexpr int64_t kCopyEntries = (int64_t)1 << 14;

static bool listing_copies(ccpm_graph *g, const ccpm_result *r, const Template &t) {
    if (!g->lrows_ready.load() && g->listings == 0) return true;
    if (r->counts.active_e_dir < kCopyEntries || t.n0 <= 3) return false;
    if (!r->counts.count_valid) return true;
    for (auto &e : t.edges)
        for (int x : {e.first, e.second}) {
            const int y = x == e.first ? e.second : e.first;
            // mean row of label(x) times the share of entries that lead to label(y)
            const double row = (double)g->label_rows[t.labels[x]] / (double)std::max<int64_t>(g->label_freq[t.labels[x]], 1);
            if (row * (double)g->label_rows[t.labels[y]] > 32.0 * (double)g->m) return true;
        }
    return false;
}

static int list_matches(ccpm_ctx_t ctx, ccpm_result_t r, ccpm_tmpl_t tm, const ccpm_options *opt_in,
                        int32_t *list, uint64_t list_cap, uint64_t *vertex_counts, uint64_t *entry_counts,
                        int dst_on_device, uint64_t *n_matches) {
    if (!ctx || !r || !tm || !n_matches || (list_cap > 0 && !list)) return CCPM_EINVAL;
    *n_matches = 0;
    ccpm_graph *g = r->g;
    if (g->ctx->device != ctx->device) return set_err(ctx, CCPM_EINVAL, "result lives on another device");
    Template &t = tm->t;
    if (r->tmpl_fp != tmpl_fingerprint(t)) return set_err(ctx, CCPM_EINVAL, "result was made for another template");
    ccpm_options opt;
    if (opt_in) opt = *opt_in; else ccpm_options_default(&opt);
    CU(ctx, cudaSetDevice(ctx->device));
    const int hub_deg = opt.hub_degree > 0 ? std::min(opt.hub_degree, kMaxHubDeg) : kDefaultHubDeg;
    const uint64_t budget = opt.search_budget ? opt.search_budget : ~0ull;
    const uint64_t split = opt.search_split < 0 ? 0 : (opt.search_split == 0 ? kSpillAfter : (uint64_t)opt.search_split);
    // as for a prune: with a caller's own budget, no handing on to idle warps
    const bool starve = opt.search_split >= 0 && opt.search_budget == 0;
    int rc = ws_ensure(ctx, g, hub_deg);
    if (rc) return rc;
    Workspace &w = ctx->ws;
    cudaStream_t s = ctx->stream;
    // host outputs are filled through device buffers of this call
    int32_t *d_list = list;
    unsigned long long *d_vc = (unsigned long long *)vertex_counts, *d_ec = (unsigned long long *)entry_counts;
    bool own = false;
    auto release = [&]() {
        if (own) { cudaFree(d_list); cudaFree(d_vc); cudaFree(d_ec); }
    };
    if (!dst_on_device) {
        own = true;
        d_list = nullptr; d_vc = nullptr; d_ec = nullptr;
        if ((list_cap && (rc = dalloc(ctx, &d_list, (size_t)(list_cap * (uint64_t)t.n0)))) ||
            (vertex_counts && (rc = dalloc(ctx, &d_vc, (size_t)g->n))) ||
            (entry_counts && (rc = dalloc(ctx, &d_ec, (size_t)std::max<int64_t>(g->m, 1))))) {
            release();
            return rc;
        }
    }
#define CUR(call)                                                                        \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess) {                                                         \
            release();                                                                   \
            return set_err(ctx, CCPM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
        }                                                                                \
    } while (0)
    if (d_vc) CUR(cudaMemsetAsync(d_vc, 0, sizeof(unsigned long long) * (size_t)g->n, s));
    if (d_ec) CUR(cudaMemsetAsync(d_ec, 0, sizeof(unsigned long long) * (size_t)g->m, s));
    CUR(cudaMemsetAsync(w.cnt, 0, sizeof(unsigned long long), s));
    // the root is the template vertex with the rarest label
    int root = 0;
    for (int q = 1; q < t.n0; q++)
        if (g->label_freq[t.labels[q]] < g->label_freq[t.labels[root]]) root = q;
    const uint32_t all = t.n0 == 32 ? 0xFFFFFFFFu : ((1u << t.n0) - 1u);
    build_plan(t, all, t.adj, root, g->label_freq, true, w.plans_h[0], -1, nullptr);
    CUR(cudaMemcpyAsync(w.plans, w.plans_h, sizeof(DevPlan), cudaMemcpyHostToDevice, s));
    // every match lies inside the result's vertices and entries: the search reads
    // rows that hold nothing else, label group by label group from a directory, or
    // where that does not pay the graph's own grouped rows
    Pipeline P;
    P.ctx = ctx;
    P.g = g;
    P.t = &t;
    P.lrp = g->rp;
    P.lcol = g->col;
    P.lbits = w.ebits;
    const uint32_t *om = r->om;
    if ((rc = clear_search(ctx, w))) { release(); return rc; }
    bool any = true;                      // something to search, as far as the host knows
    const bool copies = listing_copies(g, r, t);
    g->listings++;
    if (copies || ensure_label_rows(ctx, g)) {
        om = w.om[0];
        LabelMask lm;
        std::memset(&lm, 0, sizeof(lm));
        for (int q = 0; q < t.n0; q++) lm.m[t.labels[q]] |= 1u << q;
        CUR(cudaMemsetAsync(&w.ctl->init, 0, sizeof(RoundStats), s));
        CUR(cudaMemsetAsync(w.ebits, 0, sizeof(uint32_t) * (size_t)(w.words + 1), s));
        k_init<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, g->rp, g->lab, lm, r->om, w.om[0], w.om[1], nullptr,
                                                           nullptr, 0, w.small[0], w.med[0], w.chunk[0], w.acc,
                                                           &w.ctl->init, hub_deg, P.short_max, 0u, nullptr, nullptr, 0);
        CUR(cudaGetLastError());
        k_live_entries<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, g->rp, g->col, om, r->eb, w.ebits, w.deg, w.st);
        CUR(cudaGetLastError());
        if ((rc = read_control(ctx, w))) { release(); return rc; }
        const RoundStats &lists = w.ctl_h->init;
        if (lists.n_hub_slots > (unsigned)w.acc_cap || (int64_t)lists.n_chunk > w.chunk_cap) {
            release();
            return set_err(ctx, CCPM_EOVERFLOW, "hub bookkeeping overflow");
        }
        P.n_small = lists.n_small;
        P.n_med = lists.n_med;
        P.n_chunk = lists.n_chunk;
        P.last_kept = (int64_t)w.st_h->kept;
        any = P.last_kept > 0;
        if (any && ((rc = P.compact()) || (rc = clear_search(ctx, w)))) { release(); return rc; }
    }
    bool over = false;
    if (any) {
        k_collect_roots<<<grid_for(ctx, g->n, 256, 8), 256, 0, s>>>(g->n, om, 1u << root, w.roots, w.st);
        CUR(cudaGetLastError());
        SearchArgs a{};
        a.rp = g->rp;
        a.col = g->col;
        a.rl = P.gen >= 0 ? P.lrp : g->rp;
        a.lcol = P.gen >= 0 ? P.lcol : g->lcol;
        a.nlab = P.gen >= 0 ? P.lnlab : g->nlab;
        P.directory(a);
        a.om = om;
        a.roots = w.roots;
        a.n_roots = -1;
        a.plans = w.plans;
        a.heads = 1u << root;
        a.sat = w.sat;
        a.st = w.st;
        a.budget = budget;
        a.cap = ~0ull;
        a.items = w.items;
        a.items_cap = w.items_cap;
        a.enum_heads = 1;
        a.list_out = d_list;
        a.list_cap = list_cap;
        a.list_n0 = t.n0;
        a.list_count = w.cnt;
        a.vcnt = d_vc;
        a.ecnt = d_ec;
        int64_t launches = 0;
        const SearchMode mode{3, split, starve};
        if ((rc = queue_search(ctx, w, a, mode, t.n0, launches)) || (rc = read_control(ctx, w)) ||
            (!search_complete(w, mode) && (rc = finish_search(ctx, w, a, mode, launches)))) {
            release();
            return rc;
        }
        over = w.st_h->overflow != 0;
    }
    // the counters read last are the search's (or show that there was none)
    const unsigned long long found = any ? w.cnt_h[0] : 0ull;
    if (!dst_on_device) {
        const uint64_t rows = std::min<uint64_t>((uint64_t)found, list_cap);
        if (rows) CUR(cudaMemcpyAsync(list, d_list, sizeof(int32_t) * (size_t)(rows * (uint64_t)t.n0), cudaMemcpyDeviceToHost, s));
        if (d_vc) CUR(cudaMemcpyAsync(vertex_counts, d_vc, sizeof(uint64_t) * (size_t)g->n, cudaMemcpyDeviceToHost, s));
        if (d_ec) CUR(cudaMemcpyAsync(entry_counts, d_ec, sizeof(uint64_t) * (size_t)g->m, cudaMemcpyDeviceToHost, s));
        CUR(cudaStreamSynchronize(s));
    }
#undef CUR
    release();
    *n_matches = found;
    if (over) return set_err(ctx, CCPM_EBUDGET, "a listing search ran out of its window budget: outputs incomplete");
    return CCPM_OK;
}

const uint32_t *ccpm_result_omega_device(ccpm_result_t r) { return r ? r->om : nullptr; }
const uint32_t *ccpm_result_edge_bitmap_device(ccpm_result_t r) { return r ? r->eb : nullptr; }

int ccpm_result_matches(ccpm_ctx_t ctx, ccpm_result_t r, ccpm_tmpl_t tm, const ccpm_options *opt_in,
                        int32_t *list, uint64_t list_cap, uint64_t *vertex_counts, uint64_t *entry_counts,
                        int dst_on_device, uint64_t *n_matches) {
    const int rc = list_matches(ctx, r, tm, opt_in, list, list_cap, vertex_counts, entry_counts, dst_on_device, n_matches);
    if (rc != CCPM_ENOMEM || !ws_shrink(ctx, r->g)) return rc;
    return list_matches(ctx, r, tm, opt_in, list, list_cap, vertex_counts, entry_counts, dst_on_device, n_matches);
}

int ccpm_graph_batch_workers(ccpm_graph_t g) { return g ? g->tuned_workers : 0; }

int ccpm_graph_batch_tuning(ccpm_graph_t g, int *workers, int *grid_share, int *search_split, int *short_rows,
                            int *hub_degree, double *slice_ms) {
    if (!g) return CCPM_EINVAL;
    if (workers) *workers = g->tuned_workers;
    if (grid_share) *grid_share = g->tuned_share;
    if (search_split) *search_split = g->tuned_split;
    if (short_rows) *short_rows = g->tuned_short;
    if (hub_degree) *hub_degree = g->tuned_hub;
    if (slice_ms) *slice_ms = g->tuned_ms;
    return CCPM_OK;
}

void ccpm_result_destroy(ccpm_result_t r) {
    if (!r) return;
    cudaSetDevice(r->g->ctx->device);
    cudaFree(r->om);
    cudaFree(r->eb);
    delete r;
}

// ---- checkpoint/resume: one host blob per state (layout in ccpm.h)

namespace {
struct StateHeader {
    char magic[8];
    uint32_t version;
    uint32_t header_bytes;
    int64_t n, m_dir, words;
    uint64_t graph_fp, tmpl_fp;
    uint32_t counts_bytes, n_phases;
    uint64_t payload_bytes;
    uint64_t payload_fnv;
    uint64_t reserved[2];
};
static_assert(sizeof(StateHeader) == 96, "state header layout");
constexpr char kStateMagic[8] = {'C', 'C', 'P', 'M', 'S', 'T', 'A', 'T'};
constexpr uint32_t kStateVersion = 1;

size_t state_payload_bytes(int64_t n, int64_t words, size_t n_phases) {
    return sizeof(ccpm_counts) + sizeof(int32_t) * n_phases + sizeof(uint32_t) * (size_t)(n + words);
}
}  // namespace

int ccpm_state_export(ccpm_result_t r, void *buf, size_t *len) {
    if (!r || !len) return CCPM_EINVAL;
    ccpm_graph *g = r->g;
    ccpm_ctx *ctx = g->ctx;
    const int64_t words = (g->m + 31) / 32;
    const size_t payload = state_payload_bytes(g->n, words, r->phase_rounds.size());
    const size_t need = sizeof(StateHeader) + payload;
    if (!buf) { *len = need; return CCPM_OK; }
    if (*len < need) {
        *len = need;
        return set_err(ctx, CCPM_EINVAL, "state buffer too small");
    }
    StateHeader h;
    std::memset(&h, 0, sizeof(h));
    std::memcpy(h.magic, kStateMagic, 8);
    h.version = kStateVersion;
    h.header_bytes = sizeof(StateHeader);
    h.n = g->n;
    h.m_dir = g->m;
    h.words = words;
    h.graph_fp = graph_fingerprint(*g);
    h.tmpl_fp = r->tmpl_fp;
    h.counts_bytes = sizeof(ccpm_counts);
    h.n_phases = (uint32_t)r->phase_rounds.size();
    h.payload_bytes = payload;
    unsigned char *p = (unsigned char *)buf + sizeof(StateHeader);
    std::memcpy(p, &r->counts, sizeof(ccpm_counts));
    p += sizeof(ccpm_counts);
    if (!r->phase_rounds.empty()) std::memcpy(p, r->phase_rounds.data(), sizeof(int32_t) * r->phase_rounds.size());
    p += sizeof(int32_t) * r->phase_rounds.size();
    CU(ctx, cudaSetDevice(ctx->device));
    CU(ctx, cudaMemcpy(p, r->om, sizeof(uint32_t) * (size_t)g->n, cudaMemcpyDeviceToHost));
    p += sizeof(uint32_t) * (size_t)g->n;
    CU(ctx, cudaMemcpy(p, r->eb, sizeof(uint32_t) * (size_t)words, cudaMemcpyDeviceToHost));
    h.payload_fnv = fnv1a((const unsigned char *)buf + sizeof(StateHeader), payload);
    std::memcpy(buf, &h, sizeof(h));
    *len = need;
    return CCPM_OK;
}

int ccpm_state_import(ccpm_ctx_t ctx, ccpm_graph_t g, ccpm_tmpl_t tm, const void *buf, size_t len,
                      ccpm_result_t *out) {
    if (!ctx || !g || !tm || !buf || !out) return CCPM_EINVAL;
    *out = nullptr;
    if (g->ctx->device != ctx->device) return set_err(ctx, CCPM_EINVAL, "graph lives on another device");
    StateHeader h;
    if (len < sizeof(h)) return set_err(ctx, CCPM_EINVAL, "state: truncated header");
    std::memcpy(&h, buf, sizeof(h));
    if (std::memcmp(h.magic, kStateMagic, 8) != 0 || h.version != kStateVersion ||
        h.header_bytes != sizeof(StateHeader) || h.counts_bytes != sizeof(ccpm_counts))
        return set_err(ctx, CCPM_EINVAL, "state: not a saved state of this library version");
    const int64_t words = (g->m + 31) / 32;
    if (h.n != g->n || h.m_dir != g->m || h.words != words || h.graph_fp != graph_fingerprint(*g))
        return set_err(ctx, CCPM_EINVAL, "state: saved for another graph");
    if (h.tmpl_fp != tmpl_fingerprint(tm->t)) return set_err(ctx, CCPM_EINVAL, "state: saved for another template");
    if (h.n_phases > (1u << 20)) return set_err(ctx, CCPM_EINVAL, "state: bad phase count");
    const size_t payload = state_payload_bytes(g->n, words, h.n_phases);
    if (h.payload_bytes != payload || len < sizeof(h) + payload) return set_err(ctx, CCPM_EINVAL, "state: truncated");
    const unsigned char *p = (const unsigned char *)buf + sizeof(h);
    if (fnv1a(p, payload) != h.payload_fnv) return set_err(ctx, CCPM_EINVAL, "state: checksum mismatch");
    CU(ctx, cudaSetDevice(ctx->device));
    ccpm_result *r = new (std::nothrow) ccpm_result();
    if (!r) return set_err(ctx, CCPM_ENOMEM, "result: host allocation");
    r->g = g;
    r->tmpl_fp = h.tmpl_fp;
    int rc = dalloc(ctx, &r->om, (size_t)g->n);
    if (!rc) rc = dalloc(ctx, &r->eb, (size_t)words + 1);
    if (rc) {
        cudaFree(r->om); cudaFree(r->eb);
        delete r;
        return rc;
    }
    std::memcpy(&r->counts, p, sizeof(ccpm_counts));
    p += sizeof(ccpm_counts);
    r->phase_rounds.resize(h.n_phases);
    if (h.n_phases) std::memcpy(r->phase_rounds.data(), p, sizeof(int32_t) * h.n_phases);
    p += sizeof(int32_t) * h.n_phases;
    cudaError_t e = cudaMemcpy(r->om, p, sizeof(uint32_t) * (size_t)g->n, cudaMemcpyHostToDevice);
    p += sizeof(uint32_t) * (size_t)g->n;
    if (e == cudaSuccess) e = cudaMemcpy(r->eb, p, sizeof(uint32_t) * (size_t)words, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(r->eb + words, 0, sizeof(uint32_t));
    if (e != cudaSuccess) {
        cudaFree(r->om); cudaFree(r->eb);
        delete r;
        return set_err(ctx, CCPM_ECUDA, std::string("state import: ") + cudaGetErrorString(e));
    }
    *out = r;
    return CCPM_OK;
}

}  // extern "C"

// ===========================================================================
// Allocation-free LCC entry point
//
// Some callers cannot allocate device memory while they run: code that works
// inside a memory budget reserved up front, host code holding a lock in which
// cudaMalloc may block on the driver, or applications whose allocator is
// owned by someone else.  ccpm_lcc_fixpoint_noalloc runs local constraint
// checking to its fixpoint using only the caller's inputs and outputs plus a
// fixed scratch area compiled into this library.
// ===========================================================================

#include <mutex>

namespace {

// Scratch of the allocation-free entry point: the second omega buffer, the
// frontier lists, the split-row accumulators and the round counters.  It is
// part of the library image, so every GPU on which the library's kernels are
// loaded holds these bytes until the process exits.
constexpr size_t kNoAllocScratchBytes = (size_t)16 << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
// counters of the first round's lists and of two groups of queued rounds
constexpr int kNoAllocRounds = 4;
static __device__ RoundStats g_noalloc_rounds[1 + 2 * kNoAllocRounds];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kNoAllocMaxDevices] = {};
void *g_noalloc_rounds_addr[kNoAllocMaxDevices] = {};

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct NoAllocLayout {
    size_t om2, small[2], med[2], chunk[2], acc, st, total;
    int64_t chunk_cap, acc_cap;
};

NoAllocLayout noalloc_layout(int64_t n, int64_t m, int hub) {
    NoAllocLayout L{};
    L.chunk_cap = 2 * (m / hub) + 16;
    L.acc_cap = m / hub + 16;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off = up256(off + bytes); return at; };
    L.om2 = take(sizeof(uint32_t) * (size_t)n);
    for (int i = 0; i < 2; i++) L.small[i] = take(sizeof(int32_t) * (size_t)n);
    for (int i = 0; i < 2; i++) L.med[i] = take(sizeof(int32_t) * (size_t)n);
    for (int i = 0; i < 2; i++) L.chunk[i] = take(sizeof(ChunkItem) * (size_t)L.chunk_cap);
    L.acc = take(sizeof(HubAcc) * (size_t)L.acc_cap);
    L.st = take(sizeof(RoundStats));
    L.total = off;
    return L;
}

// Template tables straight from the caller's arrays (no heap use).
const char *noalloc_template(int n0, const uint8_t *labels, int m0, const int32_t *edges,
                             DevTmpl &d, LabelMask &lm) {
    if (n0 < 2 || n0 > kMaxT) return "template must have 2..32 vertices";
    if (m0 < 1 || m0 > CCPM_MAX_TMPL_EDGES || !labels || !edges) return "template needs 1..496 edges";
    std::memset(&d, 0, sizeof(d));
    std::memset(&lm, 0, sizeof(lm));
    d.n0 = n0;
    for (int i = 0; i < m0; i++) {
        int a = edges[2 * i], b = edges[2 * i + 1];
        if (a < 0 || b < 0 || a >= n0 || b >= n0 || a == b) return "bad template edge";
        if ((d.adj[a] >> b) & 1u) return "duplicate template edge";
        d.adj[a] |= 1u << b;
        d.adj[b] |= 1u << a;
    }
    int n_pairs = 0;
    uint32_t seen = 1u, fr = 1u;
    while (fr) {
        uint32_t nx = 0;
        for (int q = 0; q < n0; q++) if ((fr >> q) & 1u) nx |= d.adj[q];
        nx &= ~seen;
        seen |= nx;
        fr = nx;
    }
    if (seen != (n0 == 32 ? 0xFFFFFFFFu : ((1u << n0) - 1u))) return "template is not connected";
    for (int q = 0; q < n0; q++) {
        lm.m[labels[q]] |= 1u << q;
        uint32_t done = 0;
        for (int b = 0; b < n0; b++) {
            if (!((d.adj[q] >> b) & 1u) || ((done >> b) & 1u)) continue;
            uint32_t grp = 0;
            for (int c = 0; c < n0; c++)
                if (((d.adj[q] >> c) & 1u) && labels[c] == labels[b]) grp |= 1u << c;
            done |= grp;
            if (__builtin_popcount(grp) >= 2) {
                if (++n_pairs > kMaxCls) return "template has more than 32 label-multiplicity classes";
                add_class(d, q, grp);
            }
        }
    }
    return nullptr;
}

// The body of the entry point below; it may leave another device current.
int lcc_fixpoint_noalloc_body(int device, void *cuda_stream, int64_t n, int64_t m_dir,
                              const int64_t *row_ptr, const int32_t *col, const uint8_t *labels,
                              int n0, const uint8_t *tmpl_labels, int m0, const int32_t *tmpl_edges,
                              uint32_t *omega, uint32_t *ebits, int32_t *rounds,
                              int64_t *edges_scanned, char *errbuf, size_t errlen) {
    auto fail = [&](int code, const char *msg) {
        if (errbuf && errlen) std::snprintf(errbuf, errlen, "%s", msg);
        return code;
    };
    if (device < 0 || device >= kNoAllocMaxDevices) return fail(CCPM_EINVAL, "device index out of range");
    if (n < 1 || n >= ((int64_t)1 << 31) || m_dir < 0 || !row_ptr || !labels || !omega ||
        (m_dir > 0 && (!col || !ebits)))
        return fail(CCPM_EINVAL, "need 1 <= n < 2^31, m_dir >= 0 and non-NULL device arrays");
    DevTmpl dt;
    LabelMask lm;
    if (const char *why = noalloc_template(n0, tmpl_labels, m0, tmpl_edges, dt, lm)) return fail(CCPM_EINVAL, why);
    const int hub = kDefaultHubDeg;
    const NoAllocLayout L = noalloc_layout(n, m_dir, hub);
    if (L.total > kNoAllocScratchBytes) {
        char msg[160];
        std::snprintf(msg, sizeof(msg),
                      "graph too large for the allocation-free entry point: needs %zu bytes of scratch, "
                      "the fixed area holds %zu", L.total, kNoAllocScratchBytes);
        return fail(CCPM_EINVAL, msg);
    }
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return fail(CCPM_ECUDA, cudaGetErrorString(e));
    unsigned char *base = nullptr;
    RoundStats *rounds_dev = nullptr;
    {
        // once per device, with that device current: the device address of the
        // scratch array (the host-side symbol is only a stand-in)
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[device]) {
            void *p = nullptr, *q = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e == cudaSuccess) e = cudaGetSymbolAddress(&q, g_noalloc_rounds);
            if (e != cudaSuccess || !p || !q)
                return fail(CCPM_ECUDA, "cudaGetSymbolAddress of the scratch arrays failed");
            g_noalloc_addr[device] = p;
            g_noalloc_rounds_addr[device] = q;
        }
        rounds_dev = (RoundStats *)g_noalloc_rounds_addr[device];
        base = (unsigned char *)g_noalloc_addr[device];
    }
    int num_sms = 0;
    e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return fail(CCPM_ECUDA, cudaGetErrorString(e));
    cudaStream_t s = (cudaStream_t)cuda_stream;
    {
        // the scratch is sized from m_dir: the offsets must agree with it
        // before any kernel writes there (the two 8-byte ends, read into the
        // stack as one strided copy)
        int64_t ends[2] = {-1, -1};
        e = cudaMemcpy2DAsync(ends, sizeof(int64_t), row_ptr, sizeof(int64_t) * (size_t)n, sizeof(int64_t), 2,
                              cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return fail(CCPM_ECUDA, cudaGetErrorString(e));
        if (ends[0] != 0 || ends[1] != m_dir) return fail(CCPM_EINVAL, "row_ptr[0] must be 0 and row_ptr[n] == m_dir");
    }
    uint32_t *om[2] = {omega, (uint32_t *)(base + L.om2)};
    int32_t *small[2] = {(int32_t *)(base + L.small[0]), (int32_t *)(base + L.small[1])};
    int32_t *med[2] = {(int32_t *)(base + L.med[0]), (int32_t *)(base + L.med[1])};
    ChunkItem *chunk[2] = {(ChunkItem *)(base + L.chunk[0]), (ChunkItem *)(base + L.chunk[1])};
    HubAcc *acc = (HubAcc *)(base + L.acc);
    RoundStats *st = (RoundStats *)(base + L.st);
    RoundStats hs;
    auto grid = [&](int64_t items, int per_block) {
        int64_t need = (items + per_block - 1) / per_block;
        return (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)num_sms * 8));
    };
    auto read_stats = [&]() {
        cudaError_t r = cudaMemcpyAsync(&hs, st, sizeof(RoundStats), cudaMemcpyDeviceToHost, s);
        if (r == cudaSuccess) r = cudaStreamSynchronize(s);
        return r;
    };
#define NA_CU(call)                                          \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return fail(CCPM_ECUDA, cudaGetErrorString(e_)); \
    } while (0)
    const int64_t words = (m_dir + 31) / 32;
    // the scratch keeps whatever the previous call left: clear what must start at zero
    NA_CU(cudaMemsetAsync(acc, 0, sizeof(HubAcc) * (size_t)L.acc_cap, s));
    if (words > 0) NA_CU(cudaMemsetAsync(ebits, 0xFF, sizeof(uint32_t) * (size_t)words, s));
    int64_t scanned = 0;
    int cur = 0, li = 0;
    int32_t r = 0;
    if (dt.n_cls <= 4) {
        // rounds queued kNoAllocRounds at a time, each reading the list sizes of
        // the one before on the device
        RowArgs a{};
        a.n = n;
        a.m = m_dir;
        a.rp = row_ptr;
        a.col = col;
        a.col_vec = ((uintptr_t)col & 15) == 0;
        a.lab = labels;
        a.ebits = ebits;
        a.acc = acc;
        a.hub_deg = hub;
        a.short_max = kSmallDeg;
        a.lm = lm;
        const int wave = 4 * num_sms;
        RoundStats *prev = nullptr;
        for (int group = 0;; group++) {
            RoundStats *ring = rounds_dev + 1 + (group & 1) * kNoAllocRounds;
            NA_CU(cudaMemsetAsync(ring, 0, sizeof(RoundStats) * kNoAllocRounds, s));
            if (group == 0) NA_CU(cudaMemsetAsync(rounds_dev, 0, sizeof(RoundStats), s));
            for (int i = 0; i < kNoAllocRounds; i++) {
                a.st = ring + i;
                a.small_in = small[li];
                a.med_in = med[li];
                a.chunk_in = chunk[li];
                a.small_out = small[li ^ 1];
                a.med_out = med[li ^ 1];
                a.chunk_out = chunk[li ^ 1];
                if (!prev) {
                    a.om_out[0] = om[0];
                    a.om_out[1] = om[1];
                    a.first_med = med[li];
                    a.first_chunk = chunk[li];
                    a.first_sizes = rounds_dev;
                    a.sizes = rounds_dev;
                    const int gf = std::min(grid(n, 8), wave);
                    if (dt.n_cls == 0) {
                        k_first_round<0, kByLabel><<<gf, 256, 0, s>>>(a, dt);
                        k_rows<0, kFirst, kByLabel><<<wave, 256, 0, s>>>(a, dt);
                    } else {
                        k_first_round<4, kByLabel><<<gf, 256, 0, s>>>(a, dt);
                        k_rows<4, kFirst, kByLabel><<<wave, 256, 0, s>>>(a, dt);
                    }
                } else {
                    a.om = om[cur];
                    a.om_out[0] = om[cur ^ 1];
                    a.sizes = prev;
                    a.gate = prev;
                    if (dt.n_cls == 0) k_rows<0, kFull, kByWord><<<wave, 256, 0, s>>>(a, dt);
                    else k_rows<4, kFull, kByWord><<<wave, 256, 0, s>>>(a, dt);
                }
                NA_CU(cudaGetLastError());
                prev = ring + i;
                li ^= 1;
                cur ^= 1;
            }
            RoundStats h[kNoAllocRounds];
            NA_CU(cudaMemcpyAsync(h, ring, sizeof(h), cudaMemcpyDeviceToHost, s));
            NA_CU(cudaStreamSynchronize(s));
            bool done = false;
            for (int i = 0; i < kNoAllocRounds && !done; i++) {
                r++;
                scanned += (int64_t)h[i].scanned;
                done = !h[i].changed;
            }
            if (done) break;
            if (r > 4 * (m_dir + n) + 8) return fail(CCPM_ETIMEOUT, "LCC did not converge");
        }
        cur = 0;       // a fixpoint leaves the two buffers equal
    } else {
        NA_CU(cudaMemsetAsync(st, 0, sizeof(RoundStats), s));
        k_init<<<grid(n, 256), 256, 0, s>>>(n, row_ptr, labels, lm, nullptr, om[0], om[1], nullptr, nullptr, 0, small[0],
                                            med[0], chunk[0], acc, st, hub, kSmallDeg, 0u, nullptr, nullptr, 0);
        NA_CU(cudaGetLastError());
        if (m_dir & 31) k_set_word<<<1, 1, 0, s>>>(ebits + words - 1, (1u << (uint32_t)(m_dir & 31)) - 1u);
        NA_CU(read_stats());
        int64_t n_small = hs.n_small, n_med = hs.n_med, n_chunk = hs.n_chunk;
        for (;;) {
            NA_CU(cudaMemsetAsync(st, 0, sizeof(RoundStats), s));
            LccArgs a{};
            a.rp = row_ptr;
            a.col = col;
            a.om_cur = om[cur];
            a.om_next = om[cur ^ 1];
            a.ebits = ebits;
            a.small_in = small[li];
            a.med_in = med[li];
            a.chunk_in = chunk[li];
            a.n_small = n_small;
            a.n_med = n_med;
            a.n_chunk = n_chunk;
            a.small_out = small[li ^ 1];
            a.med_out = med[li ^ 1];
            a.chunk_out = chunk[li ^ 1];
            a.acc = acc;
            a.st = st;
            a.hub_deg = hub;
            a.med_chunk = 1;
            a.resident_warps = num_sms * 32;
            // at most one resident wave (four blocks an SM): the rows are dealt out evenly over the warps
            const int g = std::min(grid((n_chunk + n_med + n_small) * 32, 256), 4 * num_sms);
            k_lcc_round<kMaxCls, kFull><<<g, 256, 0, s>>>(a, dt);
            NA_CU(cudaGetLastError());
            NA_CU(read_stats());
            r++;
            scanned += (int64_t)hs.scanned;
            n_small = hs.n_small;
            n_med = hs.n_med;
            n_chunk = hs.n_chunk;
            li ^= 1;
            cur ^= 1;
            if (!hs.changed) break;
            if (r > 4 * (m_dir + n) + 8) return fail(CCPM_ETIMEOUT, "LCC did not converge");
        }
    }
    // both omega buffers agree at the fixpoint; the caller's buffer must hold it
    if (cur != 0) NA_CU(cudaMemcpyAsync(omega, om[cur], sizeof(uint32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
    if (m_dir > 0) {
        k_materialize<<<grid(n * 32, 256), 256, 0, s>>>(n, omega, row_ptr, col, ebits);
        NA_CU(cudaGetLastError());
    }
    NA_CU(cudaStreamSynchronize(s));
#undef NA_CU
    if (rounds) *rounds = r;
    if (edges_scanned) *edges_scanned = scanned;
    return CCPM_OK;
}

}  // namespace

// The caller's current device is the same after the call as before it.
extern "C" int ccpm_lcc_fixpoint_noalloc(int device, void *cuda_stream, int64_t n, int64_t m_dir,
                                         const int64_t *row_ptr, const int32_t *col, const uint8_t *labels,
                                         int n0, const uint8_t *tmpl_labels, int m0, const int32_t *tmpl_edges,
                                         uint32_t *omega, uint32_t *ebits, int32_t *rounds,
                                         int64_t *edges_scanned, char *errbuf, size_t errlen) {
    if (errbuf && errlen) errbuf[0] = '\0';
    int prev = -1;
    const bool have_prev = cudaGetDevice(&prev) == cudaSuccess;
    const int rc = lcc_fixpoint_noalloc_body(device, cuda_stream, n, m_dir, row_ptr, col, labels, n0, tmpl_labels,
                                             m0, tmpl_edges, omega, ebits, rounds, edges_scanned, errbuf, errlen);
    if (have_prev && prev != device) cudaSetDevice(prev);
    return rc;
}
