// ccpm_wide.cu -- local constraint checking (Alg. 3 and Alg. 4) for templates
// of up to 64 vertices, with omega in 64-bit words (the paper's LCC state
// estimate budgets eight bytes per vertex for 64 template vertices, Section
// 5.1), and with edge labels (Section 3: edges carry metadata too).
//
// The rules of Alg. 4 are read per edge label L: an entry (v,u) labelled L
// stays active iff some a in omega(v) has a template neighbour b in omega(u)
// joined to a by an edge labelled L (eta); q stays in omega(v) iff every
// template neighbour b of q, joined by label L, lies in omega(u) of a kept
// entry labelled L (the union omega' taken per edge label), and for each
// pair (vertex label, edge label) enough distinct kept neighbours reached by
// that label meet q's template neighbours of the pair (the multiplicity rule
// of Section 4.1).  With every edge label 0 these are the rules of the 32-bit
// pipeline.
//
// Schedule: rounds are snapshot rounds over two omega buffers, and an entry's
// bit is read and written only with its own row, so a row that dies is wiped
// where it dies and the last (quiescent) round leaves omega, the bitmap and the
// active totals as they are handed back.  The first round reads labels instead
// of omega and writes the bits that stay; it lists the rows by length for the
// later rounds, which read their counts on the device: four rounds are queued at
// a time, and those after the quiescent one return at once.  Rows up to kWShort
// entries go four to a warp, rows up to kWHub one to a warp, longer ones to
// blocks in chunks; the block that finishes a row's last chunk decides it.  Once
// few vertices change, their neighbours are marked and a round evaluates only
// those; the others count as what they read last.  No kernel waits on another
// block: every loop is bounded by the list or row it walks.
//
// Figures: 4M vertices, 124M entries, a sampled template of 48 vertices and 3
// edge labels; 112M, 40M, 17M, 6M and 6M entries read by the five rounds.  With
// one warp a row, every window of every row in each round, per-vertex list
// atomics and a hand-back pass over the bitmap they took 7.2, 4.9, 2.9, 0.7 and
// 0.5 ms, the hand-back 1.9 and allocations 1 ms.  Now 0.24 + 0.89, 0.89, 0.66,
// 0.37 and 0.07 ms, and 0.25 for the allocation.  What bounds them: instructions
// (45 % of the issue slots) and gather latency at 32 warps an SM.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "ccpm.h"
#include "ccpm_internal.h"

namespace ccpm {
namespace {

constexpr int kWT = 64;        // template vertices
constexpr int kWEL = 8;        // distinct edge labels one template may use
constexpr int kWCls = 64;      // label-multiplicity classes (need >= 2)
constexpr int kWEdges = 2016;  // 64 * 63 / 2
constexpr int kWShort = 32;    // rows up to this go eight lanes each
constexpr int kWHub = 1024;    // rows longer than this are walked by whole blocks
constexpr int kWChunk = 8192;  // entries a block takes of one: 1024 for each of its 8 warps
constexpr int kWTile = 128;    // listed vertices a warp looks through at a time
constexpr int kWQueue = 4;     // rounds queued per host round trip
constexpr int kWPush = 4;      // neighbours are marked once less than one active vertex in so many changes
constexpr unsigned FULL = 0xFFFFFFFFu;

// Template tables of one call (device copy, loaded into shared memory).
struct __align__(16) WideTab {
    int n0, n_el, n_cls, pad;
    uint8_t el_index[256];         // graph edge label -> edge-label index j, kWEL: used by no template edge
    uint64_t adj[kWEL][kWT];       // adj[j][q]: template neighbours of q joined by an edge of label index j
    uint64_t cls_mask[kWCls];      // template neighbours of cls_q with one vertex label, joined by label cls_j
    uint32_t cls_need[kWCls];      // their number (at least 2; a class of one is the coverage rule)
    uint64_t q_cls[kWT];           // the classes of q
    uint8_t cls_q[kWCls];
    uint8_t cls_j[kWCls];
};

struct WideRound {
    unsigned long long n_list;     // short rows listed for the next round
    unsigned long long scanned;    // active entries read (both ends live, bit set)
    unsigned long long alive;      // active vertices read
    unsigned long long moved;      // vertices whose omega changed
    unsigned int changed;          // anything did
    unsigned int pushed;           // the neighbours of those vertices are marked
};
struct WideState {
    unsigned long long n_mid, n_hub, n_part; // mid rows, chunks of longer rows, rows of several chunks
    // r[i + 1]: the i-th of the queued rounds (n_list: of the round after it);
    // r[0]: the round before them
    WideRound r[kWQueue + 1];
};

// A chunk of a long row; part: the row's place for combining its chunks, -1: it
// has only this one.
struct WideChunk {
    int32_t v, part, chunk, chunks;
};
struct WidePart {
    unsigned long long U[kWEL];
    uint32_t cnt[kWCls];
    uint32_t nN, chg, done, pad;
};

struct WideArgs {
    int64_t n;
    const int64_t *rp;
    const int32_t *col;
    const uint8_t *lab;
    const uint8_t *el;             // edge label per entry, or NULL (all 0)
    const uint64_t *lmask;         // 256: the template vertices of a label
    const uint64_t *om_in;
    uint64_t *om_out;
    uint32_t *ebits;
    uint32_t *deg;                 // active entries of an active vertex after its last evaluation
    const uint8_t *mark_in;        // vertices to evaluate in this round (value `mark`)
    uint8_t *mark_out;             // ... and in the next one (value `mark` + 1)
    uint8_t mark;
    const int32_t *list_in;        // active vertices with short rows
    int32_t *list_out;
    int32_t *mid;                  // initially active vertices with longer rows
    WideChunk *hub;
    WidePart *part;                // all 0 between rounds
    WideState *st;
    int slot;                      // of this round
    const WideTab *tab;
};

__device__ __forceinline__ uint64_t warp_or64(uint64_t x) {
    const uint32_t lo = __reduce_or_sync(FULL, (uint32_t)x), hi = __reduce_or_sync(FULL, (uint32_t)(x >> 32));
    return ((uint64_t)hi << 32) | lo;
}

// Over the eight lanes of a group.
__device__ __forceinline__ uint64_t group_or64(uint64_t x) {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) x |= __shfl_xor_sync(FULL, x, o);
    return x;
}

__device__ __forceinline__ void load_tab(WideTab &dst, const WideTab *src) {
    const uint32_t *s = reinterpret_cast<const uint32_t *>(src);
    uint32_t *d = reinterpret_cast<uint32_t *>(&dst);
    for (int i = threadIdx.x; i < (int)(sizeof(WideTab) / 4); i += blockDim.x) d[i] = s[i];
}

// Per-thread totals of a round, and the block's shared memory.
struct WideAcc {
    unsigned long long scanned = 0;
    uint32_t alive = 0, moved = 0;
    bool changed = false;
    bool push = false, marked = false;       // this round marks; the round before it did
};
struct WideShared {
    WideTab T;
    uint64_t lm[256];                        // first round: omega of a label
    uint64_t w[8][kWTile];                   // a warp's short rows: omega, vertex
    int32_t v[8][kWTile];
    uint64_t nb[8][4][kWEL + 1];             // per warp and row: template neighbours of omega(v), by edge label
    unsigned long long bU[kWEL];             // a long row's results
    uint32_t bcnt[kWCls];
    uint32_t bN, bchg;
    unsigned long long scanned, alive, moved;
    uint32_t changed, last;
};

// Rows of at most kWShort entries, eight lanes and four entries a lane each, so
// that four rows of a warp share its instructions and their loads are in flight
// together.  A row's bits are one 32-bit word in registers.  Coverage is decided
// first; only the classes of the vertices that pass it are counted.
template <bool FIRST, int NEL>
__device__ __forceinline__ void short_row(const WideArgs &a, WideShared &S, bool has, int32_t v, uint64_t wv,
                                          WideAcc &acc) {
    const WideTab &T = S.T;
    const int lane = threadIdx.x & 31, gl = lane & 7, gb = lane & 24;
    int64_t beg = 0;
    int len = 0;
    if (has) {
        beg = a.rp[v];
        len = (int)(a.rp[(int64_t)v + 1] - beg);
    }
    const int sh = (int)(beg & 31);
    uint32_t *const word = a.ebits + (beg >> 5);
    uint32_t rb = len >= 32 ? FULL : (1u << len) - 1u;
    if (!FIRST && len > 0) {
        const uint32_t lo = word[0], hi = sh + len > 32 ? word[1] : 0u;
        rb &= __funnelshift_r(lo, hi, sh);
    }
    int32_t u[4];
    uint8_t lb[4];
    uint64_t wu[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const bool act = (rb >> (8 * k + gl)) & 1u;
        u[k] = act ? a.col[beg + 8 * k + gl] : -1;
        lb[k] = act && a.el ? a.el[beg + 8 * k + gl] : (uint8_t)0;
    }
#pragma unroll
    for (int k = 0; k < 4; k++) wu[k] = u[k] >= 0 ? (FIRST ? S.lm[a.lab[u[k]]] : a.om_in[u[k]]) : 0ull;
    // template neighbours of omega(v); each lane takes eight template vertices
    uint64_t nb[NEL], U[NEL];
#pragma unroll
    for (int j = 0; j < NEL; j++) nb[j] = U[j] = 0;
    const uint32_t mine = (uint32_t)(wv >> (8 * gl)) & 0xFFu;
    for (uint32_t b = mine; b; b &= b - 1) {
        const int q = 8 * gl + __ffs(b) - 1;
#pragma unroll
        for (int j = 0; j < NEL; j++) nb[j] |= T.adj[j][q];
    }
    uint64_t *const snb = S.nb[threadIdx.x >> 5][lane >> 3];
#pragma unroll
    for (int j = 0; j < NEL; j++) {
        nb[j] = group_or64(nb[j]);
        if (gl == j) snb[j] = nb[j];
    }
    __syncwarp();
    uint32_t pm = 0;                         // entries that pass
    int jk[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int j = (int)T.el_index[lb[k]];
        const bool live = wu[k] != 0, pass = (wu[k] & snb[j]) != 0;
        if (live) acc.scanned++;
        if (live && !pass) acc.changed = true;           // eta eliminates an active entry
        jk[k] = pass ? j : -1;
#pragma unroll
        for (int i = 0; i < NEL; i++)
            U[i] |= wu[k] & (jk[k] == i ? ~0ull : 0ull);
        pm |= ((__ballot_sync(FULL, pass) >> gb) & 0xFFu) << (8 * k);
    }
    uint64_t keep = 0, open = 0;
    if (__any_sync(FULL, pm != 0)) {
#pragma unroll
        for (int j = 0; j < NEL; j++) U[j] = group_or64(U[j]);
        if (pm)
            for (uint32_t b = mine; b; b &= b - 1) {
                const int q = 8 * gl + __ffs(b) - 1;
                bool ok = true;
#pragma unroll
                for (int j = 0; j < NEL; j++) ok = ok && !(T.adj[j][q] & ~U[j]);
                if (ok) {
                    keep |= 1ull << q;
                    open |= T.q_cls[q];
                }
            }
        keep = group_or64(keep);
        if (T.n_cls) open = group_or64(open);
        while (__any_sync(FULL, open != 0)) {
            const int c = open ? __ffsll((long long)open) - 1 : 0;
            const uint64_t cm = T.cls_mask[c];
            const int cj = T.cls_j[c];
            uint32_t h = 0;
#pragma unroll
            for (int k = 0; k < 4; k++) h += jk[k] == cj && (wu[k] & cm) != 0 ? 1u : 0u;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) h += __shfl_xor_sync(FULL, h, o);
            if (open) {
                open &= open - 1;
                if (h < T.cls_need[c]) {
                    keep &= ~(1ull << T.cls_q[c]);
                    open &= ~T.q_cls[T.cls_q[c]];
                }
            }
        }
    }
    if (!has) return;                        // (no warp operation below)
    if (keep != wv) {
        acc.changed = true;
        if (gl == 0) acc.moved++;
        if (!FIRST && acc.push) {
            if (gl == 0 && keep) a.mark_out[v] = (uint8_t)(a.mark + 1);
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (jk[k] >= 0) a.mark_out[u[k]] = (uint8_t)(a.mark + 1);
        }
    }
    const uint32_t nbits = keep ? pm : 0u;   // a dead row's bits go at once
    const uint32_t d = FIRST ? nbits : rb & ~nbits;
    if (gl == 0) {
        acc.alive++;
        a.om_out[v] = keep;
        a.deg[v] = __popc(pm);
        const uint32_t lo = d << sh;
        if (lo) {
            if (FIRST) atomicOr(word, lo);
            else atomicAnd(word, ~lo);
        }
    } else if (gl == 1 && sh) {
        const uint32_t hi = d >> (32 - sh);
        if (hi) {
            if (FIRST) atomicOr(word + 1, hi);
            else atomicAnd(word + 1, ~hi);
        }
    }
}

__device__ __forceinline__ void list_chunks(const WideArgs &a, int32_t v) {
    const int64_t beg = a.rp[v], end = a.rp[(int64_t)v + 1];
    // chunks start at bitmap words
    const int chunks = (int)((end - (beg & ~31ll) + kWChunk - 1) / kWChunk);
    const int part = chunks > 1 ? (int)atomicAdd(&a.st->n_part, 1ull) : -1;
    const unsigned long long at = atomicAdd(&a.st->n_hub, (unsigned long long)chunks);
    for (int c = 0; c < chunks; c++) a.hub[at + c] = WideChunk{v, part, c, chunks};
}

// The listed (first round: all) vertices, 128 to a warp at a time: those that
// died get their zero in this buffer, the active ones with short rows are listed
// again and evaluated, and the first round lists the longer rows.
template <bool FIRST, int NEL>
__device__ __forceinline__ void short_part(const WideArgs &a, WideShared &S, int64_t n_in, WideAcc &acc) {
    constexpr int W = kWTile / 32;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    for (int64_t base = gw * kWTile; base < n_in; base += nw * kWTile) {
        int32_t v[W];
        uint64_t w[W];
#pragma unroll
        for (int k = 0; k < W; k++) {
            const int64_t i = base + 32 * k + lane;
            v[k] = i < n_in ? (FIRST ? (int32_t)i : a.list_in[i]) : -1;
        }
#pragma unroll
        for (int k = 0; k < W; k++) w[k] = v[k] >= 0 ? (FIRST ? S.lm[a.lab[v[k]]] : a.om_in[v[k]]) : 0ull;
        int len[W];                          // 0: short, 1: mid, 2: hub, -1: not active
#pragma unroll
        for (int k = 0; k < W; k++) {
            len[k] = w[k] ? 0 : -1;
            if (FIRST && w[k]) {
                const int64_t l = a.rp[(int64_t)v[k] + 1] - a.rp[v[k]];
                len[k] = l <= kWShort ? 0 : l <= kWHub ? 1 : 2;
            }
            if (v[k] >= 0 && !w[k]) a.om_out[v[k]] = 0;
            if (!FIRST && acc.marked && w[k] && a.mark_in[v[k]] != a.mark) {
                len[k] = 3;                  // nothing near it changed
                acc.alive++;
                acc.scanned += a.deg[v[k]];
                a.om_out[v[k]] = w[k];
            }
        }
        uint32_t cnt[3] = {0, 0, 0};
#pragma unroll
        for (int t = 0; t < (FIRST ? 3 : 1); t++) {
            uint32_t b[W], total = 0;
#pragma unroll
            for (int k = 0; k < W; k++) {
                b[k] = __ballot_sync(FULL, len[k] == t);
                total += __popc(b[k]);
            }
            cnt[t] = total;                  // (t = 0: rows to evaluate, listed with the skipped ones)
            if (!FIRST)
#pragma unroll
                for (int k = 0; k < W; k++) total += __popc(__ballot_sync(FULL, len[k] == 3));
            if (!total) continue;
            if (t == 2) {
#pragma unroll
                for (int k = 0; k < W; k++)
                    if (len[k] == t) list_chunks(a, v[k]);
                continue;
            }
            unsigned long long *const n_out = t == 0 ? &a.st->r[a.slot + 1].n_list : &a.st->n_mid;
            int32_t *const out = t == 0 ? a.list_out : a.mid;
            unsigned long long pos = 0;
            if (lane == 0) pos = atomicAdd(n_out, (unsigned long long)total);
            pos = __shfl_sync(FULL, pos, 0);
            uint32_t at = 0;
#pragma unroll
            for (int k = 0; k < W; k++) {
                if (len[k] == t) {
                    const uint32_t o = at + __popc(b[k] & lt);
                    out[pos + o] = v[k];
                    if (t == 0) {
                        S.v[wib][o] = v[k];
                        S.w[wib][o] = w[k];
                    }
                }
                at += __popc(b[k]);
            }
            if (!FIRST)
#pragma unroll
                for (int k = 0; k < W; k++) {
                    const uint32_t skipped = __ballot_sync(FULL, len[k] == 3);
                    if (len[k] == 3) out[pos + at + __popc(skipped & lt)] = v[k];
                    at += __popc(skipped);
                }
        }
        __syncwarp();
        for (uint32_t i0 = 0; i0 < cnt[0]; i0 += 4) {
            const uint32_t i = i0 + (lane >> 3);
            const bool has = i < cnt[0];
            short_row<FIRST, NEL>(a, S, has, has ? S.v[wib][i] : 0, has ? S.w[wib][i] : 0ull, acc);
        }
        __syncwarp();
    }
}

// Template vertices of omega(v) whose neighbours all lie in U; their classes.
template <int NEL>
__device__ __forceinline__ uint64_t covered(const WideTab &T, uint64_t wv, const uint64_t (&U)[NEL], uint64_t &cls) {
    const int lane = threadIdx.x & 31;
    bool ok[2];
    uint64_t c = 0;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int q = lane + 32 * h;
        ok[h] = (wv >> q) & 1ull;
#pragma unroll
        for (int j = 0; j < NEL; j++) ok[h] = ok[h] && !(T.adj[j][q] & ~U[j]);
        if (ok[h]) c |= T.q_cls[q];
    }
    cls = T.n_cls ? warp_or64(c) : 0ull;
    const uint64_t lo = __ballot_sync(FULL, ok[0]), hi = __ballot_sync(FULL, ok[1]);
    return lo | (hi << 32);
}

// A longer row, or a chunk of one: its arrays from the bitmap word of its first
// entry on (`off` entries into it, up to `span`).
struct WideRow {
    uint32_t *bits;
    const int32_t *col;
    const uint8_t *el;
    uint32_t off, span;
};
__device__ __forceinline__ WideRow row_of(const WideArgs &a, int32_t v) {
    const int64_t beg = a.rp[v], w = beg >> 5;
    return WideRow{a.ebits + w, a.col + (w << 5), a.el ? a.el + (w << 5) : nullptr, (uint32_t)(beg & 31),
                   (uint32_t)(a.rp[(int64_t)v + 1] - (w << 5))};
}
__device__ __forceinline__ WideRow chunk_of(const WideArgs &a, const WideChunk &h) {
    WideRow r = row_of(a, h.v);
    const uint32_t at = (uint32_t)h.chunk * kWChunk;
    r.bits += at >> 5;
    r.col += at;
    if (r.el) r.el += at;
    if (h.chunk) r.off = 0;
    r.span = min(r.span - at, (uint32_t)kWChunk);
    return r;
}
__device__ __forceinline__ uint32_t row_bits(const WideRow &r, uint32_t w) {
    uint32_t m = FULL;
    if (w == 0) m <<= r.off;
    if (r.span - 32 * w < 32) m &= (1u << (r.span - 32 * w)) - 1u;
    return m;
}

// Walks the set bits of a row (first round: all its bits), 32 bitmap words at a
// time, lane i holding word i.  An iteration takes four entries a lane, all loads
// in flight together; f(wu, j, pass) gets their neighbours' omegas (0 where there
// is no entry) and their edge-label indices, and fills in which of them pass; it
// returns whether to go on.  Either the lanes take four whole words
// (coalesced), or, where that is fewer iterations, each lane the next four bits
// of its own word: after the second round most words hold a bit or two (rounds 2
// to 4: 1.07, 0.98 and 0.65 ms with whole words only, 0.89, 0.66 and 0.37 so).  UPDATE:
// the bits become those that passed, with one atomic per changed word.
template <bool FIRST, bool UPDATE, class F>
__device__ __forceinline__ void walk(const WideArgs &a, const WideShared &S, const WideRow &r, uint32_t first_w,
                                     uint32_t w_step, F f) {
    const int lane = threadIdx.x & 31;
    bool go = true;
    for (uint32_t w0 = first_w; go && 32 * w0 < r.span; w0 += w_step) {
        uint32_t word = 0;
        if (32 * (w0 + lane) < r.span) {
            word = row_bits(r, w0 + lane);
            if (!FIRST) word &= r.bits[w0 + lane];
        }
        uint32_t groups = __ballot_sync(FULL, word != 0);
        groups |= groups >> 1;
        groups = (groups | (groups >> 2)) & 0x11111111u;
        if (!groups) continue;
        const bool own = !FIRST && __reduce_max_sync(FULL, (unsigned)__popc(word)) * 3 <= 8u * __popc(groups);
        uint32_t left = word, kept = 0;
        while (go && (own ? __any_sync(FULL, left != 0) : groups != 0)) {
            const int g = own ? 0 : __ffs(groups) - 1;
            groups &= groups - 1;
            bool bit[4];
            int32_t u[4];
            uint8_t lb[4];
            uint32_t at[4];                  // bit of `word` in own mode
#pragma unroll
            for (int k = 0; k < 4; k++) {
                uint32_t e;
                if (own) {
                    at[k] = left & (0u - left);
                    left ^= at[k];
                    bit[k] = at[k] != 0;
                    e = 32 * (w0 + lane) + (31 - __clz(at[k] | 1u));
                } else {
                    at[k] = 0;
                    bit[k] = (__shfl_sync(FULL, word, g + k) >> lane) & 1u;
                    e = 32 * (w0 + g + k) + lane;
                }
                u[k] = bit[k] ? r.col[e] : 0;
                lb[k] = bit[k] && r.el ? r.el[e] : (uint8_t)0;
            }
            uint64_t wu[4];
            int j[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                wu[k] = bit[k] ? (FIRST ? S.lm[a.lab[u[k]]] : a.om_in[u[k]]) : 0ull;
                j[k] = (int)S.T.el_index[lb[k]];
            }
            bool pass[4];
            go = f(wu, j, pass);
            if (UPDATE) {
                if (own) {
#pragma unroll
                    for (int k = 0; k < 4; k++) kept |= pass[k] ? at[k] : 0u;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const uint32_t p = __ballot_sync(FULL, pass[k]);
                        if (lane == g + k) kept = p;
                    }
                }
            }
        }
        if (UPDATE) {
            if (FIRST && kept) atomicOr(&r.bits[w0 + lane], kept);
            if (!FIRST && word != kept) atomicAnd(&r.bits[w0 + lane], ~(word & ~kept));
        }
    }
}

// A warp's share of a longer row.  A class is counted only until it is met,
// which on long rows is within the first groups, and the unions only until they
// hold all they can.  The warp that has the whole row to itself (WHOLE) counts
// classes once coverage is known, and only those of the vertices it leaves: on
// the entries in its registers if they are all, else on a second walk that ends
// when they are met.  Lane i holds the counts of classes i and i + 32.
template <int NEL>
struct RowScan {
    uint64_t U[NEL], open, keep;
    uint32_t nN, c0, c1;
    bool chg;
};

template <int NEL>
__device__ __forceinline__ void count_classes(const WideTab &T, const uint64_t (&wu)[4], const int (&jk)[4],
                                              RowScan<NEL> &R) {
    const int lane = threadIdx.x & 31;
    for (uint64_t o = R.open; o; o &= o - 1) {
        const int c = __ffsll((long long)o) - 1;
        const uint64_t cm = T.cls_mask[c];
        const int cj = T.cls_j[c];
        uint32_t h = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) h += __popc(__ballot_sync(FULL, jk[k] == cj && (wu[k] & cm) != 0));
        if (lane == (c & 31)) {
            if (c < 32) R.c0 += h;
            else R.c1 += h;
        }
    }
    if (R.open) {
        const uint64_t lo = __ballot_sync(FULL, R.c0 < T.cls_need[lane]);
        const uint64_t hi = __ballot_sync(FULL, R.c1 < T.cls_need[lane + 32]);
        R.open &= lo | (hi << 32);
    }
}

template <bool FIRST, int NEL, bool WHOLE>
__device__ __forceinline__ void scan_row(const WideArgs &a, WideShared &S, uint64_t wv, const WideRow &r,
                                         uint32_t first_w, uint32_t w_step, RowScan<NEL> &R, WideAcc &acc) {
    const WideTab &T = S.T;
    const int lane = threadIdx.x & 31;
    uint64_t *const nb = S.nb[threadIdx.x >> 5][0];
    {
        uint64_t c = 0, m[NEL];
#pragma unroll
        for (int j = 0; j < NEL; j++) m[j] = R.U[j] = 0;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int q = lane + 32 * h;
            if ((wv >> q) & 1ull) {
                c |= T.q_cls[q];
#pragma unroll
                for (int j = 0; j < NEL; j++) m[j] |= T.adj[j][q];
            }
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NEL; j++) {
            m[j] = warp_or64(m[j]);
            if (lane == j) nb[j] = m[j];
        }
        __syncwarp();
        R.open = !WHOLE && T.n_cls ? warp_or64(c) : 0ull;
    }
    R.keep = 0;
    R.nN = R.c0 = R.c1 = 0;
    R.chg = false;
    bool full = false;                       // the unions hold all they can
    uint32_t calls = 0;
    uint64_t wl[4];                          // the last iteration's entries that pass
    int jl[4];
    walk<FIRST, true>(a, S, r, first_w, w_step, [&](const uint64_t (&wu)[4], const int (&j)[4], bool (&pass)[4]) {
        uint64_t m[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            m[k] = wu[k] & nb[j[k]];
            const bool live = wu[k] != 0;
            pass[k] = m[k] != 0;
            if (live) acc.scanned++;
            if (live && !pass[k]) R.chg = true;          // eta eliminates an active entry
            if (pass[k]) R.nN++;
            wl[k] = wu[k];
            jl[k] = pass[k] ? j[k] : -1;
        }
        if (!full) {
#pragma unroll
            for (int k = 0; k < 4; k++)
#pragma unroll
                for (int i = 0; i < NEL; i++) R.U[i] |= m[k] & (jl[k] == i ? ~0ull : 0ull);
            if (calls % 4 == 1) {
                full = true;
#pragma unroll
                for (int i = 0; i < NEL; i++) {
                    R.U[i] = warp_or64(R.U[i]);
                    full = full && R.U[i] == nb[i];
                }
            }
        }
        calls++;
        if (!WHOLE) count_classes<NEL>(T, wl, jl, R);
        return true;
    });
#pragma unroll
    for (int j = 0; j < NEL; j++)
        if (!full) R.U[j] = warp_or64(R.U[j]);
    R.nN = __reduce_add_sync(FULL, R.nN);
    R.chg = __any_sync(FULL, R.chg);
    if (WHOLE && R.nN) {
        R.keep = covered<NEL>(T, wv, R.U, R.open);
        if (R.open) {
            if (calls == 1)
                count_classes<NEL>(T, wl, jl, R);
            else
                walk<FIRST, false>(a, S, r, first_w, w_step, [&](const uint64_t (&wu)[4], const int (&j)[4],
                                                                 bool (&)[4]) {
#pragma unroll
                    for (int k = 0; k < 4; k++) jl[k] = wu[k] & nb[j[k]] ? j[k] : -1;
                    count_classes<NEL>(T, wu, jl, R);
                    return R.open != 0;
                });
            for (uint64_t o = R.open; o; o &= o - 1) R.keep &= ~(1ull << T.cls_q[__ffsll((long long)o) - 1]);
        }
    }
}

// After a row's omega changed: marks the ends of its entries for the next round
// (its bits as they were read or are now: those dropped in this round were
// dropped at their other end, too) and, if it died, wipes its bits.
__device__ __forceinline__ void row_changed(const WideArgs &a, const WideRow &r, bool mark, bool dead, uint32_t first_w,
                                            uint32_t w_step) {
    const int lane = threadIdx.x & 31;
    const uint8_t next = (uint8_t)(a.mark + 1);
    for (uint32_t w = first_w; 32 * w < r.span; w += w_step) {
        uint32_t word[4];
#pragma unroll
        for (int k = 0; k < 4; k++) word[k] = 32 * (w + k) < r.span ? r.bits[w + k] & row_bits(r, w + k) : 0u;
        if (mark) {
            int32_t u[4];
#pragma unroll
            for (int k = 0; k < 4; k++) u[k] = (word[k] >> lane) & 1u ? r.col[32 * (w + k) + lane] : -1;
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (u[k] >= 0) a.mark_out[u[k]] = next;
        }
        if (dead && lane < 4 && 32 * (w + lane) < r.span) atomicAnd(&r.bits[w + lane], ~row_bits(r, w + lane));
    }
}

// The longer rows listed by the first round.
template <bool FIRST, int NEL>
__device__ __forceinline__ void long_part(const WideArgs &a, WideShared &S, WideAcc &acc) {
    const WideTab &T = S.T;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int64_t n_hub = (int64_t)a.st->n_hub, n_mid = (int64_t)a.st->n_mid;
    // chunks, one block each (block-uniform loop)
    for (int64_t i = blockIdx.x; i < n_hub; i += gridDim.x) {
        const WideChunk h = a.hub[i];
        const int32_t v = h.v;
        const uint64_t wv = FIRST ? S.lm[a.lab[v]] : a.om_in[v];
        const bool skip = !FIRST && acc.marked && a.mark_in[v] != a.mark;
        if (wv == 0 || skip) {               // dead, or nothing near it changed
            if (threadIdx.x == 0) a.om_out[v] = wv;
            if (threadIdx.x == 0 && wv && h.chunk == 0) {
                acc.alive++;
                acc.scanned += a.deg[v];
            }
            continue;
        }
        for (int c = threadIdx.x; c < kWCls; c += blockDim.x) S.bcnt[c] = 0;
        if (threadIdx.x < kWEL) S.bU[threadIdx.x] = 0ull;
        if (threadIdx.x == 0) { S.bN = 0; S.bchg = 0; }
        __syncthreads();
        RowScan<NEL> R;
        scan_row<FIRST, NEL, false>(a, S, wv, chunk_of(a, h), 32 * wib, 32 * nwb, R, acc);
        if (R.c0) atomicAdd(&S.bcnt[lane], R.c0);
        if (R.c1) atomicAdd(&S.bcnt[lane + 32], R.c1);
        if (lane == 0) {
#pragma unroll
            for (int j = 0; j < NEL; j++)
                if (R.U[j]) atomicOr(&S.bU[j], (unsigned long long)R.U[j]);
            if (R.nN) atomicAdd(&S.bN, R.nN);
            if (R.chg) atomicOr(&S.bchg, 1u);
        }
        __syncthreads();
        if (h.chunks > 1) {
            // add to the row's totals; the block that is last takes them over
            // (and leaves zeros for the next round)
            WidePart &P = a.part[h.part];
            if (threadIdx.x < kWCls) {
                const uint32_t c = S.bcnt[threadIdx.x];
                if (c) atomicAdd(&P.cnt[threadIdx.x], c);
            } else if (threadIdx.x < kWCls + NEL) {
                const unsigned long long U = S.bU[threadIdx.x - kWCls];
                if (U) atomicOr(&P.U[threadIdx.x - kWCls], U);
            } else if (threadIdx.x == kWCls + kWEL) {
                if (S.bN) atomicAdd(&P.nN, S.bN);
                if (S.bchg) atomicOr(&P.chg, 1u);
            }
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) S.last = atomicAdd(&P.done, 1u) + 1 == (uint32_t)h.chunks;
            __syncthreads();
            if (!S.last) continue;
            __threadfence();
            if (threadIdx.x < kWCls) S.bcnt[threadIdx.x] = atomicExch(&P.cnt[threadIdx.x], 0u);
            else if (threadIdx.x < kWCls + NEL) S.bU[threadIdx.x - kWCls] = atomicExch(&P.U[threadIdx.x - kWCls], 0ull);
            else if (threadIdx.x == kWCls + kWEL) {
                S.bN = atomicExch(&P.nN, 0u);
                S.bchg = atomicExch(&P.chg, 0u);
                P.done = 0;
            }
            __syncthreads();
        }
        uint64_t keep = 0;                   // every warp decides
        if (S.bN) {
            uint64_t U[NEL], cls;
#pragma unroll
            for (int j = 0; j < NEL; j++) U[j] = S.bU[j];
            keep = covered<NEL>(T, wv, U, cls);
            const uint64_t lo = __ballot_sync(FULL, S.bcnt[lane] < T.cls_need[lane]);
            const uint64_t hi = __ballot_sync(FULL, S.bcnt[lane + 32] < T.cls_need[lane + 32]);
            for (uint64_t o = cls & (lo | (hi << 32)); o; o &= o - 1)
                keep &= ~(1ull << T.cls_q[__ffsll((long long)o) - 1]);
        }
        if (threadIdx.x == 0) {
            acc.alive++;
            a.om_out[v] = keep;
            a.deg[v] = S.bN;
            if (keep != wv) acc.moved++;     // its entries: k_wide_hubs
            if (keep != wv || S.bchg) acc.changed = true;
        }
        __syncthreads();                     // bcnt / bU / bN are reused
    }
    // one warp each; a warp looks at four listed rows at a time
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = gw * 4; i0 < n_mid; i0 += nw * 4) {
        int32_t v4 = 0;
        uint64_t w4 = 0;
        if (lane < 4 && i0 + lane < n_mid) {
            v4 = a.mid[i0 + lane];
            w4 = FIRST ? S.lm[a.lab[v4]] : a.om_in[v4];
            const bool skip = !FIRST && acc.marked && w4 && a.mark_in[v4] != a.mark;
            if (!w4 || skip) a.om_out[v4] = w4;
            if (skip) {
                acc.alive++;
                acc.scanned += a.deg[v4];
                w4 = 0;
            }
        }
        for (uint32_t b = __ballot_sync(FULL, w4 != 0); b; b &= b - 1) {
            const int l = __ffs(b) - 1;
            const int32_t v = __shfl_sync(FULL, v4, l);
            const uint64_t wv = __shfl_sync(FULL, w4, l);
            const WideRow r = row_of(a, v);
            RowScan<NEL> R;
            scan_row<FIRST, NEL, true>(a, S, wv, r, 0, 32, R, acc);
            const bool mark = !FIRST && acc.push && R.keep != wv, dead = !R.keep && R.nN;
            if (mark || dead) {
                __syncwarp();                // after the scan's own bits
                row_changed(a, r, mark, dead, 0, 4);
            }
            if (lane == 0) {
                acc.alive++;
                a.om_out[v] = R.keep;
                a.deg[v] = R.nN;
                if (R.keep != wv) acc.moved++;
                if (mark && R.keep) a.mark_out[v] = (uint8_t)(a.mark + 1);
            }
            if (R.keep != wv || R.chg) acc.changed = true;
        }
    }
}

// One snapshot round; the first one is two launches, since its longer rows are
// listed by the pass over the short ones.
enum { kWFirstShort, kWFirstLong, kWLater };

// Four blocks an SM (64 registers): with 2, 3 and 5 the rounds above took 6.3,
// 3.7 and 4.1 ms in all instead of 3.2.
template <int PART, int NEL>
__global__ void __launch_bounds__(256, NEL <= 4 ? 4 : 2) k_wide_round(WideArgs a) {
    constexpr bool FIRST = PART != kWLater;
    __shared__ WideShared S;
    const WideRound before = a.st->r[a.slot];
    if (!FIRST && !before.changed) return;   // the round before was the last
    const int64_t n_in = PART == kWFirstLong ? 0 : FIRST ? a.n : (int64_t)before.n_list;
    const int nwb = blockDim.x >> 5;
    bool work = (int64_t)blockIdx.x * nwb * kWTile < n_in;
    if (PART != kWFirstShort)
        work = work || (int64_t)blockIdx.x < (int64_t)a.st->n_hub ||
               (int64_t)blockIdx.x * nwb * 4 < (int64_t)a.st->n_mid;
    if (!work) return;
    load_tab(S.T, a.tab);
    if (FIRST)
        for (int i = threadIdx.x; i < 256; i += blockDim.x) S.lm[i] = a.lmask[i];
    if (threadIdx.x == 0) { S.scanned = S.alive = S.moved = 0; S.changed = 0; }
    for (int i = threadIdx.x; i < 8 * 4; i += blockDim.x) S.nb[i >> 2][i & 3][kWEL] = 0;
    __syncthreads();
    WideAcc acc;
    if (!FIRST) {
        // without a change of an omega nothing needs a mark
        acc.marked = before.pushed || !before.moved;
        acc.push = acc.marked || before.moved * kWPush < before.alive;
    }
    if (PART != kWFirstShort) long_part<FIRST, NEL>(a, S, acc);
    if (PART != kWFirstLong) short_part<FIRST, NEL>(a, S, n_in, acc);
    // one atomic per block
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc.scanned += __shfl_xor_sync(FULL, acc.scanned, o);
    const uint32_t alive = __reduce_add_sync(FULL, acc.alive), moved = __reduce_add_sync(FULL, acc.moved);
    const bool changed = __any_sync(FULL, acc.changed);
    if (lane == 0) {
        if (acc.scanned) atomicAdd(&S.scanned, acc.scanned);
        if (alive) atomicAdd(&S.alive, (unsigned long long)alive);
        if (moved) atomicAdd(&S.moved, (unsigned long long)moved);
        if (changed) atomicOr(&S.changed, 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        WideRound *r = &a.st->r[a.slot + 1];
        if (S.scanned) atomicAdd(&r->scanned, S.scanned);
        if (S.alive) atomicAdd(&r->alive, S.alive);
        if (S.moved) atomicAdd(&r->moved, S.moved);
        if (acc.push) r->pushed = 1;
        if (S.changed) atomicOr(&r->changed, 1u);
    }
}

// The chunks of rows whose omega changed in this round, a block each: marks and
// wiping, spread like the round's own work (one block per such row left a tail).
template <bool FIRST>
__global__ void __launch_bounds__(256) k_wide_hubs(WideArgs a) {
    const WideRound &now = a.st->r[a.slot + 1];
    if (!now.moved) return;
    const int64_t n_hub = (int64_t)a.st->n_hub;
    for (int64_t i = blockIdx.x; i < n_hub; i += gridDim.x) {
        const WideChunk h = a.hub[i];
        const uint64_t wv = FIRST ? a.lmask[a.lab[h.v]] : a.om_in[h.v], keep = a.om_out[h.v];
        if (keep == wv) continue;
        const bool mark = !FIRST && now.pushed;
        if (mark && threadIdx.x == 0 && keep) a.mark_out[h.v] = (uint8_t)(a.mark + 1);
        if (mark || !keep)
            row_changed(a, chunk_of(a, h), mark, !keep, 4 * (threadIdx.x >> 5), 4 * (blockDim.x >> 5));
    }
}

template <int NEL>
void launch_round(const WideArgs &a, bool first, int grid, int hub_grid, cudaStream_t s) {
    if (first) {
        k_wide_round<kWFirstShort, NEL><<<grid, 256, 0, s>>>(a);
        k_wide_round<kWFirstLong, NEL><<<grid, 256, 0, s>>>(a);
        if (hub_grid) k_wide_hubs<true><<<hub_grid, 256, 0, s>>>(a);
    } else {
        k_wide_round<kWLater, NEL><<<grid, 256, 0, s>>>(a);
        if (hub_grid) k_wide_hubs<false><<<hub_grid, 256, 0, s>>>(a);
    }
}

int grid_of(ccpm_ctx *ctx, int64_t items, int per_block, int per_sm) {
    const int64_t need = std::max<int64_t>(1, (items + per_block - 1) / per_block);
    return (int)std::min<int64_t>(need, (int64_t)ctx_num_sms(ctx) * per_sm);
}

int popc64(uint64_t x) { return __builtin_popcountll(x); }

// Checks the template and fills the tables; returns CCPM_OK or CCPM_EINVAL
// with a message.
int build_tab(int n0, const uint8_t *labels, int m0, const int32_t *edges, const uint8_t *elab, WideTab &t,
              uint64_t *lmask, std::string &err) {
    if (n0 < 2 || n0 > kWT) { err = "wide template must have 2..64 vertices"; return CCPM_EINVAL; }
    if (m0 < 1 || m0 > kWEdges || !labels || !edges) {
        err = "wide template needs 1..2016 edges and non-NULL arrays";
        return CCPM_EINVAL;
    }
    std::memset(&t, 0, sizeof(t));
    std::memset(t.el_index, 0xFF, sizeof(t.el_index));
    t.n0 = n0;
    uint64_t any[kWT] = {};
    for (int i = 0; i < m0; i++) {
        const int a = edges[2 * i], b = edges[2 * i + 1];
        if (a < 0 || b < 0 || a >= n0 || b >= n0) { err = "template edge endpoint out of range"; return CCPM_EINVAL; }
        if (a == b) { err = "template self loop"; return CCPM_EINVAL; }
        if ((any[a] >> b) & 1ull) { err = "duplicate template edge"; return CCPM_EINVAL; }
        any[a] |= 1ull << b;
        any[b] |= 1ull << a;
        const uint8_t L = elab ? elab[i] : 0;
        if (t.el_index[L] == 0xFF) {
            if (t.n_el == kWEL) { err = "template uses more than 8 edge labels"; return CCPM_EINVAL; }
            t.el_index[L] = (uint8_t)t.n_el++;
        }
        const int j = t.el_index[L];
        t.adj[j][a] |= 1ull << b;
        t.adj[j][b] |= 1ull << a;
    }
    // connected
    uint64_t seen = 1, frontier = 1;
    while (frontier) {
        uint64_t next = 0;
        for (int q = 0; q < n0; q++)
            if ((frontier >> q) & 1ull) next |= any[q];
        frontier = next & ~seen;
        seen |= next;
    }
    const uint64_t all = n0 == 64 ? ~0ull : ((1ull << n0) - 1ull);
    if ((seen & all) != all) { err = "template is not connected"; return CCPM_EINVAL; }
    // multiplicity classes: q's neighbours of one vertex label joined by one edge label
    for (int q = 0; q < n0; q++)
        for (int j = 0; j < t.n_el; j++) {
            uint64_t done = 0;
            for (int b = 0; b < n0; b++) {
                if (!((t.adj[j][q] >> b) & 1ull) || ((done >> b) & 1ull)) continue;
                uint64_t grp = 0;
                for (int c = 0; c < n0; c++)
                    if (((t.adj[j][q] >> c) & 1ull) && labels[c] == labels[b]) grp |= 1ull << c;
                done |= grp;
                if (popc64(grp) < 2) continue;
                if (t.n_cls == kWCls) { err = "template has more than 64 label-multiplicity classes"; return CCPM_EINVAL; }
                t.cls_mask[t.n_cls] = grp;
                t.cls_need[t.n_cls] = (uint32_t)popc64(grp);
                t.cls_q[t.n_cls] = (uint8_t)q;
                t.cls_j[t.n_cls] = (uint8_t)j;
                t.q_cls[q] |= 1ull << t.n_cls;
                t.n_cls++;
            }
        }
    for (uint8_t &j : t.el_index)
        if (j == 0xFF) j = kWEL;
    std::memset(lmask, 0, sizeof(uint64_t) * 256);
    for (int q = 0; q < n0; q++) lmask[labels[q]] |= 1ull << q;
    return CCPM_OK;
}

// Device memory of one call, freed on every return path.  One allocation: ten
// of them and their releases took 1 ms on a graph of 4M vertices, this takes 0.25.
struct WideBufs {
    char *mem = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    ~WideBufs() {
        cudaFree(mem);
        for (auto e : ev) if (e) cudaEventDestroy(e);
    }
};

}  // namespace
}  // namespace ccpm

using namespace ccpm;

extern "C" int ccpm_lcc_wide(ccpm_ctx_t ctx, ccpm_graph_t g, int n0, const uint8_t *tmpl_labels, int m0,
                             const int32_t *tmpl_edges, const uint8_t *tmpl_edge_labels, uint64_t *omega,
                             uint32_t *ebits, int out_on_device, ccpm_wide_stats *stats) {
    if (!ctx || !g || !omega || !ebits) return CCPM_EINVAL;
    const GraphView G = graph_view(g);
    if (G.ctx != ctx) return ctx_set_err(ctx, CCPM_EINVAL, "lcc_wide: graph of another context");
    WideTab tab;
    uint64_t lmask[256];
    std::string err;
    int rc = build_tab(n0, tmpl_labels, m0, tmpl_edges, tmpl_edge_labels, tab, lmask, err);
    if (rc) return ctx_set_err(ctx, rc, err.c_str());
    if (cudaSetDevice(ctx_device(ctx)) != cudaSuccess) return ctx_set_err(ctx, CCPM_ECUDA, "lcc_wide: device");
    cudaStream_t s = (cudaStream_t)ctx_stream_ptr(ctx);
    const int64_t n = G.n, m = G.m, words = (m + 31) / 32;
    WideBufs B;
    auto fail = [&](cudaError_t e, const char *what) {
        return ctx_set_err(ctx, e == cudaErrorMemoryAllocation ? CCPM_ENOMEM : CCPM_ECUDA,
                           (std::string("lcc_wide: ") + what + ": " + cudaGetErrorString(e)).c_str());
    };
#define WCU(call, what)                          \
    do {                                         \
        cudaError_t e_ = (call);                 \
        if (e_ != cudaSuccess) return fail(e_, what); \
    } while (0)
    size_t size = 0;
    auto part = [&](size_t bytes) {
        const size_t at = size;
        size += (bytes + 255) / 256 * 256;
        return at;
    };
    // a row of more than k entries takes k + 1 of the m
    // (a chunked row may take one chunk more, being counted from a bitmap word)
    const int64_t max_mid = std::min(n, m / (kWShort + 1)), max_rows = std::min(n, m / (kWHub + 1)),
                  max_hub = m / kWChunk + 2 * max_rows, max_part = std::min(n, m / (kWChunk - 31));
    const size_t at_tab = part(sizeof(WideTab)), at_lm = part(sizeof(lmask)), at_st = part(sizeof(WideState)),
                 at_bits = part(sizeof(uint32_t) * (size_t)words), at_om0 = part(sizeof(uint64_t) * (size_t)n),
                 at_om1 = part(sizeof(uint64_t) * (size_t)n), at_mark0 = part((size_t)n), at_mark1 = part((size_t)n),
                 at_deg = part(sizeof(uint32_t) * (size_t)n), at_l0 = part(sizeof(int32_t) * (size_t)n),
                 at_l1 = part(sizeof(int32_t) * (size_t)n), at_mid = part(sizeof(int32_t) * (size_t)max_mid),
                 at_hub = part(sizeof(WideChunk) * (size_t)max_hub),
                 at_part = part(sizeof(WidePart) * (size_t)max_part);
    WCU(cudaMalloc(&B.mem, size), "alloc");
    uint64_t *const om[2] = {(uint64_t *)(B.mem + at_om0), (uint64_t *)(B.mem + at_om1)};
    int32_t *const list[2] = {(int32_t *)(B.mem + at_l0), (int32_t *)(B.mem + at_l1)};
    uint32_t *const bits = (uint32_t *)(B.mem + at_bits);
    WideState *const st = (WideState *)(B.mem + at_st);
    WideState sh;
    WCU(cudaEventCreate(&B.ev[0]), "event");
    WCU(cudaEventCreate(&B.ev[1]), "event");
    WCU(cudaMemcpyAsync(B.mem + at_tab, &tab, sizeof(WideTab), cudaMemcpyHostToDevice, s), "copy");
    WCU(cudaMemcpyAsync(B.mem + at_lm, lmask, sizeof(lmask), cudaMemcpyHostToDevice, s), "copy");
    WCU(cudaEventRecord(B.ev[0], s), "event");
    // counters, bits and marks 0; the first round writes om[0] in full, later ones
    // the listed vertices of the other buffer
    WCU(cudaMemsetAsync(B.mem + at_st, 0, at_om0 - at_st, s), "memset");
    WCU(cudaMemsetAsync(B.mem + at_om1, 0, at_deg - at_om1, s), "memset");
    WideArgs a;
    a.n = n;
    a.rp = G.rp;
    a.col = G.col;
    a.lab = G.lab;
    a.el = G.el;
    a.lmask = (const uint64_t *)(B.mem + at_lm);
    a.ebits = bits;
    a.deg = (uint32_t *)(B.mem + at_deg);
    a.mid = (int32_t *)(B.mem + at_mid);
    a.hub = (WideChunk *)(B.mem + at_hub);
    a.part = (WidePart *)(B.mem + at_part);
    if (max_part) WCU(cudaMemsetAsync(a.part, 0, sizeof(WidePart) * (size_t)max_part, s), "memset");
    a.st = st;
    a.tab = (const WideTab *)(B.mem + at_tab);
    const int grid = std::max(std::max(grid_of(ctx, n, 8 * kWTile, 8), grid_of(ctx, max_mid, 32, 8)),
                              grid_of(ctx, max_hub, 1, 8));
    const int hub_grid = max_hub ? grid_of(ctx, max_hub, 1, 8) : 0;
    uint8_t *const mark[2] = {(uint8_t *)(B.mem + at_mark0), (uint8_t *)(B.mem + at_mark1)};
    int64_t rounds = 0, scanned = 0, alive = 0, active_v = 0, active_e = 0;
    for (bool more = true; more;) {
        if (rounds) {
            WCU(cudaMemcpyAsync(&st->r[0], &st->r[kWQueue], sizeof(WideRound), cudaMemcpyDeviceToDevice, s), "copy");
            WCU(cudaMemsetAsync(&st->r[1], 0, sizeof(WideRound) * kWQueue, s), "memset");
        }
        for (int i = 0; i < kWQueue; i++) {
            const int64_t t = rounds + i;
            a.slot = i;
            a.mark = (uint8_t)t;             // of one of the last 256 rounds: an older one only costs time
            a.mark_in = mark[(t + 1) & 1];
            a.mark_out = mark[t & 1];
            a.om_in = om[(t + 1) & 1];
            a.om_out = om[t & 1];
            a.list_in = list[(t + 1) & 1];
            a.list_out = list[t & 1];
            if (tab.n_el <= 1) launch_round<1>(a, t == 0, grid, hub_grid, s);
            else if (tab.n_el == 2) launch_round<2>(a, t == 0, grid, hub_grid, s);
            else if (tab.n_el == 3) launch_round<3>(a, t == 0, grid, hub_grid, s);
            else launch_round<8>(a, t == 0, grid, hub_grid, s);
            WCU(cudaGetLastError(), "launch");
        }
        WCU(cudaMemcpyAsync(&sh, st, sizeof(sh), cudaMemcpyDeviceToHost, s), "copy");
        WCU(cudaStreamSynchronize(s), "sync");
        for (int i = 0; i < kWQueue && more; i++) {
            rounds++;
            const WideRound &r = sh.r[i + 1];
            scanned += (int64_t)r.scanned;
            alive += (int64_t)r.alive;
            more = r.changed != 0;
            // a round without a change read the active vertices and entries
            active_v = (int64_t)r.alive;
            active_e = (int64_t)r.scanned;
        }
    }
    WCU(cudaEventRecord(B.ev[1], s), "event");
    const cudaMemcpyKind kind = out_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    if (n > 0)
        WCU(cudaMemcpyAsync(omega, om[(rounds - 1) & 1], sizeof(uint64_t) * (size_t)n, kind, s), "copy");
    if (words > 0) WCU(cudaMemcpyAsync(ebits, bits, sizeof(uint32_t) * (size_t)words, kind, s), "copy");
    WCU(cudaStreamSynchronize(s), "sync");
#undef WCU
    if (stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, B.ev[0], B.ev[1]);
        stats->rounds = rounds;
        stats->edges_scanned = scanned;
        stats->vertices_scanned = alive;
        stats->active_v = active_v;
        stats->active_e_dir = active_e;
        stats->ms = ms;
    }
    return CCPM_OK;
}
