// Variant (iii)(a) in arrival order: the main path of a step.
//
// Edges of the hit graph are symmetric (8-adjacent or same pixel, |dToA| <=
// dt), so joining hits needs no time order inside a tile, only that each hit
// meets every hit it can be joined to.  A stream is nearly time ordered
// (Section 3.1), so those lie a short way around it.  No sort, no sorted
// copies and no gather are needed; a record is read from DRAM once.
//
//   k_arrival_tile   one CTA per time tile: tile j owns the hits of its ToA
//                    interval [cut j, cut j+1), picked from its TILE positions
//                    and a margin on both sides, and sees the hits of the dt
//                    before it.  Links in shared memory, pairs that join an
//                    earlier tile's hit go to a list, and every tile cluster's
//                    features are reduced.
//   k_arrival_cross  joins tile clusters over the listed pairs, closes the
//                    segments (watermark), and proves that every hit found its
//                    tile and every tile the hits before it; if not, the step
//                    takes the time-sorted path (link.cu), at once or, if tiles
//                    only held too many hits, after both kernels have run again
//                    for those, in parts.
//   k_arrival_roots  adds each tile cluster's features to its cluster's.
//   k_arrival_labels labels, closed flags and label flags per hit.
//   k_arrival_emit   records in label order; streaming: finalised hits, the
//                    carry of open hits and the stream state.
//
// Small steps (at most SMALL_TILES tiles) need no sorted path behind them: tiles
// own hits by position and look back over earlier positions, and a step that
// some tile is not done with (no order, too many hits within dt or on one pixel)
// is sorted and joined hit by hit (any_order).  All of it is one launch
// (k_arrival_step), a cluster of one CTA per tile.  As seven launches a call with
// 1,000 hits took 53 us (41 of them on the host) and one with 65,536 hits 96; now
// 26 and 58 (64 with 512 threads per CTA, which left an SM's issue slots idle).
//
// Owning by time keeps events whole: arrival disorder spreads an event's hits
// over a thousand positions, and tiles of positions would cut a quarter of
// the events into fragments (256x256 stream, 64 Mi hits: 522 tile clusters and
// 320 pairs across per tile by position, against 3.45 M clusters in all, 210
// per tile).
//
// Tile clusters are numbered c = tile * TILE + (index among the tile's
// clusters), so that everything kept per cluster (32-byte RootSlot, first and
// last ToA, union-find parent) is dense and a hit's cluster is one 32-bit c.
#include <cooperative_groups.h>

#include <cstddef>

#include "tpc_internal.cuh"

namespace tpc {

constexpr int AT = 512;                          // threads of k_arrival_tile (64 registers, two CTAs per SM)
constexpr int ST = 1024;                         // ... and where a CTA has an SM to itself
constexpr int AW = 32;                           // warps, at most
constexpr uint32_t A_MARGIN = 1024, A_WIDE = 2048;   // positions around the tile read at once; for tiles taken in parts
constexpr int A_GROUP = 2;                       // records per thread looked at while the next ones are in flight
constexpr int A_GROUPS = (TILE + 2 * A_WIDE) / (512 * A_GROUP);   // ... of 512 threads, at most
constexpr uint32_t A_STEP = TILE / ACHUNKS;      // positions per further round
constexpr uint32_t A_ENT = 5632;                 // hits staged: a tile's own and the earlier ones
constexpr uint32_t A_WORDS = 2304;               // 256 rows of nine 30-pixel words
constexpr uint32_t A_XTRA = 2048;                // unions beyond each hit's first
constexpr uint32_t A_LATER = 2048;               // hits beside cells of several hits
constexpr uint32_t A_FAR = 1920;                 // hits found beyond the margins (all that two CTAs per SM leave room for)
// A small step's tile is given up (S.flag) once a thread has walked over this
// many hits of crowded cells, or tried this often to hang a hit behind a cell's
// first: with hundreds of hits on a pixel both take the square of their number.
// (Not in k_arrival_tile: the counters cost it 1 percent.)
constexpr uint32_t A_WALK = 1024, A_TRIES = 256;
template <int NT>
constexpr bool GIVES_UP = NT == ST;
constexpr int A_JUMPS = 1;                       // path-shortening passes over the tile's forest
constexpr int A_ROUNDS = 4;                      // further rounds on each side
constexpr int A_BACK_ROUNDS = 16;                // rounds back of a small step's tiles
constexpr uint32_t A_NONE = 0x7FFFu;             // no hit
constexpr uint32_t A_MULTI = 0x8000u;            // head flag: the cell holds several hits
static_assert(A_WORDS <= 4096, "word indices take 12 bits");

// A cell is a pixel column x of a row (y mod R).  Occupied cells are found by
// a bitmap (30 pixels per word, the outer two bits repeating the neighbour
// words' border pixels, so that the three cells x-1..x+1 of a row are always
// in one word), and numbered by rank: word.y holds the occupied cells before
// the word, so a cell's slot is word.y + the set bits below it and the cells
// of a row's neighbourhood have consecutive slots.  head[slot] is a hit of
// the cell; further hits (a pixel hit more than once, or rows that share a
// cell on sensors taller than R) hang on next[].  113 KB: two CTAs per SM.
struct ArrivalShared {
    uint2 word[A_WORDS];         // bits; cells before the word (minus the repeated low bit)
    uint16_t head[A_ENT];
    uint16_t next[A_ENT];
    uint2 kc[A_ENT];             // key (ToA - base) and code
    uint16_t par[A_ENT];         // forest over the hits
    uint32_t xtra[A_XTRA];       // unions beyond each hit's first (k << 16 | j)
    uint16_t later[A_LATER];     // hits beside cells of several hits
    uint16_t far[A_FAR];         // hits beyond the margins: position - window start
    uint32_t red[4][AW];
    uint16_t first[AW][A_GROUPS];    // first entry of each warp's records of a group
    uint32_t cnt[2][AW], turn[2][AW];
    unsigned long long m64[2][AW];
    uint32_t cut[2];
    uint32_t nent, nown, ntail, nxtra, ncross, nlater, nroots, tsum, flag;
    uint32_t kept_tail;              // ntail of the parts that are done
    uint32_t from, to, numbered;     // the part of the tile's interval at hand; clusters of the parts before
    // After the links, in the place of what is no longer needed:
    __device__ uint32_t *where() { return reinterpret_cast<uint32_t *>(head); }   // [A_ENT] position << 16 | ToT per entry
    __device__ uint2 *tops() { return reinterpret_cast<uint2 *>(later); }         // [A_TOPS] roots of the tile's clusters
    __device__ uint32_t *sums() { return reinterpret_cast<uint32_t *>(word); }    // [2 * A_WORDS] feature sums
};
constexpr uint32_t A_TOPS = A_ENT / 32;   // words of a bitmap over the entries
static_assert(A_LATER * 2 >= A_TOPS * sizeof(uint2) && A_ENT % 32 == 0, "the bitmap fits the list");
static_assert(offsetof(ArrivalShared, next) == offsetof(ArrivalShared, head) + A_ENT * 2 && offsetof(ArrivalShared, head) % 4 == 0 &&
                  offsetof(ArrivalShared, later) % 8 == 0, "words over the heads and the lists");

// Code of a hit: word << 5 | bit of its cell, (y / R) << 17, and whether it is
// the tile's own (otherwise an earlier tile's).
constexpr uint32_t C_OWN = 1u << 31, C_CELL = C_OWN - 1u;

// Small steps stage every entry's position too, and have room for more unions.
constexpr uint32_t A_SMALL_XTRA = 8192;
struct SmallShared {
    ArrivalShared s;
    uint16_t pos[A_ENT];
    uint32_t xtra[A_SMALL_XTRA];
};
template <int NT>
constexpr uint32_t XTRA = NT == ST ? A_SMALL_XTRA : A_XTRA;
template <int NT>
__device__ __forceinline__ uint32_t *xtra_list(ArrivalShared &S) {
    if constexpr (NT == ST) return reinterpret_cast<SmallShared &>(S).xtra;   // (its first member)
    else return S.xtra;
}
constexpr int A_SMEM = (int)sizeof(ArrivalShared), A_SMALL_SMEM = (int)sizeof(SmallShared);
static_assert((unsigned long long)A_ENT * 0xFFFFu < (1ull << 32), "a tile's sum ToT fits 32 bits");

// Time window of 32-bit keys: base = 2^28 ticks before the segment's first
// hit.  A hit outside it (or a dt of 2^27 ticks and more) is "wide": a small
// step takes keys relative to its smallest ToA instead, others the
// time-sorted path.
constexpr uint64_t A_GUARD = ARRIVAL_DT;

__device__ __forceinline__ uint32_t absdiff(uint32_t a, uint32_t b) { return a > b ? a - b : b - a; }

__device__ __forceinline__ uint32_t lanes_below() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The cell grid of a W x H sensor: R rows (a power of two) of nw words.  A
// row's last word never uses its 30th pixel, so that no word repeats a pixel of
// another row.
struct Cells {
    uint32_t nw, rmask, rshift, nwords;   // words per row, R - 1, log2 R, words
    bool alias;                           // rows share cells
    __device__ Cells(uint32_t W, uint32_t H) {
        nw = W / 30u + 1u;                                 // <= 2185
        rshift = 31u - __clz((int)(A_WORDS / nw));         // at least one row
        while (rshift && (1u << (rshift - 1u)) >= H) --rshift;
        rmask = (1u << rshift) - 1u;
        nwords = nw << rshift;
        alias = H > rmask + 1u;
    }
    // y / R < 64: a row holds W * R > 30 * A_WORDS / 4 pixels when rows share cells, of at most 2^20
    __device__ __forceinline__ uint32_t code(uint32_t pix) const {
        const uint32_t x = pix & 0xFFFFu, y = pix >> 16, wi = x / 30u;
        uint32_t c = ((y & rmask) * nw + wi) * 32u + (x - wi * 30u) + 1u;
        if (alias) c |= y >> rshift << 17;
        return c;
    }
    __device__ __forceinline__ void set(ArrivalShared &S, uint32_t code) const {
        atomicOr(&S.word[(code >> 5) & 0xFFFu].x, 1u << (code & 31u));
    }
    __device__ __forceinline__ void pixel(uint32_t code, uint32_t magic, uint32_t &x, uint32_t &y) const {
        const uint32_t word = (code >> 5) & 0xFFFu, row = nw == 1u ? word : __umulhi(word, magic);
        x = (word - row * nw) * 30u + (code & 31u) - 1u;
        y = ((code & C_CELL) >> 17 << rshift) + row;
    }
    // word / nw = umulhi(word, magic) for words < 2^12, nw > 1 (nw = 1 apart: the factor would be 2^32)
    __device__ __forceinline__ uint32_t magic() const { return 0xFFFFFFFFu / nw + 1u; }
    template <int NT>
    __device__ __forceinline__ void clear(ArrivalShared &S) const {
        for (uint32_t i = threadIdx.x; i < (nwords + 1) / 2; i += NT)
            reinterpret_cast<uint4 *>(S.word)[i] = make_uint4(0, 0, 0, 0);
    }
};

// root of x with path halving (parents only move towards the root)
__device__ __forceinline__ uint32_t arrival_root(volatile uint16_t *par, uint32_t x) {
    while (true) {
        const uint32_t p = par[x];
        const uint32_t gp = par[p];
        if (p == gp) return p;
        par[x] = (uint16_t)gp;
        x = gp;
    }
}

// par[a]: a -> b if a is still a root (16-bit compare and swap)
__device__ __forceinline__ bool arrival_hook(uint16_t *par, uint32_t a, uint32_t b) {
    uint32_t *word = reinterpret_cast<uint32_t *>(par) + (a >> 1);
    const uint32_t shift = (a & 1u) * 16u;
    uint32_t old = *reinterpret_cast<volatile uint32_t *>(word);
    while (((old >> shift) & 0xFFFFu) == a) {
        const uint32_t seen = atomicCAS(word, old, (old & ~(0xFFFFu << shift)) | b << shift);
        if (seen == old) return true;
        old = seen;
    }
    return false;
}

// Links of the staged entries 0..n_e: cells numbered, heads and lists built,
// then each pair of adjacent hits met once, by the hit that is later in raster
// order (row above, left), on one pixel by the earlier hit.
// near(a, b): two keys within dt; join(e, j, linked): takes a pair; linked: e
// has been joined before.  ALIAS: rows share cells.
template <int NT, bool ALIAS, class Near, class Join>
__device__ __forceinline__ void arrival_pairs(ArrivalShared &S, const Cells &C, uint32_t n_e, Near near, Join join) {
    const int tid = threadIdx.x;
    // Heads of the cells left, above left, above and above right (A_NONE: none)
    // and of the own cell; up: y / R of the row above.
    auto around = [&](uint32_t code, uint32_t (&hd)[4], uint32_t &up) -> uint32_t {
        const uint32_t word = (code >> 5) & 0xFFFu, bit = code & 31u;
        const uint2 v0 = S.word[word];
        const uint32_t s0 = v0.y + __popc(v0.x & ~(0xFFFFFFFFu << bit));
        const uint32_t self = S.head[s0];
        hd[0] = hd[1] = hd[2] = hd[3] = A_NONE;
        if ((v0.x >> (bit - 1u)) & 1u) hd[0] = S.head[s0 - 1];
        const bool wrap = word < C.nw;   // the grid's first row: its last one lies above it
        up = (code & C_CELL) >> 17;
        const bool top = wrap && up == 0u;   // the sensor's first row
        up -= wrap ? 1u : 0u;
        const uint2 v1 = S.word[wrap ? word + C.nwords - C.nw : word - C.nw];
        const uint32_t m = top ? 0u : v1.x >> (bit - 1u);
        uint32_t s1 = v1.y + __popc(v1.x & ~(0xFFFFFFFFu << (bit - 1u)));
        if (m & 1u) hd[1] = S.head[s1];
        s1 += m & 1u;
        if (m & 2u) hd[2] = S.head[s1];
        s1 += (m >> 1) & 1u;
        if (m & 4u) hd[3] = S.head[s1];
        return self;
    };
    // Cells of several hits: on a neighbour pixel the latest hit at or before
    // this one and the earliest after it (the others within dt are joined to
    // those along their pixel), on the own pixel the next one.
    auto give_up = [](uint32_t count, uint32_t most) { return GIVES_UP<NT> && count > most; };
    uint32_t walked = 0;
    auto crowded = [&](uint32_t e) {
        const uint2 me = S.kc[e];
        const uint32_t code = me.y & C_CELL, key = me.x;
        bool linked = S.par[e] != e;
        uint32_t hd[4], up;
        const uint32_t self = around(code, hd, up);
        uint32_t multi = self & A_MULTI ? 16u : 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) multi |= hd[i] & A_MULTI ? 1u << i : 0u;
        while (multi) {
            const int i = __ffs(multi) - 1;
            multi &= multi - 1u;
            const uint32_t row = i == 0 || i == 4 ? code >> 17 : up;
            uint32_t j = (i == 4 ? self : i == 0 ? hd[0] : i == 1 ? hd[1] : i == 2 ? hd[2] : hd[3]) & A_NONE;
            uint32_t jlo = A_NONE, jhi = A_NONE, klo = 0, khi = 0xFFFFFFFFu;
            do {
                const uint2 o = S.kc[j];
                if (j != e && (!ALIAS || (o.y & C_CELL) >> 17 == row)) {
                    if (o.x < key || (o.x == key && (i != 4 || j < e))) {
                        if (o.x >= klo) { klo = o.x; jlo = j; }
                    } else if (o.x < khi || (o.x == khi && j < jhi)) {
                        khi = o.x;
                        jhi = j;
                    }
                }
                j = S.next[j];
            } while (j != A_NONE && !give_up(++walked, A_WALK));
            if (i != 4 && jlo != A_NONE && near(key, klo)) join(e, jlo, linked);
            if (jhi != A_NONE && near(khi, key)) join(e, jhi, linked);
        }
    };
#pragma unroll 1
    for (uint32_t e = tid; e < n_e; e += NT) {
        const uint2 me = S.kc[e];
        const uint32_t code = me.y & C_CELL, key = me.x;
        uint32_t hd[4], up;
        const uint32_t flags = around(code, hd, up);
        uint32_t kk[4] = {0, 0, 0, 0};
        bool ok[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (ALIAS) {
                uint2 o = make_uint2(0, 0);
                if (hd[i] < A_NONE) o = S.kc[hd[i]];   // a cell with one hit
                kk[i] = o.x;
                ok[i] = hd[i] < A_NONE && near(key, o.x) && (o.y & C_CELL) >> 17 == (i ? up : code >> 17);
            } else {
                if (hd[i] < A_NONE) kk[i] = S.kc[hd[i]].x;
                ok[i] = hd[i] < A_NONE && near(key, kk[i]);
            }
        }
        // A pair whose two hits are both within dt of a third neighbour's is
        // left out: the third one's pairs imply it.
        const bool by2 = ok[2];
        ok[1] = ok[1] && !(by2 && near(kk[2], kk[1])) && !(!by2 && ok[0] && near(kk[0], kk[1]));
        ok[0] = ok[0] && !(by2 && near(kk[2], kk[0]));
        ok[3] = ok[3] && !(by2 && near(kk[2], kk[3]));
        // the first of them, for all lanes at once; a second one is rare
        const uint32_t j = by2 ? hd[2] : ok[0] ? hd[0] : ok[1] ? hd[1] : hd[3];
        bool linked = by2 || ok[0] || ok[1] || ok[3];
        if (linked) {
            bool none = false;
            join(e, j, none);
        }
        uint32_t more = (ok[0] && by2 ? 1u : 0u) | (ok[1] && (by2 || ok[0]) ? 2u : 0u) |
                        (ok[3] && (by2 || ok[0] || ok[1]) ? 8u : 0u);
        while (more) {
            const uint32_t low = more & (0u - more);
            more ^= low;
            join(e, low == 1u ? hd[0] : low == 2u ? hd[1] : hd[3], linked);
        }
        // a tenth of the hits lie beside crowded cells: they are taken up
        // together afterwards, not by one lane of every warp
        if ((flags | hd[0] | hd[1] | hd[2] | hd[3]) & A_MULTI) {
            const uint32_t k = atomicAdd(&S.nlater, 1u);
            if (k < A_LATER) S.later[k] = (uint16_t)e;
        }
    }
    __syncthreads();
    const uint32_t listed = S.nlater;
    if (listed <= A_LATER)
        for (uint32_t i = tid; i < listed && !give_up(walked, A_WALK); i += NT) crowded(S.later[i]);
    else   // (more than the list holds: all of them, those without such cells have nothing to do)
        for (uint32_t e = tid; e < n_e && !give_up(walked, A_WALK); e += NT) crowded(e);
    if (give_up(walked, A_WALK)) S.flag = 1u;
}

template <int NT, class Near, class Join>
__device__ __forceinline__ void arrival_links(ArrivalShared &S, const Cells &C, uint32_t n_e, Near near, Join join) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();                // bits and entries are in place
    {   // repeat the border pixels in the neighbour words, and count the cells before each word
        constexpr uint32_t PER = (A_WORDS + NT - 1) / NT;
        const uint32_t i0 = tid * PER;
        uint32_t bits[PER], sum = 0;
        const uint32_t before = i0 && i0 < C.nwords ? S.word[i0 - 1].x : 0u;
#pragma unroll
        for (uint32_t i = 0; i < PER; ++i) bits[i] = i0 + i < C.nwords ? S.word[i0 + i].x : 0u;
        const uint32_t after = i0 + PER < C.nwords ? S.word[i0 + PER].x : 0u;
#pragma unroll
        for (uint32_t i = 0; i < PER; ++i) sum += __popc(bits[i]);
        uint32_t x = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) S.cnt[0][warp] = x;
        if (tid == 0) S.nlater = 0;
        __syncthreads();
        uint32_t run = x - sum + __reduce_add_sync(0xffffffffu, lane < warp ? S.cnt[0][min(lane, (NT / 32) - 1)] : 0u);
#pragma unroll
        for (uint32_t i = 0; i < PER; ++i) {
            const uint32_t l = i ? bits[i - 1] : before, r = i + 1 < PER ? bits[i + 1] : after;
            const uint32_t low = (l >> 30) & 1u;
            if (i0 + i < C.nwords) S.word[i0 + i] = make_uint2(bits[i] | low | (r & 2u) << 30, run - low);
            run += __popc(bits[i]);
        }
    }
    __syncthreads();
    constexpr int A_PER = (A_ENT + NT - 1) / NT;
    uint32_t slots[A_PER];
#pragma unroll
    for (int q = 0; q < A_PER; ++q) {   // any hit of a cell becomes its head
        const uint32_t e = q * NT + tid;
        slots[q] = 0;
        if (e < n_e) {
            const uint32_t code = S.kc[e].y;
            const uint2 v = S.word[(code >> 5) & 0xFFFu];
            slots[q] = v.y + __popc(v.x & ~(0xFFFFFFFFu << (code & 31u)));
            S.head[slots[q]] = (uint16_t)e;
            S.next[e] = (uint16_t)A_NONE;
            S.par[e] = (uint16_t)e;
        }
    }
    __syncthreads();
    auto give_up = [](uint32_t count, uint32_t most) { return GIVES_UP<NT> && count > most; };
    uint32_t tries = 0;
#pragma unroll
    for (int q = 0; q < A_PER; ++q) {   // the others hang behind it
        const uint32_t e = q * NT + tid;
        if (e >= n_e) continue;
        const uint32_t s = slots[q], h = S.head[s] & A_NONE;
        if (h == e) continue;
        uint32_t *half = reinterpret_cast<uint32_t *>(S.next) + (h >> 1);
        const uint32_t shift = (h & 1u) * 16u;
        uint32_t old = *reinterpret_cast<volatile uint32_t *>(half);
        while (true) {
            S.next[e] = (uint16_t)(old >> shift);
            const uint32_t seen = atomicCAS(half, old, (old & ~(0xFFFFu << shift)) | e << shift);
            if (seen == old) break;
            old = seen;
            if (give_up(++tries, A_TRIES)) {   // (hundreds of hits on one pixel)
                S.flag = 1u;
                break;
            }
        }
        S.head[s] = (uint16_t)(h | A_MULTI);
    }
    __syncthreads();
    if (GIVES_UP<NT> && S.flag) return;   // (by all: no thread writes it before the barrier in arrival_pairs)
    if (C.alias) arrival_pairs<NT, true>(S, C, n_e, near, join); else arrival_pairs<NT, false>(S, C, n_e, near, join);
}

// A pair: the hit's first makes the other its parent (always raster-earlier,
// or the next hit of its pixel, so parents form no cycle), others are listed.
template <int NT>
__device__ __forceinline__ void join_hits(ArrivalShared &S, uint32_t e, uint32_t j, bool &linked) {
    if (!linked) {
        S.par[e] = (uint16_t)j;
        linked = true;
        return;
    }
    const uint32_t k = atomicAdd(&S.nxtra, 1u);
    if (k < XTRA<NT>) xtra_list<NT>(S)[k] = e << 16 | j;
}

// Components of the staged hits, the clusters of the tile's own, their
// features, each own hit's cluster, and the pairs with earlier tiles (earlier
// hits in a cluster of this tile).  where()[e] (position from `origin`, ToT) of
// the entries is staged; the caller's barrier is behind it and the links.
// Earlier hits with keys from `within` on are of parts of this tile before: their
// clusters are joined at once.  false: more clusters than the tile has numbers.
template <int NT>
__device__ __forceinline__ bool arrival_clusters(const Work &w, const Seg &g, uint32_t t, ArrivalShared &S,
                                                 const Cells &C, uint32_t n_e, uint32_t origin, uint64_t base,
                                                 uint32_t within = 0xFFFFFFFFu) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int A_PER = (A_ENT + NT - 1) / NT;
    const uint32_t first_c = t * TILE + S.numbered;
    volatile uint16_t *par = S.par;
    uint2 *tops = S.tops();
    static_assert(A_TOPS <= (uint32_t)NT && A_TOPS <= 6 * 32, "a thread per word, six words per lane");
    if (tid < (int)A_TOPS) tops[tid] = make_uint2(0, 0);
    // Raster-order parents chain along a track; every hit first jumps to its
    // ancestors a few times (all hits at once, so paths shrink by half and
    // more each time) before unions and finds walk what is left.
#pragma unroll 1
    for (int r = 0; r < A_JUMPS; ++r) {
        uint32_t p[A_PER];
#pragma unroll
        for (int q = 0; q < A_PER; ++q)
            if (q * NT + tid < n_e) p[q] = par[q * NT + tid];
#pragma unroll
        for (int q = 0; q < A_PER; ++q)
            if (q * NT + tid < n_e) p[q] = par[p[q]];
#pragma unroll
        for (int q = 0; q < A_PER; ++q)
            if (q * NT + tid < n_e) p[q] = par[p[q]];
#pragma unroll
        for (int q = 0; q < A_PER; ++q)
            if (q * NT + tid < n_e) par[q * NT + tid] = (uint16_t)p[q];
    }
    __syncthreads();
    const uint32_t *xtra = xtra_list<NT>(S);
    for (uint32_t i = tid; i < min(S.nxtra, XTRA<NT>); i += NT) {
        uint32_t a = xtra[i] >> 16, b = xtra[i] & 0xFFFFu;
        while (true) {   // hook the larger root under the smaller
            a = arrival_root(S.par, a);
            b = arrival_root(S.par, b);
            if (a == b) break;
            if (a < b) { const uint32_t c = a; a = b; b = c; }
            if (arrival_hook(S.par, a, b)) break;
        }
    }
    __syncthreads();
    // Roots of all a thread's hits in step, their loads in flight together, each
    // step stored for the hits behind it (hit after hit, and marks, numbers and
    // parents in arrays: 2480 us for 64 Mi hits, in step 2364; without the
    // stores 3401, chains of a track's hits being long).
    // Roots with own hits are the tile's clusters (all are, but for earlier
    // hits that met none of this tile's): marked in a bitmap, numbered by rank.
    uint32_t top[A_PER];   // root of entry q * NT + tid
#pragma unroll
    for (int q = 0; q < A_PER; ++q) top[q] = q * NT + tid < n_e ? par[q * NT + tid] : 0u;
    for (bool more = true; more;) {
        more = false;
#pragma unroll
        for (int q = 0; q < A_PER; ++q) {
            if (q * NT + tid >= n_e) continue;
            const uint32_t p = par[top[q]];
            if (p != top[q]) {
                more = true;
                top[q] = p;
                par[q * NT + tid] = (uint16_t)p;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < A_PER; ++q) {
        const uint32_t e = q * NT + tid;
        if (e < n_e && S.kc[e].y & C_OWN) atomicOr(&tops[top[q] >> 5].x, 1u << (top[q] & 31u));
    }
    __syncthreads();
    if (warp == 0) {
        uint32_t c[6], sum = 0;
#pragma unroll
        for (uint32_t k = 0; k < 6; ++k) {
            c[k] = lane * 6 + k < A_TOPS ? __popc(tops[lane * 6 + k].x) : 0u;
            sum += c[k];
        }
        uint32_t run = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += y;
        }
        if (lane == 31) S.nroots = run;
        run -= sum;
#pragma unroll
        for (uint32_t k = 0; k < 6; ++k) {
            if (lane * 6 + k < A_TOPS) tops[lane * 6 + k].y = run;
            run += c[k];
        }
    }
    __syncthreads();
    uint32_t mine[(A_PER + 1) / 2];   // cluster (A_NONE: none) of entry q * NT + tid, two to a register
#pragma unroll
    for (int q = 0; q < A_PER; ++q) {
        const uint2 v = tops[top[q] >> 5];
        const uint32_t bit = 1u << (top[q] & 31u);
        const uint32_t c = v.x & bit ? v.y + __popc(v.x & (bit - 1u)) : A_NONE;
        mine[q >> 1] = q & 1 ? mine[q >> 1] | c << 16 : c;
    }
    auto cluster = [&](int q) { return q & 1 ? mine[q >> 1] >> 16 : mine[q >> 1] & 0xFFFFu; };
    // Features per cluster, as many clusters at once as the space holds.
    // Shared memory adds 32 bits natively and 64 by compare-and-swap loops:
    // while the tile's whole ToT keeps every sum in bounds (4096 hits of the
    // usual ToTs do, 40 times over) size and ToT share a word and the moments
    // take one each; otherwise the moments carry into a second word.
    uint32_t *A = S.sums();
    const uint32_t *where = S.where();
    const uint32_t nroots = S.nroots, tsum = S.tsum, magic = C.magic();
    if (nroots + S.numbered > TILE) return false;   // (nearly every hit alone, and more hits than positions)
    const bool streaming = g.ss != nullptr;
    const uint32_t reach = max(g.width, g.height);
    const bool slim = tsum < (1u << 19) && (unsigned long long)tsum * reach < (1ull << 32);
    static_assert(A_ENT < (1u << 13), "a size above a 19-bit sum ToT");
    constexpr uint32_t PASS = 2 * A_WORDS / 8;
    for (uint32_t r0 = 0; r0 == 0 || r0 < nroots; r0 += PASS) {
        const uint32_t nr = min(nroots - r0, PASS);
        for (uint32_t i = tid; i < nr; i += NT) {
#pragma unroll
            for (int k = 0; k < 6; ++k) A[k * PASS + i] = 0;
            A[6 * PASS + i] = A[7 * PASS + i] = 0xFFFFFFFFu;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < A_PER; ++q) {
            const uint32_t e = q * NT + tid;
            if (e >= n_e) break;
            const uint2 kc = S.kc[e];
            const uint32_t c = cluster(q), i = c - r0, pt = where[e], at = origin + (pt >> 16);
            if (!(kc.y & C_OWN)) {
                if (c != A_NONE && r0 == 0 && kc.x < within) {   // an earlier tile's hit in a cluster of this one
                    const uint32_t x = atomicAdd(&S.ncross, 1u);
                    if (x < A_PAIRS) w.xlist[(size_t)t * A_PAIRS + x] = make_uint2(first_c + c, at);
                }
                continue;
            }
            if (r0 == 0) {
                w.root_of[at] = first_c + c;
                if (w.rkey) w.rkey[at] = kc.x;
            }
            if (i < nr) {
                const uint32_t tot = pt & 0xFFFFu;
                uint32_t x, y;
                C.pixel(kc.y, magic, x, y);
                uint32_t *a = A + i;   // size (and ToT), ToT, x, carry, y, carry, first position, first key
                if (slim) {
                    atomicAdd(a, (1u << 19) + tot);
                    atomicAdd(a + 2 * PASS, tot * x);
                    atomicAdd(a + 4 * PASS, tot * y);
                } else {
                    const uint32_t vx = tot * x, vy = tot * y;
                    atomicAdd(a, 1u);
                    atomicAdd(a + PASS, tot);
                    if (atomicAdd(a + 2 * PASS, vx) > ~vx) atomicAdd(a + 3 * PASS, 1u);
                    if (atomicAdd(a + 4 * PASS, vy) > ~vy) atomicAdd(a + 5 * PASS, 1u);
                }
                atomicMin(a + 6 * PASS, pt >> 16);
                atomicMin(a + 7 * PASS, kc.x);
            }
        }
        __syncthreads();
        for (uint32_t i = tid; i < nr; i += NT) {
            const uint4 a = make_uint4(A[i], A[PASS + i], A[2 * PASS + i], A[3 * PASS + i]);
            const uint4 b = make_uint4(A[4 * PASS + i], A[5 * PASS + i], A[6 * PASS + i], A[7 * PASS + i]);
            const uint32_t cc = first_c + r0 + i;
            uint4 *slot = reinterpret_cast<uint4 *>(w.rslot + cc);
            slot[0] = make_uint4(slim ? a.x & 0x7FFFFu : a.y, 0u, a.z, a.w);
            slot[1] = make_uint4(b.x, b.y, slim ? a.x >> 19 : a.x, origin + b.z);
            w.rfirst[cc] = base + b.w;
            w.gpar[cc] = cc;
        }
        if (streaming) {   // last ToAs, in the place of the first ones
            __syncthreads();
            for (uint32_t i = tid; i < nr; i += NT) A[7 * PASS + i] = 0;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < A_PER; ++q) {
                const uint32_t e = q * NT + tid, i = cluster(q) - r0;
                if (e >= n_e) break;
                const uint2 kc = S.kc[e];
                if ((kc.y & C_OWN) && i < nr) atomicMax(&A[7 * PASS + i], kc.x);
            }
            __syncthreads();
            for (uint32_t i = tid; i < nr; i += NT) w.rlast[first_c + r0 + i] = base + A[7 * PASS + i];
        }
        __syncthreads();
    }
    if (within != 0xFFFFFFFFu) {
#pragma unroll
        for (int q = 0; q < A_PER; ++q) {
            const uint32_t e = q * NT + tid, c = cluster(q);
            if (e >= n_e) break;
            const uint2 kc = S.kc[e];
            if (!(kc.y & C_OWN) && c != A_NONE && kc.x >= within) gunion(w.gpar, first_c + c, w.root_of[origin + (where[e] >> 16)]);
        }
    }
    if (tid == 0) w.atile[t].nroots = S.numbered += nroots;
    return true;
}

// Cut before tile j of a segment: the median ToA key of 32 hits around its
// first position, the same for both tiles that need it (called by a warp).
__device__ __forceinline__ uint32_t arrival_cut(const Seg &g, uint32_t j, uint64_t base, int lane) {
    if (j == 0) return 0u;
    if (j >= g.ntiles) return 0xFFFFFFFFu;   // above every key that is not wide
    const uint32_t p = min(j * TILE - 512u + 32u * lane, g.n - 1u);
    const uint32_t key = (uint32_t)(hit_toa(ld_hit(g.hits + p)) - base);
    uint32_t rank = 0;
#pragma unroll
    for (int o = 1; o < 32; ++o) {
        const int from = (lane + o) & 31;
        const uint32_t k = __shfl_sync(0xffffffffu, key, from);
        rank += k < key || (k == key && from < lane);
    }
    return __shfl_sync(0xffffffffu, key, __ffs(__ballot_sync(0xffffffffu, rank == 16u)) - 1);
}

// Bound by issue and shared-memory latency, not by bytes: 64 Mi hits (256x256)
// take 2260 us at 16 B read and 8 B written each (the cluster, and the key that
// tpc_forest reads).  Of a tile's time the records
// take 22 percent, cell numbers and heads 9, the walk over neighbour cells 17,
// crowded cells 8, positions and ToTs 7, the forest and its roots 24, features
// 10.  Two CTAs of 512 threads at 64 registers; one of 1024 takes 2906 (its
// barriers leave nothing to run), 768 threads at 40 registers spill (2936).  Entry
// numbers are counted again for the positions instead of kept: 2324 -> 2260.
//
// PARTS: the tiles that did not fit (listed by the kernel without it), their
// intervals taken in halves (and those again, while they are a quarter of dt or
// longer), each one seeing the dt before it.  On both sides every part reads on
// while the outermost positions hold hits of the whole tile, its earlier ones
// among them, whether they are the part's or not: so all parts read the same
// positions, what is proved of the first part's earlier hits holds for the
// others' (they are among those, or the tile's own), and an own hit that a part
// meets was numbered by an earlier part.  (A part that reads on to the right for
// its own hits only misses one that arrived late and belongs to an earlier part,
// or meets one that no part numbered.)  8 M hits on 448x512 at 2.5 Ghits/s, dt
// 384, where no tile fits: 1110 us, 1300 time-sorted.  A kernel of its own: with
// the parts in the loop, their state spilled (2456 us for 64 Mi hits).
template <int NT, bool PARTS>
__global__ void __launch_bounds__(NT, 1024 / NT) k_arrival_tile(Work w) {
    constexpr uint32_t MARGIN = PARTS ? A_WIDE : A_MARGIN;
    constexpr int A_ITEMS = (TILE + 2 * MARGIN) / NT;   // records per thread
    static_assert(A_ITEMS * NT == TILE + 2 * (int)MARGIN && A_ITEMS % A_GROUP == 0 && A_ITEMS <= 32, "whole rounds");
    extern __shared__ __align__(16) unsigned char a_raw[];
    ArrivalShared &S = *reinterpret_cast<ArrivalShared *>(a_raw);
    Prob &P = *w.prob;
    const uint32_t nt = PARTS ? (P.raw_fail == RAW_PARTS ? P.parts_count : 0u) : P.ntiles, nsegs = P.nsegs;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t u = blockIdx.x; u < nt; u += gridDim.x) {
        const uint32_t t = PARTS ? w.redo[u] : u;
        const uint32_t si = nsegs == 1 ? 0u : w.tile_seg[t];
        const Seg &g = w.seg[si];
        if (!PARTS && t + gridDim.x < nt) {   // the next tile's records on their way to L2
            const uint32_t t1 = t + gridDim.x;
            const Seg &g1 = nsegs == 1 ? g : w.seg[w.tile_seg[t1]];
            const uint32_t p = (t1 - g1.tile0) * TILE + tid * (128u / sizeof(tpc_hit));
            if (p < g1.n) asm volatile("prefetch.global.L2 [%0];" ::"l"(g1.hits + p));
        }
        const uint32_t j = t - g.tile0, n = g.n, off = g.off, dt = g.dt, W = g.width, H = g.height;
        const uint64_t base = g.raw_base;
        const tpc_hit *hits = g.hits;
        const Cells C(W, H);
        bool first = true;
        while (true) {   // (once without PARTS)
        // ---- records around the tile --------------------------------------
        const int32_t p0 = (int32_t)(j * TILE) - (int32_t)MARGIN + tid;   // position (in the segment) of record 0
        uint4 v[A_GROUP];
#pragma unroll
        for (int q = 0; q < A_GROUP; ++q) {
            const int32_t p = p0 + q * NT;
            if ((uint32_t)p < n) v[q] = ld_hit(hits + p);
        }
        if (tid == 0) {
            S.flag = *reinterpret_cast<volatile uint32_t *>(&P.raw_fail) > RAW_PARTS;
            S.nent = S.nown = S.nxtra = S.nroots = S.tsum = 0;
            if (first) S.ntail = S.kept_tail = S.ncross = S.numbered = 0;
        }
        C.clear<NT>(S);
        if (first && warp < 2) {
            const uint32_t k = arrival_cut(g, j + warp, base, lane);
            if (lane == 0) S.cut[warp] = k;
            if (PARTS && lane == 0) (warp ? S.to : S.from) = k;
        }
        const uint32_t n_carry = g.n_carry, limit = (W - 1u) | (H - 1u) << 16;
        __syncthreads();
        const bool last = j + 1 == g.ntiles;
        if (PARTS && first) {   // halves from the start
            if (tid == 0 && j && j + 1 < g.ntiles && S.to > S.from && S.to - S.from >= max(dt, 2u)) S.to = S.from + (S.to - S.from) / 2;
            __syncthreads();
        }
        const uint32_t cut = PARTS ? S.from : S.cut[0], cut1 = PARTS ? S.to : S.cut[1];   // own keys: cut <= key < cut1
        if (S.flag) return;           // the time-sorted path takes the step
        if (S.cut[1] < S.cut[0]) {    // no time order to speak of
            if (tid == 0) P.raw_fail = RAW_UNORDERED;
            return;
        }
        const uint32_t lo = cut > dt ? cut - dt : 0u;             // earlier hits below it join nothing here
        const uint32_t span = cut1 - lo;                          // kept keys: key - lo < span
        const uint32_t whole = S.cut[0] > dt ? S.cut[0] - dt : 0u, reach = S.cut[1] - whole;   // (PARTS) of all parts
        const uint32_t tail = last ? 0xFFFFFFFFu : S.cut[1] > dt ? S.cut[1] - dt : 0u;   // own hits the next tile must see
        const uint32_t guard = base ? ARRIVAL_DT : 0u;
        uint32_t high = 0, bad = 0, kmin = 0xFFFFFFFFu, kmax = 0, cmin = 0xFFFFFFFFu;
        uint32_t tots[A_ITEMS / 2], staged = 0, own_sum = 0, tsum = 0, edge = 0;   // own_sum: own | tail << 16
        // one record: its key and code; whether it is staged
        auto look = [&](const uint4 &r, int32_t p, uint32_t &key, uint32_t &code) -> bool {
            key = 0;
            if ((uint32_t)p >= n) return false;   // (before the segment too)
            const uint64_t rel = hit_toa(r) - base;
            key = (uint32_t)rel;
            high |= (uint32_t)(rel >> 32);
            const uint32_t pix = __vminu2(r.x, limit);
            bad |= pix ^ r.x;
            kmin = min(kmin, key);
            kmax = max(kmax, key);
            if (n_carry && (uint32_t)p >= n_carry) cmin = min(cmin, key);
            code = C.code(pix);
            return key - lo < span;
        };
#pragma unroll
        for (int h = 0; h < A_ITEMS / A_GROUP; ++h) {
            uint32_t key[A_GROUP], code[A_GROUP], mask[A_GROUP], sum = 0;
#pragma unroll
            for (int q = 0; q < A_GROUP; ++q) {
                const int i = h * A_GROUP + q;
                const bool kept = look(v[q], p0 + i * NT, key[q], code[q]);
                mask[q] = __ballot_sync(0xffffffffu, kept);
                sum += __popc(mask[q]);
                tots[i >> 1] = i & 1 ? tots[i >> 1] | hit_tot(v[q]) << 16 : hit_tot(v[q]);
                if (kept) {
                    staged |= 1u << i;
                    if (key[q] >= cut) {
                        own_sum += key[q] >= tail && !last ? 0x10001u : 1u;
                        tsum += hit_tot(v[q]);
                        if (!PARTS && i == A_ITEMS - 1) edge |= 2u;
                    }
                    if (!PARTS && i == 0) edge |= 1u;
                }
                if (PARTS && (i == 0 || i == A_ITEMS - 1) && (uint32_t)(p0 + i * NT) < n && key[q] - whole < reach)
                    edge |= i ? 2u : 1u;
            }
            if (h + 1 < A_ITEMS / A_GROUP) {
#pragma unroll
                for (int q = 0; q < A_GROUP; ++q) {
                    const int32_t p = p0 + ((h + 1) * A_GROUP + q) * NT;
                    if ((uint32_t)p < n) v[q] = ld_hit(hits + p);
                }
            }
            uint32_t e0 = 0;
            if (lane == 0) e0 = atomicAdd(&S.nent, sum);
            if (lane == 0) S.first[warp][h] = (uint16_t)e0;   // (more than 2^16: not covered)
            e0 = __shfl_sync(0xffffffffu, e0, 0);
#pragma unroll
            for (int q = 0; q < A_GROUP; ++q) {
                const int i = h * A_GROUP + q;
                const uint32_t e = e0 + __popc(mask[q] & lanes_below());
                if (((staged >> i) & 1u) && e < A_ENT) {
                    S.kc[e] = make_uint2(key[q], code[q] | (key[q] >= cut ? C_OWN : 0u));
                    C.set(S, code[q]);
                }
                e0 += __popc(mask[q]);
            }
        }
        const bool given_up = tid == 0 && *reinterpret_cast<volatile uint32_t *>(&P.raw_fail) > RAW_PARTS;
        own_sum = __reduce_add_sync(0xffffffffu, own_sum);
        tsum = __reduce_add_sync(0xffffffffu, tsum);
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        cmin = n_carry ? __reduce_min_sync(0xffffffffu, cmin) : kmin;   // (no carry: every hit is new)
        edge = __reduce_or_sync(0xffffffffu, edge | (bad ? 4u : 0u));
        if (lane == 0) {
            atomicAdd(&S.nown, own_sum & 0xFFFFu);
            if (own_sum >> 16) atomicAdd(&S.ntail, own_sum >> 16);
            atomicAdd(&S.tsum, tsum);
            S.red[0][warp] = kmin;
            S.red[1][warp] = kmax;
            S.red[2][warp] = cmin;
            S.red[3][warp] = edge;
        }
        const bool wide = high || kmin < guard || kmax > 0xFFFFFFFFu - ARRIVAL_DT;
        if (__syncthreads_or((wide && kmin <= kmax) || given_up)) {   // (no hits: kmin > kmax)
            if (tid == 0) atomicMax(&P.raw_fail, RAW_COVER);
            return;
        }
        edge = __reduce_or_sync(0xffffffffu, S.red[3][min(lane, (NT / 32) - 1)]);
        // ---- hits beyond the margins: rounds while the outermost hits
        // read still held some of the tile --------------------------
        const uint32_t e_far = min(S.nent, A_ENT);
        if (edge & 3u) __syncthreads();   // read by all before a round adds to it
        const int32_t win = (int32_t)(j * TILE) - (int32_t)(MARGIN + A_ROUNDS * A_STEP);   // origin of positions
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            bool more = (edge >> side) & 1u;
            int32_t a = side ? (int32_t)((j + 1) * TILE + MARGIN) : (int32_t)(j * TILE) - (int32_t)(MARGIN + A_STEP);
#pragma unroll 1
            for (int r = 0; more && r < A_ROUNDS && (side ? a < (int32_t)n : a + (int32_t)A_STEP > 0); ++r) {
                bool outer = false;
#pragma unroll 1
                for (uint32_t u = tid; u < A_STEP; u += NT) {
                    const int32_t p = a + (int32_t)u;
                    uint32_t key, code;
                    uint4 x = make_uint4(0, 0, 0, 0);
                    if ((uint32_t)p < n) x = ld_hit(hits + p);
                    const bool kept = look(x, p, key, code);
                    if (PARTS) outer |= (uint32_t)p < n && key - whole < reach;
                    if (!kept) continue;
                    if (!PARTS) outer |= !side || key >= cut;
                    const uint32_t e = atomicAdd(&S.nent, 1u);
                    if (e < A_ENT && e - e_far < A_FAR) {
                        S.kc[e] = make_uint2(key, code | (key >= cut ? C_OWN : 0u));
                        S.far[e - e_far] = (uint16_t)(p - win);
                        C.set(S, code);
                    } else {
                        S.flag = 1u;
                    }
                    if (key >= cut) {
                        atomicAdd(&S.nown, 1u);
                        atomicAdd(&S.tsum, hit_tot(x));
                        if (key >= tail && !last) atomicAdd(&S.ntail, 1u);
                    }
                }
                more = __syncthreads_or(outer);
                a += side ? (int32_t)A_STEP : -(int32_t)A_STEP;
            }
        }
        const uint32_t n_e = S.nent;
        if (n_e > A_ENT || S.flag) {
            // own hits as far out as the last rounds on both sides: disorder that
            // sorting by tiles cannot mend either
            int out[2];
            for (int side = 0; side < 2; ++side) {
                bool own = false;
                for (uint32_t u = tid; u < A_STEP; u += NT) {
                    const int32_t p = side ? (int32_t)((j + 1) * TILE + MARGIN + (A_ROUNDS - 1) * A_STEP + u) : win + (int32_t)u;
                    if ((uint32_t)p < n) own |= (uint32_t)(hit_toa(ld_hit(hits + p)) - base) - S.cut[0] < S.cut[1] - S.cut[0];
                }
                out[side] = __syncthreads_count(own);
            }
            if (min(out[0], out[1]) >= 32) {
                if (tid == 0) atomicMax(&P.raw_fail, RAW_UNORDERED);
                return;
            }
            if (!PARTS) {   // left to the kernel with PARTS
                if (tid == 0) {
                    w.redo[atomicAdd(&P.parts_count, 1u)] = t;
                    atomicMax(&P.raw_fail, RAW_PARTS);
                }
                __syncthreads();   // the counters are reset for the next tile
                break;
            }
            bool lost = false;
            __syncthreads();   // (S.nent is read by all)
            if (tid == 0) {   // the first half of it
                uint32_t lowest = 0xFFFFFFFFu, highest = 0;
                for (int q = 0; q < NT / 32; ++q) {
                    lowest = min(lowest, S.red[0][q]);
                    highest = max(highest, S.red[1][q]);
                }
                const uint32_t begin = max(cut, lowest), end = min(cut1, highest + 1u);
                const uint32_t half = end > begin ? (end - begin) / 2 : 0u;
                S.to = begin + half;
                S.ntail = S.kept_tail;
                lost = n_e <= A_ENT || 4 * (uint64_t)half < dt || !half;   // too many far hits; parts too short
                if (lost) atomicMax(&P.raw_fail, RAW_COVER);
            }
            if (__syncthreads_or(lost)) return;
            first = false;
            continue;
        }
        ATile &info = w.atile[t];
        if (warp == 0) {
            kmin = __reduce_min_sync(0xffffffffu, S.red[0][min(lane, (NT / 32) - 1)]);
            kmax = __reduce_max_sync(0xffffffffu, S.red[1][min(lane, (NT / 32) - 1)]);
            cmin = __reduce_min_sync(0xffffffffu, S.red[2][min(lane, (NT / 32) - 1)]);
            if (lane == 0) {
                Seg &gw = w.seg[si];
                atomicMin(reinterpret_cast<unsigned long long *>(&gw.toa_min), (unsigned long long)(base + kmin));
                atomicMax(reinterpret_cast<unsigned long long *>(&gw.toa_max), (unsigned long long)(base + kmax));
                if (cmin != 0xFFFFFFFFu)
                    atomicMin(reinterpret_cast<unsigned long long *>(&gw.chunk_min), (unsigned long long)(base + cmin));
                atomicAdd(&gw.n_owned, S.nown);
                if (edge & 4u) atomicOr(&P.err, E_RANGE);
                if (!PARTS || cut == S.cut[0]) {
                    info.base = base;
                    info.cut = cut;
                    info.nhalo = n_e - S.nown;
                }
                info.ntail = S.ntail;
                if (PARTS) S.kept_tail = S.ntail;
            }
        }
        // ---- links -----------------------------------------------------------
        // (keys keep 2^27 from both ends of 32 bits and dt is less: the sum wraps for no far pair)
        const uint32_t dt2 = 2u * dt;
        arrival_links<NT>(S, C, n_e, [&](uint32_t a, uint32_t b) { return a - b + dt <= dt2; },
                      [&](uint32_t e, uint32_t o, bool &linked) { join_hits<NT>(S, e, o, linked); });
        __syncthreads();
        // ---- positions and ToTs of the entries, where the lists were ---------
        uint32_t *where = S.where();
#pragma unroll
        for (int h = 0; h < A_ITEMS / A_GROUP; ++h) {   // (the entries as they were counted above)
            uint32_t e0 = S.first[warp][h];
#pragma unroll
            for (int i = h * A_GROUP; i < (h + 1) * A_GROUP; ++i) {
                const uint32_t kept = __ballot_sync(0xffffffffu, (staged >> i) & 1u);
                if ((staged >> i) & 1u)
                    where[e0 + __popc(kept & lanes_below())] =
                        (uint32_t)(p0 + i * NT - win) << 16 | (tots[i >> 1] >> (i & 1) * 16 & 0xFFFFu);
                e0 += __popc(kept);
            }
        }
        for (uint32_t e = e_far + tid; e < n_e; e += NT)
            where[e] = (uint32_t)S.far[e - e_far] << 16 | hit_tot(ld_hit(hits + (win + (int32_t)S.far[e - e_far])));
        const bool listed = S.nxtra <= A_XTRA;
        __syncthreads();
        if (!listed || !arrival_clusters<NT>(w, g, t, S, C, n_e, off + (uint32_t)win, base, PARTS && cut != S.cut[0] ? S.cut[0] : 0xFFFFFFFFu) || S.ncross > A_PAIRS) {
            if (tid == 0) atomicMax(&P.raw_fail, RAW_COVER);
            return;
        }
        if (tid == 0) {
            info.nx = S.ncross;
            if (PARTS) {
                S.from = cut1;
                S.to = S.cut[1];
            }
        }
        const bool all = !PARTS || cut1 == S.cut[1];
        __syncthreads();   // the counters are reset for the next part, or tile
        if (all) break;
        first = false;
        }
    }
}

// ---------------------------------------------------------------------------
// Small steps: tiles own their positions, whatever the order.

// One tile; false: left to any_order (more hits within dt, pairs or hits of
// single pixels than it holds, or earlier hits too far back).
template <int NT>
__device__ __forceinline__ bool small_tile(const Work &w, uint32_t t, SmallShared &SS) {
    ArrivalShared &S = SS.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Seg &g = w.seg[0];   // (a small step has one segment)
    uint32_t begin, end;
    tile_range(g, t, begin, end);
    const uint32_t n_t = end - begin, dt = g.dt, W = g.width, H = g.height;
    const tpc_hit *hits = g.hits;
    const Cells C(W, H);
    ATile &info = w.atile[t];
    constexpr int OWN = (TILE + NT - 1) / NT, A_HPER = (A_STEP + NT - 1) / NT;

    // ---- the tile's own hits ---------------------------------------------
    uint64_t base = g.raw_base;
    const uint64_t low = base ? A_GUARD : 0, room = (1ull << 32) - A_GUARD - low;
    bool wide = dt >= A_GUARD;
    const uint32_t new0 = g.n_carry > begin ? g.n_carry - begin : 0;   // first new hit
    uint32_t kmin, kmax, tots[OWN];
    if (tid == 0) S.nxtra = S.ncross = S.nroots = S.tsum = S.numbered = S.flag = 0;
    C.clear<NT>(S);
    __syncthreads();
    for (int attempt = 0;; ++attempt) {
        bool bad = false;
        uint32_t cmin = 0xFFFFFFFFu;
        kmin = 0xFFFFFFFFu;
        if (tid < (int)ACHUNKS) S.cnt[1][tid] = 0;   // largest key of each chunk
        __syncthreads();
        uint4 v[OWN];
#pragma unroll
        for (int q = 0; q < OWN; ++q)
            if (q * NT + tid < n_t) v[q] = ld_hit(hits + begin + q * NT + tid);
#pragma unroll
        for (int q = 0; q < OWN; ++q) {
            const uint32_t e = q * NT + tid;
            tots[q] = 0;
            const uint32_t top = __reduce_max_sync(0xffffffffu, e < n_t ? (uint32_t)(hit_toa(v[q]) - base) : 0u);
            if (lane == 0 && e < n_t) atomicMax(&S.cnt[1][e / A_STEP], top);   // (a warp's hits share a chunk)
            if (e >= n_t) continue;
            const uint64_t rel = hit_toa(v[q]) - base;
            const uint32_t key = (uint32_t)rel, pix = clamp_pix(v[q].x, W, H), code = C.code(pix);
            wide |= rel - low > room;
            bad |= pix != v[q].x;
            tots[q] = hit_tot(v[q]);
            S.kc[e] = make_uint2(key, code | C_OWN);
            SS.pos[e] = (uint16_t)(begin + e);
            C.set(S, code);
            kmin = min(kmin, key);
            if (e >= new0) cmin = min(cmin, key);
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&w.prob->err, E_RANGE);
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        cmin = __reduce_min_sync(0xffffffffu, cmin);
        if (lane == 0) { S.red[0][warp] = kmin; S.red[1][warp] = cmin; }
        if (!__syncthreads_or(wide && attempt == 0)) break;
        // keys relative to the segment's smallest ToA (which hold its ToAs
        // unless they span 2^32 ticks: an error)
        uint64_t m = ~0ull, mx = 0;
        for (uint32_t i = tid; i < g.n; i += NT) {
            const uint64_t a = hit_toa(ld_hit(hits + i));
            m = a < m ? a : m;
            mx = a > mx ? a : mx;
        }
        m = warp_min_u64(m);
        mx = warp_max_u64(mx);
        if (lane == 0) { S.m64[0][warp] = m; S.m64[1][warp] = mx; }
        __syncthreads();
        for (int q = 0; q < (NT / 32); ++q) {
            m = S.m64[0][q] < m ? S.m64[0][q] : m;
            mx = S.m64[1][q] > mx ? S.m64[1][q] : mx;
        }
        if (tid == 0 && (mx - m) >> 32) atomicOr(&w.prob->err, E_SPAN);
        base = m;
    }
    {
        kmin = __reduce_min_sync(0xffffffffu, S.red[0][min(lane, (NT / 32) - 1)]);
        kmax = __reduce_max_sync(0xffffffffu, S.cnt[1][min(lane, (int)ACHUNKS - 1)]);
    }
    const uint32_t lo = kmin > dt ? kmin - dt : 0u;       // earlier hits below it join nothing here
    const uint64_t hi = (uint64_t)kmax + dt;
    if (warp == 0) {
        const uint32_t cmin = __reduce_min_sync(0xffffffffu, S.red[1][min(lane, (NT / 32) - 1)]);
        if (lane < (int)ACHUNKS) info.cmax[lane] = base + S.cnt[1][lane];
        if (lane == 0) {
            Seg &gw = w.seg[0];
            atomicMin(reinterpret_cast<unsigned long long *>(&gw.toa_min), (unsigned long long)(base + kmin));
            atomicMax(reinterpret_cast<unsigned long long *>(&gw.toa_max), (unsigned long long)(base + kmax));
            if (new0 < n_t)
                atomicMin(reinterpret_cast<unsigned long long *>(&gw.chunk_min), (unsigned long long)(base + cmin));
            info.base = base;
            info.lo = base + lo;
        }
    }

    // ---- links, with the earlier hits in rounds of A_STEP positions --------
    uint32_t h0 = begin;            // every position in [h0, begin) has been looked at
    uint32_t n_e = n_t;
    bool done = begin == 0;
    for (uint32_t buf = 0; !done;) {
        const uint32_t a = h0 - A_STEP;
        uint32_t kk[A_HPER], pp[A_HPER], mask[A_HPER], sum = 0;
#pragma unroll
        for (int u = 0; u < A_HPER; ++u) {
            const uint4 v = ld_hit(hits + a + u * NT + tid);
            const uint64_t rel = hit_toa(v) - base;
            kk[u] = (uint32_t)rel;
            pp[u] = C.code(clamp_pix(v.x, W, H));
            mask[u] = __ballot_sync(0xffffffffu, rel >= lo && rel <= hi);
            sum += __popc(mask[u]);
        }
        if (lane == 0) S.turn[buf][warp] = sum | (mask[0] ? 0x80000000u : 0u);
        __syncthreads();
        const uint32_t c = lane < (NT / 32) ? S.turn[buf][lane] : 0u;
        buf ^= 1u;   // the next round's barrier separates this one's reads from the round after
        const uint32_t total = __reduce_add_sync(0xffffffffu, c & 0x7FFFFFFFu);
        const bool oldest = __any_sync(0xffffffffu, c >> 31);   // some of the oldest NT positions matter
        if (n_e + total > A_ENT) return false;   // no room beside the staged ones
        uint32_t e = n_e + __reduce_add_sync(0xffffffffu, lane < warp ? c & 0x7FFFFFFFu : 0u);
#pragma unroll
        for (int u = 0; u < A_HPER; ++u) {
            if ((mask[u] >> lane) & 1u) {
                const uint32_t i = e + __popc(mask[u] & lanes_below());
                S.kc[i] = make_uint2(kk[u], pp[u]);
                SS.pos[i] = (uint16_t)(a + u * NT + tid);
                C.set(S, pp[u]);
            }
            e += __popc(mask[u]);
        }
        n_e += total;
        h0 = a;
        done = h0 == 0 || !oldest;
        if (!done && begin - h0 == A_BACK_ROUNDS * A_STEP) return false;
    }
    arrival_links<NT>(S, C, n_e, [&](uint32_t a, uint32_t b) { return absdiff(a, b) <= dt; },
                      [&](uint32_t e, uint32_t o, bool &linked) { join_hits<NT>(S, e, o, linked); });
    __syncthreads();
    if (S.nxtra > XTRA<NT> || S.flag) return false;
    uint32_t tsum = 0;
#pragma unroll
    for (int q = 0; q < OWN; ++q) {
        const uint32_t e = q * NT + tid;
        if (e < n_t) S.where()[e] = (uint32_t)SS.pos[e] << 16 | tots[q];
        tsum += tots[q];
    }
    for (uint32_t e = n_t + tid; e < n_e; e += NT) S.where()[e] = (uint32_t)SS.pos[e] << 16;
    tsum = __reduce_add_sync(0xffffffffu, tsum);
    if (lane == 0) atomicAdd(&S.tsum, tsum);
    __syncthreads();
    arrival_clusters<NT>(w, g, t, S, C, n_e, 0u, base);   // (at most TILE clusters)
    if (tid == 0) {
        info.h0 = h0;
        info.nx = S.ncross;
    }
    return true;
}

// Joins the listed pairs of a tile, `first` of NT threads.  Many pairs join the
// same two clusters: of a warp's pairs that do, one thread joins them.
template <int NT>
__device__ __forceinline__ void join_pairs(const Work &w, uint32_t t, uint32_t first) {
    const uint32_t nx = min(w.atile[t].nx, (uint32_t)A_PAIRS);
    const uint2 *list = w.xlist + (size_t)t * A_PAIRS;
    volatile uint32_t *par = w.gpar;
    for (uint32_t i = first; i < nx; i += NT) {
        const uint2 p = list[i];
        const uint32_t a = par[p.x], b = par[w.root_of[p.y]];
        const uint32_t same = __match_any_sync(__activemask(), (unsigned long long)a << 32 | b);
        if (a != b && __ffs(same) - 1 == (int)(threadIdx.x & 31)) gunion(w.gpar, a, b);
    }
}

// Joins the listed pairs, and proves that the tiles cover the step: their
// ToA intervals are disjoint, so every hit found its tile if the own hits add
// up to all hits; and a tile saw every earlier hit within dt of its interval
// if it counted as many of them as its predecessor counted own hits that
// late (which are all there are, if dt reaches no further back than the
// predecessor's interval).  A warp per tile: the few pairs of a tile of time
// (six of 64 Mi hits) are one chain of dependent reads, and with a CTA per tile
// too few of them were under way (96 us, 39 with a warp and one join per
// distinct pair of clusters).
constexpr int AX = 256;

__global__ void __launch_bounds__(AX) k_arrival_cross(Work w, cudaGraphConditionalHandle otherwise, bool parts) {
    __shared__ uint32_t s_failed;
    Prob &P = *w.prob;
    const int tid = threadIdx.x;
    bool stray = false;
    for (uint32_t s = tid; s < P.nsegs; s += AX) stray |= w.seg[s].n_owned != w.seg[s].n;
    if (tid == 0) s_failed = *reinterpret_cast<volatile uint32_t *>(&P.raw_fail);
    stray = __syncthreads_or(stray);
    const uint32_t failed = s_failed;
    const bool lost = stray || (parts ? failed > RAW_PARTS : failed != 0);
    bool fail = false;
    if (!lost) {
        const uint32_t nt = P.ntiles;
        for (uint32_t t = (blockIdx.x * AX + tid) / 32; t < nt; t += gridDim.x * (AX / 32)) {
            const Seg &g = w.seg[w.tile_seg[t]];
            if (t > g.tile0) {   // (every lane)
                const ATile &info = w.atile[t], &prev = w.atile[t - 1];
                fail |= info.nhalo != prev.ntail || (t - 1 > g.tile0 && info.cut < prev.cut + g.dt);
            }
            join_pairs<32>(w, t, tid & 31);
        }
    }
    // (one thread where all agree: a thousand of them took 10 us.  Hits beyond
    // the positions read are beyond the sorted path's merge too.)
    if (lost ? blockIdx.x == 0 && tid == 0 : fail && (tid & 31) == 0) {
        const bool again = !parts && failed == RAW_PARTS;
        if (!again) atomicMax(&P.raw_fail, stray && failed <= RAW_PARTS ? RAW_UNORDERED : RAW_COVER);
        if (otherwise) cudaGraphSetConditional(otherwise, again ? 0u : 1u);
    }
    if (blockIdx.x == 0 && (parts || failed != RAW_PARTS))
        for (uint32_t s = tid; s < P.nsegs; s += AX) seg_close(w.seg[s], P);
}

// Each tile cluster adds its features to its cluster's, and points straight
// at it.  The finds write nothing on their way: a path halved with a parent
// read before another thread's final store would undo that store.
template <int NT>
__device__ __forceinline__ void root_tile(const Work &w, uint32_t t, bool streaming) {
    const uint32_t nr = w.atile[t].nroots;
    for (uint32_t i = threadIdx.x; i < nr; i += NT) {
        const uint32_t c = t * TILE + i;
        volatile uint32_t *par = w.gpar;
        uint32_t r = c;
        for (uint32_t p = par[r]; p != r; p = par[r]) r = p;
        if (r == c) continue;
        w.gpar[c] = r;
        const RootSlot s = w.rslot[c];
        RootSlot &d = w.rslot[r];
        atomicAdd(&d.tot, s.tot);
        atomicAdd(&d.wx, s.wx);
        atomicAdd(&d.wy, s.wy);
        atomicAdd(&d.size, s.size);
        atomicMin(&d.min, s.min);
        atomicMin(reinterpret_cast<unsigned long long *>(&w.rfirst[r]), (unsigned long long)w.rfirst[c]);
        if (streaming) atomicMax(reinterpret_cast<unsigned long long *>(&w.rlast[r]), (unsigned long long)w.rlast[c]);
    }
}

__global__ void __launch_bounds__(256) k_arrival_roots(Work w) {
    const Prob &P = *w.prob;
    if (P.raw_fail > RAW_PARTS) return;
    const uint32_t nt = P.ntiles;
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) root_tile<256>(w, t, w.seg[w.tile_seg[t]].ss != nullptr);
}

// Labels of the hits at a tile's positions.  Their clusters are mostly tile
// clusters of this time tile and the two beside it: those tiles' labels are
// gathered once into shared memory (if they fit), then looked up per hit.
// Bound by DRAM and the two dependent reads behind a table entry; the hits'
// clusters are read beside those (64 Mi hits: 311 us after them, 247 so, for
// 256 MB read, 512 MB written and the clusters' slots).
constexpr uint32_t AL_CAP = 4096;

template <int NT>
__device__ __forceinline__ void label_tile(const Work &w, uint32_t t, const Seg &g, uint32_t *s_lab, uint32_t *s_cnt) {
    const int lane = threadIdx.x & 31;
    constexpr uint32_t CLOSED = 0x80000000u;   // a segment holds at most 2^31 - 1 hits
    uint32_t begin, end;
    tile_range(g, t, begin, end);
    const uint32_t mode = g.close_mode, off = g.off;
    const uint64_t mark = g.watermark;
    auto label_of = [&](uint32_t c) -> uint32_t {
        const uint32_t r = w.gpar[c];
        const bool closed = mode == CLOSE_ALL || (mode == CLOSE_WM && w.rlast[r] <= mark);
        return (w.rslot[r].min - off) | (closed ? CLOSED : 0u);
    };
    const uint32_t n0 = t > g.tile0 ? w.atile[t - 1].nroots : 0, n1 = w.atile[t].nroots;
    const uint32_t n2 = t + 1 < g.tile0 + g.ntiles ? w.atile[t + 1].nroots : 0;
    const bool table = n0 + n1 + n2 <= AL_CAP;
    constexpr int ITEMS = TILE / NT;
    uint32_t cc[ITEMS];   // the hits' clusters, on their way while the table is filled
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const uint32_t pos = begin + q * NT + threadIdx.x;
        cc[q] = pos < end ? w.root_of[pos] : 0u;
    }
    // c in [c0, c0 + n0), [c1, c1 + n1), [c2, c2 + n2): s_lab[c - c0], s_lab[n0 + c - c1], ...
    const uint32_t c1 = t * TILE, c0 = c1 - TILE, c2 = c1 + TILE;
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    if (table)
        for (uint32_t i = threadIdx.x; i < n0 + n1 + n2; i += NT)
            s_lab[i] = label_of(i < n0 ? c0 + i : i < n0 + n1 ? c1 + i - n0 : c2 + i - n0 - n1);
    __syncthreads();
    const bool direct = g.ss == nullptr;   // one-shot: every hit is final
    uint32_t c_label = 0, c_closed = 0;
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const uint32_t pos = begin + q * NT + threadIdx.x;
        bool is_label = false, closed = false;
        if (pos < end) {
            const uint32_t c = cc[q];
            uint32_t v;
            if (table && c - c1 < n1) v = s_lab[n0 + c - c1];
            else if (table && c - c0 < n0) v = s_lab[c - c0];
            else if (table && c - c2 < n2) v = s_lab[n0 + n1 + c - c2];
            else v = label_of(c);
            const uint32_t l = v & ~CLOSED;
            closed = (v & CLOSED) != 0;
            is_label = closed && l == pos - off;
            const uint64_t lab = gidx_of(g, l);
            if (direct) g.out_labels[pos - off] = lab;
            else w.lab_tmp[pos] = lab;
        }
        const uint32_t bl = __ballot_sync(0xffffffffu, is_label);
        const uint32_t bc = __ballot_sync(0xffffffffu, closed);
        if (lane == 0) {
            w.flag_label[pos >> 5] = bl;
            w.flag_closed[pos >> 5] = bc;
            c_label += __popc(bl);
            c_closed += __popc(bc);
        }
    }
    if (lane == 0) {
        atomicAdd(&s_cnt[0], c_label);
        atomicAdd(&s_cnt[1], c_closed);
    }
    __syncthreads();
    if (threadIdx.x < 2) w.tile_cnt[threadIdx.x * w.prob->tile_cap + t] = s_cnt[threadIdx.x];
    __syncthreads();
}

__global__ void __launch_bounds__(256) k_arrival_labels(Work w) {
    __shared__ uint32_t s_lab[AL_CAP];   // label position in the segment, closed flag
    __shared__ uint32_t s_cnt[2];
    const Prob &P = *w.prob;
    if (P.raw_fail > RAW_PARTS) return;
    const uint32_t nt = P.ntiles;
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) label_tile<256>(w, t, w.seg[w.tile_seg[t]], s_lab, s_cnt);
}

// Records in label order (and, streaming, the finalised hits and the carry).
// CTAs take contiguous tiles and sum the counts of their segment's earlier
// tiles themselves: a sum over 16384 counts costs less than a launch and the
// one-CTA scan it replaces.  Bound by the chain from a flag word to its
// record: small CTAs, so that more tiles are under way (64 Mi hits: 125 us with
// 256 threads, 110 with 128).
constexpr int AE = 128;

__device__ uint32_t emit_sum(const uint32_t *cnt, uint32_t n, uint32_t *s_red) {
    uint32_t m = 0;
#pragma unroll 8
    for (uint32_t i = threadIdx.x; i < n; i += AE) m += cnt[i];
    m = __reduce_add_sync(0xffffffffu, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = 0;
    for (int q = 0; q < AE / 32; ++q) m += s_red[q];
    return m;
}

// Exclusive prefix of the popcounts of a tile's 128 flag words.
__device__ uint32_t emit_prefix(uint32_t bits, uint32_t *s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t c = __popc(bits);
    uint32_t x = c;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) s_red[warp] = x;
    __syncthreads();
    x -= c;
    for (int q = 0; q < warp; ++q) x += s_red[q];
    return x;
}

__device__ void emit_totals(Seg &g, Prob &P, uint32_t n_clusters, uint32_t n_final) {
    g.n_clusters = n_clusters;
    g.n_final = n_final;
    g.n_open = g.n - n_final;
    if (n_clusters > g.out_cap) atomicOr(&P.err, E_CAP);
    if (!g.ss) return;
    StreamState &ss = *g.ss;
    if (g.n_open > g.carry_cap) atomicOr(&P.err, E_CAP);
    ss.n_carry = g.n_open <= g.carry_cap ? g.n_open : 0;
    ss.seen_max = g.seen_after;
    ss.has_seen = ss.has_seen || g.n != 0;
    if (g.close_mode == CLOSE_WM) ss.watermark = g.watermark;
}

// One tile's records, from record `rec` of its segment; streaming: its
// finalised hits from `fin` and its open ones, open_total in the segment.
template <int NT>
__device__ __forceinline__ void emit_tile(const Work &w, uint32_t t, const Seg &g, uint32_t begin, uint32_t end,
                                          uint32_t rec, uint32_t n_rec, uint32_t fin, uint32_t open_total,
                                          uint32_t *s_red, uint16_t *s_pos) {
    const uint32_t nwords = (end - begin + 31) >> 5;
    uint32_t bits = threadIdx.x < nwords ? w.flag_label[(begin >> 5) + threadIdx.x] : 0;
    uint32_t k = emit_prefix(bits, s_red);
    while (bits) {
        const int b = __ffs(bits) - 1;
        bits &= bits - 1;
        s_pos[k++] = (uint16_t)((threadIdx.x << 5) + b);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_rec; i += NT) {
        if (rec + i >= g.out_cap) break;
        const uint32_t pos = begin + s_pos[i];
        const uint32_t r = w.gpar[w.root_of[pos]];
        const RootSlot s = w.rslot[r];
        tpc_cluster out;
        out.label = gidx_of(g, pos - g.off);
        out.size = (int64_t)s.size;
        out.sum_tot = (int64_t)s.tot;
        out.first_toa = w.rfirst[r];
        // fp32 quotient of the exact integer sums: three roundings, each
        // at most 2^-24 relative (FP64 is a slow pipe on this GPU)
        const float sw = (float)s.tot;
        out.cx = (float)s.wx / sw;
        out.cy = (float)s.wy / sw;
        g.out_rec[rec + i] = out;
    }
    if (g.ss) {
        // a warp takes the 32 positions of a word together
        const bool fits = open_total <= g.carry_cap;
        const uint32_t cl = threadIdx.x < nwords ? w.flag_closed[(begin >> 5) + threadIdx.x] : 0;
        const uint32_t before = emit_prefix(cl, s_red);
        __syncthreads();   // the records have read s_pos
        if (threadIdx.x < nwords) s_pos[threadIdx.x] = (uint16_t)before;
        __syncthreads();
        const int lane = threadIdx.x & 31;
#pragma unroll 4
        for (uint32_t k = threadIdx.x >> 5; k < nwords; k += NT / 32) {
            const uint32_t pos = begin + 32 * k + lane, local = pos - g.off;
            const uint32_t bits = w.flag_closed[(begin >> 5) + k];
            const uint32_t closed = fin + s_pos[k] + __popc(bits & lanes_below());   // before this position
            if (pos >= end) continue;
            if ((bits >> lane) & 1u) {
                if (closed < g.out_cap) {
                    g.out_labels[closed] = w.lab_tmp[pos];
                    if (g.out_index) g.out_index[closed] = gidx_of(g, local);
                }
            } else if (fits) {
                const uint32_t dst = g.carry_cap - open_total + (local - closed);
                g.carry_out[dst] = g.hits[local];
                g.carry_gidx_out[dst] = gidx_of(g, local);
            }
        }
    }
}

__global__ void __launch_bounds__(AE) k_arrival_emit(Work w) {
    __shared__ uint32_t s_red[AE / 32];
    __shared__ uint16_t s_pos[TILE];
    __shared__ bool s_last;
    Prob &P = *w.prob;
    if (P.raw_fail > RAW_PARTS) return;
    const uint32_t nt = P.ntiles, cap = P.tile_cap, per = (nt + gridDim.x - 1) / gridDim.x;
    const uint32_t t0 = blockIdx.x * per, t1 = min(t0 + per, nt);
    const uint32_t *cnt = w.tile_cnt;
    if (blockIdx.x == 0) {   // segments without hits
        for (uint32_t s = threadIdx.x; s < P.nsegs; s += AE)
            if (w.seg[s].ntiles == 0) emit_totals(w.seg[s], P, 0, 0);
        __syncthreads();
    }
    uint32_t rec = 0, fin = 0, open_total = 0;
    const Seg *cur = nullptr;
    for (uint32_t t = t0; t < t1; ++t) {
        const uint32_t si = w.tile_seg[t];
        const Seg &g = w.seg[si];
        uint32_t begin, end;
        tile_range(g, t, begin, end);
        if (cur != &g) {
            cur = &g;
            rec = emit_sum(cnt + g.tile0, t - g.tile0, s_red);
            fin = emit_sum(cnt + cap + g.tile0, t - g.tile0, s_red);
            if (g.ss) open_total = g.n - emit_sum(cnt + cap + g.tile0, g.ntiles, s_red);
        }
        const uint32_t n_rec = cnt[t];
        emit_tile<AE>(w, t, g, begin, end, rec, n_rec, fin, open_total, s_red, s_pos);
        rec += n_rec;
        fin += cnt[cap + t];
        if (t + 1 == g.tile0 + g.ntiles && threadIdx.x == 0) emit_totals(w.seg[si], P, rec, fin);
        __syncthreads();   // s_pos is rewritten for the next tile
    }
    // the CTA that ends last sees every total and error bit
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&P.emitted, 1u) + 1u == gridDim.x;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    for (uint32_t s = threadIdx.x; s < P.nsegs; s += AE) write_info(w.seg[s], P);
}

// Whether the tile is done: every hit before h0 is earlier than its first by
// more than dt (first warp).
__device__ __forceinline__ void small_check(const Work &w, uint32_t t, bool linked) {
    if (threadIdx.x >= 32) return;
    const uint32_t lane = threadIdx.x;
    const ATile &info = w.atile[t];
    const uint32_t hc = linked ? info.h0 / A_STEP : 0u;   // chunks not looked at
    uint64_t m = 0;
    for (uint32_t i = lane; i < hc; i += 32) {
        const uint64_t c = w.atile[i / ACHUNKS].cmax[i % ACHUNKS];
        m = c > m ? c : m;
    }
    m = warp_max_u64(m);
    if (lane == 0) w.atile[t].redo = !linked || (hc && m >= info.lo) || info.nx > A_PAIRS;
}

// Tiles that are not done (between two barriers of the cluster).
__device__ __forceinline__ bool tiles_left(const Work &w, uint32_t nt) {
    bool any = false;
    for (uint32_t i = 0; i < nt; ++i) any |= *const_cast<volatile uint32_t *>(&w.atile[i].redo) != 0;
    return any;
}

constexpr int SORT_BITS = 10;
constexpr uint32_t DIGITS = 1u << SORT_BITS;
static_assert(DIGITS == (uint32_t)ST && DIGITS / 32 == 32, "a thread per digit, a lane per warp's sum");
static_assert(DIGITS * sizeof(uint32_t) <= A_PAIRS * sizeof(uint2), "a tile's counts fit its list of pairs");

struct SortShared {
    union {
        struct {
            uint16_t cnt[ST / 32][DIGITS];   // hits of each digit per warp, then those of the warps before
            uint32_t base[DIGITS];           // first place of this tile's hits of each digit
            uint32_t sum[32];
        };
        uint2 near[2 * TILE];                // after the sort: key and pixel of this tile's hits and of the tile before
    };
};
static_assert(sizeof(SortShared) <= sizeof(SmallShared), "in the place of a tile");

// One stable pass over SORT_BITS bits of the sort that the cluster's CTAs do
// together, each placing the entries of its tile.  hist: [tile][DIGITS].
__device__ __forceinline__ void sort_pass(const uint4 *src, uint4 *dst, uint32_t *hist, uint32_t t, uint32_t nt, uint32_t n,
                                          bool pixel, uint32_t shift, SortShared &S) {
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, first = t * TILE + warp * (TILE / (ST / 32)) + lane;
    constexpr int PER = TILE / ST;
    const bool mine = t < nt;
    uint4 e[PER];
    uint32_t rank[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r)
        if (mine && first + 32 * r < n) e[r] = src[first + 32 * r];
    for (uint32_t i = tid; i < sizeof(S.cnt) / sizeof(uint4); i += ST) reinterpret_cast<uint4 *>(S.cnt)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const bool valid = mine && first + 32 * r < n;
        const uint32_t d = valid ? ((pixel ? e[r].y : e[r].x) >> shift) & (DIGITS - 1) : DIGITS;
        const uint32_t same = __match_any_sync(0xffffffffu, d);
        if (valid) rank[r] = S.cnt[warp][d] + __popc(same & lanes_below());
        __syncwarp();
        if (valid && !(same & lanes_below())) S.cnt[warp][d] += (uint16_t)__popc(same);
        __syncwarp();
    }
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int q = 0; q < ST / 32; ++q) {
        const uint32_t c = S.cnt[q][tid];
        S.cnt[q][tid] = (uint16_t)run;
        run += c;
    }
    if (mine) hist[t * DIGITS + tid] = run;
    cluster.sync();
    uint32_t before = 0, all = 0;   // hits of this thread's digit in the tiles before, in all
#pragma unroll
    for (uint32_t q = 0; q < SMALL_TILES; ++q) {
        const uint32_t h = q < nt ? hist[q * DIGITS + tid] : 0u;
        before += q < t ? h : 0u;
        all += h;
    }
    uint32_t x = all;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) S.sum[warp] = x;
    __syncthreads();
    S.base[tid] = before + x - all + __reduce_add_sync(0xffffffffu, lane < warp ? S.sum[lane] : 0u);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        if (!mine || first + 32 * r >= n) continue;
        const uint32_t d = ((pixel ? e[r].y : e[r].x) >> shift) & (DIGITS - 1);
        dst[S.base[d] + S.cnt[warp][d] + rank[r]] = e[r];
    }
    cluster.sync();
}

// A small step whose tiles of positions are not all done: hits in no order,
// too many of them within dt or on one pixel.  The cluster sorts the step by
// pixel and time (in the place of the feature sums).  A hit is joined to the one
// before it on its pixel and, on its four neighbour pixels before it in raster
// order, to the latest at or before it and the earliest after it (the others
// within dt are joined to those along their pixel): the first of these becomes
// its parent, those that are within dt of another one beside them are left out,
// and the few that remain are joined in the forest over the sorted hits.  Any
// order, any density, any dt.  Bound by the latency of its stages on 16 SMs:
// 65,536 shuffled hits 193 us on the GPU, 27 of them the tiles of positions, 45
// the four passes of the sort, 34 the searches, 28 the features.  (Tiles of ToA
// intervals that each scanned all hits took 215, and where those held too many
// hits every tile was joined with every earlier one: 1480 at dt 384 with 4 hits a
// tick; all pairs joined at once in global memory 700.)  Out of line, so that its
// registers are not the usual path's.
__device__ __noinline__ void any_order(const Work &w, uint32_t t, uint32_t nt, SortShared &S) {
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const Seg &g = w.seg[0];
    const uint32_t tid = threadIdx.x, lane = tid & 31, n = g.n, W = g.width, H = g.height, dt = g.dt;
    const uint32_t begin = t < nt ? t * TILE : n, end = min(begin + (uint32_t)TILE, n);
    const uint64_t base = *reinterpret_cast<const volatile uint64_t *>(&g.toa_min);
    const uint64_t span = *reinterpret_cast<const volatile uint64_t *>(&g.toa_max) - base;
    const bool streaming = g.ss != nullptr;
    static_assert(sizeof(RootSlot) == 2 * sizeof(uint4), "the sort's two buffers");
    uint4 *src = reinterpret_cast<uint4 *>(w.rslot), *dst = src + (size_t)nt * TILE;   // key, pixel, position, ToT
    uint32_t *hist = reinterpret_cast<uint32_t *>(w.xlist);
    for (uint32_t i = begin + tid; i < end; i += ST) {
        const uint4 v = ld_hit(g.hits + i);
        const uint32_t pix = clamp_pix(v.x, W, H);
        src[i] = make_uint4((uint32_t)(hit_toa(v) - base), (pix >> 16) * W + (pix & 0xFFFFu), i, hit_tot(v));
    }
    cluster.sync();
    const uint32_t last_pixel = W * H - 1u;
    for (int pass = 0; pass < 8; ++pass) {
        const uint32_t shift = (uint32_t)(pass & 3) * SORT_BITS;
        if (!(pass < 4 ? span >> shift : last_pixel >> shift)) continue;
        sort_pass(src, dst, hist, t, nt, n, pass >= 4, shift, S);
        uint4 *x = src;
        src = dst;
        dst = x;
    }
    constexpr int PER = TILE / ST;
    uint32_t more[PER];        // neighbours to be joined later (bits as in `order`)
    uint32_t at01[PER], at23[PER];   // on each neighbour pixel, the first entry beyond the hit's key (two to a word)
    // In turn: the hit before (-), then of the pixels left, above left, above,
    // above right (0 to 3) the latest and the earliest after; neighbours beside one another.
    constexpr int order[9] = {-1, 2, 2, 0, 0, 1, 1, 3, 3};
    auto beside = [](int a, int b) { return a < 0 || b < 0 || a == b || a == 2 || b == 2 || (a < 2 && b < 2); };
    volatile uint32_t *par = w.gpar;   // (over the sorted hits)
    // The searches mostly end among this tile's hits and those of the tile before.
    const uint32_t near0 = begin > TILE ? begin - TILE : 0u;
    for (uint32_t i = near0 + tid; i < end; i += ST) S.near[i - near0] = *reinterpret_cast<const uint2 *>(src + i);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const uint32_t i = begin + r * ST + tid;
        more[r] = at01[r] = at23[r] = 0;
        if (i >= end) continue;
        const uint2 me = S.near[i - near0];
        const uint32_t y = me.y / W, x = me.y - y * W;
        uint32_t at[4], q[4];
        bool far = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = k == 0 ? x > 0 : y > 0 && (k == 1 ? x > 0 : k == 2 || x + 1 < W);
            q[k] = !in ? 0xFFFFFFFFu : k == 0 ? me.y - 1u : me.y - W + (uint32_t)k - 2u;
        }
        auto search = [&](uint32_t from, uint32_t to, auto entry) {   // first entry of [from, to) beyond the key, or to
            uint32_t len[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                at[k] = q[k] == 0xFFFFFFFFu ? 0u : from;
                len[k] = q[k] == 0xFFFFFFFFu ? 0u : to - from;
            }
            for (uint32_t longest = to - from; longest; longest >>= 1) {
                uint2 o[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) o[k] = len[k] ? entry(at[k] + (len[k] >> 1)) : make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool up = len[k] && (o[k].y < q[k] || (o[k].y == q[k] && o[k].x <= me.x));
                    const uint32_t half = len[k] >> 1;
                    at[k] += up ? half + 1u : 0u;
                    len[k] = up ? len[k] - half - 1u : half;
                }
            }
        };
        search(near0, i, [&](uint32_t a) { return S.near[a - near0]; });
#pragma unroll
        for (int k = 0; k < 4; ++k) far |= near0 && at[k] == near0;
        if (far) search(0u, i, [&](uint32_t a) { return *reinterpret_cast<const uint2 *>(src + a); });
        uint32_t key[9], found = 0;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            const int k = order[c];
            const bool after = c && c % 2 == 0;
            const uint32_t want = k < 0 ? me.y : q[k < 0 ? 0 : k], u = k < 0 ? i : at[k < 0 ? 0 : k];
            uint2 o = make_uint2(0, 0xFFFFFFFEu);
            const uint32_t j = after ? u : u - 1u;
            if (after || u) o = j >= near0 ? S.near[j - near0] : *reinterpret_cast<const uint2 *>(src + j);
            key[c] = o.x;
            if (o.y == want && (after ? o.x - me.x : me.x - o.x) <= dt) found |= 1u << c;
        }
        uint32_t parent = i, rest = 0;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            bool take = (found >> c) & 1u;
#pragma unroll
            for (int b = 0; b < c; ++b)
                if (beside(order[b], order[c])) take = take && !(((found >> b) & 1u) && absdiff(key[b], key[c]) <= dt);
            if (!take) continue;
            const int k = order[c];
            const uint32_t j = k < 0 ? i - 1u : at[k < 0 ? 0 : k] - (c % 2 ? 1u : 0u);
            if (parent == i) parent = j; else rest |= 1u << c;
        }
        par[i] = parent;
        more[r] = rest;
        at01[r] = at[0] | at[1] << 16;
        at23[r] = at[2] | at[3] << 16;
    }
    cluster.sync();
    // parents to roots, all in step (chains along a pixel or a track halve with every hop)
    uint32_t top[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) top[r] = begin + r * ST + tid < end ? par[begin + r * ST + tid] : 0u;
    for (bool any = true; any;) {
        any = false;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            if (begin + r * ST + tid >= end) continue;
            const uint32_t p = par[top[r]];
            if (p == top[r]) continue;
            any = true;
            top[r] = p;
            par[begin + r * ST + tid] = p;
        }
    }
    cluster.sync();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        while (more[r]) {
            const int c = __ffs(more[r]) - 1;
            more[r] &= more[r] - 1u;
            const int k = (c + 1) / 2;   // c 1, 2: above; 3, 4: left; 5, 6: above left; 7, 8: above right
            const uint32_t u = k == 1 ? at23[r] & 0xFFFFu : k == 2 ? at01[r] & 0xFFFFu : k == 3 ? at01[r] >> 16 : at23[r] >> 16;
            gunion(w.gpar, begin + r * ST + tid, u - (c % 2 ? 1u : 0u));
        }
    }
    uint4 e[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r)
        if (begin + r * ST + tid < end) e[r] = src[begin + r * ST + tid];
    cluster.sync();
#pragma unroll
    for (int r = 0; r < PER; ++r) {   // each hit's own features (only those at the roots are added to and read)
        const uint32_t i = begin + r * ST + tid;
        if (i >= end) continue;
        const uint32_t y = e[r].y / W, x = e[r].y - y * W, tot = e[r].w;
        uint4 *slot = reinterpret_cast<uint4 *>(w.rslot + i);
        slot[0] = make_uint4(tot, 0u, tot * x, 0u);
        slot[1] = make_uint4(tot * y, 0u, 1u, e[r].z);
        w.rfirst[i] = base + e[r].x;
        if (streaming) w.rlast[i] = base + e[r].x;
    }
    if (t < nt && tid == 0) {
        w.atile[t].nroots = 0;   // every hit points at its cluster's root
        w.atile[t].base = base;
    }
    cluster.sync();
    // The others' are added to their roots', a warp's hits of one cluster at once: a
    // lane sums up those of the lanes behind it in its group, twice as many with each
    // step (hit by hit 39 us for 65,536 hits, group after group 79).
#pragma unroll
    for (int r = 0; r < PER; ++r) top[r] = begin + r * ST + tid < end ? par[begin + r * ST + tid] : 0u;
    for (bool any = true; any;) {   // (nothing writes them any more)
        any = false;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const uint32_t p = par[top[r]];
            any |= p != top[r];
            top[r] = p;
        }
    }
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const uint32_t i = begin + r * ST + tid, root = top[r];
        const bool valid = i < end;
        const bool adds = valid && root != i;
        if (valid) {
            w.root_of[e[r].z] = root;
            if (w.rkey) w.rkey[e[r].z] = e[r].x;
        }
        const uint32_t y = e[r].y / W, x = e[r].y - y * W;
        uint32_t size = adds ? 1u : 0u, mn = adds ? e[r].z : 0xFFFFFFFFu, k0 = adds ? e[r].x : 0xFFFFFFFFu, k1 = adds ? e[r].x : 0u;
        uint32_t sum = adds ? e[r].w : 0u;
        unsigned long long sx = sum * x, sy = sum * y;   // (products below 2^32)
        const uint32_t same = __match_any_sync(0xffffffffu, adds ? root : 0xFFFFFFFFu), behind = same & ~(lanes_below() | 1u << lane);
        int next = adds && behind ? __ffs(behind) - 1 : 32;
        while (__any_sync(0xffffffffu, next < 32)) {
            const int from = next & 31;
            const bool has = next < 32;
            const uint32_t c1 = __shfl_sync(0xffffffffu, size, from), s1 = __shfl_sync(0xffffffffu, sum, from);
            const unsigned long long x1 = __shfl_sync(0xffffffffu, sx, from), y1 = __shfl_sync(0xffffffffu, sy, from);
            const uint32_t m1 = __shfl_sync(0xffffffffu, mn, from), a1 = __shfl_sync(0xffffffffu, k0, from),
                           b1 = __shfl_sync(0xffffffffu, k1, from);
            const int n1 = __shfl_sync(0xffffffffu, next, from);
            if (!has) continue;
            size += c1;
            sum += s1;
            sx += x1;
            sy += y1;
            mn = min(mn, m1);
            k0 = min(k0, a1);
            k1 = max(k1, b1);
            next = n1;
        }
        if (!adds || (same & lanes_below())) continue;
        RootSlot &d = w.rslot[root];
        atomicAdd(&d.tot, (unsigned long long)sum);
        atomicAdd(&d.wx, sx);
        atomicAdd(&d.wy, sy);
        atomicAdd(&d.size, size);
        atomicMin(&d.min, mn);
        atomicMin(reinterpret_cast<unsigned long long *>(&w.rfirst[root]), (unsigned long long)(base + k0));
        if (streaming) atomicMax(reinterpret_cast<unsigned long long *>(&w.rlast[root]), (unsigned long long)(base + k1));
    }
    cluster.sync();
}

// A whole small step in one launch: a cluster of SMALL_TILES CTAs or fewer,
// CTA t for tile t, with cluster barriers between the stages.  `seg`: the
// step's segment for callers that queue no copy of it (tpc_cluster_static);
// otherwise it is in w.seg.
__global__ void __launch_bounds__(ST, 1) k_arrival_step(Work w, Seg seg, uint32_t given, uint32_t tile_cap, uint64_t *counts,
                                                     uint32_t keep) {
    extern __shared__ __align__(16) unsigned char a_raw[];
    SmallShared &S = *reinterpret_cast<SmallShared *>(a_raw);
    __shared__ uint32_t s_red[ST / 32];
    __shared__ uint32_t s_cnt[2];
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const uint32_t t = blockIdx.x;
    const int tid = threadIdx.x;
    Prob &P = *w.prob;
    Seg &g = w.seg[0];
    if (t == 0 && tid == 0) {
        if (given) {
            g = seg;
            P.tile_cap = tile_cap;
            P.pos_cap = tile_cap * TILE;
        }
        uint32_t off = 0, tile = 0;
        setup_seg(g, off, tile);
        setup_prob(P, 1, tile, off, RAW_SMALL);
    }
    cluster.sync();
    const uint32_t nt = *const_cast<volatile uint32_t *>(&P.ntiles);
    const bool mine = t < nt;
    if (mine && tid == 0) w.tile_seg[t] = 0;
    const bool linked = mine && small_tile<ST>(w, t, S);
    if (mine && !linked) {   // clusters for the pairs of other tiles to be joined to, until any_order takes the step
        for (uint32_t i = t * TILE + tid; i < min((t + 1) * TILE, g.n); i += ST) w.root_of[i] = t * TILE;
        if (tid == 0) w.gpar[t * TILE] = t * TILE;
    }
    cluster.sync();
    if (mine) small_check(w, t, linked);
    if (linked) join_pairs<ST>(w, t, tid);
    if (t == 0 && tid == 0) seg_close(g, P);
    cluster.sync();
    if (tiles_left(w, nt)) any_order(w, t, nt, *reinterpret_cast<SortShared *>(a_raw));
    if (mine) root_tile<ST>(w, t, g.ss != nullptr);
    cluster.sync();
    if (mine) label_tile<ST>(w, t, g, reinterpret_cast<uint32_t *>(a_raw), s_cnt);
    cluster.sync();
    const uint32_t *cnt = w.tile_cnt, cap = P.tile_cap;
    if (mine) {
        uint32_t rec = 0, fin = 0, all = 0;   // of the tiles before, and (finalised) of all
        for (uint32_t i = 0; i < nt; ++i) {
            const uint32_t f = cnt[cap + i];
            if (i < t) { rec += cnt[i]; fin += f; }
            all += f;
        }
        uint32_t begin, end;
        tile_range(g, t, begin, end);
        emit_tile<ST>(w, t, g, begin, end, rec, cnt[t], fin, g.n - all, s_red, reinterpret_cast<uint16_t *>(a_raw));
        if (t + 1 == nt && tid == 0) emit_totals(g, P, rec + cnt[t], all);
    } else if (nt == 0 && t == 0 && tid == 0) {
        emit_totals(g, P, 0, 0);
    }
    if (tid == 0 && (nt ? t + 1 == nt : t == 0)) {
        write_info(g, P);
        if (counts) {   // tpc_cluster_static's result words
            counts[0] = g.n_clusters;
            counts[1] = P.err & keep;
        }
    }
}

// tpc_forest of a step on this path, whose union-find runs over tile clusters:
// the (ToA, input) order by the radix sort of the kept keys, every hit's parent
// its cluster's earliest hit.  What the step kept besides is written over: the
// keys become relative to its smallest ToA, and the slots' place holds each
// cluster's first sorted position and the parents.
__global__ void __launch_bounds__(256) k_forest_keys(Work w) {
    Prob &P = *w.prob;
    const Seg &g = w.seg[0];
    const uint32_t n = g.n, stride = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t *first = reinterpret_cast<uint32_t *>(w.slot);
    for (uint32_t i = i0; i < n; i += stride) {
        w.keys[0][i] = (uint32_t)(w.atile[i / TILE].base + w.rkey[i] - g.toa_min);
        w.vals[0][i] = i;
    }
    for (uint32_t c = i0; c < g.ntiles * TILE; c += stride) first[c] = 0xFFFFFFFFu;
    if (i0 == 0) {
        const uint64_t span = g.toa_max - g.toa_min;
        P.npasses = span ? (64u - __clzll((long long)span) + RADIX_BITS - 1u) / RADIX_BITS : 0u;
    }
}

__global__ void __launch_bounds__(256) k_forest_first(Work w) {
    const uint32_t *order = pick(w.vals, sorted_sel(*w.prob));
    uint32_t *first = reinterpret_cast<uint32_t *>(w.slot);
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < w.seg[0].n; s += gridDim.x * blockDim.x) {
        uint32_t *f = first + w.gpar[w.root_of[order[s]]];
        if (*reinterpret_cast<volatile uint32_t *>(f) > s) atomicMin(f, s);
    }
}

__global__ void __launch_bounds__(256) k_forest_parents(Work w, uint32_t *parent) {
    const uint32_t *order = pick(w.vals, sorted_sel(*w.prob));
    const uint32_t *first = reinterpret_cast<const uint32_t *>(w.slot);
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < w.seg[0].n; s += gridDim.x * blockDim.x)
        parent[s] = first[w.gpar[w.root_of[order[s]]]];
}

// Leaves the order in vals[npasses % 2].
void launch_forest(const Work &w, uint32_t *parent, const Launch &L) {
    k_forest_keys<<<L.fit(k_forest_keys, 256, 0), 256, 0, L.stream>>>(w);
    for (int pass = 0; pass < 4; ++pass) launch_radix_pass(w, pass, L);
    k_forest_first<<<L.fit(k_forest_first, 256, 0), 256, 0, L.stream>>>(w);
    k_forest_parents<<<L.fit(k_forest_parents, 256, 0), 256, 0, L.stream>>>(w, parent);
}

cudaError_t init_arrival_attributes() {
    cudaError_t e = cudaFuncSetAttribute(k_arrival_tile<AT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, A_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_arrival_tile<AT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, A_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_arrival_step, cudaFuncAttributeMaxDynamicSharedMemorySize, A_SMALL_SMEM);
    if (e == cudaSuccess)   // clusters of 16
        e = cudaFuncSetAttribute(k_arrival_step, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Links and the decision; `otherwise` (0: none) is the condition of what follows
// if they do not cover the step: 0 the same with parts, 1 the time-sorted path.
// parts: the tiles that did not fit.
void launch_arrival_link(const Work &w, cudaGraphConditionalHandle otherwise, bool parts, const Launch &L) {
    const int grid = L.fit(k_arrival_tile<AT, false>, AT, A_SMEM, G_LINK);
    if (parts) k_arrival_tile<AT, true><<<grid, AT, A_SMEM, L.stream>>>(w);
    else k_arrival_tile<AT, false><<<grid, AT, A_SMEM, L.stream>>>(w);
    L.mark(parts ? "k_arrival_tile_parts" : "k_arrival_tile");
    k_arrival_cross<<<L.fit(k_arrival_cross, AX, 0, G_LINK), AX, 0, L.stream>>>(w, otherwise, parts);
    L.mark("k_arrival_cross");
}

void launch_arrival_output(const Work &w, const Launch &L) {
    k_arrival_roots<<<L.fit(k_arrival_roots, 256, 0, G_ACC), 256, 0, L.stream>>>(w);
    L.mark("k_arrival_roots");
    k_arrival_labels<<<L.fit(k_arrival_labels, 256, 0, G_OUT), 256, 0, L.stream>>>(w);
    L.mark("k_arrival_labels");
    k_arrival_emit<<<L.fit(k_arrival_emit, AE, 0, G_OUT), AE, 0, L.stream>>>(w);
    L.mark("k_arrival_emit");
}

uint32_t arrival_step_cluster(uint32_t tiles) {
    uint32_t ctas = 1;
    while (ctas < tiles) ctas *= 2;
    return ctas;
}

static cudaLaunchConfig_t step_config(uint32_t ctas, cudaLaunchAttribute *a, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(ST);
    cfg.dynamicSmemBytes = A_SMALL_SMEM;
    cfg.stream = st;
    a->id = cudaLaunchAttributeClusterDimension;
    a->val.clusterDim.x = ctas;
    a->val.clusterDim.y = a->val.clusterDim.z = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    return cfg;
}

// A whole GPU holds clusters of SMALL_TILES CTAs of this size, one to an SM, in
// a GPC; a part of one (fewer SMs of a GPC for the process) may not.
int arrival_step_ctas() {
    for (uint32_t ctas = SMALL_TILES; ctas; ctas /= 2) {
        cudaLaunchAttribute a{};
        const cudaLaunchConfig_t cfg = step_config(ctas, &a, nullptr);
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_arrival_step, &cfg) == cudaSuccess && clusters > 0) return (int)ctas;
        cudaGetLastError();   // (too large is an answer)
    }
    return 0;
}

// A small step of at most `tiles` tiles; seg: its segment, or null if w.seg
// holds it already.
cudaError_t launch_arrival_step(const Work &w, const Seg *seg, uint32_t tiles, uint32_t tile_cap, uint64_t *counts,
                                uint32_t keep, const Launch &L) {
    cudaLaunchAttribute a{};
    const cudaLaunchConfig_t cfg = step_config(arrival_step_cluster(tiles), &a, L.stream);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_arrival_step, w, seg ? *seg : Seg{}, seg ? 1u : 0u, tile_cap, counts, keep);
    L.mark("k_arrival_step");
    return e;
}

}  // namespace tpc
