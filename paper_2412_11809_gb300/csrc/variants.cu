// Variants (iii)(b) and (iii)(c) of the cluster definition (paper Section 2),
// read as the time sweep of Algorithm 1: in (ToA, index) order a hit merges
// every still-open cluster with a member on one of its 9 pixels; (b) open =
// last ToA >= toa - dt, (c) open = first ToA >= toa - dt.  Both start from
// the components of variant (a), already in the global forest.
//
// (c): every (c) join is an (a) edge (the joined member lies between the
// cluster's first hit and the new hit, so within dt of it), hence (c)
// clusters split (a) components and each component can be swept on its own.
// Components are grouped by a stable radix sort on their root (keeping ToA
// order inside); one thread sweeps each component, looking back only over
// hits within dt (older members belong to clusters that are closed).
//
// (b): a closed cluster never reopens, so at any moment every open cluster
// with a member on pixel p also contains the latest hit on p (that hit joined
// it on arrival), and a (b) cluster is open exactly on [first, last + dt].
// The sweep's result is therefore the least partition, reached from the (a)
// components by merging, in which hit h is joined to L = the latest earlier
// hit on each of its 9 pixels whenever toa(h) <= last(group(L)) + dt.
// Rounds apply that rule: the first to every hit's 9 latest neighbours, the
// later ones to the edges still open, with the groups' last ToA kept at the
// roots by the unions (a lagging value only postpones a merge) and
// recomputed exactly when a round merges nothing; the partition is final
// after a round without merges on exact values.  The rounds join (a)
// components, each by a dense id; per-pixel timelines come from a stable
// radix sort of the hits by pixel.
#include <cooperative_groups.h>

#include "tpc_internal.cuh"

namespace tpc {

__device__ __forceinline__ bool adjacent_v(uint32_t a, uint32_t b) {
    const int dx = (int)(a & 0xFFFFu) - (int)(b & 0xFFFFu);
    const int dy = (int)(a >> 16) - (int)(b >> 16);
    return dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1;
}

// grouping keys: (c) the (a) root of each sorted position; (b) its pixel id
__global__ void __launch_bounds__(256) k_var_keys(Work w, VarWork v, int by_pixel) {
    const Prob &P = *w.prob;
    const uint32_t nt = P.ntiles;
    const uint32_t *sroot = pick(w.keys, sorted_sel(P) ^ 1u);
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) {
        const Seg &g = w.seg[w.tile_seg[t]];
        uint32_t begin, end;
        tile_range(g, t, begin, end);
        for (uint32_t s = begin + threadIdx.x; s < end; s += blockDim.x) {
            const uint32_t pix = w.spix[s];
            v.k[0][s] = by_pixel ? (pix >> 16) * g.width + (pix & 0xFFFFu) : sroot[s];
            v.v[0][s] = s;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *v.prob = P;
        // as many digits as the largest pixel id (< 2^20) or root has
        const uint32_t top = (by_pixel ? w.seg[0].width * w.seg[0].height : w.seg[0].off + w.seg[0].n) - 1u;
        v.prob->npasses = top ? (32 - __clz(top) + RADIX_BITS - 1) / RADIX_BITS : 0;
    }
}

// find with path halving, for a forest owned by one thread
__device__ __forceinline__ uint32_t seq_find(uint32_t *par, uint32_t x) {
    while (par[x] != x) {
        par[x] = par[par[x]];
        x = par[x];
    }
    return x;
}

// Threads and hits staged by the CTA sweep (below) of components that outgrow
// the warps' windows.
constexpr int BIG_THREADS = 512;
constexpr uint32_t BIG_CAP = 8192;
constexpr int BIG_SMEM = 3 * BIG_CAP * (int)sizeof(uint32_t);

// (c): one warp per component of the root-grouped order (components are
// contiguous there, in ToA order).  The sweep is sequential over the
// component's hits, but a hit needs few lookups: when a hit lands on a pixel
// it joins every open cluster with a member there, so of the clusters with a
// member on a pixel only the one of its latest hit can be open.
//   up to 32 hits      everything in registers: lane j holds hit j and its
//                      root; a step tests all earlier hits at once.
//   up to SW_CAP hits  staged in shared memory with a hash table from pixel
//                      to its latest hit: nine lanes look up the nine pixels
//                      of a hit, and three hits are taken per step; the
//                      second and third count only if they touch neither the
//                      pixels nor the clusters of those before (else they
//                      are taken again).
//   longer             (listed by k_static_long) two warps: one looks up the
//                      neighbours of 32 hits ahead, which no join changes,
//                      the other joins; a sliding window of the last hits,
//                      which the first writes out behind them.
// A lone warp's chain over the longest component sets the time of the step (its
// instructions follow one another at four to five cycles each), so what can
// be taken off that chain is: 8 M hits at 2.5 Ghits/s, longest component 6,544
// hits, from every earlier hit within dt tested 32 at a time (9.9 ms, and 1.9
// for components outgrowing a window of 512) to the table (2.4 ms) to the two
// warps (1.4 ms; 1.2 with what leaves the window written by the looking one and
// the next step's lookups read a step ahead).  It runs beside the sweep of the
// others (0.9 ms alone): 1.3 ms for both.
constexpr int SW_WARPS = 8;
constexpr uint32_t SW_CAP = 512;
constexpr uint32_t SW_TAB = 1024;
constexpr uint32_t SW_CHUNK = 32;
constexpr uint32_t LW_CAP = 1024;        // hits in the rings of a long component's sweep
constexpr uint32_t LW_WIN = LW_CAP - 64; // ... in the window (the looking warp is 32 to 64 ahead)
constexpr uint32_t LW_TAB = 4096;
constexpr uint32_t LW_REBUILD = 960;     // hits between two rebuilds of the window's table
constexpr uint32_t LW_FIRST = 2048;      // components this long are started first
constexpr int LW_CTAS = 3;               // per SM: room beside them for the other components' sweep
// Table entry: pixel id << 11 | index mod 2048.  Bit 31 is set in none, so no
// entry is the empty one (with 12 bits of index the last pixel of a sensor of
// 2^20 pixels had one that was).
constexpr uint32_t HASH_BITS = 11, HASH_AGE = (1u << HASH_BITS) - 1u;
constexpr uint32_t HASH_EMPTY = 0xFFFFFFFFu;
constexpr uint32_t NO_ROOT = 0xFFFFFFFFu;
static_assert(MAX_PIXELS <= 1u << (31 - HASH_BITS), "pixel ids leave the top bit clear");
// entries of a window's table: hits since its rebuild and those put back then, so lookups always end
static_assert(LW_REBUILD + 32 + LW_CAP < LW_TAB && LW_REBUILD + 32 + LW_CAP < HASH_AGE && 2 * SW_CAP <= SW_TAB,
              "free entries, unambiguous indices");

struct HashSweep {
    uint32_t key[SW_CAP];
    uint32_t tab[SW_TAB];
    uint16_t up[SW_CAP];   // distance to the parent, 0 at a root
};

// Sweep of component [q0, q0 + n), n <= SW_CAP, of the grouped order.
__device__ void sweep_hashed(HashSweep &S, const uint32_t *skey, const uint32_t *spix, const uint32_t *gv,
                             uint32_t *parent, uint32_t q0, uint32_t n, uint32_t dt, uint32_t W, uint32_t H, int lane) {
    const uint32_t bits = 32 - __clz((int)(2 * n - 1));   // table: at least twice the hits
    const uint32_t tsize = 1u << bits, tmask = tsize - 1u, shift = 32u - bits;
    for (uint32_t i = lane; i < tsize / 4; i += 32)
        reinterpret_cast<uint4 *>(S.tab)[i] = make_uint4(HASH_EMPTY, HASH_EMPTY, HASH_EMPTY, HASH_EMPTY);
    const int g = lane / 9, d = lane - 9 * g;      // hit of the step and its neighbour pixel (lanes 27..31 idle)
    const int dx = d % 3 - 1, dy = d / 3 - 1;
    auto root_of = [&](uint32_t x) -> uint32_t {
        volatile uint16_t *up = S.up;
        for (uint32_t k = up[x]; k; k = up[x]) x -= k;
        return x;
    };
    // the next 32 hits are on their way while 32 are swept
    uint32_t k = 0, p = 0, k1 = 0, p1 = 0;
    if ((uint32_t)lane < n) {
        const uint32_t se = gv[q0 + lane];
        k1 = skey[se];
        p1 = spix[se];
    }
    uint32_t se2 = 32u + lane < n ? gv[q0 + 32 + lane] : 0u;
    for (uint32_t base = 0; base < n; base += 32) {
        const uint32_t e = base + lane, cnt = n - base < 32u ? n - base : 32u;
        k = k1;
        p = p1;
        if (e + 32 < n) {
            k1 = skey[se2];
            p1 = spix[se2];
        }
        if (e + 64 < n) se2 = gv[q0 + e + 64];
        if (e < n) {
            S.key[e] = k;
            S.up[e] = 0;
        }
        __syncwarp();
        for (uint32_t c = 0; c < cnt;) {
            const uint32_t at = c + (g < 3 ? g : 0), i = base + at;
            const bool act = g < 3 && at < cnt;
            const uint32_t ki = __shfl_sync(0xffffffffu, k, at & 31), pi = __shfl_sync(0xffffffffu, p, at & 31);
            const uint32_t pa = __shfl_sync(0xffffffffu, p, c & 31), pb = __shfl_sync(0xffffffffu, p, (c + 1) & 31),
                           pc = __shfl_sync(0xffffffffu, p, (c + 2) & 31);
            const int x = (int)(pi & 0xFFFFu) + dx, y = (int)(pi >> 16) + dy;
            const bool in = act && x >= 0 && x < (int)W && y >= 0 && y < (int)H;
            const uint32_t pid = (uint32_t)y * W + (uint32_t)x;
            uint32_t slot = pid * 0x9E3779B1u >> shift, r = NO_ROOT;
            if (in) {
                uint32_t seen = S.tab[slot];
                while (seen != HASH_EMPTY && seen >> HASH_BITS != pid) {
                    slot = (slot + 1) & tmask;
                    seen = S.tab[slot];
                }
                if (seen != HASH_EMPTY) {
                    const uint32_t j = i - ((i - seen) & HASH_AGE);   // the pixel's latest hit
                    if (ki - S.key[j] <= dt) {
                        const uint32_t rj = root_of(j);
                        if (ki - S.key[rj] <= dt) {   // its cluster is open
                            r = rj;
                            S.up[j] = (uint16_t)(j - rj);   // (each pixel's latest hit is another)
                        }
                    }
                }
            }
            // hits 1 and 2 of the step must not touch what 0 and 1 change: pixels
            // nearby, a cluster, the same free table entry
            const uint32_t m0 = __reduce_min_sync(0xffffffffu, g == 0 ? r : NO_ROOT);   // the earliest root of
            const uint32_t m1 = __reduce_min_sync(0xffffffffu, g == 1 ? r : NO_ROOT);   // each hit's open clusters
            const uint32_t m2 = __reduce_min_sync(0xffffffffu, g == 2 ? r : NO_ROOT);
            const uint32_t same = __match_any_sync(0xffffffffu, r);
            const uint32_t clash = __ballot_sync(0xffffffffu, r != NO_ROOT && (same & ((1u << (9 * (g < 3 ? g : 0))) - 1u)));
            const uint32_t s0 = __shfl_sync(0xffffffffu, slot, 4), s1 = __shfl_sync(0xffffffffu, slot, 13),
                           s2 = __shfl_sync(0xffffffffu, slot, 22);
            uint32_t take = 1;
            if (c + 1 < cnt && !adjacent_v(pa, pb) && !(clash & (0x1FFu << 9)) && s0 != s1) {
                take = 2;
                if (c + 2 < cnt && !adjacent_v(pa, pc) && !adjacent_v(pb, pc) && !(clash & (0x1FFu << 18)) && s0 != s2 &&
                    s1 != s2)
                    take = 3;
            }
            const uint32_t m = g == 0 ? m0 : g == 1 ? m1 : m2;
            __syncwarp();
            if (act && (uint32_t)g < take) {
                if (r != NO_ROOT && r != m) S.up[r] = (uint16_t)(r - m);
                if (d == 4) {
                    if (m != NO_ROOT) S.up[i] = (uint16_t)(i - m);
                    S.tab[slot] = pid << HASH_BITS | (i & HASH_AGE);
                }
            }
            __syncwarp();
            c += take;
        }
    }
    for (uint32_t j = lane; j < n; j += 32) parent[gv[q0 + j]] = gv[q0 + root_of(j)];
}

// A long component: warp 1 runs a chunk of 32 hits ahead of warp 0 and lists
// each hit's neighbours, the latest hit within dt on each of its nine pixels:
// from the table (lane = hit), then from the earlier ones of the 32.  Warp 0
// joins, up to three hits at a time.  The rings hold the last LW_CAP hits: a
// (c) cluster spans at most dt, so while every hit within dt of the hit being
// swept is in the window, a hit that leaves it belongs to a cluster closed for
// every later hit: its root is final and goes to global memory (cpar), where
// finds that reach it read it.
struct LongSweep {
    uint32_t tab[LW_TAB];
    uint32_t key[LW_CAP], place[LW_CAP], pid[LW_CAP];   // by index mod LW_CAP; sorted position, pixel id
    uint16_t up[LW_CAP];       // distance to the parent, 0 at a root (at most the hits within dt, so at most the window)
    uint16_t back[2][32 * 9];  // of a chunk's hits: distance to the latest hit within dt per pixel, 0: none
    uint32_t next1[2], next2[2];   // hits beside the hit one, two before
    uint32_t job;
};

// Chunk at `base` (lane = hit).
__device__ __forceinline__ void long_look(LongSweep &S, uint32_t base, uint32_t n, uint32_t se, uint32_t k, uint32_t p,
                                          uint32_t dt, uint32_t W, uint32_t H, uint32_t &built, int lane) {
    constexpr uint32_t tmask = LW_TAB - 1u, shift = 32u - 12u;
    static_assert(LW_TAB == 1u << 12, "table size");
    const uint32_t e = base + lane;
    const int x = (int)(p & 0xFFFFu), y = (int)(p >> 16);
    const uint32_t pid = (uint32_t)y * W + (uint32_t)x;
    uint16_t *back = S.back[(base >> 5) & 1u];
    // an entry of a pixel: an empty slot, or the pixel's own with an earlier hit
    auto put = [&](uint32_t id, uint32_t i, uint32_t now) {
        uint32_t slot = id * 0x9E3779B1u >> shift, seen = S.tab[slot];
        while (true) {
            if (seen != HASH_EMPTY && seen >> HASH_BITS != id) {
                slot = (slot + 1) & tmask;
                seen = S.tab[slot];
                continue;
            }
            if (seen != HASH_EMPTY && ((now - seen) & HASH_AGE) <= ((now - i) & HASH_AGE)) return;
            const uint32_t was = atomicCAS(&S.tab[slot], seen, id << HASH_BITS | (i & HASH_AGE));
            if (was == seen) return;
            seen = was;
        }
    };
    if (base == 0 || base - built >= LW_REBUILD) {   // only hits within dt are still of use
        const uint32_t k0 = __shfl_sync(0xffffffffu, k, 0);
        for (uint32_t i = lane; i < LW_TAB / 4; i += 32)
            reinterpret_cast<uint4 *>(S.tab)[i] = make_uint4(HASH_EMPTY, HASH_EMPTY, HASH_EMPTY, HASH_EMPTY);
        __syncwarp();
        for (uint32_t i = (base > LW_WIN ? base - LW_WIN : 0u) + lane; i < base; i += 32)
            if (k0 - S.key[i % LW_CAP] <= dt) put(S.pid[i % LW_CAP], i, base);
        built = base;
    }
    if (e < n) {
        S.key[e % LW_CAP] = k;
        S.place[e % LW_CAP] = se;
        S.pid[e % LW_CAP] = pid;
        S.up[e % LW_CAP] = 0;
    }
    __syncwarp();
    uint32_t slot[9], seen[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int nx = x + q % 3 - 1, ny = y + q / 3 - 1;
        const bool in = e < n && nx >= 0 && nx < (int)W && ny >= 0 && ny < (int)H;
        slot[q] = ((uint32_t)ny * W + (uint32_t)nx) * 0x9E3779B1u >> shift;
        seen[q] = in ? S.tab[slot[q]] : HASH_EMPTY;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const uint32_t want = (uint32_t)(y + q / 3 - 1) * W + (uint32_t)(x + q % 3 - 1);
        while (seen[q] != HASH_EMPTY && seen[q] >> HASH_BITS != want) {
            slot[q] = (slot[q] + 1) & tmask;
            seen[q] = S.tab[slot[q]];
        }
        uint32_t a = 0;
        if (seen[q] != HASH_EMPTY) {
            a = (e - seen[q]) & HASH_AGE;
            if (a >= LW_WIN || k - S.key[(e - a) % LW_CAP] > dt) a = 0;   // (what has left the window is older than dt)
        }
        back[lane * 9 + q] = (uint16_t)a;
    }
    __syncwarp();
    const uint32_t cnt = n - base < 32u ? n - base : 32u;
    for (uint32_t j = 0; j + 1 < cnt; ++j) {
        const uint32_t pj = __shfl_sync(0xffffffffu, p, j), kj = __shfl_sync(0xffffffffu, k, j);
        const int ax = (int)(pj & 0xFFFFu) - x + 1, ay = (int)(pj >> 16) - y + 1;
        if ((uint32_t)lane > j && (unsigned)ax < 3u && (unsigned)ay < 3u && k - kj <= dt)
            back[lane * 9 + ay * 3 + ax] = (uint16_t)(lane - j);
    }
    const uint32_t u1 = __shfl_up_sync(0xffffffffu, p, 1), u2 = __shfl_up_sync(0xffffffffu, p, 2);
    const uint32_t next1 = __ballot_sync(0xffffffffu, adjacent_v(u1, p)), next2 = __ballot_sync(0xffffffffu, adjacent_v(u2, p));
    if (lane == 0) {
        S.next1[(base >> 5) & 1u] = next1;
        S.next2[(base >> 5) & 1u] = next2;
    }
    if (e < n) put(pid, e, base + 32);
    __syncwarp();
}

// Root of x in the window, or an index before it (whose cluster is closed).
__device__ __forceinline__ uint32_t long_root(LongSweep &S, uint32_t x, uint32_t lo) {
    volatile uint16_t *up = S.up;
    uint32_t k = x >= lo ? up[x % LW_CAP] : 0u;
    while (k) {
        x -= k;
        k = x >= lo ? up[x % LW_CAP] : 0u;
    }
    return x;
}

// Before the chunk at `base` is joined the 32 oldest hits leave the window.
// They and so their roots are older than dt: no join changes them any more,
// and the looking warp can write their parents while the other goes on.
// false: the window is too small.
__device__ __forceinline__ bool long_leave(LongSweep &S, uint32_t base, const uint32_t *gv, uint32_t *parent, uint32_t *cpar,
                                           uint32_t q0, uint32_t dt, bool &crowded, int lane) {
    const uint32_t k0 = S.key[base % LW_CAP];
    if (base >= SW_CAP && __any_sync(0xffffffffu, k0 - S.key[(base - SW_CAP + lane) % LW_CAP] <= dt)) crowded = true;
    if (base < LW_WIN) return true;
    const uint32_t j = base - LW_WIN + lane, lo = base - LW_WIN;
    if (__any_sync(0xffffffffu, k0 - S.key[j % LW_CAP] <= dt)) return false;
    uint32_t r = long_root(S, j, lo);
    const uint32_t to = r < lo ? (r = *reinterpret_cast<volatile uint32_t *>(&cpar[r]), gv[q0 + r]) : S.place[r % LW_CAP];
    __syncwarp();
    cpar[j] = r;
    parent[S.place[j % LW_CAP]] = to;
    __syncwarp();
    return true;
}

// First hit of the window while the chunk at `base` is joined.
__device__ __forceinline__ uint32_t long_first(uint32_t base) { return base >= LW_WIN ? base - LW_WIN + 32 : 0u; }

// Joins the hits of the chunk at `base`; lo: the first hit of the window.
__device__ __forceinline__ void long_join(LongSweep &S, uint32_t base, uint32_t n, uint32_t dt, uint32_t lo, int lane) {
    // lanes 0..26: hit g of the step and its neighbour pixel d; 27..29: hit g itself
    const int g = lane < 27 ? lane / 9 : lane - 27;
    const bool looks = lane < 27;
    const uint32_t cnt = n - base < 32u ? n - base : 32u;
    const uint16_t *back = S.back[(base >> 5) & 1u] + lane;   // (hit * 9 + d = (hit - g) * 9 + lane)
    // hits that must wait for the one before them, the two before them (or do not exist)
    const uint32_t none = cnt < 32u ? 0xFFFFFFFFu << cnt : 0u;
    const uint32_t next1 = S.next1[(base >> 5) & 1u] | none, next2 = S.next2[(base >> 5) & 1u] | next1;
    const uint32_t below = (1u << (9 * (looks ? g : 0))) - 1u;
    auto ahead = [&](uint32_t c) -> uint32_t { return looks && c + g < cnt ? back[c * 9] : 0u; };
    uint32_t b = ahead(0);
    for (uint32_t c = 0; c < cnt;) {
        const uint32_t b1 = ahead(c + 1), b2 = ahead(c + 2), b3 = ahead(c + 3);   // the next step's, whatever this one takes
        const uint32_t at = c + g, i = base + at;
        const bool wait1 = c + 1 >= 32u || ((next1 >> (c + 1)) & 1u), wait2 = c + 2 >= 32u || ((next2 >> (c + 2)) & 1u);
        uint32_t r = NO_ROOT;
        const uint32_t ki = S.key[i % LW_CAP];
        if (b) {
            const uint32_t rj = long_root(S, i - b, lo);
            if (rj >= lo && ki - S.key[rj % LW_CAP] <= dt) r = rj;   // its cluster is open
        }
        // hits 1 and 2 of the step must not touch what 0 and 1 change:
        // pixels nearby, a cluster
        const uint32_t m0 = __reduce_min_sync(0xffffffffu, g == 0 ? r : NO_ROOT);   // the earliest root of
        const uint32_t m1 = __reduce_min_sync(0xffffffffu, g == 1 ? r : NO_ROOT);   // each hit's open clusters
        const uint32_t m2 = __reduce_min_sync(0xffffffffu, g == 2 ? r : NO_ROOT);
        const uint32_t same = __match_any_sync(0xffffffffu, r);
        const uint32_t clash = __ballot_sync(0xffffffffu, r != NO_ROOT && (same & below));
        const bool two = !wait1 && !(clash & (0x1FFu << 9)), three = two && !wait2 && !(clash & (0x1FFu << 18));
        const uint32_t m = g == 0 ? m0 : g == 1 ? m1 : m2;
        const uint32_t x = looks ? r : i;   // a cluster joined, or the hit
        if (m != NO_ROOT && x != NO_ROOT && x != m && (g == 0 || (g == 1 && two) || (g == 2 && three)))
            S.up[x % LW_CAP] = (uint16_t)(x - m);
        __syncwarp();
        b = three ? b3 : two ? b2 : b1;
        c += three ? 3 : two ? 2 : 1;
    }
}

// Up to 32 hits: lane j holds hit j (key, pixel) and its root.
__device__ __forceinline__ void sweep_registers(const uint32_t *skey, const uint32_t *spix, const uint32_t *gv,
                                                uint32_t *parent, uint32_t q0, uint32_t n, uint32_t dt, int lane) {
    uint32_t se = 0, k = 0, p = 0, root = lane;
    if ((uint32_t)lane < n) {
        se = gv[q0 + lane];
        k = skey[se];
        p = spix[se];
    }
    for (uint32_t i = 1; i < n; ++i) {
        const uint32_t ki = __shfl_sync(0xffffffffu, k, i), pi = __shfl_sync(0xffffffffu, p, i);
        const uint32_t kr = __shfl_sync(0xffffffffu, k, root);
        const bool joins = (uint32_t)lane < i && adjacent_v(pi, p) && ki - kr <= dt;   // open: so is the hit itself within dt
        const uint32_t open = __reduce_or_sync(0xffffffffu, joins ? 1u << root : 0u);   // the roots joined
        if (open && ((open >> root) & 1u || (uint32_t)lane == i)) root = __ffs(open) - 1;
    }
    const uint32_t sr = __shfl_sync(0xffffffffu, se, root);
    if ((uint32_t)lane < n) parent[se] = sr;
}

// Lists the components of more than SW_CAP hits: a component starts at q and
// reaches beyond q + SW_CAP; its end by doubling steps, then halving ones.
__global__ void __launch_bounds__(256) k_static_long(Work w, VarWork v) {
    const uint32_t sel = v.prob->npasses & 1u;
    const uint32_t *gk = pick(v.k, sel);
    const Seg &g = w.seg[0];
    const uint32_t first = g.off, last = g.off + g.n;
    for (uint32_t q = first + blockIdx.x * blockDim.x + threadIdx.x; q < last; q += gridDim.x * blockDim.x) {
        const uint32_t key = gk[q];
        if ((q != first && gk[q - 1] == key) || last - q <= SW_CAP || gk[q + SW_CAP] != key) continue;
        uint32_t in = q + SW_CAP, step = SW_CAP;   // gk[in] == key
        while (last - in > step && gk[in + step] == key) { in += step; step *= 2; }
        uint32_t out = last - in > step ? in + step : last;
        while (out - in > 1) {
            const uint32_t mid = in + (out - in) / 2;
            if (gk[mid] == key) in = mid; else out = mid;
        }
        const uint32_t n = in + 1 - q;
        atomicAdd(&v.changed[0], 1u);
        // the list holds all of them (each has > SW_CAP hits), the longest from its end
        if (n >= LW_FIRST) v.big[v.big_cap - 1 - atomicAdd(&v.changed[5], 1u)] = make_uint2(q, n);
        else v.big[atomicAdd(&v.changed[6], 1u)] = make_uint2(q, n);
    }
}

__global__ void __launch_bounds__(SW_WARPS * 32) k_static_sweep(Work w, VarWork v) {
    extern __shared__ __align__(16) unsigned char sweep_raw[];
    const uint32_t *skey = pick(w.keys, sorted_sel(*w.prob));
    const uint32_t sel = v.prob->npasses & 1u;
    const uint32_t *gk = pick(v.k, sel), *gv = pick(v.v, sel);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    HashSweep &S = reinterpret_cast<HashSweep *>(sweep_raw)[warp];
    const Seg &g = w.seg[0];
    const uint32_t first = g.off, last = g.off + g.n, dt = g.dt, W = g.width, H = g.height;
    const uint32_t nchunks = (g.n + SW_CHUNK - 1) / SW_CHUNK;
    while (true) {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(v.work, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= nchunks) break;
        const uint32_t q = first + c * SW_CHUNK + lane;
        uint32_t starts = __ballot_sync(0xffffffffu, q < last && (q == first || gk[q] != gk[q - 1]));
        while (starts) {
            const uint32_t q0 = first + c * SW_CHUNK + (__ffs(starts) - 1);
            starts &= starts - 1;
            // the component's end: the first grouped position with another root
            const uint32_t key0 = gk[q0];
            uint32_t n = 0;
            for (uint32_t p0 = q0 + 1;; p0 += 32) {
                const uint32_t p = p0 + lane;
                const uint32_t stop = __ballot_sync(0xffffffffu, p >= last || gk[p] != key0);
                if (stop) { n = p0 + (__ffs(stop) - 1) - q0; break; }
                if (p0 - q0 > SW_CAP) break;   // listed by k_static_long (n = 0)
            }
            if (n == 1) {
                if (lane == 0) w.parent[gv[q0]] = gv[q0];
            } else if (n && n <= 32) {
                sweep_registers(skey, w.spix, gv, w.parent, q0, n, dt, lane);
            } else if (n && n <= SW_CAP) {
                sweep_hashed(S, skey, w.spix, gv, w.parent, q0, n, dt, W, H, lane);
            }
            __syncwarp();   // the staging is rewritten for the next component
        }
    }
}

__global__ void __launch_bounds__(64) k_static_sweep_long(Work w, VarWork v) {
    extern __shared__ __align__(16) unsigned char sweep_raw[];
    LongSweep &S = *reinterpret_cast<LongSweep *>(sweep_raw);
    const uint32_t *skey = pick(w.keys, sorted_sel(*w.prob));
    const uint32_t *gv = pick(v.v, v.prob->npasses & 1u);
    const int lane = threadIdx.x & 31;
    const bool looks = threadIdx.x >= 32;
    const Seg &g = w.seg[0];
    const uint32_t nfirst = v.changed[5], nlong = v.changed[0], dt = g.dt, W = g.width, H = g.height;
    while (true) {
        if (threadIdx.x == 0) S.job = atomicAdd(&v.changed[4], 1u);
        __syncthreads();
        const uint32_t job = S.job;
        if (job >= nlong) break;
        // the longest ones first: a chain started late would end alone
        const uint2 comp = job < nfirst ? v.big[v.big_cap - 1 - job] : v.big[job - nfirst];
        const uint32_t q0 = comp.x, n = comp.y;
        uint32_t *cpar = v.cpar + q0;
        uint32_t built = 0, se1 = 0, k1 = 0, p1 = 0, se2 = 0;
        bool crowded = false, kept = true;
        if (looks) {
            se1 = gv[q0 + lane];   // (n > SW_CAP)
            k1 = skey[se1];
            p1 = w.spix[se1];
            se2 = gv[q0 + 32 + lane];
        }
        for (uint32_t base = 0; base < n + 32; base += 32) {
            if (looks) {
                if (base < n) {
                    const uint32_t e = base + lane, se = se1, k = k1, p = p1;
                    se1 = se2;   // the next hits are on their way meanwhile
                    if (e + 32 < n) {
                        k1 = skey[se1];
                        p1 = w.spix[se1];
                    }
                    if (e + 64 < n) se2 = gv[q0 + e + 64];
                    if (base) kept = long_leave(S, base - 32, gv, w.parent, cpar, q0, dt, crowded, lane);
                    long_look(S, base, n, se, k, p, dt, W, H, built, lane);
                } else {
                    kept = long_leave(S, base - 32, gv, w.parent, cpar, q0, dt, crowded, lane);
                }
            } else if (base) {
                long_join(S, base - 32, n, dt, long_first(base - 32), lane);
            }
            kept = __syncthreads_and(kept);
            if (!kept) break;
        }
        if (looks) {
            if (lane == 0) {
                if (crowded) {   // diagnostics
                    atomicAdd(&v.changed[1], 1u);
                    if (n > BIG_CAP) atomicAdd(&v.changed[2], 1u);
                }
                if (!kept) v.over[atomicAdd(&v.changed[3], 1u)] = comp;
            }
        } else if (kept) {
            const uint32_t lo = long_first((n - 1) / 32 * 32);
            for (uint32_t j = lo + lane; j < n; j += 32) {   // the hits still in the window
                const uint32_t r = long_root(S, j, lo);
                w.parent[S.place[j % LW_CAP]] = r < lo ? gv[q0 + *reinterpret_cast<volatile uint32_t *>(&cpar[r])] : S.place[r % LW_CAP];
            }
        }
        __syncthreads();   // the rings are rewritten for the next component
    }
}

template <bool STAGED>
struct SweepView {
    const uint32_t *sk, *sp;   // staged keys and pixels (STAGED)
    uint32_t *sc;              // parent per component index (staged or global)
    const uint32_t *skey, *spix, *gv;
    uint32_t q;                // first grouped position of the component
    __device__ uint32_t key(uint32_t i) const { return STAGED ? sk[i] : skey[gv[q + i]]; }
    __device__ uint32_t pix(uint32_t i) const { return STAGED ? sp[i] : spix[gv[q + i]]; }
    __device__ uint32_t find(uint32_t x) const {   // path halving
        volatile uint32_t *c = sc;
        while (true) {
            const uint32_t p = c[x];
            if (p == x) return x;
            const uint32_t gp = c[p];
            if (gp == p) return p;
            c[x] = gp;
            x = gp;
        }
    }
};

// (c): components whose hits within dt outgrew the warp's window.  One CTA
// per component, the component staged whole in dynamic shared memory (up to
// BIG_CAP hits; from global memory beyond): the same sweep, with each
// step's candidates (the earlier hits within dt) spread over the CTA's
// threads instead of one warp's lanes, the earliest open root found by a
// shared-memory minimum.
template <bool STAGED>
__device__ void sweep_block(const SweepView<STAGED> &V, uint32_t n, uint32_t dt, uint32_t *s_min) {
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) V.sc[i] = i;
    if (threadIdx.x < 2) s_min[threadIdx.x] = 0xFFFFFFFFu;
    __syncthreads();
    uint32_t it = 0;   // iterations so far: s_min[it & 1] collects this one's minimum
    for (uint32_t i = 1; i < n; ++i) {
        const uint32_t ki = V.key(i), pi = V.pix(i);
        uint32_t root = 0xFFFFFFFFu;   // the earliest open root joined so far (the same in every thread)
        for (uint32_t base = 0; base < i; base += blockDim.x, ++it) {
            const bool valid = base + threadIdx.x < i;
            const uint32_t j = valid ? i - 1 - base - threadIdx.x : 0;
            const bool in = valid && ki - V.key(j) <= dt;
            uint32_t r = 0xFFFFFFFFu;
            if (in && adjacent_v(pi, V.pix(j))) {
                const uint32_t rj = V.find(j);
                if (ki - V.key(rj) <= dt) r = rj;   // that cluster is still open
            }
            uint32_t *mn = s_min + (it & 1u);
            if (r != 0xFFFFFFFFu) atomicMin(mn, r);
            const bool any_in = __syncthreads_or(in);
            const uint32_t m = *reinterpret_cast<volatile uint32_t *>(mn);
            if (threadIdx.x == 0) s_min[(it + 1) & 1u] = 0xFFFFFFFFu;   // read by nobody until the next barrier
            if (m != 0xFFFFFFFFu) {
                const uint32_t target = m < root ? m : root;
                if (r != 0xFFFFFFFFu && r != target) V.sc[r] = target;
                if (threadIdx.x == 0 && root != 0xFFFFFFFFu && root != target) V.sc[root] = target;
                root = target;
            }
            __syncthreads();
            if (!any_in) { ++it; break; }   // keys only fall further back
        }
        if (threadIdx.x == 0 && root != 0xFFFFFFFFu) V.sc[i] = root;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(BIG_THREADS) k_static_sweep_big(Work w, VarWork v) {
    extern __shared__ uint32_t big_raw[];
    __shared__ uint32_t s_min[2];
    const uint32_t *skey = pick(w.keys, sorted_sel(*w.prob));
    const uint32_t *gv = pick(v.v, v.prob->npasses & 1u);
    const uint32_t dt = w.seg[0].dt, nbig = v.changed[3];
    for (uint32_t k = blockIdx.x; k < nbig; k += gridDim.x) {
        const uint2 job = v.over[k];
        const uint32_t q0 = job.x, n = job.y;
        if (n <= BIG_CAP) {
            uint32_t *sk = big_raw, *sp = big_raw + BIG_CAP, *sc = big_raw + 2 * BIG_CAP;
            for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
                const uint32_t si = gv[q0 + i];
                sk[i] = skey[si];
                sp[i] = w.spix[si];
            }
            __syncthreads();
            const SweepView<true> V{sk, sp, sc, skey, w.spix, gv, q0};
            sweep_block(V, n, dt, s_min);
            for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) w.parent[gv[q0 + i]] = gv[q0 + V.find(i)];
        } else {
            const SweepView<false> V{nullptr, nullptr, v.cpar + q0, skey, w.spix, gv, q0};
            sweep_block(V, n, dt, s_min);
            for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) w.parent[gv[q0 + i]] = gv[q0 + V.find(i)];
        }
        __syncthreads();   // the staging is rewritten for the next component
    }
}

constexpr int SW_SMEM = SW_WARPS * (int)sizeof(HashSweep);
constexpr int LW_SMEM = (int)sizeof(LongSweep);

cudaError_t init_variants_attributes() {
    cudaError_t e = cudaFuncSetAttribute(k_static_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, SW_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_static_sweep_long, cudaFuncAttributeMaxDynamicSharedMemorySize, LW_SMEM);
    // the two sweeps run side by side on the SMs: one split of L1 and shared memory for both
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_static_sweep, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_static_sweep_long, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    return e == cudaSuccess
               ? cudaFuncSetAttribute(k_static_sweep_big, cudaFuncAttributeMaxDynamicSharedMemorySize, BIG_SMEM) : e;
}

// (b): where each pixel's timeline begins in the order the pixel sort left
// (single segment): a lower bound per pixel, whose first steps all threads
// share.  A histogram by atomics and its scan in one CTA took 510 us for 8 M
// hits and 229,376 pixels; this takes 16.
__global__ void __launch_bounds__(256) k_pixel_starts(Work w, VarWork v) {
    const Seg &g = w.seg[0];
    const uint32_t *tk = pick(v.k, v.prob->npasses & 1u) + g.off;
    const uint32_t np = g.width * g.height;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q <= np; q += gridDim.x * blockDim.x) {
        uint32_t a = 0, b = g.n;   // first entry of a pixel >= q
        while (a < b) {
            const uint32_t mid = (a + b) >> 1;
            if (tk[mid] < q) a = mid + 1; else b = mid;
        }
        v.pix_start[q] = a;
    }
}

// (b) takes the (a) components as its units: they get dense ids in the
// order of their roots (sorted positions), and the rounds find and join on
// a forest over those ids (cpar_d, with each group's last key at its root
// in clast), a tenth of the hits' count, mostly held in L2, instead of on
// the forest over sorted positions.  A component's own last key (clast0)
// is fixed.  The roots of the sorted positions after the (a) links are
// those k_sorted_roots left in the idle radix buffer.

// Components per tile: the roots among its positions.
__global__ void __launch_bounds__(256) k_comp_count(Work w, VarWork v) {
    __shared__ uint32_t s_cnt;
    const uint32_t nt = w.prob->ntiles;
    const uint32_t *sroot = pick(w.keys, sorted_sel(*w.prob) ^ 1u);
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) {
        const Seg &g = w.seg[w.tile_seg[t]];
        uint32_t begin, end;
        tile_range(g, t, begin, end);
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
        uint32_t c = 0;
        for (uint32_t s = begin + threadIdx.x; s < end; s += blockDim.x) c += sroot[s] == s ? 1u : 0u;
        c = __reduce_add_sync(0xffffffffu, c);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_cnt, c);
        __syncthreads();
        if (threadIdx.x == 0) v.tcnt[t] = s_cnt;
        __syncthreads();   // s_cnt is reset for the next tile
    }
}

// One CTA: exclusive scan of the tile counts; the total is the id count.
__global__ void __launch_bounds__(1024) k_comp_scan(Work w, VarWork v) {
    __shared__ uint32_t s_warp[32];
    const uint32_t nt = w.prob->ntiles;
    const uint32_t per = (nt + blockDim.x - 1) / blockDim.x;
    const uint32_t i0 = threadIdx.x * per;
    uint32_t local = 0;
    for (uint32_t i = i0; i < i0 + per && i < nt; ++i) local += v.tcnt[i];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = local;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t run = x - local;
    for (int q = 0; q < warp; ++q) run += s_warp[q];
    for (uint32_t i = i0; i < i0 + per && i < nt; ++i) {
        v.tbase[i] = run;
        run += v.tcnt[i];
    }
    if (threadIdx.x == blockDim.x - 1) *v.ncomp = run;
}

// Dense ids in root order: a root's id is the roots before it.  Each id
// starts as its own group.
__global__ void __launch_bounds__(256) k_comp_ids(Work w, VarWork v) {
    constexpr int ITEMS = TILE / 256;
    __shared__ uint32_t s_pre[TILE / 32];   // roots per 32 positions, then their exclusive prefix
    const uint32_t nt = w.prob->ntiles;
    const uint32_t *sroot = pick(w.keys, sorted_sel(*w.prob) ^ 1u);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t t = blockIdx.x; t < nt; t += gridDim.x) {
        const Seg &g = w.seg[w.tile_seg[t]];
        uint32_t begin, end;
        tile_range(g, t, begin, end);
        uint32_t m[ITEMS];
#pragma unroll
        for (int q = 0; q < ITEMS; ++q) {   // position begin + q * 256 + threadIdx.x: word q * 8 + warp
            const uint32_t s = begin + q * 256 + threadIdx.x;
            m[q] = __ballot_sync(0xffffffffu, s < end && sroot[s] == s);
            if (lane == 0) s_pre[q * 8 + warp] = __popc(m[q]);
        }
        __syncthreads();
        if (warp == 0) {   // 128 words, 4 per lane
            uint32_t c[4], sum = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) { c[k] = s_pre[lane * 4 + k]; sum += c[k]; }
            uint32_t x = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            uint32_t run = x - sum;
#pragma unroll
            for (int k = 0; k < 4; ++k) { s_pre[lane * 4 + k] = run; run += c[k]; }
        }
        __syncthreads();
        const uint32_t base = v.tbase[t];
#pragma unroll
        for (int q = 0; q < ITEMS; ++q) {
            if (!((m[q] >> lane) & 1u)) continue;
            const uint32_t s = begin + q * 256 + threadIdx.x;
            const uint32_t c = base + s_pre[q * 8 + warp] + __popc(m[q] & ((1u << lane) - 1u));
            v.cid_at[s] = c;
            v.croot[c] = s;
            v.cpar_d[c] = c;
            v.clast0[c] = 0;
        }
        __syncthreads();   // s_pre is rewritten for the next tile
    }
}

// Each component's last key; only hits that could raise the stored value
// issue the atomic (a long component would serialise on one address).
__global__ void __launch_bounds__(256) k_comp_last(Work w, VarWork v) {
    const Seg &g = w.seg[0];
    const uint32_t *skey = pick(w.keys, sorted_sel(*w.prob));
    const uint32_t *sroot = pick(w.keys, sorted_sel(*w.prob) ^ 1u);
    for (uint32_t s = g.off + blockIdx.x * blockDim.x + threadIdx.x; s < g.off + g.n; s += gridDim.x * blockDim.x) {
        const uint32_t c = v.cid_at[sroot[s]], k = skey[s];
        if (*reinterpret_cast<volatile uint32_t *>(&v.clast0[c]) < k) atomicMax(&v.clast0[c], k);
    }
}

// Before a full round: each hit's state, (id of its group's root, that
// group's last key, its sorted position, its key), first in position order
// (coalesced but for the ids, whose roots lie near), then gathered into
// pixel-timeline order, one 16-byte read per hit.  The groups and last keys
// are those of the moment (the last keys exact at the first round, lagging
// later): every rule applied to them is one the sweep applies.  flat: the
// first round, where every group is one component (and starts here).
__global__ void __launch_bounds__(256) k_position_state(Work w, VarWork v, int flat) {
    const Seg &g = w.seg[0];
    const uint32_t *skey = pick(w.keys, sorted_sel(*w.prob));
    const uint32_t *sroot = pick(w.keys, sorted_sel(*w.prob) ^ 1u);
    for (uint32_t s = g.off + blockIdx.x * blockDim.x + threadIdx.x; s < g.off + g.n; s += gridDim.x * blockDim.x) {
        const uint32_t r = sroot[s], c0 = v.cid_at[r];
        uint32_t c = c0, last;
        if (flat) {
            last = v.clast0[c0];
            if (r == s) v.clast[c0] = last;
        } else {
            c = gfind(v.cpar_d, c0);
            last = *reinterpret_cast<volatile uint32_t *>(&v.clast[c]);
        }
        v.pstate[s] = make_uint4(c, last, s, skey[s]);
    }
}

__global__ void __launch_bounds__(256) k_timeline_state(Work w, VarWork v) {
    const Seg &g = w.seg[0];
    const uint32_t *tl = pick(v.v, v.prob->npasses & 1u) + g.off;
    uint4 *T = v.tline + g.off;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < g.n; j += gridDim.x * blockDim.x)
        T[j] = v.pstate[tl[j]];
}

// The result on the hits' forest: each component's root hooked under its
// group's root (an earlier position: ids follow the roots' order).
__global__ void __launch_bounds__(256) k_comp_parents(Work w, VarWork v) {
    const uint32_t n = *v.ncomp;
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        const uint32_t f = gfind(v.cpar_d, c);
        if (f != c) w.parent[v.croot[c]] = v.croot[f];
    }
}

// (b) with the groups' last keys kept at their roots during the unions: when
// root b is hooked under a, a's last key takes b's (atomicMax).  A value can
// lag behind its group's (a concurrent hook of a loses it), never exceed it,
// so every union made on it is one the sweep makes; an exact recomputation
// when a round merges nothing decides the end.
__device__ __forceinline__ bool gunion_last(uint32_t *parent, uint32_t *glast, uint32_t a, uint32_t b) {
    while (true) {
        a = gfind(parent, a);
        b = gfind(parent, b);
        if (a == b) return false;
        if (a > b) { const uint32_t t = a; a = b; b = t; }
        if (atomicCAS(parent + b, b, a) == b) {
            const uint32_t lb = *reinterpret_cast<volatile uint32_t *>(&glast[b]);
            if (*reinterpret_cast<volatile uint32_t *>(&glast[a]) < lb) atomicMax(&glast[a], lb);
            return true;
        }
    }
}

// Append the warp's open edges (a node of h's group, a node of its
// neighbour's group, h's key) to list `out` (one atomic per warp); on
// overflow the list is marked and the next round takes every hit again.  Whether
// the list is full by now.
__device__ __forceinline__ bool push_edges(const VarWork &v, int out, unsigned long long *listed, uint32_t *flags, bool keep,
                                           uint32_t a, uint32_t b, uint32_t key) {
    uint2 *list = pick(v.edges, out);
    uint32_t *keys = pick(v.ekey, out);
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    if (!m) return false;
    const int lane = threadIdx.x & 31;
    unsigned long long base = 0;   // 64 bits: a full round can push more than 2^32 edges
    if (lane == __ffs(m) - 1) base = atomicAdd(listed, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
    const unsigned long long slot = base + __popc(m & ((1u << lane) - 1u));
    if (keep) {
        if (slot < v.edge_cap) {
            list[slot] = make_uint2(a, b);
            keys[slot] = key;
        } else {
            flags[1] = 1u;
        }
    }
    return base >= v.edge_cap;
}

// The first entries at or after position s of G timelines [at, at + n)
// (ascending positions), into at: binary searches in step, so that a load of
// each is in flight.
template <int G>
__device__ __forceinline__ void lane_bounds(const uint32_t *tl, uint32_t (&at)[G], uint32_t (&n)[G], uint32_t s) {
    uint32_t longest = 0;
#pragma unroll
    for (int k = 0; k < G; ++k) longest = max(longest, n[k]);
    for (; longest; longest >>= 1) {   // a search of n entries ends after as many steps as n has bits
        uint32_t e[G];
#pragma unroll
        for (int k = 0; k < G; ++k) e[k] = n[k] ? tl[at[k] + (n[k] >> 1)] : 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const uint32_t half = n[k] >> 1;
            const bool up = e[k] < s;
            at[k] += up ? half + 1 : 0u;
            n[k] = up ? n[k] - half - 1 : half;
        }
    }
}

// A round over every hit's 9 latest neighbours (the first round, and any
// round after an overflow of the edge list), in pixel-timeline order, with
// their state from the snapshot: the snapshot root starts the find of the
// neighbour's group, its last key decides most rules without a read.  Merges
// what the rule allows and lists the rest, as (node of h's group, root of the
// neighbour's group).
//
// Bound by the latency of its dependent loads (a search in each neighbour's
// timeline, the state found, the finds), so a lane takes its eight neighbour
// pixels through the searches and the first step of the finds together.  The
// warp searching for its 32 hits at once, one neighbour after another, took
// 1480 us for 8 M hits on 448x512 pixels, where 32 entries of the timelines
// span two pixels or more; together in groups of two, four and eight: 1199,
// 1078 and 943 us (416 of them the searches).  Not kept: warp-wide searches of
// four neighbours at once (1075), and second steps up, last keys and unions
// also taken together (1066, with twice the edges listed).
// A warp that finds the list full lists no more: on streams where nearly every
// edge stays open the one counter's atomics took longer than all else (8 M hits
// at 0.25 a tick, dt 128: 10.0 ms a call with three full rounds, 5.7 so; reading
// the list's mark instead cost as much).
constexpr int FIRST_THREADS = 128, FIRST_G = 8;

__global__ void __launch_bounds__(FIRST_THREADS, 5) k_global_first(Work w, VarWork v) {
    const Seg &g = w.seg[0];
    const uint32_t W = g.width, H = g.height, n = g.n, dt = g.dt;
    const uint32_t sel = v.prob->npasses & 1u;
    const uint32_t *tl = pick(v.v, sel) + g.off;   // sorted positions grouped by pixel
    const uint32_t *tk = pick(v.k, sel) + g.off;   // their pixel ids
    const uint4 *T = v.tline + g.off;
    auto state = [T](uint32_t at) { return __ldg(reinterpret_cast<const uint2 *>(T + at)); };   // (id, last key)
    const uint32_t *ps = v.pix_start;
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    bool changed = false, full = false;   // full: the list was, when this warp last listed an edge
    for (uint32_t i0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32u; i0 < n; i0 += warps * 32u) {
        const uint32_t i = i0 + (uint32_t)lane;
        const bool valid = i < n;
        const uint4 me = valid ? T[i] : make_uint4(0, 0, 0, 0);   // group id, its last key, position, key
        const uint32_t p = valid ? tk[i] : 0xFFFFFFFFu;
        uint32_t rh = me.x;   // an id of h's group, moved towards its root as the round goes
        // Any two nodes found equal are in one group (groups only merge), so
        // stale roots only cost a find; the last keys used are lower bounds of
        // the group's (nb.y: its part at the snapshot), so the rule never
        // merges more than the sweep.  up: a step up from nb.x.
        auto join = [&](const uint2 &nb, uint32_t up, bool has) {
            int r = 0;
            uint32_t rl = up;
            if (has && rl != rh) {
                rl = gfind(v.cpar_d, rl);
                if (rl != rh) rh = gfind(v.cpar_d, rh);   // h's group may have been joined since
                if (rl != rh) {
                    bool ok = (uint64_t)me.w <= (uint64_t)nb.y + dt;
                    if (!ok) ok = (uint64_t)me.w <= (uint64_t)*reinterpret_cast<volatile uint32_t *>(&v.clast[rl]) + dt;
                    if (ok) {
                        if (gunion_last(v.cpar_d, v.clast, rh, rl)) r = 1;
                        rh = min(rh, rl);
                    } else {
                        r = 2;
                    }
                }
            }
            changed |= r == 1;
            full |= push_edges(v, 0, v.ecount, v.changed, r == 2 && !full, rh, rl, me.w);
        };
        {   // its own pixel: the entry before
            const bool has = valid && i > ps[p];
            const uint2 nb = has ? state(i - 1) : make_uint2(0, 0);
            join(nb, nb.x, has);
        }
        const uint32_t py = p / W, px = p - py * W;
        {
            uint32_t q0[FIRST_G], at[FIRST_G], len[FIRST_G];   // each neighbour's timeline: begin, first entry after h
#pragma unroll
            for (int k = 0; k < FIRST_G; ++k) {
                const int d = k + (k >= 4), x = (int)px + d % 3 - 1, y = (int)py + d / 3 - 1;
                const bool inside = valid && x >= 0 && x < (int)W && y >= 0 && y < (int)H;
                const uint32_t q = (uint32_t)y * W + (uint32_t)x;
                at[k] = q0[k] = inside ? ps[q] : 0u;
                len[k] = inside ? ps[q + 1] - q0[k] : 0u;
            }
            lane_bounds<FIRST_G>(tl, at, len, me.z);
            uint2 nb[FIRST_G];
            uint32_t up[FIRST_G];
#pragma unroll
            for (int k = 0; k < FIRST_G; ++k) nb[k] = at[k] > q0[k] ? state(at[k] - 1) : make_uint2(0, 0);
#pragma unroll
            for (int k = 0; k < FIRST_G; ++k)
                up[k] = at[k] > q0[k] ? *reinterpret_cast<volatile uint32_t *>(&v.cpar_d[nb[k].x]) : 0u;
#pragma unroll
            for (int k = 0; k < FIRST_G; ++k) join(nb[k], up[k], at[k] > q0[k]);
        }
    }
    if (__syncthreads_or(changed) && threadIdx.x == 0) atomicOr(&v.changed[0], 1u);
}

// A round over the `count` open edges of list `in`, those left open listed in
// the other: both ends' first steps up the forest at once.
__device__ __forceinline__ void list_round(const VarWork &v, int in, unsigned long long count, uint32_t dt, uint32_t *flags,
                                           unsigned long long *listed) {
    const uint2 *list = pick(v.edges, in);
    const uint32_t *keys = pick(v.ekey, in);
    const uint32_t cnt = count < v.edge_cap ? (uint32_t)count : v.edge_cap;
    bool changed = false;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t e0 = blockIdx.x * blockDim.x; e0 < cnt; e0 += stride) {
        const uint32_t e = e0 + threadIdx.x;
        const bool valid = e < cnt;
        uint2 ed = make_uint2(0, 0);
        uint32_t ks = 0, ux = 0, uy = 0;
        if (valid) {   // (written by other SMs in the rounds before: not from L1)
            ed = __ldcg(list + e);
            ks = __ldcg(keys + e);
            ux = __ldcg(v.cpar_d + ed.x);
            uy = __ldcg(v.cpar_d + ed.y);
        }
        int r = 0;
        uint32_t rh = ed.x, rl = ed.y;
        if (valid) {
            rh = ux == ed.x ? ux : gfind(v.cpar_d, ux);
            rl = uy == ed.y ? uy : gfind(v.cpar_d, uy);
            if (rl != rh) {   // the rule on the group's last key as it stands (a lower bound)
                const uint32_t last = *reinterpret_cast<volatile uint32_t *>(&v.clast[rl]);
                if ((uint64_t)ks <= (uint64_t)last + dt) r = gunion_last(v.cpar_d, v.clast, rh, rl) ? 1 : 0;
                else r = 2;
            }
        }
        changed |= r == 1;
        push_edges(v, 1 - in, listed, flags, r == 2, rh, rl, ks);
    }
    if (__syncthreads_or(changed) && threadIdx.x == 0) atomicOr(flags, 1u);
}

// The rounds over the open edges after a full round (cooperative: a barrier of
// the grid between rounds), until the partition is closed under the rule: the
// last one merged nothing on exact last keys.  When a round merges nothing on
// keys that may lag, the groups' last keys are made exact: reset at the roots,
// then each id's own raised into its root's.  Ends early if a list overflowed
// (the host starts another full round).  Flags and counts of a round rotate
// through three slots, so that one is cleared while one is read and one written.
// One launch for all of them: launch by launch, the host looking at the flags
// after each, six rounds of 8 M hits took some 25 us each beside their work.
constexpr uint32_t MAX_ROUNDS = 4096;

__global__ void __launch_bounds__(256) k_global_rounds(Work w, VarWork v, uint32_t exact) {
    cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    const uint32_t dt = w.seg[0].dt, n = *v.ncomp, stride = gridDim.x * blockDim.x;
    const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x;
    volatile uint32_t *flags = v.changed;
    volatile unsigned long long *counts = v.ecount;
    uint32_t rounds = 0, checks = 0, slot = 0, over = 0;
    int in = 0;
    const unsigned long long open = counts[0];
    while (true) {   // (every thread takes the same way)
        over = flags[2 * slot + 1];
        if (flags[2 * slot]) {
            exact = 0;
        } else if (exact) {
            over = 0;
            break;
        } else {
            for (uint32_t c = first; c < n; c += stride)
                if (__ldcg(v.cpar_d + c) == c) v.clast[c] = 0;
            grid.sync();
            for (uint32_t c = first; c < n; c += stride) {
                const uint32_t f = gfind(v.cpar_d, c), k = v.clast0[c];
                if (*reinterpret_cast<volatile uint32_t *>(&v.clast[f]) < k) atomicMax(&v.clast[f], k);
            }
            grid.sync();
            exact = 1;
            ++checks;
        }
        if (over || rounds == MAX_ROUNDS) break;
        const uint32_t next = slot == 2 ? 0 : slot + 1, after = next == 2 ? 0 : next + 1;
        if (first == 0) {
            flags[2 * after] = flags[2 * after + 1] = 0;
            counts[after] = 0;
        }
        list_round(v, in, counts[slot], dt, v.changed + 2 * next, v.ecount + next);
        ++rounds;
        in = 1 - in;
        slot = next;
        grid.sync();
    }
    if (first == 0) {
        uint32_t *status = v.changed + ROUNDS_STATUS;
        status[0] = rounds;
        status[1] = checks;
        status[2] = over;
        status[3] = exact;
        status[4] = open < v.edge_cap ? (uint32_t)open : v.edge_cap;
        status[5] = rounds == MAX_ROUNDS;
        // with another full round to come, nothing for the features and outputs behind this one
        w.prob->ntiles = over ? 0u : v.prob->ntiles;
        w.prob->nsegs = over ? 0u : v.prob->nsegs;
    }
}

void launch_components(const Work &w, const VarWork &v, const Launch &L) {
    k_comp_count<<<L.fit(k_comp_count, 256, 0), 256, 0, L.stream>>>(w, v);
    k_comp_scan<<<1, 1024, 0, L.stream>>>(w, v);
    k_comp_ids<<<L.fit(k_comp_ids, 256, 0), 256, 0, L.stream>>>(w, v);
    k_comp_last<<<L.fit(k_comp_last, 256, 0), 256, 0, L.stream>>>(w, v);
    L.mark("k_components");
}

void launch_comp_parents(const Work &w, const VarWork &v, const Launch &L) {
    k_comp_parents<<<L.fit(k_comp_parents, 256, 0), 256, 0, L.stream>>>(w, v);
    L.mark("k_comp_parents");
}

// A full round into list 0 and the rounds over the edges it leaves open.  flat:
// the first one, where each group is one component; exact: the last keys are
// exact (they are then).
cudaError_t launch_global_rounds(const Work &w, const VarWork &v, bool flat, bool exact, const Launch &L) {
    cudaMemsetAsync(v.changed, 0, 6 * sizeof(uint32_t), L.stream);
    cudaMemsetAsync(v.ecount, 0, 3 * sizeof(unsigned long long), L.stream);
    k_position_state<<<L.fit(k_position_state, 256, 0), 256, 0, L.stream>>>(w, v, flat);
    k_timeline_state<<<L.fit(k_timeline_state, 256, 0), 256, 0, L.stream>>>(w, v);
    L.mark("k_timeline_state");
    k_global_first<<<L.fit(k_global_first, FIRST_THREADS, 0), FIRST_THREADS, 0, L.stream>>>(w, v);
    L.mark("k_global_first");
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(L.fit(k_global_rounds, 256, 0));
    cfg.blockDim = dim3(256);
    cfg.stream = L.stream;
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeCooperative;
    a.val.cooperative = 1;
    cfg.attrs = &a;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_global_rounds, w, v, exact ? 1u : 0u);
    L.mark("k_global_rounds");
    return e;
}

void launch_variant_keys(const Work &w, const VarWork &v, int by_pixel, const Launch &L) {
    k_var_keys<<<L.fit(k_var_keys, 256, 0), 256, 0, L.stream>>>(w, v, by_pixel);
    L.mark(by_pixel ? "k_var_keys_pixel" : "k_var_keys_root");
}

Work variant_view(const Work &w, const VarWork &v) {
    Work wv = w;
    wv.keys[0] = v.k[0];
    wv.keys[1] = v.k[1];
    wv.vals[0] = v.v[0];
    wv.vals[1] = v.v[1];
    wv.prob = v.prob;
    return wv;
}

// The sweep of the long components, a few chains, and that of all others,
// which fills the SMs, run side by side.  The long ones follow on the step's own
// stream, so that they are on the SMs before the others, which wait for an
// event; the other way around they started when the others ended (8 M hits of
// the 2.5 Ghits/s stream: 2.1 ms for both, 1.5 this way, 1.3 with the shorter
// chain).
cudaError_t launch_static_sweep(const Work &w, const VarWork &v, const Launch &L, const SideStream &side) {
    cudaMemsetAsync(v.work, 0, sizeof(uint32_t), L.stream);
    cudaMemsetAsync(v.changed, 0, 7 * sizeof(uint32_t), L.stream);
    k_static_long<<<L.fit(k_static_long, 256, 0), 256, 0, L.stream>>>(w, v);
    L.mark("k_static_long");
    cudaError_t e = cudaEventRecord(side.fork, L.stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side.stream, side.fork, 0);
    if (e != cudaSuccess) return e;
    const int fit = L.fit(k_static_sweep_long, 64, LW_SMEM), few = (L.sms > 0 ? L.sms : 1) * LW_CTAS;
    k_static_sweep_long<<<fit < few ? fit : few, 64, LW_SMEM, L.stream>>>(w, v);
    k_static_sweep<<<L.fit(k_static_sweep, SW_WARPS * 32, SW_SMEM), SW_WARPS * 32, SW_SMEM, side.stream>>>(w, v);
    e = cudaEventRecord(side.join, side.stream);
    k_static_sweep_big<<<L.fit(k_static_sweep_big, BIG_THREADS, BIG_SMEM), BIG_THREADS, BIG_SMEM, L.stream>>>(w, v);
    L.mark("k_static_sweep_long");
    const cudaError_t e2 = cudaStreamWaitEvent(L.stream, side.join, 0);   // (the step goes on after both)
    L.mark("k_static_sweep");
    return e == cudaSuccess ? e2 : e;
}

void launch_pixel_timelines(const Work &w, const VarWork &v, const Launch &L) {
    k_pixel_starts<<<L.fit(k_pixel_starts, 256, 0), 256, 0, L.stream>>>(w, v);
    L.mark("k_pixel_starts");
}

}  // namespace tpc
