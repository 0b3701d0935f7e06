// Device code of the step kernels (instantiated by gk_kernels.cu, per frame,
// gk_rollout.cu, multi-frame, gk_worklist.cu and gk_team.cu): one group of
// lanes advances one Generals.io game -- a warp, or for two-player games on
// small boards a half (two games per warp) or, in multi-frame launches, a
// quarter of one (four per warp); in small batches the warps of a CTA.
//
// Per game and step (paper Section IV) the group
//   1. stages the board (int16 armies, int8 owners, int8 terrain) in shared
//      memory with cp.async 16-byte copies;
//   2. resolves the players' moves one after another on its first lane
//      (Sec. IV-D, IV-E), with a group-wide pass for the land transfer of a
//      captured general;
//   3. applies growth (Sec. IV-C) while dot products turn the board into
//      bitsets (ownership per player, army >= 2) and total lands and armies;
//   4. decides termination and reward (Sec. III) and regenerates finished
//      games (Sec. IV-A);
//   5. widens the (team) ownership bitsets by a column to either side with
//      word shifts (Sec. IV-B);
//   6. joins the rows above and below into visibility and expands bitsets and
//      board bytes into 16-cell observation and mask chunks written with
//      128-bit streaming stores;
//   7. optionally picks the next actions with the benchmark policy: legal
//      (cell, direction) counts per chunk, a group scan to find the chunk, a
//      bisection of its legal moves to find the pair.
//
// Terrain bytes carry the cell type in bits 0-1 and, in bits 2-5, whether
// the neighbour up / down / left / right exists and is not a mountain.  The
// generator sets these bits once per map (mountains never change), so move
// validation and the mask read them instead of the neighbours.  The public
// state (gen_read_state) shows bits 0-1 only.
//
// No floating point decides anything: all game arithmetic is integer.
#pragma once
#include <cuda_runtime.h>

#include "gk_internal.h"

namespace gk {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
// games with at most two players share a warp: two (16 lanes each) up to
// kPairMaxCells padded cells, and in multi-frame launches four (8 lanes each)
// up to kQuadMaxCells (measured: per-frame launches of small boards lose with
// four, resident rollouts gain)
constexpr int kQuadMaxCells = 576;
constexpr int kPairMaxCells = 1024;
constexpr int kPairMaxPlayers = 2;
constexpr int kVisGuard = 4;  // zero words around a player's row bits: the rows above and below lie up to 64 cells away
constexpr int kFallbackCells = 1024;  // see place_generals_bfs
constexpr int kPlain = 0, kMountain = 1, kCastle = 2, kGeneral = 3;
constexpr int kArmyMax = 32767;
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ULL;
constexpr uint32_t kSplitThresh = 858993459u;  // floor(0.2 * 2^32)

// ---- SplitMix64 (Steele, Lea, Flood, OOPSLA 2014) as a counter hash -------
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
// n-th output of the SplitMix64 stream seeded with s
__device__ __forceinline__ uint64_t stream_out(uint64_t s, uint64_t n) { return mix64(s + (n + 1) * kGamma); }
__device__ __forceinline__ uint64_t hkey(uint64_t s, uint64_t a, uint64_t b, uint64_t c) {
    return stream_out(stream_out(stream_out(s, a), b), c);
}
__device__ __forceinline__ uint32_t hdraw(uint64_t k, uint64_t i) { return (uint32_t)(stream_out(k, i) >> 32); }
// uniform integer in [0, n) by multiply-shift
__device__ __forceinline__ int uniform_below(uint32_t u, uint32_t n) { return (int)__umulhi(u, n); }

// ---- a group of W lanes working on one game ----------------------------------
// The whole warp (W = 32) or one of its halves (W = 16, two games per warp).
// Collectives name only the group's lanes, so the two halves of a warp run
// their games independently (also through divergent branches).
template <int W>
struct Grp {
    static constexpr int width = W;
    int lane;       // 0 .. W-1
    int shift;      // the group's first lane in the warp
    unsigned mask;  // the group's lanes
    __device__ __forceinline__ explicit Grp(int warp_lane)
        : lane(warp_lane & (W - 1)), shift(W == 32 ? 0 : (warp_lane & (32 - W))),
          mask(W == 32 ? kFull : (((1u << W) - 1u) << (warp_lane & (32 - W)))) {}
    template <class T>
    __device__ __forceinline__ T shfl(T v, int src) const { return __shfl_sync(mask, v, src, W); }
    template <class T>
    __device__ __forceinline__ T shfl_up(T v, int d) const { return __shfl_up_sync(mask, v, d, W); }
    template <class T>
    __device__ __forceinline__ T shfl_down(T v, int d) const { return __shfl_down_sync(mask, v, d, W); }
    // the group's lanes that hold the same value as this one
    __device__ __forceinline__ unsigned match(int v) const { return (__match_any_sync(mask, v) & mask) >> shift; }
    // bit i = lane i of the group (the other half's lanes are masked off)
    __device__ __forceinline__ unsigned ballot(bool pr) const {
        if (W == 32) return __ballot_sync(kFull, pr);
        return (__ballot_sync(mask, pr) & mask) >> shift;
    }
    __device__ __forceinline__ unsigned reduce_add(unsigned v) const {
        if constexpr (W == 32) {
            return __reduce_add_sync(kFull, v);
        } else {
#pragma unroll
            for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, W);
            return v;
        }
    }
    __device__ __forceinline__ bool any(bool pr) const {
        if (W == 32) return __any_sync(kFull, pr);
        return ballot(pr) != 0u;
    }
    __device__ __forceinline__ void sync() const { __syncwarp(mask); }
};

// ---- per-warp shared-memory view --------------------------------------------
struct Smem {
    int16_t* army;
    int8_t* owner;
    uint8_t* terrain;  // type | passable-neighbour bits << 2
    uint32_t* own;     // [pmax][stride]
    uint32_t* big;     // army >= 2
    uint32_t* col0;    // first column
    uint32_t* colL;    // last column
    // each player's seen-from-the-row bits (see fog_pass), kVisGuard zero words
    // before and after every player's: [pmax][vstride()] from the first word on
    uint32_t* vis;
    uint32_t* tmp;  // scratch bitset: the first player's of vis
    uint8_t* cnt;      // [pmax][chunks]: legal (cell, direction) pairs of a player's 16-cell chunk
    int32_t* misc;     // [0..7] general cells, [8..15] land, [16..23] army
    int stride;
    __device__ __forceinline__ int vstride() const { return stride + kVisGuard; }
};
// words of the vis region of a carve
__host__ __device__ __forceinline__ int vis_region_words(int st, int pmax) { return kVisGuard + pmax * (st + kVisGuard); }

__host__ __device__ __forceinline__ int count_region_bytes(int npad_max, int pmax) {
    return (pmax * (npad_max >> 4) + 15) & ~15;
}

// A group's shared-memory geometry packed in one word: padded cells of the
// largest board (13 bits), bitset stride in words (8 bits), players (4 bits).
__host__ __device__ __forceinline__ uint32_t pack_geom(int npad_max, int nw_stride, int pmax) {
    return (uint32_t)npad_max | ((uint32_t)nw_stride << 13) | ((uint32_t)pmax << 21);
}
__device__ __forceinline__ uint32_t geom_of(const KArgs& a) { return pack_geom(a.npad_max, a.nw_stride, a.pmax); }

__device__ __forceinline__ Smem carve_dims(char* base, const int np, const int st, const int pm) {
    Smem s;
    s.army = reinterpret_cast<int16_t*>(base);
    s.owner = reinterpret_cast<int8_t*>(base + 2 * np);
    s.terrain = reinterpret_cast<uint8_t*>(base + 3 * np);
    uint32_t* w = reinterpret_cast<uint32_t*>(base + 4 * np);
    s.own = w;
    w += pm * st;
    s.big = w;
    w += st;
    s.col0 = w;
    w += st;
    s.colL = w;
    w += st;
    s.vis = s.tmp = w + kVisGuard;
    w += vis_region_words(st, pm);
    s.cnt = reinterpret_cast<uint8_t*>(w);
    w += count_region_bytes(np, pm) >> 2;
    s.misc = reinterpret_cast<int32_t*>(w);
    s.stride = st;
    return s;
}
__device__ __forceinline__ Smem carve_geom(char* base, uint32_t geom) {
    return carve_dims(base, (int)(geom & 0x1FFFu), (int)((geom >> 13) & 0xFFu), (int)((geom >> 21) & 0xFu));
}
// the launch's own geometry, straight from the kernel parameters
__device__ __forceinline__ Smem carve(char* base, const KArgs& a) {
    return carve_dims(base, a.npad_max, a.nw_stride, a.pmax);
}

struct Game {
    int H, W, N, Npad, nch, P, mode, nw;
    int64_t plane_off;
    int cell_off, player_off, n_cities, dmin;
};

__device__ __forceinline__ Game load_game(const GameInfo* gi) {
    Game g;
    g.H = gi->H;
    g.W = gi->W;
    g.N = gi->N;
    g.Npad = gi->Npad;
    g.nch = gi->Npad >> 4;
    g.P = gi->P;
    g.mode = gi->mode;
    g.nw = (gi->N + 31) >> 5;
    g.plane_off = gi->plane_off;
    g.cell_off = gi->cell_off;
    g.player_off = gi->player_off;
    g.n_cities = gi->n_cities;
    g.dmin = gi->dmin;
    return g;
}

// UNI: the launch's games all have the launch's shape (a.uniform), so every
// field is a kernel parameter or follows from gidx; a kernel compiled for it
// keeps none of them in registers.
template <bool UNI = false>
__device__ __forceinline__ Game game_of(const KArgs& a, int gidx) {
    if (!UNI && !a.uniform) return load_game(a.info + gidx);
    Game g = load_game(&a.ushape);
    g.cell_off = gidx * g.Npad;
    g.player_off = gidx * g.P;
    g.plane_off = (int64_t)gidx * g.P * g.Npad;
    return g;
}
template <bool UNI = false>
__device__ __forceinline__ uint64_t game_id_of(const KArgs& a, int gidx) {
    return (UNI || a.uniform) ? a.game_id_base + (uint64_t)gidx : a.info[gidx].game_id;
}

__device__ __forceinline__ uint32_t valid_bits(int N, int w) {
    int rem = N - 32 * w;
    if (rem >= 32) return kFull;
    if (rem <= 0) return 0u;
    return (1u << rem) - 1u;
}

// passable-neighbour bits of every cell (bits 2..5 of the terrain byte),
// from a mountain bitset so that no lane reads a byte another lane writes
template <int LW>
__device__ __forceinline__ void derive_passable(const Game& g, const Smem& s, const Grp<LW>& t) {
    const int N = g.N, W = g.W, H = g.H;
    for (int w = 0; w < g.nw; ++w) {
        unsigned m = 0;
        for (int h = 0; h < 32; h += LW) {
            const int c = 32 * w + h + t.lane;
            m |= t.ballot(c < N && (s.terrain[c] & 3) == kMountain) << h;
        }
        if (t.lane == 0) s.tmp[w] = m;
    }
    t.sync();
    for (int c = t.lane; c < N; c += LW) {
        const int r = c / W, col = c - r * W;
        auto mtn = [&](int x) { return (s.tmp[x >> 5] >> (x & 31)) & 1u; };
        uint32_t b = 0;
        if (r > 0 && !mtn(c - W)) b |= 1u;
        if (r < H - 1 && !mtn(c + W)) b |= 2u;
        if (col > 0 && !mtn(c - 1)) b |= 4u;
        if (col < W - 1 && !mtn(c + 1)) b |= 8u;
        s.terrain[c] = (uint8_t)((s.terrain[c] & 3) | (b << 2));
    }
    t.sync();
}

// ---- board geometry: first and last column bitsets -------------------------
// g_columns[W-1][0][w] has bit b set when cell 32w+b is in the first column
// of a W-wide board, [1] the last column; filled once per device.
constexpr int kColWords = (kMaxSide * kMaxSide) / 32;
__device__ __align__(16) uint32_t g_columns[kMaxSide][2][kColWords];

template <class T>
__device__ __forceinline__ void column_pass(const Game& g, const Smem& s, const T& t) {
    const uint32_t* c0 = g_columns[g.W - 1][0];
    const uint32_t* cl = g_columns[g.W - 1][1];
    for (int w = t.lane; w < g.nw; w += t.width) {
        s.col0[w] = c0[w];
        s.colL[w] = cl[w];
    }
    t.sync();
}

// ---- row bitsets (BFS of the map generator) --------------------------------
// A set of cells held in registers: lane l of the group keeps rows R*l ..
// R*l + R-1 of the board, one word of W bits each (32 or 64).  A step of a
// flood fill is then two shifts in place and the two neighbour rows (two
// shuffles), about ten instructions for a board of up to 32 x 32 with a warp
// per game and no shared memory.  The same fill as one dilation per step over
// shared-memory bitsets (a lane per 32 cells, a sync on either side) made
// 21,838 warp instructions per 24x24 map with BFS spacing and the castle
// guarantee.
template <class T, int R>
struct RowSet {
    T v[R];
};

// 32 bits of the nw-word bitset x from bit b on (b may lie outside: zeros)
__device__ __forceinline__ uint32_t bits_at(const uint32_t* x, int nw, int b) {
    const int i = b >> 5;
    const uint32_t lo = (unsigned)i < (unsigned)nw ? x[i] : 0u;
    const uint32_t hi = (unsigned)(i + 1) < (unsigned)nw ? x[i + 1] : 0u;
    return __funnelshift_r(lo, hi, b & 31);
}

// rows of the cells that are clear (invert) or set in the row-major bitset x
template <class T, int R, int LW>
__device__ __forceinline__ RowSet<T, R> load_rows(const uint32_t* x, const Game& g, bool invert, const Grp<LW>& t) {
    RowSet<T, R> s;
    const T width = g.W >= (int)(8 * sizeof(T)) ? ~(T)0 : (((T)1 << g.W) - 1);
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int r = R * t.lane + i;
        T v = bits_at(x, g.nw, r * g.W);
        if (sizeof(T) == 8) v |= (T)((uint64_t)bits_at(x, g.nw, r * g.W + 32) << 32);
        s.v[i] = r < g.H ? ((invert ? ~v : v) & width) : (T)0;
    }
    return s;
}

// one step of a flood fill through `pass`
template <class T, int R, int LW>
__device__ __forceinline__ void flood_step(RowSet<T, R>& x, const RowSet<T, R>& pass, const Grp<LW>& t) {
    T prev = t.shfl_up(x.v[R - 1], 1), below = t.shfl_down(x.v[0], 1);
    if (t.lane == 0) prev = 0;
    if (t.lane == LW - 1) below = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const T cur = x.v[i], next = i + 1 < R ? x.v[i + 1] : below;
        x.v[i] = cur | (((cur << 1) | (cur >> 1) | prev | next) & pass.v[i]);
        prev = cur;
    }
}
// n steps, or (n < 0) steps until nothing changes; either way it stops when
// four steps in a row change nothing
template <class T, int R, int LW>
__device__ __forceinline__ void flood(RowSet<T, R>& x, const RowSet<T, R>& pass, int n, const Grp<LW>& t) {
    for (; n < 0 || n >= 4; n -= n < 0 ? 0 : 4) {
        const RowSet<T, R> old = x;
#pragma unroll
        for (int m = 0; m < 4; ++m) flood_step(x, pass, t);
        bool changed = false;
#pragma unroll
        for (int i = 0; i < R; ++i) changed |= x.v[i] != old.v[i];
        if (!t.any(changed)) return;
    }
#pragma unroll 1
    for (; n > 0; --n) flood_step(x, pass, t);
}
// Keep in `allowed` the cells whose BFS distance from cell src through `pass`
// is above lo (lo < 0: no lower bound) and at most hi (hi <= 0: reachable).
// Returns the cells within hi steps.
template <class T, int R, int LW>
__device__ __forceinline__ RowSet<T, R> bfs_restrict(int src, int lo, int hi, const RowSet<T, R>& pass,
                                                     RowSet<T, R>& allowed, const Game& g, const Grp<LW>& t) {
    RowSet<T, R> vis;
    const int r = src / g.W, c = src - r * g.W;
#pragma unroll
    for (int i = 0; i < R; ++i) vis.v[i] = R * t.lane + i == r ? (T)1 << c : (T)0;
    const bool capped = hi > 0;
    int done = 0;
    if (lo >= 0) {
        done = capped ? min(lo, hi) : lo;
        flood(vis, pass, done, t);
        const T keep = capped && hi < lo ? (T)0 : ~(T)0;  // the cap lies below the bound: nothing fits
#pragma unroll
        for (int i = 0; i < R; ++i) allowed.v[i] &= ~vis.v[i] & keep;
    }
    flood(vis, pass, capped ? hi - done : -1, t);
#pragma unroll
    for (int i = 0; i < R; ++i) allowed.v[i] &= vis.v[i];
    return vis;
}

template <class T>
__device__ __forceinline__ int bits_of(T x) { return sizeof(T) == 8 ? __popcll((uint64_t)x) : __popc((uint32_t)x); }
template <class T>
__device__ __forceinline__ int lowest(T x) { return (sizeof(T) == 8 ? __ffsll((long long)x) : __ffs((int)x)) - 1; }

// the k-th (0-based, row-major) cell of x, or -1 when it holds no more than k
template <class T, int R, int LW>
__device__ __forceinline__ int kth_cell(const RowSet<T, R>& x, uint32_t k, const Game& g, const Grp<LW>& t) {
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) mine += bits_of(x.v[i]);
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < LW; o <<= 1) {
        const uint32_t y = t.shfl_up(incl, o);
        if (t.lane >= o) incl += y;
    }
    const unsigned b = t.ballot(incl > k);
    if (b == 0u) return -1;
    int cell = 0;
    uint32_t left = k - (incl - mine);
    bool open = true;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const uint32_t n = bits_of(x.v[i]);
        if (open && left < n) {
            T v = x.v[i];
            for (uint32_t z = 0; z < left; ++z) v &= v - 1;
            cell = (R * t.lane + i) * g.W + lowest(v);
            open = false;
        }
        left -= n;
    }
    return t.shfl(cell, __ffs(b) - 1);
}
// whether x holds cell (r, c), a cell of its own per lane
template <class T, int R, int LW>
__device__ __forceinline__ bool row_test(const RowSet<T, R>& x, int r, int c, const Grp<LW>& t) {
    T v = 0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const T y = t.shfl(x.v[i], r / R);
        if (r % R == i) v = y;
    }
    return (v >> c) & 1;
}

// Generals at BFS distance (through non-mountain cells) in [D, dmax] of every
// earlier general, D falling by one after each kGenAttempts rejected draws;
// at D = 0 the first cell (row-major) within the cap of every earlier general,
// else reachable from general 0, else any free cell.  Lane p returns player
// p's general in the low 16 bits; bit 20 says whether a general cannot reach
// general 0 (the L-path carve is then needed): only one of the last kind,
// since every other placement is reachable from general 0.  mtn: the
// mountains as a row-major bitset.
template <class T, int R, int LW>
__device__ __forceinline__ int place_generals_bfs(const Game& g, const uint32_t* mtn, uint64_t kgen, int dmax,
                                                  const Grp<LW>& t) {
    const int W = g.W;
    const RowSet<T, R> pass = load_rows<T, R>(mtn, g, true, t);
    RowSet<T, R> allowed = pass;
    int folded = 0;  // earlier generals whose distances `allowed` respects at this D
    uint32_t i = 0;
    int D = g.dmin;
    int my_gpos = -1;
    bool cut_off = false;
    for (int p = 0; p < g.P; ++p) {
        int placed = -1;
        while (placed < 0 && D >= 1) {
            for (; folded < p; ++folded) bfs_restrict(t.shfl(my_gpos, folded), D - 1, dmax, pass, allowed, g, t);
            int found = -1;
            for (int base = 0; base < kGenAttempts && found < 0; base += LW) {
                const int c = uniform_below(hdraw(kgen, (uint64_t)(i + base + t.lane)), (uint32_t)g.N);
                const int r = c / W;
                const unsigned b = t.ballot(row_test(allowed, r, c - r * W, t));
                if (b) {
                    const int l = __ffs(b) - 1;
                    found = base + l;
                    placed = t.shfl(c, l);
                }
            }
            if (found >= 0) {
                i += (uint32_t)found + 1;
            } else {
                i += kGenAttempts;
                D -= 1;
                allowed = pass;
                folded = 0;
            }
        }
        if (placed < 0) {
            // the fallbacks, over cells without a general -- of those in the
            // first kFallbackCells cells: later ones have never been left out
            // here, and maps are keyed by their seeds, so they stay as they are
            RowSet<T, R> open = pass, any;
            const T width = W >= (int)(8 * sizeof(T)) ? ~(T)0 : (((T)1 << W) - 1);
#pragma unroll
            for (int k = 0; k < R; ++k) any.v[k] = R * t.lane + k < g.H ? width : (T)0;
            for (int q = 0; q < p; ++q) {
                const int gq = t.shfl(my_gpos, q), r = gq / W;
#pragma unroll
                for (int k = 0; k < R; ++k)
                    if (R * t.lane + k == r && gq < kFallbackCells) {
                        const T bit = (T)1 << (gq - r * W);
                        open.v[k] &= ~bit;
                        any.v[k] &= ~bit;
                    }
            }
            RowSet<T, R> x = open;
            for (int q = 0; q < p; ++q) bfs_restrict(t.shfl(my_gpos, q), -1, dmax, pass, x, g, t);
            placed = kth_cell(x, 0u, g, t);
            if (placed < 0) {
                x = open;
                if (p > 0) bfs_restrict(t.shfl(my_gpos, 0), -1, 0, pass, x, g, t);
                placed = kth_cell(x, 0u, g, t);
            }
            if (placed < 0) {
                placed = kth_cell(any, 0u, g, t);
                cut_off |= p > 0;
            }
        }
        if (t.lane == p) my_gpos = placed;
    }
    return (my_gpos & 0xFFFF) | (cut_off ? (1 << 20) : 0);
}

// A neutral castle within a.castle_radius BFS steps of every general (s.misc
// holds the generals): where none is, one on a free plain cell of the ball,
// the k-th such cell in row-major order with k drawn uniformly.  mtn, taken
// and castles: row-major bitsets of the mountains, of the cells that are not
// neutral plain, and of the castles (updated).
template <class T, int R, int LW>
__device__ __forceinline__ void castle_guarantee(const KArgs& a, const Game& g, const Smem& s, const uint32_t* mtn,
                                                 const uint32_t* taken, uint32_t* castles, uint64_t kmap, const Grp<LW>& t) {
    const RowSet<T, R> pass = load_rows<T, R>(mtn, g, true, t);
    RowSet<T, R> free_plain = load_rows<T, R>(taken, g, true, t), built = load_rows<T, R>(castles, g, false, t);
    const uint64_t knp = stream_out(kmap, 5);
    const uint64_t kna = stream_out(kmap, 6);
    for (int p = 0; p < g.P; ++p) {
        RowSet<T, R> near = built;
        const RowSet<T, R> ball = bfs_restrict(s.misc[p], -1, a.castle_radius, pass, near, g, t);
        bool have = false;
#pragma unroll
        for (int i = 0; i < R; ++i) have |= near.v[i] != 0;
        if (t.any(have)) continue;
        RowSet<T, R> x = free_plain;
        uint32_t cnt = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            x.v[i] &= ball.v[i];
            cnt += bits_of(x.v[i]);
        }
        cnt = t.reduce_add(cnt);
        if (cnt == 0) continue;
        const int cell = kth_cell(x, (uint32_t)uniform_below(hdraw(knp, (uint64_t)p), cnt), g, t);
        if (t.lane == 0) {
            castles[cell >> 5] |= 1u << (cell & 31);
            s.army[cell] = (int16_t)(a.city_min + uniform_below(hdraw(kna, (uint64_t)p), (uint32_t)a.city_span));
        }
        const int r = cell / g.W;
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (R * t.lane + i == r) {
                const T bit = (T)1 << (cell - r * g.W);
                free_plain.v[i] &= ~bit;
                built.v[i] |= bit;
            }
    }
}

__device__ __forceinline__ bool wide_rows(const Game& g) { return g.W > 32 || g.H > 32; }

// ---- map generator (Sec. IV-A) ----------------------------------------------
// Mountains, castles and taken cells are row-major bitsets while the map is
// made; the cells' bytes are written once at the end, with the passable-
// neighbour bits.  Draws are evaluated LW at a time and accepted in draw
// order, so the draw counters advance exactly as one by one.
//
// Instructions bound it.  Resets of 65,536 24x24 games: 314.6 -> 204.7 us with
// the plain generator (castles a batch of draws at a time instead of a batch
// each, cells as bits until the end), 2,004 -> 419 us with BFS spacing and the
// castle guarantee (see RowSet; 608 MB of state and outputs need 90 us), with
// the step's newer passes 184 and 388 us.
// SPAWN: with the options of the launch (a.spawn_*, a.castle_radius).
// ROW_BITS: the word of a row bitset, 32 for boards of up to 32 rows and
// columns, else 64; 0: by the game.  Launches of one shape know it, and
// without the 64-bit rows' code the 32-bit rows keep more in registers (reset
// of 65,536 24x24 games with BFS spacing and the castle guarantee: 388 -> 349
// us; in a batch of both kinds, two generators would take turns in the
// instruction cache: 8,192 mixed games 380 -> 430 us).
template <int LW, bool SPAWN, int ROW_BITS>
__device__ __forceinline__ void generate_body(const KArgs& a, const Game& g, const Smem& s, uint64_t gid,
                                             uint32_t epoch, const Grp<LW>& t) {
    const int N = g.N, W = g.W, P = g.P, nw = g.nw;
    // bitsets in regions that the step rebuilds after a new map
    uint32_t* mtn = s.tmp;
    uint32_t* taken = s.own;
    uint32_t* castles = s.big;

    // mountains: a ballot per LW cells, draws running on from one another (the
    // stream advances by a constant) and several words' draws interleaved;
    // the board's army and owner planes cleared
    const uint64_t kmap = stream_out(stream_out(a.seed, gid), epoch);  // hkey(seed, gid, epoch, x) = stream_out(kmap, x)
    uint64_t z = stream_out(kmap, 1) + (uint64_t)(t.lane + 1) * kGamma;
#pragma unroll 2
    for (int w = 0; w < nw; ++w) {
        unsigned m = 0;
#pragma unroll
        for (int h = 0; h < 32; h += LW) {
            m |= t.ballot((uint32_t)(mix64(z) >> 32) < a.mtn_thresh) << h;
            z += (uint64_t)LW * kGamma;
        }
        if (t.lane == 0) mtn[w] = m & valid_bits(N, w);
    }
    for (int v = t.lane; v < 2 * g.nch; v += LW) reinterpret_cast<uint4*>(s.army)[v] = make_uint4(0, 0, 0, 0);
    for (int v = t.lane; v < g.nch; v += LW) reinterpret_cast<uint4*>(s.owner)[v] = make_uint4(kFull, kFull, kFull, kFull);
    for (int w = t.lane; w < nw; w += LW) castles[w] = 0u;
    t.sync();
    auto in = [](const uint32_t* x, int c) { return ((x[c >> 5] >> (c & 31)) & 1u) != 0u; };

    // generals
    const uint64_t kgen = stream_out(kmap, 2);
    const int dmax = SPAWN ? a.spawn_dmax : 0;
    int my_gpos = -1;  // lane p holds player p's general
    bool carve = true;
    const bool narrow_rows = ROW_BITS ? ROW_BITS == 32 : !wide_rows(g);
    if (SPAWN && a.spawn_bfs) {
        const int r = narrow_rows ? place_generals_bfs<uint32_t, 32 / LW>(g, mtn, kgen, dmax, t)
                                  : place_generals_bfs<uint64_t, 64 / LW>(g, mtn, kgen, dmax, t);
        my_gpos = t.lane < P ? (r & 0xFFFF) : -1;
        carve = (r >> 20) & 1;
    } else {
        uint32_t i = 0;
        int D = g.dmin;
        for (int p = 0; p < P; ++p) {
            int placed = -1;
            while (placed < 0) {
                if (D >= 1) {
                    int found = -1;
                    for (int base = 0; base < kGenAttempts; base += LW) {
                        const int c = uniform_below(hdraw(kgen, (uint64_t)(i + base + t.lane)), (uint32_t)N);
                        bool ok = !in(mtn, c);
                        const int rc = c / W, cc = c - rc * W;
                        for (int q = 0; q < p; ++q) {
                            const int gq = t.shfl(my_gpos, q);
                            const int rq = gq / W, cq = gq - rq * W;
                            const int d = abs(rc - rq) + abs(cc - cq);
                            if (d < D || (dmax > 0 && d > dmax)) ok = false;
                        }
                        const unsigned b = t.ballot(ok);
                        if (b) {
                            const int l = __ffs(b) - 1;
                            found = base + l;
                            placed = t.shfl(c, l);
                            break;
                        }
                    }
                    if (found >= 0) {
                        i += (uint32_t)found + 1;
                    } else {
                        i += kGenAttempts;
                        D -= 1;
                    }
                } else {
                    for (int base = 0; base < N && placed < 0; base += LW) {
                        const int c = base + t.lane;
                        bool ok = c < N;
                        for (int q = 0; q < p; ++q)
                            if (t.shfl(my_gpos, q) == c) ok = false;
                        const unsigned b = t.ballot(ok);
                        if (b) placed = base + __ffs(b) - 1;
                    }
                }
            }
            if (t.lane == p) my_gpos = placed;
        }
    }
    if (t.lane < P) {
        s.owner[my_gpos] = (int8_t)t.lane;
        s.army[my_gpos] = 1;
        s.misc[t.lane] = my_gpos;
        atomicAnd(mtn + (my_gpos >> 5), ~(1u << (my_gpos & 31)));
    }
    t.sync();

    // connectivity: L-path rows first, then columns, between consecutive
    // generals (in BFS mode only when some general cannot reach general 0)
    if (carve) {
        for (int p = 0; p + 1 < P; ++p) {
            const int g0 = s.misc[p], g1 = s.misc[p + 1];
            const int r0 = g0 / W, c0 = g0 - r0 * W, r1 = g1 / W, c1 = g1 - r1 * W;
            const int dr = abs(r1 - r0), dc = abs(c1 - c0);
            for (int k = t.lane; k < dr + dc; k += LW) {
                const int r = k < dr ? (r1 > r0 ? r0 + k + 1 : r0 - k - 1) : r1;
                const int c = k < dr ? c0 : (c1 > c0 ? c0 + (k - dr) + 1 : c0 - (k - dr) - 1);
                const int cell = r * W + c;
                if (in(mtn, cell)) atomicAnd(mtn + (cell >> 5), ~(1u << (cell & 31)));
            }
        }
        t.sync();
    }

    // neutral castles on neutral plain cells: castle k takes the first such
    // cell among its next kGenAttempts draws, else none.  A batch of LW draws
    // serves as many castles as it can: a draw is accepted when its cell is
    // free and no earlier draw of the batch took it.
    for (int w = t.lane; w < nw; w += LW) taken[w] = mtn[w];
    t.sync();
    if (t.lane < P) atomicOr(taken + (my_gpos >> 5), 1u << (my_gpos & 31));
    t.sync();
    const uint64_t kpos = stream_out(kmap, 3);
    const uint64_t karm = stream_out(kmap, 4);
    int k = 0;       // the castle being placed
    int misses = 0;  // its rejected draws so far
    for (uint32_t j = 0; k < g.n_cities; j += LW) {
        const int c = uniform_below(hdraw(kpos, (uint64_t)(j + t.lane)), (uint32_t)N);
        const bool open = !in(taken, c);
        const unsigned same = t.match(c);
        const bool ok = open && (same & ((1u << t.lane) - 1u)) == 0u;
        unsigned b = t.ballot(ok);
        const int first = b ? __ffs(b) - 1 : LW;
        if (misses + first >= kGenAttempts) {  // castle k's attempts end before that draw
            k += 1;
            misses -= kGenAttempts;
        }
        const int mine = k + __popc(b & ((1u << t.lane) - 1u));  // the castle an accepted draw places
        if (ok && mine < g.n_cities) {
            atomicOr(taken + (c >> 5), 1u << (c & 31));
            atomicOr(castles + (c >> 5), 1u << (c & 31));
            s.army[c] = (int16_t)(a.city_min + uniform_below(hdraw(karm, (uint64_t)mine), (uint32_t)a.city_span));
        }
        k += __popc(b);
        misses = b ? LW - 1 - (31 - __clz(b)) : misses + LW;
        t.sync();
    }

    if (SPAWN && a.castle_radius > 0) {
        if (narrow_rows)
            castle_guarantee<uint32_t, 32 / LW>(a, g, s, mtn, taken, castles, kmap, t);
        else
            castle_guarantee<uint64_t, 64 / LW>(a, g, s, mtn, taken, castles, kmap, t);
    }

    // terrain bytes, 16 cells per lane: type, and whether each neighbour
    // exists and is not a mountain
    t.sync();
    const uint16_t* col0 = reinterpret_cast<const uint16_t*>(g_columns[W - 1][0]);
    const uint16_t* colL = reinterpret_cast<const uint16_t*>(g_columns[W - 1][1]);
    auto passable = [&](int b) {  // 16 cells from b on: on the board and not a mountain
        const int i = b >> 5;
        const uint32_t lo = (unsigned)i < (unsigned)nw ? ~mtn[i] & valid_bits(N, i) : 0u;
        const uint32_t hi = (unsigned)(i + 1) < (unsigned)nw ? ~mtn[i + 1] & valid_bits(N, i + 1) : 0u;
        return __funnelshift_r(lo, hi, b & 31);
    };
    for (int ch = t.lane; ch < g.nch; ch += LW) {
        const int c0 = ch << 4;
        const uint32_t valid = valid_bits(N, c0 >> 5) >> (c0 & 16);
        const uint32_t m = mtn[c0 >> 5] >> (c0 & 16), z = castles[c0 >> 5] >> (c0 & 16);
        const uint32_t up = passable(c0 - W), dn = passable(c0 + W);
        const uint32_t lf = passable(c0 - 1) & ~(uint32_t)col0[ch], rt = passable(c0 + 1) & ~(uint32_t)colL[ch];
        uint32_t out[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int sh = 4 * q;
            auto spread = [&](uint32_t x) { return (((x >> sh) & 15u) * 0x00204081u) & 0x01010101u; };
            out[q] = spread(m & valid) | (spread(z) << 1) | (spread(up & valid) << 2) | (spread(dn & valid) << 3) |
                     (spread(lf & valid) << 4) | (spread(rt & valid) << 5);
        }
        *reinterpret_cast<uint4*>(s.terrain + c0) = make_uint4(out[0], out[1], out[2], out[3]);
    }
    t.sync();
    if (t.lane < P) s.terrain[my_gpos] = (uint8_t)((s.terrain[my_gpos] & ~3u) | kGeneral);
    t.sync();
}

// Out-of-line entry point of a new map inside a multi-frame launch or a CTA
// per game: it takes plain arguments and rebuilds the game and shared-memory views itself, so
// that the step kernel never materialises those structures in local memory
// for a call it rarely makes.
template <int LW, bool UNI, bool SPAWN>
__device__ __noinline__ void generate(const KArgs& a, int gidx, char* warp_base, uint32_t geom, uint64_t gid,
                                     uint32_t epoch, int warp_lane) {
    generate_body<LW, SPAWN, 0>(a, game_of<UNI>(a, gidx), carve_geom(warp_base, geom), gid, epoch, Grp<LW>(warp_lane));
}

// ---- one move on lane 0 (Sec. IV-D, IV-E) ----------------------------------
// Returns the captured general's cell in the low 16 bits and the loser in
// bits 16..19 (+1), or 0 when no general fell.
__device__ int resolve_move(const Game& g, const Smem& s, int p, int32_t act, uint32_t& alive, uint32_t& invalid,
                            uint32_t& sat) {
    if (act < 0 || act >= 9 * g.N) {
        invalid += 1;
        return 0;
    }
    const int c = act / 9, k = act - 9 * c;
    if (k == 0) return 0;
    const int d = (k - 1) & 3;
    const int av = s.army[c];
    // bit 2+d: the neighbour towards d exists and is not a mountain
    if (s.owner[c] != p || av < 2 || !((s.terrain[c] >> (2 + d)) & 1u)) {
        invalid += 1;
        return 0;
    }
    const int dst = c + (d == 0 ? -g.W : d == 1 ? g.W : d == 2 ? -1 : 1);
    const int moved = (k >= 5) ? (av >> 1) : (av - 1);
    s.army[c] = (int16_t)(av - moved);
    const int o = s.owner[dst];
    const int def = s.army[dst];
    if (o == p || (o >= 0 && g.mode == 1 && (o >> 1) == (p >> 1))) {
        int sum = def + moved;
        if (sum > kArmyMax) {
            sum = kArmyMax;
            sat += 1;
        }
        s.army[dst] = (int16_t)sum;
        if (o != p && (s.terrain[dst] & 3) != kGeneral) s.owner[dst] = (int8_t)p;
        return 0;
    }
    if (moved > def) {
        s.owner[dst] = (int8_t)p;
        s.army[dst] = (int16_t)(moved - def);
        if ((s.terrain[dst] & 3) == kGeneral && o >= 0) {
            s.terrain[dst] = (uint8_t)((s.terrain[dst] & ~3u) | kCastle);
            alive &= ~(1u << o);
            return dst | ((o + 1) << 16);
        }
    } else if (moved == def) {
        s.army[dst] = 0;
    } else {
        s.army[dst] = (int16_t)(def - moved);
    }
    return 0;
}

// ---- the players' moves of one turn (Sec. IV-D, IV-E) ------------------------
// In rotating priority, each checked when it runs (Q1).  my_act: lane p's is
// player p's.  alive and eliminated end up the same on every lane; invalid
// and sat count on lane 0.
template <int LW>
__device__ __forceinline__ void play_moves(const Game& g, const Smem& s, const Grp<LW>& t, uint32_t turn, int32_t my_act,
                                           uint32_t& alive, uint32_t& eliminated, uint32_t& invalid, uint32_t& sat) {
    int p = (int)(turn % (uint32_t)g.P);
    for (int k = 0; k < g.P; ++k, p = p + 1 == g.P ? 0 : p + 1) {
        const int32_t act = t.shfl(my_act, p);
        int cap = 0;
        if (t.lane == 0 && ((alive >> p) & 1u)) cap = resolve_move(g, s, p, act, alive, invalid, sat);
        cap = t.shfl(cap, 0);
        alive = t.shfl(alive, 0);
        t.sync();
        if (cap) {
            // land transfer: every other cell of the loser, army - army/2 (Q7)
            const int dst = cap & 0xFFFF, q = (cap >> 16) - 1;
            eliminated |= 1u << q;
            for (int c = t.lane; c < g.N; c += LW) {
                if (c != dst && s.owner[c] == q) {
                    s.owner[c] = (int8_t)p;
                    const int av = s.army[c];
                    s.army[c] = (int16_t)(av - (av >> 1));
                }
            }
            t.sync();
        }
    }
}

// ---- termination and reward (Sec. III, IV-D, IV-E; Q17, Q21) -------------------
// Returns the done code; lane p's reward is player p's.
__device__ __forceinline__ uint32_t outcome(const KArgs& a, const Game& g, int lane, uint32_t turn, uint32_t alive,
                                            uint32_t eliminated, float& reward) {
    uint32_t done = 0;
    if (g.mode == 1) {
        const bool dead0 = (alive & 0x3u) == 0u, dead1 = (alive & 0xCu) == 0u;
        if (dead0 || dead1) {
            done = 1;
            const bool mine_dead = ((lane >> 1) == 0) ? dead0 : dead1;
            reward = mine_dead ? -1.0f : 1.0f;
        }
    } else {
        if ((eliminated >> lane) & 1u) reward = -1.0f;
        if (__popc(alive) <= 1) {
            done = 1;
            if ((alive >> lane) & 1u) reward = 1.0f;
        }
    }
    if (!done && a.max_turns > 0 && turn >= (uint32_t)a.max_turns) done = 2;
    return done;
}

// ---- growth + bitsets + army totals, 16 cells per lane ---------------------
// Bytes are handled four at a time inside 32-bit words.  Per-cell flags are
// bytes of 0 or 1 (or 0x80); dot products do the rest: four flags times powers
// of two collect into bits (dp4a), and flags times 16-bit armies add up to a
// player's total (dp2a).  The integer ALU bounds this pass, and dot products
// run beside it; with zero-byte detection per player, multiplies to gather
// bits and armies split into low and high bytes it took about twice the
// instructions.  With it and the policy's players side by side: step of
// 65,536 24x24 1v1 games 132.5 -> 129 us, 16 frames of 32,768 ragged games
// 976 -> 870 us, 64 frames of 1,024 games 313 -> 293 us.

// bit j = flag byte j (0x01 * scale each) of the 16 bytes m, times scale
__device__ __forceinline__ uint32_t collect_lo(uint32_t m0, uint32_t m1) {
    return __dp4a(m1, 0x80402010u, __dp4a(m0, 0x08040201u, 0u));
}
// flag bytes 0x01 of the cells that player p owns: owners -1 .. PT-1, four a word
template <int PT>
__device__ __forceinline__ uint32_t owned_by(uint32_t ow, int p) {
    if (PT == 2) return (p ? ow & ~(ow >> 1) : ~ow) & 0x01010101u;
    const uint32_t b0 = (p & 1) ? ow : ~ow, b1 = (p & 2) ? ow >> 1 : ~(ow >> 1);
    const uint32_t v = b0 & b1 & (~(ow >> 7) & 0x01010101u);
    if (PT == 4) return v;
    return v & ((p & 4) ? ow >> 2 : ~(ow >> 2));
}

// the 16 armies from cell c0 on, grown where they are due: owned generals and
// castles +1 on even turns (grow_s), owned plain cells +1 every 50 (grow_p),
// saturating at 32767 (counted in sat)
__device__ __forceinline__ void grown_armies(const Smem& s, int c0, bool grow_s, bool grow_p, uint32_t (&aw)[8],
                                             uint32_t& sat) {
    const uint4 A0 = *reinterpret_cast<const uint4*>(s.army + c0);
    const uint4 A1 = *reinterpret_cast<const uint4*>(s.army + c0 + 8);
    aw[0] = A0.x, aw[1] = A0.y, aw[2] = A0.z, aw[3] = A0.w;
    aw[4] = A1.x, aw[5] = A1.y, aw[6] = A1.z, aw[7] = A1.w;
    if (!(grow_s || grow_p)) return;
    const uint4 O = *reinterpret_cast<const uint4*>(s.owner + c0);
    const uint4 T = *reinterpret_cast<const uint4*>(s.terrain + c0);
    const uint32_t ow[4] = {O.x, O.y, O.z, O.w}, tw[4] = {T.x, T.y, T.z, T.w};
    uint32_t g01[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t b1 = tw[k] >> 1;  // type bit 1: structures; neither bit: plain
        g01[k] = ~(ow[k] >> 7) & ((grow_s ? b1 : 0u) | (grow_p ? ~(tw[k] | b1) : 0u)) & 0x01010101u;
    }
    if (!(g01[0] | g01[1] | g01[2] | g01[3])) return;
    uint32_t over = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        aw[2 * k] += __byte_perm(g01[k], 0, 0x4140);
        aw[2 * k + 1] += __byte_perm(g01[k], 0, 0x4342);
        over |= aw[2 * k] | aw[2 * k + 1];
    }
    if (over & 0x80008000u) {  // 32767 + 1
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t ov = aw[k] & 0x80008000u;
            sat += __popc(ov);
            aw[k] -= ov >> 15;
        }
    }
    *reinterpret_cast<uint4*>(s.army + c0) = make_uint4(aw[0], aw[1], aw[2], aw[3]);
    *reinterpret_cast<uint4*>(s.army + c0 + 8) = make_uint4(aw[4], aw[5], aw[6], aw[7]);
}
// bit j: army j holds at least 2 (bit 15 / 31 of army + 0x7FFE per halfword)
__device__ __forceinline__ uint16_t big_bits(const uint32_t (&aw)[8]) {
    uint32_t b80[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        b80[k] = __byte_perm(aw[2 * k] + 0x7FFE7FFEu, aw[2 * k + 1] + 0x7FFE7FFEu, 0x7531) & 0x80808080u;
    return (uint16_t)((collect_lo(b80[0], b80[1]) >> 7) | (collect_lo(b80[2], b80[3]) << 1));
}
template <class T>
__device__ __forceinline__ uint32_t total_saturated(uint32_t sat, bool grow, const T& t) {
    return grow && t.any(sat != 0u) ? t.reduce_add(sat) : 0u;
}

// up to PT players at once
template <int PT, class T>
__device__ uint32_t chunk_pass(const Game& g, const Smem& s, bool grow_s, bool grow_p, const T& t) {
    const int P = g.P, nch = g.nch, st2 = 2 * s.stride;
    uint32_t sat = 0;
    uint32_t arm[PT], land[PT / 2];  // land: two players' counts per word
#pragma unroll
    for (int p = 0; p < PT; ++p) arm[p] = 0;
#pragma unroll
    for (int p = 0; p < PT / 2; ++p) land[p] = 0;
    uint16_t* own16 = reinterpret_cast<uint16_t*>(s.own);
    uint16_t* big16 = reinterpret_cast<uint16_t*>(s.big);
    for (int ch = t.lane; ch < nch; ch += t.width) {
        const int c0 = ch << 4;
        const uint4 O = *reinterpret_cast<const uint4*>(s.owner + c0);
        const uint32_t ow[4] = {O.x, O.y, O.z, O.w};
        uint32_t aw[8];
        grown_armies(s, c0, grow_s, grow_p, aw, sat);
        big16[ch] = big_bits(aw);
#pragma unroll
        for (int p = 0; p < PT; ++p) {
            if (p < P) {
                uint32_t m[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    m[k] = owned_by<PT>(ow[k], p);
                    arm[p] = __dp2a_hi(aw[2 * k + 1], m[k], __dp2a_lo(aw[2 * k], m[k], arm[p]));
                }
                const uint32_t own = collect_lo(m[0], m[1]) | (collect_lo(m[2], m[3]) << 8);
                own16[p * st2 + ch] = (uint16_t)own;
                land[p >> 1] += (uint32_t)__popc(own) << (16 * (p & 1));
            }
        }
        if ((nch & 1) && ch == nch - 1) {  // unused upper half of the last word
            big16[nch] = 0;
#pragma unroll
            for (int p = 0; p < PT; ++p)
                if (p < P) own16[p * st2 + nch] = 0;
        }
    }
#pragma unroll
    for (int p = 0; p < PT; ++p) {
        if (p < P) {
            const uint32_t army = t.reduce_add(arm[p]);
            const uint32_t cells = (p & 1) ? land[p >> 1] >> 16 : t.reduce_add(land[p >> 1]);
            if (!(p & 1)) land[p >> 1] = cells;
            if (t.lane == 0) {
                s.misc[8 + p] = (int)(cells & 0xFFFFu);
                s.misc[16 + p] = (int)army;
            }
        }
    }
    t.sync();
    return total_saturated(sat, grow_s || grow_p, t);
}

// the players one after another: more shared-memory loads, but few values
// live at once
template <class T>
__device__ uint32_t chunk_pass_in_turn(const Game& g, const Smem& s, bool grow_s, bool grow_p, const T& t) {
    const int P = g.P, nch = g.nch, st2 = 2 * s.stride;
    uint32_t sat = 0;
    uint16_t* own16 = reinterpret_cast<uint16_t*>(s.own);
    uint16_t* big16 = reinterpret_cast<uint16_t*>(s.big);
    for (int ch = t.lane; ch < nch; ch += t.width) {
        uint32_t aw[8];
        grown_armies(s, ch << 4, grow_s, grow_p, aw, sat);
        big16[ch] = big_bits(aw);
        if ((nch & 1) && ch == nch - 1) big16[nch] = 0;
    }
#pragma unroll 1
    for (int p = 0; p < P; ++p) {
        const uint32_t p4 = 0x01010101u * (uint32_t)p;
        uint32_t arm = 0, land = 0;  // arm: times 128 (at most 8 chunks of 16 armies per lane)
#pragma unroll 1
        for (int ch = t.lane; ch < nch; ch += t.width) {
            const int c0 = ch << 4;
            const uint4 O = *reinterpret_cast<const uint4*>(s.owner + c0);
            const uint4 A0 = *reinterpret_cast<const uint4*>(s.army + c0);
            const uint4 A1 = *reinterpret_cast<const uint4*>(s.army + c0 + 8);
            const uint32_t ow[4] = {O.x, O.y, O.z, O.w};
            const uint32_t aw[8] = {A0.x, A0.y, A0.z, A0.w, A1.x, A1.y, A1.z, A1.w};
            uint32_t z[4];  // 0x80 where the owner (-1 .. 7) is p
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                z[k] = ~(((ow[k] ^ p4) & 0x0F0F0F0Fu) + 0x7F7F7F7Fu) & 0x80808080u;
                arm = __dp2a_hi(aw[2 * k + 1], z[k], __dp2a_lo(aw[2 * k], z[k], arm));
            }
            const uint32_t own = (collect_lo(z[0], z[1]) >> 7) | (collect_lo(z[2], z[3]) << 1);
            own16[p * st2 + ch] = (uint16_t)own;
            land += __popc(own);
            if ((nch & 1) && ch == nch - 1) own16[p * st2 + nch] = 0;
        }
        arm = t.reduce_add(arm >> 7);
        land = t.reduce_add(land);
        if (t.lane == 0) {
            s.misc[8 + p] = (int)land;
            s.misc[16 + p] = (int)arm;
        }
    }
    t.sync();
    return total_saturated(sat, grow_s || grow_p, t);
}

// IN_TURN: games of more than four players take them one after another.  At
// the work list's 80 registers eight players at once are faster (32,768 mixed
// games: 216.6 against 223.7 us per frame, 16-frame rollouts of 4,096 585
// against 601 us), at the 64 of the per-frame kernels, where they spill,
// slower (4,096 30x30 free-for-all games: 51.3 against 50.5 us), and a
// multi-frame kernel that never runs them is faster without their code (64
// frames of 1,024 1v1 games: 293 against 286 us).
template <bool IN_TURN, class T>
__device__ __forceinline__ uint32_t cell_pass(const Game& g, const Smem& s, bool grow_s, bool grow_p, const T& t) {
    if constexpr (T::width < 32) {  // groups narrower than a warp only run games of at most kPairMaxPlayers
        static_assert(kPairMaxPlayers == 2, "narrow groups compile the two-player cell pass only");
        return chunk_pass<2, T>(g, s, grow_s, grow_p, t);
    } else {
        if (g.P <= 2) return chunk_pass<2, T>(g, s, grow_s, grow_p, t);
        if (g.P <= 4) return chunk_pass<4, T>(g, s, grow_s, grow_p, t);
        if constexpr (IN_TURN)
            return chunk_pass_in_turn(g, s, grow_s, grow_p, t);
        else
            return chunk_pass<8, T>(g, s, grow_s, grow_p, t);
    }
}

// ---- fog: 3x3 dilation of the (team) ownership bitset (Sec. IV-B) ----------
// This pass widens each player's (team's) cells by one column to either side;
// output_pass joins the row above and below as it reads a chunk's bits, for
// which the words around a player's are zero (zero_guards).  Words of all
// players share one loop, so that narrow groups fill their lanes.  Against a
// second pass over the words for the rows and a loop per player: step of
// 65,536 24x24 1v1 games 129.2 -> 120.9 us, of 32,768 mixed games 218.6 ->
// 201.2 us, 16 frames of 32,768 ragged games 870 -> 828 us.
template <class T>
__device__ __forceinline__ void zero_guards(const Game& g, const Smem& s, const T& t) {
    const int vs = s.vstride();
    if (t.lane < kVisGuard) s.vis[t.lane - kVisGuard] = 0u;
    for (int i = t.lane; i < g.P * 2 * kVisGuard; i += t.width) {
        const int p = i / (2 * kVisGuard), k = i & (2 * kVisGuard - 1);
        // past the game's own words, and past those of the carve's largest board (the next player's front)
        s.vis[p * vs + (k < kVisGuard ? g.nw + k : s.stride + k - kVisGuard)] = 0u;
    }
}
template <class T>
__device__ __forceinline__ void fog_pass(const Game& g, const Smem& s, uint32_t alive, const T& t) {
    const int nw = g.nw, st = s.stride, vs = s.vstride();
    const bool team = g.mode == 1;
    int p = 0, w = t.lane;
    while (p < g.P && w >= nw) {
        w -= nw;
        ++p;
    }
    while (p < g.P) {
        const uint32_t* own = s.own + p * st + w;
        const uint32_t* ally = s.own + (p ^ 1) * st + w;
        const uint32_t T0 = own[0] | (team ? ally[0] : 0u);
        const uint32_t Tm = w > 0 ? own[-1] | (team ? ally[-1] : 0u) : 0u;
        const uint32_t Tp = w + 1 < nw ? own[1] | (team ? ally[1] : 0u) : 0u;
        const uint32_t L = __funnelshift_l(Tm, T0, 1);  // bit c <- cell c-1
        const uint32_t R = __funnelshift_r(T0, Tp, 1);  // bit c <- cell c+1
        s.vis[p * vs + w] = ((alive >> p) & 1u) ? T0 | (L & ~s.col0[w]) | (R & ~s.colL[w]) : 0u;
        w += t.width;
        while (p < g.P && w >= nw) {
            w -= nw;
            ++p;
        }
    }
    t.sync();
}

// 4 bits -> 4 bytes of 0x01
__device__ __forceinline__ uint32_t spread4(uint32_t nib) { return (nib * 0x00204081u) & 0x01010101u; }
// low nibbles of 4 bytes -> 16 bits (byte k's nibble at bits 4k..4k+3): a dot
// product with 1, 16, 256, 4096
__device__ __forceinline__ uint32_t nibbles16(uint32_t x) {
    x &= 0x0F0F0F0Fu;
    return __dp2a_hi(0x10000100u, x, __dp2a_lo(0x00100001u, x, 0u));
}

// Legal moves of player p in chunk ch as 64 bits, 4 per cell in (cell,
// direction) order: the player owns the cell, it holds at least 2, and the
// neighbour towards the direction is passable.  The caller knows the player
// is alive and the game running.
__device__ __forceinline__ uint64_t chunk_legal64(const Smem& s, int p, int ch) {
    const int c0 = ch << 4;
    const int wi = c0 >> 5, sh = c0 & 16;
    const uint32_t mv = ((s.own[p * s.stride + wi] & s.big[wi]) >> sh) & 0xFFFFu;
    const uint4 T = *reinterpret_cast<const uint4*>(s.terrain + c0);
    const uint32_t tw[4] = {T.x, T.y, T.z, T.w};
    uint32_t nib[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) nib[k] = ((tw[k] >> 2) & 0x0F0F0F0Fu) & (spread4((mv >> (4 * k)) & 15u) * 0x0Fu);
    const uint32_t lo = nibbles16(nib[0]) | (nibbles16(nib[1]) << 16);
    const uint32_t hi = nibbles16(nib[2]) | (nibbles16(nib[3]) << 16);
    return ((uint64_t)hi << 32) | lo;
}

// ---- observation + mask chunks of 16 cells (Sec. IV-B, App. A, Sec. IV-G) --
// WRITE: store the planes; COUNT: legal (cell, direction) pairs per chunk.
template <bool WRITE, bool COUNT, class G>
__device__ void output_pass(const KArgs& a, const Game& g, const Smem& s, uint32_t alive, bool finished, const G& t,
                            int64_t frame_off) {
    const int nch = g.nch, st = s.stride, vs = s.vstride(), P = g.P;
    // a row up or down in 16-cell units and a shift
    const int ua = (g.W + 15) >> 4, us = 16 * ua - g.W, da = g.W >> 4, ds = g.W & 15;
    const uint32_t tail = (1u << (((g.N - 1) & 15) + 1)) - 1u;  // the last chunk's cells on the board
    int p = 0, ch = t.lane;
    while (p < P && ch >= nch) {
        ch -= nch;
        ++p;
    }
    while (p < P) {
        const int c0 = ch << 4;
        const int wi = c0 >> 5, sh = c0 & 16;
        uint32_t mv = 0;
        if (!finished && ((alive >> p) & 1u)) mv = ((s.own[p * st + wi] & s.big[wi]) >> sh) & 0xFFFFu;
        const uint4 T = *reinterpret_cast<const uint4*>(s.terrain + c0);
        const uint32_t tw[4] = {T.x, T.y, T.z, T.w};
        uint32_t om[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t dpb = ((tw[k] >> 2) & 0x0F0F0F0Fu) * 0x11u;
            om[k] = dpb & (spread4((mv >> (4 * k)) & 15u) * 0xFFu);
        }
        if (COUNT) {
            // legal pairs: either nibble of each mask byte, two words' side by side
            s.cnt[p * nch + ch] = (uint8_t)(__popc((om[0] & 0x0F0F0F0Fu) | (om[1] & 0xF0F0F0F0u)) +
                                            __popc((om[2] & 0x0F0F0F0Fu) | (om[3] & 0xF0F0F0F0u)));
        }
        if (WRITE) {
            const uint16_t* h = reinterpret_cast<const uint16_t*>(s.vis + p * vs) + ch;
            const uint32_t up = ((uint32_t)h[-ua] | ((uint32_t)h[1 - ua] << 16)) >> us;  // cells c0 - W ..
            const uint32_t dn = ((uint32_t)h[da] | ((uint32_t)h[da + 1] << 16)) >> ds;   // cells c0 + W ..
            const uint32_t vis16 = (h[0] | up | dn) & (ch == nch - 1 ? tail : 0xFFFFu);
            const uint4 A0 = *reinterpret_cast<const uint4*>(s.army + c0);
            const uint4 A1 = *reinterpret_cast<const uint4*>(s.army + c0 + 8);
            const uint4 O = *reinterpret_cast<const uint4*>(s.owner + c0);
            const uint32_t aw[8] = {A0.x, A0.y, A0.z, A0.w, A1.x, A1.y, A1.z, A1.w};
            const uint32_t ow[4] = {O.x, O.y, O.z, O.w};
            uint32_t oa[8], oo[4], ot[4], ov[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t v1 = spread4((vis16 >> (4 * k)) & 15u);
                const uint32_t bm = v1 * 0xFFu;
                oo[k] = (ow[k] & bm) | (0xFEFEFEFEu & ~bm);
                const uint32_t tt = tw[k] & 0x03030303u;
                const uint32_t fogc = ((tt ^ (tt >> 1)) & 0x01010101u) | 0x04040404u;
                ot[k] = (tt & bm) | (fogc & ~bm);
                ov[k] = v1;
                oa[2 * k] = aw[2 * k] & __byte_perm(bm, 0, 0x1100);
                oa[2 * k + 1] = aw[2 * k + 1] & __byte_perm(bm, 0, 0x3322);
            }
            const int64_t off = frame_off + g.plane_off + (int64_t)p * g.Npad + c0;
            uint4* pa = reinterpret_cast<uint4*>(a.obs_army + off);
            __stcs(pa, make_uint4(oa[0], oa[1], oa[2], oa[3]));
            __stcs(pa + 1, make_uint4(oa[4], oa[5], oa[6], oa[7]));
            __stcs(reinterpret_cast<uint4*>(a.obs_owner + off), make_uint4(oo[0], oo[1], oo[2], oo[3]));
            __stcs(reinterpret_cast<uint4*>(a.obs_terrain + off), make_uint4(ot[0], ot[1], ot[2], ot[3]));
            __stcs(reinterpret_cast<uint4*>(a.obs_vis + off), make_uint4(ov[0], ov[1], ov[2], ov[3]));
            __stcs(reinterpret_cast<uint4*>(a.mask + off), make_uint4(om[0], om[1], om[2], om[3]));
        }
        ch += t.width;
        while (p < P && ch >= nch) {
            ch -= nch;
            ++p;
        }
    }
    t.sync();
}

template <int LW>
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x, const Grp<LW>& t) {
#pragma unroll
    for (int o = 1; o < LW; o <<= 1) {
        const uint32_t y = t.shfl_up(x, o);
        if (t.lane >= o) x += y;
    }
    return x;
}

// ---- benchmark policy: uniform legal (cell, direction), split p = 0.2 -------
// Needs the chunk counts of output_pass<*, true>.  Players are scanned two at
// a time (16-bit counts packed in one 32-bit scan: a board has at most
// 4 x 4096 legal pairs); lane p then walks the chunks of the lane holding
// player p's pair and selects the bit by popcount bisection, every player at
// once.
// u: on lanes 2p and 2p + 1 player p's two draws (policy_draws).
// Returns, on lane p < P, player p's action; DIRECT also stores it.
__device__ __forceinline__ uint32_t policy_draws(const KArgs& a, const Game& g, uint32_t frame, uint64_t gid, int lane) {
    if (lane >= 2 * g.P) return 0u;
    return hdraw(hkey(a.policy_seed, gid, frame, (uint64_t)(lane >> 1)), (uint64_t)(lane & 1));
}
template <bool DIRECT, int LW>
__device__ int32_t policy_pass(const KArgs& a, const Game& g, const Smem& s, uint32_t alive, bool finished, uint32_t u,
                               const Grp<LW>& t) {
    const int nch = g.nch;
    const int cpl = (nch + LW - 1) / LW;  // consecutive chunks per lane
    const int c_lo = t.lane * cpl;
    const int c_hi = min(c_lo + cpl, nch);
    int my_lane = -1;     // the lane whose chunks hold this lane's player's pair
    uint32_t my_rank = 0;  // the pair's index among that lane's
    bool my_half = false;
    for (int p0 = 0; p0 < g.P; p0 += 2) {
        uint32_t mine = 0;
        for (int c = c_lo; c < c_hi; ++c) {
            mine += s.cnt[p0 * nch + c];
            if (p0 + 1 < g.P) mine += (uint32_t)s.cnt[(p0 + 1) * nch + c] << 16;
        }
        const uint32_t incl2 = warp_incl_scan(mine, t);
        const uint32_t total2 = t.shfl(incl2, LW - 1);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int p = p0 + q;
            if (p >= g.P) break;
            const uint32_t total = (total2 >> (16 * q)) & 0xFFFFu;
            const uint32_t incl = (incl2 >> (16 * q)) & 0xFFFFu;
            const uint32_t u1 = t.shfl(u, 2 * p), u2 = t.shfl(u, 2 * p + 1);
            if (total > 0) {
                const uint32_t j = (uint32_t)uniform_below(u1, total);
                const int L = __ffs(t.ballot(incl > j)) - 1;
                const uint32_t rank = j - t.shfl(incl - ((mine >> (16 * q)) & 0xFFFFu), L);
                if (t.lane == p) {
                    my_lane = L;
                    my_rank = rank;
                    my_half = u2 < kSplitThresh;
                }
            }
        }
    }
    int32_t action = 0;
    if (my_lane >= 0 && !finished && ((alive >> t.lane) & 1u)) {
        // the chunk first, so that the players' lanes part only in this loop
        const uint8_t* cnt = s.cnt + t.lane * nch;
        int c = my_lane * cpl;
        for (uint32_t n = cnt[c]; my_rank >= n; n = cnt[++c]) my_rank -= n;
        const uint64_t m = chunk_legal64(s, t.lane, c);
        uint32_t x = (uint32_t)m;
        int bit = 0;
        const uint32_t nlo = __popc(x);
        if (my_rank >= nlo) {
            my_rank -= nlo;
            x = (uint32_t)(m >> 32);
            bit = 32;
        }
#pragma unroll
        for (int w = 16; w >= 1; w >>= 1) {
            const uint32_t cw = __popc(x & ((1u << w) - 1u));
            if (my_rank >= cw) {
                my_rank -= cw;
                x >>= w;
                bit += w;
            }
        }
        const int d = bit & 3;
        action = (c * 16 + (bit >> 2)) * 9 + (my_half ? 5 + d : 1 + d);
    }
    if (DIRECT && t.lane < g.P) a.next_actions[g.player_off + t.lane] = action;
    return action;
}

// All of a board's 16-byte vectors (army, owner, terrain) copied global ->
// shared with cp.async: every copy is in flight at once and none passes
// through registers.  board_wait() completes them (a hardware wait).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
template <class T>
__device__ __forceinline__ void board_issue(const KArgs& a, const Game& g, const Smem& s, const T& t) {
    const int n16 = g.Npad >> 4;  // 16-byte vectors per int8 plane
    const uint4* ga = reinterpret_cast<const uint4*>(a.army + g.cell_off);
    const uint4* go = reinterpret_cast<const uint4*>(a.owner + g.cell_off);
    const uint4* gt = reinterpret_cast<const uint4*>(a.terrain + g.cell_off);
    uint4* sa = reinterpret_cast<uint4*>(s.army);
    uint4* so = reinterpret_cast<uint4*>(s.owner);
    uint4* st = reinterpret_cast<uint4*>(s.terrain);
    for (int v = t.lane; v < 2 * n16; v += t.width) cp_async16(sa + v, ga + v);
    for (int v = t.lane; v < n16; v += t.width) {
        cp_async16(so + v, go + v);
        cp_async16(st + v, gt + v);
    }
    if (a.do_outputs) {
        // the board's first- and last-column bitsets for the fog pass, in
        // the same group of copies (8-byte pairs of words: both regions and
        // both table rows are 8-byte aligned, the region holds an even count)
        const uint32_t* c0 = g_columns[g.W - 1][0];
        const uint32_t* cl = g_columns[g.W - 1][1];
        for (int v = t.lane; 2 * v < g.nw; v += t.width) {
            cp_async8(s.col0 + 2 * v, c0 + 2 * v);
            cp_async8(s.colL + 2 * v, cl + 2 * v);
        }
    }
}
template <class T>
__device__ __forceinline__ void board_wait(const T& t) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    t.sync();
}

template <class T>
__device__ __forceinline__ void store_board(const KArgs& a, const Game& g, const Smem& s, const T& t) {
    const int n16 = g.Npad >> 4;
    uint4* ga = reinterpret_cast<uint4*>(a.army + g.cell_off);
    uint4* go = reinterpret_cast<uint4*>(a.owner + g.cell_off);
    uint4* gt = reinterpret_cast<uint4*>(a.terrain + g.cell_off);
    const uint4* sa = reinterpret_cast<const uint4*>(s.army);
    const uint4* so = reinterpret_cast<const uint4*>(s.owner);
    const uint4* st = reinterpret_cast<const uint4*>(s.terrain);
    for (int v = t.lane; v < 2 * n16; v += t.width) ga[v] = sa[v];
    for (int v = t.lane; v < n16; v += t.width) {
        go[v] = so[v];
        gt[v] = st[v];
    }
}

}  // namespace

namespace {


// The end of a frame: outputs, the benchmark policy (whose actions, on lane
// p player p's, come back in my_act) and, per frame, the scalar outputs.
// columns: the board's column bitsets are in shared memory already.
template <bool MULTI, int LW, bool UNI>
__device__ __forceinline__ void finish_frame(const KArgs& a, const Game& g, const Smem& s, const int gidx, int f,
                                             bool columns, uint32_t alive, bool fin, uint32_t frame, float my_reward,
                                             uint32_t done, int32_t& my_act, const Grp<LW>& t) {
    if constexpr (MULTI) {
        // reward and done before the output passes and the scoreboard
        // as soon as the fog pass has counted the land: fewer values
        // live through the passes (measured faster in multi-frame
        // launches, slower per frame)
        if (a.do_outputs) {
            const int64_t soff = (int64_t)f * a.slot_stride;
            if (t.lane < g.P) a.reward[soff + g.player_off + t.lane] = my_reward;
            if (t.lane == 0) a.done[(int64_t)f * a.game_stride + gidx] = (uint8_t)done;
        }
    }
    if (a.do_outputs) {
        const int64_t poff = (int64_t)f * a.plane_stride;
        const int64_t soff = (int64_t)f * a.slot_stride;
        if (!columns) column_pass(g, s, t);
        fog_pass(g, s, alive, t);
        if constexpr (MULTI) {
            if (t.lane < g.P) {
                a.scoreboard[2 * (soff + g.player_off + t.lane) + 0] = s.misc[8 + t.lane];
                a.scoreboard[2 * (soff + g.player_off + t.lane) + 1] = s.misc[16 + t.lane];
            }
        }
        if (a.next_actions)
            output_pass<true, true>(a, g, s, alive, fin, t, poff);
        else
            output_pass<true, false>(a, g, s, alive, fin, t, poff);
        if constexpr (!MULTI) {
            if (t.lane < g.P) {
                a.reward[soff + g.player_off + t.lane] = my_reward;
                a.scoreboard[2 * (soff + g.player_off + t.lane) + 0] = s.misc[8 + t.lane];
                a.scoreboard[2 * (soff + g.player_off + t.lane) + 1] = s.misc[16 + t.lane];
            }
            if (t.lane == 0) a.done[(int64_t)f * a.game_stride + gidx] = (uint8_t)done;
        }
    } else if (a.next_actions) {
        output_pass<false, true>(a, g, s, alive, fin, t, 0);
    }
    if (a.next_actions)
        my_act = policy_pass<!MULTI, LW>(a, g, s, alive, fin, policy_draws(a, g, frame, game_id_of<UNI>(a, gidx), t.lane), t);
}

__device__ __forceinline__ void store_scalars(const KArgs& a, int gidx, uint32_t turn, uint32_t frame, uint32_t epoch,
                                              uint32_t alive, uint32_t finished, uint32_t invalid, uint32_t saturated,
                                              uint32_t err) {
    uint4* dst = reinterpret_cast<uint4*>(a.scal + gidx);
    dst[0] = make_uint4(turn, frame, epoch, alive);
    dst[1] = make_uint4(finished, invalid, saturated, err);
}

template <int LW>
__device__ __forceinline__ Game group_game(Game g) {
    if constexpr (LW < 32) {
        // narrow groups run only two-player games without teams: 1v1, or a
        // two-player free-for-all, whose rules are the same
        g.P = kPairMaxPlayers;
        g.mode = 0;
    }
    return g;
}

// The rest of a per-frame launch for a game that gets a new map (create,
// reset, a finished game): the map, the frame's end, the state stored.  Nothing returns to the step, so the step
// kernel keeps no value alive across a call: with the generator as a call
// that returned, its registers set the spills of the frames without a reset
// (65,536 1v1 games on 24x24: 135.5 us per launch with the earlier, smaller
// generator returning, 132.5 us so; with the spawn options compiled in,
// 185.7 us returning and 136.6 us so).
// sc: the counters with the frame and epoch of the new state.
template <int LW, bool UNI, bool SPAWN, int ROW_BITS>
__device__ __noinline__ void new_map(const KArgs& a, int gidx, char* warp_base, uint32_t geom, int warp_lane,
                                     uint32_t frame, uint32_t epoch, uint32_t invalid, uint32_t saturated, uint32_t err,
                                     float my_reward, uint32_t done) {
    const Grp<LW> t(warp_lane);
    const Game g = group_game<LW>(game_of<UNI>(a, gidx));
    const Smem s = carve_geom(warp_base, geom);
    if (a.op != OP_STEP && a.do_outputs) zero_guards(g, s, t);  // the step has set them
    generate_body<LW, SPAWN, ROW_BITS>(a, g, s, game_id_of<UNI>(a, gidx), epoch, t);
    const uint32_t alive = (1u << g.P) - 1u;
    cell_pass<true>(g, s, false, false, t);
    int32_t act = 0;
    finish_frame<false, LW, UNI>(a, g, s, gidx, 0, a.op == OP_STEP, alive, false, frame, my_reward, done, act, t);
    t.sync();
    store_board(a, g, s, t);
    if (t.lane == 0) store_scalars(a, gidx, 0u, frame, epoch, alive, 0u, invalid, saturated, err);
}

// geom: the packed carve geometry of the game's warp region, or 0 for the
// launch's own (kernel parameters); only the cold out-of-line paths use it.
template <bool MULTI, bool SPAWN, bool IN_TURN, int LW, bool UNI>
__device__ __forceinline__ void run_game(const KArgs& a, const Smem& s, char* warp_base, const uint32_t geom,
                                         const int gidx, const Grp<LW>& t) {
    const Game g = group_game<LW>(game_of<UNI>(a, gidx));
    GameScalars* sc = a.scal + gidx;

    uint4 s0, s1;
    if constexpr (!MULTI) {
        if (a.op == OP_CREATE || a.op == OP_RESET) {
            s0 = s1 = make_uint4(0, 0, 0, 0);
            if (a.op == OP_RESET) {
                s0 = *reinterpret_cast<const uint4*>(sc);
                s1 = *(reinterpret_cast<const uint4*>(sc) + 1);
                s0.z += 1;
            }
            const uint32_t whole = geom ? geom : geom_of(a);
            if constexpr (SPAWN && UNI) {
                if (wide_rows(g))
                    new_map<LW, UNI, SPAWN, 64>(a, gidx, warp_base, whole, t.lane + t.shift, s0.y, s0.z, s1.y, s1.z, s1.w, 0.0f, 0u);
                else
                    new_map<LW, UNI, SPAWN, 32>(a, gidx, warp_base, whole, t.lane + t.shift, s0.y, s0.z, s1.y, s1.z, s1.w, 0.0f, 0u);
            } else {
                new_map<LW, UNI, SPAWN, 0>(a, gidx, warp_base, whole, t.lane + t.shift, s0.y, s0.z, s1.y, s1.z, s1.w, 0.0f, 0u);
            }
            return;
        }
    }
    // every global load of the step is issued here, before any is used
    board_issue(a, g, s, t);
    if (a.do_outputs) zero_guards(g, s, t);
    s0 = *reinterpret_cast<const uint4*>(sc);
    s1 = *(reinterpret_cast<const uint4*>(sc) + 1);
    // player `lane`'s action for the next step (frame 0: from the caller)
    int32_t my_act = (a.op == OP_STEP && t.lane < g.P) ? a.actions[g.player_off + t.lane] : 0;
    board_wait(t);

    uint32_t turn = s0.x, frame = s0.y, epoch = s0.z, alive = s0.w;
    uint32_t finished = s1.x, invalid = s1.y, saturated = s1.z;
    const uint32_t err = s1.w;
    bool wrote_state = false;

    if constexpr (!MULTI) {
        if (a.op == OP_DERIVE) {  // recompute cached per-map bits after a state upload
            derive_passable(g, s, t);
            wrote_state = true;
        }
    }
    const int frames = (MULTI && a.op == OP_STEP) ? a.frames : 1;
    for (int f = 0; f < frames; ++f) {
        float my_reward = 0.0f;
        uint32_t done = 0;
        if (a.op == OP_STEP && !finished) {
            if (MULTI && a.action_log && t.lane < g.P)
                a.action_log[(int64_t)f * a.slot_stride + g.player_off + t.lane] = my_act;
            uint32_t eliminated = 0, inv0 = 0, sat0 = 0;
            play_moves(g, s, t, turn, my_act, alive, eliminated, inv0, sat0);
            invalid += t.shfl(inv0, 0);
            saturated += t.shfl(sat0, 0);
            turn += 1;
            saturated += cell_pass<IN_TURN>(g, s, (turn % 2u) == 0u, (turn % 50u) == 0u, t);
            done = outcome(a, g, t.lane, turn, alive, eliminated, my_reward);
            if (done) {
                if (a.auto_reset) {
                    epoch += 1;
                    if constexpr (!MULTI) {
                        const uint32_t whole = geom ? geom : geom_of(a);
                        if constexpr (SPAWN && UNI) {
                            if (wide_rows(g))
                                new_map<LW, UNI, SPAWN, 64>(a, gidx, warp_base, whole, t.lane + t.shift, frame + 1, epoch, invalid,
                                                            saturated, err, my_reward, done);
                            else
                                new_map<LW, UNI, SPAWN, 32>(a, gidx, warp_base, whole, t.lane + t.shift, frame + 1, epoch, invalid,
                                                            saturated, err, my_reward, done);
                        } else {
                            new_map<LW, UNI, SPAWN, 0>(a, gidx, warp_base, whole, t.lane + t.shift, frame + 1, epoch, invalid,
                                                       saturated, err, my_reward, done);
                        }
                        return;
                    } else {
                        generate<LW, UNI, SPAWN>(a, gidx, warp_base, geom ? geom : geom_of(a),
                                                 game_id_of<UNI>(a, gidx), epoch, t.lane + t.shift);
                        turn = 0;
                        alive = (1u << g.P) - 1u;
                        cell_pass<IN_TURN>(g, s, false, false, t);
                    }
                } else {
                    finished = 1;
                }
            }
            wrote_state = true;
        } else {
            // observe, policy, derive, or a frozen game
            saturated += cell_pass<IN_TURN>(g, s, false, false, t);
        }
        if (a.op == OP_STEP) frame += 1;
        finish_frame<MULTI, LW, UNI>(a, g, s, gidx, f, true, alive, finished != 0, frame, my_reward, done, my_act, t);
    }
    if (MULTI && a.next_actions && t.lane < g.P) a.next_actions[g.player_off + t.lane] = my_act;
    if (wrote_state) {
        t.sync();
        store_board(a, g, s, t);
    }
    if (t.lane == 0 && a.op != OP_OBSERVE && a.op != OP_POLICY)
        store_scalars(a, gidx, turn, frame, epoch, alive, finished, invalid, saturated, err);
}


}  // namespace

// One game per group of LW lanes (32: a warp; 16 or 8: two or four games per
// warp); groups walk the item list with a grid stride.  MULTI: several frames
// per launch (rollouts) with the board kept in shared memory.  UNI: every
// game of the launch has the launch's shape (uniform batches).
// Register budget: 64 per thread (4 CTAs of 8 warps per SM) for the per-frame
// form; the multi-frame form keeps more state live across frames and runs
// best with 80 (3 CTAs).
template <bool MULTI, bool SPAWN, int LW, bool UNI>
__global__ void __launch_bounds__(256, MULTI ? 3 : 4) k_generals(const KArgs a) {
    chain_entry();
    extern __shared__ __align__(16) char smem_raw[];
    constexpr int kGroups = 32 / LW;  // games per warp
    const int wl = threadIdx.x & 31;
    const Grp<LW> t(wl);
    const int grp = (threadIdx.x >> 5) * kGroups + wl / LW;  // group in the CTA
    const int gpc = (blockDim.x >> 5) * kGroups;                                // groups per CTA
    char* warp_base = smem_raw + grp * a.warp_smem;
    const Smem s = carve(warp_base, a);
    if constexpr (!MULTI) {  // the grid covers every item
        const int item = blockIdx.x * gpc + grp;
        if (item >= a.n_items) return;
        const int gidx = a.list ? a.list[item] : item;
        if (gidx < 0 || gidx >= a.n_games) return;
        run_game<MULTI, SPAWN, true, LW, UNI>(a, s, warp_base, 0u, gidx, t);
    } else {
        for (int item = blockIdx.x * gpc + grp; item < a.n_items; item += gridDim.x * gpc) {
            const int gidx = a.list ? a.list[item] : item;
            if (gidx < 0 || gidx >= a.n_games) continue;
            t.sync();
            run_game<MULTI, SPAWN, true, LW, UNI>(a, s, warp_base, 0u, gidx, t);
        }
    }
}

// Every size bucket of a ragged or mixed batch in one persistent launch.  A
// CTA takes one work item at a time (an atomic counter over a list ordered
// largest boards first), carves its shared memory for that item's bucket and
// runs one game per lane group: two per warp for two-player buckets of small
// boards, one per warp otherwise.  The CTA waits at a barrier between items,
// so that the next item may carve the same bytes differently.
// Three CTAs per SM (80 registers): with four (64), the eight-player passes
// spill and an item's shared memory holds fewer large boards (32,768 mixed
// games of 20..40 a side: 216.6 against 247.8 us per frame).
template <bool MULTI, bool SPAWN>
__global__ void __launch_bounds__(256, 3) k_worklist(const KArgs a, const WArgs w) {
    chain_entry();
    extern __shared__ __align__(16) char smem_raw[];
    __shared__ int s_item;
    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(w.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= w.n_items) {  // the same for every thread of the CTA
            // the last CTA to run out zeroes the counters for the next launch:
            // every CTA has drawn its last index by then, and a chained launch
            // reads them only after this grid has completed
            if (threadIdx.x == 0) {
                __threadfence();  // this CTA's last draw is ordered before its exit count
                if (atomicAdd(w.counter + 1, 1) == (int)gridDim.x - 1) {
                    __threadfence();  // and every other CTA's before these stores
                    w.counter[0] = 0;
                    w.counter[1] = 0;
                }
            }
            return;
        }
        const WorkItem item = w.items[it];
        const BucketGeom bg = w.geoms[item.bucket];
        if (bg.lw == 16) {
            const Grp<16> t(wl);
            const int grp = 2 * warp + (wl >> 4);
            if (grp < item.count) {
                char* base = smem_raw + grp * bg.group_smem;
                run_game<MULTI, SPAWN, false, 16, false>(a, carve_geom(base, bg.geom), base, bg.geom,
                                                  w.order[item.first + grp], t);
            }
        } else {
            const Grp<32> t(wl);
            if (warp < item.count) {
                char* base = smem_raw + warp * bg.group_smem;
                run_game<MULTI, SPAWN, false, 32, false>(a, carve_geom(base, bg.geom), base, bg.geom,
                                                  w.order[item.first + warp], t);
            }
        }
        __syncthreads();
    }
}

namespace {

__global__ void k_columns() {
    const int W = blockIdx.x + 1;
    for (int w = threadIdx.x; w < kColWords; w += blockDim.x) {
        uint32_t c0 = 0, cl = 0;
        for (int b = 0; b < 32; ++b) {
            const int c = 32 * w + b;
            if (c % W == 0) c0 |= 1u << b;
            if (c % W == W - 1) cl |= 1u << b;
        }
        g_columns[W - 1][0][w] = c0;
        g_columns[W - 1][1][w] = cl;
    }
}

// Fill this translation unit's column table; synchronous.  Returns a cudaError_t.
int fill_columns() {
    k_columns<<<kMaxSide, 128>>>();
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}

}  // namespace

using StepKernel = void (*)(KArgs);
using WorklistKernel = void (*)(KArgs, WArgs);

}  // namespace gk
