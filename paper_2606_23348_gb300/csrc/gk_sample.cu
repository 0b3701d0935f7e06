// Policy sampling over the H x W x 9 action space (Sec. IV-G; the policy
// head's H x W x 9 distribution, App. C) and the expanded legal mask.
//
// Legal entries of player p: (c, pass) where p owns c; (c, 1 + d) all-but-one
// and (c, 5 + d) half towards d where the move is legal (p alive and owning
// c, at least 2 units, the neighbour exists and is not a mountain, the game
// not finished).  Sampling is an exact integer inverse CDF, so that the same
// logits and seed pick the same action on every device:
//   m = max legal logit; w_e = floor(E(l_e - m) * 2^24) with E the
//   reproducible exponential below; S = sum of w_e (64-bit, exact);
//   r = floor(d * S / 2^64) for the 64-bit draw d = counter hash of (seed,
//   global game id, frame of the consuming step, p) at index 7; the action
//   is the first legal entry in index order whose running sum exceeds r.
// E(x) = 2^n * P(f): t = x * log2(e) in float, n = floor(t), f = t - n, P the
// degree-7 Taylor polynomial of 2^f (sum of (f ln 2)^k / k!) in Horner form
// with fused multiply-adds, 0 below t = -25.  Every operation is an IEEE
// single-precision operation with round-to-nearest written out explicitly
// (no contraction), so the weights are bit-reproducible.
//
// One warp per player (k_sample_slots), the expanded mask a CTA per game
// (k_mask9), both at once in one launch (k_sample_mask).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "gk_internal.h"

namespace gk {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr float kNegInf = -__builtin_huge_valf();
constexpr float kLowest = -3.402823466e38f;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t stream_out(uint64_t s, uint64_t n) { return mix64(s + (n + 1) * kGamma); }
__device__ __forceinline__ uint64_t hkey(uint64_t s, uint64_t a, uint64_t b, uint64_t c) {
    return stream_out(stream_out(stream_out(s, a), b), c);
}

// weight of a legal entry: floor(E(l - m) * 2^24).  E = P * 2^n exactly
// (n >= -25, P in [1, 2)), so the floor is P's 24-bit significand shifted
// right by -(n + 1) bits; equal to the float floor of the exact product.
__device__ __forceinline__ uint32_t weight_shift(float l, float m) {
    const float t = __fmul_rn(__fsub_rn(l, m), 1.4426950408889634f);
    if (t < -25.0f) return 0u;
    const float nf = floorf(t);
    const float f = __fsub_rn(t, nf);
    float p = 1.5252733804059838e-05f;
    p = __fmaf_rn(p, f, 0.00015403530393381606f);
    p = __fmaf_rn(p, f, 0.0013333558146428441f);
    p = __fmaf_rn(p, f, 0.009618129107628477f);
    p = __fmaf_rn(p, f, 0.055504108664821576f);
    p = __fmaf_rn(p, f, 0.2402265069591007f);
    p = __fmaf_rn(p, f, 0.6931471805599453f);
    p = __fmaf_rn(p, f, 1.0f);
    const int n = (int)nf;                                          // -25 .. 0
    const uint32_t sig = (__float_as_uint(p) & 0x7FFFFFu) | 0x800000u;  // P * 2^23
    return n >= 0 ? sig << 1 : sig >> (-(n + 1));
}

// Two weights at once: the same single-precision operations as weight_shift,
// issued as packed pairs (each half an IEEE operation of its own), for finite
// m >= l (l = -inf included: weight 0).  floor(t) is the round-down sum with
// 1.5 * 2^23, whose low bits are the integer (no conversion instruction), and
// the shift 24-bit significand << 1 >> -n is 0 from n = -26 on by itself.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
__device__ __forceinline__ float lo2(uint64_t x) { return __uint_as_float((uint32_t)x); }
__device__ __forceinline__ float hi2(uint64_t x) { return __uint_as_float((uint32_t)(x >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2_down(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t both(float x) { return pack2(x, x); }
constexpr float kFloorMagic = 12582912.0f;  // 1.5 * 2^23, bits 0x4B400000
__device__ __forceinline__ uint32_t weight_bits(float p, float r) {
    // P in [1, 2) (at most 1.9999988, at f = 1): its significand << 1 from the bits 0x3F800000 + mantissa
    const uint32_t sig = 2u * __float_as_uint(p) + 0x82000000u;
    return __funnelshift_rc(sig, 0u, 0x4B400000u - __float_as_uint(r));
}
// sum of the weights of l0 and l1
__device__ __forceinline__ uint32_t weight_pair(float l0, float l1, uint64_t minus_m) {
    uint64_t t = mul2(add2(pack2(l0, l1), minus_m), both(1.4426950408889634f));
    t = pack2(fmaxf(lo2(t), -64.0f), fmaxf(hi2(t), -64.0f));
    const uint64_t r = add2_down(t, both(kFloorMagic));
    const uint64_t f = add2(t, fma2(r, both(-1.0f), both(kFloorMagic)));
    uint64_t p = both(1.5252733804059838e-05f);
    p = fma2(p, f, both(0.00015403530393381606f));
    p = fma2(p, f, both(0.0013333558146428441f));
    p = fma2(p, f, both(0.009618129107628477f));
    p = fma2(p, f, both(0.055504108664821576f));
    p = fma2(p, f, both(0.2402265069591007f));
    p = fma2(p, f, both(0.6931471805599453f));
    p = fma2(p, f, both(1.0f));
    return weight_bits(lo2(p), lo2(r)) + weight_bits(hi2(p), hi2(r));
}
// sum of the weights of one cell's nine entries (-inf: illegal)
__device__ __forceinline__ uint32_t cell_weight(const float (&v)[9], float m) {
    const uint64_t mm = both(-m);
    uint32_t w = 0u;
#pragma unroll
    for (int k = 0; k < 8; k += 2) w += weight_pair(v[k], v[k + 1], mm);
    return w + weight_pair(v[8], kNegInf, mm);
}
// of two cells
__device__ __forceinline__ uint32_t cell_weight2(const float (&v)[9], const float (&u)[9], float m) {
    const uint64_t mm = both(-m);
    uint32_t w = 0u;
#pragma unroll
    for (int k = 0; k < 9; ++k) w += weight_pair(v[k], u[k], mm);
    return w;
}

// legal entries of one cell for player p as bits 0..8 (entry k of the cell)
__device__ __forceinline__ uint32_t legal9(int own_p, int army, uint32_t terrain, bool moves) {
    if (!own_p) return 0u;
    uint32_t b = 1u;  // pass
    if (moves && army >= 2) {
        const uint32_t dirs = (terrain >> 2) & 0xFu;  // neighbour exists and is not a mountain
        b |= (dirs << 1) | (dirs << 5);
    }
    return b;
}

// a game's description; of a uniform batch without a load, since the loads
// that follow would wait for it
__device__ __forceinline__ GameInfo sample_game(const SArgs& a, int gidx) {
    if (!a.uniform) return a.info[gidx];
    GameInfo gi = a.ushape;
    gi.cell_off = gidx * gi.Npad;
    gi.player_off = gidx * gi.P;
    gi.plane_off = (int64_t)gidx * gi.P * gi.Npad;
    gi.game_id = a.game_id_base + (uint64_t)gidx;
    return gi;
}

__device__ __forceinline__ uint64_t warp_incl64(uint64_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(kAll, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// ---- a warp per player ------------------------------------------------------
// The player's own cells are listed in index order (2 B each in shared
// memory): a lane compares 32 owner bytes, one scan places them all on boards
// of up to 1,024 cells.  Lane l then takes the cells k*l .. k*l + k-1 of the
// list, k = ceil(cells / 32), so that one 64-bit scan of the lanes' weight
// sums gives both S and the lane where the running sum first exceeds r; the
// entry is found with a lane per (cell, entry) of that lane's cells.
// Nothing is staged: armies and terrain are gathered for the own cells only,
// in flight with their logits.  A cell's nine logits start at any multiple of
// 4 bytes, and the three 16-byte vectors around them always hold all nine.
//
// Bound by instructions and L1 wavefronts (65,536 1v1 games of 24x24 at mid-
// game, N(0, 2) logits; the sectors of the own cells' logits and the board
// need 79 us): 270 -> 143.6 us, 1,531 -> 952 warp instructions per player
// (134 us in runs of four players per warp, below),
// against a warp per player that staged the board, loaded each logit by
// itself and summed and scanned every 32 cells; 1,000 such games 7.9 -> 7.4,
// 8,192 mixed games of 20..40 a side 243 -> 51 us (shared memory for eight
// staged players held those to four warps per scheduler).  The other spreads
// were slower at every size measured, 1 to 65,536 games and 15 to 177 own
// cells: 512 games 4.2 us against 6.9 us for a warp per game and 5.6 us for a
// CTA per player with a thread per (cell, entry).
// 36 warps per SM (56 registers): 148 us where 32 gave 157 us and 40, with
// spills, 147 us.
__host__ __device__ __forceinline__ int list_bytes(int npad_max) { return (2 * npad_max + 15) & ~15; }

// bit j = byte j of the 16 owner bytes O (-1 .. 7) equals p
__device__ __forceinline__ uint32_t equal_bytes16(uint4 O, uint32_t p4) {
    const uint32_t o[4] = {O.x, O.y, O.z, O.w};
    uint32_t z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) z[q] = ~(((o[q] ^ p4) & 0x0F0F0F0Fu) + 0x7F7F7F7Fu) & 0x80808080u;  // 0x80 where equal
    // dot products with powers of two collect the bytes' bits (times 128)
    const uint32_t lo = __dp4a(z[1], 0x80402010u, __dp4a(z[0], 0x08040201u, 0u));
    const uint32_t hi = __dp4a(z[3], 0x80402010u, __dp4a(z[2], 0x08040201u, 0u));
    return (lo >> 7) | (hi << 1);
}

// the nine logits of cell c, -inf where illegal
__device__ __forceinline__ void load_cell(float (&v)[9], const float* lg, const int16_t* army, const uint8_t* terrain,
                                          int c, bool moves) {
    const int s = c & 3;  // the cell's logits start s floats into the vectors
    const float4* x = reinterpret_cast<const float4*>(lg + (9 * c - s));
    const float4 a = __ldg(x), b = __ldg(x + 1), d = __ldg(x + 2);
    const int av = __ldg(army + c);
    const uint32_t tb = __ldg(terrain + c);
    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, d.x, d.y, d.z, d.w};
    const uint32_t dirs = moves && av >= 2 ? tb >> 2 : 0u;  // neighbour exists and is not a mountain
    float u[11];
#pragma unroll
    for (int k = 0; k < 11; ++k) u[k] = (s & 1) ? w[k + 1] : w[k];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = (s & 2) ? u[k + 2] : u[k];
#pragma unroll
    for (int d2 = 0; d2 < 4; ++d2) {
        const bool ok = (dirs >> d2) & 1u;
        v[1 + d2] = ok ? v[1 + d2] : kNegInf;
        v[5 + d2] = ok ? v[5 + d2] : kNegInf;
    }
}
// entry e of cell c, -inf where illegal
__device__ __forceinline__ float legal_logit(const float* lg, const int16_t* army, const uint8_t* terrain, int c, int e,
                                             bool moves) {
    const bool ok = e == 0 || (moves && __ldg(army + c) >= 2 && ((uint32_t)__ldg(terrain + c) >> (2 + ((e - 1) & 3))) & 1u);
    return ok ? __ldg(lg + 9 * c + e) : kNegInf;
}
// maximum that is a number only if both are
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float cell_max(const float (&v)[9], float m) {
#pragma unroll
    for (int k = 0; k < 9; ++k) m = max_nan(m, v[k]);
    return m;
}
__device__ __forceinline__ float warp_max_nan(float m) {
    asm("redux.sync.max.NaN.f32 %0, %0, 0xffffffff;" : "+f"(m));
    return m;
}

// the draw of player p
__device__ __forceinline__ uint64_t player_draw(const SArgs& a, const GameInfo& gi, const GameScalars& sc, int p) {
    return stream_out(hkey(a.seed, gi.game_id, sc.frame, (uint64_t)p), 7);
}

// player p's action in game gidx from its draw d, by one warp; list: its shared memory
__device__ __forceinline__ int32_t sample_player(const SArgs& a, const GameInfo& gi, const GameScalars& sc, int p,
                                                 uint64_t d, uint16_t* list, int lane) {
    const uint4* owner = reinterpret_cast<const uint4*>(a.owner + gi.cell_off);
    const uint32_t p4 = 0x01010101u * (uint32_t)p;
    int n = 0;
    for (int c0 = 0; c0 < gi.Npad; c0 += 1024) {  // 32 cells per lane; padding cells have owner -1
        const int c = c0 + 32 * lane;
        const uint4 none = make_uint4(kAll, kAll, kAll, kAll);
        const uint4 Oa = c < gi.Npad ? __ldg(owner + (c >> 4)) : none;
        const uint4 Ob = c + 16 < gi.Npad ? __ldg(owner + (c >> 4) + 1) : none;
        uint32_t mine = equal_bytes16(Oa, p4) | (equal_bytes16(Ob, p4) << 16);
        const int cnt = __popc(mine);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += y;
        }
        uint16_t* at = list + n + (incl - cnt);
        for (; mine; mine &= mine - 1) *at++ = (uint16_t)(c + __ffs(mine) - 1);
        n += __shfl_sync(kAll, incl, 31);
    }
    __syncwarp();
    if (n == 0) return 0;
    const bool moves = ((sc.alive >> p) & 1u) && !sc.finished;
    const float* lg = a.logits + (gi.plane_off + (int64_t)p * gi.Npad) * 9;
    const int16_t* army = a.army + gi.cell_off;
    const uint8_t* terrain = reinterpret_cast<const uint8_t*>(a.terrain + gi.cell_off);
    const int k = (n + 31) >> 5;
    const int i0 = lane * k, i1 = min(n, i0 + k);
    // pass 1: the maximum legal logit; the first two cells stay in registers
    float v0[9], v1[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) v0[q] = v1[q] = kNegInf;
    if (i0 < i1) load_cell(v0, lg, army, terrain, list[i0], moves);
    if (i0 + 1 < i1) load_cell(v1, lg, army, terrain, list[i0 + 1], moves);
    float m = cell_max(v1, cell_max(v0, kLowest));
    for (int i = i0 + 2; i < i1; ++i) {
        float v[9];
        load_cell(v, lg, army, terrain, list[i], moves);
        m = cell_max(v, m);
    }
    m = warp_max_nan(m);
    // pass 2: the lane's weight sum, every exponential once
    uint64_t mine = 0;
    if (m < -kNegInf) {
        mine = k > 1 ? cell_weight2(v0, v1, m) : cell_weight(v0, m);
        for (int i = i0 + 2; i < i1; ++i) {
            float v[9];
            load_cell(v, lg, army, terrain, list[i], moves);
            mine += cell_weight(v, m);
        }
    } else {  // a legal +inf or NaN, outside the documented domain: the maximum over what are numbers, weight_shift's weights
        m = kLowest;
        for (int e = 9 * i0; e < 9 * i1; ++e) m = fmaxf(m, legal_logit(lg, army, terrain, list[e / 9], e % 9, moves));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kAll, m, o));
        for (int e = 9 * i0; e < 9 * i1; ++e) mine += weight_shift(legal_logit(lg, army, terrain, list[e / 9], e % 9, moves), m);
    }
    const uint64_t incl = warp_incl64(mine, lane);
    const uint64_t S = __shfl_sync(kAll, incl, 31);
    const uint64_t r = __umul64hi(d, S);
    const unsigned hit = __ballot_sync(kAll, incl > r);
    if (hit == 0u) return 0;  // S = 0: only when every legal logit is -inf (outside the documented domain)
    const int L = __ffs(hit) - 1;
    uint64_t left = r - __shfl_sync(kAll, incl - mine, L);  // below lane L's sum
    // the entry among lane L's cells: three cells at a time, a lane per entry
    const int q = lane / 9, e = lane - 9 * q, end = min(n, L * k + k);
    for (int j = L * k; j < end; j += 3) {
        const int i = j + q;
        const int c = lane < 27 && i < end ? list[i] : -1;
        const uint32_t w = c >= 0 ? weight_shift(legal_logit(lg, army, terrain, c, e, moves), m) : 0u;
        uint32_t in = w;  // at most 27 * 2^25
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, in, o);
            if (lane >= o) in += y;
        }
        const unsigned b = __ballot_sync(kAll, (uint64_t)in > left);
        if (b) return __shfl_sync(kAll, 9 * c + e, __ffs(b) - 1);
        left -= __shfl_sync(kAll, in, 31);
    }
    return 0;  // not reached: the loop's weights sum to lane L's
}

// ---- the expanded mask --------------------------------------------------------
// One CTA per game: each cell's nine legal bits and owner in one 16-bit word
// of shared memory, then every thread makes 16-byte vectors of the players'
// planes, 512 contiguous bytes per warp.  A vector holds bytes of at most
// three cells; for most (vector, player) pairs none of them is the player's
// and zeros are stored.  HBM-bound by its 9 bytes per player and cell:
// 8,192 mixed games of 20..40 a side 53 us for 295 MB, about 100 us (of 343
// with the sampler) when a warp wrote single bytes to staging rows.
constexpr int kMaskThreads = 128;
// s_cell: legal bits 0..8, owner 12..15 (15: none)
__device__ __forceinline__ void mask_game(const SArgs& a, int gidx, uint16_t* s_cell, int tid) {
    const GameInfo gi = sample_game(a, gidx);
    const GameScalars sc = a.scal[gidx];
    const int Npad = gi.Npad, P = gi.P;
    for (int c = 4 * tid; c < Npad; c += 4 * kMaskThreads) {
        const uint2 av = __ldg(reinterpret_cast<const uint2*>(a.army + gi.cell_off + c));
        const uint32_t ow = __ldg(reinterpret_cast<const uint32_t*>(a.owner + gi.cell_off + c));
        const uint32_t tw = __ldg(reinterpret_cast<const uint32_t*>(a.terrain + gi.cell_off + c));
        uint32_t x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int o = (int)(int8_t)(ow >> (8 * i));
            const int army = (int)(int16_t)((i < 2 ? av.x : av.y) >> (16 * (i & 1)));
            const bool moves = o >= 0 && ((sc.alive >> o) & 1u) && !sc.finished;
            x[i] = legal9(o >= 0, army, (tw >> (8 * i)) & 0xFFu, moves) | ((uint32_t)(o & 15) << 12);
        }
        *reinterpret_cast<uint2*>(s_cell + c) = make_uint2(x[0] | (x[1] << 16), x[2] | (x[3] << 16));
    }
    if (tid < 2) s_cell[Npad + tid] = 0xF000u;  // read past the last cell, never kept
    __syncthreads();
    const int nv = (9 * Npad) >> 4;
    for (int v = tid; v < nv; v += kMaskThreads) {
        const int c = 16 * v / 9, off = 16 * v - 9 * c;  // the vector's first byte is entry `off` of cell c
        const uint32_t e0 = s_cell[c], e1 = s_cell[c + 1], e2 = s_cell[c + 2];
        uint4* out = reinterpret_cast<uint4*>(a.mask9 + gi.plane_off * 9) + v;
        for (int p = 0; p < P; ++p, out += nv) {
            uint32_t bits = ((e0 >> 12) == p ? e0 & 0x1FFu : 0u) | ((e1 >> 12) == p ? (e1 & 0x1FFu) << 9 : 0u) |
                            ((e2 >> 12) == p ? (e2 & 0x1FFu) << 18 : 0u);
            bits >>= off;
            uint4 y = make_uint4(0u, 0u, 0u, 0u);
            if (bits & 0xFFFFu) {
                auto spread = [&](int sh) { return (((bits >> sh) & 15u) * 0x00204081u) & 0x01010101u; };
                y = make_uint4(spread(0), spread(4), spread(8), spread(12));
            }
            __stcs(out, y);
        }
    }
}
__global__ void __launch_bounds__(kMaskThreads) k_mask9(const SArgs a) {
    chain_entry();
    extern __shared__ __align__(16) char smem[];
    mask_game(a, blockIdx.x, reinterpret_cast<uint16_t*>(smem), threadIdx.x);
}

// one warp per (game, player): warp b takes player b mod pmax of game b / pmax
// (those of absent players return at once).  CTAs of two warps: 2v2, 8-player
// and two-player games mix in one launch without holding slots for absent
// players.
constexpr int kSlotWarps = 2;
__device__ __forceinline__ void sample_slot(const SArgs& a, int gidx, int p, char* smem, int wid, int lane) {
    const GameInfo gi = sample_game(a, gidx);
    if (p >= gi.P) return;
    const GameScalars sc = a.scal[gidx];
    uint16_t* list = reinterpret_cast<uint16_t*>(smem + (size_t)wid * list_bytes(a.npad_max));
    const int32_t action = sample_player(a, gi, sc, p, player_draw(a, gi, sc, p), list, lane);
    if (lane == 0) a.actions[gi.player_off + p] = action;
}
__global__ void __launch_bounds__(32 * kSlotWarps, 36 / kSlotWarps) k_sample_slots(const SArgs a, int pmax) {
    chain_entry();
    extern __shared__ __align__(16) char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned item = blockIdx.x * kSlotWarps + wid;
    const int gidx = (int)(item / (unsigned)pmax), p = (int)item - gidx * pmax;
    if (gidx < a.n_games) sample_slot(a, gidx, p, smem, wid, lane);
}
// The same for large batches: `per` consecutive (game, player) items per warp,
// whose draws are hashed side by side, a lane each (a hundred instructions
// for all of them), and whose indexes are divided once.
__global__ void __launch_bounds__(32 * kSlotWarps, 36 / kSlotWarps) k_sample_runs(const SArgs a, int pmax, int per) {
    chain_entry();
    extern __shared__ __align__(16) char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint16_t* list = reinterpret_cast<uint16_t*>(smem + (size_t)wid * list_bytes(a.npad_max));
    const unsigned item = (blockIdx.x * kSlotWarps + wid) * (unsigned)per + lane;
    const int my_g = (int)(item / (unsigned)pmax), my_p = (int)item - my_g * pmax;
    uint64_t my_d = 0;
    if (lane < per && my_g < a.n_games) my_d = player_draw(a, sample_game(a, my_g), a.scal[my_g], my_p);
#pragma unroll 1
    for (int i = 0; i < per; ++i) {
        const int gidx = __shfl_sync(kAll, my_g, i), p = __shfl_sync(kAll, my_p, i);
        const uint64_t d = __shfl_sync(kAll, my_d, i);
        if (gidx >= a.n_games) return;
        const GameInfo gi = sample_game(a, gidx);
        if (p >= gi.P) continue;
        const GameScalars sc = a.scal[gidx];
        const int32_t action = sample_player(a, gi, sc, p, d, list, lane);
        if (lane == 0) a.actions[gi.player_off + p] = action;
        __syncwarp();  // the list is reused
    }
}
// The sampler and the expanded mask in one launch: per game, CTAs of four
// players and one CTA for its mask.  The sampler waits on latency and the
// mask on HBM writes, so they overlap (8,192 mixed games of 20..40 a side:
// one launch after the other 111 us, so 97 us).
__global__ void __launch_bounds__(kMaskThreads, 9) k_sample_mask(const SArgs a, int ctas_per_game) {
    chain_entry();
    extern __shared__ __align__(16) char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int gidx = blockIdx.x / ctas_per_game, part = blockIdx.x - gidx * ctas_per_game;
    if (part + 1 < ctas_per_game)
        sample_slot(a, gidx, part * (kMaskThreads / 32) + wid, smem, wid, lane);
    else
        mask_game(a, gidx, reinterpret_cast<uint16_t*>(smem), threadIdx.x);
}

}  // namespace

int launch_sample(const SArgs& a, int pmax, void* stream) {
    if (a.n_games <= 0) return 0;
    const cudaStream_t st = (cudaStream_t)stream;
    const int mask_smem = 2 * a.npad_max + 16;
    if (!a.logits) return launch_chained(k_mask9, dim3(a.n_games), dim3(kMaskThreads), mask_smem, st, a);
    if (a.mask9) {
        constexpr int per = kMaskThreads / 32;
        const int ctas_per_game = (pmax + per - 1) / per + 1;
        return launch_chained(k_sample_mask, dim3((unsigned)a.n_games * (unsigned)ctas_per_game), dim3(kMaskThreads),
                              std::max(mask_smem, per * list_bytes(a.npad_max)), st, a, ctas_per_game);
    }
    const int64_t items = (int64_t)a.n_games * pmax;
    // runs for batches of one shape (every item is a player) of many waves:
    // 65,536 24x24 1v1 games 141.5 us with one item per warp, 136.6 with two,
    // 134.3 with four; 16,384 games 39.9, 39.0 and 41.7; 4,000 games 11.5 and 11.9
    const int64_t per_sm = items / sm_count();
    const int per = !a.uniform || per_sm < 160 ? 1 : per_sm < 512 ? 2 : 4;
    if (per > 1) {
        const int64_t warps = (items + per - 1) / per;
        return launch_chained(k_sample_runs, dim3((unsigned)((warps + kSlotWarps - 1) / kSlotWarps)),
                              dim3(32 * kSlotWarps), kSlotWarps * list_bytes(a.npad_max), st, a, pmax, per);
    }
    return launch_chained(k_sample_slots, dim3((unsigned)((items + kSlotWarps - 1) / kSlotWarps)), dim3(32 * kSlotWarps),
                          kSlotWarps * list_bytes(a.npad_max), st, a, pmax);
}

}  // namespace gk
