// One game per CTA: the step for batches too small to fill the GPU with a
// warp per game, per frame and multi-frame.
//
// A game-frame is a chain of dependent passes (about 1,900 warp instructions
// on a 24x24 1v1 board with a warp per game), and a small batch leaves most
// issue slots idle while it runs.  Here the passes over the board spread over
// the CTA's threads, and after the cell pass the first warp picks the next
// actions while the others build the fog and write the outputs.  Boards of every size and mode share one launch: each CTA
// carves the launch's largest geometry for its game.
//
// Latency bounds it (per frame of 64 24x24 1v1 games 2.7 us, a warp per game
// 4.0 us): the moves are a serial chain on one lane, and each pass a few
// dependent shared-memory round trips between two barriers.
#include <algorithm>

#include "gk_game.cuh"

namespace gk {

namespace {

// some of the CTA's threads (a multiple of 32, from thread `first` on) as a
// group that meets at named barrier `bar`
struct Team {
    int lane, width, bar;
    __device__ __forceinline__ Team(int first, int threads, int barrier)
        : lane((int)threadIdx.x - first), width(threads), bar(barrier) {}
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(width) : "memory"); }
};

// growth, bitsets, land and army totals, legal moves per chunk of the players
// in `moving`: a chunk of 16 cells per thread, the players in turn; totals add
// up in s.misc (zeroed before) and *sat
__device__ __forceinline__ void team_cells(const Game& g, const Smem& s, bool grow_s, bool grow_p, uint32_t moving,
                                           uint32_t* sat) {
    const int lane = threadIdx.x & 31, nch = g.nch, st2 = 2 * s.stride;
    uint16_t* own16 = reinterpret_cast<uint16_t*>(s.own);
    uint16_t* big16 = reinterpret_cast<uint16_t*>(s.big);
    for (int ch = threadIdx.x; ch - lane < nch; ch += blockDim.x) {  // whole warps
        const bool in = ch < nch;
        const int c0 = ch << 4;
        uint4 O = make_uint4(kFull, kFull, kFull, kFull), T = make_uint4(0u, 0u, 0u, 0u);
        uint32_t aw[8] = {}, big = 0;
        if (in) {
            uint32_t over = 0;
            grown_armies(s, c0, grow_s, grow_p, aw, over);
            if (over) atomicAdd(sat, over);
            big = big_bits(aw);
            big16[ch] = (uint16_t)big;
            O = *reinterpret_cast<const uint4*>(s.owner + c0);
            T = *reinterpret_cast<const uint4*>(s.terrain + c0);
            if ((nch & 1) && ch == nch - 1) big16[nch] = 0;
        }
        const uint32_t ow[4] = {O.x, O.y, O.z, O.w};
        // passable neighbours: a nibble per cell, two words side by side
        const uint32_t d0 = ((T.x >> 2) & 0x0F0F0F0Fu) | ((T.y << 2) & 0xF0F0F0F0u);
        const uint32_t d1 = ((T.z >> 2) & 0x0F0F0F0Fu) | ((T.w << 2) & 0xF0F0F0F0u);
        for (int p = 0; p < g.P; ++p) {
            const uint32_t p4 = 0x01010101u * (uint32_t)p;
            uint32_t arm = 0, z[4];  // z: 0x80 where the owner (-1 .. 7) is p
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                z[k] = ~(((ow[k] ^ p4) & 0x0F0F0F0Fu) + 0x7F7F7F7Fu) & 0x80808080u;
                arm = __dp2a_hi(aw[2 * k + 1], z[k], __dp2a_lo(aw[2 * k], z[k], arm));
            }
            const uint32_t own = (collect_lo(z[0], z[1]) >> 7) | (collect_lo(z[2], z[3]) << 1);
            if (in) {
                own16[p * st2 + ch] = (uint16_t)own;
                const uint32_t mv = (moving >> p) & 1u ? own & big : 0u;
                const uint32_t l0 = (spread4(mv & 15u) * 0x0Fu) | (spread4((mv >> 4) & 15u) * 0xF0u);
                const uint32_t l1 = (spread4((mv >> 8) & 15u) * 0x0Fu) | (spread4((mv >> 12) & 15u) * 0xF0u);
                s.cnt[p * nch + ch] = (uint8_t)(__popc(d0 & l0) + __popc(d1 & l1));
                if ((nch & 1) && ch == nch - 1) own16[p * st2 + nch] = 0;
            }
            arm = __reduce_add_sync(kFull, arm >> 7);
            const uint32_t land = __reduce_add_sync(kFull, (uint32_t)__popc(own));
            if (lane == 0 && land) {
                atomicAdd(s.misc + 8 + p, (int)land);
                atomicAdd(s.misc + 16 + p, (int)arm);
            }
        }
    }
}

}  // namespace

template <bool SPAWN>
__global__ void __launch_bounds__(256, 4) k_team(const KArgs a) {
    chain_entry();
    extern __shared__ __align__(16) char smem_raw[];
    __shared__ uint32_t s_ctl[4];    // after the moves: alive, eliminated, invalid, saturated
    __shared__ uint32_t s_draws[32];  // the policy's
    const int gidx = a.list ? a.list[blockIdx.x] : (int)blockIdx.x;
    if (gidx < 0 || gidx >= a.n_games) return;
    const int tid = threadIdx.x, lane = tid & 31, nthreads = blockDim.x;
    const bool first = tid < 32;  // the warp that moves and draws
    const Team all(0, nthreads, 0), rest(32, nthreads - 32, 1);
    const Grp<32> warp(lane);
    const Game g = game_of(a, gidx);
    const Smem s = carve(smem_raw, a);
    const uint64_t gid = game_id_of(a, gidx);

    board_issue(a, g, s, all);
    zero_guards(g, s, all);
    const uint4 s0 = *reinterpret_cast<const uint4*>(a.scal + gidx);
    const uint4 s1 = *(reinterpret_cast<const uint4*>(a.scal + gidx) + 1);
    int32_t my_act = first && lane < g.P ? a.actions[g.player_off + lane] : 0;
    board_wait(all);
    uint32_t turn = s0.x, frame = s0.y, epoch = s0.z, alive = s0.w;
    uint32_t finished = s1.x, invalid = s1.y, saturated = s1.z;
    const uint32_t err = s1.w, all_alive = (1u << g.P) - 1u;
    bool wrote_state = false;

    for (int f = 0; f < a.frames; ++f) {
        float my_reward = 0.0f;  // lane p's, in every warp
        uint32_t done = 0, eliminated = 0;
        const bool stepping = !finished;
        // while the first warp moves, the second zeroes the totals and hashes
        // the draws of the next actions
        if (first) {
            if (stepping) {
                if (a.action_log && lane < g.P) a.action_log[(int64_t)f * a.slot_stride + g.player_off + lane] = my_act;
                uint32_t inv = 0, sat = 0;
                play_moves(g, s, warp, turn, my_act, alive, eliminated, inv, sat);
                if (lane == 0) {
                    s_ctl[0] = alive;
                    s_ctl[1] = eliminated;
                    s_ctl[2] = inv;
                    s_ctl[3] = sat;
                }
            }
        } else if (tid < 64) {
            if (lane < 16) s.misc[8 + lane] = 0;
            if (a.next_actions) s_draws[lane] = policy_draws(a, g, frame + 1, gid, lane);
        }
        all.sync();
        frame += 1;
        if (stepping) {
            alive = s_ctl[0];
            eliminated = s_ctl[1];
            invalid += s_ctl[2];
            turn += 1;
            done = outcome(a, g, lane, turn, alive, eliminated, my_reward);
            if (done && !a.auto_reset) finished = 1;
            wrote_state = true;
        }
        const bool new_map = done && a.auto_reset;
        team_cells(g, s, stepping && (turn % 2u) == 0u, stepping && (turn % 50u) == 0u, finished ? 0u : alive, s_ctl + 3);
        all.sync();
        if (stepping) saturated += s_ctl[3];
        if (new_map) {
            epoch += 1;
            turn = 0;
            alive = all_alive;
            if (first)
                generate<32, false, SPAWN>(a, gidx, smem_raw, geom_of(a), gid, epoch, lane);
            else if (tid < 48)
                s.misc[tid - 24] = 0;
            all.sync();
            team_cells(g, s, false, false, alive, s_ctl + 3);
            all.sync();
        }
        if (first) {
            const int64_t slot = (int64_t)f * a.slot_stride + g.player_off + lane;
            if (lane < g.P) {
                a.reward[slot] = my_reward;
                a.scoreboard[2 * slot + 0] = s.misc[8 + lane];
                a.scoreboard[2 * slot + 1] = s.misc[16 + lane];
            }
            if (lane == 0) a.done[(int64_t)f * a.game_stride + gidx] = (uint8_t)done;
            if (a.next_actions)
                my_act = policy_pass<false, 32>(a, g, s, alive, finished != 0, s_draws[lane], warp);
        } else {
            fog_pass(g, s, alive, rest);
            output_pass<true, false>(a, g, s, alive, finished != 0, rest, (int64_t)f * a.plane_stride);
        }
        all.sync();  // the next frame's moves change the board
    }
    if (first && a.next_actions && lane < g.P) a.next_actions[g.player_off + lane] = my_act;
    if (wrote_state) store_board(a, g, s, all);
    if (tid == 0) store_scalars(a, gidx, turn, frame, epoch, alive, finished, invalid, saturated, err);
}

// Warps per game: the first and enough others to write the outputs (16-cell
// chunks of every player) in about two rounds, one more while that asks for
// at most 20 warps per SM (32 frames of 1v1 games with one more and without:
// 700 of 24x24 107 and 109 us, 1,000 of 15x15 100 and 106; 64 frames of 1,024
// 24x24 games 245 and 239 us); fewer, down to two, when the
// games would not all run at once (64 registers: 32 warps per SM; 16 frames of
// 1,024 mixed games: 157 us, with up to 48 warps per SM asked for 214 us).
int launch_team(const KArgs& a, int sms, void* stream) {
    const bool spawn = a.spawn_dmax > 0 || a.spawn_bfs || a.castle_radius > 0;
    void (*const f)(KArgs) = spawn ? k_team<true> : k_team<false>;
    static SmemLimit limits[2];
    const void* fn = (const void*)f;
    const int e = limits[spawn].raise(&fn, 1, a.warp_smem);
    if (e != 0) return e;
    const int chunks = a.pmax * (a.npad_max >> 4);
    int warps = 1 + std::min(7, (chunks + 63) / 64);
    if (warps < 8 && (int64_t)a.n_items * (warps + 1) <= (int64_t)20 * sms) ++warps;
    while (warps > 2 && (int64_t)a.n_items * warps > (int64_t)28 * sms) --warps;
    const int threads = 32 * warps;
    return launch_chained(f, dim3(a.n_items), dim3(threads), a.warp_smem, (cudaStream_t)stream, a);
}

int fill_team_columns() { return fill_columns(); }

}  // namespace gk
