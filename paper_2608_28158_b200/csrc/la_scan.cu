// State scan of the chunk-parallel path (bf16, d_k = d_v = 128, chunk 64): the recurrence over chunk boundaries alone.
//
// Forward:  S_{c+1} = e^{b_n} S_c + sum_j k_j^T (w_j v_j)          w_j = e^{b_n - b_j}; S_c of every chunk -> workspace tile
// Backward: dS_{c-1} = e^{b_n} dS_c + sum_t q_t^T (e^{b_t} dO_t)   dS_c (gradient at the END of chunk c) -> workspace tile
// With the tiles in memory every chunk is independent of every other (la_chunk_fwd.cu, la_chunk_bwd.cu), so a problem
// whose (sequence, head) chains are fewer than the SMs still fills the GPU.
// The backward also leaves <S_c[i,:], dS_c[i,:]> of every chunk, row and 32 columns, which dg needs: the gradient is fp32 only
// here.  S_c arrives in the buffer that the gradient's tile leaves from, one to two tiles ahead, so it takes no room.
//
// What bounds it: the chain of chunks of one sequence while there are few of them, then 64 KB of traffic per (chunk, head).
// So the products, which do not depend on the chain, are taken out of it: the sum of a chunk is a tcgen05 product of its
// own (accumulators double-buffered in tensor memory), the state stays in the registers of the state warps (lane = state
// row), and a step of the chain is one multiply-add per element with the sum read from tensor memory, plus its bf16 tile.
// Roles, all coupled by mbarriers (no CTA-wide barrier inside the walk): a warp that draws the items and requests their
// rows (TMA, three to five chunks ahead), a gate warp (running sums -> weights), warps that weight the v rows in place, an
// MMA warp, the state warps, and a store warp (TMA).  A (sequence, head) is one item of NV = 128 state columns, or 2 of 64,
// or 4 of 32 (launch_sliced): the columns do not interact, so the split does not change any result.  All rounds run in one
// launch (scan_fwd below).
// Measured, cold inputs: 0.8 us per step of the longest path while the chains leave SMs idle, 0.85 backward, and 1.5 us from a sequence to the
// one that starts from it (17,695 tokens x 4 heads, 68 steps and three such: 65 us each way; 72 and 71 with table entries loaded when
// they were needed, slots written 16 bytes at a time and a step's waits one after the other); with 96 chains of 100,003 tokens x 16 heads 4.9 TB/s
// forward (345 us), 6.1 backward (470 us).
// Log-decays per channel: 1.3 us a step forward, 1.4 backward (1,047 agentic chunks x 16 heads 367 and 413 us), the weighting warps' chain.
// 454 and 539 us with a's values read one by one between the stores, which a load may not pass, with a warp that copied the rows of a first
// chunk by half its lanes and the gates 16 bytes at a time (12 us an item), and with two stages of rows where three fit (406 and 471).
#include <type_traits>

#include "kernels.h"
#include "tc_common.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int32_t make_state_map(CUtensorMap* map, const void* base, int64_t n);
int32_t make_state_slice_map(CUtensorMap* map, const void* base, int64_t n);
int32_t make_gate_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int sm_count();

namespace {

using namespace tc;

constexpr int BT = 64, D = 128;
constexpr int GATES = 4, RAW = 8, ITEMS = 4, EXPORTS = 4;      // rings: weights, raw log-decays, items, slots written (the state
                                                               // is at most OUTS = 3 tiles ahead of their stores)
constexpr int PANEL = BT * 128, S_PANEL = D * 128;
constexpr float LOG2E = 1.4426950408889634f;

template <int NV, bool GK>
struct Shape {
    static constexpr int NS = NV == 32 ? 128 : 256, NWT = NS, NT = NS + NWT + 128;   // state threads, weighting threads, four warps
    static constexpr int CW = NV * 128 / NS;               // state columns per state thread
    static constexpr int STAGES = GK ? NV == 64 ? 3 : 2 : NV == 64 ? 5 : 3;        // chunks of rows in shared memory
    static constexpr int OUTS = GK ? 2 : 3;                // state tiles on their way out
    // a 32-column slice loads the 64-column panel it lies in
    static constexpr int A = 2 * PANEL, B = (NV + 63) / 64 * PANEL, G = GK ? BT * D * 4 : 0,
                         O = D * NV * 2;
    static constexpr int a = 0, b = STAGES * A, g = b + STAGES * B, out = g + STAGES * G, misc = out + OUTS * O,
                         bytes = misc + 12288 + 1024;      // 1024: alignment of the dynamic area
};
struct Item {                // one (sequence, head, slice); seq < 0: no more
    int seq, h, slice, own_begin, n_replay, n_virtual, n_chunks, chunk_base, replay_base, init_slot, req_lo, req_hi;
    int n_steps;             // chunks whose sum enters the walk
};
struct Misc {
    float w[GATES][BT];
    float gamma[GATES];
    float raw[RAW][BT];
    float gammas[GATES][D];      // per-channel decay: e^{b_n} of every state row
    float part[2][4][D];         // and the sums of four groups of 16 rows, of every second step
    uint64_t full[5], weighted[5], stage_empty[5], u_full[2], u_empty[2], gates_full[GATES], gates_empty[GATES], out_full[3],
        out_empty[3], item_full[ITEMS], item_empty[ITEMS], part_full[2], exported[EXPORTS];
    Item items[ITEMS];
    int2 tile[3];            // backward: the tile (index, slice) a buffer is for
    uint32_t tmem;
    int dead;
};
static_assert(sizeof(Misc) <= 12288, "misc area");

// a: the operand that spans the state's rows (k forward, q backward), b: the one that spans its columns (v / dO).
// GK: a log-decay per row and state row (g [rows, H, 128]): its tile travels with the rows, and the weights go onto a.
template <bool BWD, int NV, bool GK>
__global__ void __launch_bounds__(Shape<NV, GK>::NT, NV == 32 ? 2 : 1)
scan_kernel(const harts_la_tables_t tb, int seq_lo, int n_items, int H, const __grid_constant__ CUtensorMap map_a,
            const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_g,
            const __grid_constant__ CUtensorMap map_tiles, const __grid_constant__ CUtensorMap map_s,
            const __nv_bfloat16* __restrict__ a, const __nv_bfloat16* __restrict__ b, const float* __restrict__ g,
            float* slots, float* ds0, float* __restrict__ dots, int* status, const int32_t* gate, int* flags, int* ticket, const RoundOrder order) {
    if (gate_closed(gate)) return;
    using S = Shape<NV, GK>;
    constexpr int SLICES = D / NV, NS = S::NS, NWT = S::NWT, CW = S::CW, STAGES = S::STAGES, OUTS = S::OUTS;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    Misc& m = *reinterpret_cast<Misc*>(smem + S::misc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < STAGES; i++) {
            mbar_init(&m.full[i], 1);
            mbar_init(&m.weighted[i], NWT / 32);
            mbar_init(&m.stage_empty[i], 1);
        }
        for (int i = 0; i < GATES; i++) {
            mbar_init(&m.gates_full[i], GK ? NWT / 32 : 1);
            mbar_init(&m.gates_empty[i], GK ? NS / 32 : (NS + NWT) / 32);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&m.u_full[i], 1);
            mbar_init(&m.part_full[i], NWT / 32);
            mbar_init(&m.u_empty[i], NS / 32);
        }
        for (int i = 0; i < OUTS; i++) {
            mbar_init(&m.out_full[i], NS / 32);
            mbar_init(&m.out_empty[i], 1);
        }
        for (int i = 0; i < ITEMS; i++) {
            mbar_init(&m.item_full[i], 1);
            mbar_init(&m.item_empty[i], (NS + NWT) / 32 + (GK ? 2 : 3));
        }
        for (int i = 0; i < EXPORTS; i++) mbar_init(&m.exported[i], NS / 32);
        m.dead = 0;
        fence_barrier_init();
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc<2 * NV>(&m.tmem);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = m.tmem;
    auto wait = [&](uint64_t* bar, int use) { return mbar_wait(bar, use & 1, status, &m.dead); };               // one thread
    auto wait_warp = [&](uint64_t* bar, int use) { return mbar_wait_warp(bar, use & 1, status, &m.dead); };     // a whole warp
    // the walk over an item's chunks: forward 0..n-1, the last one's sum is not needed (its end state is never exported);
    // backward n-1..0, chunk 0's sum only where somebody waits for the gradient of the initial state
    auto chunk_of = [](const Item& it, int i) { return BWD ? it.n_chunks - 1 - i : i; };

    if (warp < NS / 32) {
        // ---- state: row L, columns col0 .. col0 + CW - 1 of the slice ------------------------------------------------------
        const int L = (warp & 3) * 32 + lane, col0 = (warp >> 2) * CW;
        const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16) + col0;
        int gs = 0, gt = 0, n_exported = 0;   // steps, tiles and exports since the kernel began
        bool alive = true;
        for (int k = 0; alive && wait_warp(&m.item_full[k % ITEMS], k / ITEMS); k++) {
            const Item it = m.items[k % ITEMS];
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[k % ITEMS]);
            if (it.seq < 0) break;
            const size_t in_state = (size_t)L * D + it.slice * NV + col0;
            // gradients of initial states, which only these threads write and read: [32 columns][32 rows][four of the columns][row],
            // whatever the slices' width, so that a warp's access is 512 bytes in a row
            auto ds0_of = [&](size_t seq_head) {
                return reinterpret_cast<float4*>(ds0 + seq_head * (D * D)) + ((it.slice * NV + col0) / 32 * 4 + (warp & 3)) * 256 + lane;
            };
            auto ds0_step = [](int e) { return (e >> 3) * 1024 + (e & 7) * 32; };
            float x[CW];
#pragma unroll
            for (int e = 0; e < CW; e++) x[e] = 0.f;
            if (!BWD && it.init_slot >= 0) {
                const size_t from = (size_t)it.init_slot * H + it.h;
                const float4* src = reinterpret_cast<const float4*>(slots + from * (D * D) + in_state);
                if (order.n) alive = flag_wait_warp(flags + from * SLICES + it.slice, 1, status, &m.dead);
#pragma unroll
                for (int e = 0; e < CW / 4; e++) *reinterpret_cast<float4*>(x + 4 * e) = __ldcg(src + e);
            }
            // what the next export (backward: the next boundary with gradients) needs is asked for at the one before it: a table entry
            // that is used as soon as it is loaded holds the chain up by 0.35 us
            const int req_end = BWD ? it.req_lo - 1 : it.req_hi, way = BWD ? -1 : 1;
            int req = BWD ? it.req_hi - 1 : it.req_lo;
            int boundary = req != req_end ? tb.slot_chunk[req] : -1, boundary2 = req != req_end && req + way != req_end ? tb.slot_chunk[req + way] : -1;
            int cons_lo = 0, cons_hi = 0, who = 0;      // backward: the sequences that started from it; a lane's one of 32
            auto consumers = [&] {
                if (BWD && req != req_end) {
                    cons_lo = tb.slot_cons_ptr[req];
                    cons_hi = tb.slot_cons_ptr[req + 1];
                }
            };
            auto advance = [&] {
                req += way;
                boundary = boundary2;
                boundary2 = req != req_end && req + way != req_end ? tb.slot_chunk[req + way] : -1;
                consumers();
            };
            consumers();
            for (int i = 0; i < it.n_chunks && alive; i++) {
                const int c = chunk_of(it, i);
                if (BWD && boundary == c + 1) {   // gradients of every sequence that started from this boundary, in table order
                    unsigned there = 0;       // whose flag is up already: a lane each looks, 32 at a time
                    for (int u = cons_lo, k = 0; u < cons_hi; u++, k++) {
                        if ((k & 31) == 0) {
                            if ((k > 0 || i == 0) && u + lane < cons_hi) who = tb.slot_cons_seq[u + lane];
                            if (order.n) {
                                const bool mine = u + lane < cons_hi && ld_acquire(flags + ((size_t)who * H + it.h) * SLICES + it.slice) >= NS / 32;
                                there = __ballot_sync(0xffffffffu, mine);
                                __syncwarp();     // hands on what the lanes acquired
                            }
                        }
                        const size_t from = (size_t)__shfl_sync(0xffffffffu, who, k & 31) * H + it.h;
                        if (order.n && !(there >> (k & 31) & 1)) alive = flag_wait_warp(flags + from * SLICES + it.slice, NS / 32, status, &m.dead) && alive;
                        const float4* src = ds0_of(from);
#pragma unroll
                        for (int e = 0; e < CW / 4; e++) {
                            const float4 y = __ldcg(src + ds0_step(e));
                            x[4 * e] += y.x, x[4 * e + 1] += y.y, x[4 * e + 2] += y.z, x[4 * e + 3] += y.w;
                        }
                    }
                    advance();
                }
                if (BWD && boundary == c && cons_lo + lane < cons_hi) who = tb.slot_cons_seq[cons_lo + lane];      // of the next step
                if (!BWD || i > 0) {              // the state before this step as a bf16 tile (backward: zero after the last chunk)
                    // backward: the buffer holds S_c, which is multiplied with the gradient before that is rounded over it
                    if ((BWD || gt >= OUTS) && !wait_warp(&m.out_empty[gt % OUTS], BWD ? gt / OUTS : gt / OUTS - 1)) alive = false;
                    unsigned char* dst = smem + S::out + (gt % OUTS) * S::O + (col0 >> 6) * S_PANEL;
                    float* dot = BWD ? dots + ((size_t)(it.chunk_base + c) * H + it.h) * (4 * D) + (it.slice * NV + col0) / 32 * D + L : nullptr;
                    float d0 = 0.f, d1 = 0.f;
#pragma unroll
                    for (int v = 0; v < CW / 8; v++) {
                        uint4* at = reinterpret_cast<uint4*>(dst + (NV == 32 ? L * 64 + ((v ^ ((L >> 1) & 3)) << 4) : sw128_chunk(L, (col0 & 63) / 8 + v)));
                        if constexpr (BWD) {
                            const uint4 y = *at;
                            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&y);
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const float2 f = __bfloat1622float2(h2[e]);
                                d0 += f.x * x[8 * v + 2 * e];
                                d1 += f.y * x[8 * v + 2 * e + 1];
                            }
                            if ((v & 3) == 3) {   // 32 columns: the same sums whatever the width of the slices
                                dot[v / 4 * D] = d0 + d1;
                                d0 = d1 = 0.f;
                            }
                        }
                        *at = make_uint4(pack_bf16(x[8 * v], x[8 * v + 1]), pack_bf16(x[8 * v + 2], x[8 * v + 3]),
                                         pack_bf16(x[8 * v + 4], x[8 * v + 5]), pack_bf16(x[8 * v + 6], x[8 * v + 7]));
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.out_full[gt % OUTS]);
                    gt++;
                }
                if (!BWD && boundary == c) {
                    const size_t to = (size_t)req * H + it.h;
                    float* dst = slots + to * (D * D) + in_state;
                    // a thread's row is 512 bytes from the next one's: whole sectors at a time, where the array allows it
                    if ((reinterpret_cast<uintptr_t>(slots) & 31) == 0) {
#pragma unroll
                        for (int e = 0; e < CW; e += 8)
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + e), "f"(x[e]), "f"(x[e + 1]), "f"(x[e + 2]),
                                         "f"(x[e + 3]), "f"(x[e + 4]), "f"(x[e + 5]), "f"(x[e + 6]), "f"(x[e + 7]) : "memory");
                    } else {
#pragma unroll
                        for (int e = 0; e < CW; e += 4) *reinterpret_cast<float4*>(dst + e) = *reinterpret_cast<const float4*>(x + e);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.exported[n_exported % EXPORTS]);      // the store warp publishes it: no fence in the chain
                    n_exported++;
                    advance();
                }
                if (i >= it.n_steps) break;
                // both tries in flight together (per channel, where the weights are late, the second one is better made after the first)
                const bool gates = !GK && mbar_try(&m.gates_full[gs % GATES], gs / GATES & 1), sum = !GK && mbar_try(&m.u_full[gs & 1], gs >> 1 & 1);
                if ((GK || !__all_sync(~0u, gates && sum)) && (!wait_warp(&m.gates_full[gs % GATES], gs / GATES) || !wait_warp(&m.u_full[gs & 1], gs >> 1)))
                    alive = false;
                const float gamma = GK ? m.gammas[gs % GATES][L] : m.gamma[gs % GATES];
                tc_fence_after();
#pragma unroll
                for (int blk = 0; blk < CW / 16; blk++) {
                    uint32_t u[16];
                    tmem_ld16(tm + (gs & 1) * NV + blk * 16, u);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; e++) x[blk * 16 + e] = __fmaf_rn(gamma, x[blk * 16 + e], __uint_as_float(u[e]));
                }
                tc_fence_before();
                __syncwarp();
                if (lane < 2) mbar_arrive(lane ? &m.gates_empty[gs % GATES] : &m.u_empty[gs & 1]);
                gs++;
            }
            if (BWD && it.init_slot >= 0 && alive) {     // the hand-off into the sequence that exported this state
                const size_t to = (size_t)it.seq * H + it.h;
                float4* dst = ds0_of(to);
#pragma unroll
                for (int e = 0; e < CW / 4; e++) dst[ds0_step(e)] = *reinterpret_cast<const float4*>(x + 4 * e);
                if (order.n) flag_add_warp(flags + to * SLICES + it.slice);
            }
        }
    } else if (warp < (NS + NWT) / 32) {
        // ---- weights onto the b rows, in place -----------------------------------------------------------------------------------
        const int wt = tid - NS;
        int gs = 0;
        bool alive = true;
        for (int k = 0; alive && wait_warp(&m.item_full[k % ITEMS], k / ITEMS); k++) {
            const Item it = m.items[k % ITEMS];
            const int slice = it.slice;
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[k % ITEMS]);
            if (it.seq < 0) break;
            for (int i = 0; i < it.n_steps; i++, gs++) {
                const int st = gs % STAGES;
                if constexpr (GK) {
                    // thread = two channels x 16 rows: running sums of its rows, joined over the four row groups
                    const int i0 = 2 * (wt & 63), grp = wt >> 6, n_rows = min(BT, it.n_virtual - chunk_of(it, i) * BT);
                    const int first = BWD && chunk_of(it, i) == 0 ? it.n_replay : 0;      // rows before it carry no weight
                    alive = (gs < GATES || wait_warp(&m.gates_empty[gs % GATES], gs / GATES - 1)) && wait_warp(&m.full[st], gs / STAGES);
                    if (!alive) break;
                    const float* sg = reinterpret_cast<const float*>(smem + S::g + st * S::G) + i0;
                    float2 run[16];
                    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
                    for (int u = 0; u < 16; u++) {
                        const int t = 16 * grp + u;
                        const float2 x = *reinterpret_cast<const float2*>(sg + t * D);
                        sum.x += t < n_rows ? x.x * LOG2E : 0.f;
                        sum.y += t < n_rows ? x.y * LOG2E : 0.f;
                        run[u] = sum;
                    }
                    *reinterpret_cast<float2*>(&m.part[gs & 1][grp][i0]) = sum;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.part_full[gs & 1]);
                    if (!(alive = wait_warp(&m.part_full[gs & 1], gs >> 1))) break;
                    float2 before = make_float2(0.f, 0.f), bn = before;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const float2 x = *reinterpret_cast<const float2*>(&m.part[gs & 1][q][i0]);
                        if (q < grp) before.x += x.x, before.y += x.y;
                        bn.x += x.x, bn.y += x.y;
                    }
                    if (grp == 0) *reinterpret_cast<float2*>(&m.gammas[gs % GATES][i0]) = make_float2(ex2(bn.x), ex2(bn.y));
                    unsigned char* sa = smem + S::a + st * S::A + (i0 >> 6) * PANEL + (i0 & 7) * 2;
                    __nv_bfloat162 x[16];         // all of them first: a load does not pass a store whose address may be the same
#pragma unroll
                    for (int u = 0; u < 16; u++) x[u] = *reinterpret_cast<const __nv_bfloat162*>(sa + sw128_chunk(16 * grp + u, (i0 & 63) >> 3));
#pragma unroll
                    for (int u = 0; u < 16; u++) {
                        const int t = 16 * grp + u;
                        uint32_t* at = reinterpret_cast<uint32_t*>(sa + sw128_chunk(t, (i0 & 63) >> 3));
                        const float2 f = __bfloat1622float2(x[u]);
                        const float b0 = before.x + run[u].x, b1 = before.y + run[u].y;
                        const uint32_t y = pack_bf16(f.x * ex2(BWD ? b0 : bn.x - b0), f.y * ex2(BWD ? b1 : bn.y - b1));
                        *at = BWD && (t < first || t >= n_rows) ? 0u : y;
                    }
                } else {
                alive = wait_warp(&m.gates_full[gs % GATES], gs / GATES) && wait_warp(&m.full[st], gs / STAGES);
                if (!alive) break;
                unsigned char* sb = smem + S::b + st * S::B;
                const float* w = m.w[gs % GATES];
#pragma unroll
                for (int u = 0; u < BT * NV / 8 / NWT; u++) {
                    const int e = wt + u * NWT, t = NV == 32 ? (e >> 5) * 8 + (e >> 2 & 1) * 4 + (e >> 3 & 3) : (e >> 3) & 63, p = NV == 32 ? 0 : e >> 9;
                    const int ch = NV == 32 ? (slice & 1) * 4 + (e & 3) : e & 7;
                    uint4* at = reinterpret_cast<uint4*>(sb + p * PANEL + sw128_chunk(t, ch));
                    uint4 y = *at;
                    const float wv = w[t];
                    __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&y);
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const float2 f = __bfloat1622float2(h2[q]);
                        h2[q] = __floats2bfloat162_rn(f.x * wv, f.y * wv);
                    }
                    *at = BWD && wv == 0.f ? make_uint4(0, 0, 0, 0) : y;
                }
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&m.weighted[st]);
                    mbar_arrive(GK ? &m.gates_full[gs % GATES] : &m.gates_empty[gs % GATES]);
                }
            }
        }
    } else if (warp == (NS + NWT) / 32) {
        // ---- items and loads: the next item is drawn when the loads of the one before are on their way, not earlier (a CTA that
        // walks a long sequence must not sit on the items behind it) ---------------------------------------------------------------
        int gs = 0;
        bool alive = true;
        for (int k = 0; alive; k++) {
            if (k >= ITEMS && !(alive = wait_warp(&m.item_empty[k % ITEMS], k / ITEMS - 1))) break;
            int n = (int)blockIdx.x + k * (int)gridDim.x;
            if (order.n) {
                if (lane == 0) n = atomicAdd(ticket, 1);
                n = __shfl_sync(~0u, n, 0);
            }
            Item it;
            it.seq = -1;
            if (n < n_items) {
                it.slice = n % SLICES;
                it.h = n / SLICES % H;
                int j = n / SLICES / H, pos = seq_lo + j;
                if (BWD && order.n)               // last round first
                    for (int r = order.n - 1; r >= 0; r--) {
                        const int cnt = order.ptr[r + 1] - order.ptr[r];
                        pos = order.ptr[r] + j;
                        if (j < cnt) break;
                        j -= cnt;
                    }
                it.seq = tb.seq_order ? tb.seq_order[pos] : pos;
                // one table entry per lane
                const int32_t* from = lane < 2 ? tb.seq_own_begin + lane : lane < 4 ? tb.seq_replay_ptr + (lane - 2)
                                    : lane < 6 ? tb.seq_req_ptr + (lane - 4) : lane == 6 ? tb.seq_chunk_ptr : tb.seq_init_slot;
                const int v = from[it.seq];
                auto entry = [&](int l) { return __shfl_sync(~0u, v, l); };
                it.own_begin = entry(0);
                it.replay_base = entry(2);
                it.n_replay = entry(3) - it.replay_base;
                it.n_virtual = it.n_replay + entry(1) - it.own_begin;
                it.n_chunks = (it.n_virtual + BT - 1) / BT;
                it.req_lo = entry(4);
                it.req_hi = entry(5);
                it.chunk_base = entry(6);
                it.init_slot = entry(7);
                it.n_steps = BWD && it.init_slot >= 0 ? it.n_chunks : it.n_chunks - 1;
            }
            if (lane == 0) {
                m.items[k % ITEMS] = it;
                mbar_arrive(&m.item_full[k % ITEMS]);
            }
            if (it.seq < 0) break;
            for (int i = 0; i < it.n_steps; i++, gs++) {
                const int st = gs % STAGES, row0 = it.own_begin - it.n_replay + chunk_of(it, i) * BT;
                unsigned char *sa = smem + S::a + st * S::A, *sb = smem + S::b + st * S::B;
                const int b0 = it.slice * NV / 64 * 64;
                if (gs >= STAGES && !(alive = wait_warp(&m.stage_empty[st], gs / STAGES - 1))) break;
                // chunk 0 begins with rows from anywhere: row by row (backward: only the gates of replayed rows count)
                if ((GK || !BWD) && chunk_of(it, i) == 0 && it.n_replay > 0) {
                    int row[2];
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const int t = lane + 32 * u;
                        row[u] = t < it.n_replay ? tb.replay_row[it.replay_base + t] : min(it.own_begin + t - it.n_replay, tb.n_rows - 1);
                    }
                    if (GK) {                     // a row's 128 log-decays are one piece
                        if (lane == 0) mbar_expect_tx_only(&m.full[st], S::G);
                        __syncwarp();
#pragma unroll
                        for (int u = 0; u < 2; u++)
                            bulk_load(smem + S::g + st * S::G + (lane + 32 * u) * (D * 4), g + ((size_t)row[u] * H + it.h) * D, D * 4, &m.full[st]);
                    }
                    // every lane carries 16 bytes of every instruction: CH pieces a row, 32 / CH rows at once
                    auto gather = [&](auto ch_count, const __nv_bfloat16* from, unsigned char* to, int col) {
                        constexpr int CH = decltype(ch_count)::value, ROWS = 32 / CH;
                        const int ch = lane % CH;
#pragma unroll 8
                        for (int t0 = 0; t0 < BT; t0 += ROWS) {
                            const int t = t0 + lane / CH, r0 = __shfl_sync(~0u, row[0], t & 31), r1 = __shfl_sync(~0u, row[1], t & 31);
                            unsigned char* dst = to + (ch >> 3) * PANEL + sw128_chunk(t, ch & 7);
                            if (!BWD || t >= it.n_replay)
                                cp_async16(dst, from + ((size_t)(t0 < 32 ? r0 : r1) * H + it.h) * D + col + ch * 8, true);
                            else
                                *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
                        }
                    };
                    gather(std::integral_constant<int, 16>(), a, sa, 0);
                    gather(std::integral_constant<int, S::B / PANEL * 8>(), b, sb, b0);
                    cp_async_wait_all();
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.full[st]);
                } else if (lane == 0) {
                    mbar_expect_tx(&m.full[st], S::A + S::B + S::G);
                    if (GK) tma_load_3d(smem + S::g + st * S::G, &map_g, 0, it.h, row0, &m.full[st]);
                    for (int p = 0; p < 2; p++) tma_load_3d(sa + p * PANEL, &map_a, p * 64, it.h, row0, &m.full[st]);
                    for (int p = 0; p < S::B / PANEL; p++) tma_load_3d(sb + p * PANEL, &map_b, b0 + p * 64, it.h, row0, &m.full[st]);
                }
            }
        }
    } else if (warp == (NS + NWT) / 32 + 1) {
        // ---- products ----------------------------------------------------------------------------------------------------------
        constexpr uint32_t IDESC = instr_desc(128, NV, 1, 1);
        int gs = 0;
        bool alive = true;
        if (lane == 0)
            for (int k = 0; alive && wait(&m.item_full[k % ITEMS], k / ITEMS); k++) {
                const int seq = m.items[k % ITEMS].seq, n_steps = m.items[k % ITEMS].n_steps, slice = m.items[k % ITEMS].slice;
                mbar_arrive(&m.item_empty[k % ITEMS]);
                if (seq < 0) break;
                for (int i = 0; i < n_steps; i++, gs++) {
                    const int st = gs % STAGES;
                    alive = (gs < 2 || wait(&m.u_empty[gs & 1], (gs >> 1) - 1)) && wait(&m.weighted[st], gs / STAGES);
                    if (!alive) break;
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + S::a + st * S::A);
                    const uint32_t sb = smem_u32(smem + S::b + st * S::B) + (NV == 32 ? (slice & 1) * 64 : 0);
#pragma unroll
                    for (int ks = 0; ks < 4; ks++)
                        mma_ss(tmem + (gs & 1) * NV, desc_mnmajor<BT>(sa, ks), desc_mnmajor<BT>(sb, ks), IDESC, ks > 0);
                    mma_commit(&m.u_full[gs & 1]);
                    mma_commit(&m.stage_empty[st]);
                }
            }
    } else if (warp == (NS + NWT) / 32 + 2) {
        if constexpr (!GK) {
        // ---- gates: log-decays (four bytes each, rows are H apart) five steps ahead, running sums -> weights --------------------
        int gs = 0;
        bool alive = true;
        for (int k = 0; alive && wait_warp(&m.item_full[k % ITEMS], k / ITEMS); k++) {
            const Item it = m.items[k % ITEMS];
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[k % ITEMS]);
            if (it.seq < 0) break;
            auto request = [&](int i) {
                if (i < it.n_steps)
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const int vr = chunk_of(it, i) * BT + lane + 32 * u;
                        const int r = vr >= it.n_virtual ? -1 : (vr < it.n_replay ? tb.replay_row[it.replay_base + vr] : it.own_begin + vr - it.n_replay);
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(&m.raw[i % RAW][lane + 32 * u])),
                                     "l"(g + (size_t)(r < 0 ? 0 : r) * H + it.h), "r"(r < 0 ? 0 : 4) : "memory");
                    }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            for (int i = 0; i < 5; i++) request(i);
            for (int i = 0; i < it.n_steps; i++, gs++) {
                request(i + 5);
                asm volatile("cp.async.wait_group 5;" ::: "memory");
                float y[2] = {m.raw[i % RAW][lane] * LOG2E, m.raw[i % RAW][lane + 32] * LOG2E};
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float y0 = __shfl_up_sync(~0u, y[0], o), y1 = __shfl_up_sync(~0u, y[1], o);
                    if (lane >= o) {
                        y[0] += y0;
                        y[1] += y1;
                    }
                }
                y[1] += __shfl_sync(~0u, y[0], 31);
                const float bn = __shfl_sync(~0u, y[1], 31);
                if (gs >= GATES && !(alive = wait_warp(&m.gates_empty[gs % GATES], gs / GATES - 1))) break;
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int vr = chunk_of(it, i) * BT + lane + 32 * u;
                    // backward: rows without an output (replayed, past the end) carry no dO
                    m.w[gs % GATES][lane + 32 * u] = BWD ? (vr >= it.n_replay && vr < it.n_virtual ? ex2(y[u]) : 0.f) : ex2(bn - y[u]);
                }
                if (lane == 0) m.gamma[gs % GATES] = ex2(bn);
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.gates_full[gs % GATES]);
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
        }
        }
    } else {
        // ---- tile stores (backward: and the loads of S_c into their buffers) -----------------------------------------------------
        int gt = 0;
        bool alive = true;
        if (BWD && lane == 0) {
            int loaded = 0, k = 0, i = 0, n = 0, chunk_base = 0, h = 0, slice = 0;
            // requests S_c for the next tile, in this item or the next that has one; false: there is none
            auto request = [&] {
                while (i >= n) {
                    if (!wait(&m.item_full[k % ITEMS], k / ITEMS)) return false;
                    const Item& it = m.items[k % ITEMS];
                    const int seq = it.seq;
                    n = it.n_chunks;
                    chunk_base = it.chunk_base;
                    h = it.h;
                    slice = it.slice;
                    mbar_arrive(&m.item_empty[k++ % ITEMS]);
                    if (seq < 0) return false;
                    i = 1;
                }
                const int buf = loaded++ % OUTS, idx = (chunk_base + n - 1 - i++) * H + h;
                m.tile[buf] = make_int2(idx, slice);
                mbar_expect_tx(&m.out_empty[buf], S::O);
                for (int p = 0; p < (NV + 63) / 64; p++)
                    tma_load_3d(smem + S::out + buf * S::O + p * S_PANEL, &map_s, slice * NV + p * 64, 0, idx, &m.out_empty[buf]);
                return true;
            };
            bool more = true;
            while (more && loaded < OUTS) more = request();
            for (; gt < loaded; gt++) {
                if (!wait(&m.out_full[gt % OUTS], gt / OUTS)) break;
                const int2 tile = m.tile[gt % OUTS];
                for (int p = 0; p < (NV + 63) / 64; p++)
                    tma_store_3d(&map_tiles, smem + S::out + (gt % OUTS) * S::O + p * S_PANEL, tile.y * NV + p * 64, 0, tile.x);
                tma_store_commit();
                if (!more) continue;
                tma_store_wait_read();
                more = request();
            }
            tma_store_wait_all();
        } else if (lane == 0) {
            int n_exported = 0;
            for (int k = 0; alive && wait(&m.item_full[k % ITEMS], k / ITEMS); k++) {
                const Item it = m.items[k % ITEMS];
                mbar_arrive(&m.item_empty[k % ITEMS]);
                if (it.seq < 0) break;
                int req = it.req_lo, boundary = req < it.req_hi ? tb.slot_chunk[req] : -1;
                for (int i = 0; i < it.n_chunks; i++, gt++) {
                    if (!(alive = wait(&m.out_full[gt % OUTS], gt / OUTS))) break;
                    const int idx = (it.chunk_base + chunk_of(it, i)) * H + it.h;
                    for (int p = 0; p < (NV + 63) / 64; p++)
                        tma_store_3d(&map_tiles, smem + S::out + (gt % OUTS) * S::O + p * S_PANEL, it.slice * NV + p * 64, 0, idx);
                    tma_store_commit();
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");      // the tile before this one has left its buffer
                    if (gt > 0) mbar_arrive(&m.out_empty[(gt - 1) % OUTS]);
                    if (boundary == i) {          // the state warps have written this boundary's slot: tell the sequences that wait
                        if (!(alive = wait(&m.exported[n_exported % EXPORTS], n_exported / EXPORTS))) break;
                        n_exported++;
                        if (order.n) flag_set(flags + ((size_t)req * H + it.h) * SLICES + it.slice);
                        req++;
                        boundary = req < it.req_hi ? tb.slot_chunk[req] : -1;
                    }
                }
            }
            tma_store_wait_all();
        }
    }
    __syncwarp();
    if (__syncthreads_or(m.dead)) drain_delay();          // abandoned: copies and MMAs in flight must land before the CTA goes
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc<2 * NV>(tmem);
}

struct Launch {
    const harts_la_tables_t& tb;
    int seq_lo, seq_hi, H;
    const void *a, *b;
    const float* g;
    void* tiles;
    const void* states;      // backward: the forward's tiles
    float *slots, *ds0, *dots;
    int* status;
    const int32_t* gate;
    int* flags;              // all rounds in one launch (order.n > 0): the ticket, then counters per (slot | sequence, head, slice)
    const RoundOrder& order;
    cudaStream_t stream;
};

template <bool BWD, int NV, bool GK>
int32_t launch(const Launch& x) {
    using S = Shape<NV, GK>;
    CUtensorMap ma, mb, mg, mt, ms;
    int32_t rc;
    const int64_t n_tiles = (int64_t)x.tb.n_chunks * x.H;
    if ((rc = make_row_map(&ma, x.a, x.tb.n_rows, x.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mb, x.b, x.tb.n_rows, x.H)) != HARTS_OK) return rc;
    mg = ma;
    if (GK && (rc = make_gate_map(&mg, x.g, x.tb.n_rows, x.H)) != HARTS_OK) return rc;
    if ((rc = NV == 32 ? make_state_slice_map(&mt, x.tiles, n_tiles) : make_state_map(&mt, x.tiles, n_tiles)) != HARTS_OK) return rc;
    ms = mt;
    if (BWD && (rc = NV == 32 ? make_state_slice_map(&ms, x.states, n_tiles) : make_state_map(&ms, x.states, n_tiles)) != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(scan_kernel<BWD, NV, GK>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes) != cudaSuccess)
        return HARTS_ECUDA;
    const int n = (x.seq_hi - x.seq_lo) * x.H * (D / NV), resident = (NV == 32 ? 2 : 1) * sm_count();
    if (x.order.n) {
        const size_t n_flags = (size_t)(BWD ? x.tb.n_seq : x.tb.n_slots) * x.H * (D / NV);
        if (cudaMemsetAsync(x.flags, 0, (4 + n_flags) * sizeof(int), x.stream) != cudaSuccess) return HARTS_ECUDA;
    }
    scan_kernel<BWD, NV, GK><<<n < resident ? n : resident, S::NT, S::bytes, x.stream>>>(
        x.tb, x.seq_lo, n, x.H, ma, mb, mg, mt, ms, (const __nv_bfloat16*)x.a, (const __nv_bfloat16*)x.b, x.g, x.slots, x.ds0, x.dots, x.status, x.gate,
        x.flags + 4, x.flags, x.order);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}
// The narrower the slices, the shorter a step of the walk and the more often k is read: as narrow as leaves the chains of the
// (first) round at most one CTA per SM, but never 128 columns in the backward, where a state thread multiplies its columns with
// S_c besides.  Device time in us with 32 / 64 / 128 columns, cold inputs, as they were when the line was drawn (a step is shorter now with
// any of them): 17,695 tokens x 4 heads (4 chains in the first round) forward 78 / 93 / 141, backward 82 / 86 / 187; 65,521 x 16 (64 chains)
// 298 / 244 / 289, 406 / 293 / 451; 100,003 x 16 (96 chains) 426 / 359 / 345, 606 / 468 / 561; 149,270 x 12 (96 chains) forward 64: 401,
// 128: 400, backward 546, 573.
template <bool BWD>
int32_t launch_sliced(const Launch& x) {
    const int chains = (x.order.n ? x.order.ptr[1] - x.order.ptr[0] : x.seq_hi - x.seq_lo) * x.H;
    if (4 * chains <= sm_count()) return launch<BWD, 32, false>(x);
    if constexpr (!BWD)
        if (2 * chains > sm_count()) return launch<false, 128, false>(x);
    return launch<BWD, 64, false>(x);
}

}  // namespace

// order.n == 0: sequences [seq_lo, seq_hi) of one round; otherwise all rounds in one launch: the CTAs draw the (sequence,
// head, slice) items from a ticket counter, first round first (backward: last round first), and one that starts from an
// exported state (backward: one that exported a boundary) waits for the counters of its producer (consumers).  Those hold
// smaller tickets, a ticket is only ever held by a running CTA, and a CTA works its tickets off in order, so an ordinary
// launch cannot deadlock.
int32_t scan_fwd(const FwdArgs& a, int* flags, const RoundOrder& order) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    return launch_sliced<false>({a.tb, a.seq_lo, a.seq_hi, a.H, a.k, a.v, a.g, a.chunk_states, nullptr, a.slots, nullptr, nullptr, a.dev_status,
                                 status_gate(a.flags, a.dev_status), flags, order, a.stream});
}

int32_t scan_bwd(const BwdArgs& a, void* ds_tiles, float* dots, int* flags, const RoundOrder& order) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    float* ds0 = (float*)((char*)a.scratch + scratch_layout(a.tb, a.H, a.dk, a.dv).ds0);
    return launch_sliced<true>({a.tb, a.seq_lo, a.seq_hi, a.H, a.q, a.dO, a.g, ds_tiles, a.chunk_states, nullptr, ds0, dots, a.dev_status,
                                status_gate(a.flags, a.dev_status), flags, order, a.stream});
}

// The same with a log-decay per key channel (FwdArgs::g / BwdArgs::g point to [rows, H, 128]): two slices of 64 columns while
// that leaves every SM at most one CTA, else one of 128 (the gate tile is as large as k and v together, so slices cost more).
template <bool BWD>
static int32_t launch_gk(const Launch& x) {
    const int chains = (x.order.n ? x.order.ptr[1] - x.order.ptr[0] : x.seq_hi - x.seq_lo) * x.H;
    return 2 * chains <= sm_count() ? launch<BWD, 64, true>(x) : launch<BWD, 128, true>(x);
}
int32_t gk_scan_fwd(const FwdArgs& a, int* flags, const RoundOrder& order) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    return launch_gk<false>({a.tb, a.seq_lo, a.seq_hi, a.H, a.k, a.v, a.g, a.chunk_states, nullptr, a.slots, nullptr, nullptr, a.dev_status,
                             status_gate(a.flags, a.dev_status), flags, order, a.stream});
}
int32_t gk_scan_bwd(const BwdArgs& a, void* ds_tiles, float* dots, int* flags, const RoundOrder& order) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    float* ds0 = (float*)((char*)a.scratch + gk_scratch_layout(a.tb, a.H, a.dk, a.dv).ds0);
    return launch_gk<true>({a.tb, a.seq_lo, a.seq_hi, a.H, a.q, a.dO, a.g, ds_tiles, a.chunk_states, nullptr, ds0, dots, a.dev_status,
                            status_gate(a.flags, a.dev_status), flags, order, a.stream});
}

}  // namespace harts
