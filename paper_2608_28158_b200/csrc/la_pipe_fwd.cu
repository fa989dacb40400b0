// Pipelined forward walk of the packed chunkwise call (bf16, d_k = d_v = 128, chunk 64): states, slots and outputs in one pass.
//
//     A = Q K^T    P = A .* e^{b_t-b_j} [j<=t]    o_t = P V + e^{b_t} Q S_c    S_{c+1} = e^{b_n} S_c + K~^T V,  k~_j = e^{b_n-b_j} k_j
//
// One CTA walks the chunks of a (sequence, head) -- or of NV = 64 of its 128 state columns, which do not interact -- but no phase of a
// chunk waits for the phases of the chunk before it, except one: a multiply-add per element of the state.  The products do not
// depend on the chain (the sum K~^T V of a chunk is a tcgen05 product of its own), the state stays in the registers of the state
// warps, and everything else runs a chunk ahead of it or behind it, by warps of their own that meet at mbarriers only:
//   load warp    draws the items, requests q, k, v by TMA up to STAGES chunks ahead (replayed rows row by row), asks the L2 for one more
//   gate warp    log-decays five chunks ahead, running sums -> the chunk's record (decays, row ids, what the others need to know)
//   MMA warp     A of chunk n + 1, then the sum, S_c^T Q^T and V^T P^T of chunk n (an elected lane)
//   work warps   decay masking of A (lanes 0..63: two warps) | k rows weighted in place (the other two)
//   output warps o of a chunk out of tensor memory
//   state warps  S_c as a bf16 tile for the product and the chunk-state workspace, exported slots, S_{c+1}
//   store warp   state tiles by TMA, and word to other CTAs that a slot is written
// Outputs are staged over the q rows they were made of, and the gate warp, which reuses their chunk's record next, sends them off.
// Every wait is bounded; one that runs out latches, and the CTA leaves all loops.
//
// What bounds it: HBM where chains are many (4,696 chunks x 32 heads 2,946 -> 2,480 us, 98 KB an item: 5.9 TB/s; 2,389 x 16 in chains of
// up to 293 chunks 1,230 -> 700), else the 1.5 us of a chunk's busiest role (1,047 x 16 in 64 chains, two slices each: scan and chunk
// kernel 492 -> 400).  First figures: the synchronous walk of la_tc_fwd.cu or la_scan.cu with la_chunk_fwd.cu.  What made it:
//   * instruction memory: seven roles inlined and unrolled were 75 KB of code, 29 % of the instruction cache's requests missed, and a
//     warp waited for instructions longer than for anything else (3,090 us; slow paths of waits out of line, passes as loops: 2,885);
//   * a chunk more asked of the L2, since three stages do not cover the latency of memory under load (2,885 -> 2,710; two more 2,860);
//   * two values an instruction in the element-wise passes, masking without exponentials off the diagonal (2,710 -> 2,640);
//   * the switch to the next sequence: start state by whole sectors and asked of the L2 when the sequence is drawn, replayed rows with
//     more copies in flight (2,690 -> 2,480; 249 branchy sequences' worth of 3,439 chunks x 16: 1,383 -> 1,076).
#include "kernels.h"
#include "tc_common.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int32_t make_state_map(CUtensorMap* map, const void* base, int64_t n);
int sm_count();

namespace {

using namespace tc;

constexpr int BT = 64, D = 128;
constexpr int NS = 256, NW = 128, NO = 128, NT = NS + NW + NO + 128;       // state, weighting and output threads, four warps
// the first of the four: store, load, gate, MMA.  A warp's number mod 4 is its scheduler, and masking sits on the first two.
constexpr int FIRST = (NS + NW + NO) / 32;
constexpr int RAW = 8, ITEMS = 4, EXPORTS = 4;                 // rings: raw log-decays, items, slots written
constexpr int PANEL = BT * 128, S_PANEL = D * 128;
constexpr float LOG2E = 1.4426950408889634f;

template <int NV>
struct Shape {
    static constexpr int CW = NV / 2;                      // state columns per state thread
    static constexpr int STAGES = NV == 64 ? 4 : 3;        // chunks of rows in shared memory, and chunk records: as many, since the
                                                           // gate warp gives a stage back when it reuses the record
    static constexpr int OUTS = NV == 64 ? 2 : 1;          // state tiles
    static constexpr int OB = NV == 64 ? 2 : 1;            // output accumulators
    static constexpr int VP = NV / 64;                     // panels of 64 columns of v, the state and the outputs
    static constexpr int Q = 0, K = 2 * PANEL, V = 4 * PANEL, STAGE = V + VP * PANEL, S = VP * S_PANEL;
    static constexpr int s = STAGES * STAGE, p = s + OUTS * S, misc = p + 2 * PANEL, bytes = misc + 9216 + 1024;
    // tensor memory: sums of a chunk (two), A (two), outputs (P V and Q S side by side)
    static constexpr int COL_U = 0, COL_A = 2 * NV, COL_O = COL_A + 128, COLS = 512;
    static_assert(COL_O + OB * 128 <= COLS, "tensor memory");
};
struct Item {                // one (sequence, head, slice); seq < 0: no more
    int seq, h, slice, own_begin, n_replay, n_virtual, n_chunks, chunk_base, replay_base, init_slot, req_lo, req_hi;
};
struct Record {              // one chunk
    float nb2[BT];           // minus the running log-decay, in log2 units
    float eb[BT];            // e^{b_t}
    float part[BT];          // rows 0..31: e^{b_31 - b_j}, rows 32..63: e^{b_t - b_31}; their product is the decay between the halves
    uint2 w[BT];             // e^{b_n - b_t} as the sum of two bf16, each twice
    int code[BT];            // physical row of an output (own rows), -1 elsewhere
    float gamma;             // e^{b_n}
    int h, col0, row0;       // row0: physical row of the chunk's first row, where all 64 are own rows (full)
    int full, step, end;     // step: the state is needed behind this chunk; end: no chunk, no more to come
    int pad;
};
struct Misc {
    Record rows[4];
    float raw[RAW][BT];
    uint64_t full[4], stage_empty[4], a_full[2], ready[2], u_full[2], s_full[2], s_empty[2],
        o_full[2], o_empty[2], gates_full[4], gates_empty[4], item_full[ITEMS], item_empty[ITEMS], exported[EXPORTS];
    Item items[ITEMS];
    uint32_t tmem;
    int dead;
    int* status;
};
static_assert(sizeof(Misc) <= 9216, "misc area");

// What a wait does past its first try is out of line: see the note on instruction memory above.
static __device__ __noinline__ bool wait_on(uint64_t* bar, uint32_t parity, Misc* m) { return mbar_wait_warp(bar, parity, m->status, &m->dead); }
static __device__ __noinline__ bool wait_on_both(uint64_t* bar, uint32_t parity, uint64_t* bar2, uint32_t parity2, Misc* m) {
    return mbar_wait_warp(bar, parity, m->status, &m->dead) && mbar_wait_warp(bar2, parity2, m->status, &m->dead);
}
// a place in a ring of N and the parity of its barrier's current phase
template <int N>
struct Ring {
    int i = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next() {
        if (++i == N) {
            i = 0;
            ph ^= 1;
        }
    }
};

__device__ __forceinline__ uint32_t f2_bf16(F2 x) {
    float a, b;
    f2_split(x, a, b);
    return pack_bf16(a, b);
}
// Two bf16 values times a weight that is the sum of two bf16 (w.x: the weight cut off, w.y: the rest, above zero): rounded once but for
// 2^-17 of the product, in two instructions instead of five.
__device__ __forceinline__ uint32_t weighted(uint32_t x, uint2 w) {
    uint32_t y;
    asm("{\n\t.reg .b32 t;\n\tmul.rn.bf16x2 t, %1, %3;\n\tfma.rn.bf16x2 %0, %1, %2, t;\n\t}" : "=r"(y) : "r"(x), "r"(w.x), "r"(w.y));
    return y;
}
__device__ __forceinline__ uint2 split_weight(float w) {
    const uint32_t hi = __float_as_uint(w) & 0xffff0000u;
    // not zero even where nothing is left, so that an infinite x stays one
    const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(fmaxf(w - __uint_as_float(hi), 1.2e-38f)));
    return make_uint2(hi | (hi >> 16), lo | (lo << 16));
}

// Operand descriptors of 128-byte-swizzled panels by halves: the upper word is the same for all, a step of 16 rows or columns adds to the
// lower one.
constexpr uint32_t DESC_HI = (1024 >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo_k(uint32_t tile) { return ((tile & 0x3FFFF) >> 4) | (1u << 16); }      // K contiguous
template <int KROWS>
__device__ __forceinline__ uint32_t desc_lo_mn(uint32_t tile) { return ((tile & 0x3FFFF) >> 4) | ((uint32_t)(KROWS * 128 >> 4) << 16); }
template <bool ADD>
__device__ __forceinline__ void mma_lo(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\tsetp.ne.b32 p, %5, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n\t}" ::"r"(d), "r"(a), "r"(b), "r"(DESC_HI), "r"(idesc), "n"(ADD ? 1 : 0) : "memory");
}
// d (+)= sum over k-steps; the lower words advance by SA, SB a step, by GA more behind the fourth (K contiguous: the next panel)
template <int STEPS, int SA, int SB, int GA, int GB>
__device__ __forceinline__ void mma_steps(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc) {
    mma_lo<false>(d, a, b, idesc);
#pragma unroll
    for (int ks = 1; ks < STEPS; ks++) mma_lo<true>(d, a + ks * SA + (ks >> 2) * GA, b + ks * SB + (ks >> 2) * GB, idesc);
}

template <int NV>
__global__ void __launch_bounds__(NT, 1)
pipe_fwd_kernel(const harts_la_tables_t tb, int seq_lo, int n_items, int H, const __grid_constant__ CUtensorMap map_q,
                const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                const __grid_constant__ CUtensorMap map_cs, const __grid_constant__ CUtensorMap map_o,
                const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                const float* __restrict__ g, __nv_bfloat16* __restrict__ o, float* slots, int store_states, int* status,
                const int32_t* gate, int* flags, int* ticket) {
    if (gate_closed(gate)) return;
    using S = Shape<NV>;
    constexpr int SLICES = D / NV, CW = S::CW, STAGES = S::STAGES, OUTS = S::OUTS, OB = S::OB, VP = S::VP;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    Misc& m = *reinterpret_cast<Misc*>(smem + S::misc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int i = 0; i < STAGES; i++) {
            mbar_init(&m.full[i], 1);
            mbar_init(&m.stage_empty[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&m.a_full[i], 1);
            mbar_init(&m.ready[i], NW / 32);
            mbar_init(&m.u_full[i], 1);
            mbar_init(&m.s_full[i], NS / 32);
            mbar_init(&m.s_empty[i], 2);                   // the product that read it, and the store warp
            mbar_init(&m.o_full[i], 1);
            mbar_init(&m.o_empty[i], NV / 32);
        }
        for (int i = 0; i < STAGES; i++) {
            mbar_init(&m.gates_full[i], 1);
            mbar_init(&m.gates_empty[i], (NS + NW + NO) / 32);
        }
        for (int i = 0; i < ITEMS; i++) {
            mbar_init(&m.item_full[i], 1);
            mbar_init(&m.item_empty[i], NS / 32 + 3);
        }
        for (int i = 0; i < EXPORTS; i++) mbar_init(&m.exported[i], NS / 32);
        m.dead = 0;
        m.status = status;
        fence_barrier_init();
    }
    if (warp == 0) {
        __syncwarp();
        tmem_alloc<S::COLS>(&m.tmem);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = m.tmem;
    // a whole warp; parity: of the phase that has to be over (a barrier just initialised: 1 is over)
    auto wait = [&](uint64_t* bar, uint32_t parity) { return __builtin_expect(__all_sync(~0u, mbar_try(bar, parity)), 1) || wait_on(bar, parity, &m); };
    // two at once, both tries in flight
    auto wait_both = [&](uint64_t* bar, uint32_t parity, uint64_t* bar2, uint32_t parity2) {
        const bool one = mbar_try(bar, parity), two = mbar_try(bar2, parity2);
        return __builtin_expect(__all_sync(~0u, one && two), 1) || wait_on_both(bar, parity, bar2, parity2, &m);
    };

    if (warp < NS / 32) {
        // ---- state: row L, columns col0 .. col0 + CW - 1 of the slice ------------------------------------------------------
        const int L = (warp & 3) * 32 + lane, col0 = (warp >> 2) * CW;
        const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16) + S::COL_U + col0;
        Ring<ITEMS> ri;
        Ring<STAGES> rg;
        Ring<OUTS> rs;
        Ring<2> ru;
        int n_exported = 0;
        bool alive = true;
        for (; alive && wait(&m.item_full[ri.i], ri.ph);) {
            const Item& item = m.items[ri.i];
            const int seq = item.seq, h = item.h, slice = item.slice, n_chunks = item.n_chunks, init_slot = item.init_slot, req_hi = item.req_hi;
            int req = item.req_lo;
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[ri.i]);
            ri.next();
            if (seq < 0) break;
            const size_t in_state = (size_t)L * D + slice * NV + col0;
            F2 x[CW / 2];
#pragma unroll
            for (int e = 0; e < CW / 2; e++) x[e] = f2(0.f, 0.f);
            if (init_slot >= 0) {
                const size_t from = (size_t)init_slot * H + h;
                const float* src = slots + from * (D * D) + in_state;
                if (ticket) alive = flag_wait_warp(flags + from * SLICES + slice, 1, status, &m.dead);
                // a thread's row is 512 bytes from the next one's: whole sectors at a time, where the array allows it
                if ((reinterpret_cast<uintptr_t>(slots) & 31) == 0) {
#pragma unroll
                    for (int e = 0; e < CW / 8; e++)
                        asm volatile("ld.global.v4.b64 {%0, %1, %2, %3}, [%4];"
                                     : "=l"(x[4 * e].v), "=l"(x[4 * e + 1].v), "=l"(x[4 * e + 2].v), "=l"(x[4 * e + 3].v) : "l"(src + 8 * e) : "memory");
                } else {
#pragma unroll
                    for (int e = 0; e < CW / 4; e++) {
                        const float4 y = __ldcg(reinterpret_cast<const float4*>(src) + e);
                        x[2 * e] = f2(y.x, y.y);
                        x[2 * e + 1] = f2(y.z, y.w);
                    }
                }
            }
            int boundary = req < req_hi ? tb.slot_chunk[req] : -1;
            for (int c = 0; c < n_chunks && alive; c++) {
                if (!wait(&m.s_empty[rs.i], rs.ph ^ 1)) break;
                unsigned char* dst = smem + S::s + rs.i * S::S + (col0 >> 6) * S_PANEL;
#pragma unroll
                for (int v8 = 0; v8 < CW / 8; v8++)
                    *reinterpret_cast<uint4*>(dst + sw128_chunk(L, (col0 & 63) / 8 + v8)) =
                        make_uint4(f2_bf16(x[4 * v8]), f2_bf16(x[4 * v8 + 1]), f2_bf16(x[4 * v8 + 2]), f2_bf16(x[4 * v8 + 3]));
                tc_fence_before();                // the sum of two chunks ago has been read
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.s_full[rs.i]);
                rs.next();
                if (boundary == c) {
                    float4* to = reinterpret_cast<float4*>(slots + ((size_t)req * H + h) * (D * D) + in_state);
#pragma unroll
                    for (int e = 0; e < CW / 4; e++) {
                        float4 y;
                        f2_split(x[2 * e], y.x, y.y);
                        f2_split(x[2 * e + 1], y.z, y.w);
                        to[e] = y;
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.exported[n_exported % EXPORTS]);      // the store warp publishes it
                    n_exported++;
                    req++;
                    boundary = req < req_hi ? tb.slot_chunk[req] : -1;
                }
                const bool step = c + 1 < n_chunks;       // behind the last chunk nobody needs the state
                alive = step ? wait_both(&m.gates_full[rg.i], rg.ph, &m.u_full[ru.i], ru.ph) : wait(&m.gates_full[rg.i], rg.ph);
                if (step) {
                    const float gamma = m.rows[rg.i].gamma;
                    const F2 gamma2 = f2(gamma, gamma);
                    tc_fence_after();
#pragma unroll
                    for (int blk = 0; blk < CW / 16; blk++) {
                        uint32_t u[16];
                        tmem_ld16(tm + ru.i * NV + blk * 16, u);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 8; e++)
                            x[blk * 8 + e] = f2_fma(gamma2, x[blk * 8 + e], f2(__uint_as_float(u[2 * e]), __uint_as_float(u[2 * e + 1])));
                    }
                    ru.next();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.gates_empty[rg.i]);
                rg.next();
            }
        }
    } else if (warp < (NS + NW) / 32) {
        // ---- work: masking of A, weighting of k ---------------------------------------------------------------------------------
        const int quarter = warp & 3, t = quarter * 32 + lane;
        const uint32_t tm_lane = tmem + ((uint32_t)(quarter * 32) << 16) + S::COL_A;
        Ring<STAGES> rg;
        Ring<2> ra;
        uint32_t seen[16];                        // the diagonal's 32 columns, two to a register: ones where the row sees the column
#pragma unroll
        for (int e = 0; e < 16; e++) seen[e] = (2 * e <= lane ? 0xffffu : 0u) | (2 * e + 1 <= lane ? 0xffff0000u : 0u);
        if (quarter == 0)                         // rows 0..31 see nothing of columns 32..63, in either tile of P
#pragma unroll
            for (int u = 0; u < 8; u++)
                *reinterpret_cast<uint4*>(smem + S::p + (u >> 2) * PANEL + sw128_chunk(t, 4 + (u & 3))) = make_uint4(0, 0, 0, 0);
        for (;;) {
            if (!wait(&m.gates_full[rg.i], rg.ph)) break;
            const Record& rd = m.rows[rg.i];
            if (rd.end) break;
            if (quarter < 2) {                    // P = A .* decay: lanes 0..63 hold the rows
                // (behind A of this chunk: the product that read this tile of P two chunks ago, which was issued before it, is done too)
                if (!wait(&m.a_full[ra.i], ra.ph)) break;
                tc_fence_after();
                unsigned char* sp = smem + S::p + ra.i * PANEL;
                uint32_t x[32];
                tmem_ld32(tm_lane + ra.i * 64 + quarter * 32, x);
                // the 32 columns on the diagonal
                {
                    const float bt = -rd.nb2[t];
                    float y[32];
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        const float4 bj = *reinterpret_cast<const float4*>(rd.nb2 + quarter * 32 + e);
                        f2_split(f2_add(f2(bt, bt), f2(bj.x, bj.y)), y[e], y[e + 1]);
                        f2_split(f2_add(f2(bt, bt), f2(bj.z, bj.w)), y[e + 2], y[e + 3]);
                    }
#pragma unroll
                    for (int e = 0; e < 32; e++) y[e] = ex2(y[e]);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; e++)          // above the diagonal the product may be inf or NaN: bits taken out, not multiplied
                        x[e] = seen[e] & f2_bf16(f2_mul(f2(y[2 * e], y[2 * e + 1]), f2(__uint_as_float(x[2 * e]), __uint_as_float(x[2 * e + 1]))));
#pragma unroll
                    for (int v4 = 0; v4 < 4; v4++)
                        *reinterpret_cast<uint4*>(sp + sw128_chunk(t, quarter * 4 + v4)) = make_uint4(x[4 * v4], x[4 * v4 + 1], x[4 * v4 + 2], x[4 * v4 + 3]);
                }
                // rows 32..63 see all of columns 0..31: the decay in two factors, one of the row and one of the column
                if (quarter == 1) {
                    tmem_ld32(tm_lane + ra.i * 64, x);
                    const float f = rd.part[t];
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; e += 2) {
                        const float4 hj = *reinterpret_cast<const float4*>(rd.part + 2 * e);
                        x[e] = f2_bf16(f2_mul(f2_mul(f2(f, f), f2(hj.x, hj.y)), f2(__uint_as_float(x[2 * e]), __uint_as_float(x[2 * e + 1]))));
                        x[e + 1] = f2_bf16(f2_mul(f2_mul(f2(f, f), f2(hj.z, hj.w)), f2(__uint_as_float(x[2 * e + 2]), __uint_as_float(x[2 * e + 3]))));
                    }
#pragma unroll
                    for (int v4 = 0; v4 < 4; v4++)
                        *reinterpret_cast<uint4*>(sp + sw128_chunk(t, v4)) = make_uint4(x[4 * v4], x[4 * v4 + 1], x[4 * v4 + 2], x[4 * v4 + 3]);
                }
                tc_fence_before();
                fence_async_smem();
            } else {                              // k rows weighted in place, once A has been made of them: a panel of 64 columns per warp
                if (!wait_both(&m.full[rg.i], rg.ph, &m.a_full[ra.i], ra.ph)) break;
                if (rd.step) {
                    unsigned char* sk = smem + rg.i * S::STAGE + S::K + (quarter - 2) * PANEL;
#pragma unroll 1
                    for (int t0 = lane >> 3; t0 < BT; t0 += 16) {
                        uint4 y[4];
                        uint2 w[4];
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            y[u] = *reinterpret_cast<const uint4*>(sk + sw128_chunk(t0 + 4 * u, lane & 7));
                            w[u] = rd.w[t0 + 4 * u];
                        }
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            y[u].x = weighted(y[u].x, w[u]), y[u].y = weighted(y[u].y, w[u]), y[u].z = weighted(y[u].z, w[u]), y[u].w = weighted(y[u].w, w[u]);
                            *reinterpret_cast<uint4*>(sk + sw128_chunk(t0 + 4 * u, lane & 7)) = y[u];
                        }
                    }
                    fence_async_smem();
                }
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&m.ready[ra.i]);
                mbar_arrive(&m.gates_empty[rg.i]);
            }
            rg.next();
            ra.next();
        }
    } else if (warp < FIRST) {
        // ---- outputs: features 32 (warp & 3) .. + 31 of the slice; staged over the chunk's q rows ----------------------------------
        const int quarter = warp & 3, Lq = quarter * 32, c4 = lane & 3, f0 = Lq + 8 * (lane >> 3);
        const uint32_t tm_lane = tmem + ((uint32_t)Lq << 16);
        Ring<STAGES> ro;
        Ring<OB> rb;
        for (;;) {
            if (!wait(&m.gates_full[ro.i], ro.ph)) break;
            const Record& rd = m.rows[ro.i];
            if (rd.end) break;
            if (Lq < NV) {
                unsigned char* so = smem + ro.i * S::STAGE + S::Q;
                if (!wait(&m.o_full[rb.i], rb.ph)) break;    // every product that read the stage is done
                tc_fence_after();
#pragma unroll 1
                for (int t0 = 0; t0 < BT; t0 += 16) {
                    uint32_t x1[2][8], x2[2][8];
#pragma unroll
                    for (int l = 0; l < 2; l++) {
                        tmem_ld_frag16(tm_lane + ((uint32_t)(16 * l) << 16) + S::COL_O + rb.i * 128 + t0, x1[l]);
                        tmem_ld_frag16(tm_lane + ((uint32_t)(16 * l) << 16) + S::COL_O + rb.i * 128 + 64 + t0, x2[l]);
                    }
                    float2 e2[2];
#pragma unroll
                    for (int ta = 0; ta < 2; ta++) e2[ta] = *reinterpret_cast<const float2*>(rd.eb + t0 + ta * 8 + 2 * c4);
                    tmem_ld_wait();
#pragma unroll
                    for (int ta = 0; ta < 2; ta++) {
                        uint32_t pk[4];
#pragma unroll
                        for (int fa = 0; fa < 4; fa++) {
                            const int l = fa >> 1, r = 4 * ta + 2 * (fa & 1);
                            pk[fa] = f2_bf16(f2_fma(f2(e2[ta].x, e2[ta].y), f2(__uint_as_float(x2[l][r]), __uint_as_float(x2[l][r + 1])),
                                                    f2(__uint_as_float(x1[l][r]), __uint_as_float(x1[l][r + 1]))));
                        }
                        stmatrix_x4_trans(smem_u32(so) + (f0 >> 6) * PANEL + sw128_chunk(t0 + 8 * ta + (lane & 7), (f0 & 63) >> 3), pk);
                    }
                }
                tc_fence_before();
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.o_empty[rb.i]);
                if (!rd.full) {               // the rows of this warp that are outputs, 64 bytes of each
#pragma unroll 1
                    for (int e = lane; e < 256; e += 32) {
                        const int t = e >> 2, f = Lq + 8 * (e & 3), row = rd.code[t];
                        if (row >= 0)
                            *reinterpret_cast<uint4*>(o + ((size_t)row * H + rd.h) * D + rd.col0 + f) =
                                *reinterpret_cast<const uint4*>(so + (f >> 6) * PANEL + sw128_chunk(t, (f & 63) >> 3));
                    }
                    __syncwarp();
                }
            }
            if (lane == 0) mbar_arrive(&m.gates_empty[ro.i]);
            ro.next();
            rb.next();
        }
    } else {
    if (warp == FIRST + 1) {
        // ---- items and loads: the next item is drawn when the loads of the one before are on their way, not earlier (a CTA that
        // walks a long sequence must not sit on the items behind it) ---------------------------------------------------------------
        Ring<ITEMS> ri;
        Ring<STAGES> rt;
        bool alive = true;
        for (int kk = 0; alive; kk++) {
            if (!wait(&m.item_empty[ri.i], ri.ph ^ 1)) break;
            // one launch per round: dealt in a snake, longest sequences first
            const int G = (int)gridDim.x, b = (int)blockIdx.x;
            int pos = kk * G + ((kk & 1) ? G - 1 - b : b);
            if (ticket) {
                if (lane == 0) pos = atomicAdd(ticket, 1);
                pos = __shfl_sync(~0u, pos, 0);
            }
            Item it;
            it.seq = -1;
            if (pos < n_items) {
                it.slice = pos % SLICES;
                it.h = pos / SLICES % H;
                const int sp = seq_lo + pos / SLICES / H;
                it.seq = tb.seq_order ? tb.seq_order[sp] : sp;
                // one table entry per lane
                const int32_t* from = lane < 2 ? tb.seq_own_begin + lane : lane < 4 ? tb.seq_replay_ptr + (lane - 2)
                                    : lane < 6 ? tb.seq_req_ptr + (lane - 4) : lane == 6 ? tb.seq_chunk_ptr : tb.seq_init_slot;
                const int e = from[it.seq];
                auto entry = [&](int l) { return __shfl_sync(~0u, e, l); };
                it.own_begin = entry(0);
                it.replay_base = entry(2);
                it.n_replay = entry(3) - it.replay_base;
                it.n_virtual = it.n_replay + entry(1) - it.own_begin;
                it.n_chunks = (it.n_virtual + BT - 1) / BT;
                it.req_lo = entry(4);
                it.req_hi = entry(5);
                it.chunk_base = entry(6);
                it.init_slot = entry(7);
            }
            if (lane == 0) {
                m.items[ri.i] = it;
                mbar_arrive(&m.item_full[ri.i]);
            }
            ri.next();
            if (it.seq < 0) break;
            if (lane == 0 && it.init_slot >= 0 && it.slice == 0)      // its start state into the L2, chunks ahead of its use
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(slots + ((size_t)it.init_slot * H + it.h) * (D * D)), "n"(D * D * 4) : "memory");
            __syncwarp();
            const int v0 = it.slice * NV;
            for (int c = 0; c < it.n_chunks; c++, rt.next()) {
                const int st = rt.i, row0 = it.own_begin - it.n_replay + c * BT;
                unsigned char* tile = smem + st * S::STAGE;
                if (lane == 0 && c + 1 < it.n_chunks)
#pragma unroll 1
                    for (int p = 0; p < 2; p++) {
                        tma_prefetch_3d(&map_q, p * 64, it.h, row0 + BT);
                        tma_prefetch_3d(&map_k, p * 64, it.h, row0 + BT);
                        if (p < VP) tma_prefetch_3d(&map_v, v0 + p * 64, it.h, row0 + BT);
                    }
                __syncwarp();
                if (!(alive = wait(&m.stage_empty[st], rt.ph ^ 1))) break;
                if (c == 0 && it.n_replay > 0) {  // chunk 0 begins with rows from anywhere: row by row, two at a time
                    int row[2];
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const int t = lane + 32 * u;
                        row[u] = t >= it.n_virtual ? -1 : t < it.n_replay ? tb.replay_row[it.replay_base + t] : it.own_begin + t - it.n_replay;
                    }
                    const int ch = lane & 15;
#pragma unroll 4
                    for (int u = 0; u < BT / 2; u++) {
                        const int t = 2 * u + (lane >> 4), r0 = __shfl_sync(~0u, row[0], t & 31), r1 = __shfl_sync(~0u, row[1], t & 31);
                        const int r = u < BT / 4 ? r0 : r1;
                        const size_t off = ((size_t)max(r, 0) * H + it.h) * D;
                        unsigned char* dst = tile + (ch >> 3) * PANEL + sw128_chunk(t, ch & 7);
                        cp_async16(dst + S::Q, q + off + ch * 8, r >= 0 && t >= it.n_replay);
                        cp_async16(dst + S::K, k + off + ch * 8, r >= 0);
                        if (ch < NV / 8) cp_async16(dst + S::V, v + off + v0 + ch * 8, r >= 0);
                    }
                    cp_async_wait_all();
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.full[st]);
                } else if (lane == 0) {
                    mbar_expect_tx(&m.full[st], S::STAGE);
#pragma unroll 1
                    for (int p = 0; p < 2; p++) {
                        tma_load_3d(tile + S::Q + p * PANEL, &map_q, p * 64, it.h, row0, &m.full[st]);
                        tma_load_3d(tile + S::K + p * PANEL, &map_k, p * 64, it.h, row0, &m.full[st]);
                        if (p < VP) tma_load_3d(tile + S::V + p * PANEL, &map_v, v0 + p * 64, it.h, row0, &m.full[st]);
                    }
                }
            }
        }
    } else if (warp == FIRST + 3) {
        // ---- products ----------------------------------------------------------------------------------------------------------
        constexpr uint32_t IDESC_A = instr_desc(128, 64, 0, 0);    // Q x K, both K-major (rows 64..127 unused)
        constexpr uint32_t IDESC_O = instr_desc(128, 64, 1, 0);    // V^T x P, S^T x Q (a slice: rows 64..127 unused)
        constexpr uint32_t IDESC_U = instr_desc(128, NV, 1, 1);    // K~^T x V
        constexpr int K = 32 >> 4, KP = (BT * 128 - 4 * 32) >> 4, MN = 2048 >> 4;      // steps: along a row, to the next panel, 16 rows
        const uint32_t base = smem_u32(smem);
        Ring<ITEMS> ri;
        Ring<STAGES> ra, rt;          // stage of chunk n + 1, stage of chunk n
        Ring<2> rna, rp, ru;          // A of chunk n + 1, A and P of chunk n, sums
        Ring<OUTS> rs;
        Ring<OB> rb;
        bool alive = true;
        auto next_item = [&]() {                  // its chunks, or 0: there are no more
            for (;;) {
                if (!(alive = wait(&m.item_full[ri.i], ri.ph))) return 0;
                const int seq = m.items[ri.i].seq, chunks = m.items[ri.i].n_chunks;
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.item_empty[ri.i]);
                ri.next();
                if (seq < 0) return 0;
                if (chunks > 0) return chunks;
            }
        };
        auto product_a = [&]() {
            tc_fence_after();
            const uint32_t tile = base + ra.i * S::STAGE;
            if (elect_one()) {
                mma_steps<8, K, K, KP, KP>(tmem + S::COL_A + rna.i * 64, desc_lo_k(tile + S::Q), desc_lo_k(tile + S::K), IDESC_A);
                mma_commit(&m.a_full[rna.i]);
            }
            __syncwarp();
            ra.next();
            rna.next();
        };
        // A of chunk n + 1 goes ahead of chunk n's products if its rows are there, else behind them: waited for ahead, late rows would hold
        // up the stage that the loads after them wait for.  left: chunks of its item from n + 1 on
        int left = next_item();
        bool more = left > 0, step = false;
        for (bool begun = false; alive && (more || begun);) {
            const bool had = begun;               // chunk n exists; step: and chunk n + 1 is its item's
            // (its accumulator: P of chunk n - 1 was waited for)
            const bool early = more && had && __all_sync(~0u, mbar_try(&m.full[ra.i], ra.ph));
            if (early) product_a();
            if (had) {
                const uint32_t tile = base + rt.i * S::STAGE;
                // (the sum's accumulator: S of chunk n - 1, which was waited for, was made after the sum of chunk n - 2 was read)
                if (!(alive = wait(&m.ready[rp.i], rp.ph))) break;
                tc_fence_after();
                if (step) {
                    if (elect_one()) {
                        mma_steps<4, MN, MN, 0, 0>(tmem + S::COL_U + ru.i * NV, desc_lo_mn<BT>(tile + S::K), desc_lo_mn<BT>(tile + S::V), IDESC_U);
                        mma_commit(&m.u_full[ru.i]);
                    }
                    __syncwarp();
                    ru.next();
                }
                if (!(alive = wait_both(&m.s_full[rs.i], rs.ph, &m.o_empty[rb.i], rb.ph ^ 1))) break;
                tc_fence_after();
                const uint32_t acc = tmem + S::COL_O + rb.i * 128;
                if (elect_one()) {
                    mma_steps<8, MN, K, 0, KP>(acc + 64, desc_lo_mn<D>(base + S::s + rs.i * S::S), desc_lo_k(tile + S::Q), IDESC_O);
                    mma_commit(&m.s_empty[rs.i]);
                    mma_steps<4, MN, K, 0, 0>(acc, desc_lo_mn<BT>(tile + S::V), desc_lo_k(base + S::p + rp.i * PANEL), IDESC_O);
                    mma_commit(&m.o_full[rb.i]);
                }
                __syncwarp();
                rt.next();
                rs.next();
                rb.next();
                rp.next();
            }
            if (more && !early) {
                if (!(alive = wait(&m.full[ra.i], ra.ph))) break;
                product_a();
            }
            begun = more;                         // chunk n + 1 is the next round's n
            step = more && left > 1;
            if (more && --left == 0) left = next_item();
            more = left > 0;
        }
    } else if (warp == FIRST + 2) {
        // ---- gates: log-decays (four bytes each, rows are H apart) five chunks ahead, running sums -> the chunk's record ---------
        // and the outputs of the chunk that had the record before, which are staged now; their stage goes back to the load warp
        Ring<ITEMS> ri;
        Ring<STAGES> rg;
        int used = 0;                 // records that have had a chunk
        bool alive = true;
        auto take_record = [&]() {
            if (!wait(&m.gates_empty[rg.i], rg.ph ^ 1)) return false;
            if (used == STAGES && lane == 0) {
                const Record& rd = m.rows[rg.i];
                if (rd.full) {
#pragma unroll 1
                    for (int p = 0; p < VP; p++)
                        tma_store_3d(&map_o, smem + rg.i * S::STAGE + S::Q + p * PANEL, rd.col0 + p * 64, rd.h, rd.row0);
                    tma_store_commit();
                    tma_store_wait_read();
                }
                mbar_arrive(&m.stage_empty[rg.i]);
            }
            __syncwarp();
            return true;
        };
        for (; alive && wait(&m.item_full[ri.i], ri.ph);) {
            const Item it = m.items[ri.i];
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[ri.i]);
            ri.next();
            if (it.seq < 0) {
                if (!take_record()) break;
                if (lane == 0) {
                    m.rows[rg.i].end = 1;
                    mbar_arrive(&m.gates_full[rg.i]);
                }
#pragma unroll 1
                for (int i = 1; i < STAGES; i++) {        // what is still on its way out, oldest first
                    rg.next();
                    if (used < STAGES) used++;
                    if (!take_record()) break;
                }
                break;
            }
            auto row_of = [&](int vr) { return vr >= it.n_virtual ? -1 : vr < it.n_replay ? tb.replay_row[it.replay_base + vr] : it.own_begin + vr - it.n_replay; };
            auto request = [&](int c) {
                if (c < it.n_chunks)
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        const int r = row_of(c * BT + lane + 32 * u);
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(&m.raw[c % RAW][lane + 32 * u])),
                                     "l"(g + (size_t)(r < 0 ? 0 : r) * H + it.h), "r"(r < 0 ? 0 : 4) : "memory");
                    }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
#pragma unroll 1
            for (int c = -5; c < it.n_chunks; c++) {
                request(c + 5);
                if (c < 0) continue;
                asm volatile("cp.async.wait_group 5;" ::: "memory");
                float y[2] = {m.raw[c % RAW][lane] * LOG2E, m.raw[c % RAW][lane + 32] * LOG2E};
#pragma unroll
                for (int s = 1; s < 32; s <<= 1) {
                    const float y0 = __shfl_up_sync(~0u, y[0], s), y1 = __shfl_up_sync(~0u, y[1], s);
                    if (lane >= s) {
                        y[0] += y0;
                        y[1] += y1;
                    }
                }
                y[1] += __shfl_sync(~0u, y[0], 31);
                const float bn = __shfl_sync(~0u, y[1], 31), bh = __shfl_sync(~0u, y[0], 31);
                if (!(alive = take_record())) break;
                Record& rd = m.rows[rg.i];
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int t = lane + 32 * u, vr = c * BT + t;
                    rd.nb2[t] = -y[u];
                    rd.eb[t] = ex2(y[u]);
                    rd.w[t] = split_weight(ex2(bn - y[u]));
                    rd.code[t] = vr >= it.n_replay && vr < it.n_virtual ? it.own_begin + vr - it.n_replay : -1;
                }
                rd.part[lane] = ex2(bh - y[0]);
                rd.part[32 + lane] = ex2(y[1] - bh);
                if (lane == 0) {
                    rd.gamma = ex2(bn);
                    rd.h = it.h;
                    rd.col0 = it.slice * NV;
                    rd.row0 = it.own_begin - it.n_replay + c * BT;
                    rd.full = (c > 0 || it.n_replay == 0) && (c + 1) * BT <= it.n_virtual;
                    rd.step = c + 1 < it.n_chunks;
                    rd.end = 0;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.gates_full[rg.i]);
                rg.next();
                if (used < STAGES) used++;
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
        }
        if (lane == 0) tma_store_wait_all();
    } else {
        // ---- state tiles to the workspace; slots that the state warps have written are published to the sequences that wait ----------
        Ring<ITEMS> ri;
        Ring<OUTS> rs;
        Ring<EXPORTS> re;
        bool alive = true;
        for (; alive && wait(&m.item_full[ri.i], ri.ph);) {
            const Item& item = m.items[ri.i];
            const int seq = item.seq, h = item.h, slice = item.slice, n_chunks = item.n_chunks, chunk_base = item.chunk_base, req_hi = item.req_hi;
            int req = item.req_lo;
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.item_empty[ri.i]);
            ri.next();
            if (seq < 0) break;
            int boundary = req < req_hi ? tb.slot_chunk[req] : -1;
            for (int c = 0; c < n_chunks; c++) {
                if (!(alive = wait(&m.s_full[rs.i], rs.ph))) break;
                if (lane == 0) {
                    if (store_states) {
#pragma unroll 1
                        for (int p = 0; p < VP; p++)
                            tma_store_3d(&map_cs, smem + S::s + rs.i * S::S + p * S_PANEL, slice * NV + p * 64, 0, (chunk_base + c) * H + h);
                        tma_store_commit();
                        tma_store_wait_read();
                    }
                    mbar_arrive(&m.s_empty[rs.i]);
                }
                __syncwarp();
                rs.next();
                if (boundary == c) {
                    if (!(alive = wait(&m.exported[re.i], re.ph))) break;
                    re.next();
                    if (ticket && lane == 0) flag_set(flags + ((size_t)req * H + h) * SLICES + slice);
                    req++;
                    boundary = req < req_hi ? tb.slot_chunk[req] : -1;
                }
            }
        }
        if (lane == 0) tma_store_wait_all();
    }
    }
    __syncwarp();
    if (__syncthreads_or(m.dead)) drain_delay();          // abandoned: copies and MMAs in flight must land before the CTA goes
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc<S::COLS>(tmem);
}

template <int NV>
int32_t launch(const FwdArgs& a, int* flags, int* ticket) {
    using S = Shape<NV>;
    CUtensorMap mq, mk, mv, mcs, mo;
    int32_t rc;
    if ((rc = make_row_map(&mq, a.q, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mk, a.k, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mv, a.v, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mo, a.o, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    const void* cs = a.chunk_states ? a.chunk_states : a.q;   // a valid address for the (unused) map
    if ((rc = make_state_map(&mcs, cs, a.chunk_states ? (int64_t)a.tb.n_chunks * a.H : 1)) != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(pipe_fwd_kernel<NV>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::bytes) != cudaSuccess) return HARTS_ECUDA;
    const int n = (a.seq_hi - a.seq_lo) * a.H * (D / NV);
    pipe_fwd_kernel<NV><<<n < sm_count() ? n : sm_count(), NT, S::bytes, a.stream>>>(
        a.tb, a.seq_lo, n, a.H, mq, mk, mv, mcs, mo, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (__nv_bfloat16*)a.o, a.slots, a.chunk_states != nullptr, a.dev_status, status_gate(a.flags, a.dev_status), flags, ticket);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace

// flags == nullptr: sequences [a.seq_lo, a.seq_hi) of one round; otherwise all rounds in one launch (first_round: sequences of the first):
// the CTAs draw the (sequence, head, slice) items from a ticket counter in the plan's order, and one that starts from an exported
// state waits for the flag that its producer sets once the slot is written.  The producer holds a smaller ticket, a ticket is only
// ever held by a running CTA, and a CTA works its tickets off in order, so an ordinary launch cannot deadlock.
// flags: n_slots * H * 2 int32 behind one ticket; zeroed here on the stream.
int32_t pipe_fwd(const FwdArgs& a, int* flags, int first_round) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    const int chains = (flags ? first_round : a.seq_hi - a.seq_lo) * a.H;
    const bool narrow = 2 * chains <= sm_count();
    int *ticket = flags, *slot_flags = flags ? flags + 1 : nullptr;
    if (flags && cudaMemsetAsync(flags, 0, (1 + (size_t)a.tb.n_slots * a.H * (narrow ? 2 : 1)) * sizeof(int), a.stream) != cudaSuccess)
        return HARTS_ECUDA;
    return narrow ? launch<64>(a, slot_flags, ticket) : launch<128>(a, slot_flags, ticket);
}

}  // namespace harts
