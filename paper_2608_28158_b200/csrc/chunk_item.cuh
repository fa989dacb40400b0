// Work items of the chunk-parallel kernels: one (chunk, head), found by its position in the plan's chunk numbering.
#pragma once
#include "kernels.h"
#include "tc_common.cuh"

namespace harts {
namespace chunk {

constexpr int BT = 64, D = 128;
constexpr float LOG2E = 1.4426950408889634f;

struct Item {
    int gc, h;               // chunk (plan numbering), head; gc < 0: no more items
    int c, last;             // chunk index inside its sequence; 1: the sequence's last chunk
    int row0;                // physical row of the chunk's row 0 if all of them are own rows (TMA origin)
    int n_replay, n_rows;    // rows of this chunk that are replayed ancestor rows (first), rows in all
    int replay_base, own_begin, zero_state;
    __device__ bool gathered() const { return n_replay > 0; }
    __device__ bool full() const { return n_replay == 0 && n_rows == BT; }
};

// Called by a whole warp: the sequence that owns chunk gc (32-way search), then its record.
__device__ __forceinline__ Item find_item(const harts_la_tables_t& tb, int seq_lo, int seq_hi, int gc, int h, int lane) {
    int lo = seq_lo, hi = seq_hi;
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32, i = lo + lane * step;
        const unsigned m = __ballot_sync(~0u, i < hi && tb.seq_chunk_ptr[i] <= gc);
        lo += (__popc(m) - 1) * step;
        hi = min(hi, lo + step);
    }
    Item it;
    it.gc = gc;
    it.h = h;
    it.c = gc - tb.seq_chunk_ptr[lo];
    it.own_begin = tb.seq_own_begin[lo];
    it.replay_base = tb.seq_replay_ptr[lo];
    const int n_replay = tb.seq_replay_ptr[lo + 1] - it.replay_base;
    const int n_virtual = n_replay + tb.seq_own_begin[lo + 1] - it.own_begin;
    it.n_replay = it.c == 0 ? n_replay : 0;
    it.n_rows = min(BT, n_virtual - it.c * BT);
    it.last = (it.c + 1) * BT >= n_virtual;
    it.row0 = it.own_begin - n_replay + it.c * BT;
    it.zero_state = it.c == 0 && tb.seq_init_slot[lo] < 0;
    return it;
}

struct RowData {
    float b2[BT];            // running log-decay in log2 units
    float eb[BT];            // e^{b_t}
    float w[BT];             // e^{b_n - b_t}
    int code[BT];            // physical row (>= 0 own), -2 - row (replayed), -1 (past the end)
    float gamma;             // e^{b_n}
    float pad[3];
};

// One warp prepares a chunk's row data: lane and lane + 32 are its rows.  Split in two so that the loads of one item are in
// flight while an earlier one is worked on.
__device__ __forceinline__ void load_rows(const harts_la_tables_t& tb, const Item& it, const float* g, int H, int lane,
                                          int (&code)[2], float (&gv)[2]) {
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const int t = lane + 32 * r;
        code[r] = -1;
        gv[r] = 0.f;
        if (it.gc >= 0 && t < it.n_rows) {
            const int row = t < it.n_replay ? tb.replay_row[it.replay_base + t] : it.row0 + t;
            code[r] = t < it.n_replay ? -2 - row : row;
            gv[r] = g[(size_t)row * H + it.h];
        }
    }
}
__device__ __forceinline__ void store_rows(RowData& rd, const int (&code)[2], const float (&gv)[2], int lane) {
    float x0 = gv[0] * LOG2E, x1 = gv[1] * LOG2E;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float y0 = __shfl_up_sync(~0u, x0, o), y1 = __shfl_up_sync(~0u, x1, o);
        if (lane >= o) {
            x0 += y0;
            x1 += y1;
        }
    }
    x1 += __shfl_sync(~0u, x0, 31);
    const float bn = __shfl_sync(~0u, x1, 31);
    const float x[2] = {x0, x1};
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const int t = lane + 32 * r;
        rd.code[t] = code[r];
        rd.b2[t] = x[r];
        rd.eb[t] = tc::ex2(x[r]);
        rd.w[t] = tc::ex2(bn - x[r]);
    }
    if (lane == 0) rd.gamma = tc::ex2(bn);
}

// Matrix-fragment epilogue helpers: accumulators are transposed (tensor-memory lane = feature, column = row t of the chunk);
// tcgen05.ld 16x256b hands a warp 8x8 fragments, stmatrix.trans turns them into 16-byte pieces of rows in
// 128-byte-swizzled [row][64 features] panels.  A warp covers 32 features (its lane quarter) x 16 rows.
constexpr int PANEL = BT * 128;
__device__ __forceinline__ uint32_t frag_addr(uint32_t tile, int lane, int Lq, int t0, int ta) {
    const int f = Lq + 8 * (lane >> 3), t = t0 + 8 * ta + (lane & 7);
    return tile + (f >> 6) * PANEL + tc::sw128_chunk(t, (f & 63) >> 3);
}
__device__ __forceinline__ void frag_store(uint32_t stage, int lane, int Lq, int t0, const float (&val)[2][8]) {
#pragma unroll
    for (int ta = 0; ta < 2; ta++) {
        uint32_t pk[4];
#pragma unroll
        for (int fa = 0; fa < 4; fa++) {
            const int l = fa >> 1, r = 4 * ta + 2 * (fa & 1);
            pk[fa] = tc::pack_bf16(val[l][r], val[l][r + 1]);
        }
        tc::stmatrix_x4_trans(frag_addr(stage, lane, Lq, t0, ta), pk);
    }
}

}  // namespace chunk
}  // namespace harts
