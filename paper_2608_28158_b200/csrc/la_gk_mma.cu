// Per-channel-decay recurrence (the Diag(gamma) term of Eq. 1, Section 2.2) for bf16 tensors with d_k = d_v = 128:
// the same packed chunkwise call (Eq. 16), plan tables, slots, chunk states and scratch layout as la_gk.cu, with
// every dense product of a chunk on the tensor cores (warp-level mma.sync.m16n8k16, bf16 operands, fp32
// accumulation).  Two ways to drive them.  The walks hold the running state S (forward) / its gradient dS (backward) in the
// accumulator registers of the CTA's sixteen warps over a whole sequence, which is what register accumulators are for.  The chunk
// kernels take every (chunk, head) on its own, with S and dS from memory (la_scan.cu); they share the walks' code for the inside
// of a chunk and hold no state, so nothing but that ties them to mma.sync: 15 us per item of the backward on one CTA per SM,
// where its 240 KB of traffic would take 5.6; the shared memory's port is busy for two thirds of it (operand tiles that ldmatrix reads
// four times over: 14.4 k wavefronts an item).  What cannot be a dense product stays on the CUDA cores in fp32: the
// decay-dependent pair sums
//     A_tj      = sum_i q_t[i] k_j[i] e^{b_t[i]-b_j[i]}                          (j <= t)
//     dq_t[i]  += sum_{j<=t} dA_tj k_j[i] e^{b_t[i]-b_j[i]},   dk_j[i] += sum_{t>=j} dA_tj q_t[i] e^{b_t[i]-b_j[i]}
// for t and j in the same 16-row block of the chunk; pairs in different blocks become dense products too, through
// operands anchored at the first row of t's block (see scores_*).  Every exponent is a difference of running sums that
// is <= 0 for log-decays g <= 0: no gate value can overflow.  The operands that carry a decay (q~ = q e^{b_t},
// k~ = k e^{b_n-b_j}, the anchored operands, the scores A, the states) are rounded to bf16 as in the scalar-gate
// tensor-core kernels.
//
// Shared-memory tiles of bf16 are row-major with the 16-byte pieces of a row XOR-ed by (row & 7), so that ldmatrix
// (plain and transposed) is free of bank conflicts.
#include "kernels.h"
#include "tc_common.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int32_t make_state_map(CUtensorMap* map, const void* base, int64_t n);
int32_t make_gate_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int sm_count();

namespace {

constexpr int BT = 64;      // chunk rows
constexpr int D = 128;      // d_k = d_v
constexpr int NT = 512;     // threads: 16 warps
constexpr int NW = NT / 32;
constexpr float LOG2E = 1.4426950408889634f;

// ---- shared-memory addressing ---------------------------------------------------------------------------------------
// [rows][128] bf16 and [rows][64] bf16 (128-byte rows); c16 = index of the 16-byte piece in the row
// (a tile of 128 columns is two panels of 64, as TMA leaves them)
template <int ROWS = BT>
__device__ __forceinline__ uint32_t sw256(int r, int c16) { return (uint32_t)((c16 >> 3) * (ROWS * 128) + r * 128 + (((c16 & 7) ^ (r & 7)) << 4)); }
__device__ __forceinline__ uint32_t sw128(int r, int c16) { return (uint32_t)(r * 128 + ((c16 ^ (r & 7)) << 4)); }
// The running log-decays [64][128] fp32: where (r, col) lies.  Groups of four floats are XOR-ed so that the 8 rows x 8 columns of a fragment
// and the 32-byte pieces of two rows are read without bank conflicts (laid out plainly: 3.9 k of 17.8 k wavefronts an item of the backward).
__device__ __forceinline__ int b_at(int r, int col) {
    return r * D + ((((col >> 2) ^ ((col >> 5) & 1) ^ ((r & 3) << 1)) << 2) | (col & 3));
}
__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// 2^x by the special-function unit; the running log-decays are kept in log2 units so that no multiply precedes it
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Fragment loaders.  `tile` is the shared-memory address of a swizzled tile, ROWS its rows if it has 128 columns, 0 if it has 64.
// A operand (16 x 16) of a matrix stored [m][k]: rows m0.., columns k0..
template <int ROWS>
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], uint32_t tile, int m0, int k0, int lane) {
    const int r = m0 + (lane & 7) + ((lane >> 3) & 1) * 8, c = (k0 >> 3) + (lane >> 4);
    ldsm4(a, tile + (ROWS ? sw256<ROWS>(r, c) : sw128(r, c)));
}
// A operand (16 x 16) of the TRANSPOSE of a matrix stored [k][m]: A[m][k] = stored[k][m]
template <int ROWS>
__device__ __forceinline__ void frag_a_t(uint32_t (&a)[4], uint32_t tile, int m0, int k0, int lane) {
    const int r = k0 + (lane & 7) + (lane >> 4) * 8, c = (m0 >> 3) + ((lane >> 3) & 1);
    ldsm4t(a, tile + (ROWS ? sw256<ROWS>(r, c) : sw128(r, c)));
}
// B operands of TWO adjacent n-tiles (n0.., n0+8..) for one k-step, matrix stored [k][n]: b[0],b[1] -> tile n0;
// b[2],b[3] -> tile n0+8
template <int ROWS>
__device__ __forceinline__ void frag_b_kn(uint32_t (&b)[4], uint32_t tile, int k0, int n0, int lane) {
    const int r = k0 + (lane & 7) + ((lane >> 3) & 1) * 8, c = (n0 >> 3) + (lane >> 4);
    ldsm4t(b, tile + (ROWS ? sw256<ROWS>(r, c) : sw128(r, c)));
}
// the same for a matrix stored [n][k] (B = stored^T)
template <int ROWS>
__device__ __forceinline__ void frag_b_nk(uint32_t (&b)[4], uint32_t tile, int k0, int n0, int lane) {
    const int r = n0 + (lane & 7) + (lane >> 4) * 8, c = (k0 >> 3) + ((lane >> 3) & 1);
    ldsm4(b, tile + (ROWS ? sw256<ROWS>(r, c) : sw128(r, c)));
}

struct SeqInfo {
    int own_begin, n_replay, n_virtual, n_chunks, replay_base, init_slot, req_lo, req_hi, chunk_base;
};
__device__ __forceinline__ SeqInfo seq_info(const harts_la_tables_t& tb, int seq) {
    SeqInfo s;
    s.own_begin = tb.seq_own_begin[seq];
    int own_len = tb.seq_own_begin[seq + 1] - s.own_begin;
    s.replay_base = tb.seq_replay_ptr[seq];
    s.n_replay = tb.seq_replay_ptr[seq + 1] - s.replay_base;
    s.n_virtual = s.n_replay + own_len;
    s.n_chunks = (s.n_virtual + BT - 1) / BT;
    s.init_slot = tb.seq_init_slot[seq];
    s.req_lo = tb.seq_req_ptr[seq];
    s.req_hi = tb.seq_req_ptr[seq + 1];
    s.chunk_base = tb.seq_chunk_ptr[seq];
    return s;
}

// code of row t of chunk c: physical row >= 0 (own), -2 - row (replayed), -1 (past the end)
__device__ __forceinline__ int row_code(const harts_la_tables_t& tb, const SeqInfo& s, int c, int t) {
    const int vr = c * BT + t;
    if (vr >= s.n_virtual) return -1;
    return vr < s.n_replay ? -2 - tb.replay_row[s.replay_base + vr] : s.own_begin + (vr - s.n_replay);
}
__device__ __forceinline__ void load_codes(const harts_la_tables_t& tb, const SeqInfo& s, int c, int* srow) {
    if (threadIdx.x < BT) srow[threadIdx.x] = row_code(tb, s, c, threadIdx.x);
}

// The loads of a chunk go to shared memory by cp.async, all of them in flight at once (through registers they were a round
// trip each: backward, 1,047 chunks x 16 heads, 2.59 -> 2.20 ms); cp_async_wait_all() before the barrier that publishes them.
using tc::cp_async16;

// One [BT][128] bf16 tile of a [rows, H, 128] tensor into a swizzled tile, 16 bytes at a time.  need_own: only rows
// with an output are taken (q, dO); otherwise every valid row (k, v).  Rows that are not taken become zero.
template <class Code>
__device__ __forceinline__ void load_tile_bf16(const __nv_bfloat16* src, int H, int h, const Code& code_of, bool need_own,
                                               unsigned char* dst) {
#pragma unroll
    for (int u = 0; u < BT * 16 / NT; u++) {
        const int p = threadIdx.x + u * NT, t = p >> 4, c16 = p & 15, code = code_of(t);
        const int r = code >= 0 ? code : code == -1 ? 0 : -2 - code;
        cp_async16(dst + sw256(t, c16), src + ((size_t)r * H + h) * D + c16 * 8, need_own ? code >= 0 : code != -1);
    }
}

// g of the chunk's valid rows (fp32 [rows, H, 128]) into sB [BT][128], zero elsewhere
template <class Code>
__device__ __forceinline__ void load_g(const float* gk, int H, int h, const Code& code_of, float* sB) {
#pragma unroll
    for (int u = 0; u < BT * 32 / NT; u++) {
        const int p = threadIdx.x + u * NT, t = p >> 5, c4 = p & 31, code = code_of(t);
        const int r = code >= 0 ? code : code == -1 ? 0 : -2 - code;
        cp_async16(reinterpret_cast<unsigned char*>(sB) + p * 16, gk + ((size_t)r * H + h) * D + c4 * 4, code != -1);
    }
}

// Asks the L2 for the rows of chunk c of a [rows, H, 128] tensor (the chunk after the one being worked on: its global
// loads then find their lines in the L2 instead of waiting for HBM).  Chunks >= 1 hold own rows only, which are
// consecutive: virtual row vr is physical row own_begin - n_replay + vr.
template <typename T>
__device__ __forceinline__ void prefetch_rows(const T* base, int H, int h, const SeqInfo& s, int c) {
    constexpr int LINES = D * (int)sizeof(T) / 128;              // 128-byte lines per row and head
    for (int p = threadIdx.x; p < BT * LINES; p += NT) {
        const int vr = c * BT + p / LINES;
        if (vr < s.n_virtual) {
            const char* addr = reinterpret_cast<const char*>(base + ((size_t)(s.own_begin - s.n_replay + vr) * H + h) * D) +
                               (p % LINES) * 128;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(addr));
        }
    }
}

// The same for the CTA's next (chunk, head) item of the chunk-parallel kernels, where that is a chunk of the same sequence.
struct NextItem {
    int c, h, gc;            // c < 0: none
};
__device__ __forceinline__ NextItem next_item(const SeqInfo& s, int c, int gc, int item, int H, int n_items) {
    const int nx = item + gridDim.x, d = nx / H - item / H;
    NextItem n{c + d, nx % H, gc + d};
    if (nx >= n_items || n.c >= s.n_chunks) n.c = -1;
    return n;
}

// The chunk kernels' loads.  All 64 rows of most chunks are the sequence's own, one after the other: their tiles come by TMA, asked for by
// one thread.  By cp.async they took the threads' time (160 KB at 16 bytes a lane: 5 k of the backward's 31 k cycles an item).  Chunks with
// replayed rows or an end still come that way.
struct ChunkMaps {
    CUtensorMap q, k, v, dO, g, s, ds;
};
__device__ __forceinline__ bool whole_chunk(const SeqInfo& s, int c) { return c * BT >= s.n_replay && (c + 1) * BT <= s.n_virtual; }
__device__ __forceinline__ void tma_rows(unsigned char* tile, const CUtensorMap* map, const SeqInfo& s, int c, int h, uint64_t* bar) {
    for (int p = 0; p < 2; p++) tc::tma_load_3d(tile + p * (BT * 128), map, p * 64, h, s.own_begin - s.n_replay + c * BT, bar);
}
__device__ __forceinline__ void tma_state(unsigned char* tile, const CUtensorMap* map, int gc, int h, int H, uint64_t* bar) {
    for (int p = 0; p < 2; p++) tc::tma_load_3d(tile + p * (D * 128), map, p * 64, 0, gc * H + h, bar);
}
// asks the L2 for what the CTA's next item loads, one thread
__device__ __forceinline__ void prefetch_chunk(const ChunkMaps& m, bool backward, const SeqInfo& s, const NextItem& nx, int H) {
    const int row0 = s.own_begin - s.n_replay + nx.c * BT;
    for (int p = 0; p < 2; p++) {
        tc::tma_prefetch_3d(&m.q, p * 64, nx.h, row0);
        tc::tma_prefetch_3d(&m.k, p * 64, nx.h, row0);
        tc::tma_prefetch_3d(&m.v, p * 64, nx.h, row0);
        if (backward) tc::tma_prefetch_3d(&m.dO, p * 64, nx.h, row0);
        tc::tma_prefetch_3d(&m.s, p * 64, 0, nx.gc * H + nx.h);
        if (backward) tc::tma_prefetch_3d(&m.ds, p * 64, 0, nx.gc * H + nx.h);
    }
    tc::tma_prefetch_3d(&m.g, 0, nx.h, row0);
}

// log-decays, laid out plainly -> their running sum over the rows in log2 units (b_at), per channel: four threads per channel (16 rows each, scanned in registers), joined through
// sTmp[4][128]
__device__ __forceinline__ void cumsum_rows(float* sB, float* sTmp) {
    const int tid = threadIdx.x, i = tid & (D - 1), part = tid >> 7;
    float x[16];
#pragma unroll
    for (int u = 0; u < 16; u++) x[u] = sB[(part * 16 + u) * D + i] * LOG2E;
#pragma unroll
    for (int u = 1; u < 16; u++) x[u] += x[u - 1];
    sTmp[part * D + i] = x[15];
    __syncthreads();
    float base = 0.f;
    for (int pp = 0; pp < part; pp++) base += sTmp[pp * D + i];
#pragma unroll
    for (int u = 0; u < 16; u++) sB[b_at(part * 16 + u, i)] = x[u] + base;
    __syncthreads();
}

// Sum over the 32 lanes of a warp for each of 16 per-lane values; lane l returns the total of z[l & 15].
__device__ __forceinline__ float warp_transpose_reduce16(float (&z)[16], int lane) {
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
        const bool upper = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < s; i++) {
            float send = upper ? z[i] : z[i + s];
            float keep = upper ? z[i + s] : z[i];
            z[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return z[0] + __shfl_xor_sync(0xffffffffu, z[0], 16);
}

// ---- the scores A_tj = sum_i q_t[i] k_j[i] e^{b_t[i]-b_j[i]} (j <= t), bf16 into sP ([BT][BT], swizzled) --------------
// The chunk is cut into four blocks of 16 rows.  With a_I = b at the first row of block I (log-decays are <= 0, so b
// only falls along the rows):
//   j in an EARLIER block than t (block I):  e^{b_t-b_j} = e^{b_t-a_I} e^{a_I-b_j}, both exponents <= 0, so the block of
//     scores is the dense product of q^_t = q_t e^{b_t-a_I} and k^(I)_j = k_j e^{a_I-b_j} (tensor cores);
//   j in the SAME block as t: the exponent difference is taken directly (CUDA cores, fp32), as no anchor inside the
//     block bounds both factors.
// anchored operands: sQa [64][128] (row t anchored at its own block), sKa: k^(1) rows 0..15, k^(2) rows 0..31, k^(3)
// rows 0..47 stored one after the other (row offsets 0, 16, 48)
__device__ __forceinline__ int ka_row0(int I) { return I == 1 ? 0 : (I == 2 ? 16 : 48); }

__device__ __forceinline__ void anchored_operands(const unsigned char* sQ, const unsigned char* sK, const float* sB,
                                                  unsigned char* sQa, unsigned char* sKa) {
    // 64 rows of q^ and 16 + 32 + 48 = 96 rows of k^(I): 160 rows x 16 pieces
    for (int p = threadIdx.x; p < 160 * 16; p += NT) {
        const int rr = p >> 4, c16 = p & 15;
        int src_row, anchor_row, dst_row;
        bool is_q;
        if (rr < 64) { is_q = true; src_row = rr; anchor_row = rr & ~15; dst_row = rr; }
        else {
            is_q = false;
            const int r2 = rr - 64, I = r2 < 16 ? 1 : (r2 < 48 ? 2 : 3);
            src_row = r2 - ka_row0(I); anchor_row = 16 * I; dst_row = r2;
        }
        uint4 x = *reinterpret_cast<const uint4*>((is_q ? sQ : sK) + sw256(src_row, c16));
        uint32_t* w = reinterpret_cast<uint32_t*>(&x);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int i = c16 * 8 + e * 2;
            const float2 bs = *reinterpret_cast<const float2*>(sB + b_at(src_row, i));
            const float2 ba = *reinterpret_cast<const float2*>(sB + b_at(anchor_row, i));
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
            // q^: e^{b_t - a_I};  k^(I): e^{a_I - b_j}
            const float e0 = is_q ? ex2(bs.x - ba.x) : ex2(ba.x - bs.x);
            const float e1 = is_q ? ex2(bs.y - ba.y) : ex2(ba.y - bs.y);
            w[e] = pack2(f.x * e0, f.y * e1);
        }
        // the local row index of a k^(I) sub-tile is dst_row - its row offset; the offsets are multiples of 8, so the
        // swizzle of the stacked tile equals that of the sub-tile
        *reinterpret_cast<uint4*>(is_q ? sQa + sw256(dst_row, c16) : sKa + sw256<96>(dst_row, c16)) = x;
    }
}

// Pairs INSIDE a 16-row block: with the same anchor a_I (b at the block's first row) the key factor e^{a_I-b_j} is >= 1
// and grows to e^{a_I - b_{16I+15}} at the block's last row.  While that total decay of a block stays below 2^MILD_LOG2
// in every channel (bf16 and fp32 hold 2^127), the block on the diagonal is a dense product too: q^ (anchored at its
// block, as above) against k_j e^{a_I-b_j} for the keys of the same block, masked to j <= t afterwards -- the entries
// right of the diagonal are finite and thrown away.  A chunk in which any block decays faster takes the exact CUDA-core
// path for its diagonal blocks instead (one decision per chunk, the same for the whole CTA).
constexpr float MILD_LOG2 = 100.f;

__device__ __forceinline__ bool chunk_is_mild(const float* sB) {
    const int i = threadIdx.x & (D - 1), blk = threadIdx.x >> 7;       // 512 threads: 4 blocks x 128 channels
    const float fall = sB[b_at(16 * blk, i)] - sB[b_at(16 * blk + 15, i)];
    return __syncthreads_or(!(fall <= MILD_LOG2)) == 0;                  // also false for a NaN gate
}

// All operands of a mild chunk in one pass, a thread's 16-byte pieces of q and k: the anchored tiles, the keys anchored at
// their OWN block sKd[j] = k_j .* 2^{a_I(j) - b_j}, and where asked for q~ = q .* 2^{b_t}, k~ = k .* 2^{b_n - b_t}.  sKd
// and q~ may go over sK and sQ.
__device__ __forceinline__ void mild_operands(const unsigned char* sQ, const unsigned char* sK, const float* sB, unsigned char* sQa,
                                              unsigned char* sKa, unsigned char* sKd, unsigned char* sQt, unsigned char* sKt) {
#pragma unroll
    for (int u = 0; u < BT * 16 / NT; u++) {
        const int p = threadIdx.x + u * NT, t = p >> 4, c16 = p & 15, blk = t >> 4;
        const uint32_t off = sw256(t, c16);
        float bs[8], ba[8];
        auto row8 = [&](float (&x)[8], int r) {
            *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(sB + b_at(r, c16 * 8));
            *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(sB + b_at(r, c16 * 8 + 4));
        };
        auto scaled = [&](const uint4& x, auto exponent) {
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
            uint32_t y[4];
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
                y[e] = pack2(f.x * ex2(exponent(2 * e)), f.y * ex2(exponent(2 * e + 1)));
            }
            return make_uint4(y[0], y[1], y[2], y[3]);
        };
        row8(bs, t);
        row8(ba, 16 * blk);
        const uint4 qv = *reinterpret_cast<const uint4*>(sQ + off), kv = *reinterpret_cast<const uint4*>(sK + off);
        *reinterpret_cast<uint4*>(sQa + off) = scaled(qv, [&](int e) { return bs[e] - ba[e]; });
        if (sQt) *reinterpret_cast<uint4*>(sQt + off) = scaled(qv, [&](int e) { return bs[e]; });
        *reinterpret_cast<uint4*>(sKd + off) = scaled(kv, [&](int e) { return ba[e] - bs[e]; });
        for (int I = blk + 1; I < 4; I++) {
            row8(ba, 16 * I);
            // the row offsets of the k^(I) sub-tiles are multiples of 8, so the swizzle of the stacked tile equals theirs
            *reinterpret_cast<uint4*>(sKa + sw256<96>(ka_row0(I) + t, c16)) = scaled(kv, [&](int e) { return ba[e] - bs[e]; });
        }
        if (sKt) {
            row8(ba, BT - 1);
            *reinterpret_cast<uint4*>(sKt + off) = scaled(kv, [&](int e) { return ba[e] - bs[e]; });
        }
    }
}

// blocks left of the diagonal: warp -> row block I = warp & 3, 16-column tile J = warp >> 2; with `diag` (a mild chunk)
// the warps with J == I take the block on the diagonal from the keys anchored at their own block
__device__ __forceinline__ void scores_off_diagonal(uint32_t aQa, uint32_t aKa, unsigned char* sP, int warp, int lane,
                                                    bool diag = false, uint32_t aKd = 0) {
    const int I = warp & 3, g = lane >> 2, tq = lane & 3;
    if (diag && (warp >> 2) == I) {
        float acc[2][4];
#pragma unroll
        for (int x = 0; x < 2; x++) acc[x][0] = acc[x][1] = acc[x][2] = acc[x][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 8; ks++) {
            uint32_t a[4], b[4];
            frag_a<BT>(a, aQa, 16 * I, ks * 16, lane);
            frag_b_nk<BT>(b, aKd, ks * 16, 16 * I, lane);
            mma16816(acc[0], a, b[0], b[1]);
            mma16816(acc[1], a, b[2], b[3]);
        }
#pragma unroll
        for (int x = 0; x < 2; x++) {
            const int jc = 8 * x + 2 * tq, col = 16 * I + jc;           // jc, g: column and row inside the block
            const float v0 = jc <= g ? acc[x][0] : 0.f, v1 = jc + 1 <= g ? acc[x][1] : 0.f;
            const float v2 = jc <= g + 8 ? acc[x][2] : 0.f, v3 = jc + 1 <= g + 8 ? acc[x][3] : 0.f;
            *reinterpret_cast<uint32_t*>(sP + sw128(16 * I + g, col >> 3) + (col & 7) * 2) = pack2(v0, v1);
            *reinterpret_cast<uint32_t*>(sP + sw128(16 * I + g + 8, col >> 3) + (col & 7) * 2) = pack2(v2, v3);
        }
        return;
    }
    for (int J = warp >> 2; J < I; J += NW / 4) {
        float acc[2][4];
#pragma unroll
        for (int x = 0; x < 2; x++) acc[x][0] = acc[x][1] = acc[x][2] = acc[x][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < 8; ks++) {
            uint32_t a[4], b[4];
            frag_a<BT>(a, aQa, 16 * I, ks * 16, lane);
            frag_b_nk<96>(b, aKa, ks * 16, ka_row0(I) + 16 * J, lane);
            mma16816(acc[0], a, b[0], b[1]);
            mma16816(acc[1], a, b[2], b[3]);
        }
#pragma unroll
        for (int x = 0; x < 2; x++) {
            const int col = 16 * J + 8 * x + 2 * tq;
            *reinterpret_cast<uint32_t*>(sP + sw128(16 * I + g, col >> 3) + (col & 7) * 2) = pack2(acc[x][0], acc[x][1]);
            *reinterpret_cast<uint32_t*>(sP + sw128(16 * I + g + 8, col >> 3) + (col & 7) * 2) = pack2(acc[x][2], acc[x][3]);
        }
    }
}

// one-step decay factors 2^{b_t - b_{t-1}} of the rows 1..63 of a chunk (fp32 [BT][128]; row 0 is not used: the factors
// serve pairs inside a 16-row block only)
__device__ __forceinline__ void step_factors(const float* sB, float* sR) {
    for (int p = threadIdx.x; p < BT * 32; p += NT) {
        const int t = p >> 5, c4 = p & 31;
        if (t == 0) continue;
        const float4 hi = *reinterpret_cast<const float4*>(sB + b_at(t, c4 * 4));
        const float4 lo = *reinterpret_cast<const float4*>(sB + b_at(t - 1, c4 * 4));
        *reinterpret_cast<float4*>(sR + t * D + c4 * 4) = make_float4(ex2(hi.x - lo.x), ex2(hi.y - lo.y), ex2(hi.z - lo.z), ex2(hi.w - lo.w));
    }
}

// diagonal blocks: one warp per row t, every lane takes 4 channels of all (at most 16) pairs of the row, walking j from t
// down with the decay as a running product of the one-step factors (x_{t,j-1} = x_{t,j} r_j: every factor <= 1, no
// exponential per pair); the warp sums the lanes with a transposed reduction, lanes 0..15 then hold A[t][16 I + lane]
// (zero right of the diagonal)
__device__ __forceinline__ void scores_diagonal(const unsigned char* sQ, const unsigned char* sK, const float* sR,
                                                unsigned char* sP, int warp, int lane) {
    for (int t = warp; t < BT; t += NW) {
        const int j_lo = t & ~15;
        const uint2 qraw = *reinterpret_cast<const uint2*>(sQ + sw256(t, lane >> 1) + (lane & 1) * 8);
        const float2 q01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&qraw.x));
        const float2 q23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&qraw.y));
        float4 qx = make_float4(q01.x, q01.y, q23.x, q23.y);          // q_t .* x_{t,j}, j walking down from t
        float z[16];
#pragma unroll
        for (int u = 15; u >= 0; u--) {
            const int j = j_lo + u;
            float acc = 0.f;
            if (j <= t) {
                const uint2 kraw = *reinterpret_cast<const uint2*>(sK + sw256(j, lane >> 1) + (lane & 1) * 8);
                const float2 k01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kraw.x));
                const float2 k23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kraw.y));
                acc = qx.x * k01.x + qx.y * k01.y + qx.z * k23.x + qx.w * k23.y;
                if (u > 0) {
                    const float4 r = *reinterpret_cast<const float4*>(sR + j * D + lane * 4);
                    qx.x *= r.x; qx.y *= r.y; qx.z *= r.z; qx.w *= r.w;
                }
            }
            z[u] = acc;
        }
        const float total = warp_transpose_reduce16(z, lane);
        const float other = __shfl_down_sync(0xffffffffu, total, 1);
        if (lane < 16 && !(lane & 1)) {
            const int col = j_lo + lane;
            *reinterpret_cast<uint32_t*>(sP + sw128(t, col >> 3) + (col & 7) * 2) = pack2(total, other);
        }
    }
}

// q <- q .* e^{b_t} and k <- k .* e^{b_n - b_t} written to (possibly other) swizzled tiles
template <bool Q = true, bool K = true>
__device__ __forceinline__ void scale_qk(const unsigned char* sQ, const unsigned char* sK, const float* sB,
                                         unsigned char* dQ, unsigned char* dK) {
#pragma unroll
    for (int u = 0; u < BT * 16 / NT; u++) {
        const int p = threadIdx.x + u * NT, t = p >> 4, c16 = p & 15;
        const uint32_t off = sw256(t, c16);
        uint4 qv = *reinterpret_cast<const uint4*>((Q ? sQ : sK) + off), kv = *reinterpret_cast<const uint4*>((K ? sK : sQ) + off);
        uint32_t* qw = reinterpret_cast<uint32_t*>(&qv);
        uint32_t* kw = reinterpret_cast<uint32_t*>(&kv);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int i = c16 * 8 + e * 2;
            const float2 bt = *reinterpret_cast<const float2*>(sB + b_at(t, i));
            const float2 bn = *reinterpret_cast<const float2*>(sB + b_at(BT - 1, i));
            const float2 qf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&qw[e]));
            const float2 kf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&kw[e]));
            if (Q) qw[e] = pack2(qf.x * ex2(bt.x), qf.y * ex2(bt.y));
            if (K) kw[e] = pack2(kf.x * ex2(bn.x - bt.x), kf.y * ex2(bn.y - bt.y));
        }
        if (Q) *reinterpret_cast<uint4*>(dQ + off) = qv;
        if (K) *reinterpret_cast<uint4*>(dK + off) = kv;
    }
}

// The state fragments of a warp: rows 16 * (warp & 7) + g and + g + 8 (g = lane / 4), columns
// 64 * (warp >> 3) + 8 * n + 2 * (lane % 4) + {0, 1} of n-tile n: st[n][0..1] = row g, st[n][2..3] = row g + 8.
struct Shared {
    static constexpr int q = 0, k = 16384, v = 32768;          // bf16 [64][128]
    static constexpr int p = 49152;                             // bf16 [64][64]
    static constexpr int sb = 57344;                            // bf16 [128][128]: the state as an MMA operand
    static constexpr int b = 90112;                             // fp32 [64][128]: running log-decay (log2 units)
    static constexpr int qa = 122880;                           // bf16 [64][128]: q anchored at its 16-row block
    static constexpr int ka = qa + 16384;                       // bf16 [96][128]: k anchored at blocks 1, 2, 3
    static constexpr int r = ka + 96 * 256;                     // fp32 [64][128]: one-step decay factors
    static constexpr int tmp = r + 32768;                       // fp32 [4][128]
    static constexpr int row = tmp + 2048;                      // int  [64]
    static constexpr int fwd_bytes = row + 256;
};

// state fragments -> bf16 operand tile (swizzled [128][128])
__device__ __forceinline__ void state_to_operand(const float (&st)[8][4], unsigned char* sSb, int warp, int lane) {
    const int g = lane >> 2, tq = lane & 3, r0 = (warp & 7) * 16 + g, c0 = (warp >> 3) * 8;
#pragma unroll
    for (int n = 0; n < 8; n++) {
        *reinterpret_cast<uint32_t*>(sSb + sw256<D>(r0, c0 + n) + tq * 4) = pack2(st[n][0], st[n][1]);
        *reinterpret_cast<uint32_t*>(sSb + sw256<D>(r0 + 8, c0 + n) + tq * 4) = pack2(st[n][2], st[n][3]);
    }
}
// state fragments <-> fp32 [128][128] in global memory (slots, initial-state gradients)
// PAST_L1: the data was written during this launch by another CTA
template <bool ADD, bool PAST_L1>
__device__ __forceinline__ void state_from_global(float (&st)[8][4], const float* src, int warp, int lane) {
    const int g = lane >> 2, tq = lane & 3, r0 = (warp & 7) * 16 + g, c0 = (warp >> 3) * 64 + tq * 2;
#pragma unroll
    for (int n = 0; n < 8; n++) {
        const float2* p_lo = reinterpret_cast<const float2*>(src + (size_t)r0 * D + c0 + n * 8);
        const float2* p_hi = reinterpret_cast<const float2*>(src + (size_t)(r0 + 8) * D + c0 + n * 8);
        const float2 lo = PAST_L1 ? __ldcg(p_lo) : *p_lo;
        const float2 hi = PAST_L1 ? __ldcg(p_hi) : *p_hi;
        if (ADD) { st[n][0] += lo.x; st[n][1] += lo.y; st[n][2] += hi.x; st[n][3] += hi.y; }
        else { st[n][0] = lo.x; st[n][1] = lo.y; st[n][2] = hi.x; st[n][3] = hi.y; }
    }
}
__device__ __forceinline__ void state_to_global(const float (&st)[8][4], float* dst, int warp, int lane) {
    const int g = lane >> 2, tq = lane & 3, r0 = (warp & 7) * 16 + g, c0 = (warp >> 3) * 64 + tq * 2;
#pragma unroll
    for (int n = 0; n < 8; n++) {
        *reinterpret_cast<float2*>(dst + (size_t)r0 * D + c0 + n * 8) = make_float2(st[n][0], st[n][1]);
        *reinterpret_cast<float2*>(dst + (size_t)(r0 + 8) * D + c0 + n * 8) = make_float2(st[n][2], st[n][3]);
    }
}
// st <- Diag(2^{b_n}) st + X^T Y over the chunk's 64 rows: X stored [row][128] (its transpose is the A operand), Y
// stored [row][128]
__device__ __forceinline__ void state_update(float (&st)[8][4], const float* sB, uint32_t aX, uint32_t aY, int warp, int lane) {
    const int g = lane >> 2, r0 = (warp & 7) * 16, c0 = (warp >> 3) * 64;
    const float g_lo = ex2(sB[b_at(BT - 1, r0 + g)]), g_hi = ex2(sB[b_at(BT - 1, r0 + g + 8)]);
#pragma unroll
    for (int n = 0; n < 8; n++) {
        st[n][0] *= g_lo; st[n][1] *= g_lo; st[n][2] *= g_hi; st[n][3] *= g_hi;
    }
#pragma unroll
    for (int ks = 0; ks < 4; ks++) {
        uint32_t a[4];
        frag_a_t<BT>(a, aX, r0, ks * 16, lane);
#pragma unroll
        for (int n2 = 0; n2 < 4; n2++) {
            uint32_t b[4];
            frag_b_kn<BT>(b, aY, ks * 16, c0 + n2 * 16, lane);
            mma16816(st[2 * n2], a, b[0], b[1]);
            mma16816(st[2 * n2 + 1], a, b[2], b[3]);
        }
    }
}
// swizzled bf16 [rows][128] tile -> plain row-major global memory ([rows][128] contiguous), 16 bytes per thread and step
template <int ROWS>
__device__ __forceinline__ void tile_to_global(const unsigned char* tile, __nv_bfloat16* dst) {
    for (int p = threadIdx.x; p < ROWS * 16; p += NT)
        reinterpret_cast<uint4*>(dst)[p] = *reinterpret_cast<const uint4*>(tile + sw256<ROWS>(p >> 4, p & 15));
}

// plain row-major [128][128] bf16 in global memory -> swizzled tile
__device__ __forceinline__ void global_to_tile128(const __nv_bfloat16* src, unsigned char* tile) {
#pragma unroll
    for (int u = 0; u < D * 16 / NT; u++) {
        const int p = threadIdx.x + u * NT;
        cp_async16(tile + sw256<D>(p >> 4, p & 15), src + p * 8, true);
    }
}

// A warp's 16 x 32 block (rows 16 * mb, columns 32 * nq) of a [64][128] product: bf16 rows to global memory, 16 bytes a lane, by way of
// the block's own place in a tile nobody reads any more.  Straight from the fragments a store is 4 bytes of eight rows: with dq,
// dk, dv so, the rows' outputs were 0.2 of the backward's time.  Rows without an output (code < 0) are left out.
__device__ __forceinline__ void block_to_rows(const float (&acc)[4][4], unsigned char* tile, int mb, int nq, const int* srow,
                                              __nv_bfloat16* __restrict__ out, int H, int h, int lane) {
#pragma unroll
    for (int n2 = 0; n2 < 2; n2++) {
        const int row = 16 * mb + ((lane >> 3) & 1) * 8 + (lane & 7), c16 = 4 * nq + 2 * n2 + (lane >> 4);
        asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(s_u32(tile + sw256(row, c16))),
                     "r"(pack2(acc[2 * n2][0], acc[2 * n2][1])), "r"(pack2(acc[2 * n2][2], acc[2 * n2][3])),
                     "r"(pack2(acc[2 * n2 + 1][0], acc[2 * n2 + 1][1])), "r"(pack2(acc[2 * n2 + 1][2], acc[2 * n2 + 1][3])) : "memory");
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 2; u++) {
        const int row = 16 * mb + 8 * u + (lane >> 2), c16 = 4 * nq + (lane & 3), code = srow[row];
        const uint4 y = *reinterpret_cast<const uint4*>(tile + sw256(row, c16));
        if (code >= 0) *reinterpret_cast<uint4*>(out + ((size_t)code * H + h) * D + c16 * 8) = y;
    }
    __syncwarp();
}

// the sequence of [seq_lo, seq_hi) that owns chunk gc (every warp searches, 32 ways at a time)
__device__ __forceinline__ int owner_of(const harts_la_tables_t& tb, int seq_lo, int seq_hi, int gc) {
    const int lane = threadIdx.x & 31;
    int lo = seq_lo, hi = seq_hi;
    while (hi - lo > 1) {
        const int step = (hi - lo + 31) / 32, i = lo + lane * step;
        const unsigned m = __ballot_sync(~0u, i < hi && tb.seq_chunk_ptr[i] <= gc);
        lo += (__popc(m) - 1) * step;
        hi = min(hi, lo + step);
    }
    return lo;
}

// How a kernel is driven.
// ROUND: one launch per round, item = (sequence, head) = block index, no flags.
// CHUNKS (backward only): the boundary states, their gradients and <S, dS> are in memory (la_scan.cu), item = (chunk, head).
// ONE_LAUNCH: the grid covers the sequences of ALL rounds (numbered round by round).  Every CTA draws its work item
// from `ticket`, so an item is only ever held by a running CTA; a sequence that starts from an exported state waits for
// the flag its producer (an earlier round, a smaller ticket, hence running or done) sets after writing the slot.
enum Mode { ROUND, ONE_LAUNCH_MODE, CHUNKS_MODE };
template <int MODE>
__global__ void __launch_bounds__(NT, 1)
gk_mma_fwd_kernel(harts_la_tables_t tb, int seq_lo, int H, const __nv_bfloat16* __restrict__ q,
                  const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, const float* __restrict__ gk,
                  __nv_bfloat16* __restrict__ o, float* __restrict__ slots, __nv_bfloat16* __restrict__ chunk_states,
                  const int32_t* gate, int* status, int* slot_flags, int* ticket) {
    if (gate_closed(gate)) return;
    constexpr bool ONE_LAUNCH = MODE == ONE_LAUNCH_MODE;
    __shared__ int s_item, s_dead;
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *sQ = sm + Shared::q, *sK = sm + Shared::k, *sV = sm + Shared::v, *sP = sm + Shared::p,
                  *sSb = sm + Shared::sb, *sQa = sm + Shared::qa, *sKa = sm + Shared::ka;
    float* sB = reinterpret_cast<float*>(sm + Shared::b);
    float* sR = reinterpret_cast<float*>(sm + Shared::r);
    float* sTmp = reinterpret_cast<float*>(sm + Shared::tmp);
    int* srow = reinterpret_cast<int*>(sm + Shared::row);
    const uint32_t aQ = s_u32(sQ), aK = s_u32(sK), aV = s_u32(sV), aP = s_u32(sP), aSb = s_u32(sSb);

    // blocks are handed to the SMs in index order: with the plan's order (longest sequence of the round first) the long
    // walks start first and the short ones fill the tail
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    int item = blockIdx.x;
    if constexpr (ONE_LAUNCH) {
        if (tid == 0) {
            s_item = atomicAdd(ticket, 1);
            s_dead = 0;
        }
        __syncthreads();
        item = s_item;
    }
    const int mb = warp & 3, nq = warp >> 2;          // this warp's 16-row block and 32-column quarter of [64][128] products
    const size_t state_elems = (size_t)D * D;
    const int seq_pos = seq_lo + item / H, h = item % H;
    const int seq = tb.seq_order ? tb.seq_order[seq_pos] : seq_pos;
    const SeqInfo s = seq_info(tb, seq);

    float st[8][4];
    if (s.init_slot < 0) {
#pragma unroll
        for (int n = 0; n < 8; n++) st[n][0] = st[n][1] = st[n][2] = st[n][3] = 0.f;
    } else {
        if constexpr (ONE_LAUNCH) {
            if (tid == 0) tc::flag_wait(slot_flags + (size_t)s.init_slot * H + h, status, &s_dead);
            if (__syncthreads_or(s_dead)) return;      // the wait ran out (status word set): give the walk up
        }
        state_from_global<false, ONE_LAUNCH>(st, slots + ((size_t)s.init_slot * H + h) * state_elems, warp, lane);
    }

    int next_req = s.req_lo;
    for (int c = 0; c < s.n_chunks; c++) {
        __syncthreads();                                   // the previous chunk's readers of every tile are through
        load_codes(tb, s, c, srow);
        __syncthreads();
        auto code_of = [&](int t) { return srow[t]; };
        load_tile_bf16(k, H, h, code_of, false, sK);
        load_tile_bf16(q, H, h, code_of, true, sQ);
        load_tile_bf16(v, H, h, code_of, false, sV);
        load_g(gk, H, h, code_of, sB);
        if (c + 1 < s.n_chunks) {
            prefetch_rows(k, H, h, s, c + 1);
            prefetch_rows(q, H, h, s, c + 1);
            prefetch_rows(v, H, h, s, c + 1);
            prefetch_rows(gk, H, h, s, c + 1);
        }
        // start-of-chunk state: operand copy, kept for the backward, exported when the plan requests this boundary
        state_to_operand(st, sSb, warp, lane);
        const bool exported = next_req < s.req_hi && tb.slot_chunk[next_req] == c;
        if (exported) {
            state_to_global(st, slots + ((size_t)next_req * H + h) * state_elems, warp, lane);
            if (ONE_LAUNCH) __threadfence();               // this thread's part of the slot, before the flag below
            next_req++;
        }
        tc::cp_async_wait_all();
        __syncthreads();
        if (ONE_LAUNCH && exported && tid == 0) tc::flag_set(slot_flags + (size_t)(next_req - 1) * H + h);
        if (chunk_states) tile_to_global<D>(sSb, chunk_states + ((size_t)(s.chunk_base + c) * H + h) * state_elems);
        cumsum_rows(sB, sTmp);
        const bool mild = chunk_is_mild(sB);
        unsigned char* sKd = reinterpret_cast<unsigned char*>(sR);        // the two are never needed in the same chunk
        unsigned char* sKt = sKd + 16384;                                 // k~ of a mild chunk; its q~ goes over q
        if (mild) {
            mild_operands(sQ, sK, sB, sQa, sKa, sKd, sQ, sKt);
        } else {
            step_factors(sB, sR);
            anchored_operands(sQ, sK, sB, sQa, sKa);
        }
        __syncthreads();
        if (!mild) scores_diagonal(sQ, sK, sR, sP, warp, lane);
        scores_off_diagonal(s_u32(sQa), s_u32(sKa), sP, warp, lane, mild, s_u32(sKd));
        __syncthreads();
        if (!mild) {
            scale_qk(sQ, sK, sB, sQ, sK);
            __syncthreads();
        }
        // ---- o = P V + q~ S_c : warp -> rows 16 * mb, columns 32 * nq ----------------------------------------------
        {
            const int m0 = mb * 16, n_base = nq * 32;
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
            for (int ks = 0; ks <= mb; ks++) {              // P is zero right of the diagonal block
                uint32_t a[4];
                frag_a<0>(a, aP, m0, ks * 16, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    uint32_t b[4];
                    frag_b_kn<BT>(b, aV, ks * 16, n_base + n2 * 16, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
#pragma unroll
            for (int ks = 0; ks < 8; ks++) {
                uint32_t a[4];
                frag_a<BT>(a, aQ, m0, ks * 16, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    uint32_t b[4];
                    frag_b_kn<D>(b, aSb, ks * 16, n_base + n2 * 16, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
            const int row_lo = srow[m0 + g], row_hi = srow[m0 + g + 8];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = n_base + n * 8 + tq * 2;
                if (row_lo >= 0) *reinterpret_cast<uint32_t*>(o + ((size_t)row_lo * H + h) * D + col) = pack2(acc[n][0], acc[n][1]);
                if (row_hi >= 0) *reinterpret_cast<uint32_t*>(o + ((size_t)row_hi * H + h) * D + col) = pack2(acc[n][2], acc[n][3]);
            }
        }
        // ---- S <- Diag(e^{b_n}) S + k~^T V ---------------------------------------------------------------------------
        state_update(st, sB, mild ? s_u32(sKt) : aK, aV, warp, lane);
    }
}


// ---- forward, every (chunk, head) on its own -----------------------------------------------------------------------------
// The boundary states are in memory (la_scan.cu).  What bounds an item is its chain of phases (load, running sums, operands,
// scores, outputs), each far below the machine's rates, so two CTAs share an SM: 115 KB of shared memory and 64 registers a
// thread.  To fit, everything is worked on in place or over something dead: the running sums' scratch lies under the
// scores, k becomes the keys anchored at their own block, q becomes q~, V comes in over the anchored queries once the
// scores are done, the state over the running sums.  One pass over q and k makes all four operands of a mild chunk.
// Measured, 1,047 chunks x 16 heads, cold: 0.57 ms (0.78 with loads by cp.async and running sums laid out plainly; one CTA per SM with every
// tile in a place of its own 1.08).
struct SharedC {
    static constexpr int q = 0, k = 16384;                              // bf16 [64][128]; then q~, keys anchored at their block
    static constexpr int b = 32768;                                     // fp32 [64][128] running log-decay; then the state
    static constexpr int qa = 65536, ka = qa + 16384;                   // anchored operands; then V; step factors (not mild)
    static constexpr int p = ka + 96 * 256, row = p + 8192, misc = row + 256, bytes = misc + 64;
};
static_assert(2 * (SharedC::bytes + 1024 + 64) <= 228 * 1024, "two CTAs per SM");

__global__ void __launch_bounds__(NT, 2)
gk_chunk_fwd_kernel(harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const __nv_bfloat16* __restrict__ q,
                    const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, const float* __restrict__ gk,
                    __nv_bfloat16* __restrict__ o, const __grid_constant__ ChunkMaps maps, int* status, const int32_t* gate) {
    after_previous();
    extern __shared__ __align__(1024) unsigned char sm[];       // no static shared memory: the dynamic window starts 1024-byte aligned
    struct Misc {
        uint64_t bar_g, bar_qk, bar_s;
        int dead, closed;
    };
    Misc& m = *reinterpret_cast<Misc*>(sm + SharedC::misc);
    if (threadIdx.x == 0) {
        tc::mbar_init(&m.bar_g, 1);
        tc::mbar_init(&m.bar_qk, 1);
        tc::mbar_init(&m.bar_s, 1);
        m.dead = 0;
        m.closed = gate && *gate != 0;
        if (s_u32(sm) & 1023) {                   // never on sm_100a; the swizzled tiles would be misread
            m.closed = 1;
            if (status) atomicExch(status, tc::STATUS_TIMEOUT);
        }
        tc::fence_barrier_init();
    }
    __syncthreads();
    if (m.closed) return;
    uint32_t ph_rows = 0, ph_s = 0;
    bool ok = true;
    unsigned char *sQ = sm + SharedC::q, *sK = sm + SharedC::k, *sQa = sm + SharedC::qa, *sKa = sm + SharedC::ka,
                  *sP = sm + SharedC::p, *sV = sQa, *sS = sm + SharedC::b;
    float *sB = reinterpret_cast<float*>(sm + SharedC::b), *sTmp = reinterpret_cast<float*>(sP), *sR = reinterpret_cast<float*>(sQa);
    int* srow = reinterpret_cast<int*>(sm + SharedC::row);
    const uint32_t aQ = s_u32(sQ), aK = s_u32(sK), aP = s_u32(sP), aV = s_u32(sV), aS = s_u32(sB);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mb = warp & 3, nq = warp >> 2;          // this warp's 16-row block and 32-column quarter of [64][128] products
    const int chunk_lo = tb.seq_chunk_ptr[seq_lo], n_items = (tb.seq_chunk_ptr[seq_hi] - chunk_lo) * H;
    SeqInfo s;
    s.chunk_base = s.n_chunks = 0;
    int seq = seq_lo;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int h = item % H, gc = chunk_lo + item / H;
        if (gc >= s.chunk_base + s.n_chunks) {             // chunks come in order: often still the last one's sequence
            seq = owner_of(tb, seq, seq_hi, gc);
            s = seq_info(tb, seq);
        }
        const int c = gc - s.chunk_base;
        const bool has_s = c > 0 || s.init_slot >= 0;     // the state of a sequence that starts from zero is not read
        const bool whole = whole_chunk(s, c);
        tc::fence_async_smem();                            // what was written into the tiles, before TMA writes there
        __syncthreads();                                   // the previous item's readers of every tile are through
        load_codes(tb, s, c, srow);
        if (whole) {
            if (tid == 0) {
                tc::mbar_expect_tx(&m.bar_g, BT * D * 4);
                tc::tma_load_3d(sB, &maps.g, 0, h, s.own_begin - s.n_replay + c * BT, &m.bar_g);
                tc::mbar_expect_tx(&m.bar_qk, 2 * BT * D * 2);
                tma_rows(sQ, &maps.q, s, c, h, &m.bar_qk);
                tma_rows(sK, &maps.k, s, c, h, &m.bar_qk);
            }
        } else {
            auto code_of = [&](int t) { return row_code(tb, s, c, t); };
            load_g(gk, H, h, code_of, sB);
            tc::cp_async_commit();
            load_tile_bf16(q, H, h, code_of, true, sQ);
            load_tile_bf16(k, H, h, code_of, false, sK);
            tc::cp_async_commit();
        }
        const NextItem nx = next_item(s, c, gc, item, H, n_items);
        if (nx.c >= 0 && tid == 32) prefetch_chunk(maps, false, s, nx, H);
        if (whole) ok = tc::mbar_wait_warp(&m.bar_g, ph_rows, status, &m.dead) && ok;
        else tc::cp_async_wait_group<1>();
        __syncthreads();
        cumsum_rows(sB, sTmp);                             // while the rows come
        if (whole) {
            ok = tc::mbar_wait_warp(&m.bar_qk, ph_rows, status, &m.dead) && ok;
            ph_rows ^= 1;
        } else {
            tc::cp_async_wait_all();
        }
        const bool mild = chunk_is_mild(sB);               // (a barrier: every thread's rows are there)
        if (mild) mild_operands(sQ, sK, sB, sQa, sKa, sK, sQ, nullptr);
        else anchored_operands(sQ, sK, sB, sQa, sKa);
        tc::fence_async_smem();
        __syncthreads();
        auto load_state = [&] {                            // over the running sums
            if (has_s && tid == 0) {
                tc::mbar_expect_tx(&m.bar_s, D * D * 2);
                tma_state(sS, &maps.s, gc, h, H, &m.bar_s);
            }
        };
        if (mild) load_state();
        uint4 vv[BT * 16 / NT];                            // V, on its way while the scores are computed
#pragma unroll
        for (int u = 0; u < BT * 16 / NT; u++) {
            const int p = tid + u * NT, code = srow[p >> 4], r = code >= 0 ? code : -2 - code;
            vv[u] = code != -1 ? *reinterpret_cast<const uint4*>(v + ((size_t)r * H + h) * D + (p & 15) * 8) : make_uint4(0, 0, 0, 0);
        }
        scores_off_diagonal(s_u32(sQa), s_u32(sKa), sP, warp, lane, mild, aK);
        __syncthreads();                                   // the anchored operands are dead
        if (!mild) {
            step_factors(sB, sR);
            __syncthreads();
            scores_diagonal(sQ, sK, sR, sP, warp, lane);
            __syncthreads();
            scale_qk<true, false>(sQ, sK, sB, sQ, sK);
            tc::fence_async_smem();
            __syncthreads();
            load_state();
        }
#pragma unroll
        for (int u = 0; u < BT * 16 / NT; u++) {
            const int p = tid + u * NT;
            *reinterpret_cast<uint4*>(sV + sw256(p >> 4, p & 15)) = vv[u];
        }
        if (has_s) {
            ok = tc::mbar_wait_warp(&m.bar_s, ph_s, status, &m.dead) && ok;
            ph_s ^= 1;
        }
        if (__syncthreads_or(!ok)) {                       // a wait ran out (status word set): let what is in flight land
            tc::drain_delay();
            return;
        }
        // ---- o = P V + q~ S_c : warp -> rows 16 * mb, columns 32 * nq ----------------------------------------------
        const int m0 = mb * 16, n_base = nq * 32;
        float acc[4][4];
#pragma unroll
        for (int n = 0; n < 4; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
        for (int ks = 0; ks <= mb; ks++) {              // P is zero right of the diagonal block
            uint32_t a[4];
            frag_a<0>(a, aP, m0, ks * 16, lane);
#pragma unroll
            for (int n2 = 0; n2 < 2; n2++) {
                uint32_t b[4];
                frag_b_kn<BT>(b, aV, ks * 16, n_base + n2 * 16, lane);
                mma16816(acc[2 * n2], a, b[0], b[1]);
                mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
            }
        }
        if (has_s)
#pragma unroll
            for (int ks = 0; ks < 8; ks++) {
                uint32_t a[4];
                frag_a<BT>(a, aQ, m0, ks * 16, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    uint32_t b[4];
                    frag_b_kn<D>(b, aS, ks * 16, n_base + n2 * 16, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
        block_to_rows(acc, sK, mb, nq, srow, o, H, h, lane);       // k has been read: its anchored forms carry it
    }
}

// ---- backward ---------------------------------------------------------------------------------------------------------
// With dS the gradient of the state at the END of the chunk on entry, dA_tj = dO_t . v_j, ew_j = e^{b_n-b_j}:
//   dq_t[i] = e^{b_t[i]} (dO_t S_c^T)[i] + sum_{j<=t} dA_tj k_j[i] e^{b_t[i]-b_j[i]}
//   dk_j[i] = ew_j[i] (v_j dS^T)[i]      + sum_{t>=j} dA_tj q_t[i] e^{b_t[i]-b_j[i]}
//   dv_j    = sum_{t>=j} A_tj dO_t + (k_j .* ew_j) dS
//   dg_t[i] = sum_{tau>=t} (q_tau[i] dq_tau[i] - k_tau[i] dk_tau[i]) + e^{b_n[i]} <S_c[i,:], dS[i,:]> + sum_j k_j[i] ew_j[i] (v_j dS^T)[i]
//   dS     <- Diag(e^{b_n}) dS + (q .* e^{b})^T dO
// The pair sums are split like the scores of the forward: pairs in different 16-row blocks through the anchored
// operands (for dk the factor e^{a_I-b_j} of block I multiplies the product of dA's block with q^ afterwards, so one
// set of anchors serves both), pairs inside a block on the CUDA cores, one thread per (channel, half of the rows).
struct SharedB {
    static constexpr int q = 0, k = 16384, v = 32768, dO = 49152;    // bf16 [64][128]
    static constexpr int b = 65536;                                     // fp32 [64][128]
    static constexpr int sc = 98304;                                    // bf16 [128][128] S_c; later fp32 [64][128] dq
    static constexpr int dsb = 131072;                                  // bf16 [128][128] dS as an MMA operand
    static constexpr int qa = 163840;                                   // bf16 [64][128] anchored q  } later fp32
    static constexpr int ka = qa + 16384;                               // bf16 [96][128] anchored k  } [64][128] dk
    static constexpr int p = ka + 96 * 256;                             // bf16 [64][64] scores
    static constexpr int dab = p + 8192;                                // bf16 [64][64] dA
    static constexpr int dad = dab + 8192;                              // fp32 [64][16] dA, diagonal blocks
    static constexpr int tmp = dad + 4096;                              // fp32 [4][128]
    static constexpr int rowdot = tmp + 2048;                           // fp32 [2][128]
    static constexpr int gi = rowdot + 1024;                            // fp32 [4][128]
    static constexpr int row = gi + 2048;                               // int [64]
    static constexpr int misc = row + 256;
    static constexpr int bytes = misc + 64;
};
static_assert(SharedB::bytes + 1024 <= 232448, "backward tiles do not fit in shared memory");

template <int ROWS = BT>
__device__ __forceinline__ float2 ld_bf2(const unsigned char* tile, int r, int col) {      // [r][col], [r][col+1]; col even
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(tile + sw256<ROWS>(r, col >> 3) + (col & 7) * 2));
}


// ONE_LAUNCH: the grid covers the sequences of all rounds; every CTA draws its item from `ticket` (last round first,
// inside a round the plan's order).  A sequence publishes a flag once its initial-state gradient is in the scratch area;
// a sequence that exported a boundary waits for the flags of all sequences that started there (later rounds, smaller
// tickets, hence running or done) and sums their gradients itself in the order handoff_reduce uses.
template <int MODE>
__global__ void __launch_bounds__(NT, 1)
gk_mma_bwd_kernel(harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const __nv_bfloat16* __restrict__ q,
                  const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, const float* __restrict__ gk,
                  const __nv_bfloat16* __restrict__ dO, __nv_bfloat16* __restrict__ dq, __nv_bfloat16* __restrict__ dk_,
                  __nv_bfloat16* __restrict__ dv_, float* __restrict__ dgk, const __nv_bfloat16* __restrict__ chunk_states,
                  const float* __restrict__ dots, float* __restrict__ ds0, float* __restrict__ rk, float* __restrict__ rv, float* __restrict__ rg,
                  const int32_t* gate, int* status, int* ds0_flags, int* ticket, const RoundOrder rounds, const __grid_constant__ ChunkMaps maps) {
    after_previous();
    if (gate_closed(gate)) return;
    constexpr bool ONE_LAUNCH = MODE == ONE_LAUNCH_MODE, CHUNKS = MODE == CHUNKS_MODE;
    __shared__ int s_item, s_dead;
    extern __shared__ __align__(1024) unsigned char sm[];       // (the static variables ahead of it are padded to 1,024 bytes)
    uint64_t *bar_first = reinterpret_cast<uint64_t*>(sm + SharedB::misc), *bar_rest = bar_first + 1;
    uint32_t ph_first = 0, ph_rest = 0;
    bool ok = true;
    if (CHUNKS) {
        if (s_u32(sm) & 1023) {                       // never on sm_100a; the swizzled tiles would be misread
            if (threadIdx.x == 0 && status) atomicExch(status, tc::STATUS_TIMEOUT);
            return;
        }
        if (threadIdx.x == 0) {
            tc::mbar_init(bar_first, 1);
            tc::mbar_init(bar_rest, 1);
            s_dead = 0;
            tc::fence_barrier_init();
        }
        __syncthreads();
    }
    unsigned char *sQ = sm + SharedB::q, *sK = sm + SharedB::k, *sV = sm + SharedB::v, *sDO = sm + SharedB::dO,
                  *sSc = sm + SharedB::sc, *sdSb = sm + SharedB::dsb, *sQa = sm + SharedB::qa, *sKa = sm + SharedB::ka,
                  *sP = sm + SharedB::p, *sdAb = sm + SharedB::dab;
    float* sB = reinterpret_cast<float*>(sm + SharedB::b);
    float* sR = reinterpret_cast<float*>(sm + SharedB::sc);        // one-step decay factors, after S_c is dead
    float* sDQ = reinterpret_cast<float*>(sm + SharedB::sc);       // after the step factors are dead
    float* sDK = reinterpret_cast<float*>(sm + SharedB::qa);       // after the anchored operands are dead
    float* sdAd = reinterpret_cast<float*>(sm + SharedB::dad);
    float* sTmp = reinterpret_cast<float*>(sm + SharedB::tmp);
    float* sRowdot = reinterpret_cast<float*>(sm + SharedB::rowdot);
    float* sGi = reinterpret_cast<float*>(sm + SharedB::gi);
    int* srow = reinterpret_cast<int*>(sm + SharedB::row);
    const uint32_t aQ = s_u32(sQ), aK = s_u32(sK), aV = s_u32(sV), aDO = s_u32(sDO), aSc = s_u32(sSc), adSb = s_u32(sdSb),
                   aQa = s_u32(sQa), aKa = s_u32(sKa), aP = s_u32(sP), adAb = s_u32(sdAb);

    // blocks are handed to the SMs in index order: with the plan's order (longest sequence of the round first) the long
    // walks start first and the short ones fill the tail
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    const int chunk_lo = CHUNKS ? tb.seq_chunk_ptr[seq_lo] : 0, n_items = CHUNKS ? (tb.seq_chunk_ptr[seq_hi] - chunk_lo) * H : 0;
    int item = blockIdx.x;
    SeqInfo s;
    s.chunk_base = s.n_chunks = 0;
    int seq = seq_lo;
    // CHUNKS: q, k and the log-decays of a chunk; asked for under the outputs of a mild one before it
    bool first_there = false;
    auto load_first = [&](const SeqInfo& s_, int c_, int h_) {
        if (whole_chunk(s_, c_)) {
            if (tid == 0) {
                tc::mbar_expect_tx(bar_first, BT * D * 8);
                tc::tma_load_3d(sB, &maps.g, 0, h_, s_.own_begin - s_.n_replay + c_ * BT, bar_first);
                tma_rows(sQ, &maps.q, s_, c_, h_, bar_first);
                tma_rows(sK, &maps.k, s_, c_, h_, bar_first);
            }
            return;
        }
        auto code_of = [&](int t) { return row_code(tb, s_, c_, t); };
        load_g(gk, H, h_, code_of, sB);
        load_tile_bf16(q, H, h_, code_of, true, sQ);
        load_tile_bf16(k, H, h_, code_of, false, sK);
        tc::cp_async_commit();
    };
    do {
    if (CHUNKS && item >= n_items) break;
    int seq_pos = seq_lo + item / H, h = item % H;
    const int gc = chunk_lo + item / H;
    if constexpr (ONE_LAUNCH) {
        if (tid == 0) {
            s_item = atomicAdd(ticket, 1);
            s_dead = 0;
        }
        __syncthreads();
        int j = s_item / H;
        h = s_item % H;
        seq_pos = -1;
        for (int r = rounds.n - 1; r >= 0 && seq_pos < 0; r--) {      // last round first
            const int cnt = rounds.ptr[r + 1] - rounds.ptr[r];
            if (j < cnt) seq_pos = rounds.ptr[r] + j;
            else j -= cnt;
        }
    }
    if (!CHUNKS || gc >= s.chunk_base + s.n_chunks) {     // chunks come in order: often still the last one's sequence
        seq = CHUNKS ? owner_of(tb, seq, seq_hi, gc) : tb.seq_order ? tb.seq_order[seq_pos] : seq_pos;
        s = seq_info(tb, seq);
    }
    const int mb = warp & 3, nq = warp >> 2;          // this warp's 16-row block and 32-column quarter of [64][128] products
    const size_t state_elems = (size_t)D * D;

    float ds[8][4];                                   // dS, laid out over the warps like the forward's state
#pragma unroll
    for (int n = 0; n < 8; n++) ds[n][0] = ds[n][1] = ds[n][2] = ds[n][3] = 0.f;

    int next_req = s.req_hi - 1;                      // slots of this sequence are ordered by chunk index
    const int c_hi = CHUNKS ? gc - s.chunk_base : s.n_chunks - 1, c_lo = CHUNKS ? c_hi : 0;
    for (int c = c_hi; c >= c_lo; c--) {
        // zero, and neither read nor multiplied: the state of a sequence that starts from zero, the gradient after a last chunk
        const bool has_s = !CHUNKS || c > 0 || s.init_slot >= 0, has_ds = !CHUNKS || c + 1 < s.n_chunks;
        const bool whole = CHUNKS && whole_chunk(s, c);
        if (CHUNKS) tc::fence_async_smem();           // what was written into the tiles, before TMA writes there
        __syncthreads();                              // the previous chunk's readers of every tile are through
        // gradient arriving at boundary c+1 from the sequences that started there: one launch per round -- summed into
        // the first consumer's buffer by handoff_reduce; all rounds in one launch -- awaited and summed here, same order
        if (!CHUNKS && next_req >= s.req_lo && tb.slot_chunk[next_req] == c + 1) {
            const int cons_lo = tb.slot_cons_ptr[next_req], cons_hi = tb.slot_cons_ptr[next_req + 1];
            if constexpr (ONE_LAUNCH) {
                for (int u = cons_lo + tid; u < cons_hi; u += NT)
                    tc::flag_wait(ds0_flags + (size_t)tb.slot_cons_seq[u] * H + h, status, &s_dead);
                if (__syncthreads_or(s_dead)) return;      // a wait ran out (status word set): give the walk up
            }
            if (cons_lo < cons_hi) {
                if constexpr (ONE_LAUNCH) {
                    float a[8][4];
                    state_from_global<false, true>(a, ds0 + ((size_t)tb.slot_cons_seq[cons_lo] * H + h) * state_elems, warp, lane);
                    for (int u = cons_lo + 1; u < cons_hi; u++)
                        state_from_global<true, true>(a, ds0 + ((size_t)tb.slot_cons_seq[u] * H + h) * state_elems, warp, lane);
#pragma unroll
                    for (int n = 0; n < 8; n++) {
                        ds[n][0] += a[n][0]; ds[n][1] += a[n][1]; ds[n][2] += a[n][2]; ds[n][3] += a[n][3];
                    }
                } else {
                    state_from_global<true, false>(ds, ds0 + ((size_t)tb.slot_cons_seq[cons_lo] * H + h) * state_elems, warp, lane);
                }
            }
            next_req--;
        }
        load_codes(tb, s, c, srow);
        float dot = 0.f;                              // CHUNKS: <S_c[i,:], dS[i,:]> in four parts of 32 columns, from the scan (dS is fp32 there)
        if constexpr (CHUNKS) {
            if (!first_there) load_first(s, c, h);
            if (tid == 0 && (whole || has_s || has_ds)) {
                tc::mbar_expect_tx(bar_rest, (whole ? 2 * BT * D * 2 : 0) + (has_s ? D * D * 2 : 0) + (has_ds ? D * D * 2 : 0));
                if (whole) {
                    tma_rows(sV, &maps.v, s, c, h, bar_rest);
                    tma_rows(sDO, &maps.dO, s, c, h, bar_rest);
                }
                if (has_s) tma_state(sSc, &maps.s, gc, h, H, bar_rest);
                if (has_ds) tma_state(sdSb, &maps.ds, gc, h, H, bar_rest);
            }
            if (!whole) {
                auto code_of = [&](int t) { return row_code(tb, s, c, t); };
                load_tile_bf16(v, H, h, code_of, false, sV);
                load_tile_bf16(dO, H, h, code_of, true, sDO);
                tc::cp_async_commit();
            }
            if (tid < 2 * D && has_s && has_ds) {
                const float* part = dots + ((size_t)gc * H + h) * (4 * D) + (tid >> 7) * (2 * D) + (tid & (D - 1));
                dot = part[0] + part[D];
            }
        } else {
            __syncthreads();
            auto code_of = [&](int t) { return srow[t]; };
            load_tile_bf16(k, H, h, code_of, false, sK);
            load_tile_bf16(q, H, h, code_of, true, sQ);
            load_tile_bf16(v, H, h, code_of, false, sV);
            load_tile_bf16(dO, H, h, code_of, true, sDO);
            load_g(gk, H, h, code_of, sB);
        }
        if (!CHUNKS) global_to_tile128(chunk_states + ((size_t)(s.chunk_base + c) * H + h) * state_elems, sSc);
        if (CHUNKS) {
            const NextItem nx = next_item(s, c, gc, item, H, n_items);
            if (nx.c >= 0 && tid == 32) prefetch_chunk(maps, true, s, nx, H);
        } else if (c >= 1) {      // the next chunk of the walk (chunk 0 of a sequence with replayed rows is not consecutive)
            if (c - 1 >= 1 || s.n_replay == 0) {
                prefetch_rows(k, H, h, s, c - 1);
                prefetch_rows(q, H, h, s, c - 1);
                prefetch_rows(v, H, h, s, c - 1);
                prefetch_rows(dO, H, h, s, c - 1);
                prefetch_rows(gk, H, h, s, c - 1);
            }
            const char* st = reinterpret_cast<const char*>(chunk_states + ((size_t)(s.chunk_base + c - 1) * H + h) * state_elems);
            for (int p = tid; p < D * D * 2 / 128; p += NT) asm volatile("prefetch.global.L2 [%0];" ::"l"(st + p * 128));
        }
        if (!CHUNKS) {
            state_to_operand(ds, sdSb, warp, lane);
            tc::cp_async_wait_all();
        } else if (whole) {
            ok = tc::mbar_wait_warp(bar_first, ph_first, status, &s_dead) && ok;
            ph_first ^= 1;
        } else {
            tc::cp_async_wait_group<1>();
        }
        __syncthreads();
        cumsum_rows(sB, sTmp);                        // while the rest comes
        if (CHUNKS) {
            if (whole || has_s || has_ds) {
                ok = tc::mbar_wait_warp(bar_rest, ph_rest, status, &s_dead) && ok;
                ph_rest ^= 1;
            }
            tc::cp_async_wait_all();                  // (published by the barrier in chunk_is_mild)
        }
        const bool mild = chunk_is_mild(sB);          // diagonal blocks as dense products too (see chunk_is_mild)
        const int r_lo = 16 * mb + g, r_hi = r_lo + 8;            // this thread's rows in the [64][128] products
        // ---- dA = dO V^T, iq = dO S_c^T, ik = V dS^T, <S_c, dS> per channel -------------------------------------------
        float iq[4][4], ik[4][4];
        {
            float da[2][4];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                iq[n][0] = iq[n][1] = iq[n][2] = iq[n][3] = 0.f;
                ik[n][0] = ik[n][1] = ik[n][2] = ik[n][3] = 0.f;
            }
#pragma unroll
            for (int n = 0; n < 2; n++) da[n][0] = da[n][1] = da[n][2] = da[n][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ks++) {
                uint32_t a[4], b[4];
                frag_a<BT>(a, aDO, 16 * mb, ks * 16, lane);
                frag_b_nk<BT>(b, aV, ks * 16, 16 * nq, lane);          // dA: columns (keys) 16 * nq ..
                mma16816(da[0], a, b[0], b[1]);
                mma16816(da[1], a, b[2], b[3]);
                if (has_s)
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    frag_b_nk<D>(b, aSc, ks * 16, 32 * nq + 16 * n2, lane);
                    mma16816(iq[2 * n2], a, b[0], b[1]);
                    mma16816(iq[2 * n2 + 1], a, b[2], b[3]);
                }
                if (!has_ds) continue;
                frag_a<BT>(a, aV, 16 * mb, ks * 16, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    frag_b_nk<D>(b, adSb, ks * 16, 32 * nq + 16 * n2, lane);
                    mma16816(ik[2 * n2], a, b[0], b[1]);
                    mma16816(ik[2 * n2 + 1], a, b[2], b[3]);
                }
            }
            // dA: bf16 copy for the block products, fp32 copy of the diagonal 16-blocks for the pair sums
#pragma unroll
            for (int n = 0; n < 2; n++) {
                const int col = 16 * nq + 8 * n + 2 * tq;
                // the bf16 copy serves products that sum over j <= t (or t >= j) only: zero right of the diagonal
                const bool dg_blk = nq == mb;
                const int jc = (col & 15), tr = g;                       // column and row inside the diagonal block
                const float m0 = !dg_blk || jc <= tr ? da[n][0] : 0.f, m1 = !dg_blk || jc + 1 <= tr ? da[n][1] : 0.f;
                const float m2 = !dg_blk || jc <= tr + 8 ? da[n][2] : 0.f, m3 = !dg_blk || jc + 1 <= tr + 8 ? da[n][3] : 0.f;
                *reinterpret_cast<uint32_t*>(sdAb + sw128(r_lo, col >> 3) + (col & 7) * 2) = pack2(m0, m1);
                *reinterpret_cast<uint32_t*>(sdAb + sw128(r_hi, col >> 3) + (col & 7) * 2) = pack2(m2, m3);
                if (nq == mb) {
                    *reinterpret_cast<float2*>(sdAd + r_lo * 16 + (col & 15)) = make_float2(da[n][0], da[n][1]);
                    *reinterpret_cast<float2*>(sdAd + r_hi * 16 + (col & 15)) = make_float2(da[n][2], da[n][3]);
                }
            }
        }
        if constexpr (CHUNKS) {
            if (tid < 2 * D) sRowdot[tid] = dot;
        } else {   // <S_c[i,:], dS[i,:]> over this warp's 64 columns of its 16 state rows i (the two column halves meet later)
            const int i0 = (warp & 7) * 16 + g, c0 = (warp >> 3) * 64 + tq * 2;
            float d_lo = 0.f, d_hi = 0.f;
#pragma unroll
            for (int n = 0; n < 8; n++) {
                const float2 s_lo = ld_bf2<D>(sSc, i0, c0 + n * 8), s_hi = ld_bf2<D>(sSc, i0 + 8, c0 + n * 8);
                d_lo += s_lo.x * ds[n][0] + s_lo.y * ds[n][1];
                d_hi += s_hi.x * ds[n][2] + s_hi.y * ds[n][3];
            }
            d_lo += __shfl_xor_sync(0xffffffffu, d_lo, 1); d_lo += __shfl_xor_sync(0xffffffffu, d_lo, 2);
            d_hi += __shfl_xor_sync(0xffffffffu, d_hi, 1); d_hi += __shfl_xor_sync(0xffffffffu, d_hi, 2);
            if (tq == 0) { sRowdot[(warp >> 3) * D + i0] = d_lo; sRowdot[(warp >> 3) * D + i0 + 8] = d_hi; }
        }
        // inter-chunk parts at the fragment positions: iq <- e^{b_t} iq, ik <- ew ik, and sum_j k_j ew_j ik_j per channel
#pragma unroll
        for (int n = 0; n < 4; n++) {
            const int col = 32 * nq + 8 * n + 2 * tq;
            const float2 b_lo = *reinterpret_cast<const float2*>(sB + b_at(r_lo, col));
            const float2 b_hi = *reinterpret_cast<const float2*>(sB + b_at(r_hi, col));
            const float2 b_n = *reinterpret_cast<const float2*>(sB + b_at(BT - 1, col));
            const float2 k_lo = ld_bf2(sK, r_lo, col), k_hi = ld_bf2(sK, r_hi, col);
            iq[n][0] *= ex2(b_lo.x); iq[n][1] *= ex2(b_lo.y); iq[n][2] *= ex2(b_hi.x); iq[n][3] *= ex2(b_hi.y);
            ik[n][0] *= ex2(b_n.x - b_lo.x); ik[n][1] *= ex2(b_n.y - b_lo.y);
            ik[n][2] *= ex2(b_n.x - b_hi.x); ik[n][3] *= ex2(b_n.y - b_hi.y);
            float g0 = k_lo.x * ik[n][0] + k_hi.x * ik[n][2], g1 = k_lo.y * ik[n][1] + k_hi.y * ik[n][3];
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) {
                g0 += __shfl_xor_sync(0xffffffffu, g0, o);
                g1 += __shfl_xor_sync(0xffffffffu, g1, o);
            }
            if (g == 0) *reinterpret_cast<float2*>(sGi + mb * D + col) = make_float2(g0, g1);
        }
        // ---- scores and the anchored operands ------------------------------------------------------------------------
        // S_c and V are dead from here on; dA is visible
        if constexpr (CHUNKS) {
            if (__syncthreads_or(!ok)) {              // a wait ran out (status word set): let what is in flight land
                tc::drain_delay();
                return;
            }
        } else {
            __syncthreads();
        }
        // a mild chunk's own-block keys and q~ (where the walk goes on) over S_c, its k~ over V; otherwise step factors over S_c
        unsigned char *sKd = sSc, *sQt = sSc + 16384;
        const uint32_t aKd = aSc;
        if (mild) {
            mild_operands(sQ, sK, sB, sQa, sKa, sKd, CHUNKS ? nullptr : sQt, sV);
        } else {
            anchored_operands(sQ, sK, sB, sQa, sKa);
            step_factors(sB, sR);
        }
        __syncthreads();
        scores_off_diagonal(aQa, aKa, sP, warp, lane, mild, aKd);
        // ---- pairs in different blocks -------------------------------------------------------------------------------
        if (mb >= 1 || mild) {   // dq: rows of block mb against the keys of the blocks before it (and, in a mild
                                 // chunk, of its own block: dA is zero right of the diagonal), anchored at block mb
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
            for (int ks = 0; ks < mb + (mild ? 1 : 0); ks++) {
                uint32_t a[4], b[4];
                frag_a<0>(a, adAb, 16 * mb, 16 * ks, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    if (ks < mb) frag_b_kn<96>(b, aKa, ka_row0(mb) + 16 * ks, 32 * nq + 16 * n2, lane);
                    else frag_b_kn<BT>(b, aKd, 16 * mb, 32 * nq + 16 * n2, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                const float2 b_lo = *reinterpret_cast<const float2*>(sB + b_at(r_lo, col));
                const float2 b_hi = *reinterpret_cast<const float2*>(sB + b_at(r_hi, col));
                const float2 an = *reinterpret_cast<const float2*>(sB + b_at(16 * mb, col));
                iq[n][0] += ex2(b_lo.x - an.x) * acc[n][0]; iq[n][1] += ex2(b_lo.y - an.y) * acc[n][1];
                iq[n][2] += ex2(b_hi.x - an.x) * acc[n][2]; iq[n][3] += ex2(b_hi.y - an.y) * acc[n][3];
            }
        }
        // dk: keys of block mb against the queries of block I (in a mild chunk also I = mb: the factor e^{a_I-b_j} is then
        // >= 1 but bounded), anchored at block I
        for (int I = mild ? mb : mb + 1; I < 4; I++) {
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
            uint32_t a[4], b[4];
            frag_a_t<0>(a, adAb, 16 * mb, 16 * I, lane);
#pragma unroll
            for (int n2 = 0; n2 < 2; n2++) {
                frag_b_kn<BT>(b, aQa, 16 * I, 32 * nq + 16 * n2, lane);
                mma16816(acc[2 * n2], a, b[0], b[1]);
                mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
            }
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                const float2 b_lo = *reinterpret_cast<const float2*>(sB + b_at(r_lo, col));
                const float2 b_hi = *reinterpret_cast<const float2*>(sB + b_at(r_hi, col));
                const float2 an = *reinterpret_cast<const float2*>(sB + b_at(16 * I, col));
                ik[n][0] += ex2(an.x - b_lo.x) * acc[n][0]; ik[n][1] += ex2(an.y - b_lo.y) * acc[n][1];
                ik[n][2] += ex2(an.x - b_hi.x) * acc[n][2]; ik[n][3] += ex2(an.y - b_hi.y) * acc[n][3];
            }
        }
        if (mild) {
            // ---- dg, dq, dk straight from the fragments: q dq - k dk summed from the last row up, over the rows of this 16-row
            // block by shuffles (lanes of one column pair hold its eight row pairs), over the blocks through sTmp -----------------
            float z[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                const float2 q_lo = ld_bf2(sQ, r_lo, col), q_hi = ld_bf2(sQ, r_hi, col), k_lo = ld_bf2(sK, r_lo, col), k_hi = ld_bf2(sK, r_hi, col);
                z[n][0] = q_lo.x * iq[n][0] - k_lo.x * ik[n][0];
                z[n][1] = q_lo.y * iq[n][1] - k_lo.y * ik[n][1];
                z[n][2] = q_hi.x * iq[n][2] - k_hi.x * ik[n][2];
                z[n][3] = q_hi.y * iq[n][3] - k_hi.y * ik[n][3];
#pragma unroll
                for (int o_ = 4; o_ <= 16; o_ <<= 1)
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float y = __shfl_down_sync(~0u, z[n][e], o_);
                        if (lane + o_ < 32) z[n][e] += y;
                    }
                z[n][0] += __shfl_sync(~0u, z[n][2], tq);
                z[n][1] += __shfl_sync(~0u, z[n][3], tq);
                if (g == 0) *reinterpret_cast<float2*>(sTmp + mb * D + col) = make_float2(z[n][0], z[n][1]);
            }
            float2 gamma[4];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const float2 bn = *reinterpret_cast<const float2*>(sB + b_at(BT - 1, 32 * nq + 8 * n + 2 * tq));
                gamma[n] = make_float2(ex2(bn.x), ex2(bn.y));
            }
            if (CHUNKS) tc::fence_async_smem();
            __syncthreads();
            if constexpr (CHUNKS) {                   // q, k and the running sums have been read: the next item's come in over them
                const int next = item + gridDim.x, gc2 = chunk_lo + next / H;
                first_there = next < n_items;
                if (first_there) {
                    if (gc2 < s.chunk_base + s.n_chunks) {
                        load_first(s, gc2 - s.chunk_base, next % H);
                    } else {
                        const SeqInfo s2 = seq_info(tb, owner_of(tb, seq, seq_hi, gc2));
                        load_first(s2, gc2 - s2.chunk_base, next % H);
                    }
                }
            }
            const int code_lo = srow[r_lo], code_hi = srow[r_hi];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                auto at = [&](const float* x) { return *reinterpret_cast<const float2*>(x + col); };
                // <S_{c+1}[i,:], dS[i,:]> = e^{b_n} <S_c, dS> + sum_j k_j ew_j ik_j, and the blocks below this one
                const float2 d0 = at(sRowdot), d1 = at(sRowdot + D);
                float2 tail = make_float2(gamma[n].x * (d0.x + d1.x), gamma[n].y * (d0.y + d1.y));
#pragma unroll
                for (int b2 = 0; b2 < 4; b2++) {
                    const float2 x = at(sGi + b2 * D), y = at(sTmp + b2 * D);
                    tail.x += x.x + (b2 > mb ? y.x : 0.f);
                    tail.y += x.y + (b2 > mb ? y.y : 0.f);
                }
                auto put = [&](int code, int r, float2 dkv, float2 dgv) {      // replayed rows: fp32 to the scratch
                    if (code >= 0) {
                        *reinterpret_cast<float2*>(dgk + ((size_t)code * H + h) * D + col) = dgv;
                    } else if (code < -1) {
                        const size_t off = ((size_t)(s.replay_base + r) * H + h) * D + col;
                        *reinterpret_cast<float2*>(rk + off) = dkv;
                        *reinterpret_cast<float2*>(rg + off) = dgv;
                    }
                };
                put(code_lo, r_lo, make_float2(ik[n][0], ik[n][1]),
                    make_float2(z[n][0] + tail.x, z[n][1] + tail.y));
                put(code_hi, r_hi, make_float2(ik[n][2], ik[n][3]),
                    make_float2(z[n][2] + tail.x, z[n][3] + tail.y));
            }
            block_to_rows(iq, sQa, mb, nq, srow, dq, H, h, lane);      // over the anchored operands, which have been multiplied
            block_to_rows(ik, sKa, mb, nq, srow, dk_, H, h, lane);
        } else {
            first_there = false;
            __syncthreads();                              // the anchored operands are dead, the step factors visible
            scores_diagonal(sQ, sK, sR, sP, warp, lane);
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                *reinterpret_cast<float2*>(sDK + r_lo * D + col) = make_float2(ik[n][0], ik[n][1]);
                *reinterpret_cast<float2*>(sDK + r_hi * D + col) = make_float2(ik[n][2], ik[n][3]);
            }
            __syncthreads();                              // the step factors / own-block keys are dead
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                *reinterpret_cast<float2*>(sDQ + r_lo * D + col) = make_float2(iq[n][0], iq[n][1]);
                *reinterpret_cast<float2*>(sDQ + r_hi * D + col) = make_float2(iq[n][2], iq[n][3]);
            }
            __syncthreads();

            // ---- pairs inside a 16-block and dg: thread = (channel i, 16-row block blk) --------------------------------------
            {
                const int i = tid & (D - 1), blk = tid >> 7, t0 = 16 * blk;
                {
                    // rows ascending; xr[u] = 2^{b_t - b_u} as a running product of the one-step factors (one exponential per
                    // row instead of one per pair; every factor <= 1), the same factor for dq and dk
                    float dk_acc[16], kf[16], xr[16];
#pragma unroll
                    for (int u = 0; u < 16; u++) {
                        dk_acc[u] = 0.f;
                        kf[u] = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(sK + sw256(t0 + u, i >> 3) + (i & 7) * 2));
                    }
                    float b_prev = 0.f;
#pragma unroll
                    for (int tt = 0; tt < 16; tt++) {
                        const int t = t0 + tt;
                        const float qt = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(sQ + sw256(t, i >> 3) + (i & 7) * 2));
                        const float bt = sB[b_at(t, i)];
                        const float r = ex2(bt - b_prev);
                        b_prev = bt;
                        xr[tt] = 1.f;
                        float dq_acc = 0.f;
#pragma unroll
                        for (int u = 0; u <= tt; u++) {
                            if (u < tt) xr[u] *= r;
                            const float x = sdAd[t * 16 + u] * xr[u];
                            dq_acc += x * kf[u];
                            dk_acc[u] += x * qt;
                        }
                        sDQ[t * D + i] += dq_acc;
                    }
#pragma unroll
                    for (int tt = 0; tt < 16; tt++) sDK[(t0 + tt) * D + i] += dk_acc[tt];
                }
                float term[16], total = 0.f;                  // q dq - k dk of this thread's rows, and their sum
#pragma unroll
                for (int tt = 0; tt < 16; tt++) {
                    const int t = t0 + tt;
                    const float qt = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(sQ + sw256(t, i >> 3) + (i & 7) * 2));
                    const float kt = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(sK + sw256(t, i >> 3) + (i & 7) * 2));
                    term[tt] = qt * sDQ[t * D + i] - kt * sDK[t * D + i];
                    total += term[tt];
                }
                sTmp[blk * D + i] = total;
                __syncthreads();
                // dg_t = suffix over the rows + <S_{c+1}[i,:], dS[i,:]> = e^{b_n} <S_c, dS> + sum_j k_j ew_j ik_j
                float suffix = ex2(sB[b_at(BT - 1, i)]) * (sRowdot[i] + sRowdot[D + i]) + sGi[i] + sGi[D + i] + sGi[2 * D + i] +
                               sGi[3 * D + i];
                for (int b2 = 3; b2 > blk; b2--) suffix += sTmp[b2 * D + i];
#pragma unroll
                for (int tt = 15; tt >= 0; tt--) {
                    const int t = t0 + tt, code = srow[t];
                    if (code == -1) continue;
                    suffix += term[tt];
                    if (code >= 0) dgk[((size_t)code * H + h) * D + i] = suffix;
                    else rg[((size_t)(s.replay_base + t) * H + h) * D + i] = suffix;     // replayed rows sit in chunk 0
                }
            }
            __syncthreads();
            // ---- dq, dk out: own rows as bf16, replayed rows' dk in fp32 to the scratch -------------------------------------
#pragma unroll
            for (int u = 0; u < BT * 16 / NT; u++) {
                const int p = tid + u * NT, t = p >> 4, c16 = p & 15, code = srow[t];
                if (code == -1) continue;
                const float4 q0 = *reinterpret_cast<const float4*>(sDQ + t * D + c16 * 8), q1 = *reinterpret_cast<const float4*>(sDQ + t * D + c16 * 8 + 4);
                const float4 k0 = *reinterpret_cast<const float4*>(sDK + t * D + c16 * 8), k1 = *reinterpret_cast<const float4*>(sDK + t * D + c16 * 8 + 4);
                if (code >= 0) {
                    const size_t off = ((size_t)code * H + h) * D + c16 * 8;
                    *reinterpret_cast<uint4*>(dq + off) = make_uint4(pack2(q0.x, q0.y), pack2(q0.z, q0.w), pack2(q1.x, q1.y), pack2(q1.z, q1.w));
                    *reinterpret_cast<uint4*>(dk_ + off) = make_uint4(pack2(k0.x, k0.y), pack2(k0.z, k0.w), pack2(k1.x, k1.y), pack2(k1.z, k1.w));
                } else {
                    float* dst = rk + ((size_t)(s.replay_base + t) * H + h) * D + c16 * 8;
                    *reinterpret_cast<float4*>(dst) = k0;
                    *reinterpret_cast<float4*>(dst + 4) = k1;
                }
            }
            scale_qk<!CHUNKS, true>(sQ, sK, sB, sQ, sK);  // q~, k~ over the raw tiles, which nobody reads any more
            __syncthreads();
        }
        const uint32_t aQt = mild ? s_u32(sQt) : aQ, aKt = mild ? aV : aK;
        // ---- dv_j = sum_{t>=j} A_tj dO_t + k~_j dS : warp -> rows 16 * mb, columns 32 * nq -------------------------------
        {
            float acc[4][4];
#pragma unroll
            for (int n = 0; n < 4; n++) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
            for (int ks = mb; ks < 4; ks++) {             // A_tj = 0 for t < j
                uint32_t a[4], b[4];
                frag_a_t<0>(a, aP, 16 * mb, 16 * ks, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    frag_b_kn<BT>(b, aDO, 16 * ks, 32 * nq + 16 * n2, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
            if (has_ds)
#pragma unroll
            for (int ks = 0; ks < 8; ks++) {
                uint32_t a[4], b[4];
                frag_a<BT>(a, aKt, 16 * mb, 16 * ks, lane);
#pragma unroll
                for (int n2 = 0; n2 < 2; n2++) {
                    frag_b_kn<D>(b, adSb, 16 * ks, 32 * nq + 16 * n2, lane);
                    mma16816(acc[2 * n2], a, b[0], b[1]);
                    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
                }
            }
            const int row_lo = srow[r_lo], row_hi = srow[r_hi];
#pragma unroll
            for (int n = 0; n < 4; n++) {
                const int col = 32 * nq + 8 * n + 2 * tq;
                if (row_lo < -1) *reinterpret_cast<float2*>(rv + ((size_t)(s.replay_base + r_lo) * H + h) * D + col) = make_float2(acc[n][0], acc[n][1]);
                if (row_hi < -1) *reinterpret_cast<float2*>(rv + ((size_t)(s.replay_base + r_hi) * H + h) * D + col) = make_float2(acc[n][2], acc[n][3]);
            }
            block_to_rows(acc, sQa, mb, nq, srow, dv_, H, h, lane);
        }
        // ---- dS <- Diag(e^{b_n}) dS + q~^T dO ---------------------------------------------------------------------------
        if (!CHUNKS) state_update(ds, sB, aQt, aDO, warp, lane);
    }
    if (!CHUNKS && s.init_slot >= 0) {
        state_to_global(ds, ds0 + ((size_t)seq * H + h) * state_elems, warp, lane);
        if constexpr (ONE_LAUNCH) {
            __threadfence();                           // this thread's part, before the flag that follows the barrier
            __syncthreads();
            if (tid == 0) tc::flag_set(ds0_flags + (size_t)seq * H + h);
        }
    }
    item += gridDim.x;
    } while (CHUNKS);
}

}  // namespace

int32_t gk_mma_supported(int32_t dtype, int32_t dk, int32_t dv) { return dtype == HARTS_BF16 && dk == D && dv == D; }

int32_t gk_mma_fwd(const FwdArgs& a) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    if (cudaFuncSetAttribute(gk_mma_fwd_kernel<ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shared::fwd_bytes) !=
        cudaSuccess)
        return HARTS_ECUDA;
    const int n = (a.seq_hi - a.seq_lo) * a.H;
    gk_mma_fwd_kernel<ROUND><<<n, NT, Shared::fwd_bytes, a.stream>>>(
        a.tb, a.seq_lo, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (__nv_bfloat16*)a.o, a.slots, (__nv_bfloat16*)a.chunk_states, status_gate(a.flags, a.dev_status), a.dev_status,
        nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

int32_t gk_mma_bwd(const BwdArgs& a) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    if (cudaFuncSetAttribute(gk_mma_bwd_kernel<ROUND>, cudaFuncAttributeMaxDynamicSharedMemorySize, SharedB::bytes) !=
        cudaSuccess)
        return HARTS_ECUDA;
    const int n = (a.seq_hi - a.seq_lo) * a.H;
    const GkScratchLayout sl = gk_scratch_layout(a.tb, a.H, a.dk, a.dv);
    char* base = static_cast<char*>(a.scratch);
    gk_mma_bwd_kernel<ROUND><<<n, NT, SharedB::bytes, a.stream>>>(
        a.tb, a.seq_lo, a.seq_hi, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (const __nv_bfloat16*)a.dO, (__nv_bfloat16*)a.dq, (__nv_bfloat16*)a.dk_, (__nv_bfloat16*)a.dv_, a.dg,
        (const __nv_bfloat16*)a.chunk_states, nullptr, (float*)(base + sl.ds0), (float*)(base + sl.rk), (float*)(base + sl.rv),
        (float*)(base + sl.rg), status_gate(a.flags, a.dev_status), a.dev_status, nullptr, nullptr, RoundOrder{}, ChunkMaps{});
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

// All rounds in one launch per pass (sequences [seq_lo, seq_hi) = the whole plan).  flags: n_slots * H (forward) or
// n_seq * H (backward) int32 on the device, ticket: one int32; both zeroed here on the stream.  Offered while the
// problem has few items per SM, like the scalar-gate forms; HARTS_EUNSUPPORTED otherwise.
int32_t gk_mma_fwd_all(const FwdArgs& a, int* flags, int* ticket) {
    const int64_t n = (int64_t)(a.seq_hi - a.seq_lo) * a.H;
    if (n == 0) return HARTS_OK;
    if (n > (int64_t)ONE_LAUNCH_ITEMS_PER_CTA * sm_count()) return HARTS_EUNSUPPORTED;
    if (cudaFuncSetAttribute(gk_mma_fwd_kernel<ONE_LAUNCH_MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, Shared::fwd_bytes) !=
        cudaSuccess)
        return HARTS_ECUDA;
    if (a.tb.n_slots > 0 &&
        cudaMemsetAsync(flags, 0, (size_t)a.tb.n_slots * a.H * sizeof(int), a.stream) != cudaSuccess)
        return HARTS_ECUDA;
    if (cudaMemsetAsync(ticket, 0, sizeof(int), a.stream) != cudaSuccess) return HARTS_ECUDA;
    gk_mma_fwd_kernel<ONE_LAUNCH_MODE><<<(int)n, NT, Shared::fwd_bytes, a.stream>>>(
        a.tb, a.seq_lo, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (__nv_bfloat16*)a.o, a.slots, (__nv_bfloat16*)a.chunk_states, status_gate(a.flags, a.dev_status), a.dev_status,
        flags, ticket);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

int32_t gk_mma_bwd_all(const BwdArgs& a, int* flags, int* ticket, const RoundOrder& rounds) {
    const int64_t n = (int64_t)(a.seq_hi - a.seq_lo) * a.H;
    if (n == 0) return HARTS_OK;
    if (rounds.n < 1 || rounds.ptr[0] != a.seq_lo || rounds.ptr[rounds.n] != a.seq_hi) return HARTS_EINVAL;
    if (n > (int64_t)ONE_LAUNCH_ITEMS_PER_CTA * sm_count()) return HARTS_EUNSUPPORTED;
    if (cudaFuncSetAttribute(gk_mma_bwd_kernel<ONE_LAUNCH_MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SharedB::bytes) !=
        cudaSuccess)
        return HARTS_ECUDA;
    if (cudaMemsetAsync(flags, 0, (size_t)a.tb.n_seq * a.H * sizeof(int), a.stream) != cudaSuccess) return HARTS_ECUDA;
    if (cudaMemsetAsync(ticket, 0, sizeof(int), a.stream) != cudaSuccess) return HARTS_ECUDA;
    const GkScratchLayout sl = gk_scratch_layout(a.tb, a.H, a.dk, a.dv);
    char* base = static_cast<char*>(a.scratch);
    gk_mma_bwd_kernel<ONE_LAUNCH_MODE><<<(int)n, NT, SharedB::bytes, a.stream>>>(
        a.tb, a.seq_lo, a.seq_hi, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (const __nv_bfloat16*)a.dO, (__nv_bfloat16*)a.dq, (__nv_bfloat16*)a.dk_, (__nv_bfloat16*)a.dv_, a.dg,
        (const __nv_bfloat16*)a.chunk_states, nullptr, (float*)(base + sl.ds0), (float*)(base + sl.rk), (float*)(base + sl.rv),
        (float*)(base + sl.rg), status_gate(a.flags, a.dev_status), a.dev_status, flags, ticket, rounds, ChunkMaps{});
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

// Every (chunk, head) of sequences [seq_lo, seq_hi) on its own; the scan has left the states (and their gradients).
static int32_t chunk_maps(ChunkMaps* m, const harts_la_tables_t& tb, int32_t H, const void* q, const void* k, const void* v, const void* dO, const float* g,
                          const void* states, const void* ds_tiles) {
    const int64_t rows = tb.n_rows, tiles = (int64_t)tb.n_chunks * H;
    int32_t rc;
    if ((rc = make_row_map(&m->q, q, rows, H)) != HARTS_OK || (rc = make_row_map(&m->k, k, rows, H)) != HARTS_OK ||
        (rc = make_row_map(&m->v, v, rows, H)) != HARTS_OK || (rc = make_gate_map(&m->g, g, rows, H)) != HARTS_OK ||
        (rc = make_state_map(&m->s, states, tiles)) != HARTS_OK)
        return rc;
    m->dO = m->v;
    m->ds = m->s;
    if (dO && ((rc = make_row_map(&m->dO, dO, rows, H)) != HARTS_OK || (rc = make_state_map(&m->ds, ds_tiles, tiles)) != HARTS_OK)) return rc;
    return HARTS_OK;
}
int32_t gk_chunk_fwd(const FwdArgs& a) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    ChunkMaps maps;
    const int32_t rc = chunk_maps(&maps, a.tb, a.H, a.q, a.k, a.v, nullptr, a.g, a.chunk_states, nullptr);
    if (rc != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(gk_chunk_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SharedC::bytes) != cudaSuccess)
        return HARTS_ECUDA;
    const int64_t n = (int64_t)a.tb.n_chunks * a.H;
    launch_after(gk_chunk_fwd_kernel, (int)(n < 2 * sm_count() ? n : 2 * sm_count()), NT, SharedC::bytes, a.stream,
        a.tb, a.seq_lo, a.seq_hi, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (__nv_bfloat16*)a.o, maps, a.dev_status, status_gate(a.flags, a.dev_status));
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}
int32_t gk_chunk_bwd(const BwdArgs& a, const void* ds_tiles, const float* dots) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    ChunkMaps maps;
    const int32_t rc = chunk_maps(&maps, a.tb, a.H, a.q, a.k, a.v, a.dO, a.g, a.chunk_states, ds_tiles);
    if (rc != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(gk_mma_bwd_kernel<CHUNKS_MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, SharedB::bytes) != cudaSuccess)
        return HARTS_ECUDA;
    const int64_t n = (int64_t)a.tb.n_chunks * a.H;
    const GkScratchLayout sl = gk_scratch_layout(a.tb, a.H, a.dk, a.dv);
    char* base = static_cast<char*>(a.scratch);
    launch_after(gk_mma_bwd_kernel<CHUNKS_MODE>, (int)(n < sm_count() ? n : sm_count()), NT, SharedB::bytes, a.stream,
        a.tb, a.seq_lo, a.seq_hi, a.H, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g,
        (const __nv_bfloat16*)a.dO, (__nv_bfloat16*)a.dq, (__nv_bfloat16*)a.dk_, (__nv_bfloat16*)a.dv_, a.dg,
        nullptr, dots, (float*)(base + sl.ds0), (float*)(base + sl.rk), (float*)(base + sl.rv), (float*)(base + sl.rg),
        status_gate(a.flags, a.dev_status), a.dev_status, nullptr, nullptr, RoundOrder{}, maps);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
