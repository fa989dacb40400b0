// Chunk-parallel path for fp32 inputs, d_k = d_v = 64, chunk 64, on the CUDA cores (no reduced-precision product anywhere).
//
//   outer_kernel   U_c = sum_j (w_j k_j)^T v_j of every chunk, w_j = e^{b_n-b_j} (backward: W_c = sum_t (e^{b_t} q_t)^T dO_t), e^{b_n}
//   walk_kernel    S_{c+1} = e^{b_n} S_c + U_c along the chunks of a sequence, element by element, one launch per round; the
//                  state at the start of a chunk replaces the chunk's sum in the workspace (backward: the gradient at its end)
//   out_kernel     o_t = e^{b_t} q_t S_c + sum_{j<=t} A_tj v_j
//   grad_kernel    dq, dk, dv, dg of a chunk from its rows, S_c and dS_{c+1} (formulas: la_fma.cu)
// The kernels of la_fma.cu walk a sequence's chunks with everything in one CTA: 84 us per chunk, forward and backward, one
// after the other.  Only the walk is serial here, and its step is one multiply-add per element with the operand prefetched;
// the 64^3 products of different chunks run side by side.  What bounds it: launches and the latency of one product (256
// threads x 4x4 outputs, 2,048 cycles at 128 multiply-adds a clock) on small forests, the CUDA cores on large ones.  Forward +
// backward, cold inputs, against the walk: 718 tokens x 1 head (two rounds) 1.33 -> 0.086 ms (outer 9 + 7, walk 3 per round, out 13,
// grad 25 us), 12,000 branchy x 4 12.0 -> 0.32, 40,000 replay x 8 13.6 -> 3.9, 150,000 agentic x 4 46.4 -> 3.3 (grad 2.0, out 0.7).
// All but the first kernel of a call are on the SMs before the one ahead of them is done (launch_after).  What needs the call's inputs
// alone they do before they wait: a walk its tables, outputs and gradients the lookup, the rows, the scores and a chunk's own share --
// 718 tokens 69.7 -> 51.2 us a step, 796 items 313 -> 293, 3,824 items 1,255 -> 1,235.
// grad_kernel has one CTA an SM (141 KB): sixteen warps of 2x4 outputs instead of eight of 4x4 -- more shared-memory reads, twice the
// warps to hide them -- and diagonals that are not unrolled took it from 31.3 to 24.8 us on 13 items, 174 to 159 on 796.
#include "chunk_item.cuh"

namespace harts {

int sm_count();

namespace {

using chunk::BT;
using chunk::find_item;
using chunk::Item;
using chunk::RowData;
using tc::ex2;

constexpr int D = 64, NT = 256, LD = D + 4;      // rows of shared-memory tiles are padded: 16-byte aligned, conflict-free by column
constexpr int TILE = BT * LD;                    // floats

// Thread (ty, tx) = (tid / 16, tid % 16) owns outputs (R ty + r, tx + 16 c), r = 0..R-1, c = 0..3; a warp owns 2 R rows.  R = 4 with 256
// threads, R = 2 with 512.
template <int R>
struct AccT {
    float a[R][4];
    __device__ float* operator[](int r) { return a[r]; }
    __device__ const float* operator[](int r) const { return a[r]; }
};
template <int R>
__device__ __forceinline__ void clear(AccT<R>& a) {
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) a[r][c] = 0.f;
}
// a += X Y^T over column blocks 0..n_col-1 of 16
template <int N_COL, int R>
__device__ __forceinline__ void mul_nt(AccT<R>& a, const float* x, const float* y, int ty, int tx) {
#pragma unroll 4
    for (int i = 0; i < D; i += 4) {
        float4 xv[R];
#pragma unroll
        for (int r = 0; r < R; r++) xv[r] = *reinterpret_cast<const float4*>(x + (R * ty + r) * LD + i);
#pragma unroll
        for (int c = 0; c < N_COL; c++) {
            const float4 yv = *reinterpret_cast<const float4*>(y + (tx + 16 * c) * LD + i);
#pragma unroll
            for (int r = 0; r < R; r++) a[r][c] += xv[r].x * yv.x + xv[r].y * yv.y + xv[r].z * yv.z + xv[r].w * yv.w;
        }
    }
}
// the same where only columns <= the warp's last row are wanted (the rest of a stays as it is)
template <int R>
__device__ __forceinline__ void mul_nt_causal(AccT<R>& a, const float* x, const float* y, int ty, int tx) {
    switch (R * ty >> 4) {                       // 16-row groups
        case 0: mul_nt<1>(a, x, y, ty, tx); break;
        case 1: mul_nt<2>(a, x, y, ty, tx); break;
        case 2: mul_nt<3>(a, x, y, ty, tx); break;
        default: mul_nt<4>(a, x, y, ty, tx);
    }
}
// a += X[:, k0..k1) Y[k0..k1, :)
template <int R>
__device__ __forceinline__ void mul_nn(AccT<R>& a, const float* x, const float* y, int k0, int k1, int ty, int tx) {
#pragma unroll 2
    for (int k = k0; k < k1; k += 4) {
        float4 xv[R];
#pragma unroll
        for (int r = 0; r < R; r++) xv[r] = *reinterpret_cast<const float4*>(x + (R * ty + r) * LD + k);
#pragma unroll
        for (int kk = 0; kk < 4; kk++)
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const float yv = y[(k + kk) * LD + tx + 16 * c];
#pragma unroll
                for (int r = 0; r < R; r++) a[r][c] += (kk == 0 ? xv[r].x : kk == 1 ? xv[r].y : kk == 2 ? xv[r].z : xv[r].w) * yv;
            }
    }
}
// a += X[t0..64, :)^T Y[t0..64, :)
template <int R>
__device__ __forceinline__ void load_r(float (&x)[R], const float* from) {       // R floats in a row, aligned so
    if constexpr (R == 4) *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(from);
    else *reinterpret_cast<float2*>(x) = *reinterpret_cast<const float2*>(from);
}
template <int R>
__device__ __forceinline__ void mul_tn(AccT<R>& a, const float* x, const float* y, int t0, int ty, int tx) {
#pragma unroll 4
    for (int t = t0; t < BT; t++) {
        float xv[R];
        load_r<R>(xv, x + t * LD + R * ty);
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const float yv = y[t * LD + tx + 16 * c];
#pragma unroll
            for (int r = 0; r < R; r++) a[r][c] += xv[r] * yv;
        }
    }
}

// The 2 R columns (rows) at the diagonal of a warp's rows: what lies past the diagonal is left out, not multiplied by zero, so
// that an infinity or a NaN in a later row stays out of the rows before it.
// a += P[:, k0..k0+2R) Y[k0..k0+2R, :), columns up to the row
template <int R>
__device__ __forceinline__ void mul_nn_diagonal(AccT<R>& a, const float* x, const float* y, int k0, int ty, int tx) {
#pragma unroll 1
    for (int k = k0; k < k0 + 2 * R; k += 4) {
        float xv[R][4];
#pragma unroll
        for (int r = 0; r < R; r++) *reinterpret_cast<float4*>(xv[r]) = *reinterpret_cast<const float4*>(x + (R * ty + r) * LD + k);
#pragma unroll
        for (int kk = 0; kk < 4; kk++)
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const float yv = y[(k + kk) * LD + tx + 16 * c];
#pragma unroll
                for (int r = 0; r < R; r++) a[r][c] = k + kk <= R * ty + r ? a[r][c] + xv[r][kk] * yv : a[r][c];
            }
    }
}
// a += P[t0..t0+2R, :)^T Y[t0..t0+2R, :), rows from the column on
template <int R>
__device__ __forceinline__ void mul_tn_diagonal(AccT<R>& a, const float* x, const float* y, int t0, int ty, int tx) {
#pragma unroll 2
    for (int t = t0; t < t0 + 2 * R; t++) {
        float xv[R];
        load_r<R>(xv, x + t * LD + R * ty);
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const float yv = y[t * LD + tx + 16 * c];
#pragma unroll
            for (int r = 0; r < R; r++) a[r][c] = t >= R * ty + r ? a[r][c] + xv[r] * yv : a[r][c];
        }
    }
}

// Row data with the running log-decay to twice 32 bits (b2 + b2_lo): the decay between two rows is the exponential of a
// difference of two running sums, and after a steep gate both are large.  Summed in 64 bits by the same warp scan.
struct Rows : RowData {
    float b2_lo[BT];
    __device__ float decay(int t, int j) const { return ex2((b2[t] - b2[j]) + (b2_lo[t] - b2_lo[j])); }
};
__device__ __forceinline__ void store_gates(Rows& rd, const float (&gv)[2], int lane) {
    double x0 = gv[0] * 1.4426950408889634074, x1 = gv[1] * 1.4426950408889634074;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y0 = __shfl_up_sync(~0u, x0, o), y1 = __shfl_up_sync(~0u, x1, o);
        if (lane >= o) {
            x0 += y0;
            x1 += y1;
        }
    }
    x1 += __shfl_sync(~0u, x0, 31);
    const double bn = __shfl_sync(~0u, x1, 31), x[2] = {x0, x1};
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const int t = lane + 32 * r;
        const float hi = (float)x[r];
        rd.b2[t] = hi;
        rd.b2_lo[t] = isinf(hi) ? 0.f : (float)(x[r] - hi);
        rd.eb[t] = ex2(hi);
        rd.w[t] = ex2((float)(bn - x[r]));
    }
    if (lane == 0) rd.gamma = ex2((float)bn);
}

// Rows of a chunk into a tile; `own`: replayed rows (and rows past the end) are zero, else only rows past the end.
__device__ __forceinline__ void load_tile(float* dst, const float* src, const Rows& rd, bool own, int h, int H) {
    for (int e = threadIdx.x; e < BT * 16; e += blockDim.x) {
        const int t = e >> 4, ch = e & 15, code = rd.code[t], r = code >= 0 ? code : -2 - code;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (own ? code >= 0 : code != -1) x = *reinterpret_cast<const float4*>(src + ((size_t)r * H + h) * D + ch * 4);
        *reinterpret_cast<float4*>(dst + t * LD + ch * 4) = x;
    }
}
__device__ __forceinline__ void load_state(float* dst, const float* src) {
    for (int e = threadIdx.x; e < D * 16; e += blockDim.x)
        *reinterpret_cast<float4*>(dst + (e >> 4) * LD + (e & 15) * 4) = *reinterpret_cast<const float4*>(src + e * 4);
}
// The CTA's item `idx` of the range: warp 0 finds it and prepares its row data.  False: the range has no such item.  On return
// the record and the row codes are there for all; the gates' sums and weights are after the CTA's next barrier, so that warp 0
// works them out while the others load the tiles.
__device__ __forceinline__ bool begin_item(const harts_la_tables_t& tb, int seq_lo, int seq_hi, int H, const float* g, int idx, Rows& rd,
                                           Item& it) {
    const int gc = tb.seq_chunk_ptr[seq_lo] + idx / H, lane = threadIdx.x;
    if (gc >= tb.seq_chunk_ptr[seq_hi]) return false;
    __syncthreads();                             // the last readers of the item before are through
    float gv[2];
    if (threadIdx.x < 32) {
        const Item x = find_item(tb, seq_lo, seq_hi, gc, idx % H, lane);
        int code[2];
        chunk::load_rows(tb, x, g, H, lane, code, gv);
        rd.code[lane] = code[0];
        rd.code[lane + 32] = code[1];
        if (lane == 0) it = x;
    }
    __syncthreads();
    if (threadIdx.x < 32) store_gates(rd, gv, lane);
    return true;
}

struct __align__(16) OuterSmem {
    float x[TILE], y[TILE];
    Rows rd;
    Item it;
};
template <bool BWD>
__global__ void __launch_bounds__(NT, 5) outer_kernel(const harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const float* __restrict__ a,
                                                   const float* __restrict__ b, const float* __restrict__ g, float* __restrict__ sums,
                                                   float* __restrict__ gammas, const int32_t* gate) {
    let_next_launch();
    after_previous();
    if (gate_closed(gate)) return;
    __shared__ OuterSmem s;
    for (int idx = blockIdx.x; begin_item(tb, seq_lo, seq_hi, H, g, idx, s.rd, s.it); idx += gridDim.x) {
    const Item& it = s.it;
    if (BWD ? it.zero_state : it.last) continue; // this chunk's sum enters nothing
    load_tile(s.x, a, s.rd, BWD, it.h, H);
    float4 y[BT * 16 / NT];                      // the operand that is weighted
#pragma unroll
    for (int u = 0; u < BT * 16 / NT; u++) {
        const int e = threadIdx.x + u * NT, code = s.rd.code[e >> 4], r = code >= 0 ? code : -2 - code;
        y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (BWD ? code >= 0 : code != -1) y[u] = *reinterpret_cast<const float4*>(b + ((size_t)r * H + it.h) * D + (e & 15) * 4);
    }
    __syncthreads();                             // the weights
#pragma unroll
    for (int u = 0; u < BT * 16 / NT; u++) {
        const int e = threadIdx.x + u * NT, t = e >> 4;
        const float w = BWD ? s.rd.eb[t] : s.rd.w[t];
        *reinterpret_cast<float4*>(s.y + t * LD + (e & 15) * 4) = make_float4(y[u].x * w, y[u].y * w, y[u].z * w, y[u].w * w);
    }
    __syncthreads();
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    AccT<4> acc;
    clear(acc);
    mul_tn(acc, s.x, s.y, 0, ty, tx);
    float* dst = sums + ((size_t)it.gc * H + it.h) * (D * D);
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) dst[(4 * ty + r) * D + tx + 16 * c] = acc[r][c];
    if (threadIdx.x == 0) gammas[(size_t)it.gc * H + it.h] = s.rd.gamma;
    }
}

// One thread walks four elements of the state along a sequence; four CTAs per (sequence, head).
constexpr int AHEAD = 8;                         // sums in flight per thread
template <bool BWD>
__global__ void __launch_bounds__(NT) walk_kernel(const harts_la_tables_t tb, int seq_lo, int H, float* tiles, const float* gammas,
                                                  float* slots, float* ds0, const int32_t* gate) {
    let_next_launch();
    if (gate_closed(gate)) return after_previous();
    const int part = blockIdx.x & 3, item = blockIdx.x >> 2, h = item % H;
    const int pos = seq_lo + item / H, seq = tb.seq_order ? tb.seq_order[pos] : pos;
    const int chunk_base = tb.seq_chunk_ptr[seq], n_chunks = tb.seq_chunk_ptr[seq + 1] - chunk_base;
    const int init_slot = tb.seq_init_slot[seq], req_lo = tb.seq_req_ptr[seq], req_hi = tb.seq_req_ptr[seq + 1];
    const int n_steps = BWD && init_slot >= 0 ? n_chunks : n_chunks - 1;
    const size_t stride = (size_t)H * (D * D), el = (size_t)h * (D * D) + part * 1024 + threadIdx.x * 4;
    auto chunk_of = [&](int i) { return BWD ? n_chunks - 1 - i : i; };
    auto load = [&](int i0, float4 (&u)[AHEAD], float (&gm)[AHEAD]) {
#pragma unroll
        for (int j = 0; j < AHEAD; j++)
            if (i0 + j < n_steps) {
                const size_t gc = chunk_base + chunk_of(i0 + j);
                u[j] = *reinterpret_cast<const float4*>(tiles + gc * stride + el);
                gm[j] = gammas[gc * H + h];
            }
    };
    float4 u[AHEAD], un[AHEAD], x = make_float4(0.f, 0.f, 0.f, 0.f);
    float gm[AHEAD], gn[AHEAD];
    int req = BWD ? req_hi - 1 : req_lo;
    int boundary = (BWD ? req >= req_lo : req < req_hi) ? tb.slot_chunk[req] : -1;
    after_previous();                            // the tables are the call's inputs, the sums are not
    load(0, u, gm);
    if (!BWD && init_slot >= 0) x = *reinterpret_cast<const float4*>(slots + (size_t)init_slot * stride + el);
    for (int i0 = 0; i0 < n_chunks; i0 += AHEAD) {
        load(i0 + AHEAD, un, gn);
#pragma unroll
        for (int j = 0; j < AHEAD; j++) {
            const int i = i0 + j, c = chunk_of(i);
            if (i >= n_chunks) break;
            if (BWD && boundary == c + 1) {      // gradients of every sequence that started from this boundary, in table order
                for (int q = tb.slot_cons_ptr[req]; q < tb.slot_cons_ptr[req + 1]; q++) {
                    const float4 y = *reinterpret_cast<const float4*>(ds0 + (size_t)tb.slot_cons_seq[q] * stride + el);
                    x.x += y.x, x.y += y.y, x.z += y.z, x.w += y.w;
                }
                req--;
                boundary = req >= req_lo ? tb.slot_chunk[req] : -1;
            }
            // in place: this thread has read the chunk's sum already; backward: zero after the last chunk, not read
            if (!BWD || i > 0) *reinterpret_cast<float4*>(tiles + (size_t)(chunk_base + c) * stride + el) = x;
            if (!BWD && boundary == c) {
                *reinterpret_cast<float4*>(slots + (size_t)req * stride + el) = x;
                req++;
                boundary = req < req_hi ? tb.slot_chunk[req] : -1;
            }
            if (i < n_steps) {
                x.x = __fmaf_rn(gm[j], x.x, u[j].x), x.y = __fmaf_rn(gm[j], x.y, u[j].y);
                x.z = __fmaf_rn(gm[j], x.z, u[j].z), x.w = __fmaf_rn(gm[j], x.w, u[j].w);
            }
        }
#pragma unroll
        for (int j = 0; j < AHEAD; j++) u[j] = un[j], gm[j] = gn[j];
    }
    if (BWD && init_slot >= 0) *reinterpret_cast<float4*>(ds0 + (size_t)seq * stride + el) = x;
}

struct __align__(16) OutSmem {
    float q[TILE], k[TILE], v[TILE], s[TILE], p[TILE];
    Rows rd;
    Item it;
};
template <int R>
__global__ void __launch_bounds__(1024 / R) out_kernel(const harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const float* __restrict__ q,
                                                 const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ g,
                                                 const float* __restrict__ states, float* __restrict__ o, const int32_t* gate) {
    let_next_launch();
    if (gate_closed(gate)) return after_previous();
    bool waited = false;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    OutSmem& s = *reinterpret_cast<OutSmem*>(smem_raw);
    for (int idx = blockIdx.x; begin_item(tb, seq_lo, seq_hi, H, g, idx, s.rd, s.it); idx += gridDim.x) {
    const Item& it = s.it;
    load_tile(s.q, q, s.rd, true, it.h, H);
    load_tile(s.k, k, s.rd, false, it.h, H);
    load_tile(s.v, v, s.rd, false, it.h, H);
    const float* state = states + ((size_t)it.gc * H + it.h) * (D * D);
    if (waited && !it.zero_state) load_state(s.s, state);
    __syncthreads();
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16, warp = threadIdx.x / 32;
    AccT<R> acc;
    clear(acc);
    mul_nt_causal(acc, s.q, s.k, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int t = R * ty + r, j = tx + 16 * c;
            s.p[t * LD + j] = j <= t ? acc[r][c] * s.rd.decay(t, j) : 0.f;
        }
    __syncwarp();                                // a warp reads the rows it wrote
    AccT<R> in;                                      // the chunk's own share, summed by itself: it is small beside the state's
    clear(in);
    mul_nn(in, s.p, s.v, 0, 2 * R * warp, ty, tx);
    mul_nn_diagonal(in, s.p, s.v, 2 * R * warp, ty, tx);
    if (!waited) {                               // so far the call's inputs alone: the first item's share is made while the states are
        after_previous();
        waited = true;
        if (!it.zero_state) load_state(s.s, state);
        __syncthreads();
    }
    clear(acc);
    if (!it.zero_state) mul_nn(acc, s.q, s.s, 0, D, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int code = s.rd.code[R * ty + r];
        if (code >= 0)
#pragma unroll
            for (int c = 0; c < 4; c++)
                o[((size_t)code * H + it.h) * D + tx + 16 * c] = it.zero_state ? in[r][c] : __fmaf_rn(s.rd.eb[R * ty + r], acc[r][c], in[r][c]);
    }
    }
    if (!waited) after_previous();               // no item: the kernel behind this one must not get ahead of the one before it
}

struct __align__(16) GradSmem {
    float q[TILE], k[TILE], v[TILE], dO[TILE], s[TILE], ds[TILE], p[TILE], dp[TILE];
    Rows rd;
    Item it;
    float z[BT], part[16];
};
template <int R>
__global__ void __launch_bounds__(1024 / R, 1) grad_kernel(const harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const float* __restrict__ q,
                                                  const float* __restrict__ k, const float* __restrict__ v, const float* __restrict__ g,
                                                  const float* __restrict__ dO, const float* __restrict__ states,
                                                  const float* __restrict__ ds_tiles, float* __restrict__ dq, float* __restrict__ dk_,
                                                  float* __restrict__ dv_, float* __restrict__ dg, float* __restrict__ rk,
                                                  float* __restrict__ rv, float* __restrict__ rg, const int32_t* gate) {
    let_next_launch();
    if (gate_closed(gate)) return after_previous();
    bool waited = false;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& s = *reinterpret_cast<GradSmem*>(smem_raw);
    for (int idx = blockIdx.x; begin_item(tb, seq_lo, seq_hi, H, g, idx, s.rd, s.it); idx += gridDim.x) {
    const Item& it = s.it;
    const int h = it.h;
    const bool has_s = !it.zero_state, has_ds = !it.last;
    load_tile(s.q, q, s.rd, true, h, H);
    load_tile(s.k, k, s.rd, false, h, H);
    load_tile(s.v, v, s.rd, false, h, H);
    load_tile(s.dO, dO, s.rd, true, h, H);
    const size_t tile = ((size_t)it.gc * H + h) * (D * D);
    if (waited) {
        if (has_s) load_state(s.s, states + tile);
        if (has_ds) load_state(s.ds, ds_tiles + tile);
    }
    __syncthreads();
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16, warp = tid / 32, lane = tid & 31;
    AccT<R> acc, dacc;
    clear(acc);
    clear(dacc);
    mul_nt_causal(acc, s.q, s.k, ty, tx);
    mul_nt_causal(dacc, s.dO, s.v, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int t = R * ty + r, j = tx + 16 * c;
            const float w = j <= t ? s.rd.decay(t, j) : 0.f;
            s.p[t * LD + j] = j <= t ? acc[r][c] * w : 0.f;
            s.dp[t * LD + j] = j <= t ? dacc[r][c] * w : 0.f;
        }
    __syncthreads();
    // the chunk's own shares, by themselves as in out_kernel: of the call's inputs alone, the first item's made while the states are
    AccT<R> own_q, own_k, own_v;
    clear(own_q);
    clear(own_k);
    clear(own_v);
    mul_nn(own_q, s.dp, s.k, 0, 2 * R * warp, ty, tx);
    mul_nn_diagonal(own_q, s.dp, s.k, 2 * R * warp, ty, tx);
    mul_tn_diagonal(own_k, s.dp, s.q, 2 * R * warp, ty, tx);
    mul_tn(own_k, s.dp, s.q, 2 * R * warp + 2 * R, ty, tx);
    mul_tn_diagonal(own_v, s.p, s.dO, 2 * R * warp, ty, tx);
    mul_tn(own_v, s.p, s.dO, 2 * R * warp + 2 * R, ty, tx);
    if (!waited) {
        after_previous();
        waited = true;
        if (has_s) load_state(s.s, states + tile);
        if (has_ds) load_state(s.ds, ds_tiles + tile);
        __syncthreads();
    }
    const float gamma = s.rd.gamma;
    float g_part = 0.f;                          // this thread's share of <S_{c+1}, dS_{c+1}>
    float z[R] = {};           // its share of q.dq - k.dk, per row
    // ---- dq = e^{b_t} dO S^T + dP K
    clear(acc);
    if (has_s) mul_nt<4>(acc, s.dO, s.s, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int t = R * ty + r, code = s.rd.code[t];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const float x = has_s ? __fmaf_rn(s.rd.eb[t], acc[r][c], own_q[r][c]) : own_q[r][c];
            z[r] += s.q[t * LD + tx + 16 * c] * x;
            if (code >= 0) dq[((size_t)code * H + h) * D + tx + 16 * c] = x;
        }
    }
    // ---- dk = w_j V dS^T + dP^T Q
    clear(acc);
    if (has_ds) mul_nt<4>(acc, s.v, s.ds, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int t = R * ty + r, code = s.rd.code[t];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const float kv = s.k[t * LD + tx + 16 * c], inter = has_ds ? acc[r][c] * s.rd.w[t] : 0.f, x = own_k[r][c] + inter;
            g_part += kv * inter;
            z[r] -= kv * x;
            if (code >= 0) dk_[((size_t)code * H + h) * D + tx + 16 * c] = x;
            else if (code < -1) rk[((size_t)(it.replay_base + t) * H + h) * D + tx + 16 * c] = x;
        }
    }
    // ---- dv = w_j K dS + P^T dO
    clear(acc);
    if (has_ds) mul_nn(acc, s.k, s.ds, 0, D, ty, tx);
#pragma unroll
    for (int r = 0; r < R; r++) {
        const int t = R * ty + r, code = s.rd.code[t];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const float x = has_ds ? __fmaf_rn(s.rd.w[t], acc[r][c], own_v[r][c]) : own_v[r][c];
            if (code >= 0) dv_[((size_t)code * H + h) * D + tx + 16 * c] = x;
            else if (code < -1) rv[((size_t)(it.replay_base + t) * H + h) * D + tx + 16 * c] = x;
        }
    }
    // ---- dg_t = sum_{tau>=t} z_tau + e^{b_n} <S_c, dS> + sum_j k_j . (w_j dS v_j), every sum in a fixed order
    if (has_s && has_ds) {
        float dot = 0.f;
        for (int e = tid; e < D * D; e += 1024 / R) dot += s.s[(e >> 6) * LD + (e & 63)] * s.ds[(e >> 6) * LD + (e & 63)];
        g_part += gamma * dot;
    }
#pragma unroll
    for (int o_ = 16; o_ > 0; o_ >>= 1) g_part += __shfl_xor_sync(~0u, g_part, o_);
    if (lane == 0) s.part[warp] = g_part;
#pragma unroll
    for (int r = 0; r < R; r++) {
#pragma unroll
        for (int o_ = 8; o_ > 0; o_ >>= 1) z[r] += __shfl_xor_sync(~0u, z[r], o_);
        if (tx == 0) s.z[R * ty + r] = z[r];
    }
    __syncthreads();
    if (warp == 0) {
        float lo = s.z[lane], hi = s.z[lane + 32], G = 0.f;
#pragma unroll
        for (int o_ = 1; o_ < 32; o_ <<= 1) {
            const float y0 = __shfl_down_sync(~0u, lo, o_), y1 = __shfl_down_sync(~0u, hi, o_);
            if (lane + o_ < 32) {
                lo += y0;
                hi += y1;
            }
        }
        const float half = __shfl_sync(~0u, hi, 0);
#pragma unroll
        for (int w = 0; w < 32 / R; w++) G += s.part[w];
        const float out[2] = {lo + half + G, hi + G};
#pragma unroll
        for (int r = 0; r < 2; r++) {
            const int t = lane + 32 * r, code = s.rd.code[t];
            if (code >= 0) dg[(size_t)code * H + h] = out[r];
            else if (code < -1) rg[(size_t)(it.replay_base + t) * H + h] = out[r];
        }
    }
    }
    if (!waited) after_previous();
}

// A grid no larger than what is resident at once: the number of items of a range is in the tables on the device, and one launch
// per round would otherwise bring the whole forest's CTAs each time.
inline int grid_of(const harts_la_tables_t& tb, int32_t H, int per_sm) {
    const int64_t items = (int64_t)tb.n_chunks * H, most = (int64_t)per_sm * sm_count();
    return (int)(items < most ? items : most);
}
constexpr int OUTER_PER_SM = 5, OUT_PER_SM = 2, GRAD_PER_SM = 1;       // 47 registers a thread; 88 and 140 KB of shared memory

inline int32_t done() { return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA; }

}  // namespace

// Sequences [range[0], range[n]), range[r]..range[r+1] per round.  extra: f32_extra_bytes() behind the chunk states and flags.
int32_t f32_fwd(const FwdArgs& a, float* extra, const int32_t* range, int32_t n) {
    const int lo = range[0], hi = range[n];
    if (lo == hi) return HARTS_OK;
    const int32_t* gate = status_gate(a.flags, a.dev_status);
    float *states = (float*)a.chunk_states, *gammas = extra;
    outer_kernel<false><<<grid_of(a.tb, a.H, OUTER_PER_SM), NT, 0, a.stream>>>(a.tb, lo, hi, a.H, (const float*)a.k, (const float*)a.v, a.g, states, gammas, gate);
    for (int32_t r = 0; r < n; r++)
        if (range[r] < range[r + 1])
            launch_after(walk_kernel<false>, (range[r + 1] - range[r]) * a.H * 4, NT, 0, a.stream, a.tb, range[r], a.H, states, gammas, a.slots, nullptr, gate);
    // an item a CTA: sixteen warps hide its latency (13 items 16.4 -> 13.4 us); more: two CTAs of eight warps an SM, whose 4 x 4 outputs a
    // thread read shared memory less (796 items 55 us, 71 with sixteen)
    auto outputs = [&](auto kernel, int threads) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(OutSmem)) != cudaSuccess) return HARTS_ECUDA;
        launch_after(kernel, grid_of(a.tb, a.H, OUT_PER_SM), threads, sizeof(OutSmem), a.stream, a.tb, lo, hi, a.H, (const float*)a.q, (const float*)a.k,
                     (const float*)a.v, a.g, states, (float*)a.o, gate);
        return done();
    };
    return (int64_t)a.tb.n_chunks * a.H <= sm_count() ? outputs(out_kernel<2>, 512) : outputs(out_kernel<4>, 256);
}

int32_t f32_bwd(const BwdArgs& a, float* extra, const int32_t* range, int32_t n) {
    const int lo = range[0], hi = range[n];
    if (lo == hi) return HARTS_OK;
    const int32_t* gate = status_gate(a.flags, a.dev_status);
    const ScratchLayout sl = scratch_layout(a.tb, a.H, a.dk, a.dv);
    char* base = static_cast<char*>(a.scratch);
    float *gammas = extra, *tiles = extra + align_up((size_t)a.tb.n_chunks * a.H, 64), *ds0 = (float*)(base + sl.ds0);
    outer_kernel<true><<<grid_of(a.tb, a.H, OUTER_PER_SM), NT, 0, a.stream>>>(a.tb, lo, hi, a.H, (const float*)a.q, (const float*)a.dO, a.g, tiles, gammas, gate);
    for (int32_t r = n - 1; r >= 0; r--)
        if (range[r] < range[r + 1])
            launch_after(walk_kernel<true>, (range[r + 1] - range[r]) * a.H * 4, NT, 0, a.stream, a.tb, range[r], a.H, tiles, gammas, nullptr, ds0, gate);
    if (cudaFuncSetAttribute(grad_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(GradSmem)) != cudaSuccess) return HARTS_ECUDA;
    launch_after(grad_kernel<2>, grid_of(a.tb, a.H, GRAD_PER_SM), 512, sizeof(GradSmem), a.stream,
        a.tb, lo, hi, a.H, (const float*)a.q, (const float*)a.k, (const float*)a.v, a.g, (const float*)a.dO, (const float*)a.chunk_states,
        tiles, (float*)a.dq, (float*)a.dk_, (float*)a.dv_, a.dg, (float*)(base + sl.rk), (float*)(base + sl.rv), (float*)(base + sl.rg), gate);
    return done();
}

}  // namespace harts
