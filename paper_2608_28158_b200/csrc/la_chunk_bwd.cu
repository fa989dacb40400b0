// Gradients of the chunk-parallel backward (bf16, d_k = d_v = 128, chunk 64): with the state at the start of every chunk
// and its gradient at the end of every chunk in memory (la_scan.cu), each (chunk, head) is a work item of its own.
//     A  = Q K^T,  dA = dO V^T                        P = A .* D, dP = dA .* D   (D_tj = e^{b_t-b_j} [j<=t])
//     dq = dP K   + e^{b_t} (dO S^T)
//     dk = dP^T Q + w_j (V dS^T)                      w_j = e^{b_n-b_j}
//     dv = P^T dO + w_j (K dS)
//     dg_t = sum_{tau>=t} (q.dq - k.dk) + e^{b_n} <S, dS> + sum_j k_j . (w_j dS v_j)        <S, dS>: from the scan, where dS is fp32
// tcgen05 MMAs, every product transposed (tensor-memory lane = feature, column = row of the chunk); the 24 MMAs of the
// three state products do not need P or dP and run under the decay masking, so twelve are left after it.  One CTA per SM:
// eight 64-column accumulators take all 512 tensor-memory columns, tiles and staging 198 KB of shared memory.  Sixteen
// compute warps, one warp that issues every TMA (first lane) and MMA (an elected lane), one that prepares the next items and finishes dg.
// The dS of a sequence's last chunk and the state of a sequence that starts from zero are zero: not read, not multiplied.
// What bounds it: the dependent phases of one item (4.5 us; 178 KB of traffic would take 4.0): 0.77 ms for 1,595 chunks x 16
// heads (0.80 with the MMAs issued by the first lane).  Every wait is bounded.
#include "chunk_item.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int32_t make_state_map(CUtensorMap* map, const void* base, int64_t n);
int sm_count();

namespace {

using namespace tc;
using namespace chunk;

constexpr int NC = 512, NT = NC + 64;
constexpr int TILE = BT * D * 2, S_PANEL = D * 128;
constexpr int COL_A = 0, COL_DA = 64, COL_DQ = 128, COL_DQE = 192, COL_DK = 256, COL_DKE = 320, COL_DV = 384, COL_DVE = 448,
              TMEM_COLS = 512;

struct Smem {
    // dO directly after another tile: its MMA operand starts one panel early (rows 64..127 of the operand are dO)
    static constexpr int q = 0, k = TILE, v = 2 * TILE, dO = 3 * TILE, p = 4 * TILE, dp = p + PANEL, s = dp + PANEL,
                         ds = s + 2 * S_PANEL, stage_dq = ds + 2 * S_PANEL, stage_dk = stage_dq + TILE,
                         stage_dv = stage_dk + TILE, misc = stage_dv + TILE, bytes = misc + 6144;
};
struct Misc {
    RowData rows[3];
    Item items[3];
    float red[NC / 32][16];  // per-warp partial sums of q.dq - k.dk (warp w covers rows 16(w>>2)..+15)
    float gred[NC / 32];
    uint32_t tmem;
    uint64_t bar_tiles, bar_states, bar_a, bar_o, bar_o2, bar_o3, bar_qk_read, bar_exit;
    int dead;
};
static_assert(sizeof(Misc) <= 6144, "misc area");

// fragment register r of load l (l = 0: lanes +0, l = 1: lanes +16) -> its bf16 value in q / k fragments [ta][fa]
__device__ __forceinline__ float frag_elem(const uint32_t (&f)[2][4], int l, int r) {
    const uint32_t pair = f[r >> 2][2 * l + ((r >> 1) & 1)];
    return __uint_as_float((r & 1) ? (pair & 0xffff0000u) : (pair << 16));
}
__device__ __forceinline__ void load_acc(uint32_t tm_lane, int col, uint32_t (&x)[2][8]) {
#pragma unroll
    for (int l = 0; l < 2; l++) tmem_ld_frag16(tm_lane + ((uint32_t)(16 * l) << 16) + col, x[l]);
}

__global__ void __launch_bounds__(NT, 1)
chunk_bwd_kernel(const harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const __grid_constant__ CUtensorMap map_q,
                 const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const __grid_constant__ CUtensorMap map_do, const __grid_constant__ CUtensorMap map_s,
                 const __grid_constant__ CUtensorMap map_ds, const __grid_constant__ CUtensorMap map_dq,
                 const __grid_constant__ CUtensorMap map_dk, const __grid_constant__ CUtensorMap map_dv,
                 const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                 const float* __restrict__ g, const __nv_bfloat16* __restrict__ dO, __nv_bfloat16* __restrict__ dq,
                 __nv_bfloat16* __restrict__ dk_, __nv_bfloat16* __restrict__ dv_, float* __restrict__ dg,
                 float* __restrict__ rk, float* __restrict__ rv, float* __restrict__ rg, const float* __restrict__ dots,
                 int* status, const int32_t* gate) {
    after_previous();
    if (gate_closed(gate)) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *sQ = smem + Smem::q, *sK = smem + Smem::k, *sV = smem + Smem::v, *sDO = smem + Smem::dO, *sP = smem + Smem::p,
                  *sDP = smem + Smem::dp, *sS = smem + Smem::s, *sDS = smem + Smem::ds;
    Misc& m = *reinterpret_cast<Misc*>(smem + Smem::misc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool is_compute = warp < NC / 32, is_issuer = tid == NC, is_mma = warp == NC / 32, is_aux = warp == NC / 32 + 1;
    const int grp = warp >> 2, L = (warp & 3) * 32 + lane;

    const int chunk_lo = tb.seq_chunk_ptr[seq_lo], n_items = (tb.seq_chunk_ptr[seq_hi] - chunk_lo) * H;
    const int G = gridDim.x, n_mine = (int)blockIdx.x < n_items ? (n_items - 1 - (int)blockIdx.x) / G + 1 : 0;
    auto item_at = [&](int i) {
        const int idx = (int)blockIdx.x + i * G;
        return find_item(tb, seq_lo, seq_hi, chunk_lo + idx / H, idx % H, lane);
    };

    if (tid == 0) {
        mbar_init(&m.bar_tiles, 1);
        mbar_init(&m.bar_states, 1);
        mbar_init(&m.bar_a, 1);
        mbar_init(&m.bar_o, 1);
        mbar_init(&m.bar_o2, 1);
        mbar_init(&m.bar_o3, 1);
        mbar_init(&m.bar_qk_read, NC / 32);
        mbar_init(&m.bar_exit, 1);
        m.dead = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc<TMEM_COLS>(&m.tmem);
    int nx_code[2];
    float nx_g[2];
    if (is_aux && n_mine > 0) {
        Item it = item_at(0);
        load_rows(tb, it, g, H, lane, nx_code, nx_g);
        if (lane == 0) m.items[0] = it;
        store_rows(m.rows[0], nx_code, nx_g, lane);
        if (n_mine > 1) {
            it = item_at(1);
            load_rows(tb, it, g, H, lane, nx_code, nx_g);
            if (lane == 0) m.items[1] = it;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = m.tmem, tm_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);

    const uint32_t aQ = smem_u32(sQ), aK = smem_u32(sK), aV = smem_u32(sV), aDO = smem_u32(sDO), aP = smem_u32(sP),
                   aDP = smem_u32(sDP), aS = smem_u32(sS), aDS = smem_u32(sDS);
    constexpr uint32_t I_KK64 = instr_desc(128, 64, 0, 0), I_MK64 = instr_desc(128, 64, 1, 0), I_MM64 = instr_desc(128, 64, 1, 1);
    // operand descriptors at k-step 0: "k" = contraction dimension contiguous, "m" = the other one
    const uint64_t dQk = desc_kmajor_base(aQ), dKk = desc_kmajor_base(aK), dVk = desc_kmajor_base(aV), dDOk = desc_kmajor_base(aDO),
                   dDOk_hi = desc_kmajor_base(aDO - PANEL), dDPk = desc_kmajor_base(aDP), dDSk = desc_kmajor_base(aDS),
                   dSk = desc_kmajor_base(aS);
    const uint64_t dQm = desc_mnmajor_base<BT>(aQ), dKm = desc_mnmajor_base<BT>(aK), dDOm = desc_mnmajor_base<BT>(aDO),
                   dPm = desc_mnmajor_base<BT>(aP), dDPm = desc_mnmajor_base<BT>(aDP), dDSm = desc_mnmajor_base<D>(aDS);

    auto issue_tiles = [&](const Item& it) {
        const bool rows = !it.gathered();
        mbar_expect_tx(&m.bar_tiles, rows ? 4 * TILE : 0);
        if (rows)
            for (int p = 0; p < 2; p++) {
                tma_load_3d(sQ + p * PANEL, &map_q, p * 64, it.h, it.row0, &m.bar_tiles);
                tma_load_3d(sK + p * PANEL, &map_k, p * 64, it.h, it.row0, &m.bar_tiles);
                tma_load_3d(sDO + p * PANEL, &map_do, p * 64, it.h, it.row0, &m.bar_tiles);
                tma_load_3d(sV + p * PANEL, &map_v, p * 64, it.h, it.row0, &m.bar_tiles);
            }
        mbar_expect_tx(&m.bar_states, (it.zero_state ? 0 : 2 * S_PANEL) + (it.last ? 0 : 2 * S_PANEL));
        for (int p = 0; p < 2; p++) {
            if (!it.last) tma_load_3d(sDS + p * S_PANEL, &map_ds, p * 64, 0, it.gc * H + it.h, &m.bar_states);
            if (!it.zero_state) tma_load_3d(sS + p * S_PANEL, &map_s, p * 64, 0, it.gc * H + it.h, &m.bar_states);
        }
    };
    bool tiles_pending = false, gave_up = false;      // tiles_pending is kept by the issuing thread only
    if (is_issuer && n_mine > 0) {
        issue_tiles(m.items[0]);
        tiles_pending = true;
    }

    uint32_t ph = 0;
    for (int i = 0; i < n_mine; i++, ph ^= 1) {
        const Item& it = m.items[i % 3];
        const RowData& rd = m.rows[i % 3];
        const bool gathered = it.gathered(), full = it.full(), has_s = !it.zero_state, has_ds = !it.last;
        const int h = it.h, row0 = it.row0, replay_base = it.replay_base;
        if (gathered) {
            for (int e = tid; e < BT * 16; e += NT) {
                const int row = e >> 4, ch = e & 15, code = rd.code[row];
                uint4 kq = make_uint4(0, 0, 0, 0), vq = kq, qq = kq, oq = kq;
                if (code != -1) {
                    const size_t off = ((size_t)(code >= 0 ? code : -2 - code) * H + h) * D + ch * 8;
                    kq = *reinterpret_cast<const uint4*>(k + off);
                    vq = *reinterpret_cast<const uint4*>(v + off);
                    if (code >= 0) {
                        qq = *reinterpret_cast<const uint4*>(q + off);
                        oq = *reinterpret_cast<const uint4*>(dO + off);
                    }
                }
                const uint32_t dst = (ch >> 3) * PANEL + sw128_chunk(row, ch & 7);
                *reinterpret_cast<uint4*>(sQ + dst) = qq;
                *reinterpret_cast<uint4*>(sK + dst) = kq;
                *reinterpret_cast<uint4*>(sV + dst) = vq;
                *reinterpret_cast<uint4*>(sDO + dst) = oq;
            }
            fence_async_smem();
            __syncthreads();
        }
        if (is_mma) {                      // an elected lane issues (4,696 chunks x 32 heads, walk and chunk kernels: 5.81 -> 5.55 ms)
            bool ok = mbar_wait_warp(&m.bar_tiles, ph, status, &m.dead);
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 8; ks++) mma_ss(tmem + COL_A, dQk + kstep_kmajor<BT>(ks), dKk + kstep_kmajor<BT>(ks), I_KK64, ks > 0);
#pragma unroll
                for (int ks = 0; ks < 8; ks++)
                    mma_ss(tmem + COL_DA, dDOk_hi + kstep_kmajor<BT>(ks), dVk + kstep_kmajor<BT>(ks), I_KK64, ks > 0);
                mma_commit(&m.bar_a);
            }
            __syncwarp();
            ok = mbar_wait_warp(&m.bar_states, ph, status, &m.dead) && ok;
            if (ok) tiles_pending = false;
            tc_fence_after();
            if (elect_one()) {
                if (has_ds) {
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)       // dS V^T
                        mma_ss(tmem + COL_DKE, dDSk + kstep_kmajor<D>(ks), dVk + kstep_kmajor<BT>(ks), I_KK64, ks > 0);
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)       // dS^T K^T
                        mma_ss(tmem + COL_DVE, dDSm + kstep_mnmajor(ks), dKk + kstep_kmajor<BT>(ks), I_MK64, ks > 0);
                }
                if (has_s)
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)       // S dO^T
                        mma_ss(tmem + COL_DQE, dSk + kstep_kmajor<D>(ks), dDOk + kstep_kmajor<BT>(ks), I_KK64, ks > 0);
            }
            __syncwarp();
            if (is_issuer) tma_store_wait_read();     // the previous item's outputs have left the staging tiles
        }
        if (is_aux && i + 1 < n_mine) store_rows(m.rows[(i + 1) % 3], nx_code, nx_g, lane);
        float g_part = 0.f;                // this thread's share of <S_{c+1}, dS_{c+1}>
        if (is_compute) {
            if (has_s && has_ds) g_part = dots[((size_t)it.gc * H + h) * NC + tid];      // <S, dS>, one of its 512 parts per thread
            // ---- P (lanes 0..63), dP (lanes 64..127): 16 columns of one of them per thread --------------------------------
            mbar_wait(&m.bar_a, ph, status, &m.dead);
            tc_fence_after();
            const bool is_p = (warp & 3) < 2;
            const int t = L & 63;
            unsigned char* dst = is_p ? sP : sDP;
            if (grp * 16 > (warp & 1) * 32 + 31) {       // this warp's 32 rows x 16 columns lie entirely above the diagonal
                *reinterpret_cast<uint4*>(dst + sw128_chunk(t, grp * 2)) = make_uint4(0, 0, 0, 0);
                *reinterpret_cast<uint4*>(dst + sw128_chunk(t, grp * 2 + 1)) = make_uint4(0, 0, 0, 0);
            } else {
                const float bt = rd.b2[t];
                const int limit = rd.code[t] >= 0 ? t : -1;      // replay rows and rows past the end have no dO and no q
                uint32_t xa[16];
                tmem_ld16(tm_lane + (is_p ? COL_A : COL_DA) + grp * 16, xa);
                float bj[16];
#pragma unroll
                for (int u = 0; u < 4; u++)
                    *reinterpret_cast<float4*>(bj + 4 * u) = *reinterpret_cast<const float4*>(rd.b2 + grp * 16 + 4 * u);
                tmem_ld_wait();
#pragma unroll
                for (int v4 = 0; v4 < 2; v4++) {
                    float y[8];
#pragma unroll
                    for (int e = 0; e < 8; e++) {
                        const float p = __uint_as_float(xa[v4 * 8 + e]) * ex2(bt - bj[v4 * 8 + e]);
                        y[e] = grp * 16 + v4 * 8 + e <= limit ? p : 0.f;   // a select: the product may be inf or NaN above the diagonal
                    }
                    *reinterpret_cast<uint4*>(dst + sw128_chunk(t, grp * 2 + v4)) =
                        make_uint4(pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]), pack_bf16(y[6], y[7]));
                }
            }
            fence_async_smem();
        }
        tc_fence_before();
        __syncthreads();                   // (A) P and dP are in place, the staging tiles are free, the next record is visible
        tc_fence_after();
        if (is_mma) {
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 4; ks++) mma_ss(tmem + COL_DK, dQm + kstep_mnmajor(ks), dDPm + kstep_mnmajor(ks), I_MM64, ks > 0);
                mma_commit(&m.bar_o);
#pragma unroll
                for (int ks = 0; ks < 4; ks++) mma_ss(tmem + COL_DV, dDOm + kstep_mnmajor(ks), dPm + kstep_mnmajor(ks), I_MM64, ks > 0);
                mma_commit(&m.bar_o2);
#pragma unroll
                for (int ks = 0; ks < 4; ks++) mma_ss(tmem + COL_DQ, dKm + kstep_mnmajor(ks), dDPk + kstep_kmajor<BT>(ks), I_MK64, ks > 0);
                mma_commit(&m.bar_o3);
            }
            __syncwarp();
        }
        if (is_issuer) {
            mbar_wait(&m.bar_o3, ph, status, &m.dead);
            mbar_wait(&m.bar_qk_read, ph, status, &m.dead);      // the compute warps have taken their q and k values
            if (i + 1 < n_mine) {
                issue_tiles(m.items[(i + 1) % 3]);
                tiles_pending = true;
            }
        }
        if (is_aux && i + 2 < n_mine) {
            const Item nx = item_at(i + 2);
            load_rows(tb, nx, g, H, lane, nx_code, nx_g);
            if (lane == 0) m.items[(i + 2) % 3] = nx;
        }
        if (is_compute) {
            mbar_wait(&m.bar_tiles, ph, status, &m.dead);        // long complete: orders this thread's reads of the tiles
            const int c4 = lane & 3, mrow = lane >> 2, Lq = (warp & 3) * 32, t0 = grp * 16;
            uint32_t fq[2][4], fk[2][4];
#pragma unroll
            for (int ta = 0; ta < 2; ta++) {
                ldmatrix_x4_trans(frag_addr(aQ, lane, Lq, t0, ta), fq[ta]);
                ldmatrix_x4_trans(frag_addr(aK, lane, Lq, t0, ta), fk[ta]);
            }
            g_part *= rd.gamma;
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.bar_qk_read);
            // this thread's four rows: t0 + 2c, +1, t0 + 8 + 2c, +1
            float wv[4], ev[4];
            int code[4];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                *reinterpret_cast<float2*>(wv + 2 * u) = *reinterpret_cast<const float2*>(rd.w + t0 + 8 * u + 2 * c4);
                *reinterpret_cast<float2*>(ev + 2 * u) = *reinterpret_cast<const float2*>(rd.eb + t0 + 8 * u + 2 * c4);
                *reinterpret_cast<int2*>(code + 2 * u) = *reinterpret_cast<const int2*>(rd.code + t0 + 8 * u + 2 * c4);
            }
            // replayed rows keep fp32 and go to the scratch straight from the fragments (eight lanes = one 32-byte piece)
            auto replay_store = [&](float* dst, const float (&val)[2][8]) {
#pragma unroll
                for (int l = 0; l < 2; l++)
#pragma unroll
                    for (int r = 0; r < 8; r++) {
                        const int ti = 2 * (r >> 2) + (r & 1), t = t0 + 8 * (r >> 2) + 2 * c4 + (r & 1);
                        if (code[ti] < -1)
                            dst[((size_t)(replay_base + t) * H + h) * D + Lq + 16 * l + 8 * ((r >> 1) & 1) + mrow] = val[l][r];
                    }
            };
            float zf[4] = {0.f, 0.f, 0.f, 0.f};              // q.dq - k.dk over this thread's features, per row
            float val[2][8];
            uint32_t xi[2][8], xe[2][8];
            // ---- dk ---------------------------------------------------------------------------------------------------------
            mbar_wait(&m.bar_o, ph, status, &m.dead);
            tc_fence_after();
            load_acc(tm_lane, COL_DK + t0, xi);
            load_acc(tm_lane, COL_DKE + t0, xe);
            tmem_ld_wait();
#pragma unroll
            for (int l = 0; l < 2; l++)
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int ti = 2 * (r >> 2) + (r & 1);
                    const float kv = frag_elem(fk, l, r);
                    const float inter = has_ds ? wv[ti] * __uint_as_float(xe[l][r]) : 0.f;
                    const float dkv = __uint_as_float(xi[l][r]) + inter;
                    const bool ok = code[ti] != -1;
                    zf[ti] -= ok ? kv * dkv : 0.f;
                    g_part += ok ? kv * inter : 0.f;
                    val[l][r] = dkv;
                }
            frag_store(smem_u32(smem + Smem::stage_dk), lane, Lq, t0, val);
            if (gathered) replay_store(rk, val);
#pragma unroll
            for (int o_ = 16; o_ > 0; o_ >>= 1) g_part += __shfl_xor_sync(0xffffffffu, g_part, o_);
            if (lane == 0) m.gred[warp] = g_part;
            // ---- dv ---------------------------------------------------------------------------------------------------------
            mbar_wait(&m.bar_o2, ph, status, &m.dead);
            tc_fence_after();
            load_acc(tm_lane, COL_DV + t0, xi);
            load_acc(tm_lane, COL_DVE + t0, xe);
            tmem_ld_wait();
#pragma unroll
            for (int l = 0; l < 2; l++)
#pragma unroll
                for (int r = 0; r < 8; r++)
                    val[l][r] = __uint_as_float(xi[l][r]) + (has_ds ? wv[2 * (r >> 2) + (r & 1)] * __uint_as_float(xe[l][r]) : 0.f);
            frag_store(smem_u32(smem + Smem::stage_dv), lane, Lq, t0, val);
            if (gathered) replay_store(rv, val);
            // ---- dq ---------------------------------------------------------------------------------------------------------
            mbar_wait(&m.bar_o3, ph, status, &m.dead);
            tc_fence_after();
            load_acc(tm_lane, COL_DQ + t0, xi);
            load_acc(tm_lane, COL_DQE + t0, xe);
            tmem_ld_wait();
#pragma unroll
            for (int l = 0; l < 2; l++)
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int ti = 2 * (r >> 2) + (r & 1);
                    const float dqv = __uint_as_float(xi[l][r]) + (has_s ? ev[ti] * __uint_as_float(xe[l][r]) : 0.f);
                    zf[ti] += code[ti] >= 0 ? frag_elem(fq, l, r) * dqv : 0.f;
                    val[l][r] = dqv;
                }
            frag_store(smem_u32(smem + Smem::stage_dq), lane, Lq, t0, val);
            // rows are shared by the eight threads with the same c: sum over them, then one writer per row
#pragma unroll
            for (int u = 0; u < 4; u++) {
                zf[u] += __shfl_xor_sync(0xffffffffu, zf[u], 4);
                zf[u] += __shfl_xor_sync(0xffffffffu, zf[u], 8);
                zf[u] += __shfl_xor_sync(0xffffffffu, zf[u], 16);
            }
            if (lane < 4) {
                m.red[warp][2 * c4] = zf[0];
                m.red[warp][2 * c4 + 1] = zf[1];
                m.red[warp][8 + 2 * c4] = zf[2];
                m.red[warp][8 + 2 * c4 + 1] = zf[3];
            }
            if (full) fence_async_smem();
        }
        tc_fence_before();
        gave_up = __syncthreads_or(m.dead) != 0;      // (B) staged outputs and partial sums complete, tensor memory read
        tc_fence_after();
        if (gave_up) break;
        if (full) {
            if (is_issuer) {
                for (int p = 0; p < 2; p++) {
                    tma_store_3d(&map_dk, smem + Smem::stage_dk + p * PANEL, p * 64, h, row0);
                    tma_store_3d(&map_dv, smem + Smem::stage_dv + p * PANEL, p * 64, h, row0);
                    tma_store_3d(&map_dq, smem + Smem::stage_dq + p * PANEL, p * 64, h, row0);
                }
                tma_store_commit();
            }
        } else if (is_compute) {           // own rows only, 16 bytes at a time
            for (int e = tid; e < BT * 16 * 3; e += NC) {
                const int which = e / (BT * 16), t = (e >> 4) & 63, ch = e & 15, code = rd.code[t];
                if (code < 0) continue;
                __nv_bfloat16* out = which == 0 ? dq : (which == 1 ? dk_ : dv_);
                *reinterpret_cast<uint4*>(out + ((size_t)code * H + h) * D + ch * 8) = *reinterpret_cast<const uint4*>(
                    smem + Smem::stage_dq + which * TILE + (ch >> 3) * PANEL + sw128_chunk(t, ch & 7));
            }
        }
        if (is_aux) {
            // dg_t = sum_{tau >= t} r_tau + <S_{c+1}, dS_{c+1}>, rows `lane` and `lane + 32`
            auto row_sum = [&](int t) {
                const int g4 = (t >> 4) * 4, e = t & 15;
                return m.red[g4][e] + m.red[g4 + 1][e] + m.red[g4 + 2][e] + m.red[g4 + 3][e];
            };
            float lo = row_sum(lane), hi = row_sum(lane + 32);
#pragma unroll
            for (int o_ = 1; o_ < 32; o_ <<= 1) {
                const float y0 = __shfl_down_sync(0xffffffffu, lo, o_), y1 = __shfl_down_sync(0xffffffffu, hi, o_);
                if (lane + o_ < 32) {
                    lo += y0;
                    hi += y1;
                }
            }
            const float G32 = __shfl_sync(0xffffffffu, hi, 0);     // total of rows 32..63
            float Gs = 0.f;
#pragma unroll
            for (int w_ = 0; w_ < NC / 32; w_++) Gs += m.gred[w_];
            const float out[2] = {lo + G32 + Gs, hi + Gs};
#pragma unroll
            for (int r = 0; r < 2; r++) {
                const int t = lane + 32 * r, code = rd.code[t];
                if (code >= 0) dg[(size_t)code * H + h] = out[r];
                else if (code < -1) rg[(size_t)(replay_base + t) * H + h] = out[r];
            }
        }
    }
    if (__syncthreads_or(m.dead) && is_mma) {         // abandoned: let copies and MMAs in flight finish (bounded)
        if (is_issuer && tiles_pending) drain_delay();
        __syncwarp();
        if (elect_one()) {
            mma_commit(&m.bar_exit);
            mbar_wait_drain(&m.bar_exit, 0);
        }
    }
    if (is_issuer) tma_store_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc<TMEM_COLS>(tmem);
}

}  // namespace

// Gradients of the chunks of sequences [seq_lo, seq_hi); states in a.chunk_states, their gradients in ds_tiles, <S, dS> in dots.
int32_t chunk_bwd(const BwdArgs& a, const void* ds_tiles, const float* dots) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    CUtensorMap mq, mk, mv, mdo, ms, mds, mdq, mdk, mdv;
    int32_t rc;
    if ((rc = make_row_map(&mq, a.q, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mk, a.k, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mv, a.v, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdo, a.dO, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_state_map(&ms, a.chunk_states, (int64_t)a.tb.n_chunks * a.H)) != HARTS_OK) return rc;
    if ((rc = make_state_map(&mds, ds_tiles, (int64_t)a.tb.n_chunks * a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdq, a.dq, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdk, a.dk_, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdv, a.dv_, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(chunk_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem::bytes + 1024) != cudaSuccess)
        return HARTS_ECUDA;
    const ScratchLayout sl = scratch_layout(a.tb, a.H, a.dk, a.dv);
    char* base = static_cast<char*>(a.scratch);
    const int64_t n = (int64_t)a.tb.n_chunks * a.H;
    const int grid = (int)(n < sm_count() ? n : sm_count());
    launch_after(chunk_bwd_kernel, grid, NT, Smem::bytes + 1024, a.stream,
        a.tb, a.seq_lo, a.seq_hi, a.H, mq, mk, mv, mdo, ms, mds, mdq, mdk, mdv, (const __nv_bfloat16*)a.q,
        (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.g, (const __nv_bfloat16*)a.dO, (__nv_bfloat16*)a.dq,
        (__nv_bfloat16*)a.dk_, (__nv_bfloat16*)a.dv_, a.dg, (float*)(base + sl.rk), (float*)(base + sl.rv),
        (float*)(base + sl.rg), dots, a.dev_status, status_gate(a.flags, a.dev_status));
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
