// Outputs of the chunk-parallel forward (bf16, d_k = d_v = 128, chunk 64): with the state at the start of every chunk in
// memory (la_scan.cu) each (chunk, head) is a work item of its own.
//     A = Q K^T    P = A .* e^{b_t-b_j} [j<=t]    o_t = P V + e^{b_t} Q S_c
// tcgen05 MMAs with accumulators in tensor memory (O^T: lane = feature, column = row of the chunk); q, k, v and the
// state tile arrive by TMA.  Two CTAs per SM (106 KB of shared memory, 256 tensor-memory columns each), 8 compute warps,
// one warp that issues every TMA (first lane) and MMA (an elected lane), one that prepares the next items (record, gates, row ids).  The
// state's product does not need P, so it runs under the decay masking; only four MMAs are left after it.
// What bounds it: 96 KB of traffic per item (80 read, 16 written); 1,047 chunks x 16 heads take 0.25 ms = 6.6 TB/s.
// Every wait is bounded.
#include "chunk_item.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int32_t make_state_map(CUtensorMap* map, const void* base, int64_t n);
int sm_count();

namespace {

using namespace tc;
using namespace chunk;

constexpr int NC = 256, NT = NC + 64;
constexpr int TILE = BT * D * 2, S_PANEL = D * 128;
constexpr int COL_A = 0, COL_O1 = 64, COL_O2 = 128, TMEM_COLS = 256;

struct Smem {
    static constexpr int q = 0, k = TILE, v = 2 * TILE, p = 3 * TILE, s = p + PANEL, stage = s + 2 * S_PANEL,
                         misc = stage + TILE, bytes = misc + 4096;
};
struct Misc {
    RowData rows[3];
    Item items[3];
    uint32_t tmem;
    uint64_t bar_tiles, bar_a, bar_o, bar_exit;
    int dead;
};
static_assert(sizeof(Misc) <= 4096, "misc area");

__global__ void __launch_bounds__(NT, 2)
chunk_fwd_kernel(const harts_la_tables_t tb, int seq_lo, int seq_hi, int H, const __grid_constant__ CUtensorMap map_q,
                 const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                 const __grid_constant__ CUtensorMap map_cs, const __grid_constant__ CUtensorMap map_o,
                 const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
                 const __nv_bfloat16* __restrict__ v, const float* __restrict__ g, __nv_bfloat16* __restrict__ o,
                 int* status, const int32_t* gate) {
    after_previous();
    if (gate_closed(gate)) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *sQ = smem + Smem::q, *sK = smem + Smem::k, *sV = smem + Smem::v, *sP = smem + Smem::p, *sS = smem + Smem::s,
                  *sO = smem + Smem::stage;
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
        mbar_init(&m.bar_a, 1);
        mbar_init(&m.bar_o, 1);
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

    const uint32_t aQ = smem_u32(sQ), aK = smem_u32(sK), aV = smem_u32(sV), aP = smem_u32(sP), aS = smem_u32(sS), aO = smem_u32(sO);
    const uint64_t dQk = desc_kmajor_base(aQ), dKk = desc_kmajor_base(aK), dPk = desc_kmajor_base(aP);
    const uint64_t dVm = desc_mnmajor_base<BT>(aV), dSm = desc_mnmajor_base<D>(aS);
    constexpr uint32_t IDESC_A = instr_desc(128, 64, 0, 0);    // Q x K, both K-major (rows 64..127 of A unused)
    constexpr uint32_t IDESC_O = instr_desc(128, 64, 1, 0);    // V^T x P, S^T x Q

    auto issue_tiles = [&](const Item& it) {
        const bool rows = !it.gathered();
        mbar_expect_tx(&m.bar_tiles, (rows ? 3 * TILE : 0) + (it.zero_state ? 0 : 2 * S_PANEL));
        if (rows)
            for (int p = 0; p < 2; p++) {
                tma_load_3d(sQ + p * PANEL, &map_q, p * 64, it.h, it.row0, &m.bar_tiles);
                tma_load_3d(sK + p * PANEL, &map_k, p * 64, it.h, it.row0, &m.bar_tiles);
            }
        if (!it.zero_state)
            for (int p = 0; p < 2; p++) tma_load_3d(sS + p * S_PANEL, &map_cs, p * 64, 0, it.gc * H + it.h, &m.bar_tiles);
        if (rows)
            for (int p = 0; p < 2; p++) tma_load_3d(sV + p * PANEL, &map_v, p * 64, it.h, it.row0, &m.bar_tiles);
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
        const bool full = it.full(), zero_state = it.zero_state;
        const int h = it.h, row0 = it.row0;
        if (it.gathered()) {               // replayed rows: gathered row by row (they may come from several segments)
            for (int e = tid; e < BT * 16; e += NT) {
                const int row = e >> 4, ch = e & 15, code = rd.code[row];
                uint4 kq = make_uint4(0, 0, 0, 0), vq = kq, qq = kq;
                if (code != -1) {
                    const size_t off = ((size_t)(code >= 0 ? code : -2 - code) * H + h) * D + ch * 8;
                    kq = *reinterpret_cast<const uint4*>(k + off);
                    vq = *reinterpret_cast<const uint4*>(v + off);
                    if (code >= 0) qq = *reinterpret_cast<const uint4*>(q + off);
                }
                const uint32_t dst = (ch >> 3) * PANEL + sw128_chunk(row, ch & 7);
                *reinterpret_cast<uint4*>(sQ + dst) = qq;
                *reinterpret_cast<uint4*>(sK + dst) = kq;
                *reinterpret_cast<uint4*>(sV + dst) = vq;
            }
            fence_async_smem();
            __syncthreads();
        }
        if (is_mma) {                      // an elected lane issues
            if (mbar_wait_warp(&m.bar_tiles, ph, status, &m.dead)) tiles_pending = false;
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 8; ks++) mma_ss(tmem + COL_A, dQk + kstep_kmajor<BT>(ks), dKk + kstep_kmajor<BT>(ks), IDESC_A, ks > 0);
                mma_commit(&m.bar_a);
                if (!zero_state)
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)
                        mma_ss(tmem + COL_O2, dSm + kstep_mnmajor(ks), dQk + kstep_kmajor<BT>(ks), IDESC_O, ks > 0);
            }
            __syncwarp();
            if (is_issuer) tma_store_wait_read();     // the previous item's outputs have left the staging tile
        }
        if (is_aux && i + 1 < n_mine) store_rows(m.rows[(i + 1) % 3], nx_code, nx_g, lane);
        if (is_compute && (warp & 3) < 2) {           // P = A .* decay: lanes 0..63 hold the rows
            mbar_wait(&m.bar_a, ph, status, &m.dead);
            tc_fence_after();
            const int t = L, j0 = grp * 32;
            const float bt = rd.b2[t];
            uint32_t x[32];
            tmem_ld32(tm_lane + COL_A + j0, x);
            tmem_ld_wait();
#pragma unroll
            for (int v4 = 0; v4 < 4; v4++) {
                float bj[8], y[8];
                *reinterpret_cast<float4*>(bj) = *reinterpret_cast<const float4*>(rd.b2 + j0 + v4 * 8);
                *reinterpret_cast<float4*>(bj + 4) = *reinterpret_cast<const float4*>(rd.b2 + j0 + v4 * 8 + 4);
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const float p = __uint_as_float(x[v4 * 8 + e]) * ex2(bt - bj[e]);
                    y[e] = j0 + v4 * 8 + e <= t ? p : 0.f;       // a select: above the diagonal the product may be inf or NaN
                }
                *reinterpret_cast<uint4*>(sP + sw128_chunk(t, grp * 4 + v4)) =
                    make_uint4(pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]), pack_bf16(y[6], y[7]));
            }
            fence_async_smem();
        }
        tc_fence_before();
        __syncthreads();                   // (A) P is in place, the staging tile is free, the next record is visible
        tc_fence_after();
        if (is_mma) {
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 4; ks++)
                    mma_ss(tmem + COL_O1, dVm + kstep_mnmajor(ks), dPk + kstep_kmajor<BT>(ks), IDESC_O, ks > 0);
                mma_commit(&m.bar_o);
            }
            __syncwarp();
        }
        if (is_issuer) {
            mbar_wait(&m.bar_o, ph, status, &m.dead);
            if (i + 1 < n_mine) {          // every MMA that read the tiles is done
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
            mbar_wait(&m.bar_o, ph, status, &m.dead);
            tc_fence_after();
            const int Lq = (warp & 3) * 32, c4 = lane & 3;
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                const int t0 = grp * 32 + hf * 16;
                uint32_t x1[2][8], x2[2][8];
#pragma unroll
                for (int l = 0; l < 2; l++) {
                    tmem_ld_frag16(tm_lane + ((uint32_t)(16 * l) << 16) + COL_O1 + t0, x1[l]);
                    tmem_ld_frag16(tm_lane + ((uint32_t)(16 * l) << 16) + COL_O2 + t0, x2[l]);
                }
                const float2 elo = *reinterpret_cast<const float2*>(rd.eb + t0 + 2 * c4);
                const float2 ehi = *reinterpret_cast<const float2*>(rd.eb + t0 + 8 + 2 * c4);
                const float ev[4] = {elo.x, elo.y, ehi.x, ehi.y};
                float val[2][8];
                tmem_ld_wait();
#pragma unroll
                for (int l = 0; l < 2; l++)
#pragma unroll
                    for (int r = 0; r < 8; r++) {
                        const float intra = __uint_as_float(x1[l][r]);
                        val[l][r] = zero_state ? intra : __fmaf_rn(ev[2 * (r >> 2) + (r & 1)], __uint_as_float(x2[l][r]), intra);
                    }
                frag_store(aO, lane, Lq, t0, val);
            }
            if (full) fence_async_smem();
        }
        tc_fence_before();
        gave_up = __syncthreads_or(m.dead) != 0;      // (B) staged outputs complete, tensor memory read
        tc_fence_after();
        if (gave_up) break;
        if (full) {
            if (is_issuer) {
                for (int p = 0; p < 2; p++) tma_store_3d(&map_o, sO + p * PANEL, p * 64, h, row0);
                tma_store_commit();
            }
        } else if (is_compute) {
            for (int e = tid; e < BT * 16; e += NC) {
                const int t = e >> 4, ch = e & 15, code = rd.code[t];
                if (code >= 0)
                    *reinterpret_cast<uint4*>(o + ((size_t)code * H + h) * D + ch * 8) =
                        *reinterpret_cast<const uint4*>(sO + (ch >> 3) * PANEL + sw128_chunk(t, ch & 7));
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

// Outputs of the chunks of sequences [seq_lo, seq_hi); their states are in the workspace.
int32_t chunk_fwd(const FwdArgs& a) {
    if (a.seq_hi == a.seq_lo) return HARTS_OK;
    CUtensorMap mq, mk, mv, mcs, mo;
    int32_t rc;
    if ((rc = make_row_map(&mq, a.q, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mk, a.k, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mv, a.v, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mo, a.o, a.tb.n_rows, a.H)) != HARTS_OK) return rc;
    if ((rc = make_state_map(&mcs, a.chunk_states, (int64_t)a.tb.n_chunks * a.H)) != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(chunk_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem::bytes + 1024) != cudaSuccess)
        return HARTS_ECUDA;
    const int64_t n = (int64_t)a.tb.n_chunks * a.H;
    const int grid = (int)(n < 2 * sm_count() ? n : 2 * sm_count());
    launch_after(chunk_fwd_kernel, grid, NT, Smem::bytes + 1024, a.stream,
        a.tb, a.seq_lo, a.seq_hi, a.H, mq, mk, mv, mcs, mo, (const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k,
        (const __nv_bfloat16*)a.v, a.g, (__nv_bfloat16*)a.o, a.dev_status, status_gate(a.flags, a.dev_status));
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
