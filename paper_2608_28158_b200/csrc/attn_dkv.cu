// dK / dV of attention on compact tokens (Section 3.4: the ancestor-KV gather's backward sums every consumer into the
// ancestor's unique compact activation) for bf16, head dimension 128, on tcgen05.
//
// One work item = (piece, tile of 128 key rows, kv head).  Key rows sit on the tensor-memory lanes; the CTA keeps the
// K and V tiles in shared memory and streams every query tile (128 rows) that sees them: the rest of the key tile's
// own piece (causal inside the tile, Eq. 22) and all rows of all descendant pieces, whatever follows each other in memory as one
// run (QRuns; one warp walks them and tells the others, tile by tile), for each query head of the GQA group.  Per query tile:
//     S^T = K Q^T,  dP^T = V dO^T            operands in shared memory, results in tensor memory
//     P^T = exp2(S^T - lse_q),  dS^T = P^T (dP^T - delta_q)     one key row per thread; bf16 back over S^T / dP^T
//     dV += P^T dO,  dK += dS^T Q            A operand from tensor memory, Q / dO tiles read row-major as B
// dK (times the scale) and dV of the tile are complete when the walk ends and are written once.  Every wait is bounded.
//
// A tile pair of 128 x 128 takes 32 MMAs of 64 cycles (2,048); 64-query tiles, whose MMAs of 48 cycles do half the work, took 5,840
// cycles a pair, these 2,950.  What the rest goes to: a warp that issues MMAs gains most by having little else to execute (3,900 ->
// 3,000 with elect.sync, no commits of its own for freed stages and no branches between the MMAs), the element-wise passes (650
// of the cycles) work on two values per instruction and test for hidden columns only in warps on the diagonal.  Long sequences are
// bound by the power limit: 65,521 agentic tokens x 16 heads 11.6 -> 7.9 ms, at 1.36 GHz.
#include "kernels.h"
#include "tc_common.cuh"

#include "../../include/harts_attn.h"
#include "attn_common.cuh"

namespace harts {

int32_t make_row_map(CUtensorMap* map, const void* base, int64_t rows, int32_t H);
int sm_count();

namespace {

using namespace tc;
using namespace attn;

constexpr int NS = 256, NT = NS + 128;    // 8 element-wise warps: warp w and w + 4 share a lane quarter and split the columns
constexpr int BKV = 128;
constexpr int TILE = BQ * D * 2;          // 32 KB: two panels [128 rows][64 columns]
constexpr int QST = 3, DST = 2, VST = 2, TST = 4, IST = 2;  // stages: Q (held from S^T to dK), dO (from dP^T to dV), vectors, tile records, items
constexpr float LOG2E = 1.4426950408889634f;
constexpr int COL_S = 0, COL_DP = 128, COL_DV = 256, COL_DK = 384, TMEM_COLS = 512;

struct Smem {
    static constexpr int k = 0, v = TILE, q0 = 2 * TILE, do0 = q0 + QST * TILE, vec = do0 + DST * TILE, misc = vec + VST * 2 * BQ * 4;
    static constexpr int bytes = misc + 384;
};
struct Misc {
    uint64_t bar_kv, bar_kvfree, bar_q[QST], bar_do[DST], bar_vec[VST], bar_vfree[VST], bar_tile[TST], bar_tfree[TST], bar_item[IST], bar_ifree[IST], bar_s, bar_dp, bar_p, bar_ds, bar_o,
        bar_ofree, bar_exit;
    int4 tile[TST];  // {first row, rows, lead, 2 head + 1 if it is the item's last}: what the walker tells the other roles
    int item[IST];   // the work numbers this CTA drew
    int4 vinfo[VST]; // the same, beside a tile's vectors
    int dead;        // latch: a wait of this CTA ran out, the CTA is abandoning its work
    uint32_t tmem;
};
static_assert(sizeof(Misc) <= 384, "barriers");

// SPLIT: the work is the unit list of attn_split.cu, and a unit of a cut item leaves fp32 sums.
template <bool SPLIT>
__global__ void __launch_bounds__(NT, 1)
attn_dkv_kernel(Index ix, int Hq, int Hkv, int G, float scale, const __grid_constant__ CUtensorMap map_q,
                const __grid_constant__ CUtensorMap map_do, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const float* __restrict__ lse,
                const float* __restrict__ delta, __nv_bfloat16* __restrict__ dk_, __nv_bfloat16* __restrict__ dv_,
                int* ticket, int* status, SplitTable split) {
    after_previous();
    extern __shared__ __align__(1024) unsigned char smem[];       // no static shared memory: the dynamic window starts 1024-byte aligned
    unsigned char* sK = smem + Smem::k;
    unsigned char* sV = smem + Smem::v;
    float* sVec = reinterpret_cast<float*>(smem + Smem::vec);       // [stage][-lse (log2 units) | -delta][128]
    Misc& m = *reinterpret_cast<Misc*>(smem + Smem::misc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool is_softmax = warp < NS / 32, is_issuer = warp == NS / 32, is_producer = tid == NS + 32, is_loader = warp == NS / 32 + 2,
               is_walker = warp == NS / 32 + 3;
    if (smem_u32(smem) & 1023) {              // never on sm_100a; the swizzled tiles would be misread
        if (tid == 0 && status) atomicExch(status, STATUS_TIMEOUT);
        return;
    }
    if (tid == 0) {
        mbar_init(&m.bar_kv, 1);
        for (int s = 0; s < QST; s++) mbar_init(&m.bar_q[s], 1);
        for (int s = 0; s < DST; s++) mbar_init(&m.bar_do[s], 1);
        for (int s = 0; s < VST; s++) { mbar_init(&m.bar_vec[s], 32); mbar_init(&m.bar_vfree[s], NS / 32); }
        for (int s = 0; s < TST; s++) { mbar_init(&m.bar_tile[s], 1); mbar_init(&m.bar_tfree[s], 3); }
        for (int s = 0; s < IST; s++) { mbar_init(&m.bar_item[s], 1); mbar_init(&m.bar_ifree[s], 3 + NS / 32); }
        mbar_init(&m.bar_s, 1);
        mbar_init(&m.bar_dp, 1);
        mbar_init(&m.bar_p, NS / 32);
        mbar_init(&m.bar_ds, NS / 32);
        mbar_init(&m.bar_kvfree, 1);
        mbar_init(&m.bar_o, 1);
        mbar_init(&m.bar_ofree, NS / 32);
        mbar_init(&m.bar_exit, 1);
        m.dead = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc<TMEM_COLS>(&m.tmem);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = m.tmem;
    const uint32_t tm_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr uint32_t I_ACC = instr_desc(BKV, D, 0, 1);    // [128 keys x 128] += (P^T | dS^T) (tensor memory) . (dO | Q)
    const uint64_t dKd = desc_kmajor_base(smem_u32(sK)), dVd = desc_kmajor_base(smem_u32(sV));
    const float scale_log2 = scale * LOG2E;

    // where this thread's role stands in the rings (a fresh barrier counts as free: parity 1 has passed) and in the single barriers
    Ring<QST> rq;
    Ring<DST> rd;
    Ring<VST> rv;
    Ring<TST> rt;
    Ring<IST> ri;
    uint32_t ph_kv = 0, ph_s = 0, ph_dp = 0, ph_p = 0, ph_ds = 0, ph_o = 0;
    const int n_work = (SPLIT ? split.n_units[0] : ix.n_kv_items) * Hkv;
    // Work items come most work first and are drawn from a counter (by the walker, when it has handed out the tiles of the one
    // before): what a key tile takes differs by the length of its tree and its depth in it, and dealt in a fixed pattern the fullest
    // CTA had 1.05 (65,521 agentic tokens) to 1.9 times (67,731 branchy) an even share.  Which CTA an item falls to does not enter
    // its sums.
    while (is_softmax || is_issuer || is_producer || is_loader || is_walker) {
        int w;
        if (is_walker) {
            if (lane == 0) w = atomicAdd(ticket, 1);
            w = __shfl_sync(0xffffffffu, w, 0);
            if (!mbar_wait_warp(&m.bar_ifree[ri.st], ri.ph ^ 1, status, &m.dead)) break;       // a wait ran out: abandon the work
            if (lane == 0) {
                m.item[ri.st] = w;
                mbar_arrive(&m.bar_item[ri.st]);
            }
            __syncwarp();
        } else if (is_producer) {
            if (!mbar_wait(&m.bar_item[ri.st], ri.ph, status, &m.dead)) break;
            w = m.item[ri.st];
            mbar_arrive(&m.bar_ifree[ri.st]);
        } else {
            if (!mbar_wait_warp(&m.bar_item[ri.st], ri.ph, status, &m.dead)) break;
            w = m.item[ri.st];
            __syncwarp();
            if (lane == 0) mbar_arrive(&m.bar_ifree[ri.st]);
        }
        ri.next();
        if (w >= n_work) break;
        const int item = w / Hkv, hk = w % Hkv;
        DkvUnit unit{};
        if (SPLIT) unit = split.unit[item];
        const int piece = SPLIT ? unit.piece : ix.kv_item[2 * item], kt = SPLIT ? unit.kt : ix.kv_item[2 * item + 1];
        const bool partial = SPLIT && unit.slot >= 0;
        const int kv_row0 = ix.piece_row0[piece] + kt * BKV;
        const int kv_valid = min(BKV, ix.piece_len[piece] - kt * BKV);

        if (is_producer) {
            // ---- TMA producer: the K and V tiles, then the query and dO tiles (QST and DST deep) -----------------------------
            mbar_wait(&m.bar_kvfree, ph_kv ^ 1, status, &m.dead);    // the last item's S^T and dP^T products have read the tiles
            ph_kv ^= 1;
            mbar_expect_tx(&m.bar_kv, 2 * TILE);
            for (int p = 0; p < 2; p++)
                for (int r = 0; r < 2; r++) {
                    tma_load_3d(sK + p * (TILE / 2) + r * (TILE / 4), &map_k, p * 64, hk, kv_row0 + r * 64, &m.bar_kv);
                    tma_load_3d(sV + p * (TILE / 2) + r * (TILE / 4), &map_v, p * 64, hk, kv_row0 + r * 64, &m.bar_kv);
                }
            for (int4 t{}; !(t.w & 1); rq.next(), rd.next()) {
                if (!mbar_wait(&m.bar_tile[rt.st], rt.ph, status, &m.dead)) break;       // a wait ran out: abandon the item
                t = m.tile[rt.st];
                mbar_arrive(&m.bar_tfree[rt.st]);
                rt.next();
                const int halves = t.y > 64 ? 2 : 1;      // rows past the 64th are read by nothing then
                // S^T of the tile before (over all items) done: so are dK of three tiles ago and dV of two tiles ago, issued before
                // it, which read these stages last.  The tile is not needed before that tile's dV, 1,500 cycles later.  (Every phase
                // is waited for, and the next cannot complete before: parity is enough.)
                mbar_wait(&m.bar_s, ph_s ^ 1, status, &m.dead);
                ph_s ^= 1;
                unsigned char* sQ = smem + Smem::q0 + rq.st * TILE;
                unsigned char* sDO = smem + Smem::do0 + rd.st * TILE;
                mbar_expect_tx(&m.bar_q[rq.st], halves * (TILE / 2));
                for (int r = 0; r < halves; r++)
                    for (int p = 0; p < 2; p++)
                        tma_load_3d(sQ + p * (TILE / 2) + r * (TILE / 4), &map_q, p * 64, t.w >> 1, t.x + r * 64, &m.bar_q[rq.st]);
                mbar_expect_tx(&m.bar_do[rd.st], halves * (TILE / 2));
                for (int r = 0; r < halves; r++)
                    for (int p = 0; p < 2; p++)
                        tma_load_3d(sDO + p * (TILE / 2) + r * (TILE / 4), &map_do, p * 64, t.w >> 1, t.x + r * 64, &m.bar_do[rd.st]);
            }
        }
        if (is_walker) {
            // ---- the query tiles of this item, in order, TST ahead of the slowest role that uses them ---------------------
            QRuns r(ix, piece, kt);
            int g = 0, left = 0x7fffffff;
            if (SPLIT) {
                g = unit.g;
                left = unit.n_tiles;
                r.row = unit.row;
                r.end = unit.end;
                r.lead = unit.lead;
                r.d = unit.d;
            } else {
                r.first();
            }
            for (bool more = true; more; rt.next()) {
                int4 t = make_int4(r.row, min(BQ, r.end - r.row), r.lead, 2 * (hk * G + g));
                r.row += BQ;
                if (r.lead >= 0) r.lead += BQ;
                if (--left == 0) more = false;
                if (more && r.row >= r.end && !r.next()) {
                    more = ++g < G;
                    if (more) r.first();
                }
                t.w |= !more;
                if (!mbar_wait_warp(&m.bar_tfree[rt.st], rt.ph ^ 1, status, &m.dead)) break;       // a wait ran out: abandon the item
                if (lane == 0) {
                    m.tile[rt.st] = t;
                    mbar_arrive(&m.bar_tile[rt.st]);
                }
                __syncwarp();
            }
        }
        if (is_loader) {
            // ---- per-column -lse (log2 units) and -delta of the query tiles, in flight while the ring is full -----------
            for (int4 t{}; !(t.w & 1); rv.next()) {
                if (!mbar_wait_warp(&m.bar_tile[rt.st], rt.ph, status, &m.dead)) break;  // a wait ran out: abandon the item
                t = m.tile[rt.st];
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.bar_tfree[rt.st]);
                rt.next();
                float l4[4], d4[4];
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const int j = lane + e * 32;
                    const size_t at = (size_t)(t.x + j) * Hq + (t.w >> 1);
                    l4[e] = j < t.y ? -lse[at] * LOG2E : -INFINITY;     // columns past the end: probability 0
                    d4[e] = j < t.y ? -delta[at] : 0.f;
                }
                mbar_wait_warp(&m.bar_vfree[rv.st], rv.ph ^ 1, status, &m.dead);
                if (lane == 0) m.vinfo[rv.st] = t;
                float* to = sVec + rv.st * 2 * BQ + lane;
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    to[e * 32] = l4[e];
                    to[BQ + e * 32] = d4[e];
                }
                mbar_arrive(&m.bar_vec[rv.st]);
            }
        }
        if (is_issuer) {
            // ---- MMA issue: a tcgen05.mma holds its thread until the pipe has room, so this warp does nothing else ---------
            // Pipe order dV(n), S^T(n+1), dK(n), dP^T(n+1): P of tile n+1 is made under the last two, dS of tile n under the
            // first two.  S^T / dP^T are as wide as the tile has queries (steps of 16), dV / dK as deep.
            int4 tn{};                 // tile n + 1
            auto read_tile = [&]() {
                const bool ok = mbar_wait_warp(&m.bar_tile[rt.st], rt.ph, status, &m.dead);
                tn = m.tile[rt.st];
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.bar_tfree[rt.st]);
                rt.next();
                return ok;
            };
            Ring<QST> rq0 = rq;        // stages of tile n; rq and rd: of tile n + 1
            Ring<DST> rd0 = rd;
            auto issue_s = [&]() {
                mbar_wait_warp(&m.bar_q[rq.st], rq.ph, status, &m.dead);
                tc_fence_after();
                const uint32_t idesc = instr_desc(BKV, (tn.y + 15) & ~15, 0, 0);
                const uint64_t dQ = desc_kmajor_base(smem_u32(smem + Smem::q0 + rq.st * TILE));
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ks++) mma_ss(tmem + COL_S, dKd + kstep_kmajor<BKV>(ks), dQ + kstep_kmajor<BQ>(ks), idesc, ks > 0);
                    mma_commit(&m.bar_s);
                }
                __syncwarp();
                rq.next();
            };
            auto issue_dp = [&]() {
                mbar_wait_warp(&m.bar_do[rd.st], rd.ph, status, &m.dead);
                tc_fence_after();
                const uint32_t idesc = instr_desc(BKV, (tn.y + 15) & ~15, 0, 0);
                const uint64_t dDO = desc_kmajor_base(smem_u32(smem + Smem::do0 + rd.st * TILE));
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ks++) mma_ss(tmem + COL_DP, dVd + kstep_kmajor<BKV>(ks), dDO + kstep_kmajor<BQ>(ks), idesc, ks > 0);
                    mma_commit(&m.bar_dp);
                    if (tn.w & 1) mma_commit(&m.bar_kvfree);
                }
                __syncwarp();
                rd.next();
            };
            // dV or dK += A (tensor memory, `steps` k-steps of 16 queries) . B
            auto accumulate = [&](uint32_t d, uint32_t a, uint64_t b, int steps, bool add) {
                if (elect_one()) {
                    if (steps == 8) {
#pragma unroll
                        for (int ks = 0; ks < 8; ks++) mma_ts(d, a + (ks >> 2) * 64 + (ks & 3) * 8, b + kstep_mnmajor(ks), I_ACC, ks > 0 || add);
                    } else {
#pragma unroll 1
                        for (int ks = 0; ks < steps; ks++) mma_ts(d, a + (ks >> 2) * 64 + (ks & 3) * 8, b + kstep_mnmajor(ks), I_ACC, ks > 0 || add);
                    }
                }
                __syncwarp();
            };
            mbar_wait_warp(&m.bar_kv, ph_kv, status, &m.dead);
            ph_kv ^= 1;
            bool more = read_tile();
            issue_s();
            issue_dp();
            mbar_wait_warp(&m.bar_ofree, ph_kv, status, &m.dead);    // the last item's sums have been read (ph_kv: this item's parity, turned)
            for (int n = 0; more; n++) {
                if (*(volatile int*)&m.dead) break;       // a wait ran out: abandon the item
                const int steps = (tn.y + 15) >> 4;
                more = !(tn.w & 1);
                if (more) read_tile();
                mbar_wait_warp(&m.bar_p, ph_p, status, &m.dead);
                ph_p ^= 1;
                tc_fence_after();
                accumulate(tmem + COL_DV, tmem + COL_S, desc_mnmajor_base<BQ>(smem_u32(smem + Smem::do0 + rd0.st * TILE)), steps, n > 0);
                rd0.next();
                if (more) issue_s();
                mbar_wait_warp(&m.bar_ds, ph_ds, status, &m.dead);
                ph_ds ^= 1;
                tc_fence_after();
                accumulate(tmem + COL_DK, tmem + COL_DP, desc_mnmajor_base<BQ>(smem_u32(smem + Smem::q0 + rq0.st * TILE)), steps, n > 0);
                rq0.next();
                if (more) issue_dp();
            }
            if (elect_one()) mma_commit(&m.bar_o);
            __syncwarp();
        }
        if (is_softmax) {
            const int i = tid & 127, c = tid >> 7;             // key row inside the tile, and which 64 of the 128 query columns
            const F2 scale2 = f2(scale_log2, scale_log2);
            for (bool more = true; more; rv.next()) {
                if (!mbar_wait_warp(&m.bar_vec[rv.st], rv.ph, status, &m.dead)) break;   // a wait ran out: abandon the item
                const int4 t = m.vinfo[rv.st];
                more = !(t.w & 1);
                const bool any = c * 64 < t.y;      // columns past the tile's queries are read by nothing
                // query column j of an own tile sees key row i iff j >= i - lead; only warps on the diagonal have hidden ones.
                // Key rows past the end of the piece are other pieces' rows: computed, never stored.
                const bool masked = t.z >= 0 && (warp & 3) * 32 + 31 - t.z > c * 64;
                const int jmin = i - t.z - c * 64;
                const float* vl = sVec + rv.st * 2 * BQ + c * 64;
                F2 p[32];
                // ---- P^T = exp2(S^T - lse), bf16 over this warp's half of S^T (the other warp may still read its half) ------
                mbar_wait_warp(&m.bar_s, ph_s, status, &m.dead);
                ph_s ^= 1;
                tc_fence_after();
                if (any) {
                    uint32_t x[64];
                    tmem_ld32(tm_lane + COL_S + c * 64, x);
                    tmem_ld32(tm_lane + COL_S + c * 64 + 32, x + 32);
                    tmem_ld_wait();
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        uint32_t pk[16];
#pragma unroll
                        for (int e = h * 32; e < h * 32 + 32; e += 4) {
                            const float4 l4 = *reinterpret_cast<const float4*>(vl + e);
                            const F2 a = f2_fma(f2(__uint_as_float(x[e]), __uint_as_float(x[e + 1])), scale2, f2(l4.x, l4.y));
                            const F2 b = f2_fma(f2(__uint_as_float(x[e + 2]), __uint_as_float(x[e + 3])), scale2, f2(l4.z, l4.w));
                            float y[4];
                            f2_split(a, y[0], y[1]);
                            f2_split(b, y[2], y[3]);
#pragma unroll
                            for (int u = 0; u < 4; u++) y[u] = ex2(y[u]);
                            if (masked) {
#pragma unroll
                                for (int u = 0; u < 4; u++) y[u] = e + u >= jmin ? y[u] : 0.f;
                            }
                            p[e >> 1] = f2(y[0], y[1]);
                            p[(e >> 1) + 1] = f2(y[2], y[3]);
                            pk[(e & 31) >> 1] = pack_bf16(y[0], y[1]);
                            pk[((e & 31) >> 1) + 1] = pack_bf16(y[2], y[3]);
                        }
                        tmem_st16(tm_lane + COL_S + c * 64 + h * 16, pk);
                    }
                    tmem_st_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.bar_p);
                // ---- dS^T / scale = P^T (dP^T - delta), bf16 over this warp's half of dP^T -----------------------------
                mbar_wait_warp(&m.bar_dp, ph_dp, status, &m.dead);
                ph_dp ^= 1;
                tc_fence_after();
                if (any) {
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        uint32_t x[32], pk[16];
                        tmem_ld32(tm_lane + COL_DP + c * 64 + h * 32, x);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; e += 4) {
                            const float4 d4 = *reinterpret_cast<const float4*>(vl + BQ + h * 32 + e);
                            const F2 a = f2_mul(p[h * 16 + (e >> 1)], f2_add(f2(__uint_as_float(x[e]), __uint_as_float(x[e + 1])), f2(d4.x, d4.y)));
                            const F2 b = f2_mul(p[h * 16 + (e >> 1) + 1], f2_add(f2(__uint_as_float(x[e + 2]), __uint_as_float(x[e + 3])), f2(d4.z, d4.w)));
                            float y[4];
                            f2_split(a, y[0], y[1]);
                            f2_split(b, y[2], y[3]);
                            pk[e >> 1] = pack_bf16(y[0], y[1]);
                            pk[(e >> 1) + 1] = pack_bf16(y[2], y[3]);
                        }
                        tmem_st16(tm_lane + COL_DP + c * 64 + h * 16, pk);
                    }
                    tmem_st_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&m.bar_ds);
                    mbar_arrive(&m.bar_vfree[rv.st]);
                }
            }
            // ---- epilogue: dV, dK -> bf16 ---------------------------------------------------------------------------
            mbar_wait_warp(&m.bar_o, ph_o, status, &m.dead);
            tc_fence_after();
            const bool row_ok = i < kv_valid;
#pragma unroll 1
            for (int cc = 0; cc < 4; cc++) {
                const int which = cc >> 1, c4 = c * 2 + (cc & 1);       // dV, dV, dK, dK
                uint32_t x[32];
                tmem_ld32(tm_lane + (which ? COL_DK : COL_DV) + c4 * 32, x);
                tmem_ld_wait();
                if (cc == 3) {                 // the sums have been read: the next item's may start
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.bar_ofree);
                }
                const float f = which ? scale : 1.f;
#pragma unroll
                for (int e = 0; e < 32; e++) x[e] = __float_as_uint(__uint_as_float(x[e]) * f);
                if (partial) {                                           // fp32 sums of this unit
                    float4* to = reinterpret_cast<float4*>(split.sums + (((size_t)unit.slot * Hkv + hk) * 2 + which) * (BKV * D) + i * D + c4 * 32);
#pragma unroll
                    for (int v = 0; v < 8; v++)
                        to[v] = make_float4(__uint_as_float(x[4 * v]), __uint_as_float(x[4 * v + 1]), __uint_as_float(x[4 * v + 2]),
                                            __uint_as_float(x[4 * v + 3]));
                } else if (row_ok) {
                    __nv_bfloat16* to = (which ? dk_ : dv_) + ((size_t)(kv_row0 + i) * Hkv + hk) * D + c4 * 32;
#pragma unroll
                    for (int v4 = 0; v4 < 4; v4++) {
                        uint4 pk;
                        pk.x = pack_bf16(__uint_as_float(x[v4 * 8 + 0]), __uint_as_float(x[v4 * 8 + 1]));
                        pk.y = pack_bf16(__uint_as_float(x[v4 * 8 + 2]), __uint_as_float(x[v4 * 8 + 3]));
                        pk.z = pack_bf16(__uint_as_float(x[v4 * 8 + 4]), __uint_as_float(x[v4 * 8 + 5]));
                        pk.w = pack_bf16(__uint_as_float(x[v4 * 8 + 6]), __uint_as_float(x[v4 * 8 + 7]));
                        *reinterpret_cast<uint4*>(to + v4 * 8) = pk;
                    }
                }
            }
            ph_o ^= 1;
        }
    }
    if (__syncthreads_or(m.dead)) {               // abandoned: let the loads and MMAs in flight finish (bounded)
        if (is_issuer && elect_one()) {
            mma_commit(&m.bar_exit);
            mbar_wait_drain(&m.bar_exit, 0);
        }
        drain_delay();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc<TMEM_COLS>(tmem);
}

}  // namespace

int32_t attn_dkv_launch(const Index& ix, int n_rows, const void* q, const void* k, const void* v, const float* lse,
                        const void* dO, const float* delta, void* dk_, void* dv_, int Hq, int Hkv, float scale,
                        int* ticket, int32_t* status, const SplitTable* split, cudaStream_t st) {
    CUtensorMap mq, mdo, mk, mv;
    int32_t rc;
    if ((rc = make_row_map(&mq, q, n_rows, Hq)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdo, dO, n_rows, Hq)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mk, k, n_rows, Hkv)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mv, v, n_rows, Hkv)) != HARTS_OK) return rc;
    const auto kernel = split ? attn_dkv_kernel<true> : attn_dkv_kernel<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem::bytes) != cudaSuccess) return HARTS_ECUDA;
    const long long n_work = (long long)ix.n_kv_items * Hkv;
    const int grid = split || n_work > sm_count() ? sm_count() : (int)n_work;
    launch_after(kernel, grid, NT, Smem::bytes, st, ix, Hq, Hkv, Hq / Hkv, scale, mq, mdo, mk, mv, lse, delta, (__nv_bfloat16*)dk_,
                 (__nv_bfloat16*)dv_, ticket, status, split ? *split : SplitTable{});
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
