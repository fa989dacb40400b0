// Backward of full attention on compact tokens (Section 3.4, Eqs. 21-22) for bf16, head dimension 128, on tcgen05.
//
// Three kernels, no atomics, fixed summation orders:
//   delta_kernel   delta_t = <dO_t, o_t> per (row, head);
//   dq_kernel      one work item = (piece, tile of 128 query rows, query head); walks the key tiles the queries see,
//                  exactly like the forward:  S = Q K^T,  dP = dO V^T,  P = exp2(S - lse),  dS = P (dP - delta),
//                  dQ += dS K  (dS goes back to tensor memory over S as the A operand);
//   dkv_kernel     one work item = (piece, tile of 128 key rows, kv head); walks every query tile that sees those
//                  keys -- the rest of its own piece (causal) and all rows of all descendant pieces, for every query
//                  head of the group -- with everything transposed so that key rows sit on the tensor-memory lanes:
//                  S^T = K Q^T,  dP^T = V dO^T,  dV += P^T dO,  dK += dS^T Q.
//                  The gradient of a shared ancestor's K/V is thus accumulated on chip over all its descendants and
//                  written once: this replaces the scatter-add of the gather's backward.
// dq_kernel: S lives in two tensor-memory buffers and dP is taken into registers first, so the MMAs of tile n+1 run under the
// element-wise pass of tile n, and the roles meet at mbarriers only, so that the loads and first products of an item run under the
// output of the one before.  24 MMAs of 64 cycles a 128 x 128 tile (1,536); it takes 2,800 cycles, bound by the power limit on long
// sequences (1.36 GHz).  3,970 with eleven instructions an element instead of six: scalar fp32, the scale on every dS, a test for
// hidden columns on every element.  65,521 agentic tokens x 16 heads: 8.1 -> 6.3 ms.
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

constexpr int NS = 256, NT = NS + 64;     // 8 element-wise warps: warp w and w + 4 share a lane quarter and split the columns
constexpr int Q_BYTES = BQ * D * 2;       // 32 KB
constexpr float LOG2E = 1.4426950408889634f;

__global__ void __launch_bounds__(256) delta_kernel(const __nv_bfloat16* o,
                                                    const __nv_bfloat16* __restrict__ dO, float* __restrict__ delta,
                                                    long long n, int* ticket) {       // n = rows * Hq; one warp per (row, head)
    const long long w = (blockIdx.x * 256LL + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n) return;
    const uint2 a = reinterpret_cast<const uint2*>(o + w * D)[lane], b = reinterpret_cast<const uint2*>(dO + w * D)[lane];
    const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const float2 x = __bfloat1622float2(pa[e]), y = __bfloat1622float2(pb[e]);
        s = fmaf(x.x, y.x, fmaf(x.y, y.y, s));
    }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) delta[w] = s;
    // of attn_dkv_kernel.  It lies in dq's first eight bytes, and dq may be o's memory: written by the lane that read these bytes of o
    if (w == 0 && lane == 0) *ticket = 0;
}

// ------------------------------------------------------------------------------------------------------------------
// dQ: key tiles of 128 rows, so that every MMA has N = 128 (the N = 64 shape is bound by operand reads, not by the
// tensor pipe).  Tensor memory: S in two buffers (S of tile n+1 runs under the element-wise pass of tile n), dP, dQ.
// ------------------------------------------------------------------------------------------------------------------
constexpr int BKW = 128;                       // key rows per tile
constexpr int KW_BYTES = BKW * D * 2;          // 32 KB: two panels [128 rows][64 columns]
constexpr int KST = 3;                         // K stages (a K tile is held from S to dQ); V has two (held for dP only)
struct SmemQ {
    static constexpr int q = 0, dO = Q_BYTES, k0 = 2 * Q_BYTES, v0 = k0 + KST * KW_BYTES, misc = v0 + 2 * KW_BYTES;
    static constexpr int bytes = misc + 256;
};
struct MiscQ {
    uint64_t bar_q, bar_qfree, bar_k[KST], bar_v[2], bar_kfree[KST], bar_s[2], bar_dpfree, bar_p[2], bar_o, bar_ofree, bar_exit;
    int dead;        // latch: a wait of this CTA ran out, the CTA is abandoning its work
    uint32_t tmem;
};
constexpr int COL_DP = 256, COL_DQ = 384, TMEM_Q = 512;     // S of tile n at 128 (n & 1)
using WalkW = TileWalkT<BKW>;

__global__ void __launch_bounds__(NT, 1)
attn_dq_kernel(Index ix, int Hq, int G, float scale, const __grid_constant__ CUtensorMap map_q,
               const __grid_constant__ CUtensorMap map_do, const __grid_constant__ CUtensorMap map_k,
               const __grid_constant__ CUtensorMap map_v,
               const float* __restrict__ lse, const float* __restrict__ delta, __nv_bfloat16* __restrict__ dq,
               int* status) {
    after_previous();
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char* sQ = smem + SmemQ::q;
    unsigned char* sDO = smem + SmemQ::dO;
    MiscQ& m = *reinterpret_cast<MiscQ*>(smem + SmemQ::misc);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool is_softmax = warp < NS / 32, is_issuer = warp == NS / 32, is_producer = tid == NS + 32;
    if (tid == 0) {
        mbar_init(&m.bar_q, 1);
        for (int st = 0; st < KST; st++) {
            mbar_init(&m.bar_k[st], 1);
            mbar_init(&m.bar_kfree[st], 1);
        }
        for (int st = 0; st < 2; st++) {
            mbar_init(&m.bar_v[st], 1);
            mbar_init(&m.bar_s[st], 1);
        }
        mbar_init(&m.bar_dpfree, NS / 32);
        mbar_init(&m.bar_p[0], NS / 32);
        mbar_init(&m.bar_p[1], NS / 32);
        mbar_init(&m.bar_qfree, 1);
        mbar_init(&m.bar_o, 1);
        mbar_init(&m.bar_ofree, NS / 32);
        mbar_init(&m.bar_exit, 1);
        m.dead = 0;
        fence_barrier_init();
    }
    if (warp == 0) tmem_alloc<TMEM_Q>(&m.tmem);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = m.tmem;
    const uint32_t tm_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr uint32_t I_DQ = instr_desc(BQ, D, 0, 1);     // dQ[128 x 128] += dS (tensor memory) . K (rows = keys)
    const uint64_t dQd = desc_kmajor_base(smem_u32(sQ)), dDOd = desc_kmajor_base(smem_u32(sDO));
    const float scale_log2 = scale * LOG2E;

    // where this thread's role stands in the rings, which run on over the work items (a fresh barrier counts as free: parity 1
    // has passed)
    Ring<KST> rk;
    Ring<2> r2;              // V, S and the barriers that come in twos
    uint32_t ph_q = 0, ph_dpfree = 0, ph_o = 0;
    const int n_work = ix.n_q_items * Hq;
    // work items come most work first; dealt in a snake pattern (tier by tier, every second tier in reverse), so that no
    // CTA gets the largest item of every tier
    for (int tier = 0; tier * (int)gridDim.x < n_work; tier++) {
        const int w = tier * (int)gridDim.x + ((tier & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
        if (w >= n_work) continue;
        if (*(volatile int*)&m.dead) break;       // a wait ran out: abandon the work
        const int item = w / Hq, h = w % Hq, hk = h / G;
        const int piece = ix.q_item[2 * item], qt = ix.q_item[2 * item + 1];
        const int q_row0 = ix.piece_row0[piece] + qt * BQ;
        const int q_valid = min(BQ, ix.piece_len[piece] - qt * BQ);

        if (is_producer) {
            // ---- TMA producer: Q and dO tiles, then K and V tiles two deep (released separately) --------------------
            WalkW lw(ix, piece, qt);
            KvTile lt;
            mbar_wait(&m.bar_qfree, ph_q ^ 1, status, &m.dead);      // the last item's S and dP products have read the tiles
            ph_q ^= 1;
            mbar_expect_tx(&m.bar_q, 2 * Q_BYTES);
            for (int p = 0; p < 2; p++)
                for (int r = 0; r < 2; r++) {
                    tma_load_3d(sQ + p * (Q_BYTES / 2) + r * (Q_BYTES / 4), &map_q, p * 64, h, q_row0 + r * 64, &m.bar_q);
                    tma_load_3d(sDO + p * (Q_BYTES / 2) + r * (Q_BYTES / 4), &map_do, p * 64, h, q_row0 + r * 64, &m.bar_q);
                }
            for (; lw.next(lt); rk.next(), r2.next()) {
                if (*(volatile int*)&m.dead) break;       // a wait ran out: abandon the item
                const int halves = lt.n_valid > 64 ? 2 : 1;      // rows past the 64th are read by nothing then
                unsigned char* sK = smem + SmemQ::k0 + rk.st * KW_BYTES;
                unsigned char* sV = smem + SmemQ::v0 + r2.st * KW_BYTES;
                mbar_wait(&m.bar_kfree[rk.st], rk.ph ^ 1, status, &m.dead);      // dQ of the stage's last tile is done
                mbar_expect_tx(&m.bar_k[rk.st], halves * (KW_BYTES / 2));
                for (int r = 0; r < halves; r++)
                    for (int p = 0; p < 2; p++)
                        tma_load_3d(sK + p * (KW_BYTES / 2) + r * (KW_BYTES / 4), &map_k, p * 64, hk, lt.row + r * 64, &m.bar_k[rk.st]);
                // S and dP of the stage's last tile are done; the next phase of this barrier needs the tile loaded here
                mbar_wait(&m.bar_s[r2.st], r2.ph ^ 1, status, &m.dead);
                mbar_expect_tx(&m.bar_v[r2.st], halves * (KW_BYTES / 2));
                for (int r = 0; r < halves; r++)
                    for (int p = 0; p < 2; p++)
                        tma_load_3d(sV + p * (KW_BYTES / 2) + r * (KW_BYTES / 4), &map_v, p * 64, hk, lt.row + r * 64, &m.bar_v[r2.st]);
            }
        }
        if (is_issuer) {
            // ---- MMA issue: a tcgen05.mma holds its thread until the pipe has room, so this warp does nothing else ---------
            // Pipe order S(n+1), dP(n+1), dQ(n): the first two run under the pass of tile n (S has a second buffer, and the pass
            // takes dP(n) into registers first and says so).  S / dP are as wide as the tile has keys (steps of 16), dQ as deep.
            WalkW iw(ix, piece, qt);
            KvTile tn;
            Ring<KST> rk0 = rk;        // stages of tile n; rk and r2: of tile n + 1
            Ring<2> r0 = r2;
            KvTile tl;                 // looked up one further: whether tile n + 1 is the last
            bool more = iw.next(tn), more2 = iw.next(tl);
            auto issue_s = [&]() {
                mbar_wait_warp(&m.bar_k[rk.st], rk.ph, status, &m.dead);
                tc_fence_after();
                const uint32_t idesc = instr_desc(BQ, (tn.n_valid + 15) & ~15, 0, 0);     // (Q | dO) (K-major) . (K | V) (K-major)
                const uint64_t dK = desc_kmajor_base(smem_u32(smem + SmemQ::k0 + rk.st * KW_BYTES));
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)
                        mma_ss(tmem + r2.st * 128, dQd + kstep_kmajor<BQ>(ks), dK + kstep_kmajor<BKW>(ks), idesc, ks > 0);
                }
                __syncwarp();
                rk.next();
            };
            auto issue_dp = [&](bool ahead) {     // ahead: more key tiles follow; its commit also covers S, issued before it
                mbar_wait_warp(&m.bar_v[r2.st], r2.ph, status, &m.dead);
                tc_fence_after();
                const uint32_t idesc = instr_desc(BQ, (tn.n_valid + 15) & ~15, 0, 0);
                const uint64_t dV = desc_kmajor_base(smem_u32(smem + SmemQ::v0 + r2.st * KW_BYTES));
                if (elect_one()) {
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)
                        mma_ss(tmem + COL_DP, dDOd + kstep_kmajor<BQ>(ks), dV + kstep_kmajor<BKW>(ks), idesc, ks > 0);
                    mma_commit(&m.bar_s[r2.st]);
                    if (!ahead) mma_commit(&m.bar_qfree);
                }
                __syncwarp();
                r2.next();
            };
            mbar_wait_warp(&m.bar_q, ph_q, status, &m.dead);
            ph_q ^= 1;
            issue_s();
            issue_dp(more2);
            mbar_wait_warp(&m.bar_ofree, ph_q, status, &m.dead);     // the last item's dQ has been read (ph_q: this item's parity, turned)
            for (int n = 0; more; n++) {
                if (*(volatile int*)&m.dead) break;       // a wait ran out: abandon the item
                const int steps = (tn.n_valid + 15) >> 4;
                more = more2;
                if (more) {
                    tn = tl;
                    more2 = iw.next(tl);
                    issue_s();
                }
                mbar_wait_warp(&m.bar_dpfree, ph_dpfree, status, &m.dead);
                ph_dpfree ^= 1;
                if (more) {
                    tc_fence_after();
                    issue_dp(more2);
                }
                // dS(n) written, S(n) read.  One barrier per S buffer: a warp that is done with tile n may already work
                // on tile n+1 (its S and dP are complete) and arrive for it, and that arrival must not count for tile n.
                mbar_wait_warp(&m.bar_p[r0.st], r0.ph, status, &m.dead);
                tc_fence_after();
                const uint64_t dKm = desc_mnmajor_base<BKW>(smem_u32(smem + SmemQ::k0 + rk0.st * KW_BYTES));
                const uint32_t a = tmem + r0.st * 128;
                if (elect_one()) {
                    if (steps == 8) {
#pragma unroll
                        for (int ks = 0; ks < 8; ks++)
                            mma_ts(tmem + COL_DQ, a + (ks >> 2) * 64 + (ks & 3) * 8, dKm + kstep_mnmajor(ks), I_DQ, n > 0 || ks > 0);
                    } else {
#pragma unroll 1
                        for (int ks = 0; ks < steps; ks++)
                            mma_ts(tmem + COL_DQ, a + (ks >> 2) * 64 + (ks & 3) * 8, dKm + kstep_mnmajor(ks), I_DQ, n > 0 || ks > 0);
                    }
                    mma_commit(&m.bar_kfree[rk0.st]);
                    if (!more) mma_commit(&m.bar_o);
                }
                __syncwarp();
                rk0.next();
                r0.next();
            }
        }
        if (is_softmax) {
            WalkW walk(ix, piece, qt);
            KvTile t;
            const int i = tid & 127, c = tid >> 7;           // query row, and which 64 of a tile's 128 key columns
            const bool row_ok = i < q_valid;                 // other rows are other pieces' queries: computed, never stored
            const float lse2 = row_ok ? lse[(size_t)(q_row0 + i) * Hq + h] * LOG2E : 0.f;
            const float dl = row_ok ? delta[(size_t)(q_row0 + i) * Hq + h] : 0.f;
            const F2 scale2 = f2(scale_log2, scale_log2), nl = f2(-lse2, -lse2), nd = f2(-dl, -dl);
            for (; walk.next(t); r2.next()) {
                if (*(volatile int*)&m.dead) break;       // a wait ran out: abandon the item
                const uint32_t at = tm_lane + r2.st * 128 + c * 64;
                const bool any = c * 64 < t.n_valid;      // columns past the tile's keys are read by nothing
                mbar_wait_warp(&m.bar_s[r2.st], r2.ph, status, &m.dead);
                tc_fence_after();
                uint32_t xs[32], xp[64];
                if (any) {      // dP of this thread's 64 columns into registers: its buffer can take the next tile
                    tmem_ld32(tm_lane + COL_DP + c * 64, xp);
                    tmem_ld32(tm_lane + COL_DP + c * 64 + 32, xp + 32);
                    tmem_ld32(at, xs);
                    tmem_ld_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.bar_dpfree);
                if (any) {
                    const int limit = min(t.n_valid, t.shift == NO_DIAG ? BKW : i - t.shift + 1) - c * 64;     // visible: j < limit
                    const bool masked = !__all_sync(0xffffffffu, limit >= 64);
#pragma unroll
                    for (int cc = 0; cc < 2; cc++) {
                        uint32_t pk[16];
                        if (cc) {
                            tmem_ld32(at + 32, xs);
                            tmem_ld_wait();
                        }
#pragma unroll
                        for (int e = cc * 32; e < cc * 32 + 32; e += 2) {
                            float p0, p1, d0, d1;
                            f2_split(f2_fma(f2(__uint_as_float(xs[e & 31]), __uint_as_float(xs[(e & 31) + 1])), scale2, nl), p0, p1);
                            p0 = ex2(p0);
                            p1 = ex2(p1);
                            if (masked) {
                                p0 = e < limit ? p0 : 0.f;
                                p1 = e + 1 < limit ? p1 : 0.f;
                            }
                            f2_split(f2_mul(f2(p0, p1), f2_add(f2(__uint_as_float(xp[e]), __uint_as_float(xp[e + 1])), nd)), d0, d1);
                            pk[(e & 31) >> 1] = pack_bf16(d0, d1);
                        }
                        tmem_st16(at + cc * 16, pk);      // dS / scale, over this thread's own half of S
                    }
                    tmem_st_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&m.bar_p[r2.st]);
            }
            // ---- epilogue: dQ -> bf16 ------------------------------------------------------------------------------
            mbar_wait_warp(&m.bar_o, ph_o, status, &m.dead);
            tc_fence_after();
#pragma unroll
            for (int cc = 0; cc < 2; cc++) {
                const int c4 = c * 2 + cc;
                uint32_t x[32];
                tmem_ld32(tm_lane + COL_DQ + c4 * 32, x);
                tmem_ld_wait();
                if (cc == 1) {                 // dQ has been read: the next item's may start
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&m.bar_ofree);
                }
#pragma unroll
                for (int e = 0; e < 32; e++) x[e] = __float_as_uint(__uint_as_float(x[e]) * scale);
                if (row_ok) {
#pragma unroll
                    for (int v4 = 0; v4 < 4; v4++) {
                        uint4 pk;
                        pk.x = pack_bf16(__uint_as_float(x[v4 * 8 + 0]), __uint_as_float(x[v4 * 8 + 1]));
                        pk.y = pack_bf16(__uint_as_float(x[v4 * 8 + 2]), __uint_as_float(x[v4 * 8 + 3]));
                        pk.z = pack_bf16(__uint_as_float(x[v4 * 8 + 4]), __uint_as_float(x[v4 * 8 + 5]));
                        pk.w = pack_bf16(__uint_as_float(x[v4 * 8 + 6]), __uint_as_float(x[v4 * 8 + 7]));
                        *reinterpret_cast<uint4*>(dq + ((size_t)(q_row0 + i) * Hq + h) * D + c4 * 32 + v4 * 8) = pk;
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
    if (warp == 0) tmem_dealloc<TMEM_Q>(tmem);
}

}  // namespace

int32_t attn_dkv_launch(const Index& ix, int n_rows, const void* q, const void* k, const void* v, const float* lse,
                        const void* dO, const float* delta, void* dk_, void* dv_, int Hq, int Hkv, float scale,
                        int* ticket, int32_t* status, const SplitTable* split, cudaStream_t st);
bool attn_split_table(const Index& ix, const int32_t* hi, int G, int Hkv, void* buf, size_t bytes, SplitTable* t);
int32_t attn_split_launch(const Index& ix, int G, int Hkv, const SplitTable& t, cudaStream_t st);
int32_t attn_split_reduce(const Index& ix, int Hkv, const SplitTable& t, void* dk_, void* dv_, cudaStream_t st);

int32_t attn_bwd_launch(const int32_t* hi, const int32_t* di, const void* q, const void* k, const void* v,
                        const void* o, const float* lse, const void* dO, void* dq, void* dk_, void* dv_, float* delta,
                        int Hq, int Hkv, float scale, int32_t* status, cudaStream_t st) {
    const int n_rows = hi[0];
    if (n_rows == 0 || hi[4] == 0) return HARTS_OK;
    const long long n = (long long)n_rows * Hq;
    // the dK / dV kernel runs first: its work counter and, on skewed problems, its units and their sums lie in dq's memory
    int* ticket = static_cast<int*>(dq) + 1;
    delta_kernel<<<(unsigned)((n * 32 + 255) / 256), 256, 0, st>>>((const __nv_bfloat16*)o, (const __nv_bfloat16*)dO, delta, n, ticket);
    CUtensorMap mq, mdo, mk, mv;
    int32_t rc;
    if ((rc = make_row_map(&mq, q, n_rows, Hq)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mdo, dO, n_rows, Hq)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mk, k, n_rows, Hkv)) != HARTS_OK) return rc;
    if ((rc = make_row_map(&mv, v, n_rows, Hkv)) != HARTS_OK) return rc;
    if (cudaFuncSetAttribute(attn_dq_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemQ::bytes + 1024) !=
        cudaSuccess)
        return HARTS_ECUDA;
    const Index ix = make_index(hi, di);
    SplitTable split;
    const bool cut = attn_split_table(ix, hi, Hq / Hkv, Hkv, dq, (size_t)n_rows * Hq * D * 2, &split);
    if (cut && (rc = attn_split_launch(ix, Hq / Hkv, Hkv, split, st)) != HARTS_OK) return rc;
    if ((rc = attn_dkv_launch(ix, n_rows, q, k, v, lse, dO, delta, dk_, dv_, Hq, Hkv, scale, ticket, status, cut ? &split : nullptr, st)) != HARTS_OK)
        return rc;
    if (cut && (rc = attn_split_reduce(ix, Hkv, split, dk_, dv_, st)) != HARTS_OK) return rc;
    const long long n_work = (long long)ix.n_q_items * Hq;
    const int grid = (int)(n_work < sm_count() ? n_work : sm_count());
    launch_after(attn_dq_kernel, grid, NT, SmemQ::bytes + 1024, st, ix, Hq, Hq / Hkv, scale, mq, mdo, mk, mv, lse, delta, (__nv_bfloat16*)dq, status);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
