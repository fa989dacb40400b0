// Split of the dK / dV work of small, skewed problems (worth_cutting).  A key tile near the root is seen by every query below
// it -- for every query head of its group -- so on one tree with grouped queries a few work items are most of the work, and the
// CTA that draws the largest one is what the launch takes (9,001 tokens, 16 query heads on 4 key heads: both backward kernels 0.62
// ms; 0.39 ms with this split, 0.03 of them in split_kernel and reduce_kernel).  Here one CTA cuts every item into units of about a quarter of
// an SM's share of the whole, attn_dkv_kernel leaves the sums of a cut item in fp32, unit by unit, and reduce_kernel adds them
// in unit order (no atomics: same bits every run).
// The table and the partial sums live in the dq tensor, which is written only afterwards (the dQ kernel runs last then).
#include <memory>
#include <new>

#include "kernels.h"

#include "../../include/harts_attn.h"
#include "attn_common.cuh"

namespace harts {

int sm_count();

namespace {

using namespace attn;

constexpr int LEAST_UNIT = 8;          // query tiles

// One CTA of 1024 threads, a warp per item.
__global__ void __launch_bounds__(1024) split_kernel(Index ix, int G, int Hkv, int sms, SplitTable t) {
    after_previous();
    __shared__ int total, slots, len;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    for (int i = warp; i < ix.n_kv_items; i += 32) {          // tiles of every item
        QRuns r(ix, ix.kv_item[2 * i], ix.kv_item[2 * i + 1]);
        r.first();
        int n = r.tiles();
        while (r.next()) n += r.tiles();
        n *= G;
        if (lane == 0) {
            t.item[i].n_tiles = n;
            atomicAdd(&total, n);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) len = max(LEAST_UNIT, (int)(((long long)total * Hkv + 4 * sms - 1) / (4 * sms)));
    for (int tries = 0; tries < 20; tries++) {                // the longest unit such that the partial sums fit
        if (threadIdx.x == 0) slots = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < ix.n_kv_items; i += 1024) {
            const int n = t.item[i].n_tiles;
            if (n > len) atomicAdd(&slots, (n + len - 1) / len);
        }
        __syncthreads();
        const bool fits = slots <= t.cap_slots;
        __syncthreads();
        if (fits) break;
        if (threadIdx.x == 0) len *= 2;
    }
    __syncthreads();
    const int L = slots <= t.cap_slots ? len : 0x3fffffff;
    if (warp == 0) {                                          // units and slots before every item
        int units = 0, used = 0;
        for (int i0 = 0; i0 < ix.n_kv_items; i0 += 32) {
            const int i = i0 + lane, n = i < ix.n_kv_items ? t.item[i].n_tiles : 0;
            const int k = i < ix.n_kv_items ? (n + L - 1) / L : 0, s = k > 1 ? k : 0;
            int ku = k, su = s;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(~0u, ku, o), z = __shfl_up_sync(~0u, su, o);
                if (lane >= o) {
                    ku += y;
                    su += z;
                }
            }
            if (i < ix.n_kv_items) {
                t.item[i].n_units = k;
                t.item[i].first_unit = units + ku - k;
                t.item[i].first_slot = used + su - s;
            }
            units += __shfl_sync(~0u, ku, 31);
            used += __shfl_sync(~0u, su, 31);
        }
        if (lane == 0) t.n_units[0] = units;
    }
    __syncthreads();
    for (int i = warp; i < ix.n_kv_items; i += 32) {          // where every unit begins
        const SplitItem it = t.item[i];
        const int per_head = it.n_tiles / G, step = (it.n_tiles + it.n_units - 1) / it.n_units;
        for (int u = 0; u < it.n_units; u++) {
            DkvUnit x;
            x.piece = ix.kv_item[2 * i];
            x.kt = ix.kv_item[2 * i + 1];
            x.n_tiles = max(0, min(step, it.n_tiles - u * step));
            x.slot = it.n_units > 1 ? it.first_slot + u : -1;
            const int at = min(u * step, it.n_tiles - 1);
            x.g = at / per_head;
            int skip = at % per_head;
            QRuns r(ix, x.piece, x.kt);
            for (r.first(); skip >= r.tiles(); r.next()) skip -= r.tiles();
            x.row = r.row + skip * BQ;
            x.end = r.end;
            x.lead = r.lead < 0 ? -1 : skip * BQ;
            x.d = r.d;
            if (lane == 0) t.unit[it.first_unit + u] = x;
        }
    }
}

// dV and dK of the items that were cut: their units' sums in unit order, eight CTAs per (item, key head).
__global__ void __launch_bounds__(256) reduce_kernel(Index ix, int Hkv, SplitTable t, __nv_bfloat16* __restrict__ dk_,
                                                     __nv_bfloat16* __restrict__ dv_) {
    after_previous();
    const int part = blockIdx.x & 7, i = (blockIdx.x >> 3) / Hkv, hk = (blockIdx.x >> 3) % Hkv;
    const SplitItem it = t.item[i];
    if (it.n_units < 2) return;
    const int piece = ix.kv_item[2 * i], kt = ix.kv_item[2 * i + 1];
    const int row0 = ix.piece_row0[piece] + kt * 128, valid = min(128, ix.piece_len[piece] - kt * 128);
#pragma unroll
    for (int which = 0; which < 2; which++) {
        const int r = part * 16 + threadIdx.x / 16, ch = threadIdx.x % 16;
        if (r >= valid) return;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
#pragma unroll 4
        for (int u = 0; u < it.n_units; u++) {
            const float4* src = reinterpret_cast<const float4*>(t.sums + (((size_t)(it.first_slot + u) * Hkv + hk) * 2 + which) * (128 * D) +
                                                                r * D + ch * 8);
            const float4 x = src[0], y = src[1];
            a.x += x.x, a.y += x.y, a.z += x.z, a.w += x.w;
            b.x += y.x, b.y += y.y, b.z += y.z, b.w += y.w;
        }
        __nv_bfloat162 o[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w), __floats2bfloat162_rn(b.x, b.y),
                               __floats2bfloat162_rn(b.z, b.w)};
        *reinterpret_cast<uint4*>((which ? dk_ : dv_) + ((size_t)(row0 + r) * Hkv + hk) * D + ch * 8) = *reinterpret_cast<uint4*>(o);
    }
}

}  // namespace

// What cutting would save, from the host's copy of the index, in query tiles (1.3 to 1.5 us): uncut, a launch takes as long as its
// largest item or an even share of all, cut as long as its longest unit (split_kernel's length, from the room for partial sums) or
// the share.  That has to make up for two extra kernels, the units' starts and ends and the partial sums: 60 tiles.  Both
// backward kernels, whole -> cut, us (largest item, share):
//   worth it    9,001 branchy tokens, 16 query / 4 key heads  615 -> 385 (284, 74); 12,001 x 8/2 758 -> 418 (376, 80); 3,001 x 16/2
//               349 -> 132 (192, 20); 30,001 x 16/4 2,149 -> 1,973 (492, 429); 5,001 agentic x 8/2 367 -> 278 (160, 41);
//               6,007 replay x 8/1 806 -> 462 (376, 68)
//   not         25,001 branchy x 8/8 836 -> 855 (98, 167), 1,773 agentic x 32/32 173 -> 184 (14, 26); too little room for sums:
//               10,001 agentic x 4/1 658 -> 680 (316, 77; longest unit 304), 1,964 x 4/1 135 -> 145 (64, 4)
constexpr int CUT_LEAST = 60;
static bool worth_cutting(const int32_t* hi, int G, int Hkv, int sms, int cap_slots) {
    const int P = hi[1], n_items = hi[5];
    const int32_t *len = hi + hi[9], *parent = hi + hi[10], *item = hi + hi[17];
    auto tiles = [](int rows) { return (rows + BQ - 1) / BQ; };
    std::unique_ptr<int32_t[]> mem(new (std::nothrow) int32_t[3 * (size_t)P]());
    if (!mem) return false;
    int32_t *below = mem.get(), *kids = below + P, *todo = kids + P, n = 0;     // below: rows of all descendants
    for (int p = 0; p < P; p++)
        if (parent[p] >= 0) kids[parent[p]]++;
    for (int p = 0; p < P; p++)
        if (!kids[p]) todo[n++] = p;
    while (n) {
        const int p = todo[--n], a = parent[p];
        if (a < 0) continue;
        below[a] += below[p] + len[p];
        if (--kids[a] == 0) todo[n++] = a;
    }
    std::unique_ptr<int32_t[]> n_tiles(new (std::nothrow) int32_t[n_items]);
    if (!n_tiles) return false;
    int64_t total = 0, most = 0;
    for (int i = 0; i < n_items; i++) {
        const int piece = item[2 * i];
        const int32_t t = G * tiles(below[piece] + len[piece] - item[2 * i + 1] * 128);
        n_tiles[i] = t;
        total += (int64_t)t * Hkv;
        most = t > most ? t : most;
    }
    const int64_t share = (total + sms - 1) / sms;
    if (most - share < CUT_LEAST) return false;
    int64_t unit = (total + 4 * sms - 1) / (4 * sms);
    if (unit < LEAST_UNIT) unit = LEAST_UNIT;
    for (; unit < most; unit *= 2) {          // as split_kernel does
        int64_t slots = 0;
        for (int i = 0; i < n_items; i++)
            if (n_tiles[i] > unit) slots += (n_tiles[i] + unit - 1) / unit;
        if (slots <= cap_slots) break;
    }
    return most - (unit > share ? unit : share) >= CUT_LEAST;
}

// The table and the partial sums in `buf`; false: too small a buffer, or nothing to gain.
bool attn_split_table(const Index& ix, const int32_t* hi, int G, int Hkv, void* buf, size_t bytes, SplitTable* t) {
    const size_t max_units = (size_t)ix.n_kv_items + 5 * sm_count() + 64;       // units of a quarter share, plus one per item
    char* p = static_cast<char*>(buf);
    size_t off = 256;
    t->n_units = reinterpret_cast<int*>(p);
    t->item = reinterpret_cast<SplitItem*>(p + off);
    off = align_up(off + (size_t)ix.n_kv_items * sizeof(SplitItem), 256);
    t->unit = reinterpret_cast<DkvUnit*>(p + off);
    off = align_up(off + max_units * sizeof(DkvUnit), 256);
    t->sums = reinterpret_cast<float*>(p + off);
    if (bytes <= off) return false;
    t->cap_slots = (int)((bytes - off) / ((size_t)Hkv * 2 * 128 * D * sizeof(float)));
    return t->cap_slots > 1 && worth_cutting(hi, G, Hkv, sm_count(), t->cap_slots);
}
int32_t attn_split_launch(const Index& ix, int G, int Hkv, const SplitTable& t, cudaStream_t st) {
    launch_after(split_kernel, 1, 1024, 0, st, ix, G, Hkv, sm_count(), t);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}
int32_t attn_split_reduce(const Index& ix, int Hkv, const SplitTable& t, void* dk_, void* dv_, cudaStream_t st) {
    launch_after(reduce_kernel, ix.n_kv_items * Hkv * 8, 256, 0, st, ix, Hkv, t, (__nv_bfloat16*)dk_, (__nv_bfloat16*)dv_);
    return cudaGetLastError() == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

}  // namespace harts
