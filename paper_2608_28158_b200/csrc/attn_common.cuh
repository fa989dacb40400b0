// Shared by the attention kernels: the device view of the host index and the walk over the key tiles of a
// query tile (ancestor rows first, then the piece's own rows up to the diagonal, Eq. 22).
#pragma once
#include <cstdint>

namespace harts {
namespace attn {

constexpr int BQ = 128, BK = 64, D = 128;
constexpr int NO_DIAG = -(1 << 28);

struct Index {
    const int32_t *piece_row0, *piece_len, *anc_ptr, *anc_row0, *anc_len, *desc_ptr, *desc_piece, *q_item, *kv_item;
    int n_q_items, n_kv_items;
};
inline Index make_index(const int32_t* hi, const int32_t* di) {
    Index ix;
    ix.piece_row0 = di + hi[8];
    ix.piece_len = di + hi[9];
    ix.anc_ptr = di + hi[11];
    ix.anc_row0 = di + hi[12];
    ix.anc_len = di + hi[13];
    ix.desc_ptr = di + hi[14];
    ix.desc_piece = di + hi[15];
    ix.q_item = di + hi[16];
    ix.kv_item = di + hi[17];
    ix.n_q_items = hi[4];
    ix.n_kv_items = hi[5];
    return ix;
}

// The t-th key tile of an item: rows [row, row + n_valid), and the diagonal shift (key column j is visible to
// query row i iff j + shift <= i; NO_DIAG for ancestor rows).
struct KvTile {
    int row, n_valid, shift;
};

template <int W>
struct TileWalkT {      // enumerates the key tiles (W rows) of one item in order; run data is read once per run, not per tile
    const Index& ix;
    int run, run_end, off, own_row0, own_end, q0, cur_row0, cur_len;
    bool in_own;
    __device__ TileWalkT(const Index& ix_, int piece, int qt) : ix(ix_) {
        run = ix.anc_ptr[piece];
        run_end = ix.anc_ptr[piece + 1];
        off = 0;
        own_row0 = ix.piece_row0[piece];
        q0 = qt * BQ;
        own_end = min(ix.piece_len[piece], q0 + BQ);      // own rows up to the end of the query tile
        in_own = run == run_end;
        cur_row0 = cur_len = 0;
        if (!in_own) {
            cur_row0 = ix.anc_row0[run];
            cur_len = ix.anc_len[run];
        }
    }
    __device__ bool next(KvTile& t) {
        if (!in_own && off + W < cur_len) {       // inside a run
            t.row = cur_row0 + off;
            t.n_valid = W;
            t.shift = NO_DIAG;
            off += W;
            return true;
        }
        if (!in_own) {
            t.row = cur_row0 + off;
            t.n_valid = min(W, cur_len - off);
            t.shift = NO_DIAG;
            off += W;
            if (off >= cur_len) {
                off = 0;
                if (++run == run_end) {
                    in_own = true;
                } else {
                    cur_row0 = ix.anc_row0[run];
                    cur_len = ix.anc_len[run];
                }
            }
            return true;
        }
        if (off >= own_end) return false;
        t.row = own_row0 + off;
        t.n_valid = min(W, own_end - off);
        t.shift = off - q0;
        off += W;
        return true;
    }
};
using TileWalk = TileWalkT<BK>;

// dK / dV work of small problems, cut into units (attn_split.cu): a unit is some of the query tiles of one key tile, in the
// order of QRuns: n_tiles from head g of the group, from row `row` of the run that ends at `end` on (lead: that row's distance to the key
// tile's first row, -1 for descendants; d: the descendant behind the run).  slot: where its partial sums go, -1: the item is not cut.
struct DkvUnit {
    int piece, kt, n_tiles, slot, g, row, end, lead, d;
};
struct SplitItem {
    int n_tiles, n_units, first_unit, first_slot;
};
struct SplitTable {
    int* n_units;
    SplitItem* item;         // [n_kv_items]
    DkvUnit* unit;
    float* sums;             // [slot][Hkv][dV, dK][128][D]
    int cap_slots;
};

// The query rows that see the key tile `kt` (128 rows) of a piece, as runs [row, end) of physical rows: the rest of the piece from
// the key tile's first row on (causal inside), then all rows of every descendant piece.  Descendants that follow each other in
// memory make one run -- they all see the whole key tile -- and so does the first of them with the piece's own rest: fans of short
// branches fill their query tiles (17,111 replay tokens x 16 heads, two to a key head: dK / dV 3.0 ms piece by piece, 0.82 so; 1,773
// agentic x 32 heads 145 -> 79 us).  Used by a whole warp.
// Key row i is seen by row lead + j of the first run iff i <= lead + j; lead < 0: a run without a diagonal.
struct QRuns {
    const Index& ix;
    int piece, k0, d, d_end, row, end, lead, lane;
    __device__ QRuns(const Index& ix_, int piece_, int kt) : ix(ix_), piece(piece_), k0(kt * BQ), lane(threadIdx.x & 31) {
        d_end = ix.desc_ptr[piece + 1];
    }
    __device__ void extend(int last) {          // the run's end: behind piece `last` and those that follow it, d: the next one
        while (true) {
            const bool follows = d + lane < d_end && ix.desc_piece[d + lane] == last + 1 + lane;
            const unsigned m = __ballot_sync(0xffffffffu, follows);
            const int k = m == 0xffffffffu ? 32 : __ffs(~m) - 1;
            last += k;
            d += k;
            if (k < 32) break;
        }
        end = ix.piece_row0[last] + ix.piece_len[last];
    }
    __device__ void first() {
        d = ix.desc_ptr[piece];
        row = ix.piece_row0[piece] + k0;
        lead = 0;
        extend(piece);
    }
    __device__ bool next() {
        if (d >= d_end) return false;
        const int p = ix.desc_piece[d++];
        row = ix.piece_row0[p];
        lead = -1;
        extend(p);
        return true;
    }
    __device__ int tiles() const { return (end - row + BQ - 1) / BQ; }
};

// Position in a ring of N stages that runs on over a CTA's work items: the stage, and the parity of its barriers in this lap.
template <int N>
struct Ring {
    int st = 0;
    uint32_t ph = 0;
    __device__ void next() {
        if (++st == N) {
            st = 0;
            ph ^= 1;
        }
    }
};

}  // namespace attn
}  // namespace harts
