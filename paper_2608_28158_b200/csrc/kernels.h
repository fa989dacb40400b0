// Internal launch interface between the C ABI (api.cu) and the kernel files.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "../../include/harts_la.h"

namespace harts {

struct FwdArgs {
    harts_la_tables_t tb;
    int32_t seq_lo, seq_hi;
    const void *q, *k, *v;
    const float* g;
    void* o;
    float* slots;
    void* chunk_states;
    int32_t H, dk, dv, dtype;
    uint32_t flags;
    int32_t* dev_status;
    cudaStream_t stream;
};

struct BwdArgs {
    harts_la_tables_t tb;
    int32_t seq_lo, seq_hi;
    const void *q, *k, *v;
    const float* g;
    const void* dO;
    void *dq, *dk_, *dv_;
    float* dg;
    const void* chunk_states;
    void* scratch;
    int32_t H, dk, dv, dtype;
    uint32_t flags;
    int32_t* dev_status;
    cudaStream_t stream;
    // hand-off gradients summed in runs (HANDOFF_RUN): this range of slot_cons_seq are the launch's sequences, and each run's sum is left in
    // its first one's buffer (run_hi = 0: every sequence leaves its own); runs_below: the round after this one left its gradients so
    int32_t run_lo = 0, run_hi = 0;
    bool runs_below = false;
};

// Byte offsets inside the backward scratch buffer (each region 256-byte aligned).
struct ScratchLayout {
    size_t ds0;    // [n_seq, H, dk, dv] fp32: gradient w.r.t. each sequence's initial state
    size_t rk;     // [n_replay, H, dk] fp32: dk of replayed rows
    size_t rv;     // [n_replay, H, dv] fp32
    size_t rg;     // [n_replay, H] fp32
    size_t total;
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline ScratchLayout scratch_layout(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    ScratchLayout s;
    size_t off = 0;
    s.ds0 = off;
    off = align_up(off + (size_t)tb.n_seq * H * dk * dv * sizeof(float), 256);
    s.rk = off;
    off = align_up(off + (size_t)tb.n_replay * H * dk * sizeof(float), 256);
    s.rv = off;
    off = align_up(off + (size_t)tb.n_replay * H * dv * sizeof(float), 256);
    s.rg = off;
    off = align_up(off + (size_t)tb.n_replay * H * sizeof(float), 256);
    s.total = off < 256 ? 256 : off;
    return s;
}

// With HARTS_FLAG_CHECK_TABLES the kernels of a call run only while the status word is still zero: check_tables (a
// validation kernel ahead of them on the stream) records a bad index there, and nothing is dereferenced after it.
inline const int32_t* status_gate(uint32_t flags, const int32_t* dev_status) {
    return (flags & HARTS_FLAG_CHECK_TABLES) ? dev_status : nullptr;
}
#ifdef __CUDACC__
// A kernel that follows another one of the library in the same call is launched ahead of it (launch_after): its CTAs are on the
// SMs, and it waits here until that kernel is complete and its memory visible: before it writes anything, and before it reads anything
// but what the call was given (a call's first kernel is launched the ordinary way, so tables and inputs are complete).  Every CTA waits,
// also one without work, so that a kernel is complete only when all before it are.  A launch
// costs about a microsecond less so (nine kernels, 718 tokens x 1 head fp32: 77.6 -> 69.8 us a step; two to five kernels: 2 to 6 us).  In a kernel launched the ordinary way
// the wait does nothing.
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the kernel behind this one may come onto the SMs as soon as all CTAs of this one are there
__device__ __forceinline__ void let_next_launch() { asm volatile("griddepcontrol.launch_dependents;"); }
template <class... P, class... A>
inline cudaError_t launch_after(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchAttribute ahead{};
    ahead.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    ahead.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    c.attrs = &ahead;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ bool gate_closed(const int32_t* gate) {     // called by every thread of the CTA
    if (!gate) return false;
    __shared__ int closed;
    if (threadIdx.x == 0) closed = *reinterpret_cast<const volatile int32_t*>(gate);
    __syncthreads();
    return closed != 0;
}
#endif
int32_t check_tables(const harts_la_tables_t& tb, int32_t seq_lo, int32_t seq_hi, int32_t* dev_status, cudaStream_t stream);

// The same for the per-channel-decay calls: the replay-row gradient of g is a vector over the key channels.
struct GkScratchLayout {
    size_t ds0, rk, rv, rg, total;     // rg: [n_replay, H, dk] fp32
};
inline GkScratchLayout gk_scratch_layout(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    GkScratchLayout s;
    size_t off = 0;
    s.ds0 = off;
    off = align_up(off + (size_t)tb.n_seq * H * dk * dv * sizeof(float), 256);
    s.rk = off;
    off = align_up(off + (size_t)tb.n_replay * H * dk * sizeof(float), 256);
    s.rv = off;
    off = align_up(off + (size_t)tb.n_replay * H * dv * sizeof(float), 256);
    s.rg = off;
    off = align_up(off + (size_t)tb.n_replay * H * dk * sizeof(float), 256);
    s.total = off < 256 ? 256 : off;
    return s;
}

int32_t gk_supported(int32_t dtype, int32_t dk, int32_t dv);
int32_t gk_fwd(const FwdArgs& a);      // FwdArgs::g / BwdArgs::g, ::dg point to [rows, H, dk] arrays here
int32_t gk_bwd(const BwdArgs& a);
// bf16, d_k = d_v = 128: the dense products on the tensor cores (la_gk_mma.cu); taken unless HARTS_FLAG_FMA_KERNELS
int32_t gk_mma_supported(int32_t dtype, int32_t dk, int32_t dv);
int32_t gk_mma_fwd(const FwdArgs& a);
int32_t gk_mma_bwd(const BwdArgs& a);
int32_t gk_replay_reduce(const harts_la_tables_t& tb, void* dk_, void* dv_, float* dgk, const void* scratch, int32_t H,
                         int32_t dk, int32_t dv, int32_t dtype, cudaStream_t stream);

int32_t fma_supported(int32_t dtype, int32_t dk, int32_t dv);
int32_t fma_fwd(const FwdArgs& a);
int32_t fma_bwd(const BwdArgs& a);
int32_t tc_supported(int32_t dtype, int32_t dk, int32_t dv);
int32_t tc_fwd(const FwdArgs& a);
int32_t tc_fwd_fused(const FwdArgs& a, int* flags, int* ticket);     // all rounds in one launch

// Flags for the one-launch forms, kept behind the chunk states in the chunk-state workspace: one int32 per
// (slot, head) for the forward, one per (sequence, head) for the backward.
inline size_t chunk_state_payload(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv, size_t elem) {
    return align_up((size_t)tb.n_chunks * H * dk * dv * elem, 256);
}
// flags of the one-launch forms: n_slots * H (forward), n_seq * H (backward), then one ticket counter each
inline size_t fused_flag_count(const harts_la_tables_t& tb, int32_t H) { return ((size_t)tb.n_slots + tb.n_seq) * H; }
inline size_t fused_flag_bytes(const harts_la_tables_t& tb, int32_t H) {
    return align_up((fused_flag_count(tb, H) + 2) * sizeof(int32_t), 256);
}
// the plan's round table by value (kernel argument): sequences of round r (0-based) = [ptr[r], ptr[r + 1])
constexpr int MAX_FUSED_ROUNDS = 32;
constexpr int ONE_LAUNCH_ITEMS_PER_CTA = 8;    // the one-launch forms are offered up to this many items per resident CTA
struct RoundOrder {
    int n;
    int ptr[MAX_FUSED_ROUNDS + 1];
};
// Chunk-parallel path (bf16, d_k = d_v = 128): a scan leaves the state of every chunk boundary (backward: its gradient) in
// memory, then every (chunk, head) is a work item of its own.
int32_t scan_fwd(const FwdArgs& a, int* flags, const RoundOrder& order);      // la_scan.cu: states, exported slots
int32_t scan_bwd(const BwdArgs& a, void* ds_tiles, float* dots, int* flags, const RoundOrder& order);   // their gradients, ds0 hand-off
int32_t chunk_fwd(const FwdArgs& a);                           // la_chunk_fwd.cu
int32_t chunk_bwd(const BwdArgs& a, const void* ds_tiles, const float* dots);     // la_chunk_bwd.cu
// Taken up to 28,672 (chunk, head) items and 640 (sequence, head) pairs, with fewer than four chunks a sequence up to 128 pairs,
// or 1,152 where two sequences and more start from each exported state (fans).
// The walk kernels (la_tc_*.cu) move 240 KB per item in a whole step, this path 430 KB: with enough chains to fill the GPU the walk
// wins, with few the chain of its 3-6 us chunks is what takes the time.  Walk / chunk-parallel, time of a step (of the forward
// alone), 46 forests both ways with cold inputs:
//   inside the line the chunk path won everywhere: 304 chunks x 4 heads 2.8 (2.9); agentic 16,736 items, 384 pairs 1.78 (1.96);
//     25,576 items, 632 pairs 1.15 (1.34); 28,668 items, 636 pairs 1.20 (1.34); branchy 7,296 items, 624 pairs 1.16 (1.10);
//     replay fans, 422 items, 254 pairs 3.5 (2.9; gate per channel 3.4); 645 items, 393 pairs 3.4; 782 items, 478 pairs 3.3; 1,564
//     items, 956 pairs 2.5; beyond the line 3,128 items, 1,912 pairs 0.95, 6,256 items, 3,824 pairs 0.83 (up to 1,184 pairs the walk
//     runs all rounds in one launch, and one CTA sums all gradients of a boundary; the scan reads them 512 bytes at a time)
//   just outside it still won on agentic trees (28,144 items, 736 pairs 1.12 (1.26); 33,472 items, 768 pairs 1.05 (1.20)): the
//     line is on the safe side there
//   further out the walk wins: branchy 9,728 items, 832 pairs 0.97 (0.86); 24,768 items, 2,328 pairs 0.89 (0.76); agentic 51,152
//     items, 1,264 pairs 0.94 (0.90); 6,949 chunks of replay fans x 16 heads 0.65
// The line depends on the tables' totals only, so that a round issued alone takes the path of the whole.
constexpr int64_t CHUNK_PARALLEL_MAX = 28672, CHUNK_PARALLEL_CHAINS = 640, CHUNK_PARALLEL_FANS = 1152, CHUNK_PARALLEL_FEW = 128;
inline bool chunk_parallel(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv, int32_t dtype, uint32_t flags) {
    const int64_t chains = (int64_t)tb.n_seq * H;
    const bool fans = tb.n_slots > 0 && tb.n_seq >= 2 * (int64_t)tb.n_slots;
    return !(flags & HARTS_FLAG_FMA_KERNELS) && dtype == HARTS_BF16 && dk == 128 && dv == 128 &&
           (int64_t)tb.n_chunks * H <= CHUNK_PARALLEL_MAX &&
           chains <= (tb.n_chunks >= 4 * (int64_t)tb.n_seq ? CHUNK_PARALLEL_CHAINS : fans ? CHUNK_PARALLEL_FANS : CHUNK_PARALLEL_FEW);
}
// The pipelined forward walk (la_pipe_fwd.cu) wherever sequences have four chunks and more on average and their (sequence, head) pairs
// give every SM one, and in place of the synchronous walk also with fewer.  Time of a forward, other path / this one, cold inputs, 47
// forests: agentic 192 pairs 1.07, 384 pairs 1.23, 688 1.84, 768 1.65, 3,360 1.19; branchy 314 pairs 1.26, 436 1.24, 480 1.39, 5,024
// 1.35, 10,048 1.15.  With fewer pairs the chain of chunks decides, and the scan's 32-column slices take 0.55 us a step against 1.1:
// agentic 172 pairs 0.90, 96 pairs 0.74, 24 pairs 0.56 (120 branchy pairs 0.84).  Sequences of one or two chunks are bound by their
// start states, which the synchronous walk's two CTAs per SM overlap: replay fans, 17,088 pairs 0.97, 68,128 pairs 0.89.
// The backward has a line of its own (chunk_parallel): the chunk states are the same whoever wrote them.
constexpr int64_t PIPE_PAIRS = 192;
inline bool pipe_forward(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv, int32_t dtype, uint32_t flags) {
    return !(flags & HARTS_FLAG_FMA_KERNELS) && dtype == HARTS_BF16 && dk == 128 && dv == 128 && tb.n_chunks >= 4 * (int64_t)tb.n_seq &&
           ((int64_t)tb.n_seq * H >= PIPE_PAIRS || !chunk_parallel(tb, H, dk, dv, dtype, flags));
}
int32_t pipe_fwd(const FwdArgs& a, int* flags, int first_round);
// the boundary-state gradients of the chunk-parallel backward: bf16 [n_chunks, H, dk, dv] behind the flags, then
// <S_c, dS_c> in parts, fp32 [n_chunks, H, 4 blocks of 32 columns, dk], then the scan's ticket and counters
inline size_t ds_tiles_offset(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return align_up(chunk_state_payload(tb, H, dk, dv, 2) + fused_flag_bytes(tb, H), 1024);
}
inline size_t dots_offset(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return ds_tiles_offset(tb, H, dk, dv) + align_up(chunk_state_payload(tb, H, dk, dv, 2), 1024);
}
inline size_t scan_flags_offset(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return dots_offset(tb, H, dk, dv) + (size_t)tb.n_chunks * H * (dv / 32) * dk * sizeof(float);
}
inline size_t chunk_parallel_bytes(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return scan_flags_offset(tb, H, dk, dv) + (4 + (size_t)(tb.n_seq > tb.n_slots ? tb.n_seq : tb.n_slots) * H * 4) * sizeof(int);
}
// The same for the per-channel decay, under the same rule.  Walk / chunk-parallel, forward + backward: inside the line 1.16 (branchy
// 7,296 items, 624 pairs) to 4.0, 1.34 at 28,668 items; outside it the chunk path is ahead up to 51,152 items of agentic trees
// (1.12) and behind on branchy ones (9,728 items, 832 pairs: 0.97).
int32_t gk_scan_fwd(const FwdArgs& a, int* flags, const RoundOrder& order);
int32_t gk_scan_bwd(const BwdArgs& a, void* ds_tiles, float* dots, int* flags, const RoundOrder& order);
int32_t gk_chunk_fwd(const FwdArgs& a);
int32_t gk_chunk_bwd(const BwdArgs& a, const void* ds_tiles, const float* dots);
// The same for fp32 inputs, d_k = d_v = 64 (la_f32.cu): every problem that brings a chunk-state workspace (3.5 to 35 times as fast
// as the walk from 13 to 12,880 items, agentic, branchy and replay; least on short sequences).  extra: e^{b_n}
// [n_chunks, H] and the gradients of the boundary states [n_chunks, H, dk, dv], fp32, behind the flags.
inline bool f32_chunks(int32_t dk, int32_t dv, int32_t dtype) { return dtype == HARTS_FP32 && dk == 64 && dv == 64; }
inline size_t f32_extra_offset(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return chunk_state_payload(tb, H, dk, dv, 4) + fused_flag_bytes(tb, H);
}
inline size_t f32_extra_bytes(const harts_la_tables_t& tb, int32_t H, int32_t dk, int32_t dv) {
    return align_up((size_t)tb.n_chunks * H, 64) * sizeof(float) + chunk_state_payload(tb, H, dk, dv, 4);
}
int32_t f32_fwd(const FwdArgs& a, float* extra, const int32_t* range, int32_t n);
int32_t f32_bwd(const BwdArgs& a, float* extra, const int32_t* range, int32_t n);
int32_t gk_mma_fwd_all(const FwdArgs& a, int* flags, int* ticket);     // all rounds in one launch (la_gk_mma.cu)
int32_t gk_mma_bwd_all(const BwdArgs& a, int* flags, int* ticket, const RoundOrder& rounds);
int32_t tc_bwd(const BwdArgs& a);
int32_t tc_bwd_fused(const BwdArgs& a, int* flags, int* ticket, const RoundOrder& rounds);   // all rounds in one launch
// The tensor-core walk sums the gradients of a boundary's consumers in runs -- the positions of slot_cons_seq from one multiple of HANDOFF_RUN
// to the next -- and then the runs, both in table order, whoever does it.  Elsewhere (run = 1) one after the other.
constexpr int HANDOFF_RUN = 8;
int sm_count();
int32_t handoff_reduce(const BwdArgs& a, int run = 1);
int32_t replay_reduce(const harts_la_tables_t& tb, void* dk_, void* dv_, float* dg, const void* scratch, int32_t H,
                      int32_t dk, int32_t dv, int32_t dtype, cudaStream_t stream);

}  // namespace harts
