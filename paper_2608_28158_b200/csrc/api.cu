// C ABI: argument checks, kernel selection and launches.  No device memory is allocated here.
#include "kernels.h"
#include "plan.h"

namespace {

inline bool misaligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) != 0; }

int32_t check_common(const harts_la_tables_t* tb, int32_t seq_lo, int32_t seq_hi, int32_t H, int32_t dk, int32_t dv,
                     int32_t dtype) {
    if (!tb) return HARTS_EINVAL;
    if (seq_lo < 0 || seq_hi < seq_lo || seq_hi > tb->n_seq) return HARTS_EINVAL;
    if (H < 1 || dk < 1 || dv < 1) return HARTS_EINVAL;
    if (dtype != HARTS_FP32 && dtype != HARTS_BF16) return HARTS_EUNSUPPORTED;
    if (tb->chunk != 64) return HARTS_EUNSUPPORTED;
    if (!harts::fma_supported(dtype, dk, dv)) return HARTS_EUNSUPPORTED;
    if (!tb->seq_own_begin || !tb->seq_init_slot || !tb->seq_replay_ptr || !tb->replay_row || !tb->seq_req_ptr ||
        !tb->slot_chunk || !tb->seq_chunk_ptr || !tb->slot_cons_ptr || !tb->slot_cons_seq || !tb->rg_row ||
        !tb->rg_ptr || !tb->rg_entry)
        return HARTS_EINVAL;
    return HARTS_OK;
}

// The tensor-core kernels serve bf16 with d_k = d_v = 128 unless the caller asks for the FMA kernels.
inline bool use_tc(int32_t dtype, int32_t dk, int32_t dv, uint32_t flags) {
    return !(flags & HARTS_FLAG_FMA_KERNELS) && harts::tc_supported(dtype, dk, dv);
}

float* f32_extra(const harts_la_tables_t& tb, const void* chunk_states, int32_t H, int32_t dk, int32_t dv) {
    return reinterpret_cast<float*>(const_cast<char*>(static_cast<const char*>(chunk_states)) + harts::f32_extra_offset(tb, H, dk, dv));
}
// Whether round r of the walk backward sums its hand-off gradients in runs, and the positions of slot_cons_seq that its sequences are.  Where
// sequences are short a 64 KB gradient each is what a round writes and the next reads; in runs of eight it is an eighth of that (171,829
// replay tokens x 16 heads, 4,258 sequences of one to three chunks: reductions 759 -> 187 us, walk 5,580 -> 5,767, a step 9,644 -> 9,240; in runs
// of sixteen 134, 5,893 and 9,334).  Not where sequences are long, whose dealing by length matters
// more, nor where the runs would be fewer than four an SM.  Only inside a call for all rounds: a round issued alone leaves every sequence's own.
bool handoff_runs(const harts::Plan& p, const harts_la_tables_t& tb, int32_t r, int32_t H, int32_t (&run)[2]) {
    const int32_t lo = p.round_seq_ptr[r - 1], hi = p.round_seq_ptr[r];
    if (tb.n_chunks >= 4 * (int64_t)tb.n_seq || (int64_t)(hi - lo) * H < 4 * harts::HANDOFF_RUN * (int64_t)harts::sm_count()) return false;
    int32_t first = tb.n_slots, last = -1;
    for (int32_t s = lo; s < hi; s++) {
        if (p.seq_init_slot[s] < 0) return false;
        first = p.seq_init_slot[s] < first ? p.seq_init_slot[s] : first;
        last = p.seq_init_slot[s] > last ? p.seq_init_slot[s] : last;
    }
    if (p.slot_cons_ptr[last + 1] - p.slot_cons_ptr[first] != hi - lo) return false;
    run[0] = p.slot_cons_ptr[first];
    run[1] = p.slot_cons_ptr[last + 1];
    return true;
}
// Chunk-parallel path over sequences [range[0], range[n]), range[r]..range[r+1] per round: the scan, then all chunks at once.
harts::RoundOrder round_order(const int32_t* range, int32_t n) {
    harts::RoundOrder ro;
    ro.n = n > 1 ? n : 0;
    for (int32_t r = 0; r <= n; r++) ro.ptr[r] = range[r];
    return ro;
}
int32_t chunk_parallel_fwd(harts::FwdArgs a, const int32_t* range, int32_t n) {
    a.seq_lo = range[0];
    a.seq_hi = range[n];
    int* flags = reinterpret_cast<int*>(static_cast<char*>(a.chunk_states) + harts::scan_flags_offset(a.tb, a.H, a.dk, a.dv));
    const int32_t rc = harts::scan_fwd(a, flags, round_order(range, n));
    return rc != HARTS_OK ? rc : harts::chunk_fwd(a);
}
int32_t chunk_parallel_bwd(harts::BwdArgs a, const int32_t* range, int32_t n) {
    a.seq_lo = range[0];
    a.seq_hi = range[n];
    char* ws = const_cast<char*>(static_cast<const char*>(a.chunk_states));
    void* ds = ws + harts::ds_tiles_offset(a.tb, a.H, a.dk, a.dv);
    int* flags = reinterpret_cast<int*>(ws + harts::scan_flags_offset(a.tb, a.H, a.dk, a.dv));
    float* dots = reinterpret_cast<float*>(ws + harts::dots_offset(a.tb, a.H, a.dk, a.dv));
    const int32_t rc = harts::scan_bwd(a, ds, dots, flags, round_order(range, n));
    return rc != HARTS_OK ? rc : harts::chunk_bwd(a, ds, dots);
}

int32_t gk_chunk_parallel_fwd(harts::FwdArgs a, const int32_t* range, int32_t n) {
    a.seq_lo = range[0];
    a.seq_hi = range[n];
    int* flags = reinterpret_cast<int*>(static_cast<char*>(a.chunk_states) + harts::scan_flags_offset(a.tb, a.H, a.dk, a.dv));
    const int32_t rc = harts::gk_scan_fwd(a, flags, round_order(range, n));
    return rc != HARTS_OK ? rc : harts::gk_chunk_fwd(a);
}
int32_t gk_chunk_parallel_bwd(harts::BwdArgs a, const int32_t* range, int32_t n) {
    a.seq_lo = range[0];
    a.seq_hi = range[n];
    char* ws = const_cast<char*>(static_cast<const char*>(a.chunk_states));
    void* ds = ws + harts::ds_tiles_offset(a.tb, a.H, a.dk, a.dv);
    int* flags = reinterpret_cast<int*>(ws + harts::scan_flags_offset(a.tb, a.H, a.dk, a.dv));
    float* dots = reinterpret_cast<float*>(ws + harts::dots_offset(a.tb, a.H, a.dk, a.dv));
    const int32_t rc = harts::gk_scan_bwd(a, ds, dots, flags, round_order(range, n));
    return rc != HARTS_OK ? rc : harts::gk_chunk_bwd(a, ds, dots);
}

}  // namespace

extern "C" {

const char* harts_la_strerror(int32_t code) {
    switch (code) {
        case HARTS_OK: return "ok";
        case HARTS_EINVAL: return "invalid argument";
        case HARTS_ENOMEM: return "out of host memory";
        case HARTS_EUNSUPPORTED: return "unsupported dtype / head dimension / chunk size";
        case HARTS_ETIMEOUT: return "a bounded device-side wait ran out";
        case HARTS_EINTERNAL: return "internal error";
        case HARTS_ECUDA: return "CUDA call failed";
        case HARTS_ESCRATCH: return "scratch need exceeds the library's fixed scratch array";
        default: return "unknown status";
    }
}

int32_t harts_la_plan_upload(const harts_la_plan_t* plan, void* dev_blob, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || !dev_blob || misaligned(dev_blob)) return HARTS_EINVAL;
    cudaError_t e = cudaMemcpyAsync(dev_blob, p->blob.data(), p->blob.size() * sizeof(int32_t), cudaMemcpyHostToDevice,
                                    static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? HARTS_OK : HARTS_ECUDA;
}

int32_t harts_la_workspace_bytes(const harts_la_tables_t* tb, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                                 uint32_t flags, size_t* chunk_state_bytes, size_t* scratch_bytes) {
    if (!tb || H < 1 || dk < 1 || dv < 1) return HARTS_EINVAL;
    if (dtype != HARTS_FP32 && dtype != HARTS_BF16) return HARTS_EUNSUPPORTED;
    size_t elem = dtype == HARTS_FP32 ? 4 : 2;
    (void)flags;
    if (chunk_state_bytes) {    // the states, then the flags of the one-launch forms, then what the chunk-parallel path adds
        *chunk_state_bytes = harts::chunk_state_payload(*tb, H, dk, dv, elem) + harts::fused_flag_bytes(*tb, H);
        if (harts::f32_chunks(dk, dv, dtype)) *chunk_state_bytes += harts::f32_extra_bytes(*tb, H, dk, dv);
        if (harts::chunk_parallel(*tb, H, dk, dv, dtype, 0)) *chunk_state_bytes = harts::chunk_parallel_bytes(*tb, H, dk, dv);
    }
    if (scratch_bytes) *scratch_bytes = harts::scratch_layout(*tb, H, dk, dv).total;
    return HARTS_OK;
}

int32_t harts_la_fwd_seqs(const harts_la_tables_t* tb, int32_t seq_lo, int32_t seq_hi, const void* q, const void* k,
                          const void* v, const float* g, void* o, float* slots, void* chunk_states, int32_t H,
                          int32_t dk, int32_t dv, int32_t dtype, uint32_t flags, int32_t* dev_status, void* stream) {
    int32_t rc = check_common(tb, seq_lo, seq_hi, H, dk, dv, dtype);
    if (rc != HARTS_OK) return rc;
    if (!q || !k || !v || !g || !o || (tb->n_slots > 0 && !slots)) return HARTS_EINVAL;
    if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(g) || misaligned(o) || misaligned(slots) ||
        misaligned(chunk_states))
        return HARTS_EINVAL;
    harts::FwdArgs a{*tb, seq_lo, seq_hi, q, k, v, g, o, slots, chunk_states, H, dk, dv, dtype, flags, dev_status,
                     static_cast<cudaStream_t>(stream)};
    if (flags & HARTS_FLAG_CHECK_TABLES)
        if ((rc = harts::check_tables(*tb, seq_lo, seq_hi, dev_status, a.stream)) != HARTS_OK) return rc;
    const int32_t range[2] = {seq_lo, seq_hi};
    if (chunk_states && harts::f32_chunks(dk, dv, dtype)) return harts::f32_fwd(a, f32_extra(a.tb, chunk_states, H, dk, dv), range, 1);
    if (harts::pipe_forward(*tb, H, dk, dv, dtype, flags)) return harts::pipe_fwd(a, nullptr, 0);
    if (chunk_states && harts::chunk_parallel(*tb, H, dk, dv, dtype, flags)) return chunk_parallel_fwd(a, range, 1);
    if (use_tc(dtype, dk, dv, flags)) return harts::tc_fwd(a);
    return harts::fma_fwd(a);
}

static int32_t bwd_seqs(const harts_la_tables_t* tb, int32_t seq_lo, int32_t seq_hi, const void* q, const void* k,
                        const void* v, const float* g, const void* dO, void* dq, void* dk_, void* dv_, float* dg,
                        const void* chunk_states, void* scratch, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                        uint32_t flags, int32_t* dev_status, void* stream, int32_t run_lo, int32_t run_hi, bool runs_below) {
    int32_t rc = check_common(tb, seq_lo, seq_hi, H, dk, dv, dtype);
    if (rc != HARTS_OK) return rc;
    if (!q || !k || !v || !g || !dO || !dq || !dk_ || !dv_ || !dg || !chunk_states || !scratch) return HARTS_EINVAL;
    if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(g) || misaligned(dO) || misaligned(dq) ||
        misaligned(dk_) || misaligned(dv_) || misaligned(dg) || misaligned(chunk_states) || misaligned(scratch))
        return HARTS_EINVAL;
    harts::BwdArgs a{*tb, seq_lo, seq_hi, q, k, v, g, dO, dq, dk_, dv_, dg, chunk_states, scratch, H, dk, dv, dtype,
                     flags, dev_status, static_cast<cudaStream_t>(stream), run_lo, run_hi, runs_below};
    if (flags & HARTS_FLAG_CHECK_TABLES)
        if ((rc = harts::check_tables(*tb, seq_lo, seq_hi, dev_status, a.stream)) != HARTS_OK) return rc;
    const int32_t range[2] = {seq_lo, seq_hi};
    if (harts::f32_chunks(dk, dv, dtype)) return harts::f32_bwd(a, f32_extra(a.tb, chunk_states, H, dk, dv), range, 1);
    if (harts::chunk_parallel(*tb, H, dk, dv, dtype, flags)) return chunk_parallel_bwd(a, range, 1);
    if (use_tc(dtype, dk, dv, flags)) return harts::tc_bwd(a);
    return harts::fma_bwd(a);
}

int32_t harts_la_bwd_seqs(const harts_la_tables_t* tb, int32_t seq_lo, int32_t seq_hi, const void* q, const void* k,
                          const void* v, const float* g, const void* dO, void* dq, void* dk_, void* dv_, float* dg,
                          const void* chunk_states, void* scratch, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                          uint32_t flags, int32_t* dev_status, void* stream) {
    return bwd_seqs(tb, seq_lo, seq_hi, q, k, v, g, dO, dq, dk_, dv_, dg, chunk_states, scratch, H, dk, dv, dtype, flags, dev_status, stream, 0, 0, false);
}

int32_t harts_la_bwd_finish(const harts_la_tables_t* tb, void* dk_, void* dv_, float* dg, const void* scratch,
                            int32_t H, int32_t dk, int32_t dv, int32_t dtype, void* stream) {
    int32_t rc = check_common(tb, 0, 0, H, dk, dv, dtype);
    if (rc != HARTS_OK) return rc;
    if (!dk_ || !dv_ || !dg || !scratch) return HARTS_EINVAL;
    return harts::replay_reduce(*tb, dk_, dv_, dg, scratch, H, dk, dv, dtype, static_cast<cudaStream_t>(stream));
}

int32_t harts_la_fwd(const harts_la_plan_t* plan, const void* dev_blob, int32_t round, const void* q, const void* k,
                     const void* v, const float* g, void* o, float* slots, void* chunk_states, int32_t H, int32_t dk,
                     int32_t dv, int32_t dtype, uint32_t flags, int32_t* dev_status, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || round < 0 || round > p->n_rounds) return HARTS_EINVAL;
    harts_la_tables_t tb;
    int32_t rc = harts_la_plan_tables(plan, dev_blob, &tb);
    if (rc != HARTS_OK) return rc;
    int32_t r0 = round == 0 ? 1 : round, r1 = round == 0 ? p->n_rounds : round;
    if (round == 0 && p->n_rounds > 1 && p->n_rounds <= harts::MAX_FUSED_ROUNDS && chunk_states &&
        !(flags & HARTS_FLAG_ROUND_LAUNCHES) &&
        (use_tc(dtype, dk, dv, flags) || harts::f32_chunks(dk, dv, dtype))) {
        // every round in one launch: a sequence waits for the flag of the state it starts from instead of for the
        // end of the previous round's kernel
        rc = check_common(&tb, 0, tb.n_seq, H, dk, dv, dtype);
        if (rc != HARTS_OK) return rc;
        if (!q || !k || !v || !g || !o || (tb.n_slots > 0 && !slots)) return HARTS_EINVAL;
        if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(g) || misaligned(o) || misaligned(slots) ||
            misaligned(chunk_states))
            return HARTS_EINVAL;
        harts::FwdArgs a{tb, 0, tb.n_seq, q, k, v, g, o, slots, chunk_states, H, dk, dv, dtype, flags, dev_status,
                         static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES) {
            if (!dev_status) return HARTS_EINVAL;
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        }
        if (harts::f32_chunks(dk, dv, dtype))
            return harts::f32_fwd(a, f32_extra(tb, chunk_states, H, dk, dv), p->round_seq_ptr.data(), p->n_rounds);
        if (harts::pipe_forward(tb, H, dk, dv, dtype, flags))
            return harts::pipe_fwd(a, reinterpret_cast<int*>(static_cast<char*>(chunk_states) + harts::chunk_state_payload(tb, H, dk, dv, 2)),
                                   p->round_seq_ptr[1] - p->round_seq_ptr[0]);
        if (harts::chunk_parallel(tb, H, dk, dv, dtype, flags))
            return chunk_parallel_fwd(a, p->round_seq_ptr.data(), p->n_rounds);
        int* fl = reinterpret_cast<int*>(static_cast<char*>(chunk_states) + harts::chunk_state_payload(tb, H, dk, dv, 2));
        rc = harts::tc_fwd_fused(a, fl, fl + harts::fused_flag_count(tb, H));
        if (rc != HARTS_EUNSUPPORTED) return rc;         // else: not all CTAs can be resident, launch round by round
    }
    for (int32_t r = r0; r <= r1; r++) {
        rc = harts_la_fwd_seqs(&tb, p->round_seq_ptr[r - 1], p->round_seq_ptr[r], q, k, v, g, o, slots, chunk_states,
                               H, dk, dv, dtype, flags, dev_status, stream);
        if (rc != HARTS_OK) return rc;
    }
    return HARTS_OK;
}

int32_t harts_la_bwd(const harts_la_plan_t* plan, const void* dev_blob, int32_t round, const void* q, const void* k,
                     const void* v, const float* g, const void* dO, void* dq, void* dk_, void* dv_, float* dg,
                     const void* chunk_states, void* scratch, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                     uint32_t flags, int32_t* dev_status, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || round < 0 || round > p->n_rounds) return HARTS_EINVAL;
    harts_la_tables_t tb;
    int32_t rc = harts_la_plan_tables(plan, dev_blob, &tb);
    if (rc != HARTS_OK) return rc;
    int32_t r1 = round == 0 ? p->n_rounds : round, r0 = round == 0 ? 1 : round;
    bool done = false;
    if (round == 0 && p->n_rounds > 1 && p->n_rounds <= harts::MAX_FUSED_ROUNDS && !(flags & HARTS_FLAG_ROUND_LAUNCHES) &&
        (use_tc(dtype, dk, dv, flags) || harts::f32_chunks(dk, dv, dtype))) {
        rc = check_common(&tb, 0, tb.n_seq, H, dk, dv, dtype);
        if (rc != HARTS_OK) return rc;
        if (!q || !k || !v || !g || !dO || !dq || !dk_ || !dv_ || !dg || !chunk_states || !scratch) return HARTS_EINVAL;
        if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(g) || misaligned(dO) || misaligned(dq) ||
            misaligned(dk_) || misaligned(dv_) || misaligned(dg) || misaligned(chunk_states) || misaligned(scratch))
            return HARTS_EINVAL;
        harts::BwdArgs a{tb, 0, tb.n_seq, q, k, v, g, dO, dq, dk_, dv_, dg, chunk_states, scratch, H, dk, dv, dtype, flags,
                         dev_status, static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES) {
            if (!dev_status) return HARTS_EINVAL;
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        }
        if (harts::f32_chunks(dk, dv, dtype)) {
            rc = harts::f32_bwd(a, f32_extra(tb, chunk_states, H, dk, dv), p->round_seq_ptr.data(), p->n_rounds);
            if (rc != HARTS_OK) return rc;
            return harts_la_bwd_finish(&tb, dk_, dv_, dg, scratch, H, dk, dv, dtype, stream);
        }
        if (harts::chunk_parallel(tb, H, dk, dv, dtype, flags)) {
            if ((rc = chunk_parallel_bwd(a, p->round_seq_ptr.data(), p->n_rounds)) != HARTS_OK) return rc;
            return harts_la_bwd_finish(&tb, dk_, dv_, dg, scratch, H, dk, dv, dtype, stream);
        }
        // the flags sit behind the chunk states; the backward's come after the forward's (n_slots * H), the two
        // ticket counters after both
        int* fl = reinterpret_cast<int*>(const_cast<char*>(static_cast<const char*>(chunk_states)) +
                                         harts::chunk_state_payload(tb, H, dk, dv, 2));
        harts::RoundOrder ro;
        ro.n = p->n_rounds;
        for (int32_t r = 0; r <= p->n_rounds; r++) ro.ptr[r] = p->round_seq_ptr[r];
        rc = harts::tc_bwd_fused(a, fl + (size_t)tb.n_slots * H, fl + harts::fused_flag_count(tb, H) + 1, ro);
        if (rc == HARTS_OK) done = true;
        else if (rc != HARTS_EUNSUPPORTED) return rc;
    }
    bool runs_below = false;
    for (int32_t r = r1; r >= r0 && !done; r--) {
        int32_t run[2] = {0, 0};
        const bool runs = round == 0 && use_tc(dtype, dk, dv, flags) && handoff_runs(*p, tb, r, H, run);
        rc = bwd_seqs(&tb, p->round_seq_ptr[r - 1], p->round_seq_ptr[r], q, k, v, g, dO, dq, dk_, dv_, dg, chunk_states, scratch, H, dk, dv, dtype, flags,
                      dev_status, stream, run[0], run[1], runs_below);
        if (rc != HARTS_OK) return rc;
        runs_below = runs;
    }
    if (r0 == 1) return harts_la_bwd_finish(&tb, dk_, dv_, dg, scratch, H, dk, dv, dtype, stream);
    return HARTS_OK;
}

int32_t harts_la_step_host(const harts_la_plan_t* plan, const void* dev_blob, const void* host_q, const void* host_k,
                           const void* host_v, const float* host_g, const void* host_dO, void* host_o, void* host_dq,
                           void* host_dk, void* host_dv, float* host_dg, void* dev_q, void* dev_k, void* dev_v,
                           float* dev_g, void* dev_dO, void* dev_o, void* dev_dq, void* dev_dk, void* dev_dv,
                           float* dev_dg, float* slots, void* chunk_states, void* scratch, int32_t H, int32_t dk,
                           int32_t dv, int32_t dtype, uint32_t flags, int32_t* dev_status, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || H < 1 || dk < 1 || dv < 1) return HARTS_EINVAL;
    if (dtype != HARTS_FP32 && dtype != HARTS_BF16) return HARTS_EUNSUPPORTED;
    if (!host_q || !host_k || !host_v || !host_g || !host_dO || !host_o || !host_dq || !host_dk || !host_dv || !host_dg)
        return HARTS_EINVAL;
    const size_t elem = dtype == HARTS_FP32 ? 4 : 2, rows = (size_t)p->n_rows * H;
    const size_t nk = rows * dk * elem, nv = rows * dv * elem, ng = rows * sizeof(float);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const struct { void* dst; const void* src; size_t n; } in[5] = {
        {dev_q, host_q, nk}, {dev_k, host_k, nk}, {dev_v, host_v, nv}, {dev_g, host_g, ng}, {dev_dO, host_dO, nv}};
    for (const auto& c : in) {
        if (!c.dst) return HARTS_EINVAL;
        if (cudaMemcpyAsync(c.dst, c.src, c.n, cudaMemcpyHostToDevice, s) != cudaSuccess) return HARTS_ECUDA;
    }
    int32_t rc = harts_la_fwd(plan, dev_blob, 0, dev_q, dev_k, dev_v, dev_g, dev_o, slots, chunk_states, H, dk, dv, dtype,
                              flags, dev_status, stream);
    if (rc != HARTS_OK) return rc;
    rc = harts_la_bwd(plan, dev_blob, 0, dev_q, dev_k, dev_v, dev_g, dev_dO, dev_dq, dev_dk, dev_dv, dev_dg, chunk_states,
                      scratch, H, dk, dv, dtype, flags, dev_status, stream);
    if (rc != HARTS_OK) return rc;
    const struct { void* dst; const void* src; size_t n; } out[5] = {
        {host_o, dev_o, nv}, {host_dq, dev_dq, nk}, {host_dk, dev_dk, nk}, {host_dv, dev_dv, nv}, {host_dg, dev_dg, ng}};
    for (const auto& c : out)
        if (cudaMemcpyAsync(c.dst, c.src, c.n, cudaMemcpyDeviceToHost, s) != cudaSuccess) return HARTS_ECUDA;
    return HARTS_OK;
}

// ---- per-channel decay (the Diag(gamma) term of Eq. 1) -------------------------------------------------------------------
int32_t harts_la_gk_workspace_bytes(const harts_la_tables_t* tb, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                                    size_t* chunk_state_bytes, size_t* scratch_bytes) {
    if (!tb || H < 1 || dk < 1 || dv < 1) return HARTS_EINVAL;
    if (dtype != HARTS_FP32 && dtype != HARTS_BF16) return HARTS_EUNSUPPORTED;
    const size_t elem = dtype == HARTS_FP32 ? 4 : 2;
    if (chunk_state_bytes)      // the states, then the flags of the one-launch forms
        *chunk_state_bytes = harts::chunk_state_payload(*tb, H, dk, dv, elem) + harts::fused_flag_bytes(*tb, H);
    if (chunk_state_bytes && harts::chunk_parallel(*tb, H, dk, dv, dtype, 0))
        *chunk_state_bytes = harts::chunk_parallel_bytes(*tb, H, dk, dv);
    if (scratch_bytes) *scratch_bytes = harts::gk_scratch_layout(*tb, H, dk, dv).total;
    return HARTS_OK;
}

int32_t harts_la_gk_fwd(const harts_la_plan_t* plan, const void* dev_blob, int32_t round, const void* q, const void* k,
                        const void* v, const float* gk, void* o, float* slots, void* chunk_states, int32_t H, int32_t dk,
                        int32_t dv, int32_t dtype, uint32_t flags, int32_t* dev_status, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || round < 0 || round > p->n_rounds) return HARTS_EINVAL;
    harts_la_tables_t tb;
    int32_t rc = harts_la_plan_tables(plan, dev_blob, &tb);
    if (rc != HARTS_OK) return rc;
    if (H < 1 || tb.chunk != 64 || !harts::gk_supported(dtype, dk, dv)) return H < 1 ? HARTS_EINVAL : HARTS_EUNSUPPORTED;
    if (!q || !k || !v || !gk || !o || (tb.n_slots > 0 && !slots)) return HARTS_EINVAL;
    if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(gk) || misaligned(o) || misaligned(slots) ||
        misaligned(chunk_states))
        return HARTS_EINVAL;
    if ((flags & HARTS_FLAG_CHECK_TABLES) && !dev_status) return HARTS_EINVAL;
    const int32_t r0 = round == 0 ? 1 : round, r1 = round == 0 ? p->n_rounds : round;
    const bool chunks = chunk_states && harts::chunk_parallel(tb, H, dk, dv, dtype, flags);
    if (chunks && round == 0 && p->n_rounds <= harts::MAX_FUSED_ROUNDS && !(flags & HARTS_FLAG_ROUND_LAUNCHES)) {
        harts::FwdArgs a{tb, 0, tb.n_seq, q, k, v, gk, o, slots, chunk_states, H, dk, dv, dtype, flags, dev_status,
                         static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        return gk_chunk_parallel_fwd(a, p->round_seq_ptr.data(), p->n_rounds);
    }
    const bool one_launch = !chunks && round == 0 && p->n_rounds > 1 && p->n_rounds <= harts::MAX_FUSED_ROUNDS && chunk_states &&
                            !(flags & (HARTS_FLAG_ROUND_LAUNCHES | HARTS_FLAG_FMA_KERNELS)) &&
                            harts::gk_mma_supported(dtype, dk, dv);
    if (one_launch) {           // flags and tickets sit behind the chunk states, as for the scalar-gate calls
        harts::FwdArgs a{tb, 0, tb.n_seq, q, k, v, gk, o, slots, chunk_states, H, dk, dv, dtype, flags, dev_status,
                         static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        int* fl = reinterpret_cast<int*>(static_cast<char*>(chunk_states) + harts::chunk_state_payload(tb, H, dk, dv, 2));
        rc = harts::gk_mma_fwd_all(a, fl, fl + harts::fused_flag_count(tb, H));
        if (rc != HARTS_EUNSUPPORTED) return rc;
    }
    for (int32_t r = r0; r <= r1; r++) {
        harts::FwdArgs a{tb, p->round_seq_ptr[r - 1], p->round_seq_ptr[r], q, k, v, gk, o, slots, chunk_states, H, dk, dv,
                         dtype, flags, dev_status, static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, a.seq_lo, a.seq_hi, dev_status, a.stream)) != HARTS_OK) return rc;
        if ((rc = chunks ? gk_chunk_parallel_fwd(a, &p->round_seq_ptr[r - 1], 1) : harts::gk_fwd(a)) != HARTS_OK) return rc;
    }
    return HARTS_OK;
}

int32_t harts_la_gk_bwd(const harts_la_plan_t* plan, const void* dev_blob, int32_t round, const void* q, const void* k,
                        const void* v, const float* gk, const void* dO, void* dq, void* dk_, void* dv_, float* dgk,
                        const void* chunk_states, void* scratch, int32_t H, int32_t dk, int32_t dv, int32_t dtype,
                        uint32_t flags, int32_t* dev_status, void* stream) {
    const harts::Plan* p = harts_la_plan_internal(plan);
    if (!p || round < 0 || round > p->n_rounds) return HARTS_EINVAL;
    harts_la_tables_t tb;
    int32_t rc = harts_la_plan_tables(plan, dev_blob, &tb);
    if (rc != HARTS_OK) return rc;
    if (H < 1 || tb.chunk != 64 || !harts::gk_supported(dtype, dk, dv)) return H < 1 ? HARTS_EINVAL : HARTS_EUNSUPPORTED;
    if (!q || !k || !v || !gk || !dO || !dq || !dk_ || !dv_ || !dgk || !chunk_states || !scratch) return HARTS_EINVAL;
    if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(gk) || misaligned(dO) || misaligned(dq) ||
        misaligned(dk_) || misaligned(dv_) || misaligned(dgk) || misaligned(chunk_states) || misaligned(scratch))
        return HARTS_EINVAL;
    if ((flags & HARTS_FLAG_CHECK_TABLES) && !dev_status) return HARTS_EINVAL;
    const int32_t r1 = round == 0 ? p->n_rounds : round, r0 = round == 0 ? 1 : round;
    bool done = false;
    const bool chunks = harts::chunk_parallel(tb, H, dk, dv, dtype, flags);
    if (chunks && round == 0 && p->n_rounds <= harts::MAX_FUSED_ROUNDS && !(flags & HARTS_FLAG_ROUND_LAUNCHES)) {
        harts::BwdArgs a{tb, 0, tb.n_seq, q, k, v, gk, dO, dq, dk_, dv_, dgk, chunk_states, scratch, H, dk, dv, dtype, flags,
                         dev_status, static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        if ((rc = gk_chunk_parallel_bwd(a, p->round_seq_ptr.data(), p->n_rounds)) != HARTS_OK) return rc;
        done = true;
    }
    if (!chunks && round == 0 && p->n_rounds > 1 && p->n_rounds <= harts::MAX_FUSED_ROUNDS &&
        !(flags & (HARTS_FLAG_ROUND_LAUNCHES | HARTS_FLAG_FMA_KERNELS)) && harts::gk_mma_supported(dtype, dk, dv)) {
        harts::BwdArgs a{tb, 0, tb.n_seq, q, k, v, gk, dO, dq, dk_, dv_, dgk, chunk_states, scratch, H, dk, dv, dtype, flags,
                         dev_status, static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, 0, tb.n_seq, dev_status, a.stream)) != HARTS_OK) return rc;
        int* fl = reinterpret_cast<int*>(const_cast<char*>(static_cast<const char*>(chunk_states)) +
                                         harts::chunk_state_payload(tb, H, dk, dv, 2));
        harts::RoundOrder ro;
        ro.n = p->n_rounds;
        for (int32_t r = 0; r <= p->n_rounds; r++) ro.ptr[r] = p->round_seq_ptr[r];
        rc = harts::gk_mma_bwd_all(a, fl + (size_t)tb.n_slots * H, fl + harts::fused_flag_count(tb, H) + 1, ro);
        if (rc == HARTS_OK) done = true;
        else if (rc != HARTS_EUNSUPPORTED) return rc;
    }
    for (int32_t r = r1; r >= r0 && !done; r--) {
        harts::BwdArgs a{tb, p->round_seq_ptr[r - 1], p->round_seq_ptr[r], q, k, v, gk, dO, dq, dk_, dv_, dgk,
                         chunk_states, scratch, H, dk, dv, dtype, flags, dev_status, static_cast<cudaStream_t>(stream)};
        if (flags & HARTS_FLAG_CHECK_TABLES)
            if ((rc = harts::check_tables(tb, a.seq_lo, a.seq_hi, dev_status, a.stream)) != HARTS_OK) return rc;
        if ((rc = chunks ? gk_chunk_parallel_bwd(a, &p->round_seq_ptr[r - 1], 1) : harts::gk_bwd(a)) != HARTS_OK) return rc;
    }
    if (r0 == 1)
        return harts::gk_replay_reduce(tb, dk_, dv_, dgk, scratch, H, dk, dv, dtype, static_cast<cudaStream_t>(stream));
    return HARTS_OK;
}

int32_t harts_la_check(const int32_t* dev_status, void* stream) {
    if (!dev_status) return HARTS_EINVAL;
    int32_t host = 0;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&host, dev_status, sizeof(host), cudaMemcpyDeviceToHost, s) != cudaSuccess) return HARTS_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return HARTS_ECUDA;
    if (host == 0) return HARTS_OK;
    return host == HARTS_EINVAL ? HARTS_EINVAL : HARTS_ETIMEOUT;   // EINVAL: an index check of harts_logp_*
}

}  // extern "C"
