// fdd_decode_block: the denoising loop of one block (Sec. 3.3), driven by the library.
//
// Per step: gated attention for every layer and the unmasking step, which also writes the
// per-rollout counts of MASKED positions into host memory.  The host side is the part that matters
// here: on short steps (one scene, a few rollouts) the kernels of a step take a few tens of
// microseconds, less than an interpreter needs to marshal the same calls, so the loop lives in
// native code and runs one step ahead of the counts it reads.
#include "fdd_internal.h"

#include <algorithm>
#include <chrono>

namespace {

// Wait until every rollout's (n_left, stamp) of the step with this stamp has reached the host; their
// sum goes to *left.  The wait is bounded: it ends with an error if the stream reports one, if the
// stream has run empty without the counts arriving, or after kCountWaitSeconds.
constexpr double kCountWaitSeconds = 30.0;

fdd_status wait_for_counts(fdd_ctx* ctx, int buf, int stamp, int forks, cudaStream_t st, int* left) {
    const volatile long long* src = reinterpret_cast<const volatile long long*>(ctx->h_counts[buf]);
    const auto t0 = std::chrono::steady_clock::now();
    int f = 0, sum = 0;
    unsigned spins = 0;
    bool drained = false;
    while (f < forks) {
        const long long v = src[f];                      // one aligned 8-byte load: count in the low half, stamp in the high half
        if (static_cast<int>(v >> 32) == stamp) {
            sum += static_cast<int>(v & 0xFFFFFFFFLL);
            ++f;
            continue;
        }
        if ((++spins & 0x3FFu) == 0) {
            const double waited = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
            if (waited > 200e-6) {
                // a long wait: make sure the stream is still alive
                if (drained) {
                    ctx->last_error = "fdd_decode_block: the stream ran empty but the counts of a step never arrived";
                    return FDD_ERR_CUDA;
                }
                const cudaError_t q = cudaStreamQuery(st);
                if (q == cudaSuccess) drained = true;    // everything issued has completed: one more look at the counts, then give up
                else if (q != cudaErrorNotReady) {
                    ctx->last_error = std::string("fdd_decode_block: ") + cudaGetErrorString(q);
                    return FDD_ERR_CUDA;
                }
            }
            if (waited > kCountWaitSeconds) {
                ctx->last_error = "fdd_decode_block: timed out waiting for the counts of a step";
                return FDD_ERR_DEVICE_TIMEOUT;
            }
        }
#if defined(__x86_64__) || defined(__i386__)
        __builtin_ia32_pause();
#endif
    }
    *left = sum;
    return FDD_OK;
}

// Whether `st` belongs to a green context (a share of the SMs that its work is confined to).
bool in_green_context(cudaStream_t st) {
    using GetGreenCtx = CUresult (*)(CUstream, CUgreenCtx*);
    static const GetGreenCtx get = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult found;
        const bool ok = cudaGetDriverEntryPoint("cuStreamGetGreenCtx", &p, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess;
        return ok ? reinterpret_cast<GetGreenCtx>(p) : nullptr;
    }();
    CUgreenCtx green = nullptr;
    return get != nullptr && get(st, &green) == CUDA_SUCCESS && green != nullptr;
}

// The context's own stream of the same priority as the caller's; nullptr where there is none to be had, or none that the
// caller's limits would hold for: the attention then goes behind the unmasking on the caller's stream.
cudaStream_t side_stream_of(fdd_ctx* ctx, cudaStream_t st) {
    int priority = 0;
    if (in_green_context(st) || cudaStreamGetPriority(st, &priority) != cudaSuccess) return nullptr;
    for (const fdd_ctx::SideStream& s : ctx->side_streams)
        if (s.priority == priority) return s.stream;
    cudaStream_t made = nullptr;
    if (cudaStreamCreateWithPriority(&made, cudaStreamNonBlocking, priority) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    ctx->side_streams.push_back({priority, made});
    return made;
}

}  // namespace

fdd_status fdd_decode_block(fdd_ctx* ctx, fdd_forkset* const* sets, int n_sets, int n_layers,
                            int max_steps, int n_inputs,
                            const void* const* q, const void* const* k_blk, const void* const* v_blk,
                            void* const* out, const void* const* logits,
                            int32_t* tokens, uint8_t* state, const int32_t* block_len,
                            float scale, int causal_in_block, float threshold, float temperature,
                            uint32_t block_idx, int commit_kv,
                            int32_t* n_committed, int32_t* n_left,
                            int* steps_taken, int* masked_left,
                            fdd_step_fn before_step, void* user, void* stream) {
    CallRange range("fdd_decode_block");
    if (!ctx) return FDD_ERR_INVALID_ARG;
    if (!q || !k_blk || !v_blk || !out || !logits || !steps_taken || !n_left || !n_committed) {
        ctx->last_error = "fdd_decode_block: a required pointer is NULL";
        return FDD_ERR_INVALID_ARG;
    }
    if (n_layers < 1 || n_layers > ctx->cfg.n_layers || max_steps < 1 || n_inputs < 1 || n_sets < 1 || !sets) {
        ctx->last_error = "fdd_decode_block: n_layers must be in [1, context layers], max_steps, n_inputs and n_sets >= 1";
        return FDD_ERR_INVALID_ARG;
    }
    int forks = 0;
    for (int s = 0; s < n_sets; ++s) {
        if (!sets[s]) {
            ctx->last_error = "fdd_decode_block: a fork set is NULL";
            return FDD_ERR_INVALID_ARG;
        }
        forks += sets[s]->n_forks;
    }
    if (forks > ctx->cfg.max_forks) {
        ctx->last_error = "fdd_decode_block: more rollouts than the context was created for";
        return FDD_ERR_CAPACITY;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    *steps_taken = 0;
    if (masked_left) *masked_left = 0;

    // The attention of a step and its unmasking do not need each other (q, k, v and logits are all in place before the
    // step; attention only wants to know which rollouts the step before left undone), so they run side by side: the
    // unmasking on `st`, the attention on the context's own stream, each step's behind the unmasking of the step
    // before.  Both are chains of short kernels that leave most of the chip idle, or of long ones with uneven ends.
    // With a callback the next step's inputs are enqueued on `st` behind both, so all stays there.
    // One behind the other -> side by side, us: twelve steps of the smallest block 223 -> 157, three blocks of one rollout
    // 398 -> 260, of eight 737 -> 594, 36 layers of eight 1525 -> 1469, 32 rollouts on 16384 tokens 1879 -> 1824.
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    const bool beside = before_step == nullptr && forks <= kAttnMaxGatedForks && scale > 0.0f && cudaStreamIsCapturing(st, &capturing) == cudaSuccess && capturing == cudaStreamCaptureStatusNone &&
                        attention_beside_unmasking(ctx, sets, n_sets, n_layers, n_inputs < max_steps ? n_inputs : max_steps, q, k_blk, v_blk, out, logits,
                                                   tokens, state, block_len, n_committed, n_left);
    cudaStream_t st_attn = st;                          // (another one is looked for once the first unmasking is on its way)
    auto cuda_ok = [&](cudaError_t e) {
        if (e != cudaSuccess) ctx->last_error = std::string("fdd_decode_block: ") + cudaGetErrorString(e);
        return e == cudaSuccess;
    };
    // everything on `to` from here on follows everything on `from` so far
    auto follow = [&](cudaStream_t to, cudaStream_t from, cudaEvent_t ev) {
        return cuda_ok(cudaEventRecord(ev, from)) && cuda_ok(cudaStreamWaitEvent(to, ev, 0));
    };
    auto gate_slot = [&](int t) { return ctx->gate_slots + static_cast<size_t>(t % kGateSlots) * std::min(ctx->cfg.max_forks, kAttnMaxGatedForks); };

    int stamp_of[2] = {0, 0};
    // From the second step on, attention skips the rollouts that the step before left without a MASKED position.
    auto attend = [&](int t) -> fdd_status {
        const size_t at = static_cast<size_t>(t % n_inputs) * n_layers;
        return block_attn_layers(ctx, sets, n_sets, 0, n_layers, q + at, k_blk + at, v_blk + at, out + at, block_len, scale, causal_in_block,
                                 t == 0 ? nullptr : (beside ? gate_slot(t - 1) : n_left), st_attn, beside);
    };
    auto unmask = [&](int t) -> fdd_status {
        // the unmasking step also writes (n_left, stamp) of every rollout into host memory that the
        // device can address: the host sees the counts the moment they land, without a copy
        if (++ctx->count_stamp <= 0) ctx->count_stamp = 1;
        stamp_of[t & 1] = ctx->count_stamp;
        ctx->unmask_left_mirror = ctx->d_counts[t & 1];
        ctx->unmask_mirror_stamp = ctx->count_stamp;
        ctx->unmask_gate_out = beside ? gate_slot(t) : nullptr;
        const fdd_status rc = fdd_unmask(ctx, sets, n_sets, logits[t % n_inputs], tokens, state, block_len, threshold, temperature,
                                         block_idx, static_cast<uint32_t>(t), n_committed, n_left, nullptr, stream);
        ctx->unmask_left_mirror = nullptr;
        ctx->unmask_gate_out = nullptr;
        return rc;
    };
    // What is issued ahead of the counts of step t - 1: all of step t, or, side by side, its unmasking alone.
    auto enqueue = [&](int t) -> fdd_status {
        if (!beside) {
            if (before_step) before_step(user, t, stream);
            const fdd_status rc = attend(t);
            return rc != FDD_OK ? rc : unmask(t);
        }
        // what the attention of step t has to wait for: the unmasking of the step before (at first, whatever is on `st`)
        if (!cuda_ok(cudaEventRecord(ctx->ev_gate[t & 1], st))) return FDD_ERR_CUDA;
        // (a count's slot is written again only behind the attention that read it)
        if (t >= kGateSlots && !follow(st, st_attn, ctx->ev_end)) return FDD_ERR_CUDA;
        return unmask(t);
    };
    // Side by side, the attention of step t goes out once the step is known to be needed, behind its unmasking: that is
    // short, and the CTAs of the attention take whole SMs.
    auto enqueue_attention = [&](int t) -> fdd_status {
        if (!beside) return FDD_OK;
        if (t == 0)
            if (const cudaStream_t side = side_stream_of(ctx, st)) st_attn = side;
        return cuda_ok(cudaStreamWaitEvent(st_attn, ctx->ev_gate[t & 1], 0)) ? attend(t) : FDD_ERR_CUDA;
    };

    fdd_status rc = enqueue(0);
    if (rc == FDD_OK) rc = enqueue_attention(0);
    int t = 0, left = 0;
    while (rc == FDD_OK) {
        // step t + 1 goes out before the host knows what step t left: if the block turns out to be
        // complete, its kernels find every rollout gated off and no MASKED row, and return at once
        if (t + 1 < max_steps) rc = enqueue(t + 1);
        if (rc != FDD_OK) break;
        rc = wait_for_counts(ctx, t & 1, stamp_of[t & 1], forks, st, &left);
        if (rc != FDD_OK) break;
        ++t;
        if (left == 0 || t >= max_steps) break;
        rc = enqueue_attention(t);
    }
    // whatever follows on `st` follows the attention too
    if (beside && !follow(st, st_attn, ctx->ev_end) && rc == FDD_OK) rc = FDD_ERR_CUDA;
    if (rc != FDD_OK) return rc;
    *steps_taken = t;
    if (masked_left) *masked_left = left;
    if (commit_kv && left == 0) {
        // the block is complete: its keys and values, as the last step projected them, join every
        // rollout's private cache
        const size_t at = static_cast<size_t>((t - 1) % n_inputs) * n_layers;
        CallRange commit_range("fdd_kv_commit");
        rc = commit_layers(ctx, sets, n_sets, 0, n_layers, k_blk + at, v_blk + at, block_len, 1, stream, false);
        if (rc != FDD_OK) return rc;
    }
    return FDD_OK;
}
