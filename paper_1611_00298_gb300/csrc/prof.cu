// Kernel launch counter and optional CUDA-event timing of the hop and
// 5D-local kernels (events are recorded on the stream each kernel runs on).
#include "api_util.h"

long long g_launches = 0;

// Event pairs held at a time.  When all are taken the oldest is read (its
// launch lies PROF_PAIRS launches back) and used again, so every launch between
// start and stop is counted.
#define PROF_PAIRS 65536

// adds the oldest pair that is held to the totals of its kind
static void prof_take(Prof* p) {
    const int i = (int)(p->taken % PROF_PAIRS);
    EOFA_CUDA(cudaEventSynchronize(p->ev[2 * i + 1]));
    float ms = 0.f;
    EOFA_CUDA(cudaEventElapsedTime(&ms, p->ev[2 * i], p->ev[2 * i + 1]));
    p->launches[p->kind[i]]++;
    p->ms[p->kind[i]] += ms;
    p->sum_bytes[p->kind[i]] += p->bytes[i];
    p->taken++;
}

void prof_begin(const eofa_ctx* ctx, int kind, cudaStream_t st, double bytes) {
    Prof* p = ctx->prof;
    if (!p || !p->on) return;
    const int i = (int)(p->used % PROF_PAIRS);
    if (p->used - p->taken >= PROF_PAIRS) prof_take(p);
    EOFA_CUDA(cudaEventRecord(p->ev[2 * i], st));
    p->kind[i] = kind;
    p->bytes[i] = bytes;
}

void prof_end(const eofa_ctx* ctx, cudaStream_t st) {
    Prof* p = ctx->prof;
    if (!p || !p->on) return;
    EOFA_CUDA(cudaEventRecord(p->ev[2 * (int)(p->used % PROF_PAIRS) + 1], st));
    p->used++;
}

extern "C" {

long long eofa_kernel_launches(void) { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

int eofa_profile_start(eofa_ctx* ctx) {
    if (!ctx) return EOFA_EINVAL;
    try {
        if (!ctx->prof) {
            ctx->prof = new Prof();
            ctx->prof->ev.resize(2 * PROF_PAIRS);
            ctx->prof->kind.resize(PROF_PAIRS);
            ctx->prof->bytes.resize(PROF_PAIRS);
            for (auto& e : ctx->prof->ev) EOFA_CUDA(cudaEventCreate(&e));
        }
        ctx->prof->used = ctx->prof->taken = 0;
        for (int k = 0; k < 6; k++) {
            ctx->prof->launches[k] = 0;
            ctx->prof->ms[k] = ctx->prof->sum_bytes[k] = 0.0;
        }
        ctx->prof->on = true;
    } catch (const eofa_error& e) {
        return fail(ctx, e.code, e.msg);
    }
    return EOFA_OK;
}

int eofa_profile_stop(eofa_ctx* ctx, eofa_profile* out) {
    if (!ctx || !out) return EOFA_EINVAL;
    for (int k = 0; k < 6; k++) {
        out->launches[k] = 0;
        out->ms[k] = 0.0;
        out->bytes[k] = 0.0;
    }
    Prof* p = ctx->prof;
    if (!p) return EOFA_OK;
    try {
        p->on = false;
        while (p->taken < p->used) prof_take(p);
        for (int k = 0; k < 6; k++) {
            out->launches[k] = p->launches[k];
            out->ms[k] = p->ms[k];
            out->bytes[k] = p->sum_bytes[k];
            p->launches[k] = 0;
            p->ms[k] = p->sum_bytes[k] = 0.0;
        }
        p->used = p->taken = 0;
    } catch (const eofa_error& e) {
        return fail(ctx, e.code, e.msg);
    }
    return EOFA_OK;
}

}  // extern "C"
