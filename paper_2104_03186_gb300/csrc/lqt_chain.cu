// Chunked single-problem pipeline behind the C ABI (lqt_solve and
// lqt_riccati_sequential for the lane-group sizes): variant lookup, chunk
// geometry, workspace layout.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "lqt_chain_api.h"

namespace lqt {
namespace {

// smallest chunk the planner makes, in steps
constexpr long long kMinChunk = 4;

// Batches of the lane sizes: launches per run of tree levels, one persistent
// launch, or (the default) the per-level launches everywhere
// (lqt_batch_set_tuning).  Measured on one GB300 with the sizes side by side,
// per-level against persistent against the persistent launch only for grids of
// at most half the device: 8 mixed requests 335 / 345 / 345 us, 48 658 / 1142 /
// 696, 200 1.53 / 2.56 / 1.63 ms, 512 problems of T <= 1024 1.01 / 1.48 / 1.01,
// the 4096-problem batch 19.8 / 21.5 / 19.8 ms.  A cooperative launch waits
// until its whole grid is resident, so it holds up the other sizes.
std::atomic<int> g_batch_mode{LQT_BATCH_AUTO};

// Tuned chunk lengths of batches (lqt_batch_set_tuning): entry e applies to
// problems of state size n = e.n with T <= e.t_max (the first such entry).
constexpr int kMaxTune = 64;
std::mutex g_tune_mu;
lqt_batch_tune_entry g_tune[kMaxTune];
int g_tune_count = 0;

// A copy of the table, for the problems of one batch.
std::vector<lqt_batch_tune_entry> tune_table() {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    return std::vector<lqt_batch_tune_entry>(g_tune, g_tune + g_tune_count);
}

// The tuned chunk length for a problem, or 0 (none).
long long tuned_chunk(const std::vector<lqt_batch_tune_entry>& table, int n, long long T) {
    for (const lqt_batch_tune_entry& e : table)
        if (e.n == n && T <= e.t_max) return e.chunk_steps;
    return 0;
}

const ChainVariant* find_chain(int dtype, int n, int m, bool mixed) {
    const ChainVariant* (*tables[])(int*) = {&chain_variants_n4, &chain_variants_n8,
                                             &chain_variants_n16, &chain_variants_n32};
    for (auto t : tables) {
        int cnt = 0;
        const ChainVariant* v = t(&cnt);
        for (int i = 0; i < cnt; ++i)
            if (v[i].dtype == dtype && v[i].n == n && v[i].m == m &&
                (dtype == LQT_F64 || (v[i].mixed != 0) == mixed))
                return &v[i];
    }
    return nullptr;
}

// Resident lane groups of the fold kernel on the whole device.
lqt_status fold_slots(const ChainVariant& v, long long* slots) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LQT_ECUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return LQT_ECUDA;
    const size_t smem = v.fold_smem();
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(v.fold_kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
        return LQT_ECUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, v.fold_kernel(),
                                                      v.fold_threads(), smem) != cudaSuccess)
        return LQT_ECUDA;
    *slots = (long long)sms * (per_sm > 0 ? per_sm : 1) * v.fold_groups();
    return LQT_OK;
}

lqt_status geometry(const ChainVariant& v, const lqt_problem* P, bool sequential, int* NC,
                    long long* B) {
    const long long T = P->T;
    if (sequential) {
        *NC = 1;
        *B = T > 0 ? T : 1;
        return LQT_OK;
    }
    long long slots = 0;
    const lqt_status st = fold_slots(v, &slots);
    if (st != LQT_OK) return st;
    long long cap = T / kMinChunk;
    if (cap > slots) cap = slots;
    if (cap > (1LL << 24)) cap = 1LL << 24;
    long long nc = 1;
    while (nc * 2 <= cap) nc *= 2;
    *NC = (int)nc;
    *B = T > 0 ? (T + nc - 1) / nc : 1;
    return LQT_OK;
}

// Chunk geometry of a batch of one variant: a chunk length B* from the
// total work over the resident fold groups, clamped to [kMinChunk,
// kMaxBatchChunk] so that no problem's latency grows with the batch, or the
// tuned length of the problem's (n, T) where it is shorter than the unclamped
// fill length; each problem takes the largest power-of-two chunk count with
// chunks of at least that many steps.  Problems sorted by decreasing chunk
// count.
constexpr long long kMaxBatchChunk = 64;

lqt_status batch_geometry(const ChainVariant& v, const lqt_batch_item* items, const int* idx,
                          int count, std::vector<ChainProblem>* out) {
    long long slots = 0;
    const lqt_status st = fold_slots(v, &slots);
    if (st != LQT_OK) return st;
    long long total = 0;
    for (int i = 0; i < count; ++i) total += items[idx[i]].problem.T;
    long long fill = (total + slots - 1) / (slots > 0 ? slots : 1);
    if (fill < kMinChunk) fill = kMinChunk;
    const long long Bt = fill < kMaxBatchChunk ? fill : kMaxBatchChunk;
    const std::vector<lqt_batch_tune_entry> table = tune_table();
    out->resize((size_t)count);
    for (int i = 0; i < count; ++i) {
        const lqt_batch_item& it = items[idx[i]];
        const long long T = it.problem.T;
        // a tuned length applies up to the one that fills the device: a batch
        // with less work than that keeps every resident group busy instead
        const long long tuned = tuned_chunk(table, it.problem.n, T);
        const long long Bi = tuned > 0 ? (tuned < fill ? tuned : fill) : Bt;
        long long nc = 1;
        while (nc * 2 * Bi <= T && nc < (1LL << 20)) nc *= 2;
        ChainProblem& cp = (*out)[(size_t)i];
        cp.problem = &it.problem;
        cp.solution = &it.solution;
        cp.NC = (int)nc;
        cp.B = T > 0 ? (T + nc - 1) / nc : 1;
    }
    std::stable_sort(out->begin(), out->end(),
                     [](const ChainProblem& a, const ChainProblem& b) {
                         return a.NC != b.NC ? a.NC > b.NC : a.B > b.B;
                     });
    return LQT_OK;
}

}  // namespace

bool chain_supported(int dtype, int n, int m) {
    return n >= 8 && find_chain(dtype, n, m, false) != nullptr;
}

bool chain_small_supported(int dtype, int n, int m) {
    return n < 8 && find_chain(dtype, n, m, false) != nullptr;
}

lqt_status chain_workspace(const lqt_problem* P, bool refine, bool newton, bool sequential,
                           bool method2, bool lean, size_t* bytes, int* NC, long long* B,
                           int* kernels) {
    if (P->p > 2 * P->n || P->pT > 2 * P->n) return LQT_EUNSUPPORTED;
    // FP64 tree levels with the FULL refinement (the Newton step); FP32 otherwise
    const bool mixed = refine && newton && P->dtype == LQT_F32;
    const ChainVariant* v = find_chain(P->dtype, P->n, P->m, mixed);
    if (!v) return LQT_EUNSUPPORTED;
    int nc = 1;
    long long b = 1;
    const lqt_status st = geometry(*v, P, sequential, &nc, &b);
    if (st != LQT_OK) return st;
    ChainProblem cp{P, nullptr, nc, b};
    const bool rf = refine && P->T > 0;
    const bool vector = rf && !method2 && !sequential && !lean;
    if (bytes) *bytes = v->workspace(&cp, 1, rf, rf && newton, method2, vector);
    if (NC) *NC = nc;
    if (B) *B = b;
    if (kernels) *kernels = v->kernels(nc, rf, rf && newton, sequential, method2, vector);
    return LQT_OK;
}

lqt_status chain_solve(const lqt_problem* P, const lqt_solution* sol, bool refine, bool newton,
                       bool sequential, bool method2, bool lean, void* ws, size_t ws_bytes,
                       cudaStream_t s, Prof* prof) {
    if (P->p > 2 * P->n || P->pT > 2 * P->n) return LQT_EUNSUPPORTED;
    const bool mixed = refine && newton && P->dtype == LQT_F32;
    const ChainVariant* v = find_chain(P->dtype, P->n, P->m, mixed);
    if (!v) return LQT_EUNSUPPORTED;
    int NC = 1;
    long long B = 1;
    const lqt_status st = geometry(*v, P, sequential, &NC, &B);
    if (st != LQT_OK) return st;
    ChainProblem cp{P, sol, NC, B};
    const bool rf = refine && P->T > 0;
    ChainCall call{&cp, 1, rf, rf && newton, sequential, method2, ws, ws_bytes, nullptr};
    call.vector = rf && !method2 && !sequential && !lean;
    return v->run(call, s, prof);
}

lqt_status chain_batch_plan(const lqt_batch_item* items, const int* idx, int count,
                            ChainPlan* plan) {
    const lqt_problem& P0 = items[idx[0]].problem;
    plan->variant = find_chain(LQT_F32, P0.n, P0.m, false);
    if (!plan->variant) return LQT_EUNSUPPORTED;
    const lqt_status st = batch_geometry(*plan->variant, items, idx, count, &plan->probs);
    if (st != LQT_OK) return st;
    plan->bytes = plan->variant->workspace(plan->probs.data(), count, false, false, false, false);
    return LQT_OK;
}

lqt_status chain_batch_solve(const ChainPlan& plan, void* ws, int* status, cudaStream_t s) {
    ChainCall call{plan.probs.data(), (int)plan.probs.size(), false, false, false, false, ws,
                   plan.bytes, status};
    call.persistent = g_batch_mode.load() == LQT_BATCH_PERSISTENT;
    return plan.variant->run(call, s, nullptr);
}

bool chain_warm_supported(int dtype, int n, int m) {
    return find_chain(dtype, n, m, false) != nullptr;
}

namespace {

// Chunk geometry of a warm call: one problem as lqt_solve cuts it, a batch as
// lqt_solve_batched does.
lqt_status warm_geometry(const ChainVariant& v, const lqt_batch_item* items, const int* idx,
                         int count, std::vector<ChainProblem>* probs) {
    if (count == 1) {
        const lqt_batch_item& it = items[idx[0]];
        int nc = 1;
        long long b = 1;
        const lqt_status st = geometry(v, &it.problem, false, &nc, &b);
        if (st != LQT_OK) return st;
        probs->assign(1, ChainProblem{&it.problem, &it.solution, nc, b});
        return LQT_OK;
    }
    return batch_geometry(v, items, idx, count, probs);
}

}  // namespace

lqt_status chain_warm_plan(const lqt_batch_item* items, const int* idx, int count,
                           ChainPlan* plan) {
    const lqt_problem& P0 = items[idx[0]].problem;
    plan->variant = find_chain(P0.dtype, P0.n, P0.m, false);
    if (!plan->variant) return LQT_EUNSUPPORTED;
    const lqt_status st = warm_geometry(*plan->variant, items, idx, count, &plan->probs);
    if (st != LQT_OK) return st;
    plan->bytes = plan->variant->workspace(plan->probs.data(), count, false, false, false, false);
    return LQT_OK;
}

lqt_status chain_warm_solve(const ChainPlan& plan, void* ws, int* status, cudaStream_t s) {
    ChainCall call{plan.probs.data(), (int)plan.probs.size(), false, false, false, false, ws,
                   plan.bytes, status};
    call.warm = true;
    return plan.variant->run(call, s, nullptr);
}

}  // namespace lqt

extern "C" lqt_status lqt_batch_set_tuning(const lqt_batch_tune_entry* entries, int32_t count,
                                           int32_t persistent) {
    using namespace lqt;
    if (count < 0 || count > kMaxTune || (count > 0 && !entries)) return LQT_EINVAL;
    if (persistent < LQT_BATCH_PER_LEVEL || persistent > LQT_BATCH_AUTO) return LQT_EINVAL;
    for (int i = 0; i < count; ++i)
        if (entries[i].n < 1 || entries[i].t_max < 0 || entries[i].chunk_steps < 1)
            return LQT_EINVAL;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    for (int i = 0; i < count; ++i) g_tune[i] = entries[i];
    g_tune_count = count;
    g_batch_mode.store(persistent);
    return LQT_OK;
}
