// C ABI of the warm solve (include/lqt.h: lqt_solve_warm): problems whose S_k
// and K_k are known (a receding horizon over an earlier solve's model), solved
// for v, x* and u* by the vector scans of lqt_warm.cuh.  Problems are grouped
// by (dtype, n, m); each group is one chain call with its own part of the
// workspace, and the groups run side by side: the first on the caller's stream,
// the others on auxiliary streams forked from it and joined back (lqt_fork.h).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>
#include <vector>

#include "lqt.h"
#include "lqt_chain_api.h"
#include "lqt_fork.h"

namespace lqt {
namespace {

constexpr size_t kAlignW = 256;
size_t up(size_t x) { return (x + kAlignW - 1) / kAlignW * kAlignW; }

bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

lqt_status check_warm_item(const lqt_batch_item& it) {
    const lqt_problem& P = it.problem;
    const lqt_solution& S = it.solution;
    if (P.dtype != LQT_F32 && P.dtype != LQT_F64) return LQT_EINVAL;
    if (P.n < 1 || P.m < 1 || P.T < 0 || P.p < 0 || P.pT < 0) return LQT_EINVAL;
    if (!chain_warm_supported(P.dtype, P.n, P.m)) return LQT_EUNSUPPORTED;
    if (P.p > 2 * P.n || P.pT > 2 * P.n) return LQT_EUNSUPPORTED;
    if (P.T > 0 && (!P.F.ptr || !P.L.ptr || !P.U.ptr)) return LQT_EINVAL;
    if (P.T > 0 && P.p > 0 && (!P.H.ptr || !P.X.ptr)) return LQT_EINVAL;
    if (!P.x0 || (P.pT > 0 && (!P.HT || !P.XT))) return LQT_EINVAL;
    if (!S.S || !S.v || !S.x || (P.T > 0 && (!S.K || !S.u))) return LQT_EINVAL;
    const size_t es = P.dtype == LQT_F64 ? 8 : 4;
    const int64_t n = P.n, m = P.m, p = P.p;
    const struct {
        const lqt_in* in;
        int64_t size;
    } ins[] = {{&P.F, n * n}, {&P.c, n}, {&P.L, n * m}, {&P.U, m * m},
               {&P.H, p * n}, {&P.r, p}, {&P.X, p * p}};
    for (const auto& i : ins) {
        if (!i.in->ptr) continue;
        if (!aligned_to(i.in->ptr, es)) return LQT_EINVAL;
        if (i.in->step_stride < 0 || (i.in->step_stride != 0 && i.in->step_stride < i.size))
            return LQT_EINVAL;
    }
    const void* outs[] = {S.S, S.v, S.K, S.x, S.u};
    for (const void* o : outs)
        if (o && !aligned_to(o, es)) return LQT_EINVAL;
    return LQT_OK;
}

// Indices of the items, grouped by (dtype, n, m).
std::vector<std::vector<int>> warm_groups(const lqt_batch_item* items, int32_t count) {
    std::vector<std::vector<int>> groups;
    std::vector<std::pair<int, std::pair<int, int>>> keys;
    for (int i = 0; i < count; ++i) {
        const lqt_problem& P = items[i].problem;
        const auto key = std::make_pair((int)P.dtype, std::make_pair(P.n, P.m));
        size_t g = 0;
        while (g < keys.size() && keys[g] != key) ++g;
        if (g == keys.size()) {
            keys.push_back(key);
            groups.emplace_back();
        }
        groups[g].push_back(i);
    }
    return groups;
}

// The groups' plans and the workspace bytes of the whole call (a region of its
// own for each group); 0 if a group is invalid.
size_t plan_warm(const lqt_batch_item* items, int32_t count, std::vector<ChainPlan>* plans) {
    const std::vector<std::vector<int>> groups = warm_groups(items, count);
    plans->resize(groups.size());
    size_t bytes = up(256);
    for (size_t i = 0; i < groups.size(); ++i) {
        if (chain_warm_plan(items, groups[i].data(), (int)groups[i].size(), &(*plans)[i]) !=
            LQT_OK)
            return 0;
        bytes += up((*plans)[i].bytes);
    }
    return bytes;
}

}  // namespace
}  // namespace lqt

using namespace lqt;

extern "C" size_t lqt_warm_workspace_bytes(const lqt_batch_item* items, int32_t count) {
    if (count < 0 || (count > 0 && !items)) return 0;
    for (int i = 0; i < count; ++i)
        if (check_warm_item(items[i]) != LQT_OK) return 0;
    std::vector<ChainPlan> plans;
    return plan_warm(items, count, &plans);
}

extern "C" lqt_status lqt_solve_warm(const lqt_batch_item* items, int32_t count, void* workspace,
                                     size_t workspace_bytes, void* stream) {
    if (count < 0 || (count > 0 && !items)) return LQT_EINVAL;
    if (!workspace || !aligned_to(workspace, kAlignW)) return LQT_EINVAL;
    for (int i = 0; i < count; ++i) {
        const lqt_status st = check_warm_item(items[i]);
        if (st != LQT_OK) return st;
    }
    // cut once: the sizes checked here are those the groups run with
    std::vector<ChainPlan> plans;
    const size_t need = plan_warm(items, count, &plans);
    if (need == 0 || workspace_bytes < need) return LQT_ENOMEM;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(workspace);
    int* status = reinterpret_cast<int*>(base);
    if (cudaMemsetAsync(base, 0, sizeof(int), s) != cudaSuccess) return LQT_ECUDA;
    char* ws = base + up(256);
    ForkSet* aux = plans.size() > 1 ? next_fork_set(s) : nullptr;
    if (aux && cudaEventRecord(aux->fork, s) != cudaSuccess) return LQT_ECUDA;
    // the auxiliary streams in use rejoin the caller's stream on every return
    // (their work uses the workspace, and a capture must end joined)
    int forked = 0;
    auto rejoin = [&](lqt_status st) {
        for (int i = 0; i < forked; ++i)
            if (cudaEventRecord(aux->join[i], aux->s[i]) != cudaSuccess ||
                cudaStreamWaitEvent(s, aux->join[i], 0) != cudaSuccess)
                st = st == LQT_OK ? LQT_ECUDA : st;
        return st;
    };
    for (size_t i = 0; i < plans.size(); ++i) {
        cudaStream_t gs = s;
        if (aux && i > 0) {  // group i on set stream (i - 1) mod kForkStreams
            const int q = (int)((i - 1) % kForkStreams);
            gs = aux->s[q];
            if (q >= forked) {
                if (cudaStreamWaitEvent(gs, aux->fork, 0) != cudaSuccess) return rejoin(LQT_ECUDA);
                forked = q + 1;
            }
        }
        const lqt_status st = chain_warm_solve(plans[i], ws, status, gs);
        if (st != LQT_OK) return rejoin(st);
        ws += up(plans[i].bytes);
    }
    return rejoin(LQT_OK);
}
