// Counts the plans that plan_step() makes: plan_decode() and plan_prefill() are
// defined here in front of the library's, count, and call those.  For every case
// read from stdin
//   <n_q_heads> <n_kv_heads> <n_seqs> <q_len>... <ctx_len>...
// and for workspaces from none to as much as wanted, no plan may be made twice
// (the same arguments), and a workspace that holds everything takes one prefill
// plan.  One line per case: "ok" or "FAIL <reason>".
#include <dlfcn.h>

#include <cstdio>
#include <iostream>
#include <set>
#include <string>
#include <tuple>
#include <vector>

#include "ppas_internal.h"

using namespace ppas;

static std::multiset<std::tuple<bool, int, int>> g_prefill;  // (allow_split, n_ctas, max_work)
static std::multiset<bool> g_decode;                         // fine_tail

namespace ppas {
PrefillPlan plan_prefill(int32_t n_seqs, const int32_t *q, const int32_t *c, int32_t hq, int32_t hk, bool allow_split,
                         int32_t n_ctas, int32_t max_work) {
    using Fn = PrefillPlan (*)(int32_t, const int32_t *, const int32_t *, int32_t, int32_t, bool, int32_t, int32_t);
    static const Fn next = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "_ZN4ppas12plan_prefillEiPKiS1_iibii"));
    g_prefill.insert({allow_split, n_ctas, max_work});
    return next(n_seqs, q, c, hq, hk, allow_split, n_ctas, max_work);
}
DecodePlan plan_decode(int32_t n_seqs, const int32_t *q, const int32_t *c, int32_t hq, int32_t hk, int32_t sms,
                       const DecodeClusterCaps &caps, bool fine_tail) {
    using Fn = DecodePlan (*)(int32_t, const int32_t *, const int32_t *, int32_t, int32_t, int32_t,
                              const DecodeClusterCaps &, bool);
    static const Fn next = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "_ZN4ppas11plan_decodeEiPKiS1_iiiRKNS_17DecodeClusterCapsEb"));
    g_decode.insert(fine_tail);
    return next(n_seqs, q, c, hq, hk, sms, caps, fine_tail);
}
}  // namespace ppas

static std::string check(int hq, int hk, const std::vector<int32_t> &q, const std::vector<int32_t> &c) {
    const int n = static_cast<int>(q.size());
    auto made = [&](size_t ws) -> StepPlan {
        g_prefill.clear();
        g_decode.clear();
        return plan_step(n, q.data(), c.data(), hq, hk, ws);
    };
    const StepPlan all = made(SIZE_MAX);
    if (g_prefill.empty() && g_decode.empty()) return "not counted";
    if (g_prefill.size() != 1) return "prefill plans with room for everything: " + std::to_string(g_prefill.size());
    const size_t sizes[] = {SIZE_MAX, all.total_bytes(), all.total_bytes() - 1, all.dp.total_bytes(), 256, 0};
    for (size_t ws : sizes) {
        made(ws);
        for (const auto &k : g_prefill)
            if (g_prefill.count(k) > 1) return "a prefill plan made twice";
        for (bool k : g_decode)
            if (g_decode.count(k) > 1) return "a decode plan made twice";
    }
    return "";
}

int main() {
    int hq, hk, n;
    while (std::cin >> hq >> hk >> n) {
        std::vector<int32_t> q(n), c(n);
        for (auto &x : q) std::cin >> x;
        for (auto &x : c) std::cin >> x;
        const std::string e = check(hq, hk, q, c);
        std::printf(e.empty() ? "ok\n" : "FAIL %s\n", e.c_str());
    }
    return 0;
}
