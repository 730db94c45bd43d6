// Checks the decode plan with finer splits for the last rows of a mixed step.
// For every case read from stdin
//   <sms> <n_q_heads> <n_kv_heads> <n_seqs> <q_len>... <ctx_len>...
// it verifies that the splits of every row cover its pages exactly once, none
// empty or outside the kernel's limits; that only the last third of the rows
// differs from the plain plan, and only towards shorter splits; that totals and
// workspace sizes hold them; and that plan_step() takes the finer plan when the
// workspace holds it and the plain one when it does not.  One line per case:
// "ok <plain ctas> <fine ctas>" or "FAIL <reason>".
#include <algorithm>
#include <cstdio>
#include <iostream>
#include <string>
#include <vector>

#include "ppas_internal.h"

using namespace ppas;

static std::string check(int sms, int hq, int hk, const std::vector<int32_t> &q, const std::vector<int32_t> &c,
                         long long *plain, long long *fine) {
    const int n = static_cast<int>(q.size());
    const DecodePlan a = plan_decode(n, q.data(), c.data(), hq, hk, sms);
    const DecodePlan d = plan_decode(n, q.data(), c.data(), hq, hk, sms, {}, true);
    if (d.rows != a.rows || d.cluster != 1) return "rows or cluster";
    const size_t nr = d.rows.size();
    long long np = 0;
    for (size_t k = 0; k < nr; ++k) {
        const long long pages = (c[d.rows[k]] + kPage - 1) / kPage, ns = d.n_splits[k], pps = d.pages_per_split[k];
        if (ns < 1 || ns > kMaxDecodeSplitsPerRow || pps < 1 || pps > kDecodeMaxPagesPerSplit) return "limits";
        if ((ns - 1) * pps >= pages || ns * pps < pages) return "coverage";
        if (pps < std::min<long long>(pages, kDecodeMinPagesPerSplit)) return "split shorter than the minimum";
        if (k < nr - nr / 3 && (ns != a.n_splits[k] || pps != a.pages_per_split[k])) return "a first row changed";
        if (ns < a.n_splits[k] || pps > a.pages_per_split[k]) return "longer splits";
        np += ns;
    }
    if (np != d.n_part || np * hk != d.n_ctas) return "totals";
    if (d.ml_bytes < np * hq * 2 * sizeof(float) || d.o_bytes < np * hq * kHeadDim * sizeof(float) ||
        d.counter_bytes < nr * hk * sizeof(unsigned long long))
        return "workspace";
    *plain = a.n_ctas;
    *fine = d.n_ctas;
    if (static_cast<int>(nr) == n) return d.n_ctas == a.n_ctas ? "" : "a step of decode rows only changed";
    const StepPlan all = plan_step(n, q.data(), c.data(), hq, hk, SIZE_MAX);
    const StepPlan same = plan_step(n, q.data(), c.data(), hq, hk, all.total_bytes());
    if (same.dp.n_splits != all.dp.n_splits || same.pf.n_part != all.pf.n_part) return "plan at its own workspace size";
    const StepPlan least = plan_step(n, q.data(), c.data(), hq, hk, workspace_min_size(n, q.data(), c.data(), hq, hk));
    if (least.total_bytes() != workspace_min_size(n, q.data(), c.data(), hq, hk) || least.pf.n_part)
        return "plan at the smallest workspace";
    return "";
}

int main() {
    int sms, hq, hk, n;
    while (std::cin >> sms >> hq >> hk >> n) {
        std::vector<int32_t> q(n), c(n);
        for (auto &x : q) std::cin >> x;
        for (auto &x : c) std::cin >> x;
        long long plain = 0, fine = 0;
        const std::string err = check(sms, hq, hk, q, c, &plain, &fine);
        if (err.empty())
            std::printf("ok %lld %lld\n", plain, fine);
        else
            std::printf("FAIL %s\n", err.c_str());
    }
    return 0;
}
