// Checks which phases a kernel waits for when it leaves after a timeout
// (ring_newest, ring_pair_newest), against a model of the rings' mbarriers:
// for every ring length, number of consumed blocks and number of blocks that
// each producer had issued by then, the waits end exactly when every copy
// issued has landed.  Prints "ok" or the first failure.
#include <cstdio>
#include <vector>

#include "ppas_internal.h"

using namespace ppas;

// one full barrier: an arrival count of 1 and a byte count
struct Bar {
    int phases = 0;  // completed
    int pending = 1;
    long tx = 0;
    void settle() {
        if (pending == 0 && tx == 0) {
            ++phases;
            pending = 1;
        }
    }
    void expect(long bytes) {
        tx += bytes;
        --pending;
        settle();
    }
    void land(long bytes) {
        tx -= bytes;
        settle();
    }
    // what a wait for this parity answers
    bool done(int parity) const { return ((phases - 1) & 1) == parity; }
};

static const char *run(int stages, int consumed, int issued0, int issued1, bool pair) {
    std::vector<Bar> bar(stages);
    struct Copy {
        int block, cta;
    };
    std::vector<Copy> flying;
    const int most = pair && issued1 > issued0 ? issued1 : issued0;
    for (int j = 0; j < most; ++j) {
        Bar &b = bar[j % stages];
        if (j < issued0) {
            b.expect(pair ? 2 : 1);
            if (j < consumed) b.land(1); else flying.push_back({j, 0});
        }
        if (pair && j < issued1) {
            if (j < consumed) b.land(1); else flying.push_back({j, 1});
        }
    }
    std::vector<RingPairNewest> nw(stages);
    for (int s = 0; s < stages; ++s) {
        nw[s] = pair ? ring_pair_newest(issued0, issued1, s, stages) : RingPairNewest{ring_newest(issued0, s, stages), false};
        if (nw[s].block >= most || (nw[s].block >= 0 && nw[s].block % stages != s)) return "block";
        if (nw[s].arm) {
            if (nw[s].block < issued0) return "armed twice";
            bar[s].expect(1);
        }
    }
    auto waits_over = [&](int s) { return nw[s].block < 0 || bar[s].done((nw[s].block / stages) & 1); };
    for (size_t left = flying.size(); left > 0; --left) {
        const Copy c = flying[left - 1];
        if (waits_over(c.block % stages)) return "left with a copy in flight";
        bar[c.block % stages].land(1);
    }
    for (int s = 0; s < stages; ++s) {
        // the leader armed for both and the other CTA never issued: its own copy
        // has landed, and the wait ends with its limit
        const bool half = pair && nw[s].block >= consumed && nw[s].block >= issued1;
        if (!half && !waits_over(s)) return "wait without end";
    }
    return nullptr;
}

int main() {
    for (int stages = 1; stages <= 12; ++stages)
        for (int consumed = 0; consumed <= 3 * stages; ++consumed)
            for (int i0 = consumed; i0 <= consumed + stages; ++i0) {
                const char *e = run(stages, consumed, i0, 0, false);
                for (int i1 = consumed; !e && i1 <= consumed + stages; ++i1) e = run(stages, consumed, i0, i1, true);
                if (e) {
                    std::printf("FAIL %s: stages %d, consumed %d, issued %d\n", e, stages, consumed, i0);
                    return 1;
                }
            }
    std::printf("ok\n");
    return 0;
}
