// Host check of the staging schedule of the two-component pair kernel (compiled and run by
// tests/test_stages_host.py).  The march of a work item is replayed with a model of its two
// mbarriers; a wait is made to give up at every step of every item, and the waits that the
// kernel then makes have to be for exactly the phases whose copies are still in flight.
#include <cstdio>

#include "cg_stages.cuh"

using llb::cg::Stages;

namespace {

struct Barrier {
    unsigned phase = 0;  // phases completed
    int pending = 0;     // copies armed for the current phase
    // as mbarrier.try_wait.parity: the phase with this parity has completed
    bool passes(unsigned parity) const { return (phase & 1) != parity; }
};

int fails = 0;
void expect(bool ok, const char* what, int item, int s) {
    if (ok) return;
    if (fails++ < 5) std::printf("FAIL %s: item %d step %d\n", what, item, s);
}

// Items of the given numbers of steps, the wait of step `at` of item `die` giving up.
void run(const int* steps, int items, int die, int at) {
    Barrier b[Stages::kBars];
    unsigned n = 0;
    auto stage = [&](unsigned q) {
        expect(b[Stages::bar(q)].pending == 0, "two groups on one phase", -1, (int)q);
        b[Stages::bar(q)].pending = 1;
    };
    for (int it = 0; it < items; ++it) {
        const int last = steps[it] - 1;
        stage(n);
        stage(n + 1);
        for (int s = 0; s <= last; ++s) {
            Barrier& w = b[Stages::bar(n)];
            expect(!w.passes(Stages::parity(n)), "the wait passes before its copies land", it, s);
            if (it == die && s == at) {
                for (unsigned q = n; q != Stages::in_flight_end(n, s, last); ++q) {
                    Barrier& d = b[Stages::bar(q)];
                    expect(d.pending == 1 && !d.passes(Stages::parity(q)), "a wait for no copy", it, s);
                    d.pending = 0;
                    ++d.phase;
                }
                for (const Barrier& d : b) expect(d.pending == 0, "copies left in flight", it, s);
                return;
            }
            w.pending = 0;
            ++w.phase;
            expect(w.passes(Stages::parity(n)), "the wait does not pass", it, s);
            ++n;
            if (s + 2 <= last) stage(n + 1);
        }
    }
    for (const Barrier& d : b) expect(d.pending == 0, "copies left after the last item", items, 0);
}

}  // namespace

int main() {
    const int steps[] = {6, 7, 10, 5, 6, 9};  // an item of z planes takes z + 5 steps
    for (int die = 0; die < 6; ++die)
        for (int at = 0; at < steps[die]; ++at) run(steps, 6, die, at);
    run(steps, 6, -1, 0);
    std::printf(fails ? "stages check failed\n" : "stages check ok\n");
    return fails ? 1 : 0;
}
