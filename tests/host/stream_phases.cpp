// The barrier waits of the streaming tensor-core kernel, against every state that a barrier can be in when they are made.  A wait
// tests the parity of a phase: with `done` phases complete it passes when done and the phase differ in parity.  It must not pass
// before the phase is complete, whatever the speed of the other warps: for every count of complete phases between what the
// waiting warp knows of (from its waits before) and what can have happened at most.
#include <cstdio>

#include "fdqp_plan.h"

using namespace fdqp;

static long checked = 0, failed = 0;

static void check(const char* what, int known, int most, int phase, int nb, int kb0, int n, int sets, int a, int w) {
    for (int done = known; done <= most; ++done) {
        ++checked;
        const bool passes = ((done ^ phase) & 1) != 0;
        if (passes && done <= phase && ++failed <= 20)
            std::printf("%s: phase %d passes with %d complete: K blocks %d, first %d, range %d, accumulator sets %d, stages %d + %d\n", what, phase, done,
                        nb, kb0, n, sets, w, a);
    }
}

// A range of n blocks that begins with block kb0 of a tile of nb; a: stages of converted weights, w: of packed ones.
static void range(int nb, int kb0, int n, int sets, int a, int w) {
    const int segments = (kb0 + n - 1) / nb + 1;
    auto segment_end = [&](int idx) { return (idx + 1) * nb - kb0 < n ? (idx + 1) * nb - kb0 : n; };  // blocks of the range before it ends
    // complete phases of a barrier of sums when the range's first `blocks` blocks have been through the MMAs
    auto acc_done = [&](int bar, int blocks) {
        int done = 0;
        for (int i = 0; i < segments; ++i)
            if (st_acc_wait(sets, i, i + 1 == segments).bar == bar && segment_end(i) <= blocks) ++done;
        return done;
    };
    for (int g = 0; g < 2; ++g) {  // a conversion warp takes every second block
        int mma = 0;               // blocks that it knows to have been through the MMAs
        for (int j = g; j < n; j += 2) {
            int loaded = 0;  // loads into the block's stage that it knows to be complete: of its own blocks, and of those through the MMAs
            for (int b = j % w; b < j; b += w)
                if (b < mma || b % 2 == g) ++loaded;
            check("packed weights", loaded, j / w + 1, j / w, nb, kb0, n, sets, a, w);
            int freed = 0;
            for (int b = j % a; b < mma; b += a) ++freed;
            if (j >= a) {
                check("converted weights", freed, j / a, j / a - 1, nb, kb0, n, sets, a, w);
                mma = j - a + 1;
            }
        }
        const StAccWait full = st_acc_wait(sets, segments - 1, true);
        const int walked = sets == 1 && segments > 1 ? segment_end(segments - 2) : 0;  // one set: it reads every segment
        check("last sums", acc_done(full.bar, mma > walked ? mma : walked), acc_done(full.bar, n), (int)full.phase, nb, kb0, n, sets, a, w);
    }
    // the readers of all segments but the last one: warps of their own with two sets, the conversion warps with one
    for (int idx = 0; idx + 1 < segments; ++idx) {
        const StAccWait full = st_acc_wait(sets, idx, false);
        const int before = idx ? segment_end(idx - 1) : 0;
        check("sums", acc_done(full.bar, before), acc_done(full.bar, n), (int)full.phase, nb, kb0, n, sets, a, w);
    }
}

// The last release of every stage, for which the kernel waits before it ends: the loads of a range and the uses of each stage, counted as
// the kernel makes them.
static void releases(int nb, int kb0, int n, int ksteps_last, int x_steps, int stages) {
    int loads = 0;
    for (int u = kb0; u < kb0 + n; ++u)
        for (int j = 0; j < (u % nb == nb - 1 ? ksteps_last : 4); j += x_steps) ++loads;
    const int all = st_x_loads(kb0, kb0 + n, nb, x_steps, ksteps_last);
    bool wrong = all != loads;
    for (int s = 0; s < stages; ++s) {
        int uses = 0;
        for (int i = s; i < loads; i += stages) ++uses;
        wrong |= st_stage_uses(s, all, stages) != uses;
    }
    ++checked;
    if (wrong && ++failed <= 20)
        std::printf("releases: %d loads, %d counted: K blocks %d (%d k-steps), first %d, range %d, %d stages\n", all, loads, nb, ksteps_last, kb0, n, stages);
}

int main() {
    const int forms[3][2] = {{2, 3}, {2, 2}, {1, 2}};  // accumulator sets, stages of converted weights
    for (int nb = 1; nb <= 6; ++nb)
        for (int kb0 = 0; kb0 < nb; ++kb0)
            for (int n = 1; n <= 39; ++n)
                for (const auto& f : forms)
                    for (int w = kStMinW; w <= kStMaxW; ++w) range(nb, kb0, n, f[0], f[1], w);
    for (int nb = 1; nb <= 5; ++nb)
        for (int kb0 = 0; kb0 < nb; ++kb0)
            for (int n = 1; n <= 24; ++n)
                for (int ksteps_last = 1; ksteps_last <= 4; ++ksteps_last)
                    for (int x_steps = 2; x_steps <= 4; x_steps += 2)
                        for (int stages = 2; stages <= 12; ++stages) releases(nb, kb0, n, ksteps_last, x_steps, stages);
    std::printf("%ld states, %ld wrong\n", checked, failed);
    return failed ? 1 : 0;
}
