// The waits of the rotating accumulators (csrc/rotation.h) under any timing: two MMA
// warps and the drains, stepped in random order, with barriers that answer by the parity
// of a phase as mbarriers do.  A warp may be `ring` chunks ahead of the other.  Fails
// if a warp's wait lets it use a buffer whose last use is not drained, or nothing can move.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "rotation.h"

struct Use {
    int t, buf;
};

int main(int argc, char **argv) {
    const int trials = argc > 1 ? atoi(argv[1]) : 1000;
    std::mt19937 rng(1);
    for (int trial = 0; trial < trials; trial++) {
        const int top = (const int[]){2, 6, 20, 48}[trial % 4], ring = (const int[]){4, 6, 7, 16}[rng() % 4];
        std::vector<int> nc(2 + rng() % 12);
        for (int &n : nc) n = 1 + rng() % top;
        if (trial == 0) nc = {16, 16, 12, 16, 16, 12};
        if (trial == 1) nc = {44, 44, 44};
        // the ends in the drains' order, as the kernel's drain warps take them
        std::vector<Use> ends;
        std::vector<uint32_t> signal;
        {
            AccState s;
            auto end = [&](int t) {
                ends.push_back({t, (int)s.b[t]});
                signal.push_back(s.signal());
                s.end(t);
            };
            for (int n : nc) {
                for (int c = 3; c + 1 < n; c += 4) end(drained_after(c, n));
                end(0);
                end(1);
            }
        }
        int phases[AccState::kEnds] = {};                       // completed phases of each barrier
        size_t drained = 0, committed[2] = {0, 0};              // ends drained; ends of Re and Im whose MMAs are done
        std::vector<size_t> use_of[2];                          // warp t's i-th end: its number
        for (size_t e = 0; e < ends.size(); e++) use_of[ends[e].t].push_back(e);
        struct Warp {
            AccState st;
            size_t unit = 0, uses = 0;
            int c = 0, chunk = 0;
            bool fresh = true;
        } w[2];
        // a buffer's last end before warp t's use number u
        auto last_before = [&](int t, size_t u) {
            const size_t e = use_of[t][u];
            for (long i = (long)e - 1; i >= 0; i--)
                if (ends[i].buf == ends[e].buf) return i;
            return -1l;
        };
        const unsigned seldom = (const unsigned[]){3, 12, 60}[rng() % 3];   // the drains move once in so many steps
        long idle = 0;
        while (drained < ends.size()) {
            if (++idle > 100000) return printf("trial %d: nothing moves\n", trial), 1;
            if (rng() % seldom == 0) {                          // the next end, once its MMAs are done
                const Use &u = ends[drained];
                size_t i = 0;
                while (use_of[u.t][i] != drained) i++;
                if (committed[u.t] <= i) continue;
                phases[signal[drained]]++;
                drained++;
                idle = 0;
                continue;
            }
            const int t = (int)(rng() & 1);
            Warp &a = w[t];
            if (a.unit == nc.size() || a.chunk - w[1 - t].chunk >= ring) continue;
            const int n = nc[a.unit], dr = drained_after(a.c, n);
            const bool end = a.c + 1 == n || dr == t;
            if (a.fresh) {
                const uint32_t buf = a.st.b[t], on = a.st.wait_on(buf);
                if ((uint32_t)((phases[on] + 1) & 1) != a.st.wait_parity(buf)) continue;   // not the last phase
                const long need = last_before(t, a.uses);
                if ((int)buf != ends[use_of[t][a.uses]].buf || (need >= 0 && (size_t)need >= drained))
                    return printf("trial %d: warp %d took buffer %u at chunk %d before end %ld was drained\n", trial, t, buf,
                                  a.chunk, need), 1;
            }
            idle = 0;
            a.fresh = end;
            if (end) {
                a.uses++;
                committed[t]++;
            }
            if (dr >= 0) a.st.end(dr);
            a.chunk++;
            if (++a.c == n) {
                a.st.end(0);
                a.st.end(1);
                a.c = 0;
                a.unit++;
            }
        }
    }
    puts("ok");
    return 0;
}
