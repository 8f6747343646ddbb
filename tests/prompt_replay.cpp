// Replays the order in which the prompt phase's scoring visits the key tiles, for prompts of the given lengths, and checks what
// the kernel relies on:
//   - every run of every unit's own prompt is visited once by each kind of item, in the units' order, and no other run is;
//   - between a unit's last first visit and its first second visit lie the first visits of 240 other runs at least (all that are left at the
//     end), so that its statistics are there in time, and a run's visits are no further apart than the longest prompt and those;
//   - the host's counts of runs agree with the order, also for batches that start and end inside a row, and the table of a layer's
//     runs has room for any number of rows.
//   - with run 0: the run that the host chooses leaves no CTA much more than its share of the tiles.
// usage: prompt_replay Hkv layers run P shift_0 .. shift_{B-1} (no shifts: B = 1, equal lengths)   -> "ok <items>" or a diagnostic
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "mkv_schedule.h"

using namespace mkv;

#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main(int argc, char **argv)
{
    if (argc < 5) { fprintf(stderr, "usage: %s Hkv layers run P shift...\n", argv[0]); return 2; }
    const int Hkv = atoi(argv[1]), layers = atoi(argv[2]), P = atoi(argv[4]);
    int run = atoi(argv[3]);
    std::vector<int> shift;
    for (int i = 5; i < argc; ++i) shift.push_back(atoi(argv[i]));
    const int B = shift.empty() ? 1 : (int)shift.size(), U = layers * B * Hkv;
    const int *sh = shift.empty() ? nullptr : shift.data();
    if (run == 0) {
        run = prompt_run(sh, P, Hkv, B, U, 128, true);
        int items;
        const RunOrder order = run_order(sh, P, Hkv, B, run, 0, U, &items);
        std::vector<int> before(1, 0);
        for (int e = 0; e < order.entries; ++e) before.push_back(before.back() + order.entry(e));
        std::vector<long long> cta(kPromptCtas, 0);
        long long all = 0, most = 0;
        std::vector<int> taken(items, 0);
        for (int round = 0; round * kPromptCtas < items; ++round)
        for (int c = 0; c < kPromptCtas; ++c) {                    // (as in a launch of one visit)
            const int t = round * kPromptCtas + (c + round) % kPromptCtas;
            if (t >= items) continue;
            CHECK(taken[t]++ == 0);
            const RunAt at = order.place(t, before.data());
            const int left = (at.P + 127) / 128 - at.r * run;
            const int n = left < run ? left : run;
            CHECK(n >= 1);
            all += n;
            most = std::max(most, cta[c] += n);
        }
        printf("run %d, the busiest of %d CTAs has %lld of %lld tiles\n", run, kPromptCtas, most, all);
        if (all <= prompt_apart_tiles(128)) CHECK(4 * kPromptCtas * (most - 2) <= 5 * all);            // a quarter and two tiles more than its share
    }
    const int longest = ((P + 127) / 128 + run - 1) / run;
    long long seen_total = 0;
    for (int u0 : {0, 1, Hkv, U / 3, U - 1}) {
        const int count = u0 == 0 ? U : (U - u0 + 1) / 2;
        if (u0 < 0 || u0 >= U || count < 1) continue;
        std::vector<int> unit, r;                                  // the runs, one after the other
        for (int u = u0; u < u0 + count; ++u) {
            const int len = P - (sh ? sh[(u / Hkv) % B] : 0), n = ((len + 127) / 128 + run - 1) / run;
            for (int k = 0; k < n; ++k) { unit.push_back(u); r.push_back(k); }
        }
        const int items = (int)unit.size();
        int counted = -1;
        const RunOrder order = run_order(sh, P, Hkv, B, run, u0, count, &counted);
        CHECK(counted == items);
        std::vector<int> before(1, 0);
        for (int e = 0; e < order.entries; ++e) before.push_back(before.back() + order.entry(e));
        CHECK((int)before.size() <= kRunTable + 1 && (!sh || before.back() * Hkv == order.layer));
        const int lag = prompt_lag(items, longest);
        CHECK(lag - longest >= 240 && lag - longest <= 400);
        std::vector<int> at1(items, -1), at2(items, -1);
        for (int t = 0;; ++t) {
            const RunVisit v = prompt_item(t, items, lag);
            if (!v.more) { CHECK(t == 2 * items); break; }
            const int i = v.i, kind = v.kind;
            CHECK(i >= 0 && i < items);
            const RunAt placed = order.place(i, before.data());
            CHECK(placed.unit == unit[i] && placed.r == r[i] && placed.P == P - (sh ? sh[(unit[i] / Hkv) % B] : 0));
            std::vector<int> &at = kind == 1 ? at1 : at2;
            CHECK(at[i] < 0 && (i == 0 || at[i - 1] >= 0));
            at[i] = t;
        }
        for (int i = 0; i < items; ++i) {
            CHECK(at1[i] >= 0 && at2[i] > at1[i]);
            if (r[i] != 0) continue;
            int last = i;                                          // the unit's last run
            while (last + 1 < items && unit[last + 1] == unit[i]) ++last;
            const int need = items - 1 - last < 240 ? items - 1 - last : 240;
            for (int k = 1; k <= need; ++k) CHECK(at1[last + k] < at2[i]);
            if (i + lag + 1 < items) CHECK(at1[i + lag + 1] > at2[i]);
        }
        seen_total += items;
    }
    printf("ok %lld\n", seen_total);
    return 0;
}
