// Work schedules of the tensor-core decode kernel and of the prompt phase's scoring: plain integer arithmetic, compiled for
// the device by nvcc and for the host by any C++ compiler (the CPU tests replay them: for every cache length that every
// tile has exactly one owner and that the partial slots suffice, for prompts that every run is visited once).
#pragma once

#if defined(__CUDACC__)
#define MKV_HD __host__ __device__
#else
#define MKV_HD
#endif

namespace mkv {

constexpr int kSchedTile = 128;      // keys per tile

struct Item {
    int unit, tile0, nk;      // tiles [tile0, tile0 + nk) of the unit
};

// The same deterministic walk over a CTA's items in every role of the kernel.  With nt tiles per unit at
// the current cache length, global tile i is tile i % nt of unit i / nt, and CTA c of the
// E = min(grid, U * nt) working CTAs owns tiles [c * T / E, (c + 1) * T / E), T = U * nt: every
// working CTA owns at least one tile and consecutive items belong to different units.
// Order of a CTA's items: if its range ends inside a unit, that last piece comes first, then the rest in tile order.
// A unit cut by a range boundary is then worked on early by both CTAs that hold a piece of it (the one before the
// boundary starts with it, the one after it takes it first or second), so its cross-CTA merge runs while tiles
// still stream, and the item a CTA ends with is a unit all of its own, whose epilogue needs no other CTA.
//
// Whole units: where the ranges can be cut between units at the price of less than kMergeTiles tiles on the busiest CTA,
// they are.  A unit that two CTAs share costs a partial, a ticket and a second epilogue in global memory, a chain of
// round trips of about 5 us at the end of the launch; a tile costs about 1.26 us.  (112 units x 8 heads of 600 / 1030 /
// 2030 slots on 112 CTAs against 148 in equal shares: 21.1 / 29.7 / 43.3 us per step against 26.4 / 36.3 / 43.1, shares
// longer by 1.2 / 2.2 / 3.9 tiles; 256 units of 512 slots on 128 CTAs 20.7 against 29.3, 8192 of them 443 against 493.)
constexpr int kMergeTiles = 4;

// Whether whole units pay for a context of this capacity, and then at every fill.  (WHOLE is a template parameter because the
// other kind of walk, with a run-time switch in it, cost the flagship's step 0.4 us.)
inline bool sched_whole(int U, int cap, int grid)
{
    const long long nt = (cap + kSchedTile - 1) / kSchedTile;
    return U > grid && ((U + grid - 1) / grid * (long long)grid - U) * nt < (long long)kMergeTiles * grid;
}

template <bool WHOLE>
struct WalkT {
    int tile, tile_begin, tile_end;   // the host keeps U * tiles per unit below 2^31
    int nat_end;      // end of the part of the range that is handed out in tile order
    int lead_nk;      // tiles of the piece handed out first (0: none, or already handed out)
    int nt;           // tiles per unit
    int unit, off;    // unit and tile inside it of `tile`
    int nitems;       // items returned so far (= units seen: ring loads, partials)
    int T0;           // tiles of the items already advanced over
    int eff;          // working CTAs
    int cta;          // this CTA
    long long total;
    MKV_HD WalkT(int U, int n, int grid, int cta_index)
    {
        nt = (n + kSchedTile - 1) / kSchedTile;
        total = (long long)U * nt;
        eff = (int)(total < (long long)grid ? total : (long long)grid);
        cta = cta_index;
        if (cta < eff) {
            if (WHOLE) {
                tile = (int)((unsigned)U * cta / eff) * nt;           // (at most 2^24 units)
                tile_end = (int)((unsigned)U * (cta + 1) / eff) * nt;
            } else if (narrow()) {
                tile = (int)((unsigned)total * cta / eff);
                tile_end = (int)((unsigned)total * (cta + 1) / eff);
            } else {
                tile = (int)(total * cta / eff);
                tile_end = (int)(total * (cta + 1) / eff);
            }
        } else {
            tile = tile_end = 0;
        }
        tile_begin = tile;
        unit = tile / nt;         // n >= 1: a context holds at least its prompt
        off = tile - unit * nt;
        nitems = 0; T0 = 0;
        nat_end = tile_end;
        lead_nk = 0;
        if (tile_end > tile_begin) {
            const int ul = (tile_end - 1) / nt;                 // the unit the range ends in
            const int first = ul * nt;                          // its first tile
            if (tile_end != first + nt && first > tile_begin) { // the range ends inside it and starts before it
                nat_end = first;
                lead_nk = tile_end - first;
            }
        }
    }
    MKV_HD bool next(Item &x)
    {
        if (lead_nk > 0) {
            x.unit = nat_end / nt;
            x.tile0 = 0;
            x.nk = lead_nk;
            lead_nk = 0;
            return true;
        }
        if (tile >= nat_end) return false;
        x.unit = unit;
        x.tile0 = off;
        x.nk = nt - off < nat_end - tile ? nt - off : nat_end - tile;
        tile += x.nk;
        off += x.nk;
        if (off == nt) { off = 0; ++unit; }
        return true;
    }
    MKV_HD void advance(const Item &x)
    {
        T0 += x.nk;
        ++nitems;
    }
    // the CTA that owns global tile i: the largest c with c * T / E <= i
    MKV_HD int owner(long long i) const
    {
        if (WHOLE) i = i / nt * nt + nt - 1;            // the unit's last tile: (u + 1) * nt * E / T = (u + 1) * E / U
        if (narrow()) return (int)((((unsigned)i + 1) * eff - 1) / (unsigned)total);
        return (int)(((i + 1) * eff - 1) / total);
    }
    // products of a tile and a CTA index fit in 32 bits (64-bit divisions are slow, and stand at the start of every launch)
    MKV_HD bool narrow() const { return total < (1ll << 24) && eff < 256; }
    // How many CTAs hold tiles of unit u, and this CTA's index among them.
    MKV_HD int ctas_of_unit(int u, int &my_index) const
    {
        if (WHOLE) { my_index = 0; return 1; }
        const long long i0 = (long long)u * nt;
        const int c0 = owner(i0), c1 = owner(i0 + nt - 1);
        my_index = cta - c0;
        return c1 - c0 + 1;
    }
};

using Walk = WalkT<false>;

// Grid of the persistent kernel.  `splits_hint` > 0 asks for about that many CTAs per unit (ranges of
// cap_tiles / splits_hint tiles).  Otherwise one CTA per SM, or a multiple of the units where that leaves the shares less
// than kMergeTiles / 2 tiles longer: every unit is then cut into equal parts of its own and never shared by more CTAs than
// it has parts (8 at most, what the fast epilogue merges), or is one CTA's alone, for which kMergeTiles are paid.
// (64 units of 8 tiles in 128 parts 17.4 us per step against 21.1; 32 units of 16 tiles in 128 parts 18.8 against 22.9.)
// Few units always get the 8 parts, although some SMs then stay idle: 8 units of 32 / 128 / 512 tiles take 19.2 / 46.5 / 157 us in
// 8 parts and 24 / 45 / 139 in equal shares of 148 CTAs, whose 18 partials are merged first; 1 unit of 128 44 against 67; 16 of 512
// 173 against 176.
inline int sched_grid(int U, int cap, int splits_hint, int n_sm)
{
    const long long ntiles = (cap + kSchedTile - 1) / kSchedTile, total = (long long)U * ntiles;
    long long grid = n_sm;
    if (splits_hint > 0) {
        const long long chunk = (ntiles + splits_hint - 1) / splits_hint;
        grid = (total + chunk - 1) / chunk;
        if (grid > n_sm) grid = n_sm;
    } else if (U <= n_sm) {
        long long parts = n_sm / U;
        if (parts > 8) parts = 8;
        if (parts > ntiles) parts = ntiles;
        if (ntiles * n_sm - total < (long long)kMergeTiles * n_sm) grid = U;
        else if (parts > 1 && 2 * (((ntiles + parts - 1) / parts) * n_sm - total) < (long long)kMergeTiles * n_sm) grid = U * parts;
        else if (parts == 8) grid = U * parts;
    }
    if (grid > total) grid = total;
    return (int)(grid < 1 ? 1 : grid);
}

// Upper bound, over every cache length up to cap, of the CTAs that hold tiles of one unit
// (= partial slots a unit needs).
inline int sched_partials_per_unit(int U, int cap, int grid)
{
    const int ntiles = (cap + kSchedTile - 1) / kSchedTile;
    int worst = 1;
    for (int nt = 1; nt <= ntiles; ++nt) {
        const long long total = (long long)U * nt;
        const long long eff = total < grid ? total : grid;
        const long long len = total / eff;                     // shortest range of a CTA
        long long c = (nt + len - 1) / len + 1;
        if (c > nt) c = nt;
        if (c > worst) worst = (int)c;
    }
    return worst;
}

// ---- prompt phase: the key tiles of a unit's prompt in runs of `run` tiles (the last one shorter), unit after unit
constexpr int kRunTable = 512;       // most entries of the table of the rows' runs

struct RunAt {
    int unit, r, P;                // the unit, which of its runs it is, the length of its prompt
};

struct RunOrder {
    const int *shift;              // [B] how much shorter a batch row's prompt is than the longest one, or nullptr
    int P, Hkv, B, run, most;      // most: runs of the longest prompt
    int u0;                        // first unit of the batch; with prompts of different lengths also
    int first, layer;              // the runs of the units before it, and of the units of a layer
    int step, entries;             // batch rows of a table entry, entries
    MKV_HD int runs(int b) const
    {
        const int tiles = (P - (shift != nullptr ? shift[b] : 0) + kSchedTile - 1) / kSchedTile;
        return (tiles + run - 1) / run;
    }
    // runs of one unit of each of the rows e * step .. (e + 1) * step - 1
    MKV_HD int entry(int e) const
    {
        int n = 0;
        for (int b = e * step; b < (e + 1) * step && b < B; ++b) n += runs(b);
        return n;
    }
    // The i-th run from the first one of unit u0 on.  `before`: the sum of the entries in front of each entry and, behind the last one, of them all (not used where the
    // lengths are equal).  It is on the way of a CTA's next loads, so two divisions are all it takes.
    MKV_HD RunAt place(int i, const int *before) const
    {
        if (shift == nullptr) {
            const int u = (int)((unsigned)i / (unsigned)most);
            return RunAt{u0 + u, i - u * most, P};
        }
        i += first;
        const int l = (int)((unsigned)i / (unsigned)layer);
        i -= l * layer;
        int lo = 0, hi = entries;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (before[mid] * Hkv <= i) lo = mid;
            else hi = mid;
        }
        i -= before[lo] * Hkv;
        int b = lo * step, n = before[lo + 1] - before[lo];
        if (step > 1) {
            n = runs(b);
            while (i >= n * Hkv) { i -= n * Hkv; n = runs(++b); }
        }
        const int len = P - shift[b], h = (int)((unsigned)i / (unsigned)n);
        return RunAt{(l * B + b) * Hkv + h, i - h * n, len};
    }
};

// The order of the runs of units u0 .. u0 + count - 1, and their number.
inline RunOrder run_order(const int *shift, int P, int Hkv, int B, int run, int u0, int count, int *items)
{
    RunOrder o = {shift, P, Hkv, B, run, ((P + kSchedTile - 1) / kSchedTile + run - 1) / run, u0, 0, 0, 0, 0};
    if (shift == nullptr) { *items = count * o.most; return o; }
    o.step = (B + kRunTable - 1) / kRunTable;
    o.entries = (B + o.step - 1) / o.step;
    for (int b = 0; b < B; ++b) o.layer += o.runs(b) * Hkv;
    auto before = [&](int u) {
        const int row = u / Hkv;
        int n = row / B * o.layer + (u - row * Hkv) * o.runs(row % B);
        for (int b = 0; b < row % B; ++b) n += o.runs(b) * Hkv;
        return n;
    };
    o.first = before(u0);
    *items = before(u0 + count) - o.first;
    return o;
}

constexpr int kPromptCtas = 148;         // CTAs of the scoring's launches
// Up to how many tiles one launch makes each visit, as their keys stay in L2 (96 MB) by themselves.  With two blocks of rows fewer:
// what a launch of both visits gains by mixing them grows with the work per tile.  (Prompt phase in us, both visits in one launch -> a
// launch each; units x tokens, 128 rows: 64 x 2000 97 -> 77, 256 x 1499 139 -> 131, 64 x 6107 137 -> 132, 256 x 2000 156 -> 155; 240 rows:
// 32 x 9000 161 -> 146, 128 x 3035 178 -> 190.)
MKV_HD inline int prompt_apart_tiles(int rows) { return rows <= 128 ? 3072 : 2304; }

// Tiles of a run.  Eight for many tiles: an item then brings 256 KB of keys beside the 32 KB of its queries, while the items between
// the two visits of a run stay in L2 (256 units x 6144 tokens: 355 us with four, 334 with eight, 330 with sixteen at the time).
// Where nothing is selected, and items are taken by ticket once, two items per CTA.  With a launch for each visit, the length that fills the rounds of items best, in items as short as that allows: an item's own time
// is some third of a tile's, and more where there are many statistics of its unit to merge.  Rounds of a few items less than there are
// SMs, as now and then one of them is not free when the launch starts (2 units x 259 tiles, runs of seven: 148 items 127 us or 157).
// (Before, tiles / 296 and both visits in one launch from 17 runs per unit on -> now: 8 x 25600 104 -> 91, 2 x 60000 120 -> 94, 4 x 40000 with
// 256 rows 136 -> 115, 112 x 1200 with 240 rows 115 -> 104, 32 x 1500 64 -> 54.)
inline int prompt_run(const int *shift, int P, int Hkv, int B, int units, int rows, bool select)
{
    int tiles, best = 8, least = 0;
    run_order(shift, P, Hkv, B, 1, 0, units, &tiles);
    if (tiles > prompt_apart_tiles(rows)) return best;
    const int longest = (P + kSchedTile - 1) / kSchedTile;
    if (!select) {
        const long long run = ((long long)units * longest + 2 * kPromptCtas - 1) / (2 * kPromptCtas);
        return run < best ? (int)run : best;
    }
    for (int run = longest > 1 ? 2 : 1; run <= 24 && run <= longest; ++run) {
        int items;
        const RunOrder o = run_order(shift, P, Hkv, B, run, 0, units, &items);
        const int rounds = (items + kPromptCtas - 5) / (kPromptCtas - 4);
        const int cost = rounds * (10 * run + 3 + o.most / 4) + run;      // tenths of a tile
        if (least == 0 || cost < least) { least = cost; best = run; }
    }
    return best;
}

// The t-th item of a launch that visits each of `items` runs twice (`more`: not beyond the last one).  Kind 1: the first visit of run i,
// 2: its second one, which comes behind the first visits of the `lag` runs after it.
struct RunVisit {
    int kind, i;
    bool more;
};
MKV_HD inline RunVisit prompt_item(int t, int items, int lag)
{
    if (lag > items) lag = items;
    const int s = t - lag, both = 2 * (items - lag);
    if (s < 0) return RunVisit{1, t, true};
    if (s < both) return RunVisit{1 + (s & 1), (s >> 1) + ((s & 1) ? 0 : lag), true};
    const int i = s - both + (both >> 1);
    return RunVisit{2, i, i < items};
}

// Distance of the two visits, in runs (none of which is empty, whatever the prompts' lengths).  A unit's last statistics are
// published some two items after they have been handed out, while every CTA takes two items of either kind: with fewer than some
// 200 runs in between the scores wait for them.  With more the keys in between leave L2 (400 runs of eight tiles are 105 MB), which costs
// little where the launch ends soon after.  (Prompt phase in us, 200 / 240 / 300 / 400 runs in between; units x tokens: 24 x 17600 133 / 132 / 131 /
// 120, 64 x 9000 219 / 213 / 207 / 207, 256 x 3500 195 / 190 / 182 / 181; 256 x 6144 292 / 286 / 284 / 282, but 367 at 240 and 371 at 400 with
// its first step and prompt after prompt; 2048 x 3000 1030 / 1032 / 1054 / 1068, 256 x 131072 3341 / 3319 / 3546 / 3585.)
MKV_HD inline int prompt_lag(int items, int longest_runs) { return longest_runs + (items <= 1024 ? 400 : 240); }

}  // namespace mkv
