// Host-side rules of the library that need no GPU, one per command line argument; the exit
// status is the number of failed checks.
#include <climits>
#include <cstdio>
#include <cstring>

#include "lb_internal.h"

using namespace lbsc;

static int failures = 0;

static void expect(bool ok, const char* what)
{
    if (!ok) {
        std::printf("failed: %s\n", what);
        ++failures;
    }
}

// Bounded waits: a limit runs out after that many cycles, however large it is.
static void wait_limit()
{
    const long long limits[] = {1, 2000000000LL, LLONG_MAX / 2, LLONG_MAX};
    for (long long limit : limits) {
        for (long long first : {1LL, 1LL << 40, 1LL << 52}) {
            expect(!limit_passed(first, first, limit), "not at once");
            expect(!limit_passed(first, first + 1, limit), "not a cycle later");
            expect(!limit_passed(first, first + (limit < (1LL << 53) ? limit : 1LL << 53), limit),
                   "not within the limit");
            if (limit < (1LL << 53)) expect(limit_passed(first, first + limit + 1, limit), "after it");
        }
    }
}

// Steps share a launch only where that is the faster way: either side of each line, at shapes
// that were measured on both.
static void shared_launches()
{
    // pairs: enough sites, and not for a second strip of two columns
    expect(pairs_pay(760, 760, 64, 4) && pairs_pay(2050, 1999, 128, 4) && pairs_pay(140, 7490, 64, 4) &&
               pairs_pay(64, 16384, 64, 4) && pairs_pay(246, 5284, 64, 2) && pairs_pay(241, 4149, 64, 4) && pairs_pay(241, 17404, 128, 4) &&
               pairs_pay(5, 3355444, 128, 4),
           "pairs");
    expect(!pairs_pay(500, 500, 64, 4) && !pairs_pay(122, 8000, 64, 4) && !pairs_pay(121, 138655, 128, 4) &&
               !pairs_pay(5, 52429, 64, 4) && !pairs_pay(8, 40000, 64, 4) && !pairs_pay(241, 2489, 64, 4) && !pairs_pay(241, 4149, 64, 2) &&
               !pairs_pay(140, 3214, 64, 4),
           "no pairs");
    // traced states in pairs: beyond L2 or nearly
    expect(traced_pairs_pay(1300, 1300, 128, 2) && traced_pairs_pay(8192, 8192, 128, 4) &&
               traced_pairs_pay(361, 46475, 128, 4) && traced_pairs_pay(1024, 1269, 64, 4) &&
               traced_pairs_pay(1024, 1562, 64, 2),
           "traced pairs");
    expect(!traced_pairs_pay(740, 740, 64, 4) && !traced_pairs_pay(1024, 1269, 64, 2) &&
               !traced_pairs_pay(1024, 1024, 64, 4) && !traced_pairs_pay(122, 34380, 128, 4) &&
               !traced_pairs_pay(241, 69616, 128, 4),
           "no traced pairs");
    // batches: {pairs, traced pairs} of `count` lattices at a shape of their single steps
    auto batch = [](int count, int nx, int ny, int block_x, int rows, int elem_bytes) {
        std::vector<std::pair<int, int>> sizes(count, {nx, ny});
        std::vector<int4> tiles;
        pair_tiles(sizes, elem_bytes, 152, tiles);
        const int strips = (nx + block_x - 3) / (block_x - 2);
        BatchWork w{count * strips * ((ny + rows - 1) / rows), block_x, rows < ny ? rows : ny,
                    (int)tiles.size(), 0, elem_bytes, 152};
        for (const int4& t : tiles) w.pair_chunk = t.w - t.z > w.pair_chunk ? t.w - t.z : w.pair_chunk;
        const double e = batch_paired_over_single(w);
        return std::make_pair(batch_pairs_pay(block_x, rows, (double)nx / single_columns(nx, block_x), e),
                              batch_traced_pairs_pay(block_x, rows, ny,
                                                     (double)pair_columns(nx) / single_columns(nx, block_x), e));
    };
    const struct {
        int count, nx, ny, block_x, rows, elem_bytes;
        bool pairs, traced;
    } batches[] = {{74, 125, 75, 128, 32, 2, true, true},   {8, 122, 2000, 128, 32, 4, true, true},
                   {9, 512, 512, 128, 32, 4, true, true},   {96, 64, 64, 64, 8, 4, true, true},
                   {200, 5, 5, 128, 32, 4, true, false},    {500, 5, 5, 64, 8, 2, true, false},
                   {24, 16, 16, 64, 32, 2, true, true},     {30, 128, 128, 64, 8, 2, true, false},
                   {2, 5, 20000, 128, 32, 4, true, true},   {8, 5, 20000, 64, 32, 4, false, false},
                   {500, 12, 40, 64, 8, 4, false, false},   {500, 37, 37, 64, 16, 4, false, false},
                   {24, 5, 400, 64, 8, 2, false, false},    {74, 125, 75, 128, 8, 2, false, false},
                   {8, 122, 2000, 64, 32, 4, true, false},  {74, 122, 122, 64, 32, 4, true, true}};
    for (const auto& t : batches) {
        const auto got = batch(t.count, t.nx, t.ny, t.block_x, t.rows, t.elem_bytes);
        std::printf("%d of %dx%d at %dx%d: ", t.count, t.nx, t.ny, t.block_x, t.rows);
        expect(got.first == t.pairs && (got.first && got.second) == t.traced, "pairs of a batch");
        std::printf("\n");
    }
    // held launches of few steps: not of large tiles (152 SMs)
    const struct {
        int n;
        bool om1;
        int least;
    } held[] = {{70, true, 2},   {400, true, 2},  {512, true, 3}, {560, true, 3},  {680, true, 4},
                {720, true, 5},  {400, false, 2}, {512, false, 3}, {560, false, 4}};
    for (const auto& h : held) {
        ResidentBuf b;
        expect(resident_plan(h.n, h.n, h.om1, 152, b), "a held lattice");
        expect(held_least(b.tw * b.th, h.om1) == h.least, "fewest steps of a held launch");
    }
}

// A captured graph's buffers: pairs and single steps of any count swap them alike.
static void swaps()
{
    for (int te : {0, 1, 2, 3, 4, 10})
        for (bool traced : {false, true})
            for (long long t = 0; t < 12; ++t)
                for (long long n = 0; n < 40; ++n) {
                    long long k = 0, pairs = 0, singles = pairs_made(t, n, te, traced) % 2 ? 2 : 0;
                    long long swapped = 0;
                    while (k < n) {
                        bool pair = pair_at(t + k, n - k, te, traced);
                        if (singles == 1 || (singles == 2 && pair)) {
                            --singles;
                            pair = false;
                        }
                        expect(!pair || te == 0 || (t + k + 1) % te != 0, "no pair onto a trace row");
                        k += pair ? 2 : 1;
                        pairs += pair;
                        ++swapped;
                    }
                    expect(k == n && pairs % 2 == 0 && swapped % 2 == n % 2, "swaps");
                }
}

int main(int argc, char** argv)
{
    const char* which = argc > 1 ? argv[1] : "";
    if (!std::strcmp(which, "wait_limit")) wait_limit();
    else if (!std::strcmp(which, "shared_launches")) shared_launches();
    else if (!std::strcmp(which, "swaps")) swaps();
    else expect(false, "no such check");
    return failures;
}
