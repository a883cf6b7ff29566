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
    expect(pairs_pay(760, 760, 64) && pairs_pay(2050, 1999, 128) && pairs_pay(140, 7490, 64) &&
               pairs_pay(64, 16384, 64) && pairs_pay(241, 17404, 128) && pairs_pay(5, 3355444, 128),
           "pairs");
    expect(!pairs_pay(500, 500, 64) && !pairs_pay(122, 8000, 64) && !pairs_pay(121, 138655, 128) &&
               !pairs_pay(5, 52429, 64) && !pairs_pay(8, 40000, 64) && !pairs_pay(241, 1200, 64),
           "no pairs");
    // traced states in pairs: beyond L2
    expect(traced_pairs_pay(1300, 1300, 128) && traced_pairs_pay(8192, 8192, 128) &&
               traced_pairs_pay(361, 46475, 128),
           "traced pairs");
    expect(!traced_pairs_pay(740, 740, 64) && !traced_pairs_pay(1150, 1150, 64) &&
               !traced_pairs_pay(122, 34380, 128) && !traced_pairs_pay(241, 69616, 128),
           "no traced pairs");
    auto batch = [](int count, int nx, int ny, int block_x) {
        return batch_pairs_pay((long long)count * nx * ny, pair_columns(nx) * ny * count,
                               single_columns(nx, block_x) * ny * count);
    };
    expect(batch(96, 64, 64, 128) && batch(500, 5, 5, 64) && batch(4, 5, 20000, 128) &&
               batch(12, 130, 640, 64),
           "pairs of a batch");
    expect(!batch(4, 5, 20000, 64) && !batch(300, 12, 40, 64) && !batch(8, 122, 2000, 64),
           "no pairs of a batch");
    expect(batch_traced_pairs_pay(640, 32, 4) && batch_traced_pairs_pay(16, 32, 2) &&
               batch_traced_pairs_pay(64, 8, 4),
           "traced pairs of a batch");
    expect(!batch_traced_pairs_pay(5, 32, 4) && !batch_traced_pairs_pay(16, 8, 4) &&
               !batch_traced_pairs_pay(128, 8, 2),
           "no traced pairs of a batch");
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
