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

int main(int argc, char** argv)
{
    const char* which = argc > 1 ? argv[1] : "";
    if (!std::strcmp(which, "wait_limit")) wait_limit();
    else expect(false, "no such check");
    return failures;
}
