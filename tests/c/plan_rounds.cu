// Which rounds of a plan the final reduction gives a warp each: prints, for
// every round left to a thread, its two instances' partials.  Argument: the
// number of rounds (partials: 1 .. 5 of the first instance, 0 .. 40 of the
// second).
#include <cstdio>
#include <cstdlib>

#include "internal.h"

int main(int argc, char **argv)
{
    const u32 n = argc > 1 ? (u32)atoi(argv[1]) : 0;
    Plan P;
    for (u32 k = 0; k < n; k++) {
        RoundRef R{};
        R.nchunks = 1 + k % 5;
        R.nchunks2 = k % 3 ? 0 : k % 41;
        P.rounds.push_back(R);
    }
    sort_tasks(P);
    printf("%u %zu\n", P.nbig, P.rounds.size());
    for (size_t k = P.nbig; k < P.rounds.size(); k++) printf("%u %u\n", P.rounds[k].nchunks, P.rounds[k].nchunks2);
    return 0;
}
