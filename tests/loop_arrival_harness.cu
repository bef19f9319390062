// Host program: the decisions of a drafting loop whose counter starts at `leftover`, as loop_arrival() takes them.
// Prints the number of iterations until the loop ends (at most `give_up`) and whether an overrun was seen.
#include <cstdio>
#include <cstdlib>

#include "svip_draft.cuh"

int main(int argc, char** argv) {
    if (argc != 6) return 2;
    unsigned long long counter = std::strtoull(argv[1], nullptr, 10);
    const int B = std::atoi(argv[2]), lasts = std::atoi(argv[3]), max_iters = std::atoi(argv[4]), give_up = std::atoi(argv[5]);
    int body = 0, iter = 0, overrun = 0;
    bool condition = true;
    while (condition && body < give_up) {
        ++body;
        for (int i = 0; i < B; ++i) {           // every sequence goes on until iteration `lasts`
            counter += 1ull + (body < lasts ? 1ull << 32 : 0ull);
            const svip::LoopArrival r = svip::loop_arrival(counter, B);
            if (!r.closes) continue;
            counter = 0;
            overrun |= r.overrun;
            ++iter;
            condition = r.going > 0 && iter < max_iters;
        }
    }
    std::printf("%d %d\n", body, overrun);
    return 0;
}
