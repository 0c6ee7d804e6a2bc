// Host harness of csrc/awpm_rules.h: a rule's name and its arguments from the
// command line, its value to standard output.
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "awpm_rules.h"

using namespace awpm;

int main(int argc, char **argv)
{
    auto arg = [&](int k) { return argc > k ? std::atoll(argv[k]) : 0ll; };
    const char *what = argc > 1 ? argv[1] : "";
    if (!std::strcmp(what, "max_entries"))
        std::printf("%lld\n", (long long)kMaxEntries);
    else if (!std::strcmp(what, "tile_pos"))
        std::printf("%lld\n",
                    (long long)tile_pos((int32_t)arg(2), (int32_t)arg(3), (int)arg(4)));
    else if (!std::strcmp(what, "blocks_pay")) {  // n and tiles of each matrix
        BatchLoad load;
        for (int k = 2; k + 1 < argc; k += 2)
            load.add((int32_t)arg(k), arg(k + 1));
        std::printf("%d\n", load.blocks_pay() ? 1 : 0);
    } else if (!std::strcmp(what, "small_too_many"))
        std::printf("%d\n", small_too_many((int32_t)arg(2)) ? 1 : 0);
    else if (!std::strcmp(what, "mcm_cluster"))  // tiles, n
        std::printf("%d\n", mcm_cluster((int32_t)arg(2), (int32_t)arg(3)) ? 1 : 0);
    else if (!std::strcmp(what, "weights_form"))  // tiles, n: 0 cluster, 1 thin, 2 full
        std::printf("%d\n", weights_cluster((int32_t)arg(2), (int32_t)arg(3)) ? 0
                            : weights_thin((int32_t)arg(2), (int32_t)arg(3)) ? 1 : 2);
    else
        return 1;
    return 0;
}
