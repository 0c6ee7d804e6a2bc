// Host harness of csrc/awpm_fixed.h: quotients and logarithms of pairs and
// values read from standard input (raw doubles), results to standard output.
#include <cstdio>
#include <vector>

#include "awpm_fixed.h"

using namespace awpm;
static constexpr LogTable kTable = fx_make_log_table();

int main(int argc, char **argv)
{
    const bool log_mode = argc > 1 && argv[1][0] == 'l';
    std::vector<double> out;
    double a, b;
    while (std::fread(&a, 8, 1, stdin) == 1) {
        if (log_mode) {
            out.push_back(fx_double(log_below_one(fx_bits(a), kTable.e)));
            continue;
        }
        if (std::fread(&b, 8, 1, stdin) != 1)
            return 1;
        bool ok;
        const uint64_t q = quotient(fx_bits(a), make_scale(fx_bits(b)), ok);
        out.push_back(ok ? fx_double(q) : -1.0);
    }
    std::fwrite(out.data(), 8, out.size(), stdout);
    return 0;
}
