// Prints fused_split's rows, columns and parts for one leaf of the row count and
// the column count of each pair of numbers on the command line.
#include <cstdio>
#include <cstdlib>

#include "../paper_2312_00005_gb300/csrc/bem_plan.hpp"

int main(int argc, char **argv)
{
    for (int i = 1; i + 1 < argc; i += 2) {
        const bem::FusedSplit f = bem::fused_split({std::atoll(argv[i])}, std::atoll(argv[i + 1]));
        std::printf("%d %d %d\n", f.rows, f.cols, f.parts);
    }
    return 0;
}
