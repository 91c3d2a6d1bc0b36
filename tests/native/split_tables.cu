// Prints the difference weights of the split FP64 step as hex floats: for a blend,
// a boundary kind, two metrics and a time step given on the command line, every
// row of the four tables, and whether the centre weights of a diagonal merge.
// Host code only: it needs no GPU.
#include <cstdio>
#include <cstdlib>

#include "split_tables.h"

using namespace fdlbm;

int main(int argc, char **argv)
{
    if (argc < 8) return 1;
    const double beta = std::atof(argv[1]), h = std::atof(argv[4]), dt = std::atof(argv[5]);
    const bool wx = std::atoi(argv[2]) != 0, wy = std::atoi(argv[3]) != 0;
    const int nx = std::atoi(argv[6]);
    std::vector<double> mx, my;
    for (int k = 7; k < argc; ++k) ((int)mx.size() < nx ? mx : my).push_back(std::atof(argv[k]));
    const std::vector<double> t = make_split_tables(mx, my, wx, wy, beta, h, dt);
    std::printf("merge %d\n", split_centres_merge(t, (int)mx.size(), (int)my.size()) ? 1 : 0);
    for (size_t k = 0; k < t.size(); k += 4) std::printf("%a %a %a %a\n", t[k], t[k + 1], t[k + 2], t[k + 3]);
    return 0;
}
