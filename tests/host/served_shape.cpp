// Prints 1 if a served batch of argv[2] histories takes a third of the GPU beside the
// running batches argv[3]... (its own among them); argv[1] histories fill the GPU.
#include <cstdio>
#include <cstdlib>

#include "ctd_host.h"

int main(int argc, char **argv)
{
    std::vector<double> running;
    for (int i = 3; i < argc; ++i) running.push_back(std::atof(argv[i]));
    std::printf("%d\n", ctd::host::shares_sms(std::atof(argv[2]), running, std::atof(argv[1])) ? 1 : 0);
    return 0;
}
