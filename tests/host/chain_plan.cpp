// Prints the plan of a batched call's chains: streams, then each chain's batches per
// launch, then each stream's scratch voxels.  Arguments: batches, streams, voxels...
#include <cstdio>
#include <cstdlib>

#include "ctd_host.h"

namespace ctd {
namespace host {
int fail(int code, const char *, ...) { return code; }
}  // namespace host
}  // namespace ctd

int main(int argc, char **argv)
{
    std::vector<size_t> nvox;
    for (int i = 3; i < argc; ++i) nvox.push_back(std::strtoull(argv[i], nullptr, 10));
    const ctd::host::ChainPlan p =
        ctd::host::plan_chains(nvox, std::atoi(argv[1]), std::atoi(argv[2]), ctd::host::kBatchTallyBudget);
    std::printf("%d", p.lanes);
    for (int g : p.group) std::printf(" %d", g);
    for (size_t v : p.need) std::printf(" %zu", v);
    std::puts("");
    return 0;
}
