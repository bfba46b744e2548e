// The launch rule of the one-thread-per-direction hemi-Dslash, asked without a
// GPU for a device of 152 SMs.  Arguments: precision, link format and sites per
// parity, any number of times; one line per triple, 1 where the rule takes it.
#include <cstdio>
#include <cstdlib>

#include "hmc_host.h"

using namespace hmc;

int main(int argc, char **argv) {
  for (int k = 1; k + 2 < argc; k += 3) {
    hmc_ctx ctx;
    ctx.sm_count = 152;
    DslashArgs a{};
    a.n_rhs = 1;
    a.g.Vh = atoi(argv[k + 2]);
    printf("%d\n", dslash_split_rule(&ctx, a, atoi(argv[k]), atoi(argv[k + 1])) ? 1 : 0);
  }
  return 0;
}
