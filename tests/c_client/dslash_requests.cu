// Requests to the internal hemi-Dslash launcher that no kernel it would choose
// can carry out: each must come back as HMC_EINVAL before anything is launched
// (the context below has no GPU behind it, the pointers belong to nothing).
// One line per request: name, status, message.
#include <cstdio>

#include "hmc_host.h"

using namespace hmc;

struct Request {
  const char *name;
  int prec, fmt, n_rhs, variant;
  int lattice;  // extent in each direction
  void (*set)(DslashArgs &);
};

static double num[4];
static int flag;
static char field[64];

static void cg_r(DslashArgs &a) {
  a.out = nullptr;
  a.cg_r = field;
  a.cg_alpha = num;
}
static void cg_x(DslashArgs &a) {
  cg_r(a);
  a.cg_x = field;
  a.cg_p = field;
}
static void red(DslashArgs &a) {
  a.red_src = num;
  a.red_n = 1;
  a.red_dst = num + 1;
  a.red_rr = num + 2;
  a.red_alpha = num + 3;
  a.red_flag = &flag;
}
static unsigned int counter;
static void red_total(DslashArgs &a) {
  red(a);
  a.partials = num;
  a.total = num + 3;
  a.counter = &counter;
}
static void partials(DslashArgs &a) { a.partials = num; }

int main() {
  const Request requests[] = {
      // emulated FP64: no reductions, no fused update, in none of its kernels
      {"f64e_18_large_cg_r", HMC_F64E, 18, 1, -1, 24, cg_r},
      {"f64e_18_large_red", HMC_F64E, 18, 1, -1, 24, red},
      {"f64e_18_large_partials", HMC_F64E, 18, 1, -1, 24, partials},
      {"f64e_18_small_cg_r", HMC_F64E, 18, 1, -1, 8, cg_r},
      {"f64e_12_small_cg_r", HMC_F64E, 12, 1, -1, 8, cg_r},
      {"f64e_18_variant0_red", HMC_F64E, 18, 1, 0, 8, red},
      {"f64e_12_red", HMC_F64E, 12, 1, 0, 8, red},
      // the fused batched update is the multi-right-hand-side kernel's
      {"f32_one_rhs_cg_x", HMC_F32, 12, 1, 0, 8, cg_x},
      {"f32_one_rhs_small_cg_x", HMC_F32, 12, 1, -1, 8, cg_x},
      {"f64_one_rhs_cg_x", HMC_F64, 18, 1, 2, 8, cg_x},
      {"f32_rhs2_site_cg_x", HMC_F32, 12, 2, 0, 8, cg_x},
      // which has neither an extra reduction block nor the single update
      {"f16_rhs2_red", HMC_F16, 12, 2, -1, 8, red},
      {"f32_rhs2_mr_red", HMC_F32, 12, 2, 4, 8, red},
      {"f32_rhs2_mr_cg_r", HMC_F32, 12, 2, 4, 8, cg_r},
      // totals count the launch's blocks, which the reduction block is one of
      {"f32_red_total", HMC_F32, 12, 1, 0, 8, red_total},
      {"f64_small_red_total", HMC_F64, 18, 1, -1, 8, red_total},
  };
  for (const Request &q : requests) {
    hmc_ctx ctx;
    ctx.sm_count = 152;
    ctx.ds_variant = q.variant;
    const hmc_lattice lat = {{q.lattice, q.lattice, q.lattice, q.lattice}};
    DslashArgs a{};
    a.g = make_geo(lat);
    a.n_rhs = q.n_rhs;
    a.gauge = field;
    a.in = field;
    a.out = field;
    a.cb = 1.0;
    q.set(a);
    const hmc_gauge U = {field, q.prec, q.fmt};
    const int st = dslash(&ctx, a, U, q.prec, 0, nullptr);
    printf("%s %d %s\n", q.name, st, ctx.err.c_str());
  }
  return 0;
}
