// Jerk-controlled Dubins car: parameter parsing and solver instantiation.
#include <cmath>

#include "launch.cuh"
#include "sys_dubins.cuh"

namespace to {

static int parse_dubins(const double* p, size_t np, std::vector<unsigned char>& blob64,
                        std::vector<unsigned char>& blob32, std::string& err) {
  if (np < 5) { err = "dubins params: need at least 5 values"; return -1; }
  DubinsParams<double> P{};
  P.dt = p[0]; P.wu = p[1]; P.bamp = p[2]; P.bsig = p[3];
  P.nb = (int)p[4];
  if (P.nb < 0 || P.nb > 8 || np < (size_t)(8 + 2 * P.nb)) { err = "dubins params: bad bump count"; return -1; }
  if (!(P.bsig > 0)) { err = "dubins params: bump sigma must be > 0"; return -1; }
  for (int b = 0; b < P.nb; ++b) { P.bc[b][0] = p[5 + 2 * b]; P.bc[b][1] = p[6 + 2 * b]; }
  P.wpT = p[5 + 2 * P.nb];
  P.wvT = p[6 + 2 * P.nb];
  P.waT = p[7 + 2 * P.nb];
  P.derive();
  to_blobs<DubinsParams>(P, blob64, blob32);
  return 0;
}

typedef Dispatch<SysDubins, kDepth1, 1, 8, 16, 32> DBDispatch;

// Float64 batches that leave a scheduler per instance take a whole warp: a
// float64 warp instruction holds its scheduler's FP64 pipe for 64 cycles
// however many lanes it serves, and 32 lanes share a knot's entries and the
// running costs where 8 take columns of them.  Measured (152 SMs, 3 iterations,
// ms at 8 / 16 / 32 lanes, 64-thread CTAs): B = 1 3.03 / 2.90 / 1.94, 64 2.92 /
// 2.79 / 1.96, 608 2.96 / 2.83 / 2.05, 609 2.98 / 2.90 / 2.51, 912 2.98 / 3.01 /
// 2.56, 1064 2.98 / 3.01 / 3.20, 1217 3.07 / 3.77 / 5.07, 2048 3.18 / 5.01 / 6.32.
// The line is where every instance's warp has a scheduler of its own; 32 lanes
// lead by less up to 6 instances an SM, which the rule leaves unused, and lose
// beyond.  The sizes give the same bits.
static int dubins_lanes(int prec, int B, int sms, int, int) { return prec == PREC_FP64 && B <= 4 * sms ? 32 : 8; }

static SysOps make_ops() {
  SysOps o{};
  o.sys = 5;
  fill_layout<SysDubins>(o);
  o.n_groups = 4;
  o.groups[0] = 8; o.groups[1] = 16; o.groups[2] = 32; o.groups[3] = 1;   // 1: one thread per instance
  o.default_G = 8;
  o.default_gpb[0] = 8; o.default_gpb[1] = 8;
  o.lanes = dubins_lanes;
  o.accepts_actor = false;
  o.parse = parse_dubins;
  o.max_depth = 1;
  o.launch = DepthOne<DBDispatch>::launch;
  o.occupancy = DepthOne<DBDispatch>::occupancy;
  o.knot_costs = knot_costs_one<SysDubins>;
  return o;
}

const SysOps& dubins_ops() {
  static SysOps o = make_ops();
  return o;
}

}  // namespace to
