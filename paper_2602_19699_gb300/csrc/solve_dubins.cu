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
// however many lanes it serves, and 32 lanes share a knot's entries where 8
// take columns of them.  Measured (3 iterations,
// ms at 8 / 32 lanes, both with dense products): B = 64 3.90 / 2.97, 608 3.94 /
// 3.14, 1216 3.96 / 4.97, 2048 4.15 / 9.77.  Beyond 4 instances an SM the pipes are shared and 8
// lanes, four instances an instruction, win.  The sizes give the same bits.
static int dubins_lanes(int prec, int B, int sms) { return prec == PREC_FP64 && B <= 4 * sms ? 32 : 8; }

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
