// Test harness: wall coefficients rounded to the compute type (clbm::round_heat)
// with the collision's share of the heat (clbm::heat_share), compiled for the
// host.  Not part of the library; built by tests/test_wall_balance.py.
#include "../paper_1801_04577_gb300/csrc/clbm_internal.h"
#include "../paper_1801_04577_gb300/csrc/clbm_walls.h"

// o[0..3], o[4]: FP64 weights and share; o[5..8], o[9]: the FP32 ones
extern "C" void host_round_heat(double b1, double b2, double b3, double ne, double q, int have2, int have3, double l2,
                                double cT2, double* o) {
  clbm::DevCoef c{};
  c.s_nu = c.s_b = c.s3 = c.s4 = c.l1 = c.rho0 = 1.0;
  c.l2 = l2;
  c.cT2 = cT2;
  clbm::fill_f32(c);
  double k[4], d[4];
  float f[4];
  clbm::link_heat(b1, b2, b3, ne, q, have2 != 0, have3 != 0, 0.5, 1e-5, cT2, k);
  clbm::round_heat(k, b2, clbm::heat_share(c.kd, cT2), d);
  clbm::round_heat(k, b2, clbm::heat_share(c.kf, cT2), f);
  for (int i = 0; i < 4; ++i) {
    o[i] = d[i];
    o[5 + i] = f[i];
  }
  o[4] = clbm::heat_share(c.kd, cT2);
  o[9] = clbm::heat_share(c.kf, cT2);
}
