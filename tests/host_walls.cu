// Test harness: the wall-link coefficients of the step kernels (clbm::link_heat,
// clbm::link_bounce) compiled for the host.  Not part of the library; built by
// tests/test_walls_host.py.
#include "../paper_1801_04577_gb300/csrc/clbm_walls.h"

extern "C" void host_link_heat(double b1, double b2, double b3, double ne, double q, int have2, int have3, double T0,
                               double hQ, double cT2, double* k) {
  double o[4];
  clbm::link_heat(b1, b2, b3, ne, q, have2 != 0, have3 != 0, T0, hQ, cT2, o);
  for (int i = 0; i < 4; ++i) k[i] = o[i];
}

extern "C" void host_link_bounce(double q, int have2, double* k) {
  double o[3];
  clbm::link_bounce(q, have2 != 0, o);
  for (int i = 0; i < 3; ++i) k[i] = o[i];
}
