// Test harness: the host rules for wall links whose third node lies near the
// edge of a band or slab, and the places of the link tables' entries, compiled for the host.  Not part of the library; built
// by tests/test_bands_host.py.
#include "../paper_1801_04577_gb300/csrc/clbm_walls.h"

extern "C" int host_reads_third(int dir, double q, double b1) { return clbm::reads_third(dir, q, b1); }
extern "C" int host_third_row(int y, int dir) { return clbm::third_row(y, dir); }
extern "C" int host_band_holds_third(int y, int dir, int ny, int cl, int py) {
  return clbm::band_holds_third(y, dir, ny, cl, py != 0);
}
extern "C" int host_slab_holds_third(int y, int gy, int dir, int ny, int NY, int py) {
  return clbm::slab_holds_third(y, gy, dir, ny, NY, py != 0);
}
extern "C" long long host_heat_entry(int slot, int dir) { return (long long)clbm::heat_entry(slot, dir); }
extern "C" long long host_bounce_entry(int slot, int dir) { return clbm::bounce_entry(slot, dir); }
