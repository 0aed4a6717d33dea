// Host rules of the launches for tests/test_launch_rules.py (nothing here runs on a device).
#include "mhd_launch.h"

extern "C" unsigned interp_grid_of(int nlist, int Zp, int grid_y) { return mhd::interp_grid(nlist, Zp, grid_y); }
