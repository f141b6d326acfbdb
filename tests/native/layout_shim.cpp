// Test-only C entry points over the library's layout rules (compiled by tests/test_layout_host.py with the
// host compiler; not part of the library).
#include "../../paper_1908_04443_gb300/csrc/layout.h"

extern "C" {

int layout_marches(int nx, int ny, int nz) { return lbmwet::ztma_marches(nx, ny, nz); }
int layout_pitch(int dim, int zmarch, int nx, int ny) { return lbmwet::row_pitch(dim, zmarch != 0, nx, ny); }

}  // extern "C"
