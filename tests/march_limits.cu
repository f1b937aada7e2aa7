// Calls the split launcher with bare sizes (no memory behind them), for the test of
// the limits of the march along theta against the stand-in runtime.
#include "../paper_2302_13907_gb300/csrc/cwell_internal.cuh"

extern "C" int launch_with(int storage, int code, int nth, int NR, int nr, int NZ, int NZp, int pml_z, int n_mat) {
  cwell::KParams p{};
  p.nth = nth, p.NR = NR, p.NZ = NZ, p.NZp = NZp, p.nr = nr, p.pml_r = NR - nr, p.pml_z = pml_z;
  p.plane = (long long)NR * NZp;
  p.i_hi = NR;
  p.src_i = -1;
  p.n_mat = n_mat;
  return (int)cwell::launch_hoist(storage, code, p, nullptr, nullptr, 3);
}
