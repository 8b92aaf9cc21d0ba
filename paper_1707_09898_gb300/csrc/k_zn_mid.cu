#include "k_zn.cuh"

namespace tmk {

int launch_zn_mid(int L, const ZArgs& a, cudaStream_t s) {
  switch (L) {
    case 128: return run_length<128>(a, s);
    case 144: return run_length<144>(a, s);
    case 192: return run_length<192>(a, s);
    case 256: return run_length<256>(a, s);
  }
  return -2;
}

}  // namespace tmk
