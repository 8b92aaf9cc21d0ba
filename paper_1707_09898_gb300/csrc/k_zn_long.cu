#include "k_zn.cuh"

namespace tmk {

int launch_zn_long(int L, const ZArgs& a, cudaStream_t s) {
  switch (L) {
    case 288: return run_length<288>(a, s);
    case 384: return run_length<384>(a, s);
    case 512: return run_length<512>(a, s);
    case 576: return run_length<576>(a, s);
  }
  return -2;
}

}  // namespace tmk
