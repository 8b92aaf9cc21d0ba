// The lengths of the z pass (k_zn.cuh) up to 96, and the choice of the unit that holds a length:
// three units that compile at the same time.
#include "k_zn.cuh"

namespace tmk {

namespace {

// index of the unit vector v, or -1
int axis_of(const float v[3]) {
  for (int c = 0; c < 3; c++)
    if (v[c] == 1.0f && v[(c + 1) % 3] == 0.0f && v[(c + 2) % 3] == 0.0f) return c;
  return -1;
}

}  // namespace

int launch_zn(int L, const ZArgs& in, cudaStream_t s) {
  ZArgs a = in;
  if (2 * a.n_in > L || 2 * a.n_out > L) return -2;
  for (int i = 0; i < a.nin; i++) a.axis[i] = axis_of(a.u[i]);
  for (int o = 0; o < a.nout; o++) a.oaxis[o] = axis_of(a.v[o]);
  for (int i = 0; a.nin > 1 && i < a.nin; i++)  // several inputs: components, three of them in order
    if (a.axis[i] < 0 || (a.nin == 3 && a.axis[i] != i)) return -2;
  for (int o = 0; a.nout > 1 && o < a.nout; o++)
    if (a.oaxis[o] < 0 || (a.nout == 3 && a.oaxis[o] != o)) return -2;
  if (a.nin > 1 && a.nout > 1 && (a.nin != 3 || a.nout != 3)) return -2;
  switch (L) {
#define TM_CASE(LL) \
  case LL:          \
    return run_length<LL>(a, s);
    TM_CASE(8) TM_CASE(12) TM_CASE(16) TM_CASE(18) TM_CASE(24) TM_CASE(32) TM_CASE(36) TM_CASE(48) TM_CASE(64)
    TM_CASE(72) TM_CASE(96)
#undef TM_CASE
  }
  const int r = launch_zn_mid(L, a, s);
  return r != -2 ? r : launch_zn_long(L, a, s);
}

}  // namespace tmk
