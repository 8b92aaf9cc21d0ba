// z pass of the stray-field convolution for any length and any magnetization: per column
// tile the forward z transforms of every input spectrum, the product with the tensor
// N^(k), and the inverse z transforms of every output, in one block.
//
// The product is written with the vectors u_i (inputs) and v_o (outputs) of
//     out_o = sum_i (v_o^T N^ u_i) in_i :
// one input: t = N^ u, out_o = (v_o . t) in; several inputs (u_i = e_axis): one output takes
// s = N^ v, out = sum_i s_axis(i) in_i, several take out_a = sum_b N^_ab in_b. Either way each
// of the six unique tensor components is read once per frequency and used for every input
// and output.
//
// What bounds it: instruction issue and the latency of the tensor loads (up to six 4-byte
// loads per complex value) at the 16 warps an SM holds; ncu at L = 256: 55% issue active, DRAM
// below 20%. The tiles of all inputs lie in shared memory together, so a block has two
// barriers whatever the number of inputs, and between the last forward and the first
// inverse stage each thread works on its own tile elements without any. The kernels it
// replaces ran a cluster of blocks that exchanged spectra through distributed shared memory,
// or one block per output, and formed every factor from its own masked loads, one element
// after the other. Measured per launch, before and now:
//   192 x 160 x 100, L = (512, 512, 256):  M0 along z     tilted M0      varying M0
//     one input, three outputs             572 -> 283 us  789 -> 333
//     three inputs, one output             1988 -> 310    2527 -> 353
//     three and three                                                    1950 -> 438
//   256^3, L = 512: three to one, M0 along z 1749 -> 799, tilted 3657 -> 896; three and three
//   2142 -> 1166.
//
// Zero padding and crop: inputs occupy z < L/2 and only outputs z < L/2 are kept, so the
// first stage is a half-input DFT and the last inverse stage forms the lower half only.
#pragma once
#include "fft.cuh"
#include "internal.h"

namespace tmk {

namespace {

// Two-stage plans of the z transforms, L = R0 R, R0 a power of two: the positions of the
// spectrum never leave the kernel, so the plan is free of the one that the y and x passes
// use, and with radices 6, 9, 12 and 18 beside the powers of two every length takes one
// exchange through shared memory (192 = 8 8 3 took two).
__host__ __device__ constexpr int zradix0(int L) {
  switch (L) {
    case 12: case 18: return 2;
    case 8: case 16: case 24: case 36: return 4;
    case 32: case 48: case 64: case 72: return 8;
    case 96: case 128: case 144: case 192: case 256: return 16;
    default: return 32;  // 288, 384, 512, 576
  }
}
template <int L>
struct ZPlan {
  static constexpr int R0 = zradix0(L), M0 = L / R0;  // first stage: positions j + q M0
  static constexpr int R = M0;                        // last stage: positions g R + q, k = g + q R0
  // 16 warps per SM (128 registers a thread): two blocks of 256 threads, or one of 512 at
  // L = 512, where three tiles fill the shared memory. Tiles of 8 lines would keep more
  // blocks there, but their 64-byte rows cost more than the barriers: L = 512, three to
  // three, 1.34 ms with two blocks of 8 lines and 1.17 with one of 16; L = 256, one to three,
  // 321 us with four blocks of 8 lines and 287 with two of 16.
  static constexpr int NT = L <= 144 ? 128 : L == 512 ? 512 : 256;
  static constexpr int MINB = L == 576 || L == 384 ? 1 : 512 / NT;
  static constexpr int NU0 = M0 * TB, NU = R0 * TB;
  // elements of the product whose tensor components are in flight together
  static constexpr int CH = R % 4 == 0 ? 4 : R % 3 == 0 ? 3 : 2;
  static_assert(R0 * R == L && R % CH == 0, "plan");
};

// N-point DFT of inputs 0 .. N/2 - 1 (the rest zero): X[2m] = DFT(x)[m], X[2m+1] = DFT(x W^n)[m]
template <int N, bool INV>
__device__ __forceinline__ void dft_half_input(cx<float>* v) {
  cx<float> a[N / 2], b[N / 2];
#pragma unroll
  for (int n = 0; n < N / 2; n++) {
    a[n] = v[n];
    b[n] = tw32<float, INV>(v[n], n * (32 / N));
  }
  DftF<N / 2, INV>::run(a);
  DftF<N / 2, INV>::run(b);
#pragma unroll
  for (int m = 0; m < N / 2; m++) {
    v[2 * m] = a[m];
    v[2 * m + 1] = b[m];
  }
}

// cos(10 degrees m), m = 0 .. 9
__host__ __device__ constexpr double cos36_q(int m) {
  return m == 0 ? 1.0
       : m == 1 ? 0.984807753012208059367
       : m == 2 ? 0.939692620785908384054
       : m == 3 ? 0.866025403784438646764
       : m == 4 ? 0.766044443118978035202
       : m == 5 ? 0.642787609686539326323
       : m == 6 ? 0.5
       : m == 7 ? 0.342020143325668733044
       : m == 8 ? 0.173648177666930348852
                : 0.0;
}
__host__ __device__ constexpr double cos36(int m) {  // m in [0, 36)
  return m <= 9 ? cos36_q(m) : m <= 18 ? -cos36_q(18 - m) : m <= 27 ? -cos36_q(m - 18) : cos36_q(36 - m);
}
__host__ __device__ constexpr double sin36(int m) { return cos36((m + 27) % 36); }

// R-point DFT, R a power of two or 6, 9, 12, 18: three DFTs of R / 3 points over the inputs of
// equal index mod 3, their outputs times W_R^(r k), and a DFT of 3.
template <int R, bool INV>
__device__ __forceinline__ void dft_any(cx<float>* v) {
  if constexpr (R % 3 != 0) {
    DftF<R, INV>::run(v);
  } else if constexpr (R == 3) {
    Dft<float, 3, INV>::run(v);
  } else {
    constexpr int K = R / 3;
    cx<float> e[3][K];
#pragma unroll
    for (int n = 0; n < K; n++)
#pragma unroll
      for (int r = 0; r < 3; r++) e[r][n] = v[3 * n + r];
#pragma unroll
    for (int r = 0; r < 3; r++) dft_any<K, INV>(e[r]);
#pragma unroll
    for (int k = 0; k < K; k++) {
      cx<float> x[3] = {e[0][k], e[1][k], e[2][k]};
#pragma unroll
      for (int r = 1; r < 3; r++) {
        const int m = r * k * (36 / R) % 36;
        const cx<float> w = mk(float(cos36(m)), -float(sin36(m)));
        if (m != 0) x[r] = INV ? cmulc(x[r], w) : cmul(x[r], w);
      }
      Dft<float, 3, INV>::run(x);
#pragma unroll
      for (int j = 0; j < 3; j++) v[k + K * j] = x[j];
    }
  }
}

// Twiddles of stage 0 (unit j): tw[j (R0 + 2) + q] = W_L^(j q); the padding keeps two
// neighbouring units of a warp on different banks.
template <int L>
__host__ __device__ constexpr int ztw_size() {
  return ZPlan<L>::M0 * (ZPlan<L>::R0 + 2);
}

// The product's factors of one side of kz = L/2 (sz = 1 up to it, -1 above): N^ with the
// signs of the column is S N S, S = diag(1, sy, sz), N the folded tensor.
struct Signed {
  float m[3][3];  // S_a S_b w_b
};
__device__ __forceinline__ Signed signed_by(const float w[3], float sy, float sz) {
  const float S[3] = {1.0f, sy, sz};
  Signed r;
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) r.m[a][b] = S[a] * S[b] * w[b];
  return r;
}
// component a of S N S w
__device__ __forceinline__ float row_dot(const Signed& w, const float* n, int a) {
  if (a == 0) return n[0] * w.m[0][0] + n[3] * w.m[0][1] + n[4] * w.m[0][2];
  if (a == 1) return n[3] * w.m[1][0] + n[1] * w.m[1][1] + n[5] * w.m[1][2];
  return n[4] * w.m[2][0] + n[5] * w.m[2][1] + n[2] * w.m[2][2];
}

// NI inputs (2 or 3: exactly so many), NO outputs (1, or 3 for two or three). APART (NI = NO = 1):
// the grid's third dimension is the output.
template <int L, int NI, int NO, bool APART = false>
__global__ void __launch_bounds__(ZPlan<L>::NT, ZPlan<L>::MINB) k_zn(const __grid_constant__ ZArgs a) {
  using Z = ZPlan<L>;
  constexpr int R0 = Z::R0, M0 = Z::M0, R = Z::R, NT = Z::NT, CH = Z::CH, TW = R0 + 2;
  // stage-0 twiddles held in registers where several spectra use them
  constexpr bool KEEP = NI > 1 && R0 <= 16, KEEPO = NO > 1 && R0 <= 16;
  extern __shared__ __align__(16) unsigned char smem[];
  cx<float>* tw = reinterpret_cast<cx<float>*>(smem);
  cx<float>* tile = tw + ztw_size<L>();
  const int t = threadIdx.x;
  const cx<float>* gtw = reinterpret_cast<const cx<float>*>(a.tw);
  for (int k = t; k < M0 * R0; k += NT) tw[k / R0 * TW + k % R0] = gtw[(k / R0) * (k % R0)];
  const int chunk = blockIdx.x;
  const int2 col = a.zcol[blockIdx.y];  // (ky position, ky)
  const bool ylo = col.y <= a.Ly / 2;
  const int kyf = ylo ? col.y : a.Ly - col.y;
  const float sy = ylo ? 1.0f : -1.0f;
  const unsigned zs = (unsigned)a.zstride, colo = (unsigned)(col.x * a.P + chunk * TB);
  int ilo = 0, ihi = a.n_in, olo = 0, ohi = a.n_out;
  if (a.in_ext) {
    ilo = max(a.ext[0], 0);
    ihi = min(a.ext[1], a.n_in);
  }
  if (a.out_ext) {
    olo = max(a.ext[0], 0);
    ohi = min(a.ext[1], a.n_out);
  }
  const unsigned icnt = (unsigned)max(ihi - ilo, 0), ocnt = (unsigned)max(ohi - olo, 0);
  const int nout = NO == 1 ? 1 : a.nout, o0 = APART ? (int)blockIdx.z : 0;
  __syncthreads();  // twiddles
#pragma unroll
  for (int it = 0; it < (Z::NU0 + NT - 1) / NT; it++) {  // first stage: rows z = j + q M0 < L/2 in
    const int u = it * NT + t, line = u % TB, j = u / TB;
    if (Z::NU0 % NT == 0 || u < Z::NU0) {
      const unsigned off = colo + line + j * zs;
      cx<float> w[R0];
      if (KEEP) {
#pragma unroll
        for (int q = 1; q < R0; q++) w[q] = tw[j * TW + q];
      }
#pragma unroll
      for (int i = 0; i < NI; i++) {
        const cx<float>* in = reinterpret_cast<const cx<float>*>(a.buf) + a.in_slot[i] * a.cstride;
        cx<float>* tl = tile + i * (L * TB);
        cx<float> v[R0];
#pragma unroll
        for (int q = 0; q < R0 / 2; q++)
          v[q] = (unsigned)(j + q * M0 - ilo) < icnt ? in[off + q * M0 * zs] : zero<float>();
        dft_half_input<R0, false>(v);
        if (j != 0) {
#pragma unroll
          for (int q = 1; q < R0; q++) v[q] = cmul(v[q], KEEP ? w[q] : tw[j * TW + q]);
        }
#pragma unroll
        for (int q = 0; q < R0; q++) tl[(j + q * M0) * TB + line] = v[q];
      }
    }
  }
  __syncthreads();
  // last forward stage, product, first inverse stage: unit (line, g) owns positions g R + q
  // of every tile
#pragma unroll 1
  for (int it = 0; it < (Z::NU + NT - 1) / NT; it++) {
    const int u = it * NT + t, line = u % TB, g = u / TB;
    if (Z::NU % NT != 0 && u >= Z::NU) break;
    // frequencies kz = g + q R0, g < R0: up to L/2 for 2 q + 1 < R, above it for 2 q > R, and
    // either way for the one between
    auto below = [&](int q) { return 2 * q + 1 < R ? true : 2 * q > R ? false : g + q * R0 <= L / 2; };
    const unsigned tcol = (unsigned)(kyf * a.P + chunk * TB + line);
    // tensor components of CH elements, one test per component for all their loads: the
    // branch keeps the loads together (without it they were spread between their uses and
    // waited for one by one: 425 us instead of 359 for three inputs at L = 256)
    auto load_chunk = [&](int q0, float (*n)[6]) {
      unsigned off[CH];
#pragma unroll
      for (int e = 0; e < CH; e++) {
        const int kz = g + (q0 + e) * R0;
        off[e] = tcol + (unsigned)(below(q0 + e) ? kz : L - kz) * (unsigned)a.Tz;
      }
#pragma unroll
      for (int c = 0; c < 6; c++) {
        if (a.need & (1 << c)) {
          const float* tc = a.T + (long long)c * a.Tc;
#pragma unroll
          for (int e = 0; e < CH; e++) n[e][c] = tc[off[e]];
        } else {
#pragma unroll
          for (int e = 0; e < CH; e++) n[e][c] = 0.0f;
        }
      }
    };
    cx<float> v[R];
#pragma unroll
    for (int i = 0; i < NI; i++) {
      cx<float>* tl = tile + i * (L * TB);
#pragma unroll
      for (int q = 0; q < R; q++) v[q] = tl[(g * R + q) * TB + line];
      dft_any<R, false>(v);
      if (i < NI - 1) {
#pragma unroll
        for (int q = 0; q < R; q++) tl[(g * R + q) * TB + line] = v[q];
      }
    }
#pragma unroll
    for (int q0 = 0; q0 < R; q0 += CH) {
      float n[CH][6];
      load_chunk(q0, n);
#pragma unroll
      for (int e = 0; e < CH; e++) {
        const int q = q0 + e, at = (g * R + q) * TB + line;
        const float* ne = n[e];
        const float sz = below(q) ? 1.0f : -1.0f;
        if constexpr (NI == 1 && NO == 1) {
          const float f = ne[0] * a.coef[o0][0] + ne[1] * a.coef[o0][1] + ne[2] * a.coef[o0][2] +
                          ne[3] * (a.coef[o0][3] * sy) + ne[4] * (a.coef[o0][4] * sz) + ne[5] * (a.coef[o0][5] * (sy * sz));
          v[q] = scale(v[q], f);
        } else if constexpr (NI == 1) {  // outputs are components
          const Signed w = signed_by(a.u[0], sy, sz);
          const float tx = row_dot(w, ne, 0), ty = row_dot(w, ne, 1), tz = row_dot(w, ne, 2);
          const cx<float> x = v[q];
          if (nout == 3) {
            tile[at] = scale(x, tx);
            tile[L * TB + at] = scale(x, ty);
            v[q] = scale(x, tz);
          } else {
            tile[at] = scale(x, a.oaxis[0] == 0 ? tx : a.oaxis[0] == 1 ? ty : tz);
            v[q] = scale(x, a.oaxis[1] == 0 ? tx : a.oaxis[1] == 1 ? ty : tz);
          }
        } else if constexpr (NO == 1) {  // inputs are components
          const Signed w = signed_by(a.v[0], sy, sz);
          const float sx = row_dot(w, ne, 0), sY = row_dot(w, ne, 1), sZ = row_dot(w, ne, 2);
          if constexpr (NI == 3) {
            v[q] = scale(tile[at], sx) + scale(tile[L * TB + at], sY) + scale(v[q], sZ);
          } else {
            const float s0 = a.axis[0] == 0 ? sx : a.axis[0] == 1 ? sY : sZ;
            const float s1 = a.axis[1] == 0 ? sx : a.axis[1] == 1 ? sY : sZ;
            v[q] = scale(tile[at], s0) + scale(v[q], s1);
          }
        } else {  // inputs and outputs are the three components
          const float xy = ne[3] * sy, xz = ne[4] * sz, yz = ne[5] * (sy * sz);
          const cx<float> x = tile[at], y = tile[L * TB + at], z = v[q];
          tile[at] = scale(x, ne[0]) + scale(y, xy) + scale(z, xz);
          tile[L * TB + at] = scale(x, xy) + scale(y, ne[1]) + scale(z, yz);
          v[q] = scale(x, xz) + scale(y, yz) + scale(z, ne[2]);
        }
      }
    }
    dft_any<R, true>(v);
    {
      cx<float>* tl = tile + (nout - 1) * (L * TB);
#pragma unroll
      for (int q = 0; q < R; q++) tl[(g * R + q) * TB + line] = v[q];
    }
#pragma unroll
    for (int o = 0; o < NO - 1; o++) {
      if (o < nout - 1) {
        cx<float>* tl = tile + o * (L * TB);
#pragma unroll
        for (int q = 0; q < R; q++) v[q] = tl[(g * R + q) * TB + line];
        dft_any<R, true>(v);
#pragma unroll
        for (int q = 0; q < R; q++) tl[(g * R + q) * TB + line] = v[q];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < (Z::NU0 + NT - 1) / NT; it++) {  // last inverse stage: rows z = j + q M0 < L/2 out
    const int u = it * NT + t, line = u % TB, j = u / TB;
    if (Z::NU0 % NT == 0 || u < Z::NU0) {
      const unsigned off = colo + line + j * zs;
      cx<float> w[R0];
      if (KEEPO) {
#pragma unroll
        for (int q = 1; q < R0; q++) w[q] = tw[j * TW + q];
      }
#pragma unroll
      for (int o = 0; o < NO; o++) {
        if (o < nout) {
          cx<float>* out = reinterpret_cast<cx<float>*>(a.buf) + a.out_slot[o0 + o] * a.cstride;
          const cx<float>* tl = tile + o * (L * TB);
          cx<float> v[R0];
#pragma unroll
          for (int q = 0; q < R0; q++) v[q] = tl[(j + q * M0) * TB + line];
          if (j != 0) {
#pragma unroll
            for (int q = 1; q < R0; q++) v[q] = cmulc(v[q], KEEPO ? w[q] : tw[j * TW + q]);
          }
          dft_low_half<R0, true>(v);
#pragma unroll
          for (int q = 0; q < R0 / 2; q++)
            if ((unsigned)(j + q * M0 - olo) < ocnt) out[off + q * M0 * zs] = v[q];
        }
      }
    }
  }
}

template <int L, int NI, int NO, bool APART = false>
int run_zn(const ZArgs& a, cudaStream_t s) {
  using Z = ZPlan<L>;
  const int tiles = APART ? 1 : a.nin > a.nout ? a.nin : a.nout;
  const size_t sm = (size_t)(ztw_size<L>() + tiles * L * TB) * sizeof(float2);
  if (!allow_smem<k_zn<L, NI, NO, APART>>(sm)) return -1;
  k_zn<L, NI, NO, APART><<<dim3(a.P / TB, a.Ly, APART ? a.nout : 1), Z::NT, sm, s>>>(a);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

// One input with several outputs: on few column tiles the outputs' inverse transforms in turn are
// longer than the input's forward transform once more for each, on SMs that are idle otherwise.
// The line is two blocks per SM for all outputs, three for the lengths with a factor of 9, whose
// last stage is the longest. Field with M0 along z, outputs apart and together: 24 x 24 x 72 (96
// tiles, L = 144) 24.6 and 28.7 us, 24 x 32 x 72 (128) 26.6 and 28.7, 16 x 16 x 64 (64, L = 128)
// 20.8 and 22.6; 24 x 30 x 96 (128, L = 192) 26.7 and 24.6, 32 x 32 x 128 (192, L = 256) 32.8 and
// 30.7. At L = 576 three tiles fill the shared memory of an SM and one does half of it, so rounds
// of blocks count: 32 x 32 x 288 (192 tiles) 69.6 and 82.0, 48 x 48 x 288 (384) 159 and 180; 24 x
// 30 x 288 (128) 55.8 and 50.4, 72 x 72 x 288 (720, tilted M0) 282 and 275.
template <int L>
bool outputs_apart(const ZArgs& a) {
  if (a.nout == 1) return false;
  for (int o = 0; o < a.nout; o++)
    if (a.out_slot[o] == a.in_slot[0]) return false;  // another output's block may still read it
  const long long blocks = (long long)(a.P / TB) * a.Ly;
  if (L == 576) {
    const long long apart = (blocks * a.nout + 2 * a.nsm - 1) / (2 * a.nsm), together = (blocks + a.nsm - 1) / a.nsm;
    return 3 * apart <= (a.nout + 1) * together;
  }
  return blocks * a.nout <= (L % 9 == 0 ? 3LL : 2LL) * a.nsm;
}

template <int L>
int run_length(const ZArgs& a, cudaStream_t s) {
  if (a.nin == 1) {
    if constexpr (L == 512) return -2;  // k_z1m's
    else if (outputs_apart<L>(a)) return run_zn<L, 1, 1, true>(a, s);
    else return a.nout == 1 ? run_zn<L, 1, 1>(a, s) : run_zn<L, 1, 3>(a, s);
  }
  if (a.nin == 2) return run_zn<L, 2, 1>(a, s);
  return a.nout == 1 ? run_zn<L, 3, 1>(a, s) : run_zn<L, 3, 3>(a, s);
}

}  // namespace

}  // namespace tmk
