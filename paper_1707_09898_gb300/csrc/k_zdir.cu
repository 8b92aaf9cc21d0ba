// Direct z convolution in (kx, ky, z) space for targets that occupy a few planes.
//
// After the x and y transforms the convolution of Sec. "Discretization",
// Eq. (convolution) is, per column (kx, ky), a 1-D convolution along z with the
// tensor transformed along x and y only:
//     out_o(z) = sum_{z'} sum_i s_oi(z - z') in_i(z'),   s_oi = v_o^T N~(z - z') u_i.
// When the outputs (forward field on the target planes) or the inputs (adjoint
// source on the target planes) occupy at most a few planes, summing this
// directly costs a few multiply-adds per complex value streamed from memory,
// instead of a forward and an inverse z FFT. The result is the same
// convolution (no approximation). Columns are read with consecutive threads on
// consecutive kx.
//
// Bytes bound it on large grids (inputs, outputs and the tensor rows each once), latency on
// small ones. A block takes 32 kx of the columns ky and Ly - ky, which read the same tensor
// rows, and splits z over its eight warps. Each z needs one new tensor row whatever the
// number of planes: the offset of plane p at z + 1 is that of plane p - 1 at z, so the rows
// move through registers. The tensor enters as t = N~ w with the vector of the side that has
// one component (M0, or a unit vector), and its row is formed once for every plane, input
// and output. Before, eight columns per block with no split along z and each factor from its
// own masked loads: 26 us on the 39 x 39 x 41 grid with two planes (24 blocks), now 4; at 256^3, both
// directions, one plane with three components 857 -> 247 us, varying M0 500 -> 453; four
// planes 1540 -> 314 (one component), varying M0 7703 -> 778.
#include "fft.cuh"
#include "internal.h"

namespace tmk {

namespace {

// One tensor row at one offset: the six components, signs of the odd ones (xz, yz in z; xy,
// yz in y) and the factor -i of xz and yz included by the functions below.
struct Row {
  float n[6];
};

// t = N~ w = re - i im for w on the column with y sign sy
struct Vec {
  float re[3], im[3];
};
__device__ __forceinline__ Vec apply_w(const Row& r, const float w[3], float sy) {
  const float xy = sy * r.n[3], yz = sy * r.n[5];
  Vec t;
  t.re[0] = r.n[0] * w[0] + xy * w[1];
  t.re[1] = xy * w[0] + r.n[1] * w[1];
  t.re[2] = r.n[2] * w[2];
  t.im[0] = r.n[4] * w[2];
  t.im[1] = yz * w[2];
  t.im[2] = r.n[4] * w[0] + yz * w[1];
  return t;
}
// acc += (o . t) x
__device__ __forceinline__ void add_dot(cx<float>& acc, const Vec& t, const float o[3], cx<float> x) {
  const float re = o[0] * t.re[0] + o[1] * t.re[1] + o[2] * t.re[2];
  const float im = o[0] * t.im[0] + o[1] * t.im[1] + o[2] * t.im[2];
  acc.x = __fmaf_rn(im, x.y, __fmaf_rn(re, x.x, acc.x));
  acc.y = __fmaf_rn(-im, x.x, __fmaf_rn(re, x.y, acc.y));
}
// acc += N~ x for the three components
__device__ __forceinline__ void add_full(cx<float>* acc, const Row& r, float sy, const cx<float>* x) {
  const float xy = sy * r.n[3], yz = sy * r.n[5], xz = r.n[4];
  acc[0] = acc[0] + mk(r.n[0] * x[0].x + xy * x[1].x + xz * x[2].y, r.n[0] * x[0].y + xy * x[1].y - xz * x[2].x);
  acc[1] = acc[1] + mk(xy * x[0].x + r.n[1] * x[1].x + yz * x[2].y, xy * x[0].y + r.n[1] * x[1].y - yz * x[2].x);
  acc[2] = acc[2] + mk(xz * x[0].y + yz * x[1].y + r.n[2] * x[2].x, r.n[2] * x[2].y - xz * x[0].x - yz * x[1].x);
}

enum { ONE_IN = 0, ONE_OUT = 1, FULL = 2 };  // one input; several inputs, one output; three and three

constexpr int ZP = 8;  // z parts per block, one warp each

// Blocks per SM: more warps against more registers, hence loads, per thread. One plane at
// 256^3, both directions: three and three 4 blocks 452 us, 5 470, 6 494, no bound 543; one to
// one with tilted M0 no bound 119, 6 blocks 103. The variants with three inputs or outputs spill
// (72 to 212 bytes with one plane at 6 blocks, 28 to 120 with two at 4); fewer blocks were better
// on middle grids and worse on large ones. Evaluation with tilted M0 and three weights, us, one
// plane with 6, 5 and 4 blocks: 128^3 104, 99, 113, 256^3 568, 578, 569; two planes with 4, 3 and 2:
// 128^3 126, 117, 132, 256^3 619, 638, 698 (before this kernel 512 and 1305, 709 and 3000).
__host__ __device__ constexpr int blocks_per_sm(int np, int mode) {
  return np == 1 ? (mode == FULL ? 4 : 6) : np == 2 ? 4 : np == 4 ? 2 : 1;
}

// NP: planes on the short side (at most). COLS: columns per thread (ky, Ly - ky).
// NK: inputs (ONE_OUT), outputs (ONE_IN) held: 1 or 3. SHARED: few inputs, some of whose planes are
// also output planes (a target inside the design). Inputs and outputs share a slot, and such a
// plane belongs to one warp's z range while every warp reads it, so no warp may store before all
// have their inputs. (Few outputs are stored behind a barrier anyway.) An instantiation of its own:
// in one kernel for both, the barrier made the compiler order the other direction's loads
// differently, and one plane of three and three took 100 us both ways at 128^3 (88 so), 467 at
// 256^3 (449).
template <int NP, int COLS, int MODE, int NK, bool SHARED>
__global__ void __launch_bounds__(32 * ZP, blocks_per_sm(NP, MODE)) k_zdir(const __grid_constant__ ZDirArgs a) {
  constexpr int NI = MODE == ONE_IN ? 1 : NK, NO = MODE == ONE_OUT ? 1 : NK;
  constexpr int UNR = MODE == FULL ? 1 : 2;  // z per round of loads; the others measured slower
  __shared__ cx<float> red[ZP][NP][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  const bool valid = blockIdx.x * 32 + lane < a.P;
  const int kx = SHARED ? min(blockIdx.x * 32 + lane, a.P - 1) : blockIdx.x * 32 + lane;  // SHARED: lanes past P load it
  // zcol holds ky = 0, then the pairs (ky, Ly - ky), then Ly / 2
  const int c0 = COLS == 1 ? blockIdx.y : (blockIdx.y == 0 ? 0 : 2 * blockIdx.y - 1);
  const int nc = COLS == 1 || blockIdx.y == 0 || c0 == a.Ly - 1 ? 1 : 2;
  long long colo[COLS];
  float sy[COLS];
  int kyf = 0;
#pragma unroll
  for (int c = 0; c < COLS; c++) {
    const int2 col = a.zcol[c0 + (c < nc ? c : 0)];
    const bool lo = col.y <= a.Ly / 2;
    kyf = lo ? col.y : a.Ly - col.y;
    sy[c] = lo ? 1.0f : -1.0f;
    colo[c] = (long long)col.x * a.P + kx;
  }
  const cx<float>* buf = reinterpret_cast<const cx<float>*>(a.buf);
  cx<float>* obuf = reinterpret_cast<cx<float>*>(a.buf);
  // A component that no product uses is read from the place of one that some product uses (its
  // weights are zero): a test per load kept the loads of successive rows apart (varying M0
  // at 256^3, one plane, both directions: 726 us with tests, 543 without).
  const float* T = a.Tz + kyf * (long long)a.P + kx;
  unsigned comp[6];
#pragma unroll
  for (int c = 0; c < 6; c++) comp[c] = (unsigned)((a.need & (1 << c) ? c : a.need ? __ffs(a.need) - 1 : 0) * a.Tc);
  auto row = [&](int dz) {  // offsets past the stored ones belong to planes that are not wanted
    Row r;
    const unsigned at = (unsigned)(min(abs(dz), a.ndz - 1) * a.Tdz);
#pragma unroll
    for (int c = 0; c < 6; c++) r.n[c] = T[comp[c] + at];
    if (dz < 0) {
      r.n[4] = -r.n[4];
      r.n[5] = -r.n[5];
    }
    return r;
  };
  // acc[o] += the contribution of the inputs x through row r
  auto add = [&](cx<float>* acc, const Row& r, float s, const cx<float>* x) {
    if constexpr (MODE == FULL) {
      add_full(acc, r, s, x);
    } else {
      const Vec t = apply_w(r, MODE == ONE_IN ? a.u[0] : a.v[0], s);
#pragma unroll
      for (int k = 0; k < NK; k++)
        add_dot(acc[MODE == ONE_IN ? k : 0], t, MODE == ONE_IN ? a.v[k] : a.u[k], x[MODE == ONE_IN ? 0 : k]);
    }
  };
  pdl_wait();  // inputs and outputs belong to earlier kernels
  if (a.nzout <= a.nzin) {  // few outputs: stream the inputs onto NP x NO sums
    cx<float> acc[COLS][NP][NO];
#pragma unroll
    for (int c = 0; c < COLS; c++)
#pragma unroll
      for (int p = 0; p < NP; p++)
#pragma unroll
        for (int o = 0; o < NO; o++) acc[c][p][o] = zero<float>();
    const int per = (a.nzin + ZP - 1) / ZP;
    const int z0 = a.zin0 + part * per, z1 = min(z0 + per, a.zin0 + a.nzin);
    if (valid && z0 < z1) {
      Row r[NP];
#pragma unroll
      for (int p = 0; p < NP - 1; p++) r[p] = row(a.zout0 + p + 1 - z0);  // shifted into place below
#pragma unroll UNR
      for (int z = z0; z < z1; z++) {
#pragma unroll
        for (int p = NP - 1; p > 0; p--) r[p] = r[p - 1];
        r[0] = row(a.zout0 - z);
#pragma unroll
        for (int c = 0; c < COLS; c++) {
          cx<float> x[NI];
#pragma unroll
          for (int i = 0; i < NI; i++)
            x[i] = NI == 1 || i < a.nin ? buf[a.in_slot[i] * a.cstride + z * a.zstride + colo[c]] : zero<float>();
#pragma unroll
          for (int p = 0; p < NP; p++) add(acc[c][p], r[p], sy[c], x);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < COLS; c++)
#pragma unroll
      for (int o = 0; o < NO; o++) {  // the parts in order
        if (c < nc && o < a.nout) {   // (the same for the whole block)
#pragma unroll
          for (int p = 0; p < NP; p++) red[part][p][lane] = acc[c][p][o];
          __syncthreads();
          if (part < NP && part < a.nzout && valid) {
            cx<float> s = red[0][part][lane];
#pragma unroll
            for (int q = 1; q < ZP; q++) s = s + red[q][part][lane];
            obuf[a.out_slot[o] * a.cstride + (a.zout0 + part) * a.zstride + colo[c]] = s;
          }
          __syncthreads();
        }
      }
  } else {  // few inputs: keep them, stream the outputs
    if (!SHARED && !valid) return;
    cx<float> x[COLS][NP][NI];
#pragma unroll
    for (int c = 0; c < COLS; c++)
#pragma unroll
      for (int p = 0; p < NP; p++)
#pragma unroll
        for (int i = 0; i < NI; i++)
          x[c][p][i] = p < a.nzin && (NI == 1 || i < a.nin)
                           ? buf[a.in_slot[i] * a.cstride + (a.zin0 + p) * a.zstride + colo[c]]
                           : zero<float>();
    const int per = (a.nzout + ZP - 1) / ZP;
    const int z0 = a.zout0 + part * per, z1 = min(z0 + per, a.zout0 + a.nzout);
    if (SHARED) __syncthreads();
    if (!valid || z0 >= z1) return;
    Row r[NP];
#pragma unroll
    for (int p = 0; p < NP - 1; p++) r[p] = row(z0 - 1 - a.zin0 - p);  // shifted into place below
#pragma unroll UNR
    for (int z = z0; z < z1; z++) {
#pragma unroll
      for (int p = NP - 1; p > 0; p--) r[p] = r[p - 1];
      r[0] = row(z - a.zin0);
#pragma unroll
      for (int c = 0; c < COLS; c++) {
        cx<float> acc[NO];
#pragma unroll
        for (int o = 0; o < NO; o++) acc[o] = zero<float>();
#pragma unroll
        for (int p = 0; p < NP; p++) add(acc, r[p], sy[c], x[c][p]);
        if (c < nc) {
#pragma unroll
          for (int o = 0; o < NO; o++)
            if (NO == 1 || o < a.nout) obuf[a.out_slot[o] * a.cstride + z * a.zstride + colo[c]] = acc[o];
        }
      }
    }
  }
}

template <int NP, int COLS, int MODE, int NK>
int run_zdir(const ZDirArgs& a, cudaStream_t s) {
  const dim3 grid((a.P + 31) / 32, COLS == 1 ? a.Ly : a.Ly / 2 + 1);
  const bool shared = a.nzout > a.nzin && a.zin0 < a.zout0 + a.nzout && a.zout0 < a.zin0 + a.nzin;
  auto kernel = shared ? k_zdir<NP, COLS, MODE, NK, true> : k_zdir<NP, COLS, MODE, NK, false>;
  return launch_k(kernel, grid, dim3(32 * ZP), 0, s, a.pdl != 0, a) == cudaSuccess ? 0 : -1;
}

template <int NP, int COLS>
int run_planes(const ZDirArgs& a, cudaStream_t s) {
  if (a.nin == 1) return a.nout == 1 ? run_zdir<NP, COLS, ONE_IN, 1>(a, s) : run_zdir<NP, COLS, ONE_IN, 3>(a, s);
  if (a.nout == 1) return run_zdir<NP, COLS, ONE_OUT, 3>(a, s);
  return run_zdir<NP, COLS, FULL, 3>(a, s);
}

}  // namespace

int launch_zdir(const ZDirArgs& a, cudaStream_t s) {
  const int small = a.nzout <= a.nzin ? a.nzout : a.nzin;
  if (small < 0 || small > kDirectPlanesMax) return -2;
  if (small == 0) return 0;
  if (a.nin > 1 && a.nout > 1) {  // the components go in and out: u_i = e_i, v_o = e_o
    if (a.nin != 3 || a.nout != 3) return -2;
    for (int k = 0; k < 3; k++)
      for (int c = 0; c < 3; c++)
        if (a.u[k][c] != (k == c ? 1.0f : 0.0f) || a.v[k][c] != (k == c ? 1.0f : 0.0f)) return -2;
  }
  if (small == 1) return run_planes<1, 2>(a, s);
  if (small == 2) return run_planes<2, 2>(a, s);
  if (small <= 4) return run_planes<4, 2>(a, s);
  return run_planes<kDirectPlanesMax, 1>(a, s);  // two columns would not fit in registers
}

}  // namespace tmk
