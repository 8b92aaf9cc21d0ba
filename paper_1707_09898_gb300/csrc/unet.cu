// Kernels of the learned warm start: a small 3-D U-Net that maps a target
// specification to an initial density for the optimizer. Not part of the paper
// (the paper's optimizer starts from rho = 1); the optimizer always refines the
// network's output, so the network only changes how many steps are needed.
//
// Layouts: activations channels-last [N][D][H][W][C], C a multiple of 16 (padded
// channels are zero); bfloat16 activations, float32 activation gradients.
// Weights: float32 master [27][Cin][Cout] (tap = (dz+1)*9 + (dy+1)*3 + (dx+1));
// bfloat16 copies Wf (forward) and Wb (backward data) packed in the operand layout of
// the tensor-core kernels (see pack_f / pack_b below).
// 3x3x3 convolutions (stride 1, zero padding 1), forward, data gradient and weight
// gradient, are implicit GEMMs on the fifth-generation tensor cores (tcgen05.mma,
// bfloat16 operands, float32 accumulators in tensor memory): k_conv_halo (rows of 8..64
// voxels: staged halo rows, a warp-specialized pipeline) and k_conv_dw_rows (their weight
// gradient, rows of 16..64), k_conv_dw_halo (rows of 8), k_conv_tc and k_conv_dw_tc (any grid:
// per-voxel gathers). The output gradient is rounded to bfloat16 where it is an operand.
#include <cuda_bf16.h>
#include <stdint.h>

#include <type_traits>

#include "../../include/topomag_net.h"
#include "device.cuh"
#include "unet_tc.cuh"

namespace {

using tmk::sm_count;

using bf16 = __nv_bfloat16;

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}


struct Vox {
  int n, z, y, x;
};
__device__ __forceinline__ Vox vox_of(long long v, int D, int H, int W) {
  Vox r;
  r.x = (int)(v % W);
  long long t = v / W;
  r.y = (int)(t % H);
  t /= H;
  r.z = (int)(t % D);
  r.n = (int)(t / D);
  return r;
}

// Packed bfloat16 weights for the tensor-core kernels: per (tap, 16-channel chunk kc of
// the reduced dimension) a block of N x 16 values in the MMA's B layout,
// [k-group (2)][N/8][8 rows][8 elements], rows = output channels of the GEMM.
// Forward (N = cout, reduced = ci), backward data (N = cin, reduced = co).
__host__ __device__ __forceinline__ long long pack_f(int tap, int ci, int co, int cin, int cout) {
  const int kc = ci >> 4, kk = ci & 15;
  return ((long long)tap * (cin >> 4) + kc) * (16LL * cout) + (kk >> 3) * 8LL * cout + (co >> 3) * 64 + (co & 7) * 8 +
         (kk & 7);
}
__host__ __device__ __forceinline__ long long pack_b(int tap, int ci, int co, int cin, int cout) {
  const int kc = co >> 4, kk = co & 15;
  return ((long long)tap * (cout >> 4) + kc) * (16LL * cin) + (kk >> 3) * 8LL * cin + (ci >> 3) * 64 + (ci & 7) * 8 +
         (kk & 7);
}

// Error word of the tensor-core kernels: bit 0 set when a bounded wait ran out (tmn_status).
__device__ unsigned g_net_status;

// Implicit-GEMM convolution on tcgen05: a block of 128 threads owns 128 consecutive voxels
// (the M = 128 rows of the accumulator, one tensor-memory lane per voxel) and all NO output
// channels (N). The reduction runs over (tap, 16-channel chunk) steps, K = 16 each: every
// thread gathers its voxel's 16 shifted input channels into the A tile (zero outside the
// grid), thread 0 copies the step's packed weight block into the B tile (bulk copy,
// mbarrier) and issues the MMA once the step's operands are in place; S stages of A and B
// keep the next steps' loads in flight while the tensor core works. The epilogue reads
// the accumulator from tensor memory (each warp its 32 lanes).
//   MODE 0 (forward):       out[v][co] = act(sum in[v + off][ci] W[tap][ci][co] + b[co]), bfloat16
//   MODE 1 (backward data): din[v][ci] (+)= sum dout[v - off][co] W[tap][ci][co], float32
// KC: channels of the gathered input (cin forward, cout backward).
constexpr int kTcStages = 4;
template <int NO>
__host__ __device__ constexpr unsigned tmem_cols() {
  return NO <= 32 ? 32u : (NO <= 64 ? 64u : 128u);
}
template <int NO>
constexpr size_t conv_tc_smem() {
  return (size_t)kTcStages * (128 * 32 + NO * 32) + (2 * kTcStages + 1) * 8 + 16;
}
template <int MODE, int NO>
__global__ void __launch_bounds__(128) k_conv_tc(const void* src, const bf16* Wc, const float* bias, void* dst,
                                                 int Nb, int D, int H, int W, int KC, int flag) {
  using namespace tmk;
  constexpr int S = kTcStages, AB = 128 * 32, BB = NO * 32;
  constexpr unsigned NCOLS = tmem_cols<NO>();
  constexpr unsigned IDESC = idesc_bf16(128, NO);
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* As = smem;                  // [S][2 k-groups][16 row groups][8][16 B]
  unsigned char* Bs = smem + S * AB;         // [S][2][NO/8][8][16 B]
  unsigned long long* tma_bar = reinterpret_cast<unsigned long long*>(Bs + S * BB);
  unsigned long long* mma_bar = tma_bar + S;
  unsigned* tslot = reinterpret_cast<unsigned*>(mma_bar + S);
  const int t = threadIdx.x, warp = t >> 5;
  if (t == 0) {
    for (int b = 0; b < S; b++) {
      mbar_init(tma_bar + b, 1);
      mbar_init(mma_bar + b, 1);
    }
    mbar_init_fence();
  }
  if (warp == 0) {
    tmem_alloc(tslot, NCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = *tslot;

  const long long nvox = (long long)Nb * D * H * W;
  const long long v = (long long)blockIdx.x * 128 + t;
  const bool valid = v < nvox;
  int vx = 0, vy = 0, vz = 0, vn = 0;
  if (valid) {
    long long q = v;
    vx = (int)(q % W);
    q /= W;
    vy = (int)(q % H);
    q /= H;
    vz = (int)(q % D);
    vn = (int)(q / D);
  }
  const int nk = KC >> 4, nsteps = 27 * nk;
  // bounded waits: the first one that runs out flags g_net_status and this thread skips its
  // later waits, so a broken launch ends in milliseconds instead of spinning on every step
  bool dead = false;
  auto wait = [&](unsigned long long* mb, unsigned parity) {
    if (!dead) dead = !mbar_wait_limit(mb, parity, 1 << 16, &g_net_status);
  };
  // this thread's row (m = t) in the A tile: row group t / 8, row t % 8
  const int arow = (t >> 3) * 128 + (t & 7) * 16;
  auto load_step = [&](int s, int b) {
    const int tap = s / nk, kc = s - tap * nk;
    int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    if (MODE == 1) {
      dz = -dz;
      dy = -dy;
      dx = -dx;
    }
    const int z = vz + dz, y = vy + dy, x = vx + dx;
    const bool ok = valid && z >= 0 && z < D && y >= 0 && y < H && x >= 0 && x < W;
    const long long u = ok ? (((long long)vn * D + z) * H + y) * W + x : 0;
    unsigned char* a = As + b * AB + arow;
    if constexpr (MODE == 0) {
      const bf16* p = reinterpret_cast<const bf16*>(src) + u * KC + kc * 16;
      cp_async16(a, p, ok ? 16u : 0u);             // channels 0..7: k-group 0
      cp_async16(a + 2048, p + 8, ok ? 16u : 0u);  // channels 8..15: k-group 1
    } else {
      uint4 lo = make_uint4(0u, 0u, 0u, 0u), hi = lo;
      if (ok) {
        const float4* p = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(src) + u * KC + kc * 16);
        const float4 f0 = p[0], f1 = p[1], f2 = p[2], f3 = p[3];
        lo = make_uint4(pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w));
        hi = make_uint4(pack2(f2.x, f2.y), pack2(f2.z, f2.w), pack2(f3.x, f3.y), pack2(f3.z, f3.w));
      }
      *reinterpret_cast<uint4*>(a) = lo;
      *reinterpret_cast<uint4*>(a + 2048) = hi;
    }
    if (t == 0) {
      mbar_expect_tx(tma_bar + b, BB);
      bulk_load(Bs + b * BB, Wc + ((long long)tap * nk + kc) * NO * 16, BB, tma_bar + b);
    }
  };
  for (int s = 0; s < S - 1; s++) {  // always S - 1 groups, so that the wait below counts right
    if (s < nsteps) load_step(s, s);
    cp_async_commit();
  }
  for (int s = 0; s < nsteps; s++) {
    const int b = s % S;
    const int sn = s + S - 1;  // its loads go into the buffer the MMA of step s - 1 read
    if (sn < nsteps) {
      const int bn = sn % S;
      if (s >= 1) wait(mma_bar + bn, ((s - 1) / S) & 1);
      load_step(sn, bn);
    }
    cp_async_commit();
    cp_async_wait<S - 1>();  // this thread's copies of step s have landed
    fence_proxy_async_smem();  // its A rows, written through the generic proxy, for the tensor core
    __syncthreads();
    if (t == 0) {
      wait(tma_bar + b, (s / S) & 1);  // the weight block
      tc_fence_after();
      const uint64_t ad = smem_desc(As + b * AB, 2048, 128);
      const uint64_t bd = smem_desc(Bs + b * BB, NO * 16, 128);
      tc_mma(taddr, ad, bd, IDESC, s > 0);
      tc_commit(mma_bar + b);
    }
  }
  // the last commit arrives once every MMA has completed
  wait(mma_bar + (nsteps - 1) % S, ((nsteps - 1) / S) & 1);
  cp_async_wait<0>();
  tc_fence_after();
  const unsigned trow = taddr + ((unsigned)(warp * 32) << 16);
#pragma unroll
  for (int c0 = 0; c0 < NO; c0 += 16) {
    float r[16];
    tc_ld16(trow + c0, r);
    tc_wait_ld();
    if (!valid) continue;
    if constexpr (MODE == 0) {
      uint32_t pk[8];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        float o0 = r[2 * i], o1 = r[2 * i + 1];
        if (bias) {
          o0 += bias[c0 + 2 * i];
          o1 += bias[c0 + 2 * i + 1];
        }
        if (flag) {
          o0 = fmaxf(o0, 0.0f);
          o1 = fmaxf(o1, 0.0f);
        }
        pk[i] = pack2(o0, o1);
      }
      uint4* o = reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(dst) + v * NO + c0);
      o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
    } else {
      float4* o = reinterpret_cast<float4*>(reinterpret_cast<float*>(dst) + v * NO + c0);
#pragma unroll
      for (int i = 0; i < 4; i++) {
        float4 w = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        if (flag) {  // accumulate into an existing gradient
          const float4 e = o[i];
          w.x += e.x;
          w.y += e.y;
          w.z += e.z;
          w.w += e.w;
        }
        o[i] = w;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(taddr, NCOLS);
}

template <int MODE, int NO>
int launch_conv_tc(const void* src, const bf16* Wc, const float* bias, void* dst, int Nb, int D, int H, int W, int KC,
                   int flag, cudaStream_t s) {
  constexpr size_t sm = conv_tc_smem<NO>();
  if (!tmk::allow_smem<k_conv_tc<MODE, NO>>(sm)) return -4;
  const long long nvox = (long long)Nb * D * H * W;
  const int blocks = (int)((nvox + 127) / 128);
  if (blocks > 0) k_conv_tc<MODE, NO><<<blocks, 128, sm, s>>>(src, Wc, bias, dst, Nb, D, H, W, KC, flag);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -4;
}

// compile-time loop: f(std::integral_constant<int, i>) for i in [B, E)
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}
// Stage the rows (z0 - 1 + r / RP, y0 - 1 + r % RP), r < ROWS, of batch item n, channels
// [c0, c0 + 16), into three copies shifted by dx = -1, 0, +1 in the K-major core-matrix
// layout [copy][channel half][r][x][8 channels] (copy c holds x + c - 1 at position x; zero
// outside the grid), in two parts so that other loads can be in flight in between:
// stage_halo_issue copies the unshifted rows by 16-byte asynchronous copies (all in flight);
// stage_halo_finish waits for them (block barrier) and builds the shifted copies in shared
// memory. The caller still fences the generic-proxy stores for the tensor core.
template <int W, int RP, int ROWS>
__device__ __forceinline__ void stage_halo_issue(unsigned char* As, const bf16* in, int n, int z0, int y0, int D,
                                                 int H, int KC, int c0) {
  using namespace tmk;
  constexpr int BOX = 16 * W * ROWS, ITEMS = 2 * ROWS * W;
  for (int i = threadIdx.x; i < ITEMS; i += blockDim.x) {
    const int x = i % W, r = (i / W) % ROWS, h = i / (W * ROWS);
    const int z = z0 - 1 + r / RP, y = y0 - 1 + r % RP;
    const bool ok = z >= 0 && z < D && y >= 0 && y < H;
    const long long e = ok ? ((((long long)n * D + z) * H + y) * W + x) * KC + c0 + h * 8 : c0;
    cp_async16(As + (2 + h) * BOX + (r * W + x) * 16, in + e, ok ? 16u : 0u);
  }
  cp_async_commit();
}
template <int W, int ROWS>
__device__ __forceinline__ void stage_halo_finish(unsigned char* As) {
  using namespace tmk;
  constexpr int BOX = 16 * W * ROWS, ITEMS = 2 * ROWS * W;
  cp_async_wait<0>();
  __syncthreads();
  for (int i = threadIdx.x; i < ITEMS; i += blockDim.x) {
    const int x = i % W, rest = i / W, h = rest / ROWS;  // rest = h ROWS + r
    const int o = (rest - h * ROWS) * W;                 // r W
    const uint4 v = *reinterpret_cast<const uint4*>(As + (2 + h) * BOX + (o + x) * 16);
    // copy 0 at x + 1 and copy 2 at x - 1 hold this voxel; their row ends are zero
    if (x + 1 < W) *reinterpret_cast<uint4*>(As + h * BOX + (o + x + 1) * 16) = v;
    if (x >= 1) *reinterpret_cast<uint4*>(As + (4 + h) * BOX + (o + x - 1) * 16) = v;
    if (x == 0) *reinterpret_cast<uint4*>(As + h * BOX + o * 16) = make_uint4(0u, 0u, 0u, 0u);
    if (x == W - 1) *reinterpret_cast<uint4*>(As + (4 + h) * BOX + (o + W - 1) * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Halo-tile implicit GEMM for grids whose rows hold W = 8, 16, 32 or 64 voxels (128 % W ==
// 0). A tile is TZ planes of RY = 128 / W rows of one batch item: TZ MMA tiles of M = 128, the
// RY rows of plane z0 + m in (y, x) order, one tensor-memory lane per voxel. A stage holds the
// (TZ + 2) x (RY + 2) rows around a tile for 16 channels of the reduced dimension: MODE 0 as one
// box copy brings them (32-byte rows, 32-byte swizzle, zero outside the grid), MODE 1 in the
// K-major core-matrix layout [channel half][z][y][x][8 channels], the float32 output gradient
// rounded to bfloat16 by the staging warps.
// The three taps of a row, dx = -1, 0, +1, are columns of one MMA (N = 3 NO): the A operand of
// a (dz, dy) pair is the staged rows from (m + dz + 1, dy + 1) on, unshifted, and the product
// with W(dz, dy, dx) is accumulated per dx; the epilogue adds the three, each taken from the
// lane one voxel to its side (warp shuffles, and shared memory between the two warps of a
// 64-voxel row; a voxel past the row's end is the zero padding). So 9 MMAs per stage and M
// tile instead of 27, and no dx-shifted copies of the rows: an MMA of so few columns is bound
// by reading A from shared memory (4 KB for M = 128, K = 16), and the copies were two thirds
// of the staging.
// One persistent block per SM, its warps specialized: staging (one thread for the box copies,
// or four groups of two warps, a buffer each), one thread per M tile that issues the MMAs, one
// that copies weights, and groups of four warps that read alternate accumulators (a ring in
// tensor memory) and write the output, which for MODE 1 is one bulk copy per M tile; mbarriers
// between them. The packed weights stay in shared memory where they fit, otherwise each stage
// brings its chunk's.
// Measured, 64^3 x 2: forward 48 -> 16 channels 139 -> 33 us, of which the MMAs' operand reads
// are 16 (44 cycles for M = 128, N = 48); data gradient 16 -> 48 113 -> 56 us. What bounds the
// latter is the path through L1 and shared memory, 78% busy while it runs (ncu; issue 36%, tensor
// pipe 18%, DRAM 74 MB): the float32 rows read and rounded, the operands of the MMAs and the
// output's staging all take it. Before: one block per two tiles, three shifted copies, 27 MMAs a
// chunk and nothing overlapped inside a block. On the way: 9 MMAs without the pipeline 88 and 139,
// rows staged by threads in MODE 0 59, 54 weight copies a chunk instead of one box 39.
// Two planes to a tile of 32-voxel rows in MODE 1 spill 328 bytes a thread; the layers that take
// the form are still ahead of the kernel before (32^3 x 4, 16 -> 16 channels 18.4 -> 14.4 us, 32 -> 32
// 36.9 -> 26.7).
template <int MODE, int W, int TZ, int NO>
struct Halo {
  static constexpr int RY = 128 / W, ROWS = (TZ + 2) * (RY + 2);
  static constexpr int BOX = 16 * W * ROWS;            // bytes of one channel half
  static constexpr int ABYTES = 2 * BOX;               // of one stage's rows
  static constexpr int BB = 27 * NO * 32;              // weights of one chunk
  static constexpr int CS = 3 * NO;                    // tensor-memory columns per M tile
  static constexpr int SLOTS = 512 / (TZ * CS) < 4 ? 512 / (TZ * CS) : 4;  // accumulators in the ring
  static constexpr int SW = MODE == 0 ? 0 : 8;         // staging warps
  static constexpr int EG = SLOTS >= 4 && MODE == 0 ? 4 : SLOTS > 1 ? 2 : 1;  // epilogue groups of four warps
  // the data gradient's rows of an M tile are one contiguous piece of memory: staged in shared
  // memory and written by one bulk copy
  static constexpr int OBYTES = 128 * NO * 4;
  static constexpr int THREADS = 32 * (SW + 4 * EG + TZ + 1 + (MODE == 0 ? 1 : 0));
  static_assert(SLOTS >= 1 && BB % 128 == 0, "accumulators; 128-byte aligned weights");
};
constexpr int kHaloStages = 4;
constexpr size_t kHaloTail = 8 * 64 * 4 + 64 * 4 + (2 * kHaloStages + 2 * 4 + 1) * 8 + 16;
// whether the output goes through shared memory (where a tile's rows are whole, see OBYTES)
template <int MODE, int NO>
__host__ __device__ constexpr bool halo_staged_out() {
  return MODE == 1;
}
// shared memory with ns stages: 256 bytes of slack to align the staged rows
template <int MODE, int W, int TZ, int NO>
constexpr size_t halo_smem(int ns, bool resident, int nk) {
  using HT = Halo<MODE, W, TZ, NO>;
  return 256 + (halo_staged_out<MODE, NO>() ? (size_t)HT::EG * HT::OBYTES : 0) +
         (size_t)ns * (HT::ABYTES + (resident ? 0 : HT::BB)) + (resident ? (size_t)nk * HT::BB : 0) + kHaloTail;
}
// contiguous bulk copy shared -> global (16-byte aligned, size a multiple of 16), and the wait
// until this thread's copies have read shared memory
__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n cp.async.bulk.commit_group;\n" ::"l"(dst),
               "r"(tmk::smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_store_wait() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(unsigned long long* mb) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(tmk::smem_u32(mb)) : "memory");
}

template <int MODE, int W, int TZ, int NO>
__global__ void __launch_bounds__(Halo<MODE, W, TZ, NO>::THREADS, 1)
k_conv_halo(const __grid_constant__ CUtensorMap rows, const __grid_constant__ CUtensorMap wts, const void* src,
            const float* bias, void* dst, int Nb, int D, int H, int KC, int NT,
            int ns, int resident, int flag) {
  using namespace tmk;
  using HT = Halo<MODE, W, TZ, NO>;
  constexpr int RY = HT::RY, ROWS = HT::ROWS, BOX = HT::BOX, ABYTES = HT::ABYTES, BB = HT::BB, CS = HT::CS;
  constexpr int SLOTS = HT::SLOTS, EG = HT::EG;
  constexpr unsigned IDESC = idesc_bf16(128, CS);
  extern __shared__ unsigned char smem_raw[];
  // MODE 0: [stage][z][y][x][32 B], the halves of rows 4 .. 7 of every eight exchanged (32-byte
  // swizzle); MODE 1: [stage][half][z][y][x][16 B]
  unsigned char* As = smem_raw + ((256 - (smem_u32(smem_raw) & 255)) & 255);
  const int nk = KC >> 4;
  unsigned char* Bs = As + ns * ABYTES;  // [stage or chunk][dz dy][k half][dx][NO/8][8][16 B]
  float* xs = reinterpret_cast<float*>(Bs + (resident ? nk : ns) * BB + (halo_staged_out<MODE, NO>() ? EG * HT::OBYTES : 0));  // [group][parity][row][voxel 31, 32][16] (W = 64)
  float* bs = xs + 8 * 64;  // the bias (MODE 0)
  unsigned long long* full = reinterpret_cast<unsigned long long*>(bs + 64);
  unsigned long long *empty = full + kHaloStages, *accfull = empty + kHaloStages, *accempty = accfull + 4,
                     *wbar = accempty + 4;
  unsigned* tslot = reinterpret_cast<unsigned*>(wbar + 1);
  constexpr bool STAGED = halo_staged_out<MODE, NO>();
  const bool staged = STAGED && NT == NO;
  unsigned char* Os = As + ns * ABYTES + (resident ? nk : ns) * BB;  // [group][128 voxels][NO] (STAGED)
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int SW = HT::SW, MMA0 = SW + 4 * EG, WARP_W = MMA0 + TZ;  // first issuing warp, the weights' warp
  if (t == 0) {
    for (int k = 0; k < ns; k++) {
      mbar_init(full + k, (MODE == 0 ? 1 : 64) + (resident ? 0 : 1));  // the staging group, and the weights' warp
      mbar_init(empty + k, TZ);
    }
    for (int k = 0; k < SLOTS; k++) {
      mbar_init(accfull + k, TZ);
      mbar_init(accempty + k, 128);
    }
    mbar_init(wbar, 1);
    mbar_init_fence();
  }
  if (MODE == 0 && t < NO) bs[t] = bias ? bias[blockIdx.y * NO + t] : 0.0f;
  if (warp == MMA0) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = *tslot;
  bool dead = false;  // a wait ran out: no further waits in this thread, results flagged
  auto wait = [&](unsigned long long* mb, unsigned parity) {
    if (!dead) dead = !mbar_wait_limit(mb, parity & 1, 1 << 16, &g_net_status);
  };
  const int nyt = (H + RY - 1) / RY, nzt = (D + TZ - 1) / TZ;
  const int ntiles = Nb * nzt * nyt;
  // one chunk's weights, this block's window of output channels: one copy of a box that takes the
  // packed blocks [tap][chunk][k half][NT/8][8][8] in the order [dz dy][k half][dx] (54 copies of
  // NO x 16 bytes, issued by one thread, took 2 us a chunk)
  auto load_weights = [&](unsigned char* b, int kc, unsigned long long* mb) {
    tma_load_5d(b, &wts, blockIdx.y * (NO * 2), 0, 0, 0, kc, mb);
  };
  if (MODE == 0 && warp == WARP_W + 1) {
    // ---- staging, MODE 0: one copy of a box of rows per stage, zero outside the grid
    if (lane == 0) {
      fence_proxy_async_global();  // the rows were written by ordinary stores
      int s = 0;
      unsigned phase = 0;
      for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int yt = tile % nyt, zt = (tile / nyt) % nzt, n = tile / (nyt * nzt);
        for (int kc = 0; kc < nk; kc++) {
          if (phase > 0) wait(empty + s, phase - 1);
          mbar_expect_tx(full + s, ABYTES);
          tma_load_5d(As + s * ABYTES, &rows, kc * 16, 0, yt * RY - 1, zt * TZ - 1, n, full + s);
          if (++s == ns) {
            s = 0;
            phase++;
          }
        }
      }
    }
  } else if (warp < SW) {
    // ---- staging: group g of two warps fills buffer g (a group that took turns on several
    // buffers could wait for an empty one two phases ahead of its barrier); two lanes per
    // voxel, one per channel half
    const int g = warp >> 1, tg = t & 63;
    constexpr int VPR = 32;  // voxels per round of the group
    constexpr int XP = W < VPR ? 1 : W / VPR, RPI = VPR / W < 1 ? 1 : VPR / W;  // rounds per row, rows per round
    constexpr int RIT = (ROWS + RPI - 1) / RPI, ITER = RIT * XP;
    const int h = tg & 1, xv = (tg >> 1) % W, r0 = (tg >> 1) / W;
    const long long rowp = (long long)W * KC, planep = H * rowp;
    int kc = g < ns ? g : nk;  // the group's next chunk, counted from the current tile's first
    unsigned phase = 0;        // uses of the buffer so far
    const int s = g;
    unsigned char* as = As + s * ABYTES + h * BOX + xv * 16;
    for (int tile = blockIdx.x; tile < ntiles && g < ns; tile += gridDim.x) {
      if (kc < nk) {
        const int yt = tile % nyt, zt = (tile / nyt) % nzt, n = tile / (nyt * nzt);
        const int y0 = yt * RY - 1, z0 = zt * TZ - 1;
        unsigned zok = 0, yok = 0;
#pragma unroll
        for (int q = 0; q < TZ + 2; q++) zok |= (unsigned)((unsigned)(z0 + q) < (unsigned)D) << q;
#pragma unroll
        for (int q = 0; q < RY + 2; q++) yok |= (unsigned)((unsigned)(y0 + q) < (unsigned)H) << q;
        const long long base0 = (((long long)n * D + z0) * H + y0) * rowp + (long long)xv * KC + h * 8;
        for (; kc < nk; kc += ns) {
          if (phase > 0) wait(empty + s, phase - 1);
          phase++;
          const long long base = base0 + kc * 16;
          auto row_of = [&](int it, int& r, int& zr, int& yr) {
            r = (it / XP) * RPI + r0;
            zr = r / (RY + 2);
            yr = r % (RY + 2);
          };
          {
            const float* in = reinterpret_cast<const float*>(src);
            constexpr int BATCH = 8;  // rounds whose loads are in flight together
#pragma unroll
            for (int i0 = 0; i0 < ITER; i0 += BATCH) {
              float4 f[BATCH][2];
#pragma unroll
              for (int b = 0; b < BATCH; b++) {
                int r, zr, yr;
                row_of(i0 + b, r, zr, yr);
                f[b][0] = f[b][1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (i0 + b < ITER && r < ROWS && ((zok >> zr) & (yok >> yr) & 1)) {
                  const float4* q = reinterpret_cast<const float4*>(in + base + zr * planep + yr * rowp +
                                                                    ((i0 + b) % XP) * (VPR * KC));
                  f[b][0] = q[0];
                  f[b][1] = q[1];
                }
              }
#pragma unroll
              for (int b = 0; b < BATCH; b++) {
                int r, zr, yr;
                row_of(i0 + b, r, zr, yr);
                if (i0 + b < ITER && (ROWS % RPI == 0 || r < ROWS))
                  *reinterpret_cast<uint4*>(as + (r * W + ((i0 + b) % XP) * VPR) * 16) =
                      make_uint4(pack2(f[b][0].x, f[b][0].y), pack2(f[b][0].z, f[b][0].w), pack2(f[b][1].x, f[b][1].y),
                                 pack2(f[b][1].z, f[b][1].w));
              }
            }
          }
          fence_proxy_async_smem();  // the rows, written through the generic proxy, for the tensor core
          mbar_arrive(full + s);
        }
      }
      kc -= nk;
    }
  } else if (warp == WARP_W) {
    // ---- weights: all chunks once, or each stage's chunk
    if (lane == 0) {
      fence_proxy_async_global();  // they were written by ordinary stores
      if (resident) {
        mbar_expect_tx(wbar, nk * BB);
        for (int kc = 0; kc < nk; kc++) load_weights(Bs + kc * BB, kc, wbar);
      } else {
        int s = 0;
        unsigned phase = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
          for (int kc = 0; kc < nk; kc++) {
            if (phase > 0) wait(empty + s, phase - 1);
            mbar_expect_tx(full + s, BB);
            load_weights(Bs + s * BB, kc, full + s);
            if (++s == ns) {
              s = 0;
              phase++;
            }
          }
      }
    }
  } else if (warp >= MMA0) {
    // ---- MMAs of M tile m: one thread
    const int m = warp - MMA0;
    if (lane == 0) {
      if (resident) wait(wbar, 0);
      // MODE 0: rows of 32 bytes in the 32-byte swizzle (layout type 6), eight rows 256 bytes
      const uint64_t a00 = MODE == 0 ? smem_desc(As + m * (RY + 2) * W * 32, 16, 256) | (uint64_t)6 << 61
                                     : smem_desc(As + m * (RY + 2) * W * 16, BOX, 128);
      const uint64_t b00 = smem_desc(Bs, 3 * NO * 16, 128);
      int u = 0, s = 0;
      unsigned phase = 0;
      for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, u++) {
        const int slot = u % SLOTS;
        if (u >= SLOTS) wait(accempty + slot, u / SLOTS - 1);
        const unsigned acc = taddr + (slot * TZ + m) * CS;
        for (int kc = 0; kc < nk; kc++) {
          wait(full + s, phase);
          tc_fence_after();
          const uint64_t a0 = a00 + (unsigned)(s * (ABYTES >> 4)), b0 = b00 + (unsigned)((resident ? kc : s) * (BB >> 4));
          static_for<0, 9>([&](auto pair_c) {
            constexpr int pair = decltype(pair_c)::value, sg = MODE == 1 ? -1 : 1;
            constexpr int dz = sg * (pair / 3 - 1), dy = sg * (pair % 3 - 1);
            constexpr unsigned aoff = (unsigned)(((dz + 1) * (RY + 2) + dy + 1) * W) * (MODE == 0 ? 2 : 1);
            tc_mma(acc, a0 + aoff, b0 + (unsigned)(pair * NO * 6), IDESC, kc > 0 || pair > 0);
          });
          tc_commit(empty + s);
          if (++s == ns) {
            s = 0;
            phase++;
          }
        }
        tc_commit(accfull + slot);
      }
    }
  } else {
    // ---- epilogue: group e takes accumulators e, e + EG, ..
    const int e = (warp - SW) >> 2, w4 = warp & 3, v = w4 * 32 + lane, x = v % W;
    const bool pl = x > 0, pr = x < W - 1;
    unsigned step = 0;
    int u = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, u++) {
      if (u % EG != e) continue;
      const int slot = u % SLOTS;
      const int yt = tile % nyt, zt = (tile / nyt) % nzt, n = tile / (nyt * nzt);
      const int y = yt * RY + v / W;
      wait(accfull + slot, u / SLOTS);
      __syncwarp();
      tc_fence_after();
#pragma unroll 1
      for (int m = 0; m < TZ; m++) {
        const int z = zt * TZ + m;
        const bool valid = z < D && y < H;
        const long long o0 = ((((long long)n * D + z) * H + y) * W + x) * NT + blockIdx.y * NO;
        const unsigned trow = taddr + ((unsigned)(w4 * 32) << 16) + (slot * TZ + m) * CS;
        if (staged && (u != e || m > 0)) {  // the last copy has read the buffer
          if (w4 == 0 && lane == 0) bulk_store_wait();
          __syncwarp();
          bar_named(5 + e, 128);
        }
#pragma unroll 1
        for (int c0 = 0; c0 < NO; c0 += 16) {
          // lf: the products of the voxel at x - 1, taken from its lane; rt: of the one at x + 1
          float r[16], lf[16], rt[16];
          tc_ld16(trow + (MODE == 0 ? 0 : 2) * NO + c0, lf);
          tc_ld16(trow + NO + c0, r);
          tc_ld16(trow + (MODE == 0 ? 2 : 0) * NO + c0, rt);
          tc_wait_ld();
          if (m == TZ - 1 && c0 == NO - 16) {  // the accumulator has been read
            tc_fence_before();
            mbar_arrive(accempty + slot);
          }
          if constexpr (W == 64) {  // voxels 31 and 32 of a row belong to two warps
            float* xr = xs + (e * 2 + (step & 1)) * 64 + (w4 >> 1) * 32;  // the other parity may still be read
            if ((w4 & 1) == 0 && lane == 31) {
#pragma unroll
              for (int i = 0; i < 4; i++)
                reinterpret_cast<float4*>(xr)[i] = make_float4(lf[4 * i], lf[4 * i + 1], lf[4 * i + 2], lf[4 * i + 3]);
            }
            if ((w4 & 1) == 1 && lane == 0) {
#pragma unroll
              for (int i = 0; i < 4; i++)
                reinterpret_cast<float4*>(xr + 16)[i] = make_float4(rt[4 * i], rt[4 * i + 1], rt[4 * i + 2], rt[4 * i + 3]);
            }
            __syncwarp();
            bar_named(1 + e * 2 + (w4 >> 1), 64);
            step++;
#pragma unroll
            for (int i = 0; i < 16; i++) {
              const float a = __shfl_up_sync(0xffffffffu, lf[i], 1), b = __shfl_down_sync(0xffffffffu, rt[i], 1);
              lf[i] = a;
              rt[i] = b;
            }
            const bool ml = (w4 & 1) == 1 && lane == 0, mr = (w4 & 1) == 0 && lane == 31;
#pragma unroll
            for (int i = 0; i < 4; i++) {  // every lane reads (a broadcast), one keeps it
              const float4 q = reinterpret_cast<const float4*>(xr + ((w4 & 1) ? 0 : 16))[i];
              const float w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
              for (int k = 0; k < 4; k++) {
                lf[4 * i + k] = ml ? w[k] : lf[4 * i + k];
                rt[4 * i + k] = mr ? w[k] : rt[4 * i + k];
              }
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; i++) {
              lf[i] = __shfl_up_sync(0xffffffffu, lf[i], 1);
              rt[i] = __shfl_down_sync(0xffffffffu, rt[i], 1);
            }
          }
#pragma unroll
          for (int i = 0; i < 16; i++) {
            // (selects: as conditional adds these were 16 divergent branches a step, 1000 cycles)
            r[i] += pl ? lf[i] : 0.0f;
            r[i] += pr ? rt[i] : 0.0f;
          }
          if (!valid) {
          } else if constexpr (MODE == 0) {
            uint32_t pk[8];
#pragma unroll
            for (int i = 0; i < 8; i++) {
              const float2 bb = *reinterpret_cast<const float2*>(bs + c0 + 2 * i);
              float a = r[2 * i] + bb.x, b = r[2 * i + 1] + bb.y;
              if (flag) {
                a = fmaxf(a, 0.0f);
                b = fmaxf(b, 0.0f);
              }
              pk[i] = pack2(a, b);
            }
            uint4* o = reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(dst) + o0 + c0);
            o[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            o[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
          } else {
            float4* o = reinterpret_cast<float4*>(reinterpret_cast<float*>(dst) + o0 + c0);
            if (flag) {  // accumulate into an existing gradient
#pragma unroll
              for (int i = 0; i < 4; i++) {
                const float4 old = o[i];
                r[4 * i] += old.x, r[4 * i + 1] += old.y, r[4 * i + 2] += old.z, r[4 * i + 3] += old.w;
              }
            }
            if (staged) o = reinterpret_cast<float4*>(Os + e * HT::OBYTES + (v * NO + c0) * 4);
#pragma unroll
            for (int i = 0; i < 4; i++) o[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
          }
          __syncwarp();
        }
        if (staged) {  // one bulk copy of the M tile's rows that lie in the grid
          fence_proxy_async_smem();
          bar_named(5 + e, 128);
          const int rows = z < D ? min(RY, H - yt * RY) : 0;
          if (w4 == 0 && lane == 0 && rows > 0)
            bulk_store(reinterpret_cast<float*>(dst) + ((((long long)n * D + z) * H + yt * RY) * W) * NO, Os + e * HT::OBYTES,
                       rows * W * NO * 4);
        }
      }
    }
  }
  if (staged && (t & 31) == 0) bulk_store_wait();
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == MMA0) {
    tc_fence_after();
    tmem_dealloc(taddr, 512);
  }
}

// A tensor map could not be made: nothing was launched. The gather kernels need no maps.
constexpr int kNoMap = 1;
template <int MODE, int W, int TZ, int NO>
int launch_conv_halo_tz(const void* src, const bf16* Wc, const float* bias, void* dst, int Nb, int D, int H, int KC,
                        int NT, int flag, cudaStream_t s) {
  using HT = Halo<MODE, W, TZ, NO>;
  constexpr size_t kMost = 227 * 1024;
  const int nk = KC >> 4;
  // weights resident if they leave room for three stages of rows; at least two stages either way
  const bool resident = halo_smem<MODE, W, TZ, NO>(3, true, nk) <= kMost;
  int ns = kHaloStages;
  while (ns > 2 && halo_smem<MODE, W, TZ, NO>(ns, resident, nk) > kMost) ns--;
  const size_t sm = halo_smem<MODE, W, TZ, NO>(ns, resident, nk);
  static_assert(halo_smem<MODE, W, TZ, NO>(2, false, 1) <= kMost, "shared memory of one block");
  if (!tmk::allow_smem<k_conv_halo<MODE, W, TZ, NO>>(kMost)) return -4;
  const long long tiles = (long long)Nb * ((D + TZ - 1) / TZ) * ((H + HT::RY - 1) / HT::RY);
  if (tiles > 0x7fffffffLL) return -1;
  if (tiles <= 0) return 0;
  CUtensorMap rows = {}, wts = {};
  tmk::EncodeTiledFn fn = tmk::encoder();
  if (!fn) return kNoMap;
  {  // in units of 8 bytes: channel groups, dx, k half, (dz, dy), chunk
    const cuuint64_t dims[5] = {2ull * NT, 3, 2, 9, (cuuint64_t)nk};
    const cuuint64_t pitch[4] = {32ull * NT * nk, 16ull * NT, 96ull * NT * nk, 32ull * NT};
    const cuuint32_t box[5] = {2 * NO, 3, 2, 9, 1}, step[5] = {1, 1, 1, 1, 1};
    if (fn(&wts, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, const_cast<bf16*>(Wc), dims, pitch, box, step,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return kNoMap;
  }
  if (MODE == 0) {
    const cuuint64_t dims[5] = {(cuuint64_t)KC, W, (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)Nb};
    const cuuint64_t pitch[4] = {2ull * KC, 2ull * KC * W, 2ull * KC * W * H, 2ull * KC * W * H * D};
    const cuuint32_t box[5] = {16, W, HT::RY + 2, TZ + 2, 1}, step[5] = {1, 1, 1, 1, 1};
    if (fn(&rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(src), dims, pitch, box, step,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return kNoMap;
  }
  const int windows = NT / NO, gx = sm_count() / windows;  // one block per SM
  k_conv_halo<MODE, W, TZ, NO><<<dim3((unsigned)(tiles < gx ? tiles : gx), windows), HT::THREADS, sm, s>>>(
        rows, wts, src, bias, dst, Nb, D, H, KC, NT, ns, resident, flag);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -4;
}
// Two planes per tile read each staged row for more of its taps, as far as two accumulators fit
// in tensor memory; one plane where two would leave SMs without a tile (16^3 x 2). 96 channels
// go as two windows of 48 on their own blocks: their accumulator alone would be 288 columns
// wide, so that no epilogue could run beside the next tile's MMAs. Two planes of a window fill
// the tensor memory in the same way, which pays where it saves more than the overlap: where each
// stage brings its weights (more than 32 reduced channels: 64^3 x 4, 96 from 64, 850 -> 615 us),
// and with resident weights where two planes take no more rounds of tiles than one (96 from 32,
// 64^3 x 4 447 -> 390, 32^3 19.0 -> 18.5; 24 x 32 x 32, two rounds against three, 16.4 -> 18.5).
// With 16 reduced channels the epilogue is most of a tile (64^3 x 4 272 with one plane, 283), and
// so it is for rows of 8 or 16 that add to a gradient (96 from 32, 64 x 64 x 8 x 4, 55.5 and 61.5).
template <int MODE, int W, int NO>
int launch_conv_halo(const void* src, const bf16* Wc, const float* bias, void* dst, int Nb, int D, int H, int KC,
                     int flag, cudaStream_t s) {
  constexpr int NW = NO == 96 ? 48 : NO;
  if constexpr (NW <= 32) {
    if ((long long)Nb * ((D + 1) / 2) * ((H + 128 / W - 1) / (128 / W)) >= sm_count())
      return launch_conv_halo_tz<MODE, W, 2, NW>(src, Wc, bias, dst, Nb, D, H, KC, NO, flag, s);
  }
  if constexpr (NO == 96) {
    const int ny = (H + 128 / W - 1) / (128 / W), gx = sm_count() > 1 ? sm_count() / 2 : 1;
    const long long t1 = (long long)Nb * D * ny, t2 = (long long)Nb * ((D + 1) / 2) * ny;
    const bool resident = halo_smem<MODE, W, 1, NW>(3, true, KC >> 4) <= 227 * 1024;
    if (resident ? KC > 16 && (W >= 32 || !flag) && 2 * ((t2 + gx - 1) / gx) <= (t1 + gx - 1) / gx : t2 >= gx)
      return launch_conv_halo_tz<MODE, W, 2, NW>(src, Wc, bias, dst, Nb, D, H, KC, NO, flag, s);
  }
  return launch_conv_halo_tz<MODE, W, 1, NW>(src, Wc, bias, dst, Nb, D, H, KC, NO, flag, s);
}

// the halo kernel for rows of 8 .. 64 voxels, else (or without tensor maps) the per-voxel gather
// kernel; either copies the weights in pieces of 16 bytes
template <int MODE, int NO>
int launch_conv(const void* src, const bf16* Wc, const float* bias, void* dst, int Nb, int D, int H, int W, int KC,
                int flag, cudaStream_t s) {
  if (reinterpret_cast<uintptr_t>(Wc) & 15) return -4;
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    int r = kNoMap;
    if (W == 64) r = launch_conv_halo<MODE, 64, NO>(src, Wc, bias, dst, Nb, D, H, KC, flag, s);
    if (W == 32) r = launch_conv_halo<MODE, 32, NO>(src, Wc, bias, dst, Nb, D, H, KC, flag, s);
    if (W == 16) r = launch_conv_halo<MODE, 16, NO>(src, Wc, bias, dst, Nb, D, H, KC, flag, s);
    if (W == 8) r = launch_conv_halo<MODE, 8, NO>(src, Wc, bias, dst, Nb, D, H, KC, flag, s);
    if (r != kNoMap) return r;
  }
  return launch_conv_tc<MODE, NO>(src, Wc, bias, dst, Nb, D, H, W, KC, flag, s);
}

// Weight gradient on tcgen05: dW[tap][ci][co] = sum_v in[v + off(tap)][ci] q(dout[v][co]),
// a GEMM with rows (tap, ci), columns co and the voxels as the reduction. A block owns one
// row tile of 128 = 8 taps x 16 input channels (tile = (tap group, channel chunk)) and a
// range of voxels, 16 per MMA (K = 16), kDwChunks MMAs per pipeline stage; its float32
// accumulator (128 x NO) lives in tensor memory and is written out as one partial, and
// k_dw_reduce_tc adds the partials in block order. Both operands are MN-major, so the channels-last rows go into shared memory as
// they are: A gets each (tap, voxel)'s 16 shifted input channels (two 16-byte pieces), B
// each voxel's NO output-gradient channels, taken from a bfloat16 copy made beforehand
// (rounded to nearest even, the operand precision of every product).
constexpr int kDwStages = 3, kDwChunks = 4;  // pipeline stages; 16-voxel chunks (MMAs) per stage
constexpr int kDwBlocksPerSm = 4;            // voxel blocks per SM, over all row tiles
template <int NO>
constexpr size_t dw_tc_smem() {
  return (size_t)kDwStages * kDwChunks * (128 * 32 + NO * 32) + (2 * kDwStages + 1) * 8 + 16;
}
template <int NO>
__global__ void __launch_bounds__(128) k_conv_dw_tc(const bf16* in, const bf16* g16, float* part, int Nb, int D,
                                                    int H, int W, int Cin, long long chunks_per_block) {
  using namespace tmk;
  constexpr int S = kDwStages, KS = kDwChunks, AB = 128 * 32, BB = NO * 32, PG = NO / 8;
  constexpr unsigned NCOLS = tmem_cols<NO>();
  constexpr unsigned IDESC = idesc_bf16(128, NO, true);
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* As = smem;                // [S][KS][k-group (2)][16 row groups][8 k-rows][16 B]
  unsigned char* Bs = smem + S * KS * AB;  // [S][KS][2][PG][8][16 B]
  unsigned long long* mma_bar = reinterpret_cast<unsigned long long*>(Bs + S * KS * BB);
  unsigned* tslot = reinterpret_cast<unsigned*>(mma_bar + S);
  const int t = threadIdx.x, warp = t >> 5;
  if (t == 0) {
    for (int b = 0; b < S; b++) mbar_init(mma_bar + b, 1);
    mbar_init_fence();
  }
  if (warp == 0) {
    tmem_alloc(tslot, NCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = *tslot;
  bool dead = false;
  auto wait = [&](unsigned long long* mb, unsigned parity) {
    if (!dead) dead = !mbar_wait_limit(mb, parity, 1 << 16, &g_net_status);
  };
  const long long nvox = (long long)Nb * D * H * W;
  const int tile = blockIdx.y, ncc = Cin >> 4;
  const int tg = tile / ncc, cc = tile - tg * ncc;
  // A: this thread's (tap, voxel) = (8 tg + t / 16, t % 16) of each chunk
  const int tap = 8 * tg + (t >> 4), ka = t & 15;
  const bool tap_ok = tap < 27;
  const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
  const int aoff = (t >> 4) * 2 * 128 + (ka >> 3) * 2048 + (ka & 7) * 16;
  // B: this thread's piece (voxel kb, 8 channels pg) of each chunk, if t < 16 PG
  const int kb = t / PG, pg = t - kb * PG;
  const int boff = pg * 128 + (kb >> 3) * (PG * 128) + (kb & 7) * 16;
  const long long c0 = (long long)blockIdx.x * chunks_per_block;
  const long long nch = (nvox + 15) / 16;
  const long long c1 = c0 + chunks_per_block < nch ? c0 + chunks_per_block : nch;
  const int nsteps = c1 > c0 ? (int)((c1 - c0 + KS - 1) / KS) : 0;
  // this thread's A voxel v = 16 ch + ka as a cursor (x, y, z, n) that the steps advance by
  // 16 voxels in order (no divisions in the loop)
  int cx = 0, cy = 0, cz = 0;
  long long cn = 0;
  {
    long long q = c0 * 16 + ka;
    cx = (int)(q % W);
    q /= W;
    cy = (int)(q % H);
    q /= H;
    cz = (int)(q % D);
    cn = q / D;
  }
  // step s: chunks c0 + s KS + k (k < KS) of the block's range; chunks past it read zeros
  auto load_step = [&](int s, int b) {
#pragma unroll
    for (int k = 0; k < KS; k++) {
      const long long ch = c0 + (long long)s * KS + k;
      const long long v0 = ch * 16;
      const bool in_range = ch < c1;
      {
        const long long v = v0 + ka;
        const int x = cx + dx, y = cy + dy, z = cz + dz;
        const bool ok = in_range && tap_ok && v < nvox && z >= 0 && z < D && y >= 0 && y < H && x >= 0 && x < W;
        const long long u = ok ? ((cn * D + z) * H + y) * W + x : 0;
        cx += 16;  // the cursor moves to this thread's voxel of the next chunk
        while (cx >= W) {
          cx -= W;
          if (++cy == H) {
            cy = 0;
            if (++cz == D) {
              cz = 0;
              ++cn;
            }
          }
        }
        const bf16* src = in + u * Cin + cc * 16;
        unsigned char* a = As + (b * KS + k) * AB + aoff;
        cp_async16(a, src, ok ? 16u : 0u);            // channels 0..7: row group 2 (t / 16)
        cp_async16(a + 128, src + 8, ok ? 16u : 0u);  // channels 8..15: the next row group
      }
      if (t < 16 * PG) {
        const long long v = v0 + kb;
        const bool ok = in_range && v < nvox;
        cp_async16(Bs + (b * KS + k) * BB + boff, g16 + (ok ? v : 0) * NO + pg * 8, ok ? 16u : 0u);
      }
    }
  };
  for (int s = 0; s < S - 1; s++) {  // always S - 1 groups, so that the wait below counts right
    if (s < nsteps) load_step(s, s);
    cp_async_commit();
  }
  for (int s = 0; s < nsteps; s++) {
    const int b = s % S;
    const int sn = s + S - 1;
    if (sn < nsteps) {
      const int bn = sn % S;
      if (s >= 1) wait(mma_bar + bn, ((s - 1) / S) & 1);
      load_step(sn, bn);
    }
    cp_async_commit();
    cp_async_wait<S - 1>();
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < KS; k++) {
        const uint64_t ad = smem_desc(As + (b * KS + k) * AB, 2048, 128);
        const uint64_t bd = smem_desc(Bs + (b * KS + k) * BB, PG * 128, 128);
        tc_mma(taddr, ad, bd, IDESC, s > 0 || k > 0);
      }
      tc_commit(mma_bar + b);
    }
  }
  if (nsteps > 0) wait(mma_bar + (nsteps - 1) % S, ((nsteps - 1) / S) & 1);
  cp_async_wait<0>();
  tc_fence_after();
  // row t of the tile: tap 8 tg + t / 16, channel 16 cc + t % 16
  float* pr = part + (((long long)blockIdx.x * gridDim.y + tile) * 128 + t) * NO;
  const unsigned trow = taddr + ((unsigned)(warp * 32) << 16);
#pragma unroll
  for (int q0 = 0; q0 < NO; q0 += 16) {
    float r[16];
    tc_ld16(trow + q0, r);
    tc_wait_ld();
#pragma unroll
    for (int i = 0; i < 16; i++) r[i] = nsteps > 0 ? r[i] : 0.0f;
    float4* o = reinterpret_cast<float4*>(pr + q0);
#pragma unroll
    for (int i = 0; i < 4; i++) o[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(taddr, NCOLS);
}

// Weight gradient for rows of 16, 32 or 64 voxels: dW[tap][ci][co] =
// sum_v in[v + off(tap)][ci] q(dout[v][co]) as MMAs with K = 16 voxels of one row of dout, M = 8
// input rows x 16 channels and N = 3 NO, the output channels for the three dx. A tile is TZ
// planes of RT rows; a stage holds the (TZ + 2) x (RT + 2) input rows around it for one
// 16-channel chunk, [z][y][x][16 channels] in the 32-byte swizzle as one box copy brings them.
// Read as an MN-major operand, the rows from (z, y) on are M groups one row apart: with PR = RT
// + 2 rows per plane, the input row of (dz, dy) is group dz PR + dy, so two MMAs of M = 128
// (groups 0-7 and 8-15) hold all nine for every row of the tile; the groups between are
// products that nothing reads. The output gradient, rounded to bfloat16, lies in shared memory
// as [row][dx][8 channels][x], dx-shifted (zero past the row's ends), which makes dx part of N.
// So each MMA does 9/16 x 128 x 48 useful products for NO = 16, where M = 16 output channels
// padded to 128 against N = 48 did an eighth of its columns' work and 9 MMAs per 16 voxels.
// One persistent block per SM: one thread copies input rows, eight warps round and store the
// output gradient (and add up the bias gradient from the float32 values they read), one thread
// per M tile issues MMAs; the accumulators stay in tensor memory over all tiles of the block.
// Channel chunks go in groups of 512 / (6 NO), each on its own blocks. Each block writes its
// sums as one partial, added in block order by k_dw_finish. There are as many partials as SMs
// whatever the number of groups: the tensor core's accumulation loses about a bit per doubling
// of the voxels that one accumulator adds up, and with the SMs divided among the groups (a
// quarter of the partials for 64 -> 64 channels) the sums of a 64^3 x 2 layer were off by 7.5e-6
// relative instead of 1.4e-6 (262 us; with all partials 303, k_conv_dw_halo 853).
// What bounds it: reading the operands of the MMAs from shared memory (44 cycles for M = 128, N =
// 48, K = 16). Measured, 64^3 x 2, 48 -> 16 channels with db: 432 -> 49 us.
// RMAX: rows of a tile at most.
template <int W, int NO, int RMAX>
struct DwRows {
  static constexpr int ROWB = 6 * NO * W;                     // bytes of one staged output-gradient row
  static constexpr int MAXR = 50 * 1024 / ROWB < RMAX ? 50 * 1024 / ROWB : RMAX;  // two buffers of them
  static constexpr int TZ = MAXR >= 8 ? 2 : 1, RT = MAXR >= 4 ? 4 : 2;
  static constexpr int PR = RT + 2, DROWS = TZ * RT;
  static constexpr int ABYTES = (TZ + 2) * PR * W * 32;       // one stage of input rows
  static constexpr int GBYTES = DROWS * ROWB;                 // one buffer of output-gradient rows
  static constexpr int NS = 2 * ABYTES + 2 * GBYTES > 150 * 1024 ? 2 : 3;
  static constexpr int GROUP = 512 / (6 * NO);                // channel chunks per block
  static constexpr int THREADS = 256 + 64 + 32;
  // the second M tile of the last row reads up to 16 rows past its first: they stay inside
  static constexpr size_t SMEM = 256 + (size_t)NS * ABYTES + 2 * GBYTES + 256 * 8 * 4 + (2 * NS + 5) * 8 + 16;
  static_assert(MAXR >= 2 && GROUP >= 1 && 2 * PR + 2 <= 15 && SMEM <= 227 * 1024, "tile");
  static_assert(2 * GBYTES + 256 * 8 * 4 >= 8 * W * 32, "rows read past the stages");
};
template <int W, int NO, int RMAX>
__global__ void __launch_bounds__(DwRows<W, NO, RMAX>::THREADS, 1)
k_conv_dw_rows(const __grid_constant__ CUtensorMap rows, const float* dout, float* part, int Nb, int D, int H, int Cin) {
  using namespace tmk;
  using T = DwRows<W, NO, RMAX>;
  constexpr int TZ = T::TZ, RT = T::RT, PR = T::PR, DROWS = T::DROWS, ROWB = T::ROWB, NS = T::NS, CG = NO / 8;
  constexpr unsigned IDESC = idesc_bf16(128, 3 * NO, true);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* As = smem_raw + ((256 - (smem_u32(smem_raw) & 255)) & 255);  // [stage][z][y][x][32 B], swizzled
  unsigned char* Gs = As + NS * T::ABYTES;                                     // [buffer][row][dx][CG][x][16 B]
  float* dbs = reinterpret_cast<float*>(Gs + 2 * T::GBYTES);                   // [256][8] bias sums
  unsigned long long* full = reinterpret_cast<unsigned long long*>(dbs + 256 * 8);
  unsigned long long *empty = full + NS, *gfull = empty + NS, *gempty = gfull + 2, *done = gempty + 2;
  unsigned* tslot = reinterpret_cast<unsigned*>(done + 1);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if (t == 0) {
    for (int k = 0; k < NS; k++) {
      mbar_init(full + k, 1);
      mbar_init(empty + k, 2);
    }
    for (int k = 0; k < 2; k++) {
      mbar_init(gfull + k, 256);
      mbar_init(gempty + k, 2);
    }
    mbar_init(done, 2);
    mbar_init_fence();
  }
  if (warp == 8) {
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = *tslot;
  bool dead = false;  // a wait ran out: no further waits in this thread, results flagged
  auto wait = [&](unsigned long long* mb, unsigned parity) {
    if (!dead) dead = !mbar_wait_limit(mb, parity & 1, 1 << 16, &g_net_status);
  };
  const int nyt = (H + RT - 1) / RT, nzt = (D + TZ - 1) / TZ, ntiles = Nb * nzt * nyt;
  const int kc0 = blockIdx.y * T::GROUP, kc1 = min(kc0 + T::GROUP, Cin >> 4);
  if (warp == 10) {
    if (lane == 0) {
      fence_proxy_async_global();  // the input was written by ordinary stores
      int s = 0;
      unsigned phase = 0;
      for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int yt = tile % nyt, zt = (tile / nyt) % nzt, n = tile / (nyt * nzt);
        for (int kc = kc0; kc < kc1; kc++) {
          if (phase > 0) wait(empty + s, phase - 1);
          mbar_expect_tx(full + s, T::ABYTES);
          tma_load_5d(As + s * T::ABYTES, &rows, kc * 16, 0, yt * RT - 1, zt * TZ - 1, n, full + s);
          if (++s == NS) {
            s = 0;
            phase++;
          }
        }
      }
    }
  } else if (warp >= 8) {
    const int m = warp - 8;  // M tile: row groups 8 m .. 8 m + 7
    if (lane == 0) {
      const uint64_t a00 = smem_desc(As + m * 8 * W * 32, W * 32, 256) | (uint64_t)6 << 61;
      const uint64_t b00 = smem_desc(Gs, 128, W * 16);
      int s = 0, it = 0;
      unsigned phase = 0;
      for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, it++) {
        const int d = it & 1;
        wait(gfull + d, it >> 1);
        for (int kc = kc0; kc < kc1; kc++) {
          wait(full + s, phase);
          tc_fence_after();
          const unsigned acc = taddr + ((kc - kc0) * 2 + m) * 3 * NO;
          const uint64_t a0 = a00 + (unsigned)(s * (T::ABYTES >> 4)), b0 = b00 + (unsigned)(d * (T::GBYTES >> 4));
          static_for<0, DROWS>([&](auto row_c) {
            constexpr int r = decltype(row_c)::value, slot = r / RT * PR + r % RT;
#pragma unroll
            for (int ks = 0; ks < W / 16; ks++)
              tc_mma(acc, a0 + (unsigned)((slot * W * 32 + ks * 512) >> 4), b0 + (unsigned)((r * ROWB + ks * 256) >> 4),
                     IDESC, it > 0 || r > 0 || ks > 0);
          });
          tc_commit(empty + s);
          if (++s == NS) {
            s = 0;
            phase++;
          }
        }
        tc_commit(gempty + d);
      }
      tc_commit(done);
    }
  } else {
    // the output gradient: thread t takes channel group t % CG of every (256 / CG)-th voxel
    const int cg = t % CG, v0 = t / CG;
    float db[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, it++) {
      const int d = it & 1;
      if (it >= 2) wait(gempty + d, (it >> 1) - 1);
      const int yt = tile % nyt, zt = (tile / nyt) % nzt, n = tile / (nyt * nzt);
      constexpr int VP = 256 / CG, ITER = (DROWS * W + VP - 1) / VP, BATCH = ITER < 4 ? ITER : 4;
#pragma unroll
      for (int i0 = 0; i0 < ITER; i0 += BATCH) {
        float4 f[BATCH][2];
#pragma unroll
        for (int b = 0; b < BATCH; b++) {
          const int v = (i0 + b) * VP + v0, r = v / W, x = v % W, z = zt * TZ + r / RT, y = yt * RT + r % RT;
          f[b][0] = f[b][1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (i0 + b < ITER && v < DROWS * W && z < D && y < H) {
            const float4* g = reinterpret_cast<const float4*>(dout + ((((long long)n * D + z) * H + y) * W + x) * NO + cg * 8);
            f[b][0] = g[0];
            f[b][1] = g[1];
          }
        }
#pragma unroll
        for (int b = 0; b < BATCH; b++) {
          const int v = (i0 + b) * VP + v0, r = v / W, x = v % W;
          if (i0 + b >= ITER || v >= DROWS * W) continue;
          const float4 f0 = f[b][0], f1 = f[b][1];
          db[0] += f0.x, db[1] += f0.y, db[2] += f0.z, db[3] += f0.w;
          db[4] += f1.x, db[5] += f1.y, db[6] += f1.z, db[7] += f1.w;
          const uint4 pk = make_uint4(pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w));
          unsigned char* g = Gs + d * T::GBYTES + r * ROWB + cg * W * 16;  // copy c holds the value of x + 1 - c at x
          constexpr int CP = CG * W * 16;
          *reinterpret_cast<uint4*>(g + CP + x * 16) = pk;
          if (x >= 1) *reinterpret_cast<uint4*>(g + (x - 1) * 16) = pk;
          if (x + 1 < W) *reinterpret_cast<uint4*>(g + 2 * CP + (x + 1) * 16) = pk;
          if (x == 0) *reinterpret_cast<uint4*>(g + 2 * CP) = make_uint4(0u, 0u, 0u, 0u);
          if (x == W - 1) *reinterpret_cast<uint4*>(g + (W - 1) * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
      }
      fence_proxy_async_smem();  // written through the generic proxy, read by the tensor core
      mbar_arrive(gfull + d);
    }
    const long long per = 27LL * Cin * NO, stride = per + NO;
    float* pb = part + (long long)blockIdx.x * stride;
    if (blockIdx.y == 0) {  // bias sums of the threads with the same channel group, in order
#pragma unroll
      for (int i = 0; i < 8; i++) dbs[t * 8 + i] = db[i];
      bar_named(1, 256);
      if (t < NO) {
        float a = 0.0f;
        for (int k = t / 8; k < 256; k += CG) a += dbs[k * 8 + t % 8];
        pb[per + t] = a;
      }
    }
    wait(done, 0);
    __syncwarp();
    tc_fence_after();
    // lane (16 g + ci) of M tile m: row group j = 8 m + g = dz PR + dy
    const int mrow = (warp & 3) * 32 + lane, ci = mrow & 15;
    for (int q = warp >> 2; q < 2 * (kc1 - kc0); q += 2) {
      const int kc = kc0 + (q >> 1), j = 8 * (q & 1) + (mrow >> 4), dz = j / PR, dy = j % PR;
      const bool used = dz < 3 && dy < 3;
#pragma unroll 1
      for (int c0 = 0; c0 < 3 * NO; c0 += 16) {
        float r[16];
        tc_ld16(taddr + ((unsigned)((warp & 3) * 32) << 16) + q * 3 * NO + c0, r);
        tc_wait_ld();
        if (used) {
          float4* o = reinterpret_cast<float4*>(
              pb + ((long long)(dz * 9 + dy * 3 + c0 / NO) * Cin + kc * 16 + ci) * NO + c0 % NO);
#pragma unroll
          for (int i = 0; i < 4; i++) o[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        }
        __syncwarp();
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(taddr, 512);
  }
}

// dW (n values) and db (C values) = the block partials part[nblk][n + C]: 8 threads per value add
// every eighth partial, and the eight sums are added in order (one thread per value and 152
// loads in turn took 16 us for 48 -> 16 channels, beside 25 us for a bias gradient of its own)
__global__ void __launch_bounds__(256) k_dw_finish(const float* part, int nblk, long long n, int C, float* dW, float* db) {
  __shared__ float red[8][32];
  const int x = threadIdx.x & 31, r = threadIdx.x >> 5;
  const long long i = blockIdx.x * 32LL + x, stride = n + C;
  float s = 0.0f;
  if (i < stride)
    for (int b = r; b < nblk; b += 8) s += part[b * stride + i];
  red[r][x] = s;
  __syncthreads();
  if (r == 0 && i < stride) {
    for (int k = 1; k < 8; k++) s += red[k][x];
    if (i < n) dW[i] = s;
    else db[i - n] = s;
  }
}

template <int W, int NO, int RMAX>
int launch_dw_rows_of(const bf16* in, const float* dout, float* dW, float* db, float* work, long long work_floats, int Nb,
                   int D, int H, int Cin, cudaStream_t s) {
  using T = DwRows<W, NO, RMAX>;
  const long long n = 27LL * Cin * NO;
  const int skip = (int)(-(intptr_t)(reinterpret_cast<uintptr_t>(work) >> 2) & 3);  // partials from a 16-byte boundary
  work += skip;
  work_floats -= skip;
  const long long tiles = (long long)Nb * ((D + T::TZ - 1) / T::TZ) * ((H + T::RT - 1) / T::RT);
  const int groups = ((Cin >> 4) + T::GROUP - 1) / T::GROUP;
  long long nblk = sm_count();  // as many partials as SMs, and no more than work holds
  if (nblk > tiles) nblk = tiles;
  if (nblk > work_floats / (n + NO)) nblk = work_floats / (n + NO);
  if (nblk < 1 || tiles > 0x7fffffffLL) return -1;
  CUtensorMap rows;
  const cuuint64_t dims[5] = {(cuuint64_t)Cin, W, (cuuint64_t)H, (cuuint64_t)D, (cuuint64_t)Nb};
  const cuuint64_t pitch[4] = {2ull * Cin, 2ull * Cin * W, 2ull * Cin * W * H, 2ull * Cin * W * H * D};
  const cuuint32_t box[5] = {16, W, T::PR, T::TZ + 2, 1}, step[5] = {1, 1, 1, 1, 1};
  tmk::EncodeTiledFn fn = tmk::encoder();
  if (!fn || fn(&rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16*>(in), dims, pitch, box, step,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return kNoMap;
  if (!tmk::allow_smem<k_conv_dw_rows<W, NO, RMAX>>(T::SMEM)) return -4;
  k_conv_dw_rows<W, NO, RMAX><<<dim3((unsigned)nblk, groups), T::THREADS, T::SMEM, s>>>(rows, dout, work, Nb, D, H, Cin);
  k_dw_finish<<<(unsigned)((n + NO + 31) / 32), 256, 0, s>>>(work, (int)nblk, n, NO, dW, db);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -4;
}

// Tiles of at most eight rows, or of two where there are at most 16 of the large ones, or where
// the scratch holds fewer partials than SMs: one accumulator then adds up no more voxels than it
// has to. 8 x 8 x 64, 16 -> 16 channels: eight tiles of 512 voxels, 1.6e-7 relative error and 12.7
// us; 32 of 128, 0.8e-7 and 10.4. 16 x 16 x 64, 96 -> 32: 64 tiles of 256, 1.2e-7 and 29 us, 128 of
// 128, 1.1e-7 and 36 us.
template <int W, int NO>
int launch_dw_rows(const bf16* in, const float* dout, float* dW, float* db, float* work, long long work_floats, int Nb,
                   int D, int H, int Cin, cudaStream_t s) {
  using T = DwRows<W, NO, 8>;
  if constexpr (T::DROWS > 2) {
    const long long tiles = (long long)Nb * ((D + T::TZ - 1) / T::TZ) * ((H + T::RT - 1) / T::RT);
    if (tiles <= 16 || work_floats / (27LL * Cin * NO + NO) < sm_count())
      return launch_dw_rows_of<W, NO, 2>(in, dout, dW, db, work, work_floats, Nb, D, H, Cin, s);
  }
  return launch_dw_rows_of<W, NO, 8>(in, dout, dW, db, work, work_floats, Nb, D, H, Cin, s);
}

// Weight gradient for rows of 8 voxels (half of a K = 16 step, which k_conv_dw_rows could not
// cut from its rows): dW[tap][ci][co] =
// sum_v in[v + off(tap)][ci] q(dout[v][co]) as MMAs with M = co (padded to 128), N = the
// 16 input channels of a chunk for the three dx taps at once (48), K = 16 voxels. A
// persistent block takes tiles of one plane x 128 / W rows (128 voxels): it stages the three
// planes of rows around the tile once, in the forward's three dx-shifted copies, whose
// channel halves and dx copies lie one box apart -- the uniform stride the N side needs --
// and the tile's output gradient, rounded to bfloat16, as [8 co][voxel] rows. Each of the
// nine (dz, dy) pairs then has one accumulator of 48 tensor-memory columns (432 in all),
// fed by 8 MMAs per tile from four issuing threads. After the block's tiles of a channel
// chunk its accumulators go out as one float32 partial per block; k_dw_reduce_halo adds the
// partials in block order. Same products as k_conv_dw_tc, float32 sums in another order.
template <int W>
struct DwHalo {
  static constexpr int RY = 128 / W, NV = 128, ROWS = 3 * (RY + 2);
  static constexpr int BOX = 16 * W * ROWS, ABYTES = 6 * BOX, GBYTES = 16 * NV * 16;
};
template <int W>
constexpr size_t dw_halo_smem() {
  return 128 + (size_t)DwHalo<W>::ABYTES + DwHalo<W>::GBYTES + 2 * 8 + 16;
}
template <int W, int NO>
__global__ void __launch_bounds__(128, 1) k_conv_dw_halo(const bf16* in, const float* dout, float* part, int Nb,
                                                         int D, int H, int Cin) {
  using namespace tmk;
  using HT = DwHalo<W>;
  constexpr int RY = HT::RY, NV = HT::NV, ROWS = HT::ROWS, BOX = HT::BOX;
  constexpr unsigned NCOLS = 512, IDESC = idesc_bf16(128, 48, true);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* As = smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127);  // [copy][half][plane][y][x][16 B]
  unsigned char* Gs = As + HT::ABYTES;                                         // [16 co groups][NV][16 B]
  unsigned long long* mma_bar = reinterpret_cast<unsigned long long*>(Gs + HT::GBYTES);
  unsigned* tslot = reinterpret_cast<unsigned*>(mma_bar + 1);
  const int t = threadIdx.x, warp = t >> 5;
  for (int i = t; i < (16 - NO / 8) * NV; i += 128)  // co >= NO: zero rows of A, never written again
    *reinterpret_cast<uint4*>(Gs + (NO / 8) * NV * 16 + i * 16) = make_uint4(0u, 0u, 0u, 0u);
  if (t == 0) {
    mbar_init(mma_bar, 4);  // one commit per issuer
    mbar_init_fence();
  }
  if (warp == 0) {
    tmem_alloc(tslot, NCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned taddr = *tslot;
  bool dead = false;
  auto wait = [&](unsigned long long* mb, unsigned parity) {
    if (!dead) dead = !mbar_wait_limit(mb, parity, 1 << 16, &g_net_status);
  };
  const int nyt = (H + RY - 1) / RY;
  const long long ntiles = (long long)Nb * D * nyt;
  const int nk = Cin >> 4;
  unsigned phase = 0;  // completed phases of mma_bar
  for (int kc = 0; kc < nk; kc++) {
    bool first = true;  // the block's first tile of this chunk starts the accumulators
    for (long long q = blockIdx.x; q < ntiles; q += gridDim.x) {
      const int yt = (int)(q % nyt);
      const long long rq = q / nyt;
      const int z = (int)(rq % D), n = (int)(rq / D), y0 = yt * RY;
      if (!first) {  // the previous tile's MMAs have read the staged rows
        wait(mma_bar, phase & 1);
        phase++;
      }
      if (t == 0 && kc == 0 && first) fence_proxy_async_global();  // in and dout came by ordinary stores
      stage_halo_issue<W, RY + 2, ROWS>(As, in, n, z, y0, D, H, Cin, kc * 16);  // in flight meanwhile
      // the tile's output gradient: voxel v = ty W + x, co group cg; zero outside the grid
      {
        constexpr int GI = NV * (NO / 8);
        for (int i = t; i < GI; i += 128) {
          const int v = i % NV, cg = i / NV, y = y0 + v / W;
          uint4 pk = make_uint4(0u, 0u, 0u, 0u);
          if (y < H) {
            const float4* g = reinterpret_cast<const float4*>(
                dout + ((((long long)n * D + z) * H + y) * W + v % W) * NO + cg * 8);
            const float4 f0 = g[0], f1 = g[1];
            pk = make_uint4(pack2(f0.x, f0.y), pack2(f0.z, f0.w), pack2(f1.x, f1.y), pack2(f1.z, f1.w));
          }
          *reinterpret_cast<uint4*>(Gs + cg * NV * 16 + v * 16) = pk;
        }
      }
      stage_halo_finish<W, ROWS>(As);
      fence_proxy_async_smem();  // the staged rows, written through the generic proxy, for the tensor core
      __syncthreads();
      if ((t & 31) == 0) {
        // issuer w: the (dz, dy) pairs w, w + 4, w + 8 (nine over four issuers)
        tc_fence_after();
        const uint64_t a0 = smem_desc(Gs, 128, NV * 16);  // K groups (8 voxels) 128 B, M groups (8 co) NV 16 B
        const uint64_t b0 = smem_desc(As, 128, BOX);      // K groups 128 B, N groups (half, then dx) one box
        for (int p = warp; p < 9; p += 4) {
          const int dz = p / 3 - 1, dy = p % 3 - 1;
#pragma unroll
          for (int ks = 0; ks < NV / 16; ks++) {
            const int v0 = ks * 16, ty = v0 / W, x0 = v0 % W;
            const unsigned boff = (unsigned)((((dz + 1) * (RY + 2) + ty + dy + 1) * W + x0) * 16) >> 4;
            tc_mma(taddr + p * 48, a0 + (unsigned)(v0 * 16 >> 4), b0 + boff, IDESC, !(first && ks == 0));
          }
        }
        tc_commit(mma_bar);
      }
      first = false;
    }
    if (!first) {
      wait(mma_bar, phase & 1);
      phase++;
    }
    tc_fence_after();
    // the chunk's partial: lane co of warp co / 32 holds D[co][dx 16 + ci] of pair p
    float* pb = part + (long long)blockIdx.x * 27 * Cin * NO;
    if (warp * 32 < NO) {
      const int co = t;
#pragma unroll 1
      for (int p = 0; p < 9; p++) {
#pragma unroll
        for (int dxi = 0; dxi < 3; dxi++) {
          float r[16];
          tc_ld16(taddr + ((unsigned)(warp * 32) << 16) + p * 48 + dxi * 16, r);
          tc_wait_ld();
          const int tap = p * 3 + dxi;  // (dz + 1) 9 + (dy + 1) 3 + (dx + 1)
          if (co < NO) {
#pragma unroll
            for (int i = 0; i < 16; i++) pb[((long long)tap * Cin + kc * 16 + i) * NO + co] = first ? 0.0f : r[i];
          }
        }
      }
    }
    tc_fence_before();
    __syncthreads();  // the accumulators are read before the next chunk's MMAs overwrite them
    tc_fence_after();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(taddr, NCOLS);
}

// dW = sum over the blocks p (in order) of part[p][tap][ci][co]
__global__ void k_dw_reduce_halo(const float* part, int nblk, long long n, float* dW) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    float s = 0.0f;
    for (int b = 0; b < nblk; b++) s += part[(long long)b * n + i];
    dW[i] = s;
  }
}

// dW[tap][ci][co] = sum over the voxel blocks p (in order) of part[p][tile][row][co]
__global__ void k_dw_reduce_tc(const float* part, int nblk, int ntiles, int Cin, int Cout, float* dW) {
  const long long n = 27LL * Cin * Cout;
  const int ncc = Cin >> 4;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int tap = (int)(i / ((long long)Cin * Cout));
    const int r = (int)(i - (long long)tap * Cin * Cout), ci = r / Cout, co = r - ci * Cout;
    const int tile = (tap >> 3) * ncc + (ci >> 4), row = (tap & 7) * 16 + (ci & 15);
    float s = 0.0f;
    for (int b = 0; b < nblk; b++) s += part[(((long long)b * ntiles + tile) * 128 + row) * Cout + co];
    dW[i] = s;
  }
}

// bfloat16 copy of a float32 array (round to nearest even), two values per thread step
__global__ void k_to_bf16(const float* x, bf16* y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; 2 * i < n; i += (long long)gridDim.x * blockDim.x) {
    if (2 * i + 1 < n) {
      *reinterpret_cast<uint32_t*>(y + 2 * i) = pack2(x[2 * i], x[2 * i + 1]);
    } else {
      y[2 * i] = __float2bfloat16(x[2 * i]);
    }
  }
}

// The bias gradient db[c] = sum over the voxels of dout[v][c] (float32, unrounded), in a
// fixed order: block b sums its range of voxels for every channel (consecutive threads on
// consecutive channels, then voxels), k_db_final adds the block partials in block order.
constexpr int kDbBlocks = 256;
__global__ void __launch_bounds__(256) k_db_part(const float* dout, long long nvox, int C, float* part) {
  __shared__ float red[256];
  const int t = threadIdx.x, c = t % C, lane = t / C, lanes = 256 / C;
  const long long chunk = (nvox + gridDim.x - 1) / gridDim.x;
  const long long v0 = blockIdx.x * chunk, v1 = v0 + chunk < nvox ? v0 + chunk : nvox;
  float s = 0.0f;
  for (long long v = v0 + lane; v < v1; v += lanes) s += dout[v * C + c];
  red[t] = s;
  __syncthreads();
  if (t < C) {
    float a = 0.0f;
    for (int l = 0; l < lanes; l++) a += red[l * C + t];
    part[(long long)blockIdx.x * C + t] = a;
  }
}
__global__ void k_db_final(const float* part, int nblk, int C, float* db) {
  if ((int)threadIdx.x < C) {
    float a = 0.0f;
    for (int b = 0; b < nblk; b++) a += part[(long long)b * C + threadIdx.x];
    db[threadIdx.x] = a;
  }
}
// after the weight gradient's partials are consumed, work holds the bias partials
int launch_db(const float* dout, long long nvox, int C, float* work, float* db, cudaStream_t s) {
  const int nb = (int)(nvox < kDbBlocks ? nvox : kDbBlocks);
  k_db_part<<<nb, 256, 0, s>>>(dout, nvox, C, work);
  k_db_final<<<1, 64, 0, s>>>(work, nb, C, db);
  return 0;
}

// g *= (act > 0): ReLU backward through the stored bfloat16 activation
__global__ void k_relu_bwd(float* g, const bf16* act, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    if (!(__bfloat162float(act[i]) > 0.0f)) g[i] = 0.0f;
}

// 2x2x2 average pooling and its adjoint
__global__ void k_pool(const bf16* in, bf16* out, int N, int D, int H, int W, int C) {
  const long long n = (long long)N * (D / 2) * (H / 2) * (W / 2) * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const Vox q = vox_of(i / C, D / 2, H / 2, W / 2);
    float s = 0.0f;
    for (int a = 0; a < 8; a++) {
      const int z = 2 * q.z + (a >> 2), y = 2 * q.y + ((a >> 1) & 1), x = 2 * q.x + (a & 1);
      s += __bfloat162float(in[((((long long)q.n * D + z) * H + y) * W + x) * C + c]);
    }
    out[i] = __float2bfloat16(0.125f * s);
  }
}
__global__ void k_pool_bwd(const float* gout, float* gin, int N, int D, int H, int W, int C, int accumulate) {
  const long long n = (long long)N * D * H * W * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const Vox q = vox_of(i / C, D, H, W);
    const float v =
        0.125f * gout[((((long long)q.n * (D / 2) + q.z / 2) * (H / 2) + q.y / 2) * (W / 2) + q.x / 2) * C + c];
    gin[i] = accumulate ? gin[i] + v : v;
  }
}

// out = [nearest-upsample(x) (C1 channels) | skip (C2 channels)] at the fine grid, and its adjoint
__global__ void k_upcat(const bf16* x, const bf16* skip, bf16* out, int N, int D, int H, int W, int C1, int C2) {
  const int C = C1 + C2;
  const long long n = (long long)N * D * H * W * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const long long v = i / C;
    if (c < C1) {
      const Vox q = vox_of(v, D, H, W);
      out[i] = x[((((long long)q.n * (D / 2) + q.z / 2) * (H / 2) + q.y / 2) * (W / 2) + q.x / 2) * C1 + c];
    } else {
      out[i] = skip[v * C2 + (c - C1)];
    }
  }
}
__global__ void k_upcat_bwd_x(const float* gout, float* gx, int N, int D, int H, int W, int C1, int C2) {
  // gx at the coarse grid: sum over the 8 fine children
  const int C = C1 + C2;
  const long long n = (long long)N * (D / 2) * (H / 2) * (W / 2) * C1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C1);
    const Vox q = vox_of(i / C1, D / 2, H / 2, W / 2);
    float s = 0.0f;
    for (int a = 0; a < 8; a++) {
      const int z = 2 * q.z + (a >> 2), y = 2 * q.y + ((a >> 1) & 1), x = 2 * q.x + (a & 1);
      s += gout[((((long long)q.n * D + z) * H + y) * W + x) * C + c];
    }
    gx[i] = s;
  }
}
__global__ void k_upcat_bwd_skip(const float* gout, float* gskip, long long nvox, int C1, int C2) {
  const long long n = nvox * C2;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long v = i / C2;
    gskip[i] = gout[v * (C1 + C2) + C1 + (i - v * C2)];
  }
}

// head: rho0 = sigmoid(sum_c w[c] x[c] + b); loss = mean (rho0 - target)^2 and its gradients
__global__ void k_head(const bf16* x, const float* w, const float* b, float* rho, long long nvox, int C) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nvox; v += (long long)gridDim.x * blockDim.x) {
    float s = b[0];
    for (int c = 0; c < C; c++) s += w[c] * __bfloat162float(x[v * C + c]);
    rho[v] = 1.0f / (1.0f + expf(-s));
  }
}
__global__ void k_head_bwd(const bf16* x, const float* w, const float* rho, const float* target, long long nvox, int C,
                           float* gx, float* part /* [gridDim.x][C + 2]: dw, db, loss */) {
  extern __shared__ float red[];  // [blockDim.x][C + 2]
  float loc[68];
  for (int c = 0; c < C + 2; c++) loc[c] = 0.0f;
  const float inv = 1.0f / (float)nvox;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nvox; v += (long long)gridDim.x * blockDim.x) {
    const float r = rho[v], d = r - target[v];
    const float dz = 2.0f * d * r * (1.0f - r) * inv;
    for (int c = 0; c < C; c++) {
      gx[v * C + c] = dz * w[c];
      loc[c] += dz * __bfloat162float(x[v * C + c]);
    }
    loc[C] += dz;
    loc[C + 1] += d * d * inv;
  }
  for (int c = 0; c < C + 2; c++) red[threadIdx.x * (C + 2) + c] = loc[c];
  __syncthreads();
  if (threadIdx.x < C + 2) {
    float s = 0.0f;
    for (int i = 0; i < (int)blockDim.x; i++) s += red[i * (C + 2) + threadIdx.x];
    part[blockIdx.x * (C + 2) + threadIdx.x] = s;
  }
}
__global__ void k_head_reduce(const float* part, int nblk, int n, float* out) {
  const int i = threadIdx.x;
  if (i < n) {
    float s = 0.0f;
    for (int b = 0; b < nblk; b++) s += part[b * n + i];
    out[i] = s;
  }
}

// AdamW on float32 master weights; optional bfloat16 copies in the two conv layouts
__global__ void k_adamw(float* w, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                        float eps, float wd, float c1, float c2, bf16* wf, bf16* wb, int cin, int cout) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    float wi = w[i];
    wi -= lr * ((mi / c1) / (sqrtf(vi / c2) + eps) + wd * wi);
    w[i] = wi;
    if (wf) {  // i = (tap, ci, co)
      const int tap = (int)(i / ((long long)cin * cout));
      const int r = (int)(i - (long long)tap * cin * cout), ci = r / cout, co = r - ci * cout;
      wf[pack_f(tap, ci, co, cin, cout)] = __float2bfloat16(wi);
      wb[pack_b(tap, ci, co, cin, cout)] = __float2bfloat16(wi);
    }
  }
}

// bfloat16 copies of float32 master conv weights [27][cin][cout]
__global__ void k_pack_w(const float* w, bf16* wf, bf16* wb, int cin, int cout) {
  const long long n = 27LL * cin * cout;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int tap = (int)(i / ((long long)cin * cout));
    const int r = (int)(i - (long long)tap * cin * cout), ci = r / cout, co = r - ci * cout;
    wf[pack_f(tap, ci, co, cin, cout)] = __float2bfloat16(w[i]);
    wb[pack_b(tap, ci, co, cin, cout)] = __float2bfloat16(w[i]);
  }
}

// network input from a target specification on the 64^3 design grid:
// channel 0 mask footprint, 1 Ht_z / Ms on the footprint, 2 plane height / 8 (all z)
__global__ void k_spec_input(const uint8_t* foot /* [N][H][W] */, const float* ht /* [N] */, const float* hgt /* [N] */,
                             bf16* out, int N, int D, int H, int W, int C) {
  const long long n = (long long)N * D * H * W;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const Vox q = vox_of(v, D, H, W);
    const float f = foot[((long long)q.n * H + q.y) * W + q.x] ? 1.0f : 0.0f;
    for (int c = 0; c < C; c++) {
      float val = 0.0f;
      if (c == 0) val = f;
      if (c == 1) val = f * ht[q.n];
      if (c == 2) val = hgt[q.n];
      out[v * C + c] = __float2bfloat16(val);
    }
  }
}

int grid_of(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b > 16384 ? 16384 : (b < 1 ? 1 : b));
}

int ok() { return cudaPeekAtLastError() == cudaSuccess ? 0 : -4; }

}  // namespace

extern "C" {

int tmn_conv3d_forward(const void* in, const void* Wf, const float* bias, void* out, int N, int D, int H, int W,
                       int Cin, int Cout, int relu, void* stream) {
  if (!in || !Wf || !out || Cin % 16 || Cin < 16 || (Cout != 16 && Cout != 32 && Cout != 64)) return -1;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const bf16* w = reinterpret_cast<const bf16*>(Wf);
  if (Cout == 16) return launch_conv<0, 16>(in, w, bias, out, N, D, H, W, Cin, relu, s);
  if (Cout == 32) return launch_conv<0, 32>(in, w, bias, out, N, D, H, W, Cin, relu, s);
  return launch_conv<0, 64>(in, w, bias, out, N, D, H, W, Cin, relu, s);
}

int tmn_conv3d_backward_data(const float* dout, const void* Wb, float* din, int N, int D, int H, int W, int Cin,
                             int Cout, int accumulate, void* stream) {
  if (!dout || !Wb || !din || Cout % 16 || Cout < 16 || (Cin != 16 && Cin != 32 && Cin != 48 && Cin != 64 && Cin != 96))
    return -1;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const bf16* w = reinterpret_cast<const bf16*>(Wb);
  // GEMM over k = (tap, co) with the output channels ci as the N side
  if (Cin == 16) return launch_conv<1, 16>(dout, w, nullptr, din, N, D, H, W, Cout, accumulate, s);
  if (Cin == 32) return launch_conv<1, 32>(dout, w, nullptr, din, N, D, H, W, Cout, accumulate, s);
  if (Cin == 48) return launch_conv<1, 48>(dout, w, nullptr, din, N, D, H, W, Cout, accumulate, s);
  if (Cin == 64) return launch_conv<1, 64>(dout, w, nullptr, din, N, D, H, W, Cout, accumulate, s);
  return launch_conv<1, 96>(dout, w, nullptr, din, N, D, H, W, Cout, accumulate, s);
}

int tmn_status(unsigned* out) {
  if (!out) return -1;
  unsigned z = 0;
  if (cudaMemcpyFromSymbol(out, g_net_status, sizeof(unsigned)) != cudaSuccess) return -4;
  if (cudaMemcpyToSymbol(g_net_status, &z, sizeof(unsigned)) != cudaSuccess) return -4;
  return 0;
}

long long tmn_conv3d_backward_weight_work(long long nvox, int Cin, int Cout) {
  if (nvox < 1 || Cin < 16 || Cin % 16 || Cout < 16 || Cout % 16) return -1;
  const long long copy = (nvox * Cout + 1) / 2;         // floats holding the bfloat16 copy of dout
  return (copy + 3) / 4 * 4 + 4LL * (Cin / 16) * 128 * Cout;  // partials from a 16-byte boundary, one set
}

int tmn_conv3d_backward_weight(const void* in, const float* dout, float* dW, float* db, float* work,
                               long long work_floats, int N, int D, int H, int W, int Cin, int Cout, void* stream) {
  if (!in || !dout || !dW || !db || !work || Cin % 16 || Cin < 16 || (Cout != 16 && Cout != 32 && Cout != 64))
    return -1;
  const long long nvox = (long long)N * D * H * W;
  if (nvox < 1) return -1;
  if (work_floats < tmn_conv3d_backward_weight_work(nvox, Cin, Cout)) return -5;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int nsm = sm_count();
  if ((reinterpret_cast<uintptr_t>(in) & 15) == 0) {
    const bf16* x = reinterpret_cast<const bf16*>(in);
    int r = kNoMap;
#define TMN_DW_ROWS(WW)                                                                                      \
  if (W == WW) {                                                                                             \
    if (Cout == 16) r = launch_dw_rows<WW, 16>(x, dout, dW, db, work, work_floats, N, D, H, Cin, s);          \
    else if (Cout == 32) r = launch_dw_rows<WW, 32>(x, dout, dW, db, work, work_floats, N, D, H, Cin, s);     \
    else r = launch_dw_rows<WW, 64>(x, dout, dW, db, work, work_floats, N, D, H, Cin, s);                     \
  }
    TMN_DW_ROWS(16)
    TMN_DW_ROWS(32)
    TMN_DW_ROWS(64)
#undef TMN_DW_ROWS
    if (r != kNoMap) return r;
  }
  if (W == 8 && (reinterpret_cast<uintptr_t>(in) & 15) == 0) {
    // halo tiles: one persistent block per SM, as many as the work buffer holds partials for
    const long long per = 27LL * Cin * Cout, ntl = (long long)N * D * ((H + 128 / W - 1) / (128 / W));
    long long nblk = work_floats / per;
    if (nblk > nsm) nblk = nsm;
    if (nblk > ntl) nblk = ntl;
    const bf16* x = reinterpret_cast<const bf16*>(in);
    int r = 0;
    auto run = [&](auto kernel, size_t sm) {
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
        r = -4;
      else
        kernel<<<(unsigned)nblk, 128, sm, s>>>(x, dout, work, N, D, H, Cin);
    };
#define TMN_DW_HALO(WW)                                                             \
  if (W == WW) {                                                                    \
    if (Cout == 16) run(k_conv_dw_halo<WW, 16>, dw_halo_smem<WW>());                \
    if (Cout == 32) run(k_conv_dw_halo<WW, 32>, dw_halo_smem<WW>());                \
    if (Cout == 64) run(k_conv_dw_halo<WW, 64>, dw_halo_smem<WW>());                \
  }
    TMN_DW_HALO(8)
#undef TMN_DW_HALO
    if (r) return r;
    k_dw_reduce_halo<<<grid_of(per), 256, 0, s>>>(work, (int)nblk, per, dW);
    launch_db(dout, nvox, Cout, work, db, s);
    return ok();
  }
  const long long pofs = ((nvox * Cout + 1) / 2 + 3) / 4 * 4;
  const int tiles = 4 * (Cin / 16);
  const long long per_blk = (long long)tiles * 128 * Cout;
  // voxel blocks: about four blocks per SM over all tiles (each block's loop is bound by the
  // latency of its gathers, so several of them in flight), no more than the work buffer holds
  const long long chunks = (nvox + 15) / 16;
  long long nblk = (work_floats - pofs) / per_blk;
  const long long want = ((long long)kDwBlocksPerSm * nsm + tiles - 1) / tiles;
  if (nblk > want) nblk = want;
  if (nblk > chunks) nblk = chunks;
  long long cpb = (chunks + nblk - 1) / nblk;
  if (cpb > kDwChunks) cpb = (cpb + kDwChunks - 1) / kDwChunks * kDwChunks;  // whole pipeline stages
  nblk = (chunks + cpb - 1) / cpb;
  bf16* g16 = reinterpret_cast<bf16*>(work);
  float* part = work + pofs;
  k_to_bf16<<<grid_of(nvox * Cout / 2 + 1), 256, 0, s>>>(dout, g16, nvox * Cout);
  const dim3 grid((unsigned)nblk, (unsigned)tiles);
  const bf16* x = reinterpret_cast<const bf16*>(in);
  int r = 0;
  auto run = [&](auto kernel, size_t sm) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess)
      r = -4;
    else
      kernel<<<grid, 128, sm, s>>>(x, g16, part, N, D, H, W, Cin, cpb);
  };
  if (Cout == 16) run(k_conv_dw_tc<16>, dw_tc_smem<16>());
  if (Cout == 32) run(k_conv_dw_tc<32>, dw_tc_smem<32>());
  if (Cout == 64) run(k_conv_dw_tc<64>, dw_tc_smem<64>());
  if (r) return r;
  k_dw_reduce_tc<<<grid_of(27LL * Cin * Cout), 256, 0, s>>>(part, (int)nblk, tiles, Cin, Cout, dW);
  launch_db(dout, nvox, Cout, work, db, s);
  return ok();
}

int tmn_relu_backward(float* g, const void* act, long long n, void* stream) {
  k_relu_bwd<<<grid_of(n), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(g, reinterpret_cast<const bf16*>(act), n);
  return ok();
}

int tmn_pool(const void* in, void* out, int N, int D, int H, int W, int C, void* stream) {
  k_pool<<<grid_of((long long)N * D * H * W * C / 8), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<const bf16*>(in), reinterpret_cast<bf16*>(out), N, D, H, W, C);
  return ok();
}

int tmn_pool_backward(const float* gout, float* gin, int N, int D, int H, int W, int C, int accumulate, void* stream) {
  k_pool_bwd<<<grid_of((long long)N * D * H * W * C), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      gout, gin, N, D, H, W, C, accumulate);
  return ok();
}

int tmn_upcat(const void* x, const void* skip, void* out, int N, int D, int H, int W, int C1, int C2, void* stream) {
  k_upcat<<<grid_of((long long)N * D * H * W * (C1 + C2)), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      reinterpret_cast<const bf16*>(x), reinterpret_cast<const bf16*>(skip), reinterpret_cast<bf16*>(out), N, D, H, W,
      C1, C2);
  return ok();
}

int tmn_upcat_backward(const float* gout, float* gx, float* gskip, int N, int D, int H, int W, int C1, int C2,
                       void* stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  k_upcat_bwd_x<<<grid_of((long long)N * D * H * W * C1 / 8), 256, 0, s>>>(gout, gx, N, D, H, W, C1, C2);
  k_upcat_bwd_skip<<<grid_of((long long)N * D * H * W * C2), 256, 0, s>>>(gout, gskip, (long long)N * D * H * W, C1,
                                                                        C2);
  return ok();
}

int tmn_head_forward(const void* x, const float* w, const float* b, float* rho, long long nvox, int C, void* stream) {
  k_head<<<grid_of(nvox), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(reinterpret_cast<const bf16*>(x), w, b,
                                                                             rho, nvox, C);
  return ok();
}

int tmn_head_backward(const void* x, const float* w, const float* rho, const float* target, long long nvox, int C,
                      float* gx, float* work, float* out, void* stream) {
  if (C + 2 > 68) return -1;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int nblk = 256;
  k_head_bwd<<<nblk, 128, 128 * (C + 2) * sizeof(float), s>>>(reinterpret_cast<const bf16*>(x), w, rho, target, nvox,
                                                              C, gx, work);
  k_head_reduce<<<1, 128, 0, s>>>(work, nblk, C + 2, out);
  return ok();
}

int tmn_adamw(float* w, const float* g, float* m, float* v, long long n, float lr, float b1, float b2, float eps,
              float wd, int step, void* wf, void* wb, int cin, int cout, void* stream) {
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adamw<<<grid_of(n), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      w, g, m, v, n, lr, b1, b2, eps, wd, c1, c2, reinterpret_cast<bf16*>(wf), reinterpret_cast<bf16*>(wb), cin, cout);
  return ok();
}

int tmn_pack_conv_weights(const float* w, void* wf, void* wb, int cin, int cout, void* stream) {
  if (!w || !wf || !wb || cin < 1 || cout < 1) return -1;
  k_pack_w<<<grid_of(27LL * cin * cout), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      w, reinterpret_cast<bf16*>(wf), reinterpret_cast<bf16*>(wb), cin, cout);
  return ok();
}

int tmn_spec_input(const uint8_t* foot, const float* ht, const float* hgt, void* out, int N, int D, int H, int W,
                   int C, void* stream) {
  k_spec_input<<<grid_of((long long)N * D * H * W), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      foot, ht, hgt, reinterpret_cast<bf16*>(out), N, D, H, W, C);
  return ok();
}

}  // extern "C"
