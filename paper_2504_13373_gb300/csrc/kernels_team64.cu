// FP64 block-sparse products and smoothing steps on levels with few scalar
// rows, where a thread per scalar row would leave the GPU short of warps.
//
// An SM does two FP64 FMAs a clock, a warp's instruction taking an SM quarter
// 64 clocks whether one lane is active or all, so these products are bound by
// the number of FP64 instructions.  The lanes of a warp therefore take a
// block's br * bc values side by side (lane l the values l, l + 32, ..., EPL of
// them), the same positions of every block, and keep one partial sum per
// position: every lane works on every block, the matrix is read in runs of 256
// bytes, and nothing is added up before the row's end.  A team of ES x BS warps
// owns a block row: ES share out a block's positions (at most 32 * 8 each), BS
// the blocks.  At the end the sums of a row's positions meet in shared memory;
// a few lanes add up a row in a fixed order, which depends only on the matrix
// and the team.  (A CTA per block row with a thread per row of a block, as
// before, spent half of its FP64 instructions on adding up 256 / br groups one
// after another.)
//
// Operations: y = A x, y = b - A x, y += A x for br x bc blocks up to 64 x 64,
// and the block-Jacobi step x_out = x + W (b - A x) (square blocks).
//
// GB300, Q2 128^2 V-cycle, FP64, levels of 4,096, 1,024 and 256 units (12 x 12,
// 16 x 16 and 21 x 21 blocks): these products took 1,084 us of the V-cycle and
// take 738 (smoothing steps 47.3 us on average before; now 35.6, 31.5 and 33.5).
#include <cooperative_groups.h>

#include "common.cuh"
#include "internal.h"

namespace gasa {

namespace cg = cooperative_groups;

namespace {

constexpr int kT64Values = 8;       // values of a block per lane at most
constexpr int kT64Warps = 8;        // warps per team in a CTA at most (16 for blocks beyond 2,048 values)
constexpr int kT64Cluster = 8;      // CTAs sharing a block row at most

template <int EPL>
__global__ void __launch_bounds__(512)
team64_kernel(int op, int n_brows, int br, int bc, int ES, int BS, int CS, int LPR,
              const int *__restrict__ rp,
              const int *__restrict__ col, const double *__restrict__ val,
              const double *__restrict__ Wm, const double *__restrict__ x,
              const double *__restrict__ b, double *__restrict__ y) {
  extern __shared__ double sm64[];
  __shared__ double gathered[kT64Cluster][64];     // rank 0: the CTAs' row sums
  const int rank = CS > 1 ? (int)cg::this_cluster().block_rank() : 0;
  if (CS > 1) cg::this_cluster().barrier_arrive();   // waited for before the first remote write
  const int nw = ES * BS, warps = blockDim.x >> 5, teams = warps / nw;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int team = warp / nw, wt = warp - team * nw;
  const int es = wt % ES, bs = wt / ES;
  const int u = CS > 1 ? (int)blockIdx.x / CS : (int)blockIdx.x * teams + team;
  const bool on = u < n_brows;
  const int E = br * bc, pitch = ES * EPL * 32;
  double *part = sm64 + (size_t)team * BS * pitch;              // [BS][positions]
  double *res = sm64 + (size_t)teams * BS * pitch + (size_t)team * br;
  double acc[EPL];
  int e[EPL], q[EPL];
#pragma unroll
  for (int m = 0; m < EPL; ++m) {
    // positions past the block's end repeat its last value; their sums are not used
    e[m] = min((es * EPL + m) * 32 + lane, E - 1);
    q[m] = e[m] % bc;
    acc[m] = 0.0;
  }
  if (on) {
    const int end = __ldg(rp + u + 1), step = BS * CS;
    int k = __ldg(rp + u) + rank * BS + bs;
    if constexpr (EPL <= 5) {
      // two blocks' values and entries of x in flight, in 64 registers: the next
      // blocks ahead as below take 92, and on rows of 9 blocks of 12 x 12 the warps
      // lost cost more than the loads' wait (smoothing step 34.5 -> 42 us)
      int j0 = k < end ? __ldg(col + k) : 0, j1 = k + step < end ? __ldg(col + k + step) : 0;
      for (; k + step < end; k += 2 * step) {
        const double *a0 = val + (size_t)k * E, *a1 = val + (size_t)(k + step) * E;
        const double *x0 = x + (size_t)j0 * bc, *x1 = x + (size_t)j1 * bc;
        double av0[EPL], av1[EPL], xv0[EPL], xv1[EPL];
#pragma unroll
        for (int m = 0; m < EPL; ++m) {
          av0[m] = __ldg(a0 + e[m]);
          av1[m] = __ldg(a1 + e[m]);
        }
#pragma unroll
        for (int m = 0; m < EPL; ++m) {
          xv0[m] = __ldg(x0 + q[m]);
          xv1[m] = __ldg(x1 + q[m]);
        }
        j0 = k + 2 * step < end ? __ldg(col + k + 2 * step) : 0;
        j1 = k + 3 * step < end ? __ldg(col + k + 3 * step) : 0;
#pragma unroll
        for (int m = 0; m < EPL; ++m) acc[m] = fma(av1[m], xv1[m], fma(av0[m], xv0[m], acc[m]));
      }
      if (k < end) {
        const double *a0 = val + (size_t)k * E, *x0 = x + (size_t)j0 * bc;
#pragma unroll
        for (int m = 0; m < EPL; ++m) acc[m] = fma(__ldg(a0 + e[m]), __ldg(x0 + q[m]), acc[m]);
      }
    } else {
      // one block's values and entries of x ahead of the one being multiplied, and
      // the column of the one after
      double av[EPL], xv[EPL];
      int j = k < end ? __ldg(col + k) : 0;
      if (k < end) {
        const double *a0 = val + (size_t)k * E, *x0 = x + (size_t)j * bc;
#pragma unroll
        for (int m = 0; m < EPL; ++m) av[m] = __ldg(a0 + e[m]);
#pragma unroll
        for (int m = 0; m < EPL; ++m) xv[m] = __ldg(x0 + q[m]);
        j = k + step < end ? __ldg(col + k + step) : 0;
      }
#pragma unroll 1
      for (; k < end; k += step) {
        double an[EPL], xn[EPL];
        const bool more = k + step < end;
        if (more) {
          const double *a1 = val + (size_t)(k + step) * E, *x1 = x + (size_t)j * bc;
#pragma unroll
          for (int m = 0; m < EPL; ++m) an[m] = __ldg(a1 + e[m]);
#pragma unroll
          for (int m = 0; m < EPL; ++m) xn[m] = __ldg(x1 + q[m]);
          j = k + 2 * step < end ? __ldg(col + k + 2 * step) : 0;
        }
#pragma unroll
        for (int m = 0; m < EPL; ++m) acc[m] = fma(av[m], xv[m], acc[m]);
        if (more) {
#pragma unroll
          for (int m = 0; m < EPL; ++m) {
            av[m] = an[m];
            xv[m] = xn[m];
          }
        }
      }
    }
  }
#pragma unroll
  for (int m = 0; m < EPL; ++m) part[(size_t)bs * pitch + (es * EPL + m) * 32 + lane] = acc[m];
  __syncthreads();
  if (CS > 1) cg::this_cluster().barrier_wait();     // every CTA of the cluster runs
  auto finish_row = [&](int r, double v) {
    const size_t t = (size_t)u * br + r;
    if (op == 0) y[t] = v;
    else if (op == 1) y[t] = b[t] - v;
    else if (op == 2) y[t] = y[t] + v;
    else res[r] = b[t] - v;
  };
  // LPR lanes per row: the warps' sums in order, columns sub, sub + LPR, ... in
  // order, then a tree over the lanes; warps without a row skip it
  const int sub = lane & (LPR - 1);
  for (int t0 = wt * 32; t0 < br * LPR; t0 += nw * 32) {
    const int r = (t0 + lane) / LPR;
    double v = 0.0;
    if (r < br)
      for (int s = 0; s < BS; ++s)
        for (int c = sub; c < bc; c += LPR) v += part[(size_t)s * pitch + r * bc + c];
    for (int o = LPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (on && r < br && sub == 0) {
      if (CS == 1) finish_row(r, v);
      else cg::this_cluster().map_shared_rank(&gathered[0][0], 0)[rank * 64 + r] = v;
    }
  }
  if (CS > 1) {
    cg::this_cluster().sync();
    if (rank != 0) return;
    for (int r = wt * 32 + lane; on && r < br; r += nw * 32) {
      double v = 0.0;
      for (int c = 0; c < CS; ++c) v += gathered[c][r];
      finish_row(r, v);
    }
  }
  if (op != 3) return;
  __syncthreads();
  for (int t0 = wt * 32; t0 < br * LPR; t0 += nw * 32) {
    const int r = (t0 + lane) / LPR;
    double v = 0.0;
    if (on && r < br) {
      const double *w = Wm + ((size_t)u * br + r) * br;
      for (int c = sub; c < br; c += LPR) v = fma(__ldg(w + c), res[c], v);
    }
    for (int o = LPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (on && r < br && sub == 0) {
      const size_t t = (size_t)u * br + r;
      y[t] = x[t] + v;
    }
  }
}

}  // namespace

// Warps over a block's positions (ES), over a row's blocks (BS) and CTAs over a row (CS),
// and the values per lane (EPL).
void team64_split(int n_brows, int br, int bc, int64_t nnzb, int *es, int *epl, int *bs, int *cs) {
  const int per = div_up(br * bc, 32);
  const int ES = div_up(per, kT64Values), EPL = div_up(per, ES);
  const double avg = nnzb >= 0 ? (double)nnzb / (double)n_brows : 1e9;
  // Blocks shared out over warps while each keeps eight or more and the GPU has fewer
  // than 16 warps an SM; beyond that down to one or two blocks a warp as long as the
  // GPU stays within 16 warps an SM, where a warp's own chain of blocks is all there is
  // (smoothing step, GB300, 256 rows of 17 blocks of 12 x 12: two warps 9.3 us, eight
  // 6.5; 256 rows of 27 blocks of 16 x 16: 12.5 and 9.9, four 9.5; 384 rows of 4 blocks
  // of 10 x 10: one 6.7, four 5.2).  Twice as many at 16 an SM cost more in the teams'
  // sums than they hide (1,024 rows of 17 of 12 x 12: 11.4, four 11.8).
  const long long most = 16LL * kNumSM;
  int BS = 1;
  while (ES * BS * 2 <= kT64Warps &&
         ((avg >= 16.0 * BS && (long long)n_brows * ES * BS < most) ||
          (avg >= 2.0 * BS && (long long)n_brows * ES * BS * 2 <= most)))
    BS *= 2;
  if (nnzb < 0 && BS > 4) BS = 4;
  // few long rows: a cluster of CTAs per block row, each with a share of its
  // blocks, while that keeps the GPU within 24 warps an SM and every warp eight
  // blocks; rank 0 adds up the CTAs' sums and finishes the row (64 rows of 200
  // blocks of 28 x 21: 122.8 -> 34.1 us)
  int CS = 1;
  while (nnzb >= 0 && CS < kT64Cluster && avg >= 16.0 * BS * CS &&
         (long long)n_brows * ES * BS * CS * 2 <= 24LL * kNumSM)
    CS *= 2;
  *es = ES;
  *epl = EPL;
  *bs = BS;
  *cs = CS;
}

cudaError_t launch_team64(int op, int n_brows, int br, int bc, int64_t nnzb, const int *rp,
                          const int *col, const double *val, const double *W, const double *x,
                          const double *b, double *y, cudaStream_t s) {
  if (n_brows == 0) return cudaSuccess;
  if (br > 64 || bc > 64 || (op == 3 && br != bc)) return cudaErrorNotSupported;
  int ES, EPL, BS, CS;
  team64_split(n_brows, br, bc, nnzb, &ES, &EPL, &BS, &CS);
  const int nw = ES * BS, teams = CS > 1 || nw >= 4 ? 1 : 4 / nw, warps = nw * teams;
  // lanes that add up a row: two where one warp does it (fewest instructions), up
  // to sixteen where the team's warps share them (shortest chain)
  int LPR = 2;
  while (LPR < 16 && br * LPR * 2 <= nw * 32) LPR *= 2;
  const size_t smem = ((size_t)warps * 32 * EPL + (size_t)teams * br) * sizeof(double);
  auto go = [&](auto kern) {
    launch_kc(kern, CS * div_up(n_brows, teams), 32 * warps, smem, s, CS, op, n_brows, br, bc, ES, BS,
              CS, LPR, rp, col, val, W, x, b, y);
  };
  switch (EPL) {
    case 1: go(team64_kernel<1>); break;
    case 2: go(team64_kernel<2>); break;
    case 3: go(team64_kernel<3>); break;
    case 4: go(team64_kernel<4>); break;
    case 5: go(team64_kernel<5>); break;
    case 6: go(team64_kernel<6>); break;
    case 7: go(team64_kernel<7>); break;
    default: go(team64_kernel<8>); break;
  }
  note_launch();
  return cudaGetLastError();
}

}  // namespace gasa
