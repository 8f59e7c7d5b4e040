// Coarse-level block-sparse products with wide blocks (more than 8 rows or
// columns) in FP32.
//
// The Galerkin operators below level 0 of the 3-D and convection-diffusion
// workloads have blocks of 12 to 36 rows and tens to hundreds of blocks per
// block row, and at these sizes they hold more bytes than the level-0
// operator; at full rate they are bound by HBM, or by L2 where a level fits it.
//
// A lane owns a fixed run of VW columns of a block (VW = 4, 2 or 1 by what
// divides bc) in RPL of its rows: LC = bc / VW lanes read one row of the block
// side by side, G = 32 / LC rows at once, so every load instruction reads one
// contiguous run of the block whatever its width, the entries of x are loaded
// once per block, and the lane keeps one or two partial sums per row over all blocks.
// (A lane per row reads a 13-wide block with 4-byte loads 52 bytes apart, eleven
// 128-byte lines each; low blocks and short rows take it all the same, see
// wide_by_rows.)  A team of ES x BS warps
// owns a block row: ES of them share out the rows of a block (at most
// kTeamRows each), BS the blocks (block beg + b, beg + b + BS, ...).  The
// partial sums meet in shared memory and four lanes add up a row in a fixed
// order, so every row is summed in an order that depends only on the matrix
// and the team.
//
// Operations: y = A x, y = b - A x, y += A x for any br x bc blocks (at most
// 40 x 40), the block-Jacobi step x_out = x + W (b - A x) of Alg. 1 (W = w D^{-1},
// square blocks, at most 32 wide where read an entry at a time), and the fused
// residual and restriction y = R b - (R A) x of Alg. 2 with the next level's
// first step W y.
//
// GB300, FP32: level 1 of a P2 16^3 tet hierarchy (3,072 rows of about 25 blocks
// of 13 x 13, 53 MB), with a lane per row and with teams: product 16.0 -> 14.8 us,
// smoothing step 20.4 -> 17.0 us;
// level 2 (384 rows of about 98 blocks of 17 x 17, 44 MB): step 35.6 ->
// 19.0 us; fused restriction of level 1 92.4 -> 23.7 us (the last two with a
// cluster of CTAs per block row; 22.5 and 64.7 us without).  GMRES on Q2 96^2:
// 5.97 -> 4.38 ms.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace gasa {

namespace cg = cooperative_groups;

namespace {

constexpr int kTeamCluster = 8;     // CTAs sharing a block row at most
constexpr int kWideMaxRows = 40;    // rows and columns of a block at most
constexpr int kTeamRows = 8;        // rows per lane at most
constexpr int kTeamWarps = 8;       // warps per team in a CTA at most

enum { WIDE_ASSIGN = 0, WIDE_RESID = 1, WIDE_ADD = 2, WIDE_SWEEP = 3, WIDE_RFUSED = 4 };

// adds sign * (rows r0, r0 + rstep, ... of the blocks k0, k0 + BS, ... < end,
// columns c .. c + VW) . x to acc; two blocks in flight, and the column indices
// of the next two.
// Rounding: one FP32 sum over a whole row's blocks lost up to half a bit against
// summing block by block (25 blocks of 12 x 12, random values: rms error 1.4e-7 of
// the sums' rms, block by block 8.8e-8).  So a pair of blocks is summed by itself
// before it joins the row's sum, alternately one of two sums where blocks are narrow
// and rows therefore short (8.3e-8); the widest blocks, where those additions would
// take a tenth of the time and the registers another warp (3,000 rows of 12 blocks of
// 24 x 24: 16.5 us, with pairs 20.4), keep a sum for the first and one for the second
// block of the pairs (12 blocks of 24 x 24: 1.0e-7 -> 8.7e-8, block by block 8.8e-8).
template <int VW, int RPL>
struct TeamSums {
  static constexpr bool pairs = VW < 4 || RPL <= 4;
  static constexpr int n = !pairs || (VW > 1 && VW * RPL <= 8) ? 2 : 1;
};

template <int VW, int RPL>
__device__ __forceinline__ void team_blocks(int k0, int end, int step, int br, int bc, int r0,
                                            int rstep, int c, const int *__restrict__ col,
                                            const float *__restrict__ val,
                                            const float *__restrict__ x, float sign,
                                            float (&acc)[TeamSums<VW, RPL>::n][RPL]) {
  constexpr int NA = TeamSums<VW, RPL>::n;
  const float *vp = val + (size_t)r0 * bc + c;
  const size_t bb = (size_t)br * bc;
  const float *xc = x + c;
  bool row[RPL];
#pragma unroll
  for (int m = 0; m < RPL; ++m) row[m] = r0 + m * rstep < br;
  int k = k0;
  int j0 = k < end ? __ldg(col + k) : 0, j1 = k + step < end ? __ldg(col + k + step) : 0;
  for (; k + step < end; k += 2 * step) {
    float a0[RPL][VW], a1[RPL][VW], x0[VW], x1[VW];
    const float *p0 = vp + (size_t)k * bb, *p1 = vp + (size_t)(k + step) * bb;
#pragma unroll
    for (int m = 0; m < RPL; ++m) {
      if (row[m]) load_vec<float, VW>(p0 + (size_t)m * rstep * bc, a0[m]);
      if (row[m]) load_vec<float, VW>(p1 + (size_t)m * rstep * bc, a1[m]);
    }
    load_vec<float, VW>(xc + (size_t)j0 * bc, x0);
    load_vec<float, VW>(xc + (size_t)j1 * bc, x1);
    j0 = k + 2 * step < end ? __ldg(col + k + 2 * step) : 0;
    j1 = k + 3 * step < end ? __ldg(col + k + 3 * step) : 0;
#pragma unroll
    for (int m = 0; m < RPL; ++m) {
      if (!row[m]) continue;
      if constexpr (!TeamSums<VW, RPL>::pairs) {
#pragma unroll
        for (int v = 0; v < VW; ++v) {
          acc[0][m] = fmaf(sign * a0[m][v], x0[v], acc[0][m]);
          acc[1][m] = fmaf(sign * a1[m][v], x1[v], acc[1][m]);
        }
      } else {
        float t0 = sign * a0[m][0] * x0[0];
        if (NA == 1) {
#pragma unroll
          for (int v = 1; v < VW; ++v) t0 = fmaf(sign * a0[m][v], x0[v], t0);
#pragma unroll
          for (int v = 0; v < VW; ++v) t0 = fmaf(sign * a1[m][v], x1[v], t0);
        } else {
          float t1 = sign * a1[m][0] * x1[0];
#pragma unroll
          for (int v = 1; v < VW; ++v) {
            t0 = fmaf(sign * a0[m][v], x0[v], t0);
            t1 = fmaf(sign * a1[m][v], x1[v], t1);
          }
          t0 += t1;
        }
        const float other = acc[NA - 1][m];
        acc[NA - 1][m] = acc[0][m] + t0;
        if (NA == 2) acc[0][m] = other;
      }
    }
  }
  if (k < end) {
    float a0[RPL][VW], x0[VW];
    const float *p0 = vp + (size_t)k * bb;
#pragma unroll
    for (int m = 0; m < RPL; ++m)
      if (row[m]) load_vec<float, VW>(p0 + (size_t)m * rstep * bc, a0[m]);
    load_vec<float, VW>(xc + (size_t)j0 * bc, x0);
#pragma unroll
    for (int m = 0; m < RPL; ++m) {
      if (!row[m]) continue;
      float t0 = sign * a0[m][0] * x0[0];
#pragma unroll
      for (int v = 1; v < VW; ++v) t0 = fmaf(sign * a0[m][v], x0[v], t0);
      acc[0][m] += t0;
    }
  }
}

// op WIDE_ASSIGN / RESID / ADD / SWEEP on (rp, col, val); WIDE_RFUSED: the
// fused residual and restriction y = R b - (R A) x with R = (rp, col, val),
// R A = (rp2, col2, val2), and, with Wm (the next level's w D^{-1}), its first
// smoothing step x2o = Wm y.  blockDim = 32 * ES * BS * teams; dynamic shared
// memory: 32 * RPL floats per warp and 40 per team.
// 64 registers (32 warps an SM) wherever the two blocks in flight fit them: at 80,
// which the compiler took when left alone, the steps of 16 x 16 blocks went from
// 8.8 to 11.6 us
template <int VW, int RPL>
__global__ void __launch_bounds__(32 * kTeamWarps, VW * RPL < 14 || VW == 2 && RPL == 8 ? 4
                                                 : VW * RPL <= 20 ? 3 : 2)
bsr_team_kernel(int op, int n_brows, int br, int bc, int ES, int BS, int CS,
                const int *__restrict__ rp,
                const int *__restrict__ col, const float *__restrict__ val,
                const float *__restrict__ Wm, const float *__restrict__ x,
                const float *__restrict__ b, float *__restrict__ y, const int *__restrict__ rp2,
                const int *__restrict__ col2, const float *__restrict__ val2,
                float *__restrict__ x2o) {
  extern __shared__ float sm[];
  __shared__ float gathered[kTeamCluster][kWideMaxRows];   // rank 0: the CTAs' row sums
  const int rank = CS > 1 ? (int)cg::this_cluster().block_rank() : 0;
  if (CS > 1) cg::this_cluster().barrier_arrive();         // waited for before the first remote write
  const int nw = ES * BS, warps = blockDim.x >> 5, teams = warps / nw;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int team = warp / nw, wt = warp - team * nw;
  const int es = wt % ES, bs = wt / ES;
  const int LC = bc / VW, G = 32 / LC;
  const int g = lane / LC, cl = lane - g * LC;
  float *part = sm + (size_t)team * nw * 32 * RPL;            // [nw][RPL][32]
  float *res = sm + (size_t)warps * 32 * RPL + team * kWideMaxRows;
  const bool smooth = op == WIDE_SWEEP || (op == WIDE_RFUSED && Wm);
  const int u = CS > 1 ? (int)blockIdx.x / CS : (int)blockIdx.x * teams + team;
  const bool on = u < n_brows;
  auto finish_row = [&](int r, float v) {
    const size_t t = (size_t)u * br + r;
    if (op == WIDE_ASSIGN) y[t] = v;
    else if (op == WIDE_RESID) y[t] = b[t] - v;
    else if (op == WIDE_ADD) y[t] = y[t] + v;
    else if (op == WIDE_RFUSED) {
      y[t] = v;
      res[r] = v;
    } else {
      res[r] = b[t] - v;
    }
  };
  if (smooth && on) {
    // the block of Wm is needed last: bring it into L2 meanwhile
    const int lines = (br * br * 4 + 127) / 128 + 1;
    for (int q = wt * 32 + lane; q < lines; q += nw * 32) {
      const int o = min(q * 32, br * br - 1);
      asm volatile("prefetch.global.L2 [%0];" ::"l"(Wm + (size_t)u * br * br + o));
    }
  }
  constexpr int NA = TeamSums<VW, RPL>::n;
  float acc[NA][RPL];
#pragma unroll
  for (int m = 0; m < RPL; ++m) acc[0][m] = acc[NA - 1][m] = 0.f;
  if (on && g < G) {
    const int r0 = es * G + g, rs = ES * G;
    const int first = rank * BS + bs, step = BS * CS;
    const int beg = __ldg(rp + u), end = __ldg(rp + u + 1);
    if (op == WIDE_RFUSED) {
      const int beg2 = __ldg(rp2 + u), end2 = __ldg(rp2 + u + 1);
      team_blocks<VW, RPL>(beg + first, end, step, br, bc, r0, rs, cl * VW, col, val, b, 1.f, acc);
      team_blocks<VW, RPL>(beg2 + first, end2, step, br, bc, r0, rs, cl * VW, col2, val2, x, -1.f, acc);
    } else {
      team_blocks<VW, RPL>(beg + first, end, step, br, bc, r0, rs, cl * VW, col, val, x, 1.f, acc);
    }
  }
#pragma unroll
  for (int m = 0; m < RPL; ++m) part[(wt * RPL + m) * 32 + lane] = NA == 2 ? acc[0][m] + acc[NA - 1][m] : acc[0][m];
  __syncthreads();
  if (CS > 1) cg::this_cluster().barrier_wait();         // every CTA of the cluster runs
  // four lanes per row add the row's BS * LC partial sums: a warp's columns sub,
  // sub + 4, ... in order, the warps in order, then the four
  const int sub = lane & 3;
  const int rounds = (br * 4 + nw * 32 - 1) / (nw * 32);
  for (int it = 0; it < rounds; ++it) {
    const int r = (it * nw * 32 + wt * 32 + lane) >> 2;
    float v = 0.f;
    if (r < br) {
      const int m = r / (ES * G), q = r - m * ES * G;
      const float *p = part + ((size_t)(q / G) * RPL + m) * 32 + (q % G) * LC;
      for (int s = 0; s < BS; ++s) {
        float w = 0.f;
        for (int c = sub; c < LC; c += 4) w += p[(size_t)s * ES * RPL * 32 + c];
        v += w;
      }
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (on && r < br && sub == 0) {
      if (CS == 1) finish_row(r, v);
      else cg::this_cluster().map_shared_rank(&gathered[0][0], 0)[rank * kWideMaxRows + r] = v;
    }
  }
  if (CS > 1) {
    cg::this_cluster().sync();
    if (rank != 0) return;
    for (int r = wt * 32 + lane; on && r < br; r += nw * 32) {
      float v = 0.f;
      for (int c = 0; c < CS; ++c) v += gathered[c][r];
      finish_row(r, v);
    }
  }
  if (!smooth) return;
  __syncthreads();
  // SWEEP: x_out = x + W (b - A x); RFUSED: x2o = Wm y, four lanes per row
  for (int it = 0; it < rounds; ++it) {
    const int r = (it * nw * 32 + wt * 32 + lane) >> 2;
    float v = 0.f;
    if (on && r < br) {
      const float *w = Wm + ((size_t)u * br + r) * br;
      for (int c = sub; c < br; c += 4) v = fmaf(__ldg(w + c), res[c], v);
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (on && r < br && sub == 0) {
      const size_t t = (size_t)u * br + r;
      if (op == WIDE_SWEEP) y[t] = x[t] + v;
      else x2o[t] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Narrow or low blocks: a lane per row of a block (two rows a lane beyond 32).  The
// lanes of a warp form G = 32 / br groups of br lanes and group g of warp w takes the
// blocks beg + w G + g, beg + (w + nw) G + g, ...; lane r of a group reads row r of its
// block and the block's bc entries of x, even and odd columns in sums of their own.
// The partial sums of the team's nw warps meet in shared memory and its first warp adds
// them, warps in order, then groups.
// LONG: only the block rows of at least min_len blocks, the others being the
// thread-per-row kernels': a CTA looks through `chunk` rows at once and its warps take the
// long ones among them in turn, a warp each (8,000 rows of 15 blocks of 10 x 10: with 256
// rows a CTA and their long ones one team after another 170 us; so 18.8).
// Several short blocks per instruction and next to nothing per block row: the team kernel
// above brings a block in fewer L1 lines, but half-fills its lanes with low blocks, and a
// row's sums cost it as much as ten blocks.
// ---------------------------------------------------------------------------
// one lane's rows (r0 and, with two, r0 + 32) over the blocks kbeg, kbeg + step, ... < end
// of one block row: adds sign * (row . x_col) to a0, a1
template <int VW>
__device__ __forceinline__ void lane_rows(int kbeg, int end, int step, int br, int bc, int r0,
                                          bool two, const int *__restrict__ col,
                                          const float *__restrict__ val,
                                          const float *__restrict__ x, float sign, float &a0,
                                          float &a1) {
  for (int k = kbeg; k < end; k += step) {
    const int j = __ldg(col + k);
    const float *ar0 = val + ((size_t)k * br + r0) * bc;
    const float *ar1 = ar0 + (size_t)32 * bc;
    const float *xj = x + (size_t)j * bc;
    constexpr int W = VW == 1 ? 2 : VW;          // columns per turn: at least an even and an odd one
    float s[2] = {0.f, 0.f}, t[2] = {0.f, 0.f};
    int c = 0;
    for (; VW == 1 ? c + 1 < bc : c < bc; c += W) {
      float xv[W], av[W];
#pragma unroll
      for (int q = 0; q < W; q += VW) load_vec<float, VW>(xj + c + q, xv + q);
#pragma unroll
      for (int q = 0; q < W; q += VW) load_vec<float, VW>(ar0 + c + q, av + q);
#pragma unroll
      for (int q = 0; q < W; ++q) s[q & 1] = fmaf(av[q], xv[q], s[q & 1]);
      if (two) {
#pragma unroll
        for (int q = 0; q < W; q += VW) load_vec<float, VW>(ar1 + c + q, av + q);
#pragma unroll
        for (int q = 0; q < W; ++q) t[q & 1] = fmaf(av[q], xv[q], t[q & 1]);
      }
    }
    if (VW == 1 && c < bc) {
      const float xc = __ldg(xj + c);
      s[0] = fmaf(__ldg(ar0 + c), xc, s[0]);
      if (two) t[0] = fmaf(__ldg(ar1 + c), xc, t[0]);
    }
    a0 += sign * (s[0] + s[1]);
    a1 += sign * (t[0] + t[1]);
  }
}

template <int OP, int VW, bool LONG>
__global__ void __launch_bounds__(32 * kTeamWarps)
bsr_rows_kernel(int n_brows, int br, int bc, int nw, int chunk, int min_len,
                const int *__restrict__ rp,
                const int *__restrict__ col, const float *__restrict__ val,
                const float *__restrict__ Wm, const float *__restrict__ x,
                const float *__restrict__ b, float *__restrict__ y, const int *__restrict__ rp2,
                const int *__restrict__ col2, const float *__restrict__ val2,
                float *__restrict__ x2o) {
  // red[warp][slot]: each lane's partial row sums (slot = lane, lane + 32)
  __shared__ float red[kTeamWarps][kWideMaxRows];
  __shared__ float res[kTeamWarps][kWideMaxRows];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = br <= 32 ? 32 / br : 1;          // block groups per warp
  const int g = br <= 32 ? lane / br : 0;
  const int r0 = br <= 32 ? lane - g * br : lane;
  const bool lane_on = g < G && r0 < br;
  const bool two = br > 32 && lane + 32 < br;    // second row of this lane
  // block row u by warp wt of nw of a team
  auto block_row = [&](int u, bool on, int wt, int nw) {
    float a0 = 0.f, a1 = 0.f;
    if (on && lane_on) {
      const int step = nw * G, off = wt * G + g;
      if (OP == WIDE_RFUSED) {
        lane_rows<VW>(__ldg(rp + u) + off, __ldg(rp + u + 1), step, br, bc, r0, two, col, val, b,
                      1.f, a0, a1);
        lane_rows<VW>(__ldg(rp2 + u) + off, __ldg(rp2 + u + 1), step, br, bc, r0, two, col2, val2, x,
                      -1.f, a0, a1);
      } else {
        lane_rows<VW>(__ldg(rp + u) + off, __ldg(rp + u + 1), step, br, bc, r0, two, col, val, x,
                      1.f, a0, a1);
      }
    }
    if (lane_on) red[warp][br <= 32 ? g * br + r0 : r0] = a0;
    if (two) red[warp][lane + 32] = a1;
    if (LONG) __syncwarp();
    else __syncthreads();
    if (!on || wt != 0) return;
    const int w0 = warp;                         // the team's first warp
    for (int r = lane; r < br; r += 32) {
      float v = 0.f;
      for (int w = 0; w < nw; ++w) {
        if (br <= 32) {
          for (int q = 0; q < G; ++q) v += red[w0 + w][q * br + r];
        } else {
          v += red[w0 + w][r];
        }
      }
      const size_t t = (size_t)u * br + r;
      if (OP == WIDE_ASSIGN) y[t] = v;
      else if (OP == WIDE_RESID) y[t] = b[t] - v;
      else if (OP == WIDE_ADD) y[t] = y[t] + v;
      else if (OP == WIDE_RFUSED) {
        y[t] = v;
        res[w0][r] = v;
      } else {
        res[w0][r] = b[t] - v;
      }
    }
    if (OP != WIDE_SWEEP && (OP != WIDE_RFUSED || !Wm)) return;
    __syncwarp();
    // SWEEP: x_out = x + W (b - A x); RFUSED: x2o = Wm y (W row r against res)
    for (int r = lane; r < br; r += 32) {
      const float *w = Wm + ((size_t)u * br + r) * br;
      float o[2] = {0.f, 0.f};
      int c = 0;
      for (; c + 1 < br; c += 2) {
        o[0] = fmaf(__ldg(w + c), res[w0][c], o[0]);
        o[1] = fmaf(__ldg(w + c + 1), res[w0][c + 1], o[1]);
      }
      if (c < br) o[0] = fmaf(__ldg(w + c), res[w0][c], o[0]);
      const size_t t = (size_t)u * br + r;
      if (OP == WIDE_SWEEP) y[t] = x[t] + (o[0] + o[1]);
      else x2o[t] = o[0] + o[1];
    }
  };
  if constexpr (LONG) {
    __shared__ unsigned longs[kTeamWarps];
    const int base = blockIdx.x * chunk, i = base + threadIdx.x;
    const unsigned mine =
        __ballot_sync(0xffffffffu, (int)threadIdx.x < chunk && i < n_brows &&
                                       __ldg(rp + i + 1) - __ldg(rp + i) >= min_len);
    if (lane == 0) longs[warp] = mine;
    if (!__syncthreads_or(mine != 0)) return;
    int turn = 0;
    for (int w = 0; w < kTeamWarps; ++w)
      for (unsigned m = longs[w]; m; m &= m - 1u)
        if (turn++ % kTeamWarps == warp) {
          block_row(base + w * 32 + __ffs(m) - 1, true, 0, 1);
          __syncwarp();                          // red and res serve the next row
        }
  } else {
    const int team = warp / nw, u = blockIdx.x * (kTeamWarps / nw) + team;
    block_row(u, u < n_brows, warp - team * nw, nw);
  }
}

bool al(const void *p, size_t a) { return p == nullptr || ((uintptr_t)p % a) == 0; }

// widest run the block width and every pointer allow
int wide_vec(int bc, const void *v1, const void *x1, const void *v2, const void *x2) {
  if (bc % 4 == 0 && al(v1, 16) && al(x1, 16) && al(v2, 16) && al(x2, 16)) return 4;
  if (bc % 2 == 0 && al(v1, 8) && al(x1, 8) && al(v2, 8) && al(x2, 8)) return 2;
  return 1;
}

template <int VW>
cudaError_t team_go(int op, int n_brows, int br, int bc, double avg, const int *rp, const int *col,
                    const float *val, const float *W, const float *x, const float *b, float *y,
                    const int *rp2, const int *col2, const float *val2, float *x2o,
                    cudaStream_t s) {
  const int LC = bc / VW, G = 32 / LC;
  const int rows = div_up(br, G);                  // row steps of one warp over a block
  const int ES = div_up(rows, kTeamRows);
  const int RPL = div_up(rows, ES);
  // blocks shared out over warps while each keeps four or more and the GPU has
  // fewer than 40 warps an SM; twice as many warps (or half as many blocks each)
  // cost more in the teams' sums than they hide: 14.8 -> 16.7 us (25.0 us) for
  // the 13 x 13 product above
  int BS = 1;
  while (ES * BS * 2 <= kTeamWarps && avg >= 8.0 * BS &&
         (long long)n_brows * ES * BS < 40LL * kNumSM)
    BS *= 2;
  if (avg > 1e8) BS = std::min(BS, 4);   // rows of unknown length
  // Few long rows: a cluster of CTAs per block row, each with a share of its
  // blocks, while it keeps the GPU within one wave (32 warps an SM) and every
  // warp eight blocks; rank 0 adds up the CTAs' sums and finishes the row.  384
  // rows of 98 blocks of 17 x 17: step 22.5 -> 19.0 us; the fused restriction to
  // them 64.7 -> 23.7 us; 64 rows of 28 x 21 blocks 29.4 -> 12.5 us.
  int CS = 1;
  while (CS < kTeamCluster && avg < 1e8 && avg >= 16.0 * BS * CS &&
         (long long)n_brows * ES * BS * CS * 2 <= 32LL * kNumSM)
    CS *= 2;
  const int nw = ES * BS, teams = CS > 1 || nw >= 8 ? 1 : 8 / nw, warps = nw * teams;
  const size_t smem = ((size_t)warps * 32 * RPL + teams * kWideMaxRows) * sizeof(float);
  const int grid = CS * div_up(n_brows, teams);
  auto go = [&](auto kern) {
    launch_kc(kern, grid, 32 * warps, smem, s, CS, op, n_brows, br, bc, ES, BS, CS, rp, col, val, W, x, b, y,
             rp2, col2, val2, x2o);
  };
#define GASA_TEAM(N) \
  case N: go(bsr_team_kernel<VW, N>); break;
  switch (RPL) {
    GASA_TEAM(1) GASA_TEAM(2) GASA_TEAM(3) GASA_TEAM(4) GASA_TEAM(5) GASA_TEAM(6) GASA_TEAM(7)
    GASA_TEAM(8)
  }
#undef GASA_TEAM
  note_launch();
  return cudaGetLastError();
}

template <int OP, int VW>
cudaError_t rows_go(int n_brows, int br, int bc, double avg, const int *rp, const int *col,
                    const float *val, const float *W, const float *x, const float *b, float *y,
                    const int *rp2, const int *col2, const float *val2, float *x2o, int min_len,
                    cudaStream_t s) {
  auto go = [&](auto kern, int grid, int nw, int chunk) {
    launch_k(kern, grid, 32 * kTeamWarps, 0, s, n_brows, br, bc, nw, chunk, min_len, rp, col, val, W,
             x, b, y, rp2, col2, val2, x2o);
    note_launch();
    return cudaGetLastError();
  };
  if constexpr (OP != WIDE_RFUSED) {
    if (min_len > 0) {
      // as many rows a CTA as give an SM eight CTAs, a row a warp at least
      const int chunk = std::min(32 * kTeamWarps, div_up(div_up(n_brows, 8 * kNumSM), kTeamWarps) * kTeamWarps);
      return go(bsr_rows_kernel<OP, VW, true>, div_up(n_brows, chunk), 1, chunk);
    }
  }
  // warps per block row: about four blocks per group, at most a CTA; without the average
  // as many as give an SM 16
  const int G = br <= 32 ? 32 / br : 1;
  int nw = 1;
  while (nw < kTeamWarps && (avg < 1e8 ? nw * G * 4 < avg : (long long)n_brows * nw < 16LL * kNumSM))
    nw *= 2;
  return go(bsr_rows_kernel<OP, VW, false>, div_up(n_brows, kTeamWarps / nw), nw, 0);
}

cudaError_t team_launch(int op, int n_brows, int br, int bc, int64_t nnzb, const int *rp,
                        const int *col, const float *val, const float *W, const float *x,
                        const float *b, float *y, const int *rp2, const int *col2,
                        const float *val2, float *x2o, int min_len, cudaStream_t s) {
  // unknown: long enough for the number of rows alone to decide (team_go caps it)
  const double avg = nnzb >= 0 ? (double)nnzb / (double)n_brows : 1e9;
  // RFUSED multiplies val with b and val2 with x
  const int vw = op == WIDE_RFUSED ? wide_vec(bc, val, b, val2, x)
                                   : wide_vec(bc, val, x, nullptr, nullptr);
  if (min_len > 0 || wide_by_rows(op, n_brows, br, bc, nnzb, vw)) {
#define GASA_ROWS(OP)                                                                             \
  case OP:                                                                                        \
    return vw == 4 ? rows_go<OP, 4>(n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2,     \
                                    val2, x2o, min_len, s)                                        \
           : vw == 2 ? rows_go<OP, 2>(n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2,   \
                                      val2, x2o, min_len, s)                                      \
                     : rows_go<OP, 1>(n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2,   \
                                      val2, x2o, min_len, s);
    switch (op) {
      GASA_ROWS(WIDE_ASSIGN) GASA_ROWS(WIDE_RESID) GASA_ROWS(WIDE_ADD) GASA_ROWS(WIDE_SWEEP)
      GASA_ROWS(WIDE_RFUSED)
    }
#undef GASA_ROWS
  }
  if (bc / vw > 32) return cudaErrorNotSupported;
  if (vw == 4)
    return team_go<4>(op, n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2, val2, x2o, s);
  if (vw == 2)
    return team_go<2>(op, n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2, val2, x2o, s);
  return team_go<1>(op, n_brows, br, bc, avg, rp, col, val, W, x, b, y, rp2, col2, val2, x2o, s);
}

}  // namespace

// Lanes on rows of blocks instead of teams (GB300, us with lanes on rows / with teams):
//  - products with widths of 33 to 40 that have to be read an entry at a time, more than
//    a team's lanes (300 rows of 30 blocks of 37 x 37 18.3, with the general kernels, which
//    they fell to, 35.2); smoothing steps stay there (300 rows of 10 11.0 / 16.0);
//  - low blocks, at most 8 rows by 16 columns: 32,768 rows of 16 blocks of 4 x 10
//    24.6 / 42.1, 4,000 rows 4.7 / 7.6, 20,000 rows of 10 of 8 x 12 16.8 / 20.6 (wider
//    ones: 4,000 rows of 16 of 4 x 31 17.6 / 10.1);
//  - blocks up to 15 x 15 where the GPU has blocks enough to be busy but rows are short or
//    the blocks few enough to come from L2: smoothing step, 1,000 rows of 40 blocks of
//    9 x 9 6.4 / 10.5, 8,000 of 12 12.2 / 14.7, 2,000 of 12 of 12 x 12 5.9 / 6.8, 1,000 of
//    28 of 14 x 14 7.2 / 8.5 (256 of 20 of 12 x 12 5.1 / 4.8, 4,000 of 20 16.6 / 12.7,
//    2,000 of 40 of 13 x 13 20.4 / 16.2);
//  - the fused restriction likewise: 1,024 rows of 45 blocks of 10 x 8 5.7 / 9.9, of
//    12 x 12 10.1 / 11.5 (4,096 rows of 36 of 12 x 12 30.7 / 18.1); and with odd widths
//    of 17 to 20, which leave a third of a team's lanes idle, on tall blocks: 2,500 rows
//    of 36 of 22 x 17 41.3 / 57.3 (64 rows of 90 13.4 / 8.6, a cluster a row).
bool wide_by_rows(int op, int n_brows, int br, int bc, int64_t nnzb, int vw) {
  if (bc / vw > 32) return op != WIDE_SWEEP;
  if (br <= 8 && bc <= 16) return true;
  if (nnzb < 0) return false;
  const int b = std::max(br, bc);
  const int64_t k = 1000;
  if (op == WIDE_RFUSED) {
    if (vw == 1 && bc >= 17 && bc <= 20 && br >= 20) return n_brows > 128;
    return br <= 16 && bc <= 12 && nnzb >= 14 * k && nnzb <= (br <= 10 && bc <= 10 ? 100 : 60) * k;
  }
  if (b > 15 || nnzb < 14 * k) return false;
  const int short_row = b <= 10 ? 24 : b <= 12 ? 14 : 10;
  const int64_t few = (b <= 10 ? 72 : b <= 12 ? 60 : 30) * k;
  return nnzb < (int64_t)short_row * n_brows || nnzb <= few;
}

bool wide_applies(int br, int bc, int n_brows, int64_t nnzb) {
  return (br > 8 || bc > 8) && br <= kWideMaxRows && bc <= kWideMaxRows && n_brows > 0 &&
         nnzb >= (long long)kLongRow * n_brows;
}

// widths beyond a team's lanes: the general kernels when the row length is unknown, too
// (1,000 rows of 12 of 37 x 37: product 32.9 us, lanes on rows 28.8; step 28.7 and 32.8)
bool wide_shape(int br, int bc, const float *val, const float *x) {
  return (br > 8 || bc > 8) && br <= kWideMaxRows && bc <= kWideMaxRows &&
         bc / wide_vec(bc, val, x, nullptr, nullptr) <= 32;
}

cudaError_t launch_wide(int op, int n_brows, int br, int bc, int64_t nnzb, const int *rp,
                        const int *col, const float *val, const float *W, const float *x,
                        const float *b, float *y, cudaStream_t s, int min_len) {
  if (n_brows == 0) return cudaSuccess;
  if (br > kWideMaxRows || bc > kWideMaxRows || (op == WIDE_SWEEP && br != bc))
    return cudaErrorNotSupported;
  return team_launch(op, n_brows, br, bc, nnzb, rp, col, val, W, x, b, y, nullptr, nullptr, nullptr,
                     nullptr, min_len, s);
}

cudaError_t launch_wide_restrict(int n_brows, int br, int bc, int64_t nnzb, const int *rrp,
                                 const int *rcol, const float *rval, const int *arp,
                                 const int *acol, const float *aval, const float *b,
                                 const float *x, float *y, const float *Wn, float *xn,
                                 cudaStream_t s) {
  if (n_brows == 0) return cudaSuccess;
  if (br > kWideMaxRows || bc > kWideMaxRows) return cudaErrorNotSupported;
  return team_launch(WIDE_RFUSED, n_brows, br, bc, nnzb, rrp, rcol, rval, Wn, x, b, y, arp, acol,
                     aval, xn, 0, s);
}

}  // namespace gasa
