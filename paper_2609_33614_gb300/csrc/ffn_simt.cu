// CUDA-core expert FFN kernels: the path for fp32 layers (full fp32 arithmetic, no tensor-core
// rounding) over grouped, gathered rows.  SwiGLU experts (§3.1 expert FFN; the configurations use
// SwiGLU): act = silu(x Wg^T) * (x Wu^T) fused in the first kernel's epilogue; the second kernel
// is the down projection act Wd^T, written per slot in fp32 for the combine.
//
// A block computes BR rows x BC weight rows (gate and up rows of BC / 2 features, or BC down
// features) of one group.  Operands go through shared memory as they lie in memory (K contiguous,
// cp.async, rows padded by 16 bytes so that eight rows' 16-byte pieces cover all banks); a warp
// owns a (4 TM) x (8 TN) tile, lane (l / 8, l % 8) the rows l / 8 + 4 i and columns l % 8 + 8 j,
// and reads TM + TN 16-byte pieces per TM * TN * 4 FMAs.  KG groups of warps take equal shares of
// each K chunk and their tiles are added through shared memory in group order.
//
// What bounds it: a large call the shared-memory reads (8 x 8 outputs per thread need one 16-byte
// read per 16 FMAs), a small call the latency of one block's tile lookup, copies and sums.  Hence
// three shapes, by the call's (selected rows) x (expert width); the layer of 8 experts, K = 2, width
// 512 and d_model 256, us per forward call in a graph (small / mid / large shape):
//   tokens   64   128   384   512   768  1300  1536  1850  1999  2200  3000  4096
//   small  25.7  33.5  55.0  64.7  90.5 137.1 157.7 189.1 200.0 218.8 286.9 382.8
//   mid    35.8  41.2  58.0  64.2  77.2  95.5 106.5 135.7 144.6 150.3 186.3 248.4
//   large  57.9  59.1  73.4  96.1 100.3 122.4 135.6 141.5 141.9 142.4 177.1 246.4
// The line between small and mid lies there for the other layers measured too (64 experts, K = 8,
// width 1024, d 2048: 64 tokens 389 / 382; 16 experts, K = 2, width 1024, d 512: 200 85 / 84, 300 116 /
// 118; 8 experts, width 2048, d 2048: 64 202 / 261, 128 345 / 314).  Mid and large cross at 200 to 500
// rows per expert, which the toy layer reaches at its line (1953 tokens) and wider layers later than
// theirs: the layer of 64 experts mid / large 300 tokens 1107 / 1298, 1300 3723 / 3784, 1536 4311 /
// 4232; that of 16 experts 1300 273 / 300, 1536 312 / 303, 1999 406 / 430, 3000 574 / 568; 8 experts of
// width 2048 512 806 / 1026, 1000 1436 / 1456, 2200 2911 / 2803.
// (the kernels before, 32 x 64 tiles with 2 x 4 outputs per thread and one chunk in flight: gate/up
// and down 26.6 + 46.1 us at 64 tokens, 108 + 95 us at 1999.)
#include "eat_internal.cuh"

namespace eat {

namespace {

// BR, BC: rows and weight rows of a block; TM, TN: outputs per thread; KG: warp groups along K;
// BK: columns of a K chunk; ST: chunks in flight; GATEUP: gate and up rows, or down rows.
template <bool GATEUP_, int WR_, int WC_, int TM_, int TN_, int KG_, int BK_, int ST_, int MINB_>
struct SimtCfg {
  static constexpr bool GATEUP = GATEUP_;
  static constexpr int WR = WR_, WC = WC_, TM = TM_, TN = TN_, KG = KG_, BK = BK_, ST = ST_;
  static constexpr int MINB = MINB_;  // blocks an SM should hold (register bound)
  static constexpr int BR = WR * 4 * TM, BC = WC * 8 * TN;
  static constexpr int FEAT = GATEUP ? BC / 2 : BC;  // output features of a block
  static constexpr int THREADS = 32 * WR * WC * KG;
  static constexpr int LD = BK + 4;  // floats between the rows of a chunk in shared memory
  static constexpr int STAGE = (BR + BC) * LD;
  static constexpr int RED = KG > 1 ? KG * BR * (BC + 1) : 0;  // partial tiles (reuse the ring)
  static constexpr int SMEM = 4 * (ST * STAGE > RED ? ST * STAGE : RED);
  static_assert(BK % (4 * KG) == 0, "K share of a warp group in 16-byte pieces");
};
using SimtLargeUp = SimtCfg<true, 2, 2, 8, 8, 1, 32, 3, 2>;
using SimtLargeDown = SimtCfg<false, 1, 2, 8, 8, 2, 32, 3, 2>;
using SimtMidUp = SimtCfg<true, 1, 1, 8, 8, 4, 64, 2, 3>;
using SimtMidDown = SimtCfg<false, 1, 1, 8, 8, 4, 64, 2, 3>;
using SimtSmallUp = SimtCfg<true, 1, 1, 4, 4, 8, 256, 2, 1>;
using SimtSmallDown = SimtCfg<false, 1, 1, 4, 4, 8, 256, 2, 1>;
static_assert(SimtLargeUp::BR == simt_rows_up(SimtShape::kLarge) &&
                  SimtLargeDown::BR == simt_rows_down(SimtShape::kLarge) &&
                  SimtMidUp::BR == simt_rows_up(SimtShape::kMid) &&
                  SimtMidDown::BR == simt_rows_down(SimtShape::kMid) &&
                  SimtSmallUp::BR == simt_rows_up(SimtShape::kSmall) &&
                  SimtSmallDown::BR == simt_rows_down(SimtShape::kSmall),
              "row tiles the permute is told");

// The row tile of block u, found by one warp in two round trips: the group is the number of tile
// prefixes at or below u (32 groups per step; loads bypass L1, which may hold an earlier call's).
struct TileInfo {
  int g, slot0, nrows;
};
template <int BR>
__device__ __forceinline__ TileInfo find_tile(const GroupMap& gm, int u, int lane) {
  const unsigned full = 0xffffffffu;
  TileInfo ti{0, 0, 0};
  if (gm.tile_offs) {
    const int G = gm.n_groups;
    int cnt = 0, first = 0, beg = 0, end = 0;
    for (int b = 0; b < G; b += 32) {
      const int e = b + lane;
      const int te = e < G ? __ldcg(gm.tile_offs + e) : 0x7fffffff;
      const int oe = e < G ? __ldcg(gm.row_offs + e) : 0;
      const int on = e < G ? __ldcg(gm.row_offs + e + 1) : 0;
      const unsigned m = __ballot_sync(full, te <= u);
      if (m) {  // (prefixes ascend: the last group at or below u is the highest set lane)
        const int l = 31 - __clz(m);
        first = __shfl_sync(full, te, l);
        beg = __shfl_sync(full, oe, l);
        end = __shfl_sync(full, on, l);
      }
      cnt += __popc(m);
    }
    ti.g = cnt - 1;
    ti.slot0 = beg + (u - first) * BR;
    ti.nrows = min(BR, end - ti.slot0);  // <= 0 past the last group's tiles
  } else {
    const int tpg = (gm.uniform_rows + BR - 1) / BR;
    if (u >= tpg * gm.n_groups) return ti;
    ti.g = u / tpg;
    const int r0 = (u - ti.g * tpg) * BR;
    ti.slot0 = ti.g * gm.uniform_rows + r0;
    ti.nrows = min(BR, gm.uniform_rows - r0);
  }
  return ti;
}

__device__ __forceinline__ int in_row(const GroupMap& gm, int g, int s) {
  if (gm.row_mode == kRowGather) return __ldcg(gm.row_tok + s);
  if (gm.row_mode == kRowSlot) return s;
  return s - g * gm.uniform_rows;
}

template <class C>
__global__ void __launch_bounds__(C::THREADS, C::MINB)
ffn_simt_kernel(const float* __restrict__ in, const float* __restrict__ w0,
                const float* __restrict__ w1, int Fout, int Kdim, GroupMap gm,
                float* __restrict__ out) {
  constexpr int BR = C::BR, BC = C::BC, BK = C::BK, LD = C::LD, ST = C::ST, TM = C::TM,
                TN = C::TN, KG = C::KG, NT = C::THREADS;
  constexpr int PIECES = BK / 4;          // 16-byte pieces of a chunk row
  constexpr int HALF = 4 * TN;            // gate (then up) columns of a warp tile
  extern __shared__ __align__(16) float smem_f[];
  __shared__ TileInfo s_tile;
  __shared__ int s_row[BR];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the gate/up launch follows the permute; the down launch is two launches behind it, so its
  // tile and weights need not wait for the gate/up kernel
  if (C::GATEUP) pdl_wait();
  if (warp == 0) {
    const TileInfo ti = find_tile<BR>(gm, blockIdx.y, lane);
    if (lane == 0) s_tile = ti;
    if (C::GATEUP || gm.row_mode != kRowGather)
      for (int r = lane; r < BR; r += 32)
        s_row[r] = ti.nrows > 0 ? in_row(gm, ti.g, ti.slot0 + min(r, ti.nrows - 1)) : 0;
  }
  __syncthreads();
  const TileInfo ti = s_tile;
  if (ti.nrows <= 0) {
    if (!C::GATEUP) pdl_wait();
    pdl_launch_dependents();
    return;
  }
  const int f0 = blockIdx.x * C::FEAT;
  // weight row r of the block's tile: per warp column, HALF gate rows then HALF up rows of the
  // same features, or consecutive down rows; rows past Fout repeat the last one (never stored)
  auto w_row = [&](int r) -> const float* {
    if (C::GATEUP) {
      const int wc = r / (2 * HALF), q = r % (2 * HALF);
      const int f = min(f0 + wc * HALF + q % HALF, Fout - 1);
      return (q < HALF ? w0 : w1) + ((size_t)ti.g * Fout + f) * Kdim;
    }
    return w0 + ((size_t)ti.g * Fout + min(f0 + r, Fout - 1)) * Kdim;
  };
  const int chunks = (Kdim + BK - 1) / BK;
  // rows past the tile's repeat its last one (their outputs are never stored); K is a multiple of
  // 64, and a last chunk shorter than BK is copied and summed up to K
  auto load_w = [&](int c) {
    float* st = smem_f + (c % ST) * C::STAGE + BR * LD;
    const int k0 = c * BK, np = min(PIECES, (Kdim - k0) / 4);
    for (int i = tid; i < BC * PIECES; i += NT) {
      const int r = i / PIECES, p = i % PIECES;
      if (p < np)
        cp_async16((uint32_t)__cvta_generic_to_shared(st + r * LD + p * 4), w_row(r) + k0 + p * 4);
    }
  };
  auto load_x = [&](int c) {
    float* st = smem_f + (c % ST) * C::STAGE;
    const int k0 = c * BK, np = min(PIECES, (Kdim - k0) / 4);
    for (int i = tid; i < BR * PIECES; i += NT) {
      const int r = i / PIECES, p = i % PIECES;
      if (p < np)
        cp_async16((uint32_t)__cvta_generic_to_shared(st + r * LD + p * 4),
                   in + (size_t)s_row[r] * Kdim + k0 + p * 4);
    }
  };
#pragma unroll
  for (int c = 0; c < ST - 1; ++c)
    if (c < chunks) load_w(c);
  if (!C::GATEUP) pdl_wait();
  pdl_launch_dependents();
#pragma unroll
  for (int c = 0; c < ST - 1; ++c) {
    if (c < chunks) load_x(c);
    cp_async_commit();
  }

  const int kg = warp / (C::WR * C::WC), wt = warp % (C::WR * C::WC);
  const int wr = wt / C::WC, wc = wt % C::WC;
  const int lr = lane >> 3, lc = lane & 7;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  for (int c = 0; c < chunks; ++c) {
    cp_async_wait<ST - 2>();
    __syncthreads();  // chunk c is there for everyone, and chunk c - 1's buffer is free
    if (c + ST - 1 < chunks) {
      load_w(c + ST - 1);
      load_x(c + ST - 1);
    }
    cp_async_commit();
    const int kc = min(BK, Kdim - c * BK) / KG;  // this warp group's columns (K % 64 == 0)
    const float* as = smem_f + (c % ST) * C::STAGE + (wr * 4 * TM + lr) * LD + kg * kc;
    const float* bs = smem_f + (c % ST) * C::STAGE + (BR + wc * 8 * TN + lc) * LD + kg * kc;
#pragma unroll 2
    for (int kk = 0; kk < kc; kk += 4) {
      float4 b[TN];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = *(const float4*)(bs + 8 * j * LD + kk);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 a = *(const float4*)(as + 4 * i * LD + kk);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc[i][j] = fmaf(a.x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a.y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a.z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a.w, b[j].w, acc[i][j]);
        }
      }
    }
  }
  cp_async_wait<0>();

  if constexpr (KG == 1) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = wr * 4 * TM + lr + 4 * i;
      if (r >= ti.nrows) continue;
      float* o = out + (size_t)(ti.slot0 + r) * Fout;
      if constexpr (C::GATEUP) {
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
          const int f = f0 + wc * HALF + lc + 8 * j;
          const float g = acc[i][j];
          if (f < Fout) o[f] = g / (1.0f + expf(-g)) * acc[i][j + TN / 2];
        }
      } else {
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int f = f0 + wc * 8 * TN + lc + 8 * j;
          if (f < Fout) o[f] = acc[i][j];
        }
      }
    }
  } else {
    // the warp groups' tiles into shared memory (the ring is no longer read), then their sums
    constexpr int RL = BC + 1;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        smem_f[(kg * BR + wr * 4 * TM + lr + 4 * i) * RL + wc * 8 * TN + lc + 8 * j] = acc[i][j];
    __syncthreads();
    for (int q = tid; q < BR * C::FEAT; q += NT) {
      const int r = q / C::FEAT, fl = q % C::FEAT, f = f0 + fl;
      if (r >= ti.nrows || f >= Fout) continue;
      // column of the feature's first (gate or only) weight row in the tile
      const int col = C::GATEUP ? fl / HALF * (2 * HALF) + fl % HALF : fl;
      float g = 0.f, u = 0.f;
#pragma unroll
      for (int s = 0; s < KG; ++s) {
        g += smem_f[(s * BR + r) * RL + col];
        if (C::GATEUP) u += smem_f[(s * BR + r) * RL + col + HALF];
      }
      out[(size_t)(ti.slot0 + r) * Fout + f] = C::GATEUP ? g / (1.0f + expf(-g)) * u : g;
    }
  }
}

template <class C>
cudaError_t configure_simt() {
  return cudaFuncSetAttribute(ffn_simt_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              C::SMEM);
}

template <class C>
cudaError_t launch_simt(const float* in, const float* w0, const float* w1, int Fout, int Kdim,
                        const GroupMap& gm, float* out, cudaStream_t st) {
  const dim3 grid((Fout + C::FEAT - 1) / C::FEAT, gm.max_tiles);
  if (grid.y == 0) return cudaSuccess;
  return launch_pdl(ffn_simt_kernel<C>, grid, dim3(C::THREADS), C::SMEM, st, in, w0, w1, Fout,
                    Kdim, gm, out);
}

}  // namespace

cudaError_t simt_configure() {
  cudaError_t e = configure_simt<SimtLargeUp>();
  if (e == cudaSuccess) e = configure_simt<SimtLargeDown>();
  if (e == cudaSuccess) e = configure_simt<SimtMidUp>();
  if (e == cudaSuccess) e = configure_simt<SimtMidDown>();
  if (e == cudaSuccess) e = configure_simt<SimtSmallUp>();
  if (e == cudaSuccess) e = configure_simt<SimtSmallDown>();
  return e;
}

SimtShape simt_shape(int T, int K, int F) {
  // selected rows x width: where the columns of the table at the top of this file cross
  const long long work = (long long)T * K * F;
  return work >= 2000000 ? SimtShape::kLarge
                         : work >= 512 * 1024 ? SimtShape::kMid : SimtShape::kSmall;
}

cudaError_t launch_ffn_gateup_simt(const float* in, const float* wg, const float* wu, int Fout,
                                   int Kdim, GroupMap gm, SimtShape shape, float* act,
                                   cudaStream_t st) {
  if (shape == SimtShape::kLarge)
    return launch_simt<SimtLargeUp>(in, wg, wu, Fout, Kdim, gm, act, st);
  if (shape == SimtShape::kMid)
    return launch_simt<SimtMidUp>(in, wg, wu, Fout, Kdim, gm, act, st);
  return launch_simt<SimtSmallUp>(in, wg, wu, Fout, Kdim, gm, act, st);
}

cudaError_t launch_ffn_down_simt(const float* act, const float* wd, int Dout, int Kdim,
                                 GroupMap gm, SimtShape shape, float* out, cudaStream_t st) {
  gm.row_mode = kRowSlot;  // act rows are in slot order, the shared experts' too
  if (shape == SimtShape::kLarge)
    return launch_simt<SimtLargeDown>(act, wd, nullptr, Dout, Kdim, gm, out, st);
  if (shape == SimtShape::kMid)
    return launch_simt<SimtMidDown>(act, wd, nullptr, Dout, Kdim, gm, out, st);
  return launch_simt<SimtSmallDown>(act, wd, nullptr, Dout, Kdim, gm, out, st);
}

}  // namespace eat
