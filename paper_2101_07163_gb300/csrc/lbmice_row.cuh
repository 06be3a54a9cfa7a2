// One step of the stencils and folds other than the default scheme (E2, E6, E8, four-fold), on any
// grid and storage.
#pragma once

#include "lbmice_step.cuh"

namespace lbmice {

// A tile of W - 2 rows of 30 columns per CTA of W warps: warp w collides row y0 - 1 + w on all 32
// lanes, one node per thread, and the inner rows and lanes pull. Every thread collides once: a
// 32 x 8 tile whose threads also collided its one-node ring, a second collision for a third of
// them, took 22.8 us per step for E8 at 800^2 without flow and 3.7 at 100^2; this one 21.3 and 2.7.
// 8 warps, 4 CTAs per SM: the shape with the least waiting at the two barriers (16 warps 22.6,
// 10 warps 22.5, although fewer of their collisions are redundant). g and f collided ahead of the
// barrier, as the two-step kernels do, cost 2% here.
template <int W, int R>
struct RowTile {
  static constexpr int H = R + 1;
  static constexpr int PW = 30 + 2 * H, PH = W - 2 + 2 * H, PN = PW * PH;
  static constexpr int SN = 32 * W;
  template <bool FLOW>
  static constexpr size_t smem_bytes() {
    return sizeof(float) * (PostTile::floats<FLOW>(SN) + PN);
  }
};
template <int W, bool FLOW, class S, int R>
__global__ void __launch_bounds__(32 * W, 32 / W)
    row_kernel(const Consts C, const StepPtrs P) {
  using T = RowTile<W, R>;
  extern __shared__ __align__(16) float smem[];
  const int x0 = ((int)blockIdx.x + start_after_previous()) * 30;
  // tiles above one another in y and, beyond the 65,535 a launch may have there (393,210 rows), z
  const int y0 = (int)(blockIdx.z * gridDim.y + blockIdx.y) * (W - 2);
  if (y0 >= C.ny) return;
  const PostTile post = PostTile::at<FLOW>(smem, T::SN);
  float* sphi = smem + PostTile::floats<FLOW>(T::SN);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int X = x0 - 1 + lane, Y = y0 - 1 + w;
  OwnIn<S, FLOW> own;  // in flight while the phi tile loads
  own_load<S, FLOW>(C, P, X, Y, own);
  load_phi_tile<T::PW, T::PH>(C, P, x0, y0, T::H, R, sphi, threadIdx.x, 32 * W);
  const auto view_at = [=](int shx, int shy) {
    return TileView{sphi, (w + shy + R) * T::PW + (lane + shx + R), T::PW, T::PN, R};
  };
  __syncthreads();
  float hown[9];
  if (X <= C.nx && Y <= C.ny)
    collide_source<FLOW, S, true, R>(C, P, X, Y, w * 32 + lane, view_at, post, hown, &own);
  __syncthreads();
  if (w < 1 || w > W - 2 || lane < 1 || lane > 30 || X >= C.nx || Y >= C.ny) return;
  if (!in_range((w - 1) * 32 + lane - 1, T::SN, OOB_SHARED) ||
      !in_range((w + 1) * 32 + lane + 1, T::SN, OOB_SHARED))
    return;
  pull_store<FLOW, S>(C, P, X, Y,
                      [&](int a) { return (w - cy_of(a)) * 32 + (lane - cx_of(a)); }, post, hown);
}

// 32 x 8 tiles whose threads also collide the one-node ring: fewer CTAs, each 1.55 times as long. For
// grids that lose by the 30 columns and 6 rows of a row tile: those it takes beyond one wave and a tile
// does not, or whose strips it leaves nearly empty (32 or 64 columns); one_step_tiles has the line.
template <bool FLOW, class S>
__global__ void __launch_bounds__(256, 4)
    tile_kernel(const Consts C, const StepPtrs P) {
  extern __shared__ __align__(16) float smem[];
  const int x0 = ((int)blockIdx.x + start_after_previous()) * 32;
  step_tile<32, 8, FLOW, S, 2, true>(C, P, x0, blockIdx.y * 8, smem);
}

}  // namespace lbmice
