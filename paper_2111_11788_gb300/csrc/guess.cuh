// Nested initial guess: cubic interpolation of the coarse-mesh solution.
//
// The fine solve of a coupled sample starts from its coarse partner's
// solution. Bilinear interpolation leaves an oscillatory residual of the
// size of b (||r|| / ||b|| = 1.6 at 512^2), cubic interpolation one that falls with
// the mesh (2.7e-3 at 512^2, 3e-2 at 64^3): about one CG iteration less in
// FP64, one to two refinement steps less in the mixed form.
#pragma once

namespace mlmc {

// Along an axis of nc coarse cells, the fine node between coarse nodes I and
// I + 1 takes the cubic through the coarse nodes b .. b + 3 around it (at the
// ends of the axis the first or the last four).
constexpr int CUBIC_MIN_CELLS = 4;   // coarse cells per side from which the guess is cubic

__device__ __forceinline__ int cubic_base(int I, int nc) { return I == 0 ? 0 : (I >= nc - 1 ? nc - 3 : I - 1); }
__device__ __forceinline__ double cubic_mid(int I, int nc, double a, double b, double c, double d) {
  const bool lo = I == 0, hi = I == nc - 1;
  double v = (lo ? 0.3125 : (hi ? 0.0625 : -0.0625)) * a;
  v = fma(lo ? 0.9375 : (hi ? -0.3125 : 0.5625), b, v);
  v = fma(lo ? -0.3125 : (hi ? 0.9375 : 0.5625), c, v);
  return fma(lo ? 0.0625 : (hi ? 0.3125 : -0.0625), d, v);
}
// at(k): the coarse value k; the value at fine node i of the axis
template <class F>
__device__ __forceinline__ double cubic_at(int i, int nc, F&& at) {
  const int I = i >> 1;
  if (!(i & 1)) return at(I);
  const int b = cubic_base(I, nc);
  return cubic_mid(I, nc, at(b), at(b + 1), at(b + 2), at(b + 3));
}

// The coarse values of four consecutive coarse slabs (rows or planes),
// carried while the fine slabs are walked in increasing order.
struct CubicWindow {
  double v[4];
  int b;
  template <class F>
  __device__ __forceinline__ void start(int i, int nc, F&& at) {
    b = cubic_base(i >> 1, nc);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = at(b + k);
  }
  template <class F>
  __device__ __forceinline__ void advance(int i, int nc, F&& at) {
    const int nb = cubic_base(i >> 1, nc);
    while (b < nb) {
      v[0] = v[1];
      v[1] = v[2];
      v[2] = v[3];
      v[3] = at(b + 4);
      ++b;
    }
  }
  __device__ __forceinline__ double value(int i, int nc) const {
    const int I = i >> 1, k = I - b;
    if (i & 1) return cubic_mid(I, nc, v[0], v[1], v[2], v[3]);
    return k == 0 ? v[0] : (k == 1 ? v[1] : (k == 2 ? v[2] : v[3]));
  }
};

// A warp owns 32 coarse columns, one per lane from I0 - GUESS_HALO on, and
// makes the fine columns 2I and 2I + 1 of the GUESS_COLS columns whose four
// neighbours it holds; `v` is the value at coarse column I of the row being
// made. Returns the value at 2I + 1.
constexpr int GUESS_HALO = 2, GUESS_COLS = 27;
__device__ __forceinline__ double guess_odd(int I, int nc, double v) {
  constexpr unsigned FULL = 0xffffffffu;
  const double m1 = __shfl_up_sync(FULL, v, 1), m2 = __shfl_up_sync(FULL, v, 2);
  const double p1 = __shfl_down_sync(FULL, v, 1), p2 = __shfl_down_sync(FULL, v, 2), p3 = __shfl_down_sync(FULL, v, 3);
  const bool lo = I == 0, hi = I == nc - 1;
  return cubic_mid(I, nc, lo ? v : (hi ? m2 : m1), lo ? p1 : (hi ? m1 : v), lo ? p2 : (hi ? v : p1),
                   lo ? p3 : (hi ? p1 : p2));
}

}  // namespace mlmc
