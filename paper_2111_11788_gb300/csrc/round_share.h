// How many CTAs the resident solves (resident.cu) of an allocation round may
// take beside the solves on larger meshes, and for how long. Host code without
// CUDA.
#pragma once

#include <cstdint>

namespace mlmc {

// The CTAs of resident solves that fit the GPU: three per SM.
constexpr int64_t RESIDENT_ALL_CTAS = 456;

// The solves of a round, in unknowns times samples; a Jacobi solve's iterations
// grow with the cells per side, a multigrid solve's do not.
struct RoundWork {
  double resident = 0.0;
  double beside = 0.0;   // on larger meshes, of levels without a resident solve
  static double of(int dim, int n, bool jacobi, int64_t samples) {
    double w = (double)samples * (jacobi ? n : 1);
    for (int d = 0; d < dim; ++d) w *= n - 1;
    return w;
  }
  // a level's coupled samples: the work on its mesh and on the next coarser one
  // (0 on level 0), and which of them are resident
  void add_level(double fine, bool fine_resident, double coarse, bool coarse_resident) {
    if (fine_resident) resident += fine;
    if (coarse_resident) resident += coarse;
    if (!fine_resident && !coarse_resident) beside += fine + coarse;
  }
};

// The limit on the CTAs of a round's resident solves, 0: as many as the batch
// has. A resident solve holds all its CTAs' registers while it waits on
// barriers, and the larger meshes' kernels, which fill the HBM or the FP64 pipe,
// run beside it: so it is held to a quarter of the GPU where it ends long before
// them, to half where it is about as long, and not where it dominates. A level
// whose coarse mesh is resident and whose fine mesh is not gains nothing from a
// limit: its own fine solve waits for it. ms with 114 / 228 / any number of CTAs
// by resident / beside:
//   mixed 32^2..512^2   0.13: 19.3/19.6/20.1, 0.49: 9.5/9.6/10.0, 2.6: 7.4/6.7/7.1, 24: 16.3/10.1/8.1
//   mixed 32^2..1024^2  0.20: 20.1/20.4/20.5, 0.32: 16.2/16.1/16.2, 0.83: 14.0/11.8/11.9
//   mixed 8^3..128^3    0.20: 29.2/28.6/28.8, 0.50: 26.3/19.4/19.6, 1.4: 25.8/15.5/15.1
//   FP64 32^2..512^2    0.13: 43.3/44.2/44.6, 0.49: 20.2/20.9/21.1, 1.3 (large batches): 75.1/67.8/68.0, 2.5: 70.1/62.9/59.3
//   FP64 32^2..1024^2   0.48: 28.7/30.3/30.4, 0.97: 25.2/24.6/24.8
//   nothing beside: mixed 32^2..256^2, 100 samples a level 10.4/7.9/7.3; 1000 FP64 samples of 128^2 and one of 256^2
//   71.0/44.9/32.1
inline int64_t resident_limit(const RoundWork& w, bool mixed) {
  if (w.resident <= (mixed ? 0.25 : 0.5) * w.beside) return RESIDENT_ALL_CTAS / 4;
  return w.resident <= 2.0 * w.beside ? RESIDENT_ALL_CTAS / 2 : 0;
}

// Sets `value` for the rest of a scope, whichever way it is left.
class ScopedLimit {
 public:
  ScopedLimit(int64_t& where, int64_t value) : where_(where), was_(where) { where_ = value; }
  ~ScopedLimit() { where_ = was_; }
  ScopedLimit(const ScopedLimit&) = delete;
  ScopedLimit& operator=(const ScopedLimit&) = delete;

 private:
  int64_t& where_;
  const int64_t was_;
};

}  // namespace mlmc
