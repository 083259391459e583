// The limit on the CTAs of the resident solves (resident.cu) while an
// allocation round is captured. Host code without CUDA.
#pragma once

#include <cstdint>

namespace mlmc {

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
