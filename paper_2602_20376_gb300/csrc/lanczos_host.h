// lanczos_host.h -- host-side pieces of the Lanczos driver (k_lanczos.cu) that
// need no GPU.
#pragma once

#include <utility>
#include <vector>

namespace lrq {

// Largest sum |h_c| / ||w|| for which the correction sum_c U_c h_c over nc unit
// vectors may run in FP32: an entry's FMA chain has at most 2 nc roundings
// (complex; eight partial chains and their sum add 8), U and h are truncated to
// FP32 (2^-23 each), so its error is below (2 nc + 12) 2^-24 sum |h_c| |U_c| and
// w moves by less than 2^-52 ||w|| (13 for 12: the gate's own rounding).
constexpr float lz_fp32_gate(int nc) { return 0x1p-28f / (2.0f * static_cast<float>(nc) + 13.0f); }

// Host buffers that copies enqueued on a stream read: CUDA may read pageable
// memory after the call returns, so they stay until `sync` has waited for the
// stream, on every way out of the scope.
template <class Sync>
class HostCopies {
 public:
  explicit HostCopies(Sync sync) : sync_(sync) {}
  HostCopies(const HostCopies&) = delete;
  HostCopies& operator=(const HostCopies&) = delete;
  ~HostCopies() {
    if (!kept_.empty()) sync_();
  }
  const double* keep(std::vector<double>&& v) {
    kept_.push_back(std::move(v));  // moves of a vector leave its elements in place
    return kept_.back().data();
  }

 private:
  Sync sync_;
  std::vector<std::vector<double>> kept_;
};

}  // namespace lrq
