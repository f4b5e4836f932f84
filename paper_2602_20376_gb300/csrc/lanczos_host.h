// lanczos_host.h -- host-side pieces of the Lanczos driver (k_lanczos.cu) that
// need no GPU.
#pragma once

#include <utility>
#include <vector>

namespace lrq {

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
