// cc_chunks.h - which chunks of a graph the filtered phase of a batch gives to
// which warp of a block (host and device: plain integer arithmetic).
#ifndef CC_CHUNKS_H
#define CC_CHUNKS_H

#include <stdint.h>

#ifdef __CUDACC__
#define CC_HOST_DEVICE __host__ __device__
#else
#define CC_HOST_DEVICE
#endif

namespace cc {

// The chunks of [c0, c1) that were not sampled (index not a multiple of stride,
// stride >= 2), shared out in turn: number k of the unsampled chunks is
// k + k / (stride - 1) + 1, and warp w of nw takes numbers w, w + nw, ... from the
// first of the range. (Every nw-th chunk with the sampled ones skipped left the
// warps that met only sampled ones without work: half of 16 with a stride of 2.)
class UnsampledChunks {
 public:
  CC_HOST_DEVICE UnsampledChunks(uint32_t c0, uint32_t stride, uint32_t w, uint32_t nw)
      : period_(stride - 1u), dq_(nw / (stride - 1u)), dr_(nw % (stride - 1u)) {
    const uint32_t k = c0 - (c0 + stride - 1u) / stride + w;  // unsampled chunks before c0, then w more
    q_ = k / period_;
    r_ = k % period_;
  }
  // The chunk; at or past the range when there is none left.
  CC_HOST_DEVICE uint32_t chunk() const { return q_ * (period_ + 1u) + r_ + 1u; }
  CC_HOST_DEVICE void next() {
    q_ += dq_;
    r_ += dr_;
    if (r_ >= period_) {
      r_ -= period_;
      ++q_;
    }
  }

 private:
  uint32_t period_, dq_, dr_, q_, r_;
};

}  // namespace cc

#endif
