// Size of the cull's workspace (host code).
#pragma once

#include <stdint.h>

namespace gfs {

// The cull takes its tiles in chunks of at most kCullBytes of workspace, and
// of an eighth of the memory that is free, so that the build's other buffers
// still fit.  More chunks cost launches and partly filled ones: 96^3 samples at
// tau 3 with gradients take 67.0 ms at 1 GB (3 chunks), 69.5 at 256 MB, 74.8 at
// 64 MB; a batch of 16 shapes 62.6, 64.1, 67.2; 64^3 samples and 16.2M points
// 48.2, 48.4, 49.4.
constexpr int64_t kCullBytes = (int64_t(1) << 26) * 17;  // 1.06 GiB

// tiles of a chunk: bytes of workspace per tile, `free_bytes` on the device
inline int64_t cull_chunk(int64_t tiles, int64_t bytes, int64_t free_bytes) {
  const int64_t room = free_bytes / 8 < kCullBytes ? free_bytes / 8 : kCullBytes;
  const int64_t most = room / bytes;
  return most < 1 ? 1 : (most < tiles ? most : tiles);
}

// reserve(size), with the size halved while that returns `oom`; its last result
template <class Reserve>
int shrink_until(int64_t size, int oom, Reserve reserve) {
  int r = reserve(size);
  while (r == oom && size > 1) r = reserve(size /= 2);
  return r;
}

}  // namespace gfs
