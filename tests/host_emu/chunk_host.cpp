// The cull's workspace sizes (csrc/gfs_chunk.h) against a fake device that has
// `fits` tiles of room: *tried counts the attempts, the result is the tiles
// reserved, or minus the error.
#include "gfs_chunk.h"

extern "C" long long chunk_host(long long tiles, long long bytes, long long free_bytes) {
  return gfs::cull_chunk(tiles, bytes, free_bytes);
}
extern "C" long long shrink_host(long long size, long long fits, int other, int* tried) {
  long long got = 0;
  *tried = 0;
  const int r = gfs::shrink_until(size, 2, [&](int64_t s) {
    ++*tried;
    if (other && *tried == other) return 3;
    if (s > fits) return 2;
    got = s;
    return 0;
  });
  return r ? -r : got;
}
