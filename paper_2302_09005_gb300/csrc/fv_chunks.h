// fv_chunks.h -- how fv_patch_update_host cuts a batch into chunks of
// consecutive patches when the caller does not say: by bytes, whatever the
// patches' sizes and the gaps between them.  (Cut by patch 0's size, 4,000
// patches of 8^3 behind one of 1^3 were one chunk, without overlap and with
// 37 times the staging.)  Host code.
#pragma once

#include <stdint.h>

namespace fv {

constexpr int64_t kChunkMin = 4ll << 20, kChunkMax = 256ll << 20;

// Bytes of a chunk: on pinned memory an eighth of the batch, rounded up to whole
// patches (eight chunks hold it: a ninth of a few patches costs as much as any;
// no further, since chunks of 1,025 patches of 17x17 copied 5 % slower than the
// better aligned ones of 1,024), 4 to 256 MB.  The
// copy in, the update and the copy out overlap only from chunk to chunk, and a
// chunk costs the host some 20 us.  One chunk / eighths, us per call: 94.6 MB (8,192 2D
// patches of 17x17, FP64) 1299 / 876, 31.4 MB 660 / 596, 450 MB 4591 / 2847;
// 5.9 MB 121 / 99 in two, 155 in eight; 3.6 GB in 256 MB chunks 19.8 ms, in
// 128 MB chunks 20.3.  Copies of pageable memory hold the calling thread and do
// not overlap, so there only the cost of a chunk is left: 256 MB always (256 MB /
// eighths, us per call in place: 5.9 MB 123 / 164, 56 MB 608 / 1131, 94.6 MB 1237 /
// 1566, 450 MB 4331 / 4826).
inline int64_t chunk_bytes(int64_t batch_bytes, int64_t patch_bytes, bool pinned) {
  const int64_t want = pinned ? batch_bytes / 8 + patch_bytes - 1 : kChunkMax;
  return want < kChunkMin ? kChunkMin : want > kChunkMax ? kChunkMax : want;
}

// The patch after the last one of the chunk that starts at p0: as many as
// span at most `want` bytes, at least one.  off: element offsets; len(i):
// elements of patch i; es: bytes of an element.  The patches ascend without
// overlap, so their ends ascend and a binary search finds the last one.
template <typename Len>
inline int64_t chunk_end(int64_t p0, int64_t n, const int64_t* off, const Len& len, int64_t es,
                         int64_t want) {
  const int64_t last = off[p0] + want / es;
  int64_t lo = p0 + 1, hi = n;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const int64_t mid = lo + (hi - lo) / 2;
    if (off[mid] + len(mid) <= last)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

}  // namespace fv
