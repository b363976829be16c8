// Small transfers between page-locked host memory and the device by a kernel (the request payload of the host-buffer
// joins and the mask that goes back).  A request's payload is six or seven arrays of a few bytes to a few hundred
// kilobytes; as one copy each they queue up behind one another, several microseconds apiece however short they are, and
// the join waits for the last.  One kernel reads all of them over the link at once.  Bound by the link's latency for small
// payloads and its rate for larger ones.  Through L2 (__ldcg): loads that bypass it (__ldcv) cross the link in 32-byte
// requests (193 KB 35 us a call instead of 22 us).  A launch sees what the host has written before it.
// One request of 30,000 candidates, rows left on the device: 57 us with copies, 22 us this way; 500 candidates 47 -> 17 us;
// four requests (770 KB) 88 -> 58 us; eight (1.6 MB) 118 -> 98 us.
#pragma once

#include "ccr_device.cuh"

namespace ccr {

constexpr int kCopySegments = 8;
constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 4;  // 16-byte pieces a thread has in flight (one: no difference)

struct CopyArgs {
  const uint8_t* src[kCopySegments];  // 16-byte aligned; null = zeros
  uint8_t* dst[kCopySegments];        // 16-byte aligned
  long long bytes[kCopySegments];
  int n;
};

// Piece c of the concatenated segments (every segment in whole 16-byte pieces, the last one of a segment possibly short).
__global__ void __launch_bounds__(kCopyThreads) copy_segments_kernel(const CopyArgs a) {
  chain_enter(false);
  long long total = 0;
  for (int s = 0; s < a.n; ++s) total += (a.bytes[s] + 15) >> 4;
  const long long stride = static_cast<long long>(gridDim.x) * kCopyThreads;
  for (long long c0 = blockIdx.x * static_cast<long long>(kCopyThreads) + threadIdx.x; c0 < total; c0 += stride * kCopyUnroll) {
    uint4 v[kCopyUnroll];
    uint8_t* to[kCopyUnroll];
    const uint8_t* from[kCopyUnroll];
    int len[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      long long c = c0 + u * stride;
      len[u] = 0;
      v[u] = make_uint4(0u, 0u, 0u, 0u);
      if (c >= total) continue;
      int s = 0;
      for (; s < a.n - 1 && c >= (a.bytes[s] + 15) >> 4; ++s) c -= (a.bytes[s] + 15) >> 4;
      const long long left = a.bytes[s] - c * 16;
      len[u] = left < 16 ? static_cast<int>(left) : 16;
      to[u] = a.dst[s] + c * 16;
      from[u] = a.src[s] != nullptr ? a.src[s] + c * 16 : nullptr;
      if (len[u] == 16 && from[u] != nullptr && CCR_CHK(from[u], 16)) v[u] = __ldcg(reinterpret_cast<const uint4*>(from[u]));
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      if (len[u] == 16) {
        gstore(reinterpret_cast<uint4*>(to[u]), v[u]);
      } else {
        for (int i = 0; i < len[u]; ++i)
          gstore(to[u] + i, from[u] != nullptr && CCR_CHK(from[u] + i, 1) ? *reinterpret_cast<const volatile uint8_t*>(from[u] + i) : 0);
      }
    }
  }
}

}  // namespace ccr
