// Algorithm 1 step 1 of the paper on the device: per request, sort the viewer's affinity records by author
// id (a_sorted, idx = sort(a); F_sorted = gather(F, idx)) so that unsorted request payloads can be joined.
//
// The order is on (key, index of the record in its list), which makes the result the stable sort.  Lists of up to
// kListMax records (every batch whose length bound says so) are radix sorted in shared memory, one cluster of blocks per
// list, and the rows follow in a launch of their own (short lists: in the same one); see sort_lists_kernel.  Batches with
// longer lists are cut into chunks of 4,096 records: one block sorts a chunk as packed words, key << bits | index (a
// merge sort: four words per thread in registers, then runs doubled per pass along merge paths), the sorted chunks
// are merged pairwise by grid-wide launches (merge path again, one output tile per block), and the rows follow their keys
// in one grid-wide gather.  A batch with a key that leaves no room for the index is then sorted list by list by one
// 1024-thread block each.
#pragma once

#include "ccr_device.cuh"

namespace ccr {

constexpr int kSortThreads = 1024;
constexpr int kSortSmemMaxKeys = 19000;  // 12 bytes per record (int64 key + int32 index) within 227 KB

// One pass structure for both element types: for partner mask j, the pairs (i, i ^ j) with i < i ^ j are
// exactly the i whose bit `top(j)` is clear; pair number p (0 .. n/2) maps to i by inserting a zero there.
__device__ __forceinline__ int pair_low_index(int p, int top_bit) {
  const int low = p & ((1 << top_bit) - 1);
  return ((p >> top_bit) << (top_bit + 1)) | low;
}

// (key, index) records in two arrays, ordered by key then index.
__device__ __forceinline__ void sort_pairs_bitonic(long long* keys, int* idx, int n) {
  if (n < 2) return;
  for (int k = 2;; k <<= 1) {
    // flip: i pairs with its mirror inside the block of k; then disperse at distances k/4, k/8, ..., 1
    for (int j = k - 1;;) {
      const int top = 31 - __clz(j);
      for (int p = threadIdx.x;; p += blockDim.x) {
        const int i = pair_low_index(p, top), l = i ^ j;
        if (i >= n) break;  // i grows with p
        if (l < n) {
          const long long ki = keys[i], kl = keys[l];
          const int ii = idx[i], il = idx[l];
          if (ki > kl || (ki == kl && ii > il)) {
            keys[i] = kl;
            keys[l] = ki;
            idx[i] = il;
            idx[l] = ii;
          }
        }
      }
      __syncthreads();
      if (j == k - 1) j = k >> 2; else j >>= 1;
      if (j == 0) break;
    }
    if (k >= n) break;
  }
}

// M consecutive disperse steps of the network (partner distances 2^b, 2^(b-1), ..., 2^(b-M+1)) in one pass:
// the 2^M elements whose indices differ only in those M bits form a closed group, so a thread loads the group,
// runs the M rounds of compare-exchanges in registers and stores it — one barrier and one trip through shared
// memory instead of M.  Elements at or beyond n count as +infinity (every real word is below 2^63).
template <int M>
__device__ __forceinline__ void disperse_fused(unsigned long long* w, int n, int b) {
  const int sh = b - M + 1;
  for (int g = threadIdx.x;; g += blockDim.x) {
    const int base = ((g >> sh) << (b + 1)) | (g & ((1 << sh) - 1));
    if (base >= n) break;  // base grows with g
    unsigned long long v[1 << M];
#pragma unroll
    for (int m = 0; m < (1 << M); ++m) {
      const int i = base + (m << sh);
      v[m] = i < n ? w[i] : ~0ull;
    }
#pragma unroll
    for (int s = M - 1; s >= 0; --s) {
#pragma unroll
      for (int m = 0; m < (1 << M); ++m) {
        if ((m & (1 << s)) == 0) {
          const int p = m | (1 << s);
          const unsigned long long lo = min(v[m], v[p]), hi = max(v[m], v[p]);
          v[m] = lo;
          v[p] = hi;
        }
      }
    }
#pragma unroll
    for (int m = 0; m < (1 << M); ++m) {
      const int i = base + (m << sh);
      if (i < n) w[i] = v[m];
    }
  }
  __syncthreads();
}

// Every step whose partner distance is below 32 stays inside 32 consecutive elements, so a warp holding one
// element per lane runs those steps with shuffles: no shared-memory traffic, no bank conflicts, no barriers.
// FIRST: the whole network up to blocks of 32 (flip and disperse steps of k = 2 .. 32); otherwise the last five
// disperse steps (distances 16 .. 1) of a larger block.  The lane with the lower index keeps the minimum.
template <bool FIRST>
__device__ __forceinline__ void warp_steps(unsigned long long* w, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  for (int c = warp; c * 32 < n; c += n_warps) {
    const int i = c * 32 + lane;
    unsigned long long v = i < n ? w[i] : ~0ull;
    if (FIRST) {
#pragma unroll
      for (int L = 1; L <= 5; ++L) {
        const unsigned long long pf = __shfl_xor_sync(0xffffffffu, v, (1 << L) - 1);  // flip: mirror inside the block
        v = (lane & (1 << (L - 1))) == 0 ? min(v, pf) : max(v, pf);
#pragma unroll
        for (int d = (1 << L) >> 2; d >= 1; d >>= 1) {
          const unsigned long long pv = __shfl_xor_sync(0xffffffffu, v, d);
          v = (lane & d) == 0 ? min(v, pv) : max(v, pv);
        }
      }
    } else {
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long pv = __shfl_xor_sync(0xffffffffu, v, d);
        v = (lane & d) == 0 ? min(v, pv) : max(v, pv);
      }
    }
    if (i < n) w[i] = v;
  }
  __syncthreads();
}

// The same network on single 64-bit words (key << shift | index): half the shared-memory traffic; steps at
// distances below 32 run in registers (warp_steps), the others are fused up to three at a time
// (disperse_fused, always at strides of 32 words or more, which keeps them free of bank conflicts).
__device__ __forceinline__ void sort_words_bitonic(unsigned long long* w, int n) {
  if (n < 2) return;
  warp_steps<true>(w, n);  // blocks of 32 are sorted
  for (int k = 64, log_k = 6; (k >> 1) < n; k <<= 1, ++log_k) {
    {  // flip: i pairs with its mirror inside the block of k
      const int j = k - 1, top = log_k - 1;
      for (int p = threadIdx.x;; p += blockDim.x) {
        const int i = pair_low_index(p, top), l = i ^ j;
        if (i >= n) break;  // i grows with p
        if (l < n) {
          const unsigned long long wi = w[i], wl = w[l];
          if (wi > wl) {
            w[i] = wl;
            w[l] = wi;
          }
        }
      }
      __syncthreads();
    }
    // disperse at distances k/4 ... 32 in shared memory, 16 ... 1 in registers
    for (int b = log_k - 2; b >= 5;) {
      const int m = b - 4 >= 3 ? 3 : b - 4;
      if (m == 3) disperse_fused<3>(w, n, b);
      else if (m == 2) disperse_fused<2>(w, n, b);
      else disperse_fused<1>(w, n, b);
      b -= m;
    }
    warp_steps<false>(w, n);
  }
}

// Merge passes over sorted runs of `run` words in shared memory (n <= IPT * blockDim.x distinct words): runs are
// merged pairwise, doubling per pass; in a pass a thread produces IPT consecutive output words, from the point of
// its pair of runs that the merge path (a binary search along its diagonal) assigns to it, into registers, and
// writes them back after a barrier.  Two barriers per pass.
template <int IPT>
__device__ __forceinline__ void merge_passes(unsigned long long* w, int n, int run) {
  const int t0 = static_cast<int>(threadIdx.x) * IPT;
  unsigned long long v[IPT];
  for (; run < n; run <<= 1) {
    const int pb = (t0 / (2 * run)) * (2 * run);
    const int lenA = max(0, min(run, n - pb)), lenB = max(0, min(run, n - pb - run));
    const unsigned long long* A = w + pb;
    const unsigned long long* B = A + run;
    const int d = min(t0 - pb, lenA + lenB);
    int lo = max(0, d - lenB), hi = min(d, lenA);
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (A[mid] < B[d - 1 - mid]) lo = mid + 1; else hi = mid;
    }
    int i = lo, j = d - lo;
#pragma unroll
    for (int u = 0; u < IPT; ++u) {
      const bool has_a = i < lenA, has_b = j < lenB;
      const unsigned long long va = has_a ? A[i] : ~0ull, vb = has_b ? B[j] : ~0ull;
      const bool take_a = has_a && (!has_b || va < vb);
      v[u] = take_a ? va : vb;
      i += take_a ? 1 : 0;
      j += take_a ? 0 : 1;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < IPT; ++u)
      if (t0 + u < n) w[t0 + u] = v[u];
    __syncthreads();
  }
}

// Merge sort of n <= IPT * blockDim.x distinct words in shared memory: every thread sorts IPT consecutive words in
// registers (odd-even transposition), then log2(n / IPT) merge passes.
template <int IPT>
__device__ __forceinline__ void sort_words_merge(unsigned long long* w, int n) {
  const int t0 = static_cast<int>(threadIdx.x) * IPT;
  unsigned long long v[IPT];
#pragma unroll
  for (int u = 0; u < IPT; ++u) v[u] = t0 + u < n ? w[t0 + u] : ~0ull;
#pragma unroll
  for (int rd = 0; rd < IPT; ++rd) {
#pragma unroll
    for (int u = rd & 1; u + 1 < IPT; u += 2) {
      const unsigned long long lo = min(v[u], v[u + 1]), hi = max(v[u], v[u + 1]);
      v[u] = lo;
      v[u + 1] = hi;
    }
  }
#pragma unroll
  for (int u = 0; u < IPT; ++u)
    if (t0 + u < n) w[t0 + u] = v[u];
  __syncthreads();
  merge_passes<IPT>(w, n, IPT);
}

// The same for n <= 4 * blockDim.x with the first seven doublings in registers: a warp holds 128 consecutive words,
// lane-strided (word e in register e / 32 of lane e % 32, so its loads and stores are to consecutive words), and
// sorts them with a bitonic network whose steps at distances 32 and 64 pair registers of one lane and the others
// lanes (shuffles): no shared memory, no barriers.  Measured per 4,096-word chunk (two blocks resident per SM):
// 8 us for this start + 13 us for the five merge passes behind it, against 30 us for ten merge passes from runs of
// four, and 23 us with the merge passes done warp-wise on strided registers as well (bitonic merges of 128).
template <int J, typename Up>
__device__ __forceinline__ void warp128_step(unsigned long long (&v)[4], int lane, Up up) {
  if constexpr (J >= 32) {
    constexpr int dr = J >> 5;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if ((r & dr) == 0) {
        const unsigned long long lo = min(v[r], v[r | dr]), hi = max(v[r], v[r | dr]);
        const bool u = up((r << 5) | lane);  // the pair holding word e goes in ascending order
        v[r] = u ? lo : hi;
        v[r | dr] = u ? hi : lo;
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const unsigned long long pv = __shfl_xor_sync(0xffffffffu, v[r], J);
      const bool keep_min = ((lane & J) == 0) == up((r << 5) | lane);
      v[r] = keep_min ? min(v[r], pv) : max(v[r], pv);
    }
  }
}
// the steps of one block size K of the network: partner distances K/2 ... 1
template <int K, typename Up>
__device__ __forceinline__ void warp128_block(unsigned long long (&v)[4], int lane, Up up) {
  if constexpr (K >= 128) warp128_step<64>(v, lane, up);
  if constexpr (K >= 64) warp128_step<32>(v, lane, up);
  if constexpr (K >= 32) warp128_step<16>(v, lane, up);
  if constexpr (K >= 16) warp128_step<8>(v, lane, up);
  if constexpr (K >= 8) warp128_step<4>(v, lane, up);
  if constexpr (K >= 4) warp128_step<2>(v, lane, up);
  warp128_step<1>(v, lane, up);
}
__device__ __forceinline__ void sort_words_merge128(unsigned long long* w, int n) {
  const int lane = threadIdx.x & 31, o = (static_cast<int>(threadIdx.x) >> 5) * 128;
  if (o < n) {  // (a warp behind the last word has nothing but padding: 256 lists of 300 records 18.1 -> 12.7 us)
    unsigned long long v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = o + (r << 5) + lane;
      v[r] = i < n ? w[i] : ~0ull;  // padding sorts last
    }
    // blocks of K words alternate in direction until the last, which is ascending
    warp128_block<2>(v, lane, [](int e) { return (e & 2) == 0; });
    warp128_block<4>(v, lane, [](int e) { return (e & 4) == 0; });
    warp128_block<8>(v, lane, [](int e) { return (e & 8) == 0; });
    warp128_block<16>(v, lane, [](int e) { return (e & 16) == 0; });
    warp128_block<32>(v, lane, [](int e) { return (e & 32) == 0; });
    warp128_block<64>(v, lane, [](int e) { return (e & 64) == 0; });
    warp128_block<128>(v, lane, [](int) { return true; });
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = o + (r << 5) + lane;
      if (i < n) w[i] = v[r];
    }
  }
  __syncthreads();
  merge_passes<4>(w, n, 128);
}

// Rows follow their keys: output chunk c (16 bytes) comes from row source_of(c / row_ch) of the input.  One block moves the rows of
// n records, every thread with kSortGatherUnroll loads in flight; a thread steps from chunk to chunk by additions.
constexpr int kSortGatherUnroll = 8;
template <typename SourceOf>
__device__ __forceinline__ void gather_rows(const uint4* src, uint4* dst, int n, int row_ch, SourceOf source_of) {
  const int threads = static_cast<int>(blockDim.x), step_row = threads / row_ch, step_piece = threads - step_row * row_ch;
  int row = static_cast<int>(threadIdx.x) / row_ch, piece = static_cast<int>(threadIdx.x) - row * row_ch;
  const long long chunks = static_cast<long long>(n) * row_ch;
  for (long long c0 = threadIdx.x; c0 < chunks; c0 += static_cast<long long>(threads) * kSortGatherUnroll) {
    uint4 v[kSortGatherUnroll];
#pragma unroll
    for (int u = 0; u < kSortGatherUnroll; ++u) {
      if (row < n) v[u] = ldg128(src + source_of(row) * row_ch + piece);
      row += step_row;
      piece += step_piece;
      if (piece >= row_ch) {
        piece -= row_ch;
        ++row;
      }
    }
#pragma unroll
    for (int u = 0; u < kSortGatherUnroll; ++u) {
      const long long c = c0 + static_cast<long long>(u) * threads;
      if (c < chunks) st128_stream(dst + c, v[u]);
    }
  }
}

struct SortArgs {
  int* call_flag;          // chunked path: device word, zero between calls; set when a key of the batch cannot share a word with its index
  int rows_here;             // sort_lists_kernel moves the rows itself
  int more_follow;           // another kernel of the same ccr_sort_edges call is launched behind this one
  int n_req;
  const int64_t* keys_in;
  const uint8_t* feats_in;
  const int64_t* edge_offsets;
  int row_ch;            // 16-byte chunks per feature row
  int64_t* keys_out;
  uint8_t* feats_out;
  int* perm_out;         // may be null on the whole-list path
  int smem_keys;         // (key, index) records the dynamic shared memory can hold: 12 bytes each
  int smem_words;        // packed key|index words it can hold: 8 bytes each
  int max_len;           // the host's bound on the list length: longer lists are cut there (their tail is left alone)
};

#ifndef CCR_SORT_CHUNK_LOG
#define CCR_SORT_CHUNK_LOG 12
#endif
#ifndef CCR_SORT_CHUNK_THREADS
#define CCR_SORT_CHUNK_THREADS 1024
#endif
#ifndef CCR_SORT_CHUNK_BLOCKS
#define CCR_SORT_CHUNK_BLOCKS 2  // resident per SM: one block's loads hide behind the other's merging (32 registers, no spill)
#endif
constexpr int kSortChunkLog = CCR_SORT_CHUNK_LOG;
constexpr int kSortChunk = 1 << kSortChunkLog;  // records one block of the multi-block path sorts in shared memory
constexpr int kSortChunkThreads = CCR_SORT_CHUNK_THREADS;

__device__ __forceinline__ int sort_index_bits(int K) {
  int idx_bits = 1;
  while ((1 << idx_bits) < K) ++idx_bits;
  return idx_bits;
}

// Block-wide: do the K keys leave room for the record index in one 64-bit word (non-negative, below
// 2^(63 - idx_bits))?  All threads of the block must call.
__device__ __forceinline__ bool list_is_packable(const int64_t* keys, int K, int idx_bits) {
  long long kmax = 0;
  int negative = 0;
#pragma unroll 8
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const long long k = gload(keys + i);
    kmax = max(kmax, k);
    negative |= (k < 0);
  }
  return __syncthreads_or(negative || (kmax >> (63 - idx_bits)) != 0) == 0;
}

__global__ void __launch_bounds__(kSortThreads, 1) sort_edges_kernel(const SortArgs a) {
  chain_enter(a.more_follow != 0);
  extern __shared__ __align__(16) unsigned char smem_sort[];
  const int r = blockIdx.x;
  const long long e0 = gload(a.edge_offsets + r);
  const long long Kl = min(static_cast<long long>(gload(a.edge_offsets + r + 1) - e0), static_cast<long long>(a.max_len));
  if (Kl <= 0) return;
  const int K = static_cast<int>(Kl);
  // keys that leave room for the record index in one 64-bit word (non-negative, below 2^(63 - index bits)) are
  // sorted as single words: key << shift | index orders like (key, index), needs 8 bytes per record and no
  // index array at all (the word's low bits are the index)
  if (gload(a.call_flag) == 0) return;  // the chunked kernels have sorted every list
  const int idx_bits = sort_index_bits(K);
  const bool packable = list_is_packable(a.keys_in + e0, K, idx_bits);

  if (packable && K <= a.smem_words) {
    unsigned long long* w = reinterpret_cast<unsigned long long*>(smem_sort);
    for (int i = threadIdx.x; i < K; i += blockDim.x)
      w[i] = (static_cast<unsigned long long>(gload(a.keys_in + e0 + i)) << idx_bits) | static_cast<unsigned>(i);
    __syncthreads();
    // merge sort while a thread's share of the list fits its registers, the network beyond
    if (K <= 4 * kSortThreads) sort_words_merge128(w, K);
    else if (K <= 8 * kSortThreads) sort_words_merge<8>(w, K);
    else if (K <= 16 * kSortThreads) sort_words_merge<16>(w, K);
    else sort_words_bitonic(w, K);
    const unsigned long long low = (1ull << idx_bits) - 1;
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      const unsigned long long v = w[i];
      gstore(a.keys_out + e0 + i, v >> idx_bits);
      gstore(a.perm_out + e0 + i, v & low);
    }
    return;
  }

  const bool in_smem = K <= a.smem_keys;
  long long* keys = in_smem ? reinterpret_cast<long long*>(smem_sort) : reinterpret_cast<long long*>(a.keys_out + e0);
  int* idx = in_smem ? reinterpret_cast<int*>(smem_sort + static_cast<size_t>(a.smem_keys) * 8) : a.perm_out + e0;
  if (packable) {  // only reached by lists too long for shared memory: the words live in the key output array
    unsigned long long* w = reinterpret_cast<unsigned long long*>(keys);
    for (int i = threadIdx.x; i < K; i += blockDim.x)
      w[i] = (static_cast<unsigned long long>(gload(a.keys_in + e0 + i)) << idx_bits) | static_cast<unsigned>(i);
    __syncthreads();
    sort_words_bitonic(w, K);
    const unsigned long long low = (1ull << idx_bits) - 1;
    for (int i = threadIdx.x; i < K; i += blockDim.x) {  // unpack; each thread rewrites only its own slots
      const unsigned long long v = w[i];
      idx[i] = static_cast<int>(v & low);
      keys[i] = static_cast<long long>(v >> idx_bits);
    }
    __syncthreads();
  } else {
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      keys[i] = gload(a.keys_in + e0 + i);
      idx[i] = i;
    }
    __syncthreads();
    sort_pairs_bitonic(keys, idx, K);
  }
  if (in_smem) {
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      gstore(a.keys_out + e0 + i, keys[i]);
      gstore(a.perm_out + e0 + i, idx[i]);
    }
  }
}


// ---------------------------------------------------------------------------------------------------
// Multi-block path.  One block per list leaves a 19,000-record list to a single SM while the others idle.  Here
// chunks of kSortChunk records are sorted in shared memory by one block each (packed words) and the sorted chunks
// are then merged pairwise, one launch per doubling of the run length, every block producing kSortMergeTile
// consecutive output words from the two stretches of its pair of runs that the merge path assigns to them.
// Packing needs keys that leave room for the index (non-negative, below 2^(63 - index bits)).  Every chunk block
// checks the keys it loads; one that cannot be packed sets the call's flag word, and the batch is then sorted
// list by list by sort_edges_kernel instead (what the chunked kernels wrote is overwritten).  The row gather at the
// end of the call puts the word back to zero.

__device__ __forceinline__ bool list_on_multi_path(const SortArgs& a, int r, long long& e0, int& K) {
  e0 = gload(a.edge_offsets + r);
  const long long Kl = min(static_cast<long long>(gload(a.edge_offsets + r + 1) - e0), static_cast<long long>(a.max_len));
  K = Kl > 0 ? static_cast<int>(Kl) : 0;
  // (read-only in every kernel that tests it, so the load may be cached: ten thousand blocks reading one word
  // past L1 queue up at a single L2 slice — 15 us on a 256-list batch)
  return K > 0 && gload(a.call_flag) == 0;
}

// The grids of this path have one block per (list, tile of the longest list), either folded into x with lists
// varying fastest, or lists along x and tiles along y.  Either way the blocks that have work (every list has a
// first tile, few have a twentieth) come first and the ones that leave at once are the tail of the launch.  Which
// form a kernel gets is a measurement on a 256-list batch: the row gather was 9 us faster on the two-dimensional
// grid (it falls back to the folded one when a list has more tiles than a grid has rows), the chunk and merge kernels
// together 6 us faster on the folded one.
__device__ __forceinline__ void sort_block_item(const SortArgs& a, int& r, long long& y) {
  if (gridDim.y > 1) {
    r = static_cast<int>(blockIdx.x);
    y = blockIdx.y;
  } else {
    y = blockIdx.x / static_cast<unsigned>(a.n_req);
    r = static_cast<int>(blockIdx.x - static_cast<unsigned>(y) * static_cast<unsigned>(a.n_req));
  }
}

// Merging the sorted chunks.  Phase p = 1, 2, ... merges neighbouring runs of kSortChunk << (p - 1) words into
// runs of twice that length, out of place: the words alternate between the key output array and a scratch area
// inside the list's own output rows (8 bytes per record; a row has at least 16), which
// nothing else uses until the rows are gathered at the end.  A list takes part in a phase while it is longer than
// the phase's input runs, so a list of K records goes through P = sort_merge_phases(K) phases.  Its last phase
// writes keys and source indices instead of words (a single-chunk list gets them from the chunk kernel), and so
// that this never overwrites words another block still has to read, the last phase must read from the scratch
// area: phase p reads it when P - p is even, and the chunk kernel writes there when P is odd.
__device__ __host__ __forceinline__ int sort_merge_phases(long long K) {
  int p = 0;
  while ((static_cast<long long>(kSortChunk) << p) < K) ++p;
  return p;
}
__device__ __forceinline__ unsigned long long* sort_words_at(const SortArgs& a, long long e0, bool scratch) {
  return scratch ? reinterpret_cast<unsigned long long*>(a.feats_out + e0 * a.row_ch * 16)
                 : reinterpret_cast<unsigned long long*>(a.keys_out + e0);
}

// One block per chunk of kSortChunk records of a list: the chunk sorted in shared memory, as packed words
__global__ void __launch_bounds__(kSortChunkThreads, CCR_SORT_CHUNK_BLOCKS) sort_chunks_kernel(const SortArgs a) {
  chain_enter(a.more_follow != 0);
  __shared__ unsigned long long w[kSortChunk];
  int r;
  long long y;
  sort_block_item(a, r, y);
  const long long e0 = gload(a.edge_offsets + r);
  const int K = static_cast<int>(min(static_cast<long long>(gload(a.edge_offsets + r + 1) - e0), static_cast<long long>(a.max_len)));
  if (y * kSortChunk >= K) return;  // also K <= 0
  const int c0 = static_cast<int>(y) * kSortChunk;
  const int idx_bits = sort_index_bits(K);
  const int n = min(kSortChunk, K - c0);
  int bad = 0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const long long k = gload(a.keys_in + e0 + c0 + t);
    bad |= (k < 0 || (k >> (63 - idx_bits)) != 0) ? 1 : 0;
    w[t] = (static_cast<unsigned long long>(k) << idx_bits) | static_cast<unsigned>(c0 + t);
  }
  if (__syncthreads_or(bad)) {  // a key that cannot share a word with its index: the batch goes to the one-block path
    if (threadIdx.x == 0) gatomic_or(a.call_flag, 1);
    return;
  }
  static_assert(kSortChunk == 4 * kSortChunkThreads, "a warp of a chunk block owns 128 words");
  sort_words_merge128(w, n);
  const int P = sort_merge_phases(K);
  if (P == 0) {  // the whole list: done
    const unsigned long long low = (1ull << idx_bits) - 1;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      gstore(a.keys_out + e0 + t, w[t] >> idx_bits);
      gstore(a.perm_out + e0 + t, w[t] & low);
    }
    return;
  }
  unsigned long long* W = sort_words_at(a, e0, (P & 1) != 0);
  for (int t = threadIdx.x; t < n; t += blockDim.x) gstore(W + c0 + t, w[t]);
}

// Merge path, warp-cooperative: how many of the first d words of merge(A, B) come from A.  All words are distinct
// (the record index is part of the word).  A[i] is among the first d exactly when A[i] < B[d - 1 - i]; that holds for
// i below the answer and fails from it on, so the warp probes the last element of up to 32 equal sub-ranges at once
// and narrows the range by a factor of 32 per round trip to memory (three rounds for runs of 16,384).
__device__ __forceinline__ int merge_path_warp(const unsigned long long* A, int lenA, const unsigned long long* B, int lenB,
                                               int d, int lane) {
  int lo = max(0, d - lenB), hi = min(d, lenA);
  while (lo < hi) {
    const int span = hi - lo, s = (span + 31) >> 5;
    const int i = lo + lane * s + s - 1;
    const bool before = i < hi && gload(A + i) < gload(B + d - 1 - i);
    const int cnt = __popc(__ballot_sync(0xffffffffu, before));  // the predicate is monotone: the first cnt probes hold
    const int first_fail = lo + cnt * s + s - 1;                 // probe number cnt failed or lies beyond the range
    lo += cnt * s;
    hi = min(hi, first_fail);
  }
  return lo;
}

// One block per kSortMergeTile consecutive output words of phase `phase` of a list.  Small blocks, several per
// SM: the grid is sized for the longest list, and the blocks beyond the end of a shorter one leave after reading
// the offsets — side by side rather than one after the other.
constexpr int kSortMergeThreads = 256;
constexpr int kSortMergePerThread = 4;
constexpr int kSortMergeTile = kSortMergeThreads * kSortMergePerThread;
__global__ void __launch_bounds__(kSortMergeThreads) sort_merge_kernel(const SortArgs a, int phase) {
  chain_enter(a.more_follow != 0);
  __shared__ unsigned long long w[kSortMergeTile];
  __shared__ int split[2];
  long long e0, y;
  int K, r;
  sort_block_item(a, r, y);
  const long long run = static_cast<long long>(kSortChunk) << (phase - 1);
  if (!list_on_multi_path(a, r, e0, K) || run >= K || y * kSortMergeTile >= K) return;
  const int o0 = static_cast<int>(y) * kSortMergeTile;  // first output word of this block, within the list
  const int P = sort_merge_phases(K);
  const unsigned long long* src = sort_words_at(a, e0, ((P - phase) & 1) == 0);
  unsigned long long* dst = sort_words_at(a, e0, ((P - phase) & 1) != 0);
  const int pb = static_cast<int>((o0 / (2 * run)) * (2 * run));  // the pair of runs this block's words belong to
  const int lenA = static_cast<int>(min(run, static_cast<long long>(K - pb)));
  const int lenB = static_cast<int>(min(run, static_cast<long long>(K - pb - lenA)));
  const unsigned long long* A = src + pb;
  const unsigned long long* B = A + lenA;
  const int d0 = o0 - pb, d1 = min(d0 + kSortMergeTile, lenA + lenB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < 2) {
    const int ia = merge_path_warp(A, lenA, B, lenB, warp == 0 ? d0 : d1, lane);
    if (lane == 0) split[warp] = ia;
  }
  __syncthreads();
  const int ia0 = split[0], ia1 = split[1], ib0 = d0 - ia0, ib1 = d1 - ia1;
  const int nA = ia1 - ia0, nB = ib1 - ib0, n = nA + nB;
  if (nA < 0 || nB < 0 || n > kSortMergeTile) return;  // only if the runs were not sorted: touch nothing out of range
  for (int t = threadIdx.x; t < n; t += kSortMergeThreads) w[t] = t < nA ? gload(A + ia0 + t) : gload(B + ib0 + t - nA);
  __syncthreads();
  // every thread merges kSortMergePerThread consecutive output words: its own split of the tile by binary search
  const unsigned long long* sa = w;
  const unsigned long long* sb = w + nA;
  const int d = min(static_cast<int>(threadIdx.x) * kSortMergePerThread, n);
  int lo = max(0, d - nB), hi = min(d, nA);
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (sa[mid] < sb[d - 1 - mid]) lo = mid + 1; else hi = mid;
  }
  int i = lo, j = d - lo;
  unsigned long long out[kSortMergePerThread];
#pragma unroll
  for (int u = 0; u < kSortMergePerThread; ++u) {
    const bool has_a = i < nA, has_b = j < nB;
    const unsigned long long va = has_a ? sa[i] : ~0ull, vb = has_b ? sb[j] : ~0ull;
    const bool take_a = has_a && (!has_b || va < vb);
    out[u] = take_a ? va : vb;
    i += take_a ? 1 : 0;
    j += take_a ? 0 : 1;
  }
  if (phase == P) {  // the list's last merge: keys and source indices (src is the scratch area here)
    const int idx_bits = sort_index_bits(K);
    const unsigned long long low = (1ull << idx_bits) - 1;
#pragma unroll
    for (int u = 0; u < kSortMergePerThread; ++u) {
      if (d + u < n) {
        gstore(a.keys_out + e0 + o0 + d + u, out[u] >> idx_bits);
        gstore(a.perm_out + e0 + o0 + d + u, out[u] & low);
      }
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < kSortMergePerThread; ++u)
    if (d + u < n) gstore(dst + o0 + d + u, out[u]);
}

// One block per kSortGatherTile 16-byte chunks of a list's rows: rows follow their keys, for every list of the
// batch, kSortGatherUnroll chunks per thread in flight; small blocks for the same reason as in the merge kernel
constexpr int kSortGatherThreads = 256;
constexpr int kSortGatherTile = kSortGatherThreads * kSortGatherUnroll;
__global__ void __launch_bounds__(kSortGatherThreads) gather_all_kernel(const SortArgs a) {
  chain_enter(a.more_follow != 0);
  int r;
  long long y;
  sort_block_item(a, r, y);
  if (r == 0 && y == 0 && threadIdx.x == 0) gstore(a.call_flag, 0);  // every reader of the word has finished: ready for the next call
  const long long e0 = gload(a.edge_offsets + r);
  const long long K = min(static_cast<long long>(gload(a.edge_offsets + r + 1) - e0), static_cast<long long>(a.max_len));
  const long long chunks = K * a.row_ch;
  const long long first = y * kSortGatherTile;
  if (first >= chunks) return;
  const uint4* src = reinterpret_cast<const uint4*>(a.feats_in) + e0 * a.row_ch;
  uint4* dst = reinterpret_cast<uint4*>(a.feats_out) + e0 * a.row_ch;
  const int* perm = a.perm_out + e0;
  uint4 v[kSortGatherUnroll];
#pragma unroll
  for (int u = 0; u < kSortGatherUnroll; ++u) {
    const long long c = first + static_cast<long long>(u) * kSortGatherThreads + threadIdx.x;
    if (c < chunks) {
      const int row = static_cast<int>(c / a.row_ch), piece = static_cast<int>(c - static_cast<long long>(row) * a.row_ch);
      v[u] = ldg128(src + static_cast<long long>(gload(perm + row)) * a.row_ch + piece);
    }
  }
#pragma unroll
  for (int u = 0; u < kSortGatherUnroll; ++u) {
    const long long c = first + static_cast<long long>(u) * kSortGatherThreads + threadIdx.x;
    if (c < chunks) st128_stream(dst + c, v[u]);  // written once, read by a later kernel at the earliest
  }
}

// ---------------------------------------------------------------------------------------------------
// Whole lists by radix sort, one cluster of blocks each: lists of up to kListBlockMax records per block of the cluster.
// A record's word is what its key has behind the list's common prefix, above the record's index in the list.  The words
// are sorted by the bits that differ anywhere in the list, seven a pass and lowest first (stable, so equal keys keep
// their order); a digit that is the same throughout costs nothing.  Between the passes the words are in registers: a
// warp owns 32 * R consecutive ones (R = words per thread this list needs), counts its digits, a scan over (digit, block,
// warp) turns the counts into places, and the warp hands its words out in order — into the shared memory of the block
// that owns the place — the lanes that share a digit found with one ballot per digit bit.  Keys whose differing bits
// leave no room for the index (the far outlier of a clustered list is enough) are sorted in two rounds: by their low 32
// bits, then by the rest.
// Five passes and more are replaced by three over a prefix of the differing bits when few records share one (every warp looks at 32
// records: four with the same prefix say no); the records that do share one are then put in order by comparing each with its
// neighbours, and a list where more than 64 do after all takes every pass.  Spread keys cost the same whatever their range is: one list of
// 4,096 records over 2^26 / 2^40 / 2^64 21.2 / 22.5 / 23.4 us (a pass per digit: 23.7 / 31.7 / 48.9; chunks and merges 30.5 /
// 30.5 / 73.1), 16 lists of 20,000 34.5 / 40.5 / 44.0 us (37.1 / 48.0 / 75.4; 55.7 / 55.7 / 651).  From four passes on, or by two
// digits, it does not pay: the comparing costs more than a pass (production batch 98 and 104 us).
// A pass is bound by instruction issue (about 50 instructions a word and pass; over 20,000 words on one SM 11 us), hence
// the cluster: a list takes as many blocks as hold it, the others of its cluster leave at once.  Blocks of up to 4,096
// records each, 512 threads of 8 words, 2 resident per SM: a single list of 4,096 records at 2^26 21.2 us against 25.8 with 256
// threads of 16 words, the 256-list batch below 89.8 against 87.7 (less of a pass is latency, but 8 of a block's warps idle on
// lists below half its share); less than 4,096 wanted per block is slower (cluster barriers and blocks that leave at once).
// Lists of up to kListCount records: the place of a record is the number of those in front of it (256 lists of 22 records 9.5 us by the
// network, or 14.7-22.5 for wide keys, 8.7 us this way).  Up to kListNetwork there are too few words for the passes to pay:
// sort_words_merge128, once or, for wide keys, once by each half.
// 256 lists <= 20,000 (700,000 records of 128-byte rows): 141 us as chunks and merges, 90 us this way, at 2^40 94 us.
constexpr int kListRadixBits = 7, kListDigits = 1 << kListRadixBits;
constexpr int kListStride = kListDigits + 1;  // counters of a warp; odd, so that the scan's column reads spread over the banks
constexpr int kListThreads = 512, kListPer = 8, kListWarps = kListThreads / 32;
constexpr int kListScanThreads = kListWarps / 4;  // threads that share a digit in the scan over the warps' counters
constexpr int kListBlockMax = kListThreads * kListPer;  // 4,096 words of a block: 16 registers of a thread
constexpr int kListCount = 256;     // lists up to this length are sorted by counting
constexpr int kListNetwork = 1024;  // ... up to this length as one block's merge sort behind a register network
constexpr int kListRowsHere = 512;  // batches of lists up to this length move their rows in the sorting kernel
// prefix passes: digits of the prefix, fewest passes they replace, most records that share a prefix on either side of one that are still
// put in order, most of a warp's 32 sampled records that may share one
constexpr int kListPrefixDigits = 3, kListPrefixMin = 5, kListPrefixTies = 64, kListSampleSame = 3;
static_assert(kListCount <= kListThreads, "a record per thread");
static_assert(kListNetwork <= 4 * kListThreads, "sort_words_merge128 takes four words a thread");
static_assert(kListNetwork + kListNetwork / 2 <= kListBlockMax, "wide keys keep an index per record behind their words");
static_assert(kListWarps * kListStride * 4 >= kListBlockMax, "the counters' memory holds a byte per word between the passes");
constexpr int kListMaxCluster = 8;                      // the portable size
constexpr int kListMax = kListBlockMax * kListMaxCluster;
static_assert(kListDigits * kListWarps == 4 * kListThreads, "in the scan a thread has four warps' counters of one digit");
static_assert(kListScanThreads >= 1 && 32 % kListScanThreads == 0, "a digit's counters lie within one warp");

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Barrier over the blocks of the cluster that are still running, with their shared-memory writes made visible.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t smem, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem), "r"(rank));
  return r;
}
__device__ __forceinline__ unsigned cluster_ld32(uint32_t addr) {
  unsigned v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long cluster_ld64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_st64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__global__ void __launch_bounds__(kListThreads, 2) sort_lists_kernel(const SortArgs a) {
  chain_enter(a.more_follow != 0);
  __shared__ unsigned long long w[kListBlockMax];
  __shared__ unsigned cnt[kListWarps * kListStride];       // [warp][digit]
  __shared__ unsigned block_count[kListDigits];            // this block's words with each digit, read by the whole cluster
  __shared__ unsigned digit_base[kListDigits];             // place of this block's first word with each digit
  __shared__ unsigned warp_total[kListWarps], or_bits[2], votes[2];
  // kept here and not in registers, which the passes need: the list's first record, its first key
  __shared__ volatile long long s_e0;
  __shared__ volatile unsigned long long s_key0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int cs = static_cast<int>(cluster_size()), rank = static_cast<int>(cluster_rank());
  const int list = blockIdx.x / cs;
  const long long e0 = gload(a.edge_offsets + list);
  const long long Kl = min(static_cast<long long>(gload(a.edge_offsets + list + 1) - e0), static_cast<long long>(a.max_len));
  if (Kl <= 0) return;
  const int K = static_cast<int>(Kl);
  const int blocks = min(cs, (K + kListBlockMax - 1) / kListBlockMax);
  const int R = (K + blocks * kListThreads - 1) / (blocks * kListThreads), per = R * kListThreads;  // words per thread, per block
  const int n = min(per, K - rank * per);  // words of this block
  if (rank >= blocks || n <= 0) return;    // (nobody reads the shared memory of a block without words)
  if (K <= kListCount) {  // a record per thread: its place is the number of records in front of it
    const int i = static_cast<int>(threadIdx.x);
    const int64_t k = i < K ? gload(a.keys_in + e0 + i) : 0;
    if (i < K) w[i] = static_cast<unsigned long long>(k);
    __syncthreads();
    if (i < K) {
      int p = 0;
#pragma unroll 8
      for (int j = 0; j < K; ++j) {
        const int64_t o = static_cast<int64_t>(w[j]);
        p += (o < k || (o == k && j < i)) ? 1 : 0;
      }
      gstore(a.keys_out + e0 + p, k);
      if (a.perm_out) gstore(a.perm_out + e0 + p, i);
      cnt[p] = static_cast<unsigned>(i);
    }
    if (a.rows_here) {
      __syncthreads();
      gather_rows(reinterpret_cast<const uint4*>(a.feats_in) + e0 * a.row_ch, reinterpret_cast<uint4*>(a.feats_out) + e0 * a.row_ch, K, a.row_ch,
                  [&](int row) { return static_cast<long long>(cnt[row]); });
    }
    return;
  }
  const int used_blocks = (K + per - 1) / per;
  auto sync_all = [&]() {
    if (used_blocks > 1) cluster_sync();
    else __syncthreads();
  };
  const int first = warp * 32 * R + lane;  // word r of this thread: first + 32 * r of the block's
  const int64_t* keys = a.keys_in + e0;
  const unsigned per_inv = 0xffffffffu / static_cast<unsigned>(per) + 1u;  // place / per for places below 2^16: exact

  constexpr unsigned long long kSign = 0x8000000000000000ull;  // signed keys as unsigned words of the same order
  const unsigned long long key0 = static_cast<unsigned long long>(gload(keys)) ^ kSign;
  if (threadIdx.x == 0) {
    s_e0 = e0;
    s_key0 = key0;
  }
  unsigned long long v[kListPer];
  unsigned lo = 0, hi = 0;
  if (threadIdx.x < 2) or_bits[threadIdx.x] = 0u;
#pragma unroll
  for (int r = 0; r < kListPer; ++r) {
    v[r] = key0;
    if (r < R && first + 32 * r < n) v[r] = static_cast<unsigned long long>(gload(keys + rank * per + first + 32 * r)) ^ kSign;
    lo |= static_cast<unsigned>(v[r] ^ key0);
    hi |= static_cast<unsigned>((v[r] ^ key0) >> 32);
  }
  lo = __reduce_or_sync(kFull, lo);
  hi = __reduce_or_sync(kFull, hi);
  __syncthreads();
  if (lane == 0) {
    atomicOr(or_bits, lo);
    atomicOr(or_bits + 1, hi);
  }
  sync_all();
  lo = hi = 0;
  if (used_blocks > 1) {
    if (lane < used_blocks) {
      const uint32_t at = cluster_addr(smem_u32(or_bits), static_cast<uint32_t>(lane));
      lo = cluster_ld32(at);
      hi = cluster_ld32(at + 4);
    }
    lo = __reduce_or_sync(kFull, lo);
    hi = __reduce_or_sync(kFull, hi);
  } else {
    lo = or_bits[0];
    hi = or_bits[1];
  }
  const unsigned long long used = (static_cast<unsigned long long>(hi) << 32) | lo;  // bits that differ within the list
  // No block may leave while another can still read its shared memory.  The passes end in a barrier of the whole cluster
  // behind their last remote access; a list of equal keys (`used` is the same in every block) makes no pass and needs one here.
  if (used_blocks > 1 && used == 0) cluster_sync();
  const unsigned long long suffix = used == 0 ? 0 : ~0ull >> __clzll(static_cast<long long>(used));
  const int idx_bits = sort_index_bits(K);
  const unsigned low = (1u << idx_bits) - 1u;
  const bool two = (suffix >> (63 - idx_bits)) != 0;
#pragma unroll
  for (int r = 0; r < kListPer; ++r)
    v[r] = ((v[r] & (two ? 0xffffffffull : suffix)) << idx_bits) | static_cast<unsigned>(rank * per + first + 32 * r);

  const auto key_at = [&](unsigned i) { return static_cast<unsigned long long>(gload(a.keys_in + s_e0 + i)) ^ kSign; };
  const bool network = K <= kListNetwork;
  if (network) {
    unsigned* from = reinterpret_cast<unsigned*>(w + kListNetwork);  // wide keys: the record at each place of the first round
    for (int round = 0;; ++round) {
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) w[first + 32 * r] = v[r];
      __syncthreads();
      sort_words_merge128(w, n);
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) v[r] = w[first + 32 * r];
      if (!two || round == 1) break;
      // sorted by the low half; the second round is by the high half and, so that equal ones keep this order, the place
#pragma unroll
      for (int r = 0; r < kListPer; ++r) {
        if (r < R && first + 32 * r < n) {
          const unsigned i = static_cast<unsigned>(v[r]) & low;
          from[first + 32 * r] = i;
          v[r] = ((key_at(i) >> 32) << idx_bits) | static_cast<unsigned>(first + 32 * r);
        }
      }
    }
    if (two) {
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) v[r] = from[static_cast<unsigned>(v[r]) & low];  // (the key is read from the input below)
    }
  }
  // the words of the records this thread holds: key bits of `mask`, those below `base` left out
  const auto make_words = [&](unsigned long long mask, int base) {
#pragma unroll
    for (int r = 0; r < kListPer; ++r) {
      if (r < R && first + 32 * r < n) {
        const unsigned i = static_cast<unsigned>(v[r]) & low;
        v[r] = (((key_at(i) & mask) >> base) << idx_bits) | i;
      }
    }
  };
  const auto any_of_list = [&](bool mine, int slot) -> bool {
    const int here = __syncthreads_or(mine);
    if (used_blocks == 1) return here != 0;
    if (threadIdx.x == 0) votes[slot] = static_cast<unsigned>(here);
    cluster_sync();
    const unsigned x = lane < used_blocks ? cluster_ld32(cluster_addr(smem_u32(votes + slot), static_cast<uint32_t>(lane))) : 0u;
    return __any_sync(kFull, x != 0);
  };
  const auto put_word = [&](unsigned p, unsigned long long x) {  // to place p of the list
    if (used_blocks > 1) {
      const unsigned q = __umulhi(p, per_inv);
      cluster_st64(cluster_addr(smem_u32(w + (p - q * per)), q), x);
    } else {
      w[p] = x;
    }
  };
  const auto word_at = [&](unsigned p) {
    if (used_blocks == 1) return w[p];
    const unsigned q = __umulhi(p, per_inv);
    return q == static_cast<unsigned>(rank) ? w[p - q * per] : cluster_ld64(cluster_addr(smem_u32(w + (p - q * per)), q));
  };
  const auto digits_of = [](unsigned long long m) {
    int c = 0;
    for (; m != 0; ++c) m &= ~(static_cast<unsigned long long>(kListDigits - 1) << (__ffsll(static_cast<long long>(m)) - 1));
    return c;
  };

  const unsigned long long low_used = two ? used & 0xffffffffull : used;
  const int passes = network ? 0 : digits_of(low_used) + (two ? digits_of(used >> 32) : 0);
  int drop = 0, cut = 0;  // prefix passes: key bits left out of the word to make room for the index, lowest key bit of the prefix
  bool prefix = passes >= kListPrefixMin;
  if (prefix) {
    unsigned long long m = used;
#pragma unroll
    for (int d = 0; d < kListPrefixDigits; ++d) {
      if (m != 0) cut = max(64 - kListRadixBits - __clzll(static_cast<long long>(m)), 0);
      m &= (1ull << cut) - 1;
    }
    drop = two ? 1 + idx_bits - __clzll(static_cast<long long>(used)) : 0;
    prefix = cut >= drop;
  }
  if (prefix) {
    const bool live = first < n;
    unsigned long long t = ~static_cast<unsigned long long>(lane);
    if (live) t = two ? (key_at(static_cast<unsigned>(rank * per + first)) & suffix) >> cut : v[0] >> (idx_bits + cut);
    prefix = !any_of_list(__popc(__match_any_sync(kFull, t)) > kListSampleSame, 0);
    if (prefix && two) make_words(suffix, drop);
  }
  for (int round = 0; passes > 0; ++round) {
    if (round == 1) make_words(~0ull << 32, 32);
    const int base = prefix ? drop : (round == 1 ? 32 : 0);  // the key bit that is the word's lowest
    unsigned long long bits = (prefix ? (used >> cut) << cut : (round == 1 ? used : low_used)) >> base;
    while (bits != 0) {
      const int bit = __ffsll(static_cast<long long>(bits)) - 1, shift = idx_bits + bit;
      bits &= ~(static_cast<unsigned long long>(kListDigits - 1) << bit);
      for (int t = threadIdx.x; t < kListWarps * kListStride; t += kListThreads) cnt[t] = 0u;
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) atomicAdd(cnt + warp * kListStride + (static_cast<unsigned>(v[r] >> shift) & (kListDigits - 1)), 1u);
      __syncthreads();
      // counts -> places: a thread has four warps' counters of digit d; kListScanThreads neighbouring threads share a digit
      const int d = threadIdx.x / kListScanThreads, part = threadIdx.x % kListScanThreads, w0 = part * 4;
      unsigned c[4], sum = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        c[j] = cnt[(w0 + j) * kListStride + d];
        sum += c[j];
      }
      unsigned upto = sum;  // words with digit d of this thread's warps and the ones before them
#pragma unroll
      for (int s = 1; s < kListScanThreads; s <<= 1) {
        const unsigned t = __shfl_up_sync(kFull, upto, s);
        if (part >= s) upto += t;
      }
      const unsigned in_block = __shfl_sync(kFull, upto, lane | (kListScanThreads - 1));
      if (part == 0) block_count[d] = in_block;
      sync_all();
      unsigned total = in_block, before_me = 0;  // words with digit d in the list, in the blocks before this one
      if (used_blocks > 1) {
        total = 0;
        const uint32_t mine = smem_u32(block_count + d);
#pragma unroll
        for (int q = 0; q < kListMaxCluster; ++q) {
          if (q < used_blocks) {
            const unsigned x = cluster_ld32(cluster_addr(mine, static_cast<uint32_t>(q)));
            total += x;
            before_me += q < rank ? x : 0u;
          }
        }
      }
      unsigned incl = part == 0 ? total : 0u;  // one of the threads of a digit carries it
      const unsigned own = incl;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const unsigned t = __shfl_up_sync(kFull, incl, s);
        if (lane >= s) incl += t;
      }
      if (lane == 31) warp_total[warp] = incl;
      __syncthreads();
      const unsigned warps_before = __reduce_add_sync(kFull, lane < warp ? warp_total[lane & (kListWarps - 1)] : 0u);
      if (part == 0) digit_base[d] = warps_before + incl - own + before_me;
      __syncwarp();
      unsigned at = digit_base[d] + upto - sum;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        cnt[(w0 + j) * kListStride + d] = at;
        at += c[j];
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kListPer; ++r) {
        if (r < R && first - lane + 32 * r < n) {  // warp-uniform
          const bool live = first + 32 * r < n;
          const unsigned dg = static_cast<unsigned>(v[r] >> shift) & (kListDigits - 1);
          unsigned same = __ballot_sync(kFull, live);
#pragma unroll
          for (int b = 0; b < kListRadixBits; ++b) {
            const unsigned vote = __ballot_sync(kFull, (dg >> b) & 1u);
            same &= ((dg >> b) & 1u) ? vote : ~vote;
          }
          const unsigned before = __popc(same & lt);
          unsigned* c2 = cnt + warp * kListStride + dg;
          const unsigned start = *c2;
          __syncwarp();
          if (live && before == 0) *c2 = start + __popc(same);
          __syncwarp();
          if (live) {
            const unsigned p = start + before;
            put_word(p, v[r]);
          }
        }
      }
      sync_all();
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) v[r] = w[first + 32 * r];      // (the next pass writes any block's w only behind a barrier that every block reaches after these loads)
    }
    if (!prefix) {
      if (!two || round == 1) break;
      continue;
    }
    // Words with the same prefix stand together.  Each counts those in front of it that belong behind it, and the reverse.
    const int tie = idx_bits + cut - drop;
    signed char* moved = reinterpret_cast<signed char*>(cnt);  // by how many places; a byte per word of the block
    bool too_many = false;
#pragma unroll 4
    for (int r = 0; r < R; ++r) {
      const int e = first + 32 * r, p = rank * per + e;
      if (e >= n) break;
      const unsigned long long x = w[e];
      const unsigned long long before = e > 0 ? w[e - 1] : (rank > 0 ? word_at(static_cast<unsigned>(p - 1)) : ~x);
      const unsigned long long after = e < n - 1 ? w[e + 1] : (p < K - 1 ? word_at(static_cast<unsigned>(p + 1)) : ~x);
      int by = 0;
      if ((before >> tie) == (x >> tie) || (after >> tie) == (x >> tie)) {
        for (int side = -1; side <= 1; side += 2) {
          for (int q = p + side; q >= 0 && q < K; q += side) {
            const unsigned long long u = word_at(static_cast<unsigned>(q));
            if ((u >> tie) != (x >> tie)) break;
            if (side * (q - p) > kListPrefixTies) {
              too_many = true;
              break;
            }
            bool u_first = u < x;
            if (drop > 0 && (u >> idx_bits) == (x >> idx_bits)) {  // the bits that were left out decide
              const unsigned long long ku = key_at(static_cast<unsigned>(u) & low), kx = key_at(static_cast<unsigned>(x) & low);
              u_first = ku != kx ? ku < kx : u_first;
            }
            if (u_first == (side > 0)) by += side;
          }
        }
      }
      moved[e] = static_cast<signed char>(by);
    }
    if (!any_of_list(too_many, 1)) {
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) put_word(static_cast<unsigned>(rank * per + first + 32 * r + moved[first + 32 * r]), v[r]);
      sync_all();
#pragma unroll
      for (int r = 0; r < kListPer; ++r)
        if (r < R && first + 32 * r < n) v[r] = w[first + 32 * r];
      break;
    }
    // too many share a prefix after all: all passes, from the words as they stand (equal keys have kept their order)
    prefix = false;
    make_words(two ? 0xffffffffull : suffix, 0);
    round = -1;
  }
#pragma unroll
  for (int r = 0; r < kListPer; ++r) {
    const int e = first + 32 * r;
    if (r < R && e < n) {
      const unsigned i = static_cast<unsigned>(v[r]) & low;
      const long long k = two ? static_cast<long long>(key_at(i) ^ kSign) : static_cast<long long>(((s_key0 & ~suffix) | (v[r] >> idx_bits)) ^ kSign);
      gstore(a.keys_out + s_e0 + rank * per + e, k);
      if (a.perm_out) gstore(a.perm_out + s_e0 + rank * per + e, static_cast<int>(i));
      if (a.rows_here) w[e] = v[r];
    }
  }
  if (a.rows_here) {
    __syncthreads();
    gather_rows(reinterpret_cast<const uint4*>(a.feats_in) + s_e0 * a.row_ch, reinterpret_cast<uint4*>(a.feats_out) + (s_e0 + rank * per) * a.row_ch,
                n, a.row_ch, [&](int row) { return static_cast<long long>(static_cast<unsigned>(w[row]) & low); });
  }
}

// Rows of sorted lists follow the permutation.  Work is dealt out in units of kSortRowsTile records of the flat record
// range: list r owns the items [start(r), start(r + 1)), start(r) = e_r / unit - e_0 / unit + r, at least as many as its
// units, so no block is launched for a length that a list does not have; a warp finds an item's list by a 32-way search.
constexpr int kSortRowsTileLog = 8, kSortRowsTile = 1 << kSortRowsTileLog;
__global__ void __launch_bounds__(kSortRowsTile) sort_rows_kernel(const SortArgs a) {
  chain_enter(false);
  __shared__ int s_src[kSortRowsTile];
  const int lane = threadIdx.x & 31;
  const long long base = gload(a.edge_offsets) >> kSortRowsTileLog;
  const long long n_items = (gload(a.edge_offsets + a.n_req) >> kSortRowsTileLog) - base + a.n_req;
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    int r = 0, m = a.n_req;
    while (m > 1) {
      const int step = (m + 31) >> 5, p = r + lane * step;
      const bool holds = lane * step < m && (gload(a.edge_offsets + p) >> kSortRowsTileLog) - base + p <= item;
      const int c = max(1, __popc(__ballot_sync(kFull, holds)));  // starts ascend: the first c probes hold
      r += (c - 1) * step;
      m = min(step, m - (c - 1) * step);
    }
    const long long e0 = gload(a.edge_offsets + r);
    const long long K = min(static_cast<long long>(gload(a.edge_offsets + r + 1) - e0), static_cast<long long>(a.max_len));
    const long long first = (item - ((e0 >> kSortRowsTileLog) - base + r)) << kSortRowsTileLog;
    if (first < 0 || first >= K) continue;  // block-uniform
    const int n = static_cast<int>(min(static_cast<long long>(kSortRowsTile), K - first));
    if (static_cast<int>(threadIdx.x) < n) s_src[threadIdx.x] = gload(a.perm_out + e0 + first + threadIdx.x);
    __syncthreads();
    gather_rows(reinterpret_cast<const uint4*>(a.feats_in) + e0 * a.row_ch, reinterpret_cast<uint4*>(a.feats_out) + (e0 + first) * a.row_ch,
                n, a.row_ch, [&](int row) { return static_cast<long long>(s_src[row]); });
    __syncthreads();  // s_src is rewritten by the next item
  }
}

}  // namespace ccr
