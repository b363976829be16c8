// Document-id resolution on the GPU (Section 6.3.1 of the paper, "Document ID Resolution", Eq. 6):
// pos(q) = position of id q in the index, or -1.  The paper stored the id -> position map as a sorted array
// in HBM, resolved queries with a binary-search kernel (~5 ms per request over a few hundred million ids,
// ~47 ms at batch 8, every probe a dependent HBM access) and then moved the step to a CPU hash map.
//
// Here the sorted ids are cut into regions of up to kIdRegion consecutive ones, and every region is a small hash table in
// HBM: buckets of one 32-byte sector that hold the ids and their positions.  A query finds its region by the regions' last ids
// (a static search tree of sampled levels, fan-out 8, whose top level sits in shared memory; up to 8.4M ids that is all of
// it) and then reads one sector, seldom two.  What bounds a query is the number of random reads: HBM serves about 35 G of them a
// second whatever their width up to 64 bytes, L2 150-220 G, and the sector is read a lane per query (a 64-byte bucket read by
// four lanes took 27 us where this takes 12, 1.92M queries in L2).  A tree down to the ids, which this replaces, read a 64-byte
// window per level: six dependent rounds over 300M ids, two or three of them from HBM.
// A region is built in shared memory by one block and written once, front to back: building costs about what copying the
// ids does (one table over 300M ids filled by global atomics takes 18-30 ms).
#pragma once

#include "ccr_device.cuh"

namespace ccr {

constexpr int kIdRegionLog = 12;
constexpr long long kIdRegion = 1LL << kIdRegionLog;  // most ids of a region: its table is built in shared memory
constexpr int kResolveFanLog2 = 3;                 // 8 keys = one 64-byte window per level
constexpr int kResolveMaxLevels = 5;               // 2,048 x 8^4 regions: more than int32 positions can name
constexpr int kResolveTopMax = 2048;               // keys of the top level (16 KB of shared memory)
constexpr int kResolveThreads = 256;
constexpr int kResolveBlocksPerSm = 8;
constexpr int kResolveUnroll = 4;                  // queries a group of lanes descends with at a time
constexpr int kIdBuildThreads = 512;
constexpr unsigned kIdBucketSmem = 36;             // shared memory of a bucket while its region is built: the sector and a counter
constexpr long long kResolveInf = 0x7fffffffffffffffLL;  // stands for the keys beyond the end of a level

// A bucket is a 32-byte sector.  Narrow: four entries {low 32 bits of the id, position}, used when the ids of every region span
// less than 2^32, so that the low bits name an id within its region.  Wide: two entries {id, position, unused}.  Slots without an
// id repeat the first entry (so a bucket is full exactly when its last entry differs from its first); a bucket without any
// repeats the region's first id, which no query that belongs there can equal.  An id that finds its bucket full goes to the
// next one of the region that is not: a query that finds no match in a full bucket goes on there.
template <bool WIDE>
struct IdBucket {
  static constexpr int kSlots = WIDE ? 2 : 4, kStep = 8 / kSlots;  // entries, words from one to the next
  static __host__ __device__ unsigned buckets(long long ids) { return static_cast<unsigned>(WIDE ? ids + 1 : ids / 2 + 1); }
  static __device__ __forceinline__ void put(unsigned* e, int64_t id, int pos) {
    e[0] = static_cast<unsigned>(id);
    if (WIDE) e[1] = static_cast<unsigned>(static_cast<unsigned long long>(id) >> 32);
    e[WIDE ? 2 : 1] = static_cast<unsigned>(pos);
  }
  static __device__ __forceinline__ bool holds(const U32x8& x, int s, int64_t id) {
    return x.v[s * kStep] == static_cast<unsigned>(id) && (!WIDE || x.v[s * kStep + 1] == static_cast<unsigned>(static_cast<unsigned long long>(id) >> 32));
  }
  static __device__ __forceinline__ int pos(const U32x8& x, int s) { return static_cast<int>(x.v[s * kStep + (WIDE ? 2 : 1)]); }
  static __device__ __forceinline__ bool full(const U32x8& x) {
    const int l = (kSlots - 1) * kStep;
    return x.v[l] != x.v[0] || (WIDE && x.v[l + 1] != x.v[1]);
  }
};

struct ResolveArgs {
  const int64_t* level[kResolveMaxLevels];  // level[0] = last id of every region but the last, level[n_levels - 1] = top
  int count[kResolveMaxLevels];
  int n_levels;
  const unsigned* table;                    // [n_regions][n_buckets][8]
  unsigned n_buckets;                       // of a region
  int64_t min_id, max_id;
  long long n_queries;
  const int64_t* queries;
  int32_t* out_pos;
};

// Every bit of the id reaches the high bits, whatever regular pattern the ids follow: xor-shift and multiply, twice, with the multiplier of
// the public 64-bit mixer known as degski64 (in C. Wellons's hash-prospector collection).
__device__ __forceinline__ unsigned id_bucket(int64_t id, unsigned n_buckets) {
  unsigned long long h = static_cast<unsigned long long>(id);
  h = (h ^ (h >> 32)) * 0xD6E8FEB86659FD93ull;
  h = (h ^ (h >> 32)) * 0xD6E8FEB86659FD93ull;
  return __umulhi(static_cast<unsigned>(h >> 32), n_buckets);
}

// Regions first_region .. first_region + gridDim.x - 1 of an index of n ids, `per_region` each; ids[0] is the first one of them.
template <bool WIDE>
__global__ void __launch_bounds__(kIdBuildThreads) build_regions_kernel(const int64_t* ids, const int32_t* positions, long long n, int per_region,
                                                                        long long first_region, unsigned* table, unsigned n_buckets) {
  using Bucket = IdBucket<WIDE>;
  extern __shared__ __align__(16) unsigned char smem_build[];
  unsigned* tab = reinterpret_cast<unsigned*>(smem_build);
  unsigned* came = tab + n_buckets * 8;  // ids that came to a bucket, those that found it full included
  const long long region = first_region + blockIdx.x, rank0 = region * per_region, at0 = static_cast<long long>(blockIdx.x) * per_region;
  const int m = static_cast<int>(min(static_cast<long long>(per_region), n - rank0));
  for (unsigned b = threadIdx.x; b < n_buckets; b += kIdBuildThreads) came[b] = 0u;
  __syncthreads();
#pragma unroll 4
  for (int i = threadIdx.x; i < m; i += kIdBuildThreads) {
    const int64_t id = ids[at0 + i];
    if (i > 0 && ids[at0 + i - 1] == id) continue;  // a repeated id: the first occurrence answers
    unsigned b = id_bucket(id, n_buckets), s;
    while ((s = atomicAdd(came + b, 1u)) >= static_cast<unsigned>(Bucket::kSlots)) b = b + 1 == n_buckets ? 0u : b + 1;
    Bucket::put(tab + b * 8 + s * Bucket::kStep, id, positions != nullptr ? positions[at0 + i] : static_cast<int>(rank0 + i));
  }
  __syncthreads();
  // out they go, half a bucket a thread, the slots without an id filled on the way
  const uint4* from = reinterpret_cast<const uint4*>(tab);
  uint4* to = reinterpret_cast<uint4*>(table + static_cast<size_t>(region) * n_buckets * 8);
  const int64_t id0 = ids[at0];
  const int pos0 = positions != nullptr ? positions[at0] : static_cast<int>(rank0);
  for (unsigned c = threadIdx.x; c < n_buckets * 2; c += kIdBuildThreads) {
    const unsigned b = c >> 1, got = came[b], s = (c & 1u) * (Bucket::kSlots / 2);  // s: first slot of this half
    uint4 x = from[c];
    if (WIDE) {
      if (got <= s) x = got > 0 ? from[c - 1] : make_uint4(static_cast<unsigned>(id0), static_cast<unsigned>(static_cast<unsigned long long>(id0) >> 32), static_cast<unsigned>(pos0), 0u);
      x.w = 0u;
    } else if (got <= s + 1) {
      uint2 f = make_uint2(static_cast<unsigned>(id0), static_cast<unsigned>(pos0));
      if (got > 0) f = *reinterpret_cast<const uint2*>(tab + b * 8);
      if (got <= s) {
        x.x = f.x;
        x.y = f.y;
      }
      x.z = f.x;
      x.w = f.y;
    }
    to[c] = x;
  }
}

// Last ids of all regions but the last one, and whether the ids of some region (with the gap in front of it) span 2^32 or more.
__global__ void region_ends_kernel(const int64_t* ids, long long n, int per_region, int64_t* last, int n_regions, int* wide) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_regions) return;
  const int64_t end = ids[min(n, static_cast<long long>(r + 1) * per_region) - 1];
  const int64_t begin = ids[r > 0 ? static_cast<long long>(r) * per_region - 1 : 0];
  if (r < n_regions - 1) last[r] = end;
  if (((static_cast<unsigned long long>(end) - static_cast<unsigned long long>(begin)) >> 32) != 0) atomicExch(wide, 1);
}

__global__ void build_level_kernel(const int64_t* below, int64_t* above, int n_above) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_above) above[i] = below[((static_cast<long long>(i) + 1) << kResolveFanLog2) - 1];
}

// Every level is followed by kResolvePad keys of +infinity, so that the window a query reads (window c of a level
// with n keys, c <= n / 8) needs no bounds checks; the allocation of a level leaves room for them.
constexpr int kResolvePad = 2 << kResolveFanLog2;
__global__ void pad_level_kernel(int64_t* level, int n) {
  if (threadIdx.x < kResolvePad) level[n + threadIdx.x] = kResolveInf;
}

// 16-byte window piece of a level.
__device__ __forceinline__ longlong2 resolve_load(const longlong2* p) {
  if (!CCR_CHK(p, 16)) return make_longlong2(kResolveInf, kResolveInf);  // reads like the padding behind a level
  return __ldg(p);
}

// A warp takes 32 queries at a time, a lane each: the search of the top level, and at the end the sector of the bucket.  DESCEND:
// there are levels below the top; for their windows the queries are handed by shuffles to groups of G lanes that share a
// query, 16 bytes of the window each, kResolveUnroll groups of queries in flight.
template <bool DESCEND, bool WIDE>
__global__ void __launch_bounds__(kResolveThreads, DESCEND ? 5 : kResolveBlocksPerSm) resolve_kernel(const __grid_constant__ ResolveArgs a) {
  chain_enter(false);
  extern __shared__ __align__(16) unsigned char smem_res[];
  using Bucket = IdBucket<WIDE>;
  int64_t* top = reinterpret_cast<int64_t*>(smem_res);
  const int top_l = a.n_levels - 1, n_top = a.count[top_l];
  const int lane = threadIdx.x & 31;
  const long long step = static_cast<long long>(gridDim.x) * kResolveThreads;
  long long first = blockIdx.x * static_cast<long long>(kResolveThreads) + (threadIdx.x & ~31u);
  int64_t q = first + lane < a.n_queries ? gload(a.queries + first + lane) : 0;
  for (int i = threadIdx.x; i < n_top; i += kResolveThreads) top[i] = gload(a.level[top_l] + i);
  __syncthreads();
  while (first < a.n_queries) {  // warp-uniform
    unsigned region = static_cast<unsigned>(lower_bound_smem(top, n_top, q));  // keys of the level below q
    if constexpr (DESCEND) {
      constexpr int G = 1 << (kResolveFanLog2 - 1), kPerRound = 32 / G;
      const unsigned sub = lane & (G - 1);
      constexpr int kParts = 32 / (kPerRound * kResolveUnroll);
      static_assert(kParts * kResolveUnroll * kPerRound == 32, "the queries of a warp are handed out in whole rounds");
      const unsigned above = region;
#pragma unroll 1
      for (int part = 0; part < kParts; ++part) {
        unsigned c[kResolveUnroll];
        int64_t qg[kResolveUnroll];
#pragma unroll
        for (int u = 0; u < kResolveUnroll; ++u) {
          const int src = (part * kResolveUnroll + u) * kPerRound + lane / G;
          qg[u] = __shfl_sync(kFull, q, src);
          c[u] = __shfl_sync(kFull, above, src);
        }
        // c keys of level l + 1 below q: windows 0..c-1 of level l are below q, the answer is in window c
        for (int l = top_l - 1; l >= 0; --l) {
          const longlong2* lev = reinterpret_cast<const longlong2*>(a.level[l]);
          longlong2 k[kResolveUnroll];
#pragma unroll
          for (int u = 0; u < kResolveUnroll; ++u) k[u] = resolve_load(lev + (static_cast<size_t>(c[u]) * G + sub));
#pragma unroll
          for (int u = 0; u < kResolveUnroll; ++u) {
            unsigned v = (k[u].x < qg[u] ? 1u : 0u) + (k[u].y < qg[u] ? 1u : 0u);
#pragma unroll
            for (int d = 1; d < G; d <<= 1) v += __shfl_xor_sync(kFull, v, d);
            c[u] = (c[u] << kResolveFanLog2) + v;
          }
        }
#pragma unroll
        for (int u = 0; u < kResolveUnroll; ++u) {  // back to the lane that asked
          const unsigned v = __shfl_sync(kFull, c[u], (lane % kPerRound) * G);
          if (lane / kPerRound == part * kResolveUnroll + u) region = v;
        }
      }
    }
    const long long j = first + lane;
    int pos = -1;
    if (j < a.n_queries && q >= a.min_id && q <= a.max_id) {
      const unsigned* sectors = a.table + static_cast<size_t>(region) * a.n_buckets * 8;
      unsigned b = id_bucket(q, a.n_buckets);
      for (;;) {
        const U32x8 x = ldg256(sectors + static_cast<size_t>(b) * 8);
        bool hit = false;
#pragma unroll
        for (int s = 0; s < Bucket::kSlots; ++s) {
          if (Bucket::holds(x, s, q)) {
            hit = true;
            pos = Bucket::pos(x, s);
          }
        }
        if (hit || !Bucket::full(x)) break;
        b = b + 1 == a.n_buckets ? 0u : b + 1;
      }
    }
    first += step;
    q = first + lane < a.n_queries ? gload(a.queries + first + lane) : 0;
    if (j < a.n_queries) gstore(a.out_pos + j, pos);
    __syncwarp();
  }
}

}  // namespace ccr
