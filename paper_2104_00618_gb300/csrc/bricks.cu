// Brick occupancy and slot tables of a VCT_LAYOUT_BRICKS pyramid (Ch. 5.1:
// sparse storage in place of a full 3D texture): which 8^3 bricks of every
// bricked level hold a non-zero texel, and where in the pool each occupied
// brick goes.
#include <algorithm>

#include "vct_internal.cuh"

namespace vct {

namespace {

struct TableArgs {
  uint32_t *tbl[VCT_MAX_LEVELS];  // slot table of each bricked level
  uint64_t nb[VCT_MAX_LEVELS];    // bricks of each bricked level
  int nbricked;                   // bricked levels are 0 .. nbricked-1
  uint32_t *status;
  unsigned long long *count;
  uint32_t *plan;                 // the tables' shape word (plan_word)
  uint64_t capacity;              // pool bricks, the zero brick included
};

// One warp per level-0 brick: where any channel of its 512 texels is
// non-zero, the brick and the bricks above it in every bricked level are
// flagged (the flags start at 0; warps that share a coarser brick store the
// same 1); `small`: each level-0 flag is written, 0 or 1, and no other.  level0
// is dense [z][y][x][4]; the brick's rows of 8 texels are 128 bytes.  512^3:
// 0.32 ms for 2.15 GB, the HBM copy rate.
__global__ void __launch_bounds__(256) occupancy_kernel(const float4 *level0, int n,
                                                        const __grid_constant__ TableArgs a,
                                                        bool small) {
  const int lane = threadIdx.x & 31;
  const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t b = warp; b < a.nb[0]; b += nwarps) {
    const uint32_t id = (uint32_t)b;  // Morton id of the brick
    const int bx = compact3(id), by = compact3(id >> 1), bz = compact3(id >> 2);
    bool any = false;
    // lane k reads texels k, k + 32, ...: each pass covers 4 rows of 8 texels
    for (int k = lane; k < 512; k += 32) {
      const int x = k & 7, y = (k >> 3) & 7, z = k >> 6;
      const float4 v = __ldcs(level0 + ((size_t)(8 * bz + z) * n + (8 * by + y)) * n + 8 * bx + x);
      any |= (v.x != 0.0f) | (v.y != 0.0f) | (v.z != 0.0f) | (v.w != 0.0f);
    }
    any = __any_sync(0xffffffffu, any);
    if (small) {
      if (lane == 0) a.tbl[0][id] = any ? 1u : 0u;
    } else if (any && lane < a.nbricked) {
      a.tbl[lane][id >> (3 * lane)] = 1u;
    }
  }
}

// Flags -> slots, by an exclusive scan over all bricked levels in level order:
// the tables follow one another without gaps (a level of 64 bricks or more
// fills 256-byte lines, the last one has 8), so they are scanned as one array.
// kScanCtas CTAs take a part each; count_kernel leaves the parts' sums in the
// header's free words, slots_kernel adds those before its own.  At 512^3 (300 K
// flags) one CTA alone took 232 us with one flag per thread and pass, 69 us
// with 16 (its SM's share of the L2 bandwidth).
constexpr int kScanThreads = 1024;
constexpr int kScanRun = 8;    // consecutive flags per thread and pass
constexpr int kScanCtas = 56;  // sums in header words 4 .. 59
constexpr int kScanPass = kScanThreads * kScanRun;
static_assert(16 + 4 * kScanCtas <= kHeaderPlanOff, "the parts' sums lie in the header");

struct ScanArgs {
  uint32_t *flags, *sums;  // sums: null where one pass of one CTA holds every flag
  uint64_t words, part;  // part: words per CTA, a multiple of kScanPass
  uint64_t bricks0;      // level 0's
  uint32_t *status;
  unsigned long long *count;
  uint64_t capacity;
  uint32_t *plan;  // the tables' shape word (plan_word)
  uint32_t plan_value;
};

__device__ __forceinline__ uint32_t load_flags(const ScanArgs &a, uint64_t e, uint64_t end) {
  uint32_t f = 0u;
#pragma unroll
  for (int j = 0; j < kScanRun / 4; ++j) {
    if (e + 4 * j >= end) break;
    const uint4 v = *reinterpret_cast<const uint4 *>(a.flags + e + 4 * j);
    f |= (v.x | v.y << 1 | v.z << 2 | v.w << 3) << (4 * j);
  }
  return f;
}

__global__ void __launch_bounds__(kScanThreads) count_kernel(const __grid_constant__ ScanArgs a) {
  __shared__ uint32_t s_sum;
  if (threadIdx.x == 0) s_sum = 0u;
  __syncthreads();
  const uint64_t begin = blockIdx.x * a.part, end = min(begin + a.part, a.words);
  uint32_t n = 0u;
  for (uint64_t e = begin + (uint64_t)threadIdx.x * kScanRun; e < end; e += kScanPass)
    n += __popc(load_flags(a, e, end));
  n = __reduce_add_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(&s_sum, n);
  __syncthreads();
  if (threadIdx.x == 0) a.sums[blockIdx.x] = s_sum;
}

__global__ void __launch_bounds__(kScanThreads) slots_kernel(const __grid_constant__ ScanArgs a) {
  __shared__ uint32_t s_warp[2][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // (every warp sums the parts; kScanCtas <= 64)
  uint32_t before_part = 0u, total = 0u;
  for (int i = lane; a.sums != nullptr && i < (int)gridDim.x; i += 32) {
    const uint32_t c = a.sums[i];
    total += c;
    if (i < (int)blockIdx.x) before_part += c;
  }
  total = __reduce_add_sync(0xffffffffu, total);
  if (a.sums == nullptr) {  // one part of one pass: the coarser flags and the count here
    const uint32_t *child = a.flags;
    // (nb: bricks of the next level, whose flags start at `at`)
    for (uint64_t nb = a.bricks0 >> 3, at = a.bricks0; at < a.words; at += nb, nb >>= 3) {
      for (uint64_t p = threadIdx.x; p < nb; p += blockDim.x) {
        const uint4 u = *reinterpret_cast<const uint4 *>(child + 8 * p);
        const uint4 v = *reinterpret_cast<const uint4 *>(child + 8 * p + 4);
        a.flags[at + p] = u.x | u.y | u.z | u.w | v.x | v.y | v.z | v.w;
      }
      child = a.flags + at;
      __syncthreads();
    }
    const uint64_t e = (uint64_t)threadIdx.x * kScanRun;
    const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(load_flags(a, e, a.words)));
    if (lane == 0) s_warp[1][wid] = c;
    __syncthreads();
    total = __reduce_add_sync(0xffffffffu, s_warp[1][lane]);
  }
  uint32_t run = 1u + __reduce_add_sync(0xffffffffu, before_part);  // next slot of this part
  const bool fits = 1ull + total <= a.capacity;  // else: leave every brick empty, report it
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.count = total;
    *a.plan = a.plan_value;
    if (!fits) atomicExch(a.status, (uint32_t)VCT_ERR_WORKSPACE);
  }
  const uint64_t begin = blockIdx.x * a.part, end = min(begin + a.part, a.words);
  int pass = 0;
  for (uint64_t base = begin; base < end; base += kScanPass, ++pass) {
    const uint64_t e = base + (uint64_t)threadIdx.x * kScanRun;
    const uint32_t f = load_flags(a, e, end);
    const uint32_t cnt = __popc(f);
    uint32_t x = cnt;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, m);
      if (lane >= m) x += y;
    }
    uint32_t *sw = s_warp[pass & 1];
    if (lane == 31) sw[wid] = x;
    __syncthreads();  // (the other half of s_warp may still be read)
    uint32_t w = sw[lane];
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, m);
      if (lane >= m) w += y;
    }
    const uint32_t before = __shfl_sync(0xffffffffu, w, (wid + 31) & 31);
    // slot 1 + (occupied bricks before this one); 0 for an empty brick
    uint32_t slot = run + (wid ? before : 0u) + x - cnt;
#pragma unroll
    for (int j = 0; j < kScanRun / 4; ++j) {
      if (e + 4 * j >= end) break;
      uint4 o;
      o.x = (f >> (4 * j)) & 1u ? slot++ : 0u;
      o.y = (f >> (4 * j + 1)) & 1u ? slot++ : 0u;
      o.z = (f >> (4 * j + 2)) & 1u ? slot++ : 0u;
      o.w = (f >> (4 * j + 3)) & 1u ? slot++ : 0u;
      if (!fits) o = make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4 *>(a.flags + e + 4 * j) = o;
    }
    run += __shfl_sync(0xffffffffu, w, 31);
  }
}

// Tables and brick count made elsewhere for the same grid shape (`src`: the
// words at the tables' place there) into this pyramid; slots_kernel's check
// of the pool.  Those words are the caller's: tables of another shape are
// taken as a pool too small, and a slot above the count, which slots_kernel
// never hands out, becomes (with the rest of its four words) that of an empty
// brick, so that no slot outside the pool reaches the kernels that store
// through it; both are reported (512^3: 4.2 us, 3.7 for the copy alone).
__global__ void __launch_bounds__(256) adopt_tables_kernel(const __grid_constant__ TableArgs a,
                                                           const uint4 *src, uint4 *dst,
                                                           uint64_t words,
                                                           const unsigned long long *count,
                                                           const uint32_t *plan,
                                                           uint32_t plan_value) {
  const bool same = *plan == plan_value;
  const unsigned long long total = same ? *count : a.capacity;
  const bool fits = same && total < a.capacity;  // 1 + total bricks
  bool bad = false;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (fits) {
      v = src[i];
      if (v.x > total || v.y > total || v.z > total || v.w > total) {
        bad = true;
        v = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    dst[i] = v;
  }
  if (bad) atomicExch(a.status, (uint32_t)VCT_ERR_WORKSPACE);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.count = total;
    *a.plan = plan_value;
    if (!fits) atomicExch(a.status, (uint32_t)VCT_ERR_WORKSPACE);
  }
}

// Marks tables made for this shape (the places of a pyramid's tables depend on
// nothing else).
uint32_t plan_word(int n, int levels) {
  return 0x56435400u | (uint32_t)ilog2(n) << 4 | (uint32_t)levels;
}

}  // namespace

cudaError_t launch_brick_tables(const float *level0, int n, int levels, const Layout &L,
                                uint8_t *base, uint64_t capacity, cudaStream_t s,
                                const uint8_t *planned) {
  TableArgs a{};
  a.nbricked = 0;
  for (int l = 0; l < levels; ++l)
    if ((L.bricked >> l) & 1u) {
      a.tbl[l] = reinterpret_cast<uint32_t *>(base + L.level_off[l]);
      a.nb[l] = level_bricks(n, l);
      a.nbricked = l + 1;
    }
  a.status = reinterpret_cast<uint32_t *>(base);
  a.count = reinterpret_cast<unsigned long long *>(base + kHeaderCountOff);
  a.plan = reinterpret_cast<uint32_t *>(base + kHeaderPlanOff);
  a.capacity = capacity;
  if (a.nbricked == 0) {
    cudaError_t e = cudaMemsetAsync(base + kHeaderCountOff, 0, 8, s);
    return e;
  }
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  uint8_t *first = reinterpret_cast<uint8_t *>(a.tbl[0]);
  const int last = a.nbricked - 1;
  const uint64_t bytes =
      (uint64_t)(reinterpret_cast<uint8_t *>(a.tbl[last]) - first) + a.nb[last] * 4;
  if (planned != nullptr) {
    const uint64_t words = bytes / 16;
    const int grid = (int)std::min<uint64_t>((words + 255) / 256, (uint64_t)sms * 4);
    adopt_tables_kernel<<<grid, 256, 0, s>>>(
        a, reinterpret_cast<const uint4 *>(planned + L.level_off[0]),
        reinterpret_cast<uint4 *>(first), words,
        reinterpret_cast<const unsigned long long *>(planned + kHeaderCountOff),
        reinterpret_cast<const uint32_t *>(planned + kHeaderPlanOff), plan_word(n, levels));
    return cudaGetLastError();
  }
  // A grid whose flags one pass of one CTA holds (n <= 128) needs two launches.
  const bool small = bytes / 4 <= (uint64_t)kScanPass;
  cudaError_t e = small ? cudaSuccess : cudaMemsetAsync(first, 0, bytes, s);
  if (e != cudaSuccess) return e;
  const uint64_t warps = a.nb[0];
  const int grid = (int)std::min<uint64_t>((warps + 7) / 8, (uint64_t)sms * 16);
  occupancy_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<const float4 *>(level0), n, a,
                                        small);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  ScanArgs c{};
  c.flags = reinterpret_cast<uint32_t *>(first);
  c.sums = reinterpret_cast<uint32_t *>(base + 16);
  c.words = bytes / 4;
  c.part = (c.words + kScanCtas - 1) / kScanCtas;
  c.part = (c.part + kScanPass - 1) / kScanPass * kScanPass;
  c.status = a.status;
  c.count = a.count;
  c.capacity = capacity;
  c.plan = a.plan;
  c.plan_value = plan_word(n, levels);
  const int parts = (int)((c.words + c.part - 1) / c.part);
  c.bricks0 = a.nb[0];
  if (small) {
    c.sums = nullptr;
  } else {
    count_kernel<<<parts, kScanThreads, 0, s>>>(c);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  slots_kernel<<<parts, kScanThreads, 0, s>>>(c);
  return cudaGetLastError();
}

}  // namespace vct
