// Condense: Adaptive Pixel Compressor (Sec. 3.2, Eq. 1-6) and the bicubic resize (App. B.3).
//
// Density, four kernels on the caller's stream, each started before the one before it has drained
// (programmatic dependent launch): apc_zero clears the sums, then
//   apc_pass1  strips of up to 32 patches of one patch row, their 14 image rows staged in shared
//              memory: |x|^2 of each patch gives the inverse token norm 1/|T_i|; the weighted column
//              sums sum_i x_ik / (255 |T_i|) (and sum_i 1/|T_i| for the constant coordinate) are added
//              to a per-image 589-vector of 64-bit whole numbers, exactly, whatever the order.
//   apc_pass2  same strips: c = sums / N, phi = |c|^2, c_hat = c / |c| (recomputed per CTA from the
//              589 integers), then d_i = |t_i - c_hat| from exact dot products (no cancellation),
//              counted and summed (fixed point) in the tail's value buckets (global atomics).
//   apc_tail   the k_tail-th largest's bucket from the counts, its members from the distances, the
//              tail mean, rho_d, rho, r and the target size.  The token and pixel-statistic
//              densities share it (their pass 2 fills the buckets the same way).
// Resize: apc_resample, four CTAs per SM walking the output tiles of the batch; downscales of up to 8x
// per side are filtered vertically in registers, then horizontally from shared memory, small outputs
// in small staged tiles with the same sums, steeper downscales on a generic path with per-tap weights.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <cstddef>
#include <mutex>

#include <cooperative_groups.h>

#include "pace_common.cuh"
#include "pace_ptx.cuh"
#include "pace_select.cuh"

namespace pace {
namespace {

namespace cg = cooperative_groups;

constexpr int kPatch = 14;
constexpr int kPatchBytes = kPatch * kPatch * 3;     // 588
constexpr int kTokDim = kPatchBytes + 1;             // 589: pixels + constant coordinate
constexpr int kStrip = 32;                           // patches per strip
constexpr int kApcThreads = 256;
constexpr int kApcMaxB = 64;
// Column sums are 2^-32 fixed point in 64-bit integers.  The conversions below use only 32-bit
// conversions and fp32 (no fp64, which is a slow pipe on this GPU); fix32 rounds exactly like
// rounding v * 2^32 to the nearest integer (ties to even).
__device__ __forceinline__ unsigned long long fix32(float v) {   // 0 <= v < 2^31
  const float h = floorf(v);
  return (static_cast<unsigned long long>(static_cast<uint32_t>(h)) << 32) +
         __float2uint_rn((v - h) * 4294967296.0f);   // v - h is exact; the product is an exact scaling
}
__device__ __forceinline__ unsigned long long fix32_signed(float v) {   // |v| < 2^31, two's complement
  return v >= 0.f ? fix32(v) : 0ull - fix32(-v);
}
// sum * 2^-32 * inv_n for a non-negative (or, with SIGNED, two's-complement) fixed-point sum: of distances (at
// most 2 each) or of coordinates of unit vectors.  Rounded to fp32 once below 2^56, which fewer than 2^23
// patches or tokens (an image has fewer) can't pass.
template <bool SIGNED>
__device__ __forceinline__ float unfix32(unsigned long long sum, float inv_n) {
  const bool neg = SIGNED && static_cast<long long>(sum) < 0;
  const unsigned long long m = neg ? 0ull - sum : sum;
  const float hi = static_cast<float>(static_cast<uint32_t>(m >> 32));   // below 2^24
  const float v = fmaf(static_cast<float>(static_cast<uint32_t>(m)), 0x1p-32f, hi) * inv_n;
  return neg ? -v : v;
}
// m 2^-32 rounded to fp32 once, whatever m: its top 32 bits, the lowest of them standing for all that follow.
__device__ __forceinline__ float round32(unsigned long long m) {
  const int s = min(__clzll(static_cast<long long>(m)), 63);
  const unsigned long long x = m << s;
  const uint32_t top = static_cast<uint32_t>(x >> 32) | (static_cast<uint32_t>(x) != 0u ? 1u : 0u);
  return __uint2float_rn(top) * __uint_as_float(static_cast<uint32_t>(127 - s) << 23);   // 2^-s
}

struct ApcTable {
  int64_t off[kApcMaxB];    // byte offset of image b
  int H[kApcMaxB];
  int W[kApcMaxB];
  int gw[kApcMaxB];         // patches per row
  int chunks[kApcMaxB];     // strips per patch row
  int patch0[kApcMaxB];     // first global patch (or token) of image b
  int n[kApcMaxB];          // patches (or tokens) of image b
  int ktail[kApcMaxB];
  int unit_prefix[kApcMaxB + 1];
  int nb;
  int b_base;               // global index of image 0 of this table
  int strip_log2[kApcMaxB]; // log2 of the patches per strip of image b
  float2 col_scale[kApcMaxB]; // 2 / (255 n) as a sum of two floats: the mean of a column of image b from its sum
                              // in units of 2^-31 / 255
};

__device__ __forceinline__ int find_image(const ApcTable& t, int unit) {
  int b = 0;
  while (b + 1 < t.nb && t.unit_prefix[b + 1] <= unit) ++b;
  return b;
}

// Asynchronous 4-byte global -> shared copies (no register round trip, all in flight at once).
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
// 16 bytes, of which the first `bytes` are read and the others become zeros.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the warp, in every lane (below 2^64).
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
  const unsigned p0 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(v) & 0xFFFFu);
  const unsigned p1 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(v) >> 16);
  const unsigned p2 = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(v >> 32));
  return (static_cast<unsigned long long>(p2) << 32) + (static_cast<unsigned long long>(p1) << 16) + p0;
}

// ------------------------------------------------------------------------------------------------
// density on raw pixels
// ------------------------------------------------------------------------------------------------
// Both passes run one CTA per SM over its share of consecutive strips (so that it meets few images):
// three groups of 320 threads take the strips of an image in turn, each with its own buffers, the next
// strip being copied (TMA bulk copies, one per image row) while the current one is worked on.  One CTA
// per SM, because each ends an image with 589 64-bit atomics, which run at about one in 1.5 ns to a
// line (four CTAs per SM: 15 us of a 4K image's pass; clusters that add up before the atomics leave
// SMs idle).  They are bound by instruction issue, not by memory (the image is read once from
// HBM and once from L2), so both reduce to dot products of bytes that run four to an instruction
// (dp4a), exactly, in integers:
//   pass 1  |x|^2 of every patch, and the column sums of x_ik / |T_i|: 1/|T_i| in fp32 is a whole
//           multiple of 2^-31 (it lies in [2^-5, 1]), so its four bytes are the weights of four dp4a
//           over four patches at a time and the sums have no rounding at all;
//   pass 2  the dot products x_i . c_hat with c_hat in 2^-32 fixed point, four dp4a per four
//           coordinates, and |t_i - c_hat|^2 = |t_i|^2 + |c_hat|^2 - 2 t_i . c_hat in fp64 from those
//           whole numbers, so that nothing is lost when t_i is close to c_hat.
// Everything works on the 84 bytes of a patch pair's image row as 21 words: one 4-byte shared load
// brings four coordinates.  Word 10 holds the last two coordinates of the first patch and the first
// two of the second; a single last patch has an absent partner with weight 0.  On a 4K image the two
// passes took 19.9 + 15.8 us with a byte-to-float conversion and a packed fp32 FMA per coordinate, now
// 11.4 + 12.4 (three to four strips per group, each two group barriers and a wait for its rows).
constexpr int kDThreads = 320;                       // threads of a group
constexpr int kDGroups = 3;                          // groups of a CTA
constexpr int kDAll = kDThreads * kDGroups;
constexpr int kPairWords = 21;                       // words of a pair's image row
constexpr int kPairBytes = 4 * kPairWords;
constexpr int kStageRow = 1472;                      // bytes per staged row: 1344 + 16 slack, = 16 words mod 32
constexpr int kStageBytes = kPatch * kStageRow;      // so that two rows' pairs take different banks
constexpr int kWordSlots = kPatch * kPairWords;      // 294: word positions of a pair
constexpr int kStripLog2 = 5, kMinStripLog2 = 3;     // strips of 32 patches, 16 or 8
static_assert(kStrip == 1 << kStripLog2, "strip width");
constexpr int kSumSlots = 4;                         // copies of an image's column sums that the atomics spread over
constexpr int kGroups = kStrip / 8;                  // groups of four pairs in a full strip
// A dp4a of pass 1 adds at most 4 * 255^2 and a strip kGroups of them: the 32-bit digit sums are
// folded into 64 bits before they can overflow.
constexpr int kFoldStrips = 2048;
static_assert(static_cast<int64_t>(kFoldStrips) * kGroups * 4 * 255 * 255 < (int64_t{1} << 32), "digit sums");
// The strips [first, end) of this CTA.
__device__ __forceinline__ int2 unit_range(int units) {
  const int each = units / static_cast<int>(gridDim.x), extra = units - each * static_cast<int>(gridDim.x);
  const int i = static_cast<int>(blockIdx.x), first = i * each + min(i, extra);
  return make_int2(first, first + each + (i < extra ? 1 : 0));
}

// Zeroes a call's sums and tail scratch (two ranges of 16-byte words); the first pass of the density
// starts beside it and waits for it before its first atomic.  A memset in its place is a full stop in
// the stream: 2.3 us.
__global__ void __launch_bounds__(256) apc_zero(uint4* __restrict__ a, unsigned na, uint4* __restrict__ b, unsigned nb) {
  ptx::begin_call();
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < na + nb; i += gridDim.x * blockDim.x)
    *(i < na ? a + i : b + (i - na)) = make_uint4(0u, 0u, 0u, 0u);
}

struct alignas(16) StripRef {
  int b, py, px0, np;
  int pairs_log2;   // log2 of the pairs of a full strip
  uint32_t first;   // byte of the image at which the strip's first row starts (an image is below 2^32 bytes)
  uint32_t pitch;   // bytes per image row
  int patch;        // the first patch's number in the call
};
__device__ __forceinline__ void strip_place(const ApcTable& t, StripRef& q) {
  q.np = min(2 << q.pairs_log2, t.gw[q.b] - q.px0);
  q.first = static_cast<uint32_t>(q.py) * kPatch * q.pitch + static_cast<uint32_t>(q.px0) * (kPatch * 3);
  q.patch = t.patch0[q.b] + q.py * t.gw[q.b] + q.px0;
}
__device__ __forceinline__ void strip_image(const ApcTable& t, StripRef& q) {
  q.pairs_log2 = t.strip_log2[q.b] - 1;
  q.pitch = static_cast<uint32_t>(t.W[q.b]) * 3u;
}
__device__ __forceinline__ StripRef strip_ref(const ApcTable& t, int unit) {
  StripRef q;
  q.b = find_image(t, unit);
  const int u = unit - t.unit_prefix[q.b];
  q.py = u / t.chunks[q.b];
  strip_image(t, q);
  q.px0 = (u - q.py * t.chunks[q.b]) << (q.pairs_log2 + 1);
  strip_place(t, q);
  return q;
}
// The strip n on in the same image.
__device__ __forceinline__ void strip_advance(const ApcTable& t, StripRef& q, int n) {
  q.px0 += n << (q.pairs_log2 + 1);
  while (q.px0 >= t.chunks[q.b] << (q.pairs_log2 + 1)) {
    q.px0 -= t.chunks[q.b] << (q.pairs_log2 + 1);
    ++q.py;
  }
  strip_place(t, q);
}
// Row y of a strip is staged from the 16-byte boundary at or before its first byte: this many bytes on.
__device__ __forceinline__ uint32_t row_phase(const StripRef& q, int y) {
  return (q.first + static_cast<uint32_t>(y) * q.pitch) & 15u;
}

// Called by one whole warp: copies a strip's 14 rows to s (a lane per row), counted on the mbarrier
// `bar`, and the strip's place to `slot`.  Nothing past the image is read: the last row's last few bytes,
// which do not fill a 16-byte piece, are stored by the lane itself, before the warp's arrival on the barrier.
__device__ __forceinline__ void copy_strip(const uint8_t* __restrict__ img, const ApcTable& t, const StripRef& q, uint8_t* s,
                                           uint32_t bar, StripRef* slot) {
  const int lane = threadIdx.x & 31;
  uint32_t bytes = 0u;
  int64_t a = 0;
  const uint8_t* base = img + t.off[q.b];
  if (lane < kPatch) {
    const uint32_t ph = row_phase(q, lane);
    a = static_cast<int64_t>(q.first) + static_cast<int64_t>(lane) * q.pitch - ph;
    bytes = (ph + static_cast<uint32_t>(q.np) * (kPatch * 3) + 15u) & ~15u;
    const int64_t left = static_cast<int64_t>(t.H[q.b]) * q.pitch - a;
    if (bytes > left) {
      bytes = static_cast<uint32_t>(left) & ~15u;
      for (uint32_t i = bytes; i < left; i += 4u)   // an image holds a multiple of 4 bytes
        *reinterpret_cast<uint32_t*>(s + lane * kStageRow + i) = __ldg(reinterpret_cast<const uint32_t*>(base + a + i));
      ptx::fence_proxy_async_shared();
    }
  }
  const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
  __syncwarp();
  if (lane == 0) {
    *slot = q;
    ptx::mbar_arrive_expect_tx(bar, total);
  }
  __syncwarp();
  if (bytes > 0u) ptx::bulk_load(ptx::smem_u32(s + lane * kStageRow), base + a, bytes, bar);
}

// The words of a pair's row that starts at byte `a` of shared memory.  ALIGNED: a is a multiple of
// 4 (every image an even number of patches wide); otherwise a is even and each word is put together
// from two aligned ones.
template <bool ALIGNED>
struct RowWords {
  const uint32_t* w;
  uint32_t cur, sh;
  __device__ __forceinline__ explicit RowWords(const uint8_t* a) {
    if (ALIGNED) {
      w = reinterpret_cast<const uint32_t*>(a);
    } else {
      sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a) & 2u) * 8u;
      w = reinterpret_cast<const uint32_t*>(a - (sh >> 3));
      cur = w[0];
    }
  }
  __device__ __forceinline__ uint32_t get(int j) {   // j = 0, 1, 2, .. in order
    if (ALIGNED) return w[j];
    const uint32_t nxt = w[j + 1];
    const uint32_t v = __funnelshift_r(cur, nxt, sh);
    cur = nxt;
    return v;
  }
};
// One word at byte `a` (4-byte aligned if ALIGNED, else 2-byte: sh = 8 (a mod 4)).
template <bool ALIGNED>
__device__ __forceinline__ uint32_t word_at(const uint8_t* a, uint32_t sh) {
  if (ALIGNED) return *reinterpret_cast<const uint32_t*>(a);
  const uint32_t* w = reinterpret_cast<const uint32_t*>(a - (sh >> 3));
  return __funnelshift_r(w[0], w[1], sh);
}

// 1/|T_i| of a patch from its |x|^2.
__device__ __forceinline__ float inv_norm_of(uint32_t ss) {
  return 1.0f / sqrtf(static_cast<float>(ss) * (1.0f / 65025.0f) + 1.0f);
}

// Waits for use `use` of a group's buffers (two, used in turn).  After a wait that runs out the group's waits
// end at once, *gave_up holding 2; before that (1) both buffers get one more limit, so that no copy lands
// after the CTA has ended.
template <uint64_t LIMIT_NS>
__device__ __noinline__ void strip_wait(uint64_t* bars, volatile int* gave_up, unsigned use, int* status, int kernel) {
  auto wait = [&](unsigned u) { return ptx::mbar_wait(ptx::smem_u32(&bars[u & 1]), (u >> 1) & 1u, LIMIT_NS); };
  if (*gave_up == 0) {
    if (wait(use)) return;
    record_error(status, PACE_ERR_TIMEOUT, kernel);
    *gave_up = 1;
  }
  if (*gave_up == 1) {
    wait(use);
    wait(use + 1);
    *gave_up = 2;
  }
}

// A group's strips of one image (first, first + STEP, .. below end), which one of its warps copies into
// its two buffers.  `used` counts the strips that the group has worked on, i.e. the uses of its buffers.
// A group that has given up copies nothing any more and works on what its buffers hold, from the places that
// the copying warp last gave them (empty ones at the start), so within the call's images.
template <int STEP, uint64_t LIMIT_NS = kWaitLimitNs>
struct StripPipe {
  uint8_t (*s2)[kStageBytes];
  uint64_t* bars;
  StripRef* ref;
  volatile int* gave_up;
  unsigned used;
  // by one thread of the group, before the others come past a barrier
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      ptx::mbar_init(ptx::smem_u32(&bars[k]), 1);
      ref[k] = StripRef{};
    }
    *gave_up = 0;
    ptx::fence_mbar_init();
  }
  __device__ __forceinline__ void copy(const uint8_t* img, const ApcTable& t, const StripRef& q, unsigned use) {
    copy_strip(img, t, q, s2[use & 1], ptx::smem_u32(&bars[use & 1]), &ref[use & 1]);
  }
  __device__ __forceinline__ bool stopped() const { return __any_sync(0xffffffffu, *gave_up != 0); }
  // the image's first two strips (called by the copying warp of a group that is done with its buffers)
  __device__ __forceinline__ void begin(const uint8_t* img, const ApcTable& t, int first, int end) {
    if (first >= end || stopped()) return;
    StripRef q = strip_ref(t, first);
    copy(img, t, q, used);
    if (first + STEP < end) {
      strip_advance(t, q, STEP);
      copy(img, t, q, used + 1);
    }
  }
  __device__ __forceinline__ void wait(int* status, int kernel) {
    if (!ptx::mbar_try_wait(ptx::smem_u32(&bars[used & 1]), (used >> 1) & 1u))
      strip_wait<LIMIT_NS>(bars, gave_up, used, status, kernel);
  }
  __device__ __forceinline__ const uint8_t* data() const { return s2[used & 1]; }
  __device__ __forceinline__ const StripRef& place() const { return ref[used & 1]; }
  // the strip after `cur`, once the group is done with the strip before it (called by the copying warp)
  __device__ __forceinline__ void next(const uint8_t* img, const ApcTable& t, const StripRef& cur) {
    if (stopped()) return;
    StripRef q = cur;
    strip_advance(t, q, STEP);
    copy(img, t, q, used + 1);
  }
};

// Strips whose rows never land: the first wait runs out after a millisecond, the ones after it end at once, and
// the strips are empty.
__global__ void __launch_bounds__(64) strip_selftest(int* status) {
  __shared__ __align__(16) uint8_t s2[2][kStageBytes];
  __shared__ uint64_t bars[2];
  __shared__ StripRef ref[2];
  __shared__ int gave_up;
  StripPipe<1, 1000000ull> pipe{s2, bars, ref, &gave_up, 0u};
  if (threadIdx.x == 0) pipe.init();
  __syncthreads();
  const uint64_t start = ptx::globaltimer_ns();
  for (int i = 0; i < 1000; ++i, ++pipe.used) {
    pipe.wait(nullptr, K_SELFTEST);
    const StripRef cur = pipe.place();
    if (gave_up == 0 || cur.np != 0 || cur.first != 0u || cur.pitch != 0u || cur.patch != 0)
      record_error(status, PACE_ERR_INVALID_ARG, K_SELFTEST);
  }
  if (!pipe.stopped() || ptx::globaltimer_ns() - start > 500000000ull) record_error(status, PACE_ERR_INVALID_ARG, K_SELFTEST);
}

struct Pass1Group {
  uint8_t s2[2][kStageBytes];
  uint32_t ssq[kPatch][kStrip];
  // the four bytes of the weights 2^31 / |T_i|: [group of four pairs][first or second patch][byte]
  uint8_t wdig[kGroups][2][4][4];
  unsigned long long col[kTokDim + 1];
  uint64_t bars[2];
  StripRef ref[2];
  int gave_up[4];
};
static_assert(kStageBytes % 16 == 0 && offsetof(Pass1Group, wdig) % 16 == 0 && sizeof(Pass1Group) % 16 == 0, "shared layout");

template <bool ALIGNED>
__global__ void __launch_bounds__(kDAll, 1) apc_pass1(const uint8_t* __restrict__ img, const __grid_constant__ ApcTable t,
                                                      int units, uint32_t* __restrict__ sumsq,
                                                      unsigned long long* __restrict__ sums, int* status) {
  extern __shared__ __align__(16) unsigned char d_smem[];
  ptx::launch_dependents();
  const int tid = threadIdx.x, grp = threadIdx.y, warp = tid >> 5;   // thread and warp of the group
  Pass1Group* all = reinterpret_cast<Pass1Group*>(d_smem);
  Pass1Group& sh = all[grp];
  auto group_sync = [&]() { ptx::named_barrier_sync(1 + grp, kDThreads); };
  const int2 range = unit_range(units);
  constexpr int kCopyWarp = kDThreads / 32 - 1;
  StripPipe<kDGroups> pipe{sh.s2, sh.bars, sh.ref, sh.gave_up, 0u};
  if (tid == 0) pipe.init();
  group_sync();
  // thread j < 294 owns the four columns of word position j (row j / 21): their digit sums; lane 0 of
  // warp 0 the constant coordinate
  uint32_t acc[4][4] = {};
  unsigned long long one = 0ull;
  const int wy = tid / kPairWords, wj = tid - wy * kPairWords;
  int strips = 0;   // in the digit sums
  // moves the digit sums to (or adds them to) the group's 64-bit column sums (a column has two owners:
  // the first and the second patch of a pair)
  auto fold = [&](bool add) {
    auto put = [&](bool second) {
      if (tid < kWordSlots) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = 4 * wj + q;   // byte of the pair's row
          const unsigned long long v = acc[q][0] + (static_cast<unsigned long long>(acc[q][1]) << 8) +
                                       (static_cast<unsigned long long>(acc[q][2]) << 16) +
                                       (static_cast<unsigned long long>(acc[q][3]) << 24);
          if ((c >= 42) == second) {
            unsigned long long* p = &sh.col[wy * 42 + (second ? c - 42 : c)];
            *p = (second || add ? *p : 0ull) + v;
          }
        }
      }
      if (tid == 0 && !second) sh.col[kPatchBytes] = (add ? sh.col[kPatchBytes] : 0ull) + one;
    };
    put(false);
    group_sync();
    put(true);
    group_sync();
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int d = 0; d < 4; ++d) acc[q][d] = 0u;
    one = 0ull;
    strips = 0;
  };
  int first = range.x;
  for (int b = first < range.y ? find_image(t, first) : 0; first < range.y; ++b) {   // the CTA's strips of image b
    const int end = min(range.y, t.unit_prefix[b + 1]);
    if (warp == kCopyWarp) pipe.begin(img, t, first + grp, end);
    bool folded = false;
    for (int unit = first + grp; unit < end; unit += kDGroups, ++pipe.used) {
      pipe.wait(status, K_APC_PASS1);
      const StripRef cur = pipe.place();
      const uint8_t* s = pipe.data();
      if (strips == kFoldStrips) {
        fold(folded);
        folded = true;
      }
      ++strips;
      const int npair = (cur.np + 1) >> 1;
      const int iy = tid >> cur.pairs_log2, ip = tid & ((1 << cur.pairs_log2) - 1);
      if (iy < kPatch && ip < npair) {   // |x|^2 of one image row of a pair
        RowWords<ALIGNED> w(s + iy * kStageRow + row_phase(cur, iy) + ip * kPairBytes);
        uint32_t p = 0u, q = 0u;
#pragma unroll
        for (int j = 0; j < kPairWords; ++j) {
          const uint32_t v = w.get(j);
          if (j < 10) p = __dp4a(v, v, p);
          else if (j > 10) q = __dp4a(v, v, q);
          else {
            p = __dp4a(v & 0xFFFFu, v, p);
            q = __dp4a(v & 0xFFFF0000u, v, q);
          }
        }
        *reinterpret_cast<uint2*>(&sh.ssq[iy][2 * ip]) = make_uint2(p, q);
      }
      group_sync();   // (the group is also done with its other buffer)
      // (the image's first two strips were requested at its start)
      if (warp == kCopyWarp && unit >= first + kDGroups && unit + kDGroups < end) pipe.next(img, t, cur);
      if (warp == 0) {   // lane p: patch p of the strip
        uint32_t weight = 0u;
        if (tid < cur.np) {
          uint32_t ss = 0u;
#pragma unroll
          for (int y = 0; y < kPatch; ++y) ss += sh.ssq[y][tid];
          sumsq[cur.patch + tid] = ss;
          weight = __float2uint_rn(inv_norm_of(ss) * 2147483648.0f);   // exact
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) sh.wdig[tid >> 3][tid & 1][d][(tid >> 1) & 3] = static_cast<uint8_t>(weight >> (8 * d));
        const uint32_t lo = __reduce_add_sync(0xffffffffu, weight & 0xFFFFu), hi = __reduce_add_sync(0xffffffffu, weight >> 16);
        if (tid == 0) one += lo + (static_cast<unsigned long long>(hi) << 16);
      }
      group_sync();
      if (tid < kWordSlots) {
        const uint32_t off = row_phase(cur, wy) + 4u * wj;
        const uint8_t* wp = s + wy * kStageRow + off;
        const uint32_t shf = (off & 2u) * 8u;
        const uint4* wl = reinterpret_cast<const uint4*>(sh.wdig) + (wj <= 10 ? 0 : 1);   // patch of the word's first two bytes
        const uint4* wh = reinterpret_cast<const uint4*>(sh.wdig) + (wj < 10 ? 0 : 1);    // and of its last two
        auto take = [&](int g) {   // four pairs: their bytes column by column, against the weights' digits
          uint32_t w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) w[r] = word_at<ALIGNED>(wp + (4 * g + r) * kPairBytes, shf);
          const uint32_t a0 = __byte_perm(w[0], w[1], 0x5140), a1 = __byte_perm(w[0], w[1], 0x7362);
          const uint32_t b0 = __byte_perm(w[2], w[3], 0x5140), b1 = __byte_perm(w[2], w[3], 0x7362);
          const uint32_t c[4] = {__byte_perm(a0, b0, 0x5410), __byte_perm(a0, b0, 0x7632), __byte_perm(a1, b1, 0x5410),
                                 __byte_perm(a1, b1, 0x7632)};
          const uint4 l = wl[2 * g], h = wh[2 * g];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint4 d = k < 2 ? l : h;
            acc[k][0] = __dp4a(c[k], d.x, acc[k][0]);
            acc[k][1] = __dp4a(c[k], d.y, acc[k][1]);
            acc[k][2] = __dp4a(c[k], d.z, acc[k][2]);
            acc[k][3] = __dp4a(c[k], d.w, acc[k][3]);
          }
        };
        if (npair > 4 * (kGroups - 1)) {
#pragma unroll
          for (int g = 0; g < kGroups; ++g) take(g);
        } else {
          for (int g = 0; 4 * g < npair; ++g) take(g);
        }
      }
    }
    // the image's sums: the groups' added up, one atomic per column
    fold(folded);
    ptx::grid_dependency_wait();   // the zeroed sums
    __syncthreads();
    const int k = grp * kDThreads + tid;
    if (k < kTokDim) {
      unsigned long long x = 0ull;
#pragma unroll
      for (int g = 0; g < kDGroups; ++g) x += all[g].col[k];
      atomicAdd(sums + (static_cast<int64_t>(t.b_base + b) * kSumSlots + blockIdx.x % kSumSlots) * kTokDim + k, x);
    }
    first = end;
    if (first < range.y) __syncthreads();   // the column sums are rewritten
  }
  static_assert(kWordSlots <= kDThreads - 32 + 6 && kPatch * (kStrip / 2) <= kDThreads && kStrip == 32 && kTokDim <= kDAll,
                "thread roles");
}

struct TailParams {
  float alpha, gamma, r_min, r_max;
  int align;
};

constexpr int kTailBins = 4096;            // level-1 buckets of the tail select

// Bucket of a distance d >= 0: floor(2048 d), capped at the top bucket (monotone in d; NaN goes to
// bucket 0).  Full-rate arithmetic only (no float-to-integer conversion): once clamped to
// [0, 4095], 2048 d + 2^23 rounded toward zero holds floor(2048 d) in its low mantissa bits.
__device__ __forceinline__ int tail_bucket(float v) {
  const float x = fminf(fmaxf(v * 2048.0f, 0.0f), static_cast<float>(kTailBins - 1));
  return __float_as_int(__fadd_rz(x, 8388608.0f)) - 0x4B000000;
}

// Scratch of the density tail, filled by pass 2 with atomics (exact, so in any order): the count
// and the 2^-32 fixed-point sum of the distances of each bucket.
struct TailWork {
  unsigned long long sum[kTailBins];
  unsigned hist[kTailBins];
};
// Counts and sums the distances of a warp (all lanes call it; those with `live` have one).  Additions to
// one address run at about one in 1.5 ns, which a picture with much background (42000 equal distances)
// feels: the lanes of the first live lane's bucket, and then those of the last remaining one's, are
// added together, the rest one by one.  The density call on a 4K picture, 90 % one colour: 28.2 us, with
// every distance added by itself 47.1; a picture without background 26.0 either way.  (One addition per
// different bucket, by __match_any_sync and reductions over its masks, cost the latter 18 us: the
// reductions of a warp's different masks run one after the other.)
__device__ __forceinline__ void tail_count_warp(TailWork* w, float d, bool live) {
  const int b = tail_bucket(d);
  const unsigned long long v = fix32(d);   // below 2^38 (a distance is at most 2): three sums of 32 parts
  unsigned left = __ballot_sync(0xffffffffu, live);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (left == 0u) return;   // warp-uniform
    const int lead = k == 0 ? __ffs(left) - 1 : 31 - __clz(left);
    const unsigned lane = threadIdx.x & 31;
    const bool in = b == __shfl_sync(0xffffffffu, b, lead) && ((left >> lane) & 1u);
    const unsigned peers = __ballot_sync(0xffffffffu, in);
    if (__popc(peers) < 4) continue;   // warp-uniform
    const unsigned p0 = __reduce_add_sync(0xffffffffu, in ? static_cast<unsigned>(v) & 0xFFFFu : 0u);
    const unsigned p1 = __reduce_add_sync(0xffffffffu, in ? static_cast<unsigned>(v) >> 16 : 0u);
    const unsigned p2 = __reduce_add_sync(0xffffffffu, in ? static_cast<unsigned>(v >> 32) : 0u);
    if (lane == static_cast<unsigned>(lead)) {
      atomicAdd(&w->hist[b], static_cast<unsigned>(__popc(peers)));
      atomicAdd(&w->sum[b],
                (static_cast<unsigned long long>(p2) << 32) + (static_cast<unsigned long long>(p1) << 16) + p0);
    }
    left &= ~peers;
  }
  if ((left >> (threadIdx.x & 31)) & 1u) {
    atomicAdd(&w->hist[b], 1u);
    atomicAdd(&w->sum[b], v);
  }
}
// The same for a warp whose lanes hold few different values that may all lie in other buckets (the edge
// density of noise has about ten among 32 patches): one addition per different value, 47 us against 57
// for the call on a noise image of 42000 patches.  A sum of equal values needs no reduction.
__device__ __forceinline__ void tail_count_values(TailWork* w, float d, bool live) {
  const unsigned act = __ballot_sync(0xffffffffu, live);
  if (!live) return;
  const unsigned peers = __match_any_sync(act, __float_as_uint(d));
  if ((threadIdx.x & 31) != static_cast<unsigned>(__ffs(peers) - 1)) return;
  const unsigned n = static_cast<unsigned>(__popc(peers));
  const int b = tail_bucket(d);
  atomicAdd(&w->hist[b], n);
  atomicAdd(&w->sum[b], fix32(d) * n);
}
// The same for one thread that meets distances one after the other: consecutive ones of a bucket are
// added together (tokens of 1280 on a 4K picture, 90 % of them equal: 45.1 us, one by one 64.4).
struct TailRun {
  TailWork* w;
  int b = 0;
  unsigned n = 0u;
  unsigned long long sum = 0ull;
  __device__ __forceinline__ explicit TailRun(TailWork* work) : w(work) {}
  __device__ __forceinline__ void flush() {
    if (n == 0u) return;
    atomicAdd(&w->hist[b], n);
    atomicAdd(&w->sum[b], sum);
    n = 0u;
    sum = 0ull;
  }
  __device__ __forceinline__ void add(float d) {
    const int bd = tail_bucket(d);
    if (bd != b) flush();
    b = bd;
    ++n;
    sum += fix32(d);
  }
};

struct Pass2Group {
  uint8_t s2[2][kStageBytes];
  unsigned long long part[2][kPatch][kStrip];   // x . c_hat of one image row of a patch
  uint64_t bars[2];
  StripRef ref[2];
  int gave_up[4];
};
struct Pass2Smem {
  Pass2Group g[kDGroups];
  // the four bytes of c_hat (2^-32 fixed point) of a pair's words, the two patches one after the
  // other: [image row][word][byte][coordinate of the word]
  uint8_t cdig[kPatch][kPairWords][4][4];
  float craw[kTokDim + 3];
  unsigned long long redq[kDAll / 32], redc[kDAll / 32];
};
static_assert(sizeof(Pass2Group) % 16 == 0 && offsetof(Pass2Smem, cdig) % 16 == 0, "shared layout");

template <bool ALIGNED>
__global__ void __launch_bounds__(kDAll, 1) apc_pass2(const uint8_t* __restrict__ img, const __grid_constant__ ApcTable t,
                                                      int units, const uint32_t* __restrict__ sumsq,
                                                      const unsigned long long* __restrict__ sums, float* __restrict__ d_out,
                                                      pace_apc_stats* __restrict__ stats, TailWork* __restrict__ work,
                                                      int* status) {
  extern __shared__ __align__(16) unsigned char d_smem[];
  Pass2Smem& sh = *reinterpret_cast<Pass2Smem*>(d_smem);
  ptx::launch_dependents();
  const int tid = threadIdx.x, grp = threadIdx.y, warp = tid >> 5, lane = tid & 31;   // thread and warp of the group
  const int ct = grp * kDThreads + tid;                                               // thread of the CTA
  Pass2Group& my = sh.g[grp];
  auto group_sync = [&]() { ptx::named_barrier_sync(1 + grp, kDThreads); };
  constexpr int kCopyWarp = kDThreads / 32 - 1;
  const int2 range = unit_range(units);
  StripPipe<kDGroups> pipe{my.s2, my.bars, my.ref, my.gave_up, 0u};
  if (tid == 0) pipe.init();
  group_sync();
  int first = range.x;
  for (int b = first < range.y ? find_image(t, first) : 0; first < range.y; ++b) {   // the CTA's strips of image b
    const int end = min(range.y, t.unit_prefix[b + 1]);
    if (warp == kCopyWarp) pipe.begin(img, t, first + grp, end);   // (the image does not depend on pass 1)
    ptx::grid_dependency_wait();
    // c = sums / N, |c|^2 (fixed summation order), c_hat = c / |c|
    const int N = t.n[b];
    const unsigned long long* sb = sums + static_cast<int64_t>(t.b_base + b) * (kSumSlots * kTokDim);
    float c = 0.f;
    if (ct < kTokDim) {   // a thread per coordinate
      unsigned long long x = 0ull;
#pragma unroll
      for (int r = 0; r < kSumSlots; ++r) x += __ldcg(sb + r * kTokDim + ct);
      // sums are multiples of 2^-31 (and, but for the constant coordinate, of 1/255); the factor of all
      // coordinates in two floats, since its rounding would move phi, and 1 - phi more.  The high word of a
      // sum passes 2^24 from about 186000 patches on (one byte of 255 in each: 90 per patch).
      const float v = round32(x);
      c = fmaf(v, t.col_scale[b].y, v * t.col_scale[b].x) * (ct < kPatchBytes ? 1.0f : 255.0f);
      if (ct == kPatchBytes) sh.craw[0] = c;
    }
    // |c|^2 in 2^-62 fixed point (c <= 1), so that 1 - phi is exact too
    const uint32_t cu = __float2uint_rn(c * 2147483648.0f);
    const unsigned long long p2 = warp_sum_u64(static_cast<unsigned long long>(cu) * cu);
    if (lane == 0) sh.redq[ct >> 5] = p2;
    __syncthreads();
    unsigned long long phi62 = 0ull;
#pragma unroll
    for (int w = 0; w < (kTokDim + 31) / 32; ++w) phi62 += sh.redq[w];
    const float phi = static_cast<float>(phi62) * 0x1p-62f;
    const float inv_c = 1.0f / sqrtf(phi);
    unsigned long long sq = 0ull;   // square, 2^-56 fixed point
    if (ct < kPatchBytes) {
      const int y = ct / 42, x = ct - y * 42;
      const uint32_t v = __float2uint_rn(fminf(c * inv_c, 0.99999994f) * 4294967296.0f);
      sq = static_cast<unsigned long long>(v) * v >> 8;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const uint8_t byte = static_cast<uint8_t>(v >> (8 * d));
        sh.cdig[y][x >> 2][d][x & 3] = byte;
        sh.cdig[y][(x + 42) >> 2][d][(x + 42) & 3] = byte;
      }
    }
    sq = warp_sum_u64(sq);
    if (lane == 0) sh.redc[ct >> 5] = sq;
    __syncthreads();
    double cc = 0.0, c1 = 0.0;   // a group's warp 0: |c_hat|^2 and the constant coordinate of c_hat
    if (warp == 0) {             // (fp64 is slow on this GPU: one warp's worth per group and strip)
      sq = 0ull;
#pragma unroll
      for (int w = 0; w < (kPatchBytes + 31) / 32; ++w) sq += sh.redc[w];
      c1 = static_cast<double>(sh.craw[0] * inv_c);
      cc = fma(static_cast<double>(sq), 0x1p-56, c1 * c1);
    }
    if (first == t.unit_prefix[b] && ct == 0) {
      stats[t.b_base + b].phi = phi;
      stats[t.b_base + b].rho_g = static_cast<float>(static_cast<long long>((1ull << 62) - phi62)) * 0x1p-62f;
      stats[t.b_base + b].n_patches = N;
      stats[t.b_base + b].k_tail = t.ktail[b];
    }
    for (int unit = first + grp; unit < end; unit += kDGroups, ++pipe.used) {
      pipe.wait(status, K_APC_PASS2);
      const StripRef cur = pipe.place();
      const uint8_t* s = pipe.data();
      auto& part = my.part[pipe.used & 1];
      const int p0 = cur.patch;
      const int npair = (cur.np + 1) >> 1;
      const int iy = tid >> cur.pairs_log2, ip = tid & ((1 << cur.pairs_log2) - 1);   // this thread's (row, pair)
      uint32_t ss = 0u;
      if (warp == 0 && lane < cur.np) ss = __ldcg(sumsq + p0 + lane);
      // x . c_hat over one image row of a pair
      if (iy < kPatch && ip < npair) {
        RowWords<ALIGNED> w(s + iy * kStageRow + row_phase(cur, iy) + ip * kPairBytes);
        const uint4* cd = reinterpret_cast<const uint4*>(sh.cdig[iy]);
        uint32_t p[4] = {}, q[4] = {};
        auto dot = [](uint32_t v, const uint4& d, uint32_t (&x)[4]) {
          x[0] = __dp4a(v, d.x, x[0]);
          x[1] = __dp4a(v, d.y, x[1]);
          x[2] = __dp4a(v, d.z, x[2]);
          x[3] = __dp4a(v, d.w, x[3]);
        };
#pragma unroll
        for (int j = 0; j < kPairWords; ++j) {
          const uint32_t v = w.get(j);
          const uint4 d = cd[j];
          if (j < 10) dot(v, d, p);
          else if (j > 10) dot(v, d, q);
          else {
            dot(v & 0xFFFFu, d, p);
            dot(v & 0xFFFF0000u, d, q);
          }
        }
        auto join = [](const uint32_t (&x)[4]) {
          return x[0] + (static_cast<unsigned long long>(x[1]) << 8) + (static_cast<unsigned long long>(x[2]) << 16) +
                 (static_cast<unsigned long long>(x[3]) << 24);
        };
        *reinterpret_cast<ulonglong2*>(&part[iy][2 * ip]) = make_ulonglong2(join(p), join(q));
      }
      group_sync();   // (the group is also done with its other buffer)
      if (warp == kCopyWarp && unit >= first + kDGroups && unit + kDGroups < end) pipe.next(img, t, cur);
      if (warp == 0) {
        const bool live = lane < cur.np;
        unsigned long long x = 0ull;
#pragma unroll
        for (int y = 0; y < kPatch; ++y) x += live ? part[y][lane] : 0ull;
        const double iv = static_cast<double>(inv_norm_of(ss));
        const double dot = iv * fma(static_cast<double>(x), 0x1p-32 / 255.0, c1);                  // t . c_hat
        const double tt = iv * iv * fma(static_cast<double>(ss), 1.0 / 65025.0, 1.0);              // |t|^2
        const float dv = sqrtf(fmaxf(static_cast<float>(tt + cc - 2.0 * dot), 0.f));
        if (live) d_out[p0 + lane] = dv;
        tail_count_warp(work + t.b_base + b, dv, live);
      }
    }
    first = end;
    if (first < range.y) __syncthreads();   // c_hat is rewritten, and every group is done with its buffers
  }
}

// ------------------------------------------------------------------------------------------------
// density on preview tokens (Sec. 3.2 "Shallow Feature Preview": T_v from the first ViT block)
// ------------------------------------------------------------------------------------------------
// Same Eq. 1-6 as the pixel path, on caller-supplied bf16 tokens [sum N, D].  A token of zero
// norm counts as t_hat = 0 (its cosine with any token is taken as 0); if every token of an
// image is zero, c_hat = 0.
constexpr int kTokChunk = 32;    // tokens per CTA
constexpr int kTokMaxD = 4096;   // longest token accepted (c_hat is staged in shared memory)

struct TokTable {
  int64_t tok0[kApcMaxB];        // first token of image b
  int n[kApcMaxB];               // tokens of image b
  int unit_prefix[kApcMaxB + 1]; // chunks of kTokChunk tokens (pass 2)
  int unit_prefix1[kApcMaxB + 1]; // chunks of rows1 tokens (pass 1)
  int ktail[kApcMaxB];
  int nb;
  int b_base;
  int D;
  int rows1;                     // tokens per pass-1 chunk (a chunk fits a 40 KB stage)
  int run_prefix[kApcMaxB + 1];  // runs of kTokRun tokens (the register kernels)
};

constexpr int kTok1StageBytes = 40960;   // one pass-1 stage: rows1 token rows
constexpr int kTok1MaxSlots = kTokMaxD / 2 / kApcThreads;   // column pairs per thread (8)

__device__ __forceinline__ int find_tok_image(const TokTable& t, int unit) {
  int b = 0;
  while (b + 1 < t.nb && t.unit_prefix[b + 1] <= unit) ++b;
  return b;
}

__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// Pass 1: 1/|T_i| per token (warp per token) and the column sums of t_hat = T_i / |T_i|, as
// signed 2^-32 fixed point (exact, order-independent).  A grid of resident CTAs walks chunks of
// rows1 tokens; each chunk is staged in shared memory with cp.async while the previous one is
// worked on, so T is read once.  Per-chunk sums are rounded and added in registers; one atomic
// per column when the CTA moves to another image or ends.
__device__ __forceinline__ void tok_issue_chunk(const uint32_t* __restrict__ T, const TokTable& t, int unit,
                                                uint32_t* dst) {
  int b = 0;
  while (b + 1 < t.nb && t.unit_prefix1[b + 1] <= unit) ++b;
  const int r0 = (unit - t.unit_prefix1[b]) * t.rows1;
  const int nt = min(t.rows1, t.n[b] - r0);
  const int words = t.D >> 1;
  const uint32_t* src = T + (t.tok0[b] + r0) * words;
  for (int i = threadIdx.x; i < nt * words; i += kApcThreads) cp_async4(dst + i, src + i);
  cp_async_commit();
}

__global__ void __launch_bounds__(kApcThreads) apc_tok_pass1(const uint32_t* __restrict__ T,
                                                             const __grid_constant__ TokTable t, int units,
                                                             float* __restrict__ inv_norm,
                                                             unsigned long long* __restrict__ sums) {
  extern __shared__ __align__(16) uint32_t tok_smem[];   // two stages of rows1 x words
  __shared__ float inv[2][32];
  int unit = blockIdx.x;
  if (unit >= units) return;
  const int words = t.D >> 1;   // bf16 pairs per token
  const int stage = t.rows1 * words;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long acc[kTok1MaxSlots][2];
#pragma unroll
  for (int q = 0; q < kTok1MaxSlots; ++q) acc[q][0] = acc[q][1] = 0ull;
  int cur_b = -1;
  auto flush = [&]() {
    if (cur_b < 0) return;
    unsigned long long* sb = sums + static_cast<int64_t>(t.b_base + cur_b) * kSumSlots * t.D;   // the first copy
#pragma unroll
    for (int q = 0; q < kTok1MaxSlots; ++q) {
      const int w = threadIdx.x + q * kApcThreads;
      if (w < words) {
        atomicAdd(sb + 2 * w, acc[q][0]);
        atomicAdd(sb + 2 * w + 1, acc[q][1]);
      }
      acc[q][0] = acc[q][1] = 0ull;
    }
  };
  tok_issue_chunk(T, t, unit, tok_smem);
  for (int i = 0; unit < units; ++i, unit += gridDim.x) {
    const int next = unit + static_cast<int>(gridDim.x);
    if (next < units) {
      tok_issue_chunk(T, t, next, tok_smem + ((i + 1) & 1) * stage);
      cp_async_wait_group<1>();
    } else {
      cp_async_wait_group<0>();
    }
    __syncthreads();
    int b = 0;
    while (b + 1 < t.nb && t.unit_prefix1[b + 1] <= unit) ++b;
    const int r0 = (unit - t.unit_prefix1[b]) * t.rows1;
    const int nt = min(t.rows1, t.n[b] - r0);
    if (b != cur_b) {
      flush();
      cur_b = b;
    }
    const uint32_t* rows = tok_smem + (i & 1) * stage;
    float* iv_s = inv[i & 1];
    for (int p = warp; p < nt; p += kApcThreads / 32) {
      const uint32_t* row = rows + p * words;
      float ss = 0.f;
      for (int w = lane; w < words; w += 32) {
        const uint32_t v = row[w];
        const float lo = bf16_lo(v), hi = bf16_hi(v);
        ss = fmaf(lo, lo, fmaf(hi, hi, ss));
      }
      ss = warp_sum_f(ss);
      if (lane == 0) {
        const float iv = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
        iv_s[p] = iv;
        inv_norm[t.tok0[b] + r0 + p] = iv;
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kTok1MaxSlots; ++q) {
      const int w = threadIdx.x + q * kApcThreads;
      if (w < words) {
        float2 a = make_float2(0.f, 0.f);
        for (int p = 0; p < nt; ++p) {
          const uint32_t v = rows[p * words + w];
          const float iv = iv_s[p];
          a = ptx::ffma2(make_float2(iv, iv), make_float2(bf16_lo(v), bf16_hi(v)), a);
        }
        acc[q][0] += fix32_signed(a.x);
        acc[q][1] += fix32_signed(a.y);
      }
    }
    __syncthreads();   // this stage is refilled two chunks on
  }
  flush();
}

// Pass 2: c = sums / N, phi = |c|^2, c_hat = c / |c|, then d_i = |t_hat_i - c_hat| directly
// (warp per token).
__global__ void __launch_bounds__(kApcThreads) apc_tok_pass2(const uint32_t* __restrict__ T,
                                                             const __grid_constant__ TokTable t,
                                                             const float* __restrict__ inv_norm,
                                                             const unsigned long long* __restrict__ sums,
                                                             float* __restrict__ d_out,
                                                             pace_apc_stats* __restrict__ stats,
                                                             TailWork* __restrict__ work) {
  __shared__ __align__(16) float chat[kTokMaxD];
  __shared__ float red[kApcThreads / 32];
  const int unit = blockIdx.x;
  const int b = find_tok_image(t, unit);
  const int c0 = (unit - t.unit_prefix[b]) * kTokChunk;
  const int nt = min(kTokChunk, t.n[b] - c0);
  const int N = t.n[b], D = t.D, words = D >> 1;
  const float inv_n = 1.0f / static_cast<float>(N);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned long long* sb = sums + static_cast<int64_t>(t.b_base + b) * kSumSlots * D;
  float part = 0.f;
  for (int k = threadIdx.x; k < D; k += kApcThreads) {
    const float cv = unfix32<true>(sb[k], inv_n);
    chat[k] = cv;
    part = fmaf(cv, cv, part);
  }
  part = warp_sum_f(part);
  if (lane == 0) red[warp] = part;
  __syncthreads();
  float phi = 0.f;
#pragma unroll
  for (int w = 0; w < kApcThreads / 32; ++w) phi += red[w];
  const float inv_c = phi > 0.f ? 1.0f / sqrtf(phi) : 0.f;
  for (int k = threadIdx.x; k < D; k += kApcThreads) chat[k] *= inv_c;
  if (c0 == 0 && threadIdx.x == 0) {
    stats[t.b_base + b].phi = phi;
    stats[t.b_base + b].rho_g = 1.0f - phi;
    stats[t.b_base + b].n_patches = N;
    stats[t.b_base + b].k_tail = t.ktail[b];
  }
  __syncthreads();
  const uint32_t* base = T + (t.tok0[b] + c0) * words;
  const float2* chat2 = reinterpret_cast<const float2*>(chat);
  TailRun tail(work + t.b_base + b);   // lane 0's
  for (int p = warp; p < nt; p += kApcThreads / 32) {
    const uint32_t* row = base + static_cast<int64_t>(p) * words;
    const float iv = inv_norm[t.tok0[b] + c0 + p];
    float acc0 = 0.f, acc1 = 0.f;
    for (int w = lane; w < words; w += 32) {
      const uint32_t v = row[w];
      const float2 ch = chat2[w];
      const float e0 = fmaf(bf16_lo(v), iv, -ch.x), e1 = fmaf(bf16_hi(v), iv, -ch.y);
      acc0 = fmaf(e0, e0, acc0);
      acc1 = fmaf(e1, e1, acc1);
    }
    const float acc = warp_sum_f(acc0 + acc1);
    if (lane == 0) {
      const float dv = sqrtf(acc);
      d_out[t.tok0[b] + c0 + p] = dv;
      tail.add(dv);
    }
  }
  tail.flush();
}

// Token widths of up to 1536 in whole 16-byte vectors (the ViT widths): a warp per token, lane l
// holding vectors l, l + 32, .. in registers, so a token is read once per pass straight into the
// norm, the column sums and the distance, with no staging and no block barrier.  Pass 1 is bound by a
// warp's chain per token (load, sum of squares over the lanes, square root and division, column sums),
// pass 2 by L2 and HBM.  42196 tokens of 1280: 84.5 us for the call staged, 55.5 in registers (passes
// 38.8 + 31.9, now 25.3 + 28).  Other widths, and tokens off a 16-byte boundary, take the staged kernels
// above: with six vectors a lane of pass 1 has its 168 registers full (two rows in flight, a row unpacked
// and its column sums, 8 per vector each), and a seventh would spill in every token's chain.
constexpr int kTokVecMax = 6;            // 16-byte vectors per lane
constexpr int kTokThreads = 384;         // of pass 1: one CTA per SM, since each ends an image with D atomics
constexpr int kTokAhead = 2;             // tokens a warp of pass 1 has in flight
constexpr int kTokRun = 8;               // tokens (from a multiple of it on) whose column sums stay in fp32
                                         // before they are rounded, whatever the batch and the grid
static_assert(kTokRun % kTokAhead == 0, "a run's tokens keep to their buffers");
// A finite sum over a run is at most this: a coordinate of a normalised token is at most 1, or sqrt(3/2)
// when |T|^2 is so small that it is rounded to a multiple of 2^-149.
constexpr float kTokMost = 2.0f * kTokRun;
static_assert(kTokMost < 512.0f, "the range of fix_add");

// 2^-32 fixed point without conversions: v + 1.5 2^11 leaves v rounded to 2^-12 in the low mantissa
// bits, the exact remainder times 2^32 plus 1.5 2^23 the rest, so acc collects
// bits(hi) 2^20 + bits(lo), i.e. round(v 2^32) (ties to even, |v| < 2^9) plus the constant kFixBias,
// which the caller takes off again once per addition.
constexpr unsigned long long kFixBias = (0x45400000ull << 20) + 0x4B400000ull;
__device__ __forceinline__ void fix_add(unsigned long long& acc, float v) {
  const float m = v + 3072.0f;
  const float l = fmaf(v - (m - 3072.0f), 4294967296.0f, 12582912.0f);
  acc += static_cast<unsigned long long>(__float_as_uint(m)) * 1048576ull;
  acc += __float_as_uint(l);
}

template <int V>
struct TokRow {
  uint4 v[V];
};
template <int V>
__device__ __forceinline__ void tok_load(TokRow<V>& r, const uint4* __restrict__ T, int64_t token, int vecs) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int c = lane + 32 * i;
    r.v[i] = i < V - 1 || c < vecs ? __ldg(T + token * vecs + c) : make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ float2 bf16_pair(uint32_t v) { return make_float2(bf16_lo(v), bf16_hi(v)); }
__device__ __forceinline__ uint32_t word_of(const uint4& v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }

// CTA c's share [a0, a1) of the table's runs of kTokRun tokens, counted over the images.
__device__ __forceinline__ void tok_share(const TokTable& t, int& a0, int& a1) {
  const int64_t runs = t.run_prefix[t.nb];
  a0 = static_cast<int>(runs * blockIdx.x / gridDim.x);
  a1 = static_cast<int>(runs * (blockIdx.x + 1) / gridDim.x);
}

// Pass 1: the warps take the runs of their CTA's share in turn.
template <int V>
__global__ void __launch_bounds__(kTokThreads, 1) apc_tok_vec1(const uint4* __restrict__ T,
                                                               const __grid_constant__ TokTable t,
                                                               float* __restrict__ inv_norm,
                                                               unsigned long long* __restrict__ sums) {
  // [warps][kRow]: a warp's totals, lane-contiguous (no bank conflicts): entry 2 (32 (4 i + e) + lane)
  // + u is column 8 (lane + 32 i) + 2 e + u
  extern __shared__ __align__(16) unsigned long long tok_acc[];
  ptx::launch_dependents();
  constexpr int kWarps = kTokThreads / 32;
  const int D = t.D, vecs = D >> 3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kRow = V * 256;
  unsigned long long* own = tok_acc + warp * kRow;
  auto clear_own = [&]() {
#pragma unroll
    for (int i = 0; i < 4 * V; ++i) reinterpret_cast<ulonglong2*>(own)[32 * i + lane] = make_ulonglong2(0ull, 0ull);
  };
  int a0, a1, cur_b = -1, runs = 0;
  // adds the CTA's totals of image cur_b (`runs` additions to each column) to the image's sums
  auto finish = [&]() {
    ptx::grid_dependency_wait();   // the zeroed sums
    __syncthreads();
    if (cur_b < 0) return;
    const unsigned long long bias = kFixBias * static_cast<unsigned>(runs);
    unsigned long long* sb = sums + (static_cast<int64_t>(t.b_base + cur_b) * kSumSlots + blockIdx.x % kSumSlots) * D;
    for (int k = threadIdx.x; k < kRow; k += kTokThreads) {
      const int c = ((k >> 1) & 31) + 32 * (k >> 8), e = (k >> 6) & 3;   // entry k's vector and word
      if (c >= vecs) continue;
      unsigned long long x = 0ull;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) x += tok_acc[w * kRow + k];
      atomicAdd(sb + 8 * c + 2 * e + (k & 1), x - bias);
    }
  };
  tok_share(t, a0, a1);
  clear_own();
  for (int b = 0; b < t.nb; ++b) {
    const int lo = max(a0, t.run_prefix[b]), hi = min(a1, t.run_prefix[b + 1]);
    if (lo >= hi) continue;
    if (cur_b >= 0) {   // the CTA moves to the next image
      finish();
      __syncthreads();
      clear_own();
    }
    cur_b = b;
    runs = hi - lo;
    const int64_t end = t.tok0[b] + t.n[b];
    auto token = [&](int run, int q) { return t.tok0[b] + static_cast<int64_t>(run - t.run_prefix[b]) * kTokRun + q; };
    TokRow<V> buf[kTokAhead];
    auto fetch = [&](TokRow<V>& r, int run, int q) {
      const int64_t tok = token(run, q);
      if (run < hi && tok < end) tok_load<V>(r, T, tok, vecs);
    };
#pragma unroll
    for (int r = 0; r < kTokAhead; ++r) fetch(buf[r], lo + warp, r);
    for (int run = lo + warp; run < hi; run += kWarps) {
      float2 col[V][4];
#pragma unroll
      for (int i = 0; i < V; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) col[i][e] = make_float2(0.f, 0.f);
#pragma unroll
      for (int r = 0; r < kTokRun; ++r) {
        TokRow<V>& row = buf[r % kTokAhead];
        if (token(run, r) < end) {   // warp-uniform
          float2 x[V][4];
          float2 ss2 = make_float2(0.f, 0.f), ss3 = ss2;
#pragma unroll
          for (int i = 0; i < V; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              x[i][e] = bf16_pair(word_of(row.v[i], e));
              if (e & 1) ss3 = ptx::ffma2(x[i][e], x[i][e], ss3);
              else ss2 = ptx::ffma2(x[i][e], x[i][e], ss2);
            }
          if (r + kTokAhead < kTokRun) fetch(row, run, r + kTokAhead);
          else fetch(row, run + kWarps, r + kTokAhead - kTokRun);
          ss2 = ptx::fadd2(ss2, ss3);
          const float ss = warp_sum_f(ss2.x + ss2.y);
          const float iv = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
          if (lane == 0) inv_norm[token(run, r)] = iv;
          const float2 iv2 = make_float2(iv, iv);
#pragma unroll
          for (int i = 0; i < V; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) col[i][e] = ptx::ffma2(iv2, x[i][e], col[i][e]);
        }
      }
      // the run's sums, rounded to fixed point, into this warp's totals
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int c = lane + 32 * i;
        if (i < V - 1 || c < vecs) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            ulonglong2* p = reinterpret_cast<ulonglong2*>(own) + 32 * (4 * i + e) + lane;
            ulonglong2 x = *p;
            fix_add(x.x, fabsf(col[i][e].x) <= kTokMost ? col[i][e].x : 0.f);   // (a NaN counts as 0)
            fix_add(x.y, fabsf(col[i][e].y) <= kTokMost ? col[i][e].y : 0.f);
            *p = x;
          }
        }
      }
    }
  }
  finish();
}

// Pass 2: c = sums / N, phi = |c|^2, c_hat = c / |c| in registers, then d_i = |t_hat_i - c_hat|
// directly.  The tokens are taken from the last to the first: the last ones read by pass 1 are the
// ones still in L2.
template <int V>
__global__ void __launch_bounds__(kApcThreads, 2) apc_tok_vec2(const uint4* __restrict__ T,
                                                               const __grid_constant__ TokTable t,
                                                               const float* __restrict__ inv_norm,
                                                               const unsigned long long* __restrict__ sums,
                                                               float* __restrict__ d_out,
                                                               pace_apc_stats* __restrict__ stats,
                                                               TailWork* __restrict__ work) {
  __shared__ __align__(16) float chat[kTokVecMax * 256];
  __shared__ float red[kApcThreads / 32];
  ptx::launch_dependents();
  bool waited = false;
  constexpr int kWarps = kApcThreads / 32;
  const int D = t.D, vecs = D >> 3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t first = t.tok0[0], total = t.tok0[t.nb - 1] + t.n[t.nb - 1] - first;
  const int64_t a0 = first + total * blockIdx.x / gridDim.x, a1 = first + total * (blockIdx.x + 1) / gridDim.x;
  for (int b = t.nb - 1; b >= 0; --b) {
    const int64_t lo = max(a0, t.tok0[b]), hi = min(a1, t.tok0[b] + t.n[b]);
    if (lo >= hi) continue;
    int64_t tok = hi - 1 - warp;
    TokRow<V> buf[2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (tok - r * kWarps >= lo) tok_load<V>(buf[r], T, tok - r * kWarps, vecs);
    if (!waited) ptx::grid_dependency_wait();   // (the tokens do not depend on pass 1)
    waited = true;
    float inv[2];   // the rows' inverse norms, loaded with them
#pragma unroll
    for (int r = 0; r < 2; ++r) inv[r] = tok - r * kWarps >= lo ? __ldcg(inv_norm + tok - r * kWarps) : 0.f;
    const int N = t.n[b];
    const float inv_n = 1.0f / static_cast<float>(N);
    const unsigned long long* sb = sums + static_cast<int64_t>(t.b_base + b) * kSumSlots * D;
    float part = 0.f;
    for (int k = threadIdx.x; k < D; k += kApcThreads) {
      unsigned long long x = 0ull;
#pragma unroll
      for (int r = 0; r < kSumSlots; ++r) x += __ldcg(sb + r * D + k);
      const float cv = unfix32<true>(x, inv_n);
      chat[k] = cv;
      part = fmaf(cv, cv, part);
    }
    part = warp_sum_f(part);
    if (lane == 0) red[warp] = part;
    __syncthreads();
    float phi = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) phi += red[w];
    const float inv_c = phi > 0.f ? 1.0f / sqrtf(phi) : 0.f;
    float2 nch[V][4];   // -c_hat of this lane's columns
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int c = lane + 32 * i;
      const bool has = i < V - 1 || c < vecs;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 x = has ? *reinterpret_cast<const float2*>(chat + 8 * c + 2 * q) : make_float2(0.f, 0.f);
        nch[i][q] = make_float2(-x.x * inv_c, -x.y * inv_c);
      }
    }
    if (lo == t.tok0[b] && threadIdx.x == 0) {
      stats[t.b_base + b].phi = phi;
      stats[t.b_base + b].rho_g = 1.0f - phi;
      stats[t.b_base + b].n_patches = N;
      stats[t.b_base + b].k_tail = t.ktail[b];
    }
    TailRun tail(work + t.b_base + b);   // lane 0's
    while (tok >= lo) {
#pragma unroll
      for (int r = 0; r < 2; ++r, tok -= kWarps) {
        if (tok < lo) break;
        const float2 iv2 = make_float2(inv[r], inv[r]);
        float2 acc = make_float2(0.f, 0.f), acc1 = acc;
#pragma unroll
        for (int i = 0; i < V; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 e = ptx::ffma2(bf16_pair(word_of(buf[r].v[i], q)), iv2, nch[i][q]);
            if (q & 1) acc1 = ptx::ffma2(e, e, acc1);
            else acc = ptx::ffma2(e, e, acc);
          }
        if (tok - 2 * kWarps >= lo) {
          tok_load<V>(buf[r], T, tok - 2 * kWarps, vecs);
          inv[r] = __ldcg(inv_norm + tok - 2 * kWarps);
        }
        acc = ptx::fadd2(acc, acc1);
        const float d2 = warp_sum_f(acc.x + acc.y);
        if (lane == 0) {
          const float dv = sqrtf(d2);
          d_out[tok] = dv;
          tail.add(dv);
        }
      }
    }
    tail.flush();
    __syncthreads();   // chat and red are rewritten for the next image
  }
}

// Called by all 1024 threads, thread t holding the counts of bins top .. top - PER + 1 (top =
// PER * 1024 - 1 - PER * t): the bin holding the r-th largest entry, counting from the last bin down
// (1 <= r <= total): sel[0] = that bin, sel[1] = entries in the bins above it, *count = entries in it.
// wsum: 32 words.
template <int PER>
__device__ __forceinline__ void select_from_counts(const unsigned (&c)[PER], int top, unsigned r, unsigned* sel,
                                                   unsigned* wsum, unsigned* count) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned own = 0u;
#pragma unroll
  for (int q = 0; q < PER; ++q) own += c[q];
  unsigned incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  incl += __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0u);   // entries in the warps before
  const unsigned excl = incl - own;
  if (excl < r && incl >= r) {   // exactly one thread
    unsigned above = excl;
    int q = 0;
#pragma unroll
    for (int qq = 0; qq < PER - 1; ++qq)
      if (q == qq && above + c[qq] < r) {
        above += c[qq];
        q = qq + 1;
      }
    unsigned n = c[0];
#pragma unroll
    for (int qq = 1; qq < PER; ++qq)
      if (q == qq) n = c[qq];
    sel[0] = static_cast<unsigned>(top - q);
    sel[1] = above;
    *count = n;
  }
  __syncthreads();
}

// The same for NBINS counts in shared memory; returns the entries in the bin.
template <int NBINS>
__device__ __forceinline__ unsigned select_from_top(const unsigned* bins, unsigned r, unsigned* sel, unsigned* wsum) {
  constexpr int PER = NBINS / 1024;   // bins per thread
  static_assert(PER >= 1 && PER * 1024 == NBINS, "bins");
  __shared__ unsigned count;
  const int top = NBINS - 1 - PER * static_cast<int>(threadIdx.x);
  static_assert(PER == 4, "one 16-byte read per thread");
  const uint4 v = *reinterpret_cast<const uint4*>(bins + top - 3);
  const unsigned c[4] = {v.w, v.z, v.y, v.x};
  select_from_counts<4>(c, top, r, sel, wsum, &count);
  return count;
}

// Eq. 5-6 and R3-R4 from the tail mean d_top of image b: rho_d, rho, r and the target size.
__device__ __forceinline__ void tail_finish(const ApcTable& t, int b, const TailParams& prm,
                                            pace_apc_stats* __restrict__ stats, float rho_g, float d_top) {
  const float rho_d = fminf(d_top / prm.gamma, 1.0f);
  const float rho = prm.alpha * rho_g + (1.0f - prm.alpha) * rho_d;
  const float r = fminf(fmaxf(rho, prm.r_min), prm.r_max);
  const float sr = sqrtf(fmaxf(r, 0.0f));
  const int al = prm.align;
  const int H = t.H[b], W = t.W[b];
  int ho = al * static_cast<int>(floorf(static_cast<float>(H) * sr / al + 0.5f));
  int wo = al * static_cast<int>(floorf(static_cast<float>(W) * sr / al + 0.5f));
  ho = min(H, max(al, ho));
  wo = min(W, max(al, wo));
  pace_apc_stats& st = stats[t.b_base + b];
  st.d_top = d_top;
  st.rho_d = rho_d;
  st.rho = rho;
  st.r = r;
  st.h_out = ho;
  st.w_out = wo;
}

// The density tail (Eq. 5: the mean of the k_tail largest d_i, then Eq. 6 and R3-R4).  Pass 2 has
// counted and summed the distances in 4096 value buckets of width 1/2048 (the top one also takes
// anything above), so the k-th largest's bucket and the sum of everything above it follow from the
// counts alone, and only that bucket's members are looked for in the distances.  A cluster of
// CTAs per image: every CTA selects the bucket for itself, scans its share of the distances
// (loaded before the selection, so that the two latencies overlap) and appends the members to the
// first CTA's shared list, with one reservation per warp (a remote atomic and its answer take about
// half a microsecond, and one per distance row made eight in a row); after one cluster barrier the
// first CTA narrows the members to the k-th largest distance T (at most kTailRank: each ranked
// against the others; else rounds of 4096 bins over the key offsets from the smallest member) and
// writes the statistics.  A bucket with too many different members for the list is narrowed over the
// whole array by such rounds.  Everything is latency: a chain of L2 reads and block barriers.
constexpr int kTailList = 4096;    // members listed
// Members ranked directly: c^2 comparisons over 1024 threads take 1.0 us at 68 members, 4.6 at 229, 16
// at 1024; a round of bins about 1 us whatever their number.  The line lies where rank_in_list goes from
// eight threads per member to four.
constexpr int kTailRank = 128;
constexpr int kTailAhead = 8;      // distances per thread loaded ahead of the selection
constexpr int kTailCluster = 8;    // CTAs per image above kTailAhead * 1024 distances

__global__ void __launch_bounds__(1024) apc_tail(const __grid_constant__ ApcTable t, const float* __restrict__ d,
                                                 TailParams prm, pace_apc_stats* __restrict__ stats,
                                                 const TailWork* __restrict__ work) {
  __shared__ unsigned list[kTailList];
  __shared__ __align__(16) unsigned bins[kTailBins];   // bins of the narrowing rounds
  __shared__ unsigned sel[2], selb[2];
  __shared__ unsigned cred[32];
  __shared__ unsigned long long fred[32];
  __shared__ unsigned list_n, key_min, key_max;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(blockIdx.x), ncta = static_cast<int>(gridDim.x);
  if (tid == 0) {
    list_n = 0u;
    key_min = 0xFFFFFFFFu;
    key_max = 0u;
  }
  if (ncta > 1) ptx::cluster_arrive();   // the first CTA's list is ready: waited for before the first append
  ptx::begin_call();   // (nothing of this call follows: the next call's first kernel)
  const int b = blockIdx.y;
  const int N = t.n[b];
  const TailWork* w = work + (t.b_base + b);
  const float* db = d + t.patch0[b];
  const unsigned k = static_cast<unsigned>(t.ktail[b]);
  // this CTA's distances rank * 1024 + tid, + 1024 ncta, ..
  const int i0 = rank * 1024 + tid, step = ncta * 1024;
  float ahead[kTailAhead];
#pragma unroll
  for (int q = 0; q < kTailAhead; ++q) {
    const int i = i0 + q * step;
    ahead[q] = i < N ? __ldcg(db + i) : 0.f;
  }
  // level 1: thread t holds buckets 4095 - 4t .. 4092 - 4t
  const int top = kTailBins - 1 - 4 * tid;
  const uint4 cv = __ldcg(reinterpret_cast<const uint4*>(w->hist + top - 3));
  const unsigned c4[4] = {cv.w, cv.z, cv.y, cv.x};
  unsigned long long s_fix = 0ull;
  ulonglong2 s01, s23;
  float rho_g = 0.f;
  if (rank == 0) {
    s23 = __ldcg(reinterpret_cast<const ulonglong2*>(w->sum + top - 3));
    s01 = __ldcg(reinterpret_cast<const ulonglong2*>(w->sum + top - 1));
    if (tid == 0) rho_g = __ldcg(&stats[t.b_base + b].rho_g);
  }
  select_from_counts<4>(c4, top, k, sel, cred, selb);
  const int tb = static_cast<int>(sel[0]);
  const unsigned above_n = sel[1];     // entries in the buckets above it
  const unsigned cb = selb[0];         // entries in the k-th largest's bucket
  if (rank == 0) {                     // the sum of the distances in the buckets above it
    if (top > tb) s_fix += s01.y;
    if (top - 1 > tb) s_fix += s01.x;
    if (top - 2 > tb) s_fix += s23.y;
    if (top - 3 > tb) s_fix += s23.x;
  }
  const bool listed = cb <= kTailList;
  unsigned* list0 = list;
  unsigned *n0 = &list_n, *min0 = &key_min, *max0 = &key_max;
  if (ncta > 1) {
    ptx::cluster_wait();
    list0 = cluster.map_shared_rank(list, 0);
    n0 = cluster.map_shared_rank(&list_n, 0);
    min0 = cluster.map_shared_rank(&key_min, 0);
    max0 = cluster.map_shared_rank(&key_max, 0);
  }
  // this CTA's members of the bucket: the keys lo .. lo + span - 1 (bucket 0 also takes NaN, whose key
  // lies elsewhere)
  unsigned lo = __float_as_uint(static_cast<float>(tb) * (1.0f / 2048.0f));
  unsigned span = (tb == kTailBins - 1 ? 0x7F800001u : __float_as_uint(static_cast<float>(tb + 1) * (1.0f / 2048.0f))) - lo;
  const unsigned bucket_lo = lo, bucket_span = span;
  unsigned kmin = 0xFFFFFFFFu, kmax = 0u;
  for (int base = rank * 1024; base < N; base += kTailAhead * step) {   // uniform trip count per CTA
    unsigned members = 0u;   // bit q: ahead[q] is one
#pragma unroll
    for (int q = 0; q < kTailAhead; ++q) {
      const bool in = tb != 0 ? __float_as_uint(ahead[q]) - bucket_lo < bucket_span   // (0 past the end: no member)
                              : base + tid + q * step < N && tail_bucket(ahead[q]) == 0;
      members |= in ? 1u << q : 0u;
    }
    const unsigned mine = static_cast<unsigned>(__popc(members)), all = __reduce_add_sync(0xffffffffu, mine);
    if (all != 0u) {   // warp-uniform
      unsigned slot = 0u;
      if (listed) {
        unsigned incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned n = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += n;
        }
        if (lane == 0) slot = atomicAdd(n0, all);
        slot = __shfl_sync(0xffffffffu, slot, 0) + incl - mine;
      }
#pragma unroll
      for (int q = 0; q < kTailAhead; ++q) {
        if (!((members >> q) & 1u)) continue;
        const unsigned key = __float_as_uint(ahead[q]);
        kmin = min(kmin, key);
        kmax = max(kmax, key);
        if (listed) list0[slot++] = key;
      }
    }
    if (base + kTailAhead * step < N) {
#pragma unroll
      for (int q = 0; q < kTailAhead; ++q) {
        const int i = base + tid + (kTailAhead + q) * step;
        ahead[q] = i < N ? __ldcg(db + i) : 0.f;
      }
    }
  }
  if (!listed) {
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0 && kmax >= kmin) {
      atomicMin(min0, kmin);
      atomicMax(max0, kmax);
    }
  }
  if (ncta > 1) cluster.sync();
  else __syncthreads();
  if (rank != 0) return;
  // level 2: T = the k-th largest distance; the members of the bucket above T are summed in fixed
  // point (c counts every distance above T)
  unsigned remaining = k - above_n, cnt = 0u;
  unsigned prefix;
  if (cb <= kTailRank) {
    // one member per thread, ranked against the whole list: a member with fewer than `remaining`
    // members at or above it lies above the k-th largest (and is summed); with fewer than
    // `remaining` above it but at least that many at or above it, it is the k-th largest
    int mi;
    unsigned gt, ge;
    if (rank_in_list(list, cb, mi, gt, ge)) {
      const unsigned mine = list[mi];
      if (ge < remaining) {
        s_fix += fix32(__uint_as_float(mine));
        ++cnt;
      } else if (gt < remaining) {
        selb[1] = mine;   // the same key from every member equal to it
      }
    }
    __syncthreads();
    prefix = selb[1];
  } else if (listed) {
    unsigned mn = 0xFFFFFFFFu, mx = 0u;
    for (int i = tid; i < static_cast<int>(cb); i += blockDim.x) {
      mn = min(mn, list[i]);
      mx = max(mx, list[i]);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) {
      atomicMin(&key_min, mn);
      atomicMax(&key_max, mx);
    }
    static_assert(kTailBins == 4 * 1024, "one 16-byte store per thread clears the bins");
    reinterpret_cast<uint4*>(bins)[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    lo = key_min;
    span = key_max - lo + 1u;
    unsigned only = 0u;   // the k-th largest is the one member among this many keys from lo on
    while (span > 1u) {   // (one key: every member is the same distance)
      const int bits = 32 - __clz(span - 1u);
      const int shift = bits > 12 ? bits - 12 : 0;
      for (int base = 0; base < static_cast<int>(cb); base += blockDim.x) {
        const unsigned off = base + tid < static_cast<int>(cb) ? list[base + tid] - lo : span;   // wraps for keys below lo
        const unsigned bin = off < span ? off >> shift : kTailBins;
        const unsigned first = __shfl_sync(0xffffffffu, bin, 0);
        if (__all_sync(0xffffffffu, bin == first)) {   // equal distances: one addition
          if (lane == 0 && first < kTailBins) atomicAdd(&bins[first], 32u);
        } else if (bin < kTailBins) {
          atomicAdd(&bins[bin], 1u);
        }
      }
      __syncthreads();
      const unsigned in_bin = select_from_top<kTailBins>(bins, remaining, sel, cred);
      lo += sel[0] << shift;
      remaining -= sel[1];
      if (shift == 0) break;
      if (in_bin == 1u) {
        only = 1u << shift;
        break;
      }
      span = min(span - (sel[0] << shift), 1u << shift);
      __syncthreads();   // everyone has read sel and the bins
      reinterpret_cast<uint4*>(bins)[tid] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
    prefix = lo;
    if (only != 0u) {
      for (int i = tid; i < static_cast<int>(cb); i += blockDim.x)
        if (list[i] - lo < only) selb[1] = list[i];
      __syncthreads();
      prefix = selb[1];
    }
    for (int i = tid; i < static_cast<int>(cb); i += blockDim.x) {
      const unsigned key = list[i];
      if (key > prefix) {
        s_fix += fix32(__uint_as_float(key));
        ++cnt;
      }
    }
  } else if (key_min == key_max) {   // every member is the same distance
    prefix = key_min;
  } else {
    // a crowded bucket: its members by key offset from its first key over the whole array,
    // 4096 offsets (2^shift keys each) at a time, until one key is left
    while (true) {
      const int bits = 32 - __clz(span - 1u);
      const int shift = bits > 12 ? bits - 12 : 0;
      __syncthreads();                               // everyone has read sel and the bins
      for (int i = tid; i < kTailBins; i += blockDim.x) bins[i] = 0u;
      __syncthreads();
      for (int base = 0; base < N; base += blockDim.x) {   // uniform trip count: __match_any_sync below
        const int i = base + tid;
        const unsigned off = i < N ? __float_as_uint(__ldcg(db + i)) - lo : span;   // wraps for keys below lo
        const bool in = off < span;
        const unsigned digit = in ? off >> shift : kTailBins;
        const unsigned members = __ballot_sync(0xffffffffu, in);
        if (__popc(members) > 4) {
          const unsigned peers = __match_any_sync(0xffffffffu, digit);
          if (in && lane == __ffs(peers) - 1) atomicAdd(&bins[digit], static_cast<unsigned>(__popc(peers)));
        } else if (in) {
          atomicAdd(&bins[digit], 1u);
        }
      }
      __syncthreads();
      select_from_top<kTailBins>(bins, remaining, sel, cred);
      lo += sel[0] << shift;
      remaining -= sel[1];
      if (shift == 0) break;
      span = min(span - (sel[0] << shift), 1u << shift);
    }
    prefix = lo;
    for (int i = tid; i < N; i += blockDim.x) {   // the bucket's members above T
      const unsigned key = __float_as_uint(__ldcg(db + i));
      if (key > prefix && key - bucket_lo < bucket_span) {
        s_fix += fix32(__uint_as_float(key));
        ++cnt;
      }
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  for (int o = 16; o > 0; o >>= 1) s_fix += __shfl_xor_sync(0xffffffffu, s_fix, o);
  __syncthreads();   // the earlier reads of cred are done
  if (lane == 0) {
    cred[warp] = cnt;
    fred[warp] = s_fix;
  }
  __syncthreads();
  if (warp == 0) {
    const unsigned c = above_n + __reduce_add_sync(0xffffffffu, cred[lane]);
    unsigned long long f = fred[lane];
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) {
      const float T = __uint_as_float(prefix);   // k-th largest d
      const float tot = unfix32<false>(f, 1.0f) + static_cast<float>(k - c) * T;   // the rest equal T
      tail_finish(t, b, prm, stats, rho_g, tot / static_cast<float>(k));
    }
  }
}

// ------------------------------------------------------------------------------------------------
// pixel-statistic previews (App. "Shallow Feature Preview Ablation"): one small token per patch,
// then Eq. 1-6 on those tokens
// ------------------------------------------------------------------------------------------------
// Token of patch i: kPixDim floats, zero-padded.  Feature codes as pace_apc_feature.
constexpr int kPixDim = 8;
constexpr int kFeatRgb = 0, kFeatEntropy = 1, kFeatEdge = 2, kFeatLaplacian = 3;
constexpr int kLumaR = 299, kLumaG = 587, kLumaB = 114;   // Y' = 299 R + 587 G + 114 B (BT.601, thousandths)
constexpr int kLumaScale = 255000;                         // Y' of white
constexpr long long kEdgeThr2 = 63750LL * 63750LL;         // (0.25 * 255000)^2: Sobel magnitude test in integers

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int warp_sum_i(int v) { return __reduce_add_sync(0xffffffffu, v); }

// One warp computes the feature token of the patch whose pixel (y, x) is staged at px(y, x), the same
// in every lane.  Lane x + 14 h walks down column x, in half h of the rows: no index arithmetic per
// pixel, and the 3 x 3 operators take their neighbours from the next lanes and from the rows before (with
// a pixel per lane and step and the luma in shared memory the edge density of 1904 x 1064 took
// 10.3 us, now 7.0; bound by issue).  `hist` (48 ints) is the warp's scratch in shared memory.
template <typename Pixel>
__device__ __forceinline__ void patch_feature(Pixel px, int feature, int* hist, float (&tok)[kPixDim]) {
  const int lane = threadIdx.x & 31;
  const int h = lane >= kPatch ? 1 : 0, x = lane - kPatch * h;
  const bool live = lane < 2 * kPatch;
#pragma unroll
  for (int k = 0; k < kPixDim; ++k) tok[k] = 0.f;
  if (feature == kFeatRgb) {
    uint32_t s[3] = {0u, 0u, 0u}, q[3] = {0u, 0u, 0u};
    if (live) {
#pragma unroll
      for (int k = 0; k < kPatch / 2; ++k) {
        const uint8_t* p = px(kPatch / 2 * h + k, x);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const uint32_t v = p[c];
          s[c] += v;
          q[c] += v * v;
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const uint32_t S = __reduce_add_sync(0xffffffffu, s[c]);
      const uint32_t Q = __reduce_add_sync(0xffffffffu, q[c]);
      constexpr float kInv = 1.0f / (196.0f * 255.0f);
      tok[c] = static_cast<float>(S) * kInv;
      tok[3 + c] = sqrtf(static_cast<float>(196u * Q - S * S)) * kInv;   // 196 Q - S^2 >= 0, < 2^32
    }
    tok[6] = 1.f;
  } else if (feature == kFeatEntropy) {
    for (int i = lane; i < 48; i += 32) hist[i] = 0;
    __syncwarp();
    if (live) {
#pragma unroll
      for (int k = 0; k < kPatch / 2; ++k) {
        const uint8_t* p = px(kPatch / 2 * h + k, x);
#pragma unroll
        for (int c = 0; c < 3; ++c) atomicAdd(&hist[c * 16 + (p[c] >> 4)], 1);
      }
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float e = 0.f;
      if (lane < 16) {
        const int n = hist[c * 16 + lane];
        if (n > 0) {
          const float pr = static_cast<float>(n) * (1.0f / 196.0f);
          e = -pr * log2f(pr);
        }
      }
      e = warp_sum_f(e);
      tok[c] = e * 0.25f;
    }
    tok[3] = 1.f;
    __syncwarp();   // hist is rewritten by the warp's next patch
  } else {
    // rows 6 h .. 6 h + 7: the interior rows 6 h + 1 .. 6 h + 6 and their neighbours; a column's left and
    // right neighbours are the lanes beside it (columns 1 to 12 have them in their own half)
    constexpr int kRows = kPatch / 2 + 1;
    const bool inner = live && x >= 1 && x <= kPatch - 2;
    const int xs = min(x, kPatch - 1);
    auto luma = [&](int k) {
      const uint8_t* p = px((kPatch / 2 - 1) * h + k, xs);
      return kLumaR * p[0] + kLumaG * p[1] + kLumaB * p[2];
    };
    if (feature == kFeatEdge) {
      int cnt = 0, d0 = 0, d1 = 0, s0 = 0, s1 = 0;   // of the two rows before: right - left, left + 2 own + right
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int own = luma(k), left = __shfl_up_sync(0xffffffffu, own, 1), right = __shfl_down_sync(0xffffffffu, own, 1);
        const int d = right - left, sm = left + 2 * own + right;
        if (k >= 2) {
          const long long gx = d0 + 2 * d1 + d, gy = sm - s0;
          cnt += (gx * gx + gy * gy > kEdgeThr2) ? 1 : 0;
        }
        d0 = d1;
        d1 = d;
        s0 = s1;
        s1 = sm;
      }
      tok[0] = static_cast<float>(warp_sum_i(inner ? cnt : 0)) * (1.0f / 144.0f);
    } else {
      int sl = 0, above = 0, centre = 0, beside = 0;   // of the rows before: row k - 2, row k - 1 and its neighbours
      long long sl2 = 0;
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int own = luma(k), left = __shfl_up_sync(0xffffffffu, own, 1), right = __shfl_down_sync(0xffffffffu, own, 1);
        if (k >= 2) {
          const int l = beside + above + own - 4 * centre;
          sl += l;
          sl2 += static_cast<long long>(l) * l;
        }
        above = centre;
        centre = own;
        beside = left + right;
      }
      const long long S = static_cast<long long>(warp_sum_i(inner ? sl : 0)), Q = warp_sum_ll(inner ? sl2 : 0ll);
      const long long num = 144 * Q - S * S;   // 144^2 var in Y'^2 units, exact
      tok[0] = sqrtf(static_cast<float>(num)) * (1.0f / (144.0f * static_cast<float>(kLumaScale)));
    }
    tok[1] = 1.f;
  }
}

// Feature tokens of every patch: a resident grid over the strips (as the density passes),
// a warp per patch.  DENSITY: the tokens are stored l2-normalised and their column sums added to
// `sums` in 2^-32 fixed point (each token exactly rounded, so the order does not matter): one atomic
// per coordinate and CTA into one of kPixSlots copies, which keeps the CTAs off each other's words.
constexpr int kPixSlots = 16;
constexpr int kPixCtasPerSm = 4;
template <bool DENSITY>
__global__ void __launch_bounds__(kApcThreads, kPixCtasPerSm) apc_pix_features(const uint8_t* __restrict__ img,
                                                                               const __grid_constant__ ApcTable t,
                                                                               int units, int feature,
                                                                               float* __restrict__ tokens,
                                                                               unsigned long long* __restrict__ sums,
                                                                               int* status) {
  constexpr int kWarps = kApcThreads / 32;
  __shared__ __align__(16) uint8_t s2[2][kStageBytes];
  __shared__ int hist[kWarps][48];
  __shared__ unsigned long long part[kWarps][kPixDim];
  __shared__ uint64_t bars[2];
  __shared__ StripRef ref[2];
  __shared__ int gave_up;
  // (for the tokens alone this is the call's first kernel, and its last)
  if (DENSITY) ptx::launch_dependents();
  else ptx::begin_call();
  const int2 range = unit_range(units);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long acc = 0ull;   // lane k < kPixDim: coordinate k
  StripPipe<1> pipe{s2, bars, ref, &gave_up, 0u};
  if (threadIdx.x == 0) pipe.init();
  __syncthreads();
  int first = range.x;
  for (int b = first < range.y ? find_image(t, first) : 0; first < range.y; ++b) {   // the CTA's strips of image b
    const int end = min(range.y, t.unit_prefix[b + 1]);
    if (warp == 0) pipe.begin(img, t, first, end);
    for (int unit = first; unit < end; ++unit, ++pipe.used) {
      pipe.wait(status, K_APC_PASS1);
      const StripRef cur = pipe.place();
      const uint8_t* s = pipe.data();
      if (unit > first && unit + 1 < end) {
        __syncthreads();   // everyone is done with the other buffer
        if (warp == 0) pipe.next(img, t, cur);
      }
      const int64_t p0 = cur.patch;
      for (int p = warp; p < cur.np; p += kWarps) {
        float tok[kPixDim];
        patch_feature([&](int y, int x) { return s + y * kStageRow + row_phase(cur, y) + (p * kPatch + x) * 3; }, feature,
                      hist[warp], tok);
        if (DENSITY) {
          float n2 = 0.f;
#pragma unroll
          for (int k = 0; k < kPixDim; ++k) n2 = fmaf(tok[k], tok[k], n2);
          const float iv = n2 > 0.f ? 1.0f / sqrtf(n2) : 0.f;
#pragma unroll
          for (int k = 0; k < kPixDim; ++k) tok[k] *= iv;
        }
        float v = tok[0];
#pragma unroll
        for (int k = 1; k < kPixDim; ++k)
          if (lane == k) v = tok[k];
        if (lane < kPixDim) {
          tokens[(p0 + p) * kPixDim + lane] = v;
          if (DENSITY) acc += fix32_signed(v);
        }
      }
    }
    if (DENSITY) {   // the image's sums
      if (lane < kPixDim) part[warp][lane] = acc;
      acc = 0ull;
      ptx::grid_dependency_wait();   // the zeroed sums
    }
    __syncthreads();
    if (DENSITY && threadIdx.x < kPixDim) {
      unsigned long long x = 0ull;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) x += part[w][threadIdx.x];
      atomicAdd(sums + (static_cast<int64_t>(t.b_base + b) * kPixSlots + blockIdx.x % kPixSlots) * kPixDim + threadIdx.x, x);
    }
    first = end;
    if (DENSITY && first < range.y) __syncthreads();   // `part` is rewritten
  }
}

// The density of the normalised tokens: a CTA takes kApcThreads tokens of one image, a thread per
// token.
struct PixTable {
  int tok0[kApcMaxB];
  int n[kApcMaxB];
  int ktail[kApcMaxB];
  int unit_prefix[kApcMaxB + 1];
  int nb;
  int b_base;
};

__device__ __forceinline__ int find_pix_image(const PixTable& t, int unit) {
  int b = 0;
  while (b + 1 < t.nb && t.unit_prefix[b + 1] <= unit) ++b;
  return b;
}

// Pass 2: c = sums / N, phi = |c|^2, c_hat = c / |c|, d_i = |t_hat_i - c_hat| (thread per token).
__global__ void __launch_bounds__(kApcThreads) apc_pix_pass2(const __grid_constant__ PixTable t,
                                                             const float* __restrict__ tokens,
                                                             const unsigned long long* __restrict__ sums,
                                                             float* __restrict__ d_out,
                                                             pace_apc_stats* __restrict__ stats,
                                                             TailWork* __restrict__ work) {
  __shared__ unsigned long long csum[kPixDim];
  ptx::launch_dependents();
  ptx::grid_dependency_wait();
  const int b = find_pix_image(t, blockIdx.x);
  const int u = blockIdx.x - t.unit_prefix[b];
  const int i = u * kApcThreads + threadIdx.x;
  const int N = t.n[b];
  const bool live = i < N;
  const float4* row = reinterpret_cast<const float4*>(tokens + (static_cast<int64_t>(t.tok0[b]) + (live ? i : 0)) * kPixDim);
  const float4 a = __ldcg(row), e = __ldcg(row + 1);
  if (threadIdx.x < kPixDim) {
    const unsigned long long* sb = sums + static_cast<int64_t>(t.b_base + b) * kPixSlots * kPixDim + threadIdx.x;
    unsigned long long x = 0ull;
#pragma unroll
    for (int k = 0; k < kPixSlots; ++k) x += __ldcg(sb + k * kPixDim);
    csum[threadIdx.x] = x;
  }
  __syncthreads();
  const float inv_n = 1.0f / static_cast<float>(N);
  float c[kPixDim];
  float phi = 0.f;
#pragma unroll
  for (int k = 0; k < kPixDim; ++k) {
    c[k] = unfix32<true>(csum[k], inv_n);
    phi = fmaf(c[k], c[k], phi);
  }
  const float inv_c = phi > 0.f ? 1.0f / sqrtf(phi) : 0.f;
  if (u == 0 && threadIdx.x == 0) {
    stats[t.b_base + b].phi = phi;
    stats[t.b_base + b].rho_g = 1.0f - phi;
    stats[t.b_base + b].n_patches = N;
    stats[t.b_base + b].k_tail = t.ktail[b];
  }
  const float v[kPixDim] = {a.x, a.y, a.z, a.w, e.x, e.y, e.z, e.w};
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < kPixDim; ++k) {
    const float x = v[k] - c[k] * inv_c;
    acc = fmaf(x, x, acc);
  }
  const float dv = sqrtf(acc);
  if (live) d_out[t.tok0[b] + i] = dv;
  tail_count_values(work + t.b_base + b, dv, live);
}

// ------------------------------------------------------------------------------------------------
// resample
// ------------------------------------------------------------------------------------------------
constexpr int kRsThreads = 128;  // threads of a resample CTA
constexpr int kRsTH = 4;         // output rows of a generic tile (kRsTH x kRsTW = kRsThreads)
constexpr int kRsTall = 8;       // and of a tall one
constexpr int kRsTW = 32;        // output columns of a generic tile
constexpr int kRsChunk = 8;      // input rows filtered per step of the generic path

struct ResampleTable {
  int64_t src_off[kApcMaxB];
  int64_t dst_off[kApcMaxB];
  int H[kApcMaxB];
  int W[kApcMaxB];
  int Ho[kApcMaxB];  // used when stats == nullptr
  int Wo[kApcMaxB];
  int nb;
  int b_base;
};

__device__ __forceinline__ float cubic_w(float t) {
  // Keys' cubic convolution, a = -0.5
  t = fabsf(t);
  const float inner = (1.5f * t - 2.5f) * t * t + 1.0f, outer = ((-0.5f * t + 2.5f) * t - 4.0f) * t + 2.0f;
  return t < 1.0f ? inner : t < 2.0f ? outer : 0.0f;
}

__device__ __forceinline__ int div_up(int a, int b) { return (a + b - 1) / b; }

// Window of output index o (reading R5) in exact integer arithmetic.  With s = n_in / n_out
// and fs = max(s, 1), the centre is c = (2o + 1) n_in / (2 n_out), the taps are
// lo .. lo + n - 1 with lo = max(0, floor(c - 2 fs)) and lo + n = min(n_in, ceil(c + 2 fs)),
// and tap i sits at (lo + i + 0.5 - c) / fs = (num0 + i * step) * inv_den with integer
// num0 = (2 lo + 1) n_out - (2o + 1) n_in, step = 2 n_out and den = 2 n_out fs.
struct Win {
  int lo, n, num0, step;
  float inv_den;
};
__device__ __forceinline__ Win exact_window(int o, int n_in, int n_out) {
  const bool down = n_in > n_out;
  const int64_t cn = (2 * static_cast<int64_t>(o) + 1) * n_in;                   // c * 2 n_out
  const int64_t sup = 4 * static_cast<int64_t>(down ? n_in : n_out);           // 2 fs * 2 n_out
  const int64_t d = 2 * static_cast<int64_t>(n_out);
  int64_t a = max(cn - sup, static_cast<int64_t>(0)), e = cn + sup + d - 1;
  if (e < (int64_t{1} << 32)) {   // a 32-bit division is several times cheaper
    a = static_cast<uint32_t>(a) / static_cast<uint32_t>(d);
    e = static_cast<uint32_t>(e) / static_cast<uint32_t>(d);
  } else {
    a /= d;
    e /= d;
  }
  if (e > n_in) e = n_in;
  Win w;
  w.lo = static_cast<int>(a);
  w.n = static_cast<int>(e - a);
  w.num0 = static_cast<int>((2 * a + 1) * n_out - cn);
  w.step = 2 * n_out;
  w.inv_den = 1.0f / static_cast<float>(down ? 2 * n_in : 2 * n_out);
  return w;
}

// Window [lo, lo + n) of taps for output index o, the tap offset of lo, its step, 1/sum(weights).
__device__ __forceinline__ void window_1d(int o, int n_in, int n_out, int& lo, int& n, float& off0, float& ifs,
                                          float& inorm) {
  const Win w = exact_window(o, n_in, n_out);
  lo = w.lo;
  n = w.n;
  off0 = static_cast<float>(w.num0) * w.inv_den;
  ifs = static_cast<float>(w.step) * w.inv_den;
  float s = 0.f;
  for (int i = 0; i < n; ++i) s += cubic_w(static_cast<float>(w.num0 + i * w.step) * w.inv_den);
  inorm = 1.0f / s;
}

// Steep downscales: one 4 x 32 or 8 x 32 output tile, weights evaluated per tap, input read through L1.
// It is bound by the horizontal pass, which works on (rows + 3) fs input rows per tile, so a call with
// tall tiles for three quarters of the grid takes those (8 images of 4K at 8.5 per side, 3840 tall tiles:
// 1000 us, in tiles of four rows 1214; one such image, 480: 150 and 165) and others have twice the tiles
// (one at 15 per side, 144: 224 us, in tall ones 326).  Not inlined: it needs none of the caller's values.
struct GenericSmem {
  int xlo[kRsTW], xn[kRsTW];
  float xoff[kRsTW], xifs[kRsTW], xnorm[kRsTW];
  int ylo[kRsTall], yn[kRsTall];
  float yoff[kRsTall], yifs[kRsTall], ynorm[kRsTall];
  float hbuf[kRsChunk][kRsTW][3];
};
template <int ROWS>
__device__ __noinline__ void resample_tile_generic(const uint8_t* __restrict__ img, int H, int W, int Ho, int Wo, int ox0,
                                                   int oy0, int nrows, uint8_t* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  GenericSmem& sh = *reinterpret_cast<GenericSmem*>(rs_smem);
  auto &xlo = sh.xlo, &xn = sh.xn;
  auto &xoff = sh.xoff, &xifs = sh.xifs, &xnorm = sh.xnorm;
  auto &ylo = sh.ylo, &yn = sh.yn;
  auto &yoff = sh.yoff, &yifs = sh.yifs, &ynorm = sh.ynorm;
  auto& hbuf = sh.hbuf;
  if (ox0 >= Wo || oy0 >= Ho) return;
  const int tid = threadIdx.x;
  if (tid < kRsTW) {
    const int ox = min(ox0 + tid, Wo - 1);
    window_1d(ox, W, Wo, xlo[tid], xn[tid], xoff[tid], xifs[tid], xnorm[tid]);
  } else if (tid >= 32 && tid < 32 + nrows) {
    const int i = tid - 32;
    const int oy = oy0 + i;
    window_1d(oy, H, Ho, ylo[i], yn[i], yoff[i], yifs[i], ynorm[i]);
  }
  __syncthreads();
  const int iy_lo = ylo[0];
  const int iy_hi = ylo[nrows - 1] + yn[nrows - 1];  // exclusive
  const int64_t pitch = static_cast<int64_t>(W) * 3;
  // this thread's output pixels: rows my_r and, of a tall tile, my_r + 4
  const int my_r = tid / kRsTW, my_c = tid % kRsTW;
  float acc[ROWS / kRsTH][3] = {};
  for (int r0 = iy_lo; r0 < iy_hi; r0 += kRsChunk) {
    // horizontal pass: kRsChunk rows x 32 columns x 3 channels
    for (int v = tid; v < kRsChunk * kRsTW * 3; v += kRsThreads) {
      const int rr = v / (kRsTW * 3), rem = v - rr * (kRsTW * 3);
      const int cc = rem / 3, ch = rem - cc * 3;
      const int iy = r0 + rr;
      float h = 0.f;
      if (iy < iy_hi) {
        const uint8_t* row = img + iy * pitch + ch;
        const int lo = xlo[cc], n = xn[cc];
        const float off = xoff[cc], ifs = xifs[cc];
        for (int i = 0; i < n; ++i) h = fmaf(cubic_w(fmaf(static_cast<float>(i), ifs, off)),
                                             static_cast<float>(__ldg(row + 3 * (lo + i))), h);
        h *= xnorm[cc];
      }
      hbuf[rr][cc][ch] = h;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < ROWS / kRsTH; ++q) {
      const int r = my_r + q * kRsTH;
      if (r >= nrows) break;
      const int lo = ylo[r], n = yn[r];
      const float off = yoff[r], ifs = yifs[r];
      for (int rr = 0; rr < kRsChunk; ++rr) {
        const int i = r0 + rr - lo;
        if (i >= 0 && i < n) {
          const float w = cubic_w(fmaf(static_cast<float>(i), ifs, off));
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) acc[q][ch] = fmaf(w, hbuf[rr][my_c][ch], acc[q][ch]);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < ROWS / kRsTH; ++q) {
    const int r = my_r + q * kRsTH, oy = oy0 + r, ox = ox0 + my_c;
    if (r < nrows && ox < Wo) {
      const float nrm = ynorm[r];
      uint8_t* o = out + (static_cast<int64_t>(oy) * Wo + ox) * 3;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) o[ch] = static_cast<uint8_t>(min(255, max(0, __float2int_rn(acc[q][ch] * nrm))));
    }
  }
  __syncthreads();   // shared tile buffers are reused by the next call
}

// Downscales of up to 8 per side: a tile of up to kVPx input columns, filtered vertically first.
//
// Bound by instructions and their latency, so every input byte is turned into a float once per tile and
// used from registers: a thread owns four pixels (12 bytes) of a column strip and walks down the input rows,
// adding each to the (at most) four output rows whose windows hold it; a finished pair of rows goes
// to shared memory as float2 (row, row + 1), and after four rows the CTA filters them horizontally,
// a thread per column, one packed FMA per tap, channel and two rows.  Input rows come through a
// per-thread ring of asynchronous copies (no barrier: a thread reads only what it
// copied itself).  At most four windows hold an input row because they are
// 4 fs wide and fs apart (fs = n_in / n_out >= 1), so four accumulators, reused in turn, are enough
// and the row loop needs no rotation once it is unrolled over four output rows.
// Byte-wise taps in the horizontal pass first (the reverse order) cost a shared load and a
// conversion for every tap of every input row: 4K at r = 0.248 took 57 us, now 30.0.
constexpr int kVThreads = 128;
constexpr int kVPx = 4 * kVThreads;          // input columns of a tile
constexpr int kVHalf = kVPx / 2 + 4;         // even (odd) columns of a plane, and slack for the last taps
constexpr int kVPlane = 2 * kVHalf;
constexpr int kVGroup = 4;                   // output rows per horizontal pass: two pairs
constexpr int kVMaxTH = 32;                  // output rows of a tile, at most
constexpr int kVMaxRows = 96;                // and input rows
constexpr int kVMaxScale = 8;
constexpr int kVWeights = 2560;              // horizontal weights of a tile
constexpr int kVMaxCols = kVPx;
constexpr int kVCtasPerSm = 4;
constexpr int kVWidths = 2;                  // tile widths: up to kVPx columns, or up to kVThreads
static_assert(kVPx >> 2 == kVThreads, "the narrow width");
// The input ring, taken two rows at a time: aligned rows are three words per thread, others four.
template <bool ALIGNED>
struct Ring {
  static constexpr int kWords = ALIGNED ? 3 : 4;
  static constexpr int kSlots = ALIGNED ? 8 : 4;
  static constexpr int kAhead = kSlots - 2;   // rows in flight
};
constexpr int kVRingWords = 24;              // words per thread of the larger ring
static_assert(Ring<true>::kWords * Ring<true>::kSlots <= kVRingWords && Ring<false>::kWords * Ring<false>::kSlots <= kVRingWords,
              "ring size");
struct ResampleSmem {
  float2 v[kVGroup / 2][3][kVPlane];         // filtered row pairs: channel planes, even columns then odd
  float2 wy[kVMaxRows][4];                   // (w, w) of input row y for output rows r .. r + 3, r the first unfinished
  uint32_t raw[kVRingWords][kVThreads];      // [row, word][thread] of the input ring
  float wx[kVWeights];                       // [tap][column]
  int xlo[kVMaxCols];
  int last[kVMaxTH];                         // last input row of output row r
  float ynorm[kVMaxTH];
};

// Four bytes as floats, exactly (2^23 + b by byte permutes, one packed subtract per pair).
__device__ __forceinline__ void word_to_floats(uint32_t v, float2& lo, float2& hi) {
  const float2 m = make_float2(-8388608.0f, -8388608.0f);
  lo = ptx::fadd2(make_float2(__uint_as_float(__byte_perm(v, 0x4B000000u, 0x7540)),
                              __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7541))),
                  m);
  hi = ptx::fadd2(make_float2(__uint_as_float(__byte_perm(v, 0x4B000000u, 0x7542)),
                              __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7543))),
                  m);
}

// Taps of every window of a downscale by s (a window has at most floor(4 s) + 2), made even.
__device__ __forceinline__ int tap_count(float s) { return (static_cast<int>(4.0f * s) + 3) & ~1; }

static_assert(sizeof(GenericSmem) <= sizeof(ResampleSmem), "one buffer for both kinds of tile");

// Tiles of a Ho x Wo output: columns per tile (its window, starting up to 3 pixels early, fits kVPx
// and its taps kVWeights; `limit` at most), spread evenly.
__device__ __forceinline__ int cols_per_tile(int W, int Wo, int limit) {
  const float s = static_cast<float>(W) / static_cast<float>(Wo);
  const int taps = tap_count(s);
  const int most = max(1, min(min(static_cast<int>((static_cast<float>(kVPx - 8) - 4.0f * s) / s), kVWeights / taps), limit));
  return div_up(Wo, div_up(Wo, most));
}

// Starts the copy of four pixels (12 bytes) at byte `off` of the image into a slot of the thread's
// ring; nothing past the image's last word is read (what lies there is never used).
template <bool ALIGNED>
__device__ __forceinline__ void fetch_px4(const uint8_t* __restrict__ img, uint32_t off, uint32_t last, uint32_t* slot) {
  const uint32_t a = ALIGNED ? off : off & ~3u;
#pragma unroll
  for (int k = 0; k < (ALIGNED ? 3 : 4); ++k) cp_async4(slot + k * kVThreads, img + min(a + 4u * k, last));
}

// The last of n_in inputs whose centre lies in the window of output index o.
__device__ __forceinline__ int last_input(int o, int n_in, int n_out) {
  const int64_t reach = (2 * static_cast<int64_t>(o) + 1) * n_in + 4 * static_cast<int64_t>(max(n_in, n_out)) - 1 - n_out;   // centre + 2 fs
  const int64_t d = 2 * static_cast<int64_t>(n_out);
  const int64_t i = reach < (int64_t{1} << 32) ? static_cast<int64_t>(static_cast<uint32_t>(reach) / static_cast<uint32_t>(d))
                                               : reach / d;
  return static_cast<int>(min(static_cast<int64_t>(n_in - 1), i));
}

template <bool ALIGNED>
__device__ __forceinline__ void resample_tile(ResampleSmem& sh, const uint8_t* __restrict__ img, int H, int W, int Ho,
                                              int Wo, int ox0, int ncol, int oy0, int nrow, uint8_t* __restrict__ out) {
  const int tid = threadIdx.x;
  const float sx = static_cast<float>(W) / static_cast<float>(Wo);
  const int taps = tap_count(sx);
  // the first input rows are requested before the weights are worked out
  const int x0 = exact_window(ox0, W, Wo).lo & ~3;
  const int y0 = exact_window(oy0, H, Ho).lo, y1 = last_input(oy0 + nrow - 1, H, Ho) + 1;
  const uint32_t pitch = static_cast<uint32_t>(W) * 3u;
  const uint32_t last_word = static_cast<uint32_t>(static_cast<int64_t>(H) * pitch - 4);
  const int px = x0 + 4 * tid;                     // this thread's four columns
  const bool works = px < exact_window(ox0 + ncol - 1, W, Wo).lo + taps; // some window may reach them
  uint32_t off = static_cast<uint32_t>(y0) * pitch + static_cast<uint32_t>(px) * 3u;   // of the next row to fetch
  const uint32_t shr = (off & 2u) * 8u, flip = ALIGNED ? 0u : (pitch & 2u) * 8u;        // alignment of a row, of the next
  uint32_t sft = ALIGNED ? 0u : shr;
  using R = Ring<ALIGNED>;
  uint32_t* ring = &sh.raw[0][tid];
  constexpr int kRow = R::kWords * kVThreads;   // words from slot to slot
  int y = y0, head = 0;   // the next row to filter, and its slot
  auto fetch_next = [&](int row, int slot) {    // one group of copies per row, empty past the tile's last
    if (works && row < y1) fetch_px4<ALIGNED>(img, off, last_word, ring + slot * kRow);
    cp_async_commit();
    off += pitch;
  };
#pragma unroll
  for (int k = 0; k < R::kAhead; ++k) fetch_next(y0 + k, k);
  // horizontal windows and normalised weights (reading R5), padded to an even number of taps
  for (int c = tid; c < ncol; c += kVThreads) {
    const Win w = exact_window(ox0 + c, W, Wo);
    sh.xlo[c] = w.lo;
    float sum = 0.f;
#pragma unroll 4
    for (int i = 0; i < taps; ++i) {
      const float x = i < w.n ? cubic_w(static_cast<float>(w.num0 + i * w.step) * w.inv_den) : 0.f;
      sh.wx[i * ncol + c] = x;
      sum += x;
    }
    const float inv = 1.0f / sum;
#pragma unroll 4
    for (int i = 0; i < taps; ++i) sh.wx[i * ncol + c] *= inv;
  }
  // vertical windows (by the threads that have fewest columns): the last input row whose centre lies
  // inside, 1 / sum of the weights
  const int vt = kVThreads - 1 - tid;
  if (vt < nrow) {
    const int o = oy0 + vt;
    const Win w = exact_window(o, H, Ho);
    float sum = 0.f;
#pragma unroll 4
    for (int i = 0; i < w.n; ++i) sum += cubic_w(static_cast<float>(w.num0 + i * w.step) * w.inv_den);
    sh.ynorm[vt] = 1.0f / sum;
    sh.last[vt] = last_input(o, H, Ho);
  }
  __syncthreads();
  const float inv_den = 1.0f / static_cast<float>(2 * max(H, Ho));
  for (int i = tid; i < (y1 - y0) * 4; i += kVThreads) {
    const int y = y0 + (i >> 2);
    int r = 0;
    for (int half = kVMaxTH / 2; half > 0; half >>= 1)   // first row that ends at y or later
      if (r + half <= nrow && sh.last[r + half - 1] < y) r += half;
    if (r < nrow && sh.last[r] < y) ++r;
    const int rr = r + (i & 3);
    float w = 0.f;
    if (rr < nrow) {
      const int64_t num = (2 * static_cast<int64_t>(y) + 1) * Ho - (2 * static_cast<int64_t>(oy0 + rr) + 1) * H;
      w = cubic_w(static_cast<float>(num) * inv_den) * sh.ynorm[rr];
    }
    sh.wy[y - y0][i & 3] = make_float2(w, w);
  }
  __syncthreads();
  float2 acc[4][6];                                // four output rows x 12 bytes
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int e = 0; e < 6; ++e) acc[j][e] = make_float2(0.f, 0.f);
  // filters the next NR input rows; acc[(PH + j) & 3] is output row r + j of the phase's row r
  auto rows = [&](auto phase, auto count) {
    constexpr int PH = decltype(phase)::value, NR = decltype(count)::value;
    cp_async_wait_group<R::kAhead - NR>();
    uint32_t w[NR][3];
    float4 wy[NR][2];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const uint32_t* slot = ring + ((head + i) & (R::kSlots - 1)) * kRow;
      uint32_t x[R::kWords];
#pragma unroll
      for (int k = 0; k < R::kWords; ++k) x[k] = slot[k * kVThreads];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if constexpr (ALIGNED) w[i][k] = x[k];
        else w[i][k] = __funnelshift_r(x[k], x[k + 1], sft);
      }
      sft ^= flip;
      const float4* wp = reinterpret_cast<const float4*>(sh.wy[y + i - y0]);
      wy[i][0] = wp[0];
      wy[i][1] = wp[1];
    }
#pragma unroll
    for (int i = 0; i < NR; ++i) fetch_next(y + R::kAhead + i, (head + R::kAhead + i) & (R::kSlots - 1));
    y += NR;
    head = (head + NR) & (R::kSlots - 1);
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      float2 f[6];
#pragma unroll
      for (int k = 0; k < 3; ++k) word_to_floats(w[i][k], f[2 * k], f[2 * k + 1]);
      const float2 wj[4] = {make_float2(wy[i][0].x, wy[i][0].y), make_float2(wy[i][0].z, wy[i][0].w),
                            make_float2(wy[i][1].x, wy[i][1].y), make_float2(wy[i][1].z, wy[i][1].w)};
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 6; ++e) acc[(PH + j) & 3][e] = ptx::ffma2(wj[j], f[e], acc[(PH + j) & 3][e]);
    }
  };
  // the input rows up to the last one of the phase's output row, two at a time
  auto advance = [&](auto phase, int upto) {
    while (y < upto) rows(phase, std::integral_constant<int, 2>{});
    if (y == upto) rows(phase, std::integral_constant<int, 1>{});
  };
  // byte 3 i + ch of the thread's 12 is channel ch of its pixel i
  auto byte_of = [](const float2 (&v)[6], int b) { return (b & 1) ? v[b >> 1].y : v[b >> 1].x; };
  for (int g = 0; g < nrow; g += kVGroup) {
    float2 held[6];
    auto finish = [&](auto phase) {
      constexpr int PH = decltype(phase)::value;
      advance(phase, g + PH < nrow ? sh.last[g + PH] : -1);
      if constexpr ((PH & 1) == 0) {
#pragma unroll
        for (int e = 0; e < 6; ++e) held[e] = acc[PH][e];
      } else if (works) {
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          float2* plane = sh.v[PH >> 1][ch];
#pragma unroll
          for (int odd = 0; odd < 2; ++odd)   // pixels odd and odd + 2
            *reinterpret_cast<float4*>(plane + odd * kVHalf + 2 * tid) =
                make_float4(byte_of(held, 3 * odd + ch), byte_of(acc[PH], 3 * odd + ch), byte_of(held, 3 * odd + 6 + ch),
                            byte_of(acc[PH], 3 * odd + 6 + ch));
        }
      }
#pragma unroll
      for (int e = 0; e < 6; ++e) acc[PH][e] = make_float2(0.f, 0.f);
    };
    finish(std::integral_constant<int, 0>{});
    finish(std::integral_constant<int, 1>{});
    finish(std::integral_constant<int, 2>{});
    finish(std::integral_constant<int, 3>{});
    __syncthreads();
    // horizontal pass of these four rows: a thread per column, all three channels
    for (int c = tid; c < ncol; c += kVThreads) {
      const int x = sh.xlo[c] - x0;
      const float2* even = sh.v[0][0] + (x & 1) * kVHalf + (x >> 1);           // taps 0, 2, ..
      const float2* odd = sh.v[0][0] + ((x + 1) & 1) * kVHalf + ((x + 1) >> 1);   // taps 1, 3, ..
      const float* w = sh.wx + c;
      float2 a[2][3];
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) a[p][ch] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int k = 0; k < taps; k += 2, w += 2 * ncol, ++even, ++odd) {
        const float2 w0 = make_float2(w[0], w[0]), w1 = make_float2(w[ncol], w[ncol]);
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) {
            a[p][ch] = ptx::ffma2(w0, even[(3 * p + ch) * kVPlane], a[p][ch]);
            a[p][ch] = ptx::ffma2(w1, odd[(3 * p + ch) * kVPlane], a[p][ch]);
          }
      }
      uint8_t* o = out + (static_cast<int64_t>(oy0 + g) * Wo + ox0 + c) * 3;
      auto put = [&](uint8_t* q, float v) { *q = static_cast<uint8_t>(ptx::round_u8(v)); };
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (g + r >= nrow) break;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) put(o + ch, (r & 1) ? a[r >> 1][ch].y : a[r >> 1][ch].x);
        o += static_cast<int64_t>(Wo) * 3;
      }
    }
    __syncthreads();   // the row pairs are rewritten
  }
}

// Small outputs, downscaled by up to 2.75 per side: an 8 x 32 tile whose input window is staged in shared
// memory, warp w filtering rows 2 w and 2 w + 1 vertically (a lane per four bytes) and then horizontally
// (a lane per column).  Such a call is all latency: the wide tiles above spend 9000 to 10000 cycles on a
// rating, windows and weights before their first row, these on four window edges at once and on one
// window per lane (one image of 448 x 448 at r = 0.25: 6.2 us, in wide tiles 10.2; at r = 0.8 7.2 and
// 10.3).  Every sum is taken in the same order with the same weights as there, so the bytes do not
// depend on which tiles a call gets.  A launch after other work fetches its instructions from memory, so
// this code comes first in the kernel, once for rows on any boundary, and its loops are not unrolled: behind a
// flush and other kernels such a call on 448 x 448 takes 10.3 us, 15.2 with the code behind that of the wide tiles,
// twice and unrolled by four, 14.1 in wide tiles; a call in wide tiles of 4K 34.7, as without this code (36.0
// with it twice).
constexpr int kSTH = 8, kSTW = 32;           // output rows and columns
constexpr int kSTaps = 14;                   // a window has at most floor(4 * 2.75) + 2 taps
constexpr int kSRows = 36;                   // 7 * 2.75 + 4 * 2.75 + 2 input rows, and two read with weight 0
constexpr int kSPx = 102;                    // 31 * 2.75 + 4 * 2.75 + 2 input columns, starting up to 3 early
constexpr int kSPitch = 336;                 // 15 bytes of alignment, 3 kSPx, in 16-byte pieces
constexpr int kSLine = 308;                  // 3 kSPx in fours
static_assert(4 * kSRows >= 4 * 2 + 11 * 7 + 11 * 4 + 8 && 4 * kSPx >= 11 * 31 + 11 * 4 + 8 + 12, "staged window");
static_assert(kSPitch >= (15 + 3 * kSPx + 3 + 15) / 16 * 16 && kSPitch % 16 == 0 && kSPitch <= 32 * 16 && kSLine >= 3 * kSPx,
              "staged row");
struct SmallSmem {
  uint8_t raw[kSRows][kSPitch];              // input rows, from the 16-byte boundary before the window
  float v[kSTH][kSLine];                     // vertically filtered rows
  float wx[kSTaps][kSTW];
  float wy[kSTH][kSTaps];
  int xlo[kSTW], xn[kSTW], ylo[kSTH], yn[kSTH];
};
static_assert(sizeof(SmallSmem) <= sizeof(ResampleSmem), "one buffer for every kind of tile");
__device__ __forceinline__ bool small_scale(int H, int W, int Ho, int Wo) { return 4 * H <= 11 * Ho && 4 * W <= 11 * Wo; }

__device__ __forceinline__ void resample_tile_small(SmallSmem& sh, const uint8_t* __restrict__ img, int H, int W, int Ho,
                                                    int Wo, int ox0, int oy0, uint8_t* __restrict__ out) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ncol = min(kSTW, Wo - ox0), nrow = min(kSTH, Ho - oy0);
  // the input window: lane 0 works out its left edge, lanes 1 to 3 the top, the right and the bottom one
  const bool rows = lane & 1, far = lane & 2;
  const Win e = exact_window(rows ? oy0 + (far ? nrow - 1 : 0) : ox0 + (far ? ncol - 1 : 0), rows ? H : W, rows ? Ho : Wo);
  const int edge = far ? e.lo + e.n : e.lo;
  const int x0 = __shfl_sync(0xffffffffu, edge, 0) & ~3, y0 = __shfl_sync(0xffffffffu, edge, 1);
  const int x1 = __shfl_sync(0xffffffffu, edge, 2), y1 = __shfl_sync(0xffffffffu, edge, 3);
  const uint32_t pitch = static_cast<uint32_t>(W) * 3u, bytes = static_cast<uint32_t>(H) * pitch;   // below 2^32
  const uint32_t first = static_cast<uint32_t>(y0) * pitch + static_cast<uint32_t>(x0) * 3u;
  const uint32_t span = static_cast<uint32_t>(x1 - x0) * 3u;
  for (int r = warp; r < y1 - y0; r += kVThreads / 32) {   // a warp per row, a lane per 16 bytes
    const uint32_t b = first + static_cast<uint32_t>(r) * pitch, a = (b & ~15u) + 16u * lane;
    if (a < b + span && a < bytes) cp_async16(sh.raw[r] + 16 * lane, img + a, min(16u, bytes - a));
  }
  cp_async_commit();
  // the windows' weights: columns by the first warp, rows by the second
  if (warp < 2 && lane < (warp == 0 ? ncol : nrow)) {
    const int o = warp == 0 ? ox0 + lane : oy0 + lane, n_in = warp == 0 ? W : H, n_out = warp == 0 ? Wo : Ho;
    const Win w = exact_window(o, n_in, n_out);
    float* to = warp == 0 ? &sh.wx[0][lane] : &sh.wy[lane][0];
    const int step = warp == 0 ? kSTW : 1, n = min(w.n, kSTaps);
    float sum = 0.f;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const float x = cubic_w(static_cast<float>(w.num0 + i * w.step) * w.inv_den);
      to[i * step] = x;
      sum += x;
    }
    const float inv = 1.0f / sum;
#pragma unroll 1
    for (int i = 0; i < n; ++i) to[i * step] *= inv;
    (warp == 0 ? sh.xlo : sh.ylo)[lane] = w.lo;
    (warp == 0 ? sh.xn : sh.yn)[lane] = warp == 0 ? n : min(n, last_input(o, n_in, n_out) - w.lo + 1);
  }
  cp_async_wait_group<0>();
  __syncthreads();
  const int ra = 2 * warp, rb = min(ra + 1, nrow - 1);
  if (ra < nrow) {
    const int la = sh.ylo[ra], na = sh.yn[ra], lb = sh.ylo[rb], nb = sh.yn[rb];
    for (int j = lane; 4 * j < static_cast<int>(span); j += 32) {
      float2 acc[2][2] = {};
      auto take = [&](int row, float w, float2 (&a)[2]) {   // one staged row into an output row
        const uint32_t ph = (first + static_cast<uint32_t>(row) * pitch) & 15u;
        const uint32_t* p = reinterpret_cast<const uint32_t*>(sh.raw[row] + (ph & 12u)) + j;
        const uint32_t word = __funnelshift_r(p[0], (ph & 2u) != 0u ? p[1] : 0u, (ph & 2u) * 8u);   // (warp-uniform)
        float2 lo, hi;
        word_to_floats(word, lo, hi);
        const float2 w2 = make_float2(w, w);
        a[0] = ptx::ffma2(w2, lo, a[0]);
        a[1] = ptx::ffma2(w2, hi, a[1]);
      };
#pragma unroll 1
      for (int i = 0; i < max(na, nb); ++i) {
        take(la - y0 + i, i < na ? sh.wy[ra][i] : 0.f, acc[0]);
        take(lb - y0 + i, i < nb ? sh.wy[rb][i] : 0.f, acc[1]);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4*>(&sh.v[ra + q][4 * j]) = make_float4(acc[q][0].x, acc[q][0].y, acc[q][1].x, acc[q][1].y);
    }
    __syncwarp();
    if (lane < ncol) {
      const float* va = &sh.v[ra][(sh.xlo[lane] - x0) * 3];
      const int n = sh.xn[lane];
      float acc[2][3] = {};
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        const float w = sh.wx[k][lane];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int ch = 0; ch < 3; ++ch) acc[q][ch] = fmaf(w, va[q * kSLine + 3 * k + ch], acc[q][ch]);
      }
      uint8_t* o = out + (static_cast<int64_t>(oy0 + ra) * Wo + ox0 + lane) * 3;
#pragma unroll
      for (int q = 0; q < 2; ++q, o += static_cast<int64_t>(Wo) * 3) {
        if (ra + q >= nrow) break;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) o[ch] = static_cast<uint8_t>(ptx::round_u8(acc[q][ch]));
      }
    }
  }
  __syncthreads();   // the shared buffers are reused by the next tile
}
// The small tiles of a batch: lane l of every warp holds images l and l + 32, their sizes and numbers of tiles.
__device__ __forceinline__ void resample_small(SmallSmem& sh, const uint8_t* __restrict__ src, const ResampleTable& t,
                                               uint8_t* __restrict__ dst, const int (&ho)[2], const int (&wo)[2],
                                               const uint32_t (&n)[2]) {
  const int lane = threadIdx.x & 31;
  uint32_t end0 = n[0], end1 = n[1];   // tiles up to the image's last one
  if (t.nb > 1) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up0 = __shfl_up_sync(0xffffffffu, end0, o), up1 = __shfl_up_sync(0xffffffffu, end1, o);
      if (lane >= o) {
        end0 += up0;
        end1 += up1;
      }
    }
    end1 += __shfl_sync(0xffffffffu, end0, 31);
  }
  const uint32_t total = t.nb > 1 ? __shfl_sync(0xffffffffu, end1, 31) : __shfl_sync(0xffffffffu, n[0], 0);
  for (uint32_t g = blockIdx.x; g < total; g += gridDim.x) {
    int b = 0;
    if (t.nb > 1) {
      b = __popc(__ballot_sync(0xffffffffu, end0 <= g));
      if (b == 32) b += __popc(__ballot_sync(0xffffffffu, end1 <= g));
    }
    const int Ho = __shfl_sync(0xffffffffu, b < 32 ? ho[0] : ho[1], b & 31);
    const int Wo = __shfl_sync(0xffffffffu, b < 32 ? wo[0] : wo[1], b & 31);
    const int l = static_cast<int>(g - __shfl_sync(0xffffffffu, b < 32 ? end0 - n[0] : end1 - n[1], b & 31));
    const int nx = (Wo + kSTW - 1) / kSTW, row = l / nx;
    const int H = t.H[b], W = t.W[b], ox0 = (l - row * nx) * kSTW, oy0 = row * kSTH;
    resample_tile_small(sh, src + t.src_off[b], H, W, Ho, Wo, ox0, oy0, dst + t.dst_off[b]);
  }
}
// Tiles x scale per CTA of the grid (a quarter more where rows start on 2-byte boundaries, which costs a
// second word per read) up to which a call takes small tiles.  Both kinds, in us: 2.9 rounds at 1 (672 x 672)
// 10.3 and 12.3, 2.1 at 1.6 (896 x 896, 3.3) 13.3 and 14.3, 3.2 at 1.3 (896 x 896, 4.1) 15.4 and 14.3, 2.1 at 2.4
// (1344 x 1344, 5.0) 18.2 and 16.4.
constexpr float kSmallWork = 3.8f;

// Wide and generic tiles of the batch, ho and wo as in resample_small.
__device__ __forceinline__ void resample_large(ResampleSmem& sh, const uint8_t* __restrict__ src, const ResampleTable& t,
                                               uint8_t* __restrict__ dst, const int (&ho)[2], const int (&wo)[2]) {
  __shared__ int tile_prefix[kApcMaxB + 1];
  __shared__ int sho[kApcMaxB], swo[kApcMaxB];
  __shared__ int stw[kVWidths][kApcMaxB];   // columns per tile (0: generic tiles), for each limit
  __shared__ int s_tw;                      // which limit
  __shared__ int swide[kVWidths][kApcMaxB]; // tiles per row of tiles, for each limit
  __shared__ int smost[kApcMaxB];           // rows per tile, at most
  __shared__ uint32_t srcp[kApcMaxB];       // the reciprocal of a quarter of that
  __shared__ int srows[kApcMaxB], snx[kApcMaxB];   // rows per tile, tiles per row of tiles
  const int tid = threadIdx.x;
  auto rcp = [](uint32_t m) { return 0xFFFFFFFFu / m + 1u; };   // 2^32 / m, rounded up (m > 1)
  static_assert(kVThreads == kVWidths * kApcMaxB, "a thread per image and width");
  if (const int b = tid & (kApcMaxB - 1), k = tid / kApcMaxB; b < t.nb) {
    const int Ho = b < 32 ? ho[0] : ho[1], Wo = b < 32 ? wo[0] : wo[1], H = t.H[b], W = t.W[b];
    const bool tiles = Ho > 0 && H <= kVMaxScale * Ho && W <= kVMaxScale * Wo;
    const int tw = tiles ? cols_per_tile(W, Wo, kVPx >> (2 * k)) : 0;
    stw[k][b] = tw;
    swide[k][b] = tw > 0 ? div_up(Wo, tw) : 0;
    // no more rows than the input rows that a tile can hold
    const int most = max(4, static_cast<int>(static_cast<float>(kVMaxRows - 4) * Ho / H - 3.0f) & ~3);
    if (k == 0) {
      sho[b] = Ho;
      swo[b] = Wo;
      smost[b] = most;
    } else {
      srcp[b] = rcp(static_cast<uint32_t>(min(most, kVMaxTH)) / 4u);
    }
  }
  __syncthreads();
  // Rows per tile, a multiple of four, and columns, as many as fit or at most a thread each: a tile reads
  // (rows + 4) fs input rows, so tall tiles filter least twice and wide ones share the set-up, but the
  // tiles should also fill the SMs.  Lane 8 k + l of warp 0 rates 4 (l + 1) rows in width k: a tile's time
  // is about rows + 4 + 3 (the set-up) times 3 + the columns per thread when it has an SM to itself, and
  // hardly more beside others as long as the SM holds them all: n tiles on an SM take about max(1, n / 4)
  // times that (rated at 0.4 n, one of 4K at r = 0.25 took three tall tiles per SM and 34.8 us, now four and
  // 30.0; rated at 0.2 n 33.5, with 8 images of 1344 x 1008 at r = 0.18 57.7 against 44.0).  More than four
  // narrow tiles are not considered (8 such images at r = 0.25: 39.5 us in wide tiles, 52.5 in five
  // narrow ones per SM; one of 448 x 448 at r = 0.8: 13.8 in wide ones, 9.7 in narrow ones).  What an image
  // adds to each rating costs no division: with two, one image after the other, 64 images of 224 x 224
  // at r = 0.25 took 38.9 us, 15 of them here, now 29.
  if (tid < 32) {
    const int th = 4 * ((tid & 7) + 1), k = min(tid >> 3, kVWidths - 1);
    static_assert(kVMaxTH == 32 && kVWidths == 2, "eight heights, two widths");
    auto rows_of = [&](int b, int rows) { return min(rows, smost[b]); };
    const uint32_t rcp_th = rcp(static_cast<uint32_t>(th) / 4u);
    uint32_t tiles = 0u, turns = 1u;   // (an image has fewer than 2^30 pixels)
#pragma unroll 4
    for (int b = 0; b < t.nb; ++b) {
      const uint32_t m = static_cast<uint32_t>(rows_of(b, th)) / 4u, q = static_cast<uint32_t>(sho[b] + 3) / 4u + m - 1u;
      // ceil(Ho / 4 m) with 1 <= m <= 8, exact below 2^29
      tiles += static_cast<uint32_t>(swide[k][b]) * (m == 1u ? q : __umulhi(q, th <= smost[b] ? rcp_th : srcp[b]));
      turns = max(turns, static_cast<uint32_t>(stw[k][b] + kVThreads - 1) / kVThreads);
    }
    const uint32_t sms = gridDim.x / kVCtasPerSm, per_sm = min(1u << 16, (tiles + sms - 1u) / sms);
    const uint32_t load = k == 0 ? max(10u, (5u * per_sm + 1u) / 2u) : per_sm <= 3u ? 10u : 11u;
    const uint32_t cost = k > 0 && per_sm > 4u ? 0xFFFFFFFFu : (3u + turns) * load * static_cast<uint32_t>(th + 7);
    const unsigned best = __reduce_min_sync(0xffffffffu, cost);
    const int who = __ffs(__ballot_sync(0xffffffffu, cost == best)) - 1;
    const int best_th = 4 * ((who & 7) + 1), best_k = min(who >> 3, kVWidths - 1);
    if (tid == 0) s_tw = best_k;
    // images in generic tiles: rows by the tall tiles that the call has
    uint32_t tall = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (const int b = tid + 32 * h; b < t.nb && stw[0][b] == 0)
        tall += min(1u << 20, static_cast<uint32_t>(swo[b] + kRsTW - 1) / kRsTW * (static_cast<uint32_t>(sho[b] + kRsTall - 1) / kRsTall));
    const int generic_rows = __reduce_add_sync(0xffffffffu, tall) >= gridDim.x / 4u * 3u ? kRsTall : kRsTH;
    // the images' first tiles, lane l taking images l and l + 32 (one thread after the other took 2 us of a
    // batch of 16)
    int n[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int b = tid + 32 * h;
      n[h] = 0;
      if (b < t.nb) {
        const int tw = stw[best_k][b];
        srows[b] = tw > 0 ? rows_of(b, best_th) : generic_rows;
        snx[b] = tw > 0 ? swide[best_k][b] : div_up(swo[b], kRsTW);
        n[h] = div_up(sho[b], srows[b]) * snx[b];
      }
    }
    int incl[2] = {n[0], n[1]};
    if (t.nb > 1) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int up = __shfl_up_sync(0xffffffffu, incl[h], o);
          if (tid >= o) incl[h] += up;
        }
    } else {
      incl[0] = __shfl_sync(0xffffffffu, n[0], 0);
    }
    const int half = __shfl_sync(0xffffffffu, incl[0], 31);
    tile_prefix[tid] = incl[0] - n[0];
    tile_prefix[tid + 32] = half + incl[1] - n[1];
    if (tid == 31) tile_prefix[kApcMaxB] = half + incl[1];
  }
  __syncthreads();
  const int* cols = stw[s_tw];
  const int total = tile_prefix[t.nb];
  for (int g = blockIdx.x; g < total; g += gridDim.x) {
    int b = 0;   // the last image whose first tile is g or before
#pragma unroll
    for (int step = kApcMaxB / 2; step > 0; step >>= 1)
      if (b + step < t.nb && tile_prefix[b + step] <= g) b += step;
    const int Ho = sho[b], Wo = swo[b], H = t.H[b], W = t.W[b];
    const int th = srows[b], tw = cols[b] > 0 ? cols[b] : kRsTW, nx = snx[b];
    const int l = g - tile_prefix[b];
    const int row = l / nx;
    const int oy0 = row * th, ox0 = (l - row * nx) * tw;
    const uint8_t* img = src + t.src_off[b];
    uint8_t* out = dst + t.dst_off[b];
    if (cols[b] > 0) {
      const int ncol = min(tw, Wo - ox0), nrow = min(th, Ho - oy0);
      if (W % 4 == 0) resample_tile<true>(sh, img, H, W, Ho, Wo, ox0, ncol, oy0, nrow, out);
      else resample_tile<false>(sh, img, H, W, Ho, Wo, ox0, ncol, oy0, nrow, out);
    } else {
      const int nrow = min(th, Ho - oy0);
      if (th == kRsTall) resample_tile_generic<kRsTall>(img, H, W, Ho, Wo, ox0, oy0, nrow, out);
      else resample_tile_generic<kRsTH>(img, H, W, Ho, Wo, ox0, oy0, nrow, out);
    }
  }
}

// Every CTA walks the output tiles of the whole batch (target sizes read from the density statistics
// on the device, or given), so the grid never holds empty CTAs.
__global__ void __launch_bounds__(kVThreads, kVCtasPerSm) apc_resample(const uint8_t* __restrict__ src,
                                                                       const __grid_constant__ ResampleTable t,
                                                                       const pace_apc_stats* __restrict__ stats,
                                                                       uint8_t* __restrict__ dst) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  ptx::begin_call();
  const int lane = threadIdx.x & 31;
  auto size_of = [&](int b, int& Ho, int& Wo) {
    Ho = stats ? __ldcg(&stats[t.b_base + b].h_out) : t.Ho[b];
    Wo = stats ? __ldcg(&stats[t.b_base + b].w_out) : t.Wo[b];
    if (Ho < 1 || Wo < 1 || Ho > t.H[b] || Wo > t.W[b]) Ho = Wo = 0;   // nothing to write
  };
  // every warp: lane l holds images l and l + 32, their sizes and their small tiles (and the work of these,
  // too much to count where an image can't have them); of a batch the first warp works them out, since the
  // lanes read the table one after the other (64 images of 224 x 224: by every warp 3 us more)
  static_assert(kApcMaxB == 64, "two images per lane");
  constexpr float kNoSmall = static_cast<float>(1 << 20);
  __shared__ int s_ho[kApcMaxB], s_wo[kApcMaxB];
  __shared__ uint32_t s_small[kApcMaxB], s_work;
  int ho[2] = {}, wo[2] = {};
  uint32_t small_n[2] = {}, total_work = 0u;
  if (t.nb == 1 || threadIdx.x < 32) {
    float work = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int b = lane + 32 * h;
      if (b >= t.nb) continue;
      size_of(b, ho[h], wo[h]);
      if (ho[h] == 0) continue;
      const int H = t.H[b], W = t.W[b];
      small_n[h] = static_cast<uint32_t>(wo[h] + kSTW - 1) / kSTW * (static_cast<uint32_t>(ho[h] + kSTH - 1) / kSTH);
      const float scale = fmaxf(__fdividef(static_cast<float>(W), static_cast<float>(wo[h])),
                                __fdividef(static_cast<float>(H), static_cast<float>(ho[h])));
      work += small_scale(H, W, ho[h], wo[h])
                  ? fminf(kNoSmall, static_cast<float>(small_n[h]) * scale * (W % 4 == 0 ? 1.0f : 1.25f)) : kNoSmall;
    }
    total_work = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(work));
  }
  if (t.nb > 1) {
    if (threadIdx.x < 32) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        s_ho[lane + 32 * h] = ho[h];
        s_wo[lane + 32 * h] = wo[h];
        s_small[lane + 32 * h] = small_n[h];
      }
      if (lane == 0) s_work = total_work;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ho[h] = s_ho[lane + 32 * h];
      wo[h] = s_wo[lane + 32 * h];
      small_n[h] = s_small[lane + 32 * h];
    }
    total_work = s_work;
  }
  if (static_cast<float>(total_work) <= kSmallWork * static_cast<float>(gridDim.x)) {   // (this code first: see there)
    resample_small(*reinterpret_cast<SmallSmem*>(rs_smem), src, t, dst, ho, wo, small_n);
    return;
  }
  resample_large(*reinterpret_cast<ResampleSmem*>(rs_smem), src, t, dst, ho, wo);
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
struct DensityLayout {
  size_t sums_off, work_off, zero_bytes, sumsq_off, d_off, total;   // [0, zero_bytes) is zeroed per call
  int64_t n_total;
};

DensityLayout density_layout(int B, const int32_t* H, const int32_t* W) {
  DensityLayout L{};
  int64_t n = 0;
  for (int b = 0; b < B; ++b) n += static_cast<int64_t>(H[b] / kPatch) * (W[b] / kPatch);
  L.n_total = n;
  L.sums_off = 0;
  L.work_off = align_up(static_cast<size_t>(B) * kSumSlots * kTokDim * sizeof(unsigned long long), 256);
  L.zero_bytes = L.work_off + static_cast<size_t>(B) * sizeof(TailWork);
  L.sumsq_off = align_up(L.zero_bytes, 256);
  L.d_off = L.sumsq_off + align_up(static_cast<size_t>(n) * sizeof(float), 256);
  L.total = L.d_off + align_up(static_cast<size_t>(n) * sizeof(float), 256);
  return L;
}

// Launches apc_tail on one ApcTable: a cluster of CTAs per image, one CTA when every image's
// distances fit its first loads.
pace_status_t launch_tail(const ApcTable& t, const float* d, TailParams tp, pace_apc_stats* stats, TailWork* work,
                          cudaStream_t stream) {
  int most = 0;
  for (int i = 0; i < t.nb; ++i) most = std::max(most, t.n[i]);
  const unsigned ctas = most <= kTailAhead * 1024 ? 1u : kTailCluster;
  return launch_dependent(apc_tail, dim3(ctas, static_cast<unsigned>(t.nb)), 1024, 0, ctas, stream, t, d, tp, stats,
                          static_cast<const TailWork*>(work));
}

pace_status_t launch_zero(void* a, size_t a_bytes, void* b, size_t b_bytes, cudaStream_t stream) {
  const size_t na = a_bytes / 16, nb = b_bytes / 16;
  return launch_dependent(apc_zero, static_cast<unsigned>(std::min<size_t>((na + nb + 1023) / 1024, 2048)), 256, 0, 1, stream,
                          static_cast<uint4*>(a), static_cast<unsigned>(na), static_cast<uint4*>(b), static_cast<unsigned>(nb));
}

// Strip table of images c0 .. c0 + nb - 1; patch0 runs on over the calls.  The strips have the largest
// width of which the table has at least `enough` (else the smallest): a small call is all latency
// (448 x 448: 32 strips of 32 patches, 128 of 8), a large one all issue, and wide strips spend
// least of it on barriers.  With the width chosen per image, 16 images of 672 x 672 took 48.9 us in
// strips of 8, now 32.8; the line at a strip per SM, not two, 8 images of 448 x 448 16.4 against 22.5
// and one of 896 x 896 16.4 against 18.4.  The sums are exact, so the width moves no result.
void fill_strip_table(ApcTable& t, int c0, int nb, const int64_t* img_off, const int32_t* H, const int32_t* W,
                      float tail_frac, int enough, int& patch0) {
  t = ApcTable{};
  t.nb = nb;
  t.b_base = c0;
  t.unit_prefix[0] = 0;
  int lg = kStripLog2 + 1;
  for (int64_t strips = 0; lg > kMinStripLog2 && strips < enough;) {
    --lg;
    strips = 0;
    for (int b = c0; b < c0 + nb; ++b) strips += static_cast<int64_t>((W[b] / kPatch + (1 << lg) - 1) >> lg) * (H[b] / kPatch);
  }
  for (int i = 0; i < nb; ++i) {
    const int b = c0 + i;
    t.off[i] = img_off[b];
    t.H[i] = H[b];
    t.W[i] = W[b];
    t.gw[i] = W[b] / kPatch;
    t.strip_log2[i] = lg;
    t.chunks[i] = (t.gw[i] + (1 << lg) - 1) >> lg;
    t.patch0[i] = patch0;
    const int N = (H[b] / kPatch) * t.gw[i];
    t.n[i] = N;
    const double scale = 2.0 / (255.0 * N);
    t.col_scale[i].x = static_cast<float>(scale);
    t.col_scale[i].y = static_cast<float>(scale - static_cast<double>(t.col_scale[i].x));
    double kt = std::floor(static_cast<double>(tail_frac) * N + 0.5);
    if (kt < 1) kt = 1;
    if (kt > N) kt = N;
    t.ktail[i] = static_cast<int>(kt);
    patch0 += N;
    t.unit_prefix[i + 1] = t.unit_prefix[i] + (H[b] / kPatch) * t.chunks[i];
  }
}

// Whether every image row of the table starts on a 4-byte boundary (an even number of patches wide).
bool rows_aligned(const ApcTable& t) {
  bool all = true;
  for (int i = 0; i < t.nb; ++i) all = all && t.gw[i] % 2 == 0;
  return all;
}

pace_status_t check_params(const pace_apc_params* params, pace_apc_params& p) {
  if (params) p = *params;
  else pace_apc_params_default(&p);
  if (!(p.tail_frac > 0.f && p.tail_frac <= 1.f) || !(p.gamma > 0.f) || !(p.alpha >= 0.f && p.alpha <= 1.f) ||
      !(p.r_min <= p.r_max) || p.align < 1)
    return PACE_ERR_INVALID_ARG;
  return PACE_OK;
}

// The three density kernels, after the kernel that zeroes their sums and tail scratch.
pace_status_t run_density(const uint8_t* img, const int64_t* img_off, const int32_t* H, const int32_t* W, int B,
                          const pace_apc_params& p, float* d, pace_apc_stats* stats, unsigned long long* sums,
                          TailWork* work, uint32_t* sumsq, cudaStream_t stream) {
  int sms = 0, dev = 0;
  PACE_CHECK(sm_count(&sms));
  PACE_CUDA(cudaGetDevice(&dev));
  static DeviceOnce once;   // opt in to the passes' shared memory
  if (!once.done(dev)) {
    for (auto* k : {apc_pass1<true>, apc_pass1<false>})
      PACE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kDGroups * sizeof(Pass1Group)));
    for (auto* k : {apc_pass2<true>, apc_pass2<false>})
      PACE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(Pass2Smem)));
    once.mark(dev);
  }
  int* status = device_status_word();
  int patch0 = 0;
  for (int c0 = 0; c0 < B; c0 += kApcMaxB) {
    const int nb = std::min(kApcMaxB, B - c0);
    ApcTable t;
    fill_strip_table(t, c0, nb, img_off, H, W, p.tail_frac, sms, patch0);
    const int units = t.unit_prefix[nb];
    const unsigned grid = static_cast<unsigned>(std::min(units, sms));
    const dim3 block(kDThreads, kDGroups);
    const bool aligned = rows_aligned(t);
    PACE_CHECK(launch_dependent(aligned ? apc_pass1<true> : apc_pass1<false>, grid, block, kDGroups * sizeof(Pass1Group), 1,
                                stream, img, t, units, sumsq, sums, status));
    PACE_CHECK(launch_dependent(aligned ? apc_pass2<true> : apc_pass2<false>, grid, block, sizeof(Pass2Smem), 1, stream, img,
                                t, units, static_cast<const uint32_t*>(sumsq), static_cast<const unsigned long long*>(sums), d,
                                stats, work, status));
    const TailParams tp{p.alpha, p.gamma, p.r_min, p.r_max, p.align};
    PACE_CHECK(launch_tail(t, d, tp, stats, work, stream));
  }
  return PACE_OK;
}

pace_status_t check_images(const uint8_t* img, const int64_t* off, const int32_t* H, const int32_t* W, int B) {
  if (B < 0) return PACE_ERR_INVALID_ARG;
  if (B == 0) return PACE_OK;
  if (img == nullptr || off == nullptr || H == nullptr || W == nullptr) return PACE_ERR_INVALID_ARG;
  for (int b = 0; b < B; ++b) {
    if (H[b] < kPatch || W[b] < kPatch || H[b] % kPatch || W[b] % kPatch) return PACE_ERR_INVALID_ARG;
    if (off[b] < 0 || (reinterpret_cast<uintptr_t>(img) + off[b]) % 16) return PACE_ERR_INVALID_ARG;
    if (static_cast<int64_t>(H[b]) * W[b] > (int64_t{1} << 30)) return PACE_ERR_INVALID_ARG;
  }
  return PACE_OK;
}

}  // namespace

pace_status_t launch_strip_selftest(int* status, cudaStream_t stream) {
  strip_selftest<<<1, 64, 0, stream>>>(status);
  return check_launch();
}
}  // namespace pace

using namespace pace;

extern "C" size_t pace_apc_density_workspace_size(int B, const int32_t* H, const int32_t* W) {
  if (B <= 0 || H == nullptr || W == nullptr) return 0;
  for (int b = 0; b < B; ++b)
    if (H[b] < kPatch || W[b] < kPatch) return 0;
  return density_layout(B, H, W).total;
}

extern "C" pace_status_t pace_apc_density(const uint8_t* img, const int64_t* img_off, const int32_t* H,
                                          const int32_t* W, int B, const pace_apc_params* params, float* d_out,
                                          pace_apc_stats* stats, void* ws, size_t ws_bytes,
                                          pace_stream_t stream) {
  PACE_CHECK(check_images(img, img_off, H, W, B));
  if (B == 0) return PACE_OK;
  if (stats == nullptr) return PACE_ERR_INVALID_ARG;
  pace_apc_params p;
  PACE_CHECK(check_params(params, p));
  const DensityLayout L = density_layout(B, H, W);
  if (ws == nullptr || ws_bytes < L.total || reinterpret_cast<uintptr_t>(ws) % 16) return PACE_ERR_WORKSPACE;
  PACE_CHECK(check_device());
  uint8_t* w8 = static_cast<uint8_t*>(ws);
  float* d = d_out ? d_out : reinterpret_cast<float*>(w8 + L.d_off);
  PACE_CHECK(launch_zero(w8, L.zero_bytes, nullptr, 0, stream));   // column sums and tail scratch
  return run_density(img, img_off, H, W, B, p, d, stats, reinterpret_cast<unsigned long long*>(w8 + L.sums_off),
                     reinterpret_cast<TailWork*>(w8 + L.work_off), reinterpret_cast<uint32_t*>(w8 + L.sumsq_off), stream);
}

static pace_status_t resample_impl(const uint8_t* src, const int64_t* src_off, const int32_t* H, const int32_t* W,
                                   const int32_t* Ho, const int32_t* Wo, const pace_apc_stats* stats,
                                   uint8_t* dst, const int64_t* dst_off, int B, pace_stream_t stream) {
  PACE_CHECK(check_images(src, src_off, H, W, B));
  if (B == 0) return PACE_OK;
  if (dst == nullptr || dst_off == nullptr) return PACE_ERR_INVALID_ARG;
  if (stats == nullptr) {
    if (Ho == nullptr || Wo == nullptr) return PACE_ERR_INVALID_ARG;
    for (int b = 0; b < B; ++b)
      if (Ho[b] < 1 || Wo[b] < 1 || Ho[b] > H[b] || Wo[b] > W[b]) return PACE_ERR_INVALID_ARG;
  }
  for (int b = 0; b < B; ++b)
    if (dst_off[b] < 0) return PACE_ERR_INVALID_ARG;
  PACE_CHECK(check_device());
  int sms = 0, dev = 0;
  PACE_CHECK(sm_count(&sms));
  PACE_CUDA(cudaGetDevice(&dev));
  static DeviceOnce once;   // opt in to the tiles' shared memory
  if (!once.done(dev)) {
    PACE_CUDA(cudaFuncSetAttribute(apc_resample, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(ResampleSmem)));
    once.mark(dev);
  }
  for (int c0 = 0; c0 < B; c0 += kApcMaxB) {
    const int nb = (B - c0) < kApcMaxB ? (B - c0) : kApcMaxB;
    ResampleTable t{};
    t.nb = nb;
    t.b_base = c0;
    for (int i = 0; i < nb; ++i) {
      const int b = c0 + i;
      t.src_off[i] = src_off[b];
      t.dst_off[i] = dst_off[b];
      t.H[i] = H[b];
      t.W[i] = W[b];
      t.Ho[i] = stats ? H[b] : Ho[b];
      t.Wo[i] = stats ? W[b] : Wo[b];
    }
    PACE_CHECK(launch_dependent(apc_resample, static_cast<unsigned>(kVCtasPerSm * sms), kVThreads, sizeof(ResampleSmem), 1,
                                stream, src, t, stats, dst));
  }
  return PACE_OK;
}

extern "C" pace_status_t pace_apc_resample(const uint8_t* src, const int64_t* src_off, const int32_t* H,
                                           const int32_t* W, const pace_apc_stats* stats, uint8_t* dst,
                                           const int64_t* dst_off, int B, pace_stream_t stream) {
  if (B > 0 && stats == nullptr) return PACE_ERR_INVALID_ARG;
  return resample_impl(src, src_off, H, W, nullptr, nullptr, stats, dst, dst_off, B, stream);
}

extern "C" pace_status_t pace_apc_resample_to(const uint8_t* src, const int64_t* src_off, const int32_t* H,
                                              const int32_t* W, const int32_t* H_out, const int32_t* W_out,
                                              uint8_t* dst, const int64_t* dst_off, int B, pace_stream_t stream) {
  return resample_impl(src, src_off, H, W, H_out, W_out, nullptr, dst, dst_off, B, stream);
}

// ------------------------------------------------------------------------------------------------
// pace_apc_density_static: the same density computation with library-owned scratch
// ------------------------------------------------------------------------------------------------
// Scratch of pace_apc_density_static, in a file-scope device array instead of caller memory:
// the per-image 589-entry fixed-point column sums (kSumSlots copies), the tail's buckets, then |x|^2 per patch.
// Every GPU that loads the library holds this array until the process exits.
namespace pace {
namespace {
constexpr size_t kStaticSumsBytes =
    static_cast<size_t>(PACE_APC_STATIC_MAX_IMAGES) * kSumSlots * kTokDim * sizeof(unsigned long long);
constexpr size_t kStaticWorkOff = (kStaticSumsBytes + 255) / 256 * 256;
constexpr size_t kStaticZeroBytes = kStaticWorkOff + static_cast<size_t>(PACE_APC_STATIC_MAX_IMAGES) * sizeof(TailWork);
constexpr size_t kStaticSumsqOff = (kStaticZeroBytes + 255) / 256 * 256;
constexpr size_t kStaticBytes = kStaticSumsqOff + static_cast<size_t>(PACE_APC_STATIC_MAX_PATCHES) * sizeof(uint32_t);

static __device__ __align__(256) unsigned char g_apc_static_scratch[kStaticBytes];

std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};
DeviceOnce g_static_once;

// Device address of the array for the current device.  The name g_apc_static_scratch in host
// code is only a host-side handle, so the address is looked up once per device and set-up
// generation (pace_init starts a new one, e.g. after cudaDeviceReset).
pace_status_t static_scratch(unsigned char** out) {
  int dev = -1;
  PACE_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return PACE_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(g_static_mutex);
  if (!g_static_once.done(dev)) {
    void* p = nullptr;
    PACE_CUDA(cudaGetSymbolAddress(&p, g_apc_static_scratch));
    if (p == nullptr) return set_cuda_error(cudaErrorInvalidSymbol);
    g_static_ptr[dev] = p;
    g_static_once.mark(dev);
  }
  *out = static_cast<unsigned char*>(g_static_ptr[dev]);
  return PACE_OK;
}
}  // namespace
}  // namespace pace

extern "C" pace_status_t pace_apc_density_static(const uint8_t* img, const int64_t* img_off, const int32_t* H,
                                                 const int32_t* W, int B, const pace_apc_params* params,
                                                 float* d_out, pace_apc_stats* stats, pace_stream_t stream) {
  PACE_CHECK(check_images(img, img_off, H, W, B));
  if (B == 0) return PACE_OK;
  if (stats == nullptr || d_out == nullptr) return PACE_ERR_INVALID_ARG;
  if (B > PACE_APC_STATIC_MAX_IMAGES) return PACE_ERR_INVALID_ARG;
  int64_t n_total = 0;
  for (int b = 0; b < B; ++b) n_total += static_cast<int64_t>(H[b] / kPatch) * (W[b] / kPatch);
  if (n_total > PACE_APC_STATIC_MAX_PATCHES) return PACE_ERR_INVALID_ARG;
  pace_apc_params p;
  PACE_CHECK(check_params(params, p));
  PACE_CHECK(check_device());
  unsigned char* scratch = nullptr;
  PACE_CHECK(static_scratch(&scratch));
  auto* sums = reinterpret_cast<unsigned long long*>(scratch);
  auto* work = reinterpret_cast<TailWork*>(scratch + kStaticWorkOff);
  // the array keeps the previous call's contents: the column sums and the tail scratch of the
  // call's images must start from zero
  PACE_CHECK(launch_zero(sums, static_cast<size_t>(B) * kSumSlots * kTokDim * sizeof(unsigned long long), work,
                         static_cast<size_t>(B) * sizeof(TailWork), stream));
  return run_density(img, img_off, H, W, B, p, d_out, stats, sums, work,
                     reinterpret_cast<uint32_t*>(scratch + kStaticSumsqOff), stream);
}

// ------------------------------------------------------------------------------------------------
// pace_apc_density_tokens: Eq. 1-6 on preview tokens
// ------------------------------------------------------------------------------------------------
namespace pace {
namespace {
// Opts pass 1 of the token density into two 40 KB stages (once per device).
pace_status_t tok_pass1_attr() {
  static DeviceOnce once;
  int dev = 0;
  PACE_CUDA(cudaGetDevice(&dev));
  if (once.done(dev)) return PACE_OK;
  PACE_CUDA(cudaFuncSetAttribute(apc_tok_pass1, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kTok1StageBytes));
  once.mark(dev);
  return PACE_OK;
}

// Grid of pass 1: the CTAs resident at once (capped by the chunks).
unsigned tok_pass1_grid(int units) {
  static std::atomic<int> cap[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  int c = cap[dev & 63].load(std::memory_order_relaxed);
  if (c == 0) {
    int nsm = 0, per = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apc_tok_pass1, kApcThreads, 2 * kTok1StageBytes);
    c = std::max(1, nsm * std::max(per, 1));
    cap[dev & 63].store(c, std::memory_order_relaxed);
  }
  return static_cast<unsigned>(std::max(1, std::min(units, c)));
}

// The two register kernels for V 16-byte vectors per lane.
template <int V>
pace_status_t launch_tok_vec_n(const uint4* T, const TokTable& t, unsigned grid, float* d, pace_apc_stats* stats, float* inv,
                               unsigned long long* sums, TailWork* work, cudaStream_t stream) {
  constexpr size_t kWarps = kTokThreads / 32;
  int dev = 0;
  PACE_CUDA(cudaGetDevice(&dev));
  static DeviceOnce once;
  if (!once.done(dev)) {
    PACE_CUDA(cudaFuncSetAttribute(apc_tok_vec1<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(kWarps * V * 256 * sizeof(unsigned long long))));
    once.mark(dev);
  }
  PACE_CHECK(launch_dependent(apc_tok_vec1<V>, grid, kTokThreads, kWarps * V * 256 * sizeof(unsigned long long), 1, stream, T,
                              t, inv, sums));
  return launch_dependent(apc_tok_vec2<V>, 2 * grid, kApcThreads, 0, 1, stream, T, t, static_cast<const float*>(inv),
                          static_cast<const unsigned long long*>(sums), d, stats, work);
}

pace_status_t launch_tok_vec(const void* T, const TokTable& t, int64_t tokens, float* d, pace_apc_stats* stats, float* inv,
                             unsigned long long* sums, TailWork* work, cudaStream_t stream) {
  int sms = 0;
  PACE_CHECK(sm_count(&sms));
  const unsigned grid = static_cast<unsigned>(std::min<int64_t>(sms, (tokens + 7) / 8));
  const uint4* T4 = static_cast<const uint4*>(T);
  switch ((t.D + 255) / 256) {
    case 1: return launch_tok_vec_n<1>(T4, t, grid, d, stats, inv, sums, work, stream);
    case 2: return launch_tok_vec_n<2>(T4, t, grid, d, stats, inv, sums, work, stream);
    case 3: return launch_tok_vec_n<3>(T4, t, grid, d, stats, inv, sums, work, stream);
    case 4: return launch_tok_vec_n<4>(T4, t, grid, d, stats, inv, sums, work, stream);
    case 5: return launch_tok_vec_n<5>(T4, t, grid, d, stats, inv, sums, work, stream);
    default: return launch_tok_vec_n<6>(T4, t, grid, d, stats, inv, sums, work, stream);
  }
}

struct TokLayout {
  size_t sums_off, work_off, zero_bytes, inv_off, total;   // [0, zero_bytes) is zeroed per call
};
TokLayout tok_layout(int B, const int32_t* cu, int D) {
  TokLayout L{};
  L.sums_off = 0;
  L.work_off = align_up(static_cast<size_t>(B) * kSumSlots * D * sizeof(unsigned long long), 256);
  L.zero_bytes = L.work_off + static_cast<size_t>(B) * sizeof(TailWork);
  L.inv_off = align_up(L.zero_bytes, 256);
  L.total = L.inv_off + align_up(static_cast<size_t>(cu[B]) * sizeof(float), 256);
  return L;
}
}  // namespace
}  // namespace pace

extern "C" size_t pace_apc_density_tokens_workspace_size(int B, const int32_t* cu_tokens, int D) {
  if (B <= 0 || cu_tokens == nullptr || D < 2) return 0;
  return tok_layout(B, cu_tokens, D).total;
}

extern "C" pace_status_t pace_apc_density_tokens(const void* T, const int32_t* cu_tokens, int B, int D,
                                                 const int32_t* H, const int32_t* W,
                                                 const pace_apc_params* params, float* d_out,
                                                 pace_apc_stats* stats, void* ws, size_t ws_bytes,
                                                 pace_stream_t stream) {
  if (B < 0) return PACE_ERR_INVALID_ARG;
  if (B == 0) return PACE_OK;
  if (T == nullptr || cu_tokens == nullptr || H == nullptr || W == nullptr || d_out == nullptr || stats == nullptr)
    return PACE_ERR_INVALID_ARG;
  if (D < 2 || D > kTokMaxD || D % 2 != 0 || reinterpret_cast<uintptr_t>(T) % 4 != 0) return PACE_ERR_INVALID_ARG;
  if (cu_tokens[0] != 0) return PACE_ERR_INVALID_ARG;
  for (int b = 0; b < B; ++b)
    if (cu_tokens[b + 1] - cu_tokens[b] < 1 || H[b] < 1 || W[b] < 1) return PACE_ERR_INVALID_ARG;
  pace_apc_params p;
  PACE_CHECK(check_params(params, p));
  const TokLayout L = tok_layout(B, cu_tokens, D);
  if (ws == nullptr || ws_bytes < L.total || reinterpret_cast<uintptr_t>(ws) % 16) return PACE_ERR_WORKSPACE;
  PACE_CHECK(check_device());
  uint8_t* w8 = static_cast<uint8_t*>(ws);
  auto* sums = reinterpret_cast<unsigned long long*>(w8 + L.sums_off);
  auto* work = reinterpret_cast<TailWork*>(w8 + L.work_off);
  auto* inv = reinterpret_cast<float*>(w8 + L.inv_off);
  PACE_CHECK(launch_zero(w8, L.zero_bytes, nullptr, 0, stream));   // column sums and tail scratch
  const uint32_t* T32 = static_cast<const uint32_t*>(T);
  for (int c0 = 0; c0 < B; c0 += kApcMaxB) {
    const int nb = (B - c0) < kApcMaxB ? (B - c0) : kApcMaxB;
    TokTable tt{};
    ApcTable at{};   // what the tail kernel reads: sizes, token ranges, k_tail
    tt.nb = at.nb = nb;
    tt.b_base = at.b_base = c0;
    tt.D = D;
    tt.rows1 = std::max(1, std::min(32, kTok1StageBytes / (D * 2)));
    tt.unit_prefix[0] = 0;
    tt.unit_prefix1[0] = 0;
    tt.run_prefix[0] = 0;
    for (int i = 0; i < nb; ++i) {
      const int b = c0 + i;
      const int N = cu_tokens[b + 1] - cu_tokens[b];
      tt.tok0[i] = cu_tokens[b];
      tt.n[i] = at.n[i] = N;
      double kt = std::floor(static_cast<double>(p.tail_frac) * N + 0.5);
      if (kt < 1) kt = 1;
      if (kt > N) kt = N;
      tt.ktail[i] = at.ktail[i] = static_cast<int>(kt);
      tt.unit_prefix[i + 1] = tt.unit_prefix[i] + (N + kTokChunk - 1) / kTokChunk;
      tt.unit_prefix1[i + 1] = tt.unit_prefix1[i] + (N + tt.rows1 - 1) / tt.rows1;
      tt.run_prefix[i + 1] = tt.run_prefix[i] + (N + kTokRun - 1) / kTokRun;
      at.H[i] = H[b];
      at.W[i] = W[b];
      at.patch0[i] = cu_tokens[b];
    }
    const TailParams tp{p.alpha, p.gamma, p.r_min, p.r_max, p.align};
    // whole 16-byte vectors and at most kTokVecMax of them per lane: the register kernels
    if (D % 8 == 0 && D <= kTokVecMax * 256 && reinterpret_cast<uintptr_t>(T) % 16 == 0) {
      PACE_CHECK(launch_tok_vec(T, tt, static_cast<int64_t>(cu_tokens[c0 + nb]) - cu_tokens[c0], d_out, stats, inv, sums,
                                work, stream));
      PACE_CHECK(launch_tail(at, d_out, tp, stats, work, stream));
      continue;
    }
    const int units = tt.unit_prefix[nb];
    const int units1 = tt.unit_prefix1[nb];
    const size_t smem1 = 2 * static_cast<size_t>(tt.rows1) * D * 2;
    PACE_CHECK(tok_pass1_attr());
    apc_tok_pass1<<<tok_pass1_grid(units1), kApcThreads, smem1, stream>>>(T32, tt, units1, inv, sums);
    PACE_CHECK(check_launch());
    apc_tok_pass2<<<units, kApcThreads, 0, stream>>>(T32, tt, inv, sums, d_out, stats, work);
    PACE_CHECK(check_launch());
    PACE_CHECK(launch_tail(at, d_out, tp, stats, work, stream));
  }
  return PACE_OK;
}

// ------------------------------------------------------------------------------------------------
// pixel-statistic previews
// ------------------------------------------------------------------------------------------------
namespace pace {
namespace {

// Fills t for images c0 .. c0 + nb - 1 and launches the feature kernel on them (sums: null for the
// tokens alone).
pace_status_t launch_pix_features(const uint8_t* img, ApcTable& t, int c0, int nb, const int64_t* img_off, const int32_t* H,
                                  const int32_t* W, float tail_frac, int& patch0, int feature, float* tokens,
                                  unsigned long long* sums, cudaStream_t stream) {
  int sms = 0;
  PACE_CHECK(sm_count(&sms));
  fill_strip_table(t, c0, nb, img_off, H, W, tail_frac, kPixCtasPerSm * sms, patch0);
  const int units = t.unit_prefix[nb];
  const unsigned grid = static_cast<unsigned>(std::min(units, kPixCtasPerSm * sms));
  int* status = device_status_word();
  if (sums != nullptr)
    return launch_dependent(apc_pix_features<true>, grid, kApcThreads, 0, 1, stream, img, t, units, feature, tokens, sums, status);
  return launch_dependent(apc_pix_features<false>, grid, kApcThreads, 0, 1, stream, img, t, units, feature, tokens, sums, status);
}

int64_t total_patches(int B, const int32_t* H, const int32_t* W) {
  int64_t n = 0;
  for (int b = 0; b < B; ++b) n += static_cast<int64_t>(H[b] / kPatch) * (W[b] / kPatch);
  return n;
}

}  // namespace
}  // namespace pace

extern "C" pace_status_t pace_apc_pixel_features(const uint8_t* img, const int64_t* img_off, const int32_t* H,
                                                 const int32_t* W, int B, int feature, float* tokens,
                                                 pace_stream_t stream) {
  PACE_CHECK(check_images(img, img_off, H, W, B));
  if (B == 0) return PACE_OK;
  if (feature < kFeatRgb || feature > kFeatLaplacian || tokens == nullptr || reinterpret_cast<uintptr_t>(tokens) % 16)
    return PACE_ERR_INVALID_ARG;
  PACE_CHECK(check_device());
  int patch0 = 0;
  for (int c0 = 0; c0 < B; c0 += kApcMaxB) {
    ApcTable t;
    PACE_CHECK(launch_pix_features(img, t, c0, std::min(kApcMaxB, B - c0), img_off, H, W, 0.1f, patch0, feature, tokens,
                                   nullptr, stream));
  }
  return PACE_OK;
}

extern "C" size_t pace_apc_density_pixel_workspace_size(int B, const int32_t* H, const int32_t* W) {
  if (B <= 0 || H == nullptr || W == nullptr) return 0;
  for (int b = 0; b < B; ++b)
    if (H[b] < kPatch || W[b] < kPatch) return 0;
  return align_up(static_cast<size_t>(total_patches(B, H, W)) * kPixDim * sizeof(float), 256) +
         align_up(static_cast<size_t>(B) * kPixSlots * kPixDim * sizeof(unsigned long long), 256) +
         static_cast<size_t>(B) * sizeof(TailWork);
}

extern "C" pace_status_t pace_apc_density_pixel(const uint8_t* img, const int64_t* img_off, const int32_t* H,
                                                const int32_t* W, int B, int feature, const pace_apc_params* params,
                                                float* d_out, pace_apc_stats* stats, void* ws, size_t ws_bytes,
                                                pace_stream_t stream) {
  PACE_CHECK(check_images(img, img_off, H, W, B));
  if (B == 0) return PACE_OK;
  if (feature < kFeatRgb || feature > kFeatLaplacian || d_out == nullptr || stats == nullptr)
    return PACE_ERR_INVALID_ARG;
  pace_apc_params p;
  PACE_CHECK(check_params(params, p));
  const size_t tok_bytes = align_up(static_cast<size_t>(total_patches(B, H, W)) * kPixDim * sizeof(float), 256);
  if (ws == nullptr || ws_bytes < pace_apc_density_pixel_workspace_size(B, H, W) ||
      reinterpret_cast<uintptr_t>(ws) % 16)
    return PACE_ERR_WORKSPACE;
  PACE_CHECK(check_device());
  auto* tokens = static_cast<float*>(ws);
  auto* sums = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(ws) + tok_bytes);
  const size_t sums_bytes = align_up(static_cast<size_t>(B) * kPixSlots * kPixDim * sizeof(unsigned long long), 256);
  auto* work = reinterpret_cast<TailWork*>(reinterpret_cast<uint8_t*>(sums) + sums_bytes);
  PACE_CHECK(launch_zero(sums, sums_bytes, work, static_cast<size_t>(B) * sizeof(TailWork), stream));
  int patch0 = 0;
  for (int c0 = 0; c0 < B; c0 += kApcMaxB) {
    const int nb = std::min(kApcMaxB, B - c0);
    ApcTable at;
    PACE_CHECK(launch_pix_features(img, at, c0, nb, img_off, H, W, p.tail_frac, patch0, feature, tokens, sums, stream));
    PixTable pt{};
    pt.nb = nb;
    pt.b_base = c0;
    pt.unit_prefix[0] = 0;
    for (int i = 0; i < nb; ++i) {
      pt.tok0[i] = at.patch0[i];
      pt.n[i] = at.n[i];
      pt.ktail[i] = at.ktail[i];
      pt.unit_prefix[i + 1] = pt.unit_prefix[i] + (at.n[i] + kApcThreads - 1) / kApcThreads;
    }
    const int units = pt.unit_prefix[nb];
    PACE_CHECK(launch_dependent(apc_pix_pass2, static_cast<unsigned>(units), kApcThreads, 0, 1, stream, pt,
                                static_cast<const float*>(tokens), static_cast<const unsigned long long*>(sums), d_out,
                                stats, work));
    TailParams tp{p.alpha, p.gamma, p.r_min, p.r_max, p.align};
    PACE_CHECK(launch_tail(at, d_out, tp, stats, work, stream));
  }
  return PACE_OK;
}
