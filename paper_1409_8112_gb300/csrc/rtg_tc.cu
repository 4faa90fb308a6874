// Exact all-pairs r-NN (the problem of Sec. I of arXiv:1409.8112) with the distances taken
// from tensor-core tiles: d^2 = |x|^2 + |y|^2 - 2 x.y with x.y from tcgen05.mma (FP16 or BF16
// inputs, FP32 accumulation in tensor memory), and every pair whose FP32 d^2 lies within a
// band around fl(r^2) decided again with the FP64 reference sequence, so that the reported
// set is the same as the FP64 definition's.
//
// Each coordinate is centred on the bounding box and split as x = hi + lo (both half
// precision); x.y is approximated by hi.hi + hi.lo + lo.hi.  For d <= 9 the three products and
// the norms share one row of 32 halves (one or two K = 16 MMAs per tile pair); for d <= 12 the
// norms ride in the hi block of three MMAs; beyond, three MMAs give x.y and the epilogue adds
// the norms.  Operands sit in shared memory in the K-major layout without
// swizzle: core matrices of 8 rows x 16 bytes, 128 bytes apart along K and 512 bytes apart
// along M or N.  A CTA of ten warps (copies, MMAs, eight of epilogue) owns two 128 x 256 FP32
// accumulators, all 512 TMEM columns of its SM (k_brute_tc).  The band is max(1e-3 r^2, 1.25 E),
// and for unasked tiles at least what the CUDA-core filter keeps; E bounds the error of the FP32
// d^2: the hi/lo representation and dropped lo.lo term, FP32 accumulation of the products, the
// norms, the epilogue and the centring (tc_plan_band).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <limits>
#include <mutex>
#include <type_traits>

#include "rtg_internal.cuh"
#include "rtg_tc.cuh"

namespace rtg {

namespace {

constexpr int kTcRows = 128;
constexpr int kTcK = 32;                          // hi (16) + lo (16)
constexpr int kTcTileBytes = kTcRows * kTcK * 2;  // 8 KB per 128-point tile
// Epilogue warps, one TMEM load in flight each: a probe of tcgen05.ld.32x32b.x32 read 249 bytes
// a clock and SM with 4 warps, 323 with 8 and 60 with 16 (two loads in flight: 235 with 8).
constexpr int kTcEpiWarps = 8;
constexpr int kTcThreads = (kTcEpiWarps + 2) * 32;  // and one that copies tiles, one for the MMAs
constexpr int kTcSlots = 3;                       // pairs of column tiles in shared memory
constexpr int kTcPrepThreads = 256;
constexpr int kTcSample = 16;  // the plan's sample: pairs per thread of a block
// Unasked, the tiles are taken while no more than this share of the sampled pairs may lie within r
// (r^2 + band): each costs a check that the epilogue waits for, and on the CUDA cores, which also
// pay for every reported pair, far less.  30,011 points in 6-D,
// tiles against CUDA cores: 212 / 1075 us at a share of 0.03%, 1.5 / 6.1 ms at 3%, 3.3 / 9.1 at 10%,
// 8.5 / 11.2 at 30%, 14.9 / 13.0 at 60%.  Counting only: 188 / 1049 us, 0.86 / 1.10 ms at 3%, 1.13
// / 1.14 at 5%, 1.79 / 1.24 at 10%.  (16,000 points: 10% 1.0 / 2.7 ms, 60% 4.3 / 3.7.)
constexpr double kTcShareEmit = 0.4, kTcShareCount = 0.03;
// MMA completion waits: the context's spin limit times this (a commit takes far longer than
// one look-back step)
constexpr unsigned int kTcWaitScale = 16;

__device__ __forceinline__ double load_coord(const void* pts, int dtype, long long i, int d,
                                             int l) {
  return dtype == 0 ? __ldg((const double*)pts + i * d + l)
                    : (double)__ldg((const float*)pts + i * d + l);
}

// Centre of the bounding box on axis l, and the half extent.
__device__ __forceinline__ double tc_center(const unsigned long long* bbox, long long n, int l,
                                            double* half) {
  const double hi = n > 0 ? dec_double(bbox[l * 2 + 0]) : 0.0;
  const double lo = n > 0 ? dec_double(~bbox[l * 2 + 1]) : 0.0;
  *half = 0.5 * (hi - lo);
  return 0.5 * (lo + hi);
}

// Band and thresholds of instance 0 (one thread); whether the error bound lets the tiles be taken.
__device__ bool tc_plan_band(const Inst* __restrict__ inst, const unsigned long long* bbox,
                             const InstPlan* __restrict__ iplan, TcPlan* tp, int bf16, int fold,
                             int always) {
  const Inst I = inst[0];
  const int d = I.d;
  double M = 0.0;
  for (int l = 0; l < d; ++l) {
    double half;
    tc_center(bbox, I.n, l, &half);
    M = fmax(M, half * (1.0 + 1e-12) + 1e-300);
  }
  // Error bound of the FP32 d^2 (absolute), with u16 the unit roundoff of the half type:
  //   centring to FP32             8 sqrt(d) 2^-24 M (2 sqrt(d) M)
  //   hi/lo split + dropped lo.lo  2 d M^2 (2 u16^2 + 2^-22) + 2 d 2^-24 M   (x2 for -2x.y)
  //   FP32 accumulation of 48 terms 2 * 48 * 2^-24 * 2 d M^2, times 4 for an unknown order
  //   norms (two sums of d squares) 2 d 2^-24 d M^2
  //   epilogue (two roundings)      3 2^-24 (4 d M^2)
  const double E = fold ? tc_error_bound_folded(M, d, bf16 != 0) : tc_error_bound(M, d, bf16 != 0);
  const InstPlan IP = iplan[0];
  const double rr = IP.rr;
  double band = fmax(1e-3 * rr, 1.25 * E);
  // Unasked, the pairs the tiles leave are decided as on the CUDA cores, by the FP32 rows first:
  // every pair that filter would keep (FP32 d^2 <= s_hi, so d^2 <= s_hi + (s_hi - rr)) is left.
  if (!always && IP.filter_on)
    band = fmax(band, 2.0 * ((double)IP.s_hi - rr) * (1.0 + 1e-6) + 1.25 * E);
  tp->band = band;
  tp->bound = E;
  tp->lo = __double2float_rd(rr - band);
  tp->hi = __double2float_ru(rr + band);
  // Unasked, the tiles are taken when the band they need stays below an eighth of r^2 (so few
  // pairs fall inside it) and nothing overflows a half (coordinates doubled, norms).
  const double most = bf16 ? 1e30 : 60000.0;
  return always ||
         (band <= 0.125 * rr && 2.0 * M < most && (double)d * M * M < most);
}

// FP32 squared distance of two rows, in the order the CUDA-core kernels take it (their padding
// adds zeros).
__device__ __forceinline__ float tc_row_dist2(const float* pa, const float* pb, int d) {
  float s = 0.0f;
  for (int v = 0; 4 * v < d; ++v) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(pa) + v);
    const float4 y = __ldg(reinterpret_cast<const float4*>(pb) + v);
    float e = x.x - y.x;
    s = fmaf(e, e, s);
    e = x.y - y.y;
    s = fmaf(e, e, s);
    e = x.z - y.z;
    s = fmaf(e, e, s);
    e = x.w - y.w;
    s = fmaf(e, e, s);
  }
  return s;
}

// What the operand rows hold.  kTcPlain: [hi | lo], 16 halves each.  kTcFold (d <= 12): the
// tiles come in two versions, the A operand's ([-2 x, |x|^2 hi, |x|^2 lo, 1, 1] in the hi block)
// and the B operand's ([x, 1, 1, |y|^2 hi, |y|^2 lo]), so that the MMAs accumulate
// |x|^2 + |y|^2 - 2 x.y.  kTcPacked (3 d + 4 <= 32): A = [-2 hi, -2 hi, -2 lo, |x|^2 hi, |x|^2 lo,
// 1, 1] against B = [hi, lo, hi, 1, 1, |y|^2 hi, |y|^2 lo] in consecutive slots: the same
// products in two K = 16 MMAs instead of three (one for d <= 4), 64 of the 192 clocks a tile
// pair holds the tensor pipe.
enum TcForm : int { kTcPlain = 0, kTcFold = 1, kTcPacked = 2 };
inline TcForm tc_form(int d) { return d >= 1 && d <= 9 ? kTcPacked : (d <= 12 ? kTcFold : kTcPlain); }

// The plan's block: band and thresholds, and whether the tiles are taken: always when asked for,
// else by their error bound and by the share of a sample of the pairs that may lie within r.
__device__ void tc_plan_block(const Inst* __restrict__ inst, const unsigned long long* bbox,
                              const InstPlan* __restrict__ iplan, TcPlan* tp, Status* st, int bf16,
                              int fold, int always, const float* __restrict__ pf, int dpad,
                              unsigned int most_near) {
  __shared__ unsigned int s_near;
  __shared__ bool s_use;
  const Inst I = inst[0];
  float s[kTcSample];
  if (!always) {
#pragma unroll
    for (int q = 0; q < kTcSample; ++q) {
      // the multiples of 1 / p and 1 / p^2, p the plastic number, modulo 1 (a Kronecker sequence):
      // spread evenly over the index square
      const unsigned int k = threadIdx.x * kTcSample + q + 1;
      const long long i = ((long long)(k * 3242174889u) * I.n) >> 32;
      const long long j = ((long long)(k * 2447445414u) * I.n) >> 32;
      s[q] = i == j ? FLT_MAX : tc_row_dist2(pf + i * dpad, pf + j * dpad, I.d);
    }
  }
  if (threadIdx.x == 0) {
    s_near = 0;
    s_use = tc_plan_band(inst, bbox, iplan, tp, bf16, fold, always);
  }
  __syncthreads();
  if (!always) {
    const float hi = tp->hi;
    unsigned int near = 0;
#pragma unroll
    for (int q = 0; q < kTcSample; ++q) near += s[q] <= hi ? 1u : 0u;
    near = __reduce_add_sync(0xffffffffu, near);
    if ((threadIdx.x & 31) == 0 && near) atomicAdd(&s_near, near);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const bool use = s_use && s_near <= most_near;
    tp->use = use ? 1 : 0;
    if (use) st->tc_band = tp->band;
  }
}

// Half-precision rows in the tile layout, and FP32 norms of the centred points (read by the
// plain form only).  Block 0 makes the plan meanwhile (a launch of its own: 114 us a call for 4096
// points in 6-D, 109 so).
template <bool BF16, int FORM>
__global__ void __launch_bounds__(kTcPrepThreads) k_tc_prep(
    const Inst* __restrict__ inst, int dtype, const unsigned long long* __restrict__ bbox,
    const InstPlan* __restrict__ iplan, TcPlan* tp, Status* st, int always,
    const float* __restrict__ pf, int dpad, unsigned int most_near,
    unsigned char* __restrict__ tiles, float* __restrict__ norms, long long n_pad) {
  using H = typename std::conditional<BF16, __nv_bfloat16, __half>::type;
  auto to_h = [](float v) -> H {
    if constexpr (BF16) return __float2bfloat16_rn(v); else return __float2half_rn(v);
  };
  auto to_f = [](H v) -> float {
    if constexpr (BF16) return __bfloat162float(v); else return __half2float(v);
  };
  if (blockIdx.x == 0) {
    tc_plan_block(inst, bbox, iplan, tp, st, BF16 ? 1 : 0, FORM != kTcPlain ? 1 : 0, always, pf,
                  dpad, most_near);
    return;
  }
  __shared__ double s_center[kMaxDim];
  const Inst I = inst[0];
  if (threadIdx.x < kMaxDim) {
    double half;
    s_center[threadIdx.x] =
        (int)threadIdx.x < I.d ? tc_center(bbox, I.n, (int)threadIdx.x, &half) : 0.0;
  }
  __syncthreads();
  const long long i = (blockIdx.x - 1) * (long long)blockDim.x + threadIdx.x;
  if (i >= n_pad) return;
  const long long ntile = n_pad / kTcRows;
  unsigned char* tile = tiles + (i / kTcRows) * (long long)kTcTileBytes;
  unsigned char* tileB = FORM != kTcPlain ? tile + ntile * (long long)kTcTileBytes : tile;
  const int m = (int)(i % kTcRows);
  const int d = I.d;
  auto put = [&](unsigned char* t, int k, H v) { *reinterpret_cast<H*>(t + tile_off(m, k)) = v; };
  float nrm = 0.0f;
  const int width = FORM == kTcPacked ? d : 16;
  for (int k = 0; k < width; ++k) {
    float xc = 0.0f;
    if (i < I.n && k < d)
      xc = __double2float_rn(__dsub_rn(load_coord(I.pts, dtype, i, d, k), s_center[k]));
    nrm = fmaf(xc, xc, nrm);
    const H h = to_h(xc);
    const H l = to_h(xc - to_f(h));
    // A version: -2 x (exact scaling by a power of two)
    const H h2 = to_h(-2.0f * to_f(h)), l2 = to_h(-2.0f * to_f(l));
    if (FORM == kTcPacked) {
      put(tile, k, h2);
      put(tile, d + k, h2);
      put(tile, 2 * d + k, l2);
      put(tileB, k, h);
      put(tileB, d + k, l);
      put(tileB, 2 * d + k, h);
    } else {
      put(tile, k, FORM == kTcFold ? h2 : h);
      put(tile, 16 + k, FORM == kTcFold ? l2 : l);
      if (FORM == kTcFold) {
        put(tileB, k, h);
        put(tileB, 16 + k, l);
      }
    }
  }
  if (FORM != kTcPlain) {
    const int q = FORM == kTcPacked ? 3 * d : d;  // the four slots of the norms
    const H nh = to_h(nrm), nl = to_h(nrm - to_f(nh)), one = to_h(1.0f);
    put(tile, q, nh);
    put(tile, q + 1, nl);
    put(tile, q + 2, one);
    put(tile, q + 3, one);
    put(tileB, q, one);
    put(tileB, q + 1, one);
    put(tileB, q + 2, nh);
    put(tileB, q + 3, nl);
    if (FORM == kTcPacked)
      for (int k = q + 4; k < kTcK; ++k) {
        put(tile, k, to_h(0.0f));
        put(tileB, k, to_h(0.0f));
      }
  }
  norms[i] = nrm;
}

struct TcSink {
  unsigned int* row_cnt;
  unsigned long long* pair_buf;
  long long pair_cap;
  unsigned long long* emitted;
  int symmetric;
};

__device__ __forceinline__ double exact_dist2(const void* pts, int dtype, long long i, long long j,
                                           int d) {
  double s = 0.0;
  for (int l = 0; l < d; ++l) {
    const double e = __dsub_rn(load_coord(pts, dtype, i, d, l), load_coord(pts, dtype, j, d, l));
    s = __fma_rn(e, e, s);
  }
  return s;
}

// What a warp's candidates add up to in one drain.
struct TcTally {
  unsigned int pairs = 0, owned = 0, rechecks = 0, near_r = 0;
  float max_err = 0.0f;
};

// Whether a pair the tile did not reject lies within r.  With rows (pf; the unasked tiles, where
// the FP32 filter holds) as the CUDA-core kernel decides it: FP32 outside its band, else the FP64
// reference sequence.  Without, by the FP64 sequence.  Only rejections rely on the tile's error
// bound; [lo, hi] is where the tile alone could not decide.
__device__ __forceinline__ bool tc_decide(float d2, unsigned int gi, unsigned int gj, const Inst* Ip,
                                          const InstPlan* IPp, int dtype, float lo_thr,
                                          const float* pf, int dpad, TcTally& tl) {
  const Inst& I = *Ip;  // (read where it is used: the epilogue has no registers to spare)
  bool open = !(d2 < lo_thr);  // (with a band 1e-3 r^2 wide, all within 1e-12 r of r are open)
  if (pf) {
    const float s = tc_row_dist2(pf + (size_t)gi * dpad, pf + (size_t)gj * dpad, I.d);
    if (s > IPp->s_hi) return false;
    ++tl.owned;
    if (s < IPp->s_lo) return true;
    open = true;
  } else {
    ++tl.owned;
  }
  const double s = exact_dist2(I.pts, dtype, gi, gj, I.d);
  tl.max_err = fmaxf(tl.max_err, (float)fabs((double)d2 - s));
  if (open) {
    ++tl.rechecks;
    if (fabs(__dsub_rn(__dsqrt_rn(s), I.r)) <= __dmul_rn(1e-12, I.r)) ++tl.near_r;
  }
  return s <= IPp->rr;
}

// Candidates queued per warp before their exact check.  A check waits on the points' loads for
// about two microseconds, and the accumulators wait with it, so a warp collects many: the
// warps of a CTA then mostly check at the same time (at the end, at 200k points).  The check is
// inlined: a call makes the compiler keep the accumulators a warp holds in local memory.
constexpr int kTcQueue = 768;
static_assert(kTcQueue <= 32 * 32, "a bit per 32 candidates");

// A CTA's sums.  64 bits: a CTA takes up to 2^30 jobs of 2^16 pairs (1.2 million points with every
// pair within r pass 2^32 on 152 CTAs).
using TcCount = unsigned long long;
constexpr int kTcJobPairs = 256 * 256;
constexpr long long kTcMaxJobs = 1LL << 30;
static_assert(std::numeric_limits<TcCount>::max() / kTcJobPairs >= (TcCount)kTcMaxJobs,
              "a CTA's pairs must be countable");
struct TcCounts {
  TcCount pairs, owned, rechecks, near_r;
  unsigned int max_err;  // float bits
};

// Decides the qn queued candidates of a warp, 32 at a time (one per lane), delivers the pairs and
// adds up in cnt (shared memory).  Called by all lanes.
__device__ __forceinline__ void tc_drain(const unsigned int* q_i, const unsigned int* q_j,
                                         const float* q_d, unsigned int qn, int lane,
                                         const Inst* I, const InstPlan* IP, int dtype,
                                         float lo_thr, const float* pf, int dpad,
                                         const TcSink& sk, bool emit, TcCounts* cnt,
                                         unsigned int* errors) {
  const unsigned int full = 0xffffffffu;
  __syncwarp();
  TcTally tl;
  const unsigned int p0 = (unsigned int)I->p0;
  unsigned int kept = 0;  // bit k: this lane's candidate of the k-th 32 is a pair
  for (unsigned int k = 0; 32 * k < qn; ++k) {
    const unsigned int e = 32 * k + lane;
    if (e < qn && tc_decide(q_d[e], q_i[e], q_j[e], I, IP, dtype, lo_thr, pf, dpad, tl)) {
      kept |= 1u << k;
      atomicAdd(&sk.row_cnt[p0 + q_i[e]], 1u);
      if (sk.symmetric) atomicAdd(&sk.row_cnt[p0 + q_j[e]], 1u);
    }
  }
  tl.pairs = __reduce_add_sync(full, (unsigned int)__popc(kept));
  tl.owned = __reduce_add_sync(full, tl.owned);
  tl.rechecks = __reduce_add_sync(full, tl.rechecks);
  tl.near_r = __reduce_add_sync(full, tl.near_r);
  if (emit && tl.pairs) {  // one reservation for the drain
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(sk.emitted, (unsigned long long)tl.pairs);
    long long slot = (long long)__shfl_sync(full, base, 0);
    if (lane == 0 && slot + tl.pairs > sk.pair_cap) atomicOr(errors, kErrPairOverflow);
    for (unsigned int k = 0; 32 * k < qn; ++k) {
      const unsigned int mask = __ballot_sync(full, (kept >> k) & 1u);
      const long long at = slot + __popc(mask & ((1u << lane) - 1u));
      if (((kept >> k) & 1u) && at < sk.pair_cap)
        sk.pair_buf[at] = ((unsigned long long)(p0 + q_i[32 * k + lane]) << 32) |
                          (p0 + q_j[32 * k + lane]);
      slot += __popc(mask);
    }
  }
  const unsigned int err = __reduce_max_sync(full, __float_as_uint(tl.max_err));
  if (lane == 0) {
    atomicAdd(&cnt->pairs, (TcCount)tl.pairs);
    atomicAdd(&cnt->owned, (TcCount)tl.owned);
    atomicAdd(&cnt->rechecks, (TcCount)tl.rechecks);
    if (tl.near_r) atomicAdd(&cnt->near_r, (TcCount)tl.near_r);
    atomicMax(&cnt->max_err, err);
  }
  __syncwarp();  // the queue may be filled again
}

// The smaller of three values, NaN if any is NaN.
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Bounded wait that also ends when another thread of the block has given up.
__device__ __forceinline__ bool tc_wait(const uint64_t* bar, uint32_t parity, unsigned int limit,
                                        volatile int* late) {
  const uint32_t addr = smem_u32(bar);
  for (unsigned int it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
    if (*late) return false;
  }
  *late = 1;
  return false;
}

// One thread: copy `bytes` (a multiple of 16, both ends 16-byte aligned) to shared memory,
// counted on bar (whose expected bytes the caller has set).
__device__ __forceinline__ void tc_bulk_copy(void* dst, const void* src, uint32_t bytes,
                                             const uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tc_expect(const uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void tc_commit(const uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// Jobs of the brute force: blocks of 256 rows (row tiles 2 I and 2 I + 1) against blocks of 256
// columns, J >= I, I-major.  First job of I among nb blocks.
__host__ __device__ inline long long tc_first_job(long long I, long long nb) {
  return I * nb - I * (I - 1) / 2;
}

// Shared memory of k_brute_tc: two pairs of row tiles, the column tiles, the candidate queues.
constexpr size_t kTcSmem = (4 + 2 * kTcSlots) * (size_t)kTcTileBytes +
                           (size_t)kTcEpiWarps * 3 * kTcQueue * 4 + 1024;

// One lane of a converged warp.
__device__ __forceinline__ bool tc_elect() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e != 0u;
}

// Persistent, one CTA per SM, each with a contiguous range of jobs.  One warp copies the tiles in
// (bulk copies: column tiles up to kTcSlots jobs ahead, row tiles one change ahead), one issues
// the MMAs, 128 x 256 each: a job's two row tiles are the two accumulators of 256 columns, so
// that the MMAs of one overlap the reads of the other.  Both run their loops as whole warps and
// elect a lane for the copies and MMAs (a single lane running the loop, copies included, took
// 1500 clocks a 256 x 128 job).  Eight epilogue warps read the accumulators in turn: warp w the
// rows of its quadrant w % 4, columns 128 (w / 4) on, in four loads of 32 columns, two at a
// time; then the accumulator is free again.  No block barrier in the loop.
// An epilogue chunk of 32 columns is first reduced to its smallest d^2 with three-input minima
// (16 instructions for 32 values); only a chunk that holds a value not above the threshold (one
// in eleven at 200k points, degree 24) builds the mask of its candidates.  A job of 256 x 256
// costs 16 KB of column tiles for four tile pairs (8 KB for each would be near 60 bytes a clock
// and SM of L2 bandwidth).
// 200k points in 6-D (2e10 pair tests), FP16: 7.26 ms with 128 x 128 jobs, 4 CTAs per SM, block
// barriers and a mask for every chunk; 3.28 now: 1.84 without candidates (the TMEM reads alone
// would take 0.8, the MMAs 0.5), the rest for the 1.8 million candidates, for each of which a
// warp stops about 800 clocks and the others wait for its accumulator.
template <bool BF16, bool EMIT, int FORM>
__global__ void __launch_bounds__(kTcThreads, 1) k_brute_tc(
    const unsigned char* __restrict__ tiles, const float* __restrict__ norms,
    const Inst* __restrict__ inst, const InstPlan* __restrict__ iplan,
    const TcPlan* __restrict__ tp, int dtype, const float* __restrict__ rows, int dpad, Status* st,
    TcSink sk, long long nt, unsigned int wait_limit, unsigned int inject) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* s_a = smem;                      // row tiles 2 I, 2 I + 1, of two I
  unsigned char* s_b = smem + 4 * kTcTileBytes;   // kTcSlots pairs of column tiles
  __shared__ __align__(8) uint64_t b_full[kTcSlots], b_empty[kTcSlots], acc_full[2], acc_empty[2],
      a_full[2], a_empty[2], all_done, b_idle;  // b_idle: test hook, a barrier nothing arrives on
  __shared__ uint32_t tmem_base;
  __shared__ TcCounts s_cnt;
  __shared__ int s_late;  // some wait ran out
  const unsigned int full = 0xffffffffu;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (!tp->use) return;  // the CUDA-core kernel takes the pairs
  const long long nb = (nt + 1) / 2;  // blocks of 256 points
  const long long jobs = tc_first_job(nb, nb);
  const long long per = (jobs + gridDim.x - 1) / gridDim.x;
  const long long j0 = min(jobs, (long long)blockIdx.x * per), j1 = min(jobs, j0 + per);
  if (tid == 0) {
    s_cnt = TcCounts{};
    s_late = 0;
    auto init = [](const uint64_t* bar, int count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
    };
    for (int q = 0; q < kTcSlots; ++q) {
      init(&b_full[q], 1);
      init(&b_empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      init(&acc_full[q], 1);
      init(&acc_empty[q], kTcEpiWarps);
      init(&a_full[q], 1);
      init(&a_empty[q], 1);
    }
    init(&all_done, 1);
    init(&b_idle, 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
    asm volatile("fence.proxy.async.shared::cta;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  // first (I, J) of this CTA
  long long I0 = 0, J0 = 0;
  if (j0 < j1) {
    long long lo = 0, hi = nb - 1;
    while (lo < hi) {  // the last I whose first job is <= j0
      const long long mid = (lo + hi + 1) >> 1;
      if (tc_first_job(mid, nb) <= j0) lo = mid; else hi = mid - 1;
    }
    I0 = lo;
    J0 = lo + (j0 - tc_first_job(lo, nb));
  }
  const int count = (int)(j1 - j0);  // (at most 2^30)
  const int ntile = (int)nt, nblk = (int)nb;

  if (warp == kTcEpiWarps) {
    // copies.  (unless plain, the B operand's tiles follow the A operand's, and hold the norms)
    const unsigned char* tilesB = FORM != kTcPlain ? tiles + nt * (long long)kTcTileBytes : tiles;
    int I = (int)I0, J = (int)J0, change = 0, a_copied = 0, p = 0;
    bool ok = true, fresh = true;
    for (; p < count; ++p) {
      if (fresh) {  // the next pair of row tiles (in use until the MMAs of the pair before last end)
        const int as = change & 1;
        if (change >= 2) ok = tc_wait(&a_empty[as], (uint32_t)(((change >> 1) - 1) & 1), wait_limit, &s_late);
        ok = __all_sync(full, ok);
        if (!ok) break;
        const bool two = 2 * I + 1 < ntile;  // (else the second tile lies beyond n: ignored)
        if (tc_elect()) {
          tc_expect(&a_full[as], two ? 2 * kTcTileBytes : kTcTileBytes);
          const unsigned char* src = tiles + 2LL * I * kTcTileBytes;
          tc_bulk_copy(s_a + as * 2 * kTcTileBytes, src, kTcTileBytes, &a_full[as]);
          if (two)
            tc_bulk_copy(s_a + (as * 2 + 1) * kTcTileBytes, src + kTcTileBytes, kTcTileBytes,
                         &a_full[as]);
        }
        ++change;
        a_copied = change;
        fresh = false;
      }
      const int slot = p % kTcSlots;
      if (p >= kTcSlots)
        ok = tc_wait(&b_empty[slot], (uint32_t)((p / kTcSlots - 1) & 1), wait_limit, &s_late);
      ok = __all_sync(full, ok);
      if (!ok) break;
      if (tc_elect()) {
        const bool two = 2 * J + 1 < ntile;
        tc_expect(&b_full[slot], two ? 2 * kTcTileBytes : kTcTileBytes);
        tc_bulk_copy(s_b + slot * 2 * kTcTileBytes, tilesB + 2LL * J * kTcTileBytes,
                     two ? 2 * kTcTileBytes : kTcTileBytes, &b_full[slot]);
      }
      if (++J == nblk) {
        J = ++I;
        fresh = true;
      }
    }
    // no copy is left in flight when the block ends (bounded waits, each on a copy's newest phase)
    int never = 0;
    for (int z = max(0, p - kTcSlots); z < p; ++z)
      tc_wait(&b_full[z % kTcSlots], (uint32_t)((z / kTcSlots) & 1), wait_limit, &never);
    for (int z = max(0, a_copied - 2); z < a_copied; ++z)
      tc_wait(&a_full[z & 1], (uint32_t)((z >> 1) & 1), wait_limit, &never);
    __syncwarp();
  } else if (warp == kTcEpiWarps + 1) {
    // MMAs
    const uint32_t idesc = (1u << 4) | ((BF16 ? 1u : 0u) << 7) | ((BF16 ? 1u : 0u) << 10) |
                           ((256u >> 3) << 17) | ((128u >> 4) << 24);
    const bool one_part = FORM == kTcPacked && 3 * inst[0].d + 4 <= 16;
    const uint64_t adesc = make_desc(smem_u32(s_a)), bdesc = make_desc(smem_u32(s_b));
    int I = (int)I0, J = (int)J0, change = 0;
    bool ok = true, fresh = true;
    for (int q = 0; q < count; ++q) {
      const int slot = q % kTcSlots;
      if (fresh) {
        ok = tc_wait(&a_full[change & 1], (uint32_t)((change >> 1) & 1), wait_limit, &s_late);
        ++change;
        fresh = false;
      }
      if (ok) ok = tc_wait(&b_full[slot], (uint32_t)((q / kTcSlots) & 1), wait_limit, &s_late);
      const uint64_t ad0 = adesc + (uint64_t)(((change - 1) & 1) * 2 * (kTcTileBytes / 16));
      const uint64_t bd0 = bdesc + (uint64_t)(slot * 2 * (kTcTileBytes / 16));
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        if (ok && q >= 1)  // the epilogue has read this accumulator's last job
          ok = tc_wait(&acc_empty[mt], (uint32_t)((q - 1) & 1), wait_limit, &s_late);
        ok = __all_sync(full, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tc_elect()) {
          // plain and folded: hi.hi + hi.lo + lo.hi, A parts (0, 0, 1), B parts (0, 1, 0);
          // packed: parts (0, 0), (1, 1); 256 bytes per part
          const uint32_t d = tmem + (uint32_t)(mt * 256);
          const uint64_t am = ad0 + (uint64_t)(mt * (kTcTileBytes / 16));
#pragma unroll
          for (int part = 0; part < (FORM == kTcPacked ? 2 : 3); ++part) {
            if (part == 1 && one_part) break;
            const uint64_t ad = am + (FORM == kTcPacked ? part * 16u : (part == 2 ? 16u : 0u));
            const uint64_t bd = bd0 + (part == 1 ? 16u : 0u);
            asm volatile(
                "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                "l"(ad), "l"(bd), "r"(idesc), "r"(part > 0 ? 1u : 0u));
          }
          tc_commit(&acc_full[mt]);
          if (mt == 1) {
            tc_commit(&b_empty[slot]);
            if (J + 1 == nblk) tc_commit(&a_empty[(change - 1) & 1]);
          }
        }
        __syncwarp();
      }
      if (!ok) break;
      if (++J == nblk) {
        J = ++I;
        fresh = true;
      }
    }
    // nor an MMA
    int never = 0;
    if (tc_elect()) tc_commit(&all_done);
    __syncwarp();
    tc_wait(&all_done, 0u, wait_limit, &never);
    __syncwarp();
  } else {
    const float hi_thr = tp->hi;
    const int quad = warp & 3, half = warp >> 2;
    unsigned int* q_i = reinterpret_cast<unsigned int*>(smem + (4 + 2 * kTcSlots) * kTcTileBytes) +
                        (size_t)warp * 3 * kTcQueue;  // rows, columns, tile d^2
    unsigned int* q_j = q_i + kTcQueue;
    float* q_d = reinterpret_cast<float*>(q_j + kTcQueue);
    unsigned int qn = 0;  // entries queued (warp-uniform)
    // the rows that decide, where the tiles were not asked for and the FP32 filter holds
    const float* pf = iplan[0].filter_on ? rows : nullptr;
    int I = (int)I0, J = (int)J0;
    for (int unit = 0; unit < 2 * count; ++unit) {
      const int q = unit >> 1, mt = unit & 1;
      const bool ok = tc_wait((inject & kInjectTcWait) ? &b_idle : &acc_full[mt],
                              (uint32_t)(q & 1), wait_limit, &s_late);
      if (!__all_sync(full, ok)) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const long long gi = (2LL * I + mt) * kTcRows + quad * 32 + lane;
      const unsigned int cbase = (unsigned int)(2 * J + half) * kTcRows;  // first column
      // a job on the diagonal, or with columns past the points
      const bool edge = J == I || J == nblk - 1;
      const uint32_t acc =
          tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(mt * 256 + half * 128);
      // 64 columns at a time: a warp that held all 128 would spill
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        float d2[2][32], least[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t r[32];
          tc_ld32(acc + (uint32_t)(g * 64 + h * 32), r);
          if (FORM == kTcPlain) {
            const float nrow = gi < nt * kTcRows ? __ldg(norms + gi) : 0.0f;
            const float4* nb = reinterpret_cast<const float4*>(
                norms + min((long long)cbase, (nt - 1) * kTcRows) + g * 64 + h * 32);
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              const float4 c4 = __ldg(nb + v);
              d2[h][4 * v] = (nrow + c4.x) - 2.0f * __uint_as_float(r[4 * v]);
              d2[h][4 * v + 1] = (nrow + c4.y) - 2.0f * __uint_as_float(r[4 * v + 1]);
              d2[h][4 * v + 2] = (nrow + c4.z) - 2.0f * __uint_as_float(r[4 * v + 2]);
              d2[h][4 * v + 3] = (nrow + c4.w) - 2.0f * __uint_as_float(r[4 * v + 3]);
            }
          } else {
#pragma unroll
            for (int v = 0; v < 32; ++v) d2[h][v] = __uint_as_float(r[v]);
          }
          float m0 = d2[h][0], m1 = d2[h][1];
#pragma unroll
          for (int v = 2; v + 3 < 32; v += 4) {
            m0 = min3_nan(m0, d2[h][v], d2[h][v + 1]);
            m1 = min3_nan(m1, d2[h][v + 2], d2[h][v + 3]);
          }
          m0 = min3_nan(m0, d2[h][30], d2[h][31]);
          least[h] = min3_nan(m0, m1, m1);
        }
        if (g == 1) {  // read: the accumulator is free
          asm volatile("tcgen05.fence::before_thread_sync;");
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[mt]))
                         : "memory");
        }
        // Candidates go to the warp's shared-memory queue, kept across jobs, and are decided 32 at
        // a time, one per lane, so that the FP64 checks and their global loads run in parallel.
        const bool found = __any_sync(
            full, !(min3_nan(least[0], least[1], least[1]) > hi_thr));
        if (found) {  // (NaN too)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!__any_sync(full, !(least[h] > hi_thr))) continue;
            const unsigned int col0 = cbase + g * 64 + h * 32;
            // NaN (overflowed tiles) goes to FP64; four chains, for the latency
            uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              if (!(d2[h][v] > hi_thr)) m0 |= 1u << v;
              if (!(d2[h][8 + v] > hi_thr)) m1 |= 1u << (8 + v);
              if (!(d2[h][16 + v] > hi_thr)) m2 |= 1u << (16 + v);
              if (!(d2[h][24 + v] > hi_thr)) m3 |= 1u << (24 + v);
            }
            uint32_t hits = (m0 | m1) | (m2 | m3);
            if (edge) {  // columns v with gi < col0 + v < n
              const long long vlo = gi - (long long)col0 + 1, vhi = (long long)inst->n - (long long)col0;
              uint32_t valid = 0;
              if (vlo < 32 && vhi > 0) {
                const int a0 = vlo > 0 ? (int)vlo : 0, a1 = vhi < 32 ? (int)vhi : 32;
                if (a1 > a0) valid = (a1 - a0 == 32 ? full : ((1u << (a1 - a0)) - 1u)) << a0;
              }
              hits &= valid;
            }
            // one candidate a lane and round: a lane's only one is its smallest value (the usual
            // round), others are picked out of the registers
            uint32_t who = __ballot_sync(full, hits != 0u);
            bool only = !edge && (hits & (hits - 1u)) == 0u;
            while (who) {
              if (qn + 32u > (unsigned int)kTcQueue) {
                tc_drain(q_i, q_j, q_d, qn, lane, inst, iplan, dtype, tp->lo, pf, dpad, sk, EMIT,
                         &s_cnt, &st->errors);
                qn = 0;
              }
              if (hits) {
                const int v = __ffs(hits) - 1;
                float x = least[h];
                if (!only) {
#pragma unroll
                  for (int z = 0; z < 32; ++z) x = z == v ? d2[h][z] : x;
                }
                const unsigned int pos = qn + (unsigned int)__popc(who & ((1u << lane) - 1u));
                q_i[pos] = (unsigned int)gi;
                q_j[pos] = col0 + (unsigned int)v;
                q_d[pos] = x;
                hits &= hits - 1u;
              }
              qn += (unsigned int)__popc(who);
              who = __ballot_sync(full, hits != 0u);
            }
          }
        }
      }
      if (mt == 1 && ++J == nblk) J = ++I;
    }
    if (qn)  // the candidates still queued
      tc_drain(q_i, q_j, q_d, qn, lane, inst, iplan, dtype, tp->lo, pf, dpad, sk, EMIT, &s_cnt,
               &st->errors);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (tid == 0) {
    if (s_late) atomicOr(&st->errors, kErrTimeout);
    if (s_cnt.pairs) atomicAdd(&st->pairs, s_cnt.pairs);
    if (rows && s_cnt.owned) atomicAdd(&st->owned_candidates, s_cnt.owned);
    if (s_cnt.rechecks) atomicAdd(&st->dist_rechecks, s_cnt.rechecks);
    if (s_cnt.near_r) atomicAdd(&st->near_r, s_cnt.near_r);
    atomicMax(&st->tc_max_err_bits, s_cnt.max_err);
  }
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

}  // namespace

size_t tc_tiles_bytes(long long n) {
  const long long nt = (n + kTcRows - 1) / kTcRows;
  return 2 * (size_t)nt * kTcTileBytes;  // A and B versions (norms folded into the MMA)
}

int launch_brute_tc(const BuildArgs& a, bool bf16, Mode mode, unsigned char* tiles, float* norms,
                    TcPlan* tp, bool always, cudaStream_t s) {
  const long long n = a.n_total;
  const long long nt = (n + kTcRows - 1) / kTcRows;
  const long long n_pad = nt * kTcRows;
  const TcForm form = tc_form(a.d_max);  // (one instance: its d)
  const unsigned pblocks = (unsigned)((n_pad + kTcPrepThreads - 1) / kTcPrepThreads) + 1;
  const bool emit = mode == kEmit;
  const double share = always ? 1.0 : (emit ? kTcShareEmit : kTcShareCount);
  auto prep = bf16 ? (form == kTcPacked ? k_tc_prep<true, kTcPacked>
                                        : (form == kTcFold ? k_tc_prep<true, kTcFold>
                                                           : k_tc_prep<true, kTcPlain>))
                   : (form == kTcPacked ? k_tc_prep<false, kTcPacked>
                                        : (form == kTcFold ? k_tc_prep<false, kTcFold>
                                                           : k_tc_prep<false, kTcPlain>));
  prep<<<pblocks, kTcPrepThreads, 0, s>>>(a.inst, a.dtype, a.bbox, a.iplan, tp, a.st,
                                          always ? 1 : 0, a.pf, a.dpad,
                                          (unsigned int)(share * kTcSample * kTcPrepThreads), tiles,
                                          norms, n_pad);
  TcSink sk{a.row_cnt, a.pair_buf, a.pair_cap, &a.st->emitted, a.symmetric};
  // one CTA per SM (it takes all 512 TMEM columns): more than half of the shared memory
  const size_t smem = kTcSmem > 120 * 1024 ? kTcSmem : 120 * 1024;
  const long long nb = (nt + 1) / 2, jobs = tc_first_job(nb, nb);
  // (more CTAs than that only where a CTA's jobs would not be counted in 31 bits)
  const unsigned grid = (unsigned)std::max<long long>(std::min<long long>(jobs, a.num_sms),
                                                      (jobs + kTcMaxJobs - 1) / kTcMaxJobs);
#define RTG_TC_LAUNCH1(B, E, F)                                                                \
  do {                                                                                         \
    static size_t attr[64] = {};                                                               \
    int dev = 0;                                                                               \
    cudaGetDevice(&dev);                                                                       \
    std::lock_guard<std::mutex> lk(launch_attr_mutex());                                       \
    if (dev < 0 || dev >= 64 || attr[dev] < smem) {                                            \
      cudaFuncSetAttribute(k_brute_tc<B, E, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                           (int)smem);                                                         \
      if (dev >= 0 && dev < 64) attr[dev] = smem;                                              \
    }                                                                                          \
    k_brute_tc<B, E, F><<<grid, kTcThreads, smem, s>>>(tiles, norms, a.inst, a.iplan, tp,       \
                                                       a.dtype, always ? nullptr : a.pf, a.dpad, \
                                                    a.st, sk, nt,                              \
                                                    spin_limit_of(a.spin_limit) * kTcWaitScale, \
                                                    a.inject);                                 \
  } while (0)
#define RTG_TC_LAUNCH(B, E)             \
  do {                                   \
    if (form == kTcPacked) RTG_TC_LAUNCH1(B, E, kTcPacked); \
    else if (form == kTcFold) RTG_TC_LAUNCH1(B, E, kTcFold); \
    else RTG_TC_LAUNCH1(B, E, kTcPlain);     \
  } while (0)
  if (grid > 0) {
    if (bf16 && emit) RTG_TC_LAUNCH(true, true);
    else if (bf16) RTG_TC_LAUNCH(true, false);
    else if (emit) RTG_TC_LAUNCH(false, true);
    else RTG_TC_LAUNCH(false, false);
  }
#undef RTG_TC_LAUNCH
#undef RTG_TC_LAUNCH1
  return grid > 0 ? 2 : 1;
}

}  // namespace rtg
