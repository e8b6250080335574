// The FP32 Gaussian kernel block on the tensor cores (tcgen05): FP32 rows in
// three FP16 slices, products exact where it matters.
//
//   out[n][m] = exp(-max(0, |p|^2 + |q|^2 - 2 p.q) / (2 sigma^2))
//
// Every row is scaled by a power of two so that its largest |value| lies in
// [2^14, 2^15), and a scaled value is cut into hi + mid + lo: hi a multiple of
// 2^7 with at most 256 steps, mid the rest (at most 64) rounded to FP16, lo
// what mid leaves (at most 2^-6) rounded to FP16.  The product p.q is then six
// FP16 products: hi.hi, hi.mid, mid.hi, mid.mid, hi.lo and lo.hi.  Slicing the
// operands so that the leading products sum without error is the method of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012).
//
// Accuracy: a tensor-core accumulator drops the bits below its last place at
// every step, which would bias a long FP32 sum by parts in 10^6.  hi.hi is
// kept exact instead: its products are multiples of 2^14 of at most 2^16
// steps, so 256 of them stay below 2^24 steps and no bit is dropped.  The
// other five products share a second accumulator, small for most rows and
// never more than 80 steps long: every 256 values of K the epilogue adds both
// to FP32 sums in registers (rounded to nearest).  The three products left out
// (mid.lo and smaller) come to about 0.23 sqrt(2 d) in scaled units.  Measured
// against 64 bits (rms error of the squared distance in 2^-24 (|p|^2 + |q|^2),
// FFMA kernel in brackets): k/255 features of 784 values 0.82 (0.89), normal
// values 0.83 (0.83), normal + 100 0.84 (1.28); rows whose largest value stands
// far out, 0.1 to 0.4 with one 4.0 (64 values) 0.79 (0.86), with one 8.0 (784)
// 0.83 (0.94), with one 30.0 0.69 (0.68), log-normal of sigma 2 0.85 (0.86) at
// 784 and 0.89 (0.88) at 2,048 values.  (mid and lo as multiples of 2^-2 and
// 2^-11 and one second sum per tile, as before, gave 1.63, 3.34, 1.78, 1.38
// and 1.69 on those five.)  Rows beyond those bounds are left to FFMA sums, row
// by row (see split_rows_kernel).
//
// What bounds it: six FP16 products of 2 d flop per entry.  At 784 values a
// 3,001 x 15,013 block takes 0.27 ms (1.57 PFLOP/s of FP16 products, 0.82 of
// the measured BF16 rate) against 1.57 ms for the FFMA kernel (45 of the 74
// TFLOP/s that independent FFMAs reach).  A tile's exponentials and stores took
// 20,000 clocks as one chain behind a column test each, longer than the 8
// stages of MMAs that cover them, so the next chunk waited 4,300: computed in
// eights without the test (full tiles) and with an elected issuer it is 0.27
// instead of 0.29 ms.  Pairs of SMs (cta_group::2) measured 0.29-0.31 ms.
//
// Structure (persistent, one CTA of ten warps per SM, 128 samples x 256
// references): warp 0 fills three 72 KB stages by TMA (32 values of K, the
// three slices of both sides, 64-byte swizzle), warp 1 issues the MMAs, warps
// 2..9 drain and finish.  hi.hi has tensor-memory columns 0..255, the rest
// 256..511.  In a stage the ten MMAs of the second accumulator go first, so
// the drain of one accumulator runs beside MMAs into the other; running totals
// live in registers (128 per epilogue thread), so the next tile's MMAs start
// when the accumulators are read, before the exponentials and the stores.
// Every wait is bounded, and the issuing warp's lanes leave a wait together; a
// CTA ends only when its copies and MMAs have.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace kkm {

constexpr int SP_M = 128;
constexpr int SP_K = 32;                         // values of K per stage (64-byte rows)
constexpr int SP_STAGES = 3;
constexpr int SP_A_BYTES = SP_M * SP_K * 2;      // a slice of the sample tile
constexpr int SP_CHUNK = 256 / SP_K;             // stages whose hi.hi products sum exactly
constexpr int SP_THREADS = 320;
// N references per tile: 256, or 64 when tiles of 256 would leave half of the
// SMs idle (a few samples: one tile's 25 stages of d = 784 are then a chain of
// 10 us on a few SMs, against 3 us).  An entry's sums do not depend on N.
template <int N>
struct SpCfg {
  static constexpr int kBBytes = N * SP_K * 2;   // a slice of the reference tile
  static constexpr int kStageBytes = 3 * (SP_A_BYTES + kBBytes);
  static constexpr size_t kSmem = (size_t)SP_STAGES * kStageBytes + 1024;
  static constexpr int kTmemCols = 2 * N;
};

// kind::f16, FP32 accumulator, F16 A and B, both K-major.
__host__ __device__ constexpr uint32_t sp_idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(SP_M >> 4) << 24);
}
// K-major operand tile of 64-byte rows with the 64-byte swizzle (8-row atoms,
// 512 bytes apart).
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

struct SplitShared {
  uint64_t full[SP_STAGES], empty[SP_STAGES];
  uint64_t hfull, hempty;  // hi.hi sums of a chunk ready / read
  uint64_t rfull, rempty;  // the other products' sums of a chunk ready / read
  uint64_t mma_idle;       // every MMA of the CTA has finished
  uint32_t tmem_base;
  int abort_flag, n_tiles;
  float2 ns[8][128];  // norm and scale of a warp's references
};

// static and dynamic share together: 227 KB
static_assert((sizeof(SplitShared) + 1023) / 1024 * 1024 + SpCfg<256>::kSmem <= 227 * 1024, "shared memory");

template <int SP_N>
__global__ void __launch_bounds__(SP_THREADS, 1)
gram_split_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapP, int nQ, int nP,
                  int capQ, int capP, int dk, const float* __restrict__ normQ, const float* __restrict__ normP,
                  const float* __restrict__ scaleQ, const float* __restrict__ scaleP, float neg_scale,
                  float* __restrict__ out, int64_t ldo, int* __restrict__ words, int look, uint32_t polls) {
  constexpr int SP_B_BYTES = SpCfg<SP_N>::kBBytes, SP_STAGE_BYTES = SpCfg<SP_N>::kStageBytes;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* const stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ SplitShared sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* const err = words + kSplitErr;
  const int tiles_m = (nQ + SP_M - 1) / SP_M, tiles_n = (nP + SP_N - 1) / SP_N;
  const int nk = (dk + SP_K - 1) / SP_K;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SP_STAGES; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    mbar_init(&sh.hfull, 1);
    mbar_init(&sh.hempty, 8);
    mbar_init(&sh.rfull, 1);
    mbar_init(&sh.rempty, 8);
    mbar_init(&sh.mma_idle, 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_base, SpCfg<SP_N>::kTmemCols);
    tmem_relinquish();
  }
  // nothing to do when a whole side is wide: every value is then the FFMA sums'
  // (not looked up where there is one tile a CTA: the reads are 1 us of 20)
  if (threadIdx.x == 64)
    sh.n_tiles = !look || (words[kSplitWideP] < nP && words[kSplitWideQ] < nQ) ? tiles_m * tiles_n : 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  const int n_tiles = sh.n_tiles;

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        const int tm = t % tiles_m, tn = t / tiles_m;
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(&sh.empty[s], ph ^ 1u, &sh.abort_flag, polls)) {
            ok = false;
            break;
          }
          uint8_t* const a = stages + (size_t)s * SP_STAGE_BYTES;
          uint8_t* const b = a + 3 * SP_A_BYTES;
          mbar_expect_tx(&sh.full[s], SP_STAGE_BYTES);
          // slice v of row r is row v * cap + r of the slice array
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            tma_load_2d(&mapQ, &sh.full[s], a + v * SP_A_BYTES, kb * SP_K, v * capQ + tm * SP_M);
            tma_load_2d(&mapP, &sh.full[s], b + v * SP_B_BYTES, kb * SP_K, v * capP + tn * SP_N);
          }
          if (++s == SP_STAGES) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        atomicExch(err, 1);
        sh.abort_flag = 1;
      }
      drain_copies(sh.full, SP_STAGES, s, ph, err);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    {
      const bool issuer = elect_one();
      int s = 0;
      uint32_t ph = 0, hph = 1, rph = 1;  // parities of the next "read" waits
      bool ok = true;
      const uint32_t idesc = sp_idesc(SP_N);
      const uint32_t dh = tmem, dr = tmem + SP_N;
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        for (int kb = 0; kb < nk; ++kb) {
          const bool first = kb % SP_CHUNK == 0, last = kb % SP_CHUNK == SP_CHUNK - 1 || kb == nk - 1;
          if (!mbar_wait_warp(&sh.full[s], ph, &sh.abort_flag, polls) ||
              (first && !mbar_wait_warp(&sh.rempty, rph, &sh.abort_flag, polls))) {
            ok = false;
            break;
          }
          if (first) rph ^= 1u;
          tc_fence_after();
          const uint32_t a = smem_u32(stages + (size_t)s * SP_STAGE_BYTES);
          const uint32_t b = a + 3 * SP_A_BYTES;
          if (issuer) {
#pragma unroll
            for (int k = 0; k < SP_K / 16; ++k) {
              const uint64_t ah = sw64_desc(a + k * 32), am = sw64_desc(a + SP_A_BYTES + k * 32),
                             al = sw64_desc(a + 2 * SP_A_BYTES + k * 32);
              const uint64_t bh = sw64_desc(b + k * 32), bm = sw64_desc(b + SP_B_BYTES + k * 32),
                             bl = sw64_desc(b + 2 * SP_B_BYTES + k * 32);
              umma_f16(dr, al, bh, idesc, !(first && k == 0));
              umma_f16(dr, ah, bl, idesc, 1);
              umma_f16(dr, am, bm, idesc, 1);
              umma_f16(dr, am, bh, idesc, 1);
              umma_f16(dr, ah, bm, idesc, 1);
            }
            if (last) umma_commit(&sh.rfull);
          }
          __syncwarp();
          if (first) {
            if (!mbar_wait_warp(&sh.hempty, hph, &sh.abort_flag, polls)) {
              ok = false;
              break;
            }
            hph ^= 1u;
            tc_fence_after();
          }
          if (issuer) {
#pragma unroll
            for (int k = 0; k < SP_K / 16; ++k)
              umma_f16(dh, sw64_desc(a + k * 32), sw64_desc(b + k * 32), idesc, !(first && k == 0));
            umma_commit(&sh.empty[s]);
            if (last) umma_commit(&sh.hfull);
          }
          __syncwarp();
          if (++s == SP_STAGES) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        if (issuer) atomicExch(err, 2);
        sh.abort_flag = 1;
      }
      if (issuer) drain_mmas(&sh.mma_idle, err);
    }
  } else {
    // ---------------- epilogue (warps 2..9)
    const int q = warp & 3, ew = warp - 2, half = ew >> 2;
    const uint32_t th = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * (SP_N / 2));
    const int chunks = (nk + SP_CHUNK - 1) / SP_CHUNK;
    uint32_t cph = 0;
    bool ok = true;
    // adds an accumulator's sums (when they are ready) to the totals and gives it back
    float tot[SP_N / 2];
    auto drain = [&](uint64_t* full, uint64_t* empty, int col) {
      if (lane == 0) ok = mbar_wait(full, cph, &sh.abort_flag, polls);
      ok = __shfl_sync(kFull, ok ? 1 : 0, 0) != 0;
      if (!ok) return;
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < SP_N / 2; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(th + (uint32_t)(col + c0), r);
#pragma unroll
        for (int c = 0; c < 32; ++c) tot[c0 + c] += __uint_as_float(r[c]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(empty);
    };
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
      const int tm = t % tiles_m, tn = t / tiles_m;
      const int n0 = tn * SP_N + half * (SP_N / 2);
      __syncwarp();
      for (int c = lane; c < SP_N / 2; c += 32) {
        const int n = n0 + c;
        sh.ns[ew][c] = n < nP ? make_float2(normP[n], scaleP[n]) : make_float2(0.0f, 0.0f);
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < SP_N / 2; ++c) tot[c] = 0.0f;
      for (int ch = 0; ch < chunks; ++ch) {
        drain(&sh.rfull, &sh.rempty, SP_N);
        if (ok) drain(&sh.hfull, &sh.hempty, 0);
        if (!ok) break;
        cph ^= 1u;
      }
      if (!ok) {
        if (lane == 0) {
          atomicExch(err, 3);
          sh.abort_flag = 1;
        }
        break;
      }
      const int m = tm * SP_M + q * 32 + lane;
      const int ncols = min(SP_N / 2, nP - n0);
      if (m < nQ) {
        const float nq = normQ[m], sq = scaleQ[m];
        float* o = out + (int64_t)n0 * ldo + m;
        auto value = [&](int c) {
          const float2 ns = sh.ns[ew][c];
          const float dot = tot[c] * sq * ns.y;
          return exp2f(fmaxf(nq + ns.x - 2.0f * dot, 0.0f) * neg_scale);
        };
        if (ncols >= SP_N / 2) {
#pragma unroll
          for (int c = 0; c < SP_N / 2; c += 8) {  // eight chains of exponentials at a time, then their stores
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = value(c + e);
#pragma unroll
            for (int e = 0; e < 8; ++e, o += ldo) st_global(o, v[e]);
          }
        } else {
#pragma unroll
          for (int c = 0; c < SP_N / 2; ++c, o += ldo)
            if (c < ncols) *o = value(c);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, SpCfg<SP_N>::kTmemCols);
  }
}

// ------------------------------------------------------------- row slices
// One warp per row of the two sets (references, then samples): the squared norm
// (when asked), the power-of-two scale and the three slices.
//
// A row whose values the slices do not hold as well as FP32 does is wide: it
// gets no slices, and its pairs come from the FFMA sums (launch_gram_wide).
// That is a row with NaN or Inf, one whose squared norm leaves the FP32 range
// (the scaled sums would meet it as Inf - Inf), and one whose largest value
// stands so far out that the products left out matter: against the FFMA
// kernel's error of about 0.8 units of 2^-24 (|p|^2 + |q|^2) they add
// 0.23 sqrt(2 d) 2^24 / |scaled row|^2, at most 0.08 from 2^26 sqrt(d) on (the
// largest value at most 11 to 21 times the root mean square at d = 784, 7 to 13
// times at d = 128).
// The slices stay at their rows' places (compacted, with the block's rows
// through a list, a 3,001 x 15,013 x 784 call took 375 instead of 360 us), so
// a block with wide rows pays for their tensor-core pairs as well, unless a whole
// side is wide.  That call with wide rows of values like the others' (host wait
// included): none 0.38 ms, one 0.49, 1 % 0.55, 10 % 0.86, half 1.71, 90 % 2.19,
// all 1.81; the FFMA kernel alone 1.67.
struct SplitSource {
  const float* X;
  int64_t ld, n, cap;
  __half* v;
  float *scale, *norm_out;
  const float* norm;
  int32_t* rows;
  int vec;  // 16-byte loads
};
static float wide_below(int64_t d) { return 0x1p26f * sqrtf((float)d); }

__global__ void __launch_bounds__(256)
split_rows_kernel(SplitSource P, SplitSource Q, int d, int ks, float least, int* __restrict__ words) {
  const int lane = threadIdx.x & 31;
  int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= P.n + Q.n) return;
  const bool sample = row >= P.n;
  if (sample) row -= P.n;
  const SplitSource S = sample ? Q : P;
  const float* x = S.X + row * S.ld;
  auto load4 = [&](int c) -> float4 {  // values c..c+3, zero past d
    if (S.vec) return c < d ? __ldg(reinterpret_cast<const float4*>(x + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
    return make_float4(c < d ? __ldg(x + c) : 0.f, c + 1 < d ? __ldg(x + c + 1) : 0.f,
                       c + 2 < d ? __ldg(x + c + 2) : 0.f, c + 3 < d ? __ldg(x + c + 3) : 0.f);
  };
  float norm = S.norm ? __ldg(S.norm + row) : 0.0f;
  float2 acc = make_float2(0.0f, 0.0f);
  uint32_t top = 0;  // the largest |value|, as an integer (NaN and Inf sort above)
  for (int c = lane * 4; c < d; c += 128) {
    const float4 v = load4(c);
    top = max(max(top, max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu)),
              max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu));
    if (!S.norm) acc = df_add_sq(df_add_sq(df_add_sq(df_add_sq(acc, v.x), v.y), v.z), v.w);
  }
  top = __reduce_max_sync(kFull, top);
  if (!S.norm) {
    norm = __shfl_sync(kFull, df_to_float(warp_sum_df(acc)), 0);  // one answer for the warp
    if (lane == 0) S.norm_out[row] = norm;
  }
  // scaled maximum in [2^14, 2^15); the exponents stay within the normal range
  const int up = min(141 - (int)(top >> 23), 126);  // 14 - (e - 127), e biased (0: zero or subnormal)
  const float s = __uint_as_float((uint32_t)(127 + up) << 23);
  const float scaled = norm * s * s;
  const bool wide = top != 0 && !(scaled >= least && scaled <= 3.4028235e38f);
  if (lane == 0) {
    S.scale[row] = wide ? 0.0f : __uint_as_float((uint32_t)(127 - up) << 23);  // (0 marks it for the lists)
    if (wide) {
      const int at = atomicAdd(words + (sample ? kSplitWideQ : kSplitWideP), 1);
      if (sample) S.rows[at] = (int32_t)row;
    }
  }
  if (wide) return;  // (its slices would enter its own pairs only, which are written again)
  __half* const o = S.v + row * ks;
  const int64_t slice = S.cap * (int64_t)ks;
  for (int c = lane * 4; c < ks; c += 128) {
    const float4 v = load4(c);
    const float t[4] = {v.x * s, v.y * s, v.z * s, v.w * s};
    __half h[3][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float hi = rintf(t[q] * 0x1p-7f) * 0x1p7f;
      const float r1 = t[q] - hi;  // exact
      const __half mid = __float2half_rn(r1);
      h[0][q] = __float2half_rn(hi);
      h[1][q] = mid;
      h[2][q] = __float2half_rn(r1 - __half2float(mid));  // an exact difference
    }
#pragma unroll
    for (int w = 0; w < 3; ++w) *reinterpret_cast<uint2*>(o + w * slice + c) = *reinterpret_cast<const uint2*>(h[w]);
  }
}

static cudaError_t launch_split_rows(const SplitSide& P, const SplitBufs& bP, int64_t nP, const SplitSide& Q,
                                     const SplitBufs& bQ, int64_t nQ, int64_t d, int ks, int* words, cudaStream_t st) {
  if (nP + nQ <= 0) return cudaSuccess;
  auto source = [&](const SplitSide& r, const SplitBufs& b, int64_t n) {
    const int vec = d % 4 == 0 && r.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(r.X) & 15) == 0;
    return SplitSource{r.X, r.ld, n, b.cap, b.v, b.scale, b.norm, r.norm, b.rows, vec};
  };
  split_rows_kernel<<<(unsigned)ceil_div(nP + nQ, 8), 256, 0, st>>>(source(P, bP, nP), source(Q, bQ, nQ), (int)d, ks,
                                                                    wide_below(d), words);
  return cudaGetLastError();
}

// The references without slices and the others, listed from the scales.  A pass
// of its own, run only before launch_gram_wide: appending every reference as its
// slices are cut cost 4 us of a call of 95.
__global__ void __launch_bounds__(256)
split_list_kernel(const float* __restrict__ scale, int n, int32_t* __restrict__ rows, int* __restrict__ words) {
  if (words[kSplitWideP] == 0) return;  // (row a is the a-th of the others)
  const int r = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31;
  const bool wide = r < n && scale[r] == 0.0f;
  const unsigned w = __ballot_sync(kFull, wide), c = __ballot_sync(kFull, r < n && !wide);
  int at = 0;
  if (lane == 0 && c) at = atomicAdd(words + kSplitListed, __popc(c));
  if (lane == 1 && w) at = atomicAdd(words + kSplitWideListed, __popc(w));
  const int c0 = __shfl_sync(kFull, at, 0), w0 = __shfl_sync(kFull, at, 1);
  const unsigned below = (1u << lane) - 1;
  if (wide) rows[n - 1 - (w0 + __popc(w & below))] = r;
  else if (r < n) rows[c0 + __popc(c & below)] = r;
}
cudaError_t launch_split_list(SplitScratch& t, int64_t nP, cudaStream_t st) {
  if (nP <= 0 || t.listed) return cudaSuccess;
  t.listed = true;
  split_list_kernel<<<(unsigned)ceil_div(nP, 256), 256, 0, st>>>(t.P.scale, (int)nP, t.P.rows, t.words);
  return cudaGetLastError();
}

// 2-D map of a slice array [3 n][ks], box = 32 values x box_rows, 64-byte swizzle.
static bool split_map(CUtensorMap* map, const __half* base, int64_t n, int ks, int box_rows) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)ks, (cuuint64_t)(3 * n)};
  cuuint64_t strides[1] = {(cuuint64_t)(ks * 2)};
  cuuint32_t box[2] = {SP_K, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static cudaError_t launch_gram_split(const SplitBufs& bP, const float* normP, int64_t nP, const SplitBufs& bQ,
                                     const float* normQ, int64_t nQ, int ks, float neg_scale, float* out, int64_t ldo,
                                     int* words, int n_sms, cudaStream_t st, uint32_t polls) {
  if (ks % 8 != 0 || (reinterpret_cast<uintptr_t>(bP.v) & 15) || (reinterpret_cast<uintptr_t>(bQ.v) & 15) ||
      nP > bP.cap || nQ > bQ.cap || 3 * bP.cap > INT32_MAX || 3 * bQ.cap > INT32_MAX)
    return cudaErrorInvalidValue;
  alignas(64) CUtensorMap mq, mp;
#define KKM_SPLIT_LAUNCH(N)                                                                                    \
  do {                                                                                                         \
    if (!split_map(&mq, bQ.v, bQ.cap, ks, SP_M) || !split_map(&mp, bP.v, bP.cap, ks, N))                       \
      return cudaErrorInvalidValue;                                                                            \
    const cudaError_t attr = cudaFuncSetAttribute(                                                             \
        gram_split_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SpCfg<N>::kSmem);              \
    if (attr != cudaSuccess) return attr;                                                                      \
    const int64_t tiles = ceil_div(nQ, SP_M) * ceil_div(nP, N);                                                \
    gram_split_kernel<N><<<(unsigned)std::min<int64_t>(tiles, std::max(n_sms, 1)), SP_THREADS, SpCfg<N>::kSmem, st>>>( \
        mq, mp, (int)nQ, (int)nP, (int)bQ.cap, (int)bP.cap, ks, normQ, normP, bQ.scale, bP.scale, neg_scale, out, ldo, \
        words, tiles > n_sms, polls);                                                                                         \
  } while (0)
  if (2 * ceil_div(nQ, SP_M) * ceil_div(nP, 256) <= n_sms) KKM_SPLIT_LAUNCH(64);
  else KKM_SPLIT_LAUNCH(256);
#undef KKM_SPLIT_LAUNCH
  return cudaGetLastError();
}

kkm_status split_block(SplitScratch& t, const SplitSide& P, int64_t nP, const SplitSide& Q, int64_t nQ, int64_t d,
                       int dp, float neg_scale, float* out, int64_t ldo, bool p_ready, bool q_ready, int n_sms,
                       cudaStream_t st, uint32_t polls) {
  if (nP <= 0 || nQ <= 0) return KKM_OK;
  // the error word lasts, the counts start anew with their side
  const int from = t.fresh ? kSplitErr : q_ready ? kSplitWideP : kSplitWideQ, to = p_ready ? kSplitWideP : kSplitWords;
  if (from < to) {
    KKM_CK(cudaMemsetAsync(t.words + from, 0, 4 * (to - from), st));
    t.fresh = false;
    if (!p_ready) t.listed = false;
    KKM_RUN("split_rows", st,
            launch_split_rows(P, t.P, p_ready ? 0 : nP, Q, t.Q, q_ready ? 0 : nQ, d, dp, t.words, st));
  }
  KKM_RUN("gram_split", st,
          launch_gram_split(t.P, P.norm ? P.norm : t.P.norm, nP, t.Q, Q.norm ? Q.norm : t.Q.norm, nQ, dp, neg_scale, out,
                            ldo, t.words, n_sms, st, polls));
  return KKM_OK;
}

kkm_status split_wide_pairs(SplitScratch& t, const SplitSide& P, int64_t nP, const SplitSide& Q, int64_t nQ, int64_t d,
                            int dp, float neg_scale, float* out, int64_t ldo, int n_sms, cudaStream_t st) {
  KKM_RUN("split_list", st, launch_split_list(t, nP, st));
  KKM_RUN("gram_wide", st, launch_gram_wide(t, P, nP, Q, nQ, d, dp, neg_scale, out, ldo, n_sms, st));
  return KKM_OK;
}

// out[a][b] = out[b][a] for a > b: the matrix of a set with itself.  The second
// accumulator adds lo.hi before hi.lo, so an entry and its mirror image may
// differ in their last bit, which no other kernel block does.  32 x 32 tiles
// through shared memory: 3,000 x 3,000 take 10 us.
__global__ void __launch_bounds__(256)
mirror_kernel(float* __restrict__ out, int n, int64_t ldo) {
  __shared__ float t[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;  // the tile read, on or above the diagonal
  if (r0 > c0) return;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int r = y; r < 32; r += 8)
    if (r0 + r < n && c0 + x < n) t[r][x] = out[(int64_t)(r0 + r) * ldo + c0 + x];
  __syncthreads();
  for (int r = y; r < 32; r += 8) {
    const int a = c0 + r, b = r0 + x;
    if (a < n && a > b) out[(int64_t)a * ldo + b] = t[x][r];
  }
}
cudaError_t launch_mirror(float* out, int64_t n, int64_t ldo, cudaStream_t st) {
  const int64_t tiles = ceil_div(n, 32);
  if (n <= 0) return cudaSuccess;
  if (tiles > 65535) return cudaErrorInvalidValue;
  mirror_kernel<<<dim3((unsigned)tiles, (unsigned)tiles), 256, 0, st>>>(out, (int)n, ldo);
  return cudaGetLastError();
}

}  // namespace kkm
