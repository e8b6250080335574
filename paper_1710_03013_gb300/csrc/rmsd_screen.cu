// The MD kernel's screen on the tensor cores (tcgen05): the 3 x 3 correlation
// of every pair of frames, and from it whether the pair is certainly far.
//
// P (references) and Q (samples) hold centred frames as rows of split BF16:
// row 3 f + c is plane c of frame f, three segments of kp values ((hi, lo, hi)
// on the reference side, (hi, hi, lo) on the sample side), so that the product
// over K = 3 kp is the correlation to ~1e-5 relative.  A tile is 40 samples x
// 80 references: M = 128 (each tensor-memory lane quarter takes 30 rows, ten
// whole samples, so a warp's lanes hold whole pairs; two rows of a quarter are
// unused), N = 240.  For sample s and reference l the accumulator's 3 x 3
// block at rows 3 s.., columns 3 l.. is H^T.
//
// Epilogue (16 warps): lane 3 s + j of a warp reads row j of sample s for
// three references (nine columns), the warp regroups them through shared
// memory (rows of nine floats), and lane 3 s + i gets the whole correlation of
// reference i.  Then a sign test of the QCP polynomial certifies the pair
// beyond the refine threshold, or the pair gets a bit in `near` and the
// optimal rotation (a unit quaternion) for the exact pass.  The block and the
// bits are zeroed beforehand: a certified pair's value is 0.
//
// What bounds it: the epilogue's instructions, about 300 for 30 pairs (ncu: 0.6
// issued a cycle and scheduler, tensor pipe 38 % active); with the far test
// taken out the rest runs in 1.28 ms of the figures below.  10,000 x 10,000
// frames of 300 atoms: 1.71 ms, 1,250 references x 25,000 samples 0.55 ms.
// Before, 2.47 and 0.81 ms: frames in four planes (x, y, z, 0), tiles of 32 x
// 64 frames (1.6 times the operand bytes and products a pair), eight epilogue
// warps.  Tried: eight warps here 3.0 ms, twenty 1.77, the regrouping by
// shuffles 1.95, near pairs queued so that rotations fill whole warps 2.0 (the
// queue takes a stage of the ring).
// The sums of each correlation entry are the same products in the same order.
//
// Every mbarrier wait is bounded, and a CTA ends only when its copies and MMAs
// have, as in the BF16 block (gram_tc.cu).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "qcp.cuh"
#include "tc_common.cuh"

namespace kkm {

constexpr int SC_M = 128, SC_N = 240;
constexpr int SC_FQ = 40, SC_FP = 80;            // samples and references of a tile
constexpr int SC_K = 64;                         // K values per stage (one 128-byte swizzle row)
constexpr int SC_STAGES = 4;
constexpr int SC_A_BYTES = SC_M * SC_K * 2;
constexpr int SC_B_BYTES = SC_N * SC_K * 2;
constexpr int SC_STAGE_BYTES = SC_A_BYTES + SC_B_BYTES;
constexpr int SC_TX_BYTES = (4 * 30 + SC_N) * SC_K * 2;
constexpr int SC_EPI = 16;                       // epilogue warps
constexpr int SC_THREADS = 64 + 32 * SC_EPI;
constexpr int SC_PART = SC_FP / (SC_EPI / 4);    // references of an epilogue warp
constexpr size_t SC_SMEM = (size_t)SC_STAGES * SC_STAGE_BYTES + 1024 + SC_EPI * 32 * 9 * sizeof(float);
static_assert(SC_STAGE_BYTES % 1024 == 0 && SC_A_BYTES % 1024 == 0, "swizzle atoms");

// kind::f16, FP32 accumulator, BF16 A and B, both K-major.
__host__ __device__ constexpr uint32_t sc_idesc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SC_N >> 3) << 17) | ((uint32_t)(SC_M >> 4) << 24);
}

__device__ __forceinline__ void tmem_ld9(uint32_t taddr, float (&v)[9]) {
  uint32_t r[9];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[8]) : "r"(taddr + 8));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int q = 0; q < 9; ++q) v[q] = __uint_as_float(r[q]);
}

// Tile t: bands of SC_BAND reference tiles, sample tiles within a band, so that
// CTAs running side by side share sample rows as well as references.
constexpr int SC_BAND = 4;
__device__ __forceinline__ void screen_tile(int64_t t, int tiles_m, int tiles_n, int& tm, int& tn) {
  const int64_t per = (int64_t)SC_BAND * tiles_m;
  const int band = (int)(t / per), r = (int)(t - band * per), w = min(SC_BAND, tiles_n - band * SC_BAND);
  tm = r / w;
  tn = band * SC_BAND + r % w;
}

struct ScreenShared {
  uint64_t full[SC_STAGES], empty[SC_STAGES];
  uint64_t tfull[2], tempty[2];
  uint64_t mma_idle;  // every MMA of the CTA has finished
  uint32_t tmem_base;
  int abort_flag;
};

// LIMITED: waits of `polls` polls, for tests.  A limit in a register instead of a
// constant costs 1.5 % (1.736 ms against 1.709, 10,000 x 10,000 frames of 300 atoms).
template <bool LIMITED>
__global__ void __launch_bounds__(SC_THREADS, 1)
rmsd_screen_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapP, int nQ, int nP,
                   int dk, const float* __restrict__ gQ, const float* __restrict__ gP, float n_r2_far,
                   float4* __restrict__ quat, int64_t ldo, uint32_t* __restrict__ near, int64_t pitch_words,
                   int* __restrict__ err, uint32_t polls) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* const stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ ScreenShared sh;
  const uint32_t limit = LIMITED ? polls : kTcSpinLimit;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = (nQ + SC_FQ - 1) / SC_FQ, tiles_n = (nP + SC_FP - 1) / SC_FP;
  const int64_t n_tiles = (int64_t)tiles_m * tiles_n;
  const int nk = dk / SC_K;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SC_STAGES; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sh.tfull[b], 1);
      mbar_init(&sh.tempty[b], SC_EPI);
    }
    mbar_init(&sh.mma_idle, 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        int tm, tn;
      screen_tile(t, tiles_m, tiles_n, tm, tn);
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(&sh.empty[s], ph ^ 1u, &sh.abort_flag, limit)) {
            ok = false;
            break;
          }
          uint8_t* const a = stages + (size_t)s * SC_STAGE_BYTES;
          mbar_expect_tx(&sh.full[s], SC_TX_BYTES);
#pragma unroll
          for (int q = 0; q < 4; ++q)  // ten samples to a lane quarter
            tma_load_2d(&mapQ, &sh.full[s], a + q * 32 * SC_K * 2, kb * SC_K, tm * 3 * SC_FQ + q * 30);
          tma_load_2d(&mapP, &sh.full[s], a + SC_A_BYTES, kb * SC_K, tn * SC_N);
          if (++s == SC_STAGES) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok) {
        atomicExch(err, 1);
        sh.abort_flag = 1;
      }
      drain_copies(sh.full, SC_STAGES, s, ph, err);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int s = 0, lt = 0;
      uint32_t ph = 0;
      bool ok = true;
      const uint32_t idesc = sc_idesc();
      for (int64_t t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++lt) {
        const int buf = lt & 1;
        if (!mbar_wait(&sh.tempty[buf], ((uint32_t)(lt >> 1) & 1u) ^ 1u, &sh.abort_flag, limit)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem + (uint32_t)(buf * 256);
        for (int kb = 0; kb < nk; ++kb) {
          if (!mbar_wait(&sh.full[s], ph, &sh.abort_flag, limit)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a = smem_u32(stages + (size_t)s * SC_STAGE_BYTES);
          const uint32_t b = a + SC_A_BYTES;
#pragma unroll
          for (int k = 0; k < SC_K / 16; ++k)
            umma_bf16(d_tmem, sw128_desc(a + k * 32), sw128_desc(b + k * 32), idesc, (kb | k) != 0);
          umma_commit(&sh.empty[s]);
          if (++s == SC_STAGES) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok) umma_commit(&sh.tfull[buf]);
      }
      if (!ok) {
        atomicExch(err, 2);
        sh.abort_flag = 1;
      }
      drain_mmas(&sh.mma_idle, err);
    }
  } else {
    // ---------------- epilogue
    const int q = warp & 3, part = (warp - 2) >> 2;
    const int ps = lane / 3, i = lane - 3 * ps;  // sample of the quarter; own row, then own reference of three
    float* const xs = reinterpret_cast<float*>(stages + (size_t)SC_STAGES * SC_STAGE_BYTES) + (warp - 2) * 32 * 9;
    const float* const mine = xs + min(ps, 9) * 27 + 3 * i;
    int lt = 0;
    for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x, ++lt) {
      int tm, tn;
      screen_tile(t, tiles_m, tiles_n, tm, tn);
      const int buf = lt & 1;
      const int sf = tm * SC_FQ + q * 10 + ps;
      const bool valid = ps < 10 && sf < nQ;
      const float gy = valid ? gQ[sf] : 0.0f;
      bool ok = true;
      __syncwarp();
      if (lane == 0) ok = mbar_wait(&sh.tfull[buf], (uint32_t)(lt >> 1) & 1u, &sh.abort_flag, limit);
      ok = __shfl_sync(kFull, ok ? 1 : 0, 0) != 0;
      if (!ok) {
        if (lane == 0) {
          atomicExch(err, 3);
          sh.abort_flag = 1;
        }
        break;
      }
      tc_fence_after();
      const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 256 + part * SC_PART * 3);
#pragma unroll 1
      for (int g = 0; g < SC_PART; g += 3) {
        float v[9], H[9];  // v[3 l + c] = component c of reference l against the lane's own row
        tmem_ld9(tb + (uint32_t)(3 * g), v);
        // H[c1][c2] = sum_a x_a[c1] y_a[c2] of reference i, x the reference frame
#pragma unroll
        for (int c = 0; c < 9; ++c) xs[lane * 9 + c] = v[c];
        __syncwarp();
#pragma unroll
        for (int c1 = 0; c1 < 3; ++c1)
#pragma unroll
          for (int c2 = 0; c2 < 3; ++c2) H[3 * c1 + c2] = mine[9 * c2 + c1];
        __syncwarp();
        const int l = g + i, lf = tn * SC_FP + part * SC_PART + l;
        if (valid && l < SC_PART && lf < nP) {
          const float gx = gP[lf];
          if (!qcp_certainly_far(H, gx, gy, n_r2_far)) {
            float qv[4];
            qcp_quaternion(H, gx, gy, qv);
            quat[(int64_t)lf * ldo + sf] = make_float4(qv[0], qv[1], qv[2], qv[3]);
            atomicOr(near + (int64_t)lf * pitch_words + (sf >> 5), 1u << (sf & 31));
          }
        }
        __syncwarp();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.tempty[buf]);
    }
  }
  // teardown: every role is done issuing; the TMEM owner frees tensor memory
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// 2-D map of split rows [3 n][dk], box = box_rows x 128 bytes, 128-byte swizzle.
static bool screen_map(CUtensorMap* map, const __nv_bfloat16* base, int64_t n, int dk, int box_rows) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)dk, (cuuint64_t)(3 * n)};
  cuuint64_t strides[1] = {(cuuint64_t)(dk * 2)};
  cuuint32_t box[2] = {SC_K, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_rmsd_screen(const __nv_bfloat16* P, int64_t nP, const __nv_bfloat16* Q, int64_t nQ, int dk,
                               const float* gP, const float* gQ, int n_atoms, float neg_scale, float* out,
                               float4* quat, uint8_t* near, int64_t pitch, int64_t ldo, int* err, int n_sms,
                               cudaStream_t st, uint32_t polls) {
  if (nP <= 0 || nQ <= 0) return cudaSuccess;
  if (dk % SC_K != 0 || (reinterpret_cast<uintptr_t>(P) & 15) || (reinterpret_cast<uintptr_t>(Q) & 15) || n_atoms <= 0 ||
      !quat || !near || pitch % 16 != 0 || 8 * pitch < nQ || 3 * (nP + SC_FP) > INT32_MAX || 3 * (nQ + SC_FQ) > INT32_MAX)
    return cudaErrorInvalidValue;
  alignas(64) CUtensorMap mq, mp;
  if (!screen_map(&mq, Q, nQ, dk, 30) || !screen_map(&mp, P, nP, dk, SC_N)) return cudaErrorInvalidValue;
  auto* const kernel = polls == kTcSpinLimit ? rmsd_screen_kernel<false> : rmsd_screen_kernel<true>;
  const cudaError_t attr = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SC_SMEM);
  if (attr != cudaSuccess) return attr;
  cudaError_t e = ldo == nQ ? cudaMemsetAsync(out, 0, (size_t)nP * nQ * 4, st)
                            : cudaMemset2DAsync(out, (size_t)ldo * 4, 0, (size_t)nQ * 4, (size_t)nP, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(near, 0, (size_t)(nP * pitch), st);
  if (e != cudaSuccess) return e;
  // n rmsd^2 at which the kernel value falls to kRmsdRefine
  const float n_r2_far = (log2f(kRmsdRefine) / neg_scale) / (1.0f / (float)n_atoms);
  const int64_t tiles = ceil_div(nQ, SC_FQ) * ceil_div(nP, SC_FP);
  kernel<<<(unsigned)std::min<int64_t>(tiles, std::max(n_sms, 1)), SC_THREADS, SC_SMEM, st>>>(
      mq, mp, (int)nQ, (int)nP, dk, gQ, gP, n_r2_far, quat, ldo, reinterpret_cast<uint32_t*>(near), pitch / 4, err,
      polls);
  return cudaGetLastError();
}

}  // namespace kkm
