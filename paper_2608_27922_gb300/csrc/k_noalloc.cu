// dkv_candidate_order_noalloc: candidate scoring and ordering for callers that
// cannot allocate device memory.
//
// The regular path (dkv_bank_admit) keeps its intermediates in a workspace the
// caller allocates.  Some callers cannot allocate at all: code that runs inside a
// framework that owns every device byte through its own pool, real-time or
// embedded hosts where allocation is forbidden after start-up, or plugins that only
// receive pre-sized input and output buffers.  This entry point needs nothing but
// the caller's inputs and outputs: the one scratch buffer it uses (the per-
// candidate scores between the scoring kernel and the ordering kernel) is the
// file-scope device array below, of a fixed size.
//
// The scoring kernel is the fp32 direct-difference variant of the Eq. 6 pass for
// one head, on the tiled pair code of the fp32 score mode of dkv_bank_admit
// (simt_pairs.cuh), whose sums have one order for any tile size; one division by m.
// Its scores are therefore bit-identical to admit's in that mode.  The ordering
// kernel places every candidate at the number of candidates that come before it
// (smaller score, or equal score and smaller source index): the stable ascending
// order, without a buffer to sort in and over as many blocks as there are candidates.
// Measured at 2,070 MHz, d = 128, bf16, 9,360 bank keys x 4,680 candidates: the
// whole call 4,885 us before (one thread per candidate, one block sorting) -> 531.
#include "../../include/dkv.h"
#include "dkv_internal.h"
#include "simt_pairs.cuh"

#include <climits>
#include <cmath>
#include <mutex>

namespace dkv {
namespace {

// Score of a candidate whose sum a hand-over never reached (simt::Chain): a NaN that no
// arithmetic returns (results are 0x7fffffff), so it is told from a NaN of the inputs.  Written
// and recognised as integers only (nvcc 13.0 took a float compared with it bit by bit for it
// whenever the float was any NaN).
constexpr uint32_t NO_SCORE = 0xfffffffeu, NO_SCORE_KEY = ~NO_SCORE;   // (key: fkey's)

// Scratch shared by every call on a device, held until the process exits.
static __device__ __align__(256) float g_noalloc_scores[DKV_NOALLOC_MAX_N];

template <typename T, int D, int RT>
__global__ void __launch_bounds__(simt::NT) noalloc_score(const T* Kb, const float* base, int m, const T* Kc, int N,
                                                          KParams kp, bool vec, int cluster, float* scratch) {
  extern __shared__ __align__(16) float smem[];
  __shared__ int4 mail[RT];
  const int C = cluster, z = blockIdx.x % C;   // the cluster is C neighbouring blocks
  const int row0 = blockIdx.x / C * RT;
  const int sr = simt::scan_row<RT>();
  simt::Chain<RT> chain(mail, z, C, (m + simt::CT - 1) / simt::CT);
  float acc = 0.f;
  int lost = 0;
  simt::pair_tiles<T, D, false, RT>(Kc, nullptr, row0, N, Kb, nullptr, base, 0, m, kp, vec, smem, z, C,
                                    [&](int t0, int nc, const float* w, const float* inv) {
                                      const int t = t0 / simt::CT;
                                      chain.take(sr, t, acc, lost);
                                      simt::for_columns(nc, w, [&](int c, float x) { acc = __fmaf_rn(x, inv[c], acc); });
                                      chain.give(sr, t, acc, lost);
                                    });
  chain.finish();
  if (chain.last() && sr >= 0 && row0 + sr < N)
    reinterpret_cast<uint32_t*>(scratch)[row0 + sr] = lost != chain.LOST ? __float_as_uint(__fdiv_rn(acc, (float)m)) : NO_SCORE;
}

// Block b places candidates [32 b, 32 b + 32): thread (i, g) = (t % 32, t / 32) counts, for
// candidate i, those that come before it among every 8th run of ORD_RUN candidates; the
// eight counts are added through shared memory.  Every block sees every score: if one is
// missing (NO_SCORE) there is no order, and all of them write -1.  2 N^2 / 32 warp comparisons in all: at
// N = 16,384 about 8 M a phase, less than the single block of a sort in shared memory took
// for its 91 to 105 barrier-separated exchange phases.
constexpr int ORD_RUN = 256;
constexpr int ORD_GROUPS = 8;

__global__ void __launch_bounds__(32 * ORD_GROUPS) noalloc_order(const float* scratch, int N, int m, int32_t* perm,
                                                                 float* scores) {
  __shared__ __align__(16) uint32_t keys[ORD_GROUPS][ORD_RUN];
  __shared__ int s_cnt[ORD_GROUPS][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  if (m == 0) {   // empty bank: source order (Alg. 1, m = 0 branch)
    if (g == 0 && i < N) {
      perm[i] = i;
      if (scores) scores[i] = 0.f;
    }
    return;
  }
  const float mine = i < N ? scratch[i] : 0.f;
  const uint32_t key = fkey(mine);
  int cnt = 0;
  bool missing = false;
  for (int r0 = g * ORD_RUN; r0 < N; r0 += ORD_GROUPS * ORD_RUN) {   // warp-uniform
    const int n = min(ORD_RUN, N - r0);
    for (int k = lane; k < n; k += 32) {
      const uint32_t x = fkey(scratch[r0 + k]);
      missing = missing || x == NO_SCORE_KEY;
      keys[g][k] = x;
    }
    __syncwarp();
    // candidates of the run before index i precede it at equal scores
    const int below = min(max(i - r0, 0), n);
    if (n == ORD_RUN && (below == 0 || below == n)) {
      if (below) {
#pragma unroll 8
        for (int k = 0; k < ORD_RUN; k += 4) {
          const uint4 x = *reinterpret_cast<const uint4*>(&keys[g][k]);
          cnt += (x.x <= key) + (x.y <= key) + (x.z <= key) + (x.w <= key);
        }
      } else {
#pragma unroll 8
        for (int k = 0; k < ORD_RUN; k += 4) {
          const uint4 x = *reinterpret_cast<const uint4*>(&keys[g][k]);
          cnt += (x.x < key) + (x.y < key) + (x.z < key) + (x.w < key);
        }
      }
    } else {
      for (int k = 0; k < n; ++k) cnt += k < below ? keys[g][k] <= key : keys[g][k] < key;
    }
    __syncwarp();
  }
  s_cnt[g][lane] = cnt;
  missing = __syncthreads_or(missing);
  if (g == 0 && i < N) {
    int pos = 0;
#pragma unroll
    for (int q = 0; q < ORD_GROUPS; ++q) pos += s_cnt[q][lane];
    // (keys with their index are distinct: positions cover [0, N))
    if (missing) perm[i] = -1;
    else perm[pos] = i;
    if (scores) scores[i] = mine;
  }
}

template <typename T, int D, int RT>
cudaError_t launch_score(const void* Kb, const float* base, int m, const void* Kc, int N, const KParams& kp,
                         int C, float* scratch, cudaStream_t s) {
  // this entry point asks no alignment of its key arrays beyond the element's
  const bool vec = ((reinterpret_cast<uintptr_t>(Kb) | reinterpret_cast<uintptr_t>(Kc)) & 15u) == 0;
  return launch_kernel(noalloc_score<T, D, RT>, dim3((N + RT - 1) / RT * C), simt::NT, simt::Lay<D, false, RT>::SMEM, C,
                       false, s, static_cast<const T*>(Kb), base, m, static_cast<const T*>(Kc), N, kp, vec, C, scratch);
}

template <typename T, int D>
cudaError_t launch_score(const void* Kb, const float* base, int m, const void* Kc, int N, const KParams& kp,
                         float* scratch, cudaStream_t s) {
  const simt::Shape p = simt::pick_shape(1, N, m, D, sm_count(), true);
  return p.rows == 64   ? launch_score<T, D, 64>(Kb, base, m, Kc, N, kp, p.cluster, scratch, s)
         : p.rows == 32 ? launch_score<T, D, 32>(Kb, base, m, Kc, N, kp, p.cluster, scratch, s)
                        : launch_score<T, D, 16>(Kb, base, m, Kc, N, kp, p.cluster, scratch, s);
}

// Set-up per device, with that device current: the device address of the scratch
// array (in host code the array's name is only a host-side stand-in) and the
// shared-memory opt-in of the scoring kernels.  Only a complete success is kept; a
// failed attempt leaves nothing behind, so the next call on that device tries again.
constexpr int kMaxDevices = 64;
struct DeviceSetup {
  bool ready = false;
  float* scratch = nullptr;
};
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mu;

cudaError_t setup_device(int dev, float** scratch) {
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mu);
  DeviceSetup& s = g_setup[dev];
  if (!s.ready) {
    void* p = nullptr;
    cudaError_t err = cudaGetSymbolAddress(&p, g_noalloc_scores);
    auto opt_in = [&](auto k, size_t bytes) {
      if (err == cudaSuccess) err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    opt_in(noalloc_score<__nv_bfloat16, 128, 64>, simt::Lay<128, false, 64>::SMEM);
    opt_in(noalloc_score<__nv_bfloat16, 128, 32>, simt::Lay<128, false, 32>::SMEM);
    opt_in(noalloc_score<__nv_bfloat16, 128, 16>, simt::Lay<128, false, 16>::SMEM);
    opt_in(noalloc_score<__nv_bfloat16, 64, 64>, simt::Lay<64, false, 64>::SMEM);
    opt_in(noalloc_score<__nv_bfloat16, 64, 32>, simt::Lay<64, false, 32>::SMEM);
    opt_in(noalloc_score<__nv_bfloat16, 64, 16>, simt::Lay<64, false, 16>::SMEM);
    opt_in(noalloc_score<float, 128, 64>, simt::Lay<128, false, 64>::SMEM);
    opt_in(noalloc_score<float, 128, 32>, simt::Lay<128, false, 32>::SMEM);
    opt_in(noalloc_score<float, 128, 16>, simt::Lay<128, false, 16>::SMEM);
    opt_in(noalloc_score<float, 64, 64>, simt::Lay<64, false, 64>::SMEM);
    opt_in(noalloc_score<float, 64, 32>, simt::Lay<64, false, 32>::SMEM);
    opt_in(noalloc_score<float, 64, 16>, simt::Lay<64, false, 16>::SMEM);
    if (err != cudaSuccess) {
      (void)cudaGetLastError();   // do not leave the failure to the next unrelated check
      return err;
    }
    s.scratch = static_cast<float*>(p);
    s.ready = true;
  }
  *scratch = s.scratch;
  return cudaSuccess;
}

}  // namespace
}  // namespace dkv

extern "C" dkv_status_t dkv_candidate_order_noalloc(const void* K_bank, const float* base, int32_t m,
                                                    const void* Kc, int32_t N, int32_t d, int32_t dtype,
                                                    const dkv_params_t* params, float* scores_out,
                                                    int32_t* perm_out, void* stream) {
  using namespace dkv;
  if (!Kc || !perm_out || !params || (m > 0 && (!K_bank || !base))) return DKV_ERR_ARG;
  if (dtype != DKV_DTYPE_BF16 && dtype != DKV_DTYPE_FP32) return DKV_ERR_ARG;
  if (N < 1 || N > DKV_NOALLOC_MAX_N || m < 0 || m > 262144 || (d != 64 && d != 128)) return DKV_ERR_SHAPE;
  const dkv_params_t& p = *params;
  if (!(p.tau > 1.0f) || !(p.eps > 0.0f) || !(p.delta > 0.0f) || !(p.sigma >= 0.0f) ||
      !(p.p == 1.0f || p.p == 2.0f || p.p == 4.0f) || !std::isfinite(p.sigma) || !std::isfinite(p.eps))
    return DKV_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DKV_ERR_CUDA;
  float* scratch = nullptr;
  if (setup_device(dev, &scratch) != cudaSuccess) return DKV_ERR_CUDA;
  const float sg = p.sigma > 0.0f ? p.sigma : std::sqrt((float)d / 2.0f);
  KParams kp{};
  kp.inv_s2 = 1.0f / (sg * sg);
  kp.eps = p.eps;
  kp.tau = p.tau;
  kp.delta = p.delta;
  kp.p = (int)p.p;
  kp.sync_heads = 1;
  cudaStream_t s = (cudaStream_t)stream;
  if (m > 0) {
    cudaError_t e;
    if (dtype == DKV_DTYPE_BF16)
      e = d == 128 ? launch_score<__nv_bfloat16, 128>(K_bank, base, m, Kc, N, kp, scratch, s)
                   : launch_score<__nv_bfloat16, 64>(K_bank, base, m, Kc, N, kp, scratch, s);
    else
      e = d == 128 ? launch_score<float, 128>(K_bank, base, m, Kc, N, kp, scratch, s)
                   : launch_score<float, 64>(K_bank, base, m, Kc, N, kp, scratch, s);
    if (e != cudaSuccess) return DKV_ERR_CUDA;
  }
  noalloc_order<<<(N + 31) / 32, 32 * ORD_GROUPS, 0, s>>>(scratch, N, m, perm_out, scores_out);
  return cudaGetLastError() == cudaSuccess ? DKV_OK : DKV_ERR_CUDA;
}
