// fp32 "exactness mode" kernels: every candidate/bank interaction is evaluated
// on the CUDA cores as a direct sum of squared differences,
//   d2 = sum_k (a_k - b_k)^2   (fp32, sequential fused multiply-adds),
// then w = (eps + d2 / sigma^2)^(-p) (Eq. 2).  These kernels serve fp32 banks
// and the DKV_SCORE_FP32 mode of bf16 banks.
//
// The pair passes share one tiled kernel (simt_pairs.cuh): a row's interactions are formed
// by many threads and added in column order by one, so the running sums of Eq. C.2 have the
// same order in the crossing pass and in the projection pass that later resumes them from a
// snapshot, and sums do not depend on the tile size.
// Measured at 2,070 MHz (us, two threads per row pair before -> tiled), 12 heads, bf16, d =
// 128: scores 1,560 x 9,360 6,957 -> 1,784, crossings 9,360 x 1,560 1,934 -> 1,792, survivors
// 7,800 x 1,560 1,590 -> 1,449, new baselines 1,560 x 9,360 4,263 -> 1,789 (25 T fp32
// operations/s, the packed pipe about 70% busy); 2 heads, fp32, d = 64, scores 256 x 512
// 144 -> 16 (over clusters of 4 blocks, Chain in simt_pairs.cuh).
#include "dkv_internal.h"
#include "simt_pairs.cuh"

#include <climits>

namespace dkv {

namespace {

enum PMode { PM_SCORE = 0, PM_CROSS = 1, PM_PROJECT = 2, PM_SUB = 3, PM_NEWBASE = 4 };

// The cluster's size and this block's rank (1 and 0 in a launch without clusters), its
// barrier, and reads of the same shared-memory address in the cluster's block z.
__device__ __forceinline__ uint32_t simt_cluster_size() {
  uint32_t x;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(x));
  return x;
}
__device__ __forceinline__ uint32_t simt_cluster_rank() {
  uint32_t x;
  asm("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(x));
  return x;
}
__device__ __forceinline__ void simt_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t remote_addr(const float* p, int z) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(z));
  return r;
}
__device__ __forceinline__ float simt_remote(const float* p, int z) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(remote_addr(p, z)) : "memory");
  return x;
}
__device__ __forceinline__ float2 simt_remote2(const float* p, int z) {
  float2 x;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(x.x), "=f"(x.y) : "r"(remote_addr(p, z)) : "memory");
  return x;
}

template <typename T>
__device__ __forceinline__ void store2(T* p, float a, float b) {
  if constexpr (sizeof(T) == 2) *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
  else *reinterpret_cast<float2*>(p) = make_float2(a, b);
}

struct PairJob {
  int mode;          // PMode
  const void* rk;    // row keys of head 0
  int64_t rk_hs;     // row-key head stride (elements)
  const void* ck;    // column keys of head 0
  int64_t ck_hs;     // column-key head stride (elements)
  const void* rv;    // row values ([K; V] descriptor; same layout as rk)
  const void* cv;    // column values (same layout as ck)
  Bank b;
  Ws w;
  KParams kp;
};

template <typename T>
__device__ __forceinline__ const T* ptr(const void* p, int64_t off) {
  return reinterpret_cast<const T*>(p) + off;
}

template <typename T, int D, bool KV, int RT>
__global__ void __launch_bounds__(simt::NT, RT == 64 || KV ? 2 : RT == 32 ? 3 : 4) simt_pairs(PairJob j) {
  extern __shared__ __align__(16) float smem[];
  pdl_wait();
  pdl_trigger();
  __shared__ int4 mail[RT];
  const int h = blockIdx.y;
  const int mode = j.mode;   // uniform
  const int C = simt_cluster_size(), z = simt_cluster_rank();
  const DevHead hd = j.w.hd[h];
  const int N = layer_of(j.w, h)->N;
  const int rmax = layer_of(j.w, h)->rmax;
  int nrows = 0, c0 = 0, c1 = 0;
  if (mode == PM_SCORE) { nrows = hd.empty ? 0 : N;                 c1 = hd.m_old; }
  if (mode == PM_CROSS) { nrows = hd.empty ? 0 : hd.m_old;          c1 = rmax; }
  if (mode == PM_PROJECT) {
    nrows = hd.empty ? 0 : hd.m_old;
    c0 = (hd.r / SNAP) * SNAP;
    c1 = hd.r;
    // the whole tested range: the crossing pass's final sums are in the slot after the last
    // full snapshot, no column is left to add
    if (hd.r == rmax) c0 = c1 = (hd.r + SNAP - 1) / SNAP * SNAP;
  }
  if (mode == PM_SUB) { nrows = hd.empty ? 0 : hd.m_old - hd.e;     c1 = hd.e; }
  if (mode == PM_NEWBASE) { nrows = hd.r;                           c1 = hd.m_new; }
  const int row0 = blockIdx.x / C * RT;
  if (row0 >= nrows) return;   // (all of a cluster)
  const int sr = simt::scan_row<RT>();
  const int row = row0 + sr;
  const bool active = sr >= 0 && row < nrows;
  simt::Chain<RT> chain(mail, z, C, c1 > c0 ? (c1 - c0 + simt::CT - 1) / simt::CT : 0);
  const int64_t bh = (int64_t)h * j.b.M_max;   // bank head offset (rows)

  // state of this thread's row
  float S = 0.f, thr = 0.f;
  int cross = INT_MAX, self = -1, slot = -1;
  float* snap_row = nullptr;
  if (active) {
    if (mode == PM_CROSS) {
      S = j.b.rho[bh + row];
      thr = __fmul_rn(j.kp.tau, j.b.base[bh + row]);
      if (S >= thr) cross = 0;
      snap_row = j.w.snap + (bh + row) * j.w.snap_stride;
      if (z == 0) snap_row[0] = S;
    } else if (mode == PM_PROJECT) {
      S = j.w.snap[(bh + row) * j.w.snap_stride + c0 / SNAP];
    } else if (mode == PM_SUB) {
      // with no eviction every state survives in place and rho := rho~(r) (Eq. C.4)
      slot = hd.e == 0 ? row : j.w.surv_list[bh + row];
    } else if (mode == PM_NEWBASE) {
      self = j.w.slot_new[(int64_t)h * j.b.n_max + row];
    }
  }
  simt::pair_tiles<T, D, KV, RT>(
      ptr<T>(j.rk, (int64_t)h * j.rk_hs), KV ? ptr<T>(j.rv, (int64_t)h * j.rk_hs) : nullptr, row0, nrows,
      ptr<T>(j.ck, (int64_t)h * j.ck_hs), KV ? ptr<T>(j.cv, (int64_t)h * j.ck_hs) : nullptr,
      mode == PM_SCORE ? j.b.base + bh : nullptr, c0, c1, j.kp, true, smem, z, C,
      [&](int t0, int nc, const float* w, const float* meta) {
        const int t = (t0 - c0) / simt::CT;
        chain.take(sr, t, S, cross);
        if (mode == PM_SCORE) {
          simt::for_columns(nc, w, [&](int c, float x) { S = __fmaf_rn(x, meta[c], S); });
        } else if (mode == PM_CROSS) {
          simt::for_columns(nc, w, [&](int c, float x) {
            S = __fadd_rn(S, x);
            if (cross == INT_MAX && S >= thr) cross = t0 + c + 1;
          });
          static_assert(simt::CT == SNAP, "a snapshot at every tile end");
          // (a partial last tile's is the sum over all columns)
          if (active && cross != chain.LOST) snap_row[(t0 + simt::CT) / SNAP] = S;
        } else if (mode == PM_NEWBASE) {
          simt::for_columns(nc, w, [&](int c, float x) { S = __fadd_rn(S, t0 + c == self ? 0.f : x); });
        } else {
          simt::for_columns(nc, w, [&](int c, float x) { S = __fadd_rn(S, x); });
        }
        chain.give(sr, t, S, cross);
      });
  chain.finish();
  if (!active || !chain.last()) return;
  if (cross == chain.LOST) {   // an incomplete sum is not stored
    dev_fail(j.w.L, DEV_TIMEOUT, 6500 + mode);
    return;
  }
  if ((mode == PM_SUB && (slot < 0 || slot >= hd.m_old)) || (mode == PM_NEWBASE && (self < 0 || self >= hd.M))) {
    dev_fail(j.w.L, DEV_INCONSISTENT, 6000 + mode);   // a list entry out of range: skip the write
    return;
  }
  if (mode == PM_SCORE) {
    j.w.score[(int64_t)h * j.b.n_max + row] = __fdiv_rn(S, (float)hd.m_old);
  } else if (mode == PM_CROSS) {
    j.w.cross[bh + row] = cross;
    const int bin = cross == INT_MAX ? rmax + 1 : cross;
    atomicAdd(&j.w.hist[(int64_t)h * j.w.hist_stride + bin], 1);
  } else if (mode == PM_PROJECT) {
    j.w.rho_t[bh + row] = S;
  } else if (mode == PM_SUB) {
    const float rho = __fsub_rn(j.w.rho_t[bh + slot], S);
    j.b.rho[bh + slot] = rho;
    if (j.kp.refresh) {   // refreshed-baseline policy: b follows the current density
      const float bnew = fmaxf(rho, j.kp.delta);
      j.b.base[bh + slot] = bnew;
      j.w.invb[(int64_t)h * j.w.invb_stride + slot] = __frcp_rn(bnew);
    }
  } else {
    j.b.rho[bh + self] = S;
    const float bnew = fmaxf(S, j.kp.delta);
    j.b.base[bh + self] = bnew;
    j.w.invb[(int64_t)h * j.w.invb_stride + self] = __frcp_rn(bnew);
  }
}

template <typename T, int D, bool KV, int RT>
cudaError_t launch_tile(int max_rows, int C, cudaStream_t s, const PairJob& j) {
  const bool after = j.mode == PM_SCORE || j.mode == PM_CROSS;   // follows another kernel of the same call
  return launch_kernel(simt_pairs<T, D, KV, RT>, dim3((max_rows + RT - 1) / RT * C, j.b.H), simt::NT,
                       simt::Lay<D, KV, RT>::SMEM, C, after, s, j);
}

template <typename T, int D, bool KV>
cudaError_t launch_rows(int max_rows, int max_cols, cudaStream_t s, const PairJob& j) {
  const simt::Shape p = simt::pick_shape(j.b.H, max_rows, max_cols, KV ? 2 * D : D, sm_count(), !KV);
  switch (p.rows) {
    case 64:
      if constexpr (!KV) return launch_tile<T, D, KV, 64>(max_rows, p.cluster, s, j);
      [[fallthrough]];
    case 32: return launch_tile<T, D, KV, 32>(max_rows, p.cluster, s, j);
    default: return launch_tile<T, D, KV, 16>(max_rows, p.cluster, s, j);
  }
}

template <typename T, int D>
cudaError_t launch_desc(int max_rows, int max_cols, cudaStream_t s, const PairJob& j) {
  return j.rv ? launch_rows<T, D, true>(max_rows, max_cols, s, j) : launch_rows<T, D, false>(max_rows, max_cols, s, j);
}

// rv / cv: the row and column values, non-null only with the [K; V] descriptor.
cudaError_t launch_pairs(int mode, const Bank& b, const Ws& w, const KParams& kp, const void* rk, int64_t rk_hs,
                         const void* ck, int64_t ck_hs, const void* rv, const void* cv, int max_rows,
                         int max_cols, cudaStream_t s, Timer* t, const char* name) {
  PairJob j{mode, rk, rk_hs, ck, ck_hs, rv, cv, b, w, kp};
  if (max_rows <= 0) return cudaSuccess;
  timer_begin(t, name, s);
  cudaError_t e;
  if (b.bf16)
    e = b.d == 128 ? launch_desc<__nv_bfloat16, 128>(max_rows, max_cols, s, j)
                   : launch_desc<__nv_bfloat16, 64>(max_rows, max_cols, s, j);
  else
    e = b.d == 128 ? launch_desc<float, 128>(max_rows, max_cols, s, j) : launch_desc<float, 64>(max_rows, max_cols, s, j);
  timer_end(t, s);
  return e;
}

// ---------------------------------------------------------------- attention
// Online softmax over tiles of 128 keys for RT queries a block, everything in fp32.  What
// bounds it: 2 D fused multiply-adds a (query, key) pair in packed fp32x2 form, and the
// shared-memory reads that feed them.  A thread holds RT / 8 queries x 8 keys of the scores and
// RT / 8 queries x D / 16 dimensions of the output (16 queries: 4 x 4 and 4 x D / 32), so a value
// read serves 4 to 8 products.  Keys come in chunks of 32 dimensions, transposed, values in
// chunks of 32 keys, through one pair of staging buffers, the next chunk in registers while
// this one is used; one barrier a chunk.
// Small grids over long key ranges: a cluster of up to 8 blocks takes the key tiles of one
// query tile in equal parts, and each block merges a share of the rows from the others'
// shared memory.
// Measured at 2,070 MHz (us, one thread per query before -> this): 12 heads,
// fp32, d = 128, 1,560 queries x 6,240 keys 4,743 -> 1,306 (46 TFLOP/s); 12 heads, d = 64,
// 4,680 x 9,360 5,576 -> 3,227; 2 heads, d = 64, 256 x 768 315 -> 20; 1 head, d = 64,
// 139 x 7,681 2,919 -> 41.
constexpr int ANT = 128;   // threads per block
constexpr int AK = 128;    // keys per tile
constexpr int AC = 32;     // dimensions (keys) per staged chunk of keys (values)

template <int D, int RT>
struct LayA {
  static constexpr int TR = RT == 64 ? 8 : 4;        // queries per thread
  static constexpr int TC = RT == 16 ? 4 : 8;        // keys per thread
  static constexpr int CG = AK / TC;                 // key groups == dimension groups
  static constexpr int DPT = D / CG;                 // output dimensions per thread (2, 4 or 8)
  static constexpr int NK = D / AC, NV = AK / AC;    // chunks of a tile's keys and values
  static constexpr int PS = RT + 4;                  // row stride of the weights
  static constexpr int Q = 0;                        // [D][RT], scaled by log2(e) / sqrt(d)
  static constexpr int C = Q + D * RT;               // [2 stages][AC][128]
  static constexpr int P = C + 2 * AC * 128;         // [AK][PS] weights, key-major
  static constexpr int ML = P + AK * PS;             // [2][RT] maximum and sum (merge)
  static constexpr size_t SMEM = (size_t)(ML + 2 * RT) * 4;
  static_assert(SMEM <= 227 * 1024, "shared memory per block");
  static_assert((RT / TR) * CG == ANT && RT * D <= AK * PS, "thread tiling; merge rows fit over the weights");
};

template <typename T, int D, int RT>
__global__ void __launch_bounds__(ANT, RT == 64 ? 2 : 3)
    simt_attend(const T* __restrict__ Q, int Nq, const T* __restrict__ Kw, const T* __restrict__ Vw, int W,
                T* __restrict__ O, Bank b, float qscale) {
  using L = LayA<D, RT>;
  constexpr int TR = L::TR, TC = L::TC, CG = L::CG, DPT = L::DPT, NK = L::NK, NV = L::NV;
  constexpr int LV = AC * D / 8 / ANT;               // 8-element loads per thread and value chunk
  extern __shared__ __align__(16) float smem[];
  float* qs = smem + L::Q;
  float* cbuf = smem + L::C;
  float* ps = smem + L::P;
  float* ml = smem + L::ML;
  const int tid = threadIdx.x;
  const int h = blockIdx.y;
  const int nsplit = (int)simt_cluster_size(), part = (int)simt_cluster_rank();
  const int q0 = (int)blockIdx.x / nsplit * RT;
  const int m = min(max(b.occ[h], 0), b.M_max);
  const int nkeys = m + W;
  const int ntot = (nkeys + AK - 1) / AK;
  const int tbeg = (int)((int64_t)ntot * part / nsplit), tend = (int)((int64_t)ntot * (part + 1) / nsplit);
  const T* kb = reinterpret_cast<const T*>(b.k) + (int64_t)h * b.M_max * D;
  const T* vb = reinterpret_cast<const T*>(b.v) + (int64_t)h * b.M_max * D;
  const T* kw = Kw + (int64_t)h * W * D;
  const T* vw = Vw + (int64_t)h * W * D;
  float pre[AC / 8][8];
  auto load = [&](int key, int dim, const T* bank, const T* win, float (&x)[8]) {
    if (key < nkeys) {
      simt::load8<T>(key < m ? bank + (int64_t)key * D + dim : win + (int64_t)(key - m) * D + dim, true, x);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = 0.f;
    }
  };
  // chunk ch of tile t: dimensions [32 ch, +32) of the keys, staged as the pair passes' columns,
  // then values of keys [32 (ch - NK), +32) (8-element group e: key e / (D / 8)).  Four threads
  // share a key's chunk with fp32 keys (1,387 -> 1,306 us at 1,560 x 6,240, d = 128); with bf16
  // keys, half as many lines a load, one thread per key is faster (98 against 118 us at 4 heads
  // x 300 x 2,300)
  constexpr bool SHARED = sizeof(T) == 4;
  auto load_key = [&](int u) { return SHARED ? u * 32 + tid / (AC / 8) : tid; };
  auto load_dim = [&](int u) { return 8 * (SHARED ? tid % (AC / 8) : u); };
  auto fetch = [&](int t, int ch) {
    if (ch < NK) {
#pragma unroll
      for (int u = 0; u < AC / 8; ++u) load(t * AK + load_key(u), ch * AC + load_dim(u), kb, kw, pre[u]);
    } else {
#pragma unroll
      for (int u = 0; u < LV; ++u) {
        const int e = u * ANT + tid;
        load(t * AK + (ch - NK) * AC + e / (D / 8), 8 * (e % (D / 8)), vb, vw, pre[u]);
      }
    }
  };
  int stage = 0;
  // the fetched chunk into its stage, the fetch of the next one, and the barrier that publishes
  // it (a stage is written again two chunks later)
  auto advance = [&](int t, int ch) -> const float* {
    float* cs = cbuf + stage * AC * 128;
    stage ^= 1;
    if (ch < NK) {
#pragma unroll
      for (int u = 0; u < AC / 8; ++u)
#pragma unroll
        for (int k = 0; k < 8; ++k)
          cs[(load_dim(u) + k) * AK + simt::swz(load_key(u), load_dim(u) + k)] = pre[u][k];
    } else {
#pragma unroll
      for (int u = 0; u < LV; ++u) {
        const int e = u * ANT + tid;
        float4* p = reinterpret_cast<float4*>(cs + (e / (D / 8)) * D + 8 * (e % (D / 8)));
        p[0] = make_float4(pre[u][0], pre[u][1], pre[u][2], pre[u][3]);
        p[1] = make_float4(pre[u][4], pre[u][5], pre[u][6], pre[u][7]);
      }
    }
    if (ch + 1 < NK + NV) fetch(t, ch + 1);
    else if (t + 1 < tend) fetch(t + 1, 0);
    __syncthreads();
    return cs;
  };
  for (int e = tid; e < RT * D / 8; e += ANT) {
    const int r = e % RT, dim = 8 * (e / RT);
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = 0.f;
    if (q0 + r < Nq) simt::load8<T>(Q + ((int64_t)h * Nq + q0 + r) * D + dim, true, x);
#pragma unroll
    for (int k = 0; k < 8; ++k) qs[(dim + k) * RT + r] = x[k] * qscale;
  }
  // this thread: queries 4 rg + i (and RT / 2 + 4 rg + i), keys 4 cg + c (and 64 + 4 cg + c),
  // output dimensions 4 cg + k (and D / 2 + 4 cg + k), or 2 cg + k
  const int rg = tid / CG, cg = tid % CG;
  auto row_of = [&](int i) { return (i >> 2) * (RT / 2) + 4 * rg + (i & 3); };
  float2 o[TR][DPT / 2];
  float mrun[TR], l[TR];
#pragma unroll
  for (int i = 0; i < TR; ++i) {
    mrun[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int k = 0; k < DPT / 2; ++k) o[i][k] = make_float2(0.f, 0.f);
  }
  if (tbeg < tend) fetch(tbeg, 0);
  for (int t = tbeg; t < tend; ++t) {
    float2 s2[TR][TC / 2];                           // neighbouring keys
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int c = 0; c < TC / 2; ++c) s2[i][c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int ch = 0; ch < NK; ++ch) {
      const float* kc = advance(t, ch);
      const float* qp = qs + ch * AC * RT + 4 * rg;
#pragma unroll 1
      for (int k4 = 0; k4 < AC; k4 += 4) {   // (one swizzle)
        const float* kp = kc + simt::swz(4 * cg, k4);
#pragma unroll
        for (int k = k4; k < k4 + 4; ++k) {
          float qv[TR];
          float2 kv[TC / 2];
#pragma unroll
          for (int i = 0; i < TR / 4; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(qp + k * RT + i * (RT / 2));
            qv[4 * i] = x.x; qv[4 * i + 1] = x.y; qv[4 * i + 2] = x.z; qv[4 * i + 3] = x.w;
          }
#pragma unroll
          for (int c = 0; c < TC / 4; ++c) {
            const float4 x = *reinterpret_cast<const float4*>(kp + k * AK + c * (AK / 2));
            kv[2 * c] = make_float2(x.x, x.y);
            kv[2 * c + 1] = make_float2(x.z, x.w);
          }
#pragma unroll
          for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int c = 0; c < TC / 2; ++c) s2[i][c] = __ffma2_rn(make_float2(qv[i], qv[i]), kv[c], s2[i][c]);
        }
      }
    }
    bool raised = false;
    float alpha[TR];
    const int lim = nkeys - t * AK - 4 * cg;         // (keys past the end have weight 0)
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < TC; ++c) {
        float& x = c & 1 ? s2[i][c / 2].y : s2[i][c / 2].x;
        if ((c >> 2) * (AK / 2) + (c & 3) >= lim) x = -INFINITY;
        mx = fmaxf(mx, x);
      }
#pragma unroll
      for (int w = 1; w < CG; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
      const bool up = mx > mrun[i];
      alpha[i] = up ? exp2f(mrun[i] - mx) : 1.f;
      raised = raised || up;
      if (up) mrun[i] = mx;
      l[i] *= alpha[i];
#pragma unroll
      for (int c = 0; c < TC; ++c) {
        float& x = c & 1 ? s2[i][c / 2].y : s2[i][c / 2].x;
        x = exp2f(x - mrun[i]);
        l[i] += x;
      }
    }
    // (the barriers of this tile's key chunks stand between the last tile's reads and this)
#pragma unroll
    for (int c = 0; c < TC; ++c)
#pragma unroll
      for (int i = 0; i < TR / 4; ++i) {
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = c & 1 ? s2[4 * i + e][c / 2].y : s2[4 * i + e][c / 2].x;
        *reinterpret_cast<float4*>(ps + ((c >> 2) * (AK / 2) + 4 * cg + (c & 3)) * L::PS + i * (RT / 2) + 4 * rg) =
            make_float4(x[0], x[1], x[2], x[3]);
      }
    if (raised) {
#pragma unroll
      for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int k = 0; k < DPT / 2; ++k) o[i][k] = __fmul2_rn(o[i][k], make_float2(alpha[i], alpha[i]));
    }
#pragma unroll
    for (int ch = 0; ch < NV; ++ch) {
      const float* vp = advance(t, NK + ch) + (DPT < 4 ? 2 : 4) * cg;
      const float* pp = ps + ch * AC * L::PS + 4 * rg;
#pragma unroll 4
      for (int c = 0; c < AC; ++c) {
        float p[TR];
        float2 v[DPT / 2];
#pragma unroll
        for (int i = 0; i < TR / 4; ++i) {
          const float4 x = *reinterpret_cast<const float4*>(pp + c * L::PS + i * (RT / 2));
          p[4 * i] = x.x; p[4 * i + 1] = x.y; p[4 * i + 2] = x.z; p[4 * i + 3] = x.w;
        }
        if constexpr (DPT == 2) {
          v[0] = *reinterpret_cast<const float2*>(vp + c * D);
        } else {
#pragma unroll
          for (int k = 0; k < DPT / 4; ++k) {
            const float4 x = *reinterpret_cast<const float4*>(vp + c * D + k * (D / 2));
            v[2 * k] = make_float2(x.x, x.y);
            v[2 * k + 1] = make_float2(x.z, x.w);
          }
        }
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
          for (int k = 0; k < DPT / 2; ++k) o[i][k] = __ffma2_rn(make_float2(p[i], p[i]), v[k], o[i][k]);
      }
    }
  }
  auto dim_of = [&](int k) { return DPT == 2 ? 2 * cg : (k >> 1) * (D / 2) + 4 * cg + 2 * (k & 1); };   // of pair k
  // each query's sum over its CG threads
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int w = 1; w < CG; w <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], w);
  if (nsplit == 1) {
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const int r = row_of(i);
      if (q0 + r >= Nq) continue;
      const float inv = l[i] > 0.f ? 1.f / l[i] : 0.f;
      T* op = O + ((int64_t)h * Nq + q0 + r) * D;
#pragma unroll
      for (int k = 0; k < DPT / 2; ++k) store2(op + dim_of(k), o[i][k].x * inv, o[i][k].y * inv);
    }
    return;
  }
  // ---- merge over the cluster: unnormalised rows [RT][D] over the weights, (m, l) beside
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TR; ++i) {
    const int r = row_of(i);
#pragma unroll
    for (int k = 0; k < DPT / 2; ++k) *reinterpret_cast<float2*>(ps + r * D + dim_of(k)) = o[i][k];
    if (cg == 0) {
      ml[r] = mrun[i];
      ml[RT + r] = l[i];
    }
  }
  simt_cluster_sync();
  for (int e = part * ANT + tid; e < RT * D / 2; e += nsplit * ANT) {
    const int r = e / (D / 2), k = e % (D / 2);
    if (q0 + r >= Nq) continue;
    float mx = -INFINITY;
    for (int z = 0; z < nsplit; ++z) mx = fmaxf(mx, simt_remote(ml + r, z));
    float2 x = make_float2(0.f, 0.f);
    float den = 0.f;
    for (int z = 0; z < nsplit; ++z) {
      const float mz = simt_remote(ml + r, z), lz = simt_remote(ml + RT + r, z);
      const float a = mz == -INFINITY ? 0.f : exp2f(mz - mx);   // (no key in that part: nothing to add)
      const float2 oz = simt_remote2(ps + r * D + 2 * k, z);
      den = fmaf(a, lz, den);
      x.x = fmaf(a, oz.x, x.x);
      x.y = fmaf(a, oz.y, x.y);
    }
    const float inv = den > 0.f ? 1.f / den : 0.f;
    store2(O + ((int64_t)h * Nq + q0 + r) * D + 2 * k, x.x * inv, x.y * inv);
  }
  simt_cluster_sync();                               // the others may still read this block's rows
}

}  // namespace

// With the [K; V] descriptor every pass also reads the values beside its keys: the
// candidates' (source order; pi order: vperm), the bank's, and the survivors' and evicted
// states' copies (vsurv, vevict) taken by commit.
cudaError_t launch_score_fp32(const Bank& b, const Ws& w, const void* Kc, const void* Vc, int N, const KParams& kp,
                              cudaStream_t s, Timer* t) {
  // rows: candidates in source order; columns: bank keys [0, m)
  const bool kv = w.vperm != nullptr;
  return launch_pairs(PM_SCORE, b, w, kp, Kc, (int64_t)N * b.d, b.k, (int64_t)b.M_max * b.d, kv ? Vc : nullptr,
                                kv ? b.v : nullptr, N, b.M_max, s, t, "score_fp32");
}

cudaError_t launch_cross_fp32(const Bank& b, const Ws& w, const KParams& kp, cudaStream_t s, Timer* t) {
  const bool kv = w.vperm != nullptr;
  return launch_pairs(PM_CROSS, b, w, kp, b.k, (int64_t)b.M_max * b.d, w.kperm, (int64_t)b.n_max * b.d,
                                kv ? b.v : nullptr, w.vperm, b.M_max, b.n_max, s, t, "cross_fp32");
}

cudaError_t launch_project_fp32(const Bank& b, const Ws& w, const KParams& kp, cudaStream_t s, Timer* t) {
  const bool kv = w.vperm != nullptr;
  return launch_pairs(PM_PROJECT, b, w, kp, b.k, (int64_t)b.M_max * b.d, w.kperm, (int64_t)b.n_max * b.d,
                                  kv ? b.v : nullptr, w.vperm, b.M_max, SNAP, s, t, "project_fp32");
}

cudaError_t launch_subtract_fp32(const Bank& b, const Ws& w, const KParams& kp, cudaStream_t s, Timer* t) {
  return launch_pairs(PM_SUB, b, w, kp, w.ksurv, (int64_t)b.M_max * b.d, w.kevict, (int64_t)b.n_max * b.d,
                              w.vsurv, w.vevict, b.M_max, b.n_max, s, t, "subtract_fp32");
}

cudaError_t launch_newbase_fp32(const Bank& b, const Ws& w, const KParams& kp, cudaStream_t s, Timer* t) {
  const bool kv = w.vperm != nullptr;
  return launch_pairs(PM_NEWBASE, b, w, kp, w.kperm, (int64_t)b.n_max * b.d, b.k, (int64_t)b.M_max * b.d,
                                  w.vperm, kv ? b.v : nullptr, b.n_max, b.M_max, s, t, "newbase_fp32");
}

namespace {

template <typename T, int D, int RT>
cudaError_t launch_attend_t(const Bank& b, const void* Q, int Nq, const void* Kw, const void* Vw, int W, void* O,
                            int split, cudaStream_t s) {
  const float qscale = 1.4426950408889634f / sqrtf((float)D);   // log2(e) / sqrt(d)
  return launch_kernel(simt_attend<T, D, RT>, dim3((unsigned)((Nq + RT - 1) / RT * split), b.H), ANT,
                       LayA<D, RT>::SMEM, split, false, s, (const T*)Q, Nq, (const T*)Kw, (const T*)Vw, W, (T*)O, b,
                       qscale);
}

template <typename T, int D>
cudaError_t launch_attend_d(const Bank& b, const void* Q, int Nq, const void* Kw, const void* Vw, int W, void* O,
                            cudaStream_t s) {
  switch (simt::pick_shape(b.H, Nq, 1, D, sm_count(), true).rows) {   // (its key split: below)
    case 64: return launch_attend_t<T, D, 64>(b, Q, Nq, Kw, Vw, W, O, 1, s);
    case 32: return launch_attend_t<T, D, 32>(b, Q, Nq, Kw, Vw, W, O, 1, s);
    default: break;
  }
  // few queries: while there are fewer blocks than SMs, twice as many parts of the key range,
  // each of three tiles at least (a part's merge costs about two).  Like the queries per block
  // above, from the handle's heads and budgets and the call's sizes alone
  const int64_t blocks = (int64_t)b.H * ((Nq + 15) / 16);
  const int tiles = (int)(((int64_t)b.M_max + W + AK - 1) / AK);
  int split = 1;
  while (split < 8 && blocks * split < sm_count() && tiles >= 6 * split) split *= 2;
  return launch_attend_t<T, D, 16>(b, Q, Nq, Kw, Vw, W, O, split, s);
}

}  // namespace

cudaError_t launch_attend_fp32(const Bank& b, const void* Q, int Nq, const void* Kw, const void* Vw, int W,
                               void* O, cudaStream_t s, Timer* t) {
  timer_begin(t, "attend_fp32", s);
  cudaError_t e;
  if (b.bf16) {
    e = b.d == 128 ? launch_attend_d<__nv_bfloat16, 128>(b, Q, Nq, Kw, Vw, W, O, s)
                   : launch_attend_d<__nv_bfloat16, 64>(b, Q, Nq, Kw, Vw, W, O, s);
  } else {
    e = b.d == 128 ? launch_attend_d<float, 128>(b, Q, Nq, Kw, Vw, W, O, s)
                   : launch_attend_d<float, 64>(b, Q, Nq, Kw, Vw, W, O, s);
  }
  timer_end(t, s);
  return e;
}

// Dynamic shared memory above 48 KB must be opted into once per kernel.
namespace {

template <typename K>
void opt_in(cudaError_t& e, K k, size_t bytes) {
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T, int D>
void opt_in_all(cudaError_t& e) {
  opt_in(e, simt_pairs<T, D, false, 64>, simt::Lay<D, false, 64>::SMEM);
  opt_in(e, simt_pairs<T, D, false, 32>, simt::Lay<D, false, 32>::SMEM);
  opt_in(e, simt_pairs<T, D, false, 16>, simt::Lay<D, false, 16>::SMEM);
  opt_in(e, simt_pairs<T, D, true, 32>, simt::Lay<D, true, 32>::SMEM);
  opt_in(e, simt_pairs<T, D, true, 16>, simt::Lay<D, true, 16>::SMEM);
  opt_in(e, simt_attend<T, D, 64>, LayA<D, 64>::SMEM);
  opt_in(e, simt_attend<T, D, 32>, LayA<D, 32>::SMEM);
  opt_in(e, simt_attend<T, D, 16>, LayA<D, 16>::SMEM);
}

}  // namespace

cudaError_t simt_set_smem_limits() {
  cudaError_t e = cudaSuccess;
  opt_in_all<float, 128>(e);
  opt_in_all<float, 64>(e);
  opt_in_all<__nv_bfloat16, 128>(e);
  opt_in_all<__nv_bfloat16, 64>(e);
  return e;
}

}  // namespace dkv
