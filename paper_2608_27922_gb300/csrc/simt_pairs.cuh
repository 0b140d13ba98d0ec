// Tiled fp32 pair interactions on the CUDA cores, shared by the exactness mode's passes and
// the allocation-free scores.
//
// A pair's squared distance is the sum of two parts: dimensions [0, D/2) and [D/2, D) of the
// key, or with the [K; V] descriptor the key and the value.  Each part is a chain of fused
// multiply-adds over its dimensions in increasing order, the parts are joined by one rounded
// add, and w follows from riesz_w (Eq. 2).  Every pass and every tile size does exactly this,
// so all of them give the same bits for a pair.
//
// What bounds it: 2 D fp32 operations a pair (a difference and a fused multiply-add per
// dimension), in packed fp32x2 instructions over two neighbouring columns (each lane rounds
// like the scalar form; 37 T operations/s over the GPU, as the scalar form, with half the
// issue slots, which pay for the loads and the row operand's broadcast).  A block of 128
// threads takes RT rows against 128 columns at a time; a thread holds RT / 8 x 8 partial sums
// (16 rows: 4 x 4), so an element read from shared memory serves 4 or 8 pairs: with 4 x 8
// the reads alone kept the shared-memory pipe busy as long as the arithmetic took.  Rows are
// staged once, columns negated (r - c as r + (-c)) in chunks of 32 dimensions, the next
// chunk in registers while this one is used; four neighbouring threads load a column's chunk
// (one thread per column touched 32 cache lines with every load) and store it transposed, in
// 16-byte groups of columns swizzled by the dimension, so that neither side meets a bank
// conflict (12-head update of 1,560 x 9,360: 7,109 -> 6,842 us).  The 128 columns' w of a
// row then go through shared memory to one thread, which adds them in column order: a pass's
// row sums keep one fixed order for any tile size.
// Few rows: a cluster of C blocks takes a block's rows, block z the column tiles z, z + C, ..,
// and the running sums go from each tile's block to the next one's through shared memory
// (Chain), so the order of the additions stays the same.
#pragma once

#include "dkv_device.cuh"

namespace dkv {
namespace simt {

constexpr int NT = 128;   // threads per block
constexpr int CT = 128;   // columns per tile
constexpr int KC = 32;    // dimensions per staged column chunk
constexpr double CHAIN_COST = 10.0;   // see pick_shape
constexpr int WS = CT + 4;   // row stride of the w tile (odd in 16-byte units: no bank conflicts)

template <int D, bool KV, int RT>
struct Lay {
  static constexpr int PART = KV ? D : D / 2;        // dimensions per part
  static constexpr int NQ = 2 * PART / KC;           // column chunks per tile
  static constexpr int TR = RT == 64 ? 8 : 4;        // rows per thread
  static constexpr int TC = RT == 16 ? 4 : 8;        // columns per thread
  static constexpr int CG = CT / TC;                 // column groups
  static constexpr int ROWS = 0;                     // float [2 PART][RT]
  static constexpr int COLS = ROWS + 2 * PART * RT;  // float [2 stages][KC][CT]
  static constexpr int W = COLS + 2 * KC * CT;       // float [RT][WS]
  static constexpr int META = W + RT * WS;           // float [CT]
  static constexpr int FLOATS = META + CT;
  static constexpr size_t SMEM = (size_t)FLOATS * 4;
  static_assert(SMEM + RT * 16 <= 227 * 1024, "shared memory per block (with a Chain's mailboxes)");
  static_assert((RT / TR) * CG == NT, "one thread per tile of partial sums");
};

// Hands a row's running state from the block that has added column tile t to the one that
// adds tile t + 1 (rank (t + 1) % C of the cluster; nothing to do with C = 1).  Each scanning
// thread sends to the same thread of that block: its two words, then the tile they are for.
// A mailbox is free again when it is written next: that state has been through the receiver.
// A row whose hand-over did not come within WAIT_NS (far above any legitimate wait) has LOST as
// its second word from there on (which the scans leave alone): its later hand-overs carry that,
// nobody waits again, and the block that holds the row's last state must not store it.
// All of a block's threads construct and finish().
template <int RT, uint64_t WAIT_NS = 2000000000ull>
struct Chain {
  int4* mail;      // [RT] of this block: state x, y; tile
  int z, C, tiles;
  static constexpr int LOST = -2147483647 - 1;
  __device__ __forceinline__ Chain(int4* m, int rank, int size, int ntiles) : mail(m), z(rank), C(size), tiles(ntiles) {
    if (C == 1) return;
    if (threadIdx.x < RT) mail[threadIdx.x].z = 0;
    sync();
  }
  __device__ __forceinline__ void sync() const {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  // no block leaves while another may still write to it
  __device__ __forceinline__ void finish() const {
    if (C > 1) sync();
  }
  // this block holds the state after the last tile
  __device__ __forceinline__ bool last() const { return z == (tiles > 0 ? (tiles - 1) % C : 0); }
  // the state before tile t
  __device__ __forceinline__ void take(int sr, int t, float& x, int& y) {
    if (C == 1 || t == 0 || y == LOST) return;
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(mail + sr));
    uint64_t t0 = 0;
    for (uint32_t it = 1;; ++it) {
      int tag;
      asm volatile("ld.acquire.cluster.shared::cta.b32 %0, [%1];" : "=r"(tag) : "r"(a + 8) : "memory");
      if (tag == t) break;
      if ((it & 255u) == 0u) {
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > WAIT_NS) {
          y = LOST;
          return;
        }
      }
    }
    const volatile int4* m = mail + sr;
    x = __int_as_float(m->x);
    y = m->y;
  }
  __device__ __forceinline__ void give(int sr, int t, float x, int y) const {
    if (C == 1 || t + 1 >= tiles) return;
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(a)
        : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(mail + sr))), "r"((z + 1) % C));
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(__float_as_int(x)), "r"(y) : "memory");
    asm volatile("st.release.cluster.shared::cluster.b32 [%0], %1;" ::"r"(a + 8), "r"(t + 1) : "memory");
  }
};

// Rows and cluster size for H heads of `rows` rows against `cols` columns of `dims` elements.
// The SM with the most blocks sets the time, each costing its rows and tiles (16-row blocks
// read more shared memory per pair: 1.3 times), and one block alone on its SM leaves latencies
// open (1.5 times); in a cluster every block adds its start, end and hand-overs (CHAIN_COST).
// The smallest cluster and the tallest block of equals.  Both sides, us (16 rows, one block |
// chosen | next best): 1 head x 1,560 rows x 9,360 columns 564 | 196 (32 rows, 8 blocks) | 242;
// x 4,680 x 9,360 660 | 531 (64, 4) | 561; 2 heads x 256 x 512, d = 64 23.9 | 16.2 (16, 4) |
// 17.4; 8 x 128 x 4,000 218 | 77 (32, 8) | 82.  More blocks lose where rows fill the SMs: 1 x
// 9,360 x 1,560 189 (32, 1) | 204 (32, 4); 12 x 9,360 x 1,560 1,800 (64, 1) | 1,939 (64, 2).
struct Shape {
  int rows, cluster;
};
inline Shape pick_shape(int64_t H, int64_t rows, int64_t cols, int dims, int64_t n_sm, bool tall) {
  const int64_t tiles = cols > CT ? (cols + CT - 1) / CT : 1;
  const double unit = dims / 128.0;   // cost of one row and tile (1: 0.19 us)
  Shape best{16, 1};
  double least = 1e300;
  for (int C = 1; C <= 8 && C <= tiles; C *= 2)
    for (int rt = tall ? 64 : 32; rt >= 16; rt /= 2) {
      const int64_t blocks = H * ((rows + rt - 1) / rt) * C;
      const int64_t most = (blocks + n_sm - 1) / (n_sm > 0 ? n_sm : 1);
      const double per = rt == 64 ? 1.0 : rt == 32 ? 1.05 : 1.3;
      double c = unit * per * rt * (double)most * (double)((tiles + C - 1) / C) * (most == 1 ? 1.5 : 1.0);
      if (C > 1) c += CHAIN_COST * (double)most;
      if (c < least) {
        least = c;
        best = Shape{rt, C};
      }
    }
  return best;
}

// Place of column c in row k (dimension) of a staged chunk: groups of four columns, permuted
// within every 8 groups by k / 4.
__device__ __forceinline__ int swz(int c, int k) { return c ^ (((k >> 2) & 7) << 2); }

// 8 consecutive elements as floats; vec: p is 16-byte aligned.
template <typename T>
__device__ __forceinline__ void load8(const T* p, bool vec, float (&x)[8]) {
  if (!vec) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = to_f<T>(p[k]);
    return;
  }
  if constexpr (sizeof(T) == 2) {
    const uint4 u = *reinterpret_cast<const uint4*>(p);
    const uint32_t v[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {   // a bf16 is the upper half of its float
      x[2 * k] = __uint_as_float(v[k] << 16);
      x[2 * k + 1] = __uint_as_float(v[k] & 0xffff0000u);
    }
  } else {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  }
}

// Row of the tile whose column sums this thread forms (-1: none): RT / 4 rows per warp.
template <int RT>
__device__ __forceinline__ int scan_row() {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  return lane < RT / 4 ? warp * (RT / 4) + lane : -1;
}

// The interactions of rows [row0, row0 + RT) (those from nrows on are not used) with columns
// [c0, c1).  rk, ck (rv, cv: values, [K; V] descriptor) point at row 0 and column 0 of the
// head, D elements each.  For each tile of up to 128 columns from column t0, scan(t0, nc, w,
// meta) is called in the threads with scan_row() >= 0: w[c] for the thread's row, meta[c] =
// 1 / cbase[t0 + c] (if cbase is given).  Tiles z, z + C, .. only.
template <typename T, int D, bool KV, int RT, typename Scan>
__device__ __forceinline__ void pair_tiles(const T* rk, const T* rv, int row0, int nrows, const T* ck, const T* cv,
                                           const float* cbase, int c0, int c1, const KParams& kp, bool vec,
                                           float* smem, int z, int C, Scan scan) {
  using L = Lay<D, KV, RT>;
  constexpr int TR = L::TR, TC = L::TC, CG = L::CG;
  const int tid = threadIdx.x;
  float* rows = smem + L::ROWS;
  float* cols = smem + L::COLS;
  float* wt = smem + L::W;
  float* meta = smem + L::META;
  {
    const int r = tid % RT;
    const int row = row0 + r;
    for (int g = tid / RT; g < 2 * L::PART / 8; g += NT / RT) {
      float x[8];
      if (row < nrows) {
        const T* p = KV && 8 * g >= D ? rv + (int64_t)row * D + (8 * g - D) : rk + (int64_t)row * D + 8 * g;
        load8<T>(p, vec, x);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = 0.f;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) rows[(8 * g + k) * RT + r] = x[k];
    }
  }
  const int ntiles = (c1 - c0 + CT - 1) / CT;
  if (z >= ntiles) return;
  // column loads: 8 dimensions at a time, 8 (tid % 4) .., of columns tid / 4 + 32 u of the tile
  const int lc = tid / (KC / 8), lk = tid % (KC / 8) * 8;
  float pre[KC / 8][8];
  auto fetch = [&](int t, int q) {
    const int dim = q * KC + lk;
#pragma unroll
    for (int u = 0; u < KC / 8; ++u) {
      const int col = c0 + t * CT + u * (CT / (KC / 8)) + lc;
      if (col < c1) {
        load8<T>(KV && dim >= D ? cv + (int64_t)col * D + (dim - D) : ck + (int64_t)col * D + dim, vec, pre[u]);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) pre[u][k] = 0.f;
      }
    }
  };
  static_assert(NT == CT && KC == 32, "four threads per column and chunk, 32 columns a round");
  // this thread's pairs: rows 4 rg + i (and RT / 2 + 4 rg + i), columns 4 cg + j (and CT / 2
  // + 4 cg + j): 16-byte reads of neighbouring threads are neighbours
  const int rg = tid / CG, cg = tid % CG;
  auto row_of = [&](int i) { return (i >> 2) * (RT / 2) + 4 * rg + (i & 3); };
  const int sr = scan_row<RT>();
  fetch(z, 0);
  int stage = 0;
  for (int t = z; t < ntiles; t += C) {
    const int t0 = c0 + t * CT;
    const int nc = min(CT, c1 - t0);
    float cm = 1.f;
    if (cbase && tid < nc) cm = cbase[t0 + tid];
    float2 q[TR][TC / 2];
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int j = 0; j < TC / 2; ++j) q[i][j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int ch = 0; ch < L::NQ; ++ch) {
      float* cs = cols + stage * KC * CT;
#pragma unroll
      for (int u = 0; u < KC / 8; ++u)
#pragma unroll
        for (int k = 0; k < 8; ++k) cs[(lk + k) * CT + swz(u * (CT / (KC / 8)) + lc, lk + k)] = -pre[u][k];
      if (ch + 1 < L::NQ) fetch(t, ch + 1);
      else if (t + C < ntiles) fetch(t + C, 0);
      // one barrier per chunk: a stage is written again two chunks later
      __syncthreads();
      if (ch == L::NQ / 2) {   // the second part begins: the first waits in this thread's w slots
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
          for (int j = 0; j < TC / 4; ++j) {
            *reinterpret_cast<float4*>(wt + row_of(i) * WS + j * (CT / 2) + 4 * cg) =
                make_float4(q[i][2 * j].x, q[i][2 * j].y, q[i][2 * j + 1].x, q[i][2 * j + 1].y);
            q[i][2 * j] = q[i][2 * j + 1] = make_float2(0.f, 0.f);
          }
      }
      const float* rp = rows + ch * KC * RT + 4 * rg;
#pragma unroll 1
      for (int k4 = 0; k4 < KC; k4 += 4) {   // (one swizzle)
        const float* cp = cs + swz(4 * cg, k4);
#pragma unroll
        for (int k = k4; k < k4 + 4; ++k) {
          float r[TR];
          float2 c[TC / 2];
#pragma unroll
          for (int i = 0; i < TR / 4; ++i) {
            const float4 x = *reinterpret_cast<const float4*>(rp + k * RT + i * (RT / 2));
            r[4 * i] = x.x; r[4 * i + 1] = x.y; r[4 * i + 2] = x.z; r[4 * i + 3] = x.w;
          }
#pragma unroll
          for (int j = 0; j < TC / 4; ++j) {
            const float4 x = *reinterpret_cast<const float4*>(cp + k * CT + j * (CT / 2));
            c[2 * j] = make_float2(x.x, x.y);
            c[2 * j + 1] = make_float2(x.z, x.w);
          }
#pragma unroll
          for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC / 2; ++j) {
              const float2 d = __fadd2_rn(make_float2(r[i], r[i]), c[j]);
              q[i][j] = __ffma2_rn(d, d, q[i][j]);
            }
        }
      }
      stage ^= 1;
    }
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int j = 0; j < TC / 4; ++j) {
        float4* p = reinterpret_cast<float4*>(wt + row_of(i) * WS + j * (CT / 2) + 4 * cg);
        const float4 a = *p;   // the first part
        const float2 x = __fadd2_rn(make_float2(a.x, a.y), q[i][2 * j]);
        const float2 y = __fadd2_rn(make_float2(a.z, a.w), q[i][2 * j + 1]);
        *p = make_float4(riesz_w(x.x, kp), riesz_w(x.y, kp), riesz_w(y.x, kp), riesz_w(y.y, kp));
      }
    if (cbase) meta[tid] = __frcp_rn(cm);
    // (the next tile's chunk barriers stand between this scan and the next write of wt)
    __syncthreads();
    if (sr >= 0) scan(t0, nc, wt + sr * WS, meta);
  }
}

// In-order column loop of a scan: f(column offset, w), unrolled over full tiles.
template <typename F>
__device__ __forceinline__ void for_columns(int nc, const float* w, F f) {
  if (nc == CT) {
#pragma unroll 8
    for (int c = 0; c < CT; c += 4) {
      const float4 x = *reinterpret_cast<const float4*>(w + c);
      f(c, x.x); f(c + 1, x.y); f(c + 2, x.z); f(c + 3, x.w);
    }
  } else {
    for (int c = 0; c < nc; ++c) f(c, w[c]);
  }
}

}  // namespace simt
}  // namespace dkv
