// Block-Jacobi PCG with the textbook recurrences, one scene per launch, in 32-row units
// with the direction replicated on the halo (the linear solve of Algorithm 1; Sec. 4.1
// "Linear Solvers", Sec. 5.1).  Two users: the FP64 scenes (T = double, the arithmetic of
// k_pcg_s<double>) and ppn_pcg_solve_static (T = float, the arithmetic of k_pcg<float, 4>:
// FP32 vectors, FP64 sums and scalars).  Both give the bits of those kernels.
//
// What bounds it.  FP64 issues at two fused multiply-adds per clock and SM here, so what
// counts is how many SMs share the FP64 work and how much of it there is; next come the
// two grid-wide exchanges of an iteration (about 1.2 us each) and the latency of the
// FP64 chains between them.  Hence:
//   - the rows go to the CTAs in units of 32 (a reduction tile is four of them), so that
//     a small scene uses up to four times the CTAs that 128-row tiles would;
//   - a CTA keeps the direction d of its rows and of its halo (the rows of other CTAs that
//     its columns refer to) in shared memory and forms d = z + beta d once per row there,
//     not once per gathered block; what crosses CTAs is z of the halo rows;
//   - in FP64 the SpMV and the updates go component by component over the threads, so that
//     all four sub-partitions of an SM work on 32 rows; sums run only where rows are;
//   - a warp's FP64 instruction holds its sub-partition for 64 cycles whatever its lanes do:
//     levels of a tree that add only zeros are left out, comparisons look at the bits, both
//     sums of the FP32 form share one warp's tree, and rows past the end hold zeros (a branch
//     there ran the last CTA's sums once per side: 546 rows, 6.2 -> 5.5 us per CG iteration);
//   - every value crosses the grid as 64-bit words that carry 32 bits and a 32-bit stamp
//     (single-copy atomic: a word with the expected stamp carries the value, no fence).
// Fixed order.  A unit's sum is the warp's tree over its rows (FP64 scenes: d.q by 16-row
// halves), a tile's sum its units in order, a scene's sum the tiles lane-strided over a
// warp and its tree: the order of the kernels named above.  What is posted is a unit's
// sums, or a whole tile's where a CTA has several tiles anyway (RdPlan).  A post's words are
// rewritten two exchanges later, after every CTA has read them.  All waits are bounded.
#include <algorithm>
#include <type_traits>

#include "pcg_common.cuh"
#include "pcg_units.cuh"

namespace ppn {

using namespace pcgdev;

namespace {

constexpr int RD_NT = 512;  // threads per CTA
constexpr int RD_NW = RD_NT / 32;
// 64-bit words per post: two 128-byte lines that one CTA writes, one per exchange (d.q, then the
// failed blocks of the set-up; r.z and r.r).  Packing several posts' words in a line measured slower
// (32000 rows, the d.q exchange 7.4 -> 13 k cycles), and so did both exchanges' words in one line (546
// rows, r.z 4.6 -> 5.9 k cycles): every poll of a line delays the stores to it.
constexpr int RD_LINE = 32, RD_DQ = 0, RD_FAIL = 8, RD_RZ = 16;

template <typename T>
struct RdCfg;
template <>
struct RdCfg<double> {
  static constexpr int G = 2;     // lanes per row in the SpMV
  static constexpr int DQ = 2;    // d.q sums per unit
};
template <>
struct RdCfg<float> {
  static constexpr int G = 4;
  static constexpr int DQ = 1;
};

template <typename T>
struct RdSmem {
  double *w, *t;            // the posts' and the tiles' sums of an exchange
  double* u;                // the CTA's unit sums (posts of whole tiles)
  int *lrp, *lkb, *lgb;     // local row pointers, first global block of each row, first slot step of each group
  int *lcol, *href;         // local columns by slot; halo rows
  T* lval;                  // blocks by slot step: nine runs of 32 values
  int *hkey, *hidx;         // (same memory) set-up: hash of the halo rows
  T *dx, *dy, *dz;          // double: directions of the own rows, then of the halo
  float4* d4;               // float: the same as records
  T *zx, *zy, *zz;          // z of the own and halo rows (float: d4-like records in z4)
  float4* z4;
  T *qx, *qy, *qz;          // q = H d of the own rows
  T *rx, *ry, *rz, *P;      // double: r and the block-Jacobi inverse of the own rows
};

__host__ __device__ inline size_t rd_up16(size_t b) { return (b + 15) & ~size_t(15); }

template <typename T>
__host__ __device__ inline size_t rd_carve(char* base, int n_posts, int n_tiles, int rows, int slots, bool resident, int nh, int hs,
                                           RdSmem<T>* out) {
  size_t off = 0;
  auto take = [&](size_t b) {
    char* p = base ? base + off : nullptr;
    off += rd_up16(b);
    return p;
  };
  RdSmem<T> s{};
  constexpr bool D = sizeof(T) == 8;
  const int gr = 32 / RdCfg<T>::G;
  s.w = (double*)take(sizeof(double) * 2 * n_posts);
  s.t = (double*)take(sizeof(double) * 2 * n_tiles);
  s.u = (double*)take(sizeof(double) * 2 * (rows / 32));
  s.lrp = (int*)take(sizeof(int) * (rows + 1));
  s.lkb = (int*)take(sizeof(int) * rows);
  s.lgb = (int*)take(sizeof(int) * (rows / gr + 1));
  s.lcol = (int*)take(sizeof(int) * slots);
  s.href = (int*)take(sizeof(int) * nh);
  const size_t vb = resident ? sizeof(T) * 9 * (size_t)slots : 0, hb = 2 * sizeof(int) * (size_t)hs;
  s.lval = (T*)take(vb > hb ? vb : hb);
  s.hkey = (int*)s.lval;
  s.hidx = s.hkey + hs;
  if (D) {
    s.dx = (T*)take(sizeof(T) * (rows + nh));
    s.dy = (T*)take(sizeof(T) * (rows + nh));
    s.dz = (T*)take(sizeof(T) * (rows + nh));
    s.zx = (T*)take(sizeof(T) * (rows + nh));
    s.zy = (T*)take(sizeof(T) * (rows + nh));
    s.zz = (T*)take(sizeof(T) * (rows + nh));
    s.rx = (T*)take(sizeof(T) * rows);
    s.ry = (T*)take(sizeof(T) * rows);
    s.rz = (T*)take(sizeof(T) * rows);
    s.P = (T*)take(sizeof(T) * 9 * rows);
  } else {
    s.d4 = (float4*)take(sizeof(float4) * (rows + nh));
    s.z4 = (float4*)take(sizeof(float4) * (rows + nh));
  }
  s.qx = (T*)take(sizeof(T) * rows);
  s.qy = (T*)take(sizeof(T) * rows);
  s.qz = (T*)take(sizeof(T) * rows);
  if (out) *out = s;
  return off;
}

// ---- stamped words: 32 bits of a value and the 32-bit stamp
__device__ __forceinline__ unsigned long long rd_word(unsigned s, unsigned v) {
  return ((unsigned long long)s << 32) | v;
}
__device__ __forceinline__ void rd_st2(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void rd_ld2(const unsigned long long* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void rd_post(unsigned long long* p, unsigned s, double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  rd_st2(p, rd_word(s, (unsigned)(b >> 32)), rd_word(s, (unsigned)b));
}
__device__ __forceinline__ double rd_join(unsigned long long a, unsigned long long b) {
  return __longlong_as_double((long long)((a << 32) | (b & 0xffffffffull)));
}
// three products summed as the kernels named above sum them
__device__ __forceinline__ double rd_dot(double a0, double b0, double a1, double b1, double a2, double b2) {
  return __fma_rn(a2, b2, __fma_rn(a0, b0, __dmul_rn(a1, b1)));
}
__device__ __forceinline__ float rd_dot(float a0, float b0, float a1, float b1, float a2, float b2) {
  return __fmaf_rn(a2, b2, __fmaf_rn(a0, b0, __fmul_rn(a1, b1)));
}
// after_dq and after_rz with their comparisons on the bits: FP64 compares cost as much as adds
__device__ __forceinline__ bool rd_nan(double v) {
  return ((unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
__device__ __forceinline__ void rd_after_dq(SState<double>& s, double dq) {
  s.dq = dq;
  if (rd_nan(dq)) {
    s.nonfinite = 1;
    s.done = 1;
  } else if (__double_as_longlong(dq) <= 0) {  // negative or zero of either sign
    s.ind = 1;
    s.done = 1;
  } else {
    s.alpha = s.rz / dq;
  }
}
// stop: the squared tolerance times the squared norm of b (not negative, as r2)
__device__ __forceinline__ void rd_after_rz(SState<double>& s, double rz, double r2, double stop, int max_iter) {
  s.iters += 1;
  s.rr = r2;
  if (rd_nan(r2) || rd_nan(rz)) {
    s.nonfinite = 1;
    s.done = 1;
  } else if (!rd_nan(stop) && __double_as_longlong(r2) <= __double_as_longlong(stop)) {
    s.done = 1;
  } else if (s.iters >= max_iter) {
    s.hitmax = 1;
    s.done = 1;
  } else {
    s.beta = rz / s.rz;
    s.rz = rz;
  }
}
// A tile sum as k_pcg_s<double> exchanges it (hi and lo words with 16 stamp bits each):
// exact for every ordinary value; an infinite sum becomes a NaN and the last bits of a
// denormal one are dropped.
__device__ __forceinline__ double rd_exchanged(double v) {
  const unsigned e = (unsigned)((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ffu;
  if (e > 64u && e < 0x7ffu) return v;
  unsigned long long w[2];
  Words<double>::split(v, 0u, w);
  return Words<double>::join(w);
}

}  // namespace

template <typename T>
size_t pcg_rd_smem_bytes(const RdPlan& p, int slots, bool resident, int nh) {
  return rd_carve<T>(nullptr, p.n_posts, (p.nv + 127) / 128, p.rows(), slots, resident, nh, rd_hash_size(nh), nullptr);
}
template size_t pcg_rd_smem_bytes<double>(const RdPlan&, int, bool, int);
template size_t pcg_rd_smem_bytes<float>(const RdPlan&, int, bool, int);

// RES: the blocks stay in shared memory; else they are read from L2 every iteration
template <typename T, bool RES>
__global__ void __launch_bounds__(RD_NT, 1) k_pcg_rd(RdLaunch<T> A) {
  constexpr bool D = sizeof(T) == 8;
  constexpr int G = RdCfg<T>::G, GR = 32 / G, DQ = RdCfg<T>::DQ;
  extern __shared__ __align__(16) char dyn[];
  __shared__ SceneLite<T> S;
  __shared__ SState<double> st;
  __shared__ double s_sum[2], s_stop;
  __shared__ int s_bad[RD_NW];
  __shared__ int s_to, s_nh, s_fail, s_scan[RD_NW];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grid = (int)gridDim.x, n_posts = A.plan.n_posts, n_tiles = (A.plan.nv + PCG_TILE - 1) / PCG_TILE;
  const int p0 = rd_post0((int)blockIdx.x, n_posts, grid), p1 = rd_post0((int)blockIdx.x + 1, n_posts, grid);
  const int per = D ? 32 : A.plan.post_rows;        // rows per post: a unit (32) or a tile (128)
  const int row0 = per * p0, rows = per * (p1 - p0);  // (rows past the scene's last one are idle)
  unsigned long long* const my_words = A.words + (size_t)p0 * RD_LINE;
  const int hs = rd_hash_size(A.halo_cap);
  RdSmem<T> L;
  rd_carve<T>(dyn, n_posts, n_tiles, rows, A.slots, RES, A.halo_cap, hs, &L);
  GridBar* bar = A.bar;
  if (tid == 0) {
    load_lite(S, *A.scene);
    s_to = s_nh = s_fail = 0;
  }
  if (tid < RD_NW) s_bad[tid] = 0;
  for (int h = tid; h < hs; h += RD_NT) L.hkey[h] = -1;
  __syncthreads();
  const int nv = S.nv;

  // ---------------- local row pointers and the groups' slot steps
  {
    int len = 0;
    const int i = row0 + tid;
    if (tid < rows) {
      const int kb = i < nv ? S.row_ptr[i] : 0;
      len = i < nv ? S.row_ptr[i + 1] - kb : 0;
      L.lkb[tid] = kb;
    }
    int v = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane == 31) s_scan[warp] = v;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += s_scan[w];
    if (tid < rows) {
      L.lrp[tid] = before + v - len;
      if (tid == rows - 1) L.lrp[rows] = before + v;
    }
    __syncthreads();
    if (tid < rows / GR) {
      int m = 0;
      for (int r = GR * tid; r < GR * tid + GR; ++r) m = max(m, L.lrp[r + 1] - L.lrp[r]);
      L.lgb[tid + 1] = (m + G - 1) / G;
    }
    __syncthreads();
    if (tid == 0) {
      L.lgb[0] = 0;
      for (int g = 0; g < rows / GR; ++g) L.lgb[g + 1] += L.lgb[g];
      if (32 * L.lgb[rows / GR] > A.slots) s_to = 5;  // sized too small: refused before anything is stored
    }
    __syncthreads();
  }
  // ---------------- the halo rows (a hash of the columns outside the CTA's rows) and the local columns
  if (!s_to) {
    for (int item = warp; item < rows; item += RD_NW) {
      const int kb = L.lkb[item], len = L.lrp[item + 1] - L.lrp[item];
      for (int k = lane; k < len; k += 32) {
        const int j = S.col[kb + k];
        if ((j < row0 || j >= row0 + rows) && !rd_insert(L.hkey, hs, j)) s_to = 5;
      }
    }
    __syncthreads();
    rd_rank<RD_NT>(L.hkey, L.hidx, L.href, hs, A.halo_cap, &s_nh);
    if (s_nh > A.halo_cap) s_to = 5;
  }
  __syncthreads();
  if (s_to) {  // (the planner's counts are exact, so this is never reached; the others' waits run out)
    if (tid == 0) atomicExch(&bar->timeout, 1);
    return;
  }
  const int nh = s_nh, n_items = rows + nh;
  // block k of local row item -> its slot
  auto slot_of = [&](int item, int k) { return (L.lgb[item / GR] + k / G) * 32 + (k % G) * GR + item % GR; };
  for (int item = warp; item < rows; item += RD_NW) {
    const int kb = L.lkb[item], len = L.lrp[item + 1] - L.lrp[item];
    for (int k = lane; k < len; k += 32) {
      const int j = S.col[kb + k];
      int c = j - row0;
      if (c < 0 || c >= rows) {
        unsigned h = rd_hash(j) & (unsigned)(hs - 1);
        while (L.hkey[h] != j) h = (h + 1) & (unsigned)(hs - 1);
        c = rows + L.hidx[h];
      }
      L.lcol[slot_of(item, k)] = c;
    }
  }
  __syncthreads();  // (the hash's memory becomes the blocks')
  const size_t nnzb = (size_t)S.nnzb;
  if constexpr (RES) {
    for (int item = warp; item < rows; item += RD_NW) {
      const int kb = L.lkb[item], len = L.lrp[item + 1] - L.lrp[item];
      for (int k = lane; k < len; k += 32) {
        const int q = slot_of(item, k);
        T* v = L.lval + (q >> 5) * 288 + (q & 31);
#pragma unroll
        for (int c = 0; c < 9; ++c) v[32 * c] = S.val[c * nnzb + kb + k];
      }
    }
  }

  // ---------------- exchanges
  auto has = [](unsigned long long w, unsigned s) { return (unsigned)(w >> 32) == s; };
  // two words of one value once both carry stamp s (bounded)
  auto wait2 = [&](const unsigned long long* p, unsigned s, unsigned long long& a, unsigned long long& b) {
    for (unsigned spins = 0; !(has(a, s) && has(b, s)); ++spins) {
      if (spins > kWaitSpins || *(volatile int*)&s_to) {
        s_to = 1;
        return;
      }
      rd_ld2(p, a, b);
    }
  };
  // s_to set: record the timeout and give up
  auto gave_up = [&]() -> bool {
    if (!s_to) return false;
    if (tid == 0) atomicExch(&bar->timeout, 1);
    return true;
  };
  // The scene's sums of NQ quantities from the posts' words at word offset `at` (VU values per
  // quantity): to shared memory, a tile's units in order, then one warp per quantity.  Levels of the
  // warp's tree that would only add the zeros of lanes without a tile are left out: a warp's FP64
  // instruction costs 64 cycles whatever its lanes do.  f(sums) runs in one thread; every thread
  // returns after it.
  auto sums = [&](unsigned s, int at, auto nq_, auto vu_, auto&& first, auto&& f) {
    constexpr int NQ = decltype(nq_)::value, VU = decltype(vu_)::value, NV = NQ * VU;
    first();
    for (int u = tid; u < n_posts; u += RD_NT) {
      const unsigned long long* p = A.words + (size_t)u * RD_LINE + at;
      unsigned long long w[2 * NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) rd_ld2(p + 2 * q, w[2 * q], w[2 * q + 1]);
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        wait2(p + 2 * q, s, w[2 * q], w[2 * q + 1]);
        L.w[NV * u + q] = rd_join(w[2 * q], w[2 * q + 1]);
      }
    }
    __syncthreads();
    if (s_to) return;
    // the sum of tile t of quantity q (values of units past the last one are zero)
    auto tile_sum = [&](int t, int q) {
      if (per == PCG_TILE) return L.w[NQ * t + q];
      constexpr int NA = NQ == 1 ? 4 * VU : 4, step = NQ == 1 ? 1 : NV;
      const double* w = L.w + 4 * NV * t + (NQ == 1 ? 0 : q);
      const int n = min(4, n_posts - 4 * t) * (NQ == 1 ? VU : 1);
      double v[NA];
#pragma unroll
      for (int u = 0; u < NA; ++u) v[u] = u < n ? w[step * u] : 0.0;
#pragma unroll
      for (int u = 1; u < NA; ++u) v[0] += v[u];
      return D ? rd_exchanged(v[0]) : v[0];
    };
    const bool two = n_tiles > 32 && per != PCG_TILE;  // tile sums by all threads first
    if (two) {
      for (int x = tid; x < NQ * n_tiles; x += RD_NT) L.t[x] = tile_sum(x % n_tiles, x / n_tiles);
      __syncthreads();
    }
    if (warp < NQ) {
      double acc = 0.0;
      if (lane < n_tiles) {
        acc = two ? L.t[warp * n_tiles + lane] : tile_sum(lane, warp);
        for (int k = lane + 32; k < n_tiles; k += 32) acc += two ? L.t[warp * n_tiles + k] : L.w[NQ * k + warp];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (o < n_tiles) acc += __shfl_down_sync(0xffffffffu, acc, o);  // (uniform)
      if (lane == 0) {
        s_sum[warp] = acc;
        if (NQ == 1) f(s_sum);
      }
    }
    __syncthreads();
    if (NQ > 1) {
      if (tid == 0) f(s_sum);
      __syncthreads();
    }
  };
  // unit lu's sum v (in one lane) of quantity q: posted at once, or kept for its tile's post
  auto unit_sum = [&](int lu, int q, int at, unsigned s, double v) {
    if (per == PCG_TILE)
      L.u[2 * lu + q] = v;
    else
      rd_post(my_words + (size_t)lu * RD_LINE + at, s, v);
  };
  // the posts of whole tiles: nq sums of four units each, in unit order
  auto post_tiles = [&](int nq, int at, unsigned s) {
    if (per != PCG_TILE) return;
    __syncthreads();
    for (int x = tid; x < nq * (rows / PCG_TILE); x += RD_NT) {
      const int q = x % nq, t = x / nq;
      const double* u = L.u + 8 * t + q;
      rd_post(my_words + (size_t)t * RD_LINE + at + 2 * q, s, ((u[0] + u[2]) + u[4]) + u[6]);
    }
  };
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  auto nothing = [] {};

  // z of the own rows out (stamp s), z of the halo rows in (before the sums' words, which are posted
  // later, and by the last threads first, which have no such words to wait for)
  // The words lie by component, so that a warp's rows store and load whole runs.
  auto z_pair = [&](int c, int i) {  // double: the two words of component c of row i
    return reinterpret_cast<unsigned long long*>(c < 2 ? S.z : S.q) + 2 * ((size_t)(c & 1) * nv + i);
  };
  auto read_halo = [&](unsigned s) {
    if constexpr (D) {
      for (int x = RD_NT - 1 - tid; x < 3 * nh; x += RD_NT) {
        const int c = (x >= nh) + (x >= 2 * nh), h = x - c * nh;
        const unsigned long long* p = z_pair(c, L.href[h]);
        unsigned long long a, b;
        rd_ld2(p, a, b);
        wait2(p, s, a, b);
        (c == 0 ? L.zx : c == 1 ? L.zy : L.zz)[rows + h] = rd_join(a, b);
      }
    } else {
      for (int h = RD_NT - 1 - tid; h < nh; h += RD_NT) {
        const unsigned long long* p = A.z_words + L.href[h];
        unsigned long long w[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = ld_relaxed_u64(p + (size_t)c * nv);
        for (unsigned spins = 0; !(has(w[0], s) && has(w[1], s) && has(w[2], s)); ++spins) {
          if (spins > kWaitSpins || *(volatile int*)&s_to) {
            s_to = 1;
            break;
          }
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if (!has(w[c], s)) w[c] = ld_relaxed_u64(p + (size_t)c * nv);
        }
        L.z4[rows + h] = make_float4(__uint_as_float((unsigned)w[0]), __uint_as_float((unsigned)w[1]),
                                     __uint_as_float((unsigned)w[2]), 0.0f);
      }
    }
  };

  // ---------------- the rows' state.  double: thread t < 3 rows holds component t / rows of row t % rows
  // (x, r and a row of P); float: thread t < rows holds row t
  const int my_c = D ? tid / rows : 0, my_item = D ? tid - my_c * rows : tid;
  const int my_i = row0 + my_item;
  const bool own = (D ? tid < 3 * rows : tid < rows) && my_i < nv;
  T x[3] = {(T)0, (T)0, (T)0}, r[3] = {(T)0, (T)0, (T)0}, P[9];  // (zero where there is no row: no branch
#pragma unroll                                                   // splits a warp before its sums)
  for (int c = 0; c < 9; ++c) P[c] = (T)0;

  // z = P r, r.z and r.r of the own rows, posted with stamp s
  auto precondition = [&](unsigned s) {
    if constexpr (D) {
      // r (just updated) of all components through shared memory, then z, then the sums
      T* lr = my_c == 0 ? L.rx : my_c == 1 ? L.ry : L.rz;
      T* lz = my_c == 0 ? L.zx : my_c == 1 ? L.zy : L.zz;
      if (tid < 3 * rows) lr[my_item] = r[0];
      __syncthreads();
      if (tid < 3 * rows) {
        const T r0 = L.rx[my_item], r1 = L.ry[my_item], rr2 = L.rz[my_item];
        const T z = rd_dot(P[0], r0, P[1], r1, P[2], rr2);
        if (own) rd_post(z_pair(my_c, my_i), s, z);
        lz[my_item] = z;
      }
      __syncthreads();
      // unit u's r.z by warp u, its r.r by the warp `units` further
      const int units = rows / 32;
      for (int w = warp; w < 2 * units; w += RD_NW) {
        const int u = w % units, item = 32 * u + lane;
        const T r0 = L.rx[item], r1 = L.ry[item], rr2 = L.rz[item];
        T v;
        if (w < units) {
          const T z0 = L.zx[item], z1 = L.zy[item], z2 = L.zz[item];
          v = rd_dot(r0, z0, r1, z1, rr2, z2);
        } else {
          v = rd_dot(r0, r0, r1, r1, rr2, rr2);
        }
        v = warp_sum(v);
        if (lane == 0) unit_sum(u, w < units ? 0 : 1, RD_RZ + (w < units ? 0 : 2), s, v);
      }
    } else {
      if (warp < rows / 32) {  // (warp-uniform)
        const T z0 = rd_dot(P[0], r[0], P[1], r[1], P[2], r[2]);
        const T z1 = rd_dot(P[3], r[0], P[4], r[1], P[5], r[2]);
        const T z2 = rd_dot(P[6], r[0], P[7], r[1], P[8], r[2]);
        if (own) {
          unsigned long long* p = A.z_words + my_i;
          st_relaxed_u64(p, rd_word(s, __float_as_uint(z0)));
          st_relaxed_u64(p + nv, rd_word(s, __float_as_uint(z1)));
          st_relaxed_u64(p + 2 * (size_t)nv, rd_word(s, __float_as_uint(z2)));
        }
        L.z4[tid] = make_float4(z0, z1, z2, 0.0f);
        const double rz = (double)rd_dot(r[0], z0, r[1], z1, r[2], z2);
        const double r2 = (double)rd_dot(r[0], r[0], r[1], r[1], r[2], r[2]);
        // both trees in one warp: lanes 0-15 take the halves of r.z, lanes 16-31 those of r.r
        // (warp_sum pairs lane l with l + 16 first, then both halves alike)
        const double give = lane < 16 ? r2 : rz, keep = lane < 16 ? rz : r2;
        double v = keep + __shfl_xor_sync(0xffffffffu, give, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((lane & 15) == 0) unit_sum(warp, lane >> 4, RD_RZ + (lane >> 3), s, v);
      }
      post_tiles(2, RD_RZ, s);
    }
  };

  // ---------------- set-up: block-Jacobi inverse, r = b, z = P r, d = 0, x = 0
  unsigned epoch = 1;
  {
    bool ok = true;
    const int i = row0 + tid;
    if (tid < rows && i < nv) {  // the inverse: thread per row
      T Dg[9], Pm[9];
      const size_t kd = (size_t)S.diag_idx[i];
#pragma unroll
      for (int c = 0; c < 9; ++c) Dg[c] = S.val[c * nnzb + kd];
      ok = spd_inv3(Dg, Pm);
      if constexpr (D) {
        T* Pg = S.Pinv + (size_t)9 * i;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
          Pg[c] = Pm[c];
          L.P[9 * tid + c] = Pm[c];
        }
      } else {
#pragma unroll
        for (int c = 0; c < 9; ++c) P[c] = Pm[c];
      }
    }
    const unsigned bad = __ballot_sync(0xffffffffu, !ok);
    if (lane == 0 && bad) atomicAdd(&s_bad[32 * warp / per], __popc(bad));
    for (int item = tid; item < n_items; item += RD_NT) {
      if constexpr (D)
        L.dx[item] = L.dy[item] = L.dz[item] = (T)0;
      else
        L.d4[item] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncthreads();
    if (own) {
      if constexpr (D) {
#pragma unroll
        for (int k = 0; k < 3; ++k) P[k] = L.P[9 * my_item + 3 * my_c + k];
        if (A.b_from_g) {
          const double* g = reinterpret_cast<const double*>(S.g + my_i);
          r[0] = (T)(-g[my_c]);
        } else {
          r[0] = __ldcg(reinterpret_cast<const double*>(S.r + my_i) + my_c);
        }
      } else {
        const float4 b = __ldcg(reinterpret_cast<const float4*>(S.r) + my_i);
        r[0] = b.x, r[1] = b.y, r[2] = b.z;
      }
    }
    precondition(epoch);
    __syncthreads();  // (the counts)
    if (tid < p1 - p0) st_relaxed_u64(my_words + (size_t)tid * RD_LINE + RD_FAIL, rd_word(epoch, (unsigned)s_bad[tid]));
    // the failed blocks of every post, then the start of the recurrences
    for (int u = tid; u < n_posts; u += RD_NT) {
      const unsigned long long* p = A.words + (size_t)u * RD_LINE + RD_FAIL;
      unsigned long long w = ld_relaxed_u64(p);
      for (unsigned spins = 0; !has(w, epoch); ++spins) {
        if (spins > kWaitSpins || *(volatile int*)&s_to) {
          s_to = 1;
          break;
        }
        w = ld_relaxed_u64(p);
      }
      if ((unsigned)w) atomicAdd(&s_fail, (int)(unsigned)w);
    }
    sums(epoch, RD_RZ, I2{}, I1{}, [&] { read_halo(epoch); }, [&](const double* v) {
      init_state(st, v[0], v[1], (double)s_fail);
      s_stop = (double)S.tol2 * st.rr0;
    });
    if (gave_up()) return;
  }

  while (!st.done) {
    // ---------------- d = z + beta d (own and halo rows), q = H d, d.q
    {
      const T beta = (T)st.beta;
      if constexpr (D) {
        for (int y = tid; y < 3 * n_items; y += RD_NT) {
          const int c = y / n_items, item = y - c * n_items;
          T* d = c == 0 ? L.dx : c == 1 ? L.dy : L.dz;
          const T* z = c == 0 ? L.zx : c == 1 ? L.zy : L.zz;
          d[item] = z[item] + beta * d[item];
        }
      } else {
        for (int item = tid; item < n_items; item += RD_NT) {
          const float4 z = L.z4[item], p = L.d4[item];
          L.d4[item] = make_float4(z.x + beta * p.x, z.y + beta * p.y, z.z + beta * p.z, 0.0f);
        }
      }
      __syncthreads();
    }
    const int ng = rows / GR;
    if constexpr (D) {
      // a warp: 16 rows x 2 lanes, one component
      for (int w = warp; w < 3 * ng; w += RD_NW) {
        const int g = w / 3, c = w - 3 * g, item = GR * g + lane % GR, h = lane / GR;
        const int len = L.lrp[item + 1] - L.lrp[item], j0 = L.lgb[g], nj = L.lgb[g + 1] - j0;
        T a = 0;
#pragma unroll 4
        for (int j = 0; j < nj; ++j)
          if (G * j + h < len) {
            const int cl = L.lcol[(j0 + j) * 32 + lane];
            const T* v = L.lval + (j0 + j) * 288 + 96 * c + lane;
            const T dj0 = L.dx[cl], dj1 = L.dy[cl], dj2 = L.dz[cl];
            a += rd_dot(v[0], dj0, v[32], dj1, v[64], dj2);
          }
        a += __shfl_xor_sync(0xffffffffu, a, 16);
        if (h == 0) (c == 0 ? L.qx : c == 1 ? L.qy : L.qz)[item] = a;
      }
    } else {
      // a warp: 8 rows x 4 lanes
      for (int g = warp; g < ng; g += RD_NW) {
        const int item = GR * g + lane % GR, h = lane / GR;
        const int len = L.lrp[item + 1] - L.lrp[item], j0 = L.lgb[g], nj = L.lgb[g + 1] - j0;
        const int kb = L.lkb[item];
        T ax = 0, ay = 0, az = 0;
#pragma unroll 4
        for (int j = 0; j < nj; ++j)
          if (G * j + h < len) {
            const float4 d = L.d4[L.lcol[(j0 + j) * 32 + lane]];
            T v[9];
            if constexpr (RES) {
#pragma unroll
              for (int c = 0; c < 9; ++c) v[c] = L.lval[(j0 + j) * 288 + 32 * c + lane];
            } else {
#pragma unroll
              for (int c = 0; c < 9; ++c) v[c] = __ldg(S.val + c * nnzb + kb + G * j + h);
            }
            const T dj0 = d.x, dj1 = d.y, dj2 = d.z;
            ax += rd_dot(v[0], dj0, v[1], dj1, v[2], dj2);
            ay += rd_dot(v[3], dj0, v[4], dj1, v[5], dj2);
            az += rd_dot(v[6], dj0, v[7], dj1, v[8], dj2);
          }
#pragma unroll
        for (int o = 16; o >= 8; o >>= 1) {
          ax += __shfl_xor_sync(0xffffffffu, ax, o);
          ay += __shfl_xor_sync(0xffffffffu, ay, o);
          az += __shfl_xor_sync(0xffffffffu, az, o);
        }
        if (h == 0) {
          L.qx[item] = ax;
          L.qy[item] = ay;
          L.qz[item] = az;
        }
      }
    }
    __syncthreads();
    ++epoch;
    if (warp < rows / 32) {  // unit u0 + warp: a lane per row
      const T ax = L.qx[tid], ay = L.qy[tid], az = L.qz[tid];
      if constexpr (D) {
        const T d0 = L.dx[tid], d1 = L.dy[tid], d2 = L.dz[tid];
        T dq = row0 + tid < nv ? rd_dot(d0, ax, d1, ay, d2, az) : (T)0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) dq += __shfl_xor_sync(0xffffffffu, dq, o);
        if ((lane & 15) == 0) rd_post(my_words + (size_t)warp * RD_LINE + RD_DQ + (lane >> 3), epoch, dq);
      } else {
        const float4 di = L.d4[tid];
        double dq = row0 + tid < nv ? (double)rd_dot(di.x, ax, di.y, ay, di.z, az) : 0.0;
        dq = warp_sum(dq);
        if (lane == 0) unit_sum(warp, 0, RD_DQ, epoch, dq);
      }
    }
    if constexpr (!D) post_tiles(1, RD_DQ, epoch);
    sums(epoch, RD_DQ, I1{}, std::integral_constant<int, DQ>{}, nothing, [&](const double* v) { rd_after_dq(st, v[0]); });
    if (gave_up()) return;
    if (st.done) break;

    // ---------------- x += alpha d, r -= alpha q, z = P r
    ++epoch;
    const T alpha = own ? (T)st.alpha : (T)0;
    T d_own = (T)0;
    if (tid < (D ? 3 : 1) * rows) {  // (the rows past the scene's last one stay zero)
      if constexpr (D) {
        d_own = (my_c == 0 ? L.dx : my_c == 1 ? L.dy : L.dz)[my_item];
        const T q = (my_c == 0 ? L.qx : my_c == 1 ? L.qy : L.qz)[my_item];
        r[0] = r[0] - alpha * q;
      } else {
        const float4 di = L.d4[tid];
        x[0] += alpha * di.x;
        x[1] += alpha * di.y;
        x[2] += alpha * di.z;
        r[0] -= alpha * L.qx[tid];
        r[1] -= alpha * L.qy[tid];
        r[2] -= alpha * L.qz[tid];
      }
    }
    precondition(epoch);
    if (D && tid < 3 * rows) x[0] += alpha * d_own;  // (off the chain to the sums; idle warps would hold the FP64 pipe)
    sums(epoch, RD_RZ, I2{}, I1{}, [&] { read_halo(epoch); },
         [&](const double* v) { rd_after_rz(st, v[0], v[1], s_stop, S.max_iter); });
    if (gave_up()) return;
  }

  // x of this CTA's rows; CTA 0 publishes the scalars
  if (own) {
    if constexpr (D) {
      double* o = reinterpret_cast<double*>(S.dx + my_i);
      o[my_c] = x[0];
      if (my_c == 0) o[3] = 0.0;
    } else {
      st_v(S.dx + my_i, mk<float4, float>(x[0], x[1], x[2]));
    }
  }
  if (blockIdx.x == 0 && tid == 0) publish(st, S.ctl);
}

// before a solve: the barrier and the stamped words, which carry stamps of one launch only
template <typename T>
__global__ void k_rd_clear(RdLaunch<T> A, int nv) {
  const int n_thr = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (t0 == 0) *A.bar = GridBar{};
  const ulonglong2 zero = make_ulonglong2(0, 0);
  ulonglong2* w = reinterpret_cast<ulonglong2*>(A.words);
  for (int k = t0; k < A.plan.n_posts * (RD_LINE / 2); k += n_thr) w[k] = zero;
  if constexpr (sizeof(T) == 8) {
    ulonglong2 *z = reinterpret_cast<ulonglong2*>(A.scene->z), *q = reinterpret_cast<ulonglong2*>(A.scene->q);
    for (int k = t0; k < 2 * nv; k += n_thr) z[k] = q[k] = zero;
  } else {
    ulonglong2* z = reinterpret_cast<ulonglong2*>(A.z_words);
    for (int k = t0; k < 2 * nv; k += n_thr) z[k] = zero;
  }
}

// Block slots and halo rows of the largest CTA of a plan, for a device-resident pattern; a CTA with more than HS / 2 halo rows reports more than any plan
// takes.  Skips a pattern that `error` says is malformed.
__global__ void __launch_bounds__(RD_NT) k_rd_plan(const int* row_ptr, const int* col, RdPlan plan, int g_lanes,
                                                   const int* error, int* most_slots, int* most_halo) {
  constexpr int HS = 8192;
  __shared__ int key[HS];
  __shared__ int s_nh, s_steps;
  if (*error) return;
  const int tid = threadIdx.x, gr = 32 / g_lanes;
  for (int h = tid; h < HS; h += RD_NT) key[h] = -1;
  if (tid == 0) s_nh = s_steps = 0;
  __syncthreads();
  const int row0 = plan.post_rows * rd_post0((int)blockIdx.x, plan.n_posts, plan.grid);
  const int rend = plan.post_rows * rd_post0((int)blockIdx.x + 1, plan.n_posts, plan.grid);
  const int r1 = min(plan.nv, rend);
  for (int g = row0 + gr * tid; g < r1; g += gr * RD_NT) {
    int m = 0;
    for (int r = g; r < min(r1, g + gr); ++r) m = max(m, row_ptr[r + 1] - row_ptr[r]);
    atomicAdd(&s_steps, (m + g_lanes - 1) / g_lanes);
  }
  const int kb = row_ptr[row0], ke = row_ptr[r1];
  for (int k = kb + tid; k < ke; k += RD_NT) {
    const int j = col[k];
    if (j >= row0 && j < rend) continue;
    unsigned h = rd_hash(j) & (HS - 1);
    while (*(volatile int*)&s_nh <= HS / 2) {  // (a racy read only lets an over-full table grow a little more)
      const int o = atomicCAS(&key[h], -1, j);
      if (o == -1) atomicAdd(&s_nh, 1);
      if (o == -1 || o == j) break;
      h = (h + 1) & (HS - 1);
    }
  }
  __syncthreads();
  if (tid == 0) {
    atomicMax(most_slots, 32 * s_steps);
    atomicMax(most_halo, s_nh > HS / 2 ? 1 << 24 : s_nh);
  }
}

cudaError_t launch_rd_plan(const int* row_ptr, const int* col, const RdPlan& plan, const int* error, int* most_slots,
                           int* most_halo, cudaStream_t st) {
  k_rd_plan<<<plan.grid, RD_NT, 0, st>>>(row_ptr, col, plan, RdCfg<float>::G, error, most_slots, most_halo);
  return cudaGetLastError();
}

template <typename T>
static const void* rd_kernel(bool resident) {
  if constexpr (sizeof(T) == 8) return (const void*)k_pcg_rd<double, true>;
  return resident ? (const void*)k_pcg_rd<float, true> : (const void*)k_pcg_rd<float, false>;
}

template <typename T>
int pcg_rd_max_grid(int device, size_t smem, bool resident) {
  const void* k = rd_kernel<T>(resident);
  int n_sm = 0, per_sm = 0;
  if (allow_shared(k, smem) != cudaSuccess ||
      cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, RD_NT, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * n_sm;
}
template int pcg_rd_max_grid<double>(int, size_t, bool);
template int pcg_rd_max_grid<float>(int, size_t, bool);

template <typename T>
cudaError_t launch_pcg_rd(const RdLaunch<T>& L, cudaStream_t st) {
  const RdPlan& p = L.plan;
  const int nv = p.nv;
  if (!L.scene || !L.bar || !L.words || nv <= 0 || (p.post_rows != 32 && (p.post_rows != PCG_TILE || sizeof(T) == 8)) ||
      p.n_posts != (nv + p.post_rows - 1) / p.post_rows || p.grid < 1 || p.grid > p.n_posts ||
      p.rows() > (sizeof(T) == 8 ? RD_ROWS_MAX_F64 : RD_NT) || (sizeof(T) == 4 && !L.z_words))
    return cudaErrorInvalidValue;
  k_rd_clear<T><<<std::min(sm_count(), 1 + nv / 128), 256, 0, st>>>(L, nv);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const void* k = rd_kernel<T>(L.resident);
  e = allow_shared(k, L.smem_bytes);
  if (e != cudaSuccess) return e;
  RdLaunch<T> a = L;
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel(k, dim3(p.grid), dim3(RD_NT), args, L.smem_bytes, st);
}
template cudaError_t launch_pcg_rd<double>(const RdLaunch<double>&, cudaStream_t);
template cudaError_t launch_pcg_rd<float>(const RdLaunch<float>&, cudaStream_t);

}  // namespace ppn
