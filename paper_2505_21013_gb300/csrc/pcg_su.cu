// Single-reduction block-Jacobi PCG (the recurrences of pcg_sr.cu, with the same bits) for one
// scene of at most one row tile per SM (the linear solve of Algorithm 1;
// Sec. 4.1 "Linear Solvers", Sec. 5.1).
//
// What bounds it: an iteration's latency.  In the halo layout of pcg_sr.cu a one-tile CTA took
// 6200 cycles per iteration: 2600 for the SpMV of 128 rows with its sums and posts, 1900 for the
// grid's reduction, 740 for the scalar step of one thread between two barriers, 750 for updates
// through shared memory and their barriers.  One way between two SMs through L2 is 500 to 850
// cycles, so a reduction cannot take less than about 1000.  Here (756 rows 3.11 -> 2.17 us per CG
// iteration, 4096 rows 3.27 -> 2.35, 15872 rows 3.39 -> 2.55, where the halo layout, which has had some
// of this since, takes 2.53, 2.75 and 2.78; about 4300 cycles: SpMV 900, its sums
// 390, post and wait 1700, the scene's sums 400, scalar step 440, update and barriers 400):
//   - a CTA has 32, 64 or 128 rows, as few as the SMs allow: the tile sum
//     ((w0 + w1) + (w2 + w3)) + ((w4 + w5) + (w6 + w7)) of eight 16-row groups splits there, so that
//     each CTA posts the sum of its part and every CTA finishes the same tree;
//   - a block's values come as two 16-byte words and one 4-byte word per lane: the few warps of a
//     small CTA wait on the number of loads, not on their bytes;
//   - what crosses the grid is 16-byte words of three values and a stamp, one per row and one per CTA,
//     instead of three 8-byte words: polling loads are what L2 is busy with (4000 rows 3.05 -> 2.41);
//   - the state of the halo rows (r, s, the inverse) stays in registers, as that of the own rows,
//     each in threads of its own.
// Data: blocks by step, as the resident blocks of pcg_sr.cu (16 rows x 2 lanes per warp), u of the
// own and halo rows in shared memory.  A row's w goes out as one stamped 16-byte word, in two parity
// buffers; a CTA's sums likewise, in a line of its own per parity.  A buffer is overwritten two iterations later: by then its writer has the sums of the
// iteration between, which every CTA posted after its reads.  All waits are bounded.
#include <algorithm>

#include "pcg_sr.cuh"
#include "pcg_units.cuh"

namespace ppn {

using namespace pcgdev;

namespace {

constexpr int SU_NT = 512, SU_NW = SU_NT / 32;
constexpr int SU_LINE = 8;  // 16-byte words of a post and parity: gamma, delta, rho; failed blocks (set-up)

struct SuSmem {
  float* w;                // [3][posts of whole tiles] the posts' sums
  float* g;                // [4][8] the CTA's group sums
  int *lkb, *lrp, *lgb;    // first global block and length of each row, first step of each group
  int *lcol, *href;
  float* lval;             // blocks by step: 32 x 16 bytes (values 0..3), 32 x 16 (4..7), 32 x 4 (8)
  int *hkey, *hidx;        // (same memory) set-up: hash of the halo rows
  float4* u;               // own rows, then halo rows
};

__host__ __device__ inline size_t su_carve(char* base, int n_tiles, int rows, int slots, int nh, int hs, SuSmem* out) {
  size_t off = 0;
  auto take = [&](size_t b) {
    char* p = base ? base + off : nullptr;
    off += (b + 15) & ~size_t(15);
    return p;
  };
  SuSmem s{};
  s.w = (float*)take(sizeof(float) * 12 * n_tiles);
  s.g = (float*)take(sizeof(float) * 4 * 8);
  s.lkb = (int*)take(sizeof(int) * rows);
  s.lrp = (int*)take(sizeof(int) * rows);
  s.lgb = (int*)take(sizeof(int) * (rows / 16 + 1));
  s.lcol = (int*)take(sizeof(int) * slots);
  s.href = (int*)take(sizeof(int) * nh);
  const size_t vb = sizeof(float) * 9 * (size_t)slots, hb = 2 * sizeof(int) * (size_t)hs;
  s.lval = (float*)take(vb > hb ? vb : hb);
  s.hkey = (int*)s.lval;
  s.hidx = s.hkey + hs;
  s.u = (float4*)take(sizeof(float4) * (rows + nh));
  if (out) *out = s;
  return off;
}

}  // namespace

size_t pcg_su_smem_bytes(const RdPlan& p, int slots, int nh) {
  return su_carve(nullptr, (p.nv + PCG_TILE - 1) / PCG_TILE, p.rows(), slots, nh, rd_hash_size(nh), nullptr);
}

// ROWS: rows per CTA; HPT: halo rows per thread
template <int ROWS, int HPT>
__global__ void __launch_bounds__(SU_NT, 1) k_pcg_su(SuLaunch A) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ SceneLite<float> S;
  __shared__ SState<float> st;
  __shared__ int s_to, s_nh, s_widx;
  __shared__ unsigned s_seen;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_posts = A.plan.n_posts, n_tiles = (A.plan.nv + PCG_TILE - 1) / PCG_TILE;
  constexpr int rows = ROWS, per_tile = PCG_TILE / rows, ng = rows / 16;
  const int row0 = rows * (int)blockIdx.x;  // (rows past the scene's last one are idle)
  const int hs = rd_hash_size(A.halo_cap);
  SuSmem L;
  su_carve(dyn, n_tiles, rows, A.slots, A.halo_cap, hs, &L);
  if (tid == 0) {
    load_lite(S, *A.scene);
    s_to = s_nh = 0;
    s_widx = -1;
    s_seen = 0;
    st.done = 0;
  }
  for (int h = tid; h < hs; h += SU_NT) L.hkey[h] = -1;
  for (int k = tid; k < 12 * n_tiles; k += SU_NT) L.w[k] = 0.0f;  // (units past the last one)
  __syncthreads();
  const int nv = S.nv;

  // ---------------- set-up: row lengths and the units' steps, the halo, the blocks
  if (tid < rows) {
    const int i = row0 + tid, kb = i < nv ? S.row_ptr[i] : 0;
    L.lkb[tid] = kb;
    L.lrp[tid] = i < nv ? S.row_ptr[i + 1] - kb : 0;
  }
  __syncthreads();
  if (tid == 0) {
    L.lgb[0] = 0;
    for (int g = 0; g < ng; ++g) {
      int m = 0;
      for (int r = 16 * g; r < 16 * g + 16; ++r) m = max(m, L.lrp[r]);
      L.lgb[g + 1] = L.lgb[g] + ((m + 1) >> 1);
    }
    if (32 * L.lgb[ng] > A.slots) s_to = 5;  // sized too small: refused before anything is stored
  }
  for (int item = warp; item < rows; item += SU_NW)
    for (int k = lane; k < L.lrp[item]; k += 32) {
      const int j = S.col[L.lkb[item] + k];
      if ((j < row0 || j >= row0 + rows) && !rd_insert(L.hkey, hs, j)) s_to = 5;
    }
  __syncthreads();
  rd_rank<SU_NT>(L.hkey, L.hidx, L.href, hs, A.halo_cap, &s_nh);
  constexpr int n_row_thr = 2 * rows, n_halo_thr = SU_NT - n_row_thr;
  const int nh = s_nh;
  if (tid == 0 && (nh > A.halo_cap || nh > HPT * n_halo_thr)) s_to = 5;
  __syncthreads();
  if (s_to) {  // (the planner's counts are exact, so this is never reached; the others' waits run out)
    if (tid == 0) atomicExch(&A.bar->timeout, 1);
    return;
  }
  for (int item = warp; item < rows; item += SU_NW)
    for (int k = lane; k < L.lrp[item]; k += 32) {
      const int j = S.col[L.lkb[item] + k];
      int c = j - row0;
      if (c < 0 || c >= rows) {
        unsigned h = rd_hash(j) & (unsigned)(hs - 1);
        while (L.hkey[h] != j) h = (h + 1) & (unsigned)(hs - 1);
        c = rows + L.hidx[h];
      }
      L.lcol[(L.lgb[item >> 4] + (k >> 1)) * 32 + 16 * (k & 1) + (item & 15)] = c;
    }
  __syncthreads();  // (the hash's memory becomes the blocks')
  const size_t nnzb = (size_t)S.nnzb;
  for (int item = warp; item < rows; item += SU_NW)
    for (int k = lane; k < L.lrp[item]; k += 32) {
      float* v = L.lval + (L.lgb[item >> 4] + (k >> 1)) * 288;
      const int ln = 16 * (k & 1) + (item & 15);
#pragma unroll
      for (int c = 0; c < 9; ++c) v[c < 8 ? 128 * (c >> 2) + 4 * ln + (c & 3) : 256 + ln] = S.val[c * nnzb + L.lkb[item] + k];
    }

  // ---------------- the rows' state: a row warp's lanes 0..15 own its rows (slot 0 of the arrays), the
  // threads past the row warps HPT halo rows each
  const bool row_thr = tid < n_row_thr, halo_thr = !row_thr;
  const int h2 = lane >> 4, my_item = 16 * warp + (lane & 15);
  const bool mine = row_thr && h2 == 0;
  const int my_i = row0 + my_item;
  const bool own = mine && my_i < nv;
  float r[HPT][3], sv[HPT][3], P[HPT][6], w[HPT][3], x[3] = {0.f, 0.f, 0.f}, p[3] = {0.f, 0.f, 0.f};
  float u[3] = {0.f, 0.f, 0.f};
  int hrow[HPT], hitem[HPT];
  bool failed = false;
#pragma unroll
  for (int k = 0; k < HPT; ++k) {
    const int h = tid - n_row_thr + k * n_halo_thr;
    const bool halo = halo_thr && h < nh;
    const int i = mine ? (k == 0 && own ? my_i : -1) : halo ? L.href[h] : -1;
    hrow[k] = halo ? i : -1;
    hitem[k] = rows + h;
#pragma unroll
    for (int c = 0; c < 3; ++c) r[k][c] = sv[k][c] = w[k][c] = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) P[k][c] = 0.f;
    if (i >= 0) {
      float D[9], Pm[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) D[c] = S.val[c * nnzb + S.diag_idx[i]];
      const bool ok = spd_inv3(D, Pm);
      sym6(Pm, P[k]);
      if (A.b_from_g) {
        const double4 g = ld_d4(S.g + i);
        r[k][0] = (float)(-g.x);
        r[k][1] = (float)(-g.y);
        r[k][2] = (float)(-g.z);
      } else {
        const float4 rv = __ldcg(reinterpret_cast<const float4*>(S.r) + i);
        r[k][0] = rv.x;
        r[k][1] = rv.y;
        r[k][2] = rv.z;
      }
      float uu[3];
      prec6(P[k], r[k], uu);
      L.u[mine ? my_item : hitem[k]] = make_float4(uu[0], uu[1], uu[2], 0.0f);
      if (mine) {
        failed = !ok;
        float* Pg = S.Pinv + (size_t)9 * i;
#pragma unroll
        for (int c = 0; c < 9; ++c) Pg[c] = Pm[c];
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = uu[c];
      }
    } else if (mine && k == 0) {
      L.u[my_item] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  {
    const int n = __popc(__ballot_sync(0xffffffffu, failed));
    if (lane == 0 && warp < ng) L.g[24 + warp] = (float)n;
  }

  const float tol2 = (float)S.tol2;
  const int max_iter = S.max_iter;
  float4* const zw = reinterpret_cast<float4*>(S.zrec);
  float4* const my_line = A.words + (size_t)blockIdx.x * 2 * SU_LINE;
  // after a wait ran out: the first word found without stamp s, for the timeout record (looked for here, as
  // the waits' loops are the kernel's pace: 2.18 -> 2.27 us per CG iteration when they kept it)
  auto note_missing = [&](const float4* q, unsigned s, int index) {
    unsigned long long a, b;
    ld_word4(q, a, b);
    if (word4_stamp(b) != s && atomicCAS(&s_widx, -1, index) == -1) s_seen = word4_stamp(b);
  };

  for (int it = 0;; ++it) {
    const unsigned s = (unsigned)it + 1;
    const int par = it & 1;
    float4* const wpar = zw + (size_t)par * nv;
    __syncthreads();  // set-up, or the previous update, before the SpMV
    if (row_thr) {
      // ---- w = A u of the group's rows (two lanes per row: even and odd blocks), w out, the group's sums
      const int len = L.lrp[my_item], g0 = L.lgb[warp], nj = L.lgb[warp + 1] - g0;
      float ax = 0.f, ay = 0.f, az = 0.f;
      for (int jb = 0; jb < nj; jb += 4) {
        float4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (2 * (jb + q) + h2 < len) v[q] = L.u[L.lcol[(g0 + jb + q) * 32 + lane]];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (2 * (jb + q) + h2 < len) {
            const float* b = L.lval + (g0 + jb + q) * 288;
            const float4 b0 = reinterpret_cast<const float4*>(b)[lane], b1 = reinterpret_cast<const float4*>(b + 128)[lane];
            const float a[9] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w, b[256 + lane]};
            blk_mv(a, v[q].x, v[q].y, v[q].z, ax, ay, az);
          }
      }
      ax += __shfl_xor_sync(0xffffffffu, ax, 16);
      ay += __shfl_xor_sync(0xffffffffu, ay, 16);
      az += __shfl_xor_sync(0xffffffffu, az, 16);
      w[0][0] = ax, w[0][1] = ay, w[0][2] = az;
      // lanes 0..15: gamma = r.u and rho = r.r, lanes 16..31: delta = w.u (r is zero there and past the
      // scene's last row: no branch)
      const float4 uv = L.u[my_item];
      float g = dot3(h2 ? ax : r[0][0], h2 ? ay : r[0][1], h2 ? az : r[0][2], uv.x, uv.y, uv.z);
      float rho = dot3(r[0][0], r[0][1], r[0][2], r[0][0], r[0][1], r[0][2]);
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) {
        g += __shfl_xor_sync(0xffffffffu, g, d);
        rho += __shfl_xor_sync(0xffffffffu, rho, d);
      }
      if (lane == 0) {
        L.g[warp] = g;
        L.g[16 + warp] = rho;
      }
      if (lane == 16) L.g[8 + warp] = g;
      if (own) st_word4(wpar + my_i, ax, ay, az, s);
    }
    __syncthreads();  // (also: polling that starts before the stores slows them)
    if (warp == 0) {  // ---- the sums of this CTA's part of a tile out (a lane per quantity)
      const float* g = L.g + 8 * (lane & 3);
      float v = g[0] + g[1];
      if (ng > 2) v += g[2] + g[3];
      if (ng > 4) v += (g[4] + g[5]) + (g[6] + g[7]);
      const float del = __shfl_sync(0xffffffffu, v, 1), rho = __shfl_sync(0xffffffffu, v, 2);
      const float bad = __shfl_sync(0xffffffffu, v, 3);
      if (lane == 0) {
        st_word4(my_line + par * SU_LINE, v, del, rho, s);
        if (it == 0) st_word4(my_line + 1, bad, 0.f, 0.f, s);
      }
    }
    if (halo_thr) {
      // ---- w of this thread's halo rows, then the posts' sums (from the last thread down)
#pragma unroll
      for (int k = 0; k < HPT; ++k)
        if (hrow[k] >= 0) {
          unsigned long long va, vb;
          ld_word4(wpar + hrow[k], va, vb);
          for (unsigned spins = 0; word4_stamp(vb) != s; ++spins) {
            if (spins > A.wait_limit || *(volatile int*)&s_to) {
              s_to = 3;
              break;
            }
            ld_word4(wpar + hrow[k], va, vb);
          }
          w[k][0] = __uint_as_float((unsigned)va);
          w[k][1] = __uint_as_float((unsigned)(va >> 32));
          w[k][2] = __uint_as_float((unsigned)vb);
        }
      for (int un = SU_NT - 1 - tid; un < n_posts; un += n_halo_thr) {
        const float4* line = A.words + (size_t)un * 2 * SU_LINE;
        for (int z = it == 0 ? 1 : 0; z >= 0; --z) {  // (set-up: also the failed blocks)
          unsigned long long va, vb;
          const float4* q = z ? line + 1 : line + par * SU_LINE;
          ld_word4(q, va, vb);
          for (unsigned spins = 0; word4_stamp(vb) != s; ++spins) {
            if (spins > A.wait_limit || *(volatile int*)&s_to) {
              s_to = 2;
              break;
            }
            ld_word4(q, va, vb);
          }
          if (z) {
            if (__uint_as_float((unsigned)va) > 0.0f) s_nh = -1;  // (the count of halo rows is not needed any more)
          } else {
            L.w[un] = __uint_as_float((unsigned)va);
            L.w[per_tile * n_tiles + un] = __uint_as_float((unsigned)(va >> 32));
            L.w[2 * per_tile * n_tiles + un] = __uint_as_float((unsigned)vb);
          }
        }
      }
    }
    __syncthreads();
    if (s_to) {
      const int site = s_to;  // (a halo row's word and a post's may both be missing: the one noted last names the wait)
      if (halo_thr) {
        if (site == 3) {
          for (int k = 0; k < HPT; ++k)
            if (hrow[k] >= 0) note_missing(wpar + hrow[k], s, hrow[k]);
        } else {
          for (int un = SU_NT - 1 - tid; un < n_posts; un += n_halo_thr)
            note_missing(A.words + (size_t)un * 2 * SU_LINE + par * SU_LINE, s, un);
        }
      }
      __syncthreads();
      if (tid == 0) {
        if (atomicCAS(&A.bar->to_site, 0, s_to) == 0) {
          A.bar->to_iter = (unsigned)it;
          A.bar->to_seen = s_seen;
          A.bar->to_index = s_widx;
          A.bar->to_cta = (int)blockIdx.x;
        }
        atomicExch(&A.bar->timeout, 1);
      }
      return;
    }
    // ---- the scene's sums (tiles lane-strided over a warp, its tree) and the scalar step
    if (warp == 0) {
      float acc[3] = {0.f, 0.f, 0.f};
      for (int t = lane; t < n_tiles; t += 32)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float* v = L.w + (q * n_tiles + t) * per_tile;
          if constexpr (per_tile == 4) {
            const float4 p4 = *reinterpret_cast<const float4*>(v);
            acc[q] += (p4.x + p4.y) + (p4.z + p4.w);
          } else if constexpr (per_tile == 2) {
            const float2 p2 = *reinterpret_cast<const float2*>(v);
            acc[q] += p2.x + p2.y;
          } else {
            acc[q] += v[0];
          }
        }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
#pragma unroll
        for (int q = 0; q < 3; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], d);
      if (lane == 0)
        sr_step_fast(st, acc[0], acc[1], acc[2], it == 0 && s_nh < 0 ? 1.0f : 0.0f, it, tol2, max_iter);
    }
    __syncthreads();
    if (st.done) break;
    // ---- p = u + beta p, x += alpha p, s = w + beta s, r -= alpha s, u = M r; the halo rows without p and x
    const float a = st.alpha, b = st.beta;
    if (mine) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        upd_px(a, b, u[c], p[c], x[c]);
        upd_sr(a, b, w[0][c], sv[0][c], r[0][c]);
      }
      prec6(P[0], r[0], u);
      L.u[my_item] = make_float4(u[0], u[1], u[2], 0.0f);
    } else if (halo_thr) {
#pragma unroll
      for (int k = 0; k < HPT; ++k)
        if (hrow[k] >= 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) upd_sr(a, b, w[k][c], sv[k][c], r[k][c]);
          float uu[3];
          prec6(P[k], r[k], uu);
          L.u[hitem[k]] = make_float4(uu[0], uu[1], uu[2], 0.0f);
        }
    }
    if (tid == 0) st.iters += 1;
  }

  if (own) st_v(S.dx + my_i, mk<float4, float>(x[0], x[1], x[2]));
  if (blockIdx.x == 0 && tid == 0) publish(st, S.ctl);
}

// before a solve: the barrier and the stamped words, which carry stamps of one launch only
__global__ void k_su_clear(SuLaunch A) {
  const int n_thr = gridDim.x * blockDim.x, t0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (t0 == 0) *A.bar = GridBar{};
  const ulonglong2 zero = make_ulonglong2(0, 0);
  ulonglong2 *w = reinterpret_cast<ulonglong2*>(A.words), *z = reinterpret_cast<ulonglong2*>(A.scene->zrec);
  for (int k = t0; k < A.plan.n_posts * 2 * SU_LINE; k += n_thr) w[k] = zero;
  for (int k = t0; k < 2 * A.plan.nv; k += n_thr) z[k] = zero;
}

static const void* su_kernel(int rows, int hpt) {
  if (rows == 32) return hpt == 1 ? (const void*)k_pcg_su<32, 1> : (const void*)k_pcg_su<32, 2>;
  if (rows == 64) return hpt == 1 ? (const void*)k_pcg_su<64, 1> : (const void*)k_pcg_su<64, 2>;
  return hpt == 1 ? (const void*)k_pcg_su<128, 1> : (const void*)k_pcg_su<128, 2>;
}

int pcg_su_hpt(const RdPlan& p, int nh) {
  const int thr = SU_NT - 2 * p.post_rows;
  return p.post_rows > PCG_TILE ? 0 : nh <= thr ? 1 : nh <= 2 * thr ? 2 : 0;
}

int pcg_su_max_grid(int device, size_t smem, int rows, int hpt) {
  const void* k = su_kernel(rows, hpt);
  int n_sm = 0, per_sm = 0;
  if (allow_shared(k, smem) != cudaSuccess ||
      cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, SU_NT, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * n_sm;
}

cudaError_t launch_pcg_su(const SuLaunch& L, cudaStream_t st) {
  const RdPlan& p = L.plan;
  const int hpt = pcg_su_hpt(p, L.halo_cap);
  if (!L.scene || !L.bar || !L.words || p.nv <= 0 ||
      (p.post_rows != 32 && p.post_rows != 64 && p.post_rows != PCG_TILE) ||
      p.n_posts != (p.nv + p.post_rows - 1) / p.post_rows || p.grid != p.n_posts || !hpt)
    return cudaErrorInvalidValue;
  k_su_clear<<<std::min(sm_count(), 1 + p.nv / 64), 256, 0, st>>>(L);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const void* k = su_kernel(p.post_rows, hpt);
  e = allow_shared(k, L.smem_bytes);
  if (e != cudaSuccess) return e;
  SuLaunch a = L;
  void* args[] = {(void*)&a};
  return cudaLaunchCooperativeKernel(k, dim3(p.grid), dim3(SU_NT), args, L.smem_bytes, st);
}

}  // namespace ppn
