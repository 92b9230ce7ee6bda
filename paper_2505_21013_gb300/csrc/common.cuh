// Device-side data layout shared by every kernel of the library.
//
// A launch covers one or more scenes.  Each scene is described by a SceneDev
// record in device memory; work is cut into fixed-size tiles of one scene
// (TILE tets or vertices, PCG_TILE matrix rows) and a launch gets a table of
// TileRef entries, one CTA (or one PCG work unit) per tile.  Reductions write
// one partial per tile and are summed per scene in tile order, so a scene's
// arithmetic is the same whether it runs alone or inside a batch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "tetmath.cuh"

namespace ppn {

constexpr int TILE = 256;      // tets or vertices per element/vertex tile (= CTA size)
constexpr int PCG_TILE = 128;  // BSR rows per PCG reduction tile
constexpr int HE_STRIDE = 96;  // values per element Hessian record (10 blocks x 9, padded)
constexpr int GE_STRIDE = 12;  // values per element gradient record
constexpr int TETC_STRIDE = 12;  // Dm^-1 (9), V, mu, lam_s
constexpr int SELL_STEP = 320;   // words of a block step: 32 x 4 (values 0..3), 32 x 4 (4..7), 32 (8), 32 columns

template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<double> { using type = double4; };
template <typename T> using vec4_t = typename Vec4<T>::type;

// analytic obstacle of the contact model (contact.cuh)
constexpr int OBST_PLANE = 0, OBST_CYLINDER_IN = 1, OBST_SPHERE_OUT = 2;
constexpr int MAX_OBST = 8;
struct ObstDev {
  int type, pad;
  double p[3];  // plane point / axis point / centre
  double a[3];  // plane unit normal / cylinder unit axis
  double r;     // radius
};
struct ObstSet {  // a scene's obstacles, in device memory (updated between steps)
  int n, pad;
  ObstDev o[MAX_OBST];
};

// Per-scene control block: written by kernels, copied to the host at sync points.
struct Ctl {
  double grad[4];        // ||g||_2^2, ||s||_2^2 (residual scale), contact elements, ||g||_inf
  double ccd;            // 1 / (first contact time along dx), from the contact-time kernel
  double gap[4];         // 1 / (smallest free-vertex distance) to obstacles k0..k0+3 (inf: not feasible)
  double energy[3];      // incremental potential, g^T dx, max |dx| over free vertices
  double pcg_rr0, pcg_rr, pcg_rz, pcg_dq, pcg_alpha, pcg_beta;
  int n_new;             // elements selected by the last selection
  int n_new_c;           // contact elements selected by the last selection
  int n_ties;            // selection ties of the last selection (|r_e - delta| <= tie_band delta)
  int n_touched;         // BSR blocks touched by the elements of the last selection (incremental update)
  int pcg_iters;         // CG updates performed (x = sum of alpha d)
  int pcg_ind;           // negative curvature or a non-SPD diagonal block
  int pcg_precond_fail;
  int pcg_hit_max;
  int pcg_done;
  int error;             // bit flags, see kErr*
  int pad0;
  unsigned tiles_done[5];  // last-tile counters of the reductions (gradient, energy, ccd, gap, g^T dx)
};

constexpr int kErrTimeout = 1;
constexpr int kErrNonFinite = 2;

template <typename T>
struct SceneDev {
  // sizes
  int nv, nt, nnzb, nmap;
  int n_vtiles, n_ttiles, n_ptiles;  // vertex, tet and PCG-row tiles
  // constant geometry and topology
  const int4* tets;
  const T* tetc;           // nt x TETC_STRIDE
  const double* mass;      // nv
  const uint8_t* fixed;    // nv
  const double4* X;        // nv rest positions
  const int* vt_ptr;       // nv+1 vertex -> incident (tet << 2 | corner)
  const int* vt_src;
  const int* row_ptr;      // nv+1 BSR rows
  const int* col;          // nnzb
  const int* blk_row;      // nnzb
  const int* blk_ptr;      // nnzb+1 block -> contributions (tet << 4 | a << 2 | b)
  const int* blk_src;
  const unsigned char* blk_lane;  // nmap: the block of each contribution, modulo 32 (its lane in k_assemble)
  const int* diag_idx;     // nv
  const int* tet_blk;      // nt x 16: BSR block of each (a, b) corner pair of a tet
  // state
  double4* u;              // displacement x - X
  double4* u_n;
  double4* vel;
  double4* uhat;           // xhat - X
  double4* u_probe;        // scratch displacement for probes
  // per-iteration
  double* ge;              // nt x GE_STRIDE element gradients (FP64 in both precisions)
  T* He;                   // nt x HE_STRIDE
  T* dH;                   // nt x HE_STRIDE, clamping updates
  double4* g;              // assembled gradient
  double* gmax;            // per-vertex |g_v|_inf
  T* val;                  // BSR values, component-major: val[c * nnzb + k]
  int* proj_stamp;         // Newton-iteration id at which the element was projected
  int* round_stamp;        // selection-round id at which it was projected
  int* sel_list;           // compacted newly selected elements
  int* blk_mark;           // nnzb: selection round that last listed the block as touched
  int* touched;            // nnzb: blocks touched by the last selection (n_touched of them)
  // PCG vectors (nv each) and block-Jacobi inverse (nv x 9)
  vec4_t<T>* dx;
  vec4_t<T>* r;
  vec4_t<T>* z;
  vec4_t<T>* q;
  vec4_t<T>* d0;
  vec4_t<T>* d1;
  T* Pinv;
  // reduction scratch: partials[tile * 4 + k]
  double* vpart;           // vertex tiles
  double* tpart;           // tet tiles
  double* ppart;           // PCG tiles
  unsigned long long* pword;  // PCG tile partials as stamped words, [4][n_ptiles][<= 2]
  const int* gstep;           // FP32 path: ceil(nv / 16) + 1 first block steps of the 16-row groups (streamed PCG layouts)
  T* steps;                   // FP32 path: room for the blocks by step (SELL_STEP words each), or null; the memory of
                              // dH, which nothing reads between a solve's start and the next projection
  T* zrec;                    // FP32 path: [2][nv] 32-byte records {z, 0, d_prev, 0} of the resident PCG
  double* psi_out;         // optional per-element energies (probes)
  Ctl* ctl;
  // scalars of the current phase
  double dt, inv_dt2;
  double grav[3];
  double delta, eps_delta, eig_eps;
  double tie_band;         // relative half-width of the tie band around delta (counted, not selected)
  double gamma;
  double pcg_tol2;
  int pcg_max_iter;
  int it_id, round_id;
  int mode;
  int proj_kind;           // ppn_projection: 0 clamp, 1 mirror
  int init_guess;          // 0: x_n ; 1: x_n + dt v_n
  // contact against analytic obstacles
  const ObstSet* obs;       // device: the scene's obstacles (obs->n = 0: no contact)
  double kappa, dhat;
  int* cproj_stamp;        // nv: Newton-iteration id at which the contact element was projected
  int* cround_stamp;       // nv: selection round of that projection
  T* dHc;                  // nv x 9: clamping update of the contact element
  T* Hc;                   // nv x 9: Hessian of the vertex's contact potential at the iterate of the last gradient
  // Dirichlet by penalty (pen_k > 0): constrained vertices are free and carry pen_k m / (2 dt^2) |u - t|^2
  double pen_k;
  const uint8_t* con;      // nv: 1 for a constrained vertex
  double4* tgt;            // nv: its target displacement
  int active;              // the scene takes part in the current launch
};

struct TileRef {
  int scene;
  int tile;
};

// Spacing, in 64-bit words, of the stamped tile partials of the single-reduction PCG.
// Every CTA polls every tile's word once per CG iteration; packed 16 to a 128-byte L2
// line, the words of a few hundred tiles sit in a few dozen lines that all 152 SMs poll
// at once, and the requests queue at those lines' L2 slices.  One word per line spreads
// them over the slices (a 250-tile reduction fell from 4.2 to 1.4 us per iteration in
// a same-box A/B); past a few hundred tiles the extra lines cost more than the queueing,
// and two words per 16 bytes measured best (2000 tiles).  The partials' array holds
// 8 x n_ptiles x pword_stride(n_ptiles) words.
__host__ __device__ inline int pword_stride(int n_ptiles) { return n_ptiles <= 512 ? 16 : 2; }

// ---- small helpers ----
__device__ __forceinline__ double4 ld_d4(const double4* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  double2 a = q[0], b = q[1];
  return make_double4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_d4(double4* p, double4 v) {
  double2* q = reinterpret_cast<double2*>(p);
  q[0] = make_double2(v.x, v.y);
  q[1] = make_double2(v.z, v.w);
}

// FP32 to FP64 by moving bits: a conversion instruction costs an FP64 issue slot (64 cycles
// of a warp's sub-partition), twelve integer ones about a third of that.  Zeros are handled,
// denormals, infinities and NaN (any of the N) take the instruction.
template <int N>
__device__ __forceinline__ void widen(const float* x, double* d) {
  bool odd = false;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const unsigned m = __float_as_uint(x[k]) & 0x7fffffffu;
    odd |= m != 0u && m - 0x00800000u >= 0x7f000000u;
  }
  if (odd) {
#pragma unroll
    for (int k = 0; k < N; ++k) d[k] = (double)x[k];
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned b = __float_as_uint(x[k]), m = b & 0x7fffffffu;
      d[k] = __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(b << 29));
    }
  }
}
template <int N>
__device__ __forceinline__ void widen(const double* x, double* d) {
#pragma unroll
  for (int k = 0; k < N; ++k) d[k] = x[k];
}

// Fixed-order reductions of K values per thread over a CTA of TILE threads (N_SUM sums, then
// maxima, which are of values >= 0: negative ones and NaN count as 0).  An FP64 instruction
// costs a warp 64 cycles however few of its lanes matter, so the sums of a warp share the
// lanes after their first steps (5 additions for two sums, 6 for four, instead of 5 each),
// the second stage takes all K values at once, and maxima compare bits as integers.  The
// sums' tree is that of a shuffle-down per value: offsets 16, 8, 4, 2, 1, twice.
// Result k in lane 8 k of warp 0; sm: 8 K doubles.
__device__ __forceinline__ double max_bits(double a, double b) {  // of two results of max_clamp
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return x > y ? a : b;
}
__device__ __forceinline__ double max_clamp(double a) {
  const long long x = __double_as_longlong(a);
  return x < 0 || x > 0x7ff0000000000000ll ? 0.0 : a;
}
template <int K, int N_SUM>
__device__ __forceinline__ double block_reduce(const double* v, double* sm) {
  static_assert(TILE == 256 && K <= 4 && N_SUM <= K, "eight warps, four groups of eight lanes");
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  auto xadd = [](double x, int o) { return x + __shfl_xor_sync(0xffffffffu, x, o); };
  // two sums into one register: lanes with bit o clear go on with a, the others with b
  auto fold = [&](double a, double b, int o) {
    return (l & o ? b : a) + __shfl_xor_sync(0xffffffffu, l & o ? a : b, o);
  };
  if constexpr (N_SUM > 0) {
    double x;
    if constexpr (N_SUM == 1) {
      x = xadd(xadd(v[0], 16), 8);
    } else if constexpr (N_SUM == 2) {
      x = xadd(fold(v[0], v[1], 16), 8);
    } else {
      double d = 0.0;
      if constexpr (N_SUM > 3) d = v[3];
      x = fold(fold(v[0], v[1], 16), fold(v[2], d, 16), 8);
    }
    x = xadd(xadd(xadd(x, 4), 2), 1);
    const int k = N_SUM == 1 ? l : N_SUM == 2 ? (l >> 4) + (l & 15) * 4 : (l >> 4) + ((l >> 2) & 2) + (l & 7) * 4;
    if (k < N_SUM) sm[8 * k + w] = x;
  }
#pragma unroll
  for (int k = N_SUM; k < K; ++k) {
    double x = max_clamp(v[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = max_bits(x, __shfl_xor_sync(0xffffffffu, x, o));
    if (l == 0) sm[8 * k + w] = x;
  }
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    double x = l < 8 * K ? sm[l] : 0.0, m = x;
    if constexpr (N_SUM > 0) x = xadd(xadd(xadd(x + 0.0, 4), 2), 1);
    if constexpr (N_SUM < K)
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
    r = l < 8 * N_SUM ? x : m;
  }
  return r;
}

// A per-scene reduction: the CTA writes its tile's K results to part[tile * 4 + k]; the CTA
// that completes the count reduces them in tile order and writes out[0..K).
template <int K, int N_SUM>
__device__ __forceinline__ void scene_reduce(const double* v, double* part, int tile, unsigned* counter, int n_tiles,
                                             double* out) {
  __shared__ double sm[8 * K];
  __shared__ int is_last;
  const int l = threadIdx.x & 31;
  const double r = block_reduce<K, N_SUM>(v, sm);
  if (threadIdx.x < 32) {
    if (l < 8 * K && (l & 7) == 0) part[4 * tile + (l >> 3)] = r;
    __syncwarp();
    if (l == 0) {  // the counting lane's fence, after the barrier, covers the other lanes' stores
      __threadfence();
      is_last = atomicAdd(counter, 1u) == (unsigned)(n_tiles - 1);
    }
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[k] = 0.0;
  // thread t takes tiles t, t + TILE, ... in order; then a fixed tree
  for (int t = threadIdx.x; t < n_tiles; t += TILE) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const double x = __ldcg(part + 4 * t + k);
      if (k < N_SUM)
        acc[k] = t < TILE ? x : acc[k] + x;
      else
        acc[k] = max_bits(acc[k], x);
    }
  }
  const double tot = block_reduce<K, N_SUM>(acc, sm);
  if (threadIdx.x < 32 && l < 8 * K && (l & 7) == 0) out[l >> 3] = tot;
  if (threadIdx.x == 0) *counter = 0u;
}

}  // namespace ppn
