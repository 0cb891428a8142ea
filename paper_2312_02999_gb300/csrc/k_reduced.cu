// Reduced contact system of Sec. 3.2.
//
// Eq. 10-11: Sigma-hat^-1 y2 = u - Sigma^-1 Q^T v with u = Sigma^-1 y2 and,
// in the push-through form (B-check is PSD and usually singular, so it is
// never inverted), v = (I + B S)^-1 B u_c, S = Sigma^-1[c, c] (x) I_3.  With
// S = L L^T (L = L_s (x) I_3) this is v = L^-T (I + L^T B L)^-1 L^T B u_c and
// I + L^T B L is SPD with eigenvalues >= 1, so both factorisations are plain
// Cholesky.  Steps:
//   1 gather S = Sigma^-1[c,c], the block-row lists of B
//   2 S = L_s L_s^T
//   3 X = B (L_s (x) I_3)
//   4 N = I + (L_s (x) I_3)^T X
//   5 N = L_N L_N^T
//   6 y = B u_c, v = (L_s (x) I_3)^-T N^-1 (L_s (x) I_3)^T y
//   7 refinement, rho = y - v - B (S v) in float64, v += L^-T N^-1 L^T rho:
//     one step with float64 factors (it takes back what solving with explicit
//     inverse factors loses against substitution); float32 factors refine to
//     a stopping test.  The error of v reaches the global residual as
//     Q^T rho itself, so the stopping test compares |rho| with |y2| (the
//     Schur right-hand side), not with |y| = |B u_c|, which carries the
//     barrier stiffness and can be many orders larger.  At most
//     kMixedRefineSteps steps: where cond(N) nears 1 / u32 (a pair at
//     ~1e-3 d0 with every vertex of the reduced set in contact) a float32
//     factor gains only 4-10x per step, and 4 steps left |rho| near
//     1e-3 |y2|; the stopping rule ends well-conditioned solves after 1-2.
//     Beyond cond(N) of a few 1e6 a step may gain nothing or lose (a pair at 5.7e-4
//     d0: |rho| 2 to 40 |y2|, with every pivot positive), so the v of the smaller
//     residual is kept and, if that is above kAcceptRho |y2|, the solve is
//     reported (kInfoStalled): the caller solves it again with float64 factors.
//   8 z2 = u - (Sigma^-1[:, c] (x) I_3) v
// Steps 1-5 need only B-check and Sigma^-1, so they run on a side stream while
// the forward solve makes u.  Two forms: the grid form (float64, and float32
// with n_c > 128), and for float32 n_c <= 128 the one-CTA and cluster kernels
// k_small_s/x/n/v, k_clus_v, k_small_u and k_small_solve.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <utility>
#include <vector>

#include "df64.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace fsim {

namespace {

constexpr int kRT = 256;   // threads per CTA
// Largest |rho| / |y2| a refined float32 solve may leave: rho reaches the step as
// (Sigma + B)^-1 rho.  Solves with cond(N) below 1e6 end at 1e-7 or less, those that
// stop gaining end at 1e-3 to 40, so the line may lie anywhere between.
constexpr double kAcceptRho = 1e-5;

// Padded packed lower storage: row i holds columns 0..i, padded to a
// multiple of 4 floats, so 32-column segments of a row are 16-byte aligned.
__host__ __device__ constexpr int prow(int i) {
  const int q = i >> 2;
  return 8 * q * (q + 1) + (i - 4 * q) * 4 * (q + 1);
}

template <typename FT>
struct RedArgs {
  int nc, n2, refine;
  const int* nc_dev;    // n_c on the device (set by the contact-marking scan)
  FT* base;             // FT workspace: S, X, N, 1/diag, FT vectors (offsets from n_c)
  double* dtail_end;    // end of the float64 workspace; float64 vectors sit before it
  int* ibase;           // int workspace after the block occupancy: lists, counts
  const int* clist;
  const double* Sinv;   // n2 x n2
  const double* Bc;     // (3nc)^2, row-major
  const int* bocc;      // nc x nc block occupancy
  int* list;            // nc x nc block-row lists
  int* cnt;             // nc
  const double* u;      // n2 * 3
  const FT* y2;         // n2 * 3: right-hand side of the Schur system (u = Sigma^-1 y2)
  double* z2;           // n2 * 3 (out)
  FT* S;                // nc x nc  -> L_s
  FT* X;                // n3 x n3, then L_N^-1
  FT* N;                // packed lower N -> L_N, diagonal blocks inverted
  FT* Vs;               // small forms: nc x nc L_s^-1
  FT* fv;               // 2 * n3 scratch in FT
  double* y;            // n3: B u_c
  double* v;            // n3
  double* rho;          // n3
  double* w;            // n3
  double* vp;           // n3: v before the last refinement step
  double* nrm;          // 3: |rho|^2 of a refinement step (two slots), |y2|^2
  double* S64;          // small forms: Sigma^-1[c, c] in float64 (n_c x n_c)
  int* info;
  int small_lim;        // n_c handled by the small forms (0: none)
  int active;           // lock-step batches: the frame takes part in the launch
  int one_cta_max;      // largest n_c of the one-CTA path (float32 factors); the
                        // 4-CTA cluster takes n_c up to kClusNc above it
  FT* spk;              // small forms: L_s packed, its diagonal blocks inverted
  unsigned* bar;        // grid form: counters of its two kernels' barriers
};

// Offsets of the workspace for a given n_c (every kernel of the reduced solve
// derives them from the n_c it reads on the device).  red_tail: the float64
// vectors and the block lists, where both forms have them; red_layout: those
// and the matrices of the one-CTA and cluster forms.
template <typename FT>
__device__ __forceinline__ void red_tail(RedArgs<FT>& a, int nc) {
  const int n3 = 3 * nc;
  a.nc = nc;
  a.y = a.dtail_end - 5 * (size_t)n3 - 8;
  a.v = a.y + n3; a.rho = a.v + n3; a.w = a.rho + n3; a.vp = a.w + n3; a.nrm = a.vp + n3;
  a.S64 = a.y - (size_t)nc * nc;
  a.list = a.ibase;
  a.cnt = a.list + (size_t)nc * nc;
}
template <typename FT>
__device__ __forceinline__ void red_layout(RedArgs<FT>& a, int nc) {
  const int n3 = 3 * nc;
  red_tail(a, nc);
  // every segment starts on a 16-byte boundary (vector loads)
  constexpr size_t q = 16 / sizeof(FT);
  auto al = [](size_t x) { return (x + q - 1) / q * q; };
  a.S = a.base;
  a.X = a.S + al((size_t)nc * nc);
  a.N = a.X + al((size_t)n3 * n3);
  a.Vs = a.N + al(prow(n3));
  a.fv = a.Vs + al((size_t)nc * nc);
  a.spk = a.fv + al(2 * (size_t)n3);
}

// z2 = u - (Sigma^-1[:, c] (x) I_3) v, one warp per row (warp w of nw): the
// form for a single frame, which has few rows to spread over the GPU
template <typename FT>
__device__ void z2_update(const RedArgs<FT>& a, int nc, int w, int nw) {
  const int lane = threadIdx.x & 31;
  for (int q = w; q < a.n2; q += nw) {
    const double* srow = a.Sinv + (size_t)q * a.n2;
    double a0 = 0, a1 = 0, a2 = 0;
    for (int m = lane; m < nc; m += 32) {
      if (!FSIM_CHECK_IDX(a.clist[m], a.n2, CHECK_CLIST)) continue;
      const double sv = srow[a.clist[m]];
      a0 += sv * a.v[3 * m]; a1 += sv * a.v[3 * m + 1]; a2 += sv * a.v[3 * m + 2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      a1 += __shfl_xor_sync(0xffffffffu, a1, o);
      a2 += __shfl_xor_sync(0xffffffffu, a2, o);
    }
    if (lane == 0) {
      a.z2[3 * q] = a.u[3 * q] - a0;
      a.z2[3 * q + 1] = a.u[3 * q + 1] - a1;
      a.z2[3 * q + 2] = a.u[3 * q + 2] - a2;
    }
  }
}

// The same with one row per lane (warp w of nw takes rows 32 w .. 32 w + 31,
// then strides by 32 nw): the form for batches, whose frames together give
// enough warps.  Sigma^-1 is stored exactly symmetric (both triangles from
// one product), so row q's entries at the contact columns are read as
// Sigma^-1[c_m][q]: consecutive lanes read consecutive addresses and no
// cross-lane reduction is needed (each float64 warp instruction costs about
// 64 cycles of its SM sub-partition on GB300, so this halves the cost)
template <typename FT>
__device__ void z2_update_rows(const RedArgs<FT>& a, int nc, int w, int nw) {
  const int lane = threadIdx.x & 31;
  for (int q0 = 32 * w; q0 < a.n2; q0 += 32 * nw) {
    const int q = q0 + lane;
    if (q >= a.n2) continue;
    double a0 = 0, a1 = 0, a2 = 0;
    for (int m = 0; m < nc; ++m) {
      const int c = a.clist[m];
      if (!FSIM_CHECK_IDX(c, a.n2, CHECK_CLIST)) continue;
      const double sv = a.Sinv[(size_t)c * a.n2 + q];
      a0 += sv * a.v[3 * m]; a1 += sv * a.v[3 * m + 1]; a2 += sv * a.v[3 * m + 2];
    }
    a.z2[3 * q] = a.u[3 * q] - a0;
    a.z2[3 * q + 1] = a.u[3 * q + 1] - a1;
    a.z2[3 * q + 2] = a.u[3 * q + 2] - a2;
  }
}

// The z2 update alone (plain launch) after the one-CTA or cluster path; with
// n_c = 0 it copies z2 = u.
__device__ __forceinline__ void k_z2_update_body(RedArgs<float> a, bool rows) {
  const int nc = *a.nc_dev;
  if (nc == 0) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 3 * a.n2; e += gridDim.x * blockDim.x)
      a.z2[e] = a.u[e];
    return;
  }
  if (nc > a.small_lim) return;         // the grid form updates its own z2
  red_layout(a, nc);
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  if (rows) z2_update_rows(a, nc, w, nw);
  else z2_update(a, nc, w, nw);
}
__global__ void __launch_bounds__(256) k_z2_update(RedArgs<float> a) {
  k_z2_update_body(a, false);
}

// ---------------------------------------------------------------------------
// Diagonal blocks and panels of the grid form.
// ---------------------------------------------------------------------------
constexpr int kBk = 32;                     // block edge

// x 2^-e and the significand of x (x = m 2^e, 1 <= m < 2), x positive and normal
__device__ __forceinline__ int exponent_of(float x) {
  return ((__float_as_int(x) >> 23) & 255) - 127;
}
__device__ __forceinline__ float significand(float x) {
  return __int_as_float((__float_as_int(x) & 0x007fffff) | 0x3f800000);
}
__device__ __forceinline__ float scale_down(float x, int e) {
  return x * __int_as_float((127 - max(-126, min(126, e))) << 23);
}
__device__ __forceinline__ int exponent_of(double x) {
  return ((__double2hiint(x) >> 20) & 2047) - 1023;
}
__device__ __forceinline__ double significand(double x) {
  return __hiloint2double((__double2hiint(x) & 0x000fffff) | 0x3ff00000, __double2loint(x));
}
__device__ __forceinline__ double scale_down(double x, int e) {   // integer work only
  const int h = __double2hiint(x), ne = ((h >> 20) & 2047) - e;
  return ne > 0 && ne < 2047 && ((h >> 20) & 2047) != 0
             ? __hiloint2double(h - (int)((unsigned)e << 20), __double2loint(x))
             : 0.0;
}
__device__ __forceinline__ float rsqrt_ft(float v) {
  float r = rsqrtf(v);
  return r * (1.5f - 0.5f * v * r * r);
}

// element e of the lower triangle of a 32 x 32 block, columns from the last to
// the first: the elements of the columns > j are then the first ones, so that
// the work left after column j fills whole warps
__device__ __forceinline__ void tri_element(int e, int& r, int& c) {
  int m = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);      // column 31 - m holds m + 1 elements
  while ((m + 1) * (m + 2) / 2 <= e) ++m;
  while (m * (m + 1) / 2 > e) --m;
  c = kBk - 1 - m;
  r = c + e - m * (m + 1) / 2;
}

// A panel's diagonal factor (Lt[q][r] = L[r][q], dv = 1 / diag) and the columns of
// its elimination.
struct ChSm {
  float Lt[32][32];
  float dv[32], rs[32];
  float col[32][33];
};
constexpr int kDT = 256;                   // threads of diag_factor (the whole CTA)

// Factor of the diagonal block with entries load(r, c) - P_r . P_c (r >= c; P the
// panel before, transposed: P_r[l] = Pt[l ldp + r], none if Pt is null), into
// sm.Lt / sm.dv and store(r, c, L[r][c]).  The elimination is free of divisions:
// with pivot p = ph 2^e (1 <= ph < 2),
//   D[r][c] <- D[r][c] ph - D[r][j] (D[c][j] 2^-e),
// which is the Schur complement times ph, so that after column j every entry
// carries the product of the ph so far (at most 2^31).  A column then costs two
// dependent operations and one barrier; the square roots of all columns are
// taken at once at the end.  Every thread owns two elements of the triangle (16
// threads a third one, in column 0, which no step changes).
template <typename Load, typename Store>
__device__ __forceinline__ void diag_factor(ChSm& sm, const float* Pt, int ldp, int* info,
                                            Load load, Store store) {
  const int tid = threadIdx.x;
  float v[3];
  int er[3], ec[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int e = tid + q * kDT;
    er[q] = 0;
    ec[q] = -1;
    if (e >= 32 * 33 / 2) continue;
    tri_element(e, er[q], ec[q]);
    float x = load(er[q], ec[q]);
    if (Pt) {
      float a0 = 0.f, a1 = 0.f;
#pragma unroll 8
      for (int l = 0; l < 32; l += 2) {
        a0 += Pt[l * ldp + er[q]] * Pt[l * ldp + ec[q]];
        a1 += Pt[(l + 1) * ldp + er[q]] * Pt[(l + 1) * ldp + ec[q]];
      }
      x -= a0 + a1;
    }
    v[q] = x;
    if (ec[q] == 0) sm.col[0][er[q]] = x;
  }
  for (int j = 0; j + 1 < 32; ++j) {
    __syncthreads();
    if (ec[0] <= j && ec[1] <= j) continue;
    float p = sm.col[j][j];
    if (!(p > 0.f)) p = 1.f;                         // reported below
    const int e = exponent_of(p);
    const float ph = significand(p);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (ec[q] <= j) continue;
      const float w = scale_down(sm.col[j][ec[q]], e);
      v[q] = v[q] * ph - sm.col[j][er[q]] * w;
      if (ec[q] == j + 1) sm.col[j + 1][er[q]] = v[q];
    }
  }
  __syncthreads();
  if (tid < 32) {
    float p = sm.col[tid][tid];
    const bool bad = !(p > 0.f);
    if (bad) { atomicOr(info, kInfoPivot); p = 1.f; }
    float pi = significand(p);
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const float x = __shfl_up_sync(0xffffffffu, pi, s);
      if (tid >= s) pi *= x;
    }
    pi = __shfl_up_sync(0xffffffffu, pi, 1);
    if (tid == 0) pi = 1.f;
    const float rs = rsqrt_ft(p * pi);
    sm.rs[tid] = rs;
    sm.dv[tid] = pi * rs;
    if (bad) sm.col[tid][tid] = 1.f;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (ec[q] < 0) continue;
    const float x = sm.col[ec[q]][er[q]] * sm.rs[ec[q]];
    sm.Lt[ec[q]][er[q]] = x;
    store(er[q], ec[q], x);
  }
}

// x L_kk^T = a for one row in registers (right-looking: the dependent chain is
// one FMA per column; four entries of the factor per shared-memory read)
__device__ __forceinline__ void panel_row(const ChSm& sm, float x[32]) {
#pragma unroll
  for (int q = 0; q < 32; ++q) {
    x[q] *= sm.dv[q];
#pragma unroll
    for (int l4 = (q + 1) / 4; l4 < 8; ++l4) {
      const float4 f = *reinterpret_cast<const float4*>(&sm.Lt[q][4 * l4]);
      const float fv[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (4 * l4 + u > q) x[4 * l4 + u] -= x[q] * fv[u];
    }
  }
}

// ---------------------------------------------------------------------------
// Grid form: n_c of any size, float64 or float32 factors, the matrices in
// global memory (L2) and G CTAs per system.
//
// k_grid_prepare does steps 1-5.  The time of a blocked Cholesky this small
// (32 ceil(n / 32), n = 3 n_c of a few hundred) is its chain of panels, so each
// panel is two phases with a barrier after each, and its serial part, the
// 32 x 32 diagonal factor, is made by CTA 0 while the other CTAs update the
// trailing tiles (look-ahead).  The identity is carried along below the
// matrix: its rows become U = L^-T, so every later solve is two products with
// U, which spread over the grid, in place of a chain of 2 n / 32 dependent
// blocks.  The matrices are padded to whole blocks by the identity.
// k_grid_solve does steps 6-8 once u is known.
//
// Measured (one system, all SMs): float64 n_c = 93: 311 us of preparation, of
// which the forward solve covers about 200, and 48 us of solve, where one
// launch after the forward solve took 723 us (a diagonal factor with three
// barriers per column, one-CTA solves); float32 n_c = 242: 426 + 105 us from
// 1,676.  A batch's systems run side by side, each on a share of the CTAs,
// where they ran one after the other (60k face, 8 frames, two of them with
// n_c > 128: 1,760 -> 375 us per iteration).
// ---------------------------------------------------------------------------
constexpr int kSpinLimit = 1 << 21;         // polls of a barrier before it gives up (about a second)

// systems of a launch: grid = G n CTAs, CTA b works on system b / G
struct GridFrames {
  static constexpr int kMax = 64;
  int n, G;
  unsigned char id[kMax];
};

template <typename FT>
struct GridLay {
  int nc, n3, nbs, nbn, lds, ldn;
  FT *S, *Us, *N, *U, *dg, *t, *l;
};
template <typename FT>
__host__ __device__ __forceinline__ GridLay<FT> grid_layout(FT* base, int nc) {
  GridLay<FT> g;
  g.nc = nc;
  g.n3 = 3 * nc;
  g.nbs = (nc + kBk - 1) / kBk;
  g.nbn = (g.n3 + kBk - 1) / kBk;
  g.lds = g.nbs * kBk;
  g.ldn = g.nbn * kBk;
  g.S = base;                                   // L_s
  g.Us = g.S + (size_t)g.lds * g.lds;           // L_s^-T
  g.N = g.Us + (size_t)g.lds * g.lds;           // L_N
  g.U = g.N + (size_t)g.ldn * g.ldn;            // X, then L_N^-T
  g.dg = g.U + (size_t)g.ldn * g.ldn;           // two diagonal factors (by parity) + 1 / diag
  g.t = g.dg + 2 * (kBk * kBk + kBk);           // vectors of ldn
  g.l = g.t + g.ldn;
  return g;
}
int64_t grid_front_elems(int nc) {
  const GridLay<float> g = grid_layout<float>(nullptr, nc);
  return (int64_t)2 * g.lds * g.lds + 2 * (int64_t)g.ldn * g.ldn + 2 * (kBk * kBk + kBk) +
         2 * (int64_t)g.ldn + 16;
}

// Barrier of a system's CTAs: a counter that only grows within the launch
// (the last CTA to leave resets it).  All CTAs are resident (cooperative
// launch).  A wait that runs out sets the info flag, and the CTA waits no more.
struct GroupBar {
  unsigned* word;       // [0] arrivals, [1] departures
  unsigned target;
  int G;
  int* info;
  bool dead;
};
__device__ __forceinline__ void group_sync(GroupBar& b) {
  __syncthreads();
  if (b.G > 1) {
    if (threadIdx.x == 0) {
      b.target += b.G;
      __threadfence();
      atomicAdd(b.word, 1u);
      int polls = 0;
      while (!b.dead) {
        unsigned v;
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(b.word) : "memory");
        if ((int)(v - b.target) >= 0) break;
        if (++polls > kSpinLimit) {
          atomicOr(b.info, kInfoTimeout);
          b.dead = true;
        }
      }
      __threadfence();
    }
    __syncthreads();
  }
}
// arrive without waiting (the CTA's stores before it are published)
__device__ __forceinline__ void group_arrive(GroupBar& b) {
  __syncthreads();
  if (threadIdx.x == 0 && b.G > 1) {
    b.target += b.G;
    __threadfence();
    atomicAdd(b.word, 1u);
  }
}
// the last CTA to leave resets the counters (of `more` too)
__device__ __forceinline__ void group_leave(GroupBar& b, unsigned* more) {
  __syncthreads();
  if (threadIdx.x == 0 && b.G > 1) {
    __threadfence();
    if (atomicAdd(b.word + 1, 1u) == (unsigned)b.G - 1u) {
      b.word[0] = 0;
      b.word[1] = 0;
      if (more) more[0] = 0;
      __threadfence();
    }
  }
}

// cross-CTA data is read past L1
template <typename T>
__device__ __forceinline__ T ldg2(const T* p) { return __ldcg(p); }

template <typename FT>
struct GridSmem {
  union {
    struct {                       // float32 diagonal blocks (CTA 0), block row's panel
      ChSm ch;
      float Pt[kBk][kBk + 1];      // [l][row]
    } c;
    struct {                       // float64 diagonal block (CTA 0)
      FT P[kBk][kBk + 1];
      FT col[kBk][kBk + 1];        // col[j][r]: column j before its scaling
      FT rs[kBk], dv[kBk];
    } d;
    struct {                       // panel: the diagonal factor, L[r][q] at [q][r]
      FT Lt[kBk][kBk];
      FT dv[kBk];
    } p;
    float tile[4][2][kBk][kBk + 4];        // float32 trailing tiles, four at a time
    struct {                       // float64 trailing sub-tiles; tiles of step 4
      FT a[16][kBk + 1];
      FT b[16][kBk + 1];
    } q;
    struct {
      FT X[48][kBk];
      FT L[16][12];
    } n;
    struct {
      FT b[64][9];
      int j[64];
    } x;
    FT part[8][kBk];
    double red[kRT / 32];
  };
};

// float64, CTA 0: D = A(k, k) - P P^T (P the block row's panel of the step
// before; none when kp < 0), its Cholesky factor into A, and the factor
// transposed with 1 / diag into dg.  The elimination is diag_factor's; in
// float64 the reciprocal it avoids would be half a dozen dependent operations
// of about 66 cycles per column.  All global loads are issued together.
__device__ void grid_diag(double* A, int k, int ld, int kp, double* dg, int* info,
                          GridSmem<double>& sm) {
  const int tid = threadIdx.x;
  const size_t o = (size_t)kBk * k * ld + kBk * k;
  double v[3], pre[4];
  int er[3], ec[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int e = tid + q * kRT;
    er[q] = 0;
    ec[q] = -1;
    if (e >= kBk * (kBk + 1) / 2) continue;
    tri_element(e, er[q], ec[q]);
    v[q] = ldg2(A + o + (size_t)er[q] * ld + ec[q]);
  }
  if (kp >= 0)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = tid + q * kRT;
      pre[q] = ldg2(A + (size_t)(kBk * k + (e >> 5)) * ld + kBk * kp + (e & 31));
    }
  __syncthreads();
  if (kp >= 0)
#pragma unroll
    for (int q = 0; q < 4; ++q) sm.d.P[(tid + q * kRT) >> 5][tid & 31] = pre[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (ec[q] < 0) continue;
    if (kp >= 0) {
      double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
      for (int l = 0; l < kBk; l += 2) {
        a0 += sm.d.P[er[q]][l] * sm.d.P[ec[q]][l];
        a1 += sm.d.P[er[q]][l + 1] * sm.d.P[ec[q]][l + 1];
      }
      v[q] -= a0 + a1;
    }
    if (ec[q] == 0) sm.d.col[0][er[q]] = v[q];
  }
  for (int j = 0; j + 1 < kBk; ++j) {
    __syncthreads();
    if (ec[0] <= j && ec[1] <= j) continue;          // (elements 0 and 1 exist for every thread)
    double p = sm.d.col[j][j];
    if (!(p > 0.0)) p = 1.0;                         // reported below
    const int e = exponent_of(p);
    const double ph = significand(p);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (ec[q] <= j) continue;
      const double w = scale_down(sm.d.col[j][ec[q]], e);
      v[q] = v[q] * ph - sm.d.col[j][er[q]] * w;
      if (ec[q] == j + 1) sm.d.col[j + 1][er[q]] = v[q];
    }
  }
  __syncthreads();
  if (tid < kBk) {
    // pi = product of the significands before column tid; the true pivot is
    // col[j][j] / pi, so L[r][j] = col[j][r] / sqrt(col[j][j] pi)
    double p = sm.d.col[tid][tid];
    const bool bad = !(p > 0.0);
    if (bad) { atomicOr(info, kInfoPivot); p = 1.0; }
    double pi = significand(p);
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const double x = __shfl_up_sync(0xffffffffu, pi, s);
      if (tid >= s) pi *= x;
    }
    pi = __shfl_up_sync(0xffffffffu, pi, 1);
    if (tid == 0) pi = 1.0;
    const double rs = rsqrt(p * pi);
    sm.d.rs[tid] = rs;
    sm.d.dv[tid] = pi * rs;
    dg[kBk * kBk + tid] = pi * rs;
    if (bad) sm.d.col[tid][tid] = 1.0;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (ec[q] < 0) continue;
    const double x = sm.d.col[ec[q]][er[q]] * sm.d.rs[ec[q]];
    A[o + (size_t)er[q] * ld + ec[q]] = x;
    dg[ec[q] * kBk + er[q]] = x;
  }
}

// float32, CTA 0, which also solves the panel rows of the next block itself: it
// has the factor of block k in shared memory, so block k + 1 waits neither for
// the other CTAs' panel nor for theirs to reach it.  `step` is called when the
// panel rows are stored.  (A mixed slabs frame, n_c > 128: 4 % less time than with
// the block factored after the trailing update.)
template <typename Step>
__device__ void grid_next_diag(float* A, int k1, int ld, float* dg, int* info, GridSmem<float>& sm,
                               Step step) {
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t o = (size_t)kBk * k1 * ld + kBk * k1;
  float pre[3];                  // this thread's elements of the block, on their way
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int r, c;
    if (tid + q * kDT >= kBk * (kBk + 1) / 2) continue;
    tri_element(tid + q * kDT, r, c);
    pre[q] = ldg2(A + o + (size_t)r * ld + c);
  }
  if (k1 > 0 && tid < 32) {
    float4* row = reinterpret_cast<float4*>(A + (size_t)(kBk * k1 + lane) * ld + kBk * (k1 - 1));
    float x[32];
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      const float4 f = ldg2(row + l);
      x[4 * l] = f.x; x[4 * l + 1] = f.y; x[4 * l + 2] = f.z; x[4 * l + 3] = f.w;
    }
    panel_row(sm.c.ch, x);
#pragma unroll
    for (int l = 0; l < 8; ++l)
      row[l] = make_float4(x[4 * l], x[4 * l + 1], x[4 * l + 2], x[4 * l + 3]);
#pragma unroll
    for (int l = 0; l < 32; ++l) sm.c.Pt[l][lane] = x[l];
  }
  __syncthreads();
  if (k1 > 0) step();
  int nth = 0;                   // diag_factor asks for the elements in that order
  diag_factor(
      sm.c.ch, k1 > 0 ? &sm.c.Pt[0][0] : nullptr, kBk + 1, info, [&](int, int) { return pre[nth++]; },
      [&](int r, int c, float x) {
        A[o + (size_t)r * ld + c] = x;
        dg[c * kBk + r] = x;
      });
  __syncthreads();
  if (tid < kBk) dg[kBk * kBk + tid] = sm.c.ch.dv[tid];
}

// Panel k: every row below the diagonal block (float32: not those of block k + 1,
// which CTA 0 solves) and every identity row so far, x L_kk^T = a.  A row is one
// thread with its 32 values in registers (float32),
// or one warp (float64: 32 x 2 dependent warp instructions per row where a
// thread per row would need 528 per warp), four rows per CTA at a time so that
// each SM sub-partition has one.
__device__ void grid_panel(float* A, float* U, int k, int nb, int ld, const float* dg, int rank, int G,
                           GridSmem<float>& sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (rank >= nb) return;
  for (int e = tid; e < (kBk * kBk + kBk) / 4; e += kRT)      // Lt, dv
    reinterpret_cast<float4*>(&sm.c.ch)[e] = ldg2(reinterpret_cast<const float4*>(dg) + e);
  __syncthreads();
  for (int b = rank + wid * G; b < nb; b += (kRT / 32) * G) {
    if (b == k + 1) continue;
    float* row = (b > k ? A : U) + (size_t)(kBk * b + lane) * ld + kBk * k;
    float x[kBk];
    if (b == k) {
#pragma unroll
      for (int l = 0; l < kBk; ++l) x[l] = l == lane ? 1.f : 0.f;
    } else {
#pragma unroll
      for (int l = 0; l < kBk / 4; ++l) {
        const float4 f = ldg2(reinterpret_cast<const float4*>(row) + l);
        x[4 * l] = f.x; x[4 * l + 1] = f.y; x[4 * l + 2] = f.z; x[4 * l + 3] = f.w;
      }
    }
    panel_row(sm.c.ch, x);
#pragma unroll
    for (int l = 0; l < kBk / 4; ++l)
      reinterpret_cast<float4*>(row)[l] = make_float4(x[4 * l], x[4 * l + 1], x[4 * l + 2], x[4 * l + 3]);
  }
}
__device__ void grid_panel(double* A, double* U, int k, int nb, int ld, const double* dg, int rank,
                           int G, GridSmem<double>& sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (rank >= nb * (kBk / 4)) return;
  for (int e = tid; e < kBk * kBk; e += kRT) (&sm.p.Lt[0][0])[e] = ldg2(dg + e);
  if (tid < kBk) sm.p.dv[tid] = ldg2(dg + kBk * kBk + tid);
  __syncthreads();
  for (int g = rank + (wid >> 2) * G; g < nb * (kBk / 4); g += 2 * G) {
    const int r = 4 * g + (wid & 3), b = r >> 5;
    double* row = (b > k ? A : U) + (size_t)r * ld + kBk * k;
    double x = b == k ? ((r & 31) == lane ? 1.0 : 0.0) : ldg2(row + lane);
#pragma unroll 4
    for (int q = 0; q < kBk; ++q) {
      const double xq = __shfl_sync(0xffffffffu, x, q) * sm.p.dv[q];
      if (lane == q) x = xq;
      if (lane > q) x -= xq * sm.p.Lt[q][lane];
    }
    row[lane] = x;
  }
}

// Trailing update of step k, without the diagonal block of step k + 1 (CTA 0's):
// A(i, j) -= P_i P_j^T for k < j <= i, and the identity rows
// U(i, j) -= P_i P_j^T for i <= k < j (U(k, j) starts at zero).
__device__ void grid_trail(float* A, float* U, int k, int nb, int ld, int slot, int nslots,
                           GridSmem<float>& sm) {
  // four 32 x 32 tiles per CTA, 64 threads each, 4 x 4 values per thread: rows
  // ti + 8 p, columns tj + 8 q, so that the float4 reads of a quarter warp fall
  // in different banks
  const int m = nb - k - 1, tri = m * (m + 1) / 2, total = tri + (k + 1) * m;
  const int qd = threadIdx.x >> 6, tq = threadIdx.x & 63, ti = tq >> 3, tj = tq & 7;
  float(*Pi)[kBk + 4] = sm.tile[qd][0];
  float(*Pj)[kBk + 4] = sm.tile[qd][1];
  for (int t = slot + qd * nslots; t < total; t += 4 * nslots) {
    if (t == 0) continue;                  // the diagonal block
    int i, j;
    if (t < tri) {
      int I = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while ((I + 1) * (I + 2) / 2 <= t) ++I;
      while (I * (I + 1) / 2 > t) --I;
      i = k + 1 + I;
      j = k + 1 + t - I * (I + 1) / 2;
    } else {
      i = (t - tri) / m;
      j = k + 1 + (t - tri) % m;
    }
    const float* src_i = (i > k ? A : U) + (size_t)kBk * i * ld + kBk * k;
    const float* src_j = A + (size_t)kBk * j * ld + kBk * k;
    float* dst = (i > k ? A : U) + (size_t)kBk * i * ld + kBk * j;
    const bool first = i == k;
    float4 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tq + 64 * u;
      a[u] = ldg2(reinterpret_cast<const float4*>(src_i + (size_t)(e >> 3) * ld) + (e & 7));
      b[u] = ldg2(reinterpret_cast<const float4*>(src_j + (size_t)(e >> 3) * ld) + (e & 7));
    }
    float acc[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        acc[p][q] = first ? 0.f : ldg2(dst + (size_t)(ti + 8 * p) * ld + tj + 8 * q);
    asm volatile("bar.sync %0, 64;" ::"r"(qd + 1) : "memory");   // the tile before is read
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tq + 64 * u;
      *reinterpret_cast<float4*>(&Pi[e >> 3][4 * (e & 7)]) = a[u];
      *reinterpret_cast<float4*>(&Pj[e >> 3][4 * (e & 7)]) = b[u];
    }
    asm volatile("bar.sync %0, 64;" ::"r"(qd + 1) : "memory");
#pragma unroll 2
    for (int l = 0; l < kBk; l += 4) {
      float4 x[4], y[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) x[p] = *reinterpret_cast<const float4*>(&Pi[ti + 8 * p][l]);
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(&Pj[tj + 8 * q][l]);
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          acc[p][q] -= x[p].x * y[q].x + x[p].y * y[q].y + x[p].z * y[q].z + x[p].w * y[q].w;
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) dst[(size_t)(ti + 8 * p) * ld + tj + 8 * q] = acc[p][q];
  }
}
__device__ void grid_trail(double* A, double* U, int k, int nb, int ld, int slot, int nslots,
                           GridSmem<double>& sm) {
  // 16 x 16 sub-tiles, one value per thread: a 32 x 32 tile would hold an SM's
  // float64 pipes for 8 us
  const int m = nb - k - 1, m2 = 2 * m, tri = m2 * (m2 + 1) / 2, total = tri + 2 * (k + 1) * m2;
  const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
  // sub-tiles 0..2 are the diagonal block
  for (int t = 3 + slot; t < total; t += nslots) {
    int i, j;                              // sub-tile rows and columns, in units of 16
    bool low;
    if (t < tri) {
      int I = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while ((I + 1) * (I + 2) / 2 <= t) ++I;
      while (I * (I + 1) / 2 > t) --I;
      i = 2 * (k + 1) + I;
      j = 2 * (k + 1) + t - I * (I + 1) / 2;
      low = true;
    } else {
      i = (t - tri) / m2;
      j = 2 * (k + 1) + (t - tri) % m2;
      low = false;
    }
    const double* src_i = (low ? A : U) + (size_t)16 * i * ld + kBk * k;
    const double* src_j = A + (size_t)16 * j * ld + kBk * k;
    double* dst = (low ? A : U) + (size_t)(16 * i + r) * ld + 16 * j + c;
    const double a0 = ldg2(src_i + (size_t)r * ld + c), a1 = ldg2(src_i + (size_t)r * ld + c + 16);
    const double b0 = ldg2(src_j + (size_t)r * ld + c), b1 = ldg2(src_j + (size_t)r * ld + c + 16);
    double acc = !low && (i >> 1) == k ? 0.0 : ldg2(dst);
    __syncthreads();
    sm.q.a[r][c] = a0; sm.q.a[r][c + 16] = a1;
    sm.q.b[r][c] = b0; sm.q.b[r][c + 16] = b1;
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < kBk; ++l) acc -= sm.q.a[r][l] * sm.q.b[c][l];
    *dst = acc;
  }
}

// A = L L^T (nb x nb blocks, lower; L in place) and U = L^-T (upper)
__device__ void grid_chol(double* A, double* U, int nb, int ld, double* dg, GroupBar& bar, int rank,
                          GridSmem<double>& sm) {
  constexpr int kDg = kBk * kBk + kBk;
  if (rank == 0) grid_diag(A, 0, ld, -1, dg, bar.info, sm);
  group_sync(bar);
  for (int k = 0; k < nb; ++k) {
    grid_panel(A, U, k, nb, ld, dg + (k & 1) * kDg, rank, bar.G, sm);
    group_sync(bar);
    if (k + 1 < nb) {
      if (rank == 0) {
        grid_diag(A, k + 1, ld, k, dg + ((k + 1) & 1) * kDg, bar.info, sm);
        __syncthreads();
      }
      if (bar.G == 1) grid_trail(A, U, k, nb, ld, 0, 1, sm);
      else if (rank > 0) grid_trail(A, U, k, nb, ld, rank - 1, bar.G - 1, sm);
      group_sync(bar);
    }
  }
}
// float32: CTA 0 only arrives at the first barrier of a panel (with its rows of
// it stored) and makes the next diagonal factor; the others share the rest of
// the panel and the trailing update.  `panel` counts the arrivals of the first
// barrier apart from the second's, which CTA 0 may reach early.
__device__ void grid_chol(float* A, float* U, int nb, int ld, float* dg, GroupBar& bar, GroupBar& panel,
                          int rank, GridSmem<float>& sm) {
  constexpr int kDg = kBk * kBk + kBk;
  const bool lone = bar.G == 1;
  if (rank == 0) grid_next_diag(A, 0, ld, dg, bar.info, sm, [] {});
  group_sync(bar);
  for (int k = 0; k < nb; ++k) {
    if (rank == 0) {
      if (k + 1 < nb)
        grid_next_diag(A, k + 1, ld, dg + ((k + 1) & 1) * kDg, bar.info, sm, [&] { group_arrive(panel); });
      else
        group_arrive(panel);
    }
    if (rank > 0 || lone) {
      if (lone) __syncthreads();
      grid_panel(A, U, k, nb, ld, dg + (k & 1) * kDg, lone ? 0 : rank - 1, lone ? 1 : bar.G - 1, sm);
      if (k + 1 < nb) {
        if (lone) __syncthreads();
        else group_sync(panel);
        grid_trail(A, U, k, nb, ld, lone ? 0 : rank - 1, lone ? 1 : bar.G - 1, sm);
      } else if (!lone) {
        group_arrive(panel);
      }
    }
    group_sync(bar);
    if (lone && k + 1 < nb) {        // the factor of block k + 1 back into shared memory
      for (int e = threadIdx.x; e < kDg / 4; e += kRT)
        reinterpret_cast<float4*>(&sm.c.ch)[e] =
            ldg2(reinterpret_cast<const float4*>(dg + ((k + 1) & 1) * kDg) + e);
      __syncthreads();
    }
  }
}

// CTAs of the launch that a system of this size uses: with more, the barriers
// cost more than the extra CTAs give (float32: four tiles at a time per CTA)
template <typename FT>
__device__ __forceinline__ int grid_ctas(int nbn, int G) {
  const int want = std::is_same<FT, double>::value ? 2 * nbn * nbn : 8 + nbn * nbn / 8;
  return want < G ? want : G;
}

template <typename FT>
__device__ void grid_prepare(RedArgs<FT> a, int rank, int G, GridSmem<FT>& sm) {
  const int nc = *a.nc_dev;
  if (nc == 0 || nc <= a.small_lim) return;
  const GridLay<FT> g = grid_layout(a.base, nc);
  red_tail(a, nc);
  G = grid_ctas<FT>(g.nbn, G);
  if (rank >= G) return;
  GroupBar bar{a.bar, 0u, G, a.info, false}, panel{a.bar + 4, 0u, G, a.info, false};
  auto chol = [&](FT* M, FT* V, int nb, int ld) {
    if constexpr (std::is_same<FT, double>::value) grid_chol(M, V, nb, ld, g.dg, bar, rank, sm);
    else grid_chol(M, V, nb, ld, g.dg, bar, panel, rank, sm);
  };
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, n3 = g.n3;
  const int gwarp = rank * (kRT / 32) + wid, nwarps = G * (kRT / 32);
  // 1. S (lower, padded by the identity) and the block-row lists
  for (int i = gwarp; i < g.lds; i += nwarps) {
    const double* srow = i < nc ? a.Sinv + (size_t)a.clist[i] * a.n2 : nullptr;
    for (int j = lane; j <= i; j += 32)
      g.S[(size_t)i * g.lds + j] = i < nc ? (FT)srow[a.clist[j]] : (i == j ? FT(1) : FT(0));
    if (i >= nc) continue;
    int base = 0;
    for (int j0 = 0; j0 < nc; j0 += 32) {
      const int j = j0 + lane;
      const bool f = j < nc && a.bocc[(size_t)i * nc + j] != 0;
      const unsigned msk = __ballot_sync(0xffffffffu, f);
      if (f) a.list[(size_t)i * nc + base + __popc(msk & ((1u << lane) - 1u))] = j;
      base += __popc(msk);
    }
    if (lane == 0) a.cnt[i] = base;
  }
  group_sync(bar);
  // 2. L_s, U_s
  chol(g.S, g.Us, g.nbs, g.lds);
  // 3. X[(i,a),(k,b)] = sum_{j in row i, j >= k} B[(i,a),(j,b)] L_s[j][k]: a CTA
  // takes block row i and 256 columns k, the row's blocks of B staged (64 at a
  // time) in the factor's type; a thread keeps the nine values of one k
  for (int it = rank; it < nc * ((nc + kRT - 1) / kRT); it += G) {
    const int i = it % nc, k = (it / nc) * kRT + tid, ci = ldg2(a.cnt + i);
    FT acc[3][3];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) acc[p][q] = FT(0);
    for (int e0 = 0; e0 < ci; e0 += 64) {
      const int en = min(64, ci - e0);
      __syncthreads();
      for (int e = tid; e < 9 * en; e += kRT) {
        const int u = e / 9, pq = e % 9, j = ldg2(a.list + (size_t)i * nc + e0 + u);
        sm.x.b[u][pq] = (FT)a.Bc[(size_t)(3 * i + pq / 3) * n3 + 3 * j + pq % 3];
        if (pq == 0) sm.x.j[u] = j;
      }
      __syncthreads();
      if (k < nc) {
#pragma unroll 4
        for (int u = 0; u < en; ++u) {
          const int j = sm.x.j[u];
          if (j < k) continue;
          const FT L = ldg2(g.S + (size_t)j * g.lds + k);
#pragma unroll
          for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) acc[p][q] += sm.x.b[u][3 * p + q] * L;
        }
      }
    }
    if (k < nc)
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) g.U[(size_t)(3 * i + p) * g.ldn + 3 * k + q] = acc[p][q];
  }
  group_sync(bar);
  // 4. N = I + (L_s (x) I)^T X, lower triangle, by tiles of 32 x 32 (float32) or
  // 16 x 16 (float64): N[(i, ax)][col] sums L_s[j][i] X[(j, ax)][col] over
  // j >= i, 16 values of j staged at a time.  float32: each stage's sum joins
  // a two-term total (two-sum), so the long sums round like one addition
  {
    constexpr bool f32 = std::is_same<FT, float>::value;
    constexpr int TS = f32 ? 32 : 16, kV = TS * TS / kRT;
    const int nt = g.ldn / TS;
    const int c = tid % TS, r0 = tid / TS;
    for (int t = rank; t < nt * (nt + 1) / 2; t += G) {
      int ti = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
      while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
      while (ti * (ti + 1) / 2 > t) --ti;
      const int tj = t - ti * (ti + 1) / 2, R0 = TS * ti, C0 = TS * tj, i0 = R0 / 3;
      FT hi[kV], lo[kV];
#pragma unroll
      for (int q = 0; q < kV; ++q) {
        hi[q] = R0 + r0 + q * (kRT / TS) == C0 + c ? FT(1) : FT(0);
        lo[q] = FT(0);
      }
      for (int j0 = i0; j0 < nc; j0 += 16) {
        __syncthreads();
        for (int e = tid; e < 48 * TS; e += kRT) {
          const int xr = 3 * j0 + e / TS, xc = C0 + e % TS;
          sm.n.X[e / TS][e % TS] = xr < n3 && xc < n3 ? ldg2(g.U + (size_t)xr * g.ldn + xc) : FT(0);
        }
        for (int e = tid; e < 16 * 12; e += kRT) {
          const int j = j0 + e / 12, i = i0 + e % 12;
          sm.n.L[e / 12][e % 12] = j < nc && i < nc && j >= i ? ldg2(g.S + (size_t)j * g.lds + i) : FT(0);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kV; ++q) {
          const int row = R0 + r0 + q * (kRT / TS), iv = row / 3 - i0, ax = row % 3;
          FT s = f32 ? FT(0) : hi[q];
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) s += sm.n.L[jj][iv] * sm.n.X[3 * jj + ax][c];
          if (f32) {
            const FT h = hi[q] + s, bb = h - hi[q];
            lo[q] += (hi[q] - (h - bb)) + (s - bb);
            hi[q] = h;
          } else {
            hi[q] = s;
          }
        }
      }
#pragma unroll
      for (int q = 0; q < kV; ++q)
        g.N[(size_t)(R0 + r0 + q * (kRT / TS)) * g.ldn + C0 + c] = hi[q] + lo[q];
    }
  }
  group_sync(bar);
  // 5. L_N, U_N (over X)
  chol(g.N, g.U, g.nbn, g.ldn);
  group_leave(bar, a.bar + 4);
}

// out = (L_s (x) I_3)^T p (padded with zeros), one warp per entry
template <typename FT>
__device__ __forceinline__ void grid_lt(const GridLay<FT>& g, const double* p, FT* out, int gwarp,
                                        int nwarps) {
  const int lane = threadIdx.x & 31;
  for (int e = gwarp; e < g.ldn; e += nwarps) {
    const int i = e / 3, ax = e % 3;
    double acc = 0.0;
    if (e < g.n3)
      for (int j = i + lane; j < g.nc; j += 32)
        acc += (double)g.S[(size_t)j * g.lds + i] * ldg2(p + 3 * j + ax);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[e] = (FT)acc;
  }
}
// out = U^T x: a CTA per block column, its 8 warps share the rows (lane = column)
template <typename FT>
__device__ __forceinline__ void grid_ut(const GridLay<FT>& g, const FT* x, FT* out, int rank, int G,
                                        GridSmem<FT>& sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int b = rank; b < g.nbn; b += G) {
    const int j = kBk * b + lane;
    FT acc = 0;
#pragma unroll 8
    for (int i = wid; i < kBk * (b + 1); i += kRT / 32)
      acc += (i <= j ? g.U[(size_t)i * g.ldn + j] : FT(0)) * ldg2(x + i);
    __syncthreads();
    sm.part[wid][lane] = acc;
    __syncthreads();
    if (wid == 0) {
      FT s = 0;
#pragma unroll
      for (int w = 0; w < kRT / 32; ++w) s += sm.part[w][lane];
      out[j] = s;
    }
  }
}
// out = U x, one warp per row
template <typename FT>
__device__ __forceinline__ void grid_u(const GridLay<FT>& g, const FT* x, FT* out, int gwarp,
                                       int nwarps) {
  const int lane = threadIdx.x & 31;
  for (int i = gwarp; i < g.ldn; i += nwarps) {
    FT acc = 0;
#pragma unroll 4
    for (int j = (i & ~31) + lane; j < g.ldn; j += 32)
      acc += (j >= i ? g.U[(size_t)i * g.ldn + j] : FT(0)) * ldg2(x + j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[i] = acc;
  }
}

// Refinement of a float32 factor's solve by |rho|^2 (tot; of the step before:
// prev, negative before the first) and |y2|^2 (ys).  refined: no further step;
// step_lost: the last one is taken back; accepted: what is left is small enough.
// A NaN ends the steps, is taken back where that helps and is not accepted.
__device__ __forceinline__ bool refined(double tot, double prev, double ys, int it, int steps) {
  return !(tot > 1e-14 * ys) || (prev >= 0.0 && !(tot < 0.25 * prev)) || it >= steps;
}
__device__ __forceinline__ bool step_lost(double tot, double prev) {
  return prev >= 0.0 && !(tot <= prev);
}
__device__ __forceinline__ bool accepted(double tot, double prev, double ys) {
  return (step_lost(tot, prev) ? prev : tot) <= kAcceptRho * kAcceptRho * ys;
}

template <typename FT>
__device__ void grid_solve(RedArgs<FT> a, int rank, int Gall, GridSmem<FT>& sm) {
  const int nc = *a.nc_dev;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (nc == 0 || nc <= a.small_lim) return;
  const GridLay<FT> g = grid_layout(a.base, nc);
  red_tail(a, nc);
  const int G = Gall, n3 = g.n3;     // the z2 update has a row per x2 vertex: all CTAs
  GroupBar bar{a.bar + 2, 0u, G, a.info, false};
  const int gtid = rank * kRT + tid, gsz = G * kRT;
  const int gwarp = rank * (kRT / 32) + wid, nwarps = G * (kRT / 32);
  // 6. y = B u_c (a warp per block row: its lanes share the row's blocks), |y2|^2
  if (gtid == 0) { a.nrm[0] = 0.0; a.nrm[1] = 0.0; a.nrm[2] = 0.0; }
  for (int i = gwarp; i < nc; i += nwarps) {
    const double* b0 = a.Bc + (size_t)(3 * i) * n3;
    const int ci = a.cnt[i];
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int e = lane; e < ci; e += 32) {
      const int j = a.list[(size_t)i * nc + e];
      const double* uj = a.u + 3 * (size_t)a.clist[j];
      const double u0 = uj[0], u1 = uj[1], u2 = uj[2];
      const double* bp = b0 + 3 * j;
      s0 += bp[0] * u0 + bp[1] * u1 + bp[2] * u2;
      s1 += bp[n3] * u0 + bp[n3 + 1] * u1 + bp[n3 + 2] * u2;
      s2 += bp[2 * n3] * u0 + bp[2 * n3 + 1] * u1 + bp[2 * n3 + 2] * u2;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) { a.y[3 * i] = s0; a.y[3 * i + 1] = s1; a.y[3 * i + 2] = s2; }
  }
  group_sync(bar);
  if (!std::is_same<FT, double>::value) {
    double q = 0.0;
    for (int e = gtid; e < 3 * a.n2; e += gsz) q += (double)a.y2[e] * (double)a.y2[e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (lane == 0 && q != 0.0) atomicAdd(&a.nrm[2], q);
  }
  // v (+)= (U_s (x) I) U U^T (L_s (x) I)^T p
  auto apply = [&](const double* p, bool add) {
    grid_lt(g, p, g.t, gwarp, nwarps);
    group_sync(bar);
    grid_ut(g, g.t, g.l, rank, G, sm);
    group_sync(bar);
    grid_u(g, g.l, g.t, gwarp, nwarps);
    group_sync(bar);
    for (int i = gwarp; i < nc; i += nwarps) {
      FT s0 = 0, s1 = 0, s2 = 0;
#pragma unroll 4
      for (int j = i + lane; j < nc; j += 32) {
        const FT u = g.Us[(size_t)i * g.lds + j];
        s0 += u * ldg2(g.t + 3 * j);
        s1 += u * ldg2(g.t + 3 * j + 1);
        s2 += u * ldg2(g.t + 3 * j + 2);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      }
      if (lane < 3) {
        const double d = (double)(lane == 0 ? s0 : lane == 1 ? s1 : s2);
        const double v0 = add ? ldg2(a.v + 3 * i + lane) : 0.0;
        if (add) a.vp[3 * i + lane] = v0;
        a.v[3 * i + lane] = v0 + d;
      }
    }
    group_sync(bar);
  };
  apply(a.y, false);
  // 7. refinement with float64 residuals: a.refine steps with float64 factors;
  //    with float32 factors until |rho| <= 1e-7 |y2|, until a step fails to
  //    halve |rho|, or after a.refine steps, and the v of the smaller |rho|
  //    stays.  |rho|^2 alternates between two accumulators
  constexpr bool f64 = std::is_same<FT, double>::value;
  double prev = -1.0;
  for (int it = 0; !f64 || it < a.refine; ++it) {
    // w = S v with S = Sigma^-1[c, c] (x) I_3 in float64, a warp per row
    for (int i = gwarp; i < nc; i += nwarps) {
      const double* srow = a.Sinv + (size_t)a.clist[i] * a.n2;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
      for (int j = lane; j < nc; j += 32) {
        const double sv = srow[a.clist[j]];
        s0 += sv * ldg2(a.v + 3 * j);
        s1 += sv * ldg2(a.v + 3 * j + 1);
        s2 += sv * ldg2(a.v + 3 * j + 2);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      }
      if (lane < 3) a.w[3 * i + lane] = lane == 0 ? s0 : lane == 1 ? s1 : s2;
    }
    group_sync(bar);
    if (gtid == 0) a.nrm[(it + 1) & 1] = 0.0;
    double r2 = 0.0;
    for (int i = gwarp; i < nc; i += nwarps) {
      const double* b0 = a.Bc + (size_t)(3 * i) * n3;
      const int ci = a.cnt[i];
      double s0 = 0.0, s1 = 0.0, s2 = 0.0;
      for (int e = lane; e < ci; e += 32) {
        const int j = a.list[(size_t)i * nc + e];
        const double w0 = ldg2(a.w + 3 * j), w1 = ldg2(a.w + 3 * j + 1), w2 = ldg2(a.w + 3 * j + 2);
        const double* bp = b0 + 3 * j;
        s0 += bp[0] * w0 + bp[1] * w1 + bp[2] * w2;
        s1 += bp[n3] * w0 + bp[n3 + 1] * w1 + bp[n3 + 2] * w2;
        s2 += bp[2 * n3] * w0 + bp[2 * n3 + 1] * w1 + bp[2 * n3 + 2] * w2;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      }
      if (lane < 3) {
        const int row = 3 * i + lane;
        const double rr = ldg2(a.y + row) - ldg2(a.v + row) - (lane == 0 ? s0 : lane == 1 ? s1 : s2);
        a.rho[row] = rr;
        r2 += rr * rr;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if (!f64) {
      __syncthreads();
      if (lane == 0) sm.red[wid] = r2;
      __syncthreads();
      if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < kRT / 32; ++w) s += sm.red[w];
        if (s != 0.0) atomicAdd(&a.nrm[it & 1], s);
      }
    }
    group_sync(bar);
    if (!f64) {
      // the same values for every thread of the system: a uniform decision
      const double tot = ldg2(a.nrm + (it & 1)), ys = ldg2(a.nrm + 2);
      if (refined(tot, prev, ys, it, a.refine)) {
        if (step_lost(tot, prev)) {
          for (int e = gtid; e < n3; e += gsz) a.v[e] = ldg2(a.vp + e);
          group_sync(bar);
        }
        if (gtid == 0 && !accepted(tot, prev, ys)) atomicOr(a.info, kInfoStalled);
        break;
      }
      prev = tot;
    }
    apply(a.rho, true);
  }
  // 8. z2 = u - (Sigma^-1[:, c] (x) I_3) v
  z2_update(a, nc, gwarp, nwarps);
  group_leave(bar, nullptr);
}

// A: per-system arguments on the device (batches), else `one`
template <typename FT>
__global__ void __launch_bounds__(kRT) k_grid_prepare(RedArgs<FT> one, const RedArgs<FT>* A,
                                                      GridFrames fr) {
  __shared__ __align__(16) GridSmem<FT> sm;
  grid_prepare<FT>(A ? A[fr.id[blockIdx.x / fr.G]] : one, blockIdx.x % fr.G, fr.G, sm);
}
template <typename FT>
__global__ void __launch_bounds__(kRT) k_grid_solve(RedArgs<FT> one, const RedArgs<FT>* A,
                                                    GridFrames fr) {
  __shared__ __align__(16) GridSmem<FT> sm;
  grid_solve<FT>(A ? A[fr.id[blockIdx.x / fr.G]] : one, blockIdx.x % fr.G, fr.G, sm);
}

// ---------------------------------------------------------------------------
// Small forms (float32 factors, 0 < n_c <= kClusNc).  Every kernel reads n_c on
// the device.  On the side stream, while the forward solve makes u:
//   k_small_s     (1 CTA)  S = Sigma^-1[c,c], L_s, block lists of B
//   k_small_x     (grid)   X = B (L_s (x) I_3)
//   k_small_n     (grid)   N = I + (L_s (x) I_3)^T X  (lower part, packed)
//   k_small_v     (1 CTA, n_c <= kSmallNc) or k_clus_v (4-CTA cluster): L_N, the
//                          whole matrix in shared memory, so no grid-wide barrier
//   k_small_u     (CTA per block column)  V = L_N^-1, V_s = L_s^-1
// and after it
//   k_small_solve (8-CTA cluster)  y = B u_c, v and its float64 refinement
//   k_z2_update   (grid)   z2
// With explicit inverses a solve is four products that spread over the cluster;
// substitution would be a chain of 2 n / 32 + n_c / 32 dependent blocks, each a
// cluster barrier or two CTA barriers.  n_c = 93, one frame: 16 + 240 us stood
// between u and v; now 67 us do, with the factor and the inverses (104 + 45 us)
// beside the forward solve.
// ---------------------------------------------------------------------------
constexpr int kSmallNc = 96;               // 3 n_c <= 288 fits in one CTA's shared memory
constexpr int kSmallN3 = 3 * kSmallNc;
constexpr int kClusNc = 128;               // 3 n_c <= 384 fits in a 4-CTA cluster
constexpr int kClusN3 = 3 * kClusNc;
constexpr int kCl = 4;                     // CTAs per cluster
constexpr int kST = 512;                   // threads of the one-CTA kernels
constexpr int kSW = kST / 32;

constexpr int kPtLd = kSmallN3;            // panel scratch: 32 x kPtLd floats
constexpr int kPanelsDone = 16;            // word of RedArgs::bar: panels of N factored

// Outer-product elimination of the unscaled 32 x 32 diagonal block Ds: after
// step j, Ds[i][c] (c > j) holds the Schur complement; Ds[.][j] (j < i) stays
// the unscaled column and Ds[j][j] the pivot.  Thread (r0, c) = (tid / 32,
// tid % 32) owns rows r0 and r0 + 16 of column c; needs 512 threads.  The
// pivot reciprocal is the hardware approximation (within 2 ulp for pivots
// in [2^-126, 2^126]; those of N = I + L^T B L are >= 1, those of
// S = Sigma^-1[c, c] are positive and far from either end): the IEEE
// division sat on the dependent chain of every step, and these float32
// factors are refined in float64 (N) or feed only the float32 products and
// solves of the reduced system (S).  Two columns per barrier measured no
// faster.
__device__ __forceinline__ void eliminate_diag(float (*Ds)[33], int kb) {
  const int tid = threadIdx.x, r0 = tid >> 5, c = tid & 31;
  for (int j = 0; j < kb; ++j) {
    const float inv = __fdividef(1.f, Ds[j][j]);
    if (c > j) {
      const float lcj = Ds[c][j] * inv;
      if (r0 >= c) Ds[r0][c] -= Ds[r0][j] * lcj;
      if (r0 + 16 >= c) Ds[r0 + 16][c] -= Ds[r0 + 16][j] * lcj;
    }
    __syncthreads();
  }
}

// Blocked right-looking Cholesky of the packed n x n matrix A in shared
// memory by one CTA (kST threads); 32-wide panels.  Per panel: the diagonal
// block is factored in shared memory by all threads (outer-product form, one
// barrier per column), every row below solves its own panel segment by
// substitution (one thread per row) while the last warp inverts the
// diagonal block, and the trailing update A -= P P^T runs with 4 x 4
// register tiles from a transposed copy Pt of the panel.
// With `out`, every panel goes to the packed matrix out in global memory as
// soon as it is solved, its diagonal block inverted, and *done then counts it.
// DIout, if given, receives the inverted diagonal blocks.  Loops stay rolled:
// straight-line code this size would run out of the instruction cache.
__device__ void cta_chol_packed(float* A, int n, float* Pt, int* info, float* out, unsigned* done,
                                float* DIout) {
  __shared__ float Ds[32][33];
  __shared__ float Li[32][33];
  __shared__ float dv[32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int k0 = 0; k0 < n; k0 += 32) {
    const int kb = min(32, n - k0), k1 = k0 + kb, m = n - k1;
    for (int e = tid; e < 32 * 32; e += kST) {
      const int i = e >> 5, j = e & 31;
      Ds[i][j] = (i < kb && j <= i) ? A[prow(k0 + i) + k0 + j] : 0.f;
    }
    __syncthreads();
    // outer-product elimination on the unscaled block; Ds[.][j] is scaled below
    eliminate_diag(Ds, kb);
    if (tid < kb) {
      float d = Ds[tid][tid];
      if (!(d > 0.f)) {
        atomicOr(info, kInfoPivot);
        d = 1.f;
        Ds[tid][tid] = 1.f;
      }
      float rs = rsqrtf(d);
      rs = rs * (1.5f - 0.5f * d * rs * rs);
      dv[tid] = rs;
    } else if (tid < 32) {
      dv[tid] = 1.f;        // padding of a last, narrower block
    }
    __syncthreads();
    for (int e = tid; e < kb * 32; e += kST) {
      const int i = e >> 5, j = e & 31;
      if (j < i) Ds[i][j] *= dv[j];
    }
    __syncthreads();
    if (tid < kb) Ds[tid][tid] = Ds[tid][tid] * dv[tid];    // sqrt(d)
    __syncthreads();
    if (tid < m) {
      // row k1 + tid: x L_kk^T = a in registers (right-looking, so the
      // dependent chain is one FMA per column), then its transposed copy
      float* row = A + prow(k1 + tid) + k0;
      float x[32];
#pragma unroll
      for (int l = 0; l < 32; ++l) x[l] = row[l];
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        x[q] *= dv[q];
#pragma unroll
        for (int l = q + 1; l < 32; ++l) x[l] -= x[q] * Ds[l][q];
      }
#pragma unroll
      for (int l = 0; l < 32; ++l) {
        row[l] = x[l];
        Pt[l * kPtLd + tid] = x[l];
      }
      if (out) {
        float4* o = reinterpret_cast<float4*>(out + prow(k1 + tid) + k0);
#pragma unroll
        for (int l = 0; l < 8; ++l)
          o[l] = make_float4(x[4 * l], x[4 * l + 1], x[4 * l + 2], x[4 * l + 3]);
      }
    } else if (wid == kSW - 1) {
      // Li = L_kk^-1, column `lane` in registers (right-looking)
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = (i == lane) ? 1.f : 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        x[i] *= dv[i];
#pragma unroll
        for (int l = i + 1; l < 32; ++l) x[l] -= Ds[l][i] * x[i];
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) Li[i][lane] = (i >= lane) ? x[i] : 0.f;
      if (out)
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (lane <= i && i < kb) out[prow(k0 + i) + k0 + lane] = x[i];
    }
    __syncthreads();
    if (out && tid == kST - 1) {     // (a thread of the last, least loaded warp)
      __threadfence();
      asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(done), "r"((unsigned)(k0 >> 5) + 1u)
                   : "memory");
    }
    if (m > 0) {
      // trailing update A -= P P^T, 4 x 4 tiles of the lower triangle
      const int mb = (m + 3) >> 2, nt = mb * (mb + 1) / 2;
      for (int t = tid; t < nt; t += kST) {
        int I = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
        while ((I + 1) * (I + 2) / 2 <= t) ++I;
        while (I * (I + 1) / 2 > t) --I;
        const int J = t - I * (I + 1) / 2;
        float acc[4][4];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][q] = 0.f;
#pragma unroll 4
        for (int l = 0; l < 32; ++l) {
          const float4 av = *reinterpret_cast<const float4*>(Pt + l * kPtLd + 4 * I);
          const float4 bv = *reinterpret_cast<const float4*>(Pt + l * kPtLd + 4 * J);
          const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[p][q] += ar[p] * br[q];
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const int i = 4 * I + p;
          if (i >= m) break;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int jj = 4 * J + q;
            if (jj <= i) A[prow(k1 + i) + k1 + jj] -= acc[p][q];
          }
        }
      }
    }
    // the diagonal block
    for (int e = tid; e < kb * 32; e += kST) {
      const int i = e >> 5, j = e & 31;
      if (j <= i) A[prow(k0 + i) + k0 + j] = Ds[i][j];
      if (DIout) DIout[(size_t)(k0 >> 5) * 1024 + e] = (j <= i) ? Li[i][j] : 0.f;
    }
    __syncthreads();
  }
}

// k_small_s: S = Sigma^-1[c, c], its factor (plain, row-major into a.S for
// the products; packed with inverted diagonal blocks into a.spk for the
// solves) and the block-row lists of B.
__device__ __forceinline__ void k_small_s_body(RedArgs<float> a) {
  extern __shared__ float smem_f[];
  const int nc = *a.nc_dev;
  if (nc == 0 || nc > a.small_lim) return;
  red_layout(a, nc);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float* P = smem_f;                      // prow(kClusNc) floats
  float* Pt = P + prow(kClusNc);          // 32 x kPtLd
  if (tid == 0) { a.nrm[2] = 0.0; a.bar[kPanelsDone] = 0; }
  for (int i = wid; i < nc; i += kSW) {
    if (!FSIM_CHECK_IDX(a.clist[i], a.n2, CHECK_CLIST)) continue;
    const double* srow = a.Sinv + (size_t)a.clist[i] * a.n2;
#pragma unroll 4
    for (int j = lane; j < nc; j += 32) {
      if (!FSIM_CHECK_IDX(a.clist[j], a.n2, CHECK_CLIST)) continue;
      const double sv = srow[a.clist[j]];
      a.S64[(size_t)i * nc + j] = sv;
      if (j <= i) P[prow(i) + j] = (float)sv;
    }
  }
  for (int i = wid; i < nc; i += kSW) {
    bool f[kClusNc / 32];                 // all occupancy flags of the row first
#pragma unroll
    for (int q = 0; q < kClusNc / 32; ++q) {
      const int j = 32 * q + lane;
      f[q] = j < nc && a.bocc[(size_t)i * nc + j] != 0;
    }
    int base = 0;
#pragma unroll
    for (int q = 0; q < kClusNc / 32; ++q) {
      const unsigned msk = __ballot_sync(0xffffffffu, f[q]);
      if (f[q]) a.list[(size_t)i * nc + base + __popc(msk & ((1u << lane) - 1u))] = 32 * q + lane;
      base += __popc(msk);
    }
    if (lane == 0) a.cnt[i] = base;
  }
  __syncthreads();
  // L_s: row-major into a.S (for the grid products), packed plain into
  // a.spk followed by its inverted diagonal blocks (for the one-CTA solves)
  cta_chol_packed(P, nc, Pt, a.info, nullptr, nullptr, a.spk + prow(nc));
  for (int e = tid; e < nc * nc; e += kST) {
    const int i = e / nc, j = e % nc;
    a.S[e] = (j <= i) ? P[prow(i) + j] : 0.f;
  }
  for (int e = tid; e < prow(nc); e += kST) a.spk[e] = P[e];
}
__global__ void __launch_bounds__(kST) k_small_s(RedArgs<float> a) {
  k_small_s_body(a);
}

// k_small_x (grid): X = B (L_s (x) I_3) by blocks of kXRows rows: the block's
// rows of B-check are converted to float32 once into shared memory (a float64
// conversion costs a float64-pipe issue on GB300), then every thread forms
// entries of the block from them
constexpr int kXRows = 4;                  // rows of X per staged block
__device__ __forceinline__ void k_small_x_body(RedArgs<float> a) {
  const int nc = *a.nc_dev;
  if (nc == 0 || nc > a.small_lim) return;
  red_layout(a, nc);
  const int n3 = 3 * nc;
  __shared__ float bs[kXRows][3 * kClusNc];
  const int nblk = (n3 + kXRows - 1) / kXRows;
  for (int rb = blockIdx.x; rb < nblk; rb += gridDim.x) {
    const int r0 = rb * kXRows;
    __syncthreads();
    for (int e = threadIdx.x; e < kXRows * n3; e += blockDim.x) {
      const int rr = e / n3, c = e - rr * n3, row = r0 + rr;
      bs[rr][c] = row < n3 ? (float)a.Bc[(size_t)row * n3 + c] : 0.f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kXRows * n3; e += blockDim.x) {
      const int rr = e / n3, colx = e - rr * n3, row = r0 + rr;
      if (row >= n3) continue;
      const int i = row / 3, k = colx / 3, b = colx % 3;
      float acc = 0.f;
      const int ci = a.cnt[i];
#pragma unroll 4
      for (int q = 0; q < ci; ++q) {
        const int j = a.list[(size_t)i * nc + q];
        if (j >= k) acc += bs[rr][3 * j + b] * a.S[(size_t)j * nc + k];
      }
      a.X[(size_t)row * n3 + colx] = acc;
    }
  }
}
__global__ void __launch_bounds__(256) k_small_x(RedArgs<float> a) {
  k_small_x_body(a);
}

// k_small_n (grid): N = I + (L_s (x) I_3)^T X, lower part, packed.
// N = I + (L_s (x) I_3)^T X, lower triangle, by 32 x 32 tiles: CTA `tile`
// takes row tile ti and column tile tj <= ti of the lower triangle (tiles
// beyond 3 n_c exit).  Entry (row = 3 i + ax, col) is 1[row == col] plus the
// sum over j >= i of L_s[j][i] X[3 j + ax][col], accumulated in increasing j.
// X rows 3 j + ax and the tile's L_s entries are staged in shared memory
// kNJ values of j at a time; a thread keeps 4 rows of one column.
constexpr int kNJ = 16;
constexpr int kNTiles = (3 * kClusNc + 31) / 32 * ((3 * kClusNc + 31) / 32 + 1) / 2;
__device__ __forceinline__ void k_small_n_body(RedArgs<float> a, int tile) {
  __shared__ float Xs[3 * kNJ][32];
  __shared__ float Ls[kNJ][12];
  const int nc = *a.nc_dev;
  if (nc == 0 || nc > a.small_lim) return;
  const int n3 = 3 * nc, nt = (n3 + 31) / 32;
  if (tile >= nt * (nt + 1) / 2) return;
  int ti = 0;
  while ((ti + 1) * (ti + 2) / 2 <= tile) ++ti;
  const int tj = tile - ti * (ti + 1) / 2;
  red_layout(a, nc);
  const int R0 = 32 * ti, C0 = 32 * tj, i0 = R0 / 3;
  const int tid = threadIdx.x, col = tid & 31, rw = tid >> 5;
  int iv[4], ax[4];
  float acc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = R0 + rw + 8 * q;
    iv[q] = row / 3 - i0;            // 0 .. 11
    ax[q] = row % 3;
    acc[q] = (row == C0 + col) ? 1.f : 0.f;
  }
  for (int j0 = i0; j0 < nc; j0 += kNJ) {
    __syncthreads();
    for (int e = tid; e < 3 * kNJ * 32; e += blockDim.x) {
      const int rr = e >> 5, c = e & 31, xr = 3 * j0 + rr;
      Xs[rr][c] = (xr < n3 && C0 + c < n3) ? a.X[(size_t)xr * n3 + C0 + c] : 0.f;
    }
    for (int e = tid; e < kNJ * 12; e += blockDim.x) {
      const int jj = e / 12, ii = e % 12, j = j0 + jj, i = i0 + ii;
      Ls[jj][ii] = (j < nc && i < nc && j >= i) ? a.S[(size_t)j * nc + i] : 0.f;
    }
    __syncthreads();
    const int jn = min(kNJ, nc - j0);
    for (int jj = 0; jj < jn; ++jj)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += Ls[jj][iv[q]] * Xs[3 * jj + ax[q]][col];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = R0 + rw + 8 * q, c = C0 + col;
    if (row < n3 && c <= row) a.N[prow(row) + c] = acc[q];   // packed lower (k_small_v's layout)
  }
}
__global__ void __launch_bounds__(256) k_small_n(RedArgs<float> a) {
  k_small_n_body(a, blockIdx.x);
}

// Float64 refinement products.  GB300 issues a warp-wide float64 FMA about
// every 64 cycles per SM sub-partition, so these loops are laid out to keep
// the number of float64 warp instructions small: thread (vertex i, part q)
// of kRP parts accumulates the three rows of vertex i over every kRP-th
// term, the kRP parts (consecutive lanes) are summed by shuffles.  t is the
// thread's index among nt threads taking part (nt a multiple of 32, the
// same loop trip count in every lane).
constexpr int kRP = 16;

// w = S v with S = Sigma^-1[c, c] (x) I_3 (S64 gathered by k_small_s)
__device__ void refine_sv(const RedArgs<float>& a, int nc, int t, int nt) {
  const int total = kRP * nc;
  for (int base = 0; base < total; base += nt) {
    const int item = base + t;
    const bool ok = item < total;
    const int i = ok ? item / kRP : 0, q = item % kRP;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (ok) {
      const double* srow = a.S64 + (size_t)i * nc;
      for (int j = q; j < nc; j += kRP) {
        const double sij = srow[j];
        s0 += sij * a.v[3 * j];
        s1 += sij * a.v[3 * j + 1];
        s2 += sij * a.v[3 * j + 2];
      }
    }
#pragma unroll
    for (int o = kRP / 2; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (ok && q == 0) {
      a.w[3 * i] = s0;
      a.w[3 * i + 1] = s1;
      a.w[3 * i + 2] = s2;
    }
  }
}

// rho = y - v - B w over the block-row lists of B; returns this thread's
// share of |rho|^2
__device__ double refine_rho(const RedArgs<float>& a, int nc, int t, int nt) {
  const int total = kRP * nc, n3 = 3 * nc;
  double r2 = 0.0;
  for (int base = 0; base < total; base += nt) {
    const int item = base + t;
    const bool ok = item < total;
    const int i = ok ? item / kRP : 0, q = item % kRP;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (ok) {
      const double* b0 = a.Bc + (size_t)(3 * i) * n3;
      const double* b1 = b0 + n3;
      const double* b2 = b1 + n3;
      const int* li = a.list + (size_t)i * nc;
      const int ci = a.cnt[i];
      for (int e = q; e < ci; e += kRP) {
        const int j3 = 3 * li[e];
        const double w0 = a.w[j3], w1 = a.w[j3 + 1], w2 = a.w[j3 + 2];
        s0 += b0[j3] * w0 + b0[j3 + 1] * w1 + b0[j3 + 2] * w2;
        s1 += b1[j3] * w0 + b1[j3 + 1] * w1 + b1[j3 + 2] * w2;
        s2 += b2[j3] * w0 + b2[j3 + 1] * w1 + b2[j3 + 2] * w2;
      }
    }
#pragma unroll
    for (int o = kRP / 2; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (ok && q == 0) {
      const double acc[3] = {s0, s1, s2};
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const int row = 3 * i + ax;
        const double rr = a.y[row] - a.v[row] - acc[ax];
        a.rho[row] = rr;
        r2 += rr * rr;
      }
    }
  }
  return r2;
}

// Block column j of V = L^-1 (n x n, row-major) from the packed factor P:
// V_jj = L_jj^-1, then down the column V_kj = -L_kk^-1 sum_{i = j .. k-1} L_ki V_ij.
// The sums are formed as the blocks V_kj become known: a group of 64 threads owns
// the block rows 1 + group and 9 + group and keeps their sums in registers (4 x 4
// values per thread: rows ti + 8 p, columns tj + 8 q), so a step is one product per
// row and the product with the inverted diagonal block.  The diagonal blocks of P
// are inverted ones, unless DI holds those.  `done`, if given, counts the panels
// of P that are there, and step k waits for panel k.
constexpr int kULd = 36;
constexpr size_t kInvSmem = sizeof(float) * (size_t)(3 + 16) * 32 * kULd;
__device__ __forceinline__ void inverse_column(const float* P, const float* DI, float* V, int n, int j,
                                               const unsigned* done, int* info, float* sm) {
  const int nb = (n + 31) / 32;
  const int tid = threadIdx.x, gr = tid >> 6, tq = tid & 63, ti = tq >> 3, tj = tq & 7;
  const int lane = tid & 31, wid = tid >> 5;
  float(*VT)[kULd] = reinterpret_cast<float(*)[kULd]>(sm);     // V_kj [column][row]
  float(*St)[kULd] = VT + 32;                                  // the sum of row k [column][row]
  float(*Di)[kULd] = St + 32;                                  // L_kk^-1
  float(*Lk)[kULd] = Di + 32 + gr * 64;                        // L_ik of the group's rows
  float acc[2][4][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[h][p][q] = 0.f;
  for (int k = j; k < nb; ++k) {
    if (done && tid == 0) {
      int polls = 0;
      unsigned v;
      do {
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
      } while (v <= (unsigned)k && ++polls <= kSpinLimit);
      if (v <= (unsigned)k) {      // (gave up: the step fails, later panels are not waited for)
        atomicOr(info, kInfoTimeout);
        done = nullptr;
      }
      __threadfence();
    }
    __syncthreads();               // and the tiles of the step before are read
    // (past L1: a line read for an earlier panel may hold the start of this one)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = 1 + gr + 8 * h;
      if (i <= k || i >= nb) continue;
      float4 f[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tq + 64 * u, r = 32 * i + (e >> 3);
        f[u] = r < n ? __ldcg(reinterpret_cast<const float4*>(P + prow(r) + 32 * k) + (e & 7))
                     : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tq + 64 * u;
        *reinterpret_cast<float4*>(&Lk[32 * h + (e >> 3)][4 * (e & 7)]) = f[u];
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = tid + kST * h, r = e >> 5, c = e & 31;
      float v = 0.f;               // zero above the diagonal and past n
      if (c <= r && 32 * k + r < n)
        v = DI ? __ldcg(DI + 1024 * k + e) : __ldcg(P + prow(32 * k + r) + 32 * k + c);
      Di[r][c] = v;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = 1 + gr + 8 * h;
      if (i == k) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) St[tj + 8 * q][ti + 8 * p] = acc[h][p][q];
      }
    }
    __syncthreads();
    // row `lane`, columns wid and wid + 16 of V_kj
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = wid + 16 * h;
      float o = 0.f;
      if (k == j) {
        o = Di[lane][c];
      } else {
#pragma unroll
        for (int l = 0; l < 32; l += 4) {
          const float4 dv = *reinterpret_cast<const float4*>(&Di[lane][l]);
          const float4 sv = *reinterpret_cast<const float4*>(&St[c][l]);
          o -= dv.x * sv.x + dv.y * sv.y + dv.z * sv.z + dv.w * sv.w;
        }
      }
      VT[c][lane] = o;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = wid + 16 * h;
      if (32 * k + r < n && 32 * j + lane < n)
        V[(size_t)(32 * k + r) * n + 32 * j + lane] = VT[lane][r];
      const int i = 1 + gr + 8 * h;
      if (i <= k || i >= nb) continue;
#pragma unroll 2
      for (int l = 0; l < 32; l += 4) {
        float4 x[4], y[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) x[p] = *reinterpret_cast<const float4*>(&Lk[32 * h + ti + 8 * p][l]);
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(&VT[tj + 8 * q][l]);
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            acc[h][p][q] += x[p].x * y[q].x + x[p].y * y[q].y + x[p].z * y[q].z + x[p].w * y[q].w;
      }
    }
  }
  __syncthreads();                 // (the next column reuses the tiles)
}

// k_small_v: a cluster of kVCl CTAs.  CTA 0 factors N in its shared memory and
// publishes every panel; the others form the inverses beside it, V_s = L_s^-1
// and then the columns of V = L_N^-1, each step as soon as its panel is there,
// so that all but the last step of every column is done when the factor is.
// (They wait for CTA 0 only; the CTAs of a cluster run together.)  As a kernel of
// its own after the factor, V took 62 us of a 536 us iteration (30k face, n_c =
// 92, under a tracer); beside it a frame takes 36.3 -> 35.4 ms (5k: 27.1 -> 26.4).
constexpr int kVCl = 8;
__device__ __forceinline__ void k_small_v_body(RedArgs<float> a) {
  extern __shared__ __align__(16) float smem_f[];
  const int nc = *a.nc_dev;
  if (nc == 0 || nc > a.one_cta_max) return;
  red_layout(a, nc);
  const int n3 = 3 * nc, cta = blockIdx.x % kVCl;
  if (cta == 0) {
    float* A = smem_f;                      // prow(kSmallN3) floats
    float* Pt = A + prow(kSmallN3);         // 32 x kPtLd
    // packed N (padding included: prow(n3) is a multiple of 4)
    const float4* gN = reinterpret_cast<const float4*>(a.N);
    float4* sN = reinterpret_cast<float4*>(A);
#pragma unroll 4
    for (int e = threadIdx.x; e < prow(n3) / 4; e += kST) sN[e] = gN[e];
    __syncthreads();
    cta_chol_packed(A, n3, Pt, a.info, a.N, a.bar + kPanelsDone, nullptr);
    return;
  }
  const int w = cta - 1, nw = kVCl - 1;
  // one column of V_s for the CTAs with the shorter columns of V
  for (int j = nw - 1 - w; 32 * j < nc; j += nw)
    inverse_column(a.spk, a.spk + prow(nc), a.Vs, nc, j, nullptr, a.info, smem_f);
  for (int b = 0; 32 * b * nw < n3; ++b) {      // columns forth and back over the CTAs
    const int j = b * nw + (b & 1 ? nw - 1 - w : w);
    if (32 * j < n3)
      inverse_column(a.N, nullptr, a.X, n3, j, a.bar + kPanelsDone, a.info, smem_f);
  }
}
__global__ void __launch_bounds__(kST) k_small_v(RedArgs<float> a) {
  k_small_v_body(a);
}

// k_small_u: the inverses after the factor of the cluster form, a CTA per block
// column (the first kUN CTAs V of L_N, the others V_s of L_s)
constexpr int kUN = kClusN3 / 32, kUCtas = kUN + kClusNc / 32;
__device__ __forceinline__ void k_small_u_body(RedArgs<float> a, int cta) {
  extern __shared__ __align__(16) float smem_f[];
  const int nc = *a.nc_dev;
  if (nc <= a.one_cta_max || nc > a.small_lim) return;
  red_layout(a, nc);
  const int n3 = 3 * nc, j = cta < kUN ? cta : cta - kUN;
  if (cta < kUN) {
    if (32 * j < n3) inverse_column(a.N, nullptr, a.X, n3, j, nullptr, a.info, smem_f);
  } else if (32 * j < nc) {
    inverse_column(a.spk, a.spk + prow(nc), a.Vs, nc, j, nullptr, a.info, smem_f);
  }
}
__global__ void __launch_bounds__(kST) k_small_u(RedArgs<float> a) {
  k_small_u_body(a, blockIdx.x);
}

// k_small_solve: y = B u_c, v = (V_s (x) I)^T V^T V (L_s (x) I)^T y and its
// float64-residual refinement (same stopping rule as the grid form), on a
// cluster of kSolveCl CTAs: the vectors live in global memory and a cluster
// barrier separates the products.  Warps and threads are numbered interleaved
// over the CTAs, so that every SM gets its share of the float64 work.
// (512 threads a CTA: 2.4 % more time for a 5k face's frame, 0.3 % for 60k faces.)
constexpr int kSolveCl = 8, kSolveT = 256;
constexpr int kSolveW = kSolveT / 32;       // warps per CTA
__device__ __forceinline__ void k_small_solve_body(RedArgs<float> a) {
  namespace cgx = cooperative_groups;
  cgx::cluster_group cl = cgx::this_cluster();
  __shared__ float part[3][kSolveW][32];
  __shared__ double wred[kSolveW];
  __shared__ double nrm_parts[2][kSolveCl];
  const int nc = *a.nc_dev;
  if (nc == 0 || nc > a.small_lim) return;          // uniform over the cluster
  // every CTA of the cluster has to have started before another one stores into
  // its shared memory: arrive here, wait just before the first such store
  auto started = cl.barrier_arrive();
  red_layout(a, nc);
  const int n3 = 3 * nc, rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int gw = wid * kSolveCl + rank, nw = kSolveW * kSolveCl;
  const int gt = 32 * gw + lane, nt = 32 * nw;
  float* t = a.fv;
  float* l = a.fv + n3;
  const float* V = a.X;
  // sum over the cluster in slot `slot` (one barrier; the same value everywhere)
  auto cluster_sum = [&](double v, int slot) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) wred[wid] = v;
    __syncthreads();
    if (tid < kSolveCl) {
      double s = 0.0;
      for (int w = 0; w < kSolveW; ++w) s += wred[w];
      cl.map_shared_rank(&nrm_parts[slot][0], tid)[rank] = s;
    }
    cl.sync();
    double s = 0.0;
    for (int q = 0; q < kSolveCl; ++q) s += nrm_parts[slot][q];
    return s;
  };
  auto apply = [&](const double* p, bool add) {
    // t = (L_s (x) I)^T p, one warp per entry
    for (int e = gw; e < n3; e += nw) {
      const int i = e / 3, ax = e % 3;
      float acc = 0.f;
#pragma unroll 4
      for (int j = i + lane; j < nc; j += 32) acc += a.S[(size_t)j * nc + i] * (float)p[3 * j + ax];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) t[e] = acc;
    }
    cl.sync();
    // l = V t, one warp per two rows (their loads in flight together)
    for (int i = gw; i < n3; i += 2 * nw) {
      const int i1 = i + nw;
      float a0 = 0.f, a1 = 0.f;
#pragma unroll 4
      for (int j = lane; j < n3; j += 32) {
        const float tv = t[j];
        if (j <= i) a0 += V[(size_t)i * n3 + j] * tv;
        if (j <= i1 && i1 < n3) a1 += V[(size_t)i1 * n3 + j] * tv;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        a1 += __shfl_xor_sync(0xffffffffu, a1, o);
      }
      if (lane == 0) {
        l[i] = a0;
        if (i1 < n3) l[i1] = a1;
      }
    }
    cl.sync();
    // t = V^T l: block column b on CTA b, its warps share the rows (lane = column)
    for (int b = rank; 32 * b < n3; b += kSolveCl) {
      const int j = 32 * b + lane;
      float acc = 0.f;
      if (j < n3)
#pragma unroll 8
        for (int i = 32 * b + wid; i < n3; i += kSolveW) acc += V[(size_t)i * n3 + j] * l[i];
      __syncthreads();
      part[0][wid][lane] = acc;
      __syncthreads();
      if (wid == 0 && j < n3) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kSolveW; ++w) s += part[0][w][lane];
        t[j] = s;
      }
    }
    cl.sync();
    // v (+)= (V_s (x) I)^T t
    for (int b = rank; 32 * b < nc; b += kSolveCl) {
      const int i = 32 * b + lane;
      float s0 = 0.f, s1 = 0.f, s2 = 0.f;
      if (i < nc)
#pragma unroll 4
        for (int j = 32 * b + wid; j < nc; j += kSolveW) {
          const float vs = a.Vs[(size_t)j * nc + i];
          s0 += vs * t[3 * j];
          s1 += vs * t[3 * j + 1];
          s2 += vs * t[3 * j + 2];
        }
      __syncthreads();
      part[0][wid][lane] = s0;
      part[1][wid][lane] = s1;
      part[2][wid][lane] = s2;
      __syncthreads();
      if (wid < 3 && i < nc) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kSolveW; ++w) s += part[wid][w][lane];
        const double v0 = add ? a.v[3 * i + wid] : 0.0;
        if (add) a.vp[3 * i + wid] = v0;
        a.v[3 * i + wid] = v0 + (double)s;
      }
    }
    cl.sync();
  };
  // y = B u_c over the block lists (kRP lanes per block row), |y2|^2
  for (int base = 0; base < kRP * nc; base += nt) {
    const int item = base + gt;
    const bool ok = item < kRP * nc;
    const int i = ok ? item / kRP : 0, q = item % kRP;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if (ok) {
      const double* b0 = a.Bc + (size_t)(3 * i) * n3;
      const double* b1 = b0 + n3;
      const double* b2 = b1 + n3;
      const int ci = a.cnt[i];
      for (int e = q; e < ci; e += kRP) {
        const int j = a.list[(size_t)i * nc + e];
        if (!FSIM_CHECK_IDX(a.clist[j], a.n2, CHECK_CLIST)) continue;
        const double* uj = a.u + 3 * (size_t)a.clist[j];
        const double u0 = uj[0], u1 = uj[1], u2 = uj[2];
        const int j3 = 3 * j;
        s0 += b0[j3] * u0 + b0[j3 + 1] * u1 + b0[j3 + 2] * u2;
        s1 += b1[j3] * u0 + b1[j3 + 1] * u1 + b1[j3 + 2] * u2;
        s2 += b2[j3] * u0 + b2[j3 + 1] * u1 + b2[j3 + 2] * u2;
      }
    }
#pragma unroll
    for (int o = kRP / 2; o > 0; o >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if (ok && q == 0) {
      a.y[3 * i] = s0;
      a.y[3 * i + 1] = s1;
      a.y[3 * i + 2] = s2;
    }
  }
  double ys = 0.0;
  for (int e = gt; e < 3 * a.n2; e += nt) ys += (double)a.y2[e] * (double)a.y2[e];
  cl.barrier_wait(std::move(started));
  ys = cluster_sum(ys, 0);
  apply(a.y, false);
  double prev = -1.0;
  for (int it = 0;; ++it) {
    refine_sv(a, nc, gt, nt);
    cl.sync();
    // two slots in turn: a CTA may still read the one of the step before
    const double r2 = cluster_sum(refine_rho(a, nc, gt, nt), (it + 1) & 1);
    if (refined(r2, prev, ys, it, a.refine)) {
      if (step_lost(r2, prev))
        for (int e = gt; e < n3; e += nt) a.v[e] = a.vp[e];
      if (gt == 0 && !accepted(r2, prev, ys)) atomicOr(a.info, kInfoStalled);
      break;
    }
    prev = r2;
    apply(a.rho, true);
  }
  cl.sync();       // no CTA leaves while its shared memory may still be written
}
__global__ void __launch_bounds__(kSolveT) k_small_solve(RedArgs<float> a) {
  k_small_solve_body(a);
}

// ---------------------------------------------------------------------------
// k_clus_v: the same factorisation for kSmallNc < n_c <= kClusNc on a cluster
// of kCl CTAs.  32-row blocks of the packed N are spread block-cyclically over
// the CTAs' shared memory.  Per panel the owner factors its diagonal block and
// the others copy it through distributed shared memory; each CTA solves its own
// rows of the panel and stores them into the panel copy of every CTA
// (distributed shared-memory stores, visible after the cluster barrier that
// follows), then updates only its own rows.  The diagonal blocks are
// inverted after the factorisation, one warp per block, and the rows go back to
// global memory.
// ---------------------------------------------------------------------------
constexpr int kClusRowsMax = 32 * ((kClusN3 / 32 + kCl - 1) / kCl);   // own rows per CTA
// largest packed storage of the rows one CTA owns (padded row lengths)
constexpr int clus_aloc() {
  int mx = 0;
  for (int rank = 0; rank < kCl; ++rank) {
    int tot = 0;
    for (int b = rank; b < kClusN3 / 32; b += kCl)
      for (int rr = 0; rr < 32; ++rr) tot += 4 * ((32 * b + rr + 4) / 4);
    mx = tot > mx ? tot : mx;
  }
  return mx + 64;
}
constexpr int kClusALoc = clus_aloc();
static_assert(kClusALoc % 4 == 0, "panel scratch must stay 16-byte aligned");
constexpr size_t kClusSmem =
    sizeof(float) * ((size_t)kClusALoc + 32 * (size_t)kClusN3);

// (__maxnreg__ rather than __launch_bounds__: with the latter ptxas settles
// on 64 registers and spills; 512 threads x 128 registers fill one SM)
__device__ __forceinline__ void k_clus_v_body(RedArgs<float> a) {
  namespace cgx = cooperative_groups;
  cgx::cluster_group cl = cgx::this_cluster();
  extern __shared__ float smem_f[];
  __shared__ float Ds[32][33];
  __shared__ float dv[32];
  __shared__ float dvown[kClusRowsMax];            // 1 / L_ii of own rows
  __shared__ float Dinv[kClusRowsMax / 32][32][33];  // own diagonal blocks, inverted at the end
  __shared__ int loff[kClusRowsMax];
  const int nc = *a.nc_dev;
  if (nc <= a.one_cta_max || nc > kClusNc) return;  // uniform over the cluster
  red_layout(a, nc);
  const int n3 = 3 * nc, nblk = (n3 + 31) / 32;
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float* A = smem_f;                               // own rows, packed
  float* Pt = A + kClusALoc;                       // 32 x kClusN3, panel by global row - k1
  // own rows: block b is owned by b % kCl; local row lb * 32 + (r % 32)
  auto lrow = [&](int r) { return ((r >> 5) / kCl) * 32 + (r & 31); };
  if (tid < kClusRowsMax) {
    int off = 0;
    for (int lr = 0; lr < tid; ++lr) {
      const int r = ((lr >> 5) * kCl + rank) * 32 + (lr & 31);
      off += 4 * ((r + 4) / 4);                    // padded length of row r
    }
    loff[tid] = off;
  }
  __syncthreads();
  auto Ael = [&](int r, int c) -> float& { return A[loff[lrow(r)] + c]; };
  // load own rows of the packed N.  A packed row r is a 16-byte
  // aligned run of 4 (r / 4 + 1) floats in both layouts (padding included,
  // never read), so rows move as float4: warp w takes own rows w, w + 16, ..
  // two rows and all their loads in flight at once (a row has <= 96 float4)
  static_assert(kClusN3 / 4 <= 96, "a packed row must fit three float4 per lane");
  for (int lr0 = wid; lr0 < kClusRowsMax; lr0 += 2 * kSW) {
    float4 v[2][3];
    int len4[2];
    const float4* src[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int lr = lr0 + h * kSW;
      const int r = 32 * (((lr >> 5) * kCl) + rank) + (lr & 31);
      len4[h] = (lr < kClusRowsMax && r < n3) ? (r >> 2) + 1 : 0;
      src[h] = reinterpret_cast<const float4*>(a.N + prow(r < n3 ? r : 0));
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (lane + 32 * u < len4[h]) v[h][u] = src[h][lane + 32 * u];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (len4[h] == 0) continue;
      float4* dst = reinterpret_cast<float4*>(A + loff[lr0 + h * kSW]);
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (lane + 32 * u < len4[h]) dst[lane + 32 * u] = v[h][u];
    }
  }
  __syncthreads();

  // ---- Cholesky of N over the cluster --------------------------------------
  for (int k = 0; k < nblk; ++k) {
    const int k0 = 32 * k, kb = min(32, n3 - k0), k1 = k0 + kb, m = n3 - k1;
    const int owner = k % kCl;
    if (rank == owner) {
      for (int e = tid; e < 32 * 32; e += kST) {
        const int i = e >> 5, j = e & 31;
        Ds[i][j] = (i < kb && j <= i) ? Ael(k0 + i, k0 + j) : 0.f;
      }
      __syncthreads();
      eliminate_diag(Ds, kb);
      if (tid < kb) {
        float d = Ds[tid][tid];
        if (!(d > 0.f)) {
          atomicOr(a.info, kInfoPivot);
          d = 1.f;
          Ds[tid][tid] = 1.f;
        }
        float rs = rsqrtf(d);
        rs = rs * (1.5f - 0.5f * d * rs * rs);
        dv[tid] = rs;
      } else if (tid < 32) {
        dv[tid] = 1.f;
      }
      __syncthreads();
      for (int e = tid; e < kb * 32; e += kST) {
        const int i = e >> 5, j = e & 31;
        if (j < i) Ds[i][j] *= dv[j];
      }
      __syncthreads();
      if (tid < kb) Ds[tid][tid] = Ds[tid][tid] * dv[tid];
      if (tid < 32) dvown[lrow(k0) + tid] = dv[tid];   // kept for the inverse below
      __syncthreads();
    }
    cl.sync();
    if (rank != owner) {     // the owner's diagonal factor and 1/diag
      const float* rD = cl.map_shared_rank(&Ds[0][0], owner);
      const float* rv = cl.map_shared_rank(&dv[0], owner);
#pragma unroll
      for (int e = tid; e < 32 * 33; e += kST) (&Ds[0][0])[e] = rD[e];
      if (tid < 32) dv[tid] = rv[tid];
    }
    __syncthreads();
    // own panel rows: x L_kk^T = a (registers), into A and into the panel
    // copy of every CTA of the cluster (remote stores, made visible by the
    // cluster barrier below); one warp per own block below the panel
    for (int idx = tid; idx < kClusRowsMax; idx += kST) {
      const int b = ((idx >> 5) * kCl) + rank;
      const int r = 32 * b + (idx & 31);
      if (b > k && r < n3) {
        float* row = &Ael(r, k0);
        float x[32];
#pragma unroll
        for (int l = 0; l < 32; ++l) x[l] = row[l];
#pragma unroll
        for (int q = 0; q < 32; ++q) {
          x[q] *= dv[q];
#pragma unroll
          for (int l = q + 1; l < 32; ++l) x[l] -= x[q] * Ds[l][q];
        }
#pragma unroll
        for (int l = 0; l < 32; ++l) row[l] = x[l];
#pragma unroll
        for (int l = 0; l < 32; ++l) Pt[l * kClusN3 + (r - k1)] = x[l];
        for (int q = 1; q < kCl; ++q) {
          float* dst = cl.map_shared_rank(Pt, (rank + q) % kCl);
#pragma unroll
          for (int l = 0; l < 32; ++l) dst[l * kClusN3 + (r - k1)] = x[l];
        }
      }
    }
    // the owner keeps the plain diagonal factor (inverted after the loop)
    if (rank == owner)
      for (int e = tid; e < kb * 32; e += kST) {
        const int i = e >> 5, j = e & 31;
        if (j <= i) Ael(k0 + i, k0 + j) = Ds[i][j];
      }
    cl.sync();
    // trailing update of own rows: A(i, j) -= P_i . P_j, 4 x 4 tiles
    if (m > 0) {
      // only this CTA's 4-row tiles (tile I covers rows k1 + 4I ..; a 32-row
      // block b below the panel holds tiles (32b - k1)/4 + 0..7, each with
      // I + 1 column tiles J <= I), numbered consecutively over the threads
      const int mb = (m + 3) >> 2;
      int bfirst = rank;
      while (bfirst <= k) bfirst += kCl;
      int total = 0;
      for (int b = bfirst; 32 * b < n3; b += kCl) {
        const int I0 = (32 * b - k1) >> 2, ns = min(8, mb - I0);
        total += ns * (I0 + 1) + ns * (ns - 1) / 2;
      }
      for (int u = tid; u < total; u += kST) {
        int rem = u, I = 0, J = 0;
        for (int b = bfirst; 32 * b < n3; b += kCl) {
          const int I0 = (32 * b - k1) >> 2, ns = min(8, mb - I0);
          const int cnt = ns * (I0 + 1) + ns * (ns - 1) / 2;
          if (rem < cnt) {
            int s2 = 0;
            while (rem >= I0 + s2 + 1) { rem -= I0 + s2 + 1; ++s2; }
            I = I0 + s2;
            J = rem;
            break;
          }
          rem -= cnt;
        }
        float acc[4][4];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[p][q] = 0.f;
#pragma unroll 4
        for (int l = 0; l < 32; ++l) {
          const float4 av = *reinterpret_cast<const float4*>(Pt + l * kClusN3 + 4 * I);
          const float4 bv = *reinterpret_cast<const float4*>(Pt + l * kClusN3 + 4 * J);
          const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[p][q] += ar[p] * br[q];
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const int i = 4 * I + p;
          if (i >= m) break;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int jj = 4 * J + q;
            if (jj <= i) Ael(k1 + i, k1 + jj) -= acc[p][q];
          }
        }
      }
    }
    __syncthreads();
  }
  // L_kk^-1 of every own diagonal block (for the solves), one warp per
  // block, all blocks at once: column `lane` by substitution in registers
  {
    const int b = rank + kCl * wid;
    if (b < nblk) {
      const int k0 = 32 * b, kb = min(32, n3 - k0), lb = lrow(k0);
      float (*D)[33] = Dinv[wid];
      for (int i = 0; i < 32; ++i)
        D[i][lane] = (i < kb && lane <= i) ? A[loff[lb + i] + k0 + lane] : 0.f;
      __syncwarp();
      float x[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) x[i] = (i == lane) ? 1.f : 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        x[i] *= dvown[lb + i];
#pragma unroll
        for (int l = i + 1; l < 32; ++l) x[l] -= D[l][i] * x[i];
      }
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < kb && i >= lane) A[loff[lb + i] + k0 + lane] = x[i];
    }
  }
  __syncthreads();
  // own rows back to the packed N
  for (int lr = wid; lr < kClusRowsMax; lr += kSW) {
    const int r = 32 * (((lr >> 5) * kCl) + rank) + (lr & 31);
    if (r >= n3) continue;
    const float4* src = reinterpret_cast<const float4*>(A + loff[lr]);
    float4* dst = reinterpret_cast<float4*>(a.N + prow(r));
    for (int u = lane; u < (r >> 2) + 1; u += 32) dst[u] = src[u];
  }
  cl.sync();       // no CTA leaves while its shared memory may still be read
}
__global__ void __maxnreg__(128) k_clus_v(RedArgs<float> a) {
  k_clus_v_body(a);
}

constexpr size_t kSmallSmemS = sizeof(float) * ((size_t)prow(kClusNc) + 32 * kPtLd);
constexpr size_t kSmallSmemV = sizeof(float) * ((size_t)prow(kSmallN3) + 32 * kPtLd);
static_assert(kInvSmem <= kSmallSmemV, "the CTAs beside the factor use its shared memory");

template <typename FT>
RedArgs<FT> make_args(const DevMesh& m, const double* u, const FT* y2, double* z2, int* info,
                      int refine) {
  RedArgs<FT> a{};
  a.n2 = m.n2; a.refine = refine;
  a.nc_dev = m.counters + 3;
  a.base = std::is_same<FT, double>::value ? (FT*)m.red : (FT*)m.redf;
  a.dtail_end = m.red + m.red_cap;      // float64 vectors at the tail of m.red
  a.ibase = m.bocc + (size_t)m.nc_cap * m.nc_cap;
  a.clist = m.clist; a.Sinv = m.Sinv; a.Bc = m.Bc; a.bocc = m.bocc;
  a.u = u; a.y2 = y2; a.z2 = z2;
  a.info = info;
  a.small_lim = std::is_same<FT, float>::value ? kClusNc : 0;
  a.one_cta_max = std::max(0, std::min(m.one_cta_max, kSmallNc));
  a.bar = reinterpret_cast<unsigned*>(m.bocc + 2 * (size_t)m.nc_cap * m.nc_cap + m.nc_cap);
  return a;
}

// Launch one of the cluster kernels: a cluster of `ctas` CTAs per system.
template <typename K, typename A>
cudaError_t launch_clusters(cudaStream_t s, K kernel, int ctas, int threads, size_t smem, int nsys,
                            const A& arg) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, nsys);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, arg);
  count_launch();
  return e;
}

// The two kernels of the grid form for one frame: cooperative launches, since
// their CTAs wait on one another (all of them are resident together).
template <typename FT>
cudaError_t launch_grid(cudaStream_t s, RedArgs<FT> a, int ctas, bool prepare) {
  GridFrames fr{};
  fr.n = 1;
  fr.G = std::max(1, ctas);
  const RedArgs<FT>* none = nullptr;
  void* args[] = {&a, &none, &fr};
  ProfScope ps(PROF_CHOL, s);
  const void* k = prepare ? (const void*)k_grid_prepare<FT> : (const void*)k_grid_solve<FT>;
  const cudaError_t e = cudaLaunchCooperativeKernel(k, dim3(fr.G), dim3(kRT), args, 0, s);
  count_launch();
  return e;
}

// float32 factors, n_c <= kClusNc, on the side stream: one-CTA factor up to
// one_cta_max, beside the inverses of both factors; the 4-CTA cluster above it,
// then the inverses.
// No cooperative launch (whose grid must find all of its SMs free at once when
// other solves share the GPU).
cudaError_t launch_small_prepare(cudaStream_t s2, const RedArgs<float>& a, int num_sms, int nc) {
  ProfScope ps(PROF_CHOL, s2);
  k_small_s<<<1, kST, kSmallSmemS, s2>>>(a);
  k_small_x<<<2 * std::max(1, num_sms), 256, 0, s2>>>(a);
  k_small_n<<<kNTiles, 256, 0, s2>>>(a);
  count_launch(3);
  if (nc <= a.one_cta_max) return launch_clusters(s2, k_small_v, kVCl, kST, kSmallSmemV, 1, a);
  const cudaError_t e = launch_clusters(s2, k_clus_v, kCl, kST, kClusSmem, 1, a);
  if (e != cudaSuccess) return e;
  k_small_u<<<kUCtas, kST, kInvSmem, s2>>>(a);
  count_launch();
  return cudaGetLastError();
}
// the solve, and the z2 update as a plain launch
cudaError_t launch_small(cudaStream_t s, const DevMesh& m, const RedArgs<float>& a, int num_sms,
                         int nc) {
  ProfScope ps(PROF_CHOL, s);
  const int zgrid = std::max(1, std::min(2 * std::max(1, num_sms), (m.n2 + 7) / 8));
  if (nc > 0) {
    const cudaError_t e = launch_clusters(s, k_small_solve, kSolveCl, kSolveT, 0, 1, a);
    if (e != cudaSuccess) return e;
  }
  k_z2_update<<<zgrid, 256, 0, s>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

int64_t reduced_workspace_elems(int nc) {
  const int64_t n3 = 3 * (int64_t)nc;
  // small forms: S, X, packed N, L_s^-1, two FT vectors, packed L_s with its
  // inverted diagonal blocks (each rounded up to 16 bytes)
  const int64_t small = 2 * (int64_t)nc * nc + n3 * n3 + n3 * (n3 + 4) / 2 + 8 + 2 * n3 +
                        (int64_t)nc * (nc + 4) / 2 + 8 + 1024 * (((int64_t)nc + 31) / 32) + 64;
  // at the tail of the float64 buffer five float64 vectors, three norms and S64
  return std::max(small, grid_front_elems(nc)) + 5 * n3 + (int64_t)nc * nc + 64;
}

// Most float64 refinement steps of a float32 reduced factor (see step 7).
constexpr int kMixedRefineSteps = 12;

int reduced_path(int nc_host, int precision, int one_cta_max) {
  if (precision == 0 || nc_host > kClusNc) return 0;   // grid form
  if (nc_host == 0) return 1;
  return nc_host <= std::min(one_cta_max, kSmallNc) ? 2 : 3;
}

cudaError_t reduced_solve(cudaStream_t s, const DevMesh& m, const double* u, const void* y2,
                          double* z2, int* info, int num_sms, int precision, int nc_host) {
  if (nc_host <= 0)       // z2 = u
    return launch_small(s, m, make_args<float>(m, u, nullptr, z2, info, 0), num_sms, 0);
  // S .. L_N come from the side stream (reduced_prepare)
  if (cudaStreamWaitEvent(s, m.ev_join, 0) != cudaSuccess) return cudaGetLastError();
  if (precision == 0)
    return launch_grid(s, make_args<double>(m, u, (const double*)y2, z2, info, 1), num_sms, false);
  const RedArgs<float> a = make_args<float>(m, u, (const float*)y2, z2, info, kMixedRefineSteps);
  if (nc_host > kClusNc) return launch_grid(s, a, num_sms, false);
  return launch_small(s, m, a, num_sms, nc_host);
}

namespace {

// x1 = bx1 + Phi[:, c] v.  A CTA covers 32 consecutive x1 solver positions
// (coalesced reads of the rows of Phi_t) with kPhiSplit warps, each summing
// a strided share of the n_c columns; v (as float) and the c list are staged
// in shared memory.  The work is bound by load latency, hence the split.
// PAIRS: v and the sums as float pairs.  The forces v of a pair nearly cancel in
// x1; with float32 sums the worst entry's error is 0.73 u32 of the contact-free step
// at n_c = 162 (median of 40 states), with pairs 0.48, which is Phi's own rounding.
// Taken for n_c > 128, where x1 would otherwise be a backward solve from z2 on the
// solve's own stream (40 to 60k faces: 11 to 14 % more time a frame); float32 sums
// there made the whole step's median error 1.15 to 1.6 times that of the solve.
// Below, pairs would cost 0.5 to 0.9 % of a frame.
constexpr int kPhiSplit = 8;
template <bool PAIRS>
__global__ void __launch_bounds__(32 * kPhiSplit) k_phi_apply(RedArgs<float> a, int n1,
                                                             const float* __restrict__ phi_t,
                                                             const float* __restrict__ bx1,
                                                             double* __restrict__ x1) {
  constexpr int kParts = PAIRS ? 2 : 1;            // high parts, then low parts
  __shared__ float vs[kParts][3 * kClusNc];
  __shared__ int cs[kClusNc];
  __shared__ float part[kParts][kPhiSplit][3][32];
  const int nc = *a.nc_dev;
  if (nc > 0) red_tail(a, nc);
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float c[3] = {0.f, 0.f, 0.f}, e[3] = {0.f, 0.f, 0.f};
  auto add = [&](int d, float h, float l) {        // c + e += h + l
    const df s = df_two_sum(c[d], h);
    c[d] = s.hi;
    e[d] += s.lo + l;
  };
  for (int k0 = 0; k0 < nc; k0 += kClusNc) {       // n_c in chunks of the staging size
    const int kn = min(kClusNc, nc - k0);
    __syncthreads();
    for (int k = threadIdx.x; k < kn; k += blockDim.x) {
      const bool okc = FSIM_CHECK_IDX(a.clist[k0 + k], a.n2, CHECK_CLIST);
      cs[k] = okc ? a.clist[k0 + k] : 0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double v = okc ? a.v[3 * (k0 + k) + d] : 0.0;
        vs[0][3 * k + d] = (float)v;
        if (PAIRS) vs[kParts - 1][3 * k + d] = df_from_double(v).lo;
      }
    }
    __syncthreads();
    if (p < n1) {
#pragma unroll 4
      for (int k = wq; k < kn; k += kPhiSplit) {
        const float f = phi_t[(size_t)cs[k] * n1 + p];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (PAIRS) {
            const df t = df_two_prod(f, vs[0][3 * k + d]);
            add(d, t.hi, __fmaf_rn(f, vs[kParts - 1][3 * k + d], t.lo));
          } else {
            c[d] += f * vs[0][3 * k + d];
          }
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    part[0][wq][d][lane] = c[d];
    if (PAIRS) part[kParts - 1][wq][d][lane] = e[d];
  }
  __syncthreads();
  if (wq < 3 && p < n1) {
    const float b = bx1[3 * (size_t)p + wq];
    c[0] = PAIRS ? b : 0.f;
    e[0] = 0.f;
#pragma unroll
    for (int q = 0; q < kPhiSplit; ++q) {
      if (PAIRS) add(0, part[0][q][wq][lane], part[kParts - 1][q][wq][lane]);
      else c[0] += part[0][q][wq][lane];
    }
    x1[3 * (size_t)p + wq] = (double)c[0] + (double)(PAIRS ? e[0] : b);
  }
}

// ---- lock-step batches: blockIdx.y = frame, RedArgs per frame on the device
__global__ void __launch_bounds__(256) k_small_x_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_x_body(a);
}
__global__ void __launch_bounds__(kST) k_small_u_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_u_body(a, blockIdx.x);
}
__global__ void __launch_bounds__(kSolveT) k_small_solve_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_solve_body(a);       // uniform over a cluster
}
__global__ void __launch_bounds__(kST) k_small_s_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_s_body(a);
}
__global__ void __launch_bounds__(256) k_small_n_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_n_body(a, blockIdx.x);
}
__global__ void __launch_bounds__(kST) k_small_v_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_small_v_body(a);
}
// one 4-CTA cluster per frame: the cluster spans blockIdx.x, the frame is
// blockIdx.y, so the inactive test is uniform over a cluster
__global__ void __maxnreg__(128) k_clus_v_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_clus_v_body(a);
}
__global__ void __launch_bounds__(256) k_z2_update_b(const RedArgs<float>* __restrict__ A) {
  const RedArgs<float> a = A[blockIdx.y];
  if (a.active) k_z2_update_body(a, true);
}

// x1 = bx1 + Phi[:, c] v for every frame and any n_c (v from whichever path
// solved the reduced system), with bx1 read from a multi-right-hand-side
// buffer: frame f's three columns start at column col_f of rows of nr floats.
__global__ void __launch_bounds__(32 * kPhiSplit) k_phi_apply_b(const RedArgs<float>* __restrict__ A,
                                                               const int* __restrict__ cols, int n1,
                                                               const float* __restrict__ phi_t,
                                                               const float* __restrict__ bxm, int nr,
                                                               double* const* __restrict__ x1s) {
  RedArgs<float> a = A[blockIdx.y];
  if (!a.active) return;
  __shared__ float vs[3 * kClusNc];
  __shared__ int cs[kClusNc];
  __shared__ float part[kPhiSplit][3][32];
  const int nc = *a.nc_dev;
  const int col = cols[blockIdx.y];
  double* x1 = x1s[blockIdx.y];
  if (nc > 0) red_tail(a, nc);
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float c0 = 0.f, c1 = 0.f, c2 = 0.f;
  for (int k0 = 0; k0 < nc; k0 += kClusNc) {       // n_c in chunks of the staging size
    const int kn = min(kClusNc, nc - k0);
    __syncthreads();
    for (int k = threadIdx.x; k < kn; k += blockDim.x) {
      const bool okc = FSIM_CHECK_IDX(a.clist[k0 + k], a.n2, CHECK_CLIST);
      cs[k] = okc ? a.clist[k0 + k] : 0;
      vs[3 * k] = okc ? (float)a.v[3 * (k0 + k)] : 0.f;
      vs[3 * k + 1] = okc ? (float)a.v[3 * (k0 + k) + 1] : 0.f;
      vs[3 * k + 2] = okc ? (float)a.v[3 * (k0 + k) + 2] : 0.f;
    }
    __syncthreads();
    if (p < n1) {
#pragma unroll 4
      for (int k = wq; k < kn; k += kPhiSplit) {
        const float f = phi_t[(size_t)cs[k] * n1 + p];
        c0 += f * vs[3 * k];
        c1 += f * vs[3 * k + 1];
        c2 += f * vs[3 * k + 2];
      }
    }
  }
  part[wq][0][lane] = c0;
  part[wq][1][lane] = c1;
  part[wq][2][lane] = c2;
  __syncthreads();
  if (wq < 3 && p < n1)  {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < kPhiSplit; ++q) t += part[q][wq][lane];
    x1[3 * (size_t)p + wq] = (double)bxm[(size_t)p * nr + col + wq] + (double)t;
  }
}

}  // namespace

size_t reduced_args_bytes() { return sizeof(RedArgs<float>); }

void reduced_args_fill(void* dst, const DevMesh& m, int active) {
  RedArgs<float> a = make_args<float>(m, m.u, (const float*)(m.rf + 3 * (size_t)m.n1),
                                      m.r + 3 * (size_t)m.n1, m.counters + 6, kMixedRefineSteps);
  a.active = active;
  std::memcpy(dst, &a, sizeof(a));
}

namespace {
// Frames of a batch whose n_c takes the grid form, as few launches as fit:
// every frame gets an equal share of the ctas (at least kGridMinCtas).
constexpr int kGridMinCtas = 8;
cudaError_t launch_grid_b(cudaStream_t s, const RedArgs<float>* A, const RedArgs<float>* H, int nb,
                          const int* nc_host, int ctas, bool prepare) {
  std::vector<int> todo;
  for (int f = 0; f < nb; ++f)
    if (H[f].active && nc_host[f] > kClusNc) todo.push_back(f);
  const int per = std::max(1, std::min<int>(GridFrames::kMax, ctas / kGridMinCtas));
  for (size_t i = 0; i < todo.size(); i += per) {
    GridFrames fr{};
    fr.n = (int)std::min<size_t>(per, todo.size() - i);
    fr.G = std::max(1, ctas / fr.n);
    for (int q = 0; q < fr.n; ++q) fr.id[q] = (unsigned char)todo[i + q];
    RedArgs<float> unused{};
    void* args[] = {&unused, &A, &fr};
    const void* k = prepare ? (const void*)k_grid_prepare<float> : (const void*)k_grid_solve<float>;
    const cudaError_t e =
        cudaLaunchCooperativeKernel(k, dim3(fr.G * fr.n), dim3(kRT), args, 0, s);
    count_launch();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t reduced_prepare_b(cudaStream_t s2, const void* args_dev, const void* args_host, int nb,
                              const int* nc_host, int coop_ctas) {
  const auto* A = static_cast<const RedArgs<float>*>(args_dev);
  const auto* H = static_cast<const RedArgs<float>*>(args_host);
  bool any_small = false, any_clus = false;
  for (int f = 0; f < nb; ++f) {
    if (!H[f].active) continue;
    any_small |= nc_host[f] > 0 && nc_host[f] <= H[f].one_cta_max;
    any_clus |= nc_host[f] > H[f].one_cta_max && nc_host[f] <= kClusNc;
  }
  ProfScope ps(PROF_CHOL, s2);
  cudaError_t e = cudaSuccess;
  if (any_small || any_clus) {
    k_small_s_b<<<dim3(1, nb), kST, kSmallSmemS, s2>>>(A);
    k_small_x_b<<<dim3((3 * kClusNc + kXRows - 1) / kXRows, nb), 256, 0, s2>>>(A);
    k_small_n_b<<<dim3(kNTiles, nb), 256, 0, s2>>>(A);
    count_launch(3);
    if (any_small) {
      e = launch_clusters(s2, k_small_v_b, kVCl, kST, kSmallSmemV, nb, A);
      if (e != cudaSuccess) return e;
    }
    if (any_clus) {
      e = launch_clusters(s2, k_clus_v_b, kCl, kST, kClusSmem, nb, A);
      if (e != cudaSuccess) return e;
      k_small_u_b<<<dim3(kUCtas, nb), kST, kInvSmem, s2>>>(A);
      count_launch();
    }
  }
  // n_c beyond the cluster path: the grid form, all such frames side by side
  e = launch_grid_b(s2, A, H, nb, nc_host, coop_ctas, true);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t reduced_solve_b(cudaStream_t s, const void* args_dev, const void* args_host, int nb,
                            const int* nc_host, int coop_ctas) {
  const auto* A = static_cast<const RedArgs<float>*>(args_dev);
  const auto* H = static_cast<const RedArgs<float>*>(args_host);
  bool any = false;
  for (int f = 0; f < nb; ++f) any |= H[f].active && nc_host[f] > 0 && nc_host[f] <= kClusNc;
  ProfScope ps(PROF_CHOL, s);
  if (any) {
    const cudaError_t e = launch_clusters(s, k_small_solve_b, kSolveCl, kSolveT, 0, nb, A);
    if (e != cudaSuccess) return e;
  }
  const cudaError_t eg = launch_grid_b(s, A, H, nb, nc_host, coop_ctas, false);
  if (eg != cudaSuccess) return eg;
  // float64 row products, one row per lane: 256 rows per CTA of 8 warps,
  // enough CTAs to cover the rows of every frame (at least 2 per frame, also
  // for the n_c = 0 copy)
  const int zgrid = std::max(2, (H[0].n2 + 255) / 256);
  k_z2_update_b<<<dim3(zgrid, nb), 256, 0, s>>>(A);
  count_launch();
  return cudaGetLastError();
}

cudaError_t phi_apply_b(cudaStream_t s, const void* args_dev, const int* cols_dev, int nb, int n1,
                        const float* phi_t, const float* bxm, int nr, double* const* x1s_dev) {
  const auto* A = static_cast<const RedArgs<float>*>(args_dev);
  k_phi_apply_b<<<dim3((n1 + 31) / 32, nb), 32 * kPhiSplit, 0, s>>>(A, cols_dev, n1, phi_t, bxm, nr,
                                                                    x1s_dev);
  count_launch();
  return cudaGetLastError();
}

cudaError_t phi_apply(cudaStream_t s, const DevMesh& m, const double* u, const void* y2, double* z2,
                      int* info, const float* bx1, double* x1, int nc_host) {
  const RedArgs<float> a = make_args<float>(m, u, (const float*)y2, z2, info, kMixedRefineSteps);
  const auto kernel = nc_host > kClusNc ? k_phi_apply<true> : k_phi_apply<false>;
  kernel<<<(m.n1 + 31) / 32, 32 * kPhiSplit, 0, s>>>(a, m.n1, m.Phi_t, bx1, x1);
  count_launch();
  return cudaGetLastError();
}

cudaError_t reduced_prepare(cudaStream_t s, const DevMesh& m, const double* u, const void* y2,
                            double* z2, int* info, int num_sms, int precision, int nc_host) {
  if (nc_host <= 0) return cudaSuccess;
  cudaStream_t s2 = m.aux_stream;
  if (cudaEventRecord(m.ev_fork, s) != cudaSuccess || cudaStreamWaitEvent(s2, m.ev_fork, 0) != cudaSuccess)
    return cudaGetLastError();
  cudaError_t e = cudaSuccess;
  if (precision == 0) {
    e = launch_grid(s2, make_args<double>(m, u, (const double*)y2, z2, info, 1), num_sms, true);
  } else {
    const RedArgs<float> a = make_args<float>(m, u, (const float*)y2, z2, info, kMixedRefineSteps);
    e = nc_host > kClusNc ? launch_grid(s2, a, num_sms, true)
                          : launch_small_prepare(s2, a, num_sms, nc_host);
  }
  // the join is recorded even if a launch failed, so the fork always closes
  const cudaError_t ej = cudaEventRecord(m.ev_join, s2);
  return e != cudaSuccess ? e : ej;
}

}  // namespace fsim

namespace fsim {
void set_reduced_smem_limits() {
  cudaFuncSetAttribute(k_small_s, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemS);
  cudaFuncSetAttribute(k_small_v, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemV);
  cudaFuncSetAttribute(k_clus_v, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusSmem);
  cudaFuncSetAttribute(k_small_s_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemS);
  cudaFuncSetAttribute(k_small_v_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemV);
  cudaFuncSetAttribute(k_clus_v_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusSmem);
  cudaFuncSetAttribute(k_small_u, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kInvSmem);
  cudaFuncSetAttribute(k_small_u_b, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kInvSmem);
}
FSIM_CHECK_READER(check_word_reduced)

}  // namespace fsim
