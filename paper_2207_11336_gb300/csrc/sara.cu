// uSARA's handcrafted denoiser (App. B): the prox of gamma lambda ||W Psi^T x||_1 + iota_+(x) for
// the SARA dictionary Psi (the Dirac basis and the 2-D Daubechies bases db1..db8, each a multi-level
// separable DWT with periodic extension, divided by 3 so that Psi Psi^T = I), by dual
// forward-backward sub-iterations:
//   x = max(0, z - Psi u),   u <- clip(u + Psi^T x, -t, t),   t = gamma lambda w,
// warm-started from the previous call's u, and the reweighting w = rho / (rho + |Psi^T x|) that
// majorises the log-sum prior at the current image.
//
// Each DWT level works on its m x m block, analysis along axis 0 then 1,
// a[j] = sum_k f[k] x[(2 j + k) mod m] (low half, then high half), synthesis along axis 1 then 0 as the gather
// x[p] = sum_{k : p - k even} lo[k] a[((p - k) mod m) / 2] + hi[k] d[((p - k) mod m) / 2].
// The Daubechies filters are computed on the host by spectral factorisation (minimum-phase roots
// of z^(N-1) P_N((2 - z - 1/z) / 4), Durand-Kerner iteration with Newton polish).
//
// A dual sub-iteration is 2 x levels launches for all bases together: dwt_level transforms both axes of a tile in
// shared memory and applies the dual step to the coefficients that its level finishes; idwt_level rebuilds one
// level; the last one, level 0 (idwt_primal), adds up all bases in registers and forms x.  Filter lengths are
// compile-time (a block works on one basis at a time) and the filters kernel parameters, so a tap is one FMA with a
// constant operand; a lane slides along its row or column with the window in registers.
// Bound by the FMA issue and the shared-memory reads at 1024^2 (u and w, 72 MB, stay in L2) and by the u and w
// traffic, 16 B per coefficient, above.  Denoise of 10 dual iterations, before (a launch per pass, level and basis,
// elementwise steps of their own, ~150 launches per iteration) and now: 1024^2 10.46 -> 1.68 ms.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "daubechies.h"

namespace pnp {
namespace {

constexpr int SARA_FILTERS = 8, SARA_BASES = 9, MAXTAP = 16;

struct Filters {
  float f[SARA_FILTERS][2][MAXTAP];  // db1..db8: low-pass, high-pass (zero padded)
};

struct SaraState {
  int n = 0, levels = 0, iters = 0;
  double gl = 0, rho = 0;   // gamma lambda (threshold scale), log-sum floor
  Filters filt;
  float *u = nullptr, *w = nullptr;            // 9 n^2: dual variable, weights
  float *LL[2] = {nullptr, nullptr};           // approximations of the 8 bases: (n/2)^2 (odd levels), (n/4)^2 (even)
};

// r mod m for any r; a loop, since the coarsest levels' blocks can be shorter than a filter
__device__ __forceinline__ int wrap_any(int r, int m) {
  while (r >= m) r -= m;
  while (r < 0) r += m;
  return r;
}

__device__ __forceinline__ float dual_step(float u, float c, float w, float gl) {
  const float t = gl * w;
  return fminf(t, fmaxf(-t, u + c * (1.f / 3.f)));
}

// asynchronous 4-byte copy global -> shared
__device__ __forceinline__ void copy4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// ---- analysis of one level
enum { SARA_DUAL = 0, SARA_WEIGHTS = 1, SARA_COEFFS = 2 };  // what the finished coefficients c become
struct DwtArgs {
  const float* x;     // level 0: the image (n x n); else NULL
  const float* in;    // other levels: approximations [basis][m][m]
  float* ll;          // the next level's approximations [basis][m/2][m/2]
  float* out;         // [9][n][n]: u (SARA_DUAL), w (SARA_WEIGHTS) or c / 3 (SARA_COEFFS)
  const float* w;     // SARA_DUAL: weights
  int n, m, mode;
  bool last;          // the level's approximation is final too
  float gl, rho;
};
constexpr int DW_TO = 32;                       // coefficients of a tile per axis and band
constexpr int DW_THREADS = 320;                 // 79 columns x 4 runs of the widest first pass
constexpr int DW_SMEM = (79 * 79 + 64 * 79) * 4;

__device__ __forceinline__ void finish_coeff(const DwtArgs& A, int basis, int row, int col, float c) {
  const size_t at = ((size_t)basis * A.n + row) * A.n + col;
  if (A.mode == SARA_DUAL) A.out[at] = dual_step(A.out[at], c, A.w[at], A.gl);
  else if (A.mode == SARA_WEIGHTS) A.out[at] = A.rho / (A.rho + fabsf(c * (1.f / 3.f)));
  else A.out[at] = c * (1.f / 3.f);
}

template <int L>
__device__ __forceinline__ void dwt_tile(const DwtArgs& A, const float (&f)[2][MAXTAP], int basis, float* sm) {
  constexpr int IN = 2 * DW_TO + L - 1, RUN = 8, WIN = 2 * RUN + L - 2;  // IN is odd: rows of it are conflict-free
  const int half = A.m / 2, i0 = blockIdx.x * DW_TO, j0 = blockIdx.y * DW_TO;
  float* t = sm;            // [IN][IN] input
  float* s2 = sm + IN * IN; // [2 DW_TO][IN]: low rows, then high rows
  const float* src = A.x ? A.x : A.in + (size_t)(basis - 1) * A.m * A.m;
  const int rows = min(IN, 2 * (half - j0) + L - 2), cols = min(IN, 2 * (half - i0) + L - 2);
  const int lane = threadIdx.x % 32;
  const int c0 = wrap_any(2 * i0 + lane, A.m), c1 = wrap_any(2 * i0 + lane + 32, A.m), c2 = wrap_any(2 * i0 + lane + 64, A.m);
  for (int r = threadIdx.x / 32; r < rows; r += DW_THREADS / 32) {  // asynchronous: every row's loads are in flight
    const float* line = src + (size_t)wrap_any(2 * j0 + r, A.m) * A.m;
    float* to = t + r * IN + lane;
    if (lane < cols) copy4(to, line + c0);
    if (lane + 32 < cols) copy4(to + 32, line + c1);
    if (lane + 64 < cols) copy4(to + 64, line + c2);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int e = threadIdx.x; e < IN * (DW_TO / RUN); e += DW_THREADS) {  // axis 0: a run of 8 rows of one column
    const int c = e % IN, run = e / IN;
    if (c >= cols || 2 * RUN * run >= rows) continue;
    float v[WIN];
#pragma unroll
    for (int k = 0; k < WIN; ++k) v[k] = t[(2 * RUN * run + k) * IN + c];
#pragma unroll
    for (int j = 0; j < RUN; ++j) {
      float lo = 0.f, hi = 0.f;
#pragma unroll
      for (int k = 0; k < L; ++k) {
        lo = fmaf(f[0][k], v[2 * j + k], lo);
        hi = fmaf(f[1][k], v[2 * j + k], hi);
      }
      s2[(RUN * run + j) * IN + c] = lo;
      s2[(DW_TO + RUN * run + j) * IN + c] = hi;
    }
  }
  __syncthreads();
  constexpr int OP = DW_TO + 1;
  float* o = t;  // [4][DW_TO][OP]: bands (row low/high, column low/high)
  for (int e = threadIdx.x; e < 2 * DW_TO * (DW_TO / RUN); e += DW_THREADS) {  // axis 1: a run of 8 of one row
    const int r = e % (2 * DW_TO), run = e / (2 * DW_TO), band = r < DW_TO ? 0 : 2, j = r % DW_TO;
    float v[WIN];
#pragma unroll
    for (int k = 0; k < WIN; ++k) v[k] = s2[r * IN + 2 * RUN * run + k];
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
      float lo = 0.f, hi = 0.f;
#pragma unroll
      for (int k = 0; k < L; ++k) {
        lo = fmaf(f[0][k], v[2 * i + k], lo);
        hi = fmaf(f[1][k], v[2 * i + k], hi);
      }
      o[(band * DW_TO + j) * OP + RUN * run + i] = lo;
      o[((band + 1) * DW_TO + j) * OP + RUN * run + i] = hi;
    }
  }
  __syncthreads();
  // the coefficients of a row of a band, one per lane; the loads of a batch of rows before their stores
  constexpr int NB = 7, ROWS = 4 * DW_TO, STEP = DW_THREADS / 32;
  for (int e0 = threadIdx.x / 32; e0 < ROWS; e0 += NB * STEP) {
    float uo[NB], wo[NB];
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const int e = e0 + k * STEP, band = e / DW_TO, j = e % DW_TO;
      const bool in = e < ROWS && j0 + j < half && i0 + lane < half && !(band == 0 && !A.last);
      const size_t at = ((size_t)basis * A.n + (band >> 1) * half + j0 + j) * A.n + (band & 1) * half + i0 + lane;
      uo[k] = in && A.mode == SARA_DUAL ? A.out[at] : 0.f;
      wo[k] = in && A.mode == SARA_DUAL ? A.w[at] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const int e = e0 + k * STEP, band = e / DW_TO, j = e % DW_TO;
      if (e >= ROWS || j0 + j >= half || i0 + lane >= half) continue;
      const float c = o[e * OP + lane];
      const size_t at = ((size_t)basis * A.n + (band >> 1) * half + j0 + j) * A.n + (band & 1) * half + i0 + lane;
      if (band == 0 && !A.last) A.ll[((size_t)(basis - 1) * half + j0 + j) * half + i0 + lane] = c;
      else if (A.mode == SARA_DUAL) A.out[at] = dual_step(uo[k], c, wo[k], A.gl);
      else finish_coeff(A, basis, (band >> 1) * half + j0 + j, (band & 1) * half + i0 + lane, c);
    }
  }
}

// grid (tiles, tiles, 8, at level 0 one more for the Dirac basis); basis = 1 + blockIdx.z, the longest first
__global__ void __launch_bounds__(DW_THREADS) dwt_level(DwtArgs A, const __grid_constant__ Filters F) {
  extern __shared__ float sm[];
  switch (blockIdx.z) {
    case 0: dwt_tile<16>(A, F.f[7], 8, sm); break;
    case 1: dwt_tile<14>(A, F.f[6], 7, sm); break;
    case 2: dwt_tile<12>(A, F.f[5], 6, sm); break;
    case 3: dwt_tile<10>(A, F.f[4], 5, sm); break;
    case 4: dwt_tile<8>(A, F.f[3], 4, sm); break;
    case 5: dwt_tile<6>(A, F.f[2], 3, sm); break;
    case 6: dwt_tile<4>(A, F.f[1], 2, sm); break;
    case 7: dwt_tile<2>(A, F.f[0], 1, sm); break;
    default:  // the Dirac basis: the coefficients are the image
      for (int e = threadIdx.x; e < 4 * DW_TO * DW_TO; e += DW_THREADS) {
        const int row = 2 * DW_TO * blockIdx.y + e / (2 * DW_TO), col = 2 * DW_TO * blockIdx.x + e % (2 * DW_TO);
        if (row < A.n && col < A.n) finish_coeff(A, 0, row, col, A.x[(size_t)row * A.n + col]);
      }
  }
}

// ---- synthesis of one level
constexpr int ID_P0 = 32, ID_P1 = 64;           // output rows and columns of a tile
constexpr int ID_THREADS = 256;
constexpr int ID_COEF = 4 * 23 * 39;            // coefficients of a tile: 4 bands, 16 + L/2 - 1 rows, 32 + L/2 - 1
constexpr int ID_MID = 46 * (ID_P1 + 1);        // after axis 1: low rows, then high rows

struct IdwtArgs {
  const float* c;     // [9][n][n] coefficients
  const float* ll;    // approximations of the level [basis][m/2][m/2], NULL: they are in c (the last level)
  float* out;         // idwt_level: [basis][m][m]; idwt_primal: the n x n image
  const float* z;     // idwt_primal: x = max(0, z - Psi c) (pos) or z - Psi c; NULL: Psi c
  int n, m;
  bool pos;
};

// copies the coefficients of the tile's outputs (both axes' taps) into q, [band][C0][C1]
template <int L>
__device__ __forceinline__ void idwt_stage(const IdwtArgs& A, int basis, float* q) {
  constexpr int C0 = ID_P0 / 2 + L / 2 - 1, C1 = ID_P1 / 2 + L / 2 - 1;
  const int half = A.m / 2, jb0 = (int)blockIdx.y * (ID_P0 / 2) - L / 2 + 1, jb1 = (int)blockIdx.x * (ID_P1 / 2) - L / 2 + 1;
  const float* cb = A.c + (size_t)basis * A.n * A.n;
  const float* ll = A.ll ? A.ll + (size_t)(basis - 1) * half * half : cb;
  const int lp = A.ll ? half : A.n;
  for (int e = threadIdx.x; e < C0 * C1; e += ID_THREADS) {
    const int r = e / C1, k = e - r * C1, j = wrap_any(jb0 + r, half), i = wrap_any(jb1 + k, half);
    const float* src[4] = {ll + (size_t)j * lp + i, cb + (size_t)j * A.n + half + i, cb + (size_t)(half + j) * A.n + i,
                           cb + (size_t)(half + j) * A.n + half + i};
#pragma unroll
    for (int b = 0; b < 4; ++b) copy4(q + b * C0 * C1 + e, src[b]);
  }
}

// outputs 2 a and 2 a + 1 of one run from the low and high windows (entry q of a window is offset -q)
template <int L, int PAIRS>
__device__ __forceinline__ void synth_run(const float (&lo)[PAIRS + L / 2 - 1], const float (&hi)[PAIRS + L / 2 - 1],
                                          const float (&f)[2][MAXTAP], float (&out)[2 * PAIRS]) {
#pragma unroll
  for (int p = 0; p < 2 * PAIRS; ++p) {
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < L / 2; ++q) {
      const int k = 2 * q + (p & 1), e = p / 2 + L / 2 - 1 - q;
      acc = fmaf(f[0][k], lo[e], fmaf(f[1][k], hi[e], acc));
    }
    out[p] = acc;
  }
}

// the tile of basis (filter f) from its staged coefficients; thread (column, run of 8 rows) gets v
template <int L>
__device__ __forceinline__ void idwt_tile(const float (&f)[2][MAXTAP], const float* q, float* mid, float (&v)[8]) {
  constexpr int C0 = ID_P0 / 2 + L / 2 - 1, C1 = ID_P1 / 2 + L / 2 - 1, MP = ID_P1 + 1;
  for (int e = threadIdx.x; e < 2 * C0 * 4; e += ID_THREADS) {  // axis 1: a run of 16 outputs of one coefficient row
    const int r = e % (2 * C0), run = e / (2 * C0), band = r < C0 ? 0 : 2, rr = r < C0 ? r : r - C0;
    float lo[8 + L / 2 - 1], hi[8 + L / 2 - 1], o[16];
#pragma unroll
    for (int k = 0; k < 8 + L / 2 - 1; ++k) {
      lo[k] = q[(band * C0 + rr) * C1 + 8 * run + k];
      hi[k] = q[((band + 1) * C0 + rr) * C1 + 8 * run + k];
    }
    synth_run<L, 8>(lo, hi, f, o);
#pragma unroll
    for (int k = 0; k < 16; ++k) mid[r * MP + 16 * run + k] = o[k];
  }
  __syncthreads();
  const int col = threadIdx.x % ID_P1, run = threadIdx.x / ID_P1;  // axis 0: a run of 8 rows of one column
  float lo[4 + L / 2 - 1], hi[4 + L / 2 - 1];
#pragma unroll
  for (int k = 0; k < 4 + L / 2 - 1; ++k) {
    lo[k] = mid[(4 * run + k) * MP + col];
    hi[k] = mid[(C0 + 4 * run + k) * MP + col];
  }
  synth_run<L, 4>(lo, hi, f, v);
}

template <int L>
__device__ __forceinline__ void idwt_one(const IdwtArgs& A, const float (&f)[2][MAXTAP], int basis, float* sm) {
  idwt_stage<L>(A, basis, sm);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  float v[8];
  idwt_tile<L>(f, sm, sm + ID_COEF, v);
  const int col = blockIdx.x * ID_P1 + threadIdx.x % ID_P1, row = blockIdx.y * ID_P0 + threadIdx.x / ID_P1 * 8;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (row + k < A.m && col < A.m) A.out[((size_t)(basis - 1) * A.m + row + k) * A.m + col] = v[k];
}

// grid (tiles, tiles, 8): levels above 0
__global__ void __launch_bounds__(ID_THREADS) idwt_level(IdwtArgs A, const __grid_constant__ Filters F) {
  __shared__ float sm[ID_COEF + ID_MID];
  switch (blockIdx.z) {
    case 0: idwt_one<16>(A, F.f[7], 8, sm); break;
    case 1: idwt_one<14>(A, F.f[6], 7, sm); break;
    case 2: idwt_one<12>(A, F.f[5], 6, sm); break;
    case 3: idwt_one<10>(A, F.f[4], 5, sm); break;
    case 4: idwt_one<8>(A, F.f[3], 4, sm); break;
    case 5: idwt_one<6>(A, F.f[2], 3, sm); break;
    case 6: idwt_one<4>(A, F.f[1], 2, sm); break;
    default: idwt_one<2>(A, F.f[0], 1, sm); break;
  }
}

// basis b of idwt_primal: the next basis's coefficients are copied while this one's are transformed
template <int L>
__device__ __forceinline__ void primal_basis(const IdwtArgs& A, const float (&f)[2][MAXTAP], float* sm, float (&acc)[8]) {
  constexpr int B = L / 2;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();  // this basis's coefficients are in; the previous basis is done with the other buffer and mid
  if constexpr (L < MAXTAP) idwt_stage<L + 2>(A, B + 1, sm + (B & 1) * ID_COEF);
  float v[8];
  idwt_tile<L>(f, sm + ((B + 1) & 1) * ID_COEF, sm + 2 * ID_COEF, v);
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] += v[k] * (1.f / 3.f);
}

// level 0 of all bases and x = max(0, z - Psi u); the FP64 sums ||x - prev||^2, ||x||^2 go to acc2 (NULL: not formed)
__global__ void __launch_bounds__(ID_THREADS) idwt_primal(IdwtArgs A, const __grid_constant__ Filters F,
                                                          const float* __restrict__ prev, double* acc2) {
  __shared__ float sm[2 * ID_COEF + ID_MID];
  const int col = blockIdx.x * ID_P1 + threadIdx.x % ID_P1, row = blockIdx.y * ID_P0 + threadIdx.x / ID_P1 * 8;
  idwt_stage<2>(A, 1, sm);
  float acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    acc[k] = row + k < A.n && col < A.n ? A.c[(size_t)(row + k) * A.n + col] * (1.f / 3.f) : 0.f;  // the Dirac basis
  primal_basis<2>(A, F.f[0], sm, acc);
  primal_basis<4>(A, F.f[1], sm, acc);
  primal_basis<6>(A, F.f[2], sm, acc);
  primal_basis<8>(A, F.f[3], sm, acc);
  primal_basis<10>(A, F.f[4], sm, acc);
  primal_basis<12>(A, F.f[5], sm, acc);
  primal_basis<14>(A, F.f[6], sm, acc);
  primal_basis<16>(A, F.f[7], sm, acc);
  double s0 = 0.0, s1 = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (row + k >= A.n || col >= A.n) continue;
    const size_t at = (size_t)(row + k) * A.n + col;
    float x = acc[k];
    if (A.z) {
      x = A.z[at] - x;
      if (A.pos) x = fmaxf(0.f, x);
    }
    A.out[at] = x;
    const double d = (double)x - (prev ? prev[at] : 0.f);
    s0 += d * d;
    s1 += (double)x * x;
  }
  if (!acc2) return;
  __shared__ double red[2][ID_THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
  }
  if (threadIdx.x % 32 == 0) {
    red[0][threadIdx.x / 32] = s0;
    red[1][threadIdx.x / 32] = s1;
  }
  __syncthreads();
  if (threadIdx.x) return;
  for (int k = 1; k < ID_THREADS / 32; ++k) {
    s0 += red[0][k];
    s1 += red[1][k];
  }
  atomicAdd(&acc2[0], s0);
  atomicAdd(&acc2[1], s1);
}

__global__ void sara_fill(float* __restrict__ p, int64_t count, float v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

int grid1(int64_t count) { return (int)std::min<int64_t>((count + 255) / 256, 4096); }

// all bases' coefficients of the image x into `out` as `mode` says
int analyse(SaraState* S, cudaStream_t s, const float* x, int mode, float* out) {
  static bool attr = false;
  if (!attr) {
    PNP_CUDA(cudaFuncSetAttribute(dwt_level, cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM));
    attr = true;
  }
  for (int l = 0; l < S->levels; ++l) {
    const int m = S->n >> l, tiles = (m / 2 + DW_TO - 1) / DW_TO;
    DwtArgs A{l == 0 ? x : nullptr, l == 0 ? nullptr : S->LL[(l - 1) & 1], S->LL[l & 1], out, S->w, S->n, m, mode,
              l == S->levels - 1, (float)S->gl, (float)S->rho};
    dwt_level<<<dim3(tiles, tiles, l == 0 ? 9 : 8), DW_THREADS, DW_SMEM, s>>>(A, S->filt);
    PNP_CHECK_LAUNCH();
  }
  return PNP_OK;
}

// out = max(0, z - Psi c), z - Psi c (no positivity) or Psi c (z = NULL); FP64 norms into acc if given
int synthesise(SaraState* S, cudaStream_t s, const float* c, const float* z, float* out, bool pos, const float* prev,
               double* acc) {
  for (int l = S->levels - 1; l >= 0; --l) {
    const int m = S->n >> l;
    IdwtArgs A{c, l == S->levels - 1 ? nullptr : S->LL[l & 1], l == 0 ? out : S->LL[(l - 1) & 1], z, S->n, m, pos};
    const dim3 grid((m + ID_P1 - 1) / ID_P1, (m + ID_P0 - 1) / ID_P0, l == 0 ? 1 : SARA_FILTERS);
    if (l == 0) idwt_primal<<<grid, ID_THREADS, 0, s>>>(A, S->filt, prev, acc);
    else idwt_level<<<grid, ID_THREADS, 0, s>>>(A, S->filt);
    PNP_CHECK_LAUNCH();
  }
  return PNP_OK;
}

}  // namespace

int sara_create(pnp_den* d, int n, int levels, double gl, double rho, int iters) {
  SaraState* S = new SaraState();
  S->n = n;
  S->levels = levels;
  S->iters = iters;
  S->gl = gl;
  S->rho = rho;
  S->filt = Filters{};
  for (int N = 1; N <= SARA_FILTERS; ++N) {
    const std::vector<double> h = daub::daubechies(N);
    const int L = (int)h.size();
    if (L != 2 * N) {  // the factorisation must keep exactly N - 1 roots inside the unit circle
      d->impl = S;
      return fail(PNP_ERR_UNSUPPORTED, "internal: Daubechies factorisation failed for N = " + std::to_string(N));
    }
    for (int k = 0; k < L; ++k) {
      S->filt.f[N - 1][0][k] = (float)h[k];
      S->filt.f[N - 1][1][k] = (float)((k & 1 ? -1.0 : 1.0) * h[L - 1 - k]);
    }
  }
  const size_t N2 = (size_t)n * n;
  bool ok = cudaMalloc(&S->u, SARA_BASES * N2 * 4) == cudaSuccess &&
            cudaMalloc(&S->w, SARA_BASES * N2 * 4) == cudaSuccess &&
            cudaMalloc(&S->LL[0], SARA_FILTERS * (N2 / 4) * 4) == cudaSuccess &&
            cudaMalloc(&S->LL[1], SARA_FILTERS * std::max<size_t>(1, N2 / 16) * 4) == cudaSuccess;
  d->impl = S;
  if (!ok) {
    cudaGetLastError();
    return fail(PNP_ERR_OOM, "SARA denoiser allocation failed");
  }
  PNP_CUDA(cudaMemset(S->u, 0, SARA_BASES * N2 * 4));
  sara_fill<<<grid1((int64_t)(SARA_BASES * N2)), 256>>>(S->w, (int64_t)(SARA_BASES * N2), 1.f);  // w = 1
  PNP_CHECK_LAUNCH();
  PNP_CUDA(cudaDeviceSynchronize());
  return PNP_OK;
}

void sara_destroy(pnp_den* d) {
  SaraState* S = static_cast<SaraState*>(d->impl);
  if (!S) return;
  for (float* p : {S->u, S->w, S->LL[0], S->LL[1]}) cudaFree(p);
  delete S;
  d->impl = nullptr;
}

// the prox by S->iters dual-FB iterations from the kept u; out = x; FP64 norms into acc[0..1]
int sara_denoise(pnp_den* d, cudaStream_t s, const float* z, float* out, int n, double* acc, const float* x_prev,
                 bool positivity) {
  SaraState* S = static_cast<SaraState*>(d->impl);
  if (!S || n != S->n) return fail(PNP_ERR_INVALID_ARG, "image side differs from the SARA denoiser's");
  for (int it = 0; it <= S->iters; ++it) {  // x from the kept u, then u and x in turn
    if (it > 0)
      if (int rc = analyse(S, s, out, SARA_DUAL, S->u)) return rc;
    const bool end = it == S->iters;
    if (int rc = synthesise(S, s, S->u, z, out, positivity, end ? x_prev : nullptr, end ? acc : nullptr)) return rc;
  }
  return PNP_OK;
}

int sara_reweight(pnp_den* d, const float* x) {
  SaraState* S = static_cast<SaraState*>(d->impl);
  return analyse(S, d->stream, x, SARA_WEIGHTS, S->w);
}

// direction 1: out (9 n^2) = Psi^T in;  direction -1: out (n^2) = Psi in
int sara_transform(pnp_den* d, const float* in, float* out, int direction) {
  SaraState* S = static_cast<SaraState*>(d->impl);
  if (direction > 0) return analyse(S, d->stream, in, SARA_COEFFS, out);
  return synthesise(S, d->stream, in, nullptr, out, false, nullptr, nullptr);
}

}  // namespace pnp
