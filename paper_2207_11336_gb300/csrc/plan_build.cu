// Construction of the measurement operator Phi = G F Z (Eq. 1; App. E).
//
// Host side (once per plan, O(M)): KB shape parameter and grid-correction
// table, FFT twiddles, per-row tap windows, a stable counting sort of the rows
// by (grid tile of the first tap, data block), CSR row offsets and the work
// units of the gridding kernels.
//
// Device side: one warp per row evaluates the row's separable weights
//   g(t) = sum_d w_hat[d] psi(t + d),  psi(t) = I0(beta sqrt(1 - (2t/J)^2)),
// on the J_m taps nearest kappa along each axis, and writes the two factors (complex64
// plans) or their J_m^2 outer products (BF16 plans).  w_hat is the K-point DFT of the
// paraxial w-chirp exp(i pi a q(p)), a = w dl^2, whose phase profile q equals
// p^2 on the image and is continued smoothly (C^2) to a flat value at |p| = K/2
// (App. E reading: the w-kernel of each row folded into its KB row).  It is
// evaluated from its Taylor series in b = pi a (n/2)^2 about the mid value of
// the normalised profile, using moments mu_j[d] = K^-1 sum_p (qn(p) - c0)^j
// cos(2 pi d p / K) precomputed here in FP64.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>

#include "common.cuh"

namespace pnp {
namespace {

constexpr int MAX_TERMS = 64;
constexpr int MAX_D = 15;  // |d| <= MAX_D, so 2 MAX_D + 1 <= 32 lanes

struct RowGeom : RowKey {
  int64_t unit;          // offset of the stored row, 16-byte units (export: of the row's taps)
  int s0, s1;            // first tap (unwrapped) per axis
  int J;                 // row support J_m
  int cell;              // first tap's cell in its coarse tile, row << 5 | column
};

struct BuildArgs {
  int64_t M;
  int J;
  double beta, bscale, c0;   // b = bscale * a ; series centre c0
  int nterms, D;
  const double* mu;          // [nterms][2D+1]
  const RowGeom* geom;       // sorted order
  unsigned char* rows;       // stored rows (zero: the padding stays)
  int bf16;
  float2* taps;              // export: the J x J taps (k1-major) in the place of the stored rows, and their columns
  int32_t* cols;
  int logK;
};

__device__ __forceinline__ double kb_psi(double t, int J, double beta) {
  const double z = 1.0 - (2.0 * t / J) * (2.0 * t / J);
  return z >= 0.0 ? cyl_bessel_i0(beta * sqrt(z)) : 0.0;
}

// one warp per row
__global__ void __launch_bounds__(256) build_rows(BuildArgs A) {
  __shared__ double2 s_wh[8][2 * MAX_D + 1];
  __shared__ double s_psi[8][2][32];
  __shared__ double2 s_g[8][2][16];
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const int64_t row = (int64_t)blockIdx.x * 8 + wl;
  if (row >= A.M) return;
  const RowGeom g = A.geom[row];
  const int Jm = g.J, D = A.D;
  const bool has_w = g.a != 0.0;
  // w-kernel values w_hat[d], d = -D..D
  if (has_w && lane <= 2 * D) {
    const double b = A.bscale * g.a;
    // sum_j (i b)^j / j! mu_j[d]
    double tr = 1.0, ti = 0.0, sr = 0.0, si = 0.0;
    for (int j = 0; j < A.nterms; ++j) {
      const double m = A.mu[j * (2 * D + 1) + lane];
      sr += tr * m;
      si += ti * m;
      const double nr = -ti * b / (j + 1), ni = tr * b / (j + 1);
      tr = nr;
      ti = ni;
    }
    double sn, cs;
    sincos(b * A.c0, &sn, &cs);
    s_wh[wl][lane] = make_double2(sr * cs - si * sn, sr * sn + si * cs);
  }
  // psi(t0 + e) for the integers e with |t0 + e| <= J/2, per axis
  const int ax = lane >> 4, sl = lane & 15;
  const double kap = ax ? g.kap1 : g.kap0;
  const int st = ax ? g.s1 : g.s0;
  const double t0 = kap - st;
  const int emin = (int)ceil(-t0 - 0.5 * A.J);
  s_psi[wl][ax][sl] = kb_psi(t0 + emin + sl, A.J, A.beta);
  __syncwarp();
  if (sl < Jm) {
    double gr = 0.0, gi = 0.0;
    if (has_w) {
      for (int i = 0; i <= A.J; ++i) {
        const double ps = s_psi[wl][ax][i];
        const int d = emin + i + sl;
        if (ps != 0.0 && d >= -D && d <= D) {
          const double2 w = s_wh[wl][d + D];
          gr += w.x * ps;
          gi += w.y * ps;
        }
      }
    } else {
      gr = kb_psi(t0 - sl, A.J, A.beta);
    }
    s_g[wl][ax][sl] = make_double2(gr, gi);
  }
  __syncwarp();
  if (A.taps) {
    const int Km = (1 << A.logK) - 1;
    for (int t = lane; t < Jm * Jm; t += 32) {
      const int i1 = t / Jm, i0 = t - i1 * Jm;
      const double2 a = s_g[wl][0][i0], b = s_g[wl][1][i1];
      float2 w = make_float2((float)(g.d * (a.x * b.x - a.y * b.y)), (float)(g.d * (a.x * b.y + a.y * b.x)));
      if (A.bf16) w = __bfloat1622float2(__floats2bfloat162_rn(w.x, w.y));
      A.taps[g.unit + t] = w;
      A.cols[g.unit + t] = (((g.s0 + i0) & Km) << A.logK) | ((g.s1 + i1) & Km);
    }
    return;
  }
  const int jp = tap_pairs(Jm);
  float* out = reinterpret_cast<float*>(A.rows + (g.unit << 4));
  if (!A.bf16) {
    // the k1 factors, scaled by the data weight, as (re, re, im, im) per tap pair; then the k0 factors
    if (sl < Jm) {
      const double2 v = s_g[wl][ax][sl];
      if (ax) {
        const int i1 = sl + ((g.cell >> 5) & 1);
        float* o = out + 4 * (i1 >> 1) + (i1 & 1);
        o[0] = (float)(g.d * v.x);
        o[2] = (float)(g.d * v.y);
      } else {
        out[4 * jp + 2 * sl] = (float)v.x;
        out[4 * jp + 2 * sl + 1] = (float)v.y;
      }
    }
    if (lane == 0) reinterpret_cast<int*>(out)[row_cell_at(jp, false) / 4] = g.cell;
    return;
  }
  if (lane == 0) reinterpret_cast<int*>(out)[row_cell_at(jp, true) / 4] = g.cell;
  __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(out);
  for (int t = lane; t < Jm * Jm; t += 32) {
    const int i1 = t / Jm, i0 = t - i1 * Jm;
    const double2 a = s_g[wl][0][i0], b = s_g[wl][1][i1];
    const float wr = (float)(g.d * (a.x * b.x - a.y * b.y)), wi = (float)(g.d * (a.x * b.y + a.y * b.x));
    const int e1 = i1 + ((g.cell >> 5) & 1);
    __nv_bfloat16* o = ob + ((e1 >> 1) * 2 * jp + i0) * 4 + (e1 & 1);
    o[0] = __float2bfloat16_rn(wr);
    o[2] = __float2bfloat16_rn(wi);
  }
}

double kb_beta(int J, double sigma) {
  return M_PI * std::sqrt((J / sigma) * (J / sigma) * (sigma - 0.5) * (sigma - 0.5) - 0.8);
}

double kb_correction(double p, int J, double beta, int K) {
  const double s = M_PI * J * p / K, r2 = beta * beta - s * s;
  if (r2 > 0) {
    const double r = std::sqrt(r2);
    return J * std::sinh(r) / r;
  }
  if (r2 < 0) {
    const double r = std::sqrt(-r2);
    return J * std::sin(r) / r;
  }
  return J;
}

// normalised frozen-chirp phase profile qn(p) = q(p) / (n/2)^2
double chirp_q(double p, int n, int K) {
  const double a = std::fabs(p), h = n / 2.0;
  if (a <= h) return a * a / (h * h);
  const double u = (a - h) / (K / 2.0 - h);
  const double q = h * h + n * (K / 2.0 - h) * (u + u * u / 2.0 - u * u * u * u + 2.0 * std::pow(u, 5) / 5.0);
  return q / (h * h);
}

template <typename T>
int dev_alloc(pnp_plan* p, T** ptr, size_t count) {
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(ptr), count * sizeof(T));
  if (e != cudaSuccess) {
    *ptr = nullptr;
    cudaGetLastError();
    return fail(PNP_ERR_OOM, "cudaMalloc of " + std::to_string(count * sizeof(T)) + " bytes failed");
  }
  p->device_bytes += (int64_t)(count * sizeof(T));
  return PNP_OK;
}

BuildArgs build_args(const pnp_plan* p, int64_t nrows, const RowGeom* d_geom) {
  BuildArgs A{};
  A.M = nrows;
  A.J = p->J;
  A.beta = p->beta;
  A.bscale = p->bscale;
  A.c0 = p->series_c0;
  A.nterms = p->nterms;
  A.D = p->series_D;
  A.mu = p->d_mu;
  A.geom = d_geom;
  A.bf16 = p->wdtype == PNP_W_BF16C;
  A.logK = p->logK;
  return A;
}

// first tap per axis of a row of support J
int first_tap(double kap, int J) { return (int)std::floor(kap - 0.5 * J) + 1; }

// Tile side and kind of the work units, before the rows are sorted for them.  Where the units of the classes are thin
// (few rows of one support in a GT x GT tile), staging and flushing their regions costs more than their rows; larger
// tiles whose regions all supports share then do better: the cells that the flushes add, a row, fall about threefold.
// Fused pass, classes -> mixed: 4096^2 grid, uniform coverage, J 7-16: 3e5 rows (1.2 a unit, 5.7 units a 16 x 16 tile)
// 455 -> 342 us, 1e6 rows (1.9, 12) 899 -> 604 us, 4e6 rows (6.0, 16) 1583 -> 1655 us; a track of 1e5 rows (2.1, 3.9) 108 ->
// 135 us; 1024^2 grid, 3e4 rows in 2700 tiles (1.4, 7.9) 47 -> 51 us: fewer than two tiles per resident warp (12 an SM).
// key: (coarse tile, block); startc: tile within the coarse tile << 6 | cell; supports: bit J for each J of the plan.
void pick_tile(pnp_plan* p, const std::vector<RowGeom>& geom, const std::vector<int32_t>& key,
               const std::vector<uint16_t>& startc, const int32_t* stack, unsigned supports) {
  constexpr int SUBS = (GKT / GT) * (GKT / GT);
  const int64_t coarse = p->nkeys * p->nstacks;
  // too many rows for thin units, or a mask of more than half a gigabyte
  if (p->M >= 3 * coarse * SUBS * __builtin_popcount(supports) || coarse * SUBS > (int64_t(1) << 28)) return;
  std::vector<uint16_t> mask(coarse * SUBS, 0);  // per GT x GT tile, block and stack: its supports (bit J - 2)
  for (int64_t m = 0; m < p->M; ++m)
    mask[((stack ? (int64_t)stack[m] * p->nkeys : 0) + key[m]) * SUBS + (startc[m] >> 6)] |= (uint16_t)(1u << (geom[m].J - 2));
  int64_t units = 0, tiles = 0;
  for (int64_t k = 0; k < coarse; ++k) {
    unsigned seen = 0;  // its MIX_TILE x MIX_TILE tiles with rows
    for (int sub = 0; sub < SUBS; ++sub) {
      const unsigned u = mask[k * SUBS + sub];
      units += __builtin_popcount(u);
      if (u) seen |= 1u << (sub / (GKT / GT) * GT / MIX_TILE * (GKT / MIX_TILE) + sub % (GKT / GT) * GT / MIX_TILE);
    }
    tiles += __builtin_popcount(seen);
  }
  p->mixed = p->M < 3 * units && units >= 5 * tiles && tiles >= (int64_t)24 * p->num_sms * p->nstacks;
  p->tile = p->mixed ? MIX_TILE : GT;
}

}  // namespace

int build_units(pnp_plan* p) {
  ++p->epoch;  // a captured FB graph launches the old work list: it must be captured again
  std::vector<Unit> units, cls[TAP_CLASSES];
  const int64_t M = p->M;
  std::vector<int64_t> bounds(1, 0);
  // Taps per unit of each class of supports: an eighth of the unit_nnz setting (a unit is one warp's work),
  // less where the class is small, so that every resident warp (16 to 24 per SM) gets several units, but
  // enough rows to pay for staging and flushing the unit's region.
  int64_t cap[TAP_CLASSES] = {};
  for (int64_t r = 0; r < M; ++r)
    cap[p->mixed ? 0 : tap_class(tap_pairs(p->h_J[r]), tap_lanes(p->h_J[r]))] += p->h_J[r] * p->h_J[r];
  for (int64_t& c : cap)
    c = std::min<int64_t>(p->unit_nnz, std::max<int64_t>(2048, std::min<int64_t>(p->unit_nnz / 8, c / (p->num_sms * 100))));
  const int cpt = p->K / GKT, per = GKT / p->tile;  // coarse tiles per side, tiles per coarse tile side
  int of_sub[(GKT / GT) * (GKT / GT)];              // a row's tile within its coarse tile: row * per + column
  for (int sub = 0; sub < (GKT / GT) * (GKT / GT); ++sub)
    of_sub[sub] = sub / (GKT / GT) * GT / p->tile * per + sub % (GKT / GT) * GT / p->tile;
  auto tile_of = [&](int64_t r) { return of_sub[p->h_start[r] >> 6]; };
  int64_t i = 0;
  for (int st = 0; st < p->nstacks; ++st) {
    int32_t last_key = -1;
    int last_t = -1;
    int64_t held = 0;  // mixed: taps of the tile's units since the last `first`
    while (i < M && p->h_key[i] / p->nkeys == st) {
      const int32_t key = p->h_key[i];
      const int t = tile_of(i), J = p->h_J[i], ct = (int)((key % p->nkeys) / p->nblocks);
      Unit u{};
      u.row_begin = i;
      u.row_unit = p->h_unit[i];
      u.J = J;
      u.tile = ((ct / cpt) * per + t / per) * p->ntc + (ct % cpt) * per + t % per;
      const int c = p->mixed ? 0 : tap_class(tap_pairs(J), tap_lanes(J));
      int64_t taps = 0;
      while (i < M && p->h_key[i] == key && tile_of(i) == t && p->h_J[i] == J &&
             (taps == 0 || taps + (int64_t)J * J <= cap[c])) {
        taps += (int64_t)J * J;
        ++u.nrows;
        ++i;
      }
      held += taps;
      u.first = !p->mixed || key != last_key || t != last_t || held > cap[c];
      if (u.first) held = taps;
      last_key = key;
      last_t = t;
      cls[c].push_back(u);
    }
    for (auto& v : cls) {
      units.insert(units.end(), v.begin(), v.end());
      bounds.push_back((int64_t)units.size());
      v.clear();
    }
  }
  if (i != M) return fail(PNP_ERR_INVALID_ARG, "internal: rows out of stack order");
  if (p->d_units) {
    cudaFree(p->d_units);
    p->device_bytes -= std::max<int64_t>(1, p->n_units) * (int64_t)sizeof(Unit);
    p->d_units = nullptr;
  }
  p->n_units = (int64_t)units.size();
  p->h_class_units.swap(bounds);
  if (int rc = dev_alloc(p, &p->d_units, units.size())) return rc;
  if (!units.empty())
    PNP_CUDA(cudaMemcpy(p->d_units, units.data(), units.size() * sizeof(Unit), cudaMemcpyHostToDevice));
  return PNP_OK;
}

int plan_build(pnp_plan* p, const double* uvw, const int8_t* Jrow, const int32_t* block, const int32_t* stack,
               const double* row_scale) {
  const int n = p->n, K = p->K, J = p->J;
  const int64_t M = p->M;
  p->beta = kb_beta(J, (double)K / n);

  // grid correction and twiddles
  std::vector<float2> cinv(n);
  for (int a = 0; a < n; ++a) {
    const double c = 1.0 / kb_correction(a - n / 2, J, p->beta, K);
    cinv[a] = make_float2((float)c, (float)(c - (double)(float)c));
  }
  std::vector<float2> tw(K);
  for (int j = 0; j < K; ++j) {
    const double ang = -2.0 * M_PI * j / K;
    tw[j] = make_float2((float)std::cos(ang), (float)std::sin(ang));
  }

  // per-row geometry, keys
  const int cpt = K / GKT;  // coarse tiles per grid side
  std::vector<RowGeom> geom(M);
  p->h_rowkey.reserve(M);
  unsigned supports = 0;
  std::vector<int32_t> key(M);
  std::vector<uint16_t> startc(M);  // tile within the coarse tile << 6 | first tap's cell within the tile
  int Jmax = J;
  double amax = 0.0;
  for (int64_t m = 0; m < M; ++m) {
    RowGeom g;
    g.kap0 = uvw[3 * m] * (K / (2.0 * M_PI));
    g.kap1 = uvw[3 * m + 1] * (K / (2.0 * M_PI));
    if (stack && (stack[m] < 0 || stack[m] >= p->nstacks))
      return fail(PNP_ERR_INVALID_ARG, "stack id out of range at row " + std::to_string(m));
    // w-stacking (App. E): the row kernel carries only the offset from its stack's centre
    const double wres = uvw[3 * m + 2] - (stack ? p->w_centres[stack[m]] : 0.0);
    g.a = p->dl > 0 ? wres * p->dl * p->dl : 0.0;
    g.J = Jrow ? Jrow[m] : J;
    g.d = row_scale ? row_scale[m] : 1.0;
    if (!(g.d > 0.0) || !std::isfinite(g.d))
      return fail(PNP_ERR_INVALID_ARG, "row scale must be finite and > 0 at row " + std::to_string(m));
    if (!(std::isfinite(g.kap0) && std::isfinite(g.kap1) && std::isfinite(g.a)))
      return fail(PNP_ERR_INVALID_ARG, "non-finite uvw at row " + std::to_string(m));
    if (std::fabs(uvw[3 * m]) > 4 * M_PI || std::fabs(uvw[3 * m + 1]) > 4 * M_PI)
      return fail(PNP_ERR_INVALID_ARG, "omega outside [-4 pi, 4 pi] at row " + std::to_string(m));
    if (g.J < J || g.J > 16)
      return fail(PNP_ERR_INVALID_ARG, "J_per_row must lie in [J, 16]; row " + std::to_string(m));
    if (block && (block[m] < 0 || block[m] >= p->nblocks))
      return fail(PNP_ERR_INVALID_ARG, "block id out of range at row " + std::to_string(m));
    g.s0 = first_tap(g.kap0, g.J);
    g.s1 = first_tap(g.kap1, g.J);
    const int f0 = ((g.s0 % K) + K) % K, f1 = ((g.s1 % K) + K) % K;
    key[m] = ((f1 / GKT) * cpt + (f0 / GKT)) * p->nblocks + (block ? block[m] : 0);
    const int sub = (f1 % GKT) / GT * (GKT / GT) + (f0 % GKT) / GT;
    startc[m] = (uint16_t)((sub << 6) | ((f1 % GT) << 3) | (f0 % GT));
    Jmax = std::max(Jmax, g.J);
    amax = std::max(amax, std::fabs(g.a));
    supports |= 1u << g.J;
    geom[m] = g;
    p->h_rowkey.push_back(g);
  }
  p->Jmax = Jmax;

  const int64_t nkeys = (int64_t)cpt * cpt * p->nblocks;
  if (nkeys * p->nstacks > INT32_MAX) return fail(PNP_ERR_UNSUPPORTED, "too many (stack, tile, block) keys");
  p->nkeys = nkeys;
  pick_tile(p, geom, key, startc, p->nstacks > 1 ? stack : nullptr, supports);
  // stable LSD counting sort: by (T x T tile within the coarse tile, support J, first tap's cell in the tile with the
  // cells of one gridding window together), then by (coarse tile, block) key and w-stack, so that the rows of one
  // tile come out grouped by J and, within that, rows sharing a window are adjacent (the gridding pass
  // keeps it in registers)
  {
    const int T = p->tile, per = GKT / T;
    std::vector<int32_t> by_j(M);
    {
      auto bin = [&](int64_t m) {
        const int J = geom[m].J, q = T == GT ? tap_quant(tap_pairs(J), tap_lanes(J)) : 1;
        const int sub = startc[m] >> 6, cell = startc[m] & 63;
        const int r = sub / (GKT / GT) * GT + (cell >> 3), c = sub % (GKT / GT) * GT + (cell & 7);  // in the coarse tile
        const int lr = r % T, lc = c % T;
        return ((r / T * per + c / T) * 17 + J) * T * T + (((lr >> 1) * (T / q) + lc / q) * 2 + (lr & 1)) * q + lc % q;
      };
      std::vector<int64_t> cc((size_t)17 * GKT * GKT + 1, 0);
      for (int64_t m = 0; m < M; ++m) cc[bin(m) + 1]++;
      for (size_t c = 1; c < cc.size(); ++c) cc[c] += cc[c - 1];
      for (int64_t m = 0; m < M; ++m) by_j[cc[bin(m)]++] = (int32_t)m;
    }
    std::vector<int64_t> cnt(nkeys + 1, 0);
    for (int64_t m = 0; m < M; ++m) cnt[key[m] + 1]++;
    for (int64_t k = 0; k < nkeys; ++k) cnt[k + 1] += cnt[k];
    p->h_perm.assign(M, 0);
    for (int64_t i = 0; i < M; ++i) {
      const int32_t m = by_j[i];
      p->h_perm[cnt[key[m]]++] = m;
    }
    if (stack && p->nstacks > 1) {  // most significant: the w-stack
      std::vector<int64_t> cs(p->nstacks + 1, 0);
      for (int64_t m = 0; m < M; ++m) cs[stack[m] + 1]++;
      for (int s = 0; s < p->nstacks; ++s) cs[s + 1] += cs[s];
      for (int64_t i = 0; i < M; ++i) {
        const int32_t m = p->h_perm[i];
        by_j[cs[stack[m]]++] = m;
      }
      p->h_perm.swap(by_j);
    }
  }
  p->ntc = K / p->tile;
  p->pitch = p->mixed ? p->tile - 1 + 16 : GT - tap_quant(tap_pairs(Jmax), tap_lanes(Jmax)) + tap_lanes(Jmax);
  p->h_inv.assign(M, 0);
  for (int64_t i = 0; i < M; ++i) p->h_inv[p->h_perm[i]] = (int32_t)i;
  std::vector<RowGeom> sgeom(M);
  p->h_key.assign(M, 0);
  p->h_start.assign(M, 0);
  p->h_unit.assign(M + 1, 0);
  p->h_J.assign(M, 0);
  p->nnz = 0;
  for (int64_t i = 0; i < M; ++i) {
    const int64_t m = p->h_perm[i];
    sgeom[i] = geom[m];
    p->h_key[i] = (int32_t)((stack ? (int64_t)stack[m] : 0) * nkeys + key[m]);
    p->h_start[i] = startc[m];
    p->h_J[i] = (uint8_t)geom[m].J;
    sgeom[i].unit = p->h_unit[i];
    const int sub = startc[m] >> 6, cell = startc[m] & 63;
    sgeom[i].cell = (sub / (GKT / GT) * GT + (cell >> 3)) << 5 | (sub % (GKT / GT) * GT + (cell & 7));
    p->h_unit[i + 1] = p->h_unit[i] + row_units(geom[m].J, p->wdtype == PNP_W_BF16C);
    p->nnz += (int64_t)geom[m].J * geom[m].J;
  }
  // uv support of G: per grid row k1 the largest centred |k0| of its taps, and the band of rows
  std::vector<int> rowh(K, -1);
  {
    auto centred = [K](int k) {
      k = ((k % K) + K) % K;
      return k < K / 2 ? k : k - K;
    };
    for (int64_t m = 0; m < M; ++m) {
      const RowGeom& g = geom[m];
      const int c0 = centred(g.s0), c0e = c0 + g.J - 1;  // the row's k0 taps, centred (may wrap)
      const int hm = c0e >= K / 2 ? K / 2 : std::max(std::abs(c0), std::abs(c0e));
      for (int t = 0; t < g.J; ++t) {
        int& h = rowh[((g.s1 + t) % K + K) % K];
        h = std::max(h, hm);
      }
    }
    p->band = -1;
    for (int k = 0; k < K; ++k)
      if (rowh[k] >= 0) p->band = std::max(p->band, std::abs(centred(k)));
    int64_t cells = 0;  // of a grid that the FFT passes read and write: the uv support, all of it unless n = K/2
    for (int k = 0; k < K; ++k) cells += n == K / 2 ? std::clamp(2 * rowh[k] + 1, 0, K) : K;
    int l2 = 0;
    PNP_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, p->device));
    // Adjoint gridding of uniform and track coverage without and with the lines fetched ahead: 16 MB of support 75 and
    // 55 us (1e6 track rows, J = 7: 92 and 70 us), 41 MB 232 and 89 us; 5 MB 32.4 and 32.8 us.
    p->support_in_l2 = cells * (int64_t)sizeof(float2) <= l2 / 16;
  }
  std::vector<RowGeom>().swap(geom);

  // w-kernel series: b = bscale * a, qn in [0, qmax], centred at c0 = qmax / 2
  const double h = n / 2.0;
  const double bscale = M_PI * h * h;
  const double qmax = chirp_q(K / 2.0, n, K), c0 = qmax / 2.0;
  const int D = (Jmax + J + 1) / 2 + 1;
  if (D > MAX_D) return fail(PNP_ERR_UNSUPPORTED, "kernel support too large");
  int nterms = 1;
  {
    const double x = bscale * amax * c0;  // largest |b (qn - c0)|
    double term = 1.0;
    while (nterms < MAX_TERMS) {
      term *= x / nterms;
      ++nterms;
      if (term < 1e-18 && nterms > x) break;
    }
    if (nterms >= MAX_TERMS && x > 0)
      return fail(PNP_ERR_UNSUPPORTED, "w-term too large for the w-kernel series (increase K or reduce dl)");
    if (amax == 0.0) nterms = 1;
  }
  std::vector<double> mu((size_t)nterms * (2 * D + 1), 0.0);
  if (amax > 0.0) {
    std::vector<double> qc(K);
    for (int j = 0; j < K; ++j) qc[j] = chirp_q(j - K / 2, n, K) - c0;
    for (int d = -D; d <= D; ++d) {
      std::vector<double> pw(K, 1.0);
      std::vector<double> cs(K);
      for (int j = 0; j < K; ++j) cs[j] = std::cos(2.0 * M_PI * d * (double)(j - K / 2) / K);
      for (int t = 0; t < nterms; ++t) {
        double s = 0.0;
        for (int j = 0; j < K; ++j) {
          s += pw[j] * cs[j];
          pw[j] *= qc[j];
        }
        mu[(size_t)t * (2 * D + 1) + (d + D)] = s / K;
      }
    }
  }

  // device buffers
  const size_t KK = (size_t)K * K;
  if (int rc = dev_alloc(p, &p->d_cinv, n)) return rc;
  if (int rc = dev_alloc(p, &p->d_tw, K)) return rc;
  if (int rc = dev_alloc(p, &p->d_twp, TWP_ENTRIES)) return rc;
  if (int rc = dev_alloc(p, &p->d_gridA, KK)) return rc;
  if (int rc = dev_alloc(p, &p->d_gridB, KK)) return rc;
  if (int rc = dev_alloc(p, &p->d_gridB_lo, KK)) return rc;
  if (int rc = dev_alloc(p, &p->d_tmp, (size_t)K * n)) return rc;
  if (int rc = dev_alloc(p, &p->d_rowh, (size_t)K)) return rc;
  {
    const size_t bytes = (size_t)std::max<int64_t>(1, p->h_unit[M]) * 16;
    cudaError_t e = cudaMalloc(&p->d_rows, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      p->d_rows = nullptr;
      return fail(PNP_ERR_OOM, "cudaMalloc of the rows of G (" + std::to_string(bytes) + " bytes) failed");
    }
    p->device_bytes += (int64_t)bytes;
    PNP_CUDA(cudaMemset(p->d_rows, 0, bytes));  // the padding taps
  }
  if (int rc = dev_alloc(p, &p->d_perm, (size_t)M)) return rc;
  if (int rc = dev_alloc(p, &p->d_sched, (size_t)2 * p->nstacks * TAP_CLASSES)) return rc;
  PNP_CUDA(cudaMemset(p->d_sched, 0, (size_t)2 * p->nstacks * TAP_CLASSES * sizeof(unsigned)));
  if (int rc = dev_alloc(p, &p->d_ysorted, (size_t)M)) return rc;
  PNP_CUDA(cudaMemset(p->d_ysorted, 0, (size_t)M * sizeof(float2)));
  if (int rc = dev_alloc(p, &p->d_acc, 8)) return rc;
  if (int rc = dev_alloc(p, &p->d_status, 4)) return rc;
  for (int i = 0; i < 3; ++i)
    if (int rc = dev_alloc(p, &p->d_img[i], (size_t)n * n)) return rc;
  if (p->nstacks > 1) {
    // Z_s of stack s: the paraxial w-modulation of the stack centre, separable per axis
    std::vector<float2> ch((size_t)p->nstacks * n);
    for (int s = 0; s < p->nstacks; ++s) {
      const double as = p->w_centres[s] * p->dl * p->dl;
      for (int a = 0; a < n; ++a) {
        const double q = (double)(a - n / 2), ph = M_PI * as * q * q;
        ch[(size_t)s * n + a] = make_float2((float)std::cos(ph), (float)std::sin(ph));
      }
    }
    if (int rc = dev_alloc(p, &p->d_chirp, ch.size())) return rc;
    if (int rc = dev_alloc(p, &p->d_gacc, (size_t)n * n)) return rc;
    PNP_CUDA(cudaMemcpy(p->d_chirp, ch.data(), ch.size() * sizeof(float2), cudaMemcpyHostToDevice));
  }
  PNP_CUDA(cudaMemcpy(p->d_cinv, cinv.data(), n * sizeof(float2), cudaMemcpyHostToDevice));
  PNP_CUDA(cudaMemcpy(p->d_tw, tw.data(), K * sizeof(float2), cudaMemcpyHostToDevice));
  {
    std::vector<float2> twp(TWP_ENTRIES);
    for (int q = 1, off = 0; q <= 2; off += 16 * (1 << (4 * q)), ++q) {
      const int Ns = 1 << (4 * q);
      for (int r = 0; r < 16; ++r)
        for (int k = 0; k < Ns; ++k) {
          const double ang = -2.0 * M_PI * (double)(r * k) / (16.0 * Ns);
          twp[off + r * Ns + k] = make_float2((float)std::cos(ang), (float)std::sin(ang));
        }
    }
    PNP_CUDA(cudaMemcpy(p->d_twp, twp.data(), TWP_ENTRIES * sizeof(float2), cudaMemcpyHostToDevice));
  }
  // the forward grid outside G's support is never written (the split passes prune it) and reads as 0
  PNP_CUDA(cudaMemset(p->d_gridA, 0, KK * sizeof(float2)));
  PNP_CUDA(cudaMemset(p->d_gridB, 0, KK * sizeof(float2)));
  PNP_CUDA(cudaMemset(p->d_gridB_lo, 0, KK * sizeof(__nv_bfloat162)));
  PNP_CUDA(cudaMemcpy(p->d_rowh, rowh.data(), K * sizeof(int), cudaMemcpyHostToDevice));
  PNP_CUDA(cudaMemset(p->d_acc, 0, 8 * sizeof(double)));
  PNP_CUDA(cudaMemset(p->d_status, 0, 4 * sizeof(int)));
  if (M) PNP_CUDA(cudaMemcpy(p->d_perm, p->h_perm.data(), M * sizeof(int32_t), cudaMemcpyHostToDevice));
  if (M && row_scale) {  // the data weights in the caller's row order, for pnp_plan_scale_data
    std::vector<float> d(M);
    for (int64_t m = 0; m < M; ++m) d[m] = (float)row_scale[m];
    if (int rc = dev_alloc(p, &p->d_rowscale, (size_t)M)) return rc;
    PNP_CUDA(cudaMemcpy(p->d_rowscale, d.data(), M * sizeof(float), cudaMemcpyHostToDevice));
  }

  // build G rows on the GPU
  if (M) {
    RowGeom* d_geom = nullptr;
    if (int rc = dev_alloc(p, &p->d_mu, mu.size())) return rc;
    if (cudaMalloc(&d_geom, M * sizeof(RowGeom)) != cudaSuccess) {
      cudaGetLastError();
      return fail(PNP_ERR_OOM, "plan build scratch allocation failed");
    }
    PNP_CUDA(cudaMemcpy(d_geom, sgeom.data(), M * sizeof(RowGeom), cudaMemcpyHostToDevice));
    PNP_CUDA(cudaMemcpy(p->d_mu, mu.data(), mu.size() * sizeof(double), cudaMemcpyHostToDevice));
    p->nterms = nterms;
    p->series_D = D;
    p->bscale = bscale;
    p->series_c0 = c0;
    BuildArgs A = build_args(p, M, d_geom);
    A.rows = static_cast<unsigned char*>(p->d_rows);
    build_rows<<<(unsigned)((M + 7) / 8), 256, 0, p->stream>>>(A);
    cudaError_t e = cudaGetLastError();
    g_launches.fetch_add(1);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    cudaFree(d_geom);
    if (e != cudaSuccess) return fail(PNP_ERR_CUDA, std::string("build_rows: ") + cudaGetErrorString(e));
  }
  return build_units(p);
}

int export_rows_impl(const pnp_plan* p, const int64_t* rows, int64_t nrows, int64_t* offsets,
                     float* weights, int32_t* cols) {
  // evaluated anew in FP64: a stored complex64 row holds two rounded factors, whose products carry 1.8 times the error
  // (1e4 rows: 0.96 -> 1.55 ms against reading the stored rows)
  std::vector<RowGeom> geom(weights && cols ? nrows : 0);
  offsets[0] = 0;
  for (int64_t i = 0; i < nrows; ++i) {
    if (rows[i] < 0 || rows[i] >= p->M) return fail(PNP_ERR_INVALID_ARG, "export row index out of range");
    RowGeom g{};
    static_cast<RowKey&>(g) = p->h_rowkey[rows[i]];
    g.J = p->h_J[p->h_inv[rows[i]]];
    g.s0 = first_tap(g.kap0, g.J);
    g.s1 = first_tap(g.kap1, g.J);
    g.unit = offsets[i];
    if (!geom.empty()) geom[i] = g;
    offsets[i + 1] = offsets[i] + (int64_t)g.J * g.J;
  }
  if (!weights || !cols || nrows == 0) return PNP_OK;
  const int64_t total = offsets[nrows];
  RowGeom* d_geom = nullptr;
  float2* d_w = nullptr;
  int32_t* d_c = nullptr;
  int rc = PNP_OK;
  if (cudaMalloc(&d_geom, nrows * sizeof(RowGeom)) || cudaMalloc(&d_w, total * sizeof(float2)) ||
      cudaMalloc(&d_c, total * sizeof(int32_t))) {
    cudaGetLastError();
    rc = fail(PNP_ERR_OOM, "export scratch allocation failed");
  }
  if (!rc) {
    cudaError_t e = cudaMemcpy(d_geom, geom.data(), nrows * sizeof(RowGeom), cudaMemcpyHostToDevice);
    // a small copy may still be on its way, and p->stream need not wait for it
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e == cudaSuccess) {
      BuildArgs A = build_args(p, nrows, d_geom);
      A.taps = d_w;
      A.cols = d_c;
      build_rows<<<(unsigned)((nrows + 7) / 8), 256, 0, p->stream>>>(A);
      g_launches.fetch_add(1);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
    if (e == cudaSuccess) e = cudaMemcpy(weights, d_w, total * sizeof(float2), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cols, d_c, total * sizeof(int32_t), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) rc = fail(PNP_ERR_CUDA, std::string("export_rows: ") + cudaGetErrorString(e));
  }
  cudaFree(d_geom);
  cudaFree(d_w);
  cudaFree(d_c);
  return rc;
}

}  // namespace pnp
