// De-gridding y = G X (Eq. 1) and gridding G^H r (App. A), separately or fused
// into one pass over G that forms the residual r = G X - y and grids it.
//
// Every row of G is an outer product of two length-J vectors (the KB kernel along
// each grid axis, convolved with the row's w-kernel).  With complex64 weights the
// plan therefore keeps the 2 J factors of a row instead of its J^2 taps, and no
// column indices: a row's taps are the J x J block of cells from its first tap on.
// A BF16 plan keeps the rounded taps themselves (their rounding does not factor).
//
// Rows are sorted by grid tile (GT x GT first-tap cells), support and first tap.
// A work unit is a run of consecutive rows of one tile and support, processed by
// ONE WARP that owns a private shared-memory copy of the tile's input cells and a
// private accumulator of its output cells, so neither shared-memory atomics nor CTA
// barriers are needed; the accumulator is flushed to the output grid with vector
// atomics at the unit's end.
//
// The warp's lanes form groups of W = 8 (J <= 8) or 16 lanes; each group walks its own
// share of the unit's rows, one row per step, lane i0 owning the taps (i1, i0).  Per row
//   s(i0) = g0[i0] sum_i1 g1[i1] X[i1][i0],   r = sum_i0 s(i0) - y   (W-lane sum),
//   t(i0) = conj(g0[i0]) r,   sum[i1][i0] += conj(g1[i1]) t(i0),
// 8 FMA per tap as packed FP32x2 FMAs over pairs of tap rows i1, with g1 (stored as pairs)
// read as shared-memory broadcasts.  While a group's consecutive rows share a window, its
// X and sums stay in registers; when it changes, the group adds its sums to the warp's
// accumulator and loads the next window.  On sparse uv coverage consecutive rows seldom
// share their first tap, so a window covers 2 x Q first taps: Q columns by the lanes that J
// taps leave idle (a row's lanes are shifted by its column), and two rows because tap
// pairs start at an even grid row of the tile (g1 is stored with a leading zero where the
// first tap is odd).  Both regions hold pairs of grid rows, (re, re, im, im) per cell pair:
// one 16-byte access per pair of taps.
// The rows stream through a per-warp ring of cp.async copies.
//
// Where rows are so sparse that the units hold one or two (pick_tile in plan_build.cu), larger tiles are taken and
// one kernel walks the units of all supports of a tile with the same regions.  Elsewhere the rows of each class of
// supports run as a kernel of their own: its registers and regions are sized for that class, and all warps of an SM
// execute the same code (one kernel for every class spent 42% of its warp time on instruction fetches).  Warps take
// batches of units from a counter; a launch of one batch per warp takes none.
//
// What bounds it: issue slots and latency (53 to 62% of issue slots at 15 to 19 warps per SM, DRAM 15 to 19%), no longer
// the traffic of G: 32 tap_pairs instead of 10 J^2 bytes per row.  Fused pass, before (CTA-wide tiles, dense
// taps, shared-memory float atomics) and now: 4096^2 image / 2e7 rows J 7-16: 6.30 -> 2.50 ms; 2048^2 /
// 5e6 rows: 1.90 -> 0.79 ms; 256^2 / 2e5 rows J = 7: 105 -> 30 us.
// Grid layout: grid[k1*K + k0].
#include <algorithm>

#include "common.cuh"

namespace pnp {
namespace {

struct GArgs {
  int K, logK, ntc;             // grid side, log2 K, tiles per side
  const Unit* units;
  unsigned u_begin, n_units;    // this launch walks units [u_begin, n_units) (one w-stack and class)
  const unsigned char* rows;    // stored rows (row_units(J) 16-byte units each)
  const int* rowh;              // uv support: per grid row the largest centred |k0| of a tap (-1: none)
  unsigned* sched;              // [0] batches taken, [1] warps done; both zero between launches.  NULL: a batch per warp
  unsigned batch;               // units per batch
  int prefetch;                 // the cells of gridB that taps reach do not stay in L2
  const int32_t* perm;
  const float2* y_in;   // sorted order (G_GRID, G_FUSED); NULL in G_FUSED = no data term
  float2* y_out;        // caller order (G_DEGRID)
  const float2* gridA;  // input grid (G_DEGRID, G_FUSED)
  float2* gridB;        // output grid (G_GRID, G_FUSED)
  __nv_bfloat162* gridB_lo;  // compensation grid: the rounding errors of the flushes into gridB, or NULL
  int* status;          // bit 2 (4): inconsistent work list (unit skipped)
};

// Rounding error of the float sum s = a + b (Knuth's TwoSum): a + b = s + err exactly.  The
// intrinsics keep the compiler from contracting or reassociating the sequence.
__device__ __forceinline__ float two_sum_err(float a, float b, float s) {
  const float bb = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Pairs of floats, kept as 64-bit values so that packed operations take them without moves.
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float x, float y) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float hsum(f2 a) {  // x + y
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return x + y;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// the two BF16 halves of a word as floats
__device__ __forceinline__ f2 bf2(uint32_t v) { return pk(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }

// Sums of re and im over the W lanes of each row group, returned to every lane: the first
// butterfly stage trades the two values, the rest sum one.
template <int W>
__device__ __forceinline__ void group_sum(float& re, float& im, int lane) {
  const bool up = (lane & (W / 2)) != 0;
  float v = up ? im : re;
  v += __shfl_xor_sync(0xffffffffu, up ? re : im, W / 2);
#pragma unroll
  for (int o = W / 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const float w = __shfl_xor_sync(0xffffffffu, v, W / 2);
  re = up ? w : v;
  im = up ? v : w;
}

// Whether a cell of an accumulator goes to the output grid.  The padding tap rows of a window hold exact zeros
// unless a visibility is not finite; the NaN they hold then must not reach a cell outside the uv support, which
// nothing zeroes again.
__device__ __forceinline__ bool flushed(const GArgs& A, float2 v, int k1, int k0) {
  return !(v.x == 0.f && v.y == 0.f) && ((v.x == v.x && v.y == v.y) || min(k0, A.K - k0) <= A.rowh[k1]);
}

// Compensated flush of a region: the atomic returns the value it added to, so the lane forms the exact rounding error
// of the (round-to-nearest) sum (TwoSum) and adds it to the compensation grid; the atomics of FB row pairs are in flight
// together.
template <typename L>
__device__ __forceinline__ void flush_compensated(const GArgs& A, ulonglong2* sy, int r0, int c0, int lane) {
  constexpr int PR = L::PR, NC = L::NC, RL = L::RL, RI = 32 / RL, FB = L::flush_pairs();
  const int Km = A.K - 1, jc = lane % RL, gc = (c0 + jc) & Km;
  if (jc >= NC) return;
  for (int i0 = lane / RL; i0 < PR; i0 += FB * RI) {
    float2 v[2 * FB], old[2 * FB];
    bool on[2 * FB];
#pragma unroll
    for (int f = 0; f < 2 * FB; ++f) {
      const int i = i0 + (f >> 1) * RI, k1 = (r0 + 2 * i + (f & 1)) & Km;
      on[f] = false;
      if (i < PR) {
        const float4 q = *reinterpret_cast<const float4*>(&sy[i * NC + jc]);
        v[f] = f & 1 ? make_float2(q.y, q.w) : make_float2(q.x, q.z);
        if (f & 1) sy[i * NC + jc] = make_ulonglong2(0, 0);
        on[f] = flushed(A, v[f], k1, gc);
        if (on[f]) old[f] = atomicAdd(&A.gridB[((size_t)k1 << A.logK) + gc], v[f]);
      }
    }
#pragma unroll
    for (int f = 0; f < 2 * FB; ++f) {
      if (!on[f]) continue;
      const size_t g = ((size_t)((r0 + 2 * (i0 + (f >> 1) * RI) + (f & 1)) & Km) << A.logK) + gc;
      const float ex = two_sum_err(old[f].x, v[f].x, __fadd_rn(old[f].x, v[f].x));
      const float ey = two_sum_err(old[f].y, v[f].y, __fadd_rn(old[f].y, v[f].y));
      if (ex != 0.f || ey != 0.f) atomicAdd(&A.gridB_lo[g], __floats2bfloat162_rn(ex, ey));
    }
  }
}

// Adds a warp's accumulator (the region from grid row r0 and column c0 on) to the output grid and clears it.
template <typename L, bool COMP>
__device__ __forceinline__ void flush_region(const GArgs& A, ulonglong2* sy, int r0, int c0, int lane) {
  constexpr int NC = L::NC, RL = L::RL, RI = 32 / RL;
  if constexpr (COMP) {
    flush_compensated<L>(A, sy, r0, c0, lane);
    return;
  }
  const int Km = A.K - 1, jc = lane % RL, gc = (c0 + jc) & Km;
  if (jc >= NC) return;
#pragma unroll 2
  for (int i = lane / RL; i < L::PR; i += RI) {
    const float4 v = *reinterpret_cast<const float4*>(&sy[i * NC + jc]);
    sy[i * NC + jc] = make_ulonglong2(0, 0);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 c = h ? make_float2(v.y, v.w) : make_float2(v.x, v.z);
      const int k1 = (r0 + 2 * i + h) & Km;
      if (flushed(A, c, k1, gc)) atomicAdd(&A.gridB[((size_t)k1 << A.logK) + gc], c);
    }
  }
}

// shared memory of one warp: the groups' rings of rows and of visibilities (or output positions), the
// accumulator region and the input region, both PR pairs of grid rows by NC columns of (re, re, im, im)
template <int MODE, bool BF, int JP, int W_, bool MIX>
struct Layout {
  static constexpr int WARPS = MIX ? 2 : 4;  // per CTA (they work independently)
  static constexpr int RING = MIX && BF ? 2 : 4;  // rows of each lane group's ring
  static constexpr int W = W_, NG = 32 / W;
  static constexpr int UNITS = BF ? JP * JP : 2 * JP, RBYTES = 16 * UNITS;  // of the largest support
  static constexpr int T = MIX ? MIX_TILE : GT;           // tile side
  static constexpr int Q = MIX ? 1 : tap_quant(JP, W);    // first-tap columns of a window
  static constexpr int PR = T / 2 - 1 + JP, NC = T - Q + W, CELLS = PR * NC;
  static constexpr int RL = NC <= 16 ? 16 : 32;           // lanes on a row pair of a region
  // row pairs of a compensated flush in flight: two, but the fused JP = 9 kernel spills in its row loop then (1e6 rows of
  // J = 16: 241 us with one, 270 with two, 280 with three out of line)
  static constexpr int flush_pairs() { return MODE == G_FUSED && JP >= 9 ? 1 : 2; }
  static constexpr int YR = NG * RING * RBYTES, YB = NG * RING * 8;
  static constexpr int OUT = YR + YB, IN = OUT + (MODE == G_DEGRID ? 0 : CELLS * 16);
  static constexpr int BYTES = (IN + (MODE == G_GRID ? 0 : CELLS * 16) + 127) & ~127;
};

// resident CTAs the registers allow for, per class
template <int JP, bool MIX>
constexpr int min_ctas() {
  return MIX ? (JP <= 6 ? 8 : 6) : JP <= 6 ? 5 : 4;
}

// MIX: the units of a plan whose units are thin (pick_tile), of any support with tap_pairs <= JP; the regions are kept
// from one unit of a tile to the next.  Otherwise the units hold rows of the class of supports (JP, W).  COMP: the flushes
// are compensated.
template <int MODE, bool BF, int JP, int W, bool MIX, bool COMP>
__global__ void __launch_bounds__(32 * Layout<MODE, BF, JP, W, MIX>::WARPS, min_ctas<JP, MIX>()) gpass(const __grid_constant__ GArgs A) {
  using L = Layout<MODE, BF, JP, W, MIX>;
  constexpr int NG = L::NG, NC = L::NC, Q = L::Q, T = L::T, RING = L::RING;
  extern __shared__ __align__(128) unsigned char sm[];
  const int lane = threadIdx.x & 31;
  const int gi = lane / W, li = lane % W;
  unsigned char* ws = sm + (threadIdx.x >> 5) * L::BYTES;
  const unsigned char* ring = ws + gi * RING * L::RBYTES;  // this group's
  const unsigned char* yring = ws + L::YR + gi * RING * 8;
  ulonglong2* sy = reinterpret_cast<ulonglong2*>(ws + L::OUT);
  ulonglong2* sx = reinterpret_cast<ulonglong2*>(ws + L::IN);
  const int Km = A.K - 1;
  const ulonglong2 zero4 = make_ulonglong2(0, 0);
  // the next class's kernel may take the SMs' free slots from here on: it reads nothing that this one writes
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // zeros: the accumulator, and the rings (a group without a row in a step reads a stale slot)
  for (int c = lane; c < L::OUT / 16; c += 32) reinterpret_cast<ulonglong2*>(ws)[c] = zero4;
  if (MODE != G_DEGRID)
    for (int c = lane; c < L::CELLS; c += 32) sy[c] = zero4;
  const uint32_t ring_a = smem_u32(ring) + li * 16, yring_a = smem_u32(yring);
  // This form of the loop keeps the fused JP = 9 kernel, at its limit of 128 registers, from spilling in its row loop (the
  // first batch by index where there is a counter too: 212 instead of 200 us for 1e6 rows of J = 16).
  unsigned nb = blockIdx.x * L::WARPS + (threadIdx.x >> 5);
  if (A.sched && lane == 0) nb = atomicAdd(A.sched, 1u);
  nb = __shfl_sync(0xffffffffu, nb, 0);
  unsigned u = A.u_begin + nb * A.batch;  // units are no more than rows: the sums stay below 2^32
  while (u < A.n_units) {
    const unsigned ue = min(u + A.batch, A.n_units);
    if (A.sched && lane == 0) nb = atomicAdd(A.sched, 1u);  // the next batch, known by the end of this one
    int held = -1;  // MIX: the tile whose regions are staged
    for (; u < (MIX ? A.n_units : ue); ++u) {
      const Unit U = A.units[u];
      if (MIX) {  // a batch is the tiles that start in it
        if (U.first && u >= ue) break;
        if (!U.first && held < 0) continue;
        if (MODE != G_DEGRID && U.first && held >= 0)
          flush_region<L, COMP>(A, sy, held / A.ntc * T, held % A.ntc * T, lane);
      }
      const int t1 = U.tile / A.ntc, t0 = U.tile - t1 * A.ntc;
      const int r0 = t1 * T, c0 = t0 * T, J = U.J;
      const bool fresh = !MIX || U.first;
      if (MIX) held = U.tile;
      if (J < 2 || (MIX ? tap_pairs(J) > JP : tap_pairs(J) != JP || tap_lanes(J) != W)) {
        if (lane == 0) atomicOr(A.status, 4);  // inconsistent work list: skip the unit
        continue;
      }
      const int jp = MIX ? tap_pairs(J) : JP, units = MIX ? row_units(J, BF) : L::UNITS;
      const int n = (U.nrows + NG - 1) / NG;  // steps; rows of this group:
      const int q0 = min(gi * n, U.nrows), mine = min(n, U.nrows - q0);
      const unsigned char* src = A.rows + ((size_t)U.row_unit << 4) + (size_t)q0 * (16 * units) + li * 16;
      const unsigned yrow = (unsigned)U.row_begin + q0;  // rows are below 2^31
      const bool has_y = A.y_in != nullptr;
      auto fetch = [&](int s) {  // copies of the group's row s, s = 0, 1, ... (one group of copies per call)
        if (s < mine) {
          const uint32_t slot = s % RING;
#pragma unroll
          for (int c = 0; c < L::UNITS; c += W)
            if ((!MIX && c + W <= L::UNITS) || c + li < units) cp16(ring_a + slot * L::RBYTES + c * 16, src + c * 16);
          src += 16 * units;
          if (li == 0) {
            if (MODE == G_DEGRID) cp4(yring_a + slot * 8, A.perm + yrow + s);
            else if (has_y) cp8(yring_a + slot * 8, A.y_in + yrow + s);
          }
        }
        cp_commit();
      };
      // Atomics on lines that are not in L2 are served far below the rate of plain fetches, so the lines that the
      // unit's flush will add to are fetched ahead (adjoint of 3e5 J = 7 rows spread over a 4096^2 grid: 285 -> 128 us,
      // 1e6 rows of J 7-16: 1050 -> 595 us).
      if (MODE != G_DEGRID && A.prefetch && fresh && lane < 2 * L::PR) {
        const float2* g = A.gridB + ((size_t)((r0 + lane) & Km) << A.logK);
#pragma unroll
        for (int c = 0; c < NC; c += 8) asm volatile("prefetch.global.L2 [%0];" ::"l"(g + ((c0 + c) & Km)));
      }
      __syncwarp();  // the previous unit's reads (and the zeros above)
#pragma unroll
      for (int s = 0; s < RING - 1; ++s) fetch(s);
      // this lane's column of the regions (two row pairs at a time where 16 lanes hold a row)
      constexpr int RL = L::RL, RI = 32 / RL;
      if (MODE != G_GRID) {
        const int jc = lane % RL, ri = lane / RL, gc = (c0 + jc) & Km;
        if (fresh && jc < NC) {
#pragma unroll 3
          for (int i = ri; i < L::PR; i += RI) {
            const float2 a = A.gridA[((size_t)((r0 + 2 * i) & Km) << A.logK) + gc];
            const float2 b = A.gridA[((size_t)((r0 + 2 * i + 1) & Km) << A.logK) + gc];
            sx[i * NC + jc] = make_ulonglong2(pk(a.x, b.x), pk(a.y, b.y));
          }
        }
      }
      int win = -1, base = 0;  // the window held in registers
      f2 xr[JP], xi[JP], sr[JP], si[JP];
#pragma unroll
      for (int p = 0; p < JP; ++p) xr[p] = xi[p] = sr[p] = si[p] = 0;
      // adds the sums of the groups in `who` to the accumulator, one group at a time (windows may overlap)
      auto retire = [&](unsigned who) {
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          if ((who >> (g * W)) & 1u) {
            if (gi == g && win >= 0) {
#pragma unroll
              for (int p = 0; p < JP; ++p) {
                ulonglong2 o = sy[base + p * NC];
                o.x = add2(o.x, sr[p]);
                o.y = add2(o.y, si[p]);
                sy[base + p * NC] = o;
              }
            }
            __syncwarp();
          }
        }
      };
      for (int s = 0; s < n; ++s) {
        fetch(s + RING - 1);
        cp_wait<RING - 1>();  // row s has landed
        __syncwarp();
        const unsigned char* rp = ring + (s % RING) * L::RBYTES;
        const unsigned char* yp = yring + (s % RING) * 8;
        const bool act = s < mine;
        const int cell = *reinterpret_cast<const int*>(rp + row_cell_at(jp, BF)) & ((T - 1) * 33);
        const int nw = cell & ((T - 2) << 5 | (T - Q));  // row pair and window columns of the first tap
        const int i0 = li - (cell & (Q - 1));            // this lane's tap column of the row
        const bool tap = (unsigned)i0 < (MIX ? (unsigned)J : 2u * JP - 1);  // the taps beyond J are stored zeros
        const bool moved = act && nw != win;
        const unsigned who = __ballot_sync(0xffffffffu, moved);
        if (who) {
          if (MODE != G_DEGRID) retire(who);
          if (moved) {
            win = nw;
            base = (nw >> 6) * NC + (nw & 31) + li;
#pragma unroll
            for (int p = 0; p < JP; ++p) {
              if (MODE != G_GRID) {
                const ulonglong2 x = sx[base + p * NC];
                xr[p] = x.x;
                xi[p] = x.y;
              }
              sr[p] = si[p] = 0;
            }
          }
        }
        float2 g0 = make_float2(0.f, 0.f);
        if constexpr (!BF) {
          if (tap) g0 = reinterpret_cast<const float2*>(rp + 16 * jp)[i0];
        }
        auto pair = [&](int p, f2& gx, f2& gy) {  // weights of tap rows 2 p and 2 p + 1
          if constexpr (BF) {
            const uint2 w = reinterpret_cast<const uint2*>(rp)[p * 2 * jp + (tap ? i0 : 0)];
            gx = bf2(w.x);
            gy = bf2(w.y);
          } else {
            const ulonglong2 g = reinterpret_cast<const ulonglong2*>(rp)[p];
            gx = g.x;
            gy = g.y;
          }
        };
        float2 r = make_float2(0.f, 0.f);
        if (MODE != G_GRID) {
          f2 a0 = 0, a1 = 0, a2 = 0, a3 = 0;
#pragma unroll
          for (int p = 0; p < JP; ++p) {
            if (MIX && p >= jp) break;
            f2 gx, gy;
            pair(p, gx, gy);
            a0 = fma2(gx, xr[p], a0);
            a1 = fma2(gy, xi[p], a1);
            a2 = fma2(gx, xi[p], a2);
            a3 = fma2(gy, xr[p], a3);
          }
          const float re = hsum(a0) - hsum(a1), im = hsum(add2(a2, a3));
          if constexpr (BF) {
            if (tap) r = make_float2(re, im);
          } else {
            r = make_float2(fmaf(g0.x, re, -g0.y * im), fmaf(g0.x, im, g0.y * re));
          }
          group_sum<W>(r.x, r.y, lane);
        }
        if (MODE == G_DEGRID) {
          if (act && li == 0) A.y_out[*reinterpret_cast<const int32_t*>(yp)] = r;
        } else {
          if (MODE == G_GRID || has_y) {
            const float2 yv = *reinterpret_cast<const float2*>(yp);
            r = MODE == G_GRID ? yv : csub(r, yv);
          }
          if (!act || (BF && !tap)) r = make_float2(0.f, 0.f);
          if constexpr (!BF) r = make_float2(fmaf(g0.x, r.x, g0.y * r.y), fmaf(g0.x, r.y, -g0.y * r.x));
          const f2 tx = pk(r.x, r.x), ty = pk(r.y, r.y), nx = pk(-r.x, -r.x);
#pragma unroll
          for (int p = 0; p < JP; ++p) {
            if (MIX && p >= jp) break;
            f2 gx, gy;
            pair(p, gx, gy);
            sr[p] = fma2(gx, tx, fma2(gy, ty, sr[p]));  // += conj(g1) t
            si[p] = fma2(gx, ty, fma2(gy, nx, si[p]));
          }
        }
        __syncwarp();  // the slot of row s is refilled by the next step
      }
      if (MODE != G_DEGRID) {
        retire(0xffffffffu);
        if (!MIX) flush_region<L, COMP>(A, sy, U.tile / A.ntc * T, U.tile % A.ntc * T, lane);
      }
    }
    if (MIX && MODE != G_DEGRID && held >= 0) flush_region<L, COMP>(A, sy, held / A.ntc * T, held % A.ntc * T, lane);
    if (!A.sched) break;
    nb = __shfl_sync(0xffffffffu, nb, 0);
    u = A.u_begin + nb * A.batch;
  }
  // This kernel ends only after the previous class's kernel has (when it was launched as its dependent), so that
  // the end of the last class's kernel is the end of the pass.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (lane == 0 && A.sched && atomicAdd(A.sched + 1, 1u) == gridDim.x * L::WARPS - 1) {  // the last warp: every batch is taken
    A.sched[0] = 0;
    A.sched[1] = 0;
  }
}

__global__ void permute_kernel(const float2* __restrict__ y, const int32_t* __restrict__ perm,
                               float2* __restrict__ out, int64_t M, float scale) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float2 v = y[perm[i]];
    out[i] = make_float2(v.x * scale, v.y * scale);
  }
}

// The classes' kernels of one pass only add to the grid (or write their own rows), so each after the first is launched
// as a programmatic dependent of the one before: its CTAs fill the tail of that kernel instead of waiting for its end.
template <int MODE, bool BF, int JP, int W, bool MIX, bool COMP>
int launch_class(pnp_plan* p, GArgs A, int s, bool* first) {
  using L = Layout<MODE, BF, JP, W, MIX>;
  const int c = s * TAP_CLASSES + (MIX ? 0 : tap_class(JP, W));
  A.u_begin = (unsigned)p->h_class_units[c];
  A.n_units = (unsigned)p->h_class_units[c + 1];
  const long long count = (long long)A.n_units - A.u_begin;
  if (count <= 0) return PNP_OK;
  const int smem = L::WARPS * L::BYTES;
  static int per_sm = 0;
  auto kernel = gpass<MODE, BF, JP, W, MIX, COMP>;
  if (per_sm == 0) {
    PNP_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    PNP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, L::WARPS * 32, smem));
    if (per_sm < 1) return fail(PNP_ERR_UNSUPPORTED, "gridding regions do not fit in shared memory");
  }
  const long long grid = std::min((long long)per_sm * p->num_sms, (count + L::WARPS - 1) / L::WARPS);
  // about 16 batches per warp: the counter is taken seldom, the last batches are short
  A.batch = (unsigned)std::max(1ll, std::min(16ll, count / (grid * L::WARPS * 16)));
  // one batch per warp needs no counter (3 of 10 us where the whole pass is one unit per warp)
  A.sched = count > grid * L::WARPS * A.batch ? p->d_sched + 2 * c : nullptr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(L::WARPS * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = p->stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = *first ? 0 : 1;
  *first = false;
  PNP_CUDA(cudaLaunchKernelEx(&cfg, kernel, A));
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return PNP_OK;
}

template <int MODE, bool BF, bool COMP>
int launch_classes(pnp_plan* p, const GArgs& A, int s) {
  bool first = true;
  if (p->mixed)
    return tap_pairs(p->Jmax) <= 5 ? launch_class<MODE, BF, 5, 16, true, COMP>(p, A, s, &first)
                                   : launch_class<MODE, BF, 9, 16, true, COMP>(p, A, s, &first);
  // the largest supports first: the short classes fill the tails
  if (int rc = launch_class<MODE, BF, 9, 16, false, COMP>(p, A, s, &first)) return rc;
  if (int rc = launch_class<MODE, BF, 8, 16, false, COMP>(p, A, s, &first)) return rc;
  if (int rc = launch_class<MODE, BF, 7, 16, false, COMP>(p, A, s, &first)) return rc;
  if (int rc = launch_class<MODE, BF, 6, 16, false, COMP>(p, A, s, &first)) return rc;
  if (int rc = launch_class<MODE, BF, 5, 16, false, COMP>(p, A, s, &first)) return rc;
  if (int rc = launch_class<MODE, BF, 5, 8, false, COMP>(p, A, s, &first)) return rc;
  return launch_class<MODE, BF, 4, 8, false, COMP>(p, A, s, &first);
}

template <int MODE>
int dispatch(pnp_plan* p, const GArgs& A, int s) {
  const bool bf = p->wdtype == PNP_W_BF16C;
  if (MODE != G_DEGRID && A.gridB_lo) {
    constexpr bool C = MODE != G_DEGRID;
    return bf ? launch_classes<MODE, true, C>(p, A, s) : launch_classes<MODE, false, C>(p, A, s);
  }
  return bf ? launch_classes<MODE, true, false>(p, A, s) : launch_classes<MODE, false, false>(p, A, s);
}

}  // namespace

int permute_y(pnp_plan* p, const float2* y_user, float scale) {
  if (p->M == 0) return PNP_OK;
  const int threads = 256;
  long long blocks = (p->M + threads - 1) / threads;
  if (blocks > 8L * p->num_sms * 8) blocks = 8L * p->num_sms * 8;
  permute_kernel<<<(unsigned)blocks, threads, 0, p->stream>>>(y_user, p->d_perm, p->d_ysorted, p->M, scale);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}

// mode G_DEGRID: y_out (caller order) = G gridA.
// mode G_GRID:   gridB += G^H d_ysorted.
// mode G_FUSED:  gridB += G^H (G gridA - d_ysorted)  (no data term when y_user == NULL).
int gridding_pass(pnp_plan* p, int mode, const float2* y_user, float2* y_out, int s) {
  if (p->M == 0 || p->n_units == 0) return PNP_OK;
  if (s < 0 || s >= p->nstacks) return fail(PNP_ERR_INVALID_ARG, "internal: stack index out of range");
  GArgs A{};
  A.K = p->K;
  A.logK = p->logK;
  A.ntc = p->ntc;
  A.units = p->d_units;
  A.rows = static_cast<const unsigned char*>(p->d_rows);
  A.rowh = p->d_rowh;
  A.prefetch = p->support_in_l2 ? 0 : 1;
  A.perm = p->d_perm;
  A.y_in = (mode == G_DEGRID || y_user == nullptr) ? nullptr : p->d_ysorted;
  A.y_out = y_out;
  A.gridA = p->d_gridA;
  A.gridB = p->d_gridB;
  A.gridB_lo = p->compensated ? p->d_gridB_lo : nullptr;
  A.status = p->d_status;
  cudaEvent_t ev;
  if (int rc = stage_begin(p, 1, &ev)) return rc;
  int rc;
  switch (mode) {
    case G_DEGRID: rc = dispatch<G_DEGRID>(p, A, s); break;
    case G_GRID: rc = dispatch<G_GRID>(p, A, s); break;
    default: rc = dispatch<G_FUSED>(p, A, s); break;
  }
  if (rc) return rc;
  return stage_end(p, 1, ev);
}

}  // namespace pnp
