// Training of the residual CNN denoiser (App. C): l1 loss
//   E || D(u + sigma n) - u ||_1,  D(z) = z - N(z)   (Eq. training_loss, without
// the firm non-expansiveness term), Adam updates, hand-written forward and
// backward kernels.  The Gaussian draws n are inputs.
//
// Precision: weights are kept in FP32 (master copy) and rounded to BF16 for
// every convolution, as in inference; hidden activations and the back-propagated
// pre-activation gradients are BF16 in memory; the loss gradient, weight
// gradients and Adam moments are FP32.
//
// Per step:
//   forward   z = u + sigma n; layer 1 (CUDA cores) -> act1; layers 2..7 on the
//             tensor cores (conv64 forward mode) -> act2..act7; layer 8 and the
//             l1 loss and its gradient g = dL/dN (CUDA cores);
//   backward  dpre7 = (W8^T g) * [act7 > 0];  for k = 6..1: dW_{k+1} from
//             (dpre_{k+1}, act_k) on the tensor cores (mma.sync, the pixels as the
//             contraction) and dpre_k = conv(dpre_{k+1}, flipped W_{k+1}^T)
//             * [act_k > 0] on the tensor cores (conv64 backward-data mode);
//             dW1 from (dpre_1, z) and dW8 on CUDA cores (one channel); bias
//             gradients are pixel sums of dpre;
//   update    Adam on the FP32 master weights, then re-pack the BF16 operands.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace pnp {
namespace {

constexpr int CH = 64;
constexpr int NW1 = CH * 9, NB1 = CH, NWM = CH * CH * 9, NBM = CH, NW8 = CH * 9;
constexpr int64_t OFF_W1 = 0, OFF_B1 = NW1;
constexpr int64_t OFF_MID = NW1 + NB1;  // 6 x (W, b)
constexpr int64_t MID_STRIDE = NWM + NBM;
constexpr int64_t OFF_W8 = OFF_MID + 6 * MID_STRIDE, OFF_B8 = OFF_W8 + NW8;
constexpr int64_t NPARAM = OFF_B8 + 1;

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// master FP32 weights -> BF16-rounded first/last layers, biases, packed middle-layer operands
__global__ void prep_weights(const float* __restrict__ w, float* __restrict__ w1r, float* __restrict__ w8r,
                             float* __restrict__ bias, __nv_bfloat16* __restrict__ wf,
                             __nv_bfloat16* __restrict__ wb) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < 6 * (int64_t)NWM) {
    const int l = (int)(i / NWM), r = (int)(i % NWM);
    const int co = r / (CH * 9), ci = (r / 9) % CH, t = r % 9;
    const __nv_bfloat16 v = __float2bfloat16_rn(w[OFF_MID + l * MID_STRIDE + r]);
    // forward operand: tap (dy, dx), input ci, output co
    wf[(size_t)l * NWM + conv_wpack_index(t / 3, t % 3, ci, co)] = v;
    // backward-data operand: the flipped tap (2 - dy, 2 - dx) with input and output channels swapped
    wb[(size_t)l * NWM + conv_wpack_index(2 - t / 3, 2 - t % 3, co, ci)] = v;
  }
  if (i < NW1) w1r[i] = bf16r(w[OFF_W1 + i]);
  if (i < NW8) {
    const int ci = (int)(i / 9), t = (int)(i % 9);
    w8r[t * CH + ci] = bf16r(w[OFF_W8 + i]);
  }
  if (i < 8 * CH) {
    const int l = (int)(i / CH), c = (int)(i % CH);
    float b = 0.f;
    if (l == 0) b = w[OFF_B1 + c];
    else if (l < 7) b = w[OFF_MID + (l - 1) * MID_STRIDE + NWM + c];
    else if (c == 0) b = w[OFF_B8];
    bias[i] = b;
  }
}

__global__ void make_z(const float* __restrict__ u, const float* __restrict__ nz, float sigma, float* __restrict__ z,
                       int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    z[i] = u[i] + sigma * nz[i];
}

struct Dims {
  int B, s, Hc, Wc;
};

__device__ __forceinline__ size_t cidx(const Dims& d, int b, int y, int x, int c) {
  return canvas_index(b, y, x, c, d.Hc, d.Wc);
}

// ------------------------------------------------------------ the one-channel ends (layers 1 and 8)
// Tap t of a 3 x 3 stencil sits at off_t = (t / 3 - 1, t % 3 - 1); FLIP takes the pixels p - off_t in the
// place of p + off_t (a transposed convolution).  Pixels outside the image are zero.
constexpr int END_COLS = 32;  // columns of a block of the walks below: one per lane, a warp per channel block

// pairs of floats, kept as 64-bit values so that packed FMAs take them without moves
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float x, float y) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 unpk(f2 a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {  // two FP32 FMAs, one instruction
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// the two BF16 halves of a word as a pair of floats
__device__ __forceinline__ f2 bf2(uint32_t v) { return pk(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }

// rows y0 - 1 .. y0 + rows and columns x0 - 1 .. x0 + END_COLS of image b, zero outside, into shared memory
__device__ __forceinline__ void stage_window(const Dims& d, const float* __restrict__ img, int b, int y0, int x0,
                                             int rows, float (*zt)[END_COLS + 2]) {
  for (int i = threadIdx.x; i < (rows + 2) * (END_COLS + 2); i += blockDim.x) {
    const int r = i / (END_COLS + 2), c = i % (END_COLS + 2), y = y0 + r - 1, x = x0 + c - 1;
    zt[r][c] = y >= 0 && y < d.s && x >= 0 && x < d.s ? img[((int64_t)b * d.s + y) * d.s + x] : 0.f;
  }
  __syncthreads();
}
constexpr int END_ROWS = 64;  // rows of a block at most
constexpr int END_BATCH = 4;  // rows whose canvas loads a lane issues together (one at a time left HBM at 1.5 TB/s)

// 1 -> 64 with a ReLU mask: out[p][c] = [mask[p][c] > 0] sum_t W[c][t] img[p + off_t] (FLIP: p - off_t).
//   layer 8 backward: W = W8 stored [t][c], FLIP;  layer 1 tangent: W = W1 stored [c][t].
// Warp w forms channel block w of 32 columns row after row with its 72 weights in registers: one 16-byte load
// (mask) and store per lane and row, whole 512-byte runs per warp.  Bound by that traffic (256 B a pixel).
// 16 x 256^2: 82 -> 62 us against a thread per pixel with the weights read from shared memory.
template <bool FLIP>
__global__ void __launch_bounds__(256) one_to_many(Dims d, int rows, const __nv_bfloat16* __restrict__ mask,
                                                   const float* __restrict__ w, const float* __restrict__ img,
                                                   __nv_bfloat16* __restrict__ out) {
  __shared__ float zt[END_ROWS + 2][END_COLS + 2];
  const int b = blockIdx.z, y0 = blockIdx.y * rows, x0 = blockIdx.x * END_COLS;
  const int cb = threadIdx.x >> 5, lane = threadIdx.x & 31;
  stage_window(d, img, b, y0, x0, rows, zt);
  f2 wt[4][9];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int c = 8 * cb + 2 * q;
      wt[q][t] = FLIP ? pk(w[t * CH + c], w[t * CH + c + 1]) : pk(w[c * 9 + t], w[(c + 1) * 9 + t]);
    }
  const int x = x0 + lane, ye = min(rows, d.s - y0);
  if (x >= d.s) return;
  const size_t step = (size_t)d.Wc * CH;
  size_t at = cidx(d, b, y0, x, 8 * cb);
  for (int rb = 0; rb < ye; rb += END_BATCH) {
    uint4 m[END_BATCH];
#pragma unroll
    for (int k = 0; k < END_BATCH; ++k)
      if (rb + k < ye) m[k] = *reinterpret_cast<const uint4*>(mask + at + k * step);
#pragma unroll
    for (int k = 0; k < END_BATCH; ++k, at += step) {
      const int r = rb + k;
      if (r >= ye) break;
      const uint4 mc = m[k];
      f2 v[4] = {0, 0, 0, 0};
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const float g = FLIP ? zt[r + 2 - t / 3][lane + 2 - t % 3] : zt[r + t / 3][lane + t % 3];
        const f2 gg = pk(g, g);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = fma2(wt[q][t], gg, v[q]);
      }
      uint4 o;
      const uint32_t* mw = reinterpret_cast<const uint32_t*>(&mc);
      uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 a = unpk(bf2(mw[q])), u = unpk(v[q]);
        const __nv_bfloat162 h = __floats2bfloat162_rn(a.x > 0.f ? u.x : 0.f, a.y > 0.f ? u.y : 0.f);
        ow[q] = *reinterpret_cast<const uint32_t*>(&h);
      }
      *reinterpret_cast<uint4*>(out + at) = o;
    }
  }
}

// Gradients of a one-channel layer: dW[c][t] += sum_p cv[p][c] img[p + off_t] (FLIP: p - off_t), and
//   FLIP (layer 8: cv = act7, img = g):     db[0] += sum_p img[p]
//   else (layer 1: cv = dpre1, img = z):    db[c] += sum_p cv[p][c].
// Same walk as one_to_many, a block taking tiles of 32 columns by `rows` rows until none are left: a lane keeps
// the 8 x 9 sums of its column, the warp adds them up by exchanging halves (80 values in 80 shuffles) and writes
// them to the block's slice of a workspace, which onechannel_reduce adds up (as global atomics on the 576 sums
// they took 30 us however small the batch).  Bound by the canvas read.  16 x 256^2: 3040 -> 67 us (8 x 128^2: 1085 -> 19 us) against a
// thread per (tap, channel) that walked 2048 pixels one after the other.
constexpr int ONE_SUMS = 8 * 80;  // a block's partial sums: [channel block][t][8 channels], t = 9: the bias
template <bool FLIP>
__global__ void __launch_bounds__(256) wgrad_onechannel(Dims d, int rows, const float* __restrict__ img,
                                                        const __nv_bfloat16* __restrict__ cv, float* __restrict__ part) {
  __shared__ float zt[END_ROWS + 2][END_COLS + 2];
  const int cb = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tx = (d.s + END_COLS - 1) / END_COLS, ty = (d.s + rows - 1) / rows, tiles = tx * ty * d.B;
  f2 acc[9][4], bias[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    bias[q] = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) acc[t][q] = 0;
  }
  const size_t step = (size_t)d.Wc * CH;
  const f2 one = pk(1.f, 1.f);
  float isum = 0.f;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int x0 = tile % tx * END_COLS, y0 = tile / tx % ty * rows, b = tile / (tx * ty);
    __syncthreads();  // the previous tile's window
    stage_window(d, img, b, y0, x0, rows, zt);
    const int x = x0 + lane, ye = x < d.s ? min(rows, d.s - y0) : 0;
    const __nv_bfloat16* src = cv + cidx(d, b, y0, min(x, d.s - 1), 8 * cb);
    for (int rb = 0; rb < ye; rb += END_BATCH) {
      uint4 m[END_BATCH];
#pragma unroll
      for (int k = 0; k < END_BATCH; ++k)
        m[k] = rb + k < ye ? *reinterpret_cast<const uint4*>(src + (rb + k) * step) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int k = 0; k < END_BATCH; ++k) {
        const int r = rb + k;
        if (r >= ye) break;
        const f2 ch[4] = {bf2(m[k].x), bf2(m[k].y), bf2(m[k].z), bf2(m[k].w)};
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          const float g = FLIP ? zt[r + 2 - t / 3][lane + 2 - t % 3] : zt[r + t / 3][lane + t % 3];
          const f2 gg = pk(g, g);
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[t][q] = fma2(ch[q], gg, acc[t][q]);
        }
        if (FLIP) {
          isum += zt[r + 1][lane + 1];
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) bias[q] = fma2(ch[q], one, bias[q]);
        }
      }
    }
  }
  float v[80];  // [t][8 channels], then 8 bias sums (FLIP: the image's sum in the first)
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int t = 0; t < 10; ++t) {
      const float2 u = unpk(t < 9 ? acc[t < 9 ? t : 0][q] : bias[q]);
      v[8 * t + 2 * q] = FLIP && t == 9 && q == 0 ? isum : u.x;
      v[8 * t + 2 * q + 1] = u.y;
    }
  }
  int base = 0;  // the values this lane ends up with: v[0..4] = totals of base .. base + 4
#pragma unroll
  for (int n = 40, o = 16; n >= 5; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const float send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    base += up ? n : 0;
  }
  float* o = part + (size_t)blockIdx.x * ONE_SUMS + 80 * cb + base;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1);
    if (!(lane & 1)) o[k] = v[k];
  }
}

// dW[c][t] += and db += the sums of the `parts` slices (layer 8: one bias, in channel block 0); block (32, 8)
__global__ void __launch_bounds__(256) onechannel_reduce(const float* __restrict__ part, int parts, int layer8,
                                                         float* __restrict__ dW, float* __restrict__ db) {
  __shared__ float red[8][32];
  const int e = blockIdx.x * 32 + threadIdx.x;
  float s = 0.f;
  for (int k = threadIdx.y; k < parts; k += 8) s += part[(size_t)k * ONE_SUMS + e];
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y) return;
  for (int k = 1; k < 8; ++k) s += red[k][threadIdx.x];
  const int cb = e / 80, t = e % 80 / 8, c = e % 8;
  if (t < 9) dW[(8 * cb + c) * 9 + t] += s;
  else if (!layer8) db[8 * cb + c] += s;
  else if (e == 72) db[0] += s;
}

// 64 -> 1: N[p] = init + sum_{t, c} W[t][c] cv[p + off_t][c] (FLIP: p - off_t), then
//   M2O_LOSS: r = z - N - u, loss += |r| / count, out = dL/dN = -sign(r) / count  (layer 8 forward)
//   M2O_JAC:  out = v - 2 N                                                       (J_Q v and J_Q^T w)
// A thread holds one column of M2O_ROWS output rows and walks the M2O_ROWS + 2 canvas rows that they read, so
// each 8-channel vector is loaded 3 (M2O_ROWS + 2) / M2O_ROWS times per pixel instead of 9.  The terms of a pixel
// are added in the order t, c as one chain (the sign of r, and through it every gradient, hangs on the last bit
// of N).  Bound by those FMA (576 a pixel) and the loads of the weights.  16 x 256^2: 184 -> 95 us.
constexpr int M2O_LOSS = 0, M2O_JAC = 1, M2O_THREADS = 128;
template <int MODE, bool FLIP, int ROWS>
__global__ void __launch_bounds__(M2O_THREADS) many_to_one(Dims d, const __nv_bfloat16* __restrict__ cv,
                                                           const float* __restrict__ w, int w_taps_first,
                                                           const float* __restrict__ bias, const float* __restrict__ v,
                                                           const float* __restrict__ u, float* __restrict__ out,
                                                           double* loss) {
  __shared__ __align__(16) float sw[9 * CH];
  __shared__ double red[M2O_THREADS / 32];
  for (int i = threadIdx.x; i < 9 * CH; i += blockDim.x) sw[w_taps_first ? i : (i % 9) * CH + i / 9] = w[i];
  __syncthreads();
  const int b = blockIdx.z, y0 = blockIdx.y * ROWS, x = blockIdx.x * M2O_THREADS + threadIdx.x;
  float acc[ROWS];
  const float init = MODE == M2O_LOSS ? bias[7 * CH] : 0.f;
#pragma unroll
  for (int k = 0; k < ROWS; ++k) acc[k] = init;
#pragma unroll
  for (int rr = 0; rr < ROWS + 2; ++rr) {
    // canvas rows in the order in which every output row meets its taps
    const int k0 = FLIP ? ROWS - rr : rr - 1;  // canvas row y0 + k0
    const int y = y0 + k0;
    const bool row_in = y >= 0 && y < d.s;
#pragma unroll 1
    for (int dx = 0; dx < 3; ++dx) {
      const int xx = FLIP ? x + 1 - dx : x + dx - 1;
      const bool in = row_in && xx >= 0 && xx < d.s;
      const __nv_bfloat16* src = cv + cidx(d, b, in ? y : 0, in ? xx : 0, 0);
      const size_t plane = (size_t)d.Wc * 8;
#pragma unroll 2
      for (int cb = 0; cb < 8; ++cb) {
        const uint4 a = in ? *reinterpret_cast<const uint4*>(src + cb * plane) : make_uint4(0, 0, 0, 0);
        const uint32_t* aw = reinterpret_cast<const uint32_t*>(&a);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 av = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[q]));
#pragma unroll
          for (int ty = 0; ty < 3; ++ty) {
            const int k = FLIP ? k0 + ty - 1 : k0 - ty + 1;  // the output row for which this row is tap row ty
            if (k < 0 || k >= ROWS) continue;
            const float2 wv = *reinterpret_cast<const float2*>(&sw[(3 * ty + dx) * CH + 8 * cb + 2 * q]);
            acc[k] = fmaf(wv.x, av.x, fmaf(wv.y, av.y, acc[k]));
          }
        }
      }
    }
  }
  double sum = 0.0;
  const float inv = 1.f / (float)((int64_t)d.B * d.s * d.s);
#pragma unroll
  for (int k = 0; k < ROWS; ++k) {
    if (x >= d.s || y0 + k >= d.s) continue;
    const int64_t p = ((int64_t)b * d.s + y0 + k) * d.s + x;
    if (MODE == M2O_LOSS) {
      const float r = v[p] - acc[k] - u[p];
      sum += fabs((double)r);
      out[p] = r > 0.f ? -inv : (r < 0.f ? inv : 0.f);
    } else {
      out[p] = v[p] - 2.f * acc[k];
    }
  }
  if (MODE == M2O_LOSS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < M2O_THREADS / 32; ++k) sum += red[k];
      atomicAdd(loss, sum * (double)inv);
    }
  }
}

// Weight and bias gradients of a 64 -> 64 layer on the tensor cores (mma.sync m16n8k16, BF16 in, FP32
// accumulate): dW[co][ci][t] = sum_p dpre[p][co] act[p + off_t][ci] is, per tap t, a 64 x 64 GEMM whose
// contraction runs over the pixels.  The image rows of all 64-pixel column segments form one sequence that is
// cut evenly over the CTAs.  A CTA walks down a segment: per row it copies one dpre row (64 px x 64 ch) and the
// next activation row (66 px with the dx halo, zero outside the image) into rings in shared memory with cp.async,
// WGT_AHEAD rows ahead, as [pixel][channel] rows padded to 72 channels (conflict-free ldmatrix); each activation
// row serves three dpre rows.  Warp w owns tap w / 2 and output channels 32 (w % 2) .. + 31: 2 x 8 tiles of
// 16 x 8 accumulators.  Both operands are stored pixel-major, so the fragments load with ldmatrix.trans.  Bias
// gradients (sums of dpre over the pixels) come from the fragments of the centre tap's warps.  Each
// CTA writes its partial sums to its slice of a workspace and wgrad64_reduce adds the slices up (as global atomics
// the 36864 sums of each CTA cost about as much as the contraction).
// Bound by the tensor pipe as mma.sync drives it (math pipe throttle, 330 TFLOP/s).  16 x 256^2: 381 -> 244 us
// with the reduction (8 x 128^2: 106 -> 45 us) against restaging three activation rows per row, two stages deep,
// a serial bias sum and atomics.
constexpr int WGT_PX = 64;                    // pixels per segment (4 K steps of 16)
constexpr int WGT_LD = 72;                    // staged row length (channels + 8 of padding)
constexpr int WGT_WARPS = 18;                 // 9 taps x 2 output-channel halves
constexpr int WGT_THREADS = WGT_WARPS * 32;
constexpr int WGT_AHEAD = 3;                  // rows whose copies are in flight
constexpr int WGT_NA = WGT_AHEAD + 3, WGT_ND = WGT_AHEAD + 1;   // ring slots: activation and dpre rows
constexpr int WGT_AROW = (WGT_PX + 2) * WGT_LD, WGT_DROW = WGT_PX * WGT_LD;  // elements of a slot
constexpr int WGT_SMEM = (WGT_NA * WGT_AROW + WGT_ND * WGT_DROW) * 2;
constexpr int WGT_SUMS = 9 * CH * CH + CH;    // a CTA's partial sums: [t][co][ci], then [co] of the bias

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], const void* p) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a));
}
// 16-byte asynchronous copy global -> shared; nbytes = 0 fills the destination with zeros
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int nbytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(static_cast<uint32_t>(
                   __cvta_generic_to_shared(dst))),
               "l"(src), "r"(nbytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// copies PX pixels x .. of canvas row y of image b (zero outside the image) into dst, [px][WGT_LD]
template <int PX>
__device__ __forceinline__ void wgt_row(const Dims& d, const __nv_bfloat16* __restrict__ cv, int b, int y, int x,
                                        __nv_bfloat16* dst) {
  const bool row_in = y >= 0 && y < d.s;
  for (int e = threadIdx.x; e < 8 * PX; e += WGT_THREADS) {
    const int kb = e / PX, px = e - kb * PX, xx = x + px;
    const bool in = row_in && xx >= 0 && xx < d.s;
    cp_async16(dst + px * WGT_LD + 8 * kb, in ? cv + cidx(d, b, y, xx, 8 * kb) : cv, in ? 16 : 0);
  }
}

__global__ void __launch_bounds__(WGT_THREADS, 1) wgrad64_tc(Dims d, const __nv_bfloat16* __restrict__ dpre,
                                                             const __nv_bfloat16* __restrict__ act,
                                                             float* __restrict__ part) {
  extern __shared__ __align__(16) __nv_bfloat16 wsm[];
  __nv_bfloat16* sA = wsm;                        // activation ring, row y in slot (y + 1) mod WGT_NA
  __nv_bfloat16* sD = wsm + WGT_NA * WGT_AROW;    // dpre ring, row y in slot y mod WGT_ND
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = warp >> 1, dy = t / 3, dx = t % 3, co0 = 32 * (warp & 1);
  const int segs = (d.s + WGT_PX - 1) / WGT_PX;
  const int64_t total = (int64_t)d.B * segs * d.s;
  int64_t l = total * blockIdx.x / gridDim.x;
  const int64_t le = total * (blockIdx.x + 1) / gridDim.x;
  float acc[2][8][4] = {}, bsum[2][2] = {};
  const int i = lane >> 3, r = lane & 7;
  while (l < le) {
    const int strip = (int)(l / d.s), ya = (int)(l % d.s), yb = (int)min((int64_t)d.s, ya + (le - l));
    const int b = strip / segs, x0 = strip % segs * WGT_PX;
    auto fetch = [&](int y) {  // the copies of step y: dpre row y and activation row y + 1
      if (y < yb) {
        wgt_row<WGT_PX>(d, dpre, b, y, x0, sD + y % WGT_ND * WGT_DROW);
        wgt_row<WGT_PX + 2>(d, act, b, y + 1, x0 - 1, sA + (y + 2) % WGT_NA * WGT_AROW);
      }
      cp_async_commit();
    };
    __syncthreads();  // every warp is done with the previous strip's rings
    wgt_row<WGT_PX + 2>(d, act, b, ya - 1, x0 - 1, sA + ya % WGT_NA * WGT_AROW);
    wgt_row<WGT_PX + 2>(d, act, b, ya, x0 - 1, sA + (ya + 1) % WGT_NA * WGT_AROW);
    for (int y = ya; y < ya + WGT_AHEAD; ++y) fetch(y);
    for (int y = ya; y < yb; ++y) {
      cp_async_wait<WGT_AHEAD - 1>();  // this thread's copies of step y have landed
      __syncthreads();                 // and everyone's; the slots filled next were last read in step y - 1
      fetch(y + WGT_AHEAD);
      const __nv_bfloat16* pD = sD + y % WGT_ND * WGT_DROW;
      const __nv_bfloat16* pA = sA + (y + dy) % WGT_NA * WGT_AROW;  // activation row y + dy - 1
#pragma unroll
      for (int kk = 0; kk < WGT_PX / 16; ++kk) {
        uint32_t a[2][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
          ldsm_x4_trans(a[mt], pD + (16 * kk + r + 8 * (i >> 1)) * WGT_LD + co0 + 16 * mt + 8 * (i & 1));
#pragma unroll
        for (int np = 0; np < 4; ++np) {
          uint32_t bq[4];
          ldsm_x4_trans(bq, pA + (16 * kk + r + 8 * (i & 1) + dx) * WGT_LD + 16 * np + 8 * (i >> 1));
#pragma unroll
          for (int mt = 0; mt < 2; ++mt) {
            mma16816(acc[mt][2 * np], a[mt], bq[0], bq[1]);
            mma16816(acc[mt][2 * np + 1], a[mt], bq[2], bq[3]);
          }
        }
        if (t == 4) {  // warp-uniform: the pixel sums of dpre, rows g and g + 8 of the fragments
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a[mt][h]));
              const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a[mt][2 + h]));
              bsum[mt][h] += (lo.x + lo.y) + (hi.x + hi.y);
            }
        }
      }
    }
    l += yb - ya;
  }
  cp_async_wait<0>();
  const int g = lane >> 2, tq = lane & 3;
  float* o = part + (size_t)blockIdx.x * WGT_SUMS;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int co = co0 + 16 * mt + g + 8 * h;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
        *reinterpret_cast<float2*>(&o[(t * CH + co) * CH + 8 * nt + 2 * tq]) =
            make_float2(acc[mt][nt][2 * h], acc[mt][nt][2 * h + 1]);
      if (t == 4) {
        float v = bsum[mt][h];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (tq == 0) o[9 * CH * CH + co] = v;
      }
    }
}

// dW[co][ci][t] and db[co] += the sums of the `parts` slices; block (32, 8): 32 sums, the slices dealt to 8 rows
__global__ void __launch_bounds__(256) wgrad64_reduce(const float* __restrict__ part, int parts,
                                                      float* __restrict__ dW, float* __restrict__ db) {
  __shared__ float red[8][32];
  const int e = blockIdx.x * 32 + threadIdx.x;
  float s = 0.f;
  if (e < WGT_SUMS)
    for (int k = threadIdx.y; k < parts; k += 8) s += part[(size_t)k * WGT_SUMS + e];
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y || e >= WGT_SUMS) return;
  for (int k = 1; k < 8; ++k) s += red[k][threadIdx.x];
  if (e < 9 * CH * CH) dW[(size_t)(e % (CH * CH)) * 9 + e / (CH * CH)] += s;
  else db[e - 9 * CH * CH] += s;
}

int device_sms(int* sms) {
  int dev = 0;
  PNP_CUDA(cudaGetDevice(&dev));
  PNP_CUDA(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return PNP_OK;
}

int wgrad64_launch(cudaStream_t s, const Dims& d, const __nv_bfloat16* dpre, const __nv_bfloat16* act, float* part,
                   int parts, float* dW, float* db) {
  static bool attr = false;
  if (!attr) {
    PNP_CUDA(cudaFuncSetAttribute(wgrad64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, WGT_SMEM));
    attr = true;
  }
  wgrad64_tc<<<parts, WGT_THREADS, WGT_SMEM, s>>>(d, dpre, act, part);
  PNP_CHECK_LAUNCH();
  wgrad64_reduce<<<(WGT_SUMS + 31) / 32, dim3(32, 8), 0, s>>>(part, parts, dW, db);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}

// launch shape of one_to_many and wgrad_onechannel: as many rows per block (8 to 64) as leave three blocks per SM
dim3 end_grid(const Dims& d, int sms, int* rows) {
  const int cols = (d.s + END_COLS - 1) / END_COLS;
  *rows = END_ROWS;
  while (*rows > 8 && (int64_t)cols * ((d.s + *rows - 1) / *rows) * d.B < 3 * sms) *rows >>= 1;
  return dim3(cols, (d.s + *rows - 1) / *rows, d.B);
}

template <int MODE, bool FLIP>
int many_to_one_launch(cudaStream_t s, const Dims& d, int sms, const __nv_bfloat16* cv, const float* w,
                       int w_taps_first, const float* bias, const float* v, const float* u, float* out, double* loss) {
  const int cols = (d.s + M2O_THREADS - 1) / M2O_THREADS;
  if ((int64_t)cols * ((d.s + 7) / 8) * d.B >= 4 * sms)
    many_to_one<MODE, FLIP, 8><<<dim3(cols, (d.s + 7) / 8, d.B), M2O_THREADS, 0, s>>>(d, cv, w, w_taps_first, bias, v, u, out, loss);
  else
    many_to_one<MODE, FLIP, 2><<<dim3(cols, (d.s + 1) / 2, d.B), M2O_THREADS, 0, s>>>(d, cv, w, w_taps_first, bias, v, u, out, loss);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}

// ---------------------------------------------------------------- Jacobian of Q = 2D - I
// With D(z) = z - N(z), J_Q = I - 2 J_N, and J_N at z is the network with its ReLU masks at z
// frozen and no biases.  Layers 2-7 of J_N v run on the tensor cores (conv64 backward-data mode
// with the forward weights and the masks [act_{k+1} > 0]); J_N^T w is the back-propagation of
// the training step; the one-channel ends of both chains are one_to_many and many_to_one.

// n2[b] += sum_p x[b][p]^2 (FP64); grid (blocks per image, B)
__global__ void __launch_bounds__(256) image_norm2(const float* __restrict__ x, int64_t plane, double* n2) {
  __shared__ double red[256];
  const float* xb = x + (int64_t)blockIdx.y * plane;
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < plane; i += (int64_t)gridDim.x * blockDim.x)
    s += (double)xb[i] * xb[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x >> 1; k > 0; k >>= 1) {
    if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(&n2[blockIdx.y], red[0]);
}

// v[b][p] = u[b][p] / sqrt(n2[b]) (a zero image stays zero)
__global__ void __launch_bounds__(256) image_unit(const float* __restrict__ u, const double* __restrict__ n2,
                                                  int64_t plane, int B, float* __restrict__ v) {
  const int64_t total = plane * B;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const double n = n2[i / plane];
    v[i] = n > 0.0 ? (float)(u[i] / sqrt(n)) : 0.f;
  }
}

// Cotangent of the soft firm non-expansiveness penalty lam/B sum_b max(||w_b||^2, 1 - eps) with
// w = J_Q v: c[b][p] = -4 lam/B w[b][p] where ||w_b||^2 > 1 - eps, else 0.
__global__ void __launch_bounds__(256) fne_cotangent(const float* __restrict__ w, const double* __restrict__ n2,
                                                     int64_t plane, int B, float scale, double floor_,
                                                     float* __restrict__ c) {
  const int64_t total = plane * B;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
    c[i] = n2[i / plane] > floor_ ? -4.f * scale * w[i] : 0.f;
}

// Adam (Kingma & Ba 2015) on the master weights; the gradient is cleared for the next step.
// omb1 = 1 - b1 and omb2 = 1 - b2 come from the host in double precision: formed in FP32 from
// b2 = 0.999f, 1 - b2 would be off by 1.3e-5 relative, and the step m^/sqrt(v^) by half that.
__global__ void adam_step(float* __restrict__ w, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                          int64_t count, float lr, float b1, float b2, float omb1, float omb2, float eps, float c1,
                          float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + omb1 * gi;
    const float vi = b2 * v[i] + omb2 * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    g[i] = 0.f;
  }
}

__global__ void zero_f(float* p, int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = 0.f;
}

int nblocks(int64_t count, int threads = 256) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (int)std::max<int64_t>(1, std::min<int64_t>((count + threads - 1) / threads, 8L * sms));
}

}  // namespace
}  // namespace pnp

struct pnp_cnn_trainer {
  pnp::Dims d{};
  cudaStream_t stream = nullptr;
  int n_strips = 0, conv_grid = 0, t = 0, sms = 0;
  int parts = 0;          // CTAs of the weight-gradient kernel
  float* part = nullptr;  // their partial sums (parts x WGT_SUMS)
  double lr = 1e-4, b1 = 0.9, b2 = 0.999, eps = 1e-8;
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  float *w1r = nullptr, *w8r = nullptr, *bias = nullptr;
  __nv_bfloat16 *wf = nullptr, *wb = nullptr;
  __nv_bfloat16* act[8] = {};
  __nv_bfloat16* dp[2] = {};
  float *z = nullptr, *gout = nullptr;
  int4 *facets = nullptr, *strips = nullptr;
  double* loss = nullptr;
  int* status = nullptr;
  float *jv = nullptr, *jw = nullptr, *ju = nullptr;  // Jacobian power iteration images (B x s x s)
  double* jn2 = nullptr;                                // their per-image squared norms [B]
  __nv_bfloat16* tan[8] = {};                           // tangents t_1..t_7 of the penalty's J_N v
  float* junk = nullptr;                                // bias-gradient sink of the tangent network [64]
  alignas(64) unsigned char map_tan[8][256];            // TMA descriptors of tan[1..6]
  alignas(64) unsigned char map_act[8][256];  // TMA descriptors (main, halo) of act[1..7]
  alignas(64) unsigned char map_dp[2][256];   // and of the two gradient canvases
};

using namespace pnp;

namespace {
void trainer_free(pnp_cnn_trainer* T) {
  if (!T) return;
  for (void* p : {(void*)T->w, (void*)T->g, (void*)T->m, (void*)T->v, (void*)T->w1r, (void*)T->w8r, (void*)T->bias,
                  (void*)T->wf, (void*)T->wb, (void*)T->z, (void*)T->gout, (void*)T->facets, (void*)T->strips,
                  (void*)T->loss, (void*)T->status, (void*)T->jv, (void*)T->jw, (void*)T->ju, (void*)T->jn2, (void*)T->part})
    cudaFree(p);
  for (auto p : T->act) cudaFree(p);
  for (auto p : T->dp) cudaFree(p);
  for (auto p : T->tan) cudaFree(p);
  cudaFree(T->junk);
  delete T;
}

int prep(pnp_cnn_trainer* T) {
  prep_weights<<<nblocks(6 * (int64_t)NWM), 256, 0, T->stream>>>(T->w, T->w1r, T->w8r, T->bias, T->wf, T->wb);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}
}  // namespace

namespace {
// per-image squared norms of x into T->jn2
int image_norms(pnp_cnn_trainer* T, const float* x) {
  const int64_t plane = (int64_t)T->d.s * T->d.s;
  PNP_CUDA(cudaMemsetAsync(T->jn2, 0, T->d.B * sizeof(double), T->stream));
  const int bx = (int)std::min<int64_t>((plane + 255) / 256, 64);
  image_norm2<<<dim3(bx, T->d.B), 256, 0, T->stream>>>(x, plane, T->jn2);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}
}  // namespace

namespace {
// dpre7 = [act7 > 0] W8^T g into dp[0]
int layer8_back(pnp_cnn_trainer* T, const float* g) {
  int rows;
  const dim3 grid = end_grid(T->d, T->sms, &rows);
  one_to_many<true><<<grid, 256, 0, T->stream>>>(T->d, rows, T->act[7], T->w8r, g, T->dp[0]);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}
// t1 = [act1 > 0] W1 v
int layer1_tangent(pnp_cnn_trainer* T, const float* v, __nv_bfloat16* t1) {
  int rows;
  const dim3 grid = end_grid(T->d, T->sms, &rows);
  one_to_many<false><<<grid, 256, 0, T->stream>>>(T->d, rows, T->act[1], T->w1r, v, t1);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}
template <bool LAYER8>
int onechannel_grads(pnp_cnn_trainer* T, const float* img, const __nv_bfloat16* cv, float* dW, float* db) {
  int rows;
  const dim3 tiles = end_grid(T->d, T->sms, &rows);
  // two blocks per SM are resident; the workspace holds more than 57 slices per weight-gradient CTA
  const int blocks = (int)std::min<int64_t>((int64_t)tiles.x * tiles.y * tiles.z, 2 * T->parts);
  wgrad_onechannel<LAYER8><<<blocks, 256, 0, T->stream>>>(T->d, rows, img, cv, T->part);
  PNP_CHECK_LAUNCH();
  onechannel_reduce<<<ONE_SUMS / 32, dim3(32, 8), 0, T->stream>>>(T->part, blocks, LAYER8 ? 1 : 0, dW, db);
  PNP_CHECK_LAUNCH();
  return PNP_OK;
}

// the forward pass at z that fixes the ReLU masks (activations act[1..7])
int primal_forward(pnp_cnn_trainer* T, const float* z) {
  const Dims d = T->d;
  cudaStream_t s = T->stream;
  if (int rc = cnn_first_launch(s, z, d.s, (int64_t)d.s * d.s, T->facets, d.B, d.Hc, d.Wc, T->w1r, T->bias,
                                T->act[1]))
    return rc;
  for (int k = 1; k <= 6; ++k)
    if (int rc = conv64_launch(s, T->map_act[k], T->act[k + 1], T->wf + (size_t)(k - 1) * NWM, T->bias + k * CH,
                               T->strips, T->n_strips, T->conv_grid, d.Hc, d.Wc, 0, nullptr, T->status))
      return rc;
  return PNP_OK;
}

// Power iteration on J_Q^T J_Q at the current activations from v0 (normalised per image):
// T->jv ends as the last unit iterate; sigma_host (if given) gets ||J_Q v|| of the last step.
int power_iterate(pnp_cnn_trainer* T, const float* v0, int iters, double* sigma_host) {
  const Dims d = T->d;
  const int64_t plane = (int64_t)d.s * d.s, npx = plane * d.B;
  cudaStream_t s = T->stream;
  if (int rc = image_norms(T, v0)) return rc;
  image_unit<<<nblocks(npx), 256, 0, s>>>(v0, T->jn2, plane, d.B, T->jv);
  PNP_CHECK_LAUNCH();
  for (int it = 0; it < iters; ++it) {
    // w = J_Q v: tangents through layers 1..7 (masks [act_k > 0]), then layer 8
    if (int rc = layer1_tangent(T, T->jv, T->dp[0])) return rc;
    int cur = 0;
    for (int k = 1; k <= 6; ++k) {
      if (int rc = conv64_launch(s, T->map_dp[cur], T->dp[1 - cur], T->wf + (size_t)(k - 1) * NWM, nullptr, T->strips,
                                 T->n_strips, T->conv_grid, d.Hc, d.Wc, 1, T->act[k + 1], T->status))
        return rc;
      cur = 1 - cur;
    }
    if (int rc = many_to_one_launch<M2O_JAC, false>(s, d, T->sms, T->dp[cur], T->w8r, 1, nullptr, T->jv, nullptr, T->jw, nullptr))
      return rc;
    // u = J_Q^T w: the training step's back-propagation with cotangent w
    if (int rc = layer8_back(T, T->jw)) return rc;
    cur = 0;
    for (int k = 6; k >= 1; --k) {
      if (int rc = conv64_launch(s, T->map_dp[cur], T->dp[1 - cur], T->wb + (size_t)(k - 1) * NWM, nullptr, T->strips,
                                 T->n_strips, T->conv_grid, d.Hc, d.Wc, 1, T->act[k], T->status))
        return rc;
      cur = 1 - cur;
    }
    if (int rc = many_to_one_launch<M2O_JAC, true>(s, d, T->sms, T->dp[cur], T->w1r, 0, nullptr, T->jw, nullptr, T->ju, nullptr))
      return rc;
    if (sigma_host && it == iters - 1) {  // sigma = ||J_Q v|| for the current unit v
      if (int rc = image_norms(T, T->jw)) return rc;
      PNP_CUDA(cudaMemcpyAsync(sigma_host, T->jn2, d.B * sizeof(double), cudaMemcpyDeviceToHost, s));
      PNP_CUDA(cudaStreamSynchronize(s));
      for (int b = 0; b < d.B; ++b) sigma_host[b] = std::sqrt(sigma_host[b]);
    }
    if (int rc = image_norms(T, T->ju)) return rc;
    image_unit<<<nblocks(npx), 256, 0, s>>>(T->ju, T->jn2, plane, d.B, T->jv);
    PNP_CHECK_LAUNCH();
  }
  return PNP_OK;
}

// Adam on the accumulated gradients, then the BF16 operands are re-packed
int adam_update(pnp_cnn_trainer* T) {
  T->t += 1;
  const float c1 = (float)(1.0 - std::pow(T->b1, T->t)), c2 = (float)(1.0 - std::pow(T->b2, T->t));
  adam_step<<<nblocks(NPARAM), 256, 0, T->stream>>>(T->w, T->g, T->m, T->v, NPARAM, (float)T->lr, (float)T->b1,
                                                    (float)T->b2, (float)(1.0 - T->b1), (float)(1.0 - T->b2),
                                                    (float)T->eps, c1, c2);
  PNP_CHECK_LAUNCH();
  return prep(T);
}
}  // namespace

extern "C" {

int pnp_cnn_trainer_create(pnp_cnn_trainer** out, const float* weights_host, int batch, int size, double lr,
                           void* stream) {
  if (!out || !weights_host || batch < 1 || size < 8 || !(lr > 0)) return fail(PNP_ERR_INVALID_ARG, "bad argument");
  *out = nullptr;
  pnp_cnn_trainer* T = new pnp_cnn_trainer();
  T->stream = reinterpret_cast<cudaStream_t>(stream);
  T->lr = lr;
  T->d = Dims{batch, size, size, (size + 127) / 128 * 128};
  if (int rc = device_sms(&T->sms)) {
    delete T;
    return rc;
  }
  // a CTA per SM, and at least four image rows each
  T->parts = (int)std::max<int64_t>(1, std::min<int64_t>(T->sms, (int64_t)batch * ((size + WGT_PX - 1) / WGT_PX) * size / 4));
  const size_t canvas = (size_t)batch * T->d.Hc * T->d.Wc * CH;
  const int64_t npx = (int64_t)batch * size * size;
  auto al = [&](void** p, size_t bytes) -> bool {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return true;
  };
  bool ok = al((void**)&T->w, NPARAM * 4) && al((void**)&T->g, NPARAM * 4) && al((void**)&T->m, NPARAM * 4) &&
            al((void**)&T->v, NPARAM * 4) && al((void**)&T->w1r, NW1 * 4) && al((void**)&T->w8r, NW8 * 4) &&
            al((void**)&T->bias, 8 * CH * 4) && al((void**)&T->wf, 6 * (size_t)NWM * 2) &&
            al((void**)&T->wb, 6 * (size_t)NWM * 2) && al((void**)&T->z, npx * 4) && al((void**)&T->gout, npx * 4) &&
            al((void**)&T->facets, batch * sizeof(int4)) && al((void**)&T->loss, sizeof(double)) &&
            al((void**)&T->status, 4 * sizeof(int)) && al((void**)&T->jv, npx * 4) && al((void**)&T->jw, npx * 4) &&
            al((void**)&T->ju, npx * 4) && al((void**)&T->jn2, batch * sizeof(double)) &&
            al((void**)&T->junk, CH * sizeof(float)) && al((void**)&T->part, (size_t)T->parts * WGT_SUMS * sizeof(float));
  for (int i = 1; ok && i <= 7; ++i) ok = al((void**)&T->act[i], canvas * 2);
  for (int i = 0; ok && i < 2; ++i) ok = al((void**)&T->dp[i], canvas * 2);
  for (int i = 1; ok && i <= 7; ++i) ok = al((void**)&T->tan[i], canvas * 2);
  std::vector<int4> facets(batch, make_int4(0, 0, size, size));
  const std::vector<int> sides(batch, size);
  const std::vector<int4> strips = conv_strips(batch, sides.data(), sides.data(), T->sms, &T->conv_grid);
  T->n_strips = (int)strips.size();
  ok = ok && al((void**)&T->strips, strips.size() * sizeof(int4));
  if (!ok) {
    trainer_free(T);
    return fail(PNP_ERR_OOM, "trainer allocation failed");
  }
  cudaError_t e = cudaMemcpy(T->w, weights_host, NPARAM * 4, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(T->g, 0, NPARAM * 4);
  if (e == cudaSuccess) e = cudaMemset(T->m, 0, NPARAM * 4);
  if (e == cudaSuccess) e = cudaMemset(T->v, 0, NPARAM * 4);
  if (e == cudaSuccess) e = cudaMemset(T->status, 0, 4 * sizeof(int));
  for (int i = 1; e == cudaSuccess && i <= 7; ++i) e = cudaMemset(T->act[i], 0, canvas * 2);
  for (int i = 0; e == cudaSuccess && i < 2; ++i) e = cudaMemset(T->dp[i], 0, canvas * 2);
  for (int i = 1; e == cudaSuccess && i <= 7; ++i) e = cudaMemset(T->tan[i], 0, canvas * 2);
  if (e == cudaSuccess) e = cudaMemcpy(T->facets, facets.data(), batch * sizeof(int4), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(T->strips, strips.data(), strips.size() * sizeof(int4), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaGetLastError();
    trainer_free(T);
    return fail(PNP_ERR_CUDA, std::string("trainer set-up: ") + cudaGetErrorString(e));
  }
  for (int i = 1; i <= 7; ++i)
    if (int rc = canvas_map_create(T->map_act[i], T->act[i], batch, T->d.Hc, T->d.Wc)) {
      trainer_free(T);
      return rc;
    }
  for (int i = 0; i < 2; ++i)
    if (int rc = canvas_map_create(T->map_dp[i], T->dp[i], batch, T->d.Hc, T->d.Wc)) {
      trainer_free(T);
      return rc;
    }
  for (int i = 1; i <= 6; ++i)
    if (int rc = canvas_map_create(T->map_tan[i], T->tan[i], batch, T->d.Hc, T->d.Wc)) {
      trainer_free(T);
      return rc;
    }
  if (int rc = prep(T)) {
    trainer_free(T);
    return rc;
  }
  *out = T;
  return PNP_OK;
}

void pnp_cnn_trainer_destroy(pnp_cnn_trainer* T) {
  if (T) cudaStreamSynchronize(T->stream);
  trainer_free(T);
}

int pnp_cnn_train_step(pnp_cnn_trainer* T, const float* u, const float* noise, double sigma, int update,
                       double* loss_host) {
  if (!T || !u || !noise || !(sigma >= 0)) return fail(PNP_ERR_INVALID_ARG, "bad argument");
  const Dims d = T->d;
  const int64_t npx = (int64_t)d.B * d.s * d.s;
  cudaStream_t s = T->stream;
  // ---------------- forward
  make_z<<<nblocks(npx), 256, 0, s>>>(u, noise, (float)sigma, T->z, npx);
  PNP_CHECK_LAUNCH();
  if (int rc = cnn_first_launch(s, T->z, d.s, (int64_t)d.s * d.s, T->facets, d.B, d.Hc, d.Wc, T->w1r, T->bias,
                                T->act[1]))
    return rc;
  for (int k = 1; k <= 6; ++k)
    if (int rc = conv64_launch(s, T->map_act[k], T->act[k + 1], T->wf + (size_t)(k - 1) * NWM, T->bias + k * CH,
                               T->strips, T->n_strips, T->conv_grid, d.Hc, d.Wc, 0, nullptr, T->status))
      return rc;
  PNP_CUDA(cudaMemsetAsync(T->loss, 0, sizeof(double), s));
  if (int rc = many_to_one_launch<M2O_LOSS, false>(s, d, T->sms, T->act[7], T->w8r, 1, T->bias, T->z, u, T->gout, T->loss))
    return rc;
  // ---------------- backward
  if (int rc = layer8_back(T, T->gout)) return rc;
  if (int rc = onechannel_grads<true>(T, T->gout, T->act[7], T->g + OFF_W8, T->g + OFF_B8)) return rc;
  int cur = 0;
  for (int k = 6; k >= 1; --k) {
    float* gW = T->g + OFF_MID + (k - 1) * MID_STRIDE;
    if (int rc = wgrad64_launch(s, d, T->dp[cur], T->act[k], T->part, T->parts, gW, gW + NWM)) return rc;
    if (int rc = conv64_launch(s, T->map_dp[cur], T->dp[1 - cur], T->wb + (size_t)(k - 1) * NWM, nullptr,
                               T->strips, T->n_strips, T->conv_grid, d.Hc, d.Wc, 1, T->act[k], T->status))
      return rc;
    cur = 1 - cur;
  }
  if (int rc = onechannel_grads<false>(T, T->z, T->dp[cur], T->g + OFF_W1, T->g + OFF_B1)) return rc;
  // ---------------- update
  if (update)
    if (int rc = adam_update(T)) return rc;
  if (loss_host) {
    PNP_CUDA(cudaMemcpyAsync(loss_host, T->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    PNP_CUDA(cudaStreamSynchronize(s));
  }
  return PNP_OK;
}

int pnp_cnn_jacobian_norm(pnp_cnn_trainer* T, const float* z, const float* v0, int iters, double* sigma_host,
                          float* v_out) {
  if (!T || !z || !v0 || iters < 1 || iters > 100000 || !sigma_host) return fail(PNP_ERR_INVALID_ARG, "bad argument");
  const Dims d = T->d;
  const int64_t npx = (int64_t)d.s * d.s * d.B;
  if (int rc = primal_forward(T, z)) return rc;  // fixes the ReLU masks
  if (int rc = power_iterate(T, v0, iters, sigma_host)) return rc;
  if (v_out) PNP_CUDA(cudaMemcpyAsync(v_out, T->jv, npx * sizeof(float), cudaMemcpyDeviceToDevice, T->stream));
  PNP_CUDA(cudaStreamSynchronize(T->stream));
  return PNP_OK;
}

int pnp_cnn_train_step_fne(pnp_cnn_trainer* T, const float* u, const float* noise, double sigma, const float* v0,
                           int iters, double lambda, double eps, int update, double* loss_host,
                           double* penalty_host) {
  if (!T || !u || !noise || !v0 || !(sigma >= 0) || iters < 0 || iters > 100000 || !(lambda >= 0) ||
      !std::isfinite(lambda) || !(eps >= 0) || !(eps <= 1))
    return fail(PNP_ERR_INVALID_ARG, "bad argument");
  const Dims d = T->d;
  const int64_t plane = (int64_t)d.s * d.s, npx = plane * d.B;
  cudaStream_t s = T->stream;
  // the l1 term: forward at z = u + sigma n (activations kept), gradients accumulated, no update
  if (int rc = pnp_cnn_train_step(T, u, noise, sigma, 0, loss_host)) return rc;
  // v: the leading right singular vector of J_Q at z, by power iteration (iters = 0: v0 itself)
  if (iters > 0) {
    if (int rc = power_iterate(T, v0, iters, nullptr)) return rc;
  } else {
    if (int rc = image_norms(T, v0)) return rc;
    image_unit<<<nblocks(npx), 256, 0, s>>>(v0, T->jn2, plane, d.B, T->jv);
    PNP_CHECK_LAUNCH();
  }
  // w = J_Q v with every tangent kept for the weight gradients
  if (int rc = layer1_tangent(T, T->jv, T->tan[1])) return rc;
  for (int k = 1; k <= 6; ++k)
    if (int rc = conv64_launch(s, T->map_tan[k], T->tan[k + 1], T->wf + (size_t)(k - 1) * NWM, nullptr, T->strips,
                               T->n_strips, T->conv_grid, d.Hc, d.Wc, 1, T->act[k + 1], T->status))
      return rc;
  if (int rc = many_to_one_launch<M2O_JAC, false>(s, d, T->sms, T->tan[7], T->w8r, 1, nullptr, T->jv, nullptr, T->jw, nullptr))
    return rc;
  if (int rc = image_norms(T, T->jw)) return rc;
  fne_cotangent<<<nblocks(npx), 256, 0, s>>>(T->jw, T->jn2, plane, d.B, (float)(lambda / d.B), 1.0 - eps, T->gout);
  PNP_CHECK_LAUNCH();
  // back-propagation of the cotangent through the tangent network (no bias gradients)
  if (int rc = onechannel_grads<true>(T, T->gout, T->tan[7], T->g + OFF_W8, T->junk)) return rc;
  if (int rc = layer8_back(T, T->gout)) return rc;
  int cur = 0;
  for (int k = 6; k >= 1; --k) {
    if (int rc = wgrad64_launch(s, d, T->dp[cur], T->tan[k], T->part, T->parts,
                                T->g + OFF_MID + (k - 1) * MID_STRIDE, T->junk))
      return rc;
    if (int rc = conv64_launch(s, T->map_dp[cur], T->dp[1 - cur], T->wb + (size_t)(k - 1) * NWM, nullptr, T->strips,
                               T->n_strips, T->conv_grid, d.Hc, d.Wc, 1, T->act[k], T->status))
      return rc;
    cur = 1 - cur;
  }
  if (int rc = onechannel_grads<false>(T, T->jv, T->dp[cur], T->g + OFF_W1, T->junk)) return rc;
  if (penalty_host) {
    std::vector<double> n2(d.B);
    PNP_CUDA(cudaMemcpyAsync(n2.data(), T->jn2, d.B * sizeof(double), cudaMemcpyDeviceToHost, s));
    PNP_CUDA(cudaStreamSynchronize(s));
    double P = 0.0;
    for (double q : n2) P += lambda / d.B * std::max(q, 1.0 - eps);
    *penalty_host = P;
  }
  if (update) return adam_update(T);
  return PNP_OK;
}

int pnp_cnn_trainer_read(pnp_cnn_trainer* T, float* weights_host, float* grads_host, int clear_grads) {
  if (!T) return fail(PNP_ERR_INVALID_ARG, "NULL trainer");
  PNP_CUDA(cudaStreamSynchronize(T->stream));
  if (weights_host) PNP_CUDA(cudaMemcpy(weights_host, T->w, NPARAM * 4, cudaMemcpyDeviceToHost));
  if (grads_host) PNP_CUDA(cudaMemcpy(grads_host, T->g, NPARAM * 4, cudaMemcpyDeviceToHost));
  if (clear_grads) {
    zero_f<<<nblocks(NPARAM), 256, 0, T->stream>>>(T->g, NPARAM);
    PNP_CHECK_LAUNCH();
  }
  int st = 0;
  PNP_CUDA(cudaMemcpy(&st, T->status, sizeof(int), cudaMemcpyDeviceToHost));
  if (st) return fail(PNP_ERR_TIMEOUT, "a bounded wait in the tensor-core convolution gave up");
  return PNP_OK;
}

int pnp_cnn_trainer_apply_update(pnp_cnn_trainer* T) {
  if (!T) return fail(PNP_ERR_INVALID_ARG, "NULL trainer");
  return adam_update(T);
}

int pnp_cnn_trainer_set_lr(pnp_cnn_trainer* T, double lr) {
  if (!T || !(lr > 0)) return fail(PNP_ERR_INVALID_ARG, "bad argument");
  T->lr = lr;
  return PNP_OK;
}

int64_t pnp_cnn_num_params(void) { return NPARAM; }

}  // extern "C"
