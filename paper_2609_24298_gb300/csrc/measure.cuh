// Measured per-head distortion tables (App. E, "Exact DP over measured distortion").
//
// For every head, its calibration tokens go through the deployed quantizer once per candidate
// (r, b) and the reconstruction error is measured in the allocator's units:
//   D(r, b) = (1/N) sum_t sum_k omega_k (u_k . (x_t - x^_t))^2,
// omega_k = 1 (MSE objective) or sigma_Q,k^2 (attention-KL objective).  In the eigen
// coordinates c = U^T (x - mu) the error splits exactly into the energy past r,
// sum_{k >= r} omega_k c_k^2, and the quantisation error of the kept coordinates rotated back,
// H_r^T (y - y^) with y = H_r c_r (W = U_r H_r^T, so W^T (x - mu) = H_r c_r).
//
//   coords_kernel   c = (x - mu) U per head, fp32, by the shared-memory projection of compress.cuh
//                   (one CTA per head and 128 tokens).
//   measure_kernel  one CTA per (head, r): four lanes per token, 32 coordinates each, run the block
//                   Walsh-Hadamard transform y = H_r c_r (blocks of the binary digits of r, largest
//                   first, signs on the columns) by butterflies, then for every b the codes, the
//                   error y - y^, its transform back and the weighted sum.
//
// Bound: instruction issue (no memory traffic to speak of).  The lane split keeps five of the seven
// butterfly distances in registers (two are shuffles) and only the first r coordinates, in groups
// of 16, are computed at all.  256 heads x 512 tokens x 65 ranks x 8 widths with KL weights: 5.5 ms
// (3.8 G warp-instructions, 0.57 of the issue slots), against 19.3 ms with one warp per token (every
// distance below 32 a shuffle, all 128 coordinates whatever r).
#pragma once

#include "compress.cuh"

namespace cobra {

constexpr int kMeasureMaxR = 65;  // candidate ranks per call
constexpr int kMeasureMaxB = 16;  // candidate bit widths per call

struct MeasureArgs {
  const float* x;        // [n_heads][n_tok][kD] calibration tokens
  const float* U;        // [n_heads][kD * kD] basis, column k = u_k (allocator order)
  const double* lam;     // [n_heads][kD] eigenvalues in the same order
  const double* w;       // [n_heads][kD] allocator weights in the same order (lambda or sigma_Q^2 lambda)
  const float* mu;       // [n_heads][kD]
  const int8_t* signs;   // [n_heads][kD] Hadamard column signs
  float* coords;         // [n_heads][n_tok][kD] workspace: c = (x - mu) U
  double* D;             // [n_heads][n_r][n_b]
  int n_tok, n_r, n_b;
  int r[kMeasureMaxR];
  int b[kMeasureMaxB];
  double L[kMeasureMaxB];  // loading factor of b[j]
};

// c = (x - mu) U for up to kCoordTok tokens of one head per CTA, 32 at a time.
constexpr int kCoordTok = 128;
__global__ void __launch_bounds__(kAppendThreads, 2) coords_kernel(MeasureArgs a) {
  extern __shared__ __align__(16) float cosm[];
  const ProjSmem sm(cosm);
  const int h = blockIdx.y, tid = threadIdx.x;
  const int t0 = blockIdx.x * kCoordTok, t1 = min(a.n_tok, t0 + kCoordTok);
  const float* U = a.U + (size_t)h * kD * kD;  // only 4-byte aligned in general
#pragma unroll 16
  for (int idx = tid; idx < kD * kD; idx += kAppendThreads) sm.Ws[(idx >> 7) * kProjLd + (idx & 127)] = U[idx];
  const float m = a.mu[(size_t)h * kD + (tid & 127)];
  for (int s0 = t0; s0 < t1; s0 += 32) {
    const int nt = min(32, t1 - s0);
    const float* x = a.x + ((size_t)h * a.n_tok + s0) * kD;
#pragma unroll 16
    for (int idx = tid; idx < nt * kD; idx += kAppendThreads) sm.Xs[idx] = x[idx] - m;  // idx % 128 = tid % 128
    __syncthreads();
    project(sm, nt, kD);
    __syncthreads();
    float* c = a.coords + ((size_t)h * a.n_tok + s0) * kD;
    for (int idx = tid; idx < nt * kD; idx += kAppendThreads) c[idx] = sm.Os[(idx >> 7) * kProjLd + (idx & 127)];
  }
}

// Coordinate k of a token sits in lane (k / 4) % 4 of its four lanes, register 4 (k / 16) + k % 4:
// distances 1, 2, 16, 32 and 64 pair registers, 4 and 8 pair lanes.  The butterfly of distance d
// acts on the coordinates in blocks of at least 2 d elements, the first r & ~(2 d - 1) ones.
struct WhtLane {
  int r, sub;      // sub: lane % 4
  float s4, s8;    // +1 in the lane with the lower index of the pair, -1 in the other
};

// distances 1 to 8 within the 16-coordinate group v (all of it inside blocks of 16 or more)
__device__ __forceinline__ void wht_full16(float* v, const WhtLane& w) {
  const float a0 = v[0] + v[1], a1 = v[0] - v[1], a2 = v[2] + v[3], a3 = v[2] - v[3];
  v[0] = a0 + a2;
  v[2] = a0 - a2;
  v[1] = a1 + a3;
  v[3] = a1 - a3;
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = fmaf(w.s4, v[i], __shfl_xor_sync(0xffffffffu, v[i], 1));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = fmaf(w.s8, v[i], __shfl_xor_sync(0xffffffffu, v[i], 2));
}
// the same for the last group, of which only the first t = r % 16 coordinates are kept
__device__ __forceinline__ void wht_tail16(float* v, const WhtLane& w, int t) {
  const int k = 4 * w.sub;
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    const float a = v[i] + v[i + 1], b = v[i] - v[i + 1];
    const bool on = k + i < (t & ~1);
    v[i] = on ? a : v[i];
    v[i + 1] = on ? b : v[i + 1];
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float a = v[i] + v[i + 2], b = v[i] - v[i + 2];
    const bool on = k < (t & ~3);
    v[i] = on ? a : v[i];
    v[i + 2] = on ? b : v[i + 2];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float o = fmaf(w.s4, v[i], __shfl_xor_sync(0xffffffffu, v[i], 1));
    v[i] = (k & 8) < (t & ~7) ? o : v[i];
  }
}
__device__ __forceinline__ void wht_pairs(float* v, float* u) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = v[i] + u[i], b = v[i] - u[i];
    v[i] = a;
    u[i] = b;
  }
}
// distances 16, 32 and 64 over the groups
__device__ __forceinline__ void wht_groups(float (&v)[32], int r) {
#pragma unroll
  for (int m = 0; m < 8; m += 2)
    if (16 * m + 32 <= r) wht_pairs(v + 4 * m, v + 4 * m + 4);
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (64 * q + 64 <= r) {
      wht_pairs(v + 16 * q, v + 16 * q + 8);
      wht_pairs(v + 16 * q + 4, v + 16 * q + 12);
    }
  if (r == kD) {
#pragma unroll
    for (int m = 0; m < 4; ++m) wht_pairs(v + 4 * m, v + 16 + 4 * m);
  }
}

// size of the Hadamard block that holds coordinate k of r (0 past r)
__device__ __forceinline__ int hadamard_block(int r, int k) {
  int o = 0;
  for (int p = 7; p >= 0; --p)
    if (r & (1 << p)) {
      if (k < o + (1 << p)) return 1 << p;
      o += 1 << p;
    }
  return 0;
}

constexpr int kMeasureThreads = 256;
constexpr float kMeasureMagic = 12582912.0f;  // 1.5 * 2^23: fp32 spacing 1

// Quantisation error of y at one width: s = u 2^-b saturated, then floor(u) by rounding the sum with
// kMeasureMagic down (exact: its spacing is 1), clamped at the top; u = y / Delta + 2^{b-1}.
struct MeasureQuant {
  float il, scale, top, back, dl;  // il 2^-b, 2^b, magic + 2^b - 1, 2^{b-1} - 1/2, Delta
  __device__ __forceinline__ float error(float y) const {
    const float s = __saturatef(fmaf(y, il, 0.5f));
    const float t = fminf(__fmaf_rd(s, scale, kMeasureMagic), top);
    // (a code may differ from the exact division's at a cell boundary, where both cells leave an
    // error of the same size)
    return fmaf(-dl, (t - kMeasureMagic) - back, y);
  }
};

__global__ void __launch_bounds__(kMeasureThreads, 2) measure_kernel(MeasureArgs a) {
  const int h = blockIdx.y, ri = a.n_r - 1 - (int)blockIdx.x;  // the largest ranks first
  const int r = a.r[ri];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // per coordinate: Hadamard sign, 1 / sqrt(block), error weight (past r), error weight / block size
  __shared__ __align__(16) float fwd[kD], inv[kD], om[kD], ob[kD];
  __shared__ MeasureQuant quant[kMeasureMaxB];
  __shared__ float accs[kMeasureMaxB][kMeasureThreads];
  __shared__ double red[kMeasureThreads / 32][kMeasureMaxB + 1];
  const double* lam = a.lam + (size_t)h * kD;
  int nonunit = 0;
  if (tid < kD) {
    const int size = hadamard_block(r, tid);
    // error weight omega_k = w_k / lambda_k: 1 for the MSE objective, sigma_Q,k^2 for attention-KL
    const float w = lam[tid] > 0.0 ? (float)(a.w[(size_t)h * kD + tid] / lam[tid]) : 0.f;
    fwd[tid] = size > 0 ? (float)a.signs[(size_t)h * kD + tid] : 0.f;
    inv[tid] = size > 0 ? rsqrtf((float)size) : 0.f;
    om[tid] = w;
    ob[tid] = size > 0 ? w / (float)size : 0.f;
    nonunit = w != 1.f;
  }
  if (tid < a.n_b) {
    // Delta per b, as the stored fp32 step: 2 L_b sigma_bar / 2^b, sigma_bar^2 = mean lambda_{<r}
    double lsum = 0.0;
    for (int k = 0; k < r; ++k) lsum += lam[k];
    const double sigma = r > 0 ? sqrt(lsum / r) : 0.0;
    const int b = a.b[tid];
    const float dl = (float)(2.0 * a.L[tid] * sigma / (double)(1 << b));
    const float scale = (float)(1 << b);
    quant[tid] = MeasureQuant{(dl > 0.f ? 1.f / dl : 0.f) / scale, scale, kMeasureMagic + scale - 1.f, 0.5f * scale - 0.5f, dl};
  }
  // with unit weights (the MSE objective) the rotation back preserves the norm: the error is
  // summed in the rotated coordinates and the second transform is skipped
  const bool unit_w = !__syncthreads_or(nonunit);
  WhtLane w;
  w.r = r;
  w.sub = lane & 3;
  w.s4 = (lane & 1) ? -1.f : 1.f;
  w.s8 = (lane & 2) ? -1.f : 1.f;
  const int tail = r & 15, ng = (r + 15) >> 4;  // groups that hold kept coordinates
  for (int j = 0; j < a.n_b; ++j) accs[j][tid] = 0.f;
  float acc_trunc = 0.f;
  // every lane of a warp runs the same number of rounds (the shuffles need them all)
  for (int t0 = 8 * warp; t0 < a.n_tok; t0 += kMeasureThreads / 4) {
    const bool live = t0 + (lane >> 2) < a.n_tok;
    const float* c = a.coords + ((size_t)h * a.n_tok + min(t0 + (lane >> 2), a.n_tok - 1)) * kD + 4 * w.sub;
    float y[32], trunc = 0.f;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      float cv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) cv[i] = live ? c[16 * m + i] : 0.f;
      if (16 * m + 16 > r) {  // energy past r
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (16 * m + 4 * w.sub + i >= r) trunc = fmaf(om[16 * m + 4 * w.sub + i] * cv[i], cv[i], trunc);
      }
      const float4 f = *reinterpret_cast<const float4*>(fwd + 16 * m + 4 * w.sub);
      y[4 * m + 0] = cv[0] * f.x;
      y[4 * m + 1] = cv[1] * f.y;
      y[4 * m + 2] = cv[2] * f.z;
      y[4 * m + 3] = cv[3] * f.w;
    }
    acc_trunc += trunc;
    if (r == 0) continue;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      if (16 * m + 16 <= r)
        wht_full16(y + 4 * m, w);
      else if (16 * m < r)
        wht_tail16(y + 4 * m, w, tail);
    }
    wht_groups(y, r);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const float4 f = *reinterpret_cast<const float4*>(inv + 16 * m + 4 * w.sub);
      y[4 * m + 0] *= f.x;
      y[4 * m + 1] *= f.y;
      y[4 * m + 2] *= f.z;
      y[4 * m + 3] *= f.w;
    }
#pragma unroll 1
    for (int j = 0; j < a.n_b; ++j) {
      const MeasureQuant qz = quant[j];
      float sum[2] = {0.f, 0.f};
      if (unit_w) {
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          if (m >= ng) break;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float e = qz.error(y[4 * m + i]);
            if (16 * m + 16 > r && 16 * m + 4 * w.sub + i >= r) e = 0.f;
            sum[i & 1] = fmaf(e, e, sum[i & 1]);
          }
        }
      } else {
        // back to the eigen coordinates: H_r^T = diag(s) blockdiag(H_n / sqrt n) (H_n symmetric)
        float e[32];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          if (16 * m + 16 <= r) {
#pragma unroll
            for (int i = 0; i < 4; ++i) e[4 * m + i] = qz.error(y[4 * m + i]);
            wht_full16(e + 4 * m, w);
          } else if (16 * m < r) {
#pragma unroll
            for (int i = 0; i < 4; ++i) e[4 * m + i] = 4 * w.sub + i < tail ? qz.error(y[4 * m + i]) : 0.f;
            wht_tail16(e + 4 * m, w, tail);
          }
        }
        wht_groups(e, r);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          if (m >= ng) break;
          const float4 o = *reinterpret_cast<const float4*>(ob + 16 * m + 4 * w.sub);
          sum[0] = fmaf(o.x * e[4 * m + 0], e[4 * m + 0], sum[0]);
          sum[1] = fmaf(o.y * e[4 * m + 1], e[4 * m + 1], sum[1]);
          sum[0] = fmaf(o.z * e[4 * m + 2], e[4 * m + 2], sum[0]);
          sum[1] = fmaf(o.w * e[4 * m + 3], e[4 * m + 3], sum[1]);
        }
      }
      if (live) accs[j][tid] += sum[0] + sum[1];
    }
  }
  // reduce over the warp, then over the warps in fp64
#pragma unroll
  for (int o = 16; o; o >>= 1) acc_trunc += __shfl_xor_sync(0xffffffffu, acc_trunc, o);
  if (lane == 0) red[warp][kMeasureMaxB] = acc_trunc;
  for (int j = 0; j < a.n_b; ++j) {
    float v = accs[j][tid];
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][j] = v;
  }
  __syncthreads();
  if (tid < a.n_b) {
    double tr = 0.0, kept = 0.0;
    for (int k = 0; k < kMeasureThreads / 32; ++k) {
      tr += red[k][kMeasureMaxB];
      kept += red[k][tid];
    }
    a.D[((size_t)h * a.n_r + ri) * a.n_b + tid] = (tr + kept) / (double)a.n_tok;
  }
}

}  // namespace cobra
