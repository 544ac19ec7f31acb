// The compress kernels' arguments, the projection that the append shares with the query
// projection, and the single-token append (Table alg:kvrobin step 7): y = W^T (x - mu), the fused
// projection + Hadamard as one multiply (Sec. 3.4), code = clamp(floor(y / Delta + 2^{b-1}), 0,
// 2^b - 1), in code rows of format v1 (include/cobra.h).
//
// append_kernel    one CTA per (layer, kv head) and run of sequences: projects the new tokens in
//                  fp32 on CUDA cores and ORs their codes into the rows (other tokens' bits
//                  untouched).
// The bulk compress over 128-token tiles runs on the tensor cores (compress_tc.cuh).
#pragma once

#include "common.cuh"

namespace cobra {

struct CompressArgs {
  const unsigned char* block;
  const __nv_bfloat16* x;
  unsigned char* cache;
  const int* page_table;
  const int* pos;
  long long sl, ss, st, sh;
  int head0, layer_stride, n_layers, n_kv, side, n_seqs, rows_per_seq, pages_per_seq;
  int t0, n_tok;
};

__device__ __forceinline__ uint32_t pack_bf16(float lo_col, float hi_col) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo_col, hi_col);
  return *reinterpret_cast<uint32_t*>(&h);
}

// a8: single-token append, and the projection it shares with the query projection (qproj_kernel):
// both need O[v][i] = sum_d W[i][d] X[v][d] for a few vectors v of a head.  One CTA of 256 threads
// stages the head's basis in shared memory once (row stride kProjLd floats, so that a warp's
// 16-byte row reads are conflict-free) and its warps share out (4 vectors) x (32, 64 or 128
// channels) units, so that one sequence's vectors keep every warp busy as well as 32 vectors do.
// Each output is summed over d in the same order whatever the split: the codes do not depend on it.
constexpr int kAppendThreads = 256;
constexpr int kProjWarps = kAppendThreads / 32;
constexpr int kProjLd = 132;
constexpr int kProjVecs = 40;  // vectors per pass (32 queries and the new tokens of their sequences)
__host__ __device__ constexpr size_t proj_smem_bytes() {
  return sizeof(float) * ((size_t)kD * kProjLd + (size_t)kProjVecs * kD + (size_t)kProjVecs * kProjLd + kD + kProjVecs);
}
// the shared memory of a projecting CTA
struct ProjSmem {
  float* Ws;   // [kD][kProjLd] basis row i = channel i (rows past r are not written)
  float* Xs;   // [kProjVecs][kD] vectors of this pass
  float* Os;   // [kProjVecs][kProjLd] their projections
  float* wmu;  // [kD] W^T mu
  int* pos;    // [kProjVecs] positions of the pass's new tokens
  __device__ explicit ProjSmem(float* base)
      : Ws(base), Xs(Ws + kD * kProjLd), Os(Xs + kProjVecs * kD), wmu(Os + kProjVecs * kProjLd),
        pos(reinterpret_cast<int*>(wmu + kD)) {}
};

// nv vectors of 128 bf16 into Xs; row(v) is vector v's address.  `wide`: every row is 16-byte
// aligned (in general they are only 2-byte aligned).
template <typename Row>
__device__ __forceinline__ void proj_load(int nv, bool wide, Row row, float* Xs) {
  if (wide) {
#pragma unroll 3
    for (int idx = threadIdx.x; idx < nv * (kD / 8); idx += kAppendThreads) {
      const int v = idx / (kD / 8), c = idx % (kD / 8);
      const uint4 u = reinterpret_cast<const uint4*>(row(v))[c];
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
      float f[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        f[2 * k] = __uint_as_float(w[k] << 16);
        f[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
      }
      float4* o = reinterpret_cast<float4*>(Xs + v * kD + 8 * c);
      o[0] = make_float4(f[0], f[1], f[2], f[3]);
      o[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
  } else {
#pragma unroll 16
    for (int idx = threadIdx.x; idx < nv * kD; idx += kAppendThreads) Xs[idx] = __bfloat162float(row(idx / kD)[idx % kD]);
  }
}

// A warp's unit: vectors 4 vg .. 4 vg + 3 times CB blocks of 32 channels from block cb.  Rows of
// Ws past r hold anything; their results are not stored.
template <int CB>
__device__ __forceinline__ void proj_unit(const ProjSmem& sm, int vg, int cb, int nv, int r) {
  const int lane = threadIdx.x & 31;
  float acc[CB][4];
#pragma unroll
  for (int c = 0; c < CB; ++c)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[c][v] = 0.f;
  const float* Wp = sm.Ws + (lane + 32 * cb) * kProjLd;
  const float* Xp = sm.Xs + 4 * vg * kD;
#pragma unroll 4
  for (int d = 0; d < kD; d += 4) {
    float4 w[CB], x[4];
#pragma unroll
    for (int c = 0; c < CB; ++c) w[c] = *reinterpret_cast<const float4*>(Wp + 32 * c * kProjLd + d);
#pragma unroll
    for (int v = 0; v < 4; ++v) x[v] = *reinterpret_cast<const float4*>(Xp + v * kD + d);
#pragma unroll
    for (int c = 0; c < CB; ++c)
#pragma unroll
      for (int v = 0; v < 4; ++v)
        acc[c][v] += w[c].x * x[v].x + w[c].y * x[v].y + w[c].z * x[v].z + w[c].w * x[v].w;
  }
#pragma unroll
  for (int c = 0; c < CB; ++c) {
    const int ch = lane + 32 * (cb + c);
    if (ch >= r) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (4 * vg + v < nv) sm.Os[(4 * vg + v) * kProjLd + ch] = acc[c][v];
  }
}
// Os <- projections of the nv vectors in Xs on the r channels.  Wider units read each basis value
// for more vectors' worth of work per shared-memory access; they are used once there are enough
// of them for the 8 warps, and no wider than the head's channels.
template <int CB>
__device__ __forceinline__ void proj_units(const ProjSmem& sm, int nv, int r) {
  const int ng = (nv + 3) >> 2, nc = ((r + 31) / 32 + CB - 1) / CB;
  for (int u = threadIdx.x >> 5; u < ng * nc; u += kProjWarps) proj_unit<CB>(sm, u / nc, CB * (u % nc), nv, r);
}
__device__ __forceinline__ void project(const ProjSmem& sm, int nv, int r) {
  const int units = ((nv + 3) >> 2) * ((r + 31) / 32);
  if (units <= kProjWarps)
    proj_units<1>(sm, nv, r);
  else if (units <= 2 * kProjWarps || r <= 64)
    proj_units<2>(sm, nv, r);
  else
    proj_units<4>(sm, nv, r);
}

// Issues the copies of a head's W^T mu and basis rows [0, r) (parameters: this may run before the
// wait for the kernel ahead).  The caller waits with cp_async_wait_all and synchronises the block.
// W^T mu is r floats; the pool is padded to 32 floats, so whole 16-byte chunks stay in it.
__device__ __forceinline__ void proj_stage_issue(const ProjSmem& sm, const float* pool, const HeadEntry& he) {
  const int tid = threadIdx.x;
  if (tid < (he.r + 3) / 4) cp_async16(smem_addr(sm.wmu + 4 * tid), pool + he.wmu_off + 4 * tid);
  const float* W = pool + he.w_off;
  for (int idx = tid; idx < he.r * (kD / 4); idx += kAppendThreads)
    cp_async16(smem_addr(sm.Ws + (idx >> 5) * kProjLd + 4 * (idx & 31)), W + (size_t)idx * 4);
}

// Every row of the new tokens is 16-byte aligned.
__device__ __forceinline__ bool append_wide(const CompressArgs& a) {
  return ((reinterpret_cast<uintptr_t>(a.x) | (uintptr_t)(2 * a.sl) | (uintptr_t)(2 * a.ss) | (uintptr_t)(2 * a.sh)) & 15) == 0;
}

// Quantises the projections of the new tokens of sequences seq0 .. seq0 + ns - 1 (rows v0 .. of
// Os) and writes their codes: y = W^T x - W^T mu, codes into the token's bits of its row with
// atomics (the row's other tokens are untouched).
__device__ __forceinline__ void append_codes(const CompressArgs& a, const HeadEntry& he, const ProjSmem& sm, int v0,
                                             int seq0, int ns) {
  const int r = he.r, b = he.b;
  const uint32_t rb = 16u * r * b;
  const float inv_delta = he.inv_delta, half = (float)(1 << (b - 1));
  const int cmax = (1 << b) - 1;
  for (int idx = threadIdx.x; idx < ns * kD; idx += kAppendThreads) {
    const int v = idx / kD, i = idx % kD, seq = seq0 + v;
    if (i >= r) continue;
    const int p = sm.pos[v], row = p >> 7, tt = p & 127;
    const bool in_range = p >= 0 && (a.page_table ? (row >> 1) < a.pages_per_seq : row < a.rows_per_seq);
    if (!in_range) {  // a position past the cache's capacity is never written
      if (i == 0) atomicOr(&g_status, 2u);
      continue;
    }
    uint8_t* rowp = a.cache + row_offset(he.cache_off, rb, seq, row, a.page_table, a.pages_per_seq, a.rows_per_seq);
    const int tau = tt >> 4, t16 = tt & 15, rho = 2 * tau + (t16 >> 3);
    const float y = sm.Os[(v0 + v) * kProjLd + i] - sm.wmu[i];
    int code = (int)floorf(fmaf(y, inv_delta, half));
    code = code < 0 ? 0 : (code > cmax ? cmax : code);
    int piece, h;
    if (a.side == 0) {
      piece = t16 & 7;
      h = i & 1;
    } else {
      piece = 4 * (i & 1) + ((t16 >> 1) & 3);
      h = t16 & 1;
    }
    uint32_t* words = reinterpret_cast<uint32_t*>(rowp + (i >> 1) * 32 * b + piece * 4 * b);
    const int x0 = rho * b;
    const int w0 = x0 >> 4, o0 = x0 & 15;
    const int n0 = min(b, 16 - o0);
    const uint32_t m0 = ((1u << n0) - 1u) << (16 * h + o0);
    atomicAnd(words + w0, ~m0);
    atomicOr(words + w0, ((uint32_t)code << (16 * h + o0)) & m0);
    if (n0 < b) {
      const uint32_t m1 = ((1u << (b - n0)) - 1u) << (16 * h);
      atomicAnd(words + w0 + 1, ~m1);
      atomicOr(words + w0 + 1, ((uint32_t)code >> n0) << (16 * h) & m1);
    }
  }
}

// The append of sequences [seq0, seq1) of (layer, kv head) number `blk` by one CTA of
// kAppendThreads threads, with proj_smem_bytes() of shared memory at `base`.  Run by append_kernel
// and, in the decode step, by the V-side CTAs of the query projection's launch.
__device__ __forceinline__ void append_block(const CompressArgs& a, int blk, int seq0, int seq1, float* base) {
  const ProjSmem sm(base);
  const int layer = blk / a.n_kv, kv = blk % a.n_kv;
  const HeadEntry he = head_table(a.block)[a.head0 + layer * a.layer_stride + kv];
  if (he.r == 0) {
    grid_dep_wait();
    return;
  }
  proj_stage_issue(sm, param_pool(a.block), he);
  // the tokens, positions and the cache may be produced or read by the kernels ahead
  grid_dep_wait();
  const bool wide = append_wide(a);
  const __nv_bfloat16* x = a.x + layer * a.sl + kv * a.sh;
  for (int s0 = seq0; s0 < seq1; s0 += kProjVecs) {
    const int ns = min(kProjVecs, seq1 - s0);
    proj_load(ns, wide, [&](int v) { return x + (long long)(s0 + v) * a.ss; }, sm.Xs);
    if (threadIdx.x < ns) sm.pos[threadIdx.x] = a.pos[s0 + threadIdx.x];
    cp_async_wait_all();
    __syncthreads();
    project(sm, ns, he.r);
    __syncthreads();
    append_codes(a, he, sm, 0, s0, ns);
    __syncthreads();  // pos and Os are rewritten by the next pass
  }
}

// grid: (layer, kv head) x splits of the sequences, `spb` sequences each
__global__ void __launch_bounds__(kAppendThreads) append_kernel(CompressArgs a, int n_split, int spb) {
  extern __shared__ __align__(16) float apsm[];
  grid_dep_launch();
  const int s0 = (int)(blockIdx.x % n_split) * spb;
  append_block(a, blockIdx.x / n_split, s0, min(a.n_seqs, s0 + spb), apsm);
}

}  // namespace cobra
