// Per-head kernels of decode attention (Table alg:kvrobin step 8; App. G): the query
// projection ahead of the scan of decode.cuh (optionally fused with the K-side append of one
// new token, step 7, and carrying the V-side append's CTAs in the same launch) and the
// combine + back-projection after it.
#pragma once

#include <type_traits>

#include "compress.cuh"
#include "decode.cuh"

namespace cobra {

// ---------------------------------------------------------------------------------------
// Per-head kernels: the query projection has one CTA of 256 threads per (layer, kv head) and run
// of sequences, 32 query vectors per pass, with the head's basis staged in shared memory once; the
// combine has one per (layer, kv head) and one or two sequences.  The workspace's head-group table
// gives the group of (head, seq).
// ---------------------------------------------------------------------------------------
constexpr int kHeadThreads = 256;
constexpr int kVecPass = 32;  // query vectors (sequences x G) per pass
static_assert(kVecPass + kVecPass / 4 <= kProjVecs, "a pass holds its queries and their sequences' new tokens");
constexpr int kWtChunk = 64;  // chunk weights held in shared memory per vector and round

// ---------------------------------------------------------------------------------------
// a4: query projection
//   q~_g = (Delta_K / sqrt d) log2(e) W_K^T q_g per query head, scaled by a power of two so
//   that max |q~| of the group lands in [256, 512), split into fp16 hi + lo and laid out as
//   the scan's MMA B fragments; Qsum_g = sum over channels of the fed hi + lo values.
//   With ak.x set, the CTA also appends the new K tokens of its sequences (a8), which project
//   through the same staged W_K: they are further vectors of the same projection.  With av.x set,
//   the grid has a second half of CTAs (blockIdx.x >= n_qblocks) that append the new V tokens of
//   the same runs of sequences, so that both appends and the projection run in one launch.
//
//   A latency kernel: a chain of dependent loads (plan, head table, basis), then short phases.
//   The sequences of a head are spread over n_split CTAs when the heads alone leave SMs idle
//   (see proj_split), and every phase uses all eight warps whatever the number of vectors.  A warp's
//   vectors are worked on together and the q~ blocks' addresses looked up once per pass: with one
//   vector at a time and a look-up per stored fragment, 32 layers of 8 heads and 64 sequences took
//   156 us with the appends and 108 without, now 141 and 96.
// ---------------------------------------------------------------------------------------
static_assert(kAppendThreads == kHeadThreads, "the V append runs in the query projection's CTAs");
template <int G>
__global__ void __launch_bounds__(kHeadThreads, 2) qproj_kernel(DecodeArgs a, CompressArgs ak, CompressArgs av,
                                                             int n_qblocks, int n_split, int spb) {
  extern __shared__ __align__(16) float qsm[];
  grid_dep_launch();
  const int blk = (int)blockIdx.x % n_qblocks, head = blk / n_split;
  const int seq0 = (blk % n_split) * spb;
  if ((int)blockIdx.x >= n_qblocks) {
    append_block(av, head, seq0, min(av.n_seqs, seq0 + spb), qsm);
    return;
  }
  constexpr int NTK = Heads<G>::NTK, SPP = kVecPass / G;
  __shared__ float amax_s[kVecPass], up_s[SPP];
  __shared__ unsigned char* qt_s[SPP];  // the q~ blocks of the pass's sequences
  const ProjSmem sm(qsm);
  const WsHeader* wh = reinterpret_cast<const WsHeader*>(a.ws);
  const WsGroup* groups = reinterpret_cast<const WsGroup*>(a.ws + wh->groups_off);
  const int S = wh->n_seqs;
  const int* hg = reinterpret_cast<const int*>(a.ws + wh->hg_off) + (size_t)head * S;
  const WsGroup g0 = groups[hg[0]];
  const HeadEntry hk = head_table(a.block)[g0.k_head];
  const int r = hk.r, layer = g0.layer, kv = g0.kv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int seq1 = min(S, seq0 + spb);
  const float scale = hk.delta * 0.088388347648318440f * 1.4426950408889634f;  // Delta/sqrt(128)*log2(e)
  // the basis is a parameter: its copy overlaps the end of the kernel ahead; the queries, the
  // new tokens, the cache and the q~ blocks of the workspace are touched only after the wait
  const bool append = ak.x != nullptr && r > 0;
  proj_stage_issue(sm, param_pool(a.block), hk);
  int grp = tid < min(SPP, seq1 - seq0) ? hg[seq0 + tid] : 0;  // thread i: group of the pass's sequence i
  grid_dep_wait();
  const bool wide =
      ((reinterpret_cast<uintptr_t>(a.q) | (uintptr_t)(2 * a.q_sl) | (uintptr_t)(2 * a.q_ss)) & 15) == 0 &&
      (!append || append_wide(ak));
  const __nv_bfloat16* q = a.q + layer * a.q_sl + (long long)(kv * G) * kD;
  const __nv_bfloat16* x = append ? ak.x + layer * ak.sl + kv * ak.sh : nullptr;
  for (int s0 = seq0; s0 < seq1; s0 += SPP) {
    const int ns = min(SPP, seq1 - s0), nq = ns * G, nv = nq + (append ? ns : 0);
    // vectors: the queries of the pass's sequences, then their new tokens
    proj_load(
        nv, wide,
        [&](int v) {
          return v < nq ? q + (long long)(s0 + v / G) * a.q_ss + (v % G) * kD : x + (long long)(s0 + v - nq) * ak.ss;
        },
        sm.Xs);
    if (append && tid < ns) sm.pos[tid] = ak.pos[s0 + tid];
    if (tid < ns) qt_s[tid] = a.ws + wh->qt_off + (size_t)grp * wh->qt_stride;
    if (tid < min(SPP, seq1 - s0 - SPP)) grp = hg[s0 + SPP + tid];
    cp_async_wait_all();
    __syncthreads();  // basis and vectors staged
    project(sm, nv, r);
    __syncthreads();
    if (append) append_codes(ak, hk, sm, nq, s0, ns);
    // a warp's query vectors vw .. vw + nw - 1, worked on together.  In a full pass of 4 query heads
    // these are one sequence's, and the warps need not wait for one another.
    const int vpw = (nq + kProjWarps - 1) / kProjWarps, vw = warp * vpw, nw = min(vpw, nq - vw);
    const bool own = vpw == G;
    auto sync = [&] {
      if (own)
        __syncwarp();
      else
        __syncthreads();
    };
    auto scales = [&](auto nu) {
      constexpr int NU = decltype(nu)::value;  // vectors per warp at most
      // largest |q~| of each vector
      const float* o = sm.Os + vw * kProjLd;
      float red[NU] = {};
#pragma unroll 1
      for (int i = lane; i < r; i += 32)
#pragma unroll
        for (int u = 0; u < NU; ++u)
          if (u < nw) red[u] = fmaxf(red[u], fabsf(o[u * kProjLd + i] * scale));
#pragma unroll
      for (int m = 16; m; m >>= 1)
#pragma unroll
        for (int u = 0; u < NU; ++u) red[u] = fmaxf(red[u], __shfl_xor_sync(0xffffffffu, red[u], m));
#pragma unroll
      for (int u = 0; u < NU; ++u)
        if (u < nw && lane == u) amax_s[vw + u] = red[u];
      sync();
      // the power-of-two scale of each vector's group (lane u: of vector vw + u), Qsum of the hi/lo split
      float up_l = 1.f, down_l = 1.f;
      if (lane < nw) {
        const float* am = amax_s + (vw + lane) / G * G;
        float amax = 0.f;
#pragma unroll
        for (int k = 0; k < G; ++k) amax = fmaxf(amax, am[k]);
        int e = 0;
        if (amax > 0.f) {
          int ex;
          frexpf(amax, &ex);  // amax = m 2^ex, m in [0.5, 1)
          e = 9 - ex;
        }
        up_l = ldexpf(1.f, e);
        down_l = ldexpf(1.f, -e);
      }
      float up[NU];
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        up[u] = __shfl_sync(0xffffffffu, up_l, u);
        red[u] = 0.f;
      }
#pragma unroll 1
      for (int i = lane; i < r; i += 32)
#pragma unroll
        for (int u = 0; u < NU; ++u)
          if (u < nw) {
            const float y = o[u * kProjLd + i] * scale * up[u];
            const __half h = __float2half_rn(y);
            const __half l = __float2half_rn(y - __half2float(h));
            red[u] += __half2float(h) + __half2float(l);
          }
#pragma unroll
      for (int m = 16; m; m >>= 1)
#pragma unroll
        for (int u = 0; u < NU; ++u) red[u] += __shfl_xor_sync(0xffffffffu, red[u], m);
#pragma unroll
      for (int u = 0; u < NU; ++u)
        if (u < nw && lane == u) {
          const int sl = (vw + u) / G, g = (vw + u) % G;
          float* qhdr = reinterpret_cast<float*>(qt_s[sl]);
          qhdr[g] = red[u];
          if (g == 0) {
            qhdr[8] = down_l;
            up_s[sl] = up_l;
          }
        }
    };
    if (vpw == 1)  // few sequences: the short way through
      scales(std::integral_constant<int, 1>{});
    else
      scales(std::integral_constant<int, kVecPass / kProjWarps>{});
    sync();
    // element (k, n) of fragment (kappa, nt) = hi or lo part of q~ of channel 16 kappa + k
    // for the query head of column n (see Heads)
    const int f0 = own ? 256 * NTK * warp + lane : tid, f1 = 256 * NTK * (own ? min(warp + 1, ns) : ns);
    for (int idx = f0; idx < f1; idx += own ? 32 : kHeadThreads) {
      const int fl = idx & 31, nt = (idx >> 5) % NTK, kap = (idx / (32 * NTK)) & 7, sl = idx / (256 * NTK);
      const int j = fl & 3, n = fl >> 2;
      const int g = Heads<G>::col_head(nt, n), lo = Heads<G>::col_lo(nt, n);
      const float* og = sm.Os + (sl * G + g) * kProjLd;
      const float ups = up_s[sl];
      float e4[4];
      const int ks[4] = {2 * j, 2 * j + 1, 2 * j + 8, 2 * j + 9};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ch = 16 * kap + ks[u];
        float v = 0.f;
        if (ch < r) {
          const float y = og[ch] * scale * ups;
          const float h = __half2float(__float2half_rn(y));
          v = lo ? (y - h) : h;
        }
        e4[u] = v;
      }
      reinterpret_cast<uint2*>(qt_s[sl] + kQtHeaderBytes)[(kap * NTK + nt) * 32 + fl] =
          make_uint2(pack_f16(e4[0], e4[1]), pack_f16(e4[2], e4[3]));
    }
    __syncthreads();  // Os, pos, the scales and the block addresses are rewritten by the next pass
  }
}

// ---------------------------------------------------------------------------------------
// a7: combine chunks + back-projection
//   per query head: m* = max over chunks, l* = sum 2^(m - m*) l, zbar = Delta_V (sum 2^(m - m*)
//   acc / l* - 2^{b-1} + 1/2), o = mu_V + W_V zbar (zeros for an empty sequence).
//
// One CTA of 256 threads per (layer, kv head) and run of NS sequences.  The kernel is a chain of
// memory round trips (chunk maxima, chunk sums, the rows of W_V), so every phase spreads its loads
// over all threads and issues them together; a head's W_V is read again for each run (from L2).
// Two forms (combine_many), us alone, against 20, 33.5 and 112 with one CTA per head and run of 16
// query vectors, for 32 layers x 8 heads of 4 query heads and 8, 16 and 64 sequences:
//   kCombineFew   one sequence, 3 CTAs per SM, eight loads in flight per thread: the most CTAs for a
//                 call, 24, 47 and 185.  A step over 1 layer x 8 kv heads takes 23 us for 25.9 (1 x 2048
//                 tokens), 50 for 67 (24 ragged sequences at 3 bpd) and 63 for 80 (8 x 32768).
//   kCombineMany  runs of 8 query vectors, 4 CTAs per SM, four loads in flight: the most sequences at a
//                 time, 17, 30 and 108.
// ---------------------------------------------------------------------------------------
constexpr int kCombineFew = 3, kCombineMany = 4;  // resident CTAs per SM
template <int G, int NS, int CTAS>
__global__ void __launch_bounds__(kHeadThreads, CTAS) combine_kernel(DecodeArgs a) {
  constexpr int UB = CTAS == kCombineMany ? 4 : 8;  // loads in flight per thread
  constexpr int V = G * NS;  // query vectors of the CTA: vector v = query head v % G of sequence s0 + v / G
  static_assert(V <= kHeadThreads / 32, "a warp per vector");
  __shared__ float wts[V][kWtChunk];          // weights 2^(m_k - m*) / l* of a round of chunks
  __shared__ float m_s[V], inv_l_s[V];
  __shared__ __align__(16) float red[kHeadThreads * 4];  // partial chunk sums, then zbar [channel][V]
  const WsHeader* wh = reinterpret_cast<const WsHeader*>(a.ws);
  const WsGroup* groups = reinterpret_cast<const WsGroup*>(a.ws + wh->groups_off);
  const float* parts = reinterpret_cast<const float*>(a.ws + wh->part_off);
  const int S = wh->n_seqs, pstride = wh->part_stride, gstride = wh->g_stride;
  const int runs = (S + NS - 1) / NS, s0 = (int)(blockIdx.x % runs) * NS;
  const int* hg = reinterpret_cast<const int*>(a.ws + wh->hg_off) + (size_t)(blockIdx.x / runs) * S;
  const WsGroup g0 = groups[hg[s0]], g1 = groups[hg[min(s0 + NS, S) - 1]];  // (NS <= 2)
  const HeadEntry hv = head_table(a.block)[g0.v_head];
  const float* pool = param_pool(a.block);
  const int rv = hv.r, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* W = pool + hv.w_off;
  // W_V is pulled into L2 here, while the scan ahead of this kernel is still finishing (the first
  // run's CTA of a head does it for all)
  if (s0 == 0)
    for (int idx = tid; idx < rv * (kD / 32); idx += kHeadThreads) prefetch_l2(W + 32 * idx);
  const int d0 = 16 * warp + 4 * (lane & 3);  // dims of the back-projection: d0 .. d0 + 3
  float mu_a[4];
  const float* mu = pool + hv.mu_off + d0;
  if (hv.mu_off % 4 == 0) {
    const float4 m4 = *reinterpret_cast<const float4*>(mu);
    mu_a[0] = m4.x, mu_a[1] = m4.y, mu_a[2] = m4.z, mu_a[3] = m4.w;
  } else {  // (another tool's block)
#pragma unroll
    for (int k = 0; k < 4; ++k) mu_a[k] = mu[k];
  }
  // the appends of the next step may start their parameter staging meanwhile
  grid_dep_launch();
  // everything above is independent of the scan; its partials are read only from here on
  grid_dep_wait();
  const int n0 = a.seq_lens[g0.seq] > 0 ? g0.n_items : 0;
  const int n1 = NS > 1 && s0 + 1 < S && a.seq_lens[g1.seq] > 0 ? g1.n_items : 0, nmax = max(n0, n1);
  // chunks of a vector's sequence, and the first one's partial
  auto chunks = [&](int v) { return NS == 1 || v < G ? n0 : n1; };
  auto first = [&](int v) {
    return parts + (size_t)(NS == 1 || v < G ? g0 : g1).first_item * pstride + (v % G) * gstride;
  };
  // (1) warp v: m* and l* of vector v, lanes over chunks, merged online (a chunk with no tokens
  //     has m = -inf and no value entries; its weight is zero).  The m of the first kWtChunk chunks
  //     stay in shared memory and become the weights of the first round of (2).
  if (warp < V) {
    const float* pg = first(warp);
    const int n = chunks(warp);
    float M = -INFINITY, Ls = 0.f;
    for (int k = lane; k < n; k += 32) {
      const float mk = pg[(size_t)k * pstride], lk = pg[(size_t)k * pstride + 1];
      if (k < kWtChunk) wts[warp][k] = mk;
      if (mk == -INFINITY) continue;
      const float mn = fmaxf(M, mk);
      Ls = Ls * exp2f(M - mn) + lk * exp2f(mk - mn);
      M = mn;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const float mo = __shfl_xor_sync(0xffffffffu, M, o), lo = __shfl_xor_sync(0xffffffffu, Ls, o);
      const float mn = fmaxf(M, mo);
      if (mn != -INFINITY) {
        Ls = Ls * exp2f(M - mn) + lo * exp2f(mo - mn);
        M = mn;
      }
    }
    const float inv_l = n > 0 ? 1.f / Ls : 0.f;
    if (lane == 0) {
      m_s[warp] = M;
      inv_l_s[warp] = inv_l;
    }
    // the same lane wrote wts[..][k] above for k < n
    for (int k = lane; k < min(n, kWtChunk); k += 32) {
      const float mk = wts[warp][k];
      wts[warp][k] = mk != -INFINITY ? exp2f(mk - M) * inv_l : 0.f;
    }
  }
  __syncthreads();
  // (2) weighted chunk sums: thread (channel quad cq, vector v, chunk share p) of rw = r_V
  //     rounded up to 32, 64 or 128 channels sums 16-byte entries of chunks p, p + np, ..., UB loads
  //     in flight; the shares are added through shared memory.
  const int rw = rv <= 32 ? 32 : rv <= 64 ? 64 : kD;
  const int nq = rw / 4, np = kHeadThreads / (nq * V);  // np >= 1 (V = 8, rw = 128)
  {
    const int cq = tid % nq, v = (tid / nq) % V, p = tid / (nq * V), n = chunks(v);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = 0; k0 < nmax; k0 += kWtChunk) {
      if (k0 > 0) {  // later rounds: one weight per thread into shared memory
        __syncthreads();
        for (int idx = tid; idx < V * kWtChunk; idx += kHeadThreads) {
          const int vw = idx / kWtChunk, k = k0 + idx % kWtChunk;
          float w = 0.f;
          if (k < chunks(vw)) {
            const float mk = first(vw)[(size_t)k * pstride];
            if (mk != -INFINITY) w = exp2f(mk - m_s[vw]) * inv_l_s[vw];
          }
          wts[vw][idx % kWtChunk] = w;
        }
        __syncthreads();
      }
      if (4 * cq >= rv) continue;
      // the partial's channels start 4 floats in and every stride is a multiple of 4 floats
      const float4* px = reinterpret_cast<const float4*>(first(v) + (size_t)k0 * pstride + 4 + 4 * cq);
      const int kr = min(kWtChunk, n - k0);
      for (int kb = p; kb < kr; kb += UB * np) {
        float4 x[UB];
        float w[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int k = kb + u * np;
          w[u] = k < kr ? wts[v][k] : 0.f;
          // an empty chunk's value entries were never written
          x[u] = w[u] != 0.f ? px[(size_t)k * (pstride / 4)] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          acc.x += w[u] * x[u].x;
          acc.y += w[u] * x[u].y;
          acc.z += w[u] * x[u].z;
          acc.w += w[u] * x[u].w;
        }
      }
    }
    *reinterpret_cast<float4*>(red + 4 * tid) = acc;
  }
  __syncthreads();
  // zbar = Delta (sum_k w_k acc_k - 2^{b-1} + 1/2), written back as [channel][V]
  {
    const float cen = rv > 0 ? (float)(1 << (hv.b - 1)) - 0.5f : 0.f;
    float z[V / 2];  // at most V rw / 256 <= V / 2 values per thread
#pragma unroll
    for (int u = 0; u < V / 2; ++u) {
      const int idx = tid + u * kHeadThreads;  // v rw + channel
      float sum = 0.f;
      if (idx < V * rw)
        for (int p = 0; p < np; ++p) sum += red[p * V * rw + idx];
      z[u] = chunks(idx / rw) > 0 ? hv.delta * (sum - cen) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < V / 2; ++u) {
      const int idx = tid + u * kHeadThreads;
      if (idx < V * rw) red[(idx % rw) * V + idx / rw] = z[u];
    }
  }
  __syncthreads();
  // (3) o = mu_V + W_V zbar: a warp has 16 dims, its lanes 4 dims x every eighth row of W_V (UB
  //     16-byte loads in flight); the eight row shares are added by halving exchanges, after which
  //     a lane holds V / 2 consecutive outputs.
  float o[4 * V];
#pragma unroll
  for (int k = 0; k < 4 * V; ++k) o[k] = 0.f;
  const int sl = lane >> 2;
  const float4* W4 = reinterpret_cast<const float4*>(W + d0);
  for (int i0 = sl; i0 < rv; i0 += 8 * UB) {
    float4 w[UB];
#pragma unroll
    for (int u = 0; u < UB; ++u)
      w[u] = i0 + 8 * u < rv ? __ldg(W4 + (i0 + 8 * u) * (kD / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      // rows past r_V have w = 0; their zbar is finite (zeros, or within rw <= 128 rows)
      const float* zr = red + (i0 + 8 * u < rv ? i0 + 8 * u : 0) * V;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float zz = zr[v];
        o[4 * v + 0] += w[u].x * zz;
        o[4 * v + 1] += w[u].y * zz;
        o[4 * v + 2] += w[u].z * zz;
        o[4 * v + 3] += w[u].w * zz;
      }
    }
  }
#pragma unroll
  for (int st = 0; st < 3; ++st) {
    const int half = (4 * V) >> (st + 1), bit = 16 >> st;
    const bool up = lane & bit;
#pragma unroll
    for (int k = 0; k < (4 * V) >> 1; ++k) {
      if (k < half) {
        const float send = up ? o[k] : o[half + k], keep = up ? o[half + k] : o[k];
        o[k] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
      }
    }
  }
  // lane share sl holds outputs [sl V / 2, (sl + 1) V / 2) of the 4 V (vector, dim) values: 2 or 4
  // consecutive dims c0 .. of vector v, which leave in one store where the output's rows are aligned
  // (it may be host memory, where every store costs: a step that writes 4 MB there by element took
  // 0.84 ms for 0.77)
  const int v = sl * (V / 2) >> 2, c0 = sl * (V / 2) & 3;
  const WsGroup& gr = NS == 1 || v < G ? g0 : g1;
  if (NS > 1 && v >= G && s0 + 1 >= S) return;
  float* dst = a.out + gr.layer * a.o_sl + gr.seq * a.o_ss + (long long)(gr.kv * G + v % G) * kD + d0 + c0;
  const bool wide = ((reinterpret_cast<uintptr_t>(a.out) | (uintptr_t)(4 * a.o_sl) | (uintptr_t)(4 * a.o_ss)) & 15) == 0;
  float res[V / 2];
#pragma unroll
  for (int k = 0; k < V / 2; ++k) {
    const float muk = (V == 8) ? mu_a[k & 3] : ((sl & 1) ? mu_a[2 + k] : mu_a[k]);
    res[k] = chunks(v) > 0 ? muk + o[k] : 0.f;
  }
  if (!wide) {  // 4-byte aligned in general
#pragma unroll
    for (int k = 0; k < V / 2; ++k) dst[k] = res[k];
  } else if constexpr (V == 8) {
    *reinterpret_cast<float4*>(dst) = make_float4(res[0], res[1], res[2], res[3]);
  } else {
    *reinterpret_cast<float2*>(dst) = make_float2(res[0], res[1]);
  }
}

}  // namespace cobra
