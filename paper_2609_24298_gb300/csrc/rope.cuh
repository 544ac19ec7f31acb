// Decode attention for models with the rotary position embedding (RoPE).
//
// The paper compresses K before the rotation (Sec. 5, "Scope"; App. "Post-RoPE experiments":
// after it the per-head covariance depends on the position), so such a model attends with
// every reconstructed key turned to its own position t and the query to its position p:
//   s_t = <R(p) q, R(t) K^_t> / sqrt(d),   K^_t = mu_K + W_K Delta_K (c_t - 2^{b-1} + 1/2),
// R(x) turning channel pair (j, j + d/2) by the angle x omega_j, omega_j = theta^(-2j/d).
// R(t) differs per token, so W_K cannot be folded into one projected query as in the rank-
// space scan of decode.cuh: each key is rebuilt in the d-dimensional space on the tensor
// cores, turned, and scored.
//
//   rope_table_kernel  cos and sin of x omega_j in fp64, for x = i < 16 (fine rows) and
//                      x = 16 m (coarse rows); any position x = 16 m + i composes from one of
//                      each by the angle-addition formulas.
//   rope_scan_kernel   CTAs of one to three warpgroups, each with a warp that issues its MMAs and
//                      copies, take runs of the decode plan's chunks; a warpgroup takes every other
//                      128-token row of a run.  Per row, with thread t owning token t (TMEM lane t):
//                        unpack   the token's codes, as f16, into TMEM (the MMAs' A operand)
//                        rebuild  X = A W' + mu'/Delta by tcgen05.mma (W' = W_K^T, f16 hi + lo, in
//                                 shared memory; fp32 accumulators in TMEM)
//                        turn     by R(t): t = 128 row + tau, and R(128 row) is applied to the
//                                 query instead, so a thread's angles (of tau) never change
//                        score    in fp32 on the CUDA cores
//                      then the online softmax, and the rank-space accumulation of V (not rotated)
//                      on mma.sync with the probabilities shared through shared memory.
//   combine_kernel     (decode_heads.cuh) as for the plain decode.
//
// Operands.  A code c goes into the A operand as the f16 value c - (2^{b-1} - 1/2), exact for any
// width: the code's bits in 512 + c (whose spacing is 1/2) less 512 + 2^{b-1} - 1/2.  mu'/Delta comes
// from three f16 limbs against a block of constant A columns, so X = K^'/Delta with no offset to
// cancel; the factor Delta / sqrt(d) is in the query.  A head with r_K = 0 has X = mu' (Delta taken
// as 1).  Column P = 4 (j / 2) + 2 e + j % 2 of X holds model channel j + e d/2, so a thread reads the
// halves of two channel pairs as four neighbours.
//
// Bound: the CUDA cores and shared memory, 6 + 3 G instructions per token and two channel pairs (the
// angles' load, the turn in packed fp32 pairs, per query head one broadcast load and two packed
// fused multiply-adds).  With 8 or 12 warps per SM the latencies between the steps count: X is kept in two
// halves of 64 columns, so that the next row's MMAs run on the half that has been read while the
// warps score the other one and accumulate the values.  4 layers x 8 kv heads x 8 x 32768 tokens at
// 1 bpd: 0.92 to 0.94 ms per call, against 1.80 with the rebuild and the scores on mma.sync (hi + lo of
// every operand, one warp per row); 1 layer x 8 heads x 8191 tokens at 2 bpd: 33 to 35 us, against 390-450
// with one CTA per (sequence, layer, kv head).
#pragma once

#include "compress_tc.cuh"
#include "decode.cuh"

namespace cobra {

constexpr int kRopeFine = 16;         // positions per coarse step (fine rows 0..15)
constexpr int kRopeRowFloats = 128;   // floats per table row: [jj 4][n 16][cos, sin]
// Warpgroups (128 threads and an issuing warp) per CTA at most.  Three cap a thread at 128 registers,
// which 4 query heads fit but for a few spills: calls of many rows gain from the third warpgroup (4
// layers x 8 heads x 8 x 32768 tokens at 1 bpd: 943 against 998 us), short ones lose more to the cap
// (34.8 against 32.5 us for 1 x 8191) and use the build with two; 8 query heads always do.
constexpr int kRopeMaxWg = 3;
// A raised reference lies this far below the maximum, so that fewer of the small probabilities fall
// into fp16's subnormals (fed values stay below 2^kTau).
constexpr float kRopeLift = 4.f;

// Table entry of pair j = 4 n + jj within a row: [(jj * 16 + n) * 2 + (0: cos, 1: sin)].
__host__ __device__ constexpr int rope_entry(int j) { return ((j & 3) * 16 + (j >> 2)) * 2; }

__host__ __device__ constexpr size_t rope_table_floats(int n_coarse) {
  return (size_t)(kRopeFine + n_coarse) * kRopeRowFloats;
}

struct RopeArgs {
  const float* table;  // [kRopeFine + n_coarse][kRopeRowFloats]
  const int* q_pos;    // [n_seqs] query positions, or null: seq_len - 1
  int n_coarse;        // positions < 16 n_coarse are covered
  int stage_bytes;     // one stage: channel tiles of a K row + a V row
  int n_stage;         // stages per warpgroup (1 or 2)
  int batch;           // plan chunks taken at a time
};

// Shared memory of a CTA: W' hi (128 positions x up to 144 channels: three 64-channel swizzle
// atoms) and lo (two atoms), the angles of the row's tokens, then per-warpgroup buffers.
constexpr int kRopeAtomBytes = 16384;
constexpr int kRopeWBytes = 5 * kRopeAtomBytes;
constexpr int kRopeTrigBytes = 32 * 128 * 16;
constexpr int kRopePLd = kD + 8;  // halves per query head of a probability buffer
template <int G>
struct RopeWgSmem {
  float4 q[2][32 * G];          // the query turned by -128 row: [j / 2][g] (a0, a1, b0, b1)
  __half p[2][G * kRopePLd];    // fed probabilities [g][token]
  float wmax[4][G];             // row maxima of the four warps
  float cl[2][G], cle[2][G];    // the constant rows' sums c and l, and their rounding errors
  int fail[4];                  // per warp: a wait has expired
  // K stage full [2], V stage full [2], X half full [2] (MMA commits); A written and X half 0 read,
  // X half 1 read (one arrival per warp)
  unsigned long long bars[8];
};
template <int G>
struct RopeSmem {
  float4 qbase[32 * G];         // R(p) q, scaled
  float merge[kRopeMaxWg - 1][G][4 + kD];  // m, l, -, -, O of the warpgroups after the first
  uint32_t tmem;
  int batch, fail;
  alignas(16) RopeWgSmem<G> wg[1];  // one per warpgroup
};
template <int G>
__host__ __device__ constexpr size_t rope_vars_bytes(int nwg) {
  return (sizeof(RopeSmem<G>) + (nwg - 1) * sizeof(RopeWgSmem<G>) + 127) / 128 * 128;
}
template <int G>
__host__ __device__ constexpr size_t rope_fixed_bytes(int nwg) {
  return 1024 + kRopeWBytes + kRopeTrigBytes + rope_vars_bytes<G>(nwg);
}

// (cos, sin) of x omega_j for x = 16 m + i from the coarse (m) and fine (i) entries
__device__ __forceinline__ void rope_compose(float cm, float sm, float ci, float si, float& c, float& s) {
  c = fmaf(cm, ci, -sm * si);
  s = fmaf(sm, ci, cm * si);
}

// two fp32 operations at a time
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// ---------------------------------------------------------------------------------------
// Angle tables: row x < 16 holds position x, row 16 + m position 16 m (fp64 angles, rounded
// once to fp32).
// ---------------------------------------------------------------------------------------
__global__ void rope_table_kernel(float* table, int n_rows, double theta) {
  // an earlier decode may still read the table being overwritten
  grid_dep_wait();
  grid_dep_launch();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_rows * (kD / 2)) return;
  const int x = idx / (kD / 2), j = idx % (kD / 2);
  const double pos = x < kRopeFine ? (double)x : 16.0 * (double)(x - kRopeFine);
  const double om = pow(theta, -2.0 * (double)j / (double)kD);
  double s, c;
  sincos(pos * om, &s, &c);
  float* e = table + (size_t)x * kRopeRowFloats + rope_entry(j);
  e[0] = (float)c;
  e[1] = (float)s;
}

// ---------------------------------------------------------------------------------------
// Instruction descriptor, kind::f16 with f16 A and B, fp32 D, both K-major, M = 128, N = 64.
constexpr uint32_t kRopeIdesc = (1u << 4) | ((64u >> 3) << 17) | ((128u >> 4) << 24);

// 8 consecutive TMEM columns of the warp's 32 lanes: column (taddr + j) of this lane = v[j]
__device__ __forceinline__ void tc_st32x8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// named barrier of a warpgroup, and the same returning whether `p` holds in any of its threads
__device__ __forceinline__ void wg_sync(int wg) { asm volatile("bar.sync %0, 128;" ::"r"(1 + wg) : "memory"); }
__device__ __forceinline__ bool wg_any(int wg, bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %1, 0;\n bar.red.or.pred q, %2, 128, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((int)p), "r"(1 + wg)
      : "memory");
  return r != 0;
}

// The codes of token t of a K row into the A operand: TMEM lane t, column s = channels (2 s, 2 s + 1),
// nk tiles of 8 columns.  Codes of strips past the row are whatever the buffer holds (finite, against
// zero columns of W').  The rotation brings the code to mantissa bit 1; what wraps around is masked.
template <int B>
__device__ __forceinline__ void rope_unpack(const uint8_t* krow, int nk, int t, uint32_t a_tmem) {
  const int p = t & 7, rho = 2 * (t >> 4) + ((t >> 3) & 1);
  const int wi = (rho * B) >> 4, off = (rho * B) & 15, nlo = min(B, 16 - off), rot = (off + 31) & 31;
  const uint32_t m0 = (((1u << nlo) - 1u) << 1) * 0x00010001u;
  const uint32_t m1 = ((((1u << B) - 1u) & ~((1u << nlo) - 1u)) << 1) * 0x00010001u;
  const __half2 cen = __float2half2_rn(512.f + (float)(1 << (B - 1)) - 0.5f);
  const uint8_t* src = krow + p * 4 * B + 4 * wi;
  const int next = wi + 1 < B ? 4 : 0;
#pragma unroll 2
  for (int kt = 0; kt < nk; ++kt) {
    uint32_t v[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const uint8_t* w = src + (8 * kt + s) * 32 * B;
      const uint32_t x = *reinterpret_cast<const uint32_t*>(w);
      uint32_t c = (__funnelshift_r(x, x, rot) & m0) | 0x60006000u;
      if constexpr (16 % B != 0)  // a code may straddle two words
        c |= (*reinterpret_cast<const uint32_t*>(w + next) << (nlo + 1)) & m1;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&c), cen);
      v[s] = *reinterpret_cast<const uint32_t*>(&h);
    }
    tc_st32x8(a_tmem + 8 * kt, v);
  }
}
__device__ __forceinline__ void rope_unpack_dispatch(int b, const uint8_t* krow, int nk, int t, uint32_t a_tmem) {
  switch (b) {
    case 1: rope_unpack<1>(krow, nk, t, a_tmem); break;
    case 2: rope_unpack<2>(krow, nk, t, a_tmem); break;
    case 3: rope_unpack<3>(krow, nk, t, a_tmem); break;
    case 4: rope_unpack<4>(krow, nk, t, a_tmem); break;
    case 5: rope_unpack<5>(krow, nk, t, a_tmem); break;
    case 6: rope_unpack<6>(krow, nk, t, a_tmem); break;
    case 7: rope_unpack<7>(krow, nk, t, a_tmem); break;
    default: rope_unpack<8>(krow, nk, t, a_tmem); break;
  }
}

// Adds half of the thread's scores against the G query heads (log2 units): the 64 columns of X at
// x_tmem, turned by the token's angles (trig[j / 2][t]: c0, c1, s0, s1), dotted with the row's query.
template <int G>
__device__ __forceinline__ void rope_scores32(const uint32_t (&x)[32], const float4* trig_t, const float4* q,
                                              f32x2 (&acc)[2 * G]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float4 tr = trig_t[k * 128];
    const float a0 = __uint_as_float(x[4 * k]), a1 = __uint_as_float(x[4 * k + 1]);
    const f32x2 a = pack2(a0, a1), b = pack2(__uint_as_float(x[4 * k + 2]), __uint_as_float(x[4 * k + 3]));
    const f32x2 c2 = pack2(tr.x, tr.y), s2 = pack2(tr.z, tr.w);
    const float2 bs = unpack2(mul2(b, s2));
    const f32x2 ka = pack2(fmaf(a0, tr.x, -bs.x), fmaf(a1, tr.y, -bs.y));
    const f32x2 kb = fma2(a, s2, mul2(b, c2));
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float4 qq = q[k * G + g];
      acc[2 * g] = fma2(pack2(qq.x, qq.y), ka, acc[2 * g]);
      acc[2 * g + 1] = fma2(pack2(qq.z, qq.w), kb, acc[2 * g + 1]);
    }
  }
}
template <int G>
__device__ __forceinline__ void rope_scores_half(uint32_t x_tmem, const float4* trig_t, const float4* q,
                                                 f32x2 (&acc)[2 * G]) {
  uint32_t x0[32], x1[32];
  tc_ld32(x_tmem, x0);
  tc_wait_ld(x0);
  tc_ld32(x_tmem + 32, x1);  // in flight while the first half is scored
  rope_scores32<G>(x0, trig_t, q, acc);
  tc_wait_ld(x1);
  rope_scores32<G>(x1, trig_t + 8 * 128, q + 8 * G, acc);
}

// Running sums with the rounding errors of their additions kept beside them (o + e is the sum): the
// sums are dominated by the unit code offsets, and a stretch may run over hundreds of rows.
template <int NO>
struct RopeAcc {
  float o[3][NO], e[3][NO];
  __device__ __forceinline__ void add(int i, int k, float d) {
    const float t = o[i][k] + d;
    e[i][k] += d - (t - o[i][k]);
    o[i][k] = t;
  }
};

// Adds one V row's contribution to the warp's channel tiles wq, wq + 4, wq + 8 (see
// v_row_accumulate): the accumulators stay in registers.
template <int G, int B>
__device__ __forceinline__ void rope_v_tiles(const uint8_t* vrow, int rv, int wq, const uint32_t (&bv)[8][2], uint32_t one,
                                             RopeAcc<OAcc<G>::N>& o) {
  constexpr int NO = OAcc<G>::N;
  const int lane = threadIdx.x & 31;
  const int P = rv >> 1, nfull = P >> 3;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int mu = wq + 4 * i;
    if (mu > nfull) break;
    const uint8_t* pa = vrow + (8 * mu + (lane >> 3)) * 32 * B + (lane & 7) * 4 * B;
    const int sA = 8 * mu + (lane >> 3);
    uint32_t wa[B], wb[B];
    load_piece_or_zero<B>(pa, sA < P, wa);
    load_piece_or_zero<B>(pa + 4 * 32 * B, sA + 4 < P, wb);
    // lanes that feed the normaliser row (strip P, odd channel)
    const bool la = B <= 2 && sA == P && (lane & 4), lb = B <= 2 && sA + 4 == P && (lane & 4);
    float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      uint32_t a0 = unpack_reg<B>(wa, 2 * t, one), a1 = unpack_reg<B>(wb, 2 * t, one);
      uint32_t a2 = unpack_reg<B>(wa, 2 * t + 1, one), a3 = unpack_reg<B>(wb, 2 * t + 1, one);
      if constexpr (B <= 2) {
        a0 = la ? unshift_h2<B>(2 * t) : a0;
        a2 = la ? unshift_h2<B>(2 * t + 1) : a2;
        a1 = lb ? unshift_h2<B>(2 * t) : a1;
        a3 = lb ? unshift_h2<B>(2 * t + 1) : a3;
      }
      mma_f16(d[t & 1], a0, a1, a2, a3, bv[t][0], bv[t][1]);
    }
    if constexpr (NO == 2) {
      o.add(i, 0, d[0][0] + d[1][0]);
      o.add(i, 1, d[0][2] + d[1][2]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) o.add(i, k, d[0][k] + d[1][k]);
    }
  }
}
// b = 0 stands for a head with r_V = 0: only the constant rows (one window class)
template <int G>
__device__ __forceinline__ void rope_v_dispatch(int b, const uint8_t* vrow, int rv, int wq, const __half* p, uint32_t one,
                                                RopeAcc<OAcc<G>::N>& o) {
  // the V MMA's B fragments: column n = lane / 4 holds query head n / 2 in its even columns (G = 4)
  // or n (G = 8); element k = token 2 j, 2 j + 1 (+ 8)
  const int lane = threadIdx.x & 31, n = lane >> 2, j = lane & 3;
  uint32_t bv[8][2];
  const uint32_t* pw = reinterpret_cast<const uint32_t*>(p + (G == 4 ? n >> 1 : n) * kRopePLd) + j;
  const bool on = G == 8 || !(n & 1);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    bv[t][0] = on ? pw[8 * t] : 0u;
    bv[t][1] = on ? pw[8 * t + 4] : 0u;
  }
  switch (b) {
    case 1: rope_v_tiles<G, 1>(vrow, rv, wq, bv, one, o); break;
    case 2: rope_v_tiles<G, 2>(vrow, rv, wq, bv, one, o); break;
    case 3: rope_v_tiles<G, 3>(vrow, rv, wq, bv, one, o); break;
    case 4: rope_v_tiles<G, 4>(vrow, rv, wq, bv, one, o); break;
    case 5: rope_v_tiles<G, 5>(vrow, rv, wq, bv, one, o); break;
    case 6: rope_v_tiles<G, 6>(vrow, rv, wq, bv, one, o); break;
    case 7: rope_v_tiles<G, 7>(vrow, rv, wq, bv, one, o); break;
    case 8: rope_v_tiles<G, 8>(vrow, rv, wq, bv, one, o); break;
    default: rope_v_tiles<G, 3>(vrow, 0, wq, bv, one, o); break;
  }
}

// ---------------------------------------------------------------------------------------
// The scan.  A CTA takes `batch` consecutive plan chunks at a time from the plan's counter and runs
// over stretches of consecutive rows of one group (W_K is staged when the K head changes); the
// stretch's sums go to its first chunk's slot and its other chunks are left empty.
// ---------------------------------------------------------------------------------------
template <int G, int MAXWG>
__global__ void __launch_bounds__(MAXWG * 160, 1) rope_scan_kernel(DecodeArgs a, RopeArgs ra) {
  constexpr int NO = OAcc<G>::N;
  extern __shared__ uint8_t smem_raw[];
  // the combine kernel may be scheduled as CTAs of this grid exit (it waits for the results)
  grid_dep_launch();
  const uint32_t raw = smem_addr(smem_raw);
  uint8_t* wsm = smem_raw + (((raw + 1023u) & ~1023u) - raw);  // W' hi atoms 0..2, lo atoms 3, 4
  float4* trig = reinterpret_cast<float4*>(wsm + kRopeWBytes);
  RopeSmem<G>& sh = *reinterpret_cast<RopeSmem<G>*>(wsm + kRopeWBytes + kRopeTrigBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the compute warps of all warpgroups, then one warp per warpgroup that issues MMAs and copies
  const int nwg = blockDim.x / 160;
  const bool mma_warp = tid >= 128 * nwg;
  const int wg = mma_warp ? warp - 4 * nwg : tid >> 7, wq = warp & 3, t = tid & 127;
  RopeWgSmem<G>& ws = sh.wg[wg];
  const int ns = ra.n_stage;
  uint8_t* stage0 = wsm + kRopeWBytes + kRopeTrigBytes + rope_vars_bytes<G>(nwg) + (size_t)wg * ns * ra.stage_bytes;
  const uint32_t bar0 = smem_addr(ws.bars);
  auto bar_k = [&](int i) { return bar0 + 8u * i; };
  auto bar_v = [&](int i) { return bar0 + 16u + 8u * i; };
  auto bar_x = [&](int h) { return bar0 + 32u + 8u * h; };
  const uint32_t bar_a = bar0 + 48u, bar_h1 = bar0 + 56u;
  if (mma_warp && lane == 0) {
    for (int i = 0; i < 8; ++i) mbar_init(bar0 + 8u * i, i < 6 ? 1 : 4);
    fence_mbar_init();
  }
  if (tid == 0) sh.fail = 0;
  if (warp == 0) tmem_alloc(smem_addr(&sh.tmem), 512);
  // the queries and the cache come from the kernels ahead (also the table's own kernel)
  grid_dep_wait();
  const WsHeader* wh = reinterpret_cast<const WsHeader*>(a.ws);
  const WsGroup* groups = reinterpret_cast<const WsGroup*>(a.ws + wh->groups_off);
  const WsItem* items = reinterpret_cast<const WsItem*>(a.ws + wh->items_off);
  const HeadEntry* heads = head_table(a.block);
  const float* pool = param_pool(a.block);
  float* parts = reinterpret_cast<float*>(a.ws + wh->part_off);
  const int n_items = wh->n_items, gstride = wh->g_stride, pstride = wh->part_stride;
  unsigned int* next_item = const_cast<unsigned int*>(&wh->next_item);
  const float* coarse = ra.table + (size_t)kRopeFine * kRopeRowFloats;
  for (int idx = tid; idx < 32 * 128; idx += blockDim.x) {
    const int j2 = idx >> 7, tau = idx & 127;
    const float* f = ra.table + (size_t)(tau & 15) * kRopeRowFloats;
    const float* m = coarse + (size_t)min(tau >> 4, ra.n_coarse - 1) * kRopeRowFloats;
    float c[2], s[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int e = rope_entry(2 * j2 + k);
      rope_compose(m[e], m[e + 1], f[e], f[e + 1], c[k], s[k]);
    }
    trig[idx] = make_float4(c[0], c[1], s[0], s[1]);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem;
  const uint32_t lanes = (uint32_t)(32 * wq) << 16;                          // this warp's TMEM lanes
  const float4* trig_t = trig + t;
  const uint32_t one = a.one;
  const int rho_t = 2 * (t >> 4) + ((t >> 3) & 1);  // V register of the thread's token
  uint32_t ph_k = 0, ph_v = 0;                      // parity of the next wait per stage
  int total = 0;                                    // rows of this warpgroup before this stretch
  int staged_head = -1;

  // waits of a warp; after a failed one the warpgroup leaves its rows at the next barrier
  bool expired = false;
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, kWaitLimitNs))) {
      if (lane == 0) atomicOr(&g_status, 1u);
      expired = true;
    }
  };
  // barrier of the warpgroup: whether `raise` holds in any thread, and (`failed`) whether a wait of
  // any of its warps has expired - the same answers in all threads
  auto row_barrier = [&](bool raise, bool& failed) {
    const bool any = wg_any(wg, raise || expired);
    failed = false;
    if (any) {
      if (lane == 0) ws.fail[wq] = expired;
      wg_sync(wg);
      failed = ws.fail[0] | ws.fail[1] | ws.fail[2] | ws.fail[3];
      if (failed && t == 0) sh.fail = 1;
    }
    return any;
  };

  for (;;) {
    if (tid == 0) sh.batch = (int)atomicAdd(next_item, 1u);
    __syncthreads();
    const long long first = (long long)sh.batch * ra.batch;
    if (first >= n_items || sh.fail) break;
    const int i_end = min(n_items, (int)first + ra.batch);
    for (int i0 = (int)first; i0 < i_end;) {
      // ---- a stretch: chunks i0 .. i1 - 1, consecutive rows of one group ----
      const WsItem it0 = items[i0];
      int i1 = i0 + 1, row_end = it0.row_end, last_slot = it0.slot;
      while (i1 < i_end) {
        const WsItem x = items[i1];
        if (x.group != it0.group || x.row_begin != row_end) break;
        row_end = x.row_end;
        last_slot = x.slot;
        ++i1;
      }
      const WsGroup gr = groups[it0.group];
      const HeadEntry hk = heads[gr.k_head], hv = heads[gr.v_head];
      const int rk = hk.r, kb = hk.b, vr = hv.r, vb = hv.b, nk = (rk + 15) >> 4;
      const int T = a.seq_lens[gr.seq];
      const int rows_valid = (T + kRowTokens - 1) / kRowTokens;
      // a group's last chunk takes every row that is left (never past the cache's rows)
      const int cap_rows = a.page_table ? 2 * a.pages_per_seq : a.rows_per_seq;
      const int row0 = it0.row_begin;
      const int row1 = last_slot == gr.first_item + gr.n_items - 1 ? min(rows_valid, cap_rows) : min(rows_valid, row_end);
      const uint32_t rbk = rk > 0 ? 16u * rk * kb : 0u, rbv = vr > 0 ? 16u * vr * vb : 0u;
      const uint32_t kst = rk > 0 ? 256u * kb * nk : 0u;  // whole channel tiles (the last may read past the row)
      // TMEM's 512 columns hold X (128) and A (8 nk + 8) of three warpgroups up to nk = 4, of two beyond
      const int nact = nk <= 4 ? nwg : min(nwg, 2);
      const uint32_t x_col = tmem + 128u * wg, a_col = tmem + 128u * nact + (nact == 3 ? 40u : 72u) * wg;
      const bool fits = kst + ((rbv + 127u) & ~127u) <= (uint32_t)ra.stage_bytes;
      if (!fits && tid == 0) atomicOr(&g_status, 2u);
      if (T > kRopeFine * ra.n_coarse && tid == 0) atomicOr(&g_status, 2u);  // positions past the table
      const int n_rows = fits && wg < nact && row1 > row0 + wg ? (row1 - row0 - wg + nact - 1) / nact : 0;  // of this warpgroup
      const uint8_t* kbase = a.cache + hk.cache_off;
      const uint8_t* vbase = a.cache + hv.cache_off;
      // copies of the n-th row's K or V into its stage (one thread)
      auto load_k = [&](int n) {
        const int st = n % ns, row = row0 + wg + n * nact;
        mbar_arrive_expect_tx(bar_k(st), rbk);
        bulk_g2s(smem_addr(stage0 + (size_t)st * ra.stage_bytes),
                 kbase + row_offset(0, rbk, gr.seq, row, a.page_table, a.pages_per_seq, a.rows_per_seq), rbk, bar_k(st));
      };
      auto load_v = [&](int n) {
        const int st = n % ns, row = row0 + wg + n * nact;
        mbar_arrive_expect_tx(bar_v(st), rbv);
        bulk_g2s(smem_addr(stage0 + (size_t)st * ra.stage_bytes + kst),
                 vbase + row_offset(0, rbv, gr.seq, row, a.page_table, a.pages_per_seq, a.rows_per_seq), rbv, bar_v(st));
      };
      if (mma_warp && lane == 0) {  // the stages are free: every read of them is before the last block barrier
        fence_proxy_async_smem();
        for (int n = 0; n < min(ns, n_rows); ++n) {
          if (rbk) load_k(n);
          if (rbv) load_v(n);
        }
      }
      const float dk = (rk > 0 && hk.delta > 0.f) ? hk.delta : 1.f;
      if (gr.k_head != staged_head) {
        staged_head = gr.k_head;
        if (!mma_warp) {
        const float* W = pool + hk.w_off;  // d x r, column c at W + c d
        const int dm = t, j = dm & 63, P = 4 * (j >> 1) + 2 * (dm >> 6) + (j & 1);
        auto put = [&](int limb_atom, int c, uint32_t v) {  // channels c, c + 1 of position P, 128-byte swizzle
          const int atom = limb_atom + (c >> 6);
          *reinterpret_cast<uint32_t*>(wsm + atom * kRopeAtomBytes + P * 128 + ((((c & 63) >> 3) ^ (P & 7)) << 4) +
                                       (c & 7) * 2) = v;
        };
#pragma unroll 8
        for (int c = 2 * wg; c < 16 * nk; c += 2 * nwg) {
          const float x0 = c < rk ? W[(size_t)c * kD + dm] : 0.f, x1 = c < rk ? W[(size_t)(c + 1) * kD + dm] : 0.f;
          const __half2 h = __floats2half2_rn(x0, x1);
          const float2 f = __half22float2(h);
          const __half2 l = __floats2half2_rn(x0 - f.x, x1 - f.y);
          put(0, c, *reinterpret_cast<const uint32_t*>(&h));
          put(3, c, *reinterpret_cast<const uint32_t*>(&l));
        }
        // the constant A columns: 1 in the first three elements of tile nk
        const uint32_t cst[8] = {0x3C003C00u, 0x00003C00u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (wg < nact) tc_st32x8(a_col + lanes + 8 * nk, cst);
        tc_wait_st();
        tc_fence_before();
        if (wg == 0) {  // mu' / Delta in three limbs
          const float mu = pool[hk.mu_off + dm];
          const float beta = rk > 0 ? mu / hk.delta : mu;
          const float h0 = __half2float(__float2half_rn(beta)), h1 = __half2float(__float2half_rn(beta - h0));
          const float h2 = beta - h0 - h1;
          put(0, 16 * nk, pack_f16(h0, h1));
          put(0, 16 * nk + 2, pack_f16(h2, 0.f));
#pragma unroll
          for (int c = 4; c < 16; c += 2) put(0, 16 * nk + c, 0u);
        }
        fence_proxy_async_smem();  // W' is read by the tensor cores (async proxy)
        }
      }
      // ---- the group's query, turned to its position ----
      {
        int p = ra.q_pos ? ra.q_pos[gr.seq] : T - 1;
        // an empty sequence (default position -1) has no output; any other position outside the
        // table is reported and clamped
        const int max_pos = kRopeFine * ra.n_coarse;
        const bool bad = p < 0 ? (ra.q_pos != nullptr) : p >= max_pos;
        if (bad && tid == 0) atomicOr(&g_status, 2u);
        p = min(max(p, 0), max_pos - 1);
        const float fac = dk * 0.088388347648318440f * 1.4426950408889634f;  // Delta/sqrt(128) log2(e)
        const float* fine = ra.table + (size_t)(p & 15) * kRopeRowFloats;
        const float* crs = coarse + (size_t)(p >> 4) * kRopeRowFloats;
        for (int idx = tid; idx < 32 * G && !mma_warp; idx += 128 * nwg) {
          const int j2 = idx / G, g = idx % G;
          const __nv_bfloat16* qp = a.q + gr.layer * a.q_sl + (long long)gr.seq * a.q_ss + (long long)(gr.kv * G + g) * kD;
          float qa[2], qb[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int j = 2 * j2 + k, e = rope_entry(j);
            float c, s;
            rope_compose(crs[e], crs[e + 1], fine[e], fine[e + 1], c, s);
            const float xa = __bfloat162float(qp[j]), xb = __bfloat162float(qp[j + kD / 2]);
            qa[k] = fac * fmaf(xa, c, -xb * s);
            qb[k] = fac * fmaf(xa, s, xb * c);
          }
          sh.qbase[idx] = make_float4(qa[0], qa[1], qb[0], qb[1]);
        }
      }
      __syncthreads();
      tc_fence_after();

      // ---- this warpgroup's rows ----
      const int vc = (vr > 0 && vb <= 2) ? vb : 0, vbd = vr > 0 ? vb : 0;
      const float vout = vr == 0 ? 0.f : (float)(1 << (vb == 1 ? 5 : vb == 2 ? 6 : vb));
      const float pshift = vc == 1 ? (float)(Window<1>::kmin() - Window<1>::k(rho_t))
                                   : vc == 2 ? (float)(Window<2>::kmin() - Window<2>::k(rho_t)) : 0.f;
      const int ntile = (vr >> 4) + 1;  // V accumulator tiles incl. the constant rows
      RopeAcc<NO> o;
      float mref[G], s[G];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int u = 0; u < NO; ++u) o.o[k][u] = o.e[k][u] = 0.f;
#pragma unroll
      for (int g = 0; g < G; ++g) mref[g] = -INFINITY;
      // angles of R(128 row) for the thread's share of the query: (j2, g) = (t / G.., t % G)
      constexpr int QN = G / 4;
      float2 ang[QN][2];
      auto load_angles = [&](int n) {
        const float* crs = coarse + (size_t)min(8 * (row0 + wg + n * nact), ra.n_coarse - 1) * kRopeRowFloats;
#pragma unroll
        for (int u = 0; u < QN; ++u)
#pragma unroll
          for (int k = 0; k < 2; ++k)
            ang[u][k] = __ldg(reinterpret_cast<const float2*>(crs + rope_entry(2 * ((t + 128 * u) / G) + k)));
      };
      if (n_rows > 0 && !mma_warp) load_angles(0);
      // probabilities of the thread's token against the reference maxima, as fed to the V MMA
      auto put_p = [&](int buf) {
#pragma unroll
        for (int g = 0; g < G; ++g) ws.p[buf][g * kRopePLd + t] = __float2half_rn(ex2_approx(s[g] + (pshift - mref[g])));
      };
      // the values of row n: its probabilities are in buffer n & 1 unless a score exceeded its
      // reference by more than kTau (`raise`); then the reference moves to the row's maxima and the
      // accumulators are rescaled first
      auto values = [&](int n, bool raise) {
        if (raise) {
#pragma unroll
          for (int g = 0; g < G; ++g) {
            float mx = s[g];
#pragma unroll
            for (int m = 16; m; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
            if (lane == 0) ws.wmax[wq][g] = mx;
          }
          wg_sync(wg);
          float alpha[NO];
#pragma unroll
          for (int k = 0; k < NO; ++k) alpha[k] = 1.f;
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float mx = fmaxf(fmaxf(ws.wmax[0][g], ws.wmax[1][g]), fmaxf(ws.wmax[2][g], ws.wmax[3][g]));
            const bool mv = mx > mref[g] + kTau;
            const float al = mv ? ex2_approx(mref[g] - (mx - kRopeLift)) : 1.f;
            mref[g] = mv ? mx - kRopeLift : mref[g];
#pragma unroll
            for (int k = 0; k < NO; ++k)
              if (g == (G == 4 ? (lane & 3) : 2 * (lane & 3) + (k & 1))) alpha[k] = al;
          }
#pragma unroll
          for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < NO; ++k) {
              o.o[i][k] *= alpha[k];
              o.e[i][k] *= alpha[k];
            }
          put_p(n & 1);
          wg_sync(wg);
        }
        const int st = n % ns;
        if (rbv) {
          wait(bar_v(st), (ph_v >> st) & 1u);
          ph_v ^= 1u << st;
        }
        rope_v_dispatch<G>(vbd, stage0 + (size_t)st * ra.stage_bytes + kst, vr, wq, ws.p[n & 1], one, o);
      };
      bool failed = false;
      if (mma_warp) {
        // ---- MMAs and copies of the warpgroup's rows, by one thread ----
        if (lane == 0) {
          const uint64_t wdesc = umma_desc_sw128(smem_addr(wsm));
          for (int n = 0; n < n_rows && !expired; ++n) {
            const uint32_t par = (uint32_t)(total + n) & 1u;
            if (!mbar_wait_bounded(bar_a, par, kWaitLimitNs)) {
              expired = true;
              break;
            }
            tc_fence_after();
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              if (h && n > 0 && !mbar_wait_bounded(bar_h1, par ^ 1u, kWaitLimitNs)) {
                expired = true;
                break;
              }
              if (h) tc_fence_after();
              const uint64_t dh = wdesc + (uint64_t)(h * (64 * 128 >> 4));  // positions 64 h ..
              for (int kt = 0; kt <= nk; ++kt)
                tc_mma_bf16_ts(x_col + 64 * h, a_col + 8 * kt, dh + (kt >> 2) * (kRopeAtomBytes >> 4) + (kt & 3) * 2,
                               kRopeIdesc, kt > 0);
              for (int kt = 0; kt < nk; ++kt)
                tc_mma_bf16_ts(x_col + 64 * h, a_col + 8 * kt, dh + (3 + (kt >> 2)) * (kRopeAtomBytes >> 4) + (kt & 3) * 2,
                               kRopeIdesc, 1);
              tc_commit(bar_x(h));
              if (h == 0) {
                // A of row n written: every thread is past its reads of that row's K stage, and of the
                // V stage of row n - 2 (it takes the values of a row before it unpacks the second next)
                fence_proxy_async_smem();
                if (rbk && n + ns < n_rows) load_k(n + ns);
                if (rbv && n >= 2 && n - 2 + ns < n_rows) load_v(n - 2 + ns);
              }
            }
          }
          // the last V rows of a single stage: row n - 1's is free once row n's scores are in, which the
          // second half's last read tells
          if (rbv && ns == 1 && n_rows >= 2 && !expired) {
            if (mbar_wait_bounded(bar_h1, (uint32_t)(total + n_rows - 1) & 1u, kWaitLimitNs)) {
              fence_proxy_async_smem();
              load_v(n_rows - 1);
            } else {
              expired = true;
            }
          }
          if (expired) atomicOr(&g_status, 1u);
        }
        __syncwarp();
      } else {
        // the A operand of row n: its codes, once the copies have landed
        auto unpack = [&](int n) {
          const int st = n % ns;
          if (rbk) {
            wait(bar_k(st), (ph_k >> st) & 1u);
            ph_k ^= 1u << st;
            rope_unpack_dispatch(kb, stage0 + (size_t)st * ra.stage_bytes, nk, t, a_col + lanes);
            tc_wait_st();
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_a);
        };
        // the query turned by -128 row
        auto turn_query = [&](int n) {
#pragma unroll
          for (int u = 0; u < QN; ++u) {
            const float4 qb = sh.qbase[t + 128 * u];
            ws.q[n & 1][t + 128 * u] =
                make_float4(fmaf(qb.x, ang[u][0].x, qb.z * ang[u][0].y), fmaf(qb.y, ang[u][1].x, qb.w * ang[u][1].y),
                            fmaf(qb.z, ang[u][0].x, -qb.x * ang[u][0].y), fmaf(qb.w, ang[u][1].x, -qb.y * ang[u][1].y));
          }
        };
        if (n_rows > 0) {
          turn_query(0);
          if (n_rows > 1) load_angles(1);
          unpack(0);
          wg_sync(wg);  // publishes the first row's query
        }
        for (int n = 0; n < n_rows; ++n) {
          const int row = row0 + wg + n * nact;
          const uint32_t par = (uint32_t)(total + n) & 1u;
          const float4* q = ws.q[n & 1];
          f32x2 acc[2 * G];
#pragma unroll
          for (int g = 0; g < 2 * G; ++g) acc[g] = 0ull;
          wait(bar_x(0), par);
          tc_fence_after();
          rope_scores_half<G>(x_col + lanes, trig_t, q, acc);
          // both halves' MMAs done: A can take the next row's codes
          wait(bar_x(1), par);
          tc_fence_after();
          if (n + 1 < n_rows) {
            unpack(n + 1);
            turn_query(n + 1);
            if (n + 2 < n_rows) load_angles(n + 2);
          }
          rope_scores_half<G>(x_col + 64 + lanes, trig_t + 16 * 128, q + 16 * G, acc);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_h1);
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float2 v = unpack2(acc[2 * g]), u = unpack2(acc[2 * g + 1]);
            // only the last row of a sequence has masked tokens
            s[g] = row * kRowTokens + t < T ? (v.x + v.y) + (u.x + u.y) : -INFINITY;
          }
          bool exceed = false;
#pragma unroll
          for (int g = 0; g < G; ++g) exceed |= s[g] > mref[g] + kTau;
          put_p(n & 1);
          // publishes the probabilities and the next row's query
          const bool raise = row_barrier(exceed, failed);
          if (failed) break;
          values(n, raise);
        }
      }
      // a wait that no row barrier has reported (a last row's values, an issuing thread's) ends the CTA
      // all the same, before its stages are filled again
      if (expired) sh.fail = 1;
      // ---- the stretch's sums (m, l, (O - c) 2^(10 - kmin)): the second warpgroup's through shared
      //      memory into the first one's, which go to the first slot ----
      const int cr = vr & 15, ct = vr >> 4;
      if (!mma_warp) wg_sync(wg);
      if (!mma_warp && wq == (ct & 3)) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // constant rows r and r + 1
          const int rr = cr + e;
          if ((lane >> 2) == (rr & 7)) {
#pragma unroll
            for (int k = 0; k < NO; ++k) {
              if ((NO == 2 ? k : k >> 1) != (rr >> 3)) continue;
              const int g = G == 4 ? (lane & 3) : 2 * (lane & 3) + (k & 1);
              float v = o.o[0][k], w = o.e[0][k];
              if ((ct >> 2) == 1) v = o.o[1][k], w = o.e[1][k];
              if ((ct >> 2) == 2) v = o.o[2][k], w = o.e[2][k];
              ws.cl[e][g] = v;
              ws.cle[e][g] = w;
            }
          }
        }
      }
      if (!mma_warp) wg_sync(wg);
      float lsum[G];
#pragma unroll
      for (int g = 0; g < G; ++g) lsum[g] = ws.cl[1][g] + ws.cle[1][g];
      // f(g, channel, value) of this lane's entries
      auto entries = [&](auto f) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int mu = wq + 4 * i;
          if (mu >= ntile) break;
#pragma unroll
          for (int k = 0; k < NO; ++k) {
            const int g = G == 4 ? (lane & 3) : 2 * (lane & 3) + (k & 1);
            const int ch = 16 * mu + (lane >> 2) + 8 * (NO == 2 ? k : k >> 1);
            if (ch < vr) f(g, ch, ((o.o[i][k] - ws.cl[0][g]) + (o.e[i][k] - ws.cle[0][g])) * vout);
          }
        }
      };
      if (wg > 0 && wg < nact && !mma_warp) {
        entries([&](int g, int ch, float v) { sh.merge[wg - 1][g][4 + ch] = v; });
        if (t == 0) {
#pragma unroll
          for (int g = 0; g < G; ++g) {
            sh.merge[wg - 1][g][0] = mref[g];
            sh.merge[wg - 1][g][1] = lsum[g];
          }
        }
      }
      __syncthreads();
      if (wg == 0 && !mma_warp) {
        float* part = parts + (size_t)it0.slot * pstride;
        // e: the entry of a warpgroup's block (1: l, 4 + channel: O); v0: this warpgroup's value
        auto merged = [&](int g, float m0, int e, float v0, float& M) {
          M = m0;
          for (int x = 0; x < nact - 1; ++x) M = fmaxf(M, sh.merge[x][g][0]);
          float r = m0 != -INFINITY ? exp2f(m0 - M) * v0 : 0.f;
          for (int x = 0; x < nact - 1; ++x)
            if (sh.merge[x][g][0] != -INFINITY) r += exp2f(sh.merge[x][g][0] - M) * sh.merge[x][g][e];
          return r;
        };
        if (t == 0) {
#pragma unroll
          for (int g = 0; g < G; ++g) {
            float M;
            const float l = merged(g, mref[g], 1, lsum[g], M);
            part[g * gstride] = M;
            part[g * gstride + 1] = l;
          }
        }
        entries([&](int g, int ch, float v) {
          float m0 = mref[0], M;
#pragma unroll
          for (int k = 1; k < G; ++k) m0 = g == k ? mref[k] : m0;
          part[g * gstride + 4 + ch] = merged(g, m0, 4 + ch, v, M);
        });
        for (int i = i0 + 1 + t / G; i < i1; i += 128 / G) {  // the stretch's other chunks
          float* pg = parts + (size_t)items[i].slot * pstride + (t % G) * gstride;
          pg[0] = -INFINITY;
          pg[1] = 0.f;
        }
      }
      total += n_rows;
      __syncthreads();  // the merge area, the stages and W' are free for the next stretch
      if (sh.fail) break;  // set by a failed warpgroup before the barrier
      i0 = i1;
    }
  }
  if (sh.fail && mma_warp && lane == 0) {
    // after an expired wait: whatever this warpgroup still has in flight is given time to land before
    // the shared memory and TMEM go away
    tc_commit(bar_x(0));
    for (int k = 0; k < 6; ++k) mbar_wait_bounded(bar0 + 8u * k, 0, 1000000ull);
    for (int k = 0; k < 6; ++k) mbar_wait_bounded(bar0 + 8u * k, 1, 1000000ull);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
  // the last CTA to run out of items puts the work counter back to 0 for the next launch
  if (tid == 0) {
    unsigned int* done = const_cast<unsigned int*>(&wh->done_ctas);
    if (atomicAdd(done, 1u) == gridDim.x - 1) {
      atomicExch(next_item, 0u);
      atomicExch(done, 0u);
    }
  }
}

}  // namespace cobra
