// Internal layouts shared by the host code and the CUDA kernels of libcobra (not part of
// the public ABI in include/cobra.h).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace cobra {

constexpr int kD = 128;                 // head dimension
constexpr int kRowTokens = 128;         // tokens per code row
constexpr uint32_t kBlockMagic = 0x52424F43u;  // "COBR"
constexpr uint32_t kWsMagic = 0x53574F43u;     // "COWS"

// Device parameter block: header | head table | float pool.
struct BlockHeader {
  uint32_t magic;
  uint32_t version;
  int32_t n_heads;
  int32_t d;
  uint64_t heads_off;    // bytes from block start
  uint64_t pool_off;     // bytes from block start
  uint64_t pool_floats;
  uint64_t checksum;     // FNV-1a 64 of the whole block with this field zero
  uint64_t reserved[2];
};
static_assert(sizeof(BlockHeader) == 64, "header size");

struct HeadEntry {
  int32_t r, b;
  float delta, inv_delta;
  uint64_t cache_off;  // bytes into the cache buffer
  uint64_t w_off;      // floats into the pool: W, d x r column-major
  uint64_t mu_off;     // floats into the pool: mu, d
  uint64_t wmu_off;    // floats into the pool: W^T mu, r
  uint64_t reserved[2];
};
static_assert(sizeof(HeadEntry) == 64, "head entry size");

// Decode workspace: header | groups | items | head-group table | q~ blocks | partials.
struct WsHeader {
  uint32_t magic;
  uint32_t version;
  int32_t n_groups;
  int32_t n_items;
  int32_t group;      // G
  int32_t n_layers;
  int32_t n_kv;
  int32_t n_seqs;
  uint64_t groups_off, items_off, qt_off, part_off;  // bytes from workspace start
  int32_t part_stride;  // floats per item partial
  int32_t g_stride;     // floats per query head inside a partial: [m, l, -, -, O[0..max_rv)]
  int32_t qt_stride;    // bytes per group q~ block
  int32_t max_rv;
  int32_t max_row_bytes;  // largest K or V code row among the planned heads
  int32_t reserved0;
  uint64_t hg_off;        // int32 [n_layers * n_kv][n_seqs]: group index of (head, seq)
  int32_t reserved[6];
  uint32_t done_ctas;     // scan CTAs that have finished taking items in the running launch
  uint32_t next_item;     // scan work counter: 0 between launches (the scan's last CTA resets it)
};
static_assert(sizeof(WsHeader) == 128, "ws header size");

// A group's chunks write their partials to slots first_item .. first_item + n_items - 1.
struct WsGroup {
  int32_t seq, layer, kv, first_item;
  int32_t n_items, k_head, v_head, reserved;
};
// Work items in the order the scan takes them; slot is the partial the chunk writes.
struct WsItem {
  int32_t group, row_begin, row_end, slot;
};

// q~ block per group: Qsum[8] (fp32, sum of the fp16 hi+lo values per query head),
// scale (fp32, 2^-e), then B fragments [kappa 0..7][ntile 0..1][lane 0..31] of uint2.
constexpr int kQtHeaderBytes = 64;
constexpr int kQtStride = kQtHeaderBytes + 8 * 2 * 32 * 8;

constexpr size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The scan's per-warp staging ring for code rows of at most `max_row` bytes: a K and a V row.
constexpr size_t scan_ring_bytes(size_t max_row) {
  const size_t two = 2 * align_up(max_row, 128);
  return two > 8192 ? two : 8192;
}

// The scan's shared memory per warp besides the ring: V accumulators and query fragments.
constexpr size_t scan_state_bytes(int group) { return group == 4 ? 4352 : 8704; }

// Resident scan warps per SM that the registers allow: 128 a thread with 4 query heads per kv head, 168
// with 8 (the scan's launch bounds are made of these).
constexpr int kScanCtaWarps = 4;  // per CTA at most
constexpr int scan_reg_warps(int group) { return group == 4 ? 16 : 12; }

// Warps per scan CTA and resident warps per SM (at most what the registers allow): 4, 2 or 1 warps,
// whichever fits the most into 228 KB of shared memory (1 KB of it per CTA is the system's); the
// larger CTA of equals, whose launches are fewer.  A layer of 8 kv heads x 8 x 32768 tokens at 1 bpd
// (8 KB rings) takes 57 us per step with 4, 60 with 2 and 65 with 1; 2 layers x 32 ragged sequences at
// 4 bpd (24 to 32 KB rings) 639, 547 and 541.  With 8 query heads the layer takes 67 us; 76 in CTAs of
// one warp and chunks for the 13 warps per SM that shared memory alone would hold.
struct ScanShape {
  int cta_warps, sm_warps;
};
constexpr ScanShape scan_shape(size_t ring, int group) {
  ScanShape best{1, 0};
  for (int nw = kScanCtaWarps; nw >= 1; nw /= 2) {
    const size_t cta = nw * (ring + scan_state_bytes(group)) + 1024;
    const int n = (int)(233472 / cta) * nw, limit = scan_reg_warps(group) / nw * nw;
    const int warps = n < limit ? n : limit;
    if (warps > best.sm_warps) best = ScanShape{nw, warps};
  }
  return best;
}

}  // namespace cobra
