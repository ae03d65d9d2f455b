// plan.cuh -- how the fills of a batch are cut into work items (host side, shared
// by prng_batch_* and prng_batcher_*).
#pragma once

#include <algorithm>

#include "../../include/prng.h"
#include "batch.cuh"
#include "handle.cuh"
#include "ranlux_tc.cuh"

namespace prng {

// Whether a batch's requests of a RANLUX family are faster on the tensor cores, in
// cycles: the chain by its longest stream or by its warps' throughput, as for a
// plain fill (ranlux_auto_tile), against two launches, the starts and the
// products.  us, tensor cores / chain, in back-to-back serving ticks of 4,096 streams
// a client: 1 client 25 / 19, 4 83 / 70, 12 109 / 95; 6, one of them
// with a long fill, 180 / 487.
inline bool lux_tensor_pays(int p, const LuxSplit& sp, uint64_t warp_blocks, uint64_t longest) {
  const uint64_t sms = (uint64_t)sm_count();
  const uint64_t chain = std::max<uint64_t>(longest * ((49 * p + 5900) / 10),
                                            warp_blocks * ((17 * p + 1120) / 4) / (4 * sms));
  const uint64_t len = sp.cut ? std::min<uint64_t>(longest, 1ull << sp.lgb) : longest;
  const uint64_t product = std::max<uint64_t>(len * 1712, warp_blocks * 2873 / (16 * sms));
  return chain > 30000 + product;
}

struct ItemPlan {
  bool tensor = true;            // false: RANLUX on the borrow chain (no room for the segments' starts)
  bool lux_pays[FAM_COUNT];      // RANLUX families worth the tensor cores
  Tile tile[FAM_COUNT];
  LuxSplit split[FAM_COUNT];     // tensor-core families
  uint32_t max_seg[FAM_COUNT] = {};
  uint32_t mt_rows = 2;          // MT19937 streams per item, one after the other
  uint32_t ranmar_seed_rows = 256;

  ItemPlan() {
    for (int f = 0; f < FAM_COUNT; f++) {
      tile[f] = tile_of(f);
      lux_pays[f] = true;
    }
  }
  // RANLUX families whose fills run on the tensor cores.
  bool is_lux_tc(int f) const {
    return tensor && lux_pays[f] && kind_of(f) >= FAM_LUX24 && kind_of(f) < FAM_KINDS && lux_p_of(f) >= kLuxTcMinP;
  }
  // The segment length of every tensor-core family, from all its requests;
  // without `cut` each stream is one segment and MT19937 items are coarser.
  void choose(const prng_fill_req* reqs, uint32_t n, bool cut) {
    mt_rows = cut ? 1 : 2;
    ranmar_seed_rows = cut ? 16 : 256;
    for (int f = 0; f < FAM_COUNT; f++) lux_pays[f] = true;
    uint64_t wb[FAM_COUNT] = {}, longest[FAM_COUNT] = {}, xor_odd = 0;
    for (uint32_t i = 0; i < n; i++) {
      if (reqs[i].st->gen == XOR128 && (((reinterpret_cast<uintptr_t>(reqs[i].d_out) >> 2) | reqs[i].n_per_stream) & 7))
        xor_odd += reqs[i].st->n_streams;
      if (reqs[i].st->gen != RANLUX || reqs[i].n_per_stream == 0) continue;
      const int f = fill_family(reqs[i].st->gen, reqs[i].st->p, reqs[i].f32 != 0);
      if (!is_lux_tc(f)) continue;
      const uint64_t nb = reqs[i].n_per_stream / 24;
      wb[f] += (reqs[i].st->n_streams + 31) / 32 * (nb + 1);
      longest[f] = std::max(longest[f], nb);
    }
    // XOR128: items of 64 streams, whose tail is shorter, unless many streams' rows
    // start inside a 32-byte sector, which 64-column tiles store faster (items of 64 /
    // 128, us: 2,000 requests, 42,141 such streams 1,544 / 1,524, 5,000 with 112,220
    // 3,906 / 3,737, 20,000 with 386,965 15,235 / 14,695; but 500 with 8,456 409 / 435,
    // 20,000 short ones with 10,158 1,554 / 1,732).
    const bool fine = cut && !tile_chosen(XOR128, 0) && xor_odd < 32768;
    tile[FAM_XOR128] = tile[FAM_XOR128 + FAM_F32] = fine ? Tile{64, 32, 1} : tile_of(FAM_XOR128);
    for (int f = 0; f < FAM_COUNT; f++) {
      split[f] = LuxSplit{};
      max_seg[f] = 0;
      if (cut && longest[f] > 0) split[f] = lux_split(wb[f], longest[f]);
      if (split[f].cut) max_seg[f] = (uint32_t)(segments(f, 24 * longest[f]) - 1);
      if (is_lux_tc(f) && !lux_tensor_pays(lux_p_of(f), split[f], wb[f], longest[f])) {
        lux_pays[f] = false;
        split[f] = LuxSplit{};
        max_seg[f] = 0;
      }
    }
  }
  // Segments of a request of n draws per stream.
  uint64_t segments(int f, uint64_t n) const { return split[f].cut ? lux_segments(n, split[f].lgb) : 1; }
  // Streams per re-seeding item.
  uint32_t seed_rows(const prng_state* st) const { return st->gen == RANMAR ? ranmar_seed_rows : 256u; }
  uint32_t rows(int f) const { return kind_of(f) == FAM_MT ? mt_rows : rows_per_item(f, tile[f]); }
  uint64_t count(int f, const prng_state* st, uint64_t n) const {
    if (is_lux_tc(f)) return (st->n_streams + 31) / 32 * segments(f, n);
    const uint32_t per = rows(f);
    return (st->n_streams + per - 1) / per;
  }
  // Of a tensor-core family's items, those that start a group of segments.
  bool first(const BatchItem& it) const { return it.rows % kLuxGroup == 0; }
  // Work of the request's longest item, in draws or blocks of one thread.
  uint64_t cost(int f, uint64_t n) const {
    if (is_lux_tc(f)) return split[f].cut ? std::min<uint64_t>(n / 24, 1ull << split[f].lgb) : n / 24;
    return n;
  }
  // The request's items, in order.
  template <class Push>
  void items(int f, uint32_t req, const prng_state* st, uint64_t n, Push push) const {
    if (is_lux_tc(f)) {
      const uint64_t segs = segments(f, n);
      for (uint64_t s = 0; s < segs; s++)
        for (uint64_t r0 = 0; r0 < st->n_streams; r0 += 32) push(BatchItem{req, (uint32_t)s, r0});
      return;
    }
    const uint32_t per = rows(f);
    for (uint64_t r0 = 0; r0 < st->n_streams; r0 += per)
      push(BatchItem{req, (uint32_t)std::min<uint64_t>(per, st->n_streams - r0), r0});
  }
};

// Tensor map of a request's output, up to its limit's last whole row.
inline bool request_map(const prng_fill_req& r, CUtensorMap* map) {
  const uint64_t full = r.st->n_streams * r.n_per_stream;
  const uint64_t limit = (r.n_valid == 0 || r.n_valid > full) ? full : r.n_valid;
  return r.n_per_stream > 0 && lux_out_map(r.d_out, r.n_per_stream, limit / r.n_per_stream, map);
}

// The kernel of family f (not the seeding) on stream s; starts: the family's
// segment starts, lux_start_bytes(q.n_items), and the n_groups items that start
// a group of segments, for a tensor-core family.
inline cudaError_t launch_family(int f, const BatchQueue& q, const ItemPlan& plan, const CUtensorMap* maps,
                                 uint32_t* starts, const uint32_t* firsts, uint32_t n_groups, cudaStream_t s) {
  const bool f32 = is_f32_family(f);
  const Tile t = plan.tile[f];
  switch (kind_of(f)) {
    case FAM_MLCG: return launch_batch_mlcg(q, t, s);
    case FAM_XOR128: return launch_batch_xor128(q, t, f32, s);
    case FAM_RANMAR: return launch_batch_ranmar(q, t, f32, s);
    case FAM_MT: return launch_batch_mt(q, t, f32, s);
    default: break;
  }
  if (!plan.is_lux_tc(f)) return launch_batch_ranlux(q, lux_p_of(f), t, f32, s);
  LuxJob job{};
  job.reqs = q.reqs;
  job.items = q.items;
  job.maps = maps;
  job.counter = q.counter;
  job.starts = starts;
  job.firsts = plan.max_seg[f] > 0 ? firsts : nullptr;
  job.n_groups = plan.max_seg[f] > 0 ? n_groups : q.n_items;
  job.n_items = q.n_items;
  job.max_seg = plan.max_seg[f];
  job.lgb = plan.split[f].lgb;
  return launch_lux_job(job, lux_p_of(f), f32 ? OUT_F32 : OUT_U32, s);
}

}  // namespace prng
