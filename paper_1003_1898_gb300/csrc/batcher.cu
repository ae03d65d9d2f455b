// batcher.cu -- prng_batcher_*: a reusable batched-fill engine whose request
// set changes from launch to launch (the serving loop's per-tick pass).
//
// prng_batch_* plans one fixed request list and replays it as a graph.  A
// server instead forms a new set every tick from whatever has arrived, so
// the batcher owns a ring of NSLOT staging slots sized for a maximum number
// of requests and work items: each launch plans the new set into the next
// slot (pinned host buffers), copies it to the slot's device buffers, zeroes
// the slot's work counters and launches the family kernels on the caller's
// stream.  A slot is reused only after the launch that last used it has
// finished (its event), so the host can plan tick t+1 while tick t runs.
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/prng.h"
#include "plan.cuh"
#include "scratch.cuh"

using namespace prng;

namespace {

constexpr int kSlots = 4;

struct Slot {
  BatchReq* h_reqs = nullptr;     // pinned
  BatchItem* h_items = nullptr;   // pinned
  uint32_t* h_firsts = nullptr;   // pinned; items that begin a group of RANLUX segments
  uint32_t* d_firsts = nullptr;
  CUtensorMap* h_maps = nullptr;  // pinned; outputs of the tensor-core RANLUX requests
  BatchReq* d_reqs = nullptr;
  BatchItem* d_items = nullptr;
  CUtensorMap* d_maps = nullptr;
  uint32_t* d_counters = nullptr;
  cudaEvent_t done = nullptr;
  bool pending = false;
};


}  // namespace

struct prng_batcher {
  uint32_t max_requests = 0;
  uint64_t max_items = 0;
  Slot slot[kSlots];
  int next = 0;
  std::vector<const prng_state*> handles;   // duplicate check, sized once
  std::vector<uint64_t> order, sorted;      // requests, longest rows first: 2^32 - 1 - length, index
};

namespace {

// Sorts keys whose low words are already in order, by their high words: byte by
// byte, those that all keys share left out.  (Comparing the requests themselves
// took a third of a launch of 1,000 short ones.)
void sort_keys(std::vector<uint64_t>& keys, std::vector<uint64_t>& tmp) {
  if (keys.size() < 2) return;
  uint64_t differ = 0;
  for (uint64_t k : keys) differ |= k ^ keys[0];
  tmp.resize(keys.size());   // within its reserve
  for (int shift = 32; shift < 64; shift += 8) {
    if (((differ >> shift) & 255) == 0) continue;
    uint32_t at[257] = {};
    for (uint64_t k : keys) at[((k >> shift) & 255) + 1]++;
    for (int i = 0; i < 256; i++) at[i + 1] += at[i];
    for (uint64_t k : keys) tmp[at[(k >> shift) & 255]++] = k;
    keys.swap(tmp);
  }
}

void destroy_batcher(prng_batcher* b) {
  if (b == nullptr) return;
  for (auto& u : b->slot) {
    // The event of a captured launch cannot be waited for; the error stays here.
    if (u.pending && u.done && cudaEventSynchronize(u.done) != cudaSuccess) cudaGetLastError();
    if (u.done) cudaEventDestroy(u.done);
    if (u.h_reqs) cudaFreeHost(u.h_reqs);
    if (u.h_items) cudaFreeHost(u.h_items);
    if (u.h_firsts) cudaFreeHost(u.h_firsts);
    if (u.d_firsts) cudaFree(u.d_firsts);
    if (u.h_maps) cudaFreeHost(u.h_maps);
    if (u.d_maps) cudaFree(u.d_maps);
    if (u.d_reqs) cudaFree(u.d_reqs);
    if (u.d_items) cudaFree(u.d_items);
    if (u.d_counters) cudaFree(u.d_counters);
  }
  delete b;
}

}  // namespace

extern "C" {

int prng_batcher_create(prng_batcher** out, uint32_t max_requests, uint64_t max_items) {
  if (out == nullptr) return PRNG_ENULL;
  *out = nullptr;
  if (max_requests == 0 || max_items == 0 || max_items > 0xFFFFFFFFull) return PRNG_ESIZE;
  prng_batcher* b = new (std::nothrow) prng_batcher;
  if (b == nullptr) return PRNG_EALLOC;
  b->max_requests = max_requests;
  b->max_items = max_items;
  try {
    b->handles.reserve(max_requests);
    b->order.reserve(max_requests);
    b->sorted.reserve(max_requests);
  } catch (...) {
    delete b;
    return PRNG_EALLOC;
  }
  for (auto& u : b->slot) {
    if (cudaMallocHost(&u.h_reqs, max_requests * sizeof(BatchReq)) != cudaSuccess ||
        cudaMallocHost(&u.h_items, max_items * sizeof(BatchItem)) != cudaSuccess ||
        cudaMallocHost(&u.h_firsts, max_items * sizeof(uint32_t)) != cudaSuccess ||
        cudaMalloc(&u.d_firsts, max_items * sizeof(uint32_t)) != cudaSuccess ||
        cudaMallocHost(&u.h_maps, max_requests * sizeof(CUtensorMap)) != cudaSuccess ||
        cudaMalloc(&u.d_maps, max_requests * sizeof(CUtensorMap)) != cudaSuccess ||
        cudaMalloc(&u.d_reqs, max_requests * sizeof(BatchReq)) != cudaSuccess ||
        cudaMalloc(&u.d_items, max_items * sizeof(BatchItem)) != cudaSuccess ||
        cudaMalloc(&u.d_counters, FAM_COUNT * sizeof(uint32_t)) != cudaSuccess) {
      cudaGetLastError();
      destroy_batcher(b);
      return PRNG_EALLOC;
    }
    if (cudaEventCreateWithFlags(&u.done, cudaEventDisableTiming) != cudaSuccess) {
      destroy_batcher(b);
      return PRNG_ECUDA;
    }
  }
  *out = b;
  return PRNG_OK;
}

int prng_batcher_launch(prng_batcher* b, const prng_fill_req* reqs, uint32_t n_reqs, void* stream) {
  if (b == nullptr) return PRNG_ENULL;
  if (n_reqs == 0) return PRNG_OK;
  if (reqs == nullptr) return PRNG_ENULL;
  if (n_reqs > b->max_requests) return PRNG_ESIZE;
  for (uint32_t i = 0; i < n_reqs; i++) {
    const prng_fill_req& r = reqs[i];
    if (r.st == nullptr) return PRNG_ENULL;
    if (r.n_per_stream > 0 && r.d_out == nullptr) return PRNG_ENULL;
    if ((reinterpret_cast<uintptr_t>(r.d_out) & 3) != 0) return PRNG_ESIZE;
    if (r.n_per_stream > 0 && r.st->n_streams > UINT64_MAX / r.n_per_stream) return PRNG_ESIZE;
    if (handle_failed(r.st)) return PRNG_ECUDA;
  }
  // Items per family: RANLUX streams cut into segments where the slot has room
  // for them, whole otherwise.
  ItemPlan plan;
  uint64_t fam_n[FAM_COUNT], total = 0;
  uint32_t fam_off[FAM_COUNT];
  auto count = [&](bool cut) {
    plan.choose(reqs, n_reqs, cut);
    std::fill(fam_n, fam_n + FAM_COUNT, 0);
    for (uint32_t i = 0; i < n_reqs; i++) {
      const prng_fill_req& r = reqs[i];
      if (r.reseed) fam_n[FAM_SEED] += (r.st->n_streams + plan.seed_rows(r.st) - 1) / plan.seed_rows(r.st);
      if (r.n_per_stream == 0) continue;
      const int f = fill_family(r.st->gen, r.st->p, r.f32 != 0);
      fam_n[f] += plan.count(f, r.st, r.n_per_stream);
    }
    total = 0;
    for (int f = 0; f < FAM_COUNT; f++) {
      fam_off[f] = (uint32_t)std::min<uint64_t>(total, b->max_items);
      total += fam_n[f];
    }
    return total <= b->max_items;
  };
  if (!count(true)) count(false);
  if (total > b->max_items) return PRNG_ESIZE;
  // A handle may appear once per launch (its streams advance once): sorted
  // copy of the handles, adjacent equal ones rejected.
  b->handles.clear();
  for (uint32_t i = 0; i < n_reqs; i++) b->handles.push_back(reqs[i].st);
  std::sort(b->handles.begin(), b->handles.end());
  if (std::adjacent_find(b->handles.begin(), b->handles.end()) != b->handles.end()) return PRNG_EBLOB;

  Slot& u = b->slot[b->next];
  if (u.pending) {
    if (cudaEventSynchronize(u.done) != cudaSuccess) return PRNG_ECUDA;
    u.pending = false;
  }
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint32_t* starts = nullptr;   // of the RANLUX segments, for this launch
  uint64_t lux_items = 0;
  for (int f = 0; f < FAM_COUNT; f++)
    if (plan.is_lux_tc(f)) lux_items += fam_n[f];
  // A captured launch takes no scratch, as captured fills: an allocation would
  // become a node of the graph, which could then be instantiated once only.
  if (lux_items > 0 &&
      (capturing(s) ||
       scratch_alloc(reinterpret_cast<void**>(&starts), lux_start_bytes(lux_items), s) != cudaSuccess)) {
    cudaGetLastError();
    starts = nullptr;
    plan.tensor = false;        // the borrow chain, with no more items than uncut streams
    count(false);
  }
  bool maps = false;
  uint32_t at[FAM_COUNT];
  std::memcpy(at, fam_off, sizeof(at));
  for (uint32_t i = 0; i < n_reqs; i++) {
    const prng_fill_req& r = reqs[i];
    prng_state* st = r.st;
    BatchReq& q = u.h_reqs[i];
    const uint64_t full = st->n_streams * r.n_per_stream;
    std::memset(&q, 0, sizeof(q));
    q.d.state = st->d_state;
    q.d.out = r.d_out;
    q.d.n_rows = st->n_streams;
    q.d.n_per = r.n_per_stream;
    q.d.pitch = r.n_per_stream;
    q.d.limit = (r.n_valid == 0 || r.n_valid > full) ? full : r.n_valid;
    q.d.pos = r.reseed ? initial_pos(st->gen) : st->pos;
    q.d.p = st->p;
    q.d.x0 = fill_multiplier(st->gen, r.n_per_stream);
    q.d.mode = r.f32 ? OUT_F32 : OUT_U32;
    q.seed = r.seed;
    q.gen = st->gen;
    q.reseed = r.reseed ? 1 : 0;
    st->pos = advance_pos(st->gen, q.d.pos, r.n_per_stream);
    if (r.reseed) {
      const uint32_t per = plan.seed_rows(st);
      for (uint64_t r0 = 0; r0 < st->n_streams; r0 += per)
        u.h_items[at[FAM_SEED]++] = BatchItem{i, (uint32_t)std::min<uint64_t>(per, st->n_streams - r0), r0};
    }
    if (r.n_per_stream > 0) {
      const int f = fill_family(r.st->gen, r.st->p, r.f32 != 0);
      if (plan.is_lux_tc(f)) {
        q.tiles = request_map(r, &u.h_maps[i]) ? 1 : 0;
        maps = true;
      }
    }
  }
  // Items, the requests with the longest rows first (a request's items all cost
  // the same but for the last, so ordering the requests orders the items).
  b->order.clear();
  for (uint32_t i = 0; i < n_reqs; i++)
    if (reqs[i].n_per_stream > 0)
      b->order.push_back((UINT32_MAX - std::min<uint64_t>(reqs[i].n_per_stream, UINT32_MAX)) << 32 | i);
  sort_keys(b->order, b->sorted);
  for (uint64_t key : b->order) {
    const uint32_t i = (uint32_t)key;
    const prng_fill_req& r = reqs[i];
    const int f = fill_family(r.st->gen, r.st->p, r.f32 != 0);
    plan.items(f, i, r.st, r.n_per_stream, [&](const BatchItem& it) { u.h_items[at[f]++] = it; });
  }
  uint32_t groups[FAM_COUNT] = {}, group0[FAM_COUNT] = {}, n_firsts = 0;
  for (int f = 0; f < FAM_COUNT; f++) {
    if (!plan.is_lux_tc(f) || plan.max_seg[f] == 0) continue;
    group0[f] = n_firsts;
    for (uint32_t k = 0; k < fam_n[f]; k++)
      if (plan.first(u.h_items[fam_off[f] + k])) u.h_firsts[n_firsts++] = k;
    groups[f] = n_firsts - group0[f];
  }
  auto fail = [&](int rc) {
    cudaGetLastError();
    if (starts != nullptr) scratch_free(starts, s);
    return rc;
  };
  if (cudaMemcpyAsync(u.d_reqs, u.h_reqs, n_reqs * sizeof(BatchReq), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      (total > 0 && cudaMemcpyAsync(u.d_items, u.h_items, total * sizeof(BatchItem),
                                    cudaMemcpyHostToDevice, s) != cudaSuccess) ||
      (n_firsts > 0 && cudaMemcpyAsync(u.d_firsts, u.h_firsts, n_firsts * sizeof(uint32_t), cudaMemcpyHostToDevice,
                                       s) != cudaSuccess) ||
      (maps && cudaMemcpyAsync(u.d_maps, u.h_maps, n_reqs * sizeof(CUtensorMap), cudaMemcpyHostToDevice, s) !=
                   cudaSuccess) ||
      cudaMemsetAsync(u.d_counters, 0, FAM_COUNT * sizeof(uint32_t), s) != cudaSuccess)
    return fail(PRNG_ECUDA);
  auto queue = [&](int f) {
    return BatchQueue{u.d_reqs, u.d_items + fam_off[f], (uint32_t)fam_n[f], u.d_counters + f};
  };
  cudaError_t e = launch_batch_seed(queue(FAM_SEED), s);
  uint64_t lux_at = 0;
  for (int f = FAM_MLCG; f < FAM_COUNT && e == cudaSuccess; f++) {
    if (fam_n[f] == 0) continue;
    uint32_t* st = nullptr;
    if (plan.is_lux_tc(f)) {
      st = starts + lux_start_bytes(lux_at) / sizeof(uint32_t);
      lux_at += fam_n[f];
    }
    e = launch_family(f, queue(f), plan, u.d_maps, st, u.d_firsts + group0[f], groups[f], s);
  }
  if (e != cudaSuccess) return fail(PRNG_ECUDA);
  if (starts != nullptr && scratch_free(starts, s) != cudaSuccess) return PRNG_ECUDA;
  if (cudaEventRecord(u.done, s) != cudaSuccess) return PRNG_ECUDA;
  u.pending = true;
  b->next = (b->next + 1) % kSlots;
  return PRNG_OK;
}

void prng_batcher_destroy(prng_batcher* b) { destroy_batcher(b); }

}  // extern "C"
