// Eviction for streaming tables (Section 1, "Dynamic Features": under an endless stream the set of live
// features changes over time; Section 5, "Dynamic Hash Table").  The paper's table has lookup, insert and
// update; a table that can only grow fits no memory for long, so keys can be removed here: by list, or by
// age (rows carry the table's clock value of their insertion / last update).
//
// A maintenance operation, not part of the training step: it synchronises on entry and once at the end.
//   mark      a bit per row to go (by probing the listed keys, or by comparing age stamps), the counts per
//             shard, and the list of the slots concerned
//   starts    for every removed key, the start of the run of occupied slots it lies in; shards that need a rebuild
//   pair      the freed rows below a shard's new size m (ascending) are paired with the surviving rows at or
//             beyond m (ascending): one block per shard walks the shard's bits in order
//   move      the surviving row's weights and state are copied into the freed row
//   repair    linear probing must never meet a deleted slot, and there are no tombstones: the run of
//             occupied slots around a removed key is put back in order by one thread.  Runs are disjoint
//             and short (a handful of slots at load 0.5), so this costs per removed key, not per key of the table
//             (emptying and refilling the shards' regions took 107 us for 0.25 M of 1.25 M keys; this takes 25 us and
//             its cost does not grow with the table).
//   relabel   survivors that changed rows get their new row number (one pass over the slots, only when any did)
// A shard whose region is rebuilt instead (all threads take part: collected, emptied, put back): one with a run of more than
// EV_RUN slots around a removed key, which one thread would walk and probe for milliseconds; one without an empty slot;
// and one that holds keys without a row (their insert met a full shard), which an eviction drops.
// The host learns the outcome with one copy at the end; nothing in between waits for it, and the temporaries
// stay with the table unless they are large (allocating and freeing them took 1.8 ms a call).  Only where a shard is rebuilt
// nothing is changed before that copy, so that the memory for it is there before the first row moves.
// Every loop is bounded (probes by the region size); a full region raises the sticky status word.
#include <cstdlib>

#include "des_internal.cuh"

#define EV_NONE 0xFFFFFFFFu
#define EV_KEEP_BYTES (64ull << 20)                    // temporaries up to this size stay allocated with the table
#ifdef DES_DEBUG
#define EV_RUN 64u                                     // (checking build: small tables get there)
#else
#define EV_RUN 2048u                                   // slots of the longest run that one thread repairs
#endif

struct EvictCtl {                                      // zero at the start of a call
  uint32_t gone[DES_MAX_SHARDS];                       // rows to go
  uint32_t pairs[DES_MAX_SHARDS];                      // rows that move
  uint32_t n_list;                                     // slots of keys to go
  uint32_t owned[DES_MAX_SHARDS];                      // a run of the shard has found its start
  uint32_t rebuild[DES_MAX_SHARDS];                    // a run is too long, or there are keys without a row
  uint32_t any_pairs;
  uint32_t n_live;                                     // (rebuild only)
};

struct __align__(16) LiveKey { unsigned long long key; uint32_t row, shard; };

__device__ __forceinline__ int shard_of_pos(const unsigned long long* __restrict__ base, int S, unsigned long long i) {
  int lo = 0, hi = S;                                  // base[lo] <= i < base[hi]
  while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (base[mid] <= i) lo = mid; else hi = mid; }
  return lo;
}

// the rows' bits: shard s starts a word of its own at word row_base[s] / 32 + s
__device__ __forceinline__ unsigned long long ev_word0(const DevMeta* __restrict__ meta, int s) {
  return (meta->row_base[s] >> 5) + (unsigned long long)s;
}
__device__ __forceinline__ bool ev_gone(const uint32_t* __restrict__ bits, const DevMeta* __restrict__ meta, int s, uint32_t row) {
  return (bits[ev_word0(meta, s) + (row >> 5)] >> (row & 31)) & 1u;
}
__device__ __forceinline__ uint32_t ev_append(uint32_t* counter, bool want) {   // whole warp; position for the lanes that want
  const unsigned m = __ballot_sync(0xFFFFFFFFu, want);
  const int lane = threadIdx.x & 31;
  uint32_t base = 0;
  if (m && lane == __ffs(m) - 1) base = atomicAdd(counter, __popc(m));
  base = __shfl_sync(0xFFFFFFFFu, base, m ? __ffs(m) - 1 : 0);
  return base + __popc(m & ((1u << lane) - 1u));
}

// A shard that loses keys has a run that starts behind an empty slot — unless its region has no empty slot at all.
__host__ __device__ __forceinline__ bool ev_rebuilt(const EvictCtl* ctl, int s) {
  return ctl->gone[s] && (!ctl->owned[s] || ctl->rebuild[s]);
}
// The kernels that change the table are launched once, and again (`planned`) when the host has seen that a shard is to
// be rebuilt: the first time they then do nothing.  Whole block.
__device__ __forceinline__ bool ev_wait(const EvictCtl* ctl, int S, int planned) {
  bool any = false;
  if (!planned) for (int s = threadIdx.x; s < S; s += blockDim.x) any |= ev_rebuilt(ctl, s);
  return __syncthreads_or(any);
}

// by list: one thread per key (HASH: the key's own shard; FIELD: thread (key, shard) looks in every shard)
__global__ void __launch_bounds__(256) evict_mark_keys_kernel(const unsigned long long* __restrict__ keys, long long n,
                                                              int S, int partition, uint32_t mod_M, uint32_t mod_two32,
                                                              const Slot* __restrict__ slots, const DevMeta* __restrict__ meta,
                                                              uint32_t* __restrict__ bits, uint32_t* __restrict__ list,
                                                              EvictCtl* ctl) {
  __shared__ uint32_t cnt[DES_MAX_SHARDS];
  for (int i = threadIdx.x; i < S; i += 256) cnt[i] = 0;
  __syncthreads();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long per = partition == DES_PART_HASH ? 1 : S;
  uint32_t slot = EV_NONE;
  if (i < n * per) {
    const unsigned long long key = keys[i / per];
    const unsigned long long h = des_mix64(key);
    const uint32_t s = partition == DES_PART_HASH ? des_mod_small(h, (uint32_t)S, mod_M, mod_two32) : (uint32_t)(i % per);
    const uint32_t lo = (uint32_t)meta->slot_base[s], hi = (uint32_t)meta->slot_base[s + 1], cap = hi - lo;
    uint32_t cur = des_slot_home(h, lo, cap);
    for (uint32_t probe = 0; key != DES_KEY_EMPTY && probe < cap; ++probe) {
      const Slot sl = slots[cur];
      if (sl.key == key) {
        if (sl.row != DES_ROW_NONE && sl.row < meta->n_rows[s]) {
          const uint32_t bit = 1u << (sl.row & 31);
          if (!(atomicOr(bits + ev_word0(meta, s) + (sl.row >> 5), bit) & bit)) {   // (a key listed twice goes once)
            slot = cur;
            atomicAdd(&cnt[s], 1u);
          }
        }
        break;
      }
      if (sl.key == DES_KEY_EMPTY) break;
      cur = cur + 1 == hi ? lo : cur + 1;
    }
  }
  const uint32_t at = ev_append(&ctl->n_list, slot != EV_NONE);
  if (slot != EV_NONE) list[at] = slot;
  __syncthreads();
  for (int s = threadIdx.x; s < S; s += 256) if (cnt[s]) atomicAdd(&ctl->gone[s], cnt[s]);
}

// by age: one warp per word of 32 rows
__global__ void __launch_bounds__(256) evict_mark_stale_kernel(const float* __restrict__ W, int k, int stride, int S,
                                                              unsigned long long n_words, uint32_t min_clock,
                                                              const DevMeta* __restrict__ meta, uint32_t* __restrict__ bits,
                                                              EvictCtl* ctl) {
  const unsigned long long w = (unsigned long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w >= n_words) return;                            // whole warp
  int lo = 0, hi = S;                                  // the shard whose words hold w
  while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (ev_word0(meta, mid) <= w) lo = mid; else hi = mid; }
  const int lane = threadIdx.x & 31;
  const unsigned long long row = (w - ev_word0(meta, lo)) * 32 + lane;
  const bool dead = row < meta->n_rows[lo] && __float_as_uint(W[(meta->row_base[lo] + row) * stride + k + 2]) < min_clock;
  const unsigned m = __ballot_sync(0xFFFFFFFFu, dead);
  if (lane == 0 && m) { bits[w] = m; atomicAdd(&ctl->gone[lo], __popc(m)); }
}

// by age: the slots of the marked rows
__global__ void __launch_bounds__(256) evict_list_kernel(const Slot* __restrict__ slots, unsigned long long total_slots, int S,
                                                        const DevMeta* __restrict__ meta, const uint32_t* __restrict__ bits,
                                                        uint32_t* __restrict__ list, EvictCtl* ctl) {
  const unsigned long long st = (unsigned long long)gridDim.x * blockDim.x;
  const unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long rounds = (total_slots + st - 1) / st;       // whole warps
  for (unsigned long long r = 0; r < rounds; ++r) {
    const unsigned long long i = i0 + r * st;
    bool dead = false;
    if (i < total_slots) {
      const Slot sl = slots[i];
      if (sl.key != DES_KEY_EMPTY && sl.row != DES_ROW_NONE) dead = ev_gone(bits, meta, shard_of_pos(meta->slot_base, S, i), sl.row);
    }
    const uint32_t at = ev_append(&ctl->n_list, dead);
    if (dead) list[at] = (uint32_t)i;
  }
}

// where shard s's lists of freed and moving rows start: each shard needs at most min(rows to go, rows that stay)
__device__ __forceinline__ unsigned long long ev_list_off(const DevMeta* __restrict__ meta, const EvictCtl* ctl, int s) {
  unsigned long long off = 0;
  for (int i = 0; i < s; ++i) off += min(ctl->gone[i], meta->n_rows[i] - ctl->gone[i]);
  return off;
}

// one block per shard walks its bits in ascending order, 1024 words at a time: freed rows below the new size and
// surviving rows at or beyond it, each list in ascending order
__global__ void __launch_bounds__(1024) evict_pair_kernel(const uint32_t* __restrict__ bits, const DevMeta* __restrict__ meta,
                                                          EvictCtl* ctl, uint32_t* __restrict__ holes,
                                                          uint32_t* __restrict__ movers) {
  __shared__ uint32_t wh[32], wm[32], carry_h, carry_m;
  const int s = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t e = ctl->gone[s];
  if (e == 0) return;
  const uint32_t n = meta->n_rows[s], m = n - e;
  const uint32_t* b = bits + ev_word0(meta, s);
  const unsigned long long off = ev_list_off(meta, ctl, s);
  if (threadIdx.x == 0) { carry_h = 0; carry_m = 0; }
  __syncthreads();
  const uint32_t nw = (n + 31) / 32;
  auto below = [](uint32_t w, uint32_t x) { return x <= w * 32 ? 0u : x >= w * 32 + 32 ? 0xFFFFFFFFu : (1u << (x - w * 32)) - 1u; };
  for (uint32_t chunk = 0; chunk < nw; chunk += 1024) {
    const uint32_t w = chunk + threadIdx.x;
    uint32_t hb = 0, mb = 0;                            // bits: freed rows below m; surviving rows in [m, n)
    if (w < nw) {
      const uint32_t v = b[w], bm = below(w, m);
      hb = v & bm;
      mb = ~v & ~bm & below(w, n);
    }
    uint32_t ih = __popc(hb), im = __popc(mb);
    const uint32_t ch = ih, cm = im;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, ih, d), y = __shfl_up_sync(0xFFFFFFFFu, im, d);
      if (lane >= d) { ih += x; im += y; }
    }
    if (lane == 31) { wh[warp] = ih; wm[warp] = im; }
    __syncthreads();
    uint32_t ph = carry_h, pm = carry_m;
    for (int i = 0; i < warp; ++i) { ph += wh[i]; pm += wm[i]; }
    unsigned long long oh = off + ph + ih - ch, om = off + pm + im - cm;
    for (; hb; hb &= hb - 1) holes[oh++] = w * 32 + __ffs(hb) - 1;
    for (; mb; mb &= mb - 1) movers[om++] = w * 32 + __ffs(mb) - 1;
    __syncthreads();
    if (threadIdx.x == 1023) { carry_h = ph + ih; carry_m = pm + im; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {                               // (as many freed rows below m as survivors beyond it)
    ctl->pairs[s] = carry_h;
    if (carry_h) ctl->any_pairs = 1u;
  }
}

// one warp per pair: the surviving row's weights and state move into the freed row
__global__ void __launch_bounds__(256) evict_move_kernel(const DevMeta* __restrict__ meta, const EvictCtl* ctl,
                                                         const uint32_t* __restrict__ holes, const uint32_t* __restrict__ movers,
                                                         int S, int planned, int stride, float* W, float* A, float* A2) {
  if (ev_wait(ctl, S, planned)) return;
  const int s = blockIdx.y, lane = threadIdx.x & 31;
  const uint32_t np = ctl->pairs[s];
  if (np == 0) return;
  const unsigned long long base = meta->row_base[s], off = ev_list_off(meta, ctl, s);
  for (uint32_t i = blockIdx.x * 8 + (threadIdx.x >> 5); i < np; i += gridDim.x * 8) {
    const unsigned long long to = base + holes[off + i], from = base + movers[off + i];
    for (int c = lane; c < stride; c += 32) {
      W[to * stride + c] = W[from * stride + c];
      if (A) A[to * stride + c] = A[from * stride + c];
      if (A2) A2[to * stride + c] = A2[from * stride + c];
    }
  }
}

// list[i]: a removed key's slot -> the first slot of the run of occupied slots it lies in, or EV_NONE when another
// removed key of the same run comes before it (that one repairs the run).  Reads only.
__global__ void __launch_bounds__(256) evict_starts_kernel(const Slot* __restrict__ slots, int S, const DevMeta* __restrict__ meta,
                                                          const uint32_t* __restrict__ bits, const uint32_t* __restrict__ list,
                                                          uint32_t* __restrict__ starts, EvictCtl* ctl) {
  const uint32_t n = ctl->n_list;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t cur = list[i];
    const int s = shard_of_pos(meta->slot_base, S, cur);
    const uint32_t lo = (uint32_t)meta->slot_base[s], hi = (uint32_t)meta->slot_base[s + 1], cap = hi - lo;
    uint32_t start = EV_NONE, len = 1;
    bool rebuild = meta->rowless[s];
    while (!rebuild && len < cap) {                     // back to the run's start
      const uint32_t prev = cur == lo ? hi - 1 : cur - 1;
      const Slot sl = slots[prev];
      if (sl.key == DES_KEY_EMPTY) { start = cur; break; }
      if (sl.row != DES_ROW_NONE && ev_gone(bits, meta, s, sl.row)) break;
      cur = prev;
      rebuild = ++len > EV_RUN;
    }
    cur = list[i];
    while (!rebuild && start != EV_NONE) {              // on to its end: an empty slot, at the latest the one before the start
      cur = cur + 1 == hi ? lo : cur + 1;
      if (slots[cur].key == DES_KEY_EMPTY) break;
      rebuild = ++len > EV_RUN;
    }
    starts[i] = rebuild ? EV_NONE : start;
    if (rebuild && !ctl->rebuild[s]) ctl->rebuild[s] = 1u;
    if (start != EV_NONE && !ctl->owned[s]) ctl->owned[s] = 1u;
  }
}

// Slots of a run are taken out one after the other and, unless removed, put back from their home slot: everything
// between the home and the slot just emptied has been through this, so a key never lands behind where it was,
// and the result is what inserting the survivors in that order gives.
__global__ void __launch_bounds__(128) evict_repair_kernel(Slot* slots, int S, const DevMeta* __restrict__ meta,
                                                          const uint32_t* __restrict__ bits, const uint32_t* __restrict__ starts,
                                                          const EvictCtl* ctl, int planned) {
  if (ev_wait(ctl, S, planned)) return;
  const uint32_t n = ctl->n_list;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t cur = starts[i];
    if (cur == EV_NONE) continue;
    const int s = shard_of_pos(meta->slot_base, S, cur);
    if (ev_rebuilt(ctl, s)) continue;
    const uint32_t lo = (uint32_t)meta->slot_base[s], hi = (uint32_t)meta->slot_base[s + 1], cap = hi - lo;
    Slot empty; empty.key = DES_KEY_EMPTY; empty.row = DES_ROW_NONE; empty.first_occ = DES_ROW_NONE;
    for (uint32_t step = 0; step < cap; ++step) {
      const Slot sl = slots[cur];
      if (sl.key == DES_KEY_EMPTY) break;               // the run's end
      if (ev_gone(bits, meta, s, sl.row)) {
        slots[cur] = empty;
      } else {
        uint32_t at = des_slot_home(des_mix64(sl.key), lo, cap);
        for (uint32_t p = 0; p < cap && at != cur && slots[at].key != DES_KEY_EMPTY; ++p) at = at + 1 == hi ? lo : at + 1;
        if (at != cur) { slots[at] = sl; slots[cur] = empty; }
      }
      cur = cur + 1 == hi ? lo : cur + 1;
    }
  }
}

// survivors that changed rows
__global__ void __launch_bounds__(256) evict_relabel_kernel(Slot* slots, unsigned long long total_slots, int S,
                                                           const DevMeta* __restrict__ meta, const EvictCtl* ctl,
                                                           const uint32_t* __restrict__ holes, const uint32_t* __restrict__ movers,
                                                           int planned) {
  if (!ctl->any_pairs || ev_wait(ctl, S, planned)) return;
  __shared__ unsigned long long off[DES_MAX_SHARDS];
  for (int s = threadIdx.x; s < S; s += blockDim.x) off[s] = ev_list_off(meta, ctl, s);
  __syncthreads();
  unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long st = (unsigned long long)gridDim.x * blockDim.x;
  for (; i < total_slots; i += st) {
    const Slot sl = slots[i];
    if (sl.key == DES_KEY_EMPTY || sl.row == DES_ROW_NONE) continue;
    const int s = shard_of_pos(meta->slot_base, S, i);
    if (sl.row < meta->n_rows[s] - ctl->gone[s] || !ctl->pairs[s] || ev_rebuilt(ctl, s)) continue;
    const uint32_t* mv = movers + off[s];
    uint32_t a = 0, b = ctl->pairs[s];                  // mv[a] <= row < mv[b]: the row is in the list
    while (b - a > 1) { const uint32_t mid = (a + b) >> 1; if (mv[mid] <= sl.row) a = mid; else b = mid; }
    slots[i].row = holes[off[s] + a];
  }
}

__global__ void evict_finish_kernel(DevMeta* meta, const EvictCtl* ctl, int S) {
  const int s = threadIdx.x;
  if (s >= S) return;
  meta->n_rows[s] -= ctl->gone[s];
  if (ev_rebuilt(ctl, s)) meta->rowless[s] = 0u;
}

// Rebuilt shards: the survivors are collected, the regions emptied, the survivors put back.  Runs before evict_finish_kernel.
__global__ void __launch_bounds__(256) evict_collect_kernel(const Slot* __restrict__ slots, unsigned long long total_slots,
                                                            int S, const DevMeta* __restrict__ meta, EvictCtl* ctl,
                                                            const uint32_t* __restrict__ bits, const uint32_t* __restrict__ holes,
                                                            const uint32_t* __restrict__ movers, LiveKey* __restrict__ live) {
  unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long st = (unsigned long long)gridDim.x * blockDim.x;
  for (; i < total_slots; i += st) {
    const int s = shard_of_pos(meta->slot_base, S, i);
    if (!ev_rebuilt(ctl, s)) continue;
    const Slot sl = slots[i];
    if (sl.key == DES_KEY_EMPTY || sl.row == DES_ROW_NONE || ev_gone(bits, meta, s, sl.row)) continue;
    LiveKey lk; lk.key = sl.key; lk.row = sl.row; lk.shard = (uint32_t)s;
    if (sl.row >= meta->n_rows[s] - ctl->gone[s]) {
      const unsigned long long off = ev_list_off(meta, ctl, s);
      uint32_t a = 0, b = ctl->pairs[s];
      while (b - a > 1) { const uint32_t mid = (a + b) >> 1; if (movers[off + mid] <= sl.row) a = mid; else b = mid; }
      lk.row = holes[off + a];
    }
    live[atomicAdd(&ctl->n_live, 1u)] = lk;
  }
}

__global__ void __launch_bounds__(256) evict_clear_kernel(Slot* slots, unsigned long long total_slots, int S,
                                                          const DevMeta* __restrict__ meta, const EvictCtl* ctl) {
  unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long st = (unsigned long long)gridDim.x * blockDim.x;
  for (; i < total_slots; i += st) {
    if (!ev_rebuilt(ctl, shard_of_pos(meta->slot_base, S, i))) continue;
    Slot e; e.key = DES_KEY_EMPTY; e.row = DES_ROW_NONE; e.first_occ = DES_ROW_NONE;
    slots[i] = e;
  }
}

__global__ void __launch_bounds__(256) evict_reinsert_kernel(Slot* slots, DevMeta* meta, const LiveKey* __restrict__ live,
                                                             const EvictCtl* ctl) {
  const uint32_t n = ctl->n_live;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const LiveKey lk = live[i];
    const uint32_t lo = (uint32_t)meta->slot_base[lk.shard], hi = (uint32_t)meta->slot_base[lk.shard + 1], cnt = hi - lo;
    uint32_t cur = des_slot_home(des_mix64(lk.key), lo, cnt);
    bool placed = false;
    for (uint32_t probe = 0; probe < cnt && !placed; ++probe) {
      if (atomicCAS(&slots[cur].key, DES_KEY_EMPTY, lk.key) == DES_KEY_EMPTY) {
        slots[cur].row = lk.row;                       // (first_occ stays at "never touched")
        placed = true;
      }
      cur = cur + 1 == hi ? lo : cur + 1;
    }
    if (!placed) des_raise(meta, DES_ERR_CAPACITY);      // cannot happen: the region held these keys before
  }
}

static bool ev_no_memory() {
#ifdef DES_DEBUG
  return getenv("DES_DEBUG_EVICT_NO_MEMORY") != nullptr;   // checking build only: the memory for a rebuild is not to be had
#else
  return false;
#endif
}

static des_status_t evict_run(des_table_t* t, const uint64_t* d_keys, int64_t n, uint64_t min_clock, int by_age,
                              uint64_t* h_n_evicted) {
  if (h_n_evicted) *h_n_evicted = 0;
  int dev = 0;
  DES_CUDA(cudaGetDevice(&dev));
  if (dev != t->device) return DES_ERR_INVALID_ARG;
  DES_CUDA(cudaDeviceSynchronize());
  des_api_begin(t, 0);
  if (!by_age && n == 0) return DES_OK;
  const int S = (int)t->S;
  // temporaries: [ctl | bits] cleared per call, then the lists
  const uint64_t n_words = t->total_rows / 32 + S + 1;
  const uint64_t per = t->cfg.partition == DES_PART_HASH ? 1 : S;
  const uint64_t most = by_age || (uint64_t)n * per > t->total_rows ? t->total_rows : (uint64_t)n * per;   // rows to go
  const uint64_t most_pairs = most < t->total_rows / 2 + 1 ? most : t->total_rows / 2 + 1;
  const size_t clear = ((sizeof(EvictCtl) + n_words * 4) + 255) / 256 * 256;
  const size_t bytes = clear + (2 * most + 2 * most_pairs) * 4;
  unsigned char* ws = (unsigned char*)t->evict_ws;
  if (bytes > t->evict_ws_bytes) {
    cudaFree(ws);
    t->evict_ws = nullptr; t->evict_ws_bytes = 0;
    ws = nullptr;
    if (cudaMalloc(&ws, bytes) != cudaSuccess) { cudaGetLastError(); return DES_ERR_CUDA; }
    if (bytes <= EV_KEEP_BYTES) { t->evict_ws = ws; t->evict_ws_bytes = bytes; }
  }
  LiveKey* live = nullptr;
  auto bail = [&](des_status_t code) {
    if (code != DES_OK) { cudaDeviceSynchronize(); cudaGetLastError(); }
    if ((void*)ws != t->evict_ws) cudaFree(ws);
    cudaFree(live);
    return code;
  };
#define EV_CUDA(x) do { if ((x) != cudaSuccess) return bail(DES_ERR_CUDA); } while (0)
#define EV_LAUNCH(name) do { if (des_prof_mark(t, name, 1)) return bail(DES_ERR_CUDA); } while (0)
  EvictCtl* ctl = (EvictCtl*)ws;
  uint32_t* bits = (uint32_t*)(ws + sizeof(EvictCtl));
  uint32_t *list = (uint32_t*)(ws + clear), *starts = list + most, *holes = starts + most, *movers = holes + most_pairs;
  const unsigned wide = (unsigned)(t->sm_count * 8);
  EV_CUDA(cudaMemsetAsync(ws, 0, clear, 0));
  if (by_age) {
    const uint32_t mc = min_clock > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)min_clock;
    evict_mark_stale_kernel<<<(unsigned)((n_words + 7) / 8), 256>>>(t->W, (int)t->k, (int)t->stride, S, n_words, mc, t->meta, bits, ctl);
    EV_LAUNCH("evict_mark_stale_kernel");
    evict_list_kernel<<<wide, 256>>>(t->slots, t->total_slots, S, t->meta, bits, list, ctl);
    EV_LAUNCH("evict_list_kernel");
  } else {
    uint32_t M, two32;
    des_mod_consts(t->S, &M, &two32);
    evict_mark_keys_kernel<<<(unsigned)((n * per + 255) / 256), 256>>>((const unsigned long long*)d_keys, n, S,
                                                                      (int)t->cfg.partition, M, two32, t->slots, t->meta, bits, list, ctl);
    EV_LAUNCH("evict_mark_keys_kernel");
  }
  evict_starts_kernel<<<wide, 256>>>(t->slots, S, t->meta, bits, list, starts, ctl);
  EV_LAUNCH("evict_starts_kernel");
  evict_pair_kernel<<<S, 1024>>>(bits, t->meta, ctl, holes, movers);
  EV_LAUNCH("evict_pair_kernel");
  auto change = [&](int planned) {
    evict_move_kernel<<<dim3((unsigned)((t->sm_count * 8 + S - 1) / S), (unsigned)S), 256>>>(t->meta, ctl, holes, movers, S, planned,
                                                                                           (int)t->stride, t->W, t->A, t->A2);
    if (des_prof_mark(t, "evict_move_kernel", 1)) return false;
    evict_repair_kernel<<<wide * 2, 128>>>(t->slots, S, t->meta, bits, starts, ctl, planned);
    if (des_prof_mark(t, "evict_repair_kernel", 1)) return false;
    evict_relabel_kernel<<<wide, 256>>>(t->slots, t->total_slots, S, t->meta, ctl, holes, movers, planned);
    return !des_prof_mark(t, "evict_relabel_kernel", 1);
  };
  if (!change(0)) return bail(DES_ERR_CUDA);
  EvictCtl h;
  EV_CUDA(cudaMemcpy(&h, ctl, sizeof(h), cudaMemcpyDeviceToHost));
  uint64_t n_live = 0;                                 // rows of the shards to rebuild
  bool rebuild = false;
  for (int s = 0; s < S; ++s)
    if (ev_rebuilt(&h, s)) { rebuild = true; n_live += t->h_row_base[s + 1] - t->h_row_base[s]; }
  if (rebuild) {
    if (ev_no_memory() || cudaMalloc(&live, n_live * sizeof(LiveKey)) != cudaSuccess) { live = nullptr; return bail(DES_ERR_CUDA); }
    if (!change(1)) return bail(DES_ERR_CUDA);
    evict_collect_kernel<<<wide, 256>>>(t->slots, t->total_slots, S, t->meta, ctl, bits, holes, movers, live);
    EV_LAUNCH("evict_collect_kernel");
    evict_clear_kernel<<<wide, 256>>>(t->slots, t->total_slots, S, t->meta, ctl);
    EV_LAUNCH("evict_clear_kernel");
    evict_reinsert_kernel<<<wide, 256>>>(t->slots, t->meta, live, ctl);
    EV_LAUNCH("evict_reinsert_kernel");
  }
  evict_finish_kernel<<<1, DES_MAX_SHARDS>>>(t->meta, ctl, S);
  EV_LAUNCH("evict_finish_kernel");
  EV_CUDA(cudaDeviceSynchronize());
#undef EV_CUDA
#undef EV_LAUNCH
  uint64_t total = 0;
  for (int s = 0; s < S; ++s) total += h.gone[s];
  if (h_n_evicted) *h_n_evicted = total;
  return bail(DES_OK);
}

extern "C" des_status_t des_table_evict_keys(des_table_t* t, const uint64_t* d_keys, int64_t n, uint64_t* h_n_evicted) {
  if (!t || n < 0 || (n > 0 && !d_keys)) return DES_ERR_INVALID_ARG;
  return evict_run(t, d_keys, n, 0, 0, h_n_evicted);
}

extern "C" des_status_t des_table_evict_stale(des_table_t* t, uint64_t min_clock, uint64_t* h_n_evicted) {
  if (!t) return DES_ERR_INVALID_ARG;
  return evict_run(t, nullptr, 0, min_clock, 1, h_n_evicted);
}

extern "C" des_status_t des_table_clock(des_table_t* t, uint64_t* h_clock) {
  if (!t || !h_clock) return DES_ERR_INVALID_ARG;
  DES_CUDA(cudaDeviceSynchronize());
  unsigned long long c = 0;
  DES_CUDA(cudaMemcpy(&c, &t->meta->clock, 8, cudaMemcpyDeviceToHost));
  *h_clock = c;
  return DES_OK;
}
