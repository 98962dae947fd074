// Kernels of the batched prefix-cache step (PrefixShield, arXiv 2608.01657).
//
// One step is a fixed sequence of launches on the caller's stream.  Nothing on
// the path goes back to the host: every size (tokens, blocks, claims, victims)
// lives in device memory, grids are sized from the handle's bounds, and a
// thread whose item does not exist exits at once.  Apart from the one-CTA
// scans, every stage runs a thread per block position, per request or per
// victim, so a long prompt is spread over many warps instead of serializing
// one.  Each kernel's comment names the stage and the passage it implements.
#include <climits>
#include <cstdio>

#include <vector>

#include "ps_device.cuh"
#include "ps_launch.cuh"

namespace ps {

constexpr int kFinCap = 8192;  // split lists up to this size are finished by one CTA in shared memory
constexpr int kFinRows = 32;   // rows k_list_finish counts at once (32 KB)
constexpr int kFinCountCap = 512;  // split lists up to this size may be ranked by counting,
constexpr int kFinShort = 128;     // and up to this size are

// 128-bit compare-and-swap (sm_90+): installs the (p, group) identity of a
// history entry atomically, so two requests of one (group, prefix) that race
// to insert it agree on the slot.
__device__ __forceinline__ void cas128(void* addr, uint64_t exp_lo, uint64_t exp_hi, uint64_t new_lo,
                                       uint64_t new_hi, uint64_t* old_lo, uint64_t* old_hi) {
  uint64_t lo, hi;
  asm volatile(
      "{\n\t.reg .b128 e, n, d;\n\t"
      "mov.b128 e, {%2, %3};\n\t"
      "mov.b128 n, {%4, %5};\n\t"
      "atom.global.cas.b128 d, [%6], e, n;\n\t"
      "mov.b128 {%0, %1}, d;\n\t}"
      : "=l"(lo), "=l"(hi)
      : "l"(exp_lo), "l"(exp_hi), "l"(new_lo), "l"(new_hi), "l"(addr)
      : "memory");
  *old_lo = lo;
  *old_hi = hi;
}

__device__ __forceinline__ uint64_t step_tag(uint64_t step, uint32_t req) {
  return (step << 32) | (uint64_t)(0xFFFFFFFFu - req);
}
// The request index stored in a step tag, or UINT32_MAX if the tag is older.
__device__ __forceinline__ uint32_t tag_req(uint64_t tag, uint64_t step) {
  return (tag >> 32) == step ? 0xFFFFFFFFu - (uint32_t)tag : 0xFFFFFFFFu;
}
__device__ __forceinline__ int64_t refill(int64_t b, int64_t beta, int64_t rho, int64_t dt) {
  // Eq. 1, min{beta, b + rho*dt}, without overflow and without a division.
  // rho*dt >= need decides it; a product past 64 bits is past any need.
  const int64_t need = beta - b;
  const uint64_t add = (uint64_t)rho * (uint64_t)dt;
  if (need <= 0 || __umul64hi((uint64_t)rho, (uint64_t)dt) != 0 || add >= (uint64_t)need) return beta;
  return b + (int64_t)add;
}
// floor(a * b / c) for a >= 0 and 0 < b <= c.  A 128-bit division is a call of
// about a microsecond, so the cases without one go first: nothing owed, equal
// rates (one contract, or the slowest one), a product that fits 64 bits.
__device__ __forceinline__ int64_t muldiv(int64_t a, int64_t b, int64_t c) {
  if (a == 0) return 0;
  if (b == c) return a;
  if (__umul64hi((uint64_t)a, (uint64_t)b) == 0) return (int64_t)(((uint64_t)a * (uint64_t)b) / (uint64_t)c);
  return (int64_t)(((__int128)a * (__int128)b) / (__int128)c);
}

// ---- arithmetic modulo p = 2^61 - 1 (Mersenne reduction: 2^61 == 1) ------
__device__ __forceinline__ uint64_t red61(uint64_t x) {  // any 64-bit x -> [0, p)
  const uint64_t r = (x & kP61) + (x >> 61);
  return r >= kP61 ? r - kP61 : r;
}
// A chain of products keeps its values below p + 8 instead of below p, and
// reduces fully only where a value leaves it: k x + c from four 32-bit
// products and one reduction is half the instructions of a full product, a
// full sum and their two compares and subtractions.
__device__ __forceinline__ uint64_t weak61(uint64_t x) { return (x & kP61) + (x >> 61); }  // any 64-bit x -> <= p + 7
__device__ __forceinline__ uint64_t mad61(uint64_t k, uint64_t x, uint64_t c) {  // k < p, x <= p + 7, c <= 2 (p + 7)
  const uint32_t k0 = (uint32_t)k, k1 = (uint32_t)(k >> 32), x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32);  // x1 <= 2^29
  const uint64_t mid = (uint64_t)k0 * x1 + (uint64_t)k1 * x0, low = (uint64_t)k0 * x0;                    // mid <= 2^62
  uint64_t r = (uint64_t)(k1 << 3) * x1 + c;  // 2^64 = 8 (mod p); at most 3 2^61 so far, 5 2^61 in all
  r += (low & kP61) + (low >> 61);
  r += ((uint64_t)((uint32_t)mid & 0x1FFFFFFFu) << 32) + (mid >> 29);  // 2^32 mid
  return weak61(r);
}

// ---- native prefix table ---------------------------------------------------
// Lookup by one thread: the home bucket's 32-byte tag sector (a 16-bit tag per
// way, and the overflow count), then the entry of each way whose tag matches,
// then following buckets while the overflow count says some key probed past.
// A miss reads one sector instead of the whole 128-byte bucket, a hit one more:
// at 2^20 blocks the tags are 16 MB, which stay in L2, beside a 64 MB table.
// Tags are never cleared (a delete that cleared one could land after a later
// insert's): a stale tag costs a look at an empty or another key's entry.
__device__ __forceinline__ uint32_t table_tag(uint64_t key, uint32_t g) {
  const uint64_t x = (key ^ ((uint64_t)(g + 1) * 0x9E3779B97F4A7C15ull)) * 0xD6E8FEB86659FD93ull;
  const uint32_t t = (uint32_t)(x >> 16) & 0xFFFFu;  // away from the bits that choose the bucket
  return t ? t : 1u;
}
// The ways of a bucket whose tag matches: way 2k at bit k, way 2k + 1 at bit
// 16 + k; and the way of the lowest such bit.
__device__ __forceinline__ uint32_t tag_matches(const uint4& t, uint32_t tag) {
  const uint32_t t2 = tag * 0x10001u;
  return (__vcmpeq2(t.x, t2) & 0x10001u) | (__vcmpeq2(t.y, t2) & 0x20002u) | (__vcmpeq2(t.z, t2) & 0x40004u) |
         (__vcmpeq2(t.w, t2) & 0x80008u);
}
__device__ __forceinline__ uint32_t tag_bit(uint32_t w) { return 1u << ((w >> 1) + 16 * (w & 1)); }
__device__ __forceinline__ int tag_way(uint32_t m) {
  const int k = __ffs((int)m) - 1;
  return k < 16 ? 2 * k : 2 * (k - 16) + 1;
}
__device__ uint32_t table_find(const DevState& s, uint64_t key, uint32_t g) {
  const uint32_t mask = (1u << s.tb_nbuckets_log2) - 1;
  const uint32_t tag = table_tag(key, g);
  uint32_t b = table_home(key, g, s.tb_nbuckets_log2);
  for (uint32_t it = 0; it <= mask; ++it) {
    const uint4 tg = __ldg(reinterpret_cast<const uint4*>(s.tags + b));
    const uint32_t ovf = __ldg(&s.tags[b].ovf);  // issued with the tags: a miss needs no second trip
    for (uint32_t m = tag_matches(tg, tag); m; m &= m - 1) {
      const uint4 raw = __ldg(reinterpret_cast<const uint4*>(s.table + (size_t)b * kTableWays + tag_way(m)));
      if (raw.z != kNone && raw.x == (uint32_t)key && raw.y == (uint32_t)(key >> 32) && raw.w == g) return raw.z;
    }
    if (ovf == 0) return kNone;
    b = (b + 1) & mask;
  }
  return kNone;
}

// The way of its home bucket where a key's insertion tries first.
__device__ __forceinline__ uint32_t table_way0(uint64_t key) { return (uint32_t)(key >> 7) & (kTableWays - 1); }

// The same for two keys of a thread, in one round of loads where possible:
// both tag sectors and, beside them, the entry each key's insertion tries
// first (at a quarter load it is usually there).  The first entry of another
// matching way costs a second trip; a key not settled by these (several ways'
// tags match, or keys probed past the bucket) takes the general walk.
__device__ __forceinline__ void table_find2(const DevState& s, uint64_t keyA, uint64_t keyB, uint32_t g, bool doA,
                                            bool doB, uint32_t* blkA, uint32_t* blkB) {
  const uint32_t bA = table_home(keyA, g, s.tb_nbuckets_log2), bB = table_home(keyB, g, s.tb_nbuckets_log2);
  const uint32_t wA = table_way0(keyA), wB = table_way0(keyB);
  uint4 tA = make_uint4(0, 0, 0, 0), tB = tA, eA = make_uint4(0, 0, kNone, 0), eB = eA;
  uint32_t oA = 0, oB = 0;
  if (doA) {
    tA = __ldg(reinterpret_cast<const uint4*>(s.tags + bA));
    oA = __ldg(&s.tags[bA].ovf);
    eA = __ldg(reinterpret_cast<const uint4*>(s.table + (size_t)bA * kTableWays + wA));
  }
  if (doB) {
    tB = __ldg(reinterpret_cast<const uint4*>(s.tags + bB));
    oB = __ldg(&s.tags[bB].ovf);
    eB = __ldg(reinterpret_cast<const uint4*>(s.table + (size_t)bB * kTableWays + wB));
  }
  auto is_key = [&](const uint4& e, uint64_t key) {
    return e.z != kNone && e.x == (uint32_t)key && e.y == (uint32_t)(key >> 32) && e.w == g;
  };
  bool hitA = is_key(eA, keyA), hitB = is_key(eB, keyB);
  // other ways with the key's tag
  const uint32_t mA = hitA ? 0u : tag_matches(tA, table_tag(keyA, g)) & ~tag_bit(wA);
  const uint32_t mB = hitB ? 0u : tag_matches(tB, table_tag(keyB, g)) & ~tag_bit(wB);
  if (mA) {
    eA = __ldg(reinterpret_cast<const uint4*>(s.table + (size_t)bA * kTableWays + tag_way(mA)));
    hitA = is_key(eA, keyA);
  }
  if (mB) {
    eB = __ldg(reinterpret_cast<const uint4*>(s.table + (size_t)bB * kTableWays + tag_way(mB)));
    hitB = is_key(eB, keyB);
  }
  *blkA = hitA ? eA.z : ((mA & (mA - 1)) != 0 || oA != 0 ? table_find(s, keyA, g) : kNone);
  *blkB = hitB ? eB.z : ((mB & (mB - 1)) != 0 || oB != 0 ? table_find(s, keyB, g) : kNone);
}

// Returns the slot, with kDisplaced set when it lies past the home bucket
// (then a delete must repair the overflow counters on the way).  The swap
// starts at a way chosen by the key's own bits: at a quarter load that way
// is usually free, so most inserts take one atomic and no load.  (No key is
// inserted twice, so no swaps pile up on one way.)
constexpr uint32_t kDisplaced = 0x80000000u;
__device__ uint32_t table_insert(const DevState& s, uint64_t key, uint32_t g, uint32_t blk) {
  const uint32_t mask = (1u << s.tb_nbuckets_log2) - 1;
  uint32_t b = table_home(key, g, s.tb_nbuckets_log2);
  const uint32_t w0 = table_way0(key);
  const uint16_t tag = (uint16_t)table_tag(key, g);
  for (uint32_t it = 0; it <= mask; ++it) {
    TableEntry* e = s.table + (size_t)b * kTableWays;
    for (int q = 0; q < kTableWays; ++q) {
      const int w = (int)((w0 + (uint32_t)q) & (kTableWays - 1));
      if (atomicCAS(&e[w].blk, kNone, blk) == kNone) {
        e[w].key = key;
        e[w].grp = g;
        s.tags[b].tag[w] = tag;
        return (b * kTableWays + w) | (it ? kDisplaced : 0u);
      }
    }
    atomicAdd(&s.tags[b].ovf, 1u);
    b = (b + 1) & mask;
  }
  return kNone;  // unreachable: the table is at most a quarter full
}

// An entry is empty exactly when its block field is kNone (lookups test it
// first), so a delete clears only that field: an insert that takes the slot
// at once then writes its own key and group, and no late clearing store of
// the delete can land on them.
// The same from the block's record as already loaded (slot with its flag,
// key, group).
__device__ __forceinline__ void table_delete_known(const DevState& s, uint32_t tagged, uint64_t key, uint32_t g) {
  const uint32_t mask = (1u << s.tb_nbuckets_log2) - 1;
  const uint32_t slot = tagged & ~kDisplaced;
  s.table[slot].blk = kNone;
  if (!(tagged & kDisplaced)) return;  // in its home bucket: no counter passed
  const uint32_t bucket = slot / kTableWays;
  uint32_t x = table_home(key, g, s.tb_nbuckets_log2);
  for (uint32_t it = 0; x != bucket && it <= mask; ++it, x = (x + 1) & mask) atomicSub(&s.tags[x].ovf, 1u);
}
__device__ void table_delete(const DevState& s, uint32_t blk) {
  const uint32_t mask = (1u << s.tb_nbuckets_log2) - 1;
  const uint32_t tagged = s.blk_slot[blk];
  const uint32_t slot = tagged & ~kDisplaced;
  s.table[slot].blk = kNone;
  if (!(tagged & kDisplaced)) return;  // in its home bucket: no counter passed
  const uint32_t bucket = slot / kTableWays;
  uint32_t x = table_home(s.blk_key[blk], s.blk_group[blk], s.tb_nbuckets_log2);
  for (uint32_t it = 0; x != bucket && it <= mask; ++it, x = (x + 1) & mask) atomicSub(&s.tags[x].ovf, 1u);
}

// ---- per-step claim map ------------------------------------------------------
// The bucket's keys are loaded first, so the many requests that claim one
// popular key in a step mostly find it with a plain load and swap nothing
// (a swap first would serialize them on one address).  Keys kept apart from
// the entries, a bucket's in one sector, took 171 us a step at 2^20 blocks
// against 155: a second scattered line a claim costs more than the sectors.
__device__ uint32_t claim_insert(const DevState& s, uint64_t key, uint32_t req) {
  const uint32_t mask = (1u << s.cl_nbuckets_log2) - 1;
  uint32_t b = claim_home(key, s.cl_nbuckets_log2);
  for (uint32_t it = 0; it <= mask; ++it) {
    // the bucket's keys in one round of loads.  Keys only arrive during a
    // step, each in the first free way, so walking the ways in order with a
    // CAS on each free one meets the key wherever another thread put it.
    ClaimEntry* e = s.claims + (size_t)b * kClaimWays;
    uint64_t cur[kClaimWays];
#pragma unroll
    for (int w = 0; w < kClaimWays; ++w) cur[w] = ldcg_u64(&e[w].key);
#pragma unroll
    for (int w = 0; w < kClaimWays; ++w) {
      uint64_t v = cur[w];
      if (v == 0) v = atomicCAS(reinterpret_cast<unsigned long long*>(&e[w].key), 0ull, (unsigned long long)key);
      if (v == 0 || v == key) {
        atomicMin(&e[w].minreq, req);
        return b * kClaimWays + w;
      }
    }
    b = (b + 1) & mask;
  }
  return kNone;  // unreachable: the map has a slot for every block of a step
}

// ---- block state changes -----------------------------------------------------
// Remove a resident block from the pool (eviction or invalidation); returns
// its group.  Callers account the per-group statistics, warp-aggregated.
// clear_res: also clear the resident bit (evictions leave it: the id is
// allocated again in the same step, and k_bm_write sets the allocated bits).
__device__ uint32_t drop_block(const DevState& s, uint32_t b, bool clear_res = true) {
  table_delete(s, b);
  const uint32_t g = s.blk_group[b];
  s.blk_flags[b] = 0;
  if (clear_res) atomicAnd(s.res_bits + (b >> 5), ~(1u << (b & 31)));
  return g;
}

// Position -> (request, position within the request).
struct PosRef {
  uint32_t i;
  int m;
};
__device__ __forceinline__ bool pos_ref(const DevState& s, int64_t pos, PosRef* r) {
  if (pos >= s.ctl->nblocks) return false;
  r->i = s.pos_req[pos];  // both loads in one round trip
  r->m = (int)s.pos_m[pos];
  return true;
}
// The position of a position-parallel kernel, false past the step's blocks or
// in a failed step.  The step's status and size and the position's record are
// loaded in one round trip: the records reach to max_blocks whatever the
// step's size, so they may be loaded before it is known.  (A status looked at
// first cost every such kernel two trips before its work began.)
__device__ __forceinline__ bool pos_open(const DevState& s, const Ctl* c, int64_t pos, PosRef* r) {
  const int32_t st = c->status;
  const int64_t nb = c->nblocks;
  const bool in = pos < s.max_blocks;
  r->i = in ? s.pos_req[pos] : 0u;
  r->m = in ? (int)s.pos_m[pos] : 0;
  return st == PS_OK && pos < nb;
}

// ===========================================================================
// Init: an empty pool, every balance at beta (Sec. III-B, B = beta at t = 0).
__global__ void k_init_blocks(DevState s) {
  const int64_t nclaims = (int64_t)kClaimWays << s.cl_nbuckets_log2;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nclaims; c += (int64_t)gridDim.x * blockDim.x) {
    s.claims[c] = empty_claim();
  }
}
__global__ void k_init_ctl(DevState s) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    Ctl c{};
    c.step = 1;
    c.stamp_base = 1;
    *s.ctl = c;
  }
  for (int i = threadIdx.x; i < s.G * s.C; i += blockDim.x) s.ledger[i] = s.beta[i % s.C];
}

// ===========================================================================
// Stage 0: validation of the step's inputs; n_i, block positions and the
// chunk descriptors of the hashing stage.  One CTA per kValTile requests;
// the exclusive scans of blocks and chunks over the requests take each
// tile's base from its predecessors' published totals (a decoupled look-back
// without inclusive prefixes: a tile sums every earlier tile's total, and no
// total waits on anything).  The last CTA to finish sets the call's status
// and per-step scalars, and clears the tile words for the next call.
// A probe (probe_status set: where its outcome goes) skips the clock and step
// checks.  Every write is bounds-checked, so
// inputs that turn out invalid write nothing outside the scratch arrays.
// A warp's requests' chunk descriptors, a lane per chunk: its request is found
// among the warp's by the chunks before it, and the request's values come by
// shuffles (a loop over the requests took a pass of mostly idle lanes each).
__device__ __forceinline__ void write_chunks(const DevState& s, int32_t ns, int32_t n, int64_t o0, int32_t sbase,
                                             int32_t pbase, uint32_t i, uint32_t g) {
  const int lane = lane_id();
  const int32_t incl = warp_incl_scan(ns), ex = incl - ns;
  const int32_t tot = __shfl_sync(kFull, incl, 31);
  for (int q0 = 0; q0 < tot; q0 += 32) {
    const int q = q0 + lane;
    int src = 0;  // the last request with at most q chunks before it
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (__shfl_sync(kFull, ex, src + st) <= q) src += st;
    ChunkDesc d;
    d.o0 = __shfl_sync(kFull, o0, src);
    d.req = __shfl_sync(kFull, i, src);
    d.n = __shfl_sync(kFull, n, src);
    d.pbase = __shfl_sync(kFull, pbase, src);
    d.k = q - __shfl_sync(kFull, ex, src);
    d.group = __shfl_sync(kFull, g, src);
    d.sb = __shfl_sync(kFull, sbase, src);
    if (q < tot) {
      s.chunks[d.sb + d.k] = d;
      s.seg_word[d.sb + d.k] = 0;
    }
  }
}

constexpr uint64_t kTileFlag = 1ull << 63;

__global__ void __launch_bounds__(kValTile) k_validate(DevState s, int32_t* probe_status) {
  s = with_args(s);
  __shared__ uint64_t s_base;
  __shared__ bool s_last;
  const bool probe = probe_status != nullptr;
  Ctl* c = s.ctl;
  const int R = s.R;
  const int tile = blockIdx.x;
  const int i = tile * kValTile + (int)threadIdx.x;
  const bool in = i < R;
  bool bad = false;
  int32_t n = 0, ns = 0, cid = 0, g = 0;
  int64_t o0 = 0;
  if (in) {
    o0 = s.in_offsets[i];
    const int64_t o1 = s.in_offsets[i + 1];
    g = s.in_group[i];
    const int64_t nb = (o1 - o0) >> (__ffs(s.bs) - 1);  // a power of two
    bad = o1 < o0 || g < 0 || g >= s.G || nb > (int64_t)kMaxPos;
    if (s.in_contract) {
      cid = s.in_contract[i];
      bad |= cid < 0 || cid >= s.C;
    } else if (!probe && !bad) {
      cid = s.contract_of_group[g];
    }
    if (s.in_prefix) bad |= s.in_prefix[i] == 0;
    n = bad ? 0 : (int32_t)nb;
  }
  ns = (n + kChunkBlocks - 1) / kChunkBlocks;
  const int tile_bad = __syncthreads_or(bad);
  // blocks in the high half, chunks in the low half of one scanned word
  uint64_t tot;
  const uint64_t ex = block_excl_scan<uint64_t>((uint64_t)n << 32 | (uint64_t)ns, &tot);
  if (threadIdx.x == 0) st_relaxed_u64(s.val_tile + tile, tot | kTileFlag);
  if (threadIdx.x < 32 && tile * kValTile < R) {  // the tile's base: every earlier tile's total
    const int lane = threadIdx.x;
    uint64_t sum = 0;
    bool ok = true;
    for (int t0 = 0; t0 < tile; t0 += 32) {
      if (t0 + lane < tile) {
        const uint64_t v = wait_word(s.val_tile + t0 + lane, kTileFlag);
        ok = ok && v != 0;
        sum += v & ~kTileFlag;
      }
    }
    sum = warp_sum(sum);
    if (!__all_sync(kFull, ok) && lane == 0) atomicOr(&c->v_bad, 2u);  // never expected
    if (lane == 0) s_base = sum;
  } else if (threadIdx.x == 0) {
    s_base = 0;  // a tile past the step's requests writes nothing
  }
  __syncthreads();
  const uint64_t e = s_base + ex;
  const int64_t pbase = (int64_t)(e >> 32), sbase = (int64_t)(uint32_t)e;
  if (in && pbase + n <= s.max_blocks && sbase + ns <= s.max_segments) {
    s.rq_n[i] = n;
    s.rq_h[i] = n;
    s.rq_s[i] = n;
    s.rq_fu[i] = kNone;
    s.rq_pbase[i] = (int32_t)pbase;
    if (!probe) {
      s.rq_cid[i] = cid;
      s.rq_hs[i] = kNone;  // a request with no full block has no history entry
      s.rq_p[i] = 0;
    }
  }
  write_chunks(s, in && pbase + n <= s.max_blocks && sbase + ns <= s.max_segments ? ns : 0, n, o0, (int32_t)sbase,
               (int32_t)pbase, (uint32_t)i, (uint32_t)g);
  if (!probe && tile == 0) {  // per-step counts accumulated by later kernels
    if (s.policy == PS_STATICQUOTA)
      for (int gg = threadIdx.x; gg < s.G; gg += blockDim.x) s.grp_pinned[gg] = 0;
    for (int r = threadIdx.x; r < s.G * kClasses; r += blockDim.x) {  // the candidate counts (k_cand)
      if (r < s.G) s.grp_qsize[r] = 0;
      s.cls[r] = ClsRange{0, ~0u, 0, ~0u, 0};
    }
  }
  // the last CTA to finish: status and per-call scalars
  if (threadIdx.x == 0) {
    if (tile_bad) atomicOr(&c->v_bad, 1u);
    if (tot) atomicAdd(reinterpret_cast<unsigned long long*>(&c->v_sum), (unsigned long long)tot);
    __threadfence();
    s_last = atomicAdd(&c->v_ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int t = threadIdx.x; t < (int)gridDim.x; t += blockDim.x) s.val_tile[t] = 0;
  if (threadIdx.x != 0) return;
  // every value the verdict needs, loaded up front so the loads overlap
  const uint32_t vb = ldcg_u32(&c->v_bad);
  const uint64_t all = ldcg_u64(&c->v_sum);  // blocks (high half) and chunks (low half) of the step
  const int64_t T = R > 0 ? s.in_offsets[R] : 0;
  const int64_t first_off = R > 0 ? s.in_offsets[0] : 0;
  const int32_t sticky = c->sticky, lost = c->lg_lost;
  const int64_t t_prev = c->t_prev;
  const uint64_t step = c->step;
  c->v_bad = 0;
  c->v_ticket = 0;
  c->v_sum = 0;
  int32_t st = PS_OK;
  if (!probe && sticky != PS_OK) st = sticky;
  else if (!probe && lost) st = PS_ERR_DEVICE_STATUS;
  else if (!probe && s.now < t_prev) st = PS_ERR_CLOCK;
  else if (!probe && step > kMaxStep) st = PS_ERR_CAPACITY;
  else if (vb || first_off != 0 || T > s.max_tokens) st = PS_ERR_INVALID_ARG;
  c->status = st;
  if (probe) *probe_status = st;
  c->T = T;
  c->hash_ticket = 0;
  if (st != PS_OK) {
    c->nblocks = 0;
    c->nsegs = 0;
    return;
  }
  c->nblocks = (int64_t)(all >> 32);
  c->nsegs = (int64_t)(uint32_t)all;
  if (!probe) {
    c->pinned = 0; c->n_inval = 0; c->total_claims = 0; c->avail = 0; c->need = 0;
    c->nfree = 0; c->ftake = 0; c->mvict = 0; c->hist_new = 0; c->n_evicted = 0;
    c->n_alloc = 0; c->m_fb = 0; c->sel_ntie = 0; c->sel_k = 0; c->ticket = 0;
    c->internal_error = (vb & 2) ? 1 : 0;
    c->nlaunch = 1;  // this kernel; every later kernel of the step adds itself
  }
}

// ===========================================================================
// Stages 1-2 in one kernel: chained block hashing (Sec. III-B native content
// key), the longest cached prefix (n_cached of Alg. 1), the pins of the
// cached prefix, the claims of every block past it, and each request's
// history entry (OnRequest of Alg. 1).
//
// A chunk is up to kChunkBlocks = 64 consecutive blocks of one prompt; one
// warp takes one chunk, lane l its blocks l and 32 + l (two halves).  Chunks
// are numbered in request order (a request's chunks are consecutive) and CTAs
// draw their chunks in that order from a ticket, so every chunk's
// predecessors belong to warps that have already started.  Each lane reads
// its blocks' tokens with 16-byte loads and forms the block digests D_m
// itself.  The chain C_m = Kc C_{m-1} + D_m (mod 2^61 - 1) composes affine
// maps, so a warp scan of each half gives each block its chain value B_m
// relative to the half's start (value 0 entering it); the chunk's total, the
// second half's total plus Kc^(its blocks) times the first's, is published
// under a flag.  (Two blocks a lane halve the chunks, and with them the
// chain of dependent accesses each one pays: ticket, descriptor,
// predecessors' totals and miss bits.)  The value entering chunk k of a
// request is then
//   Kc^(64k) C_seed + sum_{l<k} Kc^(64(k-1-l)) total_l,
// and no total waits on anything, so the warp folds its k predecessors'
// totals directly, in windows of 32 (one lane each).  With C_m the lanes form
// their keys and probe the table.  A block is in the cached prefix iff no
// block before it in its request misses: the chunk's "some block missed" bit
// is the second published flag, and the warp ORs its predecessors'.  The
// cached prefix is pinned for the step; every block past it is claimed in the
// claim map (lowest request index wins: one materialization, one charge, I1).
// The warp of a request's first chunk installs the request's history entry.
//
// Each chunk publishes one 64-bit word (seg_word, zeroed per call by
// k_validate): bits 0-60 its chain total (a value mod 2^61 - 1), bit 61 set
// once the total is there, bit 62 once its miss bit (bit 63) is.  Value and
// flags travel in one aligned 64-bit store, read with one relaxed 64-bit
// load, so no fence orders them.  Every wait is bounded; a wait that runs
// out reports an internal error.
constexpr uint64_t kWordTotal = 1ull << 61, kWordMiss = 1ull << 62, kWordMissBit = 1ull << 63;
// A chunk descriptor in two 16-byte loads.
__device__ __forceinline__ ChunkDesc load_chunk(const ChunkDesc* p) {
  const uint4 a = __ldg(reinterpret_cast<const uint4*>(p)), b = __ldg(reinterpret_cast<const uint4*>(p) + 1);
  ChunkDesc d;
  d.o0 = (int64_t)((uint64_t)a.y << 32 | a.x);
  d.req = a.z;
  d.n = (int32_t)a.w;
  d.pbase = (int32_t)b.x;
  d.k = (int32_t)b.y;
  d.group = b.z;
  d.sb = (int32_t)b.w;
  return d;
}

// NH sums over a piece of PIECE tokens held in w[] from word OFF on (OFF the
// warp-uniform word offset, a compile-time constant in each of four forms),
// with key words from pair index kk0 on.  Summing straight from w[] keeps
// no second, re-indexed copy of the tokens live.
template <int OFF, int PIECE, int NWORDS>
__device__ __forceinline__ void nh_piece(const uint32_t (&w)[NWORDS], const uint32_t* sk, int kk0, uint64_t* a1,
                                         uint64_t* a2) {
#pragma unroll
  for (int k = 0; k < PIECE / 2; ++k) {
    const int kk = kk0 + k;
    const uint32_t tx = w[OFF + 2 * k], ty = w[OFF + 2 * k + 1];
    *a1 += (uint64_t)(tx + sk[2 * kk]) * (uint64_t)(ty + sk[2 * kk + 1]);
    *a2 += (uint64_t)(tx + sk[2 * kk + 2]) * (uint64_t)(ty + sk[2 * kk + 3]);
  }
}

// The two NH sums of one block (bs tokens from token index g0).  r is the
// request's word offset (g0 mod 4, the same for all its blocks); with a
// 16-byte aligned token buffer the block's tokens are read as the 16-byte
// words that cover them, 16 tokens at a time, otherwise token by token (as
// they are near the step's last token, where the covering words could pass
// it).
template <int BS>
__device__ __forceinline__ void block_nh(const DevState& s, const uint32_t* sk, int64_t g0, int r, bool vec, int64_t T,
                                         uint64_t* d1, uint64_t* d2) {
  constexpr int PIECE = BS < 16 ? BS : 16;  // tokens per piece
  uint64_t a1 = 0, a2 = 0;
#pragma unroll
  for (int q0 = 0; q0 < BS; q0 += PIECE) {
    const int64_t a0 = g0 + q0 - r;
    bool done = false;
    if constexpr (PIECE % 4 == 0) {
      constexpr int NW = PIECE / 4 + 1;  // 16-byte words covering a piece at any word offset
      if (vec && a0 + 4 * NW <= T) {
        uint32_t w[4 * NW];
        const uint4* src = reinterpret_cast<const uint4*>(s.in_tokens + a0);
#pragma unroll
        for (int q = 0; q < NW; ++q) {
          const uint4 v = __ldg(src + q);
          w[4 * q] = v.x;
          w[4 * q + 1] = v.y;
          w[4 * q + 2] = v.z;
          w[4 * q + 3] = v.w;
        }
        switch (r) {  // warp-uniform
          case 0: nh_piece<0, PIECE>(w, sk, q0 / 2, &a1, &a2); break;
          case 1: nh_piece<1, PIECE>(w, sk, q0 / 2, &a1, &a2); break;
          case 2: nh_piece<2, PIECE>(w, sk, q0 / 2, &a1, &a2); break;
          default: nh_piece<3, PIECE>(w, sk, q0 / 2, &a1, &a2); break;
        }
        done = true;
      }
    }
    if (!done) {
      uint32_t w[PIECE];
#pragma unroll
      for (int j = 0; j < PIECE; ++j) w[j] = (uint32_t)s.in_tokens[g0 + q0 + j];
      nh_piece<0, PIECE>(w, sk, q0 / 2, &a1, &a2);
    }
  }
  *d1 = a1;
  *d2 = a2;
}

// One chunk (j) of k_hash_lookup, by one warp.  Returns false if a wait for
// a predecessor ran out (never expected).
template <int BS>
__device__ __forceinline__ bool hash_lookup_chunk(const DevState& s, Ctl* c, const uint32_t* sk, const uint64_t* kc,
                                                  int64_t j, int32_t* probe_out) {
  const int lane = lane_id();
  const ChunkDesc d = load_chunk(s.chunks + j);
  const uint32_t i = d.req;
  const int n = d.n;
  const int64_t sb = d.sb;
  const int k = d.k;  // chunk index within the request
  const int m0 = k * kChunkBlocks;
  const int nb = tmin(kChunkBlocks, n - m0);
  const int nbA = tmin(kSegBlocks, nb), nbB = nb - nbA;  // blocks of the two halves
  const int64_t o0 = d.o0;
  const int pbase = d.pbase;
  const uint32_t g = d.group;
  const int64_t T = c->T;
  const int mA = m0 + lane, mB = m0 + kSegBlocks + lane;
  // D_m of the lane's two blocks, then the inclusive scans of the affine maps
  // x -> Kc x + D, one per half
  uint64_t bA = 0, bB = 0;
  // The halves' digests in a rolled loop: half the code, and no spills with
  // blocks of up to 16 tokens (32 and 64 spill 20 bytes a thread): 155.2 -> 152.8
  // us a step at 2^20 blocks; it cost 0.4 us with a few chunks in all.
  // The second half's tokens are on their way from DRAM meanwhile (-> 152.2).
  if (lane < nbB) {
    const int32_t* src = s.in_tokens + o0 + (int64_t)mB * BS;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
    if (BS >= 16) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + BS / 2));
  }
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
    uint64_t D = 0;
    if (lane < (half ? nbB : nbA)) {
      uint64_t d1, d2;
      block_nh<BS>(s, sk, o0 + (int64_t)(half ? mB : mA) * BS, (int)(o0 & 3), s.tokens_aligned16 != 0, T, &d1, &d2);
      D = mad61(s.digest_mul, weak61(d2), weak61(d1));
    }
    if (half) bB = D;
    else bA = D;
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const uint64_t tA = __shfl_up_sync(kFull, bA, 1 << q);
    const uint64_t tB = __shfl_up_sync(kFull, bB, 1 << q);
    if (lane >= (1 << q)) {
      bA = mad61(kc[1 << q], tA, bA);
      bB = mad61(kc[1 << q], tB, bB);
    }
  }
  const uint64_t totA = __shfl_sync(kFull, bA, nbA - 1);
  const uint64_t totB = __shfl_sync(kFull, bB, nbB > 0 ? nbB - 1 : 0);
  // a second half follows a full first half (Kc^32 times it)
  const uint64_t total = red61(nbB > 0 ? mad61(kc[nbB], totA, totB) : totA);
  if (lane == 0) st_relaxed_u64(s.seg_word + j, total | kWordTotal);
  // the chain value entering the chunk
  bool ok = true;
  uint64_t cin = red61(chain_seed(s.hash_seed, (int32_t)g));
  for (int l0 = 0; l0 < k; l0 += 32) {
    const int w = tmin(32, k - l0);
    uint64_t term = 0;
    if (lane < w) {
      const uint64_t v = wait_word(s.seg_word + sb + l0 + lane, kWordTotal);
      ok = ok && v != 0;
      term = mad61(kc[(kSegBlocks + 1) + (w - 1 - lane)], v & kP61, 0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      term += __shfl_xor_sync(kFull, term, o);
      if (o == 8 || o == 2) term = weak61(term);  // four terms at most are below 2^64
    }
    cin = mad61(kc[(kSegBlocks + 1) + w], cin, term);
  }
  // the lane's keys and their table probes
  uint64_t keyA = 0, keyB = 0;
  uint32_t blkA = kNone, blkB = kNone;
  if (lane < nbA) {
    const uint64_t C = red61(mad61(kc[lane + 1], cin, bA));
    keyA = fix_reserved(mix64(C ^ ((uint64_t)(mA + 1) * 0xD1B54A32D192ED03ull)));
  }
  if (lane < nbB) {
    const uint64_t cinB = mad61(kc[kSegBlocks], cin, totA);
    const uint64_t C = red61(mad61(kc[lane + 1], cinB, bB));
    keyB = fix_reserved(mix64(C ^ ((uint64_t)(mB + 1) * 0xD1B54A32D192ED03ull)));
  }
  table_find2(s, keyA, keyB, g, lane < nbA, lane < nbB, &blkA, &blkB);
  // What place() below swaps is fetched into L2 while the warp waits for its
  // predecessors' misses: a hit's pin, a miss's claim bucket (152.6 -> 149.8 us
  // a step at 2^20 blocks).  A hit past the first miss is claimed after all and
  // only goes without.
  auto ahead = [&](uint64_t key, uint32_t blk) {
    const void* p = blk == kNone ? (const void*)(s.claims + (size_t)claim_home(key, s.cl_nbuckets_log2) * kClaimWays)
                                 : (const void*)(s.blk_pin + blk);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  };
  if (!probe_out) {
    if (lane < nbA) ahead(keyA, blkA);
    if (lane < nbB) ahead(keyB, blkB);
  }
  const unsigned missA = __ballot_sync(kFull, lane < nbA && blkA == kNone);
  const unsigned missB = __ballot_sync(kFull, lane < nbB && blkB == kNone);
  const bool anymiss = (missA | missB) != 0;
  if (lane == 0) st_relaxed_u64(s.seg_word + j, total | kWordTotal | kWordMiss | (anymiss ? kWordMissBit : 0));
  // did any earlier block of the request miss?
  bool missbefore = false;
  for (int l0 = 0; l0 < k && !missbefore; l0 += 32) {
    const int w = tmin(32, k - l0);
    bool mb = false;
    if (lane < w) {
      const uint64_t v = wait_word(s.seg_word + sb + l0 + lane, kWordMiss);
      ok = ok && v != 0;
      mb = (v & kWordMissBit) != 0;
    }
    missbefore = __any_sync(kFull, mb);
  }
  if (!__all_sync(kFull, ok)) return false;  // a predecessor never published
  // first miss in this chunk
  const int first = missA ? __ffs(missA) - 1 : (missB ? kSegBlocks + __ffs(missB) - 1 : kChunkBlocks);
  if (probe_out) {  // the chunk of the first miss, or the last chunk, knows the count
    if (lane == 0 && !missbefore && (anymiss || m0 + nb == n)) probe_out[i] = anymiss ? m0 + first : n;
    return true;
  }
  if (!missbefore && anymiss && lane == 0) s.rq_h[i] = m0 + first;  // h_i: its only writer
  const uint32_t step32 = (uint32_t)c->step;
  // the cached prefix is pinned, every later block claimed
  auto place = [&](bool act, int half, uint64_t key, uint32_t blk, uint32_t* klass) -> bool {
    if (!act) return false;
    const int mm = m0 + half * kSegBlocks + lane;
    const int64_t p = pbase + mm;
    s.pos_key[p] = key;
    s.pos_req[p] = i;
    s.pos_m[p] = (uint32_t)mm;
    s.pos_blk[p] = blk;
    bool pinned = false;
    if (!missbefore && half * kSegBlocks + lane < first) {
      pinned = atomicExch(s.blk_pin + blk, step32) != step32;
      if (pinned && s.lg_on) *klass = s.blk_klass[blk];
      s.pos_claim[p] = kNone;
    } else {
      s.pos_claim[p] = claim_insert(s, key, i);
    }
    return pinned;
  };
  uint32_t klassA = 0, klassB = 0;
  const bool pinA = place(lane < nbA, 0, keyA, blkA, &klassA);
  const bool pinB = place(lane < nbB, 1, keyB, blkB, &klassB);
  const int np = __popc(__ballot_sync(kFull, pinA)) + __popc(__ballot_sync(kFull, pinB));
  if (lane == 0 && np) atomic_add_i64(&c->pinned, np);
  // hits are namespaced by group: every block the warp pins is group g's
  if (s.policy == PS_STATICQUOTA && lane == 0 && np) atomic_add_i64(s.grp_pinned + g, np);
  if (s.lg_on) {  // a pinned block is no candidate: it leaves its queues' live counts (applied in k_lg_cand)
    const int32_t A1 = lg_log_a(s, g, klassA), B1 = lg_log_b(s, klassA);
    agg_add_i64(s.lg_pin, (uint32_t)A1, 1, pinA && A1 >= 0);
    agg_add_i64(s.lg_pin, (uint32_t)B1, 1, pinA && B1 >= 0);
    const int32_t A2 = lg_log_a(s, g, klassB), B2 = lg_log_b(s, klassB);
    agg_add_i64(s.lg_pin, (uint32_t)A2, 1, pinB && A2 >= 0);
    agg_add_i64(s.lg_pin, (uint32_t)B2, 1, pinB && B2 >= 0);
  }
  const uint64_t key = keyA;  // block 0's key, in the first chunk's lane 0
  // OnRequest of Alg. 1: the request's (group, prefix) history entry
  if (k == 0 && lane == 0) {
    const uint64_t pid = s.in_prefix ? s.in_prefix[i] : key;  // default: block 0's key
    uint32_t hs = kNone;
    const uint32_t hmask = (1u << s.hist_cap_log2) - 1;
    uint32_t x = hist_home(pid, g, s.hist_cap_log2);
    for (uint32_t it = 0; it <= hmask; ++it, x = (x + 1) & hmask) {
      uint64_t olo, ohi;
      cas128(s.hist + x, 0ull, 0ull, pid, (uint64_t)(g + 1), &olo, &ohi);
      if (olo == 0 && ohi == 0) {
        atomic_add_i64(&c->hist_new, 1);
        hs = x;
        break;
      }
      if (olo == pid && (uint32_t)ohi == g + 1) {
        hs = x;
        break;
      }
    }
    if (hs != kNone)
      atomicMax(reinterpret_cast<unsigned long long*>(&s.hist[hs].ftag), (unsigned long long)step_tag(c->step, i));
    s.rq_hs[i] = hs;
    s.rq_p[i] = pid;
  }
  return true;
}

// The kernel: persistent warps.  Each warp takes chunk tickets one at a time,
// each only once it is free to start the chunk, so a chunk's predecessors
// (lower tickets) have always started hashing before it, and their totals
// arrive about when its own does.  A chunk waits only on chunks of lower
// tickets, each held by a running warp: the waits always make progress.
// What bounds it: the memory system under scattered accesses, not instructions
// (34% of issue slots) or DRAM bandwidth (20%).  Clocks read inside it at 2^20
// blocks, before the digests were rolled and the pins and claims fetched ahead,
// in thousands of cycles a chunk: ticket 12, descriptor 3, tokens and digests 13,
// scan 4, predecessors' totals 9, table 20, predecessors' misses 8, pins and
// claims 14.  Measured there and not kept (155 us a step): tokens read
// coalesced, four lanes a block (159 to 171), a CTA's first tickets drawn at
// once (156), a warp's next ticket drawn early (158), two claims at a time
// (155), no way loaded before its tag matched (155).
// probe_out: the read-only probe (ps_cached_prefix) stores h_i there; no pins,
// claims, history or per-position records.
constexpr int kHashCtasPerSm = 5;
template <int BS>
__global__ void __launch_bounds__(256, kHashCtasPerSm) k_hash_lookup(DevState s, int32_t* probe_out) {
  s = with_args(s);
  __shared__ uint32_t sk[BS + 2];                // the NH key words (read by every lane alike)
  __shared__ uint64_t kc[2 * (kSegBlocks + 1)];  // Kc^j, then Kc^(64 t)
  Ctl* c = s.ctl;
  const int64_t nsegs = c->nsegs;  // none in a failed call
  for (int k = threadIdx.x; k < BS + 2; k += blockDim.x) sk[k] = s.key_words[k];
  for (int k = threadIdx.x; k < 2 * (kSegBlocks + 1); k += blockDim.x) kc[k] = s.kc_pow[k];
  __syncthreads();
  const int lane = lane_id();
  if (probe_out && c->status == PS_OK)  // a prompt without a full block has no chunk
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.R; i += gridDim.x * blockDim.x)
      if (s.rq_n[i] == 0) probe_out[i] = 0;
  for (;;) {
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(&c->hash_ticket, 1u);
    t = __shfl_sync(kFull, t, 0);
    if ((int64_t)t >= nsegs) return;
    if (!hash_lookup_chunk<BS>(s, c, sk, kc, (int64_t)t, probe_out)) {
      if (lane == 0) c->internal_error = 1;
      return;
    }
  }
}


// A step whose new (group, prefix) entries would overflow the history map
// fails as a whole, leaving the pool as it was (Alg. 1's hooks change state
// only for a request that goes ahead).  k_hash_lookup has written three things
// by then, undone here thread by thread over the same positions and requests:
//  - pin tags of the cached prefix: set to a tag no step compares against
//    (the previous step's), so the retried step pins them afresh;
//  - claim-map entries: cleared (the map holds only this step's keys);
//  - history entries: an entry with no committed reference was installed by
//    this step and is removed (entries are never removed otherwise, so no
//    probe sequence ran through it); every other touched entry loses the
//    step's first-reference tag.
// The error itself is raised by k_grant, after every thread here is done.
__device__ __forceinline__ bool history_overflows(const DevState& s, const Ctl* c) {
  return c->hist_live + c->hist_new > s.history_capacity;
}
__device__ void undo_pin_claim(const DevState& s, const Ctl* c, int64_t t) {
  const int64_t nb = c->nblocks;
  const uint32_t step32 = (uint32_t)c->step;
  if (t < nb) {
    PosRef r;
    pos_ref(s, t, &r);
    if (r.m < s.rq_h[r.i]) {
      s.blk_pin[s.pos_blk[t]] = step32 - 1u;
    } else {
      const uint32_t slot = s.pos_claim[t];
      if (slot != kNone) s.claims[slot] = empty_claim();
    }
  } else if (t < nb + s.R) {
    const uint32_t hs = s.rq_hs[t - nb];
    if (hs != kNone) {
      HistEntry* e = s.hist + hs;
      if (ldcg_u32(&e->refadm) == 0) *e = HistEntry{};
      else e->ftag = 0;
    }
  }
}

// A history entry from L2 (two 16-byte loads that skip L1: a tag may have
// been updated by an atomic since another CTA on this SM read the line).
__device__ __forceinline__ HistEntry ldcg_hist(const HistEntry* p) {
  const uint4 a = __ldcg(reinterpret_cast<const uint4*>(p)), b = __ldcg(reinterpret_cast<const uint4*>(p) + 1);
  HistEntry e;
  e.p = (uint64_t)a.y << 32 | a.x;
  e.g1 = a.z;
  e.refadm = a.w;
  e.ftag = (uint64_t)b.y << 32 | b.x;
  e.atag = (uint64_t)b.w << 32 | b.z;
  return e;
}

// Stage 2 (cont.): the first own claim s_i of each request, and orphans.  A
// resident block past a request's first miss cannot be reached by lookup; it
// is dropped (invalidated) unless some request pinned it.  Threads past the
// positions take the requests (used only to undo a failing step).
__global__ void __launch_bounds__(kThreads) k_claims(DevState s) {
  s = with_args(s);
  Ctl* c = s.ctl;
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  PosRef r;
  const bool overflow = history_overflows(s, c);
  const uint32_t step32 = (uint32_t)c->step;
  const bool valid = pos_open(s, c, pos, &r);
  if (overflow) {
    if (c->status == PS_OK) undo_pin_claim(s, c, pos);
    return;
  }
  bool inv = false;
  uint32_t ginv = 0, kinv = 0;
  bool own = false;
  if (valid) {
    // the position's records in one round of loads, then what they point to
    const int h = s.rq_h[r.i];
    const uint32_t slot = s.pos_claim[pos], b = s.pos_blk[pos];
    const bool past = r.m > h && b != kNone;
    const uint32_t minreq = r.m >= h ? ldcg_u32(&s.claims[slot].minreq) : kNone;
    const uint32_t pin = past ? ldcg_u32(s.blk_pin + b) : step32;
    own = minreq == r.i;
    if (past) {
      if (pin != step32 && atomicExch(s.blk_inval + b, step32) != step32) {
        ginv = drop_block(s, b);
        if (s.lg_on) kinv = s.blk_klass[b];
        atomicOr(s.bm_inval + (b >> 5), 1u << (b & 31));
        inv = true;
      }
    }
  }
  // s_i = the first own claim: one atomic per request per warp
  agg_min_u32(reinterpret_cast<uint32_t*>(s.rq_s), valid ? r.i : 0u, valid ? (uint32_t)r.m : 0u, own);
  if (s.lg_on) {  // an invalidated block leaves its queues
    const int32_t A = lg_log_a(s, ginv, kinv), B = lg_log_b(s, kinv);
    agg_add_i64(s.lg_live, (uint32_t)A, -1, inv && A >= 0);
    agg_add_i64(s.lg_live, (uint32_t)B, -1, inv && B >= 0);
  }
  agg_stat(s, ginv, PS_STAT_INVALIDATED_BLOCKS, 1, inv);
  agg_stat(s, ginv, PS_STAT_RESIDENT_BLOCKS, -1, inv);
  const int ni = __popc(__ballot_sync(kFull, inv));
  if (lane_id() == 0 && ni) {
    atomic_add_i64(&c->n_inval, ni);
    atomic_add_i64(&c->n_resident, -ni);
  }
}

// ===========================================================================
// Stage 3: grant new blocks against the pool.  avail = free + unpinned
// resident = N - pinned; claims are ranked in (request, position) order; the
// first avail ranks are materialized.  One CTA.
__global__ void __launch_bounds__(1024) k_grant(DevState s0) {
  // Contract arrays are read from the parameter block: indexing the per-step
  // copy by a run-time contract would move the whole copy to local memory.
  const DevState s = with_args(s0);
  extern __shared__ unsigned long long g_sum[];  // [G * C] the step's charges per (group, contract)
  Ctl* c = s.ctl;
  // the first tile's claims (see below) in the status's round trip
  int32_t n4[4], s4[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = u * (int)blockDim.x + (int)threadIdx.x;
    n4[u] = i < s.R ? s.rq_n[i] : 0;
    s4[u] = i < s.R ? s.rq_s[i] : 0;
  }
  const int64_t pinned = c->pinned, n_resident = c->n_resident, t_prev = c->t_prev;
  const bool overflow = history_overflows(s, c);
  if (c->status != PS_OK) return;
  if (overflow) {  // undone by k_claims; the error is sticky
    if (threadIdx.x == 0) { c->status = PS_ERR_CAPACITY; c->sticky = PS_ERR_CAPACITY; }
    return;
  }
  const int R = s.R;
  const int C = s.C;
  const bool quota = s.policy == PS_STATICQUOTA;  // a_i already granted per group
  for (int k = threadIdx.x; k < s.G * C; k += blockDim.x) g_sum[k] = 0;
  __syncthreads();
  const int64_t avail = s.N - pinned;
  // Granted ranks are the first avail in (request, position) order, so the
  // grants before request i number min(avail, base_i), base_i the claims
  // before it, and a_i = min(avail, base_i + c_i) - min(avail, base_i).  One
  // scanned word per request: claims in the high half, StaticQuota grants in
  // the low; four 1024-request sub-tiles a pass.
  uint64_t carry = 0;
  const int tile = 4 * (int)blockDim.x;
  for (int t0 = 0; t0 < R; t0 += tile) {
    uint64_t v[4], ex[4];
    int32_t cl[4], aq[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = t0 + u * (int)blockDim.x + (int)threadIdx.x;
      const bool in = i < R;
      if (t0 > 0) {
        n4[u] = in ? s.rq_n[i] : 0;
        s4[u] = in ? s.rq_s[i] : 0;
      }
      cl[u] = n4[u] - s4[u];
      aq[u] = in && quota ? s.rq_a[i] : 0;
      v[u] = (uint64_t)cl[u] << 32 | (uint64_t)aq[u];
    }
    uint64_t tot;
    block_excl_scan4(v, ex, &tot);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = t0 + u * (int)blockDim.x + (int)threadIdx.x;
      if (i < R) {
        const uint64_t e = carry + ex[u];
        const int64_t base_c = (int64_t)(e >> 32);
        const int64_t lo = quota ? (int64_t)(uint32_t)e : tmin(avail, base_c);
        const int32_t a = quota ? aq[u] : (int32_t)(tmin(avail, base_c + cl[u]) - lo);
        // granted keys are paired with the allocated ids in (request,
        // position) order: request i's first granted key is the lo-th
        s.rq_cbase[i] = (int32_t)lo;
        s.rq_qbase[i] = (int32_t)base_c;
        s.rq_a[i] = a;
        s.out.admitted_blocks[i] = a;
        s.out.admitted_offsets[i] = (int32_t)lo;
        if (a > 0) atomicAdd(&g_sum[s.in_group[i] * C + s.rq_cid[i]], (unsigned long long)a);
      }
    }
    carry += tot;
  }
  const int64_t carry_c = (int64_t)(carry >> 32);
  const int64_t carry_a = quota ? (int64_t)(uint32_t)carry : tmin(avail, carry_c);
  int64_t qv = 0;  // StaticQuota: the groups' overflows are the victims
  if (quota) {
    for (int g = threadIdx.x; g < s.G; g += blockDim.x) qv += s.grp_x[g];
    qv = block_sum(qv);
  }
  if (threadIdx.x == 0) {
    const int64_t need = carry_a;
    s.out.admitted_offsets[R] = (int32_t)need;
    const int64_t nfree = s.N - n_resident;
    c->avail = avail;
    c->total_claims = carry_c;
    c->need = need;
    c->nfree = nfree;
    c->ftake = quota ? need - qv : tmin(need, nfree);
    c->mvict = need - c->ftake;
  }
  // The step's balances and debts (Eq. 1-3, 5) follow from each (group,
  // contract)'s total charge, so they are settled here and the select need
  // not wait for the per-request metering (which reads the refilled opening
  // balances from ledger_b0).
  __syncthreads();
  const int64_t unit = (int64_t)1 << s.fp_shift;
  for (int g = threadIdx.x; g < s.G; g += blockDim.x) {
    // the Eq. 8 decrement of the largest indebted rate is the smallest one
    int64_t raw = 0, norm = 0, delta = 0;
    for (int cc = 0; cc < C; ++cc) {
      const int64_t b0 = refill(s.ledger[g * C + cc], s0.beta[cc], s0.rho[cc], s.now - t_prev);
      s.ledger_b0[g * C + cc] = b0;
      const int64_t b = b0 - (int64_t)g_sum[g * C + cc] * unit;  // Eq. 2 over the step's charges
      s.ledger[g * C + cc] = b;
      const int64_t def = tmax<int64_t>(0, -b);
      raw += def;                                    // Eq. 3
      norm += muldiv(def, s.rho_min, s0.rho[cc]);    // Eq. 5
      if (b < 0 && (delta == 0 || s0.delta[cc] < delta)) delta = s0.delta[cc];
    }
    int64_t* row = s.stats + (int64_t)g * PS_NUM_STATS;
    row[PS_STAT_DEBT_RAW] = raw;
    row[PS_STAT_DEBT_NORM] = norm;
    s.out.debt_raw[g] = raw;
    s.out.debt_norm[g] = norm;
    s.grp_P[g] = norm;
    s.grp_delta[g] = delta;  // 1/W_g of Eq. 8
    SelSeg z{};
    z.kmin = ~0ull;
    z.kmax = 0;
    z.qmin = ~0ull;
    z.qmax = 0;
    s.sel[g] = z;
  }
}

// StaticQuota (Sec. V-A) grants, one CTA per group: the group's claims, in
// (request, position) order, while its partition of Q = floor(N / G) blocks
// minus its pinned ones holds them; its overflow m_g = granted - (Q -
// resident) is what it must reclaim from its own blocks.
__global__ void __launch_bounds__(1024) k_grant_quota(DevState s) {
  s = with_args(s);
  Ctl* c = s.ctl;
  if (c->status != PS_OK) return;
  const int g = blockIdx.x;
  const int64_t Q = s.N / s.G;
  const int64_t avail = Q - s.grp_pinned[g];
  const int R = s.R;
  int64_t carry = 0, granted = 0;
  for (int t0 = 0; t0 < R; t0 += blockDim.x) {
    const int i = t0 + threadIdx.x;
    const bool member = i < R && s.in_group[i] == g;
    const int32_t cl = member ? s.rq_n[i] - s.rq_s[i] : 0;
    int32_t tot;
    const int32_t ex = block_excl_scan(cl, &tot);
    if (member) {
      const int64_t a = tmin<int64_t>(cl, tmax<int64_t>(0, avail - (carry + ex)));
      s.rq_a[i] = (int32_t)a;
      granted += a;
    }
    carry += tot;
  }
  granted = block_sum(granted);
  if (threadIdx.x == 0) {
    const int64_t resident = s.stats[(int64_t)g * PS_NUM_STATS + PS_STAT_RESIDENT_BLOCKS];
    s.grp_x[g] = tmax<int64_t>(0, granted - (Q - resident));
  }
}

// In-step hits: positions of [h_i, s_i) belong to earlier requests' claims;
// the leading granted ones are hits.  A position whose owner's key was not
// granted lowers the request's first-ungranted mark.  The positions from s_i
// on are the request's own claims: they are listed for the insertion.
__global__ void __launch_bounds__(kThreads) k_instep(DevState s) {
  s = with_args(s);
  const Ctl* c = s.ctl;
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  PosRef r;
  bool past = false;
  const bool valid = pos_open(s, c, pos, &r);
  int h = 0, sown = 0;
  uint32_t slot = kNone;
  if (valid) {  // one round of loads
    h = s.rq_h[r.i];
    sown = s.rq_s[r.i];
    slot = s.pos_claim[pos];
    const int32_t qb = s.rq_qbase[r.i];
    if (r.m >= sown) s.claim_pos[qb + (r.m - sown)] = (uint64_t)r.i << 32 | (uint64_t)(uint32_t)pos;
  }
  if (valid && r.m >= h && r.m < sown) {
    // the owner's claims are ranked consecutively: its key here is granted
    // iff it is among the owner's first a_j
    const uint32_t j = s.claims[slot].minreq;
    past = r.m - s.rq_s[j] >= s.rq_a[j];
  }
  agg_min_u32(s.rq_fu, valid ? r.i : 0u, valid ? (uint32_t)r.m : 0u, past);
}

// ===========================================================================
// Stages 3-4: metering (Eq. 1-3, OnCacheFullBlocks of Alg. 1), in request
// order, one CTA per group.  The CTA compacts its group's requests of each
// tile of kMeterTile requests into shared memory (in request order), then
// works on the members only: block-wide exclusive scans give each member the
// charges of the group's earlier requests per contract, hence
//   D_g before the request (the gate of OnTouch, Eq. 4),
//   B_{g,c} after the request's own charge (the class of its new blocks).
// q_r >= 1 and "(g,p) was admitted" come from the history entry as it stood at
// the start of the step and the first request of the step that referenced /
// admitted it.  Also writes the group's request statistics; the balances
// and debts after the step are k_grant's (from the same charges).
constexpr int kMeterThreads = 512;
constexpr int kMeterTile = 4 * kMeterThreads;  // requests compacted per pass
__global__ void __launch_bounds__(kMeterThreads) k_meter(DevState s0) {
  // Contract arrays are read from the parameter block: indexing the per-step
  // copy by a run-time contract would move the whole copy to local memory.
  const DevState s = with_args(s0);
  Ctl* c = s.ctl;
  if (c->status != PS_OK) return;
  const int g = blockIdx.x;
  const int C = s.C;
  const int64_t unit = (int64_t)1 << s.fp_shift;
  const uint64_t step = c->step;
  __shared__ int64_t B0[PS_MAX_CONTRACTS];
  __shared__ unsigned long long s_st[7];  // the group's request statistics
  __shared__ int32_t s_mem[kMeterTile];   // this tile's members, in request order
  if (threadIdx.x < C) B0[threadIdx.x] = s.ledger_b0[g * C + threadIdx.x];  // refilled by k_grant
  if (threadIdx.x < 7) s_st[threadIdx.x] = 0;
  __syncthreads();
  int64_t carry[PS_MAX_CONTRACTS];
#pragma unroll
  for (int cc = 0; cc < PS_MAX_CONTRACTS; ++cc) carry[cc] = 0;
  int64_t st_req = 0, st_ptok = 0, st_full = 0, st_hit = 0, st_inst = 0, st_adm = 0, st_ungr = 0;
  const int R = s.R;
  for (int base = 0; base < R; base += kMeterTile) {
    // members of this tile: four consecutive requests a thread, compacted by
    // a block scan of their counts (the order is request order)
    const int i0 = base + 4 * (int)threadIdx.x;
    int32_t gg[4] = {-1, -1, -1, -1};
    if (i0 + 3 < R && (reinterpret_cast<uintptr_t>(s.in_group + i0) & 15) == 0) {
      const int4 v = *reinterpret_cast<const int4*>(s.in_group + i0);
      gg[0] = v.x; gg[1] = v.y; gg[2] = v.z; gg[3] = v.w;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < R) gg[u] = s.in_group[i0 + u];
    }
    int cnt = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) cnt += gg[u] == g;
    int nmem;
    int at = block_excl_scan(cnt, &nmem);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (gg[u] == g) s_mem[at++] = i0 + u;
    __syncthreads();
    for (int k0 = 0; k0 < nmem; k0 += kMeterThreads) {
      const int k = k0 + (int)threadIdx.x;
      const bool mem = k < nmem;
      const int i = mem ? s_mem[k] : 0;
      int n = 0, a = 0, cid = 0, rh = 0, re = 0, rs = 0;
      uint32_t hs = kNone, fu = kNone;
      int64_t ptok = 0;
      if (mem) {
        n = s.rq_n[i]; a = s.rq_a[i]; cid = s.rq_cid[i]; hs = s.rq_hs[i];
        rh = s.rq_h[i]; rs = s.rq_s[i]; fu = s.rq_fu[i];
        ptok = s.in_offsets[i + 1] - s.in_offsets[i];
        // in-step hits: the leading positions of [h_i, s_i) before the first
        // ungranted one; hit_i = h_i + e_i
        re = (int)tmin<uint32_t>(fu, (uint32_t)rs) - rh;
        s.rq_e[i] = re;
        s.out.hit_blocks[i] = rh + re;
        // the first admitting request of the (group, prefix) entry in this
        // step: only requests of this group share its entries, and every one
        // of them is this CTA's
        if (a > 0 && hs != kNone)
          atomicMax(reinterpret_cast<unsigned long long*>(&s.hist[hs].atag), (unsigned long long)step_tag(step, (uint32_t)i));
      }
      const bool pol = mem && n > 0;
      __syncthreads();  // every member's admission tag is in place
      HistEntry he{};
      if (pol && hs != kNone) he = ldcg_hist(s.hist + hs);
      // charges of this group's earlier requests, per contract
      int64_t S[PS_MAX_CONTRACTS];
#pragma unroll
      for (int cc = 0; cc < PS_MAX_CONTRACTS; ++cc) {
        S[cc] = 0;
        if (cc < C) {
          int64_t tot;
          const int64_t ex = block_excl_scan<int64_t>((pol && cid == cc) ? a : 0, &tot);
          S[cc] = carry[cc] + ex;
          carry[cc] += tot;
        }
      }
      if (pol) {
        // the raw debt before this request's charge (Eq. 3) and its balance after
        int64_t d = 0, b_after = 0;
#pragma unroll
        for (int cc = 0; cc < PS_MAX_CONTRACTS; ++cc) {
          if (cc < C) {
            d += tmax<int64_t>(0, -(B0[cc] - S[cc] * unit));
            if (cid == cc) b_after = B0[cc] - (S[cc] + a) * unit;
          }
        }
        const bool gate = (s.flags & PS_FLAG_NO_DEBT_GATE) || d <= s.eps;
        const uint32_t refadm = he.refadm;
        const bool q_ge1 = (refadm & 0x7FFFFFFFu) >= 1 || tag_req(he.ftag, step) < (uint32_t)i;
        const bool adm_before = (refadm >> 31) || tag_req(he.atag, step) < (uint32_t)i;
        const bool proven = q_ge1 && adm_before;
        s.rq_flags[i] = (uint8_t)((proven ? 1 : 0) | (gate ? 2 : 0));
        s.rq_knew[i] = (uint8_t)((b_after < -s.eps || !adm_before) ? kProb : kNormal);
        st_full += n; st_hit += rh + re; st_inst += re; st_adm += a; st_ungr += (n - rs) - a;
      }
      if (mem) { st_req += 1; st_ptok += ptok; }
    }
    __syncthreads();  // s_mem is rewritten by the next tile
  }
  {
    const int64_t v[7] = {st_req, st_ptok, st_full, st_hit, st_inst, st_adm, st_ungr};
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      const int64_t w = warp_sum(v[k]);
      if (lane_id() == 0 && w) atomicAdd(&s_st[k], (unsigned long long)w);
    }
  }
  __syncthreads();
  st_req = (int64_t)s_st[0]; st_ptok = (int64_t)s_st[1]; st_full = (int64_t)s_st[2]; st_hit = (int64_t)s_st[3];
  st_inst = (int64_t)s_st[4]; st_adm = (int64_t)s_st[5]; st_ungr = (int64_t)s_st[6];
  if (threadIdx.x == 0) {
    int64_t* row = s.stats + (int64_t)g * PS_NUM_STATS;
    row[PS_STAT_REQUESTS] += st_req;
    row[PS_STAT_PROMPT_TOKENS] += st_ptok;
    row[PS_STAT_FULL_BLOCKS] += st_full;
    row[PS_STAT_HIT_BLOCKS] += st_hit;
    row[PS_STAT_INSTEP_HIT_BLOCKS] += st_inst;
    row[PS_STAT_HIT_TOKENS] += st_hit * s.bs;
    row[PS_STAT_ADMITTED_BLOCKS] += st_adm;
    row[PS_STAT_UNGRANTED_BLOCKS] += st_ungr;
  }
}

// ===========================================================================
// Stage 4: OnTouch (Alg. 1, Eq. 4) for every hit block, resident or in-step,
// thread per position.  Pass 1 applies the access updates (stamp = max,
// access count, S3-FIFO frequency) and records, per block, the lowest request
// whose touch promotes it.  Pass 2 counts the gated touches that precede the
// promotion (or all of them when none promotes) and applies the promotion of
// resident blocks.
__global__ void __launch_bounds__(kThreads) k_touch(DevState s) {
  s = with_args(s);
  const Ctl* c = s.ctl;
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const uint64_t step = c->step, base = c->stamp_base;
  PosRef r;
  if (!pos_open(s, c, pos, &r)) return;
  // every record of the position and its request in one round of loads (an
  // atomic in between would hold back the loads after it), then the block's
  const uint32_t i = r.i;
  const int m = r.m;
  const int h = s.rq_h[i], re = s.rq_e[i], n = s.rq_n[i], pbase = s.rq_pbase[i], cid = s.rq_cid[i];
  const uint8_t fl = s.rq_flags[i];
  const uint64_t p = s.rq_p[i];
  const uint32_t b = s.pos_blk[pos], slot = s.pos_claim[pos];
  if (m >= h + re) return;
  const bool proven = fl & 1, gate = fl & 2;
  const uint64_t stamp = make_stamp(base, pbase, n, m);
  bool elig;
  if (m < h) {
    const uint8_t bc = s.blk_contract[b], bk = s.blk_klass[b];
    const uint64_t bp = s.blk_prefix[b];
    atomicMax(reinterpret_cast<unsigned long long*>(s.blk_stamp + b), (unsigned long long)stamp);
    if (s.lg_on) s.lg_slot[pbase + (n - 1 - m)] = b;  // the queues' append reads it back
    atomicAdd(s.blk_acc + b, 1u);
    atomicAdd(s.blk_freq + b, 1u);
    elig = proven && bc == cid && bp == p && bk != kReuse;
    if (elig && gate)
      atomicMax(reinterpret_cast<unsigned long long*>(s.blk_promo + b), (unsigned long long)step_tag(step, i));
  } else {
    ClaimEntry* e = s.claims + slot;
    const uint32_t j = e->minreq;
    const int jc = s.rq_cid[j];
    const uint64_t jp = s.rq_p[j];
    // later requests give larger stamps: the maximum is the latest touch's
    atomicMax(reinterpret_cast<unsigned long long*>(&e->stamp), (unsigned long long)stamp);
    atomicAdd(&e->tcnt, 1u);
    elig = proven && jc == cid && jp == p;  // new blocks are never Reuse yet
    if (elig && gate) atomicMin(&e->promo, i);
  }
  s.pos_elig[pos] = elig;
}

__global__ void __launch_bounds__(kThreads) k_touch2(DevState s) {
  s = with_args(s);
  const Ctl* c = s.ctl;
  const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  PosRef r;
  bool gated = false, promoted = false;
  uint32_t g = 0;
  bool elig = false;
  int h = 0;
  uint32_t b = kNone, slot = kNone;
  uint8_t fl = 0;
  const uint64_t step = c->step;
  if (pos_open(s, c, pos, &r)) {  // one round of loads (an untouched position's eligibility is stale, and not used)
    const uint8_t el = s.pos_elig[pos];
    const int re = s.rq_e[r.i];
    h = s.rq_h[r.i];
    b = s.pos_blk[pos];
    slot = s.pos_claim[pos];
    fl = s.rq_flags[r.i];
    g = (uint32_t)s.in_group[r.i];
    elig = r.m < h + re && el;
  }
  if (elig) {
    const uint32_t i = r.i;
    const bool gate = fl & 2;
    uint32_t promoter;
    if (r.m < h) {
      promoter = tag_req(ldcg_u64(s.blk_promo + b), step);
    } else {
      b = kNone;
      promoter = ldcg_u32(&s.claims[slot].promo);
    }
    if (!gate) {
      gated = i < promoter;
    } else if (i == promoter) {
      promoted = true;
      if (b != kNone) s.blk_klass[b] = kReuse;
    }
  }
  agg_stat(s, g, PS_STAT_GATED_REUSES, 1, gated);
  agg_stat(s, g, PS_STAT_PROMOTIONS, 1, promoted);
}

// ===========================================================================
// Stage 5: reclamation.  Candidates are resident blocks not hit in this step.
// The order key is (class, stamp) for prefixshield (Eq. 9; stamp only with
// the no-segmentation ablation) and the stamp for lru.  Per (segment, class):
// the candidates and their stamp range, so the radix select can start inside
// the class that holds its rank and skip the bytes the class's stamps share.
__global__ void __launch_bounds__(1024) k_cand(DevState s) {
  s = with_args(s);
  extern __shared__ uint32_t cand_smem[];  // 5 arrays of nseg * kClasses
  // runs beside S3-S4: the victim count is not known yet, and a failed step
  // ignores what is written here
  const Ctl* c = s.ctl;
  const uint32_t step32 = (uint32_t)c->step;
  // segments: groups for prefixshield and staticquota, one for lru; retention
  // classes only for prefixshield
  const bool ps = s.policy == PS_PREFIXSHIELD || s.policy == PS_STATICQUOTA;
  const bool seg = s.policy == PS_PREFIXSHIELD && !(s.flags & PS_FLAG_NO_SEGMENTATION);
  const int nrow = (ps ? s.G : 1) * kClasses;
  uint32_t* s_cnt = cand_smem;
  uint32_t* s_hmin = s_cnt + nrow;
  uint32_t* s_hmax = s_hmin + nrow;
  uint32_t* s_lmin = s_hmax + nrow;
  uint32_t* s_lmax = s_lmin + nrow;
  for (int r = threadIdx.x; r < nrow; r += blockDim.x) {
    s_cnt[r] = 0;
    s_hmin[r] = s_lmin[r] = ~0u;
    s_hmax[r] = s_lmax[r] = 0;
  }
  __syncthreads();
  // kU blocks a thread per iteration, their loads issued together; the trip
  // count is warp-uniform.  Lanes of one (segment, class) combine their
  // ranges and counts with warp reductions; one lane updates shared memory.
  constexpr int kU = 4;
  const int64_t span = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b0 = blockIdx.x * (int64_t)blockDim.x; b0 < s.N; b0 += span * kU) {
    uint8_t fl[kU], kl[kU];
    uint32_t pin[kU];
    uint16_t grp[kU];
    uint64_t st[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t b = b0 + u * span + threadIdx.x;
      fl[u] = 0;
      if (b < s.N) {
        fl[u] = s.blk_flags[b];
        kl[u] = s.blk_klass[b];
        pin[u] = s.blk_pin[b];
        grp[u] = s.blk_group[b];
        st[u] = s.blk_stamp[b];
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t b = b0 + u * span + threadIdx.x;
      uint64_t key = ~0ull;
      uint32_t row = ~0u;
      if ((fl[u] & 1) && pin[u] != step32) {
        key = seg ? (st[u] | (uint64_t)kl[u] << 62) : st[u];
        row = (ps ? (uint32_t)grp[u] : 0u) * kClasses + (seg ? kl[u] : 0u);
      }
      const unsigned peers = __match_any_sync(kFull, row);
      if (row != ~0u) {
        const uint32_t hi = (uint32_t)(st[u] >> 32), lo = (uint32_t)st[u];
        const uint32_t hmin = __reduce_min_sync(peers, hi), hmax = __reduce_max_sync(peers, hi);
        const uint32_t lmin = __reduce_min_sync(peers, lo), lmax = __reduce_max_sync(peers, lo);
        if (lane_id() == __ffs(peers) - 1) {
          atomicAdd(&s_cnt[row], (unsigned)__popc(peers));
          atomicMin(&s_hmin[row], hmin);
          atomicMax(&s_hmax[row], hmax);
          atomicMin(&s_lmin[row], lmin);
          atomicMax(&s_lmax[row], lmax);
        }
      }
      if (b < s.N) s.csk[b] = key;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < nrow; r += blockDim.x) {
    if (!s_cnt[r]) continue;
    if (ps) atomic_add_i64(s.grp_qsize + r / kClasses, s_cnt[r]);
    ClsRange* d = s.cls + r;
    atomicAdd(&d->cnt, s_cnt[r]);
    atomicMin(&d->hmin, s_hmin[r]);
    atomicMax(&d->hmax, s_hmax[r]);
    atomicMin(&d->lmin, s_lmin[r]);
    atomicMax(&d->lmax, s_lmax[r]);
  }
}

// Stamp range of a class from its two half ranges: exact below the top half
// when every member shares its top 32 bits, conservative otherwise.
__device__ __forceinline__ void cls_stamp_range(const ClsRange& r, uint64_t* lo, uint64_t* hi) {
  const bool same_hi = r.hmin == r.hmax;
  *lo = ((uint64_t)r.hmin << 32) | (same_hi ? r.lmin : 0u);
  *hi = ((uint64_t)r.hmax << 32) | (same_hi ? r.lmax : 0xFFFFFFFFu);
}

// Start a segment's search from its per-class candidates: the class holding
// the rank-th smallest key is fixed (lower classes are all below it), the rank
// becomes a rank inside that class, and the key range is the class's.
// cnt[k] and [lo[k], hi[k]] describe class k (unsegmented keys: class 0 only).
// Classes are picked without run-time array indexing (registers only).
__device__ __forceinline__ void sel_start_cls(SelSeg& z, const int64_t (&cnt)[kClasses], const uint64_t (&lo)[kClasses],
                                              const uint64_t (&hi)[kClasses], bool segmented) {
  static_assert(kClasses == 3, "class choice below is written for three classes");
  int k = 0;
  int64_t below = 0;
  if (segmented && z.rank > cnt[0]) {
    below = cnt[0];
    k = 1;
    if (z.rank > cnt[0] + cnt[1]) {
      below += cnt[1];
      k = 2;
    }
  }
  const int64_t ck = k == 0 ? cnt[0] : k == 1 ? cnt[1] : cnt[2];
  const uint64_t lk = k == 0 ? lo[0] : k == 1 ? lo[1] : lo[2];
  const uint64_t hk = k == 0 ? hi[0] : k == 1 ? hi[1] : hi[2];
  const uint64_t cb = segmented ? (uint64_t)k << 62 : 0ull;
  if (z.active && ck > 0) {
    z.rank -= below;
    z.kmin = cb | lk;
    z.kmax = cb | hk;
  } else {
    z.kmin = z.kmax = cb;
  }
}
__device__ __forceinline__ void sel_start_group(const DevState& s, int g, SelSeg& z, bool segmented) {
  int64_t cnt[kClasses];
  uint64_t lo[kClasses], hi[kClasses];
#pragma unroll
  for (int k = 0; k < kClasses; ++k) {
    const ClsRange r = s.cls[g * kClasses + k];
    cnt[k] = r.cnt;
    cls_stamp_range(r, &lo[k], &hi[k]);
  }
  sel_start_cls(z, cnt, lo, hi, segmented);
}

// One global segment: all candidates for lru, or (fallback) the candidates
// the debt phase of prefixshield left, in (class, stamp) order (Eq. 9).  The
// debt phase took group g's x_g smallest keys, so of class k it took
// clamp(x_g - (members of lower classes), 0, members of class k).
// One warp: the segment-0 state of a global select (lru, or the fallback).
__device__ void start_global_select(const DevState& s, Ctl* c, int fallback) {
  const int lane = lane_id();
  int64_t m = 0;
  if (c->status == PS_OK) m = fallback ? c->m_fb : c->mvict;
  const bool segmented = s.policy == PS_PREFIXSHIELD && !(s.flags & PS_FLAG_NO_SEGMENTATION);
  int64_t cnt[kClasses];
  uint64_t lo[kClasses], hi[kClasses];
  for (int k = 0; k < kClasses; ++k) { cnt[k] = 0; lo[k] = ~0ull; hi[k] = 0; }
  if (m > 0) {
    const int nseg = fallback ? s.G : 1;
    for (int g = lane; g < nseg; g += 32) {
      int64_t taken = fallback ? s.grp_x[g] : 0;
      for (int k = 0; k < kClasses; ++k) {
        const ClsRange r = s.cls[g * kClasses + k];
        const int64_t t = tmin<int64_t>(taken, (int64_t)r.cnt);
        taken -= t;
        if ((int64_t)r.cnt > t) {
          uint64_t a, b;
          cls_stamp_range(r, &a, &b);
          cnt[k] += (int64_t)r.cnt - t;
          lo[k] = tmin(lo[k], a);
          hi[k] = tmax(hi[k], b);
        }
      }
    }
    for (int k = 0; k < kClasses; ++k)
      for (int o = 16; o > 0; o >>= 1) {
        cnt[k] += __shfl_xor_sync(kFull, cnt[k], o);
        lo[k] = tmin(lo[k], (uint64_t)__shfl_xor_sync(kFull, lo[k], o));
        hi[k] = tmax(hi[k], (uint64_t)__shfl_xor_sync(kFull, hi[k], o));
      }
  }
  if (lane != 0) return;
  SelSeg z{};
  z.rank = m;
  z.active = m > 0;
  z.incl = 1;
  z.qmin = ~0ull;
  z.qmax = 0;
  sel_start_cls(z, cnt, lo, hi, segmented);
  s.sel[0] = z;
  c->lst_n = 0;
  if (!fallback) c->sel_mode = kSelGlobal;
}
__global__ void __launch_bounds__(32) k_sel_single(DevState s) {
  s = with_args(s);
  start_global_select(s, s.ctl, 0);
}

// StaticQuota: each group reclaims its overflow m_g from its own blocks, in
// recency order (one segment per group, no global fallback).
__global__ void __launch_bounds__(1024) k_quota_sel(DevState s) {
  s = with_args(s);
  Ctl* c = s.ctl;
  const int64_t m = c->status == PS_OK ? c->mvict : 0;
  for (int g = threadIdx.x; g < s.G; g += blockDim.x) {
    SelSeg z = s.sel[g];
    z.rank = m > 0 ? s.grp_x[g] : 0;
    z.active = z.rank > 0;
    z.incl = 1;
    sel_start_group(s, g, z, false);
    s.sel[g] = z;
  }
  if (threadIdx.x == 0) { c->m_fb = 0; c->sel_ntie = 0; c->sel_k = 0; c->lst_n = 0; c->sel_mode = kSelGroups; }
}

// Alg. 2 in closed form (one CTA).  Group g's j-th victim would be taken at
// projected value v_{g,j} = P_g - j*delta_g (Eq. 8) while v_{g,j} > epsilon
// (Eq. 6); each group's sequence strictly decreases, so the per-victim argmax
// loop (Eq. 7) takes items in order of (value descending, candidate key
// ascending).  The m-th largest value tau splits the items: every item above
// tau is taken; among the groups holding an item at exactly tau (at most one
// each) the ones with the smallest candidate keys are taken (resolved after
// the radix select finds those keys).  What the debt phase cannot cover goes
// to the global fallback in (class, stamp) order.
//
// A thread holds a group (PS_MAX_GROUPS threads) with everything loaded in one
// round trip; sums over the groups take one barrier each (per-warp partials,
// every warp adding them up for itself).  tau is bracketed first: a group with
// m items of its own puts tau at or above its m-th, and some group gives at
// least ceil(m / groups) of the m items, so tau is at most the largest such
// item.  The search then narrows the bracket to one decrement, within which
// each group has at most one item: tau is one of those.  (One indebted group
// needs no search at all; the search over all values took four to six rounds.)
// (PS_MAX_GROUPS threads; contract arrays are read from the parameter block s0, see k_grant)
__device__ __forceinline__ void waterfill(const DevState& s, const DevState& s0, Ctl* c) {
  __shared__ int64_t hP[PS_MAX_GROUPS], hD[PS_MAX_GROUPS], hQ[PS_MAX_GROUPS];  // the groups that can give victims
  __shared__ uint64_t hRcp[PS_MAX_GROUPS];
  __shared__ int64_t w_a[32], w_b[32], w_c[32], w_d[32];  // per-warp partials
  __shared__ int32_t w_n[32], w_f[32];
  __shared__ int64_t s_tau;
  const int g = (int)threadIdx.x, warp = g >> 5, lane = lane_id();
  const bool mine = g < s.G;
  const int64_t eps = s.eps;
  const bool seg = !(s.flags & PS_FLAG_NO_SEGMENTATION);
  const int32_t st = c->status;
  const int64_t mv = c->mvict;
  const int64_t P = mine ? s.grp_P[g] : 0, d = mine ? s.grp_delta[g] : 0, q = mine ? s.grp_qsize[g] : 0;
  ClsRange r[kClasses];
#pragma unroll
  for (int k = 0; k < kClasses; ++k) r[k] = mine ? s.cls[g * kClasses + k] : ClsRange{0, ~0u, 0, ~0u, 0};
  const int64_t m = st == PS_OK ? mv : 0;
  if (m == 0) {
    if (mine) { s.sel[g].active = 0; s.grp_x[g] = 0; s.grp_full[g] = 0; }
    if (g == 0) c->m_fb = 0;
    return;
  }
  uint64_t rcp = 0;  // floor((2^64 - 1) / d): d is some contract's decrement
  for (int cc = 0; cc < s.C; ++cc)
    if (s0.delta[cc] == d) rcp = s0.delta_rcp[cc];
  // floor(x / d) for x >= 0 from the reciprocal: the estimate is at most two
  // below the quotient, and the correction makes it exact
  auto div_d = [](uint64_t x, uint64_t dd, uint64_t rr) -> uint64_t {
    if (dd == 1) return x;
    uint64_t z = __umul64hi(x, rr);
    while (x - z * dd >= dd) ++z;
    return z;
  };
  // items of a group with value > t: min(q, floor((P - t - 1) / d) + 1) if P > t
  auto items_gt = [&](int64_t pp, int64_t dd, int64_t qq, uint64_t rr, int64_t t) -> int64_t {
    return (pp > t && dd > 0) ? tmin<int64_t>(qq, (int64_t)div_d((uint64_t)(pp - t - 1), (uint64_t)dd, rr) + 1) : 0;
  };
  // a segment started over the group's rank smallest candidates
  auto start = [&](int64_t rank, int incl) {
    SelSeg z{};
    z.rank = rank;
    z.active = 1;
    z.incl = incl;
    z.qmin = ~0ull;
    int64_t cnt[kClasses];
    uint64_t lo[kClasses], hi[kClasses];
#pragma unroll
    for (int k = 0; k < kClasses; ++k) {
      cnt[k] = r[k].cnt;
      cls_stamp_range(r[k], &lo[k], &hi[k]);
    }
    sel_start_cls(z, cnt, lo, hi, seg);
    s.sel[g] = z;
  };
  const int64_t x = items_gt(P, d, q, rcp, eps);  // the group's items above epsilon
  const bool holds = x > 0, full = holds && x == q;
  const unsigned hb = __ballot_sync(kFull, holds);
  const unsigned fl = (__ballot_sync(kFull, full) ? 1u : 0u) | (__ballot_sync(kFull, holds && !full) ? 2u : 0u);
  {
    const int64_t e = warp_sum(x);
    int64_t dm = holds ? d : INT64_MAX;
    for (int o = 16; o > 0; o >>= 1) dm = tmin(dm, (int64_t)__shfl_xor_sync(kFull, dm, o));
    if (lane == 0) {
      w_a[warp] = e;
      w_d[warp] = dm;
      w_n[warp] = __popc(hb);
      w_f[warp] = (int32_t)fl;
    }
  }
  __syncthreads();
  const int64_t E = warp_sum(w_a[lane]);
  const int32_t nw = w_n[lane], nin = warp_incl_scan(nw);
  const int ng = __shfl_sync(kFull, nin, 31);
  const int hbase = __shfl_sync(kFull, nin - nw, warp);
  int64_t dmin = w_d[lane];
  for (int o = 16; o > 0; o >>= 1) dmin = tmin(dmin, (int64_t)__shfl_xor_sync(kFull, dmin, o));
  const uint32_t flags = __reduce_or_sync(kFull, (uint32_t)w_f[lane]);
  if (E <= m) {
    // a group that gives all its candidates needs no select: the split takes
    // them whole
    if (mine) {
      s.grp_x[g] = x;
      s.grp_full[g] = full ? 1 : 0;
    }
    if (holds && !full) start(x, 1);
    const bool part = flags & 2u;
    if (g == 0) {
      c->m_fb = m - E; c->sel_ntie = 0; c->sel_k = 0; c->lst_n = 0;
      c->sel_mode = part ? kSelGroups : ((flags & 1u) ? kSelWhole : kSelGlobal);
    }
    // No group gives only some of its candidates (nothing is owed, or the
    // indebted groups go whole): what is left is one global select, which the
    // select's first pass does, and the fallback's pass has nothing to do.
    if (!part && !s.lg_on) {
      __syncthreads();
      if (warp == 0) start_global_select(s, c, 1);
    }
    return;
  }
  // tau = max{t > eps : the items at or above t number at least m}
  if (holds) {
    const int k = hbase + __popc(hb & ((1u << lane) - 1u));
    hP[k] = P;
    hD[k] = d;
    hQ[k] = q;
    hRcp[k] = rcp;
  }
  {
    const int64_t share = (m + ng - 1) / ng;
    int64_t lo = holds && x >= m ? P - (m - 1) * d : eps + 1;
    int64_t hi = holds && x >= share ? P - (share - 1) * d : eps + 1;
    for (int o = 16; o > 0; o >>= 1) {
      lo = tmax(lo, (int64_t)__shfl_xor_sync(kFull, lo, o));
      hi = tmax(hi, (int64_t)__shfl_xor_sync(kFull, hi, o));
    }
    if (lane == 0) {
      w_b[warp] = lo;
      w_c[warp] = hi;
    }
    if (g == 0) s_tau = eps;
  }
  __syncthreads();
  int64_t lo = w_b[lane], hi = w_c[lane];
  for (int o = 16; o > 0; o >>= 1) {
    lo = tmax(lo, (int64_t)__shfl_xor_sync(kFull, lo, o));
    hi = tmax(hi, (int64_t)__shfl_xor_sync(kFull, hi, o));
  }
  // Each round tests T thresholds spread over the bracket, L lanes (a power of
  // two covering the groups, at most 32) splitting the groups of one: each
  // evaluation is a chain of dependent 64-bit steps, so one per thread and
  // more rounds beat several per thread and fewer rounds.
  int logL = 0;
  while ((1 << logL) < ng && logL < 5) ++logL;
  const int L = 1 << logL, logT = 10 - logL, T = 1 << logT;  // blockDim.x == 1024 == T * L
  const int jt = g >> logL, gl = g & (L - 1);
  auto at_least = [&](int64_t t) -> int64_t {  // items at or above t, by the L lanes of a threshold
    int64_t cnt = 0;
    for (int k = gl; k < ng; k += L) cnt += items_gt(hP[k], hD[k], hQ[k], hRcp[k], t - 1);
    for (int o = L / 2; o > 0; o >>= 1) cnt += __shfl_xor_sync(kFull, cnt, o);
    return cnt;
  };
  while (hi - lo >= dmin) {
    const int64_t span = hi - lo;
    const int64_t stride = tmax<int64_t>(1, (span + T - 1) >> logT);
    const int64_t l0 = lo, h0 = hi;
    auto thr = [&](int jj) -> int64_t { return jj == T - 1 ? h0 : tmin<int64_t>(h0, l0 + 1 + stride * jj); };
    const int64_t cnt = at_least(thr(jt));
    // J = the largest threshold still holding m items: counts fall as the
    // threshold rises, so it is the number of such thresholds less one, and
    // the round's one barrier counts them
    const int J = __syncthreads_count(gl == 0 && cnt >= m) - 1;
    if (J < 0) {
      hi = lo;
    } else {
      lo = thr(J);
      hi = tmax(lo, J + 1 < T ? thr(J + 1) - 1 : h0);
    }
  }
  // each group's one item inside the bracket, if any; tau is the largest of
  // these with m items at or above it
  for (int k0 = 0; k0 < ng; k0 += T) {
    const int k = k0 + jt;
    int64_t v = eps;
    if (k < ng) {
      const int64_t dk = hD[k], pk = hP[k];
      const int64_t j = pk > hi ? (int64_t)div_d((uint64_t)(pk - hi + dk - 1), (uint64_t)dk, hRcp[k]) : 0;
      if (j < hQ[k] && pk - j * dk >= lo) v = pk - j * dk;
    }
    const int64_t cnt = at_least(tmax(v, eps + 1));
    if (gl == 0 && v > eps && cnt >= m)
      atomicMax(reinterpret_cast<long long*>(&s_tau), (long long)v);
  }
  __syncthreads();
  const int64_t tau = s_tau;
  const int64_t xa = mine ? items_gt(P, d, q, rcp, tau) : 0;
  const uint64_t qt = (mine && d > 0 && P >= tau) ? div_d((uint64_t)(P - tau), (uint64_t)d, rcp) : 0;
  const bool tied = mine && d > 0 && P >= tau && qt * (uint64_t)d == (uint64_t)(P - tau) && (int64_t)qt < q;
  if (mine) {
    s.grp_x[g] = xa + (tied ? 1 : 0);
    s.grp_full[g] = 0;
  }
  if (xa > 0 || tied) start(xa + (tied ? 1 : 0), tied ? 2 : 1);  // 2: taken only if the tie rule chooses it
  const int64_t above = warp_sum(xa);
  const int nt = __popc(__ballot_sync(kFull, tied));
  if (lane == 0) {
    w_a[warp] = above;
    w_n[warp] = nt;
  }
  __syncthreads();
  if (warp == 0) {
    const int64_t a = warp_sum(w_a[lane]);
    const int32_t n = warp_sum(w_n[lane]);
    if (lane == 0) {
      c->m_fb = 0;
      c->lst_n = 0;
      c->sel_mode = kSelGroups;
      c->sel_ntie = n;
      c->sel_k = (int32_t)(m - a);  // tied items to take, 1..ntie
    }
  }
}
__global__ void __launch_bounds__(PS_MAX_GROUPS) k_waterfill(DevState s0) {
  const DevState s = with_args(s0);
  waterfill(s, s0, s.ctl);
}

// ---- exact segmented select -------------------------------------------------
// Each active segment (a group in the debt phase, one global segment for lru
// and for the fallback) looks for the rank-th smallest key among its
// candidates of one class.  The class's key range [kmin, kmax] is cut into
// 4096 or 65536 equal buckets (a power of two wide), the candidates are counted
// by bucket, and the bucket holding the rank is found; candidates below it are
// victims, its members go to a short list that one CTA finishes exactly.
//
// Stamps are dense (a step's blocks take consecutive ones), so a range cut
// into 4096 buckets leaves a few members a segment on the list.  Cutting the
// range instead of two fixed bytes of the key keeps a segment's counts in
// 16 KB (a byte-aligned 16-bit digit took 256 KB a segment: 16.7 MB of
// histogram at 64 groups, zeroed again every step) and needs no coarse
// histogram beside it.  Measured a step, byte digits against this: staticquota
// over 100,003 blocks 90.2 -> 82.0 us, prefixshield over 256 blocks 76.2 ->
// 71.9 us and over 2^20 blocks 186.3 -> 184.5 us (the launches dominate).
//
// A class that holds blocks much older than the rest has a range far wider than
// its dense parts (a group that stood idle, a pool of hot prompts that starts to
// turn over), and a 4096th of it can hold most of a step's blocks: a list of
// thousands of members for the one CTA of list_finish.  Past 2^kWideRange stamps
// a segment is therefore cut into 65536 buckets.  Measured a step of the
// 2^20-block workloads whose stamps jump by a gap before every step, the pool
// holding a few such gaps, 4096 buckets against 65536: lru 155 -> 151 us at a
// gap of 2^22, 198 -> 154 at 2^25, 413 -> 173 at 2^28, 597 -> 230 at 2^30;
// prefixshield of 2 groups 118 -> 112, 251 -> 118, 304 -> 179, 306 -> 290.  At a
// range of 2^22 and below the longer resolve shows instead (149 -> 155, 108 ->
// 116).  2^25 is where a bucket (2^13 stamps) still leaves room for 64 groups'
// bitmaps in list_finish.  Counters for 65536 buckets are 16 MB at 64 groups; a
// handle of more groups, whose segments are shorter, keeps 4096, and so does a
// pool whose whole list fits one CTA's shared memory (4096 blocks: no
// difference at any gap).

// SMALL: of a pool of at most kWidePool blocks.
template <bool SMALL>
__device__ __forceinline__ int dig_row_log2(const DevState& s) {
  return SMALL ? kDigBits : dig_row_bits(s.N, s.G);
}
// A segment whose range takes 2^kWideBits buckets.
template <bool SMALL>
__device__ __forceinline__ bool wide_range(const DevState& s, uint64_t kmin, uint64_t kmax) {
  return ((kmax - kmin) >> kWideRange) != 0 && dig_row_log2<SMALL>(s) == kWideBits;
}
// The bucket width of a range, as a shift.
template <bool SMALL>
__device__ __forceinline__ int bucket_shift(const DevState& s, uint64_t kmin, uint64_t kmax) {
  const int bits = 64 - __clzll((long long)(kmax - kmin)), dig = wide_range<SMALL>(s, kmin, kmax) ? kWideBits : kDigBits;
  return bits > dig ? bits - dig : 0;
}
template <bool SMALL>
__device__ __forceinline__ uint4* dig_row(const DevState& s, int g) {
  return reinterpret_cast<uint4*>(s.dig_bins + ((size_t)g << dig_row_log2<SMALL>(s)));
}

// A segment as the counting pass sees it (shared memory).
struct CountSmem {
  uint64_t kmin[PS_MAX_GROUPS];
  uint64_t span[PS_MAX_GROUPS];   // kmax - kmin of a selecting segment
  uint8_t shift[PS_MAX_GROUPS];   // 64: the segment does not select
};

// Counts by bucket, thread per candidate, kU candidates a thread per
// iteration with their loads issued together (the trip count is CTA-uniform,
// as the warp-aggregated increment needs).  Neighbouring blocks were mostly
// admitted together and share buckets, so a warp's increments combine.
// Bound by the scan of N keys (8 B) and groups (2 B).
template <bool SMALL>
__device__ __forceinline__ void select_count(const DevState& s, CountSmem& sm, int mode, int fallback, int bid,
                                             int nb) {
  // indexed by group, or one entry for all
  const int nseg = mode == kSelGlobal ? 1 : s.G;
  int any = 0;
  for (int g = threadIdx.x; g < nseg; g += blockDim.x) {
    const SelSeg z = s.sel[mode == kSelGroups ? g : 0];
    const bool on = z.active && !(mode == kSelWhole && s.grp_full[g]);
    sm.kmin[g] = z.kmin;
    sm.span[g] = z.kmax - z.kmin;
    sm.shift[g] = on ? (uint8_t)bucket_shift<SMALL>(s, z.kmin, z.kmax) : (uint8_t)64;
    any |= on;
  }
  constexpr int kU = 4;
  const int64_t span = (int64_t)nb * blockDim.x;
  const int row = dig_row_log2<SMALL>(s);
  uint64_t key[kU];
  int seg[kU];
  uint32_t vw[kU];
  auto load = [&](int64_t b0) {
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t e = b0 + u * span + threadIdx.x;
      key[u] = ~0ull;
      seg[u] = 0;
      vw[u] = 0;
      if (e < s.N) {
        key[u] = s.csk[e];
        if (mode != kSelGlobal) seg[u] = s.blk_group[e];
        if (fallback) vw[u] = s.bm_victim[e >> 5];
      }
    }
  };
  load(bid * (int64_t)blockDim.x);  // the first batch beside the segments' state
  if (!__syncthreads_or(any)) return;
  for (int64_t b0 = bid * (int64_t)blockDim.x; b0 < s.N; b0 += span * kU) {
    if (b0 != bid * (int64_t)blockDim.x) load(b0);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t e = b0 + u * span + threadIdx.x;
      bool act = false;
      uint32_t idx = 0;
      if (key[u] != ~0ull && !((vw[u] >> (e & 31)) & 1)) {
        const int sh = sm.shift[seg[u]];
        const uint64_t d = key[u] - sm.kmin[seg[u]];  // keys below the range wrap past any span
        act = sh < 64 && d <= sm.span[seg[u]];
        idx = (mode == kSelGroups ? (uint32_t)seg[u] << row : 0u) + (act ? (uint32_t)(d >> sh) : 0u);
      }
      agg_inc(s.dig_bins, idx, act);
    }
  }
}

// One warp: of the 128 'rows' buckets from bucket d0 on ('bins' is the lane's
// place in the first 128; 'before' of the segment's keys lie below them), the
// one holding the segment's rank-th key, if any, as a key range [blo, bhi], and
// the rank left inside it.  The counts are cleared.
template <bool SMALL>
__device__ __forceinline__ void resolve_rows(const DevState& s, int g, const SelSeg& z, uint4* bins, int rows,
                                             uint32_t d0, uint64_t before) {
  const int lane = lane_id();
  const uint64_t rank = (uint64_t)z.rank;
  constexpr int kV = 8;  // loads in flight
  for (int k0 = 0; k0 < rows; k0 += kV) {
    uint4 v[kV];
#pragma unroll
    for (int u = 0; u < kV; ++u) v[u] = __ldcg(bins + 32 * (k0 + u));
#pragma unroll
    for (int u = 0; u < kV; ++u) {
      bins[32 * (k0 + u)] = make_uint4(0, 0, 0, 0);
      const uint32_t sum = v[u].x + v[u].y + v[u].z + v[u].w;
      if (!__any_sync(kFull, sum != 0)) continue;
      const uint32_t incl = warp_incl_scan(sum);
      uint64_t run = before + incl - sum;
      if (run < rank && rank <= run + sum) {  // one lane
        uint32_t d = d0 + 128u * (uint32_t)(k0 + u) + 4u * (uint32_t)lane;
        if (rank > run + v[u].x) { run += v[u].x; ++d;
          if (rank > run + v[u].y) { run += v[u].y; ++d;
            if (rank > run + v[u].z) { run += v[u].z; ++d; } } }
        const int sh = bucket_shift<SMALL>(s, z.kmin, z.kmax);
        SelSeg* o = s.sel + g;
        o->blo = z.kmin + ((uint64_t)d << sh);
        o->bhi = tmin<uint64_t>(o->blo + ((1ull << sh) - 1), z.kmax);
        o->rank = (int64_t)(rank - run);
      }
      before += __shfl_sync(kFull, incl, 31);
    }
  }
}
// A wide range's buckets, by a CTA of 32 warps: each sums a 32nd of them, and
// the one whose share holds the rank looks through it.
__device__ __forceinline__ void select_resolve_wide(const DevState& s, int g, const SelSeg& z) {
  __shared__ uint32_t w_sum[32];
  constexpr int kRows = (1 << kWideBits) / 128 / 32, kV = 8;
  const int warp = (int)(threadIdx.x >> 5), lane = lane_id();
  uint4* bins = dig_row<false>(s, g) + warp * kRows * 32 + lane;
  uint32_t sum = 0;
  for (int k0 = 0; k0 < kRows; k0 += kV) {
    uint4 v[kV];
#pragma unroll
    for (int u = 0; u < kV; ++u) v[u] = __ldcg(bins + 32 * (k0 + u));
#pragma unroll
    for (int u = 0; u < kV; ++u) sum += v[u].x + v[u].y + v[u].z + v[u].w;
  }
  sum = __reduce_add_sync(kFull, sum);
  if (lane == 0) w_sum[warp] = sum;
  __syncthreads();
  const uint32_t ws = w_sum[lane], ex = warp_incl_scan(ws) - ws;
  const uint64_t before = __shfl_sync(kFull, ex, warp), rank = (uint64_t)z.rank;
  if (before < rank && rank <= before + sum) {
    resolve_rows<false>(s, g, z, bins, kRows, (uint32_t)(warp * kRows) * 128u, before);
  } else if (sum) {
#pragma unroll
    for (int k = 0; k < kRows; ++k) bins[32 * k] = make_uint4(0, 0, 0, 0);
  }
}

// One CTA per segment: the bucket holding the segment's rank-th key, as a key
// range [blo, bhi], and the rank left inside it.  The counts are cleared for
// the next select.
template <bool SMALL>
__device__ __forceinline__ void select_resolve(const DevState& s, int g, const SelSeg& z) {
  if (!z.active) return;
  if (!SMALL && wide_range<SMALL>(s, z.kmin, z.kmax)) {
    select_resolve_wide(s, g, z);
    return;
  }
  constexpr int kV = 4;  // bins a thread reads at once
  uint4* bins = dig_row<SMALL>(s, g);
  uint64_t before = 0;
  for (int base = 0; base < kDigBins / kV; base += blockDim.x) {
    const int k = base + (int)threadIdx.x;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (k < kDigBins / kV) {
      v = __ldcg(bins + k);
      bins[k] = make_uint4(0, 0, 0, 0);
    }
    uint32_t tot;
    const uint64_t ex = before + block_excl_scan<uint32_t>(v.x + v.y + v.z + v.w, &tot);
    const uint64_t rank = (uint64_t)z.rank;
    if (ex < rank && rank <= ex + v.x + v.y + v.z + v.w) {  // one thread
      uint64_t run = ex;
      uint32_t d = 4u * (uint32_t)k;
      if (rank > run + v.x) { run += v.x; ++d;
        if (rank > run + v.y) { run += v.y; ++d;
          if (rank > run + v.z) { run += v.z; ++d; } } }
      const int sh = bucket_shift<SMALL>(s, z.kmin, z.kmax);
      SelSeg* o = s.sel + g;
      o->blo = z.kmin + ((uint64_t)d << sh);
      o->bhi = tmin<uint64_t>(o->blo + ((1ull << sh) - 1), z.kmax);
      o->rank = (int64_t)(rank - run);
    }
    before += tot;
  }
}

// Split: candidates below their segment's bucket are victims; the bucket's
// members go to the list, with the list's key range per segment.
struct SplitSmem {
  uint64_t lo[PS_MAX_GROUPS], hi[PS_MAX_GROUPS];  // the bucket; a segment taken whole: [~0, ~0]
  uint8_t act[PS_MAX_GROUPS];
};
__device__ __forceinline__ void select_split(const DevState& s, Ctl* c, SplitSmem& sm, int mode, int fallback,
                                             int bid, int nb) {
  const int nseg = mode == kSelGlobal ? 1 : s.G;
  const bool whole = mode != kSelGlobal && s.policy == PS_PREFIXSHIELD;
  int any = 0;
  for (int g = threadIdx.x; g < nseg; g += blockDim.x) {
    const SelSeg z = s.sel[mode == kSelGroups ? g : 0];
    const bool w = whole && s.grp_full[g];
    sm.lo[g] = w ? ~0ull : z.blo;
    sm.hi[g] = w ? ~0ull : z.bhi;
    sm.act[g] = w || z.active;
    any |= sm.act[g];
  }
  constexpr int kU = 4;
  const int64_t span = (int64_t)nb * blockDim.x;
  uint64_t key[kU];
  int seg[kU];
  uint32_t vw[kU];
  auto load = [&](int64_t b0) {
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t b = b0 + u * span + threadIdx.x;
      key[u] = ~0ull;
      seg[u] = 0;
      vw[u] = 0;
      if (b < s.N) {
        key[u] = s.csk[b];
        if (mode != kSelGlobal) seg[u] = s.blk_group[b];
        if (fallback) vw[u] = s.bm_victim[b >> 5];
      }
    }
  };
  load(bid * (int64_t)blockDim.x);  // the first batch beside the segments' state
  if (!__syncthreads_or(any)) return;
  for (int64_t b0 = bid * (int64_t)blockDim.x; b0 < s.N; b0 += span * kU) {
    if (b0 != bid * (int64_t)blockDim.x) load(b0);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t b = b0 + u * span + threadIdx.x;
      bool v = false, to_list = false;
      if (key[u] != ~0ull && !((vw[u] >> (b & 31)) & 1) && sm.act[seg[u]]) {
        v = key[u] < sm.lo[seg[u]];
        to_list = !v && key[u] <= sm.hi[seg[u]];
      }
      const unsigned bits = __ballot_sync(kFull, v);
      if (bits && lane_id() == 0) atomicOr(s.bm_victim + ((b - lane_id()) >> 5), bits);
      const unsigned lm = __ballot_sync(kFull, to_list);
      if (!lm) continue;
      const uint32_t row = mode == kSelGroups ? (uint32_t)seg[u] : 0u;
      unsigned long long base = 0;
      if (lane_id() == 0) base = atomicAdd(reinterpret_cast<unsigned long long*>(&c->lst_n), (unsigned long long)__popc(lm));
      base = __shfl_sync(kFull, base, 0);
      if (to_list) {
        const int64_t slot = (int64_t)base + __popc(lm & ((1u << lane_id()) - 1));
        s.lst_key[slot] = key[u];
        s.lst_blk[slot] = (uint32_t)b;
        s.lst_seg[slot] = (uint16_t)row;
      }
      // the list's key range per segment (lanes of one segment combined)
      const unsigned peers = __match_any_sync(kFull, to_list ? row : ~0u);
      if (to_list) {
        const uint32_t hi = (uint32_t)(key[u] >> 32), lo = (uint32_t)key[u];
        const uint32_t hmin = __reduce_min_sync(peers, hi), hmax = __reduce_max_sync(peers, hi);
        const uint32_t lmin = __reduce_min_sync(peers, hi == hmin ? lo : ~0u);
        const uint32_t lmax = __reduce_max_sync(peers, hi == hmax ? lo : 0u);
        if (lane_id() == __ffs(peers) - 1) {
          atomicMin(reinterpret_cast<unsigned long long*>(&s.sel[row].qmin), ((unsigned long long)hmin << 32) | lmin);
          atomicMax(reinterpret_cast<unsigned long long*>(&s.sel[row].qmax), ((unsigned long long)hmax << 32) | lmax);
        }
      }
    }
  }
}

// What a pass of the select has to do: its mode, or -1 for nothing.
__device__ __forceinline__ int select_mode(const Ctl* c, int fallback) {
  const int32_t st = c->status, mode = c->sel_mode;  // one round trip
  const int64_t m = c->mvict, mf = c->m_fb;
  if (st != PS_OK || m == 0) return -1;
  if (!fallback) return mode;
  return mode == kSelGroups && mf > 0 ? kSelGlobal : -1;
}
__global__ void __launch_bounds__(256) k_sel_count(DevState s, int fallback) {
  s = with_args(s);
  __shared__ CountSmem sm;
  const int mode = select_mode(s.ctl, fallback);
  if (mode >= 0) select_count<false>(s, sm, mode, fallback, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(1024) k_sel_resolve(DevState s, int fallback) {
  s = with_args(s);
  const SelSeg z = s.sel[blockIdx.x];  // in the mode's round trip
  const int mode = select_mode(s.ctl, fallback);
  if (mode == kSelGroups || (mode > 0 && blockIdx.x == 0)) select_resolve<false>(s, blockIdx.x, z);
}
__global__ void __launch_bounds__(256) k_sel_split(DevState s, int fallback) {
  s = with_args(s);
  __shared__ SplitSmem sm;
  const int mode = select_mode(s.ctl, fallback);
  if (mode >= 0) select_split(s, s.ctl, sm, mode, fallback, blockIdx.x, gridDim.x);
}

// The digits of the list's finish: bytes, from the highest one where the
// list's keys of a segment differ.
// Highest byte where kmin and kmax differ, as a shift; -1 if equal.
__device__ __forceinline__ int first_shift(uint64_t kmin, uint64_t kmax) {
  const uint64_t d = kmin ^ kmax;
  return d == 0 ? -1 : ((63 - __clzll((long long)d)) / 8) * 8;
}
// Bytes above 'shift' (shift a multiple of 8 in [0, 56]).
__device__ __forceinline__ uint64_t above_mask(int shift) { return shift >= 56 ? 0ull : (~0ull << (shift + 8)); }
// The next unresolved digit under a byte-aligned prefix mask, or -1.
__device__ __forceinline__ int next_shift(uint64_t mask) {
  if (mask == ~0ull) return -1;
  if (mask == 0) return 56;
  return __ffsll((long long)mask) - 1 - 8;
}

// The lowest 'want' set bits of f, 0 <= want <= popc(f) (a search for the
// want-th set bit by halves; __fns is a loop of up to 32 rounds).
__device__ __forceinline__ uint32_t lowest_bits(uint32_t f, int want) {
  if (want == 0) return 0;
  int left = want, p = 0;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1) {
    const int n = __popc((f >> p) & ((1u << st) - 1u));
    if (left > n) {
      left -= n;
      p += st;
    }
  }
  return f & ((2u << p) - 1u);
}
// The rest of a select on one CTA, with every segment's state in shared
// memory.  The segments' thresholds come from bitmaps of their buckets where
// those are narrow (the usual case: a bucket is a 4096th of the class's
// stamps), else from ranking the list by counting (at most kFinCountCap
// members) or from the remaining radix digits, one round per digit, over the
// list in shared memory (at most kFinCap members) or in global memory; then
// Eq. 7's tie rule, then the list's victims.  One launch for every list
// length keeps the step graph free of conditional nodes here.
struct FinSeg {
  uint64_t prefix, mask;
  int64_t rank;
  int32_t active, incl;
};
constexpr size_t kFinList = (size_t)kFinCap * 8 + (size_t)kFinRows * kRadixBins * 4 + (size_t)kFinCap * 2;
constexpr int kFinWords = (int)(kFinList / 4);  // bitmap words in the list's place
constexpr int kFinSegWords = 1024;              // of one segment (one warp searches them)
constexpr size_t kFinSmem = kFinList + (size_t)PS_MAX_GROUPS * (sizeof(FinSeg) + 8 + 4 + 2);

__device__ __forceinline__ void list_finish(const DevState& s, Ctl* c, unsigned char* fin_smem, int mode, int64_t n) {
  FinSeg* sl = reinterpret_cast<FinSeg*>(fin_smem);
  uint64_t* blo = reinterpret_cast<uint64_t*>(sl + PS_MAX_GROUPS);  // the segments' buckets
  int32_t* woff = reinterpret_cast<int32_t*>(blo + PS_MAX_GROUPS);  // and bitmaps
  int16_t* wlen = reinterpret_cast<int16_t*>(woff + PS_MAX_GROUPS);
  uint64_t* lkey = reinterpret_cast<uint64_t*>(wlen + PS_MAX_GROUPS);
  uint32_t* fh = reinterpret_cast<uint32_t*>(lkey + kFinCap);
  uint16_t* lseg = reinterpret_cast<uint16_t*>(fh + kFinRows * kRadixBins);
  __shared__ int16_t row_of[PS_MAX_GROUPS];
  __shared__ int16_t seg_of_row[PS_MAX_GROUPS];
  __shared__ int s_nrows;
  const bool single = mode != kSelGroups;
  // a pass over the groups also starts the fallback's select (the groups'
  // final take counts are known here)
  const bool start_fb = !single && s.policy == PS_PREFIXSHIELD;
  const int nseg = single ? 1 : s.G;
  if (n == 0) {  // no segment selects
    if (start_fb && threadIdx.x < 32) start_global_select(s, c, 1);
    return;
  }
  const bool small = n <= kFinCap;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  // each thread's first member, loaded beside the segments' state
  uint64_t my_key = 0;
  uint32_t my_blk = 0;
  int my_seg = 0;
  if ((int64_t)threadIdx.x < n) {
    my_key = s.lst_key[threadIdx.x];
    my_blk = s.lst_blk[threadIdx.x];
    my_seg = s.lst_seg[threadIdx.x];
  }
  // A segment's list members lie in its bucket [blo, bhi], and stamps are
  // unique: where the buckets are narrow enough, each segment gets a bitmap of
  // its bucket, the members set their bits, and the rank-th set bit is the
  // threshold, whatever the list's length.
  uint32_t* words = reinterpret_cast<uint32_t*>(lkey);  // lkey, fh and lseg: not in use on this path
  bool by_bits = n > kFinShort;  // counting a short list needs no bitmaps set up
  int64_t wtot = 0;
  for (int g0 = 0; g0 < nseg; g0 += blockDim.x) {
    const int g = g0 + (int)threadIdx.x;
    int64_t nw = 0;
    if (g < nseg) {
      const SelSeg z = s.sel[g];
      const bool listed = z.qmin <= z.qmax;
      // the list's members share the bits above the highest byte where their
      // smallest and largest key differ: those are fixed already
      const int fs = listed ? first_shift(z.qmin, z.qmax) : 56;
      const uint64_t mask = fs < 0 ? ~0ull : above_mask(fs);
      sl[g] = FinSeg{listed ? z.qmin & mask : 0ull, listed ? mask : ~0ull, z.rank, listed ? z.active : 0, z.incl};
      blo[g] = z.blo;
      if (by_bits && sl[g].active) nw = (int64_t)tmin<uint64_t>((z.bhi - z.blo) >> 5, kFinSegWords) + 1;
    }
    by_bits = by_bits && !__syncthreads_or(nw > kFinSegWords);
    if (!by_bits) continue;
    int64_t tot;
    const int64_t ex = wtot + block_excl_scan(nw, &tot);
    if (g < nseg) {
      woff[g] = (int32_t)tmin<int64_t>(ex, kFinWords);
      wlen[g] = (int16_t)nw;
    }
    wtot += tot;
  }
  by_bits = by_bits && wtot <= kFinWords;
  __syncthreads();
  if (by_bits) {
    for (int w = threadIdx.x; w < (int)wtot; w += blockDim.x) words[w] = 0;
    __syncthreads();
    for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
      const bool mine = e == (int64_t)threadIdx.x;
      const int g = mine ? my_seg : (int)s.lst_seg[e];
      const uint64_t d = (mine ? my_key : ldcg_u64(s.lst_key + e)) - blo[g];
      if (sl[g].active) atomicOr(&words[woff[g] + (int)(d >> 5)], 1u << (d & 31));
    }
    __syncthreads();
    for (int g = warp; g < nseg; g += blockDim.x >> 5) {
      if (!sl[g].active) continue;
      const int nw = wlen[g];
      int64_t left = sl[g].rank;
      for (int w0 = 0; w0 < nw; w0 += 32) {
        const uint32_t x = w0 + lane < nw ? words[woff[g] + w0 + lane] : 0u;
        const int p = __popc(x), incl = warp_incl_scan(p);
        const int tot = __shfl_sync(kFull, incl, 31);
        if (left > tot) {
          left -= tot;
          continue;
        }
        if (incl - p < left && left <= incl) {  // one lane
          const uint32_t low = lowest_bits(x, (int)(left - (incl - p)));
          sl[g].prefix = blo[g] + (uint64_t)(w0 + lane) * 32 + (uint64_t)(31 - __clz((int)low));
          sl[g].mask = ~0ull;
        }
        break;
      }
    }
  } else if (small) {
    for (int64_t e = threadIdx.x; e < n; e += blockDim.x) { lkey[e] = s.lst_key[e]; lseg[e] = s.lst_seg[e]; }
  }
  __syncthreads();
  auto key_at = [&](int64_t e) -> uint64_t { return small ? lkey[e] : ldcg_u64(s.lst_key + e); };
  auto seg_at = [&](int64_t e) -> int { return small ? (int)lseg[e] : (int)s.lst_seg[e]; };
  // A short list (the usual case): a segment's threshold key is its member
  // whose rank among the segment's list members (keys are unique) is its
  // remaining rank - 1; L lanes rank one member by counting, so no digit
  // rounds (and their barriers) are needed.
  const bool by_count = !by_bits && small && n <= kFinCountCap;
  if (by_count) {
    int L = 32;
    while (L * (int)n > (int)blockDim.x) L >>= 1;  // kFinCountCap <= blockDim.x: L >= 1
    const int e = (int)threadIdx.x / L, l = (int)threadIdx.x % L;
    const bool in = e < n && sl[lseg[e]].active;
    const int g = in ? lseg[e] : -1;
    const uint64_t key = in ? lkey[e] : 0;
    int below = 0;
    if (in)
      for (int j = l; j < n; j += L) below += (lseg[j] == g && lkey[j] < key) ? 1 : 0;
    for (int o = L / 2; o > 0; o >>= 1) below += __shfl_xor_sync(kFull, below, o);
    // one member per segment matches; nothing here writes the ranks read
    if (in && l == 0 && below == sl[g].rank - 1) {
      sl[g].prefix = key;
      sl[g].mask = ~0ull;
    }
    __syncthreads();
  }
  for (int iter = 0; !by_bits && !by_count && iter < 8; ++iter) {  // at most 8 digits in a 64-bit key
    {
      int k = 0;
      for (int base = 0; base < nseg; base += blockDim.x) {
        const int g = base + threadIdx.x;
        const bool counts = g < nseg && sl[g].active && next_shift(sl[g].mask) >= 0;
        int tot;
        const int ex = block_excl_scan((int)counts, &tot);
        if (g < nseg) row_of[g] = counts ? (int16_t)(k + ex) : (int16_t)-1;
        if (counts) seg_of_row[k + ex] = (int16_t)g;
        k += tot;
      }
      if (threadIdx.x == 0) s_nrows = k;
      __syncthreads();
    }
    const int nrows = s_nrows;
    if (nrows == 0) break;
    for (int r0 = 0; r0 < nrows; r0 += kFinRows) {
      const int rn = tmin(kFinRows, nrows - r0);
      for (int k = threadIdx.x; k < rn * kRadixBins; k += blockDim.x) fh[k] = 0;
      __syncthreads();
      for (int64_t e0 = 0; e0 < n; e0 += blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        bool act = false;
        uint32_t idx = 0;
        if (e < n) {
          const int seg = seg_at(e);
          const int row = row_of[seg];
          if (row >= r0 && row < r0 + rn) {
            const uint64_t key = key_at(e);
            if ((key & sl[seg].mask) == sl[seg].prefix) {
              act = true;
              const int sh = next_shift(sl[seg].mask);
              idx = (uint32_t)(row - r0) * kRadixBins + (uint32_t)((key >> sh) & (kRadixBins - 1));
            }
          }
        }
        agg_inc(fh, idx, act);
      }
      __syncthreads();
      for (int r = warp; r < rn; r += blockDim.x >> 5) {
        const int seg = seg_of_row[r0 + r];
        const int sh = next_shift(sl[seg].mask);
        const int64_t rank = sl[seg].rank;
        uint32_t v[kRadixBins / 32];
        uint32_t sum = 0;
#pragma unroll
        for (int j = 0; j < kRadixBins / 32; ++j) { v[j] = fh[r * kRadixBins + lane * (kRadixBins / 32) + j]; sum += v[j]; }
        const uint32_t incl = warp_incl_scan(sum);
        const uint32_t excl = incl - sum;
        if ((uint64_t)excl < (uint64_t)rank && (uint64_t)rank <= (uint64_t)incl) {
          uint32_t run = excl;
          int d = 0;
          for (int j = 0; j < kRadixBins / 32; ++j) {
            if ((uint64_t)rank <= (uint64_t)(run + v[j])) { d = lane * (kRadixBins / 32) + j; break; }
            run += v[j];
          }
          sl[seg].prefix |= (uint64_t)d << sh;
          sl[seg].mask |= (uint64_t)(kRadixBins - 1) << sh;
          sl[seg].rank = rank - run;
        }
      }
      __syncthreads();
    }
  }
  // Eq. 7's tie rule at tau: among the groups holding an item at exactly tau,
  // the sel_k with the smallest candidate keys take it
  if (!single && c->sel_ntie > 0) {
    const int64_t k = c->sel_k;
    for (int g = threadIdx.x; g < nseg; g += blockDim.x) {
      if (!(sl[g].active && sl[g].incl == 2)) continue;
      int rank = 0;
      const uint64_t own = sl[g].prefix;
#pragma unroll 4
      for (int h = 0; h < nseg; ++h)
        rank += (int)(sl[h].active != 0) & (int)(sl[h].incl == 2) & (int)(sl[h].prefix < own);
      const bool chosen = rank < k;
      s.grp_x[g] -= chosen ? 0 : 1;
      fh[g] = chosen ? 1 : 0;  // applied after every thread has read the flags
    }
    __syncthreads();
    for (int g = threadIdx.x; g < nseg; g += blockDim.x)
      if (sl[g].active && sl[g].incl == 2) sl[g].incl = (int32_t)fh[g];
    __syncthreads();
  }
  // the list's victims: keys below (or at, if incl) the threshold
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    const bool mine = e == (int64_t)threadIdx.x;
    const uint64_t key = mine ? my_key : ldcg_u64(s.lst_key + e);
    const FinSeg& f = sl[mine ? my_seg : (int)s.lst_seg[e]];
    if (f.active && (key < f.prefix || (f.incl && key == f.prefix))) {
      const uint32_t b = mine ? my_blk : s.lst_blk[e];
      atomicOr(s.bm_victim + (b >> 5), 1u << (b & 31));
    }
  }
  if (start_fb) {
    __syncthreads();  // every reader of segment 0's state is done
    if ((threadIdx.x >> 5) == 0) start_global_select(s, c, 1);
  }
}
__global__ void __launch_bounds__(1024) k_list_finish(DevState s, int fallback) {
  s = with_args(s);
  extern __shared__ __align__(16) unsigned char fin_smem[];
  const int64_t n = s.ctl->lst_n;  // in the mode's round trip
  const int mode = select_mode(s.ctl, fallback);
  if (mode >= 0) list_finish(s, s.ctl, fin_smem, mode, n);
}

// TakeTrueFree (Alg. 2) and the step's id lists (allocated, evicted,
// invalidated), all ascending, from the bitmaps.  Each CTA owns kBmChunk
// bitmap words.  Pass 1 counts each chunk's free, evicted and invalidated
// ids.  Pass 2: the ftake smallest free ids are taken greedily from low ids,
// so a chunk takes min(ftake, free before it + its own) - min(ftake, free
// before it) of its free ids, its lowest ones; with the victims they form the
// allocated set, whose ids become resident.
__device__ __forceinline__ uint32_t free_word(const DevState& s, int64_t w) {
  uint32_t f = ~s.res_bits[w];
  const int64_t hi = (w + 1) * 32;
  if (hi > s.N) f &= (1u << (uint32_t)(32 - (hi - s.N))) - 1u;
  return f;
}
__global__ void __launch_bounds__(kBmChunk) k_bm_count(DevState s) {
  s = with_args(s);
  const Ctl* c = s.ctl;
  const int64_t w = (int64_t)blockIdx.x * kBmChunk + threadIdx.x;
  const int nchunks = gridDim.x;
  const bool in = w < s.nwords;
  const int32_t st = c->status;
  const int64_t ftake = c->ftake;
  const int nv = in ? __popc(s.bm_victim[w]) : 0;
  const int ni = in ? __popc(s.bm_inval[w]) : 0;
  const int fr = in ? __popc(free_word(s, w)) : 0;
  if (st != PS_OK) return;
  const int nf = ftake > 0 ? fr : 0;
  const int tv = block_sum(nv), ti = block_sum(ni), tf = block_sum(nf);
  if (threadIdx.x == 0) {
    s.bm_chunk_cnt[0 * nchunks + blockIdx.x] = tf;
    s.bm_chunk_cnt[1 * nchunks + blockIdx.x] = tv;
    s.bm_chunk_cnt[2 * nchunks + blockIdx.x] = ti;
  }
}
// Counts are packed into one 64-bit word (three 21-bit fields: a chunk holds
// at most 8192 ids of each kind), so one block scan carries all three.
__device__ __forceinline__ uint64_t pack3(uint64_t a, uint64_t b, uint64_t c) { return a | b << 21 | c << 42; }
__device__ __forceinline__ int64_t field3(uint64_t v, int k) { return (int64_t)((v >> (21 * k)) & 0x1FFFFF); }
// The ids of nw bitmap words from w0 on to the three lists: a warp takes a
// word, a lane an id, so a list's stores coalesce (a thread a word wrote up to
// 32 ids one after the other, in as many rounds as the fullest word).
struct ListSmem {
  uint32_t word[3][kBmChunk];  // allocated, evicted, invalidated ids of each word
  int32_t base[3][kBmChunk];   // where they go
};
__device__ __forceinline__ void write_ids(const DevState& s, const ListSmem& sm, int64_t w0, int nw) {
  int32_t* outs[3] = {s.out.admitted_ids, s.out.evicted_ids, s.out.invalidated_ids};
  const int lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  for (int w = (int)(threadIdx.x >> 5); w < nw; w += (int)(blockDim.x >> 5)) {
    if (!(sm.word[0][w] | sm.word[2][w])) continue;  // victims are allocated again
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t bits = sm.word[k][w];
      const int64_t o = (int64_t)sm.base[k][w] + __popc(bits & lt);
      if (((bits >> lane) & 1u) && o < s.max_blocks) outs[k][o] = (int32_t)((w0 + w) * 32 + lane);
    }
  }
}
constexpr int kBmThreads = 512;
template <int NT>  // threads of the CTA
__device__ __forceinline__ void list_chunk(const DevState& s, Ctl* c, ListSmem& sm, int chunk, int nchunks) {
  const int32_t st = c->status;
  const int t = (int)threadIdx.x;
  const int64_t w0 = (int64_t)chunk * kBmChunk, w = w0 + t;
  const bool in = t < kBmChunk && w < s.nwords;  // the first kBmChunk threads hold a word each
  const int64_t ftake = c->ftake;
  const uint32_t vic = in ? s.bm_victim[w] : 0u, inv = in ? s.bm_inval[w] : 0u;
  const uint32_t fw = in ? free_word(s, w) : 0u;
  if (st != PS_OK) return;
  // earlier chunks' free, evicted and invalidated ids
  int64_t fb = 0, vb = 0, ib = 0;
  for (int j = t; j < chunk; j += NT) {  // (none in a single chunk)
    fb += s.bm_chunk_cnt[0 * nchunks + j];
    vb += s.bm_chunk_cnt[1 * nchunks + j];
    ib += s.bm_chunk_cnt[2 * nchunks + j];
  }
  {
    __shared__ int64_t s_before[3][NT / 32];
    fb = warp_sum(fb); vb = warp_sum(vb); ib = warp_sum(ib);
    if (lane_id() == 0) { s_before[0][t >> 5] = fb; s_before[1][t >> 5] = vb; s_before[2][t >> 5] = ib; }
    __syncthreads();
    const bool hold = lane_id() < NT / 32;
    fb = warp_sum(hold ? s_before[0][lane_id()] : (int64_t)0);
    vb = warp_sum(hold ? s_before[1][lane_id()] : (int64_t)0);
    ib = warp_sum(hold ? s_before[2][lane_id()] : (int64_t)0);
  }
  const uint32_t f = ftake > 0 ? fw : 0u;
  uint64_t tot1;
  const uint64_t ex1 = block_excl_scan<uint64_t>(pack3(__popc(f), __popc(vic), __popc(inv)), &tot1);
  // this word's taken free ids: the chunk's lowest take_here free ids
  const int64_t take_here = tmin(ftake, fb + field3(tot1, 0)) - tmin(ftake, fb);
  const int64_t fl = field3(ex1, 0);
  const int64_t want = tmin<int64_t>(tmax<int64_t>(take_here - fl, 0), __popc(f));
  const uint32_t alloc = lowest_bits(f, (int)want) | vic;
  // taken ids before the word: the free ones before it, up to take_here
  const int64_t ex2 = tmin(fl, take_here) + field3(ex1, 1);
  if (in) {
    s.res_bits[w] |= alloc;  // every allocated id is resident after the step
    s.bm_victim[w] = 0;
    s.bm_inval[w] = 0;
  }
  if (t < kBmChunk) {
    sm.word[0][t] = alloc;
    sm.word[1][t] = vic;
    sm.word[2][t] = inv;
    sm.base[0][t] = (int32_t)(vb + tmin(ftake, fb) + ex2);
    sm.base[1][t] = (int32_t)(vb + field3(ex1, 1));
    sm.base[2][t] = (int32_t)(ib + field3(ex1, 2));
  }
  if (chunk == nchunks - 1 && t == 0) {
    c->n_alloc = vb + tmin(ftake, fb) + take_here + field3(tot1, 1);
    c->n_evicted = vb + field3(tot1, 1);
  }
  __syncthreads();
  write_ids(s, sm, w0, (int)tmin<int64_t>(kBmChunk, s.nwords - w0));
}
__global__ void __launch_bounds__(kBmThreads, 3) k_bm_write(DevState s) {
  s = with_args(s);
  __shared__ ListSmem sm;
  list_chunk<kBmThreads>(s, s.ctl, sm, blockIdx.x, gridDim.x);
}

// The whole select of a small pool, and its id lists, by one CTA: the stage
// kernels above as phases between CTA barriers.  With a few thousand blocks
// each of those kernels is a launch and a chain of dependent loads around a
// few hundred instructions, ten launches under PrefixShield (four of them the
// fallback's, which mostly finds nothing to do) and six under LRU.
// Measured a step, stage kernels against this: prefixshield over 512 blocks
// 55.9 -> 50.7 us, over 2048 59.5 -> 53.4, over 4096 66.2 -> 65.5 (2 groups)
// and 62.6 -> 57.0 (32); over 8192 it lost from 16 groups on (65.7 -> 72.7 us
// with 32).  LRU has no fallback to skip: 50.7 -> 48.3 us over 512 blocks,
// 53.7 -> 53.1 over 2048, 56.4 -> 57.1 over 4096.  StaticQuota selects in
// every group on every step, which one CTA does more slowly (2048 blocks,
// 8 groups: 57.5 -> 58.5 us; 32 groups: 58.7 -> 65.2), so it is left alone.
constexpr int kSmallThreads = 1024;
constexpr int kSmallPool = 4 * kSmallThreads;     // one batch of loads a thread in the counts and in the split
static_assert(kSmallPool <= kWidePool, "a warp resolves a small pool's segment: no 2^kWideBits buckets there");
constexpr int kSmallPoolLru = 2 * kSmallThreads;
constexpr int kSmallGroups = kSmallThreads / 32;  // a warp for each segment
inline bool small_select(const DevState& s) {
  if (s.lg_on) return false;
  return s.policy == PS_PREFIXSHIELD ? s.N <= kSmallPool && s.G <= kSmallGroups
                                     : s.policy == PS_LRU && s.N <= kSmallPoolLru;
}
// select_resolve by one warp (4096 buckets).
__device__ __forceinline__ void select_resolve_warp(const DevState& s, int g) {
  const SelSeg z = s.sel[g];
  if (z.active) resolve_rows<true>(s, g, z, dig_row<true>(s, g) + lane_id(), kDigBins / 128, 0, 0);
}
__device__ __forceinline__ void small_pass(const DevState& s, Ctl* c, unsigned char* smem, int mode, int fallback) {
  select_count<true>(s, *reinterpret_cast<CountSmem*>(smem), mode, fallback, 0, 1);
  __syncthreads();
  if (mode == kSelGroups) {
    const int g = (int)(threadIdx.x >> 5);
    if (g < s.G) select_resolve_warp(s, g);
  } else {
    const SelSeg z = s.sel[0];
    select_resolve<true>(s, 0, z);
  }
  __syncthreads();
  select_split(s, c, *reinterpret_cast<SplitSmem*>(smem), mode, fallback, 0, 1);
  __syncthreads();
  list_finish(s, c, smem, mode, c->lst_n);
  __syncthreads();
}
__global__ void __launch_bounds__(kSmallThreads) k_small_select(DevState s0) {
  const DevState s = with_args(s0);
  extern __shared__ __align__(16) unsigned char fin_smem[];
  Ctl* c = s.ctl;
  if (s.policy == PS_LRU) {
    if (threadIdx.x < 32) start_global_select(s, c, 0);
  } else {
    waterfill(s, s0, c);
  }
  __syncthreads();
  const int mode = select_mode(c, 0);
  if (mode >= 0) {
    small_pass(s, c, fin_smem, mode, 0);
    const int again = s.policy == PS_PREFIXSHIELD ? select_mode(c, 1) : -1;
    if (again >= 0) small_pass(s, c, fin_smem, again, 1);
  }
  list_chunk<kSmallThreads>(s, c, *reinterpret_cast<ListSmem*>(fin_smem), 0, 1);
}

// Stage 6: place granted claims, a thread per claim of the step (k_instep
// listed them; a thread per position left most lanes idle: at 2^20 blocks half
// of the positions are hits).  The allocated ids (ascending) go to the granted
// keys in (request, position) order; each new block carries the metadata
// OnCacheFullBlocks attached plus any in-step touches.  An allocated id that
// is still resident is a victim (every victim is allocated again in its step):
// its old content leaves the pool first, in the same thread (Alg. 2 Evict:
// table entry and record), so no other thread ever sees the block between its
// two contents.  Each claim's thread then clears its claim-map slot (no other
// thread reads it here).  The first R threads also commit a request's
// OnRequest / RecordSuccessfulAdmission history update each.
__global__ void __launch_bounds__(kThreads, 5) k_insert(DevState s) {
  s = with_args(s);
  Ctl* c = s.ctl;
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // in one round trip (the claims' list reaches to max_blocks)
  const int32_t st = c->status;
  const int64_t nclaims = c->total_claims, n_alloc = c->n_alloc;
  const uint64_t base = c->stamp_base;
  const uint64_t cp = q < s.max_blocks ? s.claim_pos[q] : 0ull;
  if (st != PS_OK) return;
  bool placed = false, evicted = false;
  uint32_t g = 0, gold = 0;
  if (q < nclaims) {
    // Rounds of loads, each issued as a whole before anything is stored (a
    // store or an atomic in between would hold back the loads after it): the
    // claim's position; its and its request's records; the id and the claim;
    // the id's old record.
    const uint32_t i = (uint32_t)(cp >> 32);
    const int64_t pos = (int64_t)(uint32_t)cp;
    const int si = s.rq_s[i], a = s.rq_a[i], cbase = s.rq_cbase[i], n = s.rq_n[i], pbase = s.rq_pbase[i];
    const int cid = s.rq_cid[i];
    const uint64_t p = s.rq_p[i], key = s.pos_key[pos];
    const uint8_t knew = s.rq_knew[i];
    const uint32_t slot = s.pos_claim[pos];
    g = (uint32_t)s.in_group[i];
    const int m = (int)(pos - pbase);
    const bool grant = m < si + a;
    const int64_t rank = (int64_t)cbase + (m - si);
    ClaimEntry e{};
    uint32_t b = kNone;
    if (grant) {
      e = s.claims[slot];
      if (rank < n_alloc) b = (uint32_t)s.out.admitted_ids[rank];
    }
    uint8_t ofl = 0;
    uint32_t oslot = 0;
    uint64_t okey = 0;
    uint16_t ogrp = 0;
    if (b < (uint64_t)s.N) {
      // a resident id is a victim, whose old content (table entry, record)
      // leaves first
      ofl = s.blk_flags[b];
      oslot = s.blk_slot[b];
      okey = s.blk_key[b];
      ogrp = s.blk_group[b];
    }
    if (grant) {
      if (b >= (uint64_t)s.N) {
        c->internal_error = 1;  // the allocated set is short: never expected
      } else {
        if (ofl & 1) {
          table_delete_known(s, oslot, okey, ogrp);
          gold = ogrp;
          evicted = true;
        }
        const uint32_t nslot = table_insert(s, key, g, b);
        // the latest request that touched it: an in-step toucher's stamp, or
        // the owner's own
        const uint64_t st = tmax<uint64_t>(e.stamp, make_stamp(base, pbase, n, m));
        s.blk_key[b] = key;
        s.blk_group[b] = (uint16_t)g;
        s.blk_contract[b] = (uint8_t)cid;
        s.blk_prefix[b] = p;
        s.blk_klass[b] = e.promo != kNone ? (uint8_t)kReuse : knew;
        s.blk_stamp[b] = st;
        if (s.lg_on) s.lg_slot[st - base] = b;
        s.blk_acc[b] = e.tcnt;
        s.blk_freq[b] = e.tcnt;
        s.blk_flags[b] = 1;
        s.blk_slot[b] = nslot;
        placed = true;  // its resident bit was set with the allocated set
      }
    }
    s.claims[slot] = empty_claim();
  }
  if (q < s.R) {  // history commit of request q (no entry: no full block)
    const uint32_t hs = s.rq_hs[q];
    const int a = s.rq_a[q];
    if (hs != kNone) {
      atomicAdd(&s.hist[hs].refadm, 1u);
      if (a > 0) atomicOr(&s.hist[hs].refadm, 0x80000000u);
    }
  }
  if (q == 0) c->hist_live += c->hist_new;
  agg_stat(s, gold, PS_STAT_EVICTED_BLOCKS, 1, evicted);
  agg_stat(s, gold, PS_STAT_RESIDENT_BLOCKS, -1, evicted);
  agg_stat(s, g, PS_STAT_RESIDENT_BLOCKS, 1, placed);
  const int k = __popc(__ballot_sync(kFull, placed)) - __popc(__ballot_sync(kFull, evicted));
  if (lane_id() == 0 && k) atomic_add_i64(&c->n_resident, k);
}

// Step end: the outputs' counts and status, then the clock, the step index
// and the next step's first recency stamp.
__global__ void k_finalize(DevState s) {
  s = with_args(s);
  Ctl* c = s.ctl;
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int32_t st = c->internal_error ? PS_ERR_DEVICE_STATUS : c->status;
  s.out.counts[3] = st;
  // the queues' logs no longer agree with the pool: no later step uses them
  if (c->internal_error && s.lg_on) c->lg_lost = 1;
  if (c->status != PS_OK) return;
  s.out.counts[0] = (int32_t)c->need;
  s.out.counts[1] = (int32_t)c->n_evicted;
  s.out.counts[2] = (int32_t)c->n_inval;
  c->t_prev = s.now;
  c->step += 1;
  c->stamp_base += c->nblocks;
  if (s.policy == PS_S3FIFO) {  // the queue arrays the step wrote become current
    const S3Plan* pl = s.s3_plan;
    const int64_t n_ins = c->need < c->n_alloc ? c->need : c->n_alloc;
    c->s3_len[0] = pl->nKeepS + n_ins - pl->hits;
    c->s3_len[1] = pl->nKeepM + pl->nMid + pl->hits;
    c->s3_buf ^= 1;
    c->s3_ctr = pl->ctr_end + (uint64_t)n_ins;
    c->ghost_live -= pl->hits;
    c->s3_nS = c->s3_len[0];
    c->s3_nM = c->s3_len[1];
  }
}

// ===========================================================================
// host launchers
static int grid_for(int64_t items, int threads, int max_ctas) {
  int64_t g = (items + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > max_ctas) g = max_ctas;
  return (int)g;
}

void launch_init(const DevState& s, cudaStream_t st) {
  k_init_blocks<<<grid_for((int64_t)kClaimWays << s.cl_nbuckets_log2, 256, 152 * 8), 256, 0, st>>>(s);
  k_init_ctl<<<1, 1024, 0, st>>>(s);
  launch_queue_init(s, st);
}

template <int BS>
static void launch_hash_lookup_t(const DevState& s, cudaStream_t st, int32_t* probe_out) {
  // persistent: the CTAs that fit at once (more only queue behind them)
  int dev = 0, nsm = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // 8 warps a CTA, or fewer where all chunks have a warp then and more SMs
  // share them (a chunk's probes keep an SM's L1 busy: 8 warps on each of 37
  // SMs took longer than 2 on each of 148)
  int warps = 8;
  while (warps > 1 && s.max_segments <= (int64_t)nsm * (warps / 2)) warps >>= 1;
  const int64_t want = (s.max_segments + warps - 1) / warps;
  const int64_t most = (int64_t)nsm * kHashCtasPerSm * 8 / warps;
  const int grid = (int)(want < most ? want : most);
  k_hash_lookup<BS><<<grid > 0 ? grid : 1, 32 * warps, 0, st>>>(s, probe_out);
}
static int32_t launch_hash_lookup(const DevState& s, cudaStream_t st, int32_t* probe_out) {
  switch (s.bs) {
    case 2: launch_hash_lookup_t<2>(s, st, probe_out); break;
    case 4: launch_hash_lookup_t<4>(s, st, probe_out); break;
    case 8: launch_hash_lookup_t<8>(s, st, probe_out); break;
    case 16: launch_hash_lookup_t<16>(s, st, probe_out); break;
    case 32: launch_hash_lookup_t<32>(s, st, probe_out); break;
    case 64: launch_hash_lookup_t<64>(s, st, probe_out); break;
    default: return PS_ERR_INVALID_ARG;
  }
  return PS_OK;
}

void configure_kernels(const DevState& s) {
  (void)s;
  cudaFuncSetAttribute(k_list_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinSmem);
  cudaFuncSetAttribute(k_small_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinSmem);
  cudaFuncSetAttribute(k_cand, cudaFuncAttributeMaxDynamicSharedMemorySize, PS_MAX_GROUPS * kClasses * 5 * 4);
  cudaFuncSetAttribute(k_grant, cudaFuncAttributeMaxDynamicSharedMemorySize, PS_MAX_GROUPS * PS_MAX_CONTRACTS * 8);
}

int32_t launch_step(const DevState& s, cudaStream_t st, StepTrace* tr, const CaptureCtx* cap) {
  // grids depend only on the handle's bounds (a captured graph serves any step)
  const int R = s.max_requests;
  const int pgrid = grid_for(s.max_blocks, kThreads, 1 << 30);
  const int prgrid = grid_for(s.max_blocks + R, kThreads, 1 << 30);
  const int igrid = grid_for(s.max_blocks > R ? s.max_blocks : R, kThreads, 1 << 30);
  // The select's scans, four CTAs an SM: with eight, a step that has nothing to
  // select waits for as many CTAs to come and go four times (prefixshield over
  // 2^20 blocks: a step of one request 69.4 -> 66.0 us, of 4096 147.6 -> 142.6).
  const int cgrid = grid_for(s.N, 256, 152 * 4);
  int launches = 0;
  auto mark = [&](int stage) {
    // under capture an external record becomes an event-record node of the
    // graph (the flag is refused outside a capture)
    if (tr && tr->timing) {
      if (cap) cudaEventRecordWithFlags(tr->ev[stage], st, cudaEventRecordExternal);
      else cudaEventRecord(tr->ev[stage], st);
    }
  };
#define PS_LAUNCH(...) do { __VA_ARGS__; ++launches; } while (0)
  mark(0);
  PS_LAUNCH(launch_k(k_validate, grid_for(R, kValTile, 1 << 20), kValTile, 0, st, s, nullptr));
  mark(1);
  if (launch_hash_lookup(s, st, nullptr) != PS_OK) return PS_ERR_INVALID_ARG;
  ++launches;
  mark(2);
  PS_LAUNCH(launch_k(k_claims, prgrid, kThreads, 0, st, s));
  mark(3);
  // The candidates read pins and residency (final from here on) and the class
  // and stamp of unpinned blocks, which S3-S4 leave alone: under capture
  // they are counted on a side branch that runs beside the rest of S3-S4.
  // The candidate scan writes per-step scratch only, so it forks beside the
  // grants (a step the grant then fails ignores what it wrote); the indexed
  // queues' count applies the step's pins to persistent counts, so it waits
  // for the grant's verdict.
  const bool fork = cap && s.policy != PS_S3FIFO;
  const bool early = fork && !s.lg_on;
  cudaStream_t cs = st;
  auto launch_cand = [&]() -> int32_t {
    if (fork) {
      if (cudaEventRecord(cap->fork, st) != cudaSuccess || cudaStreamWaitEvent(cap->side, cap->fork, 0) != cudaSuccess)
        return PS_ERR_CUDA;
      cs = cap->side;
    }
    const int cand_smem = (s.policy == PS_PREFIXSHIELD || s.policy == PS_STATICQUOTA ? s.G : 1) * kClasses * 5 * 4;
    if (s.lg_on) {
      if (launch_queue_cand(s, cs, &launches) != PS_OK) return PS_ERR_CUDA;
    } else if (s.policy != PS_S3FIFO) {
      // two 512-thread CTAs an SM, less than all of them: the grants' CTA holds
      // an SM meanwhile, and CTAs left over would run as a second wave
      PS_LAUNCH(k_cand<<<fork ? 2 * 152 - 8 : grid_for(s.N, 1024 * 4, 152), fork ? 512 : 1024, cand_smem, cs>>>(s));
    }
    if (fork && cudaEventRecord(cap->join, cs) != cudaSuccess) return PS_ERR_CUDA;
    return PS_OK;
  };
  if (early && launch_cand() != PS_OK) return PS_ERR_CUDA;
  if (s.policy == PS_STATICQUOTA) PS_LAUNCH(launch_k(k_grant_quota, s.G, 1024, 0, st, s));
  PS_LAUNCH(launch_k(k_grant, 1, 1024, (size_t)s.G * s.C * 8, st, s));
  if (!early && launch_cand() != PS_OK) return PS_ERR_CUDA;
  // The in-step hits, the metering and the touch passes feed the insertion
  // (the claims' in-step touches, the new blocks' class) and the statistics;
  // the select needs only the step's debts, which k_grant settles.  Under
  // capture they run on a second parallel branch beside the select, joined
  // before the insertion (which reads, then clears, the claim entries).
  // The S3-FIFO select reads only unpinned blocks' frequencies, pin tags and
  // residency, none of which these kernels write (a touch changes hit, so
  // pinned, blocks), so it runs beside them too.  The indexed queues keep
  // them in line (their select reads the touched blocks' new stamps).
  const bool fork2 = cap != nullptr && !s.lg_on;
  cudaStream_t ms = st;
  if (fork2) {
    if (cudaEventRecord(cap->fork2, st) != cudaSuccess || cudaStreamWaitEvent(cap->side2, cap->fork2, 0) != cudaSuccess)
      return PS_ERR_CUDA;
    ms = cap->side2;
    // (Held back until the candidate scan was done they cost more than they
    // slow it down: prefixshield over 2^20 blocks 149.3 us a step of 4096
    // requests against 148.1, and 71.6 against 68.2 for one of a single one.)
  }
  PS_LAUNCH(launch_k(k_instep, pgrid, kThreads, 0, ms, s));
  if (s.policy == PS_S3FIFO) {
    if (launch_s3_probe(s, ms, &launches) != PS_OK) return PS_ERR_CUDA;
    // the plan trims the ghost: it waits for the lookups
    if (fork2 && cudaEventRecord(cap->fork, ms) != cudaSuccess) return PS_ERR_CUDA;
  }
  mark(4);
  PS_LAUNCH(launch_k(k_meter, s.G, 512, 0, ms, s));
  mark(5);
  PS_LAUNCH(launch_k(k_touch, pgrid, kThreads, 0, ms, s));
  PS_LAUNCH(launch_k(k_touch2, pgrid, kThreads, 0, ms, s));
  if (fork2 && cudaEventRecord(cap->join2, cap->side2) != cudaSuccess) return PS_ERR_CUDA;
  mark(6);
  if (fork && cudaStreamWaitEvent(st, cap->join, 0) != cudaSuccess) return PS_ERR_CUDA;
  if (s.lg_on) {
    // indexed queues: the same victims, taken from the queues' heads
    if (s.policy == PS_PREFIXSHIELD) {
      // the first kernel after the side branch's join depends on two nodes:
      // a plain launch (a programmatic edge takes a single kernel predecessor)
      PS_LAUNCH(k_waterfill<<<1, 1024, 0, st>>>(s));
      if (launch_queue_select(s, st, 0, false, &launches) != PS_OK) return PS_ERR_CUDA;
      // the fallback: its plan finds nothing owed when the debts covered all
      if (launch_queue_select(s, st, 1, false, &launches) != PS_OK) return PS_ERR_CUDA;
    } else if (launch_queue_select(s, st, s.policy == PS_LRU ? 2 : 3, fork, &launches) != PS_OK) {
      return PS_ERR_CUDA;
    }
  }
  // One exact segmented select: a digit over the candidates, the split, then
  // the split list finished by one CTA.  Every phase is launched on every
  // step (a kernel of a phase with nothing to select returns at once): a
  // conditional graph node measured about 10 us a step even when its body
  // was skipped, more than the phase's early-returning launches.
  auto select = [&](int fallback) {
    PS_LAUNCH(launch_k(k_sel_count, cgrid, 256, 0, st, s, fallback));
    PS_LAUNCH(launch_k(k_sel_resolve, fallback || s.policy == PS_LRU ? 1 : s.G, 1024, 0, st, s, fallback));
    PS_LAUNCH(launch_k(k_sel_split, cgrid, 256, 0, st, s, fallback));
    PS_LAUNCH(launch_k(k_list_finish, 1, 1024, kFinSmem, st, s, fallback));
  };
  // stage timing tells the select from the lists, so it runs them apart
  const bool one_cta = small_select(s) && !(tr && tr->timing);
  if (s.lg_on) {
    // selected above
  } else if (one_cta) {
    PS_LAUNCH(k_small_select<<<1, kSmallThreads, kFinSmem, st>>>(s));  // after the join: plain
  } else if (s.policy == PS_PREFIXSHIELD) {
    PS_LAUNCH(k_waterfill<<<1, 1024, 0, st>>>(s));  // after the join: plain
    select(0);
    select(1);  // the global fallback, started by the debt phase's finish
  } else if (s.policy == PS_STATICQUOTA) {
    PS_LAUNCH(k_quota_sel<<<1, 1024, 0, st>>>(s));  // after the join: plain
    select(0);
  } else if (s.policy == PS_LRU) {
    PS_LAUNCH(k_sel_single<<<1, 32, 0, st>>>(s));  // after the join: plain
    select(0);
  } else {
    if (launch_s3_count(s, st, fork2, &launches) != PS_OK) return PS_ERR_CUDA;
    if (fork2 && cudaStreamWaitEvent(st, cap->fork, 0) != cudaSuccess) return PS_ERR_CUDA;
    if (launch_s3_select(s, st, fork2, &launches) != PS_OK) return PS_ERR_CUDA;
  }
  // The ghost pushes run beside the id lists (the candidate scan's branch,
  // which S3-FIFO has no use for), joined before the insertion.
  const bool fork3 = cap != nullptr && s.policy == PS_S3FIFO;
  if (fork3) {
    if (cudaEventRecord(cap->fork, st) != cudaSuccess || cudaStreamWaitEvent(cap->side, cap->fork, 0) != cudaSuccess ||
        launch_s3_push(s, cap->side, true, &launches) != PS_OK || cudaEventRecord(cap->join, cap->side) != cudaSuccess)
      return PS_ERR_CUDA;
  } else if (s.policy == PS_S3FIFO && launch_s3_push(s, st, false, &launches) != PS_OK) {
    return PS_ERR_CUDA;
  }
  mark(7);
  const int nchunks = (int)((s.nwords + kBmChunk - 1) / kBmChunk);
  // a pool of one chunk (8192 blocks) has no earlier chunks to count
  if (nchunks > 1) {
    if (fork3) PS_LAUNCH((k_bm_count<<<nchunks, kBmChunk, 0, st>>>(s)));  // after the fork: plain
    else PS_LAUNCH(launch_k(k_bm_count, nchunks, kBmChunk, 0, st, s));
  }
  if (one_cta) {
    // listed already
  } else if (fork3 && nchunks == 1) PS_LAUNCH((k_bm_write<<<nchunks, kBmThreads, 0, st>>>(s)));
  else PS_LAUNCH(launch_k(k_bm_write, nchunks, kBmThreads, 0, st, s));
  mark(8);
  // (evictions happen in k_insert: every victim is allocated again in its step)
  mark(9);
  if (fork3 && cudaStreamWaitEvent(st, cap->join, 0) != cudaSuccess) return PS_ERR_CUDA;
  if (fork2) {  // the touch branch joins the insertion
    if (cudaStreamWaitEvent(st, cap->join2, 0) != cudaSuccess) return PS_ERR_CUDA;
    PS_LAUNCH((k_insert<<<igrid, kThreads, 0, st>>>(s)));  // after the join: plain
  } else {
    PS_LAUNCH(launch_k(k_insert, igrid, kThreads, 0, st, s));
  }
  if (s.policy == PS_S3FIFO && launch_s3_insert(s, st, &launches) != PS_OK) return PS_ERR_CUDA;
  if (s.lg_on && launch_queue_append(s, st, &launches) != PS_OK) return PS_ERR_CUDA;
  mark(10);
  PS_LAUNCH(launch_k(k_finalize, 1, 32, 0, st, s));
  mark(11);
#undef PS_LAUNCH
  if (tr) tr->launches = launches;
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

// The step's outputs into the caller's page-locked host buffers (one pass,
// grid-stride; the id lists by the counts the step wrote).
__global__ void __launch_bounds__(256) k_host_out(ps_step_out_t d, ps_step_out_t h, int32_t R, int32_t G) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  const bool ok = d.counts[3] == PS_OK;
  const int64_t n0 = ok ? d.counts[0] : 0, n1 = ok ? d.counts[1] : 0, n2 = ok ? d.counts[2] : 0;
  if (h.counts && t < 4) h.counts[t] = d.counts[t];
  for (int64_t i = t; i < R; i += nt) {
    if (h.hit_blocks) h.hit_blocks[i] = d.hit_blocks[i];
    if (h.admitted_blocks) h.admitted_blocks[i] = d.admitted_blocks[i];
  }
  if (h.admitted_offsets)
    for (int64_t i = t; i <= R; i += nt) h.admitted_offsets[i] = d.admitted_offsets[i];
  for (int64_t i = t; i < G; i += nt) {
    if (h.debt_raw) h.debt_raw[i] = d.debt_raw[i];
    if (h.debt_norm) h.debt_norm[i] = d.debt_norm[i];
  }
  if (h.admitted_ids)
    for (int64_t i = t; i < n0; i += nt) h.admitted_ids[i] = d.admitted_ids[i];
  if (h.evicted_ids)
    for (int64_t i = t; i < n1; i += nt) h.evicted_ids[i] = d.evicted_ids[i];
  if (h.invalidated_ids)
    for (int64_t i = t; i < n2; i += nt) h.invalidated_ids[i] = d.invalidated_ids[i];
}

void launch_host_out(const ps_step_out_t& dev, const ps_step_out_t& host, int32_t R, int32_t G, cudaStream_t st) {
  k_host_out<<<152 * 2, 256, 0, st>>>(dev, host, R, G);
}

// A step's inputs from the caller's page-locked host buffers into the staging
// area, one pass of all SMs over the host link: a small call's five copies
// took longer to issue, one after the other, than to run.
struct HostIn {
  const void* src[5];
  void* dst[5];
  int64_t words[5];  // 32-bit words
};
__global__ void __launch_bounds__(256) k_host_in(HostIn a) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int64_t n = a.words[k];
    const uint32_t* src = static_cast<const uint32_t*>(a.src[k]);
    uint32_t* dst = static_cast<uint32_t*>(a.dst[k]);
    const int64_t nv = (reinterpret_cast<uintptr_t>(src) & 15) ? 0 : n / 4;  // the staging areas are aligned
    for (int64_t i = t; i < nv; i += nt) reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(src)[i];
    for (int64_t i = 4 * nv + t; i < n; i += nt) dst[i] = src[i];
  }
}
void launch_host_in(const void* const* src, void* const* dst, const int64_t* words, cudaStream_t st) {
  HostIn a{};
  for (int k = 0; k < 5; ++k) {
    a.src[k] = src[k];
    a.dst[k] = dst[k];
    a.words[k] = src[k] ? words[k] : 0;
  }
  k_host_in<<<152 * 4, 256, 0, st>>>(a);
}

int32_t launch_probe(const DevState& s, cudaStream_t st, int32_t* out, int32_t* status) {
  DevState p = s;
  p.args = nullptr;  // the probe's kernels take every argument by value
  k_validate<<<grid_for(p.max_requests, kValTile, 1 << 20), kValTile, 0, st>>>(p, status);
  if (s.R > 0 && launch_hash_lookup(p, st, out) != PS_OK) return PS_ERR_INVALID_ARG;
  return cudaGetLastError() == cudaSuccess ? PS_OK : PS_ERR_CUDA;
}

}  // namespace ps
