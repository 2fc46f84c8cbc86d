// pctree_tree_attention: one grouped-query attention layer of the target's
// tree-verification forward (Sec. 4.2; Appendix A "Tensor implementation"):
// every drafted node attends to the verified prefix, itself and its
// root-to-node ancestors.
//
// Work items: request r, KV head h, a query tile and a range of keys.  A
// tile's rows are (node, query head of the group) pairs, node-major: row t =
// node_local * G + g, R = G * nodes_per_tile <= 128; the G query heads sharing
// KV head h read each K/V block once.  The kernel is persistent: one CTA per
// SM takes items in rounds of gridDim.x, forwards and backwards in turn, over
// a list ordered by decreasing request length (longest first keeps the last
// round short), so its set-up (barriers, TMEM) is paid once and every
// pipeline runs on across items.
//
//   warp 0      TMA producer: each item's Q tile (two buffers), then its K and
//               V blocks (128 keys x 128 dims, two 64-dim halves each,
//               128-byte swizzle), K and V in turn, into a ring of 32 KB slots
//   warp 1      S issuer: S_b = Q K_b^T (tcgen05.mma, M=128, N=128 keys, K=128
//               dims) into one of two TMEM buffers
//   warp 2      PV issuer: O_h += P_b V_b over each half h of the block's keys
//               (M=128, N=128 dims, K=64 keys; P read from TMEM, V the MN-major
//               shared-memory operand)
//   warp 3      planner: the facts of the CTA's next items, and their
//               ancestor-or-self masks from the packed parents
//   warps 4..7  output: the two O of a finished item, combined and normalised,
//               to bf16 rows (or the split's partial), while the softmax goes on
//   warps 8..15 softmax, two threads per TMEM lane = tile row, 64 keys of a
//               block each with its own running maximum, sum and O (so the two
//               warps of a sub-partition never wait for one another and one's
//               exponentials overlap the other's loads): the S row is read
//               from TMEM once, masked and scaled; P = 2^(s - m_used) rounded to
//               bf16 pairs is written back over the S columns it came from
//               (the TMEM A operand of the PV product)
//
// What bounds it, and why this split: per block of keys each role pays fixed
// costs (a wait on a barrier that is already complete ~250 cycles, a commit
// ~130), and straight-line code runs at 2 - 4 cycles an instruction (it does
// not stay in the innermost instruction cache), so the softmax of a block, not
// its MMAs, set the pace: 1500 cycles per 64 keys and tile with one thread
// per row.  128 keys per block halve the fixed costs and let the S products
// run at full rate (at N = 64 they take 54 cycles an MMA instead of 64 for
// twice the keys); two threads per row halve the softmax chain; output and
// planning took 4 - 9 thousand cycles of the softmax warps' time per item and
// have warps of their own.
// Measured against one thread per row, 64-key blocks and two tiles per CTA (us
// per layer, alternating graph replays): 14B-shaped (batch 32, 40 / 8 heads,
// 128-node trees, prefixes to 1024) 97.9 -> 64.9; 8B-shaped (batch 16, 64 nodes)
// 25.9 -> 19.7; 4B-shaped (batch 1, prefix 2048, split keys) 16.9 -> 15.5.  Two tiles
// per CTA with 128-key blocks, one S buffer each and setmaxnreg ran 125 us on
// the 14B shape: with a single S buffer softmax and MMAs of a tile alternate.
// Key ranges of a request may be split over several items (few requests,
// long prefixes); each then writes (max, sum, unnormalised O) of its rows and
// a second kernel merges the splits, spread over all SMs.  All waits are
// bounded (1 s) and end in PCTREE_ERR_TIMEOUT.
#include <cuda_bf16.h>

#include "pctree_common.cuh"
#include "sm103_ptx.cuh"

namespace pct {
namespace {

constexpr int kBK = 128;                  // keys per block
// The unit of the key split over items: whole blocks, since an item of 64 keys
// takes a block's time (us per layer, units of 64 / 128: 25 requests of 6 nodes
// with prefixes to 246 14.1 / 9.5, 7 of 5 nodes to 115 10.3 / 6.8, one of 64
// nodes to 8000 26.0 / 20.6).
constexpr int kSplitKeys = kBK;
constexpr int kHalfBytes = 128 * 128;     // 128 rows x 64 bf16 (one dim half)
constexpr int kTileBytes = 2 * kHalfBytes;   // a Q tile, or a K or V block
constexpr int kMaskWords = PCTREE_ATTN_MAX_N / 32;
constexpr uint64_t kAttnLimitNs = 1000000000ull;

constexpr int kMaxOrder = 256;            // requests ordered by length in shared memory
constexpr int kItemRing = 4;              // items planned ahead

// One CTA: two Q buffers and a ring of K and V blocks in shared memory; in
// TMEM two S buffers (128 fp32 columns each; the P of a 64-key half, packed
// bf16 pairs, overwrites the first 32 columns of its half) and an O of 128
// columns for each half.
constexpr int kAttnThreads = 512;         // roles above
constexpr int kSlots = 4;                 // K or V blocks in the ring
constexpr int kKVOff = 2 * kTileBytes;
constexpr int kTailOff = kKVOff + kSlots * kTileBytes;
constexpr uint32_t kOCol = 2 * kBK;
constexpr uint32_t kTmemCols = 512;

// One work item: request r, KV head kvh, query tile qt and the keys key0 ..
// key1-1 of the request's Tp + n, in nblk blocks.  A tile that holds no node
// of the request's tree (a tree may use less than the budget N, and tile
// counts round up) has none: its rows are written as 0 without any product.
// (Computing every tile cost the 14B-shaped layer, whose trees fill 3 to 6 of
// 6 tiles, a fifth of its time.)
struct AttnItem {
  int r, kvh, qt, split, Tp, n, key0, key1, nblk;
};

// Barriers count blocks over the CTA's whole item sequence: K or V block x in
// ring slot x % kSlots (K of the g-th block x = 2 g, its V x = 2 g + 1), S/P
// buffer g & 1 of the g-th block, ancestor buffer k & 1 and item slot k %
// kItemRing of the k-th item.
struct AttnTail {
  uint64_t q_full[2], q_empty[2];
  uint64_t kv_full[kSlots], kv_empty[kSlots];
  uint64_t s_full[2];                      // S written
  uint64_t p_full[2];                      // P written over it
  uint64_t p_empty[2];                     // PV product done: buffer free
  uint64_t o_full, o_empty;                // an item's O and row sums / read
  uint64_t anc_full[2], anc_empty[2];
  uint64_t item_full[kItemRing], item_empty[kItemRing];
  uint64_t done;
  uint32_t tmem_base;
  int abort;
  AttnItem item[kItemRing];
  float row_l[2][128], row_m[2][128];      // row sums and references of each half
  alignas(16) uint8_t stage[4][32 * 64];   // output staging, per output warp
  alignas(16) uint32_t anc[2][PCTREE_ATTN_MAX_N][kMaskWords];   // ancestor-or-self bits
  int16_t par[PCTREE_ATTN_MAX_N];          // next ancestor not yet in a node's bits
  int32_t pre[kMaxOrder], nn[kMaxOrder];   // validated prefix / node counts
  int16_t lt[kMaxOrder];                   // tiles that hold nodes
  int16_t order[kMaxOrder];                // requests by decreasing key count
  int32_t first[kMaxOrder + 1];            // items with nodes before the i-th of them
};

constexpr size_t kAttnSmem = kTailOff + sizeof(AttnTail) + 1024;
static_assert(kAttnSmem <= 227 * 1024, "shared memory per CTA");

struct AttnArgs {
  const int32_t* prefix;
  const int32_t* n_nodes;
  const int32_t* parent;
  uint16_t* out;          // bf16 [batch][N][Hq][128]
  float* part_o;          // [unit][split][32][128][4]: dims / 4, tile rows, 4 dims
  float2* part_ml;        // [unit][split][128]  (max in log2 units, sum)
  int32_t* status;
  int batch, N, Hq, Hkv, G, npt, R, nqt, max_slots, n_split, bps;
  int items;              // batch * Hkv * nqt * n_split
  float scale_log2;       // softmax scale * log2(e)
};

// A request with an impossible prefix or tree size attends to nothing (its
// rows are written as 0 and the launch reports PCTREE_ERR_INVALID_ARG).
__device__ __forceinline__ bool request_ok(const AttnArgs& a, int Tp, int n) {
  return Tp >= 0 && n >= 0 && n <= a.N && static_cast<long long>(Tp) + n <= a.max_slots;
}

// Tiles of a request of n nodes that hold any of them.
__device__ __forceinline__ int live_tiles(const AttnArgs& a, int n) {
  return (n + a.npt - 1) / a.npt;
}

// Item `idx` of the item list.  Not `ranked`: the items of request idx /
// per_req as (split, KV head, tile) triples.  `ranked` (the validated request
// sizes are in shared memory): requests in the longest-first order, first
// the items whose tiles hold nodes (so the CTAs' rounds are dealt from items
// that do work), then the rest.
__device__ __forceinline__ AttnItem item_facts(const AttnArgs& a, const AttnTail* T, int idx,
                                               bool ranked) {
  AttnItem it;
  const int per_req = a.Hkv * a.nqt * a.n_split;
  int tiles = a.nqt, tile0 = 0, rest;
  if (ranked) {
    const int live = T->first[a.batch];
    const bool dead = idx >= live;
    const int x = dead ? idx - live : idx;
    // the request i with begin(i) <= x < begin(i + 1), begin(i) its first
    // item in the list of items with (or without) nodes
    int lo = 0, hi = a.batch;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      const int begin = dead ? mid * per_req - T->first[mid] : T->first[mid];
      if (begin <= x) lo = mid; else hi = mid;
    }
    it.r = T->order[lo];
    rest = x - (dead ? lo * per_req - T->first[lo] : T->first[lo]);
    const int lt = T->lt[it.r];
    tiles = dead ? a.nqt - lt : lt;
    tile0 = dead ? lt : 0;
    it.Tp = T->pre[it.r];
    it.n = T->nn[it.r];
  } else {
    it.r = idx / per_req;
    rest = idx - it.r * per_req;
    it.Tp = a.prefix[it.r];
    it.n = a.n_nodes[it.r];
    if (!request_ok(a, it.Tp, it.n)) it.Tp = it.n = 0;
  }
  const int head = rest / tiles;               // split * Hkv + KV head
  it.split = head / a.Hkv;
  it.kvh = head - it.split * a.Hkv;
  it.qt = tile0 + rest - head * tiles;
  it.key0 = it.split * a.bps * kSplitKeys;
  it.key1 = it.qt * a.npt < it.n ? min(it.key0 + a.bps * kSplitKeys, it.Tp + it.n) : 0;
  it.nblk = max(0, (it.key1 - it.key0 + kBK - 1) / kBK);
  return it;
}

// Position in the longest-first list of this CTA's k-th item: rounds of
// gridDim.x items, taken forwards and backwards in turn, so every CTA gets a
// mix of long and short items.
__device__ __forceinline__ long long item_pos(int k) {
  const long long base = static_cast<long long>(k) * gridDim.x;
  return (k & 1) ? base + gridDim.x - 1 - blockIdx.x : base + blockIdx.x;
}

// 32 lanes x 8 columns of 32-bit TMEM words from registers: thread t of the
// warp writes lane (taddr.lane + t), columns taddr.col .. +7.
__device__ __forceinline__ void tmem_st_32x32b_x8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// 32 lanes x 16 columns of 32-bit TMEM words from registers (see
// tmem_st_32x32b_x8).
__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15])
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]: the A operand (M = 128 rows on the TMEM
// lanes, 16 K elements as 8 columns of bf16 pairs, the lower half holding the
// even element) is read from tensor memory.  Issued by one thread.
__device__ __forceinline__ void tc_mma_bf16_tmem_a(uint32_t d_tmem, uint32_t a_tmem,
                                                   uint64_t b_desc, uint32_t idesc,
                                                   uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Records the first error in the optional status word.
__device__ __forceinline__ void report(int32_t* status, int code) {
  if (status != nullptr) atomicCAS(status, 0, code);
}

// Allowed-key bits of 32 consecutive slots kc0 .. kc0+31 for a row whose
// node has ancestor-or-self bits `anc`: the whole prefix (slots < T) and
// the tree slots T + m of its ancestors (the bits are 0 past the tree).
__device__ __forceinline__ uint32_t allowed_bits(int kc0, int T,
                                                 const uint32_t* anc) {
  uint32_t bits = 0;
  const int pm = T - kc0;                       // prefix slots in the chunk
  if (pm >= 32) return 0xffffffffu;
  if (pm > 0) bits = (1u << pm) - 1u;
  const int m0 = kc0 - T;                       // tree index of slot kc0
  if (m0 >= 0) {
    const int w = m0 >> 5, sh = m0 & 31;
    uint32_t lo = w < kMaskWords ? anc[w] : 0u;
    uint32_t hi = (w + 1) < kMaskWords ? anc[w + 1] : 0u;
    bits |= sh == 0 ? lo : ((lo >> sh) | (hi << (32 - sh)));
  } else if (m0 > -32) {
    bits |= anc[0] << (-m0);
  }
  return bits;
}

// 112 registers a thread (of the 128 that 512 threads could have): the rest of
// the register file lets the merge kernel's CTAs start while this kernel
// finishes (with 128 the 4B-shaped layer took 3 us more).
__global__ void __maxnreg__(112)
tree_attn_kernel(const __grid_constant__ CUtensorMap tm_q,
                 const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, AttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  AttnTail* T = reinterpret_cast<AttnTail*>(sm + kTailOff);
  uint8_t* sq = sm;                            // Q buffer k & 1 of the k-th item
  uint8_t* skv = sm + kKVOff;                // ring slot s at skv + s * kTileBytes
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long n_items = a.items;
  // the longest-first order only matters when CTAs take several items; the
  // request sizes are then staged in shared memory too
  const bool ranked = a.batch <= kMaxOrder && n_items > static_cast<long long>(gridDim.x);
  volatile int* abort_v = &T->abort;

  // ---------------- set-up (once per CTA) ----------------
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&T->kv_full[s], 1);
      mbar_init(&T->kv_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&T->q_full[s], 1);
      mbar_init(&T->q_empty[s], 1);
      mbar_init(&T->s_full[s], 1);
      mbar_init(&T->p_full[s], 8);         // every softmax warp
      mbar_init(&T->p_empty[s], 1);
      mbar_init(&T->anc_full[s], 1);
      mbar_init(&T->anc_empty[s], 8);
    }
    for (int s = 0; s < kItemRing; ++s) {
      mbar_init(&T->item_full[s], 1);
      mbar_init(&T->item_empty[s], 3 + 4 + 8);   // every role's copy
    }
    mbar_init(&T->o_full, 1 + 8);          // the PV issuer, the softmax warps
    mbar_init(&T->o_empty, 4);             // the output warps
    mbar_init(&T->done, 2);              // one commit from each MMA issuer
    T->abort = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    tma_prefetch_desc(&tm_v);
  }
  // rows R..127 of the Q buffers are never loaded: zero them once (read by
  // the MMA)
  const int zq = (128 - a.R) * 8;                  // 16-byte chunks per half
  for (int i = threadIdx.x; i < 2 * 2 * zq; i += blockDim.x) {
    const int j = i / (2 * zq), half = (i / zq) & 1, rem = i % zq;
    *reinterpret_cast<uint4*>(sq + j * kTileBytes + half * kHalfBytes + (a.R + rem / 8) * 128 +
                              (rem % 8) * 16) = make_uint4(0, 0, 0, 0);
  }
  fence_proxy_async_smem();
  if (warp == 1) tmem_alloc(&T->tmem_base, kTmemCols);
  // programmatic dependent launch: the launch and the set-up above overlap
  // the previous kernel of the stream; every global access (request sizes,
  // Q, K, V, the output) comes after it is complete
  pdl_launch_dependents();
  pdl_wait();
  // requests: validated sizes (reported once) and, when ranked, staged and
  // ordered by key count
  if (ranked || blockIdx.x == 0) {
    for (int u = threadIdx.x; u < a.batch; u += blockDim.x) {
      int Tp = a.prefix[u], n = a.n_nodes[u];
      if (!request_ok(a, Tp, n)) {
        if (blockIdx.x == 0) report(a.status, PCTREE_ERR_INVALID_ARG);
        Tp = n = 0;
      }
      if (ranked) {
        T->pre[u] = Tp;
        T->nn[u] = n;
        T->lt[u] = static_cast<int16_t>(live_tiles(a, n));
      }
    }
  }
  if (ranked) {
    __syncthreads();
    for (int u = threadIdx.x; u < a.batch; u += blockDim.x) {
      const int ku = T->nn[u] > 0 ? T->pre[u] + T->nn[u] : 0;
      int rank = 0, before = 0;
      for (int v = 0; v < a.batch; ++v) {
        const int kv = T->nn[v] > 0 ? T->pre[v] + T->nn[v] : 0;
        const bool ahead = kv > ku || (kv == ku && v < u);
        rank += ahead ? 1 : 0;
        before += ahead ? T->lt[v] : 0;
      }
      const int per_tile = a.Hkv * a.n_split;
      T->order[rank] = static_cast<int16_t>(u);
      T->first[rank] = before * per_tile;
      if (rank == a.batch - 1) T->first[a.batch] = (before + T->lt[u]) * per_tile;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = T->tmem_base;

  // a warp whose lanes all saw the phase complete continues together, so the
  // warp-collective tcgen05 operations that follow never diverge
  auto wwait = [&](uint64_t* bar, uint32_t parity) -> bool {
    return __all_sync(kFull, mbar_wait_bounded(bar, parity, abort_v, kAttnLimitNs));
  };
  auto give_up = [&]() {
    *abort_v = 1;
    report(a.status, PCTREE_ERR_TIMEOUT);
  };
  // the k-th item's facts, copied so that its slot can be planned again
  auto fetch_one = [&](int k, AttnItem& it) -> bool {          // one thread
    const int s = k % kItemRing;
    if (!mbar_wait_bounded(&T->item_full[s], (k / kItemRing) & 1, abort_v, kAttnLimitNs))
      return false;
    it = T->item[s];
    mbar_arrive(&T->item_empty[s]);
    return true;
  };
  auto fetch_warp = [&](int k, AttnItem& it) -> bool {         // a whole warp
    const int s = k % kItemRing;
    if (!wwait(&T->item_full[s], (k / kItemRing) & 1)) return false;
    it = T->item[s];
    __syncwarp();
    if (lane == 0) mbar_arrive(&T->item_empty[s]);
    return true;
  };

  if (warp < 4) {
    if (warp == 0 && lane == 0) {
      // ---------------- TMA producer: Q tiles, K and V blocks ----------------
      int slot = 0, issued = 0, q = 0;           // ring slot, blocks, Q tiles
      uint32_t phase = 0;
      bool ok = true;
      AttnItem it;
      for (int k = 0; ok && item_pos(k) < n_items; ++k) {
        if (!(ok = fetch_one(k, it))) break;
        if (it.nblk == 0) continue;
        // Q buffer q & 1 is free once the S products of two items ago are done
        const int qb = q & 1;
        if (!(ok = mbar_wait_bounded(&T->q_empty[qb], ((q >> 1) & 1) ^ 1, abort_v, kAttnLimitNs)))
          break;
        mbar_arrive_expect_tx(&T->q_full[qb], 2u * static_cast<uint32_t>(a.R) * 128u);
        tma_load_4d(sq + qb * kTileBytes, &tm_q, &T->q_full[qb], 0, it.kvh * a.G, it.qt * a.npt,
                    it.r);
        tma_load_4d(sq + qb * kTileBytes + kHalfBytes, &tm_q, &T->q_full[qb], 64, it.kvh * a.G,
                    it.qt * a.npt, it.r);
        ++q;
        for (int b = 0; ok && b < it.nblk; ++b) {
          const int key = it.key0 + b * kBK;
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            if (!(ok = mbar_wait_bounded(&T->kv_empty[slot], phase ^ 1u, abort_v, kAttnLimitNs)))
              break;
            uint8_t* dst = skv + slot * kTileBytes;
            const CUtensorMap* map = v == 0 ? &tm_k : &tm_v;
            mbar_arrive_expect_tx(&T->kv_full[slot], static_cast<uint32_t>(kTileBytes));
            tma_load_4d(dst, map, &T->kv_full[slot], 0, it.kvh, key, it.r);
            tma_load_4d(dst + kHalfBytes, map, &T->kv_full[slot], 64, it.kvh, key, it.r);
            ++issued;
            if (++slot == kSlots) {
              slot = 0;
              phase ^= 1u;
            }
          }
        }
      }
      if (!ok) give_up();
      // copies still in flight land before the CTA may exit
      volatile int never = 0;
      for (int x = issued > kSlots ? issued - kSlots : 0; x < issued; ++x)
        (void)mbar_wait_bounded(&T->kv_full[x % kSlots], (x / kSlots) & 1, &never, kAttnLimitNs);
      for (int x = q > 2 ? q - 2 : 0; x < q; ++x)
        (void)mbar_wait_bounded(&T->q_full[x & 1], (x >> 1) & 1, &never, kAttnLimitNs);
    } else if (warp == 1 && lane == 0) {
      // ---------------- S issuer ----------------
      // Every wait and MMA of the two issuers is on the layer's critical
      // path: their loops keep counters and descriptors in registers.
      constexpr uint32_t idS = idesc_bf16_f32(128, kBK);
      int slot = 0, q = 0, g = 0;                  // K's ring slot, Q tiles, blocks
      uint32_t phase = 0;
      const uint64_t q_desc = desc_kmajor_sw128(smem_u32(sq));
      const uint64_t k_desc = desc_kmajor_sw128(smem_u32(skv));
      bool ok = true;
      AttnItem it;
      for (int k = 0; ok && item_pos(k) < n_items; ++k) {
        if (!(ok = fetch_one(k, it))) break;
        if (it.nblk == 0) continue;
        const int qb = q & 1;
        if (!(ok = mbar_wait_bounded(&T->q_full[qb], (q >> 1) & 1, abort_v, kAttnLimitNs))) break;
        ++q;
        const uint64_t qd = q_desc + qb * (kTileBytes >> 4);
        for (int b = 0; b < it.nblk; ++b, ++g) {
          const int sb = g & 1;
          // S buffer sb holds the P of two blocks ago until its PV product
          // is done
          ok = mbar_wait_bounded(&T->kv_full[slot], phase, abort_v, kAttnLimitNs) &&
               mbar_wait_bounded(&T->p_empty[sb], ((g >> 1) & 1) ^ 1, abort_v, kAttnLimitNs);
          if (!ok) break;
          const uint64_t kd = k_desc + slot * (kTileBytes >> 4);
          tc_fence_after_sync();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) {      // 128 dims in steps of 16
            const int off = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
            tc_mma_bf16(tmem + sb * kBK, qd + off, kd + off, idS, kk > 0 ? 1u : 0u);
          }
          tc_commit(&T->s_full[sb]);
          tc_commit(&T->kv_empty[slot]);
          slot += 2;
          if (slot >= kSlots) {
            slot -= kSlots;
            phase ^= 1u;
          }
        }
        tc_commit(&T->q_empty[qb]);      // arrives once the item's S products are done
      }
      if (!ok) give_up();
      tc_commit(&T->done);               // every MMA this thread issued has finished
      volatile int never = 0;
      (void)mbar_wait_bounded(&T->done, 0, &never, kAttnLimitNs);
    } else if (warp == 2 && lane == 0) {
      // ---------------- PV issuer ----------------
      constexpr uint32_t idO = idesc_bf16_f32_bmn(128, 128);
      int slot = 1, g = 0;                         // V's ring slot, blocks
      uint32_t phase = 0;
      const uint64_t v_desc = desc_mnmajor_sw128(smem_u32(skv), kHalfBytes, 1024);
      bool ok = true;
      AttnItem it;
      for (int k = 0; ok && item_pos(k) < n_items; ++k) {
        if (!(ok = fetch_one(k, it))) break;
        // O (and the row sums) of the previous item have been read
        auto wait_o = [&]() {
          return mbar_wait_bounded(&T->o_empty, (k & 1) ^ 1, abort_v, kAttnLimitNs);
        };
        if (it.nblk == 0) {                              // no product to wait for
          if (!(ok = wait_o())) break;
          mbar_arrive(&T->o_full);
        }
        for (int b = 0; b < it.nblk; ++b, ++g) {
          const int sb = g & 1;
          // V has landed; P_b, and with it S_b, is complete; with short items
          // O is free last
          ok = mbar_wait_bounded(&T->kv_full[slot], phase, abort_v, kAttnLimitNs) &&
               mbar_wait_bounded(&T->p_full[sb], (g >> 1) & 1, abort_v, kAttnLimitNs) &&
               (b > 0 || wait_o());
          if (!ok) break;
          const uint64_t vd = v_desc + slot * (kTileBytes >> 4);
          tc_fence_after_sync();
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            // A: 16 keys of P = 8 TMEM columns; B: 16 keys = 16 rows of 128 B
            // of V, the dims 64..127 half kHalfBytes further on
            const int h = kk >> 2;
            tc_mma_bf16_tmem_a(tmem + kOCol + h * 128, tmem + sb * kBK + h * 64 + (kk & 3) * 8,
                               vd + ((kk * 16 * 128) >> 4), idO,
                               (b > 0 || (kk & 3) > 0) ? 1u : 0u);   // O accumulates over the item
          }
          tc_commit(&T->p_empty[sb]);
          if (b + 1 == it.nblk) tc_commit(&T->o_full);
          tc_commit(&T->kv_empty[slot]);
          slot += 2;
          if (slot >= kSlots) {
            slot -= kSlots;
            phase ^= 1u;
          }
        }
      }
      if (!ok) give_up();
      tc_commit(&T->done);
      volatile int never = 0;
      (void)mbar_wait_bounded(&T->done, 0, &never, kAttnLimitNs);
    } else if (warp == 3) {
      // ---------------- planner: item facts two ahead, ancestor masks ----------------
      // (A lane works out one of the CTA's next 32 items: one by one the divisions
      // and the search of item_facts took ~2 thousand cycles an item, which set
      // the pace of short ones.  With the packed products of the output warps
      // and the PV issuer's wait for O last, us per layer: 32 requests of up to 64
      // nodes with prefixes to 64 19.5 -> 17.8, the 14B shape 65.6 -> 64.9.)
      AttnItem mine = {};
      auto plan = [&](int k) -> bool {
        if (item_pos(k) >= n_items) return true;
        if ((k & 31) == 0)
          mine = item_facts(a, T, static_cast<int>(min(item_pos(k + lane), n_items - 1)), ranked);
        const int s = k % kItemRing;
        if (!wwait(&T->item_empty[s], ((k / kItemRing) & 1) ^ 1)) return false;
        if (lane == (k & 31)) {
          T->item[s] = mine;
          mbar_arrive(&T->item_full[s]);
        }
        __syncwarp();
        return true;
      };
      // Ancestor-or-self bits of a request's nodes, by pointer jumping:
      // bits[x] holds the nodes from x up to, not including, par[x]; a node
      // takes over its par's bits and par until none is left (about
      // log2(depth) rounds; 32 nodes read, then write, together, so the pair
      // is always consistent).  Walking up from each node took 3 - 7 thousand
      // cycles an item (one dependent load per level and node), more than a
      // short item's products.
      auto ancestor_bits = [&](int r, int n, int ab) {
        uint32_t(*bits)[kMaskWords] = T->anc[ab];
        for (int i = lane; i < n; i += 32) {
          const int p = a.parent[static_cast<size_t>(r) * a.N + i];
          T->par[i] = static_cast<int16_t>(p >= 0 && p < i ? p : -1);   // parents precede children
#pragma unroll
          for (int w = 0; w < kMaskWords; ++w) bits[i][w] = w == (i >> 5) ? 1u << (i & 31) : 0u;
        }
        __syncwarp();
        for (int round = 0; round < 9; ++round) {   // 2^8 levels at most
          bool more = false;
          for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const int p = i < n ? T->par[i] : -1;
            uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
            int pp = -1;
            if (p >= 0) {
              pp = T->par[p];
              lo = *reinterpret_cast<const uint4*>(&bits[p][0]);
              if (n > 128) hi = *reinterpret_cast<const uint4*>(&bits[p][4]);
            }
            __syncwarp();
            if (p >= 0) {
              uint4* w = reinterpret_cast<uint4*>(&bits[i][0]);
              const uint4 l0 = w[0];
              w[0] = make_uint4(l0.x | lo.x, l0.y | lo.y, l0.z | lo.z, l0.w | lo.w);
              if (n > 128) {
                const uint4 h0 = w[1];
                w[1] = make_uint4(h0.x | hi.x, h0.y | hi.y, h0.z | hi.z, h0.w | hi.w);
              }
              T->par[i] = static_cast<int16_t>(pp);
              more |= pp >= 0;
            }
            __syncwarp();
          }
          if (!__any_sync(kFull, more)) break;
        }
        __syncwarp();                      // all lanes done with par and the masks
      };
      bool ok = plan(0) && plan(1);
      for (int k = 0; ok && item_pos(k) < n_items; ++k) {
        const int ab = k & 1;
        const int r = T->item[k % kItemRing].r;
        // a range of prefix keys alone needs no masks
        const int n = T->item[k % kItemRing].key1 > T->item[k % kItemRing].Tp
                          ? T->item[k % kItemRing].n : 0;
        // buffer ab was last read by the softmax warps for item k - 2
        if (!(ok = wwait(&T->anc_empty[ab], ((k >> 1) & 1) ^ 1))) break;
        ancestor_bits(r, n, ab);
        if (lane == 0) mbar_arrive(&T->anc_full[ab]);
        ok = plan(k + 2);
      }
      if (!ok && lane == 0) give_up();
    }
  } else if (warp < 8) {
    // ---------------- output, one thread per tile row ----------------
    // Kept short and rolled: straight-line code that runs once an item comes
    // from the instruction cache at ~4 cycles an instruction.
    const int quad = warp & 3;               // TMEM lanes quad*32 .. +31
    const int t = quad * 32 + lane;          // tile row
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    uint8_t* stg = T->stage[quad];           // 32 rows x 64 bytes
    // the rows this lane stores: 8 i + lane / 4 of the warp's 32, piece
    // lane % 4 of a 64-byte segment; their tile-local nodes (a value no item
    // reaches past the tile's rows) and offsets from the item's first node
    // and head
    int out_nl[4], out_off[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ti = quad * 32 + 8 * i + (lane >> 2), ni = ti / a.G;
      out_nl[i] = ti < a.R ? ni : 0x7fffffff;
      out_off[i] = (ni * a.Hq + ti - ni * a.G) * 128 + (lane & 3) * 8;
    }
    bool ok = true;
    for (int k = 0; ok && item_pos(k) < n_items; ++k) {
      AttnItem it;
      if (!(ok = fetch_warp(k, it))) break;
      if (!(ok = wwait(&T->o_full, k & 1))) break;
      tc_fence_after_sync();
      const int node0 = it.qt * a.npt;
      uint16_t* oitem =
          a.out + ((static_cast<size_t>(it.r) * a.N + node0) * a.Hq + it.kvh * a.G) * 128;
      const size_t part = static_cast<size_t>((it.r * a.Hkv + it.kvh) * a.nqt + it.qt) * a.n_split +
                          it.split;
      if (it.nblk == 0) {
        // no keys or no nodes: nothing to read, zeros for the tile's rows (through
        // the code below each such item took 3 thousand cycles; us per layer: the
        // 14B shape 68.4 -> 65.5, 27 requests of up to 36 nodes with prefixes to
        // 52 14.2 -> 13.2)
        if (lane == 0) mbar_arrive(&T->o_empty);
        if (a.n_split > 1) {
          a.part_ml[part * 128 + t] = make_float2(-INFINITY, 0.0f);
        } else {
#pragma unroll 1
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (out_nl[i] < a.N - node0)
                *reinterpret_cast<uint4*>(oitem + out_off[i] + c * 32) = make_uint4(0, 0, 0, 0);
        }
        continue;
      }
      // the halves' sums and O relative to the larger of their references (a
      // sum is 0 where a half or a row sees no key; one that a non-finite
      // score made NaN counts, and makes the row NaN)
      const float l0 = T->row_l[0][t], l1 = T->row_l[1][t];
      const float m0 = l0 != 0.0f ? T->row_m[0][t] : -INFINITY;
      const float m1 = l1 != 0.0f ? T->row_m[1][t] : -INFINITY;
      const float m = fmaxf(m0, m1);
      float f0 = l0 != 0.0f ? exp2f(m0 - m) : 0.0f;
      float f1 = l1 != 0.0f ? exp2f(m1 - m) : 0.0f;
      const float l = l0 * f0 + l1 * f1;
      const uint32_t o_col = lane_base + kOCol;
      if (a.n_split == 1 && l != 0.0f) {
        const float inv = 1.0f / l;
        f0 *= inv;
        f1 *= inv;
      }
      const uint32_t keep = l != 0.0f ? 0xffffffffu : 0u;   // else O may hold anything
      if (a.n_split > 1) a.part_ml[part * 128 + t] = make_float2(l != 0.0f ? m : -INFINITY, l);
      // tcgen05.ld is warp-collective, so every lane loads and only valid
      // rows store
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {          // 32 dims at a time
        float y[32];
        {
          uint32_t y0[32], y1[32];
          tmem_ld_32x32b_x32(o_col + c * 32, y0);
          tmem_ld_32x32b_x32(o_col + 128 + c * 32, y1);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const uint64_t a0 = pack2(__uint_as_float(y0[i]), __uint_as_float(y0[i + 1]));
            const uint64_t a1 = pack2(__uint_as_float(y1[i]), __uint_as_float(y1[i + 1]));
            unpack2(fma2(a0, pack2(f0, f0), mul2(a1, pack2(f1, f1))), y[i], y[i + 1]);
          }
        }
        if (c == 3) {                        // O and the row sums are read
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&T->o_empty);
        }
        if (a.n_split > 1) {
          // [dim / 4][row][4]: a store covers 32 rows x 16 contiguous bytes
          float4* po = reinterpret_cast<float4*>(a.part_o + part * 128 * 128) + c * 8 * 128 + t;
          if (l != 0.0f) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              po[q * 128] = make_float4(y[4 * q], y[4 * q + 1], y[4 * q + 2], y[4 * q + 3]);
          }
          continue;
        }
        // 32 dims of the row as bf16 through shared memory (16-byte pieces,
        // swizzled), so that a store writes 64 contiguous bytes of eight rows
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t w[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const int i = q * 8 + 2 * h;
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(y[i], y[i + 1]);
            w[h] = *reinterpret_cast<const uint32_t*>(&b2) & keep;
          }
          *reinterpret_cast<uint4*>(stg + lane * 64 + ((q ^ (lane >> 1)) & 3) * 16) =
              make_uint4(w[0], w[1], w[2], w[3]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = 8 * i + (lane >> 2);
          const uint4 v = *reinterpret_cast<const uint4*>(
              stg + row * 64 + (((lane & 3) ^ (row >> 1)) & 3) * 16);
          if (out_nl[i] < a.N - node0)
            *reinterpret_cast<uint4*>(oitem + out_off[i] + c * 32) = v;
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) give_up();
  } else {
    // ---------------- softmax, two threads per tile row ----------------
    // Thread (row, half) takes keys 64 half .. +63 of each block.  Its O
    // accumulates in TMEM through the PV MMA with P = 2^(s - m_used); the
    // reference m_used moves (and O and the sum are rescaled in place) only
    // when a block's maximum exceeds it by more than 2^8, so P stays <= 256.
    const int half = (warp - 8) >> 2;
    const int quad = warp & 3;               // TMEM lanes quad*32 .. +31
    const int t = quad * 32 + lane;          // tile row
    const int nl = t / a.G;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    const uint32_t o_col = lane_base + kOCol + half * 128;
    const float sc = a.scale_log2;
    int g = 0;                               // blocks so far
    bool ok = true;
    for (int k = 0; ok && item_pos(k) < n_items; ++k) {
      AttnItem it;
      const int ab = k & 1;
      bool have_anc = false;                   // waited for where first needed
      if (!(ok = fetch_warp(k, it))) break;
      const int node = it.qt * a.npt + nl;
      const bool row_ok = it.nblk > 0 && t < a.R && node < it.n;
      const uint32_t* anc = T->anc[ab][row_ok ? node : 0];
      const int Tp = it.Tp, n_keys = it.Tp + it.n, key1 = it.key1, nblk = it.nblk;
      float m_used = -INFINITY, l_sum = 0.0f;  // O and l_sum are relative to m_used
      for (int b = 0; b < nblk; ++b, ++g) {
        const int sb = g & 1;
        const int key0 = it.key0 + b * kBK, hkey0 = key0 + half * 64;
        if (!(ok = wwait(&T->s_full[sb], (g >> 1) & 1))) break;
        tc_fence_after_sync();
        const uint32_t s_col = lane_base + sb * kBK + half * 64;
        float x[64];
        {
          uint32_t* xu = reinterpret_cast<uint32_t*>(x);
#pragma unroll
          for (int c = 0; c < 2; ++c)
            tmem_ld_32x32b_x32(s_col + c * 32,
                               *reinterpret_cast<uint32_t(*)[32]>(xu + c * 32));
          tmem_ld_wait();
        }
        // keys the row may not see become -inf (rows that store nothing take
        // part unmasked in blocks of prefix keys: their sums are dropped at
        // the item's end)
        if (hkey0 + 64 > min(Tp, key1)) {
          if (!have_anc && hkey0 + 64 > Tp) {
            if (!(ok = wwait(&T->anc_full[ab], (k >> 1) & 1))) break;
            have_anc = true;
          }
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t al = row_ok ? allowed_bits(hkey0 + c * 32, Tp, anc) : 0u;
            const int left = key1 - hkey0 - c * 32;   // keys of this range
            if (left < 32) al = left <= 0 ? 0u : al & ((1u << left) - 1u);
#pragma unroll
            for (int k2 = 0; k2 < 32; ++k2)
              x[c * 32 + k2] = ((al >> k2) & 1u) ? x[c * 32 + k2] : -INFINITY;
          }
        }
        float m8[8];                         // independent running maxima
#pragma unroll
        for (int u = 0; u < 8; ++u) m8[u] = x[u];
#pragma unroll
        for (int k2 = 8; k2 < 64; ++k2) m8[k2 & 7] = fmaxf(m8[k2 & 7], x[k2]);
        const float mx = fmaxf(fmaxf(fmaxf(m8[0], m8[1]), fmaxf(m8[2], m8[3])),
                         fmaxf(fmaxf(m8[4], m8[5]), fmaxf(m8[6], m8[7]))) * sc;
        // the last block of the request: V rows past the tree hold whatever
        // the cache held there; zero them so that 0 * (non-finite) cannot
        // reach O
        const int valid = n_keys - key0;
        if (valid < kBK) {
          const int xv = 2 * g + 1;          // V's place in the ring sequence
          if (!(ok = wwait(&T->kv_full[xv % kSlots], (xv / kSlots) & 1))) break;
          uint8_t* v = skv + (xv % kSlots) * kTileBytes;
          for (int i = half * 128 + t; i < 2 * (kBK - valid) * 8; i += 256) {
            const int vh = i >= (kBK - valid) * 8, rem = i - vh * (kBK - valid) * 8;
            *reinterpret_cast<uint4*>(v + vh * kHalfBytes + (valid + rem / 8) * 128 +
                                      (rem % 8) * 16) = make_uint4(0, 0, 0, 0);
          }
          fence_proxy_async_smem();          // the PV product reads V after p_full
        }
        // move the reference up where a row needs it (rare after an item's
        // first block); tcgen05.ld / st are warp-collective, so the warp
        // rescales together (alpha = 1 for rows that keep their reference)
        if (__any_sync(kFull, mx > m_used + 8.0f)) {
          const bool mine = mx > m_used + 8.0f;
          const float alpha = mine ? ex2_approx(m_used - mx) : 1.0f;   // 0 from -inf
          if (b >= 1) {
            // O must hold every block before b: the PV product of block b - 1
            // has finished
            if (!(ok = wwait(&T->p_empty[(g - 1) & 1], ((g - 1) >> 1) & 1))) break;
            tc_fence_after_sync();
            // eight columns at a time: the block's scores stay live meanwhile
#pragma unroll 2
            for (int c = 0; c < 16; ++c) {
              uint32_t y[8];
              tmem_ld_32x32b_x8(o_col + c * 8, y);
              tmem_ld_wait();
#pragma unroll
              for (int k2 = 0; k2 < 8; ++k2)
                y[k2] = __float_as_uint(__uint_as_float(y[k2]) * alpha);
              tmem_st_32x32b_x8(o_col + c * 8, y);
            }
            tmem_st_wait();
          }
          if (mine) {
            l_sum *= alpha;
            m_used = mx;
          }
        }
        // P = 2^(s - m_used) in bf16 pairs over the first 32 of the half's S
        // columns: the TMEM A operand of the PV MMA.  The scaling and the sums
        // go two at a time (fma / add .f32x2).
        const float mref = m_used == -INFINITY ? 0.0f : m_used;
        const uint64_t sc2 = pack2(sc, sc), nm2 = pack2(-mref, -mref);
        uint64_t ls[4] = {0, 0, 0, 0};
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int h = 0; h < 16; ++h) {
            float e0, e1;
            unpack2(fma2(pack2(x[c * 32 + 2 * h], x[c * 32 + 2 * h + 1]), sc2, nm2), e0, e1);
            const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);
            ls[h & 3] = add2(ls[h & 3], pack2(p0, p1));
            const __nv_bfloat162 pb = __floats2bfloat162_rn(p0, p1);
            pk[h] = *reinterpret_cast<const uint32_t*>(&pb);
          }
          tmem_st_32x32b_x16(s_col + c * 16, pk);
        }
        tmem_st_wait();
        {
          float s0, s1;
          unpack2(add2(add2(ls[0], ls[1]), add2(ls[2], ls[3])), s0, s1);
          l_sum += s0 + s1;
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&T->p_full[sb]);
      }
      if (!ok) break;
      // the ancestor bits of this item are no longer needed
      if (!have_anc && !(ok = wwait(&T->anc_full[ab], (k >> 1) & 1))) break;
      __syncwarp();
      if (lane == 0) mbar_arrive(&T->anc_empty[ab]);
      // the item's row sums, once the output warps have read the last item's
      if (!(ok = wwait(&T->o_empty, (k & 1) ^ 1))) break;
      T->row_l[half][t] = row_ok ? l_sum : 0.0f;
      T->row_m[half][t] = m_used;
      __syncwarp();
      if (lane == 0) mbar_arrive(&T->o_full);
    }
    if (!ok && lane == 0) give_up();
  }
  // ---------------- teardown ----------------
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// Merges the key splits of every (request, KV head, tile) unit: one thread
// per four output dims of a row, 16 rows x 32 dims per CTA.  Per row the
// splits' maxima and sums give weights 2^(m_s - m*); the weighted partial
// outputs are summed U splits at a time (their loads in flight together) and
// normalised.  At most 64 registers a thread, so that its CTAs fit beside the
// attention kernel's.  U follows the number of splits: the loads and weights
// of eight cost a unit of two splits 2 us more (us per layer, U = 8 / this: 26
// requests of 20 nodes with prefixes to 387 15.1 / 13.5, 10 of 16 to 586 16.0 /
// 14.3; U = 2 with four such columns a thread 15.0, 16.7: its code runs cold).
constexpr int kMergeThreads = 128;
constexpr int kMergeRows = 16;

template <int U>
__global__ void __launch_bounds__(kMergeThreads, 8)
tree_attn_merge_kernel(AttnArgs a) {
  // launched while the attention kernel finishes: its partials are read
  // after it is complete
  pdl_launch_dependents();
  pdl_wait();
  const int unit = blockIdx.x;
  const int row = blockIdx.y * kMergeRows + (threadIdx.x >> 3);   // tile row
  const int quad = blockIdx.z * 8 + (threadIdx.x & 7);            // dims 4 quad .. +3
  const int qt = unit % a.nqt;
  const int kvh = (unit / a.nqt) % a.Hkv;
  const int r = unit / (a.nqt * a.Hkv);
  const int nl = row / a.G, g = row - nl * a.G;
  const int node = qt * a.npt + nl;
  if (row >= a.R || node >= a.N) return;
  const size_t s_first = static_cast<size_t>(unit) * a.n_split;
  const float2* ml = a.part_ml + s_first * 128 + row;
  const float4* po = reinterpret_cast<const float4*>(a.part_o) + s_first * 32 * 128 + quad * 128 + row;
  float m = -INFINITY, lsum = 0.0f;
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int s0 = 0; s0 < a.n_split; s0 += U) {
    float2 w[U];
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = s0 + u < a.n_split;
      w[u] = in ? ml[static_cast<size_t>(s0 + u) * 128] : make_float2(-INFINITY, 0.0f);
      // a split without keys (sum 0) wrote no O: its values are not used
      v[u] = in ? po[static_cast<size_t>(s0 + u) * 32 * 128] : acc;
    }
    float mn = m;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (w[u].y != 0.0f) mn = fmaxf(mn, w[u].x);
    const float f0 = mn > m && m > -INFINITY ? exp2f(m - mn) : 1.0f;
    lsum *= f0;
    acc.x *= f0;
    acc.y *= f0;
    acc.z *= f0;
    acc.w *= f0;
    m = mn;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (w[u].y != 0.0f) {
        const float f = exp2f(w[u].x - m);
        lsum = fmaf(w[u].y, f, lsum);
        acc.x = fmaf(v[u].x, f, acc.x);
        acc.y = fmaf(v[u].y, f, acc.y);
        acc.z = fmaf(v[u].z, f, acc.z);
        acc.w = fmaf(v[u].w, f, acc.w);
      }
    }
  }
  const float inv = lsum != 0.0f ? 1.0f / lsum : 0.0f;   // (NaN stays)
  uint16_t* orow =
      a.out + ((static_cast<size_t>(r) * a.N + node) * a.Hq + kvh * a.G + g) * 128 + quad * 4;
  const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x * inv, acc.y * inv);
  const __nv_bfloat162 hi = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(orow) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo),
                                               *reinterpret_cast<const uint32_t*>(&hi));
}

}  // namespace
}  // namespace pct

namespace pct {
namespace {

// Tiling of a configuration: query tiles per (request, KV head) and
// the split of each request's keys (in units of a block) over items.  Splits are
// chosen so that there are about as many items as the 152 SMs of a GB300 when
// there are few (request, KV head, tile) units; they depend only on the
// configuration, so the workspace size does too.  Caches of fewer than 12 blocks
// get no more items than SMs: the second item of some CTAs and the merge cost more
// than the shorter ranges save; longer ones gain, since the prefixes differ
// (us per layer, more / no more: 14 requests of 4 nodes with prefixes to 174, 64
// heads 14.0 / 8.2; 16 of 4 to 1128 18.4 / 14.5; 12 of 21 to 1393, 40 heads 17.3 /
// 17.3; 14 of 20 to 2854 25.5 / 28.8; 13 of 15 to 6108 49.9 / 56.7).
struct AttnGeom {
  int G, npt, R, nqt, nb_max, n_split, bps;
  long long units;                    // (request, KV head, query tile) triples
};

AttnGeom attn_geom(const pctree_attn_config& c) {
  AttnGeom g{};
  g.G = c.Hq / c.Hkv;
  g.npt = 128 / g.G < c.N ? 128 / g.G : c.N;
  g.R = g.G * g.npt;
  g.nqt = (c.N + g.npt - 1) / g.npt;
  g.units = static_cast<long long>(c.batch) * c.Hkv * g.nqt;
  g.nb_max = (c.max_slots + kSplitKeys - 1) / kSplitKeys;
  long long want = ((g.nb_max < 12 ? 0 : g.units - 1) + 152) / g.units;
  if (want > g.nb_max) want = g.nb_max;
  if (want < 1) want = 1;
  g.bps = static_cast<int>((g.nb_max + want - 1) / want);
  g.n_split = (g.nb_max + g.bps - 1) / g.bps;
  return g;
}

pctree_status attn_check(const pctree_attn_config* c) {
  if (c == nullptr) return PCTREE_ERR_INVALID_ARG;
  if (c->batch < 1 || c->N < 1 || c->Hq < 1 || c->Hkv < 1 || c->D < 1 ||
      c->max_slots < c->N || !(c->scale > 0.0f) || !(c->scale < 1e30f))
    return PCTREE_ERR_INVALID_ARG;
  if (c->Hq % c->Hkv != 0) return PCTREE_ERR_INVALID_ARG;
  if (c->D != 128 || c->Hq / c->Hkv > 128 || c->N > PCTREE_ATTN_MAX_N ||
      c->batch > 65535 || c->Hkv > 65535)
    return PCTREE_ERR_UNSUPPORTED;
  const AttnGeom g = attn_geom(*c);
  if (static_cast<long long>(c->batch) * c->Hkv * g.nqt * g.n_split > 0x7fffffffll)
    return PCTREE_ERR_UNSUPPORTED;
  return PCTREE_OK;
}

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

struct AttnWs {
  size_t part_o, part_ml, total;
};

AttnWs attn_ws(const pctree_attn_config& c, const AttnGeom& g) {
  AttnWs w{};
  if (g.n_split <= 1) return w;
  const size_t slots = static_cast<size_t>(g.units) * g.n_split * 128;
  w.part_o = 0;
  w.part_ml = align256(w.part_o + slots * 128 * sizeof(float));
  w.total = align256(w.part_ml + slots * sizeof(float2));
  return w;
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace
}  // namespace pct

extern "C" {

size_t pctree_tree_attention_workspace_bytes(const pctree_attn_config* cfg) {
  if (pct::attn_check(cfg) != PCTREE_OK) return 0;
  return pct::attn_ws(*cfg, pct::attn_geom(*cfg)).total;
}

pctree_status pctree_tree_attention(const pctree_attn_config* cfg, const void* q,
                                    const void* k_cache, const void* v_cache,
                                    const int32_t* prefix_len,
                                    const int32_t* n_nodes, const int32_t* parent,
                                    void* out, void* workspace,
                                    size_t workspace_bytes, int32_t* status,
                                    void* stream_ptr) {
  pct::NvtxRange range("pctree_tree_attention");
  using namespace pct;
  pctree_status st = attn_check(cfg);
  if (st != PCTREE_OK) return st;
  const pctree_attn_config& c = *cfg;
  if (q == nullptr || k_cache == nullptr || v_cache == nullptr ||
      prefix_len == nullptr || n_nodes == nullptr || parent == nullptr ||
      out == nullptr || !al16(q) || !al16(k_cache) || !al16(v_cache) || !al16(out))
    return PCTREE_ERR_INVALID_ARG;
  const AttnGeom g = attn_geom(c);
  const AttnWs w = attn_ws(c, g);
  if (w.total > 0 && (workspace == nullptr || workspace_bytes < w.total ||
                      (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0))
    return PCTREE_ERR_WORKSPACE;
  int num_sms = 0;
  st = device_facts(&num_sms);
  if (st != PCTREE_OK) return st;
  CUtensorMap tm_q, tm_k, tm_v;
  const uint64_t hd = 128 * 2;                       // bytes of one head row
  {
    const uint64_t dims[4] = {128, static_cast<uint64_t>(c.Hq),
                              static_cast<uint64_t>(c.N), static_cast<uint64_t>(c.batch)};
    const uint64_t str[3] = {hd, hd * c.Hq, hd * c.Hq * c.N};
    const uint32_t box[4] = {64, static_cast<uint32_t>(g.G), static_cast<uint32_t>(g.npt), 1};
    st = encode_bf16_map_nd(&tm_q, q, 4, dims, str, box);
    if (st != PCTREE_OK) return st;
  }
  {
    const uint64_t dims[4] = {128, static_cast<uint64_t>(c.Hkv),
                              static_cast<uint64_t>(c.max_slots),
                              static_cast<uint64_t>(c.batch)};
    const uint64_t str[3] = {hd, hd * c.Hkv, hd * c.Hkv * c.max_slots};
    const uint32_t box[4] = {64, 1, static_cast<uint32_t>(kBK), 1};
    st = encode_bf16_map_nd(&tm_k, k_cache, 4, dims, str, box);
    if (st != PCTREE_OK) return st;
    st = encode_bf16_map_nd(&tm_v, v_cache, 4, dims, str, box);
    if (st != PCTREE_OK) return st;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(stream_ptr);
  AttnArgs a{};
  a.prefix = prefix_len;
  a.n_nodes = n_nodes;
  a.parent = parent;
  a.out = static_cast<uint16_t*>(out);
  a.status = status;
  a.batch = c.batch;
  a.N = c.N;
  a.Hq = c.Hq;
  a.Hkv = c.Hkv;
  a.G = g.G;
  a.npt = g.npt;
  a.R = g.R;
  a.nqt = g.nqt;
  a.items = static_cast<int>(static_cast<long long>(c.batch) * c.Hkv * g.nqt * g.n_split);
  a.max_slots = c.max_slots;
  a.n_split = g.n_split;
  a.bps = g.bps;
  a.scale_log2 = static_cast<float>(static_cast<double>(c.scale) * 1.4426950408889634);
  if (w.total > 0) {
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    a.part_o = reinterpret_cast<float*>(ws + w.part_o);
    a.part_ml = reinterpret_cast<float2*>(ws + w.part_ml);
  }
  // a dummy status word is not needed: kernels test for NULL
  static SmemLimit limit;
  if (limit.ensure(reinterpret_cast<const void*>(tree_attn_kernel), kAttnSmem) != cudaSuccess)
    return PCTREE_ERR_CUDA;
  // persistent: one CTA per SM walks its share of the items; both kernels
  // are launched with programmatic stream serialization (each waits for its
  // predecessor before touching global memory)
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(static_cast<unsigned>(a.items < num_sms ? a.items : num_sms));
  lc.stream = stream;
  lc.attrs = attr;
  lc.numAttrs = 1;
  lc.blockDim = dim3(kAttnThreads);
  lc.dynamicSmemBytes = kAttnSmem;
  if (cudaLaunchKernelEx(&lc, tree_attn_kernel, tm_q, tm_k, tm_v, a) != cudaSuccess)
    return PCTREE_ERR_CUDA;
  if (g.n_split > 1) {
    lc.gridDim = dim3(static_cast<unsigned>(g.units), (g.R + kMergeRows - 1) / kMergeRows, 4);
    lc.blockDim = dim3(kMergeThreads);
    lc.dynamicSmemBytes = 0;
    const cudaError_t e = g.n_split <= 2   ? cudaLaunchKernelEx(&lc, tree_attn_merge_kernel<2>, a)
                          : g.n_split <= 4 ? cudaLaunchKernelEx(&lc, tree_attn_merge_kernel<4>, a)
                                           : cudaLaunchKernelEx(&lc, tree_attn_merge_kernel<8>, a);
    if (e != cudaSuccess) return PCTREE_ERR_CUDA;
  }
  return PCTREE_OK;
}

}  // extern "C"
