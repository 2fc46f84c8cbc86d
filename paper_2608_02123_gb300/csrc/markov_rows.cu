// Markov projection of one PCTree stage with the stage's log-softmax
// normaliser and per-parent top-k folded into the epilogue (Eqs. 2-3), for
// bf16 heads and any number of Markov rows:
//
//   z[row][v] = L_d[req(row)][v] + sum_h X[row][h] * W_out[v][h]
//
// is formed tile by tile in tensor memory and never written to HBM.  For
// every parent row a CTA keeps, over its share of the vocabulary, a running
// log-sum-exp and a sorted top-k list; at the end it publishes them as one
// partial per (row, vocabulary slot), which the stage's merge combines into
// the row's normaliser and children.
//
// Layout of the work.  The parent rows are the MMA's M, the vocabulary its N:
// TMEM lane = parent row, so that each epilogue thread owns one row, reads its
// logits column by column and keeps the row's sums and list in registers (with
// the vocabulary as M every 64 x 128 chunk went through shared memory to be
// transposed, and its row reductions through warp shuffles).
//   rows <= 128: one CTA per vocabulary slot, tcgen05.mma M = 128, N = 256.
//   rows > 128:  a pair of CTAs (cta_group::2) per (slot, group of 256 rows),
//                M = 256, N = 256; each CTA stages its 128 rows of X and half
//                of the W_out tile, 32 KB for a K chunk where a single CTA with
//                256 rows needs 48: the pass was bound by the bytes it could
//                keep in flight.  Pairs of different row groups take the same
//                vocabulary tile at the same time, so W_out comes from HBM
//                once a stage for any number of rows.
// A slot owns a contiguous range of the vocabulary in units of 16 to 128
// entries (all slots equal to within one unit; the unit's rows are one TMA box
// of W_out: a box costs the issuing thread ~145 ns whatever its size, so a tile
// loaded in 16-row boxes streams at half the HBM rate), in tiles of up to
// 256.  Warp 0 streams X and W_out with TMA into a shared-memory ring, warp
// 1 issues the MMAs into two 256-column TMEM buffers, warps 2..9 are the
// epilogue: warp quadrant = TMEM lanes, four warps for the columns 0..127 of a
// tile and four for 128..255; the two lists of a row meet at the end (few rows:
// a warp to a row, see few_rows).
//
// The slots also share, per row, the best k-th list entry any of them holds
// (a 64-bit word in global memory raised with atomicMax after each tile): a
// logit below it is beaten by k logits of that list alone, so it cannot be one
// of the row's k children and is not inserted.  The shared value only removes
// candidates that lose anyway, so the merged children do not depend on when a
// thread reads it.  Rows are always handled by the same threads in the same
// order.
//
// Measured against the vocabulary as M (us per round, alternating runs): 14B-
// shaped (512 rows, H 5120) 10540 -> 8804 under the power cap: the MMA pipe is
// busy 84 % of its cycles at ~1.45 GHz; 8B-shaped (128 rows, H 4096) 1451 ->
// 1360, 0.955 of the copy rate; 151936 x 64 with 64 rows 460 -> 298, 30000 x
// 1024 with 512 rows 1120 -> 489 (epilogue-bound before).  With what the comments
// below add: 14B-shaped 8660, 8B-shaped 1320, 4B-shaped (8 rows, H 2560, 16
// stages) 2017 -> 1840 against the fused round it had, W_out at the copy rate.
#include <cuda_runtime.h>

#include "pctree_common.cuh"
#include "sm103_ptx.cuh"

namespace pct {
namespace {

constexpr int kBN = 256;          // vocabulary entries per tile (MMA N)
constexpr int kBK = 64;           // K elements per ring slot (128 B of bf16)
constexpr int kUmmaK = 16;        // K per tcgen05.mma kind::f16
constexpr int kEpiWarps = 8;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kRowBytes = kBK * 2;
constexpr int kMaxStages = 12;
constexpr int kBarBytes = 512;
constexpr int kSmemLimit = 227 * 1024;
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s per bounded wait
constexpr float kNegInf = -INFINITY;
constexpr float kPosInf = INFINITY;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kNoToken = 0x7fffffff;
constexpr long long kStreamBytes = 384ll << 20;   // heads above: three times L2

struct RowsArgs {
  const float* L;          // base logits of depth d, request 0
  long long l_req_stride;  // floats between two requests' rows
  int V, H, k, rows, rows_per_req;
  int n_stages;            // ring slots
  int stage_bytes;         // bytes of a ring slot
  int x_box;               // parent rows per CTA and TMA box
  int unit;                // vocabulary entries per unit of the slots' ranges
  int small_box;           // W_out rows of tmap_ws's boxes
  int groups;              // row groups (of 128, or 256 for pairs)
  int tile;                // most entries of a tile
  int n_slots;             // vocabulary slots = partials per row
  int z_bytes;             // FEW: shared memory of a tile's accumulators
  int tiled;               // 1: W_out in the tiled layout (PCTREE_HEAD_TILED)
  int l_vec;               // 1: base logits can be read as float4
  float* part_m;           // [rows][n_slots] largest logit
  float* part_s;           // [rows][n_slots] sum of exp relative to it
  float* part_z;           // [rows][n_slots][k] top-k logits, best first
  int32_t* part_t;         // [rows][n_slots][k] their tokens
  // [rows] per row: (tag << 32) | order key of the best k-th list entry of
  // any slot; entries of earlier stages carry smaller tags and count as empty
  unsigned long long* gthr;
  unsigned tag;            // stage + 1
  int32_t* status;
};

// The vocabulary range of a slot, in units, and its tiles.  PAIR: up to the
// next multiple of 256, so that nearly every W_out box is a whole 128-row
// block.  Else tiles of equal numbers of units: a short one would stream with
// fewer bytes in flight (a last tile of 64 entries cost as much as one of 192).
template <bool PAIR, bool STREAM>
struct Range {
  int lo, hi;              // entries [lo, hi)
  int n;                   // tiles
  int unit;
  bool flip;
  // walk from the last tile (and K chunk) to the first
  __device__ __forceinline__ bool back() const { return STREAM && flip; }
  __device__ __forceinline__ Range(int V, int unit_, int slot, int n_slots, int tile_, bool flip_)
      : unit(unit_), flip(flip_) {
    const long long units = (V + unit - 1) / unit;
    lo = static_cast<int>(units * slot / n_slots) * unit;
    hi = static_cast<int>(units * (slot + 1) / n_slots) * unit;
    n = PAIR ? (hi + kBN - 1 - lo / kBN * kBN) / kBN : (hi - lo + tile_ - 1) / tile_;
  }
  __device__ __forceinline__ int start(int i) const {
    if constexpr (PAIR) return i == n ? hi : max(lo, lo / kBN * kBN + i * kBN);
    return lo + (hi - lo) / unit * i / n * unit;
  }
  // the i-th tile of the walk
  __device__ __forceinline__ void tile(int i, int& t_lo, int& t_n) const {
    const int at = back() ? n - 1 - i : i;
    t_lo = start(at);
    t_n = start(at + 1) - t_lo;
  }
};

// Sorted top-KL list of one row in a thread's registers, best first, as order
// keys with tokens.  For k < KL the first KL - k entries hold the largest key
// and never move, so the k-th best is always the last entry.
template <int KL>
struct RegList {
  uint32_t key[KL];
  int tok[KL];
  __device__ __forceinline__ void reset(int k) {
#pragma unroll
    for (int j = 0; j < KL; ++j) {
      key[j] = j < KL - k ? 0xffffffffu : 0u;
      tok[j] = kNoToken;
    }
  }
  __device__ __forceinline__ uint32_t kth() const { return key[KL - 1]; }
  // Inserts a candidate whose token is above every token of the list (it
  // goes behind equal keys); one not better than the last entry drops out, as
  // does key 0 (no candidate).
  __device__ __forceinline__ void insert_later(uint32_t c, int t) {
#pragma unroll
    for (int j = KL - 1; j > 0; --j) {
      const bool up = c > key[j - 1], here = c > key[j];
      key[j] = up ? key[j - 1] : (here ? c : key[j]);
      tok[j] = up ? tok[j - 1] : (here ? t : tok[j]);
    }
    const bool here = c > key[0];
    key[0] = here ? c : key[0];
    tok[0] = here ? t : tok[0];
  }
  // Takes over the k entries KL - k .. KL - 1 of another such list, read by
  // `entry`: the better of entry i of this one and entry KL - 1 - i of those
  // (padded with empty ones) are the KL best of both, in a bitonic order that
  // log2 KL steps of compare-exchange sort.  (k inserts took 1 - 5 us.)
  template <typename Entry>
  __device__ __forceinline__ void merge(int k, Entry entry) {
    auto swap_if_better = [&](uint32_t& ka, int& ta, uint32_t kb, int tb) {
      const bool b = (kb > ka) | ((kb == ka) & (tb < ta));
      ka = b ? kb : ka;
      ta = b ? tb : ta;
      return b;
    };
#pragma unroll
    for (int i = 0; i < KL; ++i) {
      const int j = KL - k + KL - 1 - i;   // the other list's entry
      uint32_t c = 0u;
      int t = kNoToken;
      if (j < KL) entry(j, c, t);
      (void)swap_if_better(key[i], tok[i], c, t);
    }
#pragma unroll
    for (int d = KL / 2; d >= 1; d /= 2) {
#pragma unroll
      for (int i = 0; i < KL; ++i) {
        if ((i & d) == 0) {
          const uint32_t ka = key[i];
          const int ta = tok[i];
          const bool b = swap_if_better(key[i], tok[i], key[i + d], tok[i + d]);
          key[i + d] = b ? ka : key[i + d];
          tok[i + d] = b ? ta : tok[i + d];
        }
      }
    }
  }
  // The same as insert_later for any token: (key desc, token asc) order.
  __device__ __forceinline__ void insert(uint32_t c, int t) {
    auto better = [&](int j) { return (c > key[j]) | ((c == key[j]) & (t < tok[j])); };
#pragma unroll
    for (int j = KL - 1; j > 0; --j) {
      const bool up = better(j - 1), here = better(j);
      key[j] = up ? key[j - 1] : (here ? c : key[j]);
      tok[j] = up ? tok[j - 1] : (here ? t : tok[j]);
    }
    const bool here = better(0);
    key[0] = here ? c : key[0];
    tok[0] = here ? t : tok[0];
  }
};

// Sorts 16 values in registers, largest first (Batcher's odd-even merge sort;
// step (P, K) compares a with a + K inside blocks of 2 P).
template <int P, int K>
__device__ __forceinline__ void sort_step(float (&x)[16]) {
#pragma unroll
  for (int a = 0; a + K < 16; ++a) {
    if (a >= K % P && (a - K % P) % (2 * K) < K && a / (2 * P) == (a + K) / (2 * P)) {
      const float hi = fmaxf(x[a], x[a + K]), lo = fminf(x[a], x[a + K]);
      x[a] = hi;
      x[a + K] = lo;
    }
  }
}
__device__ __forceinline__ void sort16_desc(float (&x)[16]) {
  sort_step<1, 1>(x);
  sort_step<2, 2>(x);
  sort_step<2, 1>(x);
  sort_step<4, 4>(x);
  sort_step<4, 2>(x);
  sort_step<4, 1>(x);
  sort_step<8, 8>(x);
  sort_step<8, 4>(x);
  sort_step<8, 2>(x);
  sort_step<8, 1>(x);
}

__device__ __forceinline__ void epi_barrier() { named_barrier(1, kEpiThreads); }

// exp(z - R) for z <= R, R finite.  The difference is taken before it is scaled
// to a power of two: z log2 e alone overflows for a mask of the lowest float,
// and its rounding error grows with |z| (one of the logits near the maximum,
// which carry the sum, is exact here).
__device__ __forceinline__ float exp_diff(float z, float R) {
  return ex2_approx((z - R) * kLog2e);
}

// The largest of z, NaN if any is: every row's logits pass here, so that one
// that is NaN or +inf is seen also among -inf alone, where no sum of exp is formed.
__device__ __forceinline__ float max_of(const float (&z)[8]) {
  const float m = max_nan(z[0], z[1], z[2]);
  return max_nan(max_nan(m, z[3], z[4]), max_nan(z[5], z[6], z[7]));
}
__device__ __forceinline__ float max_of(const float (&z)[32]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = max_nan(z[3 * i], z[3 * i + 1], z[3 * i + 2]);
#pragma unroll
  for (int e = 12; e < 32; e += 2) m[e / 2 & 3] = max_nan(m[e / 2 & 3], z[e], z[e + 1]);
  return max_nan(max_nan(m[0], m[1]), m[2], m[3]);
}

// The sum of exp(z[e] - R) over e, two at a time.
template <int N>
__device__ __forceinline__ float sum_exp(const float (&z)[N], float R) {
  constexpr int kSums = N >= 32 ? 4 : 2;   // independent chains
  const uint64_t nr = pack2(-R, -R), sc = pack2(kLog2e, kLog2e);
  float s[kSums];
#pragma unroll
  for (int i = 0; i < kSums; ++i) s[i] = 0.0f;
#pragma unroll
  for (int e = 0; e < N; e += 2) {
    float x0, x1;
    unpack2(mul2(add2(pack2(z[e], z[e + 1]), nr), sc), x0, x1);
    s[e % kSums] += ex2_approx(x0);
    s[e % kSums + 1] += ex2_approx(x1);
  }
  if constexpr (kSums == 4) return (s[0] + s[1]) + (s[2] + s[3]);
  return s[0] + s[1];
}

// The epilogue for few rows.  Only one warp in four can read the accumulators
// of rows 0..31, so with a thread to a row two warps of eight and half their
// lanes would do all of it (16 rows with lists of 16 spent 27 of a stage's 41
// thousand cycles so).  Instead those two warps put each tile's accumulators into
// shared memory and each of the eight takes OWN whole rows (ew, ew + 8, ...) of
// it: lane l the columns 4 l .. 4 l + 3 and 128 more, a sorted list spread over
// the lanes.  us per round of 7 stages, a thread to a row / this: 12000 x 1024
// with 8 rows 147 / 119, with 16 rows and lists of 16 235 / 163; 32000 x 4096 379
// / 341; 4000 x 256 94 / 80; 151936 x 2560 in 16 stages with 8 rows 1886 / 1840,
// with one 1826 / 1780.
template <bool STREAM, int OWN>
__device__ __forceinline__ void few_rows(const RowsArgs& a, const Range<false, STREAM>& range,
                                         uint32_t tmem_base, uint64_t* bars, uint64_t* acc_full,
                                         uint64_t* acc_empty, volatile int* abort_v,
                                         int* stop_flag, int slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ew = warp - 2;
  const bool reader = (warp & 3) == 0;     // TMEM lanes 0..31
  float* zs = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(bars) + kBarBytes);
  const int pitch = (a.tile <= 128 ? 128 : 256) + 4;
  const int own = a.rows > ew ? (a.rows - ew + 7) / 8 : 0;   // rows ew, ew + 8, ...
  // base logits of this lane's columns of a tile, loaded one tile ahead
  float l[OWN][8];
  auto load_row = [&](int row, int t_lo, int end, float (&dst)[8]) {
    const float* Lr = a.L + static_cast<long long>(row / a.rows_per_req) * a.l_req_stride;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int v = t_lo + 128 * j + 4 * lane;
      if (a.l_vec && v + 3 < end) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(Lr + v));
        dst[4 * j] = f.x;
        dst[4 * j + 1] = f.y;
        dst[4 * j + 2] = f.z;
        dst[4 * j + 3] = f.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[4 * j + e] = v + e < end ? __ldg(Lr + v + e) : 0.0f;
      }
    }
  };
  auto load_l = [&](int i) {
    if (i >= range.n) return;
    int t_lo, t_n;
    range.tile(i, t_lo, t_n);
    const int end = min(t_lo + t_n, a.V);
#pragma unroll
    for (int o = 0; o < OWN; ++o)
      if (o < own) load_row(ew + 8 * o, t_lo, end, l[o]);
  };
#pragma unroll
  for (int i = 0; i < 8 * OWN; ++i) l[i / 8][i % 8] = 0.0f;
  load_l(0);
  pdl_wait();
  // per row: sum of exp(z - R) over this lane's columns, R their largest; its list
  float Rs[OWN], Ss[OWN];
  WarpList lists[OWN];
#pragma unroll
  for (int o = 0; o < OWN; ++o) {
    Rs[o] = kNegInf;
    Ss[o] = 0.0f;
    lists[o].reset();
  }
  bool bad = false, ok = true;
  int acc = 0;
  uint32_t acc_phase = 0;
  for (int i = 0; i < range.n; ++i) {
    int t_lo, t_n;
    range.tile(i, t_lo, t_n);
    const int end = min(t_lo + t_n, a.V);
    // the shared thresholds, read past L1 while the tile is still computed
    unsigned long long words[OWN];
#pragma unroll
    for (int o = 0; o < OWN; ++o) words[o] = i > 0 && o < own ? __ldcg(a.gthr + ew + 8 * o) : 0ull;
    // (a warp whose wait runs out still meets the others at the barriers)
    if (ok)
      ok = __all_sync(kFull, mbar_wait_bounded(&acc_full[acc], acc_phase, abort_v, kWaitLimitNs));
    tc_fence_after_sync();
    if (i > 0) epi_barrier();              // the last tile has been read
    if (ok && reader) {
      for (int c = warp == 4 ? 0 : 32; c < t_n; c += 64) {
        uint32_t r[32];
        tmem_ld_32x32b_x32(tmem_base + static_cast<uint32_t>(acc * kBN + c), r);
        tmem_ld_wait();
        if (lane < a.rows) {
          uint4* to = reinterpret_cast<uint4*>(zs + lane * pitch + c);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            to[q] = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
        }
      }
      tc_fence_before_sync();
    }
    __syncwarp();
    if (ok && lane == 0) mbar_arrive(&acc_empty[acc]);
    epi_barrier();
#pragma unroll 1
    for (int o = 0; o < own && ok; ++o) {      // (one copy of this code: it runs cold)
      const int row = ew + 8 * o;
      WarpList lst;
      lst = lists[0];
#pragma unroll
      for (int q = 1; q < OWN; ++q) {
        lst.v = o == q ? lists[q].v : lst.v;
        lst.t = o == q ? lists[q].t : lst.t;
      }
      float R = pick(Rs, o), S = pick(Ss, o);
      const unsigned long long w = pick(words, o);
      float lv[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) lv[e] = l[0][e];
#pragma unroll
      for (int q = 1; q < OWN; ++q)
#pragma unroll
        for (int e = 0; e < 8; ++e) lv[e] = o == q ? l[q][e] : lv[e];
      const float gl = static_cast<unsigned>(w >> 32) == a.tag
                           ? key_float(static_cast<uint32_t>(w)) : kNegInf;
      float z[8];
      float mn = kPosInf;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = 128 * j + 4 * lane;
        float4 b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (128 * j < t_n) b = *reinterpret_cast<const float4*>(zs + row * pitch + c);
        const float bb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const bool in = t_lo + c + e < end;
          mn = fminf(mn, in ? bb[e] : kPosInf);
          z[4 * j + e] = in ? bb[e] + lv[4 * j + e] : kNegInf;
        }
      }
      // a Markov bias of -inf shows here; one that is NaN or +inf, and a NaN or
      // +inf base logit, in the logits (-inf base logits are legal)
      bad |= mn == kNegInf;
      const float lm = max_of(z);
      bad |= !(lm < kPosInf);
      if (lm > R) {
        S *= exp_diff(R, lm);
        R = lm;
      }
      if (R > kNegInf) S += sum_exp(z, R);
      const int tbase = t_lo + 4 * lane;
      unsigned skip = 0;
      if (i == 0) {
        // the list starts from the lanes' best logits (one sort instead of
        // inserts into an empty list)
        int li = 0;
#pragma unroll
        for (int e = 7; e >= 0; --e)
          if (z[e] == lm) li = e;
        const bool any = lm > kNegInf;
        lst.seed(any ? lm : kNegInf, any ? tbase + (li >> 2) * 128 + (li & 3) : kNoToken, a.k);
        if (any) skip = 1u << li;
      }
      const float tv = __shfl_sync(kFull, lst.v, a.k - 1);
      const int tt = __shfl_sync(kFull, lst.t, a.k - 1);
      // (a NaN is no candidate, but the logits beside it may be)
      if (__any_sync(kFull, !(lm < tv) && !(lm < gl))) {
        unsigned marks = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int t = tbase + (e >> 2) * 128 + (e & 3);
          marks |= static_cast<unsigned>((z[e] >= gl) &
                                         cand_better(z[e], t < end ? t : kNoToken, tv, tt))
                   << e;
        }
        marks &= ~skip;
        while (__any_sync(kFull, marks != 0)) {
          const int sel = marks != 0 ? __ffs(marks) - 1 : 0;
          const float cv = marks != 0 ? pick(z, sel) : kNegInf;
          const int ct = marks != 0 ? tbase + (sel >> 2) * 128 + (sel & 3) : kNoToken;
          marks &= marks - 1;
          lst.offer(cv, ct, a.k);
        }
      }
      // publish the row's k-th entry for the other slots
      const float kv = __shfl_sync(kFull, lst.v, a.k - 1);
      if (lane == 0 && kv > gl && (i == 0 || kv > tv))
        atomicMax(a.gthr + row, (static_cast<unsigned long long>(a.tag) << 32) | float_key(kv));
#pragma unroll
      for (int q = 0; q < OWN; ++q) {
        lists[q].v = o == q ? lst.v : lists[q].v;
        lists[q].t = o == q ? lst.t : lists[q].t;
        Rs[q] = o == q ? R : Rs[q];
        Ss[q] = o == q ? S : Ss[q];
      }
    }
    load_l(i + 1);
    if (++acc == 512 / kBN) {
      acc = 0;
      acc_phase ^= 1u;
    }
  }
  if (bad) set_status(a.status, PCTREE_ERR_NONFINITE);
  if (!ok && lane == 0) {
    *abort_v = 1;
    set_status(a.status, PCTREE_ERR_TIMEOUT);
  }
  // one decision for the eight warps
  epi_barrier();
  if (threadIdx.x == 64) *stop_flag = *abort_v;
  epi_barrier();
  if (*stop_flag) return;
#pragma unroll
  for (int o = 0; o < OWN; ++o) {
    if (o >= own) break;
    const int row = ew + 8 * o;
    const float R = Rs[o];
    float Rm = R, S = Ss[o];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) Rm = fmaxf(Rm, __shfl_xor_sync(kFull, Rm, d));
    S = R > kNegInf ? S * exp_diff(R, Rm) : 0.0f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) S += __shfl_xor_sync(kFull, S, d);
    const size_t p = static_cast<size_t>(row) * a.n_slots + slot;
    if (lane == 0) {
      a.part_m[p] = Rm;
      a.part_s[p] = S;
    }
    if (lane < a.k) {
      a.part_z[p * a.k + lane] = lists[o].v;
      a.part_t[p * a.k + lane] = lists[o].t;
    }
  }
}

// STREAM: W_out is far larger than L2 (see launch_markov_rows)
// FEW: at most 8 FEW rows (see few_rows), or 0
template <int KL, bool PAIR, bool STREAM, int FEW>
__global__ void __launch_bounds__(kThreads, 1)
markov_rows_kernel(const __grid_constant__ CUtensorMap tmap_w,     // 128-row boxes
                   const __grid_constant__ CUtensorMap tmap_ws,    // small_box rows
                   const __grid_constant__ CUtensorMap tmap_x,
                   const __grid_constant__ RowsArgs a) {
  constexpr bool EARLY = !PAIR;
  constexpr int kM = PAIR ? 256 : 128;
  constexpr int kAccBufs = 512 / kBN;
  constexpr uint32_t kTmemCols = kAccBufs * kBN;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int n_stages = a.n_stages;
  // ring slot: this CTA's X rows (K-major, 128 bytes each), then its W rows
  const int a_bytes = a.x_box * kRowBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + n_stages * a.stage_bytes);
  uint64_t* full = bars;                              // [kMaxStages]
  uint64_t* empty = full + kMaxStages;                // [kMaxStages]
  uint64_t* acc_full = empty + kMaxStages;            // [kAccBufs]
  uint64_t* acc_empty = acc_full + kAccBufs;          // [kAccBufs]
  uint64_t* drain = acc_empty + kAccBufs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  int* stop_flag = abort_flag + 1;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = PAIR ? static_cast<int>(cluster_ctarank()) : 0;
  const int unit_id = PAIR ? static_cast<int>(blockIdx.x) >> 1 : static_cast<int>(blockIdx.x);
  const int group = unit_id % a.groups, slot = unit_id / a.groups;
  const int row0 = group * kM + rank * 128;           // this CTA's first row
  const int n_k = (a.H + kBK - 1) / kBK;
  // odd stages of a streamed head walk backwards, so that a stage begins with
  // the W_out the last one read last, part of which is still in L2
  const Range<PAIR, STREAM> range(a.V, a.unit, slot, a.n_slots, a.tile, (a.tag & 1u) == 0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < kAccBufs; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], kEpiWarps * (PAIR ? 2 : 1));   // one arrival per warp
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    *stop_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmap_w);
    tma_prefetch_desc(&tmap_ws);
    tma_prefetch_desc(&tmap_x);
  }
  if (warp == 1) {
    if constexpr (PAIR) tmem_alloc_pair(tmem_slot, kTmemCols);
    else tmem_alloc(tmem_slot, kTmemCols);
  }
  tc_fence_before_sync();
  __syncthreads();
  // the peer's barriers are initialised before anything arrives on them
  if constexpr (PAIR) cluster_sync();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  volatile int* abort_v = abort_flag;
  // The set-up above overlaps the previous kernel of the stream, the merge that
  // writes this stage's parent rows.  EARLY: each role waits for it before it
  // touches what the round writes; stage 0 waits here, and lets later kernels
  // launch only then: those then know that everything before the round is
  // complete, so that from stage 1 on W_out and the base logits, which no
  // kernel of the round writes, are loaded before the wait (us per round of 7
  // stages: 12000 x 1024 152 -> 146, 151936 x 1024 404 -> 386, 32000 x 4096 389 ->
  // 379).  Pairs, bound by their MMAs: nothing below runs before the merge is
  // complete.
  if (EARLY && a.tag == 1) pdl_wait();
  pdl_launch_dependents();
  if (!EARLY) pdl_wait();

  if (warp == 0) {
    // --------------------------------------------------------------- producer
    if (lane == 0) {
      // W_out is read once by a single row group, else again by the others'
      // pairs at about the same time: leave it in L2 for them
      const uint64_t w_policy = a.groups == 1 ? l2_policy_evict_first() : l2_policy_evict_normal();
      const uint64_t x_policy = l2_policy_evict_normal();
      int stage = 0;
      uint32_t phase = 0;
      // ring slots armed here (by the even CTA of a pair for both), and the
      // phase each was armed in
      uint32_t armed = 0, armed_phase = 0;
      bool ok = true;
      auto load = [&](int st, unsigned char* to, const CUtensorMap* map, int x, int y,
                      uint64_t policy) {
        if constexpr (PAIR) tma_load_2d_pair(to, map, mapa_shared(&full[st], 0), x, y, policy);
        else tma_load_2d_hint(to, map, &full[st], x, y, policy);
      };
      auto load_x = [&](int st, int kx) {
        load(st, ring + st * a.stage_bytes, &tmap_x, kx * kBK, row0, x_policy);
      };
      // slots that still lack their parent rows; -1 once those can be loaded
      int held = EARLY && a.tag > 1 ? 0 : -1;
      auto parents = [&]() {        // the merge is complete: load them
        pdl_wait();
        for (int s = 0; s < held; ++s) load_x(s, range.back() ? n_k - 1 - s % n_k : s % n_k);
        held = -1;
      };
      for (int i = 0; i < range.n && ok; ++i) {
        int t_lo, t_n;
        range.tile(i, t_lo, t_n);
        const int b_rows = PAIR ? t_n / 2 : t_n;      // W rows of this CTA
        const int b_lo = t_lo + rank * b_rows;
        for (int kc = 0; kc < n_k; ++kc) {
          // the ring is full of slots waiting for the parent rows
          if (EARLY && held == n_stages) parents();
          if (!mbar_wait_bounded(&empty[stage], phase ^ 1u, abort_v, kWaitLimitNs)) {
            ok = false;
            break;
          }
          const int kx = range.back() ? n_k - 1 - kc : kc;
          unsigned char* dst = ring + stage * a.stage_bytes;
          if (rank == 0) {
            mbar_arrive_expect_tx(&full[stage], static_cast<uint32_t>(
                                                    (PAIR ? 2 : 1) * (a_bytes + b_rows * kRowBytes)));
            armed |= 1u << stage;
            armed_phase = (armed_phase & ~(1u << stage)) | (phase << stage);
          }
          // the W rows, in whole 128-row blocks where the range allows
          for (int r = 0; r < b_rows;) {
            const int v = b_lo + r, in = v & 127;
            const bool whole = in == 0 && b_rows - r >= 128;
            const int y = a.tiled ? ((v >> 7) * n_k + kx) * 128 + in : v;
            load(stage, dst + a_bytes + r * kRowBytes, whole ? &tmap_w : &tmap_ws,
                 a.tiled ? 0 : kx * kBK, y, w_policy);
            r += whole ? 128 : a.small_box;
          }
          if (EARLY && held >= 0) ++held;
          else load_x(stage, kx);
          if (++stage == n_stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (EARLY && held >= 0) parents();     // (also after a wait that ran out: every armed
                                    // slot gets its bytes)
      if (!ok) {
        *abort_v = 1;
        set_status(a.status, PCTREE_ERR_TIMEOUT);
      }
      // every copy armed here must land before the CTA may exit
      volatile int never = 0;
      for (int s = 0; s < n_stages; ++s)
        if ((armed >> s) & 1u)
          mbar_wait_bounded(&full[s], (armed_phase >> s) & 1u, &never, kWaitLimitNs);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------- MMA issue
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      const uint64_t a_desc0 = desc_kmajor_sw128(smem_u32(ring));
      const uint64_t b_desc0 = desc_kmajor_sw128(smem_u32(ring) + a_bytes);
      for (int i = 0; i < range.n && ok; ++i) {
        int t_lo, t_n;
        range.tile(i, t_lo, t_n);
        const uint32_t idesc = idesc_bf16_f32(kM, t_n);
        if (!mbar_wait_bounded(&acc_empty[acc], acc_phase ^ 1u, abort_v, kWaitLimitNs)) {
          ok = false;
          break;
        }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kBN);
        for (int kc = 0; kc < n_k; ++kc) {
          if (!mbar_wait_bounded(&full[stage], phase, abort_v, kWaitLimitNs)) {
            ok = false;
            break;
          }
          tc_fence_after_sync();
          const uint64_t off = static_cast<uint64_t>(stage) * (a.stage_bytes >> 4);
#pragma unroll
          for (int kk = 0; kk < kBK / kUmmaK; ++kk) {
            const uint64_t ad = a_desc0 + off + (kk * kUmmaK * 2 >> 4);
            const uint64_t bd = b_desc0 + off + (kk * kUmmaK * 2 >> 4);
            const uint32_t keep = (kc | kk) != 0 ? 1u : 0u;
            if constexpr (PAIR) tc_mma_bf16_pair(d_tmem, ad, bd, idesc, keep);
            else tc_mma_bf16(d_tmem, ad, bd, idesc, keep);
          }
          // frees the ring slot (of both CTAs) once read
          if constexpr (PAIR) tc_commit_pair(&empty[stage]);
          else tc_commit(&empty[stage]);
          if (++stage == n_stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        // accumulator ready for the epilogue (of both CTAs)
        if constexpr (PAIR) tc_commit_pair(&acc_full[acc]);
        else tc_commit(&acc_full[acc]);
        if (++acc == kAccBufs) {
          acc = 0;
          acc_phase ^= 1u;
        }
      }
      if (!ok) {
        *abort_v = 1;
        set_status(a.status, PCTREE_ERR_TIMEOUT);
      }
      // every MMA issued here must be complete before TMEM is released
      if constexpr (PAIR) tc_commit_pair(drain);
      else tc_commit(drain);
    }
    // (the odd CTA of a pair waits too: the last arrivals on its barriers have
    // landed before it may exit)
    if (lane == 0) {
      volatile int never = 0;
      mbar_wait_bounded(drain, 0, &never, 2 * kWaitLimitNs);
    }
  } else {
    if constexpr (FEW != 0) {
      few_rows<STREAM, FEW>(a, range, tmem_base, bars, acc_full, acc_empty, abort_v, stop_flag, slot);
    } else {
    // --------------------------------------------------------------- epilogue
    const int quad = warp & 3;               // TMEM lanes 32*quad .. +31
    const int half = (warp - 2) >> 2;        // tile columns 128*half .. +127
    const int trow = quad * 32 + lane;       // row of this CTA's 128
    const int row = row0 + trow;
    const bool live = row < a.rows;
    const bool warp_live = row0 + quad * 32 < a.rows;
    const int tid = threadIdx.x - 64;
    // (base logits are loaded before the wait below)
    const float* Lr = a.L + static_cast<long long>((live ? row : 0) / a.rows_per_req) *
                                a.l_req_stride;
    unsigned long long* gword = a.gthr + (live ? row : 0);
    const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
    // Base logits of 32 columns from v, in columns below v_end (no others are
    // used); loaded one chunk ahead.
    auto load_l = [&](int v, int v_end, float (&dst)[32]) {
      if (!live) return;
      if (a.l_vec && v + 32 <= v_end) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 f = __ldg(reinterpret_cast<const float4*>(Lr + v) + q);
          dst[4 * q] = f.x;
          dst[4 * q + 1] = f.y;
          dst[4 * q + 2] = f.z;
          dst[4 * q + 3] = f.w;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) dst[e] = v + e < v_end ? __ldg(Lr + v + e) : 0.0f;
      }
    };
    // columns [v, v_end) of tile i that this warp's half takes (whole chunks
    // of 32 for the first half), and the first one's accumulator column
    auto my_columns = [&](int i, int& v, int& v_end) {
      int t_lo, t_n;
      range.tile(i, t_lo, t_n);
      const int mid = ((t_n + 63) >> 6) << 5;
      v = t_lo + (half ? mid : 0);
      v_end = min(t_lo + (half ? t_n : min(mid, t_n)), a.V);
      return half ? mid : 0;
    };
    float lcur[32];
#pragma unroll
    for (int e = 0; e < 32; ++e) lcur[e] = 0.0f;
    // the base logits of this half's first chunk in tile i
    auto load_first = [&](int i) {
      if (i >= range.n) return;
      int v, v_end;
      my_columns(i, v, v_end);
      if (v < v_end) load_l(v, v_end, lcur);
    };
    RegList<KL> lst;
    lst.reset(a.k);
    // running sum of exp(z - R) of the row, R the largest logit so far
    float R = kNegInf, S = 0.0f;
    bool bad = false;
    load_first(0);
    if (EARLY) pdl_wait();
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int i = 0; i < range.n; ++i) {
      int v0, v_end;
      const int col0 = my_columns(i, v0, v_end);
      // the shared threshold, read past L1 while the tile is still computed
      float gl = kNegInf;
      if (live && i > 0) {
        const unsigned long long w = __ldcg(gword);
        if (static_cast<unsigned>(w >> 32) == a.tag) gl = key_float(static_cast<uint32_t>(w));
      }
      // the lanes agree before the warp-collective TMEM loads
      ok = __all_sync(kFull, mbar_wait_bounded(&acc_full[acc], acc_phase, abort_v, kWaitLimitNs));
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t kth_before = lst.kth();
      const uint32_t shared_before = gl > kNegInf ? float_key(gl) : 0u;
      bool held = true;                      // the accumulator buffer
      auto release = [&]() {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) mbar_arrive_cluster(mapa_shared(&acc_empty[acc], 0));
          else mbar_arrive(&acc_empty[acc]);
        }
        held = false;
      };
      if (warp_live) {
        // accumulators of the chunk at v plus its base logits; columns past
        // v_end give -inf
        auto chunk_logits = [&](int v, float (&z)[32]) {
          uint32_t r[32];
          tmem_ld_32x32b_x32(t_lane + static_cast<uint32_t>(acc * kBN + col0 + v - v0), r);
          tmem_ld_wait();
          const int nv = v_end - v;
          if (nv < 32) {
#pragma unroll
            for (int e = 0; e < 32; ++e) r[e] = e < nv ? r[e] : 0u;
          }
          // a Markov bias of -inf shows here; one that is NaN or +inf, and a
          // NaN or +inf base logit, in the logits (-inf base logits are
          // legal)
          float mn = kPosInf;
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float b = __uint_as_float(r[e]);
            mn = fminf(mn, b);
            z[e] = b + lcur[e];
          }
          bad |= mn == kNegInf;
          if (nv < 32) {
#pragma unroll
            for (int e = 0; e < 32; ++e) z[e] = e < nv ? z[e] : kNegInf;
          }
        };
        if (KL <= 16 && i == 0) {
          // A lower bound of the k-th best of the slot's first columns before
          // any list exists: the k-th best of 16 group maxima (each the best of
          // distinct columns).  Without it the empty lists take nearly every
          // logit of the first chunks (~60 insertions a row instead of ~15).
          float gm[16];
#pragma unroll
          for (int g = 0; g < 16; ++g) gm[g] = kNegInf;
#pragma unroll 1
          for (int v = v0; v < v_end; v += 32) {
            float z[32];
            chunk_logits(v, z);
            load_l(v + 32 < v_end ? v + 32 : v0, v_end, lcur);
#pragma unroll
            for (int g = 0; g < 16; ++g) gm[g] = fmaxf(gm[g], fmaxf(z[g], z[g + 16]));
          }
          sort16_desc(gm);
          float bound = kNegInf;
#pragma unroll
          for (int g = 0; g < 16; ++g) bound = g == a.k - 1 ? gm[g] : bound;
          gl = fmaxf(gl, bound);
        }
#pragma unroll 1
        for (int v = v0; v < v_end; v += 32) {
          float z[32];
          chunk_logits(v, z);
          if (v + 32 >= v_end) release();    // this warp's last TMEM read of the tile
          const int nv = min(32, v_end - v);
          // the next chunk's base logits
          if (v + 32 < v_end) load_l(v + 32, v_end, lcur);
          else load_first(i + 1);
          const float mc = max_of(z);
          bad |= !(mc < kPosInf);
          // log-sum-exp (Eq. 2)
          if (mc > R) {
            S *= exp_diff(R, mc);
            R = mc;
          }
          if (R > kNegInf) S += sum_exp(z, R);
          // top-k: logits that reach the list's last entry (any, while the list
          // is not full) and are not below the shared threshold.  On a forward
          // walk tokens rise, so an equal one stays out.
          const uint32_t kth = lst.kth();
          const float kf = kth != 0u ? key_float(kth) : kNegInf;
          uint32_t mk = 0;
          if (__any_sync(kFull, live && !(mc < gl) &&
                                    (!(mc <= kf) || (range.back() && mc == kf) || kth == 0u))) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              mk |= static_cast<uint32_t>((z[e] > kf) | (range.back() & (z[e] == kf))) << e;
            if (kth == 0u) mk = nv == 32 ? 0xffffffffu : (1u << nv) - 1u;
            if (gl > kNegInf) {
              uint32_t mg = 0;
#pragma unroll
              for (int e = 0; e < 32; ++e) mg |= static_cast<uint32_t>(z[e] >= gl) << e;
              mk &= mg;
            }
            if (!live) mk = 0;
            while (__any_sync(kFull, mk != 0)) {
              const int e = mk != 0 ? __ffs(mk) - 1 : 0;
              const float ze = pick(z, e);
              const uint32_t c = mk != 0 && ze == ze ? float_key(ze) : 0u;   // (not a NaN)
              mk &= mk - 1;
              if (range.back()) {
                if (__any_sync(kFull, c >= lst.kth() && c != 0u))
                  lst.insert(c, c != 0u ? v + e : kNoToken);
              } else {
                if (__any_sync(kFull, c > lst.kth())) lst.insert_later(c, v + e);
              }
            }
          }
        }
      }
      if (held) {                            // no column or no row of this tile
        release();
        load_first(i + 1);
      }
      // publish the row's k-th entry for the other slots
      if (live && lst.kth() > kth_before && lst.kth() > shared_before)
        atomicMax(gword, (static_cast<unsigned long long>(a.tag) << 32) | lst.kth());
      if (++acc == kAccBufs) {
        acc = 0;
        acc_phase ^= 1u;
      }
    }
    if (live && bad) set_status(a.status, PCTREE_ERR_NONFINITE);
    if (!ok && lane == 0) {
      *abort_v = 1;
      set_status(a.status, PCTREE_ERR_TIMEOUT);
    }
    // one decision for the eight warps, which meet at named barriers
    epi_barrier();
    if (tid == 0) *stop_flag = *abort_v;
    epi_barrier();
    if (!*stop_flag) {
      // The two halves of a row meet in the ring's memory: every accumulator
      // is complete, so no copy or MMA uses it any more.
      float* hm = reinterpret_cast<float*>(ring);              // [128] R, then S
      uint32_t* hk = reinterpret_cast<uint32_t*>(hm + 256);    // [KL][128] keys
      int* ht = reinterpret_cast<int*>(hk + KL * 128);         // [KL][128] tokens
      if (half == 1) {
        hm[trow] = R;
        hm[128 + trow] = S;
#pragma unroll
        for (int j = 0; j < KL; ++j) {
          hk[j * 128 + trow] = lst.key[j];
          ht[j * 128 + trow] = lst.tok[j];
        }
      }
      epi_barrier();
      if (half == 0 && warp_live) {
        const float R1 = hm[trow], S1 = hm[128 + trow];
        const float Rm = fmaxf(R, R1);
        if (Rm > kNegInf) {
          S = (R > kNegInf ? S * exp_diff(R, Rm) : 0.0f) +
              (R1 > kNegInf ? S1 * exp_diff(R1, Rm) : 0.0f);
          R = Rm;
        }
        lst.merge(a.k, [&](int j, uint32_t& c, int& t) {
          c = hk[j * 128 + trow];
          t = ht[j * 128 + trow];
        });
        if (live) {
          const size_t p = static_cast<size_t>(row) * a.n_slots + slot;
          a.part_m[p] = R;
          a.part_s[p] = S;
#pragma unroll
          for (int j = 0; j < KL; ++j) {
            const int o = j - (KL - a.k);
            if (o >= 0) {
              a.part_z[p * a.k + o] = lst.key[j] != 0u ? key_float(lst.key[j]) : kNegInf;
              a.part_t[p * a.k + o] = lst.tok[j];
            }
          }
        }
      }
    }
  }
  }

  tc_fence_before_sync();
  __syncthreads();
  // neither CTA of a pair exits while the other may still use its memory
  if constexpr (PAIR) cluster_sync();
  tc_fence_after_sync();
  if (warp == 1) {
    if constexpr (PAIR) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <int KL, bool PAIR, bool STREAM, int FEW = 0>
cudaError_t launch_kl(const ProjMaps& maps, const RowsArgs& a, cudaStream_t stream) {
  const size_t smem = 1024 + static_cast<size_t>(a.n_stages) * a.stage_bytes + kBarBytes + a.z_bytes;
  static SmemLimit limit;
  cudaError_t e = limit.ensure(reinterpret_cast<const void*>(markov_rows_kernel<KL, PAIR, STREAM, FEW>),
                               kSmemLimit);
  if (e != cudaSuccess) return e;
  // programmatic dependent launch: may be scheduled while the kernel before
  // it finishes (the kernel waits for it before touching memory)
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(a.n_slots * a.groups * (PAIR ? 2 : 1)));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = PAIR ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, markov_rows_kernel<KL, PAIR, STREAM, FEW>, maps.w,
                            maps.w_small, maps.x, a);
}

template <int KL>
cudaError_t launch_any(const ProjMaps& maps, const RowsArgs& a, bool pair, bool from_hbm,
                       cudaStream_t stream) {
  if constexpr (KL <= 16)
    if (from_hbm) return launch_kl<KL, false, true>(maps, a, stream);
  return pair ? launch_kl<KL, true, false>(maps, a, stream)
              : launch_kl<KL, false, false>(maps, a, stream);
}

}  // namespace

ProjPlan proj_plan(int V, int H, int rows, int num_sms) {
  ProjPlan p{};
  // a pair's 256 rows would be at most half used by 128
  p.pair = rows > 128;
  const int m = p.pair ? 256 : 128;
  p.groups = (rows + m - 1) / m;
  const int ctas = num_sms < kProjMaxSlots ? num_sms : kProjMaxSlots;
  p.slots = ctas / (p.pair ? 2 : 1) / p.groups;
  if (p.slots < 1) p.slots = 1;
  // The unit of the slots' ranges.  Pairs (MMA-bound): 64 entries, so that
  // slots differ by a quarter tile at most, 32 where a slot would get none.
  // Single CTAs: the unit with the least estimated time of the busiest slot:
  // per K chunk the larger of its W_out bytes at ~50 GB/s and its TMA boxes at
  // ~145 ns each (a coarse unit leaves slots uneven: 80000 entries in 128s give
  // some slots 5 blocks where 4.1 would do, 20 % of a stage; a fine one is box-
  // bound), then the epilogue's chunks of 2 x 32 columns.  Tiles are as few as
  // can be and equal, and the ring's slots hold just such a tile, so that as many
  // bytes are in flight as with tiles of 256 (us per round, slots for 256 and
  // boxes counted as if a tile started mid-block / so: 40000 x 2048 with 64 rows
  // 333 / 281, 45000 x 3072 with 128 452 / 418, 80000 x 4096 with one 548 / 500).
  int unit = 64;
  p.tile = kBN;
  if (p.pair) {
    if ((V + 63) / 64 < p.slots) unit = 32;
  } else {
    double best = 0.0;
    for (int u = 128; u >= 16; u /= 2) {
      const int n = (V + u - 1) / u;
      const int slots = p.slots < n ? p.slots : n;
      const int cols = (n + slots - 1) / slots * u;
      const int tiles = (cols + kBN - 1) / kBN;
      const int tile = (cols / u + tiles - 1) / tiles * u;
      // boxes of a tile, over the places it can start at in a 128-row block
      int boxes = 0;
      for (int in = 0; in < 128; in += u)
        for (int r = 0; r < tile; ++boxes) r += ((in + r) & 127) == 0 && tile - r >= 128 ? 128 : u;
      const double box_ns = 145.0 * tiles * (static_cast<double>(boxes) / (128 / u) + 1.0);
      const double chunk = 2.56 * cols > box_ns ? 2.56 * cols : box_ns;
      const double ns = (H + kBK - 1) / kBK * chunk + 700.0 * ((cols + 63) / 64);
      if (u == 128 || ns < best) {
        best = ns;
        unit = u;
        p.tile = tile;
      }
    }
  }
  p.unit = unit;
  p.small_box = p.pair ? unit / 2 : unit;
  const int units = (V + unit - 1) / unit;
  if (p.slots > units) p.slots = units;
  // Two 128-row blocks in nearly every slot: two tiles, so that the first's
  // epilogue runs under the second's stream (36808 x 2816, 78 rows: 412 -> 380
  // us a round; 32000 x 4096, where a third of the slots has one block and two
  // tiles only halve the others' loads in flight, 385 -> 398 and stays at one).
  const int most = (units + p.slots - 1) / p.slots * unit;
  if (!p.pair && unit == 128 && most == 2 * 128 && 8 * units >= 14 * p.slots) p.tile = 128;
  return p;
}

cudaError_t launch_markov_rows(const ProjMaps& maps, const ProjPlan& plan, const float* L,
                               long long l_req_stride, int V, int H, int k, int rows,
                               int rows_per_req, int x_box, int tiled, float* part_m,
                               float* part_s, float* part_z, int32_t* part_t,
                               unsigned long long* gthr, unsigned tag, int32_t* status,
                               cudaStream_t stream) {
  RowsArgs a{};
  a.L = L;
  a.l_req_stride = l_req_stride;
  a.V = V;
  a.H = H;
  a.k = k;
  a.rows = rows;
  a.rows_per_req = rows_per_req;
  a.x_box = x_box;
  a.groups = plan.groups;
  a.unit = plan.unit;
  a.small_box = plan.small_box;
  a.n_slots = plan.slots;
  a.tiled = tiled;
  a.l_vec = (reinterpret_cast<uintptr_t>(L) & 15u) == 0 && (l_req_stride & 3) == 0;
  a.part_m = part_m;
  a.part_s = part_s;
  a.part_z = part_z;
  a.part_t = part_t;
  a.gthr = gthr;
  a.tag = tag;
  a.status = status;
  // A warp to a row of logits: up to 16 rows, up to 32 where a thread's own list
  // would be long (us per round, a thread / a warp to a row: 32 rows of 12000 x
  // 512 with k 16 215 / 174, of 32000 x 2048 with k 12 294 / 255, of 150000 x 2560
  // with k 32 in 4 stages 718 / 684, of 2500 x 4096 with k 16 310 / 316; with k 8 of
  // 12000 x 512 137 / 137, of 80000 x 1024 267 / 287).
  const bool few = rows <= (k > 10 ? 32 : 16);
  // Where W_out comes from HBM every stage, stages alternate their direction; a
  // head that stays in L2 gains nothing from that, and a thread's list inserts
  // compare tokens too on a backward walk (us per round, without / with it and
  // early loads: 151936 x 2560, 8 rows, B 16 1945 / 1900; 151936 x 4096, 128 rows
  // 1327 / 1323; 60001 x 2048, 60 rows 359 / 364; lists of 32 768 / 807).
  const bool from_hbm =
      !plan.pair && (few || k <= 16) && static_cast<long long>(V) * H * 2 > kStreamBytes;
  a.tile = plan.tile;
  // A ring slot holds the largest tile's W rows.  At least 16 KB: the MMA reads
  // 128 rows of A from the slot's start, however few are loaded (the rest gives
  // accumulator rows that nobody reads).
  a.stage_bytes = x_box * kRowBytes + (plan.pair ? a.tile / 2 : a.tile) * kRowBytes;
  if (a.stage_bytes < 128 * kRowBytes) a.stage_bytes = 128 * kRowBytes;
  a.z_bytes = few ? rows * ((a.tile <= 128 ? 128 : 256) + 4) * 4 : 0;
  const int room = kSmemLimit - 1024 - kBarBytes - a.z_bytes;
  a.n_stages = room / a.stage_bytes < kMaxStages ? room / a.stage_bytes : kMaxStages;
  if (few) {
    if (rows <= 16)
      return from_hbm ? launch_kl<8, false, true, 2>(maps, a, stream)
                      : launch_kl<8, false, false, 2>(maps, a, stream);
    return from_hbm ? launch_kl<8, false, true, 4>(maps, a, stream)
                    : launch_kl<8, false, false, 4>(maps, a, stream);
  }
  if (k <= 8) return launch_any<8>(maps, a, plan.pair, from_hbm, stream);
  if (k <= 16) return launch_any<16>(maps, a, plan.pair, from_hbm, stream);
  return launch_any<32>(maps, a, plan.pair, from_hbm, stream);
}

}  // namespace pct
