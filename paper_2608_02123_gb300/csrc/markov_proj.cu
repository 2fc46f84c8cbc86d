// Markov projection of one PCTree stage (Eq. 3) for float32 heads:
//
//   Z[row][v] = L_d[req(row)][v] + sum_h W_out[v][h] * X[row][h]
//
// where X[row] = E_in[parent token of row] (gathered by the previous stage),
// so that sum_h W_out[v][h] X[row][h] is the Markov head's bias for that
// parent.  A CUDA-core kernel with float32 accumulation in ascending h
// (tensor cores would round float32 inputs to tf32); the stage logits Z go to
// the workspace and partials_kernel reduces them.  bf16 heads take
// markov_rows.cu, which never writes Z.
//
// What bounds it: the issue of FMAs and of what feeds them, once W_out sits in
// L2 and enough of it is on its way.  A CTA computes 128 vocabulary entries for
// up to 32 rows with two sets of 4 warps = RG row groups of 8 rows x 4 / RG
// vocabulary groups; each set takes half of every K chunk (one set leaves an SM
// 4 to 8 warps, too few to cover shared-memory latency).  A thread keeps 8 rows x
// RG entries (lane + 32 j) in registers as pairs of sums over even and odd k and
// reads RG + 8 float4 (4 k each; the rows' are a broadcast) for 16 RG packed
// FMAs.  K chunks of 32 come with cp.async into three stages, rows padded to 36
// words (float4 reads of 32 rows are conflict-free); rows beyond 32 are more
// CTAs (grid.y).  The first W_out chunks and the base logits load while the
// merge before the stage still runs.  The four sums of a logit run over ascending
// h, one FMA each, and are added at the end.
// Measured (us per round, alternating runs): 32000 x 256 with 32 rows 232 ->
// 210, 65536 x 512 with 64 rows 925 -> 876, 20000 x 512 with 8 rows 220 -> 189,
// 50257 x 770 with 12 rows 459 -> 409, 4096 x 128 with 64 rows 106 -> 79, 1024 x
// 64 with 4 rows 47 -> 41 against one set of warps with scalar FMAs and loads
// behind the wait; that was 846 -> 242 on the first against chunks loaded
// between barriers.
#include "pctree_common.cuh"
#include "sm103_ptx.cuh"

namespace pct {

namespace {

constexpr int kF32Threads = 256;
constexpr int kF32V = 128;        // vocabulary entries per CTA
constexpr int kF32K = 32;         // K chunk per stage
constexpr int kF32Ld = kF32K + 4; // row stride in shared memory, in words
constexpr int kF32Group = 8;      // rows per thread
constexpr int kF32Stages = 3;

template <int RG>
constexpr int kF32StageWords = (kF32V + RG * kF32Group) * kF32Ld;
// the stages, then the tile's base logits
template <int RG>
constexpr int kF32Words = kF32Stages * kF32StageWords<RG> + RG * kF32Group * kF32V;

// Asynchronous copies of 16 or 4 bytes to shared memory, of which the first
// `bytes` are read and the others zeros; `ok` false: all zeros.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(ok ? 4 : 0)
               : "memory");
}

// RG: row groups of 8 (1, 2 or 4); VEC: H % 4 == 0 (rows on 16-byte
// boundaries: 16-byte copies).
template <int RG, bool VEC>
__global__ void __launch_bounds__(kF32Threads, 2)
markov_f32_kernel(const float* __restrict__ W, const float* __restrict__ X,
                  const float* __restrict__ L, long long l_req_stride,
                  float* __restrict__ Z, int ldz, int V, int H, int rows,
                  int rows_per_req, int l_vec, int first, int32_t* status) {
  constexpr int kRows = RG * kF32Group;
  extern __shared__ __align__(16) float sm[];
  float* ls = sm + kF32Stages * kF32StageWords<RG>;       // [kRows][kF32V]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v0 = blockIdx.x * kF32V, r0 = blockIdx.y * kRows;
  const int half = warp >> 2;                             // its 16 of a chunk's 32 k
  const int rg = (warp & 3) % RG;                         // this warp's row group
  const int vl = (warp & 3) / RG * 32 * RG + lane;        // its first entry
  const int n_chunks = (H + kF32K - 1) / kF32K;
  // Chunk c of W (128 rows) and X (kRows rows) into its stage.  A thread copies
  // the same columns of the same rows of every chunk: rows and columns
  // out of range are not read (zeros), and their source is a place in range.
  constexpr int kWCopies = VEC ? 4 : 16, kXCopies = VEC ? 1 : RG;
  const int w_row = VEC ? warp * 16 + (lane >> 3) : warp * 16;
  const int x_row = VEC ? threadIdx.x >> 3 : warp;
  const int col = VEC ? (lane & 7) * 4 : lane;           // 8 or 32 lanes to a row
  constexpr int kWStep = VEC ? 4 : 1, kXStep = 8;
  const int w_live = min(kF32V, V - v0), x_live = min(kRows, rows - r0);
  const float* wp = W + static_cast<size_t>(v0) * H + (col < H ? col : 0);
  const float* xp = X + static_cast<size_t>(r0) * H + (col < H ? col : 0);
  auto copy = [&](float* dst, const float* src, bool ok) {
    if constexpr (VEC) cp_async16(dst, src, ok ? 16 : 0);
    else cp_async4(dst, src, ok);
  };
  auto load_w = [&](int c, int slot) {
    float* ws = sm + slot * kF32StageWords<RG> + w_row * kF32Ld + col;
    const bool in = c * kF32K + col < H;
    const float* src = wp + (in ? c * kF32K : 0);
#pragma unroll 4
    for (int i = 0; i < kWCopies; ++i) {
      const int vr = w_row + i * kWStep;
      copy(ws + i * kWStep * kF32Ld, src + static_cast<size_t>(min(vr, w_live - 1)) * H,
           in && vr < w_live);
    }
  };
  auto load_x = [&](int c, int slot) {
    float* xs = sm + slot * kF32StageWords<RG> + (kF32V + x_row) * kF32Ld + col;
    const bool in = c * kF32K + col < H;
    const float* src = xp + (in ? c * kF32K : 0);
    if (VEC && x_row >= kRows) return;
#pragma unroll
    for (int i = 0; i < kXCopies; ++i) {
      const int xr = x_row + i * kXStep;
      copy(xs + i * kXStep * kF32Ld, src + static_cast<size_t>(min(xr, x_live - 1)) * H,
           in && xr < x_live);
    }
  };
  // launched while the kernels before it finish.  X is the previous stage's
  // output; W and the base logits are the round's inputs, and any stage but the
  // first knows them complete (its predecessors started after them).
  if (first) pdl_wait();
#pragma unroll
  for (int c = 0; c < kF32Stages - 1; ++c)
    if (c < n_chunks) load_w(c, c);
  if (l_vec) {
#pragma unroll
    for (int i = 0; i < kRows * kF32V / 4 / kF32Threads; ++i) {
      const int rl = i * (kF32Threads / 32) + warp, left = V - (v0 + 4 * lane);
      const bool ok = rl < x_live && left > 0;
      cp_async16(ls + rl * kF32V + 4 * lane,
                 ok ? L + static_cast<long long>((r0 + rl) / rows_per_req) * l_req_stride + v0 +
                          4 * lane
                    : L,
                 ok ? 4 * min(4, left) : 0);
    }
  } else {
#pragma unroll 1
    for (int rl = warp; rl < x_live; rl += kF32Threads / 32) {
      const float* Lr = L + static_cast<long long>((r0 + rl) / rows_per_req) * l_req_stride + v0;
#pragma unroll
      for (int i = lane; i < kF32V; i += 32)
        cp_async4(ls + rl * kF32V + i, i < w_live ? Lr + i : L, i < w_live);
    }
  }
  if (!first) pdl_wait();
#pragma unroll
  for (int c = 0; c < kF32Stages - 1; ++c) {
    if (c < n_chunks) load_x(c, c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  uint64_t acc[kF32Group][RG];         // sums over even and odd k
#pragma unroll
  for (int g = 0; g < kF32Group; ++g)
#pragma unroll
    for (int j = 0; j < RG; ++j) acc[g][j] = 0ull;
  int slot = 0;                        // c % kF32Stages
  for (int c = 0; c < n_chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kF32Stages - 2) : "memory");
    __syncthreads();                   // chunk c is here; chunk c - 1 has been read
    if (c + kF32Stages - 1 < n_chunks) {
      const int next = slot == 0 ? kF32Stages - 1 : slot - 1;
      load_w(c + kF32Stages - 1, next);
      load_x(c + kF32Stages - 1, next);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* ws = sm + slot * kF32StageWords<RG> + vl * kF32Ld + half * 16;
    const float* xs = sm + slot * kF32StageWords<RG> + (kF32V + rg * kF32Group) * kF32Ld + half * 16;
    slot = slot + 1 == kF32Stages ? 0 : slot + 1;
#pragma unroll
    for (int q = 0; q < 16; q += 4) {
      ulonglong2 w[RG];
#pragma unroll
      for (int j = 0; j < RG; ++j)
        w[j] = *reinterpret_cast<const ulonglong2*>(ws + 32 * j * kF32Ld + q);
#pragma unroll
      for (int g = 0; g < kF32Group; ++g) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(xs + g * kF32Ld + q);
#pragma unroll
        for (int j = 0; j < RG; ++j) {
          acc[g][j] = fma2(w[j].x, x.x, acc[g][j]);
          acc[g][j] = fma2(w[j].y, x.y, acc[g][j]);
        }
      }
    }
  }
  // (not earlier: CTAs of later kernels that become resident beside a running
  // grid leave uneven room for the next projection's)
  pdl_launch_dependents();
  // each half hands the other the sums of four of its eight rows
  __syncthreads();                     // the last chunk has been read
  float* mine = sm + (half * 4 + (warp & 3)) * 32 * (kF32Group / 2 * RG) + lane;
  float* other = sm + ((half ^ 1) * 4 + (warp & 3)) * 32 * (kF32Group / 2 * RG) + lane;
  float sum[kF32Group / 2][RG];
#pragma unroll
  for (int g = 0; g < kF32Group; ++g)
#pragma unroll
    for (int j = 0; j < RG; ++j) {
      float lo, hi;
      unpack2(acc[g][j], lo, hi);
      // (both halves' registers are indexed by constants)
      if ((g >= kF32Group / 2) == (half == 1))
        sum[g % (kF32Group / 2)][j] = lo + hi;
      else
        other[32 * (g % (kF32Group / 2) * RG + j)] = lo + hi;
    }
  __syncthreads();
  bool bad = false;
#pragma unroll
  for (int g = 0; g < kF32Group / 2; ++g) {
    const int rl = rg * kF32Group + half * (kF32Group / 2) + g, row = r0 + rl;
    if (row >= rows) break;
#pragma unroll
    for (int j = 0; j < RG; ++j) {
      const int v = v0 + vl + 32 * j;
      if (v < V) {
        const float lval = ls[rl * kF32V + vl + 32 * j];
        const float z = lval + (sum[g][j] + mine[32 * (g * RG + j)]);
        bad |= !(fabsf(z) < INFINITY) && !(lval == -INFINITY && z == z);
        Z[static_cast<size_t>(row) * ldz + v] = z;
      }
    }
  }
  if (bad) set_status(status, PCTREE_ERR_NONFINITE);
}

}  // namespace

cudaError_t launch_markov_f32(const float* W_out, const float* X,
                              const float* L, long long l_req_stride, float* Z,
                              int ldz, int V, int H, int rows,
                              int rows_per_req, int stage, int32_t* status,
                              cudaStream_t stream) {
  const int l_vec = (reinterpret_cast<uintptr_t>(L) & 15u) == 0 && (l_req_stride & 3) == 0;
  const int rg = rows <= 8 ? 1 : rows <= 16 ? 2 : 4;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((V + kF32V - 1) / kF32V, (rows + 8 * rg - 1) / (8 * rg));
  cfg.blockDim = dim3(kF32Threads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static SmemLimit limits[6];
  auto go = [&](auto kernel, int words, SmemLimit& limit) {
    cfg.dynamicSmemBytes = static_cast<size_t>(words) * sizeof(float);
    const cudaError_t e =
        limit.ensure(reinterpret_cast<const void*>(kernel), cfg.dynamicSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, kernel, W_out, X, L, l_req_stride, Z, ldz, V, H, rows,
                              rows_per_req, l_vec, stage == 0 ? 1 : 0, status);
  };
  if (H % 4 == 0) {
    if (rg == 1) return go(markov_f32_kernel<1, true>, kF32Words<1>, limits[0]);
    if (rg == 2) return go(markov_f32_kernel<2, true>, kF32Words<2>, limits[1]);
    return go(markov_f32_kernel<4, true>, kF32Words<4>, limits[2]);
  }
  if (rg == 1) return go(markov_f32_kernel<1, false>, kF32Words<1>, limits[3]);
  if (rg == 2) return go(markov_f32_kernel<2, false>, kF32Words<2>, limits[4]);
  return go(markov_f32_kernel<4, false>, kF32Words<4>, limits[5]);
}

}  // namespace pct
