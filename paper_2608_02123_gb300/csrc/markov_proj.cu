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
// What bounds it: FFMA issue (128 FMA per clock and SM) once W_out sits in L2,
// as long as enough of W_out is on its way.  A CTA computes 128 vocabulary
// entries for up to 32 rows: 4 warps = RG row groups of 8 rows x 4 / RG
// vocabulary groups; a thread keeps 8 rows x RG entries (lane + 32 j) in
// registers and reads RG + 8 float4 (4 k each; the rows' are a broadcast) for
// 32 RG FMAs.  K chunks of 32 come with cp.async into three stages, rows
// padded to 36 words (float4 reads of 32 rows are conflict-free); rows beyond
// 32 are more CTAs (grid.y).  Sums run over ascending h, one FMA each.
// Measured (us per round, alternating runs; with the finer chunks of the partials
// pass): 32000 x 256 with 32 rows 846 -> 242; 65536 x 512 with 64 rows 2812 ->
// 501; 20000 x 512 with 8 rows 454 -> 196; 1024 x 64 with 4 rows 83 -> 49.
// One W word read per 8 FMAs and chunks loaded between barriers took 128 us a
// stage on the first; register-staged chunks one ahead 33; cp.async 26.
#include "pctree_common.cuh"
#include "sm103_ptx.cuh"

namespace pct {

namespace {

constexpr int kF32Threads = 128;
constexpr int kF32V = 128;        // vocabulary entries per CTA
constexpr int kF32K = 32;         // K chunk per stage
constexpr int kF32Ld = kF32K + 4; // row stride in shared memory, in words
constexpr int kF32Group = 8;      // rows per thread
constexpr int kF32Stages = 3;

template <int RG>
constexpr int kF32StageWords = (kF32V + RG * kF32Group) * kF32Ld;

// Asynchronous copies of 16 or 4 bytes to shared memory; `ok` false: zeros.
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
               "r"(ok ? 16 : 0)
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
__global__ void __launch_bounds__(kF32Threads)
markov_f32_kernel(const float* __restrict__ W, const float* __restrict__ X,
                  const float* __restrict__ L, long long l_req_stride,
                  float* __restrict__ Z, int ldz, int V, int H, int rows,
                  int rows_per_req, int32_t* status) {
  constexpr int kRows = RG * kF32Group;
  extern __shared__ __align__(16) float sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v0 = blockIdx.x * kF32V, r0 = blockIdx.y * kRows;
  const int rg = warp % RG;                               // this warp's row group
  const int vl = (warp / RG) * 32 * RG + lane;            // its first entry
  const int n_chunks = (H + kF32K - 1) / kF32K;
  // chunk c of W (128 rows) and X (kRows rows) into its stage; sources of
  // rows and columns out of range are not read
  auto load = [&](int c) {
    float* ws = sm + (c % kF32Stages) * kF32StageWords<RG>;
    float* xs = ws + kF32V * kF32Ld;
    const int h0 = c * kF32K;
    if constexpr (VEC) {
      const int q = (lane & 7) * 4, h = h0 + q;           // 8 lanes to a row
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int vr = warp * 32 + i * 4 + (lane >> 3);
        const bool ok = v0 + vr < V && h < H;
        cp_async16(ws + vr * kF32Ld + q, ok ? W + static_cast<size_t>(v0 + vr) * H + h : W, ok);
      }
#pragma unroll
      for (int i = 0; i < (kRows + 15) / 16; ++i) {
        const int xr = i * 16 + (threadIdx.x >> 3);
        const bool ok = r0 + xr < rows && h < H;
        if (xr < kRows)
          cp_async16(xs + xr * kF32Ld + q, ok ? X + static_cast<size_t>(r0 + xr) * H + h : X, ok);
      }
    } else {
      const int h = h0 + lane;                            // 32 lanes to a row
#pragma unroll 8
      for (int i = 0; i < 32; ++i) {
        const int vr = warp * 32 + i;
        const bool ok = v0 + vr < V && h < H;
        cp_async4(ws + vr * kF32Ld + lane, ok ? W + static_cast<size_t>(v0 + vr) * H + h : W, ok);
      }
#pragma unroll
      for (int i = 0; i < kRows / 4; ++i) {
        const int xr = i * 4 + warp;
        const bool ok = r0 + xr < rows && h < H;
        cp_async4(xs + xr * kF32Ld + lane, ok ? X + static_cast<size_t>(r0 + xr) * H + h : X, ok);
      }
    }
  };
  float acc[kF32Group][RG];
#pragma unroll
  for (int g = 0; g < kF32Group; ++g)
#pragma unroll
    for (int j = 0; j < RG; ++j) acc[g][j] = 0.0f;
  // launched while the kernel before it finishes: X is its output
  pdl_wait();
#pragma unroll
  for (int c = 0; c < kF32Stages - 1; ++c) {
    if (c < n_chunks) load(c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int c = 0; c < n_chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kF32Stages - 2) : "memory");
    __syncthreads();                   // chunk c is here; chunk c - 1 has been read
    if (c + kF32Stages - 1 < n_chunks) load(c + kF32Stages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* ws = sm + (c % kF32Stages) * kF32StageWords<RG> + vl * kF32Ld;
    const float* xs = sm + (c % kF32Stages) * kF32StageWords<RG> +
                      (kF32V + rg * kF32Group) * kF32Ld;
#pragma unroll 2
    for (int q = 0; q < kF32K; q += 4) {
      float4 w[RG], x[kF32Group];
#pragma unroll
      for (int j = 0; j < RG; ++j)
        w[j] = *reinterpret_cast<const float4*>(ws + 32 * j * kF32Ld + q);
#pragma unroll
      for (int g = 0; g < kF32Group; ++g)
        x[g] = *reinterpret_cast<const float4*>(xs + g * kF32Ld + q);
#pragma unroll
      for (int g = 0; g < kF32Group; ++g)
#pragma unroll
        for (int j = 0; j < RG; ++j) {
          acc[g][j] = fmaf(w[j].x, x[g].x, acc[g][j]);
          acc[g][j] = fmaf(w[j].y, x[g].y, acc[g][j]);
          acc[g][j] = fmaf(w[j].z, x[g].z, acc[g][j]);
          acc[g][j] = fmaf(w[j].w, x[g].w, acc[g][j]);
        }
    }
  }
  // (not earlier: CTAs of later kernels that become resident beside a running
  // grid leave uneven room for the next projection's)
  pdl_launch_dependents();
  bool bad = false;
#pragma unroll
  for (int g = 0; g < kF32Group; ++g) {
    const int row = r0 + rg * kF32Group + g;
    if (row >= rows) break;
    const float* Lr = L + static_cast<long long>(row / rows_per_req) * l_req_stride;
#pragma unroll
    for (int j = 0; j < RG; ++j) {
      const int v = v0 + vl + 32 * j;
      if (v < V) {
        const float lval = Lr[v];
        const float z = lval + acc[g][j];
        bad |= isnan(z) || (isinf(z) && !(isinf(lval) && lval < 0.0f));
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
                              int rows_per_req, int32_t* status,
                              cudaStream_t stream) {
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
    cfg.dynamicSmemBytes = static_cast<size_t>(words) * kF32Stages * sizeof(float);
    const cudaError_t e =
        limit.ensure(reinterpret_cast<const void*>(kernel), cfg.dynamicSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, kernel, W_out, X, L, l_req_stride, Z, ldz, V, H, rows,
                              rows_per_req, status);
  };
  if (H % 4 == 0) {
    if (rg == 1) return go(markov_f32_kernel<1, true>, kF32StageWords<1>, limits[0]);
    if (rg == 2) return go(markov_f32_kernel<2, true>, kF32StageWords<2>, limits[1]);
    return go(markov_f32_kernel<4, true>, kF32StageWords<4>, limits[2]);
  }
  if (rg == 1) return go(markov_f32_kernel<1, false>, kF32StageWords<1>, limits[3]);
  if (rg == 2) return go(markov_f32_kernel<2, false>, kF32StageWords<2>, limits[4]);
  return go(markov_f32_kernel<4, false>, kF32StageWords<4>, limits[5]);
}

}  // namespace pct
