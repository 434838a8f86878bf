// Ramp filter F of the filtered least-squares loss (Sec. 2):
//   L_FLS(z, y) = 1/2 (z - y)^T F (z - y),  dL/dz = F (z - y)   (Sec. 3, after Algorithm 1).
// F convolves every detector row (fixed view, and fixed detector row v for the
// cone) along the bin axis with the band-limited ramp (Ram-Lak) kernel of the
// textbook FBP, sampled at the bin pitch tau = du * (2/N) at the isocentre:
//   (F r)_b = tau * sum_k h[k] r_{b-k},  h[0] = 1/(4 tau^2),
//   h[k] = -1/(pi^2 k^2 tau^2) for odd k, 0 for even k != 0;
// bins outside the detector count as zero.  F is symmetric, so the same
// kernel gives the gradient.
#include <math.h>

#include <algorithm>

#include "filter.cuh"
#include "projector.cuh"

namespace inrct {

typedef unsigned long long f32x2;  // two FP32 values in one 64-bit register
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 dup2(float v) { return pack2(v, v); }
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// h[k] vanishes for even k != 0, so apart from h[0] the even bins depend on the odd bins only and the odd on the
// even: per row two Toeplitz products of half the length.  A thread computes the four even and four odd outputs
// 2 i0 .. 2 i0 + 7 of M = 2 rows; the inputs are kept in shared memory by parity, reversed (jr = n - 1 - j, so
// that the taps a thread needs rise with jr) and with the two rows side by side, so that a step of four inputs
// costs 2 tap loads of 16 bytes and 8 broadcast input loads of 8 for 64 multiply-adds, packed in pairs of rows.
// One thread per output with both neighbours loaded per tap, as before, was bound by its shared loads.
// 256^3 scan, 15,360 rows of 384 bins: the call takes 389 us before, 84 us now (the multiply-adds alone 28 us at
// the nominal rate; the three steps around a thread's own outputs read their inputs lane by lane).  Four rows per
// thread took 127 us (128 registers), blocks of 256 threads 96 us.
// gs[y] = h[|2 (y + 1 - n) - 1|]: the tap between even output i and odd input j is gs[i + jr], between odd output
// i and even input j gs[i + jr + 1].
constexpr int M = 2, kRampThreads = 128;
__global__ void __launch_bounds__(kRampThreads)
    ramp_kernel(const float* __restrict__ r, float* __restrict__ out, int A, int n, int64_t rows, int groups, float tau,
                double* __restrict__ loss_part) {
  extern __shared__ __align__(16) float sh[];
  float* gs = sh;              // [2 n]
  float* in = sh + 2 * n;      // [group][parity][jr][M]
  const float inv_t2 = 1.f / (tau * tau);
  for (int y = threadIdx.x; y < 2 * n; y += blockDim.x) {
    const int k = abs(2 * (y + 1 - n) - 1);
    gs[y] = -inv_t2 / (float)(M_PI * M_PI * (double)k * k);
  }
  const int64_t row0 = (int64_t)blockIdx.x * groups * M;
  for (int q = 0; q < groups * M; ++q) {
    const int64_t row = row0 + q;
    float* dst = in + (size_t)(q / M) * 2 * n * M + q % M;
    for (int b = threadIdx.x; b < 2 * n; b += blockDim.x)
      dst[((b & 1) * n + n - 1 - (b >> 1)) * M] = b < A && row < rows ? r[row * A + b] : 0.f;
  }
  __syncthreads();
  float lsum = 0.f;
  const int tiles = n / 4;
  const bool vec = A % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;  // rows 16-byte aligned
  for (int item = threadIdx.x; item < groups * tiles; item += blockDim.x) {
    const int grp = item / tiles, i0 = 4 * (item - grp * tiles);
    const float* ev = in + (size_t)grp * 2 * n * M;
    const float* od = ev + n * M;
    auto step = [&](int jr, f32x2 (&acc)[2][4]) {
      float t[8];
      *reinterpret_cast<float4*>(t) = *reinterpret_cast<const float4*>(gs + i0 + jr);
      *reinterpret_cast<float4*>(t + 4) = *reinterpret_cast<const float4*>(gs + i0 + jr + 4);
      f32x2 d[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) d[k] = dup2(t[k]);
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const f32x2 e = *reinterpret_cast<const f32x2*>(ev + (jr + jj) * M);
        const f32x2 o = *reinterpret_cast<const f32x2*>(od + (jr + jj) * M);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          fma2(acc[0][k], d[k + jj], o);
          fma2(acc[1][k], d[k + jj + 1], e);
        }
      }
    };
    // The far taps are small and sum by themselves; the three steps around the thread's own outputs start from the
    // h[0] term, which they mostly cancel, and the two sums meet at the end.  One running sum over all inputs would
    // round most of its additions at the size of h[0] r (3.3e-7 -> 1.1e-6 relative error on a smooth residual).
    f32x2 far[2][4], acc[2][4];
    const float h0 = 0.25f * inv_t2;
    const int own = n - 4 - i0;  // the step that holds the outputs' own places
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int k = 0; k < 4; ++k) far[p][k] = 0ull;
    for (int jr = 0; jr < n; jr += 4)
      if (abs(jr - own) > 4) step(jr, far);
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float* c = (p ? od : ev) + (own + 3 - k) * M;
        acc[p][k] = pack2(h0 * c[0], h0 * c[1]);
      }
    for (int jr = max(0, own - 4); jr <= min(n - 4, own + 4); jr += 4) step(jr, acc);
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int64_t row = row0 + grp * M + m;
      if (row < rows) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const f32x2 a2 = acc[p][k], f2 = far[p][k];
            v[2 * k + p] = (__uint_as_float((uint32_t)(m ? a2 >> 32 : a2)) +
                            __uint_as_float((uint32_t)(m ? f2 >> 32 : f2))) * tau;
            if (2 * (i0 + k) + p < A) lsum = fmaf((p ? od : ev)[(own + 3 - k) * M + m], v[2 * k + p], lsum);
          }
        float* dst = out + row * A + 2 * i0;
        if (vec && 2 * i0 + 8 <= A) {  // eight single stores 32 bytes apart across lanes would each cost a sector
          reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
          reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (2 * i0 + k < A) dst[k] = v[k];
        }
      }
    }
  }
  __shared__ float red[kRampThreads / 32];
  for (int o = 16; o; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lsum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    loss_part[blockIdx.x] = 0.5 * s;
  }
}

static int64_t ramp_rows(const inrct_geom* g) {
  return (int64_t)g->n_views * (g->kind == INRCT_CONE3D ? g->n_bins_v : 1);
}

size_t ramp_ws_bytes(const inrct_geom* geom) {
  return align_up(sizeof(double) * ramp_rows(geom), 256) + 256;
}

int ramp_filter_impl(const inrct_geom* geom, const inrct_grid* grid, const float* r, float* out,
                     double* loss_out, void* ws, size_t ws_bytes, cudaStream_t st) {
  INRCT_TRY(check_geom(geom, grid));
  INRCT_REQUIRE(r && out && loss_out, "r, out and loss_out must not be NULL");
  INRCT_REQUIRE(r != out, "ramp filter cannot run in place");
  INRCT_REQUIRE(geom->n_bins_u <= 6144, "ramp filter supports at most 6144 bins per row");
  const size_t need = ramp_ws_bytes(geom);
  if (!ws || ws_bytes < need) {
    set_error("ramp filter: workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  const int64_t rows = ramp_rows(geom);
  const int A = geom->n_bins_u;
  const float tau = (float)(geom->du * 2.0 / grid->N);
  double* part = static_cast<double*>(ws);
  const int n = (A + 7) / 8 * 4;  // inputs and outputs per parity, a multiple of 4
  // as many row groups per block as fill its threads
  const int groups = (int)std::min<int64_t>(std::max(1, kRampThreads / (n / 4)), ceil_div(rows, M));
  const size_t sm = sizeof(float) * (size_t)(2 * n) * (1 + groups * M);  // at most 74 KB (6144 bins)
  const unsigned blocks = ceil_div(rows, (int64_t)groups * M);
  const cudaError_t e = cudaFuncSetAttribute(ramp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) {
    set_error("ramp filter shared memory (%zu bytes): %s", sm, cudaGetErrorString(e));
    return INRCT_ERR_CUDA;
  }
  ramp_kernel<<<blocks, kRampThreads, sm, st>>>(r, out, A, n, rows, groups, tau, part);
  INRCT_CHECK_LAUNCH("ramp filter");
  return reduce_f64(part, blocks, loss_out, st);
}

}  // namespace inrct
