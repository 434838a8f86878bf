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
#include <type_traits>

#include "filter.cuh"
#include "projector.cuh"

namespace inrct {

typedef unsigned long long f32x2;  // two FP32 values in one 64-bit register
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// h[k] vanishes for even k != 0, so apart from h[0] an output depends on the bins of the other parity only:
//   out[b] = tau (h[0] r[b] + sum over odd k of h[k] (r[b - k] + r[b + k])),
// summed outwards from b, so that the large terms, which cancel on smooth residuals, meet first (one running sum
// over the row instead rounds most additions at the size of h[0] r: error 3.3e-7 -> 1.1e-6).  A thread takes four
// neighbouring outputs of one parity (bins 2 (i0 + q) + p) of two rows, the rows packed.  Its two windows of
// neighbours move outwards by one bin of the other parity per k, so four k cost two blocks of four bins and
// four taps from shared memory, 16 packed additions and 16 packed multiply-adds.  The kernel this replaced loaded
// two neighbours and a tap per output and k.  256^3 scan, 15,360 rows of 384 bins: the call takes 389 us before,
// 115 us now, with the same bits (148 with warps of mixed parities; 84 without the order of the sums,
// which the half-precision networks' FLS steps would pass on to their roundings).
// Shared memory: [group][parity][half][block] of 16 bytes: bins 4 block + 2 half, + 1 of that parity, each the two
// rows' values side by side (lanes take neighbouring blocks: no bank conflicts), then the taps, then the results.
constexpr int kRampThreads = 384;
// FULL: kRampThreads threads, and rows as long as that.  Loops over rows one after the other then (98 us for 15,360 rows
// of 384 bins, 104 with the loops that also take rows side by side).
template <bool FULL>
__global__ void __launch_bounds__(kRampThreads)
    ramp_kernel(const float* __restrict__ r, float* __restrict__ out, int A, int n, int64_t rows, int groups, float tau,
                double* __restrict__ loss_part) {
  extern __shared__ __align__(16) float sh[];
  const int nb = n / 4;                      // blocks of four bins per parity
  float* in = sh;                            // groups x 2 parities x 2 halves x nb x 4
  float* h = in + (size_t)groups * 16 * nb;  // h[2 m + 1], m < n
  float* res = h + n;                        // [2 groups rows][2 n]
  const float inv_t2 = 1.f / (tau * tau);
  for (int m = threadIdx.x; m < n; m += blockDim.x) {
    const int k = 2 * m + 1;
    h[m] = -inv_t2 / (float)(M_PI * M_PI * (double)k * k);
  }
  const int64_t row0 = (int64_t)blockIdx.x * groups * 2;
  auto put = [&](int q, int b) {
    const int64_t row = row0 + q;
    const int i = b >> 1;
    in[((((q >> 1) * 2 + (b & 1)) * 2 + ((i >> 1) & 1)) * nb + (i >> 2)) * 4 + (i & 1) * 2 + (q & 1)] =
        b < A && row < rows ? r[row * A + b] : 0.f;
  };
  // not FULL: threads per row, whole warps, and rows side by side, so that the block's loads are in flight together
  const int tw = min((int)blockDim.x, (2 * n + 31) & ~31), side = blockDim.x / tw;
  const int qt = threadIdx.x / tw < side ? threadIdx.x / tw : groups * 2, bt = threadIdx.x % tw;
  if constexpr (FULL) {
    for (int q = 0; q < groups * 2; ++q)
      for (int b = threadIdx.x; b < 2 * n; b += blockDim.x) put(q, b);
  } else {
    for (int q = qt; q < groups * 2; q += side)
      for (int b = bt; b < 2 * n; b += tw) put(q, b);
  }
  __syncthreads();
  float lsum = 0.f;
  const int half = (nb + 1) / 2;
  // Segments of whole warps: left halves of the even outputs, of the odd, then the right halves: a warp's outputs
  // have one parity and run out of neighbours on the same side.
  const int seg = (groups * half + 31) & ~31;
  for (int item = threadIdx.x; item < 4 * seg; item += blockDim.x) {
    const int sg = item / seg, idx = item - sg * seg, p = sg & 1;
    const bool right = sg >= 2;
    const int grp = idx / half, t = idx - grp * half + (right ? half : 0), gp = 2 * grp + p, i0 = 4 * t;
    if (grp >= groups || t >= nb) continue;
    const ulonglong2* own = reinterpret_cast<const ulonglong2*>(in) + (size_t)gp * 2 * nb;
    const ulonglong2* oth = reinterpret_cast<const ulonglong2*>(in) + (size_t)(gp ^ 1) * 2 * nb;
    auto block = [&](int bl, f32x2* x) {
      const bool ok = (unsigned)bl < (unsigned)nb;
      const ulonglong2 none = make_ulonglong2(0ull, 0ull);
      *reinterpret_cast<ulonglong2*>(x) = ok ? oth[bl] : none;
      *reinterpret_cast<ulonglong2*>(x + 2) = ok ? oth[nb + bl] : none;
    };
    f32x2 x0[4], acc[4];
    *reinterpret_cast<ulonglong2*>(x0) = own[t];
    *reinterpret_cast<ulonglong2*>(x0 + 2) = own[nb + t];
    const float h0 = 0.25f * inv_t2;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float u, v;
      unpack2(x0[q], u, v);
      acc[q] = pack2(h0 * u, h0 * v);
    }
    // windows of eight bins of the other parity: lw[e] = bin i0 - m4 - 4 + e, rw[e] = bin i0 + m4 + e; output q takes
    // for k = 2 (m4 + s) + 1 the bins i0 + q - (m4 + s) - 1 + p and i0 + q + (m4 + s) + p
    f32x2 lw[8], rw[8];
    block(t, lw + 4);
    block(t, rw);
    auto outwards = [&](auto pc) {
      constexpr int po = decltype(pc)::value;
      // four k on both sides, or past the nearer end of the row on the farther side only (the other adds zeros)
      auto step = [&](int s4, auto left, auto rght) {
        constexpr bool kL = decltype(left)::value, kR = decltype(rght)::value;
        if (kL) block(t - s4 - 1, lw);
        if (kR) block(t + s4 + 1, rw + 4);
        const float4 hv = *reinterpret_cast<const float4*>(h + 4 * s4);
        const float hs[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const f32x2 hk = pack2(hs[s], hs[s]);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const f32x2 l = lw[q - s + 3 + po], x = rw[q + s + po];
            fma2(acc[q], hk, kL && kR ? add2(l, x) : kL ? l : x);
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (kL) lw[4 + e] = lw[e];
          if (kR) rw[e] = rw[4 + e];
        }
      };
      for (int s4 = 0; s4 < half; ++s4) step(s4, std::true_type{}, std::true_type{});
      if (right)
        for (int s4 = half; s4 < t + 1; ++s4) step(s4, std::true_type{}, std::false_type{});
      else
        for (int s4 = half; s4 < nb - t; ++s4) step(s4, std::false_type{}, std::true_type{});
    };
    if (p) outwards(std::integral_constant<int, 1>{});
    else outwards(std::integral_constant<int, 0>{});
    auto finish = [&](auto inside) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int b = 2 * (i0 + q) + p;
        float v[2], x[2];
        unpack2(acc[q], v[0], v[1]);
        unpack2(x0[q], x[0], x[1]);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          res[(size_t)(2 * grp + m) * 2 * n + b] = v[m] * tau;
          // past the row 0 times an infinite sum would be NaN
          if (decltype(inside)::value || b < A) lsum = fmaf(x[m], v[m] * tau, lsum);
        }
      }
    };
    if (2 * i0 + 8 <= A) finish(std::true_type{});
    else finish(std::false_type{});
  }
  __syncthreads();
  if constexpr (FULL) {
    for (int q = 0; q < groups * 2; ++q)
      if (row0 + q < rows)
        for (int b = threadIdx.x; b < A; b += blockDim.x) out[(row0 + q) * A + b] = res[(size_t)q * 2 * n + b];
  } else {
    for (int q = qt; q < groups * 2; q += side)
      if (row0 + q < rows)
        for (int b = bt; b < A; b += tw) out[(row0 + q) * A + b] = res[(size_t)q * 2 * n + b];
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
  const int n = (A + 7) / 8 * 4;  // bins per parity, a multiple of 4
  // As many row pairs per block as fill its threads, but no more than leave two blocks per SM of a 152-SM GPU; a block
  // of one or few short pairs is as small as its work.  (Filled blocks whose rows were loaded one after the other took
  // 70 us for 180 rows of 16 bins and 19 us for 60 rows of 183; 8 and 10 us now.)
  const int half = (n / 4 + 1) / 2;
  const int64_t pairs = ceil_div(rows, 2);
  const int groups = (int)std::max<int64_t>(1, std::min<int64_t>(kRampThreads / 4 / half, ceil_div(pairs, 2 * 152)));
  const int threads = std::min(kRampThreads, 4 * ((groups * half + 31) & ~31));
  const size_t sm = sizeof(float) * ((size_t)groups * 8 * n + n);  // at most 111 KB (6144 bins)
  const unsigned blocks = ceil_div(pairs, groups);
  const bool full = threads == kRampThreads && 2 * n > kRampThreads - 32;
  const auto kernel = full ? ramp_kernel<true> : ramp_kernel<false>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) {
    set_error("ramp filter shared memory (%zu bytes): %s", sm, cudaGetErrorString(e));
    return INRCT_ERR_CUDA;
  }
  kernel<<<blocks, threads, sm, st>>>(r, out, A, n, rows, groups, tau, part);
  INRCT_CHECK_LAUNCH("ramp filter");
  return reduce_f64(part, blocks, loss_out, st);
}

}  // namespace inrct
