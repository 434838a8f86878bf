// Joseph ray-driven projector P and its exactly matched adjoint P^T on sm_103a.
//
// The paper factorises the projection as z = P E{f} with a discrete projector
// P in R^{m x n} and needs v = P^T r (Sec. 3; Algorithm 1).  The
// model implemented here is Joseph's: a ray picks the grid axis along which it
// advances fastest (the driving axis), crosses every slice of that axis, and
// linearly (2-D) or bilinearly (3-D) interpolates the image at the crossing,
// with zero outside the grid; the sum is scaled by the path length per slice.
//
// Arithmetic layout
// -----------------
// * Per-ray constants are computed once per call in FP64 by a table kernel
//   (driving axis, crossing at the middle slice, slope, step length); the
//   crossing is then carried in 32.32 fixed point and stepped by exact integer
//   addition (see the table section), so its error stays near 1e-7 pixel.
// * Across the driving axis P and the gather-form adjoint evaluate the
//   crossing with the same integer operations and convert it to weights with
//   the same FP32 operations, so in 2-D P^T is the transpose of P up to the
//   FP32 summation order only.  Along z (cone) the kernels differ by rounding:
//   the column projector rounds a row's z pitch at a slice to 2^-32 voxel and
//   the tile adjoint forms row distances in FP32 from an exact reference row.
//   Both are closer to the FP64 operator than the kernels that step z in fixed
//   point (figures at the kernels), and <P x, y> and <x, P^T y> agree to FP32
//   rounding (501^3: 5e-8).
// * Forward: neighbouring rays cross neighbouring pixels of the same slice, so
//   warp loads coalesce.  2-D and the cone's other plans: blocks of 32 rays x
//   SEG segments of each ray, rays driven along x reading a transposed copy of
//   the image so that their two taps are also contiguous.  Cone: detector
//   columns over a z-fastest copy, or row patches.
// * Adjoint: gather form (2-D: tiles of pixels, cone: tiles, columns or chunks
//   of voxels).  Every pixel enumerates, view by view, the few detector bins
//   whose rays can reach it, recomputes their weights from the same ray table
//   and sums locally: deterministic, no atomics.
#include <math.h>

#include <algorithm>
#include <map>
#include <vector>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "common.cuh"
#include "projector.cuh"

namespace inrct {

// ---------------------------------------------------------------------------
// ray tables (FP64 set-up, fixed-point result)
//
// Crossings are carried in 32.32 fixed point: U = round(u * 2^32) in an int64,
// where u is the fractional transverse index.  Along a ray u is affine in the
// slice index j, u(j) = U0 + (j - jref) * S with jref = N/2, so the forward
// kernel steps it by integer addition and the adjoint evaluates the same
// integer expression directly: both get the same bits, with a position error
// of about 1e-7 pixel (instead of ~1e-5 for an FP32 crossing at N = 512).
// The interpolation weights are f = (low 32 bits) * 2^-32 and 1 - f in FP32.
// ---------------------------------------------------------------------------
constexpr double kFx32 = 4294967296.0;         // 2^32
constexpr double kFx30 = 1073741824.0;         // 2^30 (slopes, |slope| <= 1)
constexpr double kFx48 = 281474976710656.0;    // 2^48 (cone z-slope coefficient)

__device__ __forceinline__ bool drive_x(double ex, double ey) {
  // x drives unless |e_y| exceeds |e_x| by more than a relative 1e-12
  return !(fabs(ey) > fabs(ex) * (1.0 + 1e-12));
}

__device__ __forceinline__ int4 pack_ray(double uref, double slope, float scale_signed) {
  const long long U0 = __double2ll_rn(uref * kFx32);
  const int S = (int)__double2ll_rn(slope * kFx30);
  return make_int4((int)(unsigned)(U0 & 0xffffffffll), (int)(U0 >> 32), S,
                   __float_as_int(scale_signed));
}

__device__ __forceinline__ int64_t ray_U0(const int4& t) {
  return ((int64_t)t.y << 32) | (int64_t)(uint32_t)t.x;
}

// The tables of a geometry persist in the workspace between calls.  A block of the table launch owns the entries of
// kTabViews views x kTabBins bins (columns), each of its warps those of one view and one 64-bit checksum of them, seeded
// with a fingerprint of the geometry: entries that are still what a block of this geometry left behind are kept, any
// others are built, and the checksums with them.  What else was written to the workspace in between, and where, does
// not matter, and the blocks need nothing of one another.  A block forms the FP64 cosines and sines of its views and
// bins once.
// First projection of a 512^2 fan scan with 180 views: 246 us with the finished blocks counted in one word, which marked
// the tables as a whole; 107 us with a checksum per 256 rays of the scan, each forming its own bin's sine; 93 us now
// (later ones 66 us).  The check is kept short, wide multiply-adds, warp sums by one instruction and one barrier: a later
// projection of 128^2 with 60 views keeps the device 12.4 us with 64-bit products, shuffles and two barriers, 10.4 so.
// It reads the tables, which after an L2 flush costs the graph of 16 problems 1 % (7.66 -> 7.74 ms a step) against
// trusting a mark beside them.
constexpr int kTabViews = 8, kTabBins = 32, kTabThreads = kTabViews * kTabBins;
static_assert(kTabBins == 32, "a warp per view");
struct TableArgs {
  ProjTables t;
  unsigned long long fp;
  unsigned blocks;
};
struct TableBlock {
  int k0, b0;  // first view and bin
  int k, b;    // this thread's entry
  int sum;     // this warp's checksum
  bool in;
};
__device__ __forceinline__ TableBlock table_place(const GeomDev& g, unsigned block) {
  const int nb = (g.A + kTabBins - 1) / kTabBins, bb = (int)block % nb;
  TableBlock p;
  p.k0 = (int)block / nb * kTabViews;
  p.b0 = bb * kTabBins;
  p.k = p.k0 + (int)threadIdx.x / kTabBins;
  p.b = p.b0 + (int)threadIdx.x % kTabBins;
  p.sum = p.k * nb + bb;
  p.in = p.k < g.V && p.b < g.A;
  return p;
}

// Checksum of the warp's entries (and, for the first bins, of its view's FP32 cosine and sine) as they stand in memory,
// to every lane.  Each entry's words, multiplied by odd constants and added to a seed of its index, are mixed once more
// by a product with the index; the lanes' two halves are added separately.
__device__ __forceinline__ uint2 table_sum(const GeomDev& g, const TableArgs& a, const TableBlock& p) {
  unsigned long long h = 0;
  if (p.in) {
    const int r = p.k * g.A + p.b;  // V A <= 2^26
    auto add = [&](unsigned w, unsigned odd) { h += (unsigned long long)w * odd; };
    auto add4 = [&](const int4& v, unsigned odd) {
      add(v.x, odd);
      add(v.y, odd * 3u);
      add(v.z, odd * 5u);
      add(v.w, odd * 7u);
    };
    h = a.fp + (unsigned long long)(unsigned)r * 0x9E3779B9u;  // 2^32 over the golden ratio, as below
    add4(a.t.tab0[r], 0x9E3779B9u);
    if (g.kind == INRCT_CONE3D) {
      add4(a.t.tab1[r], 0x9E3779B9u * 9u);
      add(__float_as_uint(a.t.tab2[r]), 0x9E3779B9u * 11u);
    }
    if (p.b == 0) {
      const float2 v = a.t.views[p.k];
      add(__float_as_uint(v.x), 0x9E3779B9u * 13u);
      add(__float_as_uint(v.y), 0x9E3779B9u * 15u);
    }
    h += (unsigned long long)((unsigned)(h >> 32) ^ (unsigned)h) * (2u * (unsigned)r + 0x9E3779B9u);
  }
  return make_uint2(__reduce_add_sync(0xffffffffu, (unsigned)h), __reduce_add_sync(0xffffffffu, (unsigned)(h >> 32)));
}

__device__ __forceinline__ void build_ray2d(const GeomDev& g, double2 view, double2 bin, int4* __restrict__ tab, int b, int r) {
  const double D = 2.0 / g.N;
  const double cb = view.x, sb = view.y;
  double px, py, ex, ey;
  if (g.kind == INRCT_PAR2D) {
    const double t = ((double)b - 0.5 * (g.A - 1)) * g.du * D;
    px = t * cb;
    py = t * sb;
    ex = -sb;
    ey = cb;
  } else {
    const double R = g.sod * D;
    const double cg = bin.x, sg = bin.y;
    ex = -(cb * cg - sb * sg);
    ey = -(sb * cg + cb * sg);
    const double Sx = R * cb, Sy = R * sb;
    const double dot = Sx * ex + Sy * ey;  // point of the ray nearest the isocentre
    px = Sx - dot * ex;
    py = Sy - dot * ey;
  }
  const bool xd = drive_x(ex, ey);
  const double ea = xd ? ex : ey, eq = xd ? ey : ex;
  const double pa = xd ? px : py, pq = xd ? py : px;
  const double a0 = (pa + 1.0) / D - 0.5;  // fractional slice index of the reference point
  const double q0 = (pq + 1.0) / D - 0.5;  // its fractional transverse index
  const double slope = eq / ea;
  const double uref = q0 + ((double)(g.N / 2) - a0) * slope;
  const float sc = (float)(D / fabs(ea));
  tab[r] = pack_ray(uref, slope, xd ? sc : -sc);
}

__device__ __forceinline__ void build_col3d(const GeomDev& g, double2 view, int4* __restrict__ t0,
                                            int4* __restrict__ t1, float* __restrict__ t2, int a, int r) {
  const double D = 2.0 / g.N;
  const double cb = view.x, sb = view.y;
  const double R = g.sod * D;
  const double pu = g.du * D * g.sdd / g.sod;
  const double pv = g.dv * D * g.sdd / g.sod;
  const double ua = ((double)a - 0.5 * (g.A - 1)) * pu;
  const double dc = -(g.sdd - g.sod) * D;
  const double Sx = R * cb, Sy = R * sb;
  const double ex = (dc * cb - ua * sb) - Sx;  // bin - source, xy part (depends on the column only)
  const double ey = (dc * sb + ua * cb) - Sy;
  const double L2 = ex * ex + ey * ey;
  const double tau0 = -(Sx * ex + Sy * ey) / L2;  // nearest point to the z axis
  const double px = Sx + tau0 * ex, py = Sy + tau0 * ey;
  const bool xd = drive_x(ex, ey);
  const double ea = xd ? ex : ey, eq = xd ? ey : ex;
  const double pa = xd ? px : py, pq = xd ? py : px;
  const double a0 = (pa + 1.0) / D - 0.5;
  const double q0 = (pq + 1.0) / D - 0.5;
  const double slope = eq / ea;
  const double jref = (double)(g.N / 2);
  const float sa = (float)(D / fabs(ea));
  t0[r] = pack_ray(q0 + (jref - a0) * slope, slope, xd ? sa : -sa);
  // z crossing: u_z(j) = Cz + vb * G(j), vb = m_r * pv/2 (m_r = 2 row - (B-1)),
  // G(j) = tau(j)/D = G_ref + (j - jref) / e_a
  const double Gref = tau0 / D + (jref - a0) / ea;
  const long long Hh = __double2ll_rn(0.5 * pv * Gref * kFx32);
  const long long Kk = __double2ll_rn(0.5 * pv / ea * kFx48);
  t1[r] = make_int4((int)(unsigned)(Hh & 0xffffffffll), (int)(Hh >> 32),
                    (int)(unsigned)(Kk & 0xffffffffll), (int)(Kk >> 32));
  t2[r] = (float)L2;
}

// One block's part of the tables: rays (2-D) or (view, column) entries (cone).
__device__ __forceinline__ void table_block(const GeomDev& g, const TableArgs& a, unsigned block) {
  __shared__ double2 sv[kTabViews], sb[kTabBins];  // cosine and sine of the view angles, of the fan angles
  const TableBlock p = table_place(g, block);
  const int t = threadIdx.x, w = t >> 5, l = t & 31;
  const bool kept = a.t.sums && p.k < g.V;  // the warp has a checksum
  if (a.t.sums) {
    bool stale = false;
    if (kept) {
      const uint2 was = a.t.sums[p.sum], is = table_sum(g, a, p);
      stale = was.x != is.x || was.y != is.y;
    }
    if (!__syncthreads_or(stale)) return;
  }
  double s, c;
  if (w == 0 && l < kTabViews && p.k0 + l < g.V) {
    sincos(g.angle0 + g.span * (double)(p.k0 + l) / (double)g.V, &s, &c);
    sv[l] = make_double2(c, s);
    if (p.b0 == 0) a.t.views[p.k0 + l] = make_float2((float)c, (float)s);
  }
  if (w == 1 && g.kind == INRCT_FAN2D) {
    sincos(((double)(p.b0 + l) - 0.5 * (g.A - 1)) * g.du / g.sod, &s, &c);
    sb[l] = make_double2(c, s);
  }
  __syncthreads();
  if (p.in) {
    const int r = p.k * g.A + p.b;
    const double2 view = sv[p.k - p.k0];
    if (g.kind == INRCT_CONE3D) build_col3d(g, view, a.t.tab0, a.t.tab1, a.t.tab2, p.b, r);
    else build_ray2d(g, view, sb[p.b - p.b0], a.t.tab0, p.b, r);
  }
  if (!kept) return;
  const uint2 sum = table_sum(g, a, p);
  if (l == 0) a.t.sums[p.sum] = sum;
}

__global__ void __launch_bounds__(kTabThreads) tables_kernel(GeomDev g, const __grid_constant__ TableArgs a) {
  table_block(g, a, blockIdx.x);
}

// ---------------------------------------------------------------------------
// shared helpers: identical integer/FP32 operations in P and P^T
// ---------------------------------------------------------------------------
__device__ __forceinline__ void split_fx(int64_t u, int& i0, float& f) {
  i0 = (int)(u >> 32);
  f = __uint2float_rn((uint32_t)(u & 0xffffffffll)) * 2.3283064365386963e-10f;  // * 2^-32
}

// Interpolation weight that crossing u gives to integer index q
// (the forward gives 1 - f to floor(u) and f to floor(u) + 1).
__device__ __forceinline__ float tap_weight(int64_t u, int q) {
  int i0;
  float f;
  split_fx(u, i0, f);
  return q == i0 ? __fsub_rn(1.f, f) : (q == i0 + 1 ? f : 0.f);
}

__device__ __forceinline__ int64_t slope_fx(const int4& t) { return (int64_t)t.z << 2; }

struct ConeRay {
  int64_t Z0, Sz;  // z crossing at jref and its step, 32.32
  float vb;        // v coordinate of the detector row (world units)
};

__device__ __forceinline__ ConeRay cone_ray(const int4& t1, int mr, int64_t CzF, float pv_half) {
  const int64_t Hh = ((int64_t)t1.y << 32) | (int64_t)(uint32_t)t1.x;
  const int64_t Kk = ((int64_t)t1.w << 32) | (int64_t)(uint32_t)t1.z;
  ConeRay c;
  c.Z0 = CzF + (int64_t)mr * Hh;
  c.Sz = ((int64_t)mr * Kk) >> 16;
  c.vb = __fmul_rn((float)mr, pv_half);
  return c;
}

__device__ __forceinline__ float cone_scale(float vb, float L2, float sa) {
  return __fmul_rn(__fsqrt_rn(__fmaf_rn(vb, vb, L2)), sa);
}

// Slices j in [lo, hi) where u(j) = uref + (j - jref) * slope may lie in (-1, N).
__device__ __forceinline__ void active_range(float uref, float slope, int jref, int N, int& lo,
                                             int& hi) {
  if (fabsf(slope) < 1e-12f) {
    if (uref > -1.f && uref < (float)N) {
      lo = 0;
      hi = N;
    } else {
      lo = hi = 0;
    }
    return;
  }
  const float ja = (float)jref + (-1.f - uref) / slope, jb = (float)jref + ((float)N - uref) / slope;
  float l = fminf(ja, jb), h = fmaxf(ja, jb);
  l = fmaxf(l - 1.f, -1.f);
  h = fminf(h + 1.f, (float)N + 1.f);
  lo = max(0, (int)floorf(l));
  hi = min(N, (int)ceilf(h) + 1);
  if (hi < lo) hi = lo;
}

__device__ __forceinline__ float fx_to_float(int64_t u) { return (float)((double)u * (1.0 / kFx32)); }

// ---------------------------------------------------------------------------
// transposes (x-driven rays read img^T so that their taps are contiguous)
// ---------------------------------------------------------------------------
// The 2-D projection's preparation in one launch: the first a.blocks blocks are the table launch, the others transpose
// 32 x 32 tiles of the image (128^2, 60 views: four launches of a projection become two, 29 -> 24 us a call).
__global__ void __launch_bounds__(kTabThreads)
    prep2d_kernel(GeomDev g, const __grid_constant__ TableArgs a, const float* __restrict__ in, float* __restrict__ out) {
  if (blockIdx.x < a.blocks) {
    table_block(g, a, blockIdx.x);
    return;
  }
  __shared__ float tile[32][33];
  const int N = g.N, nx = (N + 31) / 32, i = blockIdx.x - a.blocks;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, x0 = (i % nx) * 32, y0 = (i / nx) * 32;
  for (int yy = ty; yy < 32; yy += kTabThreads / 32)
    if (x0 + tx < N && y0 + yy < N) tile[yy][tx] = in[(size_t)(y0 + yy) * N + x0 + tx];
  __syncthreads();
  for (int xx = ty; xx < 32; xx += kTabThreads / 32)
    if (x0 + xx < N && y0 + tx < N) out[(size_t)(x0 + xx) * N + y0 + tx] = tile[tx][xx];
}

__global__ void transpose_xy_kernel(const float* __restrict__ in, float* __restrict__ out, int N) {
  __shared__ float tile[32][33];
  const size_t zoff = (size_t)blockIdx.z * N * N;
  int x = blockIdx.x * 32 + threadIdx.x;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    int y = blockIdx.y * 32 + yy;
    if (x < N && y < N) tile[yy][threadIdx.x] = in[zoff + (size_t)y * N + x];
  }
  __syncthreads();
  int y = blockIdx.y * 32 + threadIdx.x;
  for (int xx = threadIdx.y; xx < 32; xx += blockDim.y) {
    int xo = blockIdx.x * 32 + xx;
    if (xo < N && y < N) out[zoff + (size_t)xo * N + y] = tile[threadIdx.x][xx];
  }
}

// Volume [z][y][x] -> [y][x][z] with columns of Zp >= N voxels, zeros past N.
__global__ void transpose_z_kernel(const float* __restrict__ in, float* __restrict__ out, int N, int Zp) {
  __shared__ float tile[32][33];
  const int y = blockIdx.z, x = blockIdx.x * 32 + threadIdx.x;
  for (int zz = threadIdx.y; zz < 32; zz += blockDim.y) {
    const int z = blockIdx.y * 32 + zz;
    tile[zz][threadIdx.x] = x < N && z < N ? in[((size_t)z * N + y) * N + x] : 0.f;
  }
  __syncthreads();
  const int z = blockIdx.y * 32 + threadIdx.x;
  for (int xx = threadIdx.y; xx < 32; xx += blockDim.y) {
    const int xo = blockIdx.x * 32 + xx;
    if (xo < N && z < Zp) out[((size_t)y * N + xo) * Zp + z] = tile[threadIdx.x][xx];
  }
}

// ---------------------------------------------------------------------------
// forward projection
// ---------------------------------------------------------------------------
template <int SEG>
__global__ void __launch_bounds__(32 * SEG)
    project2d_kernel(const int4* __restrict__ tab, int m, int N, const float* __restrict__ img,
                     const float* __restrict__ imgT, float* __restrict__ sino,
                     const float* __restrict__ y, float* __restrict__ resid,
                     double* __restrict__ loss_part) {
  __shared__ float part[SEG][33];
  const int lane = threadIdx.x, s = threadIdx.y;
  const int r = blockIdx.x * 32 + lane;
  const int jref = N / 2;
  float sum = 0.f, sc = 0.f;
  if (r < m) {
    const int4 P = __ldg(tab + r);
    sc = __int_as_float(P.w);
    const float* base = sc > 0.f ? imgT : img;
    sc = fabsf(sc);
    const int64_t U0 = ray_U0(P), S4 = slope_fx(P);
    int lo, hi;
    active_range(fx_to_float(U0), (float)P.z * 9.313225746154785e-10f, jref, N, lo, hi);
    const int per = (hi - lo + SEG - 1) / SEG;
    const int j0 = lo + s * per, j1 = min(hi, j0 + per);
    int64_t u = U0 + (int64_t)(j0 - jref) * S4;
    int jN = j0 * N;  // 32-bit row offset: N^2 <= 4096^2
    for (int j = j0; j < j1; ++j, u += S4, jN += N) {
      int i0;
      float f;
      split_fx(u, i0, f);
      const float* row = base + jN;
      // 0 <= i0 < N and -1 <= i0 < N - 1 as unsigned compares
      const float v0 = (unsigned)i0 < (unsigned)N ? __ldg(row + i0) : 0.f;
      const float v1 = (unsigned)(i0 + 1) < (unsigned)N ? __ldg(row + i0 + 1) : 0.f;
      sum = fmaf(__fsub_rn(1.f, f), v0, fmaf(f, v1, sum));
    }
  }
  part[s][lane] = sum;
  __syncthreads();
  if (s == 0) {
    float z = 0.f;
#pragma unroll
    for (int k = 0; k < SEG; ++k) z += part[k][lane];
    z *= sc;
    float l = 0.f;
    if (r < m) {
      sino[r] = z;
      if (y) {
        const float d = z - y[r];
        resid[r] = d;
        l = d * d;
      }
    }
    if (y) {
#pragma unroll
      for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) loss_part[blockIdx.x] = 0.5 * (double)l;
    }
  }
}

template <int SEG>
__global__ void __launch_bounds__(32 * SEG)
    project3d_kernel(const int4* __restrict__ t0, const int4* __restrict__ t1,
                     const float* __restrict__ t2, int A, int B, int N, float pv_half, int64_t CzF,
                     const float* __restrict__ vol, const float* __restrict__ volT,
                     float* __restrict__ sino, const float* __restrict__ y,
                     float* __restrict__ resid, double* __restrict__ loss_part) {
  __shared__ float part[SEG][33];
  const int lane = threadIdx.x, s = threadIdx.y;
  // grid (column groups, views, rows): the blocks of one detector row run together for all
  // views; their rays cross nearly the same z-band of the volume, which then stays in L2
  const int a = blockIdx.x * 32 + lane, k = blockIdx.y, row = blockIdx.z;
  const int jref = N / 2;
  float sum = 0.f, sc = 0.f;
  if (a < A) {
    const size_t ci = (size_t)k * A + a;
    const int4 P = __ldg(t0 + ci);
    const ConeRay cr = cone_ray(__ldg(t1 + ci), 2 * row - (B - 1), CzF, pv_half);
    const float sa = __int_as_float(P.w);
    sc = cone_scale(cr.vb, __ldg(t2 + ci), fabsf(sa));
    const float* base = sa > 0.f ? volT : vol;
    const int64_t Uq = ray_U0(P), Sq = slope_fx(P);
    int lo, hi, lz, hz;
    active_range(fx_to_float(Uq), (float)P.z * 9.313225746154785e-10f, jref, N, lo, hi);
    active_range(fx_to_float(cr.Z0), fx_to_float(cr.Sz), jref, N, lz, hz);
    lo = max(lo, lz);
    hi = min(hi, hz);
    if (hi < lo) hi = lo;
    const int per = (hi - lo + SEG - 1) / SEG;
    const int j0 = lo + s * per, j1 = min(hi, j0 + per);
    const size_t NN = (size_t)N * N;
    int64_t uq = Uq + (int64_t)(j0 - jref) * Sq;
    int64_t uz = cr.Z0 + (int64_t)(j0 - jref) * cr.Sz;
    for (int j = j0; j < j1; ++j, uq += Sq, uz += cr.Sz) {
      int iq, iz;
      float fq, fz;
      split_fx(uq, iq, fq);
      split_fx(uz, iz, fz);
      const float wq0 = __fsub_rn(1.f, fq), wz0 = __fsub_rn(1.f, fz);
      const bool q0ok = iq >= 0 && iq < N, q1ok = iq >= -1 && iq + 1 < N;
      const bool z0ok = iz >= 0 && iz < N, z1ok = iz >= -1 && iz + 1 < N;
      const float* p0 = base + (ptrdiff_t)iz * (ptrdiff_t)NN + (ptrdiff_t)j * N + iq;
      const float* p1 = p0 + NN;
      const float v00 = (z0ok && q0ok) ? __ldg(p0) : 0.f;
      const float v01 = (z0ok && q1ok) ? __ldg(p0 + 1) : 0.f;
      const float v10 = (z1ok && q0ok) ? __ldg(p1) : 0.f;
      const float v11 = (z1ok && q1ok) ? __ldg(p1 + 1) : 0.f;
      sum = fmaf(wz0 * wq0, v00, sum);
      sum = fmaf(wz0 * fq, v01, sum);
      sum = fmaf(fz * wq0, v10, sum);
      sum = fmaf(fz * fq, v11, sum);
    }
  }
  part[s][lane] = sum;
  __syncthreads();
  if (s == 0) {
    float z = 0.f;
#pragma unroll
    for (int q = 0; q < SEG; ++q) z += part[q][lane];
    z *= sc;
    float l = 0.f;
    const size_t r = ((size_t)k * B + row) * A + a;
    if (a < A) {
      sino[r] = z;
      if (y) {
        const float d = z - y[r];
        resid[r] = d;
        l = d * d;
      }
    }
    if (y) {
#pragma unroll
      for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0)
        loss_part[((size_t)k * B + row) * gridDim.x + blockIdx.x] = 0.5 * (double)l;
    }
  }
}

// Cone forward projection, plan seg = 1 in row patches: each thread takes a whole ray and a block holds 32
// detector columns of kRowsPerBlock consecutive detector rows of one view.  Rays of neighbouring
// rows cross nearly the same slices at z about 2/3 voxel apart, so the warps of a block re-read
// one another's lines from L1 (project3d_kernel's blocks hold one row, and the blocks of the
// neighbouring rows run far apart in launch order).  Same samples and weights as
// project3d_kernel; the sum runs in two accumulators, even and odd samples, added at the end, so
// its rounding chain is as short as that of the two-segment plan (sinograms agree with it to
// about 4e-7 relative) and the two FMA chains are independent.  OFF32 (N <= 1024, so N^3 + N^2 <
// 2^31) forms the tap addresses from 32-bit offsets, stepping j N by N along the ray.
constexpr int kRowsPerBlock = 4;
template <bool OFF32>
__global__ void __launch_bounds__(32 * kRowsPerBlock)
    project3d_rows_kernel(const int4* __restrict__ t0, const int4* __restrict__ t1,
                          const float* __restrict__ t2, int A, int B, int N, float pv_half, int64_t CzF,
                          const float* __restrict__ vol, const float* __restrict__ volT,
                          float* __restrict__ sino, const float* __restrict__ y,
                          float* __restrict__ resid, double* __restrict__ loss_part) {
  __shared__ float part[kRowsPerBlock];
  const int lane = threadIdx.x, w = threadIdx.y;
  const int a = blockIdx.x * 32 + lane, k = blockIdx.y, row = blockIdx.z * kRowsPerBlock + w;
  const int jref = N / 2;
  float sum = 0.f, sc = 0.f;
  const bool live = a < A && row < B;
  if (live) {
    const size_t ci = (size_t)k * A + a;
    const int4 P = __ldg(t0 + ci);
    const ConeRay cr = cone_ray(__ldg(t1 + ci), 2 * row - (B - 1), CzF, pv_half);
    const float sa = __int_as_float(P.w);
    sc = cone_scale(cr.vb, __ldg(t2 + ci), fabsf(sa));
    const float* base = sa > 0.f ? volT : vol;
    const int64_t Uq = ray_U0(P), Sq = slope_fx(P);
    int lo, hi, lz, hz;
    active_range(fx_to_float(Uq), (float)P.z * 9.313225746154785e-10f, jref, N, lo, hi);
    active_range(fx_to_float(cr.Z0), fx_to_float(cr.Sz), jref, N, lz, hz);
    lo = max(lo, lz);
    hi = min(hi, hz);
    if (hi < lo) hi = lo;
    const size_t NN = (size_t)N * N;
    // two accumulators, even and odd samples of the ray, added at the end: a shorter rounding
    // chain than one sequence (and two independent FMA chains)
    float s0 = 0.f, s1 = 0.f;
    int64_t uq = Uq + (int64_t)(lo - jref) * Sq;
    int64_t uz = cr.Z0 + (int64_t)(lo - jref) * cr.Sz;
    const int NN32 = N * N;
    int jN = lo * N;
    auto sample = [&](int j, float& acc) {
      int iq, iz;
      float fq, fz;
      split_fx(uq, iq, fq);
      split_fx(uz, iz, fz);
      const float wq0 = __fsub_rn(1.f, fq), wz0 = __fsub_rn(1.f, fz);
      // 0 <= i < N and -1 <= i < N - 1 as unsigned compares
      const bool q0ok = (unsigned)iq < (unsigned)N, q1ok = (unsigned)(iq + 1) < (unsigned)N;
      const bool z0ok = (unsigned)iz < (unsigned)N, z1ok = (unsigned)(iz + 1) < (unsigned)N;
      const float* p0;
      const float* p1;
      if constexpr (OFF32) {
        p0 = base + (iz * NN32 + jN + iq);
        p1 = p0 + NN32;
        jN += N;
      } else {
        p0 = base + (ptrdiff_t)iz * (ptrdiff_t)NN + (ptrdiff_t)j * N + iq;
        p1 = p0 + NN;
      }
      const float v00 = (z0ok && q0ok) ? __ldg(p0) : 0.f;
      const float v01 = (z0ok && q1ok) ? __ldg(p0 + 1) : 0.f;
      const float v10 = (z1ok && q0ok) ? __ldg(p1) : 0.f;
      const float v11 = (z1ok && q1ok) ? __ldg(p1 + 1) : 0.f;
      acc = fmaf(wz0 * wq0, v00, acc);
      acc = fmaf(wz0 * fq, v01, acc);
      acc = fmaf(fz * wq0, v10, acc);
      acc = fmaf(fz * fq, v11, acc);
      uq += Sq;
      uz += cr.Sz;
    };
    int j = lo;
    for (; j + 1 < hi; j += 2) {
      sample(j, s0);
      sample(j + 1, s1);
    }
    if (j < hi) sample(j, s0);
    sum = s0 + s1;
  }
  const float z = sum * sc;
  float l = 0.f;
  if (live) {
    const size_t r = ((size_t)k * B + row) * A + a;
    sino[r] = z;
    if (y) {
      const float d = z - y[r];
      resid[r] = d;
      l = d * d;
    }
  }
  if (y) {
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) part[w] = l;
    __syncthreads();
    if (w == 0 && lane == 0) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < kRowsPerBlock; ++q) t += part[q];
      loss_part[((size_t)k * gridDim.z + blockIdx.z) * gridDim.x + blockIdx.x] = 0.5 * (double)t;
    }
  }
}

// Cone forward projection, plan seg = 1 by columns (cols_fit, cols_faster): one warp per (view, detector column) and chunk of
// 32 R detector rows, lane l taking rows l, l + 32, ...  All rows of a detector column cross a slice at the same
// transverse place, so a slice is first interpolated across once for the whole column,
//   T[z] = (1 - f) vol[q][z] + f vol[q + 1][z],
// by 16-byte loads from the z-fastest copy of the volume (both driving axes read the same copy), and every row then
// takes two neighbouring T from shared memory: full lines per T and two shared loads per sample, instead of four
// gathers of about two lines each.  The next slice's voxels are in flight while the rows of this one are sampled.
// The warp's shared T holds `pad` zeros on both sides, so rows of four 32-row groups that partly miss the volume
// need no test; fours that miss it are skipped.
// z crossings: u(row, j) = Cz + m_row G(j) in 32.32 fixed point with G(j) = (Hh 2^16 + (j - jref) Kk) / 2^16, so a
// slice costs one 64-bit product per lane and a group one 64-bit addition.  What depends on the slice alone is
// computed for 32 slices at a time, one per lane, and handed round; a ray's sum over those 32 is added to its total
// in shared memory.  Two groups are weighted and added by packed FP32 instructions.
// A block holds kColsPerBlock neighbouring columns, whose transverse taps overlap in L1; the results leave through
// shared memory in runs of the block's columns.
// 501^3 x 60 views x 768^2: 14.28 -> 9.36 ms with the transpose (project3d_rows_kernel: L1 86 % busy), error against
// FP64 3.4e-7 -> 1.0e-7.  Now bound by the latency of the volume's lines at 24 warps per SM and by issue (65 %
// active; L1 60 %, L2 27 %, DRAM 3.2 of 6.8 TB/s).  Measured beside it: three pieces ahead with 20 warps 10.4 ms,
// 8 columns per block 9.46, 12 columns 9.70, 24 rows per lane 12.5, prefetches into L1 or L2 no change.
constexpr int kColsPerBlock = 4, kColsAhead = 2;  // 128-voxel pieces of the next slice held in registers
typedef unsigned long long f32x2;  // two FP32 values in one 64-bit register
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2r(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
template <int R>
__global__ void __launch_bounds__(32 * kColsPerBlock, 6)
    project3d_cols_kernel(const int4* __restrict__ t0, const int4* __restrict__ t1, const float* __restrict__ t2, int A,
                          int B, int N, int Zp, int pad, float pv_half, int64_t CzF, const float* __restrict__ volz,
                          float* __restrict__ sino, const float* __restrict__ y, float* __restrict__ resid,
                          double* __restrict__ loss_part) {
  constexpr int RP = R / 2;                     // pairs of row groups
  constexpr unsigned kFull = 0xffffffffu;
  extern __shared__ __align__(16) float csm[];  // [kColsPerBlock][Zp + 2 pad], then [kColsPerBlock][32 R + 1]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int a = blockIdx.x * kColsPerBlock + w, k = blockIdx.y, rbase = blockIdx.z * 32 * R;
  const int ts = Zp + 2 * pad;
  float* T = csm + w * ts + pad;
  float* res = csm + kColsPerBlock * ts + w * (32 * R + 1);  // this column's sums, then the block's [column][row]
#pragma unroll
  for (int i = 0; i < R; ++i) res[lane + 32 * i] = 0.f;
  if (a < A) {
    for (int i = lane; i < ts; i += 32) T[i - pad] = 0.f;
    __syncwarp();  // other lanes write the same words below
    const size_t ci = (size_t)k * A + a;
    const int jref = N / 2;
    int lo, hi;
    bool xd;
    {
      const int4 P = __ldg(t0 + ci);
      xd = __int_as_float(P.w) > 0.f;
      active_range(fx_to_float(ray_U0(P)), (float)P.z * 9.313225746154785e-10f, jref, N, lo, hi);
    }
    const int qstep = xd ? N * Zp : Zp;
    // this lane's slice of the batch: offset of its first voxel, weight, z pitch, and packed: first and last four
    // row groups (4 bits each), whether its two taps are inside, end and begin of the voxels in fours
    int e_off = 0;
    float e_f = 0.f;
    int64_t e_G = 0;
    unsigned e_meta = 0;  // no voxels: the slice is skipped
    auto batch = [&](int jb) {
      // the column's table entries are read again for each batch: kept, they would cost ten registers
      const int4 P = __ldg(t0 + ci), Q = __ldg(t1 + ci);
      const int64_t Hh = ((int64_t)Q.y << 32) | (int64_t)(uint32_t)Q.x;
      const int64_t Kk = ((int64_t)Q.w << 32) | (int64_t)(uint32_t)Q.z;
      const float hf = fx_to_float(Hh), kf = (float)((double)Kk * (1.0 / kFx48));
      const float Bm1 = (float)(B - 1), Cz = 0.5f * (float)N - 0.5f;
      const int j = jb + lane;
      const int64_t dj = j - jref;
      int iq;
      split_fx(ray_U0(P) + dj * slope_fx(P), iq, e_f);
      e_G = ((Hh << 16) + dj * Kk + 32768) >> 16;
      // the row groups that can meet the volume, in FP32 (a row of margin), and the z their rows reach
      const float g = fmaf((float)dj, kf, hf), inv = __frcp_rn(g);
      const int rl = (int)floorf(fmaf(0.5f, fmaf(-1.f - Cz, inv, Bm1), -1.f)) - rbase;
      const int rh = (int)ceilf(fminf(fmaf(0.5f, fmaf((float)N - Cz, inv, Bm1), 1.f), Bm1)) - rbase;
      const int il = max(0, rl >> 7), ih = min(R / 4 - 1, rh >> 7);
      const bool q0 = (unsigned)iq < (unsigned)N, q1 = (unsigned)(iq + 1) < (unsigned)N;
      const float m0 = (float)(2 * (rbase + 128 * il)) - Bm1, m1 = fminf((float)(2 * (rbase + 128 * ih + 127)) - Bm1, Bm1);
      const int z0 = max(0, ((int)floorf(fmaf(m0, g, Cz)) - 1) & ~3), z1 = min(N, (int)floorf(fmaf(m1, g, Cz)) + 3);
      e_off = j * (xd ? Zp : N * Zp) + iq * qstep + z0;
      e_meta = j < hi && il <= ih && (q0 || q1) && z0 < z1
                   ? (unsigned)il | (unsigned)ih << 4 | (q0 ? 256u : 0u) | (q1 ? 512u : 0u) |
                         (unsigned)((z1 + 3) >> 2) << 10 | (unsigned)(z0 >> 2) << 19
                   : 0u;
    };
    auto pieces = [](unsigned meta) { return ((int)((meta >> 10) & 511u) - (int)(meta >> 19) + 31) >> 5; };
    float4 v0[kColsAhead], v1[kColsAhead];
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load = [&](int off, unsigned meta, int n, float4& x0, float4& x1) {
      const bool in = (int)(meta >> 19) + lane + 32 * n < (int)((meta >> 10) & 511u);
      const float* c = volz + (off + 4 * lane + 128 * n);
      x0 = in && (meta & 256u) ? __ldg(reinterpret_cast<const float4*>(c)) : none;
      x1 = in && (meta & 512u) ? __ldg(reinterpret_cast<const float4*>(c + qstep)) : none;
    };
    auto put = [&](unsigned meta, float f, int n, const float4& x0, const float4& x1) {
      const int z4 = (int)(meta >> 19) + lane + 32 * n;
      const float w0 = __fsub_rn(1.f, f);
      if (z4 < (int)((meta >> 10) & 511u))
        *reinterpret_cast<float4*>(T + 4 * z4) = make_float4(fmaf(f, x1.x, w0 * x0.x), fmaf(f, x1.y, w0 * x0.y),
                                                        fmaf(f, x1.z, w0 * x0.z), fmaf(f, x1.w, w0 * x0.w));
    };
    int off;
    unsigned meta;
    float f;
    int64_t G;
    auto next = [&](int j) {  // slice j's values to all lanes, its first pieces in flight
      const int t = (j - lo) & 31;
      if (t == 0) batch(j);
      off = __shfl_sync(kFull, e_off, t);
      f = __shfl_sync(kFull, e_f, t);
      G = __shfl_sync(kFull, e_G, t);
      meta = __shfl_sync(kFull, e_meta, t);
      const int np = pieces(meta);
#pragma unroll
      for (int n = 0; n < kColsAhead; ++n)
        if (n < np) load(off, meta, n, v0[n], v1[n]);
    };
    const f32x2 kScale = pack2(2.3283064365386963e-10f, 2.3283064365386963e-10f), kOne = pack2(1.f, 1.f),
                kMinus = pack2(-1.f, -1.f);
    f32x2 acc[RP];
#pragma unroll
    for (int i = 0; i < RP; ++i) acc[i] = 0ull;
    auto flush = [&]() {  // add the sums of up to 32 slices to the column's (short rounding chains, few registers)
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        float s0, s1;
        unpack2(acc[i], s0, s1);
        res[lane + 64 * i] += s0;
        res[lane + 64 * i + 32] += s1;
        acc[i] = 0ull;
      }
    };
    if (lo < hi) next(lo);
    for (int j = lo; j < hi; ++j) {
      const unsigned m = meta;
      const int64_t Gc = G;
      const int np = pieces(m), il = m & 15, ih = (m >> 4) & 15;
#pragma unroll
      for (int n = 0; n < kColsAhead; ++n)
        if (n < np) put(m, f, n, v0[n], v1[n]);
      for (int n = kColsAhead; n < np; ++n) {
        float4 x0, x1;
        load(off, m, n, x0, x1);
        put(m, f, n, x0, x1);
      }
      __syncwarp();
      if (j + 1 < hi) next(j + 1);
      if (np > 0) {
        int64_t u = CzF + (int64_t)(2 * (rbase + lane) - (B - 1)) * Gc;
        const int64_t du = 64 * Gc;
#pragma unroll
        for (int i = 0; i < R / 4; ++i) {
          if (i >= il && i <= ih) {
            const int64_t uu[4] = {u, u + du, u + 2 * du, u + 3 * du};
            float ta[4], tb[4], fr[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float* pt = T + (int)(uu[q] >> 32);
              ta[q] = pt[0];
              tb[q] = pt[1];
              fr[q] = __uint2float_rn((uint32_t)uu[q]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const f32x2 f2 = mul2(pack2(fr[2 * h], fr[2 * h + 1]), kScale);
              fma2(acc[2 * i + h], fma2r(f2, kMinus, kOne), pack2(ta[2 * h], ta[2 * h + 1]));
              fma2(acc[2 * i + h], f2, pack2(tb[2 * h], tb[2 * h + 1]));
            }
          }
          u += 4 * du;
        }
      }
      if (((j - lo) & 31) == 31) flush();
      __syncwarp();
    }
    flush();
  }
  float sa = 0.f, L2 = 0.f;
  if (a < A) {
    sa = fabsf(__int_as_float(__ldg(t0 + (size_t)k * A + a).w));
    L2 = __ldg(t2 + (size_t)k * A + a);
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
    res[lane + 32 * i] *= cone_scale(__fmul_rn((float)(2 * (rbase + lane + 32 * i) - (B - 1)), pv_half), L2, sa);
  __syncthreads();
  double l = 0.0;
  const int c = threadIdx.x % kColsPerBlock, ac = blockIdx.x * kColsPerBlock + c;
  for (int r = threadIdx.x / kColsPerBlock; r < 32 * R; r += 32) {
    const int row = rbase + r;
    if (ac >= A || row >= B) continue;
    const size_t o = ((size_t)k * B + row) * A + ac;
    const float z = csm[kColsPerBlock * ts + c * (32 * R + 1) + r];
    sino[o] = z;
    if (y) {
      const float d = z - y[o];
      resid[o] = d;
      l += (double)(d * d);
    }
  }
  if (y) {
    __shared__ double part[kColsPerBlock];
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) part[w] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < kColsPerBlock; ++q) t += part[q];
      loss_part[((size_t)blockIdx.z * gridDim.y + k) * gridDim.x + blockIdx.x] = 0.5 * t;
    }
  }
}

// Deterministic FP64 sum of n partials into out[0]: one block, eight loads in flight per thread.  Bound by the FP64
// pipe (16 cycles per warp instruction on this part), so few warps and one addition per value: 344 partials took
// 8.3 us with 32 warps and eight sums per thread, 3.6 us now.
constexpr int kSumThreads = 256;
__global__ void __launch_bounds__(kSumThreads)
    reduce_f64_kernel(const double* __restrict__ in, int64_t n, double* __restrict__ out) {
  __shared__ double sh[kSumThreads];
  const int t = threadIdx.x;
  double s = 0.0;
  for (int64_t i = t; i < n; i += 8 * kSumThreads) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i + u * kSumThreads < n) v[u] = in[i + u * kSumThreads];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i + u * kSumThreads < n) s += v[u];
  }
  sh[t] = s;
  __syncthreads();
  if (t >= 32) return;
  s = 0.0;
#pragma unroll
  for (int w = 0; w < kSumThreads / 32; ++w)
    if (32 * w < n) s += sh[t + 32 * w];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (t == 0) out[0] = s;
}

int reduce_f64(const double* in, int64_t n, double* out, cudaStream_t st) {
  reduce_f64_kernel<<<1, kSumThreads, 0, st>>>(in, n, out);
  INRCT_CHECK_LAUNCH("FP64 sum");
  return INRCT_OK;
}

// ---------------------------------------------------------------------------
// adjoint (gather form)
// ---------------------------------------------------------------------------
// 2-D adjoint, tile-driven.  A block owns a 32 x 32 pixel tile; its warps take
// disjoint subsets of the views.  For one view, a warp walks the rays whose
// window can reach the tile (the bin range spanned by the tile's corners plus
// the interpolation reach), and lane l evaluates each ray at the tile's slice l
// of the ray's driving axis: the ray's fixed-point crossing there, identical
// to the forward projector's, gives the two taps 1 - f and f on transverse
// indices floor(u) and floor(u) + 1, which are added into the warp's
// accumulator of the tile.  A crossing is thus evaluated once per (ray, slice)
// instead of once per (pixel, candidate ray).  The accumulator is laid out
// [transverse][slice] (row stride 32), so that lane l always writes bank l: no
// conflicts and no atomics.  y-driven rays are walked first, x-driven rays second,
// with one accumulator per warp for the two in turn; a view's window is walked twice
// only where both kinds occur in it (its first and last ray differ; for small launches
// see TWO below).  The windows of
// 32 views are computed at a time, one per lane.  The warps' accumulators are summed
// in a fixed order (deterministic).
// 512^2 fan, 90 views: the call takes 99 us with two accumulators per warp (three blocks
// per SM, so the 512 blocks ran as one wave and a nearly empty one) and every lane
// computing every window, 74 us now, with the same bits (1024^2 parallel, 180 views: 438 ->
// 297 us).  Bound by the chain through the accumulator and by warps waiting for the others
// of their block (issue 49 % active, 31.6 M instructions).
constexpr int kBpTile = 32, kBpWarps = 8;
// When an image has few tiles, each tile's views are split over S blocks that write S
// partial images, summed in a fixed order afterwards: S is the smallest split that
// gives about three blocks per SM of a 152-SM GPU.
constexpr int kBpTargetBlocks = 3 * 152;
constexpr int kBpTwoBlocks = 3 * 152;  // see TWO below
constexpr size_t bp_smem(bool two) {
  return sizeof(float) * ((size_t)(two ? 2 : 1) * kBpWarps * kBpTile * kBpTile + kBpTile * (kBpTile + 1));
}

// TWO: an accumulator for each kind of ray, so that a view is walked once and the block waits once.  Three blocks per SM
// instead of five, so for launches of no more blocks than that: small images, where a warp has few views and the set-up
// and the wait between the kinds are what a call costs (fan 96^2, 24
// views: 28.2 us with one accumulator, 22.7 with two; 362^2 and 60 views: the same).
template <bool TWO>
__global__ void __launch_bounds__(32 * kBpWarps)
    backproject2d_tile_kernel(GeomDev g, const int4* __restrict__ tab, const float2* __restrict__ views,
                              const float* __restrict__ sino, float* __restrict__ out, int nsplit) {
  // view split blockIdx.z of nsplit writes its own partial image (the image itself if nsplit == 1)
  constexpr unsigned kFull = 0xffffffffu;
  float* img = out + (size_t)blockIdx.z * g.N * g.N;
  extern __shared__ float bsm[];
  float* acc = bsm + (size_t)threadIdx.y * kBpTile * kBpTile;  // this warp's taps [q][lane]
  constexpr int kAcc = kBpWarps * kBpTile * kBpTile;           // TWO: the x-driven rays' accumulators follow
  float* fin = bsm + (TWO ? 2 : 1) * kAcc;                     // sums of the y-driven taps, [row][col], stride 33
  const int lane = threadIdx.x, wv = threadIdx.y;
  const int N = g.N, A = g.A;
  const int jref = N / 2;
  const int x0 = blockIdx.x * kBpTile, y0 = blockIdx.y * kBpTile;
  const float D = 2.f / (float)N;
  // pixel-centre box of the tile (clipped to the image)
  const float xlo = -1.f + ((float)x0 + 0.5f) * D, xhi = -1.f + ((float)min(x0 + kBpTile, N) - 0.5f) * D;
  const float ylo = -1.f + ((float)y0 + 0.5f) * D, yhi = -1.f + ((float)min(y0 + kBpTile, N) - 0.5f) * D;
  const float cA = 0.5f * (float)(A - 1);
  const bool par = g.kind == INRCT_PAR2D;
  const float inv_pitch = (float)(1.0 / (g.du * (2.0 / N)));  // parallel: bins per world unit
  const float inv_dgam = (float)(g.sod / g.du);                // fan: bins per radian
  const float R = (float)(g.sod * (2.0 / N));
  const float hpar = (float)(1.0 / g.du) + 0.02f;
  const int k0 = blockIdx.z * kBpWarps + wv, kstep = nsplit * kBpWarps;
  const int t = wv * 32 + lane;
  // sums over the block's warps: y-driven taps to fin, x-driven ones with them to the image
  auto add_warps = [&](bool xphase) {
    const float* a = bsm + (TWO && xphase ? kAcc : 0);
    __syncthreads();
    for (int i = t; i < kBpTile * kBpTile; i += 32 * kBpWarps) {
      const int u = i >> 5, v = i & 31;  // y-driven: column u, row v; x-driven: row u, column v
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < kBpWarps; ++w) s += a[w * kBpTile * kBpTile + u * kBpTile + v];
      if (!xphase) fin[v * (kBpTile + 1) + u] = s;
      else if (y0 + u < N && x0 + v < N) img[(size_t)(y0 + u) * N + x0 + v] = s + fin[u * (kBpTile + 1) + v];
    }
  };
  // slices and transverse places of the rays being added: x-driven rays' slices are columns
  int dj4, qbase;  // slopes are in 2.30, crossings in 32.32
  unsigned qlim;   // places inside tile and image
  float* kacc;
  auto aim = [&](bool xd) {
    const int j = (xd ? x0 : y0) + lane;
    qbase = xd ? y0 : x0;
    dj4 = 4 * (j - jref);
    qlim = j < N ? (unsigned)min(kBpTile, N - qbase) : 0u;
    kacc = acc + (TWO && xd ? kAcc : 0);
  };
  int b0 = 0, b1 = -1, kinds = 0;  // this lane's view of the batch
  const bool one_batch = k0 + 32 * kstep >= g.V;
#pragma unroll 1
  for (int phase = 0; phase < (TWO ? 1 : 2); ++phase) {
    const bool xphase = phase == 1;
    for (int i = lane; i < kBpTile * kBpTile; i += 32) {
      acc[i] = 0.f;
      if (TWO) acc[kAcc + i] = 0.f;
    }
    __syncwarp();
    if (!TWO) aim(xphase);
    for (int kb = k0; kb < g.V; kb += 32 * kstep) {
      // this lane's view of the batch: the bins whose window (centre +- h, as for a single pixel) can reach a pixel
      // of the tile, and the kinds of its rays: 1 driven along y, 2 along x, 3 both
      const int kl = kb + lane * kstep;
      if (!(xphase && one_batch)) {
        b0 = 0, b1 = -1, kinds = 0;
      }
      if (kl < g.V && !(xphase && one_batch)) {
        const float2 cs = views[kl];
        const float cb = cs.x, sb = cs.y;
        float blo, bhi;
        if (par) {
          const float c00 = (xlo * cb + ylo * sb), c10 = (xhi * cb + ylo * sb);
          const float c01 = (xlo * cb + yhi * sb), c11 = (xhi * cb + yhi * sb);
          blo = fmaf(fminf(fminf(c00, c10), fminf(c01, c11)), inv_pitch, cA) - hpar;
          bhi = fmaf(fmaxf(fmaxf(c00, c10), fmaxf(c01, c11)), inv_pitch, cA) + hpar;
        } else {
          // fan angle of a point seen from the source, as a bin coordinate; extreme at the corners
          const float sx = R * cb, sy = R * sb;
          auto bin_of = [&](float px, float py) {
            const float wx = px - sx, wy = py - sy;
            return fmaf(atan2f(sb * wx - cb * wy, -(wx * cb + wy * sb)), inv_dgam, cA);
          };
          const float b00 = bin_of(xlo, ylo), b10 = bin_of(xhi, ylo), b01 = bin_of(xlo, yhi), b11 = bin_of(xhi, yhi);
          // the widest single-pixel window: the tile point closest to the source
          const float qx = fminf(fmaxf(sx, xlo), xhi) - sx, qy = fminf(fmaxf(sy, ylo), yhi) - sy;
          const float x = D * rsqrtf(qx * qx + qy * qy);
          const float h = x * (1.f + x * x * (1.f / 6.f) + 4e-3f) * inv_dgam + 0.02f;
          blo = fminf(fminf(b00, b10), fminf(b01, b11)) - h;
          bhi = fmaxf(fmaxf(b00, b10), fmaxf(b01, b11)) + h;
        }
        b0 = max(0, (int)ceilf(blo));
        b1 = min(A - 1, (int)floorf(bhi));
        if (b0 <= b1) {
          // the driving axis changes every 90 degrees of ray direction: between two rays of one kind less than that
          // apart there is no other kind
          const float s0 = __int_as_float(__ldg(tab + (size_t)kl * A + b0).w);
          const float s1 = __int_as_float(__ldg(tab + (size_t)kl * A + b1).w);
          kinds = (s0 > 0.f ? 2 : 1) | (s1 > 0.f ? 2 : 1);
          if (!par && (float)(b1 - b0) > inv_dgam) kinds = 3;
        }
      }
      const int cnt = min(32, (g.V - kb + kstep - 1) / kstep);
      for (int i = 0; i < cnt; ++i) {
        const int kd = __shfl_sync(kFull, kinds, i), ba = __shfl_sync(kFull, b0, i), be = __shfl_sync(kFull, b1, i);
        if (TWO ? kd == 0 : !(kd & (xphase ? 2 : 1))) continue;
        const size_t row = (size_t)(kb + i * kstep) * A;
        const int4* trow = tab + row;
        const float* srow = sino + row;
        auto ray = [&](const int4& P, float s) {
          const float asc = fabsf(__int_as_float(P.w));
          int i0;
          float f;
          split_fx(ray_U0(P) + (int64_t)dj4 * P.z, i0, f);
          const float w0 = __fsub_rn(1.f, f);
          const int q0 = i0 - qbase;
          const bool p0 = (unsigned)q0 < qlim && w0 != 0.f, p1 = (unsigned)(q0 + 1) < qlim && f != 0.f;
          float* a = kacc + q0 * kBpTile + lane;
          const float v0 = p0 ? a[0] : 0.f, v1 = p1 ? a[kBpTile] : 0.f;
          if (p0) a[0] = fmaf(w0 * asc, s, v0);
          if (p1) a[kBpTile] = fmaf(f * asc, s, v1);
        };
        if (TWO) aim(kd == 2);
        if (kd != 3) {
#pragma unroll 4  // independent table loads and crossings of four rays in flight
          for (int b = ba; b <= be; ++b) ray(__ldg(trow + b), __ldg(srow + b));
        } else if (TWO) {
#pragma unroll 4
          for (int b = ba; b <= be; ++b) {
            const int4 P = __ldg(trow + b);
            aim(__int_as_float(P.w) > 0.f);
            ray(P, __ldg(srow + b));
          }
        } else {
          for (int b = ba; b <= be; ++b) {
            const int4 P = __ldg(trow + b);
            if ((__int_as_float(P.w) > 0.f) == xphase) ray(P, __ldg(srow + b));
          }
        }
      }
    }
    if (!TWO) {
      add_warps(xphase);
      __syncthreads();
    }
  }
  if (TWO) {
    add_warps(false);
    add_warps(true);
  }
}

// Sum of the nsplit partial images in split order.
__global__ void bp_sum_kernel(const float* __restrict__ part, int nsplit, int64_t n, float* __restrict__ img) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float acc = part[i];
  for (int s = 1; s < nsplit; ++s) acc += part[(int64_t)s * n + i];
  img[i] = acc;
}

// Cone adjoint, gather form with the per-ray factor sqrt(v_b^2 + |e_xy|^2) |s_a| (the ray's
// step length per slice) applied once per ray by a pre-pass, and the z crossing of
// consecutive rows stepped exactly in integers.
__global__ void cone_prescale_kernel(GeomDev g, const int4* __restrict__ t0, const float* __restrict__ t2,
                                     float pv_half, const float* __restrict__ sino, float* __restrict__ out) {
  const int64_t m = (int64_t)g.V * g.B * g.A;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int a = (int)(i % g.A);
  const int64_t kb = i / g.A;
  const int b = (int)(kb % g.B), k = (int)(kb / g.B);
  const size_t ci = (size_t)k * g.A + a;
  const float sa = fabsf(__int_as_float(__ldg(t0 + ci).w));
  const float vb = __fmul_rn((float)(2 * b - (g.B - 1)), pv_half);
  out[i] = sino[i] * cone_scale(vb, __ldg(t2 + ci), sa);
}

// As cone_prescale_kernel, written column-major per view ([view][column][row]) for the column
// kernel below, which stages one detector column's rows at a time.
__global__ void cone_prescale_t_kernel(GeomDev g, const int4* __restrict__ t0, const float* __restrict__ t2,
                                       float pv_half, const float* __restrict__ sino, float* __restrict__ out) {
  const int64_t m = (int64_t)g.V * g.B * g.A;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int a = (int)(i % g.A);
  const int64_t kb = i / g.A;
  const int b = (int)(kb % g.B), k = (int)(kb / g.B);
  const size_t ci = (size_t)k * g.A + a;
  const float sa = fabsf(__int_as_float(__ldg(t0 + ci).w));
  const float vb = __fmul_rn((float)(2 * b - (g.B - 1)), pv_half);
  out[ci * g.B + b] = sino[i] * cone_scale(vb, __ldg(t2 + ci), sa);
}

// Cone adjoint, one warp per (x, y) column of the volume: lane l gathers voxels l*VL .. l*VL+VL-1.
// For a view and a detector column, the window, the tap weight and the row pitch are the same
// for the whole warp, so the lanes run the row sweep of backproject3d_kernel in step (there,
// neighbouring lanes are neighbouring x with their own windows and row counts, and about half
// of the lanes idle on average).  The warp first stages the detector column's rows that can reach
// the volume ([view][column][row] sinogram: one coalesced read) in shared memory; each lane then
// sweeps its chunk exactly as backproject3d_kernel<VL> does.  N <= 32 VL, at most kColStrip rows.
// With V4 (B a multiple of 4 and sino_t 16-byte aligned) the strip is staged in 16-byte copies
// from the aligned row at or below its first row.
constexpr int kColStrip = 1024;
constexpr int kColWarps = 8;
template <int VL, bool V4>
__global__ void __launch_bounds__(32 * kColWarps, 4) backproject3d_col_kernel(GeomDev g, const int4* __restrict__ t0,
    const int4* __restrict__ t1, const float2* __restrict__ views, int64_t CzF,
    const float* __restrict__ sino_t, float* __restrict__ vol) {
  // [V] view directions (padded to an even count: the strips start 16-byte aligned), then
  // kColWarps strips of kColStrip rows
  extern __shared__ float2 sv[];
  float* strips = reinterpret_cast<float*>(sv + ((g.V + 1) & ~1));
  for (int k = threadIdx.x; k < g.V; k += blockDim.x) sv[k] = views[k];
  __syncthreads();
  const int N = g.N, A = g.A, B = g.B;
  const int jref = N / 2;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int ix = blockIdx.x * kColWarps + wi, iy = blockIdx.y;
  if (ix >= N) return;  // a whole warp
  float* strip = strips + wi * kColStrip;
  const int z0 = lane * VL;
  const float D = 2.f / (float)N;
  const float px = -1.f + ((float)ix + 0.5f) * D, py = -1.f + ((float)iy + 0.5f) * D;
  const float cA = 0.5f * (float)(A - 1), Bm1 = (float)(B - 1);
  const float Cz = 0.5f * (float)N - 0.5f;
  const float R = (float)(g.sod * (2.0 / N));
  const float kcol = (float)(g.sod / g.du);
  const float kha = (float)(1.3 * (2.0 / N) * g.sod / g.du);
  float acc[VL];
#pragma unroll
  for (int q = 0; q < VL; ++q) acc[q] = 0.f;
  for (int k = 0; k < g.V; ++k) {
    const float cb = sv[k].x, sb = sv[k].y;
    const float depth = R - (cb * px + sb * py);
    const float ucoord = -sb * px + cb * py;
    const float ac = fmaf(ucoord / depth, kcol, cA);
    const float ha = kha / depth + 0.02f;
    const int a0i = max(0, (int)ceilf(ac - ha));
    const int a1i = min(A - 1, (int)floorf(ac + ha));
    for (int a = a0i; a <= a1i; ++a) {
      const size_t ci = (size_t)k * A + a;
      const int4 P = __ldg(t0 + ci);
      const float sa = __int_as_float(P.w);
      const bool xd = sa > 0.f;
      const int j = xd ? ix : iy, q = xd ? iy : ix;
      const int64_t dj = j - jref;
      const float wq = tap_weight(ray_U0(P) + dj * slope_fx(P), q);
      if (wq == 0.f) continue;
      const int4 T1 = __ldg(t1 + ci);
      const int64_t Hh = ((int64_t)T1.y << 32) | (int64_t)(uint32_t)T1.x;
      const int64_t Kk = ((int64_t)T1.w << 32) | (int64_t)(uint32_t)T1.z;
      const float hg = fmaf((float)dj,
                            fmaf(__uint2float_rn((uint32_t)T1.z), 3.552713678800501e-15f,
                                 __int2float_rn(T1.w) * 1.52587890625e-05f),
                            fmaf(__uint2float_rn((uint32_t)T1.x), 2.3283064365386963e-10f, __int2float_rn(T1.y)));
      const float inv_hg = __frcp_rn(hg);
      const float hb = 0.5f * fabsf(inv_hg) * 1.001f + 0.02f;
      const float* scol = sino_t + ci * B;  // this view's detector column, rows contiguous
      if (fabsf(hg) > 1e-3f) {
        // the rows that can reach any voxel of the column (the chunks' bounds, united)
        const float cz0 = 0.5f * fmaf(-Cz, inv_hg, Bm1);
        const float cz1 = 0.5f * fmaf((float)(N - 1) - Cz, inv_hg, Bm1);
        const int sl = max(0, (int)ceilf(fminf(cz0, cz1) - hb));
        const int sh = min(B - 1, (int)floorf(fmaxf(cz0, cz1) + hb));
        if (sl > sh) continue;
        __syncwarp();  // the previous strip is no longer read
        int s0 = sl;   // the row held in strip[0]
        if constexpr (V4) {
          // rows s0 .. 4 floor(sh / 4) + 3: inside the column (B % 4 == 0) and at most B rows
          s0 = sl & ~3;
          const float4* src = reinterpret_cast<const float4*>(scol + s0);
          float4* dst = reinterpret_cast<float4*>(strip);
#pragma unroll 2
          for (int i = lane; i <= (sh - s0) >> 2; i += 32) dst[i] = __ldg(src + i);
        } else {
          for (int i = lane; i <= sh - sl; i += 32) strip[i] = __ldg(scol + sl + i);
        }
        __syncwarp();
        if (z0 >= N) continue;
        // this lane's chunk: the row sweep of backproject3d_kernel, its rows clipped to the strip
        const float bzA = 0.5f * fmaf((float)z0 - Cz, inv_hg, Bm1);
        const float bzB = 0.5f * fmaf((float)(z0 + VL - 1) - Cz, inv_hg, Bm1);
        const int bl = max(sl, (int)ceilf(fminf(bzA, bzB) - hb));
        const int bh = min(sh, (int)floorf(fmaxf(bzA, bzB) + hb));
        if (bl > bh) continue;
        const int dir = hg > 0.f ? 1 : -1;
        const int bfirst = dir > 0 ? bl : bh;
        const float nrow = (float)(bh - bl + 1);
        const int mr = 2 * bfirst - (B - 1);
        const int64_t Zf = CzF + (int64_t)mr * Hh + dj * (((int64_t)mr * Kk) >> 16) - ((int64_t)z0 << 32);
        const float u0 = (float)Zf * 2.3283064365386963e-10f;  // * 2^-32
        const float du = 2.f * fabsf(hg);
        const float* sp = strip + (bfirst - s0);
        // u = fma(rr, du, u0) rises strictly with rr (du > 2e-3 is far above the float spacing
        // of u here), so rr < nrow holds exactly when u < ulim, and each loop below tests u alone
        const float ulim = fmaf(nrow, du, u0);
        float rr = 0.f, u = u0;
        const float lm1 = fminf(-1.f, ulim), l0 = fminf(0.f, ulim);
        while (u < lm1) {
          rr += 1.f;
          sp += dir;
          u = fmaf(rr, du, u0);
        }
        while (u < l0) {  // floor(u) = -1: f = u + 1 to voxel 0
          acc[0] = fmaf(wq * (u + 1.f), *sp, acc[0]);
          rr += 1.f;
          sp += dir;
          u = fmaf(rr, du, u0);
        }
#pragma unroll
        for (int zq = 0; zq < VL; ++zq) {
          const float lz = fminf((float)(zq + 1), ulim);
          while (u < lz) {  // floor(u) = zq
            const float ws = wq * *sp;
            const float f = u - (float)zq;
            acc[zq] = fmaf(-f, ws, acc[zq] + ws);
            if (zq + 1 < VL) acc[zq + 1] = fmaf(f, ws, acc[zq + 1]);
            rr += 1.f;
            sp += dir;
            u = fmaf(rr, du, u0);
          }
        }
        continue;
      }
      if (z0 >= N) continue;
#pragma unroll
      for (int zq = 0; zq < VL; ++zq) {
        const int iz = z0 + zq;
        if (iz >= N) break;
        const float bz = 0.5f * fmaf((float)iz - Cz, inv_hg, Bm1);
        const int bb0 = max(0, (int)ceilf(bz - hb));
        const int bb1 = min(B - 1, (int)floorf(bz + hb));
        int mr = 2 * bb0 - (B - 1);
        int64_t Zb = CzF + (int64_t)mr * Hh, Pk = (int64_t)mr * Kk;
        for (int b = bb0; b <= bb1; ++b, Zb += 2 * Hh, Pk += 2 * Kk) {
          const float wz = tap_weight(Zb + dj * (Pk >> 16), iz);
          if (wz != 0.f) acc[zq] = fmaf(wq * wz, __ldg(scol + b), acc[zq]);
        }
      }
    }
  }
#pragma unroll
  for (int zq = 0; zq < VL; ++zq) {
    const int iz = z0 + zq;
    if (iz < N) vol[((size_t)iz * N + iy) * N + ix] = acc[zq];
  }
}

// As cone_prescale_t_kernel for the tile kernel below: [view][column][row] with kRowPad zero rows before and after
// each column, transposed through shared memory (both sides in runs of 32).
constexpr int kRowPad = 4;
__global__ void cone_prescale_pad_kernel(GeomDev g, const int4* __restrict__ t0, const float* __restrict__ t2,
                                         float pv_half, const float* __restrict__ sino, float* __restrict__ out) {
  __shared__ float tile[32][33];
  const int k = blockIdx.z, a = blockIdx.x * 32 + threadIdx.x, Bp = g.B + 2 * kRowPad;
  float sa = 0.f, L2 = 0.f;
  if (a < g.A) {
    sa = fabsf(__int_as_float(__ldg(t0 + (size_t)k * g.A + a).w));
    L2 = __ldg(t2 + (size_t)k * g.A + a);
  }
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int b = blockIdx.y * 32 + r - kRowPad;
    tile[r][threadIdx.x] = a < g.A && b >= 0 && b < g.B
                               ? sino[((size_t)k * g.B + b) * g.A + a] *
                                     cone_scale(__fmul_rn((float)(2 * b - (g.B - 1)), pv_half), L2, sa)
                               : 0.f;
  }
  __syncthreads();
  const int b = blockIdx.y * 32 + threadIdx.x;
  for (int c = threadIdx.y; c < 32; c += blockDim.y) {
    const int ac = blockIdx.x * 32 + c;
    if (ac < g.A && b < Bp) out[((size_t)k * g.A + ac) * Bp + b] = tile[threadIdx.x][c];
  }
}

// Cone adjoint, plan zc = 0 where it fits (tile_fit): a block owns a 4 x 4 tile of (x, y) and all z.  The two taps of
// a detector column at a slice share the same sum over its rows,
//   S[z] = sum_b hat(u_b - z) s_b,  v[q][z] += (1 - f) S[z],  v[q + 1][z] += f S[z],
// so a warp takes one slice j of the tile and its four transverse places q: it forms S once for a column and adds it
// to the four accumulators with their tap weights (the columns that reach four places are about 5.5, against 2 for
// each place alone).  Lanes are consecutive z (Z groups of 32 per lane).  With a reference row near the middle of
// the warp's z range, whose distance d_ref to the middle voxel is formed exactly in the forward's 32.32 fixed point,
// a lane rounds up to the first row that can reach its voxel (a hundredth of a row of margin), takes that row's
// distance d as db p - dz + d_ref (the row pitch p in two FP32 terms, the difference of the large terms rounded
// once, at the size of the result), and steps by p over the two to four rows whose hat reaches it.  No lane waits
// for another's row count, and the rows of neighbouring lanes are neighbours in memory.
// (In backproject3d_col_kernel each place sweeps the rows of its own columns, every row once per tap, in loops whose
// length differs between lanes.)  Columns, weights and reference rows are formed for four views at a time, eight
// lanes each, and read back from shared memory; two z groups share a packed FP32 instruction.  Rays driven along y
// (slices of constant y, q = x) are gathered first, those driven along x (slices of constant x, q = y) second; the
// two meet in shared memory.
// 501^3 x 60 views x 768^2: 20.08 -> 11.32 ms with the ray scale, error against FP64 6.9e-7 -> 1.8e-7; 256^3 x 40
// views 2285 -> 1010 us, 64^3 x 20 views 113 -> 80 us; bound by instruction issue (80 % active; 33 instructions per column, z group and warp, of them
// about 13 the taps).  Measured beside it: 8 z groups per lane 16.1 ms (distances in 64 bits, 14.1 with 4), 2 z
// groups 16.0, row loads only where the hat reaches 12.4, views tested for their driving axis first 12.5.
struct __align__(16) ColEntry {
  f32x2 w[4];              // tap weights of the four places, each twice
  float p_hi, p_lo, ip, c;  // row pitch, 1 / p, rounding offset: first row db = round(dz ip + c)
  float d_ref;
  int base;                // index of the reference row in the padded sinogram
  int b_ref;
  int kind;                // rows per voxel (2 to 4), + 8 if some row lies off the padded column
};
constexpr float kRoundF = 12582912.f;  // 1.5 2^23: adding it rounds to an integer in the low mantissa bits
template <int Z>
__global__ void __launch_bounds__(512, 2)
    backproject3d_tile_kernel(GeomDev g, const int4* __restrict__ t0, const int4* __restrict__ t1,
                              const float2* __restrict__ views, int64_t CzF, const float* __restrict__ sino_p,
                              float* __restrict__ vol) {
  constexpr unsigned kFull = 0xffffffffu;
  extern __shared__ __align__(16) float tsm[];  // [warp][32] column entries, then the tile [4 y][4 x][zs]
  const int N = g.N, A = g.A, B = g.B, Bp = B + 2 * kRowPad;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, jj = w & 3;
  ColEntry* ent = reinterpret_cast<ColEntry*>(tsm) + 32 * w;
  float* tile = tsm + (size_t)(blockDim.x >> 5) * 32 * (sizeof(ColEntry) / sizeof(float));
  const int zbase = (w >> 2) * 32 * Z, zs = (blockDim.x >> 7) * 32 * Z + 2, zr = zbase + 16 * Z;
  const int x0 = blockIdx.x * 4, y0 = blockIdx.y * 4, jref = N / 2;
  const float D = 2.f / (float)N;
  const float cA = 0.5f * (float)(A - 1), Bm1 = (float)(B - 1), Cz = 0.5f * (float)N - 0.5f;
  const float R = (float)(g.sod * (2.0 / N)), kcol = (float)(g.sod / g.du);
  const float kha = (float)(1.3 * (2.0 / N) * g.sod / g.du);
  const float dz0 = (float)(lane - 16 * Z);
#pragma unroll 1
  for (int phase = 0; phase < 2; ++phase) {
    const int j = (phase ? x0 : y0) + jj, q0 = phase ? y0 : x0;
    f32x2 acc[4][Z / 2];  // z groups 2 i and 2 i + 1
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < Z / 2; ++i) acc[q][i] = 0ull;
    const float pj = -1.f + ((float)j + 0.5f) * D;
    const float pa = -1.f + ((float)q0 + 0.5f) * D, pb = -1.f + ((float)q0 + 3.5f) * D;
    const int64_t dj = j - jref;
    for (int kb = 0; kb < g.V && j < N; kb += 4) {
      const int k = kb + (lane >> 3);
      int a = 1, a1 = 0;
      if (k < g.V) {  // the columns whose window can reach one of the four places
        const float2 cs = __ldg(views + k);
        const float px0 = phase ? pj : pa, py0 = phase ? pa : pj, px1 = phase ? pj : pb, py1 = phase ? pb : pj;
        const float d0 = 1.f / (R - (cs.x * px0 + cs.y * py0)), d1 = 1.f / (R - (cs.x * px1 + cs.y * py1));
        const float c0 = fmaf((cs.x * py0 - cs.y * px0) * d0, kcol, cA), c1 = fmaf((cs.x * py1 - cs.y * px1) * d1, kcol, cA);
        const float ha = kha * fmaxf(d0, d1) + 0.02f;
        a = max(0, (int)ceilf(fminf(c0, c1) - ha)) + (lane & 7);
        a1 = min(A - 1, (int)floorf(fmaxf(c0, c1) + ha));
      }
      while (__any_sync(kFull, a <= a1)) {
        float wq[4] = {0.f, 0.f, 0.f, 0.f};
        int4 P;
        const int ci = k * A + a;
        if (a <= a1) {
          P = __ldg(t0 + ci);
          if ((__int_as_float(P.w) > 0.f) == (phase == 1)) {
            const int64_t uq = ray_U0(P) + dj * slope_fx(P);
#pragma unroll
            for (int q = 0; q < 4; ++q) wq[q] = q0 + q < N ? tap_weight(uq, q0 + q) : 0.f;
          }
        }
        const bool on = wq[0] != 0.f || wq[1] != 0.f || wq[2] != 0.f || wq[3] != 0.f;
        const unsigned todo = __ballot_sync(kFull, on);
        if (on) {
          const int4 Q = __ldg(t1 + ci);
          const int64_t Hh = ((int64_t)Q.y << 32) | (int64_t)(uint32_t)Q.x;
          const int64_t Kk = ((int64_t)Q.w << 32) | (int64_t)(uint32_t)Q.z;
          const int64_t G = ((Hh << 16) + dj * Kk + 32768) >> 16;  // as the forward's; 0 < G < 2^32 (tile_fit)
          ColEntry e;
#pragma unroll
          for (int q = 0; q < 4; ++q) e.w[q] = pack2(wq[q], wq[q]);
          const float gf = __uint2float_rn((unsigned)G);
          e.p_hi = gf * 4.656612873077393e-10f;  // 2 G 2^-32
          e.p_lo = (float)(int)((unsigned)G - (unsigned)gf) * 4.656612873077393e-10f;
          e.ip = __frcp_rn(e.p_hi);
          e.b_ref = __float2int_rn(fmaf((float)zr - Cz, e.ip, 0.5f * Bm1));
          const int64_t u = CzF + (int64_t)(2 * e.b_ref - (B - 1)) * G - ((int64_t)zr << 32);
          e.d_ref = (float)(int)(u >> 4) * 3.725290298461914e-09f;  // 28 fractional bits, |d_ref| < 2
          e.c = fmaf(-1.f - e.d_ref, e.ip, 0.49f);
          e.base = ci * Bp + kRowPad + e.b_ref;
          const int K = (int)ceilf(fmaf(2.f, e.ip, 0.02f));
          const float first = fmaf((float)(-16 * Z), e.ip, e.c) - 1.f, last = fmaf((float)(16 * Z), e.ip, e.c) + 1.f;
          const bool off = (float)e.b_ref + first < (float)-kRowPad || (float)(e.b_ref + K) + last > (float)(B + kRowPad);
          e.kind = max(K, 2) + (off ? 8 : 0);
          ent[__popc(todo & ((1u << lane) - 1))] = e;
        }
        __syncwarp();
        const int n = __popc(todo);
        for (int c = 0; c < n; ++c) {
          const ColEntry& e = ent[c];
          const f32x2 w0 = e.w[0], w1 = e.w[1], w2 = e.w[2], w3 = e.w[3];
          const bool on0 = w0 != 0ull, on1 = w1 != 0ull, on2 = w2 != 0ull, on3 = w3 != 0ull;
          const float p_hi = e.p_hi, p_lo = e.p_lo, ip = e.ip, cc = e.c, d_ref = e.d_ref;
          const float* s = sino_p + (e.base - __float_as_int(kRoundF));
          // rows off the padded column read its zeros: clamps of the row index, where some row needs them
          const int lo = __float_as_int(kRoundF) - kRowPad - e.b_ref, hi = __float_as_int(kRoundF) + B - e.b_ref;
          auto rows = [&](auto kc, auto clamp) {
            constexpr int K = decltype(kc)::value;
#pragma unroll
            for (int i = 0; i < Z / 2; ++i) {
              float S[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const float dz = dz0 + (float)(32 * (2 * i + h));
                const float y = fmaf(dz, ip, cc) + kRoundF;
                const float db = y - kRoundF;
                float d = fmaf(db, p_lo, fmaf(db, p_hi, -dz)) + d_ref;
                int r = __float_as_int(y);
                if constexpr (decltype(clamp)::value) r = min(max(r, lo), hi);
                const float* sp = s + r;
                S[h] = 0.f;
#pragma unroll
                for (int t = 0; t < K; ++t) {
                  const float m = fabsf(d);
                  const float sv = __ldg(sp + t);  // loaded in any case: all loads in flight at once
                  if (m < 1.f) S[h] = fmaf(1.f - m, sv, S[h]);
                  d += p_hi;
                }
              }
              const f32x2 S2 = pack2(S[0], S[1]);
              // only the places the column reaches (0 times a value that is not finite would spread it)
              if (on0) fma2(acc[0][i], w0, S2);
              if (on1) fma2(acc[1][i], w1, S2);
              if (on2) fma2(acc[2][i], w2, S2);
              if (on3) fma2(acc[3][i], w3, S2);
            }
          };
          const int kind = e.kind;
          if (kind == 2) rows(std::integral_constant<int, 2>{}, std::false_type{});
          else if (kind == 3) rows(std::integral_constant<int, 3>{}, std::false_type{});
          else if (kind == 4) rows(std::integral_constant<int, 4>{}, std::false_type{});
          else rows(std::integral_constant<int, 4>{}, std::true_type{});
        }
        __syncwarp();  // the entries are no longer read
        a += 8;
      }
    }
    if (phase) __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < Z / 2; ++i) {
        float* t = tile + (phase ? q * 4 + jj : jj * 4 + q) * zs + zbase + lane + 64 * i;
        float v0, v1;
        unpack2(acc[q][i], v0, v1);
        t[0] = phase ? t[0] + v0 : v0;
        t[32] = phase ? t[32] + v1 : v1;
      }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 16 * N; e += blockDim.x) {
    const int c = e & 15, z = e >> 4, x = x0 + (c & 3), y = y0 + (c >> 2);
    if (x < N && y < N) vol[((size_t)z * N + y) * N + x] = tile[c * zs + z];
  }
}

// Launch bound: eight blocks of 128 threads per SM (at most 64 registers).  The 32-voxel chunk
// then spills a little but runs fastest (501^3: 30.1 ms against 32.1 ms for 16 voxels without a
// bound, whose 92 registers leave fewer warps resident); the smaller chunks fit in 64 registers.
template <int ZC>
__global__ void __launch_bounds__(128, 8) backproject3d_kernel(GeomDev g, const int4* __restrict__ t0, const int4* __restrict__ t1,
                            const float2* __restrict__ views, int64_t CzF,
                            const float* __restrict__ sino_s, float* __restrict__ vol) {
  extern __shared__ float2 sv[];
  for (int k = threadIdx.y * blockDim.x + threadIdx.x; k < g.V; k += blockDim.x * blockDim.y)
    sv[k] = views[k];
  __syncthreads();
  const int N = g.N, A = g.A, B = g.B;
  const int jref = N / 2;
  const int ix = blockIdx.x * blockDim.x + threadIdx.x;
  const int iy = blockIdx.y * blockDim.y + threadIdx.y;
  const int z0 = blockIdx.z * ZC;
  if (ix >= N || iy >= N) return;
  const float D = 2.f / (float)N;
  const float px = -1.f + ((float)ix + 0.5f) * D, py = -1.f + ((float)iy + 0.5f) * D;
  const float cA = 0.5f * (float)(A - 1), Bm1 = (float)(B - 1);
  const float Cz = 0.5f * (float)N - 0.5f;
  const float R = (float)(g.sod * (2.0 / N));
  const float kcol = (float)(g.sod / g.du);
  const float kha = (float)(1.3 * (2.0 / N) * g.sod / g.du);
  float acc[ZC];
#pragma unroll
  for (int q = 0; q < ZC; ++q) acc[q] = 0.f;
  for (int k = 0; k < g.V; ++k) {
    const float cb = sv[k].x, sb = sv[k].y;
    const float depth = R - (cb * px + sb * py);
    const float ucoord = -sb * px + cb * py;
    const float ac = fmaf(ucoord / depth, kcol, cA);
    const float ha = kha / depth + 0.02f;
    const int a0i = max(0, (int)ceilf(ac - ha));
    const int a1i = min(A - 1, (int)floorf(ac + ha));
    for (int a = a0i; a <= a1i; ++a) {
      const size_t ci = (size_t)k * A + a;
      const int4 P = __ldg(t0 + ci);
      const float sa = __int_as_float(P.w);
      const bool xd = sa > 0.f;
      const int j = xd ? ix : iy, q = xd ? iy : ix;
      const int64_t dj = j - jref;
      const float wq = tap_weight(ray_U0(P) + dj * slope_fx(P), q);
      if (wq == 0.f) continue;
      const int4 T1 = __ldg(t1 + ci);
      const int64_t Hh = ((int64_t)T1.y << 32) | (int64_t)(uint32_t)T1.x;
      const int64_t Kk = ((int64_t)T1.w << 32) | (int64_t)(uint32_t)T1.z;
      // z pitch of this column's rows at slice j, (Hh 2^16 + dj Kk) / 2^48, from the 32-bit
      // halves in FP32: it only bounds the rows searched below (with a 0.1 % + 0.02-row
      // margin), the weights come from the exact fixed-point crossings
      const float hg = fmaf((float)dj,
                            fmaf(__uint2float_rn((uint32_t)T1.z), 3.552713678800501e-15f,
                                 __int2float_rn(T1.w) * 1.52587890625e-05f),
                            fmaf(__uint2float_rn((uint32_t)T1.x), 2.3283064365386963e-10f, __int2float_rn(T1.y)));
      const float inv_hg = __frcp_rn(hg);
      const float hb = 0.5f * fabsf(inv_hg) * 1.001f + 0.02f;
      const float* scol = sino_s + (size_t)k * B * A + a;
      if (fabsf(hg) > 1e-3f) {
        // One sweep over the rows that can reach this z-chunk, in increasing z: a row's
        // crossing u (in voxels, relative to the chunk's first voxel z0) gives 1 - f to voxel
        // floor(u) and f to floor(u) + 1 (the forward's taps), so while the voxel loop below is
        // unrolled every row lands in registers known at compile time.  The first row's
        // crossing is formed exactly in the forward's 32.32 fixed point; the following ones
        // step by the row pitch 2 |hg| in FP32 (one FMA from the first, no accumulation),
        // which keeps them within a few 1e-6 voxel of the forward's (|u| < ZC + 2): the weights
        // match the forward's to FP32 rounding.  With |pitch| > 1e-3 voxel per row the
        // crossings are strictly increasing.  The rows are those of the per-voxel windows
        // below, united over the chunk.
        const float bzA = 0.5f * fmaf((float)z0 - Cz, inv_hg, Bm1);
        const float bzB = 0.5f * fmaf((float)(z0 + ZC - 1) - Cz, inv_hg, Bm1);
        const int bl = max(0, (int)ceilf(fminf(bzA, bzB) - hb));
        const int bh = min(B - 1, (int)floorf(fmaxf(bzA, bzB) + hb));
        if (bl > bh) continue;
        const int dir = hg > 0.f ? 1 : -1;
        const int bfirst = dir > 0 ? bl : bh;
        const float nrow = (float)(bh - bl + 1);
        const int mr = 2 * bfirst - (B - 1);
        const int64_t Zf = CzF + (int64_t)mr * Hh + dj * (((int64_t)mr * Kk) >> 16) - ((int64_t)z0 << 32);
        const float u0 = (float)Zf * 2.3283064365386963e-10f;  // * 2^-32
        const float du = 2.f * fabsf(hg);
        const float* sp = scol + (ptrdiff_t)bfirst * A;
        const ptrdiff_t step = (ptrdiff_t)dir * A;
        float rr = 0.f, u = u0;
        while (rr < nrow && u < -1.f) {
          rr += 1.f;
          sp += step;
          u = fmaf(rr, du, u0);
        }
        while (rr < nrow && u < 0.f) {  // floor(u) = -1: f = u + 1 to voxel 0
          acc[0] = fmaf(wq * (u + 1.f), __ldg(sp), acc[0]);
          rr += 1.f;
          sp += step;
          u = fmaf(rr, du, u0);
        }
#pragma unroll
        for (int zq = 0; zq < ZC; ++zq) {
          while (rr < nrow && u < (float)(zq + 1)) {  // floor(u) = zq
            const float ws = wq * __ldg(sp);
            const float f = u - (float)zq;
            acc[zq] = fmaf(-f, ws, acc[zq] + ws);
            if (zq + 1 < ZC) acc[zq + 1] = fmaf(f, ws, acc[zq + 1]);
            rr += 1.f;
            sp += step;
            u = fmaf(rr, du, u0);
          }
        }
        continue;
      }
#pragma unroll
      for (int zq = 0; zq < ZC; ++zq) {
        const int iz = z0 + zq;
        if (iz >= N) break;
        const float bz = 0.5f * fmaf((float)iz - Cz, inv_hg, Bm1);
        const int bb0 = max(0, (int)ceilf(bz - hb));
        const int bb1 = min(B - 1, (int)floorf(bz + hb));
        int mr = 2 * bb0 - (B - 1);
        int64_t Zb = CzF + (int64_t)mr * Hh, Pk = (int64_t)mr * Kk;
        for (int b = bb0; b <= bb1; ++b, Zb += 2 * Hh, Pk += 2 * Kk) {
          const float wz = tap_weight(Zb + dj * (Pk >> 16), iz);
          if (wz != 0.f) acc[zq] = fmaf(wq * wz, __ldg(scol + (size_t)b * A), acc[zq]);
        }
      }
    }
  }
#pragma unroll
  for (int zq = 0; zq < ZC; ++zq) {
    const int iz = z0 + zq;
    if (iz < N) vol[((size_t)iz * N + iy) * N + ix] = acc[zq];
  }
}


// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int check_geom(const inrct_geom* geom, const inrct_grid* grid) {
  INRCT_REQUIRE(geom && grid, "geometry and grid descriptors must not be NULL");
  INRCT_REQUIRE(grid->N > 0 && grid->N <= 4096, "grid side N=%d out of range (1..4096)", grid->N);
  INRCT_REQUIRE(grid->fov == 0 || grid->fov == 1, "grid fov=%d must be 0 or 1", grid->fov);
  INRCT_REQUIRE(geom->n_views > 0 && geom->n_views <= 4096, "n_views=%d out of range (1..4096)",
                geom->n_views);
  INRCT_REQUIRE(geom->n_bins_u > 0 && geom->n_bins_u <= 16384, "n_bins_u=%d out of range",
                geom->n_bins_u);
  INRCT_REQUIRE(geom->du > 0, "du must be positive");
  if (geom->kind == INRCT_PAR2D || geom->kind == INRCT_FAN2D) {
    INRCT_REQUIRE(grid->d == 2, "2-D geometry needs a 2-D grid (d=%d)", grid->d);
  } else if (geom->kind == INRCT_CONE3D) {
    INRCT_REQUIRE(grid->d == 3, "cone geometry needs a 3-D grid (d=%d)", grid->d);
    INRCT_REQUIRE(geom->n_bins_v > 0 && geom->n_bins_v <= 16384, "n_bins_v=%d out of range",
                  geom->n_bins_v);
    INRCT_REQUIRE(geom->dv > 0, "dv must be positive");
  } else {
    set_error("unknown geometry kind %d", geom->kind);
    return INRCT_ERR_INVALID_ARG;
  }
  if (geom->kind != INRCT_PAR2D) {
    INRCT_REQUIRE(geom->sod > 0 && geom->sdd > geom->sod,
                  "need 0 < sod < sdd (sod=%g, sdd=%g)", geom->sod, geom->sdd);
    // the source must lie outside the grid's circumscribed circle/sphere
    const double rmax = 0.5 * grid->N * sqrt((double)grid->d);
    INRCT_REQUIRE(geom->sod > rmax, "source inside the grid (sod=%g <= %g pixels)", geom->sod,
                  rmax);
  }
  if (geom->kind == INRCT_CONE3D) {
    // z must never be the driving axis: |e_z| < max(|e_x|, |e_y|) on every ray
    const double vmax = 0.5 * (geom->n_bins_v - 1) * geom->dv;
    if (!(vmax < geom->sod / sqrt(2.0) * 0.999)) {
      set_error("cone angle too wide: z would drive some rays (unsupported)");
      return INRCT_ERR_UNSUPPORTED;
    }
  }
  return INRCT_OK;
}

GeomDev to_dev(const inrct_geom* geom, const inrct_grid* grid) {
  GeomDev g;
  g.kind = geom->kind;
  g.N = grid->N;
  g.V = geom->n_views;
  g.A = geom->n_bins_u;
  g.B = geom->kind == INRCT_CONE3D ? geom->n_bins_v : 1;
  g.du = geom->du;
  g.dv = geom->dv;
  g.sod = geom->sod;
  g.sdd = geom->sdd;
  g.angle0 = geom->angle0;
  g.span = geom->angle_span;
  return g;
}

int64_t num_rays(const inrct_geom* geom) {
  if (!geom) return 0;
  const int64_t rows = geom->kind == INRCT_CONE3D ? geom->n_bins_v : 1;
  return (int64_t)geom->n_views * rows * geom->n_bins_u;
}

// Ray tables of one geometry (built by the projection or the adjoint, in a grad_step by the
// projection for both).
static void tables_layout(const inrct_geom* geom, Carver& c, ProjTables* t) {
  const bool cone = geom->kind == INRCT_CONE3D;
  const int64_t entries = cone ? (int64_t)geom->n_views * geom->n_bins_u : num_rays(geom);
  t->tab0 = c.take<int4>(entries);
  t->tab1 = cone ? c.take<int4>(entries) : nullptr;
  t->tab2 = cone ? c.take<float>(entries) : nullptr;
  t->views = c.take<float2>(geom->n_views);
  t->sums = nullptr;
}
static unsigned table_blocks(int V, int A) { return ceil_div(V, kTabViews) * ceil_div(A, kTabBins); }
// Their checksums, last in a workspace.
static void sums_layout(const inrct_geom* geom, Carver& c, ProjTables* t) {
  t->sums = c.take<uint2>((size_t)geom->n_views * ceil_div(geom->n_bins_u, kTabBins));
}

// Fingerprint of a geometry: FNV-1a over the geometry and the grid.
static unsigned long long tables_fp(const GeomDev& g) {
  unsigned long long h = 1469598103934665603ull;
  auto mix = [&](const void* p, size_t n) {
    const unsigned char* b = static_cast<const unsigned char*>(p);
    for (size_t i = 0; i < n; ++i) h = (h ^ b[i]) * 1099511628211ull;
  };
  mix(&g.kind, sizeof(int) * 5);
  const double dd[6] = {g.du, g.dv, g.sod, g.sdd, g.angle0, g.span};
  mix(dd, sizeof(dd));
  return h;
}

size_t tables_bytes(const inrct_geom* geom) {
  Carver c(nullptr, 0);
  ProjTables t;
  tables_layout(geom, c, &t);
  sums_layout(geom, c, &t);
  return c.off + 256;
}

int place_tables(const inrct_geom* geom, const inrct_grid* grid, void* ws, size_t ws_bytes, ProjTables* t) {
  INRCT_TRY(check_geom(geom, grid));
  Carver c(ws, ws_bytes);
  tables_layout(geom, c, t);
  sums_layout(geom, c, t);
  if (!ws || !c.ok) {
    set_error("ray tables: workspace of %zu bytes too small", ws_bytes);
    return INRCT_ERR_WORKSPACE;
  }
  return INRCT_OK;
}

static TableArgs table_args(const GeomDev& g, const ProjTables& t) {
  return TableArgs{t, tables_fp(g), table_blocks(g.V, g.A)};
}

static int build_tables(const GeomDev& g, const ProjTables& t, cudaStream_t st) {
  const TableArgs a = table_args(g, t);
  tables_kernel<<<a.blocks, kTabThreads, 0, st>>>(g, a);
  INRCT_CHECK_LAUNCH("ray table");
  return INRCT_OK;
}

// Per-call workspace: [ray tables unless given], transposed image (P only), loss partials (P only).
struct ProjWs {
  ProjTables t;
  float* imgT;
  double* loss_part;
  float* bp_part;  // 2-D adjoint: partial images of the view splits (NULL: one split)
  int bp_splits;
  float* sino_s;   // cone adjoint: the sinogram times each ray's step length
};

// Default number of view splits of the 2-D adjoint (see backproject2d_tile_kernel).
static int default_bp_splits(const inrct_geom* geom, const inrct_grid* grid) {
  if (geom->kind == INRCT_CONE3D) return 1;
  const int tiles = ceil_div(grid->N, kBpTile) * ceil_div(grid->N, kBpTile);
  const int want = ceil_div(kBpTargetBlocks, tiles);
  const int most = std::max(1, geom->n_views / kBpWarps);
  return std::max(1, std::min(want, most));
}

// ---------------------------------------------------------------------------
// Launch plans and the autotuner (inrct_tune)
//
// A plan fixes the launch shape of P and P^T for one geometry: the ray segments per
// block of the forward (2-D 4, 8 or 16; cone 2, 4 or 8, or 1, the cone default: whole rays,
// one warp per detector column, project3d_cols_kernel, or in patches of kRowsPerBlock detector
// rows, project3d_rows_kernel; by default the one expected to be faster (cols_faster), when tuned
// the one that was, when pinned columns where they fit; 501^3 P 18.5 ms with 2 segments, 9.36 and
// 14.3 ms), the view splits of the 2-D
// adjoint (1 up to twice the default, at most one split per 8 views) and the voxels per
// thread along z of the cone adjoint (4, 8, 16 or 32; 0 selects backproject3d_tile_kernel, 4 x 4 tiles
// of (x, y), where tile_fit, else backproject3d_col_kernel, one warp per (x, y) column: N <= 512, at
// most kColStrip detector rows; 501^3 P^T 30.1 ms with 32 voxels per thread, 11.3 and 20.1 ms).
// Without tuning the defaults above apply;
// tune_impl times every candidate on the caller's stream and keeps the fastest in a
// process-wide table keyed by the geometry's kind and sizes and by which kernels its plans
// mean (PlanKey), which every later call consults.  Workspaces are sized for the largest candidate,
// so a workspace sized before tuning stays valid after it.
// ---------------------------------------------------------------------------
static int max_bp_splits(const inrct_geom* geom, const inrct_grid* grid) {
  if (geom->kind == INRCT_CONE3D) return 1;
  const int most = std::max(1, geom->n_views / kBpWarps);
  return std::max(1, std::min(most, 2 * default_bp_splits(geom, grid)));
}

// The cone adjoint's column kernel (plan zc = 0: one warp per (x, y) column) takes volumes of
// side N <= 512 and detector columns of at most kColStrip rows.
static bool col_kernel_fits(const inrct_geom* geom, const inrct_grid* grid) {
  return geom->kind == INRCT_CONE3D && grid->N <= 512 && geom->n_bins_v <= kColStrip;
}

// Where the tile kernel runs under plan zc = 0 (which needs N <= 512): N >= 64 (4 warps per 128 voxels of z, at most
// 16), row pitches within [1/2, 2) voxel throughout the volume (two to four rows reach a voxel, 32-bit pitch) and a
// padded sinogram of less than 2^31 values (32-bit indices).
constexpr int kTileZ = 4;
static bool tile_fit(const inrct_geom* geom, const inrct_grid* grid) {
  if (!col_kernel_fits(geom, grid) || grid->N < 64) return false;
  const double reach = 0.7072 * (grid->N + 8) / geom->sod;
  return geom->dv * (1.0 - reach) >= 0.51 && geom->dv * (1.0 + reach) < 1.98 &&
         (int64_t)geom->n_views * geom->n_bins_u * (geom->n_bins_v + 2 * kRowPad) < ((int64_t)1 << 31) - (1 << 20);
}

// The column form of the cone projector (project3d_cols_kernel): voxels per column of the volume's z-fastest copy,
// zeros on both sides of a warp's interpolated column (four row groups plus the margin of its range test), rows
// per lane, and its shared memory.
struct ColsPlan {
  int Zp, pad, R, chunks;
  size_t smem;
};
static ColsPlan cols_plan(const inrct_geom* geom, const inrct_grid* grid) {
  ColsPlan c;
  const int N = grid->N;
  c.Zp = (N + 3) & ~3;
  // largest z pitch of a detector row, in voxels, where a ray is within a pixel of the volume
  const double pitch = geom->dv * (geom->sod + 0.7072 * (N + 2)) / geom->sod;
  c.pad = (int)std::min(1e6, 132.0 * pitch + 8.0) & ~3;
  const int groups = ceil_div(geom->n_bins_v, 32);
  c.chunks = ceil_div(groups, 12);
  const int per = ceil_div(groups, c.chunks);
  c.R = per <= 4 ? 4 : per <= 8 ? 8 : 12;
  c.smem = sizeof(float) * kColsPerBlock * ((size_t)c.Zp + 2 * (size_t)c.pad + 32 * c.R + 1);
  return c;
}
// Where the column form can run: N >= 128 (100^3 x 20 views 96 us by row patches, 103 by columns), N <= 1024 (32-bit
// offsets into the copy), at least 32 detector rows (a warp's lanes are rows), rows no finer than 1e-4 voxel (row
// numbers at the volume's edges fit an int), and a column of the volume with its zeros in shared memory.  With
// N >= 32 every crossing within a pixel of the volume lies in front of the source (sod > 0.866 N), so the row pitch is
// positive.
static bool cols_fit(const inrct_geom* geom, const inrct_grid* grid) {
  return geom->kind == INRCT_CONE3D && grid->N >= 128 && grid->N <= 1024 && geom->n_bins_v >= 32 && geom->dv >= 1e-4 &&
         cols_plan(geom, grid).smem <= 100 * 1024;
}
// Where it is expected to be faster than the row patches, by an estimate of both calls in us.  A warp's slice costs the
// column form a latency (few warps: 300 ns, and per piece of 128 voxels and group of 128 rows) or its share of the chip
// (many), whichever is more, whether the detector's rows are few or many; the row patches pay per ray.  So columns
// win on scans of many rows and views (501^3 x 60 views x 768^2: 9.36 ms, row patches 14.28; 256^3 x 40 views x 384^2:
// 884 and 1423 us) and lose on short detectors, coarse row pitches and few columns (501^3 x 6 views x 752 x 32: 664 and
// 442 us; 256^3 x 2 views x 384^2: 282 and 156 us).  Fitted to 875 scans of 128^3 to 1024^3, 1 to 120 views, 32 to 2000
// rows of 1/4 to 8 voxels, timed by both: the form chosen is at most 17 % slower than the row patches (2 % of the
// scans by more than 3 %), 20 % than the columns, 0.3 % than the better one on average.
static bool cols_faster(const inrct_geom* geom, const inrct_grid* grid) {
  const double N = grid->N, B = geom->n_bins_v, z = std::min(N, B * geom->dv);
  const double rows = std::min(B, 1.05 * N / geom->dv + 1), chunks = cols_plan(geom, grid).chunks;  // rows that meet the volume
  const double columns = geom->n_views * std::min((double)geom->n_bins_u, 1.3 * N / geom->du);
  const int R = cols_plan(geom, grid).R;
  const double fours = ceil(rows / 128), pieces = ceil(std::min(z, std::min(32.0 * R, B) * geom->dv) / 128);
  const double patches = 2.0e-6 * N * N * N + N * (0.31 + columns * (1.3e-6 * rows + 2.9e-8 * B));
  const double latency = 0.30 + 0.14 * pieces + 0.12 * std::min(fours, R / 4.0);
  // beyond 320^3 the copy does not stay in L2
  const double share = columns * (5.4e-5 * chunks + (N > 320 ? 4.7e-5 : 3.1e-5) * (ceil(z / 128) + chunks - 1) + 5.1e-5 * fours);
  return 2.4e-6 * N * N * N + N * sqrt(latency * latency + share * share) < patches;
}

static ProjPlan default_plan(const inrct_geom* geom, const inrct_grid* grid) {
  ProjPlan p;
  p.seg = geom->kind == INRCT_CONE3D ? 1 : 8;
  p.cols = cols_fit(geom, grid) && cols_faster(geom, grid);
  p.bp_splits = default_bp_splits(geom, grid);
  p.zc = col_kernel_fits(geom, grid) ? 0 : 8;
  return p;
}

// A plan holds for the scans of one kind and set of sizes that its launch shapes mean the same kernels for: plan
// seg = 1 and zc = 0 stand for one kernel or another by the row pitch and the source distance as well.
typedef std::tuple<int, int, int, int, int, bool, bool> PlanKey;

static PlanKey plan_key(const inrct_geom* geom, const inrct_grid* grid) {
  return PlanKey(geom->kind, grid->N, geom->n_views, geom->n_bins_u, geom->kind == INRCT_CONE3D ? geom->n_bins_v : 1,
                 cols_fit(geom, grid), tile_fit(geom, grid));
}

static std::mutex g_plan_mu;
static std::map<PlanKey, ProjPlan> g_plans;

bool plan_lookup(const inrct_geom* geom, const inrct_grid* grid, ProjPlan* out) {
  std::lock_guard<std::mutex> lk(g_plan_mu);
  auto it = g_plans.find(plan_key(geom, grid));
  if (it == g_plans.end()) {
    *out = default_plan(geom, grid);
    return false;
  }
  *out = it->second;
  return true;
}

void plan_reset() {
  std::lock_guard<std::mutex> lk(g_plan_mu);
  g_plans.clear();
}

int plan_set(const inrct_geom* geom, const inrct_grid* grid, const ProjPlan& p) {
  INRCT_TRY(check_geom(geom, grid));
  const bool cone = geom->kind == INRCT_CONE3D;
  const bool seg_ok = cone ? (p.seg == 1 || p.seg == 2 || p.seg == 4 || p.seg == 8)
                           : (p.seg == 4 || p.seg == 8 || p.seg == 16);
  INRCT_REQUIRE(seg_ok, "segments per ray %d not a candidate for this geometry", p.seg);
  INRCT_REQUIRE(p.bp_splits >= 1 && p.bp_splits <= max_bp_splits(geom, grid), "view splits %d out of range (1..%d)",
                p.bp_splits, max_bp_splits(geom, grid));
  INRCT_REQUIRE(p.zc == 4 || p.zc == 8 || p.zc == 16 || p.zc == 32 || (p.zc == 0 && (!cone || col_kernel_fits(geom, grid))),
                "voxels per thread along z %d not 4, 8, 16 or 32 (or 0: the column kernel, N <= 512 and at most %d "
                "detector rows)", p.zc, kColStrip);
  ProjPlan q = p;
  q.cols = cols_fit(geom, grid);
  std::lock_guard<std::mutex> lk(g_plan_mu);
  g_plans[plan_key(geom, grid)] = q;
  return INRCT_OK;
}

static ProjPlan plan_for(const inrct_geom* geom, const inrct_grid* grid) {
  ProjPlan p;
  plan_lookup(geom, grid, &p);
  return p;
}

static size_t proj_layout(const inrct_geom* geom, const inrct_grid* grid, void* ws, size_t cap,
                          ProjWs* out, bool forward, bool with_tables, bool cols, bool* ok, bool sums = true) {
  Carver c(ws, cap);
  const bool cone = geom->kind == INRCT_CONE3D;
  ProjWs w;
  if (with_tables) tables_layout(geom, c, &w.t);
  // the transposed image, or the volume's z-fastest copy with padded columns
  const size_t img_floats = cols ? (size_t)grid->N * grid->N * cols_plan(geom, grid).Zp : (size_t)grid_points(grid);
  w.imgT = forward ? c.take<float>(img_floats) : nullptr;
  const int64_t blocks = cone ? (int64_t)ceil_div(geom->n_bins_u, 32) * geom->n_bins_v * geom->n_views
                              : (int64_t)ceil_div(num_rays(geom), 32);
  w.loss_part = forward ? c.take<double>(blocks) : nullptr;
  const int bp_max = forward ? 1 : max_bp_splits(geom, grid);  // any plan's split count fits
  w.bp_splits = 1;
  w.bp_part = bp_max > 1 ? c.take<float>((size_t)bp_max * grid_points(grid)) : nullptr;
  // the scaled sinogram, with zero rows around each column for the tile kernel (cols)
  const size_t sino_floats = cols ? (size_t)geom->n_views * geom->n_bins_u * (geom->n_bins_v + 2 * kRowPad)
                                  : (size_t)num_rays(geom);
  w.sino_s = (!forward && cone) ? c.take<float>(sino_floats) : nullptr;
  if (with_tables && sums) sums_layout(geom, c, &w.t);  // without them every call builds the tables
  if (out) *out = w;
  if (ok) *ok = c.ok;
  return c.off + 256;
}

size_t project_ws_bytes(const inrct_geom* geom, const inrct_grid* grid, bool with_tables) {
  if (check_geom(geom, grid) != INRCT_OK) return 0;
  return proj_layout(geom, grid, nullptr, 0, nullptr, true, with_tables, cols_fit(geom, grid), nullptr);
}

size_t backproject_ws_bytes(const inrct_geom* geom, const inrct_grid* grid, bool with_tables) {
  if (check_geom(geom, grid) != INRCT_OK) return 0;
  return proj_layout(geom, grid, nullptr, 0, nullptr, false, with_tables, tile_fit(geom, grid), nullptr);
}

// Per-geometry cone constants shared by P and P^T: half the row pitch (world
// units) and the z index of the grid's lower face in 32.32 fixed point.
static void cone_consts(const GeomDev& g, float* pv_half, int64_t* CzF) {
  const double D = 2.0 / g.N;
  *pv_half = (float)(0.5 * g.dv * D * g.sdd / g.sod);
  *CzF = (int64_t)llrint((0.5 * g.N - 0.5) * 4294967296.0);
}

static int project_run(const inrct_geom* geom, const inrct_grid* grid, const float* image, float* sino,
                       const float* y, float* resid, double* loss_out, void* ws, size_t ws_bytes,
                       cudaStream_t st, const ProjTables* pre, const ProjPlan& plan, bool sums = true) {
  INRCT_TRY(check_geom(geom, grid));
  INRCT_REQUIRE(image && sino, "image and sino must not be NULL");
  INRCT_REQUIRE(!y || (resid && loss_out), "y given: resid and loss_out must not be NULL");
  ProjWs w;
  bool ok;
  // the column form also wants its padded columns to fit the workspace and 16-byte loads from it
  bool cols = plan.seg == 1 && plan.cols && cols_fit(geom, grid);
  size_t need = 0;
  if (cols) {
    need = proj_layout(geom, grid, ws, ws_bytes, &w, true, pre == nullptr, true, &ok, sums);
    cols = ok && reinterpret_cast<uintptr_t>(w.imgT) % 16 == 0;
  }
  if (!cols) need = proj_layout(geom, grid, ws, ws_bytes, &w, true, pre == nullptr, false, &ok, sums);
  if (!ws || !ok) {
    set_error("project: workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  const GeomDev g = to_dev(geom, grid);
  if (pre) w.t = *pre;
  const int N = g.N;
  if (g.kind == INRCT_CONE3D) INRCT_TRY(build_tables(g, w.t, st));  // 2-D: below, with the transpose
  dim3 tb(32, 8);
  if (cols) {
    float pvh;
    int64_t CzF;
    cone_consts(g, &pvh, &CzF);
    const ColsPlan c = cols_plan(geom, grid);
    transpose_z_kernel<<<dim3(ceil_div(N, 32), ceil_div(c.Zp, 32), N), tb, 0, st>>>(image, w.imgT, N, c.Zp);
    INRCT_CHECK_LAUNCH("transpose");
    const dim3 grd(ceil_div(g.A, kColsPerBlock), g.V, c.chunks);
    auto launch = [&](auto kernel) {
      const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem);
      if (e != cudaSuccess) {
        set_error("project3d: shared memory attribute: %s", cudaGetErrorString(e));
        return INRCT_ERR_CUDA;
      }
      kernel<<<grd, 32 * kColsPerBlock, c.smem, st>>>(w.t.tab0, w.t.tab1, w.t.tab2, g.A, g.B, N, c.Zp, c.pad, pvh, CzF,
                                                      w.imgT, sino, y, resid, w.loss_part);
      INRCT_CHECK_LAUNCH("project3d (columns)");
      return INRCT_OK;
    };
    INRCT_TRY(c.R == 4 ? launch(project3d_cols_kernel<4>)
                       : c.R == 8 ? launch(project3d_cols_kernel<8>) : launch(project3d_cols_kernel<12>));
    return y ? reduce_f64(w.loss_part, (int64_t)grd.x * grd.y * grd.z, loss_out, st) : INRCT_OK;
  }
  if (g.kind == INRCT_CONE3D) {
    transpose_xy_kernel<<<dim3(ceil_div(N, 32), ceil_div(N, 32), N), tb, 0, st>>>(image, w.imgT, N);
    INRCT_CHECK_LAUNCH("transpose");
    float pvh;
    int64_t CzF;
    cone_consts(g, &pvh, &CzF);
    if (plan.seg == 1) {  // project3d_rows_kernel
      dim3 grr(ceil_div(g.A, 32), g.V, ceil_div(g.B, kRowsPerBlock));
#define INRCT_PR(OFF32)                                                                                 \
  project3d_rows_kernel<OFF32><<<grr, dim3(32, kRowsPerBlock), 0, st>>>(w.t.tab0, w.t.tab1, w.t.tab2, g.A, g.B, N, \
                                                                      pvh, CzF, image, w.imgT, sino, y, resid,  \
                                                                      w.loss_part)
      if (N <= 1024) INRCT_PR(true);
      else INRCT_PR(false);
#undef INRCT_PR
      INRCT_CHECK_LAUNCH("project3d (rows)");
      if (y) {
        INRCT_TRY(reduce_f64(w.loss_part, (int64_t)grr.x * grr.y * grr.z, loss_out, st));
      }
      return INRCT_OK;
    }
    dim3 grd(ceil_div(g.A, 32), g.V, g.B);
#define INRCT_P3(SEG)                                                                                  \
  project3d_kernel<SEG><<<grd, dim3(32, SEG), 0, st>>>(w.t.tab0, w.t.tab1, w.t.tab2, g.A, g.B, N, pvh, CzF, \
                                                       image, w.imgT, sino, y, resid, w.loss_part)
    if (plan.seg == 2) INRCT_P3(2);
    else if (plan.seg == 8) INRCT_P3(8);
    else INRCT_P3(4);
#undef INRCT_P3
    INRCT_CHECK_LAUNCH("project3d");
    if (y) {
      INRCT_TRY(reduce_f64(w.loss_part, (int64_t)grd.x * grd.y * grd.z, loss_out, st));
    }
  } else {
    const int64_t m = num_rays(geom);
    const unsigned nb = ceil_div(m, 32);
    const TableArgs a = table_args(g, w.t);
    prep2d_kernel<<<a.blocks + ceil_div(N, 32) * ceil_div(N, 32), kTabThreads, 0, st>>>(g, a, image, w.imgT);
    INRCT_CHECK_LAUNCH("projection tables and transpose");
#define INRCT_P2(SEG)                                                                                       \
  project2d_kernel<SEG><<<nb, dim3(32, SEG), 0, st>>>(w.t.tab0, (int)m, N, image, w.imgT, sino, y, resid, \
                                                      w.loss_part)
    if (plan.seg == 4) INRCT_P2(4);
    else if (plan.seg == 16) INRCT_P2(16);
    else INRCT_P2(8);
#undef INRCT_P2
    INRCT_CHECK_LAUNCH("project2d");
    if (y) {
      INRCT_TRY(reduce_f64(w.loss_part, nb, loss_out, st));
    }
  }
  return INRCT_OK;
}

int project_impl(const inrct_geom* geom, const inrct_grid* grid, const float* image, float* sino,
                 const float* y, float* resid, double* loss_out, void* ws, size_t ws_bytes,
                 cudaStream_t st, const ProjTables* pre) {
  return project_run(geom, grid, image, sino, y, resid, loss_out, ws, ws_bytes, st, pre, plan_for(geom, grid));
}

static int backproject_run(const inrct_geom* geom, const inrct_grid* grid, const float* sino, float* image,
                           void* ws, size_t ws_bytes, cudaStream_t st, const ProjTables* pre,
                           const ProjPlan& plan) {
  INRCT_TRY(check_geom(geom, grid));
  INRCT_REQUIRE(image && sino, "image and sino must not be NULL");
  ProjWs w;
  bool ok;
  // the tile kernel also wants its padded columns to fit the workspace
  bool tiles = plan.zc == 0 && tile_fit(geom, grid);
  size_t need = 0;
  if (tiles) {
    need = proj_layout(geom, grid, ws, ws_bytes, &w, false, pre == nullptr, true, &ok);
    tiles = ok;
  }
  if (!tiles) need = proj_layout(geom, grid, ws, ws_bytes, &w, false, pre == nullptr, false, &ok);
  if (!ws || !ok) {
    set_error("backproject: workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  const GeomDev g = to_dev(geom, grid);
  if (pre) w.t = *pre;  // built by the projection before
  else INRCT_TRY(build_tables(g, w.t, st));
  if (g.kind == INRCT_CONE3D) {
    float pvh;
    int64_t CzF;
    cone_consts(g, &pvh, &CzF);
    const int64_t m = num_rays(geom);
    if (tiles) {
      cone_prescale_pad_kernel<<<dim3(ceil_div(g.A, 32), ceil_div(g.B + 2 * kRowPad, 32), g.V), dim3(32, 8), 0, st>>>(
          g, w.t.tab0, w.t.tab2, pvh, sino, w.sino_s);
      INRCT_CHECK_LAUNCH("backproject3d (ray scale)");
      const int nz = ceil_div(g.N, 32 * kTileZ);
      const size_t smem = sizeof(ColEntry) * 32 * 4 * nz + sizeof(float) * 16 * ((size_t)nz * 32 * kTileZ + 2);
      const cudaError_t e = cudaFuncSetAttribute(backproject3d_tile_kernel<kTileZ>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) {
        set_error("backproject3d: shared memory attribute: %s", cudaGetErrorString(e));
        return INRCT_ERR_CUDA;
      }
      backproject3d_tile_kernel<kTileZ><<<dim3(ceil_div(g.N, 4), ceil_div(g.N, 4)), 128 * nz, smem, st>>>(
          g, w.t.tab0, w.t.tab1, w.t.views, CzF, w.sino_s, image);
      INRCT_CHECK_LAUNCH("backproject3d (tile kernel)");
      return INRCT_OK;
    }
    if (plan.zc == 0) {
      // one warp per (x, y) column (see backproject3d_col_kernel); plan_set and default_plan
      // only give zc = 0 when the kernel fits the geometry
      INRCT_REQUIRE(col_kernel_fits(geom, grid), "column kernel: N=%d or %d detector rows out of range", g.N, g.B);
      cone_prescale_t_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, st>>>(g, w.t.tab0, w.t.tab2, pvh, sino, w.sino_s);
      INRCT_CHECK_LAUNCH("backproject3d (ray scale)");
      const size_t smem = sizeof(float2) * ((g.V + 1) & ~1) + sizeof(float) * kColWarps * kColStrip;  // < 48 KB
      const bool v4 = g.B % 4 == 0 && reinterpret_cast<uintptr_t>(w.sino_s) % 16 == 0;
      dim3 grd(ceil_div(g.N, kColWarps), g.N);
#define INRCT_COL(VL, V4)                                                                                    \
  backproject3d_col_kernel<VL, V4><<<grd, 32 * kColWarps, smem, st>>>(g, w.t.tab0, w.t.tab1, w.t.views, CzF, \
                                                                      w.sino_s, image)
      if (g.N <= 256) {
        if (v4) INRCT_COL(8, true); else INRCT_COL(8, false);
      } else {
        if (v4) INRCT_COL(16, true); else INRCT_COL(16, false);
      }
#undef INRCT_COL
      INRCT_CHECK_LAUNCH("backproject3d (column kernel)");
      return INRCT_OK;
    }
    cone_prescale_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, st>>>(g, w.t.tab0, w.t.tab2, pvh, sino, w.sino_s);
    INRCT_CHECK_LAUNCH("backproject3d (ray scale)");
    dim3 blk(32, 4);
    if (plan.zc == 4) {
      dim3 grd(ceil_div(g.N, 32), ceil_div(g.N, 4), ceil_div(g.N, 4));
      backproject3d_kernel<4><<<grd, blk, sizeof(float2) * g.V, st>>>(g, w.t.tab0, w.t.tab1, w.t.views, CzF,
                                                                      w.sino_s, image);
    } else if (plan.zc == 32) {
      dim3 grd(ceil_div(g.N, 32), ceil_div(g.N, 4), ceil_div(g.N, 32));
      backproject3d_kernel<32><<<grd, blk, sizeof(float2) * g.V, st>>>(g, w.t.tab0, w.t.tab1, w.t.views, CzF,
                                                                       w.sino_s, image);
    } else if (plan.zc == 16) {
      dim3 grd(ceil_div(g.N, 32), ceil_div(g.N, 4), ceil_div(g.N, 16));
      backproject3d_kernel<16><<<grd, blk, sizeof(float2) * g.V, st>>>(g, w.t.tab0, w.t.tab1, w.t.views, CzF,
                                                                       w.sino_s, image);
    } else {
      dim3 grd(ceil_div(g.N, 32), ceil_div(g.N, 4), ceil_div(g.N, 8));
      backproject3d_kernel<8><<<grd, blk, sizeof(float2) * g.V, st>>>(g, w.t.tab0, w.t.tab1, w.t.views, CzF,
                                                                      w.sino_s, image);
    }
    INRCT_CHECK_LAUNCH("backproject3d");
  } else {
    w.bp_splits = plan.bp_splits;
    if (w.bp_splits < 1 || w.bp_splits > max_bp_splits(geom, grid)) {
      set_error("backproject: %d view splits out of range (1..%d)", w.bp_splits, max_bp_splits(geom, grid));
      return INRCT_ERR_INVALID_ARG;
    }
    dim3 blk(32, kBpWarps);
    dim3 grd(ceil_div(g.N, kBpTile), ceil_div(g.N, kBpTile), w.bp_splits);
    auto launch = [&](auto kernel, size_t smem) {
      const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) {
        set_error("backproject2d: shared memory attribute: %s", cudaGetErrorString(e));
        return INRCT_ERR_CUDA;
      }
      kernel<<<grd, blk, smem, st>>>(g, w.t.tab0, w.t.views, sino, w.bp_splits > 1 ? w.bp_part : image, w.bp_splits);
      INRCT_CHECK_LAUNCH("backproject2d");
      return INRCT_OK;
    };
    const bool two = (int64_t)grd.x * grd.y * grd.z <= kBpTwoBlocks;
    INRCT_TRY(two ? launch(backproject2d_tile_kernel<true>, bp_smem(true))
                  : launch(backproject2d_tile_kernel<false>, bp_smem(false)));
    if (w.bp_splits > 1) {
      const int64_t n = (int64_t)g.N * g.N;
      bp_sum_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(w.bp_part, w.bp_splits, n, image);
      INRCT_CHECK_LAUNCH("backproject2d (split sum)");
    }
  }
  return INRCT_OK;
}

int backproject_impl(const inrct_geom* geom, const inrct_grid* grid, const float* sino, float* image,
                     void* ws, size_t ws_bytes, cudaStream_t st, const ProjTables* pre) {
  return backproject_run(geom, grid, sino, image, ws, ws_bytes, st, pre, plan_for(geom, grid));
}

// ---------------------------------------------------------------------------
// The tuner: times every candidate plan of one geometry (see "Launch plans" above)
// ---------------------------------------------------------------------------
__global__ void tune_fill_kernel(float* __restrict__ a, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = 1.0f + 0.001f * (float)(i % 7);
}

size_t tune_ws_bytes(const inrct_geom* geom, const inrct_grid* grid) {
  if (check_geom(geom, grid) != INRCT_OK) return 0;
  const size_t pw = std::max(project_ws_bytes(geom, grid, true), backproject_ws_bytes(geom, grid, true));
  return align_up(sizeof(float) * grid_points(grid), 256) + align_up(sizeof(float) * num_rays(geom), 256) + pw + 512;
}

int tune_impl(const inrct_geom* geom, const inrct_grid* grid, void* ws, size_t ws_bytes, cudaStream_t st,
              ProjPlan* out) {
  INRCT_TRY(check_geom(geom, grid));
  const size_t need = tune_ws_bytes(geom, grid);
  if (!ws || ws_bytes < need) {
    set_error("inrct_tune: workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  Carver c(ws, ws_bytes);
  const int64_t n = grid_points(grid), m = num_rays(geom);
  float* image = c.take<float>(n);
  float* sino = c.take<float>(m);
  const size_t rest_off = align_up(c.off, 256);  // need leaves at least the projection scratch here
  void* rest = static_cast<char*>(ws) + rest_off;
  const size_t rest_bytes = ws_bytes - rest_off;
  tune_fill_kernel<<<ceil_div(n, 256), 256, 0, st>>>(image, n);
  INRCT_CHECK_LAUNCH("tune fill");
  tune_fill_kernel<<<ceil_div(m, 256), 256, 0, st>>>(sino, m);
  INRCT_CHECK_LAUNCH("tune fill");
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    set_error("inrct_tune: event creation failed");
    return INRCT_ERR_CUDA;
  }
  constexpr int kReps = 5;
  int rc = INRCT_OK;
  // mean time of kReps calls after one untimed call (which also builds the ray tables)
  auto timed = [&](auto&& call, float* ms) -> int {
    INRCT_TRY(call());
    cudaEventRecord(e0, st);
    for (int r = 0; r < kReps; ++r) INRCT_TRY(call());
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(ms, e0, e1) != cudaSuccess) {
      set_error("inrct_tune: timing failed: %s", cudaGetErrorString(cudaGetLastError()));
      return INRCT_ERR_CUDA;
    }
    return INRCT_OK;
  };
  const bool cone = geom->kind == INRCT_CONE3D;
  ProjPlan best = default_plan(geom, grid);
  float best_ms = 0.f;
  // (segments, columns) of the cone's candidates: plan seg = 1 in both its forms
  const std::pair<int, bool> segs2[3] = {{4, false}, {8, false}, {16, false}},
                             segs3[5] = {{1, false}, {2, false}, {4, false}, {8, false}, {1, true}};
  for (int i = 0; i < (cone ? (cols_fit(geom, grid) ? 5 : 4) : 3) && rc == INRCT_OK; ++i) {
    ProjPlan p = best;
    std::tie(p.seg, p.cols) = cone ? segs3[i] : segs2[i];
    float ms = 0.f;
    rc = timed([&] { return project_run(geom, grid, image, sino, nullptr, nullptr, nullptr, rest, rest_bytes, st,
                                        nullptr, p); }, &ms);
    if (rc == INRCT_OK && (i == 0 || ms < best_ms)) {
      best.seg = p.seg;
      best.cols = p.cols;
      best_ms = ms;
    }
  }
  std::vector<int> cands;
  if (cone) {
    cands = {4, 8, 16, 32};
    if (col_kernel_fits(geom, grid)) cands.insert(cands.begin(), 0);
  } else {
    const int mx = max_bp_splits(geom, grid), df = default_bp_splits(geom, grid);
    for (int k = 1; k < mx; k *= 2) cands.push_back(k);
    cands.push_back(mx);
    if (std::find(cands.begin(), cands.end(), df) == cands.end()) cands.push_back(df);
  }
  float best_bp_ms = 0.f;
  for (size_t i = 0; i < cands.size() && rc == INRCT_OK; ++i) {
    ProjPlan p = best;
    if (cone) p.zc = cands[i];
    else p.bp_splits = cands[i];
    float ms = 0.f;
    rc = timed([&] { return backproject_run(geom, grid, sino, image, rest, rest_bytes, st, nullptr, p); }, &ms);
    if (rc == INRCT_OK && (i == 0 || ms < best_bp_ms)) {
      best.zc = p.zc;
      best.bp_splits = p.bp_splits;
      best_bp_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != INRCT_OK) return rc;
  {
    std::lock_guard<std::mutex> lk(g_plan_mu);
    g_plans[plan_key(geom, grid)] = best;
  }
  if (out) *out = best;
  return INRCT_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free projection
//
// For callers that must not allocate device memory themselves: for example a
// host application whose device memory is owned by another framework's pool
// (a cudaMalloc behind its back would break its budget or fragment it), or a
// reconstruction loop on a scanner that reserves all memory once at start-up
// and allows no allocation afterwards.  The projection's scratch (ray tables,
// transposed image, loss partials) then lives in one file-scope device array
// of fixed size, which every GPU that loads this library holds until the
// process exits.
// ---------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_project_scratch[INRCT_NOALLOC_SCRATCH_BYTES];

static std::mutex g_project_scratch_mu;
static void* g_project_scratch_addr[256] = {};  // device address of the array, per device ordinal

// Device address of the array on the current device.  Host code cannot use the array's
// name as a device pointer, so the address is looked up with cudaGetSymbolAddress: on every
// call outside stream capture (the lookup is cheap, and a device reset or a re-created primary
// context then never leaves a stale address behind), and from the per-device cache while the
// stream is being captured (where the lookup is not allowed to run).
static int project_scratch_address(cudaStream_t st, void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 256) {
    set_error("project_noalloc: no usable current device (%s)", cudaGetErrorString(e));
    return INRCT_ERR_CUDA;
  }
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool capturing = cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
  std::lock_guard<std::mutex> lk(g_project_scratch_mu);
  if (!capturing || !g_project_scratch_addr[dev]) {
    if (capturing) {
      set_error("project_noalloc: the first call on a device must not be made during stream capture");
      return INRCT_ERR_INVALID_ARG;
    }
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_project_scratch);
    if (e != cudaSuccess || !p) {
      set_error("project_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return INRCT_ERR_CUDA;
    }
    g_project_scratch_addr[dev] = p;
  }
  *out = g_project_scratch_addr[dev];
  return INRCT_OK;
}

int project_noalloc_impl(const inrct_geom* geom, const inrct_grid* grid, const float* image,
                         float* sino, const float* y, float* resid, double* loss_out, cudaStream_t st) {
  INRCT_TRY(check_geom(geom, grid));
  // without the column form's padding and the tables' checksums, which the array holds only where they fit
  const size_t need = proj_layout(geom, grid, nullptr, 0, nullptr, true, true, false, nullptr, false);
  if (need > (size_t)INRCT_NOALLOC_SCRATCH_BYTES) {
    set_error("project_noalloc: this geometry needs %zu bytes of scratch, more than the %zu-byte "
              "static buffer; use project() with a caller-provided workspace",
              need, (size_t)INRCT_NOALLOC_SCRATCH_BYTES);
    return INRCT_ERR_WORKSPACE;
  }
  void* ws = nullptr;
  INRCT_TRY(project_scratch_address(st, &ws));
  // What the projection reads from the array: the ray tables, the transposed image and the
  // loss partials.  The last two are written earlier in the same call.  Ray tables left by an
  // earlier call are kept only where they still have this geometry's checksums; those of any
  // other geometry, or overwritten in between, are rebuilt first.  So nothing needs clearing.
  const bool sums = proj_layout(geom, grid, nullptr, 0, nullptr, true, true, false, nullptr) <= INRCT_NOALLOC_SCRATCH_BYTES;
  return project_run(geom, grid, image, sino, y, resid, loss_out, ws, (size_t)INRCT_NOALLOC_SCRATCH_BYTES, st, nullptr,
                     plan_for(geom, grid), sums);
}

}  // namespace inrct
