// FP32 SIMT path of the INR: the plain comparator of the BF16 tensor-core path.
//
// Computes E{f_theta} on the grid (Sec. 3) and the weighted Jacobian-transpose
// product sum_i w_i grad_theta f(x_i) with w_i = scale * v_i at listed points
// (Sec. 3, Eq. 2; with every grid point listed it is the full gradient).
//
// Layout: theta follows inrct.h (W row-major [out][in], then b[out]).  The weights are copied once per
// call into aligned rows (WeightCopies).  A VJP runs per chunk of at most kVjpChunk points:
//   1. point_kernel: forward at the chunk's points, storing the layer-1 input E, the activations A_l
//      and (SIREN) sigma'(z_l), then the backward chain delta_l = (W_{l+1}^T delta_{l+1}) sigma'(z_l), which
//      overwrites sigma' (scratch grows with the chunk, never with the grid); the sums over a block's
//      points that need no stored operand (output layer, SIREN first layer) leave it as partials;
//   2. dw_kernel: dW_l = sum_points delta_l a_{l-1}^T and db_l = sum delta_l as a split-K GEMM, FP32
//      partials per split;
//   3. reduce_kernel: the partials into the FP64 gradient (accumulated over chunks).
//
// Hash-encoded INR (Sec. 4, "Hash Enc."): the layer-1 input is gathered from the
// tables at theta[0, n_table) by the forward kernel; the backward kernel finishes
// with g = W_1^T delta_1 per point and scatters w_v g into the 2^d vertex entries
// of every level with FP64 atomics (the encoding is linear in the entries).
#include <math.h>

#include "mlp.cuh"

namespace inrct {

namespace {

struct NetDev {
  int kind, d, F, W, L, K0, N;
  float omega0;
  const float* B;
  int hL, hF, hlog2T;
  unsigned hdense;  // bit l: level l is looked up densely
  float rcp2N;      // 1 / (2N) rounded to FP32
  int fov;          // listed points outside the field of view carry no weight
  int hres[kMaxHashLevels];
};

struct LayerOffs {
  int64_t W[kMaxLayers], b[kMaxLayers];
};

NetDev dev_of(const Net& n, int N) {
  NetDev d;
  d.kind = n.kind;
  d.d = n.d;
  d.F = n.F;
  d.W = n.W;
  d.L = n.L;
  d.K0 = n.K0;
  d.N = N;
  d.omega0 = n.omega0;
  d.B = n.B;
  d.hL = n.hL;
  d.hF = n.hF;
  d.hlog2T = n.hlog2T;
  d.hdense = 0;
  d.rcp2N = 1.0f / (2.0f * (float)N);
  d.fov = n.fov;
  for (int l = 0; l < kMaxHashLevels; ++l) {
    d.hres[l] = l < n.hL ? n.hres[l] : 0;
    if (l < n.hL) {
      int64_t cells = 1;
      for (int a = 0; a < n.d; ++a) cells *= (int64_t)n.hres[l] + 1;
      if (cells <= ((int64_t)1 << n.hlog2T)) d.hdense |= 1u << l;
    }
  }
  return d;
}

__device__ __forceinline__ int64_t grid_size(const NetDev& n) {
  return n.d == 3 ? (int64_t)n.N * n.N * n.N : (int64_t)n.N * n.N;
}

// Level l of the hash encoding at the grid point with per-axis indices k[0..D): the
// table entries of its 2^D surrounding vertices and their multilinear weights.  The
// level coordinate (2k + 1) N_l / (2N) is split exactly into its integer part c0 and
// remainder r: while the numerator stays below 2^24 (exact in FP32) the quotient from
// the FP32 reciprocal is within one of the floor, and one integer correction makes it
// exact; larger numerators divide in 32 or 64-bit integers.  The fraction is r / (2N)
// in FP32 (exact when 2N is a power of two).  D is a template parameter so that every
// loop unrolls and the vertex state stays in registers.
template <int D>
__device__ __forceinline__ void hash_vertices(const NetDev& n, int l, const int* k, uint32_t (&ent)[1 << D],
                                              float (&w)[1 << D]) {
  const uint32_t Nl = (uint32_t)n.hres[l];
  const uint32_t twoN = 2u * (uint32_t)n.N;
  uint32_t c0[D];
  float fr[D];
  // (2k + 1) N_l < 2N N_l
  const uint64_t bound = (uint64_t)twoN * Nl;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    uint32_t rem;
    if (bound <= (1u << 24)) {
      // |num * fl(1/2N) - num / 2N| < 2 num 2^-24 / 2N < 1: truncation is off by at most one
      const uint32_t num = (2u * (uint32_t)k[a] + 1u) * Nl;
      uint32_t q = (uint32_t)((float)num * n.rcp2N);
      int r = (int)num - (int)(q * twoN);
      if (r < 0) {
        q -= 1;
        r += (int)twoN;
      } else if (r >= (int)twoN) {
        q += 1;
        r -= (int)twoN;
      }
      c0[a] = q;
      rem = (uint32_t)r;
    } else if (bound <= 0xFFFFFFFFull) {
      const uint32_t num = (2u * (uint32_t)k[a] + 1u) * Nl;
      c0[a] = num / twoN;
      rem = num - c0[a] * twoN;
    } else {
      const uint64_t num = (2ull * (uint32_t)k[a] + 1ull) * Nl;
      c0[a] = (uint32_t)(num / twoN);
      rem = (uint32_t)(num - (uint64_t)c0[a] * twoN);
    }
    fr[a] = (float)rem * n.rcp2N;
  }
  const bool dense = (n.hdense >> l) & 1u;
  const uint32_t mask = (1u << n.hlog2T) - 1u;
  constexpr uint32_t kPrime[3] = {1u, 2654435761u, 805459861u};
#pragma unroll
  for (int v = 0; v < (1 << D); ++v) {
    float wv = 1.f;
    uint32_t lin = 0, stride = 1, h = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const uint32_t bit = (v >> a) & 1;
      const uint32_t c = c0[a] + bit;
      wv *= bit ? fr[a] : 1.f - fr[a];
      lin += c * stride;  // dense levels have (N_l + 1)^D <= T <= 2^24 entries: no wrap
      stride *= Nl + 1u;
      h ^= c * kPrime[a];  // 32-bit unsigned, wraps by definition
    }
    ent[v] = dense ? lin : (h & mask);
    w[v] = wv;
  }
}

// Features of level l at the point: sum_v w_v table[ent_v][f] to out[f stride], f < F.
template <int D>
__device__ __forceinline__ void hash_gather(const NetDev& n, const float* __restrict__ theta, int l,
                                            const int* k, float* out, int stride) {
  uint32_t ent[1 << D];
  float w[1 << D];
  hash_vertices<D>(n, l, k, ent, w);
  const float* tab = theta + ((int64_t)l << n.hlog2T) * n.hF;
  if (n.hF == 2) {
    // both features of a vertex in one 8-byte load (theta is 8-byte aligned, see
    // check_theta_alignment, and every table and entry offset is even)
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int v = 0; v < (1 << D); ++v) {
      const float2 e = __ldg(reinterpret_cast<const float2*>(tab) + ent[v]);
      a0 = fmaf(w[v], e.x, a0);
      a1 = fmaf(w[v], e.y, a1);
    }
    out[0] = a0;
    out[stride] = a1;
    return;
  }
  for (int f = 0; f < n.hF; ++f) {
    float a = 0.f;
#pragma unroll
    for (int v = 0; v < (1 << D); ++v) a = fmaf(w[v], __ldg(tab + (int64_t)ent[v] * n.hF + f), a);
    out[f * stride] = a;
  }
}

// Table gradient of level l (the same for the warp) at one point per lane: entry ent_v, feature f receives
// w_v g[f stride].  Called by all 32 lanes of a warp together (ok = false: the lane adds
// nothing).  Runs of consecutive lanes whose vertex is the same entry are summed
// by a segmented scan (up to 5 shuffle steps, no divergence) and the last lane of each run
// issues the one atomic: neighbouring points of a sorted index set share vertices at
// coarse levels.  An entry that recurs after another one simply starts a new run, so the
// result holds for any order of the points.  The runs come from one ballot, and the scan ends with the longest run
// of the warp (none at the fine levels): shuffles bound this part, which took 33 of the hash step's 532 us with
// run flags spread by shuffles and all five steps always taken and takes 30 now; the atomics are 10 of it.
template <int D>
__device__ __forceinline__ void hash_scatter_warp(const NetDev& n, double* __restrict__ gtab, int l, const int* k,
                                                  const float* g, int stride, bool ok) {
  const unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint32_t ent[1 << D];
  float w[1 << D];
#pragma unroll
  for (int v = 0; v < (1 << D); ++v) ent[v] = 0;
  if (ok) hash_vertices<D>(n, l, k, ent, w);
  const unsigned live = __ballot_sync(kFull, ok);
  // lanes that cannot continue a run: the first, those that add nothing, and those after one
  const bool alone = lane == 0 || !ok || !(live >> (lane - 1) & 1u);
  double* gl = gtab + ((int64_t)l << n.hlog2T) * n.hF;
#pragma unroll
  for (int v = 0; v < (1 << D); ++v) {
    const uint32_t prev = __shfl_up_sync(kFull, ent[v], 1);
    const unsigned heads = __ballot_sync(kFull, alone || prev != ent[v]);
    const int back = lane - (31 - __clz(heads & (kFull >> (31 - lane))));  // lanes since the run's head
    const bool tail = lane == 31 || (heads >> (lane + 1) & 1u);
    const int longest = __reduce_max_sync(kFull, back);
    for (int ff = 0; ff < n.hF; ++ff) {
      float val = ok ? w[v] * g[ff * stride] : 0.f;
      for (int off = 1; off <= longest; off <<= 1) {
        const float up = __shfl_up_sync(kFull, val, off);
        if (back >= off) val += up;
      }
      if (ok && tail) atomicAdd(gl + (int64_t)ent[v] * n.hF + ff, (double)val);
    }
  }
}

// ---------------------------------------------------------------------------
// weight layouts: W^T of every hidden layer ([in][out], the forward's rows), and for the VJP the
// layers W itself ([out][in], the backward chain's rows), one launch.  Copies, so that the rows are
// 16-byte aligned whatever theta's alignment is; the hash networks' W_1 rows are padded to 64.
// ---------------------------------------------------------------------------
struct WeightCopies {
  int64_t Wt[kMaxLayers], Wc[kMaxLayers];  // offsets in the copy buffer (Wc: -1 where not needed)
  int64_t total;
};

WeightCopies weight_copies(const Net& n, bool vjp) {
  WeightCopies c;
  int64_t off = 0;
  for (int l = 0; l < n.L; ++l) {
    c.Wt[l] = off;
    off += (int64_t)n.in_dim[l] * n.W;
    c.Wc[l] = -1;
  }
  if (vjp) {
    for (int l = n.kind == INRCT_HASH ? 0 : 1; l < n.L; ++l) {
      c.Wc[l] = off;
      off += (int64_t)n.W * (l == 0 ? 64 : n.W);
    }
  }
  c.total = off;
  return c;
}

struct CopyArgs {
  int L, W;
  int in[kMaxLayers];
  int64_t offW[kMaxLayers], Wt[kMaxLayers], Wc[kMaxLayers];
};

__global__ void __launch_bounds__(256)
    copy_weights_kernel(const float* __restrict__ theta, const __grid_constant__ CopyArgs a, float* __restrict__ out) {
  const int l = blockIdx.y, in = a.in[l], W = a.W;
  const float* w = theta + a.offW[l];
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = t0; t < (int64_t)in * W; t += step) {
    const int k = (int)(t / W), o = (int)(t - (int64_t)k * W);
    out[a.Wt[l] + t] = w[(int64_t)o * in + k];
  }
  if (a.Wc[l] >= 0) {
    const int ld = l == 0 ? 64 : W;
    for (int64_t t = t0; t < (int64_t)W * ld; t += step) {
      const int o = (int)(t / ld), k = (int)(t - (int64_t)o * ld);
      out[a.Wc[l] + t] = k < in ? w[(int64_t)o * in + k] : 0.f;
    }
  }
}

// ---------------------------------------------------------------------------
// asynchronous copies and packed FMAs
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// n = 16: copy; n = 0: zero fill (src must still be a valid address)
__device__ __forceinline__ void cp16(float* dst, const float* src, int n) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm_addr(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp4(float* dst, const float* src, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sm_addr(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// acc[PT][4] += a[PT] (x) w[8]: PT points by 8 columns, the columns in four packed pairs (w0, w1 as
// loaded, 16 bytes each).  A point's value is packed with itself.
template <int PT>
__device__ __forceinline__ void outer8(f32x2 (&acc)[PT][4], const float* a, ulonglong2 w0, ulonglong2 w1) {
#pragma unroll
  for (int p = 0; p < PT; ++p) {
    const f32x2 d = dup2(a[p]);
    acc[p][0] = fma2(d, w0.x, acc[p][0]);
    acc[p][1] = fma2(d, w0.y, acc[p][1]);
    acc[p][2] = fma2(d, w1.x, acc[p][2]);
    acc[p][3] = fma2(d, w1.y, acc[p][3]);
  }
}

// ---------------------------------------------------------------------------
// The point kernel: forward chain of a block's points and, for the VJP, the backward chain.
//
// A block holds P = 8 PT points and 2 NW warps (W = 64 NW).  Activations (then deltas) live in
// shared memory as [unit][point], one buffer for all layers; a warp owns 4 PT points x 64 units
// and a thread PT points x 8 units, so each step of the contraction costs a thread PT/4 + 2
// 16-byte shared loads for 8 PT multiply-adds (packed in pairs).  The rows of the weight matrix
// stream through a ring of kStages chunks of kKc rows by cp.async; all blocks read the same rows,
// from L2.  The kernel this replaced kept one unit per thread and 16 points per block: 16
// broadcast 16-byte loads and 4 weight loads per 64 multiply-adds, bound by the load/store unit.
// 512^2 evaluation of the SIREN 5 x 256: 4.78 -> 2.64 ms (52 of the nominal 80.5 TFLOP/s); VJP of 65,536 points,
// point kernel 2.72 -> 1.47 ms.  What bounds it: the FMA pipe (67 % busy over the launch, the sine passes
// included).  Measured beside it: scalar FMAs in place of the packed ones 3.24 ms (issue slots), chunks of 8
// rows in a ring of 4 2.76 ms, operands of the next step fetched ahead in registers 2.86 ms.
//
// The activations are applied in a second pass over the thread's own values through shared memory
// (a loop, not 8 PT inlined sines).  In that pass a lane starts with another one of its four
// points than its neighbours (rot), so that the 32 lanes hit 32 banks.
// ---------------------------------------------------------------------------
constexpr int kKc = 16, kStages = 2;

struct PointArgs {
  const float* theta;
  const float* wbuf;  // weight copies (WeightCopies)
  WeightCopies wc;
  int64_t npts;
  const int32_t* idx;  // NULL: grid order
  float* out_f;        // evaluation: f(x)
  int rows;            // rows of the shared activation buffer
  // VJP
  const float* v;
  float scale;
  float* A;  // [l][npts][W] activations
  float* D;  // [l][npts][W] sigma' (SIREN), then the deltas
  float* E;  // [npts][K0] layer-1 input (Fourier features, hash)
  float* bpart;    // [block][bp] partial sums (see block_partial_cols)
  double* vpart;   // [block] partial sums of the virtual loss
  double* gtab;    // hash table gradient
};

// Columns of a block's partial sums: dW_out[W], db_out, and for the SIREN dW_1 [W][d], db_1 [W] (its
// layer-1 input is the point's coordinates, so those sums come from the deltas in shared memory).
__host__ __device__ inline int block_partial_cols(int kind, int W, int d) {
  return W + 1 + (kind == INRCT_SIREN ? W * (d + 1) : 0);
}

template <int PT, int WW, typename Row>
__device__ __forceinline__ void gemm_rows(const float* __restrict__ act, float* __restrict__ wst, Row row, int K,
                                          int nthreads, int pbase, int wbase, bool active, f32x2 (&acc)[PT][4]) {
  constexpr int S = 8 * PT + 4;
  const int t = threadIdx.x, chunks = (K + kKc - 1) / kKc;
  auto load = [&](int c) {
    if (c < chunks) {
      const int rows = min(kKc, K - c * kKc);
      float* st = wst + (c % kStages) * (kKc * WW);
      for (int e = t; e < rows * (WW / 4); e += nthreads) {
        const int r = e / (WW / 4), q = e % (WW / 4);
        cp16(st + r * WW + 4 * q, row(c * kKc + r) + 4 * q, 16);
      }
    }
    cp_commit();
  };
#pragma unroll
  for (int c = 0; c < kStages - 1; ++c) load(c);
  const float* ap = act + pbase;
  for (int c = 0; c < chunks; ++c) {
    cp_wait<kStages - 2>();
    __syncthreads();  // chunk c has landed for every thread, and chunk c - 1 is no longer read
    load(c + kStages - 1);
    if (active) {
      const float* wp = wst + (c % kStages) * (kKc * WW) + wbase;
      auto step = [&](int r) {
        float a[PT];
        *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(ap + r * S);
        if constexpr (PT == 8)
          *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(ap + r * S + 16);
        outer8<PT>(acc, a, *reinterpret_cast<const ulonglong2*>(wp + r * WW),
                   *reinterpret_cast<const ulonglong2*>(wp + r * WW + 32));
      };
      const int rows = K - c * kKc;
      if (rows >= kKc) {
#pragma unroll
        for (int r = 0; r < kKc; ++r) step(r);
      } else {
        for (int r = 0; r < rows; ++r) step(r);
      }
    }
    ap += kKc * S;
  }
  cp_wait<0>();
  __syncthreads();  // the buffers may be written again
}

// Layer-1 input of a block's points to E: buffer rows [0, rows) are columns k0 on (half > 0: the first half are, the
// others follow column F + k0).  Four columns at a time where they stay together and aligned: a lane writes a row of
// its own, so a column at a time costs a sector for four bytes (128^2 points of 128 columns, the step's VJP kernel
// 49.9 -> 41.8 us).  Not inlined: in line it cost the SIREN's VJP, which never comes here, 0.2 % by its registers.
template <int P, int S, int T>
__device__ __noinline__ void store_inputs(const float* act, float* E, int K0, int F, int k0, int rows, int half,
                                          int64_t p0, int64_t npts) {
  const int t = threadIdx.x;
  if (((K0 | rows | half | k0 | (half ? F : 0)) & 3) == 0) {
    for (int e = t; e < (rows >> 2) * P; e += T) {
      const int p = e % P, r = (e / P) * 4;
      const int k = half ? (r < half ? k0 + r : F + k0 + r - half) : r;
      const float* a = act + r * S + p;
      if (p0 + p < npts)
        *reinterpret_cast<float4*>(E + (p0 + p) * K0 + k) = make_float4(a[0], a[S], a[2 * S], a[3 * S]);
    }
    return;
  }
  for (int e = t; e < rows * P; e += T) {
    const int p = e % P, r = e / P;
    const int k = half ? (r < half ? k0 + r : F + k0 + r - half) : r;
    if (p0 + p < npts) E[(p0 + p) * K0 + k] = act[r * S + p];
  }
}

template <int PT, int NW, bool VJP>
__global__ void __launch_bounds__(64 * NW, 8 / NW)
    point_kernel(const __grid_constant__ NetDev net, const __grid_constant__ LayerOffs lo,
                 const __grid_constant__ PointArgs g) {
  constexpr int P = 8 * PT, S = P + 4, W = 64 * NW, T = 64 * NW;
  extern __shared__ __align__(16) float sh[];
  float* act = sh;                    // [rows][S]
  float* wst = sh + g.rows * S;       // [kStages][kKc][W]
  __shared__ float xs[P][3];
  __shared__ int ks[P][3];
  __shared__ float dsc[P];
  __shared__ float red[T / P > 0 ? T / P : 1][P];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int lq = lane & 7, lp = lane >> 3, wo = warp % NW, pw = warp / NW;
  const int pbase = pw * 4 * PT + 4 * lp;  // the thread's points: pbase + {0..3} (+ 16 + {0..3})
  const int obase = wo * 64 + 4 * lq;      // its units: obase + {0..3} and + 32 + {0..3}
  const int rot = lq >> 1;
  const int64_t p0 = (int64_t)blockIdx.x * P;
  const int K0 = net.K0, L = net.L;
  for (int p = t; p < P; p += T) {
    // places past the last point repeat it without weight: 0 times a value that is not finite would reach the block's
    // sums, and must not come from a point that is not listed
    const bool live = p0 + p < g.npts;
    const int64_t q = live ? p0 + p : g.npts - 1;
    int64_t i = g.idx ? (int64_t)g.idx[q] : q;
    const bool in = i >= 0 && i < grid_size(net);
    if (VJP) dsc[p] = live && in && (!net.fov || in_fov(i, net.N)) ? g.scale * g.v[i] : 0.f;
    if (!in) i = 0;  // out-of-range indices contribute nothing
    point_coords(i, net.N, net.d, xs[p]);
    ks[p][0] = (int)(i % net.N);
    ks[p][1] = (int)((i / net.N) % net.N);
    ks[p][2] = net.d == 3 ? (int)(i / ((int64_t)net.N * net.N)) : 0;
  }
  __syncthreads();

  f32x2 acc[PT][4];
  // acc = the layer's bias
  auto init_bias = [&](int l) {
    const float* b = g.theta + lo.b[l] + obase;
    const f32x2 b0 = pack2(b[0], b[1]), b1 = pack2(b[2], b[3]), b2 = pack2(b[32], b[33]), b3 = pack2(b[34], b[35]);
#pragma unroll
    for (int p = 0; p < PT; ++p) {
      acc[p][0] = b0;
      acc[p][1] = b1;
      acc[p][2] = b2;
      acc[p][3] = b3;
    }
  };
  // acc to the thread's own places of the activation buffer
  auto put_acc = [&]() {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float u[2][PT];
#pragma unroll
      for (int p = 0; p < PT; ++p) unpack2(acc[p][q], u[0][p], u[1][p]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float* d = act + (obase + (q >> 1) * 32 + (q & 1) * 2 + h) * S + pbase;
        *reinterpret_cast<float4*>(d) = make_float4(u[h][0], u[h][1], u[h][2], u[h][3]);
        if constexpr (PT == 8)
          *reinterpret_cast<float4*>(d + 16) = make_float4(u[h][4], u[h][5], u[h][6], u[h][7]);
      }
    }
  };
  // fn(point, values of its 8 units, from the buffer and back) over the thread's points
  auto each_point = [&](auto&& fn) {
#pragma unroll 1
    for (int it = 0; it < PT; ++it) {
      const int p = pbase + (it & 4) * 4 + ((it + rot) & 3);
      float u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = act[(obase + (q >> 2) * 32 + (q & 3)) * S + p];
      fn(p, u);
#pragma unroll
      for (int q = 0; q < 8; ++q) act[(obase + (q >> 2) * 32 + (q & 3)) * S + p] = u[q];
    }
  };
  auto store8 = [&](float* base, const float* u) {
    *reinterpret_cast<float4*>(base) = make_float4(u[0], u[1], u[2], u[3]);
    *reinterpret_cast<float4*>(base + 32) = make_float4(u[4], u[5], u[6], u[7]);
  };
  auto load8 = [&](const float* base, float* u) {
    *reinterpret_cast<float4*>(u) = *reinterpret_cast<const float4*>(base);
    *reinterpret_cast<float4*>(u + 4) = *reinterpret_cast<const float4*>(base + 32);
  };
  auto place = [&](int l, int p) { return ((int64_t)l * g.npts + p0 + p) * W + obase; };
  auto store_E = [&](int k0, int rows, int half) {
    store_inputs<P, S, T>(act, g.E, K0, net.F, k0, rows, half, p0, g.npts);
  };

  // ---- layer 1 ----
  init_bias(0);
  const float* wt0 = g.wbuf + g.wc.Wt[0];
  if (net.kind == INRCT_FFN_RELU) {
    // the whole input where it fits the buffer (columns in order), else chunks of rows / 2 features, their cosines
    // and their sines
    const float inv_N = 1.f / (float)net.N;
    const int fmax = K0 <= g.rows ? net.F : g.rows / 2;
    for (int f0 = 0; f0 < net.F; f0 += fmax) {
      const int nf = min(fmax, net.F - f0);
#pragma unroll 4
      for (int e = t; e < P * nf; e += T) {
        const int p = e % P, f = e / P;
        const float* Bf = net.B + (int64_t)(f0 + f) * net.d;
        const int m[3] = {2 * ks[p][0] + 1 - net.N, 2 * ks[p][1] + 1 - net.N,
                          net.d == 3 ? 2 * ks[p][2] + 1 - net.N : 0};
        float s, c;
        sincospif(2.f * ffn_phase_exact(Bf[0], Bf[1], net.d == 3 ? Bf[2] : 0.f, m, net.d, net.N, inv_N), &s, &c);
        act[f * S + p] = c;
        act[(nf + f) * S + p] = s;
      }
      __syncthreads();
      if (VJP) store_E(f0, 2 * nf, nf);
      const int F = net.F;
      gemm_rows<PT, W>(act, wst, [=](int r) { return wt0 + (int64_t)(r < nf ? f0 + r : F + f0 + r - nf) * W; }, 2 * nf,
                       T, pbase, obase, true, acc);
    }
  } else {
    if (net.kind == INRCT_HASH) {
      // one thread per (level, point): interpolate the level's features
      for (int e = t; e < P * net.hL; e += T) {
        const int p = e % P, l = e / P;
        if (net.d == 3) hash_gather<3>(net, g.theta, l, ks[p], act + l * net.hF * S + p, S);
        else hash_gather<2>(net, g.theta, l, ks[p], act + l * net.hF * S + p, S);
      }
    } else {
      for (int e = t; e < P * net.d; e += T) act[(e / P) * S + e % P] = xs[e % P][e / P];
    }
    __syncthreads();
    if (VJP && net.kind == INRCT_HASH) store_E(0, K0, 0);
    gemm_rows<PT, W>(act, wst, [=](int r) { return wt0 + (int64_t)r * W; }, K0, T, pbase, obase, true, acc);
  }

  // ---- hidden layers ----
  for (int l = 0;; ++l) {
    put_acc();
    if (net.kind == INRCT_SIREN) {
      each_point([&](int p, float* u) {
        if (VJP) {
          float c[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float z = net.omega0 * u[q];
            u[q] = sinf(z);
            c[q] = net.omega0 * cosf(z);
          }
          if (p0 + p < g.npts) {
            store8(g.A + place(l, p), u);
            store8(g.D + place(l, p), c);
          }
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) u[q] = sinf(net.omega0 * u[q]);
        }
      });
    } else {
      each_point([&](int p, float* u) {
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = fmaxf(u[q], 0.f);
        if (VJP && p0 + p < g.npts) store8(g.A + place(l, p), u);
      });
    }
    __syncthreads();
    if (l + 1 == L) break;
    init_bias(l + 1);
    const float* wt = g.wbuf + g.wc.Wt[l + 1];
    gemm_rows<PT, W>(act, wst, [=](int r) { return wt + (int64_t)r * W; }, W, T, pbase, obase, true, acc);
  }

  // ---- f(x) = w_out . a + b_out: T / P threads per point ----
  const float* wout = g.theta + lo.W[L];
  if (g.out_f || (VJP && g.vpart)) {
    static_assert(T >= P, "at least one thread per point");
    constexpr int G = T / P, KG = W / G;
    const int p = t % P, gr = t / P;
    // a tree over pairs of units: a chain of the KG units would round at the size of the sum KG times
    constexpr int H = KG / 2;
    float s[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int o = gr * KG + i;
      s[i] = fmaf(act[(o + H) * S + p], __ldg(wout + o + H), act[o * S + p] * __ldg(wout + o));
    }
#pragma unroll
    for (int d = H / 2; d; d /= 2)
#pragma unroll
      for (int i = 0; i < d; ++i) s[i] += s[i + d];
    red[gr][p] = s[0];
    __syncthreads();
    if (t < P) {
      float f = g.theta[lo.b[L]];
#pragma unroll
      for (int q = 0; q < G; ++q) f += red[q][t];
      if (!VJP) {
        if (p0 + t < g.npts) g.out_f[p0 + t] = f;
      } else {
        red[0][t] = f;  // read by this thread's column only
      }
    }
    if (VJP) {
      __syncthreads();
      if (t < 32) {  // the block's share of the virtual loss, FP64 in a fixed order
        double s2 = 0.0;
        for (int q = t; q < P; q += 32) s2 += (double)dsc[q] * (double)red[0][q];
#pragma unroll
        for (int o = 16; o; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        if (t == 0) g.vpart[blockIdx.x] = s2;
      }
    }
  }
  if constexpr (VJP) {
    // sum over the block's points of dsc a, per unit (T == W threads); lanes start at different points (banks)
    float* bp = g.bpart + (int64_t)blockIdx.x * block_partial_cols(net.kind, W, net.d);
    const int start = lane >> 3;
    {
      float s[4] = {}, sb[4] = {};  // four chains of P / 4 points
      for (int q = 0; q < P / 4; ++q)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int p = (q + h * (P / 4) + start) & (P - 1);
          s[h] = fmaf(dsc[p], act[t * S + p], s[h]);
          sb[h] += dsc[p];
        }
      bp[t] = (s[0] + s[1]) + (s[2] + s[3]);
      if (t == 0) bp[W] = (sb[0] + sb[1]) + (sb[2] + sb[3]);
    }
    __syncthreads();
    // delta_{L-1} = dsc w_out sigma'(z_{L-1})
    {
      float w[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q] = wout[obase + (q >> 2) * 32 + (q & 3)];
      each_point([&](int p, float* u) {
        const bool live = p0 + p < g.npts;
        float c[8];
        if (net.kind == INRCT_SIREN) {
          if (live) load8(g.D + place(L - 1, p), c);
        } else {
#pragma unroll
          for (int q = 0; q < 8; ++q) c[q] = u[q] > 0.f ? 1.f : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = live ? dsc[p] * w[q] * c[q] : 0.f;
        if (live) store8(g.D + place(L - 1, p), u);
      });
    }
    __syncthreads();
    // delta_{l-1} = (W_l^T delta_l) sigma'(z_{l-1})
    for (int l = L - 1; l >= 1; --l) {
#pragma unroll
      for (int p = 0; p < PT; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = 0ull;
      const float* wl = g.wbuf + g.wc.Wc[l];
      gemm_rows<PT, W>(act, wst, [=](int r) { return wl + (int64_t)r * W; }, W, T, pbase, obase, true, acc);
      put_acc();
      each_point([&](int p, float* u) {
        const bool live = p0 + p < g.npts;
        float c[8];
        if (live) load8((net.kind == INRCT_SIREN ? g.D : g.A) + place(l - 1, p), c);
        if (net.kind != INRCT_SIREN) {
#pragma unroll
          for (int q = 0; q < 8; ++q) c[q] = c[q] > 0.f ? 1.f : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = live ? u[q] * c[q] : 0.f;
        if (live) store8(g.D + place(l - 1, p), u);
      });
      __syncthreads();
    }
    if (net.kind == INRCT_SIREN) {
      float s[3] = {0.f, 0.f, 0.f}, sb = 0.f;
      for (int q = 0; q < P; ++q) {
        const int p = (q + start) & (P - 1);
        const float d = act[t * S + p];
        s[0] = fmaf(d, xs[p][0], s[0]);
        s[1] = fmaf(d, xs[p][1], s[1]);
        s[2] = fmaf(d, xs[p][2], s[2]);
        sb += d;
      }
      float* b1 = bp + W + 1 + t * (net.d + 1);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k < net.d) b1[k] = s[k];
      b1[net.d] = sb;
    }
    if (net.kind == INRCT_HASH) {
      // hash tables: g = W_1^T delta_1 is the gradient of the layer-1 input; each vertex entry of each
      // level receives its weight times the level's slice of g.  64 columns: the warps of unit group 0.
#pragma unroll
      for (int p = 0; p < PT; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = 0ull;
      const float* w0 = g.wbuf + g.wc.Wc[0];
      gemm_rows<PT, 64>(act, wst, [=](int r) { return w0 + (int64_t)r * 64; }, W, T, pbase, 4 * lq, wo == 0, acc);
      if (wo == 0) put_acc();
      __syncthreads();
      // level-major items: a warp holds consecutive points of one level
      static_assert(P % 32 == 0, "whole warps per level");
      for (int e = t; e < P * net.hL; e += T) {  // T is a multiple of 32: warps stay whole
        const int l = e / P, p = e % P;
        const bool ok = dsc[p] != 0.f;
        const float* gl = act + l * net.hF * S + p;
        if (net.d == 3) hash_scatter_warp<3>(net, g.gtab, l, ks[p], gl, S, ok);
        else hash_scatter_warp<2>(net, g.gtab, l, ks[p], gl, S, ok);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// dW_l and db_l of the layers whose input is stored, as a split-K GEMM over the points:
//   C[o][k] = sum_q X[q][o] Y[q][k] (k < K) and C[o][K] = sum_q X[q][o], X the deltas, Y the layer's input.
// Tiles of TM x TM outputs, 8 x 8 per thread; G thread groups of one block take every G-th slab of points and
// are added in group order at the end.  Slabs of kDk points come by cp.async (both operands are [point][column],
// the layout the multiply reads).  The kernel this replaced (64 x 64 tiles, 4 x 4 per thread, one layer per
// launch, sines recomputed per tile) took 460 us per 256 x 256 layer and 65,536 points, this one 170 us; it is
// bound by the FMA pipe (68 % busy).  64-wide networks take 64 x 64 tiles (their whole layer).
// ---------------------------------------------------------------------------
constexpr int kDk = 16, kDStages = 3;

struct DwJob {
  const float *X, *Y;
  int O, K, tiles_k, first;  // first: the job's first tile in blockIdx.x
  int runs, run_rounds;      // FP32 sums a block forms one after the other, rounds of G slabs in each (see dw_runs)
  int64_t part;              // offset of its partials, [split][run][O][K + 1]
};
struct DwArgs {
  int n;
  int64_t npts;
  DwJob job[kMaxLayers];
};

template <int TM, int G>
__global__ void __launch_bounds__(TM * TM / 64 * G)
    dw_kernel(const __grid_constant__ DwArgs a, float* __restrict__ part) {
  constexpr int TG = TM * TM / 64, T = TG * G;  // threads of a group, of the block
  constexpr int SLAB = 2 * kDk * TM;            // floats of one group's slab: X then Y
  extern __shared__ __align__(16) float sh[];   // [kDStages][G][SLAB], then (G > 1) [TM][TM] sums and [TM] bias sums
  int j = 0;
  while (j + 1 < a.n && (int)blockIdx.x >= a.job[j + 1].first) ++j;
  const DwJob& J = a.job[j];
  const int tile = blockIdx.x - J.first, to = tile / J.tiles_k, tk = tile % J.tiles_k, sp = blockIdx.y;
  const int O = J.O, K = J.K, o0 = to * TM, k0 = tk * TM;
  const int64_t q0 = (int64_t)sp * J.runs * J.run_rounds * (kDk * G);
  const int rounds = J.runs * J.run_rounds;
  const int t = threadIdx.x, grp = t / TG, tg = t % TG;
  // 32 x 64 outputs per warp: lanes 4 x 8, a thread takes rows 4 lp + {0..3}, + 16 and columns 4 lq + {0..3}, + 32
  const int lane = t & 31, wg = tg >> 5;
  const int orow = (wg / (TM / 64)) * 32 + 4 * (lane >> 3), kcol = (wg % (TM / 64)) * 64 + 4 * (lane & 7);
  const bool yvec = (K & 3) == 0;  // rows of Y 16-byte aligned (its base is)
  auto load = [&](int c) {
    const int64_t qb = q0 + (int64_t)(c * G + grp) * kDk;
    if (c < rounds) {
      float* xs = sh + ((c % kDStages) * G + grp) * SLAB;
      float* ys = xs + kDk * TM;
      for (int e = tg; e < kDk * TM / 4; e += TG) {
        const int r = e / (TM / 4), col = 4 * (e % (TM / 4));
        const bool in = qb + r < a.npts;
        cp16(xs + r * TM + col, in ? J.X + (qb + r) * O + o0 + col : J.X, in ? 16 : 0);  // O is a multiple of TM
        if (yvec) {
          const bool iy = in && k0 + col < K;
          cp16(ys + r * TM + col, iy ? J.Y + (qb + r) * K + k0 + col : J.Y, iy ? 16 : 0);
        } else {
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const bool iy = in && k0 + col + h < K;
            cp4(ys + r * TM + col + h, iy ? J.Y + (qb + r) * K + k0 + col + h : J.Y, iy ? 4 : 0);
          }
        }
      }
    }
    cp_commit();
  };
  f32x2 acc[8][4];
  constexpr int OB = (TM + TG - 1) / TG;  // bias columns per thread
  float sb[OB];
  auto clear = [&]() {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int h = 0; h < 4; ++h) acc[i][h] = 0ull;
#pragma unroll
    for (int b = 0; b < OB; ++b) sb[b] = 0.f;
  };
  clear();
#pragma unroll
  for (int c = 0; c < kDStages - 1; ++c) load(c);
  float* out = part + J.part + (int64_t)sp * J.runs * O * (K + 1);
  int left = J.run_rounds;
  for (int c = 0; c < rounds; ++c) {
    cp_wait<kDStages - 2>();
    __syncthreads();
    load(c + kDStages - 1);
    const float* xs = sh + ((c % kDStages) * G + grp) * SLAB;
    const float* ys = xs + kDk * TM;
#pragma unroll
    for (int r = 0; r < kDk; ++r) {
      float x[8];
      *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(xs + r * TM + orow);
      *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(xs + r * TM + orow + 16);
      outer8<8>(acc, x, *reinterpret_cast<const ulonglong2*>(ys + r * TM + kcol),
                *reinterpret_cast<const ulonglong2*>(ys + r * TM + kcol + 32));
    }
    if (tk == 0) {
#pragma unroll
      for (int b = 0; b < OB; ++b)
        if (tg + b * TG < TM)
#pragma unroll
          for (int r = 0; r < kDk; ++r) sb[b] += xs[r * TM + tg + b * TG];
    }
    if (--left) continue;
    // the end of a run of FP32 sums: its partials leave, the copies of the next slabs are under way
    left = J.run_rounds;
    if constexpr (G > 1) {
      // add the groups in order through shared memory (one group writes at a time)
      float* sum = sh + kDStages * G * SLAB;
      float* bsum = sum + TM * TM;
      for (int q = 0; q < G; ++q) {
        if (grp == q) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int h = 0; h < 4; ++h) {
              float* d = sum + (orow + (i >> 2) * 16 + (i & 3)) * TM + kcol + (h >> 1) * 32 + (h & 1) * 2;
              float lo, hi;
              unpack2(acc[i][h], lo, hi);
              d[0] = q ? d[0] + lo : lo;
              d[1] = q ? d[1] + hi : hi;
            }
#pragma unroll
          for (int b = 0; b < OB; ++b)
            if (tg + b * TG < TM) bsum[tg + b * TG] = q ? bsum[tg + b * TG] + sb[b] : sb[b];
        }
        __syncthreads();
      }
      for (int e = t; e < TM * TM; e += T) {
        const int o = e / TM, k = e % TM;
        if (k0 + k < K) out[(int64_t)(o0 + o) * (K + 1) + k0 + k] = sum[e];
      }
      if (tk == 0 && t < TM) out[(int64_t)(o0 + t) * (K + 1) + K] = bsum[t];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int o = o0 + orow + (i >> 2) * 16 + (i & 3), k = k0 + kcol + (h >> 1) * 32 + (h & 1) * 2;
          float lo, hi;
          unpack2(acc[i][h], lo, hi);
          if (k < K) out[(int64_t)o * (K + 1) + k] = lo;
          if (k + 1 < K) out[(int64_t)o * (K + 1) + k + 1] = hi;
        }
      if (tk == 0) {
#pragma unroll
        for (int b = 0; b < OB; ++b)
          if (tg + b * TG < TM) out[(int64_t)(o0 + tg + b * TG) * (K + 1) + K] = sb[b];
      }
    }
    clear();
    out += (int64_t)O * (K + 1);
  }
  cp_wait<0>();
}

// ---------------------------------------------------------------------------
// The partial sums into the FP64 gradient, every layer in one launch.  A job's entry e sums S partials `stride`
// floats apart; its gradient place is off + e, or, for rows of K weights and a bias, offW / offb.  An entry's
// partials go to `ways` threads, each sums its share (sum_parts), and the shares are added in FP64 in a fixed order,
// so nothing depends on timing.  The FP64 pipe bounds the launch unless an entry costs few FP64 instructions: one
// thread per entry where S is small or the entries many (they alone fill the chip), 8 or 32 where it is not (a block then reads 32
// or 8 neighbouring entries, whole sectors).  FP32 sums of two or three partials by 32 warps, FP64 from there: 16.8 us
// for 16.6K entries of 76 partials; this form 7.9.
// ---------------------------------------------------------------------------
constexpr int kRedThreads = 256;
int red_ways(int64_t S, int64_t entries) {
  return S <= 64 || (S <= 128 && entries >= 65536) ? 1 : S <= 256 ? 8 : 32;
}
struct RedJob {
  const float* part;
  int64_t stride, S, entries;
  int K;  // > 0: entry e is (row e / (K + 1), column e % (K + 1)), the last column the bias
  int ways;
  int64_t offW, offb;
  int first;  // first block
};
struct RedArgs {
  int n;
  RedJob job[kMaxLayers + 2];
  const double* vpart;  // virtual loss: per-block FP64 sums (NULL: none), added by the last block
  int64_t nv;
  double* value;
};

__global__ void __launch_bounds__(kRedThreads)
    reduce_kernel(const __grid_constant__ RedArgs a, int accumulate, double* __restrict__ grad) {
  __shared__ double red[kRedThreads];
  const int t = threadIdx.x;
  if (a.vpart && blockIdx.x == gridDim.x - 1) {
    double s = 0.0;
    for (int64_t i = t; i < a.nv; i += kRedThreads) s += a.vpart[i];
    red[t] = s;
    __syncthreads();
    if (t < 32) {
      s = 0.0;
#pragma unroll
      for (int w = 0; w < kRedThreads / 32; ++w) s += red[t + 32 * w];
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (t == 0) *a.value = accumulate ? *a.value + s : s;
    }
    return;
  }
  int j = 0;
  while (j + 1 < a.n && (int)blockIdx.x >= a.job[j + 1].first) ++j;
  const RedJob& J = a.job[j];
  const int per = kRedThreads / J.ways;  // entries per block
  const int64_t e = (int64_t)(blockIdx.x - J.first) * per + t % per;
  double tot = e < J.entries ? sum_parts(J.part + e, J.stride, t / per, J.ways, J.S) : 0.0;
  if (J.ways > 1) {
    red[t] = tot;
    __syncthreads();
    if (t >= per) return;
    double s[4] = {};
    for (int w = 0; w < J.ways; w += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += red[t + (w + u) * per];
    tot = (s[0] + s[1]) + (s[2] + s[3]);
  }
  if (e >= J.entries) return;
  const int row = J.K + 1, o = (int)e / row, k = (int)e % row;  // entries < 2^31
  const int64_t dst = k < J.K ? J.offW + (int64_t)o * J.K + k : J.offb + o;
  grad[dst] = accumulate ? grad[dst] + tot : tot;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Rows of the shared activation buffer: W, or the layer-1 input up to 256 columns.
int act_rows(const Net& n) { return std::max(n.W, std::min((n.K0 + 1) & ~1, 256)); }

// Points per thread: 8, or 4 where the points are too few to give every SM eight warps of 8-point threads
// (128^2 points, width 64: 512 warps over 152 SMs).  Fewer points per thread load more weights per multiply-add.
int points_per_thread(const Net& n, int64_t npts) {
  return (npts + 63) / 64 * (n.W / 32) < 8 * 152 ? 4 : 8;
}

size_t point_smem(const Net& n, int pt) {
  return sizeof(float) * ((size_t)act_rows(n) * (8 * pt + 4) + (size_t)kStages * kKc * n.W);
}

template <int PT, int NW, bool VJP>
int launch_points_t(const Net& n, const NetDev& nd, const LayerOffs& lo, const PointArgs& g, cudaStream_t st) {
  const size_t sm = point_smem(n, PT);
  const cudaError_t e = cudaFuncSetAttribute(point_kernel<PT, NW, VJP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) {
    set_error("point kernel shared memory (%zu bytes): %s", sm, cudaGetErrorString(e));
    return INRCT_ERR_CUDA;
  }
  point_kernel<PT, NW, VJP><<<ceil_div(g.npts, 8 * PT), 64 * NW, sm, st>>>(nd, lo, g);
  INRCT_CHECK_LAUNCH("point kernel");
  return INRCT_OK;
}

template <bool VJP>
int launch_points(const Net& n, const NetDev& nd, const LayerOffs& lo, const PointArgs& g, cudaStream_t st) {
  const bool big = points_per_thread(n, g.npts) == 8;
  switch (n.W) {
    case 64: return big ? launch_points_t<8, 1, VJP>(n, nd, lo, g, st) : launch_points_t<4, 1, VJP>(n, nd, lo, g, st);
    case 128: return big ? launch_points_t<8, 2, VJP>(n, nd, lo, g, st) : launch_points_t<4, 2, VJP>(n, nd, lo, g, st);
    default: return big ? launch_points_t<8, 4, VJP>(n, nd, lo, g, st) : launch_points_t<4, 4, VJP>(n, nd, lo, g, st);
  }
}

void layer_offs(const Net& n, LayerOffs* lo) {
  for (int l = 0; l <= n.L; ++l) {
    lo->W[l] = n.offW[l];
    lo->b[l] = n.offb[l];
  }
}

int copy_weights(const Net& n, const float* theta, const WeightCopies& wc, float* buf, cudaStream_t st) {
  CopyArgs a;
  a.L = n.L;
  a.W = n.W;
  int64_t most = 0;
  for (int l = 0; l < n.L; ++l) {
    a.in[l] = n.in_dim[l];
    a.offW[l] = n.offW[l];
    a.Wt[l] = wc.Wt[l];
    a.Wc[l] = wc.Wc[l];
    most = std::max<int64_t>(most, (int64_t)n.in_dim[l] * n.W);
  }
  copy_weights_kernel<<<dim3((unsigned)std::min<int64_t>(ceil_div(most, 256), 512), n.L), 256, 0, st>>>(theta, a, buf);
  INRCT_CHECK_LAUNCH("weight copies");
  return INRCT_OK;
}

// Layers with a dW GEMM: those whose input is stored (the SIREN's first and the output layer come from the
// point kernel's block sums).
int first_dw_layer(const Net& n) { return n.kind == INRCT_SIREN ? 1 : 0; }
int dw_tile(const Net& n) { return n.W >= 128 ? 128 : 64; }
int64_t dw_tiles(const Net& n) {
  const int tm = dw_tile(n);
  int64_t c = 0;
  for (int l = first_dw_layer(n); l < n.L; ++l) c += (int64_t)(n.W / tm) * ceil_div(n.in_dim[l], tm);
  return c;
}
// Splits of the points: enough (tile, split) blocks for two waves of two per SM of a 152-SM part (64-wide networks,
// whose blocks add kDwGroups groups of points themselves: one wave), at least 64 points per split.  A fixed SM count
// keeps the workspace size a function of the network and the chunk alone.
constexpr int kDwGroups = 4;
int dw_splits(const Net& n, int64_t npts) {
  const int64_t tiles = dw_tiles(n);
  if (tiles == 0) return 0;
  const int64_t S = std::min<int64_t>(std::max<int64_t>((dw_tile(n) == 128 ? 4 : 2) * 152 / tiles, 1), ceil_div(npts, 64));
  return (int)std::max<int64_t>(S, 1);
}
// FP32 sums that a block forms one after the other for layer l.  The splits serve all layers together, so those of many
// layers are long, and with them the sums (SIREN 9 x 256 and 2^16 points: 3450 points in a row, error of the gradient
// against 64 bits 1.5e-7 -> 2.9e-7): a layer takes as many as four blocks per SM of 64 x 64 tiles would make for it
// alone (1725 points, 1.5e-7), unless the splits make two thirds of them.  VJP of 2^14 points of a ReLU 8 x 256: 1050
// us without, 1068 with; of 2^12, where the partials double, 364 and 402.  More splits instead, for the layer or for
// all, end in a wave that is nearly empty (ReLU 3 x 256, 2^16 points: 1279 us for 1211).
int dw_runs(const Net& n, int l, int64_t npts) {
  const int64_t tiles64 = (int64_t)(n.W / 64) * ceil_div(n.in_dim[l], 64);
  const int64_t sums = std::min<int64_t>(ceil_div(4 * 152, tiles64), ceil_div(npts, 64));
  const int64_t shared = (int64_t)dw_splits(n, npts) * (dw_tile(n) == 128 ? 1 : kDwGroups);
  return 2 * sums <= 3 * shared ? 1 : (int)ceil_div(sums, shared);
}

struct VjpWs {
  float *wbuf, *E, *A, *D, *part, *bpart;
  double* vpart;
};

size_t vjp_layout(const Net& n, int64_t chunk, void* ws, size_t cap, VjpWs* out, bool* ok) {
  Carver c(ws, cap);
  VjpWs w;
  w.wbuf = c.take<float>(weight_copies(n, true).total);
  w.E = n.kind == INRCT_SIREN ? nullptr : c.take<float>(chunk * n.K0);
  w.A = c.take<float>(chunk * n.L * n.W);
  w.D = c.take<float>(chunk * n.L * n.W);
  int64_t pe = 0;
  for (int l = first_dw_layer(n); l < n.L; ++l) pe += (int64_t)n.W * (n.in_dim[l] + 1) * dw_splits(n, chunk) * dw_runs(n, l, chunk);
  w.part = c.take<float>(pe);
  const int64_t blocks = ceil_div(chunk, 32);  // the most blocks either point kernel takes
  w.bpart = c.take<float>(blocks * block_partial_cols(n.kind, n.W, n.d));
  w.vpart = c.take<double>(blocks);
  if (out) *out = w;
  if (ok) *ok = c.ok;
  return c.off + 256;
}

int launch_dw(const Net& n, const VjpWs& w, int64_t np, RedArgs* R, int* red_blocks, cudaStream_t st) {
  const int tm = dw_tile(n), S = dw_splits(n, np);
  const int G = tm == 128 ? 1 : kDwGroups;  // 64-wide networks: groups of 64 threads share a tile (fewer partials)
  DwArgs a;
  a.n = 0;
  a.npts = np;
  int tile = 0;
  int64_t off = 0;
  auto red = [&](const float* part, int64_t stride, int64_t S, int64_t rows, int K, int64_t offW, int64_t offb) {
    RedJob& J = R->job[R->n++];
    J.part = part;
    J.stride = stride;
    J.S = S;
    J.entries = rows * (K + 1);
    J.K = K;
    J.offW = offW;
    J.offb = offb;
    J.first = *red_blocks;
    J.ways = red_ways(S, J.entries);
    *red_blocks += ceil_div(J.entries, kRedThreads / J.ways);
  };
  for (int l = first_dw_layer(n); l < n.L; ++l) {
    DwJob& J = a.job[a.n++];
    J.X = w.D + (int64_t)l * np * n.W;
    J.Y = l == 0 ? w.E : w.A + (int64_t)(l - 1) * np * n.W;
    J.O = n.W;
    J.K = n.in_dim[l];
    J.tiles_k = ceil_div(J.K, tm);
    J.first = tile;
    J.part = off;
    J.runs = dw_runs(n, l, np);
    const int64_t sums = (int64_t)S * J.runs;
    J.run_rounds = (int)ceil_div(ceil_div(np, sums), kDk * G);
    tile += (n.W / tm) * J.tiles_k;
    red(w.part + off, (int64_t)n.W * (J.K + 1), sums, n.W, J.K, n.offW[l], n.offb[l]);
    off += sums * n.W * (J.K + 1);
  }
  if (tile > 0) {
    const size_t sm = sizeof(float) * (kDStages * G * 2 * kDk * tm + (G > 1 ? tm * tm + tm : 0));  // two blocks per SM
    const void* fn = tm == 128 ? (const void*)dw_kernel<128, 1> : (const void*)dw_kernel<64, kDwGroups>;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) {
      set_error("dW kernel shared memory (%zu bytes): %s", sm, cudaGetErrorString(e));
      return INRCT_ERR_CUDA;
    }
    if (tm == 128) dw_kernel<128, 1><<<dim3(tile, S), 256, sm, st>>>(a, w.part);
    else dw_kernel<64, kDwGroups><<<dim3(tile, S), 256, sm, st>>>(a, w.part);
    INRCT_CHECK_LAUNCH("dW");
  }
  const int64_t blocks = ceil_div(np, 8 * points_per_thread(n, np));
  const int cols = block_partial_cols(n.kind, n.W, n.d);
  red(w.bpart, cols, blocks, 1, n.W, n.offW[n.L], n.offb[n.L]);
  if (n.kind == INRCT_SIREN) red(w.bpart + n.W + 1, cols, blocks, n.W, n.d, n.offW[0], n.offb[0]);
  return INRCT_OK;
}

}  // namespace

// The kernels take an input of any width; the bound is the path's documented range (tested up to it), which was the
// shared memory of 16 points' inputs and activations.
bool simt_supported(const Net& n, char* why, size_t len) {
  constexpr int kMaxColumns = 3618;
  if (n.K0 + n.W <= kMaxColumns) return true;
  snprintf(why, len, "%d input columns exceed %d at width %d", n.K0, kMaxColumns - n.W, n.W);
  return false;
}

size_t simt_eval_ws_bytes(const Net& n) { return align_up(sizeof(float) * weight_copies(n, false).total, 256) + 256; }

// The hash gather reads both features of a vertex in one 8-byte load.
int check_theta_alignment(const Net& n, const float* theta, const char* who) {
  if (n.kind == INRCT_HASH && (reinterpret_cast<uintptr_t>(theta) & 7) != 0) {
    set_error("%s: theta must be 8-byte aligned for the hash-encoded INR", who);
    return INRCT_ERR_INVALID_ARG;
  }
  return INRCT_OK;
}

// The asynchronous copies and vector accesses want the scratch on 16-byte boundaries; the sizes carry 256 bytes
// for a workspace that does not start on one.
void align_ws(void*& ws, size_t& ws_bytes) {
  const size_t shift = ws ? (16 - (reinterpret_cast<uintptr_t>(ws) & 15)) & 15 : 0;
  if (shift == 0 || ws_bytes < shift) return;
  ws = static_cast<char*>(ws) + shift;
  ws_bytes -= shift;
}

// A step's evaluation and VJP read the same weights: copied once for both, where the step's workspace has room (one
// launch of 3.8 us less; a call by itself copies its own).
size_t simt_weights_bytes(const Net& n) { return sizeof(float) * weight_copies(n, true).total + 256; }

int simt_prepare(const Net& n, const float* theta, void* buf, size_t bytes, cudaStream_t st) {
  INRCT_TRY(check_theta_alignment(n, theta, "inr_eval_grid"));
  align_ws(buf, bytes);
  return copy_weights(n, theta, weight_copies(n, true), static_cast<float*>(buf), st);
}

int simt_eval(const Net& n, const float* theta, int N, int64_t npts, float* image, void* ws,
              size_t ws_bytes, cudaStream_t st, const void* prepared) {
  INRCT_TRY(check_theta_alignment(n, theta, "inr_eval_grid"));
  const size_t need = simt_eval_ws_bytes(n);
  const WeightCopies wc = weight_copies(n, prepared != nullptr);
  if (!ws || ws_bytes < need) {
    set_error("inr_eval_grid (fp32): workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  void* buf = prepared ? const_cast<void*>(prepared) : ws;
  size_t room = prepared ? simt_weights_bytes(n) : ws_bytes;
  align_ws(buf, room);
  float* wbuf = static_cast<float*>(buf);
  if (!prepared) INRCT_TRY(copy_weights(n, theta, wc, wbuf, st));
  LayerOffs lo;
  layer_offs(n, &lo);
  PointArgs g{};
  g.theta = theta;
  g.wbuf = wbuf;
  g.wc = wc;
  g.npts = npts;
  g.out_f = image;
  g.rows = act_rows(n);
  prof_mark(kMarkEvalKernel, st);
  INRCT_TRY(launch_points<false>(n, dev_of(n, N), lo, g, st));
  prof_mark(kMarkEvalDone, st);
  return INRCT_OK;
}

size_t simt_vjp_ws_bytes(const Net& n, int64_t n_idx) {
  const int64_t chunk = n_idx < kVjpChunk ? n_idx : kVjpChunk;
  return vjp_layout(n, chunk, nullptr, 0, nullptr, nullptr);
}

int simt_vjp(const Net& n, const float* theta, int N, const int32_t* idx, int64_t n_idx,
             const float* v, double scale, double* grad_f64, float* grad_f32, double* value_out,
             void* ws, size_t ws_bytes, cudaStream_t st, const void* prepared) {
  INRCT_TRY(check_theta_alignment(n, theta, "inr_weighted_vjp"));
  const int64_t chunk = n_idx < kVjpChunk ? n_idx : kVjpChunk;
  VjpWs w;
  bool ok;
  align_ws(ws, ws_bytes);
  const size_t need = vjp_layout(n, chunk, ws, ws_bytes, &w, &ok);
  if (!ws || !ok) {
    set_error("inr_weighted_vjp (fp32): workspace of %zu bytes too small (need %zu)", ws_bytes, need);
    return INRCT_ERR_WORKSPACE;
  }
  LayerOffs lo;
  layer_offs(n, &lo);
  PointArgs g{};
  g.theta = theta;
  g.wbuf = w.wbuf;
  g.wc = weight_copies(n, true);
  g.rows = act_rows(n);
  g.v = v;
  g.scale = (float)scale;
  g.A = w.A;
  g.D = w.D;
  g.E = w.E;
  g.bpart = w.bpart;
  g.vpart = value_out ? w.vpart : nullptr;
  g.gtab = n.n_table > 0 ? grad_f64 : nullptr;
  if (prepared) {
    void* buf = const_cast<void*>(prepared);
    size_t room = simt_weights_bytes(n);
    align_ws(buf, room);
    g.wbuf = static_cast<float*>(buf);
  } else {
    INRCT_TRY(copy_weights(n, theta, g.wc, w.wbuf, st));
  }
  if (n.n_table > 0) {
    const cudaError_t e = cudaMemsetAsync(grad_f64, 0, sizeof(double) * n.n_table, st);
    if (e != cudaSuccess) {
      set_error("hash table gradient clear: %s", cudaGetErrorString(e));
      return INRCT_ERR_CUDA;
    }
  }
  const NetDev nd = dev_of(n, N);
  for (int64_t c0 = 0; c0 < n_idx; c0 += chunk) {
    const int64_t np = std::min(chunk, n_idx - c0);
    g.npts = np;
    g.idx = idx + c0;
    if (c0 == 0) prof_mark(kMarkVjpKernel, st);
    INRCT_TRY(launch_points<true>(n, nd, lo, g, st));
    if (c0 == 0) prof_mark(kMarkVjpKernelDone, st);
    RedArgs R{};
    int blocks = 0;
    INRCT_TRY(launch_dw(n, w, np, &R, &blocks, st));
    if (value_out) {
      R.vpart = w.vpart;
      R.nv = ceil_div(np, 8 * points_per_thread(n, np));
      R.value = value_out;
      ++blocks;
    }
    reduce_kernel<<<blocks, kRedThreads, 0, st>>>(R, c0 > 0, grad_f64);
    INRCT_CHECK_LAUNCH("gradient reduce");
  }
  if (grad_f32) INRCT_TRY(f64_to_f32(grad_f64, grad_f32, n.p, st));
  return INRCT_OK;
}

}  // namespace inrct
