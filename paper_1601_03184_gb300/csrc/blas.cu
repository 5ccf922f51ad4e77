// BLAS-like operations on interleaved multi-RHS arrays (Sec. 5 of the paper:
// with the right-hand sides innermost these are elementwise per RHS; the
// global sums are taken for all right-hand sides in one pass).
// Arrays are `rows` complex rows of [2][N]: element (row, re/im, rhs).
// Reductions use a fixed two-level tree (per-CTA partials, then a fixed-order
// sum), so results are bitwise reproducible.
#include <algorithm>
#include <cstdint>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace mrhs {
namespace {

constexpr int kBlock = 256;

int n_chunks(size_t rows, int N) {
  size_t work = rows * (size_t)N;
  size_t ch = work / (kBlock * 64);
  if (ch < 1) ch = 1;
  if (ch > 2048) ch = 2048;
  return (int)ch;
}

// partial[k][chunk][r] = sum over the chunk's rows of conj(X_k) * Y, for the
// group of up to KG vectors k = KG*blockIdx.y + j: every element of Y read
// serves the whole group. A thread takes VEC right-hand sides of a row (VEC =
// 4: FP32, N % 4 == 0, 16-byte loads), Q = N / VEC threads a row, and a warp
// 32 / Q rows at a time (a row spans warps when Q > 32). Bound by the loads when
// there are enough rows; at few rows (coarse fields) by the sums across the
// threads, and there by FP64, which this GPU adds at 2 per clock and SM.
// Without PAIR a thread adds its (FP32) sums of kFlush rows in FP64 and the threads are
// joined by a tree in FP64. With PAIR (FP32 data, N <= 32 VEC) a thread sums its rows, at
// most kMaxRows or with VEC = 1 kFlush, in FP32, and the threads are joined, by shuffles
// and then across the warps, in pairs of FP32 numbers (two-sums: 48 bits, where the rows'
// own sums have 24); a pair that leaves the range of FP32 sends the CTA to the same joins
// in FP64. (Over plain FP32 shuffles, five roundings more, the pairs cost 1 us of a call
// of 16384 x 32.)
// A chunk is one CTA, or a cluster of two, four or eight while all CTAs still run
// together, two to an SM: the ranks take equal parts of the chunk and the first adds their
// sums in order, so that the partials, and the workspace they need, stay one per chunk.
// More CTAs than that only repeat the joins: with clusters of eight below 304 CTAs
// altogether (before) and by this rule, 152 SMs, per call: 1, 5, 10 and 20 vectors of 16384 x 32
// 12.4, 20.6, 30.8, 53.7 -> 12.3, 16.5, 18.5, 28.7 us; of 12800 x 20 12.4, 16.5, 24.6, 38.8
// -> 12.4, 16.5, 18.5, 30.8; of 98304 x 24 36, 96, 79, 146 -> 16, 53, 79, 145. 1 vector
// of 4096 rows, one CTA a chunk and a serial FP64 sum: 97 us; now 10.
constexpr int kKG = 4;          // vectors per group (its sums: up to 40 KB of shared memory)
constexpr int kKGWide = 2;      // the same for VEC = 4 and more than kWide right-hand sides
constexpr int kWide = 64;
constexpr int kFlush = 32;
constexpr int kMaxRows = 128;
constexpr int kClusterCtas = 8;
template <class S, int VEC>
__device__ __forceinline__ void ld_row(const S* p, typename Real<S>::type v[VEC]) {
  if constexpr (VEC == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
  } else {
    v[0] = to_r(p[0]);
  }
}

// rows that one pass of a CTA covers
__host__ __device__ __forceinline__ int dot_lanes(int Q) { return Q <= 32 ? (kBlock / 32) * (32 / Q) : kBlock / Q; }

// (hi, lo) += (h, l)
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h, float l) {
  const float s = __fadd_rn(hi, h), b = __fsub_rn(s, hi);
  lo = __fadd_rn(__fadd_rn(lo, l), __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(h, b)));
  hi = s;
}

template <class S, int VEC, int KG, bool PAIR>
__global__ void __launch_bounds__(kBlock, 2) k_multi_dot(const S* __restrict__ X, size_t stride, int K,
                                                         const S* __restrict__ Y, size_t rows, int N, int nchunk,
                                                         int ranks, double* __restrict__ part) {
  using R = typename Real<S>::type;
  // the threads' sums [KG][lanes][N], lanes N <= kBlock; or the warps' pairs
  // [KG][8 warps][N] float4, KG N <= 64 VEC
  constexpr int kN = PAIR ? (VEC == 4 ? kBlock : 32 * KG) : KG * kBlock;
  __shared__ double2 buf[PAIR ? 8 * kN : kN];
  __shared__ double2 res[kN];  // [KG][N]
  const int k0 = blockIdx.y * KG, ch = blockIdx.x / ranks, rank = blockIdx.x % ranks;
  const int nk = min(KG, K - k0);
  size_t r0 = rows * ch / nchunk, r1 = rows * (ch + 1) / nchunk;
  if (ranks > 1) {
    const size_t n = r1 - r0, base = r0;
    r0 = base + n * rank / ranks, r1 = base + n * (rank + 1) / ranks;
  }
  const int tid = threadIdx.x, Q = N / VEC, lanes = dot_lanes(Q);
  const bool warp_rows = Q <= 32;
  const int lw = warp_rows ? 32 / Q : 1;                      // rows of a warp
  const int wlane = warp_rows ? (tid & 31) / Q : 0;           // this thread's row among them
  const int q = warp_rows ? (tid & 31) % Q : tid % Q;
  const int lane = warp_rows ? (tid >> 5) * lw + wlane : tid / Q;
  const bool on = warp_rows ? wlane < lw : lane < lanes;
  constexpr bool FLUSH = !PAIR;
  static_assert(PAIR || VEC == 1, "lanes N <= kBlock");
  double are[FLUSH ? KG : 1][VEC], aim[FLUSH ? KG : 1][VEC];
  R pre[KG][VEC], pim[KG][VEC];
#pragma unroll
  for (int j = 0; j < KG; ++j)
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      if (FLUSH) are[j][e] = aim[j][e] = 0;
      pre[j][e] = pim[j][e] = 0;
    }
  if (on) {
    int cnt = 0;
    for (size_t row = r0 + lane; row < r1; row += lanes) {
      R yr[VEC], yi[VEC];
      ld_row<S, VEC>(Y + fidx(row, 0, N, VEC * q), yr);
      ld_row<S, VEC>(Y + fidx(row, 1, N, VEC * q), yi);
#pragma unroll
      for (int j = 0; j < KG; ++j) {
        if (j < nk) {
          const S* Xk = X + (size_t)(k0 + j) * stride;
          R xr[VEC], xi[VEC];
          ld_row<S, VEC>(Xk + fidx(row, 0, N, VEC * q), xr);
          ld_row<S, VEC>(Xk + fidx(row, 1, N, VEC * q), xi);
#pragma unroll
          for (int e = 0; e < VEC; ++e) {
            pre[j][e] = fma(xr[e], yr[e], fma(xi[e], yi[e], pre[j][e]));
            pim[j][e] = fma(xr[e], yi[e], fma(-xi[e], yr[e], pim[j][e]));
          }
        }
      }
      if (FLUSH && ++cnt == kFlush) {
#pragma unroll
        for (int j = 0; j < KG; ++j)
#pragma unroll
          for (int e = 0; e < VEC; ++e)
            are[j][e] += pre[j][e], aim[j][e] += pim[j][e], pre[j][e] = pim[j][e] = 0;
        cnt = 0;
      }
    }
  }
  if constexpr (FLUSH) {
#pragma unroll
    for (int j = 0; j < KG; ++j)
      if (on && j < nk)
        buf[j * kBlock + lane * N + q] = make_double2(are[j][0] + (double)pre[j][0], aim[j][0] + (double)pim[j][0]);
    __syncthreads();
    int half = 1;  // the largest power of two below the number of lanes
    while (2 * half < lanes) half *= 2;
    if (lanes > 1)
      for (int h = half; h > 0; h >>= 1) {
        for (int e = tid; e < h * N && e + h * N < lanes * N; e += kBlock)
          for (int j = 0; j < nk; ++j) {
            double2& t = buf[j * kBlock + e];
            const double2 o = buf[j * kBlock + e + h * N];
            t.x += o.x, t.y += o.y;
          }
        __syncthreads();
      }
    for (int e = tid; e < nk * N; e += kBlock) res[e] = buf[(e / N) * kBlock + e % N];
  } else {
    float4* wsum = reinterpret_cast<float4*>(buf);  // (re hi, re lo, im hi, im lo)
    constexpr int kWarps = kBlock / 32;
    const int unit = tid >> 5;
    int half = 1;
    while (2 * half < lw) half *= 2;
    if (lw == 1) half = 0;
#pragma unroll
    for (int j = 0; j < KG; ++j) {
      if (j >= nk) break;
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        float a = pre[j][e], b = pim[j][e], al = 0.f, bl = 0.f;
        for (int h = half; h > 0; h >>= 1) {
          const float oa = __shfl_down_sync(0xffffffffu, a, h * Q), ob = __shfl_down_sync(0xffffffffu, b, h * Q);
          float ol = 0.f, pl = 0.f;
          if (h < half) ol = __shfl_down_sync(0xffffffffu, al, h * Q), pl = __shfl_down_sync(0xffffffffu, bl, h * Q);
          if (wlane < h && wlane + h < lw) pair_add(a, al, oa, ol), pair_add(b, bl, ob, pl);
        }
        if (on && wlane == 0) wsum[(j * kWarps + unit) * N + VEC * q + e] = make_float4(a, al, b, bl);
      }
    }
    __syncthreads();
    bool left = false;  // the range of FP32 (or the data are not finite)
    for (int e = tid; e < nk * N; e += kBlock) {
      const float4* w = wsum + (size_t)(e / N) * kWarps * N + e % N;
      float4 t = w[0];
#pragma unroll
      for (int u = 1; u < kWarps; ++u) {
        const float4 o = w[u * N];
        pair_add(t.x, t.y, o.x, o.y), pair_add(t.z, t.w, o.z, o.w);
      }
      left = left || !isfinite(t.x) || !isfinite(t.z);
      res[e] = make_double2((double)t.x + (double)t.y, (double)t.z + (double)t.w);
    }
    if (__syncthreads_or(left)) {
#pragma unroll
      for (int j = 0; j < KG; ++j) {
        if (j >= nk) break;
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
          double a = pre[j][e], b = pim[j][e];
          for (int h = half; h > 0; h >>= 1) {
            const double oa = __shfl_down_sync(0xffffffffu, a, h * Q), ob = __shfl_down_sync(0xffffffffu, b, h * Q);
            if (wlane < h && wlane + h < lw) a += oa, b += ob;
          }
          if (on && wlane == 0) buf[unit * N + VEC * q + e] = make_double2(a, b);
        }
        __syncthreads();
        for (int r = tid; r < N; r += kBlock) {
          double2 t = buf[r];
          for (int u = 1; u < kWarps; ++u) t.x += buf[u * N + r].x, t.y += buf[u * N + r].y;
          res[j * N + r] = t;
        }
        __syncthreads();
      }
    }
  }
  if (ranks > 1) cg::this_cluster().sync();
  else __syncthreads();
  if (rank == 0) {
    for (int e = tid; e < nk * N; e += kBlock) {
      double2 t = res[e];
      for (int c = 1; c < ranks; ++c) {
        const double2 o = *cg::this_cluster().map_shared_rank(&res[e], c);
        t.x += o.x, t.y += o.y;
      }
      *reinterpret_cast<double2*>(part + (((size_t)(k0 + e / N) * nchunk + ch) * N + e % N) * 2) = t;
    }
  }
  if (ranks > 1) cg::this_cluster().sync();  // the ranks' shared memory stays until it has been read
}

// out[k][r] = sum over the chunks of part[k][chunk][r]: one warp per (k, r),
// lane l adds chunks l, l+32, ... and the lanes are joined by a fixed
// butterfly, so the order of the sum does not depend on timing; out32 (may be
// null): the same rounded to FP32, the coefficients of a following multi_axpy
__global__ void k_sum_chunks(const double* part, int K, int nchunk, int N, double* out, float* out32) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (t >= K * N) return;
  const int k = t / N, r = t % N;
  double a = 0, b = 0;
  for (int ch = lane; ch < nchunk; ch += 32) {
    a += part[(((size_t)k * nchunk + ch) * N + r) * 2];
    b += part[(((size_t)k * nchunk + ch) * N + r) * 2 + 1];
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    out[2 * t] = a;
    out[2 * t + 1] = b;
    if (out32) *reinterpret_cast<float2*>(out32 + 2 * t) = make_float2((float)a, (float)b);
  }
}

// coefficients in the compute precision, once per (k, r)
__global__ void k_coef_to_float(const double* coef, float* out, int n) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) out[t] = (float)coef[t];
}

template <class S, class C>
__global__ void k_multi_axpy(const S* X, size_t stride, int K, S* Y, size_t rows, int N, const C* coef, C sign) {
  using R = typename Real<S>::type;
  size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= rows * N) return;
  int r = (int)(t % N);
  size_t row = t / N;
  R yr = to_r(Y[fidx(row, 0, N, r)]), yi = to_r(Y[fidx(row, 1, N, r)]);
  for (int k = 0; k < K; ++k) {
    R cr = (R)(sign * coef[((size_t)k * N + r) * 2]), ci = (R)(sign * coef[((size_t)k * N + r) * 2 + 1]);
    const S* Xk = X + (size_t)k * stride;
    R xr = to_r(Xk[fidx(row, 0, N, r)]), xi = to_r(Xk[fidx(row, 1, N, r)]);
    yr = fma(cr, xr, fma(-ci, xi, yr));
    yi = fma(cr, xi, fma(ci, xr, yi));
  }
  Y[fidx(row, 0, N, r)] = from_r<S>(yr);
  Y[fidx(row, 1, N, r)] = from_r<S>(yi);
}

// FP32, N % 4 == 0: four right-hand sides per thread, 16-byte loads and
// stores (the scalar kernel's operations in its order: the same bits)
__global__ void k_multi_axpy4(const float* __restrict__ X, size_t stride, int K, float* __restrict__ Y, size_t rows,
                              int N, const float* __restrict__ coef, float sign) {
  const int Q = N / 4;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= rows * Q) return;
  const int q = (int)(t % Q);
  const size_t row = t / Q;
  float4* py = reinterpret_cast<float4*>(Y + fidx(row, 0, N, 4 * q));
  float4* pyi = reinterpret_cast<float4*>(Y + fidx(row, 1, N, 4 * q));
  const float4 y0 = *py, y1 = *pyi;
  float yr[4] = {y0.x, y0.y, y0.z, y0.w}, yi[4] = {y1.x, y1.y, y1.z, y1.w};
  for (int k = 0; k < K; ++k) {
    const float4 c01 = *reinterpret_cast<const float4*>(coef + ((size_t)k * N + 4 * q) * 2);
    const float4 c23 = *reinterpret_cast<const float4*>(coef + ((size_t)k * N + 4 * q) * 2 + 4);
    const float cr[4] = {sign * c01.x, sign * c01.z, sign * c23.x, sign * c23.z};
    const float ci[4] = {sign * c01.y, sign * c01.w, sign * c23.y, sign * c23.w};
    const float* Xk = X + (size_t)k * stride;
    const float4 x0 = *reinterpret_cast<const float4*>(Xk + fidx(row, 0, N, 4 * q));
    const float4 x1 = *reinterpret_cast<const float4*>(Xk + fidx(row, 1, N, 4 * q));
    const float xr[4] = {x0.x, x0.y, x0.z, x0.w}, xi[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      yr[e] = fmaf(cr[e], xr[e], fmaf(-ci[e], xi[e], yr[e]));
      yi[e] = fmaf(cr[e], xi[e], fmaf(ci[e], xr[e], yi[e]));
    }
  }
  *py = make_float4(yr[0], yr[1], yr[2], yr[3]);
  *pyi = make_float4(yi[0], yi[1], yi[2], yi[3]);
}

// s[r] = 1/sqrt(nrm2[r]) (0 for a zero vector), once per right-hand side
__global__ void k_inv_sqrt(const double* nrm2, double* s, int N) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  double n = nrm2[2 * r];
  s[r] = n > 0 ? 1.0 / sqrt(n) : 0.0;
}

// X[., r] *= s[r]
template <class S>
__global__ void k_scale_by(S* X, size_t rows, int N, const double* s) {
  using R = typename Real<S>::type;
  size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= rows * N) return;
  int r = (int)(t % N);
  size_t row = t / N;
  R f = (R)s[r];
  X[fidx(row, 0, N, r)] = from_r<S>(to_r(X[fidx(row, 0, N, r)]) * f);
  X[fidx(row, 1, N, r)] = from_r<S>(to_r(X[fidx(row, 1, N, r)]) * f);
}

// the four-RHS kernels need FP32, N % 4 == 0 and 16-byte aligned rows
bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }
bool use_dot4(const void* X, size_t stride, const void* Y, int N, int dtype) {
  return dtype == MRHS_F32 && N % 4 == 0 && N <= 128 && aligned16(X) && aligned16(Y) && stride % 4 == 0;
}

}  // namespace

size_t multi_dot_partials_bytes(size_t rows, int N, int K) {
  return sizeof(double) * 2 * (size_t)K * n_chunks(rows, N) * N;
}

// part: a buffer of multi_dot_partials_bytes(rows, N, K) bytes
void multi_dot_ws(mrhs_ctx c, const void* X, size_t stride, int K, const void* Y, size_t rows, int N, int dtype,
                  double* out, double* part, float* out32) {
  MRHS_REQUIRE(N >= 1 && N <= kBlock && K >= 1, MRHS_ERR_ARG, "multi_dot: bad sizes");
  const int nch = n_chunks(rows, N);
  const bool four = use_dot4(X, stride, Y, N, dtype);
  // rows that a thread would sum with one CTA per chunk
  auto thread_rows = [&](int vec) { return (rows / nch) / dot_lanes(N / vec) + 1; };
  const bool four_ok = four && thread_rows(4) <= kMaxRows;
  const int kg = four_ok && N > kWide ? kKGWide : kKG;
  const int groups = (K + kg - 1) / kg;
  int ranks = kClusterCtas;
  while (ranks > 1 && nch * groups * ranks > 2 * c->num_sms) ranks /= 2;
  const bool one_ok = dtype == MRHS_F32 && N <= 32 && thread_rows(1) / ranks + 1 <= kFlush;
  Prof pr(c, "multi_dot");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nch * ranks, groups);
  cfg.blockDim = dim3(kBlock);
  cfg.stream = c->stream;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ranks, at.val.clusterDim.y = 1, at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = ranks > 1 ? 1 : 0;
  if (four_ok || one_ok) {
    auto kern = !four_ok ? k_multi_dot<float, 1, kKG, true>
                : kg == kKG ? k_multi_dot<float, 4, kKG, true> : k_multi_dot<float, 4, kKGWide, true>;
    MRHS_CUDA(cudaLaunchKernelEx(&cfg, kern, (const float*)X, stride, K, (const float*)Y, rows, N, nch, ranks, part));
  } else {
    MRHS_DISPATCH(dtype, S, {
      MRHS_CUDA(cudaLaunchKernelEx(&cfg, k_multi_dot<S, 1, kKG, false>, (const S*)X, stride, K, (const S*)Y, rows, N, nch,
                                   ranks, part));
    });
  }
  MRHS_LAUNCH_CHECK("multi_dot");
  k_sum_chunks<<<grid_for((size_t)K * N * 32, 256), 256, 0, c->stream>>>(part, K, nch, N, out, out32);
  MRHS_LAUNCH_CHECK("sum_chunks");
}

void multi_dot(mrhs_ctx c, const void* X, size_t stride, int K, const void* Y, size_t rows, int N, int dtype,
               double* out, float* out32) {
  MRHS_REQUIRE(N >= 1 && N <= kBlock && K >= 1, MRHS_ERR_ARG, "multi_dot: bad sizes");
  double* part = (double*)scratch(c, SC_RED, multi_dot_partials_bytes(rows, N, K));
  multi_dot_ws(c, X, stride, K, Y, rows, N, dtype, out, part, out32);
}

// out[r] (as [N][2], imaginary part 0) = |X_r|^2
void norms(mrhs_ctx c, const void* X, size_t rows, int N, int dtype, double* out) {
  multi_dot(c, X, 0, 1, X, rows, N, dtype, out);
}

// coef32 (may be null): the coefficients in FP32 as a multi_dot has left them;
// otherwise they are converted here
void multi_axpy(mrhs_ctx c, const void* X, size_t stride, int K, void* Y, size_t rows, int N, int dtype,
                const double* coef, double sign, const float* coef32) {
  size_t work = rows * N;
  Prof pr(c, "multi_axpy");
  if (dtype == MRHS_F64) {
    k_multi_axpy<double, double><<<grid_for(work, kBlock), kBlock, 0, c->stream>>>((const double*)X, stride, K, (double*)Y, rows, N, coef, sign);
  } else {
    MRHS_REQUIRE(K <= 65 && N <= 256, MRHS_ERR_ARG, "multi_axpy: K <= 65 and N <= 256");
    if (!coef32) {
      const int n = 2 * K * N;
      k_coef_to_float<<<grid_for(n, 256), 256, 0, c->stream>>>(coef, c->coef32, n);
      coef32 = c->coef32;
    }
    const float sg = sign < 0 ? -1.f : 1.f;
    if (dtype == MRHS_F32 && N % 4 == 0 && aligned16(X) && aligned16(Y) && stride % 4 == 0)
      k_multi_axpy4<<<grid_for(rows * (N / 4), kBlock), kBlock, 0, c->stream>>>((const float*)X, stride, K, (float*)Y,
                                                                                rows, N, coef32, sg);
    else
      MRHS_DISPATCH(dtype, S, (k_multi_axpy<S, float><<<grid_for(work, kBlock), kBlock, 0, c->stream>>>((const S*)X, stride, K, (S*)Y, rows, N, coef32, sg)));
  }
  MRHS_LAUNCH_CHECK("multi_axpy");
}

// normalise every right-hand side of X to unit 2-norm
namespace {
// |X[., r]|^2 of a fine FP32 field (N / 4 divides 256, 16-byte aligned rows):
// thread (quad of right-hand sides, lane) over a grid-stride range of rows,
// FP32 sums over 64 rows at a time added into FP64; the lanes of a quad summed
// in a fixed order, then the CTAs (k_norm2_sum)
constexpr int kNormCtas = 608;
__global__ void __launch_bounds__(kBlock) k_norm2_4(const float* __restrict__ X, size_t rows, int N,
                                                    double* __restrict__ part) {
  __shared__ double sh[kBlock * 4];
  const int nq = N / 4, lanes = kBlock / nq;
  const int q = threadIdx.x % nq, lane = threadIdx.x / nq;
  double acc[4] = {0, 0, 0, 0};
  float f[4] = {0.f, 0.f, 0.f, 0.f};
  int cnt = 0;
  for (size_t row = (size_t)blockIdx.x * lanes + lane; row < rows; row += (size_t)gridDim.x * lanes) {
    const float4 re = __ldg(reinterpret_cast<const float4*>(X + row * 2 * N + 4 * q));
    const float4 im = __ldg(reinterpret_cast<const float4*>(X + row * 2 * N + N + 4 * q));
    f[0] = fmaf(re.x, re.x, fmaf(im.x, im.x, f[0]));
    f[1] = fmaf(re.y, re.y, fmaf(im.y, im.y, f[1]));
    f[2] = fmaf(re.z, re.z, fmaf(im.z, im.z, f[2]));
    f[3] = fmaf(re.w, re.w, fmaf(im.w, im.w, f[3]));
    if (++cnt == 64) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[e] += f[e], f[e] = 0.f;
      cnt = 0;
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) sh[lane * N + 4 * q + e] = acc[e] + f[e];
  __syncthreads();
  if (threadIdx.x < N) {
    double t = 0;
    for (int l = 0; l < lanes; ++l) t += sh[l * N + threadIdx.x];
    part[(size_t)blockIdx.x * N + threadIdx.x] = t;
  }
}
__global__ void k_norm2_sum(const double* part, int nblk, int N, double* out) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  double t = 0;
  for (int b = 0; b < nblk; ++b) t += part[(size_t)b * N + r];
  out[2 * r] = t;
  out[2 * r + 1] = 0;
}

// tv = (X[., r] * s[r]) * scale in the storage type of tv: the normalised
// vectors converted in one pass (the same two roundings as scaling X in
// place and converting it)
template <class SI, class SO>
__global__ void k_scale_convert(const SI* __restrict__ X, SO* __restrict__ T, size_t rows, int N,
                                const double* __restrict__ s, float scale) {
  using R = typename Real<SI>::type;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t >= rows * 2 * N) return;
  const int r = (int)(t % N);
  const R v = (R)(to_r(X[t]) * (R)s[r]);
  T[t] = from_r<SO>(v * (R)scale);
}

// the same four values at a time for FP32 X (N % 4 == 0, 16-byte aligned)
template <class SO>
__device__ __forceinline__ void store4(SO* p, float a, float b, float c, float d);
template <>
__device__ __forceinline__ void store4<float>(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<double>(double* p, float a, float b, float c, float d) {
  p[0] = a, p[1] = b, p[2] = c, p[3] = d;
}
template <>
__device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float a, float b, float c, float d) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
template <>
__device__ __forceinline__ void store4<__half>(__half* p, float a, float b, float c, float d) {
  __half2 lo = __floats2half2_rn(a, b), hi = __floats2half2_rn(c, d);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
// resident CTAs per SM of k_scale_convert4 (256 threads each)
constexpr int kScaleCtasPerSm = 8;
// loads in flight per thread in k_scale_convert4
constexpr int kScaleUnroll = 4;

// the same four values at a time for FP32 X on a persistent grid: the
// grid-stride step is a multiple of N/4 float4, so a thread keeps the same
// four right-hand sides (and their factors) throughout, and it keeps
// kScaleUnroll loads in flight; the products are those of k_scale_convert
template <class SO>
__global__ void __launch_bounds__(kBlock) k_scale_convert4(const float* __restrict__ X, SO* __restrict__ T, size_t n4,
                                                           int N, const double* __restrict__ s, float scale) {
  const int nq = N / 4;
  const size_t G = (size_t)gridDim.x * blockDim.x;
  const size_t step = G - G % (size_t)nq;
  const size_t t0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (t0 >= step) return;
  const int r = 4 * (int)(t0 % (size_t)nq);
  const float s0 = (float)s[r], s1 = (float)s[r + 1], s2 = (float)s[r + 2], s3 = (float)s[r + 3];
  const float4* X4 = reinterpret_cast<const float4*>(X);
  size_t t = t0;
  for (; t + (kScaleUnroll - 1) * step < n4; t += kScaleUnroll * step) {
    float4 v[kScaleUnroll];
#pragma unroll
    for (int u = 0; u < kScaleUnroll; ++u) v[u] = __ldg(X4 + t + u * step);
#pragma unroll
    for (int u = 0; u < kScaleUnroll; ++u)
      store4<SO>(T + 4 * (t + u * step), (v[u].x * s0) * scale, (v[u].y * s1) * scale, (v[u].z * s2) * scale,
                 (v[u].w * s3) * scale);
  }
  for (; t < n4; t += step) {
    const float4 v = __ldg(X4 + t);
    store4<SO>(T + 4 * t, (v.x * s0) * scale, (v.y * s1) * scale, (v.z * s2) * scale, (v.w * s3) * scale);
  }
}

void norms_of_field(mrhs_ctx c, const void* X, size_t rows, int N, int dtype, double* nrm) {
  if (dtype == MRHS_F32 && N % 4 == 0 && kBlock % (N / 4) == 0 && aligned16(X)) {
    double* part = (double*)scratch(c, SC_RED, sizeof(double) * kNormCtas * (size_t)N);
    Prof pr(c, "norms");
    k_norm2_4<<<kNormCtas, kBlock, 0, c->stream>>>((const float*)X, rows, N, part);
    MRHS_LAUNCH_CHECK("norm2_4");
    k_norm2_sum<<<grid_for(N, 64), 64, 0, c->stream>>>(part, kNormCtas, N, nrm);
    MRHS_LAUNCH_CHECK("norm2_sum");
    return;
  }
  norms(c, X, rows, N, dtype, nrm);
}
}  // namespace

// T = X / |X[., r]| * scale in T's storage type (X unchanged)
void normalise_into(mrhs_ctx c, const void* X, int dx, void* T, int dt, size_t rows, int N, float scale) {
  double* nrm = (double*)scratch(c, SC_MISC, sizeof(double) * 3 * N);
  norms_of_field(c, X, rows, N, dx, nrm);
  k_inv_sqrt<<<grid_for(N, 64), 64, 0, c->stream>>>(nrm, nrm + 2 * N, N);
  MRHS_LAUNCH_CHECK("inv_sqrt");
  const size_t work = rows * 2 * N;
  Prof pr(c, "normalise");
  const size_t n4 = work / 4;
  const int grid = (int)std::min<size_t>((size_t)std::max(c->num_sms, 1) * kScaleCtasPerSm, (n4 + kBlock - 1) / kBlock);
  // (the persistent form needs a grid of at least N/4 threads)
  if (dx == MRHS_F32 && dt != MRHS_F64 && N % 4 == 0 && aligned16(X) && aligned16(T) &&
      (size_t)grid * kBlock >= (size_t)(N / 4)) {
    MRHS_DISPATCH(dt, SO, (k_scale_convert4<SO><<<grid, kBlock, 0, c->stream>>>((const float*)X, (SO*)T, n4, N, nrm + 2 * N, scale)));
    MRHS_LAUNCH_CHECK("scale_convert4");
    return;
  }
  MRHS_DISPATCH(dx, SI, MRHS_DISPATCH(dt, SO, (k_scale_convert<SI, SO><<<grid_for(work, kBlock), kBlock, 0, c->stream>>>((const SI*)X, (SO*)T, rows, N, nrm + 2 * N, scale))));
  MRHS_LAUNCH_CHECK("scale_convert");
}

void normalise_rhs(mrhs_ctx c, void* X, size_t rows, int N, int dtype) {
  double* nrm = (double*)scratch(c, SC_MISC, sizeof(double) * 3 * N);
  norms_of_field(c, X, rows, N, dtype, nrm);
  k_inv_sqrt<<<grid_for(N, 64), 64, 0, c->stream>>>(nrm, nrm + 2 * N, N);
  MRHS_LAUNCH_CHECK("inv_sqrt");
  size_t work = rows * N;
  Prof pr(c, "normalise");
  MRHS_DISPATCH(dtype, S, (k_scale_by<S><<<grid_for(work, kBlock), kBlock, 0, c->stream>>>((S*)X, rows, N, nrm + 2 * N)));
  MRHS_LAUNCH_CHECK("normalise");
}

}  // namespace mrhs
