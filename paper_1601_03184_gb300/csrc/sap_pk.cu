// SAP sweep (Sec. 2 of the paper; red-black multiplicative Schwarz with
// minimal-residual block solves) with the domain on chip and the arithmetic
// on packed pairs of right-hand sides.
//
// Per colour, one CTA per (domain, chunk of 4 right-hand sides), as in
// sap_tm.cu, but a thread owns one SITE and a PAIR of right-hand sides
// (thread t: site t/2, pair t%2 of the chunk) instead of two (site, rhs)
// items: every complex operation is one .f32x2 instruction on the pair, and
// the links and the clover term of the site are loaded once for both
// right-hand sides of the pair.
//   shared memory  rho [12][Va][2] float4 = (re_a, re_b, im_a, im_b) of the
//                  pair and the domain-local neighbour table [8][Va] (the
//                  domain's halved links [20][Va+1] float4 too in the "2s"
//                  form; by default the links are read through L1);
//   tensor memory  the running solution x_B of the thread's pair
//                  (48 columns: 12 components x (re_a, re_b, im_a, im_b)) and
//                  a copy of the clover term of the thread's site (72
//                  columns), staged once per CTA: the five applications of D
//                  per chunk read it there instead of from global memory;
//   registers      q = D_B rho between the reduction for alpha and the
//                  update.
// Per colour and chunk: r = b - D x on the domain (neighbours outside it from
// x in global memory, owned by the other colour and not written during the
// launch), then n_mr MR steps e += alpha rho, rho -= alpha q with
// alpha = <q, rho> / <q, q> per right-hand side, then x_B += e.
#include <algorithm>
#include <cstdlib>
#include <string>

#include "stencil.cuh"
#include "tc.cuh"

namespace mrhs {
namespace {

// PP pairs of right-hand sides per chunk: PP = 2 (512 threads for a 256-site
// domain, one CTA per SM) or PP = 1 (256 threads, two CTAs per SM); LG: the
// links read from global memory (through L1) instead of staged in shared
// memory, which leaves room for the second CTA
constexpr int kPCols = 48;    // tensor-memory columns of one thread's x_B
constexpr int kPClov = 72;    // tensor-memory columns of its site's clover term
constexpr int kPWarpCols = kPCols + kPClov;

struct DomP {
  const float4* sR;  // [12][Va][PP]
  const float4* sU;  // [20][Va+1]: float4 k of link mu at row mu*5 + k
  const int* sN;     // [8][Va]: neighbour inside the domain (local) or ~(device site)
  uint32_t tclov;    // tensor-memory address of the thread's copy of its site's clover term
  int Va, l, p;
  size_t s0;
};

template <int PP>
__device__ __forceinline__ c2 ldR(const DomP& d, int c, int n) {
  const float4 v = d.sR[(c * d.Va + n) * PP + d.p];
  return mk2(make_float2(v.x, v.y), make_float2(v.z, v.w));
}

__device__ __forceinline__ void ld_link(const float4* src, int stride, float u[20]) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float4 t = src[k * stride];
    u[4 * k] = t.x, u[4 * k + 1] = t.y, u[4 * k + 2] = t.z, u[4 * k + 3] = t.w;
  }
}
// link mu of device site n from global memory (read-only path)
__device__ __forceinline__ void ld_link_g(const float* __restrict__ U20, size_t n, int mu, float u[20]) {
  const float4* src = reinterpret_cast<const float4*>(U20 + (n * 4 + mu) * 20);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float4 t = __ldg(src + k);
    u[4 * k] = t.x, u[4 * k + 1] = t.y, u[4 * k + 2] = t.z, u[4 * k + 3] = t.w;
  }
}

// o += hop (MU, DIR) at the thread's site for its pair: the neighbour spinor
// from shared memory inside the domain; outside it (RESID only) from x, with
// the link of a backward hop from global memory. The two halves of the
// projected spinor (h_0 from spins 0 and SB0, h_1 from spins 1 and SB1) are
// done one after the other, so that only one half is live in registers; each
// half feeds one upper and one lower spin of o.
template <int MU, int DIR, int SP>
__device__ __forceinline__ void half_pk(c2 o[12], const c2 h[3], const float u[20]) {
  using Tb = BTab<MU>;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    c2 ch;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      // U[a][b] forward, conj(U[b][a]) backward (the sign of the time
      // boundary and the factor 1/2 are folded into the stored links)
      const int q = DIR > 0 ? a * 3 + b : b * 3 + a;
      const float2 ure = bc2(u[2 * q]);
      const float2 uim = bc2(DIR > 0 ? u[2 * q + 1] : -u[2 * q + 1]);
      const float2 nuim = bc2(DIR > 0 ? -u[2 * q + 1] : u[2 * q + 1]);
      const c2 hv = h[b];
      if (b == 0) {
        ch.re = mul2(ure, hv.re);
        ch.im = mul2(ure, hv.im);
      } else {
        ch.re = fma2(ure, hv.re, ch.re);
        ch.im = fma2(ure, hv.im, ch.im);
      }
      ch.re = fma2(nuim, hv.im, ch.re);
      ch.im = fma2(uim, hv.re, ch.im);
    }
    // upper spin SP -= chi_SP; the lower spin that B^dag takes chi_SP to
    o[3 * SP + a] = o[3 * SP + a] - ch;
    if (Tb::SD0 == SP) o[6 + a] = axpy_ph<Tb::KD0, DIR>(o[6 + a], ch);
    if (Tb::SD1 == SP) o[9 + a] = axpy_ph<Tb::KD1, DIR>(o[9 + a], ch);
  }
}

template <int MU, int DIR, bool RESID, int PP, bool LG>
__device__ __forceinline__ void hop_pk(const DomP& d, c2 o[12], const float* __restrict__ x,
                                       const float* __restrict__ U20, int N, int r0) {
  using Tb = BTab<MU>;
  const int e = d.sN[((DIR > 0 ? 0 : 4) + MU) * d.Va + d.l];
  if (!RESID && e < 0) return;
  float u[20];
  const float* xn = nullptr;
  if (e >= 0) {
    if (LG) ld_link_g(U20, d.s0 + (DIR > 0 ? d.l : e), MU, u);
    else ld_link(d.sU + MU * 5 * (d.Va + 1) + (DIR > 0 ? d.l : e), d.Va + 1, u);
  } else {
    const size_t n = (size_t)(~e);
    xn = x + n * 24 * N + r0 + 2 * d.p;
    if (DIR > 0) {
      if (LG) ld_link_g(U20, d.s0 + d.l, MU, u);
      else ld_link(d.sU + MU * 5 * (d.Va + 1) + d.l, d.Va + 1, u);
    } else {
      ld_link(reinterpret_cast<const float4*>(U20 + (n * 4 + MU) * 20), 1, u);
    }
  }
  auto ld = [&](int comp) -> c2 {
    if (e >= 0) return ldR<PP>(d, comp, e);
    return mk2(*reinterpret_cast<const float2*>(xn + (2 * comp) * N),
               *reinterpret_cast<const float2*>(xn + (2 * comp + 1) * N));
  };
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_ph<Tb::KB0, -DIR>(ld(c), ld(3 * Tb::SB0 + c));
    half_pk<MU, DIR, 0>(o, h, u);
  }
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_ph<Tb::KB1, -DIR>(ld(3 + c), ld(3 * Tb::SB1 + c));
    half_pk<MU, DIR, 1>(o, h, u);
  }
}

// o = D x (RESID: x inside the domain from shared memory, outside from global
// memory) or o = D_B rho (couplings leaving the domain dropped)
template <bool RESID, int PP, bool LG>
__device__ __forceinline__ void apply_pk(const DomP& d, c2 o[12], const float* __restrict__ Acl,
                                         const float* __restrict__ x, const float* __restrict__ U20, int N,
                                         int r0) {
  {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float q[36];
      tc::tmem_ld36(d.tclov + 36 * h, q);
      c2 ps[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) ps[a] = ldR<PP>(d, 6 * h + a, d.l);
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        const float2 qa = bc2(q[a]);
        c2 acc = mk2(mul2(ps[a].re, qa), mul2(ps[a].im, qa));
#pragma unroll
        for (int b2 = 0; b2 < 6; ++b2) {
          if (b2 == a) continue;
          const int ei = b2 > a ? herm_idx(a, b2) : herm_idx(b2, a);
          const float mim = b2 > a ? q[ei + 1] : -q[ei + 1];
          const float2 mre2 = bc2(q[ei]), mim2 = bc2(mim), nmim2 = bc2(-mim);
          acc.re = fma2(mre2, ps[b2].re, acc.re);
          acc.re = fma2(nmim2, ps[b2].im, acc.re);
          acc.im = fma2(mre2, ps[b2].im, acc.im);
          acc.im = fma2(mim2, ps[b2].re, acc.im);
        }
        o[6 * h + a] = acc;
      }
    }
  }
  // one hop per iteration of a loop the compiler keeps rolled, so that it does
  // not start the loads of later hops early (they would not fit in the
  // registers next to o)
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    switch (k) {
      case 0: hop_pk<0, +1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 1: hop_pk<1, +1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 2: hop_pk<2, +1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 3: hop_pk<3, +1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 4: hop_pk<0, -1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 5: hop_pk<1, -1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      case 6: hop_pk<2, -1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
      default: hop_pk<3, -1, RESID, PP, LG>(d, o, x, U20, N, r0); break;
    }
  }
}

// a pair of right-hand sides of b (two consecutive values) in FP32
__device__ __forceinline__ float2 ld_pair(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 ld_pair(const double* p) { return make_float2((float)p[0], (float)p[1]); }
__device__ __forceinline__ float2 ld_pair(const __nv_bfloat16* p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}
__device__ __forceinline__ float2 ld_pair(const __half* p) {
  return __half22float2(*reinterpret_cast<const __half2*>(p));
}

__device__ __forceinline__ void xb_put(uint32_t ta, const c2 v[12]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float f[16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const c2 t = v[4 * k + i];
      f[4 * i] = t.re.x, f[4 * i + 1] = t.re.y, f[4 * i + 2] = t.im.x, f[4 * i + 3] = t.im.y;
    }
    tc::tmem_st16(ta + 16 * k, f);
  }
}

template <class SB, int PP, bool LG>
__global__ void __launch_bounds__(256 * PP, 3 - PP) k_sap_pk(const SB* __restrict__ b, float* __restrict__ x,
                                                      const float* __restrict__ U20, const float* __restrict__ Acl,
                                                      const int* __restrict__ nbr, int N, int Va,
                                                      const int* __restrict__ blist, int n_mr, uint32_t tm_cols,
                                                      int cpb, int x0z) {
  extern __shared__ float4 smem4[];
  const int T = blockDim.x;
  constexpr int kG = 2 * PP;                                          // right-hand sides per chunk
  float4* sU = smem4;                                                 // [20][Va+1] (not LG)
  float4* sR = LG ? smem4 : sU + 20 * (Va + 1);                       // [12][Va][PP]
  float2* sred = reinterpret_cast<float2*>(sR + 12 * PP * Va);        // [T/32][PP][3]
  int* sN = reinterpret_cast<int*>(sred + (T / 32) * PP * 3);        // [8][Va]
  __shared__ uint32_t s_tmem;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  DomP d;
  d.Va = Va;
  d.l = tid / PP;
  d.p = tid % PP;
  const bool valid = d.l < Va;
  if (!valid) d.l = 0;  // idle threads read site 0 and write nothing
  d.s0 = (size_t)blist[blockIdx.x / cpb] * Va;
  d.sR = sR;
  d.sU = sU;
  d.sN = sN;

  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, tm_cols);
    tc::tmem_relinquish();
  }
  {
    const float4* U4 = reinterpret_cast<const float4*>(U20) + d.s0 * 20;
    if (!LG)
      for (int i = tid; i < 20 * Va; i += T) sU[(i % 20) * (Va + 1) + i / 20] = __ldg(U4 + i);
    for (int i = tid; i < 8 * Va; i += T) {
      const int l = i >> 3, k = i & 7;
      const int n = __ldg(nbr + (d.s0 + l) * 8 + k) & 0x3fffffff;
      const int nl = n - (int)d.s0;
      sN[k * Va + l] = (nl >= 0 && nl < Va) ? nl : ~n;
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  // lane quarter of the warp; warps w, w+4, w+8, w+12 share it and take
  // disjoint column ranges of kPCols
  const uint32_t tm = s_tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * kPWarpCols);
  d.tclov = tm + kPCols;
  {
    // the clover term of the thread's site -> tensor memory (72 columns)
    const float4* A4 = reinterpret_cast<const float4*>(Acl + (d.s0 + d.l) * 72);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float f[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = __ldg(A4 + 4 * k + i);
        f[4 * i] = v.x, f[4 * i + 1] = v.y, f[4 * i + 2] = v.z, f[4 * i + 3] = v.w;
      }
      tc::tmem_st16(d.tclov + 16 * k, f);
    }
    float f[8];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 v = __ldg(A4 + 16 + i);
      f[4 * i] = v.x, f[4 * i + 1] = v.y, f[4 * i + 2] = v.z, f[4 * i + 3] = v.w;
    }
    tc::tmem_st8(d.tclov + 64, f);
    tc::tmem_wait_st();
  }

  for (int r0 = (blockIdx.x % cpb) * kG; r0 < N; r0 += cpb * kG) {
    // stage x0: one (component c, site l) per unit, the real and imaginary
    // rows of the chunk's right-hand sides become the pairs' float4
    // (re_a, re_b, im_a, im_b)
    // (x0z: x = 0 everywhere, the stage and D x0 are skipped)
    for (int u = x0z ? 12 * Va : tid; u < 12 * Va; u += T) {
      const int c = u / Va, l = u % Va;
      const float* xs = x + ((d.s0 + l) * 24 + 2 * c) * N + r0;
      if (PP == 2) {
        const float4 re = *reinterpret_cast<const float4*>(xs);
        const float4 im = *reinterpret_cast<const float4*>(xs + N);
        sR[(c * Va + l) * 2] = make_float4(re.x, re.y, im.x, im.y);
        sR[(c * Va + l) * 2 + 1] = make_float4(re.z, re.w, im.z, im.w);
      } else {
        const float2 re = *reinterpret_cast<const float2*>(xs);
        const float2 im = *reinterpret_cast<const float2*>(xs + N);
        sR[c * Va + l] = make_float4(re.x, re.y, im.x, im.y);
      }
    }
    __syncthreads();
    c2 o[12];
    // x_B = x0 of the thread's pair -> tensor memory; then q0 = D x0
#pragma unroll
    for (int c = 0; c < 12; ++c) o[c] = x0z ? mk2(make_float2(0.f, 0.f), make_float2(0.f, 0.f)) : ldR<PP>(d, c, d.l);
    xb_put(tm, o);
    if (!x0z) apply_pk<true, PP, LG>(d, o, Acl, x, U20, N, r0);
    tc::tmem_wait_st();
    __syncthreads();  // every read of x0 in shared memory is done
    // rho = b - D x0 at the thread's site
    if (valid) {
      const SB* bs = b + (d.s0 + d.l) * 24 * N + r0 + 2 * d.p;
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        const float2 bre = ld_pair(bs + (2 * c) * N), bim = ld_pair(bs + (2 * c + 1) * N);
        const c2 r = mk2(sub2(bre, o[c].re), sub2(bim, o[c].im));
        sR[(c * Va + d.l) * PP + d.p] = make_float4(r.re.x, r.re.y, r.im.x, r.im.y);
      }
    }
    __syncthreads();
    for (int step = 0; step < n_mr; ++step) {
      float2 pr = make_float2(0.f, 0.f), pi = pr, pq = pr;
      apply_pk<false, PP, LG>(d, o, Acl, x, U20, N, r0);  // o = q = D_B rho
      if (valid) {
#pragma unroll
        for (int c = 0; c < 12; ++c) {
          const c2 r = ldR<PP>(d, c, d.l);
          pr = fma2(o[c].re, r.re, fma2(o[c].im, r.im, pr));
          pi = fma2(o[c].re, r.im, fma2(make_float2(-o[c].im.x, -o[c].im.y), r.re, pi));
          pq = fma2(o[c].re, o[c].re, fma2(o[c].im, o[c].im, pq));
        }
      }
      // sums over the sites of the warp (lanes of the same pair parity),
      // then over the warps in order: every thread of a pair gets the same
      // alpha for both of its right-hand sides
#pragma unroll
      for (int s = PP; s < 32; s <<= 1) {
        pr.x += __shfl_xor_sync(0xffffffffu, pr.x, s);
        pr.y += __shfl_xor_sync(0xffffffffu, pr.y, s);
        pi.x += __shfl_xor_sync(0xffffffffu, pi.x, s);
        pi.y += __shfl_xor_sync(0xffffffffu, pi.y, s);
        pq.x += __shfl_xor_sync(0xffffffffu, pq.x, s);
        pq.y += __shfl_xor_sync(0xffffffffu, pq.y, s);
      }
      if (lane < PP) {
        sred[(warp * PP + lane) * 3] = pr;
        sred[(warp * PP + lane) * 3 + 1] = pi;
        sred[(warp * PP + lane) * 3 + 2] = pq;
      }
      __syncthreads();
      float2 a = make_float2(0.f, 0.f), bb = a, cc = a;
      for (int w = 0; w < T / 32; ++w) {
        const float2 t0 = sred[(w * PP + d.p) * 3], t1 = sred[(w * PP + d.p) * 3 + 1],
                     t2 = sred[(w * PP + d.p) * 3 + 2];
        a.x += t0.x, a.y += t0.y;
        bb.x += t1.x, bb.y += t1.y;
        cc.x += t2.x, cc.y += t2.y;
      }
      const float2 alr = make_float2(cc.x > 0.f ? a.x / cc.x : 0.f, cc.y > 0.f ? a.y / cc.y : 0.f);
      const float2 ali = make_float2(cc.x > 0.f ? bb.x / cc.x : 0.f, cc.y > 0.f ? bb.y / cc.y : 0.f);
      const float2 nali = make_float2(-ali.x, -ali.y);
      // x_B += alpha rho (tensor memory), rho -= alpha q (shared memory)
      // four components (16 tensor-memory columns) at a time
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float f[16];
        tc::tmem_ld16(tm + 16 * k, f);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 4 * k + i;
            c2 xv = mk2(make_float2(f[4 * i], f[4 * i + 1]), make_float2(f[4 * i + 2], f[4 * i + 3]));
            c2 r = ldR<PP>(d, c, d.l);
            xv.re = fma2(alr, r.re, xv.re);
            xv.re = fma2(nali, r.im, xv.re);
            xv.im = fma2(alr, r.im, xv.im);
            xv.im = fma2(ali, r.re, xv.im);
            // rho += alpha (-q)
            const c2 nq = mk2(make_float2(-o[c].re.x, -o[c].re.y), make_float2(-o[c].im.x, -o[c].im.y));
            r.re = fma2(alr, nq.re, r.re);
            r.re = fma2(nali, nq.im, r.re);
            r.im = fma2(alr, nq.im, r.im);
            r.im = fma2(ali, nq.re, r.im);
            sR[(c * Va + d.l) * PP + d.p] = make_float4(r.re.x, r.re.y, r.im.x, r.im.y);
            f[4 * i] = xv.re.x, f[4 * i + 1] = xv.re.y, f[4 * i + 2] = xv.im.x, f[4 * i + 3] = xv.im.y;
          }
        }
        tc::tmem_st16(tm + 16 * k, f);
      }
      tc::tmem_wait_st();
      __syncthreads();
    }
    // x = x_B for the thread's site and pair
    {
      float* xs = x + (d.s0 + d.l) * 24 * N + r0 + 2 * d.p;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float f[16];
        tc::tmem_ld16(tm + 16 * k, f);
        if (valid) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 4 * k + i;
            *reinterpret_cast<float2*>(xs + (2 * c) * N) = make_float2(f[4 * i], f[4 * i + 1]);
            *reinterpret_cast<float2*>(xs + (2 * c + 1) * N) = make_float2(f[4 * i + 2], f[4 * i + 3]);
          }
        }
      }
    }
    __syncthreads();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(s_tmem, tm_cols);
}

// ---------------------------------------------------------------------------
// The form for domains of more than 128 sites and at least two sweeps: one pair of
// right-hand sides per CTA, a thread per site, two CTAs per SM, on copies of x and b
// laid out as the CTA reads them: per (domain, pair) a tile [12][Va] of (re_a, re_b,
// im_a, im_b). In the fields' own layout a chunk of right-hand sides is 8 or 16 bytes
// of every 128-byte row, and each warp access of that many rows took 34 cycles of the
// load/store unit: 53,000 of the 161,000 cycles of a k_sap_pk CTA (b 13,000, x0 7,000,
// the neighbours' faces 18,000, the clover term 4,000, x 11,000; 4^4 domain, 4 MR
// steps). From the tiles every access is a run of 16 bytes (the x faces) to 512. The
// copies cost one pass over b and two over x per call, not per launch.
//   - x0 of the domain goes into the rho tile and the neighbours' faces into slots
//     by cp.async: nF slots beside the rho tile (two at 4^4 domains, so that L1 keeps
//     the 82 KB of the domain's links for the SM's two CTAs) and, once D_B x0 is done,
//     as many as fit in the rho tile itself;
//   - b of the thread's site goes straight into the residual's registers;
//   - the residual is D_B x0 from shared memory like an MR step's product, then one
//     pass per direction over the sites at either face: a lane at the forward face
//     takes U h, one at the backward face U^dag h', with the signs and the
//     conjugate-transposed link selected per lane;
//   - the links have the sites innermost (k_links), so that a warp's 16-byte loads fall
//     into 4 lines each, not 32.
// What bounds it now: the packed FMAs (9,000 cycles of the 11,000 to 13,000 that two
// CTAs take for an application of D_B side by side) and, in the residual, the
// latency of its four copies in turn. Measured at 16^3x32, 4 sweeps of 4 steps, the
// copies included: 32 right-hand sides 8.66 -> 7.33 ms, 20: 5.41 -> 4.74; 32^3x64,
// 24, 5 sweeps: 122.2 -> 106.9 ms; 8^4, 20: 588 -> 388 us. Two pairs per CTA (one CTA
// of 512 threads per SM) took 8.20, 5.36 ms and 586 us, four right-hand sides per
// thread 10 ms. Domains of 128 sites and fewer fill half a CTA or less of this form
// and stay with k_sap_pk (16^4, 128 sites, 20: 2.60 against 2.54 ms; 81 sites: 5.68
// against 5.61; 16 sites: 8.2 against 12.6); a single sweep does not pay for the
// copies (3 passes, about 0.3 of a sweep).
struct SapGeo {
  int a[4], S[4], nf[4];  // extents, strides and face sizes of a domain
  int slot;               // float4 of a face slot (the largest face)
  int nF, nR;             // slots beside the rho tile and in it
};

// o += sg phase(ch): lower spins of a hop, sg = +1 (forward) or -1 per lane
template <int K>
__device__ __forceinline__ c2 axpy_sg(c2 a, c2 x, float sg) {
  constexpr bool nre = !(K == 0 || K == 3), nim = !(K == 0 || K == 1);
  return mk2(fma2(bc2(nre ? -sg : sg), (K & 1) ? x.im : x.re, a.re),
             fma2(bc2(nim ? -sg : sg), (K & 1) ? x.re : x.im, a.im));
}

// one half (SP) of a face hop; u is the link, conjugate-transposed already
// where the lane's hop is a backward one
template <int MU, int SP>
__device__ __forceinline__ void half_face(c2 o[12], const c2 h[3], const float u[18], float sg) {
  using Tb = BTab<MU>;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    c2 ch;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int q = a * 3 + b;
      const float2 ure = bc2(u[2 * q]), uim = bc2(u[2 * q + 1]), nuim = bc2(-u[2 * q + 1]);
      if (b == 0) {
        ch.re = mul2(ure, h[b].re);
        ch.im = mul2(ure, h[b].im);
      } else {
        ch.re = fma2(ure, h[b].re, ch.re);
        ch.im = fma2(ure, h[b].im, ch.im);
      }
      ch.re = fma2(nuim, h[b].im, ch.re);
      ch.im = fma2(uim, h[b].re, ch.im);
    }
    o[3 * SP + a] = o[3 * SP + a] - ch;
    if (Tb::SD0 == SP) o[6 + a] = axpy_sg<Tb::KD0>(o[6 + a], ch, sg);
    if (Tb::SD1 == SP) o[9 + a] = axpy_sg<Tb::KD1>(o[9 + a], ch, sg);
  }
}

struct DomH {
  const float4* sR;   // [12][Va]
  const float4* UQd;  // [20][Va]: the domain's links
  uint32_t tclov;
  int Va, l;
  int x[4];  // coordinates of the thread's site in the domain
};
__device__ __forceinline__ c2 ldH(const DomH& d, int c, int n) {
  const float4 v = d.sR[c * d.Va + n];
  return mk2(make_float2(v.x, v.y), make_float2(v.z, v.w));
}

// the face hops of direction MU: sx the slot of the face that the thread's
// site sees (its own side's), f the site's index in the face
template <int MU>
__device__ __forceinline__ void hop_face(const DomH& d, c2 o[12], const float4* sx, int nf, int f, bool fwd,
                                         const float4* __restrict__ UQ, int B, const SapGeo& g) {
  using Tb = BTab<MU>;
  float u[20];
  {
    const int ln = d.l + (g.a[MU] - 1) * g.S[MU];  // the neighbour of a backward hop, in its domain
    ld_link((fwd ? d.UQd + d.l : UQ + (size_t)B * 20 * d.Va + ln) + 5 * MU * d.Va, d.Va, u);
    if (!fwd) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        u[2 * (4 * i) + 1] = -u[2 * (4 * i) + 1];
#pragma unroll
        for (int j = i + 1; j < 3; ++j) {
          const int q = 3 * i + j, t = 3 * j + i;
          const float re = u[2 * q], im = u[2 * q + 1];
          u[2 * q] = u[2 * t], u[2 * q + 1] = -u[2 * t + 1];
          u[2 * t] = re, u[2 * t + 1] = -im;
        }
      }
    }
  }
  const float sg = fwd ? 1.f : -1.f;
  // slot: [12][nf]
  const float4* s4 = sx + f;
  auto ld = [&](int c) {
    const float4 v = s4[c * nf];
    return mk2(make_float2(v.x, v.y), make_float2(v.z, v.w));
  };
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_sg<Tb::KB0>(ld(c), ld(3 * Tb::SB0 + c), -sg);
    half_face<MU, 0>(o, h, u, sg);
  }
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_sg<Tb::KB1>(ld(3 + c), ld(3 * Tb::SB1 + c), -sg);
    half_face<MU, 1>(o, h, u, sg);
  }
}

template <int MU, int DIR>
__device__ __forceinline__ void hop_dom(const DomH& d, c2 o[12], const SapGeo& g) {
  using Tb = BTab<MU>;
  if (DIR > 0 ? d.x[MU] == g.a[MU] - 1 : d.x[MU] == 0) return;
  const int e = DIR > 0 ? d.l + g.S[MU] : d.l - g.S[MU];
  float u[20];
  ld_link(d.UQd + 5 * MU * d.Va + (DIR > 0 ? d.l : e), d.Va, u);
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_ph<Tb::KB0, -DIR>(ldH(d, c, e), ldH(d, 3 * Tb::SB0 + c, e));
    half_pk<MU, DIR, 0>(o, h, u);
  }
  {
    c2 h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) h[c] = axpy_ph<Tb::KB1, -DIR>(ldH(d, 3 + c, e), ldH(d, 3 * Tb::SB1 + c, e));
    half_pk<MU, DIR, 1>(o, h, u);
  }
}

__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
// o = D_B rho, or o = D_B rho - o (ADD)
template <bool ADD>
__device__ __forceinline__ void apply_dom(const DomH& d, c2 o[12], const SapGeo& g) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float q[36];
    tc::tmem_ld36(d.tclov + 36 * h, q);
    c2 ps[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) ps[a] = ldH(d, 6 * h + a, d.l);
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const float2 qa = bc2(q[a]);
      c2 acc;
      if (ADD) acc = mk2(fma2(ps[a].re, qa, neg2(o[6 * h + a].re)), fma2(ps[a].im, qa, neg2(o[6 * h + a].im)));
      else acc = mk2(mul2(ps[a].re, qa), mul2(ps[a].im, qa));
#pragma unroll
      for (int b2 = 0; b2 < 6; ++b2) {
        if (b2 == a) continue;
        const int ei = b2 > a ? herm_idx(a, b2) : herm_idx(b2, a);
        const float mim = b2 > a ? q[ei + 1] : -q[ei + 1];
        const float2 mre2 = bc2(q[ei]), mim2 = bc2(mim), nmim2 = bc2(-mim);
        acc.re = fma2(mre2, ps[b2].re, acc.re);
        acc.re = fma2(nmim2, ps[b2].im, acc.re);
        acc.im = fma2(mre2, ps[b2].im, acc.im);
        acc.im = fma2(mim2, ps[b2].re, acc.im);
      }
      o[6 * h + a] = acc;
    }
  }
  // (rolled for the same reason as in apply_pk)
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    switch (k) {
      case 0: hop_dom<0, +1>(d, o, g); break;
      case 1: hop_dom<1, +1>(d, o, g); break;
      case 2: hop_dom<2, +1>(d, o, g); break;
      case 3: hop_dom<3, +1>(d, o, g); break;
      case 4: hop_dom<0, -1>(d, o, g); break;
      case 5: hop_dom<1, -1>(d, o, g); break;
      case 6: hop_dom<2, -1>(d, o, g); break;
      default: hop_dom<3, -1>(d, o, g); break;
    }
  }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// start the copies of faces k0 <= k < k1 (k = 2 mu + (0 forward, 1 backward)) of
// the neighbouring domains' tiles into consecutive slots [12][face site]
__device__ __forceinline__ void fetch_faces(float4* slots, int k0, int k1, const int* nbd, const float4* xq, int nch,
                                            int ch, int Va, const SapGeo& g, int tid, int T) {
  for (int k = k0; k < k1; ++k) {
    const int mu = k >> 1, S = g.S[mu], a = g.a[mu], nf = g.nf[mu];
    const float4* xd = xq + ((size_t)nbd[k] * nch + ch) * 12 * Va;
    float4* dst = slots + (k - k0) * g.slot;
    const int side = (k & 1) ? (a - 1) * S : 0;
    if (T % nf == 0) {  // a thread keeps its face site
      const int f = tid % nf, l = f % S + f / S * S * a + side;
      for (int c = tid / nf; c < 12; c += T / nf) cp_async16(dst + c * nf + f, xd + c * Va + l);
    } else {
      for (int i = tid; i < 12 * nf; i += T) {
        const int f = i % nf, l = f % S + f / S * S * a + side;
        cp_async16(dst + i, xd + i / nf * Va + l);
      }
    }
  }
}

// xq, bq: tiles [domain][nch pairs][12][Va]; x is updated in place
__global__ void __launch_bounds__(256, 2) k_sap_face(const float4* __restrict__ bq, float4* xq,
                                                     const float4* __restrict__ UQ, const float* __restrict__ Acl,
                                                     const int* __restrict__ aggnbr, int nch, int Va,
                                                     const int* __restrict__ blist, int n_mr, uint32_t tm_cols, int x0z,
                                                     const __grid_constant__ SapGeo g) {
  extern __shared__ float4 smem4[];
  const int T = blockDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float4* sR = smem4;                                         // [12][Va]
  float4* sF = sR + 12 * Va;                                  // [nF][slot]
  float2* sred = reinterpret_cast<float2*>(sF + g.nF * g.slot);  // [T/32][3]
  int* nbd = reinterpret_cast<int*>(sred + (T / 32) * 3);    // [8]: the neighbouring domains, 2 mu + side
  __shared__ uint32_t s_tmem;
  const int A = blist[blockIdx.x / nch], ch = blockIdx.x % nch;
  const size_t tile = ((size_t)A * nch + ch) * 12 * Va;
  const size_t s0 = (size_t)A * Va;
  DomH d;
  d.Va = Va;
  d.l = tid;
  const bool valid = d.l < Va;
  if (!valid) d.l = 0;  // idle threads read site 0 and write nothing
  d.sR = sR;
  d.UQd = UQ + (size_t)A * 20 * Va;
  {
    int l = d.l;
#pragma unroll
    for (int m = 0; m < 4; ++m) d.x[m] = l % g.a[m], l /= g.a[m];
  }
  if (tid < 8) nbd[tid] = aggnbr[A * 8 + (tid & 1) * 4 + (tid >> 1)];
  if (!x0z)
    for (int i = tid; i < 12 * Va; i += T) cp_async16(sR + i, xq + tile + i);
  cp_commit();
  if (warp == 0) {
    tc::tmem_alloc(&s_tmem, tm_cols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (!x0z) fetch_faces(sF, 0, min(g.nF, 8), nbd, xq, nch, ch, Va, g, tid, T);
  cp_commit();
  // b of the thread's site and pair -> the residual's registers (negated where
  // they are first used, so that nothing waits for them here)
  c2 o[12];
  {
    const float4* bs = bq + tile + d.l;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const float4 v = __ldg(bs + c * Va);
      o[c] = mk2(make_float2(v.x, v.y), make_float2(v.z, v.w));
    }
  }
  const uint32_t tm = s_tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * kPWarpCols);
  d.tclov = tm + kPCols;
  {
    const float4* A4 = reinterpret_cast<const float4*>(Acl + (s0 + d.l) * 72);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float f[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = __ldg(A4 + 4 * k + i);
        f[4 * i] = v.x, f[4 * i + 1] = v.y, f[4 * i + 2] = v.z, f[4 * i + 3] = v.w;
      }
      tc::tmem_st16(d.tclov + 16 * k, f);
    }
    float f[8];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 v = __ldg(A4 + 16 + i);
      f[4 * i] = v.x, f[4 * i + 1] = v.y, f[4 * i + 2] = v.z, f[4 * i + 3] = v.w;
    }
    tc::tmem_st8(d.tclov + 64, f);
    tc::tmem_wait_st();
  }
  if (x0z) {
    // x_B = 0
    float f[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) f[i] = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) tc::tmem_st16(tm + 16 * k, f);
    tc::tmem_wait_st();
  } else {
    cp_wait<1>();  // x0 (the faces may still be on their way)
    __syncthreads();
    // x_B = x0 -> tensor memory
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float f[16];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const c2 t = ldH(d, 4 * k + i, d.l);
        f[4 * i] = t.re.x, f[4 * i + 1] = t.re.y, f[4 * i + 2] = t.im.x, f[4 * i + 3] = t.im.y;
      }
      tc::tmem_st16(tm + 16 * k, f);
    }
    tc::tmem_wait_st();
    apply_dom<true>(d, o, g);
    __syncthreads();  // every read of x0 in shared memory is done
    // the faces, in turn from the slots beside the rho tile and those in it;
    // both sides of a direction always come together
    int k0 = 0, k1 = min(g.nF, 8);  // the faces that have been fetched first
    bool in_f = true;
    while (k0 < 8) {
      const int k2 = min(k1 + (in_f ? g.nR : g.nF), 8);
      if (k2 > k1) fetch_faces(in_f ? sR : sF, k1, k2, nbd, xq, nch, ch, Va, g, tid, T);
      cp_commit();
      cp_wait<1>();
      __syncthreads();
      const float4* slots = in_f ? sF : sR;
#pragma unroll 1
      for (int mu = k0 >> 1; mu < (k1 >> 1); ++mu) {
        const int xm = mu == 0 ? d.x[0] : mu == 1 ? d.x[1] : mu == 2 ? d.x[2] : d.x[3];
        const int f = d.l % g.S[mu] + d.l / (g.S[mu] * g.a[mu]) * g.S[mu];
        // a domain one site wide sees both faces from every site
        for (int side = 0; side < (g.a[mu] == 1 ? 2 : 1); ++side) {
          const bool fwd = g.a[mu] == 1 ? side == 0 : xm == g.a[mu] - 1;
          if (fwd || xm == 0) {
            const int k = 2 * mu + (fwd ? 0 : 1);
            const float4* sx = slots + (k - k0) * g.slot;
            const int B = nbd[k];
            switch (mu) {
              case 0: hop_face<0>(d, o, sx, g.nf[0], f, fwd, UQ, B, g); break;
              case 1: hop_face<1>(d, o, sx, g.nf[1], f, fwd, UQ, B, g); break;
              case 2: hop_face<2>(d, o, sx, g.nf[2], f, fwd, UQ, B, g); break;
              default: hop_face<3>(d, o, sx, g.nf[3], f, fwd, UQ, B, g); break;
            }
          }
        }
      }
      __syncthreads();  // the slots are free
      k0 = k1, k1 = k2, in_f = !in_f;
    }
  }
  // rho = b - D x0 at the thread's site (o holds D x0 - b, or b itself)
  const float sgr = x0z ? 1.f : -1.f;
  if (valid) {
#pragma unroll
    for (int c = 0; c < 12; ++c)
      sR[c * Va + d.l] = make_float4(sgr * o[c].re.x, sgr * o[c].re.y, sgr * o[c].im.x, sgr * o[c].im.y);
  }
  __syncthreads();
  for (int step = 0; step < n_mr; ++step) {
    float2 pr = make_float2(0.f, 0.f), pi = pr, pq = pr;
    apply_dom<false>(d, o, g);  // o = q = D_B rho
    if (valid) {
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        const c2 r = ldH(d, c, d.l);
        pr = fma2(o[c].re, r.re, fma2(o[c].im, r.im, pr));
        pi = fma2(o[c].re, r.im, fma2(make_float2(-o[c].im.x, -o[c].im.y), r.re, pi));
        pq = fma2(o[c].re, o[c].re, fma2(o[c].im, o[c].im, pq));
      }
    }
    // sums over the sites of the warp, then over the warps
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      pr.x += __shfl_xor_sync(0xffffffffu, pr.x, s);
      pr.y += __shfl_xor_sync(0xffffffffu, pr.y, s);
      pi.x += __shfl_xor_sync(0xffffffffu, pi.x, s);
      pi.y += __shfl_xor_sync(0xffffffffu, pi.y, s);
      pq.x += __shfl_xor_sync(0xffffffffu, pq.x, s);
      pq.y += __shfl_xor_sync(0xffffffffu, pq.y, s);
    }
    if (lane == 0) sred[warp * 3] = pr, sred[warp * 3 + 1] = pi, sred[warp * 3 + 2] = pq;
    __syncthreads();
    // every warp adds the warps' sums (at most 8): lane w takes one, by a butterfly
    float2 a = make_float2(0.f, 0.f), bb = a, cc = a;
    if (lane < T / 32) a = sred[lane * 3], bb = sred[lane * 3 + 1], cc = sred[lane * 3 + 2];
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, s), a.y += __shfl_xor_sync(0xffffffffu, a.y, s);
      bb.x += __shfl_xor_sync(0xffffffffu, bb.x, s), bb.y += __shfl_xor_sync(0xffffffffu, bb.y, s);
      cc.x += __shfl_xor_sync(0xffffffffu, cc.x, s), cc.y += __shfl_xor_sync(0xffffffffu, cc.y, s);
    }
    const float2 alr = make_float2(cc.x > 0.f ? a.x / cc.x : 0.f, cc.y > 0.f ? a.y / cc.y : 0.f);
    const float2 ali = make_float2(cc.x > 0.f ? bb.x / cc.x : 0.f, cc.y > 0.f ? bb.y / cc.y : 0.f);
    const float2 nali = make_float2(-ali.x, -ali.y);
    // x_B += alpha rho (tensor memory), rho -= alpha q (shared memory; nothing
    // reads it after the last step), four components at a time
    const bool more = step + 1 < n_mr;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float f[16];
      tc::tmem_ld16(tm + 16 * k, f);
      if (valid) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = 4 * k + i;
          c2 xv = mk2(make_float2(f[4 * i], f[4 * i + 1]), make_float2(f[4 * i + 2], f[4 * i + 3]));
          c2 r = ldH(d, c, d.l);
          xv.re = fma2(alr, r.re, xv.re);
          xv.re = fma2(nali, r.im, xv.re);
          xv.im = fma2(alr, r.im, xv.im);
          xv.im = fma2(ali, r.re, xv.im);
          if (more) {
            // rho += alpha (-q)
            const c2 nq = mk2(make_float2(-o[c].re.x, -o[c].re.y), make_float2(-o[c].im.x, -o[c].im.y));
            r.re = fma2(alr, nq.re, r.re);
            r.re = fma2(nali, nq.im, r.re);
            r.im = fma2(alr, nq.im, r.im);
            r.im = fma2(ali, nq.re, r.im);
            sR[c * Va + d.l] = make_float4(r.re.x, r.re.y, r.im.x, r.im.y);
          }
          f[4 * i] = xv.re.x, f[4 * i + 1] = xv.re.y, f[4 * i + 2] = xv.im.x, f[4 * i + 3] = xv.im.y;
        }
      }
      tc::tmem_st16(tm + 16 * k, f);
    }
    tc::tmem_wait_st();
    __syncthreads();
  }
  // x = x_B for the thread's site and pair
  {
    float4* xs = xq + tile + d.l;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float f[16];
      tc::tmem_ld16(tm + 16 * k, f);
      if (valid) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          xs[(4 * k + i) * Va] = make_float4(f[4 * i], f[4 * i + 1], f[4 * i + 2], f[4 * i + 3]);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(s_tmem, tm_cols);
}

// the links with the sites of a domain innermost: float4 k of link mu at row 5 mu + k of
// [domain][20][Va]. Made anew by every call (a read and a write of 320 bytes a site, 42 MB
// each at 16^3 x 32) rather than held by the context beside U20. CTA (domain, kLinkSites
// of its sites), through shared memory (rows of 21 float4: reads of a column fall into
// different banks), so that both sides are runs of 1 KB and more.
constexpr int kLinkSites = 64;
__global__ void __launch_bounds__(256) k_links(const float4* __restrict__ U20, float4* __restrict__ UQ, int Va) {
  __shared__ float4 sm[kLinkSites * 21];
  const int l0 = blockIdx.y * kLinkSites, n = min(kLinkSites, Va - l0);
  const float4* src = U20 + ((size_t)blockIdx.x * Va + l0) * 20;
  float4* dst = UQ + (size_t)blockIdx.x * 20 * Va + l0;
  for (int i = threadIdx.x; i < 20 * n; i += 256) sm[i / 20 * 21 + i % 20] = __ldg(src + i);
  __syncthreads();
  for (int i = threadIdx.x; i < 20 * kLinkSites; i += 256) {
    const int l = i % kLinkSites, row = i / kLinkSites;
    if (l < n) dst[row * Va + l] = sm[l * 21 + row];
  }
}

// four consecutive right-hand sides of a row, FP32
__device__ __forceinline__ float4 ld_four(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <class S>
__device__ __forceinline__ float4 ld_four(const S* p) {
  const float2 a = ld_pair(p), b = ld_pair(p + 2);
  return make_float4(a.x, a.y, b.x, b.y);
}

// Right-hand sides r0 .. r0 + G - 1 of a field to the tiles of k_sap_face and back
// (FP32 field, OUT). CTA (A, c, block of ns sites): the block's two rows of
// component c go through shared memory ([part][site][G + 2] floats: the 8-byte
// accesses of 16 sites fall into different banks), so that the field is read or
// written by whole rows and the tiles by runs of ns sites.
template <class S, bool OUT>
__global__ void __launch_bounds__(256) k_tiles(S* __restrict__ f, float4* __restrict__ q, int N, int r0, int G, int Va,
                                               int ns) {
  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  const int A = blockIdx.x, c = blockIdx.y, l0 = blockIdx.z * ns, n = min(ns, Va - l0);
  const int ld = G + 2, Q = G / 4, nch = G / 2;
  S* fs = f + (((size_t)A * Va + l0) * 24 + 2 * c) * N + r0;
  auto fine = [&](auto move) {  // (site, part, four right-hand sides)
    for (int i = threadIdx.x; i < 2 * n * Q; i += 256) {
      const int k = i % Q, part = i / Q & 1, l = i / (2 * Q);
      move(fs + ((size_t)l * 24 + part) * N + 4 * k, reinterpret_cast<float2*>(sm + (part * ns + l) * ld + 4 * k));
    }
  };
  auto tile = [&](auto move) {  // (pair, site)
    for (int i = threadIdx.x; i < nch * n; i += 256) {
      const int l = i % n, ch = i / n;
      float2* re = reinterpret_cast<float2*>(sm + l * ld + 2 * ch);
      move(q + (((size_t)A * nch + ch) * 12 + c) * Va + l0 + l, re, re + ns * ld / 2);
    }
  };
  if constexpr (!OUT) {
    fine([](const S* g, float2* t) {
      const float4 v = ld_four(g);
      t[0] = make_float2(v.x, v.y), t[1] = make_float2(v.z, v.w);
    });
    __syncthreads();
    tile([](float4* g, const float2* re, const float2* im) { *g = make_float4(re->x, re->y, im->x, im->y); });
  } else {
    tile([](const float4* g, float2* re, float2* im) {
      const float4 v = *g;
      *re = make_float2(v.x, v.y), *im = make_float2(v.z, v.w);
    });
    __syncthreads();
    fine([](S* g, const float2* t) {
      *reinterpret_cast<float4*>(g) = make_float4(t[0].x, t[0].y, t[1].x, t[1].y);
    });
  }
}

}  // namespace

// the form of the kernel: MRHS_SAP_PK = "2g" (default: two pairs per CTA,
// links read through L1), "2s" (links staged in shared memory) or "1g" (one
// pair per CTA, two CTAs per SM). Measured at 48^3x96 with 32 right-hand
// sides: 83.2 ms per colour launch (2g), 88.8 (2s), 108.7 (1g): the links of
// a domain stay in L1 across the hops, and staging them cost more than it
// saved; two CTAs per SM each restage the clover term and re-read the links
// for half the right-hand sides.
struct PkForm {
  int pp;
  bool lg;
};
static PkForm pk_form() {
  static const PkForm f = [] {
    const char* e = std::getenv("MRHS_SAP_PK");
    const std::string v = e ? e : "";
    if (v == "1g") return PkForm{1, true};
    if (v == "2s") return PkForm{2, false};
    return PkForm{2, true};
  }();
  return f;
}

static int sap_pk_threads(int Va, int pp) { return 128 * ((pp * Va + 127) / 128); }

static size_t sap_pk_smem(int Va, int T, PkForm f) {
  return sizeof(float4) * ((f.lg ? 0 : 20 * (size_t)(Va + 1)) + 12 * (size_t)f.pp * Va) +
         sizeof(float2) * (T / 32) * f.pp * 3 + sizeof(int) * 8 * (size_t)Va;
}

bool sap_pk_ok(mrhs_ctx c, int nrhs) {
  const int Va = c->g.Va;
  const PkForm f = pk_form();
  if (Va > 256 || !c->U20 || nrhs % (2 * f.pp) != 0) return false;
  int maxsm = 0;
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  return sap_pk_smem(Va, sap_pk_threads(Va, f.pp), f) <= (size_t)maxsm;
}

// k_sap_face's slots for this context's domains; nF = 0: it does not fit
static SapGeo sap_face_geo(mrhs_ctx c, int T, size_t* smem) {
  SapGeo g;
  const int Va = c->g.Va;
  int S = 1;
  g.slot = 0;
  for (int m = 0; m < 4; ++m) {
    g.a[m] = c->g.a[m], g.S[m] = S, g.nf[m] = Va / c->g.a[m];
    S *= c->g.a[m];
    g.slot = std::max(g.slot, 12 * g.nf[m]);
  }
  // both sides of a direction come together, so slots come in pairs
  g.nR = 12 * Va / g.slot / 2 * 2;
  const size_t fixed = sizeof(float4) * 12 * (size_t)Va + sizeof(float2) * (T / 32) * 3 + sizeof(int) * 8;
  g.nF = 2;
  while (g.nF < 8 && sizeof(float4) * (g.nF + 2) * g.slot <= (size_t)25 * 1024) g.nF += 2;
  *smem = fixed + sizeof(float4) * g.nF * g.slot;
  int maxsm = 0;
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  if (*smem > (size_t)maxsm) g.nF = 0;
  return g;
}

// Right-hand sides smoothed together on tile copies: all of them when the workspace (the
// links and two copies) takes at most tile_limit bytes (20 GB; or 3/4 of what is free),
// else fewer, so that the largest lattices keep their memory for the setup, in multiples
// of 8: of a row's 128 bytes (32 right-hand sides) whole 64-byte pieces come from memory,
// so copies of four at a time cost as much as of eight (48^3 x 96, 32 vectors, a setup:
// 545 ms in fours, 236 ms in eights, 16 GB). A group is at most kTileGroup, so that
// k_tiles' rows of one site fit in shared memory. 0: not even four fit, the caller takes
// the form without copies.
constexpr int kTileGroup = 2048;
static int sap_group(mrhs_ctx c, int nrhs, size_t links) {
  const size_t four = 2 * sizeof(float) * fine_elems(c, 4);
  const size_t held = tiles_held(c);
  size_t room = c->tile_limit;
  if (held < std::min(room, links + four * (std::min(nrhs, kTileGroup) / 4))) {
    const Unrecorded u;
    size_t free_b = 0, total_b = 0;
    MRHS_CUDA(cudaMemGetInfo(&free_b, &total_b));
    room = std::max(held, std::min(room, (free_b + held) / 4 * 3));
  }
  if (room < links + four) return 0;
  const int group = std::min(kTileGroup, 4 * (int)std::min<size_t>(nrhs / 4, (room - links) / four));
  return group < nrhs && group > 8 ? group & ~7 : group;
}

// the smoother on tile copies; false: they or the kernel do not fit, or b does not
// start on the 16 bytes that the copies of FP32 fields take at a time
static bool sap_face(mrhs_ctx c, const void* b, int bdtype, void* x, int nrhs, int n_sweeps, int n_mr, bool x0_zero) {
  const int Va = c->g.Va, T = sap_pk_threads(Va, 1);
  if (c->work_dtype != MRHS_F32) return false;
  if (bdtype == MRHS_F32 && ((uintptr_t)b & 15) != 0) return false;
  size_t smem = 0;
  const SapGeo geo = sap_face_geo(c, T, &smem);
  const size_t links = sizeof(float) * 80 * c->g.V;
  const int group = geo.nF > 0 ? sap_group(c, nrhs, links) : 0;
  if (group == 0) return false;
  uint32_t cols = 32;
  while (cols < (uint32_t)(T / 128) * kPWarpCols) cols <<= 1;
  const size_t tiles = sizeof(float) * fine_elems(c, group);
  const TileSpace ws(c, links + 2 * tiles);
  if (!ws.p) return false;
  float4* uq = (float4*)ws.p;
  float4* xq = uq + links / sizeof(float4);
  float4* bq = xq + tiles / sizeof(float4);
  MRHS_CUDA(cudaFuncSetAttribute(k_sap_face, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  for (int g0 = 0; g0 < nrhs; g0 += group) {
    const int G = std::min(group, nrhs - g0), nch = G / 2;
    const int ns = std::max(1, std::min(Va, (int)(32 * 1024 / (8 * (G + 2)))));  // sites per block: 32 KB
    const size_t smem_t = sizeof(float) * 2 * ns * (G + 2);
    const dim3 grid(c->g.nagg, 12, (Va + ns - 1) / ns);
    {
      Prof pr(c, "sap_tiles");
      if (g0 == 0)
        k_links<<<dim3(c->g.nagg, (Va + kLinkSites - 1) / kLinkSites), 256, 0, c->stream>>>((const float4*)c->U20, uq, Va);
      MRHS_DISPATCH(bdtype, SB, (k_tiles<const SB, false><<<grid, 256, smem_t, c->stream>>>((const SB*)b, bq, nrhs, g0, G, Va, ns)));
      if (x0_zero) MRHS_CUDA(cudaMemsetAsync(xq, 0, sizeof(float) * fine_elems(c, G), c->stream));
      else k_tiles<const float, false><<<grid, 256, smem_t, c->stream>>>((const float*)x, xq, nrhs, g0, G, Va, ns);
      MRHS_LAUNCH_CHECK("tiles_in");
    }
    for (int sw = 0; sw < n_sweeps; ++sw)
      for (int col = 0; col < 2; ++col) {
        const int* blist = c->blocks_col + (col ? c->ncol[0] : 0);
        Prof pr(c, "sap_pk");
        k_sap_face<<<c->ncol[col] * nch, T, smem, c->stream>>>(bq, xq, uq, c->A32, c->aggnbr, nch, Va, blist, n_mr, cols,
                                                               x0_zero && sw == 0 && col == 0, geo);
        MRHS_LAUNCH_CHECK("sap_face");
      }
    Prof pr(c, "sap_tiles");
    k_tiles<float, true><<<grid, 256, smem_t, c->stream>>>((float*)x, xq, nrhs, g0, G, Va, ns);
    MRHS_LAUNCH_CHECK("tiles_out");
  }
  return true;
}

void sap_pk(mrhs_ctx c, const void* b, int bdtype, void* x, int nrhs, int n_sweeps, int n_mr, bool x0_zero) {
  const int Va = c->g.Va;
  const PkForm f = pk_form();
  const int T = sap_pk_threads(Va, f.pp);
  const size_t smem = sap_pk_smem(Va, T, f);
  const int kG = 2 * f.pp;
  // x_B and the clover copy: kPWarpCols columns per thread, (T / 128) warps
  // per lane quarter (at most 4 x 120 = 480 of the 512 columns)
  uint32_t cols = 32;
  while (cols < (uint32_t)(T / 128) * kPWarpCols) cols <<= 1;
  // CTAs per domain: by default one chunk each, so that a domain's CTAs run
  // side by side and share the 32-byte sectors of x and b in L2;
  // MRHS_SAP_CPB = c: c CTAs per domain, each looping over nrhs / (4 c) chunks
  // (the links and clover term staged once per CTA serve all its chunks)
  static const int cpb_env = [] {
    const char* e = std::getenv("MRHS_SAP_CPB");
    return e ? std::atoi(e) : 0;
  }();
  const int cpb = cpb_env > 0 ? std::min(cpb_env, nrhs / kG) : nrhs / kG;
  static const bool switched = std::getenv("MRHS_SAP_PK") || cpb_env > 0;
  MRHS_DISPATCH(bdtype, SB, {
    auto kern = f.pp == 1 ? k_sap_pk<SB, 1, true> : f.lg ? k_sap_pk<SB, 2, true> : k_sap_pk<SB, 2, false>;
    // (in front of both forms: it also loads the kernel, which a first launch inside a
    // capture must not have to do)
    MRHS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // The copies live as long as a call, and a recorded call may be replayed at any time,
    // also beside a direct one: while the stream is captured, the form that touches only
    // the caller's fields and the tables that live as long as the context.
    if (!switched && n_sweeps >= 2 && Va > 128 && !capturing(c) &&
        sap_face(c, b, bdtype, x, nrhs, n_sweeps, n_mr, x0_zero))
      return;
    for (int sw = 0; sw < n_sweeps; ++sw)
      for (int col = 0; col < 2; ++col) {
        const int* blist = c->blocks_col + (col ? c->ncol[0] : 0);
        Prof pr(c, "sap_pk");
        kern<<<c->ncol[col] * cpb, T, smem, c->stream>>>((const SB*)b, (float*)x, c->U20, c->A32, c->nbr, nrhs, Va,
                                                         blist, n_mr, cols, cpb, x0_zero && sw == 0 && col == 0);
        MRHS_LAUNCH_CHECK("sap_pk");
      }
  });
}

}  // namespace mrhs
