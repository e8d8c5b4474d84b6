// Semblance kernels: K1 (forward, three forms), its small-launch split form,
// K2 (adjoint gradient) and the stacked output, as templates over the
// operator, window, storage type and position form. Each operator's
// instantiations are compiled in a translation unit of their own
// (semblance_op_*.cu) and reached through pick_kernel / pick_stack.
//
// Work decomposition: (domain, individual) pairs are laid out domain-major;
// a warp owns 64 consecutive pairs, so with NP = 64 it covers one domain,
// and consecutive warps cover adjacent t0 at the same m0. Consecutive
// domains share a group (same m0, same aperture), so every lane of a warp
// walks the same aperture entries in the same order: the geometry-table load
// is a warp-uniform broadcast and the 2w+2 samples each lane reads from a
// trace row sit at nearby addresses for nearby t0 and for a converging
// population, which the L1 cache turns into reuse.
//
// Per aperture trace i (Sec. 2, the W_l x T_a inner loop of eq. order), in
// sample units (A' = A/dt, B' = B/dt^2, C' = C/dt^2, p0 = it0), the position
// u = t/dt of the window centre is found, then
//   j = floor(u), f = u - j, g = 1 - f,
//   a_k = g x[j+k] + f x[j+k+1],  s_k += a_k,  E += a_k^2
// and S = sum_k s_k^2 / (N E) (0 when E = 0).
//
// Two ways to find u, chosen by the record length at launch:
//  * direct (records up to 2048 samples, u <= 2048 + w):
//      q = p0 + A' dm,  U = q^2 + B' dm^2 + C' h^2,  u = sqrt(U)
//    whose FP32 rounding stays within ~1e-4 samples there;
//  * moveout (longer records): u = p0 + du with du the root of
//      du^2 + 2 p0 du - V = 0,  V = x (x + 2 p0) + B' dm^2 + C' h^2,  x = A' dm,
//    taken as du0 = U r - p0 (r ~ U^-1/2 from the hardware, one rounding)
//    refined by one Newton step du = du0 - (du0 (du0 + 2 p0) - V) r / 2.
//    p0 is an exact integer and du is tens of samples for deep events, so
//    the fraction keeps ~1e-5-sample accuracy where u itself (thousands of
//    samples) would round at ~1e-4 samples.
// U < 0 (no real traveltime) gives NaN, which the clamp maps to ns + w: a
// window of padding zeros. The scalar and the packed code run the same
// operations; no product is ever rounded and then added (a pattern a compiler
// may fuse), so they agree bit for bit.
#pragma once

#include <cooperative_groups.h>

#include "de_kernels.cuh"
#include "tt_internal.cuh"

namespace tt {
namespace sk {


// The two halves of a cluster barrier: work between them overlaps the other
// blocks' arrival. The relaxed arrival orders no memory (no fence to wait for).
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <typename T>
__device__ __forceinline__ float ld_sample(const T* p);
template <>
__device__ __forceinline__ float ld_sample<float>(const float* p) {
  return __ldg(p);
}
template <>
__device__ __forceinline__ float ld_sample<__nv_bfloat16>(const __nv_bfloat16* p) {
  unsigned short u = __ldg(reinterpret_cast<const unsigned short*>(p));
  return __uint_as_float(unsigned(u) << 16);
}

// Per-lane constants of one (domain, individual) pair.
struct Lane {
  int d, e0, e1, p0i;
  float p0, ca, cb, cc, inv_dt;
  float cah, cbh;      // FO-CRS: Ah / dt and Bmh / dt^2
  float two_p0, p0sq;  // 2 p0, p0^2 + 1e-30 (the bias keeps U = 0 finite under rsqrt)
  float lim, neg_p0;   // moveout: du is clamped to [-p0, ns + w - p0]
  float umax;          // direct: u is clamped to ns + w
};

// Domain of pair q = d P + p. A 64-bit division costs about a hundred
// instructions a lane, which the short-lived warps of the split kernels feel.
__device__ __forceinline__ int dom_of(long long q, int P) {
  if (P == 1) return int(q);
  if (q <= 0x7fffffffll) return int(unsigned(q) / unsigned(P));
  return int(q / P);
}

// L.d is the local domain (indexing theta and S); its geometry comes from the
// global domain dom_map[L.d] when a map is given (a subset evaluation).
// The operator's coefficients of parameter vector th in sample units.
template <int OP>
__device__ __forceinline__ void set_theta(Lane& L, const float* th) {
  const float i2 = L.inv_dt * L.inv_dt;
  L.cah = 0.f;
  L.cbh = 0.f;
  if (OP == TT_OP_CMP) {
    L.ca = 0.f;
    L.cb = 0.f;
    L.cc = th[0] * i2;
  } else if (OP == TT_OP_CRS) {
    L.ca = th[0] * L.inv_dt;
    L.cb = th[1] * i2;
    L.cc = th[2] * i2;
  } else {  // (Am, Ah, Bmm, Bmh, Bhh): ca, cah slopes, cb, cbh, cc curvatures
    L.ca = th[0] * L.inv_dt;
    L.cah = th[1] * L.inv_dt;
    L.cb = th[2] * i2;
    L.cbh = th[3] * i2;
    L.cc = th[4] * i2;
  }
}

template <int OP, bool DIV32 = false>
__device__ __forceinline__ bool lane_setup(const EvalArgs& a, long long q, Lane& L) {
  if (q >= (long long)a.n_dom * a.P) return false;
  L.d = DIV32 ? dom_of(q, a.P) : int(q / a.P);
  const int gd = a.dom_map ? a.dom_map[L.d] : L.d;
  if (gd < 0) return false;
  const int g = a.dom_group[gd];
  L.inv_dt = a.g_inv_dt[g];
  L.e0 = a.ap_ptr[g];
  L.e1 = a.ap_ptr[g + 1];
  L.p0i = a.dom_it0[gd];
  L.p0 = float(L.p0i);
  const float* th = a.theta + q * op_dim(OP);
  set_theta<OP>(L, th);
  L.two_p0 = 2.f * L.p0;
  L.p0sq = __fmul_rn(L.p0, L.p0) + 1e-30f;
  L.lim = a.umax - L.p0;
  L.neg_p0 = -L.p0;
  L.umax = a.umax;
  return true;
}

// FO-CRS quadratic part in samples^2: dm (Bmm dm + Bmh dh) + (Bhh dh) dh,
// from the table entry (dm, dh, -, row)
__device__ __forceinline__ float fo_quad(const Lane& L, float4 t4) {
  return fmaf(t4.x, fmaf(L.cb, t4.x, __fmul_rn(L.cbh, t4.y)),
              __fmul_rn(__fmul_rn(L.cc, t4.y), t4.y));
}

// Position of one pair on one trace. Every operation is rounded once, in the
// same order as one lane of the packed path, so both give identical bits.
struct Pos {
  int j;       // window sample k sits at j - W + k
  float f, g;  // interpolation weights
  float u;     // clamped position (samples)
  float q;     // p0 + A' dm (for the gradient)
};

// FLOOR_FP32: the direct form's floor of 0 <= u < 2^23 by adding 2^23 rounded
// toward zero -- FP32-pipe work with the same result, for kernels that do
// little else per position; truncf and the conversion take the slow unit twice.
template <int OP, bool MOVEOUT, bool FLOOR_FP32 = false>
__device__ __forceinline__ Pos locate(const Lane& L, float4 t4) {
  Pos P;
  if (!MOVEOUT) {
    float U;
    if (OP == TT_OP_CMP) {
      P.q = L.p0;
      U = fmaf(L.cc, t4.z, __fmul_rn(L.p0, L.p0));
    } else if (OP == TT_OP_CRS) {
      P.q = fmaf(L.ca, t4.x, L.p0);
      U = fmaf(L.cb, t4.y, fmaf(L.cc, t4.z, __fmul_rn(P.q, P.q)));
    } else {
      P.q = fmaf(L.ca, t4.x, fmaf(L.cah, t4.y, L.p0));
      U = fmaf(P.q, P.q, fo_quad(L, t4));
    }
    P.u = fminf(sqrt_approx(U), L.umax);
    if (FLOOR_FP32) {
      const float big = __fadd_rz(P.u, 8388608.f);
      const float fl = __fsub_rn(big, 8388608.f);
      P.f = __fsub_rn(P.u, fl);
      P.j = int(__float_as_uint(big) - 0x4b000000u);
    } else {
      const float fl = truncf(P.u);
      P.f = __fsub_rn(P.u, fl);
      P.j = int(fl);
    }
    P.g = __fsub_rn(1.f, P.f);
    return P;
  }
  float V, x;
  if (OP == TT_OP_CMP) {
    x = 0.f;
    V = __fmul_rn(L.cc, t4.z);
  } else if (OP == TT_OP_CRS) {
    x = __fmul_rn(L.ca, t4.x);
    const float w = fmaf(L.cb, t4.y, __fmul_rn(L.cc, t4.z));
    V = fmaf(x, __fadd_rn(x, L.two_p0), w);
  } else {
    x = fmaf(L.ca, t4.x, __fmul_rn(L.cah, t4.y));
    V = fmaf(x, __fadd_rn(x, L.two_p0), fo_quad(L, t4));
  }
  const float U = __fadd_rn(L.p0sq, V);
  const float r = rsqrt_approx(U);
  const float du0 = fmaf(U, r, L.neg_p0);
  const float res = fmaf(du0, __fadd_rn(du0, L.two_p0), __fmul_rn(V, -1.f));
  float du = fmaf(res, __fmul_rn(r, -0.5f), du0);
  du = fmaxf(fminf(du, L.lim), L.neg_p0);
  const float fl = floorf(du);
  P.f = fmaf(fl, -1.f, du);
  P.g = fmaf(P.f, -1.f, 1.f);
  P.j = L.p0i + int(fl);
  P.u = L.p0 + du;
  P.q = L.p0 + x;
  return P;
}

// Final normalisation S = Q / (N E). FP32-stored traces: E is one FP32
// sum over the aperture. BF16-stored traces (long apertures, reduced-
// precision data): E is accumulated in FP32 within chunks of 32 aperture
// traces and the chunk sums are added in FP64, so the energy's rounding
// error stays that of a 32-trace FP32 sum; the division is done in FP64.
template <typename T>
struct Chunk {
  static constexpr bool kF64 = false;
  static constexpr int kTraces = 1 << 30;  // one chunk: the whole aperture
};
template <>
struct Chunk<__nv_bfloat16> {
  static constexpr bool kF64 = true;
  static constexpr int kTraces = 32;
};

template <typename T>
__device__ __forceinline__ float normalise(float Q, int N, float E, double Ed) {
  if (Chunk<T>::kF64) return (Ed > 0.0) ? float(double(Q) / (double(N) * Ed)) : 0.f;
  return (E > 0.f) ? Q / (float(N) * E) : 0.f;
}

__device__ __forceinline__ void store_S(const EvalArgs& a, long long q, int d, float S) {
  if (a.slots) {
    const int slot = a.slots[q];
    if (slot >= 0) a.S[(size_t)d * a.np_out + slot] = S;
  } else {
    a.S[q] = S;
  }
}

// Accumulate one pair over aperture entries [r0, r1): the stack sums s_k and
// the energy -- one FP32 sum over the range (FP32 storage), or the FP64 sum
// of FP32 sums over 32-entry chunks from r0 (BF16 storage).
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void acc_scalar(const EvalArgs& a, const Lane& L, int r0, int r1,
                                           float* s, float& E, double& Ed) {
  constexpr int K = 2 * W + 1;
  const T* __restrict__ tr = static_cast<const T*>(a.traces);
  for (int c0 = r0, c1; c0 < r1; c0 = c1) {
    c1 = (r1 - c0 > Chunk<T>::kTraces) ? c0 + Chunk<T>::kTraces : r1;
    float Ec = 0.f;
    for (int e = c0; e < c1; ++e) {
      const float4 t4 = __ldg(a.ap_tab + e);
      const Pos P = locate<OP, MV>(L, t4);
      const T* x = tr + (__float_as_uint(t4.w) + P.j - W);
      float xv[K + 1];
#pragma unroll
      for (int k = 0; k <= K; ++k) xv[k] = ld_sample<T>(x + k);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float ak = fmaf(P.f, xv[k + 1], __fmul_rn(P.g, xv[k]));
        s[k] = __fadd_rn(s[k], ak);
        Ec = fmaf(ak, ak, Ec);
      }
    }
    if (Chunk<T>::kF64) Ed += double(Ec); else E = Ec;
  }
}

// The same for two pairs sharing an aperture, with packed FP32x2 arithmetic:
// sample k of the two pairs forms one register pair, so every interpolation,
// stack and energy update is one f32x2 instruction for both (same operations
// and bits as two acc_scalar calls).
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void acc_packed(const EvalArgs& a, const Lane& L0, const Lane& L1,
                                           int r0, int r1, float2* s, float2& E, double& Ed0,
                                           double& Ed1) {
  constexpr int K = 2 * W + 1;
  const T* __restrict__ tr = static_cast<const T*>(a.traces);
  const float2 ca = make_float2(L0.ca, L1.ca), cb = make_float2(L0.cb, L1.cb),
               cc = make_float2(L0.cc, L1.cc), two_p0 = make_float2(L0.two_p0, L1.two_p0),
               p0sq = make_float2(L0.p0sq, L1.p0sq), neg_p0 = make_float2(L0.neg_p0, L1.neg_p0),
               p0v = make_float2(L0.p0, L1.p0);
  const float2 cah = make_float2(L0.cah, L1.cah), cbh = make_float2(L0.cbh, L1.cbh);
  const float2 p0p0 = __fmul2_rn(p0v, p0v);
  // FO-CRS quadratic part, the packed twin of fo_quad
  auto fo_quad2 = [&](float2 dm, float2 dh) {
    return __ffma2_rn(dm, __ffma2_rn(cb, dm, __fmul2_rn(cbh, dh)),
                      __fmul2_rn(__fmul2_rn(cc, dh), dh));
  };
  const float2 m1 = make_float2(-1.f, -1.f), one = make_float2(1.f, 1.f),
               mhalf = make_float2(-0.5f, -0.5f);
  for (int c0 = r0, c1; c0 < r1; c0 = c1) {
    c1 = (r1 - c0 > Chunk<T>::kTraces) ? c0 + Chunk<T>::kTraces : r1;
    float2 Ec = make_float2(0.f, 0.f);
    for (int e = c0; e < c1; ++e) {
      const float4 t4 = __ldg(a.ap_tab + e);
      float2 f, g;
      int j0, j1;
      if constexpr (!MV) {
        float2 U;
        if (OP == TT_OP_CMP) {
          U = __ffma2_rn(cc, make_float2(t4.z, t4.z), p0p0);
        } else if (OP == TT_OP_CRS) {
          const float2 qv = __ffma2_rn(ca, make_float2(t4.x, t4.x), p0v);
          U = __ffma2_rn(cc, make_float2(t4.z, t4.z), __fmul2_rn(qv, qv));
          U = __ffma2_rn(cb, make_float2(t4.y, t4.y), U);
        } else {
          const float2 dm = make_float2(t4.x, t4.x), dh = make_float2(t4.y, t4.y);
          const float2 qv = __ffma2_rn(ca, dm, __ffma2_rn(cah, dh, p0v));
          U = __ffma2_rn(qv, qv, fo_quad2(dm, dh));
        }
        const float u0 = fminf(sqrt_approx(U.x), L0.umax), u1 = fminf(sqrt_approx(U.y), L1.umax);
        const float fl0 = truncf(u0), fl1 = truncf(u1);
        f = make_float2(__fsub_rn(u0, fl0), __fsub_rn(u1, fl1));
        g = make_float2(__fsub_rn(1.f, f.x), __fsub_rn(1.f, f.y));
        j0 = int(fl0);
        j1 = int(fl1);
      } else {
        float2 V;
        if (OP == TT_OP_CMP) {
          V = __fmul2_rn(cc, make_float2(t4.z, t4.z));
        } else if (OP == TT_OP_CRS) {
          const float2 x = __fmul2_rn(ca, make_float2(t4.x, t4.x));
          const float2 w = __ffma2_rn(cb, make_float2(t4.y, t4.y),
                                      __fmul2_rn(cc, make_float2(t4.z, t4.z)));
          V = __ffma2_rn(x, __fadd2_rn(x, two_p0), w);
        } else {
          const float2 dm = make_float2(t4.x, t4.x), dh = make_float2(t4.y, t4.y);
          const float2 x = __ffma2_rn(ca, dm, __fmul2_rn(cah, dh));
          V = __ffma2_rn(x, __fadd2_rn(x, two_p0), fo_quad2(dm, dh));
        }
        const float2 U = __fadd2_rn(p0sq, V);
        const float2 r = make_float2(rsqrt_approx(U.x), rsqrt_approx(U.y));
        const float2 du0 = __ffma2_rn(U, r, neg_p0);
        const float2 res = __ffma2_rn(du0, __fadd2_rn(du0, two_p0), __fmul2_rn(V, m1));
        float2 du = __ffma2_rn(res, __fmul2_rn(r, mhalf), du0);
        du.x = fmaxf(fminf(du.x, L0.lim), L0.neg_p0);
        du.y = fmaxf(fminf(du.y, L1.lim), L1.neg_p0);
        const float2 fl = make_float2(floorf(du.x), floorf(du.y));
        f = __ffma2_rn(fl, m1, du);
        g = __ffma2_rn(f, m1, one);
        j0 = L0.p0i + int(fl.x);
        j1 = L1.p0i + int(fl.y);
      }
      const unsigned base = __float_as_uint(t4.w) - W;
      const T* x0 = tr + (base + j0);
      const T* x1 = tr + (base + j1);
      float2 xv[K + 1];
#pragma unroll
      for (int k = 0; k <= K; ++k) xv[k] = make_float2(ld_sample<T>(x0 + k), ld_sample<T>(x1 + k));
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float2 ak = __ffma2_rn(f, xv[k + 1], __fmul2_rn(g, xv[k]));
        s[k] = __fadd2_rn(s[k], ak);
        Ec = __ffma2_rn(ak, ak, Ec);
      }
    }
    if (Chunk<T>::kF64) {
      Ed0 += double(Ec.x);
      Ed1 += double(Ec.y);
    } else {
      E = Ec;
    }
  }
}

// Scalar evaluation of one (domain, individual) pair over its aperture.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ float eval_scalar(const EvalArgs& a, const Lane& L) {
  constexpr int K = 2 * W + 1;
  float s[K];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k] = 0.f;
  float E = 0.f;
  double Ed = 0.0;
  acc_scalar<OP, W, T, MV>(a, L, L.e0, L.e1, s, E, Ed);
  float Q = 0.f;
#pragma unroll
  for (int k = 0; k < K; ++k) Q = fmaf(s[k], s[k], Q);
  return normalise<T>(Q, L.e1 - L.e0, E, Ed);
}

__device__ __forceinline__ bool same_aperture(const Lane& L0, const Lane& L1) {
  return L1.e0 == L0.e0 && L1.e1 == L0.e1 && L1.inv_dt == L0.inv_dt;
}

// One 64-pair unit: each thread evaluates pairs q and q + 32 (either may be
// absent: past the end, or a domain the map skips). When both lie in one
// group (the common case: same aperture, possibly different t0) the
// aperture is walked once with packed arithmetic; otherwise each pair is
// evaluated on its own (same operations, same bits).
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void eval_unit(const EvalArgs& a, long long unit, int lane) {
  constexpr int K = 2 * W + 1;
  const long long q0 = unit * 64 + lane, q1 = q0 + 32;
  Lane L0, L1;
  const bool v0 = lane_setup<OP>(a, q0, L0);
  const bool v1 = lane_setup<OP>(a, q1, L1);
  if (!v0 || !v1 || !same_aperture(L0, L1)) {
    if (v0) store_S(a, q0, L0.d, eval_scalar<OP, W, T, MV>(a, L0));
    if (v1) store_S(a, q1, L1.d, eval_scalar<OP, W, T, MV>(a, L1));
    return;
  }
  float2 s[K];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k] = make_float2(0.f, 0.f);
  float2 E = make_float2(0.f, 0.f);
  double Ed0 = 0.0, Ed1 = 0.0;
  acc_packed<OP, W, T, MV>(a, L0, L1, L0.e0, L0.e1, s, E, Ed0, Ed1);
  float2 Q = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < K; ++k) Q = __ffma2_rn(s[k], s[k], Q);
  const int N = L0.e1 - L0.e0;
  store_S(a, q0, L0.d, normalise<T>(Q.x, N, E.x, Ed0));
  store_S(a, q1, L1.d, normalise<T>(Q.y, N, E.y, Ed1));
}

// K1 for small launches (few 64-pair units): the aperture of a unit's pairs is
// cut into 8 B contiguous slices, whose partial sums are added eight at a time
// in slice order and the B sums of eight in order. B is 9 up to half a unit
// per SM, 7 up to 2 units per SM, 2 below 12 per SM and 1 above (76, 304 and
// 1824 units on a 152-SM device). The summation order depends on B and differs
// from the one-warp-per-unit kernel, so B is chosen by launch size alone --
// every variant of a launch gives the same bits -- and results stay
// reproducible. Three kernels run it, with the same bits:
//  * k_semblance_split: a warp per slice, eight warps per block, a cluster of
//    B blocks per unit (for long apertures, at some sizes, B single blocks whose
//    sums meet in global scratch: scratch_wins). A cluster's blocks push their
//    sums into the first one's shared memory and leave; no fence, ticket or
//    re-read. Latency bound (44% issue, 43% of the warps resident): a CRS launch of 118 units x
//    1008 traces, w = 5, takes 30.9 us against 37.5 us through global scratch,
//    258 units 63.0 us against 70.9 us, 24 units of 48 traces 9.7 against 12.5.
//  * k_semblance_short: a warp per eight slices, walked one after the other,
//    for apertures too short to feed 8 B warps (258 units x 48 traces: 10.4 us
//    against 18.5 us with a warp per slice and 29.1 us through scratch).
//  * k_search_short: the same walk inside a whole search.
constexpr int kSplitWarps = 8;

// Slice sl of nsl of a pair's aperture: entries floor(n sl / nsl) to
// floor(n (sl + 1) / nsl), from n = h nsl + m in 32 bits (m sl < nsl^2).
__device__ __forceinline__ void slice_of(const Lane& L, int nsl, int sl, int& r0, int& r1) {
  const unsigned n = unsigned(L.e1 - L.e0), u = unsigned(nsl), h = n / u, m = n - h * u;
  r0 = L.e0 + int(h * sl + m * sl / u);
  r1 = L.e0 + int(h * (sl + 1) + m * (sl + 1) / u);
}

// What the end of a split launch needs of its unit's pairs: the aperture size
// (-1 for an absent pair), kept in shared memory by one warp.
__device__ __forceinline__ void keep_sizes(int* size, int lane, bool v0, const Lane& L0, bool v1,
                                           const Lane& L1) {
  size[lane] = v0 ? L0.e1 - L0.e0 : -1;
  size[lane + 32] = v1 ? L1.e1 - L1.e0 : -1;
}

// shared rows of 64 floats per set of sums: s_k and E; BF16 storage adds a row
// of 64 doubles per set
template <typename T>
constexpr size_t split_set_bytes(int W) {
  return 64 * (sizeof(float) * (2 * W + 2) + (Chunk<T>::kF64 ? sizeof(double) : 0));
}
// k_semblance_split: the block's eight slices, and (used by the cluster's
// first block) the B blocks' sums it receives -- unless those would leave room
// for three blocks on an SM instead of four (windows of 15 samples and more,
// BF16 storage from 13): the first block then reads them where they are, and
// the others wait for it (w = 8, 258 units x 1008 traces: 93 us, against 105 us
// at three blocks an SM and 99 us through global scratch).
template <typename T>
constexpr bool split_pulls(int W) {
  return split_set_bytes<T>(W) * size_t(kSplitWarps + kSplitSmallBlocks) > 55 * 1024;
}
template <typename T>
constexpr size_t split_smem_bytes_of(int B, int W) {
  return split_set_bytes<T>(W) * size_t(kSplitWarps + (B > 1 && !split_pulls<T>(W) ? B : 0));
}
static_assert(split_smem_bytes_of<__nv_bfloat16>(1, TT_MAX_HALF_WINDOW) + 512 <= 48 * 1024,
              "a block's own sets fit without an opt-in");
inline size_t split_smem_bytes(int B, int W, bool bf16) {
  return bf16 ? split_smem_bytes_of<__nv_bfloat16>(B, W) : split_smem_bytes_of<float>(B, W);
}
// k_semblance_short and k_search_short: the unit's B sums
inline size_t short_smem_bytes(int B, int W, bool bf16) {
  const size_t set = bf16 ? split_set_bytes<__nv_bfloat16>(W) : split_set_bytes<float>(W);
  return set * size_t(B);
}

// S of pair q (row entry p) from its summed rows; N = -1 marks an absent pair.
// The rows themselves are kept where a gradient is to follow (a.sums).
template <int W, typename T>
__device__ __forceinline__ void finish_pair(const EvalArgs& a, long long q, int N,
                                            const float* tot, double Ed) {
  constexpr int K = 2 * W + 1;
  if (N < 0) return;
  if (a.sums) {
    float* out = a.sums + (q >> 6) * ((K + 1) * 64) + (q & 63);
#pragma unroll
    for (int k = 0; k <= K; ++k) out[k * 64] = tot[k * 64];
    if (Chunk<T>::kF64) a.sums_Ed[q] = Ed;
  }
  float Q = 0.f;
#pragma unroll
  for (int k = 0; k < K; ++k) Q = fmaf(tot[k * 64], tot[k * 64], Q);
  store_S(a, q, a.slots ? dom_of(q, a.P) : 0, normalise<T>(Q, N, tot[K * 64], Ed));
}

// GLOBAL: no clusters; the blocks' sums meet in the launch's scratch, where the
// unit's last block to arrive adds them (launch_split says when).
template <int OP, int W, typename T, bool MV, bool GLOBAL>
__global__ void __launch_bounds__(32 * kSplitWarps, 4) k_semblance_split(const EvalArgs a) {
  constexpr int K = 2 * W + 1, R = K + 1;
  constexpr int S = kSplitWarps, NT = 32 * S;
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char split_smem[];
  constexpr bool PULL = split_pulls<T>(W);
  const int B = a.split_blocks;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long unit = blockIdx.x / B;
  const int rank = int(blockIdx.x - unit * B);
  double* part_Ed = reinterpret_cast<double*>(split_smem);  // [S][64], then [B][64]
  double* recv_Ed = part_Ed + S * 64;
  const int sets = S + (B > 1 && !PULL && !GLOBAL ? B : 0);
  float* part = reinterpret_cast<float*>(part_Ed + (Chunk<T>::kF64 ? sets * 64 : 0));
  float* recv = part + S * R * 64;  // [B][R][64], in the cluster's first block
  // met by cluster_wait below: every block has started
  if (B > 1 && !PULL && !GLOBAL) cluster_arrive_relaxed();
  const long long q0 = unit * 64 + lane, q1 = q0 + 32;
  Lane L0, L1;
  const bool v0 = lane_setup<OP, true>(a, q0, L0);
  const bool v1 = lane_setup<OP, true>(a, q1, L1);
  __shared__ int size[64];
  if (w == 0) keep_sizes(size, lane, v0, L0, v1, L1);
  const int nsl = S * B, sl = rank * S + w;
  int r0, r1;
  if (v0 && v1 && same_aperture(L0, L1)) {
    slice_of(L0, nsl, sl, r0, r1);
    float2 s[K];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = make_float2(0.f, 0.f);
    float2 E = make_float2(0.f, 0.f);
    double Ed0 = 0.0, Ed1 = 0.0;
    acc_packed<OP, W, T, MV>(a, L0, L1, r0, r1, s, E, Ed0, Ed1);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      part[(w * R + k) * 64 + lane] = s[k].x;
      part[(w * R + k) * 64 + lane + 32] = s[k].y;
    }
    part[(w * R + K) * 64 + lane] = E.x;
    part[(w * R + K) * 64 + lane + 32] = E.y;
    if (Chunk<T>::kF64) {
      part_Ed[w * 64 + lane] = Ed0;
      part_Ed[w * 64 + lane + 32] = Ed1;
    }
  } else {
    for (int h = 0; h < 2; ++h) {
      float s[K], E = 0.f;
      double Ed = 0.0;
#pragma unroll
      for (int k = 0; k < K; ++k) s[k] = 0.f;
      if (h ? v1 : v0) {
        const Lane& L = h ? L1 : L0;
        slice_of(L, nsl, sl, r0, r1);
        acc_scalar<OP, W, T, MV>(a, L, r0, r1, s, E, Ed);
      }
      const int p = lane + 32 * h;
#pragma unroll
      for (int k = 0; k < K; ++k) part[(w * R + k) * 64 + p] = s[k];
      part[(w * R + K) * 64 + p] = E;
      if (Chunk<T>::kF64) part_Ed[w * 64 + p] = Ed;
    }
  }
  __syncthreads();
  // the block's sums, slices in order: to the cluster's first block, or the scratch
  float* to = part;
  double* to_d = part_Ed;
  if constexpr (GLOBAL) {
    to = a.part + blockIdx.x * size_t(R * 64);
    to_d = a.part_Ed + blockIdx.x * size_t(64);
  } else if (B > 1 && !PULL) {
    cluster_wait();
    to = cl.map_shared_rank(recv, 0) + rank * R * 64;
    to_d = cl.map_shared_rank(recv_Ed, 0) + rank * 64;
  }
  for (int i = threadIdx.x; i < R * 64; i += NT) {
    float t = 0.f;
#pragma unroll
    for (int v = 0; v < S; ++v) t = __fadd_rn(t, part[v * R * 64 + i]);
    to[i] = t;
  }
  if (Chunk<T>::kF64 && threadIdx.x < 64) {
    double t = 0.0;
    for (int v = 0; v < S; ++v) t += part_Ed[v * 64 + threadIdx.x];
    to_d[threadIdx.x] = t;
  }
  double Ed = 0.0;
  if constexpr (GLOBAL) {  // no block waits
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(a.ticket + unit, 1u) == unsigned(B - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) a.ticket[unit] = 0u;  // ready for the next launch
    const size_t set0 = size_t(unit) * B;
    for (int i = threadIdx.x; i < R * 64; i += NT) {
      float t = 0.f;
      for (int b = 0; b < B; ++b) t = __fadd_rn(t, __ldcg(a.part + (set0 + b) * (R * 64) + i));
      part[i] = t;
    }
    if (Chunk<T>::kF64 && threadIdx.x < 64)
      for (int b = 0; b < B; ++b) Ed += __ldcg(a.part_Ed + (set0 + b) * 64 + threadIdx.x);
  } else if (B > 1 && !PULL) {
    __syncwarp();
    cluster_arrive();
    if (rank) return;  // done with: nothing of this block's shared memory is read by others
    cluster_wait();
    for (int i = threadIdx.x; i < R * 64; i += NT) {
      float t = 0.f;
      for (int b = 0; b < B; ++b) t = __fadd_rn(t, recv[b * R * 64 + i]);
      part[i] = t;
    }
    if (Chunk<T>::kF64 && threadIdx.x < 64)
      for (int b = 0; b < B; ++b) Ed += recv_Ed[b * 64 + threadIdx.x];
  } else if (B > 1) {
    cl.sync();
    if (rank == 0) {
      for (int i = threadIdx.x; i < R * 64; i += NT) {
        float t = 0.f;
        for (int b = 0; b < B; ++b) t = __fadd_rn(t, cl.map_shared_rank(part, b)[i]);
        part[i] = t;
      }
      if (Chunk<T>::kF64 && threadIdx.x < 64)
        for (int b = 0; b < B; ++b) Ed += cl.map_shared_rank(part_Ed, b)[threadIdx.x];
    }
    cl.sync();  // no block leaves while its sums are read
    if (rank) return;
  }
  __syncthreads();
  if (threadIdx.x < 64) {
    if (Chunk<T>::kF64 && !GLOBAL && B == 1) Ed = part_Ed[threadIdx.x];
    finish_pair<W, T>(a, unit * 64 + threadIdx.x, size[threadIdx.x], part + threadIdx.x, Ed);
  }
}

// kSplitWarps consecutive slices of a pair's aperture, from slice sl0 of nsl:
// entries e0 to e1, the first slice's end, and what the next ends take --
// slice ends lie h or h + 1 entries apart, n = h nsl + m, as the remainder
// `rem` of m times the slice number passes nsl. Set up once (the divisions
// are as long as an entry's loads), walked without dividing.
struct Slices {
  int e0, e1, end, h, m, rem, nsl;
  __device__ __forceinline__ void set(const Lane& L, int nsl_, int sl0) {
    int r;
    nsl = nsl_;
    slice_of(L, nsl, sl0, e0, end);
    slice_of(L, nsl, sl0 + kSplitWarps - 1, r, e1);
    const int n = L.e1 - L.e0;
    h = n / nsl;
    m = n - h * nsl;
    rem = m * (sl0 + 1) % nsl;
  }
  __device__ __forceinline__ void next() {
    end += h;
    rem += m;
    if (rem >= nsl) {
      rem -= nsl;
      ++end;
    }
  }
};

// Sums of kSplitWarps consecutive slices of two pairs sharing an aperture, as
// acc_packed gives each and added in slice order. Apertures of no more traces
// than slices have at most one entry in a slice, whose amplitudes are the
// slice's sums: they are added directly.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void acc_slices(const EvalArgs& a, const Lane& L0, const Lane& L1,
                                           Slices at, float2* t, float2& tE, double& tEd0,
                                           double& tEd1) {
  constexpr int K = 2 * W + 1;
  if (at.h == 0) {
    const T* __restrict__ tr = static_cast<const T*>(a.traces);
    for (int e = at.e0; e < at.e1; ++e) {
      const float4 t4 = __ldg(a.ap_tab + e);
      const Pos P0 = locate<OP, MV, true>(L0, t4), P1 = locate<OP, MV, true>(L1, t4);
      const unsigned base = __float_as_uint(t4.w) - W;
      const T* x0 = tr + (base + P0.j);
      const T* x1 = tr + (base + P1.j);
      float2 xv[K + 1];
#pragma unroll
      for (int k = 0; k <= K; ++k) xv[k] = make_float2(ld_sample<T>(x0 + k), ld_sample<T>(x1 + k));
      const float2 f = make_float2(P0.f, P1.f), g = make_float2(P0.g, P1.g);
      float2 E = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float2 ak = __ffma2_rn(f, xv[k + 1], __fmul2_rn(g, xv[k]));
        t[k] = __fadd2_rn(t[k], ak);
        E = __ffma2_rn(ak, ak, E);
      }
      if (Chunk<T>::kF64) {
        tEd0 += double(E.x);
        tEd1 += double(E.y);
      } else {
        tE = __fadd2_rn(tE, E);
      }
    }
    return;
  }
  for (int v = 0, r0 = at.e0; v < kSplitWarps; ++v) {
    float2 s[K], E = make_float2(0.f, 0.f);
    double Ed0 = 0.0, Ed1 = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = make_float2(0.f, 0.f);
    acc_packed<OP, W, T, MV>(a, L0, L1, r0, at.end, s, E, Ed0, Ed1);
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = __fadd2_rn(t[k], s[k]);
    tE = __fadd2_rn(tE, E);
    tEd0 += Ed0;
    tEd1 += Ed1;
    r0 = at.end;
    at.next();
  }
}

// The same for one pair.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void acc_slices_scalar(const EvalArgs& a, const Lane& L, Slices at,
                                                  float* t, float& tE, double& tEd) {
  constexpr int K = 2 * W + 1;
  for (int v = 0, r0 = at.e0; v < kSplitWarps; ++v) {
    float s[K], E = 0.f;
    double Ed = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = 0.f;
    acc_scalar<OP, W, T, MV>(a, L, r0, at.end, s, E, Ed);
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = __fadd_rn(t[k], s[k]);
    tE = __fadd_rn(tE, E);
    tEd += Ed;
    r0 = at.end;
    at.next();
  }
}

// One of the unit's sums of eight slices, into row set `set` [K + 1][64] and
// energies set_Ed [64]. A0, A1: the slices of the lane's pairs.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void unit_slices(const EvalArgs& a, bool v0, const Lane& L0,
                                            const Slices& A0, bool v1, const Lane& L1,
                                            const Slices& A1, int lane, float* set,
                                            double* set_Ed) {
  constexpr int K = 2 * W + 1;
  if (v0 && v1 && same_aperture(L0, L1)) {
    float2 t[K], E = make_float2(0.f, 0.f);
    double Ed0 = 0.0, Ed1 = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = make_float2(0.f, 0.f);
    acc_slices<OP, W, T, MV>(a, L0, L1, A0, t, E, Ed0, Ed1);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      set[k * 64 + lane] = t[k].x;
      set[k * 64 + lane + 32] = t[k].y;
    }
    set[K * 64 + lane] = E.x;
    set[K * 64 + lane + 32] = E.y;
    if (Chunk<T>::kF64) {
      set_Ed[lane] = Ed0;
      set_Ed[lane + 32] = Ed1;
    }
    return;
  }
  for (int h = 0; h < 2; ++h) {
    float t[K], E = 0.f;
    double Ed = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = 0.f;
    if (h ? v1 : v0)
      acc_slices_scalar<OP, W, T, MV>(a, h ? L1 : L0, h ? A1 : A0, t, E, Ed);
    const int p = lane + 32 * h;
#pragma unroll
    for (int k = 0; k < K; ++k) set[k * 64 + p] = t[k];
    set[K * 64 + p] = E;
    if (Chunk<T>::kF64) set_Ed[p] = Ed;
  }
}

// The B sets of a unit added in order, into the first, by its 32 B threads.
template <int W, int B>
__device__ __forceinline__ void add_sets(float* set, int tid) {
  constexpr int R = 2 * W + 2;
#pragma unroll
  for (int i0 = 0; i0 < R * 64; i0 += 32 * B) {
    const int i = i0 + tid;
    if (i >= R * 64) break;
    float t = 0.f;
#pragma unroll
    for (int c = 0; c < B; ++c) t = __fadd_rn(t, set[c * R * 64 + i]);
    set[i] = t;
  }
}

template <int OP, int W, typename T, bool MV>
__global__ void __launch_bounds__(32 * kSplitSmallBlocks, 2) k_semblance_short(const EvalArgs a) {
  constexpr int B = kSplitSmallBlocks;
  extern __shared__ __align__(16) unsigned char split_smem[];
  __shared__ int size[64];
  const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
  const long long unit = blockIdx.x;
  double* set_Ed = reinterpret_cast<double*>(split_smem);  // [B][64]
  float* set = reinterpret_cast<float*>(set_Ed + (Chunk<T>::kF64 ? B * 64 : 0));
  Lane L0, L1;
  const bool v0 = lane_setup<OP, true>(a, unit * 64 + lane, L0);
  const bool v1 = lane_setup<OP, true>(a, unit * 64 + lane + 32, L1);
  if (b == 0) keep_sizes(size, lane, v0, L0, v1, L1);
  Slices A0{}, A1{};
  if (v0) A0.set(L0, kSplitWarps * B, kSplitWarps * b);
  if (v1) A1.set(L1, kSplitWarps * B, kSplitWarps * b);
  unit_slices<OP, W, T, MV>(a, v0, L0, A0, v1, L1, A1, lane, set + b * (2 * W + 2) * 64,
                            set_Ed + b * 64);
  __syncthreads();
  add_sets<W, B>(set, threadIdx.x);
  __syncthreads();
  const int p = threadIdx.x;
  if (p >= 64) return;
  double Ed = 0.0;
  if (Chunk<T>::kF64)
    for (int c = 0; c < B; ++c) Ed += set_Ed[c * 64 + p];
  finish_pair<W, T>(a, unit * 64 + p, size[p], set + p, Ed);
}

// The search of short apertures and few domains, generation after generation
// in one launch: nothing but the neighbour exchange couples domains, so a block
// of B warps takes the 64 / NP domains of a unit and runs evaluation and DE
// step in turn on populations that stay in shared memory. A generation of such
// a search is a few microseconds of dependent work; as two launches it costs
// as much again in launch latency, and each kernel reads what the one before
// wrote from L2. Each pair's semblance is that of the stepwise search bit for
// bit: the same 8 B slices of its aperture, B by the size of the stepwise
// launch; so are the DE steps (de_kernels.cuh). Bound by the latency of the
// seven warps' instructions (about 6,000 of a generation's 9,000 cycles are
// the evaluation). 128 registers, so that two blocks fit an SM: 500 CMP
// domains x 48 traces, DE 32 x 50: 239 us, against 526 us stepwise with
// k_semblance_short and 1,525 us before that.
template <int OP, int W, typename T, bool MV>
__global__ void __maxnreg__(128)
    k_search_short(const EvalArgs a, const DeArgs de, const FusedArgs fa) {
  constexpr int K = 2 * W + 1, R = K + 1;
  constexpr int D = op_dim(OP);
  extern __shared__ __align__(16) unsigned char split_smem[];
  __shared__ float pop[64 * D], trial[64 * D], fit[64], tfit[64];
  __shared__ int size[64];
  const int B = blockDim.x >> 5, nt = blockDim.x, NP = a.P;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* set_Ed = reinterpret_cast<double*>(split_smem);  // [B][64]
  float* set = reinterpret_cast<float*>(set_Ed + (Chunk<T>::kF64 ? B * 64 : 0));
  const int per = 64 / NP, dom0 = blockIdx.x * per;  // the block's domains
  const int nd = min(per, a.n_dom - dom0), n = nd * NP;  // and pairs
  // a lane without a second pair walks its first one twice
  const bool v0 = lane < n, v1 = lane + 32 < n;
  const int p1 = v1 ? lane + 32 : lane;
  Lane L0, L1;
  lane_setup<OP, true>(a, (long long)dom0 * NP + (v0 ? lane : 0), L0);
  lane_setup<OP, true>(a, (long long)dom0 * NP + (v0 ? p1 : 0), L1);
  if (w == 0) keep_sizes(size, lane, v0, L0, v1, L1);
  Slices A0, A1;
  A0.set(L0, kSplitWarps * B, kSplitWarps * w);
  A1.set(L1, kSplitWarps * B, kSplitWarps * w);
  auto evaluate = [&](const float* th, float* S) {
    if (v0) {
      set_theta<OP>(L0, th + lane * D);
      set_theta<OP>(L1, th + p1 * D);
    }
    unit_slices<OP, W, T, MV>(a, v0, L0, A0, v0, L1, A1, lane, set + w * R * 64, set_Ed + w * 64);
    __syncthreads();
    if (B == kSplitSmallBlocks)
      add_sets<W, kSplitSmallBlocks>(set, threadIdx.x);
    else
      add_sets<W, kSplitTinyBlocks>(set, threadIdx.x);
    __syncthreads();
    if (threadIdx.x < n) {
      const int p = threadIdx.x;
      double Ed = 0.0;
      if (Chunk<T>::kF64)
        for (int c = 0; c < B; ++c) Ed += set_Ed[c * 64 + p];
      float Q = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) Q = fmaf(set[k * 64 + p], set[k * 64 + p], Q);
      S[p] = normalise<T>(Q, size[p], set[K * 64 + p], Ed);
    }
    __syncthreads();
  };
  auto step = [&](int gen, int sel_gen, bool select, bool mutate) {
    for (int i = w; i < nd; i += B) {
      const int o = i * NP;
      de::DePop p;
      p.pop = p.spop = pop + o * D;
      p.fit = p.sfit = fit + o;
      p.trial = select ? trial + o * D : nullptr;
      p.tfit = tfit + o;
      p.next = mutate ? trial + o * D : nullptr;
      de::de_step<D>(de, dom0 + i, uint32_t(de.dom_base + dom0 + i), uint32_t(gen),
                     uint32_t(sel_gen), p, lane);
    }
    __syncthreads();
  };
  const size_t row = (size_t)dom0 * NP;
  if (fa.first == 0) {
    for (int i = w; i < nd; i += B)
      de::de_init<D>(de, dom0 + i, uint32_t(de.dom_base + dom0 + i), pop + i * NP * D, lane);
    __syncthreads();
    evaluate(pop, fit);
  } else {
    for (int i = threadIdx.x; i < n * D; i += nt) pop[i] = de.pop[row * D + i];
    for (int i = threadIdx.x; i < n; i += nt) fit[i] = de.fit[row + i];
    __syncthreads();
  }
  const int g0 = fa.first ? fa.first : 1;
  for (int g = g0; g <= fa.last; ++g) {
    step(g, g - 1, g > g0, true);
    evaluate(trial, tfit);
  }
  if (fa.last >= g0) step(fa.last + 1, fa.last, true, false);
  for (int i = threadIdx.x; i < n * D; i += nt) de.pop[row * D + i] = pop[i];
  for (int i = threadIdx.x; i < n; i += nt) de.fit[row + i] = fit[i];
}

// Blocks of kBlock threads that K1 asks the compiler to fit on an SM: 4 (64
// registers) for FO-CRS and for BF16 storage at windows up to 11 samples, where
// the compiler left to itself takes 72 and more (w = 5, 128-thread blocks:
// FO-CRS 18,000 domains x 64 2.09 -> 1.93 ms, moveout form 3.78 -> 3.60 ms, BF16
// moveout form 5.83 -> 5.53 ms); 0, no request, for the others (asking for 4
// costs the FP32 CRS direct form, at 64 registers either way, 1.4%).
template <int OP, int W, typename T>
constexpr int k1_blocks() {
  return W <= 5 && (OP == TT_OP_FOCRS || sizeof(T) == 2) ? 4 : 0;
}

// K1, grid-mapped (queue == nullptr: one 64-pair unit per warp, the grid
// covers every unit) or persistent (a grid sized to the GPU; after its first
// unit a warp takes the next one from an atomic counter, so warps whose
// apertures are short take more units).
template <int OP, int W, typename T, bool MV>
__global__ void __launch_bounds__(kBlock, k1_blocks<OP, W, T>()) k_semblance(const EvalArgs a) {
  const int lane = threadIdx.x & 31;
  const long long n_units = ((long long)a.n_dom * a.P + 63) / 64;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  long long unit = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  while (unit < n_units) {
    eval_unit<OP, W, T, MV>(a, unit, lane);
    if (!a.queue) break;
    __syncwarp();
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(a.queue, 1ull);
    unit = warps + (long long)__shfl_sync(0xffffffffu, next, 0);
  }
}

// K1, one (domain, individual) pair per thread.
template <int OP, int W, typename T, bool MV>
__global__ void __launch_bounds__(kBlock) k_semblance_scalar(const EvalArgs a) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  Lane L;
  if (!lane_setup<OP>(a, q, L)) return;
  store_S(a, q, L.d, eval_scalar<OP, W, T, MV>(a, L));
}

// K2: two passes over the aperture. Pass 1 = K1 (s_k, E, S). With
// alpha = 2/(N E), beta = 2 S / E, dS/da_ik = alpha s_k - beta a_ik, so pass 2
// forms dS/du_i = sum_k (alpha s_k - beta a_ik)(x[j+k+1] - x[j+k]) and
// chains it through du/dtheta (u = p0 + du in samples, q = p0 + A' dm):
//   du/dA = q dm / (u dt),  du/dB = dm^2 / (2 u dt^2),  du/dC = h^2 / (2 u dt^2).
// u = 0 contributes nothing, and positions clamped to the all-zero window give
// zero by themselves.

// 1 / u of two positions, 0 where u = 0 (a product rather than a skipped term, so
// that a NaN passes on as it does in the unsplit form). The hardware's reciprocal
// is up to 1 ulp off; a Newton step y + y (1 - u y) on the FMA pipe leaves the
// rounding of the result, as the unsplit form's division has. Positions are below
// 2^25 and, where not 0, above 1e-19: nothing here leaves the normal range.
__device__ __forceinline__ float2 inv_u(float u0, float u1) {
  const float2 u = make_float2(u0, u1);
  const float2 y = make_float2(u0 > 0.f ? rcp_approx(u0) : 0.f, u1 > 0.f ? rcp_approx(u1) : 0.f);
  const float2 e = __ffma2_rn(__fmul2_rn(u, make_float2(-1.f, -1.f)), y, make_float2(1.f, 1.f));
  return __ffma2_rn(y, e, y);
}

// Pass 2 of one pair over aperture entries [r0, r1): G += the entries' terms
// (without the 1/dt factors). nbeta = -beta.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void adj_scalar(const EvalArgs& a, const Lane& L, int r0, int r1,
                                           const float* s, float alpha, float nbeta, float* G) {
  constexpr int K = 2 * W + 1;
  const T* __restrict__ tr = static_cast<const T*>(a.traces);
  for (int e = r0; e < r1; ++e) {
    const float4 t4 = __ldg(a.ap_tab + e);
    const Pos P = locate<OP, MV>(L, t4);
    const T* x = tr + (__float_as_uint(t4.w) + P.j - W);
    float xv[K + 1];
#pragma unroll
    for (int k = 0; k <= K; ++k) xv[k] = ld_sample<T>(x + k);
    float sg = 0.f, ag = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float gk = __fsub_rn(xv[k + 1], xv[k]);
      const float ak = fmaf(P.f, xv[k + 1], __fmul_rn(P.g, xv[k]));
      sg = fmaf(s[k], gk, sg);
      ag = fmaf(ak, gk, ag);
    }
    const float c = __fmul_rn(fmaf(alpha, sg, __fmul_rn(nbeta, ag)), inv_u(P.u, P.u).x);
    const float hc = __fmul_rn(0.5f, c), cq = __fmul_rn(c, P.q);
    if (OP == TT_OP_FOCRS) {  // dU = 2q dm, 2q dh, dm^2, dm dh, dh^2
      const float hm = __fmul_rn(hc, t4.x), hh = __fmul_rn(hc, t4.y);
      G[0] = fmaf(cq, t4.x, G[0]);
      G[1] = fmaf(cq, t4.y, G[1]);
      G[2] = fmaf(hm, t4.x, G[2]);
      G[3] = fmaf(hm, t4.y, G[3]);
      G[4] = fmaf(hh, t4.y, G[4]);
    } else if (OP == TT_OP_CRS) {
      G[0] = fmaf(cq, t4.x, G[0]);
      G[1] = fmaf(hc, t4.y, G[1]);
      G[2] = fmaf(hc, t4.z, G[2]);
    } else {
      G[0] = fmaf(hc, t4.z, G[0]);
    }
  }
}

// The same for two pairs sharing an aperture, with packed FP32x2 arithmetic.
template <int OP, int W, typename T, bool MV>
__device__ __forceinline__ void adj_packed(const EvalArgs& a, const Lane& L0, const Lane& L1,
                                           int r0, int r1, const float2* s, float2 alpha,
                                           float2 nbeta, float2* G) {
  constexpr int K = 2 * W + 1;
  const T* __restrict__ tr = static_cast<const T*>(a.traces);
  const float2 m1 = make_float2(-1.f, -1.f), half = make_float2(0.5f, 0.5f);
  for (int e = r0; e < r1; ++e) {
    const float4 t4 = __ldg(a.ap_tab + e);
    const Pos P0 = locate<OP, MV>(L0, t4), P1 = locate<OP, MV>(L1, t4);
    const unsigned base = __float_as_uint(t4.w) - W;
    const T* x0 = tr + (base + P0.j);
    const T* x1 = tr + (base + P1.j);
    float2 xv[K + 1];
#pragma unroll
    for (int k = 0; k <= K; ++k) xv[k] = make_float2(ld_sample<T>(x0 + k), ld_sample<T>(x1 + k));
    const float2 f = make_float2(P0.f, P1.f), g = make_float2(P0.g, P1.g);
    float2 sg = make_float2(0.f, 0.f), ag = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float2 gk = __ffma2_rn(xv[k], m1, xv[k + 1]);
      const float2 ak = __ffma2_rn(f, xv[k + 1], __fmul2_rn(g, xv[k]));
      sg = __ffma2_rn(s[k], gk, sg);
      ag = __ffma2_rn(ak, gk, ag);
    }
    const float2 d = __ffma2_rn(alpha, sg, __fmul2_rn(nbeta, ag));
    const float2 c = __fmul2_rn(d, inv_u(P0.u, P1.u));
    const float2 hc = __fmul2_rn(half, c), cq = __fmul2_rn(c, make_float2(P0.q, P1.q));
    const float2 tx = make_float2(t4.x, t4.x), ty = make_float2(t4.y, t4.y),
                 tz = make_float2(t4.z, t4.z);
    if (OP == TT_OP_FOCRS) {
      const float2 hm = __fmul2_rn(hc, tx), hh = __fmul2_rn(hc, ty);
      G[0] = __ffma2_rn(cq, tx, G[0]);
      G[1] = __ffma2_rn(cq, ty, G[1]);
      G[2] = __ffma2_rn(hm, tx, G[2]);
      G[3] = __ffma2_rn(hm, ty, G[3]);
      G[4] = __ffma2_rn(hh, ty, G[4]);
    } else if (OP == TT_OP_CRS) {
      G[0] = __ffma2_rn(cq, tx, G[0]);
      G[1] = __ffma2_rn(hc, ty, G[1]);
      G[2] = __ffma2_rn(hc, tz, G[2]);
    } else {
      G[0] = __ffma2_rn(hc, tz, G[0]);
    }
  }
}

// S, alpha and -beta from a pair's sums; false (and both zero) when the energy
// is 0 or NaN. An infinite energy has a gradient like its S: NaN.
template <typename T>
__device__ __forceinline__ bool grad_factors(float Q, int N, float E, double Ed, float& S,
                                             float& alpha, float& nbeta) {
  S = normalise<T>(Q, N, E, Ed);
  const float En = Chunk<T>::kF64 ? float(Ed) : E;
  const bool ok = En > 0.f;
  alpha = ok ? 2.f / (float(N) * En) : 0.f;
  nbeta = ok ? -2.f * S / En : 0.f;
  return ok;
}

// dS of pair q: the 1/dt factors; zero without an energy to divide by.
template <int OP>
__device__ __forceinline__ void store_grad(const EvalArgs& a, long long q, float inv_dt, bool ok,
                                           const float* G) {
  constexpr int D = op_dim(OP);
  constexpr int n1 = OP == TT_OP_FOCRS ? 2 : OP == TT_OP_CRS ? 1 : 0;  // slopes: 1/dt
  const float i2 = inv_dt * inv_dt;
  float* out = a.dS + q * D;
#pragma unroll
  for (int d = 0; d < D; ++d) out[d] = ok ? G[d] * (d < n1 ? inv_dt : i2) : 0.f;
}

// K2 with one pair per thread, both passes in entry order: the form of the
// polish (which compares the S of successive iterates, so its sums may not
// depend on the launch), of splitting off and of short apertures. U entries
// are in flight at a time: their table rows, positions and windows are loaded
// before the first is added. A small launch of one pair per domain has few
// warps to hide an L2 load behind and takes U = 6 (1008 traces, w = 5, 1,500 /
// 60,000 domains: one entry at a time 808 / 956 us, two 563 / 761, four 412 /
// 623, six 364 / 581); a large one has the warps and takes U = 1 (300,000
// domains 2126 us, four at a time 2305 us). U does not change a bit.
template <int OP, int W, typename T, bool MV, int U, typename F>
__device__ __forceinline__ void each_window(const EvalArgs& a, const Lane& L, F&& add) {
  constexpr int K = 2 * W + 1;
  const T* __restrict__ tr = static_cast<const T*>(a.traces);
  for (int e = L.e0; e < L.e1; e += U) {
    float4 t4[U];
    Pos P[U];
    float xv[U][K + 1];
#pragma unroll
    for (int v = 0; v < U; ++v) t4[v] = __ldg(a.ap_tab + min(e + v, L.e1 - 1));
#pragma unroll
    for (int v = 0; v < U; ++v) {
      P[v] = locate<OP, MV, true>(L, t4[v]);
      const T* x = tr + (__float_as_uint(t4[v].w) + P[v].j - W);
#pragma unroll
      for (int k = 0; k <= K; ++k) xv[v][k] = ld_sample<T>(x + k);
    }
#pragma unroll
    for (int v = 0; v < U; ++v)
      if (e + v < L.e1) add(t4[v], P[v], xv[v]);
  }
}

template <int OP, int W, typename T, bool MV, int U>
__global__ void __launch_bounds__(128) k_semblance_grad(const EvalArgs a) {
  constexpr int K = 2 * W + 1;
  constexpr int D = op_dim(OP);
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  Lane L;
  if (!lane_setup<OP>(a, q, L)) return;
  float s[K];
#pragma unroll
  for (int k = 0; k < K; ++k) s[k] = 0.f;
  float E = 0.f;
  each_window<OP, W, T, MV, U>(a, L, [&](float4, const Pos& P, const float* xv) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const float ak = fmaf(P.f, xv[k + 1], __fmul_rn(P.g, xv[k]));
      s[k] += ak;
      E = fmaf(ak, ak, E);
    }
  });
  float Q = 0.f;
#pragma unroll
  for (int k = 0; k < K; ++k) Q = fmaf(s[k], s[k], Q);
  const float N = float(L.e1 - L.e0);
  const float S = (E > 0.f) ? Q / (N * E) : 0.f;
  float G[D];
#pragma unroll
  for (int d = 0; d < D; ++d) G[d] = 0.f;
  if (E > 0.f) {
    const float alpha = 2.f / (N * E);
    const float beta = 2.f * S / E;
    each_window<OP, W, T, MV, U>(a, L, [&](float4 t4, const Pos& P, const float* xv) {
      float sg = 0.f, ag = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float gk = xv[k + 1] - xv[k];
        const float ak = fmaf(P.f, xv[k + 1], __fmul_rn(P.g, xv[k]));
        sg = fmaf(s[k], gk, sg);
        ag = fmaf(ak, gk, ag);
      }
      const float dSdu = fmaf(alpha, sg, -beta * ag);
      const float inv_u = (P.u > 0.f && P.u < L.umax) ? 1.f / P.u : 0.f;
      const float c = dSdu * inv_u;
      if (OP == TT_OP_FOCRS) {  // dU = 2q dm, 2q dh, dm^2, dm dh, dh^2
        G[0] = fmaf(c * P.q, t4.x, G[0]);
        G[1] = fmaf(c * P.q, t4.y, G[1]);
        G[2] = fmaf(0.5f * c, t4.x * t4.x, G[2]);
        G[3] = fmaf(0.5f * c, t4.x * t4.y, G[3]);
        G[4] = fmaf(0.5f * c, t4.y * t4.y, G[4]);
      } else if (OP == TT_OP_CRS) {
        G[0] = fmaf(c * P.q, t4.x, G[0]);
        G[1] = fmaf(0.5f * c, t4.y, G[1]);
        G[2] = fmaf(0.5f * c, t4.z, G[2]);
      } else {
        G[0] = fmaf(0.5f * c, t4.z, G[0]);
      }
    });
  }
  a.S[q] = S;
  constexpr int n1 = OP == TT_OP_FOCRS ? 2 : OP == TT_OP_CRS ? 1 : 0;  // slopes: 1/dt
  const float i2 = L.inv_dt * L.inv_dt;
#pragma unroll
  for (int d = 0; d < D; ++d) a.dS[q * D + d] = G[d] * (d < n1 ? L.inv_dt : i2);
}

// K2 split: a cluster of B blocks of kGradWarps warps shares one 64-pair unit,
// warp w of block b walking slice b kGradWarps + w of every pair's aperture in
// both passes. Each pass's partial sums meet in shared memory (slices in
// order) and across the cluster's blocks through distributed shared memory
// (blocks in order); the cluster barriers take the place of a second launch.
// The gradient usually has one pair per domain, so that a thread per pair
// leaves a few warps per SM, each waiting on 1008 x 2 dependent window loads:
// 60,000 CRS domains, 1008 traces, w = 5: 880 us (572 us with six entries in
// flight), now 473 us; 1500 domains 700 us (319 us), now 28 us. Three blocks per
// SM (80 registers) hide more load latency than two (540 us); it stays bound by
// its window loads (two passes at K1's rate). From sums that the evaluation kept
// (a.sums) it is the second pass alone.
constexpr int kGradWarps = 8;

// shared memory of a block: FP64 energies [kGradWarps + 1][64]; rows of 64
// floats that hold the slice sums of s and E [kGradWarps][K + 1], later the
// unit's s and E, alpha, -beta and the slices' G [kGradWarps][D]; and the
// block's sums [K + 1] (later its G [D])
constexpr int grad_rows(int W, int D) {
  const int R = 2 * W + 2, first = kGradWarps * R, second = R + 2 + kGradWarps * D;
  return first > second ? first : second;
}
constexpr size_t grad_smem_bytes(int W, int D) {
  const int R = 2 * W + 2;
  return 64 * (sizeof(float) * size_t(grad_rows(W, D) + (R > D ? R : D)) +
               sizeof(double) * size_t(kGradWarps + 1));
}
static_assert(grad_smem_bytes(TT_MAX_HALF_WINDOW, 5) <= 48 * 1024, "fits without an opt-in");

template <int OP, int W, typename T, bool MV>
__global__ void __launch_bounds__(32 * kGradWarps, 3) k_semblance_grad_split(const EvalArgs a) {
  constexpr int K = 2 * W + 1, R = K + 1;  // R rows of 64: s_k and E
  constexpr int D = op_dim(OP);
  constexpr int S = kGradWarps, NT = 32 * S;
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char grad_smem[];
  double* part_Ed = reinterpret_cast<double*>(grad_smem);      // [S][64]
  double* blk_Ed = part_Ed + S * 64;                           // [64]
  float* part = reinterpret_cast<float*>(blk_Ed + 64);         // [S][R][64]
  float* blk = part + grad_rows(W, D) * 64;                    // [R][64]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int B = int(cl.num_blocks()), rank = int(cl.block_rank());
  const long long unit = blockIdx.x / B;
  const long long q0 = unit * 64 + lane, q1 = q0 + 32;
  Lane L0, L1;
  const bool v0 = lane_setup<OP, true>(a, q0, L0), v1 = lane_setup<OP, true>(a, q1, L1);
  const bool both = v0 && v1 && same_aperture(L0, L1);
  __shared__ int size[64];
  if (w == 0) keep_sizes(size, lane, v0, L0, v1, L1);
  int r0 = 0, r1 = 0;
  if (both) slice_of(L0, S * B, rank * S + w, r0, r1);
  if (!a.sums) {  // pass 1, unless the forward launch has kept its sums
    if (both) {
      float2 s[K];
#pragma unroll
      for (int k = 0; k < K; ++k) s[k] = make_float2(0.f, 0.f);
      float2 E = make_float2(0.f, 0.f);
      double Ed0 = 0.0, Ed1 = 0.0;
      acc_packed<OP, W, T, MV>(a, L0, L1, r0, r1, s, E, Ed0, Ed1);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        part[(w * R + k) * 64 + lane] = s[k].x;
        part[(w * R + k) * 64 + lane + 32] = s[k].y;
      }
      part[(w * R + K) * 64 + lane] = E.x;
      part[(w * R + K) * 64 + lane + 32] = E.y;
      if (Chunk<T>::kF64) {
        part_Ed[w * 64 + lane] = Ed0;
        part_Ed[w * 64 + lane + 32] = Ed1;
      }
    } else {
      for (int h = 0; h < 2; ++h) {
        float s[K], E = 0.f;
        double Ed = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] = 0.f;
        if (h ? v1 : v0) {
          const Lane& L = h ? L1 : L0;
          slice_of(L, S * B, rank * S + w, r0, r1);
          acc_scalar<OP, W, T, MV>(a, L, r0, r1, s, E, Ed);
        }
        const int p = lane + 32 * h;
#pragma unroll
        for (int k = 0; k < K; ++k) part[(w * R + k) * 64 + p] = s[k];
        part[(w * R + K) * 64 + p] = E;
        if (Chunk<T>::kF64) part_Ed[w * 64 + p] = Ed;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < R * 64; i += NT) {
      float t = 0.f;
#pragma unroll
      for (int v = 0; v < S; ++v) t = __fadd_rn(t, part[v * R * 64 + i]);
      blk[i] = t;
    }
    if (Chunk<T>::kF64 && threadIdx.x < 64) {
      double t = 0.0;
      for (int v = 0; v < S; ++v) t += part_Ed[v * 64 + threadIdx.x];
      blk_Ed[threadIdx.x] = t;
    }
    if (B > 1) cl.sync(); else __syncthreads();
  }
  // the unit's sums, in every block, over the slice sums that are done with
  float* tot = part;                     // [R][64]
  float* fac = part + R * 64;            // alpha [64], -beta [64]
  float* gsl = fac + 2 * 64;             // [S][D][64]
  for (int i = threadIdx.x; i < R * 64; i += NT) {
    float t = 0.f;
    if (a.sums)
      t = a.sums[unit * (R * 64) + i];
    else
      for (int b = 0; b < B; ++b)
        t = __fadd_rn(t, B > 1 ? cl.map_shared_rank(blk, b)[i] : blk[i]);
    tot[i] = t;
  }
  __syncthreads();
  bool ok = false;  // thread p < 64: pair p has an energy
  if (threadIdx.x < 64 && size[threadIdx.x] >= 0) {
    const int p = threadIdx.x;
    float Q = 0.f, Sv, al, nb;
#pragma unroll
    for (int k = 0; k < K; ++k) Q = fmaf(tot[k * 64 + p], tot[k * 64 + p], Q);
    double Ed = 0.0;
    if (Chunk<T>::kF64 && a.sums)
      Ed = a.sums_Ed[unit * 64 + p];
    else if (Chunk<T>::kF64)
      for (int b = 0; b < B; ++b) Ed += B > 1 ? cl.map_shared_rank(blk_Ed, b)[p] : blk_Ed[p];
    ok = grad_factors<T>(Q, size[p], tot[K * 64 + p], Ed, Sv, al, nb);
    fac[p] = al;
    fac[64 + p] = nb;
    if (rank == 0 && !a.sums) a.S[unit * 64 + p] = Sv;
  }
  if (B > 1 && !a.sums) cl.sync(); else __syncthreads();  // every block has read blk: it is free
  // pass 2
  if (both) {
    float2 s[K], G[D];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = make_float2(tot[k * 64 + lane], tot[k * 64 + lane + 32]);
#pragma unroll
    for (int d = 0; d < D; ++d) G[d] = make_float2(0.f, 0.f);
    adj_packed<OP, W, T, MV>(a, L0, L1, r0, r1, s, make_float2(fac[lane], fac[lane + 32]),
                             make_float2(fac[64 + lane], fac[96 + lane]), G);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      gsl[(w * D + d) * 64 + lane] = G[d].x;
      gsl[(w * D + d) * 64 + lane + 32] = G[d].y;
    }
  } else {
    for (int h = 0; h < 2; ++h) {
      const int p = lane + 32 * h;
      float s[K], G[D];
#pragma unroll
      for (int d = 0; d < D; ++d) G[d] = 0.f;
      if (h ? v1 : v0) {
        const Lane& L = h ? L1 : L0;
        slice_of(L, S * B, rank * S + w, r0, r1);
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] = tot[k * 64 + p];
        adj_scalar<OP, W, T, MV>(a, L, r0, r1, s, fac[p], fac[64 + p], G);
      }
#pragma unroll
      for (int d = 0; d < D; ++d) gsl[(w * D + d) * 64 + p] = G[d];
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < D * 64; i += NT) {
    float t = 0.f;
#pragma unroll
    for (int v = 0; v < S; ++v) t = __fadd_rn(t, gsl[v * D * 64 + i]);
    blk[i] = t;
  }
  if (B > 1) cl.sync(); else __syncthreads();
  if (rank == 0 && threadIdx.x < 64) {
    const int p = threadIdx.x;
    Lane L;
    if (lane_setup<OP>(a, unit * 64 + p, L)) {
      float G[D];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        G[d] = 0.f;
        for (int b = 0; b < B; ++b)
          G[d] = __fadd_rn(G[d], B > 1 ? cl.map_shared_rank(blk, b)[d * 64 + p] : blk[d * 64 + p]);
      }
      store_grad<OP>(a, unit * 64 + p, L.inv_dt, ok, G);
    }
  }
  if (B > 1) cl.sync();  // no block leaves while another may read its sums
}

using KFn = void (*)(const EvalArgs);

// Stacked output (P = 1, theta [n_dom][D]): 32 strided sums of the centre
// amplitudes -- sum l takes aperture entries e0 + l, e0 + l + 32, ... in order
// -- added in a butterfly (sums 16 apart, then 8, ...), and the mean is one
// FP32 division. Positions are those of the semblance window's centre sample
// (same clamp: T < 0 or past the record reads the zero padding). Two forms
// with the same operations, so the same bits.
template <int OP, typename T, bool MV>
__device__ __forceinline__ float centre(const EvalArgs& a, const Lane& L, int e, float s) {
  const float4 t4 = __ldg(a.ap_tab + e);
  const Pos P = locate<OP, MV, true>(L, t4);
  const T* x = static_cast<const T*>(a.traces) + (__float_as_uint(t4.w) + P.j);
  return __fadd_rn(s, fmaf(P.f, ld_sample<T>(x + 1), __fmul_rn(P.g, ld_sample<T>(x))));
}

// Domains with apertures of their own: one warp per domain, lane l taking sum l.
template <int OP, typename T, bool MV>
__global__ void __launch_bounds__(256) k_stack(const EvalArgs a, float* __restrict__ out) {
  const long long d = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  Lane L;
  if (!lane_setup<OP>(a, d, L)) return;  // warp-uniform: the whole warp leaves
  float s = 0.f;
  for (int e = L.e0 + lane; e < L.e1; e += 32) s = centre<OP, T, MV>(a, L, e, s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
  if (lane == 0) {
    const int N = L.e1 - L.e0;
    out[L.d] = N > 0 ? __fdiv_rn(s, float(N)) : 0.f;
  }
}

// Domains that share apertures (consecutive t0 of one midpoint): one lane per
// domain, so that a warp walks the same entries and reads one trace row at 32
// neighbouring positions (a line or two a request, against 32 lines where a
// warp spreads over 32 rows). 32 / R warps share 32 domains, each holding R of
// their sums in registers; the sums meet in shared memory.
template <int OP, typename T, bool MV, int R>
__global__ void __launch_bounds__(R == 1 ? 1024 : 256) k_stack_rows(const EvalArgs a,
                                                                     float* __restrict__ out) {
  constexpr int NW = R == 1 ? 32 : 8;  // warps per block
  constexpr int per = 32 / R;          // warps per 32 domains
  __shared__ float sums[NW / per][32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = w / per, l0 = (w - g * per) * R;
  const long long d = ((long long)blockIdx.x * (NW / per) + g) * 32 + lane;
  Lane L;
  const bool valid = lane_setup<OP>(a, d, L);
  float s[R];
#pragma unroll
  for (int r = 0; r < R; ++r) s[r] = 0.f;
  if (valid) {
    int e = L.e0 + l0;
    for (; e + R <= L.e1; e += 32) {
#pragma unroll
      for (int r = 0; r < R; ++r) s[r] = centre<OP, T, MV>(a, L, e + r, s[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (e + r < L.e1) s[r] = centre<OP, T, MV>(a, L, e + r, s[r]);
  }
#pragma unroll
  for (int r = 0; r < R; ++r) sums[g][lane][l0 + r] = s[r];
  __syncthreads();
  if (l0 != 0 || !valid) return;
  float t[32];
#pragma unroll
  for (int l = 0; l < 32; ++l) t[l] = sums[g][lane][l];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int l = 0; l < o; ++l) t[l] = __fadd_rn(t[l], t[l + o]);
  const int N = L.e1 - L.e0;
  out[L.d] = N > 0 ? __fdiv_rn(t[0], float(N)) : 0.f;
}

// Member order of one population for the evaluation that follows: one warp
// per domain ranks the domain's P members (P <= kOrderMaxP) by the position
// of their window on the domain's middle aperture entry (ties by index; an
// empty aperture keeps the index order), then writes member i's parameters
// to row rank(i) of theta_out and i to slots[d * P + rank(i)]. Evaluating
// theta_out with those slots as the scatter map gives every member its own
// semblance bit for bit (a pair's arithmetic does not depend on its lane),
// while the 32 lanes of a warp read windows that lie close together.
constexpr int kOrderWarps = 8;

template <int OP, bool MV>
__global__ void __launch_bounds__(32 * kOrderWarps) k_member_order(const EvalArgs a,
                                                                   float* __restrict__ theta_out,
                                                                   int* __restrict__ slots) {
  __shared__ float key[kOrderWarps][kOrderMaxP];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long d = (long long)blockIdx.x * kOrderWarps + w;
  if (d >= a.n_dom) return;  // warp-uniform
  const int P = a.P;
  for (int i = lane; i < P; i += 32) {
    Lane L;
    float k = 0.f;
    if (lane_setup<OP>(a, d * P + i, L) && L.e1 > L.e0) {
      k = locate<OP, MV>(L, __ldg(a.ap_tab + ((L.e0 + L.e1) >> 1))).u;
      if (!(k == k)) k = 3.0e38f;
    }
    key[w][i] = k;
  }
  __syncwarp();
  constexpr int D = op_dim(OP);
  for (int i = lane; i < P; i += 32) {
    const float ki = key[w][i];
    int rank = 0;
    for (int j = 0; j < P; ++j) {
      const float kj = key[w][j];
      rank += (kj < ki || (kj == ki && j < i)) ? 1 : 0;
    }
    const float* src = a.theta + (d * P + i) * D;
    float* dst = theta_out + (d * P + rank) * D;
#pragma unroll
    for (int k = 0; k < D; ++k) dst[k] = src[k];
    slots[d * P + rank] = i;
  }
}

using FFn = void (*)(const EvalArgs, const DeArgs, const FusedArgs);

template <int OP, typename T, bool MV>
FFn pick_fused_w(int W) {
  switch (W) {
    case 0: return k_search_short<OP, 0, T, MV>;
    case 1: return k_search_short<OP, 1, T, MV>;
    case 2: return k_search_short<OP, 2, T, MV>;
    case 3: return k_search_short<OP, 3, T, MV>;
    case 4: return k_search_short<OP, 4, T, MV>;
    case 5: return k_search_short<OP, 5, T, MV>;
    case 6: return k_search_short<OP, 6, T, MV>;
    case 7: return k_search_short<OP, 7, T, MV>;
    case 8: return k_search_short<OP, 8, T, MV>;
  }
  return nullptr;
}

template <int OP>
FFn pick_fused(int storage, int W, bool mv) {
  const bool bf = storage == TT_STORE_BF16;
  if (mv)
    return bf ? pick_fused_w<OP, __nv_bfloat16, true>(W) : pick_fused_w<OP, float, true>(W);
  return bf ? pick_fused_w<OP, __nv_bfloat16, false>(W) : pick_fused_w<OP, float, false>(W);
}

using OFn = void (*)(const EvalArgs, float*, int*);

template <int OP>
OFn pick_order(bool mv) {
  return mv ? k_member_order<OP, true> : k_member_order<OP, false>;
}

using SFn = void (*)(const EvalArgs, float*);
enum KernelKind {
  kKindPacked = 0, kKindScalar = 1, kKindSplit = 2, kKindGrad = 3, kKindGradSplit = 4,
  kKindGradAhead = 5, kKindShort = 6, kKindSplitGlobal = 7
};

template <int OP, int W, typename T, bool MV>
KFn pick_kind(int kind) {
  switch (kind) {
    case kKindPacked: return k_semblance<OP, W, T, MV>;
    case kKindScalar: return k_semblance_scalar<OP, W, T, MV>;
    case kKindSplit: return k_semblance_split<OP, W, T, MV, false>;
    case kKindSplitGlobal: return k_semblance_split<OP, W, T, MV, true>;
    case kKindShort: return k_semblance_short<OP, W, T, MV>;
    case kKindGrad: return k_semblance_grad<OP, W, T, MV, 1>;
    case kKindGradAhead: return k_semblance_grad<OP, W, T, MV, 6>;
    case kKindGradSplit: return k_semblance_grad_split<OP, W, T, MV>;
  }
  return nullptr;
}

template <int OP, typename T, bool MV>
KFn pick_w(int kind, int W) {
  switch (W) {
    case 0: return pick_kind<OP, 0, T, MV>(kind);
    case 1: return pick_kind<OP, 1, T, MV>(kind);
    case 2: return pick_kind<OP, 2, T, MV>(kind);
    case 3: return pick_kind<OP, 3, T, MV>(kind);
    case 4: return pick_kind<OP, 4, T, MV>(kind);
    case 5: return pick_kind<OP, 5, T, MV>(kind);
    case 6: return pick_kind<OP, 6, T, MV>(kind);
    case 7: return pick_kind<OP, 7, T, MV>(kind);
    case 8: return pick_kind<OP, 8, T, MV>(kind);
  }
  return nullptr;
}

// The kernel of one kind for operator OP, storage type and half window W;
// mv selects the moveout form of the position.
template <int OP>
KFn pick_kernel(int kind, int storage, int W, bool mv) {
  const bool bf = storage == TT_STORE_BF16;
  if (mv) return bf ? pick_w<OP, __nv_bfloat16, true>(kind, W) : pick_w<OP, float, true>(kind, W);
  return bf ? pick_w<OP, __nv_bfloat16, false>(kind, W) : pick_w<OP, float, false>(kind, W);
}

// The stack kernel of operator OP: rows = 0 the warp-per-domain form, else the
// lane-per-domain form with that many sums per warp.
template <int OP, typename T, bool MV>
SFn pick_stack_rows(int rows) {
  switch (rows) {
    case 0: return k_stack<OP, T, MV>;
    case 1: return k_stack_rows<OP, T, MV, 1>;
    case 8: return k_stack_rows<OP, T, MV, 8>;
  }
  return nullptr;
}

template <int OP>
SFn pick_stack(int storage, bool mv, int rows) {
  const bool bf = storage == TT_STORE_BF16;
  if (mv)
    return bf ? pick_stack_rows<OP, __nv_bfloat16, true>(rows)
              : pick_stack_rows<OP, float, true>(rows);
  return bf ? pick_stack_rows<OP, __nv_bfloat16, false>(rows)
            : pick_stack_rows<OP, float, false>(rows);
}

}  // namespace sk
}  // namespace tt
