// Launch logic and entry points of the semblance kernels (semblance_kernels.cuh):
// forward evaluation (K1 in its packed, persistent, scalar and small-launch
// split forms), the adjoint gradient (K2) and the stacked output.
#include "semblance_kernels.cuh"

#include <cmath>

namespace tt {
namespace sk {
extern template KFn pick_kernel<TT_OP_CMP>(int, int, int, bool);
extern template KFn pick_kernel<TT_OP_CRS>(int, int, int, bool);
extern template KFn pick_kernel<TT_OP_FOCRS>(int, int, int, bool);
extern template SFn pick_stack<TT_OP_CMP>(int, bool, int);
extern template SFn pick_stack<TT_OP_CRS>(int, bool, int);
extern template SFn pick_stack<TT_OP_FOCRS>(int, bool, int);
extern template OFn pick_order<TT_OP_CMP>(bool);
extern template OFn pick_order<TT_OP_CRS>(bool);
extern template OFn pick_order<TT_OP_FOCRS>(bool);
extern template FFn pick_fused<TT_OP_CMP>(int, int, bool);
extern template FFn pick_fused<TT_OP_CRS>(int, int, bool);
extern template FFn pick_fused<TT_OP_FOCRS>(int, int, bool);
}  // namespace sk

namespace {

using sk::KFn;

constexpr int kDirectMax = 2048;  // direct position up to u = 2048 samples

KFn pick(int kind, const EvalArgs& a, bool mv) {
  switch (a.op) {
    case TT_OP_CMP: return sk::pick_kernel<TT_OP_CMP>(kind, a.storage, a.W, mv);
    case TT_OP_CRS: return sk::pick_kernel<TT_OP_CRS>(kind, a.storage, a.W, mv);
    case TT_OP_FOCRS: return sk::pick_kernel<TT_OP_FOCRS>(kind, a.storage, a.W, mv);
  }
  return nullptr;
}

// A block's shared memory above 48 KB, the kernel's own arrays included, has
// to be asked for. The limit belongs to the kernel, for every context and host
// thread: `most` is the largest size any launch of fn takes, so that no call
// lowers the limit between another's setting it and launching.
template <typename Fn>
cudaError_t allow_smem(Fn fn, size_t most) {
  if (most <= 40 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most));
}

// Sums of eight slices per pair of a split launch (see semblance_kernels.cuh).
int split_blocks(long long units, int n_sm) {
  return units * 2 <= n_sm                              ? kSplitTinyBlocks
         : units <= (long long)n_sm * kSplitSmallPerSm ? kSplitSmallBlocks
         : units < (long long)n_sm * kSplitMultiPerSm  ? 2
                                                       : 1;
}

// Whether a launch of B blocks a unit adds its blocks' sums through the scratch (if
// it has one) rather than in clusters. A launch takes as long as the SM with the most
// blocks, and clusters, placed whole within a part of the chip, do not fill every
// SM: 61 of nine blocks and 83 of seven fit at four blocks an SM (occupancy query)
// where 67 and 86 times as many single blocks do, 0.905 and (over all numbers of
// blocks an SM) 0.93 of them. Where that is one block more for some SM, single blocks
// win (FP32, w = 5, 5000 traces, 48 / 62 / 125 / 149 / 167 / 299 units 52 / 65 / 112 /
// 128 / 143 / 237 us against 62 / 75 / 125 / 147 / 154 / 250; BF16, w = 8, 62 / 149
// units 104 / 208 us against 121 / 244); elsewhere the way through global memory costs
// 2 to 5 us more (36 / 77 / 119 / 179 units 52 / 79 / 112 / 157 against 51 / 77 / 109 /
// 157), which apertures below 1500 traces do not win back either way (1008 traces,
// 118 / 152 / 282 units 34 / 41 / 64 against 32 / 40 / 61).
bool scratch_wins(const EvalArgs& a, long long units, int B) {
  if (B < kSplitSmallBlocks || a.mean_ap < kSplitScratchMinAp) return false;
  const double per_sm = double(units * B) / a.n_sm;
  return std::ceil(per_sm / (B == kSplitTinyBlocks ? 0.905 : 0.93)) > std::ceil(per_sm);
}

cudaError_t launch_split(EvalArgs& a, long long units, bool mv, cudaStream_t s) {
  const bool bf = a.storage == TT_STORE_BF16;
  const int B = split_blocks(units, a.n_sm);
  a.split_blocks = B;
  // 7 warps a unit instead of 56 while they are not walked for longer than the
  // 56 take to come and go: 48 traces 118 / 258 units 8.7 / 10.4 us against
  // 10.5 / 18.5 us, 144 traces 258 units 18.6 against 22.8 us; 336 traces 118 /
  // 258 units 20.7 / 34.9 us against 16.7 / 31.1 us
  // The launch ends with its longest aperture, which eight times fewer warps walk:
  // 300 units of 40 traces, one of 2000: 121 us against 25 us; ten of 240 / 320 20.6 /
  // 25.8 against 22.3 / 22.8; 160 units of 40, ten of 120 / 160 14.1 / 16.3 against
  // 12.6 / 13.3; 300 units of 150, twenty of 250 26.7 against 30.6.
  if (B == kSplitSmallBlocks && a.mean_ap <= 0.6f * float(units) &&
      float(a.max_ap) <= 0.7f * float(units) + 0.5f * a.mean_ap) {
    const KFn fn = pick(sk::kKindShort, a, mv);
    if (!fn) return cudaErrorInvalidValue;
    const size_t smem = sk::short_smem_bytes(kSplitSmallBlocks, a.W, bf);
    const cudaError_t e = allow_smem(fn, smem);
    if (e != cudaSuccess) return e;
    fn<<<unsigned(units), 32 * kSplitSmallBlocks, smem, s>>>(a);
    return cudaGetLastError();
  }
  if (a.part && scratch_wins(a, units, B)) {  // a block's own eight sets fit without asking
    const KFn fn = pick(sk::kKindSplitGlobal, a, mv);
    if (!fn) return cudaErrorInvalidValue;
    fn<<<unsigned(units * B), 32 * sk::kSplitWarps, sk::split_smem_bytes(1, a.W, bf), s>>>(a);
    return cudaGetLastError();
  }
  const KFn fn = pick(sk::kKindSplit, a, mv);
  if (!fn) return cudaErrorInvalidValue;
  const size_t smem = sk::split_smem_bytes(B, a.W, bf);
  cudaError_t e = allow_smem(fn, sk::split_smem_bytes(kSplitTinyBlocks, a.W, bf));
  if (e == cudaSuccess && B > 8)  // more blocks than every device has to offer
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  // load-balancing rather than spread placement of the clusters: ENS 5 x 1 sweep
  // 19.3 -> 18.6 ms, 125 units x 6120 traces 168 -> 160 us
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(B);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
  attr[1].val.clusterSchedulingPolicyPreference = cudaClusterSchedulingPolicyLoadBalancing;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(units * B));
  cfg.blockDim = dim3(32 * sk::kSplitWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, fn, a);
}

// Split gradient launches: where forward launches split (their sums then agree
// bit for bit, and so does S), with apertures of 256 traces or more (1008
// traces: 24 / 282 / 938 / 4688 units 28 / 189 / 473 / 1962 us against 319 / 374 /
// 572 / 2217 us with one pair per thread), with shorter ones down to 16 traces
// while the launch has fewer than 16 units per SM (144 traces: 469 units 60 us
// against 67 us, 4688 units 322 us against 307 us; 48 traces: 16 units 16 us
// against 19 us, 9375 units 284 us against 217 us).
bool grad_split(const EvalArgs& a, long long units) {
  return a.split && units < (long long)a.n_sm * kSplitUnitsPerSm &&
         (a.mean_ap >= 256.f || (a.mean_ap >= 16.f && units < 16ll * a.n_sm));
}

// Pairs times aperture entries (half as many in BF16 storage, whose S is evaluated
// as well) up to which a differentiated evaluation takes the adjoint at once. Both
// ways a pass forward and backward is host time there, and the backward's own launch
// adds 40 to 60 us of it (4,000 x 1008: 220 against 279 us); a value whose backward
// never comes takes the adjoint's time instead of the evaluation's, at most some 80
// us more (4,000 x 1008: 52 against 33 us; 16 million: about 140 against 60).
constexpr double kGradTogetherMax = 16777216.0;

// The cluster has the forward launch's B blocks, 9, 7, 2 or 1, so that S agrees
// with it (1008 traces, clusters of 1 / 2 / 4 / 7 / 8 / 9: 24 units 107 / 61 / 36 /
// 32 / 27 / 27 us, 282 units 290 / 217 / 176 / 189 / 185 / 189 us, 938 units 560 /
// 473 / 468 / 574 / 565 / 591 us, 4688 units 1964 / 1972 / 2157 / 2767 / 2740 / 2888
// us: the rule's 9, 7, 2 and 1 lie within 8% of the best).
cudaError_t launch_grad_split(const EvalArgs& a, long long units, bool mv, cudaStream_t s) {
  const KFn fn = pick(sk::kKindGradSplit, a, mv);
  if (!fn) return cudaErrorInvalidValue;
  const int B = split_blocks(units, a.n_sm);
  if (B > 8) {
    const cudaError_t e =
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  if (units * B > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = unsigned(B);
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(units * B));
  cfg.blockDim = dim3(32 * sk::kGradWarps);
  cfg.dynamicSmemBytes = sk::grad_smem_bytes(a.W, op_dim(a.op));
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, a);
}

cudaError_t launch(const EvalArgs& a, cudaStream_t s, bool grad) {
  const long long n = (long long)a.n_dom * a.P;
  if (n == 0) return cudaSuccess;
  const int block = (a.block == 128) ? 128 : 256;
  // records longer than kDirectMax samples use the moveout form of the position
  const bool mv = a.umax > float(kDirectMax);
  KFn fn;
  long long blocks;
  EvalArgs b = a;
  if (grad) {
    const long long units = (n + 63) / 64;
    if (a.sums || grad_split(a, units)) return launch_grad_split(a, units, mv, s);
    // few pairs: several entries in flight, in small blocks that spread over the SMs
    const bool few = n < 768ll * a.n_sm;
    fn = pick(few ? sk::kKindGradAhead : sk::kKindGrad, a, mv);
    if (!fn) return cudaErrorInvalidValue;
    const int threads = few ? 32 : 128;
    blocks = (n + threads - 1) / threads;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    fn<<<unsigned(blocks), threads, 0, s>>>(a);
    return cudaGetLastError();
  } else if (a.split && (n + 63) / 64 < (long long)a.n_sm * kSplitUnitsPerSm) {
    // too few units to fill the GPU: each unit's aperture split over warps
    return launch_split(b, (n + 63) / 64, mv, s);
  } else if (a.kernel == TT_KERNEL_SCALAR) {
    fn = pick(sk::kKindScalar, a, mv);
    blocks = (n + block - 1) / block;
  } else {
    fn = pick(sk::kKindPacked, a, mv);
    const long long units = (n + 63) / 64;
    blocks = (units + block / 32 - 1) / (block / 32);
    if (a.kernel == TT_KERNEL_PERSISTENT && a.queue) {
      int per_sm = 0;
      cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, 0);
      if (e != cudaSuccess) return e;
      const long long resident = (long long)a.n_sm * (per_sm > 0 ? per_sm : 1);
      if (resident < blocks) blocks = resident;
      e = cudaMemsetAsync(a.queue, 0, sizeof(unsigned long long), s);
      if (e != cudaSuccess) return e;
    } else {
      b.queue = nullptr;
    }
  }
  if (!fn) return cudaErrorInvalidValue;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  fn<<<unsigned(blocks), block, 0, s>>>(b);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_semblance(const EvalArgs& a, cudaStream_t s) { return launch(a, s, false); }

cudaError_t launch_stack(const EvalArgs& a, float* out, cudaStream_t s) {
  if (a.n_dom == 0) return cudaSuccess;
  if (a.P != 1) return cudaErrorInvalidValue;
  const bool mv = a.umax > float(kDirectMax);
  // One lane per domain where consecutive domains mostly share an aperture: runs
  // of 4 domains of a group on average already win (2000 groups of 4, 1008 traces:
  // 29 us against 42 us with a warp per domain; of 1500: below). Groups whose
  // domains are scattered (200 groups x 1500 with the group changing at every
  // domain: 1734 us against 761 us) keep the warp per domain. One warp per
  // sum until the launch has 16 groups of 32 domains per SM, then 8 sums per
  // warp (20 / 60 / 200 CMPs x 1500 samples, 1008 traces, one sum a warp 36 /
  // 87 / 305 us, eight 45 / 88 / 241 us, a warp per domain 93 / 265 / 843 us).
  const long long groups32 = ((long long)a.n_dom + 31) / 32;
  const int rows = a.n_dom < 4ll * a.n_runs ? 0 : groups32 < 16ll * a.n_sm ? 1 : 8;
  sk::SFn fn = nullptr;
  switch (a.op) {
    case TT_OP_CMP: fn = sk::pick_stack<TT_OP_CMP>(a.storage, mv, rows); break;
    case TT_OP_CRS: fn = sk::pick_stack<TT_OP_CRS>(a.storage, mv, rows); break;
    case TT_OP_FOCRS: fn = sk::pick_stack<TT_OP_FOCRS>(a.storage, mv, rows); break;
  }
  if (!fn) return cudaErrorInvalidValue;
  const int threads = rows == 1 ? 1024 : 256;
  // warps that the launch needs: one per domain, or 32 / rows per 32 domains
  const long long warps = rows ? groups32 * (32 / rows) : a.n_dom;
  const long long blocks = (warps * 32 + threads - 1) / threads;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  fn<<<unsigned(blocks), threads, 0, s>>>(a, out);
  return cudaGetLastError();
}

cudaError_t launch_semblance_grad(const EvalArgs& a, cudaStream_t s) { return launch(a, s, true); }

// How a differentiated evaluation runs: its value now, its gradient later or
// never. The sums of a split evaluation are kept and the gradient starts from
// them (60,000 domains x 1008 traces: the value 197 us, with its gradient 483 us
// through autograd, against 459 and 478 us with the adjoint at once and 197 and
// 675 us with a launch of each; 300,000 x 144: 129 and 336 us, 307 and 325 us, 129
// and 460 us). Where a pass is host time either way, the adjoint gives value and
// gradient at once (kGradTogetherMax). What the evaluation does not split, or holds
// apertures too short for split gradients, is evaluated and differentiated by
// launches of their own.
long long grad_sums_bytes(const EvalArgs& a) {
  const long long n = (long long)a.n_dom * a.P, units = (n + 63) / 64;
  if (!a.split || n == 0 || units >= (long long)a.n_sm * kSplitUnitsPerSm || a.mean_ap < 16.f)
    return 0;
  const double work = double(n) * a.mean_ap * (a.storage == TT_STORE_BF16 ? 2.0 : 1.0);
  if (work <= kGradTogetherMax && grad_split(a, units)) return -1;
  return units * (long long)(a.storage == TT_STORE_BF16 ? sk::split_set_bytes<__nv_bfloat16>(a.W)
                                                        : sk::split_set_bytes<float>(a.W));
}

// Apertures of up to 160 traces, or of 1.5 per unit where the 64 slots of a
// block are nearly full: DE 32 x 30 on 38 / 150 / 300 units of 48 traces 144 /
// 134 / 173 us against 291 / 302 / 344 us stepwise, of 144 traces 253 / 267 /
// 370 against 289 / 504 / 525, of 336 traces 446 / 665 / 799 against 341 / 672
// / 1122, of 1008 traces 1258 / 1898 / 2164 against 602 / 1352 / 2297. A block
// holds 64 / NP whole domains, so that populations of 33 to 60 members fill it
// less and a launch may need a second wave: up to 120 traces then (NP 33, 589
// blocks for 304 units, 48 / 120 / 160 traces 319 / 630 / 769 us against 393 / 647
// / 749 us). A search ends with its longest aperture, by seven warps where the
// stepwise launch has 56: 76 domains, mean 66 to 70 traces, longest 180 / 240 / 600
// 295 / 356 / 781 us against 287 / 299 / 352 us; 300 of mean 22, longest 250 / 310
// 365 / 472 against 378 / 380; 600 of mean 99 to 110, longest 400 / 450 798 / 1023
// against 838 / 864.
bool fused_search_fits(const EvalArgs& a) {
  const long long units = ((long long)a.n_dom * a.P + 63) / 64;
  if (!a.split || a.P > 64 || a.dom_map || units > (long long)a.n_sm * kSplitSmallPerSm)
    return false;
  const int per = 64 / a.P;
  const long long blocks = (a.n_dom + per - 1) / per;
  if (float(a.max_ap) > a.mean_ap + 110.f + 0.75f * float(units)) return false;
  return a.mean_ap <= (blocks > 2ll * a.n_sm ? 120.f : 160.f) ||
         (a.mean_ap <= 1.5f * float(units) && per * a.P * 6 >= 64 * 5);
}

cudaError_t launch_fused_search(const EvalArgs& a, const DeArgs& de, const FusedArgs& f,
                                cudaStream_t s) {
  if (a.n_dom == 0) return cudaSuccess;
  const bool mv = a.umax > float(kDirectMax);
  sk::FFn fn = nullptr;
  switch (a.op) {
    case TT_OP_CMP: fn = sk::pick_fused<TT_OP_CMP>(a.storage, a.W, mv); break;
    case TT_OP_CRS: fn = sk::pick_fused<TT_OP_CRS>(a.storage, a.W, mv); break;
    case TT_OP_FOCRS: fn = sk::pick_fused<TT_OP_FOCRS>(a.storage, a.W, mv); break;
  }
  const int B = split_blocks(((long long)a.n_dom * a.P + 63) / 64, a.n_sm);
  // the kernel adds kSplitSmallBlocks or kSplitTinyBlocks sets, no fewer
  if (!fn || a.P > 64 || B < kSplitSmallBlocks) return cudaErrorInvalidValue;
  const int per = 64 / a.P;
  const bool bf = a.storage == TT_STORE_BF16;
  const size_t smem = sk::short_smem_bytes(B, a.W, bf);
  const cudaError_t e = allow_smem(fn, sk::short_smem_bytes(kSplitTinyBlocks, a.W, bf));
  if (e != cudaSuccess) return e;
  fn<<<(a.n_dom + per - 1) / per, 32 * B, smem, s>>>(a, de, f);
  return cudaGetLastError();
}

cudaError_t launch_member_order(const EvalArgs& a, float* theta_out, int* slots,
                                cudaStream_t s) {
  if (a.n_dom == 0) return cudaSuccess;
  if (a.P < 1 || a.P > kOrderMaxP || a.dom_map) return cudaErrorInvalidValue;
  const bool mv = a.umax > float(kDirectMax);
  sk::OFn fn = nullptr;
  switch (a.op) {
    case TT_OP_CMP: fn = sk::pick_order<TT_OP_CMP>(mv); break;
    case TT_OP_CRS: fn = sk::pick_order<TT_OP_CRS>(mv); break;
    case TT_OP_FOCRS: fn = sk::pick_order<TT_OP_FOCRS>(mv); break;
  }
  if (!fn) return cudaErrorInvalidValue;
  const long long blocks = ((long long)a.n_dom + sk::kOrderWarps - 1) / sk::kOrderWarps;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
  fn<<<unsigned(blocks), 32 * sk::kOrderWarps, 0, s>>>(a, theta_out, slots);
  return cudaGetLastError();
}

// L1 load-bandwidth probe: every warp streams 4-byte loads (the instruction
// K1 gathers its windows with), 32 consecutive floats per warp request, from
// a 24 KiB window that stays in L1. Each iteration starts at another line of
// the window (a multiple of 37 lines, modulo 64), so no load repeats an
// earlier iteration's address and none can be moved out of the loop; their
// sum is written so that none is dropped. The grid is one wave of resident
// blocks (at most 8 of 256 threads per SM).
constexpr int kProbeThreads = 256, kProbeBlocksPerSm = 8, kProbeLoads = 32;
__global__ void __launch_bounds__(kProbeThreads, 4) k_l1_probe(const float* buf, int iters,
                                                               float* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* base = buf + ((warp & 1) * 3072 + lane);
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int it = 0; it < iters; ++it) {
    const float* p = base + ((it * 37) & 63) * 32;
#pragma unroll
    for (int u = 0; u < kProbeLoads; ++u) acc[u & 7] += __ldg(p + u * 32);
  }
  float t = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) t += acc[u];
  if (t == 1.2345f) out[0] = t;  // practically never: keeps the loads live
}

cudaError_t launch_l1_probe(const float* buf, float* out, int n_sm, int iters, double* bytes,
                            cudaStream_t s) {
  // one wave: as many blocks as stay resident on every SM at once
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_l1_probe,
                                                                kProbeThreads, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  if (per_sm > kProbeBlocksPerSm) per_sm = kProbeBlocksPerSm;
  const long long blocks = (long long)n_sm * per_sm;
  *bytes = double(blocks) * kProbeThreads * double(iters) * kProbeLoads * sizeof(float);
  k_l1_probe<<<unsigned(blocks), kProbeThreads, 0, s>>>(buf, iters, out);
  return cudaGetLastError();
}

}  // namespace tt

extern "C" tt_status tt_semblance_eval(tt_ctx* ctx, const float* theta, int32_t P, float* S,
                                       void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (P < 1) return tt_fail(ctx, TT_ERR_INVALID_ARG, "P must be >= 1");
  if (ctx->n_dom > 0 && (!theta || !S)) return tt_fail(ctx, TT_ERR_INVALID_ARG, "NULL array");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const tt::EvalArgs a = ctx->call_args(theta, P, S, s);
  return tt_cuda_check(ctx, ctx->semblance(a, s, false), "semblance launch");
}

extern "C" tt_status tt_stack(tt_ctx* ctx, const float* theta, float* out, void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (ctx->n_dom > 0 && (!theta || !out)) return tt_fail(ctx, TT_ERR_INVALID_ARG, "NULL array");
  tt::EvalArgs a = ctx->eval_args(theta, 1, nullptr);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return tt_cuda_check(ctx, ctx->counted(tt::launch_stack(a, out, s)), "stack launch");
}

extern "C" tt_status tt_semblance_grad(tt_ctx* ctx, const float* theta, int32_t P, float* S,
                                       float* dS, void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (P < 1) return tt_fail(ctx, TT_ERR_INVALID_ARG, "P must be >= 1");
  if (ctx->n_dom > 0 && (!theta || !S || !dS))
    return tt_fail(ctx, TT_ERR_INVALID_ARG, "NULL array");
  tt::EvalArgs a = ctx->eval_args(theta, P, S);
  a.dS = dS;
  return tt_cuda_check(ctx, ctx->semblance(a, static_cast<cudaStream_t>(stream), true),
                       "semblance gradient launch");
}

extern "C" tt_status tt_semblance_sums_size(tt_ctx* ctx, int32_t P, int64_t* bytes) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (P < 1) return tt_fail(ctx, TT_ERR_INVALID_ARG, "P must be >= 1");
  if (!bytes) return tt_fail(ctx, TT_ERR_INVALID_ARG, "bytes is NULL");
  *bytes = tt::grad_sums_bytes(ctx->eval_args(nullptr, P, nullptr));
  return TT_OK;
}

namespace {

// The two parts of a buffer of sums (the same whatever the launch's slices).
void set_sums(tt::EvalArgs& a, void* sums) {
  const size_t units = ((size_t)a.n_dom * a.P + 63) / 64;
  a.sums_Ed = a.storage == TT_STORE_BF16 ? static_cast<double*>(sums) : nullptr;
  a.sums = a.sums_Ed ? reinterpret_cast<float*>(a.sums_Ed + units * 64)
                     : static_cast<float*>(sums);
}

}  // namespace

extern "C" tt_status tt_semblance_eval_sums(tt_ctx* ctx, const float* theta, int32_t P, float* S,
                                            void* sums, void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (P < 1) return tt_fail(ctx, TT_ERR_INVALID_ARG, "P must be >= 1");
  if (!theta || !S || !sums) return tt_fail(ctx, TT_ERR_INVALID_ARG, "NULL array");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  tt::EvalArgs a = ctx->call_args(theta, P, S, s);
  if (tt::grad_sums_bytes(a) <= 0)
    return tt_fail(ctx, TT_ERR_INVALID_ARG, "this launch keeps no sums");
  set_sums(a, sums);
  return tt_cuda_check(ctx, ctx->semblance(a, s, false), "semblance launch");
}

extern "C" tt_status tt_semblance_grad_sums(tt_ctx* ctx, const float* theta, int32_t P,
                                            const void* sums, float* dS, void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (P < 1) return tt_fail(ctx, TT_ERR_INVALID_ARG, "P must be >= 1");
  if (ctx->n_dom > 0 && (!theta || !sums || !dS))
    return tt_fail(ctx, TT_ERR_INVALID_ARG, "NULL array");
  tt::EvalArgs a = ctx->eval_args(theta, P, nullptr);
  a.dS = dS;
  set_sums(a, const_cast<void*>(sums));
  return tt_cuda_check(ctx, ctx->semblance(a, static_cast<cudaStream_t>(stream), true),
                       "semblance gradient launch");
}

extern "C" tt_status tt_ctx_probe_l1(tt_ctx* ctx, int32_t iters, double* bytes, void* stream) {
  if (!ctx) return tt_fail(nullptr, TT_ERR_INVALID_ARG, "ctx is NULL");
  if (iters < 1 || !bytes) return tt_fail(ctx, TT_ERR_INVALID_ARG, "iters < 1 or bytes is NULL");
  // the window and the sink live in the context (no allocation)
  return tt_cuda_check(ctx,
                       ctx->counted(tt::launch_l1_probe(ctx->probe, ctx->probe + 8192,
                                                        ctx->n_sm, iters, bytes,
                                                        static_cast<cudaStream_t>(stream))),
                       "L1 probe launch");
}
