// Kernels of the ARA engine outside the layer's hot loop: input checks and
// per-record preparation at load time, the quantile tables, the check kernels,
// the scan and the per-layer event index.  The two layer kernels are in
// ara_layer.cu.
#include <cuda_runtime.h>

#include <cstdint>

#include "ara_df.cuh"
#include "ara_batch.h"

namespace ara {

namespace {

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// Exclusive block scan of one uint32 per thread.  s_warp needs 33 words.
// All threads of the block must call it.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* s_warp, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_warps = (blockDim.x + 31) >> 5;
  const uint32_t incl = warp_inclusive_scan(v);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint32_t x = (lane < n_warps) ? s_warp[lane] : 0u;
    const uint32_t xi = warp_inclusive_scan(x);
    s_warp[lane] = xi - x;
    if (lane == 31) s_warp[32] = xi;
  }
  __syncthreads();
  const uint32_t r = s_warp[warp] + incl - v;
  *total = s_warp[32];
  __syncthreads();
  return r;
}

}  // namespace

// =============================================================== load-time checks
__global__ void k_check_offsets(const int64_t* off, int64_t n_trials, int64_t n_events, uint32_t* flags) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  uint32_t f = 0;
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < n_trials; t += stride) {
    const int64_t a = off[t], b = off[t + 1];
    if (b < a) f |= kBadOffsets;
    if (b - a >= static_cast<int64_t>(kMaxTrialEvents)) f |= kLongTrial;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (off[0] != 0 || off[n_trials] != n_events) f |= kBadOffsets;
  }
  if (f) atomicOr(flags, f);
}

__global__ void k_check_ids(const int32_t* ids, int64_t n, int32_t catalogue, uint32_t* flags) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  bool bad = false;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    const int32_t e = ids[i];
    bad |= (e < 0) | (e >= catalogue);
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flags, kBadEventId);
}

// The YET upload from pinned host memory: each thread moves int4 groups of
// ids (four groups in flight) when the source is 16-byte aligned, single ids
// otherwise, and flags any id outside [0, catalogue).  A few blocks keep
// enough reads in flight to fill the host link.
constexpr int kUploadBlocks = 32;
constexpr int kUploadThreads = 512;

__device__ __forceinline__ bool id_bad(int32_t e, uint32_t cat) { return static_cast<uint32_t>(e) >= cat; }

__global__ void __launch_bounds__(kUploadThreads) k_upload_ids(const int32_t* __restrict__ src,
                                                               int32_t* __restrict__ dst, int64_t n,
                                                               int32_t catalogue, uint32_t* flags) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t tid = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint32_t cat = static_cast<uint32_t>(catalogue);
  bool bad = false;
  int64_t k0 = 0;  // first id of the single-id tail
  if ((reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
    const int4* s4 = reinterpret_cast<const int4*>(src);
    int4* d4 = reinterpret_cast<int4*>(dst);
    const int64_t n4 = n >> 2;
    int64_t i = tid;
    for (; i + 3 * stride < n4; i += 4 * stride) {
      int4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = s4[i + j * stride];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        d4[i + j * stride] = v[j];
        bad |= id_bad(v[j].x, cat) | id_bad(v[j].y, cat) | id_bad(v[j].z, cat) | id_bad(v[j].w, cat);
      }
    }
    for (; i < n4; i += stride) {
      const int4 v = s4[i];
      d4[i] = v;
      bad |= id_bad(v.x, cat) | id_bad(v.y, cat) | id_bad(v.z, cat) | id_bad(v.w, cat);
    }
    k0 = 4 * n4;
  }
  for (int64_t k = k0 + tid; k < n; k += stride) {
    const int32_t e = src[k];
    dst[k] = e;
    bad |= id_bad(e, cat);
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flags, kBadEventId);
}

cudaError_t launch_upload_ids(const int32_t* src, int32_t* dst, int64_t n, int32_t catalogue, uint32_t* flags,
                              cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  k_upload_ids<<<kUploadBlocks, kUploadThreads, 0, s>>>(src, dst, n, catalogue, flags);
  return cudaGetLastError();
}

cudaError_t launch_check_offsets(const int64_t* off, int64_t n_trials, int64_t n_events, uint32_t* flags,
                                 cudaStream_t s) {
  const int64_t blocks = (n_trials + 255) / 256;
  k_check_offsets<<<static_cast<int>(blocks < 4096 ? (blocks > 0 ? blocks : 1) : 4096), 256, 0, s>>>(
      off, n_trials, n_events, flags);
  return cudaGetLastError();
}

cudaError_t launch_check_ids(const int32_t* ids, int64_t n, int32_t catalogue, uint32_t* flags, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t blocks = (n + 1023) / 1024;
  k_check_ids<<<static_cast<int>(blocks < 8192 ? blocks : 8192), 1024, 0, s>>>(ids, n, catalogue, flags);
  return cudaGetLastError();
}

// =============================================================== record preparation (FP64)
namespace {

// Continued fraction of I_x(a, b) (A&S 26.5.8) in FP64; returns 1/K with
// K = 1 + d1/(1 + d2/(1 + ...)), d_n = p_n / q_n:
//   n = 2m+1: p_n = -(a + m)(a + b + m) x, q_n = (a + 2m)(a + 2m + 1),
//   n = 2m:   p_n = m (b - m) x,            q_n = (a + 2m - 1)(a + 2m).
// The equivalence transformation with c_n = q_n clears the denominators
// (partial numerators q_{n-1} p_n, partial denominators q_n), so the forward
// recurrence A_n = b'_n A_{n-1} + a'_n A_{n-2} (and B_n alike) needs only
// multiply-adds; every 8 terms the pairs are rescaled by 1/B_n, which is where
// convergence of A_n / B_n is tested.  FP64 divisions are slow on this GPU, so
// this costs about a tenth of the modified Lentz method.
__device__ double beta_cf_f64_ref(double a, double b, double x) {
  double A2 = 1.0, B2 = 0.0;  // A_{n-2}, B_{n-2}
  double A1 = 1.0, B1 = 1.0;  // A_{n-1}, B_{n-1}
  double q_prev = 1.0, f_prev = 1.0;
  for (int n = 1; n <= 40000; ++n) {
    const double h = static_cast<double>(n >> 1);
    double pn, qn;
    if (n & 1) {
      pn = -(a + h) * (a + b + h) * x;
      qn = (a + 2.0 * h) * (a + 2.0 * h + 1.0);
    } else {
      pn = h * (b - h) * x;
      qn = (a + 2.0 * h - 1.0) * (a + 2.0 * h);
    }
    const double an = q_prev * pn;  // q_0 = 1 gives a'_1 = p_1
    const double A0 = fma(qn, A1, an * A2);
    const double B0 = fma(qn, B1, an * B2);
    A2 = A1;
    B2 = B1;
    A1 = A0;
    B1 = B0;
    q_prev = qn;
    if ((n & 7) == 0) {
      const double inv = 1.0 / B1;
      A1 *= inv;
      A2 *= inv;
      B2 *= inv;
      B1 = 1.0;
      if (fabs(A1 - f_prev) <= 1e-15 * fabs(A1)) break;
      f_prev = A1;
    }
  }
  return B1 / A1;
}

// The continued fraction of beta_cf_f64_ref in double-float arithmetic, two
// terms (the odd and the even one of each m) per iteration: FP64 runs at a
// small fraction of the FP32 rate on this GPU, and 48 bits carry the value to
// the 1e-13 relative tolerance used here (the table nodes are FP32; their
// polish and check need the CDF to about 1e-10).  FP32's exponent range is
// kept by rescaling the four convergents by a power of two each iteration
// (exact; the ratio is unchanged).  False when a value leaves the FP32 range or
// the iteration does not converge, for the FP64 fallback.
__device__ bool beta_cf_df(double a, double b, double x, double* num, double* den) {
  const DF X = df_of(x);
  DF v = df_of(a);          // a + m
  DF w = df_of(a + b);      // a + b + m
  DF y = df_of(b - 1.0);    // b - m - 1
  DF u = df_of(a);          // a + 2m
  DF A2{1.0f, 0.0f}, B2{0.0f, 0.0f}, A1{1.0f, 0.0f}, B1{1.0f, 0.0f};
  DF q_prev{1.0f, 0.0f};
  double Ap = 1.0, Bp = 1.0;  // the convergent of the last test
  for (int m = 0; m < 20000; ++m) {
    const DF u1 = df_add_f(u, 1.0f), u2 = df_add_f(u, 2.0f);
    // odd term n = 2m + 1: p = -(a + m)(a + b + m) x, q = (a + 2m)(a + 2m + 1)
    const DF qo = df_mul(u, u1);
    const DF ao = df_mul(q_prev, df_neg(df_mul(df_mul(v, w), X)));
    DF A0 = df_add(df_mul(qo, A1), df_mul(ao, A2));
    DF B0 = df_add(df_mul(qo, B1), df_mul(ao, B2));
    // even term n = 2m + 2: p = (m + 1)(b - m - 1) x, q = (a + 2m + 1)(a + 2m + 2)
    const DF qe = df_mul(u1, u2);
    const DF ae = df_mul(qo, df_mul(df_mul(DF{static_cast<float>(m + 1), 0.0f}, y), X));
    const DF Ae = df_add(df_mul(qe, A0), df_mul(ae, A1));
    const DF Be = df_add(df_mul(qe, B0), df_mul(ae, B1));
    A2 = A0;
    B2 = B0;
    A1 = Ae;
    B1 = Be;
    q_prev = qe;
    v = df_add_f(v, 1.0f);
    w = df_add_f(w, 1.0f);
    y = df_add_f(y, -1.0f);
    u = u2;
    const float big = fmaxf(fabsf(A1.hi), fabsf(B1.hi));
    if (!(big < 3.0e38f) || !(big > 0.0f)) return false;
    const int k = -f_exponent(big);
    A1 = df_scale(A1, k);
    A2 = df_scale(A2, k);
    B1 = df_scale(B1, k);
    B2 = df_scale(B2, k);
    if ((m & 3) == 3) {
      // |A1/B1 - Ap/Bp| <= 1e-13 |A1/B1|, cross-multiplied in FP64 (the quotients' divisions and the conversions
      // took a third of the table build)
      const double An = df_val_fast(A1), Bn = df_val_fast(B1), f = An * Bp;
      if (fabs(fma(-Ap, Bn, f)) <= 1e-13 * fabs(f)) {
        *num = Bn;
        *den = An;
        return true;
      }
      Ap = An;
      Bp = Bn;
    }
  }
  return false;
}

// The continued fraction of I_x(a, b), num / den: double-float, else FP64.
__device__ void beta_cf_f64(double a, double b, double x, double* num, double* den) {
  if (beta_cf_df(a, b, x, num, den) && isfinite(*num) && isfinite(*den) && *den != 0.0) return;
  *num = beta_cf_f64_ref(a, b, x);
  *den = 1.0;
}

}  // namespace

// Section 3.3 per record: sigma_b = sigma / max_l, mu_b = mu / max_l,
// sigma_bmax = sqrt(mu_b (1 - mu_b)), sigma_b clipped to (1 - 1e-6) sigma_bmax,
// alpha = mu_b ((sigma_bmax / sigma_b)^2 - 1), beta = (1 - mu_b)(...).  With a
// correlated part sigma_C (Section 3.1), sigma = sigma_I + sigma_C
// (Section 3.2 step i) and a record with sigma_C > 0 is of kind kKindBetaC,
// with weights (sigma_I, sigma_C) / sqrt(sigma_I^2 + sigma_C^2) for the
// combination of its two normal variables.
// blockIdx.y is the ELT, of records [rec_off[y], rec_off[y + 1]), with its
// results at elts + kEltWords y.
__global__ void k_prepare_records(const int32_t* events, const float* mean, const float* sigma,
                                  const float* exposure, const int64_t* rec_off, Pair* out, BetaShape* shapes,
                                  uint32_t* elts, const float* sigma_c, float2* weights) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t begin = rec_off[blockIdx.y], end = rec_off[blockIdx.y + 1];
  uint32_t* flags = elts + static_cast<int64_t>(blockIdx.y) * kEltWords;
  int32_t* max_event = reinterpret_cast<int32_t*>(flags + kEltMaxEvent);
  uint32_t* max_loss = flags + kEltMaxLoss;
  uint32_t f = 0;
  int32_t emax = -1;
  float lmax = 0.0f;
  for (int64_t i = begin + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < end; i += stride) {
    const int32_t e = events[i];
    emax = max(emax, e);
    if (e < 0) f |= kBadEventId;
    if (i > begin && events[i - 1] >= e) f |= kBadOrder;
    const double mu = mean[i], si = sigma[i], ex = exposure[i];
    const double sc = sigma_c ? static_cast<double>(sigma_c[i]) : 0.0;
    const double sg = si + sc;
    Pair p;
    p.a = p.b = p.m0 = p.c = p.p_half = 0.0f;
    p.max_l = static_cast<float>(ex);
    p.mu = static_cast<float>(mu);
    uint32_t kind = kKindBeta;
    double sa = 0.0, sb_ = 0.0, slnb = 0.0;
    float2 w = make_float2(1.0f, 0.0f);
    if (!(mu >= 0.0) || !(si >= 0.0) || !(sc >= 0.0) || !isfinite(mu) || !isfinite(sg) || !isfinite(ex)) {
      f |= kBadValue;
      kind = kKindZero;
    } else if (mu == 0.0) {
      kind = kKindZero;
    } else if (sg == 0.0) {
      kind = kKindMean;
    } else if (!(ex > mu)) {
      f |= kBadExposure;
      kind = kKindZero;
    } else {
      const double mb = mu / ex, sb0 = sg / ex;
      const double smax = sqrt(mb * (1.0 - mb));
      const double sb = (sb0 >= (1.0 - 1e-6) * smax) ? (1.0 - 1e-6) * smax : sb0;
      const double k = (smax / sb) * (smax / sb) - 1.0;
      const double a = mb * k, b = (1.0 - mb) * k;
      const double x0 = a / (a + b), y0 = b / (a + b);
      const double lnB = lgamma(a) + lgamma(b) - lgamma(a + b);
      const double c = a * log(x0) + b * log(y0) - lnB;
      // I_{1/2}(a, b), only used to pick the side of the root
      const double lfront = -(a + b) * 0.69314718055994530942 - lnB;
      double ph, num, den;
      if (0.5 < (a + 1.0) / (a + b + 2.0)) {
        beta_cf_f64(a, b, 0.5, &num, &den);
        ph = exp(lfront) * num / (den * a);
      } else {
        beta_cf_f64(b, a, 0.5, &num, &den);
        ph = 1.0 - exp(lfront) * num / (den * b);
      }
      p.a = static_cast<float>(a);
      p.b = static_cast<float>(b);
      sa = a;
      sb_ = b;
      slnb = lnB;
      p.m0 = (x0 <= y0) ? -static_cast<float>(x0) : static_cast<float>(y0);
      p.c = static_cast<float>(c);
      p.p_half = static_cast<float>(ph);
      if (sc > 0.0) {
        kind = kKindBetaC;
        f |= kHasCorrelated;
        const double nrm = sqrt(si * si + sc * sc);
        w = make_float2(static_cast<float>(si / nrm), static_cast<float>(sc / nrm));
      }
    }
    p.meta = (kind << kMetaKindShift) | (static_cast<uint32_t>(i - begin) << kMetaRecShift);
    if (kind != kKindZero) lmax = fmaxf(lmax, fmaxf(p.max_l, p.mu));
    out[i] = p;
    shapes[i] = BetaShape{sa, sb_, slnb, 0.0};
    if (weights) weights[i] = w;
  }
  if (f) atomicOr(flags, f);
  // block max of event ids, then one atomic per warp
  for (int d = 16; d > 0; d >>= 1) {
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, d));
    lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, d));
  }
  if ((threadIdx.x & 31) == 0 && emax >= 0) atomicMax(max_event, emax);
  // non-negative floats order as their bit patterns
  if ((threadIdx.x & 31) == 0 && lmax > 0.0f) atomicMax(max_loss, __float_as_uint(lmax));
}

cudaError_t launch_prepare_records(const int32_t* events, const float* mean, const float* sigma,
                                   const float* exposure, const int64_t* rec_off, int n_elts, int64_t longest,
                                   Pair* out, BetaShape* shapes, uint32_t* elts, cudaStream_t s, const float* sigma_c,
                                   float2* weights, int* n_launch) {
  if (longest == 0) return cudaSuccess;
  const int64_t blocks = (longest + 127) / 128;
  for (int y = 0; y < n_elts; y += 65535) {  // the grid's y limit
    const dim3 grid(static_cast<int>(blocks < 65535 ? blocks : 65535), n_elts - y < 65535 ? n_elts - y : 65535);
    k_prepare_records<<<grid, 128, 0, s>>>(events, mean, sigma, exposure, rec_off + y, out, shapes,
                                           elts + static_cast<int64_t>(y) * kEltWords, sigma_c, weights);
    if (n_launch) *n_launch += 1;
  }
  return cudaGetLastError();
}

// =============================================================== quantile tables (FP64, load time)
namespace {

// I_x(a, b) and 1 - I_x(a, b), each without cancellation (A&S 26.5.8 with
// symmetry).  *front_out (optional) receives x^a (1-x)^b / B(a, b), which is
// x (1 - x) f(x) for the Beta density f.
__device__ void beta_inc_pair_f64(double x, double a, double b, double lnB, double* I, double* Ic,
                                  double* front_out = nullptr, double* lx_out = nullptr, double* l1mx_out = nullptr) {
  if (!(x > 0.0)) {
    *I = 0.0;
    *Ic = 1.0;
    if (front_out) *front_out = 0.0;
    return;
  }
  if (!(x < 1.0)) {
    *I = 1.0;
    *Ic = 0.0;
    if (front_out) *front_out = 0.0;
    return;
  }
  const double lx = log(x), l1mx = log1p(-x);
  const double front = exp(a * lx + b * l1mx - lnB);
  if (front_out) *front_out = front;
  if (lx_out) *lx_out = lx;
  if (l1mx_out) *l1mx_out = l1mx;
  // the fraction on the side where it converges fast: the side is chosen per
  // lane and the fraction called once, so that the lanes of a warp do not
  // run it twice
  const bool lower = x * (a + b + 2.0) < a + 1.0;
  const double p = lower ? a : b, q = lower ? b : a, y = lower ? x : 1.0 - x;
  double num, den;
  beta_cf_f64(p, q, y, &num, &den);
  const double v = front * num / (den * p);
  *I = lower ? v : 1.0 - v;
  *Ic = lower ? 1.0 - v : v;
}

// Root r of I_r(A, B) = p (p <= 1/2) by bracketed Newton in FP64 from `guess`.
// The nodes are stored in FP32, so the iteration stops at 2e-10 relative:
// well below FP32 resolution, and above the ~1e-12 relative noise of the FP64
// evaluation of I for large shapes (cancellation in ln B(A, B)), which a
// tighter tolerance would chase for the whole iteration budget.
__device__ double beta_root_f64(double p, double A, double B, double lnB, double guess) {
  double lo = 0.0, hi = 1.0;
  double r = (guess > 0.0 && guess < 1.0) ? guess : A / (A + B);
  for (int it = 0; it < 60; ++it) {
    double I, Ic;
    beta_inc_pair_f64(r, A, B, lnB, &I, &Ic);
    const double f = I - p;
    if (f == 0.0) return r;
    if (f < 0.0) lo = r; else hi = r;
    const double lpdf = (A - 1.0) * log(r) + (B - 1.0) * log1p(-r) - lnB;
    double rn = r - f * exp(-lpdf);
    if (!(rn > lo && rn < hi)) {
      const double l = fmax(lo, 1e-300);
      if (lo == 0.0 && hi <= 1e-300) return hi;
      rn = (hi > 4.0 * l) ? sqrt(l) * sqrt(hi) : 0.5 * (lo + hi);
    } else if (fabs(rn - r) <= 2e-10 * rn) {
      return rn;
    }
    r = rn;
  }
  return r;
}

// ln(1 + e), e^q - 1: a short series near 0 (to 1e-16 relative below 1e-3),
// where the polish below nearly always is; the library's functions elsewhere.
__device__ __forceinline__ double log1p_near(double e) {
  if (!(fabs(e) < 1e-3)) return log1p(e);
  return e * fma(e, fma(e, fma(e, fma(e, 0.2, -0.25), 1.0 / 3.0), -0.5), 1.0);
}
__device__ __forceinline__ double expm1_near(double q) {
  if (!(fabs(q) < 1e-3)) return expm1(q);
  return q * fma(q, fma(q, fma(q, fma(q, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5), 1.0);
}

// A root r of I_r(A, B) = p, with ln r, ln(1 - r) and B(A, B) / (r^A (1 - r)^B).
struct BetaRoot {
  double r, lr, l1mr, inv_front;
};

__device__ __noinline__ BetaRoot beta_root_of(double p, double A, double B, double lnB, double guess) {
  BetaRoot x;
  x.r = beta_root_f64(p, A, B, lnB, guess);
  x.lr = log(x.r);
  x.l1mr = log1p(-x.r);
  x.inv_front = exp(lnB - A * x.lr - B * x.l1mr);
  return x;
}

// Newton on u = ln r in FP64 from r towards the root of I_r(A, B) = p (p <=
// 1/2), where I ~ r^A near 0 makes the step almost exact: up to `steps` steps,
// ended by one of |du| < tol.  The last step's logarithms and front factor are
// moved along by du, a short series, in place of new ones, and one division
// serves a step.  False when it does not converge; r is then where it stood.
__device__ bool beta_newton_f64(double p, double A, double B, double lnB, int steps, double tol, double* r_io,
                                BetaRoot* out) {
  double r = *r_io;
  for (int it = 0; it < steps; ++it) {
    if (!(r > 0.0 && r < 1.0)) return false;
    double I, Ic, front, lr, l1mr;
    beta_inc_pair_f64(r, A, B, lnB, &I, &Ic, &front, &lr, &l1mr);
    if (!(I > 0.0) || !(front > 0.0)) return false;
    const double y = 1.0 - r;
    const double inv = 1.0 / (y * front * p);
    const double e = (I - p) * (inv * y * front);              // (I - p) / p
    const double du = -log1p_near(e) * (y * y * I * p * inv);  // d ln I / d ln r = front / ((1 - r) I)
    if (!(fabs(du) < 0.5)) return false;
    const double rn = fma(r, expm1_near(du), r);
    if (!(rn > 0.0 && rn < 1.0)) return false;
    if (fabs(du) < tol) {
      const double dl = log1p_near((r - rn) * (inv * front * p));  // ln((1 - rn) / (1 - r))
      const double inv_front = inv * y * p * (1.0 + expm1_near(-(A * du + B * dl)));
      if (!(inv_front > 0.0) || !isfinite(inv_front)) return false;
      *out = BetaRoot{rn, lr + du, l1mr + dl, inv_front};
      return true;
    }
    r = rn;
    *r_io = rn;
  }
  return false;
}

// The root where the polish of the plain seed failed (a root near 1 whose
// complement the seed has lost, one below the FP32 range): the same steps from
// the seed of the root's own side, or from the power law I ~ r^A / (A B(A, B))
// where that is the root to FP64 precision.  They end at |du| < 1e-7, so that
// what is left (du^2) is below the bracketed solver's 2e-10, which takes what
// does not converge here (dozens of FP64 fractions a root: with it alone the
// stress recipe's tables took five times as long as the plain recipe's).
__device__ __noinline__ BetaRoot beta_root_again(double p, double A, double B, double lnB, double own_seed,
                                                 double guess) {
  const double lpow = (log(p) + log(A) + lnB) / A;
  double r = lpow < -46.0 ? exp(lpow) : own_seed;  // below 1e-20
  BetaRoot x;
  if (r > 1e-290 && beta_newton_f64(p, A, B, lnB, 6, 1e-7, &r, &x)) return x;
  return beta_root_of(p, A, B, lnB, guess);
}

// Polish of an FP32 root r of I_r(A, B) = p (p <= 1/2).  The seed is good to
// ~1e-6, so a step |du| < 1e-5 leaves an error of order du^2 (~1e-10, below
// the FP32 resolution of the stored node) and ends the iteration; at most 3
// steps.
__device__ BetaRoot beta_polish_f64(double p, double A, double B, double lnB, double seed, double own_seed) {
  BetaRoot x;
  double r = seed;
  // (a seed more than a factor of two off its own side's fails at the first step)
  if (seed < 2.1 * own_seed && own_seed < 2.1 * seed && beta_newton_f64(p, A, B, lnB, 3, 1e-5, &r, &x)) return x;
  return beta_root_again(p, A, B, lnB, own_seed, seed > 0.0 && seed < 1.0 ? r : -1.0);
}

// What a table's nodes need of t alone: the smaller tail Phi(-|t|) and the
// normal density.
struct TabPoint {
  double t, zl, phi;
};
__device__ TabPoint tab_point(double t) {
  return TabPoint{t, normcdf(-fabs(t)), exp(-0.5 * t * t - 0.91893853320467274178)};
}

}  // namespace

// One node of a record's quantile table at t: the FP64 root x (seeded by the
// FP32 Halley solver), w = ln x, and the derivatives in t, w' = phi(t) / (x f(x))
// and w'' = w' (-t - w' (a - (b-1) x/(1-x))).  Returns {x, 0, h w', h^2 w''}
// (the caller fills in w_{j+1} - w_j) and w.
__device__ float4 table_node(const Pair& pr, double a, double b, double lnB, const TabPoint& q, double h,
                             double* w_out) {
  const double t = q.t, zl = q.zl;
  // FP32 seed, then FP64 polish on the side where the root keeps relative precision
  BetaSolveStats st;
  const float zf = (t <= 0.0) ? static_cast<float>(zl) : static_cast<float>(1.0 - zl);
  const float z = fminf(fmaxf(zf, 5.9604645e-08f), 0.99999994f);
  bool is_x;
  const float root = pair_root_newton(pr, z, -1.0f, &st, &is_x);
  const float seed = is_x ? root : 1.0f - root;
  // the root x (t <= 0) or y = 1 - x (t > 0): the shapes are swapped per lane
  // and the polish called once (ln B is symmetric), so that the two halves of
  // the warp do not run it in turn
  const bool lo = t <= 0.0;
  const BetaRoot v = beta_polish_f64(zl, lo ? a : b, lo ? b : a, lnB,
                                     lo ? static_cast<double>(seed) : 1.0 - static_cast<double>(seed),
                                     lo == is_x ? static_cast<double>(root) : 1.0 - static_cast<double>(root));
  const double x = lo ? v.r : 1.0 - v.r, y = lo ? 1.0 - v.r : v.r;
  const double D = q.phi * y * v.inv_front;  // phi / (x f(x)), as x (1 - x) f(x) is the front factor
  const double E = D * (-t - D * (a - (b - 1.0) * (x / y)));
  *w_out = lo ? v.lr : v.l1mr;
  return make_float4(static_cast<float>(x), 0.0f, static_cast<float>(h * D), static_cast<float>(h * h * E));
}

// Accuracy of the segment [t, t + h] of a table (node nd = {x, dw, h w', h^2 w''}
// at t; d1, e1 the derivative terms of the next node), checked at the midpoint
// tq = t + h / 2, zq = Phi(-|tq|),
// where the error kernel s^3 (1-s)^3 of quintic Hermite interpolation peaks:
// the FP32 interpolant (as the hot path evaluates it) against the FP64 CDF.
// True when the implied relative error of x there is within kTabTol (a bound
// set by the FP32 evaluation of the interpolant, ~2e-7, more than by the
// interpolation error, which elsewhere in the segment is below its midpoint
// value), or x < 1e-30 (negligible losses).
__device__ bool table_segment_ok(float4 nd, float d1, float e1, double tq, double zq, double a, double b, double lnB) {
  if (!(isfinite(nd.x) && isfinite(nd.y) && isfinite(nd.z) && isfinite(nd.w))) return false;
  const float xq = (nd.x > 0.0f) ? nd.x * expf(tab_increment(0.5f, nd.y, nd.z, nd.w, d1, e1)) : 0.0f;
  if (!(xq >= 1e-30f)) return true;
  double I, Ic, front, rel;
  if (xq >= 1.0f) {
    // the FP32 ceiling: fine iff the quantile itself is within 2^-24 of 1
    beta_inc_pair_f64(1.0 - 5.9604644775390625e-08, a, b, lnB, &I, &Ic);
    rel = (tq > 0.0 && Ic >= zq) ? 0.0 : INFINITY;
  } else {
    const double xd = static_cast<double>(xq);
    beta_inc_pair_f64(xd, a, b, lnB, &I, &Ic, &front);
    const double err_z = (tq <= 0.0) ? (I - zq) : (Ic - zq);
    rel = fabs(err_z) * (1.0 - xd) / front;  // |dz| / (x f(x))
  }
  return (rel <= kTabTol) && isfinite(rel);
}

// Coarse tables: a block builds those of 32 records, lane l of every warp the
// record order[32 block + l] (or that record itself without an order), warp w
// the nodes j = w, w + 8, .. at t_j = -T1 + j h, then the segments' checks.  A
// load of few records takes 8 a block and a thread a node, whose chain of nodes
// and checks is a quarter as long (1 record 142 us a load against 230, 1,000
// 382 and 534, 8,000 663 and 667, 16,000 972 and 900).  The stored float4 is
// {x_j, w_{j+1} - w_j, h w'_j, h^2 w''_j}.  need[rec] = 1 for a Beta record whose
// coarse table is not exact (a candidate for a fine table).
// The iteration and fraction lengths follow the shapes and t: with the records
// in order of a + b a warp's lanes, at the same t, run about equally long,
// where a warp per record with a lane per node ran 13 of its 32 lanes (30 now).
// Bound by the FP64 pipe (77% active: logs, exps and divisions around the
// double-float fraction).  150,000 records of the plain recipe: 3.9 ms (3.6 with
// the fraction's stop test in double-float too), a warp per record 10.7, and
// 15.1 with an FP64 division for each test of the fraction and new logarithms
// and exponentials after the last Newton step; of the stress recipe 4.5 ms (4.2),
// 19.8 with the bracketed solver for the roots near 1.  Against those new
// logarithms a node's FP64 root agrees to about 1e-15, and its FP32 value was
// another in one of 100 million nodes compared.
constexpr int kTabThreads = 256;

// kTabRecs: records of a block, thread t the record t mod kTabRecs.
template <int kTabRecs>
__global__ void __launch_bounds__(kTabThreads, 2) k_build_tables(Pair* recs, const BetaShape* shapes, int64_t n,
                                                                 const int64_t* order, float4* tab, uint32_t* need) {
  constexpr int kGroups = kTabThreads / kTabRecs;  // threads of a record
  static_assert(kTabRecs <= 32 && kGroups <= kTabNodes && kTabNodes == 32, "a bit a record, a lane a node");
  // the nodes' and midpoints' normal values, the same for every record
  __shared__ TabPoint pt[kTabNodes];
  __shared__ double mid_t[kTabNodes], mid_z[kTabNodes];
  __shared__ double s_w[kTabRecs][kTabNodes + 1];
  __shared__ float4 s_node[kTabRecs][kTabNodes + 1];
  __shared__ int64_t s_rec[kTabRecs];
  __shared__ uint32_t s_bad;  // records with a segment that fails its check
  const double h = 2.0 * kTabT1 / (kTabNodes - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int own = threadIdx.x % kTabRecs, group = threadIdx.x / kTabRecs;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * kTabRecs + own;
  const int64_t rec = i < n ? (order ? order[i] : i) : -1;
  if (group == 0) s_rec[own] = rec;
  if (warp == 0) {
    const double t = -kTabT1 + h * lane;
    pt[lane] = tab_point(t);
    if (lane == 0) s_bad = 0u;
  } else if (warp == 1) {
    const double t = -kTabT1 + h * lane + 0.5 * h;
    mid_t[lane] = t;
    mid_z[lane] = normcdf(-fabs(t));
  }
  __syncthreads();
  Pair pr{};
  double a = 0.0, b = 0.0, lnB = 0.0;
  bool beta = false;
  if (rec >= 0) {
    pr = recs[rec];
    beta = kind_is_beta(pair_kind(pr.meta));
    a = shapes[rec].a;
    b = shapes[rec].b;
    lnB = shapes[rec].lnB;
  }
#pragma unroll 1
  for (int j = group; j < kTabNodes; j += kGroups) {
    double w = 0.0;
    float4 node = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (beta) node = table_node(pr, a, b, lnB, pt[j], h, &w);
    s_w[own][j] = w;
    s_node[own][j] = node;
  }
  __syncthreads();
#pragma unroll 1
  for (int j = group; j < kTabNodes; j += kGroups) {
    float4 node = s_node[own][j];
    bool ok = true;
    if (j < kTabNodes - 1) {
      node.y = static_cast<float>(s_w[own][j + 1] - s_w[own][j]);
      s_node[own][j].y = node.y;
      const float4* next = &s_node[own][j + 1];
      if (beta) ok = table_segment_ok(node, next->z, next->w, mid_t[j], mid_z[j], a, b, lnB);
    } else {
      ok = isfinite(node.x) && isfinite(node.z) && isfinite(node.w);
    }
    if (!ok) atomicOr(&s_bad, 1u << own);
  }
  __syncthreads();
#pragma unroll 1
  for (int r = warp; r < kTabRecs; r += kTabThreads / 32)
    if (s_rec[r] >= 0) tab[s_rec[r] * kTabNodes + lane] = s_node[r][lane];
  if (group == 0 && rec >= 0) {
    const bool all_ok = ((s_bad >> own) & 1u) == 0u;
    if (beta && all_ok) recs[rec].meta = pr.meta | (1u << kMetaExactBit);
    need[rec] = beta && !all_ok ? 1u : 0u;
  }
}

// Keys that put records with like shapes together: a + b in steps of a quarter
// of its power of two, then the mean a / (a + b) in 64 steps (0 for records
// without a Beta).
__global__ void k_shape_keys(const BetaShape* shapes, int64_t n, unsigned long long* keys, int64_t* order) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    const float sum = static_cast<float>(shapes[i].a + shapes[i].b), mean = static_cast<float>(shapes[i].a) / sum;
    keys[i] = sum > 0.0f ? (((__float_as_uint(sum) >> 21) & 0x3FFu) << 6) | static_cast<uint32_t>(63.0f * mean) : 0u;
    order[i] = i;
  }
}

// Fine tables: global block b is slot b - slot_begin of the job (ELT) whose
// slot range holds b, for that job's (b - slot_begin)-th candidate in record
// order (slots = exclusive prefix of all records' need flags); thread j = node j at
// t_j = -T1 + j h / kTabRefine.  The record's meta then addresses its fine
// table (by the ELT-local slot); it is table-exact if the fine table passes
// the check.
// A block takes slots blockIdx.x, blockIdx.x + gridDim.x, .., so that the nodes'
// and midpoints' normal values are computed once a block.
__global__ void __launch_bounds__(kTabFineStride, 2) k_build_fine(Pair* recs, const BetaShape* shapes,
                                                                 const FineJob* jobs, int n_jobs, const uint32_t* slots,
                                                                 int64_t total_slots, float4* tabf) {
  __shared__ double s_w[kTabFineStride];
  __shared__ float4 s_node[kTabFineStride];
  __shared__ int64_t s_rec;
  __shared__ uint32_t s_ls;
  const double h = 2.0 * kTabT1 / (kTabFineNodes - 1);
  const int j = threadIdx.x;
  const double t = -kTabT1 + h * (j < kTabFineNodes ? j : kTabFineNodes - 1);
  const TabPoint pt = tab_point(t);
  const double mid_z = normcdf(-fabs(t + 0.5 * h));
  for (int64_t gb = blockIdx.x; gb < total_slots; gb += gridDim.x) {
    if (threadIdx.x == 0) {
      int lo = 0, hi = n_jobs - 1;  // the last job with slot_begin <= gb
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].slot_begin <= gb) lo = mid; else hi = mid - 1;
      }
      const FineJob jb = jobs[lo];
      const uint32_t ls = static_cast<uint32_t>(gb - jb.slot_begin);
      int64_t rec = -1;
      const uint32_t* slot = slots + jb.rec_begin;
      if (jb.n > 0 && ls < jb.cap && ls < slot[jb.n] - slot[0]) {
        int64_t l = 0, hh = jb.n - 1;  // the first r with slot[r + 1] > ls
        while (l < hh) {
          const int64_t mid = (l + hh) >> 1;
          if (slot[mid + 1] - slot[0] > ls) hh = mid; else l = mid + 1;
        }
        rec = jb.rec_begin + l;
      }
      s_rec = rec;
      s_ls = ls;
    }
    __syncthreads();
    const int64_t rec = s_rec;
    const uint32_t ls = s_ls;
    if (rec < 0) {
      __syncthreads();  // the next slot rewrites s_rec
      continue;
    }
    const Pair pr = recs[rec];
    const double a = shapes[rec].a, b = shapes[rec].b, lnB = shapes[rec].lnB;
    double w = 0.0;
    float4 node = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (j < kTabFineNodes) node = table_node(pr, a, b, lnB, pt, h, &w);
    s_w[j] = w;
    s_node[j] = node;
    __syncthreads();
    bool ok = true;
    if (j < kTabFineNodes - 1) {
      node.y = static_cast<float>(s_w[j + 1] - w);
      ok = table_segment_ok(node, s_node[j + 1].z, s_node[j + 1].w, t + 0.5 * h, mid_z, a, b, lnB);
    } else if (j == kTabFineNodes - 1) {
      ok = isfinite(node.x) && isfinite(node.z) && isfinite(node.w);
    }
    if (j < kTabFineNodes) tabf[gb * kTabFineStride + j] = node;
    const bool all_ok = __syncthreads_and(ok) != 0;
    if (j == 0)
      recs[rec].meta = (pr.meta & ((1u << kMetaFineBit) - 1u)) | (1u << kMetaFineBit) |
                       (all_ok ? (1u << kMetaExactBit) : 0u) | (ls << kMetaRecShift);
  }
}

constexpr int64_t kTabFew = 8000;  // records up to which a block takes 8 and not 32

size_t build_tables_work_words(int64_t n) { return 2 * static_cast<size_t>(n) + 1 + scan_tmp_words(n); }

uint32_t fine_table_cap(int64_t n) {
  const int64_t cap = n / 16 + 16;
  return static_cast<uint32_t>(cap < n ? cap : n);
}

size_t shape_order_bytes(int64_t n) {
  return static_cast<size_t>(n) * (sizeof(unsigned long long) + sizeof(int64_t)) + sort_pairs_scratch_bytes(n) + 256;
}

cudaError_t launch_shape_order(const BetaShape* shapes, int64_t n, void* scratch, int64_t** order, cudaStream_t s,
                               int* n_launch) {
  unsigned long long* keys = static_cast<unsigned long long*>(scratch);
  *order = reinterpret_cast<int64_t*>(keys + n);
  const int64_t blocks = (n + 255) / 256;
  k_shape_keys<<<static_cast<int>(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(shapes, n, keys, *order);
  if (n_launch) *n_launch += 1;
  const cudaError_t err = cudaGetLastError();
  return err != cudaSuccess ? err : sort_pairs_ascending(keys, *order, n, 16, *order + n, s, n_launch);
}

// Each job's candidates for fine tables, from the scan of the need flags.
__global__ void k_fine_counts(const FineJob* jobs, int n_jobs, const uint32_t* slots, uint32_t* elts) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_jobs; i += gridDim.x * blockDim.x)
    elts[static_cast<int64_t>(jobs[i].elt) * kEltWords + kEltFine] =
        slots[jobs[i].rec_begin + jobs[i].n] - slots[jobs[i].rec_begin];
}

cudaError_t launch_build_tables(Pair* recs, const BetaShape* shapes, int64_t n, const int64_t* order,
                                const FineJob* jobs, int n_jobs, int64_t total_slots, float4* tab, float4* tabf,
                                uint32_t* work, uint32_t* elts, cudaStream_t s, int* n_launch) {
  if (n == 0) return cudaSuccess;
  uint32_t *need = work, *slots = work + n, *tmp = slots + n + 1;
  if (n <= kTabFew)
    k_build_tables<8><<<static_cast<int>((n + 7) / 8), kTabThreads, 0, s>>>(recs, shapes, n, order, tab, need);
  else
    k_build_tables<32><<<static_cast<int>((n + 31) / 32), kTabThreads, 0, s>>>(recs, shapes, n, order, tab, need);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if ((err = scan_exclusive_u32(need, slots, n, tmp, s, n_launch)) != cudaSuccess) return err;
  k_fine_counts<<<(n_jobs + 255) / 256, 256, 0, s>>>(jobs, n_jobs, slots, elts);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  const int64_t most = 4096;
  k_build_fine<<<static_cast<int>(total_slots < most ? total_slots : most), kTabFineStride, 0, s>>>(
      recs, shapes, jobs, n_jobs, slots, total_slots, tabf);
  if (n_launch) *n_launch += 3;
  return cudaGetLastError();
}

// =============================================================== check kernels
__global__ void k_debug_uniforms(uint32_t seed_lo, uint32_t seed_hi, int64_t n, const int64_t* trials,
                                 const int32_t* ks, const int32_t* elts, float* out) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride)
    out[i] = philox_uniform(seed_lo, seed_hi, trials[i], static_cast<uint32_t>(ks[i]), static_cast<uint32_t>(elts[i]));
}

__global__ void k_debug_losses(const Pair* recs, const float4* tab, const float4* tabf, const float* z, int64_t n,
                               int newton_only, float* out, int32_t* iters) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    BetaSolveStats st;
    const Pair pr = recs[i];
    const int64_t r = pair_rec(pr.meta);
    const float4* tb = pair_fine(pr.meta) ? tabf + r * kTabFineStride : tab + r * kTabNodes;
    out[i] = pair_loss(pr, z[i], false, tb, newton_only != 0, &st);
    if (iters) iters[i] = st.converged ? st.iters : -st.iters;
  }
}

cudaError_t launch_debug_uniforms(uint32_t seed_lo, uint32_t seed_hi, int64_t n, const int64_t* trials,
                                  const int32_t* ks, const int32_t* elts, float* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t b = (n + 255) / 256;
  k_debug_uniforms<<<static_cast<int>(b < 65535 ? b : 65535), 256, 0, s>>>(seed_lo, seed_hi, n, trials, ks, elts, out);
  return cudaGetLastError();
}

cudaError_t launch_debug_losses(const Pair* recs, const float4* tab, const float4* tabf, const float* z, int64_t n,
                                int newton_only, float* out, int32_t* iters, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int64_t b = (n + 127) / 128;
  k_debug_losses<<<static_cast<int>(b < 65535 ? b : 65535), 128, 0, s>>>(recs, tab, tabf, z, n, newton_only, out,
                                                                         iters);
  return cudaGetLastError();
}

// =============================================================== exclusive scan (uint32)
namespace {
constexpr int kScanThreads = 1024;
constexpr int kScanPerThread = 8;
constexpr int kScanTile = kScanThreads * kScanPerThread;

// Per-tile sums.
__global__ void k_scan_tile_sums(const uint32_t* in, int64_t n, uint32_t* sums) {
  __shared__ uint32_t s_warp[33];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile + threadIdx.x * kScanPerThread;
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < kScanPerThread; ++j) {
    const int64_t i = base + j;
    if (i < n) v += in[i];
  }
  uint32_t total;
  block_exclusive_scan(v, s_warp, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Exclusive scan of each tile with a starting offset per tile.
__global__ void k_scan_tiles(const uint32_t* in, uint32_t* out, int64_t n, const uint32_t* tile_off,
                             int write_total) {
  __shared__ uint32_t s_warp[33];
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile + threadIdx.x * kScanPerThread;
  uint32_t vals[kScanPerThread];
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < kScanPerThread; ++j) {
    const int64_t i = base + j;
    vals[j] = (i < n) ? in[i] : 0u;
    v += vals[j];
  }
  uint32_t total;
  uint32_t run = block_exclusive_scan(v, s_warp, &total) + (tile_off ? tile_off[blockIdx.x] : 0u);
#pragma unroll
  for (int j = 0; j < kScanPerThread; ++j) {
    const int64_t i = base + j;
    if (i < n) out[i] = run;
    run += vals[j];
  }
  if (write_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = run;
}
}  // namespace

size_t scan_tmp_words(int64_t n) {
  // each level keeps its tile sums and their scan (tiles + tiles + 1 words)
  size_t words = 0;
  int64_t m = n;
  while (m > kScanTile) {
    const int64_t tiles = (m + kScanTile - 1) / kScanTile;
    words += 2 * static_cast<size_t>(tiles) + 1;
    m = tiles;
  }
  return words + 1;
}

cudaError_t scan_exclusive_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* tmp, cudaStream_t s,
                               int* n_launch) {
  if (n <= 0) {
    return cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
  }
  if (n <= kScanTile) {
    k_scan_tiles<<<1, kScanThreads, 0, s>>>(in, out, n, nullptr, 1);
    if (n_launch) *n_launch += 1;
    return cudaGetLastError();
  }
  if (n_launch) *n_launch += 2;
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  uint32_t* sums = tmp;
  uint32_t* sums_scanned = tmp + tiles;  // tiles + 1 words are reserved after the sums by scan_tmp_words
  k_scan_tile_sums<<<static_cast<int>(tiles), kScanThreads, 0, s>>>(in, n, sums);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  // recursive scan of the tile sums (into the space after them)
  err = scan_exclusive_u32(sums, sums_scanned, tiles, tmp + 2 * tiles + 1, s, n_launch);
  if (err != cudaSuccess) return err;
  k_scan_tiles<<<static_cast<int>(tiles), kScanThreads, 0, s>>>(in, out, n, sums_scanned, 1);
  return cudaGetLastError();
}

// =============================================================== layer index
namespace {

// The layer index in four launches and one memset, each bound by its launch and
// the latency of a few dependent loads (15 ELTs of 10,000 records over 2M ids:
// 37 us a build; 14 launches, with a scan for each of the three sums and a
// search for each record's ELT, took 94 us).  A slot's first pair follows from
// its word's pairs and the slots of the word before it, so the slots need no
// scan of their own, and the slots are an indexed pass's distinct events.
// Grids below: blockIdx.y is the ELT position, blockIdx.x strides over its records.

__global__ void k_mark_members(const __grid_constant__ LayerEltRefs r, uint32_t* bits, uint32_t* word_cnt) {
  const int p = blockIdx.y;
  const int32_t* ev = r.events[p];
  const int64_t n = r.rec_begin[p + 1] - r.rec_begin[p];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    const int32_t e = ev[i];
    atomicOr(&bits[e >> 5], 1u << (e & 31));
    atomicAdd(&word_cnt[e >> 5], 1u);  // every record is one (event, ELT) pair
  }
}

// slot_base and pair_base: exclusive sums over the words of the member events
// and of the records.  Block b sums the words before its own 1,024 itself (at
// most kBasesWords of them, from L2): one launch of 8 us for both sums at
// 62,500 words, where two scans took six launches and 23 us.
constexpr int kBasesThreads = 1024;
constexpr int64_t kBasesWords = 1 << 17;

__global__ void __launch_bounds__(kBasesThreads) k_word_bases(const uint32_t* __restrict__ bits,
                                                              const uint32_t* __restrict__ word_cnt, int64_t n_words,
                                                              uint32_t* slot_base, uint32_t* pair_base) {
  __shared__ uint32_t s_warp[33];
  uint32_t slots = 0u, pairs = 0u;
  const int64_t b0 = static_cast<int64_t>(blockIdx.x) * kBasesThreads;
#pragma unroll 4
  for (int64_t i = 4 * static_cast<int64_t>(threadIdx.x); i < b0; i += 4 * kBasesThreads) {
    const uint4 x = *reinterpret_cast<const uint4*>(bits + i), c = *reinterpret_cast<const uint4*>(word_cnt + i);
    slots += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
    pairs += c.x + c.y + c.z + c.w;
  }
  const int64_t w = b0 + threadIdx.x;
  const uint32_t my_slots = w < n_words ? __popc(bits[w]) : 0u, my_pairs = w < n_words ? word_cnt[w] : 0u;
  uint32_t before_slots, before_pairs, total;
  block_exclusive_scan(slots, s_warp, &before_slots);
  block_exclusive_scan(pairs, s_warp, &before_pairs);
  const uint32_t s = before_slots + block_exclusive_scan(my_slots, s_warp, &total);
  const uint32_t q = before_pairs + block_exclusive_scan(my_pairs, s_warp, &total);
  if (w < n_words) {
    slot_base[w] = s;
    pair_base[w] = q;
    if (w == n_words - 1) {
      slot_base[n_words] = s + my_slots;
      pair_base[n_words] = q + my_pairs;
    }
  }
}

__global__ void k_word_popc(const uint32_t* bits, int64_t n_words, uint32_t* cnt) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t w = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; w < n_words; w += stride)
    cnt[w] = __popc(bits[w]);
}

// Where the pairs of a member event e are: its word, and its rank in the word.
struct Place {
  uint32_t slot0, pair0, below;  // the word's first slot and pair, the word's events below e
  bool several;                  // the word holds an event with several pairs
};
__device__ __forceinline__ Place place_of(const uint32_t* __restrict__ bits, const uint32_t* __restrict__ slot_base,
                                          const uint32_t* __restrict__ pair_base, int32_t e) {
  const int32_t w = e >> 5;
  const uint32_t b = bits[w];
  Place pl;
  pl.slot0 = slot_base[w];
  pl.pair0 = pair_base[w];
  pl.below = __popc(b & ((1u << (e & 31)) - 1u));
  pl.several = pair_base[w + 1] - pl.pair0 != static_cast<uint32_t>(__popc(b));
  return pl;
}

__global__ void k_mark_positions(const __grid_constant__ LayerEltRefs r, const uint32_t* __restrict__ bits,
                                 const uint32_t* __restrict__ slot_base, const uint32_t* __restrict__ pair_base,
                                 unsigned long long* mask) {
  const int p = blockIdx.y;
  const int32_t* ev = r.events[p];
  const int64_t n = r.rec_begin[p + 1] - r.rec_begin[p];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) {
    const Place pl = place_of(bits, slot_base, pair_base, ev[i]);
    if (pl.several) atomicOr(&mask[pl.slot0 + pl.below], 1ull << p);
  }
}

// One word's rank-directory entry and its slots' first pairs and events.
__device__ __forceinline__ void fill_word(const LayerIndex& ix, int64_t w) {
  const uint32_t b = ix.bits[w], slot0 = ix.slot_base[w], pair0 = ix.pair_base[w];
  const uint32_t n = __popc(b), n_pairs = ix.pair_base[w + 1] - pair0;
  uint32_t y = pair0;
  if (n_pairs == n) {
    for (uint32_t i = 0; i < n; ++i) ix.slot_start[slot0 + i] = pair0 + i;
  } else {
    y = kRankSlots | slot0;
    uint32_t at = pair0, left = b;
    for (uint32_t i = 0; i < n; ++i) {
      const uint32_t c = __popcll(ix.mask[slot0 + i]);
      ix.slot_start[slot0 + i] = at;
      at += c;
      if (n_pairs == n + 1u && c == 2u && pair0 <= kRankBaseMask)
        y = kRankTwo | (static_cast<uint32_t>(__ffs(left) - 1) << kRankTwoShift) | pair0;
      left &= left - 1u;
    }
  }
  ix.rankdir[w] = make_uint2(b, y);
  if (ix.slot_event) {
    uint32_t left = b;
    for (uint32_t i = 0; i < n; ++i, left &= left - 1u)
      ix.slot_event[slot0 + i] = static_cast<int32_t>(32 * w + __ffs(left) - 1);
  }
  if (w == ix.n_words - 1) ix.slot_start[slot0 + n] = pair0 + n_pairs;
}

// The pairs in (event, position) order; the blocks of the last blockIdx.y fill
// the words' directory entries and slots.
__global__ void k_fill_pairs(const __grid_constant__ LayerEltRefs r, const __grid_constant__ LayerIndex ix) {
  const int p = blockIdx.y;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t i0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (p == r.n_elts) {
    for (int64_t w = i0; w < ix.n_words; w += stride) fill_word(ix, w);
    return;
  }
  const int32_t* ev = r.events[p];
  const Pair* recs = r.recs[p];
  const float2* wts = r.wts[p];
  const int64_t n = r.rec_begin[p + 1] - r.rec_begin[p];
  for (int64_t j = i0; j < n; j += stride) {
    const int32_t e = ev[j];
    Pair q = recs[j];
    const Place pl = place_of(ix.bits, ix.slot_base, ix.pair_base, e);
    uint32_t at = pl.pair0 + pl.below;
    if (pl.several) {
      at = pl.pair0;
      for (uint32_t k = 0; k < pl.below; ++k) at += __popcll(ix.mask[pl.slot0 + k]);
      at += __popcll(ix.mask[pl.slot0 + pl.below] & ((1ull << p) - 1ull));
    }
    q.meta = (q.meta & ~kMetaPosMask) | static_cast<uint32_t>(p);
    ix.pairs[at] = q;
    PairHot hq;
    hq.max_l = q.max_l;
    hq.mu = q.mu;
    hq.meta = q.meta;
    hq.node = pair_rec(q.meta) * (pair_fine(q.meta) ? kTabFineStride : kTabNodes);
    ix.hot[at] = hq;
    if (ix.pw && wts) ix.pw[at] = wts[j];
    if (ix.pev) ix.pev[at] = e;
  }
}

inline int grid_for(int64_t n, int threads, int cap = 4096) {
  const int64_t b = (n + threads - 1) / threads;
  return static_cast<int>(b < 1 ? 1 : (b > cap ? cap : b));
}

inline int64_t round4(int64_t n) { return (n + 3) & ~int64_t(3); }

}  // namespace

size_t index_marks_bytes(int64_t n_words, int64_t n_recs) {
  return sizeof(unsigned long long) * static_cast<size_t>((n_recs + 2) & ~int64_t(1)) +
         2 * sizeof(uint32_t) * static_cast<size_t>(round4(n_words));
}

void index_place_marks(LayerIndex& ix, void* marks) {
  ix.mask = static_cast<unsigned long long*>(marks);
  ix.bits = reinterpret_cast<uint32_t*>(ix.mask + ((ix.n_recs + 2) & ~int64_t(1)));
  ix.word_cnt = ix.bits + round4(ix.n_words);
  ix.marks_bytes = index_marks_bytes(ix.n_words, ix.n_recs);
}

size_t index_scan_words(int64_t n_words) { return n_words > kBasesWords ? scan_tmp_words(n_words) : 1; }

cudaError_t build_layer_index(const LayerEltRefs& refs, LayerIndex& ix, cudaStream_t s, int* n_launch) {
  const int64_t n_recs = refs.rec_begin[refs.n_elts];
  cudaError_t err;
  if ((err = cudaMemsetAsync(ix.mask, 0, ix.marks_bytes, s)) != cudaSuccess) return err;
  int launched = 0;
  int64_t longest = 0;
  for (int p = 0; p < refs.n_elts; ++p) {
    const int64_t n = refs.rec_begin[p + 1] - refs.rec_begin[p];
    longest = n > longest ? n : longest;
  }
  const dim3 by_elt(grid_for(longest, 256, 64), refs.n_elts);
  if (n_recs > 0) {
    k_mark_members<<<by_elt, 256, 0, s>>>(refs, ix.bits, ix.word_cnt);
    ++launched;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  if (ix.n_words <= kBasesWords) {
    k_word_bases<<<grid_for(ix.n_words, kBasesThreads), kBasesThreads, 0, s>>>(ix.bits, ix.word_cnt, ix.n_words,
                                                                              ix.slot_base, ix.pair_base);
    ++launched;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  } else {
    k_word_popc<<<grid_for(ix.n_words, 256), 256, 0, s>>>(ix.bits, ix.n_words, ix.slot_base);
    ++launched;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    // in place: each tile reads its inputs before writing
    if ((err = scan_exclusive_u32(ix.slot_base, ix.slot_base, ix.n_words, ix.scan_tmp, s, &launched)) != cudaSuccess ||
        (err = scan_exclusive_u32(ix.word_cnt, ix.pair_base, ix.n_words, ix.scan_tmp, s, &launched)) != cudaSuccess)
      return err;
  }
  if (n_recs > 0) {
    k_mark_positions<<<by_elt, 256, 0, s>>>(refs, ix.bits, ix.slot_base, ix.pair_base, ix.mask);
    ++launched;
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  k_fill_pairs<<<dim3(64, refs.n_elts + 1), 256, 0, s>>>(refs, ix);
  ++launched;
  if (n_launch) *n_launch += launched;
  return cudaGetLastError();
}

}  // namespace ara
