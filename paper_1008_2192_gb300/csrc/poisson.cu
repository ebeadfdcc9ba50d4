// The POISSON work function (declarations and contract in include/crb.h).
//
// CRBLASTER measures the cost of its own framework by swapping L.A.Cosmic for
// a work function with an equal, known load per pixel and no overlap regions
// (Sec. 6.3.2): each output pixel is a Poisson deviate whose mean is the input
// pixel, drawn with Knuth's multiplicative method (Algorithm Q, Seminumerical
// Algorithms Sec. 3.4.1): uniforms are multiplied until the product falls
// below e^-mu, and the number of factors taken before that is the deviate.
// Its cost grows linearly with mu.
//
// One thread per pixel over all frames of a call. The uniforms come from
// SplitMix64 (Steele, Lea and Flood 2014) used as a counter-based generator,
// so a pixel's draws depend only on its frame's seed, its index and the draw
// number: value(s, j) = mix13(s + (j + 1) * gamma); pixel p draws from the
// stream keyed by value(seed, p), its j-th uniform being the top 53 bits of
// value(key, j) times 2^-53. e^-mu is formed by fixed IEEE double steps
// (Cody-Waite reduction -mu = n ln2 + r, the Taylor polynomial of e^r to
// degree 13 by Horner's rule, scaling by 2^n), with the rounded operations
// spelled out so that no multiply-add is fused; the comparisons q >= e^-mu are
// therefore those of any implementation that takes the same steps (a product
// in float decides all but the closest of them, see poisson_kernel). mu <= 0 or
// NaN gives 0, mu above 700 is taken as 700, and at most 4096 factors are
// drawn, which bounds every thread's loop.

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>

#include "crb.h"

void crb_detail_set_error(const char* msg);  // crb.cu

namespace {

constexpr uint64_t kGamma = 0x9e3779b97f4a7c15ULL;
constexpr double kMuMax = 700.0;
constexpr int kQMax = 4096;
constexpr int kPThreads = 128;
constexpr int kFramesPerLaunch = 256;  // the frame table travels in the launch parameters

struct PFrame {
  const float* in;
  float* out;
  long long pix0;  // first pixel of the frame in the launch's pixel index
  uint64_t seed;
};

struct PLaunch {
  PFrame f[kFramesPerLaunch];
  int n;
  long long total;
  double c[14];  // 1/i!
  double ln2_hi, ln2_lo, inv_ln2;
};

__device__ __forceinline__ uint64_t mix13(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t stream_value(uint64_t s, uint64_t j) { return mix13(s + (j + 1) * kGamma); }

// (v >> 11) * 2^-53, built from its bits with integer operations (the value
// is exact either way): the FP64 pipe is left to the product.
__device__ __forceinline__ double uniform53(uint64_t v) {
  const uint64_t m = v >> 11;
  if (m == 0) return 0.0;
  const int e = 63 - __clzll((long long)m);  // top bit of m, 0 .. 52
  const uint64_t frac = (m << (52 - e)) & ((uint64_t(1) << 52) - 1);
  return __longlong_as_double((long long)((uint64_t(e - 53 + 1023) << 52) | frac));
}

__device__ __forceinline__ double exp_neg(double mu, const PLaunch& P) {
  const double x = -mu;
  const double n = rint(__dmul_rn(x, P.inv_ln2));
  const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(n, P.ln2_hi)), __dmul_rn(n, P.ln2_lo));
  double p = P.c[13];
#pragma unroll
  for (int i = 12; i >= 0; --i) p = __dadd_rn(__dmul_rn(p, r), P.c[i]);
  return ldexp(p, int(n));
}

// The deviate of pixel p by the defining steps in double: every product and
// comparison as stated in the header. After the first draw eight at a time, their
// uniforms ahead of the chain of products, which fall monotonically: a product
// above e^-mu has none below it before. One pixel's chain holds up a small image's call
// (64 x 64 of mean 690, 3 such pixels: 121 us with one draw at a time, so 97).
__device__ __noinline__ int deviate_exact(float mean, uint64_t key, const PLaunch& P) {
  // q and e^-mu are non-negative doubles, which order as their bit patterns
  const long long L = __double_as_longlong(exp_neg(fmin(double(mean), kMuMax), P));
  auto draw = [&](int j) { return uniform53(mix13(key + uint64_t(j + 1) * kGamma)); };
  double q = draw(0);
  if (__double_as_longlong(q) < L) return 0;
  for (int k = 1; k < kQMax; k += 8) {
    double u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) u[i] = draw(k + i);
    double q8 = q;
#pragma unroll
    for (int i = 0; i < 8; ++i) q8 = __dmul_rn(q8, u[i]);
    if (__double_as_longlong(q8) >= L) {
      q = q8;
      continue;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      q = __dmul_rn(q, u[i]);
      if (__double_as_longlong(q) < L) return min(k + i, kQMax);
    }
  }
  return kQMax;
}

// hi * 2^-32 in float, rounded once: the top 23 bits and the low 9 as
// significands of 2^23 + x, so that no conversion instruction is needed (they
// run on the FP64 pipe here: 2 lanes per clock and SM).
__device__ __forceinline__ float unit_float(uint32_t hi) {
  const float a = __fsub_rn(__uint_as_float(__funnelshift_r(hi, 0x96u, 9)), 0x1p23f);  // hi >> 9, exact
  const float b = __fmaf_rn(__uint_as_float((hi & 511u) | 0x4b000000u), 0x1p-32f, -0x1p-9f);  // exact
  return __fmaf_rn(a, 0x1p-23f, b);
}

// The state after mix13's second product: its top 32 bits are those of the
// output but for the lowest, since the last XOR (by z >> 31) moves the high word
// by one at most.
__device__ __forceinline__ uint64_t mix_head(uint64_t s) {
  const uint64_t z = (s ^ (s >> 30)) * 0xbf58476d1ce4e5b9ULL;
  return (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
}

// The uniform of a draw in float, with a relative error below 3 * 2^-24 against
// the 53-bit one: 2^-24 of the rounding and 2/hi of the bits left out, where
// the 32 bits taken (hi) are at least 2^24. kSmall: the top word is less (one
// draw in 256); then the 32 bits eight places further down, with the same
// bound, or for a still smaller value the whole output.
template <bool kSmall>
__device__ __forceinline__ float uniform_approx(uint64_t z) {
  const uint32_t hi = uint32_t(z >> 32);
  if (!kSmall || hi >= (1u << 24)) return unit_float(hi);
  const uint32_t w = uint32_t(z >> 24);
  if (w >= (1u << 24)) return unit_float(w) * 0x1p-8f;
  return __ull2float_rn((z ^ (z >> 31)) >> 11) * 0x1p-53f;
}

// The defining steps decide only where the running product falls below e^-mu,
// so the product is first taken in float with a bound on its relative error:
// 4 * 2^-24 per factor (the uniform above and the rounded product), and 2^-20
// for e^-mu in float. Only where the product lands within that bound of e^-mu
// (about 4e-5 of the pixels at mu = 24) is the pixel drawn again in double
// (deviate_exact); the deviates are the same bits.
// What bounds it: the ALU pipe (69 % active, issue 76 %), the shifts, XORs and
// 64-bit products of each draw's mix, and the lanes of a warp that wait for its
// longest draw (22.5 of 32 active). The form that multiplied in double was bound
// by the FP64 pipe (2 lanes per clock and SM, 81 % active): 94.2 us on a 750x750
// image of mean 24.3, against 31.1 us (with an integer-to-float conversion
// instruction, which runs on the FP64 pipe too, 47.8 us), and 29.7 launched ahead of time. Two draws per step with
// one comparison: the products fall monotonically, so the second one alone
// tells whether to go on.
// mu > 60, where e^-mu leaves float's range: the product is scaled up by 2^64
// each time it falls below 2^-64, until the rest of e^-mu lies above 2^-90.
// Launched while the kernel ahead of it on the stream runs; it waits for that one's results first.
__global__ void __launch_bounds__(kPThreads) poisson_kernel(const __grid_constant__ PLaunch P) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < P.total;
       t += (long long)gridDim.x * blockDim.x) {
    int lo = 0, hi = P.n - 1;  // frame of pixel t
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (P.f[mid].pix0 <= t) lo = mid; else hi = mid - 1;
    }
    const PFrame& f = P.f[lo];
    const long long p = t - f.pix0;
    const float mean = __ldg(f.in + p);
    int k = 0;
    if (mean > 0.f) {
      const float mu = fminf(mean, float(kMuMax));
      const uint64_t key = stream_value(f.seed, uint64_t(p));
      // e^-mu = 2^-e * m, m in [2^-0.5, 2^0.5]: mu * log2(e) in two floats
      constexpr float kLog2eHi = 1.44269502f, kLog2eLo = 1.92596299e-8f;
      const float h = __fmul_rn(mu, kLog2eHi);
      const float l = __fmaf_rn(mu, kLog2eHi, -h) + mu * kLog2eLo;
      const float n = rintf(h);
      const float m = exp2f(-((h - n) + l));
      int e = int(n);
      const int kmax = int(2.f * mu) + 64;  // factors the error bound below allows for
      const float delta = float(kmax + 16) * 0x1p-22f;
      const float mhi = m * (1.f + delta), mlow = m * (1.f - delta);
      uint64_t ctr = key;
      float q = 1.f, q1 = 1.f, thr;
      bool exact = false;
      for (;;) {
        const bool last = e <= 90;
        thr = last ? mhi * __int_as_float((127 - e) << 23) : 0x1p-64f;
        // two tiny factors in a row: the product below the threshold already, or before its scaling below 2^-126,
        // where float loses bits that the error bound does not count
        if (q < fmaxf(thr, 0x1p-62f)) {
          exact = true;
          break;
        }
        for (;;) {
          const uint64_t z1 = mix_head(ctr + kGamma);
          ctr += 2 * kGamma;
          const uint64_t z2 = mix_head(ctr);
          float u1 = uniform_approx<false>(z1), u2 = uniform_approx<false>(z2);
          if (min(uint32_t(z1 >> 32), uint32_t(z2 >> 32)) < (1u << 24)) {
            u1 = uniform_approx<true>(z1);
            u2 = uniform_approx<true>(z2);
          }
          q1 = q * u1;
          q = q1 * u2;
          if (q < thr || k >= kmax) break;
          k += 2;
        }
        if (last || k >= kmax) break;
        k += 2;
        q *= 0x1p64f;
        e -= 64;
      }
      // the factor that crossed: the first of the pair unless q1 is still above
      const bool first = q1 < thr;
      const float qc = first ? q1 : q, low = mlow * __int_as_float((127 - e) << 23);
      k += first ? 0 : 1;
      if (exact || k >= kmax || qc >= low) k = deviate_exact(mean, key, P);
    }
    f.out[p] = float(k);
  }
}

int fail(int code, const std::string& msg) {
  crb_detail_set_error(msg.c_str());
  return code;
}

// The constants of exp_neg, by the same steps on the host: ln2 rounded to
// double, its high part with the low 20 significand bits cleared (n * ln2_hi is
// exact for |n| < 2^20), the remainder, and 1/i! by repeated division.
void fill_constants(PLaunch& P) {
  const double ln2 = 0.693147180559945309417232121458;
  uint64_t bits;
  std::memcpy(&bits, &ln2, 8);
  bits &= ~((uint64_t(1) << 20) - 1);
  std::memcpy(&P.ln2_hi, &bits, 8);
  P.ln2_lo = ln2 - P.ln2_hi;
  P.inv_ln2 = 1.0 / ln2;
  P.c[0] = 1.0;
  for (int i = 1; i < 14; ++i) P.c[i] = P.c[i - 1] / double(i);
}

int launch(PLaunch& P, cudaStream_t stream) {
  // a pixel per thread: blocks that draw long are balanced by the blocks still to start
  const long long blocks = std::min<long long>((P.total + kPThreads - 1) / kPThreads, 1 << 22);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(std::max<long long>(blocks, 1)));
  cfg.blockDim = dim3(kPThreads);
  cfg.stream = stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, poisson_kernel, P);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(CRB_ECUDA, std::string("crb_poisson launch: ") + cudaGetErrorString(e));
  return CRB_OK;
}

}  // namespace

extern "C" int crb_poisson_batch(int n, const float* const* imgs, const int* ws, const int* hs, const uint64_t* seeds,
                                 float* const* outs, cudaStream_t stream) {
  if (n < 0 || (n > 0 && (!imgs || !ws || !hs || !seeds || !outs)))
    return fail(CRB_EINVAL, "crb_poisson_batch: invalid batch arrays");
  for (int i = 0; i < n; ++i) {
    if (ws[i] < 1 || hs[i] < 1 || (long long)ws[i] * hs[i] >= (1LL << 31))
      return fail(CRB_EINVAL, "crb_poisson_batch: frame " + std::to_string(i) + ": sizes");
    if (!imgs[i] || !outs[i]) return fail(CRB_EINVAL, "crb_poisson_batch: frame " + std::to_string(i) + ": null");
  }
  PLaunch P;  // about 8 KB, passed by value in the launch parameters
  for (int a = 0; a < n; a += kFramesPerLaunch) {
    const int m = std::min(kFramesPerLaunch, n - a);
    fill_constants(P);
    P.n = m;
    P.total = 0;
    for (int i = 0; i < m; ++i) {
      const long long px = (long long)ws[a + i] * hs[a + i];
      P.f[i] = PFrame{imgs[a + i], outs[a + i], P.total, seeds[a + i]};
      P.total += px;
    }
    const int rc = launch(P, stream);
    if (rc) return rc;
  }
  return CRB_OK;
}

extern "C" int crb_poisson(const float* img, int w, int h, uint64_t seed, float* out, cudaStream_t stream) {
  if (!img || !out) return fail(CRB_EINVAL, "crb_poisson: null image or output pointer");
  const float* const imgs[1] = {img};
  float* const outs[1] = {out};
  return crb_poisson_batch(1, imgs, &w, &h, &seed, outs, stream);
}
