// device_common.cuh -- device helpers shared by the shot kernel and the
// adjoint kernel (complex arithmetic, packed keys, Philox4x32-10).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"

namespace soft {
namespace dev {

// Aligned to its size, so that both components move in one load or store of 8 or 16 bytes.
template <typename R>
struct alignas(2 * sizeof(R)) Cx {
  R x, y;
};
// Real arithmetic with fixed rounding: explicit round-to-nearest intrinsics, so that no
// product is contracted into a fused multiply-add differently in different kernels (the
// noiseless-run snapshots come from one kernel and must equal, bit for bit, what the shot
// kernels compute on the same events). A negated operand of a product or a fused
// multiply-add is an instruction modifier, not an operation.
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double addr(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float addr(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double subr(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float subr(float a, float b) { return __fsub_rn(a, b); }
// a b: each component one product and one fused multiply-add
template <typename R>
__device__ __forceinline__ Cx<R> cmul(Cx<R> a, Cx<R> b) {
  return {fmar(a.x, b.x, mulr(-a.y, b.y)), fmar(a.x, b.y, mulr(a.y, b.x))};
}
template <typename R>
__device__ __forceinline__ Cx<R> cadd(Cx<R> a, Cx<R> b) {
  return {addr(a.x, b.x), addr(a.y, b.y)};
}
template <typename R>
__device__ __forceinline__ Cx<R> csub(Cx<R> a, Cx<R> b) {
  return {subr(a.x, b.x), subr(a.y, b.y)};
}
template <typename R>
__device__ __forceinline__ Cx<R> cscale(Cx<R> a, R s) {
  return {mulr(a.x, s), mulr(a.y, s)};
}
// a v + b w as one chain of fused multiply-adds per component
template <typename R>
__device__ __forceinline__ Cx<R> cmad2(Cx<R> a, Cx<R> v, Cx<R> b, Cx<R> w) {
  return {fmar(a.x, v.x, fmar(-a.y, v.y, fmar(b.x, w.x, mulr(-b.y, w.y)))),
          fmar(a.x, v.y, fmar(a.y, v.x, fmar(b.x, w.y, mulr(b.y, w.x))))};
}
// -x by flipping the sign bit, for a negated value that is stored or selected rather than
// fed to an arithmetic instruction. For FP64 the flip is an explicit 32-bit xor of the
// high word in inline PTX: written as a plain negation (or a bit flip the compiler
// recognizes as one) it becomes a DADD on GB300's narrow FP64 pipe, which measured
// 0.91 G DADDs per 2^22 shots of the FP64 lane kernel, 22 % of its time.
__device__ __forceinline__ double negr(double x) {
  int hi = __double2hiint(x);
  const int lo = __double2loint(x);
  asm("xor.b32 %0, %0, 0x80000000;" : "+r"(hi));
  return __hiloint2double(hi, lo);
}
__device__ __forceinline__ float negr(float x) { return -x; }
// v * i^e
template <typename R>
__device__ __forceinline__ Cx<R> ipow(Cx<R> v, uint32_t e) {
  Cx<R> r = (e & 1u) ? Cx<R>{negr(v.y), v.x} : v;
  if (e & 2u) r = {negr(r.x), negr(r.y)};
  return r;
}
template <typename R>
__device__ __forceinline__ R norm2(Cx<R> v) {
  return fmar(v.x, v.x, mulr(v.y, v.y));
}

// The pruning test |v|^2 < tau, decided exactly as the norm computed in R decides it.
// FP64: when both |re| and |im| lie below sqrt(tau/2) (1 - 2^-18), or either lies above
// sqrt(tau) (1 + 2^-18), integer compares of their high words settle it (the computed
// norm's rounding cannot cross tau there); only values in that narrow band compute the
// norm on the FP64 pipe, GB300's narrowest.
template <typename R>
struct PruneTest {
  R tau;
  uint32_t lo = 0, hi = 0;  // high words of the two bounds above (FP64)
  __device__ explicit PruneTest(const PruneBounds &b) : tau((R)b.tau), lo(b.lo), hi(b.hi) {}
  __device__ __forceinline__ bool small(Cx<R> v) const {
    if (sizeof(R) == 4) return norm2(v) < tau;
    const uint32_t hx = (uint32_t)((unsigned long long)__double_as_longlong((double)v.x) >> 32) & 0x7FFFFFFFu;
    const uint32_t hy = (uint32_t)((unsigned long long)__double_as_longlong((double)v.y) >> 32) & 0x7FFFFFFFu;
    if (hx > hi || hy > hi) return false;
    if (hx < lo && hy < lo) return true;
    return norm2(v) < tau;
  }
};
// ---- scaled FP64 maps (the lane kernels and affine_kernel). The map's entries are
// e^{i phi} v / sqrt(N): a squared norm N per shot, and the circuit's global phase phi (pi/8
// times the event's ev_phase), which is the same in every shot and only needed when a state
// is read out. A rotation c I - i s Z is then v' = v - i (s / c) xi v_partner with N / c^2,
// two fused multiply-adds per entry instead of two complex products (eight operations), and
// a measurement keeps its outcome's sum as the new N instead of scaling every entry. GB300
// issues an FP64 instruction per 76 cycles and SM partition whatever its active lanes, and
// that pipe bounded every FP64 map (random 40-qubit circuit, 0.2 M shots: 2.9 -> 1.8 ms; w97,
// 0.5 M: 19.1 -> 17.8 ms; w42, 2^22: 12.5 -> 11.3 ms).
// The sign bit of a 64-bit float as a value to XOR into its high word.
__device__ __forceinline__ double xor_hi(double x, uint32_t flip) {
  return __hiloint2double((int)((uint32_t)__double2hiint(x) ^ flip), __double2loint(x));
}
// i^(eo) (-1)^neg k: what multiplies the two components of an entry's partner
struct ScaledTurn {
  double kx, ky;  // for the new re and im
  bool swap;      // odd eo: re takes the partner's im
  __device__ __forceinline__ ScaledTurn(double k, uint32_t eo)
      : kx(xor_hi(k, ((eo ^ (eo >> 1)) & 1u) << 31)), ky(xor_hi(k, (eo & 2u) << 30)), swap((eo & 1u) != 0u) {}
  // base + i^eo (-1)^neg k w
  __device__ __forceinline__ Cx<double> add(Cx<double> base, Cx<double> w, uint32_t neg) const {
    const double p = swap ? w.y : w.x, q = swap ? w.x : w.y;
    return {__fma_rn(xor_hi(kx, neg << 31), p, base.x), __fma_rn(xor_hi(ky, neg << 31), q, base.y)};
  }
};
// x >= 0 as a float, rounded toward zero to 21 bits (0 below 2^-125, inf from 2^126), without
// the FP64 pipe's conversion
__device__ __forceinline__ float low_float(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  return h < (898u << 20) ? 0.0f : h >= (1149u << 20) ? __uint_as_float(0x7F800000u) : __uint_as_float((h - (896u << 20)) << 3);
}
// The pruning test |v|^2 < tau N. The bounds of PruneTest, widened to 2^-16 and multiplied by
// sqrt(N) in FP32 (N truncated to 21 bits), are compared with the high words of |re| and
// |im|; only values between them compute the norm on the FP64 pipe.
struct ScaledPrune {
  double tau;
  float klo, khi;
  uint32_t lo = 0, hi = 0;
  __device__ explicit ScaledPrune(const PruneBounds &b) : tau(b.tau), klo(b.klo), khi(b.khi) {}
  __device__ __forceinline__ void set(double N) {  // N in range
    const float n = low_float(N), r = n * rsqrtf(n);
    lo = (__float_as_uint(klo * r) >> 3) + (896u << 20);
    hi = (__float_as_uint(khi * r) >> 3) + (896u << 20) + 1u;
  }
  __device__ __forceinline__ bool small(Cx<double> v, double N) const {
    const uint32_t hx = (uint32_t)__double2hiint(v.x) & 0x7FFFFFFFu, hy = (uint32_t)__double2hiint(v.y) & 0x7FFFFFFFu;
    if (hx > hi || hy > hi) return false;
    if (hx < lo && hy < lo) return true;
    return norm2(v) < mulr(tau, N);
  }
  // N within [2^-64, 2^96]: outside, the entries take the factor fit(N) (a power of two:
  // exact) and N its square
  __device__ __forceinline__ static bool in_range(double N) {
    const uint32_t h = (uint32_t)__double2hiint(N);
    return h >= ((1023u - 64u) << 20) && h < ((1023u + 96u) << 20);
  }
  __device__ __forceinline__ static double fit(double N) { return N > 1.0 ? 0x1p-32 : 0x1p32; }
};
// e^{i pi ph / 8}
__device__ __forceinline__ Cx<double> phase_of(uint32_t ph) {
  double s, c;
  sincospi(0.125 * (double)ph, &s, &c);
  return {c, s};
}

// e^{i pi ph / 8} / sqrt(N): what multiplies a scaled map's entries when they are read out
__device__ __forceinline__ Cx<double> readout(uint32_t ph, double N) { return cscale(phase_of(ph), rsqrt(N)); }

template <typename R>
__device__ __forceinline__ double norm2d(Cx<R> v) {
  const double a = (double)v.x, b = (double)v.y;
  return __fma_rn(a, a, __dmul_rn(b, b));
}
// |v|^2 as it enters the FP64 probability sums of a measurement: computed in FP64 for FP64
// maps; for FP32 maps computed in FP32 (its rounding, 2^-24 relative, is that of the
// coefficients themselves) and widened, which keeps two conversions and two FP64 products
// per entry off GB300's narrow FP64 pipe (w42 FP32: 622 -> 660 M shots/s). The sums stay FP64.
template <typename R>
__device__ __forceinline__ double pnorm(Cx<R> v) {
  if (sizeof(R) == 4) return (double)norm2(v);
  return norm2d(v);
}

// Parity of the set bits of a 64-bit word: the halves are folded first, so that one 32-bit
// population count (a quarter-rate instruction at best) serves instead of two.
__device__ __forceinline__ uint32_t wordpar(uint64_t x) {
  return (uint32_t)__popc((uint32_t)x ^ (uint32_t)(x >> 32)) & 1u;
}
// Bytes (4, 8 or 16) from global to shared memory without passing through registers; the
// thread's own copies are complete after copies_done().
template <int Bytes>
__device__ __forceinline__ void copy_async(void *shared, const void *global) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(shared)),
               "l"(global), "n"(Bytes)
               : "memory");
}
// A hint to bring the line that holds global address p into L1.
__device__ __forceinline__ void prefetch_line(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }
// For a warp that walks the events on its own (the noiseless runs): event `ev` is next. Once per
// 32 events the lanes ask for the ones after the next 32, an event each, and for the coefficients
// and case-B constants of those, so that the walk finds them in L1: the loads of a lone warp were
// a third of its time (with cold caches, w42's noiseless run in FP64 454 -> 389 us, the
// gradient's 404 -> 329; the events alone gained nothing, each case-B measurement's constants
// were the long waits).
template <int W>
__device__ __forceinline__ void prefetch_events(const Ev<W> *evs, const Coef *coef, const CaseB *cb, uint32_t ev, uint32_t n_events, uint32_t lane) {
  if (ev & 31u) return;
  for (uint32_t k = ev ? ev + 32u + lane : lane; k < n_events && k < ev + 64u; k += 32) {
    const unsigned char *q = reinterpret_cast<const unsigned char *>(evs + k);
    prefetch_line(q);
    prefetch_line(q + sizeof(Ev<W>) - 16);
    const uint32_t type = ev_type(__ldg(&evs[k].w0));
    if (type == EV_ROT || type == EV_ROT_DIAG) prefetch_line(coef + __ldg(&evs[k].a));
    if (type == EV_MEAS_B) {
      const unsigned char *c = reinterpret_cast<const unsigned char *>(cb + (uint32_t)__ldg(&evs[k].beta[0]));
      for (uint32_t o = 0; o < sizeof(CaseB); o += 128) prefetch_line(c + o);
      prefetch_line(c + sizeof(CaseB) - 16);
    }
  }
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int W>
struct Key {
  uint64_t w[W];
};
template <int W>
__device__ __forceinline__ Key<W> kxor(const Key<W> &a, const uint64_t *b) {
  Key<W> r;
#pragma unroll
  for (int i = 0; i < W; ++i) r.w[i] = a.w[i] ^ b[i];
  return r;
}
template <int W>
__device__ __forceinline__ uint32_t kpar(const Key<W> &a, const uint64_t *b) {
  uint64_t t = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) t ^= a.w[i] & b[i];
  return wordpar(t);
}
template <int W>
__device__ __forceinline__ bool keq(const Key<W> &a, const Key<W> &b) {
  bool e = true;
#pragma unroll
  for (int i = 0; i < W; ++i) e = e && (a.w[i] == b.w[i]);
  return e;
}
// word (i >> 6) of a W-word vector without dynamic register indexing
template <int W>
__device__ __forceinline__ uint64_t word_of(const uint64_t *a, uint32_t i) {
  return (W == 1 || (i >> 6) == 0u) ? a[0] : a[W - 1];
}
template <int W>
__device__ __forceinline__ uint32_t kbit(const Key<W> &a, uint32_t i) {
  return (uint32_t)((word_of<W>(a.w, i) >> (i & 63)) & 1ull);
}
template <int W>
__device__ __forceinline__ uint32_t khash(const Key<W> &a) {
  uint64_t h = a.w[0];
  if (W == 2) h ^= a.w[W - 1] * 0xC2B2AE3D27D4EB4Full;
  h *= 0x9E3779B97F4A7C15ull;
  return (uint32_t)(h >> 32);
}
template <int W>
__device__ __forceinline__ uint32_t wpar(const uint64_t *a, const uint64_t *b) {
  uint64_t t = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) t ^= a[i] & b[i];
  return wordpar(t);
}
// parity of a . b + c . d over GF(2)
template <int W>
__device__ __forceinline__ uint32_t wpar2(const uint64_t *a, const uint64_t *b, const uint64_t *c, const uint64_t *d) {
  uint64_t t = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) t ^= (a[i] & b[i]) ^ (c[i] & d[i]);
  return wordpar(t);
}
template <int W>
__device__ __forceinline__ uint32_t wbit(const uint64_t *a, uint32_t i) {
  return (uint32_t)((word_of<W>(a, i) >> (i & 63)) & 1ull);
}
// The lowest set bit of a nonzero W-word vector (64 W for zero). A reversal and a leading-zero
// count: with __ffsll(x) - 1 here a build of affine.cu failed the random-circuit tests, and a
// print in a scratch copy of it showed -1 beside a residual of 8. Why was not found.
template <int W>
__device__ __forceinline__ uint32_t wlow(const uint64_t *x) {
  const bool first = W == 1 || x[0] != 0ull;
  return (first ? 0u : 64u) + (uint32_t)__clzll((long long)__brevll(first ? x[0] : x[W - 1]));
}
template <int W>
__device__ __forceinline__ void wflip(uint64_t *a, uint32_t i) {
#pragma unroll
  for (int w = 0; w < W; ++w)
    if ((int)(i >> 6) == w) a[w] ^= 1ull << (i & 63);
}

// Philox4x32-10, counter (shot_lo, shot_hi, stream, index), key = seed. Rolled: the
// round loop is not unrolled, for kernels whose instruction fetch limits them (the lane
// kernel: 3.6 % faster on w42 FP32); same values.
template <bool Rolled = false>
__device__ __forceinline__ uint4 philox(uint64_t seed, uint64_t shot, uint32_t stream, uint32_t idx) {
  uint32_t c0 = (uint32_t)shot, c1 = (uint32_t)(shot >> 32), c2 = stream, c3 = idx;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll (Rolled ? 1 : 10)
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  return make_uint4(c0, c1, c2, c3);
}



}  // namespace dev
}  // namespace soft
