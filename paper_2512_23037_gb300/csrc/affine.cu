// affine.cu -- shot kernel with one warp per shot and the coefficient map in affine form.
//
// It runs the shots that lanes cannot hold: those whose maps outgrow a lane (from the
// lane's hand-over record, or again from their start), and the circuits whose noiseless
// maps have no lane size. The map is the lane kernel's cube (see lanes.cu): slot s of 2^d
// holds the value of key alpha0 ^ XOR over the set bits k of s of B[k], zero where no entry
// lives (a live entry is never zero: pruning drops |v|^2 < tau). What a lane does with
// loops over its rows and slots, a warp does at once: lane k keeps B[k] and its dual D[k]
// in registers, so that the parities of a vector with the whole basis are one population
// count and one ballot, its coordinates another, and its residual a warp-wide XOR
// reduction; the values are in shared memory, a pair of slots per lane and step. No key is
// stored or searched. The sparse form's hash index, of 4 slots per entry, its probes and
// its rebuilds after each pruning made the warp-per-shot kernel of kernels.cu 3 to 6 times
// slower on these shots.
//
// A map whose live entries span P.aff_dim directions, however many they are, goes at the next
// rotation that adds one to the pass at the circuit's cap, which runs it from its start with the
// sparse form of kernels.cu. The arithmetic is the lane kernel's, product by product, in both
// precisions: which shots come here from a lane depends on the order of claims and on which warps
// end first, and no entry may depend on that. Only the FP64 sums over a map's entries run in
// another order, since this kernel packs a map into fewer slots sooner (their last bit).
#include <type_traits>

#include "device_common.cuh"
#include "kernels.cuh"
#include "shot_common.cuh"

namespace soft {
namespace {

using namespace dev;

enum : int { AS_RUN = -1, AS_KEPT = 0, AS_DISC = 1, AS_OVF = 2, AS_ERR = 3, AS_RERUN = 4 };
constexpr uint32_t kAll = 0xFFFFFFFFu;
constexpr int kAffBlock = 128;
constexpr uint32_t kAffRecWords = 32;  // lane w keeps record word w (a circuit has at most 16)

// events held ahead of a warp in shared memory
constexpr uint32_t kRing = 4;
template <typename R, int W>
__host__ __device__ constexpr size_t aff_warp_bytes(uint32_t dim) {
  return (sizeof(Cx<R>) << dim) + kRing * sizeof(Ev<W>);
}

__device__ __forceinline__ uint64_t shfl64(uint64_t x, uint32_t src) {
  return (uint64_t)__shfl_sync(kAll, (unsigned long long)x, (int)src);
}
// XOR over the lanes of x
__device__ __forceinline__ uint64_t xor_all(uint64_t x) {
  return (uint64_t)__reduce_xor_sync(kAll, (uint32_t)x) | ((uint64_t)__reduce_xor_sync(kAll, (uint32_t)(x >> 32)) << 32);
}
// Both sums over the lanes: the halves of the warp trade one of them first, so that one
// chain of additions carries both (6 FP64 additions instead of 10).
__device__ __forceinline__ void sum_both(double &a, double &b) {
  const bool up = (threadIdx.x & 16u) != 0u;
  double x = (up ? b : a) + __shfl_xor_sync(kAll, up ? a : b, 16);
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(kAll, x, off);
  a = __shfl_sync(kAll, x, 0);
  b = __shfl_sync(kAll, x, 16);
}
// acc + |v|^2 as it enters a probability: FP32 norms widened (see pnorm), FP64 fused
__device__ __forceinline__ double addn(double acc, Cx<float> v) { return acc + pnorm(v); }
__device__ __forceinline__ double addn(double acc, Cx<double> v) { return __fma_rn(v.x, v.x, __fma_rn(v.y, v.y, acc)); }
__device__ __forceinline__ uint32_t par32(uint32_t x) { return (uint32_t)__popc(x) & 1u; }
// i with a zero bit inserted at position q
__device__ __forceinline__ uint32_t open_bit(uint32_t i, uint32_t q) {
  const uint32_t lo = (1u << q) - 1u;
  return (i & lo) | ((i & ~lo) << 1);
}

template <typename R, int W>
struct AffShot {
  const ShotParams &P;
  const CircDev *C = nullptr;
  const uint32_t lane;
  Cx<R> *v;             // 2^aff_dim values (shared memory)
  unsigned char *ring;  // kRing events (shared memory)
  uint64_t B[W], D[W];  // lane k < d: direction k and its dual; 0 in the other lanes
  uint64_t a0[W];       // alpha0 (every lane)
  uint64_t recw;        // lane w: record word w
  uint64_t shot;
  uint64_t sd[W], ss[W];
  uint32_t d;
  NoiseCursor nc;
  int status, chain, logical, lastm;
  double fid;
  bool force;
  static constexpr bool kScaled = sizeof(R) == 8;  // FP64 maps are scaled (see ScaledPrune)
  double nrm = 1.0;                                // their squared norm
  typename std::conditional<kScaled, ScaledPrune, PruneTest<R>>::type pt;  // |v|^2 < tau

  __device__ AffShot(const ShotParams &p, unsigned char *base)
      : P(p), lane(threadIdx.x & 31u), v(reinterpret_cast<Cx<R> *>(base)), ring(base + (sizeof(Cx<R>) << p.aff_dim)), pt(p.prune) {}
  // x, or zero where it is below tau
  __device__ __forceinline__ Cx<R> pruned(Cx<R> x) const {
    bool sm;
    if constexpr (kScaled) sm = pt.small(x, nrm);
    else sm = pt.small(x);
    return sm ? Cx<R>{0, 0} : x;
  }

  __device__ __forceinline__ uint32_t size() const { return 1u << d; }
  __device__ __forceinline__ static bool nonzero(const Cx<R> &x) { return x.x != (R)0 || x.y != (R)0; }

  // bit k: g . B[k]; g0: g . alpha0
  __device__ __forceinline__ uint32_t parities(const uint64_t *g, uint32_t &g0) const {
    g0 = wpar<W>(a0, g);
    return __ballot_sync(kAll, wpar<W>(B, g) != 0u);
  }
  // coordinates of x (bit k: D[k] . x) and its residual, zero iff x lies in the span
  __device__ __forceinline__ uint32_t coords(const uint64_t *x, uint64_t *r) const {
    const bool in = wpar<W>(D, x) != 0u;
#pragma unroll
    for (int w = 0; w < W; ++w) r[w] = x[w] ^ xor_all(in ? B[w] : 0ull);
    return __ballot_sync(kAll, in);
  }
  __device__ __forceinline__ static bool wnonzero(const uint64_t *x) { return (x[0] | x[W - 1]) != 0ull; }
  // the vector z with z . B[k] = 0 for every k and z . r = 1, for a residual r
  __device__ __forceinline__ void co_dual(const uint64_t *r, uint64_t *z) const {
    const uint32_t p = wlow<W>(r);
    const bool in = wbit<W>(B, p) != 0u;
#pragma unroll
    for (int w = 0; w < W; ++w)
      z[w] = xor_all(in ? D[w] : 0ull) ^ (((int)(p >> 6) == w) ? (1ull << (p & 63u)) : 0ull);
  }
  // B[d] = r (a residual: D[k] . r = 0 for k < d)
  __device__ __forceinline__ void add_dim(const uint64_t *r) {
    uint64_t z[W];
    co_dual(r, z);
    if (lane == d) {
#pragma unroll
      for (int w = 0; w < W; ++w) {
        B[w] = r[w];
        D[w] = z[w];
      }
    }
    ++d;
  }
  // Every live slot s has parity(s & g) = t, and g's highest bit is q: drop coordinate q
  // (alpha0 ^= t B[q], B[k] ^= B[q] for the other k of g; the other duals stay dual). The
  // values, scaled by sc (1: as they are), move to the slots without bit q; scaled values
  // below tau become zero.
  __device__ void remove_dim(uint32_t q, uint32_t g, uint32_t t, bool scaled, R sc) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint64_t bq = shfl64(B[w], q);
      if (t) a0[w] ^= bq;
      if (lane != q && ((g >> lane) & 1u)) B[w] ^= bq;
      const uint32_t src = lane < q || lane == 31u ? lane : lane + 1u;  // (lane 31 holds no row: d <= 31)
      B[w] = shfl64(B[w], src);
      D[w] = shfl64(D[w], src);
    }
    --d;
    const uint32_t n = size();
#pragma unroll 1
    for (uint32_t b = 0; b < n; b += 32) {  // sources lie at or above their targets, chunk by chunk
      const uint32_t s2 = b + lane;
      Cx<R> x{0, 0};
      if (s2 < n) {
        uint32_t s = open_bit(s2, q);
        s |= (par32(s & g) ^ t) << q;
        x = v[s];
        if (scaled) {
          x = pruned(cscale(x, sc));
        }
      }
      __syncwarp();
      if (s2 < n) v[s2] = x;
    }
    __syncwarp();
  }
  // One coordinate that the live slots' affine span does not need, if there is one: the
  // constraints g (lane k's candidate) that every difference of two live slots satisfies
  // are found by elimination, a violating slot per dropped candidate. False if none is left.
  __device__ bool compact_one(uint32_t &gl, uint32_t &g0) {
    uint32_t s0 = 0;
    bool found = false;
    for (uint32_t b = 0; b < size() && !found; b += 32) {
      const uint32_t m = __ballot_sync(kAll, b + lane < size() && nonzero(v[b + lane]));
      if (m) {
        s0 = b + (uint32_t)__ffs(m) - 1u;
        found = true;
      }
    }
    uint32_t G = lane < d ? 1u << lane : 0u;
    for (uint32_t k = 0; k < d; ++k) {
      const uint32_t g = __shfl_sync(kAll, G, (int)k);
      const uint32_t t = par32(s0 & g);
      uint32_t x = kAll;
      for (uint32_t b = 0; b < size(); b += 32) {
        const uint32_t s = b + lane;
        const uint32_t m = __ballot_sync(kAll, s < size() && par32(s & g) != t && nonzero(v[s]));
        if (m) {
          x = b + (uint32_t)__ffs(m) - 1u;
          break;
        }
      }
      if (x == kAll) {
        const uint32_t q = 31u - __clz(g), lo = (1u << q) - 1u;
        if ((gl >> q) & 1u) {  // the parities follow the rows
          gl ^= g & lo;
          g0 ^= t;
        }
        gl = (gl & lo) | ((gl >> (q + 1u)) << q);
        remove_dim(q, g, t, false, (R)1);
        return true;
      }
      if (lane > k && par32((x ^ s0) & G)) G ^= g;
    }
    return false;
  }
  // live slots, and the last of them
  __device__ uint32_t live_count(uint32_t *last = nullptr) const {
    uint32_t n = 0;
    for (uint32_t b = 0; b < size(); b += 32) {
      const uint32_t m = __ballot_sync(kAll, b + lane < size() && nonzero(v[b + lane]));
      n += __popc(m);
      if (last && m) *last = b + 31u - __clz(m);
    }
    return n;
  }
  // Before the map grows: where half the slots or more are empty, drop the coordinates that the
  // live ones do not need. Rotations that undo earlier ones (the T^dag after a T) leave such
  // maps, down to a single entry; compacting only at the map's limit left 75 slots on average
  // on w97 where 30 do. True if a coordinate went (coordinates and residuals are then stale).
  __device__ bool compact(uint32_t &gl, uint32_t &g0) {
    if (d < 3u) return false;
    uint32_t s0 = 0;
    const uint32_t n = live_count(&s0);
    if (n > (size() >> 1) && d < P.aff_dim) return false;
    if (n == 1u) {  // one entry: alpha0 takes its key
#pragma unroll
      for (int w = 0; w < W; ++w) {
        a0[w] ^= xor_all(((s0 >> lane) & 1u) ? B[w] : 0ull);
        B[w] = D[w] = 0ull;
      }
      g0 ^= par32(s0 & gl);
      gl = 0;
      d = 0;
      if (s0 && lane == 0) v[0] = v[s0];
      __syncwarp();
      return true;
    }
    bool any = false;
    while (compact_one(gl, g0)) any = true;
    return any;
  }

  __device__ void fail_check(uint32_t code, uint64_t value) {
    status = AS_ERR;
    if (lane == 0 && P.diag && atomicAdd(&P.diag[0], 1ull) == 0ull) {
      P.diag[1] = ((unsigned long long)code << 32);
      P.diag[2] = shot;
      P.diag[3] = value;
    }
  }
  __device__ __forceinline__ int pick(uint32_t ord, double sp, double sm) {
    return pick_outcome<false>(P.seed, shot, ord, sp, sm, force, fid, nullptr);
  }
  __device__ __forceinline__ static R inv_sqrt(double x) {
    if (sizeof(R) == 4) return (R)rsqrtf((float)x);
    return (R)rsqrt(x);
  }

  // ---- start: the noiseless run's state at event e (its map in affine form, as computed
  // when the circuit was compiled)
  __device__ void load_snapshot(uint32_t e) {
    const unsigned char *in = C->traj + (size_t)e * C->traj_stride;
    const SnapHdr *h = reinterpret_cast<const SnapHdr *>(in);
    const uint64_t *r_in = reinterpret_cast<const uint64_t *>(in + sizeof(SnapHdr));
    const SnapAffine<R, W> *a = reinterpret_cast<const SnapAffine<R, W> *>(in + snap_affine_off<R, W>(C->rw));
    chain = (int)__ldg(&h->chain);
    logical = (int)__ldg(&h->logical);
    lastm = (int)__ldg(&h->lastm);
    fid = __ldg(&h->fid);
    nrm = 1.0;
    recw = lane < C->rw ? __ldg(&r_in[lane]) : 0ull;
    d = __ldg(&a->d);
    if (d > P.aff_dim || d > kSnapDim) {
      d = 0;
      status = AS_RERUN;
      return;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] = __ldg(&h->sd[w]);
      ss[w] = __ldg(&h->ss[w]);
      a0[w] = __ldg(&a->rows[0][w]);
      B[w] = lane < d ? __ldg(&a->rows[1 + lane][w]) : 0ull;
      D[w] = lane < d ? __ldg(&a->rows[1 + kSnapDim + lane][w]) : 0ull;
    }
    for (uint32_t s = lane; s < size(); s += 32) v[s] = a->v[s];
    __syncwarp();
  }
  // ---- resumption from a lane's record (eviction or hand-over), which holds the same form.
  // Returns the event to resume at.
  __device__ uint32_t load_spill(uint32_t r) {
    const Spill<R, W> S(P.sp, P.rw_max, kLaneDim);
    unsigned char *p = S.at(r);
    const uint4 a = S.ha(p), b = S.hb(p);
    d = a.w & 255u;
    chain = (int)((a.w >> 8) & 1u);
    logical = (int)((a.w >> 9) & 1u);
    lastm = (int)(int8_t)((a.w >> 16) & 255u);
    nc = NoiseCursor{b.x, b.y, b.z};
    fid = S.fid(p);
    if constexpr (kScaled) nrm = S.norm(p);
    recw = lane < C->rw ? S.rec(p)[lane] : 0ull;
    if (d > kLaneDim || d > P.aff_dim || a.y >= C->n_events) {  // a record never holds more, nor resumes past the end
      fail_check(CHK_NNZ, d);
      return C->n_events;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] = S.sd(p)[w];
      ss[w] = S.ss(p)[w];
      a0[w] = S.rows(p)[w];
      B[w] = lane < d ? S.rows(p)[(1 + lane) * W + w] : 0ull;
      D[w] = lane < d ? S.rows(p)[(1 + kLaneDim + lane) * W + w] : 0ull;
    }
    if (lane < size()) v[lane] = ((a.z >> lane) & 1u) ? S.vals(p)[lane] : Cx<R>{0, 0};
    __syncwarp();
    return a.y;
  }

  // ---- Paulis: v'_{a^beta} = i^{e + 2 gamma.a} v_a: phases per entry, then alpha0 moves
  __device__ void apply_pauli(const uint64_t *beta, const uint64_t *gamma, uint32_t e) {
    uint32_t g0;
    const uint32_t gl = parities(gamma, g0);
    e += 2u * g0;
    if (gl || (e & 3u))
      for (uint32_t s = lane; s < size(); s += 32) v[s] = ipow(v[s], e + 2u * par32(s & gl));
#pragma unroll
    for (int w = 0; w < W; ++w) a0[w] ^= beta[w];
    __syncwarp();
  }
  __device__ void apply_error(uint32_t s) {
    if (s >= C->n_sites) {
      fail_check(CHK_SITE, s);
      return;
    }
    // the site's record, 16 bytes per lane, in one load; its words are combined by reductions
    const uint32_t pp = nc.pair(), need = site_images(pp);
    constexpr uint32_t kParts = sizeof(SiteDev<W>) / 16, kSig = W == 1 ? 4u : 8u;  // (lane kSig: the signs)
    const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2 *>(reinterpret_cast<const SiteDev<W> *>(C->sites) + s) +
                               (lane < kParts ? lane : 0u));
    uint64_t beta[W], gamma[W], pe = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      uint64_t esd, ess;
      if (W == 1) {  // lane j: image j's beta and gamma
        const bool in = lane < 4u && ((need >> lane) & 1u);
        beta[w] = xor_all(in ? q.x : 0ull);
        gamma[w] = xor_all(in ? q.y : 0ull);
        esd = shfl64(q.x, kSig);
        ess = shfl64(q.y, kSig);
      } else {  // lanes 2j, 2j + 1: image j's two words of beta, of gamma
        const uint64_t y = w ? q.y : q.x;
        const bool in = lane < 8u && ((need >> (lane >> 1)) & 1u);
        beta[w] = xor_all(in && !(lane & 1u) ? y : 0ull);
        gamma[w] = xor_all(in && (lane & 1u) ? y : 0ull);
        esd = shfl64(y, kSig);
        ess = shfl64(y, kSig + 1u);
      }
      pe ^= ((sd[w] ^ esd) & beta[w]) ^ ((ss[w] ^ ess) & gamma[w]);
    }
    const uint32_t c0 = __shfl_sync(kAll, (uint32_t)(q.y >> 32), (int)kParts - 1);
    apply_pauli(beta, gamma, nc.phase(((c0 >> (2u * pp)) + 2u * wordpar(pe)) & 3u));
  }

  // ---- a I + b Z_q; FP32 as in LaneShot::rot (lanes.cu): the phase xi folded into b (bq, or its
  // negation bn), one fused chain per component (with a zero partner it rounds as one product)
  __device__ void rot(uint32_t w0, uint32_t ci, const uint64_t *beta, const uint64_t *gamma, bool diag) {
    const uint32_t e = (ev_e0(w0) + 2u * wpar2<W>(sd, beta, ss, gamma)) & 3u;  // (beta = 0 when diagonal)
    if (ci >= C->n_coef) {
      fail_check(CHK_COEF, ci);
      return;
    }
    uint32_t g0, gl = parities(gamma, g0), c = 0;
    bool fresh = false;
    uint64_t r[W];
    if (!diag) {
      c = coords(beta, r);
      fresh = wnonzero(r);  // beta outside the span: every entry gains a partner
      if (fresh && compact(gl, g0)) {
        c = coords(beta, r);
        fresh = wnonzero(r);
      }
      if (fresh && d == P.aff_dim) {
        status = AS_RERUN;
        return;
      }
    }
    const Coef *cf = C->coef + ci;
    if constexpr (kScaled) {
      rot_scaled(cf, e, diag, fresh, gl, g0, c, r);
    } else {
      const float4 f = __ldg(reinterpret_cast<const float4 *>(&cf->fa_re));
      const Cx<R> a{(R)f.x, (R)f.y}, bq = ipow(Cx<R>{(R)f.z, (R)f.w}, e), bn{negr(bq.x), negr(bq.y)};
      if (diag) {
        const Cx<R> c0 = cadd(a, bq), c1 = cadd(a, bn);
        for (uint32_t s = lane; s < size(); s += 32) v[s] = pruned(cmul(g0 ^ par32(s & gl) ? c1 : c0, v[s]));
        __syncwarp();
        return;
      }
      if (fresh) {
        const uint32_t n = size(), t0 = c | n;  // slot s gains the partner s ^ t0
        add_dim(r);
        for (uint32_t s = lane; s < n; s += 32) {
          const Cx<R> x = v[s];
          v[s] = pruned(cmul(a, x));
          v[s ^ t0] = pruned(cmul(g0 ^ par32(s & gl) ? bn : bq, x));
        }
      } else {
        const uint32_t q = (uint32_t)__ffs(c) - 1u, flip = par32(c & gl), np = size() >> 1;
        for (uint32_t i = lane; i < np; i += 32) {  // a pair of slots per lane
          const uint32_t s = open_bit(i, q), t = s ^ c, ps = g0 ^ par32(s & gl);
          const Cx<R> vs = v[s], vt = v[t];
          v[s] = pruned(cmad2(a, vs, ps ^ flip ? bn : bq, vt));
          v[t] = pruned(cmad2(a, vt, ps ? bn : bq, vs));
        }
      }
    }
    __syncwarp();
    if (!diag && size() > C->cap && live_count() > C->cap) status = AS_OVF;
  }
  // (rare: many rotations, or very unlikely outcomes, since the last sampled outcome)
  __device__ __forceinline__ void fit_norm() {
    for (int k = 0; k < 32 && !ScaledPrune::in_range(nrm); ++k) {  // (bounded: an empty map has norm 0)
      const double f = ScaledPrune::fit(nrm);
      for (uint32_t s = lane; s < size(); s += 32) v[s] = cscale(v[s], (R)f);
      __syncwarp();
      nrm = nrm * f * f;
    }
  }
  // the scaled form: v' = cm v + i^{e + 3} k (-1)^{gamma.key} v_partner, n2 left to the norm
  __device__ __forceinline__ void rot_scaled(const Coef *cf, uint32_t e, bool diag, bool fresh, uint32_t gl,
                                             uint32_t g0, uint32_t c, const uint64_t *r) {
    const double2 kc = __ldg(reinterpret_cast<const double2 *>(&cf->k));
    const bool plain = __double2hiint(kc.y) != 0x3FF00000;
    if (!plain) nrm = mulr(nrm, __ldg(&cf->n2));
    fit_norm();
    pt.set(nrm);
    const ScaledTurn turn(kc.x, (e + 3u) & 3u);
    auto base = [&](Cx<R> x) { return plain ? cscale(x, (R)kc.y) : x; };
    if (diag) {
      for (uint32_t s = lane; s < size(); s += 32) {
        const Cx<R> x = v[s];
        v[s] = pruned(turn.add(base(x), x, g0 ^ par32(s & gl)));
      }
    } else if (fresh) {  // the old entries stay as they are, but for cm
      const uint32_t n = size(), t0 = c | n;
      add_dim(r);
      for (uint32_t s = lane; s < n; s += 32) {
        const Cx<R> x = v[s];
        v[s] = pruned(base(x));
        v[s ^ t0] = pruned(turn.add(Cx<R>{0, 0}, x, g0 ^ par32(s & gl)));
      }
    } else if (size() <= 32u) {
      // a slot per lane: an FP64 instruction holds its pipe alike for 16 lanes (a pair each,
      // two outputs one after the other) and for 32
      const bool in = lane < size();
      const uint32_t t = lane ^ c;
      Cx<R> x{0, 0}, y{0, 0};
      if (in) {
        x = v[lane];
        y = v[t];
      }
      __syncwarp();
      if (in) v[lane] = pruned(turn.add(base(x), y, g0 ^ par32(t & gl)));
    } else {
      const uint32_t q = (uint32_t)__ffs(c) - 1u, flip = par32(c & gl), np = size() >> 1;
      for (uint32_t i = lane; i < np; i += 32) {  // a pair of slots per lane
        const uint32_t s = open_bit(i, q), t = s ^ c, ps = g0 ^ par32(s & gl);
        const Cx<R> vs = v[s], vt = v[t];
        v[s] = pruned(turn.add(base(vs), vt, ps ^ flip));
        v[t] = pruned(turn.add(base(vt), vs, ps));
      }
    }
  }

  // ---- measurement of P, beta = 0: lambda_a = c (-1)^{gamma.a}
  __device__ int meas_a(uint32_t w0, uint32_t ord, const uint64_t *gamma) {
    const uint32_t e = (ev_e0(w0) + 2u * wpar<W>(ss, gamma)) & 3u;
    if (e & 1u) {
      fail_check(CHK_PHASE, e);
      return 1;
    }
    uint32_t g0;
    const uint32_t gl = parities(gamma, g0);
    const uint32_t sgn = (e >> 1) ^ g0;  // slot s: eigenvalue -1 iff parity(s & gl) != sgn
    if (!gl) return sgn ? -1 : 1;
    bool h0 = false, h1 = false;
    for (uint32_t s = lane; s < size(); s += 32)
      if (nonzero(v[s])) {
        if (par32(s & gl) ^ sgn) h1 = true;
        else h0 = true;
      }
    h0 = __any_sync(kAll, h0);
    h1 = __any_sync(kAll, h1);
    int m;
    bool scaled = false;
    R sc = (R)1;
    if (!(h0 && h1)) {  // decided (all eigenvalues equal): integer test only, no scaling
      m = h1 ? -1 : 1;
    } else {
      // a lane's slots 32 apart change sides with the high part of gl: acc[0] takes the rows of
      // its first slot's side
      double acc[2] = {0.0, 0.0};
      for (uint32_t b = 0; b < size(); b += 32) {
        const uint32_t s = b + lane;
        const Cx<R> x = s < size() ? v[s] : Cx<R>{0, 0};
        if (par32(b & gl)) acc[1] = addn(acc[1], x);
        else acc[0] = addn(acc[0], x);
      }
      const bool first_neg = (par32(lane & gl) ^ sgn) != 0u;
      double sp = first_neg ? acc[1] : acc[0], sm = first_neg ? acc[0] : acc[1];
      sum_both(sp, sm);
      m = pick(ord, sp, sm);
      if constexpr (kScaled) {
        nrm = m == 1 ? sp : sm;
      } else {
        sc = inv_sqrt(m == 1 ? sp : sm);
        scaled = true;
      }
    }
    __syncwarp();
    // the kept slots share parity(s & gl): one coordinate fewer
    remove_dim(31u - __clz(gl), gl, sgn ^ (m == -1 ? 1u : 0u), scaled, sc);
    return m;
  }

  // ---- measurement of P, beta != 0 (case B): row operations on the signs, relabel,
  // pairing, replacement (see LaneShot::meas_b in lanes.cu)
  __device__ int meas_b(uint32_t ord, uint32_t cbi) {
    if (cbi >= C->n_cb) {
      fail_check(CHK_CASEB, cbi);
      return 1;
    }
    const CaseB *Bc = C->cb + cbi;
    const uint32_t p = __ldg(&Bc->p);
    uint64_t J[W], g2[W], ep[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      J[w] = __ldg(&Bc->J[w]);
      g2[w] = __ldg(&Bc->gamma2[w]);
      ep[w] = ((int)(p >> 6) == w) ? (1ull << (p & 63)) : 0ull;
    }
    const uint32_t ssp = wbit<W>(ss, p);
    const uint32_t sdJ = wpar<W>(sd, J);
#pragma unroll
    for (int w = 0; w < W; ++w) ss[w] ^= (ssp ? J[w] : 0ull) ^ __ldg(&Bc->Hs[w]);
    if (sdJ ^ __ldg(&Bc->hdp)) wflip<W>(sd, p);
    const uint32_t e2 = (__ldg(&Bc->e0b) + 2u * (wbit<W>(sd, p) + wpar<W>(ss, g2))) & 3u;
    // relabel a_j ^= a_p (j in J): alpha0 and the directions through it, the duals through its transpose
    const bool a0p0 = wbit<W>(a0, p) != 0u, bp0 = wbit<W>(B, p) != 0u, dj = wpar<W>(D, J) != 0u;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (a0p0) a0[w] ^= J[w];
      if (bp0) B[w] ^= J[w];
      if (dj) D[w] ^= ep[w];
    }
    uint32_t g20;
    const uint32_t gl2 = parities(g2, g20);
    const uint32_t a0p = wbit<W>(a0, p);
    const uint32_t bp = __ballot_sync(kAll, wbit<W>(B, p) != 0u);  // slot s: key bit p = a0p ^ parity(s & bp)
    uint64_t rr[W];
    const uint32_t c = coords(ep, rr);
    const bool lone = wnonzero(rr);  // e_p outside the span: no entry has a partner
    const uint32_t q = lone ? 0u : (uint32_t)__ffs(c) - 1u;
    const uint32_t n = lone ? size() : size() >> 1;
    // v0 (the entry with bit p clear) and x1 = xi_{a1} v_{a1} of item i; s: its slot, t: the other's
    auto pair = [&](uint32_t i, uint32_t &s, uint32_t &t, Cx<R> &v0, Cx<R> &x1) {
      s = lone ? i : open_bit(i, q);
      t = lone ? i : s ^ c;
      const bool hi = (a0p ^ par32(s & bp)) != 0u;
      if (!lone && hi) {
        const uint32_t y = s;
        s = t;
        t = y;
      }
      v0 = (lone && hi) ? Cx<R>{0, 0} : v[s];
      x1 = (lone && !hi) ? Cx<R>{0, 0} : ipow(v[t], e2 + 2u * (g20 ^ par32(t & gl2)));
    };
    int m;
    if constexpr (kScaled) {
      if (lone) {
        // p = 1/2 exactly: one random bit; the entries with key bit p become m xi v, the norm stays
        m = force ? 1 : (philox(P.seed, shot, 1u, ord).x >> 31) ? -1 : 1;
        if (force) fid *= 0.5;
        for (uint32_t s = lane; s < n; s += 32)
          if (a0p ^ par32(s & bp)) v[s] = ipow(v[s], e2 + 2u * (g20 ^ par32(s & gl2)) + (m == -1 ? 2u : 0u));
      } else {
        // sp, sm = (N +- 2 C) / 2 with N the norm and C = sum Re conj(v0) x1; the kept side's own
        // norm is summed from the values it keeps
        double sn = 0.0, cr = 0.0;
        for (uint32_t i = lane; i < n; i += 32) {
          uint32_t s, t;
          Cx<R> v0, x1;
          pair(i, s, t, v0, x1);
          sn = addn(addn(sn, v0), x1);
          cr = fmar((double)v0.x, (double)x1.x, fmar((double)v0.y, (double)x1.y, cr));
        }
        sum_both(sn, cr);
        const double sp = fmar(0.5, sn, cr), sm = fmar(0.5, sn, -cr);
        m = pick(ord, sp, sm);
        nrm = 2.0 * (m == 1 ? sp : sm);
        fit_norm();
        pt.set(nrm);
        double kn = 0.0, none = 0.0;
        for (uint32_t i = lane; i < n; i += 32) {
          uint32_t s, t;
          Cx<R> v0, x1;
          pair(i, s, t, v0, x1);
          const Cx<R> nv = cadd(v0, m == 1 ? x1 : Cx<R>{negr(x1.x), negr(x1.y)});
          kn = addn(kn, nv);
          v[t] = Cx<R>{0, 0};
          v[s] = pruned(nv);
        }
        sum_both(kn, none);
        nrm = kn;
      }
    } else {
      double sp = 0.0, sm = 0.0;
      for (uint32_t i = lane; i < n; i += 32) {
        uint32_t s, t;
        Cx<R> v0, x1;
        pair(i, s, t, v0, x1);
        sp += 0.5 * pnorm(cadd(v0, x1));
        sm += 0.5 * pnorm(csub(v0, x1));
      }
      sum_both(sp, sm);
      m = pick(ord, sp, sm);
      const R sc = inv_sqrt(2.0 * (m == 1 ? sp : sm));
      for (uint32_t i = lane; i < n; i += 32) {
        uint32_t s, t;
        Cx<R> v0, x1;
        pair(i, s, t, v0, x1);
        const Cx<R> nv = cscale(m == 1 ? cadd(v0, x1) : csub(v0, x1), sc);
        v[t] = Cx<R>{0, 0};
        v[s] = pruned(nv);  // (t = s when alone)
      }
    }
    __syncwarp();
    if (lone) {
      // every key loses bit p, injectively; the duals lose it through z (z . B[k] = 0 and
      // z[p] = 1, since e_p's residual is z's): D[k] ^= D[k][p] z keeps D . B and clears bit p
      uint64_t z[W];
      co_dual(rr, z);
      const bool dp = wbit<W>(D, p) != 0u, bb = wbit<W>(B, p) != 0u;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        if (dp) D[w] ^= z[w];
        if (bb) B[w] ^= ep[w];
        if (a0p) a0[w] ^= ep[w];
      }
    } else if (bp) {
      remove_dim(31u - __clz(bp), bp, a0p, false, (R)1);  // the kept keys have bit p clear
    }
    // replacement: d_j <- d_j s_p (j in G), d_p <- old s_p, s_p <- m P
#pragma unroll
    for (int w = 0; w < W; ++w) sd[w] ^= (ssp ? __ldg(&Bc->G[w]) : 0ull) ^ __ldg(&Bc->Hd[w]);
    if (wbit<W>(sd, p) != ssp) wflip<W>(sd, p);
    const uint32_t newsp = (m == -1 ? 1u : 0u) ^ __ldg(&Bc->rP);
    if (wbit<W>(ss, p) != newsp) wflip<W>(ss, p);
    return m;
  }

  __device__ __forceinline__ uint32_t rec_bit(int32_t r) const {
    const bool ok = r >= 0 && (uint32_t)r < 64u * C->rw;
    const uint64_t w = shfl64(recw, ok ? (uint32_t)r >> 6 : 0u);
    return ok ? (uint32_t)((w >> (r & 63)) & 1ull) : 0u;
  }

  // past the first error: the one after it, drawn by the warp (next_site of shot_common.cuh with
  // the candidates of U's bucket compared at once)
  __device__ __forceinline__ void advance() {
    if (nc.second != kNotDrawn) {
      nc.first = nc.second;
      nc.second = kNotDrawn;
      return;
    }
    uint32_t cur = nc.site() + 1u;
    draw(cur);
  }
  __device__ void draw(uint32_t cur) {
    const uint32_t n_sites = C->n_sites;
    for (uint32_t guard = 0; guard <= n_sites; ++guard) {
      if (cur >= n_sites) {
        nc.first = pack_error(kAll, 0u);
        return;
      }
      const uint4 w = philox(P.seed, shot, 0u, nc.kblk++);
      const uint64_t U = (uint64_t)w.x | ((uint64_t)w.y << 32);
      const uint32_t rem = n_sites - cur, b = (uint32_t)(U >> (64 - kThrTabBits));
      const uint32_t t0 = __ldg(&C->thr_tab[b]), t1 = __ldg(&C->thr_tab[b + 1]);
      uint32_t lo = t0 < rem ? t0 : rem;
      const uint32_t hi = t1 < rem ? t1 : rem;
      while (lo < hi) {  // (a bucket spans few sites)
        const uint32_t n = hi - lo < 32u ? hi - lo : 32u;
        const uint32_t below = __popc(__ballot_sync(kAll, lane < n && !(U < __ldg(&C->thr[lo + (lane < n ? lane : 0u)]))));
        lo += below;
        if (below < n) break;
      }
      if (lo == rem) {
        nc.first = pack_error(kAll, 0u);
        return;
      }
      const uint32_t s = cur + lo;
      cur = s + 1u;
      const uint32_t kind = __ldg(&C->site_kind[s]);
      if ((kind & kSiteThinned) && !(w.w < __ldg(&C->site_thin[s]))) continue;
      nc.first = pack_error(s, (kind & 3u) == SITE_DEPOL2 ? __umulhi(w.z, 15u) + 1u
                               : (kind & 3u) == SITE_FLIP ? kind & 12u
                                                          : (__umulhi(w.z, 3u) + 1u) << 2);
      return;
    }
    status = AS_ERR;
  }

  // one event (its copy in shared memory)
  __device__ void step(const Ev<W> *ev) {
    const uint4 hdr = *reinterpret_cast<const uint4 *>(ev);
    const uint64_t *body = ev->dsd;  // dsd, dss, beta, gamma
    while (nc.site() < hdr.y && status == AS_RUN) {
      apply_error(nc.site());
      advance();
    }
    if (status != AS_RUN) return;
    const uint64_t *beta = body + 2 * W, *gamma = body + 3 * W;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] ^= body[w];
      ss[w] ^= body[W + w];
    }
    const uint32_t w0 = hdr.x, type = ev_type(w0), flags = ev_flags(w0);
    if (type == EV_MEAS_A || type == EV_MEAS_B) {
      force = P.fid_mode && (flags & F_FIDELITY);
      const int m = (type == EV_MEAS_A) ? meas_a(w0, hdr.z, gamma) : meas_b(hdr.z, (uint32_t)beta[0]);
      if (status != AS_RUN) return;
      if (force && m == -1) {  // +1 impossible: F = 0, the shot ends kept
        fid = 0.0;
        status = AS_KEPT;
        return;
      }
      lastm = m;
      if (flags & F_RECORD) {
        if (hdr.w >= 64u * C->rw) {
          fail_check(CHK_RECORD, hdr.w);
          return;
        }
        if (m < 0 && lane == (hdr.w >> 6)) recw |= 1ull << (hdr.w & 63u);
      }
      if ((flags & F_COND_LAST) && m == -1) {  // fused reset correction
        uint64_t xb[W], xg[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
          xb[w] = ev->xbeta[w];
          xg[w] = ev->xgamma[w];
        }
        apply_pauli(xb, xg, (ev_xe0(w0) + 2u * wpar2<W>(sd, xb, ss, xg)) & 3u);
      }
      if ((flags & F_DETECTOR) && ((m == -1 ? 1u : 0u) ^ ((flags & F_INVERT) ? 1u : 0u))) status = AS_DISC;
    } else if (type == EV_ROT || type == EV_ROT_DIAG) {
      rot(w0, hdr.z, beta, gamma, type == EV_ROT_DIAG);
    } else if (type == EV_PAULI) {
      const uint32_t cond = (flags & F_COND_LAST) ? (uint32_t)(lastm == -1)
                                                  : rec_bit((int32_t)hdr.z) ^ rec_bit((int32_t)hdr.w);
      if (cond) apply_pauli(beta, gamma, (ev_e0(w0) + 2u * wpar2<W>(sd, beta, ss, gamma)) & 3u);
    } else if (type == EV_PARITY) {
      const int par = chain ^ (int)rec_bit((int32_t)hdr.z) ^ (int)rec_bit((int32_t)hdr.w) ^ ((flags & F_INVERT) ? 1 : 0);
      if (flags & F_CHAIN) {
        chain = par;
      } else {
        chain = 0;
        if ((flags & F_DETECTOR) && par) status = AS_DISC;
        if ((flags & F_OBSERVABLE) && par) logical = 1;
      }
    }
  }
  // event e into its place of the ring, 16 bytes per lane (one copy group per event, empty past
  // the end, so that the groups count the events)
  __device__ __forceinline__ void fetch_event(const Ev<W> *evs, uint32_t e, uint32_t n_events) {
    if (e < n_events && lane < sizeof(Ev<W>) / 16)
      copy_async<16>(ring + (e % kRing) * sizeof(Ev<W>) + lane * 16u, reinterpret_cast<const unsigned char *>(evs + e) + lane * 16u);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // the shot of item `local` (chunk-local), from spill record r or (kNoRecord) from its start
  // event
  __device__ void run(uint64_t s, uint32_t local, uint32_t r) {
    shot = s;
    status = AS_RUN;
    force = false;
    uint32_t ev;
    if (r != kNoRecord) {
      ev = load_spill(r);
    } else {
      // the pre-pass drew the first errors (and put the shot on this pass's list, or a lane did)
      const uint4 k = reinterpret_cast<const uint4 *>(P.al_cursor)[local];
      nc = NoiseCursor{k.x, k.y, k.z};
      if (nc.kblk == kAll) status = AS_ERR;
      ev = k.w;
      load_snapshot(ev);
    }
    const Ev<W> *evs = reinterpret_cast<const Ev<W> *>(C->ev);
    const uint32_t n_events = C->n_events;
    ev_top = ev;
    if (status == AS_RUN) {
      for (uint32_t k = 0; k + 1u < kRing; ++k) fetch_event(evs, ev + k, n_events);
      while (ev < n_events && status == AS_RUN) {  // the events after this one are on their way
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
        __syncwarp();
        fetch_event(evs, ev + kRing - 1u, n_events);
        step(reinterpret_cast<const Ev<W> *>(ring + (ev % kRing) * sizeof(Ev<W>)));
        ev_top = ++ev;
      }
      copies_done();  // (the next shot writes the ring again)
      __syncwarp();
    }
    if (status == AS_RUN) status = AS_KEPT;
  }
  // tallies, status, records, captured state; off: the shot's offset within its circuit
  __device__ void finish(uint32_t local, uint64_t off, uint32_t ci, unsigned long long (*btally)[5]) {
    if (status == AS_RERUN) {
      if (lane == 0) {
        const unsigned long long i = atomicAdd(P.n_rerun, 1ull);
        if (i < P.rerun_cap) P.rerun[i] = local;
        if (P.n_rerun_total) atomicAdd(P.n_rerun_total, 1ull);
      }
      return;
    }
    if (lane == 0) {
      atomicAdd(&btally[ci][0], 1ull);
      if (status == AS_DISC) atomicAdd(&btally[ci][1], 1ull);
      else if (status == AS_OVF) atomicAdd(&btally[ci][2], 1ull);
      else if (status == AS_KEPT) {
        atomicAdd(&btally[ci][3], 1ull);
        if (logical) atomicAdd(&btally[ci][4], 1ull);
        if (P.fid_mode && C->fsum) atomicAdd(C->fsum, fid);
      }
      if (off < C->out_limit && C->status) C->status[off] = (uint8_t)status;
    }
    if (off < C->out_limit && C->records && lane < C->rw) C->records[off * C->rw + lane] = recw;
    if (ci == 0 && off < P.st_limit) capture(off);
  }
  uint32_t ev_top;  // the event after the last one that the shot ran
  __device__ void capture(uint64_t off) const {
    Cx<double> f{1.0, 0.0};
    if constexpr (kScaled) f = readout(top_phase<W>(C, ev_top), nrm);
    if (lane == 0) {
      P.st_signs[off * 4 + 0] = sd[0];
      P.st_signs[off * 4 + 1] = (W == 2) ? sd[W - 1] : 0ull;
      P.st_signs[off * 4 + 2] = ss[0];
      P.st_signs[off * 4 + 3] = (W == 2) ? ss[W - 1] : 0ull;
    }
    uint32_t n = 0;
    for (uint32_t b = 0; b < size(); b += 32) {
      const uint32_t s = b + lane;
      const bool live = s < size() && nonzero(v[s]);
      const uint32_t m = __ballot_sync(kAll, live);
      uint64_t k[W];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        k[w] = a0[w];
        for (uint32_t j = 0; j < d; ++j) {
          const uint64_t x = shfl64(B[w], j);
          if ((s >> j) & 1u) k[w] ^= x;
        }
      }
      const uint32_t i = n + __popc(m & ((1u << lane) - 1u));
      if (live && i < P.st_stride) {
        const size_t o = (size_t)off * P.st_stride + i;
        P.st_keys[2 * o] = k[0];
        P.st_keys[2 * o + 1] = (W == 2) ? k[W - 1] : 0ull;
        Cx<R> x = v[s];
        if constexpr (kScaled) x = cmul(f, x);
        P.st_vals[2 * o] = (double)x.x;
        P.st_vals[2 * o + 1] = (double)x.y;
      }
      n += __popc(m);
    }
    if (lane == 0) P.st_nnz[off] = n;
  }
};

template <typename R, int W>
__global__ void __launch_bounds__(kAffBlock, sizeof(R) == 4 && W == 1 ? 6 : 5) affine_kernel(
    const __grid_constant__ ShotParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long btally[kMaxCirc][5];
  const uint32_t n_circ = P.n_circ < (uint32_t)kMaxCirc ? P.n_circ : (uint32_t)kMaxCirc;
  for (uint32_t i = threadIdx.x; i < 5 * n_circ; i += blockDim.x) btally[i / 5][i % 5] = 0ull;
  __syncthreads();
  AffShot<R, W> s(P, smem + (threadIdx.x / 32) * aff_warp_bytes<R, W>(P.aff_dim));
  const unsigned long long n_items = *P.n_items_dev < P.rerun_cap ? *P.n_items_dev : P.rerun_cap;  // the list's entries
  const unsigned long long item_base = P.item_base_dev ? *P.item_base_dev : P.item_base;
  for (;;) {
    unsigned long long item = 0;
    if (s.lane == 0) item = atomicAdd(P.next_item, 1ull);
    item = __shfl_sync(kAll, item, 0);
    if (item >= n_items) break;
    uint32_t local = P.list[item];
    uint32_t rec = kNoRecord;  // an entry naming a spill record resumes the shot a lane handed over
    if ((local & kSpillRef) && P.sp) {
      rec = local & ~kSpillRef;
      if (rec >= P.sp_cap) break;  // never: records are taken below the pool's capacity
      const Spill<R, W> S(P.sp, P.rw_max, kLaneDim);
      local = S.ha(S.at(rec)).x;
    }
    const uint64_t g = item_base + local;
    uint32_t lo = 0, hi = n_circ;  // the circuit of item g
    while (hi - lo > 1u) {
      const uint32_t mid = (lo + hi) >> 1;
      if (P.circ[mid].item_begin <= g) lo = mid;
      else hi = mid;
    }
    s.C = &P.circ[lo];
    const uint64_t off = g - s.C->item_begin;
    s.run(s.C->first_shot + off, local, rec);
    s.finish(local, off, lo, btally);
    __syncwarp();
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < 5 * n_circ; i += blockDim.x)
    if (btally[i / 5][i % 5]) atomicAdd(&P.circ[i / 5].tally[i % 5], btally[i / 5][i % 5]);
}

}  // namespace

cudaError_t prepare_affine(const ShotParams &p, int fp32, uint32_t W, int blocks_per_sm, LaunchCfg *cfg) {
  if (!p.list || !p.n_items_dev || p.aff_dim > 12 || p.rw_max > kAffRecWords) return cudaErrorInvalidConfiguration;
  const void *kern = fp32 ? (W == 1 ? reinterpret_cast<const void *>(affine_kernel<float, 1>)
                                    : reinterpret_cast<const void *>(affine_kernel<float, 2>))
                          : (W == 1 ? reinterpret_cast<const void *>(affine_kernel<double, 1>)
                                    : reinterpret_cast<const void *>(affine_kernel<double, 2>));
  const size_t smem =
      (kAffBlock / 32) * (fp32 ? (W == 1 ? aff_warp_bytes<float, 1>(p.aff_dim) : aff_warp_bytes<float, 2>(p.aff_dim))
                               : (W == 1 ? aff_warp_bytes<double, 1>(p.aff_dim) : aff_warp_bytes<double, 2>(p.aff_dim)));
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kAffBlock, smem)) != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  if (blocks_per_sm > 0 && blocks_per_sm < occ) occ = blocks_per_sm;
  cfg->kern = kern;
  cfg->grid = (unsigned)(occ * sms);
  cfg->block = kAffBlock;
  cfg->smem = smem;
  return cudaSuccess;
}

}  // namespace soft
