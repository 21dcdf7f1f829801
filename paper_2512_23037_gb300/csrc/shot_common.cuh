// shot_common.cuh -- per-shot device pieces shared by the shot kernels: the
// noise stream's next accepted site, the event a shot starts at, the layout of
// the noiseless run's snapshots, and the spill records through which a shot
// moves between lanes of later rounds, or from a lane to a warp.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "device_common.cuh"
#include "kernels.cuh"

namespace soft {
namespace dev {

// The next accepted error site at or after `cur` of shot `shot`: geometric gaps
// of the noise stream against the thresholds thr (the smallest gap g with
// U < thr[g]), then thinning. nxt = the site (0xFFFFFFFF if none), pp = its Pauli
// pair (pa << 2 | pb, codes 1 X, 2 Y, 3 Z; pb = 0 at a one-qubit site).
// False if the guard ran out (impossible for valid tables).
template <bool Rolled = false>
__device__ __forceinline__ bool next_site(const CircDev *C, uint64_t seed, uint64_t shot, uint32_t &cur,
                                          uint32_t &kblk, uint32_t &nxt, uint32_t &pp) {
  const uint32_t n_sites = C->n_sites;
  const uint64_t *thr = C->thr;
  for (uint32_t guard = 0; guard <= n_sites; ++guard) {
    if (cur >= n_sites) {
      nxt = 0xFFFFFFFFu;
      return true;
    }
    uint4 w = philox<Rolled>(seed, shot, 0u, kblk++);
    uint64_t U = (uint64_t)w.x | ((uint64_t)w.y << 32);
    const uint32_t rem = n_sites - cur;
    uint32_t lo = 0, hi = rem;
    if (C->thr_tab) {  // U's bucket bounds the answer: search between its entry and the next
      const uint32_t b = (uint32_t)(U >> (64 - kThrTabBits));
      const uint32_t t0 = __ldg(&C->thr_tab[b]), t1 = __ldg(&C->thr_tab[b + 1]);
      lo = t0 < rem ? t0 : rem;
      hi = t1 < rem ? t1 : rem;
    }
    while (lo < hi) {
      uint32_t mid = (lo + hi) >> 1;
      if (U < __ldg(&thr[mid])) hi = mid;
      else lo = mid + 1u;
    }
    if (lo == rem) {
      cur = n_sites;
      nxt = 0xFFFFFFFFu;
      return true;
    }
    uint32_t s = cur + lo;
    cur = s + 1u;
    const uint32_t kind = __ldg(&C->site_kind[s]);
    if ((kind & kSiteThinned) && !(w.w < __ldg(&C->site_thin[s]))) continue;
    nxt = s;
    pp = (kind & 3u) == SITE_DEPOL2 ? __umulhi(w.z, 15u) + 1u
         : (kind & 3u) == SITE_FLIP ? kind & 12u
                                    : (__umulhi(w.z, 3u) + 1u) << 2;
    return true;
  }
  nxt = 0xFFFFFFFFu;
  return false;
}

// The image of the error pp at site s, relative to signs (sd, ss) at the previous event:
// i^e d_beta s_gamma. Every load is independent of the others.
template <int W>
__device__ __forceinline__ uint32_t site_pauli(const CircDev *C, uint32_t s, uint32_t pp, const uint64_t *sd,
                                               const uint64_t *ss, uint64_t *beta, uint64_t *gamma) {
  const SiteDev<W> *S = reinterpret_cast<const SiteDev<W> *>(C->sites) + s;
  const uint32_t need = site_images(pp);
#pragma unroll
  for (int w = 0; w < W; ++w) beta[w] = gamma[w] = 0ull;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint64_t m = 0ull - (uint64_t)((need >> j) & 1u);
    const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(S->img[j]);
    const ulonglong2 x = __ldg(p);
    if (W == 1) {
      beta[0] ^= x.x & m;
      gamma[0] ^= x.y & m;
    } else {
      const ulonglong2 y = __ldg(p + 1);
      beta[0] ^= x.x & m;
      beta[W - 1] ^= x.y & m;
      gamma[0] ^= y.x & m;
      gamma[W - 1] ^= y.y & m;
    }
  }
  uint64_t pe = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) pe ^= ((sd[w] ^ __ldg(&S->dsd[w])) & beta[w]) ^ ((ss[w] ^ __ldg(&S->dss[w])) & gamma[w]);
  return ((__ldg(&S->c0) >> (2u * pp)) + 2u * wordpar(pe)) & 3u;
}

// A shot's place in its noise stream: the next error, the one after it once drawn (`drawn`;
// the lanes' pre-pass draws both, whose Philox blocks and searches would run with a few
// active lanes in the lane kernel), and the next Philox block. Packed: site | pair << 28.
// (site kMaxPackedSites: no error left)
constexpr uint32_t kNotDrawn = 0x10000000u;  // (no second error: it would be at site 0)
__device__ __forceinline__ uint32_t pack_error(uint32_t nxt, uint32_t pp) {
  return nxt == 0xFFFFFFFFu ? 0x0FFFFFFFu : nxt | (pp << 28);
}
// kblk carries kPhaseKnown and the first error's phase (bits 30-31) while the shot starts at a
// later event than the one that applies it, and the same of the second three bits further down
// where that holds for it too (only with a fate table, so for at most kFateMaxSites sites, whose
// block numbers stay below these bits; reading the second's phase from the table as it comes up
// took 2 % of a random 40-qubit circuit's run and 5 % of w97's in FP64).
constexpr uint32_t kPhaseKnown = 0x20000000u, kSecondKnown = kPhaseKnown >> 3, kBlockMask = kSecondKnown - 1u;
static_assert(kFateMaxSites < kBlockMask, "block numbers below the flags");
struct NoiseCursor {
  uint32_t first, second, kblk;
  // the first error's phase: that of its site, e, or the one it brought along
  __device__ __forceinline__ uint32_t phase(uint32_t e) {
    if (kblk & kPhaseKnown) {
      e = kblk >> 30;
      kblk = (kblk & kBlockMask) | ((kblk & (7u * kSecondKnown)) << 3);
    }
    return e;
  }
  __device__ __forceinline__ uint32_t site() const { return first & 0x0FFFFFFFu; }
  __device__ __forceinline__ uint32_t pair() const { return first >> 28; }
  // past the first error
  template <bool Rolled = false>
  __device__ __forceinline__ bool advance(const CircDev *C, uint64_t seed, uint64_t shot) {
    bool ok = true;
    if (second == kNotDrawn) {
      uint32_t cur = site() + 1u, nxt = 0xFFFFFFFFu, pp = 0;
      ok = next_site<Rolled>(C, seed, shot, cur, kblk, nxt, pp);
      first = pack_error(nxt, pp);
    } else {
      first = second;
      second = kNotDrawn;
    }
    return ok;
  }
};

// The event a shot whose first error is at site nxt starts at: the event that
// applies that error, capped at the last valid event of the noiseless run
// (fidelity mode: of its part before the first observed measurement).
__device__ __forceinline__ uint32_t first_event(const CircDev *C, int fid_mode, uint32_t nxt) {
  const uint32_t stop = fid_mode && C->traj_fid_stop < C->traj_stop ? C->traj_fid_stop : C->traj_stop;
  if (nxt < C->n_sites) {
    const uint32_t e = __ldg(&C->site_ev[nxt]);
    return e < stop ? e : stop;
  }
  return stop;
}

// Where a shot starts whose next two errors nc holds: at the event that applies the first, or
// later (see fate_kernel). Its first error is carried to the event where its fate is decided; if
// the second comes in before that, the two are carried to the earlier of their events, if that
// comes before the third error, which is drawn here for it (and again where the shot runs: the
// cursor holds two). With the second error carried the pre-pass discards 71 % of w42's shots and
// 78 % of w97's (60 and 61 % with the first alone) and the others run fewer events (per shot w42
// 10.7 -> 9.1, w97 13.4 -> 9.2): w42 FP32 2^24 shots 8.56 -> 7.6 ms, w97 FP64 500 k 4.7 -> 3.5.
// At the latest it starts where its next error comes in or the recorded noiseless run ends.
// resolved: the shot ends at the returned event, discarded by its detector (whose record is
// flipped), with nothing left to run. ahead: false for shots whose final state is captured (they
// run from their first error).
__device__ __forceinline__ uint32_t start_event(const CircDev *C, int fid_mode, uint64_t seed, uint64_t shot,
                                                NoiseCursor &nc, bool ahead, bool &resolved) {
  const uint32_t stop = fid_mode && C->traj_fid_stop < C->traj_stop ? C->traj_fid_stop : C->traj_stop;
  resolved = false;
  const uint32_t s = nc.site();
  if (s == kMaxPackedSites) return stop;
  const uint32_t e1 = __ldg(&C->site_ev[s]);
  if (e1 > stop) return stop;
  if (!C->fate || !ahead) return e1;
  const uint32_t f = __ldg(&C->fate[(size_t)s * 16 + nc.pair()]), s2 = nc.second & kMaxPackedSites;
  uint32_t F = f & kFateEvent, discard = f & kFateDiscard, second = 0;
  uint32_t next = s2 == kMaxPackedSites ? 0xFFFFFFFFu : __ldg(&C->site_ev[s2]);  // where the next error comes in
  if (next <= (F < stop ? F : stop)) {
    const uint32_t f2 = __ldg(&C->fate[(size_t)s2 * 16 + (nc.second >> 28)]), F2 = f2 & kFateEvent;
    uint32_t cur = s2 + 1u, kblk = nc.kblk, s3 = 0, p3 = 0;
    if ((F2 > next || (f2 & kFateDiscard)) && next_site(C, seed, shot, cur, kblk, s3, p3)) {
      // an event that neither of them passes may be one that their product passes: the shot runs it
      discard = F2 < F ? f2 & kFateDiscard : F2 == F ? 0u : discard;
      F = F2 < F ? F2 : F;
      next = s3 == 0xFFFFFFFFu ? s3 : __ldg(&C->site_ev[s3]);
      second = kSecondKnown | ((f2 & 0xC0000000u) >> 3);
    }
  }
  if (discard && F <= stop && next > F) {
    resolved = true;
    return F;
  }
  const uint32_t at = F < next ? F : next;
  nc.kblk |= kPhaseKnown | second | (f & 0xC0000000u);
  return at < stop ? at : stop;
}

// Snapshot of the noiseless run at the top of an event: header, rw record words,
// kSnapMax keys (W words each), kSnapMax values.
// The phase of the events before e (Ev::w0, in units of pi/8): the top of event e.
template <int W>
__device__ __forceinline__ uint32_t top_phase(const CircDev *C, uint32_t e) {
  return e ? ev_phase(__ldg(&reinterpret_cast<const Ev<W> *>(C->ev)[e - 1u].w0)) : 0u;
}
struct SnapHdr {
  uint32_t nnz, chain, logical, lastm;
  double fid;
  uint64_t sd[2], ss[2];
  uint64_t pad;
};
static_assert(sizeof(SnapHdr) == 64, "snapshot header");
constexpr uint32_t kSnapMax = 64;
// where the keys start (a multiple of 16, so that FP64 values are aligned)
__host__ __device__ constexpr size_t snap_keys_off(uint32_t rw) { return sizeof(SnapHdr) + (size_t)((rw + 1u) & ~1u) * 8; }

// The snapshot's map in the affine form of the lane kernels (lanes.cu): d directions
// (0xFFFFFFFF: more than kSnapDim), the live slots (bit s: slot s), rows alpha0,
// B[0..kSnapDim), Dual[0..kSnapDim), and the values of 2^kSnapDim slots (zero where not
// live; FP64: without the global phase, as scaled maps hold them). Computed once per circuit
// and precision, after the noiseless run.
constexpr uint32_t kSnapDim = 6;
template <typename R, int W>
struct SnapAffine {
  uint32_t d, live_lo, live_hi, pad;  // live: the slot set, in two words
  uint64_t rows[2 + 2 * kSnapDim][W];  // (one row of padding: v is 16-byte aligned)
  Cx<R> v[1u << kSnapDim];
};
template <typename R, int W>
__host__ __device__ constexpr size_t snap_affine_off(uint32_t rw) {
  return (snap_keys_off(rw) + kSnapMax * (size_t)W * 8 + kSnapMax * sizeof(Cx<R>) + 15) & ~(size_t)15;
}
template <typename R, int W>
__host__ __device__ constexpr size_t snap_stride(uint32_t rw) {
  return (snap_affine_off<R, W>(rw) + sizeof(SnapAffine<R, W>) + 15) & ~(size_t)15;
}

#ifndef SOFT_LANE_CAP
#define SOFT_LANE_CAP 16
#endif
constexpr uint32_t kLaneCap = SOFT_LANE_CAP;  // map entries per lane
static_assert(kLaneCap >= 2 && kLaneCap <= 16, "lane map capacity (partner indices are 4-bit)");

// A rerun-list entry with this bit names a spill record (a shot handed from its
// lane to a warp) instead of an item.
constexpr uint32_t kSpillRef = 0x80000000u;
constexpr uint32_t kNoRecord = 0xFFFFFFFFu;

// The outcome +1 (or -1) of a measurement with unnormalised probabilities sp and sm: +1 iff
// u < p, p = sp / (sp + sm) snapped to 0 or 1 within 1e-12, decided as u (sp + sm) < sp. The
// random words are Philox's for the measurement's ordinal. Sums whose 21-bit truncations
// settle the snap and the comparison (all but 1 in 10^5) are decided in FP32, which keeps
// eight instructions off the FP64 pipe; the others exactly. force: fidelity mode, projects
// onto +1 with weight p in fid. *undecided is set where the outcome depended on u.
template <bool Rolled>
__device__ __forceinline__ int pick_outcome(uint64_t seed, uint64_t shot, uint32_t ord, double sp, double sm, bool force,
                                            double &fid, bool *undecided) {
  const float a = low_float(sp), t = a + low_float(sm);
  const bool clear = a > 1e-5f * t && a < (1.0f - 1e-5f) * t;
  if (!clear || force) {
    const double tot = sp + sm;
    if (!(tot > 0.0)) return -1;
    const bool zero = sp < 1e-12 * tot, one = sp > (1.0 - 1e-12) * tot;
    if (undecided && !zero && !one) *undecided = true;
    if (force) {
      if (zero) return -1;
      fid *= one ? 1.0 : sp / tot;
      return 1;
    }
    if (zero) return -1;
    if (one) return 1;
  }
  if (undecided) *undecided = true;
  const uint4 w = philox<Rolled>(seed, shot, 1u, ord);
  const float diff = (float)w.x * 0x1p-32f * t - a;
  if (fabsf(diff) > 1e-5f * t) return diff < 0.0f ? 1 : -1;
  const uint64_t m = ((uint64_t)w.x << 21) ^ (uint64_t)(w.y >> 11);
  return (double)m * 0x1p-53 * (sp + sm) < sp ? 1 : -1;
}

// A spill record holds one shot's whole state at the top of an event, with its map in a
// lane's affine form of `dim` directions: item, resume event, live slots (low word), d and
// flags (chain, logical, last outcome); the noise cursor and the live slots' high word; F;
// FP64: the squared norm; the signs; the record words; the rows alpha0, B[0..dim),
// Dual[0..dim); the values of the 2^dim slots (those of live slots below 2^d, rows below d,
// are written). A lane or a warp reads a whole record at once, so its words are contiguous.
template <typename R, int W>
struct Spill {
  unsigned char *base;
  uint32_t rw, dim;
  size_t stride;
  __host__ __device__ static size_t fixed(uint32_t rw) {
    return 48 + (size_t)2 * W * 8 + (size_t)rw * 8;
  }
  __host__ __device__ static size_t vals_off(uint32_t rw, uint32_t dim) {
    return (fixed(rw) + (size_t)(1 + 2 * dim) * W * 8 + 15) & ~(size_t)15;
  }
  __host__ __device__ static size_t record_bytes(uint32_t rw, uint32_t dim) {
    return (vals_off(rw, dim) + (sizeof(Cx<R>) << dim) + 15) & ~(size_t)15;
  }
  __device__ Spill(unsigned char *b, uint32_t rw_, uint32_t dim_)
      : base(b), rw(rw_), dim(dim_), stride(record_bytes(rw_, dim_)) {}
  __device__ __forceinline__ unsigned char *at(uint32_t r) const { return base + (size_t)r * stride; }
  __device__ __forceinline__ static uint4 &ha(unsigned char *p) { return reinterpret_cast<uint4 *>(p)[0]; }
  __device__ __forceinline__ static uint4 &hb(unsigned char *p) { return reinterpret_cast<uint4 *>(p)[1]; }
  __device__ __forceinline__ static double &fid(unsigned char *p) { return reinterpret_cast<double *>(p)[4]; }
  __device__ __forceinline__ static double &norm(unsigned char *p) { return reinterpret_cast<double *>(p)[5]; }
  __device__ __forceinline__ static uint64_t *sd(unsigned char *p) { return reinterpret_cast<uint64_t *>(p + 48); }
  __device__ __forceinline__ static uint64_t *ss(unsigned char *p) { return sd(p) + W; }
  __device__ __forceinline__ static uint64_t *rec(unsigned char *p) { return sd(p) + 2 * W; }
  __device__ __forceinline__ uint64_t *rows(unsigned char *p) const { return reinterpret_cast<uint64_t *>(p + fixed(rw)); }
  __device__ __forceinline__ Cx<R> *vals(unsigned char *p) const {
    return reinterpret_cast<Cx<R> *>(p + vals_off(rw, dim));
  }
  __device__ __forceinline__ static uint32_t meta(uint32_t d, int chain, int logical, int lastm) {
    return d | ((uint32_t)(chain & 1) << 8) | ((uint32_t)(logical & 1) << 9) | (((uint32_t)lastm & 255u) << 16);
  }
};
constexpr uint32_t kLaneDim = 4;  // directions of a first-round lane's records (kLaneCap = 2^kLaneDim)
static_assert(kLaneCap == (1u << kLaneDim), "lane map");

}  // namespace dev
}  // namespace soft
