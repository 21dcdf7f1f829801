// lanes.cu -- shot kernel with one shot per lane, 32 shots per warp, all at the
// same event.
//
// Shots are first bucketed by the event they start at (start_event: where their first
// errors come to matter, at most the end of the circuit's recorded noiseless run).
// Every warp then walks the events in order. Its idle lanes claim shots from the
// bucket of the event it is at, load the noiseless run's state there, and the
// warp executes each event once for all its lanes: the event is decoded once,
// and every lane updates its own shot's coefficient map, kept in shared memory
// (entry i of lane l at row i, column l). A rotation whose map would outgrow
// kLaneCap entries hands the shot over: its state at the top of that event goes
// to a spill record, which the wide round's lanes or the affine warp pass (affine.cu)
// resume. The per-shot arithmetic is that of the warp-per-shot kernels (the same
// formulas, pruning thresholds and outcome rule), entry by entry. In a batch, each circuit
// has its own range of buckets and a warp serves one circuit at a time. Circuits
// whose noiseless maps outgrow kLaneCap get lanes of 32 or (FP32) 64 entries, one
// launch per size over that size's buckets; the shots of circuits beyond those go
// straight to the warp pass.
//
// Most shots end at the first detector after their first error, but a few run to
// the end of the circuit, and they would hold a warp with a few active lanes. So a
// warp left with few active lanes (lane_evict) writes their shots' state to a
// spill pool and moves on to fresh shots. The next round (another launch) buckets
// the evicted shots by the event they resume at, and packs them into warps again; in
// small runs the affine warp pass takes them instead. The last round evicts nothing, until
// most of its warps have ended (lane_tail): the affine pass takes the others' shots. Which lane or
// warp runs a shot depends on the order of claims, so all of them share one arithmetic, entry by
// entry; FP64 sums over a map's entries alone run in another order in the affine pass.
//
// A warp's time went to waits rather than to the maps (clock counters, w42 FP32: claims 22 %,
// errors 17 %, finished and evicted shots 13 %, the search for the next bucket 7 %). So the
// pre-pass draws each shot's first two errors and leaves its cursor in bucket order; a claim
// issues the snapshot's copies to shared memory before its atomic answers; bucket bounds are
// read one event ahead; tallies are ballots; and 32 buckets are searched at a time. w42 FP32
// at 2^24 shots 19.6 -> 16.8 ms, FP64 at 2^22 11.2 -> 9.7 ms, w97 FP32 at 2 M 24.9 -> 21.7 ms,
// a batch of 64 circuits (7.7 M shots) 31.7 -> 16.6 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "device_common.cuh"
#include "kernels.cuh"
#include "shot_common.cuh"

namespace soft {
namespace {

using namespace dev;
namespace cg = cooperative_groups;

enum : int { LS_RUN = -1, LS_KEPT = 0, LS_DISC = 1, LS_OVF = 2, LS_ERR = 3, LS_RERUN = 4, LS_HAND = 5 };
constexpr int kLaneBlock = 128;
// threads per block of a lane launch: 2 warps for 32-entry lanes (their shared memory per
// warp fits more warps per SM in small blocks: FP64 10 against 8, FP32 18 against 16; w42
// FP64 406.5 -> 421.0 M shots/s, FP32 713 -> 720 M through the wide round), 4 otherwise
template <uint32_t Cap>
__host__ __device__ constexpr int lane_block() { return Cap == 32u ? 64 : kLaneBlock; }
constexpr uint32_t kLaneMaxBuckets = 50000;  // the pre-pass histogram of all buckets: 200 KB of shared memory
#ifndef SOFT_LANE_ROUNDS
#define SOFT_LANE_ROUNDS 2
#endif
constexpr uint32_t kLaneRounds = SOFT_LANE_ROUNDS;  // rounds per chunk, the last without eviction
static_assert(kLaneRounds >= 1 && kLaneRounds <= 8, "lane rounds");

// The wide round's lanes: shots handed over by the first rounds continue in lanes
// of twice the map.
constexpr uint32_t kWideCap = 2 * kLaneCap;
// First-pass lanes for circuits whose noiseless maps outgrow kLaneCap: 32 entries (kWideCap)
// or, with FP32 coefficients, 64 entries. These never hand over: a shot whose map outgrows
// them runs again from its start in a warp.
constexpr uint32_t kLaneBigCap = 4 * kLaneCap;

// Lane map in affine form. The keys of a shot's coefficient map lie in an affine
// space alpha0 ^ span(B[0..d)) of dimension d <= kDim (Sec. II-C: the support of v
// grows by one direction per rotation whose beta is new, Theorem 1 (3), and shrinks
// with measurements and cancellations). Slot s (s < 2^d) holds the entry of key
//   key(s) = alpha0 ^ XOR over the set bits k of s of B[k],
// with its value in row s of the lane's value column, and `live` marks the slots that
// hold entries (values elsewhere are never read). Dual[k] (Dual[k] . B[j] = 1 iff
// k = j, over GF(2)) gives the coordinates of a vector x of the span: x = XOR over
// the k with Dual[k] . x = 1 of B[k]. So the partner key(s) ^ beta of a rotation is
// slot s ^ c (c: beta's coordinates), a parity gamma . key(s) is g0 ^ parity(s & gl)
// (g0 = gamma . alpha0, bit k of gl = gamma . B[k]), and a Pauli error moves alpha0
// only: per entry only values are read and written, and no key is stored. The live
// slots are the paper's sparse map: updates, pruning at tau and the overflow rule
// apply to them exactly as to a sparse map.
__host__ __device__ constexpr uint32_t lane_dim(uint32_t cap) { return cap <= 16u ? 4u : cap <= 32u ? 5u : 6u; }
// A set of slots: one bit per slot of the lane's cube (32 bits up to 32 slots, 64 for 64).
template <uint32_t Cap>
struct SlotSet {
  using T = uint32_t;
};
template <>
struct SlotSet<64> {
  using T = unsigned long long;
};
// (of a nonempty set)
__device__ __forceinline__ uint32_t mffs(uint32_t m) { return (uint32_t)__ffs(m); }
__device__ __forceinline__ uint32_t mffs(unsigned long long m) { return 1u + (uint32_t)__clzll((long long)__brevll(m)); }
__device__ __forceinline__ uint32_t mpopc(uint32_t m) { return (uint32_t)__popc(m); }
__device__ __forceinline__ uint32_t mpopc(unsigned long long m) { return (uint32_t)__popcll(m); }

template <typename R, int W, uint32_t Cap>
__host__ __device__ inline size_t lane_warp_bytes(uint32_t rw) {
  // values of Cap slots; alpha0, kDim basis and kDim dual vectors (W words each); record words
  return (size_t)Cap * sizeof(Cx<R>) * 32 + (size_t)(1 + 2 * lane_dim(Cap)) * W * 8 * 32 + (size_t)rw * 8 * 32;
}

// Slot masks over a cube of up to 32 (M = uint32_t) or 64 slots: the slots whose index has
// bit k set.
template <typename M>
__device__ __forceinline__ M slot_bit_mask(uint32_t k) {
  if (sizeof(M) == 4)
    return (M)(k == 0u ? 0xAAAAAAAAu : k == 1u ? 0xCCCCCCCCu : k == 2u ? 0xF0F0F0F0u : k == 3u ? 0xFF00FF00u : 0xFFFF0000u);
  return (M)(k == 0u   ? 0xAAAAAAAAAAAAAAAAull
             : k == 1u ? 0xCCCCCCCCCCCCCCCCull
             : k == 2u ? 0xF0F0F0F0F0F0F0F0ull
             : k == 3u ? 0xFF00FF00FF00FF00ull
             : k == 4u ? 0xFFFF0000FFFF0000ull
                       : 0xFFFFFFFF00000000ull);
}
// The slots s with parity(s & g) = 1, in a cube of Dim coordinates.
template <typename M, uint32_t Dim>
__device__ __forceinline__ M slot_par_mask(uint32_t g) {
  M m = 0;
#pragma unroll
  for (uint32_t k = 0; k < Dim; ++k)
    if ((g >> k) & 1u) m ^= slot_bit_mask<M>(k);
  return m;
}
// A slot set moved by s -> s ^ c.
template <typename M, uint32_t Dim>
__device__ __forceinline__ M slot_xor_perm(M L, uint32_t c) {
#pragma unroll
  for (uint32_t k = 0; k < Dim; ++k)
    if ((c >> k) & 1u) {
      const M B = slot_bit_mask<M>(k);
      const uint32_t sh = 1u << k;
      L = ((L & B) >> sh) | ((L & ~B) << sh);
    }
  return L;
}
__device__ __forceinline__ uint32_t spar(uint32_t s, uint32_t g) { return (uint32_t)__popc(s & g) & 1u; }
template <int W>
__device__ __forceinline__ bool wnonzero(const uint64_t *x) {
  uint64_t o = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) o |= x[w];
  return o != 0ull;
}
template <typename R, int W, uint32_t Cap>
struct LaneShot {
  static constexpr uint32_t kDim = lane_dim(Cap);
  static_assert(Cap == (1u << kDim), "a lane holds a cube of slots");
  static constexpr uint32_t kRowB = 1, kRowD = 1 + kDim;  // rows: alpha0, B[0..kDim), Dual[0..kDim)
  using Mask = typename SlotSet<Cap>::T;  // a set of the cube's slots
  const ShotParams &P;
  const CircDev *C;
  uint32_t lane;
  Cx<R> *vals;     // [slot][lane]
  uint64_t *rows;  // [row][w][lane]
  uint64_t *rec;   // [w][lane]
  // per-lane shot state
  uint64_t shot;
  uint32_t d;
  Mask live;
  uint64_t sd[W], ss[W];
  NoiseCursor nc;
  int status, chain, logical, lastm;
  double fid;
  bool force;
  static constexpr bool kScaled = sizeof(R) == 8;  // FP64 maps are scaled (see ScaledPrune)
  double nrm;  // their squared norm

  typename std::conditional<kScaled, ScaledPrune, PruneTest<R>>::type pt;  // |v|^2 < tau

  __device__ LaneShot(const ShotParams &p, unsigned char *base) : P(p), C(&p.circ[0]), nrm(1.0), pt(p.prune) {
    lane = threadIdx.x & 31u;
    const size_t vb = (size_t)Cap * sizeof(Cx<R>) * 32, rb = (size_t)(1 + 2 * kDim) * W * 8 * 32;
    vals = reinterpret_cast<Cx<R> *>(base);
    rows = reinterpret_cast<uint64_t *>(base + vb);
    rec = reinterpret_cast<uint64_t *>(base + vb + rb);
  }

  __device__ __forceinline__ Cx<R> val(uint32_t s) const { return vals[(size_t)s * 32 + lane]; }
  __device__ __forceinline__ void set_val(uint32_t s, Cx<R> v) { vals[(size_t)s * 32 + lane] = v; }
  __device__ __forceinline__ uint64_t row(uint32_t r, int w) const { return rows[((size_t)r * W + w) * 32 + lane]; }
  __device__ __forceinline__ void set_row(uint32_t r, int w, uint64_t x) { rows[((size_t)r * W + w) * 32 + lane] = x; }
  __device__ __forceinline__ void get_row(uint32_t r, uint64_t *x) const {
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = row(r, w);
  }
  __device__ __forceinline__ void put_row(uint32_t r, const uint64_t *x) {
#pragma unroll
    for (int w = 0; w < W; ++w) set_row(r, w, x[w]);
  }
  __device__ __forceinline__ void xor_row(uint32_t r, const uint64_t *x) {
#pragma unroll
    for (int w = 0; w < W; ++w) set_row(r, w, row(r, w) ^ x[w]);
  }
  __device__ __forceinline__ uint32_t row_par(uint32_t r, const uint64_t *g) const {
    uint64_t t = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) t ^= row(r, w) & g[w];
    return wordpar(t);
  }
  __device__ __forceinline__ uint32_t row_bit(uint32_t r, uint32_t p) const {
    return (uint32_t)((row(r, (W == 2 && p >= 64u) ? W - 1 : 0) >> (p & 63u)) & 1ull);
  }
  __device__ __forceinline__ Mask cube() const {
    if (sizeof(Mask) == 4) return (Mask)(d >= 5u ? 0xFFFFFFFFu : (1u << (1u << d)) - 1u);
    return (Mask)(d >= 6u ? ~0ull : (1ull << (1u << d)) - 1ull);
  }
  __device__ __forceinline__ uint32_t nnz() const { return mpopc(live); }
  // the slots whose key has gamma . key = 1 (gl, g0: gamma's parities with the basis and
  // alpha0): computed once per event, an entry's parity is then one shift instead of a
  // population count (with the folded word parities, w42 FP32 at 2^24 shots: 23.4 -> 20.5 ms)
  __device__ __forceinline__ Mask par_mask(uint32_t gl, uint32_t g0) const {
    const Mask m = slot_par_mask<Mask, kDim>(gl);
    return g0 ? ~m : m;
  }
  __device__ __forceinline__ static uint32_t in_mask(Mask m, uint32_t s) { return (uint32_t)(m >> s) & 1u; }

  // g . alpha0 into g0; bit k of the result: g . B[k]
  __device__ uint32_t parities(const uint64_t *g, uint32_t &g0) const {
    g0 = row_par(0, g);
    uint32_t m = 0;
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k) m |= row_par(kRowB + k, g) << k;
    return m;
  }
  // coordinates c of x (bit k: Dual[k] . x) and the residual r = x ^ XOR_{k in c} B[k],
  // zero iff x lies in the span (otherwise Dual[k] . r = 0 for every k)
  __device__ uint32_t coords(const uint64_t *x, uint64_t *r) const {
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) r[w] = x[w];
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k)
      if (row_par(kRowD + k, x)) {
        c |= 1u << k;
#pragma unroll
        for (int w = 0; w < W; ++w) r[w] ^= row(kRowB + k, w);
      }
    return c;
  }
  // z with z . B[k] = 0 for every k and z . r = 1, for a residual r (nonzero, Dual[k] . r = 0):
  // e_p ^ XOR_k B[k][p] Dual[k] for the lowest set bit p of r
  __device__ __forceinline__ void co_dual(const uint64_t *r, uint64_t *z) const {
    const uint32_t p = wlow<W>(r);
#pragma unroll
    for (int w = 0; w < W; ++w) z[w] = ((int)(p >> 6) == w) ? (1ull << (p & 63u)) : 0ull;
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k)
      if (row_bit(kRowB + k, p)) {
#pragma unroll
        for (int w = 0; w < W; ++w) z[w] ^= row(kRowD + k, w);
      }
  }
  // B[d] = r, a residual; the old duals stay dual
  __device__ void add_dim(const uint64_t *r) {
    uint64_t z[W];
    co_dual(r, z);
    put_row(kRowB + d, r);
    put_row(kRowD + d, z);
    ++d;
  }
  // Every live slot s has parity(s & g) = t, and g has bit q set (q < d): bit q of a live
  // slot follows from the others, so the map needs one coordinate less. alpha0 ^= t B[q],
  // B[k] ^= B[q] for the other k of g; B[q] and Dual[q] go (the other duals stay dual);
  // each live slot drops bit q of its index.
  __device__ void remove_dim(uint32_t q, uint32_t g, uint32_t t) {
    remove_rows(q, g, t);
    const uint32_t lo = (1u << q) - 1u;
    Mask nl = 0;
#pragma unroll 1
    for (Mask m = live; m; m &= m - (Mask)1) {  // ascending: a slot moves down onto a vacated one
      const uint32_t s = mffs(m) - 1, s2 = (s & lo) | ((s >> (q + 1u)) << q);
      if (s2 != s) set_val(s2, val(s));
      nl |= (Mask)1 << s2;
    }
    live = nl;
  }
  // the rows' part of remove_dim (d decreases); the caller moves the slots
  __device__ void remove_rows(uint32_t q, uint32_t g, uint32_t t) {
    uint64_t bq[W];
    get_row(kRowB + q, bq);
    if (t) xor_row(0, bq);
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k)
      if (k != q && ((g >> k) & 1u)) xor_row(kRowB + k, bq);
#pragma unroll 1
    for (uint32_t k = q; k + 1u < d; ++k) {
      uint64_t x[W];
      get_row(kRowB + k + 1u, x);
      put_row(kRowB + k, x);
      get_row(kRowD + k + 1u, x);
      put_row(kRowD + k, x);
    }
    --d;
  }
  // after a measurement: all live slots share parity(s & g); drop a coordinate if g != 0
  __device__ __forceinline__ void restrict_to(uint32_t g) {
    g &= (d >= 32u) ? 0xFFFFFFFFu : ((1u << d) - 1u);
    if (!g || !live) return;
    const uint32_t t = spar(mffs(live) - 1, g);
    remove_dim(31u - __clz(g), g, t);
  }
  // Drop the coordinates that the live slots' affine span does not need: any g with the
  // same parity(s & g) for every live slot s removes its highest coordinate. Cancelled
  // entries leave such slanted flats as often as unused coordinates: with unused ones
  // alone dropped, 1 shot in 6 of the 97-qubit workload left its lane although its
  // entries spanned no more than the lane's directions (FP32, 2 M shots: 45.9 -> 26.9 ms
  // with the span; w42's hand-overs fall too). gl, g0: parities that follow the
  // rows. Constraints below 2^q do not involve the coordinates that a removal moves, so
  // the scan goes on at 2^q.
  __device__ void compact_span(uint32_t &gl, uint32_t &g0) {
    uint32_t g = 1;
#pragma unroll 1
    while (g < (1u << d)) {
      const Mask x = live & slot_par_mask<Mask, kDim>(g);
      if (x && x != live) {
        ++g;
        continue;
      }
      const uint32_t q = 31u - __clz(g), lo = (1u << q) - 1u, t = x ? 1u : 0u;
      if ((gl >> q) & 1u) {
        gl ^= g & lo;
        g0 ^= t;
      }
      gl = (gl & lo) | ((gl >> (q + 1u)) << q);
      remove_dim(q, g, t);
      g = 1u << q;
    }
  }
  // key of slot s
  __device__ Key<W> key_of(uint32_t s) const {
    Key<W> k;
#pragma unroll
    for (int w = 0; w < W; ++w) k.w[w] = row(0, w);
#pragma unroll 1
    for (uint32_t j = 0; j < d; ++j)
      if ((s >> j) & 1u) {
#pragma unroll
        for (int w = 0; w < W; ++w) k.w[w] ^= row(kRowB + j, w);
      }
    return k;
  }
  __device__ void fail_capacity() { status = P.small_pass ? LS_RERUN : LS_OVF; }
  __device__ void fail_check(uint32_t code, uint64_t value) {
    status = LS_ERR;
    if (P.diag && atomicAdd(&P.diag[0], 1ull) == 0ull) {
      P.diag[1] = ((unsigned long long)code << 32);
      P.diag[2] = shot;
      P.diag[3] = value;
    }
  }

  __device__ __forceinline__ int pick(uint32_t ord, double sp, double sm) {
    return pick_outcome<true>(P.seed, shot, ord, sp, sm, force, fid, nullptr);
  }
  __device__ __forceinline__ R inv_sqrt(double x) const {
    if (sizeof(R) == 4) return (R)rsqrtf((float)x);
    return (R)rsqrt(x);
  }

  __device__ __forceinline__ void fetch_row(uint32_t r, const uint64_t *src) {
#pragma unroll
    for (int w = 0; w < W; ++w) copy_async<8>(&rows[((size_t)r * W + w) * 32 + lane], src + w);
  }
  __device__ __forceinline__ void fetch_val(uint32_t s, const Cx<R> *src) {
    copy_async<(int)sizeof(Cx<R>)>(&vals[(size_t)s * 32 + lane], src);
  }
  // ---- start at event e of the noiseless run (its map in affine form, computed once per
  // snapshot when the circuit was compiled): everything but the shot's own cursor. The map
  // goes to the lane's columns in asynchronous copies (complete after copies_done()), issued
  // before the claim's atomic has answered
  __device__ void begin(uint32_t e) {
    status = LS_RUN;
    force = false;
    nrm = 1.0;
    const unsigned char *in = C->traj + (size_t)e * C->traj_stride;
    const SnapHdr *h = reinterpret_cast<const SnapHdr *>(in);
    const uint64_t *r_in = reinterpret_cast<const uint64_t *>(in + sizeof(SnapHdr));
    const SnapAffine<R, W> *a = reinterpret_cast<const SnapAffine<R, W> *>(in + snap_affine_off<R, W>(C->rw));
    const uint2 dl = __ldg(reinterpret_cast<const uint2 *>(&a->d));  // d and the low word of live
    const uint4 h0 = __ldg(reinterpret_cast<const uint4 *>(h));
    chain = (int)h0.y;
    logical = (int)h0.z;
    lastm = (int)h0.w;
    fid = __ldg(&h->fid);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] = __ldg(&h->sd[w]);
      ss[w] = __ldg(&h->ss[w]);
    }
    live = 0;
    d = 0;
    if (dl.x > kDim) {
      fail_capacity();
      return;
    }
    d = dl.x;
    live = (Mask)dl.y;  // (no slot at or above 2^kDim is live)
    if (sizeof(Mask) == 8) live |= (Mask)__ldg(&a->live_hi) << 16 << 16;
#pragma unroll 1
    for (uint32_t s = 0; s < (1u << d); ++s) fetch_val(s, &a->v[s]);
    fetch_row(0, a->rows[0]);
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k) {
      fetch_row(kRowB + k, a->rows[1 + k]);
      fetch_row(kRowD + k, a->rows[1 + kSnapDim + k]);
    }
#pragma unroll 1
    for (uint32_t w = 0; w < C->rw; ++w) copy_async<8>(&rec[(size_t)w * 32 + lane], &r_in[w]);
  }
  __device__ __forceinline__ void start(uint64_t s, const uint4 &cursor) {
    shot = s;
    nc = NoiseCursor{cursor.x, cursor.y, cursor.z};
    if (cursor.z == 0xFFFFFFFFu) status = LS_ERR;
  }

  // ---- eviction: the shot's whole state into record r, to resume at event ev
  __device__ void evict(const Spill<R, W> &S, uint32_t r, uint32_t item, uint32_t ev) const {
    unsigned char *p = S.at(r);
    S.ha(p) = make_uint4(item, ev, (uint32_t)live, S.meta(d, chain, logical, lastm));
    S.hb(p) = make_uint4(nc.first, nc.second, nc.kblk, sizeof(Mask) == 8 ? (uint32_t)((unsigned long long)live >> 32) : 0u);
    S.fid(p) = fid;
    if constexpr (kScaled) S.norm(p) = nrm;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      S.sd(p)[w] = sd[w];
      S.ss(p)[w] = ss[w];
    }
#pragma unroll 1
    for (uint32_t w = 0; w < C->rw; ++w) S.rec(p)[w] = rec[(size_t)w * 32 + lane];
    uint64_t *q = S.rows(p);
#pragma unroll 1
    for (uint32_t k = 0; k <= d; ++k)
#pragma unroll
      for (int w = 0; w < W; ++w) {
        q[k * W + w] = row(k, w);
        if (k < d) q[(1 + S.dim + k) * W + w] = row(kRowD + k, w);
      }
    Cx<R> *qv = S.vals(p);
#pragma unroll 1
    for (Mask m = live; m; m &= m - (Mask)1) qv[mffs(m) - 1] = val(mffs(m) - 1);
  }
  // ---- resumption from record r (asynchronous copies, as begin); returns the shot's item
  // (chunk-local index)
  __device__ uint32_t resume(const Spill<R, W> &S, uint32_t r, uint64_t first) {
    unsigned char *p = S.at(r);
    const uint4 a = S.ha(p), b = S.hb(p);
    shot = first + a.x;
    status = LS_RUN;
    force = false;
    chain = (int)((a.w >> 8) & 1u);
    logical = (int)((a.w >> 9) & 1u);
    lastm = (int)(int8_t)((a.w >> 16) & 255u);
    nc = NoiseCursor{b.x, b.y, b.z};
    fid = S.fid(p);
    if constexpr (kScaled) nrm = S.norm(p);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] = S.sd(p)[w];
      ss[w] = S.ss(p)[w];
    }
#pragma unroll 1
    for (uint32_t w = 0; w < C->rw; ++w) copy_async<8>(&rec[(size_t)w * 32 + lane], S.rec(p) + w);
    d = 0;
    live = 0;
    const uint32_t rd = a.w & 255u;
    if (rd > S.dim || rd > kDim) {  // a record never holds more; checked so that a bad record cannot index past the map
      fail_check(CHK_NNZ, rd);
      return a.x;
    }
    d = rd;
    live = (Mask)a.z;
    if (sizeof(Mask) == 8) live |= (Mask)b.w << 16 << 16;
    live &= cube();
    const uint64_t *q = S.rows(p);
    fetch_row(0, q);
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k) {
      fetch_row(kRowB + k, q + (1 + k) * W);
      fetch_row(kRowD + k, q + (1 + S.dim + k) * W);
    }
#pragma unroll 1
    for (Mask m = live; m; m &= m - (Mask)1) fetch_val(mffs(m) - 1, S.vals(p) + (mffs(m) - 1));
    return a.x;
  }
  // ---- the shot's final state (signs, keys, values) for state capture at offset off; ph: the
  // circuit's global phase where it ended
  __device__ void capture(uint64_t off, uint32_t ph) const {
    Cx<double> f{1.0, 0.0};
    if constexpr (kScaled) f = readout(ph, nrm);
    P.st_nnz[off] = nnz();
    P.st_signs[off * 4 + 0] = sd[0];
    P.st_signs[off * 4 + 1] = (W == 2) ? sd[W - 1] : 0ull;
    P.st_signs[off * 4 + 2] = ss[0];
    P.st_signs[off * 4 + 3] = (W == 2) ? ss[W - 1] : 0ull;
    uint32_t i = 0;
#pragma unroll 1
    for (Mask m = live; m && i < P.st_stride; m &= m - (Mask)1, ++i) {
      const uint32_t s = mffs(m) - 1;
      const Key<W> k = key_of(s);
      Cx<R> v = val(s);
      if constexpr (kScaled) v = cmul(f, v);
      const size_t o = (size_t)off * P.st_stride + i;
      P.st_keys[2 * o] = k.w[0];
      P.st_keys[2 * o + 1] = (W == 2) ? k.w[W - 1] : 0ull;
      P.st_vals[2 * o] = (double)v.x;
      P.st_vals[2 * o + 1] = (double)v.y;
    }
  }

  // ---- Paulis: v'_{a^beta} = i^{e + 2 gamma.a} v_a: phases per entry, then alpha0 moves
  __device__ void apply_pauli(const uint64_t *beta, const uint64_t *gamma, uint32_t e) {
    uint32_t g0;
    const uint32_t gl = parities(gamma, g0);
    const Mask odd = par_mask(gl, g0);
#pragma unroll 1
    for (Mask m = live; m; m &= m - (Mask)1) {
      const uint32_t s = mffs(m) - 1;
      set_val(s, ipow(val(s), e + 2u * in_mask(odd, s)));
    }
    xor_row(0, beta);
  }
  __device__ void apply_error(uint32_t s) {
    if (s >= C->n_sites) {
      fail_check(CHK_SITE, s);
      return;
    }
    uint64_t beta[W], gamma[W];
    const uint32_t e = site_pauli<W>(C, s, nc.pair(), sd, ss, beta, gamma);
    apply_pauli(beta, gamma, nc.phase(e));
  }

  // (rare: many rotations, or very unlikely outcomes, since the last sampled outcome)
  __device__ __forceinline__ void fit_norm() {
    for (int k = 0; k < 32 && !ScaledPrune::in_range(nrm); ++k) {  // (bounded: an empty map has norm 0)
      const double f = ScaledPrune::fit(nrm);
#pragma unroll 1
      for (Mask m = live; m; m &= m - (Mask)1) set_val(mffs(m) - 1, cscale(val(mffs(m) - 1), (R)f));
      nrm = nrm * f * f;
    }
  }
  // ---- a I + b Z_q: v'_a = a v_a + b xi_{a^beta} v_{a^beta}; xi = i^e (-1)^{gamma.key}
  // folded into b (b or -b per entry, exact), and a diagonal rotation (beta = 0) is one
  // product (a + b xi) v per entry. gl, g0: gamma's parities with the basis and alpha0 on
  // entry (they follow the basis through the changes made here).
  __device__ void rot(uint32_t w0, uint32_t ci, const uint64_t *beta, const uint64_t *gamma, bool diag, uint32_t gl,
                      uint32_t g0) {
    const uint32_t pe = wpar2<W>(sd, beta, ss, gamma);  // (beta = 0 when diagonal)
    const uint32_t e = (ev_e0(w0) + 2u * pe) & 3u;
    if (ci >= C->n_coef) {
      fail_check(CHK_COEF, ci);
      return;
    }
    const Coef *cf = C->coef + ci;
    Cx<R> a{0, 0}, bq{0, 0}, bn{0, 0};  // FP32: a, and b with the phase folded in, and its negation
    double k = 0.0, cm = 1.0;           // FP64: v' = cm v + i^{e + 3} k (-1)^{gamma.key} v_partner
    if constexpr (!kScaled) {
      const float4 f = __ldg(reinterpret_cast<const float4 *>(&cf->fa_re));
      a = Cx<R>{(R)f.x, (R)f.y};
      bq = ipow(Cx<R>{(R)f.z, (R)f.w}, e);
      bn = Cx<R>{negr(bq.x), negr(bq.y)};
    } else {
      const double2 kc = __ldg(reinterpret_cast<const double2 *>(&cf->k));
      k = kc.x;
      cm = kc.y;
    }
    const bool plain = kScaled && __double2hiint(cm) != 0x3FF00000;
    const ScaledTurn turn(k, (e + 3u) & 3u);
    auto base = [&](Cx<R> v) { return plain ? cscale(v, (R)cm) : v; };
    // the norm takes its factor once the event is certain to happen
    auto scale = [&]() {
      if constexpr (kScaled) {
        if (!plain) nrm = mulr(nrm, __ldg(&cf->n2));
        fit_norm();
        pt.set(nrm);
      }
    };
    auto small = [&](Cx<R> v) {
      if constexpr (kScaled) return pt.small(v, nrm);
      else return pt.small(v);
    };
    Mask drop = 0;
    if (diag) {
      const Cx<R> c0 = kScaled ? a : cadd(a, bq), c1 = kScaled ? a : cadd(a, bn);
      const Mask odd = par_mask(gl, g0);
      scale();
#pragma unroll 1
      for (Mask m = live; m; m &= m - (Mask)1) {
        const uint32_t s = mffs(m) - 1;
        Cx<R> nv = val(s);
        if constexpr (kScaled) nv = turn.add(base(nv), nv, in_mask(odd, s));
        else nv = cmul(in_mask(odd, s) ? c1 : c0, nv);
        const bool sm = small(nv);
        if (!sm) set_val(s, nv);
        drop |= (Mask)sm << s;
      }
      live &= ~drop;
      return;
    }
    uint64_t r[W];
    uint32_t c;
    bool fresh;
#pragma unroll 1
    for (uint32_t pass = 0;; ++pass) {
      c = coords(beta, r);
      fresh = wnonzero<W>(r);  // beta outside the span: every entry gains a partner
      if (!fresh || d < kDim) break;
      if (pass) {
        // the map would outgrow the lane: nothing has been written yet, so the shot can be
        // taken over at the top of this event (by the wide round's lanes, or a warp);
        // otherwise (the wide round) it reruns in a warp
        if (P.lane_hand && P.sp && P.small_pass && C->cap > Cap) status = LS_HAND;
        else fail_capacity();
        return;
      }
      compact_span(gl, g0);
    }
    if (fresh) {
      add_dim(r);
      c |= 1u << (d - 1u);
      gl |= row_par(kRowB + d - 1u, gamma) << (d - 1u);
    }
    const Mask odd = par_mask(gl, g0);
    const Mask spread = live | slot_xor_perm<Mask, kDim>(live, c);
    const Mask lead = spread & ~slot_bit_mask<Mask>(__ffs(c) - 1) & cube();  // one member of each pair
    scale();
#pragma unroll 1
    for (Mask m = lead; m; m &= m - (Mask)1) {
      const uint32_t s = mffs(m) - 1, t = s ^ c;
      const uint32_t ls = in_mask(live, s), lt = in_mask(live, t);
      const Cx<R> vs = ls ? val(s) : Cx<R>{0, 0}, vt = lt ? val(t) : Cx<R>{0, 0};
      Cx<R> ns, nt;
      if constexpr (kScaled) {
        ns = base(vs);
        nt = base(vt);
        if (lt) ns = turn.add(ns, vt, in_mask(odd, t));  // (skipped by a warp whose entries gain partners)
        if (ls) nt = turn.add(nt, vs, in_mask(odd, s));
      } else {
        // one fused chain per component; with a zero partner it rounds as the single product
        const Cx<R> bs = in_mask(odd, s) ? bn : bq, bt = in_mask(odd, t) ? bn : bq;
        ns = cmad2(a, vs, bt, vt);
        nt = cmad2(a, vt, bs, vs);
      }
      const bool ss_ = small(ns), st_ = small(nt);
      if (!ss_) set_val(s, ns);
      if (!st_) set_val(t, nt);
      drop |= ((Mask)ss_ << s) | ((Mask)st_ << t);
    }
    live = spread & ~drop;
    if (nnz() > C->cap) status = LS_OVF;  // the overflow rule, for circuits whose cap is below the lane's
  }

  // ---- measurement of P, beta = 0: lambda_a = c (-1)^{gamma.a}; gl, g0: gamma's parities
  // with the basis and alpha0
  __device__ int meas_a(uint32_t w0, uint32_t ord, const uint64_t *gamma, const uint32_t gl, const uint32_t g0) {
    const uint32_t e = (ev_e0(w0) + 2u * wpar<W>(ss, gamma)) & 3u;
    if (e & 1u) {
      fail_check(CHK_PHASE, e);
      return 1;
    }
    const uint32_t sgn = e >> 1;
    const Mask pm = slot_par_mask<Mask, kDim>(gl) & cube();
    const Mask neg = live & (((sgn ^ g0) & 1u) ? ~pm : pm);  // slots with eigenvalue -1
    const Mask pos = live & ~neg;
    int m;
    R sc = (R)1;
    Mask keep;
    if (!neg || !pos) {  // decided (all eigenvalues equal): integer test only, no scaling
      m = neg ? -1 : 1;
      keep = live;
      if (!gl || !live) return m;
    } else {
      double sp = 0.0, sm = 0.0;
      if constexpr (kScaled) {  // two fused multiply-adds per entry, one side after the other
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
          double acc = 0.0;
#pragma unroll 1
          for (Mask mm = side ? neg : pos; mm; mm &= mm - (Mask)1) {
            const Cx<R> v = val(mffs(mm) - 1);
            acc = __fma_rn((double)v.x, (double)v.x, __fma_rn((double)v.y, (double)v.y, acc));
          }
          sp = side ? sp : acc;
          sm = acc;
        }
      } else {
#pragma unroll 1
        for (Mask mm = live; mm; mm &= mm - (Mask)1) {
          const uint32_t s = mffs(mm) - 1;
          const double a2 = pnorm(val(s));
          if ((neg >> s) & 1u) sm += a2;
          else sp += a2;
        }
      }
      m = pick(ord, sp, sm);
      if constexpr (kScaled) nrm = m == 1 ? sp : sm;
      else sc = inv_sqrt(m == 1 ? sp : sm);
      keep = (m == 1) ? pos : neg;
    }
    // the kept slots share parity(s & gl) = t, so bit q of their index is redundant; each is
    // scaled straight into its slot of the restricted map. A decided outcome goes through
    // the same loop with the scale 1 (exact; no kept value is below tau), so that the
    // restriction is inlined once (w42 FP32: 676 -> 708 M shots/s)
    const uint32_t q = 31u - __clz(gl), lo = (1u << q) - 1u, t = spar(mffs(keep) - 1, gl);
    Mask nl = 0;
#pragma unroll 1
    for (Mask mm = keep; mm; mm &= mm - (Mask)1) {  // ascending: a write lands on a slot already read
      const uint32_t s = mffs(mm) - 1, s2 = (s & lo) | ((s >> (q + 1u)) << q);
      if constexpr (kScaled) {  // (normalising raises every entry: none falls below tau)
        set_val(s2, val(s));
        nl |= (Mask)1 << s2;
      } else {
        const Cx<R> v = cscale(val(s), sc);
        if (!pt.small(v)) {
          set_val(s2, v);
          nl |= (Mask)1 << s2;
        }
      }
    }
    if (nl) remove_rows(q, gl, t);
    live = nl;
    return m;
  }

  // ---- measurement of P, beta != 0 (case B): row operations on the signs, relabel,
  // pairing, replacement
  __device__ int meas_b(uint32_t ord, uint32_t cbi) {
    if (cbi >= C->n_cb) {
      fail_check(CHK_CASEB, cbi);
      return 1;
    }
    const CaseB *B = C->cb + cbi;
    const uint32_t p = __ldg(&B->p);
    uint64_t J[W], g2[W], ep[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      J[w] = __ldg(&B->J[w]);
      g2[w] = __ldg(&B->gamma2[w]);
      ep[w] = ((int)(p >> 6) == w) ? (1ull << (p & 63)) : 0ull;
    }
    const uint32_t ssp = wbit<W>(ss, p);
    const uint32_t sdJ = wpar<W>(sd, J);
#pragma unroll
    for (int w = 0; w < W; ++w) ss[w] ^= (ssp ? J[w] : 0ull) ^ __ldg(&B->Hs[w]);
    if (sdJ ^ __ldg(&B->hdp)) wflip<W>(sd, p);
    const uint32_t e2 = (__ldg(&B->e0b) + 2u * (wbit<W>(sd, p) + wpar<W>(ss, g2))) & 3u;
    // relabel a_j ^= a_p (j in J), a linear map L of the keys: alpha0 and every B[k] go
    // through it, and the duals through its transpose (D ^= (D . J) e_p; L is its own inverse)
#pragma unroll 1
    for (uint32_t k = 0; k <= d; ++k) {
      const uint32_t rr = k == 0 ? 0u : kRowB + k - 1u;
      if (row_bit(rr, p)) xor_row(rr, J);
    }
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k)
      if (row_par(kRowD + k, J)) xor_row(kRowD + k, ep);
    // pair a0 (key bit p clear) with a1 = a0 ^ e_p: first the outcome probabilities, then
    // the combined values (v0 + m x1) / sqrt(2 p_m), x1 = xi_{a1} v_{a1}
    uint32_t g20;
    const uint32_t gl2 = parities(g2, g20);
    const Mask odd = par_mask(gl2, g20);
    uint32_t bp = 0;  // bit k: B[k][p]
#pragma unroll 1
    for (uint32_t k = 0; k < d; ++k) bp |= row_bit(kRowB + k, p) << k;
    const Mask cb = cube();
    const Mask kb = (row_bit(0, p) ? ~slot_par_mask<Mask, kDim>(bp) : slot_par_mask<Mask, kDim>(bp)) & cb;  // slots whose key has bit p
    uint64_t rr[W];
    const uint32_t c = coords(ep, rr);
    const bool lone = wnonzero<W>(rr);  // e_p outside the span: no entry has a partner
    const Mask spread = lone ? live : (live | slot_xor_perm<Mask, kDim>(live, c));
    const Mask lead = lone ? live : (spread & ~kb);  // a0 members (lone: every entry)
    int m;
    Mask nl = 0;
    if constexpr (kScaled) {
      if (lone) {
        // every entry stays, those with key bit p as m xi v: p = 1/2 exactly, so the outcome is
        // one random bit and the norm stays
        m = force ? 1 : (philox<true>(P.seed, shot, 1u, ord).x >> 31) ? -1 : 1;
        if (force) fid *= 0.5;
#pragma unroll 1
        for (Mask mm = live & kb; mm; mm &= mm - (Mask)1) {
          const uint32_t s = mffs(mm) - 1;
          set_val(s, ipow(val(s), e2 + 2u * in_mask(odd, s) + (m == -1 ? 2u : 0u)));
        }
        nl = live;
      } else {
        // sp, sm = (N +- 2 C) / 2 with N the pairs' norm and C = sum Re conj(v0) x1; the kept
        // side's own norm is summed from the values it keeps
        double sn = 0.0, cr = 0.0;
#pragma unroll 1
        for (Mask mm = lead; mm; mm &= mm - (Mask)1) {
          const uint32_t s = mffs(mm) - 1, t = s ^ c;
          Cx<R> v0{0, 0}, x1{0, 0};
          if (in_mask(live, s)) v0 = val(s);
          if (in_mask(live, t)) x1 = ipow(val(t), e2 + 2u * in_mask(odd, t));
          sn = fmar((double)v0.x, (double)v0.x, fmar((double)v0.y, (double)v0.y, sn));
          sn = fmar((double)x1.x, (double)x1.x, fmar((double)x1.y, (double)x1.y, sn));
          cr = fmar((double)v0.x, (double)x1.x, fmar((double)v0.y, (double)x1.y, cr));
        }
        const double sp = fmar(0.5, sn, cr), sm = fmar(0.5, sn, -cr);
        m = pick(ord, sp, sm);
        nrm = 2.0 * (m == 1 ? sp : sm);
        fit_norm();
        pt.set(nrm);
        const uint32_t flip = m == -1 ? 2u : 0u;
        double kn = 0.0;
#pragma unroll 1
        for (Mask mm = lead; mm; mm &= mm - (Mask)1) {
          const uint32_t s = mffs(mm) - 1, t = s ^ c;
          Cx<R> v0{0, 0}, x1{0, 0};
          if (in_mask(live, s)) v0 = val(s);
          if (in_mask(live, t)) x1 = ipow(val(t), e2 + flip + 2u * in_mask(odd, t));
          const Cx<R> nv = cadd(v0, x1);
          kn = fmar((double)nv.x, (double)nv.x, fmar((double)nv.y, (double)nv.y, kn));
          if (!pt.small(nv, nrm)) {
            set_val(s, nv);
            nl |= (Mask)1 << s;
          }
        }
        nrm = kn;
      }
    } else {
      double sp = 0.0, sm = 0.0;
#pragma unroll 1
      for (Mask mm = lead; mm; mm &= mm - (Mask)1) {
        const uint32_t s = mffs(mm) - 1;
        Cx<R> v0{0, 0}, x1{0, 0};
        if (lone) {
          if (in_mask(kb, s)) x1 = ipow(val(s), e2 + 2u * in_mask(odd, s));
          else v0 = val(s);
        } else {
          const uint32_t t = s ^ c;
          if (in_mask(live, s)) v0 = val(s);
          if (in_mask(live, t)) x1 = ipow(val(t), e2 + 2u * in_mask(odd, t));
        }
        sp += 0.5 * pnorm(cadd(v0, x1));
        sm += 0.5 * pnorm(csub(v0, x1));
      }
      m = pick(ord, sp, sm);
      const R sc = inv_sqrt(2.0 * (m == 1 ? sp : sm));
#pragma unroll 1
      for (Mask mm = lead; mm; mm &= mm - (Mask)1) {
        const uint32_t s = mffs(mm) - 1;
        Cx<R> v0{0, 0}, x1{0, 0};
        if (lone) {
          if (in_mask(kb, s)) x1 = ipow(val(s), e2 + 2u * in_mask(odd, s));
          else v0 = val(s);
        } else {
          const uint32_t t = s ^ c;
          if (in_mask(live, s)) v0 = val(s);
          if (in_mask(live, t)) x1 = ipow(val(t), e2 + 2u * in_mask(odd, t));
        }
        const Cx<R> nv = cscale(m == 1 ? cadd(v0, x1) : csub(v0, x1), sc);
        if (!pt.small(nv)) {
          set_val(s, nv);
          nl |= (Mask)1 << s;
        }
      }
    }
    live = nl;
    if (lone) {
      // every key loses bit p (a1 keys become a1 ^ e_p); injective on the space since e_p is
      // not in the span, so the slots stay. With z . B[k] = 0 for every k and z[p] = 1 (the dual
      // of e_p's residual), D[k] ^= D[k][p] z clears bit p of the duals and keeps them dual
      uint64_t z[W];
      co_dual(rr, z);
#pragma unroll 1
      for (uint32_t k = 0; k < d; ++k)
        if (row_bit(kRowD + k, p)) xor_row(kRowD + k, z);
#pragma unroll 1
      for (uint32_t k = 0; k <= d; ++k) {
        const uint32_t r2 = k == 0 ? 0u : kRowB + k - 1u;
        if (row_bit(r2, p)) xor_row(r2, ep);
      }
    } else {
      restrict_to(bp);  // the kept keys have bit p clear: parity(s & bp) = alpha0[p]
    }
    // replacement: d_j <- d_j s_p (j in G), d_p <- old s_p, s_p <- m P
#pragma unroll
    for (int w = 0; w < W; ++w) sd[w] ^= (ssp ? __ldg(&B->G[w]) : 0ull) ^ __ldg(&B->Hd[w]);
    if (wbit<W>(sd, p) != ssp) wflip<W>(sd, p);
    const uint32_t newsp = (m == -1 ? 1u : 0u) ^ __ldg(&B->rP);
    if (wbit<W>(ss, p) != newsp) wflip<W>(ss, p);
    return m;
  }

  __device__ uint32_t rec_bit(int32_t r) const {
    return (r < 0 || (uint32_t)r >= 64u * C->rw) ? 0u : (uint32_t)((rec[(size_t)(r >> 6) * 32 + lane] >> (r & 63)) & 1ull);
  }

  // one event for this lane's shot
  __device__ void step(uint32_t ev, const uint4 &hdr, const uint64_t *body, const Ev<W> *E) {
    while (nc.site() < hdr.y && status == LS_RUN) {
      apply_error(nc.site());
      if (!nc.template advance<true>(C, P.seed, shot)) status = LS_ERR;
    }
    if (status != LS_RUN) return;
    const uint64_t *dsd = body, *dss = body + W, *beta = body + 2 * W, *gamma = body + 3 * W;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] ^= dsd[w];
      ss[w] ^= dss[w];
    }
    const uint32_t w0 = hdr.x, type = ev_type(w0), flags = ev_flags(w0);
    // gamma's parities with alpha0 and the basis, once for the event types that use them.
    // This kernel is bound by instruction fetch, so each helper is inlined at as few sites as
    // possible: one parity computation here instead of one per handler, one rotation handler
    // for both kinds, and the handlers in a chain of tests in order of frequency (a `break`
    // leaves the chain) rather than a jump table (w42: FP32 660 -> 675 M shots/s, FP64
    // 352 -> 382 M).
    uint32_t g0 = 0, gl = 0;
    if (type == EV_ROT || type == EV_ROT_DIAG || type == EV_MEAS_A) gl = parities(gamma, g0);
    do {
      if (type == EV_MEAS_A || type == EV_MEAS_B) {
        force = P.fid_mode && (flags & F_FIDELITY);
        const int m = (type == EV_MEAS_A) ? meas_a(w0, hdr.z, gamma, gl, g0) : meas_b(hdr.z, (uint32_t)beta[0]);
        if (status != LS_RUN) break;
        if (force && m == -1) {
          fid = 0.0;
          status = LS_KEPT;
          break;
        }
        lastm = m;
        if (flags & F_RECORD) {
          const uint32_t r = hdr.w;
          if (r >= 64u * C->rw) {
            fail_check(CHK_RECORD, r);
            break;
          }
          if (m < 0) rec[(size_t)(r >> 6) * 32 + lane] |= 1ull << (r & 63);
        }
        if ((flags & F_COND_LAST) && m == -1) {
          uint64_t xb[W], xg[W];
#pragma unroll
          for (int w = 0; w < W; ++w) {
            xb[w] = __ldg(&E->xbeta[w]);
            xg[w] = __ldg(&E->xgamma[w]);
          }
          apply_pauli(xb, xg, (ev_xe0(w0) + 2u * wpar2<W>(sd, xb, ss, xg)) & 3u);
        }
        if ((flags & F_DETECTOR) && ((m == -1 ? 1u : 0u) ^ ((flags & F_INVERT) ? 1u : 0u))) status = LS_DISC;
        break;
      }
      if (type == EV_ROT || type == EV_ROT_DIAG) {
        rot(w0, hdr.z, beta, gamma, type == EV_ROT_DIAG, gl, g0);
        break;
      }
      if (type == EV_PAULI) {
        uint32_t cond;
        if (flags & F_COND_LAST) cond = (lastm == -1);
        else cond = rec_bit((int32_t)hdr.z) ^ rec_bit((int32_t)hdr.w);
        if (cond) {
          apply_pauli(beta, gamma, (ev_e0(w0) + 2u * wpar2<W>(sd, beta, ss, gamma)) & 3u);
        }
        break;
      }
      if (type == EV_PARITY) {
        const int par = chain ^ (int)rec_bit((int32_t)hdr.z) ^ (int)rec_bit((int32_t)hdr.w) ^
                        ((flags & F_INVERT) ? 1 : 0);
        if (flags & F_CHAIN) {
          chain = par;
        } else {
          chain = 0;
          if ((flags & F_DETECTOR) && par) status = LS_DISC;
          if ((flags & F_OBSERVABLE) && par) logical = 1;
        }
        break;
      }
    } while (false);
    if (status == LS_HAND) {  // back to the top of the event: the signs as before its XOR
#pragma unroll
      for (int w = 0; w < W; ++w) {
        sd[w] ^= dsd[w];
        ss[w] ^= dss[w];
      }
    }
    (void)ev;
  }
};

// ---- the affine form (SnapAffine) of every valid snapshot of a noiseless run (events
// [0, stop[0]]), a warp per snapshot, once per compiled circuit and precision; the
// largest dimension goes to stop[3] (0xFF where a map needs more than kSnapDim). Each direction is
// found by all keys at once, their residuals in registers, two a lane (w42 FP64 26 -> 5.6 us, w97
// 77 -> 7.8 against a thread per snapshot with its rows in local memory).
template <typename R, int W>
__global__ void __launch_bounds__(128) snap_affine_kernel(unsigned char *traj, uint32_t n_snap, uint32_t stride, uint32_t rw,
                                                          uint32_t *stop, const void *ev) {
  static_assert(kSnapMax == 64, "two keys a lane");
  const uint32_t e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31u;
  if (e >= n_snap || e > stop[0]) return;
  unsigned char *in = traj + (size_t)e * stride;
  const SnapHdr *h = reinterpret_cast<const SnapHdr *>(in);
  const uint64_t *k_in = reinterpret_cast<const uint64_t *>(in + snap_keys_off(rw));
  const Cx<R> *v_in = reinterpret_cast<const Cx<R> *>(k_in + kSnapMax * W);
  SnapAffine<R, W> *out = reinterpret_cast<SnapAffine<R, W> *>(in + snap_affine_off<R, W>(rw));
  const uint32_t n = h->nnz < kSnapMax ? h->nnz : kSnapMax;
  Cx<R> turn{(R)1, (R)0};  // FP64: the circuit's global phase is taken out (scaled maps)
  if constexpr (sizeof(R) == 8) turn = phase_of(e ? (16u - ev_phase(reinterpret_cast<const Ev<W> *>(ev)[e - 1u].w0)) & 15u : 0u);
  uint64_t a0[W], B[kSnapDim][W], D[kSnapDim][W], r[2][W];  // r: the keys' residuals
#pragma unroll
  for (int w = 0; w < W; ++w) {
    a0[w] = n ? k_in[w] : 0ull;
#pragma unroll
    for (int i = 0; i < 2; ++i) r[i][w] = lane + 32u * i < n ? k_in[(lane + 32u * i) * W + w] ^ a0[w] : 0ull;
  }
  uint32_t d = 0, c[2] = {0, 0};
  bool done = false, ok = true;
  // the first key outside the span, in the map's order, is the next direction
#pragma unroll
  for (uint32_t j = 0; j <= kSnapDim; ++j) {
    const uint32_t m0 = __ballot_sync(0xFFFFFFFFu, wnonzero<W>(r[0])), m1 = __ballot_sync(0xFFFFFFFFu, wnonzero<W>(r[1]));
    const uint32_t m = m0 ? m0 : m1, src = m ? 31u - (uint32_t)__clz((int)(m & (0u - m))) : 0u;
    done = done || !m;
    if (j == kSnapDim) {
      ok = done;
      break;
    }
    uint64_t x[W], z[W];
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = __shfl_sync(0xFFFFFFFFu, (unsigned long long)(m0 ? r[0][w] : r[1][w]), src);
    const uint32_t p = done ? 0u : wlow<W>(x);  // its dual (as in LaneShot::add_dim)
#pragma unroll
    for (int w = 0; w < W; ++w) z[w] = !done && (int)(p >> 6) == w ? 1ull << (p & 63u) : 0ull;
#pragma unroll
    for (uint32_t k = 0; k < j; ++k)
      if (!done && wbit<W>(B[k], p))
#pragma unroll
        for (int w = 0; w < W; ++w) z[w] ^= D[k][w];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      B[j][w] = x[w];  // (zero once done)
      D[j][w] = z[w];
    }
    d += done ? 0u : 1u;
#pragma unroll
    for (int i = 0; i < 2; ++i)  // (residuals lie outside the span so far: its duals are zero on them)
      if (wpar<W>(z, r[i])) {
        c[i] |= 1u << j;
#pragma unroll
        for (int w = 0; w < W; ++w) r[i][w] ^= x[w];
      }
  }
  uint32_t live[2] = {0, 0};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    out->v[lane + 32u * i] = Cx<R>{0, 0};
    if (lane + 32u * i < n) live[c[i] >> 5] |= 1u << (c[i] & 31u);
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (lane + 32u * i < n) out->v[c[i]] = sizeof(R) == 8 ? cmul(turn, v_in[lane + 32u * i]) : v_in[lane + 32u * i];
  const uint32_t lo = __reduce_or_sync(0xFFFFFFFFu, live[0]), hi = __reduce_or_sync(0xFFFFFFFFu, live[1]);
  if (lane == 0) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      out->rows[0][w] = a0[w];
#pragma unroll
      for (uint32_t k = 0; k < kSnapDim; ++k) {
        out->rows[1 + k][w] = B[k][w];
        out->rows[1 + kSnapDim + k][w] = D[k][w];
      }
    }
    out->d = ok ? d : 0xFFFFFFFFu;
    out->live_lo = lo;
    out->live_hi = hi;
    atomicMax(&stop[3], ok ? d : 0xFFu);
  }
}

// ---- the fate of each site's errors, once per compiled circuit and precision.
// Before its first error a shot is the noiseless run. An error E commutes past every event that
// leaves it alone: a rotation whose generator commutes with it, a decided measurement whose
// outcome it does not flip (its corrections commuting with E too), a parity of unflipped
// records. Up to such an event the shot is E applied to the noiseless run's state there, to
// rounding: E permutes and phases the entries exactly, and rotations round alike on values times
// i^k; but the state comes from the sparse kernel's form of the maps (FP64: unscaled), and the norm
// that decides on pruning rounds differently for a value and i times it. So the shot may start at
// the first event that does not leave E alone, and if that
// is a measurement with a detector on it, E flips it and the shot ends there, discarded: the
// pre-pass finishes such shots without running them (60 % of w42's and w97's; the others
// start 10 to 20 events later; events run per shot: w42 25.7 -> 10.7, w97 46 -> 13.4). Two errors
// are carried to the earlier of their events (start_event).
// Entry: that event (at most the recorded run's last), kFateDiscard, and E's phase i^e relative to
// the signed rows, which the Clifford gates in between leave as it is.
// A warp takes a site and tests 32 events at once, a lane each: whether the event leaves an error
// alone is linear in its generators' images, so one look at an event serves all 15 pairs (w42: 70 ->
// 15 us against a thread per site and pair that walks event by event, each step a load's latency;
// w97 141 -> 46).
template <int W>
__global__ void __launch_bounds__(128) fate_kernel(const __grid_constant__ CircDev C, const uint32_t *stop_at, uint32_t *out) {
  const uint32_t s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31u, pp = lane & 15u;
  if (s >= C.n_sites) return;
  const SiteDev<W> *S = reinterpret_cast<const SiteDev<W> *>(C.sites) + s;
  const uint32_t at = __ldg(&C.site_ev[s]), stop = *stop_at < C.n_events ? *stop_at : C.n_events;
  // lane pp: its pair's event and kind, and the errors' phase (others are no errors, or never used)
  const bool error = lane < 16u && pp && ((__ldg(&S->kind) & 3u) == SITE_DEPOL2 || !(pp & 3u)) && at <= stop;
  uint32_t e = error ? stop : at, kind = 0;
  if (error) {
    const SnapHdr *h = reinterpret_cast<const SnapHdr *>(C.traj + (size_t)at * C.traj_stride);
    uint64_t b[W], g[W], sd[W], ss[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      sd[w] = h->sd[w];
      ss[w] = h->ss[w];
    }
    kind = site_pauli<W>(&C, s, pp, sd, ss, b, g) << 30;
  }
  uint64_t img[4][2 * W];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int w = 0; w < 2 * W; ++w) img[j][w] = __ldg(&S->img[j][w]);
  const Ev<W> *evs = reinterpret_cast<const Ev<W> *>(C.ev);
  uint32_t open = __ballot_sync(0xFFFFFFFFu, error);
  for (uint32_t base = at; base < stop && open; base += 32) {
    const uint32_t k = base + lane;
    uint32_t flip = 0, turn = 0;  // per generator: it anticommutes with the event, with its correction
    bool halt = false, ends = false;
    if (k < stop) {
      const Ev<W> *E = evs + k;
      const uint32_t w0 = __ldg(&E->w0), type = ev_type(w0), flags = ev_flags(w0);
      uint64_t be[W], ga[W];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        be[w] = __ldg(&E->beta[w]);
        ga[w] = __ldg(&E->gamma[w]);
      }
      if (type == EV_ROT || type == EV_ROT_DIAG) {
#pragma unroll
        for (int j = 0; j < 4; ++j) flip |= wpar2<W>(be, img[j] + W, ga, img[j]) << j;
      } else if (type == EV_MEAS_A) {
        ends = (flags & F_DETECTOR) != 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) flip |= wpar<W>(ga, img[j]) << j;
        if ((flags & F_COND_LAST) &&  // the noiseless run applies the correction
            (int)reinterpret_cast<const SnapHdr *>(C.traj + (size_t)(k + 1u) * C.traj_stride)->lastm == -1) {
          uint64_t xb[W], xg[W];
#pragma unroll
          for (int w = 0; w < W; ++w) {
            xb[w] = __ldg(&E->xbeta[w]);
            xg[w] = __ldg(&E->xgamma[w]);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) turn |= wpar2<W>(xb, img[j] + W, xg, img[j]) << j;
        }
      } else {
        halt = type != EV_PARITY && type != EV_END;
      }
    }
    for (uint32_t m = open; m; m &= m - 1u) {
      const uint32_t q = 31u - (uint32_t)__clz((int)(m & (0u - m))), need = site_images(q);
      const bool f = (__popc(flip & need) & 1) != 0;
      const uint32_t hit = __ballot_sync(0xFFFFFFFFu, halt || f || (__popc(turn & need) & 1)), end = __ballot_sync(0xFFFFFFFFu, ends && f);
      if (hit) {
        const uint32_t first = hit & (0u - hit);
        if (lane == q) {
          e = base + (31u - (uint32_t)__clz((int)first));
          kind |= (end & first) ? kFateDiscard : 0u;
        }
        open &= ~(1u << q);
      }
    }
  }
  if (lane < 16u) out[(size_t)s * 16 + pp] = e | kind;
}

// ---- bucketing pre-pass. Buckets: per circuit of the run, one per event plus one
// (shots that start past the end), circuit after circuit from circuit.bucket0.
// The circuit of item g: the last one whose item range starts at or before g.
__device__ __forceinline__ uint32_t circ_of_item(const ShotParams &P, uint64_t g) {
  uint32_t lo = 0, hi = P.n_circ;
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (P.circ[mid].item_begin <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}
// The circuit of bucket g: the last one whose first bucket is at or before g.
__device__ __forceinline__ uint32_t circ_of_bucket(const ShotParams &P, uint32_t g) {
  uint32_t lo = 0, hi = P.n_circ;
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    if (P.circ[mid].bucket0 <= g) lo = mid;
    else hi = mid;
  }
  return lo;
}
// Exclusive scan of the bucket sizes by one block of 1024 threads: each thread sums a contiguous
// range, the warps scan their sums by shuffles (a serial pass over 1024 partial sums took 7 us).
__device__ void scan_buckets(const ShotParams &P) {
  __shared__ uint32_t part[32];
  const uint32_t nb = P.al_nb, tid = threadIdx.x, nt = blockDim.x, ln = tid & 31u;
  const uint32_t per = (nb + nt - 1) / nt, lo = tid * per < nb ? tid * per : nb, hi = lo + per < nb ? lo + per : nb;
  uint32_t sum = 0;
  for (uint32_t k = lo; k < hi; ++k) sum += P.al_count[k];
  auto scan = [&](uint32_t v) {  // inclusive, over the warp
#pragma unroll
    for (uint32_t off = 1; off < 32; off <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, v, off);
      if (ln >= off) v += u;
    }
    return v;
  };
  const uint32_t inc = scan(sum);
  if (ln == 31u) part[tid / 32] = inc;
  __syncthreads();
  if (tid < 32) part[tid] = scan(tid < nt / 32 ? part[tid] : 0u);
  __syncthreads();
  uint32_t run = inc - sum + (tid >= 32 ? part[tid / 32 - 1] : 0u);
  if (tid == nt - 1) P.al_start[nb] = run + sum;
  for (uint32_t k = lo; k < hi; ++k) {
    P.al_start[k] = run;
    run += P.al_count[k];
  }
}
__global__ void __launch_bounds__(1024) lane_scan_kernel(const __grid_constant__ ShotParams P) { scan_buckets(P); }
// ---- round r >= 1: its records are those taken since round r - 1 began (the pool's
// count, capped at its capacity: reservations past it were not written)
__device__ __forceinline__ void round_setup(const ShotParams &P) {
  const uint32_t r = P.lane_round;
  if (P.lane_wide_round) {  // the wide round: the handed-over shots' records
    const unsigned long long cap = P.sp_cap - P.sp_evict_cap;
    P.lr[2 + 2 * r] = P.sp_evict_cap;
    P.lr[3 + 2 * r] = P.lr[1] < cap ? P.lr[1] : cap;
    return;
  }
  for (uint32_t k = 0; k < P.rs_n; ++k) {
    unsigned long long *lr = P.rs_lr[k];
    const unsigned long long used = lr[0] < P.rs_cap[k] ? lr[0] : P.rs_cap[k];
    const unsigned long long first = r == 1 ? 0ull : lr[2 + 2 * (r - 1)] + lr[3 + 2 * (r - 1)];
    lr[2 + 2 * r] = first;
    lr[3 + 2 * r] = used > first ? used - first : 0ull;
  }
}
// the items of a resume pre-pass: the round's records of every pool
__device__ __forceinline__ unsigned long long resumed_items(const ShotParams &P) {
  unsigned long long n = 0;
  for (uint32_t k = 0; k < P.rs_n; ++k) n += P.rs_lr[k][3 + 2 * P.lane_round];
  return n;
}
// item i's pool; i becomes its number within the pool
__device__ __forceinline__ uint32_t resumed_pool(const ShotParams &P, unsigned long long &i) {
  uint32_t k = 0;
  while (k + 1u < P.rs_n && i >= P.rs_lr[k][3 + 2 * P.lane_round]) i -= P.rs_lr[k++][3 + 2 * P.lane_round];
  return k;
}
__global__ void lane_round_setup_kernel(const __grid_constant__ ShotParams P) { round_setup(P); }
// ---- block-binned pre-pass: each block ranks its contiguous range of items per
// bucket with shared-memory atomics, then takes one global atomic per non-empty
// bucket for its base. The first errors cluster in a few buckets, and global
// atomics on one address serialise.
// Items of circuits whose maps outgrow a lane go to the warp pass's list instead: the
// block ranks them too and reserves their slots with one global atomic.
// Shots that their first errors discard are finished here (start_event): their status, their
// record (the noiseless run's, with the failing measurement's bit flipped) and their count.
constexpr uint32_t kResolved = 0xFFFFFFFEu;  // as a bucket
template <bool Resume, typename R, int W>
__device__ __forceinline__ void bin_items(const ShotParams &P, uint32_t *hist) {
  const uint32_t nb = P.al_nb;
  uint32_t *ended = hist + nb + 1;  // per circuit: shots discarded here
  for (uint32_t k = threadIdx.x; k <= nb + (Resume ? 0u : P.n_circ); k += blockDim.x) hist[k] = 0u;
  __syncthreads();
  const unsigned long long n_items =
      Resume ? resumed_items(P) : (P.n_items_dev ? *P.n_items_dev : P.n_items);
  const unsigned long long per = (n_items + gridDim.x - 1) / gridDim.x;
  const unsigned long long i0 = blockIdx.x * per, i1 = i0 + per < n_items ? i0 + per : n_items;
  const unsigned long long base = P.item_base_dev ? *P.item_base_dev : P.item_base;
  for (unsigned long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    uint32_t e;
    const CircDev *C;
    if (Resume) {
      unsigned long long j = i;
      const uint32_t k = resumed_pool(P, j);
      const Spill<R, W> S(P.rs_sp[k], P.rw_max, P.rs_dim[k]);
      const uint4 a = S.ha(S.at((uint32_t)(P.rs_lr[k][2 + 2 * P.lane_round] + j)));
      C = &P.circ[circ_of_item(P, base + a.x)];
      e = a.y < C->n_events ? a.y : C->n_events;  // a record always resumes at an event of its circuit
    } else {
      const uint32_t ci = circ_of_item(P, base + i);
      C = &P.circ[ci];
      // the shot's first error and the one after it: nearly every shot applies the first as it
      // starts, and here all lanes of a warp draw
      uint32_t cur = 0, nxt = 0, pp = 0, n2 = 0, p2 = 0;
      NoiseCursor nc{0, 0, 0};
      const uint64_t off = base + i - C->item_begin, shot = C->first_shot + off;
      bool ok = next_site(C, P.seed, shot, cur, nc.kblk, nxt, pp);
      if (ok && nxt != 0xFFFFFFFFu) ok = next_site(C, P.seed, shot, cur, nc.kblk, n2, p2);
      else n2 = 0xFFFFFFFFu;
      nc.first = pack_error(nxt, pp);
      nc.second = pack_error(n2, p2);
      if (!ok) nc = NoiseCursor{kMaxPackedSites, kMaxPackedSites, 0xFFFFFFFFu};
      bool resolved = false;
      e = start_event(C, P.fid_mode, P.seed, shot, nc, ok && !(ci == 0u && off < P.st_limit), resolved);
      if (resolved) {
        reinterpret_cast<uint2 *>(P.al_ev)[i] = make_uint2(kResolved, 0u);
        atomicAdd(&ended[ci], 1u);
        if (off < C->out_limit) {
          if (C->status) C->status[off] = (uint8_t)LS_DISC;
          if (C->records) {
            const Ev<W> *E = reinterpret_cast<const Ev<W> *>(C->ev) + e;
            const uint32_t r = __ldg(&E->b);
            const uint64_t *rec = reinterpret_cast<const uint64_t *>(C->traj + (size_t)e * C->traj_stride + sizeof(SnapHdr));
            const bool one = !(ev_flags(__ldg(&E->w0)) & F_INVERT);  // the outcome that fails the detector
            for (uint32_t w = 0; w < C->rw; ++w)
              C->records[off * C->rw + w] = __ldg(&rec[w]) | (one && w == (r >> 6) ? 1ull << (r & 63u) : 0ull);
          }
        }
        continue;
      }
      reinterpret_cast<uint4 *>(P.al_cursor)[i] = make_uint4(nc.first, nc.second, nc.kblk, e);
      if (C->lanes_off) {
        reinterpret_cast<uint2 *>(P.al_ev)[i] = make_uint2(kNoRecord, atomicAdd(&hist[nb], 1u));
        continue;
      }
    }
    e += C->bucket0;
    reinterpret_cast<uint2 *>(P.al_ev)[i] = make_uint2(e, atomicAdd(&hist[e], 1u));
  }
  __syncthreads();
  for (uint32_t k = threadIdx.x; k < nb; k += blockDim.x) {
    const uint32_t c = hist[k];
    P.al_base[(size_t)blockIdx.x * (nb + 1) + k] = c ? atomicAdd(&P.al_count[k], c) : 0u;
  }
  if (threadIdx.x == 0)
    P.al_base[(size_t)blockIdx.x * (nb + 1) + nb] = hist[nb] ? (uint32_t)atomicAdd(P.n_rerun, (unsigned long long)hist[nb]) : 0u;
  if (!Resume)
    for (uint32_t k = threadIdx.x; k < P.n_circ; k += blockDim.x)
      if (ended[k]) {
        atomicAdd(&P.circ[k].tally[0], (unsigned long long)ended[k]);
        atomicAdd(&P.circ[k].tally[1], (unsigned long long)ended[k]);
      }
}
template <bool Resume, typename R, int W>
__global__ void __launch_bounds__(256) lane_bin_kernel(const __grid_constant__ ShotParams P) {
  extern __shared__ uint32_t hist[];  // nb buckets, then the block's count of warp-pass items
  bin_items<Resume, R, W>(P, hist);
}
// (same grid as lane_bin_kernel: it fixes each item's block)
template <bool Resume>
__device__ __forceinline__ void scatter_items(const ShotParams &P) {
  const uint32_t nb = P.al_nb;
  const unsigned long long n_items =
      Resume ? resumed_items(P) : (P.n_items_dev ? *P.n_items_dev : P.n_items);
  const unsigned long long per = (n_items + gridDim.x - 1) / gridDim.x;
  const unsigned long long i0 = blockIdx.x * per, i1 = i0 + per < n_items ? i0 + per : n_items;
  for (unsigned long long i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const uint2 er = reinterpret_cast<const uint2 *>(P.al_ev)[i];
    if (er.x == kResolved) continue;
    if (er.x == kNoRecord) {  // a shot of a circuit without lanes: the warp pass's list
      const unsigned long long slot = P.al_base[(size_t)blockIdx.x * (nb + 1) + nb] + er.y;
      if (slot < P.rerun_cap) P.rerun[slot] = (uint32_t)i;
      continue;
    }
    const uint32_t at = P.al_start[er.x] + P.al_base[(size_t)blockIdx.x * (nb + 1) + er.x] + er.y;
    if (Resume) {
      unsigned long long j = i;
      resumed_pool(P, j);
      P.al_order[at] = (uint32_t)j;
    } else {
      const uint4 k = reinterpret_cast<const uint4 *>(P.al_cursor)[i];
      reinterpret_cast<uint4 *>(P.al_rec)[at] = make_uint4(k.x, k.y, k.z, (uint32_t)i);
    }
  }
}

template <bool Resume>
__global__ void __launch_bounds__(256) lane_bin_scatter_kernel(const __grid_constant__ ShotParams P) {
  scatter_items<Resume>(P);
}
// The whole pre-pass in one block, for few items: a launch instead of three (four with the
// round's setup), which cost more than the work (6-qubit circuit, 4096 shots: 18 + 17 us).
template <bool Resume, typename R, int W>
__global__ void __launch_bounds__(1024, 1) lane_bin_one_kernel(const __grid_constant__ ShotParams P) {
  extern __shared__ uint32_t hist[];
  if (Resume) {
    if (threadIdx.x == 0) round_setup(P);
    __syncthreads();
  }
  bin_items<Resume, R, W>(P, hist);
  __syncthreads();
  scan_buckets(P);
  __syncthreads();
  scatter_items<Resume>(P);
}

// Register budget: resident blocks per SM the compiler must allow. FP32 16-slot lanes: 8
// (64 registers; the shared memory allows 8 on w42; measured 617 M shots/s against 604 M
// at 6 blocks and 76 registers); 32-slot lanes (blocks of 2 warps): 8 in FP32, 4 in FP64,
// which leave the registers they use (shared memory allows 9 and 5); 64-slot lanes: 2;
// FP64 16-slot lanes: 5 (its shared memory allows 5; 272.8 M against 266.7 M at 4).
template <typename R, uint32_t Cap>
constexpr int kLaneMinBlocks() {
  return sizeof(R) == 4 ? (Cap <= 16 ? 8 : Cap <= 32 ? 8 : 2) : (Cap == 32 ? 4 : 5);
}

// Multi: the run holds several circuits (a warp serves one at a time); the single-
// circuit instantiation keeps circuit 0 and bucket offset 0 as constants. Cap: map
// entries per lane (kLaneCap in the first rounds, kWideCap in the wide round, or
// kWideCap / kLaneBigCap as the first pass of circuits with larger noiseless maps).
template <typename R, int W, bool Multi, uint32_t Cap>
__global__ void __launch_bounds__(lane_block<Cap>(), kLaneMinBlocks<R, Cap>()) lane_kernel(const __grid_constant__ ShotParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t warp = threadIdx.x / 32, lane = threadIdx.x & 31u;
  LaneShot<R, W, Cap> s(P, smem + (size_t)warp * lane_warp_bytes<R, W, Cap>(P.rw_max));
  const unsigned long long base = P.item_base_dev ? *P.item_base_dev : P.item_base;
  const unsigned long long n_items =
      P.lane_round ? P.lr[3 + 2 * P.lane_round] : (P.n_items_dev ? *P.n_items_dev : P.n_items);
  const unsigned long long rec0 = P.lane_round ? P.lr[2 + 2 * P.lane_round] : 0ull;
  const Spill<R, W> S(P.sp, P.rw_max, P.sp_dim);
  // a batch's launch serves the buckets [P.al_lo, P.al_hi) of its lane map size's circuits
  // (read from the launch parameters where used, so that no register holds them through the
  // loop); a single circuit's, all of them
  if (Multi && P.al_hi <= P.al_lo) return;
  // one bit per bucket: a warp of this block found it exhausted
  uint32_t *empty = reinterpret_cast<uint32_t *>(smem + (size_t)(blockDim.x / 32) * lane_warp_bytes<R, W, Cap>(P.rw_max));
  for (uint32_t k = threadIdx.x; k < (P.al_nb + 31u) / 32u; k += blockDim.x) empty[k] = 0u;
  __syncthreads();
  // warps start spread evenly over the buckets, so that they meet buckets that still hold shots
  const unsigned long long gw = (unsigned long long)blockIdx.x * (blockDim.x / 32) + warp;
  const unsigned long long nw = (unsigned long long)gridDim.x * (blockDim.x / 32);
  uint32_t g = (Multi ? P.al_lo : 0u) + (uint32_t)((gw * (unsigned long long)(Multi ? P.al_hi - P.al_lo : P.al_nb)) / nw);
  uint32_t ci = Multi ? circ_of_bucket(P, g) : 0u;
  const CircDev *C = &P.circ[ci];
  uint32_t n_ev = C->n_events, e = Multi ? g - C->bucket0 : g;
  const Ev<W> *evs = reinterpret_cast<const Ev<W> *>(C->ev);
  s.C = C;
  // the warp's tallies of its current circuit, lane k counter k (shots, discarded, overflow,
  // kept, logical), counted by ballots; added to the circuit's when the warp moves to another
  // circuit and at the end
  uint32_t cnt = 0;
  auto flush = [&]() {
    if (lane < 5 && cnt) atomicAdd(&C->tally[lane], (unsigned long long)cnt);
    cnt = 0;
  };
  bool active = false;
  uint32_t item = 0;
  uint32_t from = kNoRecord;  // wide round: the shot's hand-over record, from which a warp may run it again
  // the current bucket: its first record and the next bucket's
  uint32_t b0 = __ldg(&P.al_start[g]), b1 = __ldg(&P.al_start[g + 1]);
  const unsigned long long limit = (n_items + 2ull) * ((Multi ? P.al_hi - P.al_lo : P.al_nb) + 2ull) + 64ull;
  for (unsigned long long guard = 0; guard < limit; ++guard) {
    g = Multi ? C->bucket0 + e : e;
    // the event's header and body, loaded before the claims so that their latency overlaps
    // the claims' (w42 FP32: 710.8 -> 715.0 M shots/s)
    const Ev<W> *E = evs + e;
    uint4 hdr = make_uint4(0u, 0u, 0u, 0u);
    uint64_t body[4 * W];
#pragma unroll
    for (int k = 0; k < 4 * W; ++k) body[k] = 0ull;
    if (e < n_ev) {  // (no event past the last)
      hdr = __ldg(reinterpret_cast<const uint4 *>(E));
      const ulonglong2 *bp = reinterpret_cast<const ulonglong2 *>(&E->dsd[0]);
#pragma unroll
      for (int k = 0; k < 2 * W; ++k) {
        const ulonglong2 v = __ldg(bp + k);
        body[2 * k] = v.x;
        body[2 * k + 1] = v.y;
      }
    }
    // idle lanes claim shots that start at event e of circuit ci (one atomic per warp). The
    // snapshot's copies are issued before the atomic answers: a lane that gets no shot has
    // only filled columns that nobody reads.
    const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !active);
    bool claim = idle && b1 != b0;
    if (claim) {
      // (other warps change both words meanwhile, so the lanes may read different values: the warp
      // decides as one, by a vote)
      bool shut = ((*(volatile uint32_t *)&empty[g >> 5] >> (g & 31u)) & 1u) != 0u;
      if (!shut && *(volatile unsigned int *)&P.al_next[g] >= b1 - b0) {  // once per block and bucket
        if (lane == 0) atomicOr(&empty[g >> 5], 1u << (g & 31u));
        shut = true;
      }
      claim = !__any_sync(0xFFFFFFFFu, shut);
    }
    if (claim) {
      uint32_t got0 = 0;
      const uint32_t leader = __ffs(idle) - 1;
      if (lane == leader) got0 = atomicAdd(&P.al_next[g], __popc(idle));
      if (!active && !P.lane_round) s.begin(e);
      got0 = __shfl_sync(0xFFFFFFFFu, got0, leader);
      if (!active) {
        const uint32_t k = got0 + __popc(idle & ((1u << lane) - 1u));
        if (k < b1 - b0) {
          const uint64_t first = C->first_shot + base - (Multi ? C->item_begin : 0ull);  // shot of item i: first + i
          if (P.lane_round) {
            item = __ldg(&P.al_order[b0 + k]);
            if (item < n_items) {
              active = true;
              if (Cap == kWideCap && P.lane_wide_round) from = (uint32_t)(rec0 + item);
              item = s.resume(S, (uint32_t)(rec0 + item), first);
            }
          } else {
            const uint4 rc = __ldg(reinterpret_cast<const uint4 *>(P.al_rec) + (b0 + k));
            item = rc.w;
            if (item < n_items) {
              active = true;
              s.start(first + item, rc);
            }
          }
        }
      }
      copies_done();
    }
    if (e < n_ev && __any_sync(0xFFFFFFFFu, active && s.status == LS_RUN)) {
      if (active && s.status == LS_RUN) s.step(e, hdr, body, E);
    }
    // the end of the next bucket, used when the warp walks on
    const uint32_t b2 = __ldg(&P.al_start[g + 2u < P.al_nb ? g + 2u : P.al_nb]);
    // a spill record to write (a hand-over or an eviction), written once below
    uint32_t ev_r = 0xFFFFFFFFu, ev_e = 0;
    // finish: ended, or past the last event
    const bool done = active && (s.status != LS_RUN || e + 1u >= n_ev);
    if (__any_sync(0xFFFFFFFFu, done)) {
      if (done && s.status == LS_RUN) s.status = LS_KEPT;
      const bool out = done && s.status < LS_RERUN;  // (the others run again, or go on, in a later pass)
      {
        const uint32_t all = __ballot_sync(0xFFFFFFFFu, out), kept = __ballot_sync(0xFFFFFFFFu, out && s.status == LS_KEPT);
        const uint32_t disc = __ballot_sync(0xFFFFFFFFu, out && s.status == LS_DISC);
        const uint32_t ovf = __ballot_sync(0xFFFFFFFFu, out && s.status == LS_OVF);
        const uint32_t log = __ballot_sync(0xFFFFFFFFu, out && s.status == LS_KEPT && s.logical);
        cnt += __popc(lane == 0 ? all : lane == 1 ? disc : lane == 2 ? ovf : lane == 3 ? kept : lane == 4 ? log : 0u);
      }
      if (out) {
        const uint64_t off = base + item - (Multi ? C->item_begin : 0ull);  // the shot's offset within its circuit
        if (P.fid_mode && s.status == LS_KEPT && C->fsum) atomicAdd(C->fsum, s.fid);
        if (!Multi && off < P.st_limit) s.capture(off, top_phase<W>(C, e < n_ev ? e + 1u : n_ev));
        if (off < C->out_limit) {
          if (C->status) C->status[off] = (uint8_t)s.status;
          if (C->records)
#pragma unroll 1
            for (uint32_t w = 0; w < C->rw; ++w) C->records[off * C->rw + w] = s.rec[(size_t)w * 32 + lane];
        }
      } else if (done) {
        uint32_t entry = item;  // a rerun starts the shot again from its start (or its hand-over)
        if (Cap == kWideCap && from != kNoRecord) entry = kSpillRef | from;
        bool listed = true;
        if (s.status == LS_HAND) {  // or it resumes from its state at the top of event e
          const unsigned long long h = atomicAdd(&P.lr[1], 1ull);
          if (h < (unsigned long long)(P.sp_cap - P.sp_evict_cap)) {
            const uint32_t r = P.sp_evict_cap + (uint32_t)h;
            ev_r = r;
            ev_e = e;
            entry = kSpillRef | r;    // in a warp, from the rerun list,
            listed = !P.lane_wide;    // or in the wide round, which takes every such record
          }
        }
        if (listed) {
          const unsigned long long i = atomicAdd(P.n_rerun, 1ull);
          if (i < P.rerun_cap) P.rerun[i] = entry;
        }
        if (P.n_rerun_total) atomicAdd(P.n_rerun_total, 1ull);
      }
      if (done) active = false;
    }
    // few active lanes: their shots go to the spill pool (when it has room), to resume in
    // the next round packed with others, and the warp moves on to fresh shots
    if (P.lane_evict || P.lane_tail) {
      const uint32_t am = __ballot_sync(0xFFFFFFFFu, active);
      bool out = (uint32_t)__popc(am) <= P.lane_evict;  // or few warps are left (every 8th event: the read waits)
      // (a vote: lanes may read different values of the counter)
      if ((e & 7u) == 0u && P.lane_tail)
        out = __any_sync(0xFFFFFFFFu, out || *(volatile unsigned int *)P.lane_done >= P.lane_tail);
      if (am && out && e + 1u < n_ev) {
        const uint32_t leader = __ffs(am) - 1;
        unsigned long long r0 = 0;
        const bool again = !P.sp || (Cap > kLaneCap && P.lane_round);  // no record to write
        if (lane == leader) r0 = atomicAdd(again ? P.n_rerun : &P.lr[0], (unsigned long long)__popc(am));
        r0 = __shfl_sync(0xFFFFFFFFu, r0, leader);
        if (active) {
          const unsigned long long r = r0 + __popc(am & ((1u << lane) - 1u));
          if (again) {  // (only with lane_list) the warp pass runs them from their start, or their hand-over
            if (r < P.rerun_cap) P.rerun[r] = Cap == kWideCap && from != kNoRecord ? kSpillRef | from : item;
            active = false;
          } else if (r < P.sp_evict_cap) {
            ev_r = (uint32_t)r;
            ev_e = e + 1u;
            active = false;
            if (P.lane_list) {
              const unsigned long long i = atomicAdd(P.n_rerun, 1ull);
              if (i < P.rerun_cap) P.rerun[i] = kSpillRef | (uint32_t)r;
            }
          }
          if (!active && P.lane_list && P.n_rerun_total) atomicAdd(P.n_rerun_total, 1ull);
        }
      }
    }
    if (ev_r != 0xFFFFFFFFu) s.evict(S, ev_r, item, ev_e);
    uint32_t en = e + 1u > n_ev ? 0u : e + 1u;  // (within the circuit, cyclically)
    if (__any_sync(0xFFFFFFFFu, active)) {
      if (en) {
        b0 = b1;
        b1 = b2;
      }
    } else {
      // all lanes idle: the next bucket of any circuit (cyclically) that still has shots, or
      // stop; 32 buckets per step, one per lane
      uint32_t found = 0xFFFFFFFFu;
      const uint32_t b_lo = Multi ? P.al_lo : 0u, nb = Multi ? P.al_hi - P.al_lo : P.al_nb;
      const uint32_t g1 = (Multi ? C->bucket0 : 0u) + en - b_lo;
      for (uint32_t k = 0; k < nb; k += 32) {
        uint32_t c = g1 + k + lane;
        if (c >= nb) c -= nb;  // (g1 < nb, k + lane < nb where it counts)
        bool has = false;
        if (k + lane < nb) has = *(volatile unsigned int *)&P.al_next[b_lo + c] < __ldg(&P.al_start[b_lo + c + 1]) - __ldg(&P.al_start[b_lo + c]);
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, has);
        if (m) {
          found = __shfl_sync(0xFFFFFFFFu, b_lo + c, __ffs(m) - 1);
          break;
        }
      }
      if (found == 0xFFFFFFFFu) break;
      if (Multi) {
        const uint32_t cn = circ_of_bucket(P, found);
        if (cn != ci) {
          flush();
          ci = cn;
          C = &P.circ[ci];
          n_ev = C->n_events;
          evs = reinterpret_cast<const Ev<W> *>(C->ev);
          s.C = C;
        }
        en = found - C->bucket0;
      } else {
        en = found;
      }
    }
    if (!en || !__any_sync(0xFFFFFFFFu, active)) {  // not the bucket after the last one
      const uint32_t gn = Multi ? C->bucket0 + en : en;
      b0 = __ldg(&P.al_start[gn]);
      b1 = __ldg(&P.al_start[gn + 1]);
    }
    e = en;
  }
  flush();
  if (P.lane_tail && lane == 0) atomicAdd(P.lane_done, 1u);
}

}  // namespace

template <uint32_t Cap>
static size_t lane_smem_bytes_t(int fp32, uint32_t W, uint32_t rw) {
  const size_t per = fp32 ? (W == 1 ? lane_warp_bytes<float, 1, Cap>(rw) : lane_warp_bytes<float, 2, Cap>(rw))
                          : (W == 1 ? lane_warp_bytes<double, 1, Cap>(rw) : lane_warp_bytes<double, 2, Cap>(rw));
  return per * (lane_block<Cap>() / 32);
}
size_t lane_smem_bytes(int fp32, uint32_t W, uint32_t rw, uint32_t cap) {
  return cap == kLaneBigCap ? lane_smem_bytes_t<kLaneBigCap>(fp32, W, rw)
         : cap == kWideCap  ? lane_smem_bytes_t<kWideCap>(fp32, W, rw)
                            : lane_smem_bytes_t<kLaneCap>(fp32, W, rw);
}

uint32_t lane_map_cap() { return kLaneCap; }
uint32_t lane_map_dim() { return lane_dim(kLaneCap); }
uint32_t lane_first_cap(uint32_t max_n, uint32_t max_d, int fp32) {
  if (max_n <= kLaneCap && max_d <= lane_dim(kLaneCap)) return kLaneCap;
  if (max_n <= kWideCap && max_d <= lane_dim(kWideCap)) return kWideCap;
  if (fp32 && max_n <= kLaneBigCap && max_d <= lane_dim(kLaneBigCap)) return kLaneBigCap;
  return 0;
}

cudaError_t launch_snap_affine(unsigned char *traj, uint32_t n_snap, uint32_t rw, int fp32, uint32_t W,
                               uint32_t *stop, const void *ev, cudaStream_t st) {
  const unsigned grid = (n_snap + 3) / 4;
  if (fp32) {
    if (W == 1) snap_affine_kernel<float, 1><<<grid, 128, 0, st>>>(traj, n_snap, (uint32_t)snap_stride<float, 1>(rw), rw, stop, ev);
    else snap_affine_kernel<float, 2><<<grid, 128, 0, st>>>(traj, n_snap, (uint32_t)snap_stride<float, 2>(rw), rw, stop, ev);
  } else {
    if (W == 1) snap_affine_kernel<double, 1><<<grid, 128, 0, st>>>(traj, n_snap, (uint32_t)snap_stride<double, 1>(rw), rw, stop, ev);
    else snap_affine_kernel<double, 2><<<grid, 128, 0, st>>>(traj, n_snap, (uint32_t)snap_stride<double, 2>(rw), rw, stop, ev);
  }
  return cudaGetLastError();
}
cudaError_t launch_fate(const CircDev &c, uint32_t W, const uint32_t *stop, uint32_t *fate, cudaStream_t st) {
  if (!c.n_sites) return cudaSuccess;
  const unsigned grid = (c.n_sites + 3u) / 4u;
  if (W == 1) fate_kernel<1><<<grid, 128, 0, st>>>(c, stop, fate);
  else fate_kernel<2><<<grid, 128, 0, st>>>(c, stop, fate);
  return cudaGetLastError();
}
uint32_t lane_rounds() { return kLaneRounds; }
uint32_t lane_max_buckets() { return kLaneMaxBuckets; }
uint32_t lane_prepass_grid(uint64_t items) {
  if (items <= 8192) return 1;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (uint32_t)std::min<uint64_t>((uint64_t)(sms > 0 ? sms : 1) * 8u, (items + 255) / 256);
}

size_t lane_spill_bytes(int fp32, uint32_t W, uint32_t rw, uint32_t cap, uint32_t dim) {
  return (size_t)cap * (fp32 ? (W == 1 ? Spill<float, 1>::record_bytes(rw, dim) : Spill<float, 2>::record_bytes(rw, dim))
                             : (W == 1 ? Spill<double, 1>::record_bytes(rw, dim) : Spill<double, 2>::record_bytes(rw, dim)));
}

// the histogram of all buckets in shared memory (above 48 KB by the opt-in attribute)
template <bool Resume, typename R, int W>
static cudaError_t launch_bin(const ShotParams &p, cudaStream_t st) {
  const size_t sh = ((size_t)p.al_nb + 1 + p.n_circ) * sizeof(uint32_t);
  if (sh > 48 * 1024) {
    const void *kern = p.al_grid == 1 ? reinterpret_cast<const void *>(lane_bin_one_kernel<Resume, R, W>)
                                      : reinterpret_cast<const void *>(lane_bin_kernel<Resume, R, W>);
    // (the largest that any run asks for: see prepare_lanes)
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)((kLaneMaxBuckets + 1 + kMaxCirc) * sizeof(uint32_t)));
    if (e != cudaSuccess) return e;
  }
  if (p.al_grid == 1) {
    lane_bin_one_kernel<Resume, R, W><<<1, 1024, sh, st>>>(p);
    return cudaGetLastError();
  }
  lane_bin_kernel<Resume, R, W><<<p.al_grid, 256, sh, st>>>(p);
  lane_scan_kernel<<<1, 1024, 0, st>>>(p);
  lane_bin_scatter_kernel<Resume><<<p.al_grid, 256, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_lane_resume_prepass(const ShotParams &p, int fp32, uint32_t W, cudaStream_t st) {
  if (p.al_grid > 1) lane_round_setup_kernel<<<1, 1, 0, st>>>(p);
  if (fp32) return W == 1 ? launch_bin<true, float, 1>(p, st) : launch_bin<true, float, 2>(p, st);
  return W == 1 ? launch_bin<true, double, 1>(p, st) : launch_bin<true, double, 2>(p, st);
}

cudaError_t launch_lane_prepass(const ShotParams &p, uint32_t W, cudaStream_t st) {
  return W == 1 ? launch_bin<false, float, 1>(p, st) : launch_bin<false, float, 2>(p, st);
}

template <uint32_t Cap>
static const void *lane_kernel_for(int fp32, uint32_t W, bool multi) {
  if (fp32)
    return W == 1 ? (multi ? reinterpret_cast<const void *>(lane_kernel<float, 1, true, Cap>)
                           : reinterpret_cast<const void *>(lane_kernel<float, 1, false, Cap>))
                  : (multi ? reinterpret_cast<const void *>(lane_kernel<float, 2, true, Cap>)
                           : reinterpret_cast<const void *>(lane_kernel<float, 2, false, Cap>));
  if constexpr (Cap == kLaneBigCap) {
    return nullptr;  // 64-entry lanes: FP32 only (an FP64 warp's map would not leave room for two blocks)
  } else {
    return W == 1 ? (multi ? reinterpret_cast<const void *>(lane_kernel<double, 1, true, Cap>)
                           : reinterpret_cast<const void *>(lane_kernel<double, 1, false, Cap>))
                  : (multi ? reinterpret_cast<const void *>(lane_kernel<double, 2, true, Cap>)
                           : reinterpret_cast<const void *>(lane_kernel<double, 2, false, Cap>));
  }
}

cudaError_t prepare_lanes(const ShotParams &p, int fp32, uint32_t W, int blocks_per_sm, LaunchCfg *cfg, uint32_t cap) {
  const bool multi = p.n_circ > 1;
  const void *kern = cap == kLaneBigCap ? lane_kernel_for<kLaneBigCap>(fp32, W, multi)
                     : cap == kWideCap  ? lane_kernel_for<kWideCap>(fp32, W, multi)
                                        : lane_kernel_for<kLaneCap>(fp32, W, multi);
  if (!kern) return cudaErrorInvalidConfiguration;
  const size_t smem = lane_smem_bytes(fp32, W, p.rw_max, cap) + (size_t)((p.al_nb + 31u) / 32u) * 4u;
  constexpr int kSmemLimit = 227 * 1024;
  if (smem > kSmemLimit) return cudaErrorInvalidConfiguration;
  // The attribute is the kernel's, not the launch's, and a launch's shared memory depends on its
  // circuits' events and records: a thread that set its own size could lower it under another's
  // launch. So every run sets the same.
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int block = cap == kWideCap ? lane_block<kWideCap>() : kLaneBlock;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, block, smem)) != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  if (blocks_per_sm > 0 && blocks_per_sm < occ) occ = blocks_per_sm;
  cfg->kern = kern;
  cfg->grid = (unsigned)(occ * sms);
  cfg->block = (unsigned)block;
  cfg->smem = smem;
  return cudaSuccess;
}

}  // namespace soft
