// compile.cpp -- host compiler: op list + noise model -> per-shot device program.
//
// One pass over the circuit evolves the X/Z words of the tableau (the part
// that is the same in every shot), accumulates each Clifford gate's sign
// flips into XOR masks, numbers the noise sites of the uniform depolarizing
// model (Sec. III of arxiv 2512.23037) and emits one event per non-Clifford
// step: T/T^dag/Rz (Eq. T_gate), Z measurement (Theorem 1 (2)), conditional
// Paulis, parity checks.
//
// Clifford conjugation is derived from each gate's images of X and Z on its
// qubits (U X U^dag, U Z U^dag); the image of any row follows by Pauli
// multiplication, and its sign bit at zero input sign is the XOR mask entry.
#include "compile.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace soft {
namespace {

inline int pc(uint64_t v) { return __builtin_popcountll(v); }

// i^e X^x Z^z on n <= 128 qubits.
struct Pz {
  uint64_t x[2] = {0, 0}, z[2] = {0, 0};
  int e = 0;
};
struct Row {
  uint64_t x[2] = {0, 0}, z[2] = {0, 0};
};

Pz pmul(const Pz &a, const Pz &b) {
  Pz o;
  int t = 0;
  for (int w = 0; w < 2; ++w) {
    o.x[w] = a.x[w] ^ b.x[w];
    o.z[w] = a.z[w] ^ b.z[w];
    t += pc(a.z[w] & b.x[w]);
  }
  o.e = (a.e + b.e + 2 * t) & 3;
  return o;
}

// The Hermitian Pauli of a row with sign bit 0.
Pz herm(const Row &r) {
  Pz p;
  for (int w = 0; w < 2; ++w) {
    p.x[w] = r.x[w];
    p.z[w] = r.z[w];
  }
  p.e = (pc(r.x[0] & r.z[0]) + pc(r.x[1] & r.z[1])) & 3;
  return p;
}

// Sign bit of a Hermitian Pauli written i^e X^x Z^z; -1 if not Hermitian.
int sign_bit(const Pz &p) {
  int d = (p.e - pc(p.x[0] & p.z[0]) - pc(p.x[1] & p.z[1])) & 3;
  return (d & 1) ? -1 : (d >> 1);
}

Row row_of(const Pz &p) {
  Row r;
  for (int w = 0; w < 2; ++w) {
    r.x[w] = p.x[w];
    r.z[w] = p.z[w];
  }
  return r;
}

inline int bit(const uint64_t *v, uint32_t i) { return (int)((v[i >> 6] >> (i & 63)) & 1u); }
inline void flip(uint64_t *v, uint32_t i) { v[i >> 6] ^= 1ull << (i & 63); }

// Local two-qubit Pauli i^e X^x Z^z (bit 0 = first qubit, bit 1 = second).
struct L2 {
  uint32_t x, z;
  int e;
};
L2 l2mul(L2 a, L2 b) { return {a.x ^ b.x, a.z ^ b.z, (a.e + b.e + 2 * pc(a.z & b.x)) & 3}; }

// Row update table: input nibble (xa, za, xb, zb) -> output nibble, sign flip.
struct GateTab {
  uint8_t out[16];
  uint8_t flipb[16];
};

GateTab make_tab(L2 iXa, L2 iZa, L2 iXb, L2 iZb) {
  GateTab t{};
  for (uint32_t in = 0; in < 16; ++in) {
    uint32_t xa = in & 1, za = (in >> 1) & 1, xb = (in >> 2) & 1, zb = (in >> 3) & 1;
    L2 acc{0, 0, (int)((xa & za) + (xb & zb))};
    if (xa) acc = l2mul(acc, iXa);
    if (za) acc = l2mul(acc, iZa);
    if (xb) acc = l2mul(acc, iXb);
    if (zb) acc = l2mul(acc, iZb);
    int d = (acc.e - pc(acc.x & acc.z)) & 3;
    t.out[in] = (uint8_t)((acc.x & 1) | ((acc.z & 1) << 1) | (((acc.x >> 1) & 1) << 2) | (((acc.z >> 1) & 1) << 3));
    t.flipb[in] = (uint8_t)((d >> 1) | ((d & 1) << 7));  // bit 7 marks an impossible odd phase
  }
  return t;
}

struct Tabs {
  GateTab g[8];
  L2 back[8][4];  // U^dag Q U for Q = X_a, Z_a, X_b, Z_b
  Tabs() {
    const L2 Xa{1, 0, 0}, Za{0, 1, 0}, Xb{2, 0, 0}, Zb{0, 2, 0};
    const L2 inv[8][4] = {{Za, Xa, Xb, Zb},                       // H
                          {L2{1, 1, 3}, Za, Xb, Zb},              // S: X -> -Y backwards
                          {L2{1, 1, 1}, Za, Xb, Zb},              // S^dag: X -> Y backwards
                          {Xa, L2{0, 1, 2}, Xb, Zb},              // X
                          {L2{1, 0, 2}, L2{0, 1, 2}, Xb, Zb},     // Y
                          {L2{1, 0, 2}, Za, Xb, Zb},              // Z
                          {L2{3, 0, 0}, Za, Xb, L2{0, 3, 0}},     // CX
                          {L2{1, 2, 0}, Za, L2{2, 1, 0}, Zb}};    // CZ
    std::memcpy(back, inv, sizeof back);
    g[SOFT_H] = make_tab(Za, Xa, Xb, Zb);
    g[SOFT_S] = make_tab(L2{1, 1, 1}, Za, Xb, Zb);       // X -> Y
    g[SOFT_S_DAG] = make_tab(L2{1, 1, 3}, Za, Xb, Zb);   // X -> -Y
    g[SOFT_X] = make_tab(Xa, L2{0, 1, 2}, Xb, Zb);       // Z -> -Z
    g[SOFT_Y] = make_tab(L2{1, 0, 2}, L2{0, 1, 2}, Xb, Zb);
    g[SOFT_Z] = make_tab(L2{1, 0, 2}, Za, Xb, Zb);       // X -> -X
    g[SOFT_CX] = make_tab(L2{3, 0, 0}, Za, Xb, L2{0, 3, 0});        // Xa -> XaXb, Zb -> ZaZb
    g[SOFT_CZ] = make_tab(L2{1, 2, 0}, Za, L2{2, 1, 0}, Zb);        // Xa -> XaZb, Xb -> ZaXb
  }
};
const Tabs &tabs() {
  static Tabs t;
  return t;
}

// 64 x 64 bit matrix, transposed in place by exchanging blocks of 32, 16, ... 1 bits (the
// recursive method of Warren, Hacker's Delight, sec. 7-3).
void transpose64(uint64_t a[64]) {
  uint64_t m = 0x00000000FFFFFFFFull;
  for (uint32_t j = 32; j; j >>= 1, m ^= m << j)
    for (uint32_t k = 0; k < 64; k = (k + j + 1) & ~j) {
      const uint64_t t = ((a[k] >> j) ^ a[k + j]) & m;
      a[k] ^= t << j;
      a[k + j] ^= t;
    }
}

struct Tableau {
  uint32_t n = 0;
  // The tableau by columns (per qubit: bit i of xd is row d_i's X bit there): a gate is a few
  // word operations. Rows are taken from them where products of rows are needed.
  struct Col {
    uint64_t xd[2] = {0, 0}, zd[2] = {0, 0}, xs[2] = {0, 0}, zs[2] = {0, 0};
  };
  std::vector<Col> col;
  mutable std::vector<Row> d, s;
  mutable bool rows_ok = false;
  uint64_t pend_d[2] = {0, 0}, pend_s[2] = {0, 0};  // sign XOR since the last event
  // X_q and Z_q as i^e d_beta s_gamma, kept through the Clifford gates: with the rows' signs
  // of the gates so far (all_d, all_s) a gate changes only its own qubits' images, to products
  // of them. A noise site takes its images from here; decomposing over the rows for each site
  // was most of the compile time, and
  // the rows' updates by gates most of the rest (soft_compile_circuit: w42 3.1 -> 1.0 ms,
  // w97 22.4 -> 3.1 ms; the same programs byte for byte).
  struct Image {
    uint64_t b[2] = {0, 0}, g[2] = {0, 0};
    uint32_t e = 0;
  };
  std::vector<Image> ix, iz;
  uint64_t all_d[2] = {0, 0}, all_s[2] = {0, 0};

  static Image times(const Image &p, const Image &q) {
    Image o;
    o.e = (p.e + q.e + 2u * (uint32_t)(pc(p.g[0] & q.b[0]) + pc(p.g[1] & q.b[1]))) & 3u;
    for (int w = 0; w < 2; ++w) {
      o.b[w] = p.b[w] ^ q.b[w];
      o.g[w] = p.g[w] ^ q.g[w];
    }
    return o;
  }
  uint32_t gate_signs(const Image &i) const {
    return (uint32_t)(pc(all_d[0] & i.b[0]) + pc(all_d[1] & i.b[1]) + pc(all_s[0] & i.g[0]) + pc(all_s[1] & i.g[1]));
  }
  void gate_images(int op, uint32_t a, uint32_t b, bool two) {
    const L2 *to = tabs().back[op];
    const Image xa = ix[a], za = iz[a], xb = two ? ix[b] : Image{}, zb = two ? iz[b] : Image{};
    auto image = [&](const L2 &l) {
      Image o;
      o.e = (uint32_t)l.e & 3u;
      if (l.x & 1u) o = times(o, xa);
      if (l.x & 2u) o = times(o, xb);
      if (l.z & 1u) o = times(o, za);
      if (l.z & 2u) o = times(o, zb);
      return o;
    };
    ix[a] = image(to[0]);
    iz[a] = image(to[1]);
    if (two) {
      ix[b] = image(to[2]);
      iz[b] = image(to[3]);
    }
  }
  // X_q (code 1), Y_q = i X_q Z_q (2) or Z_q (3) at zero signs
  void image(int code, uint32_t q, uint64_t beta[2], uint64_t gamma[2], uint32_t *e0) const {
    Image i = code == 3 ? iz[q] : ix[q];
    if (code == 2) {
      i = times(i, iz[q]);
      i.e += 1u;
    }
    for (int w = 0; w < 2; ++w) {
      beta[w] = i.b[w];
      gamma[w] = i.g[w];
    }
    *e0 = (i.e + 2u * gate_signs(i)) & 3u;
  }

  // any i^e X^x Z^z at zero signs
  void image(const Pz &p, uint64_t beta[2], uint64_t gamma[2], uint32_t *e0) const {
    Image o;
    for (uint32_t q = 0; q < n; ++q)
      if (bit(p.x, q)) o = times(o, ix[q]);
    for (uint32_t q = 0; q < n; ++q)
      if (bit(p.z, q)) o = times(o, iz[q]);
    for (int w = 0; w < 2; ++w) {
      beta[w] = o.b[w];
      gamma[w] = o.g[w];
    }
    *e0 = (o.e + (uint32_t)p.e + 2u * gate_signs(o)) & 3u;
  }

  void init(uint32_t nq) {
    n = nq;
    ix.assign(n, Image{});
    iz.assign(n, Image{});
    for (uint32_t q = 0; q < n; ++q) {
      flip(ix[q].b, q);
      flip(iz[q].g, q);
    }
    col.assign(n, Col{});
    for (uint32_t i = 0; i < n; ++i) {
      flip(col[i].xd, i);
      flip(col[i].zs, i);
    }
    rows_ok = false;
  }
  // one part of the rows (X or Z words of d or s) from the columns', or back
  template <typename Get, typename Set>
  static void transpose(uint32_t rows_in, uint32_t rows_out, Get get, Set set) {
    for (uint32_t ob = 0; ob < rows_out; ob += 64)
      for (uint32_t ib = 0; ib < rows_in; ib += 64) {
        uint64_t m[64];
        for (uint32_t k = 0; k < 64; ++k) m[k] = ib + k < rows_in ? get(ib + k, ob >> 6) : 0ull;
        transpose64(m);
        for (uint32_t k = 0; k < 64 && ob + k < rows_out; ++k) set(ob + k, ib >> 6, m[k]);
      }
  }
  void rows() const {
    if (rows_ok) return;
    d.assign(n, Row{});
    s.assign(n, Row{});
    transpose(n, n, [&](uint32_t q, uint32_t w) { return col[q].xd[w]; }, [&](uint32_t i, uint32_t w, uint64_t v) { d[i].x[w] = v; });
    transpose(n, n, [&](uint32_t q, uint32_t w) { return col[q].zd[w]; }, [&](uint32_t i, uint32_t w, uint64_t v) { d[i].z[w] = v; });
    transpose(n, n, [&](uint32_t q, uint32_t w) { return col[q].xs[w]; }, [&](uint32_t i, uint32_t w, uint64_t v) { s[i].x[w] = v; });
    transpose(n, n, [&](uint32_t q, uint32_t w) { return col[q].zs[w]; }, [&](uint32_t i, uint32_t w, uint64_t v) { s[i].z[w] = v; });
    rows_ok = true;
  }
  // the columns of changed rows
  void rows_changed() {
    transpose(n, n, [&](uint32_t i, uint32_t w) { return d[i].x[w]; }, [&](uint32_t q, uint32_t w, uint64_t v) { col[q].xd[w] = v; });
    transpose(n, n, [&](uint32_t i, uint32_t w) { return d[i].z[w]; }, [&](uint32_t q, uint32_t w, uint64_t v) { col[q].zd[w] = v; });
    transpose(n, n, [&](uint32_t i, uint32_t w) { return s[i].x[w]; }, [&](uint32_t q, uint32_t w, uint64_t v) { col[q].xs[w] = v; });
    transpose(n, n, [&](uint32_t i, uint32_t w) { return s[i].z[w]; }, [&](uint32_t q, uint32_t w, uint64_t v) { col[q].zs[w] = v; });
  }
  // The images after a case-B measurement of P. The row operations (s_j = +-s'_j s_p for j in J,
  // d_p = +-d'_p prod d_J) keep d's and s's apart; then s_p becomes d''_p, d'_j (j in G)
  // +-d''_j d''_p, and d'_p = i^-e0b P s_gamma2 with P = +-s''_p.
  void case_b_images(const CaseB &B) {
    const uint32_t p = B.p;
    auto without_p = [&](uint64_t v[2]) { v[p >> 6] &= ~(1ull << (p & 63)); };
    auto par = [](const uint64_t *a, const uint64_t *b) { return (uint32_t)(pc(a[0] & b[0]) + pc(a[1] & b[1])); };
    Image dp, sp;  // d'_p and s_p in the new rows
    flip(sp.b, p);
    for (int w = 0; w < 2; ++w) dp.g[w] = B.gamma2[w];
    without_p(dp.g);
    flip(dp.g, p);
    dp.e = (4u - (B.e0b & 3u) + 2u * B.rP) & 3u;
    if (bit(B.gamma2, p)) dp = times(dp, sp);
    for (uint32_t q = 0; q < 2 * n; ++q) {
      Image &im = q < n ? ix[q] : iz[q - n];
      uint32_t e = im.e + 2u * gate_signs(im);  // at zero signs
      uint64_t b[2] = {im.b[0], im.b[1]}, g[2] = {im.g[0], im.g[1]};
      const bool bp = bit(b, p) != 0;
      if (bp) {
        for (int w = 0; w < 2; ++w) b[w] ^= B.J[w];
        e += 2u * B.hdp;
      }
      e += 2u * par(g, B.Hs);
      if (par(g, B.J) & 1u) flip(g, p);
      const bool gp = bit(g, p) != 0;
      Image o, sg;
      for (int w = 0; w < 2; ++w) {
        o.b[w] = b[w];
        sg.g[w] = g[w];
      }
      without_p(o.b);
      without_p(sg.g);
      e += 2u * par(o.b, B.Hd);
      if (par(o.b, B.G) & 1u) flip(o.b, p);
      o.e = e & 3u;
      if (bp) o = times(o, dp);
      o = times(o, sg);
      if (gp) o = times(o, sp);
      o.e = (o.e + 2u * gate_signs(o)) & 3u;
      im = o;
    }
  }

  // Rows by rows of the table: which inputs flip the sign, and the (linear) outputs, as word
  // operations on the qubits' columns.
  void gate(int op, uint32_t a, uint32_t b) {
    const GateTab &t = tabs().g[op];
    const bool two = (op == SOFT_CX || op == SOFT_CZ);
    rows_ok = false;
    const uint32_t nw = (n + 63u) / 64u;
    auto part = [&](uint64_t *xa, uint64_t *za, uint64_t *xb, uint64_t *zb, uint64_t *pend, uint64_t *all) {
      for (uint32_t w = 0; w < nw; ++w) {
        const uint64_t v[4] = {xa[w], za[w], two ? xb[w] : 0ull, two ? zb[w] : 0ull};
        uint64_t f = 0;
        for (uint32_t in = 1; in < (two ? 16u : 4u); ++in)
          if (t.flipb[in] & 1u) {
            uint64_t m = ~0ull;
            for (uint32_t k = 0; k < (two ? 4u : 2u); ++k) m &= ((in >> k) & 1u) ? v[k] : ~v[k];
            f |= m;
          }
        uint64_t o[4] = {0, 0, 0, 0};
        for (uint32_t k = 0; k < (two ? 4u : 2u); ++k)
          for (uint32_t j = 0; j < 4; ++j)
            if ((t.out[1u << k] >> j) & 1u) o[j] ^= v[k];
        xa[w] = o[0];
        za[w] = o[1];
        if (two) {
          xb[w] = o[2];
          zb[w] = o[3];
        }
        pend[w] ^= f;
        all[w] ^= f;
      }
    };
    Col &ca = col[a], &cb = col[two ? b : a];
    part(ca.xd, ca.zd, cb.xd, cb.zd, pend_d, all_d);
    part(ca.xs, ca.zs, cb.xs, cb.zs, pend_s, all_s);
    gate_images(op, a, b, two);
  }

  // Q = i^e0 d_beta s_gamma at zero signs. NW: the 64-bit words in use. Bits are set
  // without branches and the product runs over the set bits in increasing order,
  // accumulating X, Z and the phase in place (the data-dependent branches and the
  // second word were most of the compile time).
  template <int NW>
  bool decompose_w(const Pz &q, uint64_t beta[2], uint64_t gamma[2], uint32_t *e0) const {
    beta[0] = beta[1] = gamma[0] = gamma[1] = 0;
    for (uint32_t i = 0; i < n; ++i) {
      int ts = 0, td = 0;
      for (int w = 0; w < NW; ++w) {
        ts += pc((q.x[w] & s[i].z[w]) ^ (q.z[w] & s[i].x[w]));
        td += pc((q.x[w] & d[i].z[w]) ^ (q.z[w] & d[i].x[w]));
      }
      beta[i >> 6] |= (uint64_t)(ts & 1) << (i & 63);
      gamma[i >> 6] |= (uint64_t)(td & 1) << (i & 63);
    }
    // acc <- acc * herm(r): phase + herm's own (popc(x & z)) + 2 popc(acc.z & r.x)
    uint64_t ax[2] = {0, 0}, az[2] = {0, 0};
    int ae = 0;
    auto mul = [&](const Row &r) {
      for (int w = 0; w < NW; ++w) {
        ae += pc(r.x[w] & r.z[w]) + 2 * pc(az[w] & r.x[w]);
        ax[w] ^= r.x[w];
        az[w] ^= r.z[w];
      }
    };
    for (int w = 0; w < NW; ++w)
      for (uint64_t m = beta[w]; m; m &= m - 1) mul(d[64 * w + __builtin_ctzll(m)]);
    for (int w = 0; w < NW; ++w)
      for (uint64_t m = gamma[w]; m; m &= m - 1) mul(s[64 * w + __builtin_ctzll(m)]);
    for (int w = 0; w < 2; ++w)
      if (ax[w] != q.x[w] || az[w] != q.z[w]) return false;
    *e0 = (uint32_t)((q.e - ae) & 3);
    return true;
  }
  bool decompose(const Pz &q, uint64_t beta[2], uint64_t gamma[2], uint32_t *e0) const {
    rows();
    return n <= 64 ? decompose_w<1>(q, beta, gamma, e0) : decompose_w<2>(q, beta, gamma, e0);
  }
};

Pz single(int code, uint32_t q) {
  Pz p;
  if (code == 1 || code == 2) flip(p.x, q);
  if (code == 3 || code == 2) flip(p.z, q);
  p.e = (code == 2) ? 1 : 0;
  return p;
}

bool is1q(int op) {
  return op == SOFT_H || op == SOFT_S || op == SOFT_S_DAG || op == SOFT_X || op == SOFT_Y || op == SOFT_Z ||
         op == SOFT_T || op == SOFT_T_DAG || op == SOFT_RZ;
}
bool is2q(int op) { return op == SOFT_CX || op == SOFT_CZ; }
bool isclifford(int op) { return op <= SOFT_CZ; }

// log_q: log1p(-p)
uint64_t gap_thr(double log_q, uint64_t g) {
  double q = -std::expm1((double)(g + 1) * log_q);
  if (!(q > 0.0)) return 0;
  if (q >= 1.0) return UINT64_MAX;
  double t = std::ldexp(q, 64);
  if (t >= 18446744073709551615.0) return UINT64_MAX;
  return (uint64_t)t;
}

// Peephole pass: fold a reset's conditional X and a single-record detector
// into the measurement event right before them. Folding is exact when the
// folded event adds no noise sites and no Clifford sign masks in between and
// no parity chain is pending.
void fuse_events(std::vector<Ev<2>> &ev) {
  std::vector<Ev<2>> out;
  out.reserve(ev.size());
  bool chain_pending = false;
  auto quiet = [](const Ev<2> &e, const Ev<2> &prev) {
    return e.site_begin == prev.site_begin && !(e.dsd[0] | e.dsd[1] | e.dss[0] | e.dss[1]);
  };
  for (const Ev<2> &e : ev) {
    const uint32_t type = ev_type(e.w0), fl = ev_flags(e.w0);
    if (!out.empty()) {
      Ev<2> &m = out.back();
      const uint32_t mt = ev_type(m.w0), mf = ev_flags(m.w0);
      const bool is_meas = (mt == EV_MEAS_A || mt == EV_MEAS_B);
      if (is_meas && type == EV_PAULI && (fl & F_COND_LAST) && !(mf & (F_COND_LAST | F_DETECTOR)) && quiet(e, m)) {
        m.w0 |= (F_COND_LAST << 4) | (ev_e0(e.w0) << 24);
        m.xbeta[0] = e.beta[0];
        m.xbeta[1] = e.beta[1];
        m.xgamma[0] = e.gamma[0];
        m.xgamma[1] = e.gamma[1];
        continue;
      }
      if (is_meas && type == EV_PARITY && (fl & F_DETECTOR) && !(fl & F_CHAIN) && !chain_pending &&
          (mf & F_RECORD) && !(mf & F_DETECTOR) && e.a == m.b && e.b == kNoRec && quiet(e, m)) {
        m.w0 |= (F_DETECTOR << 4) | ((fl & F_INVERT) ? (F_INVERT << 4) : 0u);
        continue;
      }
    }
    if (type == EV_PARITY) chain_pending = (fl & F_CHAIN) != 0;
    out.push_back(e);
  }
  ev.swap(out);
}

}  // namespace

int compile_program(const soft_op *ops, size_t n_ops, uint32_t n, const soft_noise *noise, uint32_t cap,
                    HostProgram &P, std::string &err) {
  if (!noise || (!ops && n_ops)) {
    err = "null argument";
    return SOFT_E_ARG;
  }
  if (n == 0 || n > 128) {
    err = "n_qubits must be in 1..128";
    return SOFT_E_QUBIT_RANGE;
  }
  if (cap == 0 || cap > 65536) {
    err = "coeff_cap must be in 1..65536";
    return SOFT_E_ARG;
  }
  const double ps[4] = {noise->p1, noise->p2, noise->p_meas, noise->p_reset};
  for (double p : ps)
    if (!(p >= 0.0 && p < 1.0)) {
      err = "noise probabilities must be in [0, 1)";
      return SOFT_E_ARG;
    }
  if (noise->p_idle != 0.0) {
    err = "idle noise is not supported (p_idle must be 0)";
    return SOFT_E_UNSUPPORTED_OP;
  }
  P = HostProgram{};
  P.n = n;
  P.W = n <= 64 ? 1 : 2;
  P.cap = cap;
  P.pmax = std::fmax(std::fmax(noise->p1, noise->p2), std::fmax(noise->p_meas, noise->p_reset));
  Tableau tb;
  tb.init(n);
  bool noiseless = false;
  uint32_t nrec = 0, ord = 0;

  // kind: SITE_DEPOL1, SITE_DEPOL2, or SITE_FLIP | code << 2
  auto add_site = [&](uint32_t q0, uint32_t q1, uint32_t kind, double p) -> bool {
    const bool two = (kind & 3u) == SITE_DEPOL2;
    Site s{};
    s.dsd[0] = tb.pend_d[0];
    s.dsd[1] = tb.pend_d[1];
    s.dss[0] = tb.pend_s[0];
    s.dss[1] = tb.pend_s[1];
    s.kind = kind;
    // X_q and Z_q of each site qubit: Q = i^e d_beta s_gamma at zero signs
    uint32_t ex[2] = {0, 0}, ez[2] = {0, 0};
    for (int k = 0; k < (two ? 2 : 1); ++k) {
      uint32_t q = k == 0 ? q0 : q1;
      tb.image(1, q, s.bx[k], s.gx[k], &ex[k]);
      tb.image(3, q, s.bz[k], s.gz[k], &ez[k]);
    }
    // Phases of the other Paulis by composition. With P = i^a d_b s_c and
    // Q = i^a' d_b' s_c', PQ = i^(a + a' + 2 |c & b'|) d_(b^b') s_(c^c'): s_j
    // anticommutes with d_j only, and the d's (and the s's) commute and square to I.
    // |c & b'| counts modulo 2 and is linear in either operand, so four parities per pair of
    // qubits give all 15 codes.
    auto dot = [&](const uint64_t *c, const uint64_t *b2) { return (uint32_t)(pc(c[0] & b2[0]) + pc(c[1] & b2[1])); };
    uint32_t e1[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};  // phases of 1 X, 2 Y = i X Z, 3 Z per qubit
    for (int k = 0; k < (two ? 2 : 1); ++k) {
      e1[k][1] = ex[k];
      e1[k][2] = 1u + ex[k] + ez[k] + 2u * dot(s.gx[k], s.bz[k]);
      e1[k][3] = ez[k];
    }
    uint32_t c0 = 0;
    if (!two) {
      for (int code = 1; code <= 3; ++code) {
        c0 |= (e1[0][code] & 3u) << (2 * code);
        c0 |= (e1[0][code] & 3u) << (8 * code);  // also at code << 2, the site's Pauli pair (see Site)
      }
    } else {
      const uint32_t cr[2][2] = {{dot(s.gx[0], s.bx[1]), dot(s.gx[0], s.bz[1])}, {dot(s.gz[0], s.bx[1]), dot(s.gz[0], s.bz[1])}};
      for (int code = 1; code <= 15; ++code) {
        const int pa = code >> 2, pb = code & 3;
        const int ax = pa == 1 || pa == 2, az = pa >= 2, bx = pb == 1 || pb == 2, bz = pb >= 2;
        const uint32_t x = (ax && bx ? cr[0][0] : 0u) + (ax && bz ? cr[0][1] : 0u) + (az && bx ? cr[1][0] : 0u) +
                           (az && bz ? cr[1][1] : 0u);
        c0 |= ((e1[0][pa] + e1[1][pb] + 2u * x) & 3u) << (2 * code);
      }
    }
    s.c0 = c0;
    if (p >= P.pmax) {
      s.always = 1;
      s.thin = 0xFFFFFFFFu;
    } else {
      s.always = 0;
      s.thin = (uint32_t)std::floor(std::ldexp(p / P.pmax, 32));
    }
    P.sites.push_back(s);
    P.site_kind.push_back((uint8_t)(kind | (s.always ? 0u : kSiteThinned)));
    return true;
  };

  auto new_event = [&](uint32_t type, uint32_t flags, uint32_t e0, uint32_t lowbit) -> Ev<2> & {
    Ev<2> e{};
    e.w0 = ev_pack(type, flags, e0, lowbit);
    e.site_begin = (uint32_t)P.sites.size();
    e.dsd[0] = tb.pend_d[0];
    e.dsd[1] = tb.pend_d[1];
    e.dss[0] = tb.pend_s[0];
    e.dss[1] = tb.pend_s[1];
    tb.pend_d[0] = tb.pend_d[1] = tb.pend_s[0] = tb.pend_s[1] = 0;
    e.a = e.b = kNoRec;
    P.ev.push_back(e);
    return P.ev.back();
  };

  auto pauli_event = [&](int code, uint32_t q, uint32_t flags, int32_t r0, int32_t r1) -> bool {
    uint64_t beta[2], gamma[2];
    uint32_t e0;
    tb.image(code, q, beta, gamma, &e0);
    Ev<2> &e = new_event(EV_PAULI, flags, e0, 0);
    e.a = (uint32_t)r0;
    e.b = (uint32_t)r1;
    std::memcpy(e.beta, beta, sizeof beta);
    std::memcpy(e.gamma, gamma, sizeof gamma);
    return true;
  };

  std::vector<int32_t> coef_phase;  // per coefficient: its global phase in units of pi/8
  // fixed angles share entries by value; a parameterised angle gets one entry per (parameter, sign)
  auto coef_index = [&](double ar, double ai, double br, double bi, double co, double si, int32_t phase,
                        int32_t param) -> uint32_t {
    for (size_t k = 0; k < P.coefs.size(); ++k) {
      const Coef &c = P.coefs[k];
      if (param >= 0 ? P.coef_param[k] == param
                     : (P.coef_param[k] < 0 && c.a_re == ar && c.a_im == ai && c.b_re == br && c.b_im == bi))
        return (uint32_t)k;
    }
    const bool scaled = std::fabs(si) <= std::sqrt(3.0) * std::fabs(co);
    Coef c{ar, ai, br, bi, (float)ar, (float)ai, (float)br, (float)bi, scaled ? si / co : si, scaled ? 1.0 : co,
           scaled ? 1.0 / (co * co) : 1.0, 0.0};
    P.coefs.push_back(c);
    P.coef_param.push_back(param);
    coef_phase.push_back(phase);
    return (uint32_t)(P.coefs.size() - 1);
  };
  // records read by OBSERVABLE ops (fidelity measurements of gradient runs)
  std::vector<uint8_t> observed;
  {
    uint32_t nr = 0;
    for (size_t i = 0; i < n_ops; ++i) {
      int op = ops[i].op;
      if (op == SOFT_M || op == SOFT_MR || (op == SOFT_MPP && !(ops[i].flags & SOFT_MPP_MORE))) nr++;
      if (op == SOFT_OBSERVABLE)
        for (int k = 0; k < 2; ++k)
          if (ops[i].rec[k] >= 0 && (uint32_t)ops[i].rec[k] < nr) {
            if (observed.size() <= (size_t)ops[i].rec[k]) observed.resize(ops[i].rec[k] + 1, 0);
            observed[ops[i].rec[k]] = 1;
          }
    }
  }

  // One Pauli measurement of P (Theorem 1 (2)): case A when P commutes with
  // every stabilizer row, else case B with its row operations and
  // replacement constants. Returns false on an internal inconsistency.
  auto meas_event = [&](const Pz &Pm, int zq, bool recd) -> bool {  // zq: P is Z on this qubit (-1: not)
    uint64_t beta[2], gamma[2];
    uint32_t e0;
    if (zq >= 0) tb.image(3, (uint32_t)zq, beta, gamma, &e0);
    else tb.image(Pm, beta, gamma, &e0);
    const uint32_t fidf = (recd && nrec < observed.size() && observed[nrec]) ? F_FIDELITY : 0u;
    if ((beta[0] | beta[1]) == 0) {
      Ev<2> &e = new_event(EV_MEAS_A, (recd ? F_RECORD : 0) | fidf, e0, 0);
      std::memcpy(e.gamma, gamma, sizeof gamma);
      e.a = ord;
      e.b = recd ? nrec : 0;
      return true;
    }
    CaseB cb{};
    tb.rows();
    uint32_t p = beta[0] ? (uint32_t)__builtin_ctzll(beta[0]) : 64u + (uint32_t)__builtin_ctzll(beta[1]);
    cb.p = p;
    cb.J[0] = beta[0];
    cb.J[1] = beta[1];
    flip(cb.J, p);
    // s_j <- s_j s_p
    for (uint32_t j = 0; j < n; ++j)
      if (bit(cb.J, j)) {
        Pz prod = pmul(herm(tb.s[j]), herm(tb.s[p]));
        int sb = sign_bit(prod);
        if (sb < 0) return false;
        if (sb) flip(cb.Hs, j);
        tb.s[j] = row_of(prod);
      }
    // d_p <- d_p prod_{j in J} d_j
    {
      Pz acc = herm(tb.d[p]);
      for (uint32_t j = 0; j < n; ++j)
        if (bit(cb.J, j)) acc = pmul(acc, herm(tb.d[j]));
      int sb = sign_bit(acc);
      if (sb < 0) return false;
      cb.hdp = (uint32_t)sb;
      tb.d[p] = row_of(acc);
    }
    uint64_t b2[2];
    if (!tb.decompose(Pm, b2, cb.gamma2, &cb.e0b)) return false;
    if (b2[0] != (p < 64 ? (1ull << p) : 0) || b2[1] != (p >= 64 ? (1ull << (p - 64)) : 0)) return false;
    Row old_sp = tb.s[p];
    for (uint32_t j = 0; j < n; ++j)
      if (j != p && bit(cb.gamma2, j)) {
        flip(cb.G, j);
        Pz prod = pmul(herm(tb.d[j]), herm(old_sp));
        int sb = sign_bit(prod);
        if (sb < 0) return false;
        if (sb) flip(cb.Hd, j);
        tb.d[j] = row_of(prod);
      }
    tb.d[p] = old_sp;
    // s_p <- m P: the row of P with P's own sign bit, flipped on the device when m = -1
    const int rp = sign_bit(Pm);
    if (rp < 0) return false;
    tb.s[p] = row_of(Pm);
    cb.rP = (uint32_t)rp;
    Ev<2> &e = new_event(EV_MEAS_B, (recd ? F_RECORD : 0) | fidf, 0, 0);
    e.a = ord;
    e.b = recd ? nrec : 0;
    e.beta[0] = P.cb.size();
    P.cb.push_back(cb);
    tb.rows_changed();
    tb.case_b_images(cb);
    return true;
  };

  Pz mpp_acc;                     // product of the open MPP chain's factors
  uint64_t mpp_q[2] = {0, 0};     // its qubits
  bool mpp_open = false, seen_observed = false;
  for (size_t i = 0; i < n_ops; ++i) {
    const soft_op &o = ops[i];
    int op = o.op;
    if (op > SOFT_MPP) {
      err = "unknown op code at op " + std::to_string(i);
      return SOFT_E_UNSUPPORTED_OP;
    }
    if (mpp_open && op != SOFT_MPP) {
      err = "an MPP chain is continued by a non-MPP op at op " + std::to_string(i);
      return SOFT_E_ARG;
    }
    bool needs_q = is1q(op) || is2q(op) || op == SOFT_M || op == SOFT_R || op == SOFT_MR || op == SOFT_CPAULI ||
                   op == SOFT_MPP;
    if (needs_q && o.q0 >= n) {
      err = "qubit out of range at op " + std::to_string(i);
      return SOFT_E_QUBIT_RANGE;
    }
    if (is2q(op) && (o.q1 >= n || o.q1 == o.q0)) {
      err = "bad second qubit at op " + std::to_string(i);
      return SOFT_E_QUBIT_RANGE;
    }
    const bool mpp_first = op == SOFT_MPP && !mpp_open;
    if (op == SOFT_MPP) {
      const int pa = o.flags & 3, pb = (o.flags >> 2) & 3;
      if (pa == 0 || (o.flags & ~(uint32_t)(15 | SOFT_MPP_MORE))) {
        err = "bad MPP flags at op " + std::to_string(i);
        return SOFT_E_ARG;
      }
      if (pb && (o.q1 >= n || o.q1 == o.q0)) {
        err = "bad second MPP qubit at op " + std::to_string(i);
        return SOFT_E_QUBIT_RANGE;
      }
      if (bit(mpp_q, o.q0) || (pb && bit(mpp_q, o.q1))) {
        err = "MPP chain repeats a qubit at op " + std::to_string(i);
        return SOFT_E_ARG;
      }
      if ((o.flags & SOFT_MPP_MORE) && i + 1 == n_ops) {
        err = "MPP chain left open at the end of the circuit";
        return SOFT_E_ARG;
      }
    }
    if (op == SOFT_DETECTOR && seen_observed) P.fid_ok = false;
    if (op == SOFT_DETECTOR || op == SOFT_OBSERVABLE || op == SOFT_CPAULI) {
      for (int k = 0; k < 2; ++k)
        if (o.rec[k] >= 0 && (uint32_t)o.rec[k] >= nrec) {
          err = "record reference to a future measurement at op " + std::to_string(i);
          return SOFT_E_RECORD_REF;
        }
    }
    if (op == SOFT_NOISELESS_BEGIN) noiseless = true;
    if (op == SOFT_NOISELESS_END) noiseless = false;

    if (!noiseless && noise->p_meas > 0) {
      if (op == SOFT_M || op == SOFT_MR) {
        if (!add_site(o.q0, 0, SITE_FLIP | (1u << 2), noise->p_meas)) goto internal;
      } else if (mpp_first) {
        const uint32_t fc = (o.flags & 3) == 1 ? 3u : 1u;  // anticommutes with the first factor
        if (!add_site(o.q0, 0, SITE_FLIP | (fc << 2), noise->p_meas)) goto internal;
      }
    }

    if (isclifford(op)) {
      tb.gate(op, o.q0, o.q1);
    } else if (op == SOFT_T || op == SOFT_T_DAG || op == SOFT_RZ) {
      uint64_t beta[2], gamma[2];
      uint32_t e0;
      tb.image(3, o.q0, beta, gamma, &e0);
      bool diag = (beta[0] | beta[1]) == 0;
      double ar, ai, br, bi, co, si;  // a phase times co I - i si Z
      int32_t phase = 0;
      if (op == SOFT_RZ) {
        co = std::cos(0.5 * o.angle);
        si = std::sin(0.5 * o.angle);
        ar = co;
        ai = 0.0;
        br = 0.0;
        bi = -si;
        if (co < 0.0) {  // c I - i s Z = e^{i pi} (-c I + i s Z)
          co = -co;
          si = -si;
          phase = 8;
        }
      } else {
        // diag(1, e^{+-i pi/4}) = (1 + w)/2 I + (1 - w)/2 Z with w = e^{+-i pi/4}
        double c = std::cos(0.25 * M_PI), sn = (op == SOFT_T ? 1.0 : -1.0) * std::sin(0.25 * M_PI);
        ar = 0.5 * (1.0 + c);
        ai = 0.5 * sn;
        br = 0.5 * (1.0 - c);
        bi = -0.5 * sn;
        phase = op == SOFT_T ? 1 : -1;
        co = std::cos(0.125 * M_PI);
        si = phase * std::sin(0.125 * M_PI);
      }
      uint32_t lowbit = 0;
      if (!diag) lowbit = beta[0] ? (uint32_t)__builtin_ctzll(beta[0]) : 64u + (uint32_t)__builtin_ctzll(beta[1]);
      int32_t param = -1;
      if (op == SOFT_RZ && o.pad > 0) {
        param = (int32_t)(((o.pad - 1) << 1) | (o.flags & 1));
        P.n_params = std::max<uint32_t>(P.n_params, o.pad);
      }
      uint32_t ci = coef_index(ar, ai, br, bi, co, si, phase, param);
      Ev<2> &e = new_event(diag ? EV_ROT_DIAG : EV_ROT, 0, e0, lowbit);
      e.a = ci;
      e.b = param >= 0 ? (uint32_t)param : kNoRec;
      P.n_rot++;
      std::memcpy(e.beta, beta, sizeof beta);
      std::memcpy(e.gamma, gamma, sizeof gamma);
    } else if (op == SOFT_M || op == SOFT_R || op == SOFT_MR) {
      bool recd = (op != SOFT_R);
      if (recd && nrec < observed.size() && observed[nrec]) seen_observed = true;
      if (!meas_event(single(3, o.q0), (int)o.q0, recd)) goto internal;
      ord++;
      if (recd) nrec++;
      if (op == SOFT_R || op == SOFT_MR)
        if (!pauli_event(1, o.q0, F_COND_LAST, -1, -1)) goto internal;
    } else if (op == SOFT_MPP) {
      if (!mpp_open) mpp_acc = Pz{};
      mpp_acc = pmul(mpp_acc, single(o.flags & 3, o.q0));
      flip(mpp_q, o.q0);
      if ((o.flags >> 2) & 3) {
        mpp_acc = pmul(mpp_acc, single((o.flags >> 2) & 3, o.q1));
        flip(mpp_q, o.q1);
      }
      mpp_open = (o.flags & SOFT_MPP_MORE) != 0;
      if (!mpp_open) {
        mpp_q[0] = mpp_q[1] = 0;
        if (nrec < observed.size() && observed[nrec]) seen_observed = true;
        if (!meas_event(mpp_acc, -1, true)) goto internal;
        ord++;
        nrec++;
      }
    } else if (op == SOFT_CPAULI) {
      int code = o.flags & 3;
      if (code) {
        if (!pauli_event(code, o.q0, F_COND_REC, o.rec[0], o.rec[1])) goto internal;
      }
    } else if (op == SOFT_DETECTOR || op == SOFT_OBSERVABLE) {
      uint32_t fl = (op == SOFT_DETECTOR ? F_DETECTOR : F_OBSERVABLE) | ((o.flags & SOFT_FLAG_CHAIN) ? F_CHAIN : 0) |
                    ((o.flags & SOFT_FLAG_INVERT) ? F_INVERT : 0);
      Ev<2> &e = new_event(EV_PARITY, fl, 0, 0);
      e.a = (uint32_t)o.rec[0];
      e.b = (uint32_t)o.rec[1];
    }

    if (!noiseless) {
      if (is1q(op) && noise->p1 > 0) {
        if (!add_site(o.q0, 0, SITE_DEPOL1, noise->p1)) goto internal;
      } else if (is2q(op) && noise->p2 > 0) {
        if (!add_site(o.q0, o.q1, SITE_DEPOL2, noise->p2)) goto internal;
      } else if ((op == SOFT_R || op == SOFT_MR) && noise->p_reset > 0) {
        if (!add_site(o.q0, 0, SITE_FLIP | (1u << 2), noise->p_reset)) goto internal;
      }
    }
  }
  new_event(EV_END, 0, 0, 0);
  fuse_events(P.ev);
  {
    uint32_t ph = 0;  // (units of pi/8, modulo 16)
    for (auto &e : P.ev) {
      if (ev_type(e.w0) == EV_ROT || ev_type(e.w0) == EV_ROT_DIAG) ph += (uint32_t)coef_phase[e.a];
      e.w0 |= (ph & 15u) << 26;
    }
  }
  P.n_records = nrec;
  P.rw = nrec ? (nrec + 63) / 64 : 1;
  if (P.rw > 16) {
    err = "at most 1024 recorded measurements are supported";
    return SOFT_E_ARG;
  }
  P.n_sites = (uint32_t)P.sites.size();
  P.thr.resize(P.n_sites ? P.n_sites : 1);
  {
    const double log_q = std::log1p(-P.pmax);
    for (uint32_t g = 0; g < P.n_sites; ++g) P.thr[g] = gap_thr(log_q, g);
  }
  // thr increases with g, so the first g with U < thr[g] for every U of a bucket of the top
  // bits lies between the bucket's entry and the next one's
  P.thr_tab.assign((1u << kThrTabBits) + 1u, P.n_sites);
  for (uint32_t b = 0, at = 0; b < (1u << kThrTabBits); ++b) {
    const uint64_t U = (uint64_t)b << (64 - kThrTabBits);
    while (at < P.n_sites && P.thr[at] <= U) ++at;  // (both increase)
    P.thr_tab[b] = at;
  }
  P.site_ev.assign(P.thr.size(), (uint32_t)P.ev.size());
  {
    uint32_t e = 0;
    for (uint32_t s = 0; s < P.n_sites; ++s) {
      while (e < P.ev.size() && P.ev[e].site_begin <= s) ++e;
      P.site_ev[s] = e;
    }
  }
  tb.rows();
  P.fin_x.assign(4 * (size_t)n, 0);
  P.fin_z.assign(4 * (size_t)n, 0);
  for (uint32_t i = 0; i < n; ++i)
    for (int w = 0; w < 2; ++w) {
      P.fin_x[2 * i + w] = tb.d[i].x[w];
      P.fin_z[2 * i + w] = tb.d[i].z[w];
      P.fin_x[2 * (n + i) + w] = tb.s[i].x[w];
      P.fin_z[2 * (n + i) + w] = tb.s[i].z[w];
    }
  return SOFT_OK;
internal:
  err = "internal tableau inconsistency";
  return SOFT_E_ARG;
}

}  // namespace soft
