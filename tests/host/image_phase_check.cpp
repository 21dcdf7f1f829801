// Host check of the Pauli images that the compiler keeps per qubit: at every noise site and
// rotation, against the decomposition of the Pauli over the tableau's rows (words and phase),
// the phases of a site's 15 pairs against those of the products.
// The rows follow the gates by their columns and a case-B measurement by its constants.
// Usage: image_phase_check <ops file> <n_qubits> <p>; prints "ok <sites> <rotations> <case B>".
#include <cstdio>
#include <cstdlib>
#include <fstream>
#include <iterator>

#include "../../paper_2512_23037_gb300/csrc/compile.cpp"

using namespace soft;

static Tableau tb;
static size_t n_site = 0, n_rot = 0, n_cb = 0;

static void stop(const char *what, size_t i) {
  std::printf("%s %zu differs\n", what, i);
  std::exit(1);
}
static bool same(const uint64_t *a, const uint64_t *b) { return a[0] == b[0] && a[1] == b[1]; }

static void site(const HostProgram &hp, uint32_t q0, uint32_t q1, bool two) {
  if (n_site >= hp.sites.size()) stop("site count", n_site);
  const Site &s = hp.sites[n_site];
  uint64_t b[2], g[2];
  uint32_t e;
  for (int k = 0; k < (two ? 2 : 1); ++k) {
    const uint32_t q = k ? q1 : q0;
    if (!tb.decompose(single(1, q), b, g, &e) || !same(b, s.bx[k]) || !same(g, s.gx[k])) stop("X image of site", n_site);
    if (!tb.decompose(single(3, q), b, g, &e) || !same(b, s.bz[k]) || !same(g, s.gz[k])) stop("Z image of site", n_site);
  }
  for (int pp = 1; pp < 16; ++pp) {
    const int pa = pp >> 2, pb = pp & 3;
    if (!two && pb) continue;
    Pz p{};
    if (pa) p = pmul(p, single(pa, q0));
    if (pb) p = pmul(p, single(pb, q1));
    if (!tb.decompose(p, b, g, &e) || ((s.c0 >> (2 * pp)) & 3u) != e) stop("phase at site", n_site);
  }
  ++n_site;
}

// the rows' words after a case-B measurement of P
static void measure(const HostProgram &hp, const Pz &P) {
  uint64_t b[2], g[2];
  uint32_t e;
  if (!tb.decompose(P, b, g, &e)) stop("measured Pauli", n_cb);
  if (!(b[0] | b[1])) return;
  if (n_cb >= hp.cb.size()) stop("case-B count", n_cb);
  const CaseB &B = hp.cb[n_cb++];
  const uint32_t p = B.p;
  auto add = [](Row &r, const Row &o) {
    for (int w = 0; w < 2; ++w) {
      r.x[w] ^= o.x[w];
      r.z[w] ^= o.z[w];
    }
  };
  for (uint32_t j = 0; j < tb.n; ++j)
    if (bit(B.J, j)) {
      add(tb.s[j], tb.s[p]);
      add(tb.d[p], tb.d[j]);
    }
  for (uint32_t j = 0; j < tb.n; ++j)
    if (bit(B.G, j)) add(tb.d[j], tb.s[p]);
  tb.d[p] = tb.s[p];
  tb.s[p] = row_of(P);
  tb.rows_changed();
}

int main(int argc, char **argv) {
  if (argc < 4) return 2;
  std::ifstream f(argv[1], std::ios::binary);
  std::vector<char> buf((std::istreambuf_iterator<char>(f)), std::istreambuf_iterator<char>());
  const soft_op *ops = reinterpret_cast<const soft_op *>(buf.data());
  const size_t n_ops = buf.size() / sizeof(soft_op);
  const double p = std::atof(argv[3]);
  const soft_noise nz{p, p, p, p, 0.0};
  HostProgram hp;
  std::string err;
  if (compile_program(ops, n_ops, (uint32_t)std::atoi(argv[2]), &nz, 256, hp, err) != 0) {
    std::printf("compile failed: %s\n", err.c_str());
    return 1;
  }
  tb.init((uint32_t)std::atoi(argv[2]));
  size_t ev = 0;
  bool quiet = false, open = false;
  Pz product;
  for (size_t i = 0; i < n_ops; ++i) {
    const soft_op &o = ops[i];
    const int op = o.op;
    if (op == SOFT_NOISELESS_BEGIN || op == SOFT_NOISELESS_END) quiet = op == SOFT_NOISELESS_BEGIN;
    if (!quiet && (op == SOFT_M || op == SOFT_MR || (op == SOFT_MPP && !open))) site(hp, o.q0, 0, false);
    if (isclifford(op)) {
      tb.gate(op, o.q0, o.q1);
    } else if (op == SOFT_T || op == SOFT_T_DAG || op == SOFT_RZ) {
      while (ev < hp.ev.size() && ev_type(hp.ev[ev].w0) != EV_ROT && ev_type(hp.ev[ev].w0) != EV_ROT_DIAG) ++ev;
      uint64_t b[2], g[2];
      uint32_t e;
      if (ev == hp.ev.size() || !tb.decompose(single(3, o.q0), b, g, &e) || !same(b, hp.ev[ev].beta) ||
          !same(g, hp.ev[ev].gamma) || ev_e0(hp.ev[ev].w0) != e)
        stop("rotation", n_rot);
      ++ev;
      ++n_rot;
    } else if (op == SOFT_M || op == SOFT_R || op == SOFT_MR) {
      measure(hp, single(3, o.q0));
    } else if (op == SOFT_MPP) {
      if (!open) product = Pz{};
      product = pmul(product, single(o.flags & 3, o.q0));
      if ((o.flags >> 2) & 3) product = pmul(product, single((o.flags >> 2) & 3, o.q1));
      open = (o.flags & SOFT_MPP_MORE) != 0;
      if (!open) measure(hp, product);
    }
    if (!quiet && is1q(op)) site(hp, o.q0, 0, false);
    if (!quiet && is2q(op)) site(hp, o.q0, o.q1, true);
    if (!quiet && (op == SOFT_R || op == SOFT_MR)) site(hp, o.q0, 0, false);
  }
  if (n_site != hp.sites.size() || n_cb != hp.cb.size()) stop("count", n_site);
  std::printf("ok %zu %zu %zu\n", n_site, n_rot, n_cb);
  return 0;
}
