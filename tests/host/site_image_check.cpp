// Host check of the compiled sites' Pauli images: at every site X and Z of a
// qubit anticommute, and those of different qubits commute (Clifford gates and
// the frame changes of measurements keep the symplectic product).
// Usage: site_image_check <ops file> <n_qubits> <p> ; prints "ok <sites>" or the first failure.
#include <cstdio>
#include <cstdlib>
#include <fstream>
#include <iterator>
#include <string>
#include <vector>

#include "../../paper_2512_23037_gb300/csrc/compile.h"

// the symplectic product of (b1, g1) and (b2, g2)
static int product(const uint64_t *b1, const uint64_t *g1, const uint64_t *b2, const uint64_t *g2) {
  int s = 0;
  for (int w = 0; w < 2; ++w) s ^= __builtin_parityll(b1[w] & g2[w]) ^ __builtin_parityll(g1[w] & b2[w]);
  return s;
}

int main(int argc, char **argv) {
  if (argc < 4) return 2;
  std::ifstream f(argv[1], std::ios::binary);
  std::vector<char> buf((std::istreambuf_iterator<char>(f)), std::istreambuf_iterator<char>());
  const double p = std::atof(argv[3]);
  const soft_noise nz{p, p, p, p, 0.0};
  soft::HostProgram hp;
  std::string err;
  if (soft::compile_program(reinterpret_cast<const soft_op *>(buf.data()), buf.size() / sizeof(soft_op),
                            (uint32_t)std::atoi(argv[2]), &nz, 256, hp, err) != 0) {
    std::printf("compile failed: %s\n", err.c_str());
    return 1;
  }
  size_t k = 0;
  for (const soft::Site &s : hp.sites) {
    const int two = (s.kind & 3u) == soft::SITE_DEPOL2 ? 2 : 1;
    for (int q = 0; q < two; ++q)
      if (product(s.bx[q], s.gx[q], s.bz[q], s.gz[q]) != 1) {
        std::printf("site %zu: X and Z of its qubit %d commute\n", k, q);
        return 1;
      }
    if (two == 2 && (product(s.bx[0], s.gx[0], s.bx[1], s.gx[1]) || product(s.bx[0], s.gx[0], s.bz[1], s.gz[1]) ||
                     product(s.bz[0], s.gz[0], s.bx[1], s.gx[1]) || product(s.bz[0], s.gz[0], s.bz[1], s.gz[1]))) {
      std::printf("site %zu: Paulis of its two qubits anticommute\n", k);
      return 1;
    }
    ++k;
  }
  std::printf("ok %zu\n", k);
  return 0;
}
