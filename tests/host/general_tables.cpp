// Host check of the interface stencil tables of general meshes (csrc/mesh.cpp,
// build_general_if_tables): every row against the sub-stencils of the node's
// copies, summed node by node through the node keys' order.  No CUDA call.
//
// usage: general_tables nv nt R dir kind [faulty id...]
// dir holds verts.bin (nv x 3 doubles) and tets.bin (nt x 4 int32).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include <vector>

#include "../../paper_1506_06185_gb300/csrc/hhg_internal.h"

using namespace hhg;

template <class T>
static std::vector<T> readv(const std::string& fn, size_t n) {
  std::vector<T> v(n);
  FILE* f = fopen(fn.c_str(), "rb");
  if (!f || fread(v.data(), sizeof(T), n, f) != n) exit(2);
  fclose(f);
  return v;
}
#define CHECK(c)                                        \
  if (!(c)) {                                           \
    printf("line %d: %s (level %zu)\n", __LINE__, #c, l); \
    return 1;                                           \
  }

int main(int argc, char** argv) {
  const int nv = atoi(argv[1]), nt = atoi(argv[2]), R = atoi(argv[3]), kind = atoi(argv[5]);
  const std::string dir = argv[4];
  const auto verts = readv<double>(dir + "/verts.bin", 3 * (size_t)nv);
  const auto tets = readv<int>(dir + "/tets.bin", 4 * (size_t)nt);
  HostMesh m;
  build_general_mesh(m, verts.data(), nv, tets.data(), nt, R, 2, nullptr);
  std::vector<unsigned char> faulty(m.n_macro, 0);
  for (int a = 6; a < argc; ++a) faulty[atoi(argv[a])] = 1;
  HostProblem p;
  build_general_problem(m, kind, faulty, p);
  long rows = 0;
  for (size_t l = 1; l < m.lv.size(); ++l) {
    const HostLevel& L = m.lv[l];
    const int N = L.N;
    const HostProblemLevel& P = p.lv[l];
    const std::vector<int>& cptr = kind == 3 ? P.cptr : L.if_cptr;
    const std::vector<Copy>& copies = kind == 3 ? P.copies : L.if_copy;
    // node of every block slot: interface nodes, then n_if + slot
    std::map<int64_t, int64_t> node;
    for (int n = 0; n < L.n_if; ++n)
      for (int c = L.if_cptr[n]; c < L.if_cptr[n + 1]; ++c) {
        const Copy& cp = L.if_copy[c];
        node[(int64_t)cp.macro * L.block + lidx(L.SL.data(), N, cp.i, cp.j, cp.k)] = n;
      }
    auto id = [&](int64_t slot) {
      auto it = node.find(slot);
      return it == node.end() ? (int64_t)L.n_if + slot : it->second;
    };
    std::vector<uint32_t> ptr, nb;
    std::vector<int> len;
    std::vector<double> w, diag;
    CHECK(build_general_if_tables(m, (int)l, P.free_if, P.class_off, cptr, copies, ptr, len, nb, w, diag));
    CHECK(ptr.size() == P.free_if.size() && len.size() == ptr.size() && diag.size() == ptr.size());
    for (size_t q = 0; q < P.free_if.size(); ++q, ++rows) {
      const int n = P.free_if[q];
      std::map<int64_t, double> want;
      double dg = 0.0;
      for (int c = cptr[n]; c < cptr[n + 1]; ++c) {
        const Copy& cp = copies[c];
        const double* wm = &L.W[((size_t)cp.macro * 16 + node_class(cp.i, cp.j, cp.k, N)) * NDIR];
        dg += wm[0];
        for (int d = 1; d < NDIR; ++d) {
          int di, dj, dk;
          dir_ijk(d, di, dj, dk);
          if (wm[d] == 0.0 || !in_lattice(cp.i + di, cp.j + dj, cp.k + dk, N)) continue;
          want[id((int64_t)cp.macro * L.block + lidx(L.SL.data(), N, cp.i + di, cp.j + dj, cp.k + dk))] += wm[d];
        }
      }
      CHECK(diag[q] == dg);
      CHECK(len[q] % 4 == 0 && len[q] >= (int)want.size());
      CHECK((size_t)ptr[q] + 32 * (size_t)(len[q] - 1) < nb.size());
      std::map<int64_t, double> got;
      for (int e = 0; e < len[q]; ++e) {
        const int64_t v = id(nb[ptr[q] + 32 * e]);
        CHECK(v != n);                                   // padding does not read the node itself
        if (e < (int)want.size()) CHECK(got.find(v) == got.end());
        if (e >= (int)want.size()) CHECK(w[ptr[q] + 32 * e] == 0.0);
        got[v] += w[ptr[q] + 32 * e];
      }
      CHECK(got == want);                                // same sums in the same order of copies
    }
  }
  // offsets beyond 31 bits: no tables
  const size_t l = 1;
  HostMesh big = m;
  big.lv[1].block = (int64_t(1) << 31) / m.n_macro + 1;
  std::vector<uint32_t> ptr, nb;
  std::vector<int> len;
  std::vector<double> w, diag;
  CHECK(!build_general_if_tables(big, 1, p.lv[1].free_if, p.lv[1].class_off, big.lv[1].if_cptr, big.lv[1].if_copy, ptr,
                                 len, nb, w, diag));
  CHECK(ptr.empty() && nb.empty() && w.empty());
  printf("ok %ld rows\n", rows);
  return 0;
}
