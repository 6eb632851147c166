// Checks of the coarse space's kernels on their own, compared with the same sums
// in long double on the host.  Test infrastructure only.
//   coarse_main weights <leaves.bin> <level>   R against P^T in FP64
//   coarse_main gather <entries>               sums of the operator build in float
// Prints one number: the largest error over its bound.
#include "coarse.cu"

#include <cstdio>
#include <cstdlib>
#include <cstring>

using namespace chns;

namespace {
void must(cudaError_t e) {
  if (e != cudaSuccess) { std::fprintf(stderr, "%s\n", cudaGetErrorString(e)); std::exit(3); }
}

chns_mesh *read_mesh(const char *path) {
  FILE *f = std::fopen(path, "rb");
  int64_t n = 0;
  int32_t dim = 0, ml = 0;
  if (!f || std::fread(&n, 8, 1, f) != 1 || std::fread(&dim, 4, 1, f) != 1 || std::fread(&ml, 4, 1, f) != 1)
    std::exit(2);
  std::vector<uint8_t> lv(static_cast<size_t>(n));
  std::vector<uint32_t> an(size_t(n) * dim);
  if (std::fread(lv.data(), 1, lv.size(), f) != lv.size() || std::fread(an.data(), 4, an.size(), f) != an.size())
    std::exit(2);
  std::fclose(f);
  chns_mesh *m = nullptr;
  if (chns_mesh_create(dim, n, lv.data(), an.data(), ml, nullptr, nullptr, &m) != CHNS_OK) {
    std::fprintf(stderr, "%s\n", chns_last_error());
    std::exit(3);
  }
  return m;
}

double uniform(uint64_t &s) {  // in (0.5, 1)
  s = s * 6364136223846793005ull + 1442695040888963407ull;
  return 0.5 + double(s >> 11) / 18014398509481984.0;
}

// rc = P^T v (with the identity as coarse inverse): the sums of L terms may be off
// by their L + 1 roundings and by three of a weight in double
double weights(const char *path, int level) {
  chns_mesh *m = read_mesh(path);
  if (coarse_setup(m, level) != CHNS_OK) std::exit(3);
  Coarse &C = m->coarse;
  const int nf = m->nf, dim = m->dim;
  std::vector<double> I(size_t(C.nc) * C.nc, 0.0), v(size_t(m->n_nodes) * nf);
  for (int64_t k = 0; k < C.nc; ++k) I[size_t(k) * C.nc + k] = 1.0;
  must(cudaMemcpy(C.M.p, I.data(), sizeof(double) * I.size(), cudaMemcpyHostToDevice));
  C.ready = true;
  uint64_t s = 1;
  for (double &x : v) x = uniform(s);
  DevBuf dv, dz;
  if (dv.ensure(sizeof(double) * v.size()) != CHNS_OK || dz.ensure(sizeof(double) * v.size()) != CHNS_OK) std::exit(3);
  must(cudaMemcpy(dv.p, v.data(), sizeof(double) * v.size(), cudaMemcpyHostToDevice));
  must(cudaDeviceSynchronize());
  precond_apply<double>(m, nullptr, true, dv.as<double>(), dz.as<double>(), nullptr);
  std::vector<double> rc(static_cast<size_t>(C.nc));
  must(cudaMemcpy(rc.data(), C.vec.p, sizeof(double) * rc.size(), cudaMemcpyDeviceToHost));
  // hat functions from the node coordinates
  std::vector<long double> ref(size_t(C.nc), 0.0L);
  std::vector<int64_t> cnt(size_t(C.ncn), 0);
  const long double h = std::ldexp(1.0L, level - m->max_level);
  for (int64_t i = 0; i < m->n_nodes; ++i)
    for (int64_t c = 0; c < C.ncn; ++c) {
      long double w = 1.0L;
      int64_t r = c;
      for (int a = 0; a < dim; ++a) {
        w *= std::max(0.0L, 1.0L - std::fabs((long double)(m->node_xyz[i * dim + a]) * h - (long double)(r % C.nc1)));
        r /= C.nc1;
      }
      if (w == 0.0L) continue;
      ++cnt[c];
      for (int q = 0; q < nf; ++q) ref[c * nf + q] += w * (long double)v[i * nf + q];
    }
  double worst = 0.0;
  for (int64_t k = 0; k < C.nc; ++k)
    worst = std::max(worst, double(std::fabs((long double)rc[k] - ref[k]) / (ref[k] * (cnt[k / nf] + 4) * 0x1p-53L)));
  chns_mesh_destroy(m);
  return worst;
}

// A list of n entries of weight 1 around one coarse node, all in one slot: a one,
// then terms of just under half its last place, each of which is lost when it is
// added to a sum that holds the one.  Of the most roundings on the way of a term,
// 11, each is off by at most 2^-24 of the sum.
double gather_sums(int n) {
  constexpr int NF = 6, DIM = 3;
  // level 1: three coarse nodes an axis, the middle one (1, 1, 1) has number 13;
  // probe 13 NF: colour (1, 1, 1), whose node is the owner of the mesh nodes
  std::vector<int32_t> node(n), piece{13};
  std::vector<int64_t> begin{0, n};
  std::vector<float> w(n, 1.0f), pos(size_t(n) * DIM, 1.0f), y(size_t(n) * NF);
  long double ref[NF] = {0};
  for (int e = 0; e < n; ++e) {
    node[e] = e;
    for (int q = 0; q < NF; ++q) {
      y[size_t(e) * NF + q] = e == 0 ? 1.0f : 0x1.fffffep-25f * float(q + 1) / NF;
      ref[q] += (long double)y[size_t(e) * NF + q];
    }
  }
  int32_t *dpiece = nullptr, *dnode = nullptr;
  int64_t *dbegin = nullptr;
  float *dw = nullptr, *dpos = nullptr, *dy = nullptr;
  if (upload(&dpiece, piece) || upload(&dnode, node) || upload(&dbegin, begin) || upload(&dw, w) ||
      upload(&dpos, pos) || upload(&dy, y))
    std::exit(3);
  DevBuf part;
  if (part.ensure(sizeof(double) * 8 * NF) != CHNS_OK) std::exit(3);
  must(cudaDeviceSynchronize());
  CGeo g{DIM, NF, 3, n, 27, 27 * NF, 0};
  k_gather_coarse<float, NF, DIM><<<1, kChunk>>>(g, dpiece, dbegin, dnode, dw, dpos, 13 * NF, dy, part.as<double>());
  double out[8 * NF], worst = 0.0;
  must(cudaMemcpy(out, part.p, sizeof(out), cudaMemcpyDeviceToHost));
  for (int s = 0; s < 8; ++s)
    for (int q = 0; q < NF; ++q) {
      const long double want = s == 0 ? ref[q] : 0.0L;
      worst = std::max(worst, double(std::fabs((long double)out[s * NF + q] - want) / (11 * 0x1p-24L * ref[q])));
    }
  return worst;
}
}  // namespace

int main(int argc, char **argv) {
  double r = -1.0;
  if (argc == 4 && !std::strcmp(argv[1], "weights")) r = weights(argv[2], std::atoi(argv[3]));
  if (argc == 3 && !std::strcmp(argv[1], "gather")) r = gather_sums(std::atoi(argv[2]));
  if (r < 0.0) return 2;
  std::printf("%.6g\n", r);
  return 0;
}
