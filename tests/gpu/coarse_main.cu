// Checks of the coarse space's kernels on their own, compared with the same sums
// in long double on the host.  Test infrastructure only.
//   coarse_main weights <leaves.bin> <level>   R against P^T in FP64
//   coarse_main gather <entries>               sums of the operator build in float
//   coarse_main restrict <entries>             sums of the restriction in float
//   coarse_main pieces <pieces>                the restriction's sum over a list's pieces
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

// n terms a component: a one, then terms of just under half its last place, each
// of which is lost when it is added to a sum that holds the one.  Of the `most`
// roundings on the way of a term each is off by at most 2^-24 of the sum.
constexpr int NF = 6;
struct Terms {
  std::vector<float> y;
  long double ref[NF] = {0};
  explicit Terms(int n) : y(size_t(n) * NF) {
    for (int e = 0; e < n; ++e)
      for (int q = 0; q < NF; ++q) {
        y[size_t(e) * NF + q] = e == 0 ? 1.0f : 0x1.fffffep-25f * float(q + 1) / NF;
        ref[q] += (long double)y[size_t(e) * NF + q];
      }
  }
  double error(const double *out, int most) const {
    double worst = 0.0;
    for (int q = 0; q < NF; ++q)
      worst = std::max(worst, double(std::fabs((long double)out[q] - ref[q]) / (most * 0x1p-24L * ref[q])));
    return worst;
  }
};

template <class T>
T *on_device(const std::vector<T> &x) {
  T *d = nullptr;
  if (upload(&d, x) != CHNS_OK || uploads_done(d, int64_t(x.size())) != CHNS_OK) std::exit(3);
  return d;
}

// a list of n entries of weight 1 around one coarse node, all in one slot
double gather_sums(int n) {
  constexpr int DIM = 3;
  // level 1: three coarse nodes an axis, the middle one (1, 1, 1) has number 13;
  // probe 13 NF: colour (1, 1, 1), whose node is the owner of the mesh nodes
  std::vector<int32_t> node(n), piece{13};
  for (int e = 0; e < n; ++e) node[e] = e;
  const std::vector<int64_t> begin{0, n};
  const std::vector<float> w(n, 1.0f), pos(size_t(n) * DIM, 1.0f);
  const Terms t(n);
  DevBuf part;
  if (part.ensure(sizeof(double) * 8 * NF) != CHNS_OK) std::exit(3);
  CGeo g{DIM, NF, 3, n, 27, 27 * NF, 0};
  k_gather_coarse<float, NF, DIM><<<1, kChunk>>>(g, on_device(piece), on_device(begin), on_device(node), on_device(w),
                                                 on_device(pos), 13 * NF, on_device(t.y), part.as<double>());
  double out[8 * NF];
  must(cudaMemcpy(out, part.p, sizeof(out), cudaMemcpyDeviceToHost));
  for (int k = NF; k < 8 * NF; ++k)
    if (out[k] != 0.0) return 1e30;
  return t.error(out, 11);
}

// the restriction of one piece of n entries of weight 1, or of n pieces
double restrict_sums(int n, bool pieces) {
  const Terms t(n);
  DevBuf rc;
  if (rc.ensure(sizeof(float) * NF) != CHNS_OK) std::exit(3);
  if (pieces) {
    const std::vector<int32_t> node_piece{0, n};
    k_restrict_pieces<float><<<1, kB>>>(NF, NF, on_device(node_piece), on_device(t.y), rc.as<float>());
  } else {
    std::vector<int32_t> node(n);
    for (int e = 0; e < n; ++e) node[e] = e;
    const std::vector<int64_t> begin{0, n};
    const std::vector<float> w(n, 1.0f);
    k_restrict_lists<float, NF><<<1, kGroups * 8>>>(on_device(begin), on_device(node), on_device(w), on_device(t.y),
                                                    rc.as<float>());
  }
  float f[NF];
  must(cudaMemcpy(f, rc.p, sizeof(f), cudaMemcpyDeviceToHost));
  double out[NF];
  for (int q = 0; q < NF; ++q) out[q] = f[q];
  return t.error(out, pieces ? (n + 7) / 8 + 3 : 15);
}
}  // namespace

int main(int argc, char **argv) {
  double r = -1.0;
  if (argc == 4 && !std::strcmp(argv[1], "weights")) r = weights(argv[2], std::atoi(argv[3]));
  if (argc == 3 && !std::strcmp(argv[1], "gather")) r = gather_sums(std::atoi(argv[2]));
  if (argc == 3 && !std::strcmp(argv[1], "restrict")) r = restrict_sums(std::atoi(argv[2]), false);
  if (argc == 3 && !std::strcmp(argv[1], "pieces")) r = restrict_sums(std::atoi(argv[2]), true);
  if (r < 0.0) return 2;
  std::printf("%.6g\n", r);
  return 0;
}
