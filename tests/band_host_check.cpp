// Host check of the dense inverse of small meshes (band_order, band_inverse): run by tests/test_host_band_inverse.py on
// matrices written as CSR. Prints "OK <time of band_inverse / time of build_amg>", or what is wrong.
#include <chrono>
#include <cstdio>

#include "../paper_2502_10872_gb300/csrc/amg_setup.cpp"
#include "../paper_2502_10872_gb300/csrc/host_mesh.cpp"

using namespace shl;

static double now() {
  return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

int main(int argc, char **argv) {
  FILE *f = argc > 1 ? fopen(argv[1], "rb") : nullptr;
  int32_t head[2];
  if (!f || fread(head, 4, 2, f) != 2) return 2;
  HostCsr A;
  const int n = A.n = A.m = head[0];
  A.ptr.resize(n + 1);
  A.col.resize(head[1]);
  A.val.resize(head[1]);
  if (fread(A.ptr.data(), 4, n + 1, f) != (size_t)n + 1 || fread(A.col.data(), 4, head[1], f) != (size_t)head[1] ||
      fread(A.val.data(), 8, head[1], f) != (size_t)head[1])
    return 2;
  fclose(f);
  HostTopo T;
  T.nv = n;
  T.row_ptr = A.ptr;
  const HostSell S = to_sell(A);
  T.n_slices = S.n_slices;
  T.sl_ptr = S.sl_ptr;
  T.sl_col = S.sl_col;
  std::vector<uint8_t> skip(n, 1);
  std::vector<double> d(n);
  for (int i = 0; i < n; ++i)
    for (int k = A.ptr[i]; k < A.ptr[i + 1]; ++k) {
      if (A.col[k] != i && A.val[k] != 0.0) skip[i] = 0;
      if (A.col[k] == i) d[i] = std::sqrt(A.val[k]);
    }
  std::vector<int32_t> perm;
  const int band = band_order(T, skip.data(), &perm);
  std::vector<char> seen(n, 0);
  for (int32_t p : perm) {
    if (p < 0 || p >= n || seen[p]) return printf("not a permutation\n"), 1;
    seen[p] = 1;
  }
  std::vector<double> X;
  const double u = 0x1p-53;
  if (!band_inverse(A, perm, band, u, &X)) return printf("rejected\n"), 1;
  // S Y = I, S the matrix with unit diagonal and Y its inverse; a column's residual is bounded by c n u |S| |y|
  double snorm = 0.0;
  for (int i = 0; i < n; ++i) {
    double r = 0.0;
    for (int k = A.ptr[i]; k < A.ptr[i + 1]; ++k) r += std::fabs(A.val[k]) / (d[i] * d[A.col[k]]);
    snorm = std::max(snorm, r);
  }
  for (int j = 0; j < n; ++j) {
    double big = 0.0;
    for (int i = 0; i < n; ++i) {
      big = std::max(big, std::fabs(X[(size_t)i * n + j]) * d[i] * d[j]);
      if (X[(size_t)i * n + j] != X[(size_t)j * n + i]) return printf("not symmetric\n"), 1;
    }
    for (int i = 0; i < n; ++i) {
      double s = i == j ? -1.0 : 0.0;
      for (int k = A.ptr[i]; k < A.ptr[i + 1]; ++k)
        s += A.val[k] / (d[i] * d[A.col[k]]) * (X[(size_t)A.col[k] * n + j] * d[A.col[k]] * d[j]);
      if (!(std::fabs(s) <= 4.0 * n * u * snorm * big)) return printf("residual %g at (%d, %d)\n", s, i, j), 1;
    }
  }
  std::vector<double> B;
  if (band_inverse(A, perm, band, 0.5, &B)) return printf("held in one bit\n"), 1;   // |S| |Y| >= 1
  double t_inv = 1e300, t_amg = 1e300;
  for (int k = 0; k < 15; ++k) {
    const double t0 = now();
    band_inverse(A, perm, band, u, &B);
    const double t1 = now();
    HostAmg H;
    build_amg(A, &H);
    t_inv = std::min(t_inv, t1 - t0);
    t_amg = std::min(t_amg, now() - t1);
  }
  if (B != X) return printf("not reproducible\n"), 1;
  HostCsr N = A;   // indefinite: a free row's diagonal negated
  for (int i = n / 2; i < n; ++i)
    if (!skip[i]) {
      for (int k = N.ptr[i]; k < N.ptr[i + 1]; ++k)
        if (N.col[k] == i) N.val[k] *= 1e-3;
      break;
    }
  if (band_inverse(N, perm, band, u, &B)) return printf("indefinite matrix accepted\n"), 1;
  printf("OK %.3f\n", t_inv / t_amg);
  return 0;
}
