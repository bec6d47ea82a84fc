// Host check of the reflection-basis weights (k_sym.cu's tables, built by
// capi.cu): the blocks, contracted as the kernels contract them, equal the
// direct contraction with the plan's weight functions on random rows.
#include "capi.cu"

#include <random>

namespace {

double unfold(const double* L, int upper, const int par[3]) {  // L[s], s bit q: sign (0 +)
  double v = 0;
  for (int s = 0; s < 8; ++s) {
    double f = 1;
    for (int q = 0; q < 3; ++q)
      if (!((upper >> q) & 1)) f *= ((s >> q) & 1 ? -1.0 : 1.0) * (par[q] ? -1.0 : 1.0);
    v += f * L[s];
  }
  return v;
}

// B[s][k] of one component: A over positions -m .. 2m - 1 per axis (x fastest)
double block_value(const std::vector<double>& A, int m, int k, int s, int par) {
  const int n = 3 * m, h = n / 2;
  const int kk[3] = {k % h, (k / h) % h, k / (h * h)};
  double v = 0;
  for (int e = 0; e < 8; ++e) {
    int idx = 0, str = 1;
    double f = 1;
    for (int q = 0; q < 3; ++q) {
      const int lo = (e >> q) & 1;
      idx += str * (m + (lo ? m / 2 - 1 - kk[q] : m / 2 + kk[q]));
      str *= n;
      if (lo) f *= ((s >> q) & 1 ? -1.0 : 1.0) * ((par >> q) & 1 ? -1.0 : 1.0);
    }
    v += f * A[idx];
  }
  return v;
}

bool m2l_case(int p, int mo, int lo) {
  MultiIndex mi;
  mi.init(p);
  if (mo >= 0) mi.mo = mo;
  if (lo >= 0) mi.lo = lo;
  TaylorTable tt;
  tt.build(mi);
  SymHost H;
  sym_m2l_weights(mi, tt, H, true);
  const SymTab& T = H.tab;
  const std::vector<int> red = harmonic_components(mi);
  const int nk = T.nk;
  std::mt19937 rng(100 + p);
  std::uniform_real_distribution<double> U(-1, 1);
  std::vector<std::vector<double>> A(nk, std::vector<double>(216));
  for (auto& a : A)
    for (double& v : a) v = U(rng);
  double err = 0;
  for (int b = 0; b < nk; ++b) {
    const int u = b / 8, n = b % 8;
    double Lz[8] = {}, Lr[8] = {};  // z-run weights, row-form weights
    for (int a = 0; a < T.n1[u]; ++a) {
      const int nl = a < T.n8[u] ? 8 : a < T.n4[u] ? 4 : 1;
      if (n < nl) {
        const long long wo = T.w_off[u] + 216LL * (a < T.n8[u]   ? 8 * a
                                                   : a < T.n4[u] ? 8 * T.n8[u] + 4 * (a - T.n8[u])
                                                                 : 8 * T.n8[u] + 4 * (T.n4[u] - T.n8[u]) + a - T.n4[u]);
        for (int k = 0; k < 27; ++k)
          for (int s = 0; s < 8; ++s)
            Lz[s] += block_value(A[a], 2, k, s, T.par[a]) *
                     H.Ws[wo + ((((k % 9) * 4 + (s & 3)) * 3 + k / 9) * nl + n) * 2 + (s >> 2)];
      }
      if (a < T.kb[b])
        for (int k = 0; k < 27; ++k)
          for (int s = 0; s < 8; ++s)
            Lr[s] += block_value(A[a], 2, k, s, T.par[a]) * H.Wq[(size_t)k * T.q_len + T.q_off[a] + b * 8 + s];
    }
    for (int a = T.n1[u]; a < nk; ++a)
      if (a < T.kb[b]) return false;  // a pair no unit holds
    const int par[3] = {T.par[b] & 1, (T.par[b] >> 1) & 1, (T.par[b] >> 2) & 1};
    for (int c = 0; c < 8; ++c) {
      double ref = 0, sabs = 0;
      for (int a = 0; a < nk; ++a)
        for (int d = 0; d < 27; ++d)
          for (int cs = 0; cs < 8; ++cs) {
            const int D[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
            int idx = 0, str = 1;
            for (int q = 0; q < 3; ++q) idx += str * (2 + 2 * D[q] + ((cs >> q) & 1)), str *= 6;
            const double t = A[a][idx] * m2l_entry(mi, tt, d, red[a] * 8 + cs, red[b] * 8 + c);
            ref += t;
            sabs += std::fabs(t);
          }
      const double e = std::max(std::fabs(unfold(Lz, c, par) - ref), std::fabs(unfold(Lr, c, par) - ref));
      if (sabs > 0) err = std::max(err, e / sabs);
      else if (e != 0) return false;
    }
  }
  std::printf("reflection m2l p=%d mo=%d lo=%d: err/sum|terms| %.1e\n", p, mi.mo, mi.lo, err);
  return err <= 1e-13;
}

bool near_case() {
  std::vector<double> W;
  sym_near4_weights(W);
  std::mt19937 rng(7);
  std::uniform_real_distribution<double> U(0, 1);
  std::vector<double> A(1728);
  for (double& v : A) v = U(rng);
  double err = 0;
  for (int n = 0; n < 8; ++n) {
    double L[8] = {};
    for (int k = 0; k < 216; ++k)
      for (int s = 0; s < 8; ++s)
        L[s] += block_value(A, 4, k, s, 0) * W[((((k % 36) * 4 + (s & 3)) * 6 + k / 36) * 8 + n) * 2 + (s >> 2)];
    const int par[3] = {0, 0, 0};
    for (int c = 0; c < 8; ++c) {
      int t[3];
      for (int q = 0; q < 3; ++q) t[q] = (c >> q) & 1 ? 2 + ((n >> q) & 1) : 1 - ((n >> q) & 1);
      double ref = 0;
      for (int d = 0; d < 27; ++d) {
        const int D[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
        for (int sc = 0; sc < 64; ++sc) {
          const int j[3] = {sc % 4, (sc / 4) % 4, sc / 16};
          const int idx = (4 + 4 * D[0] + j[0]) + 12 * (4 + 4 * D[1] + j[1]) + 144 * (4 + 4 * D[2] + j[2]);
          ref += A[idx] * near_entry(4, D, sc, t[0] + 4 * t[1] + 16 * t[2]);
        }
      }
      err = std::max(err, std::fabs(unfold(L, c, par) / ref - 1));
    }
  }
  std::printf("reflection near: err %.1e\n", err);
  return err <= 1e-13;
}

bool near2_case() {
  SymHost H;
  sym_near2_weights(H);
  std::mt19937 rng(8);
  std::uniform_real_distribution<double> U(0, 1);
  std::vector<double> A(216);
  for (double& v : A) v = U(rng);
  double L[8] = {}, err = 0;
  for (int k = 0; k < 27; ++k)
    for (int s = 0; s < 8; ++s)
      L[s] += block_value(A, 2, k, s, 0) * H.Ws[(((k % 9) * 4 + (s & 3)) * 3 + k / 9) * 2 + (s >> 2)];
  const int par[3] = {0, 0, 0};
  for (int c = 0; c < 8; ++c) {
    double ref = 0;
    for (int d = 0; d < 27; ++d)
      for (int sc = 0; sc < 8; ++sc) {
        const int D[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
        int idx = 0, str = 1;
        for (int q = 0; q < 3; ++q) idx += str * (2 + 2 * D[q] + ((sc >> q) & 1)), str *= 6;
        ref += A[idx] * near_entry(2, D, sc, c);
      }
    err = std::max(err, std::fabs(unfold(L, c, par) / ref - 1));
  }
  std::printf("reflection near leaf 2: err %.1e\n", err);
  return err <= 1e-13 && H.tab.n1[0] == 1 && H.tab.n8[0] == 0;
}

bool m2p_case(int p, int b, int mo) {
  MultiIndex mi;
  mi.init(p);
  if (mo >= 0) mi.mo = mo;
  M2pTable tab;
  tab.build(mi, b);
  SymHost H;
  sym_m2p_weights(mi, tab, b, H);
  const SymTab& T = H.tab;
  const std::vector<int> red = harmonic_components(mi);
  const int b3 = b * b * b;
  std::mt19937 rng(30 + p);
  std::uniform_real_distribution<double> U(-1, 1);
  std::vector<std::vector<double>> A(T.nk, std::vector<double>(216));
  for (auto& a : A)
    for (double& v : a) v = U(rng);
  double err = 0;
  for (int cell = 0; cell < b3; ++cell) {
    double L[8] = {};
    for (int a = 0; a < T.nk; ++a)
      for (int k = 0; k < 27; ++k)
        for (int s = 0; s < 8; ++s)
          L[s] += block_value(A[a], 2, k, s, T.par[a]) *
                  H.Ws[T.w_off[cell / 8] + (long long)a * 216 * 8 +
                       ((((k % 9) * 4 + (s & 3)) * 3 + k / 9) * 8 + cell % 8) * 2 + (s >> 2)];
    const int par[3] = {0, 0, 0}, o[3] = {cell % b, (cell / b) % b, cell / (b * b)};
    for (int c = 0; c < 8; ++c) {
      int t[3];
      for (int q = 0; q < 3; ++q) t[q] = (c >> q) & 1 ? o[q] : b - 1 - o[q];
      double ref = 0, sabs = 0;
      for (int a = 0; a < T.nk; ++a)
        for (int d = 0; d < 27; ++d)
          for (int cs = 0; cs < 8; ++cs) {
            const int D[3] = {d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1};
            int idx = 0, str = 1;
            for (int q = 0; q < 3; ++q) idx += str * (2 + 2 * D[q] + ((cs >> q) & 1)), str *= 6;
            const double v = A[a][idx] * m2p_entry(mi, tab, d, red[a] * 8 + cs, c * b3 + (t[2] * b + t[1]) * b + t[0]);
            ref += v;
            sabs += std::fabs(v);
          }
      err = std::max(err, std::fabs(unfold(L, c, par) - ref) / sabs);
    }
  }
  std::printf("reflection M2P p=%d b=%d mo=%d: err/sum|terms| %.1e\n", p, b, mi.mo, err);
  return err <= 1e-13;
}

}  // namespace

int main() {
  bool ok = near_case() && near2_case() && m2p_case(3, 2, 2) && m2p_case(4, 4, -1) && m2p_case(6, 2, -1);
  for (int p = 2; p <= 8; ++p) ok &= m2l_case(p, -1, -1);
  ok &= m2l_case(3, 2, -1) && m2l_case(3, -1, 2) && m2l_case(6, 4, -1) && m2l_case(6, -1, 4) && m2l_case(4, 0, -1);
  return ok ? 0 : 1;
}
