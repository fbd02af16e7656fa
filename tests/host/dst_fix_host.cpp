// Host run of the fixed-point DST phases (one simulated thread at a time, a
// barrier between phases) for checking index arithmetic and error on the
// CPU.  stdin (binary): int32 N, RS, then 32 columns of N-1 float64 values;
// stdout (binary): the 32 transformed columns.
#include <cmath>
#include <cstdio>
#include <vector>

#include "dst_fix.cuh"

using namespace kfbi::fixdst;

template <int N, int RS>
int run() {
  using G = Geo<N, RS>;
  std::vector<double> s((size_t)N * RS, 0.0), x((size_t)32 * (N - 1));
  if (std::fread(x.data(), sizeof(double), x.size(), stdin) != x.size()) return 1;
  for (int c = 0; c < 32; ++c)
    for (int j = 1; j < N; ++j) s[(size_t)j * RS + c] = x[(size_t)c * (N - 1) + j - 1];
  const long double pi = 3.14159265358979323846264338327950288L;
  std::vector<double> tw(4 * N);
  for (int j = 0; j < 2 * N; ++j) {
    tw[2 * j] = (double)std::cos(pi * j / N);
    tw[2 * j + 1] = (double)std::sin(pi * j / N);
  }
  std::vector<cfx> sp(N / 2), lv(N / 2);
  std::vector<fx> sinv(N / 2);
  for (int i = 0; i < N / 2; ++i) table_entry<N>(i, tw.data(), sp.data(), lv.data(), sinv.data());
  std::vector<int> mx(256);
  std::vector<uint32_t> sm(256);
  std::vector<ll> tot(256);
  std::vector<State<G>> st(256);
  ll* si = reinterpret_cast<ll*>(s.data());
  c2* ex = reinterpret_cast<c2*>(s.data());
  for (int t = 0; t < 256; ++t) phase_0<G>(st[t], s.data(), mx.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_s<G>(st[t], mx.data(), sm.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_1<G>(st[t], si, sm.data(), sinv.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_a1<G>(st[t], si, sp.data(), lv.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_a2<G>(st[t], ex, t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_c<G>(st[t], ex, t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_d<G>(st[t], si, sp.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_e1<G>(st[t], si, tot.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_e2<G>(st[t], si, tot.data(), t >> 5, t & 31);
  for (int t = 0; t < 256; ++t) phase_f<G>(st[t], s.data(), t >> 5, t & 31);
  for (int c = 0; c < 32; ++c)
    for (int j = 1; j < N; ++j) x[(size_t)c * (N - 1) + j - 1] = s[(size_t)j * RS + c];
  std::fwrite(x.data(), sizeof(double), x.size(), stdout);
  return 0;
}

int main() {
  int32_t p[2];
  if (std::fread(p, sizeof(int32_t), 2, stdin) != 2) return 1;
  const bool pad = p[1] != 32;
  switch (p[0]) {
    case 32: return pad ? run<32, 33>() : run<32, 32>();
    case 64: return pad ? run<64, 33>() : run<64, 32>();
    case 128: return pad ? run<128, 33>() : run<128, 32>();
    case 256: return pad ? run<256, 33>() : run<256, 32>();
    case 384: return pad ? run<384, 33>() : run<384, 32>();
    case 512: return pad ? run<512, 33>() : run<512, 32>();
    default: return 2;
  }
}
