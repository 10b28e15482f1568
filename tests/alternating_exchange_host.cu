// Host check of the alternating exchange layouts (Line<P, Q, T>, P = T, in
// csrc/dos_fft.cuh) on every compiled line shape, compiled by nvcc as host
// code, no GPU needed.  A forward DFT in the normal layout is followed by an
// inverse one in the transposed layout on the same buffer, thread by thread
// with no barrier between the second step of the first and the first step of
// the second: thread t writes its transposed entries before thread t + 1 has
// read its normal ones.  The round trip must give M x back.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_2604_02624_gb300/csrc/dos_fft.cuh"

using namespace dos;

template <int P, int Q, int T, int ZR>
static int check(const char* what) {
  using LF = Line<P, Q, T>;
  constexpr int M = P * Q, E = M / T;
  static_assert(LF::ALT, "compiled lines alternate");
  std::vector<float2> tw(LF::TWS + 1), z((size_t)Q * ZR + 2, make_float2(NAN, NAN));
  float2* twp = reinterpret_cast<float2*>((reinterpret_cast<size_t>(tw.data()) + 15) & ~size_t(15));
  float2* zp = reinterpret_cast<float2*>((reinterpret_cast<size_t>(z.data()) + 15) & ~size_t(15));
  const double pi = 3.14159265358979323846;
  for (int q = 0; q < Q; ++q)
    for (int k = 0; k < LF::TWP; ++k) {
      const double a = -2.0 * pi * ((q * k) % M) / M;
      twp[q * LF::TWP + k] = make_float2((float)std::cos(a), (float)std::sin(a));
    }
  std::mt19937 rng(M);
  std::normal_distribution<double> nd;
  std::vector<std::vector<float2>> r(T, std::vector<float2>(E)), x;
  for (auto& v : r)
    for (auto& e : v) e = make_float2((float)nd(rng), (float)nd(rng));
  x = r;
  auto at = [&](int t) -> float2(&)[E] { return *reinterpret_cast<float2(*)[E]>(r[t].data()); };
  double num = 0, den = 0;
  for (int pass = 0; pass < 2; ++pass) {  // the second pass meets the entries the first one left
    for (int t = 0; t < T; ++t) LF::template step1<false, P, false, false, ZR>(at(t), t, zp, twp);
    for (int t = 0; t < T; ++t) {
      LF::template step2<false, Q, false, false, ZR>(at(t), t, zp);
      LF::template step1<true, P, false, true, ZR>(at(t), t, zp, twp);
    }
    for (int t = 0; t < T; ++t) {
      LF::template step2<true, Q, false, true, ZR>(at(t), t, zp);
      for (int i = 0; i < E; ++i) {
        const double dx = r[t][i].x / M - x[t][i].x, dy = r[t][i].y / M - x[t][i].y;
        num += dx * dx + dy * dy;
        den += (double)x[t][i].x * x[t][i].x + (double)x[t][i].y * x[t][i].y;
      }
      r[t] = x[t];
    }
  }
  const double e = std::sqrt(num / den);
  // two FP32 DFTs: about 2^-24 sqrt(log2 M) each; 1e-6 is four times that at M = 512
  const bool ok = e < 1e-6;
  if (!ok) std::printf("FAIL %s M=%d pitch=%d: %.3e\n", what, M, ZR, e);
  return ok ? 0 : 1;
}

template <int P, int Q, int T>
static int shape() {
  return check<P, Q, T, Line<P, Q, T>::RP>("odd pitch") + check<P, Q, T, P + (P & 1)>("even pitch");
}

int main() {
  const int bad = shape<4, 4, 4>() + shape<4, 8, 4>() + shape<8, 8, 8>() + shape<8, 16, 8>() + shape<10, 20, 10>() +
                  shape<16, 16, 16>() + shape<20, 20, 20>() + shape<16, 32, 16>();
  std::printf("%s\n", bad ? "FAIL" : "OK");
  return bad ? 1 : 0;
}
