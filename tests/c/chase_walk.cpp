// Walks the chase's schedule (csrc/chase_schedule.cuh) on the host, one
// rotation after another, on the band as the kernel's window holds it: six
// diagonals, row 1 apart, and cells to the right of and below the matrix,
// which start at zero and take part in the rotations like any other.  For
// every m x n with n <= 14 (m = n and m = n + 1, what the spike leaves) and
// every position of u and v: finite values reduce to an upper bidiagonal, and
// with a NaN, an infinity or an overflowing entry there no rotation names a
// row or column outside the matrix.
#include <cmath>
#include <cstdio>
#include <limits>
#include <vector>

#include "chase_schedule.cuh"

using namespace bdu::chase;

struct Walk {
  int m, n;
  Phases F;
  std::vector<double> band, r1, u, v;
  int outside = 0, rotations = 0;

  Walk(int m_, int n_) : m(m_), n(n_), F(phases_of(m_, n_)), band(6 * (F.N + 16)), r1(F.N + 16), u(F.N + 16), v(F.N + 16) {}
  double &at(int i, int j) { return i == 1 ? r1[j] : band[6 * i + (j - i + 2)]; }
  static bool nz(double x) { return !(x == 0.0); }

  // One op; last: the entry the chase looks at next.  False: nothing to rotate.
  bool op(int st, int a, double &last) {
    const Geo G = geo_of(st);
    const int lo = a - G.dl;
    double &f = G.src == 1 ? u[a] : G.src == 2 ? r1[a] : G.rows ? at(a, lo) : at(lo, a);
    double &g = G.src == 1 ? u[a + 1] : G.src == 2 ? r1[a + 1] : G.rows ? at(a + 1, lo) : at(lo, a + 1);
    if (!nz(g)) return false;
    rotations++;
    if (a < 1 || a + 1 > (G.rows ? F.N : n)) outside++;
    const double r = std::copysign(std::hypot(f, g), f);
    const double c = f == 0.0 ? 0.0 : f / r, s = f == 0.0 ? 1.0 : g / r;
    auto rot = [&](double &x, double &y) {
      const double p = c * x + s * y, q = c * y - s * x;
      x = p;
      y = q;
    };
    for (int q = 0; q < G.w; q++) {
      double &x = G.rows ? at(a, lo + q) : at(lo + q, a), &y = G.rows ? at(a + 1, lo + q) : at(lo + q, a + 1);
      if (&x != &f) rot(x, y);
      last = x;
    }
    if (G.withv) rot(v[a], v[a + 1]);
    const double rr = f == 0.0 ? g : r;
    f = rr;
    g = 0.0;
    return true;
  }

  void chase(int phase, int q) {
    int st, pos;
    if (!first_op(F, n, phase, q, st, pos)) return;
    for (;;) {
      double last = 0.0;
      const bool ok = op(st, pos, last);
      const Geo G = geo_of(st);
      const bool exists = pos + G.loff <= (G.limN ? F.N : n);
      if (exists && ((ok && nz(last)) || st == S_A)) { pos += G.dpos; st = G.next; }
      else if (ok && st == S_R1 && pos + 3 <= n && nz(at(pos + 1, pos + 3))) pos += 2;
      else if (ok && st == S_CL && pos + 4 <= F.N && nz(at(pos + 4, pos + 2))) pos += 3;
      else return;
    }
  }

  void run() {
    for (int q = 0; q < F.p1; q++) chase(1, q);
    for (int j = 1; j <= n; j++) r1[j] += u[1] * v[j];
    for (int q = 0; q < F.p2; q++) chase(2, q);
    for (int q = 0; q < F.p3; q++) chase(3, q);
  }

  void fill(unsigned seed) {
    auto rnd = [&]() {
      seed = seed * 1664525u + 1013904223u;
      return (double)(seed >> 8) / (1 << 24) + 0.25;
    };
    for (int i = 1; i <= n; i++) {
      at(i, i) = 1.0 + 9.0 * rnd();
      if (i < n) at(i, i + 1) = rnd() - 0.75;
    }
    for (int i = 1; i <= F.N; i++) u[i] = rnd() - 0.75;
    for (int j = 1; j <= n; j++) v[j] = rnd() - 0.75;
  }

  double off_bidiagonal() {
    double worst = 0.0;
    for (int i = 1; i <= F.N; i++)
      for (int j = i == 1 ? 1 : (i > 3 ? i - 2 : 1); j <= (i == 1 ? n : i + 3); j++)
        if (j <= n && j != i && j != i + 1) worst = std::fmax(worst, std::fabs(at(i, j)));
    return worst;
  }
};

int main() {
  const double bad[] = {std::numeric_limits<double>::quiet_NaN(), std::numeric_limits<double>::infinity(), 1e200};
  long walks = 0, outside = 0, rotations = 0;
  double worst = 0.0;
  for (int n = 1; n <= 14; n++)
    for (int m = n; m <= n + 1; m++) {
      Walk w(m, n);
      w.fill(17 * n + m);
      w.run();
      worst = std::fmax(worst, w.off_bidiagonal());
      outside += w.outside;
      const int N = w.F.N;
      for (double x : bad)
        for (int k = 1; k <= N + n; k++) {
          Walk t(m, n);
          t.fill(31 * n + m + k);
          (k <= N ? t.u[k] : t.v[k - N]) = x;
          if (x == 1e200) (k <= N ? t.v[1 + k % n] : t.u[1 + k % N]) = 1e200;  // u v^T overflows
          t.run();
          walks++;
          outside += t.outside;
          rotations += t.rotations;
        }
    }
  std::printf("walks %ld rotations %ld outside %ld off-bidiagonal %.1e\n", walks, rotations, outside, worst);
  return outside == 0 && worst < 1e-12 ? 0 : 1;
}
