// precond_line.cu -- which grids the line kernels take, and their host tables.
#include "precond_line.cuh"

#include <cmath>

namespace gmrf {
namespace line {

// rows of a chunk and chunks of a scan lane for ny rows (must match col_launch)
static void col_plan(int ny, int& ry, int& seg) {
  ry = ny >= 4096 ? 16 : 8;
  seg = ny >= 2048 ? 16 : (ny >= 64 ? 8 : ny / 8);
}

void host_tables(int kind, int nx, int ny, double kbar2, HostTables& t) {
  const double pi = 3.14159265358979323846;
  const bool mir = kind == GMRF_PREC_MIRROR;
  const int L = nx / 2;
  t.tw.clear();
  for (int ns = 8; ns < L; ns *= 8) {
    const int rad = pass_radix(L, ns);
    for (int r = 1; r < rad; ++r)
      for (int j = 0; j < ns; ++j) {
        const double th = 2.0 * pi * j * r / ((double)ns * rad);
        t.tw.push_back(std::cos(th));
        t.tw.push_back(-std::sin(th));
      }
  }
  t.pair.clear();
  for (int k = 0; k < L / 2; ++k) {
    t.pair.push_back(std::cos(2.0 * pi * k / nx));
    t.pair.push_back(-std::sin(2.0 * pi * k / nx));
    if (!mir) continue;
    t.pair.push_back(std::cos(pi * k / (2.0 * nx)));
    t.pair.push_back(-std::sin(pi * k / (2.0 * nx)));
  }
  int ry, seg;
  col_plan(ny, ry, seg);
  t.col.clear();
  for (int i = 0; i < nx; ++i) {
    // transform index of packed position i
    const int k = i / 4, e = i % 4;
    int idx;
    if (mir) {
      const int of[4] = {k, k == 0 ? L : nx - k, k == 0 ? L / 2 : L - k, k == 0 ? nx - L / 2 : L + k};
      idx = of[e];
    } else {
      idx = k == 0 ? (e == 0 ? 0 : (e == 1 ? L : L / 2)) : (e < 2 ? k : L - k);
    }
    const double half = std::sin(mir ? pi * idx / (2.0 * nx) : pi * idx / (double)nx);
    const double s = kbar2 + 4.0 * half * half;
    const double root = std::sqrt(s * (s + 4.0));  // 1/rho - rho
    // 1 - rho = 2 s / (root + s): rho = 1 + s/2 - root/2, without the cancellation
    const double delta = 2.0 * s / (root + s);
    const double lr = std::log1p(-delta);
    const double den = -std::expm1((mir ? 2.0 : 1.0) * ny * lr);
    const double rec[8] = {delta, -std::expm1(ry * lr), std::exp(seg * ry * lr), std::exp(ny * lr), 1.0 / den,
                           2.0 / nx / root, 0.0, 0.0};
    t.col.insert(t.col.end(), rec, rec + 8);
  }
}

}  // namespace line

bool line_eligible(int power, int nx, int ny) {
  auto p2 = [](int v) { return v > 0 && (v & (v - 1)) == 0; };
  return power == 2 && p2(nx) && p2(ny) && nx >= 64 && nx <= 4096 && ny >= 8 && ny <= 4096;
}

int line_blocks_per_vector(int nx, int ny) {
  const int rb = line::block_rows(nx);
  return (ny + rb - 1) / rb;
}

}  // namespace gmrf
