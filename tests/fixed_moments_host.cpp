// The fixed-point moment sums of fixed_moments.cuh run on the host, warp by
// warp over `per` paths as the backward kernel runs them, and the same sums
// in double in the same order of lanes.
#include "host_warp.h"

#include "fixed_moments.cuh"

using namespace lsmc;

namespace {

template <int BASIS>
void fixed_sums_t(int n, int per, const double* e, const double* v, const double* z, double xK,
                  double invTh, int neg, double* out) {
  using Sums = FixedSums<BASIS>;
  std::fill(out, out + Sums::NU, 0.0);
  double part[32];
  FixWarp ws;
  run_warp([&](int lane) {
    for (int w0 = 0; w0 < n; w0 += per) {
      const int m = std::min(per, n - w0);
      Sums acc;
      acc.start(ws);
      uint32_t settled = 0;  // of this lane's paths
      auto item = [&](int j, double& ej, double& vj, double& zj) {
        ej = e[w0 + j];
        vj = v[w0 + j];
        zj = z[w0 + j];
      };
      // lists of 96 paths, as the kernel's sub-tiles give them
      for (int l0 = 0; l0 < m; l0 += 96) {
        const int full = std::min(m, l0 + 96);
        const bool more = full < m;
        bool spilt = false, any = l0 > 0;
        if (!any) acc.grow(ws, false, 0, full, more, item, xK, invTh);
        for (int j0 = l0; j0 < full;) {
          const bool have = j0 + lane < full;
          double ej, vj, zj;
          item(have ? j0 + lane : j0, ej, vj, zj);
          if (acc.add(ws.scale, ej, vj, zj, have && !spilt, xK, invTh)) {
            j0 += 32;
            spilt = false;
            any = true;
          } else {
            acc.settle_mean((uint32_t)j0 / 32 - settled);
            settled = (uint32_t)j0 / 32;
            spilt = acc.grow(ws, any, j0, full, more, item, xK, invTh);
          }
        }
      }
      long long a[Sums::NU], b[Sums::NU], oa, ob;
      int i;
      acc.settle_mean((uint32_t)(m - lane + 31) / 32 * (lane < m) - settled);
      acc.units(a, b);
      halving_units<Sums::NU, 16>(a, b, lane, 0, Sums::NU, oa, ob, i);
      if (i >= 0) part[i] = Sums::value(i, oa, ob, ws.scale, neg != 0);
      __syncwarp();
      if (lane < Sums::NU) out[lane] += ws.spilled ? part[lane] + ws.spill[lane] : part[lane];
      __syncwarp();
    }
  });
}

template <int BASIS>
void double_sums_t(int n, int per, const double* e, const double* v, const double* z, double xK,
                   double invTh, double* out) {
  using Sums = FixedSums<BASIS>;
  std::fill(out, out + Sums::NU, 0.0);
  for (int w0 = 0; w0 < n; w0 += per) {
    const int m = std::min(per, n - w0);
    double s[32][Sums::NU] = {};
    for (int j = 0; j < m; ++j) {
      const double x = std::fma(e[w0 + j], xK, -1.0), y = z[w0 + j];
      const double w = Sums::kV ? std::fma(v[w0 + j], invTh, -1.0) : 0.0;
      const double xx = x * x, xw = x * w, ww = w * w;
      const double sq[3][3] = {{1.0, w, ww}, {x, xw, 0.0}, {xx, 0.0, 0.0}};
      for (int u = 0; u < Sums::NU; ++u) {
        const uint32_t t = Sums::unit(u);
        int a = (int)(t & 15u), b = (int)((t >> 4) & 15u);
        double p = 1.0, q = y;
        if (!((t >> 8) & 15u)) {  // the second factor: a basis function of degree 2 or less
          const int a2 = std::min(a, 2), b2 = std::min(b, 2 - a2);
          q = sq[a2][b2];
          a -= a2;
          b -= b2;
        }
        p = sq[a][b];
        s[j & 31][u] = std::fma(p, q, s[j & 31][u]);
      }
    }
    for (int o = 16; o > 0; o >>= 1)
      for (int l = 0; l < o; ++l)
        for (int u = 0; u < Sums::NU; ++u) s[l][u] += s[l + o][u];
    for (int u = 0; u < Sums::NU; ++u) out[u] += s[0][u];
  }
}

}  // namespace

extern "C" void fixed_sums(int sv2, int n, int per, const double* e, const double* v,
                           const double* z, double xK, double invTh, int neg, double* out) {
  if (sv2) fixed_sums_t<kBasisSV2>(n, per, e, v, z, xK, invTh, neg, out);
  else fixed_sums_t<kBasisS2>(n, per, e, v, z, xK, invTh, neg, out);
}

extern "C" void double_sums(int sv2, int n, int per, const double* e, const double* v,
                            const double* z, double xK, double invTh, double* out) {
  if (sv2) double_sums_t<kBasisSV2>(n, per, e, v, z, xK, invTh, out);
  else double_sums_t<kBasisS2>(n, per, e, v, z, xK, invTh, out);
}
