// Host side of the double-precision tensor-core passes: digit tables of the
// derivative matrices, tile geometries, launches. See ts_emu.cuh.
#include "ts_emu.cuh"

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <vector>

#include "ts_launch.cuh"

namespace ts {

namespace {

// Matrix entries are formed in long double (64 bits and more): the digits hold 62
// bits of a row, and the rounding of the entries to double would be the largest
// error left in a contraction. Long double is software on Arm: every function value
// is formed once, by its index.
typedef long double Wide;
const Wide kPi = 3.14159265358979323846264338327950288L;

// The Chebyshev-Gauss-Lobatto and periodic Fourier derivative matrices of ts_api.cu.
std::vector<Wide> cheb_wide(int Nr, double R1, double R2) {
  const int N = Nr - 1;
  std::vector<Wide> D((size_t)Nr * Nr, 0.0L);
  auto w = [&](int i) { return ((i % 2) ? -1.0L : 1.0L) * (i == 0 || i == N ? 0.5L : 1.0L); };
  const Wide s = 2.0L / ((Wide)R2 - (Wide)R1);
  std::vector<Wide> sn(2 * N + 1);   // sin(pi q / (2 N))
  for (int q = 0; q <= 2 * N; ++q) sn[q] = sinl(kPi * q / (2.0L * N));
  for (int i = 0; i < Nr; ++i) {
    Wide diag = 0.0L;
    for (int j = 0; j < Nr; ++j) {
      if (i == j) continue;
      const Wide dx = 2.0L * sn[i + j] * (i > j ? sn[i - j] : -sn[j - i]);
      const Wide v = w(j) / w(i) / dx * s;
      D[(size_t)i * Nr + j] = v;
      diag -= v;
    }
    D[(size_t)i * Nr + i] = diag;
  }
  return D;
}
std::vector<Wide> fourier_wide(int M) {
  std::vector<Wide> D((size_t)M * M, 0.0L), c(M, 0.0L);
  for (int q = 1; q < M; ++q)   // cot(pi / 2) = 0
    if (2 * q != M) c[q] = 0.5L * (q % 2 ? -1.0L : 1.0L) / tanl(q * kPi / M);
  for (int j = 0; j < M; ++j)
    for (int k = 0; k < M; ++k) D[(size_t)j * M + k] = j >= k ? c[j - k] : -c[k - j];
  return D;
}

typedef std::vector<std::vector<Wide>> Mat;   // [output][K element]

// An f16 integer of magnitude at most 2048.
uint16_t f16_int(int v) {
  if (v == 0) return 0;
  const int a = std::abs(v);
  int e = 0;
  while ((2 << e) <= a) ++e;
  return (uint16_t)((v < 0 ? 0x8000 : 0) | ((e + 15) << 10) | (((a - (1 << e)) << 10) >> e));
}

// The scale of a row (see digits_of), at most smax.
int scale_of(const std::vector<Wide>& row, int smax) {
  double mx = 0.0, tot = 0.0;
  for (const Wide& w : row) {
    const double a = std::fabs((double)w);
    mx = std::max(mx, a);
    tot += a;
  }
  if (mx == 0.0) return smax;
  return std::min(std::min(62 - (std::ilogb(mx) + 1), 65 - (std::ilogb(tot) + 1)), smax);
}
// The digits of a row: value 2^s rounded to an integer below 2^62, s the largest with
// sum |Dfix| < 2^65; digits balanced, most significant first.
struct Row {
  int s = 0;
  std::vector<std::array<int, 8>> e;
};
Row digits_of(const std::vector<Wide>& row, int smax) {
  Row r;
  r.e.resize(row.size());
  for (auto& e : r.e) e.fill(0);
  r.s = scale_of(row, smax);
  for (size_t k = 0; k < row.size(); ++k) {
    if (row[k] == 0.0L) continue;
    long long v = llrintl(ldexpl(row[k], r.s));
    for (int j = 7; j >= 0; --j) {
      const int q = j == 0 ? (int)v : (int)((((v + 128) % 256) + 256) % 256) - 128;
      r.e[k][j] = q;
      v = (v - q) / 256;
    }
  }
  return r;
}

// Builds the operand of `m` (K elements already in core order, -1 columns zero):
// `left` (>= 0): that K element rides in the bias MMA. False if an accumulator
// could leave the range in which its bit pattern is linear.
bool build_operand(const Mat& m, const std::vector<int>& order, int left, bool common, EmuMat* out,
                   std::vector<uint16_t>* bits, std::vector<int>* se) {
  out->nout = (int)m.size();
  out->n = (out->nout + 7) / 8 * 8;
  out->rows = 8 * out->n + 16;
  out->kc = (int)order.size() / 8;
  out->extra = left >= 0 ? 1 : 0;
  const size_t core = (size_t)out->rows * 8;
  bits->assign(core * (1 + out->extra + out->kc), 0);
  se->assign(out->n, 3);
  uint16_t* bias = bits->data();
  uint16_t* ext = bias + core;
  uint16_t* main = bias + core * (1 + out->extra);
  int smin = 1 << 20;   // the scale every row has where they share one
  for (const auto& row : m) smin = std::min(smin, scale_of(row, 1 << 20));
  if (smin == 1 << 20) smin = 60;   // a matrix of zeros
  out->s = smin;
  for (int o = 0; o < out->nout; ++o) {
    Row r = digits_of(m[o], common ? smin : 1 << 20);
    auto largest = [&]() {
      long long worst = 0;
      for (int od = 0; od < 8; ++od) {
        long long a = 0;
        for (const auto& e : r.e)
          for (int j = 0; j <= od; ++j) a += std::abs(e[j]);
        worst = std::max(worst, 128 * a);
      }
      return worst;
    };
    if (largest() >= (1 << 22))
      for (auto& e : r.e) e[7] = 0;   // the last digit (2^-56 of the row) makes room
    if (largest() >= (1 << 22)) return false;
    (*se)[o] = 3 - r.s;
    for (int od = 0; od < 8; ++od) {
      long long tot = 0;
      for (const auto& e : r.e)
        for (int j = 0; j <= od; ++j) tot += e[j];
      const long long c = -tot;
      const int c0 = (int)(((c + 32) % 64 + 64) % 64) - 32, c1 = (int)((c - c0) / 64);
      if (std::abs(c1) > 2048) return false;
      uint16_t* b = bias + (size_t)(od * out->n + o) * 8;
      b[0] = 0x3C00;           // 1.0 x 0.75
      b[1] = f16_int(c1);      // x 2^-11 = 128 x 64 units
      b[2] = f16_int(c0);      // x 2^-17 = 128 units
      if (left >= 0)
        for (int i = 0; i <= od; ++i)
          ext[(size_t)(od * out->n + o) * 8 + i] = f16_int(r.e[left][od - i]);
    }
    for (int j = 0; j < 8; ++j)
      for (size_t x = 0; x < order.size(); ++x)
        if (order[x] >= 0)
          main[(x / 8) * core + (size_t)(j * out->n + o) * 8 + x % 8] = f16_int(r.e[order[x]][j]);
  }
  // accumulators of padded outputs stay at zero bits or small sums: never read
  return true;
}

// K order of a DFS axis of N nodes: the line's cores and the partner line's, each
// padded to 8; with an odd number of cores the two last ones make up one step.
std::vector<int> dfs_order(int N) {
  const int k = (N + 7) / 8, full = k / 2 * 2;
  std::vector<int> o;
  auto put = [&](int side, int c) {
    for (int z = 0; z < 8; ++z) o.push_back(c * 8 + z < N ? side * N + c * 8 + z : -1);
  };
  for (int side = 0; side < 2; ++side)
    for (int c = 0; c < full; ++c) put(side, c);
  if (k & 1)
    for (int side = 0; side < 2; ++side) put(side, k - 1);
  return o;
}
std::vector<int> plain_order(int N, int cores) {
  std::vector<int> o;
  for (int z = 0; z < cores * 8; ++z) o.push_back(z < N ? z : -1);
  return o;
}

int pow2_at_least(int n) {
  int c = 32;
  while (c < n) c *= 2;
  return c;
}
int region(int n) { return 8 * n + (n % 16 ? 16 : 0); }

constexpr int kTwoCtas = 113 * 1024;   // shared memory of each of two CTAs on an SM
constexpr int kOneCta = 227 * 1024;

bool geometry2_form(int xw, bool seq, int Na, int Nb, const EmuMat& D, const EmuMat& F, int nf,
                    int nz, bool adj, EmuGeo* out) {
  EmuGeo g{};
  g.xw = xw;
  g.seq = seq ? 1 : 0;
  g.Na = Na;
  g.Nb = Nb;
  g.hb = Nb / 2;
  g.ka = (Na + 7) / 8;
  g.kb = (Nb + 7) / 8;
  g.nf = nf;
  g.nz = nz;
  g.kc1 = D.kc;
  g.kc2 = F.kc;
  g.n1 = D.n;
  g.n2 = F.n;
  g.r1 = D.rows;
  g.r2 = F.rows;
  g.mt1 = (Nb * xw + 127) / 128;
  g.mt2 = (Na * xw + 127) / 128;
  const int hg = g.hb * xw / 8;   // row groups of half the Fourier axis
  // copy 1: 16 (32) bytes more per row group, so that the stores of a warp (consecutive
  // b; or pairs of a) fall on distinct banks
  g.sb1 = g.ka * 128 + (xw == 8 ? 16 : 32);
  g.d1 = 3 * hg * g.sb1;
  g.sb2 = g.kb * 128;
  g.d2 = (Na * xw + 7) / 8 * g.sb2;
  g.exP = Na * xw + 8;
  const int exB = Nb * g.exP * 8;
  const bool alias =
      xw == 8 && g.mt2 == 1 && Na % 8 == 0 && Nb % 8 == 0 && exB <= 8 * g.d2;
  int o = 0;
  auto take = [&](int bytes) {
    const int at = o;
    o += (bytes + 127) / 128 * 128;
    return at;
  };
  g.oC1 = take(seq ? 8 * std::max(g.d1, g.d2) : 8 * g.d1);
  g.oC2 = seq ? g.oC1 : take(8 * g.d2);
  g.oB1 = take(D.bytes());
  g.oB2 = take(F.bytes());
  g.oCA = take(2 * 128 * 16);
  g.oEx = alias ? g.oC2 : take(exB);
  // header, scalars, moments; angular: weights and shares; plane: shifts
  const int kf = nf >= 5 ? 2 : nf >= 3 ? 1 : 0;
  const int shares = std::max(4 * emu_moments(kf), adj ? g.mt1 * 16 : 0) * 8;
  g.oMs = take(96 + (128 + 80 + (nf ? emu_weights(kf) * Na + shares : Na)) * 8);
  g.oLn = take((g.hb + Na) * xw * 2);
  // a 128-row tile may read row groups past the last one: inside the allocation
  const int over = std::max(g.oC1 + 7 * g.d1 + (16 * g.mt1 + hg) * g.sb1 + 256,
                            g.oC2 + 7 * g.d2 + 16 * g.mt2 * g.sb2 + 256);
  g.bytes = (std::max(o, over) + 127) / 128 * 128;
  const int reg = std::max(region(g.n1), region(g.n2));
  if (reg > 512 || Na * Nb > 1024) return false;
  if (xw == 8 && g.bytes <= kTwoCtas && reg <= 256 && Na * Nb <= 256) {
    g.threads = 256;
    g.half = pow2_at_least(reg);
    g.dual = g.half <= 128 && (g.mt2 == 1 || !alias);
    g.cols = g.dual ? 2 * g.half : g.half;
  } else if (g.bytes <= kOneCta) {
    g.threads = 512;
    g.half = pow2_at_least(reg);
    g.dual = g.half <= 256;
    g.cols = g.dual ? 2 * g.half : g.half;
  } else {
    return false;
  }
  if ((xw == 4 ? (Na + 1) / 2 : Na) * Nb > g.threads) return false;   // one unit a thread
  if (seq && g.mt2 > (g.dual ? 2 : 1)) return false;
  *out = g;
  return true;
}
// Eight x where both copies fit; else four (which need whole pairs in each half of the
// Fourier axis), with the copies in one buffer if need be.
bool geometry2(int Na, int Nb, const EmuMat& D, const EmuMat& F, int nf, int nz, bool adj,
               EmuGeo* out) {
  if (geometry2_form(8, false, Na, Nb, D, F, nf, nz, adj, out)) return true;
  if (Nb % 4) return false;
  return geometry2_form(4, false, Na, Nb, D, F, nf, nz, adj, out) ||
         geometry2_form(4, true, Na, Nb, D, F, nf, nz, adj, out);
}

bool geometry_radial(int Nr, EmuRadGeo* out) {
  EmuRadGeo g{};
  g.Nr = Nr;
  g.left = Nr % 16 == 1 ? 1 : 0;
  g.kc = g.left ? (Nr - 1) / 8 : (Nr + 15) / 16 * 2;
  g.sb = g.kc * 128 + 16;
  g.d = 16 * g.sb;
  // two CTAs on an SM; one; one with the matrices streamed through two buffers
  for (int form = 0; form < 3; ++form) {
    const bool two = form == 0;
    for (int go = 32; go >= 8; go -= 8) {   // outputs per group: whole cores, fewest groups
      const int ng = (Nr + go - 1) / go;
      if (ng > 8) break;
      g.ng = ng;
      g.nb = form == 2 ? 2 : ng;
      if (form == 2 && ng < 3) continue;
      g.go = (Nr + ng - 1) / ng;
      g.n = (g.go + 7) / 8 * 8;
      g.rows = 8 * g.n + 16;
      const int reg = region(g.n);
      if (reg > 256) continue;
      g.bB = (1 + g.left + g.kc) * g.rows * 16;
      int o = 0;
      auto take = [&](int bytes) {
        const int at = o;
        o += (bytes + 127) / 128 * 128;
        return at;
      };
      g.oA = take(8 * g.d + 256);
      g.oB = take(g.nb * g.bB);
      g.oCA = take(2 * 128 * 16);
      g.oMs = take(64 + (ng * g.n * 4 + 15) / 16 * 16 + 128 * 8 + 2 * 128 * 4);
      g.bytes = o;
      if (g.bytes > (two ? kTwoCtas : kOneCta)) continue;
      g.threads = two ? 256 : 512;
      if (Nr * 16 > kEmuRadUnits * g.threads) continue;
      g.half = pow2_at_least(reg);
      g.dual = g.half <= (two ? 128 : 256) && ng > 1;
      g.cols = g.dual ? 2 * g.half : g.half;
      if (form == 2 && !g.dual) continue;
      *out = g;
      return true;
    }
  }
  return false;
}

struct Upload {
  std::vector<unsigned char> host;
  std::vector<std::pair<EmuMat*, std::pair<size_t, size_t>>> fix;
  void add(EmuMat* m, const std::vector<uint16_t>& b, const std::vector<int>& se) {
    auto put = [&](const void* p, size_t n) {
      const size_t at = (host.size() + 255) / 256 * 256;
      host.resize(at + n);
      std::memcpy(host.data() + at, p, n);
      return at;
    };
    const size_t a = put(b.data(), b.size() * 2), s = put(se.data(), se.size() * 4);
    fix.push_back({m, {a, s}});
  }
};

bool add_matrix(const Mat& m, const std::vector<int>& order, int left, bool common, EmuMat* out,
                Upload* up) {
  std::vector<uint16_t> b;
  std::vector<int> se;
  if (!build_operand(m, order, left, common, out, &b, &se)) return false;
  up->add(out, b, se);
  return true;
}

}  // namespace

EmuPlan* emu_create(const ts_grid_desc& g, cudaError_t* err) {
  *err = cudaSuccess;
  const int Nr = g.Nr, Nt = g.Ntheta, Np = g.Nphi, NT = g.NTheta, NP = g.NPhi;
  const bool cons = g.form == TS_FORM_CONSERVATIVE;
  const Wide odd = cons ? -1.0L : 1.0L;
  auto sine = [](int m, int n) {   // sin(2 pi m / n), exactly zero at 0 and pi
    return 2 * m % n ? sinl(2.0L * kPi * m / n) : 0.0L;
  };
  EmuPlan* e = new EmuPlan();
  Upload up;
  {
    // angular: Theta' = sinTh (A u + B partner) [conservative: + cosTh P u],
    // Phi' = sinPh D u [conservative: D (sinPh u)]; the sign and 1/r, and sinTh cot th
    // of the Phi term, are the epilogue's. A, B: the halves of the doubled circle
    // (B times -1 for the odd continuation of the conservative form)
    const std::vector<Wide> DT = fourier_wide(2 * NT), DP = fourier_wide(NP);
    Mat mD(NT, std::vector<Wide>(2 * NT)), mF(NP + 5, std::vector<Wide>(NP));
    for (int k = 0; k < NT; ++k) {
      const Wide Th = kPi * (k + 0.5L) / NT, st = sinl(Th), ct = cosl(Th);
      for (int q = 0; q < NT; ++q) {
        mD[k][q] = st * DT[(size_t)k * 2 * NT + q];
        mD[k][NT + q] = odd * st * DT[(size_t)k * 2 * NT + 2 * NT - 1 - q];
        if (cons) {   // P: the Nyquist bin of the doubled circle taken out
          const Wide alt = ((k + q) % 2 ? -1.0L : 1.0L) / (2.0L * NT);
          mD[k][q] += ct * ((k == q ? 1.0L : 0.0L) - alt);
          mD[k][NT + q] -= ct * alt;
        }
      }
    }
    std::vector<Wide> sP(NP);
    for (int m = 0; m < NP; ++m) sP[m] = sine(m, NP);
    for (int q = 0; q < NP; ++q) {
      const Wide c = cosl(2.0L * kPi * q / NP), s = sP[q];
      for (int m = 0; m < NP; ++m) mF[m][q] = (cons ? s : sP[m]) * DP[(size_t)m * NP + q];
      mF[NP][q] = 1.0L;
      mF[NP + 1][q] = c;
      mF[NP + 2][q] = s;
      mF[NP + 3][q] = c * c;
      mF[NP + 4][q] = c * s;
    }
    e->ang = add_matrix(mD, dfs_order(NT), -1, true, &e->angD, &up);
    for (int f = 0; f < kEmuForms && e->ang; ++f) {
      // sinPh vanishes at Phi = 0 and pi: the first functionals take those rows of the
      // advective form, the others follow behind the derivatives
      const int nf = emu_functionals(f), nz = cons ? 0 : std::min(nf, 2);
      Mat part(mF.begin(), mF.begin() + NP);
      for (int q = 0; q < nf; ++q) {
        if (q < nz) part[q * (NP / 2)] = mF[NP + q];
        else part.push_back(mF[NP + q]);
      }
      e->ang = add_matrix(part, plain_order(NP, (NP + 15) / 16 * 2), -1, true, &e->angF[f], &up) &&
               geometry2(NT, NP, e->angD, e->angF[f], nf, nz, false, &e->gAng[f]);
    }
  }
  const bool adj = !cons && g.radial == TS_RADIAL_CHEBYSHEV;   // the forms that have an adjoint
  if (adj) {
    // the transposed angular operator: D_Th^T (sinTh lt), D_Ph^T (sinPh lt)
    const std::vector<Wide> DT = fourier_wide(2 * NT), DP = fourier_wide(NP);
    Mat mD(NT, std::vector<Wide>(2 * NT)), mF(NP + 5, std::vector<Wide>(NP));
    for (int k = 0; k < NT; ++k) {
      const Wide st = sinl(kPi * (k + 0.5L) / NT);
      for (int q = 0; q < NT; ++q) {
        mD[q][k] = st * DT[(size_t)k * 2 * NT + q];
        mD[q][NT + k] = st * DT[(size_t)k * 2 * NT + 2 * NT - 1 - q];
      }
    }
    for (int m = 0; m < NP; ++m) {
      const Wide c = cosl(2.0L * kPi * m / NP), s = sine(m, NP);
      for (int q = 0; q < NP; ++q) mF[q][m] = s * DP[(size_t)m * NP + q];
      mF[NP][m] = 1.0L;
      mF[NP + 1][m] = c;
      mF[NP + 2][m] = s;
      mF[NP + 3][m] = c * c;
      mF[NP + 4][m] = c * s;
    }
    e->adj = add_matrix(mD, dfs_order(NT), -1, true, &e->adjD, &up);
    for (int f = 0; f < kEmuForms && e->adj; ++f) {
      const int nf = emu_functionals(f);
      Mat part(mF.begin(), mF.begin() + NP + nf);
      e->adj = add_matrix(part, plain_order(NP, (NP + 15) / 16 * 2), -1, true, &e->adjF[f], &up) &&
               geometry2(NT, NP, e->adjD, e->adjF[f], nf, 0, true, &e->gAdj[f]);
    }
  }
  {
    const std::vector<Wide> Dt = fourier_wide(2 * Nt), Dp = fourier_wide(Np);
    Mat mD(Nt, std::vector<Wide>(2 * Nt)), mF(Np, std::vector<Wide>(Np));
    for (int j = 0; j < Nt; ++j)
      for (int q = 0; q < Nt; ++q) {
        mD[j][q] = Dt[(size_t)j * 2 * Nt + q];
        mD[j][Nt + q] = odd * Dt[(size_t)j * 2 * Nt + 2 * Nt - 1 - q];
      }
    for (int l = 0; l < Np; ++l)
      for (int q = 0; q < Np; ++q) mF[l][q] = Dp[(size_t)l * Np + q];
    e->plane = add_matrix(mD, dfs_order(Nt), -1, true, &e->plD, &up) &&
               add_matrix(mF, plain_order(Np, (Np + 15) / 16 * 2), -1, true, &e->plF, &up) &&
               geometry2(Nt, Np, e->plD, e->plF, 0, 0, false, &e->gPl);
    if (adj && e->plane) {
      // transposed: a_th changes sign at the partner (cos(Ph + pi) = -cosPh), so it comes
      // out of the contraction with the partner's matrix negated
      Mat tD(Nt, std::vector<Wide>(2 * Nt)), tF(Np, std::vector<Wide>(Np));
      for (int j = 0; j < Nt; ++j)
        for (int q = 0; q < Nt; ++q) {
          tD[q][j] = mD[j][q];
          tD[q][Nt + j] = -mD[j][Nt + q];
        }
      for (int l = 0; l < Np; ++l)
        for (int q = 0; q < Np; ++q) tF[q][l] = mF[l][q];
      e->planeT = add_matrix(tD, dfs_order(Nt), -1, true, &e->plTD, &up) &&
                  add_matrix(tF, plain_order(Np, (Np + 15) / 16 * 2), -1, true, &e->plTF, &up);
    }
  }
  if (g.radial == TS_RADIAL_CHEBYSHEV && geometry_radial(Nr, &e->gRad)) {
    const EmuRadGeo& r = e->gRad;
    const std::vector<Wide> Dr = cheb_wide(Nr, g.R1, g.R2);
    e->rad = true;
    e->radT = adj;
    for (int tr = 0; tr < 2; ++tr) {
      bool& ok = tr ? e->radT : e->rad;
      for (int q = 0; q < r.ng && ok; ++q) {
        EmuMat* out = tr ? &e->radTM[q] : &e->radM[q];
        Mat m;
        for (int o = q * r.go; o < std::min(Nr, (q + 1) * r.go); ++o) {
          const int i = o == 0 ? 0 : o == 1 ? Nr - 1 : o - 1;
          std::vector<Wide> row(Nr);
          for (int z = 0; z < Nr; ++z) row[z] = tr ? Dr[(size_t)z * Nr + i] : Dr[(size_t)i * Nr + z];
          m.push_back(row);
        }
        while ((int)m.size() < r.go) m.push_back(std::vector<Wide>(Nr));   // equal groups
        ok = add_matrix(m, plain_order(r.left ? Nr - 1 : Nr, r.kc), r.left ? Nr - 1 : -1, false, out,
                        &up);
      }
    }
  }
  if (!e->ang && !e->plane && !e->rad) {
    delete e;
    return nullptr;
  }
  cudaError_t r = cudaMalloc(&e->mem, up.host.size());
  if (r == cudaSuccess)
    r = cudaMemcpy(e->mem, up.host.data(), up.host.size(), cudaMemcpyHostToDevice);
  if (r != cudaSuccess) {
    *err = r;
    emu_destroy(e);
    return nullptr;
  }
  for (auto& f : up.fix) {
    f.first->dev = reinterpret_cast<const uint16_t*>(static_cast<char*>(e->mem) + f.second.first);
    f.first->se = reinterpret_cast<const int*>(static_cast<char*>(e->mem) + f.second.second);
  }
  return e;
}

void emu_destroy(EmuPlan* e) {
  if (!e) return;
  if (e->mem) cudaFree(e->mem);
  delete e;
}

namespace {

// CTAs of a persistent launch: two per SM with 256 threads (the geometry keeps their
// shared and tensor memory to half an SM's, the launch bounds their registers), else one.
cudaError_t emu_ctas(int threads, long long ntiles, int* ctas) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  *ctas = (int)std::max<long long>(1, std::min<long long>(ntiles, (threads == 256 ? 2LL : 1LL) * nsm));
  return e;
}

template <int PASS, int KF, int T, int NA, int NB, int XW = 8>
cudaError_t launch2(const Problem& p, const Tables<double>& t, const EmuGeo& g, const EmuMat& D,
                    const EmuMat& F, emu::EmuArgs A, cudaStream_t s) {
  static const cudaError_t e = allow_smem(emu::k_emu2<PASS, KF, T, NA, NB, XW>);   // once per kernel
  if (e != cudaSuccess) return e;
  int ctas = 1;
  const cudaError_t e2 = emu_ctas(T, A.ntiles, &ctas);
  if (e2 != cudaSuccess) return e2;
  return launch_pass(emu::k_emu2<PASS, KF, T, NA, NB, XW>, ctas, T, g.bytes, s, p, t, g,
                     emu::MatArg{D.dev, 3 - D.s}, emu::MatArg{F.dev, 3 - F.s}, A);
}
template <int PASS, int KF>
cudaError_t launch2t(const Problem& p, const Tables<double>& t, const EmuGeo& g, const EmuMat& D,
                     const EmuMat& F, emu::EmuArgs A, cudaStream_t s) {
  const int h = g.xw / 2;
  const uintptr_t at = reinterpret_cast<uintptr_t>(A.U);
  if (PASS == emu::EP_PLANE) {   // h columns of a half circle in one load
    A.ntiles = (long long)p.d.G * p.d.Nr * p.d.NT * ((p.d.NP / 2 + h - 1) / h);
    A.vec = p.d.NP % (2 * h) == 0 && at % (8 * h) == 0;
  } else {                       // xw = 4: two points of a row (rows are of even length)
    A.ntiles = (p.d.nblk + g.xw - 1) / g.xw;
    A.vec = at % 16 == 0;
  }
  // 16 x 16 has a form of its own, as the other passes have for common sizes: the index
  // arithmetic folds away (33 x 16^4 x 4: 1509 us a step, 1585 without; conservative 1855,
  // 2030). At 32 x 32 one gives 0.3 %
  if (g.threads == 256 && g.Na == 16 && g.Nb == 16)
    return launch2<PASS, KF, 256, 16, 16>(p, t, g, D, F, A, s);
  if (g.xw == 4) return launch2<PASS, KF, 512, 0, 0, 4>(p, t, g, D, F, A, s);
  return g.threads == 256 ? launch2<PASS, KF, 256, 0, 0>(p, t, g, D, F, A, s)
                          : launch2<PASS, KF, 512, 0, 0>(p, t, g, D, F, A, s);
}

}  // namespace

cudaError_t emu_angular(const EmuPlan& e, const Problem& p, const Tables<double>& t, bool cons,
                        const double* U, double* K, double sgn, bool collision, cudaStream_t s) {
  const int kf = kernel_form(p, collision ? 1 : 0);
  emu::EmuArgs A{};
  A.U = U;
  A.K = K;
  A.sgn = sgn;
  A.collision = collision ? 1 : 0;
  A.cons = cons ? 1 : 0;
  switch (kf) {
    case KF_QUADRATIC:
      return launch2t<emu::EP_ANGULAR, KF_QUADRATIC>(p, t, e.gAng[kf], e.angD, e.angF[kf], A, s);
    case KF_LINEAR:
      return launch2t<emu::EP_ANGULAR, KF_LINEAR>(p, t, e.gAng[kf], e.angD, e.angF[kf], A, s);
    default:
      return launch2t<emu::EP_ANGULAR, KF_ISO>(p, t, e.gAng[kf], e.angD, e.angF[kf], A, s);
  }
}

namespace {
cudaError_t plane_launch(const Problem& p, const Tables<double>& t, const EmuGeo& g,
                         const EmuMat& D, const EmuMat& F, const double* U, double* K, double sgn,
                         cudaStream_t s) {
  emu::EmuArgs A{};
  A.U = U;
  A.K = K;
  A.sgn = sgn;
  return launch2t<emu::EP_PLANE, KF_ISO>(p, t, g, D, F, A, s);
}
}  // namespace

cudaError_t emu_plane(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                      const double* U, double* K, double sgn, cudaStream_t s) {
  return plane_launch(p, t, e.gPl, e.plD, e.plF, U, K, sgn, s);
}

cudaError_t emu_angular_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                          const double* lt, const double* Ubar, const double* Us, double* gk,
                          double* ge, const double* lam, const double* lam_in, double* lam_out,
                          double* Kbar, double wl, double wu, cudaStream_t s) {
  const int kf = kernel_form(p, 1);
  emu::EmuArgs A{};
  A.U = lt;
  A.K = const_cast<double*>(Ubar);   // only read
  A.sgn = -1.0;
  A.collision = 1;
  A.Us = Us;
  A.gk = gk;
  A.ge = ge;
  A.lam = lam;
  A.lam_in = lam_in;
  A.lam_out = lam_out;
  A.Kbar = Kbar;
  A.wl = wl;
  A.wu = wu;
  switch (kf) {
    case KF_QUADRATIC:
      return launch2t<emu::EP_ADJOINT, KF_QUADRATIC>(p, t, e.gAdj[kf], e.adjD, e.adjF[kf], A, s);
    case KF_LINEAR:
      return launch2t<emu::EP_ADJOINT, KF_LINEAR>(p, t, e.gAdj[kf], e.adjD, e.adjF[kf], A, s);
    default:
      return launch2t<emu::EP_ADJOINT, KF_ISO>(p, t, e.gAdj[kf], e.adjD, e.adjF[kf], A, s);
  }
}

cudaError_t emu_plane_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                        const double* lt, double* Ubar, cudaStream_t s) {
  return plane_launch(p, t, e.gPl, e.plTD, e.plTF, lt, Ubar, -1.0, s);
}

namespace {
template <int T, int MODE>
cudaError_t launch_rad(const EmuRadGeo& g, const EmuMat* mats, const Problem& p,
                       const Tables<double>& t, emu::RadArgs A, cudaStream_t s) {
  static const cudaError_t ea = allow_smem(emu::k_emu_radial<T, MODE>);   // once per kernel
  if (ea != cudaSuccess) return ea;
  int ctas = 1;
  const cudaError_t e2 = emu_ctas(T, A.ntiles, &ctas);
  if (e2 != cudaSuccess) return e2;
  emu::RadMats M{};
  for (int q = 0; q < g.ng; ++q) {
    M.dev[q] = mats[q].dev;
    M.se[q] = mats[q].se;
  }
  return launch_pass(emu::k_emu_radial<T, MODE>, ctas, T, g.bytes, s, p, t, g, M, A);
}
template <int T>
cudaError_t launch_rad_mode(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                            emu::RadArgs A, cudaStream_t s) {
  switch (A.mode) {
    case RAD_RHS: return launch_rad<T, RAD_RHS>(e.gRad, e.radM, p, t, A, s);
    case RAD_STAGE0: return launch_rad<T, RAD_STAGE0>(e.gRad, e.radM, p, t, A, s);
    case RAD_STAGE1:
    case RAD_STAGE2: return launch_rad<T, RAD_STAGE1>(e.gRad, e.radM, p, t, A, s);
    case RAD_STAGE3: return launch_rad<T, RAD_STAGE3>(e.gRad, e.radM, p, t, A, s);
    case RAD_AB2: return launch_rad<T, RAD_AB2>(e.gRad, e.radM, p, t, A, s);
    default: return launch_rad<T, RAD_AB2_START>(e.gRad, e.radM, p, t, A, s);
  }
}
}  // namespace

cudaError_t emu_radial(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                       const double* U, const double* K, double sgn, bool tau, int mode, double* F,
                       double* Acc, double* Uout, double* out, double dt, cudaStream_t s) {
  emu::RadArgs A{U, K, sgn, tau ? 1 : 0, mode, F, Acc, Uout, out, dt,
                 (long long)p.d.G * p.d.Nt * p.d.Np * ((p.d.NT * p.d.NP + 127) / 128)};
  return e.gRad.threads == 256 ? launch_rad_mode<256>(e, p, t, A, s)
                               : launch_rad_mode<512>(e, p, t, A, s);
}

cudaError_t emu_radial_T(const EmuPlan& e, const Problem& p, const Tables<double>& t,
                         const double* X, double scale, bool tau, double* lt, double* Ubar,
                         cudaStream_t s) {
  emu::RadArgs A{X, nullptr, 1.0, tau ? 1 : 0, emu::RAD_ADJOINT, nullptr, lt, nullptr, Ubar, scale,
                 (long long)p.d.G * p.d.Nt * p.d.Np * ((p.d.NT * p.d.NP + 127) / 128)};
  return e.gRad.threads == 256
             ? launch_rad<256, emu::RAD_ADJOINT>(e.gRad, e.radTM, p, t, A, s)
             : launch_rad<512, emu::RAD_ADJOINT>(e.gRad, e.radTM, p, t, A, s);
}

}  // namespace ts
