// Host program of test_fx_host.py: the arithmetic of su3_fx.cuh (the same
// functions as on the device) against long double, on Haar-like SU(3) matrices,
// on matrices with exact zeros and ones, and next to plain FP64 arithmetic.
// Prints the largest errors, in units of 2^-53.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "su3_fx.cuh"
#include "su3_fx_kp.cuh"

using namespace su3dev;
typedef long double Q;
struct cq {
  Q re, im;
};
struct M {
  double e[3][3][2];
};

static std::mt19937_64 rng(1);

static cq mulq(cq a, cq b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
static cq get(const M& m, int i, int k) { return {m.e[i][k][0], m.e[i][k][1]}; }
static cq cj(cq a) { return {a.re, -a.im}; }

static M su3(int kind) {
  std::normal_distribution<double> nd;
  M m{};
  if (kind == 1) {  // a permutation of the identity with signs: entries exactly 0, 1, -1
    const int p = (int)(rng() % 3);
    const double s = rng() & 1 ? 1.0 : -1.0;
    m.e[0][p][0] = s;
    m.e[1][(p + 1) % 3][0] = s;
    m.e[2][(p + 2) % 3][0] = 1.0;
    return m;
  }
  Q r[2][6];
  for (auto& row : r)
    for (Q& x : row) x = nd(rng) * (kind == 2 ? 1e-9 : 1.0);
  if (kind == 2) r[0][0] = r[1][2] = 1.0;  // close to the identity
  Q n = 0, d[2] = {0, 0};
  for (Q x : r[0]) n += x * x;
  for (Q& x : r[0]) x /= std::sqrt(n);
  for (int k = 0; k < 3; ++k) {
    d[0] += r[0][2 * k] * r[1][2 * k] + r[0][2 * k + 1] * r[1][2 * k + 1];
    d[1] += r[0][2 * k] * r[1][2 * k + 1] - r[0][2 * k + 1] * r[1][2 * k];
  }
  for (int k = 0; k < 3; ++k) {
    const Q a = r[0][2 * k], b = r[0][2 * k + 1];
    r[1][2 * k] -= d[0] * a - d[1] * b;
    r[1][2 * k + 1] -= d[0] * b + d[1] * a;
  }
  n = 0;
  for (Q x : r[1]) n += x * x;
  for (Q& x : r[1]) x /= std::sqrt(n);
  for (int i = 0; i < 2; ++i)
    for (int k = 0; k < 6; ++k) m.e[i][k / 2][k % 2] = (double)r[i][k];
  for (int k = 0; k < 3; ++k) {
    const int a = (k + 1) % 3, b = (k + 2) % 3;
    const cq x = mulq(get(m, 0, a), get(m, 1, b)), y = mulq(get(m, 0, b), get(m, 1, a));
    m.e[2][k][0] = (double)(x.re - y.re);
    m.e[2][k][1] = -(double)(x.im - y.im);
  }
  return m;
}

static cfx dec(const M& m, int i, int k) { return {fx_from_double(m.e[i][k][0]), fx_from_double(m.e[i][k][1])}; }
static Q val(const fx& a, int unit) { return std::ldexp((Q)a.h, unit) + std::ldexp((Q)a.l, unit - 32); }

// Errors of the fixed-point functions and of their FP64 form (root mean square
// and largest), in units of 2^-53.
struct Err {
  Q most = 0, sum = 0;
  long n = 0;
  void add(Q e) {
    e = std::fabs(e) * std::ldexp((Q)1, 53);
    most = std::fmax(most, e);
    sum += e * e;
    ++n;
  }
  Q rms() const { return std::sqrt(sum / n); }
};

static void heatbath_scalars() {
  const Q pi = std::acos((Q)-1);
  std::normal_distribution<double> nd;
  Err lg, trig, root, dir, dir64, a0, a0_64, ax, ax64, rot;
  long other = 0;
  for (int it = 0; it < 200000; ++it) {
    // uniforms over the whole range, and near 0, 1/2 and 1
    unsigned long long m = rng() >> 11;
    const int cut = (int)(rng() % 52);
    if (it % 5 == 1) m >>= cut;
    if (it % 5 == 2) m = (1ull << 53) - 1 - (m >> cut);
    if (it % 5 == 3) m = (1ull << 52) + (m >> (cut / 2 + 26));
    m |= 1;
    if (it == 0) m = 1;
    if (it == 2) m = (1ull << 53) - 1;
    const Q x = std::ldexp((Q)m, -53);
    lg.add(std::ldexp((Q)fx_neg_log(m), -57) + std::log(x));
    const fx_cs cs = fx_cossin(m);
    trig.add(val(cs.c, -30) - std::cos(2 * pi * x));
    trig.add(val(cs.s, -30) - std::sin(2 * pi * x));
    root.add(val(fx_two_root((long long)(m << 9)), -30) - 2 * std::sqrt(x * (1 - x)));

    long long r[4];
    const int scale = it % 3 == 0 ? 59 : 20 + (int)(rng() % 40);
    for (long long& c : r) c = (long long)std::ldexp(nd(rng), scale);
    if (it % 7 == 0) r[1] = r[2] = r[3] = 0;
    if (it % 11 == 0) r[1] = -r[0];
    Q k = 0;
    double kd = 0;
    for (long long c : r) {
      k += (Q)c * c;
      kd = std::fma((double)c, (double)c, kd);
    }
    if (k == 0) continue;
    k = std::sqrt(k);
    fx v[4], a[4];
    double ik;
    if (!fx_direction(r, v, &ik)) {
      std::printf("a direction was refused\n");
      std::exit(1);
    }
    for (int c = 0; c < 4; ++c) {
      dir.add(val(v[c], -30) - r[c] / k);
      dir64.add((Q)((double)r[c] * (1.0 / std::sqrt(kd))) - r[c] / k);
    }
    unsigned long long w[6];
    for (unsigned long long& y : w) y = (rng() >> 11) | 1;
    const double ia = std::pow(10.0, -2.5 + 3.0 * (double)(rng() % 1000) / 1000.0);
    Q U[6];
    double D[6];
    for (int c = 0; c < 6; ++c) U[c] = D[c] = std::ldexp((double)w[c], -53);
    const Q cq1 = std::cos(2 * pi * U[1]), delta = -(std::log(U[0]) + cq1 * cq1 * std::log(U[2])) * ia;
    const bool take = U[3] * U[3] <= 1 - delta / 2, took = fx_propose(fx_draw(w), ia, a);
    other += take != took;
    if (!take || !took) continue;
    const double cd = (double)cq1, dd = -std::fma(cd * cd, std::log(D[2]), std::log(D[0])) * ia;
    const Q rho = std::sqrt(1 - (1 - delta) * (1 - delta)), ct = 1 - 2 * U[4], sn = std::sqrt(1 - ct * ct);
    const double rhod = std::sqrt(std::fma(-(1 - dd), 1 - dd, 1.0)), ctd = 1 - 2 * D[4];
    const double snd = std::sqrt(std::fma(-ctd, ctd, 1.0));
    const Q e[4] = {1 - delta, rho * sn * std::cos(2 * pi * U[5]), rho * sn * std::sin(2 * pi * U[5]), rho * ct};
    const double f[4] = {1 - dd, rhod * snd * (double)std::cos(2 * pi * U[5]),
                         rhod * snd * (double)std::sin(2 * pi * U[5]), rhod * ctd};
    for (int c = 0; c < 4; ++c) {
      (c ? ax : a0).add(val(a[c], -30) - e[c]);
      (c ? ax64 : a0_64).add((Q)f[c] - e[c]);
    }
    cfx R0, R1;
    fx_rotation(a, v, R0, R1);
    Q n = -1;
    for (const fx& y : {R0.re, R0.im, R1.re, R1.im}) n += val(y, -30) * val(y, -30);
    rot.add(n);
  }
  std::printf("log %.3Lf trig %.3Lf root %.3Lf dir %.3Lf dir_fp %.3Lf azero %.3Lf azero_fp %.3Lf avec %.3Lf avec_fp %.3Lf "
              "unit %.3Lf flips %ld\n", lg.most, trig.most, root.most, dir.rms(), dir64.rms(), a0.rms(), a0_64.rms(), ax.rms(),
              ax64.rms(), rot.most, other);
}

int main() {
  heatbath_scalars();
  const Q u = std::ldexp((Q)1, -53);
  Q decode = 0, staple = 0, plain = 0, reunit = 0, round_trip = 0;
  for (int it = 0; it < 200000; ++it) {
    std::uniform_real_distribution<double> ud(-1, 1);
    const double special[8] = {0.0, -0.0, 1.0, -1.0, 0.5, -0.25, 1.0 - 0x1p-53, 0x1p-1060};
    const double d = it < 8 ? special[it] : std::ldexp(ud(rng), -(int)(rng() % 80));
    decode = std::fmax(decode, std::fabs(val(fx_from_double(d), -30) - d) / u);
    decode = std::fmax(decode, std::fabs(val(fx_from_double(d, 0x80000000u), -30) + d) / u);
    round_trip = std::fmax(round_trip, std::fabs((Q)fx_to_double(fx_from_double(d)) - d) / u);
  }
  for (int it = 0; it < 3000; ++it) {
    // six paths X Y^+ Z, summed, row 2 completed
    cq ref[3][3] = {};
    double f64[3][3][2] = {};
    fx_staple A;
    fx_staple_zero(A);
    const int kind = it % 4 == 3 ? 1 : (it % 4 == 2 ? 2 : 0);
    for (int path = 0; path < 6; ++path) {
      const M X = su3(kind), Y = su3(kind), Z = su3(kind);
      cq t[3][3], F[2][3];
      double td[2][3][2], Fd[2][3][2];
      fx_rows01 f;
      cfx tx[2][3];
      for (int i = 0; i < 2; ++i)
        for (int k = 0; k < 3; ++k) {
          t[i][k] = {0, 0};
          double re = 0, im = 0;
          cfacc s = cfx_zero();
          for (int j = 0; j < 3; ++j) {
            const cq p = mulq(get(X, i, j), cj(get(Y, k, j)));
            t[i][k] = {t[i][k].re + p.re, t[i][k].im + p.im};
            const double *a = X.e[i][j], *b = Y.e[k][j];
            re = std::fma(a[1], b[1], std::fma(a[0], b[0], re));
            im = std::fma(a[1], b[0], std::fma(-a[0], b[1], im));
            cfx_mac_cb(s, dec(X, i, j), dec(Y, k, j));
          }
          td[i][k][0] = re;
          td[i][k][1] = im;
          tx[i][k] = cfx_norm(s);
        }
      for (int i = 0; i < 2; ++i)
        for (int k = 0; k < 3; ++k) {
          F[i][k] = {0, 0};
          double re = 0, im = 0;
          cfacc s = cfx_zero();
          for (int j = 0; j < 3; ++j) {
            const cq p = mulq(t[i][j], get(Z, j, k));
            F[i][k] = {F[i][k].re + p.re, F[i][k].im + p.im};
            const double *a = td[i][j], *b = Z.e[j][k];
            re = std::fma(-a[1], b[1], std::fma(a[0], b[0], re));
            im = std::fma(a[1], b[0], std::fma(a[0], b[1], im));
            cfx_mac(s, tx[i][j], dec(Z, j, k));
          }
          Fd[i][k][0] = re;
          Fd[i][k][1] = im;
          const long long mr = fx_merge(s.re), mi = fx_merge(s.im);
          f.e[i][k] = cfx{fx_norm_merged(mr), fx_norm_merged(mi)};
          A.r[i][k][0] += mr;
          A.r[i][k][1] += mi;
          ref[i][k] = {ref[i][k].re + F[i][k].re, ref[i][k].im + F[i][k].im};
          f64[i][k][0] += re;
          f64[i][k][1] += im;
        }
      for (int k = 0; k < 3; ++k) {
        const int a = (k + 1) % 3, b = (k + 2) % 3;
        const cq x = mulq(F[0][a], F[1][b]), y = mulq(F[0][b], F[1][a]);
        ref[2][k] = {ref[2][k].re + x.re - y.re, ref[2][k].im - (x.im - y.im)};
        const double *p = Fd[0][a], *q = Fd[1][b], *v = Fd[0][b], *w = Fd[1][a];
        f64[2][k][0] += std::fma(p[0], q[0], std::fma(-p[1], q[1], std::fma(-v[0], w[0], v[1] * w[1])));
        f64[2][k][1] -= std::fma(p[0], q[1], std::fma(p[1], q[0], std::fma(-v[0], w[1], -v[1] * w[0])));
      }
      fx_staple_add_row2(A, f);
    }
    const fx_mat m = fx_staple_mat(A, 6);
    for (int i = 0; i < 3; ++i)
      for (int k = 0; k < 3; ++k) {
        staple = std::fmax(staple, std::fabs(val(m.e[i][k].re, -28) - ref[i][k].re) / u);
        staple = std::fmax(staple, std::fabs(val(m.e[i][k].im, -28) - ref[i][k].im) / u);
        plain = std::fmax(plain, std::fabs(f64[i][k][0] - ref[i][k].re) / u);
        plain = std::fmax(plain, std::fabs(f64[i][k][1] - ref[i][k].im) / u);
      }
    // reunitarisation of a matrix 2^-34 to 2^-53 away from SU(3)
    M Y = su3(kind);
    const double away = std::ldexp(1.0, -36 - it % 18);
    std::normal_distribution<double> nd;
    fx_mat x{};
    Q r[2][6];
    for (int i = 0; i < 2; ++i)
      for (int k = 0; k < 3; ++k) {
        for (int c = 0; c < 2; ++c) r[i][2 * k + c] = Y.e[i][k][c] += away * nd(rng);
        x.e[i][k] = dec(Y, i, k);
      }
    if (!fx_reunitarise(x)) {
      std::printf("a link %g away from SU(3) was refused\n", away);
      return 1;
    }
    Q n = 0, d[2] = {0, 0};
    for (Q y : r[0]) n += y * y;
    for (Q& y : r[0]) y /= std::sqrt(n);
    for (int k = 0; k < 3; ++k) {
      d[0] += r[0][2 * k] * r[1][2 * k] + r[0][2 * k + 1] * r[1][2 * k + 1];
      d[1] += r[0][2 * k] * r[1][2 * k + 1] - r[0][2 * k + 1] * r[1][2 * k];
    }
    for (int k = 0; k < 3; ++k) {
      const Q a = r[0][2 * k], b = r[0][2 * k + 1];
      r[1][2 * k] -= d[0] * a - d[1] * b;
      r[1][2 * k + 1] -= d[0] * b + d[1] * a;
    }
    n = 0;
    for (Q y : r[1]) n += y * y;
    for (Q& y : r[1]) y /= std::sqrt(n);
    for (int i = 0; i < 2; ++i)
      for (int k = 0; k < 3; ++k) {
        reunit = std::fmax(reunit, std::fabs(val(x.e[i][k].re, -30) - r[i][2 * k]) / u);
        reunit = std::fmax(reunit, std::fabs(val(x.e[i][k].im, -30) - r[i][2 * k + 1]) / u);
      }
    // and refused where first order does not do
    for (int k = 0; k < 3; ++k) {
      Y.e[0][k][0] *= 1.0 + 1e-7;
      Y.e[0][k][1] *= 1.0 + 1e-7;
      x.e[0][k] = dec(Y, 0, k);
    }
    if (fx_reunitarise(x)) {
      std::printf("a link 1e-7 away from SU(3) was accepted\n");
      return 1;
    }
  }
  std::printf("decode %.3Lf round_trip %.3Lf staple %.3Lf plain %.3Lf reunitarise %.3Lf\n", decode, round_trip, staple, plain, reunit);
  return 0;
}
