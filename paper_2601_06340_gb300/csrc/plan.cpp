// Host-side plan math in FP64 (compiled with -ffp-contract=off so that the
// operation order written here is the one executed).
//
// Per photon energy (Krzywinski & Halavanau, arXiv 2601.06340, Sec. 2):
//   lambda = hc / E, k = 2 pi / lambda, s = sin(theta_B(E)) = lambda / 2d
//   (the band centres +-k_d/2 in units of k, Eq. fov7), cos(alpha) =
//   sqrt(1 - s^2) (Eq. fov4), dz^ = k dz, dx^ = k dx (Eq. fov2), and the
//   Jacobi-Anger coefficients of Eqs. fov11-fov12 read with dz^:
//   a = J0(w) e^{i phi0}, b = i J1(w) e^{i phi0}, w = dz^ chi_h / cos(alpha),
//   phi0 = dz^ chi_0 / (2 cos(alpha)).
// Per band, the propagator exp(i dz^ sqrt(1 - (q +- s)^2)) of Eq. fov10 is
// split into the common phase g = exp(i dz^ cos(alpha)) and the mode part
// exp(i dz^ delta_+-(q)), delta_+-(q) = -q (q +- 2 s) /
// (sqrt(1 - (q +- s)^2) + cos(alpha)), which is the same quantity without
// the cancellation of sqrt(...) - cos(alpha).
#include <cmath>
#include <complex>
#include <string>
#include <vector>

#include "bpm_internal.h"

namespace bpm {

namespace {

using cd = std::complex<double>;

bool finite(double v) { return std::isfinite(v); }

// J_nu(w) by its power series sum_m (-1)^m (w/2)^(2m+nu) / (m! (m+nu)!).
// skip_first drops the m = 0 term (J0(w) - 1 without cancellation).
cd bessel(int nu, cd w, bool skip_first) {
  cd half = w / 2.0;
  cd term = (nu == 0) ? cd(1.0, 0.0) : half;
  double scale = std::max(std::abs(term), 1e-300);
  cd total = skip_first ? cd(0.0, 0.0) : term;
  for (int m = 1; m <= 200; ++m) {
    term = term * (-(half * half)) / double(m * (m + nu));
    total += term;
    if (std::abs(term) < 1e-18 * scale) break;
  }
  return total;
}

// exp(i z) - 1 for complex z without cancellation.
cd expm1_i(cd z) {
  double x = z.real(), y = z.imag();          // i z = -y + i x
  double ey = std::exp(-y), em = std::expm1(-y);
  double sh = std::sin(0.5 * x);
  double cosm1 = -2.0 * sh * sh;               // cos x - 1
  return cd(em * std::cos(x) + cosm1, ey * std::sin(x));
}

// exp(i x) - 1 for real x without cancellation (the same value as above, with
// the terms that are exactly 0 or 1 left out).
cd expm1_i(double x) {
  const double sh = std::sin(0.5 * x);
  return cd(-2.0 * sh * sh, std::sin(x));
}

double fftfreq_q(int k, int n, double dxh) {
  int kk = (k < n / 2) ? k : k - n;
  return kTwoPi * (double(kk) * (1.0 / (double(n) * dxh)));
}

// delta_+-(q) in the cancellation-free form (sign = +1 for psi_+).
double delta_q(double q, double s, double c, int sign) {
  double t = q + sign * s;
  double root = std::sqrt(1.0 - t * t);
  return -q * (q + sign * 2.0 * s) / (root + c);
}

}  // namespace

static void unit_root(int m, int n, double* cr, double* ci);

int validate_problem(const bpm_problem* p, std::string* why) {
  auto bad = [&](const std::string& m) { *why = m; return BPM_ERR_INVALID; };
  if (!p) return bad("problem is NULL");
  if (p->nx < 8 || p->nx > (1 << kMaxLogN) || (p->nx & (p->nx - 1)))
    return bad("nx must be a power of two in [8, " +
               std::to_string(1 << kMaxLogN) + "]");
  if (p->nz < 1) return bad("nz must be >= 1");
  if (!(p->dx_um > 0) || !finite(p->dx_um)) return bad("dx_um must be > 0");
  if (!(p->dz_um > 0) || !finite(p->dz_um)) return bad("dz_um must be > 0");
  if (!finite(p->x0_um)) return bad("x0_um must be finite");
  if (p->n_energy < 1 || !p->energy_ev) return bad("need n_energy >= 1 energies");
  if (p->n_energy > (1 << 20)) return bad("n_energy too large");
  if (!(p->e_ref_ev > 0) || !finite(p->e_ref_ev)) return bad("e_ref_ev must be > 0");
  if (!(p->theta_b_ref_rad > 0) || !(p->theta_b_ref_rad < 1.5707963267948966))
    return bad("theta_b_ref_rad must be in (0, pi/2)");
  if (!finite(p->chi0_re) || !finite(p->chi0_im) || !finite(p->chih_re) ||
      !finite(p->chih_im))
    return bad("chi values must be finite");
  if (p->record_every < 0) return bad("record_every must be >= 0");
  if (p->precision != BPM_FP64_PLAIN && p->precision != BPM_FP32_FUSED)
    return bad("precision must be BPM_FP64_PLAIN or BPM_FP32_FUSED");
  for (int j = 0; j < p->n_energy; ++j) {
    double e = p->energy_ev[j];
    if (!(e > 0) || !finite(e)) return bad("energies must be > 0");
    double s = std::sin(p->theta_b_ref_rad) * (p->e_ref_ev / e);
    if (!(s < 1.0)) return bad("no Bragg angle at energy " + std::to_string(e));
    double lam = kHcEvAngstrom / e * 1e-4;
    double k = kTwoPi / lam;
    double qmax = M_PI / (k * p->dx_um);
    if (!((qmax + s) * (qmax + s) < 1.0))
      return bad("evanescent modes: 1 - (q_max + s)^2 <= 0, refine the grid");
    // Eqs. fov11-fov12 expand the step's coupling in powers of
    // w = dz^ chi_h / cos(alpha); the series is summed in FP64, which stays
    // accurate for |w| <= 1 (steps far shorter than the extinction length)
    const double c = std::sqrt((1.0 - s) * (1.0 + s));
    const double w = k * p->dz_um * std::hypot(p->chih_re, p->chih_im) / c;
    const double phi_im = k * p->dz_um * std::fabs(p->chi0_im) / (2.0 * c);
    if (!(w <= 1.0))
      return bad("dz too long for the coupling expansion: |dz^ chi_h / cos(alpha)| = " +
                 std::to_string(w) + " > 1");
    if (!(phi_im <= 700.0)) return bad("dz too long: the per-step absorption underflows");
  }
  return BPM_OK;
}

int validate_problem3d(const bpm_problem* p, int ny, double dy_um, double y0_um,
                       std::string* why) {
  auto bad = [&](const std::string& m) { *why = m; return BPM_ERR_INVALID; };
  int rc = validate_problem(p, why);
  if (rc != BPM_OK) return rc;
  if (p->precision != BPM_FP32_FUSED) return bad("3D plans run in BPM_FP32_FUSED");
  if (p->nx < 256 || p->nx > 4096) return bad("3D plans need nx in [256, 4096]");
  if (ny < 256 || ny > 1024 || (ny & (ny - 1)))
    return bad("ny must be a power of two in [256, 1024]");
  if (!(dy_um > 0) || !finite(dy_um)) return bad("dy_um must be > 0");
  if (!finite(y0_um)) return bad("y0_um must be finite");
  for (int j = 0; j < p->n_energy; ++j) {
    double e = p->energy_ev[j];
    double s = std::sin(p->theta_b_ref_rad) * (p->e_ref_ev / e);
    double k = kTwoPi / (kHcEvAngstrom / e * 1e-4);
    double qx = M_PI / (k * p->dx_um), qy = M_PI / (k * dy_um);
    if (!((qx + s) * (qx + s) + qy * qy < 1.0))
      return bad("evanescent modes: 1 - (qx_max + s)^2 - qy_max^2 <= 0, refine the grid");
  }
  return BPM_OK;
}

void compute_energy_consts(bpm_plan_s* plan) {
  plan->ec.clear();
  for (double e : plan->energies) {
    EnergyConsts c{};
    c.e_ev = e;
    double lam_a = kHcEvAngstrom / e;
    double lam_um = lam_a * 1e-4;
    c.k_um = kTwoPi / lam_um;
    c.s = std::sin(plan->theta_b_ref) * (plan->e_ref_ev / e);
    c.c = std::sqrt((1.0 - c.s) * (1.0 + c.s));
    c.dzh = c.k_um * plan->dz_um;
    c.dxh = c.k_um * plan->dx_um;
    c.w = c.dzh * plan->chih / c.c;
    c.phi0 = c.dzh * plan->chi0 / (2.0 * c.c);
    cd ephi = std::exp(cd(0.0, 1.0) * c.phi0);
    cd j0m1 = bessel(0, c.w, true);
    cd j1 = bessel(1, c.w, false);
    c.a = (1.0 + j0m1) * ephi;
    c.b = cd(0.0, 1.0) * j1 * ephi;
    c.am1 = j0m1 * ephi + expm1_i(c.phi0);
    c.gphase = std::fmod(c.dzh * c.c, kTwoPi);
    plan->ec.push_back(c);
  }
}

// Radices of the fused kernel's passes: radix 16 while at least 16 remain,
// then one pass with the remaining power of two.
static std::vector<int> fused_radices(int logn) {
  std::vector<int> r;
  int left = logn;
  while (left > 4) { r.push_back(16); left -= 4; }
  r.push_back(1 << left);
  return r;
}

std::vector<int> fft_output_order(int logn) {
  int n = 1 << logn;
  std::vector<int> rad = fused_radices(logn);
  std::vector<int> out(n);
  for (int pos = 0; pos < n; ++pos) {
    int rem = pos, len = n, freq = 0, mult = 1;
    for (int r : rad) {
      int stride = len / r;
      int d = rem / stride;
      rem %= stride;
      freq += d * mult;
      mult *= r;
      len = stride;
    }
    out[pos] = freq;
  }
  return out;
}

// Split bands (N = M P), per band and local position pos of the local
// M-point transform's digit-reversed output, with spectral index k and
// D = (P(q) - 1)/N:
//   P = 2: [band][D(k) | D(k + M)][pos] -- the kernel forms
//          X_r = F_0 + (-1)^r W_N^k F_1 and D(k + M r) X_r itself, so each
//          table value is rounded relative to itself;
//   P = 4: [band][h][delta][pos] of E_delta[k] W_N^{s k}, s = h' - h for the
//          sender h' = (h + delta) mod 4, E_delta[k] = sum_r W_4^{delta r}
//          D[k + M r], as double-float pairs (hi, lo): float4 (hi.re,
//          hi.im, lo.re, lo.im).  Part h forms sum_delta of these times the
//          senders' local spectra F_h'.  E mixes D values of very different
//          size, so a single float would round the small ones far beyond
//          their own size, and that error repeats every step; hi + lo keeps
//          it at FP64 level.
void split_prop_table(const bpm_plan_s* plan, const std::vector<cd>& inc, int logm,
                      std::vector<float2>* out) {
  const int n = plan->nx, m = 1 << logm, parts = n / m;
  std::vector<int> local = fft_output_order(logm);
  out->assign(size_t(split_table_stride(plan, logm)), float2{0.f, 0.f});
  std::vector<cd> dk(parts), root(parts == 2 ? 0 : n);   // root[m] = W_N^m
  for (int m = 0; m < int(root.size()); ++m) {
    double cr, ci;
    unit_root(m, n, &cr, &ci);
    root[m] = cd(cr, ci);
  }
  for (int band = 0; band < 2; ++band) {
    for (int pos = 0; pos < m; ++pos) {
      for (int r = 0; r < parts; ++r) dk[r] = inc[size_t(band) * n + local[pos] + m * r];
      if (parts == 2) {
        for (int r = 0; r < 2; ++r)
          (*out)[(size_t(band) * 2 + r) * m + pos] =
              float2{float(dk[r].real()), float(dk[r].imag())};
        continue;
      }
      for (int dl = 0; dl < parts; ++dl) {
        cd e(0.0, 0.0);
        for (int r = 0; r < parts; ++r) e += root[((dl * r) % parts) * m] * dk[r];
        for (int h = 0; h < parts; ++h) {
          const int sh = h + dl < parts ? dl : dl - parts;     // h' - h
          const cd f = e * root[((sh * local[pos]) % n + n) % n];   // W_N^{sh k}
          const float fr = float(f.real()), fi = float(f.imag());
          const size_t at = 2 * (((size_t(band) * parts + h) * parts + dl) * m + pos);
          (*out)[at] = float2{fr, fi};
          (*out)[at + 1] = float2{float(f.real() - double(fr)), float(f.imag() - double(fi))};
        }
      }
    }
  }
}

int split_table_stride(const bpm_plan_s* plan, int logm) {
  const int parts = plan->nx >> logm;
  return parts == 2 ? 2 * parts * (1 << logm) : 2 * parts * parts * (1 << logm) * 2;
}

void prop_increments(const bpm_plan_s* plan, int row, double frac, std::vector<cd>* out) {
  const EnergyConsts& c = plan->ec[row];
  const int n = plan->nx;
  out->resize(2 * size_t(n));
  const double inv_n = 1.0 / double(n);
  auto value = [&](int k, int sign) {
    return expm1_i(frac * c.dzh * delta_q(fftfreq_q(k, n, c.dxh), c.s, c.c, sign)) * inv_n;
  };
  cd *up = out->data(), *down = up + n;
  for (int k = 0; k < n; ++k) up[k] = value(k, +1);
  // delta_-(q) = delta_+(-q), the same floating-point operations up to signs
  // that cancel, so psi_-'s table is psi_+'s mirrored (plan creation of FP64
  // 24 x 16384 18.7 -> 10.4 ms); 0 and -n/2 have no mirror image
  down[0] = value(0, -1);
  down[n / 2] = value(n / 2, -1);
  for (int k = 1; k < n; ++k)
    if (k != n / 2) down[k] = up[n - k];
}

void fused_prop_table(const bpm_plan_s* plan, const std::vector<cd>& inc,
                      std::vector<float2>* out) {
  if (plan->logn >= kSplitLogN) {   // N = 4096 P, P = 2 or 4
    split_prop_table(plan, inc, 12, out);
    return;
  }
  const int n = plan->nx;
  std::vector<int> order = fft_output_order(plan->logn);
  out->resize(2 * size_t(n));
  for (int band = 0; band < 2; ++band)
    for (int pos = 0; pos < n; ++pos) {
      const cd d = inc[size_t(band) * n + order[pos]];
      (*out)[size_t(band) * n + pos] = float2{float(d.real()), float(d.imag())};
    }
}

size_t nat_stride(const bpm_plan_s* plan, int tables) {
  return size_t(tables) * 2 * plan->nx + (plan->logn <= 7 ? 1 : 0);
}

void natural_prop_table(const std::vector<cd>& inc, float2* out) {
  for (size_t i = 0; i < inc.size(); ++i)
    out[i] = float2{float(inc[i].real()), float(inc[i].imag())};
}

float2 prop_form(const std::vector<cd>& inc) {
  const double n = 0.5 * double(inc.size());
  double sum = 0.0;
  for (const cd& v : inc) sum += std::norm(v);
  return sum * n * n > 2.0 * n ? float2{float(1.0 / n), 0.f} : float2{0.f, 1.f};
}

// Frequency of value j of thread t, at index j T + t (T = n/8 threads), of the
// 3D march's transforms: radix-8 passes and one of the power of two that is
// left, the last pass's group i of thread t being t + i T.
static std::vector<int> vol_order(int logn) {
  const int n = 1 << logn, T = n / 8, np = (logn + 2) / 3, rl = 1 << (logn - 3 * (np - 1));
  std::vector<int> out(n);
  for (int j = 0; j < 8; ++j)
    for (int t = 0; t < T; ++t) {
      int rem = (t + (j / rl) * T) * rl + j % rl, freq = 0, mult = 1, len = n;
      for (int p = 0; p < np; ++p) {
        const int r = p < np - 1 ? 8 : rl, stride = len / r;
        freq += (rem / stride) * mult;
        rem %= stride;
        mult *= r;
        len = stride;
      }
      out[j * T + t] = freq;
    }
  return out;
}

void vol_prop_table(const bpm_plan_s* plan, int row, std::vector<float2>* out) {
  // delta_+-(qx, qy) = sqrt(1 - (qx +- s)^2 - qy^2) - cos(alpha)
  //                  = -(qx (qx +- 2 s) + qy^2) / (sqrt(...) + cos(alpha))
  const EnergyConsts& c = plan->ec[row];
  const int nx = plan->nx, ny = plan->ny, ty = ny / 8;
  const double dyh = c.k_um * plan->dy_um;
  const std::vector<int> ox = vol_order(plan->logn), oy = vol_order(plan->logny);
  const double inv = 1.0 / (double(nx) * double(ny));
  out->resize(2 * size_t(nx) * ny);
  // [band][tile of 4 columns][j][column, t]: what thread (column, t) reads
  for (int band = 0; band < 2; ++band) {
    const double sign = band == 0 ? 1.0 : -1.0;
    for (int x = 0; x < nx; ++x) {
      const double qx = fftfreq_q(ox[x], nx, c.dxh);
      const double t = qx + sign * c.s;
      float2* col = out->data() + (size_t(band) * (nx / 4) + x / 4) * 4 * ny + (x % 4) * ty;
      for (int i = 0; i < ny; ++i) {
        const double qy = fftfreq_q(oy[i], ny, dyh);
        const double root = std::sqrt(1.0 - t * t - qy * qy);
        const double delta = -(qx * (qx + sign * 2.0 * c.s) + qy * qy) / (root + c.c);
        const cd d = expm1_i(c.dzh * delta) * inv;
        col[size_t(i / ty) * 4 * ty + i % ty] = float2{float(d.real()), float(d.imag())};
      }
    }
  }
}

std::vector<std::pair<double, double>> split_stages(int method) {
  if (method == BPM_SPLIT_VERLET) return {{0.0, 0.5}, {1.0, 0.5}};
  if (method == BPM_SPLIT_FOREST_RUTH) {
    const double t = 1.0 / (2.0 - std::cbrt(2.0));
    return {{0.0, t / 2.0}, {t, (1.0 - t) / 2.0}, {1.0 - 2.0 * t, (1.0 - t) / 2.0}, {t, t / 2.0}};
  }
  return {{1.0, 1.0}};
}

void coupling_frac(const bpm_plan_s* plan, int row, double frac, cd* a, cd* b) {
  const EnergyConsts& c = plan->ec[row];
  const cd w = frac * c.w, phi0 = frac * c.phi0;
  const cd ephi = std::exp(cd(0.0, 1.0) * phi0);
  *a = (1.0 + bessel(0, w, true)) * ephi;
  *b = cd(0.0, 1.0) * bessel(1, w, false) * ephi;
}

void plain_prop_table_frac(const bpm_plan_s* plan, int row, double frac,
                           std::vector<double2>* out) {
  const EnergyConsts& c = plan->ec[row];
  int n = plan->nx;
  out->assign(2 * size_t(n), double2{0.0, 0.0});
  double inv_n = 1.0 / double(n);
  for (int band = 0; band < 2; ++band) {
    int sign = band == 0 ? +1 : -1;
    for (int m = 0; m < n; ++m) {
      double q = fftfreq_q(m, n, c.dxh);
      double ph = frac * c.dzh * delta_q(q, c.s, c.c, sign);
      (*out)[size_t(band) * n + m] = double2{std::cos(ph) * inv_n, std::sin(ph) * inv_n};
    }
  }
}

void plain_prop_table(const bpm_plan_s* plan, int row, std::vector<double2>* out) {
  const EnergyConsts& c = plan->ec[row];
  int n = plan->nx;
  out->assign(2 * size_t(n), double2{0.0, 0.0});
  double inv_n = 1.0 / double(n);
  for (int band = 0; band < 2; ++band) {
    int sign = band == 0 ? +1 : -1;
    for (int m = 0; m < n; ++m) {
      double q = fftfreq_q(m, n, c.dxh);
      double ph = c.dzh * delta_q(q, c.s, c.c, sign);
      (*out)[size_t(band) * n + m] = double2{std::cos(ph) * inv_n, std::sin(ph) * inv_n};
    }
  }
}

static void unit_root(int m, int n, double* cr, double* ci) {
  // exp(-2 pi i m / n) with exact zeros on the axes.
  double ang = kTwoPi * (double(m) / double(n));
  double c = std::cos(ang), s = -std::sin(ang);
  if ((4 * m) % n == 0) {
    int q = (4 * m) / n;
    const double cs[4][2] = {{1, 0}, {0, -1}, {-1, 0}, {0, 1}};
    c = cs[q & 3][0];
    s = cs[q & 3][1];
  }
  *cr = c;
  *ci = s;
}

void twiddle_table_f32(int n, std::vector<float4>* out) {
  out->resize(n);
  auto put = [&](int m, double c, double s, float ch, float sh) {
    (*out)[m] = float4{ch, sh, float(c - double(ch)), float(s - double(sh))};
  };
  if (n < 8) {
    for (int m = 0; m < n; ++m) {
      double c, s;
      unit_root(m, n, &c, &s);
      put(m, c, s, float(c), float(s));
    }
    return;
  }
  // the first octant, exp(-i a) with a = 2 pi m / n <= pi / 4, and its mirror
  // images
  for (int m = 0; m <= n / 8; ++m) {
    double c, s;
    unit_root(m, n, &c, &s);
    // of the floats next to (c, s), the pair whose modulus is nearest to one:
    // a forward and an inverse pass multiply by W and its conjugate, so the
    // modulus error is the one that repeats every step at the same modes
    // (marches of 2000-6000 steps with the spread kernels' three twiddle
    // passes: relative error 4.7e-6 -> 4.3e-6 at N = 8192, 3.6e-6 -> 3.1e-6 at
    // 2048).  Weighing the phase error with 0.03 made single steps 2 % better and
    // marches of 4000 to 6000 steps 4 to 5 % worse; launches of few steps apply
    // the low part too (kFewSteps)
    float ch = float(c), sh = float(s);
    if (m != 0 && m != n / 8) {
      const float c0 = ch, s0 = sh;
      double best = 1.0;
      for (int i = -1; i <= 1; ++i)
        for (int j = -1; j <= 1; ++j) {
          const float ci = i == 0 ? c0 : std::nextafterf(c0, i * 2.f);
          const float sj = j == 0 ? s0 : std::nextafterf(s0, j * 2.f);
          const double err = std::fabs(double(ci) * ci + double(sj) * sj - 1.0);
          if (err < best) {
            best = err;
            ch = ci;
            sh = sj;
          }
        }
    }
    const int q = n / 4;
    put(m, c, s, ch, sh);                              // (c, s), s <= 0
    put(q - m, -s, -c, -sh, -ch);
    put(q + m, s, -c, sh, -ch);
    put(2 * q - m, -c, s, -ch, sh);
    if (m == 0) {
      put(2 * q, -c, -s, -ch, -sh);
      put(3 * q, -s, c, -sh, ch);
      continue;
    }
    put(2 * q + m, -c, -s, -ch, -sh);
    put(3 * q - m, s, c, sh, ch);
    put(3 * q + m, -s, c, -sh, ch);
    put(4 * q - m, c, -s, ch, -sh);
  }
}

void twiddle_table_f64(int n, std::vector<double2>* out) {
  out->resize(n);
  for (int m = 0; m < n; ++m) {
    double c, s;
    unit_root(m, n, &c, &s);
    (*out)[m] = double2{c, s};
  }
}

}  // namespace bpm
