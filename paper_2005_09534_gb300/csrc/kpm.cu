// Density of states of H~ by the kernel polynomial method (Weisse, Wellein,
// Alvermann, Fehske, Rev. Mod. Phys. 78, 275 (2006)): stochastic Chebyshev
// moments mu_n = (1/R) sum_r r^T T_n(H~) r of R random vectors, from the same
// H~ step kernel as the filter, and the Jackson-damped eigenvalue count of an
// interval.  The paper sets K from the density of states at the target
// ("POLFED algorithm" section and the Supplement's estimate of rho(0)) and
// cites iterative estimators of it; this is such an estimator.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "polfed_internal.h"

namespace polfed {

// Jackson damping factors g_n, n = 0..N-1 (Weisse et al., Eq. (71)).
void jackson_coeffs(int N, std::vector<double>& g) {
  g.assign(N, 1.0);
  const double q = M_PI / (N + 1);
  for (int n = 0; n < N; n++)
    g[n] = ((N - n + 1) * std::cos(q * n) + std::sin(q * n) / std::tan(q)) / (N + 1);
}

namespace {

// [t_n in FP64 for odd n] [mu] [partial sums]
constexpr size_t kMuBytes = (size_t)2 * (kMaxKpmMoments / 2 + 1) * sizeof(double);

}  // namespace

size_t kpm_buffer_bytes(const HamPlan& plan, int kind, int R) {
  const size_t v = (size_t)plan.geo.dim * R * sizeof(double);
  return moment_scratch_bytes(plan, kind, R) + kMuBytes + kMaxMomentCtas * 16 + std::min<size_t>(v, 1 << 20);
}

int kpm_moments(HamPlan& plan, int kind, const void* r, int R, int n_mom, double* mu, void* buf, FilterScratch& scr,
                cudaStream_t s) {
  const int half = (n_mom + 1) / 2;  // t_0 .. t_half are needed
  char* p = (char*)buf;
  char* d_mu = p + moment_scratch_bytes(plan, kind, R);
  char* part = d_mu + (((size_t)2 * half * sizeof(double) + 255) & ~(size_t)255);
  const size_t part_bytes = (size_t)(p + kpm_buffer_bytes(plan, kind, R) - part);
  PF_CHECK(moment_steps(plan, kind, r, R, half, p, part, part_bytes, (double*)d_mu, scr, s));
  std::vector<double> raw((size_t)2 * half);
  PF_CUDA(cudaMemcpyAsync(raw.data(), d_mu, raw.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
  PF_CUDA(cudaStreamSynchronize(s));
  // raw[0] = r.r, raw[1] = r.H~r; raw[2k] = t_k.t_k, raw[2k+1] = t_{k+1}.t_k
  //   T_{2k} = 2 T_k^2 - T_0,  T_{2k+1} = 2 T_{k+1} T_k - T_1
  const double m0 = raw[0], m1 = raw[1];
  for (int j = 0; j < n_mom; j++) {
    double v;
    if (j < 2)
      v = raw[j];
    else
      v = 2.0 * raw[j] - ((j & 1) ? m1 : m0);
    mu[j] = v / R;
  }
  for (int j = 0; j < n_mom; j++)
    if (!std::isfinite(mu[j]) || std::fabs(mu[j]) > 1.01 * std::fabs(mu[0]) + 1e-300)
      return fail(POLFED_EBOUNDS, "KPM moment |mu_n| > mu_0: spectrum outside [e_lo, e_hi]");
  return POLFED_OK;
}

// Fraction of the spectrum in [x_a, x_b] from Jackson-damped moments:
// the indicator's Chebyshev coefficients are c_0 = (th_a - th_b) / pi and
// c_n = 2 (sin n th_a - sin n th_b) / (n pi), th = arccos x.
double kpm_count_fraction(const double* mu, int n_mom, double x_a, double x_b) {
  std::vector<double> g;
  jackson_coeffs(n_mom, g);
  const double ta = std::acos(std::max(-1.0, std::min(1.0, x_a)));
  const double tb = std::acos(std::max(-1.0, std::min(1.0, x_b)));
  double f = (ta - tb) / M_PI * mu[0];
  for (int k = 1; k < n_mom; k++) f += g[k] * 2.0 * (std::sin(k * ta) - std::sin(k * tb)) / (k * M_PI) * mu[k];
  return f / mu[0];
}

}  // namespace polfed

using namespace polfed;

extern "C" {

int polfed_kpm_moments(const polfed_model* model, const uint32_t* d_states, int64_t dim, double e_lo, double e_hi,
                       int32_t n_mom, const void* d_R, int32_t R, int32_t dtype, double* mu, polfed_stream_t stream) {
  if (!model) return fail(POLFED_EINVAL, "model is NULL");
  if (model->L < 4 || model->L > 32 || (model->L & 1)) return fail(POLFED_EINVAL, "L must be even, 4 <= L <= 32");
  if (dim != (int64_t)binom_host(model->L, model->L / 2)) return fail(POLFED_EINVAL, "dim != C(L, L/2)");
  if (!d_states || !d_R || !mu) return fail(POLFED_EINVAL, "NULL argument");
  if (n_mom < 2 || n_mom > kMaxKpmMoments) return fail(POLFED_EINVAL, "n_mom must be in 2..65536");
  if (R < 1 || R > 128) return fail(POLFED_EINVAL, "R must be in 1..128");
  if (dtype != POLFED_F32 && dtype != POLFED_F64 && dtype != POLFED_DF64) return fail(POLFED_EINVAL, "bad dtype");
  if (!std::isfinite(e_lo) || !std::isfinite(e_hi) || !(e_lo < e_hi)) return fail(POLFED_EINVAL, "need e_lo < e_hi");
  cudaStream_t s = (cudaStream_t)stream;
  HamPlan plan;
  PF_CHECK(plan.init(model, s, true, moments_b(dtype, model->L), dtype, e_lo, e_hi));
  const size_t fb = (filter_scratch_bytes(plan, dtype, R) + 255) & ~(size_t)255;
  void* mem = nullptr;
  PF_CHECK(scratch_alloc(&mem, fb + kpm_buffer_bytes(plan, dtype, R), s));
  FilterScratch scr;
  scr.xs = mem;
  scr.bytes = fb;
  const int rc = kpm_moments(plan, dtype, d_R, R, n_mom, mu, (char*)mem + fb, scr, s);
  cudaFreeAsync(mem, s);
  cudaStreamSynchronize(s);
  return rc;
}

int polfed_kpm_count(const double* mu, int32_t n_mom, double x_a, double x_b, double* fraction) {
  if (!mu || !fraction) return fail(POLFED_EINVAL, "NULL argument");
  if (n_mom < 1 || n_mom > kMaxKpmMoments) return fail(POLFED_EINVAL, "n_mom must be in 1..65536");
  if (!(x_a <= x_b) || !(mu[0] != 0.0)) return fail(POLFED_EINVAL, "need x_a <= x_b and mu[0] != 0");
  *fraction = kpm_count_fraction(mu, n_mom, x_a, x_b);
  return POLFED_OK;
}

}  // extern "C"
