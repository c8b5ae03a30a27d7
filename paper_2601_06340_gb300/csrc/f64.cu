// FP64 plans of N = 64 .. 16384: buffers, tables and launches of the fused
// FP64 march (f64_kernel.cuh).
#include <algorithm>
#include <atomic>
#include <vector>

#include "f64_kernel.cuh"

namespace bpm {

namespace {

constexpr size_t kF64SyncBytes = 256;

template <int LOGN>
int f64_resident() {   // CTAs that the GPU keeps resident at once
  static std::atomic<int> cached{0};
  int c = cached.load(std::memory_order_relaxed);
  if (c == 0) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f64_march_kernel<LOGN>,
                                                      F64Cfg<LOGN>::T, 0) != cudaSuccess)
      cudaGetLastError();
    c = std::max(1, per * sms);
    cached.store(c, std::memory_order_relaxed);
  }
  return c;
}

template <int LOGN>
int f64_launch(F64March* a, cudaStream_t st) {
  using C = F64Cfg<LOGN>;
  // as many rounds of items as residency needs, all of the same number of
  // CTAs: a phase ends with its last item, and one alone on its SM takes as
  // long as a full round (16 rows of N = 4096 on 912 + 112 CTAs 46 us a step)
  const int items = a->nb * C::ITEMS;
  const int rounds = (items + f64_resident<LOGN>() - 1) / f64_resident<LOGN>();
  const int grid = (items + rounds - 1) / rounds;
  void* args[] = {a};
  cudaError_t e =
      cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(f64_march_kernel<LOGN>),
                                  dim3(grid), dim3(C::T), args, 0, st);
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "FP64 march launch");
}

template <typename F>
auto with_size(int logn, F f) {
  switch (logn) {
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    case 9: return f(std::integral_constant<int, 9>{});
    case 10: return f(std::integral_constant<int, 10>{});
    case 11: return f(std::integral_constant<int, 11>{});
    case 12: return f(std::integral_constant<int, 12>{});
    case 13: return f(std::integral_constant<int, 13>{});
    default: return f(std::integral_constant<int, 14>{});
  }
}

}  // namespace

bool f64_fused(const bpm_plan_s* plan) {
  return plan->precision == BPM_FP64_PLAIN && plan->logn >= 6;
}

void f64_prop_table(const bpm_plan_s* plan, const std::vector<std::complex<double>>& inc,
                    const std::vector<int>& rev, double2* out) {
  const size_t n = plan->nx;
  for (size_t b = 0; b < 2; ++b)
    for (size_t p = 0; p < n; ++p) {
      const std::complex<double>& v = inc[b * n + size_t(rev[p])];
      out[b * n + p] = make_double2(v.real(), v.imag());
    }
}

std::vector<int> bit_reversal(int bits) {
  std::vector<int> r(size_t(1) << bits, 0);
  for (size_t i = 1; i < r.size(); ++i)
    r[i] = (r[i >> 1] >> 1) | (int(i & 1) << (bits - 1));
  return r;
}

size_t f64_twiddle_count(const bpm_plan_s* plan) {
  const size_t n1 = size_t(1) << (plan->logn / 2);
  return n1 + plan->nx / n1 + 2 * size_t(plan->nx);
}

void f64_twiddles(const bpm_plan_s* plan, std::vector<double2>* out) {
  const int logn = plan->logn, a = logn / 2, b = logn - a;
  const size_t n = plan->nx, n1 = size_t(1) << a, n2 = size_t(1) << b;
  std::vector<double2> w;
  twiddle_table_f64(int(n), &w);
  const std::vector<int> ra = bit_reversal(a);
  out->assign(f64_twiddle_count(plan), double2{1.0, 0.0});
  double2 *xf = out->data(), *ki = xf + n1, *kf = ki + n2, *xi = kf + n;
  for (int s = 0; s < std::max(a, b); ++s) {
    const std::vector<int> rs = bit_reversal(s);
    for (size_t j = 0; j < size_t(1) << s; ++j) {
      const size_t at = (size_t(1) << s) + j;
      if (s < a) xf[at] = w[size_t(rs[j]) << (logn - 1 - s)];
      if (s < b) ki[at] = w[j << (logn - 1 - s)];
      if (s < b)
        for (size_t p = 0; p < n1; ++p)
          kf[p * n2 + at] = w[(size_t(rs[j]) * n1 + size_t(ra[p])) << (b - 1 - s)];
      if (s < a)
        for (size_t c = 0; c < n2; ++c) xi[c * n1 + at] = w[(j * n2 + c) << (a - 1 - s)];
    }
  }
}

size_t f64_part_bytes(const bpm_plan_s* plan) {
  return with_size(plan->logn, [&](auto L) {
    return size_t(plan->nb) * F64Cfg<decltype(L)::value>::ITEMS * 2 * sizeof(double);
  });
}

size_t f64_scratch_bytes(const bpm_plan_s* plan) {
  return kF64SyncBytes + f64_part_bytes(plan) + size_t(plan->nb) * 2 * plan->nx * sizeof(double2);
}

void f64_rows(const bpm_plan_s* plan, void* d_records, double* d_powers,
              std::vector<F64Row>* out) {
  const size_t n = plan->nx, nb = plan->nb;
  const auto stages = split_stages(plan->split);
  const bool fr = plan->split == BPM_SPLIT_FOREST_RUTH;
  out->resize(nb);
  for (size_t r = 0; r < nb; ++r) {
    F64Row& d = (*out)[r];
    d.state = static_cast<double2*>(plan->d_state) + r * 2 * n;
    d.prop = static_cast<const double2*>(fr ? plan->d_stage_prop : plan->d_prop) + r * 2 * n;
    d.prop2 = fr ? d.prop + nb * 2 * n : nullptr;
    d.phasor = static_cast<const double2*>(plan->d_phasor);
    d.records = d_records ? static_cast<double2*>(d_records) + r * plan->n_rec * 2 * n : nullptr;
    d.powers = d_powers ? d_powers + r * (plan->n_rec + 1) * 2 : nullptr;
    // a splitting form's outer couplings (its first stage's) and, of
    // Forest-Ruth, the inner ones (its second stage's); else the step's
    auto coupling = [&](double frac, double2* am1, double2* b) {
      std::complex<double> ca, cb;
      coupling_frac(plan, int(r), frac, &ca, &cb);
      *am1 = make_double2(ca.real() - 1.0, ca.imag());
      *b = make_double2(cb.real(), cb.imag());
    };
    coupling(stages.front().second, &d.am1h, &d.bh);
    coupling(stages[fr ? 1 : 0].second, &d.am1, &d.b);
    if (plan->split == BPM_SPLIT_FIRST_ORDER) {
      d.am1 = make_double2(plan->ec[r].am1.real(), plan->ec[r].am1.imag());
      d.b = make_double2(plan->ec[r].b.real(), plan->ec[r].b.imag());
    }
    d.gphase = plan->ec[r].gphase;
    d.dx_um = plan->dx_um;
  }
}

int launch_f64(bpm_plan_s* plan, int n_begin, int n_end, int n_phase0, bool records, int* status,
               cudaStream_t st) {
  char* base = static_cast<char*>(plan->d_f64);
  F64March a{};
  a.rows = static_cast<const F64Row*>(plan->d_rows);
  a.tw = static_cast<const double2*>(plan->d_tw);
  a.sync = reinterpret_cast<unsigned*>(base);
  a.part = reinterpret_cast<double*>(base + kF64SyncBytes);
  a.xbuf = reinterpret_cast<double2*>(base + kF64SyncBytes + f64_part_bytes(plan));
  a.status = status;
  a.nb = plan->nb;
  a.steps = n_end - n_begin;
  a.split = plan->split;
  a.n_begin = n_begin;
  a.n_phase0 = n_phase0;
  a.record_every = records ? plan->record_every : 0;
  cudaError_t e = cudaMemsetAsync(base, 0, kF64SyncBytes, st);
  if (e != cudaSuccess) return cuda_fail(e, "FP64 march");
  return with_size(plan->logn, [&](auto L) { return f64_launch<decltype(L)::value>(&a, st); });
}


int march_f64(bpm_plan_s* plan, int n_begin, int n_end, int n_phase0, void* d_records,
              double* d_powers, int* status, cudaStream_t st) {
  if (!f64_fused(plan)) return plain_march(plan, n_begin, n_end, n_phase0, d_records, d_powers, st);
  std::vector<F64Row> rows;
  f64_rows(plan, d_records, d_powers, &rows);
  // (pageable memory: the copy is staged before the call returns)
  cudaError_t e = cudaMemcpyAsync(plan->d_rows, rows.data(), rows.size() * sizeof(F64Row),
                                  cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "upload row descriptors");
  return launch_f64(plan, n_begin, n_end, n_phase0, d_records || d_powers, status, st);
}

}  // namespace bpm
