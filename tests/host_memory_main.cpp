// Calls of the C ABI while the host runs out of memory: the k-th `new` of a call fails, for every k up to the number
// the call makes.  No failure may come back as anything but LBCAD_E_OOM, and the context has to step on as if
// it had not happened.
// Prints "ok" and the number of failures per call, or what went wrong.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <new>
#include <vector>

#include "lbcad.h"

static long g_left = -1;  // allocations until one fails; negative: none fails

static void* take(std::size_t n) noexcept {
  if (g_left >= 0 && g_left-- == 0) return nullptr;
  return std::malloc(n ? n : 1);
}
void* operator new(std::size_t n) {
  if (void* p = take(n)) return p;
  throw std::bad_alloc();
}
void* operator new[](std::size_t n) { return operator new(n); }
void* operator new(std::size_t n, const std::nothrow_t&) noexcept { return take(n); }
void* operator new[](std::size_t n, const std::nothrow_t&) noexcept { return take(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete[](void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
void operator delete[](void* p, std::size_t) noexcept { std::free(p); }

#define NEED(what)                                                                          \
  do {                                                                                      \
    if (!(what)) {                                                                          \
      std::printf("%s:%d: %s (%s)\n", __FILE__, __LINE__, #what, lbcad_last_error(nullptr)); \
      std::exit(1);                                                                         \
    }                                                                                       \
  } while (0)

static const lbcad_grid kBox = {24, 20, 16};

static lbcad_params params(int precision) {
  lbcad_params p;
  std::memset(&p, 0, sizeof(p));
  p.tau = 1.0, p.rho0 = 1.0, p.A0 = 1.0, p.chi0 = 2.5, p.chis = 0.25, p.K = 0.04, p.q0 = 0.6, p.gammaQ = 0.3, p.xi = 0.7;
  p.a = p.b = 0.07, p.kphi = 0.14, p.M = 0.1, p.W = 0.02, p.zeta = 0.005, p.R = 5.0, p.S0 = 0.5, p.noise = 1e-3;
  p.centre[0] = 11.5, p.centre[1] = 9.5, p.centre[2] = 7.5;
  p.precision = precision;
  p.device = -1;
  return p;
}

static std::vector<char> state(lbcad_ctx* c) {
  size_t n = 0;
  NEED(lbcad_state_bytes(c, 0, &n) == LBCAD_OK);
  std::vector<char> s(n);
  NEED(lbcad_get_state(c, 0, s.data(), n, 0) == LBCAD_OK);
  return s;
}

// Fails the call's allocations one after the other, until the call needs no more; the number of failures.  (A call may
// do without an allocation that failed.)
static int fail_each(const std::function<int()>& call) {
  for (int k = 0;; ++k) {
    g_left = k;
    const int r = call();
    const bool failed = g_left < 0;
    g_left = -1;
    NEED(r == LBCAD_OK || (failed && r == LBCAD_E_OOM));
    if (!failed) return k;
    NEED(k < 1000);
  }
}

static void run(int precision) {
  const lbcad_params p = params(precision);
  const long long n = (long long)kBox.nx * kBox.ny * kBox.nz;
  std::vector<double> buf(28 * n);
  lbcad_ctx* ref = nullptr;
  NEED(lbcad_create(&kBox, &p, 7, &ref) == LBCAD_OK);
  NEED(lbcad_step(ref, 11) == LBCAD_OK);
  const std::vector<char> want = state(ref);
  lbcad_destroy(ref);

  lbcad_ctx* c = nullptr;
  std::printf("create %d", fail_each([&] {
                lbcad_destroy(c);
                return lbcad_create(&kBox, &p, 7, &c);
              }));
  NEED(lbcad_set_graph(c, 2) == LBCAD_OK && lbcad_step(c, 3) == LBCAD_OK);
  std::printf(", set_tiles %d", fail_each([&] { return lbcad_set_tiles(c, precision == LBCAD_FP32 ? 3 : 0); }));
  NEED(lbcad_step(c, 2) == LBCAD_OK);
  std::printf(", set_path %d", fail_each([&] { return lbcad_set_path(c, LBCAD_PATH_TWO_KERNEL); }));
  NEED(lbcad_set_path(c, LBCAD_PATH_FUSED) == LBCAD_OK);
  std::printf(", get_fields %d", fail_each([&] {
                return lbcad_get_fields(c, 0, LBCAD_FIELD_G | LBCAD_FIELD_U | LBCAD_FIELD_Q | LBCAD_FIELD_PSI, buf.data(),
                                        buf.size() * sizeof(double), 0);
              }));
  lbcad_obs o;
  std::printf(", observables %d", fail_each([&] { return lbcad_observables(c, 0, &o); }));
  std::printf(", step %d", fail_each([&] { return lbcad_step(c, 6); }));
  NEED(lbcad_step_count(c) == 11 && state(c) == want);
  lbcad_ctx* a = nullptr;
  NEED(lbcad_create(&kBox, &p, 7, &a) == LBCAD_OK);
  double dz, dq, J, dz1, dq1, J1;
  std::vector<double> dQ(5 * n), dQ1(5 * n);
  NEED(lbcad_adjoint(a, 11, 4, &dz, &dq, dQ.data(), &J) == LBCAD_OK);
  NEED(state(a) == want);
  lbcad_destroy(a);
  NEED(lbcad_create(&kBox, &p, 7, &a) == LBCAD_OK);
  const std::vector<char> start = state(a);
  std::printf(", adjoint %d\n", fail_each([&] {
                if (lbcad_set_state(a, 0, start.data(), start.size(), 0) != LBCAD_OK) return LBCAD_E_OOM;
                return lbcad_adjoint(a, 11, 4, &dz1, &dq1, dQ1.data(), &J1);
              }));
  NEED(dQ1 == dQ && state(a) == want);
  lbcad_destroy(a);
  lbcad_destroy(c);
}

int main() {
  run(LBCAD_FP32);
  run(LBCAD_FP64);
  std::puts("ok");
  return 0;
}
