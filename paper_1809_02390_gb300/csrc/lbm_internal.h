// Internal declarations shared by the library's translation units.
#pragma once

#include <cstddef>
#include <cstdint>

#include "lbm.h"

namespace lbm {

// Host thermodynamics and parameter derivation (lbm_thermo.cpp).
double critical_temperature(int kind, double a, double b, double R);
int maxwell(int kind, double a, double b, double R, double T, double K, double* rho_g, double* rho_l,
            double* p_star);
void interface_constants(int kind, double a, double b, double R, double T, double K, double rho_g,
                         double rho_l, double p_star, double* W1, double* sigma1);
int derive(const lb_params* p, lb_derived* d, char* err, size_t errlen);
const char* thread_error();

// Whether steps may store their results straight into a record that starts at address
// `at`, states of `bytes` bytes one behind the other.  Tensor copies read the states back
// on 16-byte boundaries; FP16 stores of lattices of even width write two nodes in 4 bytes
// (so do all their states then, `bytes` being a multiple of 4); the other stores and the
// resident run's write single elements.
inline bool record_in_place(const lb_params& p, uintptr_t at, size_t bytes, bool tensor) {
  const unsigned elem = p.precision == LB_FP64 ? 8 : p.precision == LB_FP32 ? 4 : p.nx % 2 == 0 ? 4 : 2;
  return tensor ? at % 16 == 0 && bytes % 16 == 0 : at % elem == 0;
}
inline bool record_by_elements(const lb_params& p, uintptr_t at) {
  return at % (p.precision == LB_FP64 ? 8 : p.precision == LB_FP32 ? 4 : 2) == 0;
}
void set_thread_error(const char* msg);

}  // namespace lbm
