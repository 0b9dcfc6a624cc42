// Host reader/packer for RDEMECH 1 text (see mech_layout.h for the image).
#pragma once
#include <stddef.h>

#include <string>
#include <vector>

#include "mech_layout.h"

namespace rde {

// Returns 0 on success, -1 on a syntax error, -2 on an inconsistent mechanism;
// *err receives a one-line description on failure.
// E_J, if given, receives each reaction's activation energy in J/mol (of k_inf for falloff).
int pack_mechanism(const char* text, size_t len, std::vector<unsigned char>* image, std::string* err,
                   std::vector<double>* E_J = nullptr);

// v log2(e) 2^bits rounded to an integer; false if it does not lie below 2^62.
bool scaled_log2(double v, int bits, int64_t* out);

// Fixed-point NASA polynomials of one mechanism for T in [Tlo, 8192) K (thermo_fix): per
// species and range Cp/R and the polynomial part of H/RT (10 coefficients in units of
// 2^-cp_bits), G/RT log2 e (7, in units of 2^-51) and d(Cp/R)/dT (4, 2^-dcp_bits[k]), each
// coefficient of T^j scaled by 2^(14 j).
struct FixThermo {
  std::vector<int64_t> c;   // [K][2][21]
  int cp_bits = 0;
  std::vector<int> dcp_bits;   // [K]
  double Tlo = 0.0;
};
// False where a coefficient does not fit, or where the unit of Cp/R would be coarser than
// 2^-56: the four steps of Horner's scheme lose up to 6.6 units, which with the final rounding
// is 0.71 ulp of a Cp/R between 2 and 4 at 2^-56, against 0.73 measured in FP64 (300 to
// 3,500 K, seeded H2/air; 0.52 in fixed point at its 2^-57).  Coefficients of the size of
// published fits take 2^-52 or 2^-53 and stay in FP64 (they would lose 2.8 ulp, FP64 1.2).
bool fix_thermo(const MechView& v, FixThermo* f);

// Fills the fixed-point form of every reaction's ln A, b and E/R (zA, zb, zE) and the
// header's Tfix; to be repeated when ln A or E change.
void fix_rates(unsigned char* image);

// Gather plan of the CTA-per-cell kernel (large_plan.h) for a packed image.
void build_large_plan(const unsigned char* image, std::vector<unsigned char>* plan);

}  // namespace rde
