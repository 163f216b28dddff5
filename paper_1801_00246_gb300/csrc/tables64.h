// The integer operator of the exactly sliced FP64 apply (apply_tc64.cu), built on the
// host (tables64.cpp).
#pragma once

#include <vector>

#include "dg_internal.h"

namespace dgx {

// OB of apply_tc64.cu, without (Poisson) or with the mass columns (Helmholtz). Columns
// come in chunks of 48: item i of kind c in chunk k is column (3 k + c) 16 + i, items in
// groups of eight: groups [0, gvol) hold nodes (kinds S_rr, S_rs + S_sr, S_ss),
// [gvol, gface) face nodes (kinds Dr_f^T Mf, Ds_f^T Mf, E_f Mf), those after them three
// nodes an item (mass). Entry (r, k) is x[r cols + k] 2^{ea[r] - 56}, |x| <= 2^56 + 1.
struct OutTable {
  int gvol = 0, gface = 0, chunks = 0, cols = 0;
  int k1 = 0, k2 = 0, km = 0;  // the flux, jump and mass columns are scaled by 2^k1, 2^k2, 2^km
  std::vector<int> ea;
  std::vector<long long> x;
};
void build_out_tables(const RefElem& R, OutTable (&t)[2]);  // [helmholtz]

}  // namespace dgx
