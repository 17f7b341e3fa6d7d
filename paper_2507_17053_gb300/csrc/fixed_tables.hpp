// The fixed-point tables of the 3D FP64 cell term (fixed_point.cuh), built on
// the host in double-double arithmetic.
#pragma once

#include <vector>

#include "fixed_point.cuh"

namespace sbm {

struct Tables1D;

struct FixedTables {
  fix::Block Vt, V;                  // nodal line -> scaled modes; modes -> nodal line
  std::vector<fix::Entry> xline;     // x-line operators, slot by slot (XLineOp's packed layout)
  int eoff = 0;                      // result unit: biased exponent E + eoff (to_double's eb)
};

// Tables of the pencil of t for the cell operator scaled by scale = h^(d-2);
// false if a bound the arithmetic relies on does not hold.
bool build_fixed_tables(const Tables1D& t, double scale, FixedTables* out);

}  // namespace sbm
