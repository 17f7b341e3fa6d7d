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
  // faces (face_fixed.cuh): D0 [n], M [n][n], S [n][n] (phi_j'(0), the mass
  // matrix, phi_j at the Gauss points), the result exponents of q and tm
  std::vector<fix::Entry> face;
  int face_eq = 0, face_etm = 0;
  fix::DgTab dg;                     // discontinuous Galerkin line operators (dg_apply.cu)
  bool dg_pen_in = true;             // the penalty is in dg.w[0] (else added in double)
};

// Parts of the tables: the cell term (Vt, V, xline, eoff), the faces, the DG
// line operators.
enum : int { kFixCell = 1, kFixFaces = 2, kFixDg = 4 };

// Tables of the pencil of t for the cell operator scaled by scale = h^(d-2);
// false if a bound the arithmetic relies on does not hold.  pen: h times the
// interior-face penalty (DG).  What the
// degree alone decides is made once per process (p = 1 .. 6: 4 / 11 / 22 / 43 / 70 /
// 114 us on a host core, less without the cell term); a call then takes 0 / 1 / 3 /
// 7 / 13 / 23 us for the cell term and at most 2 for the rest.
bool build_fixed_tables(const Tables1D& t, double scale, FixedTables* out, double pen = 0.0,
                        int parts = kFixCell | kFixFaces | kFixDg);

}  // namespace sbm
