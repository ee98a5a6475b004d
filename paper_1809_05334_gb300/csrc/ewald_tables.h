// Host set-up of the Ewald tables of one incidence (ewald_tables.cpp).
#pragma once
#include <vector>

#include "ewald_params.h"

namespace vie {

// Ewald parameters and tables of one incidence; status as vie_status;
// split_mult > 0: the FP32 tables' Ewald split multiplier (else the default);
// pow2: the spatial table's spacing for the far kernels (a power of two of the
// distance), else as fine as its size allows
int build_ewald_tables(double a, double b, double k0, double kx, double ky, double z_extent, bool fp64,
                       EwaldTables &E, std::vector<double> *orders, const char **why,
                       double split_mult = 0.0, bool pow2 = true);

// Polynomials of the spectral series for the far kernels (FarPoly) from the
// order map of make_ewald_f32: fp.mode = FAR_NONE where no short form applies,
// or where an order needs a degree above FP_MAX_DEG (a cell several periods
// thick); then the general tabulated form is used.  coef receives fp.n_coef
// floats.
void build_far_poly(const EwaldTables &t, const EwaldF32 &f, FarPoly &fp, std::vector<float> &coef);
// The FP64 form of a request whose tables were built with fp64 = true; f.n_blob = 0
// where it does not apply (an order of too high a degree, or too large a blob).
void build_far64(const EwaldTables &t, double k0, double kx, double ky, Far64 &f, std::vector<double> &blob);

}  // namespace vie
