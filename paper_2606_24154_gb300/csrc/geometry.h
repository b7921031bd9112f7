// geometry.h -- host-side element-table construction (see geometry.cpp).
#pragma once
#include <string>
#include <vector>

#include "nb_internal.h"

namespace nb {

// Build the device record, the interface-row diagonal term and the FP32 far-field nodes
// of one raw element (tier distances in element radii from opt).  Returns NEBEM_OK or an
// error code with a reason in `why`.
int build_element(const nebem_element& r, const nebem_options& opt, Elem& e, double& diag, FarNodes& fn,
                  std::string& why);

// Gauss-Legendre nodes and weights on [0, 1] (m <= 16), by Newton iteration on P_m.
void gauss_legendre01(int m, double* x, double* w);

// Grid (box and cell edge) of the near-pair search over the image centroids c_j + t_k; near radius of
// element j = ratio_near * rho_j.  The cell list itself is made on the device (launch_cell_list).
int near_grid_box(const std::vector<Elem>& el, const ImageTable& img, double ratio_near, NearGrid& grid,
                  std::string& why);

// The rules of the fill's node tables (launch_fill_tables): Gauss-Legendre on [0, 1] with 3, 4 and 6
// nodes, and the two orbits of the 6-point triangle rule (barycentric place, share of the area).
struct GaussRules {
    double x3[3], w3[3], x4[4], w4[4], x6[6], w6[6], tri_a[2], tri_w[2];
};
GaussRules gauss_rules();

// Image translations t = k1 a1 + k2 a2, index (k1-lo)*m + (k2-lo); lattice NULL -> one
// zero translation.
int build_images(const double* lattice, int lo, int hi, ImageTable& img, std::string& why);

}  // namespace nb
