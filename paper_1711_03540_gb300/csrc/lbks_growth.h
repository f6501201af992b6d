// Internal: the linear stability check of the constructors (lbks_params.cpp).
#pragma once

namespace lbks {

// Whether lb_ks_max_growth about rho = 0 at nk phases exceeds `limit`, decided phase by
// phase without the roots where they need not be known (each phase's largest root is
// computed only when it may lie outside the limit's circle).
bool growth_exceeds(int scheme, double dx, double dt, double tau, int dm_variant, int nk, double limit);

}  // namespace lbks
