// Internal: the linear stability check of the constructors (lbks_params.cpp).
#pragma once

namespace lbks {

// lb_ks_max_growth about rho = 0 at nk phases where it exceeds `limit`, else `limit`.  Decided
// phase by phase without the roots where they need not be known: a phase's largest root is
// computed only when it may lie outside the circle of the largest rate so far.  first: any
// rate above the limit will do (the first one found).
double growth_above(int scheme, double dx, double dt, double tau, int dm_variant, int nk, double limit, bool first);

}  // namespace lbks
