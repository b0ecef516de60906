// Host-side rules of the library's launch plans.
#include "prc_host.h"

extern "C" int host_f64_tile_rows(int nx, int ny, int num_sms)
{
    lbm_params p = {};
    p.nx = nx;
    p.ny = ny;
    p.dtype = LBM_F64;
    return prc_host::f64_tile_threads(p, num_sms) / prc::BX;
}
