// Local coordinates of the FP64 form (quad_local64) on the host: n cells of
// four corners and a point each (10 numbers); returns how many did not settle.
#include <cstring>

#include "quad_tables.h"

using namespace alelb;

extern "C" int alelb_hostcheck_local64(int n, const double *in, double *out)
{
    int bad = 0;
    for (int k = 0; k < n; ++k) {
        const double *p = in + 10 * k;
        double2 v[4], b[5];
        for (int j = 0; j < 4; ++j) v[j] = make_double2(p[2 * j], p[2 * j + 1]);
        quad_map_coefficients(v, b);
        QuadDev M{};
        M.ebd = b;
        if (!quad_local64(M, 0, 0, 0, p[8], p[9], out[2 * k], out[2 * k + 1])) ++bad;
    }
    return bad;
}
