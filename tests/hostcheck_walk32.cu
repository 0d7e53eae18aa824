// The quadrilateral walk on certified FP32 predicates (QPred32) against the
// walk on exact FP64 ones (QPred64), on the host, for every population the
// FP32 walk takes: returns the number of populations whose location differs;
// out = {populations compared, walks that needed the FP64 departure point,
// populations certified missing by the exterior cone, wrong ones among them}.
#include "hostcheck.cu"

extern "C" int alelb_hostcheck_walk32_q2(const alelb_mesh_desc *d, double t, int64_t out[4])
{
    HostTables T;
    QuadTables Q;
    std::string err;
    if (build_quad_tables(d, T, Q, err) != ALELB_OK) return -1;
    QuadDev M = quad_host_view(T, Q);
    M.cone = Q.cone.data();
    M.conek = Q.conek.data();
    MapStatic MS = T.host_map();
    const MapScalars sc = map_scalars(T.mkind, T.mp, t);
    MapScalarsF sf{};
    sf.s = (float)sc.s;
    sf.sd = (float)sc.sd;
    sf.vy = (float)sc.vy;
    sf.c = (float)sc.c;
    sf.sn = (float)sc.sn;
    sf.thd = (float)sc.thd;
    sf.cm = (float)sc.cm;
    sf.Xc = (float)T.mp[3];
    sf.Yc = (float)T.mp[4];
    sf.er0 = 2.0f;
    int bad = 0, e = 0;
    for (int k = 0; k < 4; ++k) out[k] = 0;
    for (int a = 0; a < T.N; ++a) {
        const float4 Xf = M.Xf[a];
        const FastMap F = fast_map(MS, sf, a, Xf);
        const double2 Xa = M.X[a];
        double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22, wx, wy;
        map_node(MS, sc, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
        metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
        mesh_velocity_term(a11, a12, a21, a22, ds(Vx, sc.Ux), ds(Vy, sc.Uy), false, wx, wy);
        for (int i = 0; i < NQ; ++i) {
            const float cx = (float)lat_cx(i), cy = (float)lat_cy(i);
            const float chx = F.A11 * cx + F.A12 * cy - F.W1;
            const float chy = F.A21 * cx + F.A22 * cy - F.W2;
            if (!F.ok || !(sqrtf(chx * chx + chy * chy) > 4.0f * F.eq(i))) continue;
            double hx, hy, px, py;
            departure(a11, a12, a21, a22, wx, wy, cx, cy, Xa.x, Xa.y, hx, hy, px, py);
            QPred32 p32{M, MS, sc, a, i, Xf, -chx, -chy, F.eq(i)};
            p32.have64 = false;
            const Loc L = quad_walk_t(M, p32, a, &e);
            const Loc R = quad_walk(M, a, Xa.x, Xa.y, px, py, &e);
            ++out[0];
            if (p32.have64) ++out[1];
            if (L.e != R.e || L.kind != R.kind || (R.e >= 0 && (L.sx != R.sx || L.sy != R.sy || L.vnode != R.vnode))) ++bad;
            const int ck = cone_missing(M, F, a, i);
            if (ck) {
                ++out[2];
                if (R.e != -1 || R.kind != ck) ++out[3];
            }
        }
    }
    return e ? -2 : bad;
}
