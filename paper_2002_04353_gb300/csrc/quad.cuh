// quad.cuh -- the paper's 9-node quadrilateral element (Sec. III): the
// bilinear geometry of Eq. NonLinear_Eq, the local coordinates of a
// departure point by Newton's method, the nine second-order Lagrange shape
// functions of Eq. Propagation (s = 1..9), the straight-line element walk
// over quadrilaterals and the element gradients (the kernels of a time step
// on such a mesh are in quad.cu).
//
// Node order of an element: corners v0 (-1,-1), v1 (1,-1), v2 (1,1),
// v3 (-1,1) counter-clockwise, the midside nodes of edges (v0,v1), (v1,v2),
// (v2,v3), (v3,v0), then the centre (0,0).  Edge k runs from v_k to v_k+1.
//
// The exact path: the FP64 departure point, exact orientation signs for the
// walk and the tie rules, Newton in the interpolation's arithmetic; the
// populations are stored and interpolated in the solver's precision.  A
// certified FP32 test of the previous-step element settles most populations
// before it (quad_fast_decide).
#pragma once
#include "geom.cuh"

namespace alelb {

// Index (0, 1, 2 for -1, 0, 1) of local node l's xi and eta.
ALELB_HD __forceinline__ int quad_ix(int l) { return (int)((0x11928u >> (2 * l)) & 3u); }
ALELB_HD __forceinline__ int quad_iy(int l) { return (int)((0x164a0u >> (2 * l)) & 3u); }

// Bilinear map of the corners w (x, y pairs) at (xi, eta), Eq. NonLinear_Eq:
// x = sum_k n_k w_k with n = (1 -+ xi)(1 -+ eta)/4, and its Jacobian
// J = {x_xi, x_eta, y_xi, y_eta}.
ALELB_HD __forceinline__ void quad_bilinear(const double w[8], double xi, double eta, double &x, double &y,
                                            double J[4])
{
    const double n0 = 0.25 * (1.0 - xi) * (1.0 - eta), n1 = 0.25 * (1.0 + xi) * (1.0 - eta);
    const double n2 = 0.25 * (1.0 + xi) * (1.0 + eta), n3 = 0.25 * (1.0 - xi) * (1.0 + eta);
    const double a0 = -0.25 * (1.0 - eta), a1 = 0.25 * (1.0 - eta), a2 = 0.25 * (1.0 + eta), a3 = -0.25 * (1.0 + eta);
    const double b0 = -0.25 * (1.0 - xi), b1 = -0.25 * (1.0 + xi), b2 = 0.25 * (1.0 + xi), b3 = 0.25 * (1.0 - xi);
    x = n0 * w[0] + n1 * w[2] + n2 * w[4] + n3 * w[6];
    y = n0 * w[1] + n1 * w[3] + n2 * w[5] + n3 * w[7];
    J[0] = a0 * w[0] + a1 * w[2] + a2 * w[4] + a3 * w[6];
    J[1] = b0 * w[0] + b1 * w[2] + b2 * w[4] + b3 * w[6];
    J[2] = a0 * w[1] + a1 * w[3] + a2 * w[5] + a3 * w[7];
    J[3] = b0 * w[1] + b1 * w[3] + b2 * w[5] + b3 * w[7];
}

// Newton's method on Eq. NonLinear_Eq for corners c taken relative to the
// point (so the root is x(xi, eta) = 0), in the arithmetic A of the values
// it serves: start at the centre, at most QUAD_NEWTON_ITERS steps, stopping
// once a step is below `done` (quadratic convergence: the next one would be
// below the rounding); converged when the last step is below `tol`.  The
// element choice never depends on it (exact signs decide), only the
// interpolation weights.
constexpr int QUAD_NEWTON_ITERS = 8;
// Whether any lane of `lanes` still iterates: those lanes leave the loop
// together (a lane that has converged keeps its values meanwhile), so that the
// interpolation after it runs once per warp, not once per iteration count
// (kq_fast at 150,400 nodes: 56 us with lanes leaving one by one).  Every lane
// of the mask has to come here, which only the caller can know: it votes for
// the mask before its lanes part (quad_fast_pop).  lanes = 0: the lane is on its
// own, as on the exact path, where the lanes of a warp are at different entries.
ALELB_HD __forceinline__ bool lanes_go(unsigned lanes, bool go)
{
#ifdef __CUDA_ARCH__
    if (lanes) return __any_sync(lanes, go);
#endif
    return go;
}
template <class A>
ALELB_HD __forceinline__ bool quad_newton_t(const A c[8], A done, A tol, A &xi, A &eta, unsigned lanes = 0)
{
    A a = A(0), b = A(0), da = A(0), db = A(0);
    bool go = true;
#pragma unroll 1
    for (int it = 0; it < QUAD_NEWTON_ITERS; ++it) {
        if (go) {
            const A n0 = A(0.25) * (A(1) - a) * (A(1) - b), n1 = A(0.25) * (A(1) + a) * (A(1) - b);
            const A n2 = A(0.25) * (A(1) + a) * (A(1) + b), n3 = A(0.25) * (A(1) - a) * (A(1) + b);
            const A a0 = A(-0.25) * (A(1) - b), a1 = A(0.25) * (A(1) - b), a2 = A(0.25) * (A(1) + b), a3 = -a2;
            const A b0 = A(-0.25) * (A(1) - a), b1 = A(-0.25) * (A(1) + a), b2 = -b1, b3 = -b0;
            const A rx = n0 * c[0] + n1 * c[2] + n2 * c[4] + n3 * c[6];
            const A ry = n0 * c[1] + n1 * c[3] + n2 * c[5] + n3 * c[7];
            const A J0 = a0 * c[0] + a1 * c[2] + a2 * c[4] + a3 * c[6];
            const A J1 = b0 * c[0] + b1 * c[2] + b2 * c[4] + b3 * c[6];
            const A J2 = a0 * c[1] + a1 * c[3] + a2 * c[5] + a3 * c[7];
            const A J3 = b0 * c[1] + b1 * c[3] + b2 * c[5] + b3 * c[7];
            const A inv = A(1) / (J0 * J3 - J1 * J2);
            da = (J3 * rx - J1 * ry) * inv;
            db = (-J2 * rx + J0 * ry) * inv;
            a -= da;
            b -= db;
            go = !(fabs(da) + fabs(db) < done);
        }
        if (!lanes_go(lanes, go)) break;
    }
    xi = a;
    eta = b;
    return fabs(da) <= tol && fabs(db) <= tol;
}
ALELB_HD __forceinline__ bool quad_newton(const double c[8], double &xi, double &eta)
{
    return quad_newton_t<double>(c, 1e-12, 1e-9, xi, eta);
}

// One-dimensional quadratic Lagrange polynomials through -1, 0, 1 and
// their derivatives.
template <class A> ALELB_HD __forceinline__ void lagrange3(A s, A L[3], A dL[3])
{
    L[0] = A(0.5) * s * (s - A(1));
    L[1] = (A(1) - s) * (A(1) + s);
    L[2] = A(0.5) * s * (s + A(1));
    dL[0] = s - A(0.5);
    dL[1] = A(-2) * s;
    dL[2] = s + A(0.5);
}

// N_s(xi, eta) = L_i(xi) L_j(eta) for the nine nodes (Eq. Propagation).
template <class A> ALELB_HD __forceinline__ void shape9(A xi, A eta, A N[9])
{
    A Lx[3], Ly[3], dx[3], dy[3];
    lagrange3(xi, Lx, dx);
    lagrange3(eta, Ly, dy);
#pragma unroll
    for (int s = 0; s < 9; ++s) N[s] = Lx[quad_ix(s)] * Ly[quad_iy(s)];
}

struct QuadDev {
    int N, E;
    double Lx, Ly;
    const double2 *X;      // [N]
    const double2 *ev;     // [4E] corners in each element's frame
    const int *nbr;        // [4E]
    const uint32_t *einfo; // [E] byte k: kind(2) | nbr edge(2) | dsx+1(2) | dsy+1(2)
    const int *rank;       // [E]
    const int *conn;       // [9E]
    const int *fan_ptr;    // [N + 1]
    const int2 *fan;       // (elem, local | (sx+1)<<4 | (sy+1)<<6)
    const int2 *owner;     // (elem, local)
    const int2 *bcel;      // (elem, local): wall-condition gradient element
    const uint8_t *bkind;  // [N]
    const int *wall_idx;   // [N]
    const int *probe_e;    // [NW]
    const double2 *probe_xi; // [NW]
    const double2 *wall_nrm; // [NW]
    const int *orig_elem;  // [E]
    const float4 *Xf;      // [N] node coordinates, FP32 hi + lo
    const float4 *evf;     // [4E] corners, FP32 hi + lo
    const float *bdist;    // [N] lower bound of the distance to the nearest boundary edge
    const float4 *ownJf;   // [N] owner element's J^{-1} at the node, FP32
    const double2 *ownJd;  // [2N] the same in FP64 (grad xi, grad eta)
    const double2 *ebd;    // [5E] bilinear map (QuadTables)
    const float4 *cone;    // [N] boundary node: outgoing, incoming boundary edge (as MeshDev's)
    const uint8_t *conek;  // [N]
    const uint8_t *vzero;  // [N] 1: mesh velocity exactly zero at all times
    int nvzero;            // number of those nodes
};

// The four corners of element e shifted by (sx, sy) periods.
ALELB_HD __forceinline__ void quad_frame(const QuadDev &M, int e, int sx, int sy, double w[8])
{
    const double ox = sx ? sx * M.Lx : 0.0, oy = sy ? sy * M.Ly : 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double2 v = M.ev[4 * e + k];
        w[2 * k] = sx ? v.x + ox : v.x;
        w[2 * k + 1] = sy ? v.y + oy : v.y;
    }
}

ALELB_HD __forceinline__ int quad_fan_best(const QuadDev &M, int v)
{
    int best = -1;
    for (int k = M.fan_ptr[v]; k < M.fan_ptr[v + 1]; ++k) {
        const int e = M.fan[k].x;
        if (best < 0 || M.rank[e] < M.rank[best]) best = e;
    }
    return best;
}

// Location of p in the closed element e, given its signs against the four
// edges: strictly inside; on one edge, then the better-ranked of the two
// elements sharing it (larger area, then lower original id); on a corner,
// which is named.
ALELB_HD __forceinline__ Loc quad_finish(const QuadDev &M, int e, int sx, int sy, const int o[4])
{
    Loc r;
    r.kind = 0;
    r.vnode = -1;
    const int nz = (o[0] == 0) + (o[1] == 0) + (o[2] == 0) + (o[3] == 0);
    if (nz == 1) {
        const int kz = o[0] == 0 ? 0 : o[1] == 0 ? 1 : o[2] == 0 ? 2 : 3;
        const uint32_t inf = (M.einfo[e] >> (8 * kz)) & 255u;
        if ((inf & 3) == 0) {
            const int e2 = M.nbr[4 * e + kz];
            if (M.rank[e2] < M.rank[e]) {
                e = e2;
                sx += (int)((inf >> 4) & 3) - 1;
                sy += (int)((inf >> 6) & 3) - 1;
            }
        }
    } else if (nz >= 2) {
        // the corner shared by two zero edges k, k + 1 is corner k + 1
        int vl = 0;
        for (int k = 0; k < 4; ++k)
            if (o[k] == 0 && o[(k + 1) & 3] == 0) vl = (k + 1) & 3;
        r.vnode = M.conn[9 * e + vl];
    }
    r.e = e;
    r.sx = sx;
    r.sy = sy;
    return r;
}

// Orientation provider of the walk over quadrilaterals: exact FP64 predicates
// on the FP64 departure point and the element frames.
struct QPred64 {
    const QuadDev &M;
    double Xa, Ya, px, py;
    double w[8];
    ALELB_HD void load(int e, int sx, int sy) { quad_frame(M, e, sx, sy, w); }
    ALELB_HD int vvp(int k1, int k2) { return orient(w[2 * k1], w[2 * k1 + 1], w[2 * k2], w[2 * k2 + 1], px, py); }
    ALELB_HD int avp(int k) { return orient(Xa, Ya, px, py, w[2 * k], w[2 * k + 1]); }
    // p, on the line through w_l and w_k, lies on the ray from w_l through w_k
    ALELB_HD bool fwd(int l, int k)
    {
        return (px - w[2 * l]) * (w[2 * k] - w[2 * l]) + (py - w[2 * l + 1]) * (w[2 * k + 1] - w[2 * l + 1]) > 0.0;
    }
    ALELB_HD bool p_is_node() const { return px == Xa && py == Ya; }
};

// The same in FP32 (as Pred32 on triangles): every point relative to the
// node, the departure point from the FP32 c^, the corners from their hi/lo
// splits; a sign that is not certain falls back to the exact predicate on the
// canonical FP64 departure point, computed lazily.  The caller ensures that
// |c^| > 4 F.eq(i), so the departure point is not the node.
struct QPred32 {
    const QuadDev &M;
    const MapStatic &MS;
    const MapScalars &sc;
    int a, i;
    float4 Xf;
    float rpx, rpy, ep;
    int e, sx, sy;
    float x0, x1, x2, x3, y0, y1, y2, y3, e0, e1, e2, e3; // corners relative to the node, error bounds
    bool have64;
    double Xa, Ya, px, py;
    ALELB_HD float RX(int k) const { return k == 0 ? x0 : k == 1 ? x1 : k == 2 ? x2 : x3; }
    ALELB_HD float RY(int k) const { return k == 0 ? y0 : k == 1 ? y1 : k == 2 ? y2 : y3; }
    ALELB_HD float ER(int k) const { return k == 0 ? e0 : k == 1 ? e1 : k == 2 ? e2 : e3; }
    ALELB_HD void corner(int k, float &x, float &y, float &ek) const
    {
        const float u = 5.9604644775390625e-08f;
        const float4 v = M.evf[4 * e + k];
        const float hx = v.x - Xf.x, hy = v.y - Xf.y;
        x = hx + (v.z - Xf.z);
        y = hy + (v.w - Xf.w);
        float sh = 0.0f;
        if (sx) {
            x += (float)sx * (float)M.Lx;
            sh = fabsf((float)M.Lx);
        }
        if (sy) {
            y += (float)sy * (float)M.Ly;
            sh = fmaxf(sh, fabsf((float)M.Ly));
        }
        ek = 4.0f * u * (fmaxf(fabsf(x), fabsf(y)) + fmaxf(fabsf(hx), fabsf(hy)) + sh) + 9.313225746154785e-10f;
    }
    ALELB_HD void load(int e_, int sx_, int sy_)
    {
        e = e_;
        sx = sx_;
        sy = sy_;
        corner(0, x0, y0, e0);
        corner(1, x1, y1, e1);
        corner(2, x2, y2, e2);
        corner(3, x3, y3, e3);
    }
    ALELB_HD void ensure64()
    {
        if (have64) return;
        const double2 X = M.X[a];
        double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22, wx, wy, chx, chy;
        Xa = X.x;
        Ya = X.y;
        map_node(MS, sc, a, Xa, Ya, xX, xY, yX, yY, Vx, Vy);
        metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
        mesh_velocity_term(a11, a12, a21, a22, ds(Vx, sc.Ux), ds(Vy, sc.Uy), false, wx, wy);
        departure(a11, a12, a21, a22, wx, wy, lat_cx(i), lat_cy(i), Xa, Ya, chx, chy, px, py);
        have64 = true;
    }
    ALELB_HD double2 W(int k) const
    {
        double2 v = M.ev[4 * e + k];
        if (sx) v.x = v.x + sx * M.Lx;
        if (sy) v.y = v.y + sy * M.Ly;
        return v;
    }
    ALELB_HD int vvp(int k1, int k2)
    {
        const int s = orient3_f32(RX(k1), RY(k1), ER(k1), RX(k2), RY(k2), ER(k2), rpx, rpy, ep);
        if (s) return s;
        ensure64();
        const double2 p = W(k1), q = W(k2);
        return orient(p.x, p.y, q.x, q.y, px, py);
    }
    ALELB_HD int avp(int k)
    {
        const int s = orient3_f32(0.0f, 0.0f, 0.0f, rpx, rpy, ep, RX(k), RY(k), ER(k));
        if (s) return s;
        ensure64();
        const double2 q = W(k);
        return orient(Xa, Ya, px, py, q.x, q.y);
    }
    ALELB_HD bool fwd(int l, int k)
    {
        ensure64();
        const double2 p = W(l), q = W(k);
        return (px - p.x) * (q.x - p.x) + (py - p.y) * (q.y - p.y) > 0.0;
    }
    ALELB_HD bool p_is_node() const { return false; }
};

// Straight-line walk from node a along the segment X_a -> p over the
// quadrilaterals, with exact orientation signs (the same reading of the
// departure search as on triangles: a line through a vertex passes to the
// vertex's right; a population is missing when the walk leaves the mesh
// through a boundary edge or no element of the node's fan holds the first
// piece of the segment; a segment along a boundary edge stays inside the
// closed mesh).  Exit edges follow from the side of the segment line that
// each corner lies on: the walk leaves a convex cell where the corners
// change from the right of the line to its left, counter-clockwise.
// P supplies the orientation signs, always exact.
template <class P> ALELB_HD __forceinline__ Loc quad_walk_t(const QuadDev &M, P &pr, int a, int *err)
{
    Loc r;
    r.kind = 0;
    r.vnode = -1;
    r.sx = r.sy = 0;
    if (pr.p_is_node()) {
        r.e = quad_fan_best(M, a);
        r.vnode = a;
        return r;
    }
    int e = -1, loc = 0, sx = 0, sy = 0;
    for (int k = M.fan_ptr[a]; k < M.fan_ptr[a + 1]; ++k) {
        const int2 fe = M.fan[k];
        const int ll = fe.y & 15, ssx = ((fe.y >> 4) & 3) - 1, ssy = ((fe.y >> 6) & 3) - 1;
        pr.load(fe.x, ssx, ssy);
        bool hit;
        if (ll < 4) { // corner: the sector between rays ll -> ll+1 and ll -> ll+3
            const int k1 = (ll + 1) & 3, k3 = (ll + 3) & 3;
            hit = pr.vvp(ll, k1) >= 0;
            if (hit) {
                const int s3 = pr.vvp(ll, k3);
                // along the incoming boundary edge: no other element holds that ray
                hit = s3 < 0 || (s3 == 0 && ((M.einfo[fe.x] >> (8 * k3)) & 3u) && pr.fwd(ll, k3));
            }
        } else if (ll < 8) { // midside node of edge ll - 4: the element's half-plane
            const int k0 = ll - 4, k1 = (k0 + 1) & 3;
            hit = pr.vvp(k0, k1) >= 0;
        } else { // the centre: strictly inside
            hit = true;
        }
        if (hit) {
            e = fe.x;
            loc = ll;
            sx = ssx;
            sy = ssy;
            break;
        }
    }
    if (e < 0) {
        if (!M.bkind[a]) {
            set_err(err, ERR_LOCATE);
            r.e = -2;
            return r;
        }
        r.e = -1;
        r.kind = M.bkind[a];
        return r;
    }
    pr.load(e, sx, sy);
    int o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = pr.vvp(k, (k + 1) & 3);
    if (o[0] >= 0 && o[1] >= 0 && o[2] >= 0 && o[3] >= 0) return quad_finish(M, e, sx, sy, o);
    // side of the segment line of corner k: >= 0 left (or on it), < 0 right
    auto side = [&](int k) { return pr.avp(k); };
    int kout;
    if (loc < 4) {
        kout = side((loc + 2) & 3) >= 0 ? (loc + 1) & 3 : (loc + 2) & 3;
    } else if (loc < 8) {
        const int k0 = loc - 4;
        kout = side((k0 + 2) & 3) >= 0 ? (k0 + 1) & 3 : side((k0 + 3) & 3) >= 0 ? (k0 + 2) & 3 : (k0 + 3) & 3;
    } else {
        int sd[4];
        for (int k = 0; k < 4; ++k) sd[k] = side(k);
        kout = 0;
        for (int k = 0; k < 4; ++k)
            if (sd[k] < 0 && sd[(k + 1) & 3] >= 0) kout = k;
    }
#pragma unroll 1
    for (int step = 0; step < WALK_LIMIT; ++step) {
        const uint32_t inf = (M.einfo[e] >> (8 * kout)) & 255u;
        const int kind = inf & 3;
        if (kind) {
            r.e = -1;
            r.kind = kind;
            return r;
        }
        const int kin = (inf >> 2) & 3;
        sx += (int)((inf >> 4) & 3) - 1;
        sy += (int)((inf >> 6) & 3) - 1;
        e = M.nbr[4 * e + kout];
        pr.load(e, sx, sy);
        bool in = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) { // kin was crossed from outside: p lies strictly on its inner side
            o[k] = k == kin ? 1 : pr.vvp(k, (k + 1) & 3);
            in = in && o[k] >= 0;
        }
        if (in) return quad_finish(M, e, sx, sy, o);
        kout = side((kin + 2) & 3) >= 0 ? (kin + 1) & 3 : side((kin + 3) & 3) >= 0 ? (kin + 2) & 3 : (kin + 3) & 3;
    }
    set_err(err, ERR_LOCATE);
    r.e = -2;
    return r;
}

ALELB_HD inline Loc quad_walk(const QuadDev &M, int a, double Xa, double Ya, double px, double py, int *err)
{
    QPred64 pr{M, Xa, Ya, px, py, {}};
    return quad_walk_t(M, pr, a, err);
}

// The certified FP32 decision of the deviation forms for population i of
// node a: its previous-step element (cache code c, unshifted) holds the FP64
// departure point strictly inside -- four orientation signs certified in
// FP32 against their error bounds (the departure offset -c^ carries F.eq(i)
// per component, the node-relative corners their hi/lo rounding) -- and the
// segment from the node cannot leave the mesh: the cell is one of the
// node's own (convex, it holds both ends) or the segment is shorter than
// the node's distance to any boundary.  The oracle's exhaustive search
// then picks the same cell: a point strictly inside one cell lies in no
// other.  On success cw holds the corners relative to the departure point
// (FP32) for Newton.
ALELB_HD __forceinline__ bool quad_fast_decide(const QuadDev &M, const FastMap &F, float4 Xf, int a, int i, int c,
                                               int &e, float cw[8])
{
    if (!F.ok || c < 0 || (c >> 28) != 5) return false;
    const float u = 5.9604644775390625e-08f;
    const float cx = (float)lat_cx(i), cy = (float)lat_cy(i);
    const float chx = F.A11 * cx + F.A12 * cy - F.W1;
    const float chy = F.A21 * cx + F.A22 * cy - F.W2;
    const float eq = F.eq(i);
    const float len2 = chx * chx + chy * chy;
    const float q4 = 4.0f * eq;
    if (!(len2 > q4 * q4)) return false;
    e = c & CACHE_ELEM;
    bool own = false;
#pragma unroll
    for (int k = 0; k < 9; ++k) own = own || M.conn[9 * e + k] == a;
    const float room = M.bdist[a] - eq;
    if (!(own | ((room > 0.0f) & (len2 < room * room)))) return false;
    const float px = -chx, py = -chy;
    float rx[4], ry[4], er[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 v = M.evf[4 * e + k];
        const float hx = v.x - Xf.x, hy = v.y - Xf.y;
        rx[k] = hx + (v.z - Xf.z);
        ry[k] = hy + (v.w - Xf.w);
        er[k] = 4.0f * u * (fmaxf(fabsf(rx[k]), fabsf(ry[k])) + fmaxf(fabsf(hx), fabsf(hy))) + 9.313225746154785e-10f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int k1 = (k + 1) & 3;
        if (orient3_f32(rx[k], ry[k], er[k], rx[k1], ry[k1], er[k1], px, py, eq) <= 0) return false;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        cw[2 * k] = rx[k] - px;
        cw[2 * k + 1] = ry[k] - py;
    }
    return true;
}

// Local coordinates of p in element e (frame shift sx, sy) by Newton, in
// the arithmetic A of the interpolation (the corners relative to p are
// formed in FP64, then rounded to A).
template <class A>
ALELB_HD __forceinline__ bool quad_local(const QuadDev &M, int e, int sx, int sy, double px, double py, A &xi,
                                         A &eta)
{
    double w[8];
    quad_frame(M, e, sx, sy, w);
    A c[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        c[2 * k] = (A)(w[2 * k] - px);
        c[2 * k + 1] = (A)(w[2 * k + 1] - py);
    }
    if (sizeof(A) == 8) return quad_newton_t<A>(c, A(1e-12), A(1e-9), xi, eta);
    return quad_newton_t<A>(c, A(1e-5), A(1e-4), xi, eta); // FP32: converged near 1e-7
}

// The corners of element e (frame shift sx, sy) relative to the FP64 point p,
// as FP32 numbers: the shift is taken from p in FP64, then the leading and the
// trailing parts (corner and point split in two FP32 numbers each) are
// subtracted, the former exactly, so that one rounding remains (quad_local's
// FP32 corners in eight FP64 subtractions and conversions less).
ALELB_HD __forceinline__ void quad_corners32(const QuadDev &M, int e, int sx, int sy, double px, double py, float c[8])
{
    if (sx) px = px - sx * M.Lx;
    if (sy) py = py - sy * M.Ly;
    const float hx = (float)px, hy = (float)py;
    const float lx = (float)(px - (double)hx), ly = (float)(py - (double)hy);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 v = M.evf[4 * e + k];
        c[2 * k] = (v.x - hx) + (v.z - lx);
        c[2 * k + 1] = (v.y - hy) + (v.w - ly);
    }
}

// FP64 <-> FP32 by their bits, for values whose rounding does not matter
// (the FP64 pipe runs conversions at its own low rate): truncation toward
// zero, below the normal range to zero, above it to the largest float.
ALELB_HD __forceinline__ float d2f_bits(double v)
{
#ifdef __CUDA_ARCH__
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
#else
    unsigned long long w;
    std::memcpy(&w, &v, 8);
    const unsigned hi = (unsigned)(w >> 32), lo = (unsigned)w;
#endif
    const unsigned m = hi & 0x7fffffffu;
    unsigned b = ((m - 0x38000000u) << 3) | (lo >> 29);
    if (m < 0x38100000u) b = 0u;
    if (m >= 0x47f00000u) b = 0x7f7fffffu;
    b |= hi & 0x80000000u;
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    std::memcpy(&f, &b, 4);
    return f;
#endif
}

// Local coordinates of p in element e for the FP64 form: Newton in FP32 on
// the bilinear map x = w0 + c + b1 xi + b2 eta + b3 xi eta, then corrections
// with the residual in FP64 and the FP32 inverse Jacobian.  A correction leaves
// a part k of the error it finds: the FP32 rounding of the Jacobian, 2^-20 in
// cells near a parallelogram of moderate aspect, more by the aspect ratio in
// thin cells oblique to the axes (1e-3 at 1e4).  The last two corrections give
// it, k = last / before, so what the last one leaves is last^2 / before: after
// two, more are made while that is above 2^-54 (none on the O-meshes and boxes;
// 2^-52: the rounding of the coordinates).  The residual is formed from the
// point relative to a corner, exact nearby, by fused operations; a correction
// costs 9 operations of the FP64 pipe, against about 60 for a Newton step in
// FP64.  The error against extended precision is that of Newton's method in FP64
// on the corners relative to p: in the quadratic mean over the cells 4.1e-17
// (Newton 6.4e-17) on a jittered box, 5.5e-17 (7.4e-17) on the 150k O-mesh,
// 8.6e-17 (9.1e-17) on one of 64 x 20 cells; at most 1.7e-16 (2.6e-16), 2.0e-15
// (1.1e-15), 3.9e-15 (3.0e-15).  The rounding of every operation is pinned, so
// the result is the same in every kernel.  false: the corrections did not settle
// (the last one above 1e-9), or the cell's area is beyond FP32 (an inverse of
// zero would leave any point settled).
constexpr int QUAD_CORRECTIONS = 4;
ALELB_HD __forceinline__ bool quad_local64(const QuadDev &M, int e, int sx, int sy, double px, double py,
                                           double &xi, double &eta, unsigned lanes = 0)
{
    double2 w0 = M.ebd[5 * e];
    const double2 b1 = M.ebd[5 * e + 1], b2 = M.ebd[5 * e + 2], b3 = M.ebd[5 * e + 3], c = M.ebd[5 * e + 4];
    if (sx) w0.x = da(w0.x, sx * M.Lx);
    if (sy) w0.y = da(w0.y, sy * M.Ly);
    const double dx = ds(ds(px, w0.x), c.x), dy = ds(ds(py, w0.y), c.y);
    const float fx = d2f_bits(dx), fy = d2f_bits(dy);
    const float b1x = d2f_bits(b1.x), b1y = d2f_bits(b1.y), b2x = d2f_bits(b2.x), b2y = d2f_bits(b2.y),
                b3x = d2f_bits(b3.x), b3y = d2f_bits(b3.y);
    float u = 0.f, v = 0.f, i11 = 0.f, i12 = 0.f, i21 = 0.f, i22 = 0.f, inv = 0.f;
    const auto inverse = [&]() { // J^{-1} at (u, v)
        const float j11 = ffma(b3x, v, b1x), j12 = ffma(b3x, u, b2x);
        const float j21 = ffma(b3y, v, b1y), j22 = ffma(b3y, u, b2y);
        inv = frcp(ffma(j11, j22, -fm(j12, j21)));
        i11 = fm(j22, inv);
        i12 = -fm(j12, inv);
        i21 = -fm(j21, inv);
        i22 = fm(j11, inv);
    };
    bool go = true;
#pragma unroll 1
    for (int it = 0; it < QUAD_NEWTON_ITERS; ++it) {
        if (go) {
            inverse();
            const float uv = fm(u, v);
            const float rx = fa(fx, -ffma(b3x, uv, ffma(b2x, v, fm(b1x, u))));
            const float ry = fa(fy, -ffma(b3y, uv, ffma(b2y, v, fm(b1y, u))));
            const float du = ffma(i11, rx, fm(i12, ry)), dv = ffma(i21, rx, fm(i22, ry));
            u = fa(u, du);
            v = fa(v, dv);
            go = !(fabsf(du) + fabsf(dv) < 1e-4f); // the next step would be below the FP32 rounding
        }
        if (!lanes_go(lanes, go)) break;
    }
    inverse();
    xi = f2d_bits(u);
    eta = f2d_bits(v);
    float last = 0.f, left = 0.f; // the last correction, what it leaves
    const auto correct = [&]() {
        const double q = dm(xi, eta);
        const float rx = d2f_bits(dfma(-b3.x, q, dfma(-b2.x, eta, dfma(-b1.x, xi, dx))));
        const float ry = d2f_bits(dfma(-b3.y, q, dfma(-b2.y, eta, dfma(-b1.y, xi, dy))));
        const float du = ffma(i11, rx, fm(i12, ry)), dv = ffma(i21, rx, fm(i22, ry));
        const float before = last;
        xi = da(xi, f2d_bits(du));
        eta = da(eta, f2d_bits(dv));
        last = fabsf(du) + fabsf(dv); // (a sum, so that one that is not a number stays so)
        left = fm(last, last) - fm(5.5511151231257827e-17f, before); // 2^-54
    };
    correct();
    correct();
#pragma unroll 1
    for (int it = 2; it < QUAD_CORRECTIONS && !(left <= 0.f || last <= 2.220446049250313e-16f); ++it) correct();
    return last <= 1e-9f && inv != 0.f;
}

// The pair (f_i, g_i) of the FP64 form interpolated at (xi, eta) of element
// e: the nine shape functions are products of one-dimensional ones, so three
// sums along xi and one along eta (24 operations of the FP64 pipe for the two
// fields, against 27 for nine weights and their sums); the one-dimensional
// functions are (xi^2 -+ xi)/2 and 1 - xi^2, four operations each direction.
__device__ __forceinline__ void quad_interp64(const QuadDev &M, const double *post, int N, int i, int e, double xi,
                                              double eta, double &f, double &g)
{
    int nb[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) nb[k] = M.conn[9 * e + k];
    const double hx = scale2_bits(xi, -1), hy = scale2_bits(eta, -1), x2 = dm(xi, xi), y2 = dm(eta, eta);
    const double sx = scale2_bits(x2, -1), sy = scale2_bits(y2, -1);
    const double lx[3] = {ds(sx, hx), ds(1.0, x2), da(sx, hx)};
    const double ly[3] = {ds(sy, hy), ds(1.0, y2), da(sy, hy)};
    constexpr int at[3][3] = {{0, 4, 1}, {7, 8, 5}, {3, 6, 2}}; // local node at (i, j), row j along xi
    f = 0.0;
    g = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        double rf = 0.0, rg = 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int b = nb[at[j][q]];
            const double fb = post[i * N + b], gb = post[(NQ + i) * N + b];
            rf = q ? dfma(lx[q], fb, rf) : dm(lx[q], fb);
            rg = q ? dfma(lx[q], gb, rg) : dm(lx[q], gb);
        }
        f = j ? dfma(ly[j], rf, f) : dm(ly[j], rf);
        g = j ? dfma(ly[j], rg, g) : dm(ly[j], rg);
    }
}

// d K / d X at node a in element el = (elem, local): the nine-node
// derivative (Eq. FE_Derivative in the owner element), with J^{-1} of the
// bilinear map at the node's local position (the wall forces).
template <class S>
__device__ __forceinline__ void quad_grad(const QuadDev &M, int2 el, const S *K, double &KX, double &KY)
{
    const int e = el.x, l = el.y;
    const double xi = quad_ix(l) - 1.0, eta = quad_iy(l) - 1.0;
    double w[8], x, y, J[4];
    quad_frame(M, e, 0, 0, w);
    quad_bilinear(w, xi, eta, x, y, J);
    double sxi = 0.0, seta = 0.0;
    double Lx[3], Ly[3], dx[3], dy[3];
    lagrange3(xi, Lx, dx);
    lagrange3(eta, Ly, dy);
#pragma unroll
    for (int s = 0; s < 9; ++s) {
        const double Ks = (double)K[M.conn[9 * e + s]];
        sxi += Ks * (dx[quad_ix(s)] * Ly[quad_iy(s)]);
        seta += Ks * (Lx[quad_ix(s)] * dy[quad_iy(s)]);
    }
    const double det = J[0] * J[3] - J[2] * J[1];
    KX = (J[3] * sxi - J[2] * seta) / det;
    KY = (-J[1] * sxi + J[0] * seta) / det;
}

// Gradients of three node fields at node a's position in element el, of the
// bilinear interpolants of the corner values (the first-order gradients of the
// wall condition): one Jacobian for the three, its coefficients from the
// element's table.  G[2 f], G[2 f + 1]: d K_f / d X, d K_f / d Y.
template <class S>
__device__ __forceinline__ void quad_grad3_linear(const QuadDev &M, int2 el, const S *K0, const S *K1, const S *K2,
                                                  double G[6])
{
    const int e = el.x, l = el.y;
    const int ix = quad_ix(l) - 1, iy = quad_iy(l) - 1;
    const double xi = ix < 0 ? -1.0 : ix ? 1.0 : 0.0, eta = iy < 0 ? -1.0 : iy ? 1.0 : 0.0;
    const double2 b1 = M.ebd[5 * e + 1], b2 = M.ebd[5 * e + 2], b3 = M.ebd[5 * e + 3];
    const double jxx = b1.x + b3.x * eta, jxe = b2.x + b3.x * xi, jyx = b1.y + b3.y * eta, jye = b2.y + b3.y * xi;
    const double inv = 1.0 / (jxx * jye - jyx * jxe);
    int nb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) nb[k] = M.conn[9 * e + k];
    const S *const Ks[3] = {K0, K1, K2};
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        const double k0 = (double)Ks[f][nb[0]], k1 = (double)Ks[f][nb[1]], k2 = (double)Ks[f][nb[2]],
                     k3 = (double)Ks[f][nb[3]];
        // the interpolant's coefficients, as the map's: c1 + c3 eta and c2 + c3 xi
        const double u = k1 - k0, w = k2 - k3, c3 = 0.25 * (w - u);
        const double sxi = 0.25 * (u + w) + c3 * eta, seta = 0.25 * ((k3 - k0) + (k2 - k1)) + c3 * xi;
        G[2 * f] = (jye * sxi - jyx * seta) * inv;
        G[2 * f + 1] = (-jxe * sxi + jxx * seta) * inv;
    }
}

} // namespace alelb

namespace alelb {

// Local node at grid position (i, j) of the 3 x 3 node lattice of an
// element (i along xi, j along eta; 0, 1, 2 for -1, 0, 1): 4-bit fields of
// one word, row j = 0 first (a run-time index into a constant array would
// put the array in local memory).
ALELB_HD __forceinline__ int quad_node_at(int i, int j)
{
    return (int)((0x263587140ull >> (4 * (3 * j + i))) & 15ull);
}

// d K / d X at node a in its owner element (Eq. FE_Derivative), in the
// arithmetic of the form (float, or double for FP64 fields): at a node the
// nine shape functions' xi derivatives vanish off the node's eta row and
// their eta derivatives off its xi column, so each derivative is a three-term
// sum; dL_m at the node's coordinate t in {-1, 0, 1} is t - 1/2, -2 t, t + 1/2
// (exact).
template <class S> struct QuadJ;
template <> struct QuadJ<float> {
    static __device__ __forceinline__ void get(const QuadDev &M, int a, float J[4])
    {
        const float4 v = M.ownJf[a];
        J[0] = v.x;
        J[1] = v.y;
        J[2] = v.z;
        J[3] = v.w;
    }
};
template <> struct QuadJ<double> {
    static __device__ __forceinline__ void get(const QuadDev &M, int a, double J[4])
    {
        const double2 p = M.ownJd[2 * a], q = M.ownJd[2 * a + 1];
        J[0] = p.x;
        J[1] = p.y;
        J[2] = q.x;
        J[3] = q.y;
    }
};
template <class S>
__device__ __forceinline__ void quad_owner_grad(const QuadDev &M, int a, const S *K, S &KX, S &KY)
{
    const int2 ow = M.owner[a];
    const int e = ow.x, l = ow.y;
    const int li = quad_ix(l), lj = quad_iy(l);
    const int *cn = M.conn + 9 * e;
    // the three weights by selection (t = li - 1): no FP64 conversion
    const auto w0 = [](int c) { return c == 0 ? S(-1.5) : c == 1 ? S(-0.5) : S(0.5); };
    const auto w1 = [](int c) { return c == 0 ? S(2) : c == 1 ? S(0) : S(-2); };
    const auto w2 = [](int c) { return c == 0 ? S(-0.5) : c == 1 ? S(0.5) : S(1.5); };
    const S sxi = w0(li) * K[cn[quad_node_at(0, lj)]] + w1(li) * K[cn[quad_node_at(1, lj)]] +
                  w2(li) * K[cn[quad_node_at(2, lj)]];
    const S seta = w0(lj) * K[cn[quad_node_at(li, 0)]] + w1(lj) * K[cn[quad_node_at(li, 1)]] +
                   w2(lj) * K[cn[quad_node_at(li, 2)]];
    S J[4];
    QuadJ<S>::get(M, a, J);
    KX = sxi * J[0] + seta * J[2];
    KY = sxi * J[1] + seta * J[3];
}

} // namespace alelb
