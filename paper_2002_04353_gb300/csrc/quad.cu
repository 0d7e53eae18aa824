// quad.cu -- one time step on a mesh of the paper's 9-node quadrilaterals
// (Sec. III), the element-choice report and the wall forces, plus the upload
// of the mesh tables.  The kinetic model (equilibria, collision, Grad-type
// missing populations) is the one the triangles use (kinetic.cuh); only the
// geometry differs: the walk over quadrilaterals, Newton's method for the
// local coordinates of Eq. NonLinear_Eq, the nine shape functions of
// Eq. Propagation and the element gradients (quad.cuh).  Every form first
// tries the previous-step element under a certified FP32 test
// (quad_fast_decide); the other populations take the exact FP64 path.  The
// FP64 form at 150,400 nodes (plunge): 145 + 40 us for the two passes against
// 3,881 us with every population walked and Newton in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "internal.h"

namespace alelb {
namespace {

// Population i of node a by the certified FP32 decision of the deviation
// forms: its previous-step element, accepted by quad_fast_decide, Newton in
// FP32, the nine-node interpolation.  False: left to the exact path.
template <class S, class A>
__device__ __forceinline__ bool quad_fast_pop(const QuadDev &M, const FastMap &F, float4 Xf, const StateDev<S> &st,
                                              int a, int i, unsigned lanes)
{
    const int N = M.N;
    const int c = st.cache[i * N + a];
    int e = 0;
    float cw[8];
    float xi, eta;
    bool in = quad_fast_decide(M, F, Xf, a, i, c, e, cw);
    const unsigned newton = __ballot_sync(lanes, in); // the lanes that iterate together
    if (in) in = quad_newton_t<float>(cw, 1e-5f, 1e-4f, xi, eta, newton);
    __syncwarp(lanes);
    if (!in) return false;
    A Nw[9];
    shape9<A>((A)xi, (A)eta, Nw);
    A fi = 0, gi = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int b = M.conn[9 * e + k];
        A fb, gb;
        fg_get(st.post, i, b, N, fb, gb);
        fi += Nw[k] * fb;
        gi += Nw[k] * gb;
    }
    fg_put(st.str, i, a, N, fi, gi);
    return true;
}

// The FP64 form's population: the same certified decision, then departure
// point, local coordinates and interpolation in FP64.
template <bool TR>
__device__ __forceinline__ bool quad_fast_pop64(const QuadDev &M, const FastMap &F, const Node64 &n, float4 Xf, double2 X,
                                                const StateDev<double> &st, int a, int i, int c, unsigned lanes,
                                                const DepTab &D)
{
    int e = 0;
    float cw[8];
    double px, py, xi, eta, f, g;
    bool in = quad_fast_decide(M, F, Xf, a, i, c, e, cw);
    const unsigned newton = __ballot_sync(lanes, in);
    if (in) {
        if (TR) {
            const double2 cw = D.c[i];
            px = ds(X.x, cw.x);
            py = ds(X.y, cw.y);
        } else {
            departure64<TR>(n, i, X, px, py);
        }
        in = quad_local64(M, e, 0, 0, px, py, xi, eta, newton);
    }
    __syncwarp(lanes);
    if (!in) return false;
    quad_interp64(M, st.post, M.N, i, e, xi, eta, f, g);
    fg_put(st.str, i, a, M.N, f, g);
    return true;
}

// Missing populations of Sec. IV.A at node a (all nine directions), from its
// metrics and mesh velocity at the arrival time.
template <class S, class A>
__device__ __forceinline__ void quad_missing(const QuadDev &M, const KinParams<A> &K, const StateDev<S> &st, int a,
                                             double a11, double a12, double a21, double a22, double Vx, double Vy,
                                             A fm[NQ], A gm[NQ])
{
    A rt, uxt, uyt, Tt;
    const int wi = M.wall_idx[a];
    if (wi >= 0) { // wall node: u = V_G, rho and T at the probe B
        const int pe = M.probe_e[wi];
        const double2 pxi = M.probe_xi[wi];
        A Nw[9];
        shape9<A>((A)pxi.x, (A)pxi.y, Nw);
        A r = 0, t = 0, ub = 0, vb = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int b = M.conn[9 * pe + k];
            r += Nw[k] * (A)st.rho[b];
            t += Nw[k] * (A)st.T[b];
            if (K.flags & FLAG_SLIP) {
                ub += Nw[k] * (A)st.ux[b];
                vb += Nw[k] * (A)st.uy[b];
            }
        }
        rt = r;
        Tt = t;
        uxt = (A)Vx;
        uyt = (A)Vy;
        if (K.flags & FLAG_SLIP) {
            const double2 nw = M.wall_nrm[wi];
            slip_target<A>((A)a11, (A)a12, (A)a21, (A)a22, (A)nw.x, (A)nw.y, ub, vb, (A)Vx, (A)Vy, uxt, uyt);
        }
    } else { // off-wall node: its previous-step fields (mesh velocity under R8c)
        const bool vg = (K.flags & FLAG_OFFWALL_VG) != 0;
        rt = (A)st.rho[a];
        uxt = vg ? (A)Vx : (A)st.ux[a];
        uyt = vg ? (A)Vy : (A)st.uy[a];
        Tt = (A)st.T[a];
    }
    A du[4] = {0, 0, 0, 0}, dT[2] = {0, 0};
    if (!(K.flags & FLAG_BC_EQ) && !((K.flags & FLAG_SLIP) && wi >= 0)) {
        double G[6];
        quad_grad3_linear(M, M.bcel[a], st.ux, st.uy, st.T, G);
        du[0] = (A)(a11 * G[0] + a21 * G[1]);
        du[1] = (A)(a12 * G[0] + a22 * G[1]);
        du[2] = (A)(a11 * G[2] + a21 * G[3]);
        du[3] = (A)(a12 * G[2] + a22 * G[3]);
        dT[0] = (A)(a11 * G[4] + a21 * G[5]);
        dT[1] = (A)(a12 * G[4] + a22 * G[5]);
    }
    grad_missing(K, rt, uxt, uyt, Tt, du, dT, fm, gm);
}
// The same with the map evaluated, the directions in mask written.
template <class S, class A>
__device__ __forceinline__ void quad_bc_node(const QuadDev &M, const MapStatic &MS, const MapScalars &sc,
                                             const KinParams<A> &K, const StateDev<S> &st, int a, unsigned mask)
{
    const double2 X = M.X[a];
    double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22;
    map_node(MS, sc, a, X.x, X.y, xX, xY, yX, yY, Vx, Vy);
    if (uniform_metric(MS.kind)) {
        a11 = sc.A11;
        a12 = sc.A12;
        a21 = sc.A21;
        a22 = sc.A22;
    } else {
        metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
    }
    A fm[NQ], gm[NQ];
    quad_missing(M, K, st, a, a11, a12, a21, a22, Vx, Vy, fm, gm);
#pragma unroll
    for (int i = 0; i < NQ; ++i)
        if (mask >> i & 1u) fg_put(st.str, i, a, M.N, fm[i], gm[i]);
}

// Propagation of population pairs i0 .. i0 + G - 1 of node a on the exact
// path (Eq. Propagation over the nine nodes of the departure element) and,
// for those that are missing, the condition of Sec. IV.A.  KEEP: the element
// is kept for the next step's certified check.  The moments, Q'_aaa and
// mu/(rho T) follow in k_moments, as on triangles.
// Returns the number of element walks taken.
template <int G, bool KEEP, class S, class A>
__device__ __forceinline__ unsigned quad_stream_pops(const QuadDev &M, const MapStatic &MS, const MapScalars &sc,
                                                     const MapScalars &scd, const KinParams<A> &K,
                                                     const StateDev<S> &st, int *err, int a, int i0)
{
    const int N = M.N;
    const double2 Xa = M.X[a];
    bool have64 = false;
    double a11 = 0, a12 = 0, a21 = 0, a22 = 0, wx = 0, wy = 0, Vx = 0, Vy = 0;
    int miss = 0, far = 0;
    unsigned walks = 0;
#pragma unroll 1
    for (int i = i0; i < i0 + G; ++i) {
        A fi = 0, gi = 0;
        int src = -1;
        if (!have64 && !(K.flags & FLAG_EXACT_CHAR)) {
            double xX, xY, yX, yY;
            map_node(MS, scd, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
            metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
            mesh_velocity_term(a11, a12, a21, a22, ds(Vx, scd.Ux), ds(Vy, scd.Uy), (K.flags & FLAG_LITERAL_VG) != 0,
                               wx, wy);
            have64 = true;
        }
        double chx, chy, px, py;
        if (K.flags & FLAG_EXACT_CHAR)
            exact_departure(MS, sc, scd, (double)c_cx[i], (double)c_cy[i], Xa.x, Xa.y, chx, chy, px, py);
        else
            departure(a11, a12, a21, a22, wx, wy, (double)c_cx[i], (double)c_cy[i], Xa.x, Xa.y, chx, chy, px, py);
        if (chx == 0.0 && chy == 0.0) {
            src = a;
        } else {
            ++walks;
            const Loc L = quad_walk(M, a, Xa.x, Xa.y, px, py, err);
            if (KEEP) // the element for the next step's certified check
                st.cache[i * N + a] = L.e >= 0 ? (L.e | ((L.sx + 1) << 28) | ((L.sy + 1) << 30)) : -1;
            if (L.e == -2) {
                src = a;
            } else if (L.e == -1) {
                miss |= 1 << i;
                if (L.kind == 2) far |= 1 << i;
                continue;
            } else if (L.vnode >= 0) {
                src = L.vnode;
            } else {
                if constexpr (std::is_same<S, double>::value) {
                    double xi, eta;
                    if (!quad_local64(M, L.e, L.sx, L.sy, px, py, xi, eta) &&
                        !quad_local<double>(M, L.e, L.sx, L.sy, px, py, xi, eta))
                        set_err(err, ERR_LOCATE);
                    quad_interp64(M, st.post, N, i, L.e, xi, eta, fi, gi);
                } else {
                    A xi, eta;
                    if (!quad_local<A>(M, L.e, L.sx, L.sy, px, py, xi, eta)) set_err(err, ERR_LOCATE);
                    A Nw[9];
                    shape9<A>(xi, eta, Nw);
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        const int b = M.conn[9 * L.e + k];
                        A fb, gb;
                        fg_get(st.post, i, b, N, fb, gb);
                        fi += Nw[k] * fb;
                        gi += Nw[k] * gb;
                    }
                }
            }
        }
        if (src >= 0) fg_get(st.post, i, src, N, fi, gi);
        fg_put(st.str, i, a, N, fi, gi);
    }

    if (miss) {
        if (!have64 || (K.flags & FLAG_MIDPOINT)) { // the wall condition's map: arrival time
            double xX, xY, yX, yY;
            map_node(MS, sc, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
            metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
        }
        A fm[NQ], gm[NQ];
        if (miss & ~far) {
            quad_missing(M, K, st, a, a11, a12, a21, a22, Vx, Vy, fm, gm);
        }
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            if (!(miss >> i & 1)) continue;
            const A fi = (far >> i & 1) ? K.finf[i] : fm[i];
            const A gi = (far >> i & 1) ? K.ginf[i] : gm[i];
            fg_put(st.str, i, a, N, fi, gi);
        }
    }
    return walks;
}

// The departure point of population i of node a; a translation spares the map's
// chain of operations (150,400 nodes: 1,534 us against 1,560 per 20 FP32 steps,
// 1,489 against 1,498 per 5 FP64 steps).
__device__ __forceinline__ void quad_departure64(const MapStatic &MS, const MapScalars &scd, int a, int i, double2 X,
                                                 double &px, double &py)
{
    if (MS.kind == MK_NONE || MS.kind == MK_PLUNGE)
        departure64<true>(node64<true>(MS, scd, a, X, false), i, X, px, py);
    else
        departure64<false>(node64<false>(MS, scd, a, X, false), i, X, px, py);
}

// Population i of node a on the exact path, its walk on certified FP32
// predicates: location, interpolation, far-field or wall condition.  Returns
// the number of walks (0: c^ is exactly zero).  Where no FP32 map is usable the
// FP64 departure point is walked (quad_stream_pops).
template <class S, class A>
__device__ __forceinline__ unsigned quad_slow_pop(const QuadDev &M, const MapStatic &MS, const MapScalars &sc,
                                                  const MapScalars &scd, const MapScalarsF &sfd, const KinParams<A> &K,
                                                  const StateDev<S> &st, int *err, int a, int i)
{
    const int N = M.N;
    prefetch_l1(M.X + a);
    prefetch_l1(M.fan_ptr + a);
    prefetch_l1(M.wall_idx + a);
    const float4 Xf = M.Xf[a];
    const FastMap F = fast_map(MS, sfd, a, Xf);
    const float cx = (float)lat_cx(i), cy = (float)lat_cy(i);
    const float chx = F.A11 * cx + F.A12 * cy - F.W1;
    const float chy = F.A21 * cx + F.A22 * cy - F.W2;
    if ((K.flags & (FLAG_LITERAL_VG | FLAG_EXACT_CHAR)) || !F.ok || !(sqrtf(chx * chx + chy * chy) > 4.0f * F.eq(i)))
        return quad_stream_pops<1, true>(M, MS, sc, scd, K, st, err, a, i);
    QPred32 pr{M, MS, scd, a, i, Xf, -chx, -chy, F.eq(i)};
    pr.have64 = false;
    const Loc L = quad_walk_t(M, pr, a, err);
    st.cache[i * N + a] = L.e >= 0 ? (L.e | ((L.sx + 1) << 28) | ((L.sy + 1) << 30)) : -1;
    if (L.e == -1) {
        if (L.kind == 2) fg_put(st.str, i, a, N, K.finf[i], K.ginf[i]);
        else quad_bc_node(M, MS, sc, K, st, a, 1u << i);
        return 1u;
    }
    A fi = 0, gi = 0;
    if (L.e == -2 || L.vnode >= 0) {
        fg_get(st.post, i, L.e == -2 ? a : L.vnode, N, fi, gi);
    } else if constexpr (std::is_same<S, double>::value) {
        const double2 X = M.X[a];
        double px, py, xi, eta;
        quad_departure64(MS, scd, a, i, X, px, py);
        if (!quad_local64(M, L.e, L.sx, L.sy, px, py, xi, eta) &&
            !quad_local<double>(M, L.e, L.sx, L.sy, px, py, xi, eta))
            set_err(err, ERR_LOCATE);
        quad_interp64(M, st.post, N, i, L.e, xi, eta, fi, gi);
    } else {
        const double2 X = M.X[a];
        double px, py;
        quad_departure64(MS, scd, a, i, X, px, py);
        float c[8];
        quad_corners32(M, L.e, L.sx, L.sy, px, py, c);
        float xi, eta;
        if (!quad_newton_t<float>(c, 1e-5f, 1e-4f, xi, eta)) set_err(err, ERR_LOCATE);
        A Nw[9];
        shape9<A>((A)xi, (A)eta, Nw);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            A fb, gb;
            fg_get(st.post, i, M.conn[9 * L.e + k], N, fb, gb);
            fi += Nw[k] * fb;
            gi += Nw[k] * gb;
        }
    }
    fg_put(st.str, i, a, N, fi, gi);
    return 1u;
}

// Grid (node blocks, 9 / G direction groups): G directions per thread.
template <class S, class A, int G>
__global__ void __launch_bounds__(128) kq_stream(QuadDev M, MapStatic MS, MapScalars sc, MapScalars scd,
                                                 KinParams<A> K, StateDev<S> st, int *err,
                                                 unsigned long long *stats)
{
    wait_prior_grid();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned walks = 0;
    if (a < M.N) walks = quad_stream_pops<G, false>(M, MS, sc, scd, K, st, err, a, G * blockIdx.y);
    // one atomic per warp (all lanes here: blocks of whole warps)
    const unsigned wsum = __reduce_add_sync(0xffffffffu, walks);
    if (stats && (threadIdx.x & 31u) == 0u && wsum) atomicAdd(stats, (unsigned long long)wsum);
}

// The propagation in two passes, as on triangles: kq_fast settles the
// populations whose previous-step element passes the certified FP32 test
// (grid y: 9 / G direction groups, G directions per thread) and lists the
// others; kq_slow runs the exact path over the list, spread over all blocks,
// so that the walks do not hold up the warps of settled populations.  TR: the
// map is a translation (no map, plunge).  The lanes are brought together after
// the certified test and after Newton (__syncwarp): left apart, the own and the
// other elements' lanes interpolated one after the other (150,400 nodes: 60 us
// against 33 in FP32).  The FP32 and 16-bit forms are held to 32 registers, 16
// blocks an SM, on a translation (33 us; 35 at 40 registers), and to 40, 12 blocks,
// on the other maps, which spill at 32 (150,400 nodes pitching: 37.1 us, 38.3 at
// 32 registers and 39.1 at 48; blended 37.8, 39.3, 40.1; 600,996 nodes 129 at 32
// and 40, 141 at 48).
template <class S, class A, int G, bool TR>
__global__ void __launch_bounds__(128, std::is_same<S, double>::value ? 1 : TR ? 16 : 12) kq_fast(QuadDev M, MapStatic MS, MapScalars scd, MapScalarsF sfd,
                                               KinParams<A> K, StateDev<S> st, unsigned long long *stats,
                                               const __grid_constant__ DepTab D)
{
    constexpr bool FP64 = std::is_same<S, double>::value;
    wait_prior_grid();
    const int a = blockIdx.x * blockDim.x + threadIdx.x, i0 = G * blockIdx.y;
    int code[G];
#pragma unroll
    for (int j = 0; j < G; ++j) code[j] = 0;
    const unsigned lanes = __ballot_sync(0xffffffffu, a < M.N);
    if (a < M.N) {
        const float4 Xf = M.Xf[a];
        FastMap F = TR ? fast_map_translation(sfd, Xf) : fast_map(MS, sfd, a, Xf);
        if (K.flags & (FLAG_LITERAL_VG | FLAG_EXACT_CHAR)) F.ok = false;
        Node64 n;
        double2 X;
        int c[G];
        if constexpr (FP64) {
            X = M.X[a];
            if (!TR) n = node64<TR>(MS, scd, a, X, false);
            if (!TR && i0 == 0 && st.met) { // for the derivative passes
                st.met[2 * a] = make_double2(n.a11, n.a12);
                st.met[2 * a + 1] = make_double2(n.a21, n.a22);
            }
#pragma unroll
            for (int j = 0; j < G; ++j) c[j] = st.cache[(i0 + j) * M.N + a];
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const int i = i0 + j;
            __syncwarp(lanes);
            // (a node of zero mesh velocity fails the test: its c^_0 is zero)
            bool done;
            if constexpr (FP64) done = quad_fast_pop64<TR>(M, F, n, Xf, X, st, a, i, c[j], lanes, D);
            else done = quad_fast_pop<S, A>(M, F, Xf, st, a, i, lanes);
            if (!done && F.ok) {
                const int ck = cone_missing(M, F, a, i);
                if (ck == 2) fg_put(st.str, i, a, M.N, K.finf[i], K.ginf[i]); // far field
                // 3: settled, but not by the element (the counter tells them apart)
                code[j] = ck == 2 ? 3 : ck == 1 ? 2 : 1;
            } else {
                code[j] = done ? 0 : 1;
            }
            if (i == 0 && M.vzero[a] && !(K.flags & FLAG_SHIFT)) { // c^_0 exactly zero: the node's own value
                fg_copy(st.str, st.post, 0, a, M.N);
                code[j] = 0;
            }
        }
    }
    int any = 0;
#pragma unroll
    for (int j = 0; j < G; ++j) any |= code[j];
    if (__any_sync(0xffffffffu, any != 0)) {
#pragma unroll
        for (int j = 0; j < G; ++j) {
            append_pop(st, a, M.N, i0 + j, code[j]);
            const unsigned far = __ballot_sync(0xffffffffu, code[j] == 3);
            if (!FP64 && stats && far && (threadIdx.x & 31u) == 0u) atomicAdd(stats, (unsigned long long)__popc(far));
        }
    }
}

// The exact path's walk runs on certified FP32 signs, the wall condition once
// per wall node for its cone-certified directions, its three gradients with one
// Jacobian: 30 us against 53 with every listed population walked in FP64 and
// its wall condition computed per direction (FP32, 150,400 nodes; FP64 form 40
// against 67).  Bound by the latency of one entry's chain.
// The counter: the deviation forms count the populations that the certified
// test does not settle (the nodes of zero mesh velocity among them), the FP64
// form all that are located (9 N less those whose c^ is exactly zero).
template <class S, class A>
__global__ void __launch_bounds__(128) kq_slow(QuadDev M, MapStatic MS, MapScalars sc, MapScalars scd, MapScalarsF sfd,
                                               KinParams<A> K, StateDev<S> st, int *err, unsigned long long *stats)
{
    constexpr bool FP64 = std::is_same<S, double>::value;
    wait_prior_grid();
    __shared__ unsigned pre[NQ + 1];
    if (threadIdx.x == 0) work_prefix(st.wcount, pre);
    __syncthreads();
    const unsigned n = pre[NQ];
    if (stats && blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned nz = K.flags & FLAG_SHIFT ? 0u : (unsigned)M.nvzero;
        atomicAdd(stats, FP64 ? (unsigned long long)NQ * M.N - nz : (unsigned long long)n + nz);
    }
    const unsigned total = n + st.wcount[NQ]; // then the wall nodes, with their certified directions
    for (unsigned w = spread_first(); w < total; w += spread_stride()) {
        if (w < n) {
            const int code = work_at(st.work, M.N, pre, w);
            const unsigned walks = quad_slow_pop(M, MS, sc, scd, sfd, K, st, err, code / NQ, code % NQ);
            if (FP64 && stats && !walks) atomicAdd(stats, ~0ull); // c^ exactly zero: one less
        } else {
            const int a = st.work[(size_t)NQ * M.N + (w - n)];
            const unsigned mask = st.wmask[a] & WMASK_DIRS;
            if (!FP64 && stats) atomicAdd(stats, (unsigned long long)__popc(mask));
            quad_bc_node(M, MS, sc, K, st, a, mask);
        }
    }
}

// Directions per thread of kq_stream (the FP64 form where no FP32
// certificate covers the departure point): one per population,
// the most threads to hide the walks' dependent loads (3.90 ms per launch
// at 150k nodes, against 4.00 at three and 4.12 at nine).
#ifndef ALELB_QUAD_G
#define ALELB_QUAD_G 1
#endif
static_assert(NQ % ALELB_QUAD_G == 0, "directions per thread");

// d_x K0 and d_y K1 at node a in FP64 (owner_div64 on quadrilaterals).
__device__ __forceinline__ void quad_owner_div64(const QuadDev &M, const MapStatic &MS, const MapScalars &sc,
                                                 const StateDev<double> &st, int a, const double *K0, const double *K1,
                                                 double &d0, double &d1)
{
    double X0, Y0, X1, Y1, A[4];
    quad_owner_grad(M, a, K0, X0, Y0);
    quad_owner_grad(M, a, K1, X1, Y1);
    d0 = X0;
    d1 = Y1;
    if (MS.kind == MK_NONE || MS.kind == MK_PLUNGE) return; // A = I
    metric64(MS, sc, M.X, st, a, A);
    d0 = A[0] * X0 + A[2] * Y0;
    d1 = A[1] * X1 + A[3] * Y1;
}

// D_a = (mu / rho T) d_a Q'_aaa in the owner element (Eq. Xa); FP32 in the
// deviation forms (the FP32 map and the node's FP32 owner-element J^{-1}),
// FP64 otherwise.
template <class S, class A>
__global__ void __launch_bounds__(256) kq_deriv1(QuadDev M, MapStatic MS, MapScalars sc, MapScalarsF sf,
                                                 StateDev<S> st)
{
    wait_prior_grid();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M.N) return;
    if constexpr (!std::is_same<S, double>::value) {
        const FastMap F = fast_map(MS, sf, a, M.Xf[a]);
        float KX, KY;
        quad_owner_grad(M, a, st.Qx, KX, KY);
        const float dQx = F.A11 * KX + F.A21 * KY; // d_x Q'_xxx
        quad_owner_grad(M, a, st.Qy, KX, KY);
        const float dQy = F.A12 * KX + F.A22 * KY; // d_y Q'_yyy
        const float m = (float)st.mrt[a];
        st.Dx[a] = (fld_t<S>)(m * dQx);
        st.Dy[a] = (fld_t<S>)(m * dQy);
    } else {
        double dQx, dQy;
        quad_owner_div64(M, MS, sc, st, a, st.Qx, st.Qy, dQx, dQy);
        const double m = st.mrt[a];
        st.Dx[a] = m * dQx;
        st.Dy[a] = m * dQy;
    }
}

// X_a = -d_a D_a in the owner element, then the collision (Eqs. feqn, geqn).
template <class S, class A>
__global__ void __launch_bounds__(128) kq_collide(QuadDev M, MapStatic MS, MapScalars sc, MapScalarsF sf,
                                                  KinParams<A> K, StateDev<S> st, int *err)
{
    wait_prior_grid();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M.N) return;
    const int N = M.N;
    if constexpr (std::is_same<S, double>::value) { // from the moments pass's fields
        double Xx = 0, Xy = 0;
        if (!(K.flags & (FLAG_PHI_OFF | FLAG_COLLIDE_OFF))) {
            quad_owner_div64(M, MS, sc, st, a, st.Dx, st.Dy, Xx, Xy);
            Xx = -Xx;
            Xy = -Xy;
        }
        collide_store64(K, st, N, a, Xx, Xy);
        return;
    } else {
        A Xx = 0, Xy = 0;
        if (!(K.flags & FLAG_PHI_OFF)) {
            const FastMap F = fast_map(MS, sf, a, M.Xf[a]);
            float KX, KY;
            quad_owner_grad(M, a, st.Dx, KX, KY);
            Xx = (A)(-(F.A11 * KX + F.A21 * KY));
            quad_owner_grad(M, a, st.Dy, KX, KY);
            Xy = (A)(-(F.A12 * KX + F.A22 * KY));
        }
        A f[NQ], g[NQ];
#pragma unroll
        for (int i = 0; i < NQ; ++i) fg_get(st.str, i, a, N, f[i], g[i]);
        A rho, ux, uy, T;
        if (!collide_node(K, f, g, Xx, Xy, rho, ux, uy, T)) atomicOr(err, ERR_NONFINITE);
#pragma unroll
        for (int i = 0; i < NQ; ++i) fg_put(st.post, i, a, N, f[i], g[i]);
        st.rho[a] = (fld_t<S>)rho;
        st.ux[a] = (fld_t<S>)ux;
        st.uy[a] = (fld_t<S>)uy;
        st.T[a] = (fld_t<S>)T;
    }
}

// Element choice of every population (parity report): original element id,
// -2 (the node itself) or -1 with the boundary kind.
static __global__ void kq_locate(QuadDev M, MapStatic MS, MapScalars sc, int literal, int *elem, int8_t *kind,
                                 int *err)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = M.N;
    if (a >= N) return;
    const double2 Xa = M.X[a];
    double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22, wx, wy;
    map_node(MS, sc, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
    metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
    mesh_velocity_term(a11, a12, a21, a22, ds(Vx, sc.Ux), ds(Vy, sc.Uy), literal != 0, wx, wy);
    for (int i = 0; i < NQ; ++i) {
        double chx, chy, px, py;
        departure(a11, a12, a21, a22, wx, wy, (double)lat_cx(i), (double)lat_cy(i), Xa.x, Xa.y, chx, chy, px, py);
        int e = -2, k = 0;
        if (!(chx == 0.0 && chy == 0.0)) {
            const Loc L = quad_walk(M, a, Xa.x, Xa.y, px, py, err);
            if (L.e >= 0) {
                e = M.orig_elem[L.vnode >= 0 ? quad_fan_best(M, L.vnode) : L.e];
            } else if (L.e == -1) {
                e = -1;
                k = L.kind;
            }
        }
        elem[i * N + a] = e;
        kind[i * N + a] = (int8_t)k;
    }
}

// Wall forces (reading R9): Simpson's rule on each straight 3-node wall edge
// of the mapped geometry, owner-element gradients; one thread per node of an
// edge, as on triangles (k_forces; 73 us in one block at 320 edges).
template <class S>
__global__ void __launch_bounds__(FORCE_BS) kq_forces(QuadDev M, MapStatic MS, MapScalars sc, StateDev<S> st,
                                                      const int2 *wedges, int nw, double mu, double Cv, double *part)
{
    double acc[4] = {0, 0, 0, 0};
    const int t = blockIdx.x * FORCE_BS + threadIdx.x;
    if (t < 3 * nw) {
        const int w = t / 3, j = t % 3, e = wedges[w].x, k = wedges[w].y, k1 = (k + 1) & 3;
        const int n0 = M.conn[9 * e + k], n2 = M.conn[9 * e + k1];
        const int a = j == 0 ? n0 : j == 1 ? M.conn[9 * e + 4 + k] : n2;
        const double2 A0 = M.X[n0], B0 = M.X[n2], Xa = M.X[a];
        double xa, ya, xb, yb;
        map_position(MS, sc, n0, A0.x, A0.y, xa, ya);
        map_position(MS, sc, n2, B0.x, B0.y, xb, yb);
        const double tx = xb - xa, ty = yb - ya, L = sqrt(tx * tx + ty * ty);
        const double nx = -ty / L, ny = tx / L; // out of the body, into the fluid
        double xX, xY, yX, yY, Vx, Vy, a11, a12, a21, a22;
        map_node(MS, sc, a, Xa.x, Xa.y, xX, xY, yX, yY, Vx, Vy);
        metric_inverse_T(xX, xY, yX, yY, a11, a12, a21, a22);
        double KX, KY, d[4];
        quad_grad(M, M.owner[a], st.ux, KX, KY);
        d[0] = a11 * KX + a21 * KY;
        d[1] = a12 * KX + a22 * KY;
        quad_grad(M, M.owner[a], st.uy, KX, KY);
        d[2] = a11 * KX + a21 * KY;
        d[3] = a12 * KX + a22 * KY;
        force_item(j == 1 ? 4.0 * L / 6.0 : L / 6.0, nx, ny, (double)st.rho[a], (double)st.T[a], d, mu, Cv, acc);
    }
    force_block_sums(acc, part);
}

} // namespace

alelb_status quad_mesh_upload(alelb_mesh *m)
{
    const QuadTables &Q = m->QT;
    const HostTables &T = m->T;
    cudaError_t st = cudaSuccess;
    DevBuf &B = m->buf;
    QuadDev &D = m->qdev;
    D.N = T.N;
    D.E = T.E;
    D.Lx = T.Lx;
    D.Ly = T.Ly;
    D.X = B.put(T.X, st);
    D.ev = B.put(Q.ev, st);
    D.nbr = B.put(Q.nbr, st);
    D.einfo = B.put(Q.einfo, st);
    D.rank = B.put(Q.rank, st);
    D.conn = B.put(Q.conn, st);
    D.fan_ptr = B.put(Q.fan_ptr, st);
    D.fan = B.put(Q.fan, st);
    D.owner = B.put(Q.owner, st);
    D.bcel = B.put(Q.bcel, st);
    D.bkind = B.put(Q.bkind, st);
    D.wall_idx = B.put(Q.wall_idx, st);
    D.probe_e = B.put(Q.probe_e, st);
    D.probe_xi = B.put(Q.probe_xi, st);
    D.wall_nrm = B.put(Q.wall_nrm, st);
    D.orig_elem = B.put(Q.orig, st);
    D.Xf = B.put(Q.Xf, st);
    D.evf = B.put(Q.evf, st);
    D.bdist = B.put(Q.bdist, st);
    D.ownJf = B.put(Q.ownJf, st);
    D.ownJd = B.put(Q.ownJd, st);
    D.ebd = B.put(Q.ebd, st);
    D.cone = B.put(Q.cone, st);
    D.conek = B.put(Q.conek, st);
    D.vzero = B.put(Q.vzero, st);
    D.nvzero = (int)std::count(Q.vzero.begin(), Q.vzero.end(), (uint8_t)1);
    m->d_wedges = B.put(Q.wedges, st);
    m->d_n2o = B.put(T.node_new2old, st);
    m->nw = (int)Q.wedges.size();
    m->mst = T.host_map();
    m->mst.ms = B.put(T.ms, st);
    m->mst.msf = B.put(T.msf, st);
    if (st == cudaSuccess) st = cudaDeviceSynchronize();
    if (st != cudaSuccess) {
        m->buf.release();
        m->err = cudaGetErrorString(st);
        return st == cudaErrorMemoryAllocation ? ALELB_ERR_OOM : ALELB_ERR_CUDA;
    }
    return ALELB_OK;
}

cudaError_t quad_launch(alelb_solver *s, int kernel, const MapScalars &sc, const MapScalars &scd)
{
    alelb_mesh *m = s->mesh;
    const int N = m->T.N;
    with_state(s, [&](auto &st, auto &K) {
        using S = typename std::remove_reference<decltype(st)>::type::Tag;
        using A = typename std::remove_reference<decltype(K)>::type::Arith;
        switch (kernel) {
        case KT_STREAM: {
            constexpr int G = ALELB_QUAD_G;
            launch_pdl(kq_stream<S, A, G>, dim3((N + 127) / 128, NQ / G), dim3(128), s->stream, m->qdev, m->mst, sc,
                       scd, K, st, s->d_err, s->d_stats);
            break;
        }
        case KT_FAST: {
            const MapScalarsF sfd = to_f32(scd, m->T);
            const DepTab dep = dep_table(scd);
            const bool tr = m->T.mkind == MK_NONE || m->T.mkind == MK_PLUNGE;
            const dim3 gb(128), g1((N + 127) / 128, NQ), g3(g1.x, NQ / 3);
            if (tr) {
                launch_pdl(kq_fast<S, A, 1, true>, g1, gb, s->stream, m->qdev, m->mst, scd, sfd, K, st, s->d_stats, dep);
                break;
            }
            if constexpr (std::is_same<S, double>::value) {
                // FP64: one map evaluation for three directions from 8k nodes
                // on (239k blended: 427 us against 539 at one and 446 at nine
                // per thread; 160k box 280, 318, 326; 24k 54, 62, 80), one per
                // direction below (1k box: 13, 24, 58 us)
                if (N >= FAST64_G3_NODES) {
                    launch_pdl(kq_fast<S, A, 3, false>, g3, gb, s->stream, m->qdev, m->mst, scd, sfd, K, st, s->d_stats, dep);
                    break;
                }
            }
            launch_pdl(kq_fast<S, A, 1, false>, g1, gb, s->stream, m->qdev, m->mst, scd, sfd, K, st, s->d_stats, dep);
            break;
        }
        case KT_SLOW: {
            // every block resident at once (the list spread over all of them)
            static const int per_sm = [] {
                int v = 0;
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kq_slow<S, A>, 128, 0);
                return v > 0 ? v : 1;
            }();
            launch_pdl(kq_slow<S, A>, dim3(per_sm * s->n_sm), dim3(128), s->stream, m->qdev, m->mst, sc, scd,
                       to_f32(scd, m->T), K, st, s->d_err, s->d_stats);
            break;
        }
        case KT_MOMENTS:
            launch_pdl(k_moments<S, A>, dim3((N + 255) / 256), dim3(256), s->stream, K, st, N, s->d_err);
            break;
        case KT_DERIV1:
            launch_pdl(kq_deriv1<S, A>, dim3((N + 255) / 256), dim3(256), s->stream, m->qdev, m->mst, sc,
                       to_f32(sc, m->T), st);
            break;
        default:
            launch_pdl(kq_collide<S, A>, dim3((N + 127) / 128), dim3(128), s->stream, m->qdev, m->mst, sc,
                       to_f32(sc, m->T), K, st, s->d_err);
        }
    });
    return cudaGetLastError();
}

cudaError_t quad_locate(alelb_solver *s, const MapScalars &sc, int *elem, int8_t *kind)
{
    alelb_mesh *m = s->mesh;
    kq_locate<<<(m->T.N + 127) / 128, 128, 0, s->stream>>>(m->qdev, m->mst, sc, (s->flags & ALELB_FLAG_LITERAL_VG) != 0,
                                                           elem, kind, s->d_err);
    return cudaGetLastError();
}

cudaError_t quad_forces(alelb_solver *s, const MapScalars &sc)
{
    alelb_mesh *m = s->mesh;
    with_state(s, [&](auto &st, auto &) {
        using S = typename std::remove_reference<decltype(st)>::type::Tag;
        kq_forces<S><<<force_blocks(m->nw), FORCE_BS, 0, s->stream>>>(m->qdev, m->mst, sc, st, m->d_wedges, m->nw, s->mu,
                                                                      s->Cv, s->d_scratch);
        k_forces_sum<<<1, 128, 0, s->stream>>>(s->d_scratch, force_blocks(m->nw), s->d_out);
    });
    return cudaGetLastError();
}

} // namespace alelb
