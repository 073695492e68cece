// Differentiation of a simulated trajectory by the adjoint method.  Each time step is taken as the solution of
// grad E(x_{t+1}; x~_t, theta) = 0 (Algorithm 1's minimisation), x~_t = x_t + h v_t + h^2 g, v_{t+1} = (x_{t+1} - x_t)/h.
// The implicit function theorem gives H dx_{t+1} = M dx~_t - (d grad E / d theta) d theta with H the Hessian of E at
// x_{t+1} (inertia, elastic density, barrier with the closest points frozen as in Sec. 3.2, half-space barrier), so a
// reverse step solves H lambda = abar_x(t+1) + abar_v(t+1)/h and carries abar_x~ = M lambda back:
//   abar_x(t) = M lambda - abar_v(t+1)/h,   abar_v(t) = h M lambda,   abar_E_e -= lambda_e . d g_e / d E_e.
// H is applied matrix-free (the vector form of the p^T H p terms); the solve is Jacobi-preconditioned linear CG with
// the preconditioner of Sec. 4.2.  Kinematic vertices: rows and columns of H dropped, lambda = 0 there.
#pragma once

#include "kernels.cuh"
#include "persistent.cuh"

namespace pncg {

// Vectors of this pass (v, H v, the solver's x, r, p, q) are double4_32a per vertex: one 256-bit access each.

// kinematic rows and columns of H are dropped
template <typename R> __device__ inline bool dropped(const Dev<R> &D, int i) { return D.nfix > 0 && D.xtil[i].w < 0.0; }

// Hessian times v, vertex part (inertia and half-space barrier; kinematic rows zero).  Needs the gradient pass at x
// (dg.w = mass or -1, g.w = kappa b'' of the half-space).
template <typename R>
__device__ inline double4_32a hvp_vert(const Dev<R> &D, int par, int i, const double4_32a &v)
{
    const typename V4<R>::T Dg = D.dg[par][i];
    if (!(Dg.w > R(0))) return make_double4_32a(0.0, 0.0, 0.0, 0.0);
    const double m = Dg.w;
    double4_32a o = make_double4_32a(m * v.x, m * v.y, m * v.z, 0.0);
    if (D.has_plane) {
        const R w = D.g[par][i].w;
        if (w != R(0)) {
            const double nv = D.pn[0] * v.x + D.pn[1] * v.y + D.pn[2] * v.z, k = double(w) * nv;
            o.x += k * D.pn[0]; o.y += k * D.pn[1]; o.z += k * D.pn[2];
        }
    }
    return o;
}
template <typename R>
__global__ void k_hvp_vert(Dev<R> D, int par, const double4_32a *v, double4_32a *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < D.nv) out[i] = hvp_vert<R>(D, par, i, v[i]);
}

template <typename R> __device__ inline v3<double> vload(const Dev<R> &D, const double4_32a *v, int i)
{
    if (dropped(D, i)) return mkv(0.0, 0.0, 0.0);
    const double4_32a a = ldcg4(v + i);
    return mkv(a.x, a.y, a.z);
}
template <typename R> __device__ inline void vadd(const Dev<R> &D, double4_32a *out, int i, double a, double b, double c)
{
    if (dropped(D, i)) return;
    atomicAdd(&out[i].x, a);
    atomicAdd(&out[i].y, b);
    atomicAdd(&out[i].z, c);
}

// Elastic part of one tet on the direction's edge vectors Dp: the columns of h^2 V dP Dm^-T, the corners' contributions
// of x_1..x_3 (x_0 gets minus their sum); p^T (H p) equals the p^T H p form of Sec. 3.1.  NH and SNH:
//   FP64: Dp (2 Psi_2 h^2 V M) + h^2 V Psi_33 det(Dm^-1)^2 (cof(Ds) : Dp) cof(Ds) + h^2 V Psi_3 det(Dm^-1) d cof(Ds)[Dp], with
// the scalars that the gradient pass at x left (tet_pHp_edges): about 135 FP64 operations where the form on F took 430
// (82,944 tets: 70 us a pass).  rec (or null): cof(Ds) and h^2 V Psi_3 det(Dm^-1) Ds kept by the solver, whose x stands
// still (hvp_record): 91 operations, and 15 for the corner sums and p^T H_e p.
//   FP32: (L P F^T + 2 (k1 tr(E) I + k2 E)) Ds^-T, E = L + L^T, L = Dp Ds^-1, from the gradient pass's record: the
// derivative of the quadratic form of tet_pHp_edges, in which the large terms of a rotating direction never meet.
constexpr int HVP_REC = 5;   // double4 per tet of the record
__device__ inline void hvp_record(const Dev<double> &D, int e, double4_32a *rec)
{
    const size_t n = (size_t)D.nt;
    double s[3][3], c[3][3];
    tet_ds<double>(D, D.tet[e], s);
    cof3<double>(s, c);
    const double k3 = __ldcg(D.tk + n + e);
    rec[e] = make_double4_32a(c[0][0], c[0][1], c[0][2], c[1][0]);
    rec[n + e] = make_double4_32a(c[1][1], c[1][2], c[2][0], c[2][1]);
    rec[2 * n + e] = make_double4_32a(c[2][2], k3 * s[0][0], k3 * s[0][1], k3 * s[0][2]);
    rec[3 * n + e] = make_double4_32a(k3 * s[1][0], k3 * s[1][1], k3 * s[1][2], k3 * s[2][0]);
    rec[4 * n + e] = make_double4_32a(k3 * s[2][1], k3 * s[2][2], 0.0, 0.0);
}
template <typename R>
__device__ inline void tet_hvp_edges(const Dev<R> &D, int e, const int4 &tv, const R dp[3][3], R H[3][3], const double4_32a *rec)
{
    const size_t n = (size_t)D.nt;
    if constexpr (sizeof(R) == 4) {
        const float4 q0 = __ldcg(D.tS + e), q1 = __ldcg(D.tS + n + e), q2 = __ldcg(D.tS + 2 * n + e);
        const float4 q3 = __ldcg(D.tS + 3 * n + e);
        const float hv = D.hv[e], k1 = hv * __ldcg(D.tk + e), k2 = hv * q3.w;
        const float Z[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
        const float S[3][3] = {{q2.y, q2.z, q2.w}, {q2.z, q3.x, q3.y}, {q2.w, q3.y, q3.z}};
        float L[3][3], E[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) L[a][b] = dp[a][0] * Z[b][0] + dp[a][1] * Z[b][1] + dp[a][2] * Z[b][2];
        const float kt = 4.0f * k1 * (L[0][0] + L[1][1] + L[2][2]);   // 2 k1 tr(E)
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b)
                E[a][b] = 2.0f * k2 * (L[a][b] + L[b][a]) + (a == b ? kt : 0.0f) + L[a][0] * S[0][b] + L[a][1] * S[1][b] + L[a][2] * S[2][b];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < 3; ++i) H[a][i] = E[a][0] * Z[0][i] + E[a][1] * Z[1][i] + E[a][2] * Z[2][i];
    } else {
        const double4_32a a = D.td[e], b = D.td[n + e];
        R s[3][3], c[3][3];
        if (rec) {
            const double4_32a q0 = rec[e], q1 = rec[n + e], q2 = rec[2 * n + e], q3 = rec[3 * n + e], q4 = rec[4 * n + e];
            c[0][0] = q0.x; c[0][1] = q0.y; c[0][2] = q0.z; c[1][0] = q0.w; c[1][1] = q1.x; c[1][2] = q1.y;
            c[2][0] = q1.z; c[2][1] = q1.w; c[2][2] = q2.x;
            s[0][0] = q2.y; s[0][1] = q2.z; s[0][2] = q2.w; s[1][0] = q3.x; s[1][1] = q3.y; s[1][2] = q3.z;
            s[2][0] = q3.w; s[2][1] = q4.x; s[2][2] = q4.y;
        } else {
            const R k3 = __ldcg(D.tk + n + e);
            tet_ds<R>(D, tv, s);
            cof3<R>(s, c);
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int i = 0; i < 3; ++i) s[r][i] *= k3;
        }
        R g3 = R(0);
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int i = 0; i < 3; ++i) g3 += c[r][i] * dp[r][i];
        g3 *= __ldcg(D.tk + e);
        const R M[3][3] = {{a.x, a.y, a.z}, {a.y, a.w, b.x}, {a.z, b.x, b.y}};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int u = (i + 1) % 3, w = (i + 2) % 3;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const int y = (r + 1) % 3, z = (r + 2) % 3;
                H[r][i] = dp[r][0] * M[0][i] + dp[r][1] * M[1][i] + dp[r][2] * M[2][i] + g3 * c[r][i] +
                          (dp[y][u] * s[z][w] - dp[z][u] * s[y][w]) + (s[y][u] * dp[z][w] - s[z][u] * dp[y][w]);
            }
        }
    }
}

// FCR and ARAP, on F: dP = 2 Psi_2 dF + Psi_33 (cof F : dF) cof F + Psi_3 d cof(F)[dF] + Psi_1 H1[dF] (the differential of P =
// Psi_1 R + 2 Psi_2 F + Psi_3 cof F; the I1 term from the polar decomposition, in double).
template <typename R>
__device__ inline bool tet_hvp_rotated(const Dev<R> &D, int e, const int4 &tv, const R dp[3][3], R H[3][3])
{
    TetF<R> T;
    tet_F<R>(D, e, tv, T);
    if (!(T.J > R(0))) { flag_error(D.ctrl, ERR_INVERTED); return false; }
    R dF[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) dF[a][b] = dp[a][0] * T.w[0][b] + dp[a][1] * T.w[1][b] + dp[a][2] * T.w[2][b];
    R mu, lam;
    tet_material<R>(D, e, mu, lam);
    const MatTerms<R> mt = mat_terms<R>(D.model, mu, lam, T.J);
    R g3 = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) g3 += T.cf[a][b] * dF[a][b];
    double Fd[3][3], dFd[3][3], H1[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) { Fd[a][b] = double(T.F[a][b]); dFd[a][b] = double(dF[a][b]); }
    Polar pol;
    polar_of(Fd, pol);
    polar_h1_vec(pol, dFd, H1);
    const R sc = D.hv[e];
    R dP[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int u = (i + 1) % 3, w = (i + 2) % 3;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int y = (r + 1) % 3, z = (r + 2) % 3;   // column i of d cof(F)[dF] = d(f_u x f_w)
            const R dc = (dF[y][u] * T.F[z][w] - dF[z][u] * T.F[y][w]) + (T.F[y][u] * dF[z][w] - T.F[z][u] * dF[y][w]);
            dP[r][i] = sc * (mt.c2 * dF[r][i] + mt.Psi33 * g3 * T.cf[r][i] + mt.Psi3 * dc) + sc * R(double(mt.Psi1) * H1[r][i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int a = 0; a < 3; ++a) H[a][i] = dP[a][0] * T.w[i][0] + dP[a][1] * T.w[i][1] + dP[a][2] * T.w[i][2];
    return true;
}

// out += H_e v of tet e; returns v^T H_e v, in double as every sum: in the FP32 form from v itself and the entries that were
// added, so that it is the v^T (H v) of the vectors
template <typename R, bool CO>
__device__ inline double hvp_tet(const Dev<R> &D, int e, const double4_32a *v, double4_32a *out, const double4_32a *rec = nullptr)
{
    const int4 tv = D.tet[e];
    const v3<double> V0 = vload(D, v, tv.x), V1 = vload(D, v, tv.y), V2 = vload(D, v, tv.z), V3 = vload(D, v, tv.w);
    R dp[3][3], H[3][3];
    dp[0][0] = R(V1.x) - R(V0.x); dp[1][0] = R(V1.y) - R(V0.y); dp[2][0] = R(V1.z) - R(V0.z);
    dp[0][1] = R(V2.x) - R(V0.x); dp[1][1] = R(V2.y) - R(V0.y); dp[2][1] = R(V2.z) - R(V0.z);
    dp[0][2] = R(V3.x) - R(V0.x); dp[1][2] = R(V3.y) - R(V0.y); dp[2][2] = R(V3.z) - R(V0.z);
    if constexpr (CO) {
        if (!tet_hvp_rotated<R>(D, e, tv, dp, H)) return 0.0;
    } else {
        tet_hvp_edges<R>(D, e, tv, dp, H, rec);
    }
    vadd<R>(D, out, tv.y, H[0][0], H[1][0], H[2][0]);
    vadd<R>(D, out, tv.z, H[0][1], H[1][1], H[2][1]);
    vadd<R>(D, out, tv.w, H[0][2], H[1][2], H[2][2]);
    const R h0 = -(H[0][0] + H[0][1] + H[0][2]), h1 = -(H[1][0] + H[1][1] + H[1][2]), h2 = -(H[2][0] + H[2][1] + H[2][2]);
    vadd<R>(D, out, tv.x, h0, h1, h2);
    double q = 0.0;
    if constexpr (sizeof(R) == 4) {
        q = V0.x * h0 + V0.y * h1 + V0.z * h2;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const v3<double> &V = i == 0 ? V1 : i == 1 ? V2 : V3;
            q += V.x * H[0][i] + V.y * H[1][i] + V.z * H[2][i];
        }
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int i = 0; i < 3; ++i) q += dp[a][i] * H[a][i];
    }
    return q;
}
template <typename R, bool CO>
__global__ void __launch_bounds__(EB) k_hvp_tet(Dev<R> D, const double4_32a *v, double4_32a *out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < D.nt) hvp_tet<R, CO>(D, e, v, out);
}

// Barrier pair part with the closest points frozen (Eqs. 12-13 as an operator): w = sum_j c_j v_j,
// (H v)_k += c_k (A (w . t) t + B w).  In double: the pair terms cancel in part.  Returns v^T H_k v.
template <typename R>
__device__ inline double hvp_pair(const Dev<R> &D, int k, const double4_32a *v, double4_32a *out)
{
    Active<R> ap;
    load_active<R>(D, k, ap);
    const int vid[4] = {ap.v.x, ap.v.y, ap.v.z, ap.v.w};
    double w[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const v3<double> V = vload(D, v, vid[j]);
        w[0] += double(ap.c[j]) * V.x; w[1] += double(ap.c[j]) * V.y; w[2] += double(ap.c[j]) * V.z;
    }
    const double s = w[0] * double(ap.t[0]) + w[1] * double(ap.t[1]) + w[2] * double(ap.t[2]);
    const double A = ap.A, Bc = ap.B;
    double f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) f[a] = A * s * double(ap.t[a]) + Bc * w[a];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double cj = ap.c[j];
        vadd<R>(D, out, vid[j], cj * f[0], cj * f[1], cj * f[2]);
    }
    return w[0] * f[0] + w[1] * f[1] + w[2] * f[2];
}
template <typename R>
__global__ void __launch_bounds__(EB) k_hvp_pair(Dev<R> D, const double4_32a *v, double4_32a *out)
{
    const int na = D.ctrl->n_active;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < na; k += gridDim.x * blockDim.x) hvp_pair<R>(D, k, v, out);
}

// ---- linear CG on H lambda = b (Jacobi-preconditioned) in one launch: every block stays resident and meets the others at
// the grid barriers of the persistent time step (or, on a small mesh, as one cluster: CL).  An iteration has three:
//   direction  p = z + beta p and the vertex part of q = H p, one thread per vertex
//   product    the tets and pairs add to q; p^T q accumulates beside it from the elements' own p^T H_e p, so that no pass
//              of its own reads p and q for it
//   update     alpha = r.z / p.q; x += alpha p, r -= alpha q, z = P r; the sums r.z and r.r
// It replaces six launches an iteration and a host round trip every eight (82,944 tets, about 900 iterations: 100 us an
// iteration, nearly all of it the kernels themselves, against 38 in one launch, of which the product is 28).  Convergence is
// looked at every eighth iteration.  The waits at the grid barriers are bounded as the time step's; the cluster's need not be.
constexpr int CG_PB = 256;
constexpr int CG_STRIDE = 8;      // iterations between two looks at the residual
enum { CG_RZ = 0, CG_BETA, CG_RR, CG_BB, CG_IT, CG_N };
struct CgArgs {
    double4_32a *x, *r, *p, *q, *P;   // solution, residual (the right-hand side at iteration 0), direction, H p, Jacobi entries
    double4_32a *rec;                 // FP64 form, NH and SNH: [HVP_REC][nt] (hvp_record); else, or without room for it, null
    double *cg;                       // [CG_N] scalars carried between launches
    void *part;                       // reduction partials: 16 x gridDim.x doubles
    unsigned int *count;              // barrier arrival counter (zeroed before the launch)
    int it0, it1;                     // iterations of this launch
    double tol2;                      // squared relative tolerance
};

template <typename R, bool CO, bool CL>
__global__ void __launch_bounds__(CG_PB, CL ? 1 : 2) k_cg(Dev<R> D, CgArgs A)
{
    __shared__ __align__(16) unsigned char sh_raw[sizeof(PShared<double, CG_PB, CL>)];
    PShared<double, CG_PB, CL> &sh = *reinterpret_cast<PShared<double, CG_PB, CL> *>(sh_raw);
    Ctrl *c = D.ctrl;
    RedBufs rb;
    rb.base = A.part;
    rb.n = gridDim.x;
    Bar br{A.count, 0u, nullptr, nullptr, nullptr, 0, 0};
    const Share vs = share_of(D.nv), ts = share_of(D.nt);
    const int na = min((volatile const int &)c->n_active, D.cand_cap);
    const Share as = share_of(na);
    const int nts = ts.b1 - ts.b0, nit = nts + (as.b1 - as.b0);
    const int par = 0;   // the gradient pass of the evaluation
    double rz = A.cg[CG_RZ], beta = A.cg[CG_BETA], rr = A.cg[CG_RR], bb = A.cg[CG_BB];
    grid_barrier<CL>(br, c);
    // alpha, beta and the other scalars: FP64 divisions, in one thread per block
    auto share = [&](double a, double b) {
        if (threadIdx.x == 0) { sh.o[0] = a; sh.o[1] = b; }
        __syncthreads();
    };
    constexpr bool REC = sizeof(R) == 8 && !CO;
    if (A.it0 == 0) {
        if constexpr (REC)
            for (int e = ts.b0 + (int)threadIdx.x; A.rec && e < ts.b1; e += CG_PB) hvp_record(D, e, A.rec);
        Acc<double> s[2];
        for (int i = vs.b0 + (int)threadIdx.x; i < vs.b1; i += CG_PB) {
            const typename V4<R>::T Dg = ldcg4(D.dg[par] + i);
            const bool fr = Dg.w > R(0);
            const double4_32a P = fr ? make_double4_32a(precond<R>(Dg.x, Dg.w), precond<R>(Dg.y, Dg.w), precond<R>(Dg.z, Dg.w), 0.0)
                                     : make_double4_32a(0.0, 0.0, 0.0, 0.0);
            const double4_32a r = A.r[i];
            A.P[i] = P;
            A.x[i] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
            s[0].v += r.x * (P.x * r.x) + r.y * (P.y * r.y) + r.z * (P.z * r.z);
            s[1].v += r.x * r.x + r.y * r.y + r.z * r.z;
        }
        grid_reduce<double, CG_PB, CL, 2, false>(s, 0.0, rb.sum_region<double>(), sh, br, c);
        rz = sh.res[0];
        bb = rr = sh.res[1];
        beta = 0.0;
    }
    int it = A.it0;
    for (; it < A.it1; ++it) {
        if (it % CG_STRIDE == 0 && !(bb > 0.0 && rr > A.tol2 * bb)) break;
        Acc<double> pq[1];
        for (int i = vs.b0 + (int)threadIdx.x; i < vs.b1; i += CG_PB) {
            const double4_32a r = A.r[i], P = A.P[i];
            double4_32a p = make_double4_32a(P.x * r.x, P.y * r.y, P.z * r.z, 0.0);
            if (it > 0) {
                const double4_32a p0 = A.p[i];
                p.x += beta * p0.x; p.y += beta * p0.y; p.z += beta * p0.z;
            }
            const double4_32a q = hvp_vert<R>(D, par, i, p);
            A.p[i] = p;
            A.q[i] = q;
            pq[0].v += p.x * q.x + p.y * q.y + p.z * q.z;
        }
        grid_barrier<CL>(br, c);
        for (int j = threadIdx.x; j < nit; j += CG_PB)
            pq[0].v += j < nts ? hvp_tet<R, CO>(D, ts.b0 + j, A.p, A.q, REC ? A.rec : nullptr) : hvp_pair<R>(D, as.b0 + j - nts, A.p, A.q);
        grid_reduce<double, CG_PB, CL, 1, false>(pq, 0.0, rb.sum_region<double>(), sh, br, c);
        share(threadIdx.x == 0 && sh.res[0] != 0.0 ? rz / sh.res[0] : 0.0, 0.0);
        const double al = sh.o[0];
        Acc<double> s[2];
        for (int i = vs.b0 + (int)threadIdx.x; i < vs.b1; i += CG_PB) {
            const double4_32a p = A.p[i], q = ldcg4(A.q + i), P = A.P[i];
            double4_32a x = A.x[i], r = A.r[i];
            x.x += al * p.x; x.y += al * p.y; x.z += al * p.z;
            r.x -= al * q.x; r.y -= al * q.y; r.z -= al * q.z;
            A.x[i] = x;
            A.r[i] = r;
            s[0].v += r.x * (P.x * r.x) + r.y * (P.y * r.y) + r.z * (P.z * r.z);
            s[1].v += r.x * r.x + r.y * r.y + r.z * r.z;
        }
        grid_reduce<double, CG_PB, CL, 2, false>(s, 0.0, rb.sum_region<double>(), sh, br, c);
        share(0.0, threadIdx.x == 0 && rz != 0.0 ? sh.res[0] / rz : 0.0);
        beta = sh.o[1];
        rz = sh.res[0];
        rr = sh.res[1];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.cg[CG_RZ] = rz; A.cg[CG_BETA] = beta; A.cg[CG_RR] = rr; A.cg[CG_BB] = bb; A.cg[CG_IT] = it;
    }
}

// ---- the reverse step's vertex bookkeeping
// rhs = abar_x + abar_v / h on free vertices
template <typename R>
__global__ void k_adj_rhs(Dev<R> D, const double *ax, const double *av, double4_32a *b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D.nv) return;
    double f[3];
    for (int a = 0; a < 3; ++a) f[a] = dropped(D, i) ? 0.0 : ax[3 * i + a] + av[3 * i + a] / D.h;
    b[i] = make_double4_32a(f[0], f[1], f[2], 0.0);
}
// abar_x(t) = M lambda - abar_v(t+1)/h, abar_v(t) = h M lambda (free vertices);
// kinematic: abar_x(t) = -abar_v(t+1)/h (v(t+1) = (target - x(t))/h), abar_v(t) = 0
template <typename R>
__global__ void k_adj_out(Dev<R> D, const double4_32a *lam, const double *av, double *ax_t, double *av_t)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D.nv) return;
    const double4_32a l = lam[i];
    const double m = dropped(D, i) ? 0.0 : D.mass[i], ml[3] = {m * l.x, m * l.y, m * l.z};
    for (int a = 0; a < 3; ++a) {
        ax_t[3 * i + a] = ml[a] - av[3 * i + a] / D.h;
        av_t[3 * i + a] = D.h * ml[a];
    }
}
// dE_e -= lambda_e . d g_e / d E_e: the tet's elastic gradient is linear in E_e (mu and lambda are), so its
// derivative is the gradient evaluated with E_e = 1 (D carries mu and lambda of E = 1 and no per-tet scale).  The tets' constants
// hold mu_e, which may be 0: mu h^2 V M (or its factor) is formed anew, from D_m^-1.
template <typename R, bool CO = false>
__global__ void __launch_bounds__(EB) k_adj_youngs(Dev<R> D, const double4_32a *lam, double *dE)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= D.nt) return;
    TetIn<R> in;
    load_tet_in<R, CO>(D, e, in);
    if constexpr (!CO) {
        R w[3][3];
        load_w<R>(D, e, w);
        const R f = D.mu * D.hv[e];
        if constexpr (sizeof(R) == 4) {
            double wd[3][3], k[6];
            for (int i = 0; i < 9; ++i) wd[i / 3][i % 3] = w[i / 3][i % 3];
            tri_factor(wd, sqrt((double)f), k);
            for (int i = 0; i < 6; ++i) in.m[i] = (float)k[i];
        } else {
            int q = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = i; j < 3; ++j, ++q) in.m[q] = f * (w[i][0] * w[j][0] + w[i][1] * w[j][1] + w[i][2] * w[j][2]);
        }
    }
    R gv[4][3], dv[4][3];
    if (!tet_grad_eval<R, CO>(D, in, gv, dv)) return;
    const int vid[4] = {in.tv.x, in.tv.y, in.tv.z, in.tv.w};
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double4_32a l = lam[vid[i]];
        s += l.x * double(gv[i][0]) + l.y * double(gv[i][1]) + l.z * double(gv[i][2]);
    }
    dE[e] -= s;
}

} // namespace pncg
