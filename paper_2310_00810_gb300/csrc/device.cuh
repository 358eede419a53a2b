// Device helpers shared by the forward and adjoint kernels: moments of
// shifted populations (Eq. 1-2), BGK collision (Eq. 4-5) and the pull with
// halfway bounce-back and anti-bounce-back (Eq. 3, Eq. 6).
#pragma once

#include "common.cuh"

namespace lbm {

// omega = 1 / tau.  wide: rounded from the FP64 quotient, without an FP64
// division in every thread (an FP32 quotient corrected by its residual,
// accurate to 2^-47 before the last rounding).
template <typename T>
__device__ __forceinline__ T relaxation_rate(double tau, bool wide)
{
    const T t = T(tau), w = T(1) / t;
    if constexpr (sizeof(T) == 4) {
        if (wide) {
            const float lo = (float)(tau - (double)t);  // tau = t + lo
            const float r = fmaf(fmaf(-lo, w, fmaf(-t, w, 1.0f)), w, w);
            if (isfinite(r)) return r;
        }
    }
    return w;
}

// The sum of one term per lane, valid in lane 0: in T, or (wide, FP32) to the
// accuracy of an FP64 sum as pairs of FP32 numbers: each addition keeps its
// rounding error exactly (Knuth's two-sum).  FP64 lanes would cost 80 cycles
// of an SM's FP64 pipe per warp.
template <typename T>
__device__ __forceinline__ double warp_total(T v, bool wide)
{
    if constexpr (sizeof(T) == 4) {
        if (wide) {
            float hi = v, lo = 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
                const float s = hi + h2, b = s - hi;
                lo += l2 + ((hi - (s - b)) + (h2 - b));
                hi = s;
            }
            return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return (double)v;
}


template <int Q>
__host__ __device__ constexpr long long link_offset(int i, int nx, long long plane)
{
    return (long long)Lattice<Q>::c(i, 0) + (long long)Lattice<Q>::c(i, 1) * nx +
           (long long)Lattice<Q>::c(i, 2) * plane;
}

// Moments of shifted populations: rho = 1 + sum v, rho u = sum c v.
template <int Q, typename T>
__device__ __forceinline__ void moments(const T (&v)[Q], T& drho, T& rho, T (&u)[3])
{
    using L = Lattice<Q>;
    T s = 0, j[3] = {0, 0, 0};
    if constexpr (std::is_same<T, double>::value) {  // by opposite pairs, which takes fewer additions
        s = v[0];
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if (i < L::opp(i)) {
                const T o = v[i] - v[L::opp(i)];
                s += v[i] + v[L::opp(i)];
#pragma unroll
                for (int a = 0; a < L::D; ++a)
                    if (L::c(i, a) != 0) j[a] = L::c(i, a) > 0 ? j[a] + o : j[a] - o;
            }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            s += v[i];
#pragma unroll
            for (int a = 0; a < L::D; ++a)
                if (L::c(i, a) != 0) j[a] += L::c(i, a) > 0 ? v[i] : -v[i];
        }
    }
    drho = s;
    rho = T(1) + s;
    T inv = T(1) / rho;
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = a < L::D ? j[a] * inv : T(0);
}

template <int Q, typename T>
__device__ __forceinline__ T cdot(int i, const T (&u)[3])
{
    using L = Lattice<Q>;
    T s = 0;
#pragma unroll
    for (int a = 0; a < L::D; ++a)
        if (L::c(i, a) != 0) s += L::c(i, a) > 0 ? u[a] : -u[a];
    return s;
}

// Where the equilibrium and its adjoint are evaluated by opposite pairs and
// moments: FP64, which runs at about two lanes per SM and clock, so that its
// kernels are as fast as they have few operations (64x32 D2Q9: 23.7 us per time
// level of a gradient evaluation by direction, in 64-thread blocks and Eq. 6
// link by link; 16.8 so, in 32-thread blocks and with opposite Eq. 6 links
// together).  FP32 keeps the sums by direction: its layouts
// round alike term by term, and on D3Q19 pairs gave 1 to 3 %.
template <typename T>
constexpr bool kByPairs = std::is_same<T, double>::value;

// BGK collision (Eq. 4-5) in place on shifted populations.  FUSED: the last
// product and subtraction as one rounding, which is what the compiler makes
// of it in the vectorised and TMA kernels; where a kernel also holds the MRT
// collision it rounds twice.
template <int Q, typename T, bool FUSED = false>
__device__ __forceinline__ void collide(T (&v)[Q], T omega)
{
    using L = Lattice<Q>;
    T drho, rho, u[3];
    moments<Q, T>(v, drho, rho, u);
    if constexpr (kByPairs<T>) {
        // feq of i and its opposite: w (even +- odd), the cu^2 term shared
        T uu = u[0] * u[0] + u[1] * u[1];
        if (L::D == 3) uu += u[2] * u[2];
        const T base = drho - T(1.5) * rho * uu;
        const T r3 = T(3) * rho, r45 = T(4.5) * rho;
        v[0] = v[0] - omega * (v[0] - T(L::w(0)) * base);
        const T wa = T(L::w(1)), wd = T(L::w(Q - 1));  // the axis and the diagonal links
        const T b[2] = {wa * base, wd * base}, p[2] = {wa * r3, wd * r3}, q[2] = {wa * r45, wd * r45};
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if (i < L::opp(i)) {
                const int cls = L::w(i) == L::w(1) ? 0 : 1;
                const T cu = cdot<Q, T>(i, u);
                const T even = b[cls] + q[cls] * cu * cu, odd = p[cls] * cu;
                // the difference from f^eq first: (1 - omega) f + omega f^eq is two operations shorter and
                // rounds f^eq's own size (2.1e-16 rms of the state for 1.7e-16)
                v[i] = v[i] - omega * (v[i] - (even + odd));
                v[L::opp(i)] = v[L::opp(i)] - omega * (v[L::opp(i)] - (even - odd));
            }
        return;
    }
    T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        T cu = cdot<Q, T>(i, u);
        T feq = T(L::w(i)) * (drho + rho * (T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu));
        v[i] = FUSED ? fma(-omega, v[i] - feq, v[i]) : v[i] - omega * (v[i] - feq);
    }
}

// ------------------------------------------------------------- MRT (D2Q9)
// The moment matrix of the MRT operator (section 3.4, Eq. 18) in this
// lattice's direction order; rows rho, e, epsilon, j_x, q_x, j_y, q_y, p_xx,
// p_xy (the printed p_xy row |c_x c_y| read as the orthogonal c_x c_y), and
// 1 / |row|^2 (the rows are orthogonal: M^{-1} = M^T diag(1 / |row|^2)).
__host__ __device__ constexpr int mrt_m(int r, int j)
{
    constexpr int t[9][9] = {{1, 1, 1, 1, 1, 1, 1, 1, 1},     {-4, -1, -1, -1, -1, 2, 2, 2, 2},
                             {4, -2, -2, -2, -2, 1, 1, 1, 1},  {0, 1, 0, -1, 0, 1, -1, -1, 1},
                             {0, -2, 0, 2, 0, 1, -1, -1, 1},   {0, 0, 1, 0, -1, 1, 1, -1, -1},
                             {0, 0, -2, 0, 2, 1, 1, -1, -1},   {0, 1, -1, 1, -1, 0, 0, 0, 0},
                             {0, 0, 0, 0, 0, 1, -1, 1, -1}};
    return t[r][j];
}

__host__ __device__ constexpr double mrt_inv_norm2(int r)
{
    constexpr double t[9] = {1.0 / 9, 1.0 / 36, 1.0 / 36, 1.0 / 6, 1.0 / 12, 1.0 / 6, 1.0 / 12, 1.0 / 4, 1.0 / 4};
    return t[r];
}

// Relaxation rate of moment row r: 0 for the conserved rho, j_x, j_y (their
// m - m^eq vanishes), s_e, s_eps, s_q for the free rows, omega = 1/tau for the
// stress rows p_xx, p_xy.
template <typename T>
__device__ __forceinline__ T mrt_rate(int r, T omega, const T (&s)[3])
{
    return r == 1 ? s[0] : r == 2 ? s[1] : (r == 4 || r == 6) ? s[2] : (r >= 7 ? omega : T(0));
}

// MRT collision (Eq. 16) in place on shifted populations:
// f* = f - M^{-1} S M (f - f^eq), m^eq = M f^eq with f^eq of Eq. 5.
template <typename T>
__device__ __forceinline__ void collide_mrt(T (&v)[9], T omega, const double (&rates)[3])
{
    using L = Lattice<9>;
    const T s[3] = {T(rates[0]), T(rates[1]), T(rates[2])};
    T drho, rho, u[3];
    moments<9, T>(v, drho, rho, u);
    const T uu = u[0] * u[0] + u[1] * u[1];
    T d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const T cu = cdot<9, T>(i, u);
        d[i] = v[i] - T(L::w(i)) * (drho + rho * (T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu));
    }
    T dm[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        T m = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j)
            if (mrt_m(r, j) != 0) m += T(mrt_m(r, j)) * d[j];
        dm[r] = mrt_rate<T>(r, omega, s) * m * T(mrt_inv_norm2(r));
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        T c = 0;
#pragma unroll
        for (int r = 0; r < 9; ++r)
            if (mrt_m(r, j) != 0 && r != 0 && r != 3 && r != 5) c += T(mrt_m(r, j)) * dm[r];
        v[j] -= c;
    }
}

// BGK (Eq. 4-5) or, on D2Q9 plans with Bc::mrt, MRT.
template <int Q, typename T, bool FUSED = false>
__device__ __forceinline__ void collide_any(T (&v)[Q], T omega, const Bc& bc)
{
    if constexpr (Q == 9) {
        if (bc.mrt) {
            collide_mrt<T>(v, omega, bc.mrt_rates);
            return;
        }
    }
    collide<Q, T, FUSED>(v, omega);
}

// Transpose of the MRT collision at one node, from f^t (moments drho, rho, u)
// and mu = dL/df*: with nu = M^T S diag(1/|row|^2) M mu (nu = omega mu for
// BGK), lambda_k = mu_k - nu_k + A + sum_a (B_a + G_a) (c_ka - u_a) / rho,
// A = sum_j nu_j w_j P_j, B_a = sum_j nu_j w_j rho (3 c_ja + 9 (c_j.u) c_ja - 3 u_a),
// G the Eq. 6 velocity terms.  Returns the node's dL/domega term: only the
// stress rows depend on omega, -sum_{p_xx, p_xy} (M mu)_r (M (f - f^eq))_r / |row_r|^2.
template <typename T>
__device__ __forceinline__ T adjoint_collision_mrt(const T (&f)[9], const T (&mu)[9], T drho, T rho,
                                                   const T (&u)[3], const T (&G)[3], T omega,
                                                   const double (&rates)[3], T (&lam)[9])
{
    using L = Lattice<9>;
    const T s[3] = {T(rates[0]), T(rates[1]), T(rates[2])};
    const T uu = u[0] * u[0] + u[1] * u[1];
    T d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const T cu = cdot<9, T>(i, u);
        d[i] = f[i] - T(L::w(i)) * (drho + rho * (T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu));
    }
    T sm[9], dom = T(0);
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        T mm = 0, md = 0;
#pragma unroll
        for (int j = 0; j < 9; ++j)
            if (mrt_m(r, j) != 0) {
                mm += T(mrt_m(r, j)) * mu[j];
                md += T(mrt_m(r, j)) * d[j];
            }
        if (r >= 7) dom -= mm * md * T(mrt_inv_norm2(r));
        sm[r] = mrt_rate<T>(r, omega, s) * mm * T(mrt_inv_norm2(r));
    }
    T nu[9], A = 0, B[2] = {T(0), T(0)};
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        T c = 0;
#pragma unroll
        for (int r = 0; r < 9; ++r)
            if (mrt_m(r, j) != 0 && r != 0 && r != 3 && r != 5) c += T(mrt_m(r, j)) * sm[r];
        nu[j] = c;
        const T cu = cdot<9, T>(j, u);
        const T wj = T(L::w(j));
        A += c * wj * (T(1) + T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu);
#pragma unroll
        for (int a = 0; a < 2; ++a)
            B[a] += c * wj * rho * (T(3 * L::c(j, a)) + T(9) * cu * T(L::c(j, a)) - T(3) * u[a]);
    }
    const T inv = T(1) / rho;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        T sk = mu[k] - nu[k] + A;
#pragma unroll
        for (int a = 0; a < 2; ++a) sk += (B[a] + G[a]) * inv * (T(L::c(k, a)) - u[a]);
        lam[k] = sk;
    }
    return dom;
}

// Eq. 6 with the wall velocity extrapolated to the pressure plane half a
// link outside the boundary node (Bc::uw_extrap): u_w = u(x_b) + (u(x_b) -
// u(x_b + e)) / 2, with x_b + e the inward neighbour, whose velocity comes from
// its post-collision populations (collision keeps u).  `nb` indexes the
// neighbour in a state of `stride` nodes per direction.
template <int Q, typename T>
__device__ __forceinline__ void extrapolate_wall_velocity(T (&u)[3], const T* __restrict__ src, long long stride,
                                                          long long nb)
{
    T v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = src[(long long)i * stride + nb];
    T drho, rho, ue[3];
    moments<Q, T>(v, drho, rho, ue);
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = T(1.5) * u[a] - T(0.5) * ue[a];
}

// The direction whose link starts at the inward neighbour of a boundary node:
// c = (-1, 0, 0) at the inlet (x - c = x + 1), (+1, 0, 0) at the outlet.
template <int Q>
__host__ __device__ constexpr int inward_dir(bool xin)
{
    return xin ? Lattice<Q>::opp(1) : 1;
}

// Reverse of the extrapolated u_w at one boundary node x_b with inward
// neighbour x_e.  The adjoint kernels take u_w as the node's own velocity u;
// this returns what the extrapolation changes: the velocity terms of x_b
// become 1.5 G(u_w) instead of G(u), x_e gains -0.5 G(u_w), and the inlet
// gradient changes by the difference of d(Eq. 6)/drho_w.  With
// G_a(v) = sum over the node's Eq. 6 links i of lambda_i 2 w_i rho_w (9 (c_i.v) c_ia - 3 v_a),
// the deltas are  d_b[k] = sum_a (1.5 G_a(u_w) - G_a(u)) (c_ka - u_a) / rho(x_b)
// and d_e[k] = sum_a (-0.5 G_a(u_w)) (c_ka - u_e,a) / rho(x_e).
// fb, fe: f^t at x_b and x_e; li[i]: lambda^{t+1}_i(x_b) for the Eq. 6 links
// (bit i of eq6); returns the change of dL/drho_w.
template <int Q, typename T>
__device__ __forceinline__ double adjoint_uw_delta(const T (&fb)[Q], const T (&fe)[Q], const T (&li)[Q],
                                                   uint32_t eq6, T rw, T (&db)[Q], T (&de)[Q])
{
    using L = Lattice<Q>;
    T drb, rhob, ub[3], dre, rhoe, ue[3];
    moments<Q, T>(fb, drb, rhob, ub);
    moments<Q, T>(fe, dre, rhoe, ue);
    T uw[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) uw[a] = T(1.5) * ub[a] - T(0.5) * ue[a];
    const T uub = ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2];
    const T uuw = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
    T Gw[3] = {T(0), T(0), T(0)}, Gu[3] = {T(0), T(0), T(0)};
    double dgrw = 0.0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (!((eq6 >> i) & 1u)) continue;
        const T two_w = T(2.0 * L::w(i));
        const T cw = cdot<Q, T>(i, uw), cb = cdot<Q, T>(i, ub);
        dgrw += (double)(li[i] * two_w * (T(4.5) * (cw * cw - cb * cb) - T(1.5) * (uuw - uub)));
#pragma unroll
        for (int a = 0; a < L::D; ++a) {
            Gw[a] += li[i] * two_w * rw * (T(9) * cw * T(L::c(i, a)) - T(3) * uw[a]);
            Gu[a] += li[i] * two_w * rw * (T(9) * cb * T(L::c(i, a)) - T(3) * ub[a]);
        }
    }
    const T invb = T(1) / rhob, inve = T(1) / rhoe;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        T sb = 0, se = 0;
#pragma unroll
        for (int a = 0; a < L::D; ++a) {
            sb += (T(1.5) * Gw[a] - Gu[a]) * (T(L::c(k, a)) - ub[a]);
            se += T(-0.5) * Gw[a] * (T(L::c(k, a)) - ue[a]);
        }
        db[k] = sb * invb;
        de[k] = se * inve;
    }
    return dgrw;
}

// Transpose of the collision (adjoint.cu, step 3) at one node, from f^t (its
// moments drho, rho, u) and mu = dL/df*: gives lambda^t and returns the
// node's dL/domega term.  G holds the Eq. 6 velocity terms (zero inside).
// DENSE_ROUND: f^eq in that term formed from P (as the vectorised and TMA
// kernels round it) instead of P - 1 summed without its 1.
template <int Q, typename T, bool DENSE_ROUND = false>
__device__ __forceinline__ T adjoint_collision(const T (&f)[Q], const T (&mu)[Q], T drho, T rho, const T (&u)[3],
                                               const T (&G)[3], T omega, T (&lam)[Q], const Bc& bc)
{
    using L = Lattice<Q>;
    if constexpr (Q == 9) {
        if (bc.mrt) return adjoint_collision_mrt<T>(f, mu, drho, rho, u, G, omega, bc.mrt_rates, lam);
    }
    T A = 0, B[3] = {T(0), T(0), T(0)}, domT = 0;
    if constexpr (kByPairs<T>) {
        // dL/domega by pairs of mu (e, o) and of f^eq - f, whose difference is taken before the product:
        // sum mu f^eq - sum mu f would cancel (sum over 20000 nodes: 4e-12 off for 3e-13)
        T uu = 0;
#pragma unroll
        for (int a = 0; a < L::D; ++a) uu += u[a] * u[a];
        const T fbase = drho - T(1.5) * rho * uu, r3 = T(3) * rho, r45 = T(4.5) * rho;
        domT = mu[0] * (T(L::w(0)) * fbase - f[0]);
        // sum_j mu_j w_j times 1, c and c c: A and B are quadratic in u with these coefficients
        T ea[3] = {T(0), T(0), T(0)}, oa[3] = {T(0), T(0), T(0)}, ed[3] = {T(0), T(0), T(0)},
          od[3] = {T(0), T(0), T(0)}, x[3] = {T(0), T(0), T(0)}, sd = 0;
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if (i < L::opp(i)) {
                const T e = mu[i] + mu[L::opp(i)], o = mu[i] - mu[L::opp(i)];
                const T cu = cdot<Q, T>(i, u), wi = T(L::w(i));
                domT += e * (wi * fbase + wi * r45 * cu * cu - T(0.5) * (f[i] + f[L::opp(i)]));
                domT += o * (wi * r3 * cu - T(0.5) * (f[i] - f[L::opp(i)]));
                int n = 0, sg = 1, axes = 0;
#pragma unroll
                for (int a = 0; a < L::D; ++a)
                    if (L::c(i, a) != 0) {
                        ++n;
                        sg *= L::c(i, a);
                        axes += a;
                    }
                if (n == 2) {
                    sd += e;
                    x[axes - 1] = sg > 0 ? x[axes - 1] + e : x[axes - 1] - e;  // xy, xz, yz
                }
#pragma unroll
                for (int a = 0; a < L::D; ++a)
                    if (L::c(i, a) != 0) {
                        if (n == 1) {
                            ea[a] = e;
                            oa[a] = L::c(i, a) > 0 ? o : -o;
                        } else {
                            ed[a] += e;
                            od[a] = L::c(i, a) > 0 ? od[a] + o : od[a] - o;
                        }
                    }
            }
        constexpr T wa = T(L::w(1)), wd = T(L::w(Q - 1));
        T S0 = T(L::w(0)) * mu[0] + wd * sd, S1[3], Su[3], s1u = 0, q = 0;
#pragma unroll
        for (int a = 0; a < L::D; ++a) {
            S0 += wa * ea[a];
            S1[a] = wa * oa[a] + wd * od[a];
            Su[a] = (wa * ea[a] + wd * ed[a]) * u[a];
            s1u += S1[a] * u[a];
        }
        x[0] *= wd;
        Su[0] += x[0] * u[1];
        Su[1] += x[0] * u[0];
        if (L::D == 3) {
            x[1] *= wd;
            x[2] *= wd;
            Su[0] += x[1] * u[2];
            Su[1] += x[2] * u[2];
            Su[2] += x[1] * u[0] + x[2] * u[1];
        }
#pragma unroll
        for (int a = 0; a < L::D; ++a) {
            q += Su[a] * u[a];
            B[a] = rho * (T(3) * (S1[a] - u[a] * S0) + T(9) * Su[a]);
        }
        const T A1 = T(3) * s1u + T(4.5) * q - T(1.5) * uu * S0;
        A = S0 + A1;
    } else {
        const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            const T cu = cdot<Q, T>(j, u);
            const T wj = T(L::w(j));
            const T P = T(1) + T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu;
            const T feq = wj * (drho + rho * (DENSE_ROUND ? P - T(1) : T(3) * cu + T(4.5) * cu * cu - T(1.5) * uu));
            domT += mu[j] * (feq - f[j]);
            A += mu[j] * wj * P;
#pragma unroll
            for (int a = 0; a < L::D; ++a)
                B[a] += mu[j] * wj * rho * (T(3 * L::c(j, a)) + T(9) * cu * T(L::c(j, a)) - T(3) * u[a]);
        }
    }
    const T inv = T(1) / rho;
    T Bt[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) Bt[a] = (omega * B[a] + G[a]) * inv;
    const T keep = T(1) - omega;
    if constexpr (kByPairs<T>) {
        T base = omega * A;
#pragma unroll
        for (int a = 0; a < L::D; ++a) base -= Bt[a] * u[a];
        lam[0] = keep * mu[0] + base;
#pragma unroll
        for (int i = 1; i < Q; ++i)
            if (i < L::opp(i)) {
                const T t = cdot<Q, T>(i, Bt);
                lam[i] = keep * mu[i] + (base + t);
                lam[L::opp(i)] = keep * mu[L::opp(i)] + (base - t);
            }
        return domT;
    }
    const T base = omega * A;
#pragma unroll
    for (int kk = 0; kk < Q; ++kk) {
        T s = keep * mu[kk] + base;
#pragma unroll
        for (int a = 0; a < L::D; ++a) s += Bt[a] * (T(L::c(kk, a)) - u[a]);
        lam[kk] = s;
    }
    return domT;
}

// The wall density of Eq. 6 at a node of column 0 or nx - 1.
__device__ __forceinline__ double wall_density(const Bc& bc, const Geo& g, bool xin, int y, int z)
{
    return xin ? (bc.profile ? bc.rho_in[(long long)z * g.ny + y] : bc.rho_in[0]) : bc.rho_out;
}

// Pull with boundaries: fills v with what node n (at column x) receives; rw
// is its wall density where x = 0 or nx - 1.  Every address is selected and
// then loaded unconditionally (a population that does not come from a
// neighbour starts from the node's own one of the opposite direction), so
// the loads issue together instead of one branch, and one wait, at a time.
template <int Q, typename T>
__device__ __forceinline__ void pull(T (&v)[Q], const T* src, long long n, int x, uint32_t lw, const Geo& g,
                                     const Bc& bc, double rw)
{
    using L = Lattice<Q>;
    const long long N = g.N, plane = (long long)g.nx * g.ny;
    const bool xin = x == 0, xout = x == g.nx - 1;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = L::c(i, 0);
        const bool own = ((lw >> i) & 1u) || (cx == 1 && xin) || (cx == -1 && xout);
        const T* p = own ? src + (long long)L::opp(i) * N : src + (long long)i * N - link_offset<Q>(i, g.nx, plane);
        v[i] = p[n];
    }
    if (xin || xout) {
        // the node's own velocity u(x, t) for Eq. 6, from its local state
        T loc[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) loc[i] = src[(long long)i * N + n];
        T drho, rho, u[3];
        moments<Q, T>(loc, drho, rho, u);
        if (bc.uw_extrap && !((lw >> inward_dir<Q>(xin)) & 1u))
            extrapolate_wall_velocity<Q, T>(u, src, N, xin ? n + 1 : n - 1);
        const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        const T drw = T(rw - 1.0), rwT = T(rw);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int cx = L::c(i, 0);
            if (!((lw >> i) & 1u) && ((cx == 1 && xin) || (cx == -1 && xout))) {
                const T cu = cdot<Q, T>(i, u);
                v[i] = -v[i] + T(2.0 * L::w(i)) * (drw + rwT * (T(4.5) * cu * cu - T(1.5) * uu));
            }
        }
    }
}

// Whether a lane stores its node: fluid nodes, and the solid ones (as zeros)
// of every 32-byte sector that holds a fluid node, so that DRAM never has to
// merge a partly written sector.  Called by whole warps.
__device__ __forceinline__ bool stores_node(bool fluid, bool live, const Geo& g, bool fp32)
{
    const unsigned m = __ballot_sync(0xffffffffu, fluid);
    if (!live) return false;
    const int lane = (int)(threadIdx.x & 31u);
    return !g.skip_sectors || ((m >> (fp32 ? lane & 24 : lane & 28)) & (fp32 ? 0xffu : 0xfu)) != 0u;
}

}  // namespace lbm
