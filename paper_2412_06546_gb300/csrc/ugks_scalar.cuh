// ugks_scalar.cuh -- FP64 arithmetic of one cell or face: primitive variables,
// time integrals of the interface distribution, the slope systems (internal).
#pragma once
#include "ugks_device.cuh"

namespace ugks {

struct Prim {
    double rho, U[MAXD], lam, T;
};

// a / b with ib = 1 / b: the quotient's remainder corrects the product, which
// rounds as the division does in all but rare cases, for a third of its operations
__device__ __forceinline__ double quotient(double a, double b, double ib)
{
    const double q = a * ib;
    return fma(fma(-q, b, a), ib, q);
}

// (with products by the reciprocal, U of random states was off by 0.64e-16 in the
// root mean square, where divisions and this leave 0.43e-16)
__device__ __forceinline__ Prim prim_of(const double *W, int D)
{
    Prim p;
    p.rho = W[0];
    const double ir = 1.0 / W[0];
    double ke = 0.0;
    for (int d = 0; d < MAXD; ++d) p.U[d] = 0.0;
    for (int d = 0; d < D; ++d) {
        p.U[d] = quotient(W[1 + d], W[0], ir);
        ke += p.U[d] * p.U[d];
    }
    p.T = (2.0 / 3.0) * (quotient(W[D + 1], W[0], ir) - 0.5 * ke);
    p.lam = 0.5 / p.T;
    return p;
}

// the same from a primitive row (rho, U, T)
template <int D> __device__ __forceinline__ void set_prim(const double *P, Prim &p)
{
    p.rho = P[0];
    for (int d = 0; d < MAXD; ++d) p.U[d] = d < D ? P[1 + d] : 0.0;
    p.T = P[D + 1];
    p.lam = 0.5 / p.T;
}

constexpr double LOG2E = 1.4426950408889634073599246810018921;

__device__ __forceinline__ double pref_of(double rho, double lam, int D)
{
    const double a = fma(lam, 0.3183098861837907, lam * -1.9678676675182487e-17);     // lam / pi, 1 / pi in two parts
    return D == 2 ? rho * a : rho * a * sqrt(a);
}

// Time integrals of c1..c5 over [0, dt] (Sec. 2.4), written with x = dt/tau,
// E = 1 - e^{-x}:  q1 = dt E/x, q2 = dt^2 (x e^{-x} - E)/x^2, q3 = dt (x - E)/x,
// q4 = dt^2 (2E - x(1 + e^{-x}))/x^2, q5 = dt^2 (x^2/2 - x + E)/x^2.
// Below x = 1/2 the brackets cancel; with phi_n = sum_i (-x)^i / (i + n)! they
// are phi_1, phi_2 - phi_1, x phi_2, -x (phi_2 - 2 phi_3) and x phi_3, where
// phi_4 is summed to rounding, phi_n = 1/n! - x phi_(n+1), and
// phi_2 - phi_1 = -1/2 + x (1/2 - (1 + x) phi_3), phi_2 - 2 phi_3 = 1/6 + x ((x + 2) phi_4 - 1/6).
// (Summing the five series term by term took about 500 FP64 operations; an SM
// retires 1.6 of them per cycle and lane-wise that was half of k_face_fin1.)
// Root mean square errors in units of 1e-16 against 128 bits, with those series
// and these brackets in brackets: q4 1.0 (1.8) below 1/2, 25 (29) at 0.5..0.7,
// q2 1.1 (1.4) and 2.6 (2.6), the others no larger.  E from expm1: 1 - e^{-x}
// costs q1, q2, q3 and q5 a quarter to two thirds there, and q4 a half.
__device__ __forceinline__ void time_integrals(double dt, double x, double q[5])
{
    if (x < 0.5) {
        double f = 2.0;                    // (i + 4)! upwards, folded at compile time
        double c[13];
#pragma unroll
        for (int i = 0; i < 13; ++i) {
            f *= i == 0 ? 12.0 : (double)(i + 4);
            c[i] = (i & 1 ? -1.0 : 1.0) / f;
        }
        double p4 = c[12];
#pragma unroll
        for (int i = 11; i >= 0; --i) p4 = fma(p4, x, c[i]);
        const double p3 = fma(-x, p4, 1.0 / 6.0), p2 = fma(-x, p3, 0.5), p1 = fma(-x, p2, 1.0);
        q[0] = dt * p1;
        q[1] = dt * dt * fma(x, fma(-p3, 1.0 + x, 0.5), -0.5);
        q[2] = dt * x * p2;
        q[3] = -dt * dt * x * fma(x, fma(x + 2.0, p4, -1.0 / 6.0), 1.0 / 6.0);
        q[4] = dt * dt * x * p3;
    } else {
        const double e = exp(-x);
        const double E = -expm1(-x);
        const double ix = 1.0 / x, ix2 = ix * ix;
        q[0] = dt * E * ix;
        q[1] = dt * dt * (x * e - E) * ix2;
        q[2] = dt * (x - E) * ix;
        q[3] = dt * dt * (2.0 * E - x * (1.0 + e)) * ix2;
        q[4] = dt * dt * (0.5 * x * x - x + E) * ix2;
    }
}

// A = L diag(d) L^T of a symmetric positive definite matrix (packed upper
// triangle t(i, j), i <= j); inv[i] = 1 / d_i, L below the diagonal in place of
// the entries.  Five divisions for the factor and none in the solves (the
// Cholesky form took 5 square roots and 50 divisions for the four right-hand
// sides, FP64 operations of about ten instructions each).  A pivot that is not
// positive makes the solutions NaN, as its square root would: such a matrix is no
// set of moments (a velocity set in one plane, a broken state), and the NaN is what
// ugks_check finds.
template <int M> __device__ __forceinline__ constexpr int tri(int i, int j) { return i * M - i * (i - 1) / 2 + (j - i); }

template <int M>
__device__ __forceinline__ void ldl_factor(double *A, double (&inv)[M])
{
#pragma unroll
    for (int j = 0; j < M; ++j) {
        double dj = A[tri<M>(j, j)];
        double w[M];                             // L_jk d_k
#pragma unroll
        for (int k = 0; k < j; ++k) {
            w[k] = A[tri<M>(k, j)];
            const double l = w[k] * inv[k];
            dj -= l * w[k];
        }
        inv[j] = dj > 0.0 ? 1.0 / dj : __longlong_as_double(0x7ff8000000000000ll);
        // A(j, i) for i > j: subtract sum_k L_jk d_k L_ik, kept as L_ij d_j
#pragma unroll
        for (int i = j + 1; i < M; ++i) {
            double t = A[tri<M>(j, i)];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= w[k] * inv[k] * A[tri<M>(k, i)];
            A[tri<M>(j, i)] = t;
        }
    }
    // entries (j, i) hold L_ij d_j: scale to L_ij
#pragma unroll
    for (int j = 0; j < M; ++j)
#pragma unroll
        for (int i = j + 1; i < M; ++i) A[tri<M>(j, i)] *= inv[j];
}

template <int M>
__device__ __forceinline__ void ldl_solve(const double *A, const double (&inv)[M], double *x)
{
#pragma unroll
    for (int i = 1; i < M; ++i)
#pragma unroll
        for (int k = 0; k < i; ++k) x[i] -= A[tri<M>(k, i)] * x[k];
#pragma unroll
    for (int i = 0; i < M; ++i) x[i] *= inv[i];
#pragma unroll
    for (int i = M - 2; i >= 0; --i)
#pragma unroll
        for (int k = i + 1; k < M; ++k) x[i] -= A[tri<M>(i, k)] * x[k];
}

}  // namespace ugks
