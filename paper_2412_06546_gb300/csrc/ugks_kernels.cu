// ugks_kernels.cu -- the CUDA kernels of one UGKS time step (sm_103a).
//
// One step (Algorithm 1 of arXiv:2412.06546, reorganised for the GPU):
//   k_prep        cell records from W^n, q^n; far-field ghost states     (CFL and heat-flux step, Sec. 2.5)
//   k_macro_grad  limited least-squares gradient of W                    (macroscopic reconstruction)
//   k_face_pre    face states W_L, W_R, interface macro gradient, q0     (interface equilibrium)
//   k_face_sum1   half-range moments over the velocity grid -> W0        (Sec. 2.4)
//   k_face_fin1   g0 parameters, tau0, time integrals q1..q5             (Sec. 2.4)
//   k_face_sum2   moments of g0 for the slope systems                    (Sec. 2.4)
//   k_face_fin2   spatial and time slopes of g0                          (Sec. 2.4)
//   k_wall_sum    wall density from zero net mass flux                   (Eq. maxWalldes)
//   k_flux        micro slopes and the outgoing face fluxes               (velocity loop)
//   k_stage1      flux balance, stage 1, moments of the flux residual     (velocity loop, Eq. microS1)
//   k_update_W    W^{n+1} and stage-2 coefficients                       (Eq. macroscopicUpdata)
//   k_collide     stage 2 and the heat flux of f^{n+1}                   (Eq. microS2)
// All per-velocity arithmetic is in T (double or float).  Velocity-moment sums
// are FP64 in the FP64 form.  In the FP32 form the products are FP32 and the
// sums are accumulated in FP64: the face sums from FP32 block partials of at
// most SUM_BLOCK terms per lane (see block_to_fp64), the wall density and the
// heat flux from Kahan-compensated lane sums, the moments of the flux residual
// from double-float lane and warp sums (k_stage1).  Macroscopic scalars (W, the
// equilibrium parameters, the heat flux, the collision coefficients) are
// formed in FP64.
#include "ugks_device.cuh"
#include "ugks_scalar.cuh"
#include "ugks_kernels.h"

#include <algorithm>
#include <type_traits>
#include <cmath>

namespace ugks {

// ------------------------------------------------------------ FP64 helpers (see ugks_scalar.cuh)
// dt / tau of a state, tau = mu_ref T^omega / (rho T) (VHS viscosity, p = rho T)
template <typename T>
__device__ __forceinline__ double dt_over_tau(const DevCase<T> &dc, double rho, double Tmp)
{
    return dc.dt_mu * rho * pow(Tmp, 1.0 - dc.omega);
}

// a record of Maxwellian, Shakhov and collision coefficients (CR_*) of the state
// p with heat flux q; the divisions and the power are the length of the
// kernels that form them (an FP64 operation has a latency of about 70 cycles)
template <typename T, int D>
__device__ __forceinline__ void cell_record(const DevCase<T> &dc, const Prim &p, const double *q, T *r)
{
    const double cc = 0.5 * dt_over_tau(dc, p.rho, p.T);
    const double kappa = 0.8 * (1.0 - dc.Pr) * p.lam * p.lam / p.rho;
    for (int d = 0; d < 3; ++d) r[CR_U + d] = (T)p.U[d];
    r[CR_LAM] = (T)p.lam;
    r[CR_PREF] = (T)pref_of(p.rho, p.lam, D);
    for (int d = 0; d < 3; ++d) r[CR_KQ + d] = d < D ? (T)(kappa * q[d]) : T(0);
    r[CR_C] = (T)cc;
    r[CR_INV] = (T)(1.0 / (1.0 + cc));
    r[CR_NB] = (T)(dc.nxi * p.T);
    r[CR_NL2] = (T)(-p.lam * LOG2E);
}

// ------------------------------------------------------------ launches
// The kernels of a step are launched with programmatic stream serialisation: a
// kernel is set up while the one before it drains, and waits here, before its
// first access to what that one wrote, until the one before has ended and its
// writes are visible.  Every kernel of the step waits, so the order of the whole
// step is kept.  Step times on 13 and more kernels: 20x20 squares x 24^2 119 ->
// 88 us, 2,183 triangles x 30x25 153 -> 117, 2,145 hexahedra x 4,080 446 -> 405.
// Releasing the next kernel's blocks earlier (launch_dependents at a kernel's
// start) was slower, 95, 123 and 416 us: they take the SMs' slots to wait in.
__device__ __forceinline__ void dependency_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
static cudaError_t launch(void (*kernel)(P...), int blocks, int threads, size_t smem, cudaStream_t st, const A &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// ------------------------------------------------------------ batched launches
// The per-case kernels of a step (all but the gather) are written as bodies of
// a block index.  k_X runs them for one case (block index = blockIdx.x);
// k_X_batch runs them for many cases of a batch in one launch.  Its block b
// belongs to the last case i with off[i] <= b (off[] holds the prefix sums of
// the cases' block counts, so a case without blocks is never chosen) and runs
// that case's local block b - off[i]: the same arithmetic as the single-case
// launch.  The case's DevCase is copied into shared memory, where its fields
// are read without aliasing the arrays the kernel writes.
template <typename T>
__device__ __forceinline__ const DevCase<T> &batch_case(const DevCase<T> *__restrict__ cases,
                                                       const int *__restrict__ off, int n, int &bx)
{
    __shared__ __align__(16) unsigned char raw[sizeof(DevCase<T>)];
    static_assert(sizeof(DevCase<T>) % sizeof(int) == 0, "DevCase is copied in 4-byte words");
    const int b = blockIdx.x;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= b) lo = mid;
        else hi = mid - 1;
    }
    bx = b - __ldg(off + lo);
    const int *src = reinterpret_cast<const int *>(cases + lo);
    int *dst = reinterpret_cast<int *>(raw);
    for (int w = threadIdx.x; w < (int)(sizeof(DevCase<T>) / sizeof(int)); w += blockDim.x) dst[w] = __ldg(src + w);
    __syncthreads();
    return *reinterpret_cast<const DevCase<T> *>(raw);
}

// ------------------------------------------------------------ init / moments
template <typename T, int D, int NC>
__global__ void k_init_f(DevCase<T> dc)
{
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= dc.C) return;
    Prim p = prim_of(dc.W + (size_t)c * (D + 2), D);
    T rec[GREC];
    for (int d = 0; d < 3; ++d) rec[GR_U + d] = (T)p.U[d];
    rec[GR_LAM] = (T)p.lam;
    rec[GR_PREF] = (T)pref_of(p.rho, p.lam, D);
    rec[GR_NB] = (T)(dc.nxi * p.T);
    rec[GR_NL2] = (T)(-p.lam * LOG2E);
    const size_t rs = (size_t)NC * dc.nvp;
    for (int k = lane; k < dc.nvp; k += 32) {
        T u[3] = {dc.u[0][k], dc.u[1][k], D == 3 ? dc.u[2][k] : T(0)};
        T H = maxwell_h<T, D>(rec, u);
        dc.f_cur[(size_t)c * rs + k] = H;
        if (NC == 2) dc.f_cur[(size_t)c * rs + dc.nvp + k] = rec[GR_NB] * H;
    }
}

// heat flux q = 1/2 sum_k w c (|c|^2 h + b), c = u - U(W)  (Sec. 2.1)
template <typename T, int D, int NC>
__global__ void k_heatflux(DevCase<T> dc)
{
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= dc.C) return;
    Prim p = prim_of(dc.W + (size_t)c * (D + 2), D);
    T U[3] = {(T)p.U[0], (T)p.U[1], (T)p.U[2]};
    const size_t rs = (size_t)NC * dc.nvp;
    CSum<T> acc[D];
    for (int k = lane; k < dc.nvp; k += 32) {
        T cc[D], c2 = 0;
        for (int d = 0; d < D; ++d) {
            cc[d] = dc.u[d][k] - U[d];
            c2 += cc[d] * cc[d];
        }
        T h = dc.f_cur[(size_t)c * rs + k];
        T e = c2 * h + (NC == 2 ? dc.f_cur[(size_t)c * rs + dc.nvp + k] : T(0));
        T we = dc.w[k] * e;
        for (int d = 0; d < D; ++d) acc[d].add(cc[d] * we);
    }
    for (int d = 0; d < D; ++d) {
        const double s = warp_sum(acc[d].value());
        if (lane == 0) dc.q[(size_t)c * D + d] = 0.5 * s;
    }
}

// ------------------------------------------------------------ k_prep
template <typename T, int D, int NC>
__device__ __forceinline__ void prep_body(const DevCase<T> &dc, const int bx)
{
    const int t = bx * blockDim.x + threadIdx.x;
    constexpr int M = D + 2;
    if (t < dc.C) {
        const int c = t;
        Prim p = prim_of(dc.W + (size_t)c * M, D);
        if (!(p.rho > 0.0) || !(p.T > 0.0)) atomicOr(dc.flags, 1);
        double *Pc = dc.prim + (size_t)c * M;
        Pc[0] = p.rho;
        for (int d = 0; d < D; ++d) Pc[1 + d] = p.U[d];
        Pc[D + 1] = p.T;
        cell_record<T, D>(dc, p, dc.q + (size_t)c * D, dc.crec + (size_t)c * CREC);
        return;
    }
    const int g = t - dc.C;
    if (g >= dc.G) return;
    // far-field ghost (Sec. 2.5): free stream where it enters (U_inf . n < 0),
    // zero-gradient extrapolation of the cell state elsewhere
    const int f = dc.gface[g];
    const int own = dc.fL[f];
    double un = __dmul_rn(dc.inf_W[1] / dc.inf_W[0], dc.fn_d[(size_t)f * D]);
    un = __dadd_rn(un, __dmul_rn(dc.inf_W[2] / dc.inf_W[0], dc.fn_d[(size_t)f * D + 1]));
    if (D == 3) un = __dadd_rn(un, __dmul_rn(dc.inf_W[3] / dc.inf_W[0], dc.fn_d[(size_t)f * D + 2]));
    double *Wg = dc.Wg + (size_t)g * M;
    for (int m = 0; m < M; ++m) Wg[m] = un < 0.0 ? dc.inf_W[m] : dc.W[(size_t)own * M + m];
    Prim p = prim_of(Wg, D);
    double *Pg = dc.primg + (size_t)g * M;
    Pg[0] = p.rho;
    for (int d = 0; d < D; ++d) Pg[1 + d] = p.U[d];
    Pg[D + 1] = p.T;
    T *r = dc.grec + (size_t)g * GREC;
    for (int d = 0; d < 3; ++d) r[GR_U + d] = (T)p.U[d];
    r[GR_LAM] = (T)p.lam;
    r[GR_PREF] = (T)pref_of(p.rho, p.lam, D);
    r[GR_NB] = (T)(dc.nxi * p.T);
    r[GR_NL2] = (T)(-p.lam * LOG2E);
}

template <typename T, int D, int NC>
__global__ void k_prep(DevCase<T> dc)
{
    dependency_wait();
    prep_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_prep_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    prep_body<T, D, NC>(dc, bx);
}

// ------------------------------------------------------------ k_macro_grad
// limited least-squares gradients of the primitive variables (rho, U, T) and
// the conserved-variable gradient obtained from them by the chain rule
template <typename T, int D, int NC>
__device__ __forceinline__ void macro_grad_body(const DevCase<T> &dc, const int bx)
{
    const int c = bx * blockDim.x + threadIdx.x;
    constexpr int M = D + 2;
    if (c >= dc.C) return;
    const double *Pc = dc.prim + (size_t)c * M;
    const int q0 = dc.nb_ptr[c], q1 = dc.nb_ptr[c + 1];
    const int s0 = dc.cf_ptr[c], s1 = dc.cf_ptr[c + 1];
    const double e2 = dc.eps2_d[c];
    // every neighbour's row is read once for all components; the limiter's
    // factor is taken at the largest and the most negative offset, as in
    // cell_slope, with one division per component
    double gp[D][M], vi[M];
    Extrema<double> ex[M], d2x[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        vi[m] = Pc[m];
        ex[m].set(vi[m]);
        d2x[m].set(0.0);
#pragma unroll
        for (int d = 0; d < D; ++d) gp[d][m] = 0.0;
    }
    for (int q = q0; q < q1; ++q) {
        const int id = dc.nb_id[q];
        const double *row = id >= 0 ? dc.prim + (size_t)id * M : dc.primg + (size_t)(-id - 1) * M;
        double a[D];
#pragma unroll
        for (int d = 0; d < D; ++d) a[d] = dc.nb_a_d[(size_t)q * D + d];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const double vj = row[m], df = vj - vi[m];
#pragma unroll
            for (int d = 0; d < D; ++d) gp[d][m] += a[d] * df;
            ex[m].add(vj);
        }
    }
    if (dc.limiter) {
        for (int s = s0; s < s1; ++s) {
            double r[D];
#pragma unroll
            for (int d = 0; d < D; ++d) r[d] = dc.cf_r_d[(size_t)s * D + d];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                double d2 = 0.0;
#pragma unroll
                for (int d = 0; d < D; ++d) d2 += gp[d][m] * r[d];
                d2x[m].add(d2);
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            double num[2], den[2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const double d1 = (s ? ex[m].bottom() : ex[m].top()) - vi[m];
                const double d2 = s ? d2x[m].bottom() : d2x[m].top();
                const double a2 = d1 * d1 + e2;
                num[s] = a2 + 2.0 * d1 * d2;
                den[s] = a2 + d2 * (2.0 * d2 + d1);
            }
            const double phi = min_ratio(num[0], den[0], num[1], den[1]);
#pragma unroll
            for (int d = 0; d < D; ++d) gp[d][m] *= phi;
        }
    }
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll
        for (int m = 0; m < M; ++m) dc.gradprim[((size_t)c * D + d) * M + m] = gp[d][m];
    double uu = 0.0;
    for (int e = 0; e < D; ++e) uu += Pc[1 + e] * Pc[1 + e];
    for (int d = 0; d < D; ++d) {
        double *gw = dc.gradW + ((size_t)c * D + d) * M;
        double udu = 0.0;
        gw[0] = gp[d][0];
        for (int e = 0; e < D; ++e) {
            gw[1 + e] = Pc[1 + e] * gp[d][0] + Pc[0] * gp[d][1 + e];
            udu += Pc[1 + e] * gp[d][1 + e];
        }
        gw[D + 1] = gp[d][0] * (0.5 * uu + 1.5 * Pc[D + 1]) + Pc[0] * (udu + 1.5 * gp[d][D + 1]);
    }
}

template <typename T, int D, int NC>
__global__ void k_macro_grad(DevCase<T> dc)
{
    dependency_wait();
    macro_grad_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_macro_grad_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    macro_grad_body<T, D, NC>(dc, bx);
}

// ------------------------------------------------------------ face pass
// face state P_c + gradP_c . r in primitive variables (rho, U, T); the cell
// average is used if rho or T would not be positive
template <int D>
__device__ __forceinline__ void face_state(const double *P, const double *gradP, int c, const double *r, Prim &p)
{
    constexpr int M = D + 2;
    double pf[M], av[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        double s = av[m] = P[(size_t)c * M + m];
#pragma unroll
        for (int d = 0; d < D; ++d) s += gradP[((size_t)c * D + d) * M + m] * r[d];
        pf[m] = s;
    }
    const bool ok = pf[0] > 0.0 && pf[D + 1] > 0.0;
#pragma unroll
    for (int m = 0; m < M; ++m) pf[m] = ok ? pf[m] : av[m];
    set_prim<D>(pf, p);
}

template <typename T, int D>
__device__ __forceinline__ void side_record(const Prim &p, double nxi, T *rec)
{
    for (int d = 0; d < 3; ++d) rec[GR_U + d] = (T)p.U[d];
    rec[GR_LAM] = (T)p.lam;
    rec[GR_PREF] = (T)pref_of(p.rho, p.lam, D);
    rec[GR_NB] = (T)(nxi * p.T);
    rec[GR_NL2] = (T)(-p.lam * LOG2E);
}

// Analytic half-range moments of the Maxwellian p over u.n > 0 (sigma = +1)
// or u.n < 0 (sigma = -1), added into the conserved components W.  Along the
// unit normal, with U_n = U.n and e = sigma exp(-lam U_n^2) / (2 sqrt(pi lam)):
// <1> = erfc(-sigma sqrt(lam) U_n) / 2, <u_n> = U_n <1> + e and
// <u_n^2> = (U_n^2 + 1/(2 lam)) <1> + U_n e; the D-1 tangential components
// (mean U - U_n n) and the 3-D internal ones are full Gaussians of variance
// 1/(2 lam) each, two components in all.
template <int D>
__device__ void add_half_range(const Prim &p, const double n[D], double sigma, double *W)
{
    double Un = 0.0;
    for (int d = 0; d < D; ++d) Un += p.U[d] * n[d];
    const double m0 = 0.5 * erfc(-sigma * sqrt(p.lam) * Un);
    const double e = sigma * exp(-p.lam * Un * Un) / (2.0 * sqrt(3.14159265358979323846 * p.lam));
    const double m1 = Un * m0 + e;
    const double m2 = (Un * Un + 0.5 / p.lam) * m0 + Un * e;
    double Ut2 = 0.0;
    W[0] += p.rho * m0;
    for (int d = 0; d < D; ++d) {
        const double Ut = p.U[d] - Un * n[d];
        Ut2 += Ut * Ut;
        W[1 + d] += p.rho * (m1 * n[d] + Ut * m0);
    }
    W[D + 1] += 0.5 * p.rho * (m2 + (Ut2 + 1.0 / p.lam) * m0);
}

template <typename T, int D, int NC>
__device__ __forceinline__ void face_pre_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * blockDim.x + threadIdx.x;
    constexpr int M = D + 2;
    if (f >= dc.F) return;
    const int typ = dc.ftype[f];
    if (typ == FT_WALL) return;
    const int L = dc.fL[f];
    double rL[D], rR[D];
    Prim pL, pR;
    for (int d = 0; d < D; ++d) rL[d] = dc.frL_d[(size_t)f * D + d];
    face_state<D>(dc.prim, dc.gradprim, L, rL, pL);
    double *dW0 = dc.fdW0 + (size_t)f * D * M;
    double *q0 = dc.fq0 + (size_t)f * D;
    if (typ == FT_FARFIELD) {
        set_prim<D>(dc.primg + (size_t)dc.faux[f] * M, pR);
        for (int d = 0; d < D; ++d) {
            for (int m = 0; m < M; ++m) dW0[d * M + m] = 0.5 * dc.gradW[((size_t)L * D + d) * M + m];
            q0[d] = 0.5 * dc.q[(size_t)L * D + d];
        }
    } else {
        const int R = dc.fR[f];
        for (int d = 0; d < D; ++d) rR[d] = dc.frR_d[(size_t)f * D + d];
        face_state<D>(dc.prim, dc.gradprim, R, rR, pR);
        for (int d = 0; d < D; ++d) {
            for (int m = 0; m < M; ++m)
                dW0[d * M + m] = 0.5 * (dc.gradW[((size_t)L * D + d) * M + m] + dc.gradW[((size_t)R * D + d) * M + m]);
            q0[d] = 0.5 * (dc.q[(size_t)L * D + d] + dc.q[(size_t)R * D + d]);
        }
    }
    side_record<T, D>(pL, dc.nxi, dc.fside + (size_t)f * 2 * GREC);
    side_record<T, D>(pR, dc.nxi, dc.fside + (size_t)f * 2 * GREC + GREC);
    for (int d = 0; d < D; ++d) dc.fUref[(size_t)f * D + d] = 0.5 * (pL.U[d] + pR.U[d]);
    if (dc.w0_analytic) {
        // W0 from the analytic half-range moments (continuous velocity space),
        // stored centred at U_ref as the discrete sums of k_face_sum1 are
        double n[D], W0[M];
        for (int d = 0; d < D; ++d) n[d] = dc.fn_d[(size_t)f * D + d];
        for (int m = 0; m < M; ++m) W0[m] = 0.0;
        add_half_range<D>(pL, n, 1.0, W0);
        add_half_range<D>(pR, n, -1.0, W0);
        double *S = dc.fsum1 + (size_t)f * M;
        double uS = 0.0, uu = 0.0;
        S[0] = W0[0];
        for (int d = 0; d < D; ++d) {
            const double Ur = dc.fUref[(size_t)f * D + d];
            S[1 + d] = W0[1 + d] - Ur * W0[0];
            uS += Ur * W0[1 + d];
            uu += Ur * Ur;
        }
        S[D + 1] = W0[D + 1] - uS + 0.5 * uu * W0[0];
    }
}

template <typename T, int D, int NC>
__global__ void k_face_pre(DevCase<T> dc)
{
    dependency_wait();
    face_pre_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_pre_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_pre_body<T, D, NC>(dc, bx);
}

// half-range moments: sum_k w psi_c [H(u_n) g_L + (1 - H(u_n)) g_R], centred at U_ref
template <typename T, int D, int NC>
__device__ __forceinline__ void face_sum1_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    constexpr int M = D + 2;
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    // both side records in registers; a velocity selects its upwind side's
    // values instead of loading them through a selected pointer
    T sL[GREC], sR[GREC];
#pragma unroll
    for (int i = 0; i < GREC; ++i) {
        sL[i] = dc.fside[(size_t)f * 2 * GREC + i];
        sR[i] = dc.fside[(size_t)f * 2 * GREC + GREC + i];
    }
    T n[D], Ur[D];
    for (int d = 0; d < D; ++d) {
        n[d] = dc.fn[(size_t)f * D + d];
        Ur[d] = (T)dc.fUref[(size_t)f * D + d];
    }
    // the terms of velocity k, added into a[0..M)
    auto terms = [&](int k, T *a) {
        T u[3], wk;
        load_uw(dc.uw, k, u, wk);
        T un = normal_velocity<T, D>(u, n);
        T h, b;
        if (un != T(0)) {
            T s[GREC];
#pragma unroll
            for (int i = 0; i < GREC; ++i) s[i] = un > T(0) ? sL[i] : sR[i];
            h = maxwell_h<T, D>(s, u);
            b = s[GR_NB] * h;
        } else {
            T hl = maxwell_h<T, D>(sL, u), hr = maxwell_h<T, D>(sR, u);
            h = T(0.5) * hl + T(0.5) * hr;
            b = T(0.5) * sL[GR_NB] * hl + T(0.5) * sR[GR_NB] * hr;
        }
        T c2 = 0;
        T wh = wk * h;
        a[0] += wh;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            T c = u[d] - Ur[d];
            c2 += c * c;
            a[1 + d] += c * wh;
        }
        a[D + 1] += T(0.5) * wk * (c2 * h + b);
    };
    if constexpr (std::is_same<T, float>::value) {
        // blocked sums accumulated in FP64 (SUM_BLOCK terms per lane per block)
        constexpr int NP = M <= 4 ? 4 : 8;
        double acc = 0.0;
        for (int k0 = lane; k0 < dc.nvp; k0 += 32 * SUM_BLOCK) {
            float blk[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) blk[i] = 0.f;
#pragma unroll 4
            for (int j = 0; j < SUM_BLOCK; ++j) {
                const int k = k0 + 32 * j;
                if (k >= dc.nvp) break;              // uniform: nvp is a multiple of 32
                terms(k, blk);
            }
            acc += block_to_fp64<NP>(blk);
        }
        const int vi = lane >> (NP == 4 ? 3 : 2);
        if ((lane & (NP == 4 ? 7 : 3)) == 0 && vi < M) dc.fsum1[(size_t)f * M + vi] = acc;
    } else {
        T acc[M];
#pragma unroll
        for (int m = 0; m < M; ++m) acc[m] = 0;
        for (int k = lane; k < dc.nvp; k += 32) terms(k, acc);
        for (int m = 0; m < M; ++m) {
            const double sm = warp_sum(acc[m]);
            if (lane == 0) dc.fsum1[(size_t)f * M + m] = sm;
        }
    }
}

template <typename T, int D, int NC>
__global__ void k_face_sum1(DevCase<T> dc)
{
    dependency_wait();
    face_sum1_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_sum1_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_sum1_body<T, D, NC>(dc, bx);
}

// k_face_sum1 on a tensor-product velocity grid.  With the face-state
// Maxwellians factored by axis, the half-range sums become, for every point of
// the outer axes, sums over a contiguous range of the last axis: u.n, rounded
// as everywhere (no contraction, last term added last), is monotone along that
// axis when its nodes ascend.  Prefix sums of the last axis' 1-D moments give
// every range in O(1); the range ends come from binary searches on the exact
// u.n, and nodes with u.n = 0 keep their half weight on both sides.  One warp
// per face; the prefix sums live in shared memory, 2 sides x 3 powers x
// (NL + 1) doubles per warp.
constexpr int SUM1_SEP_WARPS = 4;

template <typename T, int D, int NC>
__device__ __forceinline__ void face_sum1_sep_body(const DevCase<T> &dc, const int bx)
{
    extern __shared__ __align__(16) unsigned char psum_raw[];
    T *psum = reinterpret_cast<T *>(psum_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int f = bx * SUM1_SEP_WARPS + warp;
    constexpr int M = D + 2;
    constexpr int L = D - 1;                 // the prefix-sum axis
    const int NL = dc.cart_n[L];
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    T *P = psum + (size_t)warp * 6 * (NL + 1);
    const T *side[2] = {dc.fside + (size_t)f * 2 * GREC, dc.fside + (size_t)f * 2 * GREC + GREC};
    T n[D], Ur[D];
    for (int d = 0; d < D; ++d) {
        n[d] = dc.fn[(size_t)f * D + d];
        Ur[d] = (T)dc.fUref[(size_t)f * D + d];
    }
    // prefix sums over the last axis of w g (u - Ur)^p, p = 0, 1, 2, per side
    // (at most SUM1_SEP_MAX_NL = 512 terms each: one block of the FP32 form's
    // blocked sums)
    for (int s = 0; s < 2; ++s) {
        const T *r = side[s];
        T *Ps = P + s * 3 * (NL + 1);
        if (lane == 0) Ps[0] = Ps[NL + 1] = Ps[2 * (NL + 1)] = T(0);
        T carry[3] = {0, 0, 0};
        for (int j0 = 0; j0 < NL; j0 += 32) {
            const int j = j0 + lane;
            T v[3] = {0, 0, 0};
            if (j < NL) {
                const T a = dc.axis[L][j];
                const T dv = a - r[GR_U + L];
                const T g = dc.axw[L][j] * gauss<T>(r[GR_LAM], r[GR_NL2], dv * dv);
                const T c = a - Ur[L];
                v[0] = g;
                v[1] = g * c;
                v[2] = g * c * c;
            }
#pragma unroll
            for (int p = 0; p < 3; ++p) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const T t = __shfl_up_sync(0xffffffffu, v[p], o);
                    if (lane >= o) v[p] += t;
                }
                if (j < NL) Ps[p * (NL + 1) + j + 1] = carry[p] + v[p];
                carry[p] += __shfl_sync(0xffffffffu, v[p], 31);
            }
        }
    }
    __syncwarp();
    const T nl = n[L];
    const T *aL = dc.axis[L];
    int nouter = dc.cart_n[0];
    if (D == 3) nouter *= dc.cart_n[1];
    // the terms of outer node o (both sides), added into acc[0..M)
    auto terms = [&](int o, T *acc) {
        int idx[2] = {o % dc.cart_n[0], D == 3 ? o / dc.cart_n[0] : 0};
        T uo[2];
        uo[0] = dc.axis[0][idx[0]];
        uo[1] = D == 3 ? dc.axis[1][idx[1]] : T(0);
        T sp = mul_rn(uo[0], n[0]);
        if (D == 3) sp = add_rn(sp, mul_rn(uo[1], n[1]));
        // [ja, jb): u.n = 0; ascending u.n (nl >= 0): u.n < 0 on [0, ja), > 0 on [jb, NL);
        // descending (nl < 0): u.n > 0 on [0, ja), < 0 on [jb, NL)
        auto first = [&](int mode) {
            int lo = 0, hi = NL;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                const T v = add_rn(sp, mul_rn(aL[mid], nl));
                const bool t = mode == 0 ? v >= T(0) : mode == 1 ? v > T(0) : mode == 2 ? v <= T(0) : v < T(0);
                if (t) hi = mid;
                else lo = mid + 1;
            }
            return lo;
        };
        const bool asc = nl >= T(0);
        const int ja = first(asc ? 0 : 2), jb = first(asc ? 1 : 3);
        T co2 = 0, co[2];
#pragma unroll
        for (int e = 0; e < D - 1; ++e) {
            co[e] = uo[e] - Ur[e];
            co2 += co[e] * co[e];
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T *r = side[s];
            const T *Ps = P + s * 3 * (NL + 1);
            const bool lo_side = (s == 0) != asc;        // the full range starts at 0
            const int f0 = lo_side ? 0 : jb, f1 = lo_side ? ja : NL;
            T Y[3];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                const T *Pp = Ps + p * (NL + 1);
                Y[p] = (Pp[f1] - Pp[f0]) + T(0.5) * (Pp[jb] - Pp[ja]);
            }
            T go = r[GR_PREF];
#pragma unroll
            for (int e = 0; e < D - 1; ++e) {
                const T dv = uo[e] - r[GR_U + e];
                go *= dc.axw[e][idx[e]] * gauss<T>(r[GR_LAM], r[GR_NL2], dv * dv);
            }
            const T g = go;
            acc[0] += g * Y[0];
#pragma unroll
            for (int e = 0; e < D - 1; ++e) acc[1 + e] += g * co[e] * Y[0];
            acc[1 + L] += g * Y[1];
            acc[D + 1] += T(0.5) * g * (co2 * Y[0] + Y[2] + r[GR_NB] * Y[0]);
        }
    };
    if constexpr (std::is_same<T, float>::value) {
        // blocked sums accumulated in FP64 (SUM_BLOCK outer nodes per lane per block)
        constexpr int NP = M <= 4 ? 4 : 8;
        double acc = 0.0;
        for (int o0 = 0; o0 < nouter; o0 += 32 * SUM_BLOCK) {
            float blk[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) blk[i] = 0.f;
            for (int j = 0; j < SUM_BLOCK; ++j) {
                const int o = o0 + 32 * j + lane;
                if (o >= nouter) break;
                terms(o, blk);
            }
            acc += block_to_fp64<NP>(blk);
        }
        const int vi = lane >> (NP == 4 ? 3 : 2);
        if ((lane & (NP == 4 ? 7 : 3)) == 0 && vi < M) dc.fsum1[(size_t)f * M + vi] = acc;
    } else {
        T acc[M];
#pragma unroll
        for (int m = 0; m < M; ++m) acc[m] = 0;
        for (int o = lane; o < nouter; o += 32) terms(o, acc);
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const double sm = warp_sum(acc[m]);
            if (lane == 0) dc.fsum1[(size_t)f * M + m] = sm;
        }
    }
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(32 * SUM1_SEP_WARPS) k_face_sum1_sep(DevCase<T> dc)
{
    dependency_wait();
    face_sum1_sep_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(32 * SUM1_SEP_WARPS) k_face_sum1_sep_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_sum1_sep_body<T, D, NC>(dc, bx);
}

template <typename T, int D, int NC>
__device__ __forceinline__ void face_fin1_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * blockDim.x + threadIdx.x;
    constexpr int M = D + 2;
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    const double *S = dc.fsum1 + (size_t)f * M;
    const double *Ur = dc.fUref + (size_t)f * D;
    // shift the centred sums back: psi = L psi_c with c = u - U_ref
    double W0[M];
    W0[0] = S[0];
    double uS = 0.0, uu = 0.0;
    for (int d = 0; d < D; ++d) {
        W0[1 + d] = S[1 + d] + Ur[d] * S[0];
        uS += Ur[d] * S[1 + d];
        uu += Ur[d] * Ur[d];
    }
    W0[D + 1] = S[D + 1] + uS + 0.5 * uu * S[0];
    Prim p = prim_of(W0, D);
    double *pp = dc.fprim0 + (size_t)f * M;
    pp[0] = p.rho;
    for (int d = 0; d < D; ++d) pp[1 + d] = p.U[d];
    pp[D + 1] = p.lam;
    T *r = dc.frec + (size_t)f * FREC;
    for (int d = 0; d < 3; ++d) r[FR_U + d] = (T)p.U[d];
    r[FR_LAM] = (T)p.lam;
    r[FR_PREF] = (T)pref_of(p.rho, p.lam, D);
    r[FR_NL2] = (T)(-p.lam * LOG2E);
    time_integrals(dc.dt, dt_over_tau(dc, p.rho, p.T), dc.fqs + (size_t)f * 5);   // FP64, for k_face_fin2
}

template <typename T, int D, int NC>
__global__ void k_face_fin1(DevCase<T> dc)
{
    dependency_wait();
    face_fin1_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_fin1_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_fin1_body<T, D, NC>(dc, bx);
}

// number of unique entries of a symmetric (D+2)x(D+2) matrix
template <int D> struct Sym { static constexpr int N = (D + 2) * (D + 3) / 2; };

// The sums the slope systems need on an unstructured velocity set are the
// entries of sum_k w_k H0 psi_c psi_c^T and of the same with a factor c_d, with
// psi_c = (1, c, psi_E) and, after integrating the internal degrees of freedom,
// psi_E = (|c|^2 + nb) / 2 and psi_E^2 = (|c|^4 + 2 nb |c|^2 + xb) / 4.  Every
// one of them is a combination of fewer distinct moments R of w H0:
//   c^a for |a| <= 3 (1, c_d, pairs d <= e, triples d <= e <= g),
//   |c|^2 c_d c_e (d <= e), |c|^4 and |c|^4 c_d,
// 30 in 3D against 60 entries (16 against 30 in 2D).  k_face_sum2 reduces R;
// k_face_fin2 forms the entries in FP64 (mono_moments).
template <int D> struct Mono {
    static constexpr int N2 = D * (D + 1) / 2;                // pairs d <= e
    static constexpr int N3 = D * (D + 1) * (D + 2) / 6;      // triples d <= e <= g
    static constexpr int O1 = 1, O2 = O1 + D, O3 = O2 + N2, OQ2 = O3 + N3, OQ4 = OQ2 + N2, N = OQ4 + 1 + D;
};

// position of the pair d <= e (row-major upper triangle) and of the triple
// d <= e <= g (lexicographic), the order in which k_face_sum2 stores them
__host__ __device__ constexpr int pair_index(int D, int d, int e) { return d * D - d * (d - 1) / 2 + (e - d); }

__host__ __device__ constexpr int triple_index(int D, int d, int e, int g)
{
    // triples with a first index below d, then with (d, b < e), then (d, e, c < g)
    return (D * (D + 1) * (D + 2) - (D - d) * (D - d + 1) * (D - d + 2)) / 6 +
           ((D - d) * (D - d + 1) - (D - e) * (D - e + 1)) / 2 + (g - e);
}

// sum w H0 c_a c_b (c_g) from R, indices in any order
template <int D> __device__ __forceinline__ double mono2(const double *R, int a, int b)
{
    return R[Mono<D>::O2 + (a <= b ? pair_index(D, a, b) : pair_index(D, b, a))];
}

template <int D> __device__ __forceinline__ double mono3(const double *R, int a, int b, int g)
{
    int x = a, y = b, z = g, t;
    if (x > y) { t = x; x = y; y = t; }
    if (y > z) { t = y; y = z; z = t; }
    if (x > y) { t = x; x = y; y = t; }
    return R[Mono<D>::O3 + triple_index(D, x, y, z)];
}

// the k_face_sum2 entries (layout of sep_moments) from the distinct moments R
template <int D>
__device__ void mono_moments(const double *R, double nb, double xb, double *S)
{
    using Mo = Mono<D>;
    constexpr int NS = Sym<D>::N;
    constexpr int M = D + 2;
    double s2 = 0.0, s2c[D];                        // sum |c|^2 and sum |c|^2 c_d
#pragma unroll
    for (int e = 0; e < D; ++e) s2 += mono2<D>(R, e, e);
#pragma unroll
    for (int d = 0; d < D; ++d) {
        s2c[d] = 0.0;
#pragma unroll
        for (int e = 0; e < D; ++e) s2c[d] += mono3<D>(R, d, e, e);
    }
    int t = 0;
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
        for (int j = i; j < M; ++j) {
            double base, bc[D];
            if (j < M - 1) {                        // psi_i psi_j: a monomial of degree <= 2
                if (i == 0 && j == 0) {
                    base = R[0];
#pragma unroll
                    for (int d = 0; d < D; ++d) bc[d] = R[Mo::O1 + d];
                } else if (i == 0) {
                    base = R[Mo::O1 + j - 1];
#pragma unroll
                    for (int d = 0; d < D; ++d) bc[d] = mono2<D>(R, j - 1, d);
                } else {
                    base = mono2<D>(R, i - 1, j - 1);
#pragma unroll
                    for (int d = 0; d < D; ++d) bc[d] = mono3<D>(R, i - 1, j - 1, d);
                }
            } else if (i < M - 1) {                 // psi_i psi_E
                if (i == 0) {
                    base = 0.5 * (s2 + nb * R[0]);
#pragma unroll
                    for (int d = 0; d < D; ++d) bc[d] = 0.5 * (s2c[d] + nb * R[Mo::O1 + d]);
                } else {
                    const int a = i - 1;
                    base = 0.5 * (s2c[a] + nb * R[Mo::O1 + a]);
#pragma unroll
                    for (int d = 0; d < D; ++d)
                        bc[d] = 0.5 * (R[Mo::OQ2 + (a <= d ? pair_index(D, a, d) : pair_index(D, d, a))] +
                                       nb * mono2<D>(R, a, d));
                }
            } else {                                // psi_E^2
                base = 0.25 * (R[Mo::OQ4] + 2.0 * nb * s2 + xb * R[0]);
#pragma unroll
                for (int d = 0; d < D; ++d) bc[d] = 0.25 * (R[Mo::OQ4 + 1 + d] + 2.0 * nb * s2c[d] + xb * R[Mo::O1 + d]);
            }
            S[t] = base;
#pragma unroll
            for (int d = 0; d < D; ++d) S[NS * (1 + d) + t] = bc[d];
            ++t;
        }
}

template <typename T, int D, int NC>
__device__ __forceinline__ void face_sum2_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    constexpr int NS = Sym<D>::N;
    constexpr int S2 = NS * (D + 1);
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    const T *fr = dc.frec + (size_t)f * FREC;
    T U0[D];
#pragma unroll
    for (int d = 0; d < D; ++d) U0[d] = fr[FR_U + d];
    const T lam = fr[FR_LAM], pref = fr[FR_PREF], nl2 = fr[FR_NL2];
    using Mo = Mono<D>;
    // the distinct monomial moments of velocity k, added into r[0..Mo::N)
    auto terms = [&](int k, T *r) {
        T uk[3], wk, c[D], c2 = 0;
        load_uw(dc.uw, k, uk, wk);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            c[d] = uk[d] - U0[d];
            c2 += c[d] * c[d];
        }
        const T a = wk * pref * gauss<T>(lam, nl2, c2);
        r[0] += a;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const T a1 = a * c[d];
            r[Mo::O1 + d] += a1;
#pragma unroll
            for (int e = d; e < D; ++e) {
                const T a2 = a1 * c[e];
                r[Mo::O2 + pair_index(D, d, e)] += a2;
                r[Mo::OQ2 + pair_index(D, d, e)] += a2 * c2;
#pragma unroll
                for (int g = e; g < D; ++g) r[Mo::O3 + triple_index(D, d, e, g)] += a2 * c[g];
            }
        }
        const T a4 = a * c2 * c2;
        r[Mo::OQ4] += a4;
#pragma unroll
        for (int d = 0; d < D; ++d) r[Mo::OQ4 + 1 + d] += a4 * c[d];
    };
    if constexpr (std::is_same<T, float>::value) {
        // blocked sums accumulated in FP64 (SUM_BLOCK terms per lane per block)
        constexpr int NP = Mo::N <= 16 ? 16 : 32;
        double acc = 0.0;
        for (int k0 = lane; k0 < dc.nvp; k0 += 32 * SUM_BLOCK) {
            float blk[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) blk[i] = 0.f;
#pragma unroll 2
            for (int j = 0; j < SUM_BLOCK; ++j) {
                const int k = k0 + 32 * j;
                if (k >= dc.nvp) break;              // uniform: nvp is a multiple of 32
                terms(k, blk);
            }
            acc += block_to_fp64<NP>(blk);
        }
        const int vi = lane >> (NP == 16 ? 1 : 0);
        if ((lane & (NP == 16 ? 1 : 0)) == 0 && vi < Mo::N) dc.fsum2[(size_t)f * S2 + vi] = acc;
    } else {
        T r[Mo::N];
#pragma unroll
        for (int i = 0; i < Mo::N; ++i) r[i] = 0;
        for (int k = lane; k < dc.nvp; k += 32) terms(k, r);
#pragma unroll
        for (int i = 0; i < Mo::N; ++i) {
            const double sm = warp_sum(r[i]);
            if (lane == 0) dc.fsum2[(size_t)f * S2 + i] = sm;
        }
    }
}

template <typename T, int D, int NC>
__global__ void k_face_sum2(DevCase<T> dc)
{
    dependency_wait();
    face_sum2_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_sum2_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_sum2_body<T, D, NC>(dc, bx);
}

// The same sums as k_face_sum2 on a tensor-product velocity grid, where
// u_k = (x_i, y_j[, z_l]) and w_k = wx_i wy_j [wz_l]: every moment of g0 the slope
// systems need is sum_k w_k H0(u_k) c^alpha = pref0 prod_d m_d[alpha_d] with the
// 1-D moments m_d[p] = sum_i w_{d,i} exp(-lam0 c_{d,i}^2) c_{d,i}^p, p <= 5.
// This kernel reduces the 1-D moments (warp per face); k_face_fin2 forms the
// products (thread per face, FP64).
template <typename T, int D, int NC>
__device__ __forceinline__ void face_sum2_sep_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    constexpr int NS = Sym<D>::N;
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    const T *fr = dc.frec + (size_t)f * FREC;
    const T lam = fr[FR_LAM], nl2 = fr[FR_NL2];
    double *out = dc.fsum2 + (size_t)f * NS * (D + 1);
    for (int d = 0; d < D; ++d) {
        const T U0 = fr[FR_U + d];
        if constexpr (std::is_same<T, float>::value) {
            // blocked sums accumulated in FP64 (SUM_BLOCK nodes per lane per block)
            double acc = 0.0;
            for (int i0 = 0; i0 < dc.cart_n[d]; i0 += 32 * SUM_BLOCK) {
                float blk[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int j = 0; j < SUM_BLOCK; ++j) {
                    const int i = i0 + 32 * j + lane;
                    if (i >= dc.cart_n[d]) break;
                    const float c = dc.axis[d][i] - U0;
                    float v = dc.axw[d][i] * gauss<float>(lam, nl2, c * c);
#pragma unroll
                    for (int pw = 0; pw < 6; ++pw) {
                        blk[pw] += v;
                        v *= c;
                    }
                }
                acc += block_to_fp64<8>(blk);
            }
            if ((lane & 3) == 0 && (lane >> 2) < 6) out[d * 6 + (lane >> 2)] = acc;
        } else {
            T acc[6] = {0, 0, 0, 0, 0, 0};
            for (int i = lane; i < dc.cart_n[d]; i += 32) {
                const T c = dc.axis[d][i] - U0;
                T v = dc.axw[d][i] * gauss<T>(lam, nl2, c * c);
#pragma unroll
                for (int pw = 0; pw < 6; ++pw) {
                    acc[pw] += v;
                    v *= c;
                }
            }
#pragma unroll
            for (int pw = 0; pw < 6; ++pw) {
                const double sm = warp_sum(acc[pw]);
                if (lane == pw) out[d * 6 + pw] = sm;
            }
        }
    }
}

template <typename T, int D, int NC>
__global__ void k_face_sum2_sep(DevCase<T> dc)
{
    dependency_wait();
    face_sum2_sep_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_sum2_sep_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_sum2_sep_body<T, D, NC>(dc, bx);
}

// the distinct moments R of k_face_sum2 from the 1-D moments m[d][0..5] of a
// tensor grid: products over the axes
template <int D>
__device__ __forceinline__ void sep_moments(const double (&m)[D][6], double pref, double *R)
{
    using Mo = Mono<D>;
    auto Q = [&](int a, int b, int c) {
        const double r = pref * m[0][a] * m[1][b];
        return D == 3 ? r * m[D - 1][c] : r;
    };
    // |c|^2n times the monomial of exponents (a, b, c)
    auto Q2 = [&](int a, int b, int c) {
        const double s = Q(a + 2, b, c) + Q(a, b + 2, c);
        return D == 3 ? s + Q(a, b, c + 2) : s;
    };
    auto Q4 = [&](int a, int b, int c) {
        const double s = Q(a + 4, b, c) + Q(a, b + 4, c) + 2.0 * Q(a + 2, b + 2, c);
        return D == 3 ? s + Q(a, b, c + 4) + 2.0 * (Q(a + 2, b, c + 2) + Q(a, b + 2, c + 2)) : s;
    };
    R[0] = Q(0, 0, 0);
    R[Mo::OQ4] = Q4(0, 0, 0);
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const int x = d == 0, y = d == 1, z = d == 2;
        R[Mo::O1 + d] = Q(x, y, z);
        R[Mo::OQ4 + 1 + d] = Q4(x, y, z);
#pragma unroll
        for (int e = d; e < D; ++e) {
            const int xe = x + (e == 0), ye = y + (e == 1), ze = z + (e == 2);
            R[Mo::O2 + pair_index(D, d, e)] = Q(xe, ye, ze);
            R[Mo::OQ2 + pair_index(D, d, e)] = Q2(xe, ye, ze);
#pragma unroll
            for (int g = e; g < D; ++g)
                R[Mo::O3 + triple_index(D, d, e, g)] = Q(xe + (g == 0), ye + (g == 1), ze + (g == 2));
        }
    }
}

// slopes of g0 in the centred basis: M0 = L Mc L^T, sum_k w u_d psi psi^T g0 =
// L (Tc_d + U0_d Mc) L^T with psi = L psi_c.  Then beta_d = L^T a_d solves
// Mc beta_d = L^{-1} dW0/dx_d, and the compatibility condition gives
// beta_A = L^T A = -Mc^{-1} sum_d Tc_d beta_d - sum_d U0_d beta_d.
template <typename T, int D, int NC>
__device__ __forceinline__ void face_fin2_body(const DevCase<T> &dc, const int bx)
{
    const int f = bx * blockDim.x + threadIdx.x;
    constexpr int M = D + 2, NS = Sym<D>::N, S2 = NS * (D + 1);
    if (f >= dc.F || dc.ftype[f] == FT_WALL) return;
    const double *pp = dc.fprim0 + (size_t)f * M;
    const double rho0 = pp[0], lam0 = pp[D + 1], i2l = 0.5 / lam0;
    const double nb = dc.nxi * i2l, xb = dc.nxi * (dc.nxi + 2.0) * i2l * i2l, pref = pref_of(rho0, lam0, D);
    double R[Mono<D>::N], S[S2];
    const double *sum2 = dc.fsum2 + (size_t)f * S2;
    if (dc.sep) {
        double m1[D][6];
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int pw = 0; pw < 6; ++pw) m1[d][pw] = sum2[d * 6 + pw];
        sep_moments<D>(m1, pref, R);
    } else {
#pragma unroll
        for (int i = 0; i < Mono<D>::N; ++i) R[i] = sum2[i];
    }
    mono_moments<D>(R, nb, xb, S);
    double U0[D], uu = 0.0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        U0[d] = pp[1 + d];
        uu += U0[d] * U0[d];
    }
    // right-hand sides L^{-1} dW0_d, then B[d] = beta_d, B[D] = beta_A
    double B[(D + 1) * M], inv[M], xa[M];
    const double *dW = dc.fdW0 + (size_t)f * D * M;
    ldl_factor<M>(S, inv);                  // the first NS entries: Mc
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const double *g = dW + d * M;
        double *x = B + d * M;
        x[0] = g[0];
        double um = 0.0;
#pragma unroll
        for (int e = 0; e < D; ++e) {
            x[1 + e] = g[1 + e] - U0[e] * g[0];
            um += U0[e] * g[1 + e];
        }
        x[D + 1] = g[D + 1] - um + 0.5 * uu * g[0];
        ldl_solve<M>(S, inv, x);
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
        double s = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int j = 0; j < M; ++j) s += S[NS * (1 + d) + (i <= j ? tri<M>(i, j) : tri<M>(j, i))] * B[d * M + j];
        xa[i] = -s;
    }
    ldl_solve<M>(S, inv, xa);
#pragma unroll
    for (int i = 0; i < M; ++i) {
#pragma unroll
        for (int d = 0; d < D; ++d) xa[i] -= U0[d] * B[d * M + i];
        B[D * M + i] = xa[i];
    }

    // Expand the equilibrium part of the interface distribution,
    // q3 (g0 + g0+) + q4 u.grad g0 + q5 dg0/dt, into H0(c) P_m(c), c = u - U0:
    //   h: sh = 1 + (kq.c)(2 lam |c|^2 - D - 2), slope terms of int (beta.psi_c) g0 dxi
    //   b: sh = nb [1 + (kq.c)(2 lam |c|^2 - D)], slope terms of int xi^2 (beta.psi_c) g0 dxi
    // with u_d = c_d + U0_d.
    const double kappa = 4.0 * (1.0 - dc.Pr) * lam0 * lam0 / (5.0 * rho0);
    double kq[D];
    for (int d = 0; d < D; ++d) kq[d] = kappa * dc.fq0[(size_t)f * D + d];
    const double *qs = dc.fqs + (size_t)f * 5;   // time integrals of k_face_fin1
    using X = XRec<D>;
    T *x = dc.xrec + (size_t)f * X::LEN;
    for (int d = 0; d < D; ++d) x[X::U + d] = (T)-U0[d];
    x[X::EX] = (T)(std::is_same<T, float>::value ? -lam0 * LOG2E : -lam0);
    x[X::Q1] = (T)qs[0];
    x[X::Q2] = (T)qs[1];
    x[X::PREF] = (T)pref;
    const double pc = std::is_same<T, double>::value ? pref : 1.0;      // factor of the coefficients
    constexpr int NB = Poly<D>::NB, NP = Poly<D>::N;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const double sm = m == 0 ? 1.0 : nb;            // scale of the b moments
        const double xm = m == 0 ? nb : xb;             // xi^2 (resp. xi^4) factor of beta_E / 2
        const double sh0 = m == 0 ? 1.0 : nb;
        const double shl = m == 0 ? -(double)(D + 2) : -(double)D;
        double a0 = qs[2] * sh0, a[D], Bq[D][D], gam[D];
#pragma unroll
        for (int e = 0; e < D; ++e) {
            a[e] = qs[2] * sh0 * shl * kq[e];
            gam[e] = qs[2] * sh0 * 2.0 * lam0 * kq[e];
#pragma unroll
            for (int g = 0; g < D; ++g) Bq[e][g] = 0.0;
        }
        double diag = 0.0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const double *bd = B + d * M;                // beta^(d) in the psi_c basis
            const double alpha = sm * bd[0] + 0.5 * bd[D + 1] * xm;
            a0 += qs[3] * U0[d] * alpha;
            a[d] += qs[3] * alpha;
#pragma unroll
            for (int e = 0; e < D; ++e) {
                a[e] += qs[3] * U0[d] * sm * bd[1 + e];
                Bq[d][e] += qs[3] * sm * bd[1 + e];
            }
            diag += qs[3] * U0[d] * 0.5 * sm * bd[D + 1];
            gam[d] += qs[3] * 0.5 * sm * bd[D + 1];
        }
        const double alphaA = sm * xa[0] + 0.5 * xa[D + 1] * xm;
        a0 += qs[4] * alphaA;
#pragma unroll
        for (int e = 0; e < D; ++e) a[e] += qs[4] * sm * xa[1 + e];
        diag += qs[4] * 0.5 * sm * xa[D + 1];
        T *pm = x + X::POLY + m * NP;
        pm[0] = (T)(pc * a0);
#pragma unroll
        for (int e = 0; e < D; ++e) pm[1 + e] = (T)(pc * a[e]);
        int t = 1 + D;
#pragma unroll
        for (int e = 0; e < D; ++e)
#pragma unroll
            for (int g = e; g < D; ++g)
                pm[t++] = (T)(pc * (e == g ? Bq[e][e] + diag : Bq[e][g] + Bq[g][e]));
#pragma unroll
        for (int e = 0; e < D; ++e) pm[1 + D + NB + e] = (T)(pc * gam[e]);
    }
}

template <typename T, int D, int NC>
__global__ void k_face_fin2(DevCase<T> dc)
{
    dependency_wait();
    face_fin2_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void k_face_fin2_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    face_fin2_body<T, D, NC>(dc, bx);
}

// ------------------------------------------------------------ walls
// rho_w from zero net mass flux (Eq. maxWalldes): outgoing particles (u_n > 0)
// carry the interior reconstruction transported freely over the step,
// incoming ones the wall Maxwellian.
template <typename T, int D, int NC>
__device__ __forceinline__ void wall_sum_body(const DevCase<T> &dc, const int bx)
{
    constexpr int M = D + 2;
    constexpr int NR = 2 + 2 * M;               // num, den, outgoing moments A, incoming moments B
    __shared__ double red[NR][8];
    const int s = bx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (s >= dc.NW) return;
    const int f = dc.wface[s];
    const int c = dc.fL[f];
    const int tag = dc.ftag[f];
    const double Tw = dc.wallT[tag];
    const double lw = 1.0 / (2.0 * Tw);
    T wr[GREC];
    for (int d = 0; d < 3; ++d) wr[GR_U + d] = (T)dc.wallU[tag * 3 + d];
    wr[GR_LAM] = (T)lw;
    wr[GR_PREF] = (T)pref_of(1.0, lw, D);
    wr[GR_NB] = (T)(dc.nxi / (2.0 * lw));
    wr[GR_NL2] = (T)(-lw * LOG2E);
    wr[GREC - 1] = T(0);
    T n[D], r[D];
    for (int d = 0; d < D; ++d) {
        n[d] = dc.fn[(size_t)f * D + d];
        r[d] = dc.frL[(size_t)f * D + d];
    }
    const T dt = dc.dtT;
    const T hdt = T(0.5) * dc.dtT;
    const size_t rs = (size_t)NC * dc.nvp;
    // num / den: zero net mass flux (Eq. maxWalldes); A / B: moments (Eq.
    // macroscopicFlux) of the outgoing flux and of the incoming flux of the
    // unit-density wall Maxwellian over the step, so that F_w = A + rho_w B
    CSum<T> v[NR];
    // TW consecutive velocities per thread: the wall cell's limited slope
    // (cell_slope) reads each face entry once for all of them
    constexpr int TW = 4;
    using K = Pk<T, TW>;
    using P = typename K::P;
    int e0, ne;
    entry_range(dc, c, e0, ne);
    for (int k0 = TW * threadIdx.x; k0 < dc.nvp; k0 += TW * blockDim.x) {
        T u[3][TW], wk[TW], un[TW];
        ldv_const<T, TW>(dc.u[0] + k0, u[0]);
        ldv_const<T, TW>(dc.u[1] + k0, u[1]);
        if (D == 3) ldv_const<T, TW>(dc.u[2] + k0, u[2]);
        else
#pragma unroll
            for (int j = 0; j < TW; ++j) u[2][j] = T(0);
        ldv_const<T, TW>(dc.w + k0, wk);
        bool out = false;
#pragma unroll
        for (int j = 0; j < TW; ++j) {
            const T uj[3] = {u[0][j], u[1][j], u[2][j]};
            un[j] = normal_velocity<T, D>(uj, n);
            out = out || un[j] > T(0);
        }
        P up[K::NP][D], g[NC][K::NP][D], fi[NC][K::NP], ug[NC][K::NP];
#pragma unroll
        for (int j = 0; j < TW; ++j)
#pragma unroll
            for (int d = 0; d < D; ++d) pel<K::W>(&up[j / K::W][d], j % K::W) = u[d][j];
        if (out) {
            // FP32 in 3D: with a fixed entry count all rows are requested before the
            // first is used, where the loop over any count waits for each in turn
            // (2,114 wall faces x 4,568 velocities 214 -> 179 us, 862 x 4,080 103 ->
            // 93).  The FP64 form is bound by its arithmetic; in 2D eight mixed
            // serving cases were 1.7 % slower per step with it.
            const GlobalCell<T, D, NC, TW> src{dc, dc.f_cur + k0, c, e0};
            constexpr int NA = sizeof(T) == 4 && D == 3 ? 4 : 0, NB = sizeof(T) == 4 && D == 3 ? 6 : 0;
            if (NA > 0 && dc.nf == NA) cell_slope<T, D, NC, TW, NA>(dc, src, c, ne, up, fi, g, ug);
            else if (NB > 0 && dc.nf == NB) cell_slope<T, D, NC, TW, NB>(dc, src, c, ne, up, fi, g, ug);
            else cell_slope<T, D, NC, TW, 0>(dc, src, c, ne, up, fi, g, ug);
        }
#pragma unroll
        for (int j = 0; j < TW; ++j) {
            const T uj[3] = {u[0][j], u[1][j], u[2][j]};
            T Fh = 0, Fb = 0;
            int off = -1;
            if (un[j] > T(0)) {
                T hin = pel<K::W>(fi[0], j);
#pragma unroll
                for (int d = 0; d < D; ++d) hin += pel<K::W>(&g[0][j / K::W][d], j % K::W) * r[d];
                const T uga = pel<K::W>(ug[0], j);
                v[0].add(wk[j] * un[j] * (hin - hdt * uga));
                Fh = dt * un[j] * (hin - hdt * uga);
                if (NC == 2) {
                    T bin = pel<K::W>(fi[NC - 1], j);
#pragma unroll
                    for (int d = 0; d < D; ++d) bin += pel<K::W>(&g[NC - 1][j / K::W][d], j % K::W) * r[d];
                    Fb = dt * un[j] * (bin - hdt * pel<K::W>(ug[NC - 1], j));
                }
                off = 2;
            } else if (un[j] < T(0)) {
                const T H = maxwell_h<T, D>(wr, uj);
                v[1].add(wk[j] * un[j] * H);
                Fh = dt * un[j] * H;
                Fb = wr[GR_NB] * Fh;
                off = 2 + M;
            }
            if (off >= 0) {
                T u2 = 0;
#pragma unroll
                for (int d = 0; d < D; ++d) u2 += uj[d] * uj[d];
                T mom[M];
                mom[0] = wk[j] * Fh;
#pragma unroll
                for (int d = 0; d < D; ++d) mom[1 + d] = wk[j] * uj[d] * Fh;
                mom[D + 1] = T(0.5) * wk[j] * (u2 * Fh + (NC == 2 ? Fb : T(0)));
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    if (off == 2) v[2 + i].add(mom[i]);
                    else v[2 + M + i].add(mom[i]);
                }
            }
        }
    }
    // the warps' sums by recursive halving (16 FP64 additions per warp instead of
    // 5 NR), then one thread per value adds the warps
    double t[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) t[i] = i < NR ? v[i < NR ? i : 0].value() : 0.0;
    const double ts = warp_transpose_sum<double, 16>(t);
    if ((lane & 1) == 0 && (lane >> 1) < NR) red[lane >> 1][warp] = ts;
    __syncthreads();
    if (threadIdx.x < NR) {
        double a = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += red[threadIdx.x][w];
        red[threadIdx.x][0] = a;
    }
    __syncthreads();
    if (threadIdx.x <= M) {
        const double rw = -red[0][0] / red[1][0];
        const int m = threadIdx.x - 1;
        if (m >= 0) {
            dc.wall_F[(size_t)s * M + m] = red[2 + m][0] + rw * red[2 + M + m][0];
        } else {
            dc.rho_w[s] = rw;
            T *w = dc.wrec + (size_t)s * GREC;
            for (int i = 0; i < GREC; ++i) w[i] = wr[i];
            w[GR_PREF] = (T)pref_of(rw, lw, D);
        }
    }
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_wall_sum(DevCase<T> dc)
{
    dependency_wait();
    wall_sum_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_wall_sum_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    wall_sum_body<T, D, NC>(dc, bx);
}

// ------------------------------------------------------------ gather pass
// The velocity loop of Algorithm 1 in two passes over a chunk of velocities,
// with the chunk's face fluxes in between:
//   k_flux    every cell's limited slopes (each once), and from the registers
//             that hold them the time-integrated flux (Eq. microscopicFlux with
//             Eq. fullSolution; walls per Sec. 2.5) of those velocities that
//             leave the cell, through each of its faces.  A velocity crosses a
//             face from one side, so every flux is evaluated and stored once,
//             by the cell it comes from; a boundary face's cell stores both
//             directions.
//   k_stage1  per cell the sum of its faces' fluxes, stage 1 (Eq. microS1) in
//             place, and the moments sum_k w psi_k R_k of the flux residual for
//             the W update (Eq. macroscopicUpdata / macroscopicFlux).
// One pass over patches of cells that kept the slopes in shared memory spent
// most of its instructions on slopes recomputed for the neighbours of a patch
// (2.2 evaluations per cell of 48-cell patches), on fluxes evaluated from both
// sides of a face and on selects between the sides: 897 thread instructions
// per cell-velocity for tetrahedra against 295 of the two kernels here
// (k_flux 227, k_stage1 68 at 1,024-velocity groups).  The price is the flux
// buffer, F/C values per cell and velocity written once and read twice, which
// L2 and HBM have room for.  107k-cell tetrahedral mesh x 4,568 velocities,
// FP32: 17.2 -> 7.95 ms; 24k cells x 28^3: 18.4 -> 8.2 ms; 30k triangles x
// 60x50: 3.18 -> 1.55 ms; FP64, 8k triangles x 60x50: 21.0 -> 14.8 ms.
// A chunk bounds the buffer; velocities of different chunks do not meet, so
// the update is in place.

// One warp per cell and tile of 32 TV velocities, TV consecutive ones per lane;
// the nth / 32 warps of a patch (in CTAs of four) take its P cells in turn.  TV =
// 4 reads an entry
// or a record for twice the velocities of TV = 2 (107k-cell tetrahedral mesh:
// 9.1 against 12.4 ms of both kernels).  The next cell's rows, entries and
// records are copied to shared memory while a cell is worked on (StagedCell):
// with loads at their use the 16 warps of an SM waited for memory in 3.8 of 8.9
// cycles per instruction, now its 19 in 1.5 of 8.2, and both kernels went from 8.14
// to 7.35 ms on that mesh and from 0.266 to 0.215 on 2,145 hexahedra x 4,080.
// Bound: instruction issue (45,796 tetrahedra x 1,024 velocities: 58 % of the issue
// slots, FMA pipe 55 %, DRAM 18 %; 15,081 triangles: 54, 50 and 19 %).
constexpr int FLUX_THREADS = 128;

template <typename T, int D, int NC, int TV, int NF>
__device__ __forceinline__ void flux_body(const DevCase<T> &dc, const int bx, const int chunk)
{
    using E = GEnt<D>;
    using X = XRec<D>;
    using K = Pk<T, TV>;
    using P = typename K::P;
    constexpr int W = K::W, NP = K::NP, V = 32 * TV;
    // patches fastest: the CTAs in flight cover neighbouring patches of one
    // tile, so that the rows of f and of the flux buffer they share stay in L2
    const int split = dc.nth / FLUX_THREADS, ncta = dc.n_patches * split;
    const int tile = bx / ncta, p = (bx - tile * ncta) / split;
    const int lane = threadIdx.x & 31, nwarps = dc.nth >> 5;
    const int mine = threadIdx.x >> 5;                                // in the CTA
    const int warp = mine + (bx - tile * ncta - p * split) * (FLUX_THREADS / 32);   // on the patch
    // the lane's first velocity in the chunk and of all; the last tile may be
    // short: its lanes beyond the end repeat the tile's start and store nothing
    int kb, kn;
    chunk_span(dc, chunk, kb, kn);
    const int kl = tile * V + TV * lane;
    const bool live = kl < kn;
    const int kc = live ? kl : tile * V, k = kb + kc;
    const unsigned all = live ? (1u << TV) - 1 : 0u;
    const int cb = p * dc.P, ce = min(dc.C, cb + dc.P);
    const T *fl = dc.f_cur + k;
    P u[NP][D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        P t[NP];
        ldp_const<T, TV>(dc.u[d] + k, t);
#pragma unroll
        for (int i = 0; i < NP; ++i) u[i][d] = t[i];
    }
    const T dt = dc.dtT, hdt2 = T(0.5) * dc.dtT * dc.dtT;
    auto cell = [&](const int c, const auto &src, const int ne) {
        P fi[NC][NP], g[NC][NP][D], ug[NC][NP];
        cell_slope<T, D, NC, TV, NF>(dc, src, c, ne, u, fi, g, ug);
        auto face = [&](const int e) {
            const int4 gi = src.ids(e);
            const int type = gi.z & 255;
            if (type == FT_NONE) return;
            T rsv[4], nv[4];
            src.values(e, (E::RS / 4) * 4, rsv);
            src.values(e, E::N, nv);
            const T *r = rsv + E::RS % 4;
            P un[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) un[i] = pnormal<T, D, P>(u[i], nv, dc.one);
            // the velocities this cell evaluates: those that leave it (u.n = 0,
            // no flux, falls to the neighbour); all of a boundary face
            const bool own = (gi.z >> 8) != 0;
            unsigned on = 0;
#pragma unroll
            for (int j = 0; j < TV; ++j) on |= (gt0(pel<W>(un, j)) == own ? 1u : 0u) << j;
            on &= all;
            P F[NC][NP];
            // value of the cell at the face centre
            auto at_face = [&](int m, int i) {
                P s = fi[m][i];
#pragma unroll
                for (int d = 0; d < D; ++d) s = pfma(g[m][i][d], pbc<P>(r[d]), s);
                return s;
            };
            if (type == FT_WALL) {
                T wr[GREC];
                load_rec<GREC>(dc.wrec + (size_t)gi.w * GREC, wr);
#pragma unroll
                for (int j = 0; j < TV; ++j) {
                    const int i = j / W;
                    T uj[3] = {T(0), T(0), T(0)};
#pragma unroll
                    for (int d = 0; d < D; ++d) uj[d] = pel<W>(&u[i][d], j % W);
                    const T H = maxwell_h<T, D>(wr, uj), unj = pel<W>(un, j);
#pragma unroll
                    for (int m = 0; m < NC; ++m) {
                        P s = at_face(m, i);
                        const T out = pfma(dt, pel<W>(&s, j % W), -pmul(hdt2, pel<W>(ug[m], j)));
                        pel<W>(F[m], j) = (on >> j & 1) ? unj * out : (m == 0 ? unj * dt : unj * dt * wr[GR_NB]) * H;
                    }
                }
                on = all;
            } else {
                T x[X::LEN];
                src.record(e, gi.y, x);
                P fup[NC][NP], ugf[NC][NP];
#pragma unroll
                for (int m = 0; m < NC; ++m)
#pragma unroll
                    for (int i = 0; i < NP; ++i) {
                        fup[m][i] = at_face(m, i);
                        ugf[m][i] = ug[m][i];
                    }
                if (type == FT_FARFIELD) {                 // the ghost's Maxwellian comes in
                    T gr[GREC];
                    load_rec<GREC>(dc.grec + (size_t)gi.w * GREC, gr);
#pragma unroll
                    for (int j = 0; j < TV; ++j) {
                        if (on >> j & 1) continue;
                        T uj[3] = {T(0), T(0), T(0)};
#pragma unroll
                        for (int d = 0; d < D; ++d) uj[d] = pel<W>(&u[j / W][d], j % W);
                        const T H = maxwell_h<T, D>(gr, uj);
#pragma unroll
                        for (int m = 0; m < NC; ++m) {
                            pel<W>(fup[m], j) = m == 0 ? H : gr[GR_NB] * H;
                            pel<W>(ugf[m], j) = T(0);
                        }
                    }
                    on = all;
                }
                const P q1 = pbc<P>(x[X::Q1]), q2 = pbc<P>(x[X::Q2]);
#pragma unroll
                for (int i = 0; i < NP; ++i) {
                    P cv[D], c2;
#pragma unroll
                    for (int d = 0; d < D; ++d) {
                        cv[d] = padd(u[i][d], pbc<P>(x[X::U + d]));
                        c2 = d == 0 ? pmul(cv[0], cv[0]) : pfma(cv[d], cv[d], c2);
                    }
                    P h = gauss_ex(x[X::EX], c2);
                    if (!std::is_same<T, double>::value) h = pmul(h, pbc<P>(x[X::PREF]));   // in P in FP64
#pragma unroll
                    for (int m = 0; m < NC; ++m) {
                        const P eq = poly_eval<T, D, P>(x + X::POLY + m * Poly<D>::N, cv, c2);
                        F[m][i] = pmul(un[i], pfma(h, eq, pfma(q1, fup[m][i], pmul(q2, ugf[m][i]))));
                    }
                }
            }
            T *Fr = dc.flux + (size_t)gi.y * NC * dc.chunk + kc;
            if (on == (1u << TV) - 1) {
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    T v[TV];
#pragma unroll
                    for (int j = 0; j < TV; ++j) v[j] = pel<W>(F[m], j);
                    stv<T, TV>(Fr + (size_t)m * dc.chunk, v);
                }
            } else if (on) {
#pragma unroll
                for (int m = 0; m < NC; ++m)
#pragma unroll
                    for (int j = 0; j < TV; ++j)
                        if (on >> j & 1) Fr[(size_t)m * dc.chunk + j] = pel<W>(F[m], j);
            }
        };
        if constexpr (NF > 0 && std::is_same<T, double>::value) {
            // FP64: a lane takes its own outgoing faces one after the other, with
            // the face's record read from the stage by its own index: the warp
            // evaluates as many fluxes as its busiest lane has faces to leave
            // through (2 of 3 for triangles, 3 of 6 for hexahedra, 2 to 3 of 4
            // for tetrahedra) instead of one per face with half of the lanes
            // idle, and everything but the FP64 operations is free here.  Flux and
            // stage-1 passes: 8k triangles x 60x50 14.0 -> 10.5 ms, 11k tetrahedra
            // x 14^3 16.9 -> 12.8, 20x20 squares x 24^2 0.243 -> 0.191.
#pragma unroll
            for (int e = 0; e < NF; ++e) {
                const int type = src.ids(e).z & 255;
                if (type == FT_WALL || type == FT_FARFIELD) face(e);
            }
#pragma unroll
            for (int j = 0; j < TV; ++j) {
                T un[NF];
                unsigned m = 0;
#pragma unroll
                for (int e = 0; e < NF; ++e) {
                    const int4 gi = src.ids(e);
                    const int type = gi.z & 255;
                    un[e] = T(0);
                    if (type != FT_INTERIOR && type != FT_PERIODIC) continue;
                    T nv[4];
                    src.values(e, E::N, nv);
                    un[e] = pnormal<T, D, T>(u[j], nv, T(1));
                    m |= (live && gt0(un[e]) == ((gi.z >> 8) != 0) ? 1u : 0u) << e;
                }
                for (; m; m &= m - 1) {
                    const int e = __ffs(m) - 1;
                    T une = un[0], rsv[4], x[X::LEN];
#pragma unroll
                    for (int q = 1; q < NF; ++q) une = q == e ? un[q] : une;
                    src.values(e, (E::RS / 4) * 4, rsv);
                    src.record(e, 0, x);
                    T cv[D], c2;
#pragma unroll
                    for (int d = 0; d < D; ++d) {
                        cv[d] = u[j][d] + x[X::U + d];
                        c2 = d == 0 ? cv[0] * cv[0] : pfma(cv[d], cv[d], c2);
                    }
                    const T h = gauss_ex(x[X::EX], c2);
                    T *Fr = dc.flux + (size_t)src.ids(e).y * NC * dc.chunk + kc + j;
#pragma unroll
                    for (int q = 0; q < NC; ++q) {
                        T s = fi[q][j];
#pragma unroll
                        for (int d = 0; d < D; ++d) s = pfma(g[q][j][d], rsv[E::RS % 4 + d], s);
                        const T eq = poly_eval<T, D, T>(x + X::POLY + q * Poly<D>::N, cv, c2);
                        Fr[(size_t)q * dc.chunk] = une * pfma(h, eq, pfma(x[X::Q1], s, x[X::Q2] * ug[q][j]));
                    }
                }
            }
        } else if constexpr (NF > 0) {
#pragma unroll
            for (int e = 0; e < NF; ++e) face(e);
        } else {
            for (int e = 0; e < ne; ++e) face(e);
        }
    };
    if constexpr (NF > 0) {
        // two stages per warp: while a cell is worked on, the next one's rows,
        // entries and records are on their way, and the entry ids of the one
        // after it (which the requests need) are being loaded
        extern __shared__ __align__(16) unsigned char stages[];
        using S = StagedCell<T, D, NC, TV, NF>;
        const S st[2] = {{stages + (size_t)(2 * mine) * S::BYTES, lane}, {stages + (size_t)(2 * mine + 1) * S::BYTES, lane}};
        auto ids = [&](int c) {
            return lane < NF && c < ce ? __ldg(dc.gi + (size_t)c * NF + lane) : make_int4(0, 0, 0, 0);
        };
        int c = cb + warp;
        if (c >= ce) return;
        st[0].request(dc, fl, c, ids(c));
        int4 id = ids(c + nwarps);
        for (int b = 0; c < ce; c += nwarps, b ^= 1) {
            __syncwarp();                                 // the stage to be filled has been read
            const S &cur = st[b];
            if (c + nwarps < ce) st[b ^ 1].request(dc, fl, c + nwarps, id);
            else cp_async_commit();                       // an empty group, for the wait below
            id = ids(c + 2 * nwarps);
            cp_async_wait<1>();
            __syncwarp();
            cell(c, cur, NF);
        }
    } else {
        for (int c = cb + warp; c < ce; c += nwarps) {
            int e0, ne;
            entry_range(dc, c, e0, ne);
            cell(c, GlobalCell<T, D, NC, TV>{dc, fl, c, e0}, ne);
        }
    }
}

// dynamic shared memory of a CTA of the flux pass
template <typename T, int D, int NC, int TV, int NF> constexpr int flux_smem()
{
    if constexpr (NF == 0) return 0;
    else return FLUX_THREADS / 32 * 2 * StagedCell<T, D, NC, TV, NF>::BYTES;
}

// CTAs of four warps: 20 warps fit an SM at 96 registers (tetrahedra and
// hexahedra, FP32 at TV = 4) and 16 at the 120 of the 2D kernels, against 16 in
// CTAs of eight, and the last wave ends sooner.  Both kernels, 107k-cell
// tetrahedral mesh 7.12 -> 6.63 ms (6.88 at four CTAs per SM), 24k cells x 28^3 7.73 -> 7.38,
// 30k-cell triangulation 1.52 -> 1.49 (1.56 at five CTAs per SM, which spill in
// 2D); CTAs of six warps 7.11, 7.84 and 1.57, of two 6.62, 7.34 and 1.55.
template <typename T, int D, int TV> constexpr int flux_min_ctas() { return sizeof(T) == 4 && TV == 4 ? (D == 3 ? 5 : 4) : 0; }

template <typename T, int D, int NC, int TV, int NF>
__global__ void __launch_bounds__(FLUX_THREADS, flux_min_ctas<T, D, TV>()) k_flux(DevCase<T> dc, int chunk)
{
    dependency_wait();
    flux_body<T, D, NC, TV, NF>(dc, blockIdx.x, chunk);
}

template <typename T, int D, int NC, int TV, int NF>
__global__ void __launch_bounds__(FLUX_THREADS, flux_min_ctas<T, D, TV>())
    k_flux_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n, int chunk)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    flux_body<T, D, NC, TV, NF>(dc, bx, chunk);
}

// Moment sums of stage 1: a lane adds its terms two velocities at a time into
// double-float pairs in the FP32 form (TwoSum, the errors summed in the low
// part), plainly in the FP64 form.
template <typename P> struct MomentSum;
template <> struct MomentSum<double> {
    double s;
    __device__ __forceinline__ void zero() { s = 0.0; }
    __device__ __forceinline__ void add(double x, double) { s = __dadd_rn(s, x); }
    // between the chunks of a group: slot i of the carry buffer
    __device__ __forceinline__ void load(const double *carry, size_t i) { s = carry[i]; }
    __device__ __forceinline__ void store(double *carry, size_t i) const { carry[i] = s; }
};
template <> struct MomentSum<float2> {
    float2 h, l;
    __device__ __forceinline__ void zero() { h = l = make_float2(0.f, 0.f); }
    // every addition rounds by itself (see psum)
    __device__ __forceinline__ void add(float2 x, float one)
    {
        const float2 m1 = make_float2(-one, -one);
        const float2 s = psum(x, h, one), v = pfma(h, m1, s);     // s - h
        l = padd(l, padd(pfma(pfma(v, m1, s), m1, h), pfma(v, m1, x)));   // (h - (s - v)) + (x - v)
        h = s;
    }
    __device__ __forceinline__ void load(const float *carry, size_t i)
    {
        const float4 v = reinterpret_cast<const float4 *>(carry)[i];
        h = make_float2(v.x, v.y);
        l = make_float2(v.z, v.w);
    }
    __device__ __forceinline__ void store(float *carry, size_t i) const
    {
        reinterpret_cast<float4 *>(carry)[i] = make_float4(h.x, h.y, l.x, l.y);
    }
};

// One warp per cell and group of gvel velocities of the chunk, four consecutive
// velocities per lane.  Bound: the latency of its row loads (nf rows of the flux
// buffer and f, which is written in place); the reduction at a group's end costs
// as much as 250 velocities (see set_chunks in ugks_host.cu).
//
// The rows come through a ring of NS slots in shared memory, filled NS - 1
// iterations ahead by asynchronous copies (a lane reads back what it copied, so
// no barrier): without it a warp had the loads of one iteration in flight and
// waited for them in 11 of 15 cycles per instruction (7.35 -> 7.12 ms of both
// kernels on the 107k-cell mesh, 1.56 -> 1.52 on the 30k-cell triangulation); now it
// waits in 2.9 of 8.0 cycles for tetrahedra (DRAM 55 %) and 4.8 of 9.5 for triangles
// (65 %).
template <typename T, int NC, int NF> constexpr int stage1_stages()
{
    return (NF + 1) * NC * 4 * (int)sizeof(T) * 32 * 8 * 3 <= 64 * 1024 ? 3 : 2;
}
template <typename T, int NC, int NF> constexpr int stage1_smem()
{
    return NF == 0 ? 0 : stage1_stages<T, NC, NF>() * (NF + 1) * NC * 4 * (int)sizeof(T) * 32 * 8;
}

template <typename T, int D, int NC, int NF>
__device__ __forceinline__ void stage1_body(const DevCase<T> &dc, const int bx, const int chunk)
{
    using E = GEnt<D>;
    using K = Pk<T, 4>;
    using P = typename K::P;
    constexpr int M = D + 2, W = K::W, NP = K::NP;
    const int lane = threadIdx.x & 31;
    const int ncb = (dc.C + 7) >> 3, grp = bx / ncb;
    const int c = (bx - grp * ncb) * 8 + (threadIdx.x >> 5);
    if (c >= dc.C) return;
    int kb, kn;                                                        // chunk start, velocities
    chunk_span(dc, chunk, kb, kn);
    const int kg = grp * dc.gvel;                                      // group start in the chunk
    kn = min(kn, kg + dc.gvel);                                        // end in the chunk
    if (kg >= kn) return;                                              // the last chunk may be short
    int e0 = c * NF, ne = NF;
    if (NF == 0) entry_range(dc, c, e0, ne);
    T cs[NF > 0 ? NF : 1];
    const T *Fr[NF > 0 ? NF : 1];
    T *frow = dc.f_cur + (size_t)c * NC * dc.nvp + kb;
    constexpr int B = 4 * (int)sizeof(T), NS = stage1_stages<T, NC, NF>(), ROWS = (NF + 1) * NC;
    extern __shared__ __align__(16) unsigned char stages[];
    unsigned char *const mine = stages + ((size_t)(threadIdx.x >> 5) * NS * ROWS * 32 + lane) * B;
    // rows of the velocities at kc into ring slot q: the faces' fluxes, then f
    auto request = [&](const int kc, const int q) {
        if (kc < kn) {
            unsigned char *dst = mine + (size_t)q * ROWS * 32 * B;
#pragma unroll
            for (int e = 0; e < NF; ++e)
#pragma unroll
                for (int m = 0; m < NC; ++m)
                    cp_async_lane<B>(dst + (e * NC + m) * 32 * B, Fr[e] + (size_t)m * dc.chunk + kc);
#pragma unroll
            for (int m = 0; m < NC; ++m) cp_async_lane<B>(dst + (NF * NC + m) * 32 * B, frow + (size_t)m * dc.nvp + kc);
        }
        cp_async_commit();
    };
    if constexpr (NF > 0) {
        // a padding entry reads the first face's row with coefficient 0
        const int f0 = __ldg(dc.gi + e0).y;
#pragma unroll
        for (int e = 0; e < NF; ++e) {
            const int4 gi = __ldg(dc.gi + e0 + e);
            cs[e] = __ldg(dc.gf + (size_t)(e0 + e) * E::LEN + E::CS);
            Fr[e] = dc.flux + (size_t)(gi.z == FT_NONE ? f0 : gi.y) * NC * dc.chunk;
        }
#pragma unroll
        for (int q = 0; q < NS - 1; ++q) request(kg + 4 * lane + 128 * q, q);
    }
    T cr[CREC];
    load_rec<CREC>(dc.crec + (size_t)c * CREC, cr);
    const P ccol = pbc<P>(cr[CR_C]), kl2 = pbc<P>(T(2) * cr[CR_LAM]);
    MomentSum<P> acc[M];
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i].zero();
    // a group in several chunks: the lane's sums go on where the chunk before left them
    if (dc.parts > 1 && chunk % dc.parts > 0)
#pragma unroll
        for (int i = 0; i < M; ++i) acc[i].load(dc.carry, ((size_t)c * M + i) * 32 + lane);
    int slot = 0;
    for (int kc = kg + 4 * lane; kc < kn; kc += 128) {
        P fs[NC][NP], R[NC][NP];
#pragma unroll
        for (int m = 0; m < NC; ++m)
#pragma unroll
            for (int i = 0; i < NP; ++i) R[m][i] = pbc<P>(T(0));
        if constexpr (NF > 0) {
            request(kc + 128 * (NS - 1), slot == 0 ? NS - 1 : slot - 1);   // the slot read last
            cp_async_wait<NS - 1>();
            const unsigned char *src = mine + (size_t)slot * ROWS * 32 * B;
            slot = slot == NS - 1 ? 0 : slot + 1;
#pragma unroll
            for (int e = 0; e < NF; ++e)
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    P Fv[NP];
                    lds_pack<T, 4>(src + (e * NC + m) * 32 * B, Fv);
#pragma unroll
                    for (int i = 0; i < NP; ++i) R[m][i] = pfma(pbc<P>(cs[e]), Fv[i], R[m][i]);
                }
#pragma unroll
            for (int m = 0; m < NC; ++m) lds_pack<T, 4>(src + (NF * NC + m) * 32 * B, fs[m]);
        } else {
            for (int e = 0; e < ne; ++e) {
                const int4 gi = __ldg(dc.gi + e0 + e);
                const P ce = pbc<P>(__ldg(dc.gf + (size_t)(e0 + e) * E::LEN + E::CS));
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    P Fv[NP];
                    ldp<T, 4>(dc.flux + ((size_t)gi.y * NC + m) * dc.chunk + kc, Fv);
#pragma unroll
                    for (int i = 0; i < NP; ++i) R[m][i] = pfma(ce, Fv[i], R[m][i]);
                }
            }
#pragma unroll
            for (int m = 0; m < NC; ++m)                               // f is written below: ordinary loads
#pragma unroll
                for (int j = 0; j < 4; ++j) pel<W>(fs[m], j) = frow[(size_t)m * dc.nvp + kc + j];
        }
        P u[D][NP], wk[NP];
#pragma unroll
        for (int d = 0; d < D; ++d) ldp_const<T, 4>(dc.u[d] + kb + kc, u[d]);
        ldp_const<T, 4>(dc.w + kb + kc, wk);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            // f+ of the cell (shakhov_fplus), stage 1
            P cv[D], c2, kqc, u2, h;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                cv[d] = padd(u[d][i], pbc<P>(-cr[CR_U + d]));
                c2 = d == 0 ? pmul(cv[0], cv[0]) : pfma(cv[d], cv[d], c2);
                kqc = d == 0 ? pmul(cv[0], pbc<P>(cr[CR_KQ])) : pfma(cv[d], pbc<P>(cr[CR_KQ + d]), kqc);
                u2 = d == 0 ? pmul(u[0][i], u[0][i]) : pfma(u[d][i], u[d][i], u2);
            }
#pragma unroll
            for (int w = 0; w < W; ++w)
                pel<W>(&h, w) = cr[CR_PREF] * gauss<T>(cr[CR_LAM], cr[CR_NL2], pel<W>(&c2, w));
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const P X = pfma(kqc, pfma(kl2, c2, pbc<P>(T(m == 0 ? -(D + 2) : -D))), pbc<P>(T(1)));
                const P df = pfma(m == 0 ? h : pmul(h, pbc<P>(cr[CR_NB])), X, pmul(fs[m][i], pbc<P>(T(-1))));
                fs[m][i] = pfma(ccol, df, padd(fs[m][i], R[m][i]));
            }
            const P wr = pmul(wk[i], R[0][i]);
            acc[0].add(wr, dc.one);
#pragma unroll
            for (int d = 0; d < D; ++d) acc[1 + d].add(pmul(u[d][i], wr), dc.one);
            const P en = NC == 2 ? pfma(u2, wr, pmul(wk[i], R[NC - 1][i])) : pmul(u2, wr);
            acc[D + 1].add(pmul(pbc<P>(T(0.5)), en), dc.one);
        }
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            T v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = pel<W>(fs[m], j);
            stv<T, 4>(frow + (size_t)m * dc.nvp + kc, v);
        }
    }
    const int group = (kb + kg) / dc.gvel;
    if (dc.parts > 1 && kb + kn < min(dc.nvp, (group + 1) * dc.gvel)) {
#pragma unroll
        for (int i = 0; i < M; ++i) acc[i].store(dc.carry, ((size_t)c * M + i) * 32 + lane);
        return;
    }
    // across the warp
    constexpr int NR = M <= 4 ? 4 : 8;
    const int vi = lane >> (NR == 4 ? 3 : 2);
    double sum;
    if constexpr (std::is_same<T, float>::value) {
        float mh[NR], ml[NR], oh, ol;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            mh[i] = ml[i] = 0.f;
            if (i < M) {
                mh[i] = acc[i].h.x;
                ml[i] = acc[i].l.x;
                ff_add(mh[i], ml[i], acc[i].h.y, acc[i].l.y);
            }
        }
        warp_transpose_sum_ff2<NR>(mh, ml, oh, ol);
        sum = (double)oh + (double)ol;
    } else {
        T v[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) v[i] = i < M ? acc[i].s : T(0);
        sum = warp_transpose_sum<T, NR>(v);
    }
    if ((lane & (NR == 4 ? 7 : 3)) == 0 && vi < M)
        dc.dW_part[((size_t)c * dc.n_groups + group) * M + vi] = sum;
}

template <typename T, int D, int NC, int NF>
__global__ void __launch_bounds__(256) k_stage1(DevCase<T> dc, int chunk)
{
    dependency_wait();
    stage1_body<T, D, NC, NF>(dc, blockIdx.x, chunk);
}

template <typename T, int D, int NC, int NF>
__global__ void __launch_bounds__(256) k_stage1_batch(const DevCase<T> *__restrict__ cases,
                                                      const int *__restrict__ off, int n, int chunk)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    stage1_body<T, D, NC, NF>(dc, bx, chunk);
}

// ------------------------------------------------------------ W update
template <typename T, int D, int NC>
__device__ __forceinline__ void update_W_body(const DevCase<T> &dc, const int bx)
{
    constexpr int M = D + 2;
    const int c = bx * blockDim.x + threadIdx.x;
    double dsq[M], wsq[M];
    for (int m = 0; m < M; ++m) dsq[m] = wsq[m] = 0.0;
    if (c < dc.C) {
        double *Wc = dc.W + (size_t)c * M;
        const bool counts = !dc.owned || dc.owned[c];      // halo cells of a subdomain do not count
        for (int m = 0; m < M; ++m) {
            double s = 0.0;
            for (int t = 0; t < dc.n_groups; ++t) s += dc.dW_part[((size_t)c * dc.n_groups + t) * M + m];
            if (counts) {
                wsq[m] = Wc[m] * Wc[m];
                dsq[m] = s * s;
            }
            Wc[m] += s;
        }
        Prim p = prim_of(Wc, D);
        if (!(p.rho > 0.0) || !(p.T > 0.0) || !isfinite(p.rho) || !isfinite(p.T)) atomicOr(dc.flags, 1);
        cell_record<T, D>(dc, p, dc.q + (size_t)c * D, dc.krec + (size_t)c * CREC);
    }
    // residual partials of the warp's 32 cells, whatever the block size
    const int w = c >> 5;
    for (int m = 0; m < M; ++m) {
        const double a = warp_sum(dsq[m]), b = warp_sum(wsq[m]);
        if ((threadIdx.x & 31) == 0 && c < dc.C) {
            dc.res_part[(size_t)w * 2 * M + m] = a;
            dc.res_part[(size_t)w * 2 * M + M + m] = b;
        }
    }
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_update_W(DevCase<T> dc)
{
    dependency_wait();
    update_W_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_update_W_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off, int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    update_W_body<T, D, NC>(dc, bx);
}

// one block of RES_THREADS threads: thread sums of the partials, all values of a
// partial requested together, then the lanes in order
constexpr int RES_THREADS = 512;
template <int M>
__global__ void __launch_bounds__(RES_THREADS) k_residual(const double *res_part, int nparts, double *res)
{
    __shared__ double acc[2 * M][RES_THREADS / 32];
    const int t = threadIdx.x;
    double s[2 * M];
#pragma unroll
    for (int i = 0; i < 2 * M; ++i) s[i] = 0.0;
#pragma unroll 4
    for (int b = t; b < nparts; b += RES_THREADS)
#pragma unroll
        for (int i = 0; i < 2 * M; ++i) s[i] += res_part[(size_t)b * 2 * M + i];
#pragma unroll
    for (int i = 0; i < 2 * M; ++i) {
        const double v = warp_sum(s[i]);
        if ((t & 31) == 0) acc[i][t >> 5] = v;
    }
    __syncthreads();
    if (t < M) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < RES_THREADS / 32; ++w) {
            a += acc[t][w];
            b += acc[M + t][w];
        }
        res[t] = b > 0.0 ? sqrt(a) / sqrt(b) : sqrt(a);
    }
}

// sums of RES_FOLD consecutive partials (of 32 cells each), a thread per value
__global__ void __launch_bounds__(256) k_residual_fold(const double *res_part, int nparts, int nvals, double *out)
{
    const int t = blockIdx.x * 256 + threadIdx.x, j = t / nvals, i = t - j * nvals;
    if (j * RES_FOLD >= nparts) return;
    double s = 0.0;
    for (int b = j * RES_FOLD; b < min(nparts, (j + 1) * RES_FOLD); ++b) s += res_part[(size_t)b * nvals + i];
    out[t] = s;
}

// ------------------------------------------------------------ stage 2
template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<double> { using type = double4_32a; };

// 4 consecutive velocities per lane (rows are padded to a multiple of 32, so
// every row start is 16-byte aligned for FP32 and 32-byte aligned for FP64)
template <typename T, int D, int NC>
__device__ __forceinline__ void collide_body(const DevCase<T> &dc, const int bx)
{
    using V4 = typename Vec4<T>::type;
    const int c = bx * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= dc.C) return;
    // the cell's record in registers: read once, not again after every store of f
    T kr[CREC];
#pragma unroll
    for (int i = 0; i < CREC; ++i) kr[i] = dc.krec[(size_t)c * CREC + i];
    const T cc = kr[CR_C];
    const T inv = kr[CR_INV];
    T U[D];
#pragma unroll
    for (int d = 0; d < D; ++d) U[d] = kr[CR_U + d];
    const size_t rs = (size_t)NC * dc.nvp;
    // heat-flux terms: FP64 sums in the FP64 form; blocked sums accumulated in
    // FP64 in the FP32 form (16 terms per lane per block)
    constexpr bool F32 = std::is_same<T, float>::value;
    constexpr int NP = D == 2 ? 2 : 4;
    T blk[NP];
#pragma unroll
    for (int d = 0; d < NP; ++d) blk[d] = 0;
    double acc = 0.0;
    int nblk = 0;
    // f~ comes through a ring of COLLIDE_SLOTS slots of shared memory per lane,
    // filled by asynchronous copies COLLIDE_SLOTS - 1 iterations ahead
    T *frow = dc.f_cur + (size_t)c * rs;
    constexpr int B = 4 * (int)sizeof(T), COLLIDE_SLOTS = sizeof(T) == 4 ? 3 : 2;
    __shared__ __align__(32) unsigned char ring[8 * COLLIDE_SLOTS * NC * 32 * B];
    unsigned char *const mine = ring + ((threadIdx.x >> 5) * COLLIDE_SLOTS * NC * 32 + lane) * B;
    auto request = [&](int k0, int q) {
        if (k0 < dc.nvp)
#pragma unroll
            for (int m = 0; m < NC; ++m) cp_async_lane<B>(mine + (q * NC + m) * 32 * B, frow + (size_t)m * dc.nvp + k0);
        cp_async_commit();
    };
#pragma unroll
    for (int q = 0; q < COLLIDE_SLOTS - 1; ++q) request(128 * q + 4 * lane, q);
    int slot = 0;
    for (int k00 = 0; k00 < dc.nvp; k00 += 128) {          // uniform over the warp
        const int k0 = k00 + 4 * lane;
        request(k0 + 128 * (COLLIDE_SLOTS - 1), slot == 0 ? COLLIDE_SLOTS - 1 : slot - 1);
        cp_async_wait<COLLIDE_SLOTS - 1>();
        if (k0 < dc.nvp) {
            T ft[NC][4], fn[NC][4];
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const V4 v = *reinterpret_cast<const V4 *>(mine + (slot * NC + m) * 32 * B);
                ft[m][0] = v.x;
                ft[m][1] = v.y;
                ft[m][2] = v.z;
                ft[m][3] = v.w;
            }
            // the lane's four velocities from the per-component arrays: each load
            // of the warp covers one contiguous span (the packed [k][4] records
            // of four consecutive velocities per lane would touch four times the
            // cache lines per load)
            T uv[3][4], wv[4];
            ldv_const<T, 4>(dc.u[0] + k0, uv[0]);
            ldv_const<T, 4>(dc.u[1] + k0, uv[1]);
            if (D == 3) ldv_const<T, 4>(dc.u[2] + k0, uv[2]);
            else
#pragma unroll
                for (int j = 0; j < 4; ++j) uv[2][j] = T(0);
            ldv_const<T, 4>(dc.w + k0, wv);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const T u[3] = {uv[0][j], uv[1][j], uv[2][j]};
                const T wk = wv[j];
                T fp[NC];
                shakhov_fplus<T, D, NC>(kr, u, fp);
#pragma unroll
                for (int m = 0; m < NC; ++m) fn[m][j] = (ft[m][j] + cc * fp[m]) * inv;
                T cv[D], c2 = 0;
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    cv[d] = u[d] - U[d];
                    c2 += cv[d] * cv[d];
                }
                const T we = wk * (c2 * fn[0][j] + (NC == 2 ? fn[NC - 1][j] : T(0)));
#pragma unroll
                for (int d = 0; d < D; ++d) blk[d] += cv[d] * we;
            }
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                V4 v;
                v.x = fn[m][0];
                v.y = fn[m][1];
                v.z = fn[m][2];
                v.w = fn[m][3];
                *reinterpret_cast<V4 *>(frow + (size_t)m * dc.nvp + k0) = v;
            }
        }
        slot = slot == COLLIDE_SLOTS - 1 ? 0 : slot + 1;
        if constexpr (F32) {
            if (++nblk == SUM_BLOCK / 4 || k00 + 128 >= dc.nvp) {
                acc += block_to_fp64<NP>(blk);
#pragma unroll
                for (int d = 0; d < NP; ++d) blk[d] = 0;
                nblk = 0;
            }
        }
    }
    if constexpr (F32) {
        // lanes 16j.. (D = 2) or 8j.. (D = 3) hold component j
        const int vi = lane >> (NP == 2 ? 4 : 3);
        if ((lane & (NP == 2 ? 15 : 7)) == 0 && vi < D) dc.q[(size_t)c * D + vi] = 0.5 * acc;
    } else {
        for (int d = 0; d < D; ++d) {
            const double sm = warp_sum(blk[d]);
            if (lane == 0) dc.q[(size_t)c * D + d] = 0.5 * sm;
        }
    }
}

// four 256-thread blocks per SM in the 2D FP32 form (five would spill).  Ring of
// 3 slots on the 30k x 60x50 and the 107k x 4,568 cases: 0.304 -> 0.236 ms (6.2
// TB/s) and 0.766 -> 0.731 ms (5.4 TB/s; the latency of the arithmetic chain is
// what is left in 3D); 4 and 6 slots 0.236 and 0.245, 0.738 and 0.728.
template <typename T, int D, int NC>
__global__ void __launch_bounds__(256, sizeof(T) == 4 && D == 2 ? 4 : 0) k_collide(DevCase<T> dc)
{
    dependency_wait();
    collide_body<T, D, NC>(dc, blockIdx.x);
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_collide_batch(const DevCase<T> *__restrict__ cases, const int *__restrict__ off,
                                                       int n)
{
    int bx;
    const DevCase<T> &dc = batch_case(cases, off, n, bx);
    dependency_wait();
    collide_body<T, D, NC>(dc, bx);
}

// ------------------------------------------------------------ state I/O
// Host-layout element type S: double, or float for callers that hold the
// distribution in single precision (exact for FP32 storage).
template <typename T, int D, int NC, typename S>
__global__ void k_f_export(DevCase<T> dc, const long long *perm, int c0, int nc, S *out)
{
    // out[(i - c0)][m][k] (caller cell order i) from internal cell perm[i]
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long per = (long long)NC * dc.nv;
    if (idx >= (long long)nc * per) return;
    const int i = c0 + (int)(idx / per);
    const long long r = idx % per;
    const int m = (int)(r / dc.nv), k = (int)(r % dc.nv);
    const long long ci = perm[i];
    out[idx] = (S)dc.f_cur[(size_t)ci * NC * dc.nvp + (size_t)m * dc.nvp + k];
}

template <typename T, int D, int NC, typename S>
__global__ void k_f_import(DevCase<T> dc, const long long *perm, int c0, int nc, const S *in)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long per = (long long)NC * dc.nvp;
    if (idx >= (long long)nc * per) return;
    const int i = c0 + (int)(idx / per);
    const long long r = idx % per;
    const int m = (int)(r / dc.nvp), k = (int)(r % dc.nvp);
    const long long ci = perm[i];
    dc.f_cur[(size_t)ci * NC * dc.nvp + (size_t)m * dc.nvp + k] =
        k < dc.nv ? (T)in[((long long)(i - c0) * NC + m) * dc.nv + k] : T(0);
}

template <int D>
__global__ void k_moments_out(const double *W, const double *q, const long long *perm, int C, double *out)
{
    // out[i][0..]: rho, U[D], T, q[D] in caller order
    constexpr int M = D + 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C) return;
    const long long c = perm[i];
    Prim p = prim_of(W + (size_t)c * M, D);
    double *o = out + (size_t)i * (2 * D + 2);
    o[0] = p.rho;
    for (int d = 0; d < D; ++d) o[1 + d] = p.U[d];
    o[D + 1] = p.T;
    for (int d = 0; d < D; ++d) o[D + 2 + d] = q[(size_t)c * D + d];
}

template <int D>
__global__ void k_W_permute(const double *src, const long long *perm, int C, double *dst, int to_internal)
{
    constexpr int M = D + 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C) return;
    const long long c = perm[i];
    for (int m = 0; m < M; ++m) {
        if (to_internal) dst[(size_t)c * M + m] = src[(size_t)i * M + m];
        else dst[(size_t)i * M + m] = src[(size_t)c * M + m];
    }
}

__global__ void k_check(const double *W, int n, int M, int *flags)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const double *w = W + (size_t)c * M;
    double ke = 0.0;
    for (int d = 1; d < M - 1; ++d) ke += w[d] * w[d];
    const double e = w[M - 1] - 0.5 * ke / w[0];
    bool bad = !(w[0] > 0.0) || !(e > 0.0);
    for (int m = 0; m < M; ++m) bad |= !isfinite(w[m]);
    if (bad) atomicOr(flags, 1);
}

// Smallest and largest density over the own cells (owned == NULL: all cells).
// Densities are positive doubles, whose bit patterns order as the values do;
// a non-positive or non-finite density enters as +0.  range[0] starts at all
// ones (atomicMin), range[1] at zero (atomicMax).
__global__ void k_density_range(const double *W, int n, int M, const unsigned char *owned,
                                unsigned long long *range)
{
    unsigned long long lo = ~0ull, hi = 0ull;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        if (owned && !owned[c]) continue;
        const double r = W[(size_t)c * M];
        const unsigned long long b = (r > 0.0 && isfinite(r)) ? (unsigned long long)__double_as_longlong(r) : 0ull;
        lo = b < lo ? b : lo;
        hi = b > hi ? b : hi;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        lo = l2 < lo ? l2 : lo;
        hi = h2 > hi ? h2 : hi;
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&range[0], lo);
        atomicMax(&range[1], hi);
    }
}

// ------------------------------------------------------------ halo exchange
// Rows of the halo buffer: f of the cell in the storage type [NC][nv], padded
// to 8 bytes, then W [D+2] and q [D] in FP64.  One block per listed cell.
// Bound by the bytes of the rows: component by component, without a division
// per value, eight loads of a thread in flight before its first store: 107k rows of
// 18 KB 1.06 -> 0.65 ms (6.1 TB/s), 30k rows of 24 KB 0.405 -> 0.222 ms (6.5 TB/s).
template <typename T>
__device__ __forceinline__ void copy_row(const T *__restrict__ src, T *__restrict__ dst, int n)
{
    for (int j0 = threadIdx.x; j0 < n; j0 += 8 * blockDim.x) {
        T v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if ((int)(j0 + q * blockDim.x) < n) v[q] = src[j0 + q * blockDim.x];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if ((int)(j0 + q * blockDim.x) < n) dst[j0 + q * blockDim.x] = v[q];
    }
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_halo_pack(DevCase<T> dc, const int *cells, int n, size_t row,
                                                   unsigned char *buf)
{
    constexpr int M = D + 2;
    const int i = blockIdx.x;
    if (i >= n) return;
    const int c = cells[i];
    unsigned char *r = buf + (size_t)i * row;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        T *__restrict__ fo = reinterpret_cast<T *>(r) + (size_t)m * dc.nv;
        const T *fc = dc.f_cur + ((size_t)c * NC + m) * dc.nvp;
        copy_row(fc, fo, dc.nv);
    }
    double *tail = reinterpret_cast<double *>(r + row - (size_t)(M + D) * sizeof(double));
    if (threadIdx.x < M) tail[threadIdx.x] = dc.W[(size_t)c * M + threadIdx.x];
    else if (threadIdx.x < M + D) tail[threadIdx.x] = dc.q[(size_t)c * D + threadIdx.x - M];
}

template <typename T, int D, int NC>
__global__ void __launch_bounds__(256) k_halo_unpack(DevCase<T> dc, const int *cells, int n, size_t row,
                                                     const unsigned char *buf)
{
    constexpr int M = D + 2;
    const int i = blockIdx.x;
    if (i >= n) return;
    const int c = cells[i];
    const unsigned char *r = buf + (size_t)i * row;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        const T *__restrict__ fi = reinterpret_cast<const T *>(r) + (size_t)m * dc.nv;
        T *fc = dc.f_cur + ((size_t)c * NC + m) * dc.nvp;
        copy_row(fi, fc, dc.nv);
    }
    const double *tail = reinterpret_cast<const double *>(r + row - (size_t)(M + D) * sizeof(double));
    if (threadIdx.x < M) dc.W[(size_t)c * M + threadIdx.x] = tail[threadIdx.x];
    else if (threadIdx.x < M + D) dc.q[(size_t)c * D + threadIdx.x - M] = tail[threadIdx.x];
}

// ------------------------------------------------------------ launchers
static inline int cdiv(long long a, int b) { return (int)((a + b - 1) / b); }

// The two kernels of a chunk, for one case (cases == nullptr) or for those of a
// batch (block offsets off[0..n]).  All cases of a launch share the velocities
// per lane tv and the entry count nf.
template <typename T, int D, int NC, int TV, int NF>
static cudaError_t flux_launch(int blocks, int chunk, cudaStream_t st, const DevCase<T> *dc, const DevCase<T> *cases,
                               const int *off, int n)
{
    constexpr int smem = flux_smem<T, D, NC, TV, NF>();
    if (smem > 48 * 1024) {
        const cudaError_t e =
            cases ? cudaFuncSetAttribute(k_flux_batch<T, D, NC, TV, NF>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                  : cudaFuncSetAttribute(k_flux<T, D, NC, TV, NF>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    return cases ? launch(k_flux_batch<T, D, NC, TV, NF>, blocks, FLUX_THREADS, smem, st, cases, off, n, chunk)
                 : launch(k_flux<T, D, NC, TV, NF>, blocks, FLUX_THREADS, smem, st, *dc, chunk);
}

template <typename T, int D, int NC, int NF>
static cudaError_t flux_tiled(int tv, int blocks, int chunk, cudaStream_t st, const DevCase<T> *dc,
                              const DevCase<T> *cases, const int *off, int n)
{
    if (tv == 1) return flux_launch<T, D, NC, 1, NF>(blocks, chunk, st, dc, cases, off, n);
    if (tv == 2) return flux_launch<T, D, NC, 2, NF>(blocks, chunk, st, dc, cases, off, n);
    if (tv == 4) return flux_launch<T, D, NC, 4, NF>(blocks, chunk, st, dc, cases, off, n);
    return cudaErrorInvalidValue;
}

// entry counts with kernels of their own: triangles, quadrilaterals and
// tetrahedra, hexahedra; a mesh with another largest count takes the next one
// above, one beyond MAX_NF the kernels that loop over the cells' own counts
template <typename T>
cudaError_t launch_flux(int D, int nf, int vtile, int blocks, int chunk, cudaStream_t st, const DevCase<T> *dc,
                        const DevCase<T> *cases, const int *off, int n)
{
    const int tv = vtile / 32;
    if (blocks <= 0) return cudaSuccess;
    if (D == 2) {
        if (nf == 3) return flux_tiled<T, 2, 2, 3>(tv, blocks, chunk, st, dc, cases, off, n);
        if (nf == 4) return flux_tiled<T, 2, 2, 4>(tv, blocks, chunk, st, dc, cases, off, n);
        return flux_tiled<T, 2, 2, 0>(tv, blocks, chunk, st, dc, cases, off, n);
    }
    if (nf == 4) return flux_tiled<T, 3, 1, 4>(tv, blocks, chunk, st, dc, cases, off, n);
    if (nf == 6) return flux_tiled<T, 3, 1, 6>(tv, blocks, chunk, st, dc, cases, off, n);
    return flux_tiled<T, 3, 1, 0>(tv, blocks, chunk, st, dc, cases, off, n);
}

template <typename T, int D, int NC, int NF>
static cudaError_t stage1_launch(int blocks, int chunk, cudaStream_t st, const DevCase<T> *dc, const DevCase<T> *cases,
                                 const int *off, int n)
{
    constexpr int smem = stage1_smem<T, NC, NF>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cases ? cudaFuncSetAttribute(k_stage1_batch<T, D, NC, NF>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                                    : cudaFuncSetAttribute(k_stage1<T, D, NC, NF>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    return cases ? launch(k_stage1_batch<T, D, NC, NF>, blocks, 256, smem, st, cases, off, n, chunk)
                 : launch(k_stage1<T, D, NC, NF>, blocks, 256, smem, st, *dc, chunk);
}

template <typename T>
cudaError_t launch_stage1(int D, int nf, int blocks, int chunk, cudaStream_t st, const DevCase<T> *dc,
                          const DevCase<T> *cases, const int *off, int n)
{
    if (blocks <= 0) return cudaSuccess;
    if (D == 2) {
        if (nf == 3) return stage1_launch<T, 2, 2, 3>(blocks, chunk, st, dc, cases, off, n);
        if (nf == 4) return stage1_launch<T, 2, 2, 4>(blocks, chunk, st, dc, cases, off, n);
        return stage1_launch<T, 2, 2, 0>(blocks, chunk, st, dc, cases, off, n);
    }
    if (nf == 4) return stage1_launch<T, 3, 1, 4>(blocks, chunk, st, dc, cases, off, n);
    if (nf == 6) return stage1_launch<T, 3, 1, 6>(blocks, chunk, st, dc, cases, off, n);
    return stage1_launch<T, 3, 1, 0>(blocks, chunk, st, dc, cases, off, n);
}

template <typename T> int flux_blocks(const DevCase<T> &dc, int chunk)
{
    int kb, len;
    chunk_span(dc, chunk, kb, len);
    return len > 0 ? dc.n_patches * (dc.nth / FLUX_THREADS) * cdiv(len, dc.vtile) : 0;
}

template <typename T> int stage1_blocks(const DevCase<T> &dc, int chunk)
{
    int kb, len;
    chunk_span(dc, chunk, kb, len);
    return len > 0 ? cdiv(dc.C, 8) * cdiv(len, dc.gvel) : 0;
}

// the flux and stage-1 passes of one case over its chunks
template <typename T>
cudaError_t launch_gather(const DevCase<T> &dc, cudaStream_t st)
{
    for (int r = 0; r < dc.n_chunks; ++r) {
        cudaError_t e = launch_flux<T>(dc.D, dc.nf, dc.vtile, flux_blocks(dc, r), r, st, &dc, nullptr, nullptr, 0);
        if (e == cudaSuccess)
            e = launch_stage1<T>(dc.D, dc.nf, stage1_blocks(dc, r), r, st, &dc, nullptr, nullptr, 0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Work items, threads per block, blocks and dynamic shared memory of the per-case
// kernels of a step (SmallKernel order); 0 items: the case does not run that
// kernel.  The kernels with a thread per cell or face are chains of FP64
// operations, which an SM retires at one warp instruction in 20 cycles: on small
// meshes one-warp blocks spread them over all SMs (20 x 20 cells, 840 faces:
// k_update_W 24 -> 12.5 us, k_macro_grad 27 -> 12.6, k_face_fin1 28 -> 8.7,
// k_face_fin2 29 -> 16, with the operations saved in them).
constexpr int kSpread = 152 * 128;           // up to here one-warp blocks do not fill the chip

template <typename T>
static int sk_items(const DevCase<T> &dc, int k)
{
    const int C = dc.C, F = dc.F;
    const bool sums1 = !dc.w0_analytic;
    switch (k) {
    case SK_PREP: return C + dc.G;
    case SK_FACE_SUM1_SEP: return sums1 && dc.sep1 ? F : 0;
    case SK_FACE_SUM1: return sums1 && !dc.sep1 ? F : 0;
    case SK_FACE_SUM2_SEP: return dc.sep ? F : 0;
    case SK_FACE_SUM2: return !dc.sep ? F : 0;
    case SK_FACE_PRE:
    case SK_FACE_FIN1:
    case SK_FACE_FIN2: return F;
    case SK_WALL_SUM: return dc.NW;
    case SK_MACRO_GRAD:
    case SK_UPDATE_W:
    case SK_COLLIDE: return C;
    default: return 0;
    }
}

static int sk_threads(int k, long long items)
{
    switch (k) {
    case SK_FACE_SUM1_SEP: return 32 * SUM1_SEP_WARPS;
    case SK_FACE_SUM1:
    case SK_FACE_SUM2_SEP:
    case SK_FACE_SUM2:
    case SK_WALL_SUM:
    case SK_COLLIDE: return 256;
    case SK_FACE_FIN2: return items <= kSpread ? 32 : 64;
    default: return items <= kSpread ? 32 : 128;
    }
}

// items per block: a warp each in the sums and the collision pass, a block each
// in the wall pass, a thread each in the others
static int sk_blocks(int k, int items, int threads)
{
    switch (k) {
    case SK_WALL_SUM: return items;
    case SK_FACE_SUM1_SEP:
    case SK_FACE_SUM1:
    case SK_FACE_SUM2_SEP:
    case SK_FACE_SUM2:
    case SK_COLLIDE: return cdiv(items, threads / 32);
    default: return cdiv(items, threads);
    }
}

template <typename T, int D>
static size_t sk_smem(const DevCase<T> &dc, int k)
{
    // k_face_sum1_sep: prefix sums of the last axis, 2 sides x 3 powers per warp
    return k == SK_FACE_SUM1_SEP ? (size_t)SUM1_SEP_WARPS * 6 * (dc.cart_n[D - 1] + 1) * sizeof(T) : 0;
}

// one per-case kernel, for one case (cases == nullptr) or for the cases of a
// batch (block offsets off[0..n])
template <typename T, int D, int NC>
static cudaError_t sk_launch(int k, int blocks, int nt, size_t smem, cudaStream_t st, const DevCase<T> *dc,
                             const DevCase<T> *cases, const int *off, int n)
{
    if (blocks <= 0) return cudaSuccess;
#define UGKS_SK(ID, K)                                                                                  \
    case ID:                                                                                            \
        return cases ? launch(K##_batch<T, D, NC>, blocks, nt, smem, st, cases, off, n)                 \
                     : launch(K<T, D, NC>, blocks, nt, smem, st, *dc);
    if (k == SK_FACE_SUM1_SEP && smem > 48 * 1024) {
        cudaError_t e = cases ? cudaFuncSetAttribute(k_face_sum1_sep_batch<T, D, NC>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                              : cudaFuncSetAttribute(k_face_sum1_sep<T, D, NC>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    switch (k) {
        UGKS_SK(SK_PREP, k_prep)
        UGKS_SK(SK_MACRO_GRAD, k_macro_grad)
        UGKS_SK(SK_FACE_PRE, k_face_pre)
        UGKS_SK(SK_FACE_SUM1_SEP, k_face_sum1_sep)
        UGKS_SK(SK_FACE_SUM1, k_face_sum1)
        UGKS_SK(SK_FACE_FIN1, k_face_fin1)
        UGKS_SK(SK_FACE_SUM2_SEP, k_face_sum2_sep)
        UGKS_SK(SK_FACE_SUM2, k_face_sum2)
        UGKS_SK(SK_FACE_FIN2, k_face_fin2)
        UGKS_SK(SK_WALL_SUM, k_wall_sum)
        UGKS_SK(SK_UPDATE_W, k_update_W)
        UGKS_SK(SK_COLLIDE, k_collide)
    default: return cudaErrorInvalidValue;
    }
#undef UGKS_SK
}

template <typename T, int D, int NC>
static void sk_case(const DevCase<T> &dc, int k, cudaStream_t st)
{
    const int items = sk_items(dc, k), nt = sk_threads(k, items);
    sk_launch<T, D, NC>(k, sk_blocks(k, items, nt), nt, sk_smem<T, D>(dc, k), st, &dc, nullptr, nullptr, 0);
}

template <typename T, int D, int NC>
static void pre_gather(const DevCase<T> &dc, cudaStream_t st, cudaEvent_t *ev)
{
    auto mark = [&](int i) {
        if (ev) cudaEventRecord(ev[i], st);
    };
    mark(0);
    sk_case<T, D, NC>(dc, SK_PREP, st);
    sk_case<T, D, NC>(dc, SK_MACRO_GRAD, st);
    mark(1);
    for (int k = SK_FACE_PRE; k <= SK_FACE_FIN2; ++k) sk_case<T, D, NC>(dc, k, st);
    mark(2);
    sk_case<T, D, NC>(dc, SK_WALL_SUM, st);
    mark(3);
}

template <typename T, int D, int NC>
static void post_gather(const DevCase<T> &dc, cudaStream_t st, cudaEvent_t *ev)
{
    auto mark = [&](int i) {
        if (ev) cudaEventRecord(ev[i], st);
    };
    mark(4);
    sk_case<T, D, NC>(dc, SK_UPDATE_W, st);
    mark(5);
    sk_case<T, D, NC>(dc, SK_COLLIDE, st);
    mark(6);
}

template <typename T, int D, int NC>
static cudaError_t step_dn(const DevCase<T> &dc, cudaStream_t st, cudaEvent_t *ev)
{
    pre_gather<T, D, NC>(dc, st, ev);
    cudaError_t e = launch_gather(dc, st);
    if (e != cudaSuccess) return e;
    post_gather<T, D, NC>(dc, st, ev);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pre_gather(const DevCase<T> &dc, cudaStream_t st)
{
    if (dc.D == 2) pre_gather<T, 2, 2>(dc, st, nullptr);
    else pre_gather<T, 3, 1>(dc, st, nullptr);
    return cudaGetLastError();
}

template <typename T>
int small_kernel_items(const DevCase<T> &dc, int k)
{
    return sk_items(dc, k);
}

int small_kernel_threads(int k, long long items) { return sk_threads(k, items); }

int small_kernel_blocks(int k, int items, int threads) { return sk_blocks(k, items, threads); }

template <typename T>
size_t small_kernel_smem(const DevCase<T> &dc, int k)
{
    return dc.D == 2 ? sk_smem<T, 2>(dc, k) : sk_smem<T, 3>(dc, k);
}

template <typename T>
cudaError_t launch_small_batch(int D, int k, const DevCase<T> *cases, const int *off, int n, int blocks, int threads,
                               size_t smem, cudaStream_t st)
{
    if (D == 2) return sk_launch<T, 2, 2>(k, blocks, threads, smem, st, nullptr, cases, off, n);
    return sk_launch<T, 3, 1>(k, blocks, threads, smem, st, nullptr, cases, off, n);
}

template <typename T>
cudaError_t launch_step(const DevCase<T> &dc, cudaStream_t st, cudaEvent_t *ev)
{
    return dc.D == 2 ? step_dn<T, 2, 2>(dc, st, ev) : step_dn<T, 3, 1>(dc, st, ev);
}

template <typename T>
cudaError_t launch_init(const DevCase<T> &dc, cudaStream_t st)
{
    if (dc.D == 2) {
        k_init_f<T, 2, 2><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
        k_heatflux<T, 2, 2><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
    } else {
        k_init_f<T, 3, 1><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
        k_heatflux<T, 3, 1><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_heatflux(const DevCase<T> &dc, cudaStream_t st)
{
    if (dc.D == 2) k_heatflux<T, 2, 2><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
    else k_heatflux<T, 3, 1><<<cdiv(dc.C, 8), 256, 0, st>>>(dc);
    return cudaGetLastError();
}

template <typename T, typename S>
cudaError_t launch_f_export(const DevCase<T> &dc, const long long *perm, int c0, int nc, S *out, cudaStream_t st)
{
    long long n = (long long)nc * (dc.D == 2 ? 2 : 1) * dc.nv;
    if (n == 0) return cudaSuccess;
    if (dc.D == 2) k_f_export<T, 2, 2, S><<<cdiv(n, 256), 256, 0, st>>>(dc, perm, c0, nc, out);
    else k_f_export<T, 3, 1, S><<<cdiv(n, 256), 256, 0, st>>>(dc, perm, c0, nc, out);
    return cudaGetLastError();
}

template <typename T, typename S>
cudaError_t launch_f_import(const DevCase<T> &dc, const long long *perm, int c0, int nc, const S *in,
                            cudaStream_t st)
{
    long long n = (long long)nc * (dc.D == 2 ? 2 : 1) * dc.nvp;
    if (n == 0) return cudaSuccess;
    if (dc.D == 2) k_f_import<T, 2, 2, S><<<cdiv(n, 256), 256, 0, st>>>(dc, perm, c0, nc, in);
    else k_f_import<T, 3, 1, S><<<cdiv(n, 256), 256, 0, st>>>(dc, perm, c0, nc, in);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_halo(const DevCase<T> &dc, const int *cells, int n, size_t row, void *buf, int unpack,
                        cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    if (dc.D == 2) {
        if (unpack) k_halo_unpack<T, 2, 2><<<n, 128, 0, st>>>(dc, cells, n, row, (const unsigned char *)buf);
        else k_halo_pack<T, 2, 2><<<n, 128, 0, st>>>(dc, cells, n, row, (unsigned char *)buf);
    } else {
        if (unpack) k_halo_unpack<T, 3, 1><<<n, 128, 0, st>>>(dc, cells, n, row, (const unsigned char *)buf);
        else k_halo_pack<T, 3, 1><<<n, 128, 0, st>>>(dc, cells, n, row, (unsigned char *)buf);
    }
    return cudaGetLastError();
}
template cudaError_t launch_halo<double>(const DevCase<double> &, const int *, int, size_t, void *, int,
                                         cudaStream_t);
template cudaError_t launch_halo<float>(const DevCase<float> &, const int *, int, size_t, void *, int,
                                        cudaStream_t);

cudaError_t launch_residual(const double *res_part, int nparts, int D, double *res, cudaStream_t st)
{
    if (D == 2) k_residual<4><<<1, RES_THREADS, 0, st>>>(res_part, nparts, res);
    else k_residual<5><<<1, RES_THREADS, 0, st>>>(res_part, nparts, res);
    return cudaGetLastError();
}

cudaError_t launch_residual_fold(const double *res_part, int nparts, int D, double *out, cudaStream_t st)
{
    const int nvals = 2 * (D + 2), n = cdiv(nparts, RES_FOLD) * nvals;
    if (n > 0) k_residual_fold<<<cdiv(n, 256), 256, 0, st>>>(res_part, nparts, nvals, out);
    return cudaGetLastError();
}

cudaError_t launch_moments_out(const double *W, const double *q, const long long *perm, int C, int D,
                               double *out, cudaStream_t st)
{
    if (C == 0) return cudaSuccess;
    if (D == 2) k_moments_out<2><<<cdiv(C, 128), 128, 0, st>>>(W, q, perm, C, out);
    else k_moments_out<3><<<cdiv(C, 128), 128, 0, st>>>(W, q, perm, C, out);
    return cudaGetLastError();
}

cudaError_t launch_W_permute(const double *src, const long long *perm, int C, int D, double *dst,
                             int to_internal, cudaStream_t st)
{
    if (C == 0) return cudaSuccess;
    if (D == 2) k_W_permute<2><<<cdiv(C, 128), 128, 0, st>>>(src, perm, C, dst, to_internal);
    else k_W_permute<3><<<cdiv(C, 128), 128, 0, st>>>(src, perm, C, dst, to_internal);
    return cudaGetLastError();
}

cudaError_t launch_check(const double *W, int C, int M, int *flags, cudaStream_t st)
{
    if (C == 0) return cudaSuccess;
    k_check<<<cdiv(C, 128), 128, 0, st>>>(W, C, M, flags);
    return cudaGetLastError();
}

cudaError_t launch_density_range(const double *W, int C, int M, const unsigned char *owned,
                                 unsigned long long *range, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(&range[0], 0xff, sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(&range[1], 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess || C == 0) return e;
    k_density_range<<<std::min(cdiv(C, 256), 1024), 256, 0, st>>>(W, C, M, owned, range);
    return cudaGetLastError();
}

template cudaError_t launch_pre_gather<double>(const DevCase<double> &, cudaStream_t);
template cudaError_t launch_pre_gather<float>(const DevCase<float> &, cudaStream_t);
template int small_kernel_items<double>(const DevCase<double> &, int);
template int small_kernel_items<float>(const DevCase<float> &, int);
template size_t small_kernel_smem<double>(const DevCase<double> &, int);
template size_t small_kernel_smem<float>(const DevCase<float> &, int);
template cudaError_t launch_small_batch<double>(int, int, const DevCase<double> *, const int *, int, int, int,
                                                size_t, cudaStream_t);
template cudaError_t launch_small_batch<float>(int, int, const DevCase<float> *, const int *, int, int, int, size_t,
                                               cudaStream_t);
#define UGKS_GATHER(T)                                                                                        \
    template cudaError_t launch_flux<T>(int, int, int, int, int, cudaStream_t, const DevCase<T> *,            \
                                        const DevCase<T> *, const int *, int);                                \
    template cudaError_t launch_stage1<T>(int, int, int, int, cudaStream_t, const DevCase<T> *,               \
                                          const DevCase<T> *, const int *, int);                              \
    template int flux_blocks<T>(const DevCase<T> &, int);                                                     \
    template int stage1_blocks<T>(const DevCase<T> &, int);                                                   \
    template cudaError_t launch_gather<T>(const DevCase<T> &, cudaStream_t);                                  \
    template cudaError_t launch_step<T>(const DevCase<T> &, cudaStream_t, cudaEvent_t *);
UGKS_GATHER(double)
UGKS_GATHER(float)
#undef UGKS_GATHER
template cudaError_t launch_init<double>(const DevCase<double> &, cudaStream_t);
template cudaError_t launch_init<float>(const DevCase<float> &, cudaStream_t);
template cudaError_t launch_heatflux<double>(const DevCase<double> &, cudaStream_t);
template cudaError_t launch_heatflux<float>(const DevCase<float> &, cudaStream_t);
#define UGKS_STATE_IO(T, S)                                                                                   \
    template cudaError_t launch_f_export<T, S>(const DevCase<T> &, const long long *, int, int, S *, cudaStream_t); \
    template cudaError_t launch_f_import<T, S>(const DevCase<T> &, const long long *, int, int, const S *,          \
                                               cudaStream_t);
UGKS_STATE_IO(double, double)
UGKS_STATE_IO(double, float)
UGKS_STATE_IO(float, double)
UGKS_STATE_IO(float, float)
#undef UGKS_STATE_IO

}  // namespace ugks
