// ugks_device.cuh -- device-side data layout and per-velocity building blocks
// of the GB300 UGKS library (internal; not part of the C ABI).
//
// Layout in HBM (internal cell order = Morton order of the centroids):
//   f      [C][NC][nvp]  T   distribution, updated in place, NC = 2 (h, b) in 2D, 1 (h) in 3D,
//                            velocity contiguous, padded to a multiple of the
//                            velocity tile (padded velocities have u = 0, w = 0)
//   W      [C][D+2]      f64 conserved variables
//   q      [C][D]        f64 heat flux of f^n
//   cell records [C][CREC] T   Maxwellian / Shakhov / collision coefficients
//   flux records [F][XREC] T   interface equilibrium g0, its slopes, q1, q2
// T is the per-velocity arithmetic type (double or float).
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

namespace ugks {

constexpr int MAXD = 3;
constexpr int MAXM = 5;

// cell record: Maxwellian of the cell state plus Shakhov and collision factors
// (CR_C = dt / (2 tau) and CR_INV = 1 / (1 + dt / (2 tau)), both formed in FP64)
enum { CR_U = 0, CR_LAM = 3, CR_PREF = 4, CR_KQ = 5, CR_C = 8, CR_NB = 9, CR_NL2 = 10, CR_INV = 11, CREC = 12 };
// ghost / side / wall record: a Maxwellian
enum { GR_U = 0, GR_LAM = 3, GR_PREF = 4, GR_NB = 5, GR_NL2 = 6, GREC = 8 };
// face record: the Maxwellian g0 of the interface, read by the sums of k_face_sum2
enum { FR_U = 0, FR_LAM = 3, FR_PREF = 4, FR_NL2 = 5, FREC = 8 };

// flux record read by the flux pass: the equilibrium part of the
// time-integrated interface distribution, q3 (g0 + g0+) + q4 u.grad g0 +
// q5 dg0/dt, is H0(c) P_m(c) with c = u - U0, H0 = PREF e^{-lam |c|^2} (the factor
// PREF is multiplied into the coefficients in the FP64 form) and, per
// stored component m, P_m(c) = a0 + a.c + sum_{e<=f} B_ef c_e c_f + (gamma.c)|c|^2.
// U = -U0; EX = the coefficient gauss_ex() takes (-lam, or -lam log2 e in FP32)
template <int D> struct Poly {
    static constexpr int NB = D * (D + 1) / 2;
    static constexpr int N = 1 + D + NB + D;   // a0, a, B (packed upper, off-diagonal doubled), gamma
};
template <int D> struct XRec {
    static constexpr int U = 0, EX = D, Q1 = D + 1, Q2 = D + 2, PREF = D + 3, POLY = D + 4;
    static constexpr int LEN = (POLY + (4 - D) * Poly<D>::N + 3) / 4 * 4;   // 24 in 2D, 20 in 3D
};

// FT_NONE: an entry that pads a cell to the entry count of the mesh
enum { FT_INTERIOR = 0, FT_WALL = 1, FT_FARFIELD = 2, FT_PERIODIC = 3, FT_NONE = 4 };

// nodes of the last velocity axis the separable half-range sums hold in shared memory
constexpr int SUM1_SEP_MAX_NL = 512;

// largest face count the entries are padded to (hexahedra)
constexpr int MAX_NF = 6;

// layout of the values of one entry (cell c, face f): a = LSQ coefficient of
// the neighbour across f (0 for a wall), rs = x_f - x_c, n = unit normal of f
// pointing out of its owner, cs = -sigma S_f / |Omega_c| with sigma = 1 for the
// owner and -1 for the neighbour, so that the flux F of f in the owner's
// orientation enters c as cs F.  Grouped in 16-byte vectors so that each pass
// loads only what it reads: a and rs by the slopes, rs and n by the fluxes, cs
// by stage 1.
template <int D> struct GEnt;
template <> struct GEnt<2> {
    static constexpr int A = 0, RS = 2, N = 4, CS = 6, LEN = 8;
};
template <> struct GEnt<3> {
    static constexpr int RS = 0, CS = 3, A = 4, N = 8, LEN = 12;
};

// Everything a kernel needs, by value.  Geometry used inside velocity loops is
// held in the arithmetic type T; macroscopic data is FP64.
template <typename T>
struct DevCase {
    int D, NC;
    int C, F, G, NW;         // cells, faces, far-field ghosts, wall faces
    int nv, nvp;             // velocities, padded count
    double dt, Pr, omega, nxi;
    double dt_mu;                 // dt / mu_ref (0: collisionless)
    int limiter;
    int w0_analytic;              // 1: W0 from the analytic half-range moments
    // velocity grid (padded)
    const T *u[3], *w;
    const T *uw;                  // [nvp][4] (u_x, u_y, u_z or 0, w) packed for one vector load
    // distribution, updated in place: f^n, then f~ (stage 1), then f^{n+1}
    T *f_cur;
    // time-integrated flux of every face in its owner's orientation for one
    // chunk of velocities: [F][NC][chunk]
    T *flux;
    // macroscopic state
    double *W, *q, *gradW;
    double *prim, *primg, *gradprim;  // primitive (rho, U, T) of cells / ghosts, limited gradient
    // least squares (CSR over cells)
    const int *nb_ptr, *nb_id;    // id >= 0: cell, id < 0: ghost -(id+1)
    const double *nb_a_d;
    // faces of each cell (CSR): limiter offsets and gather entries
    const int *cf_ptr;
    const double *cf_r_d;         // x_f - x_c (periodic image on the neighbour side)
    // entries, one per (cell, face) in cf order: gi = {row, face, type + 256
    // (cell owns the face), ghost or wall slot} with row the neighbour cell
    // (interior, periodic) or the cell itself; gf = GEnt<D> values.  nf > 0:
    // every cell has nf entries (the largest face count of the mesh, if at most
    // MAX_NF), padded with FT_NONE; nf = 0: the cells' own counts (cf_ptr)
    const int4 *gi;
    const T *gf;
    int nf;
    const double *eps2_d;
    const T *eps2;
    // faces
    const int *fL, *fR, *faux;    // owner, neighbour (-1 at boundaries), ghost or wall slot
    const signed char *ftype;
    const double *fn_d, *frL_d, *frR_d;
    const T *fn, *frL;            // T copies used inside velocity loops
    T dtT;                        // dt in the arithmetic type
    T one;                        // 1 (see psum)
    // ghosts (one per far-field face)
    const int *gface;
    double *Wg;                   // [G][D+2]
    T *grec;                      // [G][GREC]
    // walls
    const int *wface;             // [NW] face id
    const double *wallT, *wallU;  // per wall tag
    const int *ftag;
    double inf_W[MAXM];
    double *rho_w;                // [NW]
    double *wall_F;               // [NW][D+2] macroscopic wall flux over the last step (Eq. macroscopicFlux)
    T *wrec;                      // [NW][GREC]
    // per-step work
    T *crec;                      // [C][CREC] stage-1 record (W^n, q^n)
    T *krec;                      // [C][CREC] stage-2 record (W^{n+1}, q^n)
    T *frec;                      // [F][FREC] face-pass work record
    T *xrec;                      // [F][XREC] flux record of the gather pass
    T *fside;                     // [F][2][GREC] Maxwellians of the face states
    double *fdW0;                 // [F][D][D+2] interface macro gradient
    double *fq0;                  // [F][D]
    double *fUref;                // [F][D]
    double *fsum1, *fsum2;        // [F][S1], [F][S2]
    double *fprim0;               // [F][D+2] rho0, U0, lam0
    double *fqs;                  // [F][5] time integrals q1..q5 of the interface
    double *dW_part;              // [C][n_groups][D+2] moments of the flux residual over gvel velocities
    double *res_part;             // [ceil(C / 32)][2(D+2)]
    const unsigned char *owned;   // [C] 1 for cells whose residual counts (a subdomain's own cells),
                                  // nullptr: every cell
    int *flags;                   // [1] numeric failure flag
    // tensor-product velocity grid (sep = 1): axes and 1-D weights per dimension
    int sep, cart_n[3];
    int sep1;                     // sep with the last axis strictly ascending and at most
                                  // SUM1_SEP_MAX_NL nodes (separable half-range sums)
    const T *axis[3], *axw[3];
    // tiling of the flux and stage-1 passes
    int P, n_patches, vtile;      // cells per patch and velocities per warp of the flux pass
    int nth;                      // threads per patch (256, or 512 for FP32 at vtile <= 64), in CTAs of 128
    int chunk, n_chunks;          // velocities per chunk, chunks (see chunk_span)
    int gvel, n_groups;           // velocities of a cell per warp of stage 1 (whole tiles, or all), groups per cell
    int parts;                    // chunks per group: 1 (a chunk holds one group or several), or more
    T *carry;                     // parts > 1: lane sums of a group between its chunks, [C][D+2][32] of MomentSum
};

// First velocity of chunk r and the number of its velocities (<= 0: the case
// has no such chunk).  A chunk holds whole groups of gvel velocities, or, where
// the flux buffer cannot hold a group, is one of the parts of a group (multiples
// of 128 velocities, so that a lane of stage 1 keeps its velocities).
template <typename T>
__host__ __device__ __forceinline__ void chunk_span(const DevCase<T> &dc, int r, int &kb, int &len)
{
    kb = r * dc.chunk;
    int end = kb + dc.chunk;
    if (dc.parts > 1) {
        const int g = r / dc.parts;
        kb += g * (dc.gvel - dc.parts * dc.chunk);
        end = kb + dc.chunk < (g + 1) * dc.gvel ? kb + dc.chunk : (g + 1) * dc.gvel;
    }
    if (end > dc.nvp) end = dc.nvp;
    len = end - kb;
}

// ------------------------------------------------------------------ math
// 2^x with the hardware approximation (relative error ~2^-22); FP32 only
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// exp(x) in FP64 for the Maxwellians, after Tang's table-driven scheme (ACM TOMS 15, 1989):
// x = (64 m + j) ln2/64 + r with |r| <= ln2/128, exp(x) = 2^m 2^(j/64) (1 + q(r)),
// q the Taylor polynomial of degree 5 of e^r - 1 (next term 3e-17).  EXP2_64[j] =
// 2^(j/64) as the nearest double and the remainder.  Eleven FP64 operations where
// the library function costs the time of fourteen multiplications (an SM retires
// 1.6 of them per cycle, which bounds the FP64 form: flux and stage-1 passes of
// 8k triangles x 60x50 14.6 -> 14.0 ms, collision pass 1.77 -> 1.62); measured on
// 10^6 arguments, error 0.81 units in the last place at most and 0.253 in the
// mean, against 0.84 and 0.255 of exp().
// Below -700 the result is 0 (the true value is under 1e-304).
__device__ const double2 EXP2_64[64] = {
    {1, 0}, {1.0108892860517005, -1.5234778603368577e-17},
    {1.0218971486541166, 5.1092250289734439e-17}, {1.0330248790212284, 7.6008388740270885e-18},
    {1.0442737824274138, 8.5518897055379649e-17}, {1.0556451783605572, 1.759325738772092e-18},
    {1.0671404006768237, -7.8998539668415821e-17}, {1.0787607977571199, -6.6566604360565926e-17},
    {1.0905077326652577, -3.0467820798124711e-17}, {1.1023825833078409, 5.2660368715706944e-17},
    {1.1143867425958924, 1.0410278456845571e-16}, {1.1265216186082418, 5.1658567587954567e-17},
    {1.1387886347566916, 8.9128126760254078e-17}, {1.1511892299529827, 3.2507102188638272e-17},
    {1.1637248587775775, 3.8292048369240935e-17}, {1.1763969916502812, 5.554203254218079e-17},
    {1.189207115002721, 3.9820152314656461e-17}, {1.2021567314527031, 6.6449814992523012e-17},
    {1.215247359980469, -7.7126306926814881e-17}, {1.22848053610687, -1.89878163130253e-17},
    {1.241857812073484, 4.6580275918369368e-17}, {1.2553807570246911, -6.7113898212968784e-18},
    {1.2690509571917332, 2.6679321313421861e-18}, {1.2828700160787783, 1.713594918243561e-17},
    {1.2968395546510096, 2.5382502794888315e-17}, {1.3109612115247644, -7.1815361355194539e-17},
    {1.3252366431597413, -2.8587312100388614e-17}, {1.3396675240533029, 8.927282594831732e-17},
    {1.3542555469368927, 7.7009483798029895e-17}, {1.3690024229745905, 9.5937979191188488e-17},
    {1.383909881963832, -6.7705116587947863e-17}, {1.3989796725383112, -9.6142132090513231e-17},
    {1.4142135623730951, -9.6672933134529135e-17}, {1.42961333839197, -1.2031642489053655e-17},
    {1.4451808069770467, -3.0237581349939873e-17}, {1.460917794180647, -5.6003771860752158e-17},
    {1.4768261459394993, -3.4839945568927958e-17}, {1.4929077282912648, 1.4192920154284036e-17},
    {1.5091644275934228, -1.016455327754295e-16}, {1.5255981507445384, -1.1024941712342561e-16},
    {1.5422108254079407, 7.9498348096976209e-17}, {1.5590044002378369, 3.7812070533575275e-17},
    {1.5759808451078865, -1.0136916471278304e-17}, {1.593142151342267, -1.0094406542311964e-16},
    {1.6104903319492543, 2.4707192569797888e-17}, {1.6280274218573478, -6.7129550847070841e-17},
    {1.6457554781539649, -1.0125679913674773e-16}, {1.6636765803267364, 5.8909926967130997e-17},
    {1.681792830507429, 8.1990100205814965e-17}, {1.7001063537185235, -8.0237193703977002e-18},
    {1.7186192981224779, -1.851380418263111e-17}, {1.7373338352737062, 3.1643892992929569e-17},
    {1.7562521603732995, 2.9601406954488733e-17}, {1.7753764925265212, 6.429731796556572e-17},
    {1.7947090750031072, 1.8227458427912087e-17}, {1.8142521755003989, -9.9695315389203488e-17},
    {1.8340080864093424, 3.2831072242456272e-17}, {1.8539791250833855, 9.7618874907275935e-17},
    {1.8741676341103, -6.1227634130041426e-17}, {1.8945759815869656, 3.4034035352165297e-17},
    {1.9152065613971474, -1.0619946056195963e-16}, {1.9360617934922943, 1.0332385960676326e-16},
    {1.9571441241754002, 8.9607677910366678e-17}, {1.9784560263879509, 4.0388753109278167e-17},
};

__device__ __forceinline__ double exp_neg(double x)
{
    const double magic = 6755399441055744.0;                 // 1.5 * 2^52: the sum's low word is the integer
    const double t = fma(x, 92.332482616893657, magic);                   // 64 / ln2
    const double k = t - magic;
    double r = fma(k, -0.010830424696249145, x);                            // ln2 / 64, high and low part
    r = fma(k, -3.6235106466348431e-19, r);
    const int n = __double2loint(t);
    const double2 s = __ldg(EXP2_64 + (n & 63));
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    const double q = fma(p, r * r, r);
    const double e = s.x + fma(s.x, q, s.y);
    const double v = __hiloint2double(__double2hiint(e) + ((n >> 6) << 20), __double2loint(e));
    if ((unsigned)(__double2hiint(x) & 0x7fffffff) < 0x4085E000u) return v;    // |x| < 700
    return x < 0.0 ? 0.0 : exp(x);                           // also NaN and a broken state's growth
}

// exp(-lambda c2) of a record: FP64 through exp_neg(), FP32 through 2^(nl2 c2)
// with nl2 = -lambda log2(e) precomputed in the record
template <typename T> __device__ __forceinline__ T gauss(T lam, T nl2, T c2);
template <> __device__ __forceinline__ double gauss<double>(double lam, double, double c2) { return exp_neg(-lam * c2); }
template <> __device__ __forceinline__ float gauss<float>(float, float nl2, float c2) { return ex2_approx(nl2 * c2); }

template <typename T> __device__ __forceinline__ T mul_rn(T a, T b);
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <typename T> __device__ __forceinline__ T add_rn(T a, T b);
template <> __device__ __forceinline__ double add_rn<double>(double a, double b) { return __dadd_rn(a, b); }
template <> __device__ __forceinline__ float add_rn<float>(float a, float b) { return __fadd_rn(a, b); }

// u . n without contraction: the upwind and half-range decisions are taken
// from exactly the same rounded value as the oracle computes
template <typename T, int D>
__device__ __forceinline__ T normal_velocity(const T u[3], const T *n)
{
    T s = mul_rn(u[0], n[0]);
    s = add_rn(s, mul_rn(u[1], n[1]));
    if (D == 3) s = add_rn(s, mul_rn(u[2], n[2]));
    return s;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------------ moment sums
// Velocity-moment sums of the FP32 form are compensated: a lane accumulates
// its FP32 terms with Kahan's correction (the running sum s and the rounding
// error c lost so far; the sum is s - c, returned in FP64), and the lanes'
// sums are combined in FP64.  The FP64 form sums plainly in FP64.  The
// corrections rely on IEEE rounding of every addition: nothing here may be
// reassociated or contracted (no fast-math flags).
template <typename T> struct CSum;
template <> struct CSum<double> {
    double s;
    __device__ __forceinline__ CSum() : s(0.0) {}
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct CSum<float> {
    float s, c;
    __device__ __forceinline__ CSum() : s(0.f), c(0.f) {}
    __device__ __forceinline__ void add(float x)
    {
        const float y = __fsub_rn(x, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// Blocked accumulation in FP64 for sums with many terms per lane and many
// values (the face sums): every lane adds at most SUM_BLOCK of its FP32 terms
// per value into blk[] (a block of 32 x SUM_BLOCK terms per warp), the warp
// combines each block value across lanes (warp_transpose_sum, FP32), and the
// block totals are accumulated in FP64, lane j holding value j >> (5 - log2 N).
// The FP32 part of every sum spans one block, so its rounding error is bounded
// by about (SUM_BLOCK + 5) units in the last place of the block's absolute sum
// whatever the number of terms.
constexpr int SUM_BLOCK = 16;

// Error-free sum of two FP32 values (Knuth's TwoSum): a + b = s + e exactly.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

// Double-float addition (hi, lo) += (bh, bl): about 44 significant bits, with
// FP32 instructions only (FP64 arithmetic is scarce on this part).
__device__ __forceinline__ void ff_add(float &hi, float &lo, float bh, float bl)
{
    float s, e;
    two_sum(hi, bh, s, e);
    e = __fadd_rn(e, __fadd_rn(lo, bl));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// warp_transpose_sum on double-float pairs (h, l): the same exchange pattern,
// with every addition a double-float addition.  On return (oh, ol) is the
// full sum of value index lane >> (5 - log2 N).
template <int N>
__device__ __forceinline__ void warp_transpose_sum_ff2(float (&h)[N], float (&l)[N], float &oh, float &ol)
{
    const int lane = threadIdx.x & 31;
    int n = N;
#pragma unroll
    for (int bit = 16; n > 1; bit >>= 1) {
        n >>= 1;
        const bool upper = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            if (i >= n) break;
            const float sh = upper ? h[i] : h[i + n], sl = upper ? l[i] : l[i + n];
            const float kh = upper ? h[i + n] : h[i], kl = upper ? l[i + n] : l[i];
            const float rh = __shfl_xor_sync(0xffffffffu, sh, bit), rl = __shfl_xor_sync(0xffffffffu, sl, bit);
            h[i] = kh;
            l[i] = kl;
            ff_add(h[i], l[i], rh, rl);
        }
    }
    constexpr int used = (N == 32) ? 5 : (N == 16) ? 4 : (N == 8) ? 3 : (N == 4 ? 2 : (N == 2 ? 1 : 0));
    float rh = h[0], rl = l[0];
#pragma unroll
    for (int bit = 16 >> used; bit > 0; bit >>= 1) {
        const float qh = __shfl_xor_sync(0xffffffffu, rh, bit), ql = __shfl_xor_sync(0xffffffffu, rl, bit);
        ff_add(rh, rl, qh, ql);
    }
    oh = rh;
    ol = rl;
}

// Sum of N (a power of two up to 32) values over the 32 lanes of a warp by
// recursive halving: at every exchange a lane keeps half of its values and
// receives the partner's partial sums of that half.  On return lane l holds
// the full sum of value index l >> (5 - log2 N) (lanes 8j..8j+7 for N = 4,
// lane j for N = 32).
template <typename T, int N>
__device__ __forceinline__ T warp_transpose_sum(T (&v)[N])
{
    const int lane = threadIdx.x & 31;
    int n = N;
#pragma unroll
    for (int bit = 16; n > 1; bit >>= 1) {
        n >>= 1;
        const bool upper = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            if (i >= n) break;
            const T send = upper ? v[i] : v[i + n];
            const T keep = upper ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
    }
    constexpr int used = (N == 32) ? 5 : (N == 16) ? 4 : (N == 8) ? 3 : (N == 4 ? 2 : (N == 2 ? 1 : 0));
    static_assert((1 << used) == N, "N must be a power of two up to 32");
    T r = v[0];
#pragma unroll
    for (int bit = 16 >> used; bit > 0; bit >>= 1) r += __shfl_xor_sync(0xffffffffu, r, bit);
    return r;
}

// the block step of the blocked FP64 accumulation (see SUM_BLOCK)
template <int N>
__device__ __forceinline__ double block_to_fp64(float (&blk)[N])
{
    return (double)warp_transpose_sum<float, N>(blk);
}

// Shakhov equilibrium f+ = (H + H+, B + B+) of a cell record at velocity u:
// H+ = kappa (c.q)(2 lam c^2 - D - 2) H,  B+ = kappa (c.q)(2 lam c^2 - D) nb H
template <typename T, int D, int NC>
__device__ __forceinline__ void shakhov_fplus(const T *rec, const T u[3], T fp[NC])
{
    T c[D], c2 = 0, kqc = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        c[d] = u[d] - rec[CR_U + d];
        c2 += c[d] * c[d];
        kqc += rec[CR_KQ + d] * c[d];
    }
    T H = rec[CR_PREF] * gauss<T>(rec[CR_LAM], rec[CR_NL2], c2);
    T l2c2 = T(2) * rec[CR_LAM] * c2;
    fp[0] = H * (T(1) + kqc * (l2c2 - T(D + 2)));
    if (NC == 2) fp[NC - 1] = H * rec[CR_NB] * (T(1) + kqc * (l2c2 - T(D)));
}

// TV consecutive values at a TV*sizeof(T)-aligned address, moved in chunks
// of at most 16 bytes.  Two kinds of loads: *_const through the non-coherent
// path, for what no kernel of a step writes (velocities, weights, geometry), and
// ordinary ones for what an earlier kernel of the step wrote (f, the fluxes, the
// records).  A kernel of a step starts before its predecessor has ended
// (dependency_wait), and a non-coherent load may be moved ahead of the wait: it
// asks for memory that is read-only as long as the kernel lives.
template <typename T, int N> struct VecOf;
template <> struct VecOf<float, 1> { using type = float; };
template <> struct VecOf<float, 2> { using type = float2; };
template <> struct VecOf<float, 4> { using type = float4; };
template <> struct VecOf<double, 1> { using type = double; };
template <> struct VecOf<double, 2> { using type = double2; };
template <typename T, int TV> constexpr int vec_chunk() { return TV * (int)sizeof(T) <= 16 ? TV : 16 / (int)sizeof(T); }

template <bool CONST, typename V> __device__ __forceinline__ V ld(const V *p)
{
    if constexpr (CONST) return __ldg(p);
    else return *p;
}
template <bool CONST, typename T, int TV>
__device__ __forceinline__ void ld_lane(const T *p, T (&x)[TV])
{
    constexpr int CH = vec_chunk<T, TV>();
    using V = typename VecOf<T, CH>::type;
#pragma unroll
    for (int i = 0; i < TV / CH; ++i) {
        const V v = ld<CONST>(reinterpret_cast<const V *>(p) + i);
        const T *e = reinterpret_cast<const T *>(&v);
#pragma unroll
        for (int j = 0; j < CH; ++j) x[i * CH + j] = e[j];
    }
}
template <typename T, int TV> __device__ __forceinline__ void ldv_const(const T *p, T (&x)[TV]) { ld_lane<true>(p, x); }
template <typename T, int TV>
__device__ __forceinline__ void stv(T *p, const T (&x)[TV])
{
    constexpr int CH = vec_chunk<T, TV>();
    using V = typename VecOf<T, CH>::type;
#pragma unroll
    for (int i = 0; i < TV / CH; ++i) {
        V v;
        T *e = reinterpret_cast<T *>(&v);
#pragma unroll
        for (int j = 0; j < CH; ++j) e[j] = x[i * CH + j];
        reinterpret_cast<V *>(p)[i] = v;
    }
}

// copy a 16-byte aligned record of N values into registers with vector loads
template <bool CONST, typename T, int N> __device__ __forceinline__ void ld_rec(const T *p, T (&r)[N])
{
    constexpr int CH = 16 / (int)sizeof(T);
    static_assert(N % CH == 0, "record length");
#pragma unroll
    for (int i = 0; i < N / CH; ++i) {
        const typename VecOf<T, CH>::type v = ld<CONST>(reinterpret_cast<const typename VecOf<T, CH>::type *>(p) + i);
        const T *e = reinterpret_cast<const T *>(&v);
#pragma unroll
        for (int j = 0; j < CH; ++j) r[i * CH + j] = e[j];
    }
}
template <int N, typename T> __device__ __forceinline__ void load_rec(const T *p, T (&r)[N]) { ld_rec<false>(p, r); }
template <int N, typename T> __device__ __forceinline__ void load_rec_const(const T *p, T (&r)[N]) { ld_rec<true>(p, r); }

// velocity k and its weight from the packed array, one 16-byte (FP32) or two
// 16-byte (FP64) loads
__device__ __forceinline__ void load_uw(const float *__restrict__ uw, int k, float u[3], float &w)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(uw) + k);
    u[0] = v.x;
    u[1] = v.y;
    u[2] = v.z;
    w = v.w;
}
__device__ __forceinline__ void load_uw(const double *__restrict__ uw, int k, double u[3], double &w)
{
    const double2 a = __ldg(reinterpret_cast<const double2 *>(uw) + 2 * k);
    const double2 b = __ldg(reinterpret_cast<const double2 *>(uw) + 2 * k + 1);
    u[0] = a.x;
    u[1] = a.y;
    u[2] = b.x;
    w = b.y;
}

// ------------------------------------------------------------ packs
// The velocities of a lane are held in packs: pairs of FP32 values worked on by
// the packed instructions (fma/add/mul .f32x2: the arithmetic of two velocities
// per issued instruction at the rounding of the scalar ones; measured on GB300
// at 1.87 packed against 3.6 scalar instructions per cycle and SM, so the
// arithmetic rate is the same but half of the issue slots are free for loads,
// compares and selects), single values otherwise.  Every contraction of the
// formulas on packs, and of what is evaluated beside them per velocity, is
// explicit, so all instantiations of a formula round alike.
template <typename T, int TV> struct Pk {
    static constexpr int W = 1, NP = TV;
    using P = T;
};
template <> struct Pk<float, 2> {
    static constexpr int W = 2, NP = 1;
    using P = float2;
};
template <> struct Pk<float, 4> {
    static constexpr int W = 2, NP = 2;
    using P = float2;
};

__device__ __forceinline__ float pfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double pfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double pmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double padd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float pneg(float a) { return -a; }
__device__ __forceinline__ double pneg(double a) { return -a; }
__device__ __forceinline__ float2 pneg(float2 a) { return __fmul2_rn(a, make_float2(-1.f, -1.f)); }

// Maxwellian H and the b-factor of a record (cell / ghost / side / wall)
template <typename T, int D>
__device__ __forceinline__ T maxwell_h(const T *rec, const T u[3])
{
    T c2 = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const T c = u[d] - rec[GR_U + d];
        c2 = pfma(c, c, c2);
    }
    return rec[GR_PREF] * gauss<T>(rec[GR_LAM], rec[GR_NL2], c2);
}

// the same value in every element
template <typename P> __device__ __forceinline__ P pbc(double v);
template <> __device__ __forceinline__ double pbc<double>(double v) { return v; }
template <typename P> __device__ __forceinline__ P pbc(float v);
template <> __device__ __forceinline__ float pbc<float>(float v) { return v; }
template <> __device__ __forceinline__ float2 pbc<float2>(float v) { return make_float2(v, v); }

// element j of a lane's velocities
template <int W, typename P> __device__ __forceinline__ auto &pel(P *x, int j)
{
    if constexpr (W == 1) return x[j];
    else return (j & 1) ? x[j >> 1].y : x[j >> 1].x;
}

// TV consecutive values into packs
template <bool CONST, typename T, int TV>
__device__ __forceinline__ void ld_pack(const T *p, typename Pk<T, TV>::P (&x)[Pk<T, TV>::NP])
{
    T v[TV];
    ld_lane<CONST>(p, v);
#pragma unroll
    for (int j = 0; j < TV; ++j) pel<Pk<T, TV>::W>(x, j) = v[j];
}
template <typename T, int TV>
__device__ __forceinline__ void ldp(const T *p, typename Pk<T, TV>::P (&x)[Pk<T, TV>::NP]) { ld_pack<false, T, TV>(p, x); }
template <typename T, int TV>
__device__ __forceinline__ void ldp_const(const T *p, typename Pk<T, TV>::P (&x)[Pk<T, TV>::NP]) { ld_pack<true, T, TV>(p, x); }

// a + b where a is a product that must not be contracted into the sum.  ptxas
// fuses a packed multiplication and addition even where both carry .rn (the
// scalar ones it leaves alone; measured: mul.rn.f32x2 + add.rn.f32x2 rounds
// once), so the packed sum is an fma with a factor of 1 that the compiler does
// not see, one = DevCase::one.
__device__ __forceinline__ float psum(float a, float b, float) { return __fadd_rn(a, b); }
__device__ __forceinline__ double psum(double a, double b, double) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 psum(float2 a, float2 b, float one) { return __ffma2_rn(a, make_float2(one, one), b); }

// u . n without contraction, as normal_velocity
template <typename T, int D, typename P>
__device__ __forceinline__ P pnormal(const P (&u)[D], const T *n, T one)
{
    P s = psum(pmul(u[0], pbc<P>(n[0])), pmul(u[1], pbc<P>(n[1])), one);
    if constexpr (D == 3) s = psum(pmul(u[D - 1], pbc<P>(n[D - 1])), s, one);
    return s;
}

// exp(-lam c2) from the record's coefficient (-lam; -lam log2 e in FP32)
__device__ __forceinline__ float gauss_ex(float ex, float c2) { return ex2_approx(__fmul_rn(ex, c2)); }
__device__ __forceinline__ double gauss_ex(double ex, double c2) { return exp_neg(ex * c2); }
__device__ __forceinline__ float2 gauss_ex(float ex, float2 c2)
{
    const float2 t = pmul(c2, make_float2(ex, ex));
    return make_float2(ex2_approx(t.x), ex2_approx(t.y));
}

// Sign tests and running extrema.  A double compare costs as much as an FP64
// multiply (an SM retires 1.6 of either per cycle), so FP64 values are compared
// as integers: the bits of a double order as its value for non-negative ones,
// and for all after the magnitude bits of the negative ones are inverted.
__device__ __forceinline__ bool gt0(float x) { return x > 0.f; }
__device__ __forceinline__ bool lt0(float x) { return x < 0.f; }
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool lt0(double x)
{
    const long long b = __double_as_longlong(x);
    return b < 0 && b != (long long)0x8000000000000000ull;
}

// min(x, 0)
__device__ __forceinline__ float min0(float x) { return fminf(x, 0.f); }
__device__ __forceinline__ double min0(double x) { return lt0(x) ? x : 0.0; }

template <typename T> struct Extrema;
template <> struct Extrema<float> {
    float hi, lo;
    __device__ __forceinline__ void set(float x) { hi = lo = x; }
    __device__ __forceinline__ void add(float x)
    {
        hi = fmaxf(hi, x);
        lo = fminf(lo, x);
    }
    // two values with one three-input instruction per extremum
    __device__ __forceinline__ void add(float x, float y)
    {
        asm("max.f32 %0, %0, %1, %2;" : "+f"(hi) : "f"(x), "f"(y));
        asm("min.f32 %0, %0, %1, %2;" : "+f"(lo) : "f"(x), "f"(y));
    }
    __device__ __forceinline__ float top() const { return hi; }
    __device__ __forceinline__ float bottom() const { return lo; }
};
template <> struct Extrema<double> {
    long long hi, lo;
    static __device__ __forceinline__ long long key(double x)
    {
        const long long b = __double_as_longlong(x);
        return b ^ ((b >> 63) & 0x7fffffffffffffffll);
    }
    static __device__ __forceinline__ double value(long long k)
    {
        return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
    }
    __device__ __forceinline__ void set(double x) { hi = lo = key(x); }
    __device__ __forceinline__ void add(double x)
    {
        const long long k = key(x);
        hi = k > hi ? k : hi;
        lo = k < lo ? k : lo;
    }
    __device__ __forceinline__ void add(double x, double y)
    {
        add(x);
        add(y);
    }
    __device__ __forceinline__ double top() const { return value(hi); }
    __device__ __forceinline__ double bottom() const { return value(lo); }
};

// a / b by the approximate reciprocal; b below the normal range counts as 0
// (the callers discard or bound the quotient there)
__device__ __forceinline__ float fdiv_ftz(float a, float b)
{
    float q;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(q) : "f"(a), "f"(b));
    return q;
}

// min(1, n1 / d1, n2 / d2) of non-negative numerators and denominators; a
// quotient 0 / 0 counts as 1.  FP32: fmin ignores the NaN of 0 / 0.  FP64: the
// smaller quotient is found by cross products, so that one division is left.
__device__ __forceinline__ float min_ratio(float n1, float d1, float n2, float d2)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(fdiv_ftz(n1, d1)), "f"(fdiv_ftz(n2, d2)), "f"(1.f));
    return r;
}
__device__ __forceinline__ double min_ratio(double n1, double d1, double n2, double d2)
{
    if (!gt0(d1)) n1 = d1 = 1.0;
    if (!gt0(d2)) n2 = d2 = 1.0;
    const bool first = __double_as_longlong(n1 * d2) < __double_as_longlong(n2 * d1);
    const double n = first ? n1 : n2, d = first ? d1 : d2;
    return __double_as_longlong(n) < __double_as_longlong(d) ? n / d : 1.0;
}

// phi theta of the positivity scaling: theta = f / (f - v) if v < 0 (0 if f <= 0;
// FP32: or below the normal range, where fdiv_ftz would see 0 / 0)
__device__ __forceinline__ float positive_scale(float phi, float f, float v)
{
    const float th = f >= 1.17549435e-38f ? fdiv_ftz(f, __fsub_rn(f, v)) : 0.f;
    return v < 0.f ? phi * th : phi;
}
__device__ __forceinline__ double positive_scale(double phi, double f, double v)
{
    if (!lt0(v)) return phi;
    return gt0(f) ? phi * (f / (f - v)) : 0.0;
}

// entries of cell c
template <typename T>
__device__ __forceinline__ void entry_range(const DevCase<T> &dc, int c, int &e0, int &ne)
{
    if (dc.nf > 0) {
        e0 = c * dc.nf;
        ne = dc.nf;
    } else {
        e0 = __ldg(dc.cf_ptr + c);
        ne = __ldg(dc.cf_ptr + c + 1) - e0;
    }
}

// The entries of cell c and the rows of f they read (TV velocities of the lane,
// fl = f_cur + its first one), from global memory.
template <typename T, int D, int NC, int TV> struct GlobalCell {
    using P = typename Pk<T, TV>::P;
    static constexpr int NP = Pk<T, TV>::NP;
    const DevCase<T> &dc;
    const T *fl;
    int c, e0;
    __device__ __forceinline__ int4 ids(int e) const { return __ldg(dc.gi + e0 + e); }
    __device__ __forceinline__ void values(int e, int at, T (&v)[4]) const
    {
        load_rec_const<4>(dc.gf + (size_t)(e0 + e) * GEnt<D>::LEN + at, v);
    }
    __device__ __forceinline__ void row_of(int cell, P (&x)[NC][NP]) const
    {
#pragma unroll
        for (int m = 0; m < NC; ++m) ldp<T, TV>(fl + ((size_t)cell * NC + m) * dc.nvp, x[m]);
    }
    __device__ __forceinline__ void own(P (&x)[NC][NP]) const { row_of(c, x); }
    __device__ __forceinline__ void row(int, const int4 &gi, P (&x)[NC][NP]) const { row_of(gi.x, x); }
    __device__ __forceinline__ void record(int, int face, T (&x)[XRec<D>::LEN]) const
    {
        load_rec<XRec<D>::LEN>(dc.xrec + (size_t)face * XRec<D>::LEN, x);
    }
};

// asynchronous copies of N bytes (4, 8 or 16) from global into shared memory
template <int N> __device__ __forceinline__ void cp_async(void *smem, const void *global)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s), "l"(global), "n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// B bytes of a lane (4 to 32) in chunks of at most 16
template <int B> __device__ __forceinline__ void cp_async_lane(void *smem, const void *global)
{
    constexpr int CB = B < 16 ? B : 16;
#pragma unroll
    for (int q = 0; q < B / CB; ++q)
        cp_async<CB>(static_cast<char *>(smem) + q * CB, static_cast<const char *>(global) + q * CB);
}

// TV values of a lane from shared memory into packs
template <typename T, int TV>
__device__ __forceinline__ void lds_pack(const unsigned char *p, typename Pk<T, TV>::P (&x)[Pk<T, TV>::NP])
{
    constexpr int CH = vec_chunk<T, TV>();
    using V = typename VecOf<T, CH>::type;
    T v[TV];
#pragma unroll
    for (int q = 0; q < TV / CH; ++q) {
        const V w = reinterpret_cast<const V *>(p)[q];
        const T *t = reinterpret_cast<const T *>(&w);
#pragma unroll
        for (int j = 0; j < CH; ++j) v[q * CH + j] = t[j];
    }
#pragma unroll
    for (int j = 0; j < TV; ++j) pel<Pk<T, TV>::W>(x, j) = v[j];
}

// The same of a cell with NF entries, staged in the warp's shared memory by
// asynchronous copies: its entries, the flux records of its faces and, per lane,
// its TV velocities of the cell's and the neighbours' rows (a lane reads back
// what it copied itself).
template <typename T, int D, int NC, int TV, int NF> struct StagedCell {
    using K = Pk<T, TV>;
    using P = typename K::P;
    using E = GEnt<D>;
    using X = XRec<D>;
    static constexpr int NP = K::NP;
    static constexpr int ROW = 32 * TV * (int)sizeof(T);
    static constexpr int GI = (NF + 1) * NC * ROW, GF = GI + NF * 16, XR = GF + NF * E::LEN * (int)sizeof(T);
    static constexpr int BYTES = XR + NF * X::LEN * (int)sizeof(T);        // a multiple of 16
    static_assert(BYTES % 16 == 0, "stages are 16-byte aligned");
    unsigned char *s;
    int lane;
    // request cell c, whose entry ids lane e < NF holds in id
    __device__ __forceinline__ void request(const DevCase<T> &dc, const T *fl, int c, const int4 &id) const
    {
        constexpr int B = TV * (int)sizeof(T);
#pragma unroll
        for (int e = 0; e <= NF; ++e) {
            const int r = e < NF ? __shfl_sync(0xffffffffu, id.x, e < NF ? e : 0) : c;
#pragma unroll
            for (int m = 0; m < NC; ++m)
                cp_async_lane<B>(s + (e * NC + m) * ROW + lane * B, fl + ((size_t)r * NC + m) * dc.nvp);
        }
        if (lane < NF) *reinterpret_cast<int4 *>(s + GI + lane * 16) = id;
        constexpr int NG = NF * E::LEN * (int)sizeof(T) / 16;
        const char *gf = reinterpret_cast<const char *>(dc.gf + (size_t)c * NF * E::LEN);
#pragma unroll
        for (int q = 0; q < (NG + 31) / 32; ++q)
            if (q * 32 + lane < NG) cp_async<16>(s + GF + (q * 32 + lane) * 16, gf + (q * 32 + lane) * 16);
        constexpr int XV = X::LEN * (int)sizeof(T) / 16, NX = NF * XV;
#pragma unroll
        for (int q = 0; q < (NX + 31) / 32; ++q) {
            const int i = q * 32 + lane, e = i / XV;
            const int face = __shfl_sync(0xffffffffu, id.y, e < NF ? e : 0);
            if (i < NX)
                cp_async<16>(s + XR + i * 16,
                             reinterpret_cast<const char *>(dc.xrec + (size_t)face * X::LEN) + (i - e * XV) * 16);
        }
        cp_async_commit();
    }
    template <int N> __device__ __forceinline__ void read(int at, T (&v)[N]) const
    {
#pragma unroll
        for (int q = 0; q < N * (int)sizeof(T) / 16; ++q) {
            const int4 w = *reinterpret_cast<const int4 *>(s + at + q * 16);
            const T *t = reinterpret_cast<const T *>(&w);
#pragma unroll
            for (int j = 0; j < 16 / (int)sizeof(T); ++j) v[q * (16 / (int)sizeof(T)) + j] = t[j];
        }
    }
    __device__ __forceinline__ int4 ids(int e) const { return *reinterpret_cast<const int4 *>(s + GI + e * 16); }
    __device__ __forceinline__ void values(int e, int at, T (&v)[4]) const
    {
        read<4>(GF + (e * E::LEN + at) * (int)sizeof(T), v);
    }
    __device__ __forceinline__ void row_of(int e, P (&x)[NC][NP]) const
    {
#pragma unroll
        for (int m = 0; m < NC; ++m) lds_pack<T, TV>(s + (e * NC + m) * ROW + lane * TV * (int)sizeof(T), x[m]);
    }
    __device__ __forceinline__ void own(P (&x)[NC][NP]) const { row_of(NF, x); }
    __device__ __forceinline__ void row(int e, const int4 &, P (&x)[NC][NP]) const { row_of(e, x); }
    __device__ __forceinline__ void record(int e, int, T (&x)[X::LEN]) const
    {
        read<X::LEN>(XR + e * X::LEN * (int)sizeof(T), x);
    }
};

// Micro reconstruction of cell c (Sec. 3.1 Step 2) for the TV consecutive
// velocities of this lane: least-squares slope grad = sum_j a_cj (f_j - f_c),
// Venkatakrishnan factor phi = min over the faces of c of (D1^2 + eps^2 +
// 2 D1 D2) / (D1^2 + 2 D2^2 + D1 D2 + eps^2), then a positivity scaling theta
// so that the reconstruction is non-negative at every face centre and at the
// foot of the characteristic after one step: with dmin = min(0, min_f D2_f),
// v = f_c + phi (dmin + min(0, -dt u.grad)); theta = f_c / (f_c - v) if v < 0.
// fi returns f_c, g the scaled slope, ug = u . g.  src gives the cell's entries
// and rows (GlobalCell or the staged ones of the flux pass).  NF > 0: ne == NF
// entries, their rows all requested before the first is used; NF = 0: any
// number.  A wall or padding entry reads the cell itself (no difference, no
// extremum).
template <typename T, int D, int NC, int TV, int NF, typename Src>
__device__ __forceinline__ void cell_slope(const DevCase<T> &dc, const Src &src, const int c, const int ne,
                                           const typename Pk<T, TV>::P (&u)[Pk<T, TV>::NP][D],
                                           typename Pk<T, TV>::P (&fi)[NC][Pk<T, TV>::NP],
                                           typename Pk<T, TV>::P (&g)[NC][Pk<T, TV>::NP][D],
                                           typename Pk<T, TV>::P (&ug)[NC][Pk<T, TV>::NP])
{
    using E = GEnt<D>;
    using K = Pk<T, TV>;
    using P = typename K::P;
    constexpr int W = K::W, NP = K::NP;
    P nfi[NC][NP];
    Extrema<T> ex[NC][TV];
    src.own(fi);
#pragma unroll
    for (int m = 0; m < NC; ++m) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            nfi[m][i] = pneg(fi[m][i]);
#pragma unroll
            for (int d = 0; d < D; ++d) g[m][i][d] = pbc<P>(T(0));
        }
#pragma unroll
        for (int j = 0; j < TV; ++j) ex[m][j].set(pel<W>(fi[m], j));
    }
    // f of the cell across an entry
    auto across = [&](const int e, P (&fj)[NC][NP]) {
        const int4 gi = src.ids(e);
        src.row(e, gi, fj);
        if ((gi.z & 255) == FT_FARFIELD) {
            T gr[GREC];
            load_rec<GREC>(dc.grec + (size_t)gi.w * GREC, gr);
#pragma unroll
            for (int j = 0; j < TV; ++j) {
                T uj[3] = {T(0), T(0), T(0)};
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    P t[NP];
#pragma unroll
                    for (int i = 0; i < NP; ++i) t[i] = u[i][d];
                    uj[d] = pel<W>(t, j);
                }
                const T H = maxwell_h<T, D>(gr, uj);
                pel<W>(fj[0], j) = H;
                if (NC == 2) pel<W>(fj[NC - 1], j) = gr[GR_NB] * H;
            }
        }
    };
    auto slope_term = [&](const int e, P (&fj)[NC][NP]) {
        T a[4];
        src.values(e, (E::A / 4) * 4, a);
#pragma unroll
        for (int m = 0; m < NC; ++m)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const P df = padd(fj[m][i], nfi[m][i]);
#pragma unroll
                for (int d = 0; d < D; ++d) g[m][i][d] = pfma(pbc<P>(a[E::A % 4 + d]), df, g[m][i][d]);
            }
    };
    auto extrema = [&](P (&x)[NC][NP], P (&y)[NC][NP], bool both, auto &q) {
#pragma unroll
        for (int m = 0; m < NC; ++m)
#pragma unroll
            for (int j = 0; j < TV; ++j) {
                if (both) q[m][j].add(pel<W>(x[m], j), pel<W>(y[m], j));
                else q[m][j].add(pel<W>(x[m], j));
            }
    };
    if constexpr (NF > 0) {
        P fj[NF][NC][NP];
#pragma unroll
        for (int e = 0; e < NF; ++e) across(e, fj[e]);
#pragma unroll
        for (int e = 0; e < NF; ++e) slope_term(e, fj[e]);
#pragma unroll
        for (int e = 0; e < NF; e += 2) extrema(fj[e], fj[e + 1 < NF ? e + 1 : e], e + 1 < NF, ex);
    } else {
        for (int e = 0; e < ne; ++e) {
            P fj[NC][NP];
            across(e, fj);
            slope_term(e, fj);
            extrema(fj, fj, false, ex);
        }
    }
    // Venkatakrishnan's factor at a face, phi(d2) = (a2 + 2 d1 d2) / (a2 + d2 (2 d2 + d1))
    // with a2 = d1^2 + eps^2 and d1 of the sign of d2, is at least 1 for
    // 0 <= d2/d1 <= 1/2 and strictly decreasing in |d2| beyond.  Its minimum over
    // the faces (clipped at 1) is therefore taken at the largest and at the most
    // negative d2, so the face loop only tracks those two, and phi is evaluated
    // twice per velocity instead of once per face.
    Extrema<T> d2x[NC][TV];
#pragma unroll
    for (int m = 0; m < NC; ++m)
#pragma unroll
        for (int j = 0; j < TV; ++j) d2x[m][j].set(T(0));
    auto offset = [&](const int e, P (&d2)[NC][NP]) {
        T r[4];
        src.values(e, (E::RS / 4) * 4, r);
#pragma unroll
        for (int m = 0; m < NC; ++m)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                P s = pmul(g[m][i][0], pbc<P>(r[E::RS % 4]));
#pragma unroll
                for (int d = 1; d < D; ++d) s = pfma(g[m][i][d], pbc<P>(r[E::RS % 4 + d]), s);
                d2[m][i] = s;
            }
    };
    if constexpr (NF > 0) {
#pragma unroll
        for (int e = 0; e < NF; e += 2) {
            P x[NC][NP], y[NC][NP];
            offset(e, x);
            if (e + 1 < NF) offset(e + 1, y);
            extrema(x, y, e + 1 < NF, d2x);
        }
    } else {
        for (int e = 0; e < ne; ++e) {
            P x[NC][NP];
            offset(e, x);
            extrema(x, x, false, d2x);
        }
    }
    const P e2 = pbc<P>(__ldg(dc.eps2 + c)), ndt = pbc<P>(-dc.dtT);
#pragma unroll
    for (int m = 0; m < NC; ++m)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            P phi = pbc<P>(T(1)), dn, dp, low;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                pel<W>(&dp, w) = d2x[m][i * W + w].top();
                pel<W>(&dn, w) = d2x[m][i * W + w].bottom();
            }
            if (dc.limiter) {
                P hi, lo, num[2], den[2];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    pel<W>(&hi, w) = ex[m][i * W + w].top();
                    pel<W>(&lo, w) = ex[m][i * W + w].bottom();
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const P d1 = padd(s ? lo : hi, nfi[m][i]), d2 = s ? dn : dp;
                    const P a2 = pfma(d1, d1, e2);
                    num[s] = pfma(padd(d1, d1), d2, a2);
                    den[s] = pfma(d2, pfma(pbc<P>(T(2)), d2, d1), a2);
                }
#pragma unroll
                for (int w = 0; w < W; ++w)
                    pel<W>(&phi, w) =
                        min_ratio(pel<W>(num, w), pel<W>(den, w), pel<W>(num + 1, w), pel<W>(den + 1, w));
            }
            P s = pmul(u[i][0], g[m][i][0]);
#pragma unroll
            for (int d = 1; d < D; ++d) s = pfma(u[i][d], g[m][i][d], s);
            const P foot = pmul(s, ndt);
#pragma unroll
            for (int w = 0; w < W; ++w) pel<W>(&low, w) = min0(pel<W>(const_cast<P *>(&foot), w));
            low = padd(dn, low);
            P v = pfma(phi, low, fi[m][i]);
#pragma unroll
            for (int w = 0; w < W; ++w)
                pel<W>(&phi, w) = positive_scale(pel<W>(&phi, w), pel<W>(&fi[m][i], w), pel<W>(&v, w));
#pragma unroll
            for (int d = 0; d < D; ++d) g[m][i][d] = pmul(g[m][i][d], phi);
            if constexpr (std::is_same<T, double>::value) {
                ug[m][i] = pmul(s, phi);               // FP64 operations are what the FP64 form spends
            } else {
                s = pmul(u[i][0], g[m][i][0]);
#pragma unroll
                for (int d = 1; d < D; ++d) s = pfma(u[i][d], g[m][i][d], s);
                ug[m][i] = s;
            }
        }
}

// P_m(c) of the flux record (see XRec); in FP64 grouped by the components of c
// (12 operations in 3D instead of 17)
template <typename T, int D, typename P>
__device__ __forceinline__ P poly_eval(const T *__restrict__ a, const P (&c)[D], const P c2)
{
    constexpr int NB = Poly<D>::NB;
    P p = pbc<P>(a[0]);
    if constexpr (std::is_same<T, double>::value) {
#pragma unroll
        for (int e = 0; e < D; ++e) {
            P r = pfma(a[1 + D + NB + e], c2, a[1 + e]);
#pragma unroll
            for (int f = e; f < D; ++f) r = pfma(a[1 + D + (e * (2 * D - e + 1)) / 2 + (f - e)], c[f], r);
            p = pfma(r, c[e], p);
        }
        return p;
    } else {
        P q, g;
#pragma unroll
        for (int e = 0; e < D; ++e) {
            p = pfma(pbc<P>(a[1 + e]), c[e], p);
            P r = pmul(pbc<P>(a[1 + D + (e * (2 * D - e + 1)) / 2]), c[e]);
#pragma unroll
            for (int f = e + 1; f < D; ++f)
                r = pfma(pbc<P>(a[1 + D + (e * (2 * D - e + 1)) / 2 + (f - e)]), c[f], r);
            q = e == 0 ? pmul(r, c[0]) : pfma(r, c[e], q);
            g = e == 0 ? pmul(pbc<P>(a[1 + D + NB]), c[0]) : pfma(pbc<P>(a[1 + D + NB + e]), c[e], g);
        }
        return pfma(g, c2, padd(p, q));
    }
}

}  // namespace ugks
