// ugks_host.cu -- C ABI of the UGKS library: validation, host preprocessing
// (cell ordering, least-squares coefficients, face entries), device state and
// the launch sequence of a time step.  The numerics live in ugks_kernels.cu.
#include "../../include/ugks.h"
#include "ugks_device.cuh"
#include "ugks_kernels.h"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <numeric>
#include <stdexcept>
#include <string>
#include <vector>

namespace {

thread_local std::string g_err;

struct Fail {
    ugks_status code;
    std::string msg;
};

[[noreturn]] void fail(ugks_status code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    throw Fail{code, buf};
}

void cuda_ok(cudaError_t e, const char *what)
{
    if (e != cudaSuccess) fail(UGKS_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

}  // namespace

struct ugks_case {
    int D = 0, NC = 0, prec = UGKS_FP64;
    int64_t C = 0, F = 0, Nv = 0, nvp = 0;
    int G = 0, NW = 0;
    double dt = 0.0;
    int64_t step = 0;
    cudaStream_t stream = nullptr;
    ugks_alloc alloc{};
    bool user_alloc = false;
    std::vector<std::pair<void *, size_t>> blocks;
    size_t device_bytes = 0, f_bytes = 0;
    size_t stage_bytes = 0;        // bytes of the flux buffer, the staging area of state I/O between steps
    ugks::DevCase<double> d64{};
    ugks::DevCase<float> d32{};
    int P = 0, vtile = 0, nth = 256, n_patches = 0, vt_group = 1;
    int nf = 0, gvel = 0, n_groups = 1, chunk = 0, n_chunks = 1, parts = 1;
    long long *perm_d = nullptr;   // caller cell i -> internal cell
    std::vector<long long> perm_h; // the same on the host
    std::vector<long long> wall_face_h;   // face id of every wall slot
    std::vector<double> wall_n_h;         // [NW][D] its normal
    double *res_d = nullptr;       // [M]
    int *flags_d = nullptr;
    unsigned long long *range_d = nullptr;   // [2] bit patterns of the min and max density
    int n_res_parts = 0;
    bool stepped = false;
    // kernel-group profiling
    std::vector<cudaEvent_t> prof_ev;
    int prof_max = 0, prof_used = 0;
    // host -> device copies of ugks_set_state (created on first use): the copy
    // stream and its events (ready, copied[2], consumed[2])
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t io_ev[5] = {};
    // domain decomposition: owned-cell mask (internal order) and the halo
    // lists registered by ugks_halo_set (internal cell ids on the device)
    unsigned char *owned_d = nullptr;
    struct HaloList {
        int *ids = nullptr;
        int n = 0;
    };
    std::vector<HaloList> halo;

    void *dalloc(size_t bytes)
    {
        if (bytes == 0) bytes = 16;
        bytes = (bytes + 255) & ~size_t(255);
        void *p = nullptr;
        if (user_alloc) {
            p = alloc.alloc(alloc.ctx, bytes, (void *)stream);
            if (!p) fail(UGKS_ENOMEM, "device allocation of %zu bytes failed", bytes);
            if ((uintptr_t)p & 255) {       // the vector loads and stores rely on it
                alloc.free(alloc.ctx, p, bytes, (void *)stream);
                fail(UGKS_EINVAL, "the allocator returned a pointer that is not 256-byte aligned");
            }
        } else {
            cudaError_t e = cudaMalloc(&p, bytes);
            if (e != cudaSuccess) {
                cudaGetLastError();
                fail(UGKS_ENOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
            }
        }
        blocks.push_back({p, bytes});
        device_bytes += bytes;
        return p;
    }

    // frees one block of dalloc (a halo list that is replaced)
    void dfree(const void *p)
    {
        if (!p) return;
        for (size_t i = 0; i < blocks.size(); ++i)
            if (blocks[i].first == p) {
                if (user_alloc) alloc.free(alloc.ctx, blocks[i].first, blocks[i].second, (void *)stream);
                else cudaFree(blocks[i].first);
                device_bytes -= blocks[i].second;
                blocks.erase(blocks.begin() + (long)i);
                return;
            }
    }

    template <typename V>
    V *upload(const std::vector<V> &h)
    {
        V *d = (V *)dalloc(h.size() * sizeof(V));
        if (!h.empty()) cuda_ok(cudaMemcpyAsync(d, h.data(), h.size() * sizeof(V), cudaMemcpyHostToDevice, stream),
                                "upload");
        return d;
    }

    void release()
    {
        if (stream) cudaStreamSynchronize(stream);
        else cudaDeviceSynchronize();
        if (copy_stream) {
            cudaStreamSynchronize(copy_stream);
            for (auto &e : io_ev) {
                if (e) cudaEventDestroy(e);
                e = nullptr;
            }
            cudaStreamDestroy(copy_stream);
            copy_stream = nullptr;
        }
        for (auto &b : blocks) {
            if (user_alloc) alloc.free(alloc.ctx, b.first, b.second, (void *)stream);
            else cudaFree(b.first);
        }
        blocks.clear();
    }
};

namespace {

// 2D / 3D Morton key of quantised centroids
uint64_t spread2(uint64_t x)
{
    x &= 0xffffffffULL;
    x = (x | (x << 16)) & 0x0000ffff0000ffffULL;
    x = (x | (x << 8)) & 0x00ff00ff00ff00ffULL;
    x = (x | (x << 4)) & 0x0f0f0f0f0f0f0f0fULL;
    x = (x | (x << 2)) & 0x3333333333333333ULL;
    x = (x | (x << 1)) & 0x5555555555555555ULL;
    return x;
}

uint64_t spread3(uint64_t x)
{
    x &= 0x1fffffULL;
    x = (x | (x << 32)) & 0x1f00000000ffffULL;
    x = (x | (x << 16)) & 0x1f0000ff0000ffULL;
    x = (x | (x << 8)) & 0x100f00f00f00f00fULL;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ULL;
    x = (x | (x << 2)) & 0x1249249249249249ULL;
    return x;
}

struct Host {
    // internal-order geometry produced by preprocessing
    std::vector<int> perm_i2u, perm_u2i;
    std::vector<int> cf_ptr, cf_face;
    std::vector<signed char> cf_side;
    std::vector<double> cf_r;
    std::vector<double> gf;          // entry values, GEnt<D>::LEN each
    std::vector<int> gi;             // entry ids, 4 each
    int nf = 0;                      // entries per cell (0: the cells' own counts)
    std::vector<int> nb_ptr, nb_id;
    std::vector<double> nb_a, eps2, vol;
    std::vector<int> fL, fR, faux, ftag, gface, wface;
    std::vector<signed char> ftype;
    std::vector<double> fn, frL, frR;
};

// CFL time step of Algorithm 1 over the first n cells of the mesh:
// dt = cfl * min_i (2 |Omega_i| / sum_f S_f) / max_k |u_k|.  Each cell's face
// areas are summed in ascending face order, so a cell gives the same value in
// any mesh that holds all of its faces in the same relative order (a
// subdomain's own cells).
double cfl_dt_of(const ugks_mesh *m, const ugks_vgrid *v, double cfl, int64_t n)
{
    const int D = m->dim;
    std::vector<double> sumS((size_t)m->n_cells, 0.0);
    for (int64_t f = 0; f < m->n_faces; ++f) {
        sumS[(size_t)m->face_cells[2 * f]] += m->face_S[f];
        const int64_t b = m->face_cells[2 * f + 1];
        if (b >= 0) sumS[(size_t)b] += m->face_S[f];
    }
    double hmin = INFINITY;
    for (int64_t i = 0; i < n; ++i) hmin = std::min(hmin, 2.0 * m->cell_vol[i] / sumS[(size_t)i]);
    double umax = 0.0;
    for (int64_t k = 0; k < v->nv; ++k) {
        double s = 0.0;
        for (int d = 0; d < D; ++d) s += v->u[k * D + d] * v->u[k * D + d];
        umax = std::max(umax, std::sqrt(s));
    }
    return cfl * hmin / umax;
}

void validate(const ugks_mesh *m, const ugks_vgrid *v, const ugks_params *p)
{
    if (!m || !v || !p) fail(UGKS_EINVAL, "mesh, vgrid and params must not be NULL");
    if (m->dim != 2 && m->dim != 3) fail(UGKS_EINVAL, "mesh dim must be 2 or 3 (got %d)", m->dim);
    if (v->dim != m->dim) fail(UGKS_EINVAL, "velocity grid dim %d != mesh dim %d", v->dim, m->dim);
    if (m->n_cells <= 0 || m->n_faces < 0) fail(UGKS_EINVAL, "mesh needs n_cells > 0, n_faces >= 0");
    if (m->n_cells > (1LL << 30) || m->n_faces > (1LL << 30)) fail(UGKS_EINVAL, "mesh too large for 32-bit indexing");
    if (v->nv <= 0 || v->nv > (1 << 24)) fail(UGKS_EINVAL, "velocity count %lld out of range", (long long)v->nv);
    if (!m->cell_xc || !m->cell_vol || !m->face_cells || !m->face_n || !m->face_S || !m->face_xc ||
        !m->face_type || !m->face_tag)
        fail(UGKS_EINVAL, "mesh arrays must not be NULL");
    if (!v->u || !v->w) fail(UGKS_EINVAL, "velocity arrays must not be NULL");
    if (p->precision != UGKS_FP64 && p->precision != UGKS_FP32) fail(UGKS_EINVAL, "unknown precision %d", p->precision);
    if (!(p->Pr > 0.0) || !(p->omega >= 0.0) || !(p->L_ref > 0.0) || !(p->Kn > 0.0))
        fail(UGKS_EINVAL, "need Kn > 0, L_ref > 0, Pr > 0, omega >= 0");
    if (!(p->dt > 0.0) && !(p->cfl > 0.0)) fail(UGKS_EINVAL, "need cfl > 0 or dt > 0");
    if (p->limiter && !(p->venkat_K > 0.0)) fail(UGKS_EINVAL, "venkat_K must be > 0 with the limiter on");
    if (p->n_walls < 0 || (p->n_walls > 0 && (!p->wall_T || !p->wall_U))) fail(UGKS_EINVAL, "wall arrays missing");
    for (int i = 0; i < p->n_walls; ++i)
        if (!(p->wall_T[i] > 0.0)) fail(UGKS_EINVAL, "wall %d temperature must be > 0", i);
    const int D = m->dim;
    for (int64_t i = 0; i < m->n_cells; ++i)
        if (!(m->cell_vol[i] > 0.0)) fail(UGKS_EINVAL, "cell %lld has non-positive volume", (long long)i);
    bool farfield = false;
    for (int64_t f = 0; f < m->n_faces; ++f) {
        const int64_t a = m->face_cells[2 * f], b = m->face_cells[2 * f + 1];
        const int t = m->face_type[f];
        if (a < 0 || a >= m->n_cells) fail(UGKS_EINVAL, "face %lld: owner out of range", (long long)f);
        if (t == UGKS_FACE_INTERIOR || t == UGKS_FACE_PERIODIC) {
            if (b < 0 || b >= m->n_cells) fail(UGKS_EINVAL, "face %lld: neighbour out of range", (long long)f);
            if (t == UGKS_FACE_PERIODIC && !m->face_shift) fail(UGKS_EINVAL, "periodic faces need face_shift");
        } else if (t == UGKS_FACE_WALL || t == UGKS_FACE_FARFIELD) {
            if (b != -1) fail(UGKS_EINVAL, "face %lld: boundary face must have neighbour -1", (long long)f);
            if (t == UGKS_FACE_WALL && (m->face_tag[f] < 0 || m->face_tag[f] >= p->n_walls))
                fail(UGKS_EINVAL, "face %lld: wall tag %d out of range", (long long)f, m->face_tag[f]);
            if (t == UGKS_FACE_FARFIELD) farfield = true;
        } else {
            fail(UGKS_EINVAL, "face %lld: unknown type %d", (long long)f, t);
        }
        if (!(m->face_S[f] > 0.0)) fail(UGKS_EINVAL, "face %lld: area must be > 0", (long long)f);
        double nn = 0.0;
        for (int d = 0; d < D; ++d) nn += m->face_n[f * D + d] * m->face_n[f * D + d];
        if (std::fabs(nn - 1.0) > 1e-8) fail(UGKS_EINVAL, "face %lld: normal is not unit length", (long long)f);
    }
    if (farfield && (!(p->inf_rho > 0.0) || !(p->inf_T > 0.0)))
        fail(UGKS_EINVAL, "far-field faces need inf_rho > 0 and inf_T > 0");
    for (int64_t k = 0; k < v->nv; ++k)
        if (!(v->w[k] >= 0.0) || !std::isfinite(v->w[k])) fail(UGKS_EINVAL, "velocity weight %lld invalid", (long long)k);
    if (p->prim_init)
        for (int64_t i = 0; i < m->n_cells; ++i)
            if (!(p->prim_init[i * (D + 2)] > 0.0) || !(p->prim_init[i * (D + 2) + D + 1] > 0.0))
                fail(UGKS_EINVAL, "initial state of cell %lld needs rho > 0 and T > 0", (long long)i);
    if (p->vtile != 0 && p->vtile != 32 && p->vtile != 64 && p->vtile != 128)
        fail(UGKS_EINVAL, "vtile must be 0, 32, 64 or 128");
    if (p->patch_cells < 0 || p->patch_cells > 4096) fail(UGKS_EINVAL, "patch_cells out of range");
    if (p->w0_analytic != 0 && p->w0_analytic != 1) fail(UGKS_EINVAL, "w0_analytic must be 0 or 1");
    if (p->gather_threads != 0 && p->gather_threads != 256 && p->gather_threads != 512)
        fail(UGKS_EINVAL, "gather_threads must be 0, 256 or 512");
    if (p->gather_threads == 512 && (p->precision != UGKS_FP32 || p->vtile > 64))
        fail(UGKS_EINVAL, "gather_threads = 512 needs UGKS_FP32 and vtile <= 64");
    if (p->gather_tile_group < 0 || p->gather_tile_group > 1024)
        fail(UGKS_EINVAL, "gather_tile_group must be in [0, 1024]");
}

// invert the DxD normal matrix by its adjugate
bool invert_small(int D, const double *A, double *Ainv)
{
    double tr = 0.0;
    for (int a = 0; a < D; ++a) tr += A[a * D + a];
    double det;
    if (D == 2) {
        det = A[0] * A[3] - A[1] * A[2];
        if (!(std::fabs(det) > 1e-12 * std::pow(tr / D, D))) return false;
        Ainv[0] = A[3] / det;
        Ainv[1] = -A[1] / det;
        Ainv[2] = -A[2] / det;
        Ainv[3] = A[0] / det;
        return true;
    }
    const double c00 = A[4] * A[8] - A[5] * A[7], c01 = A[5] * A[6] - A[3] * A[8], c02 = A[3] * A[7] - A[4] * A[6];
    det = A[0] * c00 + A[1] * c01 + A[2] * c02;
    if (!(std::fabs(det) > 1e-12 * std::pow(tr / D, D))) return false;
    Ainv[0] = c00 / det;
    Ainv[3] = c01 / det;
    Ainv[6] = c02 / det;
    Ainv[1] = (A[2] * A[7] - A[1] * A[8]) / det;
    Ainv[4] = (A[0] * A[8] - A[2] * A[6]) / det;
    Ainv[7] = (A[1] * A[6] - A[0] * A[7]) / det;
    Ainv[2] = (A[1] * A[5] - A[2] * A[4]) / det;
    Ainv[5] = (A[2] * A[3] - A[0] * A[5]) / det;
    Ainv[8] = (A[0] * A[4] - A[1] * A[3]) / det;
    return true;
}

void preprocess(const ugks_mesh *m, const ugks_params *p, Host &h)
{
    const int D = m->dim;
    const int C = (int)m->n_cells, F = (int)m->n_faces;
    // ---- cell order: Morton order of the centroids (spatially compact patches)
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int i = 0; i < C; ++i)
        for (int d = 0; d < D; ++d) {
            lo[d] = std::min(lo[d], m->cell_xc[(size_t)i * D + d]);
            hi[d] = std::max(hi[d], m->cell_xc[(size_t)i * D + d]);
        }
    std::vector<uint64_t> key(C);
    const double bits = D == 2 ? 4294967295.0 : 2097151.0;
    for (int i = 0; i < C; ++i) {
        uint64_t k = 0;
        for (int d = 0; d < D; ++d) {
            double span = hi[d] - lo[d];
            double t = span > 0 ? (m->cell_xc[(size_t)i * D + d] - lo[d]) / span : 0.0;
            uint64_t qv = (uint64_t)std::llround(t * bits);
            k |= (D == 2 ? spread2(qv) : spread3(qv)) << d;
        }
        key[i] = k;
    }
    h.perm_i2u.resize(C);
    std::iota(h.perm_i2u.begin(), h.perm_i2u.end(), 0);
    std::stable_sort(h.perm_i2u.begin(), h.perm_i2u.end(), [&](int a, int b) { return key[a] < key[b]; });
    h.perm_u2i.resize(C);
    for (int i = 0; i < C; ++i) h.perm_u2i[h.perm_i2u[i]] = i;
    auto X = [&](int ci, int d) { return m->cell_xc[(size_t)h.perm_i2u[ci] * D + d]; };
    h.vol.resize(C);
    for (int i = 0; i < C; ++i) h.vol[i] = m->cell_vol[h.perm_i2u[i]];

    // ---- faces
    h.fL.assign(F, -1);
    h.fR.assign(F, -1);
    h.faux.assign(F, -1);
    h.ftag.assign(F, 0);
    h.ftype.assign(F, 0);
    h.fn.assign((size_t)F * D, 0.0);
    h.frL.assign((size_t)F * D, 0.0);
    h.frR.assign((size_t)F * D, 0.0);
    for (int f = 0; f < F; ++f) {
        const int t = m->face_type[f];
        h.ftype[f] = (signed char)t;
        h.ftag[f] = m->face_tag[f];
        h.fL[f] = h.perm_u2i[m->face_cells[2 * f]];
        if (t == UGKS_FACE_INTERIOR || t == UGKS_FACE_PERIODIC) h.fR[f] = h.perm_u2i[m->face_cells[2 * f + 1]];
        for (int d = 0; d < D; ++d) {
            h.fn[(size_t)f * D + d] = m->face_n[(size_t)f * D + d];
            const double xf = m->face_xc[(size_t)f * D + d];
            h.frL[(size_t)f * D + d] = xf - X(h.fL[f], d);
            if (h.fR[f] >= 0) {
                const double sh = (t == UGKS_FACE_PERIODIC) ? m->face_shift[(size_t)f * D + d] : 0.0;
                h.frR[(size_t)f * D + d] = xf - sh - X(h.fR[f], d);
            }
        }
        if (t == UGKS_FACE_FARFIELD) {
            h.faux[f] = (int)h.gface.size();
            h.gface.push_back(f);
        } else if (t == UGKS_FACE_WALL) {
            h.faux[f] = (int)h.wface.size();
            h.wface.push_back(f);
        }
    }

    // ---- faces of each cell (CSR, face order within a cell)
    h.cf_ptr.assign(C + 1, 0);
    for (int f = 0; f < F; ++f) {
        h.cf_ptr[h.fL[f] + 1]++;
        if (h.fR[f] >= 0) h.cf_ptr[h.fR[f] + 1]++;
    }
    for (int i = 0; i < C; ++i) h.cf_ptr[i + 1] += h.cf_ptr[i];
    const int ncf = h.cf_ptr[C];
    h.cf_face.resize(ncf);
    h.cf_side.resize(ncf);
    h.cf_r.resize((size_t)ncf * D);
    std::vector<int> fill(C, 0);
    for (int f = 0; f < F; ++f)
        for (int s = 0; s < 2; ++s) {
            const int c = s == 0 ? h.fL[f] : h.fR[f];
            if (c < 0) continue;
            const int e = h.cf_ptr[c] + fill[c]++;
            h.cf_face[e] = f;
            h.cf_side[e] = (signed char)s;
            for (int d = 0; d < D; ++d) h.cf_r[(size_t)e * D + d] = s == 0 ? h.frL[(size_t)f * D + d] : h.frR[(size_t)f * D + d];
        }

    // ---- least squares: neighbours across non-wall faces, far-field ghosts
    //      mirrored across the face; weights 1/|d|^2; a = w M^{-1} d
    h.nb_ptr.assign(C + 1, 0);
    h.eps2.resize(C);
    std::vector<double> dvec;
    for (int c = 0; c < C; ++c) {
        double sumS = 0.0;
        const int n0 = (int)h.nb_id.size();
        for (int e = h.cf_ptr[c]; e < h.cf_ptr[c + 1]; ++e) {
            const int f = h.cf_face[e];
            sumS += m->face_S[f];
            const int t = h.ftype[f];
            if (t == UGKS_FACE_WALL) continue;
            double d[3];
            if (t == UGKS_FACE_FARFIELD) {
                double rn = 0.0;
                for (int k = 0; k < D; ++k) rn += h.frL[(size_t)f * D + k] * h.fn[(size_t)f * D + k];
                for (int k = 0; k < D; ++k) d[k] = 2.0 * rn * h.fn[(size_t)f * D + k];
                h.nb_id.push_back(-(h.faux[f] + 1));
            } else {
                // vector from this cell to the other one through the face
                const bool own = h.cf_side[e] == 0;
                const int o = own ? h.fR[f] : h.fL[f];
                for (int k = 0; k < D; ++k) {
                    const double ro = own ? h.frR[(size_t)f * D + k] : h.frL[(size_t)f * D + k];
                    d[k] = h.cf_r[(size_t)e * D + k] - ro;
                }
                h.nb_id.push_back(o);
            }
            for (int k = 0; k < D; ++k) dvec.push_back(d[k]);
        }
        const int n1 = (int)h.nb_id.size();
        h.nb_ptr[c + 1] = n1;
        double A[9] = {0}, Ai[9];
        for (int q = n0; q < n1; ++q) {
            const double *d = &dvec[(size_t)q * D];
            double dd = 0.0;
            for (int k = 0; k < D; ++k) dd += d[k] * d[k];
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) A[a * D + b] += d[a] * d[b] / dd;
        }
        const bool ok = n1 > n0 && invert_small(D, A, Ai);
        for (int q = n0; q < n1; ++q) {
            const double *d = &dvec[(size_t)q * D];
            double dd = 0.0;
            for (int k = 0; k < D; ++k) dd += d[k] * d[k];
            for (int a = 0; a < D; ++a) {
                double s = 0.0;
                if (ok)
                    for (int b = 0; b < D; ++b) s += Ai[a * D + b] * d[b];
                h.nb_a.push_back(s / dd);
            }
        }
        // limiter scale h_c = 2 D |Omega_c| / sum S (the time-step scale is cfl_dt_of's)
        const double hc = 2.0 * D * h.vol[c] / sumS;
        const double Kh = p->venkat_K * hc;
        h.eps2[c] = Kh * Kh * Kh;
    }

    // ---- entries of every (cell, face) (GEnt, DevCase::gi), padded to the same
    //      count in every cell where that is at most MAX_NF
    int most = 0;
    for (int c = 0; c < C; ++c) most = std::max(most, h.cf_ptr[c + 1] - h.cf_ptr[c]);
    // counts with kernels of their own: 3 and 4 in 2D, 4 and 6 in 3D
    h.nf = most == 0 || most > ugks::MAX_NF ? 0 : D == 2 ? (most <= 3 ? 3 : most <= 4 ? 4 : 0) : (most <= 4 ? 4 : 6);
    const int GL = D == 2 ? ugks::GEnt<2>::LEN : ugks::GEnt<3>::LEN;
    const int oA = D == 2 ? ugks::GEnt<2>::A : ugks::GEnt<3>::A;
    const int oRS = D == 2 ? ugks::GEnt<2>::RS : ugks::GEnt<3>::RS;
    const int oN = D == 2 ? ugks::GEnt<2>::N : ugks::GEnt<3>::N;
    const int oCS = D == 2 ? ugks::GEnt<2>::CS : ugks::GEnt<3>::CS;
    const size_t n_ent = h.nf > 0 ? (size_t)C * h.nf : (size_t)ncf;
    h.gf.assign(n_ent * GL, 0.0);
    h.gi.assign(n_ent * 4, 0);
    for (int c = 0; c < C; ++c) {
        int q = h.nb_ptr[c];
        size_t at = h.nf > 0 ? (size_t)c * h.nf : (size_t)h.cf_ptr[c];
        const size_t end = h.nf > 0 ? at + h.nf : (size_t)h.cf_ptr[c + 1];
        for (int e = h.cf_ptr[c]; e < h.cf_ptr[c + 1]; ++e, ++at) {
            const int f = h.cf_face[e], t = h.ftype[f];
            const bool own = h.cf_side[e] == 0, inner = t == UGKS_FACE_INTERIOR || t == UGKS_FACE_PERIODIC;
            double *g = &h.gf[at * GL];
            int *gi = &h.gi[at * 4];
            gi[0] = inner ? (own ? h.fR[f] : h.fL[f]) : c;
            gi[1] = f;
            gi[2] = t + (own ? 256 : 0);
            gi[3] = inner ? 0 : h.faux[f];
            if (t != UGKS_FACE_WALL) {
                for (int d = 0; d < D; ++d) g[oA + d] = h.nb_a[(size_t)q * D + d];
                ++q;
            }
            for (int d = 0; d < D; ++d) {
                g[oRS + d] = h.cf_r[(size_t)e * D + d];
                g[oN + d] = h.fn[(size_t)f * D + d];
            }
            g[oCS] = (own ? -1.0 : 1.0) * m->face_S[f] / h.vol[c];
        }
        for (; at < end; ++at) {
            h.gi[at * 4] = c;
            h.gi[at * 4 + 2] = ugks::FT_NONE;
        }
    }
}

template <typename T>
std::vector<T> cast(const std::vector<double> &v)
{
    return std::vector<T>(v.begin(), v.end());
}

// lane sums of stage 1 between the chunks of a group (DevCase::carry): per cell,
// moment and lane 16 bytes (two pairs) in the FP32 form, 8 in the FP64 form
size_t carry_bytes(const ugks_case *c)
{
    return (size_t)c->C * (c->D + 2) * 32 * (c->prec == UGKS_FP64 ? 8 : 16);
}

template <typename T>
void fill_case(ugks_case *c, ugks::DevCase<T> &dc, const ugks_mesh *m, const ugks_vgrid *v, const ugks_params *p,
               const Host &h)
{
    const int D = c->D, M = D + 2;
    dc.D = D;
    dc.NC = c->NC;
    dc.C = (int)c->C;
    dc.F = (int)c->F;
    dc.G = c->G;
    dc.NW = c->NW;
    dc.nv = (int)c->Nv;
    dc.nvp = (int)c->nvp;
    dc.dt = c->dt;
    dc.Pr = p->Pr;
    dc.omega = p->omega;
    dc.nxi = 3.0 - D;
    // VHS viscosity at the reference state (Bird's mean free path)
    const double mu_ref = 15.0 * std::sqrt(2.0 * M_PI) * p->Kn * p->L_ref /
                          (2.0 * (5.0 - 2.0 * p->omega) * (7.0 - 2.0 * p->omega));
    dc.dt_mu = std::isinf(p->Kn) ? 0.0 : c->dt / mu_ref;
    dc.limiter = p->limiter ? 1 : 0;
    dc.w0_analytic = p->w0_analytic ? 1 : 0;
    // velocities, padded with u = 0, w = 0
    for (int d = 0; d < 3; ++d) {
        dc.u[d] = nullptr;
    }
    for (int d = 0; d < D; ++d) {
        std::vector<double> ud(c->nvp, 0.0);
        for (int64_t k = 0; k < c->Nv; ++k) ud[k] = v->u[k * D + d];
        dc.u[d] = c->upload(cast<T>(ud));
    }
    // tensor-product grid: u_k = (x_i, y_j[, z_l]), k = i + nx (j + ny l), and
    // w_k = wx_i wy_j [wz_l]; verified exactly for the axes and to 1e-14 for the
    // weights, else the general per-velocity face sums are used
    dc.sep = 0;
    dc.sep1 = 0;
    for (int d = 0; d < 3; ++d) {
        dc.cart_n[d] = 0;
        dc.axis[d] = dc.axw[d] = nullptr;
    }
    {
        int64_t prod = 1;
        bool ok = true;
        for (int d = 0; d < D; ++d) {
            ok = ok && v->cart_n[d] > 1;
            prod *= std::max(v->cart_n[d], 1);
        }
        ok = ok && prod == c->Nv;
        if (ok) {
            const int nx = v->cart_n[0], ny = v->cart_n[1], nz = D == 3 ? v->cart_n[2] : 1;
            std::vector<std::vector<double>> ax(D), aw(D);
            auto kidx = [&](int i, int j, int l) { return (int64_t)i + (int64_t)nx * (j + (int64_t)ny * l); };
            const int nn[3] = {nx, ny, nz};
            for (int d = 0; d < D; ++d) {
                for (int i = 0; i < nn[d]; ++i) {
                    int ijk[3] = {0, 0, 0};
                    ijk[d] = i;
                    const int64_t k = kidx(ijk[0], ijk[1], ijk[2]);
                    ax[d].push_back(v->u[k * D + d]);
                    aw[d].push_back(d == 0 ? v->w[k] : v->w[k] / v->w[0]);
                }
            }
            for (int l = 0; l < nz && ok; ++l)
                for (int j = 0; j < ny && ok; ++j)
                    for (int i = 0; i < nx && ok; ++i) {
                        const int64_t k = kidx(i, j, l);
                        const int ijk[3] = {i, j, l};
                        double wp = 1.0;
                        for (int d = 0; d < D; ++d) {
                            ok = ok && v->u[k * D + d] == ax[d][ijk[d]];
                            wp *= aw[d][ijk[d]];
                        }
                        ok = ok && std::fabs(wp - v->w[k]) <= 1e-14 * std::fabs(v->w[k]) + 1e-300;
                    }
            if (ok) {
                dc.sep = 1;
                for (int d = 0; d < D; ++d) {
                    dc.cart_n[d] = nn[d];
                    dc.axis[d] = c->upload(cast<T>(ax[d]));
                    dc.axw[d] = c->upload(cast<T>(aw[d]));
                }
                // the separable half-range sums search the last axis for the
                // sign changes of u.n, so its nodes must ascend (also in T)
                const std::vector<T> last = cast<T>(ax[D - 1]);
                bool asc = last.size() <= (size_t)ugks::SUM1_SEP_MAX_NL;
                for (size_t i = 1; i < last.size(); ++i) asc = asc && last[i - 1] < last[i];
                dc.sep1 = asc ? 1 : 0;
            }
        }
    }
    std::vector<double> wd(c->nvp, 0.0);
    for (int64_t k = 0; k < c->Nv; ++k) wd[k] = v->w[k];
    dc.w = c->upload(cast<T>(wd));
    {
        std::vector<T> uw((size_t)c->nvp * 4, T(0));
        for (int64_t k = 0; k < c->Nv; ++k) {
            for (int d = 0; d < D; ++d) uw[(size_t)k * 4 + d] = (T)v->u[k * D + d];
            uw[(size_t)k * 4 + 3] = (T)v->w[k];
        }
        dc.uw = c->upload(uw);
    }
    // state
    const size_t fcount = (size_t)c->C * c->NC * c->nvp;
    dc.f_cur = (T *)c->dalloc(fcount * sizeof(T));
    // the flux buffer also stages state I/O, in host rows of up to FP64: room
    // for at least two cells' FP64 rows (one per upload slot), even on tiny meshes
    c->stage_bytes = std::max((size_t)c->F * c->NC * c->chunk * sizeof(T), (size_t)2 * c->NC * c->nvp * sizeof(double));
    dc.flux = (T *)c->dalloc(c->stage_bytes);
    std::vector<double> W((size_t)c->C * M);
    for (int64_t i = 0; i < c->C; ++i) {
        const int ci = h.perm_u2i[i];
        double pr[5];
        if (p->prim_init) {
            for (int k = 0; k < M; ++k) pr[k] = p->prim_init[i * M + k];
        } else {
            pr[0] = p->inf_rho;
            for (int d = 0; d < D; ++d) pr[1 + d] = p->inf_U[d];
            pr[D + 1] = p->inf_T;
        }
        double ke = 0.0;
        W[(size_t)ci * M] = pr[0];
        for (int d = 0; d < D; ++d) {
            W[(size_t)ci * M + 1 + d] = pr[0] * pr[1 + d];
            ke += pr[1 + d] * pr[1 + d];
        }
        W[(size_t)ci * M + D + 1] = pr[0] * (0.5 * ke + 1.5 * pr[D + 1]);
    }
    dc.W = c->upload(W);
    dc.q = (double *)c->dalloc((size_t)c->C * D * sizeof(double));
    dc.gradW = (double *)c->dalloc((size_t)c->C * D * M * sizeof(double));
    dc.gradprim = (double *)c->dalloc((size_t)c->C * D * M * sizeof(double));
    dc.prim = (double *)c->dalloc((size_t)c->C * M * sizeof(double));
    dc.primg = (double *)c->dalloc((size_t)std::max(c->G, 1) * M * sizeof(double));
    dc.nb_ptr = c->upload(h.nb_ptr);
    dc.nb_id = c->upload(h.nb_id);
    dc.nb_a_d = c->upload(h.nb_a);
    dc.cf_ptr = c->upload(h.cf_ptr);
    dc.cf_r_d = c->upload(h.cf_r);
    dc.gi = reinterpret_cast<const int4 *>(c->upload(h.gi));
    dc.gf = c->upload(cast<T>(h.gf));
    dc.nf = h.nf;
    dc.eps2_d = c->upload(h.eps2);
    dc.eps2 = c->upload(cast<T>(h.eps2));
    dc.fL = c->upload(h.fL);
    dc.fR = c->upload(h.fR);
    dc.faux = c->upload(h.faux);
    dc.ftype = c->upload(h.ftype);
    dc.ftag = c->upload(h.ftag);
    dc.fn_d = c->upload(h.fn);
    dc.frL_d = c->upload(h.frL);
    dc.frR_d = c->upload(h.frR);
    dc.fn = c->upload(cast<T>(h.fn));
    dc.frL = c->upload(cast<T>(h.frL));
    dc.dtT = (T)c->dt;
    dc.one = T(1);
    dc.gface = c->upload(h.gface);
    dc.Wg = (double *)c->dalloc((size_t)std::max(c->G, 1) * M * sizeof(double));
    dc.grec = (T *)c->dalloc((size_t)std::max(c->G, 1) * ugks::GREC * sizeof(T));
    dc.wface = c->upload(h.wface);
    std::vector<double> wT(std::max(p->n_walls, 1), 1.0), wU(3 * std::max(p->n_walls, 1), 0.0);
    for (int i = 0; i < p->n_walls; ++i) {
        wT[i] = p->wall_T[i];
        for (int d = 0; d < 3; ++d) wU[3 * i + d] = p->wall_U[3 * i + d];
    }
    dc.wallT = c->upload(wT);
    dc.wallU = c->upload(wU);
    {
        double ke = 0.0;
        dc.inf_W[0] = p->inf_rho;
        for (int d = 0; d < D; ++d) {
            dc.inf_W[1 + d] = p->inf_rho * p->inf_U[d];
            ke += p->inf_U[d] * p->inf_U[d];
        }
        dc.inf_W[D + 1] = p->inf_rho * (0.5 * ke + 1.5 * p->inf_T);
    }
    dc.rho_w = (double *)c->dalloc((size_t)std::max(c->NW, 1) * sizeof(double));
    dc.wall_F = (double *)c->dalloc((size_t)std::max(c->NW, 1) * M * sizeof(double));
    cuda_ok(cudaMemsetAsync(dc.wall_F, 0, (size_t)std::max(c->NW, 1) * M * sizeof(double), c->stream), "memset");
    c->wall_face_h.assign(h.wface.begin(), h.wface.end());
    c->wall_n_h.resize((size_t)c->NW * D);
    for (int s = 0; s < c->NW; ++s)
        for (int d = 0; d < D; ++d) c->wall_n_h[(size_t)s * D + d] = m->face_n[(size_t)h.wface[s] * D + d];
    dc.wrec = (T *)c->dalloc((size_t)std::max(c->NW, 1) * ugks::GREC * sizeof(T));
    dc.crec = (T *)c->dalloc((size_t)c->C * ugks::CREC * sizeof(T));
    dc.krec = (T *)c->dalloc((size_t)c->C * ugks::CREC * sizeof(T));
    const size_t Fm = (size_t)std::max<int64_t>(c->F, 1);
    dc.frec = (T *)c->dalloc(Fm * ugks::FREC * sizeof(T));
    dc.xrec = (T *)c->dalloc(Fm * (D == 2 ? ugks::XRec<2>::LEN : ugks::XRec<3>::LEN) * sizeof(T));
    dc.fside = (T *)c->dalloc(Fm * 2 * ugks::GREC * sizeof(T));
    dc.fdW0 = (double *)c->dalloc(Fm * D * M * sizeof(double));
    dc.fq0 = (double *)c->dalloc(Fm * D * sizeof(double));
    dc.fUref = (double *)c->dalloc(Fm * D * sizeof(double));
    dc.fsum1 = (double *)c->dalloc(Fm * M * sizeof(double));
    const int NS = M * (M + 1) / 2;
    dc.fsum2 = (double *)c->dalloc(Fm * NS * (D + 1) * sizeof(double));
    dc.fprim0 = (double *)c->dalloc(Fm * M * sizeof(double));
    dc.fqs = (double *)c->dalloc(Fm * 5 * sizeof(double));
    dc.dW_part = (double *)c->dalloc((size_t)c->C * c->n_groups * M * sizeof(double));
    // the partials, then the folded ones (residual_parts)
    dc.res_part = (double *)c->dalloc((size_t)(c->n_res_parts + c->n_res_parts / ugks::RES_FOLD + 1) * 2 * M * sizeof(double));
    dc.flags = c->flags_d;
    dc.owned = nullptr;
    dc.gvel = c->gvel;
    dc.n_groups = c->n_groups;
    dc.chunk = c->chunk;
    dc.n_chunks = c->n_chunks;
    dc.parts = c->parts;
    dc.carry = c->parts > 1 ? (T *)c->dalloc(carry_bytes(c)) : nullptr;
    dc.P = c->P;
    dc.nth = c->nth;
    dc.n_patches = c->n_patches;
    dc.vtile = c->vtile;
}

}  // namespace

namespace {

// velocity tile used when neither the caller nor the autotuner sets one
int kDefaultVtile(int prec) { return prec == UGKS_FP64 ? 32 : 64; }

// Velocities per warp of stage 1 (gvel) and per chunk of the flux buffer.
// A warp of stage 1 ends its group of velocities with a reduction over its lanes
// that costs as much as about 250 velocities of the pass itself: groups of 1024,
// fewer where the mesh has too few cells to fill the chip with one warp per cell
// and group, or where the flux buffer of a group would exceed 9/8 of a copy of f.  (The
// 107k-cell tetrahedral mesh x 4,568 velocities in FP32, flux and stage-1 passes:
// 9.10, 8.30 and 7.95 ms at 256, 512 and 1024.)  The buffer holds as many
// groups as fit 64 MB or 9/8 of a copy of f, whichever is smaller (4 MB are always
// taken): fewer launches for small cases (the 1/8 lets quadrilaterals, 2.1 faces
// per cell, do with two chunks), little memory for large ones.
// With a tiling of the caller's (patch_cells or the group given) the group depends on
// the velocities alone, so that a cell's moments are summed alike on any mesh that
// holds it, a subdomain's or the whole one.  Where the fluxes of such a group exceed
// 9/8 of a copy of f by more than the lane sums that stage 1 then keeps
// (carry_bytes), it is cut into several chunks.
void set_chunks(ugks_case *c, int tile_group, bool fixed)
{
    const int nvp = (int)c->nvp;
    const size_t per_vel = (size_t)std::max<int64_t>(c->F, 1) * c->NC * (c->prec == UGKS_FP64 ? 8 : 4);
    const size_t most = std::max((size_t)c->f_bytes + c->f_bytes / 8, (size_t)4 << 20);
    const int64_t warps = 152 * 32;
    int groups = (nvp + 1023) / 1024, step = 128;
    auto vel = [&] { return ((nvp + groups - 1) / groups + step - 1) / step * step; };
    while (!fixed && vel() > step && (c->C * groups < warps || vel() * per_vel > most)) ++groups;
    c->gvel = std::min(vel(), nvp);
    if (tile_group > 0) c->gvel = (int)std::min<int64_t>((int64_t)tile_group * c->vtile, nvp);
    c->n_groups = (nvp + c->gvel - 1) / c->gvel;
    if (fixed && c->gvel > 128 && per_vel * c->gvel > most + carry_bytes(c)) {
        const int fit = (int)std::max<size_t>(1, most / (per_vel * 128)) * 128;
        c->parts = (c->gvel + fit - 1) / fit;
        c->chunk = ((c->gvel + c->parts - 1) / c->parts + 127) / 128 * 128;
        c->parts = (c->gvel + c->chunk - 1) / c->chunk;
        const int last = nvp - (c->n_groups - 1) * c->gvel;
        c->n_chunks = (c->n_groups - 1) * c->parts + (last + c->chunk - 1) / c->chunk;
        return;
    }
    const size_t in = std::max<size_t>(1, std::min(most, (size_t)64 << 20) / (per_vel * c->gvel));
    c->n_chunks = (int)((c->n_groups + in - 1) / in);
    c->chunk = std::min((c->n_groups + c->n_chunks - 1) / c->n_chunks * c->gvel, nvp);
    c->n_chunks = (nvp + c->chunk - 1) / c->chunk;
}

// Autotuner of the flux pass: cells per patch and velocities per warp are chosen
// by timing the flux and stage-1 passes themselves on this case (before the
// state is initialised for the caller), and the choice is cached per (dimension,
// precision, velocity count, mesh-size bucket) for later cases of the same shape.
struct Tiling {
    int P = 0, vtile = 0;
};
std::mutex g_tune_mutex;
std::map<std::string, Tiling> g_tune_cache;

template <typename T>
void set_tiling(ugks_case *c, ugks::DevCase<T> &dc, int P, int vtile)
{
    dc.P = c->P = P;
    dc.n_patches = c->n_patches = (int)((c->C + P - 1) / P);
    dc.vtile = c->vtile = vtile;
}

template <typename T>
void autotune(ugks_case *c, ugks::DevCase<T> &dc, bool tune_vtile)
{
    char key[160];
    snprintf(key, sizeof(key), "D%d_nf%d_p%d_vt%d_t%d_g%d_nv%lld_c%d", c->D, c->nf, c->prec,
             tune_vtile ? 0 : c->vtile, c->nth, c->gvel, (long long)c->Nv,
             (int)std::lround(std::log2((double)c->C)));
    Tiling best;
    {
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) best = it->second;
    }
    if (best.P == 0) {
        std::vector<int> vc = {c->vtile};
        if (tune_vtile) vc = c->prec == UGKS_FP64 ? std::vector<int>{32, 64} : std::vector<int>{64, 128};
        cuda_ok(ugks::launch_pre_gather(dc, c->stream), "autotune prep");
        cudaEvent_t e0, e1;
        cuda_ok(cudaEventCreate(&e0), "event");
        cuda_ok(cudaEventCreate(&e1), "event");
        float best_ms = 0.f;
        for (int vt : vc) {
            // whole tiles per group, so that the reported tiling gives the same groups again;
            // the key holds all that this depends on
            if ((c->gvel % vt && c->gvel != c->nvp) || (c->nth == 512 && vt > 64)) continue;
            for (int P : {8, 16, 32, 64}) {
                if (P > 8 && (P < c->nth / 32 || P > std::max<int64_t>(16, c->C / 64))) continue;
                set_tiling(c, dc, P, vt);
                cuda_ok(ugks::launch_gather(dc, c->stream), "autotune gather");
                cuda_ok(cudaEventRecord(e0, c->stream), "event");
                for (int r = 0; r < 2; ++r) cuda_ok(ugks::launch_gather(dc, c->stream), "autotune gather");
                cuda_ok(cudaEventRecord(e1, c->stream), "event");
                cuda_ok(cudaEventSynchronize(e1), "event");
                float ms = 0.f;
                cuda_ok(cudaEventElapsedTime(&ms, e0, e1), "event");
                if (best.P == 0 || ms < best_ms) {
                    best = {P, vt};
                    best_ms = ms;
                }
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        std::lock_guard<std::mutex> lock(g_tune_mutex);
        g_tune_cache[key] = best;
    }
    set_tiling(c, dc, best.P, best.vtile);
}

ugks_status guard(const std::function<void()> &fn)
{
    try {
        g_err.clear();
        fn();
        return UGKS_OK;
    } catch (const Fail &e) {
        g_err = e.msg;
        return e.code;
    } catch (const std::bad_alloc &) {
        g_err = "host allocation failed";
        return UGKS_ENOMEM;
    } catch (const std::exception &e) {
        g_err = e.what();
        return UGKS_EINVAL;
    } catch (...) {
        g_err = "unknown error";
        return UGKS_EINVAL;
    }
}

template <typename Fn>
auto with_dc(ugks_case *c, Fn &&fn)
{
    if (c->prec == UGKS_FP64) return fn(c->d64);
    return fn(c->d32);
}

// f of the case into host memory, f[C][ncomp][nv] of element type S in caller
// cell order, staged through the flux buffer in chunks of cells
template <typename S>
void export_f(ugks_case *c, S *f)
{
    const size_t per = (size_t)c->NC * c->Nv;
    const size_t cap = c->stage_bytes / sizeof(S);
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>(cap / per, (size_t)c->C));
    for (int c0 = 0; c0 < (int)c->C; c0 += chunk) {
        const int nc = (int)std::min<int64_t>(chunk, c->C - c0);
        with_dc(c, [&](auto &dc) {
            S *stg = (S *)dc.flux;
            cuda_ok(ugks::launch_f_export(dc, c->perm_d, c0, nc, stg, c->stream), "f export");
            cuda_ok(cudaMemcpyAsync(f + (size_t)c0 * per, stg, (size_t)nc * per * sizeof(S), cudaMemcpyDeviceToHost,
                                    c->stream),
                    "f copy");
            cuda_ok(cudaStreamSynchronize(c->stream), "sync");
        });
    }
}

// f from host memory (layout of export_f) into the case.  The flux buffer is
// split into two staging slots; chunks of cells alternate between them.  The
// copy of a chunk runs on the case's copy stream while the case stream imports
// (reorders and converts) the chunk before it; a slot is refilled only after
// its previous import.  The first copy waits for the work already queued on
// the case stream, which may still use the buffer.
template <typename S>
void import_f(ugks_case *c, const S *f)
{
    const size_t per = (size_t)c->NC * c->Nv;
    const size_t slot = c->stage_bytes / 2 / sizeof(S);            // >= one cell's row
    int chunk = (int)std::max<size_t>(1, std::min<size_t>(slot / per, (size_t)c->C));
    chunk = std::min(chunk, (int)std::max<int64_t>(1, (c->C + 3) / 4));   // at least four chunks in flight
    if (!c->copy_stream) {
        cuda_ok(cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking), "copy stream");
        for (auto &e : c->io_ev) cuda_ok(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "event create");
    }
    cudaEvent_t ready = c->io_ev[0], *copied = c->io_ev + 1, *consumed = c->io_ev + 3;
    cuda_ok(cudaEventRecord(ready, c->stream), "event");
    cuda_ok(cudaStreamWaitEvent(c->copy_stream, ready, 0), "event wait");
    int k = 0;
    for (int c0 = 0; c0 < (int)c->C; c0 += chunk, ++k) {
        const int nc = (int)std::min<int64_t>(chunk, c->C - c0);
        const int sl = k & 1;
        if (k >= 2) cuda_ok(cudaStreamWaitEvent(c->copy_stream, consumed[sl], 0), "event wait");
        with_dc(c, [&](auto &dc) {
            S *stg = (S *)dc.flux + (size_t)sl * slot;
            cuda_ok(cudaMemcpyAsync(stg, f + (size_t)c0 * per, (size_t)nc * per * sizeof(S), cudaMemcpyHostToDevice,
                                    c->copy_stream),
                    "f upload");
            cuda_ok(cudaEventRecord(copied[sl], c->copy_stream), "event");
            cuda_ok(cudaStreamWaitEvent(c->stream, copied[sl], 0), "event wait");
            cuda_ok(ugks::launch_f_import(dc, c->perm_d, c0, nc, stg, c->stream), "f import");
            cuda_ok(cudaEventRecord(consumed[sl], c->stream), "event");
        });
    }
}

// W[C][dim+2] (caller cell order) into the case through the gradW scratch
void import_W(ugks_case *c, const double *W)
{
    const int D = c->D, M = D + 2;
    double *Wd = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
    double *stg = c->prec == UGKS_FP64 ? c->d64.gradW : c->d32.gradW;
    cuda_ok(cudaMemcpyAsync(stg, W, (size_t)c->C * M * sizeof(double), cudaMemcpyHostToDevice, c->stream),
            "W upload");
    cuda_ok(ugks::launch_W_permute(stg, c->perm_d, (int)c->C, D, Wd, 1, c->stream), "W import");
}

void export_W(ugks_case *c, double *W)
{
    const int D = c->D, M = D + 2;
    double *Wd = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
    double *stg = c->prec == UGKS_FP64 ? c->d64.gradW : c->d32.gradW;
    cuda_ok(ugks::launch_W_permute(Wd, c->perm_d, (int)c->C, D, stg, 0, c->stream), "W export");
    cuda_ok(cudaMemcpyAsync(W, stg, (size_t)c->C * M * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "W copy");
    cuda_ok(cudaStreamSynchronize(c->stream), "sync");
}

// the partial sums of the last step's residual and their number: folded by
// RES_FOLD above 65,536 cells, where copying or adding up the 32-cell partials takes
// longer than the launch (a million cells: ugks_residual_sums 0.162 -> 0.046 ms,
// ugks_residual 0.111 -> 0.052 ms; 30k cells unfolded 0.023, folded 0.027)
const double *residual_parts(ugks_case *c, int &n)
{
    double *rp = c->prec == UGKS_FP64 ? c->d64.res_part : c->d32.res_part;
    n = c->n_res_parts;
    if (n <= 2048) return rp;
    double *folded = rp + (size_t)n * 2 * (c->D + 2);
    cuda_ok(ugks::launch_residual_fold(rp, n, c->D, folded, c->stream), "residual launch");
    n = (n + ugks::RES_FOLD - 1) / ugks::RES_FOLD;
    return folded;
}

template <typename S>
ugks_status get_state(ugks_case *c, S *f, double *W)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (W) export_W(c, W);
        if (f) export_f(c, f);
    });
}

template <typename S>
ugks_status set_state(ugks_case *c, const S *f, const double *W)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (W) import_W(c, W);
        if (f) import_f(c, f);
        if (f || W) with_dc(c, [&](auto &dc) { cuda_ok(ugks::launch_heatflux(dc, c->stream), "heat flux"); });
    });
}
}  // namespace

namespace ugks {
// lets other translation units of the library report through ugks_last_error()
void set_last_error(const std::string &msg) { g_err = msg; }
}  // namespace ugks

extern "C" {

const char *ugks_last_error(void) { return g_err.c_str(); }

ugks_status ugks_create(const ugks_mesh *mesh, const ugks_vgrid *vgrid, const ugks_params *params,
                        const ugks_alloc *alloc, void *stream, ugks_case **out)
{
    if (!out) {
        g_err = "out must not be NULL";
        return UGKS_EINVAL;
    }
    *out = nullptr;
    std::unique_ptr<ugks_case> c(new ugks_case());
    ugks_status st = guard([&] {
        validate(mesh, vgrid, params);
        if (alloc && (!alloc->alloc || !alloc->free)) fail(UGKS_EINVAL, "allocator callbacks missing");
        c->D = mesh->dim;
        c->NC = mesh->dim == 2 ? 2 : 1;
        c->prec = params->precision;
        c->C = mesh->n_cells;
        c->F = mesh->n_faces;
        c->Nv = vgrid->nv;
        c->stream = (cudaStream_t)stream;
        if (alloc) {
            c->alloc = *alloc;
            c->user_alloc = true;
        }
        // velocity rows are padded to whole tiles, in 2D of 64 velocities at most (a
        // last tile of 128 may be short), as for the autotuner's choice of a tile
        c->vtile = params->vtile > 0 ? params->vtile : kDefaultVtile(c->prec);
        c->nth = params->gather_threads > 0 ? params->gather_threads : 256;
        const int most = c->D == 3 ? 128 : 64, vpad = params->vtile > 0 ? std::min(params->vtile, most) : most;
        c->P = params->patch_cells > 0 ? params->patch_cells : 16;
        Host h;
        preprocess(mesh, params, h);
        c->nf = h.nf;
        c->n_patches = (int)((c->C + c->P - 1) / c->P);
        c->nvp = (c->Nv + vpad - 1) / vpad * vpad;
        c->f_bytes = (size_t)c->C * c->NC * c->nvp * (c->prec == UGKS_FP64 ? 8 : 4);
        set_chunks(c.get(), params->gather_tile_group, params->patch_cells > 0 || params->gather_tile_group > 0);
        c->G = (int)h.gface.size();
        c->NW = (int)h.wface.size();
        // upwind CFL bound (the CFL step of Algorithm 1)
        c->dt = params->dt > 0.0 ? params->dt : cfl_dt_of(mesh, vgrid, params->cfl, mesh->n_cells);
        c->n_res_parts = (int)((c->C + 31) / 32);
        c->flags_d = (int *)c->dalloc(sizeof(int));
        cuda_ok(cudaMemsetAsync(c->flags_d, 0, sizeof(int), c->stream), "memset");
        c->range_d = (unsigned long long *)c->dalloc(2 * sizeof(unsigned long long));
        c->res_d = (double *)c->dalloc(8 * sizeof(double));
        cuda_ok(cudaMemsetAsync(c->res_d, 0, 8 * sizeof(double), c->stream), "memset");
        c->perm_h.assign(h.perm_u2i.begin(), h.perm_u2i.end());
        c->perm_d = c->upload(c->perm_h);
        with_dc(c.get(), [&](auto &dc) {
            fill_case(c.get(), dc, mesh, vgrid, params, h);
            cuda_ok(ugks::launch_init(dc, c->stream), "init");
            if (params->patch_cells == 0) {
                // the trial passes overwrite f in place: initialise it again
                autotune(c.get(), dc, params->vtile == 0);
                cuda_ok(ugks::launch_init(dc, c->stream), "init");
            }
            c->vt_group = (c->gvel + c->vtile - 1) / c->vtile;
        });
        cuda_ok(c->stream ? cudaStreamSynchronize(c->stream) : cudaDeviceSynchronize(), "create sync");
    });
    if (st != UGKS_OK) {
        std::string keep = g_err;
        c->release();
        g_err = keep;
        return st;
    }
    *out = c.release();
    return UGKS_OK;
}

ugks_status ugks_step(ugks_case *c, int32_t nsteps)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (nsteps < 0) fail(UGKS_EINVAL, "nsteps must be >= 0");
        for (int32_t s = 0; s < nsteps; ++s) {
            cudaEvent_t *ev = nullptr;
            if (c->prof_used < c->prof_max) ev = &c->prof_ev[(size_t)c->prof_used++ * (ugks::N_GROUPS + 1)];
            with_dc(c, [&](auto &dc) { cuda_ok(ugks::launch_step(dc, c->stream, ev), "step launch"); });
            ++c->step;
            c->stepped = true;
        }
    });
}

ugks_status ugks_check(ugks_case *c)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        const int M = c->D + 2;
        double *W = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
        cuda_ok(ugks::launch_check(W, (int)c->C, M, c->flags_d, c->stream), "check launch");
        int flag = 0;
        cuda_ok(cudaMemcpyAsync(&flag, c->flags_d, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "check copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "check sync");
        if (flag) fail(UGKS_ENUMERIC, "non-finite or non-positive density / temperature in the state");
    });
}

ugks_status ugks_density_range(ugks_case *c, double *range)
{
    return guard([&] {
        if (!c || !range) fail(UGKS_EINVAL, "case and range must not be NULL");
        const int M = c->D + 2;
        const double *W = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
        cuda_ok(ugks::launch_density_range(W, (int)c->C, M, c->owned_d, c->range_d, c->stream), "range launch");
        unsigned long long b[2];
        cuda_ok(cudaMemcpyAsync(b, c->range_d, sizeof(b), cudaMemcpyDeviceToHost, c->stream), "range copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "range sync");
        if (b[0] == ~0ull) b[0] = 0ull;          // no own cell
        std::memcpy(&range[0], &b[0], sizeof(double));
        std::memcpy(&range[1], &b[1], sizeof(double));
    });
}

ugks_status ugks_moments(ugks_case *c, double *rho, double *U, double *T, double *q)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        const int D = c->D;
        const size_t per = 2 * D + 2;
        double *Wd = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
        double *qd = c->prec == UGKS_FP64 ? c->d64.q : c->d32.q;
        // reuse the gradient buffer as staging ([C][D][D+2] >= [C][2D+2])
        double *out = c->prec == UGKS_FP64 ? c->d64.gradW : c->d32.gradW;
        cuda_ok(ugks::launch_moments_out(Wd, qd, c->perm_d, (int)c->C, D, out, c->stream), "moments launch");
        std::vector<double> hbuf((size_t)c->C * per);
        cuda_ok(cudaMemcpyAsync(hbuf.data(), out, hbuf.size() * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                "moments copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "moments sync");
        for (int64_t i = 0; i < c->C; ++i) {
            const double *o = &hbuf[(size_t)i * per];
            if (rho) rho[i] = o[0];
            for (int d = 0; d < D; ++d) {
                if (U) U[i * D + d] = o[1 + d];
                if (q) q[i * D + d] = o[D + 2 + d];
            }
            if (T) T[i] = o[D + 1];
        }
    });
}

ugks_status ugks_residual(ugks_case *c, double *res)
{
    return guard([&] {
        if (!c || !res) fail(UGKS_EINVAL, "case and res must not be NULL");
        const int M = c->D + 2;
        if (!c->stepped) {
            for (int m = 0; m < M; ++m) res[m] = 0.0;
            return;
        }
        int n;
        const double *rp = residual_parts(c, n);
        cuda_ok(ugks::launch_residual(rp, n, c->D, c->res_d, c->stream), "residual launch");
        cuda_ok(cudaMemcpyAsync(res, c->res_d, M * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "residual copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "residual sync");
    });
}

ugks_status ugks_get_state(ugks_case *c, double *f, double *W) { return get_state(c, f, W); }

ugks_status ugks_get_state_f32(ugks_case *c, float *f, double *W) { return get_state(c, f, W); }

ugks_status ugks_wall_quantities(ugks_case *c, int64_t *face, double *p, double *sigma, double *q)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        const int D = c->D, M = D + 2, NW = c->NW;
        if (NW == 0) return;
        std::vector<double> F((size_t)NW * M);
        const double *Fd = c->prec == UGKS_FP64 ? c->d64.wall_F : c->d32.wall_F;
        cuda_ok(cudaMemcpyAsync(F.data(), Fd, F.size() * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                "wall flux copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "sync");
        for (int s = 0; s < NW; ++s) {
            const double *Fs = &F[(size_t)s * M];
            const double *n = &c->wall_n_h[(size_t)s * D];
            double pn = 0.0, t2 = 0.0;
            for (int d = 0; d < D; ++d) pn += Fs[1 + d] * n[d];
            for (int d = 0; d < D; ++d) {
                const double t = Fs[1 + d] - pn * n[d];
                t2 += t * t;
            }
            if (face) face[s] = c->wall_face_h[s];
            if (p) p[s] = pn / c->dt;
            if (sigma) sigma[s] = std::sqrt(t2) / c->dt;
            if (q) q[s] = Fs[D + 1] / c->dt;
        }
    });
}

ugks_status ugks_get_cells(ugks_case *c, const int64_t *cells, int64_t n, double *f, double *W)
{
    return guard([&] {
        if (!c || !cells) fail(UGKS_EINVAL, "case and cells must not be NULL");
        if (n < 0 || n > c->C) fail(UGKS_EINVAL, "n = %lld outside [0, n_cells]", (long long)n);
        if (n == 0) return;
        const int D = c->D, M = D + 2;
        std::vector<long long> ids((size_t)n);
        for (int64_t i = 0; i < n; ++i) {
            if (cells[i] < 0 || cells[i] >= c->C) fail(UGKS_EINVAL, "cell id %lld out of range", (long long)cells[i]);
            ids[(size_t)i] = c->perm_h[(size_t)cells[i]];
        }
        // staging in the gradient scratch (C*D*M doubles >= n*(1 + M)): the
        // internal ids, then W; f goes through the flux buffer in chunks
        double *gW = c->prec == UGKS_FP64 ? c->d64.gradW : c->d32.gradW;
        long long *ids_d = reinterpret_cast<long long *>(gW);
        double *wst = gW + n;
        cuda_ok(cudaMemcpyAsync(ids_d, ids.data(), (size_t)n * sizeof(long long), cudaMemcpyHostToDevice, c->stream),
                "ids upload");
        if (W) {
            double *Wd = c->prec == UGKS_FP64 ? c->d64.W : c->d32.W;
            cuda_ok(ugks::launch_W_permute(Wd, ids_d, (int)n, D, wst, 0, c->stream), "W gather");
            cuda_ok(cudaMemcpyAsync(W, wst, (size_t)n * M * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                    "W copy");
        }
        if (f) {
            const size_t per = (size_t)c->NC * c->Nv;
            const size_t cap = c->stage_bytes / sizeof(double);
            const int chunk = (int)std::max<size_t>(1, std::min<size_t>(cap / per, (size_t)n));
            for (int c0 = 0; c0 < (int)n; c0 += chunk) {
                const int nc = (int)std::min<int64_t>(chunk, n - c0);
                with_dc(c, [&](auto &dc) {
                    double *stg = (double *)dc.flux;
                    cuda_ok(ugks::launch_f_export(dc, ids_d, c0, nc, stg, c->stream), "f gather");
                    cuda_ok(cudaMemcpyAsync(f + (size_t)c0 * per, stg, (size_t)nc * per * sizeof(double),
                                            cudaMemcpyDeviceToHost, c->stream),
                            "f copy");
                });
                cuda_ok(cudaStreamSynchronize(c->stream), "sync");
            }
        }
        cuda_ok(cudaStreamSynchronize(c->stream), "sync");
    });
}

ugks_status ugks_set_state(ugks_case *c, const double *f, const double *W) { return set_state(c, f, W); }

ugks_status ugks_set_state_f32(ugks_case *c, const float *f, const double *W) { return set_state(c, f, W); }

ugks_status ugks_profile_begin(ugks_case *c, int32_t max_steps)
{
    return guard([&] {
        if (!c || max_steps < 0) fail(UGKS_EINVAL, "invalid profile request");
        for (auto e : c->prof_ev) cudaEventDestroy(e);
        c->prof_ev.assign((size_t)max_steps * (ugks::N_GROUPS + 1), nullptr);
        for (auto &e : c->prof_ev) cuda_ok(cudaEventCreate(&e), "event create");
        c->prof_max = max_steps;
        c->prof_used = 0;
    });
}

ugks_status ugks_profile_end(ugks_case *c, double *ms, int32_t n, int32_t *steps)
{
    return guard([&] {
        if (!c || !ms) fail(UGKS_EINVAL, "invalid profile request");
        cuda_ok(c->stream ? cudaStreamSynchronize(c->stream) : cudaDeviceSynchronize(), "profile sync");
        for (int i = 0; i < n; ++i) ms[i] = 0.0;
        for (int s = 0; s < c->prof_used; ++s)
            for (int g = 0; g < ugks::N_GROUPS && g < n; ++g) {
                float t = 0.f;
                cudaEvent_t *e = &c->prof_ev[(size_t)s * (ugks::N_GROUPS + 1)];
                cuda_ok(cudaEventElapsedTime(&t, e[g], e[g + 1]), "event time");
                ms[g] += t;
            }
        if (steps) *steps = c->prof_used;
        for (auto e : c->prof_ev) cudaEventDestroy(e);
        c->prof_ev.clear();
        c->prof_max = c->prof_used = 0;
    });
}

ugks_status ugks_info(const ugks_case *c, ugks_info_t *info)
{
    return guard([&] {
        if (!c || !info) fail(UGKS_EINVAL, "case and info must not be NULL");
        info->dim = c->D;
        info->ncomp = c->NC;
        info->precision = c->prec;
        info->n_cells = c->C;
        info->n_faces = c->F;
        info->nv = c->Nv;
        info->nv_pad = c->nvp;
        info->dt = c->dt;
        info->step = c->step;
        info->device_bytes = c->device_bytes;
        info->f_bytes = c->f_bytes;
        info->n_patches = c->n_patches;
        info->patch_cells = c->P;
        info->vtile = c->vtile;
        info->gather_threads = c->nth;
        info->gather_tile_group = c->vt_group;
        info->kernel_launches_per_step = 4 + 2 * c->n_chunks + (c->F > 0 ? 5 : 0) + (c->NW > 0 ? 1 : 0);
        info->n_wall_faces = c->NW;
    });
}

ugks_status ugks_cfl_dt(const ugks_mesh *mesh, const ugks_vgrid *vgrid, double cfl, int64_t n_cells, double *dt)
{
    return guard([&] {
        if (!mesh || !vgrid || !dt) fail(UGKS_EINVAL, "mesh, vgrid and dt must not be NULL");
        if (!(cfl > 0.0)) fail(UGKS_EINVAL, "cfl must be > 0");
        if (n_cells < 1 || n_cells > mesh->n_cells) fail(UGKS_EINVAL, "n_cells outside [1, mesh n_cells]");
        if (!mesh->cell_vol || !mesh->face_cells || !mesh->face_S || !vgrid->u || vgrid->nv < 1 ||
            vgrid->dim != mesh->dim)
            fail(UGKS_EINVAL, "incomplete mesh or velocity grid");
        for (int64_t f = 0; f < mesh->n_faces; ++f) {
            const int64_t a = mesh->face_cells[2 * f], b = mesh->face_cells[2 * f + 1];
            if (a < 0 || a >= mesh->n_cells || b >= mesh->n_cells) fail(UGKS_EINVAL, "face %lld: cell out of range",
                                                                       (long long)f);
        }
        *dt = cfl_dt_of(mesh, vgrid, cfl, n_cells);
    });
}

ugks_status ugks_set_owned(ugks_case *c, int64_t n_owned)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (n_owned < 0 || n_owned > c->C) fail(UGKS_EINVAL, "n_owned outside [0, n_cells]");
        std::vector<unsigned char> mask((size_t)c->C, 0);
        for (int64_t i = 0; i < n_owned; ++i) mask[(size_t)c->perm_h[(size_t)i]] = 1;
        if (!c->owned_d) c->owned_d = (unsigned char *)c->dalloc((size_t)c->C);
        cuda_ok(cudaMemcpyAsync(c->owned_d, mask.data(), mask.size(), cudaMemcpyHostToDevice, c->stream), "upload");
        cuda_ok(cudaStreamSynchronize(c->stream), "sync");
        c->d64.owned = c->owned_d;
        c->d32.owned = c->owned_d;
    });
}

ugks_status ugks_residual_sums(ugks_case *c, double *sums)
{
    return guard([&] {
        if (!c || !sums) fail(UGKS_EINVAL, "case and sums must not be NULL");
        const int M = c->D + 2;
        for (int i = 0; i < 2 * M; ++i) sums[i] = 0.0;
        if (!c->stepped) return;
        int n;
        const double *rp = residual_parts(c, n);
        std::vector<double> part((size_t)n * 2 * M);
        cuda_ok(cudaMemcpyAsync(part.data(), rp, part.size() * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                "residual copy");
        cuda_ok(cudaStreamSynchronize(c->stream), "residual sync");
        for (int b = 0; b < n; ++b)
            for (int i = 0; i < 2 * M; ++i) sums[i] += part[(size_t)b * 2 * M + i];
    });
}

ugks_status ugks_halo_row_bytes(const ugks_case *c, size_t *bytes)
{
    return guard([&] {
        if (!c || !bytes) fail(UGKS_EINVAL, "case and bytes must not be NULL");
        const size_t esz = c->prec == UGKS_FP64 ? 8 : 4;
        const size_t fbytes = ((size_t)c->NC * c->Nv * esz + 7) / 8 * 8;
        *bytes = fbytes + (size_t)(2 * c->D + 2) * sizeof(double);
    });
}

ugks_status ugks_halo_set(ugks_case *c, int32_t slot, const int64_t *cells, int64_t n)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (slot < 0 || slot >= 4096) fail(UGKS_EINVAL, "slot outside [0, 4096)");
        if (n < 0 || n > c->C || (n > 0 && !cells)) fail(UGKS_EINVAL, "invalid cell list");
        std::vector<int> ids((size_t)n);
        for (int64_t i = 0; i < n; ++i) {
            if (cells[i] < 0 || cells[i] >= c->C) fail(UGKS_EINVAL, "cell id %lld out of range", (long long)cells[i]);
            ids[(size_t)i] = (int)c->perm_h[(size_t)cells[i]];
        }
        if ((size_t)slot >= c->halo.size()) c->halo.resize((size_t)slot + 1);
        auto &h = c->halo[(size_t)slot];
        if (h.ids) {
            cuda_ok(cudaStreamSynchronize(c->stream), "sync");   // queued packs may still read the old list
            c->dfree(h.ids);
            h.ids = nullptr;
        }
        h.n = (int)n;
        if (n > 0) h.ids = c->upload(ids);
        cuda_ok(cudaStreamSynchronize(c->stream), "sync");
    });
}

static ugks_status halo_move(ugks_case *c, int32_t slot, void *buf, int unpack)
{
    return guard([&] {
        if (!c) fail(UGKS_EINVAL, "case is NULL");
        if (slot < 0 || (size_t)slot >= c->halo.size()) fail(UGKS_EINVAL, "halo slot %d is not set", slot);
        const auto &h = c->halo[(size_t)slot];
        if (h.n > 0 && !buf) fail(UGKS_EINVAL, "buffer must not be NULL");
        size_t row = 0;
        ugks_halo_row_bytes(c, &row);
        with_dc(c, [&](auto &dc) {
            cuda_ok(ugks::launch_halo(dc, h.ids, h.n, row, buf, unpack, c->stream), unpack ? "halo unpack" : "halo pack");
        });
    });
}

ugks_status ugks_halo_pack(ugks_case *c, int32_t slot, void *device_buf) { return halo_move(c, slot, device_buf, 0); }

ugks_status ugks_halo_unpack(ugks_case *c, int32_t slot, const void *device_buf)
{
    return halo_move(c, slot, const_cast<void *>(device_buf), 1);
}

}  // extern "C"

struct ugks_batch {
    std::vector<ugks_case *> cases;
    int D = 0, prec = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    void *dcases = nullptr;         // device array of DevCase<T>
    // the flux and stage-1 passes, one launch each per chunk over the cases of a
    // group (same velocity tile and entry count): per chunk
    // the block offsets of both kernels over all cases of the batch
    struct Group {
        int vtile = 0, nf = 0, n_chunks = 0;
        int *off = nullptr;                  // [n_chunks][2][n + 1]
        std::vector<int> blocks;             // [n_chunks][2]
        cudaStream_t branch = nullptr;       // capture stream of the group's branch (but the first's)
        cudaEvent_t join = nullptr;
    };
    std::vector<Group> groups;
    cudaEvent_t fork = nullptr;
    // the other kernels of a step, one launch each over all cases: block offsets
    // off[k][0..n] (device, prefix sums of the cases' block counts), total
    // blocks and dynamic shared memory per kernel
    int *small_off = nullptr;
    int small_blocks[ugks::SK_COUNT] = {}, small_threads[ugks::SK_COUNT] = {};
    size_t small_smem[ugks::SK_COUNT] = {};
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<cudaEvent_t> case_ev;   // orders each case's stream with the batch stream
    cudaEvent_t done = nullptr;
};

namespace {

template <typename T>
ugks::DevCase<T> &dc_of(ugks_case *c);
template <>
ugks::DevCase<double> &dc_of<double>(ugks_case *c) { return c->d64; }
template <>
ugks::DevCase<float> &dc_of<float>(ugks_case *c) { return c->d32; }

template <typename T>
void batch_build(ugks_batch *b)
{
    const int n = (int)b->cases.size();
    std::vector<ugks::DevCase<T>> h(n);
    for (int i = 0; i < n; ++i) h[i] = dc_of<T>(b->cases[i]);
    cuda_ok(cudaMalloc(&b->dcases, sizeof(ugks::DevCase<T>) * n), "batch alloc");
    cuda_ok(cudaMemcpy(b->dcases, h.data(), sizeof(ugks::DevCase<T>) * n, cudaMemcpyHostToDevice), "batch upload");
    // offsets of the batched per-case kernels
    std::vector<int> off((size_t)ugks::SK_COUNT * (n + 1), 0);
    for (int k = 0; k < ugks::SK_COUNT; ++k) {
        int *o = &off[(size_t)k * (n + 1)];
        long long items = 0;
        for (int i = 0; i < n; ++i) items += ugks::small_kernel_items<T>(h[i], k);
        b->small_threads[k] = ugks::small_kernel_threads(k, items);
        for (int i = 0; i < n; ++i) {
            const long long nb = (long long)o[i] + ugks::small_kernel_blocks(k, ugks::small_kernel_items<T>(h[i], k),
                                                                             b->small_threads[k]);
            if (nb > INT32_MAX) fail(UGKS_EINVAL, "batch too large for one launch of kernel %d", k);
            o[i + 1] = (int)nb;
            b->small_smem[k] = std::max(b->small_smem[k], ugks::small_kernel_smem<T>(h[i], k));
        }
        b->small_blocks[k] = o[n];
    }
    cuda_ok(cudaMalloc((void **)&b->small_off, off.size() * sizeof(int)), "batch alloc");
    cuda_ok(cudaMemcpy(b->small_off, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice), "batch upload");
    for (auto *first : b->cases) {
        auto in_group = [&](const ugks_case *c) {
            return c->vtile == first->vtile && c->nf == first->nf;
        };
        if (first != *std::find_if(b->cases.begin(), b->cases.end(), in_group)) continue;   // its group is there
        ugks_batch::Group g;
        g.vtile = first->vtile;
        g.nf = first->nf;
        for (auto *c : b->cases)
            if (in_group(c)) g.n_chunks = std::max(g.n_chunks, c->n_chunks);
        std::vector<int> goff((size_t)g.n_chunks * 2 * (n + 1), 0);
        for (int r = 0; r < g.n_chunks; ++r)
            for (int k = 0; k < 2; ++k) {
                int *o = &goff[((size_t)r * 2 + k) * (n + 1)];
                for (int i = 0; i < n; ++i) {
                    long long nb = o[i];
                    if (in_group(b->cases[i])) nb += k == 0 ? ugks::flux_blocks<T>(h[i], r) : ugks::stage1_blocks<T>(h[i], r);
                    if (nb > INT32_MAX) fail(UGKS_EINVAL, "batch too large for one launch of the flux pass");
                    o[i + 1] = (int)nb;
                }
                g.blocks.push_back(o[n]);
            }
        cuda_ok(cudaMalloc((void **)&g.off, goff.size() * sizeof(int)), "batch alloc");
        b->groups.push_back(g);      // owned by the batch from here on
        if (b->groups.size() > 1) {
            cuda_ok(cudaStreamCreateWithFlags(&b->groups.back().branch, cudaStreamNonBlocking), "branch stream");
            cuda_ok(cudaEventCreateWithFlags(&b->groups.back().join, cudaEventDisableTiming), "branch event");
        }
        cuda_ok(cudaMemcpy(g.off, goff.data(), goff.size() * sizeof(int), cudaMemcpyHostToDevice), "batch upload");
    }
}

template <typename T>
void batch_capture(ugks_batch *b)
{
    cudaStream_t st = b->stream;
    const int n = (int)b->cases.size();
    const auto *dcs = (const ugks::DevCase<T> *)b->dcases;
    auto small = [&](int k) {
        cuda_ok(ugks::launch_small_batch<T>(b->D, k, dcs, b->small_off + (size_t)k * (n + 1), n, b->small_blocks[k],
                                            b->small_threads[k], b->small_smem[k], st),
                "batched step kernel");
    };
    cuda_ok(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal), "begin capture");
    for (int k = ugks::SK_PREP; k <= ugks::SK_WALL_SUM; ++k) small(k);
    // the groups' passes touch different cases: branches of the graph, so that the
    // last blocks of one run beside the first of another
    cuda_ok(cudaEventRecord(b->fork, st), "fork");
    for (size_t gi = 0; gi < b->groups.size(); ++gi) {
        const auto &g = b->groups[gi];
        cudaStream_t sg = gi == 0 ? st : g.branch;
        if (gi > 0) cuda_ok(cudaStreamWaitEvent(sg, b->fork, 0), "fork");
        for (int r = 0; r < g.n_chunks; ++r) {
            const int *off = g.off + (size_t)r * 2 * (n + 1);
            cuda_ok(ugks::launch_flux<T>(b->D, g.nf, g.vtile, g.blocks[2 * r], r, sg, nullptr, dcs, off, n),
                    "batched flux pass");
            cuda_ok(ugks::launch_stage1<T>(b->D, g.nf, g.blocks[2 * r + 1], r, sg, nullptr, dcs, off + n + 1, n),
                    "batched stage 1");
        }
        if (gi > 0) {
            cuda_ok(cudaEventRecord(g.join, sg), "join");
            cuda_ok(cudaStreamWaitEvent(st, g.join, 0), "join");
        }
    }
    small(ugks::SK_UPDATE_W);
    small(ugks::SK_COLLIDE);
    cuda_ok(cudaStreamEndCapture(st, &b->graph), "end capture");
    cuda_ok(cudaGraphInstantiate(&b->exec, b->graph, 0), "graph instantiate");
}

void batch_free(ugks_batch *b)
{
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->dcases) cudaFree(b->dcases);
    for (auto &g : b->groups) {
            if (g.off) cudaFree(g.off);
            if (g.join) cudaEventDestroy(g.join);
            if (g.branch) cudaStreamDestroy(g.branch);
        }
    if (b->small_off) cudaFree(b->small_off);
    for (auto e : b->case_ev)
        if (e) cudaEventDestroy(e);
    if (b->done) cudaEventDestroy(b->done);
    if (b->fork) cudaEventDestroy(b->fork);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
}

}  // namespace

extern "C" {

ugks_status ugks_batch_create(ugks_case *const *cases, int32_t n, void *stream, ugks_batch **out)
{
    if (!out) {
        g_err = "out must not be NULL";
        return UGKS_EINVAL;
    }
    *out = nullptr;
    std::unique_ptr<ugks_batch> b(new ugks_batch());
    ugks_status st = guard([&] {
        if (!cases || n <= 0) fail(UGKS_EINVAL, "a batch needs at least one case");
        for (int i = 0; i < n; ++i) {
            if (!cases[i]) fail(UGKS_EINVAL, "case %d is NULL", i);
            if (cases[i]->D != cases[0]->D || cases[i]->prec != cases[0]->prec)
                fail(UGKS_EINVAL, "case %d differs from case 0 in dimension or precision", i);
            for (int j = 0; j < i; ++j)
                if (cases[j] == cases[i]) fail(UGKS_EINVAL, "case %d appears twice", i);
            b->cases.push_back(cases[i]);
        }
        b->D = cases[0]->D;
        b->prec = cases[0]->prec;
        if (stream) {
            b->stream = (cudaStream_t)stream;
        } else {
            cuda_ok(cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking), "stream");
            b->own_stream = true;
        }
        cuda_ok(cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming), "event");
        cuda_ok(cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming), "event");
        b->case_ev.assign(b->cases.size(), nullptr);
        for (auto &e : b->case_ev) cuda_ok(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "event");
        // the cases' own streams must have finished their queued work
        for (auto *c : b->cases) cuda_ok(c->stream ? cudaStreamSynchronize(c->stream) : cudaDeviceSynchronize(), "sync");
        if (b->prec == UGKS_FP64) batch_build<double>(b.get());
        else batch_build<float>(b.get());
    });
    if (st != UGKS_OK) {
        std::string keep = g_err;
        batch_free(b.get());
        g_err = keep;
        return st;
    }
    *out = b.release();
    return UGKS_OK;
}

ugks_status ugks_batch_step(ugks_batch *b, int32_t nsteps)
{
    return guard([&] {
        if (!b) fail(UGKS_EINVAL, "batch is NULL");
        if (nsteps < 0) fail(UGKS_EINVAL, "nsteps must be >= 0");
        if (nsteps == 0) return;
        if (!b->exec) {
            if (b->prec == UGKS_FP64) batch_capture<double>(b);
            else batch_capture<float>(b);
        }
        // work queued on the cases' own streams comes first, and later calls
        // on a case (moments, state I/O, ugks_step) wait for the batch
        for (size_t i = 0; i < b->cases.size(); ++i) {
            cuda_ok(cudaEventRecord(b->case_ev[i], b->cases[i]->stream), "order");
            cuda_ok(cudaStreamWaitEvent(b->stream, b->case_ev[i], 0), "order");
        }
        for (int32_t s = 0; s < nsteps; ++s) cuda_ok(cudaGraphLaunch(b->exec, b->stream), "graph launch");
        cuda_ok(cudaEventRecord(b->done, b->stream), "order");
        for (auto *c : b->cases) {
            cuda_ok(cudaStreamWaitEvent(c->stream, b->done, 0), "order");
            c->step += nsteps;
            c->stepped = true;
        }
    });
}

void ugks_batch_destroy(ugks_batch *b)
{
    if (!b) return;
    batch_free(b);
    delete b;
}

void ugks_destroy(ugks_case *c)
{
    if (!c) return;
    for (auto e : c->prof_ev) cudaEventDestroy(e);
    c->prof_ev.clear();
    c->release();
    delete c;
}

}  // extern "C"
