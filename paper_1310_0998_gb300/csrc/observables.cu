// Observables of Sec. 5.3-5.4 (arXiv:1310.0998) on the device, FP64.
//
//   agent COM     c_k = x_tail + 1/2 minimg(x_head - x_tail), wrapped;
//                 v_k = (v_head + v_tail)/2                       (Sec. 5.3)
//   u_M           square window of side eps around (i + 1/2) L/M, closed,
//                 minimum image; mean COM velocity inside, 0 if empty
//                 (Sec. 5.4, Eq. filterwidth)
//   E(k)          z = u_x + i u_y, Z = FFT2(z); |uhat_x|^2 + |uhat_y|^2 summed
//                 over a shell equals |Z|^2 / (2 M^4) summed over the same
//                 shell, because k -> -k maps each shell onto itself
//                 (Eqs. fourierTrans01, ESPf)
//   g_v, L_gv     pair histogram of COM separations, sums of v_a . v_b
//                 (Eqs. VCF, spatial01)
// Window and bin decisions use the same IEEE double operations, in the same
// order, as a plain evaluation of those definitions (explicit _rn intrinsics,
// no contraction), so they are reproducible bit for bit off the device.
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "dpd.h"
#include "obs_common.cuh"
#include "vcf.cuh"
#include "sim_host.h"

namespace dpd {

struct ObsScratch {
    void *buf = nullptr;
    size_t bytes = 0;
};

// u = window mean, 0 if empty, from the window sums (2 v_x, 2 v_y, count).
__global__ void k_field_finish(const double *sx, const double *sy, const double *cnt, int MM, double2 *z)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= MM) return;
    const double n = cnt[g];
    z[g] = n > 0.0 ? make_double2(0.5 * sx[g] / n, 0.5 * sy[g] / n) : make_double2(0.0, 0.0);
}

// Scalar vorticity of the field, omega = du_y/dx - du_x/dy (Sec. 5.3), by
// second-order central differences on the periodic grid of spacing h.
__global__ void k_vorticity(const double2 *__restrict__ z, int M, double inv2h, double *__restrict__ om)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= M * M) return;
    const int iy = g / M, ix = g - iy * M;
    const int xp = ix + 1 == M ? 0 : ix + 1, xm = ix == 0 ? M - 1 : ix - 1;
    const int yp = iy + 1 == M ? 0 : iy + 1, ym = iy == 0 ? M - 1 : iy - 1;
    const double duy = __dsub_rn(z[(size_t)iy * M + xp].y, z[(size_t)iy * M + xm].y);
    const double dux = __dsub_rn(z[(size_t)yp * M + ix].x, z[(size_t)ym * M + ix].x);
    om[g] = __dsub_rn(__dmul_rn(duy, inv2h), __dmul_rn(dux, inv2h));
}

__global__ void k_shells(const double2 *Z, int M, double scale, double *E)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= M * M) return;
    const int iy = g / M, ix = g - iy * M;
    const int ky = iy < M / 2 ? iy : iy - M, kx = ix < M / 2 ? ix : ix - M;
    const int sh = shell_of(kx * kx + ky * ky);
    if (sh >= 1 && sh <= M / 2) {
        const double2 a = Z[g];
        atomicAdd(&E[sh - 1], (a.x * a.x + a.y * a.y) * scale);
    }
}

// Sum over agents of |v_COM| with v_COM = (v_head + v_tail) / 2, FP64.
__global__ void k_agent_speed(const uint4 *__restrict__ xv, int na, double *acc)
{
    double s = 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < na; k += gridDim.x * blockDim.x) {
        const uint4 h = xv[2 * k], t = xv[2 * k + 1];
        const double vx = __dmul_rn(0.5, __dadd_rn(to_double(__uint_as_float(h.z)), to_double(__uint_as_float(t.z))));
        const double vy = __dmul_rn(0.5, __dadd_rn(to_double(__uint_as_float(h.w)), to_double(__uint_as_float(t.w))));
        s += sqrt(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(acc, s);
}

}  // namespace dpd

using namespace dpd;

static ObsScratch *scratch_of(dpd_ctx *c, size_t bytes)
{
    static_assert(sizeof(void *) == 8, "64-bit only");
    auto *s = reinterpret_cast<ObsScratch *>(c->obs);
    if (!s) {
        s = new ObsScratch();
        c->obs = s;
    }
    if (s->bytes < bytes) {
        if (s->buf) cudaFree(s->buf);
        s->buf = nullptr;
        s->bytes = 0;
        if (cudaMalloc(&s->buf, bytes) != cudaSuccess) return nullptr;
        s->bytes = bytes;
    }
    return s;
}

void dpd_internal_free_obs(dpd_ctx *c)
{
    auto *s = reinterpret_cast<ObsScratch *>(c->obs);
    if (s) {
        if (s->buf) cudaFree(s->buf);
        delete s;
        c->obs = nullptr;
    }
}

#define CUO(x)                                                    \
    do {                                                          \
        const cudaError_t e_ = (x);                               \
        if (e_ != cudaSuccess)                                    \
            return e_ == cudaErrorMemoryAllocation ? DPD_ERR_OOM : DPD_ERR_CUDA; \
    } while (0)

// A result of a few values to the caller and the latched status: through the
// context's page-locked buffer, since a copy to pageable memory waits by itself.
static int small_out(dpd_ctx *c, void *to, const void *from, size_t bytes)
{
    if (bytes > H_PIN_SMALL) {
        CUO(cudaMemcpyAsync(to, from, bytes, cudaMemcpyDeviceToHost, c->st));
        return dpd_internal_latched(c);
    }
    CUO(cudaMemcpyAsync(c->h_pin, from, bytes, cudaMemcpyDeviceToHost, c->st));
    const int rc = dpd_internal_latched(c);
    std::memcpy(to, c->h_pin, bytes);
    return rc;
}

// Field on the device: z [M*M] double2 (u_x, u_y), cnt [M*M], and a tail of
// tail_bytes (cleared) for the caller.  Every sub-buffer starts on a 256-byte
// boundary (z is read as double2, which needs 16; an odd M*M must not shift it).
static int field_device(dpd_ctx *c, int M, double eps, size_t tail_bytes, double2 **z_out, double **cnt_out,
                        char **tail)
{
    const int na = c->d.n / 2;
    const size_t MM = (size_t)M * M;
    auto up = [](size_t o) { return (o + 255) & ~size_t(255); };
    const size_t o_tail = up(24 * MM), o_z = up(o_tail + tail_bytes);
    ObsScratch *s = scratch_of(c, o_z + 16 * MM + 256);
    if (!s) return DPD_ERR_OOM;
    char *b = (char *)s->buf;
    double *sum = (double *)b, *cn = sum + 2 * MM;
    double2 *z = (double2 *)(b + o_z);
    const double L = c->p.L;
    if (eps <= 0.0) eps = L * std::sqrt(10.0 / (double)na);
    CUO(cudaMemsetAsync(b, 0, o_z, c->st));
    deposit<2>(ObsState{c->d.C_xv, nullptr, na, L, c->d.ulen_d}, M, eps, sum, c->st);
    k_field_finish<<<(int)((MM + 255) / 256), 256, 0, c->st>>>(sum, sum + MM, cn, (int)MM, z);
    CUO(cudaGetLastError());
    *z_out = z;
    *cnt_out = cn;
    if (tail) *tail = b + o_tail;
    return DPD_OK;
}

extern "C" {

int dpd_velocity_field(dpd_ctx *c, int M, double eps, double *u, double *n_in)
{
    if (!c || !u || M < 2 || M > 1024) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    if (eps <= 0.0) eps = c->p.L * std::sqrt(10.0 / (double)(c->d.n / 2));
    if (eps / (c->p.L / M) > 56.0) return DPD_ERR_INVALID_ARG;   // window wider than 56 grid points
    double2 *z;
    double *cn;
    int rc = field_device(c, M, eps, 0, &z, &cn, nullptr);
    if (rc) return rc;
    const size_t MM = (size_t)M * M;
    CUO(cudaMemcpyAsync(u, z, 16 * MM, cudaMemcpyDeviceToHost, c->st));
    if (n_in) CUO(cudaMemcpyAsync(n_in, cn, 8 * MM, cudaMemcpyDeviceToHost, c->st));
    return dpd_internal_latched(c);
}

int dpd_energy_spectrum(dpd_ctx *c, int M, double eps, double *E)
{
    if (!c || !E || M < 4 || M > 1024 || (M & (M - 1))) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    if (eps <= 0.0) eps = c->p.L * std::sqrt(10.0 / (double)(c->d.n / 2));
    if (eps / (c->p.L / M) > 56.0) return DPD_ERR_INVALID_ARG;
    double2 *z;
    double *cn;
    char *tail;
    int rc = field_device(c, M, eps, 8 * (size_t)(M / 2), &z, &cn, &tail);
    if (rc) return rc;
    int logM = 0;
    while ((1 << logM) < M) ++logM;
    fft_axis(z, M, logM, 1, M, M, 0, M, c->st);   // rows (along x)
    fft_axis(z, M, logM, M, M, 1, 0, M, c->st);   // columns (along y)
    double *dE = (double *)tail;
    const double M2 = (double)M * (double)M;
    k_shells<<<(M * M + 255) / 256, 256, 0, c->st>>>(z, M, 0.5 / (M2 * M2), dE);
    CUO(cudaGetLastError());
    return small_out(c, E, dE, 8 * (size_t)(M / 2));
}

int dpd_vorticity(dpd_ctx *c, int M, double eps, double *omega)
{
    if (!c || !omega || M < 3 || M > 1024) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const int na = c->d.n / 2;
    if (eps <= 0.0) eps = c->p.L * std::sqrt(10.0 / (double)na);
    if (eps / (c->p.L / M) > 56.0) return DPD_ERR_INVALID_ARG;
    const size_t MM = (size_t)M * M;
    double2 *z;
    double *cn;
    char *tail;
    int rc = field_device(c, M, eps, 8 * MM, &z, &cn, &tail);
    if (rc) return rc;
    double *om = (double *)tail;
    k_vorticity<<<(int)((MM + 255) / 256), 256, 0, c->st>>>(z, M, (double)M / (2.0 * c->p.L), om);
    CUO(cudaGetLastError());
    CUO(cudaMemcpyAsync(omega, om, 8 * MM, cudaMemcpyDeviceToHost, c->st));
    return dpd_internal_latched(c);
}

int dpd_agent_speed(dpd_ctx *c, double *mean_speed)
{
    if (!c || !mean_speed) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const int na = c->d.n / 2;
    ObsScratch *s = scratch_of(c, 256);
    if (!s) return DPD_ERR_OOM;
    double *acc = (double *)s->buf;
    CUO(cudaMemsetAsync(acc, 0, 8, c->st));
    k_agent_speed<<<std::min((na + 255) / 256, 1024), 256, 0, c->st>>>(c->d.C_xv, na, acc);
    CUO(cudaGetLastError());
    double h = 0.0;
    const int rc = small_out(c, &h, acc, 8);
    *mean_speed = h / na;
    return rc;
}

int dpd_velocity_correlation(dpd_ctx *c, double dr, int nbins, double *g, double *L_int, double *num,
                             int64_t *cnt)
{
    if (!c || !g || !(dr > 0) || nbins < 1 || nbins > 8192) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const int na = c->d.n / 2;
    const double L = c->p.L;
    // pairs within r_max = nbins dr only: a cell grid when at least three cells
    // of side r_max fit per side, else all pairs; both give a pair the same shell
    const double rmax = (double)nbins * dr * (1.0 + 1e-9);
    const double ncv_d = std::floor(L / rmax);
    const bool few = ncv_d >= 3.0 && ncv_d <= 2048.0, cells = few || (ncv_d > 2048.0 && nbins <= 2560);
    const long long tiles = (na + 255) / 256;   // limits of the call: shells, and agents where r_max is no cell's side
    if (few ? 64 * (size_t)nbins + 20480 > 200 * 1024
            : 16 * (size_t)nbins + 8192 > 200 * 1024 || tiles * (tiles + 1) / 2 > 2147483647ll)
        return DPD_ERR_INVALID_ARG;
    int m = 0, n = 0;
    if (cells) vcf::cells_for<2>(L, rmax, na, 2048, &m, &n);
    ObsScratch *s = scratch_of(c, vcf::Layout((size_t)na, (size_t)nbins, vcf::cells_of<2>(n)).bytes);
    if (!s) return DPD_ERR_OOM;
    const vcf::State state{c->d.C_xv, nullptr, na, L, c->d.ulen_d};
    std::vector<long long> host(vcf::result_words(nbins));
    const void *res = nullptr;
    int rc = vcf::vcf_run<2>(state, dr, nbins, m, n, (char *)s->buf, c->st, &res);
    if (rc) return rc;
    rc = small_out(c, host.data(), res, 8 * host.size());
    vcf::vcf_outputs(vcf::vcf_finish<2>(host, na, nbins, n), dr, nbins, g, L_int, num, cnt);
    return rc;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// E(k) with no allocation: dpd_energy_spectrum_noalloc.
//
// Which callers cannot allocate, and why.  dpd_energy_spectrum grows a scratch
// buffer with cudaMalloc on first use (and again when a larger M or box comes
// along).  Two kinds of caller cannot accept that in the middle of a run: one
// whose simulation state was sized to fill the device's memory (the largest
// boxes), where the late cudaMalloc fails; and one that samples E(k) every few
// hundred steps from inside a pipelined run, where cudaMalloc / cudaFree
// synchronise the whole device and stall the other streams.  This variant
// keeps its scratch in one fixed static device array instead.
//
// How.  The window sums come straight from the state (k_deposit), so the
// scratch does not grow with the number of agents: per grid point the window
// sums of u_x and u_y, the window count and the complex field (5 doubles), plus
// M/2 shell sums: 2,622,464 bytes at the maximum M = 256.  Larger M is rejected.
//
// What must start at zero.  The three window sums and the shell sums are
// accumulated with atomics; every call clears them (cudaMemsetAsync on the
// caller's stream) before the deposit.  The field is overwritten in full.
//
// Sharing.  There is one array per device, shared by every context on it:
// two calls whose stream work overlaps (two host threads, or two contexts on
// different streams) race on it and return wrong values.  Serialise them.
//
// Set-up.  The first call on a device, made with that device current, looks up
// the array's device address with cudaGetSymbolAddress and keeps it for later
// calls on that device; make that first call before any stream capture.
// ---------------------------------------------------------------------------

namespace {
constexpr int NOALLOC_MAX_M = 256;
constexpr size_t NOALLOC_MAX_GRID = (size_t)NOALLOC_MAX_M * NOALLOC_MAX_M;
constexpr size_t NOALLOC_DOUBLES = 5 * NOALLOC_MAX_GRID + NOALLOC_MAX_M / 2;
constexpr int NOALLOC_MAX_DEVICES = 64;
}  // namespace

static __device__ __align__(256) double g_spectrum_scratch[NOALLOC_DOUBLES];

static double *g_spectrum_scratch_ptr[NOALLOC_MAX_DEVICES];
static std::mutex g_spectrum_scratch_mu;

// Device address of the static scratch on the context's device (set-up on the
// first call per device).  The symbol lookup answers for the current device,
// so that must be the device the context was created on.
static int spectrum_scratch(int ctx_dev, double **out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return DPD_ERR_CUDA;
    if (dev != ctx_dev) return DPD_ERR_INVALID_ARG;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return DPD_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_spectrum_scratch_mu);
    if (!g_spectrum_scratch_ptr[dev]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_spectrum_scratch);
        if (e != cudaSuccess || !p) return DPD_ERR_CUDA;
        g_spectrum_scratch_ptr[dev] = (double *)p;
    }
    *out = g_spectrum_scratch_ptr[dev];
    return DPD_OK;
}

extern "C" int dpd_energy_spectrum_noalloc(dpd_ctx *c, int M, double eps, double *E)
{
    if (!c || !E || M < 4 || M > NOALLOC_MAX_M || (M & (M - 1))) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const int na = c->d.n / 2;
    const double L = c->p.L;
    if (eps <= 0.0) eps = L * std::sqrt(10.0 / (double)na);
    if (eps / (L / M) > 56.0) return DPD_ERR_INVALID_ARG;
    double *scr = nullptr;
    const int rc = spectrum_scratch(c->dev, &scr);
    if (rc) return rc;
    const size_t MM = (size_t)M * M;
    double *sx = scr, *sy = sx + MM, *cn = sy + MM;
    double2 *z = (double2 *)(cn + MM);          // 16-byte aligned: 3 MM doubles, MM even
    double *dE = (double *)(z + MM);
    CUO(cudaMemsetAsync(sx, 0, 8 * MM * 3, c->st));
    CUO(cudaMemsetAsync(dE, 0, 8 * (size_t)(M / 2), c->st));
    deposit<2>(ObsState{c->d.C_xv, nullptr, na, L, c->d.ulen_d}, M, eps, sx, c->st);
    k_field_finish<<<(int)((MM + 255) / 256), 256, 0, c->st>>>(sx, sy, cn, (int)MM, z);
    int logM = 0;
    while ((1 << logM) < M) ++logM;
    fft_axis(z, M, logM, 1, M, M, 0, M, c->st);
    fft_axis(z, M, logM, M, M, 1, 0, M, c->st);
    const double M2 = (double)M * (double)M;
    k_shells<<<(M * M + 255) / 256, 256, 0, c->st>>>(z, M, 0.5 / (M2 * M2), dE);
    CUO(cudaGetLastError());
    return small_out(c, E, dE, 8 * (size_t)(M / 2));
}
