// Observables of Secs. 5.3-5.4 (arXiv:1310.0998) for the three-dimensional
// variant (include/dpd.h, dpd3_velocity_field / energy_spectrum / vorticity /
// velocity_correlation), FP64 on the device.
//
// The paper defines them in two dimensions; each carries over axis by axis:
//   agent COM     c_k = x_tail + 1/2 minimg(x_head - x_tail), wrapped;
//                 v_k = (v_head + v_tail) / 2
//   u_M           cubic window of side eps around (i + 1/2) L/M per axis,
//                 closed, minimum image; mean COM velocity inside, 0 if empty;
//                 default eps = L (N_f / N)^(1/3), N_f = 10 (the window holds
//                 N_f agents on average, as the square window of Eq.
//                 filterwidth does in two dimensions)
//   E(k)          uhat = M^-3 sum u e^{-2 pi i k.x/L}; E(k) = sum over
//                 nint|k| = k of (|uhat_x|^2 + |uhat_y|^2 + |uhat_z|^2) / 2,
//                 k = 1..M/2.  z1 = u_x + i u_y and z2 = u_z are transformed;
//                 k -> -k maps a shell onto itself, so the shell sum of
//                 |Z1|^2 + |Z2|^2 equals M^6 times that of the three |uhat|^2
//   omega         curl u_M by second-order central differences
//   g_v, L_gv     agent pairs a < b within r_max: bin floor(r / dr) of the
//                 COM separation r = sqrt((dx^2 + dy^2) + dz^2), sums of
//                 v_a . v_b (a cell grid of side >= r_max, or all pairs);
//                 g_v(b) = (<v_a . v_b>_b - |<v>|^2) / (<|v|^2> - |<v>|^2),
//                 L_gv by the trapezoid rule over r = 0 (g = 1) and the
//                 centres of the non-empty bins
// Window and bin decisions use the same IEEE double operations, in the same
// order, as a plain evaluation of those definitions.
#include <cmath>
#include <vector>

#include "dpd.h"
#include "obs_common.cuh"
#include "vcf.cuh"
#include "sim3d_host.h"

namespace dpd {

// u = window mean (0 if empty), stored as z1 = u_x + i u_y and z2 = u_z + 0 i.
__global__ void k3_field_finish(const double *sx, const double *sy, const double *sz, const double *cnt, long long MMM,
                                double2 *z1, double2 *z2)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= MMM) return;
    const double n = cnt[g];
    z1[g] = n > 0.0 ? make_double2(0.5 * sx[g] / n, 0.5 * sy[g] / n) : make_double2(0.0, 0.0);   // the sums hold 2 v
    z2[g] = make_double2(n > 0.0 ? 0.5 * sz[g] / n : 0.0, 0.0);
}

__global__ void k3_field_out(const double2 *z1, const double2 *z2, long long MMM, double *u)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= MMM) return;
    u[3 * g] = z1[g].x;
    u[3 * g + 1] = z1[g].y;
    u[3 * g + 2] = z2[g].x;
}

// omega = curl u by central differences on the periodic grid (spacing h):
// (d u_z/dy - d u_y/dz, d u_x/dz - d u_z/dx, d u_y/dx - d u_x/dy).
__global__ void k3_vorticity(const double2 *__restrict__ z1, const double2 *__restrict__ z2, int M, double inv2h,
                             double *__restrict__ om)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long MM = (long long)M * M;
    if (g >= MM * M) return;
    const int iz = (int)(g / MM), iy = (int)((g / M) % M), ix = (int)(g % M);
    const int xp = ix + 1 == M ? 0 : ix + 1, xm = ix == 0 ? M - 1 : ix - 1;
    const int yp = iy + 1 == M ? 0 : iy + 1, ym = iy == 0 ? M - 1 : iy - 1;
    const int zp = iz + 1 == M ? 0 : iz + 1, zm = iz == 0 ? M - 1 : iz - 1;
    auto at = [&](int z, int y, int x) { return ((long long)z * M + y) * M + x; };
    const double duz_dy = __dsub_rn(z2[at(iz, yp, ix)].x, z2[at(iz, ym, ix)].x);
    const double duy_dz = __dsub_rn(z1[at(zp, iy, ix)].y, z1[at(zm, iy, ix)].y);
    const double dux_dz = __dsub_rn(z1[at(zp, iy, ix)].x, z1[at(zm, iy, ix)].x);
    const double duz_dx = __dsub_rn(z2[at(iz, iy, xp)].x, z2[at(iz, iy, xm)].x);
    const double duy_dx = __dsub_rn(z1[at(iz, iy, xp)].y, z1[at(iz, iy, xm)].y);
    const double dux_dy = __dsub_rn(z1[at(iz, yp, ix)].x, z1[at(iz, ym, ix)].x);
    om[3 * g] = __dsub_rn(__dmul_rn(duz_dy, inv2h), __dmul_rn(duy_dz, inv2h));
    om[3 * g + 1] = __dsub_rn(__dmul_rn(dux_dz, inv2h), __dmul_rn(duz_dx, inv2h));
    om[3 * g + 2] = __dsub_rn(__dmul_rn(duy_dx, inv2h), __dmul_rn(dux_dy, inv2h));
}

// Shell sums of (|Z1|^2 + |Z2|^2) scale, per block in shared memory first.
__global__ void k3_shells(const double2 *Z1, const double2 *Z2, int M, double scale, double *E)
{
    extern __shared__ double es[];
    const int nsh = M / 2;
    for (int i = threadIdx.x; i < nsh; i += blockDim.x) es[i] = 0.0;
    __syncthreads();
    const long long MM = (long long)M * M;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < MM * M;
         g += (long long)gridDim.x * blockDim.x) {
        const int iz = (int)(g / MM), iy = (int)((g / M) % M), ix = (int)(g % M);
        const int kz = iz < M / 2 ? iz : iz - M, ky = iy < M / 2 ? iy : iy - M, kx = ix < M / 2 ? ix : ix - M;
        const int sh = shell_of(kx * kx + ky * ky + kz * kz);
        if (sh >= 1 && sh <= nsh) {
            const double2 a = Z1[g], b = Z2[g];
            atomicAdd(&es[sh - 1], (a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y) * scale);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nsh; i += blockDim.x)
        if (es[i] != 0.0) atomicAdd(&E[i], es[i]);
}

}  // namespace dpd

using namespace dpd;

#define CUO3(x)                                                                     \
    do {                                                                            \
        const cudaError_t e_ = (x);                                                 \
        if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? DPD_ERR_OOM : DPD_ERR_CUDA; \
    } while (0)

static char *scratch3(dpd3_ctx *c, size_t bytes)
{
    if (c->obs_bytes < bytes) {
        if (c->obs) cudaFree(c->obs);
        c->obs = nullptr;
        c->obs_bytes = 0;
        if (cudaMalloc(&c->obs, bytes) != cudaSuccess) return nullptr;
        c->obs_bytes = bytes;
    }
    return (char *)c->obs;
}

static double default_eps3(const dpd3_ctx *c)
{
    return c->p.L * std::cbrt(10.0 / (double)(c->s.b.n / 2));
}

// Field on the device: z1 (u_x + i u_y) and z2 (u_z) [M^3] double2, back to
// back (one FFT launch per axis covers both), cnt [M^3], and a tail of at
// least tail_bytes.  Every sub-buffer starts on a 256-byte boundary.
static int field3_device(dpd3_ctx *c, int M, double eps, size_t tail_bytes, double2 **z_out, double **cnt_out,
                         char **tail)
{
    const int na = c->s.b.n / 2;
    const size_t MMM = (size_t)M * M * M;
    auto up = [](size_t o) { return (o + 255) & ~size_t(255); };
    const size_t o_tail = up(32 * MMM), o_z = up(o_tail + tail_bytes);
    char *b = scratch3(c, o_z + 32 * MMM + 256);
    if (!b) return DPD_ERR_OOM;
    double *sx = (double *)b, *sy = sx + MMM, *sz = sy + MMM, *cn = sz + MMM;
    double2 *z = (double2 *)(b + o_z);
    const double L = c->p.L;
    CUO3(cudaMemsetAsync(b, 0, 32 * MMM, c->st));
    deposit<3>(ObsState{c->s.C_p, c->s.C_v, na, L, c->s.b.ulen_d}, M, eps, sx, c->st);
    k3_field_finish<<<(unsigned)((MMM + 255) / 256), 256, 0, c->st>>>(sx, sy, sz, cn, (long long)MMM, z, z + MMM);
    CUO3(cudaGetLastError());
    *z_out = z;
    *cnt_out = cn;
    if (tail) *tail = b + o_tail;
    return DPD_OK;
}

static int check_field_args(dpd3_ctx *c, int M, double *eps)
{
    if (!c->have_state) return DPD_ERR_STATE;
    if (*eps <= 0.0) *eps = default_eps3(c);
    if (!(*eps / (c->p.L / M) <= 28.0)) return DPD_ERR_INVALID_ARG;   // window wider than 28 grid points
    return DPD_OK;
}

extern "C" {

int dpd3_velocity_field(dpd3_ctx *c, int M, double eps, double *u, double *n_in)
{
    if (!c || !u || M < 2 || M > 256) return DPD_ERR_INVALID_ARG;
    int rc = check_field_args(c, M, &eps);
    if (rc) return rc;
    const size_t MMM = (size_t)M * M * M;
    double2 *z;
    double *cn;
    char *tail;
    rc = field3_device(c, M, eps, 24 * MMM, &z, &cn, &tail);
    if (rc) return rc;
    double *du = (double *)tail;
    k3_field_out<<<(unsigned)((MMM + 255) / 256), 256, 0, c->st>>>(z, z + MMM, (long long)MMM, du);
    CUO3(cudaGetLastError());
    CUO3(cudaMemcpyAsync(u, du, 24 * MMM, cudaMemcpyDeviceToHost, c->st));
    if (n_in) CUO3(cudaMemcpyAsync(n_in, cn, 8 * MMM, cudaMemcpyDeviceToHost, c->st));
    return dpd3_internal_latched(c);
}

int dpd3_energy_spectrum(dpd3_ctx *c, int M, double eps, double *E)
{
    if (!c || !E || M < 4 || M > 256 || (M & (M - 1))) return DPD_ERR_INVALID_ARG;
    int rc = check_field_args(c, M, &eps);
    if (rc) return rc;
    const long long MM = (long long)M * M, MMM = MM * M;
    double2 *z;
    double *cn;
    char *tail;
    rc = field3_device(c, M, eps, 8 * (size_t)(M / 2), &z, &cn, &tail);
    if (rc) return rc;
    int logM = 0;
    while ((1 << logM) < M) ++logM;
    const int lines = (int)(2 * MM);   // M^2 lines per axis in each of z1, z2
    fft_axis(z, M, logM, 1, lines, M, 0, lines, c->st);          // along x
    fft_axis(z, M, logM, M, M, 1, MM, lines, c->st);             // along y
    fft_axis(z, M, logM, MM, (int)MM, 1, MMM, lines, c->st);     // along z
    double *dE = (double *)tail;
    CUO3(cudaMemsetAsync(dE, 0, 8 * (size_t)(M / 2), c->st));
    const double M3 = (double)MMM;
    const long long blocks = std::min<long long>((MMM + 255) / 256, 4096);
    k3_shells<<<(unsigned)blocks, 256, 8 * (size_t)(M / 2), c->st>>>(z, z + MMM, M, 0.5 / (M3 * M3), dE);
    CUO3(cudaGetLastError());
    CUO3(cudaMemcpyAsync(E, dE, 8 * (size_t)(M / 2), cudaMemcpyDeviceToHost, c->st));
    return dpd3_internal_latched(c);
}

int dpd3_vorticity(dpd3_ctx *c, int M, double eps, double *omega)
{
    if (!c || !omega || M < 3 || M > 256) return DPD_ERR_INVALID_ARG;
    int rc = check_field_args(c, M, &eps);
    if (rc) return rc;
    const size_t MMM = (size_t)M * M * M;
    double2 *z;
    double *cn;
    char *tail;
    rc = field3_device(c, M, eps, 24 * MMM, &z, &cn, &tail);
    if (rc) return rc;
    double *om = (double *)tail;
    k3_vorticity<<<(unsigned)((MMM + 255) / 256), 256, 0, c->st>>>(z, z + MMM, M, (double)M / (2.0 * c->p.L), om);
    CUO3(cudaGetLastError());
    CUO3(cudaMemcpyAsync(omega, om, 24 * MMM, cudaMemcpyDeviceToHost, c->st));
    return dpd3_internal_latched(c);
}

int dpd3_velocity_correlation(dpd3_ctx *c, double dr, int nbins, double *g, double *L_int, double *num,
                              int64_t *cnt)
{
    if (!c || !g || !(dr > 0) || nbins < 1 || nbins > 4096) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const int na = c->s.b.n / 2;
    const double L = c->p.L;
    // a cell grid when at least three cells of side r_max fit per side, else all
    // agent pairs; both give a pair the same shell
    const double rmax = (double)nbins * dr * (1.0 + 1e-9);
    const double nv_d = std::floor(L / rmax);
    const bool few = nv_d >= 3.0 && nv_d <= 256.0, cells = few || (nv_d > 256.0 && nbins <= 2560);
    const long long tiles = (na + 255) / 256;   // limits of the call: shells, and agents where r_max is no cell's side
    if (few ? 64 * (size_t)nbins + 20480 > 200 * 1024
            : 16 * (size_t)nbins + 16416 > 200 * 1024 || tiles * (tiles + 1) / 2 > 2147483647ll)
        return DPD_ERR_INVALID_ARG;
    int m = 0, n = 0;
    if (cells) vcf::cells_for<3>(L, rmax, na, 256, &m, &n);
    char *buf = scratch3(c, vcf::Layout((size_t)na, (size_t)nbins, vcf::cells_of<3>(n)).bytes);
    if (!buf) return DPD_ERR_OOM;
    const vcf::State state{c->s.C_p, c->s.C_v, na, L, c->s.b.ulen_d};
    std::vector<long long> host(vcf::result_words(nbins));
    const void *res = nullptr;
    int rc = vcf::vcf_run<3>(state, dr, nbins, m, n, buf, c->st, &res);
    if (rc) return rc;
    CUO3(cudaMemcpyAsync(host.data(), res, 8 * host.size(), cudaMemcpyDeviceToHost, c->st));
    rc = dpd3_internal_latched(c);
    vcf::vcf_outputs(vcf::vcf_finish<3>(host, na, nbins, n), dr, nbins, g, L_int, num, cnt);
    return rc;
}

}  // extern "C"
