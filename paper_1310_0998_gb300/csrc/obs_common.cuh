// Device pieces shared by the two- and three-dimensional observables
// (Secs. 5.3-5.4 of arXiv:1310.0998): the canonical state, an agent's centre of
// mass, the filter windows that hold it and their sums, and a radix-2 FFT along
// one axis of a complex grid.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace dpd {

static __device__ __forceinline__ double minimg_d(double d, double L)
{
    return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

// Grid indices i whose window [x_i - eps/2, x_i + eps/2] (minimum image,
// x_i = (i + 1/2) dxg) contains coordinate c; at most min(M, maxout) of them.
static __device__ __forceinline__ int window_hits(double c, double L, double dxg, double half, int M, int *out,
                                                  int maxout)
{
    const double lo = (c - half) / dxg - 0.5, hi = (c + half) / dxg - 0.5;
    int i0 = (int)floor(lo) - 1, i1 = (int)ceil(hi) + 1;
    if (i1 - i0 + 1 > M) { i0 = 0; i1 = M - 1; }
    int n = 0;
    for (int ii = i0; ii <= i1 && n < maxout; ++ii) {
        const int i = ((ii % M) + M) % M;
        const double xm = __dmul_rn(__dadd_rn((double)i, 0.5), dxg);
        const double d = minimg_d(__dsub_rn(xm, c), L);
        if (fabs(d) <= half) out[n++] = i;
    }
    return n;
}

// Canonical state in id order; beads 2k and 2k + 1 are agent k.  In two
// dimensions the velocity is in p.z, p.w and v is unused.
struct ObsState {
    const uint4 *p;
    const float4 *v;
    int na;
    double L, ulen;
};

template <int D>
struct AgentBeads {
    uint32_t hx[D], tx[D];   // head and tail position, fixed point
    float hv[D], tv[D];      // and velocity
};

template <int D>
__device__ __forceinline__ AgentBeads<D> load_beads(const ObsState &s, int k)
{
    const uint4 h = s.p[2 * (size_t)k], t = s.p[2 * (size_t)k + 1];
    AgentBeads<D> a;
    a.hx[0] = h.x; a.hx[1] = h.y;
    a.tx[0] = t.x; a.tx[1] = t.y;
    if constexpr (D == 2) {
        a.hv[0] = __uint_as_float(h.z); a.hv[1] = __uint_as_float(h.w);
        a.tv[0] = __uint_as_float(t.z); a.tv[1] = __uint_as_float(t.w);
    } else {
        const float4 u = s.v[2 * (size_t)k], w = s.v[2 * (size_t)k + 1];
        a.hx[2] = h.z;
        a.tx[2] = t.z;
        a.hv[0] = u.x; a.hv[1] = u.y; a.hv[2] = u.z;
        a.tv[0] = w.x; a.tv[1] = w.y; a.tv[2] = w.z;
    }
    return a;
}

// Centre of mass x_tail + minimg(x_head - x_tail) / 2 in units L 2^-33, modulo
// 2^33: exact, since the state is whole numbers of L 2^-32.
__device__ __forceinline__ unsigned long long com33(uint32_t hx, uint32_t tx)
{
    return (2ull * tx + (unsigned long long)(long long)(int)(hx - tx)) & 0x1ffffffffull;
}

// The same in FP64, positions as the doubles X L / 2^32 (the definition's
// operations one by one).
__device__ __forceinline__ double com_d(uint32_t hx, uint32_t tx, double L, double ulen)
{
    const double t = __dmul_rn((double)tx, ulen);
    const double c = __dadd_rn(t, __dmul_rn(0.5, minimg_d(__dsub_rn(__dmul_rn((double)hx, ulen), t), L)));
    return __dsub_rn(c, __dmul_rn(L, floor(__ddiv_rn(c, L))));
}

// float -> double on the integer pipe (the FP64 pipe is one lane wide on this
// part, and conversions run on it); exact.
__device__ __forceinline__ double to_double(float x)
{
    const uint32_t u = __float_as_uint(x), e = (u >> 23) & 255u;
    if (e == 0u || e == 255u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Windows of one axis by whole numbers: grid points (i + 1/2) L/M within half
// of the centre c (2^-33 L), half = H 2^-33 L/M; the first index (it may lie
// outside [0, M): modulo M) and their number, or -1 where an edge is too close
// for the rounding of H, or the windows wrap onto themselves.
__device__ __forceinline__ int window_range(unsigned long long c, int M, long long H, int *first)
{
    constexpr long long ONE = 1ll << 33, NEAR = 1ll << 6;
    const long long u = (long long)(c * (unsigned long long)M) - (ONE >> 1), lo = u - H, hi = u + H;
    const long long a = lo & (ONE - 1), b = hi & (ONE - 1);
    const int i0 = (int)((lo + ONE - 1) >> 33), n = (int)(hi >> 33) - i0 + 1;
    if (a < NEAR || a > ONE - NEAR || b < NEAR || b > ONE - NEAR || n > M) return -1;
    *first = i0;
    return max(n, 0);
}

constexpr int WIN_MAX = 64;   // hits per axis (the callers keep the window below)

// Window sums of agent k by the FP64 definition of its windows.
template <int D>
__device__ __noinline__ void deposit_exact(const ObsState &s, int k, double dxg, double half, int M, double *sum)
{
    constexpr int MAXW = D == 2 ? WIN_MAX : WIN_MAX / 2;
    const AgentBeads<D> g = load_beads<D>(s, k);
    int idx[D][MAXW], n[3] = {1, 1, 1};
    for (int i = 0; i < D; ++i) n[i] = window_hits(com_d(g.hx[i], g.tx[i], s.L, s.ulen), s.L, dxg, half, M, idx[i], MAXW);
    size_t cells = 1;
    for (int i = 0; i < D; ++i) cells *= (size_t)M;
    for (int z = 0; z < n[2]; ++z)
        for (int y = 0; y < n[1]; ++y)
            for (int x = 0; x < n[0]; ++x) {
                size_t at = (size_t)idx[1][y] * M + idx[0][x];
                if constexpr (D == 3) at += (size_t)idx[2][z] * M * M;
                for (int i = 0; i < D; ++i) atomicAdd(&sum[i * cells + at], __dadd_rn((double)g.hv[i], (double)g.tv[i]));
                atomicAdd(&sum[D * cells + at], 1.0);
            }
}

// Window sums per grid point: twice the velocity (head + tail) by component,
// then the count, each M^D values; H as window_range.  With the windows found by FP64
// divisions and roundings this took 593 us (and 194 for the centres) for
// 1,572,864 agents on 128 x 128, 275 (and 80) for 393,216 on 64^3.
// W lanes share an agent's windows (1, or 32 where a window holds many points:
// 1,382 agents of 119 points each 26 us at one lane, 5 at 32).
template <int D, int W>
__global__ void __launch_bounds__(128) k_deposit(ObsState s, double dxg, double half, long long H, int M, double *sum)
{
    // (the threads of 2^27 agents on 32 lanes do not fit in 32 bits)
    const int k = (int)(blockIdx.x * (128 / W) + threadIdx.x / W), lane = threadIdx.x % W;
    if (k >= s.na) return;
    const AgentBeads<D> g = load_beads<D>(s, k);
    int f[3] = {0, 0, 0}, n[3] = {1, 1, 1};
    bool sure = true;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        n[i] = window_range(com33(g.hx[i], g.tx[i]), M, H, &f[i]);
        sure = sure && n[i] >= 0;
        f[i] %= M;
        f[i] += f[i] < 0 ? M : 0;
    }
    if (!sure) {
        if (lane == 0) deposit_exact<D>(s, k, dxg, half, M, sum);
        return;
    }
    if (n[0] == 0 || n[1] == 0 || n[2] == 0) return;
    const size_t cells = D == 2 ? (size_t)M * M : (size_t)M * M * M;
    double v[D];
#pragma unroll
    for (int i = 0; i < D; ++i) v[i] = __dadd_rn(to_double(g.hv[i]), to_double(g.tv[i]));
    auto point = [&](int x, int y, int z) {
        const int ix = f[0] + x >= M ? f[0] + x - M : f[0] + x, iy = f[1] + y >= M ? f[1] + y - M : f[1] + y;
        const int iz = f[2] + z >= M ? f[2] + z - M : f[2] + z;
        double *to = sum + ((size_t)(D == 3 ? iz : 0) * M + iy) * M + ix;
#pragma unroll
        for (int i = 0; i < D; ++i) atomicAdd(to + i * cells, v[i]);
        atomicAdd(to + D * cells, 1.0);
    };
    if constexpr (W == 1) {
        for (int z = 0; z < n[2]; ++z)
            for (int y = 0; y < n[1]; ++y)
                for (int x = 0; x < n[0]; ++x) point(x, y, z);
    } else {
        const int row = n[0], plane = row * n[1];
        for (int p = lane; p < plane * n[2]; p += W) {
            const int z = p / plane, q = p - z * plane, y = q / row;
            point(q - y * row, y, z);
        }
    }
}

// Half a window in the units of window_range (host).
static inline long long window_units(double half, double dxg) { return (long long)llrint(half / dxg * 8589934592.0); }

// Window sums of side eps on the grid of M points an axis into `sum` (cleared).
template <int D>
static inline void deposit(const ObsState &s, int M, double eps, double *sum, cudaStream_t st)
{
    const double dxg = s.L / M, w = eps / dxg, points = D == 2 ? w * w : w * w * w;
    const long long H = window_units(0.5 * eps, dxg);
    if (points < 16.0) k_deposit<D, 1><<<(s.na + 127) / 128, 128, 0, st>>>(s, dxg, 0.5 * eps, H, M, sum);
    else k_deposit<D, 32><<<(unsigned)(((long long)s.na * 32 + 127) / 128), 128, 0, st>>>(s, dxg, 0.5 * eps, H, M, sum);
}

// In-place radix-2 FFT (forward, e^{-2 pi i k n / M}) of lines of M complex
// doubles with stride `stride` between elements.  Line l starts at
// (l / inner) outer_pitch + (l % inner) inner_pitch, so one launch covers every
// line of a 2D grid along either axis, or of a 3D grid along any axis.  A block
// takes lpb neighbouring lines (M/2 threads each) and reads a strided axis
// across them; the M/2 twiddle factors are made once per block (a sine and
// cosine per butterfly was three quarters of the FP64 work: 173 us an axis of
// 64^3 x 2, 19 us an axis of 128 x 128).
static __global__ void __launch_bounds__(512) k_fft(double2 *z, int M, int logM, long long stride, int inner,
                                                    long long inner_pitch, long long outer_pitch, int lpb, int lines)
{
    extern __shared__ double2 s_fft[];
    double2 *tw = s_fft, *s = s_fft + M / 2;
    const int P = M + 1, l0 = blockIdx.x * lpb, nt = blockDim.x, hM = M >> 1, all = lpb << logM;
    for (int p = threadIdx.x; p < hM; p += nt) {
        double sn, cs;
        sincospi(-2.0 * (double)p / (double)M, &sn, &cs);
        tw[p] = make_double2(cs, sn);
    }
    auto at = [&](int t, int &l, int &i) -> double2 * {
        if (stride == 1) { l = t >> logM; i = t & (M - 1); }
        else { l = t % lpb; i = t / lpb; }
        const long long b = l0 + l;
        return z + (b / inner) * outer_pitch + (b % inner) * inner_pitch + (long long)i * stride;
    };
    for (int t = threadIdx.x; t < all; t += nt) {
        int l, i;
        const double2 *p = at(t, l, i);
        if (l0 + l < lines) s[l * P + (__brev(i) >> (32 - logM))] = *p;
    }
    __syncthreads();
    for (int lg = 1; lg <= logM; ++lg) {
        const int half = 1 << (lg - 1);
        for (int t = threadIdx.x; t < all / 2; t += nt) {
            const int l = t >> (logM - 1), b = t & (hM - 1), pos = b & (half - 1);
            double2 *x = s + l * P + ((b >> (lg - 1)) << lg) + pos;
            const double2 w = tw[pos << (logM - lg)], a = x[0], c = x[half];
            const double2 wc = make_double2(c.x * w.x - c.y * w.y, c.x * w.y + c.y * w.x);
            x[0] = make_double2(a.x + wc.x, a.y + wc.y);
            x[half] = make_double2(a.x - wc.x, a.y - wc.y);
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < all; t += nt) {
        int l, i;
        double2 *p = at(t, l, i);
        if (l0 + l < lines) *p = s[l * P + i];
    }
}

// One axis of `lines` lines: several per block where there are many.
static inline void fft_axis(double2 *z, int M, int logM, long long stride, int inner, long long inner_pitch,
                            long long outer_pitch, int lines, cudaStream_t st)
{
    const int lpb = lines <= 1024 ? 1 : M >= 512 ? 1 : 512 / M > 16 ? 16 : 512 / M;
    const int thr = lpb * M / 2 < 32 ? 32 : (lpb * M / 2 > 512 ? 512 : lpb * M / 2);
    const size_t sm = 16 * ((size_t)M / 2 + (size_t)lpb * (M + 1));
    k_fft<<<(lines + lpb - 1) / lpb, thr, sm, st>>>(z, M, logM, stride, inner, inner_pitch, outer_pitch, lpb, lines);
}

// Shell nint|k| of a squared wave number below 2^20: no sqrt of a whole number
// lies within 10^-4 of a half, so FP32 rounds it as FP64 does.
__device__ __forceinline__ int shell_of(int k2) { return (int)rintf(sqrtf((float)k2)); }

}  // namespace dpd
