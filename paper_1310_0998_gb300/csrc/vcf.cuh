// Velocity correlation of agents (Sec. 5.3, Eqs. VCF, spatial01) in two and
// three dimensions: sums of v_a . v_b and pair counts over the agent pairs
// a < b by shell floor(r / dr) of their separation, and the means of v and |v|^2.
//
// The FP64 pipe of this part is one lane wide (32 cycles per warp instruction)
// and its shared-memory FP64 add is a compare-and-swap loop, so the pass does
// its arithmetic in FP32 and whole numbers:
//   separation  from FP32 offsets inside the cells (or from the 32-bit centres
//               of mass where no cells are used).  A pair whose r / dr lies
//               within `mg` of a shell edge or of r_max, `mg` being above the
//               FP32 error, is queued, and full warps of queued pairs take the
//               FP64 expressions of the definition: every pair's shell, and
//               hence every count, is that of the FP64 evaluation.
//   products    v = (V + R 2^-32) / k, V and R whole numbers and k a power of
//               two by the fastest agent (2^29 <= |V| < 2^30 there): a component
//               is held to 2^-59 of the fastest speed.  v_a . v_b by 32 x 32 ->
//               64 bit products in units k^-2, rounded once and without
//               R_a . R_b: good to 2^-55 of the largest |v|^2.  Where the
//               fastest agent's |v|^2 is no FP32 number, or the mean |v|^2 lies
//               so far below it (256 to 1024 times) that FP64 products would be
//               the better ones, the same pass takes those, with FP64 sums (so do
//               all pairs of more than MANY shells).
//   sums        three 21-bit limbs of a product and the count go to the warp's
//               own histogram in shared memory by native 32-bit integer adds;
//               it is emptied into 64-bit global sums before a word can
//               overflow.  Whole-number sums do not depend on the order.
// A warp takes 32 agents of a cell at a time, one per lane, against the agents of
// a neighbour cell, whose data every lane reads at the same address.
// Bound by instruction issue (58 warp instructions per 32 candidates, half of
// them inside r_max).  1,572,864 agents, r < 16, 64 shells (9.5e8 pairs): 4.5 ms
// against 27.7 with FP64 products and shared FP64 adds (4.0 with FP32 cross terms,
// which left a product good to 2^-49 of the largest |v|^2); a cube of 393,216, r <
// 4: 1.4 against 6.0; all pairs of 1,382 agents (96 shells): 23 us against 410.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <vector>

#include <cuda_runtime.h>

#include "dpd.h"
#include "obs_common.cuh"
#include "sim_host.h"

namespace dpd {
namespace vcf {

using State = ObsState;

template <int D>
struct Agent {
    unsigned long long c[D];   // centre of mass in units L 2^-33
    float sh[D], sl[D];        // v_head + v_tail = sh + sl exactly
};

template <int D>
__device__ __forceinline__ Agent<D> load_agent(const State &s, int k)
{
    const AgentBeads<D> a = load_beads<D>(s, k);
    Agent<D> g;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        g.c[i] = com33(a.hx[i], a.tx[i]);
        const float x = __fadd_rn(a.hv[i], a.tv[i]), bb = __fsub_rn(x, a.hv[i]);
        g.sh[i] = x;
        g.sl[i] = __fadd_rn(__fsub_rn(a.hv[i], __fsub_rn(x, bb)), __fsub_rn(a.tv[i], bb));
    }
    return g;
}

// log2 of the velocity scale k: |v| k < 2^30 (1 + 2^-22) for the largest |v|^2,
// whose FP32 value has the bits v2, and at least 2^29 there.
__device__ __host__ __forceinline__ int scale_log2(uint32_t v2)
{
    const int e = (int)(v2 >> 23) - 127;            // |v|^2 < 2^(e + 1)
    return v2 == 0u ? 0 : 30 - ((e + 2) >> 1);      // |v| < 2^((e + 2) >> 1)
}

// V and R of one component from half the head and tail sum, R to a multiple of 4:
// what sh k / 2 and sl k / 2 leave beside their nearest whole numbers is exact.
__device__ __forceinline__ void split_v(float sh, float sl, float half_k, int &V, int &R)
{
    const float x = __fmul_rn(sh, half_k), z = __fmul_rn(sl, half_k), f = rintf(z);
    const int i = __float2int_rn(x);
    const int r = __float2int_rn(__fmul_rn(__fsub_rn(x, (float)i), 1073741824.0f)) +
                  __float2int_rn(__fmul_rn(__fsub_rn(z, f), 1073741824.0f));
    const int up = (r + (1 << 29)) >> 30;           // r - up 2^30 lies in [-2^29, 2^29)
    V = i + (int)f + up;
    R = (r - up * (1 << 30)) * 4;
}
constexpr long long HALF32 = 1ll << 31;   // rounds a following shift by 32

// Whether the pass takes FP64 products: |v|^2 of the fastest agent (bits v2) zero,
// denormal or infinite, or the mean V^2 below 2^52 (sums: as k_vcf_count's).
template <int D>
__device__ __host__ __forceinline__ bool wide_speeds(uint32_t v2, const long long *sums, int na)
{
    const uint32_t e = v2 >> 23;
    return e == 0u || e == 255u || sums[2 * D + 1] + (sums[2 * D] >> 32) < ((long long)na << 20);
}

template <int D>
__global__ void __launch_bounds__(256) k_vcf_max(State s, unsigned *vmax)
{
    unsigned m = 0u;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < s.na; k += gridDim.x * 256) {
        const Agent<D> g = load_agent<D>(s, k);
        float v2 = 0.f;
#pragma unroll
        for (int i = 0; i < D; ++i) v2 = fmaf(0.5f * g.sh[i], 0.5f * g.sh[i], v2);
        m = max(m, __float_as_uint(v2));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(vmax, m);
}

template <int D>
__device__ __forceinline__ int cell_of(const Agent<D> &g, int n)
{
    int f = 0;
#pragma unroll
    for (int i = D - 1; i >= 0; --i) f = f * n + (int)((g.c[i] * (unsigned long long)n) >> 33);
    return f;
}

// Sums over the agents (sum V, sum R per component; V^2 in two 32-bit halves and
// the rest of |v|^2) and, with cells (n > 0), each agent's rank in its cell.
template <int D>
__global__ void __launch_bounds__(256) k_vcf_count(State s, int n, const unsigned *vmax, unsigned *cnt, unsigned *rank,
                                                   long long *sums)
{
    constexpr int NS = 2 * D + 3;
    const float half_k = __int_as_float((127 + scale_log2(*vmax) - 1) << 23);
    long long a[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) a[i] = 0;
    for (int k = blockIdx.x * 256 + threadIdx.x; k < s.na; k += gridDim.x * 256) {
        const Agent<D> g = load_agent<D>(s, k);
        if (n > 0) rank[k] = atomicAdd(&cnt[cell_of<D>(g, n)], 1u);
        unsigned long long q = 0;
        long long er = HALF32;   // 2^-32
#pragma unroll
        for (int i = 0; i < D; ++i) {
            int V, R;
            split_v(g.sh[i], g.sl[i], half_k, V, R);
            a[2 * i] += V;
            a[2 * i + 1] += R;
            q += (unsigned long long)((long long)V * V);
            er += 2 * (long long)V * R + __mulhi(R, R);
        }
        a[2 * D] += (long long)(q & 0xffffffffull);
        a[2 * D + 1] += (long long)(q >> 32);
        a[2 * D + 2] += er >> 32;
    }
    __shared__ long long red[8][NS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        long long x = a[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[warp][i] = x;
    }
    __syncthreads();
    if (threadIdx.x < NS) {
        long long x = 0;
        for (int w = 0; w < 8; ++w) x += red[w][threadIdx.x];
        atomicAdd((unsigned long long *)&sums[threadIdx.x], (unsigned long long)x);
    }
}

// Agents in cell order (n > 0: offset from the cell's corner in units of dr) or
// as they come (n = 0: 32-bit centre of mass): P, Q = (Vx, Vy, Rx, Ry) or
// (Vx, Vy, Vz, Rz) with R = (Rx, Ry), and the agent's id.  For FP64 products: Q
// (and R) hold v, and wsum gets the sums of v (three) and |v|^2.
template <int D>
__global__ void __launch_bounds__(256) k_vcf_place(State s, int n, float cell_dr, const unsigned *vmax,
                                                   const long long *sums, bool real, const unsigned *start, const unsigned *rank,
                                                   float4 *P, int4 *Q, int2 *R, int *id, double *wsum)
{
    const int k = blockIdx.x * 256 + threadIdx.x;
    const bool wide = real || wide_speeds<D>(*vmax, sums, s.na);
    double w[4] = {0.0, 0.0, 0.0, 0.0};
    if (wide) {
        if (k < s.na) {
            const AgentBeads<D> g = load_beads<D>(s, k);
            for (int i = 0; i < D; ++i) {
                w[i] = __dmul_rn(0.5, __dadd_rn((double)g.hv[i], (double)g.tv[i]));
                w[3] = fma(w[i], w[i], w[3]);
            }
        }
        for (int i = 0; i < 4; ++i) {
            double t = w[i];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if ((threadIdx.x & 31) == 0) atomicAdd(&wsum[i], t);
        }
    }
    if (k >= s.na) return;
    const float half_k = __int_as_float((127 + scale_log2(*vmax) - 1) << 23);
    const Agent<D> g = load_agent<D>(s, k);
    unsigned dst = (unsigned)k;
    if (n > 0) dst = start[cell_of<D>(g, n)] + rank[k];
    if (dst >= (unsigned)s.na) return;
    float p[3] = {0.f, 0.f, 0.f};
    int v[3] = {0, 0, 0}, r[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < D; ++i) {
        if (n > 0) {
            const unsigned long long f = (g.c[i] * (unsigned long long)n) & 0x1ffffffffull;   // offset in the cell, 2^-33
            p[i] = (float)(uint32_t)(f >> 1) * 2.3283064365386963e-10f * cell_dr;
        } else {
            p[i] = __uint_as_float((uint32_t)(g.c[i] >> 1));
        }
        split_v(g.sh[i], g.sl[i], half_k, v[i], r[i]);
    }
    P[dst] = make_float4(p[0], p[1], p[2], 0.f);
    if (wide) {
        reinterpret_cast<double2 *>(Q)[dst] = make_double2(w[0], w[1]);
        if constexpr (D == 3) reinterpret_cast<double *>(R)[dst] = w[2];
    } else if constexpr (D == 2) {
        Q[dst] = make_int4(v[0], v[1], r[0], r[1]);
    } else {
        Q[dst] = make_int4(v[0], v[1], v[2], r[2]);
        R[dst] = make_int2(r[0], r[1]);
    }
    id[dst] = k;
}

// Exclusive scan of n counts in one block, 4096 coalesced counts a turn.
static __global__ void __launch_bounds__(1024) k_vcf_scan(const unsigned *cnt, int n, unsigned *start)
{
    __shared__ unsigned s_w[32];
    __shared__ unsigned s_carry;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) s_carry = 0u;
    for (int b = 0; b < n; b += 4096) {
        unsigned c[4], sum = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = b + 4 * t + i;
            c[i] = k < n ? cnt[k] : 0u;
            sum += c[i];
        }
        unsigned incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const unsigned w = s_w[lane];
            unsigned wi = w;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += v;
            }
            s_w[lane] = wi - w + s_carry;
            __syncwarp();
            if (lane == 31) s_carry += wi;
        }
        __syncthreads();
        unsigned run = s_w[warp] + incl - sum;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = b + 4 * t + i;
            if (k < n) start[k] = run;
            run += c[i];
        }
        __syncthreads();
    }
    if (t == 0) start[n] = s_carry;
}

// What the pair passes share.
struct Pass {
    State s;
    const float4 *P;
    const int4 *Q;
    const int2 *R;
    const int *id;
    double dr;
    int nbins;
    const unsigned *vmax;      // what wide_speeds takes
    const long long *sums;
    bool real;                 // FP64 products whatever the speeds
    float lim2, mg;            // (nbins + mg)^2, and the distance from a shell edge that FP32 decides
    long long *gsum;           // [3][nbins] limb sums (FP64 products: [nbins] doubles)
    unsigned long long *gcnt;  // [nbins]
};

constexpr int LIMB = 21;        // a histogram word takes 2^11 adds of a limb (the high one: of 2^18 in magnitude)
constexpr int QUEUE = 160;
// Candidates (32 adds each at most) until the counts are looked at again, where
// the largest is `most`; fewer than 32 pairs wait in the queue.
__device__ __forceinline__ int room_after(int most) { return ((1 << 11) - 32 - most) / 32 & ~3; }
constexpr int FULL_AT = 992;    // count from which the histogram is emptied at a look: room for 60 then, for 32 below

// WIDE: FP64 products and sums; the histogram is nbins doubles, and the counts where
// they are otherwise.  SHARED (and WIDE): the block's warps add to one histogram,
// nbins doubles and nbins counts, which the block clears and empties.
template <int D, bool WIDE, bool SHARED>
struct Warp {
    const Pass &p;
    int *h;            // [4][nbins]: low, middle, high limb, count (this warp's)
    uint2 *q;          // queued pairs near a shell edge (QUEUE: 31 and four candidates of 32 lanes)
    int qn, lane;
    int a;             // the lane's agent, -1 for none
    int room;          // candidates until the next look at the counts
    float x[D];
    struct Whole { int V[D], R[D]; };
    struct Real { double v[D]; };
    using Vel = std::conditional_t<WIDE, Real, Whole>;
    Vel va;

    __device__ Warp(const Pass &pass, int *hist, uint2 *queue)
        : p(pass), h(hist), q(queue), qn(0), lane(threadIdx.x & 31), a(-1), room(room_after(0))
    {
        if (!SHARED)
            for (int i = lane; i < 4 * p.nbins; i += 32) h[i] = 0;
        __syncwarp();
    }
    __device__ __forceinline__ Vel vel(int b) const
    {
        Vel v;
        if constexpr (WIDE) {
            const double2 q = reinterpret_cast<const double2 *>(p.Q)[b];
            v.v[0] = q.x;
            v.v[1] = q.y;
            if constexpr (D == 3) v.v[2] = reinterpret_cast<const double *>(p.R)[b];
            return v;
        } else {
            const int4 q = p.Q[b];
            v.V[0] = q.x;
            v.V[1] = q.y;
            if constexpr (D == 2) {
                v.R[0] = q.z;
                v.R[1] = q.w;
            } else {
                const int2 r = p.R[b];
                v.V[2] = q.z;
                v.R[0] = r.x;
                v.R[1] = r.y;
                v.R[2] = q.w;
            }
            return v;
        }
    }
    __device__ __forceinline__ void load(int k, int end)
    {
        a = k < end ? k : -1;
        const float4 P = p.P[max(a, 0)];
        const float px[3] = {P.x, P.y, P.z};
        va = vel(max(a, 0));
#pragma unroll
        for (int i = 0; i < D; ++i) x[i] = px[i];
    }
    __device__ __forceinline__ void add(int bin, double d)
    {
        atomicAdd(reinterpret_cast<double *>(h) + bin, d);
        atomicAdd(h + (SHARED ? 2 : 3) * p.nbins + bin, 1);
    }
    __device__ __forceinline__ void add(int bin, long long d)
    {
        int *w = h + bin;
        atomicAdd(w, (int)(d & ((1 << LIMB) - 1)));
        atomicAdd(w + p.nbins, (int)((d >> LIMB) & ((1 << LIMB) - 1)));
        atomicAdd(w + 2 * p.nbins, (int)(d >> (2 * LIMB)));
        atomicAdd(w + 3 * p.nbins, 1);
    }
    // v . w in units k^-2: the whole parts' product, and the cross terms (below
    // 2^63: |V| < 2^30 and |R| <= 3^1/2 2^31) rounded.
    static __device__ __forceinline__ double dot(const Real &v, const Real &w)
    {
        double d = __dadd_rn(__dmul_rn(v.v[0], w.v[0]), __dmul_rn(v.v[1], w.v[1]));
        if constexpr (D == 3) d = __dadd_rn(d, __dmul_rn(v.v[2], w.v[2]));
        return d;
    }
    static __device__ __forceinline__ long long dot(const Whole &v, const Whole &w)
    {
        long long d = 0, c = HALF32;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            d += (long long)v.V[i] * w.V[i];
            c += (long long)v.V[i] * w.R[i];
            c += (long long)v.R[i] * w.V[i];
        }
        return d + (c >> 32);
    }
    __device__ __forceinline__ void com(int id, double *c) const
    {
        const AgentBeads<D> g = load_beads<D>(p.s, id);
        for (int i = 0; i < D; ++i) c[i] = com_d(g.hx[i], g.tx[i], p.s.L, p.s.ulen);
    }
    // The last queued pairs (up to 32 of them) by the FP64 definition of their shell.
    __device__ __forceinline__ void drain()
    {
        __syncwarp();
        const int first = max(qn - 32, 0);
        if (first + lane < qn) {
            const uint2 e = q[first + lane];
            double ca[3], cb[3], d[3];
            com(p.id[e.x], ca);
            com(p.id[e.y], cb);
            const double hL = 0.5 * p.s.L;
            for (int i = 0; i < D; ++i) {
                d[i] = __dsub_rn(ca[i], cb[i]);
                d[i] = d[i] > hL ? __dsub_rn(d[i], p.s.L) : (d[i] < -hL ? __dadd_rn(d[i], p.s.L) : d[i]);
            }
            double r2 = __dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1]));
            if constexpr (D == 3) r2 = __dadd_rn(r2, __dmul_rn(d[2], d[2]));
            const double rmax2 = (double)p.nbins * p.dr * (double)p.nbins * p.dr * (1.0 + 1e-9);
            const double bf = floor(__ddiv_rn(sqrt(r2), p.dr));
            if (r2 < rmax2 && bf < (double)p.nbins) {
                add((int)bf, dot(vel((int)e.x), vel((int)e.y)));
            }
        }
        qn = first;
        __syncwarp();
    }
    __device__ __forceinline__ void flush()
    {
        __syncwarp();
        const int nb = p.nbins;
        for (int b = lane; b < nb; b += 32) {
            const int c = h[3 * nb + b];
            if (c == 0) continue;
            if constexpr (WIDE) {
                double *sum = reinterpret_cast<double *>(h) + b;
                atomicAdd(reinterpret_cast<double *>(p.gsum) + b, *sum);
                *sum = 0.0;
            } else {
                for (int w = 0; w < 3; ++w) {
                    // the low two limbs are never negative and fill their words to 2^32
                    const long long x = w < 2 ? (long long)(unsigned)h[w * nb + b] : (long long)h[w * nb + b];
                    atomicAdd((unsigned long long *)&p.gsum[w * nb + b], (unsigned long long)x);
                    h[w * nb + b] = 0;
                }
            }
            atomicAdd(&p.gcnt[b], (unsigned long long)c);
            h[3 * nb + b] = 0;
        }
        __syncwarp();
    }
    // The lane's agent, seen from `sh` (cells: the neighbour cell's corner; none:
    // ALL), against the agents [s, e) after `after`.
    template <bool ALL>
    __device__ __forceinline__ void run(int s, int e, const float *sh, int after, float unit)
    {
        constexpr float M = 12582912.0f;   // 1.5 2^23: adding it rounds to a whole number in the low bits
        float y[D];
        uint32_t X[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            y[i] = ALL ? 0.f : x[i] - sh[i];
            X[i] = __float_as_uint(x[i]);
        }
        const float lim2 = a >= 0 ? p.lim2 : -1.0f, inside = 0.5f - p.mg, last = (float)p.nbins - p.mg;
        while (s < e) {
            const int stop = SHARED ? e : min(e, s + room);
            if (!SHARED) room -= (stop - s + 3) & ~3;
            for (; s < stop; s += 4) {
                unsigned near = 0u;   // candidates whose shell FP32 does not decide
                float t2[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 P = p.P[min(s + u, stop - 1)];
                    const float px[3] = {P.x, P.y, P.z};
                    t2[u] = 0.f;
#pragma unroll
                    for (int i = 0; i < D; ++i) {
                        // whole-number difference: the periodic image nearest by wrapping
                        const float dd = ALL ? (float)(int)(X[i] - __float_as_uint(px[i])) * unit : y[i] - px[i];
                        t2[u] = fmaf(dd, dd, t2[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int b = s + u;
                    if ((b < stop) & (t2[u] < lim2) & (b > after)) {
                        float t;
                        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(t2[u]));
                        // the shell's middle nearest to t
                        const float w = t - 0.5f, z = w + M;
                        if ((fabsf(w - (z - M)) < inside) & (t < last)) add(__float_as_int(z) - 0x4B400000, dot(va, vel(b)));
                        else near |= 1u << u;
                    }
                }
                if (__any_sync(0xffffffffu, near != 0u)) {
#pragma unroll 1
                    for (int u = 0; u < 4; ++u) {
                        const bool on = (near >> u) & 1u;
                        const unsigned m = __ballot_sync(0xffffffffu, on);
                        if (on) q[qn + __popc(m & ((1u << lane) - 1u))] = make_uint2((unsigned)a, (unsigned)(s + u));
                        qn += __popc(m);
                    }
                    while (qn >= 32) drain();
                }
            }
            if (SHARED || room > 0) continue;
            __syncwarp();
            int most = 0;
            for (int b = lane; b < p.nbins; b += 32) most = max(most, h[3 * p.nbins + b]);
            most = __reduce_max_sync(0xffffffffu, most);
            if (most >= FULL_AT) {
                flush();
                most = 0;
            }
            room = room_after(most);
        }
    }
    __device__ __forceinline__ void finish()
    {
        while (qn > 0) drain();
        if (!SHARED) flush();
    }
};

__host__ __device__ inline size_t warp_smem(int nbins) { return (size_t)nbins * 16 + QUEUE * sizeof(uint2); }

// Cells: task (cell, row of neighbour cells, one of `parts` shares of the cell's
// agents), rows 0 .. of the forward half stencil of m cells each way (row 0: the own
// cell and those east of it), taken from a counter.
template <int D, bool WIDE>
__device__ __forceinline__ void cells_pass(const Pass &p, const unsigned *start, int n, int m, int rows, int parts, int tasks,
                                           float cell_dr, unsigned *next)
{
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *mine = smem + warp_smem(p.nbins) * (threadIdx.x >> 5);
    Warp<D, WIDE, false> w(p, (int *)(mine + QUEUE * sizeof(uint2)), (uint2 *)mine);
    while (true) {
        unsigned t = 0;
        if (w.lane == 0) t = atomicAdd(next, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= (unsigned)tasks) break;
        const int u = (int)t / parts, part = (int)t - u * parts, cell = u / rows, row = u - cell * rows;
        int c[3] = {cell % n, (cell / n) % n, D == 3 ? cell / (n * n) : 0};
        // row r > 0: forward rows in (dz, dy) order after (0, 0)
        int dy = row, dz = 0;
        if (D == 3 && row > m) {
            dz = 1 + (row - m - 1) / (2 * m + 1);
            dy = (row - m - 1) % (2 * m + 1) - m;
        }
        const int yy = c[1] + dy, zz = c[2] + dz;
        const int ny = yy < 0 ? yy + n : (yy >= n ? yy - n : yy), nz = zz >= n ? zz - n : zz;
        const int a0 = (int)start[cell], a1 = (int)start[cell + 1];
        for (int g = a0 + 32 * part; g < a1; g += 32 * parts) {
            w.load(g + w.lane, a1);
            for (int dx = row == 0 ? 0 : -m; dx <= m; ++dx) {
                const int xx = c[0] + dx, nx = xx < 0 ? xx + n : (xx >= n ? xx - n : xx);
                const int nb = (nz * n + ny) * n + nx;
                const float sh[3] = {dx * cell_dr, dy * cell_dr, dz * cell_dr};
                w.template run<false>((int)start[nb], (int)start[nb + 1], sh, row == 0 && dx == 0 ? w.a : -1, 0.f);
            }
        }
    }
    w.finish();
}
template <int D>
__device__ __noinline__ void cells_pass_wide(const Pass &p, const unsigned *start, int n, int m, int rows, int parts, int tasks,
                                             float cell_dr, unsigned *next)
{
    cells_pass<D, true>(p, start, n, m, rows, parts, tasks, cell_dr, next);
}
template <int D>
__global__ void __launch_bounds__(128) k_vcf_cells(const __grid_constant__ Pass p, const unsigned *start, int n, int m,
                                                   int rows, int parts, int tasks, float cell_dr, unsigned *next)
{
    if (wide_speeds<D>(*p.vmax, p.sums, p.s.na)) cells_pass_wide<D>(p, start, n, m, rows, parts, tasks, cell_dr, next);
    else cells_pass<D, false>(p, start, n, m, rows, parts, tasks, cell_dr, next);
}

// All pairs: a warp's 32 agents against a stretch of `cols` agents after them.
template <int D>
__device__ __forceinline__ void all_pass(const Pass &p, int cols, float unit)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int a0 = ((int)blockIdx.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5)) * 32;
    const int s = max(a0, (int)blockIdx.y * cols), e = min(p.s.na, ((int)blockIdx.y + 1) * cols);
    if (a0 >= p.s.na || s >= e) return;   // a whole warp at a time; no block barrier below
    unsigned char *mine = smem + warp_smem(p.nbins) * (threadIdx.x >> 5);
    Warp<D, false, false> w(p, (int *)(mine + QUEUE * sizeof(uint2)), (uint2 *)mine);
    w.load(a0 + w.lane, p.s.na);
    w.template run<true>(s, e, nullptr, w.a, unit);
    w.finish();
}
// The same with FP64 products: one histogram per block (its shared FP64 adds are
// compare-and-swap loops, which wait more than they collide), 12 bytes a shell.
__host__ __device__ inline size_t block_smem(int nbins, int warps) { return (size_t)nbins * 12 + warps * QUEUE * sizeof(uint2); }
template <int D>
__device__ __noinline__ void all_pass_wide(const Pass &p, int cols, float unit)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warps = (int)(blockDim.x >> 5), warp = (int)(threadIdx.x >> 5), nb = p.nbins;
    const int b0 = (int)blockIdx.x * warps * 32, a0 = b0 + 32 * warp, c0 = (int)blockIdx.y * cols;
    const int e = min(p.s.na, c0 + cols);
    if (b0 >= p.s.na || max(b0, c0) >= e) return;   // the whole block
    int *h = (int *)(smem + warps * QUEUE * sizeof(uint2));
    for (int i = threadIdx.x; i < 3 * nb; i += blockDim.x) h[i] = 0;
    __syncthreads();
    if (a0 < p.s.na && max(a0, c0) < e) {
        Warp<D, true, true> w(p, h, (uint2 *)smem + warp * QUEUE);
        w.load(a0 + w.lane, p.s.na);
        w.template run<true>(max(a0, c0), e, nullptr, w.a, unit);
        w.finish();
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        if (h[2 * nb + b] == 0) continue;
        atomicAdd(reinterpret_cast<double *>(p.gsum) + b, reinterpret_cast<const double *>(h)[b]);
        atomicAdd(&p.gcnt[b], (unsigned long long)(unsigned)h[2 * nb + b]);
    }
}
template <int D>
__global__ void __launch_bounds__(128) k_vcf_all(const __grid_constant__ Pass p, int cols, float unit)
{
    if (p.real || wide_speeds<D>(*p.vmax, p.sums, p.s.na)) all_pass_wide<D>(p, cols, unit);
    else all_pass<D>(p, cols, unit);
}

// All pairs of more shells than this take FP64 products: a warp's whole-number
// histogram of 8,192 shells leaves one warp to an SM (60,000 agents: 157 ms against 32
// with a block's FP64 one).  Up to here the sums that no order changes are kept, at
// 44 ms against 22 for 4,096 shells; below 2,500 they are the faster ones too (18
// against 21 for 2,048, 9 against 20 for 1,024).
constexpr int MANY = 4096;

// Host results of a pass.
struct Out {
    std::vector<double> num;
    std::vector<unsigned long long> cnt;
    double mean[3], v2;
};

// Scratch of a pass: fixed offsets for na agents, nbins shells, ncell cells.
struct Layout {
    size_t P, Q, R, id, rank, cnt, start, zero, words, bytes;   // [zero, bytes): cleared words
    Layout(size_t na, size_t nbins, size_t ncell)
    {
        auto up = [](size_t o) { return (o + 255) & ~size_t(255); };
        P = 0;
        Q = up(P + 16 * na);
        R = up(Q + 16 * na);
        id = up(R + 8 * na);
        rank = up(id + 4 * na);
        start = up(rank + (ncell ? 4 * na : 0));
        zero = up(start + 4 * (ncell + 1));
        words = zero;                    // [0] vmax, [1] task counter, 16 whole-number sums, 4 FP64 ones, the shell sums
        cnt = up(gsum() + 8 * 4 * nbins);   // cell counts
        bytes = cnt + 4 * ncell;
    }
    size_t sums() const { return words + 64; }
    size_t wsum() const { return words + 192; }
    size_t gsum() const { return words + 256; }
};
// 64-bit words of a pass's results (from Layout::words on).
static inline size_t result_words(int nbins) { return 32 + 4 * (size_t)nbins; }

#define VCF_CU(x)                                                                   \
    do {                                                                            \
        const cudaError_t e_ = (x);                                                 \
        if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? DPD_ERR_OOM : DPD_ERR_CUDA; \
    } while (0)

// Cells per r_max (m) and per side (n) for a box with room for n1 >= 3 cells of
// side r_max: half cells where they still hold warps of agents (candidates
// inside r_max: half instead of a third of them in two dimensions).  Where more
// than `limit` of them fit a side, wider cells of about two agents each: 20,000
// agents on 2048 x 2048 cells spent 7.0 of 7.1 ms in the scan of the counts
// (5.2 ms as all pairs).
template <int D>
static void cells_for(double L, double rmax, int na, int limit, int *m, int *n)
{
    if (L / rmax >= limit + 1.0) {
        *m = 1;
        *n = std::min(std::max((int)std::pow(0.5 * na, 1.0 / D), 3), limit);
        return;
    }
    const int n1 = (int)std::floor(L / rmax), n2 = (int)std::floor(2.0 * L / rmax);
    const bool half = n2 <= limit && na / std::pow((double)n2, D) >= 48.0;
    *m = half ? 2 : 1;
    *n = half ? n2 : n1;
}

template <int D>
static size_t cells_of(int n) { return D == 2 ? (size_t)n * n : (size_t)n * n * n; }

// One pass on `st`; buf holds Layout(na, nbins, n^D).bytes.  n = 0: all pairs.
// Asynchronous; *res: the result words on the device, from which (copied to the
// host) vcf_finish makes Out.
template <int D>
static int vcf_run(const State &s, double dr, int nbins, int m, int n, char *buf, cudaStream_t st, const void **res)
{
    const size_t ncell = cells_of<D>(n);
    const Layout l((size_t)s.na, (size_t)nbins, ncell);
    unsigned *vmax = (unsigned *)(buf + l.words), *next = vmax + 1;
    long long *sums = (long long *)(buf + l.sums());
    Pass p;
    p.s = s;
    p.P = (const float4 *)(buf + l.P);
    p.Q = (const int4 *)(buf + l.Q);
    p.R = (const int2 *)(buf + l.R);
    p.id = (const int *)(buf + l.id);
    p.dr = dr;
    p.nbins = nbins;
    p.real = n == 0 && nbins > MANY;
    p.vmax = vmax;
    p.sums = sums;
    // FP32 error of r / dr in half-ulps u = 2^-24.  Cells of side c (in dr): a
    // component has 2 c u from each offset, (m + 1) c u from the shift and
    // 2 nbins u from the difference and c's own rounding (m = 2: c is below 0.6
    // nbins), the square and its root 4 nbins u: in all below 22 u max(nbins,
    // 0.75 c).  Cells are wider than r_max where r_max is small beside the
    // box.  All pairs: the centres' 32 bits on top of three half-ulps.
    const double side = n > 0 ? s.L / n / dr : 0.0;
    p.mg = (float)(std::max((double)nbins, 0.75 * side) * 2e-6 + 2e-6 + (n > 0 ? 0.0 : s.L / dr * std::ldexp(1.0, -31)));
    p.lim2 = ((float)nbins + p.mg) * ((float)nbins + p.mg) * 1.000001f;
    p.gsum = (long long *)(buf + l.gsum());
    p.gcnt = (unsigned long long *)(p.gsum + 3 * (size_t)nbins);
    VCF_CU(cudaMemsetAsync(buf + l.zero, 0, l.bytes - l.zero, st));
    int dev = 0, nsm = 0;
    VCF_CU(cudaGetDevice(&dev));
    VCF_CU(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int g = std::min((s.na + 255) / 256, 8 * nsm), gp = (s.na + 255) / 256;
    const float cell_dr = n > 0 ? (float)(s.L / n / dr) : 0.f;
    unsigned *cnt = (unsigned *)(buf + l.cnt), *rank = (unsigned *)(buf + l.rank), *start = (unsigned *)(buf + l.start);
    k_vcf_max<D><<<g, 256, 0, st>>>(s, vmax);
    k_vcf_count<D><<<g, 256, 0, st>>>(s, n, vmax, cnt, rank, sums);
    if (n > 0) k_vcf_scan<<<1, 1024, 0, st>>>(cnt, (int)ncell, start);
    k_vcf_place<D><<<gp, 256, 0, st>>>(s, n, cell_dr, vmax, sums, p.real, start, rank, (float4 *)p.P, (int4 *)p.Q, (int2 *)p.R, (int *)p.id,
                                     (double *)(buf + l.wsum()));
    // warps per block: four, or one where the histograms are large.  The kernels'
    // limit on shared memory is the process's: it is always set to the largest, so
    // that no thread's call lowers it for another's.
    int wpb = warp_smem(nbins) * 4 <= 96 * 1024 ? 4 : 1;
    size_t sm = warp_smem(nbins) * wpb;
    if (n > 0) {
        VCF_CU(cudaFuncSetAttribute(k_vcf_cells<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dynamic_smem()));
        const int rows = D == 2 ? m + 1 : m + 1 + m * (2 * m + 1);
        int occ = 0;
        VCF_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_vcf_cells<D>, 32 * wpb, sm));
        // few cells: a cell's agents by shares of 32, for 24 warps an SM (400,000
        // agents in 16 cells, 64 shells: 0.12 s against 2.29; 60,000 in 400 cells,
        // 512 shells: 0.33 ms against 0.89)
        const long long each = (s.na / (long long)ncell + 31) / 32, want = 24ll * nsm / ((long long)ncell * rows);
        const int parts = (int)std::max<long long>(std::min(each, want), 1);
        const long long tasks = (long long)ncell * rows * parts;
        const long long blocks = std::min<long long>((tasks + wpb - 1) / wpb, (long long)nsm * std::max(occ, 1));
        if (tasks > 2000000000ll) return DPD_ERR_INVALID_ARG;
        k_vcf_cells<D><<<(unsigned)blocks, 32 * wpb, sm, st>>>(p, start, n, m, rows, parts, (int)tasks, cell_dr, next);
    } else {
        VCF_CU(cudaFuncSetAttribute(k_vcf_all<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dynamic_smem()));
        if (p.real) {
            wpb = 4;
            sm = block_smem(nbins, wpb);
        }
        // stretches long enough that emptying the histograms does not matter,
        // short enough for a few thousand warps
        const long long tiles = (s.na + 31) / 32;
        long long cols = tiles * s.na / 2 / (32ll * nsm) / 32 * 32;
        cols = std::min<long long>(std::max<long long>(cols, 32), 1 << 20);
        while ((s.na + cols - 1) / cols > 65535) cols *= 2;
        const dim3 grid((unsigned)((tiles + wpb - 1) / wpb), (unsigned)((s.na + cols - 1) / cols));
        k_vcf_all<D><<<grid, 32 * wpb, sm, st>>>(p, (int)cols, (float)(std::ldexp(s.L, -32) / dr));
    }
    VCF_CU(cudaGetLastError());
    *res = buf + l.words;
    return DPD_OK;
}

template <int D>
static Out vcf_finish(const std::vector<long long> &host, int na, int nbins, int n)
{
    Out o;
    const uint32_t vmax = (uint32_t)((unsigned long long)host[0] & 0xffffffffull);
    const int k = scale_log2(vmax);
    const long long *s = host.data() + 8, *g = host.data() + 32;
    o.num.resize(nbins);
    o.cnt.resize(nbins);
    for (int b = 0; b < nbins; ++b) o.cnt[b] = (unsigned long long)g[3 * nbins + b];
    if ((n == 0 && nbins > MANY) || wide_speeds<D>(vmax, s, na)) {
        double w[4];
        std::memcpy(w, host.data() + 24, sizeof w);
        for (int i = 0; i < 3; ++i) o.mean[i] = w[i] / na;
        o.v2 = w[3] / na;
        std::memcpy(o.num.data(), g, 8 * (size_t)nbins);
        return o;
    }
    for (int i = 0; i < 3; ++i)
        o.mean[i] = i < D ? std::ldexp((double)s[2 * i] + std::ldexp((double)s[2 * i + 1], -32), -k) / na : 0.0;
    const __int128 q = ((__int128)s[2 * D + 1] << 32) + s[2 * D] + s[2 * D + 2];
    o.v2 = std::ldexp((double)q, -2 * k) / na;
    const double unit = std::ldexp(1.0, -2 * k);   // (a power of two: exact)
    for (int b = 0; b < nbins; ++b) {
        const long long hi = g[2 * nbins + b], mid = g[nbins + b], lo = g[b];
        if (o.cnt[b] < 2048 && hi > -(1ll << 19) && hi < 1ll << 19) o.num[b] = (double)(hi * (1ll << (2 * LIMB)) + (mid << LIMB) + lo) * unit;
        else o.num[b] = (double)(((__int128)hi << (2 * LIMB)) + ((__int128)mid << LIMB) + lo) * unit;
    }
    return o;
}

// g, L_int, num, cnt of Eqs. (VCF), (spatial01) from the sums.
static inline void vcf_outputs(const Out &o, double dr, int nbins, double *g, double *L_int, double *num, int64_t *cnt)
{
    const double m2 = o.mean[0] * o.mean[0] + o.mean[1] * o.mean[1] + o.mean[2] * o.mean[2], den = o.v2 - m2;
    double li = 0.0, rprev = 0.0, gprev = 1.0;
    for (int k = 0; k < nbins; ++k) {
        if (o.cnt[k] > 0 && den > 0) {
            g[k] = (o.num[k] / (double)o.cnt[k] - m2) / den;
            const double r = (k + 0.5) * dr;
            li += 0.5 * (g[k] + gprev) * (r - rprev);
            rprev = r;
            gprev = g[k];
        } else {
            g[k] = NAN;
        }
        if (num) num[k] = o.num[k];
        if (cnt) cnt[k] = (int64_t)o.cnt[k];
    }
    if (L_int) *L_int = den > 0 ? li : NAN;
}

}  // namespace vcf
}  // namespace dpd
