// Three-dimensional variant of the simulator (include/dpd.h, dpd3_*).
//
// Sec. 2 states every force as a vector law, so the pair force (Eqs. DPDf,
// DPDcdr, weightFunc01), the bond (Eq. stiffSpring), propulsion and drag
// (Eq. DPDnp) and the velocity-Verlet step of Sec. 5 carry over to a periodic
// cube unchanged; only the geometry is new.  Positions are 32-bit fixed point
// per axis as in two dimensions (uniform resolution, wrap by overflow, exact
// minimum image and cell index).
//
// Layout (N beads, n_c^3 cells numbered (z n_c + y) n_c + x):
//   S    uint4[N][2] (X, Y, Z, id) of the pre-force state and the bits of its
//                   half-step velocity v_{s-1/2} (v_s at set-up), sorted by cell
//   U_p, U_v, U_rank  the next pre-force state in the order of S, with each
//                     bead's rank inside its new cell (atomic ticket)
//   slot u32[N]     id -> sorted slot (the bonded partner of bead id is id^1)
//   counts, cstart  cell populations and their exclusive scan (the same
//                   decoupled look-back scan as the 2D path)
//   C_p, C_v, C_f   canonical (X_s, v_s, f_s) in id order after each call
//   F    s64[N][4]  pair-force sums of the current step by sorted slot, in
//                   fixed point (2^-24 force units per count, as the 2D
//                   path), kept zero between steps
// One step: scan, scatter, pair forces, integration.  The pair kernel gives
// one thread per bead the half stencil (the rest of its cell and the 13
// cells ahead of it, five rows of cells), so every pair inside r_c is
// evaluated once; the pairs go through a warp queue so that their arithmetic
// runs on full warps, the force lands on the owner through shared memory and
// its reaction on the partner through 64-bit integer atomics into F (sorted
// order).  Every sum is in fixed point, so it does not depend on the order in
// which pairs are met and a run is reproducible bit for bit.  The integration kernel reads and
// clears F, adds bond, propulsion and drag, does the second half-kick, the
// FP64 thermo partials, the next half-kick and drift, and bins the new
// position.
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "dpd.h"
#include "launch.cuh"
#include "sim_host.h"
#include "sim3d_host.h"
#include "sim_kernels.cuh"

namespace dpd {


__device__ __forceinline__ int cell3(const Sys &d, uint32_t X, uint32_t Y, uint32_t Z)
{
    return (cell_coord(d, Z) * d.nc + cell_coord(d, Y)) * d.nc + cell_coord(d, X);
}

__global__ void __launch_bounds__(SCAN_NT) k3_scan(Sys d, int nblocks)
{
    __shared__ uint32_t s_buf[SCAN_BUF];
    wait_for_previous();
    scan_decoupled_t<SCAN_NT>(d, nblocks, s_buf);
    let_next_start();
}

__global__ void k3_bin(Sys3 s)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.b.n) return;
    const uint4 p = s.U_p[k];
    s.U_rank[k] = atomicAdd(&s.b.counts[cell3(s.b, p.x, p.y, p.z)], 1u);
}

__global__ void k3_scatter(Sys3 s)
{
    wait_for_previous();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.b.n) return;
    const uint4 p = s.U_p[k];
    const uint32_t dst = s.b.cstart[cell3(s.b, p.x, p.y, p.z)] + s.U_rank[k];
    if (dst >= (uint32_t)s.b.n || p.w >= (uint32_t)s.b.n) {
        set_err_at(s.b, ERR_INTERNAL, 11, k, dst, p.w);
        return;
    }
    const float4 v = s.U_v[k];
    s.S[2 * (size_t)dst] = p;
    s.S[2 * (size_t)dst + 1] = make_uint4(fbits(v.x), fbits(v.y), fbits(v.z), 0u);
    s.slot[p.w] = dst;
    s.S_pos[dst] = make_float4((float)p.x * s.b.ulen, (float)p.y * s.b.ulen, (float)p.z * s.b.ulen, 0.f);
}

// Double positions [N][3] and float velocities [N][3] (id order) -> U.
__global__ void k3_load(Sys3 s, const double *__restrict__ x, const float *__restrict__ v)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.b.n) return;
    uint32_t X[3];
    bool ok = true;
    for (int c = 0; c < 3; ++c) {
        const double u = x[3 * k + c] * s.b.inv_ulen_d;
        if (!(fabs(u) < 4503599627370496.0)) { ok = false; X[c] = 0u; }
        else X[c] = (uint32_t)(unsigned long long)llrint(u);
    }
    float4 vv = make_float4(v[3 * k], v[3 * k + 1], v[3 * k + 2], 0.f);
    if (!isfinite(vv.x) || !isfinite(vv.y) || !isfinite(vv.z)) ok = false;
    if (!ok) {
        set_err(s.b, ERR_NONFINITE);
        vv = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    s.U_p[k] = make_uint4(X[0], X[1], X[2], (uint32_t)k);
    s.U_v[k] = vv;
}

__global__ void k3_store(Sys3 s, double *__restrict__ x, float *__restrict__ v, float *__restrict__ f)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= s.b.n) return;
    const uint4 p = s.C_p[k];
    const float4 vv = s.C_v[k], ff = s.C_f[k];
    x[3 * k] = (double)p.x * s.b.ulen_d;
    x[3 * k + 1] = (double)p.y * s.b.ulen_d;
    x[3 * k + 2] = (double)p.z * s.b.ulen_d;
    v[3 * k] = vv.x; v[3 * k + 1] = vv.y; v[3 * k + 2] = vv.z;
    f[3 * k] = ff.x; f[3 * k + 1] = ff.y; f[3 * k + 2] = ff.z;
}

__global__ void k3_set_step(Sys d, long long s) { *d.step = s; }

// Pair force magnitude along e (as the 2D pair term, with dv.e in 3D).
__device__ __forceinline__ float pair_scalar3(const Sys &d, float r2, float rinv, float dve, uint32_t ia,
                                              uint32_t ib, uint32_t s_lo, uint32_t s_hi)
{
    const float r = r2 * rinv;
    const float w = 1.0f - r * d.inv_rc;
    const float nz = pair_noise(d, ia, ib, s_lo, s_hi);
    if (!d.gen_w) return __fmul_rn(w, __fmaf_rn(d.sig_r, nz, __fmaf_rn(-__fmul_rn(d.gamma, w), dve, d.a)));
    const float wr = __powf(w, d.hwexp);
    return d.a * w - d.gamma * (wr * wr) * dve + d.sig_r * wr * nz;
}

// A sorted bead's 32-byte record in one load (two 16-byte loads of scattered
// beads take twice the wavefronts).
__device__ __forceinline__ void load_bead(const uint4 *S, uint32_t q, uint4 &p, float3 &v)
{
    [[maybe_unused]] uint32_t pad;
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(p.x), "=r"(p.y), "=r"(p.z), "=r"(p.w), "=f"(v.x), "=f"(v.y), "=f"(v.z), "=r"(pad)
                 : "l"(S + 2 * (size_t)q));
}

// One queued pair (sorted slot q, owner lane o of this warp): the pair force
// on the owner, accumulated in shared memory ((hi, lo) words per component,
// as the 2D tile); its reaction on q comes back in r (Newton-3: every pair is
// evaluated once).  False: no force.  The roundings are written out, so that
// what surrounds the arithmetic cannot change its bits.
__device__ __forceinline__ bool eval3(const Sys3 &s, uint32_t q, int o, const uint4 *pis, const float4 *vis,
                                      int (*fs)[6], uint32_t s_lo, uint32_t s_hi, long long *r)
{
    const Sys &d = s.b;
    if (q >= (uint32_t)d.n) {   // cannot happen: every queued slot was read below n
        set_err_at(d, ERR_INTERNAL, 13, q, o, 0);
        return false;
    }
    uint4 pj;
    float3 vj;
    load_bead(s.S, q, pj, vj);
    const uint4 pi = pis[o];
    if ((pi.w ^ pj.w) == 1u && d.excl) return false;   // the bonded partner
    const float4 vi = vis[o];
    const float dx = mdiff(d, pi.x, pj.x), dy = mdiff(d, pi.y, pj.y), dz = mdiff(d, pi.z, pj.z);
    const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
    if (!(r2 < d.rc2) || !(r2 > 0.f)) return false;   // the walk's filter is a little wider than r_c
    const float rinv = rsqrtf(r2);
    const float ex = __fmul_rn(dx, rinv), ey = __fmul_rn(dy, rinv), ez = __fmul_rn(dz, rinv);   // e = (x_i - x_j)/r
    const float wx = __fsub_rn(vi.x, vj.x), wy = __fsub_rn(vi.y, vj.y), wz = __fsub_rn(vi.z, vj.z);
    const float dve = __fmaf_rn(wz, ez, __fmaf_rn(wx, ex, __fmul_rn(wy, ey)));
    const float F = pair_scalar3(d, r2, rinv, dve, pi.w, pj.w, s_lo, s_hi);
    if (!(fabsf(F) < FQ_MAX)) set_err(d, ERR_NONFINITE);
    const long long qx = fq(F * ex), qy = fq(F * ey), qz = fq(F * ez);
    fq_add(&fs[o][0], 1, qx);
    fq_add(&fs[o][2], 1, qy);
    fq_add(&fs[o][4], 1, qz);
    r[0] = -qx;
    r[1] = -qy;
    r[2] = -qz;
    return true;
}

// Pair forces, one thread per bead over the half stencil: the rest of its own
// cell and the 13 cells ahead of it in (z, y, x) order, so that every pair
// inside r_c is met once (n_c >= 3).  The cells of a row are consecutive in the
// sorted order, so the stencil is five runs of slots (and, for a bead whose cell
// is the first or last of its row, up to five more with the cell across the
// boundary).  As in the 2D tile, a lane tests a run in FP32 into a bit mask
// without control flow and the warp queues the hits from a scan of their
// counts; cell by cell and candidate by candidate the walk took 150 of 193 warp
// instructions per bead (the lanes of a warp step through a run together, and
// the longest of 32 three-bead cells holds eight).  Every nb-th queued
// pair goes into one evaluation, so that its atomics rarely meet on one owner.
// 786,432 beads at density 3: 123 us against 158; what bounds it now is the
// load/store pipe (scattered partners and reactions).
constexpr int PAIRS3_THREADS = 128, PAIRS3_PAD = 64, PAIRS3_Q = 224;
__global__ void __launch_bounds__(PAIRS3_THREADS, 8) k3_pairs(Sys3 s)
{
    const Sys &d = s.b;
    constexpr int NW = PAIRS3_THREADS / 32;
    const int g = blockIdx.x * PAIRS3_THREADS + threadIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    __shared__ uint4 s_pi[NW][32];
    __shared__ float4 s_vi[NW][32];
    __shared__ int s_f[NW][32][6];
    __shared__ uint32_t s_b[NW][10][32];      // first slot of each run
    __shared__ uint32_t s_l[NW][10][32];      // and its length
    __shared__ long long s_r[NW][96];         // reactions of an evaluation, three words a pair
    __shared__ uint32_t s_rq[NW][32];         // and their slots (n: none)
    wait_for_previous();
    __shared__ uint16_t s_q[NW][PAIRS3_Q];    // queued pairs: owner lane | slot in the run << 5 | run << 10
    const bool active = g < d.n;
    const long long step = *d.step;
    const uint32_t s_lo = (uint32_t)((unsigned long long)step & 0xffffffffull);
    const uint32_t s_hi = (uint32_t)((unsigned long long)step >> 32);
    const uint32_t n = (uint32_t)d.n;
    const uint4 pi = active ? s.S[2 * (size_t)g] : make_uint4(0u, 0u, 0u, 0xffffffffu);
    const uint4 vb = active ? s.S[2 * (size_t)g + 1] : make_uint4(0u, 0u, 0u, 0u);
    s_pi[warp][lane] = pi;
    s_vi[warp][lane] = make_float4(vbits(vb.x), vbits(vb.y), vbits(vb.z), 0.f);
    const float4 xi = active ? s.S_pos[g] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 6; ++c) s_f[warp][lane][c] = 0;
    const int cx = cell_coord(d, pi.x), cy = cell_coord(d, pi.y), cz = cell_coord(d, pi.z), nc = d.nc;
    const bool west = cx == 0, east = cx == nc - 1;
    const int runs = __any_sync(FULL, west | east) ? 10 : 5;
    // run k < 5: row k of the stencil inside the box, (dy, dz) = (0, 0), (1, 0),
    // (-1, 1), (0, 1), (1, 1); run 5 + k: its cell across the boundary in x
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int dy = k == 0 ? 0 : (k == 1 ? 1 : k - 3), dz = k >= 2;
        int y = cy + dy, z = cz + dz;
        y += y < 0 ? nc : (y >= nc ? -nc : 0);
        z -= z >= nc ? nc : 0;
        const uint32_t *row = d.cstart + (size_t)(z * nc + y) * nc;
        uint32_t b = 0u, e = 0u, wb = 0u, we = 0u;
        if (active) {
            b = min(row[k == 0 ? cx : max(cx - 1, 0)], n);
            e = min(row[min(cx + 2, nc)], n);
            if (k == 0) b = (uint32_t)g + 1u;
            if (east || (west && k > 0)) {
                const int c = east ? 0 : nc - 1;
                wb = min(row[c], n);
                we = min(row[c + 1], n);
            }
        }
        s_b[warp][k][lane] = b;
        s_l[warp][k][lane] = e > b ? e - b : 0u;
        s_b[warp][5 + k][lane] = wb;
        s_l[warp][5 + k][lane] = we > wb ? we - wb : 0u;
    }
    __syncwarp();
    uint32_t qn = 0;   // warp-uniform
    // Mask of the first 32 slots of run k, seen from the bead's image beside it.
    auto mask = [&](int k) -> uint32_t {
        const int r = k < 5 ? k : k - 5, dy = r == 0 ? 0 : (r == 1 ? 1 : r - 3), dz = r >= 2;
        const float x = xi.x + (k < 5 ? 0.f : (west ? d.L : -d.L));
        const float y = xi.y + (cy + dy < 0 ? d.L : (cy + dy >= nc ? -d.L : 0.f));
        const float z = xi.z + (cz + dz >= nc ? -d.L : 0.f);
        const uint32_t l = min(s_l[warp][k][lane], 32u);
        const int most = __reduce_max_sync(FULL, (int)l);
        const float4 *p = s.S_pos + (l ? s_b[warp][k][lane] : 0u);   // padded: a window reads up to 35 slots on
        uint32_t m = 0u;
#pragma unroll 1
        for (int c = 0; c < most; c += 4) {
            uint32_t h = 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 o = p[c + u];
                const float ax = x - o.x, ay = y - o.y, az = z - o.z;
                if (ax * ax + ay * ay + az * az < s.rc2f) h |= 1u << u;
            }
            m |= h << c;
        }
        return l ? m & (0xffffffffu >> (32u - l)) : 0u;
    };
    auto evaluate = [&](bool all) {
        const uint32_t nb = all ? (qn + 31u) >> 5 : qn >> 5;
        if (nb == 0u) return;
        __syncwarp();
#pragma unroll 1
        for (uint32_t b = 0; b < nb; ++b) {
            const uint32_t i = (uint32_t)lane * nb + b;
            uint32_t q = n;
            if (i < qn) {
                const uint32_t c = s_q[warp][i], o = c & 31u;
                const uint32_t slot = s_b[warp][c >> 10][o] + ((c >> 5) & 31u);
                long long r[3];
                if (eval3(s, slot, (int)o, s_pi[warp], s_vi[warp], s_f[warp], s_lo, s_hi, r)) {
                    q = slot;
                    s_r[warp][3 * lane] = r[0];
                    s_r[warp][3 * lane + 1] = r[1];
                    s_r[warp][3 * lane + 2] = r[2];
                }
            }
            s_rq[warp][lane] = q;
            __syncwarp();
            // the reactions with the three words of a bead on neighbouring
            // lanes: a third of the wavefronts of an add per component
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int w = 32 * t + lane, p = w / 3;
                const uint32_t to = s_rq[warp][p];
                if (to < n) atomicAdd((unsigned long long *)(s.F + 4 * (size_t)to + (w - 3 * p)), (unsigned long long)s_r[warp][w]);
            }
            __syncwarp();
        }
        const uint16_t left = s_q[warp][(nb << 5) + lane < PAIRS3_Q ? (nb << 5) + lane : 0u];
        __syncwarp();
        qn = all ? 0u : qn & 31u;
        if ((uint32_t)lane < qn) s_q[warp][lane] = left;
        __syncwarp();
    };
#pragma unroll 1
    for (int k = 0; k < runs; k += 2) {
        const int k2 = k + 1 < 10 ? k + 1 : k;   // (k + 1 = 5 of 5 runs: lengths zero)
        while (true) {
            uint32_t m1 = mask(k), m2 = mask(k2);
            const uint32_t c1 = (uint32_t)lane | ((uint32_t)k << 10), c2 = (uint32_t)lane | ((uint32_t)k2 << 10);
            uint32_t end = (uint32_t)(__popc(m1) + __popc(m2));
            const uint32_t cnt = end;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(FULL, end, o);
                if (lane >= o) end += v;
            }
            const uint32_t hits = __shfl_sync(FULL, end, 31);
            uint32_t done = 0;
            while (done != hits) {   // append the lanes that fit whole (64 hits at most, 31 pairs wait)
                const uint32_t lim = done + PAIRS3_Q - qn;
                const bool go = end <= lim && end > done;
                uint32_t x1 = go ? m1 : 0u, x2 = go ? m2 : 0u;
                uint16_t *to = s_q[warp] + qn + end - done - cnt;
                const int rounds = __reduce_max_sync(FULL, max(__popc(x1), __popc(x2)));
#pragma unroll 1
                for (int r = 0; r < rounds; ++r) {
                    const uint32_t p = top_bit(x1), o = top_bit(x2);
                    if (x1) *to++ = (uint16_t)(c1 + (p << 5));
                    if (x2) *to++ = (uint16_t)(c2 + (o << 5));
                    x1 ^= bit_at(p);
                    x2 ^= bit_at(o);
                }
                const uint32_t upto = hits <= lim ? hits : __reduce_max_sync(FULL, go ? end : done);
                qn += upto - done;
                done = upto;
                evaluate(false);
            }
            // runs beyond 32 slots: the queue refers to their first slots, so it
            // is emptied before they move on
            const uint32_t l1 = s_l[warp][k][lane], l2 = s_l[warp][k2][lane];
            if (!__any_sync(FULL, (l1 > 32u) | (l2 > 32u))) break;
            evaluate(true);
            if (l1 > 32u) { s_l[warp][k][lane] = l1 - 32u; s_b[warp][k][lane] += 32u; } else { s_l[warp][k][lane] = 0u; }
            if (l2 > 32u) { s_l[warp][k2][lane] = l2 - 32u; s_b[warp][k2][lane] += 32u; } else { s_l[warp][k2][lane] = 0u; }
            __syncwarp();
        }
    }
    evaluate(true);
    __syncwarp();
    if (active) {
        unsigned long long *fq_g = (unsigned long long *)(s.F + 4 * (size_t)g);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long qc = (long long)s_f[warp][lane][2 * c] * 65536ll + (long long)(unsigned)s_f[warp][lane][2 * c + 1];
            if (qc) atomicAdd(fq_g + c, (unsigned long long)qc);
        }
    }
}

// Everything after the pair sums, one thread per sorted slot: the pair force
// (reset to zero for the next step), bond and propulsion (partner id ^ 1),
// drag on the half-step velocity, the second half-kick, FP64 thermo
// partials, the next half-kick and drift, and the binning of the new position.
__global__ void __launch_bounds__(256) k3_integrate(Sys3 s, int flags)
{
    const Sys &d = s.b;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    __shared__ uint32_t s_vmax;
    __shared__ double s_big[4];
    if (threadIdx.x < 4) s_big[threadIdx.x] = 0.0;
    if (threadIdx.x == 0) s_vmax = 0u;
    wait_for_previous();
    __syncthreads();
    float tv[3] = {0.f, 0.f, 0.f};   // v_s
    const uint32_t n = (uint32_t)d.n;
    if (g < d.n) {
        const uint4 pi = s.S[2 * (size_t)g], vb = s.S[2 * (size_t)g + 1];
        const float3 vi = make_float3(vbits(vb.x), vbits(vb.y), vbits(vb.z));
        const uint32_t id = pi.w;
        longlong2 *fqg = (longlong2 *)(s.F + 4 * (size_t)g);
        const longlong2 f01 = fqg[0], f23 = fqg[1];
        fqg[0] = make_longlong2(0ll, 0ll);
        fqg[1] = make_longlong2(0ll, 0ll);
        float fx = fq_to_f(f01.x), fy = fq_to_f(f01.y), fz = fq_to_f(f23.x);
        // bond and propulsion (partner id ^ 1), drag on the half-step velocity
        const uint32_t ps = s.slot[id ^ 1u];
        if (ps < n) {
            const uint4 pp = s.S[2 * (size_t)ps];
            const float dx = mdiff(d, pi.x, pp.x), dy = mdiff(d, pi.y, pp.y), dz = mdiff(d, pi.z, pp.z);
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (r2 > 0.f) {
                const float r = sqrtf(r2), inv = 1.0f / r;
                const float fb = -d.kbond * (r - d.r0);
                const float sp = (id & 1u) ? -d.fp : d.fp;   // n_k = head - tail
                fx += (fb + sp) * dx * inv;
                fy += (fb + sp) * dy * inv;
                fz += (fb + sp) * dz * inv;
            }
        } else {
            set_err_at(d, ERR_INTERNAL, 12, g, id, ps);
        }
        float vx = vi.x, vy = vi.y, vz = vi.z;
        fx -= d.zeta * vx;
        fy -= d.zeta * vy;
        fz -= d.zeta * vz;
        if (!(flags & F_FIRST)) { vx += d.hdtm * fx; vy += d.hdtm * fy; vz += d.hdtm * fz; }
        tv[0] = vx; tv[1] = vy; tv[2] = vz;
        if (flags & F_FINAL) {
            s.C_p[id] = make_uint4(pi.x, pi.y, pi.z, 0u);
            s.C_v[id] = make_float4(vx, vy, vz, 0.f);
            s.C_f[id] = make_float4(fx, fy, fz, 0.f);
        }
        if (flags & F_ADVANCE) {
            vx += d.hdtm * fx;
            vy += d.hdtm * fy;
            vz += d.hdtm * fz;
            const float ddx = d.dt * vx, ddy = d.dt * vy, ddz = d.dt * vz;
            uint32_t nx = pi.x, ny = pi.y, nz = pi.z;
            const float lim = 0.25f * d.L;
            if (fabsf(ddx) < lim && fabsf(ddy) < lim && fabsf(ddz) < lim) {   // false for NaN too
                nx = fx_add(d, pi.x, ddx);
                ny = fx_add(d, pi.y, ddy);
                nz = fx_add(d, pi.z, ddz);
            } else {
                set_err(d, ERR_NONFINITE);
                vx = vy = vz = 0.f;
            }
            s.U_rank[g] = atomicAdd(&d.counts[cell3(d, nx, ny, nz)], 1u);
            s.U_p[g] = make_uint4(nx, ny, nz, id);
            s.U_v[g] = make_float4(vx, vy, vz, 0.f);
        }
    }
    // thermo partials as whole numbers (see ThermoQ), scaled by the block's
    // fastest bead: FP64 partials, a hundred warp instructions a block on the
    // one-lane FP64 pipe, took a third of the time (786,432 beads: 54 us against 90)
    if (flags & (F_ADVANCE | F_FINAL)) {
        const unsigned FULL = 0xffffffffu;
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
        __shared__ int buf[8][12];
        uint32_t vm = 0u;
#pragma unroll
        for (int i = 0; i < 3; ++i) vm = max(vm, __float_as_uint(tv[i]) & 0x7fffffffu);
        vm = __reduce_max_sync(FULL, vm);
        if (lane == 0) atomicMax(&s_vmax, vm);
        __syncthreads();
        ThermoQ th = thermo_q(s_vmax, 1, s_big);
        long long q[4] = {0, 0, 0, 0};   // v'^2; v' by component in 2^-24
        if (fabsf(tv[0]) * th.sc < th.lim && fabsf(tv[1]) * th.sc < th.lim && fabsf(tv[2]) * th.sc < th.lim) {
            float er = 0.f;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float w = __fmul_rn(tv[i], th.sc);
                const int a = __float2int_rn(w);
                const float r = __fsub_rn(w, (float)a);
                q[0] += (long long)a * a;
                er = __fmaf_rn(r, __fadd_rn(w, (float)a), er);
                q[1 + i] = (long long)a * 16777216 + __float2int_rn(__fmul_rn(r, 16777216.0f));
            }
            q[0] += __float2int_rn(er);
        } else if (tv[0] != 0.f || tv[1] != 0.f || tv[2] != 0.f) {
            double e = 0.0;
            for (int i = 0; i < 3; ++i) {
                e = fma((double)tv[i], (double)tv[i], e);
                atomicAdd(&s_big[1 + i], (double)tv[i]);
            }
            atomicAdd(&s_big[0], e);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int q0 = (int)__reduce_add_sync(FULL, (unsigned)(q[i] & 0x3fffffll));
            const int q1 = (int)__reduce_add_sync(FULL, (unsigned)((q[i] >> 22) & 0x3fffffll));
            const int q2 = __reduce_add_sync(FULL, (int)(q[i] >> 44));
            if (lane == 0) { buf[wid][3 * i] = q0; buf[wid][3 * i + 1] = q1; buf[wid][3 * i + 2] = q2; }
        }
        __syncthreads();
        if (tid < 4) {
            long long s0 = 0, s1 = 0, s2 = 0;
            for (int w = 0; w < 8; ++w) {
                s0 += buf[w][3 * tid];
                s1 += buf[w][3 * tid + 1];
                s2 += buf[w][3 * tid + 2];
            }
            const int x = (int)(__float_as_uint(th.sc) >> 23) - 127;   // sc = 2^x
            const int ex = th.lim == 0.0f ? 0 : (tid == 0 ? -2 * x : -x - 24);
            const double a = fma((double)s2, 17592186044416.0, fma((double)s1, 4194304.0, (double)s0)) *
                             __hiloint2double((1023 + ex) << 20, 0);
            const double b = s_big[tid];
            atomicAdd(&d.thermo[4 * (size_t)(*d.step % THERMO_CAP) + tid], b != 0.0 ? a + b : a);
        }
    }
}

}  // namespace dpd

using namespace dpd;

#define CU3(x)                                                                      \
    do {                                                                            \
        const cudaError_t e_ = (x);                                                 \
        if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? DPD_ERR_OOM : DPD_ERR_CUDA; \
    } while (0)

static int latched3(dpd3_ctx *c)
{
    int *e = (int *)(c->h_pin + 500);
    CU3(cudaMemcpyAsync(e, c->s.b.err, sizeof(int), cudaMemcpyDeviceToHost, c->st));
    CU3(cudaStreamSynchronize(c->st));
    if (*e & ERR_NONFINITE) return DPD_ERR_NONFINITE;
    if (*e & ERR_TIMEOUT) return DPD_ERR_TIMEOUT;
    if (*e & ERR_INTERNAL) return DPD_ERR_INTERNAL;
    return DPD_OK;
}

int dpd3_internal_latched(dpd3_ctx *c) { return latched3(c); }

static void iteration3(dpd3_ctx *c, int flags)
{
    const int g = (c->s.b.n + 255) / 256;
    launch_step(k3_scan, c->nscan, SCAN_NT, 0, c->st, c->s.b, c->nscan);
    launch_step(k3_scatter, g, 256, 0, c->st, c->s);
    launch_step(k3_pairs, (c->s.b.n + PAIRS3_THREADS - 1) / PAIRS3_THREADS, PAIRS3_THREADS, 0, c->st, c->s);
    launch_step(k3_integrate, g, 256, 0, c->st, c->s, flags);
}

extern "C" {

int dpd3_create(const dpd_params *p, void *stream, dpd3_ctx **out)
{
    if (!out) return DPD_ERR_INVALID_ARG;
    *out = nullptr;
    int rc = validate(p);
    if (rc) return rc;
    const int nc = n_cells_side(p->L, p->rc);
    if ((double)nc * nc * nc >= 2.0e9) return DPD_ERR_INVALID_ARG;
    dpd3_ctx *c = new (std::nothrow) dpd3_ctx();
    if (!c) return DPD_ERR_OOM;
    c->p = *p;
    if (stream) c->st = (cudaStream_t)stream;
    else {
        if (cudaStreamCreateWithFlags(&c->st, cudaStreamNonBlocking) != cudaSuccess) { delete c; return DPD_ERR_CUDA; }
        c->own_stream = true;
    }
    Sys &d = c->s.b;
    fill_physics(d, p);
    fill_geometry(d, p, 8);
    d.ncells = nc * nc * nc;
    d.ntx = 0;
    d.cap = 0;
    c->nscan = (d.ncells + SCAN_TILE - 1) / SCAN_TILE;
    const size_t n = (size_t)d.n, nce = (size_t)d.ncells;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += (bytes + 255) & ~size_t(255); return o; };
    const size_t o_S = take(32 * n), o_Up = take(16 * n), o_Uv = take(16 * n),
                 o_Cp = take(16 * n), o_Cv = take(16 * n), o_Cf = take(16 * n), o_rank = take(4 * n),
                 o_slot = take(4 * n), o_cnt = take(4 * nce), o_cst = take(4 * (nce + 1)),
                 o_th = take(32 * (size_t)THERMO_CAP), o_step = take(8), o_err = take(4), o_einfo = take(32),
                 o_ss = take(8 * (size_t)c->nscan), o_tk = take(8), o_stage = take(48 * n),
                 o_F = take(32 * n), o_pos = take(16 * (n + PAIRS3_PAD));
    if (cudaMalloc(&c->pool, off) != cudaSuccess || cudaMallocHost((void **)&c->h_pin, 4096) != cudaSuccess) {
        dpd3_destroy(c);
        return DPD_ERR_OOM;
    }
    char *b = (char *)c->pool;
    c->s.S = (uint4 *)(b + o_S);
    c->s.U_p = (uint4 *)(b + o_Up); c->s.U_v = (float4 *)(b + o_Uv);
    c->s.C_p = (uint4 *)(b + o_Cp); c->s.C_v = (float4 *)(b + o_Cv); c->s.C_f = (float4 *)(b + o_Cf);
    c->s.U_rank = (uint32_t *)(b + o_rank); c->s.slot = (uint32_t *)(b + o_slot);
    c->s.F = (long long *)(b + o_F);   // zeroed with the pool; k3_integrate keeps it zero between steps
    c->s.S_pos = (float4 *)(b + o_pos);
    // FP32 coordinates are good to 2^-23 L, a shifted one to 2^-23 L more: a
    // separation to sqrt(3) (2^-22 + 2^-23) L
    c->s.rc2f = (float)((p->rc + 8e-7 * p->L) * (p->rc + 8e-7 * p->L) * (1.0 + 1e-5));
    d.slot = c->s.slot;
    d.counts = (uint32_t *)(b + o_cnt); d.cstart = (uint32_t *)(b + o_cst);
    d.thermo = (double *)(b + o_th); d.step = (long long *)(b + o_step);
    d.err = (int *)(b + o_err); d.errinfo = (long long *)(b + o_einfo);
    d.scan_status = (unsigned long long *)(b + o_ss); d.scan_ticket = (unsigned long long *)(b + o_tk);
    d.S_xv = nullptr; d.S_id = nullptr; d.U_xv = nullptr; d.U_id = nullptr; d.U_rank = c->s.U_rank;
    d.C_xv = nullptr; d.C_f = nullptr; d.pcnt = nullptr; d.ovf = nullptr;
    c->stage = b + o_stage;
    if (cudaMemsetAsync(c->pool, 0, off, c->st) != cudaSuccess ||
        cudaStreamSynchronize(c->st) != cudaSuccess) {
        dpd3_destroy(c);
        return DPD_ERR_CUDA;
    }
    *out = c;
    return DPD_OK;
}

void dpd3_destroy(dpd3_ctx *c)
{
    if (!c) return;
    if (c->st) cudaStreamSynchronize(c->st);
    if (c->pool) cudaFree(c->pool);
    if (c->obs) cudaFree(c->obs);
    if (c->h_pin) cudaFreeHost(c->h_pin);
    if (c->own_stream && c->st) cudaStreamDestroy(c->st);
    delete c;
}

int dpd3_set_state(dpd3_ctx *c, const double *x, const float *v, int64_t step)
{
    if (!c || !x || !v) return DPD_ERR_INVALID_ARG;
    const size_t n = (size_t)c->s.b.n;
    char *st = c->stage;
    CU3(cudaMemcpyAsync(st, x, 24 * n, cudaMemcpyHostToDevice, c->st));
    CU3(cudaMemcpyAsync(st + 24 * n, v, 12 * n, cudaMemcpyHostToDevice, c->st));
    CU3(cudaMemsetAsync(c->s.b.err, 0, sizeof(int), c->st));
    CU3(cudaMemsetAsync(c->s.b.errinfo, 0, 32, c->st));
    CU3(cudaMemsetAsync(c->s.b.counts, 0, 4 * (size_t)c->s.b.ncells, c->st));
    const int g = (int)((n + 255) / 256);
    k3_load<<<g, 256, 0, c->st>>>(c->s, (const double *)st, (const float *)(st + 24 * n));
    k3_bin<<<g, 256, 0, c->st>>>(c->s);
    k3_set_step<<<1, 1, 0, c->st>>>(c->s.b, step - 1);
    iteration3(c, F_FIRST | F_FINAL | F_ADVANCE);
    CU3(cudaGetLastError());
    c->step = step;
    c->have_state = true;
    return latched3(c);
}

int dpd3_step(dpd3_ctx *c, int64_t n)
{
    if (!c || n < 0) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    for (int64_t i = 0; i < n; ++i) iteration3(c, i == n - 1 ? (F_ADVANCE | F_FINAL) : F_ADVANCE);
    CU3(cudaGetLastError());
    c->step += n;
    return DPD_OK;
}

int dpd3_sync(dpd3_ctx *c)
{
    if (!c) return DPD_ERR_INVALID_ARG;
    return latched3(c);
}

int dpd3_get_state(dpd3_ctx *c, double *x, float *v, float *f, int64_t *step)
{
    if (!c || !x || !v || !f) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    const size_t n = (size_t)c->s.b.n;
    double *dx = (double *)c->stage;
    float *dv = (float *)(dx + 3 * n), *df = dv + 3 * n;
    k3_store<<<(int)((n + 255) / 256), 256, 0, c->st>>>(c->s, dx, dv, df);
    CU3(cudaMemcpyAsync(x, dx, 24 * n, cudaMemcpyDeviceToHost, c->st));
    CU3(cudaMemcpyAsync(v, dv, 12 * n, cudaMemcpyDeviceToHost, c->st));
    CU3(cudaMemcpyAsync(f, df, 12 * n, cudaMemcpyDeviceToHost, c->st));
    if (step) *step = c->step;
    return latched3(c);
}

int dpd3_thermo(dpd3_ctx *c, double out[5])
{
    if (!c || !out) return DPD_ERR_INVALID_ARG;
    if (!c->have_state) return DPD_ERR_STATE;
    CU3(cudaMemcpyAsync(c->h_pin, c->s.b.thermo + 4 * (size_t)(c->step % THERMO_CAP), 32, cudaMemcpyDeviceToHost,
                        c->st));
    const int rc = latched3(c);
    const double m = c->p.mass, n = (double)c->s.b.n;
    out[0] = 0.5 * m * c->h_pin[0];
    out[1] = m * c->h_pin[1];
    out[2] = m * c->h_pin[2];
    out[3] = m * c->h_pin[3];
    out[4] = m * c->h_pin[0] / (3.0 * n - 3.0);
    return rc;
}

}  // extern "C"
