// Cloud-in-cell (CIC) variant of the step and its adjoint, for differentiable
// runs.  The paper's nearest-grid-point assignment (Eq. eqn:cell) has zero
// position gradient almost everywhere; this variant spreads each mass over
// the 8 cells around it with trilinear weights W, takes the grid field as
// the central difference of the potential (first term of Eq. eqn:diff) and
// interpolates it back with the same weights.  Regions, mass sets, the
// doubled-grid convolution and the combination rule of Sec. 2.1 are those of
// the NGP step; grid centres are held fixed.
//
// CIC cells: the NGP cell a of Eq. (eqn:cell) (canonical rounding) fixes the
// particle; t = Delta / l in [-1/2, 1/2] is its offset from that cell's
// centre; the lower CIC cell is a - 1 with fraction t + 1 when t < 0, else a
// with fraction t.  With a in the usable box 2..N-3 the CIC cells and their
// difference neighbours stay inside 0..N-1.
//
// Adjoint (vector-Jacobian product of the acceleration a(x, m) with a
// cotangent u per particle), with K the symmetric convolution and D the
// central difference (D^T = -D on the grid):
//   direct term  dx_i += sum_c grad W(x_i - x_c) (g[c] . u_i)
//   field term   lam_k = K sum_d D_d^T psi_k^d, psi_k^d = sum_i W u_i^d over the
//                field points that read set k; then for each particle j of mass
//                set k: dx_j += m_j sum_c grad W lam_k[c], dm_j += sum_c W lam_k[c].
// The sum_d D_d^T psi is spread directly from each particle (32 cells) as
// int64 fixed point, so the adjoint solve reuses the FFT passes unchanged.
// Pair slots are loaded so that the solver's stored outputs are the lam_k
// the mass sets need: medium a = psi_2 - psi_3, b = psi_3 (outputs
// lam_2 = a + b, lam_3 = b); coarse a = psi_4 - psi_5, b = psi_5.
//
// Bound by the atomics (32 per point and level in the adjoint spread, 80 G/s
// for unsorted points).  So the particles of nested systems run in spatial order
// (an index computed per deposit, pm_launch_order, 55 us for 1M; the rule and
// both its sides: cic_order_pays in pm_api.cu), runs of particles in one cell
// share their atomics, and each point spreads once per level.  1M points of two
// galaxies: deposit 333 -> 129 us, spread 1600 -> 558, direct term 160 -> 104.
#pragma once

#include <algorithm>

#include "pm_launch.h"
#include "pm_particle.cuh"

namespace pmk {

// Threads per block of the particle kernels of this file: small blocks, so that
// a few ten thousand particles spread evenly over the SMs (FP64 runs are bound
// by the SMs' FP64 pipes).
constexpr int CIC_THREADS = 64;

template <typename T> struct Cic {
    size_t base;          // offset of the lower cell (a0, b0, c0)
    T w[3][2];            // per axis: weights of the lower and upper cell
    T il[3];              // 1 / l per axis
};

template <typename T>
__device__ __forceinline__ Cic<T> cic_cell(const GeomK &g, const Cell &cl, T rx, T ry, T rz) {
    T d[3];
    cell_delta(g, cl, rx, ry, rz, d[0], d[1], d[2]);
    Cic<T> c;
    c.il[0] = c.il[1] = pick<T>(2.0 * g.c_gx, g.fil_xy);
    c.il[2] = pick<T>(2.0 * g.c_gz, g.fil_z);
    int idx[3] = {cl.i, cl.j, cl.k};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T t = d[a] * c.il[a];
        if (t < (T)0) { idx[a] -= 1; t += (T)1; }
        c.w[a][0] = (T)1 - t;
        c.w[a][1] = t;
    }
    c.base = ((size_t)idx[2] * g.ny + idx[1]) * g.nx + idx[0];
    return c;
}

// Central-difference field of F at the 8 CIC cells: gr[dk][dj][di][axis].
template <typename T>
__device__ __forceinline__ void cic_grad8(const GeomK &g, const T *__restrict__ F, const Cic<T> &c,
                                          T gr[2][2][2][3]) {
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
    const T *b = F + c.base;
    auto ld = [&](int di, int dj, int dk) -> T { return __ldg(b + di + dj * sy + dk * sz); };
    T cen[2][2][2];
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di) cen[dk][dj][di] = ld(di, dj, dk);
    const T hx = c.il[0] * (T)0.5, hz = c.il[2] * (T)0.5;
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj) {
            const T lo = ld(-1, dj, dk), hi = ld(2, dj, dk);
            gr[dk][dj][0][0] = (cen[dk][dj][1] - lo) * hx;
            gr[dk][dj][1][0] = (hi - cen[dk][dj][0]) * hx;
        }
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            const T lo = ld(di, -1, dk), hi = ld(di, 2, dk);
            gr[dk][0][di][1] = (cen[dk][1][di] - lo) * hx;
            gr[dk][1][di][1] = (hi - cen[dk][0][di]) * hx;
        }
#pragma unroll
    for (int dj = 0; dj < 2; ++dj)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            const T lo = ld(di, dj, -1), hi = ld(di, dj, 2);
            gr[0][dj][di][2] = (cen[1][dj][di] - lo) * hz;
            gr[1][dj][di][2] = (hi - cen[0][dj][di]) * hz;
        }
}

// acc += sum_c W g_c   (VJP == false)
// gx  += sum_c grad W (g_c . u)   (VJP == true)
template <typename T, bool VJP>
__device__ __forceinline__ void cic_field(const GeomK &g, const void *F, const Cic<T> &c, const T *u, T *out) {
    T gr[2][2][2][3];
    cic_grad8<T>(g, static_cast<const T *>(F), c, gr);
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const T *v = gr[dk][dj][di];
                if (!VJP) {
                    const T W = c.w[0][di] * c.w[1][dj] * c.w[2][dk];
                    out[0] += W * v[0];
                    out[1] += W * v[1];
                    out[2] += W * v[2];
                } else {
                    const T s = v[0] * u[0] + v[1] * u[1] + v[2] * u[2];
                    out[0] += (di ? c.il[0] : -c.il[0]) * c.w[1][dj] * c.w[2][dk] * s;
                    out[1] += (dj ? c.il[1] : -c.il[1]) * c.w[0][di] * c.w[2][dk] * s;
                    out[2] += (dk ? c.il[2] : -c.il[2]) * c.w[0][di] * c.w[1][dj] * s;
                }
            }
}

// lam_w += sum_c W F_c, lam_g += sum_c grad W F_c (the 8 CIC cells).
template <typename T>
__device__ __forceinline__ void cic_gather(const GeomK &g, const void *Fv, const Cic<T> &c, T &lw, T *lg) {
    const T *F = static_cast<const T *>(Fv) + c.base;
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const T f = __ldg(F + di + dj * sy + dk * sz);
                lw += c.w[0][di] * c.w[1][dj] * c.w[2][dk] * f;
                lg[0] += (di ? c.il[0] : -c.il[0]) * c.w[1][dj] * c.w[2][dk] * f;
                lg[1] += (dj ? c.il[1] : -c.il[1]) * c.w[0][di] * c.w[2][dk] * f;
                lg[2] += (dk ? c.il[2] : -c.il[2]) * c.w[0][di] * c.w[1][dj] * f;
            }
}

// Rounds a share, already scaled by the (power of two) fixed-point factor.
// (Integer operations in place of the conversion, which runs on the FP64 pipe,
// measured slower: adjoint spread of 1M points 558 -> 582 us.)
__device__ __forceinline__ long long cic_q(float v) { return __float2ll_rn(v); }
__device__ __forceinline__ long long cic_q(double v) { return __double2ll_rn(v); }

// Adjacent active lanes with one lower cell (the particles run in the order of
// pm_launch_order) form a run; with runs of two or more on average every cell's
// shares are summed over the run by a segmented scan (64-bit adds, exact) and
// its last lane issues the atomic.  Every lane of the warp must call start
// and add.
struct CicRuns {
    bool active, sum, tail;
    int behind, longest;   // lanes since the run's first; the warp's largest
    __device__ __forceinline__ void start(const unsigned long long *cell, bool act) {
        const unsigned FULL = 0xffffffffu;
        const int lane = (int)(threadIdx.x & 31);
        active = act;
        const unsigned long long key = act ? (unsigned long long)cell : 0ull;   // no cell lives at address 0
        const unsigned long long prev = __shfl_up_sync(FULL, key, 1);
        const unsigned heads = __ballot_sync(FULL, act && (lane == 0 || prev != key)), on = __ballot_sync(FULL, act);
        const unsigned brk = heads | ~on;
        const unsigned upto = lane == 31 ? FULL : ((2u << lane) - 1u);
        behind = act ? lane - (31 - __clz(brk & upto)) : 0;
        tail = act && (lane == 31 || ((brk >> (lane + 1)) & 1u));
        sum = 2 * __popc(heads) <= __popc(on);
        longest = sum ? (int)__reduce_max_sync(FULL, (unsigned)behind) : 0;
    }
    __device__ __forceinline__ void add(unsigned long long *addr, long long q) const {
        unsigned long long v = (unsigned long long)q;
        if (sum) {
            for (int d = 1; d <= longest; d <<= 1) {
                const unsigned long long u = __shfl_up_sync(0xffffffffu, v, d);
                if (behind >= d) v += u;
            }
            if (tail) atomicAdd(addr, v);
        } else if (active) {
            atomicAdd(addr, v);
        }
    }
};

// Forward deposit: m W into the 8 cells (fixed point; m carries the scale).
template <typename T>
__device__ __forceinline__ void cic_spread_mass(const GeomK &g, unsigned long long *rho, const Cic<T> &c, T m,
                                                bool active) {
    const int sy = g.nx, sz = g.nx * g.ny;
    unsigned long long *b = rho + c.base;
    CicRuns run;
    run.start(b, active);
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di)
                run.add(b + di + dj * sy + dk * sz, active ? cic_q(m * (c.w[0][di] * c.w[1][dj] * c.w[2][dk])) : 0);
}

// Adjoint spread: sum_d D_d^T (W u_d) into the 32 cells it touches (fixed
// point).  h[d] = u_d / (2 l_d) times the scale.
template <typename T>
__device__ __forceinline__ void cic_spread_adj(const GeomK &g, unsigned long long *rho, const Cic<T> &c, const T *h,
                                               bool active) {
    const int sy = g.nx, sz = g.nx * g.ny;
    unsigned long long *b = rho + c.base;
    CicRuns run;
    run.start(b, active);
    auto add = [&](int di, int dj, int dk, T v) { run.add(b + di + dj * sy + dk * sz, active ? cic_q(v) : 0); };
    const T(&w)[3][2] = c.w;
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const T vx = h[0] * w[1][dj] * w[2][dk] * (di ? w[0][0] : -w[0][1]);
                const T vy = h[1] * w[0][di] * w[2][dk] * (dj ? w[1][0] : -w[1][1]);
                const T vz = h[2] * w[0][di] * w[1][dj] * (dk ? w[2][0] : -w[2][1]);
                add(di, dj, dk, vx + vy + vz);
            }
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj) {
            add(-1, dj, dk, -h[0] * w[0][0] * w[1][dj] * w[2][dk]);
            add(2, dj, dk, h[0] * w[0][1] * w[1][dj] * w[2][dk]);
        }
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            add(di, -1, dk, -h[1] * w[1][0] * w[0][di] * w[2][dk]);
            add(di, 2, dk, h[1] * w[1][1] * w[0][di] * w[2][dk]);
        }
#pragma unroll
    for (int dj = 0; dj < 2; ++dj)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            add(di, dj, -1, -h[2] * w[2][0] * w[0][di] * w[1][dj]);
            add(di, dj, 2, h[2] * w[2][1] * w[0][di] * w[1][dj]);
        }
}

// Particle position relative to the system centre and to galaxy h's centre.
template <typename T> struct Rel {
    float sx, sy, sz;   // canonical FP32 offsets from the system centre (cells, lost test)
    T rsx, rsy, rsz;    // offsets from the system centre (Delta)
};
template <typename T>
__device__ __forceinline__ Rel<T> rel_sys(const SysK &s, T x, T y, T z) {
    Rel<T> r;
    r.sx = pm_canon(x, s.sc[0], s.sc_hi[0], s.sc_lo[0]);
    r.sy = pm_canon(y, s.sc[1], s.sc_hi[1], s.sc_lo[1]);
    r.sz = pm_canon(z, s.sc[2], s.sc_hi[2], s.sc_lo[2]);
    r.rsx = rel_off(x, s.sc[0], s.sc_hi[0], s.sc_lo[0]);
    r.rsy = rel_off(y, s.sc[1], s.sc_hi[1], s.sc_lo[1]);
    r.rsz = rel_off(z, s.sc[2], s.sc_hi[2], s.sc_lo[2]);
    return r;
}

// Particle j of the processing order (ord null: as stored).
__device__ __forceinline__ long long cic_at(const unsigned *ord, long long j) { return ord ? (long long)__ldg(ord + j) : j; }

// Forward CIC deposit with the lost test and mass sets of the NGP deposit.
// The loop is warp-uniform (the spreads are warp collectives).
template <typename T>
__global__ void __launch_bounds__(CIC_THREADS) k_cic_deposit(PartK<T> p, const __grid_constant__ SysK s,
                                                             const CenK *cen, const unsigned *ord) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long b = (long long)blockIdx.x * blockDim.x; b < p.n; b += stride) {
        const long long j = b + threadIdx.x;
        const long long i = j < p.n ? cic_at(ord, j) : 0;
        const uint32_t f = j < p.n ? p.flags[i] : PM_FLAG_LOST;
        bool live = !(f & PM_FLAG_LOST);
        Cic<T> kc = {}, km = {}, kf = {};
        int reg = REG_OUTER, g = 0;
        T m = 0;
        if (live) {
            const T x = p.x[i], y = p.y[i], z = p.z[i];
            g = p.gal[i];
            m = p.m[i] * pick<T>(s.mscale, s.mscale_f);   // a power of two: exact
            const Rel<T> rs = rel_sys(s, x, y, z);
            bool lost = !(pm_r2(rs.sx, rs.sy, rs.sz) < s.rsys2);
            if (g < 0 || g >= s.ngal) lost = true;
            Cell cc;
            cc.i = cc.j = cc.k = 0; cc.ok = false;
            for (int h = 0; h < s.ngal; ++h) {
                const Cell ch = pm_cells(s.gal[h].coarse, rs.sx, rs.sy, rs.sz);
                lost = lost || !ch.ok;
                if (h == g) cc = ch;
            }
            if (lost) {
                p.flags[i] = f | PM_FLAG_LOST;
                live = false;
                g = 0;
            } else {
                const GalK &G = s.gal[g];
                const Cen1 ce = load_cen(cen, g);
                Cell cf, cm;
                reg = pm_region(G, pm_canon(x, ce.c[0], ce.hi[0], ce.lo[0]), pm_canon(y, ce.c[1], ce.hi[1], ce.lo[1]),
                                pm_canon(z, ce.c[2], ce.hi[2], ce.lo[2]), cf, cm);
                kc = cic_cell<T>(G.coarse, cc, rs.rsx, rs.rsy, rs.rsz);
                if (reg != REG_OUTER) {
                    const T rx = rel_off(x, ce.c[0], ce.hi[0], ce.lo[0]);
                    const T ry = rel_off(y, ce.c[1], ce.hi[1], ce.lo[1]);
                    const T rz = rel_off(z, ce.c[2], ce.hi[2], ce.lo[2]);
                    km = cic_cell<T>(G.med, cm, rx, ry, rz);
                    if (reg == REG_CORE) kf = cic_cell<T>(G.fine, cf, rx, ry, rz);
                }
            }
        }
        const GalK &G = s.gal[g];
        cic_spread_mass<T>(G.coarse, G.rho[reg == REG_OUTER ? 4 : 3], kc, m, live);
        if (!__any_sync(0xffffffffu, live && reg != REG_OUTER)) continue;
        cic_spread_mass<T>(G.med, G.rho[reg == REG_CORE ? 1 : 2], km, m, live && reg != REG_OUTER);
        if (__any_sync(0xffffffffu, live && reg == REG_CORE))
            cic_spread_mass<T>(G.fine, G.rho[0], kf, m, live && reg == REG_CORE);
    }
}

// Field-point kernels over every galaxy's grids (combination rule):
//   MODE 0: v += dtk a, x += dtd v     MODE 1: write a
//   MODE 2: g += u^T (d a / d x_i) direct term (positions' own weights)
//   MODE 3: adjoint spread of u into the pair slots (scale qs)
template <typename T, int MODE>
__global__ void __launch_bounds__(CIC_THREADS) k_cic_field(PartK<T> p, const __grid_constant__ SysK s, const CenK *cen,
                                                           T dtk, T dtd, T *ox, T *oy, T *oz, const T *ux, const T *uy,
                                                           const T *uz, T qs, const unsigned *ord) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long b = (long long)blockIdx.x * blockDim.x; b < p.n; b += stride) {   // warp-uniform (MODE 3)
        const long long j = b + threadIdx.x;
        if (MODE != 3 && j >= p.n) continue;
        const long long i = j < p.n ? cic_at(ord, j) : 0;
        const bool live = j < p.n && !(p.flags[i] & PM_FLAG_LOST);
        if (MODE != 3 && !live) {
            if (MODE == 1) { ox[i] = 0; oy[i] = 0; oz[i] = 0; }
            continue;
        }
        T xT = 0, yT = 0, zT = 0;
        T u[3] = {0, 0, 0};
        if (live) {
            xT = p.x[i]; yT = p.y[i]; zT = p.z[i];
            if (MODE >= 2) { u[0] = ux[i]; u[1] = uy[i]; u[2] = uz[i]; }
        }
        const Rel<T> rs = rel_sys(s, xT, yT, zT);
        T out[3] = {0, 0, 0};
        for (int h = 0; h < s.ngal; ++h) {
            const GalK &G = s.gal[h];
            const Cen1 ce = load_cen(cen, h);
            Cell cf, cm;
            const int reg = pm_region(G, pm_canon(xT, ce.c[0], ce.hi[0], ce.lo[0]),
                                      pm_canon(yT, ce.c[1], ce.hi[1], ce.lo[1]),
                                      pm_canon(zT, ce.c[2], ce.hi[2], ce.lo[2]), cf, cm);
            const Cell cc = pm_cells(G.coarse, rs.sx, rs.sy, rs.sz);
            const bool on = live && cc.ok;   // not ok only after positions changed without a deposit
            if (MODE != 3 && !on) continue;
            const Cic<T> kc = cic_cell<T>(G.coarse, cc, rs.rsx, rs.rsy, rs.rsz);
            Cic<T> km = {}, kf = {};
            if (on && reg != REG_OUTER) {
                const T rx = rel_off(xT, ce.c[0], ce.hi[0], ce.lo[0]);
                const T ry = rel_off(yT, ce.c[1], ce.hi[1], ce.lo[1]);
                const T rz = rel_off(zT, ce.c[2], ce.hi[2], ce.lo[2]);
                km = cic_cell<T>(G.med, cm, rx, ry, rz);
                if (reg == REG_CORE) kf = cic_cell<T>(G.fine, cf, rx, ry, rz);
            }
            if (MODE == 3) {
                // each point once per level, into the slot of its region:
                // k_cic_slots forms the sums and differences the solve takes
                const T v[3] = {u[0] * qs, u[1] * qs, u[2] * qs};   // qs a power of two: exact
                T c3[3] = {v[0] * pick<T>(G.coarse.c_gx, G.coarse.fc_gx), v[1] * pick<T>(G.coarse.c_gx, G.coarse.fc_gx), v[2] * pick<T>(G.coarse.c_gz, G.coarse.fc_gz)};
                cic_spread_adj<T>(G.coarse, G.rho[reg == REG_OUTER ? 4 : 3], kc, c3, on);
                if (!__any_sync(0xffffffffu, on && reg != REG_OUTER)) continue;
                T m3[3] = {v[0] * pick<T>(G.med.c_gx, G.med.fc_gx), v[1] * pick<T>(G.med.c_gx, G.med.fc_gx), v[2] * pick<T>(G.med.c_gz, G.med.fc_gz)};
                cic_spread_adj<T>(G.med, G.rho[reg == REG_CORE ? 1 : 2], km, m3, on && reg != REG_OUTER);
                if (!__any_sync(0xffffffffu, on && reg == REG_CORE)) continue;
                T f3[3] = {v[0] * pick<T>(G.fine.c_gx, G.fine.fc_gx), v[1] * pick<T>(G.fine.c_gx, G.fine.fc_gx), v[2] * pick<T>(G.fine.c_gz, G.fine.fc_gz)};
                cic_spread_adj<T>(G.fine, G.rho[0], kf, f3, on && reg == REG_CORE);   // psi_1
                continue;
            }
            constexpr bool VJP = (MODE == 2);
            cic_field<T, VJP>(G.coarse, reg == REG_OUTER ? G.phi_call : G.phi_c5, kc, u, out);
            if (reg != REG_OUTER) {
                cic_field<T, VJP>(G.med, reg == REG_SHELL ? G.phi_m23 : G.phi_m3, km, u, out);
                if (reg == REG_CORE) cic_field<T, VJP>(G.fine, G.phi_fine, kf, u, out);
            }
        }
        if (MODE == 0) {
            const T vx = p.vx[i] + dtk * out[0], vy = p.vy[i] + dtk * out[1], vz = p.vz[i] + dtk * out[2];
            p.vx[i] = vx; p.vy[i] = vy; p.vz[i] = vz;
            p.x[i] = xT + dtd * vx; p.y[i] = yT + dtd * vy; p.z[i] = zT + dtd * vz;
        } else if (MODE == 1) {
            ox[i] = out[0]; oy[i] = out[1]; oz[i] = out[2];
        } else if (MODE == 2) {
            ox[i] += out[0]; oy[i] += out[1]; oz[i] += out[2];
        }
    }
}

// The pair slots of the adjoint solve from the regions' spreads: medium
// a = psi_2 - psi_3 (minus the core's), b = psi_3 (core and shell); coarse
// a = psi_4 - psi_5 (minus the inner points'), b = psi_5 (all points).
static __global__ void __launch_bounds__(256) k_cic_slots(long long *a, long long *b, long long n) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += stride) {   // n is even
        longlong2 *pa = reinterpret_cast<longlong2 *>(a) + i, *pb = reinterpret_cast<longlong2 *>(b) + i;
        longlong2 va = *pa, vb = *pb;
        vb.x += va.x; vb.y += va.y;
        va.x = -va.x; va.y = -va.y;
        *pa = va;
        *pb = vb;
    }
}

// Field term of the adjoint for each particle's own mass sets: the adjoint
// solve left lam_1 in the fine sum slot, lam_2 (medium sum), lam_3 (medium
// b), lam_4 (coarse sum) and lam_5 (coarse b, or the sum without medium).
template <typename T>
__global__ void __launch_bounds__(CIC_THREADS) k_cic_gather(PartK<T> p, const __grid_constant__ SysK s, const CenK *cen,
                                                            T *gx, T *gy, T *gz, T *gm) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    // in stored order: the few gathers gain less than the indirect sums cost
    // (1M points: 54 us, in spatial order 98)
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += stride) {
        if (p.flags[i] & PM_FLAG_LOST) continue;
        const int g = p.gal[i];
        if (g < 0 || g >= s.ngal) continue;
        const T x = p.x[i], y = p.y[i], z = p.z[i];
        const Rel<T> rs = rel_sys(s, x, y, z);
        const GalK &G = s.gal[g];
        const Cen1 ce = load_cen(cen, g);
        Cell cf, cm;
        const int reg = pm_region(G, pm_canon(x, ce.c[0], ce.hi[0], ce.lo[0]), pm_canon(y, ce.c[1], ce.hi[1], ce.lo[1]),
                                  pm_canon(z, ce.c[2], ce.hi[2], ce.lo[2]), cf, cm);
        const Cell cc = pm_cells(G.coarse, rs.sx, rs.sy, rs.sz);
        if (!cc.ok) continue;
        T lw = 0, lg[3] = {0, 0, 0};
        const Cic<T> kc = cic_cell<T>(G.coarse, cc, rs.rsx, rs.rsy, rs.rsz);
        if (reg == REG_OUTER) {
            cic_gather<T>(G.coarse, G.phi_c5, kc, lw, lg);
        } else {
            const T rx = rel_off(x, ce.c[0], ce.hi[0], ce.lo[0]);
            const T ry = rel_off(y, ce.c[1], ce.hi[1], ce.lo[1]);
            const T rz = rel_off(z, ce.c[2], ce.hi[2], ce.lo[2]);
            cic_gather<T>(G.coarse, G.phi_call, kc, lw, lg);
            const Cic<T> km = cic_cell<T>(G.med, cm, rx, ry, rz);
            if (reg == REG_CORE) {
                cic_gather<T>(G.med, G.phi_m23, km, lw, lg);
                cic_gather<T>(G.fine, G.phi_fine, cic_cell<T>(G.fine, cf, rx, ry, rz), lw, lg);
            } else {
                cic_gather<T>(G.med, G.phi_m3, km, lw, lg);
            }
        }
        const T m = p.m[i];
        gx[i] += m * lg[0];
        gy[i] += m * lg[1];
        gz[i] += m * lg[2];
        gm[i] += lw;
    }
}

// max |u| over live particles (as float bits; non-finite values give +inf).
template <typename T>
__global__ void __launch_bounds__(256) k_cic_umax(PartK<T> p, const T *ux, const T *uy, const T *uz, unsigned *out) {
    float mx = 0.f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += stride) {
        if (p.flags[i] & PM_FLAG_LOST) continue;
        const T a = fmax(fabs(ux[i]), fmax(fabs(uy[i]), fabs(uz[i])));
        const float af = (a == a) ? (float)a : __int_as_float(0x7f800000);
        mx = fmaxf(mx, af);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(mx));
}

}  // namespace pmk

// ---------------------------------------------------------------------------
// Host launchers (instantiated for float and double in pm_cic.cu)
// ---------------------------------------------------------------------------
namespace pmk_cic_host {
inline int grid_for(long long n, int threads = pmk::CIC_THREADS) {
    long long b = (n + threads - 1) / threads;
    return (int)(b < (1LL << 18) ? (b > 0 ? b : 1) : (1LL << 18));
}
}  // namespace pmk_cic_host

template <typename T>
cudaError_t pm_launch_cic_deposit(const PartK<T> &p, const SysK &sk, const CenK *cen, const unsigned *ord,
                                  cudaStream_t st) {
    if (p.n <= 0) return cudaSuccess;
    pmk::k_cic_deposit<T><<<pmk_cic_host::grid_for(p.n), pmk::CIC_THREADS, 0, st>>>(p, sk, cen, ord);
    return cudaGetLastError();
}

template <typename T>
cudaError_t pm_launch_cic_field(int mode, const PartK<T> &p, const SysK &sk, const CenK *cen, double dtk, double dtd,
                                T *ox, T *oy, T *oz, const T *ux, const T *uy, const T *uz, double qs,
                                const unsigned *ord, cudaStream_t st) {
    if (p.n <= 0) return cudaSuccess;
    const int g = pmk_cic_host::grid_for(p.n);
#define PM_CF(M) pmk::k_cic_field<T, M><<<g, pmk::CIC_THREADS, 0, st>>>(p, sk, cen, (T)dtk, (T)dtd, ox, oy, oz, ux, uy, uz, (T)qs, ord)
    switch (mode) {
        case 0: PM_CF(0); break;
        case 1: PM_CF(1); break;
        case 2: PM_CF(2); break;
        case 3: PM_CF(3); break;
        default: return cudaErrorInvalidValue;
    }
#undef PM_CF
    return cudaGetLastError();
}

static cudaError_t cic_slots(long long *a, long long *b, long long n, cudaStream_t st) {
    pmk::k_cic_slots<<<(unsigned)std::min<long long>((n / 2 + 255) / 256, 16LL * pmk_host::num_sms()), 256, 0, st>>>(a, b, n);
    return cudaGetLastError();
}

template <typename T>
cudaError_t pm_launch_cic_gather(const PartK<T> &p, const SysK &sk, const CenK *cen, T *gx, T *gy, T *gz, T *gm,
                                 cudaStream_t st) {
    if (p.n <= 0) return cudaSuccess;
    pmk::k_cic_gather<T><<<pmk_cic_host::grid_for(p.n), pmk::CIC_THREADS, 0, st>>>(p, sk, cen, gx, gy, gz, gm);
    return cudaGetLastError();
}

template <typename T>
cudaError_t pm_launch_cic_umax(const PartK<T> &p, const T *ux, const T *uy, const T *uz, unsigned *out,
                               cudaStream_t st) {
    if (p.n <= 0) return cudaSuccess;
    pmk::k_cic_umax<T><<<pmk_cic_host::grid_for(p.n, 256), 256, 0, st>>>(p, ux, uy, uz, out);
    return cudaGetLastError();
}

#define PM_CIC_INSTANTIATE(T)                                                                                  \
    template cudaError_t pm_launch_cic_deposit<T>(const PartK<T> &, const SysK &, const CenK *, const unsigned *, \
                                                  cudaStream_t);                                               \
    template cudaError_t pm_launch_cic_field<T>(int, const PartK<T> &, const SysK &, const CenK *, double,     \
                                                double, T *, T *, T *, const T *, const T *, const T *, double, \
                                                const unsigned *, cudaStream_t);                               \
    template cudaError_t pm_launch_cic_gather<T>(const PartK<T> &, const SysK &, const CenK *, T *, T *, T *,  \
                                                 T *, cudaStream_t);                                           \
    template cudaError_t pm_launch_cic_umax<T>(const PartK<T> &, const T *, const T *, const T *, unsigned *,  \
                                               cudaStream_t);
