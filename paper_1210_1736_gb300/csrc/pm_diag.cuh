// Disc diagnostics of the paper's Sec. 6 (thickness sqrt<z^2>(R), heat
// E_heat about the binned circular velocity, velocity dispersions in an
// annulus, Fourier modes A~_m in rings) as FP64 reductions over the selected
// particles, positions and velocities taken relative to a galaxy centre.
//
// Bound by the FP64 pipe (2 lanes per clock and SM), so nothing is computed
// twice and nothing returns to the host in between: one pass compacts the
// selected particles' R^2 and index; the bins' bounds, exact order statistics
// of R^2, come from a radix select over the IEEE bits of R^2 (a non-negative
// double, so its bits order like its value) whose digits are resolved on the
// device; one pass forms every sum and leaves what the heat needs.  1M
// particles, 400k selected, launches under ncu: radix passes over all particles
// 353 us (and a host step each), sums by FP64 shared atomics 318, heat 130;
// now select and radix passes 163, sums 105 (FP64 operations and read-modify-
// writes of 4 warps per SM, as many as the columns leave room for), heat 17.
// Without memory for the list every pass reads the particles (the whole call
// 389 -> 690 us).
#pragma once

#include <algorithm>

#include "pm_launch.h"
#include "pm_particle.cuh"
#include "pm_roots.cuh"

namespace pmk {

template <typename T>
__device__ __forceinline__ bool diag_take(const DiagP<T> &d, long long i) {
    if (d.flags[i] & PM_FLAG_LOST) return false;
    return d.sel ? d.sel[i] != 0 : d.gal_id[i] == d.gal;
}

// Bits of R^2 (the same operations as the FP64 reference, no contraction).
__device__ __forceinline__ unsigned long long diag_key(double dx, double dy) {
    return (unsigned long long)__double_as_longlong(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
}

// Counts the selected particles and compacts their key and index (key null:
// counts only), in blocks of 1024 particles.
template <typename T>
__global__ void __launch_bounds__(256) k_diag_select(DiagP<T> d, const CenK *cen, DiagState *st,
                                                     unsigned long long *key, long long *idx) {
    __shared__ int wtot[8];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double cx = cen->c[d.gal][0], cy = cen->c[d.gal][1];
    for (long long b = (long long)blockIdx.x * 1024; b < d.n; b += (long long)gridDim.x * 1024) {
        bool take[4];
        unsigned before[4];
        int tot = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long i = b + u * 256 + threadIdx.x;
            take[u] = i < d.n && diag_take(d, i);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned m = __ballot_sync(0xffffffffu, take[u]);
            before[u] = tot + __popc(m & ((1u << lane) - 1u));
            tot += __popc(m);
        }
        if (lane == 0) wtot[w] = tot;
        __syncthreads();
        if (threadIdx.x == 0) {
            int s = 0;
            for (int k = 0; k < 8; ++k) {
                const int v = wtot[k];
                wtot[k] = s;
                s += v;
            }
            base = s ? atomicAdd(&st->nsel, (unsigned long long)s) : 0;
        }
        __syncthreads();
        const long long o = (long long)base + wtot[w];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (take[u] && key) {
                const long long i = b + u * 256 + threadIdx.x;
                key[o + before[u]] = diag_key(__dsub_rn((double)d.x[i], cx), __dsub_rn((double)d.y[i], cy));
                idx[o + before[u]] = i;
            }
        __syncthreads();   // wtot and base are rewritten
    }
}

// The selected particles' keys: as k_diag_select left them, or from the
// particles (no memory to keep them).
struct DiagKept {
    const unsigned long long *key;
    __device__ __forceinline__ long long count(const DiagState *st) const { return (long long)st->nsel; }
    __device__ __forceinline__ bool get(long long i, unsigned long long &k) const { k = key[i]; return true; }
};
template <typename T> struct DiagRead {
    DiagP<T> d;
    const CenK *cen;
    __device__ __forceinline__ long long count(const DiagState *) const { return d.n; }
    __device__ __forceinline__ bool get(long long i, unsigned long long &k) const {
        if (!diag_take(d, i)) return false;
        k = diag_key(__dsub_rn((double)d.x[i], cen->c[d.gal][0]), __dsub_rn((double)d.y[i], cen->c[d.gal][1]));
        return true;
    }
};

// Digits of the radix select: DG_BITS bits per pass from the top, the last
// pass the remaining ones.
constexpr int DG_BITS = 11, DG_PASSES = 6, DG_ROW = 1 << DG_BITS;
__device__ __forceinline__ int diag_low(int pass) { return pass + 1 < DG_PASSES ? 64 - DG_BITS * (pass + 1) : 0; }
__device__ __forceinline__ int diag_high(int pass) { return 64 - DG_BITS * pass; }

// By the pass's last block: each boundary's digit from its prefix's counters,
// then the prefixes of the next pass (boundaries are sorted, so equal ones are
// adjacent); clears the counters.
static __device__ void diag_resolve(int pass, int nbins, int np, long long n, DiagState *st, unsigned *hist) {
    __shared__ unsigned long long nk[DIAG_MAXBINS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nb = nbins - 1;
    const int width = diag_high(pass) - diag_low(pass);
    for (int k = w; k < nb; k += 8) {
        const int j = pass ? st->which[k] : 0;
        const long long rank = pass ? st->rank[k] : ((long long)(k + 1) * n) / nbins;
        const uint4 *row = reinterpret_cast<const uint4 *>(hist + j * DG_ROW + lane * (DG_ROW / 32));
        uint4 h[DG_ROW / 128];
        unsigned sum = 0;
#pragma unroll
        for (int q = 0; q < DG_ROW / 128; ++q) {
            h[q] = __ldcg(row + q);
            sum += h[q].x + h[q].y + h[q].z + h[q].w;
        }
        unsigned incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const unsigned has = __ballot_sync(0xffffffffu, (long long)incl > rank);
        if (has == 0 && lane == 0 && n > 0) st->err = 1;   // particles changed during the call?
        if (lane == (has ? __ffs(has) - 1 : 0)) {
            long long left = rank - (long long)(incl - sum);
            int dgt = 0;
            bool done = false;
#pragma unroll
            for (int q = 0; q < DG_ROW / 128; ++q) {
                const unsigned c[4] = {h[q].x, h[q].y, h[q].z, h[q].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (!done && left < (long long)c[e]) {
                        done = true;
                        dgt = lane * (DG_ROW / 32) + q * 4 + e;
                    }
                    if (!done) left -= c[e];
                }
            }
            nk[k] = ((pass ? st->pref[j] : 0ull) << width) | (unsigned long long)dgt;
            st->rank[k] = left;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < np * DG_ROW / 4; i += 256) reinterpret_cast<uint4 *>(hist)[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        int m = 0;
        for (int k = 0; k < nb; ++k) {
            if (m == 0 || nk[k] != nk[k - 1]) st->pref[m++] = nk[k];
            st->which[k] = m - 1;
            st->edge[k] = nk[k];   // complete after the last pass
        }
        st->npref = m;
        st->done = 0;
    }
}

// One pass: keys that agree with one of the sorted prefixes (the bits above
// diag_high) count their next digit.  Lanes with one counter share an atomic
// (the first digits, exponents, take few values).  The last block to finish
// resolves the pass.
template <class KEYS>
__global__ void __launch_bounds__(256) k_diag_hist(int pass, int nbins, DiagState *st, KEYS keys, unsigned *hist) {
    __shared__ unsigned long long pref[DIAG_MAXBINS];
    __shared__ bool last;
    const int np = pass ? st->npref : 1;
    const long long n = keys.count(st);
    if (threadIdx.x < np) pref[threadIdx.x] = pass ? st->pref[threadIdx.x] : 0;
    __syncthreads();
    const int low = diag_low(pass), high = diag_high(pass);
    const unsigned mask = (1u << (high - low)) - 1u;
    for (long long b = (long long)blockIdx.x * 256; b < n; b += (long long)gridDim.x * 256) {
        const long long i = b + threadIdx.x;
        int bin = -1;
        unsigned long long k;
        if (i < n && keys.get(i, k)) {
            int j = 0;
            if (pass > 0) {
                const unsigned long long pk = k >> high;
                int lo = 0, hi = np - 1;
                j = -1;
                while (lo <= hi) {
                    const int mid = (lo + hi) >> 1;
                    if (pref[mid] == pk) { j = mid; break; }
                    if (pref[mid] < pk) lo = mid + 1; else hi = mid - 1;
                }
            }
            if (j >= 0) bin = j * DG_ROW + (int)((unsigned)(k >> low) & mask);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        if (bin >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(hist + bin, (unsigned)__popc(peers));
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) {
        __threadfence();
        diag_resolve(pass, nbins, np, (long long)st->nsel, st, hist);
    }
}

// R, the direction and the cylindrical velocities of a particle.
struct DiagPoint {
    double R, c1, s1, vR, vphi;
    __device__ __forceinline__ DiagPoint(unsigned long long key, double dx, double dy, double vx, double vy) {
        double inv;
        pmroot::root_inv(__longlong_as_double((long long)key), R, inv);
        c1 = dx * inv;
        s1 = dy * inv;
        vR = c1 * vx + s1 * vy;
        vphi = c1 * vy - s1 * vx;
    }
    // what the heat needs
    __device__ __forceinline__ double4 rest(double vz, double m) const { return make_double4(R, vphi, vR * vR + vz * vz, m); }
};

// The sums over the selected particles; KEPT: of k_diag_select's list, leaving
// what the heat needs per particle, else of the particles themselves.
// Accumulators in shared memory: with PRIVATE a column per thread (no
// conflicts, no atomics), else one set per block.
template <typename T, bool PRIVATE, bool KEPT>
__global__ void __launch_bounds__(256) k_diag_sums(DiagP<T> d, const CenK *cen, DiagQ q, const DiagState *st,
                                                   const unsigned long long *key, const long long *idx, double *acc,
                                                   double4 *rest) {
    extern __shared__ double sh[];
    __shared__ unsigned long long edge[DIAG_MAXBINS];
    const int nacc = 4 * q.nbins + 7 + 2 * q.nring * q.mmax, copies = PRIVATE ? (int)blockDim.x : 1;
    for (int k = threadIdx.x; k < nacc * copies; k += blockDim.x) sh[k] = 0.0;
    for (int k = threadIdx.x; k < q.nbins - 1; k += blockDim.x) edge[k] = st->edge[k];
    __syncthreads();
    auto add = [&](int k, double v) {
        if (PRIVATE) sh[k * copies + threadIdx.x] += v;
        else atomicAdd(sh + k, v);
    };
    const double cx = cen->c[d.gal][0], cy = cen->c[d.gal][1], cz = cen->c[d.gal][2], iw = 1.0 / q.width;
    const long long n = KEPT ? (long long)st->nsel : d.n, stride = (long long)gridDim.x * blockDim.x;
    // few warps fit beside the columns: U particles' loads in flight each
    constexpr int U = 4;
    for (long long p0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; p0 < n; p0 += U * stride) {
        unsigned long long ku[U];
        T xu[U], yu[U], zu[U], vxu[U], vyu[U], vzu[U], mu[U];
        long long iu[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long p = p0 + u * stride;
            iu[u] = -1;
            if (KEPT) {
                if (p < n) { ku[u] = key[p]; iu[u] = idx[p]; }
            } else if (p < n && diag_take(d, p)) {
                iu[u] = p;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (iu[u] >= 0) {
                const long long i = iu[u];
                xu[u] = d.x[i]; yu[u] = d.y[i]; zu[u] = d.z[i];
                vxu[u] = d.vx[i]; vyu[u] = d.vy[i]; vzu[u] = d.vz[i];
                mu[u] = d.m[i];
            }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (iu[u] < 0) continue;
            const double dx = __dsub_rn((double)xu[u], cx), dy = __dsub_rn((double)yu[u], cy);
            const unsigned long long r2k = KEPT ? ku[u] : diag_key(dx, dy);
            const double dz = __dsub_rn((double)zu[u], cz);
            const double vx = vxu[u], vy = vyu[u], vz = vzu[u], m = mu[u];
            int b = 0;   // number of edges <= key
            {
                int lo = 0, hi = q.nbins - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (edge[mid] <= r2k) lo = mid + 1; else hi = mid;
                }
                b = lo;
            }
            const DiagPoint pt(r2k, dx, dy, vx, vy);
            const double R = pt.R, c1 = pt.c1, s1 = pt.s1, vR = pt.vR, vphi = pt.vphi;
            if (KEPT) rest[p0 + u * stride] = pt.rest(vz, m);
            add(4 * b + 0, R);
            add(4 * b + 1, 1.0);
            add(4 * b + 2, dz * dz);
            add(4 * b + 3, vphi);
            if (R >= q.rlo && R < q.rhi) {
                const int a = 4 * q.nbins;
                add(a + 0, m);
                add(a + 1, m * vR);
                add(a + 2, m * vR * vR);
                add(a + 3, m * vphi);
                add(a + 4, m * vphi * vphi);
                add(a + 5, m * vz);
                add(a + 6, m * vz * vz);
            }
            if (R > 0 && R < q.r_ring) {
                // floor(R / width): the quotient is formed only near an integer
                double f = R * iw;
                const double near = rint(f);
                if (fabs(f - near) < 1e-9 * (near + 1.0)) f = __ddiv_rn(R, q.width);
                const int ring = (int)floor(f);
                if (ring < q.nring) {
                    const int a = 4 * q.nbins + 7 + 2 * ring * q.mmax;
                    // exp(-i m phi) by the angle-addition recurrence from m cos, m sin phi
                    double cm = m * c1, sm = -m * s1;
                    for (int mo = 0; mo < q.mmax; ++mo) {
                        add(a + 2 * mo, cm);
                        add(a + 2 * mo + 1, sm);
                        const double cn = cm * c1 + sm * s1;
                        sm = sm * c1 - cm * s1;
                        cm = cn;
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nacc; k += blockDim.x) {
        double v = 0.0;
        if (PRIVATE) {
            double v2 = 0.0, v3 = 0.0, v4 = 0.0;   // four chains; the columns start at k: no bank conflicts
            for (int c = 0; c < copies; c += 4) {
                v += sh[k * copies + ((c + k) & (copies - 1))];
                v2 += sh[k * copies + ((c + 1 + k) & (copies - 1))];
                v3 += sh[k * copies + ((c + 2 + k) & (copies - 1))];
                v4 += sh[k * copies + ((c + 3 + k) & (copies - 1))];
            }
            v = (v + v2) + (v3 + v4);
        } else {
            v = sh[k];
        }
        if (v != 0.0) atomicAdd(acc + k, v);
    }
}

// E_heat with vbar_c linear in R between the non-empty bins' (mean R, mean
// v_phi), held constant outside.
template <typename T, bool KEPT>
__global__ void __launch_bounds__(256) k_diag_heat(DiagP<T> d, const CenK *cen, int nbins, const DiagState *st,
                                                   const double *acc, const double4 *rest, double *heat) {
    __shared__ double xp[DIAG_MAXBINS], fp[DIAG_MAXBINS], sl[DIAG_MAXBINS], red[8];
    __shared__ int s_np;
    if (threadIdx.x < 32) {
        int base = 0;
        for (int b0 = 0; b0 < nbins; b0 += 32) {
            const int b = b0 + threadIdx.x;
            const double cnt = b < nbins ? acc[4 * b + 1] : 0.0;
            const unsigned m = __ballot_sync(0xffffffffu, cnt > 0);
            if (cnt > 0) {
                const int k = base + __popc(m & ((1u << threadIdx.x) - 1u));
                xp[k] = acc[4 * b] / cnt;
                fp[k] = acc[4 * b + 3] / cnt;
            }
            base += __popc(m);
        }
        __syncwarp();
        for (int k = threadIdx.x; k + 1 < base; k += 32) sl[k] = (fp[k + 1] - fp[k]) / (xp[k + 1] - xp[k]);
        if (threadIdx.x == 0) s_np = base;
    }
    __syncthreads();
    const int np = s_np;
    const long long n = KEPT ? (long long)st->nsel : d.n, stride = (long long)gridDim.x * blockDim.x;
    double e = 0.0;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += stride) {
        double4 v;
        if (KEPT) {
            v = rest[p];
        } else {
            if (!diag_take(d, p)) continue;
            const double dx = __dsub_rn((double)d.x[p], cen->c[d.gal][0]), dy = __dsub_rn((double)d.y[p], cen->c[d.gal][1]);
            v = DiagPoint(diag_key(dx, dy), dx, dy, d.vx[p], d.vy[p]).rest(d.vz[p], d.m[p]);
        }
        const double R = v.x;
        double vb;
        if (R <= xp[0]) vb = fp[0];
        else if (R >= xp[np - 1]) vb = fp[np - 1];
        else {
            int lo = 0, hi = np - 1;   // xp[lo] < R < xp[hi]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (xp[mid] <= R) lo = mid; else hi = mid;
            }
            vb = sl[lo] * (R - xp[lo]) + fp[lo];
        }
        const double dv = v.y - vb;
        e += 0.5 * v.w * (v.z + dv * dv);
    }
    e = warp_sum(e);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        if (s != 0.0) atomicAdd(heat, s);
    }
}

}  // namespace pmk

template <typename T, bool KEPT>
cudaError_t pm_launch_diag_k(const pmk::DiagP<T> &d, const CenK *cen, const pmk::DiagQ &q, const pmk::DiagBuf &b,
                             cudaStream_t st) {
    const int nacc = 4 * q.nbins + 7 + 2 * q.nring * q.mmax;
    // a wave of blocks: the sums' epilogues cost FP64 operations per block
    const unsigned sms = (unsigned)pmk_host::num_sms();
    const unsigned by = (unsigned)std::min<long long>((d.n + 1023) / 1024, 8 * sms);
    pmk::k_diag_select<T><<<by, 256, 0, st>>>(d, cen, b.state, b.key, b.idx);
    if (q.nbins > 1)
        for (int pass = 0; pass < pmk::DG_PASSES; ++pass) {
            const unsigned g = std::min(by, 2 * sms);
            if constexpr (KEPT) pmk::k_diag_hist<<<g, 256, 0, st>>>(pass, q.nbins, b.state, pmk::DiagKept{b.key}, b.hist);
            else pmk::k_diag_hist<<<g, 256, 0, st>>>(pass, q.nbins, b.state, pmk::DiagRead<T>{d, cen}, b.hist);
        }
    // a column of accumulators per thread while 64 or 32 threads' fit two
    // blocks on an SM
    const size_t one = sizeof(double) * nacc;
    const int threads = 64 * one <= 100u << 10 ? 64 : 32 * one <= 100u << 10 ? 32 : 0;
    if (threads) {
        const auto k = pmk::k_diag_sums<T, true, KEPT>;
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 << 10);
        if (e != cudaSuccess) return e;
        k<<<2 * sms, threads, threads * one, st>>>(d, cen, q, b.state, b.key, b.idx, b.acc, b.rest);
    } else {
        // one set per block: small blocks, as few particles as there are for
        // each, since a block's threads add to its set one after another (64
        // bins, 16 x 64 modes, whole call with 20k / 100k / 1M particles: 482, 543
        // and 1484 us; 256 threads, a block per 1024 particles 603, 628 and 1557)
        const unsigned g = (unsigned)std::min<long long>((d.n + 127) / 128, 8 * sms);
        pmk::k_diag_sums<T, false, KEPT><<<g, 128, one, st>>>(d, cen, q, b.state, b.key, b.idx, b.acc, b.rest);
    }
    pmk::k_diag_heat<T, KEPT><<<std::min(by, 4 * sms), 256, 0, st>>>(d, cen, q.nbins, b.state, b.acc, b.rest, b.acc + nacc);
    return cudaGetLastError();
}

// Every step of pm_disc_diagnostics on the device (acc: nacc + 1 sums, the
// last the heat; everything zeroed here).
template <typename T>
cudaError_t pm_launch_diag(const pmk::DiagP<T> &d, const CenK *cen, const pmk::DiagQ &q, const pmk::DiagBuf &b,
                           cudaStream_t st) {
    const int nacc = 4 * q.nbins + 7 + 2 * q.nring * q.mmax;
    cudaError_t e = cudaMemsetAsync(b.state, 0, sizeof(pmk::DiagState), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.acc, 0, sizeof(double) * (nacc + 1), st);
    if (e == cudaSuccess && q.nbins > 1)
        e = cudaMemsetAsync(b.hist, 0, sizeof(unsigned) * pmk::DG_ROW * (q.nbins - 1), st);
    if (e != cudaSuccess || d.n <= 0) return e;
    return b.key ? pm_launch_diag_k<T, true>(d, cen, q, b, st) : pm_launch_diag_k<T, false>(d, cen, q, b, st);
}

#define PM_DIAG_INSTANTIATE(T)                                                                                \
    template cudaError_t pm_launch_diag<T>(const pmk::DiagP<T> &, const CenK *, const pmk::DiagQ &, const pmk::DiagBuf &, \
                                           cudaStream_t);
