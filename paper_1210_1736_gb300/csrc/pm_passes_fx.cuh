// FFT passes of FP64 contexts: the passes of pm_passes.cuh on fixed-point
// transforms (pm_fx.cuh).  Work arrays, tiles, tensor maps and the batch walk
// are the same; what differs is the arithmetic and the shape of the code.
//
// Bound by integer instructions (a 1M-particle galaxy's y forward: ALU pipe 64 %,
// IMAD.WIDE pipe 50 %, issue 57 %, DRAM 20 %; its 256-point z pass: 53, 50, 52
// and 9 %), after the instruction cache:
// unrolled like the FP32 passes a z pass was 180 KB of code and its warps
// waited for instructions.  So every transform runs the one forward plan (an
// inverse swaps the components going in and coming out), equal stages share a
// loop body, and the conversions between FP64 and fixed point and the spectral
// factors run in rolled loops over shared memory, where each thread keeps its
// 16 values in slots only it touches.  128-thread blocks, three per SM: four
// (128 registers) and two measured the same.
//
// One step of the 1M-particle galaxy (128^3, 128^3, 128x128x32 grids), FP64
// arithmetic -> this: x forward 452 -> 120 us, y forward 826 -> 211, z 3381 ->
// 921, y inverse 942 -> 240, x inverse 497 -> 143.  Error of the potential
// against 80-bit arithmetic on grids of 16^3 to 64^3 and 256x16x64: 0.6-1.0
// times that of the FP64 transforms.
#pragma once

#include "pm_passes.cuh"

namespace pmk {

constexpr int FXT = 128;   // threads per block of the FP64 passes: three blocks per SM by registers and shared memory

// Scale of a transform's values: value = x 2^ex.  measure() publishes the
// largest butterfly sum of the group (one warp, or the block through slot),
// apply() shifts; a block-wide group synchronises in between.
template <bool BLOCK> struct FxScale {
    int ex;
    int *slot;     // block: zero before use, slot[s] for stage s
    unsigned m;
    template <int R> __device__ __forceinline__ void measure(const fx2 *v, int s) {
        m = pmfx::warp_max(pmfx::group_sum<R>(v));
        if (BLOCK && (threadIdx.x & 31) == 0) atomicMax(slot + s, (int)m);
    }
    __device__ __forceinline__ void apply(fx2 *v, int s, int top) {
        const int sh = pmfx::sum_shift(BLOCK ? (unsigned)slot[s] : m, top);
        pmfx::shift<E>(v, sh);
        ex += sh;
    }
};

template <int L> __host__ __device__ constexpr int fx_top(int s) {   // room for a closing radix-2 stage that is not rescaled
    return pmfx::FX_TOP - ((L == 32 && s == 0) || (L == 512 && s == 1) ? 1 : 0);
}

template <bool BLOCK> __device__ __forceinline__ void fx_sync() {
    if (BLOCK) __syncthreads(); else __syncwarp();
}

// Forward transform of length L on the group's scaled values: register e
// holds row t + e L/16 before and after.  Exchanges through sm (layout lay);
// the group is a warp or, BLOCK, the block, which ends synchronised.
template <int L, bool BLOCK, class LAY>
__device__ __forceinline__ void fx_fft(fx2 *v, fx2 *sm, const LAY &lay, int t, const fxw *tw, FxScale<BLOCK> &sc) {
    if constexpr (L == 256) {   // two equal stages
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
            if (s) {
                pmfft::load_stage<L, 1, false>(sm, lay, t, v);
                sc.template measure<16>(v, 1);
                fx_sync<BLOCK>();
                sc.apply(v, 1, pmfx::FX_TOP);
                const fxw *tws = tw + t;
#pragma unroll
                for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], tws[r * 16]);
            }
            pmfft::Dft<16, -1, fx2>::run(v);
            if (!s) {
                pmfft::store_stage<L, 0, false>(sm, lay, t, v);
                fx_sync<BLOCK>();
            }
        }
        return;
    }
    pmfft::stage_butterflies<L, 0, false, -1>(v, t, tw);
    if constexpr (L > 16) {
        constexpr int R1 = radix(L, 1, false);
        pmfft::store_stage<L, 0, false>(sm, lay, t, v);
        fx_sync<BLOCK>();
        pmfft::load_stage<L, 1, false>(sm, lay, t, v);
        if constexpr (R1 > 2) sc.template measure<R1>(v, 1);
        fx_sync<BLOCK>();
        if constexpr (R1 > 2) sc.apply(v, 1, fx_top<L>(1));
        pmfft::stage_butterflies<L, 1, false, -1>(v, t, tw);
    }
    if constexpr (L > 256) {
        pmfft::store_stage<L, 1, false>(sm, lay, t, v);
        fx_sync<BLOCK>();
        pmfft::load_stage<L, 2, false>(sm, lay, t, v);
        fx_sync<BLOCK>();
        pmfft::stage_butterflies<L, 2, false, -1>(v, t, tw);
    }
    if constexpr (L > 16) pmfft::regs_last_to_first<L>(v);
}

// exponent of a power of two
__device__ __forceinline__ int exponent_of(double s) { return ((__double2hiint(s) >> 20) & 0x7ff) - 1023; }

// In-place conversion of a thread's slots (at(e), e < n) between FP64 and
// fixed point, in rolled loops.
template <class AT> __device__ __forceinline__ void fx_from(int n, int em, AT &&at) {
#pragma unroll 2
    for (int e = 0; e < n; ++e) {
        int4 *p = reinterpret_cast<int4 *>(at(e));
        const double2 d = *reinterpret_cast<const double2 *>(p);
        fx2 q;
        q.x = pmfx::from_double<pmfx::FX_TOP>(d.x, em);
        q.y = pmfx::from_double<pmfx::FX_TOP>(d.y, em);
        *reinterpret_cast<fx2 *>(p) = q;
    }
}
template <bool CHECK> __device__ __forceinline__ double2 fx_out(fx2 q, int ex) {
    return make_double2(pmfx::to_double<CHECK>(q.x, ex), pmfx::to_double<CHECK>(q.y, ex));
}
template <bool CHECK, class AT> __device__ __forceinline__ void fx_to_loop(int n, int ex, AT &&at) {
#pragma unroll CHECK ? 1 : 2
    for (int e = 0; e < n; ++e) {
        fx2 *p = reinterpret_cast<fx2 *>(at(e));
        *reinterpret_cast<double2 *>(p) = fx_out<CHECK>(*p, ex);
    }
}
template <class AT> __device__ __forceinline__ void fx_to(int n, int ex, AT &&at) {
    if (pmfx::in_range(ex)) fx_to_loop<false>(n, ex, at);
    else fx_to_loop<true>(n, ex, at);
}
__device__ __forceinline__ fx2 swapped(fx2 v) { fx2 r; r.x = v.y; r.y = v.x; return r; }

// ---------------------------------------------------------------------------
// x passes.  Blocks of 32..FXT threads (the launch takes fewer where a grid
// has too few rows to give every SM a block).
// ---------------------------------------------------------------------------
template <int L> constexpr size_t fx_xsmem(int threads) {
    return (size_t)(pmfft::tw_dir_size(L, false) + threads / XShape<L>::TPC * XShape<L>::LDR) * sizeof(fx2);
}

// INV = false: integer densities in, spectrum rows out; INV: spectrum rows
// in, potentials out (as k_xfwd and k_xinv).
template <int L, bool INV, bool HALF> __global__ void __launch_bounds__(FXT, 3) k_xfx(const __grid_constant__ PassBatch B) {
    typedef XShape<L> S;
    constexpr int NX = L / 2, TPC = S::TPC;
    extern __shared__ __align__(16) unsigned char smraw[];
    fxw *tw = reinterpret_cast<fxw *>(smraw);
    fx2 *sm = reinterpret_cast<fx2 *>(tw + pmfft::tw_dir_size(L, false));
    const int tid = threadIdx.x, line = tid / TPC, t = tid % TPC, lines = blockDim.x / TPC;
    const int ny = B.a[0].ny, lgi = B.lgi;   // common to the items; read once (see k_xfwd)
    __shared__ void *ip[PM_BATCH][3];
    __shared__ int isplit[PM_BATCH];
    if (tid < B.n) {
        ip[tid][0] = INV ? B.a[tid].phi_b : const_cast<long long *>(B.a[tid].rho_a);
        ip[tid][1] = INV ? B.a[tid].phi_sum : const_cast<long long *>(B.a[tid].rho_b);
        ip[tid][2] = B.a[tid].work;
        isplit[tid] = B.a[tid].split;
    }
    pmfft::expand_stage_twiddles<L, 1, false>(tw, static_cast<const fxw *>(B.a[0].tw));
    pmfft::expand_stage_twiddles<L, 2, false>(tw, static_cast<const fxw *>(B.a[0].tw));
    __syncthreads();
    pdl_wait();
    const long long nrows = (long long)ny * B.a[0].nz >> (HALF ? 1 : 0);   // HALF: row pairs, as in k_xfwd
    const int kend = B.kend;
    const long long ngroups = (long long)B.n << lgi;
    const int lny = __ffs(ny) - 1;   // row r = z*ny + y; ny is a power of two
    const int ex0 = exponent_of(B.a[0].scale);
    const pmfft::RowLayout lay{line * S::LDR};
    auto mine = [&](int e) { return sm + lay(t + e * TPC); };
    for (long long grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
        if (grp + gridDim.x >= ngroups) pdl_release();
        const int item = (int)(grp >> lgi);
        const long long r = (grp & ((1LL << lgi) - 1)) * lines + line;
        const bool valid = r < nrows;
        const long long r1 = (HALF ? 2 : 1) * r;   // the (first) row
        const long long z = valid ? r1 >> lny : 0, y = valid ? r1 & (ny - 1) : 0;
        double2 *row = static_cast<double2 *>(ip[item][2]) + ((size_t)z * 2 * ny + y) * L;
        fx2 v[E];
        FxScale<false> sc{ex0, nullptr, 0};
        if constexpr (INV && HALF) {
            // slots k <= nx: F0(k); above: F1(L - k), and F1(0), F1(nx) beside
            unsigned m = 0;
            double2 ends = make_double2(0.0, 0.0);   // F1(0) (t = 0) and F1(nx)
#pragma unroll
            for (int e = 0; e <= E / 2; ++e) {
                const int k = t + e * TPC;
                if (k > NX) continue;
                double2 d = make_double2(0.0, 0.0), f = d;
                if (valid) {
                    d = __ldg(row + k);
                    f = __ldg(row + L + k);
                }
                m = max(m, max(max(pmfx::dmag(d.x), pmfx::dmag(d.y)), max(pmfx::dmag(f.x), pmfx::dmag(f.y))));
                *reinterpret_cast<double2 *>(sm + lay(k)) = d;
                if (k > 0 && k < NX) *reinterpret_cast<double2 *>(sm + lay(L - k)) = f;
                else if (k == 0) ends.x = f.x;   // real, up to rounding
                else ends.y = f.x;
            }
            // a bit less than FX_TOP: F0 + i F1 adds two components
            const int em = pmfx::group_em(pmfx::warp_max(m));
            sc.ex = pmfx::group_ex(em, pmfx::FX_TOP) + 1;
            __syncwarp();
            fx_from(E, em + 1, mine);
            __syncwarp();
            // F0 + i F1 at k, and at L - k from the rows' symmetry
#pragma unroll 1
            for (int e = 0; e <= E / 2; ++e) {
                const int k = t + e * TPC;
                if (k > NX) break;
                const fx2 f0 = sm[lay(k)];
                if (k == 0 || k == NX) {
                    fx2 p;
                    p.x = f0.x;
                    p.y = pmfx::from_double<pmfx::FX_TOP>(k == 0 ? ends.x : ends.y, em + 1);
                    sm[lay(k)] = p;
                    continue;
                }
                const fx2 f1 = sm[lay(L - k)];
                fx2 p, q;
                p.x = f0.x - f1.y; p.y = f0.y + f1.x;
                q.x = f0.x + f1.y; q.y = f1.x - f0.y;
                sm[lay(k)] = p;
                sm[lay(L - k)] = q;
            }
            __syncwarp();
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = swapped(*mine(e));
            __syncwarp();   // read before the exchange writes
        } else if constexpr (INV) {
            unsigned m = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                double2 d = make_double2(0.0, 0.0);
                if (valid) d = __ldg(row + t + e * TPC);
                m = max(m, max(pmfx::dmag(d.x), pmfx::dmag(d.y)));
                *reinterpret_cast<double2 *>(mine(e)) = d;
            }
            const int em = pmfx::group_em(pmfx::warp_max(m));
            sc.ex = pmfx::group_ex(em, pmfx::FX_TOP);
            fx_from(E, em, mine);
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = swapped(*mine(e));
            __syncwarp();   // read before the exchange writes
        } else {
            const long long *ra = static_cast<const long long *>(ip[item][0]) + (valid ? r1 * NX : 0);
            const long long *rb = HALF ? ra + NX : static_cast<const long long *>(ip[item][1]);
            if (!HALF && rb) rb += valid ? r * NX : 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                v[e] = czero<fx2>();
                if (e < E / 2 && valid) {   // inputs x >= nx are the zero padding
                    v[e].x = __ldg(ra + t + e * TPC);
                    if (rb) v[e].y = __ldg(rb + t + e * TPC);
                }
            }
            // densities of any size to 59 bits (the sums below see only values beyond 2^32)
            const int sh = pmfx::warp_bits<E / 2>(v) - (pmfx::FX_TOP - 1);
            pmfx::shift_full<E / 2>(v, sh);
            sc.ex += sh;
        }
        sc.template measure<16>(v, 0);
        sc.apply(v, 0, fx_top<L>(0));
        fx_fft<L, false>(v, sm, lay, t, tw, sc);
        if constexpr (HALF && !INV) {
            // rows F0, F1 from their sum F0 + i F1 at k and L - k, k = 0..nx
#pragma unroll
            for (int e = 0; e < E; ++e) *mine(e) = v[e];
            __syncwarp();
            const int ex = sc.ex - 1;   // the halves of the separation
#pragma unroll 1
            for (int e = 0; e <= E / 2; ++e) {
                const int k = t + e * TPC;
                if (k > NX || !valid) break;
                const fx2 p = sm[lay(k)], q = sm[lay((L - k) & (L - 1))];
                fx2 f0, f1;
                f0.x = p.x + q.x; f0.y = p.y - q.y;
                f1.x = p.y + q.y; f1.y = q.x - p.x;
                __stcg(row + k, fx_out<true>(f0, ex));
                __stcg(row + L + k, fx_out<true>(f1, ex));
            }
            if (valid)
                for (int k = NX + 1 + t; k < kend; k += TPC) {
                    __stcg(row + k, make_double2(0.0, 0.0));
                    __stcg(row + L + k, make_double2(0.0, 0.0));
                }
            __syncwarp();   // the slots are read before the next rows' exchange
            continue;
        }
        bool sum = false;
        if constexpr (INV && !HALF) sum = ip[item][0] && !isplit[item];   // Phi_a + Phi_b beside Phi_b
#pragma unroll
        for (int e = 0; e < (INV ? E / 2 : E); ++e) {
            if (INV) v[e] = swapped(v[e]);
            if (INV && sum) v[e].x += v[e].y;
            *mine(e) = v[e];
        }
        fx_to(INV ? E / 2 : E, sc.ex, mine);
        if (valid) {
            if constexpr (INV) {
                double *phi_b = static_cast<double *>(ip[item][0]), *phi_s = static_cast<double *>(ip[item][1]) + r1 * NX;
                if (HALF) phi_b = phi_s + NX;   // the second row
                else if (phi_b) phi_b += r * NX;
#pragma unroll
                for (int e = 0; e < E / 2; ++e) {   // outputs x < nx
                    const double2 d = *reinterpret_cast<const double2 *>(mine(e));
                    __stcg(phi_s + t + e * TPC, d.x);
                    if (phi_b) __stcg(phi_b + t + e * TPC, d.y);
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    __stcg(row + t + e * TPC, *reinterpret_cast<const double2 *>(mine(e)));
            }
        }
        __syncwarp();   // the slots are read before the next row's exchange
    }
}

// ---------------------------------------------------------------------------
// y passes (as k_col): a tile of COLS columns shares one exponent.  One input
// buffer: the next tile loads while this one is transformed.
// ---------------------------------------------------------------------------
template <int L, int MODE> constexpr size_t fx_ysmem() {
    constexpr int COLS = CShape<double, L>::COLS;
    return 256 + ((size_t)pmfft::tw_dir_size(L, false) + (size_t)L * COLS + (size_t)ColRows<MODE>::of(L) * COLS) *
                     sizeof(fx2);
}

template <int L, int MODE, bool HALF> __global__ void __launch_bounds__(FXT, 3) k_yfx(const __grid_constant__ PassBatch B) {
    typedef CShape<double, L> S;
    static_assert(S::THREADS == FXT, "tile shape");
    constexpr bool INV = MODE == COL_YINV;
    constexpr int COLS = S::COLS, TPC = S::TPC, ROWS = ColRows<MODE>::of(L), NIN = INV ? E : E / 2;
    constexpr int BOXR = ROWS < 256 ? ROWS : 256, NBOX = ROWS / BOXR;
    constexpr int OROWS = INV ? L / 2 : L, OBOX = OROWS < 256 ? OROWS : 256, NOUT = INV ? E / 2 : E;
    extern __shared__ __align__(128) unsigned char smraw[];
    unsigned char *base = aligned_smem<128>(smraw);
    fx2 *in = reinterpret_cast<fx2 *>(base);
    fx2 *sm = in + ROWS * COLS;
    fxw *tw = reinterpret_cast<fxw *>(sm + L * COLS);
    __shared__ uint64_t bar;
    __shared__ int slot[2][4];   // FxScale's and, [0], the tile's exponent; this tile's and the next's
    const int tid = threadIdx.x, c = tid % COLS, t = tid / COLS;
    const int nx2 = 2 * B.a[0].nx, ny2 = 2 * B.a[0].ny;   // the items' common shape, read once
    const long long tiles_per_z = (nx2 + COLS - 1) / COLS;
    const int ltpz = __ffs((int)tiles_per_z) - 1;
    const long long ntiles = HALF ? (long long)B.n * B.tpi : (long long)B.n << B.lgi, lmask = (1LL << B.lgi) - 1;
    auto coords = [&](long long tile, int &x, int &y) {   // and the item
        if (HALF) {
            const int item = (int)tile / B.tpi, lt = (int)tile - item * B.tpi, z = lt / B.tpr;
            x = (lt - z * B.tpr) * COLS * S::EPC;
            y = z * ny2;
            return item;
        }
        const long long lt = tile & lmask;
        x = (int)((lt & (tiles_per_z - 1)) * COLS * S::EPC);
        y = (int)((lt >> ltpz) * ny2);
        return (int)(tile >> B.lgi);
    };
    auto issue = [&](long long tile) {
        int x, y;
        const CUtensorMap *map = &B.lmap[coords(tile, x, y)];
        mbar_expect_tx(&bar, (unsigned)(ROWS * COLS * sizeof(fx2)));
#pragma unroll
        for (int k = 0; k < NBOX; ++k) tma_load_2d(in + k * BOXR * COLS, map, x, y + k * BOXR, &bar);
    };
    if (tid < 8) (&slot[0][0])[tid] = (tid & 3) ? 0 : pmfx::FX_LOW;
    if (tid == 0) {
        for (int i = 0; i < B.n; ++i)
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&B.lmap[i])) : "memory");
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pmfft::expand_stage_twiddles<L, 1, false>(tw, static_cast<const fxw *>(B.a[0].tw));
    pmfft::expand_stage_twiddles<L, 2, false>(tw, static_cast<const fxw *>(B.a[0].tw));
    __syncthreads();
    pdl_wait();
    if (tid == 0 && blockIdx.x < ntiles) issue(blockIdx.x);
    const pmfft::ColLayout lay{COLS, c};
    int it = 0;
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        if (tile + gridDim.x >= ntiles) pdl_release();
        // a tensor copy that never lands: report and stop (the only copy in flight is the one waited for)
        if (!__syncthreads_and(mbar_wait(&bar, (unsigned)(it & 1)) ? 1 : 0)) {
            if (tid == 0) atomicExch(B.a[0].err, 1);
            break;
        }
        int *const sl = slot[it & 1];
        auto at = [&](int e) { return in + (t + e * TPC) * COLS + c; };
        unsigned m = 0;
#pragma unroll
        for (int e = 0; e < NIN; ++e) {
            const double2 d = *reinterpret_cast<const double2 *>(at(e));
            m = max(m, max(pmfx::dmag(d.x), pmfx::dmag(d.y)));
        }
        // the warp's own exponent and scale; the tile takes the largest
        const int em = pmfx::group_em(pmfx::warp_max(m));
        fx_from(NIN, em, at);
        fx2 v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = czero<fx2>();
            if (e < NIN) v[e] = INV ? swapped(*at(e)) : *at(e);
        }
        // (a warp of zeros, e.g. beyond the grid's columns, has no say in it)
        FxScale<true> sc{pmfx::group_zero(em) ? pmfx::FX_LOW : pmfx::group_ex(em, pmfx::FX_TOP), sl, 0};
        sc.m = pmfx::warp_max(pmfx::group_sum<16>(v));
        if ((tid & 31) == 0) atomicMax(sl, sc.ex + pmfx::sum_shift(sc.m, fx_top<L>(0)));
        fence_async_smem();                // the buffer's conversions before the next load's writes
        if (tid == 0) bulk_wait_read();    // the previous tile's outputs have been read out of sm
        __syncthreads();
        if (tid == 0 && tile + gridDim.x < ntiles) {
            fence_async_smem();
            issue(tile + gridDim.x);
        }
        if (tid < 4) slot[(it & 1) ^ 1][tid] = tid ? 0 : pmfx::FX_LOW;   // last read before the barrier
        const int tex = sl[0] == pmfx::FX_LOW ? pmfx::FX_ZERO : sl[0];   // a tile of zeros
        pmfx::shift<E>(v, tex - sc.ex);
        sc.ex = tex;
        fx_fft<L, true>(v, sm, lay, t, tw, sc);
        // fx_fft leaves the exchange buffer free: the outputs, rows t + e TPC
        auto to = [&](int e) { return sm + (t + e * TPC) * COLS + c; };
#pragma unroll
        for (int e = 0; e < NOUT; ++e) *to(e) = INV ? swapped(v[e]) : v[e];
        fx_to(NOUT, sc.ex, to);
        fence_async_smem();   // the staged outputs are visible to the tensor copies
        __syncthreads();
        if (tid == 0) {
            int x, y;
            const CUtensorMap *smap = &B.smap[coords(tile, x, y)];
#pragma unroll
            for (int k = 0; k < OROWS / OBOX; ++k) tma_store_2d(smap, x, y + k * OBOX, sm + k * OBOX * COLS);
            bulk_commit();
        }
    }
    if (tid == 0) bulk_wait_all();
}

// ---------------------------------------------------------------------------
// z pass (as k_colw; block-synchronous at every length).  DM as there; the
// second inverse of DM = 2 reads the spectrum times H-hat kept in shared
// memory.
// ---------------------------------------------------------------------------
template <int L, int DM> constexpr size_t fx_zsmem() {
    typedef WShape<double, L> S;
    return 1024 + 2 * (size_t)S::BUF + (size_t)S::COLS * S::LDR * sizeof(fx2) * (DM == 2 ? 2 : 1) +
           (size_t)pmfft::tw_dir_size(L, false) * sizeof(fxw);
}

template <int L, int DM, bool HALF>
__global__ void __launch_bounds__(FXT, DM == 2 ? 2 : 3) k_zfx(const __grid_constant__ PassBatch B) {
    typedef WShape<double, L> S;
    static_assert(S::THREADS == FXT, "tile shape");
    constexpr int TPC = S::TPC;
    extern __shared__ __align__(128) unsigned char smraw[];
    unsigned char *base = aligned_smem<1024>(smraw);
    fx2 *xch = reinterpret_cast<fx2 *>(base + 2 * S::BUF);
    fx2 *keep = DM == 2 ? xch + S::COLS * S::LDR : xch;
    fxw *tw = reinterpret_cast<fxw *>(keep + S::COLS * S::LDR);
    __shared__ uint64_t full[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int t = lane % TPC, c = warp * (32 / TPC) + lane / TPC;   // column within the tile
    const PairArgs &a = B.a[0];   // the shape, tables and mode are the items' common ones
    const int nx2 = 2 * a.nx, ny2 = 2 * a.ny, lnx2 = __ffs(nx2) - 1;
    const int lgi = B.lgi, lmask = (1 << lgi) - 1, nt = HALF ? B.n * B.tpi : B.n << lgi;
    auto locate = [&](int tile, int &q0) {   // first column, and the item
        if (HALF) {
            const int item = tile / B.tpi, lt = tile - item * B.tpi, ky = lt / B.tpr;
            q0 = (ky << lnx2) + (lt - ky * B.tpr) * S::COLS;
            return item;
        }
        q0 = (tile & lmask) * S::COLS;
        return tile >> lgi;
    };
    auto issue_load = [&](int tile, int b) {
        int q0;
        const CUtensorMap *map = &B.lmap[locate(tile, q0)];
        mbar_expect_tx(&full[b], S::BUF);
#pragma unroll
        for (int s = 0; s < S::NSUB; ++s)
#pragma unroll
            for (int k = 0; k < S::NBOXI; ++k)
                tma_load_2d(base + b * S::BUF + s * S::RIN * S::P + k * S::BOXI * S::P, map,
                            (q0 + s * S::SW) * S::EPC, k * S::BOXI, &full[b]);
    };
    auto issue_store = [&](int q0, const unsigned char *src, const CUtensorMap *map) {
#pragma unroll
        for (int s = 0; s < S::NSUB; ++s)
#pragma unroll
            for (int k = 0; k < S::NBOXI; ++k)
                tma_store_2d(map, (q0 + s * S::SW) * S::EPC, k * S::BOXI,
                             src + s * S::RIN * S::P + k * S::BOXI * S::P);
    };
    __shared__ const double *ihhat[PM_BATCH];
    if (tid < B.n) ihhat[tid] = static_cast<const double *>(B.a[tid].hhat);
    if (tid == 0) {
        for (int i = 0; i < B.n; ++i) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&B.lmap[i])) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&B.smap[i])) : "memory");
        }
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pmfft::expand_stage_twiddles<L, 1, false>(tw, static_cast<const fxw *>(a.tw));
    pmfft::expand_stage_twiddles<L, 2, false>(tw, static_cast<const fxw *>(a.tw));
    __syncthreads();
    pdl_wait();
    int issued[2] = {0, 0};   // thread 0's count of loads per buffer
    if (tid == 0) {
        if ((int)blockIdx.x < nt) { issue_load(blockIdx.x, 0); ++issued[0]; }
        if ((int)(blockIdx.x + gridDim.x) < nt) { issue_load(blockIdx.x + gridDim.x, 1); ++issued[1]; }
    }
    const pmfft::RowLayout lay{c * S::LDR};
    auto mine = [&](int e) { return xch + lay(t + e * TPC); };
    auto kept = [&](int e) { return keep + lay(t + e * TPC); };
    int it = 0;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x, ++it) {
        if (tile + (int)gridDim.x >= nt) pdl_release();
        const int b = it & 1;
        const unsigned phase = (unsigned)((it >> 1) & 1);
        if (!__syncthreads_and(mbar_wait(&full[b], phase) ? 1 : 0)) {
            // report; the other buffer's load in flight lands before the block leaves (bounded)
            if (tid == 0) {
                atomicExch(a.err, 1);
                const int o = b ^ 1, used = (it + (b == 0 ? 0 : 1)) >> 1;   // loads of buffer o consumed so far
                if (issued[o] > used) mbar_wait(&full[o], (unsigned)(used & 1));
            }
            break;
        }
        unsigned char *in = base + b * S::BUF;
        if (tid == 0 && it > 0 && tile + (int)gridDim.x < nt) {
            // the previous tile's buffer, once its store has read it
            bulk_wait_read();
            issue_load(tile + (int)gridDim.x, b ^ 1);
            ++issued[b ^ 1];
        }
        int q0;
        const int item = locate(tile, q0), q = q0 + c;   // the column
        const int ky = q >> lnx2, kx = q & (nx2 - 1);
        const int kyr = ky <= a.ny ? ky : ny2 - ky, kxr = kx <= a.nx ? kx : nx2 - kx;
        const double *hcol = ihhat[item] + ((size_t)kyr * (a.nx + 1) + kxr) * S::HS;
        auto slot_of = [&](int e) { return in + woff<double, L, S::RIN>(t + e * TPC, c); };
        // H-hat of row kz (pm_build_hhat's order): register e of the last
        // stage's order holds row kz, entry t * 16 + e of a thread-major table
        auto hval = [&](int e) {
            if constexpr (hhat_thread_major(L)) {
                constexpr int RL = radix(L, nstages(L) - 1, false), GR = E / RL;
                return __ldg(hcol + t * E + (e % GR) * RL + e / GR);
            } else {
                const int kz = t + e * TPC;
                return __ldg(hcol + (kz <= L / 2 ? kz : L - kz));
            }
        };
        fx2 v[E];
        FxScale<false> sc{0, nullptr, 0};
        {
            unsigned m = 0;
#pragma unroll
            for (int e = 0; e < E / 2; ++e) {
                const double2 d = *reinterpret_cast<const double2 *>(slot_of(e));
                m = max(m, max(pmfx::dmag(d.x), pmfx::dmag(d.y)));
            }
            const int em = pmfx::group_em(pmfx::warp_max(m));
            sc.ex = pmfx::group_ex(em, pmfx::FX_TOP);
            fx_from(E / 2, em, slot_of);
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = e < E / 2 ? *reinterpret_cast<const fx2 *>(slot_of(e)) : czero<fx2>();
        }
        // the largest H-hat of the warp's columns
        unsigned hm = 0;
#pragma unroll 4
        for (int e = 0; e < E; ++e) hm = max(hm, pmfx::dmag(hval(e)));
        const int hem = pmfx::group_em(pmfx::warp_max(hm));
        int kex = 0;   // exponent of the kept spectrum
#pragma unroll 1
        for (int j = 0; j < (DM == 2 ? 3 : 2); ++j) {
            sc.template measure<16>(v, 0);
            sc.apply(v, 0, fx_top<L>(0));
            fx_fft<L, false>(v, xch, lay, t, tw, sc);
            if (j > 0) {
                // inverse outputs, rows below L/2, staged in the tile's buffer
#pragma unroll
                for (int e = 0; e < E / 2; ++e) *reinterpret_cast<fx2 *>(slot_of(e)) = swapped(v[e]);
                fx_to(E / 2, sc.ex, slot_of);
                fence_async_smem();   // the staged outputs are visible to the tensor copies
                __syncthreads();
                const bool last = DM != 2 || j == 2;
                if (tid == 0) {
                    // DM = 2: fx + i fy through smap, then fz + i Phi in place through lmap
                    issue_store(q0, in, DM == 2 && last ? &B.lmap[item] : &B.smap[item]);
                    bulk_commit();
                    if (!last) bulk_wait_read();   // read out before the second outputs overwrite the buffer
                }
                if (last) break;
                __syncthreads();
            } else {
                // spectrum times H-hat
#pragma unroll
                for (int e = 0; e < E; ++e) *kept(e) = v[e];
                unsigned m = 0;
#pragma unroll 2
                for (int e = 0; e < E; ++e) {
                    int h, l;
                    pmfx::split(pmfx::from_double<pmfx::FX_Q>(hval(e), hem), h, l);
                    fx2 w = *kept(e);
                    w.x = pmfx::mulr(w.x, h, l);
                    w.y = pmfx::mulr(w.y, h, l);
                    *kept(e) = w;
                    m = max(m, (unsigned)max(abs((int)(w.x >> 32)), abs((int)(w.y >> 32))));
                }
                kex = sc.ex + pmfx::factor_ex(hem);
                if constexpr (DM != 0) {   // components below 2^59: the difference factors' moduli reach sqrt(2)
                    const int sh = 64 - __clz((int)pmfx::warp_max(m + 1)) - (pmfx::FX_TOP - 1);
#pragma unroll 2
                    for (int e = 0; e < E; ++e) {
                        fx2 w[1] = {*kept(e)};
                        pmfx::shift<1>(w, sh);
                        *kept(e) = w[0];
                    }
                    kex += sh;
                }
            }
            // inputs of the next inverse: the spectrum times 1, D_x + i D_y or D_z + i
            sc.ex = kex;
            if constexpr (DM != 0) {
                if (DM == 2 ? j == 0 : a.dmode == 1) {
                    const double2 dx = static_cast<const double2 *>(a.dtx)[kx], dy = static_cast<const double2 *>(a.dty)[ky];
                    const double fr = dx.x - dy.y, fi = dx.y + dy.x;
                    const int em = pmfx::group_em(pmfx::warp_max(max(pmfx::dmag(fr), pmfx::dmag(fi))));
                    fxw f;
                    pmfx::wsplit(pmfx::from_double<pmfx::FX_Q>(fr, em), f.rh, f.rl);
                    pmfx::wsplit(pmfx::from_double<pmfx::FX_Q>(fi, em), f.ih, f.il);
#pragma unroll 2
                    for (int e = 0; e < E; ++e) *mine(e) = cmul(*kept(e), f);
                    sc.ex += pmfx::factor_ex(em);
                } else {
                    // D_z + i in units of 2^-59, the second half of D's table
                    const longlong2 *dz = static_cast<const longlong2 *>(a.dtz) + L;
#pragma unroll 2
                    for (int e = 0; e < E; ++e) {
                        const longlong2 f = dz[t + e * TPC];
                        *mine(e) = pmfx::cmulq(*kept(e), f.x, f.y);
                    }
                    sc.ex += 1;
                }
            }
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = swapped(*mine(e));
            __syncwarp();   // read before the exchange writes
        }
    }
    if (tid == 0) bulk_wait_all();
}

}  // namespace pmk
