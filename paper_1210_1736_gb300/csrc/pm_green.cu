// H-hat, the DFT of the even-extended Green's function (Sec. 2.1,
// Eq. eqn:greens and eq:symmetry), in the z pass's table order.
//
// H is known on the (nx+1)(ny+1)(nz+1) octant; its doubled-grid extension is
// even along every axis, so its DFT is real, even and separable: per axis the
// transform of length L = 2n of the even extension of n + 1 values.  Two
// columns travel as one complex transform (both results are real) in the fixed
// point of pm_fx.cuh; the first axis evaluates H, the last writes the table.
// For 128 x 128 x 32 in FP32 the three launches take 22, 15 and 17 us (the
// first bound by H's FP64 operations: 31 us before the ones that integer or FP32
// operations replace exactly were taken out) where H took 22 us, dense FP64
// cosine sums, bound by the FP64 pipe, 125 + 127 + 35 us and the table 9 us.  H-hat
// is also more exact: the FP64 potentials' error fell to a half or a third.
#include <cuda_runtime.h>

#include "pm_passes_fx.cuh"
#include "pm_roots.cuh"

namespace {

using pmfft::E;

struct HatArgs {
    double *h;               // [nz+1][ny+1][nx+1]
    void *out;               // the table (last axis)
    const fxw *tw;           // exp(-2 pi i m / 512), m < 512
    long long ncol, inner;   // columns along the axis; element stride
    int ny1;                 // ny + 1 (first axis)
    double q, h000, scale;
};

// AX 0: evaluate H, transform along x; 1: along y; 2: along z, then scale into
// T and store in the table's order (see pm_build_hhat).
template <int L, int AX, typename T> __global__ void __launch_bounds__(pmk::FXT, 3) k_hat_axis(HatArgs a) {
    constexpr int TPC = L / E, N = L / 2, LDR = L + L / 16;
    extern __shared__ __align__(16) unsigned char smraw[];
    fxw *tw = reinterpret_cast<fxw *>(smraw);
    fx2 *sm = reinterpret_cast<fx2 *>(tw + pmfft::tw_dir_size(L, false));
    const int tid = threadIdx.x, line = tid / TPC, t = tid % TPC;
    pmfft::expand_stage_twiddles<L, 1, false, 512 / L>(tw, a.tw);
    pmfft::expand_stage_twiddles<L, 2, false, 512 / L>(tw, a.tw);
    __syncthreads();
    const long long col = 2 * ((long long)blockIdx.x * (blockDim.x / TPC) + line);
    const bool va = col < a.ncol, vb = col + 1 < a.ncol;
    const pmfft::RowLayout lay{line * LDR};
    auto base = [&](long long c) { return a.h + (AX == 0 ? c * (N + 1) : (c / a.inner) * (N + 1) * a.inner + c % a.inner); };
    double *ha = base(va ? col : 0), *hb = base(vb ? col + 1 : 0);
    const long long stride = AX == 0 ? 1 : a.inner;
    // rows t + e TPC <= N of the two columns
    auto mine = [&](int e) { return sm + lay(t + e * TPC); };
    const int cnt = t == 0 ? E / 2 + 1 : E / 2;
    // first axis: a column's squared distance from the axis in its two parts
    int jj[2] = {0, 0};
    double kk[2] = {0.0, 0.0};
    if constexpr (AX == 0)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int c = (int)col + w, k = c / a.ny1, j = c - k * a.ny1;
            const double qk = a.q * (double)k;
            jj[w] = j * j;
            kk[w] = qk * qk;
        }
    const float kf[2] = {(float)kk[0], (float)kk[1]};
    unsigned m = 0;
#pragma unroll 3
    for (int e = 0; e < cnt; ++e) {
        const int i = t + e * TPC;
        double2 d = make_double2(0.0, 0.0);
        if constexpr (AX == 0) {
            auto green = [&](int w) {
                const int n = i * i + jj[w];   // exact in FP32
                return i == 0 && col + w == 0 ? a.h000 : pmroot::inv_sqrt((double)n + kk[w], (float)n + kf[w]);
            };
            if (va) d.x = green(0);
            if (vb) d.y = green(1);
        } else {
            if (va) d.x = ha[i * stride];
            if (vb) d.y = hb[i * stride];
        }
        m = max(m, max(pmfx::dmag(d.x), pmfx::dmag(d.y)));
        *reinterpret_cast<double2 *>(mine(e)) = d;
    }
    const int em = pmfx::group_em(pmfx::warp_max(m));
    pmk::fx_from(cnt, em, mine);
    __syncwarp();
    fx2 v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int r = t + e * TPC;
        v[e] = sm[lay(r <= N ? r : L - r)];   // the even extension
    }
    __syncwarp();
    pmk::FxScale<false> sc{pmfx::group_ex(em, pmfx::FX_TOP), nullptr, 0};
    sc.template measure<16>(v, 0);
    sc.apply(v, 0, pmk::fx_top<L>(0));
    pmk::fx_fft<L, false>(v, sm, lay, t, tw, sc);
#pragma unroll
    for (int e = 0; e <= E / 2; ++e)
        if (e < cnt) *mine(e) = v[e];
    pmk::fx_to(cnt, sc.ex, mine);
    if constexpr (AX < 2) {
        for (int e = 0; e < cnt; ++e) {
            const double2 d = *reinterpret_cast<const double2 *>(mine(e));
            const long long o = (t + e * TPC) * stride;
            if (va) ha[o] = d.x;
            if (vb) hb[o] = d.y;
        }
    } else {
        constexpr int HS = pm_hhat_stride(L);
        T *oa = static_cast<T *>(a.out) + col * HS, *ob = oa + HS;
        auto put = [&](int w, double2 d) {
            if (va) oa[w] = (T)(d.x * a.scale);
            if (vb) ob[w] = (T)(d.y * a.scale);
        };
        // thread-major tables hold all L values: register e of thread t (last
        // stage's order) at t * 16 + e
        auto slot = [&](int kz) {
            constexpr int RL = pmfft::radix(L, pmfft::nstages(L) - 1, false);
            return kz % TPC * E + kz / TPC % (E / RL) * RL + kz / (L / RL);
        };
        for (int e = 0; e < cnt; ++e) {
            const double2 d = *reinterpret_cast<const double2 *>(mine(e));
            const int kz = t + e * TPC;
            if constexpr (pmk::hhat_thread_major(L)) {
                put(slot(kz), d);
                if (kz > 0 && kz < N) put(slot(L - kz), d);
            } else {
                put(kz, d);
            }
        }
        if constexpr (!pmk::hhat_thread_major(L))
            for (int w = N + 1 + t; w < HS; w += TPC) put(w, make_double2(0.0, 0.0));   // padding
    }
}

template <int L, int AX, typename T> cudaError_t launch_axis(const HatArgs &a, cudaStream_t st) {
    constexpr int TPC = L / E, LDR = L + L / 16;
    // Fewer warps than the SMs have schedulers: blocks of one warp, which spread
    // over more SMs (whole calls of pm_potential_static, one after another, 32 /
    // 128 threads: FP32 8 x 8 x 128 55.6 / 59.5 us, 8 x 256 x 8 61.9 / 66.1, 64 x
    // 64 x 32 68.9 / 71.1, 16 x 16 x 256 70.7 / 68.1).  From there on both
    // measure the same (128 x 64 x 32 77.9 us).
    const int threads = a.ncol / 2 * TPC < 32LL * 4 * pmk_host::num_sms() ? 32 : pmk::FXT;
    const size_t smem = ((size_t)pmfft::tw_dir_size(L, false) + (size_t)threads / TPC * LDR) * sizeof(fx2);
    static_assert(((size_t)pmfft::tw_dir_size(L, false) + (size_t)pmk::FXT / TPC * LDR) * sizeof(fx2) <= 48 << 10, "no opt-in");
    const long long lines = (a.ncol + 1) / 2, per = threads / TPC;
    k_hat_axis<L, AX, T><<<(unsigned)((lines + per - 1) / per), threads, smem, st>>>(a);
    return cudaGetLastError();
}
template <int AX, typename T> cudaError_t axis(int n, const HatArgs &a, cudaStream_t st) {
    switch (n) {
        case 8: return launch_axis<16, AX, T>(a, st);
        case 16: return launch_axis<32, AX, T>(a, st);
        case 32: return launch_axis<64, AX, T>(a, st);
        case 64: return launch_axis<128, AX, T>(a, st);
        case 128: return launch_axis<256, AX, T>(a, st);
        case 256: return launch_axis<512, AX, T>(a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

template <typename T>
cudaError_t pm_build_hhat(double *h, T *out, const fxw *tw, int nx, int ny, int nz, double q, double h000, double scale,
                          cudaStream_t st) {
    HatArgs a;
    a.h = h;
    a.out = out;
    a.tw = tw;
    a.ny1 = ny + 1;
    a.q = q;
    a.h000 = h000;
    a.scale = scale;
    a.ncol = (long long)(nz + 1) * (ny + 1);
    a.inner = 1;
    cudaError_t e = axis<0, double>(nx, a, st);
    if (e != cudaSuccess) return e;
    a.ncol = (long long)(nz + 1) * (nx + 1);
    a.inner = nx + 1;
    if ((e = axis<1, double>(ny, a, st)) != cudaSuccess) return e;
    a.ncol = a.inner = (long long)(ny + 1) * (nx + 1);
    return axis<2, T>(nz, a, st);
}
template cudaError_t pm_build_hhat<float>(double *, float *, const fxw *, int, int, int, double, double, double, cudaStream_t);
template cudaError_t pm_build_hhat<double>(double *, double *, const fxw *, int, int, int, double, double, double, cudaStream_t);
