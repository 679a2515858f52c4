// The FP64 hopping term in block fixed-point arithmetic (dslash_fx.cuh):
// kernels, launch table and the conversion of the links.
#include "dslash_fx.cuh"

namespace wd {
namespace {

// the epilogue of one complex component (plane j, spin s) at site h: out =
// scale H in, or x + scale H in, in FP64 operations as in k_dslash<double>
template <int EPI>
__device__ __forceinline__ double2 fx_store(const DslashArgs<double> &a, long h, int cc, int s,
                                            double vr, double vi) {
    const long at = ((long)(4 * cc + s) * a.g.stride + h) * 16;
    const double ts = s < 2 ? a.twist : -a.twist;   // spins 0, 1: 1 + i t, spins 2, 3: 1 - i t
    double2 o;
    if (EPI == EPI_XPAY) {
        double2 x = ld_nc_d2((const char *)a.x + at);
        if (a.twist_on) x = make_double2(x.x - ts * x.y, x.y + ts * x.x);
        o = make_double2(x.x + a.scale * vr, x.y + a.scale * vi);
    } else {
        o = make_double2(a.scale * vr, a.scale * vi);
        if (a.twist_on) o = make_double2(o.x + ts * o.y, o.y - ts * o.x);
    }
    *reinterpret_cast<double2 *>((char *)a.out + at) = o;
    return o;
}

// The fused norm: |out|^2 per spin in FP64, the four spins and then the 32
// sites of the block's partial in double-float.  Five blocks per SM: 96
// registers; with four (122) or six (80, spilling) it is 8 to 15 % slower at
// 16^3 x 32 and above, so the kernel is not tuned per handle.
template <int EPI, int NORM>
__global__ void __launch_bounds__(FX_BLOCK, 5) k_dslash_fx(const __grid_constant__ FxArgs A) {
    __shared__ FxShared sh;
    const DslashArgs<double> &a = A.d;
    // (the shuffle tells the compiler that the warp index is uniform)
    const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const long hs = a.h0 + (long)blockIdx.x * FX_SITES + lane;
    const long h = hs < a.h1 ? hs : a.h1 - 1;
    double v[6];
    fx_site(A, (unsigned)h, w, sh, v);
    double sq = 0;
    if (hs < a.h1) {
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            const double2 o = fx_store<EPI>(a, h, cc, w, v[2 * cc], v[2 * cc + 1]);
            if (NORM) sq += o.x * o.x + o.y * o.y;
        }
    }
    if (NORM) {
        __shared__ df64 ws[4][32];
        ws[w][lane] = to_df(sq);
        __syncthreads();
        if (w == 0) {
            const df64 s = warp_sum(((ws[0][lane] + ws[1][lane]) + ws[2][lane]) + ws[3][lane]);
            if (lane == 0) a.red.partials[blockIdx.x] = s;
        }
    }
}

template <int EPI, int NORM>
__global__ void __launch_bounds__(FXW_BLOCK, 1) k_dslash_fx_wide(const __grid_constant__ FxArgs A) {
    __shared__ FxWideShared sh;
    const DslashArgs<double> &a = A.d;
    const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const long hs = a.h0 + (long)blockIdx.x * FX_SITES + lane;
    const long h = hs < a.h1 ? hs : a.h1 - 1;
    double v[2];
    fx_site_wide(A, (unsigned)h, w, sh, v);
    double sq = 0;
    if (w < 12 && hs < a.h1) {
        const double2 o = fx_store<EPI>(a, h, w >> 2, w & 3, v[0], v[1]);
        if (NORM) sq = o.x * o.x + o.y * o.y;
    }
    if (NORM) {
        __shared__ df64 ws[12][32];
        if (w < 12) ws[w][lane] = to_df(sq);
        __syncthreads();
        if (w == 0) {
            df64 t = ws[0][lane];
#pragma unroll
            for (int j = 1; j < 12; ++j) t = t + ws[j][lane];
            t = warp_sum(t);
            if (lane == 0) a.red.partials[blockIdx.x] = t;
        }
    }
}

template <int EPI, int NORM>
void launch_fx(const FxArgs &A, bool wide, cudaStream_t s) {
    const long n = A.d.h1 - A.d.h0;
    if (wide) {
        k_dslash_fx_wide<EPI, NORM><<<(unsigned)((n + FX_SITES - 1) / FX_SITES), FXW_BLOCK, 0, s>>>(A);
        return;
    }
    k_dslash_fx<EPI, NORM><<<(unsigned)((n + FX_SITES - 1) / FX_SITES), FX_BLOCK, 0, s>>>(A);
}

// Fixed-point links of one parity from its FP64 records: one thread per (site,
// direction).  With m = max(max |u|, the largest sum of absolute values of a
// row's or a column's six reals over 2.46): eu = 0 for 1/8 < m <= 1 (SU(3): at
// most sqrt(6) / 2.46 = 0.9957), else the exponent with m in (2^(eu - 1), 2^eu].
template <int RECON>
__global__ void __launch_bounds__(128)
k_gauge_fx(Geom g, const char *links, size_t dir_bytes, char *fx, size_t fx_dir_bytes,
           int16_t *ex, int *any_exp) {
    const long i = (long)blockIdx.x * 128 + threadIdx.x;
    if (i >= 4 * g.vh) return;
    const int mu = (int)(i / g.vh);
    const long site = i - mu * g.vh;
    double U[18];
    load_link<double, double, RECON>(links + mu * dir_bytes, g.stride, site, U);
    double mx = 0, row[3] = {}, col[3] = {};
    bool finite = true;
#pragma unroll
    for (int k = 0; k < 18; ++k) {
        const double u = fabs(U[k]);
        finite = finite && isfinite(u);
        mx = fmax(mx, u);
        row[k / 6] += (1 / 2.46) * u;
        col[(k / 2) % 3] += (1 / 2.46) * u;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) mx = fmax(mx, fmax(row[k], col[k]));
    finite = finite && isfinite(mx);
    int eu = 0;
    if (!finite) eu = FX_BAD_EXP;
    else if (mx > 1.0 || mx <= 0.125) {
        if (mx != 0.0) {
            const double m = frexp(mx, &eu);   // mx = m 2^eu, m in [1/2, 1)
            if (m == 0.5) eu -= 1;
        }
        if (eu < -FX_LINK_EXP || eu > FX_LINK_EXP) eu = FX_BAD_EXP;
    }
    if (eu != 0) atomicOr(any_exp, 1);
    ex[(size_t)mu * g.stride + site] = (int16_t)eu;
    char *dst = fx + mu * fx_dir_bytes + site * 16;
#pragma unroll
    for (int e = 0; e < FX_PLANES; ++e) {
        uint32_t w[4];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const long long F = eu == FX_BAD_EXP ? 0ll : __double2ll_rn(ldexp(U[2 * e + p], 62 - eu));
            const int u0 = (int)F;
            w[2 * p] = (uint32_t)u0;
            w[2 * p + 1] = (uint32_t)((F - u0) >> 32);
        }
        st_v4(dst + (long)e * g.stride * 16, make_uint4(w[0], w[1], w[2], w[3]));
    }
}

}  // namespace

cudaError_t launch_gauge_fx(const GaugeSet &gs, const Geom &g, cudaStream_t s) {
    if (gs.prec != WD_F64 || !gs.fx[0] || !gs.fx[1]) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(gs.any_exp, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((4 * g.vh + 127) / 128);
    for (int p = 0; p < 2; ++p) {
        if (gs.recon == 12)
            k_gauge_fx<12><<<grid, 128, 0, s>>>(g, (const char *)gs.ptr[p], gs.dir_bytes,
                                                (char *)gs.fx[p], gs.fx_dir_bytes, gs.fx_exp[p],
                                                gs.any_exp);
        else
            k_gauge_fx<18><<<grid, 128, 0, s>>>(g, (const char *)gs.ptr[p], gs.dir_bytes,
                                                (char *)gs.fx[p], gs.fx_dir_bytes, gs.fx_exp[p],
                                                gs.any_exp);
    }
    return cudaGetLastError();
}

cudaError_t launch_dslash_fx(const DslashLaunch &L, cudaStream_t s) {
    const GaugeSet &gs = *L.gauge;
    if (!gs.fx[0]) return cudaErrorInvalidValue;
    FxArgs A;
    cudaError_t e = fill_dslash_args<double>(L, A.d);
    if (e != cudaSuccess) return e;
    if (A.d.h1 == A.d.h0) return cudaSuccess;
    A.recon = gs.recon;
    A.dagger = L.dagger;
    const int q = 1 - L.out_parity;
    A.fx_out = (const char *)gs.fx[L.out_parity];
    A.fx_in = (const char *)gs.fx[q];
    A.fx_dir_bytes = gs.fx_dir_bytes;
    A.ex_out = gs.fx_exp[L.out_parity];
    A.ex_in = gs.fx_exp[q];
    A.any_exp = gs.any_exp;
    if (L.red) {
        launch_fx<EPI_XPAY, 1>(A, gs.fx_wide, s);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return launch_finish_partials(*L.red, (L.g.vh + 31) / 32, s);
    }
    if (L.epi == EPI_PLAIN) launch_fx<EPI_PLAIN, 0>(A, gs.fx_wide, s);
    else launch_fx<EPI_XPAY, 0>(A, gs.fx_wide, s);
    return cudaGetLastError();
}

}  // namespace wd
