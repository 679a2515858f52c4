// The other Krylov solvers of the paper's solver comparison (Sec. 5, Fig.
// "algosxp": CGNR, CRNE, MCR1 and MCR2, all on the Schur-reduced system),
// which the paper names but does not define.  Textbook readings:
//
//   CR (Saad, "Iterative Methods for Sparse Linear Systems", 2nd ed., Alg.
//   6.20) on a Hermitian B y = c minimises ||c - B y|| over K_k(B, c):
//     alpha = (r|B r) / (Bp|Bp),  y += alpha p,  r -= alpha Bp,
//     beta = (r'|B r') / (r|B r), p = r' + beta p, Bp = B r' + beta Bp.
//   CRNE: B = A A^dag, x = A^dag y.  Tracked here through x itself:
//     s = A^dag r, t = A s = B r, q = A^dag p, w = A q = B p, (r|B r) = |s|^2,
//     so x += alpha q and q = s + beta q replace the updates of y and p.
//   MCR1/MCR2: B = gamma5 A, c = gamma5 b.  gamma5 A is Hermitian because
//     A^dag = gamma5 A gamma5 (Fig. "id"); with a twisted mass that identity
//     fails (gamma5 A(mu) gamma5 = A(-mu)^dag), so MCR needs mu = 0.  MCR1
//     forms B p with the operator each iteration (two applications of A),
//     MCR2 by the recurrence (one).
//   CGNR: Alg. "CGNR", in the same host-driven form, so that the four
//     methods are compared with the same vector kernels.
// A = Mhat_p, the Schur operator of the op (Alg. "schur"), applied in FP64; x,
// r and every direction are half-lattice fields in the operator's FP64 storage
// layout (plane j of a field holds complex number j = 4 colour + spin of every
// site), so that an application is two hopping terms and nothing else.  Every
// inner product sums in FP64; the coefficients are formed on the device by the
// sums' last block, and the host reads |r|^2 once per iteration, while the
// direction update runs.  (Canonical fields, with a pack and an unpack per
// application and a host round trip per inner product: MCR2 on 16^3 x 32 took
// 27.3 ms, now 16.9.)  The solve wraps the method in the Schur preparation
// and reconstruction and accepts x only on the FP64 true residual of the full
// system; if the recursive residual met the target but the true one does not,
// the method restarts from the current x with an explicitly computed residual.
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "op.cuh"

namespace wd {

constexpr int KR_BLOCK = 256;
constexpr int KR_PLANES = 12;   // complex numbers of a site's spinor
// Two blocks per SM of a GB300, the same number for every plane (16^3 x 32, an
// iteration's sum over r and Br: 16 us with 300 blocks, 19 with 612 and 1224).
constexpr int KR_BLOCKS = 300;

// A field's entries: plane j = blockIdx.y of `vh` numbers, `stride` apart.
// (A canonical array of n numbers is read as 12 planes of n / 12.)
struct KrShape {
    long vh, stride;
};
#define KR_EACH(sh, i)                                                                      \
    _Pragma("unroll 2")                                                                     \
    for (long i = (long)blockIdx.y * sh.stride + (long)blockIdx.x * KR_BLOCK + threadIdx.x, \
              end_ = (long)blockIdx.y * sh.stride + sh.vh;                                  \
         i < end_; i += (long)gridDim.x * KR_BLOCK)

// gamma5 of the DeGrand-Rossi basis is diag(1, 1, -1, -1); spin is the
// fastest part of the plane index
__device__ __forceinline__ double kr_g5() { return (blockIdx.y & 3) < 2 ? 1.0 : -1.0; }

// The method's scalars, on the device, mirrored to the host by the sums that
// the host reads.
struct KrScalars {
    double rho = 0.0;     // CGNR, CRNE: |A^dag r|^2; MCR: Re (r|B r)
    double rr = 0.0;      // |r|^2
    double alpha = 0.0, beta = 0.0;
    int bad = 0;          // no alpha: the step leaves x and r as they are
};

// What the last block makes of the two sums
enum KrFinish {
    KR_START,   // rho = s0, rr = s1
    KR_ALPHA,   // alpha = rho / s0, s0 = |A p|^2 or |B p|^2
    KR_BETA,    // beta = s0 / rho, then as KR_START
    KR_SUM      // rr = s0
};

struct KrRed {
    double2 *partials;       // [KR_BLOCKS]
    unsigned int *counter;
    KrScalars *sc, *host;    // host: mapped
    int fin, cr;             // cr: rho = 0 is a breakdown too
};

// Sums of s0 and, if TWO, s1 over the grid in a fixed order; every thread of
// every block calls it.  The two sums share a warp's butterfly after its first
// step (lanes 0-15 go on with s0, the others with s1): an FP64 addition of a
// warp takes the pipe 16 clocks.
template <bool TWO>
__device__ __forceinline__ void kr_block_sum(double &s0, double &s1, double2 *ws) {
    const int lane = threadIdx.x & 31;
    double v = s0;
    if (TWO) {
        const double give = lane < 16 ? s1 : s0;
        v = lane < 16 ? s0 : s1;
        v += __shfl_xor_sync(0xffffffffu, give, 16);
    } else {
        v += __shfl_xor_sync(0xffffffffu, v, 16);
    }
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) ws[threadIdx.x >> 5].x = v;
    if (TWO && lane == 16) ws[threadIdx.x >> 5].y = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        s0 = ws[0].x;
        if (TWO) s1 = ws[0].y;
        for (int w = 1; w < KR_BLOCK / 32; ++w) {
            s0 += ws[w].x;
            if (TWO) s1 += ws[w].y;
        }
    }
}

template <bool TWO>
__device__ __forceinline__ void kr_reduce(const KrRed &red, double s0, double s1) {
    __shared__ double2 ws[KR_BLOCK / 32];
    __shared__ bool last;
    const int blocks = gridDim.x * gridDim.y;
    kr_block_sum<TWO>(s0, s1, ws);
    if (threadIdx.x == 0) {
        red.partials[blockIdx.y * gridDim.x + blockIdx.x] = make_double2(s0, s1);
        __threadfence();
        last = atomicAdd(red.counter, 1u) == (unsigned)blocks - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    s0 = s1 = 0.0;
    for (int i = threadIdx.x; i < blocks; i += KR_BLOCK) {
        const double2 v = __ldcg(red.partials + i);
        s0 += v.x;
        if (TWO) s1 += v.y;
    }
    __syncthreads();   // ws
    kr_block_sum<TWO>(s0, s1, ws);
    if (threadIdx.x != 0) return;
    *red.counter = 0;
    KrScalars c = *red.sc;
    if (red.fin == KR_ALPHA) {
        c.bad = !(s0 > 0.0) || !isfinite(c.rho) || (red.cr && c.rho == 0.0);
        c.alpha = c.bad ? 0.0 : c.rho / s0;
    } else if (red.fin == KR_SUM) {
        c.rr = s0;
    } else {
        if (red.fin == KR_BETA) c.beta = s0 / c.rho;
        c.rho = s0;
        c.rr = s1;
    }
    *red.sc = c;
    if (red.fin != KR_ALPHA) *red.host = c;   // the host reads nothing after KR_ALPHA
}

// <a0, b0> and, when a1 != nullptr, <a1, b1> (real parts).  Of the imaginary
// parts, which no method uses, and separate products and sums came 12 FP64
// operations per pair of entries where 4 do (24 -> 13 us on 16^3 x 32, with
// twice the entries here).
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_dot2(KrShape sh, const double2 *__restrict__ a0, const double2 *__restrict__ b0,
          const double2 *__restrict__ a1, const double2 *__restrict__ b1, const KrRed red) {
    double s0 = 0.0, s1 = 0.0;
    KR_EACH(sh, i) {
        const double2 x = a0[i], y = b0[i];
        s0 = fma(x.x, y.x, fma(x.y, y.y, s0));
        if (a1) {
            const double2 u = a1[i], v = b1[i];
            s1 = fma(u.x, v.x, fma(u.y, v.y, s1));
        }
    }
    kr_reduce<true>(red, s0, s1);
}

// f = gamma5 f with <r, f> and |r|^2 of the result, or |f|^2 when r is null.
// <r, gamma5 A r> is a small difference of two large sums, and the method
// divides by it: a thread takes the planes of spins s and s + 2 together (six
// pairs in blockIdx.y), so that the terms cancel before they are added up.
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_g5_dot(KrShape sh, double2 *__restrict__ f, const double2 *__restrict__ r, const KrRed red) {
    double s0 = 0.0, s1 = 0.0;
    const long plane = (long)((blockIdx.y >> 1) * 4 + (blockIdx.y & 1)) * sh.stride;
#pragma unroll 2
    for (long h = (long)blockIdx.x * KR_BLOCK + threadIdx.x; h < sh.vh;
         h += (long)gridDim.x * KR_BLOCK) {
        const long i = plane + h, j = i + 2 * sh.stride;
        const double2 v = f[i];
        double2 w = f[j];
        w.x = -w.x;
        w.y = -w.y;
        f[j] = w;
        const double2 u = r ? r[i] : v, t = r ? r[j] : w;
        s0 = fma(u.x, v.x, fma(t.x, w.x, fma(u.y, v.y, fma(t.y, w.y, s0))));
        if (r) s1 = fma(u.x, u.x, fma(t.x, t.x, fma(u.y, u.y, fma(t.y, t.y, s1))));
    }
    kr_reduce<true>(red, s0, s1);
}

// x += alpha p;  r -= alpha w
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_step(KrShape sh, const KrScalars *__restrict__ sc, double2 *__restrict__ x,
          const double2 *__restrict__ p, double2 *__restrict__ r, const double2 *__restrict__ w) {
    if (sc->bad) return;
    const double alpha = sc->alpha;
    KR_EACH(sh, i) {
        const double2 pv = p[i], wv = w[i];
        double2 xv = x[i], rv = r[i];
        xv.x += alpha * pv.x; xv.y += alpha * pv.y;
        rv.x -= alpha * wv.x; rv.y -= alpha * wv.y;
        x[i] = xv;
        r[i] = rv;
    }
}

// q = s + beta q
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_dir(KrShape sh, const KrScalars *__restrict__ sc, double2 *__restrict__ q,
         const double2 *__restrict__ s) {
    const double beta = sc->beta;
    KR_EACH(sh, i) {
        const double2 sv = s[i];
        double2 qv = q[i];
        qv.x = sv.x + beta * qv.x; qv.y = sv.y + beta * qv.y;
        q[i] = qv;
    }
}

// q = s + beta q, w = t + beta w and |w|^2 (the next iteration's |B p|^2)
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_dir2(KrShape sh, double2 *__restrict__ q, const double2 *__restrict__ s,
          double2 *__restrict__ w, const double2 *__restrict__ t, const KrRed red) {
    const double beta = red.sc->beta;
    double s0 = 0.0;
    KR_EACH(sh, i) {
        const double2 sv = s[i], tv = t[i];
        double2 qv = q[i], wv = w[i];
        qv.x = sv.x + beta * qv.x; qv.y = sv.y + beta * qv.y;
        wv.x = tv.x + beta * wv.x; wv.y = tv.y + beta * wv.y;
        q[i] = qv;
        w[i] = wv;
        s0 = fma(wv.x, wv.x, fma(wv.y, wv.y, s0));
    }
    kr_reduce<false>(red, s0, 0.0);
}

// out = g (a + c b), g = gamma5 when g5 != 0, else 1 (out may alias a or b)
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_comb(KrShape sh, double2 *out, const double2 *a, double c, const double2 *b, int g5) {
    KR_EACH(sh, i) {
        double2 v = a[i];
        if (b) {
            const double2 bv = b[i];
            v.x += c * bv.x; v.y += c * bv.y;
        }
        if (g5 && kr_g5() < 0.0) { v.x = -v.x; v.y = -v.y; }
        out[i] = v;
    }
}

// v = c (1 + i s gamma5) v (the twisted-mass block A = 1 + i t gamma5 and its
// inverse (1 - i t gamma5) / (1 + t^2))
__global__ void __launch_bounds__(KR_BLOCK)
k_kr_twist(KrShape sh, double2 *v, double s, double c) {
    const double sg = s * kr_g5();
    KR_EACH(sh, i) {
        const double2 a = v[i];
        v[i] = make_double2(c * (a.x - sg * a.y), c * (a.y + sg * a.x));
    }
}

}  // namespace wd

using namespace wd;

static thread_local std::string g_kr_error;
static int kr_fail(int code, const std::string &m) {
    g_kr_error = m;
    return code;
}
#define KR_CUDA(call)                                                                       \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return kr_fail(e_ == cudaErrorMemoryAllocation ? WD_ERR_NOMEM : WD_ERR_CUDA,    \
                           std::string(#call) + ": " + cudaGetErrorString(e_));             \
    } while (0)
#define KR_TRY(call)                                                                        \
    do {                                                                                    \
        int rc_ = (call);                                                                   \
        if (rc_ != WD_OK) {                                                                 \
            if (g_kr_error.empty()) g_kr_error = wd_last_error();                           \
            return rc_;                                                                     \
        }                                                                                   \
    } while (0)

struct wd_krylov {
    wd_op *op = nullptr;
    int method = 0;
    KrShape half{}, whole{};         // half-lattice fields; canonical full-lattice ones
    double2 *x = nullptr, *r = nullptr, *f[4] = {}, *bh = nullptr, *bq = nullptr;
    double2 *full = nullptr;         // canonical full-lattice work field
    double2 *partials = nullptr;
    unsigned int *counter = nullptr;
    KrScalars *sc = nullptr;         // device
    KrScalars *sc_host = nullptr, *sc_host_dev = nullptr;   // pinned, mapped
    cudaEvent_t ev = nullptr;        // a sum that the host reads
    std::vector<void *> allocs;
    long launches = 0;               // kernels queued by the current solve
    long applies = 0;                // Schur-operator applications of the current solve
};

static int kr_alloc(wd_krylov *s, void **p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return kr_fail(WD_ERR_NOMEM, "cudaMalloc failed");
    }
    s->allocs.push_back(*p);
    KR_CUDA(cudaMemset(*p, 0, bytes));
    return WD_OK;
}

static cudaStream_t kr_stream(const wd_krylov *s) { return s->op->stream; }

#define KR_LAUNCH(s, kernel, ...) KR_LAUNCH_ON(s, KR_PLANES, kernel, __VA_ARGS__)
#define KR_LAUNCH_ON(s, planes, kernel, ...)                                                \
    do {                                                                                    \
        kernel<<<dim3(KR_BLOCKS / (planes), planes), KR_BLOCK, 0, kr_stream(s)>>>(          \
            __VA_ARGS__);                                                                   \
        (s)->launches += 1;                                                                 \
        KR_CUDA(cudaGetLastError());                                                        \
    } while (0)

static KrRed kr_red(const wd_krylov *s, int fin) {
    const int cr = s->method != WD_KRYLOV_CGNR;
    return KrRed{s->partials, s->counter, s->sc, s->sc_host_dev, fin, cr};
}

// the host's copy of the scalars, after the last sum marked by kr_mark
static int kr_mark(wd_krylov *s) {
    KR_CUDA(cudaEventRecord(s->ev, kr_stream(s)));
    return WD_OK;
}
static int kr_read(wd_krylov *s, KrScalars &sc) {
    KR_CUDA(cudaEventSynchronize(s->ev));
    sc = *s->sc_host;
    return WD_OK;
}

// |v|^2 of a canonical full-lattice field, read by the host
static int kr_norm2(wd_krylov *s, const double2 *v, double &out) {
    KrScalars sc;
    KR_LAUNCH(s, k_kr_dot2, s->whole, v, v, nullptr, nullptr, kr_red(s, KR_SUM));
    KR_TRY(kr_mark(s));
    KR_TRY(kr_read(s, sc));
    out = sc.rr;
    return WD_OK;
}

static int kr_comb(wd_krylov *s, const KrShape &sh, double2 *out, const double2 *a, double c,
                   const double2 *b, int g5) {
    KR_LAUNCH(s, k_kr_comb, sh, out, a, c, b, g5);
    return WD_OK;
}

// out = Mhat_p in (dagger: Mhat_p^dag in)
static int kr_apply(wd_krylov *s, double2 *out, const double2 *in, int parity, int dagger) {
    s->applies += 1;
    s->launches += 2;   // two hopping terms
    KR_TRY(op_schur(s->op, parity, dagger, out, in));
    return WD_OK;
}

static int kr_copy(wd_krylov *s, double2 *out, const double2 *in) {
    KR_CUDA(cudaMemcpyAsync(out, in, sizeof(double2) * KR_PLANES * s->half.stride,
                            cudaMemcpyDeviceToDevice, kr_stream(s)));
    return WD_OK;
}

// v = A^-1 v on one parity (nothing for mu = 0)
static int kr_twist_inverse(wd_krylov *s, double2 *v) {
    const double t = s->op->twist(0);
    if (t == 0.0) return WD_OK;
    KR_LAUNCH(s, k_kr_twist, s->half, v, -t, 1.0 / (1.0 + t * t));
    return WD_OK;
}

// canonical full-lattice field <-> its two parities
static int kr_split(wd_krylov *s, const double2 *full, double2 *even, double2 *odd) {
    KR_CUDA(launch_pack_full(WD_F64, s->op->g, even, odd, (const double *)full, kr_stream(s)));
    s->launches += 1;
    return WD_OK;
}
static int kr_merge(wd_krylov *s, double2 *full, const double2 *even, const double2 *odd) {
    KR_CUDA(launch_unpack_full(WD_F64, s->op->g, (double *)full, even, odd, kr_stream(s)));
    s->launches += 1;
    return WD_OK;
}

// Fields per method (f[0..3]):
//   CGNR  z = f0, p = f1, Ap = f2
//   CRNE  s = f0, t = f1, q = f2, w = f3
//   MCR   Br = f0, p = f1, Bp = f2
// The scalars rho, rr (and alpha, except for CGNR) once r is known.
static int kr_start(wd_krylov *s, int p, KrScalars &st) {
    double2 **f = s->f, *Bp = nullptr;
    const KrShape sh = s->half;
    switch (s->method) {
    case WD_KRYLOV_CGNR:
        KR_TRY(kr_apply(s, f[0], s->r, p, 1));                        // z = A^dag r
        KR_TRY(kr_copy(s, f[1], f[0]));                               // p = z
        KR_LAUNCH(s, k_kr_dot2, sh, f[0], f[0], s->r, s->r, kr_red(s, KR_START));
        break;
    case WD_KRYLOV_CRNE:
        KR_TRY(kr_apply(s, f[0], s->r, p, 1));                        // s = A^dag r
        KR_TRY(kr_apply(s, f[1], f[0], p, 0));                        // t = A s
        KR_TRY(kr_copy(s, f[2], f[0]));                               // q = s
        KR_TRY(kr_copy(s, f[3], f[1]));                               // w = t
        KR_LAUNCH(s, k_kr_dot2, sh, f[0], f[0], s->r, s->r, kr_red(s, KR_START));
        Bp = f[3];
        break;
    default:                                                          // MCR1, MCR2
        KR_TRY(kr_apply(s, f[0], s->r, p, 0));
        KR_LAUNCH_ON(s, 6, k_kr_g5_dot, sh, f[0], s->r, kr_red(s, KR_START));   // Br = gamma5 A r
        KR_TRY(kr_copy(s, f[1], s->r));                               // p = r
        KR_TRY(kr_copy(s, f[2], f[0]));                               // Bp = Br
        Bp = f[2];
        break;
    }
    KR_TRY(kr_mark(s));
    if (Bp) KR_LAUNCH(s, k_kr_dot2, sh, Bp, Bp, nullptr, nullptr, kr_red(s, KR_ALPHA));
    return kr_read(s, st);
}

// One iteration; WD_ERR_BREAKDOWN, with x and r as they were, on a zero or
// non-finite denominator.
static int kr_iterate(wd_krylov *s, int p, KrScalars &st) {
    double2 **f = s->f;
    const KrShape sh = s->half;
    const KrRed alpha = kr_red(s, KR_ALPHA), beta = kr_red(s, KR_BETA);
    switch (s->method) {
    case WD_KRYLOV_CGNR:
        KR_TRY(kr_apply(s, f[2], f[1], p, 0));                        // Ap = A p
        KR_LAUNCH(s, k_kr_dot2, sh, f[2], f[2], nullptr, nullptr, alpha);
        KR_LAUNCH(s, k_kr_step, sh, s->sc, s->x, f[1], s->r, f[2]);
        KR_TRY(kr_apply(s, f[0], s->r, p, 1));                        // z = A^dag r
        KR_LAUNCH(s, k_kr_dot2, sh, f[0], f[0], s->r, s->r, beta);
        KR_TRY(kr_mark(s));
        KR_LAUNCH(s, k_kr_dir, sh, s->sc, f[1], f[0]);
        break;
    case WD_KRYLOV_CRNE:
        KR_LAUNCH(s, k_kr_step, sh, s->sc, s->x, f[2], s->r, f[3]);
        KR_TRY(kr_apply(s, f[0], s->r, p, 1));                        // s = A^dag r
        KR_TRY(kr_apply(s, f[1], f[0], p, 0));                        // t = A s = B r
        KR_LAUNCH(s, k_kr_dot2, sh, f[0], f[0], s->r, s->r, beta);
        KR_TRY(kr_mark(s));
        KR_LAUNCH(s, k_kr_dir2, sh, f[2], f[0], f[3], f[1], alpha);
        break;
    default:                                                          // MCR1, MCR2
        KR_LAUNCH(s, k_kr_step, sh, s->sc, s->x, f[1], s->r, f[2]);
        KR_TRY(kr_apply(s, f[0], s->r, p, 0));
        KR_LAUNCH_ON(s, 6, k_kr_g5_dot, sh, f[0], s->r, beta);              // Br = gamma5 A r
        KR_TRY(kr_mark(s));
        if (s->method == WD_KRYLOV_MCR2) {                            // Bp = Br + beta Bp
            KR_LAUNCH(s, k_kr_dir2, sh, f[1], s->r, f[2], f[0], alpha);
        } else {                                                      // Bp = gamma5 A p
            KR_LAUNCH(s, k_kr_dir, sh, s->sc, f[1], s->r);
            KR_TRY(kr_apply(s, f[2], f[1], p, 0));
            KR_LAUNCH_ON(s, 6, k_kr_g5_dot, sh, f[2], nullptr, alpha);
        }
        break;
    }
    KR_TRY(kr_read(s, st));
    if (st.bad)
        return kr_fail(WD_ERR_BREAKDOWN, s->method == WD_KRYLOV_CGNR
                                             ? "CGNR: |Ap| = 0"
                                             : "CR: (r|B r) or |B p| is zero");
    return WD_OK;
}

static int kr_solve(wd_krylov *s, double2 *x, const double2 *b, double tol, int maxiter,
                    int parity, wd_solve_info *info);

extern "C" {

const char *wd_krylov_last_error(void) { return g_kr_error.c_str(); }

void wd_krylov_destroy(wd_krylov *s) {
    if (!s) return;
    for (void *p : s->allocs) cudaFree(p);
    if (s->sc_host) cudaFreeHost(s->sc_host);
    if (s->ev) cudaEventDestroy(s->ev);
    delete s;
}

int wd_krylov_create(wd_krylov **out, wd_op *op, int method) {
    g_kr_error.clear();
    if (!out || !op) return kr_fail(WD_ERR_ARG, "null argument to wd_krylov_create");
    *out = nullptr;
    if (method < WD_KRYLOV_CGNR || method > WD_KRYLOV_MCR2)
        return kr_fail(WD_ERR_ARG, "method must be WD_KRYLOV_CGNR, _CRNE, _MCR1 or _MCR2");
    if (op->prec != WD_F64)
        return kr_fail(WD_ERR_ARG, "the Krylov solvers need a WD_F64 operator");
    wd_krylov *s = new wd_krylov();
    s->op = op;
    s->method = method;
    s->half = KrShape{op->g.vh, op->g.stride};
    s->whole = KrShape{2 * op->g.vh, 2 * op->g.vh};
    const size_t bytes = sizeof(double2) * KR_PLANES * op->g.stride;
    int rc = kr_alloc(s, (void **)&s->x, bytes);
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->r, bytes);
    for (int i = 0; i < 4 && rc == WD_OK; ++i) rc = kr_alloc(s, (void **)&s->f[i], bytes);
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->bh, bytes);
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->bq, bytes);
    if (rc == WD_OK)
        rc = kr_alloc(s, (void **)&s->full, sizeof(double2) * KR_PLANES * s->whole.vh);
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->partials, sizeof(double2) * KR_BLOCKS);
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->counter, sizeof(unsigned int));
    if (rc == WD_OK) rc = kr_alloc(s, (void **)&s->sc, sizeof(KrScalars));
    if (rc == WD_OK &&
        (cudaHostAlloc((void **)&s->sc_host, sizeof(KrScalars), cudaHostAllocMapped) !=
             cudaSuccess ||
         cudaHostGetDevicePointer((void **)&s->sc_host_dev, s->sc_host, 0) != cudaSuccess))
        rc = kr_fail(WD_ERR_NOMEM, "pinned host buffer");
    // (the memsets are on the legacy stream, the work is not)
    if (rc == WD_OK && cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess)
        rc = kr_fail(WD_ERR_CUDA, "initialisation of the fields");
    if (rc == WD_OK && cudaEventCreateWithFlags(&s->ev, cudaEventDisableTiming) != cudaSuccess)
        rc = kr_fail(WD_ERR_CUDA, "event");
    if (rc != WD_OK) {
        std::string m = g_kr_error;
        wd_krylov_destroy(s);
        g_kr_error = m;
        return rc;
    }
    *out = s;
    return WD_OK;
}

int wd_krylov_solve(wd_krylov *s, double *x_, const double *b_, double tol, int maxiter,
                    int parity, wd_solve_info *info) {
    g_kr_error.clear();
    if (!s || !x_ || !b_) return kr_fail(WD_ERR_ARG, "null argument to wd_krylov_solve");
    if (!(tol > 0) || maxiter < 0) return kr_fail(WD_ERR_ARG, "tol must be > 0, maxiter >= 0");
    if (parity != 0 && parity != 1) return kr_fail(WD_ERR_ARG, "parity must be 0 or 1");
    if (s->method >= WD_KRYLOV_MCR1 && s->op->mu != 0.0)
        return kr_fail(WD_ERR_ARG, "MCR needs gamma5-hermiticity: twisted mass must be 0");
    if (!s->op->gauge_loaded) return kr_fail(WD_ERR_STATE, "no gauge field loaded");
    if (info) memset(info, 0, sizeof(*info));
    s->launches = 0;
    s->applies = 0;
    KR_TRY(op_fork(s->op));
    const int rc = kr_solve(s, (double2 *)x_, (const double2 *)b_, tol, maxiter, parity, info);
    // (the caller's stream also waits for what a failed call has queued)
    const int rj = op_join(s->op);
    return rc == WD_OK && rj != WD_OK ? kr_fail(rj, wd_last_error()) : rc;
}

}  // extern "C"

static int kr_solve(wd_krylov *s, double2 *x, const double2 *b, double tol, int maxiter,
                    int parity, wd_solve_info *info) {
    auto t0 = std::chrono::steady_clock::now();
    const int p = parity, q = 1 - parity;
    const double kappa = s->op->kappa;
    const KrShape sh = s->half;
    double2 *xp = s->x, *xq = s->f[3], *bp = s->r;
    double d;

    // Alg. "schur": bhat = b_p + kappa H_pq A^-1 b_q; x_p from the caller's x
    KR_TRY(kr_split(s, b, p ? s->bq : bp, p ? bp : s->bq));
    KR_TRY(kr_norm2(s, b, d));
    const double nb = std::sqrt(d);
    const double target = tol * nb;
    KR_TRY(kr_twist_inverse(s, s->bq));
    s->launches += 1;
    KR_TRY(op_hop(s->op, p, 0, s->bh, s->bq));
    KR_TRY(kr_comb(s, sh, s->bh, bp, kappa, s->bh, 0));
    KR_TRY(kr_split(s, x, p ? xq : xp, p ? xp : xq));

    const bool mcr = s->method >= WD_KRYLOV_MCR1;
    int iters = 0, restarts = 0, status = WD_ERR_NOT_CONVERGED;
    double true_rel = 0.0;
    while (true) {
        const int iters_at_start = iters;
        // r = bhat - A x_p (gamma5 of it for MCR), the method's start
        KR_TRY(kr_apply(s, s->r, xp, p, 0));
        KR_TRY(kr_comb(s, sh, s->r, s->bh, -1.0, s->r, mcr));
        KrScalars st;
        KR_TRY(kr_start(s, p, st));
        int rc = WD_OK;
        while (std::sqrt(st.rr) > target && iters < maxiter) {
            rc = kr_iterate(s, p, st);
            if (rc != WD_OK) break;
            ++iters;
        }
        if (rc == WD_ERR_BREAKDOWN) { status = rc; break; }
        KR_TRY(rc);
        // reconstruction x_q = A^-1 (b_q + kappa H_qp x_p) and the true residual
        KR_TRY(kr_split(s, b, p ? s->bq : s->f[0], p ? s->f[0] : s->bq));
        s->launches += 1;
        KR_TRY(op_hop(s->op, q, 0, xq, xp));
        KR_TRY(kr_comb(s, sh, xq, s->bq, kappa, xq, 0));
        KR_TRY(kr_twist_inverse(s, xq));
        KR_TRY(kr_merge(s, x, p ? xq : xp, p ? xp : xq));
        // (wd_apply works on this stream, between two waits on the caller's)
        s->launches += 4;
        KR_TRY(wd_apply(s->op, (double *)s->full, (const double *)x, 0));
        KR_TRY(kr_comb(s, s->whole, s->full, b, -1.0, s->full, 0));
        KR_TRY(kr_norm2(s, s->full, d));
        restarts += 1;
        const double rn = std::sqrt(d);
        true_rel = nb > 0 ? rn / nb : 0.0;
        if (!std::isfinite(rn)) { status = WD_ERR_BREAKDOWN; break; }
        if (rn <= target) { status = WD_OK; break; }
        // a pass that could not iterate (maxiter, or a recomputed residual
        // already under the target while the true one is not) ends the solve
        if (iters >= maxiter || iters == iters_at_start) break;
    }
    KR_CUDA(cudaStreamSynchronize(kr_stream(s)));
    if (info) {
        info->iters = iters;
        info->reliable_updates = restarts;
        info->true_rel_resid = true_rel;
        // two hopping terms per Schur application, one in the preparation,
        // one per reconstruction and two per full-lattice residual
        info->dslash_hi = 2.0 * (double)s->applies + 1.0 + 3.0 * restarts;
        info->launches = (double)s->launches;
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    if (status != WD_OK) kr_fail(status, status == WD_ERR_BREAKDOWN && !g_kr_error.empty()
                                             ? g_kr_error : wd_status_string(status));
    return status;
}

