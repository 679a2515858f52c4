// One layer with 16 input channels (16 or 1 output channels) of the
// parallel-transport network in a single kernel: the transports are
// computed on the CUDA cores straight into the
// tensor cores' shared-memory operand tiles, so the gathered operand (nine
// transports x 16 channels x 4 spins x re/im per (site, colour) row, 2.3 KB
// per row in BF16) never goes to HBM.
//
//   out_c'(x)[a][s'] = sum_{k, c, s} W[c', c, k][s', s] (T_k in_c)(x)[a][s]
//
// Work split.  A persistent CTA takes tiles of 128 consecutive sites.  For
// colour a the rows of the tile are the 128 sites, so one tile is three
// 128 x N FP32 accumulators in tensor memory (N = 128 output columns for 16
// output channels, 16 for one: re/im x channels x spins, padded), one per
// colour, all multiplied by the same weight matrix.  The
// reduction (1152 real columns: re/im x 9 transports x 16 channels x 4
// spins) runs in 18 chunks of 64 columns, chunk (k, g) = transport k,
// channels 8 g .. 8 g + 7, the 32 real-part and the 32 imaginary-part
// columns.  Per chunk
//   * 16 warps compute (T_k in_c)(x) for 128 sites x 8 channels in FP32
//     (one (site, channel) item: the neighbour's 3 x 4 spinor entries and
//     one link, 36 complex multiply-adds), round to BF16 and store the
//     values in the K-major core-matrix layout of three 128 x 64 tiles;
//   * the N x 64 slice of the real block weight matrix, kept in global
//     memory as the core-matrix image, arrives by one bulk copy (295 KB in
//     all for 16 output channels: it stays in L2);
//   * one lane of another warp issues 3 x 4 tcgen05.mma (M = 128, N,
//     K = 16) into the three accumulators and commits them to the stage's
//     mbarrier.
// Chunks cycle through three 64 KB shared-memory stages; a stage is refilled
// once the commit of the chunk that last used it has arrived, so the
// transports of the next chunks overlap the MMAs of the current one.  After
// the last chunk of a tile the accumulators go through tcgen05.ld to the FP32
// output rows (x, a), which are the next layer's input rows.
//
// Measured at 16^3 x 32 (1024 tiles): 397 us for 16 -> 16 channels, 329 us for
// 16 -> 1 (484 and 372 us with 8-way bank conflicts in the weight copies and 4-way
// ones in the operand stores, a link load per item and per-lane output lines).
// What bounds it: the producers' issue slots (46 % active; the transports'
// 144 multiply-adds per item are 43 % of the instructions), then the latency of
// the neighbours' rows, which 16 warps of 112 registers hide only in part;
// tensor pipe 13 %, L1 data stage 53 %.
//
// Bounded waits as in tc_gemm.cuh: every mbarrier wait polls at most
// spin_limit times; a wait that gives up sets err = 1, no further MMA is
// issued, a final commit drains the MMAs already issued (err = 2 if even
// that wait gives up) and only then is tensor memory freed.  `withhold`
// (tests only) makes the CTA issue no MMA, so that its first stage wait
// runs out with nothing in flight.
#pragma once

#include <type_traits>

#include "tc_gemm.cuh"

namespace wd {

constexpr int PF_SITES = 128;                  // sites per tile = MMA rows
constexpr int PF_THREADS = 512;
constexpr int PF_CIN = 16;
constexpr int PF_LDF = 8 * PF_CIN;             // row stride of 16-channel activations
constexpr int PF_KHALF = PF_CIN * 36;          // 576 columns per re/im part
constexpr int PF_NCHUNK = 18;                  // 9 transports x 2 channel groups
constexpr int PF_STAGES = 3;
constexpr int PF_TILE = PF_SITES * 64 * 2;     // 16 KB: one 128 x 64 BF16 operand tile
static_assert(PF_SITES * 4 == PF_THREADS, "a thread per two sites and a channel");

// output columns of a layer with COUT output channels: re/im x COUT x 4 spins,
// at least 16 (the smallest N of an M = 128 MMA)
template <int COUT> constexpr int pf_n() { return 8 * COUT < 16 ? 16 : 8 * COUT; }
template <int COUT> constexpr int pf_stage_bytes() { return 3 * PF_TILE + pf_n<COUT>() * 64 * 2; }
template <int COUT> constexpr int pf_smem_bytes() { return PF_STAGES * pf_stage_bytes<COUT>(); }
template <int COUT> constexpr uint32_t pf_tmem_cols() {
    return 3 * pf_n<COUT>() <= 32 ? 32 : 3 * pf_n<COUT>() <= 64 ? 64 : 3 * pf_n<COUT>() <= 128 ? 128
         : 3 * pf_n<COUT>() <= 256 ? 256 : 512;
}

struct PfArgs {
    PtcGeom g;
    const float *F;            // input rows (x, a): [Re (c, s)][Im (c, s)], 16 channels,
                               // PF_LDF floats apart
    unsigned phase_on;         // bit mu set: the boundary phase of direction mu is not 1
    const float2 *U;           // links [V][4][3][3], complex64
    const __nv_bfloat16 *B;    // real block weights as the shared-memory images of the 18
                               // chunks (k_ptc_weights_fused), N x 64 each
    float *out;                // output rows (x, a), row stride ldo (>= N)
    int ldo;
    long ntiles;
    int *err;
    unsigned spin_limit;
    int withhold;              // tests: issue no MMA, so the first stage wait runs out
};

// read-only loads that stay where they are written: left to the compiler, a
// chunk's loads were spread over its arithmetic to save registers, and a warp
// made about six round trips to L2 per chunk
// (OFF: byte offset, part of the instruction)
template <int OFF>
__device__ __forceinline__ float4 pf_load4(const void *p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4 + %5];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float2 pf_load2(const void *p) {
    float2 v;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2 + %3];"
                 : "=f"(v.x), "=f"(v.y) : "l"(p), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared.v2.b32 [%0 + %3], {%1, %2};" :: "r"(addr), "r"(a), "r"(b), "n"(OFF));
}
// a site's operands of one channel group: three colours, real and imaginary
// parts of four spins
__device__ __forceinline__ void pf_load_row(const float *row, float4 re[3], float4 im[3]) {
    constexpr int C = 4 * 128, I = 4 * 64;   // bytes between colours, and to the imaginary part
    re[0] = pf_load4<0>(row);     im[0] = pf_load4<I>(row);
    re[1] = pf_load4<C>(row);     im[1] = pf_load4<C + I>(row);
    re[2] = pf_load4<2 * C>(row); im[2] = pf_load4<2 * C + I>(row);
}
// a link's elements, transposed if T
template <bool T> __device__ __forceinline__ void pf_load_link(const float2 *U, float2 u[9]) {
    u[0] = pf_load2<0>(U);           u[1] = pf_load2<T ? 24 : 8>(U);  u[2] = pf_load2<T ? 48 : 16>(U);
    u[3] = pf_load2<T ? 8 : 24>(U);  u[4] = pf_load2<32>(U);          u[5] = pf_load2<T ? 56 : 40>(U);
    u[6] = pf_load2<T ? 16 : 48>(U); u[7] = pf_load2<T ? 40 : 56>(U); u[8] = pf_load2<64>(U);
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// Warp roles: sixteen warps produce the operand tiles and run the epilogue;
// one lane of warp 16 issues the MMAs (done by a producer warp instead, the
// 850 cycles of issuing a chunk's MMAs come on top of that warp's own part, and
// every warp then waits for it: 544 against 454 us in an earlier form).  Warps 16 .. 19 form a
// register warpgroup of their own: they give registers up (setmaxnreg) and the
// producers take them, so that a producer keeps two sites' operands and links
// without spilling.  Hand-offs go through mbarriers, never a CTA-wide barrier, so
// producer warps run up to PF_STAGES chunks ahead of the tensor cores and hide
// each other's memory latency:
//   full[s]   producers -> MMA: stage s holds a chunk's operands (16 arrivals)
//   bfull[s]  bulk copy -> MMA: stage s holds the chunk's weights
//   empty[s]  MMA -> producers: the chunk's MMAs have read stage s (commit)
//   accf      MMA -> producers: the tile's accumulators are complete (commit)
//   acce      producers -> MMA: the epilogue has read the accumulators
// A wait that runs out sets `abort` in shared memory; every role checks it
// and leaves its loop, and the MMAs already issued are drained before the
// tensor memory is freed.
constexpr int PF_WARPS = PF_THREADS / 32;
constexpr int PF_ALL_THREADS = PF_THREADS + 128;
// registers per thread after the hand-over: the launch must bring their sum
constexpr int PF_REGS_PRODUCER = 112, PF_REGS_MMA = 24;
constexpr int PF_REGS_TOTAL = PF_THREADS * PF_REGS_PRODUCER + 128 * PF_REGS_MMA;

template <int COUT>
__global__ void __launch_bounds__(PF_ALL_THREADS, 1) k_ptc_layer_fused(const __grid_constant__ PfArgs p) {
    constexpr int N = pf_n<COUT>();
    constexpr int STAGE = pf_stage_bytes<COUT>();
    constexpr uint32_t TMEM_COLS = pf_tmem_cols<COUT>();
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[PF_STAGES], empty[PF_STAGES], bfull[PF_STAGES];
    __shared__ __align__(8) uint64_t accf, acce, drain;
    __shared__ __align__(16) uint4 turn[PF_WARPS][128];   // the epilogue's turning buffers
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool mma_warp = warp == PF_WARPS;

    if (mma_warp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < PF_STAGES; ++b) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&full[b])), "r"(PF_WARPS) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&empty[b])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&bfull[b])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&accf)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&acce)), "r"(PF_WARPS) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&drain)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t smem0 = smem_u32(smem);
    // a bounded wait that, when it runs out, tells every role to stop
    auto wait = [&](uint64_t *bar, uint32_t parity) {
        if (abort_flag) return false;
        if (tc_wait(smem_u32(bar), parity, p.spin_limit)) return true;
        abort_flag = 1;
        return false;
    };

    if (warp >= PF_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(PF_REGS_MMA));
        // ---- MMA issue (one lane)
        if (mma_warp && lane == 0) {
            long chunk = 0, it = 0;
            for (long tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++it) {
                if (it > 0 && !wait(&acce, (uint32_t)((it - 1) & 1))) break;
                bool ok = true;
                for (int q = 0; q < PF_NCHUNK; ++q, ++chunk) {
                    const int st = (int)(chunk % PF_STAGES);
                    const uint32_t par = (uint32_t)((chunk / PF_STAGES) & 1);
                    if (!wait(&full[st], par) || !wait(&bfull[st], par)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (!p.withhold) {
                        const uint32_t sbase = smem0 + st * STAGE, sB = sbase + 3 * PF_TILE;
#pragma unroll
                        for (int a = 0; a < 3; ++a)
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                const uint64_t ad = tc_smem_desc(sbase + a * PF_TILE + kk * 256, 128, 1024);
                                const uint64_t bd = tc_smem_desc(sB + kk * 256, 128, 1024);
                                const uint32_t acc = (q > 0 || kk > 0) ? 1u : 0u;
                                asm volatile(
                                    "{\n\t.reg .pred p;\n\t"
                                    "setp.ne.b32 p, %4, 0;\n\t"
                                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
                                    :: "r"(tmem + (uint32_t)(a * N)), "l"(ad), "l"(bd),
                                       "r"(tc_idesc_bf16<N, TC_NT>()), "r"(acc)
                                    : "memory");
                            }
                        tc_commit(&empty[st]);
                    }
                }
                if (!ok) break;
                if (!p.withhold) tc_commit(&accf);
            }
        }
        __syncwarp();
    } else {
        // ---- producers: operand tiles, then the epilogue of each tile
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(PF_REGS_PRODUCER));
        long chunk = 0, it = 0;
        // thread (two sites four apart, one channel): the eight lanes of a
        // quarter warp read one 128-byte line of a site's row.  The 8-byte
        // operand stores of a half warp would then be two sites x four channel
        // pairs, and the pairs of a site share their banks; lanes of odd
        // channel pairs store their second site first, which halves that.
        const int cl = lane & 7, odd = (cl >> 1) & 1;
        const int s0 = 8 * warp + (lane >> 3);          // sites s0 and s0 + 4
        const long sty = p.g.L[0], stz = sty * p.g.L[1], stt = stz * p.g.L[2];
        for (long tile = blockIdx.x; tile < p.ntiles; tile += gridDim.x, ++it) {
            const long x0 = tile * PF_SITES;
            const bool whole = x0 + PF_SITES <= p.g.V;
            long x[2];
            int co[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                x[j] = x0 + s0 + 4 * j < p.g.V ? x0 + s0 + 4 * j : 0;
                lex_coords(p.g, x[j], co[j]);
            }
            // operands of both sites, [site][colour] of four spins; links in the
            // order of the product (U forward, its adjoint backward); the row of
            // the neighbour and whether its hop needs the boundary phase
            float4 pre[2][3], pim[2][3];
            float2 u[2][9];
            const float *rows[2];
            bool wrap[2];
            // start the loads of site j for chunk q: the link and the neighbour
            // when a transport begins, the operands of its channel group
            auto load = [&](int j, int q) {
                const int k = q >> 1, grp = q & 1;
                if (grp == 0) {
                    long xn = x[j];
                    wrap[j] = false;
                    if (k > 0) {
                        const int mu = (k - 1) & 3;
                        const bool fwd = k <= 4;
                        const int cm = mu == 0 ? co[j][0] : mu == 1 ? co[j][1]
                                       : mu == 2 ? co[j][2] : co[j][3];
                        const long s = mu == 0 ? 1 : mu == 1 ? sty : mu == 2 ? stz : stt;
                        const int last = p.g.L[mu] - 1;
                        const bool w = cm == (fwd ? last : 0);
                        xn = fwd ? (w ? xn - last * s : xn + s) : (w ? xn + last * s : xn - s);
                        wrap[j] = w && (p.phase_on >> mu & 1u);
                        const float2 *Ul = p.U + ((fwd ? x[j] : xn) * 4 + mu) * 9;
                        if (fwd) {
                            pf_load_link<false>(Ul, u[j]);
                        } else {
                            pf_load_link<true>(Ul, u[j]);
#pragma unroll
                            for (int e = 0; e < 9; ++e) u[j][e].y = -u[j][e].y;
                        }
                    }
                    rows[j] = p.F + xn * 3 * PF_LDF + cl * 4;
                }
                pf_load_row(rows[j] + grp * 32, pre[j], pim[j]);
            };
            // colour a of site j's operand: BF16 pairs, re spins 01, 23, im 01, 23.
            // (Rows past the lattice hold site 0's values: rows do not mix, and
            // theirs are not stored.)
            auto transport = [&](int j, int a, int mu, bool fwd, bool phase, uint32_t (&o)[4]) {
                float vr[4], vi[4];
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const float wx = u[j][3 * a + b].x, wy = u[j][3 * a + b].y;
                    const float r[4] = {pre[j][b].x, pre[j][b].y, pre[j][b].z, pre[j][b].w};
                    const float m[4] = {pim[j][b].x, pim[j][b].y, pim[j][b].z, pim[j][b].w};
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        // one rounding per product, in the order of the gathered form
                        vr[s] = fmaf(-wy, m[s], b == 0 ? wx * r[s] : fmaf(wx, r[s], vr[s]));
                        vi[s] = fmaf(wy, r[s], b == 0 ? wx * m[s] : fmaf(wx, m[s], vi[s]));
                    }
                }
                if (phase) {
                    if (wrap[j]) {
                        const float pr = p.g.ph[2 * mu];
                        const float pi = fwd ? p.g.ph[2 * mu + 1] : -p.g.ph[2 * mu + 1];
#pragma unroll
                        for (int s = 0; s < 4; ++s) {
                            const float t = vr[s] * pr - vi[s] * pi;
                            vi[s] = vr[s] * pi + vi[s] * pr;
                            vr[s] = t;
                        }
                    }
                }
                o[0] = pack_bf16x2(vr[0], vr[1]);
                o[1] = pack_bf16x2(vr[2], vr[3]);
                o[2] = pack_bf16x2(vi[0], vi[1]);
                o[3] = pack_bf16x2(vi[2], vi[3]);
            };
            // K-major core-matrix layout: row = site, K column = channel * 4 + s
            // (re) or 32 + the same (im), four BF16 per store
            const uint32_t soff = (cl >> 1) * 128 + (cl & 1) * 8 + (s0 >> 3) * 1024 + (s0 & 7) * 16;
            bool ok = true;
#pragma unroll 1
            for (int q = 0; q < PF_NCHUNK; ++q, ++chunk) {
                const int st = (int)(chunk % PF_STAGES);
                const uint32_t sbase = smem0 + st * STAGE;
                load(0, q);
                load(1, q);
                const bool free_stage =
                    chunk < PF_STAGES ||
                    wait(&empty[st], (uint32_t)(((chunk - PF_STAGES) / PF_STAGES) & 1));
                if (!__all_sync(0xffffffffu, free_stage)) {   // (the warp leaves together)
                    ok = false;
                    break;
                }
                if (tid == 0) {   // the chunk's weights
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                                 :: "r"(smem_u32(&bfull[st])), "r"((uint32_t)(N * 128)) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
                                 "[%0], [%1], %2, [%3];"
                                 :: "r"(sbase + 3 * PF_TILE),
                                    "l"(p.B + (long)q * N * 64), "r"((uint32_t)(N * 128)),
                                    "r"(smem_u32(&bfull[st])) : "memory");
                }
                const uint32_t first = sbase + soff + (odd ? 64 : 0), second = sbase + soff + (odd ? 0 : 64);
                const int k = q >> 1, mu = (k - 1) & 3;
                const bool fwd = k <= 4;
                const bool phase = __any_sync(0xffffffffu, wrap[0] || wrap[1]);
                auto colour = [&](auto A) {
                    constexpr int a = decltype(A)::value, O = a * PF_TILE;
                    uint32_t o[2][4];
                    if (k == 0) {   // T_0 = 1
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            o[j][0] = pack_bf16x2(pre[j][a].x, pre[j][a].y);
                            o[j][1] = pack_bf16x2(pre[j][a].z, pre[j][a].w);
                            o[j][2] = pack_bf16x2(pim[j][a].x, pim[j][a].y);
                            o[j][3] = pack_bf16x2(pim[j][a].z, pim[j][a].w);
                        }
                    } else {
                        transport(0, a, mu, fwd, phase, o[0]);
                        transport(1, a, mu, fwd, phase, o[1]);
                    }
                    sts64<O>(first, odd ? o[1][0] : o[0][0], odd ? o[1][1] : o[0][1]);
                    sts64<O>(second, odd ? o[0][0] : o[1][0], odd ? o[0][1] : o[1][1]);
                    sts64<O + 512>(first, odd ? o[1][2] : o[0][2], odd ? o[1][3] : o[0][3]);
                    sts64<O + 512>(second, odd ? o[0][2] : o[1][2], odd ? o[0][3] : o[1][3]);
                };
                colour(std::integral_constant<int, 0>());
                colour(std::integral_constant<int, 1>());
                colour(std::integral_constant<int, 2>());
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&full[st])) : "memory");
            }
            if (!ok) break;
            // epilogue: wait for the tile's accumulators, read them, hand TMEM back
            if (!__all_sync(0xffffffffu, wait(&accf, (uint32_t)(it & 1)))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            {
                // warp w reads TMEM lanes 32 (w % 4) .. +31 (sites); column blocks
                // of 16 are dealt round-robin over the warps sharing a lane quarter.
                // A lane holds one site's 64 bytes; they pass through 2 KB of
                // shared memory per warp (16-byte slots swizzled by the row, no
                // bank conflicts), so that four lanes store a site's 64 bytes
                // together instead of every lane a line of its own (11 us of a
                // tile's 65).
                constexpr int NGROUPS = PF_WARPS / 4;
                const int quarter = warp & 3, group = warp >> 2;
                const uint32_t lane_base = (uint32_t)(32 * quarter) << 16;
                const uint32_t buf = smem_u32(turn[warp]);
                const uint32_t wr = buf + lane * 64, wsw = (lane >> 1) & 3;
#pragma unroll 1
                for (int c0 = 16 * group; c0 < 3 * N; c0 += 16 * NGROUPS) {
                    uint32_t r[16];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                          "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                          "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                        : "r"(tmem + lane_base + (uint32_t)c0));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    __syncwarp();   // the previous block's reads are done
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                                     :: "r"(wr + ((j ^ wsw) << 4)), "r"(r[4 * j]), "r"(r[4 * j + 1]),
                                        "r"(r[4 * j + 2]), "r"(r[4 * j + 3]) : "memory");
                    __syncwarp();
                    const int a = c0 / N, n0 = c0 - a * N;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int row = 8 * i + (lane >> 2), part = lane & 3;
                        uint4 v;
                        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                                     : "r"(buf + row * 64 + ((part ^ ((row >> 1) & 3)) << 4))
                                     : "memory");
                        const long xr = x0 + 32 * quarter + row;
                        if (whole || xr < p.g.V)
                            *reinterpret_cast<uint4 *>(p.out + (xr * 3 + a) * (long)p.ldo + n0 +
                                                       4 * part) = v;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&acce)) : "memory");
        }
        // a role that gave up: the weight copies still in flight land before the
        // CTA's shared memory is given back
        if (abort_flag && tid == 0)
            for (long c = chunk > PF_STAGES ? chunk - PF_STAGES : 0; c < chunk; ++c)
                tc_wait(smem_u32(&bfull[c % PF_STAGES]), (uint32_t)((c / PF_STAGES) & 1),
                        64ull * p.spin_limit);
    }
    // every role has left its loop; drain the MMAs issued if a wait ran out
    __syncthreads();
    if (abort_flag) {
        if (mma_warp && lane == 0) {
            atomicExch(p.err, 1);
            tc_commit(&drain);
            if (!tc_wait(smem_u32(&drain), 0u, 64ull * p.spin_limit)) atomicExch(p.err, 2);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (mma_warp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
}

}  // namespace wd
