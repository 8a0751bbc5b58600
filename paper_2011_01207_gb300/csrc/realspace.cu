// a2 / a5 - Real-space pair kernels over blocks of 32 atoms (paper Sec. 2.3: groups of B_size
// atoms with the paper's group-to-atom list filtering). One CTA per block walks the lists of
// its target pairs (pair_walk.cuh); pair arithmetic and a thread's sums in T (FP32 in the mixed and fixed
// modes), the sum over a target's threads compensated in FP32, stored once as FP64 (or fixed point).
//
// Bound by instruction issue and latency at the occupancy that registers and shared memory allow (63 % of the
// slots busy in the matvec at 96,000 atoms, FMA pipe 36 %, shared memory 35 %; 53, 29 and 25 % with cold caches).
// Measured on GB300, ncu, warm caches, against the kernels on 32 x 32 pair
// masks that this replaced (one side per lane, items staged and flushed with atomics):
//   matvec           96,000 atoms  61 -> 40.0 us (49.7 M -> 26.6 M warp instructions)
//   permanent field  96,000 atoms  85 -> 58.1 us
//   matvec at 6,000 atoms (quarter blocks)  16.1 -> 8.6 us
#include "common.cuh"
#include "pair_math.cuh"
#include "pair_walk.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace {

constexpr int PT = 128;   // threads of a CTA
constexpr int MV_MINB = 6, PF_MINB = 4;   // CTAs per SM asked for: the shared memory's limit

// ---------------------------------------------------------------------------------------
// a2: permanent multipole field, E_i += E(R; q_j, d_j, Q_j), with R = x_i - x_j and sigma = 0 in
// R_n for excluded pairs. The radial functions come negated, so the terms in R are collected apart
// from the others (g, f) and E = f - g.
template <class T, class Vt>
__device__ __forceinline__ void pf_contract(const Vt *R, const Vt *Mn, const typename V4<T>::type &d,
                                            const typename V4<T>::type &qa, const typename V4<T>::type &qb, Vt *f, Vt *g) {
    const Vt dx = splat2(d.x), dy = splat2(d.y), dz = splat2(d.z), qyz = splat2(qb.x);
    const Vt dR = fma2(dx, R[0], fma2(dy, R[1], mul2(dz, R[2])));
    const Vt Qx = fma2(splat2(qa.x), R[0], fma2(splat2(qa.y), R[1], mul2(splat2(qa.z), R[2])));
    const Vt Qy = fma2(splat2(qa.y), R[0], fma2(splat2(qa.w), R[1], mul2(qyz, R[2])));
    const Vt Qz = fma2(splat2(qa.z), R[0], fma2(qyz, R[1], mul2(splat2(qb.y), R[2])));
    const Vt RQR = fma2(Qx, R[0], fma2(Qy, R[1], mul2(Qz, R[2])));
    const Vt fac = fma2(splat2(qb.w), Mn[0], fma2(dR, Mn[1], mul2(mul2(RQR, splat2(T(1.0 / 3.0))), Mn[2])));
    const Vt m2 = mul2(Mn[1], splat2(T(2.0 / 3.0)));
    f[0] = fma2(Mn[0], dx, fma2(m2, Qx, f[0]));
    f[1] = fma2(Mn[0], dy, fma2(m2, Qy, f[1]));
    f[2] = fma2(Mn[0], dz, fma2(m2, Qz, f[2]));
    g[0] = fma2(fac, R[0], g[0]);
    g[1] = fma2(fac, R[1], g[1]);
    g[2] = fma2(fac, R[2], g[2]);
}

template <class T, int PARTS>
__global__ void __launch_bounds__(PT, PF_MINB) k_perm_field(ListArgs la, const typename V4<T>::type *__restrict__ posw,
                                                   const typename V4<T>::type *__restrict__ dipd,
                                                   const typename V4<T>::type *__restrict__ quad0,
                                                   const typename V4<T>::type *__restrict__ quad1,
                                                   double *__restrict__ acc, int n_pad, PairConsts<T> pc, int fixed) {
    typedef typename V4<T>::type T4;
    typedef typename Vec<T>::type Vt;
    extern __shared__ __align__(16) unsigned char raw[];
    constexpr int ROW = (AP_CHUNK + 1) * (int)sizeof(T4);
    const Layout<T, PARTS> ly;
    const RadialConsts<T> rk(pc);
    Targets<T> tg;
    tg.load(posw, ly.slot(), ly.h, pc.n, pc.rc2, rk.ta);
    Vt f[3], g[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = g[k] = splat2(T(0));
    const T4 *const src[3] = {dipd, quad0, quad1};
    for_chunks<T, PARTS>(raw, la, ly, src, [&](const unsigned *list, int words, int flagged, int) {
        auto side = [&](unsigned e, auto ex) {
            constexpr bool EX = decltype(ex)::value;
            const unsigned char *at = raw + (e & 0xfff0u) * (unsigned)(sizeof(T4) / 16);
            const T4 o = *reinterpret_cast<const T4 *>(at), d = *reinterpret_cast<const T4 *>(at + ROW);
            const T4 qa = *reinterpret_cast<const T4 *>(at + 2 * ROW), qb = *reinterpret_cast<const T4 *>(at + 3 * ROW);
            Vt R[3], Mu[3], Md[3], pen;
            bool exa, exb;
            const Vt r2 = tg.template vector<EX>(o, e, R, pen, exa, exb);
            radial<3, EX>(rk, r2, mul1(tg.w, o.w), pen, exa, exb, Mu, Md);
            pf_contract<T>(R, EX ? Md : Mu, d, qa, qb, f, g);
        };
        walk(list, words, flagged, ly.first, ly.STRIDE, [&](unsigned e) { side(e, std::true_type()); },
             [&](unsigned e) { side(e, std::false_type()); });
    });
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = sub2(f[k], g[k]);
    ly.store3(acc, n_pad, f, fixed);
}

// ---------------------------------------------------------------------------------------
// a5: dipole-field matrix-vector product, E_i += -R1 p_j + R2 (p_j.R) R, for one dipole vector
// or (NS = 2, AMOEBA's d and p dipoles) two at once: the pair tensor is evaluated once for both.
// SHORT: only the pairs closer than AP_SHORT_RANGE (the learned guess's feature), which come
// first in every list.
template <class T, int PARTS, int NS, bool SHORT>
__global__ void __launch_bounds__(PT, MV_MINB) k_matvec(ListArgs la, const typename V4<T>::type *__restrict__ posw,
                                               const typename V4<T>::type *__restrict__ pv0,
                                               const typename V4<T>::type *__restrict__ pv1, double *__restrict__ acc0,
                                               double *__restrict__ acc1, int n_pad, PairConsts<T> pc, int fixed) {
    typedef typename V4<T>::type T4;
    typedef typename Vec<T>::type Vt;
    extern __shared__ __align__(16) unsigned char raw[];
    constexpr int ROW = (AP_CHUNK + 1) * (int)sizeof(T4);
    const Layout<T, PARTS> ly;
    const RadialConsts<T> rk(pc);
    Targets<T> tg;
    tg.load(posw, ly.slot(), ly.h, pc.n, SHORT ? T(AP_SHORT_RANGE * AP_SHORT_RANGE) : pc.rc2, rk.ta);
    Vt f[3 * NS], g[3 * NS];   // E = f - g, as in the permanent field
#pragma unroll
    for (int k = 0; k < 3 * NS; ++k) f[k] = g[k] = splat2(T(0));
    const T4 *src[NS];
    src[0] = pv0;
    if constexpr (NS == 2) src[1] = pv1;
    for_chunks<T, PARTS>(raw, la, ly, src, [&](const unsigned *list, int words, int flagged, int shorts) {
        auto side = [&](unsigned e, auto ex) {
            constexpr bool EX = decltype(ex)::value;
            const unsigned char *at = raw + (e & 0xfff0u) * (unsigned)(sizeof(T4) / 16);
            const T4 o = *reinterpret_cast<const T4 *>(at);
            Vt R[3], Mn[2], pen;
            bool exa, exb;   // sigma = 1 for every pair
            const Vt r2 = tg.template vector<EX>(o, e, R, pen, exa, exb);
            radial<2, false>(rk, r2, mul1(tg.w, o.w), pen, false, false, Mn, Mn);
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                const T4 v = *reinterpret_cast<const T4 *>(at + (1 + q) * ROW);
                const Vt vx = splat2(v.x), vy = splat2(v.y), vz = splat2(v.z);
                const Vt u = mul2(fma2(vx, R[0], fma2(vy, R[1], mul2(vz, R[2]))), Mn[1]);
                f[3 * q] = fma2(Mn[0], vx, f[3 * q]);
                f[3 * q + 1] = fma2(Mn[0], vy, f[3 * q + 1]);
                f[3 * q + 2] = fma2(Mn[0], vz, f[3 * q + 2]);
                g[3 * q] = fma2(u, R[0], g[3 * q]);
                g[3 * q + 1] = fma2(u, R[1], g[3 * q + 1]);
                g[3 * q + 2] = fma2(u, R[2], g[3 * q + 2]);
            }
        };
        walk(list, SHORT ? shorts : words, flagged, ly.first, ly.STRIDE, [&](unsigned e) { side(e, std::true_type()); },
             [&](unsigned e) { side(e, std::false_type()); });
    });
#pragma unroll
    for (int k = 0; k < 3 * NS; ++k) f[k] = sub2(f[k], g[k]);
    ly.store3(acc0, n_pad, f, fixed);
    if (NS == 2) ly.store3(acc1, n_pad, f + 3 * (NS - 1), fixed);
}

template <class T>
size_t rows_bytes(int rows) { return (size_t)rows * (AP_CHUNK + 1) * sizeof(typename V4<T>::type); }

template <class T, int PARTS>
int perm_field_t(ap_ctx *ctx, cudaStream_t s) {
    typedef typename V4<T>::type T4;
    auto kern = k_perm_field<T, PARTS>;
    const size_t bytes = rows_bytes<T>(4);
    kern<<<ctx->n_blocks * PARTS, PT, bytes, s>>>(list_args(ctx), (const T4 *)ctx->posw, (const T4 *)ctx->dipd,
                                                  (const T4 *)ctx->quad0, (const T4 *)ctx->quad1, ctx->acc, ctx->n_pad,
                                                  make_consts<T>(ctx), ctx->fixed);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

// shared memory of the matvec's CTA; the autotuner's limit of `per_sm` CTAs on an SM (0: none) is
// kept by asking for more than the kernel uses
constexpr size_t SM_SMEM = 227 * 1024, CTA_RESERVE = 1024;
size_t matvec_bytes(size_t need, int per_sm) {
    if (per_sm <= 0) return need;
    return std::max(need, SM_SMEM / per_sm - CTA_RESERVE);
}

template <class T, int PARTS, int NS, bool SHORT>
int matvec_p(ap_ctx *ctx, const void *p0, const void *p1, double *acc0, double *acc1, cudaStream_t s) {
    typedef typename V4<T>::type T4;
    auto kern = k_matvec<T, PARTS, NS, SHORT>;
    const size_t bytes = matvec_bytes(rows_bytes<T>(1 + NS), NS == 1 && !SHORT ? ctx->tune_mv_per_sm : 0);
    kern<<<ctx->n_blocks * PARTS, PT, bytes, s>>>(list_args(ctx), (const T4 *)ctx->posw, (const T4 *)p0, (const T4 *)p1, acc0,
                                                  acc1, ctx->n_pad, make_consts<T>(ctx), ctx->fixed);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}
template <class T, int NS, bool SHORT>
int matvec_t(ap_ctx *ctx, const void *p0, const void *p1, double *acc0, double *acc1, cudaStream_t s) {
    return quarter_blocks(ctx) ? matvec_p<T, 4, NS, SHORT>(ctx, p0, p1, acc0, acc1, s)
                               : matvec_p<T, 1, NS, SHORT>(ctx, p0, p1, acc0, acc1, s);
}

template <class T>
int resident_t() {
    int per_sm = 0;
    const size_t bytes = rows_bytes<T>(2);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_matvec<T, 1, 1, false>, PT, bytes);
    return std::max(1, per_sm);
}

template <class T, int PARTS>
int init_p(ap_ctx *ctx) {
    AP_CUDA(allow_smem(k_perm_field<T, PARTS>, rows_bytes<T>(4)));
    AP_CUDA(allow_smem(k_matvec<T, PARTS, 1, false>, SM_SMEM));   // whatever the autotuner chooses
    AP_CUDA(allow_smem(k_matvec<T, PARTS, 1, true>, rows_bytes<T>(2)));
    AP_CUDA(allow_smem(k_matvec<T, PARTS, 2, false>, rows_bytes<T>(3)));
    return AP_OK;
}
template <class T>
int init_t(ap_ctx *ctx) {
    // (the count of resident CTAs is always the whole-block kernel's)
    AP_CUDA(allow_smem(k_matvec<T, 1, 1, false>, SM_SMEM));
    return quarter_blocks(ctx) ? init_p<T, 4>(ctx) : init_p<T, 1>(ctx);
}

template <class T>
int field_t(ap_ctx *ctx, cudaStream_t s) {
    return quarter_blocks(ctx) ? perm_field_t<T, 4>(ctx, s) : perm_field_t<T, 1>(ctx, s);
}

}  // namespace

int real_init(ap_ctx *ctx) { return ctx->prec == AP_FP64 ? init_t<double>(ctx) : init_t<float>(ctx); }

int short_matvec_launch(ap_ctx *ctx, const void *p, double *out, cudaStream_t s) {
    return ctx->prec == AP_FP64 ? matvec_t<double, 1, true>(ctx, p, nullptr, out, nullptr, s)
                                : matvec_t<float, 1, true>(ctx, p, nullptr, out, nullptr, s);
}

int real_field_launch(ap_ctx *ctx, cudaStream_t s) {
    return ctx->prec == AP_FP64 ? field_t<double>(ctx, s) : field_t<float>(ctx, s);
}

// CTAs of the real-space matvec that fit on one SM at once (the autotuner's upper bound)
int real_matvec_resident_per_sm(ap_ctx *ctx) { return ctx->prec == AP_FP64 ? resident_t<double>() : resident_t<float>(); }

int real_matvec_launch(ap_ctx *ctx, const void *p, cudaStream_t s) {
    return ctx->prec == AP_FP64 ? matvec_t<double, 1, false>(ctx, p, nullptr, ctx->acc, nullptr, s)
                                : matvec_t<float, 1, false>(ctx, p, nullptr, ctx->acc, nullptr, s);
}

int real_matvec2_launch(ap_ctx *ctx, const void *p0, const void *p1, double *acc0, double *acc1, cudaStream_t s) {
    return ctx->prec == AP_FP64 ? matvec_t<double, 2, false>(ctx, p0, p1, acc0, acc1, s)
                                : matvec_t<float, 2, false>(ctx, p0, p1, acc0, acc1, s);
}
