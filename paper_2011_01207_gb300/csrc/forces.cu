// a9 - Polarization energy and forces at fixed induced dipoles ("final force evaluation",
// paper Sec. 1.2).
//
// E_pol = -(f/2) sum_i mu_i . E_i. At the solution of A mu = E, dE_pol/dx at fixed mu is the
// gradient of  -f sum_{i<j} mu_i T_ij mu_j - f sum_i mu_i . E_i  (variational property):
//   real space: each unordered pair carries
//       U_ij = -f [mu_i . E(R; M_j) + mu_j . E(-R; M_i) + mu_i . T(R) mu_j],  R = x_i - x_j;
//   reciprocal: f <dQ_mu/dx, phi_M + phi_mu> + f <dQ_M/dx, phi_mu>, from the smooth-PME
//               potentials' derivatives up to third order at the atoms;
//   frames:     global multipoles rotate with their frame atoms: dU/d(global dipole) and
//               dU/d(global quadrupole) are chained through the frame construction.
// Pair arithmetic in T; a thread's sums over its pairs in T; those over a target's threads, and what its own
// multipoles make of them, in FP64 or compensated FP32 pairs.
//
// Virial (on request): V_ab = dE_pol/de_ab under x -> (I + e) x of positions and box, which
// the paper's real-space loop updates with the energy and the forces (Sec. 1.2.1) and sums in
// double precision (Sec. 2.2). At fixed mu it is
//   pairs:      sum over pairs of (dU/dR)_a R_b (R the image vector);
//   frames:     sum over frame vectors v of (dU/dv)_a v_b;
//   reciprocal: -f sum_j [grad phi_{M+mu} mu_j^T + grad phi_mu d_j^T + (2/3) H(phi_mu) Q_j]
//               plus the structure-factor sum of pme.cu (volume and |m| of C(m));
// accumulated per block in FP64 (fixed point in AP_FIXED) into nine device slots.
#include "common.cuh"
#include "pair_math.cuh"
#include "pair_walk.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

void unsort3(ap_ctx *ctx, const double *src, double *out, cudaStream_t s);

namespace {

// FP64 value v added to slot k of an array of FP64 numbers or (fixed) fixed-point integers,
// by the only thread that updates that slot
__device__ __forceinline__ void add_plain(double *arr, size_t k, double v, int fixed) {
    if (fixed)
        reinterpret_cast<long long *>(arr)[k] += ap_to_fx(v);
    else
        arr[k] += v;
}

// adds the nine values v of every thread of a block of NT threads to acc[0..8]: FP64 sums
// and FP64 atomics, or (FX) values already in fixed point, integer sums and integer atomics
// (order-independent, so bitwise reproducible)
template <int NT, class V>
__device__ __forceinline__ void block_add9(V *v, double *acc) {
    __shared__ V sm[NT / 32][9];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        V x = v[k];
        for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        if (l == 0) sm[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        V t = 0;
#pragma unroll
        for (int k = 0; k < NT / 32; ++k) t += sm[k][threadIdx.x];
        if constexpr (std::is_integral<V>::value)
            atomicAdd(reinterpret_cast<unsigned long long *>(acc) + threadIdx.x, (unsigned long long)t);
        else
            atomicAdd(acc + threadIdx.x, t);
    }
}

// ---- real space ----------------------------------------------------------------------------
// One CTA per block of 32 atoms over the pair lists (pair_walk.cuh). What a target's force and
// torque need of its neighbours are derivatives of two fields at the target: E of the induced
// dipoles, up to second order, for the target's charge, dipole and quadrupole, and G, the first
// derivative of the field of permanent multipoles and induced dipoles together, for its induced
// dipole. So the walk accumulates those 30 numbers per target (as the smooth-PME part does) and
// the target's own multipoles enter once at the end, instead of contracting two multipoles per
// pair side: fewer operations, and no target multipoles in the walk's registers.
// With R = x_target - x_source, u = mu.R, D = d + mu:
//   E_a = -R1 mu_a + R2 u R_a
//   E_ab = y_a R_b + y_b R_a + delta_ab sum R2 u,            y = R2 mu - (1/2) R3 u R
//   E_abc = sym(w_a R_b R_c) + (V_a delta_bc + V_b delta_ac + V_c delta_ab),
//           w = (1/3) R4 u R - R3 mu,                        V = R2 mu - R3 u R
//   G_ab = t_a R_b + t_b R_a - (2/3) R2 Q_ab + delta_ab (q R1 + R2 D.R + (1/3) R3 R.Q.R),
//           t = R2 D + (2/3) R3 Q R - (1/2) (q R2 + R3 D.R + (1/3) R4 R.Q.R) R
// and then
//   F_c / f = q E_c + sum_a d_a E_ac + (1/3) sum_ab Q_ab E_abc + sum_a mu_a G_ac
//   dU/dd / (-f) = E,   dU/dQ / (-f/3) = E_ab without its trace part (Q is traceless).
// Measured on GB300 (ncu, warm): 228 -> 132.2 us at 96,000 atoms, 44.2 -> 23.5 us at 6,000, against
// contracting both atoms' multipoles per pair side on 32 x 32 pair masks. 158 registers, so 3 CTAs
// per SM (shared memory would hold 4): what bounds it is issue at that occupancy.
// (Timed with events 135.0 us, 131.7 with the sums of a target's threads and their contraction in plain FP32.)
// Every term is linear in the R_n, which come negated, so the sums are those of -E and -G.
// Excluded pairs (sigma = 0 between permanent and induced, 1 between induced and induced) come
// first in the lists and take two sets of radial functions.
template <class V>
struct FieldSums {
    V E[3], xx, yy, zz, xy, xz, yz, tr;              // the diagonal of E_ab halved
    V S[10], W[3];                                   // xxx yyy zzz (a third) xxy xxz xyy yyz xzz yzz xyz; V
    V gxx, gyy, gzz, gxy, gxz, gyz, gtr;             // G: the diagonal's t_a R_a part halved
    V qxx, qyy, qzz;                                 // and the diagonal of -(2/3) R2 Q
};
constexpr int FS = 33, FO = 29;
// what the force is made of: E, E_ab (the diagonal halved, without its trace part) and that part, S, W, and G whole
template <class Vt>
__device__ __forceinline__ void fold(const FieldSums<Vt> &a, Vt *o) {
    const Vt *v = reinterpret_cast<const Vt *>(&a);
#pragma unroll
    for (int k = 0; k < 23; ++k) o[k] = v[k];
    o[23] = add2(add2(a.gxx, a.gxx), add2(a.gtr, a.qxx));
    o[24] = add2(add2(a.gyy, a.gyy), add2(a.gtr, a.qyy));
    o[25] = add2(add2(a.gzz, a.gzz), add2(a.gtr, a.qzz));
    o[26] = a.gxy;
    o[27] = a.gxz;
    o[28] = a.gyz;
}

template <class T>
__device__ __forceinline__ void zero_sums(FieldSums<typename Vec<T>::type> &a) {
    typename Vec<T>::type *v = reinterpret_cast<typename Vec<T>::type *>(&a);
#pragma unroll
    for (int k = 0; k < FS; ++k) v[k] = splat2(T(0));
}

// the induced dipole mu's share of E, E_ab and E_abc (radial functions Rn[0..3])
template <class T>
__device__ __forceinline__ void add_induced(FieldSums<typename Vec<T>::type> &a, const typename Vec<T>::type *R,
                                            const typename Vec<T>::type *Rn, const typename V4<T>::type &mu) {
    typedef typename Vec<T>::type Vt;
    const Vt mx = splat2(mu.x), my = splat2(mu.y), mz = splat2(mu.z);
    const Vt u = fma2(mx, R[0], fma2(my, R[1], mul2(mz, R[2])));
    const Vt u2 = mul2(Rn[1], u), u3 = mul2(Rn[2], u), n1 = mul2(Rn[0], splat2(T(-1)));
    const Vt h3 = mul2(u3, splat2(T(-0.5))), n3 = mul2(u3, splat2(T(-1))), m3 = mul2(Rn[2], splat2(T(-1)));
    const Vt u4 = mul2(mul2(Rn[3], u), splat2(T(1.0 / 3.0)));
    a.E[0] = fma2(n1, mx, fma2(u2, R[0], a.E[0]));
    a.E[1] = fma2(n1, my, fma2(u2, R[1], a.E[1]));
    a.E[2] = fma2(n1, mz, fma2(u2, R[2], a.E[2]));
    a.tr = add2(a.tr, u2);
    const Vt sx = mul2(Rn[1], mx), sy = mul2(Rn[1], my), sz = mul2(Rn[1], mz);
    const Vt yx = fma2(h3, R[0], sx), yy = fma2(h3, R[1], sy), yz = fma2(h3, R[2], sz);
    a.xx = fma2(yx, R[0], a.xx);
    a.yy = fma2(yy, R[1], a.yy);
    a.zz = fma2(yz, R[2], a.zz);
    a.xy = fma2(yx, R[1], fma2(yy, R[0], a.xy));
    a.xz = fma2(yx, R[2], fma2(yz, R[0], a.xz));
    a.yz = fma2(yy, R[2], fma2(yz, R[1], a.yz));
    a.W[0] = add2(a.W[0], fma2(n3, R[0], sx));
    a.W[1] = add2(a.W[1], fma2(n3, R[1], sy));
    a.W[2] = add2(a.W[2], fma2(n3, R[2], sz));
    const Vt wx = fma2(u4, R[0], mul2(m3, mx)), wy = fma2(u4, R[1], mul2(m3, my)), wz = fma2(u4, R[2], mul2(m3, mz));
    const Vt rxx = mul2(R[0], R[0]), ryy = mul2(R[1], R[1]), rzz = mul2(R[2], R[2]);
    const Vt rxy = mul2(R[0], R[1]), rxz = mul2(R[0], R[2]), ryz = mul2(R[1], R[2]);
    const Vt wx2 = add2(wx, wx), wy2 = add2(wy, wy), wz2 = add2(wz, wz);
    a.S[0] = fma2(wx, rxx, a.S[0]);
    a.S[1] = fma2(wy, ryy, a.S[1]);
    a.S[2] = fma2(wz, rzz, a.S[2]);
    a.S[3] = fma2(wy, rxx, fma2(wx2, rxy, a.S[3]));   // xxy
    a.S[4] = fma2(wz, rxx, fma2(wx2, rxz, a.S[4]));   // xxz
    a.S[5] = fma2(wx, ryy, fma2(wy2, rxy, a.S[5]));   // xyy
    a.S[6] = fma2(wz, ryy, fma2(wy2, ryz, a.S[6]));   // yyz
    a.S[7] = fma2(wx, rzz, fma2(wz2, rxz, a.S[7]));   // xzz
    a.S[8] = fma2(wy, rzz, fma2(wz2, ryz, a.S[8]));   // yzz
    a.S[9] = fma2(wx, ryz, fma2(wy, rxz, fma2(wz, rxy, a.S[9])));   // xyz
}

// the share in G of a multipole (q, D, Q); POLES: with charge and quadrupole
template <class T, bool POLES>
__device__ __forceinline__ void add_gradient(FieldSums<typename Vec<T>::type> &a, const typename Vec<T>::type *R,
                                             const typename Vec<T>::type *Rn, T q, T Dx, T Dy, T Dz,
                                             const typename V4<T>::type &qa, T qyz, T qzz) {
    typedef typename Vec<T>::type Vt;
    const Vt dx = splat2(Dx), dy = splat2(Dy), dz = splat2(Dz);
    const Vt DR = fma2(dx, R[0], fma2(dy, R[1], mul2(dz, R[2])));
    Vt c = mul2(Rn[2], DR), tr = mul2(Rn[1], DR);
    Vt tx = mul2(Rn[1], dx), ty = mul2(Rn[1], dy), tz = mul2(Rn[1], dz);
    if (POLES) {
        const Vt Qx = fma2(splat2(qa.x), R[0], fma2(splat2(qa.y), R[1], mul2(splat2(qa.z), R[2])));
        const Vt Qy = fma2(splat2(qa.y), R[0], fma2(splat2(qa.w), R[1], mul2(splat2(qyz), R[2])));
        const Vt Qz = fma2(splat2(qa.z), R[0], fma2(splat2(qyz), R[1], mul2(splat2(qzz), R[2])));
        const Vt RQR = mul2(fma2(Qx, R[0], fma2(Qy, R[1], mul2(Qz, R[2]))), splat2(T(1.0 / 3.0)));
        c = fma2(splat2(q), Rn[1], fma2(RQR, Rn[3], c));
        tr = fma2(splat2(q), Rn[0], fma2(RQR, Rn[2], tr));
        const Vt r3 = mul2(Rn[2], splat2(T(2.0 / 3.0))), r2 = mul2(Rn[1], splat2(T(-2.0 / 3.0)));
        tx = fma2(r3, Qx, tx);
        ty = fma2(r3, Qy, ty);
        tz = fma2(r3, Qz, tz);
        a.qxx = fma2(r2, splat2(qa.x), a.qxx);
        a.qyy = fma2(r2, splat2(qa.w), a.qyy);
        a.qzz = fma2(r2, splat2(qzz), a.qzz);
        a.gxy = fma2(r2, splat2(qa.y), a.gxy);
        a.gxz = fma2(r2, splat2(qa.z), a.gxz);
        a.gyz = fma2(r2, splat2(qyz), a.gyz);
    }
    c = mul2(c, splat2(T(-0.5)));
    tx = fma2(c, R[0], tx);
    ty = fma2(c, R[1], ty);
    tz = fma2(c, R[2], tz);
    a.gtr = add2(a.gtr, tr);
    a.gxx = fma2(tx, R[0], a.gxx);
    a.gyy = fma2(ty, R[1], a.gyy);
    a.gzz = fma2(tz, R[2], a.gzz);
    a.gxy = fma2(tx, R[1], fma2(ty, R[0], a.gxy));
    a.gxz = fma2(tx, R[2], fma2(tz, R[0], a.gxz));
    a.gyz = fma2(ty, R[2], fma2(tz, R[1], a.gyz));
}

// a target's own multipoles: charge, dipole, quadrupole (xx xy xz yy yz zz) and induced dipole
template <class X>
struct OwnPoles {
    X q, d[3], Q[6], mu[3];
};
// component C of the force (over f) of those multipoles in the fields of the sums a[0..FO-1] (order of fold)
template <int C, class X>
__device__ __forceinline__ X own_force(const X *a, const OwnPoles<X> &m) {
    const X tr = a[9];
    const X Eab[3][3] = {{2 * a[3] + tr, a[6], a[7]}, {a[6], 2 * a[4] + tr, a[8]}, {a[7], a[8], 2 * a[5] + tr}};
    const X G[3][3] = {{a[23], a[26], a[27]}, {a[26], a[24], a[28]}, {a[27], a[28], a[25]}};
    const X *S = a + 10, *W = a + 20, *Q = m.Q;
    // sum_bc Q_bc E_abc, with sum_bc Q_bc delta_bc = 0
    const X QS[3] = {Q[0] * 3 * S[0] + Q[3] * S[5] + Q[5] * S[7] + 2 * (Q[1] * S[3] + Q[2] * S[4] + Q[4] * S[9]),
                     Q[0] * S[3] + Q[3] * 3 * S[1] + Q[5] * S[8] + 2 * (Q[1] * S[5] + Q[2] * S[9] + Q[4] * S[6]),
                     Q[0] * S[4] + Q[3] * S[6] + Q[5] * 3 * S[2] + 2 * (Q[1] * S[9] + Q[2] * S[7] + Q[4] * S[8])};
    const X QW[3] = {Q[0] * W[0] + Q[1] * W[1] + Q[2] * W[2], Q[1] * W[0] + Q[3] * W[1] + Q[4] * W[2],
                     Q[2] * W[0] + Q[4] * W[1] + Q[5] * W[2]};
    return m.q * a[C] + m.d[0] * Eab[0][C] + m.d[1] * Eab[1][C] + m.d[2] * Eab[2][C] + (QS[C] + 2 * QW[C]) * X(1.0 / 3.0) +
           m.mu[0] * G[0][C] + m.mu[1] * G[1][C] + m.mu[2] * G[2][C];
}

// The same from sums in compensated FP32 pairs (hi, lo): every product with hi exact (its rounding error by an
// fma) and added to a compensated pair, the quadrupole's terms apart for their factor of a third.
struct WideDot {
    F2 s = {0.f, 0.f};
    __device__ __forceinline__ void add(float c, float2 a) {
        const float p = c * a.x;
        f2_add(s, p);
        s.lo += fmaf(c, a.y, fmaf(c, a.x, -p));
    }
    __device__ __forceinline__ double value() const { return f2d_exact(s.hi) + f2d_exact(s.lo); }
};
template <int C>
__device__ __forceinline__ double own_force_wide(const float2 *a, const OwnPoles<float> &m) {
    constexpr int X = (C + 1) % 3, Y = (C + 2) % 3;             // the other two components
    constexpr int AT[3][3] = {{0, 6, 7}, {6, 0, 8}, {7, 8, 0}};   // xy, xz, yz in E_ab; 20 further in G
    constexpr int S3[3][6] = {{0, 5, 7, 3, 4, 9}, {3, 1, 8, 5, 9, 6}, {4, 6, 2, 9, 7, 8}};   // of Q xx yy zz xy xz yz
    constexpr int QI[6] = {0, 3, 5, 1, 2, 4}, QR[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    WideDot f, t;
    f.add(m.q, a[C]);
    f.add(2 * m.d[C], a[3 + C]);
    f.add(m.d[C], a[9]);
    f.add(m.d[X], a[AT[C][X]]);
    f.add(m.d[Y], a[AT[C][Y]]);
    f.add(m.mu[C], a[23 + C]);
    f.add(m.mu[X], a[20 + AT[C][X]]);
    f.add(m.mu[Y], a[20 + AT[C][Y]]);
#pragma unroll
    for (int k = 0; k < 6; ++k) t.add((k < 3 ? 1 : 2) * m.Q[QI[k]], a[10 + S3[C][k]]);
    t.add(2 * m.Q[QI[C]], a[10 + C]);   // the diagonal's are kept as a third
#pragma unroll
    for (int k = 0; k < 3; ++k) t.add(2 * m.Q[QR[C][k]], a[20 + k]);
    return f.value() + t.value() * (1.0 / 3.0);
}

template <class T>
struct PoleArgs {
    const typename V4<T>::type *posw, *dipd, *quad0, *quad1, *mu;
};
template <class T>
__device__ __forceinline__ OwnPoles<T> own_poles(const PoleArgs<T> &a, int s, int n) {
    OwnPoles<T> m;
    typename V4<T>::type d, c, e, u;
    d.x = d.y = d.z = T(0);
    c = e = u = d;
    c.w = e.w = T(0);
    if (s < n) {
        d = a.dipd[s];
        c = a.quad0[s];
        e = a.quad1[s];
        u = a.mu[s];
    }
    m.q = e.w;
    m.d[0] = d.x; m.d[1] = d.y; m.d[2] = d.z;
    m.Q[0] = c.x; m.Q[1] = c.y; m.Q[2] = c.z; m.Q[3] = c.w; m.Q[4] = e.x; m.Q[5] = e.y;
    m.mu[0] = u.x; m.mu[1] = u.y; m.mu[2] = u.z;
    return m;
}

constexpr int FT = 128;   // threads of a CTA

// VIR: also the pairs' virial, sum over pairs of (dU/dR) R^T = -(1/2) sum over sides of F R^T,
// which needs every side's own force: its share of the sums by itself, and the targets'
// multipoles in registers.
template <class T, int PARTS, bool VIR>
__global__ void __launch_bounds__(FT, sizeof(T) == 4 && !VIR ? 3 : 1) k_pair_forces(
    ListArgs la, PoleArgs<T> src, double *__restrict__ frc, double *__restrict__ gdip, double *__restrict__ gquad,
    int n_pad, PairConsts<T> pc, double fconst, double *__restrict__ vir, int fixed) {
    typedef typename V4<T>::type T4;
    typedef typename Vec<T>::type Vt;
    constexpr int W = Vec<T>::W;
    extern __shared__ __align__(16) unsigned char raw[];
    constexpr int ROW = (AP_CHUNK + 1) * (int)sizeof(T4);
    typedef Layout<T, PARTS> LY;
    const LY ly;
    const RadialConsts<T> rk(pc);
    Targets<T> tg;
    tg.load(src.posw, ly.slot(), ly.h, pc.n, pc.rc2, rk.ta);
    FieldSums<Vt> sum;
    zero_sums<T>(sum);
    OwnPoles<T> own[W];
    Vt vs[9];                       // sum of F R^T over this thread's sides of a chunk (VIR)
    double vsum[9];                 // and over all chunks
    if constexpr (VIR) {
#pragma unroll
        for (int h = 0; h < W; ++h) own[h] = own_poles<T>(src, ly.slot() + h, pc.n);
#pragma unroll
        for (int k = 0; k < 9; ++k) vsum[k] = 0.0;
    }
    const T4 *const from[4] = {src.dipd, src.quad0, src.quad1, src.mu};
    for_chunks<T, PARTS>(raw, la, ly, from, [&](const unsigned *list, int words, int flagged, int) {
        if constexpr (VIR) {
#pragma unroll
            for (int k = 0; k < 9; ++k) vs[k] = splat2(T(0));
        }
        auto side = [&](unsigned e, auto ex) {
            constexpr bool EX = decltype(ex)::value;
            const unsigned char *at = raw + (e & 0xfff0u) * (unsigned)(sizeof(T4) / 16);
            const T4 o = *reinterpret_cast<const T4 *>(at), d = *reinterpret_cast<const T4 *>(at + ROW);
            const T4 qa = *reinterpret_cast<const T4 *>(at + 2 * ROW), qb = *reinterpret_cast<const T4 *>(at + 3 * ROW);
            const T4 mu = *reinterpret_cast<const T4 *>(at + 4 * ROW);
            Vt R[3], Mu[4], Md[4], pen;
            bool exa, exb;
            const Vt r2 = tg.template vector<EX>(o, e, R, pen, exa, exb);
            radial<4, EX>(rk, r2, mul1(tg.w, o.w), pen, exa, exb, Mu, Md);
            auto add = [&](FieldSums<Vt> &a) {
                add_induced<T>(a, R, EX ? Md : Mu, mu);
                if constexpr (EX) {
                    add_gradient<T, true>(a, R, Md, qb.w, d.x, d.y, d.z, qa, qb.x, qb.y);
                    add_gradient<T, false>(a, R, Mu, T(0), mu.x, mu.y, mu.z, qa, T(0), T(0));
                } else {
                    add_gradient<T, true>(a, R, Mu, qb.w, d.x + mu.x, d.y + mu.y, d.z + mu.z, qa, qb.x, qb.y);
                }
            };
            // in FP32 the sums take the same operations with and without the virial (in AP_FIXED the
            // forces are the same bit for bit)
            if constexpr (!VIR || W == 2) add(sum);
            if constexpr (VIR) {
                FieldSums<Vt> one;
                zero_sums<T>(one);
                add(one);
                if constexpr (W == 1) {
                    const Vt *o1 = reinterpret_cast<const Vt *>(&one);
                    Vt *t = reinterpret_cast<Vt *>(&sum);
#pragma unroll
                    for (int k = 0; k < FS; ++k) t[k] = add2(t[k], o1[k]);
                }
                Vt of[FO];
                fold(one, of);
#pragma unroll
                for (int h = 0; h < W; ++h) {
                    T v[FO], F[3];
#pragma unroll
                    for (int k = 0; k < FO; ++k) v[k] = Vec<T>::get(of[k], h);
                    F[0] = own_force<0>(v, own[h]);
                    F[1] = own_force<1>(v, own[h]);
                    F[2] = own_force<2>(v, own[h]);
#pragma unroll
                    for (int x = 0; x < 3; ++x)
#pragma unroll
                        for (int y = 0; y < 3; ++y) {
                            T *t = reinterpret_cast<T *>(&vs[3 * x + y]) + h;
                            *t = fma(F[x], Vec<T>::get(R[y], h), *t);
                        }
                }
            }
        };
        walk(list, words, flagged, ly.first, ly.STRIDE, [&](unsigned e) { side(e, std::true_type()); },
             [&](unsigned e) { side(e, std::false_type()); });
        if constexpr (VIR) {
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                vsum[k] += (double)Vec<T>::get(vs[k], 0);
                if (W == 2) vsum[k] += (double)Vec<T>::get(vs[k], 1);
            }
        }
    });
    // The sums of a target's threads through shared memory (the staged candidates are done with): number k
    // of target h at red[(W k + h) FT + tid]. In FP32 they are compensated pairs, and so is what the target's own
    // multipoles make of them.
    __syncthreads();
    T *red = reinterpret_cast<T *>(raw);
    Vt *tot = reinterpret_cast<Vt *>(red + W * FO * FT);
    {
        Vt v[FO];
        fold(sum, v);
#pragma unroll
        for (int k = 0; k < FO; ++k)
#pragma unroll
            for (int h = 0; h < W; ++h) red[(W * k + h) * FT + threadIdx.x] = Vec<T>::get(v[k], h);
    }
    __syncthreads();
    constexpr int NT = 2 * LY::PAIRS;   // targets of this CTA
    if constexpr (W == 2) {
        for (int q = threadIdx.x; q < FO * LY::PAIRS; q += FT) {
            const int k = q / LY::PAIRS, pp = q % LY::PAIRS;
            const float *r = red + 2 * k * FT + pp * LY::TP;
            float2 hi = make_float2(0.f, 0.f), lo = hi;
#pragma unroll
            for (int i = 0; i < LY::TP; i += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(r + i), b = *reinterpret_cast<const float4 *>(r + FT + i);
                if (i) f2_add(hi, lo, make_float2(a.x, b.x));
                else hi = make_float2(a.x, b.x);
                f2_add(hi, lo, make_float2(a.y, b.y));
                f2_add(hi, lo, make_float2(a.z, b.z));
                f2_add(hi, lo, make_float2(a.w, b.w));
            }
            tot[2 * pp * (FO + 1) + k] = make_float2(hi.x, lo.x);
            tot[(2 * pp + 1) * (FO + 1) + k] = make_float2(hi.y, lo.y);
        }
    } else {
        for (int q = threadIdx.x; q < FO * NT; q += FT) {
            const int k = q / NT, t = q % NT, pp = t >> 1, h = t & 1;
            const T *r = red + k * FT + pp * LY::TP + h;
            T v = T(0);
#pragma unroll
            for (int i = 0; i < LY::TP; i += 2) v += r[i];
            tot[t * (FO + 1) + k] = v;
        }
    }
    __syncthreads();
    // a warp each for the components of the force, and one for the torque sources
    const int t = threadIdx.x & 31, part = threadIdx.x >> 5;
    if (t < NT) {
        const int slot = ly.I * 32 + (int)(blockIdx.x % PARTS) * NT + t;
        const Vt *a = tot + t * (FO + 1);
        if (part < 3) {
            const OwnPoles<T> m = own_poles<T>(src, slot, pc.n);
            double F;
            if constexpr (W == 2)
                F = part == 0 ? own_force_wide<0>(a, m) : part == 1 ? own_force_wide<1>(a, m) : own_force_wide<2>(a, m);
            else
                F = part == 0 ? own_force<0>(a, m) : part == 1 ? own_force<1>(a, m) : own_force<2>(a, m);
            store_acc<double>(frc + (size_t)part * n_pad + slot, -fconst * F, fixed);
        } else {
            const int at[6] = {3, 6, 7, 4, 8, 5};   // E_ab: xx xy xz yy yz zz, the diagonal's halved
            auto value = [&](int k) {
                if constexpr (W == 2) return f2d_exact(a[k].x) + f2d_exact(a[k].y);
                else return a[k];
            };
            for (int c = 0; c < 3; ++c) store_acc<double>(gdip + (size_t)c * n_pad + slot, fconst * value(c), fixed);
            for (int c = 0; c < 6; ++c)
                store_acc<double>(gquad + (size_t)c * n_pad + slot, fconst * (c == 0 || c == 3 || c == 5 ? 2.0 / 3.0 : 1.0 / 3.0) * value(at[c]), fixed);
        }
    }
    if constexpr (VIR) {
        double v[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) v[k] = 0.5 * fconst * vsum[k];
        if (fixed) {
            long long vf[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) vf[k] = ap_to_fx(v[k]);
            block_add9<FT>(vf, vir);
        } else {
            block_add9<FT>(v, vir);
        }
    }
}

// reciprocal-space gradient and source terms per atom
// D: phi_mu derivatives [20][n_pad] then phi_M derivatives [10][n_pad] (component order of pme.cu)
// one atom's share of the reciprocal virial from its potential derivatives (layout of D as in
// k_recip_forces), its induced dipole and its global multipoles
template <class T>
__device__ __forceinline__ void recip_atom_virial(const double *__restrict__ D, const double *__restrict__ mu,
                                                  const typename V4<T>::type *__restrict__ dipd,
                                                  const typename V4<T>::type *__restrict__ quad0,
                                                  const typename V4<T>::type *__restrict__ quad1, int s, int n_pad,
                                                  double f, double *v) {
    typedef T C;
    auto Du = [&](int c) { return (C)D[(size_t)c * n_pad + s]; };
    auto DM = [&](int c) { return (C)D[(size_t)(20 + c) * n_pad + s]; };
    const C m[3] = {(C)mu[s], (C)mu[n_pad + s], (C)mu[2 * n_pad + s]};
    const typename V4<T>::type b = dipd[s], c = quad0[s], d = quad1[s];
    const C dd[3] = {b.x, b.y, b.z};
    const C Q[3][3] = {{c.x, c.y, c.z}, {c.y, c.w, d.x}, {c.z, d.x, d.y}};
    const C Hu[3][3] = {{Du(4), Du(7), Du(8)}, {Du(7), Du(5), Du(9)}, {Du(8), Du(9), Du(6)}};
    const C gu[3] = {Du(1), Du(2), Du(3)}, gM[3] = {DM(1), DM(2), DM(3)};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const C hq = Hu[a][0] * Q[0][e] + Hu[a][1] * Q[1][e] + Hu[a][2] * Q[2][e];
            v[3 * a + e] = -f * (double)((gM[a] + gu[a]) * m[e] + gu[a] * dd[e] + C(2.0 / 3.0) * hq);
        }
}

// VIR (blocks of 128 threads): also the atoms' share of the reciprocal virial,
// -f [grad phi_{M+mu} mu^T + grad phi_mu d^T + (2/3) H(phi_mu) Q]
template <class T, bool VIR>
__global__ void k_recip_forces(const double *__restrict__ D, const double *__restrict__ mu,
                               const typename V4<T>::type *__restrict__ posq,
                               const typename V4<T>::type *__restrict__ dipd,
                               const typename V4<T>::type *__restrict__ quad0,
                               const typename V4<T>::type *__restrict__ quad1, int n, int n_pad, double f,
                               double self_coef, double *__restrict__ frc, double *__restrict__ gdip,
                               double *__restrict__ gquad, int fixed, double *__restrict__ vir) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (VIR) {
        double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        if (s < n) recip_atom_virial<T>(D, mu, dipd, quad0, quad1, s, n_pad, f, v);
        if (fixed) {
            long long vf[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) vf[k] = ap_to_fx(v[k]);
            block_add9<128>(vf, vir);
        } else {
            block_add9<128>(v, vir);
        }
    }
    if (s >= n) return;
    typedef T C;   // FP32 in the mixed and fixed modes (FP64 is slow on this part), FP64 in AP_FP64
    auto Du = [&](int c) { return (C)D[(size_t)c * n_pad + s]; };
    auto DM = [&](int c) { return (C)D[(size_t)(20 + c) * n_pad + s]; };
    const C m[3] = {(C)mu[s], (C)mu[n_pad + s], (C)mu[2 * n_pad + s]};
    typename V4<T>::type a = posq[s], b = dipd[s], c = quad0[s], d = quad1[s];
    const C q = a.w, dd[3] = {b.x, b.y, b.z};
    const C Qxx = c.x, Qxy = c.y, Qxz = c.z, Qyy = c.w, Qyz = d.x, Qzz = d.y;
    // symmetric Hessians: index (xx yy zz xy xz yz) -> 4..9
    C Hu[3][3] = {{Du(4), Du(7), Du(8)}, {Du(7), Du(5), Du(9)}, {Du(8), Du(9), Du(6)}};
    C HM[3][3] = {{DM(4), DM(7), DM(8)}, {DM(7), DM(5), DM(9)}, {DM(8), DM(9), DM(6)}};
    const C gu[3] = {Du(1), Du(2), Du(3)};
    // sum_bc Q_bc T_abc with T the third derivatives of phi_mu
    const C Txxx = Du(10), Tyyy = Du(11), Tzzz = Du(12), Txxy = Du(13), Txxz = Du(14), Txyy = Du(15),
                 Tyyz = Du(16), Txzz = Du(17), Tyzz = Du(18), Txyz = Du(19);
    const C QT[3] = {
        Qxx * Txxx + Qyy * Txyy + Qzz * Txzz + 2 * (Qxy * Txxy + Qxz * Txxz + Qyz * Txyz),
        Qxx * Txxy + Qyy * Tyyy + Qzz * Tyzz + 2 * (Qxy * Txyy + Qxz * Txyz + Qyz * Tyyz),
        Qxx * Txxz + Qyy * Tyyz + Qzz * Tzzz + 2 * (Qxy * Txyz + Qxz * Txzz + Qyz * Tyzz)};
    for (int k = 0; k < 3; ++k) {
        C g = 0;
        for (int l = 0; l < 3; ++l) g += m[l] * (Hu[k][l] + HM[k][l]) + dd[l] * Hu[k][l];
        g += q * gu[k] + QT[k] * C(1.0 / 3.0);
        add_plain(frc, (size_t)k * n_pad + s, -f * (double)g, fixed);
        add_plain(gdip, (size_t)k * n_pad + s, f * (double)gu[k] - f * self_coef * (double)m[k], fixed);
    }
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int k = 0; k < 6; ++k) add_plain(gquad, (size_t)k * n_pad + s, f * (1.0 / 3.0) * (double)Hu[ia[k]][ib[k]], fixed);
}

__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }
template <class C>
__device__ __forceinline__ C dot3(const C *a, const C *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
template <class C>
__device__ __forceinline__ void cross3(const C *a, const C *b, C *o) {
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// frame chain rule: dU/dR = G_d d_l^T + 2 G_Q R Q_l, then through the axis construction
// the chain rule of one atom's frame: forces on the atom and its z- and x-atoms; with v
// given, also its frame vectors' virial (dU/dv) v^T into v[0..8]
template <class C>
__device__ __forceinline__ void frame_chain(const double *__restrict__ gdip, const double *__restrict__ gquad,
                                            const double *__restrict__ rot, const double *__restrict__ mpl,
                                            const double *__restrict__ fvec, const int *__restrict__ frame_s, int n,
                                            int n_pad, double *__restrict__ frc, int fixed, int s, double *vout) {
    if (s >= n) return;
    const int type = frame_s[3 * s];
    if (type != AP_FRAME_Z_THEN_X && type != AP_FRAME_BISECTOR) return;
    const int zs = frame_s[3 * s + 1], xs = frame_s[3 * s + 2];
    C R[3][3];
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) R[a][b] = rot[9 * s + 3 * a + b];
    const double *m = mpl + 10 * s;
    const C dl[3] = {(C)m[1], (C)m[2], (C)m[3]};
    const C Ql[3][3] = {{(C)m[4], (C)m[5], (C)m[6]}, {(C)m[5], (C)m[7], (C)m[8]}, {(C)m[6], (C)m[8], (C)m[9]}};
    const C Gd[3] = {(C)acc_value(gdip, s, fixed), (C)acc_value(gdip, (size_t)n_pad + s, fixed),
                     (C)acc_value(gdip, (size_t)2 * n_pad + s, fixed)};
    C g6[6];
    for (int k = 0; k < 6; ++k) g6[k] = (C)acc_value(gquad, (size_t)k * n_pad + s, fixed);
    const C GQ[3][3] = {{g6[0], g6[1], g6[2]}, {g6[1], g6[3], g6[4]}, {g6[2], g6[4], g6[5]}};
    C RQ[3][3], dR[3][3];
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) RQ[a][b] = R[a][0] * Ql[0][b] + R[a][1] * Ql[1][b] + R[a][2] * Ql[2][b];
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b)
            dR[a][b] = Gd[a] * dl[b] + C(2) * (GQ[a][0] * RQ[0][b] + GQ[a][1] * RQ[1][b] + GQ[a][2] * RQ[2][b]);
    C gx[3], gy[3], gz[3], xa[3], za[3];
    for (int a = 0; a < 3; ++a) {
        gx[a] = dR[a][0]; gy[a] = dR[a][1]; gz[a] = dR[a][2];
        xa[a] = R[a][0]; za[a] = R[a][2];
    }
    C t[3];
    cross3(gy, za, t);
    for (int a = 0; a < 3; ++a) gx[a] += t[a];
    cross3(xa, gy, t);
    for (int a = 0; a < 3; ++a) gz[a] += t[a];
    const C vz[3] = {(C)fvec[6 * s], (C)fvec[6 * s + 1], (C)fvec[6 * s + 2]};
    const C vx[3] = {(C)fvec[6 * s + 3], (C)fvec[6 * s + 4], (C)fvec[6 * s + 5]};
    C g_vz[3], g_vx[3];
    if (type == AP_FRAME_Z_THEN_X) {
        const C vxz = dot3(vx, za);
        C w[3];
        for (int a = 0; a < 3; ++a) w[a] = vx[a] - vxz * za[a];
        // reciprocal norms with rsqrt: FP64 division and sqrt are slow on this part
        const C inw = rsq(dot3(w, w)), inz = rsq(dot3(vz, vz));
        const C gxx = dot3(gx, xa);
        C gw[3];
        for (int a = 0; a < 3; ++a) gw[a] = (gx[a] - gxx * xa[a]) * inw;
        const C gwz = dot3(gw, za);
        for (int a = 0; a < 3; ++a) {
            g_vx[a] = gw[a] - gwz * za[a];
            gz[a] = gz[a] - gwz * vx[a] - vxz * gw[a];
        }
        const C gzz = dot3(gz, za);
        for (int a = 0; a < 3; ++a) g_vz[a] = (gz[a] - gzz * za[a]) * inz;
    } else {
        const C in1 = rsq(dot3(vz, vz)), in2 = rsq(dot3(vx, vx));
        C u1[3], u2[3], sv[3], w[3];
        for (int a = 0; a < 3; ++a) { u1[a] = vz[a] * in1; u2[a] = vx[a] * in2; sv[a] = u1[a] + u2[a]; }
        const C u2z = dot3(u2, za);
        for (int a = 0; a < 3; ++a) w[a] = u2[a] - u2z * za[a];
        const C inw = rsq(dot3(w, w)), ins = rsq(dot3(sv, sv));
        const C gxx = dot3(gx, xa);
        C gw[3], gu2[3], gs[3];
        for (int a = 0; a < 3; ++a) gw[a] = (gx[a] - gxx * xa[a]) * inw;
        const C gwz = dot3(gw, za);
        for (int a = 0; a < 3; ++a) {
            gu2[a] = gw[a] - gwz * za[a];
            gz[a] = gz[a] - gwz * u2[a] - u2z * gw[a];
        }
        const C gzz = dot3(gz, za);
        for (int a = 0; a < 3; ++a) gs[a] = (gz[a] - gzz * za[a]) * ins;
        for (int a = 0; a < 3; ++a) gu2[a] += gs[a];
        const C a1 = dot3(gs, u1), a2 = dot3(gu2, u2);
        for (int a = 0; a < 3; ++a) {
            g_vz[a] = (gs[a] - a1 * u1[a]) * in1;
            g_vx[a] = (gu2[a] - a2 * u2[a]) * in2;
        }
    }
    for (int a = 0; a < 3; ++a) {
        if (fixed) {
            unsigned long long *fx = reinterpret_cast<unsigned long long *>(frc);
            atomicAdd(fx + a * n_pad + zs, (unsigned long long)ap_to_fx(-(double)g_vz[a]));
            atomicAdd(fx + a * n_pad + xs, (unsigned long long)ap_to_fx(-(double)g_vx[a]));
            atomicAdd(fx + a * n_pad + s, (unsigned long long)ap_to_fx((double)g_vz[a] + (double)g_vx[a]));
        } else {
            atomicAdd(frc + a * n_pad + zs, -(double)g_vz[a]);
            atomicAdd(frc + a * n_pad + xs, -(double)g_vx[a]);
            atomicAdd(frc + a * n_pad + s, (double)g_vz[a] + (double)g_vx[a]);
        }
    }
    if (vout) {
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                vout[3 * a + b] = (double)g_vz[a] * (double)vz[b] + (double)g_vx[a] * (double)vx[b];
    }
}

// VIR (blocks of 128 threads): also the frames' share of the virial, sum over the frame
// vectors v of (dU/dv) v^T
template <class C, bool VIR>
__global__ void k_frame_forces(const double *__restrict__ gdip, const double *__restrict__ gquad,
                               const double *__restrict__ rot, const double *__restrict__ mpl,
                               const double *__restrict__ fvec, const int *__restrict__ frame_s, int n, int n_pad,
                               double *__restrict__ frc, int fixed, double *__restrict__ vir) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    frame_chain<C>(gdip, gquad, rot, mpl, fvec, frame_s, n, n_pad, frc, fixed, s, VIR ? v : nullptr);
    if constexpr (VIR) {
        if (fixed) {
            long long vf[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) vf[k] = ap_to_fx(v[k]);
            block_add9<128>(vf, vir);
        } else {
            block_add9<128>(v, vir);
        }
    }
}

template <class T>
__global__ void k_mu_load(const double *__restrict__ mu_in, const int *__restrict__ perm, int n, int n_pad,
                          double *__restrict__ mu_s, typename V4<T>::type *__restrict__ p) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_pad) return;
    double m[3] = {0, 0, 0};
    if (s < n) {
        int i = perm[s];
        for (int c = 0; c < 3; ++c) m[c] = mu_in[3 * i + c];
    }
    for (int c = 0; c < 3; ++c) mu_s[c * n_pad + s] = m[c];
    typename V4<T>::type v;
    v.x = (T)m[0]; v.y = (T)m[1]; v.z = (T)m[2]; v.w = (T)0;
    p[s] = v;
}

__global__ void k_energy(const double *__restrict__ mu, const double *__restrict__ E, int n_pad, double scale,
                         double *__restrict__ out, int fixed) {
    __shared__ double sm[8];
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    double v = 0.0;
    if (s < n_pad)
        for (int c = 0; c < 3; ++c) v += mu[c * n_pad + s] * E[c * n_pad + s];
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w];
        if (fixed)   // energy in fixed point with 30 fractional bits: order-independent sum
            atomicAdd(reinterpret_cast<unsigned long long *>(out), (unsigned long long)llrint(scale * t * 1073741824.0));
        else
            atomicAdd(out, scale * t);
    }
}

// fixed-point energy (30 fractional bits) -> FP64
__global__ void k_energy_out(const double *__restrict__ e, double *__restrict__ out) {
    *out = (double)*reinterpret_cast<const long long *>(e) * (1.0 / 1073741824.0);
}

// force accumulators in fixed point, sorted slots -> FP64, caller order
__global__ void k_unsort3_fx(const double *__restrict__ src, int n_pad, const int *__restrict__ iperm, int n,
                             double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int s = iperm[i];
    for (int c = 0; c < 3; ++c) out[3 * i + c] = acc_value(src, (size_t)c * n_pad + s, 1);
}

// the candidates' rows, or the reduction of the sums
template <class T>
constexpr size_t pair_forces_bytes() {
    return std::max(5 * (AP_CHUNK + 1) * sizeof(typename V4<T>::type),
                    sizeof(T) * Vec<T>::W * FO * FT + sizeof(double) * 32 * (FO + 1));
}
template <class T, int PARTS>
int init_p(ap_ctx *ctx) {
    AP_CUDA(allow_smem(k_pair_forces<T, PARTS, false>, pair_forces_bytes<T>()));
    AP_CUDA(allow_smem(k_pair_forces<T, PARTS, true>, pair_forces_bytes<T>()));
    return AP_OK;
}
template <class T>
int init_t(ap_ctx *ctx) { return quarter_blocks(ctx) ? init_p<T, 4>(ctx) : init_p<T, 1>(ctx); }

// the real-space force kernel over the current pair lists with the dipoles in ctx->p and the
// multipoles (dipd, quad0, quad1) given, written to frc, gdip and gquad; with vir given, also the
// pairs' virial added to vir[0..8]
template <class T, int PARTS>
int pair_forces_p(ap_ctx *ctx, cudaStream_t s, const PoleArgs<T> &src, double *frc, double *gdip, double *gquad,
                  double *vir) {
    auto kern = vir ? k_pair_forces<T, PARTS, true> : k_pair_forces<T, PARTS, false>;
    const size_t bytes = pair_forces_bytes<T>();
    kern<<<ctx->n_blocks * PARTS, FT, bytes, s>>>(list_args(ctx), src, frc, gdip, gquad, ctx->n_pad, make_consts<T>(ctx),
                                                  AP_COULOMB, vir, ctx->fixed);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}
template <class T>
int pair_forces_t(ap_ctx *ctx, cudaStream_t s, const void *dipd, const void *quad0, const void *quad1,
                  double *frc, double *gdip, double *gquad, double *vir = nullptr) {
    typedef typename V4<T>::type T4;
    const PoleArgs<T> src = {(const T4 *)ctx->posw, (const T4 *)dipd, (const T4 *)quad0, (const T4 *)quad1, (const T4 *)ctx->p};
    return quarter_blocks(ctx) ? pair_forces_p<T, 4>(ctx, s, src, frc, gdip, gquad, vir)
                               : pair_forces_p<T, 1>(ctx, s, src, frc, gdip, gquad, vir);
}

// `extra`, if given, runs on the force stream after the pair and reciprocal terms and before
// the frame chain rule: it may add to ctx->frc, ctx->gdip and ctx->gquad (and, while
// ctx->vir_active is set, to that virial accumulator). vir: nine device slots (FP64, or fixed
// point in AP_FIXED) cleared here and accumulating the virial, or NULL.
template <class T>
int forces_t(ap_ctx *ctx, const double *d_mu, double *d_energy, double *d_forces,
             int (*extra)(ap_ctx *, cudaStream_t), double *vir) {
    typedef typename V4<T>::type T4;
    cudaStream_t s = ctx->s0;
    const int n = ctx->n, n_pad = ctx->n_pad;
    const double f = AP_COULOMB;
    const double self_coef = 4.0 * std::pow(ctx->prm.ewald_beta, 3) / (3.0 * AP_SQRT_PI);
    if (vir) AP_CUDA(cudaMemsetAsync(vir, 0, sizeof(double) * 9, s));
    k_mu_load<T><<<ap_grid_for(n_pad, 256), 256, 0, s>>>(d_mu, ctx->perm, n, n_pad, ctx->mu_s, (T4 *)ctx->p);
    // reciprocal-space potential derivatives on the second stream, concurrent with the
    // energy and the real-space pair forces (they write only gbuf and the grid); joined
    // before the kernels that update the force arrays per atom
    const cudaStream_t aux = aux_stream(ctx, s, ctx->s1);
    if (aux != s) {
        AP_CUDA(cudaEventRecord(ctx->ev_fork, s));
        AP_CUDA(cudaStreamWaitEvent(aux, ctx->ev_fork, 0));
    }
    int rc = pme_forces_derivs(ctx, ctx->p, ctx->gbuf, aux, vir);
    if (rc) return rc;
    AP_CUDA(cudaMemsetAsync(ctx->red + 8, 0, sizeof(double), s));
    // energy
    k_energy<<<ap_grid_for(n_pad, 256), 256, 0, s>>>(ctx->mu_s, ctx->E, n_pad, -0.5 * f, ctx->red + 8, ctx->fixed);
    rc = pair_forces_t<T>(ctx, s, ctx->dipd, ctx->quad0, ctx->quad1, ctx->frc, ctx->gdip, ctx->gquad, vir);
    if (rc) return rc;
    if (aux != s) {
        AP_CUDA(cudaEventRecord(ctx->ev_join, aux));
        AP_CUDA(cudaStreamWaitEvent(s, ctx->ev_join, 0));
    }
    auto krec = vir ? k_recip_forces<T, true> : k_recip_forces<T, false>;
    krec<<<ap_grid_for(n, 128), 128, 0, s>>>(ctx->gbuf, ctx->mu_s, (const T4 *)ctx->posq, (const T4 *)ctx->dipd,
                                            (const T4 *)ctx->quad0, (const T4 *)ctx->quad1, n, n_pad, f, self_coef,
                                            ctx->frc, ctx->gdip, ctx->gquad, ctx->fixed, vir);
    AP_CUDA(cudaGetLastError());
    ctx->vir_active = vir;
    rc = extra ? extra(ctx, s) : AP_OK;
    ctx->vir_active = nullptr;
    if (rc) return rc;
    auto kfr = vir ? k_frame_forces<T, true> : k_frame_forces<T, false>;
    kfr<<<ap_grid_for(n, 128), 128, 0, s>>>(ctx->gdip, ctx->gquad, ctx->rot, ctx->mpl, ctx->fvec, ctx->frame_s, n,
                                           n_pad, ctx->frc, ctx->fixed, vir);
    AP_CUDA(cudaGetLastError());
    if (ctx->fixed) {
        k_unsort3_fx<<<ap_grid_for(n, 256), 256, 0, s>>>(ctx->frc, n_pad, ctx->iperm, n, d_forces);
        k_energy_out<<<1, 1, 0, s>>>(ctx->red + 8, d_energy);
    } else {
        unsort3(ctx, ctx->frc, d_forces, s);
        AP_CUDA(cudaMemcpyAsync(d_energy, ctx->red + 8, sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

// forces of the mutual term alone, -(f/2) mu . T mu, for caller-order dipoles d_mu: the
// single-set force path with the permanent multipoles replaced by zeros (mz: posq, dipd,
// quad0, quad1 with q, d and Q zero, positions and Thole factors kept) and without the
// permanent potential's reciprocal part or the frame chain rule. gd, gq: scratch for the
// dipole and quadrupole derivatives the kernels also write (not used). vir: as in forces_t.
template <class T>
int mutual_forces_t(ap_ctx *ctx, const double *d_mu, void *const *mz, double *gd, double *gq, double *d_forces,
                    double *vir) {
    typedef typename V4<T>::type T4;
    cudaStream_t s = ctx->s0;
    const int n = ctx->n, n_pad = ctx->n_pad;
    const double f = AP_COULOMB;
    const double self_coef = 4.0 * std::pow(ctx->prm.ewald_beta, 3) / (3.0 * AP_SQRT_PI);
    if (vir) AP_CUDA(cudaMemsetAsync(vir, 0, sizeof(double) * 9, s));
    k_mu_load<T><<<ap_grid_for(n_pad, 256), 256, 0, s>>>(d_mu, ctx->perm, n, n_pad, ctx->mu_s, (T4 *)ctx->p);
    AP_CUDA(cudaEventRecord(ctx->ev_fork, s));
    AP_CUDA(cudaStreamWaitEvent(ctx->s1, ctx->ev_fork, 0));
    int rc = pme_forces_derivs_mu(ctx, ctx->p, ctx->gbuf, ctx->s1, vir);
    if (rc) return rc;
    rc = pair_forces_t<T>(ctx, s, mz[1], mz[2], mz[3], ctx->frc, gd, gq, vir);
    if (rc) return rc;
    AP_CUDA(cudaEventRecord(ctx->ev_join, ctx->s1));
    AP_CUDA(cudaStreamWaitEvent(s, ctx->ev_join, 0));
    auto krec = vir ? k_recip_forces<T, true> : k_recip_forces<T, false>;
    krec<<<ap_grid_for(n, 128), 128, 0, s>>>(ctx->gbuf, ctx->mu_s, (const T4 *)mz[0], (const T4 *)mz[1],
                                            (const T4 *)mz[2], (const T4 *)mz[3], n, n_pad, f, self_coef, ctx->frc,
                                            gd, gq, ctx->fixed, vir);
    AP_CUDA(cudaGetLastError());
    if (ctx->fixed)
        k_unsort3_fx<<<ap_grid_for(n, 256), 256, 0, s>>>(ctx->frc, n_pad, ctx->iperm, n, d_forces);
    else
        unsort3(ctx, ctx->frc, d_forces, s);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

// d_out[0..8] = value(a) - value(b) (b optional) of two virial accumulators in FP64 or (fixed)
// fixed point
__global__ void k_virial_out(const double *__restrict__ a, const double *__restrict__ b, int fixed,
                             double *__restrict__ out) {
    const int k = threadIdx.x;
    if (k >= 9) return;
    double v = acc_value(a, k, fixed);
    if (b) v -= acc_value(b, k, fixed);
    out[k] = v;
}

}  // namespace

int forces_init(ap_ctx *ctx) { return ctx->prec == AP_FP64 ? init_t<double>(ctx) : init_t<float>(ctx); }

int pair_forces_launch(ap_ctx *ctx, cudaStream_t s) {
    return ctx->prec == AP_FP64
               ? pair_forces_t<double>(ctx, s, ctx->dipd, ctx->quad0, ctx->quad1, ctx->frc, ctx->gdip,
                                       ctx->gquad)
               : pair_forces_t<float>(ctx, s, ctx->dipd, ctx->quad0, ctx->quad1, ctx->frc, ctx->gdip,
                                      ctx->gquad);
}

int mutual_forces_run(ap_ctx *ctx, const double *d_mu, void *const *mz, double *gd, double *gq, double *d_forces,
                      double *vir) {
    return ctx->prec == AP_FP64 ? mutual_forces_t<double>(ctx, d_mu, mz, gd, gq, d_forces, vir)
                                : mutual_forces_t<float>(ctx, d_mu, mz, gd, gq, d_forces, vir);
}

// the virial accumulators: slots 16..24 of the context's reduction scratch for a force call,
// 32..40 for the mutual pass of the two-set forces
double *virial_acc(ap_ctx *ctx, int which) { return ctx->red + (which ? 32 : 16); }

int virial_out(ap_ctx *ctx, const double *a, const double *b, double *d_virial) {
    k_virial_out<<<1, 32, 0, ctx->s0>>>(a, b, ctx->fixed, d_virial);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

int forces_run(ap_ctx *ctx, const double *d_mu, double *d_energy, double *d_forces, double *d_virial) {
    double *vir = d_virial ? virial_acc(ctx, 0) : nullptr;
    const int rc = ctx->prec == AP_FP64 ? forces_t<double>(ctx, d_mu, d_energy, d_forces, nullptr, vir)
                                        : forces_t<float>(ctx, d_mu, d_energy, d_forces, nullptr, vir);
    if (rc || !d_virial) return rc;
    return virial_out(ctx, vir, nullptr, d_virial);
}

int forces_run_ex(ap_ctx *ctx, const double *d_mu, double *d_energy, double *d_forces,
                  int (*extra)(ap_ctx *, cudaStream_t), double *vir) {
    return ctx->prec == AP_FP64 ? forces_t<double>(ctx, d_mu, d_energy, d_forces, extra, vir)
                                : forces_t<float>(ctx, d_mu, d_energy, d_forces, extra, vir);
}
