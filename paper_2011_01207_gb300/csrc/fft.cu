// The smooth-PME round trip in FP32, phi = C2R[ B C R2C[Q] ], as three kernels:
//   k_fft_planes   one CTA per z-plane: real transforms along x (two rows as one complex line),
//                  then along y, in shared memory;
//   k_fft_columns  one CTA per few (y, x) columns: along z, times B C, and back along z;
//   k_fft_back     one CTA per z-plane: back along y, then along x to real numbers.
// So the grid is read and written three times, in five launches less than the library's transforms
// and a separate product, whose launches were most of their time on the grids of small systems.
//
// A line of N = R1 R2 points (both factors among the register transforms below, at most 16) takes
// two passes (the four-step decomposition: Gentleman & Sande 1966, Bailey 1990): with n = R2 a + b and
// k = k1 + R1 k2, a thread first transforms R1 points over a for one b and multiplies by
// w_N^(b k1), then R2 points over b for one k1. Both passes store where they read, so frequency k
// ends at place R2 k1 + k2 of the line; the way back undoes the passes in the opposite order, so
// nothing is ever reordered: y and z stay in that order between the kernels and the table of B C is
// laid out likewise. Other sizes, and the FP64 mode, use cuFFT.
//
// Measured on GB300: the round trip with the product, cuFFT's R2C and C2R and the product kernel -> here:
//   24^3 20.4 -> 16.3 us, 28 x 32 x 40 20.7 -> 16.7, 50^3 21.9 -> 19.8, 64^3 21.3 -> 20.3, 75^3 45.5 -> 26.2,
//   80^3 26.0 -> 22.5, 96^3 32.7 -> 26.1 (each a little above its kernels' own times: launches bound it at
//   the small end, the latency of a plane's passes at the large one). Half or a quarter of the rows at a time or
//   256 threads per plane are slower at every size (100^3: 28.8 and 36.4 for 25.7 us).
#include "common.cuh"
#include "pair_math.cuh"   // packed add2, sub2, fma2

#include <algorithm>
#include <cmath>
#include <vector>

namespace {

// ---- register transforms --------------------------------------------------------------
constexpr double cos_series(double x) {
    double t = 1.0, s = 1.0;
    for (int k = 1; k < 24; ++k) {
        t *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        s += t;
    }
    return s;
}
constexpr double sin_series(double x) {
    double t = x, s = x;
    for (int k = 1; k < 24; ++k) {
        t *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
        s += t;
    }
    return s;
}
// cos and sin of 2 pi j / R
template <int R>
struct Roots {
    float c[R], s[R];
    constexpr Roots() : c(), s() {
        for (int j = 0; j < R; ++j) {
            const double x = 2.0 * 3.14159265358979323846 * (2 * j > R ? j - R : j) / R;
            c[j] = (float)cos_series(x);
            s[j] = (float)sin_series(x);
        }
    }
};
template <int R>
__device__ constexpr Roots<R> ROOTS{};

// a complex number is a register pair, so its sums are one packed f32x2 operation each
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return sub2(a, b); }
// a w (forward, w = c - i s) or a conj(w) (INV)
template <bool INV>
__device__ __forceinline__ float2 ctw(float2 a, float c, float s) {
    return INV ? make_float2(a.x * c - a.y * s, a.y * c + a.x * s) : make_float2(a.x * c + a.y * s, a.y * c - a.x * s);
}

constexpr int first_factor(int R) {
    return R == 6 || R == 8 || R == 10 || R == 14 ? 2 : R == 9 || R == 12 || R == 15 ? 3 : R == 16 ? 4 : R;
}

// X_k = sum_n v_n e^(-/+ 2 pi i n k / R) in place
template <int R, bool INV>
struct Dft {
    static __device__ __forceinline__ void run(float2 *v) {
        if constexpr (R == 2) {
            const float2 a = v[0];
            v[0] = cadd(a, v[1]);
            v[1] = csub(a, v[1]);
        } else if constexpr (R == 4) {
            const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
            const float2 e = INV ? make_float2(-d.y, d.x) : make_float2(d.y, -d.x);   // -/+ i d
            v[0] = cadd(a, c);
            v[1] = cadd(b, e);
            v[2] = csub(a, c);
            v[3] = csub(b, e);
        } else if constexpr (first_factor(R) == R) {   // 3, 5, 7: sums and differences of v_n and v_(R-n)
            constexpr int H = (R - 1) / 2;
            float2 t[H], d[H], x0 = v[0];
#pragma unroll
            for (int n = 0; n < H; ++n) {
                t[n] = cadd(v[n + 1], v[R - 1 - n]);
                d[n] = csub(v[n + 1], v[R - 1 - n]);
            }
            float2 sum = x0;
#pragma unroll
            for (int n = 0; n < H; ++n) sum = cadd(sum, t[n]);
#pragma unroll
            for (int k = 1; k <= H; ++k) {
                float2 p = x0, q = make_float2(0.f, 0.f);
#pragma unroll
                for (int n = 0; n < H; ++n) {
                    const int j = (n + 1) * k % R;
                    p = fma2(splat2(ROOTS<R>.c[j]), t[n], p);
                    q = fma2(splat2(ROOTS<R>.s[j]), d[n], q);
                }
                const float2 iq = INV ? make_float2(-q.y, q.x) : make_float2(q.y, -q.x);
                v[k] = cadd(p, iq);
                v[R - k] = csub(p, iq);
            }
            v[0] = sum;
        } else {
            constexpr int A = first_factor(R), B = R / A;
            float2 y[R];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                float2 u[A];
#pragma unroll
                for (int a = 0; a < A; ++a) u[a] = v[B * a + b];
                Dft<A, INV>::run(u);
#pragma unroll
                for (int k = 0; k < A; ++k) y[k * B + b] = b * k ? ctw<INV>(u[k], ROOTS<R>.c[b * k], ROOTS<R>.s[b * k]) : u[k];
            }
#pragma unroll
            for (int k = 0; k < A; ++k) {
                Dft<B, INV>::run(y + k * B);
#pragma unroll
                for (int q = 0; q < B; ++q) v[k + A * q] = y[k * B + q];
            }
        }
    }
};

template <int R> struct Int { static constexpr int value = R; };
// f(Int<R>) for a runtime R among the register transforms
template <class F>
__device__ __forceinline__ void with_radix(int R, F f) {
    switch (R) {
    case 2: f(Int<2>()); break;
    case 3: f(Int<3>()); break;
    case 4: f(Int<4>()); break;
    case 5: f(Int<5>()); break;
    case 6: f(Int<6>()); break;
    case 7: f(Int<7>()); break;
    case 8: f(Int<8>()); break;
    case 9: f(Int<9>()); break;
    case 10: f(Int<10>()); break;
    case 12: f(Int<12>()); break;
    case 14: f(Int<14>()); break;
    case 15: f(Int<15>()); break;
    case 16: f(Int<16>()); break;
    }
}
bool radix_ok(int R) { return (R >= 2 && R <= 10) || R == 12 || (R >= 14 && R <= 16); }

// ---- the passes ----------------------------------------------------------------------------
struct Line {
    int N, R1, R2;
    const float2 *tw;     // (cos, sin)(2 pi m / N), m = 0..N-1
};

// `lines` lines in shared memory, point i of line l at buf[l ls + i es]. ST selects where the points
// come from and go to: ld(l, i), st(l, i, v).
// first pass of the way there (over a, for every b), or last of the way back
template <bool INV, class LD, class ST>
__device__ __forceinline__ void pass_a(const Line &L, const float2 *tw, int lines, LD ld, ST st) {
    with_radix(L.R1, [&](auto r) {
        constexpr int R = decltype(r)::value;
        const int items = lines * L.R2;
        for (int q = threadIdx.x; q < items; q += blockDim.x) {
            const int b = q / lines, l = q - b * lines;
            float2 v[R];
#pragma unroll
            for (int a = 0; a < R; ++a) v[a] = ld(l, L.R2 * a + b);
            Dft<R, INV>::run(v);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (!INV && k) {
                    const float2 w = tw[b * k];   // b k < N
                    v[k] = ctw<false>(v[k], w.x, w.y);
                }
                st(l, L.R2 * k + b, v[k]);
            }
        }
    });
}
// second pass of the way there (over b, for every k1), or first of the way back
template <bool INV, class LD, class ST>
__device__ __forceinline__ void pass_b(const Line &L, const float2 *tw, int lines, LD ld, ST st) {
    with_radix(L.R2, [&](auto r) {
        constexpr int R = decltype(r)::value;
        const int items = lines * L.R1;
        for (int q = threadIdx.x; q < items; q += blockDim.x) {
            const int k1 = q / lines, l = q - k1 * lines;
            float2 v[R];
#pragma unroll
            for (int b = 0; b < R; ++b) v[b] = ld(l, R * k1 + b);
            Dft<R, INV>::run(v);
#pragma unroll
            for (int b = 0; b < R; ++b) {
                if (INV && b) {
                    const float2 w = tw[b * k1];
                    v[b] = ctw<true>(v[b], w.x, w.y);
                }
                st(l, R * k1 + b, v[b]);
            }
        }
    });
}

struct FftShape {
    Line x, y, z;
    int Kx, Ky, Kz, hx;
    int pairs;            // row pairs of a plane transformed along x at once
    int ld;               // their line length in shared memory (odd, so that lanes on different lines
                          // use different banks)
};
// the roots of a line's size into shared memory
__device__ __forceinline__ void load_roots(const Line &L, float2 *tw) {
    for (int m = threadIdx.x; m < L.N; m += blockDim.x) tw[m] = __ldg(L.tw + m);
}
// place of frequency k in a transformed line
__device__ __forceinline__ int place(const Line &L, int k) {
    const int k2 = k / L.R1;
    return L.R2 * (k - k2 * L.R1) + k2;
}

// places of the frequencies k and N - k, k = 0..hx-1, of the lines along x
__device__ __forceinline__ void load_places(const FftShape &F, ushort2 *pl) {
    for (int k = threadIdx.x; k < F.hx; k += blockDim.x)
        pl[k] = make_ushort2((unsigned short)place(F.x, k), (unsigned short)place(F.x, k ? F.Kx - k : 0));
}

// shared memory of the plane kernels: the half plane [Ky][hx], the rows' lines, the tables
struct PlaneSmem {
    float2 *H, *Z, *twx, *twy;
    ushort2 *pl;
    __device__ __forceinline__ PlaneSmem(float2 *sh, const FftShape &F) {
        H = sh;
        Z = H + (size_t)F.Ky * F.hx;
        twx = Z + (size_t)F.pairs * F.ld;
        twy = twx + F.Kx;
        pl = reinterpret_cast<ushort2 *>(twy + F.Ky);
        load_roots(F.x, twx);
        load_roots(F.y, twy);
        load_places(F, pl);
    }
};

__global__ void __launch_bounds__(512, 1) k_fft_planes(const float *__restrict__ in, float2 *__restrict__ out, FftShape F) {
    extern __shared__ float2 sh[];
    const PlaneSmem S(sh, F);
    float2 *H = S.H, *Z = S.Z;
    const float *plane = in + (size_t)blockIdx.x * F.Ky * F.Kx;
    const int all = (F.Ky + 1) / 2;
    for (int p0 = 0; p0 < all; p0 += F.pairs) {
        const int np = min(F.pairs, all - p0);
        if (!(F.Kx & 1)) {   // two points of both rows at a time
            const int half = F.Kx / 2;
            for (int q = threadIdx.x; q < np * half; q += blockDim.x) {
                const int p = q / half, x = 2 * (q - p * half), y = 2 * (p0 + p);
                const float2 a = *reinterpret_cast<const float2 *>(plane + (size_t)y * F.Kx + x);
                const float2 b = y + 1 < F.Ky ? *reinterpret_cast<const float2 *>(plane + (size_t)(y + 1) * F.Kx + x)
                                              : make_float2(0.f, 0.f);
                Z[p * F.ld + x] = make_float2(a.x, b.x);
                Z[p * F.ld + x + 1] = make_float2(a.y, b.y);
            }
        } else {
            for (int q = threadIdx.x; q < np * F.Kx; q += blockDim.x) {
                const int p = q / F.Kx, x = q - p * F.Kx, y = 2 * (p0 + p);
                const float a = plane[(size_t)y * F.Kx + x], b = y + 1 < F.Ky ? plane[(size_t)(y + 1) * F.Kx + x] : 0.f;
                Z[p * F.ld + x] = make_float2(a, b);
            }
        }
        __syncthreads();
        auto ld = [&](int l, int i) { return Z[l * F.ld + i]; };
        auto st = [&](int l, int i, float2 v) { Z[l * F.ld + i] = v; };
        pass_a<false>(F.x, S.twx, np, ld, st);
        __syncthreads();
        pass_b<false>(F.x, S.twx, np, ld, st);
        __syncthreads();
        // the two rows' transforms from Z_k and conj Z_(N-k)
        for (int q = threadIdx.x; q < np * F.hx; q += blockDim.x) {
            const int p = q / F.hx, k = q - p * F.hx, y = 2 * (p0 + p);
            const ushort2 at = S.pl[k];
            const float2 a = Z[p * F.ld + at.x], b = Z[p * F.ld + at.y];
            H[(size_t)y * F.hx + k] = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
            if (y + 1 < F.Ky) H[(size_t)(y + 1) * F.hx + k] = make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
        }
        __syncthreads();
    }
    float2 *o = out + (size_t)blockIdx.x * F.Ky * F.hx;
    auto ld = [&](int l, int i) { return H[i * F.hx + l]; };
    pass_a<false>(F.y, S.twy, F.hx, ld, [&](int l, int i, float2 v) { H[i * F.hx + l] = v; });
    __syncthreads();
    pass_b<false>(F.y, S.twy, F.hx, ld, [&](int l, int i, float2 v) { o[(size_t)i * F.hx + l] = v; });
}

// TX columns of the half grid [Kz][plane] (plane = Ky hx points): along z, times green (laid out as
// the transformed grid), and back; or the two ways apart (the virial looks at the transform)
enum { COL_BOTH, COL_THERE, COL_BACK };
template <int TX, int WAY>
__global__ void __launch_bounds__(TX * 16) k_fft_columns(float2 *__restrict__ c, const float *__restrict__ green,
                                                        FftShape F) {
    extern __shared__ float2 sh[];
    float2 *tw = sh + (size_t)TX * F.Kz;
    load_roots(F.z, tw);
    __syncthreads();
    const int plane = F.Ky * F.hx, c0 = blockIdx.x * TX, n = min(TX, plane - c0);
    float2 *g = c + c0;
    auto ld = [&](int l, int i) { return sh[i * TX + l]; };
    auto st = [&](int l, int i, float2 v) { sh[i * TX + l] = v; };
    if constexpr (WAY != COL_BACK) {
        pass_a<false>(F.z, tw, n, [&](int l, int i) { return g[(size_t)i * plane + l]; }, st);
        __syncthreads();
    }
    with_radix(F.z.R2, [&](auto r) {
        constexpr int R = decltype(r)::value;
        const int items = n * F.z.R1;
        for (int q = threadIdx.x; q < items; q += blockDim.x) {
            const int k1 = q / n, l = q - k1 * n;
            float2 v[R];
#pragma unroll
            for (int b = 0; b < R; ++b) v[b] = WAY == COL_BACK ? g[(size_t)(R * k1 + b) * plane + l] : sh[(R * k1 + b) * TX + l];
            if constexpr (WAY != COL_BACK) Dft<R, false>::run(v);
            if constexpr (WAY == COL_THERE) {
#pragma unroll
                for (int b = 0; b < R; ++b) g[(size_t)(R * k1 + b) * plane + l] = v[b];
            } else {
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    const float w = __ldg(green + (size_t)(R * k1 + b) * plane + c0 + l);
                    v[b].x *= w;
                    v[b].y *= w;
                }
                Dft<R, true>::run(v);
#pragma unroll
                for (int b = 0; b < R; ++b) {
                    if (b) {
                        const float2 w = tw[b * k1];
                        v[b] = ctw<true>(v[b], w.x, w.y);
                    }
                    sh[(R * k1 + b) * TX + l] = v[b];
                }
            }
        }
    });
    if constexpr (WAY != COL_THERE) {
        __syncthreads();
        pass_a<true>(F.z, tw, n, ld, [&](int l, int i, float2 v) { g[(size_t)i * plane + l] = v; });
    }
}

__global__ void __launch_bounds__(512, 1) k_fft_back(const float2 *__restrict__ in, float *__restrict__ out, FftShape F) {
    extern __shared__ float2 sh[];
    const PlaneSmem S(sh, F);
    float2 *H = S.H, *Z = S.Z;
    __syncthreads();
    const float2 *src = in + (size_t)blockIdx.x * F.Ky * F.hx;
    float *plane = out + (size_t)blockIdx.x * F.Ky * F.Kx;
    auto put = [&](int l, int i, float2 v) { H[i * F.hx + l] = v; };
    pass_b<true>(F.y, S.twy, F.hx, [&](int l, int i) { return src[(size_t)i * F.hx + l]; }, put);
    __syncthreads();
    pass_a<true>(F.y, S.twy, F.hx, [&](int l, int i) { return H[i * F.hx + l]; }, put);
    __syncthreads();
    const int all = (F.Ky + 1) / 2;
    for (int p0 = 0; p0 < all; p0 += F.pairs) {
        const int np = min(F.pairs, all - p0);
        // two rows as the real and imaginary parts of one line (of k = 0 and, N even, k = N/2 the
        // transform to real numbers takes the real parts)
        for (int q = threadIdx.x; q < np * F.hx; q += blockDim.x) {
            const int p = q / F.hx, k = q - p * F.hx, y = 2 * (p0 + p);
            const ushort2 at = S.pl[k];
            float2 a = H[(size_t)y * F.hx + k], b = y + 1 < F.Ky ? H[(size_t)(y + 1) * F.hx + k] : make_float2(0.f, 0.f);
            if (k == 0 || 2 * k == F.Kx) a.y = b.y = 0.f;
            Z[p * F.ld + at.x] = make_float2(a.x - b.y, a.y + b.x);
            if (k && 2 * k != F.Kx) Z[p * F.ld + at.y] = make_float2(a.x + b.y, b.x - a.y);
        }
        __syncthreads();
        auto ld = [&](int l, int i) { return Z[l * F.ld + i]; };
        auto st = [&](int l, int i, float2 v) { Z[l * F.ld + i] = v; };
        pass_b<true>(F.x, S.twx, np, ld, st);
        __syncthreads();
        pass_a<true>(F.x, S.twx, np, ld, st);
        __syncthreads();
        if (!(F.Kx & 1)) {
            const int half = F.Kx / 2;
            for (int q = threadIdx.x; q < np * half; q += blockDim.x) {
                const int p = q / half, x = 2 * (q - p * half), y = 2 * (p0 + p);
                const float2 u = Z[p * F.ld + x], v = Z[p * F.ld + x + 1];
                *reinterpret_cast<float2 *>(plane + (size_t)y * F.Kx + x) = make_float2(u.x, v.x);
                if (y + 1 < F.Ky) *reinterpret_cast<float2 *>(plane + (size_t)(y + 1) * F.Kx + x) = make_float2(u.y, v.y);
            }
        } else {
            for (int q = threadIdx.x; q < np * F.Kx; q += blockDim.x) {
                const int p = q / F.Kx, x = q - p * F.Kx, y = 2 * (p0 + p);
                const float2 v = Z[p * F.ld + x];
                plane[(size_t)y * F.Kx + x] = v.x;
                if (y + 1 < F.Ky) plane[(size_t)(y + 1) * F.Kx + x] = v.y;
            }
        }
        __syncthreads();
    }
}

// N = R1 R2 with both factors register transforms, as even as possible
bool split(int N, int *R1, int *R2) {
    for (int a = (int)std::sqrt((double)N); a >= 2; --a)
        if (N % a == 0 && radix_ok(a) && radix_ok(N / a)) {
            *R1 = a;
            *R2 = N / a;
            return true;
        }
    return false;
}

constexpr size_t MAX_SMEM = 227 * 1024;
// Largest grid: up to here the three kernels take less than the library's transforms and the product
// (times above); at 100^3 the round trip alone is still shorter (27.5 -> 25.0 us) but a solve of 96,000 atoms,
// where it shares the GPU with the pair kernel, takes 2% longer (one CTA per plane leaves a third of the SMs out,
// and its 80 KB of shared memory wait for the pair kernel's CTAs), and at 224^3 the times are 241 -> 249 us.
constexpr size_t FFT_POINTS = 96 * 96 * 96;
size_t plane_bytes(const FftShape &F) {
    return sizeof(float2) * ((size_t)F.Ky * F.hx + (size_t)F.pairs * F.ld + F.Kx + F.Ky) + sizeof(ushort2) * F.hx;
}

FftShape shape_of(const ap_ctx *ctx) {
    FftShape F;
    F.Kx = ctx->K[0];
    F.Ky = ctx->K[1];
    F.Kz = ctx->K[2];
    F.hx = F.Kx / 2 + 1;
    F.ld = F.Kx | 1;
    Line *L[3] = {&F.x, &F.y, &F.z};
    const float2 *tw = ctx->fft_tw;
    for (int d = 0; d < 3; ++d) {
        L[d]->N = ctx->K[d];
        L[d]->tw = tw;
        if (!split(ctx->K[d], &L[d]->R1, &L[d]->R2)) L[d]->R1 = 0;
        if (tw) tw += ctx->K[d];
    }
    // all row pairs at once while they fit, else as many as do (whole warps of lines)
    F.pairs = (F.Ky + 1) / 2;
    const size_t half = sizeof(float2) * (size_t)F.Ky * F.hx;
    if (half >= MAX_SMEM) F.pairs = 0;
    else while (F.pairs > 4 && plane_bytes(F) > MAX_SMEM) F.pairs = (F.pairs + 1) / 2;
    return F;
}

}  // namespace

// whether the context's grid takes the kernels above: FP32, at most FFT_POINTS, every size a product of
// two register transforms, and a half plane with some lines beside it in shared memory
bool fft_supported(const ap_ctx *ctx) {
    if (ctx->prec == AP_FP64) return false;
    const FftShape F = shape_of(ctx);
    return ctx->ngrid <= FFT_POINTS && F.x.R1 && F.y.R1 && F.z.R1 && F.pairs && plane_bytes(F) <= MAX_SMEM;
}

// tables of roots, and B C in the order of the transformed grid (green: natural order [Kz][Ky][hx])
int fft_init(ap_ctx *ctx, const float *green) {
    const FftShape F = shape_of(ctx);
    std::vector<float2> tw;
    for (int d = 0; d < 3; ++d)
        for (int m = 0; m < ctx->K[d]; ++m) {
            const double x = 2.0 * M_PI * m / ctx->K[d];
            tw.push_back(make_float2((float)std::cos(x), (float)std::sin(x)));
        }
    AP_CUDA(cudaMalloc((void **)&ctx->fft_tw, sizeof(float2) * tw.size()));
    AP_CUDA(cudaMemcpy(ctx->fft_tw, tw.data(), sizeof(float2) * tw.size(), cudaMemcpyHostToDevice));
    auto freq = [](const Line &L, int p) { return p / L.R2 + L.R1 * (p % L.R2); };   // frequency at place p
    std::vector<float> g(ctx->ncgrid);
    for (int z = 0; z < F.Kz; ++z)
        for (int y = 0; y < F.Ky; ++y)
            std::copy_n(green + ((size_t)freq(F.z, z) * F.Ky + freq(F.y, y)) * F.hx, F.hx,
                        g.data() + ((size_t)z * F.Ky + y) * F.hx);
    AP_CUDA(cudaMalloc((void **)&ctx->fft_green, sizeof(float) * g.size()));
    AP_CUDA(cudaMemcpy(ctx->fft_green, g.data(), sizeof(float) * g.size(), cudaMemcpyHostToDevice));
    AP_CUDA(cudaFuncSetAttribute(k_fft_planes, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM));
    AP_CUDA(cudaFuncSetAttribute(k_fft_back, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM));
    const int cols = 33 * 256 * (int)sizeof(float2);   // sizes are at most 256
    AP_CUDA(cudaFuncSetAttribute(k_fft_columns<32, COL_BOTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, cols));
    AP_CUDA(cudaFuncSetAttribute(k_fft_columns<32, COL_THERE>, cudaFuncAttributeMaxDynamicSharedMemorySize, cols));
    AP_CUDA(cudaFuncSetAttribute(k_fft_columns<32, COL_BACK>, cudaFuncAttributeMaxDynamicSharedMemorySize, cols));
    return AP_OK;
}

namespace {

int plane_threads(const FftShape &F) {
    const int ty = F.hx * std::max(F.y.R1, F.y.R2), tx = F.pairs * std::max(F.x.R1, F.x.R2);
    return std::min(512, std::max(64, (std::max(tx, ty) + 31) / 32 * 32));
}

template <int WAY>
void columns(const ap_ctx *ctx, const FftShape &F, float2 *c, cudaStream_t s) {
    const int plane = F.Ky * F.hx, r = std::max(F.z.R1, F.z.R2);
    // wider tiles once there are enough columns to fill the GPU with them
    if (plane >= 32 * 2 * ctx->sm_count)
        k_fft_columns<32, WAY><<<(plane + 31) / 32, 32 * r, sizeof(float2) * 33 * F.Kz, s>>>(c, ctx->fft_green, F);
    else
        k_fft_columns<16, WAY><<<(plane + 15) / 16, 16 * r, sizeof(float2) * 17 * F.Kz, s>>>(c, ctx->fft_green, F);
}

}  // namespace

// out = C2R[ B C R2C[in] ] through the complex work grid c (in may be out)
int fft_roundtrip_own(ap_ctx *ctx, const float *in, float2 *c, float *out, cudaStream_t s) {
    const FftShape F = shape_of(ctx);
    const size_t bytes = plane_bytes(F);
    k_fft_planes<<<F.Kz, plane_threads(F), bytes, s>>>(in, c, F);
    columns<COL_BOTH>(ctx, F, c, s);
    k_fft_back<<<F.Kz, plane_threads(F), bytes, s>>>(c, out, F);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

// its two halves: c = R2C[in] in the order of the places, and out = C2R[ B C c ]
int fft_there_own(ap_ctx *ctx, const float *in, float2 *c, cudaStream_t s) {
    const FftShape F = shape_of(ctx);
    k_fft_planes<<<F.Kz, plane_threads(F), plane_bytes(F), s>>>(in, c, F);
    columns<COL_THERE>(ctx, F, c, s);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}
int fft_back_own(ap_ctx *ctx, float2 *c, float *out, cudaStream_t s) {
    const FftShape F = shape_of(ctx);
    columns<COL_BACK>(ctx, F, c, s);
    k_fft_back<<<F.Kz, plane_threads(F), plane_bytes(F), s>>>(c, out, F);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}
// frequency of place p of a transformed line along y (d = 1) or z (d = 2) is p / R2 + R1 (p mod R2);
// R1 = 1, R2 = N (the natural order) where cuFFT is used
int2 fft_factors(const ap_ctx *ctx, int d) {
    if (!ctx->fft_green) return make_int2(1, ctx->K[d]);
    const FftShape F = shape_of(ctx);
    return d == 1 ? make_int2(F.y.R1, F.y.R2) : make_int2(F.z.R1, F.z.R2);
}
