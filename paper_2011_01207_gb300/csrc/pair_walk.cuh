// How the real-space kernels walk the pair lists of a configuration (built by lists.cu).
//
// A CTA of 128 threads takes one block of 32 target atoms, or in small systems a quarter of one
// (Layout). The block's candidate atoms (those within the cutoff of any of its atoms; positions
// next to the block, in its periodic image) are staged in shared memory, at most AP_CHUNK at a
// time. Eight (or 32) threads share target pair p (slots 2 p and 2 p + 1 of the block); in FP32
// each holds both targets in the halves of two-vectors, in FP64 one of them, and walks its share
// of the pair's list: one shared-memory read of a source serves two pairs, and the whole
// evaluation is packed. Nobody else adds to these targets, so their sums stay in registers and
// are stored once: no atomics, no clearing, a fixed order. In FP32 a thread's share of a pair's list (about
// 22 entries of 175 in water at r_c = 7 A) is summed in FP32, and the threads' shares in compensated FP32 pairs.
// (Sums in FP64 from the first entry on change the errors against 64 bits by less than 2 %: those of the
// pairs' own terms are ten times what the sums add.)
//
// A list entry is 16 bits: the candidate's place in shared memory (bits 4-15) and four flags for
// the two targets: excluded pair (bits 0, 1), the target itself (bits 2, 3). An entry stands for
// an atom within the cutoff of at least one of the two targets; the walk tests both distances
// and makes the radial functions of a pair that is out of range exactly zero. A list is a table of eight columns, entry row r of column c in
// half r mod 2 of word (r / 2) 8 + c, so that threads 8 j .. 8 j + 7 read a row together; column c
// holds the candidates in places k with k mod 8 = c as far as its length allows, whose 16-byte
// rows lie in different shared-memory banks. In each column the entries with flags come first,
// then those within the short range of the learned guess, then the rest; the last rows are
// filled up with entries for a phantom candidate far away.
#pragma once
#include "common.cuh"
#include "pair_math.cuh"

struct ListArgs {
    const int *tile_off;             // [n_blocks + 1]
    const int4 *ncand;               // [n_blocks] candidates of the block's four segments
    const int *cand_j;               // slot | AP_CAND_SELF
    const void *cand_pos;            // T4: position relative to the block's origin, Thole factor
    const uint2 *meta;               // [chunk][16] entry offset; rounds of 16 entries, | those with flagged
                                     // entries << 10, | those with flagged or short-range ones << 20
    const unsigned *list;            // two entries per word
    int mult;                        // images a candidate can appear in (1 unless the box is small)
};
inline ListArgs list_args(const ap_ctx *ctx) {
    ListArgs a;
    a.tile_off = ctx->tile_off;
    a.ncand = ctx->ncand;
    a.cand_j = ctx->cand_j;
    a.cand_pos = ctx->cand_pos;
    a.meta = ctx->list_meta;
    a.list = ctx->list;
    a.mult = ctx->list_mult;
    return a;
}

// the candidates of one block: four segments (one per warp of the list kernel)
struct Cands {
    size_t start[4];
    int p1, p2, p3, n;      // ends of the first three segments in the block's order, and the total
    __device__ __forceinline__ Cands(const ListArgs &la, int I) {
        const int t0 = la.tile_off[I], nt = la.tile_off[I + 1] - t0;
        const int4 c = la.ncand[I];
#pragma unroll
        for (int w = 0; w < 4; ++w) start[w] = ((size_t)t0 + segment_tile(nt, w)) * 32 * la.mult;
        p1 = c.x;
        p2 = p1 + c.y;
        p3 = p2 + c.z;
        n = p3 + c.w;
    }
    // place of candidate k (0 <= k < n) in the candidate arrays
    __device__ __forceinline__ size_t at(int k) const {
        if (k < p1) return start[0] + k;
        if (k < p2) return start[1] + (k - p1);
        if (k < p3) return start[2] + (k - p2);
        return start[3] + (k - p3);
    }
};

// Which block, target pair and list words a thread of a CTA of 128 has. PARTS = 1: one CTA per
// block, eight threads per pair. PARTS = 4: four CTAs per block, 32 threads per pair, for systems
// whose blocks alone leave most of the GPU idle (every CTA stages the same candidates).
template <class T, int PARTS>
struct Layout {
    static constexpr int W = Vec<T>::W, TP = 8 * PARTS, PAIRS = 16 / PARTS, STRIDE = W == 2 ? TP : TP / 2;
    int I, p, s, h, first;
    __device__ __forceinline__ Layout() {
        I = blockIdx.x / PARTS;
        p = (blockIdx.x % PARTS) * PAIRS + threadIdx.x / TP;
        s = threadIdx.x % TP;
        h = W == 2 ? 0 : s & 1;              // the thread's (first) target of the pair
        first = W == 2 ? s : s >> 1;         // its first word of the list
    }
    __device__ __forceinline__ int slot() const { return I * 32 + 2 * p + h; }
    // f[3] summed over the threads that share the targets, to acc [3][n_pad]. In FP32 the sums over the
    // threads are compensated (a thread's own share of a list is a plain FP32 sum). Neighbours share them out: the
    // target by bit 0 of s, the component by bits 1 and 2 (x, y, then z twice).
    __device__ __forceinline__ void store3(double *__restrict__ acc, int n_pad, const typename Vec<T>::type *f,
                                           int fixed) const {
        const bool b0 = s & 1, b1 = s & 2, b2 = s & 4;
        const int t = s & 1;
        auto shfl = [](auto v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); };
        if constexpr (W == 2) {
            float hi[3], lo[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                hi[c] = b0 ? f[c].y : f[c].x;
                lo[c] = 0.f;
                f2_add(hi[c], lo[c], shfl(b0 ? f[c].x : f[c].y, 1));
            }
            float vh = b1 ? hi[2] : hi[0], vl = b1 ? lo[2] : lo[0];
            f2_merge(vh, vl, shfl(b1 ? hi[0] : hi[2], 2), shfl(b1 ? lo[0] : lo[2], 2));
            f2_merge(hi[1], lo[1], shfl(hi[1], 2), shfl(lo[1], 2));
            const bool give = !b1 && !b2, keep = !b1 && b2;   // y goes to the threads with bit 2
            const float oh = shfl(give ? hi[1] : vh, 4), ol = shfl(give ? lo[1] : vl, 4);
            if (keep) {
                vh = hi[1];
                vl = lo[1];
            }
            f2_merge(vh, vl, oh, ol);
#pragma unroll
            for (int off = 8; off < TP; off <<= 1) f2_merge(vh, vl, shfl(vh, off), shfl(vl, off));
            if (s < 8 && !(b1 && b2))
                store_acc<double>(acc + (size_t)(b1 ? 2 : b2 ? 1 : 0) * n_pad + I * 32 + 2 * p + t, f2d_exact(vh) + f2d_exact(vl), fixed);
        } else {
            double a[3] = {f[0], f[1], f[2]};
#pragma unroll
            for (int off = 2; off < TP; off <<= 1)
#pragma unroll
                for (int c = 0; c < 3; ++c) a[c] += shfl(a[c], off);
            const int k = s >> 1;   // a thread stores component k of target t
            if (k < 3) store_acc<double>(acc + (size_t)k * n_pad + I * 32 + 2 * p + t, k == 0 ? a[0] : k == 1 ? a[1] : a[2], fixed);
        }
    }
};

// The targets of a thread, and the limits of their r^2 (negative for padding). In FP32 a padding slot can be
// the other half of a real atom's pair, and its terms are evaluated with the rest: it lies far from every
// candidate and from the phantom, so that r^2 is neither zero nor beyond FP32 and the zero exponentials of a pair
// out of range make each of its terms exactly zero. (At the block's origin, where the middle atom of a
// molecule can lie, 1/r is infinite and the slot's sums NaN.)
constexpr float PADDING_AT = 1e6f;
template <class T> struct Targets;
template <> struct Targets<float> {
    float2 x, y, z, w, lim;
    __device__ __forceinline__ void load(const float4 *posw, int s0, int, int n, float rc2, float ta) {
        float4 a = posw[s0], b = posw[s0 + 1];
        const bool va = s0 < n, vb = s0 + 1 < n;
        if (!va) a.x = a.y = a.z = PADDING_AT;
        if (!vb) b.x = b.y = b.z = PADDING_AT;
        x = make_float2(a.x, b.x);
        y = make_float2(a.y, b.y);
        z = make_float2(a.z, b.z);
        w = make_float2(va ? ta * a.w : 0.f, vb ? ta * b.w : 0.f);
        lim = make_float2(va ? rc2 : -1.f, vb ? rc2 : -1.f);
    }
    // R = x_target - x_source of both pairs and r^2; pen: AP_OUT for a pair that is out of range or
    // (EX, by the entry's flags) no pair but the target itself; exa, exb: its excluded pairs
    template <bool EX>
    __device__ __forceinline__ float2 vector(const float4 &o, unsigned e, float2 *R, float2 &pen, bool &exa,
                                             bool &exb) const {
        R[0] = sub1(x, o.x);
        R[1] = sub1(y, o.y);
        R[2] = sub1(z, o.z);
        float2 r2 = fma2(R[0], R[0], fma2(R[1], R[1], mul2(R[2], R[2])));
        const bool ina = r2.x < lim.x && !(EX && (e & 4u)), inb = r2.y < lim.y && !(EX && (e & 8u));
        pen = make_float2(ina ? 0.f : AP_OUT, inb ? 0.f : AP_OUT);
        exa = EX && ina && (e & 1u);
        exb = EX && inb && (e & 2u);
        if (EX) r2 = make_float2(e & 4u ? 1.f : r2.x, e & 8u ? 1.f : r2.y);
        return r2;
    }
};
template <> struct Targets<double> {
    double x, y, z, w, lim;
    int h;
    __device__ __forceinline__ void load(const dvec4 *posw, int s, int half, int n, double rc2, double ta) {
        const dvec4 a = posw[s];
        const bool va = s < n;
        h = half;
        x = va ? a.x : 0.0;
        y = va ? a.y : 0.0;
        z = va ? a.z : 0.0;
        w = va ? ta * a.w : 0.0;
        lim = va ? rc2 : -1.0;
    }
    template <bool EX>
    __device__ __forceinline__ double vector(const dvec4 &o, unsigned e, double *R, double &pen, bool &exa, bool &exb) const {
        R[0] = x - o.x;
        R[1] = y - o.y;
        R[2] = z - o.z;
        e >>= h;
        const double r2 = R[0] * R[0] + R[1] * R[1] + R[2] * R[2];
        const bool in = r2 < lim && !(EX && (e & 4u));
        pen = in ? 0.0 : (double)AP_OUT;
        exa = exb = EX && in && (e & 1u);
        return in ? r2 : 1.0;
    }
};

// the phantom candidate of list padding: out of every target's range, with a Thole factor of zero
// (its multipoles are zero as well)
template <class T>
__device__ __forceinline__ typename V4<T>::type phantom_pos() {
    typename V4<T>::type v;
    v.x = v.y = v.z = T(1e10);
    v.w = T(0);
    return v;
}

// The walk of one thread over its share of a pair's list: `words` words (two entries each), every
// `stride`-th from `first` on, the far entries first: plain(entry), and from the words down that can
// hold entries with flags flagged(entry). (Sums that take their small terms first round less: the
// matvec's error against 64 bits is 4.7e-7 this way and 7.2e-7 with the near pairs first.)
// entry: byte offset of the candidate's 16-byte row (place << 4) with the flags in its low bits.
template <class FA, class FB>
__device__ __forceinline__ void walk(const unsigned *__restrict__ list, int words, int flagged_words, int first, int stride,
                                     FA flagged, FB plain) {
    if (first >= words) return;
    int w = first + (words - 1 - first) / stride * stride;
    unsigned next = __ldg(list + w);
    for (; w >= flagged_words; w -= stride) {
        const unsigned e = next;
        if (w >= stride) next = __ldg(list + w - stride);
        plain(e >> 16);
        plain(e & 0xffffu);
    }
    for (; w >= 0; w -= stride) {
        const unsigned e = next;
        if (w >= stride) next = __ldg(list + w - stride);
        flagged(e >> 16);
        flagged(e & 0xffffu);
    }
}
// a pair's list as k_pair_lists describes it: all words, and those with flagged or short-range entries
__device__ __forceinline__ int meta_words(uint2 m) { return (int)(m.y & 1023u) * 8; }
__device__ __forceinline__ int meta_flagged(uint2 m) { return (int)((m.y >> 10) & 1023u) * 8; }
__device__ __forceinline__ int meta_short(uint2 m) { return (int)(m.y >> 20) * 8; }

// asynchronous copy of one T4 to shared memory (cp.async: no registers, all of a thread's copies in
// flight together)
template <class T4>
__device__ __forceinline__ void copy_async(T4 *dst, const T4 *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const char *s = reinterpret_cast<const char *>(src);
#pragma unroll
    for (int k = 0; k < (int)sizeof(T4); k += 16)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + k), "l"(s + k) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// stages candidates k0 .. k0 + kc - 1 (row 0 positions, row r + 1 of src[r]) and the phantom
// behind them; rows of AP_CHUNK + 1. Every thread of the CTA calls it; it ends with a barrier.
template <class T4, int NS>
__device__ __forceinline__ void stage(T4 *rows, const ListArgs &la, const Cands &cs, int k0, int kc,
                                      const T4 *const (&src)[NS], const T4 &phantom) {
    constexpr int NR = AP_CHUNK + 1, PER = AP_CHUNK / 128;
    const T4 *cpos = (const T4 *)la.cand_pos;
    int j[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = threadIdx.x + i * 128;
        if (k < kc) {
            const size_t at = cs.at(k0 + k);
            j[i] = __ldg(la.cand_j + at) & ~AP_CAND_SELF;
            copy_async(rows + k, cpos + at);
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = threadIdx.x + i * 128;
        if (k < kc) {
#pragma unroll
            for (int r = 0; r < NS; ++r) copy_async(rows + (r + 1) * NR + k, src[r] + j[i]);
        }
    }
    if (threadIdx.x == 0) {
        T4 z = phantom;
        rows[kc] = z;
        z.x = z.y = z.z = z.w = 0;
        for (int r = 1; r <= NS; ++r) rows[r * NR + kc] = z;
    }
    copies_done();
    __syncthreads();
}

// The shared loop over a block's chunks: stages each and calls body(list, words, flagged, short
// words) with this thread's pair's list.
template <class T, int PARTS, int NS, class Body>
__device__ __forceinline__ void for_chunks(unsigned char *raw, const ListArgs &la, const Layout<T, PARTS> &ly,
                                           const typename V4<T>::type *const (&src)[NS], Body body) {
    typedef typename V4<T>::type T4;
    const Cands cs(la, ly.I);
    const int t0 = la.tile_off[ly.I], chunks = list_chunks(cs.n), per = list_chunk_size(cs.n);
    const unsigned *list = la.list + list_entry_base(t0, ly.I, la.mult) / 2;
    const uint2 *meta = la.meta + list_meta_base(t0, ly.I, la.mult) * 16 + ly.p;
    for (int c = 0; c < chunks; ++c) {
        const uint2 m = __ldg(meta + (size_t)c * 16);
        if (c) __syncthreads();
        stage(reinterpret_cast<T4 *>(raw), la, cs, c * per, min(per, cs.n - c * per), src, phantom_pos<T>());
        body(list + m.x / 2, meta_words(m), meta_flagged(m), meta_short(m));
    }
}

// Quarter blocks for systems of up to PARTS_BLOCKS blocks (a fixed number, so that the order of the
// sums does not depend on the device): see Layout.
constexpr int PARTS_BLOCKS = 304;
inline bool quarter_blocks(const ap_ctx *ctx) { return ctx->n_blocks <= PARTS_BLOCKS; }

// Dynamic shared memory above 48 KB has to be asked for. The limit is the kernel's on its device, shared by every
// context, so each kernel's is set when a context is made, to the most that any launch can need: set before a launch
// to what that one needs, it could be lowered by another thread's before the launch came.
template <class K>
inline cudaError_t allow_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
