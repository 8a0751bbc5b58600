// Pair lists of a configuration (paper Sec. 2.3.2, "List filtering": an atom belongs to a group's
// neighbourhood when it is within range of some atom of the group).
//
// The block-pair lists (neighbour.cu) are built with cutoff + buffer and reused for many steps;
// once the positions of a step are known they stay fixed for the field, every PCG matrix-vector
// product and the forces. So every configuration gets, for each block I of 32 atoms,
//   - its candidates: the atoms of the partner blocks (I itself among them) within r_c of some
//     atom of I, with their positions beside I and their exclusion bits;
//   - for each of its 16 target pairs the list of candidates within r_c of either target, in the
//     form pair_walk.cuh describes.
// Lists are kept for both atoms of a pair: the kernels that use them evaluate each pair once per
// side, as they did on 32 x 32 pair masks, but a side's sum stays with its target's threads, so
// no kernel adds into another's targets. (On masks, half of a kernel's time went into staging and
// flushing items of 32 x 32 slots with 124 pairs in them.)
//
// One CTA per block. Each of its four warps takes every fourth of the block's tiles (a contiguous quarter
// each left the CTA waiting for the warps with the nearest blocks, a sixth of its time):
// atoms that pass the bounding-box test queue up, and every 32 of them are tested against the
// block's atoms, a lane holding one candidate and reading the targets from shared memory (in FP32
// two at a time, packed, the sign of r^2 - r_c^2 shifted into the candidate's word); the result is
// a 32-bit word per candidate, bit i-lane. Transposed 32 x 32 bits at a time these become words
// per target pair, whose set bits eight threads per pair count and write out as entries, through shared memory so that the list goes out in whole lines.
// Measured on GB300 (ncu, warm) against filtered chunks, pair masks and work-item scans (k_filter,
// k_pairmask and five small kernels): 96,000 atoms 76 + 42 + 17 -> 137 us in one launch, 6,000 atoms
// (short box) 342 + 20 + 15 -> 55 us; the kernels that walk the lists gain 40 % and more. That took longer in
// permanent_field alone above 200,000 atoms, where nothing hides it: 693 -> 724 us at 255,552, 1,613 -> 1,752 at 648,000,
// 2,700 -> 2,936 at 1,065,000. Interleaved tiles, entries written without a search for bits, a look at whole blocks
// first, and two tiles in flight instead of four (64 registers, 8 CTAs an SM instead of 5: it is bound by issue and
// latency together, 55 % of the slots at 5, 68 % at 8) made those 605, 1,443 and 2,431: 91 us a launch at 96,000
// atoms and 3 for the boxes.
// Candidate and entry order follow the tile order, so the lists are the same in every run.
#include "common.cuh"
#include "pair_walk.cuh"

namespace {

constexpr int LT = 128;              // threads per block of atoms
constexpr int STAGE = 4096;          // entries staged in shared memory before they go out

constexpr int GROUPS = AP_CHUNK / 32;

// the block's targets as the test reads them
template <class T> struct TargetSmem;
template <> struct TargetSmem<float> {
    float4 xy[16];
    float2 z[16];
    __device__ __forceinline__ void put(int i, float x, float y, float zz) {
        float *p = reinterpret_cast<float *>(&xy[i >> 1]);
        p[i & 1] = x;
        p[2 + (i & 1)] = y;
        reinterpret_cast<float *>(&z[i >> 1])[i & 1] = zz;
    }
    // bits of the targets within sqrt(rc2) and sqrt(rs2) of the candidate
    __device__ __forceinline__ void test(const float4 &c, float rc2, float rs2, unsigned &in, unsigned &sh) const {
        const float2 cx = splat2(c.x), cy = splat2(c.y), cz = splat2(c.z), n = splat2(-rc2), ds = splat2(rc2 - rs2);
        in = sh = 0u;
#pragma unroll
        for (int p = 15; p >= 0; --p) {
            const float4 a = xy[p];
            const float2 dx = sub2(make_float2(a.x, a.y), cx), dy = sub2(make_float2(a.z, a.w), cy), dz = sub2(z[p], cz);
            const float2 d = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, n))), e = add2(d, ds);
            in = __funnelshift_l(__float_as_uint(d.y), in, 1);
            in = __funnelshift_l(__float_as_uint(d.x), in, 1);
            sh = __funnelshift_l(__float_as_uint(e.y), sh, 1);
            sh = __funnelshift_l(__float_as_uint(e.x), sh, 1);
        }
    }
    };
template <> struct TargetSmem<double> {
    double x[32], y[32], z[32];
    __device__ __forceinline__ void put(int i, double a, double b, double c) {
        x[i] = a;
        y[i] = b;
        z[i] = c;
    }
    __device__ __forceinline__ void test(const dvec4 &c, double rc2, double rs2, unsigned &in, unsigned &sh) const {
        in = sh = 0u;
#pragma unroll 4
        for (int i = 31; i >= 0; --i) {
            const double dx = x[i] - c.x, dy = y[i] - c.y, dz = z[i] - c.z, r2 = dx * dx + dy * dy + dz * dz;
            in = (in << 1) | (r2 < rc2 ? 1u : 0u);
            sh = (sh << 1) | (r2 < rs2 ? 1u : 0u);
        }
    }
    };

template <class T>
struct ListSmem {
    TargetSmem<T> tg;
    union {
        struct {
            typename V4<T>::type pos[4][64];        // each warp's queue of box-passing candidates
            int j[4][64];
            unsigned ex[4][64];
        } q;
        unsigned short stage[STAGE];
    };
    unsigned word[3][16][GROUPS + 1];   // per pair and 32 candidates: entries with flags, short, others
    unsigned ex[AP_CHUNK], own[AP_CHUNK];   // a candidate's excluded targets, and itself if it is one
    int count[4];
    int total[16];
    int2 column[16][8];                 // per pair and column of its list: first hole's number, entries
};

// 32 (or the last m) queued candidates against the block's atoms: the ones in range of any go to
// the candidate arrays at `at`, of which `room` are left, and their masks to `mask`; returns how many
template <class T>
__device__ __forceinline__ int test_queue(const ListSmem<T> &S, int w, int lane, int m, T rc2, T rs2, size_t at, int room,
                                          typename V4<T>::type *__restrict__ cand_pos, int *__restrict__ cand_j,
                                          uint4 *mask) {
    const typename V4<T>::type c = S.q.pos[w][lane];
    const int j = S.q.j[w][lane];
    unsigned in, sh;
    S.tg.test(c, rc2, rs2, in, sh);
    if (j & AP_CAND_SELF) in &= ~(1u << (j & 31));
    const bool keep = lane < m && in != 0u;
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    // (rounding at 2 r_c = L could make a third image; the room is for two)
    if (keep && __popc(b & ((1u << lane) - 1u)) < room) {
        const int k = __popc(b & ((1u << lane) - 1u));
        cand_pos[at + k] = c;
        cand_j[at + k] = j;
        // in-range, short-range and exclusion bits (bit i-lane), and j
        mask[k] = make_uint4(in, sh & in, S.q.ex[w][lane] & in, (unsigned)j);
    }
    return min(__popc(b), room);
}

// transpose of a 32 x 32 bit matrix held one row per lane (bit c of lane r -> bit r of lane
// c): five butterfly stages, each swapping the off-diagonal blocks of lanes l and l ^ j
__device__ __forceinline__ unsigned warp_transpose32(unsigned x, int lane) {
    const unsigned lo_masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int st = 0, j = 16; st < 5; ++st, j >>= 1) {
        const unsigned y = __shfl_xor_sync(0xffffffffu, x, j);
        const unsigned lo = lo_masks[st];
        x = (lane & j) ? ((x & ~lo) | ((y >> j) & lo)) : ((x & lo) | ((y & lo) << j));
    }
    return x;
}

// The blocks' boxes at their atoms' present places: centre (relative to the block's origin) and half extents, a
// little more than the atoms reach. One warp a block.
template <class T>
__global__ void k_boxes(const typename V4<T>::type *__restrict__ posw, int n_atoms, int n_blocks,
                        typename V4<T>::type *__restrict__ boxes) {
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (b >= n_blocks) return;
    const typename V4<T>::type me = posw[b * 32 + lane];
    const bool real = b * 32 + lane < n_atoms;
    const T x[3] = {me.x, me.y, me.z};
    T c[3], h[3];
    for (int d = 0; d < 3; ++d) {
        T lo = real ? x[d] : T(1e30), hi = real ? x[d] : T(-1e30);
        for (int off = 16; off; off >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        }
        c[d] = T(0.5) * (lo + hi);
        h[d] = T(0.5) * (hi - lo) + T(1e-6) * max(abs(lo), abs(hi));
    }
    if (lane == 0) {
        typename V4<T>::type v;
        v.x = c[0]; v.y = c[1]; v.z = c[2]; v.w = T(0);
        boxes[2 * b] = v;
        v.x = h[0]; v.y = h[1]; v.z = h[2];
        boxes[2 * b + 1] = v;
    }
}

// dims: bit d set where the box is so short along d that an atom may be in range of one block in
// two images (IMAGES: any); a tile's atoms are then taken in the image nearest the block and its
// neighbours along those dimensions
template <class T, bool IMAGES>
__global__ void __launch_bounds__(LT, sizeof(T) == 4 && !IMAGES ? 8 : 5) k_pair_lists(
    const TileRec *__restrict__ tiles, const int *__restrict__ tile_off, const unsigned *__restrict__ excl_mask,
    const typename V4<T>::type *__restrict__ posw, const typename V4<T>::type *__restrict__ boxes, int n_atoms, T rc2, T rs2, T Lx, T Ly, T Lz, int dims, int mult,
    int4 *__restrict__ ncand, typename V4<T>::type *__restrict__ cand_pos, int *__restrict__ cand_j,
    uint2 *__restrict__ meta, unsigned short *list) {
    typedef typename V4<T>::type T4;
    extern __shared__ __align__(16) unsigned char raw[];
    ListSmem<T> &S = *reinterpret_cast<ListSmem<T> *>(raw);
    const int I = blockIdx.x, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const T4 me = posw[I * 32 + lane];   // padding slots lie out of everybody's range
    const bool vi = I * 32 + lane < n_atoms;
    if (w == 0) S.tg.put(lane, me.x, me.y, me.z);
    // the block's box: centre and half extents
    T ctr[3] = {me.x, me.y, me.z}, half[3];
    for (int d = 0; d < 3; ++d) {
        T lo = vi ? ctr[d] : T(1e30), hi = vi ? ctr[d] : T(-1e30);
        for (int off = 16; off; off >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, off));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        }
        ctr[d] = T(0.5) * (lo + hi);
        half[d] = T(0.5) * (hi - lo) * T(1.0 + 1e-6);   // not less than the targets reach
    }
    const int t0 = tile_off[I], nt = tile_off[I + 1] - t0, te = t0 + nt;
    __syncthreads();

    const size_t seg = ((size_t)t0 + segment_tile(nt, w)) * 32 * mult;
    list += list_entry_base(t0, I, mult);
    uint4 *const masks = reinterpret_cast<uint4 *>(list + list_mask_base(nt, mult)), *const own_masks = masks + segment_tile(nt, w) * 32 * mult;
    const int room = (segment_tile(nt, w + 1) - segment_tile(nt, w)) * 32 * mult;
    int queued = 0, kept = 0;
    auto push = [&](T x, T y, T z, T wt, int j, unsigned ex, bool ok) {
        const T gx = max(T(0), abs(x - ctr[0]) - half[0]);
        const T gy = max(T(0), abs(y - ctr[1]) - half[1]);
        const T gz = max(T(0), abs(z - ctr[2]) - half[2]);
        const bool sel = ok && gx * gx + gy * gy + gz * gz < rc2;
        const unsigned b = __ballot_sync(0xffffffffu, sel);
        if (!b) return;   // a third of the tiles: lists are kept for cutoff + buffer
        if (sel) {
            const int k = queued + __popc(b & ((1u << lane) - 1u));
            T4 v;
            v.x = x; v.y = y; v.z = z; v.w = wt;
            S.q.pos[w][k] = v;
            S.q.j[w][k] = j;
            S.q.ex[w][k] = ex;
        }
        queued += __popc(b);
        __syncwarp();
        if (queued >= 32) {
            kept += test_queue<T>(S, w, lane, 32, rc2, rs2, seg + kept, room - kept, cand_pos, cand_j, own_masks + kept);
            queued -= 32;
            __syncwarp();
            if (lane < queued) {   // the rest moves to the front (read and written by the same lane)
                S.q.pos[w][lane] = S.q.pos[w][32 + lane];
                S.q.j[w][lane] = S.q.j[w][32 + lane];
                S.q.ex[w][lane] = S.q.ex[w][32 + lane];
            }
            __syncwarp();
        }
    };
    // With the boxes at hand a lane looks at one of the warp's tiles each, and those whose blocks are out of range
    // as a whole (a third: the list of tiles is made for cutoff + buffer) go no further.
    for (int base = t0 + w; base < te; base += 4 * 32) {
        const int look = base + 4 * lane;
        bool near_block = look < te;
        if (!IMAGES && boxes && near_block) {
            const TileRec t = tiles[look];
            const T4 bc = boxes[2 * t.J], bh = boxes[2 * t.J + 1];
            const T gx = max(T(0), abs((bc.x + (T)t.lx) + (T)t.hx - ctr[0]) - half[0] - bh.x);
            const T gy = max(T(0), abs((bc.y + (T)t.ly) + (T)t.hy - ctr[1]) - half[1] - bh.y);
            const T gz = max(T(0), abs((bc.z + (T)t.lz) + (T)t.hz - ctr[2]) - half[2] - bh.z);
            near_block = gx * gx + gy * gy + gz * gz < rc2;
        }
        unsigned todo = __ballot_sync(0xffffffffu, near_block);
        // two tiles' loads go out together (four would take the registers of three CTAs an SM)
        constexpr int U = 2;
        while (todo) {
            TileRec rec[U];
            int tr[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                tr[u] = todo ? base + 4 * (__ffs(todo) - 1) : te;
                todo &= todo - 1u;
            }
            T4 qv[U];
            unsigned ev[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (tr[u] < te) rec[u] = tiles[tr[u]];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (tr[u] < te) {
                    qv[u] = posw[rec[u].J * 32 + lane];
                    ev[u] = rec[u].excl >= 0 ? excl_mask[(size_t)rec[u].excl * 32 + lane] : 0u;
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (tr[u] >= te) break;   // uniform over the warp
                const TileRec &t = rec[u];
                // positions are relative to their block's origin: moved to block I's origin with the
                // tile's offset, a float pair (hi + lo), so that the result (a few A) has full FP32
                // precision at any box size
                const T x = (qv[u].x + (T)t.lx) + (T)t.hx, y = (qv[u].y + (T)t.ly) + (T)t.hy, z = (qv[u].z + (T)t.lz) + (T)t.hz;
                const int slot = t.J * 32 + lane;
                if constexpr (!IMAGES) {
                    push(x, y, z, qv[u].w, t.J == I ? slot | AP_CAND_SELF : slot, ev[u], true);
                } else {
                    // along a short dimension: the image nearest the box's centre (k0), and the next one on
                    // the other side, each only if it lies within r_c of the box along that dimension
                    const T L[3] = {Lx, Ly, Lz}, rc = sqrt(rc2);
                    T c[3] = {x, y, z}, alt[3];
                    int k0[3] = {0, 0, 0}, k1[3] = {0, 0, 0};
                    bool near[3] = {true, true, true}, far[3] = {false, false, false};
                    const bool real = slot < n_atoms;
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        alt[d] = c[d];
                        if (((dims >> d) & 1) && real) {
                            const T k = rint((c[d] - ctr[d]) / L[d]), sgn = c[d] - L[d] * k > ctr[d] ? T(1) : T(-1);
                            k0[d] = (int)k;
                            k1[d] = (int)(k + sgn);
                            c[d] = alt[d] - L[d] * k;
                            alt[d] -= L[d] * (k + sgn);
                            near[d] = abs(c[d] - ctr[d]) - half[d] < rc;
                            far[d] = abs(alt[d] - ctr[d]) - half[d] < rc;
                        }
                    }
                    for (int im = 0; im < 8; ++im) {
                        if (im & ~dims) continue;   // uniform over the launch
                        const bool i0 = im & 1, i1 = im & 2, i2 = im & 4;
                        const bool ok = (i0 ? far[0] : near[0]) && (i1 ? far[1] : near[1]) && (i2 ? far[2] : near[2]);
                        if (!__any_sync(0xffffffffu, ok)) continue;
                        const bool own = t.J == I && (i0 ? k1[0] : k0[0]) == 0 && (i1 ? k1[1] : k0[1]) == 0 && (i2 ? k1[2] : k0[2]) == 0;
                        push(i0 ? alt[0] : c[0], i1 ? alt[1] : c[1], i2 ? alt[2] : c[2], qv[u].w,
                             own ? slot | AP_CAND_SELF : slot, ev[u], ok);
                    }
                }
            }
        }
    }
    if (queued) kept += test_queue<T>(S, w, lane, queued, rc2, rs2, seg + kept, room - kept, cand_pos, cand_j, own_masks + kept);
    if (lane == 0) S.count[w] = kept;
    __syncthreads();
    if (tid == 0) ncand[I] = make_int4(S.count[0], S.count[1], S.count[2], S.count[3]);

    // ---- the lists, chunk by chunk
    const int e1 = S.count[0], e2 = e1 + S.count[1], e3 = e2 + S.count[2], n = e3 + S.count[3];
    auto seg_start = [&](int q) { return segment_tile(nt, q) * 32 * mult; };
    const int b1 = seg_start(1) - e1, b2 = seg_start(2) - e2, b3 = seg_start(3) - e3;
    const int chunks = list_chunks(n), per = list_chunk_size(n);
    const int p = tid >> 3, s = tid & 7;
    const size_t metas = list_meta_base(t0, I, mult) * 16;
    int done = 0;   // entries of the earlier chunks
    for (int c = 0; c < chunks; ++c) {
        const int k0 = c * per, kc = min(per, n - k0);
        const int groups = (kc + 31) >> 5;
        for (int g = w; g < groups; g += 4) {
            const int k = g * 32 + lane, kk = k0 + k;
            uint4 m = make_uint4(0u, 0u, 0u, 0u);
            if (k < kc) m = masks[(kk < e1 ? 0 : kk < e2 ? b1 : kk < e3 ? b2 : b3) + kk];
            unsigned in = 0u, sh = 0u, ex = 0u, own = 0u;
            if (k < kc) {
                in = m.x;
                sh = m.y;
                ex = m.z;
                own = m.w & AP_CAND_SELF ? 1u << (m.w & 31) : 0u;
                S.ex[k] = ex;
                S.own[k] = own;
            }
            unsigned ti = warp_transpose32(in, lane), ts = 0u, tf = 0u;
            ti |= __shfl_xor_sync(0xffffffffu, ti, 1);
            if (__any_sync(0xffffffffu, (ex | own) != 0u)) {
                tf = warp_transpose32(ex | own, lane);
                tf = (tf | __shfl_xor_sync(0xffffffffu, tf, 1)) & ti;
            }
            if (__any_sync(0xffffffffu, sh != 0u)) {
                ts = warp_transpose32(sh, lane);
                ts = (ts | __shfl_xor_sync(0xffffffffu, ts, 1)) & ~tf;
            }
            if (!(lane & 1)) {
                S.word[0][lane >> 1][g] = tf;
                S.word[1][lane >> 1][g] = ts;
                S.word[2][lane >> 1][g] = ti & ~tf & ~ts;
            }
        }
        __syncthreads();
        // Eight threads per pair. Thread s has the candidates in places k with k mod 8 = s, and they go
        // to column s of the list: the eight threads that walk a row of eight entries together then
        // read eight different 16-byte banks of the staged candidates (entries in plain order
        // collide, 2.6 deep on average, and shared memory was the walks' first bound). In a column
        // come the flagged entries, then the short-range ones, then the rest; what a column has
        // beyond the rows of the list fills the holes of the shorter ones, phantoms the last.
        const unsigned cls = 0x01010101u << s;
        int c0 = 0, c1 = 0, c2 = 0;
        unsigned used[2] = {0u, 0u};   // the groups with any flagged and any short-range entry
        for (int g = 0; g < groups; ++g) {
            const unsigned a = S.word[0][p][g] & cls, b = S.word[1][p][g] & cls, d = S.word[2][p][g] & cls;
            c0 += __popc(a);
            c1 += __popc(b);
            c2 += __popc(d);
            if (a) used[0] |= 1u << g;
            if (b) used[1] |= 1u << g;
        }
        const int mine = c0 + c1 + c2;
        int np = mine;
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) np += __shfl_xor_sync(0xffffffffu, np, off);
        const int rounds = (np + 15) >> 4, rows = 2 * rounds;
        const int over = max(mine - rows, 0), hole = max(rows - mine, 0);
        int po = over, ph = hole, r0 = min(c0, rows), r1 = min(c0 + c1, rows);
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) {   // inclusive prefixes over the columns, and maxima
            const int a = __shfl_up_sync(0xffffffffu, po, off, 8), b = __shfl_up_sync(0xffffffffu, ph, off, 8);
            if (s >= off) {
                po += a;
                ph += b;
            }
            r0 = max(r0, __shfl_xor_sync(0xffffffffu, r0, off));
            r1 = max(r1, __shfl_xor_sync(0xffffffffu, r1, off));
        }
        const int all_over = __shfl_sync(0xffffffffu, po, 7, 8);
        po -= over;
        ph -= hole;
        S.column[p][s] = make_int2(ph, mine);
        if (s == 0) S.total[p] = rounds * 16;
        __syncthreads();
        int off = 0, all = 0;
        for (int q = 0; q < 16; ++q) {
            if (q < p) off += S.total[q];
            all += S.total[q];
        }
        const bool staged = all <= STAGE;
        auto flags = [&](int k) { return ((S.ex[k] >> (2 * p)) & 3u) | (((S.own[k] >> (2 * p)) & 3u) << 2); };
        auto emit = [&](unsigned short *out) {
            auto put = [&](int row, int col, unsigned e) { out[(((row >> 1) * 8 + col) << 1) | (row & 1)] = (unsigned short)e; };
            // No bits are searched for: the warp goes through the groups that have any of a kind, every thread
            // looking at its four places in turn.
            int at = 0;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                while (used[q]) {
                    const int g = __ffs(used[q]) - 1;
                    used[q] &= used[q] - 1u;
                    unsigned m = S.word[q][p][g] & cls;
                    while (m) {
                        const int k = g * 32 + __ffs(m) - 1;
                        m &= m - 1u;
                        if (at < rows) put(at, s, (unsigned)k << 4 | (q == 0 ? flags(k) : 0u));
                        ++at;
                    }
                }
            }
            for (int g = 0; g < groups; ++g) {
                const unsigned m = S.word[2][p][g] >> s;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const bool on = (m >> (8 * b)) & 1u;
                    if (on && at < rows) put(at, s, (unsigned)(g * 32 + s + 8 * b) << 4);
                    at += on;
                }
            }
            // what the column has beyond the rows, from the end: hole number h is in the last column whose holes
            // start at or before it
            for (int q = 2, left = over; left; --q)
                for (int g = groups - 1; left && g >= 0; --g) {
                    unsigned m = S.word[q][p][g] & cls;
                    for (; left && m; --left) {
                        const int bit = 31 - __clz(m), k = g * 32 + bit, h = po + left - 1;
                        m ^= 1u << bit;
                        int col = 7;
                        while (S.column[p][col].x > h || S.column[p][col].y >= rows) --col;
                        put(S.column[p][col].y + h - S.column[p][col].x, col, (unsigned)k << 4 | (q == 0 ? flags(k) : 0u));
                    }
                }
            for (int k = 0; k < hole; ++k)
                if (ph + k >= all_over) put(mine + k, s, (unsigned)kc << 4);   // the phantom
        };
        emit(staged ? S.stage + off : list + done + off);
        if (s == 0)   // where it lies; its rounds of 16 entries, those with flagged and with short-range ones
            meta[metas + (size_t)c * 16 + p] = make_uint2((unsigned)(done + off), (unsigned)rounds |
                                                          ((unsigned)((r0 + 1) >> 1) << 10) | ((unsigned)((r1 + 1) >> 1) << 20));
        __syncthreads();
        if (staged) {
            const uint4 *src = reinterpret_cast<const uint4 *>(S.stage);
            uint4 *dst = reinterpret_cast<uint4 *>(list + done);
            for (int k = tid; k < all / 8; k += LT) dst[k] = src[k];
        }
        done += all;
        __syncthreads();
    }
}

// Blocks per SM from which the tiles are first tested as a whole, by the blocks' present boxes: as many CTAs as
// are resident (field, without -> with: 102.2 -> 104.8 us at 750 blocks, 165.0 -> 163.5 at 1,465, 253.4 -> 252.4 at 3,000,
// 619 -> 602.6 at 7,986; the boxes are a launch of their own, which a system of one wave waits for).
constexpr int BOXES_MIN = 8;
template <class T>
int lists_t(ap_ctx *ctx, cudaStream_t s) {
    typedef typename V4<T>::type T4;
    const ap_params &P = ctx->prm;
    // a 1e-5 margin over r_c^2: the walks decide each pair, rounding here drops none
    const T rc2 = (T)(P.cutoff * P.cutoff * (1.0 + 1e-5)), rs2 = (T)(AP_SHORT_RANGE * AP_SHORT_RANGE * (1.0 + 1e-5));
    auto kern = ctx->image_dims ? k_pair_lists<T, true> : k_pair_lists<T, false>;
    const T4 *boxes = nullptr;
    if (ctx->n_blocks >= BOXES_MIN * ctx->sm_count && !ctx->image_dims) {
        boxes = (const T4 *)ctx->boxes;
        k_boxes<T><<<ap_grid_for(32L * ctx->n_blocks, 128), 128, 0, s>>>((const T4 *)ctx->posw, ctx->n, ctx->n_blocks, (T4 *)ctx->boxes);
    }
    kern<<<ctx->n_blocks, LT, sizeof(ListSmem<T>), s>>>(ctx->tiles, ctx->tile_off, ctx->excl_mask, (const T4 *)ctx->posw, boxes,
                                                        ctx->n, rc2, rs2, (T)P.box[0], (T)P.box[1], (T)P.box[2],
                                                        ctx->image_dims, ctx->list_mult, ctx->ncand, (T4 *)ctx->cand_pos,
                                                        ctx->cand_j, ctx->list_meta,
                                                        (unsigned short *)ctx->list);
    AP_CUDA(cudaGetLastError());
    return AP_OK;
}

template <class T>
int init_t(ap_ctx *ctx) {
    AP_CUDA(allow_smem(k_pair_lists<T, true>, sizeof(ListSmem<T>)));
    AP_CUDA(allow_smem(k_pair_lists<T, false>, sizeof(ListSmem<T>)));
    return AP_OK;
}

}  // namespace

int lists_init(ap_ctx *ctx) { return ctx->prec == AP_FP64 ? init_t<double>(ctx) : init_t<float>(ctx); }

int lists_launch(ap_ctx *ctx, cudaStream_t s) {
    return ctx->prec == AP_FP64 ? lists_t<double>(ctx, s) : lists_t<float>(ctx, s);
}

// (re)allocate the candidate and list arrays after a list build. The capacities hold whatever the
// positions do: every atom of every tile a candidate, and every candidate in every target pair's
// list (times the images an atom can have beside one block in a short box), an eighth more for the next
// builds. In FP32 a tile takes 1,702 bytes: 0.52 GB at 96,000 atoms of water with r_c = 7 A and a buffer of 2 A, 5.7 GB at 1,065,000.
int lists_alloc(ap_ctx *ctx) {
    const long need = (long)ctx->n_tiles * ctx->list_mult;
    if (need <= ctx->cap_lists) return AP_OK;
    void **ptrs[] = {(void **)&ctx->cand_j, &ctx->cand_pos, (void **)&ctx->list,
                     (void **)&ctx->list_meta};
    for (void **p : ptrs) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
    ctx->cap_lists = 0;
    const size_t cap = (size_t)(need + need / 8 + 64), es = ctx->prec == AP_FP64 ? 8 : 4;
    AP_CUDA(cudaMalloc((void **)&ctx->cand_j, sizeof(int) * 32 * cap));
    AP_CUDA(cudaMalloc(&ctx->cand_pos, 4 * es * 32 * cap));
    AP_CUDA(cudaMalloc((void **)&ctx->list, 2 * (AP_LIST_PER_TILE * cap + AP_LIST_PER_BLOCK * (size_t)ctx->n_blocks)));
    AP_CUDA(cudaMalloc((void **)&ctx->list_meta, sizeof(uint2) * 16 * (cap / (AP_CHUNK / 32) + ctx->n_blocks + 1)));
    if (!ctx->ncand) AP_CUDA(cudaMalloc((void **)&ctx->ncand, sizeof(int4) * ctx->n_blocks));
    ctx->cap_lists = (long)cap;
    return AP_OK;
}
