// a1 - Neighbour blocks (paper Sec. 2.3, "Neighbor list").
//
// Atoms are sorted into a cell grid whose numbering follows one dimension contiguously
// (Sec. 2.3.1, box partitioning), then cut into groups of exactly 32 consecutive atoms
// (B_size = warp size). Interacting group pairs are those whose bounding boxes are
// within cutoff + buffer; they form the "adjacency" of Sec. 2.3.1, compacted into a
// list sorted by the first group. Bonded pairs whose scale differs from 1 are not
// stored per atom (Sec. 1.2.1 moves them out of the pair loop); here each group pair
// that holds any gets a 32 x 32-bit mask instead.
//
// GB300 choices (differences from the paper): cells are 1/4 of a 32-atom cube along x
// and the cell order snakes through x and y, so every run of 32 atoms stays compact
// without the paper's iterative refinement; the block-pair test is a brute-force
// bounding-box sweep over block pairs (n_blocks^2 tests, about a ms at 10^6 atoms),
// which needs no bit matrix at all. Block pairs are kept in both orders: the pair lists made
// from them (lists.cu) are per target atom. A rebuild with capacities that still hold allocates
// nothing and reads its results back once.
#include "common.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace {

struct CellGrid {
    int nx, ny, nz;
    double lx, ly, lz;
};

__device__ __forceinline__ double wrap1(double x, double L) {
    double w = x - L * floor(x / L);
    return (w >= L) ? 0.0 : w;
}

// cell of every atom, and the cells' counts
__global__ void k_cell_key(const double *__restrict__ xyz, int n, CellGrid g, int *__restrict__ key,
                           int *__restrict__ count) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double x = wrap1(xyz[3 * i + 0], g.lx), y = wrap1(xyz[3 * i + 1], g.ly), z = wrap1(xyz[3 * i + 2], g.lz);
    // clamp: a non-finite coordinate must not index outside the cell arrays
    int cx = isfinite(x) ? max(0, min(g.nx - 1, (int)(x / g.lx * g.nx))) : 0;
    int cy = isfinite(y) ? max(0, min(g.ny - 1, (int)(y / g.ly * g.ny))) : 0;
    int cz = isfinite(z) ? max(0, min(g.nz - 1, (int)(z / g.lz * g.nz))) : 0;
    // serpentine numbering: y reverses on odd z-planes, x reverses on odd rows
    int cyy = (cz & 1) ? (g.ny - 1 - cy) : cy;
    int row = cz * g.ny + cyy;
    int cxx = (row & 1) ? (g.nx - 1 - cx) : cx;
    key[i] = row * g.nx + cxx;
    atomicAdd(&count[key[i]], 1);
}

// exclusive scan of m ints with one block of 1024 threads (build-time only); with total given,
// the sum also to it and to out[m]
__global__ void k_scan_single(const int *__restrict__ in, int *__restrict__ out, int m, int *__restrict__ total) {
    __shared__ int sums[1024];
    int t = threadIdx.x;
    int chunk = (m + 1023) / 1024;
    int b = t * chunk, e = min(m, b + chunk);
    int s = 0;
    for (int k = b; k < e; ++k) s += in[k];
    sums[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        int v = (t >= off) ? sums[t - off] : 0;
        __syncthreads();
        sums[t] += v;
        __syncthreads();
    }
    int run = sums[t] - s;
    for (int k = b; k < e; ++k) {
        int v = in[k];
        out[k] = run;
        run += v;
    }
    if (t == 1023 && total) *total = out[m] = sums[1023];
}

__global__ void k_scatter(const int *__restrict__ key, int n, const int *__restrict__ start,
                          int *__restrict__ cursor, int *__restrict__ perm) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int k = key[i];
    perm[start[k] + atomicAdd(&cursor[k], 1)] = i;
}

// deterministic order inside each cell: ascending atom index (insertion sort; cells hold ~8)
__global__ void k_sort_cells(const int *__restrict__ start, const int *__restrict__ count, int ncell,
                             int *__restrict__ perm) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    int b = start[c], m = count[c];
    for (int a = 1; a < m; ++a) {
        int v = perm[b + a];
        int k = a - 1;
        while (k >= 0 && perm[b + k] > v) { perm[b + k + 1] = perm[b + k]; --k; }
        perm[b + k + 1] = v;
    }
}

__global__ void k_pad_perm(int *__restrict__ perm, int n, int n_pad) {
    const int s = n + threadIdx.x;
    if (s < n_pad) perm[s] = -1;
}

// One warp per block: its atoms put in an order in which slots 2 k and 2 k + 1 hold near neighbours.
// The pair kernels give a thread two such slots and walk one list for both, so a list is the
// shorter the more of the two atoms' neighbours are the same: in water 175 entries per pair at
// r_c = 7 A against 187 in the order of the cells. Greedy matching: every unmatched atom finds its
// nearest unmatched one, mutual choices are matched, and so on (each round matches at least
// the closest pair; distance ties go to the lower lane).
__global__ void k_pair_order(const double *__restrict__ xyz, int nb, double3 L, int *__restrict__ perm) {
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (b >= nb) return;
    const int a = perm[b * 32 + lane], a0 = perm[b * 32];
    float x = 0.f, y = 0.f, z = 0.f;
    if (a >= 0) {   // image nearest the block's first atom
        const double d[3] = {xyz[3 * a] - xyz[3 * a0], xyz[3 * a + 1] - xyz[3 * a0 + 1], xyz[3 * a + 2] - xyz[3 * a0 + 2]};
        x = (float)(d[0] - L.x * rint(d[0] / L.x));
        y = (float)(d[1] - L.y * rint(d[1] / L.y));
        z = (float)(d[2] - L.z * rint(d[2] / L.z));
    }
    const unsigned real = __ballot_sync(0xffffffffu, a >= 0);
    unsigned open = real, leaders = 0u;
    int partner = -1;
    for (int round = 0; round < 16 && __popc(open) > 1; ++round) {
        float best = 3e38f;
        int nn = -1;
        for (int j = 0; j < 32; ++j) {
            const float dx = x - __shfl_sync(0xffffffffu, x, j), dy = y - __shfl_sync(0xffffffffu, y, j),
                        dz = z - __shfl_sync(0xffffffffu, z, j), d = dx * dx + dy * dy + dz * dz;
            if (((open >> j) & 1u) && j != lane && d < best) {
                best = d;
                nn = j;
            }
        }
        if (!((open >> lane) & 1u)) nn = -1;
        const int back = __shfl_sync(0xffffffffu, nn, nn < 0 ? lane : nn);
        const bool mutual = nn >= 0 && back == lane;
        if (mutual) partner = nn;
        const unsigned done = __ballot_sync(0xffffffffu, mutual);
        if (!done) break;   // only with coordinates that are not numbers
        leaders |= __ballot_sync(0xffffffffu, mutual && lane < nn);
        open &= ~done;
    }
    // pairs by their first lane, then the atoms left over, then the padding
    const unsigned below = (1u << lane) - 1u;
    const int pairs = __popc(leaders);
    int slot;
    if (partner >= 0) {
        const int lead = min(lane, partner);
        slot = 2 * __popc(leaders & ((1u << lead) - 1u)) + (lane > partner);
    } else if (a >= 0) {
        slot = 2 * pairs + __popc(open & below);
    } else {
        slot = 2 * pairs + __popc(open) + __popc(~real & below);
    }
    __syncwarp();
    perm[b * 32 + slot] = a;
}

// one warp per block: bounding box of its atoms (wrapped coordinates); also the inverse order
__global__ void k_block_bbox(const double *__restrict__ xyz, const int *__restrict__ perm, int nb, int *__restrict__ iperm,
                             double lx, double ly, double lz, float4 *__restrict__ center,
                             float4 *__restrict__ half, unsigned *__restrict__ hmax_bits) {
    int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (w >= nb) return;
    int a = perm[w * 32 + lane];
    double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
    if (a >= 0) {
        iperm[a] = w * 32 + lane;
        double p[3] = {wrap1(xyz[3 * a], lx), wrap1(xyz[3 * a + 1], ly), wrap1(xyz[3 * a + 2], lz)};
        for (int d = 0; d < 3; ++d) lo[d] = hi[d] = p[d];
    }
    for (int off = 16; off; off >>= 1)
        for (int d = 0; d < 3; ++d) {
            lo[d] = fmin(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
            hi[d] = fmax(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
        }
    if (lane == 0) {
        center[w] = make_float4((float)(0.5 * (lo[0] + hi[0])), (float)(0.5 * (lo[1] + hi[1])),
                                (float)(0.5 * (lo[2] + hi[2])), 0.f);
        float h[3];
        for (int d = 0; d < 3; ++d) h[d] = (float)(0.5 * (hi[d] - lo[d])) + 1e-4f;
        half[w] = make_float4(h[0], h[1], h[2], 0.f);
        for (int d = 0; d < 3; ++d) atomicMax(&hmax_bits[d], __float_as_uint(h[d]));
    }
}

// centres lie in [0, L), so min(|d|, L - |d|) is the nearest image's distance
__device__ __forceinline__ bool blocks_near(const float4 &ci, const float4 &hi, const float4 &cj, const float4 &hj, const float3 &L,
                                            float r2) {
    const float ax = fabsf(ci.x - cj.x), ay = fabsf(ci.y - cj.y), az = fabsf(ci.z - cj.z);
    const float gx = fmaxf(0.f, fminf(ax, L.x - ax) - hi.x - hj.x);
    const float gy = fmaxf(0.f, fminf(ay, L.y - ay) - hi.y - hj.y);
    const float gz = fmaxf(0.f, fminf(az, L.z - az) - hi.z - hj.z);
    return gx * gx + gy * gy + gz * gz < r2;
}

// One warp per TILE_I blocks I: count (tiles == nullptr) or write their partners J, I among them (as
// many as fit: the caller looks at the total and grows the arrays). Two blocks per warp halve the
// loads of J, and four of those are in flight per lane. (With one block a warp, a division per dimension and the
// tiles' FP64 origins formed here by the few lanes that hit, a build and field took 625 us for 554 at 96,000 atoms
// and 4,064 for 3,605 at 648,000.)
constexpr int TILE_I = 2;
__global__ void k_tiles(const float4 *__restrict__ center, const float4 *__restrict__ half, int nb,
                        float3 L, float r2, int *__restrict__ count, const int *__restrict__ off,
                        TileRec *__restrict__ tiles, int cap) {
    const int I0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * TILE_I;
    const int lane = threadIdx.x & 31;
    if (I0 >= nb) return;
    float4 ci[TILE_I], hi[TILE_I];
    int pos[TILE_I];
#pragma unroll
    for (int i = 0; i < TILE_I; ++i) {
        const int I = min(I0 + i, nb - 1);
        ci[i] = center[I];
        hi[i] = half[I];
        pos[i] = tiles ? off[I] : 0;
    }
    constexpr int U = 4;
    for (int base = 0; base < nb; base += 32 * U) {
        float4 cj[U], hj[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int J = min(base + 32 * u + lane, nb - 1);
            cj[u] = center[J];
            hj[u] = half[J];
        }
#pragma unroll
        for (int i = 0; i < TILE_I; ++i) {
            if (I0 + i >= nb) break;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int J = base + 32 * u + lane;
                const bool hit = blocks_near(ci[i], hi[i], cj[u], hj[u], L, r2) && J < nb;
                const unsigned m = __ballot_sync(0xffffffffu, hit);
                const int k = pos[i] + __popc(m & ((1u << lane) - 1u));
                if (tiles && hit && k < cap) {
                    TileRec r = {};
                    r.J = J;
                    r.excl = I0 + i;   // until k_tile_origins
                    tiles[k] = r;
                }
                pos[i] += __popc(m);
            }
        }
    }
    if (!tiles && lane == 0)
#pragma unroll
        for (int i = 0; i < TILE_I; ++i)
            if (I0 + i < nb) count[I0 + i] = pos[i];
}

// The tiles' origins, one thread each: J's image next to I relative to I's origin, c_J - c_I + L k in
// FP64, split into float hi + lo (the centres are the blocks' position origins). Apart from k_tiles, where
// a few lanes of a warp at a time ran these FP64 instructions.
__global__ void k_tile_origins(const float4 *__restrict__ center, float3 L, double3 Ld, const int *__restrict__ total, int cap,
                               TileRec *__restrict__ tiles) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= min(*total, cap)) return;
    TileRec r = tiles[t];
    const float4 a = center[r.excl], c = center[r.J];
    const double ox = (double)c.x - (double)a.x + Ld.x * rintf((a.x - c.x) / L.x);
    const double oy = (double)c.y - (double)a.y + Ld.y * rintf((a.y - c.y) / L.y);
    const double oz = (double)c.z - (double)a.z + Ld.z * rintf((a.z - c.z) / L.z);
    r.excl = -1;
    r.hx = (float)ox;
    r.hy = (float)oy;
    r.hz = (float)oz;
    r.lx = (float)(ox - r.hx);
    r.ly = (float)(oy - r.hy);
    r.lz = (float)(oz - r.hz);
    tiles[t] = r;
}

__device__ int find_tile(const TileRec *__restrict__ tiles, int b, int e, int J) {
    while (b < e) {
        int m = (b + e) >> 1;
        int v = tiles[m].J;
        if (v == J) return m;
        if (v < J) b = m + 1; else e = m;
    }
    return -1;
}

// what a build reads back: tiles, whether an excluded pair lies outside them, exclusion slots, those
// of diagonal tiles, and the blocks' largest half extents (float bits)
enum { NB_TILES, NB_FAR, NB_SLOTS, NB_DIAG, NB_HMAX };

// Exclusion masks of the tiles, word j-lane of tile (I, J) holding the excluded i-lanes, for both
// orders of every pair. pass 0: flag the tiles (-2, diagonal ones -3); pass 1: set the mask bits.
__global__ void k_excl(const int *__restrict__ off, const int *__restrict__ atoms, int n,
                       const int *__restrict__ iperm, TileRec *__restrict__ tiles, int cap,
                       const int *__restrict__ tile_off, unsigned *__restrict__ masks, int cap_slots, int pass,
                       int *__restrict__ info) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || info[NB_TILES] > cap) return;
    for (int k = off[i]; k < off[i + 1]; ++k) {
        int j = atoms[k];
        if (j == i || j < 0 || j >= n) continue;
        const int s[2] = {iperm[i], iperm[j]};
        for (int d = 0; d < 2; ++d) {
            const int bI = s[d] >> 5, li = s[d] & 31, bJ = s[1 - d] >> 5, lj = s[1 - d] & 31;
            const int t = find_tile(tiles, tile_off[bI], tile_off[bI + 1], bJ);
            if (t < 0) { atomicExch(info + NB_FAR, 1); continue; }
            if (pass == 0) {
                tiles[t].excl = bI == bJ ? -3 : -2;
            } else {
                const int e = tiles[t].excl;
                if (e >= 0 && e < cap_slots) atomicOr(&masks[(size_t)e * 32 + lj], 1u << li);
            }
        }
    }
}

// a slot (in any order) and a cleared mask for every flagged tile
__global__ void k_assign_slots(TileRec *__restrict__ tiles, int cap, unsigned *__restrict__ masks, int cap_slots,
                               int *__restrict__ info) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (info[NB_TILES] > cap || t >= info[NB_TILES] || tiles[t].excl > -2) return;
    const int e = atomicAdd(info + NB_SLOTS, 1);
    if (tiles[t].excl == -3) atomicAdd(info + NB_DIAG, 1);
    tiles[t].excl = e;
    if (e < cap_slots)
        for (int k = 0; k < 32; ++k) masks[(size_t)e * 32 + k] = 0u;
}

// room for `need` elements; `moved` is set when the array is allocated anew
template <class P>
int grow(ap_ctx *ctx, P **ptr, int *cap, long need, size_t elem, bool *moved = nullptr) {
    if (need <= *cap) return AP_OK;
    long c = std::max<long>(need + need / 4 + 64, 1024);
    if (*ptr) AP_CUDA(cudaFree(*ptr));
    *ptr = nullptr;
    *cap = 0;
    if (moved) *moved = true;
    AP_CUDA(cudaMalloc((void **)ptr, (size_t)c * elem));
    *cap = (int)c;
    return AP_OK;
}

}  // namespace

int nb_build(ap_ctx *ctx, const double *d_xyz, const int *d_off, const int *d_atoms, int n_excl) {
    const ap_params &P = ctx->prm;
    cudaStream_t s = ctx->s0;
    const int n = ctx->n, n_pad = ctx->n_pad, nb = ctx->n_blocks;
    double vol = P.box[0] * P.box[1] * P.box[2];
    double rho = n / vol;
    double c = std::cbrt(32.0 / rho);
    CellGrid g;
    g.ny = std::max(1, (int)std::floor(P.box[1] / c));
    g.nz = std::max(1, (int)std::floor(P.box[2] / c));
    g.nx = std::max(1, (int)std::floor(4.0 * P.box[0] / c));
    g.lx = P.box[0]; g.ly = P.box[1]; g.lz = P.box[2];
    long ncell = (long)g.nx * g.ny * g.nz;
    if (ncell > (1L << 26)) return ap_fail(ctx, AP_ERR_ARG, "cell grid too large");

    int r;
    if ((r = grow(ctx, &ctx->cell_count, &ctx->cap_cells, 3 * ncell + 3, sizeof(int)))) return r;
    if ((r = grow(ctx, &ctx->tmp_int, &ctx->cap_tmp, std::max<long>(n, nb), sizeof(int)))) return r;
    // the order, the tiles and the lists change from here on: none are valid until all are done
    ctx->lists_valid = 0;
    ctx->config_valid = 0;
    int *count = ctx->cell_count, *cursor = count + ncell, *start = cursor + ncell;
    int *key = ctx->tmp_int, *info = ctx->nb_info;
    const int T = 256;

    AP_CUDA(cudaMemsetAsync(info, 0, sizeof(int) * 8, s));
    AP_CUDA(cudaMemsetAsync(count, 0, sizeof(int) * 2 * ncell, s));   // and the cursors
    k_cell_key<<<ap_grid_for(n, T), T, 0, s>>>(d_xyz, n, g, key, count);
    k_scan_single<<<1, 1024, 0, s>>>(count, start, (int)ncell, nullptr);
    k_scatter<<<ap_grid_for(n, T), T, 0, s>>>(key, n, start, cursor, ctx->perm);
    k_sort_cells<<<ap_grid_for(ncell, T), T, 0, s>>>(start, count, (int)ncell, ctx->perm);
    const double3 Ld = make_double3(P.box[0], P.box[1], P.box[2]);
    if (n_pad > n) k_pad_perm<<<1, 32, 0, s>>>(ctx->perm, n, n_pad);
    k_pair_order<<<ap_grid_for((long)nb * 32, T), T, 0, s>>>(d_xyz, nb, Ld, ctx->perm);
    k_block_bbox<<<ap_grid_for((long)nb * 32, T), T, 0, s>>>(d_xyz, ctx->perm, nb, ctx->iperm, P.box[0], P.box[1], P.box[2],
                                                           ctx->bcenter, ctx->bhalf, (unsigned *)(info + NB_HMAX));
    AP_CUDA(cudaGetLastError());
    const float3 L = make_float3((float)P.box[0], (float)P.box[1], (float)P.box[2]);
    const float rl = (float)(P.cutoff + P.buffer);
    int *bcount = key;                 // reuse: key no longer needed
    const int warps = ap_grid_for((long)(nb + TILE_I - 1) / TILE_I * 32, T);
    k_tiles<<<warps, T, 0, s>>>(ctx->bcenter, ctx->bhalf, nb, L, rl * rl, bcount, nullptr, nullptr, 0);
    k_scan_single<<<1, 1024, 0, s>>>(bcount, ctx->tile_off, nb, info + NB_TILES);
    AP_CUDA(cudaGetLastError());

    // Fill the tiles and their exclusion masks with the capacities of the last build, and read the
    // counts back; where one did not hold, grow it and fill again (the first build of a context
    // goes round twice or three times).
    bool moved = false;
    int h[8];
    for (int round = 0;; ++round) {
        if (ctx->cap_tiles > 0) {
            k_tiles<<<warps, T, 0, s>>>(ctx->bcenter, ctx->bhalf, nb, L, rl * rl, nullptr, ctx->tile_off, ctx->tiles,
                                        ctx->cap_tiles);
            k_tile_origins<<<ap_grid_for(ctx->cap_tiles, T), T, 0, s>>>(ctx->bcenter, L, Ld, info + NB_TILES, ctx->cap_tiles,
                                                                       ctx->tiles);
            if (n_excl > 0) {
                const int slots = ctx->cap_excl / 32;
                AP_CUDA(cudaMemsetAsync(info + NB_FAR, 0, sizeof(int) * 3, s));
                k_excl<<<ap_grid_for(n, T), T, 0, s>>>(d_off, d_atoms, n, ctx->iperm, ctx->tiles, ctx->cap_tiles,
                                                      ctx->tile_off, ctx->excl_mask, slots, 0, info);
                k_assign_slots<<<ap_grid_for(ctx->cap_tiles, T), T, 0, s>>>(ctx->tiles, ctx->cap_tiles, ctx->excl_mask,
                                                                           slots, info);
                k_excl<<<ap_grid_for(n, T), T, 0, s>>>(d_off, d_atoms, n, ctx->iperm, ctx->tiles, ctx->cap_tiles,
                                                      ctx->tile_off, ctx->excl_mask, slots, 1, info);
            }
            AP_CUDA(cudaGetLastError());
        }
        AP_CUDA(cudaMemcpyAsync(h, info, sizeof(h), cudaMemcpyDeviceToHost, s));
        AP_CUDA(cudaStreamSynchronize(s));
        if (h[NB_TILES] <= 0) return ap_fail(ctx, AP_ERR_ARG, "no interacting blocks");
        if (h[NB_TILES] > ctx->cap_tiles) {
            if ((r = grow(ctx, &ctx->tiles, &ctx->cap_tiles, h[NB_TILES], sizeof(TileRec)))) return r;
            continue;
        }
        if (h[NB_FAR]) return ap_fail(ctx, AP_ERR_ARG, "an excluded pair is farther apart than cutoff+buffer");
        if ((long)h[NB_SLOTS] * 32 > ctx->cap_excl) {
            if ((r = grow(ctx, &ctx->excl_mask, &ctx->cap_excl, (long)h[NB_SLOTS] * 32, sizeof(unsigned), &moved))) return r;
            continue;
        }
        break;
    }
    ctx->n_tiles = h[NB_TILES];
    ctx->n_excl_tiles = (h[NB_SLOTS] + h[NB_DIAG]) / 2;   // kept in both orders, diagonal ones once

    // one image per tile is exact along every dimension with L > 2 r_c + 4 (h_max + buffer/2);
    // along a shorter one an atom can be in range of a block in two
    int dims = 0, mult = 1;
    for (int d = 0; d < 3; ++d) {
        float hm;
        memcpy(&hm, &h[NB_HMAX + d], sizeof(float));
        if (!(P.box[d] > 2.0 * P.cutoff + 4.0 * (hm + 0.5 * P.buffer))) {
            dims |= 1 << d;
            mult *= 2;
        }
    }
    if (mult != ctx->list_mult) moved = true;
    ctx->image_dims = dims;
    ctx->list_mult = mult;
    const long held = ctx->cap_lists;
    if ((r = lists_alloc(ctx))) return r;
    if (ctx->cap_lists != held) moved = true;
    ctx->lists_valid = 1;
    if (moved) {                   // captured solve loops hold the old pointers
        ctx->graph_ok = 0;
        ctx->graph_tried = 0;
        if (ctx->solve_exec) cudaGraphExecDestroy(ctx->solve_exec);
        ctx->solve_exec = nullptr;
        diis_forget_graph(ctx);
        dp_forget_graph(ctx);
    }
    return AP_OK;
}
