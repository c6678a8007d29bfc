// amr.cuh -- the AMR refinement rule of 3D EBIT (arxiv 2509.26361, Sec. 2.5)
// and a narrow-band brick store of the state built on it.
//
// Sec. 2.5: with one marker per edge, cells of two refinement levels must
// never share the interface, so every cell within the 3x3x3 block around an
// interfacial cell is refined to the finest level.  A cell is interfacial when
// its eight corner colours differ (an edge carries a marker exactly when its
// end colours differ).  The brick store keeps the state of the 8^3 tiles that
// hold a refined cell, and one colour per other tile: such a tile contains no
// interfacial cell, so its cells share one colour, its edges carry no marker
// and its faces store their corner colour.
#pragma once
#include "band.cuh"
#include "common.cuh"

namespace ebit {

constexpr int AMR_R = TILE + 3;   // staged nodes per axis: -1 .. TILE + 1
constexpr int AMR_F = TILE + 2;   // interfacial flags of cells -1 .. TILE
constexpr int AMR_WARPS = 8;
constexpr int AMR_CHUNK = 1024;   // tiles per chunk of the compaction

// Per tile: the refinement mask of its cells (mask may be null), whether any
// of them is refined (flag), the colour of its origin node (bg, may be null),
// and the numbers of refined cells (count[0]), of flagged tiles (count[1]) and
// of flagged tiles per chunk of AMR_CHUNK (chunk).  Outputs but the mask start
// at zero where they are sums.
//
// A block takes a strip of eight tiles along x.  Its colours come as groups of 8
// cells, consecutive lanes along the rows, and are kept as one byte of bits per
// group; each warp then works on one tile, whose rows of 11 nodes it reads off
// three bytes: the flags of ten cells are a few shifts of four rows and the
// 27-cell OR of eight cells a few of nine.  The mask is written the way the
// colours are read.  Bound by the colours' way from L2 and the mask's to memory.
// (a block per tile, one byte per thread and node: 558 us at 384^3; a warp per
// tile, a lane per row: 230 us, bound by the cache lines its loads touch, one per
// lane; this form 89.)
constexpr int AMR_G = 10;  // groups of 8 nodes per row: x0 - 8 .. x0 + 71

__global__ void __launch_bounds__(32 * AMR_WARPS) refine_kernel(Grid g, const uint8_t *__restrict__ cb, long long whole,
                                                                uint8_t *__restrict__ mask, uint8_t *__restrict__ flag,
                                                                uint8_t *__restrict__ bg,
                                                                unsigned long long *__restrict__ count,
                                                                int *__restrict__ chunk) {
    __shared__ uint8_t s_col[AMR_R * AMR_R][AMR_G + 2];  // (a row of 12 bytes)
    __shared__ unsigned s_flg[AMR_WARPS][AMR_F * AMR_F];
    __shared__ uint8_t s_ref[TILE * TILE][AMR_WARPS];
    const unsigned full = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned *flg = s_flg[warp];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const long long n = (long long)nx * ny * nz;
    const int sx = (g.td[0] + AMR_WARPS - 1) / AMR_WARPS;
    const long long strips = (long long)sx * g.td[1] * g.td[2];
    unsigned nref = 0;
    for (long long st = blockIdx.x; st < strips; st += gridDim.x) {
        const int ix = (int)(st % sx), iyz = (int)(st / sx), ty = iyz % g.td[1], tz = iyz / g.td[1];
        const int x0 = ix * AMR_WARPS * TILE, y0 = ty * TILE, z0 = tz * TILE;
        int seen = 0;
#pragma unroll
        for (int q = 0; q < (AMR_R * AMR_R * AMR_G + 255) / 256; q++) {
            const int k = threadIdx.x + 256 * q;
            if (k >= AMR_R * AMR_R * AMR_G) continue;
            const int r = k / AMR_G, gr = k - r * AMR_G;
            const int y = wrapc(y0 + r % AMR_R - 1, ny), z = wrapc(z0 + r / AMR_R - 1, nz);
            const unsigned c = group_colours(cb, (z * ny + y) * nx, x0 + 8 * (gr - 1), nx, whole, n);
            s_col[r][gr] = (uint8_t)c;
            // uniform strips (of the nodes that are read) need no flags
            const unsigned used = gr == 0 ? 0x80u : (gr == AMR_G - 1 ? 0x03u : 0xFFu);
            seen |= ((c & used) ? 1 : 0) | ((~c & used) ? 2 : 0);
        }
        const int has1 = __syncthreads_or(seen & 1), has0 = __syncthreads_or(seen & 2);
        const int tx = ix * AMR_WARPS + warp, o0 = x0 + TILE * warp;
        const bool tile_ok = tx < g.td[0];
        const int tile = (tz * g.td[1] + ty) * g.td[0] + tx;
        const unsigned vx = !tile_ok ? 0u : (nx - o0 >= TILE ? 0xFFu : (1u << (nx - o0)) - 1u);
        bool any = false;
        if (has1 && has0) {
            // node row r of the warp's tile, nodes -1 .. TILE + 1
            auto row = [&](int r) -> unsigned {
                const uint8_t *c = s_col[r] + warp;
                return (unsigned)c[0] >> 7 | (unsigned)c[1] << 1 | ((unsigned)c[2] & 3u) << 9;
            };
            // interfacial flags of the cells -1 .. TILE around the tile
            for (int r = lane; r < AMR_F * AMR_F; r += 32) {
                const int i = r % AMR_F + AMR_R * (r / AMR_F);
                const unsigned p = row(i), q = row(i + 1), s = row(i + AMR_R), t = row(i + AMR_R + 1);
                const unsigned hi = p | q | s | t, lo = p & q & s & t;
                flg[r] = (hi | hi >> 1) & ~(lo & lo >> 1) & ((1u << AMR_F) - 1u);
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const int r = lane + 32 * q, ly = r & 7, lz = r >> 3;
                unsigned f = 0;
#pragma unroll
                for (int d = 0; d < 9; d++) f |= flg[ly + d % 3 + AMR_F * (lz + d / 3)];
                const unsigned ref = y0 + ly < ny && z0 + lz < nz ? (f | f >> 1 | f >> 2) & vx : 0u;
                nref += __popc(ref);
                any |= ref != 0u;
                s_ref[r][warp] = (uint8_t)ref;
            }
        } else {
            s_ref[lane][warp] = s_ref[lane + 32][warp] = 0;
        }
        const bool tile_any = __any_sync(full, any);
        if (lane == 0 && tile_ok) {
            flag[tile] = tile_any ? 1 : 0;
            if (bg) bg[tile] = s_col[1 + AMR_R][warp + 1] & 1u;  // the origin node
            if (tile_any) {
                atomicAdd(count + 1, 1ull);
                atomicAdd(chunk + tile / AMR_CHUNK, 1);
            }
        }
        __syncthreads();
        if (mask) {
#pragma unroll
            for (int q = 0; q < TILE * TILE * AMR_WARPS / 256; q++) {
                const int k = threadIdx.x + 256 * q, r = k / AMR_WARPS, gr = k % AMR_WARPS;
                const int y = y0 + (r & 7), z = z0 + (r >> 3), x = x0 + TILE * gr;
                if (y >= ny || z >= nz || x >= nx) continue;
                store_row<TILE>(mask, ((long long)z * ny + y) * nx + x, s_ref[r][gr], 0u, 0u, 0u,
                                nx - x >= TILE ? 0xFFu : (1u << (nx - x)) - 1u);
            }
        }
        __syncthreads();  // the staging is rewritten by the next strip
    }
    nref = __reduce_add_sync(full, nref);
    if (lane == 0 && nref) atomicAdd(count, (unsigned long long)nref);
}

// Ascending ids of the flagged tiles into out[0 .. cap), from the flags and the
// counts of refine_kernel: a block per chunk, which starts at the sum of the
// chunks before it.
__global__ void __launch_bounds__(256) compact_tiles_kernel(const uint8_t *__restrict__ flag, int nt,
                                                            const int *__restrict__ chunk, int *__restrict__ out,
                                                            int cap) {
    __shared__ int s_w[8], s_base;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int c = blockIdx.x; c * AMR_CHUNK < nt; c += gridDim.x) {
        if (threadIdx.x == 0) s_base = 0;
        __syncthreads();
        int sum = 0;
        for (int k = threadIdx.x; k < c; k += 256) sum += chunk[k];
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0 && sum) atomicAdd(&s_base, sum);
        const int t0 = c * AMR_CHUNK + 4 * threadIdx.x;
        int m = 0;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (t0 + j < nt && flag[t0 + j]) m |= 1 << j;
        const int cnt = __popc(m);
        unsigned total;
        const int pre = (int)warp_prefix((unsigned)cnt, &total);
        if (lane == 0) s_w[wid] = (int)total;
        __syncthreads();
        int pos = s_base + pre;
        for (int w = 0; w < wid; w++) pos += s_w[w];
        for (int j = 0; j < 4; j++)
            if ((m >> j) & 1) {
                if (pos < cap) out[pos] = t0 + j;
                pos++;
            }
        __syncthreads();
    }
}

// Brick k of the store: tile tiles[k]'s colour bytes cb[k][c] and canonical
// offsets s[k][a][c] (0 on an edge without a marker), c = cell index in the
// tile (x fastest); cells outside the grid give 0.
__global__ void __launch_bounds__(256) pack_kernel(Grid g, const uint8_t *__restrict__ cb, const double *__restrict__ s0,
                                                   const double *__restrict__ s1, const double *__restrict__ s2,
                                                   const int *__restrict__ tiles,
                                                   const unsigned long long *__restrict__ nbricks, int cap,
                                                   uint8_t *__restrict__ out_cb, double *__restrict__ out_s) {
    const int n = (int)min(*nbricks, (unsigned long long)cap);
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        int o[3];
        tile_origin(g, tiles[k], o);
        for (int c = threadIdx.x; c < TILE_CELLS; c += blockDim.x) {
            const int x = o[0] + (c & 7), y = o[1] + ((c >> 3) & 7), z = o[2] + (c >> 6);
            uint8_t b = 0;
            double v[3] = {0.0, 0.0, 0.0};
            if (x < g.n[0] && y < g.n[1] && z < g.n[2]) {
                const int id = lin(g, x, y, z);
                b = __ldg(cb + id);
                const int nb[3] = {lin(g, x + 1, y, z), lin(g, x, y + 1, z), lin(g, x, y, z + 1)};
                const double *sa[3] = {s0, s1, s2};
#pragma unroll
                for (int a = 0; a < 3; a++)
                    if (((__ldg(cb + nb[a]) ^ b) & 1) != 0) v[a] = __ldg(sa[a] + id);
            }
            out_cb[(size_t)k * TILE_CELLS + c] = b;
#pragma unroll
            for (int a = 0; a < 3; a++) out_s[((size_t)k * 3 + a) * TILE_CELLS + c] = v[a];
        }
    }
}

// slot[t] = k for tile t = tiles[k], -1 for the other tiles; ids out of range
// are counted in *bad and skipped.
__global__ void brick_slots_kernel(const int *__restrict__ tiles, int n, int nt, int *__restrict__ slot,
                                   int *__restrict__ bad) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int t = tiles[k];
        if (t < 0 || t >= nt) atomicAdd(bad, 1);
        else slot[t] = k;
    }
}

// The state from a brick store: bricks copied in, every other tile filled with
// its colour (bg: bit 0), face colours equal to it.  Both state buffers get the
// colours (a sweep leaves tiles outside its band unwritten); the offsets go to
// the first only, and only the bricks' (an offset is read where its edge
// carries a marker, and a sweep writes every marker's).  One thread per 8 cells
// of an x-row of tiles; HBM writes of two bytes per cell.
__global__ void __launch_bounds__(256) unpack_kernel(Grid g, const int *__restrict__ slot, const uint8_t *__restrict__ in_cb,
                                                     const double *__restrict__ in_s, const uint8_t *__restrict__ bg,
                                                     uint8_t *__restrict__ cb, uint8_t *__restrict__ cb2,
                                                     double *__restrict__ s0, double *__restrict__ s1,
                                                     double *__restrict__ s2) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const long long groups = (long long)g.td[0] * ny * nz, stride = (long long)gridDim.x * blockDim.x;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < groups; t += stride) {
        const int row = (int)(t / g.td[0]), tx = (int)(t - (long long)row * g.td[0]);
        const int z = row / ny, y = row - z * ny;
        const int tile = ((z >> 3) * g.td[1] + (y >> 3)) * g.td[0] + tx;
        const long long id = (long long)row * nx + 8 * tx;
        const int cnt = min(8, nx - 8 * tx);
        const int k = slot[tile];
        unsigned long long v = (bg[tile] & 1) ? 0x0F0F0F0F0F0F0F0Full : 0ull;
        if (k >= 0) {
            const int c = ((y & 7) + 8 * (z & 7)) * 8;
            const uint8_t *bc = in_cb + (size_t)k * TILE_CELLS + c;
            const double *bs = in_s + (size_t)k * 3 * TILE_CELLS + c;
            v = 0;
            for (int j = 0; j < cnt; j++) {
                v |= (unsigned long long)__ldg(bc + j) << (8 * j);
                s0[id + j] = __ldg(bs + j);
                s1[id + j] = __ldg(bs + TILE_CELLS + j);
                s2[id + j] = __ldg(bs + 2 * TILE_CELLS + j);
            }
        }
        if (cnt == 8 && (((uintptr_t)(cb + id) | (uintptr_t)(cb2 + id)) & 7) == 0) {
            *reinterpret_cast<unsigned long long *>(cb + id) = v;
            *reinterpret_cast<unsigned long long *>(cb2 + id) = v;
        } else {
            for (int j = 0; j < cnt; j++) cb[id + j] = cb2[id + j] = (uint8_t)(v >> (8 * j));
        }
    }
}

}  // namespace ebit
