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

constexpr int AMR_CHUNK = 1024;    // tiles per chunk of the compaction
constexpr int AMR_TX = 8;          // a block's tiles along x: rows of 64 cells
constexpr int AMR_TZ = 2;          // ... and along z
constexpr int AMR_THREADS = TILE * TILE * AMR_TZ;         // a thread per row of cells
constexpr int AMR_NY = TILE + 3, AMR_NZ = TILE * AMR_TZ + 3;  // node rows staged: -1 .. +1 past the end
constexpr int AMR_FY = TILE + 2, AMR_FZ = TILE * AMR_TZ + 2;  // cell rows flagged: -1 .. the end
constexpr int AMR_G = AMR_TX + 2;  // groups of 8 nodes per row: x0 - 8 .. x0 + 71

__host__ __device__ inline long long refine_blocks(const Grid &g) {
    return (long long)((g.td[0] + AMR_TX - 1) / AMR_TX) * g.td[1] * ((g.td[2] + AMR_TZ - 1) / AMR_TZ);
}

// Per tile: the refinement mask of its cells (mask may be null), whether any
// of them is refined (flag), the colour of its origin node (bg, may be null),
// and the numbers of refined cells (count[0]), of flagged tiles (count[1]) and
// of flagged tiles per chunk of AMR_CHUNK (chunk).  Outputs but the mask start
// at zero where they are sums.
//
// A block takes 64 x 8 x 16 cells.  Its node rows are kept as 64-bit words (and
// the nodes -1, 64 and 65 in a second one), read in groups of 8 colours,
// consecutive lanes along the rows; the flags of a row of 64 cells and their
// spread along x are some twenty operations on four rows, the 27-cell OR of a row
// nine words.  A block of one colour skips both.  Bound by instruction issue,
// most of it taking the colours in: hence whole words, and the two tiles along z,
// which share their halo rows.  (A block per tile, a byte per thread: 558 us at
// 384^3; a warp per tile, a lane per row: 230 us; eight tiles along x with a warp
// per tile's flags: 84 us; this form 40.)
__global__ void __launch_bounds__(AMR_THREADS) refine_kernel(Grid g, const uint8_t *__restrict__ cb, long long whole,
                                                             uint8_t *__restrict__ mask, uint8_t *__restrict__ flag,
                                                             uint8_t *__restrict__ bg,
                                                             unsigned long long *__restrict__ count,
                                                             int *__restrict__ chunk) {
    typedef unsigned long long u64;
    // nodes 0 .. 63 | nodes 64 .. 71 (byte 8), -8 .. -1 (byte 15)
    __shared__ ulonglong2 s_row[AMR_NY * AMR_NZ];
    __shared__ int s_off[AMR_NY * AMR_NZ];
    __shared__ u64 s_dil[AMR_FY * AMR_FZ];  // flagged cells and their neighbours along x
    __shared__ u64 s_ref[AMR_THREADS];
    __shared__ unsigned s_any[AMR_THREADS / 32][2];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const long long n = (long long)nx * ny * nz;
    const unsigned bx = (g.td[0] + AMR_TX - 1) / AMR_TX;
    const long long blocks = refine_blocks(g);
    const bool wide = mask && nx % 16 == 0 && ((uintptr_t)mask & 15) == 0;
    for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
        const unsigned byz = (unsigned)b / bx, bz = byz / (unsigned)g.td[1];
        const int tx0 = (int)((unsigned)b - byz * bx) * AMR_TX, ty = (int)(byz - bz * (unsigned)g.td[1]);
        const int x0 = tx0 * TILE, y0 = ty * TILE, z0 = (int)bz * AMR_TZ * TILE;
        // the rows' first nodes, once per row (rows past the last that a cell reads repeat it)
        for (int r = tid; r < AMR_NY * AMR_NZ; r += AMR_THREADS) {
            const int z = min(z0 + r / AMR_NY - 1, nz + 1), y = min(y0 + r % AMR_NY - 1, ny + 1);
            s_off[r] = (wrapc(z, nz) * ny + wrapc(y, ny)) * nx + x0 - 8;
        }
        __syncthreads();
        uint8_t *bytes = reinterpret_cast<uint8_t *>(s_row);
        unsigned has1 = 0, has0 = 0;
        auto keep = [&](int r, int gr, unsigned c) {
            bytes[16 * r + ((gr - 1) & 15)] = (uint8_t)c;
            const unsigned used = gr == 0 ? 0x80u : (gr == AMR_G - 1 ? 0x03u : 0xFFu);
            has1 |= c & used;
            has0 |= ~c & used;
        };
        constexpr int TASKS = AMR_NY * AMR_NZ * AMR_G;
        if (x0 >= 8 && x0 + 8 * (AMR_G - 1) <= nx && nx % 8 == 0 && whole > 0) {
            // no group at the seam, and rows start on 8 bytes
#pragma unroll 6
            for (int k = tid; k < TASKS; k += AMR_THREADS) {
                const int r = k / AMR_G, gr = k - r * AMR_G;
                keep(r, gr, gather_bits(__ldg(reinterpret_cast<const u64 *>(cb + (s_off[r] + 8 * gr)))));
            }
        } else {
            for (int k = tid; k < TASKS; k += AMR_THREADS) {
                const int r = k / AMR_G, gr = k - r * AMR_G;
                keep(r, gr, group_colours(cb, s_off[r] - x0 + 8, x0 + 8 * (gr - 1), nx, whole, n));
            }
        }
        const bool mixed = __syncthreads_or((int)has1) && __syncthreads_or((int)has0);
        const int y = tid & 7, z = tid >> 3;
        u64 ref = 0;
        if (mixed) {
            for (int r = tid; r < AMR_FY * AMR_FZ; r += AMR_THREADS) {
                const ulonglong2 *q = s_row + r % AMR_FY + AMR_NY * (r / AMR_FY);
                const ulonglong2 c0 = q[0], c1 = q[1], c2 = q[AMR_NY], c3 = q[AMR_NY + 1];
                const u64 hi = c0.x | c1.x | c2.x | c3.x, lo = c0.x & c1.x & c2.x & c3.x;
                const u64 he = c0.y | c1.y | c2.y | c3.y, le = c0.y & c1.y & c2.y & c3.y;
                const u64 f = (hi | hi >> 1 | he << 63) & ~(lo & (lo >> 1 | le << 63));  // cells 0 .. 63
                const u64 fm = (he >> 63 | hi) & ~(le >> 63 & lo) & 1u;                  // cell -1
                const u64 fp = (he | he >> 1) & ~(le & le >> 1);                          // cell 64: bit 0
                s_dil[r] = f | f << 1 | f >> 1 | fm | fp << 63;
            }
            __syncthreads();
            const u64 *q = s_dil + y + AMR_FY * z;
#pragma unroll
            for (int d = 0; d < 9; d++) ref |= q[d % 3 + AMR_FY * (d / 3)];
            if (nx - x0 < 64) ref &= (1ull << (nx - x0)) - 1ull;
            if (y0 + y >= ny || z0 + z >= nz) ref = 0;
            const unsigned nref = __reduce_add_sync(full, (unsigned)__popcll(ref));
            if (lane == 0 && nref) atomicAdd(count, (u64)nref);
        }
        s_ref[tid] = ref;
        const unsigned a0 = __reduce_or_sync(full, (unsigned)ref), a1 = __reduce_or_sync(full, (unsigned)(ref >> 32));
        if (lane == 0) {
            s_any[warp][0] = a0;
            s_any[warp][1] = a1;
        }
        __syncthreads();
        if (tid < AMR_TX * AMR_TZ) {  // a thread per tile
            const int k = tid % AMR_TX, zt = tid / AMR_TX, tx = tx0 + k, tz = (int)bz * AMR_TZ + zt;
            if (tx < g.td[0] && tz < g.td[2]) {
                const int tile = (tz * g.td[1] + ty) * g.td[0] + tx;
                const bool any = ((s_any[2 * zt][k >> 2] | s_any[2 * zt + 1][k >> 2]) >> (8 * (k & 3))) & 0xFFu;
                flag[tile] = any ? 1 : 0;
                if (bg) bg[tile] = (uint8_t)(s_row[1 + AMR_NY * (1 + TILE * zt)].x >> (8 * k) & 1u);  // the origin node
                if (any) {
                    atomicAdd(count + 1, 1ull);
                    atomicAdd(chunk + tile / AMR_CHUNK, 1);
                }
            }
        }
        if (wide) {
#pragma unroll 4
            for (int k = tid; k < AMR_THREADS * AMR_TX / 2; k += AMR_THREADS) {
                const int r = k / (AMR_TX / 2), q = k % (AMR_TX / 2);
                const int yy = y0 + (r & 7), zz = z0 + (r >> 3), x = x0 + 16 * q;
                if (yy >= ny || zz >= nz || x >= nx) continue;
                const unsigned w = (unsigned)(s_ref[r] >> (16 * q));
                *reinterpret_cast<ulonglong2 *>(mask + (((long long)zz * ny + yy) * nx + x)) =
                    make_ulonglong2(spread_bits(w), spread_bits(w >> 8));
            }
        } else if (mask) {
            for (int k = tid; k < AMR_THREADS * AMR_TX; k += AMR_THREADS) {
                const int r = k / AMR_TX, q = k % AMR_TX;
                const int yy = y0 + (r & 7), zz = z0 + (r >> 3), x = x0 + 8 * q;
                if (yy >= ny || zz >= nz || x >= nx) continue;
                store_row<TILE>(mask, ((long long)zz * ny + yy) * nx + x, (unsigned)(s_ref[r] >> (8 * q)) & 0xFFu, 0u, 0u,
                                0u, nx - x >= TILE ? 0xFFu : (1u << (nx - x)) - 1u);
            }
        }
        __syncthreads();  // the staging is rewritten by the next round
    }
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
// the first only, and only where an edge may carry a marker (an offset is read
// there only, and a sweep writes every marker's): the bricks', and 0 on the edges
// into a brick from a tile outside the store whose colour differs (a packed store has
// none: that tile would hold a refined cell; but any store may be unpacked, and the
// context's old offsets must not show; background_seams has the edges between two
// tiles outside it).  A warp takes 32 groups
// of up to 8 cells in a row: a lane writes its group's colours, and the bricks'
// offsets go in 16-byte pieces, lane after lane.  Two bytes per cell and the bricks
// are 17 us of traffic at 384^3; bound by issue (61 % of the slots) and latency.  (A lane per row of a brick, value by value: 68 us at 384^3;
// this form 54, with the edges into a brick 57.  A background lane's look at the next
// tiles, or a kernel of its own for them, cost 12 us in place of 3.)
__global__ void __launch_bounds__(256) unpack_kernel(Grid g, const int *__restrict__ slot, const uint8_t *__restrict__ in_cb,
                                                     const double *__restrict__ in_s, const uint8_t *__restrict__ bg,
                                                     uint8_t *__restrict__ cb, uint8_t *__restrict__ cb2,
                                                     double *__restrict__ s0, double *__restrict__ s1,
                                                     double *__restrict__ s2) {
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    const bool wide = nx % 2 == 0 && (((uintptr_t)in_s | (uintptr_t)s0 | (uintptr_t)s1 | (uintptr_t)s2) & 15) == 0;
    const long long groups = (long long)g.td[0] * ny * nz, stride = (long long)gridDim.x * blockDim.x;
    for (long long t0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < groups; t0 += stride) {
        const long long t = t0 + lane;
        int id = 0, cnt = 0, row8 = -1;  // row8: the group's row of its brick, in units of 8 cells
        if (t < groups) {
            const int row = (int)((unsigned)t / (unsigned)g.td[0]), tx = (int)t - row * g.td[0];
            const int z = row / ny, y = row - z * ny;
            const int tile = ((z >> 3) * g.td[1] + (y >> 3)) * g.td[0] + tx;
            id = row * nx + 8 * tx;
            cnt = min(8, nx - 8 * tx);
            const int k = slot[tile];
            unsigned long long v = (bg[tile] & 1) ? 0x0F0F0F0F0F0F0F0Full : 0ull;
            if (k >= 0) {
                const int c = (y & 7) + 8 * (z & 7);
                // the tile behind along each axis in which this is its first layer
                const int bx = tx ? tile - 1 : tile + g.td[0] - 1,
                          by = (y & 7) ? tile : (y ? tile : tile + g.td[1] * g.td[0]) - g.td[0],
                          bz = (z & 7) ? tile : (z ? tile : tile + g.ntiles) - g.td[1] * g.td[0];
                const int kx = slot[bx], ky = slot[by], kz = slot[bz], cx = bg[bx], cy = bg[by], cz = bg[bz];
                const uint8_t *bc = in_cb + (size_t)k * TILE_CELLS + c * 8;
                row8 = k * 3 * (TILE_CELLS / 8) + c;
                if (((uintptr_t)bc & 7) == 0) {
                    v = __ldg(reinterpret_cast<const unsigned long long *>(bc));
                } else {
                    v = 0;
                    for (int j = 0; j < 8; j++) v |= (unsigned long long)__ldg(bc + j) << (8 * j);
                }
                if (kx < 0 && ((v ^ cx) & 1)) s0[id + (tx ? -1 : nx - 1)] = 0.0;
                const unsigned colours = gather_bits(v), ok = (1u << cnt) - 1u;
                for (unsigned m = ky < 0 ? (colours ^ (cy & 1 ? 0xFFu : 0u)) & ok : 0u; m; m &= m - 1)
                    s1[id + __ffs((int)m) - 1 + (y ? -nx : (ny - 1) * nx)] = 0.0;
                for (unsigned m = kz < 0 ? (colours ^ (cz & 1 ? 0xFFu : 0u)) & ok : 0u; m; m &= m - 1)
                    s2[id + __ffs((int)m) - 1 + (z ? -ny * nx : (nz - 1) * ny * nx)] = 0.0;
            }
            if (cnt == 8 && (((uintptr_t)(cb + id) | (uintptr_t)(cb2 + id)) & 7) == 0) {
                *reinterpret_cast<unsigned long long *>(cb + id) = v;
                *reinterpret_cast<unsigned long long *>(cb2 + id) = v;
            } else {
                for (int j = 0; j < cnt; j++) cb[id + j] = cb2[id + j] = (uint8_t)(v >> (8 * j));
            }
        }
        if (!__any_sync(full, row8 >= 0)) continue;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int from = 8 * j + (lane >> 2), b = 2 * (lane & 3);
            const int r8 = __shfl_sync(full, row8, from), left = __shfl_sync(full, cnt, from) - b;
            const int at = __shfl_sync(full, id, from) + b;
            if (r8 < 0 || left <= 0) continue;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                const double *p = in_s + (size_t)(r8 + a * (TILE_CELLS / 8)) * 8 + b;
                double *q = (a == 0 ? s0 : a == 1 ? s1 : s2) + at;
                if (wide && left > 1) {
                    *reinterpret_cast<double2 *>(q) = __ldg(reinterpret_cast<const double2 *>(p));
                } else {
                    q[0] = __ldg(p);
                    if (left > 1) q[1] = __ldg(p + 1);
                }
            }
        }
    }
}

}  // namespace ebit
