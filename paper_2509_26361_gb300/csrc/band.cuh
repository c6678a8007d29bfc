// band.cuh -- the integer pass of a split sweep over the band tiles
// (arxiv 2509.26361, Sec. 2.1-2.3; the method and the kernels around it are
// described in sweep.cuh).
//
// Two warps per tile, bit-parallel over the tile's x-rows.  A row's node colours
// are one bit mask, so the colour window of all its cells, the crossings of the
// aligned markers (two masks: crossed the upper node, crossed the lower node),
// the new colours, the edges that carry a marker, the saddle faces and the
// annihilation checks are shifts and exclusive-ors of a few words; only the
// markers themselves (their bins, and the coordinates of the aligned ones that
// stay) are handled one per lane, from lists the warps compact in shared memory.
//
// What bounds it: the latency of one tile's chain (list entry, colours, bins,
// list slots and aligned coordinates: four dependent rounds through L2) and the
// issue of its about 1300 instructions.  A block of 256 threads per tile (one
// thread per two cells, 3000 warp instructions per interface tile) held four
// tiles on an SM; 64 threads hold sixteen, and their 64 lanes match the 64 rows
// of cells of an 8^3 tile (one warp per tile had the longer chain: 11 us
// against 8 for the 64 tiles of 32^3).  Measured per sweep, before and now: 66
// and 18 us at 512^3, 23 and 10 at 128^3, 12 and 8 at 32^3.
#pragma once
#include "common.cuh"
#include "sweep_args.cuh"

namespace ebit {

__host__ __device__ constexpr int tile_edge(int sh, int a) { return 1 << tile_log2(sh, a); }

// the staged region of a tile: nodes -1 .. T + 1 along the sweep axis, 0 .. T
// along the others (T: the tile's edge on that axis)
template <int D, int SH>
struct BandRegion {
    static constexpr int TX = tile_edge(SH, 0), TY = tile_edge(SH, 1), TZ = tile_edge(SH, 2);
    static_assert(TX * TY * TZ == TILE_CELLS && TX > NEAR && TY > NEAR && TZ > NEAR, "see Tile shapes");
    static constexpr int X0 = D == 0 ? -1 : 0, Y0 = D == 1 ? -1 : 0, Z0 = D == 2 ? -1 : 0;
    static constexpr int RX = TX + (D == 0 ? 3 : 1), RY = TY + (D == 1 ? 3 : 1), RZ = TZ + (D == 2 ? 3 : 1);
    static constexpr int ROWS = RY * RZ;      // x-rows
    static constexpr int CELL_ROWS = TY * TZ; // x-rows of cells
};
template <bool WIDE>
struct RowMask {
    using type = uint32_t;
};
template <>
struct RowMask<true> {
    using type = uint64_t;
};

constexpr int BAND_THREADS = 64;  // per tile

// a tile's shared memory
template <int D, int SH>
struct BandSmem {
    using R = BandRegion<D, SH>;
    using M = typename RowMask<(R::RX > 32)>::type;
    // Rows go to the 64 lanes in turn.  Each warp lists the marked edges of its
    // rows in a part of its own, and later the aligned markers of its cell rows.
    static constexpr int PER_ROW = R::RX - (D == 0);
    static constexpr int ROWS0 = (R::ROWS < 32 ? R::ROWS : 32) +
                                 (R::ROWS <= 64 ? 0 : (R::ROWS - 64 < 32 ? R::ROWS - 64 : 32));  // rows of warp 0
    static constexpr int LIST1 = ROWS0 * PER_ROW;                                                // warp 1's part
    static_assert(R::ROWS <= 128, "two rows per lane");
    static_assert(R::CELL_ROWS <= 32 ? R::CELL_ROWS * R::TX <= R::ROWS * PER_ROW
                                     : 32 * R::TX <= LIST1 && (R::CELL_ROWS - 32) * R::TX <= R::ROWS * PER_ROW - LIST1,
                  "the aligned markers fit the parts");
    M C[R::ROWS];   // node colours (bit x - X0)
    M up[R::ROWS];  // sweep-axis edges whose marker crossed the upper node (bin >= 2)
    M dn[R::ROWS];  // ... the lower node (bin < 0)
    M nc[R::ROWS];  // new colours (bit x)
    uint32_t fa[R::CELL_ROWS];  // old colours of the faces normal to the sweep (bit x)
    unsigned seen[2], near[2];  // per warp: colours staged, proximity mask
    uint16_t list[R::ROWS * PER_ROW];  // row * 64 + bit of a marked edge; later the aligned markers
};

// barrier of a tile's threads (named barrier `id`)
__device__ __forceinline__ void band_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(BAND_THREADS) : "memory");
}

__device__ __forceinline__ int ffs_mask(uint32_t m) { return __ffs((int)m); }
__device__ __forceinline__ int ffs_mask(uint64_t m) { return __ffsll((long long)m); }
__device__ __forceinline__ int popc_mask(uint32_t m) { return __popc(m); }
__device__ __forceinline__ int popc_mask(uint64_t m) { return __popcll(m); }
__device__ __forceinline__ void or_mask(uint32_t *p, uint32_t m) { atomicOr(p, m); }
__device__ __forceinline__ void or_mask(uint64_t *p, uint64_t m) {
    atomicOr(reinterpret_cast<unsigned long long *>(p), (unsigned long long)m);
}

// bit 0 of each of 8 bytes -> 8 bits
__device__ __forceinline__ unsigned gather_bits(unsigned long long v) {
    return (unsigned)(((v & 0x0101010101010101ull) * 0x0102040810204080ull) >> 56);
}
// 8 bits -> bit 0 of 8 bytes
__device__ __forceinline__ unsigned long long spread_bits(unsigned m) {
    const unsigned long long t = (unsigned long long)(m & 0xFFu) * 0x0101010101010101ull & 0x8040201008040201ull;
    return ((t + 0x7F7F7F7F7F7F7F7Full) >> 7) & 0x0101010101010101ull;
}

// Colour bytes i .. i + 7 (0 past the end of the array).  whole: the bytes from
// cb that may be read as aligned 8-byte words (0 when cb is not aligned): any
// position is then one or two word loads.
__device__ __forceinline__ unsigned long long load_colours8(const uint8_t *__restrict__ cb, long long i, long long whole,
                                                            long long n) {
    if (i + 8 <= whole) {
        const unsigned long long *w = reinterpret_cast<const unsigned long long *>(cb) + (i >> 3);
        const int sh = (int)(i & 7) * 8;
        unsigned long long v = __ldg(w);
        if (sh) v = v >> sh | __ldg(w + 1) << (64 - sh);
        return v;
    }
    unsigned long long v = 0;
    for (int k = 0; k < 8; k++)
        if (i + k < n) v |= (unsigned long long)__ldg(cb + i + k) << (8 * k);
    return v;
}

// Colours of nodes x .. x + 7 (periodic) of the row that starts at node `row`, as
// bits, for passes over whole strips of tiles; x from -8 (only node -1 is read)
// to past the end of the row.
__device__ __forceinline__ unsigned group_colours(const uint8_t *__restrict__ cb, int row, int x, int nx, long long whole,
                                                  long long n) {
    if (x < 0) return (unsigned)(__ldg(cb + row + nx - 1) & 1) << 7;
    if (x >= nx) x -= nx;
    if (x >= nx) return 0u;
    const unsigned c = gather_bits(load_colours8(cb, (long long)row + x, whole, n));
    if (x + 8 <= nx) return c;
    const int v = nx - x;
    return (c & ((1u << v) - 1u)) | ((gather_bits(load_colours8(cb, row, whole, n)) << v) & 0xFFu);
}

// The colours of nodes x0 + X0 .. x0 + X0 + RX - 1 (periodic) of the x-row that
// starts at node `row`, bit x - x0 - X0, and bit `fbit` of the bytes of the TX
// cells (bit x - x0) in *fa.
template <typename M, int TX, int X0, int RX>
__device__ __forceinline__ M load_row(const uint8_t *__restrict__ cb, int row, int x0, int nx, long long whole,
                                      long long n, int fbit, uint32_t *fa) {
    M c = 0;
    uint32_t f = 0;
    if (x0 + TX <= nx) {
#pragma unroll
        for (int g = 0; g < TX / 8; g++) {
            const unsigned long long v = load_colours8(cb, (long long)row + x0 + 8 * g, whole, n);
            c |= (M)gather_bits(v) << (8 * g - X0);
            f |= gather_bits(v >> fbit) << (8 * g);
        }
        if (X0 < 0) c |= (M)(__ldg(cb + row + wrapc(x0 - 1, nx)) & 1);
#pragma unroll
        for (int k = TX; k < RX + X0; k++) c |= (M)(__ldg(cb + row + wrapc(x0 + k, nx)) & 1) << (k - X0);
    } else {
        // the last, clipped tile of a row: `v` nodes, then the row's first ones
        // (the region wraps once at most)
        const int v = nx - x0;
        uint64_t lo = 0, fl = 0, w = 0;
#pragma unroll
        for (int g = 0; g < TX / 8; g++) {
            const unsigned long long b = load_colours8(cb, (long long)row + x0 + 8 * g, whole, n);
            lo |= (uint64_t)gather_bits(b) << (8 * g);
            fl |= (uint64_t)gather_bits(b >> fbit) << (8 * g);
        }
#pragma unroll
        for (int g = 0; g <= (TX + 1) / 8; g++)
            w |= (uint64_t)gather_bits(load_colours8(cb, (long long)row + 8 * g, whole, n)) << (8 * g);
        const uint64_t mine = ((uint64_t)1 << v) - 1;
        lo = ((lo & mine) | w << v) & (((uint64_t)1 << (RX + X0)) - 1);
        f = (uint32_t)(fl & mine);
        c = (M)(lo << -X0);
        if (X0 < 0) c |= (M)(__ldg(cb + row + wrapc(x0 - 1, nx)) & 1);
    }
    *fa = f;
    return c;
}

// The colour bytes of TX cells from node i (planes of bits: node colour and the
// three face colours), the cells of `valid` only.
template <int TX>
__device__ __forceinline__ void store_row(uint8_t *cb, long long i, uint32_t n0, uint32_t f0, uint32_t f1, uint32_t f2,
                                          uint32_t valid) {
#pragma unroll
    for (int g = 0; g < TX / 8; g++) {
        const unsigned long long v = spread_bits(n0 >> (8 * g)) | spread_bits(f0 >> (8 * g)) << 1 |
                                     spread_bits(f1 >> (8 * g)) << 2 | spread_bits(f2 >> (8 * g)) << 3;
        const uint32_t ok = (valid >> (8 * g)) & 0xFFu;
        uint8_t *p = cb + i + 8 * g;
        if (ok == 0xFFu && ((uintptr_t)p & 7) == 0) {
            *reinterpret_cast<unsigned long long *>(p) = v;
        } else {
#pragma unroll
            for (int k = 0; k < 8; k++)
                if ((ok >> k) & 1u) p[k] = (uint8_t)(v >> (8 * k));
        }
    }
}

// four nodes of a face hold a marker on every edge
__device__ __forceinline__ uint32_t saddles(uint32_t c00, uint32_t c10, uint32_t c01, uint32_t c11) {
    return ~(c00 ^ c11) & ~(c10 ^ c01) & (c00 ^ c10);
}

// events of the tiles a warp has processed (one value per lane, summed at the end)
struct BandEvents {
    unsigned markers = 0, annihilate = 0, multi = 0, inconsistent = 0;
};
// every lane of the warp must call it
__device__ __forceinline__ void flush_events(const BandEvents &e, unsigned long long *ctr) {
    const unsigned full = 0xffffffffu;
    if (!__any_sync(full, e.markers | e.annihilate | e.multi | e.inconsistent)) return;
    const unsigned v[4] = {__reduce_add_sync(full, e.markers), __reduce_add_sync(full, e.annihilate),
                           __reduce_add_sync(full, e.multi), __reduce_add_sync(full, e.inconsistent)};
    if ((threadIdx.x & 31) == 0) {
        if (v[0]) atomicAdd(ctr + C_MARKERS, (unsigned long long)v[0]);
        if (v[1]) atomicAdd(ctr + C_ANNIHILATE, (unsigned long long)v[1]);
        if (v[2]) atomicAdd(ctr + C_MULTI, (unsigned long long)v[2]);
        if (v[3]) atomicAdd(ctr + C_INCONSISTENT, (unsigned long long)v[3]);
    }
}

// exclusive prefix over the warp's lanes of `v` (three counts of 10 bits each);
// *total gets the sum
__device__ __forceinline__ unsigned warp_prefix(unsigned v, unsigned *total) {
    const int lane = threadIdx.x & 31;
    unsigned inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += t;
    }
    *total = __shfl_sync(0xffffffffu, inc, 31);
    return inc - v;
}

// One band tile of grid g, 64 threads (`bar`: a named barrier of theirs); the
// caller synchronises them before `sm` is used again.  The grid's cells start
// at `base` and its tiles at `tbase` of the arrays (0, 0 for a single context, its
// slice of the arena for an instance of a batch); `whole`: see load_colours8,
// for the colours from base on.  Ids on the lists count from the arrays' start.
// With F, data written earlier in the same launch
// (bins, advected coordinates) is read through L2.
template <int D, bool F, int SH = 0>
__device__ __forceinline__ void band_tile(const SweepArgs &a, const Grid &g, int base0, int tbase, long long whole, int tile,
                                          BandSmem<D, SH> &sm, int bar, BandEvents &ev) {
    using R = BandRegion<D, SH>;
    using M = typename BandSmem<D, SH>::M;
    constexpr int A = D, T1 = (D + 1) % 3, T2 = (D + 2) % 3;
    constexpr int TX = R::TX, TY = R::TY, TZ = R::TZ, RY = R::RY, X0 = R::X0, Y0 = R::Y0, Z0 = R::Z0;
    constexpr int RPL = (R::ROWS + 63) / 64;  // rows per lane (of cells: one, R::CELL_ROWS <= 64)
    constexpr uint32_t MT = TX == 32 ? 0xFFFFFFFFu : (1u << (TX & 31)) - 1u;
    constexpr M MR = ((M)1 << R::RX) - 1;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x & (BAND_THREADS - 1), lane = tid & 31, warp = tid >> 5;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const long long n = (long long)nx * ny * nz;
    const uint8_t *cb = a.cb + base0;
    uint16_t *list = sm.list + (warp ? BandSmem<D, SH>::LIST1 : 0);
    int o[3];
    tile_origin(g, tile, o);

    // ---- the region's colours
    M mine[RPL];
    bool any1 = false, any0 = false;
#pragma unroll
    for (int q = 0; q < RPL; q++) {
        const int r = tid + BAND_THREADS * q;
        mine[q] = 0;
        if (r >= R::ROWS) continue;
        const int ry = r % RY + Y0, rz = r / RY + Z0;
        uint32_t f;
        const M c = load_row<M, TX, X0, R::RX>(cb, (wrapc(o[2] + rz, nz) * ny + wrapc(o[1] + ry, ny)) * nx, o[0], nx,
                                              whole, n, 1 + A, &f);
        mine[q] = c;
        sm.C[r] = c;
        sm.up[r] = 0;
        sm.dn[r] = 0;
        if (ry >= 0 && ry < TY && rz >= 0 && rz < TZ) sm.fa[ry + TY * rz] = f;
        any1 |= c != 0;
        any0 |= c != MR;
    }
    const unsigned seen = (__any_sync(full, any1) ? 1u : 0u) | (__any_sync(full, any0) ? 2u : 0u);
    if (lane == 0) sm.seen[warp] = seen;
    band_sync(bar);
    const unsigned colours = sm.seen[0] | sm.seen[1];
    uint32_t vx = MT;  // the row's cells inside the grid
    if (nx - o[0] < TX) vx = (1u << (nx - o[0])) - 1u;
    // the lane's row of cells
    const int ly = tid % TY, lz = tid / TY, y = o[1] + ly, z = o[2] + lz;
    const bool row_ok = tid < R::CELL_ROWS && y < ny && z < nz;
    const int rowid = base0 + (z * ny + y) * nx + o[0];
    if (colours != 3u) {
        // Every staged node has one colour: no marker lies on an edge whose
        // crossing could change a node, face or edge of this tile's cells, so
        // the sweep leaves them as they are: canonical colour bytes, no markers,
        // no work, and nothing for Front2VOF to redo.
        const uint32_t c = colours == 1u ? MT : 0u;
        if (row_ok) store_row<TX>(a.cbo, rowid, c, c, c, c, vx);
        if (tid == 0) {
            a.tile_marker[tbase + tile] = 0u;
            if (a.band_flag) a.band_flag[tbase + tile] = 0u;
        }
        return;
    }

    // ---- the marked edges along the sweep axis, listed, then their crossings
    M mk[RPL];
    int cnt = 0;
#pragma unroll
    for (int q = 0; q < RPL; q++) {
        const int r = tid + BAND_THREADS * q;
        mk[q] = 0;
        if (r >= R::ROWS) continue;
        if (A == 0) mk[q] = (mine[q] ^ mine[q] >> 1) & (MR >> 1);
        if (A == 1 && r % RY < RY - 1) mk[q] = mine[q] ^ sm.C[r + 1];
        if (A == 2 && r / RY < R::RZ - 1) mk[q] = mine[q] ^ sm.C[r + RY];
        cnt += popc_mask(mk[q]);
    }
    unsigned total;
    int at = (int)warp_prefix((unsigned)cnt, &total);
#pragma unroll
    for (int q = 0; q < RPL; q++) {
        const int r = tid + BAND_THREADS * q;
        for (M m = mk[q]; m; m &= m - 1) list[at++] = (uint16_t)(r * 64 + ffs_mask(m) - 1);
    }
    __syncwarp();
    for (int k0 = 0; k0 < (int)total; k0 += 64) {  // two loads in flight per lane
        int code[2], b[2];
#pragma unroll
        for (int j = 0; j < 2; j++) {
            const int k = k0 + 32 * j + lane;
            code[j] = k < (int)total ? list[k] : -1;
            b[j] = 0;
            if (code[j] >= 0) {
                const int r = code[j] >> 6;
                b[j] = ld_in<F>(a.bin[A] + base0 + lin(g, o[0] + (code[j] & 63) + X0, o[1] + r % RY + Y0, o[2] + r / RY + Z0));
            }
        }
#pragma unroll
        for (int j = 0; j < 2; j++) {
            // X >= 1 <=> bin >= 2, X < 0 <=> bin < 0 (Fig. 4)
            if (b[j] >= 2) or_mask(&sm.up[code[j] >> 6], (M)1 << (code[j] & 63));
            if (b[j] < 0) or_mask(&sm.dn[code[j] >> 6], (M)1 << (code[j] & 63));
        }
    }
    band_sync(bar);

    // ---- new node colours: flipped once per marker that crossed the node
#pragma unroll
    for (int q = 0; q < RPL; q++) {
        const int r = tid + BAND_THREADS * q;
        if (r >= R::ROWS) continue;
        if (A == 0) sm.nc[r] = mine[q] >> 1 ^ sm.up[r] ^ sm.dn[r] >> 1;
        if (A == 1 && r % RY >= 1) sm.nc[r] = mine[q] ^ sm.up[r - 1] ^ sm.dn[r];
        if (A == 2 && r / RY >= 1) sm.nc[r] = mine[q] ^ sm.up[r - RY] ^ sm.dn[r];
    }
    band_sync(bar);

    // ---- the lane's cells
    // their work: unaligned edges, saddle faces and annihilation checks of the
    // two families (lists 0-5), and the aligned markers (present; landed from
    // the edge below, above; several; none)
    uint32_t wk[6] = {0, 0, 0, 0, 0, 0}, al = 0, below = 0, above = 0, many = 0, lost = 0;
    unsigned near = 0;  // proximity mask
    if (row_ok) {
        const int r0 = (ly - Y0) + RY * (lz - Z0);
        // old colours at (da, d1, d2) relative to the cells, new ones for da >= 0
        auto V = [&](int da, int d1, int d2) -> uint32_t {
            if (A == 0) return (uint32_t)(sm.C[r0 + d1 + RY * d2] >> (da + 1)) & MT;
            if (A == 1) return (uint32_t)(sm.C[r0 + da + RY * d1] >> d2) & MT;
            return (uint32_t)(sm.C[r0 + d2 + RY * da] >> d1) & MT;
        };
        auto N = [&](int da, int d1, int d2) -> uint32_t {
            if (A == 0) return (uint32_t)(sm.nc[r0 + d1 + RY * d2] >> da) & MT;
            if (A == 1) return (uint32_t)(sm.nc[r0 + da + RY * d1] >> d2) & MT;
            return (uint32_t)(sm.nc[r0 + d2 + RY * da] >> d1) & MT;
        };
        // an edge mask on the cells' own line, at offset da
        auto E = [&](const M *m, int da) -> uint32_t {
            if (A == 0) return (uint32_t)(m[r0] >> (da + 1)) & MT;
            return (uint32_t)m[r0 + (A == 1 ? da : RY * da)] & MT;
        };
        const uint32_t v000 = V(0, 0, 0), v100 = V(1, 0, 0), vm00 = V(-1, 0, 0);
        const uint32_t v010 = V(0, 1, 0), v001 = V(0, 0, 1);
        const uint32_t n0 = N(0, 0, 0), n1 = N(1, 0, 0), n01 = N(0, 1, 0), n11 = N(1, 1, 0), n02 = N(0, 0, 1),
                       n12 = N(1, 0, 1), n012 = N(0, 1, 1);
        // aligned edge (Fig. 5): presence from the new colours, landing markers
        const uint32_t pres = (n0 ^ n1) & vx;
        const uint32_t la = E(sm.up, -1), lb = (v000 ^ v100) & ~E(sm.up, 0) & ~E(sm.dn, 0), lc = E(sm.dn, 1);
        const uint32_t odd = la ^ lb ^ lc, two = (la & lb) | (la & lc) | (lb & lc);
        al = pres;
        many = pres & la & lb & lc;
        lost = pres & ~odd;
        below = la;
        above = lc;
        ev.multi += __popc(many);
        ev.inconsistent += __popc(lost);
        ev.annihilate += __popc(~pres & two & vx);
        // unaligned edges: a marker -> list; none, but a colour change around ->
        // the crossings that met there are counted (topology change, Fig. 5)
        const uint32_t p1 = (n0 ^ n01) & vx, p2 = (n0 ^ n02) & vx;
        const uint32_t along = (v000 ^ vm00) | (v100 ^ vm00);
        wk[0] = p1;
        wk[1] = p2;
        ev.markers += __popc(pres) + __popc(p1) + __popc(p2);
        wk[4] = (along | (V(-1, 1, 0) ^ vm00) | (v010 ^ vm00) | (V(1, 1, 0) ^ vm00)) & ~p1 & vx;
        wk[5] = (along | (V(-1, 0, 1) ^ vm00) | (v001 ^ vm00) | (V(1, 0, 1) ^ vm00)) & ~p2 & vx;
        // face colours: family 1 faces are normal to T2, family 2 to T1
        const uint32_t s1 = saddles(n0, n1, n01, n11), s2 = saddles(n0, n1, n02, n12), sa = saddles(n0, n01, n02, n012);
        wk[2] = s1 & vx;
        wk[3] = s2 & vx;
        uint32_t f[3];
        f[T2] = n0 & ~s1;
        f[T1] = n0 & ~s2;
        f[A] = (n0 & ~sa) | (sm.fa[tid] & sa);
        store_row<TX>(a.cbo, rowid, n0, f[0], f[1], f[2], vx);
        // cells with a marker before or after
        const uint32_t m = ((v000 ^ v100) | (v000 ^ v010) | (v000 ^ v001) | pres | p1 | p2) & vx;
        // (the layers next to the following tile, from the last cell inside the grid)
        const unsigned xs = ((m & ((1u << NEAR) - 1u)) ? 1u : 0u) | (m ? 2u : 0u) |
                            ((m >> max(min(TX, nx - o[0]) - NEAR, 0)) ? 4u : 0u);
        const unsigned ys = (ly < NEAR ? 1u : 0u) | 1u << 3 | (ly >= min(TY, ny - o[1]) - NEAR ? 1u << 6 : 0u);
        const unsigned zs = (lz < NEAR ? 1u : 0u) | 1u << 9 | (lz >= min(TZ, nz - o[2]) - NEAR ? 1u << 18 : 0u);
        near |= xs * ys * zs;
    }
    near = __reduce_or_sync(full, near);
    if (lane == 0) sm.near[warp] = near;

    // ---- slots on the lists: prefix sums over the warp, then one round of
    // independent atomics (lane k reserves list k, lane 6 the aligned markers)
    unsigned t0, t1, t2;
    const unsigned w0 = warp_prefix(__popc(wk[0]) | __popc(wk[1]) << 10 | __popc(wk[2]) << 20, &t0);
    const unsigned w1 = warp_prefix(__popc(wk[3]) | __popc(wk[4]) << 10 | __popc(wk[5]) << 20, &t1);
    const unsigned w2 = warp_prefix(__popc(al), &t2);
    int base = 0;
    if (lane < 6) {
        const unsigned c = ((lane < 3 ? t0 : t1) >> (10 * (lane % 3))) & 1023u;
        if (c) base = atomicAdd(a.wcount + lane, (int)c);
    } else if (lane == 6 && t2 && a.mk_out) {
        base = atomicAdd(a.mk_out_count, (int)t2);
    }
    // the aligned markers, compacted: cell, and which edge it came from (0
    // below, 1 the same, 2 above, 3 the median of three, 4 none)
    at = (int)w2;
    for (uint32_t m = al; m; m &= m - 1) {
        const int x = __ffs((int)m) - 1;
        const uint32_t bit = m & (0u - m);
        const int src = (lost & bit) ? 4 : (many & bit) ? 3 : (below & bit) ? 0 : (above & bit) ? 2 : 1;
        list[at++] = (uint16_t)(x | tid << 5 | src << 11);
    }
#pragma unroll
    for (int k = 0; k < 6; k++) {
        int pos = __shfl_sync(full, base, k) + (int)(((k < 3 ? w0 : w1) >> (10 * (k % 3))) & 1023u);
        // an unaligned edge is on list k or, checked for annihilation, on list
        // k + 4, never on both: the two share an array, from its two ends
        unsigned *w = k < 4 ? a.work[k] : a.work[k - 4] + (a.cells - 1);
        for (uint32_t m = wk[k]; m; m &= m - 1, pos++) w[k < 4 ? pos : -pos] = (unsigned)(rowid + __ffs((int)m) - 1);
    }
    const int bal = __shfl_sync(full, base, 6);
    __syncwarp();
    for (int k = lane; k < (int)t2; k += 32) {
        const int c = list[k], src = c >> 11, r = (c >> 5) & 63;
        const int cx = o[0] + (c & 31), cy = o[1] + r % TY, cz = o[2] + r / TY;
        const int id = base0 + (cz * ny + cy) * nx + cx;
        auto landed = [&](int e) -> double {
            const double xv =
                ld_in<F>(a.adv[A] + base0 + lin(g, cx + (A == 0 ? e : 0), cy + (A == 1 ? e : 0), cz + (A == 2 ? e : 0)));
            const double s = e == 0 ? xv : xv + (e < 0 ? -1.0 : 1.0);
            return __double_as_longlong(s) > __double_as_longlong(ONE_MINUS) ? ONE_MINUS : s;
        };
        double v;
        if (src < 3) {
            v = landed(src - 1);
        } else if (src == 3) {
            double a0 = landed(-1), a1 = landed(0), a2 = landed(1), tmp;
            if (a0 > a1) { tmp = a0; a0 = a1; a1 = tmp; }
            if (a1 > a2) { tmp = a1; a1 = a2; a2 = tmp; }
            if (a0 > a1) { tmp = a0; a0 = a1; a1 = tmp; }
            v = a1;
        } else {
            v = 0.5;
        }
        a.so[A][id] = v;
        if (a.mk_out) a.mk_out[bal + k] = (unsigned)id;
    }
    band_sync(bar);
    if (tid == 0) {
        const unsigned nm = sm.near[0] | sm.near[1];
        a.tile_marker[tbase + tile] = nm;
        a.tile_dirty[tbase + tile] = 1;
        if (a.band_flag) a.band_flag[tbase + tile] = 0u;
        if (a.mt_out && nm) a.mt_out[atomicAdd(a.mt_out_count, 1)] = tbase + tile;
    }
}

template <int D>
__global__ void __launch_bounds__(BAND_THREADS, 16) sweep_kernel(SweepArgs a) {
    __shared__ BandSmem<D, 0> sm;
    __shared__ int s_next;
    pdl_wait();
    // the first tile's id with the list's length (the list has room for every
    // tile, and the grid no more blocks than tiles)
    int tile = a.list ? a.list[blockIdx.x] : (int)blockIdx.x;
    const int ntl = a.list ? *a.count : a.g.ntiles;
    BandEvents ev;
    // after the first, each block takes tiles from a counter (tiles differ in
    // cost), read one tile ahead: the value is stored after the tile, since the
    // store waits for it, and with it all that follows in the warp
    for (int li = blockIdx.x; li < ntl;) {
        int next = li + (int)gridDim.x;
        if (threadIdx.x == 0 && a.tile_next) next = (int)gridDim.x + atomicAdd(a.tile_next, 1);
        band_tile<D, false>(a, a.g, 0, 0, a.cb_whole, tile, sm, 0, ev);
        if (threadIdx.x == 0) s_next = next;
        __syncthreads();
        li = s_next;
        if (li < ntl) tile = a.list ? a.list[li] : li;
        __syncthreads();
    }
    flush_events(ev, a.ctr);
    if (a.scan_count && blockIdx.x == 0 && threadIdx.x < 3) a.scan_count[threadIdx.x] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.ctr + C_TILES, (unsigned long long)ntl);
}

}  // namespace ebit
