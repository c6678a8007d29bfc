// f2v.cuh -- Front2VOF volume fractions (arxiv 2509.26361, Sec. 2.6, Eq. 7).
//
// Per cell: the corner colours (and the face colour on saddle faces) give the
// face segments of the six cube faces (Sec. 2.3, Fig. 7b); oriented so that the
// reference phase lies on their left seen from outside, they chain into closed
// loops, one loop per interface segment of the cell (separate loops are never
// merged, Sec. 2.4).  Each loop is fanned into triangles around the centroid of
// its markers (Eq. 7), and the reference-phase volume follows from Gauss's
// theorem with the cell's lowest corner as origin:
//     V = (A_x1 + A_y1 + A_z1) / 3 - sum_loops sum_i det(c, p_i, p_i+1) / 6,
// where A_a1 is the reference-phase area on the cube face a = 1 (the faces
// through the origin contribute nothing).  C = V clamped to [0, 1].
#pragma once
#include "band.cuh"
#include "common.cuh"

namespace ebit {

// corners of the six cube faces, counter-clockwise seen from outside
// (corner id = dx | dy<<1 | dz<<2); faces x=0, x=1, y=0, y=1, z=0, z=1
__host__ __device__ constexpr unsigned face_corners(int F) {
    return F == 0 ? 0x2640u : F == 1 ? 0x5731u : F == 2 ? 0x4510u : F == 3 ? 0x3762u : F == 4 ? 0x1320u : 0x6754u;
}
// cube edge between consecutive face corners k and k+1 (x-edges 0-3 by dy+2dz,
// y-edges 4-7 by dx+2dz, z-edges 8-11 by dx+2dy), nibble k
__host__ __device__ constexpr unsigned face_edges(int F) {
    return F == 0 ? 0x4A68u : F == 1 ? 0x97B5u : F == 2 ? 0x8290u : F == 3 ? 0x1B3Au : F == 4 ? 0x0514u : 0x6372u;
}

struct F2VArgs {
    Grid g;
    const uint8_t *__restrict__ cb;
    const double *__restrict__ s[3];
    double *__restrict__ C;
    long long cb_whole;              // see load_colours8
    uint8_t *__restrict__ dirty;     // per tile: swept since the last call (cleared here)
    int full;                        // take every tile
    unsigned *__restrict__ cut;      // cells cut by the interface (output list)
    int *__restrict__ ncut;          // its length (0 on entry)
    int *__restrict__ zero;          // the length of the next call's list, cleared here
    unsigned long long *bad;
};

__device__ __forceinline__ void cell_ids(const Grid &g, int x, int y, int z, int ids[8]) {
#pragma unroll
    for (int cid = 0; cid < 8; cid++) ids[cid] = lin(g, x + (cid & 1), y + ((cid >> 1) & 1), z + ((cid >> 2) & 1));
}

// Band pass (integers only) over the tiles swept since the last call: a cell
// with eight equal corner colours holds no marker and its fraction is that
// colour (written as a bit pattern); the others go to the global cut list (their
// fraction is written by the list kernel).
//
// 64 threads per tile, one x-row of cells each, bit-parallel as in band.cuh.
// A block finds its tiles among every gridDim-th flag, so that neighbouring
// tiles, which are swept together, fall to different blocks; that takes the
// place of a launch that listed the flagged tiles (with it and one byte load per
// cell corner: 9 us at 128^3, 25 at 512^3, 294 over every tile of 384^3; now 8,
// 14 and 152.)
template <int SH>
__global__ void __launch_bounds__(64, 16) f2v_band_kernel(F2VArgs a) {
    constexpr int TX = tile_edge(SH, 0), TY = tile_edge(SH, 1), TZ = tile_edge(SH, 2);
    constexpr int RY = TY + 1, ROWS = RY * (TZ + 1);
    constexpr uint32_t MT = TX == 32 ? 0xFFFFFFFFu : (1u << (TX & 31)) - 1u;
    using M = typename RowMask<(TX + 1 > 32)>::type;
    __shared__ M s_row[ROWS];
    __shared__ int s_tile[64], s_n;
    pdl_wait();
    if (a.zero && blockIdx.x == 0 && threadIdx.x == 0) *a.zero = 0;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31;
    const int nx = a.g.n[0], ny = a.g.n[1], nz = a.g.n[2];
    const long long n = (long long)nx * ny * nz;
    const bool even = nx % 2 == 0 && ((uintptr_t)a.C & 15) == 0;  // rows of C start on 16 bytes
    for (long long t0 = blockIdx.x; t0 < a.g.ntiles; t0 += 64ll * gridDim.x) {
        if (tid == 0) s_n = 0;
        __syncthreads();
        const long long t = t0 + (long long)tid * gridDim.x;
        bool on = false;
        if (t < a.g.ntiles) {
            const uint8_t d = a.dirty[t];
            if (d) a.dirty[t] = 0;
            on = d || a.full;
        }
        if (on) s_tile[atomicAdd(&s_n, 1)] = (int)t;
        __syncthreads();
        const int nt = s_n;
        for (int k = 0; k < nt; k++) {
            int o[3];
            tile_origin(a.g, s_tile[k], o);
#pragma unroll
            for (int q = 0; q < (ROWS + 63) / 64; q++) {
                const int r = tid + 64 * q;
                if (r >= ROWS) continue;
                uint32_t f;
                s_row[r] = load_row<M, TX, 0, TX + 1>(
                    a.cb, (wrapc(o[2] + r / RY, nz) * ny + wrapc(o[1] + r % RY, ny)) * nx, o[0], nx, a.cb_whole, n, 1, &f);
            }
            __syncthreads();
            const int ly = tid % TY, lz = tid / TY, y = o[1] + ly, z = o[2] + lz;
            const bool row_ok = tid < TY * TZ && y < ny && z < nz;
            uint32_t ones = 0, cut = 0, vx = 0;
            const int id = (z * ny + y) * nx + o[0];
            if (row_ok) {
                vx = nx - o[0] >= TX ? MT : (1u << (nx - o[0])) - 1u;
                const M *r = s_row + ly + RY * lz;
                const M all = r[0] & r[1] & r[RY] & r[RY + 1], any = r[0] | r[1] | r[RY] | r[RY + 1];
                ones = (uint32_t)(all & all >> 1) & MT;
                cut = (uint32_t)(any | any >> 1) & ~ones & vx;
            }
            unsigned total;
            int pos = (int)warp_prefix((unsigned)__popc(cut), &total);
            if (total) {
                int base = 0;
                if (lane == 0) base = atomicAdd(a.ncut, (int)total);
                pos += __shfl_sync(full, base, 0);
                for (uint32_t m = cut; m; m &= m - 1) a.cut[pos++] = (unsigned)(id + __ffs((int)m) - 1);
            }
            // the fractions, 16 bytes per lane along the rows
            constexpr int LPR = TX / 2;  // lanes per row
#pragma unroll
            for (int j = 0; j < LPR; j++) {
                const int from = j * (32 / LPR) + lane / LPR, b = 2 * (lane % LPR);
                const uint32_t w = __shfl_sync(full, ones, from) >> b, ok = __shfl_sync(full, vx, from) >> b;
                unsigned long long *p = reinterpret_cast<unsigned long long *>(a.C) + __shfl_sync(full, id, from) + b;
                const unsigned long long v0 = (w & 1u) ? 0x3FF0000000000000ull : 0ull,
                                         v1 = (w & 2u) ? 0x3FF0000000000000ull : 0ull;
                if (even && (ok & 3u) == 3u) {
                    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v0, v1);
                } else {
                    if (ok & 1u) p[0] = v0;
                    if (ok & 2u) p[1] = v1;
                }
            }
            __syncthreads();
        }
    }
}

// The band pass over every tile (8^3 tiles): a block takes 64 x 8 x 16 cells, a
// thread a row of 64.  Node rows are kept as 64-bit words (node 64 in a second
// one), read in groups of 8 colours, consecutive lanes along the rows; fractions go
// out 16 bytes per lane along the rows.  HBM bound by the fractions (a tile at a
// time, a lane per row, 152 us at 384^3; eight tiles along x, bytes of colours per
// tile row, 105; this form about 85, of which the fractions take 68).
constexpr int F2V_TX = 8, F2V_TZ = 2;                // a block's tiles along x and z
constexpr int F2V_THREADS = TILE * TILE * F2V_TZ;    // a thread per row of cells
inline long long f2v_blocks(const Grid &g) {
    return (long long)((g.td[0] + F2V_TX - 1) / F2V_TX) * g.td[1] * ((g.td[2] + F2V_TZ - 1) / F2V_TZ);
}
__global__ void __launch_bounds__(F2V_THREADS) f2v_full_kernel(F2VArgs a) {
    typedef unsigned long long u64;
    constexpr int RY = TILE + 1, RZ = TILE * F2V_TZ + 1, G = F2V_TX + 1;
    __shared__ ulonglong2 s_row[RY * RZ];  // nodes 0 .. 63 | nodes 64 .. 71 (byte 8)
    __shared__ int s_off[RY * RZ];
    __shared__ u64 s_one[F2V_THREADS];
    pdl_wait();
    if (a.zero && blockIdx.x == 0 && threadIdx.x == 0) *a.zero = 0;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nx = a.g.n[0], ny = a.g.n[1], nz = a.g.n[2];
    const long long n = (long long)nx * ny * nz;
    const bool even = nx % 2 == 0 && ((uintptr_t)a.C & 15) == 0;  // rows of C start on 16 bytes
    const unsigned bx = (a.g.td[0] + F2V_TX - 1) / F2V_TX;
    const long long blocks = (long long)bx * a.g.td[1] * ((a.g.td[2] + F2V_TZ - 1) / F2V_TZ);
    for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
        const unsigned byz = (unsigned)b / bx, bz = byz / (unsigned)a.g.td[1];
        const int tx0 = (int)((unsigned)b - byz * bx) * F2V_TX, ty = (int)(byz - bz * (unsigned)a.g.td[1]);
        const int x0 = tx0 * TILE, y0 = ty * TILE, z0 = (int)bz * F2V_TZ * TILE;
        // the rows' first nodes, once per row (rows past the last that a cell reads repeat it)
        for (int r = tid; r < RY * RZ; r += F2V_THREADS)
            s_off[r] = (wrapc(min(z0 + r / RY, nz), nz) * ny + wrapc(min(y0 + r % RY, ny), ny)) * nx + x0;
        __syncthreads();
        uint8_t *bytes = reinterpret_cast<uint8_t *>(s_row);
        constexpr int TASKS = RY * RZ * G;
        if (x0 + 8 * G <= nx && nx % 8 == 0 && a.cb_whole > 0) {
            // no group at the seam, and rows start on 8 bytes
#pragma unroll 6
            for (int k = tid; k < TASKS; k += F2V_THREADS) {
                const int r = k / G, gr = k - r * G;
                bytes[16 * r + gr] = (uint8_t)gather_bits(__ldg(reinterpret_cast<const u64 *>(a.cb + (s_off[r] + 8 * gr))));
            }
        } else {
            for (int k = tid; k < TASKS; k += F2V_THREADS) {
                const int r = k / G, gr = k - r * G;
                bytes[16 * r + gr] = (uint8_t)group_colours(a.cb, s_off[r] - x0, x0 + 8 * gr, nx, a.cb_whole, n);
            }
        }
        __syncthreads();
        const int y = tid & 7, z = tid >> 3;
        u64 one, cut;
        {
            const ulonglong2 *q = s_row + y + RY * z;
            const ulonglong2 c0 = q[0], c1 = q[1], c2 = q[RY], c3 = q[RY + 1];
            const u64 all = c0.x & c1.x & c2.x & c3.x, any = c0.x | c1.x | c2.x | c3.x;
            one = all & (all >> 1 | (c0.y & c1.y & c2.y & c3.y) << 63);
            cut = (any | any >> 1 | (c0.y | c1.y | c2.y | c3.y) << 63) & ~one;
            if (nx - x0 < 64) cut &= (1ull << (nx - x0)) - 1ull;
            if (y0 + y >= ny || z0 + z >= nz) cut = 0;
        }
        s_one[tid] = one;
        // the cut cells, tile by tile (entries next to each other on the list share
        // neighbourhoods)
        if (__any_sync(full, cut != 0)) {
            const int id = ((z0 + z) * ny + y0 + y) * nx + x0;
            for (int k = 0; k < F2V_TX; k++) {
                const unsigned m8 = (unsigned)(cut >> (8 * k)) & 0xFFu;
                if (!__any_sync(full, m8)) continue;
                unsigned total;
                int pos = (int)warp_prefix((unsigned)__popc(m8), &total);
                int base = 0;
                if (lane == 0) base = atomicAdd(a.ncut, (int)total);
                pos += __shfl_sync(full, base, 0);
                for (unsigned m = m8; m; m &= m - 1) a.cut[pos++] = (unsigned)(id + 8 * k + __ffs((int)m) - 1);
            }
        }
        if (tid < F2V_TX * F2V_TZ) {
            const int tx = tx0 + tid % F2V_TX, tz = (int)bz * F2V_TZ + tid / F2V_TX;
            if (tx < a.g.td[0] && tz < a.g.td[2]) a.dirty[(tz * a.g.td[1] + ty) * a.g.td[0] + tx] = 0;
        }
        __syncthreads();
        const int x = x0 + 2 * lane;
        if (x < nx) {
#pragma unroll 8
            for (int r = warp; r < F2V_THREADS; r += F2V_THREADS / 32) {
                const int yy = y0 + (r & 7), zz = z0 + (r >> 3);
                if (yy >= ny || zz >= nz) continue;
                const unsigned w = (unsigned)(s_one[r] >> (2 * lane));
                u64 *p = reinterpret_cast<u64 *>(a.C) + ((long long)zz * ny + yy) * nx + x;
                const u64 v0 = (w & 1u) ? 0x3FF0000000000000ull : 0ull, v1 = (w & 2u) ? 0x3FF0000000000000ull : 0ull;
                if (even) {
                    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v0, v1);
                } else {
                    p[0] = v0;
                    if (x + 1 < nx) p[1] = v1;
                }
            }
        }
        __syncthreads();  // the staging is rewritten by the next round
    }
}

// Per-cell reconstruction, registers only:
//   * face areas from closed forms -- a corner cut is the triangle l1*l2/2, a
//     cut across the face the trapezoid (l1 + l2)/2, three corners the
//     complement of a corner cut (l = distances from the cut corner or side);
//   * loops walked through successor codes packed 4 bits per edge;
//   * sum_i det(c, p_i, p_i+1) = c . sum_i (p_i x p_i+1) with c the mean of
//     the loop's markers (Eq. 7) -- the same sum reassociated, so C agrees
//     with the fan-by-fan evaluation to rounding (about 1e-16).
// Bound by the FP64 pipe on long lists and by the chain of one cell on short
// ones.  A marker's coordinates but one are 0 or 1, so of the six products of a
// cross product five are selections; the faces' cases differ by selected
// operands, not by branches, so lanes with different cuts share one instruction
// stream (72 registers, where the branching form took 160; 62 to 45 us at 512^3;
// with multiply-adds, exact halves and quotients by known reciprocals 37).
__device__ __forceinline__ double sel01(int b) { return __longlong_as_double(b ? 0x3FF0000000000000ll : 0ll); }

// a loop's number of markers (up to 12) as a double, by its bit pattern
__device__ __forceinline__ double small_count(int k) {
    const int e = 31 - __clz(k);
    return __hiloint2double((1023 + e) << 20 | (k << (20 - e) & 0xFFFFF), 0);
}

// v / 2: an exponent decrement for a normal number with a normal half
__device__ __forceinline__ double half_of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return ((b >> 52) & 0x7FF) > 1 ? __longlong_as_double((long long)(b - (1ull << 52))) : 0.5 * v;
}

// 1 / k correctly rounded, k = 1 .. 12
static __constant__ double kInverse[13] = {0.0,       1.0,       1.0 / 2.0, 1.0 / 3.0, 1.0 / 4.0,  1.0 / 5.0, 1.0 / 6.0,
                                           1.0 / 7.0, 1.0 / 8.0, 1.0 / 9.0, 1.0 / 10.0, 1.0 / 11.0, 1.0 / 12.0};

__device__ __forceinline__ void marker_xyz(int e, double s, double &x, double &y, double &z) {
    const int ax = e >> 2, r = e & 3;
    const double u = sel01(r & 1), v = sel01(r >> 1);
    x = ax == 0 ? s : u;
    y = ax == 1 ? s : (ax == 0 ? u : v);
    z = ax == 2 ? s : v;
}

// Links the segments of face F into the successor codes (a segment runs from one
// cube edge to the next with the reference phase on its left) and, for an upper
// face (odd F), returns its reference-phase area.  Of the face's edges 0 and 1
// run from corner k to k + 1, 2 and 3 back, on every face, which fixes
// whether a distance is s or 1 - s.
// eds, cors: the face's edges and corners as nibbles; upper: an odd F.
__device__ __forceinline__ double face_area_and_links(unsigned eds, unsigned cors, bool upper, int K, int phif,
                                                      const double *sE, int stride, unsigned long long &nxt) {
    int cols = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) cols |= ((K >> ((cors >> (4 * k)) & 7)) & 1) << k;
    auto edge = [&](int k) -> int { return (int)((eds >> (4 * k)) & 15u); };
    auto link = [&](int from, int to, bool on) {
        const unsigned long long m = on ? 0xFull << (4 * from) : 0ull;
        nxt = (nxt & ~m) | (((unsigned long long)to << (4 * from)) & m);
    };
    const int mm = cols ^ ((cols >> 1) | (cols & 1) << 3);  // edge k marked: corners k, k + 1 differ
    const bool saddle = mm == 15, one = mm != 0 && !saddle;
    // one segment between the marked edges ea < eb, or on a saddle the cuts of
    // the two corners m0, m0 + 2 whose colour differs from the face's
    const int m0 = (cols & 1) == phif ? 1 : 0, ea = one ? __ffs(mm) - 1 : (m0 + 3) & 3, eb = one ? 31 - __clz(mm) : m0;
    const int arc = one ? (cols >> ((ea + 1) & 3)) & 1 : !phif;
    const int ce_a = edge(ea), ce_b = edge(eb);
    link(arc ? ce_b : ce_a, arc ? ce_a : ce_b, one || saddle);
    const int ce_c = edge((ea + 2) & 3), ce_d = edge((eb + 2) & 3);  // the saddle's other cut
    link(arc ? ce_d : ce_c, arc ? ce_c : ce_d, saddle);
    if (!upper) return 0.0;
    double area = sel01(cols & 1);
    if (one) {
        // corner ea + 1 cut off (eb = ea + 1), corners ea + 1 and ea + 2 (eb =
        // ea + 2), or all but corner 0 (ea = 0, eb = 3: its complement)
        const bool rest = eb == ea + 3, side = eb == ea + 2;
        Fp l1 = sE[ce_a * stride], l2 = sE[ce_b * stride];
        if (ea < 2 && !rest) l1 = 1.0 - l1;
        if (eb >= 2 && !rest) l2 = 1.0 - l2;
        // l1 + l2 or l1 l2, in one operation
        Fp R = half_of(__fma_rn(l1.v, side ? fp_one() : l2.v, side ? l2.v : fp_minus_zero()));
        if (rest) R = 1.0 - R;
        area = arc ? R : 1.0 - R;
    } else if (saddle) {
        Fp T = 0.0;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            if (((cols >> m) & 1) == phif) continue;
            // legs from corner m back along edge m - 1 and on along edge m
            const int p = (m + 3) & 3;
            Fp lp = sE[edge(p) * stride], ln = sE[edge(m) * stride];
            if (p < 2) lp = 1.0 - lp;
            if (m >= 2) ln = 1.0 - ln;
            T += half_of(lp * ln);
        }
        area = phif ? 1.0 - T : T;
    }
    return area;
}

template <int F>
__device__ __forceinline__ double face_of(int K, int phif, const double *sE, int stride, unsigned long long &nxt) {
    constexpr unsigned eds = face_edges(F), cors = face_corners(F);
    return face_area_and_links(eds, cors, F & 1, K, phif, sE, stride, nxt);
}

// edges whose end colours differ
__device__ __forceinline__ unsigned marked_edges(int K) {
    unsigned has = 0;
    const int cx[4] = {0, 2, 4, 6}, cy[4] = {0, 1, 4, 5}, cz[4] = {0, 1, 2, 3};
#pragma unroll
    for (int r = 0; r < 4; r++) {
        has |= (unsigned)(((K >> cx[r]) ^ (K >> (cx[r] + 1))) & 1) << r;
        has |= (unsigned)(((K >> cy[r]) ^ (K >> (cy[r] + 2))) & 1) << (4 + r);
        has |= (unsigned)(((K >> cz[r]) ^ (K >> (cz[r] + 4))) & 1) << (8 + r);
    }
    return has;
}

// the volume from the upper faces' areas and the sum over the loops, clamped to
// [0, 1] by the bit pattern
__device__ __forceinline__ double volume(Fp A1, Fp A2, Fp A3, Fp acc) {
    const double six = 2.0 * ((A1 + A2) + A3) - acc;
    const double V = safe_quotient(six) ? quotient(six, 6.0, 1.0 / 6.0) : six / 6.0;
    const long long b = __double_as_longlong(V);
    if (b < 0 && (b << 1) != 0) return 0.0;
    return b > 0x3FF0000000000000ll ? 1.0 : V;
}
__device__ __forceinline__ double loop_mean(double dot, int len) {
    return safe_quotient(dot) ? quotient(dot, small_count(len), kInverse[len]) : dot / small_count(len);
}

__device__ double cell_fraction_fast(int K, const int Fc[6], const double *sE, int stride, int *bad) {
    unsigned long long nxt = ~0ull;
    face_of<0>(K, Fc[0], sE, stride, nxt);
    const Fp A1 = face_of<1>(K, Fc[1], sE, stride, nxt);
    face_of<2>(K, Fc[2], sE, stride, nxt);
    const Fp A2 = face_of<3>(K, Fc[3], sE, stride, nxt);
    face_of<4>(K, Fc[4], sE, stride, nxt);
    const Fp A3 = face_of<5>(K, Fc[5], sE, stride, nxt);
    const unsigned has = marked_edges(K);
    if (!has) return sel01(K & 1);
    unsigned todo = has;
    Fp acc = 0.0;
    while (todo) {
        const int e0 = __ffs(todo) - 1;
        double sp = sE[e0 * stride];
        const double s0 = sp;
        double px, py, pz;
        marker_xyz(e0, sp, px, py, pz);
        Fp sx = px, sy = py, sz = pz;
        Fp cxs = 0.0, cys = 0.0, czs = 0.0;
        int len = 1, e = e0;
        todo &= ~(1u << e0);
        bool closed = false;
        for (int guard = 0; guard < 12; guard++) {
            const int to = (int)((nxt >> (4 * e)) & 0xF);
            closed = to == e0;
            if (!closed && (to == 0xF || !((todo >> to) & 1))) break;
            const double sq = closed ? s0 : sE[to * stride];
            double qx, qy, qz;
            marker_xyz(to, sq, qx, qy, qz);
            // p x q: the one product of two offsets, the others selected
            const double pq = Fp(sp) * sq;
            const int ap = e >> 2, aq = to >> 2;
            auto mul = [&](double u, double v, int au, int av) -> Fp {
                // u = p's coordinate au, v = q's coordinate av
                const bool us = ap == au, vs = aq == av;
                const double w = us ? u : v;             // the factor that is an offset (or 0, 1)
                const double z = us ? v : u;             // the other one
                return (us && vs) ? pq : (__double2hiint(z) ? w : 0.0);
            };
            cxs += mul(py, qz, 1, 2) - mul(pz, qy, 2, 1);
            cys += mul(pz, qx, 2, 0) - mul(px, qz, 0, 2);
            czs += mul(px, qy, 0, 1) - mul(py, qx, 1, 0);
            if (closed) break;
            sx += qx; sy += qy; sz += qz;
            px = qx; py = qy; pz = qz;
            sp = sq;
            todo &= ~(1u << to);
            e = to;
            len++;
        }
        if (!closed) {
            *bad = 1;
            continue;
        }
        acc += loop_mean(sx * cxs + sy * cys + sz * czs, len);
    }
    return volume(A1, A2, A3, acc);
}

// FP64 pass: one thread per cut cell, full warps.
__global__ void __launch_bounds__(128) f2v_list_kernel(F2VArgs a) {
    __shared__ double sE[12 * 128];
    pdl_wait();
    const int n = *a.ncut;
    unsigned nbad = 0;
    const int stride = gridDim.x * blockDim.x;
    const int iters = (n + stride - 1) / stride;
    double *myE = sE + threadIdx.x;
    for (int it = 0; it < iters; it++) {
        const int t = list_item(it);
        if (t >= n) continue;
        const int id = (int)a.cut[t];
        const int row = (int)((unsigned)id / (unsigned)a.g.n[0]), x = id - row * a.g.n[0];
        const int z = (int)((unsigned)row / (unsigned)a.g.n[1]), y = row - z * a.g.n[1];
        int ids[8];
        cell_ids(a.g, x, y, z, ids);
        int K = 0;
#pragma unroll
        for (int cid = 0; cid < 8; cid++) K |= (__ldg(a.cb + ids[cid]) & 1) << cid;
        const uint8_t b0 = __ldg(a.cb + ids[0]);
        int F[6];
        F[0] = (b0 >> 1) & 1;
        F[1] = (__ldg(a.cb + ids[1]) >> 1) & 1;
        F[2] = (b0 >> 2) & 1;
        F[3] = (__ldg(a.cb + ids[2]) >> 2) & 1;
        F[4] = (b0 >> 3) & 1;
        F[5] = (__ldg(a.cb + ids[4]) >> 3) & 1;
        // x-edges at corners (0,dy,dz), y-edges at (dx,0,dz), z-edges at (dx,dy,0)
        const int cx[4] = {0, 2, 4, 6}, cy[4] = {0, 1, 4, 5}, cz[4] = {0, 1, 2, 3};
#pragma unroll
        for (int r = 0; r < 4; r++) {
            myE[r * 128] = (((K >> cx[r]) ^ (K >> (cx[r] + 1))) & 1) ? __ldg(a.s[0] + ids[cx[r]]) : 0.0;
            myE[(4 + r) * 128] = (((K >> cy[r]) ^ (K >> (cy[r] + 2))) & 1) ? __ldg(a.s[1] + ids[cy[r]]) : 0.0;
            myE[(8 + r) * 128] = (((K >> cz[r]) ^ (K >> (cz[r] + 4))) & 1) ? __ldg(a.s[2] + ids[cz[r]]) : 0.0;
        }
        int bad = 0;
        a.C[id] = cell_fraction_fast(K, F, myE, 128, &bad);
        nbad += bad;
    }
    unsigned v = __reduce_add_sync(0xffffffffu, nbad);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(a.bad, (unsigned long long)v);
}

}  // namespace ebit
