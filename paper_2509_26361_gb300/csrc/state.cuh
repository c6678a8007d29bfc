// state.cuh -- marker initialisation, state read-back and the active band.
#pragma once
#include "band.cuh"
#include "common.cuh"

namespace ebit {

// Marker initialisation (Sec. 3.1): colour = (phi >= 0); on every edge whose end
// colours differ, the marker sits at the linear-interpolation root of phi (or at
// a caller-given offset); saddle faces take the sign of phi at the face centre
// (the mean of the four corners when no face values are given); every other
// face stores its lowest corner's colour.
static __global__ void init_kernel(Grid g, const double *__restrict__ phi, const double *__restrict__ phif,
                            const double *__restrict__ sx, uint8_t *__restrict__ cb,
                            double *__restrict__ s0, double *__restrict__ s1, double *__restrict__ s2) {
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    double *sp[3] = {s0, s1, s2};
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < N; t += (long long)gridDim.x * blockDim.x) {
        int x = (int)(t % g.n[0]);
        int y = (int)((t / g.n[0]) % g.n[1]);
        int z = (int)(t / ((long long)g.n[0] * g.n[1]));
        const int p[3] = {x, y, z};
        const int id = (int)t;
        const double f0 = phi[id];
        const int c0 = f0 >= 0.0;
        int byte = c0;
        for (int a = 0; a < 3; a++) {
            int q[3] = {p[0], p[1], p[2]};
            q[a] += 1;
            int iq = lin3(g, q);
            double f1 = phi[iq];
            int c1 = f1 >= 0.0;
            double v = 0.0;
            if (c0 != c1) {
                double ex = sx ? sx[(long long)a * N + id] : (double)NAN;
                if (ex == ex) v = ex;
                else v = f0 / (f0 - f1);
                if (v < 0.0) v = 0.0;
                if (v > ONE_MINUS) v = ONE_MINUS;
            }
            sp[a][id] = v;
            // face normal to a: corners p, p+e1, p+e2, p+e1+e2 (e1 < e2)
            int e1 = (a == 0) ? 1 : 0, e2 = (a == 2) ? 1 : 2;
            int r1[3] = {p[0], p[1], p[2]}, r2[3] = {p[0], p[1], p[2]}, r3[3] = {p[0], p[1], p[2]};
            r1[e1] += 1;
            r2[e2] += 1;
            r3[e1] += 1;
            r3[e2] += 1;
            int i1 = lin3(g, r1), i2 = lin3(g, r2), i3 = lin3(g, r3);
            int k1 = phi[i1] >= 0.0, k2 = phi[i2] >= 0.0, k3 = phi[i3] >= 0.0;
            int bit = c0;
            if (c0 == k3 && k1 == k2 && c0 != k1) {
                double fc = phif ? phif[(long long)a * N + id]
                                 : 0.25 * ((f0 + phi[i1]) + (phi[i2] + phi[i3]));
                bit = fc >= 0.0;
            }
            byte |= bit << (1 + a);
        }
        cb[id] = (uint8_t)byte;
    }
}

// Marked edges of up to 8 cells of an x-row from the node colours: the cells
// 8 gx .. of row `row` (bits of m[0..2], per edge axis), their first node in
// *id and their number in *cnt (0 past the grid); the cells' colour bytes.
struct RowGroup {
    unsigned m[3];
    int id, cnt;
    unsigned long long bytes;
};
__device__ __forceinline__ RowGroup row_group(const Grid &g, const uint8_t *__restrict__ cb, long long whole, int gx,
                                              long long t) {
    RowGroup r{{0u, 0u, 0u}, 0, 0, 0ull};
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    if (t >= (long long)gx * ny * nz) return r;
    const long long n = (long long)nx * ny * nz;
    // (fewer groups than cells: 32-bit divisions)
    const int row = (int)((unsigned)t / (unsigned)gx), x = 8 * ((int)t - row * gx);
    const int z = row / ny, y = row - z * ny;
    r.id = row * nx + x;
    r.cnt = min(8, nx - x);
    r.bytes = load_colours8(cb, r.id, whole, n);
    const unsigned c = gather_bits(r.bytes);
    const unsigned cy = gather_bits(load_colours8(cb, (long long)(z * ny + wrapc(y + 1, ny)) * nx + x, whole, n));
    const unsigned cz = gather_bits(load_colours8(cb, (long long)(wrapc(z + 1, nz) * ny + y) * nx + x, whole, n));
    const unsigned cn = __ldg(cb + row * nx + wrapc(x + r.cnt, nx)) & 1u;  // the node after the group's last
    const unsigned last = 1u << (r.cnt - 1), ok = (last << 1) - 1u;
    const unsigned up = (c >> 1 & ~last) | (cn ? last : 0u);
    r.m[0] = (c ^ up) & ok;
    r.m[1] = (c ^ cy) & ok;
    r.m[2] = (c ^ cz) & ok;
    return r;
}
__device__ __forceinline__ void store_group(uint8_t *p, unsigned long long v, int cnt) {
    if (cnt == 8 && ((uintptr_t)p & 7) == 0) *reinterpret_cast<unsigned long long *>(p) = v;
    else
        for (int k = 0; k < cnt; k++) p[k] = (uint8_t)(v >> (8 * k));
}

// The markers of the whole grid, one list per edge axis, from the node colours
// (after a state change, in dense mode and in the allocation-free sweep).  One
// thread per 8 cells of an x-row: the row's colours and those of the next rows
// along y and z are 8-bit masks, their exclusive-ors the marked edges; a warp
// reserves its slots with one round of atomics.  list_count[3] starts at zero.
//
// With a source state (cb2 not null) the same pass takes that state in: its
// colours into cb1 and cb2 (both buffers of a context: a sweep leaves tiles
// outside its band unwritten), its offsets on marked edges into s (offsets are
// read only there, and a sweep writes every marker's, so neither the others
// nor the second buffer's are copied).
struct ScanArgs {
    Grid g;
    const uint8_t *cb;
    long long whole;
    unsigned *list[3];
    int *list_count;
    uint8_t *cb1 = nullptr, *cb2 = nullptr;
    const double *src = nullptr;  // [3][n]
    double *s[3] = {nullptr, nullptr, nullptr};
    // zeros into the offsets of an output state, before a sweep writes its markers'
    double *clear = nullptr;      // [3][n]
};
static __global__ void __launch_bounds__(256) mark_scan_kernel(ScanArgs a) {
    pdl_wait();
    const int gx = (a.g.n[0] + 7) / 8;
    const long long n = (long long)a.g.n[0] * a.g.n[1] * a.g.n[2];
    const long long groups = (long long)gx * a.g.n[1] * a.g.n[2];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (a.clear) {
        const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (((uintptr_t)a.clear & 15) == 0) {
            double2 *p = reinterpret_cast<double2 *>(a.clear);
            for (long long k = t; k < 3 * n / 2; k += stride) p[k] = make_double2(0.0, 0.0);
            if (t == 0 && (n & 1)) a.clear[3 * n - 1] = 0.0;
        } else {
            for (long long k = t; k < 3 * n; k += stride) a.clear[k] = 0.0;
        }
    }
    for (long long t0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < groups; t0 += stride) {
        const RowGroup r = row_group(a.g, a.cb, a.whole, gx, t0 + lane);
        if (a.cb2) {
            store_group(a.cb1 + r.id, r.bytes, r.cnt);
            store_group(a.cb2 + r.id, r.bytes, r.cnt);
        }
        if (!__any_sync(full, r.m[0] | r.m[1] | r.m[2])) continue;
        unsigned tot;
        const unsigned pre = warp_prefix(__popc(r.m[0]) | __popc(r.m[1]) << 10 | __popc(r.m[2]) << 20, &tot);
        int base = 0;
        if (lane < 3) {
            const unsigned c = (tot >> (10 * lane)) & 1023u;
            if (c) base = atomicAdd(a.list_count + lane, (int)c);
        }
#pragma unroll
        for (int k = 0; k < 3; k++) {
            int pos = __shfl_sync(full, base, k) + (int)((pre >> (10 * k)) & 1023u);
            for (unsigned w = r.m[k]; w; w &= w - 1) {
                const int id = r.id + __ffs((int)w) - 1;
                a.list[k][pos++] = (unsigned)id;
                if (a.cb2) a.s[k][id] = __ldg(a.src + k * n + id);
            }
        }
    }
}

// The state read back: colour bytes, and the offsets with 0 on edges that carry
// no marker (out_cb may be null: offsets only).  A warp takes 256 cells (32
// groups of up to 8 in a row) and writes each edge axis in 16-byte pieces, lane
// after lane; an offset is read only where its edge carries a marker.  Bound by
// the 24 bytes written per cell.
static __global__ void __launch_bounds__(256) state_out_kernel(Grid g, const uint8_t *__restrict__ cb, long long whole,
                                                               const double *__restrict__ s0,
                                                               const double *__restrict__ s1,
                                                               const double *__restrict__ s2,
                                                               uint8_t *__restrict__ out_cb, double *__restrict__ out) {
    const int gx = (g.n[0] + 7) / 8;
    const long long n = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long groups = (long long)gx * g.n[1] * g.n[2];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < groups; t0 += stride) {
        const RowGroup r = row_group(g, cb, whole, gx, t0 + lane);
        if (out_cb) store_group(out_cb + r.id, r.bytes, r.cnt);
        const unsigned marks = r.m[0] | r.m[1] << 8 | r.m[2] << 16;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int from = 8 * j + (lane >> 2), b = 2 * (lane & 3);
            const unsigned mk = __shfl_sync(full, marks, from) >> b;
            const int cnt = __shfl_sync(full, r.cnt, from), id = __shfl_sync(full, r.id, from) + b;
            if (b >= cnt) continue;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const double *s = k == 0 ? s0 : (k == 1 ? s1 : s2);
                const unsigned m = mk >> (8 * k);
                double v0 = 0.0, v1 = 0.0;
                if (m & 1u) v0 = __ldg(s + id);
                if ((m & 2u) && b + 1 < cnt) v1 = __ldg(s + id + 1);
                double *p = out + k * n + id;
                if (b + 1 < cnt && ((uintptr_t)p & 15) == 0) {
                    *reinterpret_cast<double2 *>(p) = make_double2(v0, v1);
                } else {
                    p[0] = v0;
                    if (b + 1 < cnt) p[1] = v1;
                }
            }
        }
    }
}

// Every tile marked for the next sweep and Front2VOF, the lists of the sweeps
// empty: the tables of a context after a state change (null where it has none).
struct MarkAllArgs {
    int ntiles;
    uint32_t *tile_marker;
    uint8_t *dirty, *clean;  // the tile flags the next Front2VOF takes, and the other set
    uint32_t *band_flag;
    int *band_count, *scan_count;
    // a brick store just unpacked (see background_seams; null otherwise)
    const int *slot = nullptr;
    const uint8_t *bg = nullptr;
    Grid g;
    double *s[3] = {nullptr, nullptr, nullptr};
};

// Offset 0 on the edges between tile t and the next one along axis d (neither in the
// brick store, their colours differ).
static __device__ __noinline__ void background_seam(const Grid &g, int t, int d, double *s) {
    int o[3];
    tile_origin(g, t, o);
    const int l0 = min(o[0] + TILE, g.n[0]) - 1, l1 = min(o[1] + TILE, g.n[1]) - 1, l2 = min(o[2] + TILE, g.n[2]) - 1;
    for (int k = 0; k < TILE * TILE; k++) {
        const int i = k & 7, j = k >> 3;
        const int x = d == 0 ? l0 : o[0] + i, y = d == 1 ? l1 : o[1] + (d == 0 ? i : j), z = d == 2 ? l2 : o[2] + j;
        if (x <= l0 && y <= l1 && z <= l2) s[((long long)z * g.n[1] + y) * g.n[0] + x] = 0.0;
    }
}
static __device__ __forceinline__ void background_seams(const MarkAllArgs &a, int t) {
    const int sy = a.g.td[0], sz = a.g.td[0] * a.g.td[1];
    const int tx = t % sy, r = t / sy, ty = r % a.g.td[1], tz = r / a.g.td[1];
    const int next[3] = {tx + 1 < a.g.td[0] ? t + 1 : t - tx, ty + 1 < a.g.td[1] ? t + sy : t - ty * sy,
                         tz + 1 < a.g.td[2] ? t + sz : t - tz * sz};
    const int own = a.slot[t], colour = a.bg[t];
    bool seam[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const int k = a.slot[next[d]], c = a.bg[next[d]];  // (one round of loads)
        seam[d] = (own & k) < 0 && ((c ^ colour) & 1);
    }
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (seam[d]) background_seam(a.g, t, d, a.s[d]);
}

static __global__ void mark_all_kernel(MarkAllArgs a) {
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x;
    for (int t = t0; t < a.ntiles; t += gridDim.x * blockDim.x) {
        if (a.slot) background_seams(a, t);
        a.tile_marker[t] = 0xFFFFFFFFu;
        a.dirty[t] = 1;
        if (a.clean) a.clean[t] = 0;
        if (a.band_flag) a.band_flag[t] = 0u;
    }
    if (a.band_count && t0 < 2) a.band_count[t0] = 0;
    if (a.scan_count && t0 < 3) a.scan_count[t0] = 0;
}

static __global__ void iota_kernel(int *list, int n, int *count) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) list[t] = t;
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = n;
}

}  // namespace ebit
