// sweep.cuh -- one split advection sweep of the 3D EBIT method.
//
// Method (arxiv 2509.26361): markers move along the sweep axis D by explicit
// Euler with the interpolated velocity (Sec. 2.1, Eqs. 1-2).  Markers on D-edges
// (aligned) stay on their grid line; a node's colour flips once per marker that
// crosses it (Sec. 2.2, Fig. 4); an edge keeps a marker iff its end colours
// differ, so two markers meeting on one edge both vanish (Fig. 5).  Markers on
// the two other edge families (unaligned) are rebuilt in the two face families
// that contain D (Sec. 2.3, Fig. 6): the old polyline of each plane (connectivity
// from the corner colours, and from the face-centre colour on saddle faces) is
// advected, and each unaligned edge whose new end colours differ receives the
// crossing of that polyline with its grid line, refined by two circle fits with
// the radius-ratio rule (Sec. 2.1, Fig. 2).
//
// GPU organisation.  GB300's FP64 pipe is narrow and a warp-level FP64
// instruction costs its issue slots whatever the number of active lanes, so all
// FP64 arithmetic runs from compacted lists with full warps, and the band pass
// over the cells is integer work:
//   mark_scan_kernel -- (state.cuh) after a state change, the markers of the
//                    whole grid listed from the colours.
//   advect_list_kernel -- every listed marker moved once (trilinear velocity):
//                    adv = its advected coordinate along D relative to its node
//                    (s + u dt/h for an aligned marker, u dt/h for an unaligned
//                    one) and bin = floor(2 adv), both in scratch arrays.
//   sweep_kernel  -- (band.cuh) per band tile, integers only: new node colours,
//                    aligned edges, canonical face colours; unaligned edges that
//                    carry a marker, saddle faces and unaligned edges whose
//                    annihilation count needs their crossings go to global
//                    work lists.
//   fp64_kernel   -- one thread per list entry (two per unaligned edge when
//                    the lists are short, the circle fits split between them):
//                    crossings, circle fits, face phases, crossing counts.
// Every crossing decision compares an advected coordinate da + adv with 0 or
// 1/2; for the integers da that occur the sum is exact near those thresholds,
// so "da + adv < 0" equals "bin < -2 da" and "da + adv < 1/2" equals
// "bin < 1 - 2 da" exactly, and the integer test gives the same answer as the
// floating-point one.  Every output word has one owner thread (face bits of
// saddle faces are OR-ed into the byte written by the band pass), and old and
// new state live in separate buffers.
#pragma once
#include "band.cuh"
#include "common.cuh"
#include "sweep_args.cuh"

namespace ebit {

struct P2 {
    Fp x, y;
};

// 2D cell edges in a plane spanned by (a, t): B a-edge at c00, R t-edge at c10,
// T a-edge at c01, L t-edge at c00.
enum { EB = 0, ER = 1, ET = 2, EL = 3 };

// Comparisons on the bit patterns: a floating-point comparison goes through
// the FP64 pipe (2 lanes per clock and SM), which bounds the long lists, and a
// circle fit has ten of them.  For the values that occur the outcomes are the
// IEEE ones: -0 equals 0, and a NaN satisfies neither in_unit nor below_zero.
__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long abs_bits(double v) { return dbits(v) & 0x7FFFFFFFFFFFFFFFull; }
// 0 <= v <= 1
__device__ __forceinline__ bool in_unit(double v) {
    const unsigned long long b = dbits(v);
    return b <= 0x3FF0000000000000ull || b == 0x8000000000000000ull;
}
// v < 0
__device__ __forceinline__ bool below_zero(double v) {
    return dbits(v) - 0x8000000000000001ull <= 0xFFF0000000000000ull - 0x8000000000000001ull;
}
// an offset clamped to [0, 1-]
__device__ __forceinline__ double clamp_offset(double y) {
    if (below_zero(y)) return 0.0;
    return __double_as_longlong(y) > __double_as_longlong(ONE_MINUS) ? ONE_MINUS : y;
}
// 2 v: an exponent increment for a normal number
__device__ __forceinline__ double twice(double v) {
    const unsigned long long b = dbits(v);
    return ((b >> 52) & 0x7FF) ? __longlong_as_double((long long)(b + (1ull << 52))) : 2.0 * v;
}

// Circle through A, B, C meeting the grid line x = 0; only roots on the edge
// (0 <= y <= 1) count, the one nearest ylin is kept (Fig. 2).  rad2 gets the
// squared radius.
__device__ __forceinline__ bool circle_root(P2 A, P2 B, P2 C, double ylin, double *root, double *rad2) {
    const Fp bx = B.x - A.x, by = B.y - A.y;
    const Fp cx = C.x - A.x, cy = C.y - A.y;
    const Fp b2 = bx * bx + by * by;
    const Fp c2 = cx * cx + cy * cy;
    const double det = twice(bx * cy - by * cx);
    if (abs_bits(det) <= dbits(1e-12 * (b2 + c2))) return false;
    const Fp nx = cy * b2 - by * c2, ny = bx * c2 - cx * b2;
    Fp ux, uy;
    // both quotients from one reciprocal
    if (safe_quotient(det) && safe_quotient(nx) && safe_quotient(ny)) {
        const double y = __drcp_rn(det);
        ux = quotient(nx, det, y);
        uy = quotient(ny, det, y);
    } else {
        ux = nx / det;
        uy = ny / det;
    }
    const Fp r2 = ux * ux + uy * uy;
    const Fp dx = A.x + ux;
    const Fp disc = r2 - dx * dx;
    if (below_zero(disc)) return false;
    const Fp sq = sqrt(disc.v);
    const Fp yc = A.y + uy;
    const Fp yp = yc + sq, ym = yc - sq;
    const bool okp = in_unit(yp), okm = in_unit(ym);
    if (!okp && !okm) return false;
    if (okp && okm) *root = (abs_bits(yp - ylin) <= abs_bits(ym - ylin)) ? yp.v : ym.v;
    else *root = okp ? yp.v : ym.v;
    *rad2 = r2;
    return true;
}

// The ratio rule's test rmax > 10 rmin with rmax = sqrt(r2max), rmin =
// sqrt(r2min), both rounded, as the method states it.  Away from the threshold
// the squared radii decide it (r2max against 100 r2min with a relative margin of
// 1e-12, far above the few units of rounding in the radii and the product), so
// the square roots are taken only within that margin.
__device__ __forceinline__ bool ratio_above_10(double r2max, double r2min) {
    const Fp t = 100.0 * Fp(r2min);
    if (dbits(r2max) > dbits(t * (1.0 + 1e-12))) return true;
    if (dbits(r2max) < dbits(t * (1.0 - 1e-12))) return false;
    return sqrt(r2max) > 10.0 * sqrt(r2min);
}

// The crossing of an unaligned edge from the advected points P1 P2 P3 P4
// (P2 -> P3 crosses the edge's grid line at ylin; P1, P4 their neighbours, if
// found): circles through P1 P2 P3 and P2 P3 P4; both valid -> the larger
// circle's root if its radius exceeds 10 times the smaller one, else the mean;
// one valid -> its root; none -> ylin; clamped to [0, 1-] (Fig. 2).  One
// out-of-line copy serves every edge family (the two fits are independent, so
// their FP64 chains interleave inside it).
static __device__ __noinline__ double circle_pair(P2 P1, P2 Pa, P2 Pb, P2 P4, double ylin, bool h1, bool h4) {
    double ya = 0.0, ra2 = 0.0, yb = 0.0, rb2 = 0.0;
    bool va = circle_root(P1, Pa, Pb, ylin, &ya, &ra2);
    bool vb = circle_root(Pa, Pb, P4, ylin, &yb, &rb2);
    va = va && h1;
    vb = vb && h4;
    double y;
    if (va && vb) {
        // above the ratio the radii differ, so the larger squared radius names
        // the larger circle
        const bool a_larger = dbits(ra2) > dbits(rb2);
        if (ratio_above_10(a_larger ? ra2 : rb2, a_larger ? rb2 : ra2)) y = a_larger ? ya : yb;
        else y = 0.5 * (Fp(ya) + yb);
    } else if (va) {
        y = ya;
    } else if (vb) {
        y = yb;
    } else {
        y = ylin;
    }
    return clamp_offset(y);
}

// circle_pair with one fit per lane of a lane pair (adjacent lanes of a warp;
// lane parity `half`: 0 fits P1 Pa Pb, 1 fits Pa Pb P4).  The pair exchanges
// root, squared radius and validity, and both lanes return the crossing
// circle_pair returns (the same operations, in the same order, per fit).
static __device__ __noinline__ double circle_pair_split(P2 P1, P2 Pa, P2 Pb, P2 P4, double ylin, bool h1, bool h4,
                                                        int half) {
    const unsigned pm = 3u << ((threadIdx.x & 31) & ~1u);
    const P2 A = half ? Pa : P1, B = half ? Pb : Pa, Cc = half ? P4 : Pb;
    double y = 0.0, r2 = 0.0;
    bool v = circle_root(A, B, Cc, ylin, &y, &r2);
    v = v && (half ? h4 : h1);
    const double yo = __shfl_xor_sync(pm, y, 1), r2o = __shfl_xor_sync(pm, r2, 1);
    const bool vo = __shfl_xor_sync(pm, (int)v, 1) != 0;
    const double ya = half ? yo : y, ra2 = half ? r2o : r2, yb = half ? y : yo, rb2 = half ? r2 : r2o;
    const bool va = half ? vo : v, vb = half ? v : vo;
    double res;
    if (va && vb) {
        const bool a_larger = dbits(ra2) > dbits(rb2);
        if (ratio_above_10(a_larger ? ra2 : rb2, a_larger ? rb2 : ra2)) res = a_larger ? ya : yb;
        else res = 0.5 * (Fp(ya) + yb);
    } else if (va) {
        res = ya;
    } else if (vb) {
        res = yb;
    } else {
        res = ylin;
    }
    return clamp_offset(res);
}

// trilinear u_D at node q shifted by s along axis e; lerps in x, y, z order
template <int D>
__device__ double interp_u(const Grid &g, const double *__restrict__ u, const int q[3], int e, double s) {
    int base[3];
    Fp t[3];
#pragma unroll
    for (int b = 0; b < 3; b++) {
        if (b == D) {
            base[b] = q[b];
            t[b] = (b == e) ? s : 0.0;
        } else if (b != e) {
            base[b] = q[b] - 1;
            t[b] = 0.5;
        } else if (s < 0.5) {
            base[b] = q[b] - 1;
            t[b] = Fp(s) + 0.5;
        } else {
            base[b] = q[b];
            t[b] = Fp(s) - 0.5;
        }
    }
    int x0 = wrapc(base[0], g.n[0]), x1 = wrapc(base[0] + 1, g.n[0]);
    int y0 = wrapc(base[1], g.n[1]), y1 = wrapc(base[1] + 1, g.n[1]);
    int z0 = wrapc(base[2], g.n[2]), z1 = wrapc(base[2] + 1, g.n[2]);
    int r00 = (z0 * g.n[1] + y0) * g.n[0], r10 = (z0 * g.n[1] + y1) * g.n[0];
    int r01 = (z1 * g.n[1] + y0) * g.n[0], r11 = (z1 * g.n[1] + y1) * g.n[0];
    // A marker off the sweep axis sits on a D-face plane (t[D] = 0): the lerp
    // along D gives (1 - 0) a + 0 b = a for finite b, so its upper samples are
    // not read (for a = -0 the sign of the zero may differ; nothing downstream
    // depends on it).
    const bool flatD = e != D;
    Fp c00, c10, c01, c11;
    if (D == 0 && flatD) {
        c00 = __ldg(u + r00 + x0);
        c10 = __ldg(u + r10 + x0);
        c01 = __ldg(u + r01 + x0);
        c11 = __ldg(u + r11 + x0);
    } else {
        c00 = (1.0 - t[0]) * __ldg(u + r00 + x0) + t[0] * __ldg(u + r00 + x1);
        c10 = (D == 1 && flatD) ? Fp(0.0) : (1.0 - t[0]) * __ldg(u + r10 + x0) + t[0] * __ldg(u + r10 + x1);
        c01 = (D == 2 && flatD) ? Fp(0.0) : (1.0 - t[0]) * __ldg(u + r01 + x0) + t[0] * __ldg(u + r01 + x1);
        c11 = (D != 0 && flatD) ? Fp(0.0) : (1.0 - t[0]) * __ldg(u + r11 + x0) + t[0] * __ldg(u + r11 + x1);
    }
    const Fp c0 = (D == 1 && flatD) ? c00 : (1.0 - t[1]) * c00 + t[1] * c10;
    if (D == 2 && flatD) return c0;
    const Fp c1 = (D == 1 && flatD) ? c01 : (1.0 - t[1]) * c01 + t[1] * c11;
    return (1.0 - t[2]) * c0 + t[2] * c1;
}

// ---------------------------------------------------------------- advection
// the counters the band pass appends to start at zero (cleared by the launch before it)
__device__ __forceinline__ void clear_sweep_counts(const SweepArgs &a) {
    if (blockIdx.x != 0) return;
    if (threadIdx.x < SWEEP_LISTS) a.wcount[threadIdx.x] = 0;
    if (threadIdx.x == 32 && a.mk_out_count) *a.mk_out_count = 0;
    if (threadIdx.x == 33 && a.mt_out_count) *a.mt_out_count = 0;
    if (threadIdx.x == 34 && a.tile_next) *a.tile_next = 0;
    if (threadIdx.x == 35 && a.band_next_count) *a.band_next_count = 0;
}

// Move the marker on the e-edge of node gid once (Eq. 2); the grid's cells start
// at base, u is u_D on its D-faces and lam = dt / h.  CFL >= 1 is counted and
// clamped; a displacement that is not finite (NaN or infinite velocity) is
// counted apart and the marker stays where it is.
template <int D>
__device__ __forceinline__ void move_marker(const SweepArgs &a, const Grid &g, int base, const double *__restrict__ u,
                                            double lam, int e, int gid, unsigned &hits, unsigned &bad) {
    const int nx = g.n[0], nxy = nx * g.n[1], id = gid - base;
    const int z = id / nxy, r = id - z * nxy;
    const int y = r / nx;
    const int q[3] = {r - y * nx, y, z};
    // selects rather than indexing, which would copy the parameter arrays to
    // local memory
    const double *se = e == 0 ? a.s[0] : (e == 1 ? a.s[1] : a.s[2]);
    double *adv = e == 0 ? a.adv[0] : (e == 1 ? a.adv[1] : a.adv[2]);
    int8_t *bin = e == 0 ? a.bin[0] : (e == 1 ? a.bin[1] : a.bin[2]);
    const double sv = __ldg(se + gid);
    double cf = Fp(interp_u<D>(g, u, q, e, sv)) * lam;
    if (!isfinite(cf)) {
        bad++;
        cf = 0.0;
    } else if (!(fabs(cf) < 1.0)) {
        hits++;
        cf = cf > 0.0 ? ONE_MINUS : -ONE_MINUS;
    }
    const double x = (e == D) ? (double)(Fp(sv) + cf) : cf;
    adv[gid] = x;
    bin[gid] = (int8_t)(int)floor(2.0 * x);
}

// Band item b (a direction) of a listed tile of grid g (its tiles start at
// tbase): the neighbour the tile's mask points to that way (bit
// near_bit(dx, dy, dz)), listed once; from tile 0 backwards, past a narrow last
// tile, also the one before it (along each such axis: up to eight tiles).
__device__ __forceinline__ void band_item(const Grid &g, int tbase, int tile, int b, const uint32_t *__restrict__ mask,
                                          uint32_t *band_flag, int *band, int *band_count) {
    if (!((__ldg(mask + tbase + tile) >> b) & 1u)) return;
    const int tx = tile % g.td[0], ty = (tile / g.td[0]) % g.td[1], tz = tile / (g.td[0] * g.td[1]);
    const int dx = b % 3 - 1, dy = (b / 3) % 3 - 1, dz = b / 9 - 1;
    const int bx = wrapc(tx + dx, g.td[0]), by = wrapc(ty + dy, g.td[1]), bz = wrapc(tz + dz, g.td[2]);
    const int ex = dx < 0 && tx == 0 && narrow_last(g, 0), ey = dy < 0 && ty == 0 && narrow_last(g, 1),
              ez = dz < 0 && tz == 0 && narrow_last(g, 2);
    auto take = [&](int x, int y, int z) {
        const int nt = tbase + (z * g.td[1] + y) * g.td[0] + x;
        if (atomicExch(band_flag + nt, 1u) == 0u) band[atomicAdd(band_count, 1)] = nt;
    };
    take(bx, by, bz);
    if (ex | ey | ez)
#pragma unroll 1
        for (int k = 1; k < 8; k++)
            if ((k & 1) <= ex && (k >> 1 & 1) <= ey && (k >> 2) <= ez) take(bx - (k & 1), by - (k >> 1 & 1), bz - (k >> 2));
}

// Advection from the marker lists (Eq. 2): one thread per marker, no tile
// staging.
template <int D>
__global__ void __launch_bounds__(256, 5) advect_list_kernel(SweepArgs a, MarkerLists m) {
    pdl_wait();
    clear_sweep_counts(a);
    // One index space: the markers, then this sweep's band items (tile of the
    // marker-tile list, direction); a thread takes one item per round, so the
    // two kinds of work run side by side rather than one after the other.
    const int n0 = *m.count[0], n1 = *m.count[1], n2 = *m.count[2];
    const int total = n0 + n1 + n2;
    const int nmt = *m.mtiles_count;
    const int all = total + 27 * nmt;
    const int stride = gridDim.x * blockDim.x;
    const int iters = (all + stride - 1) / stride;
    unsigned hits = 0, bad = 0;
    for (int it = 0; it < iters; it++) {
        const int t = list_item(it);
        if (t >= all) continue;
        if (t >= total) {
            const int tb = t - total;
            band_item(a.g, 0, __ldg(m.mtiles + tb / 27), tb % 27, a.tile_marker, a.band_flag, m.band, m.band_count);
            continue;
        }
        const int k = t < n0 ? 0 : (t < n0 + n1 ? 1 : 2);
        const int j = t - (k == 0 ? 0 : (k == 1 ? n0 : n0 + n1));
        const unsigned *lst = k == 0 ? m.list[0] : (k == 1 ? m.list[1] : m.list[2]);
        const int e = k == 0 ? m.axis[0] : (k == 1 ? m.axis[1] : m.axis[2]);
        move_marker<D>(a, a.g, 0, a.u, a.lam, e, (int)__ldg(lst + j), hits, bad);
    }
    unsigned v = __reduce_add_sync(0xffffffffu, hits);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(a.ctr + C_CFL, (unsigned long long)v);
    v = __reduce_add_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(a.ctr + C_NONFINITE, (unsigned long long)v);
}

// ----------------------------------------------------------- cell context
// the integers -2 .. 2 as doubles, by bit patterns (an integer conversion would
// go through the FP64 pipe)
__device__ __forceinline__ double small_double(int q) {
    const int hi = (q & 1) ? 0x3FF00000 : (q ? 0x40000000 : 0);
    return __hiloint2double(hi | (q & 0x80000000), 0);
}

// Segments of a 2D cell by its markers m (bits EB, ER, ET, EL) and, on a saddle,
// whether its lower-left colour equals the face colour: the endpoints of segment
// k in bits 4 k .. 4 k + 3 (first, second), the number of segments in *ns.  The
// order is the oracle's.
__device__ __forceinline__ unsigned seg_codes(unsigned m, bool same, int *ns) {
    if (m == 15u) {
        *ns = 2;
        return same ? (EB | ER << 2 | EL << 4 | ET << 6) : (EB | EL << 2 | ER << 4 | ET << 6);
    }
    *ns = m ? 1 : 0;
    return m ? (unsigned)(__ffs(m) - 1) | (unsigned)(31 - __clz(m)) << 2 : 0u;
}

// A plane of one face family through a node, offsets (da, dt) along (A, T) in
// da [-2, 2], dt [-1, 2], T the family's transverse axis.
// The window's node and face colours are two bit masks, so that segments,
// crossings and polyline neighbours are integer selects: every lane of a warp
// follows one instruction stream whatever its edges, and the marker data is
// read in two rounds of independent loads (the bins that decide the crossings
// come with the colours, then the coordinates of the four points).  With
// branches per edge code and per segment the loads of divergent lanes came one
// after another, up to twenty rounds of L2 latency: a list of a few hundred
// edges took 22 us where this form takes 10 (32^3, one sphere), and one of
// 1.4e5 edges 51 us where it takes 42 (512^3).
template <int D, bool F = false>
struct SweepCell {
    static constexpr int A = D, T1 = (D + 1) % 3, T2 = (D + 2) % 3;
    const SweepArgs &a;
    // the node, and its coordinate, the extent and the stride along A and the
    // transverse axis (T1 for family 0, T2 for family 1).  The family is a
    // run-time value: both share one copy of the code (a short list is bound by
    // instruction fetches as much as by data) and lanes of both run together.
    const int id, fam;
    int pa, pt, na, nt, sa, st;
    // bit (da + 2) + 5 (dt + 1): node colour, and the colour of the node's face
    unsigned col, face;

    // node id_ of grid g, whose cells start at base
    __device__ SweepCell(const SweepArgs &args, const Grid &g, int base, int id_, int fam_)
        : a(args), id(id_), fam(fam_) {
        const int nx = g.n[0], nxy = nx * g.n[1], l = id_ - base, z = l / nxy, r = l - z * nxy, y = r / nx;
        const int p[3] = {r - y * nx, y, z}, s[3] = {1, nx, nxy};
        pa = p[A];
        na = g.n[A];
        sa = s[A];
        pt = fam ? p[T2] : p[T1];
        nt = fam ? g.n[T2] : g.n[T1];
        st = fam ? s[T2] : s[T1];
    }
    // per-family arrays by selects (indexing would copy the arguments to local memory)
    __device__ __forceinline__ const int8_t *bin_t() const { return fam ? a.bin[T2] : a.bin[T1]; }
    __device__ __forceinline__ const double *adv_t() const { return fam ? a.adv[T2] : a.adv[T1]; }
    __device__ __forceinline__ const double *s_t() const { return fam ? a.s[T2] : a.s[T1]; }
    __device__ __forceinline__ double *so_t() const { return fam ? a.so[T2] : a.so[T1]; }
    // node at offset (da, dt)
    __device__ __forceinline__ int pid(int da, int dt) const {
        return id + (wrapc(pa + da, na) - pa) * sa + (wrapc(pt + dt, nt) - pt) * st;
    }
    __device__ __forceinline__ void loadw() {
        unsigned c = 0, f = 0;
        const int fb = 1 + (fam ? T1 : T2);
#pragma unroll
        for (int dt = -1; dt <= 2; dt++)
#pragma unroll
            for (int da = -2; da <= 2; da++) {
                const int i = (da + 2) + 5 * (dt + 1);
                const unsigned b = __ldg(a.cb + pid(da, dt));
                c |= (b & 1u) << i;
                f |= ((b >> fb) & 1u) << i;
            }
        col = c;
        face = f;
    }
    __device__ __forceinline__ static int wi(int da, int dt) { return (da + 2) + 5 * (dt + 1); }
    // markers of cell (da, dt) (bits EB, ER, ET, EL)
    __device__ __forceinline__ unsigned marks(int i) const {
        const unsigned w = col >> i;
        const unsigned c00 = w & 1u, c10 = (w >> 1) & 1u, c01 = (w >> 5) & 1u, c11 = (w >> 6) & 1u;
        return (c00 ^ c10) | (c10 ^ c11) << ER | (c01 ^ c11) << ET | (c00 ^ c01) << EL;
    }
    // does the cell's lower-left colour equal its face's?
    __device__ __forceinline__ bool same(int i) const { return (((col ^ face) >> i) & 1u) == 0u; }
    __device__ __forceinline__ unsigned segs(int da, int dt, int *ns) const {
        const int i = wi(da, dt);
        return seg_codes(marks(i), same(i), ns);
    }

    // Endpoints left of x = 0 per edge code (bits EB, ER, ET, EL) of the cells
    // (-1, 0) and (0, 0), in bits 0-3 and 4-7: x = q + adv < 0 <=> bin < -2 q for
    // the edge's node offset q.  (bins of edges without a marker are read and
    // not used)
    struct Bins {
        int B1, T1, B0, T0, L1, L0, R0;
    };
    __device__ __forceinline__ Bins load_bins() const {
        const int8_t *ba = a.bin[A], *bt = bin_t();
        return Bins{ld_in<F>(ba + pid(-1, 0)), ld_in<F>(ba + pid(-1, 1)), ld_in<F>(ba + pid(0, 0)), ld_in<F>(ba + pid(0, 1)),
                    ld_in<F>(bt + pid(-1, 0)), ld_in<F>(bt + pid(0, 0)),  ld_in<F>(bt + pid(1, 0))};
    }
    __device__ __forceinline__ static unsigned left_bits(const Bins &b) {
        const int bB1 = b.B1, bT1 = b.T1, bB0 = b.B0, bT0 = b.T0, bL1 = b.L1, bL0 = b.L0, bR0 = b.R0;
        const unsigned mid = bL0 < 0;  // the edge between the two cells
        return (unsigned)(bB1 < 2) | mid << ER | (unsigned)(bT1 < 2) << ET | (unsigned)(bL1 < 2) << EL |
               ((unsigned)(bB0 < 0) | (unsigned)(bR0 < -2) << ER | (unsigned)(bT0 < 0) << ET | mid << EL) << 4;
    }
    // number of segments of cells (-1, 0) and (0, 0) crossing x = 0
    __device__ __forceinline__ int count_crossings(unsigned left) const {
        int n = 0;
#pragma unroll
        for (int da = -1; da <= 0; da++) {
            int ns;
            const unsigned sg = segs(da, 0, &ns), lc = left >> (4 * (da + 1));
#pragma unroll
            for (int k = 0; k < 2; k++)
                if (k < ns) n += ((lc >> ((sg >> (4 * k)) & 3)) ^ (lc >> ((sg >> (4 * k + 2)) & 3))) & 1;
        }
        return n;
    }

    // a marker of the window: its node offset (qa, qt) and whether it lies on an
    // A-edge (EB, ET) or a TT-edge (EL, ER)
    struct Mark {
        int qa, qt;
        bool on_a;
    };
    __device__ __forceinline__ static Mark mark(int e, int da, int dt) {
        return Mark{da + (e == ER), dt + (e == ET), (e & 1) == 0};
    }
    // its advected position (x along A, y along TT) relative to the cell's node
    __device__ __forceinline__ P2 pos(const Mark &m) const {
        const int q = pid(m.qa, m.qt);
        const double x = ld_in<F>((m.on_a ? a.adv[A] : adv_t()) + q);
        double s = 0.0;
        if (!m.on_a) s = __ldg(s_t() + q);
        P2 r;
        r.x = Fp(small_double(m.qa)) + x;
        r.y = Fp(small_double(m.qt)) + s;
        return r;
    }
    // the marker next along the polyline beyond edge e of cell (da, dt), in the
    // cell across that edge; false when that cell has no segment ending on it
    __device__ __forceinline__ bool next_mark(int e, int da, int dt, Mark *out) const {
        const int oda = da + (e == ER) - (e == EL), odt = dt + (e == ET) - (e == EB);
        const int oe = e ^ 2;  // the same edge seen from there: EB <-> ET, EL <-> ER
        const int i = wi(oda, odt);
        const unsigned m = marks(i);
        const unsigned rest = m & ~(1u << oe);
        // two markers: the other one; a saddle: EB-ER, EL-ET or EB-EL, ER-ET
        const int other = m == 15u ? (same(i) ? oe ^ 1 : 3 - oe) : __ffs(rest) - 1;
        *out = mark(other & 3, oda, odt);
        return ((m >> oe) & 1u) && rest;
    }

    // Crossings of the advected polyline of cells (-1, 0) and (0, 0) with the
    // grid line x = 0, in scan order (cell da = -1 then 0, segment 0 then 1):
    // their number, and for the first three their left and right endpoint
    // edges and cell (scalars, so that nothing lives in local memory).
    struct Crossings {
        int n;
        int el0, er0, da0, el1, er1, da1, el2, er2, da2;
    };
    __device__ __forceinline__ Crossings crossings(unsigned left) const {
        Crossings c{};
#pragma unroll
        for (int da = -1; da <= 0; da++) {
            int ns;
            const unsigned sg = segs(da, 0, &ns), lc = left >> (4 * (da + 1));
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int e0 = (sg >> (4 * k)) & 3, e1 = (sg >> (4 * k + 2)) & 3;
                const bool l0 = (lc >> e0) & 1u, l1 = (lc >> e1) & 1u;
                if (k >= ns || l0 == l1) continue;
                const int el = l0 ? e0 : e1, er = l0 ? e1 : e0;
                if (c.n == 0) { c.el0 = el; c.er0 = er; c.da0 = da; }
                else if (c.n == 1) { c.el1 = el; c.er1 = er; c.da1 = da; }
                else if (c.n == 2) { c.el2 = el; c.er2 = er; c.da2 = da; }
                c.n++;
            }
        }
        return c;
    }
    // linear crossing height of the segment Pa Pb with x = 0
    __device__ __forceinline__ static double crossing_line(const P2 &Pa, const P2 &Pb) {
        const Fp tt = (0.0 - Pa.x) / (Pb.x - Pa.x);
        return Pa.y + tt * (Pb.y - Pa.y);
    }
    __device__ __forceinline__ double crossing_height(int el, int er, int cda) const {
        return crossing_line(pos(mark(el, cda, 0)), pos(mark(er, cda, 0)));
    }

    // Unaligned edge of the family at the cell's node (carries a marker):
    // crossings of the advected polyline with the grid line x = 0 in strip 0
    // (Fig. 1c), then the two circle fits with the ratio rule (Fig. 2).
    // half: -1 one lane per edge; 0, 1 the lanes of a pair sharing the edge
    // (the even lane counts and stores).
    __device__ __forceinline__ void unaligned(unsigned left, unsigned ev[C_N], int half = -1) const {
        const Crossings c = crossings(left);
        const bool lead = half <= 0;
        if ((c.n & 1) == 0) {
            if (lead) {
                ev[C_INCONSISTENT]++;
                so_t()[id] = 0.5;
            }
            return;
        }
        int el = c.el0, er = c.er0, cda = c.da0;
        if (c.n == 3) {
            // a fold of the polyline: the crossing with the median linear
            // height, by the same three compare-exchanges as the oracle
            // (v_k tracks yl[o_k], so the comparisons are the oracle's)
            double v0 = crossing_height(c.el0, c.er0, c.da0), v1 = crossing_height(c.el1, c.er1, c.da1),
                   v2 = crossing_height(c.el2, c.er2, c.da2), tv;
            int o0 = 0, o1 = 1, o2 = 2, tmp;
            if (v0 > v1) { tmp = o0; o0 = o1; o1 = tmp; tv = v0; v0 = v1; v1 = tv; }
            if (v1 > v2) { tmp = o1; o1 = o2; o2 = tmp; tv = v1; v1 = v2; v2 = tv; }
            if (v0 > v1) { tmp = o0; o0 = o1; o1 = tmp; tv = v0; v0 = v1; v1 = tv; }
            if (o1 == 1) { el = c.el1; er = c.er1; cda = c.da1; }
            else if (o1 == 2) { el = c.el2; er = c.er2; cda = c.da2; }
            if (lead) ev[C_MULTI]++;
        }
        // the crossing segment and its neighbours along the polyline (their own
        // ends where there is none), all loads together, then the two fits
        const Mark ma = mark(el, cda, 0), mb = mark(er, cda, 0);
        Mark m1, m4;
        const bool h1 = next_mark(el, cda, 0, &m1), h4 = next_mark(er, cda, 0, &m4);
        if (!h1) m1 = ma;
        if (!h4) m4 = mb;
        const P2 Pa = pos(ma), Pb = pos(mb), P1 = pos(m1), P4 = pos(m4);
        const double ylin = crossing_line(Pa, Pb);
        if (lead && !h1) ev[C_INCONSISTENT]++;
        if (lead && !h4) ev[C_INCONSISTENT]++;
        if (half < 0) {
            so_t()[id] = circle_pair(P1, Pa, Pb, P4, ylin, h1, h4);
        } else {
            const double y = circle_pair_split(P1, Pa, Pb, P4, ylin, h1, h4, half);
            if (lead) so_t()[id] = y;
        }
    }

    // is the endpoint on edge e of cell (da, dt) left of x = 1/2?
    __device__ __forceinline__ bool left_of_half(int e, int da, int dt) const {
        const Mark m = mark(e, da, dt);
        const int b = ld_in<F>((m.on_a ? a.bin[A] : bin_t()) + pid(m.qa, m.qt));
        return b < 1 - 2 * m.qa;
    }
    // Face-centre colour of the family's 2D cell at the node (saddle faces): the
    // phase of the advected polyline at the centre, reached from the node along
    // the a-line to x = 1/2 and then up the line x = 1/2 to y = 1/2.
    __device__ int face_phase(int ncol0) const {
        int par = ncol0;
        for (int da = -1; da <= 1; da++) {
            const int i = wi(da, 0);
            if (((col >> i) & 1u) == ((col >> (i + 1)) & 1u)) continue;
            int b = ld_in<F>(a.bin[A] + pid(da, 0));
            if (b >= -2 * da && b < 1 - 2 * da) par ^= 1;
        }
        for (int da = -1; da <= 1; da++) {
            int ns;
            const unsigned sg = segs(da, 0, &ns);
            for (int k = 0; k < ns; k++) {
                const int e0 = (sg >> (4 * k)) & 3, e1 = (sg >> (4 * k + 2)) & 3;
                bool l0 = left_of_half(e0, da, 0), l1 = left_of_half(e1, da, 0);
                if (l0 == l1) continue;
                P2 L = pos(mark(l0 ? e0 : e1, da, 0));
                P2 R = pos(mark(l0 ? e1 : e0, da, 0));
                const Fp tt = (0.5 - L.x) / (R.x - L.x);
                const double yl = L.y + tt * (R.y - L.y);
                if (yl < 0.5) par ^= 1;
            }
        }
        return par;
    }
};

// ------------------------------------------------- FP64 work lists
// Entry of list `kind` (0, 1: unaligned edges of families 1, 2; 2, 3: saddle
// faces; 4, 5: annihilation checks): node id of grid g, whose cells start at base.
template <int D, bool F>
__device__ __forceinline__ void fp64_item(const SweepArgs &a, const Grid &g, int base, int kind, int id, unsigned ev[C_N],
                                          int half = -1) {
    constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
    SweepCell<D, F> cell(a, g, base, id, kind & 1);
    const auto bins = cell.load_bins();  // (with the colours: one wait for both)
    cell.loadw();
    const unsigned left = cell.left_bits(bins);
    if (kind >= 4) {
        // an even number (>= 2) of advected crossings met on an edge that keeps
        // no marker (Fig. 5)
        if (cell.count_crossings(left) >= 2) ev[C_ANNIHILATE]++;
    } else if (kind < 2) {
        cell.unaligned(left, ev, half);
    } else {
        int ncol0 = ld_in<F>(a.cbo + id) & 1;
        const int bit = cell.face_phase(ncol0) << (1 + (kind == 2 ? T2 : T1));
        if (bit) {
            uintptr_t addr = (uintptr_t)(a.cbo + id);
            unsigned *w = (unsigned *)(addr & ~(uintptr_t)3);
            atomicOr(w, (unsigned)bit << (8 * (addr & 3)));
        }
    }
}

// The work lists of a sweep as one index space of lanes.  Unaligned edges come
// first, then saddle faces and annihilation checks, one lane each.  When the
// lists fit one round of `stride` lanes with two per unaligned edge, each edge
// gets two adjacent lanes and the circle fits are split between them: a shorter
// chain per warp where few warps run.  Long lists keep one lane per edge, since
// the pairs repeat the work before the fits.
template <bool F>
struct WorkLanes {
    int n[SWEEP_LISTS], lanes_u, lanes;
    bool pairs;
    __device__ WorkLanes(const SweepArgs &a, int stride) {
#pragma unroll
        for (int k = 0; k < SWEEP_LISTS; k++) n[k] = ld_in<F>(a.wcount + k);
        const int nu = n[0] + n[1], rest = n[2] + n[3] + n[4] + n[5];
        pairs = 2 * nu + rest <= stride;
        lanes_u = pairs ? 2 * nu : nu;
        lanes = lanes_u + rest;
    }
    // lane t's list and node, and its half of the edge (-1: all of it)
    __device__ __forceinline__ int item(const SweepArgs &a, int t, int *kind, int *half) const {
        *half = -1;
        if (t < lanes_u) {
            if (pairs) {
                *half = t & 1;
                t >>= 1;
            }
        } else {
            t += n[0] + n[1] - lanes_u;
        }
        int k = 0;
#pragma unroll
        for (int q = 0; q < SWEEP_LISTS - 1; q++)
            if (k == q && t >= n[q]) {
                t -= n[q];
                k = q + 1;
            }
        *kind = k;
        // the checks fill the unaligned lists' arrays from the end
        const unsigned *w = (k & 1) ? ((k & 2) ? a.work[3] : a.work[1]) : ((k & 2) ? a.work[2] : a.work[0]);
        return (int)ld_in<F>(k < 4 ? w + t : w + (a.cells - 1 - t));
    }
};

template <int D>
__global__ void __launch_bounds__(128, 8) fp64_kernel(SweepArgs a) {
    pdl_wait();
    unsigned ev[C_N] = {0, 0, 0, 0, 0};
    const int stride = gridDim.x * blockDim.x;
    const WorkLanes<false> w(a, stride);
    // (the trip count is uniform so that every lane reaches the warp reductions)
    const int iters = (w.lanes + stride - 1) / stride;
    for (int it = 0; it < iters; it++) {
        const int t = list_item(it);
        if (t >= w.lanes) continue;
        int kind, half;
        const int id = w.item(a, t, &kind, &half);
        fp64_item<D, false>(a, a.g, 0, kind, id, ev, half);
    }
#pragma unroll
    for (int k = 0; k < C_N; k++) {
        if (k == C_MARKERS || k == C_CFL) continue;  // counted by the band pass and the advection
        unsigned v = __reduce_add_sync(0xffffffffu, ev[k]);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(a.ctr + k, (unsigned long long)v);
    }
}

}  // namespace ebit
