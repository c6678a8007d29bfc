// hf.cuh -- height-function curvature from volume fractions.
//
// The paper computes curvature from the Front2VOF volume fractions with the
// (generalised) height-function method (Sec. 2.6).  This kernel is the standard
// form: for an interface cell (0 < C < 1) the normal n = -grad C is taken from
// the 3x3x3 block with 1-2-1 weights; along the axis of largest |n_d| (ties to
// the lower axis) the heights of a 3x3 stencil of 9-cell columns are summed; a
// column is valid when its end on the reference-phase side is full (C = 1) and
// the other end empty (C = 0).  From the heights eta,
//   kappa h = -sign(n_d) [(1+h_y^2) h_xx + (1+h_x^2) h_yy - 2 h_x h_y h_xy]
//             / (1 + h_x^2 + h_y^2)^(3/2)
// with centred differences; if a column is invalid the next axis by |n| is
// tried, and with none the status is NO_HF (no paraboloid fit).
#pragma once
#include "band.cuh"
#include "common.cuh"

namespace ebit {

constexpr int HFH = 4;  // column half-length: 9 cells

struct HFArgs {
    Grid g;
    const double *__restrict__ C;
    double *__restrict__ kh;
    uint8_t *__restrict__ st;
    const unsigned *__restrict__ prev;  // interface cells of the previous call
    const int *__restrict__ nprev;
    const unsigned *__restrict__ cand;  // candidate cells (all interface cells are among them)
    const int *__restrict__ ncand;
    unsigned *__restrict__ iface;       // interface cells of this call (output list, may be null)
    int *__restrict__ niface;
    int *zero[2];                       // counters of later launches to clear (may be null)
};

// 0 < C < 1 on the bit pattern (C is never negative; -0 and NaN fail as in IEEE)
__device__ __forceinline__ bool is_interface(double c) {
    long long b = __double_as_longlong(c);
    return b > 0 && b < 0x3FF0000000000000ll;
}

// The cell's neighbourhood: offsets along one axis are wrapped by two selects, so
// cells at a periodic seam run the same code as the others.
struct HFCell {
    const double *__restrict__ C;
    int p[3], n[3], s[3];  // coordinates, extents, strides
    int id;

    __device__ HFCell(const double *C_, const Grid &g, int id_) : C(C_), id(id_) {
        n[0] = g.n[0];
        n[1] = g.n[1];
        n[2] = g.n[2];
        s[0] = 1;
        s[1] = n[0];
        s[2] = n[0] * n[1];
        p[2] = id / s[2];
        const int r = id - p[2] * s[2];
        p[1] = r / n[0];
        p[0] = r - p[1] * n[0];
    }
    // id offset of m cells along an axis (coordinate q, extent nn, stride st)
    __device__ __forceinline__ static int off(int q, int nn, int st, int m) { return (wrapc(q + m, nn) - q) * st; }
};

// The float at or below c for c in [+0, 1], from the bit pattern (values
// under 2^-126 give 0): an error below one float ulp, at most 2^-24.
__device__ __forceinline__ float trunc_unit_float(double c) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(c);
    const int e = (int)(b >> 52);
    const unsigned f = ((unsigned)(e - 1023 + 127) << 23) | (unsigned)((b >> 29) & 0x7FFFFFull);
    return e < 1023 - 126 ? 0.0f : __uint_as_float(f);
}

// axes in the order they are tried (bits 0-5, two each) and, in bits 6-8, the
// axes with n > 0 (reference phase below)
template <typename T>
__device__ __forceinline__ int hf_order(T n0, T n1, T n2) {
    const T a0 = n0 < T(0) ? -n0 : n0, a1 = n1 < T(0) ? -n1 : n1, a2 = n2 < T(0) ? -n2 : n2;
    int o0 = 0, o1 = 1, o2 = 2, tmp;
    T f0 = a0, f1 = a1, f2 = a2, t;
    if (f1 > f0) { tmp = o0; o0 = o1; o1 = tmp; t = f0; f0 = f1; f1 = t; }
    if (f2 > f1) {
        tmp = o1; o1 = o2; o2 = tmp; t = f1; f1 = f2; f2 = t;
        if (f1 > f0) { tmp = o0; o0 = o1; o1 = tmp; }
    }
    return o0 | o1 << 2 | o2 << 4 | (n0 > T(0) ? 64 : 0) | (n1 > T(0) ? 128 : 0) | (n2 > T(0) ? 256 : 0);
}

// The order by the FP64 normal, Youngs sums in the order (b2 outer, b1 inner):
// the rare cells whose float normal does not decide.
static __device__ __noinline__ int hf_order_exact(const double *__restrict__ C, int id, const int *ox, const int *oy,
                                                  const int *oz) {
    double n[3];
    const double w[3] = {1.0, 2.0, 1.0};
    for (int d = 0; d < 3; d++) {
        double gsum = 0.0;
        for (int b2 = 0; b2 < 3; b2++)
            for (int b1 = 0; b1 < 3; b1++) {
                // the block's cells at +1 and -1 along d, b1 and b2 along the other two axes
                const int up = d == 0 ? ox[2] + oy[b1] + oz[b2] : (d == 1 ? ox[b1] + oy[2] + oz[b2] : ox[b1] + oy[b2] + oz[2]);
                const int dn = d == 0 ? ox[0] + oy[b1] + oz[b2] : (d == 1 ? ox[b1] + oy[0] + oz[b2] : ox[b1] + oy[b2] + oz[0]);
                gsum += (w[b1] * w[b2]) * (__ldg(C + id + up) - __ldg(C + id + dn));
            }
        n[d] = -gsum;
    }
    return hf_order<double>(n[0], n[1], n[2]);
}

// A value in [+0, 1] (bit pattern b) in units of 2^-58, cut off below.
__device__ __forceinline__ long long unit_fixed(unsigned long long b) {
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) << 6 | 1ull << 58;  // of a value in [1, 2)
    return (long long)(m >> min(1023 - (int)(b >> 52), 63));                   // (0 from exponent 0)
}
// v 2^-s rounded to the nearest double, ties to even
__device__ __forceinline__ double fixed_double(long long v, int s) {
    unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    if (a == 0) return 0.0;
    const int lead = __clzll((long long)a);
    a <<= lead;  // the leading one at bit 63
    // 53 bits kept; a carry out of the fraction raises the exponent
    const unsigned long long t = (a >> 11) + (((a >> 10) & 1ull) & (((a & 0x3FFull) != 0) | ((a >> 11) & 1ull)));
    const unsigned long long e = (unsigned long long)(1023 + 63 - s - lead);
    return __longlong_as_double((long long)((((unsigned long long)v >> 63) << 63) | ((e << 52) + (t - (1ull << 52)))));
}

// Height-function curvature of an interface cell: its status, and kappa h in
// *out.
//
// The axis is chosen first, by integer tests of the columns' ends alone: the
// ends of the 3x3 columns along the axis must be pure with the reference phase
// on the expected side.  The heights are then summed once, for the one axis that
// has them.  Every lane of a warp follows one instruction stream (wrapped
// offsets, the axis a run-time value, one path for both ways of ordering the
// axes): with separate code for cells at the seams, for each way of ordering and
// a whole sum per axis tried, a warp ran up to twelve sums one after another.
// The FP64 units (2 lanes per clock and SM) take about 32 operations per cell with
// heights, for the formula; its columns' 72 additions and their differences run as
// integers.  3.0e5 cells at 256^3 took 286 us, with the additions in FP64 88, and
// take 62, bound by integer issue and the gathers (issue slots 42 % busy, the FP64
// pipe 26 %); the error against 64-bit references fell
// from 8.3e-15 to 7e-15.
__device__ __forceinline__ int hf_cell(const HFCell &c, double *out) {
    int ox[3], oy[3], oz[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        ox[i] = HFCell::off(c.p[0], c.n[0], c.s[0], i - 1);
        oy[i] = HFCell::off(c.p[1], c.n[1], c.s[1], i - 1);
        oz[i] = HFCell::off(c.p[2], c.n[2], c.s[2], i - 1);
    }
    // The normal decides only the axis order and the side of the reference
    // phase.  A float normal decides them when every |n_d| and every gap
    // between two |n_d| clears the float rounding bound CANON_EPS with margin
    // (then the FP64 sums, within 2e-14 of the exact ones, order and sign them
    // the same); otherwise the FP64 sums, in the oracle's order.
    // (the bound holds for values in [+0, 1], checked on the bit patterns).
    // The floats are the doubles truncated by integer operations, not rounded
    // by conversion instructions: an input error below 2^-24 instead of 2^-25,
    // which raises the bound from 1.7e-5 to 1.8e-5, still under CANON_EPS.
    float fv[27];
    bool unit = true;
#pragma unroll
    for (int i = 0; i < 27; i++) {
        const double v = __ldg(c.C + c.id + ox[i % 3] + oy[(i / 3) % 3] + oz[i / 9]);
        unit = unit && (unsigned long long)__double_as_longlong(v) <= 0x3FF0000000000000ull;
        fv[i] = trunc_unit_float(v);
    }
    float nf[3];
    youngs<float>(fv, nf);
    const float f0 = fabsf(nf[0]), f1 = fabsf(nf[1]), f2 = fabsf(nf[2]);
    int ord;
    if (unit && f0 > CANON_EPS && f1 > CANON_EPS && f2 > CANON_EPS && fabsf(f0 - f1) > 2.0f * CANON_EPS &&
        fabsf(f0 - f2) > 2.0f * CANON_EPS && fabsf(f1 - f2) > 2.0f * CANON_EPS)
        ord = hf_order<float>(nf[0], nf[1], nf[2]);
    else
        ord = hf_order_exact(c.C, c.id, ox, oy, oz);
    // the first axis whose columns end pure, the reference phase below (above)
    int axis = -1, q = 0, nn = 0, st = 0, t1[3], t2[3];
    for (int k = 0; k < 3 && axis < 0; k++) {
        const int d = (ord >> (2 * k)) & 3;
        q = d == 0 ? c.p[0] : (d == 1 ? c.p[1] : c.p[2]);
        nn = d == 0 ? c.n[0] : (d == 1 ? c.n[1] : c.n[2]);
        st = d == 0 ? c.s[0] : (d == 1 ? c.s[1] : c.s[2]);
#pragma unroll
        for (int i = 0; i < 3; i++) {
            t1[i] = d == 0 ? oy[i] : ox[i];
            t2[i] = d == 2 ? oy[i] : oz[i];
        }
        const int lo = c.id + HFCell::off(q, nn, st, -HFH), hi = c.id + HFCell::off(q, nn, st, HFH);
        const bool below = (ord >> (6 + d)) & 1;
        bool ok = true;
#pragma unroll
        for (int b2 = 0; b2 < 3; b2++)
#pragma unroll
            for (int b1 = 0; b1 < 3; b1++) {
                // == 1.0 is one pattern, == 0.0 two (+0, -0)
                const unsigned long long l = (unsigned long long)__double_as_longlong(__ldg(c.C + lo + t1[b1] + t2[b2]));
                const unsigned long long h = (unsigned long long)__double_as_longlong(__ldg(c.C + hi + t1[b1] + t2[b2]));
                const unsigned long long f = below ? l : h, e = below ? h : l;
                ok = ok && f == 0x3FF0000000000000ull && (e << 1) == 0ull;
            }
        if (ok) axis = d;
    }
    if (axis < 0) {
        *out = 0.0;
        return 4;
    }
    // heights: the sum of a column's values in [+0, 1] as integers in units of 2^-58
    // (a value's bits below that are cut off); the differences are exact, with
    // one rounding to a double; of other values, in FP64
    const bool below = (ord >> (6 + axis)) & 1;
    int om[9];
#pragma unroll
    for (int m = 0; m < 9; m++) om[m] = HFCell::off(q, nn, st, m - HFH);
    long long e[3][3];
    bool fixed = true;
#pragma unroll
    for (int b2 = 0; b2 < 3; b2++)
#pragma unroll
        for (int b1 = 0; b1 < 3; b1++) {
            const double *col = c.C + c.id + t1[b1] + t2[b2];
            long long H = 0;
            // (the ends are 0 and 1 in every column: left out of the differences)
#pragma unroll
            for (int m = 1; m < 8; m++) {
                const unsigned long long b = (unsigned long long)__double_as_longlong(__ldg(col + om[m]));
                fixed = fixed && b <= 0x3FF0000000000000ull;
                H += unit_fixed(b);
            }
            e[b1][b2] = below ? H : -H;
        }
    Fp hx, hy, hxx, hyy, hxy;
    if (fixed) {
        hx = fixed_double(e[2][1] - e[0][1], 59);
        hy = fixed_double(e[1][2] - e[1][0], 59);
        hxx = fixed_double(e[2][1] + e[0][1] - 2 * e[1][1], 58);
        hyy = fixed_double(e[1][2] + e[1][0] - 2 * e[1][1], 58);
        hxy = fixed_double((e[2][2] - e[2][0]) - (e[0][2] - e[0][0]), 60);
    } else {
        double eta[3][3];
#pragma unroll
        for (int b2 = 0; b2 < 3; b2++)
#pragma unroll
            for (int b1 = 0; b1 < 3; b1++) {
                const double *col = c.C + c.id + t1[b1] + t2[b2];
                double H = __ldg(col + om[0]);
#pragma unroll
                for (int m = 1; m < 9; m++) H += __ldg(col + om[m]);
                eta[b1][b2] = (below ? H : HFH + 0.5) - (below ? HFH + 0.5 : H);
            }
        hx = (eta[2][1] - eta[0][1]) * 0.5;
        hy = (eta[1][2] - eta[1][0]) * 0.5;
        hxx = (eta[2][1] + eta[0][1]) - 2.0 * eta[1][1];
        hyy = (eta[1][2] + eta[1][0]) - 2.0 * eta[1][1];
        hxy = ((eta[2][2] - eta[2][0]) - (eta[0][2] - eta[0][0])) * 0.25;
    }
    const Fp num = (1.0 + hy * hy) * hxx + (1.0 + hx * hx) * hyy - 2.0 * hx * hy * hxy;
    const Fp q2 = 1.0 + hx * hx + hy * hy;
    const double kap = num / (q2 * sqrt(q2.v));
    *out = below ? -kap : kap;
    return 1 + axis;
}

// Interface-cell pass: entries [0, nprev) reset the previous interface cells
// that are no longer cut (their curvature becomes 0, status NONE); entries of
// the candidate list are computed if 0 < C < 1 and reset otherwise.  Every
// interface cell of the current C is a candidate, so the curvature field is
// complete; one thread per entry, full warps for the FP64 work.  Without
// COMPUTE the interface cells are only listed (the learned curvature writes
// them next).
// 4 blocks of 128 per SM (128 registers without spilling)
template <bool COMPUTE>
__global__ void __launch_bounds__(128, 4) hf_list_kernel(HFArgs a) {
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (a.zero[0]) *a.zero[0] = 0;
        if (a.zero[1]) *a.zero[1] = 0;
    }
    const int np = *a.nprev, nc = *a.ncand;
    const int total = np + nc;
    const int stride = gridDim.x * blockDim.x;
    const int iters = (total + stride - 1) / stride;
    for (int it = 0; it < iters; it++) {
        const int t = list_item(it);
        bool keep = false;
        int id = 0;
        if (t < total) {
            id = (int)(t < np ? a.prev[t] : a.cand[t - np]);
            bool iface = is_interface(__ldg(a.C + id));
            if (t < np) {
                if (!iface) {
                    a.kh[id] = 0.0;
                    a.st[id] = 0;
                }
            } else if (iface) {
                if (COMPUTE) {
                    double kv = 0.0;
                    const int st = hf_cell(HFCell(a.C, a.g, id), &kv);
                    a.kh[id] = kv;
                    a.st[id] = (uint8_t)st;
                }
                keep = true;
            } else {
                a.kh[id] = 0.0;
                a.st[id] = 0;
            }
        }
        const unsigned full = 0xffffffffu;
        unsigned m = __ballot_sync(full, keep);
        if (m && a.iface) {
            const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
            int base = 0;
            if (lane == leader) base = atomicAdd(a.niface, __popc(m));
            base = __shfl_sync(full, base, leader);
            if (keep) a.iface[base + __popc(m & ((1u << lane) - 1u))] = (unsigned)id;
        }
    }
}

// Full scan of any C: curvature 0 and status NONE in every cell, and the
// interface cells listed (the passes after this one write those).
//
// A block takes a brick of 64 x 8 x 8 cells, a warp a row of 64 at a time, 16
// bytes per lane: 17 bytes per cell from and to HBM in whole lines.  The
// interface cells are kept as one bit mask per row and listed by 8^3 tiles, so
// that consecutive entries share the neighbourhoods the later passes gather (a
// list in row order costs those more than the scan gains).  Reading tile rows of
// 64 bytes instead, the scan of 256^3 took 68 us; this form takes 46.
constexpr int SCAN_X = 64;
static __global__ void __launch_bounds__(256) hf_scan_kernel(Grid g, const double *__restrict__ C, double *__restrict__ kh,
                                                             uint8_t *__restrict__ st, unsigned *__restrict__ list,
                                                             int *__restrict__ count, int *__restrict__ zero0,
                                                             int *__restrict__ zero1) {
    __shared__ unsigned char s_bits[64][8];  // [row of the brick][8-cell tile along x]
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (zero0) *zero0 = 0;
        if (zero1) *zero1 = 0;
    }
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
    const int bx = (nx + SCAN_X - 1) / SCAN_X;
    const long long bricks = (long long)bx * g.td[1] * g.td[2];
    const unsigned full = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // rows of every array start on 16-byte boundaries (the status bytes on 2)
    const bool pairs = nx % 2 == 0 && (((uintptr_t)C | (uintptr_t)kh) & 15) == 0 && ((uintptr_t)st & 1) == 0;
    for (long long br = blockIdx.x; br < bricks; br += gridDim.x) {
        const int ix = (int)(br % bx), iyz = (int)(br / bx);
        const int x0 = ix * SCAN_X, y0 = (iyz % g.td[1]) * 8, z0 = (iyz / g.td[1]) * 8;
        const int x = x0 + 2 * lane;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int r = warp + 8 * q, y = y0 + (r & 7), z = z0 + (r >> 3);
            bool i0 = false, i1 = false;
            if (y < ny && z < nz && x < nx) {
                const long long id = ((long long)z * ny + y) * nx + x;
                if (pairs) {
                    const double2 c = __ldg(reinterpret_cast<const double2 *>(C + id));
                    i0 = is_interface(c.x);
                    i1 = is_interface(c.y);
                    *reinterpret_cast<double2 *>(kh + id) = make_double2(0.0, 0.0);
                    *reinterpret_cast<uint16_t *>(st + id) = 0;
                } else {
                    i0 = is_interface(__ldg(C + id));
                    kh[id] = 0.0;
                    st[id] = 0;
                    if (x + 1 < nx) {
                        i1 = is_interface(__ldg(C + id + 1));
                        kh[id + 1] = 0.0;
                        st[id + 1] = 0;
                    }
                }
            }
            // lane l holds cells 2 l, 2 l + 1: a tile's 8 cells are 4 lanes
            const unsigned b0 = __ballot_sync(full, i0), b1 = __ballot_sync(full, i1);
            if (lane < 8) {
                const unsigned e = (b0 >> (4 * lane)) & 15u, o = (b1 >> (4 * lane)) & 15u;
                unsigned m = 0;
#pragma unroll
                for (int k = 0; k < 4; k++) m |= ((e >> k) & 1u) << (2 * k) | ((o >> k) & 1u) << (2 * k + 1);
                s_bits[r][lane] = (unsigned char)m;
            }
        }
        __syncthreads();
        // warp w lists tile w of the brick, two rows per lane
        {
            const unsigned m0 = s_bits[2 * lane][warp], m1 = s_bits[2 * lane + 1][warp];
            if (__any_sync(full, m0 | m1)) {
                unsigned total;
                int pos = (int)warp_prefix(__popc(m0) + __popc(m1), &total);
                int base = 0;
                if (lane == 0) base = atomicAdd(count, (int)total);
                pos += __shfl_sync(full, base, 0);
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const int r = 2 * lane + q;
                    const int id = ((z0 + (r >> 3)) * ny + y0 + (r & 7)) * nx + x0 + 8 * warp;
                    for (unsigned m = q ? m1 : m0; m; m &= m - 1) list[pos++] = (unsigned)(id + __ffs((int)m) - 1);
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace ebit
