// coupling.cuh -- the one-fluid coupling terms of the EBIT interface
// (arxiv 2509.26361, Sec. 2.5: Eq. 6 and the surface-tension term).
//
// Eq. 6 with the Heaviside function of the reference phase taken as the
// Front2VOF fraction C: rho = C rho1 + (1 - C) rho2, mu = C mu1 + (1 - C) mu2,
// per cell.  Surface tension as a well-balanced continuum surface force on the
// faces of the MAC grid: on the a-face between cells idx - e_a and idx,
//     f_a = sigma kappa_f (C[idx] - C[idx - e_a]) / h,
// kappa = kappa_h / h on cells whose curvature is valid (height functions
// along x, y or z, or the network), kappa_f the mean of the two cells' values,
// the one valid value, or 0.  One pass over the grid, x fastest: every array
// is read and written once, coalesced; the neighbour values come through L1/L2.
#pragma once
#include "common.cuh"

namespace ebit {

struct CouplingArgs {
    Grid g;
    const double *__restrict__ C;
    const double *__restrict__ kh;
    const uint8_t *__restrict__ st;
    double sigma, rho1, rho2, mu1, mu2, h;
    double inv_h;              // 1 / h, correctly rounded
    double *__restrict__ rho;  // may be null
    double *__restrict__ mu;   // may be null
    double *__restrict__ f[3]; // null: no force
};

__device__ __forceinline__ bool curv_valid(uint8_t s) { return s == 1 || s == 2 || s == 3 || s == 5; }

// a / h (h > 0) in three operations instead of nine
__device__ __forceinline__ double over_h(const CouplingArgs &a, double v) {
    if (!safe_quotient(a.h)) return v / a.h;
    if (((unsigned long long)__double_as_longlong(v) << 1) == 0) return v;
    return safe_quotient(v) ? quotient(v, a.h, a.inv_h) : v / a.h;
}

// A dense pass of 48 bytes per cell, five sixths of them writes: bound by HBM.
// One thread per W neighbouring cells of an x-row and one round of loads and
// stores per thread: 512^3 as blocks that come and go moved 6.8 TB/s in a probe
// of the bare traffic where a resident grid looping over it reached 6.0.  With W
// = 2 every array is read and written in 16-byte pieces (the host takes it when
// rows and arrays start on 16-byte boundaries; odd rows take W = 1).  The stores
// stream past L2 (evict first), which keeps the previous plane's fractions there
// for the z neighbours.  The main path only selects: pure cells (C = 0 or 1,
// compared as bit patterns) get the end values of Eq. 6 -- the same values the
// formula gives there -- and every face force 0.  The cells the interface crosses
// are then compacted over the warp and their values written over those, in a branch
// of its own, whose registers and FP64 arithmetic (a narrow pipe) stay out of the
// main path: with each lane taking its own two cells in turn, a warp ran the
// arithmetic twice for the two or three such cells of a row (256^3, one sphere: 337
// us, 199 compacted and with quotients by 1 / h; 312 with a block per row).
// Measured at 512^3: 1592 us with a block per row and 8-byte accesses,
// 1037 with W = 2, 1025 in this form (6.3 TB/s of the 48 bytes).
template <int W>
__global__ void __launch_bounds__(256) coupling_kernel(CouplingArgs a) {
    const int nx = a.g.n[0], ny = a.g.n[1], nz = a.g.n[2];
    const unsigned per_row = (unsigned)nx / W;
    __shared__ uint8_t s_cell[8][32 * W];  // per warp: the lane and cell of each mixed cell
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    const bool in = t / per_row < (unsigned)(ny * nz);  // (others repeat the last thread's reads)
    const unsigned row = in ? t / per_row : (unsigned)(ny * nz) - 1u;
    const int x = in ? (int)(t - row * per_row) * W : nx - W;
    const int z = (int)row / ny, y = (int)row - z * ny;
    const long long nxy = (long long)nx * ny, idx = (long long)row * nx + x;
    // the cells one step back along x, y and z (periodic)
    const long long dx = x == 0 ? nx - 1 : -1, dy = y == 0 ? nxy - nx : -(long long)nx,
                    dz = z == 0 ? nxy * (nz - 1) : -nxy;
    const long long *__restrict__ Cb = reinterpret_cast<const long long *>(a.C);
    constexpr long long ONE = 0x3FF0000000000000LL;
    long long c[W];
    if (W == 2) {
        const longlong2 v = __ldg(reinterpret_cast<const longlong2 *>(Cb + idx));
        c[0] = v.x;
        c[W - 1] = v.y;
    } else {
        c[0] = __ldg(Cb + idx);
    }
    unsigned mixed = 0;  // bit k: cell k is cut, or a face force of it is not 0
    if (a.f[0]) {
        long long cy[W], cz[W];
        if (W == 2) {
            const longlong2 v = __ldg(reinterpret_cast<const longlong2 *>(Cb + idx + dy));
            const longlong2 w = __ldg(reinterpret_cast<const longlong2 *>(Cb + idx + dz));
            cy[0] = v.x;
            cy[W - 1] = v.y;
            cz[0] = w.x;
            cz[W - 1] = w.y;
        } else {
            cy[0] = __ldg(Cb + idx + dy);
            cz[0] = __ldg(Cb + idx + dz);
        }
        mixed = __ldg(Cb + idx + dx) != c[0];
#pragma unroll
        for (int k = 0; k < W; k++) mixed |= (cy[k] != c[k] || cz[k] != c[k] || (k && c[k] != c[0]) ? 1u : 0u) << k;
    }
#pragma unroll
    for (int k = 0; k < W; k++) mixed |= (c[k] != 0 && c[k] != ONE ? 1u : 0u) << k;
    auto put = [&](double *p, double v0, double v1) {
        if (W == 2) __stcs(reinterpret_cast<double2 *>(p + idx), make_double2(v0, v1));
        else __stcs(p + idx, v0);
    };
    if (in) {
        if (a.rho) put(a.rho, c[0] == 0 ? a.rho2 : a.rho1, c[W - 1] == 0 ? a.rho2 : a.rho1);
        if (a.mu) put(a.mu, c[0] == 0 ? a.mu2 : a.mu1, c[W - 1] == 0 ? a.mu2 : a.mu1);
        if (a.f[0]) {
            put(a.f[0], 0.0, 0.0);
            put(a.f[1], 0.0, 0.0);
            put(a.f[2], 0.0, 0.0);
        }
    }
    const unsigned full = 0xffffffffu;
    if (!__any_sync(full, in && mixed != 0)) return;
    const int lane = threadIdx.x & 31;
    uint8_t *list = s_cell[threadIdx.x >> 5];
    int count = 0;
#pragma unroll
    for (int k = 0; k < W; k++) {
        const bool on = in && (mixed >> k & 1);
        const unsigned m = __ballot_sync(full, on);
        if (on) list[count + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(lane | k << 5);
        count += __popc(m);
    }
    __syncwarp();  // the list, and the pure values before the cells' own
#pragma unroll 1
    for (int n0 = 0; n0 < count; n0 += 32) {
        const bool on = n0 + lane < count;
        const int who = on ? list[n0 + lane] & 31 : 0, k = on ? list[n0 + lane] >> 5 : 0;
        const long long i = __shfl_sync(full, idx, who) + k, ox = __shfl_sync(full, dx, who),
                        oy = __shfl_sync(full, dy, who), oz = __shfl_sync(full, dz, who);
        if (!on) continue;
        const long long cb = __ldg(Cb + i);
        const Fp v = __longlong_as_double(cb);
        if (cb != 0 && cb != ONE) {
            if (a.rho) a.rho[i] = v * a.rho1 + (1.0 - v) * a.rho2;
            if (a.mu) a.mu[i] = v * a.mu1 + (1.0 - v) * a.mu2;
        }
        if (!a.f[0]) continue;
        const bool ok = curv_valid(__ldg(a.st + i));
        const Fp kc = ok ? over_h(a, __ldg(a.kh + i)) : 0.0;
#pragma unroll 1
        for (int d = 0; d < 3; d++) {
            const long long j = i + (d == 0 ? (k == 0 ? ox : -1) : (d == 1 ? oy : oz));
            const long long nb = __ldg(Cb + j);
            if (nb == cb) continue;
            const bool okn = curv_valid(__ldg(a.st + j));
            const Fp kn = okn ? over_h(a, __ldg(a.kh + j)) : 0.0;
            const Fp kf = (ok && okn) ? 0.5 * (kc + kn) : (ok ? kc : (okn ? kn : Fp(0.0)));
            (d == 0 ? a.f[0] : (d == 1 ? a.f[1] : a.f[2]))[i] = over_h(a, a.sigma * kf * (v - Fp(__longlong_as_double(nb))));
        }
    }
}

}  // namespace ebit
