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
    double *__restrict__ rho;  // may be null
    double *__restrict__ mu;   // may be null
    double *__restrict__ f[3]; // null: no force
};

__device__ __forceinline__ bool curv_valid(uint8_t s) { return s == 1 || s == 2 || s == 3 || s == 5; }

// A dense pass of 48 bytes per cell, five sixths of them writes: bound by HBM.
// One thread per W neighbouring cells of an x-row and one round of loads and
// stores per thread: 512^3 as blocks that come and go moved 6.8 TB/s in a probe
// of the bare traffic where a resident grid looping over it reached 6.0.  With W
// = 2 every array is read and written in 16-byte pieces (the host takes it when
// rows and arrays start on 16-byte boundaries; odd rows take W = 1).  The stores
// stream past L2 (evict first), which keeps the previous plane's fractions there
// for the z neighbours.  The main path only selects: pure cells (C = 0 or 1,
// compared as bit patterns) get the end values of Eq. 6 -- the same values the
// formula gives there -- and every face force 0.  A cell the interface crosses
// then writes its own values over those, in a branch of its own, whose registers
// and FP64 arithmetic (a narrow pipe) stay out of the main path.
// Measured at 512^3: 1592 us with a block per row and 8-byte accesses,
// 1037 in this form (6.2 TB/s of the 48 bytes).
template <int W>
__global__ void __launch_bounds__(256) coupling_kernel(CouplingArgs a) {
    const int nx = a.g.n[0], ny = a.g.n[1], nz = a.g.n[2];
    const unsigned per_row = (unsigned)nx / W;
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    const unsigned row = t / per_row;
    const int x = (int)(t - row * per_row) * W;
    if (row >= (unsigned)(ny * nz)) return;
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
    bool mixed = false;
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
        for (int k = 0; k < W; k++) mixed = mixed || cy[k] != c[k] || cz[k] != c[k] || c[k] != c[0];
    }
#pragma unroll
    for (int k = 0; k < W; k++) mixed = mixed || (c[k] != 0 && c[k] != ONE);
    auto put = [&](double *p, double v0, double v1) {
        if (W == 2) __stcs(reinterpret_cast<double2 *>(p + idx), make_double2(v0, v1));
        else __stcs(p + idx, v0);
    };
    if (a.rho) put(a.rho, c[0] == 0 ? a.rho2 : a.rho1, c[W - 1] == 0 ? a.rho2 : a.rho1);
    if (a.mu) put(a.mu, c[0] == 0 ? a.mu2 : a.mu1, c[W - 1] == 0 ? a.mu2 : a.mu1);
    if (a.f[0]) {
        put(a.f[0], 0.0, 0.0);
        put(a.f[1], 0.0, 0.0);
        put(a.f[2], 0.0, 0.0);
    }
    if (!mixed) return;
#pragma unroll 1
    for (int k = 0; k < W; k++) {
        const long long i = idx + k;
        const long long cb = __ldg(Cb + i);
        const double v = __longlong_as_double(cb);
        if (cb != 0 && cb != ONE) {
            if (a.rho) a.rho[i] = v * a.rho1 + (1.0 - v) * a.rho2;
            if (a.mu) a.mu[i] = v * a.mu1 + (1.0 - v) * a.mu2;
        }
        if (!a.f[0]) continue;
        const bool ok = curv_valid(__ldg(a.st + i));
        const double kc = ok ? __ldg(a.kh + i) / a.h : 0.0;
#pragma unroll 1
        for (int d = 0; d < 3; d++) {
            const long long j = i + (d == 0 ? (k == 0 ? dx : -1) : (d == 1 ? dy : dz));
            const long long nb = __ldg(Cb + j);
            if (nb == cb) continue;
            const bool okn = curv_valid(__ldg(a.st + j));
            const double kn = okn ? __ldg(a.kh + j) / a.h : 0.0;
            const double kf = (ok && okn) ? 0.5 * (kc + kn) : (ok ? kc : (okn ? kn : 0.0));
            (d == 0 ? a.f[0] : (d == 1 ? a.f[1] : a.f[2]))[i] = a.sigma * kf * (v - __longlong_as_double(nb)) / a.h;
        }
    }
}

}  // namespace ebit
