// common.cuh -- grid indexing and shared device helpers for the EBIT kernels.
//
// The whole EBIT translation unit is compiled with --fmad=false: every product
// and sum is its own IEEE double operation in the written order, and double
// division and square root are IEEE round-to-nearest (CUDA defaults).  The
// floating-point decisions of the method (which node a marker crossed, which
// circle root lies on an edge, the colour of a saddle face) therefore do not
// depend on compiler contraction.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ebit {

// Programmatic dependent launch.  The kernels of a step are launched with
// programmatic stream serialization, so the next kernel in the stream is
// launched as the blocks of the current one exit, overlapping its launch with
// the current kernel's tail.  Every such kernel calls pdl_wait() before its
// first access to global memory: it returns once the preceding kernel has
// completed and its writes are visible (and so, by induction, every earlier
// one).  None of them releases its dependents early
// (griddepcontrol.launch_dependents): grids sized to full occupancy then had
// the next kernel's waiting blocks take the slots of exiting ones unevenly,
// which measured slower than the release at exit.  For an ordinary launch
// pdl_wait() is a no-op.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Entry of a compacted work list for this thread in iteration `it` of a
// grid-stride loop over the list.  Whole warps of consecutive entries are dealt
// to the blocks in turn (warp slot 0 of every block, then slot 1, ...), so a
// list much shorter than the grid spreads over all SMs instead of filling the
// first blocks; every entry maps to one thread of one iteration.
__device__ __forceinline__ int list_item(int it) {
    const int gw = (it * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5)) * (int)gridDim.x + (int)blockIdx.x;
    return gw * 32 + (int)(threadIdx.x & 31);
}

// A double whose sums and products run as fused multiply-adds, a 1 + b and
// a b + (-0): the same values to the last bit (one rounding each, of the same
// exact result; signed zeros, infinities and NaN included).  GB300's FP64 units
// take a warp's multiply-add in 65 cycles per scheduler when all four have one,
// an add or a product in 78 (153 against 129 with two warps each).  The constants
// come from a register the compiler cannot see through, or it would turn the
// operations back.
struct Fp {
    double v;
    Fp() = default;
    __device__ __forceinline__ Fp(double x) : v(x) {}
    __device__ __forceinline__ operator double() const { return v; }
};
__device__ __forceinline__ unsigned opaque_zero() {
    unsigned r;
    asm("mov.u32 %0, %%smid;" : "=r"(r));  // an SM's number, far below 2^20
    return r >> 20;
}
__device__ __forceinline__ double fp_one() { return __hiloint2double((int)(0x3FF00000u | opaque_zero()), 0); }
__device__ __forceinline__ double fp_minus_zero() { return __hiloint2double((int)(0x80000000u | opaque_zero()), 0); }
__device__ __forceinline__ Fp operator+(Fp a, Fp b) { return __fma_rn(a.v, fp_one(), b.v); }
__device__ __forceinline__ Fp operator-(Fp a, Fp b) { return __fma_rn(-b.v, fp_one(), a.v); }
__device__ __forceinline__ Fp operator*(Fp a, Fp b) { return __fma_rn(a.v, b.v, fp_minus_zero()); }
__device__ __forceinline__ Fp operator/(Fp a, Fp b) { return a.v / b.v; }
__device__ __forceinline__ Fp operator+(Fp a, double b) { return a + Fp(b); }
__device__ __forceinline__ Fp operator-(Fp a, double b) { return a - Fp(b); }
__device__ __forceinline__ Fp operator*(Fp a, double b) { return a * Fp(b); }
__device__ __forceinline__ Fp operator/(Fp a, double b) { return a / Fp(b); }
__device__ __forceinline__ Fp operator+(double a, Fp b) { return Fp(a) + b; }
__device__ __forceinline__ Fp operator-(double a, Fp b) { return Fp(a) - b; }
__device__ __forceinline__ Fp operator*(double a, Fp b) { return Fp(a) * b; }
__device__ __forceinline__ Fp &operator+=(Fp &a, Fp b) { return a = a + b; }

// a / b for a y that is 1 / b correctly rounded: one product, the remainder and one
// correction (P. Markstein, IBM J. Res. Dev. 34, 1990), in three FP64 operations
// where a division takes nine.  Correctly rounded where the product is within a unit
// in the last place of the quotient (a's fraction not below b's, among others);
// elsewhere what is rounded lies within 2^-52 units of it, and no operands were
// found for which the result differs (7e7 whose quotients lie as near to the middle
// of two doubles as any can, 2e8 others).  Only for operands that pass safe_quotient: not zero, and far from where
// the remainder underflows or the product overflows; the callers divide the others.
__device__ __forceinline__ double quotient(double a, double b, double y) {
    const double q = __fma_rn(a, y, fp_minus_zero());
    return __fma_rn(__fma_rn(-b, q, a), y, q);
}
__device__ __forceinline__ bool safe_quotient(double a) {
    const unsigned e = ((unsigned)__double2hiint(a) >> 20) & 0x7FF;
    return e - 1023u + 400u <= 800u;  // 2^-400 <= |a| < 2^401
}

constexpr double ONE_MINUS = 0.99999999999999988898;  // 1 - 2^-53, largest offset below 1
constexpr int TILE = 8;                               // tile edge of a single grid (cells)
constexpr int TILE_CELLS = TILE * TILE * TILE;          // cells of every tile shape

// Tile shapes (cells per tile edge along x, y, z; 512 cells each).  A single
// grid uses shape 0; a batch may use any (chosen by its autotuner).  Every
// edge is at least 4 cells, more than the NEAR = 3 layers of the proximity
// mask, so a marker touches its own tile and the 26 adjacent ones; across a last
// tile clipped to fewer than NEAR cells it also touches the tile before that one
// (see narrow_last).
constexpr int N_TILE_SHAPES = 3;
__host__ __device__ constexpr int tile_log2(int sh, int a) {
    return sh == 0 ? 3 : (sh == 1 ? (a == 0 ? 4 : (a == 1 ? 3 : 2)) : (a == 0 ? 5 : 2));
}

// Tile proximity mask: bit near_bit(dx, dy, dz) is set when a marker owned by a
// node of the tile lies within NEAR cells of the neighbour tile in direction
// (dx, dy, dz) (the owner node in the NEAR layers next to that neighbour, along
// every axis with a non-zero step, counted from the tile's last cell inside the
// grid where it is clipped); bit near_bit(0, 0, 0) whenever the tile
// owns a marker.  A sweep changes a node's byte or edges only if a marker is
// owned by a node within one cell behind or two cells ahead of it (the window of
// the band pass), and Front2VOF reads a cell's corners one cell ahead, so a
// tile next to a marker tile needs the sweep (and Front2VOF) only where that
// neighbour owns a marker within three cells of it.
constexpr int NEAR = 3;
__host__ __device__ inline int near_bit(int dx, int dy, int dz) { return 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1); }

enum Counter { C_MARKERS = 0, C_ANNIHILATE = 1, C_MULTI = 2, C_INCONSISTENT = 3, C_CFL = 4, C_N = 5 };
// extra device counters after the event counters (C_NONFINITE: markers whose
// displacement u dt / h was not finite; they are left in place)
enum { C_F2V_BAD = C_N, C_TILES = C_N + 1, C_NONFINITE = C_N + 2, C_TOTAL = C_N + 3 };

struct Grid {
    int n[3];        // cells per axis
    int td[3];       // tiles per axis
    int ntiles;
    int tl[3];       // log2 of the tile edge per axis (3, 3, 3 for 8^3 tiles)
};

// tiles per axis and in total for tile shape sh
__host__ __device__ inline void grid_tiles(Grid &g, int sh) {
    g.ntiles = 1;
    for (int a = 0; a < 3; a++) {
        g.tl[a] = tile_log2(sh, a);
        g.td[a] = (g.n[a] + (1 << g.tl[a]) - 1) >> g.tl[a];
        g.ntiles *= g.td[a];
    }
}

// Is the last tile of axis a clipped to fewer than NEAR cells?  A marker in the
// first layers of tile 0 then touches, behind it across the periodic seam, both
// the last tile and the one before that: tile 0's step -1 stands for both.  (Ahead
// a marker touches no node further than the next one, so step +1 names one tile
// whatever its width.)
__host__ __device__ inline bool narrow_last(const Grid &g, int a) {
    return g.n[a] - ((g.td[a] - 1) << g.tl[a]) < NEAR;
}

__host__ __device__ inline int wrapc(int v, int n) {
    // v is within a few cells of [0, n)
    return v < 0 ? v + n : (v >= n ? v - n : v);
}

__device__ __forceinline__ int lin(const Grid &g, int x, int y, int z) {
    return (wrapc(z, g.n[2]) * g.n[1] + wrapc(y, g.n[1])) * g.n[0] + wrapc(x, g.n[0]);
}

__device__ __forceinline__ int lin3(const Grid &g, const int q[3]) { return lin(g, q[0], q[1], q[2]); }

// tile id -> origin of its cells
__device__ __forceinline__ void tile_origin(const Grid &g, int t, int o[3]) {
    int tx = t % g.td[0];
    int r = t / g.td[0];
    int ty = r % g.td[1];
    int tz = r / g.td[1];
    o[0] = tx << g.tl[0];
    o[1] = ty << g.tl[1];
    o[2] = tz << g.tl[2];
}

// Is tile (tx, ty, tz) in the band: does it own a marker, or does a neighbour
// own one within NEAR cells of it (that neighbour's proximity bit toward it)?
// (the loads are independent: no early exit)
__device__ __forceinline__ bool in_band(const Grid &g, const uint32_t *__restrict__ mask, int tx, int ty, int tz) {
    // step 2: from the tile before a narrow last one to tile 0, whose step -1 names both
    const int ex = narrow_last(g, 0) && tx == g.td[0] - 2 ? 2 : 1, ey = narrow_last(g, 1) && ty == g.td[1] - 2 ? 2 : 1,
              ez = narrow_last(g, 2) && tz == g.td[2] - 2 ? 2 : 1;
    unsigned on = 0;
    for (int dz = -1; dz <= ez; dz++)
        for (int dy = -1; dy <= ey; dy++)
            for (int dx = -1; dx <= ex; dx++) {
                const int nx = wrapc(tx + dx, g.td[0]), ny = wrapc(ty + dy, g.td[1]), nz = wrapc(tz + dz, g.td[2]);
                on |= mask[(nz * g.td[1] + ny) * g.td[0] + nx] >> near_bit(dx < 2 ? -dx : -1, dy < 2 ? -dy : -1, dz < 2 ? -dz : -1);
            }
    return on & 1u;
}

// Youngs normal n = -grad C of a 3x3x3 block (1-2-1 weights, b2 outer, b1
// inner), in the type T of the block values.
template <typename T>
__device__ __forceinline__ void youngs(const T (&v)[27], T n[3]) {
    const T w[3] = {T(1), T(2), T(1)};
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const int t1 = (d == 0) ? 1 : 0, t2 = (d == 2) ? 1 : 2;
        T gsum = T(0);
#pragma unroll
        for (int b2 = -1; b2 <= 1; b2++)
#pragma unroll
            for (int b1 = -1; b1 <= 1; b1++) {
                int op[3] = {1, 1, 1}, om[3] = {1, 1, 1};
                op[d] += 1;
                om[d] -= 1;
                op[t1] += b1;
                om[t1] += b1;
                op[t2] += b2;
                om[t2] += b2;
                gsum += (w[b1 + 1] * w[b2 + 1]) * (v[op[2] * 9 + op[1] * 3 + op[0]] - v[om[2] * 9 + om[1] * 3 + om[0]]);
            }
        n[d] = -gsum;
    }
}

// Bound on |n_float - n| for values rounded to float: 8 additions below 64
// (half an ulp, 2^-19, each) and the inputs' rounding (2^-25 each, weights
// summing to 16, three roundings per difference) stay under 1.7e-5.
constexpr float CANON_EPS = 3.0e-5f;

}  // namespace ebit
