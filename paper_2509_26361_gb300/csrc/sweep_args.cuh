// sweep_args.cuh -- the arguments of a split sweep's kernels and what they share.
#pragma once
#include "common.cuh"

namespace ebit {

// work lists of a sweep: unaligned edges and saddle faces of the two face
// families, and the annihilation checks of the two families
constexpr int SWEEP_LISTS = 6;

struct SweepArgs {
    Grid g;
    const uint8_t *__restrict__ cb;  // old colour bytes
    uint8_t *__restrict__ cbo;       // new colour bytes
    const double *__restrict__ s[3]; // old offsets per edge axis
    double *__restrict__ so[3];      // new offsets (written only where a marker is)
    const double *__restrict__ u;    // u_D on D-faces
    double lam;                      // dt / h
    double *__restrict__ adv[3];     // advected coordinate of each marker (scratch)
    int8_t *__restrict__ bin[3];     // floor(2 adv) (scratch)
    const int *__restrict__ list;    // band tile ids (null: every tile of g)
    const int *__restrict__ count;   // number of band tiles (device)
    unsigned *__restrict__ work[4];  // work lists, one entry per node each: unaligned fam.1, fam.2, saddle fam.1,
                                     // fam.2; the annihilation checks of a family fill its unaligned list from
                                     // the end (an edge is on one of the two at most)
    int *__restrict__ wcount;        // [6] list lengths (device): unaligned, saddle, annihilation checks
    long long cells = 0;             // entries of each work list (a batch: the cells of its arena)
    long long cb_whole = 0;          // bytes from cb that may be read as aligned 8-byte words (see load_colours8)
    unsigned long long *ctr;         // event counters
    uint32_t *tile_marker;           // per tile: proximity mask of its markers in the input or the output
    uint8_t *tile_dirty;             // per tile: processed since the last Front2VOF
    // Lists for the next sweep (a context's band sweeps; null elsewhere).  The
    // band pass appends every aligned edge that carries a marker after the
    // sweep to mk_out (the unaligned ones are its work lists 0 and 1) and every
    // tile whose new proximity mask is not empty to mt_out; it clears the band
    // flag of each tile it processes.  The next sweep's advection builds that
    // sweep's band from mt_out and the masks.
    unsigned *mk_out = nullptr;
    int *mk_out_count = nullptr;
    int *mt_out = nullptr;
    int *mt_out_count = nullptr;
    uint32_t *band_flag = nullptr;
    // the count of the band list the following sweep builds (cleared here)
    int *band_next_count = nullptr;
    // next band tile to take (blocks of the band pass take tiles in turn from
    // this counter; null: a fixed stride over the list)
    int *tile_next = nullptr;
    // lengths of the marker lists that mark_scan_kernel fills (cleared by the
    // band pass for the next scan; null: not scanned)
    int *scan_count = nullptr;
};

// The markers of the state before a sweep, as node ids of their edges, one
// list per edge axis, and the tiles whose proximity mask is not empty (the
// previous sweep's band pass wrote them); the band this sweep processes is
// built from the latter into band / band_count, with band_flag against
// duplicates.
struct MarkerLists {
    const unsigned *list[3];
    const int *count[3];
    int axis[3];
    const int *mtiles;
    const int *mtiles_count;
    int *band;
    int *band_count;
};

// Loads of data produced earlier in the same launch (the persistent batched
// sweep, F = true) bypass the non-coherent read-only path and L1; separate
// launches (F = false) read them through the read-only cache.
template <bool F, typename T>
__device__ __forceinline__ T ld_in(const T *p) {
    if (F) return __ldcg(p);
    return __ldg(p);
}

}  // namespace ebit
