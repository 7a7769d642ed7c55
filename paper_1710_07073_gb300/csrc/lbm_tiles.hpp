// The lattice tiles of one axis that a bubble's window touches: the integer
// arithmetic the kernels and the host's capacity bounds share.  Plain C++ (the
// CPU tests compile it too).
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

// The tiles (of T cells) that hold a cell of [lo, hi], as two runs of
// consecutive ones, [first, first + n0) then [second, ...), n in all, for a
// window that does not wrap onto itself (2 n + 2 <= L on a periodic axis, as
// lbm_set_bubbles ensures): no loops, divisions or arrays.  The update and the
// binning of one bubble are a single thread's or warp's serial code, run once
// per launch, so their length is paid in instruction fetches: with the general
// list code the counting of a bubble's tiles took 7,900 cycles of k_swarm_tail.
struct AxisRun {
    int first, n0, second, n;
    LBM_HD int tile(int i) const { return i < n0 ? first + i : second + (i - n0); }
};

template <int T>
LBM_HD AxisRun axis_run(int lo, int hi, int L, bool periodic) {
    static_assert((T & (T - 1)) == 0, "tiles of a power of two");
    if (periodic) {
        if (lo < 0) lo += L;
        if (hi >= L) hi -= L;
    } else {
        lo = lo < 0 ? 0 : lo;
        hi = hi > L - 1 ? L - 1 : hi;
        if (hi < lo) return AxisRun{0, 0, 0, 0};
    }
    const int ts = lo / T, te = hi / T;   // lo, hi >= 0
    if (lo <= hi) return AxisRun{ts, te - ts + 1, 0, te - ts + 1};
    // The window wraps: the tiles up to te, then those from ts (all of them
    // when both ends lie in one tile).
    const int nt = (L + T - 1) / T;
    if (te >= ts) return AxisRun{0, nt, 0, nt};
    return AxisRun{0, te + 1, ts, te + 1 + nt - ts};
}

// The most tiles that `cells` consecutive cells touch on an axis of L cells:
// whole tiles with one more for an end inside a tile, and one more again where
// a periodic axis ends in a narrower tile, which a window across the boundary
// adds to its whole ones.
LBM_HD int axis_tile_bound(int cells, int L, bool periodic, int T) {
    const int whole = (cells + T - 1) / T + 1;
    const int nt = (L + T - 1) / T;
    return periodic && L % T != 0 && whole < nt ? whole + 1 : whole;
}

// The tile layers [l0, l1] that hold a cell of [lo, hi], a window that may be
// wider than the axis; on a periodic axis to be taken modulo their number.
// l1 < l0: none.  (The cells are wrapped before they are divided: layers of a
// window counted past a narrow last tile would be off by one.)
struct LayerRun {
    int l0, l1;
};

template <int T>
LBM_HD LayerRun layer_run(int lo, int hi, int L, bool periodic) {
    const int nt = (L + T - 1) / T;
    if (!periodic) {
        lo = lo < 0 ? 0 : lo;
        hi = hi > L - 1 ? L - 1 : hi;
        return hi < lo ? LayerRun{0, -1} : LayerRun{lo / T, hi / T};
    }
    if (hi - lo + 1 >= L) return LayerRun{0, nt - 1};
    lo %= L;
    hi %= L;
    if (lo < 0) lo += L;
    if (hi < 0) hi += L;
    const int ls = lo / T, le = hi / T;
    if (lo <= hi) return LayerRun{ls, le};
    if (le >= ls) return LayerRun{0, nt - 1};
    return LayerRun{ls, le + nt};
}

}  // namespace lbm
