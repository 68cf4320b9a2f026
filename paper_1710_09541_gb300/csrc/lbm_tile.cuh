// lbm_tile.cuh -- several time steps of a small grid in one launch.
//
// On a small grid a step is bound by its launch and by one round of latencies
// (64^2: 2.6 us a step, of which the arithmetic of 4096 nodes is a few tens of
// nanoseconds).  This kernel takes S steps per launch: a block owns a tile of
// nodes, pulls it from global memory with a halo of 2 S nodes, and keeps the
// state in shared memory between the steps, each of which computes a region
// two nodes narrower on every side than the last (a step reaches two nodes:
// one for the pull, one for the phi stencil).  One thread per node of the first
// region and its phi ring, the same node in every step; a step is
//   pull the node (step 1 from global memory, else from shared memory), its phi
//   to shared memory -- barrier -- stencil, collide, write the node in place (the
//   last step to global memory) -- barrier --
// Every value is formed by the functions of the one-step kernels in the same
// order and the shared state is in the storage format, so the result is
// theirs bit for bit.
//
// What bounds it: 1.8 us per launch (launch, first loads, stores) and then the
// latency of the steps, at up to 16 warps per SM.  Giving the threads new nodes in
// every step, so that the narrower regions filled whole warps, cost more in
// index arithmetic than it saved (64^2 1.52 us per step against 1.06); bounding
// the registers to 64 for two blocks per SM spilled (64^2 1.27 against 1.06).
#pragma once
#include "lbm_march.cuh"

namespace lbmpf {

constexpr int TILE_THREADS = 512;  // the most nodes of a first region with its phi ring

template <int ST>
struct TileSmem {
    static constexpr int LP = 4 * TILE_THREADS;  // bytes of one plane of the shared state
    static constexpr int PHI = MarchRow<ST>::RING_PLANES * LP;
    static constexpr int BYTES = PHI + LP;
};

template <int WALLS, int ST, bool CHK>
__device__ __forceinline__ void tile_block(char* smem, const MarchArgs& A, const Model& m, int x0, int y0, int tw,
                                           int th, int S, unsigned int nstep) {
    using Row = MarchRow<ST>;
    constexpr bool W = WALLS != 0;
    constexpr int LP = TileSmem<ST>::LP;
    const int nx = A.nx, ny = A.ny;
    const bool open_top = W && m.walls == 2;
    // the thread's node, the same in every step: one of the phi region of step 1
    const int mg = 2 * S - 1, w1 = tw + 2 * mg, i = threadIdx.x;
    const int ly = i / w1, xl = x0 - mg + i - ly * w1, yl = y0 - mg + ly;
    const int x = fold_x(xl, nx), y = W ? yl : fold_y(yl, ny, 0);
    // nodes from the tile (walls: none beyond the grid take part)
    int dist = max(max(x0 - xl, xl - (x0 + tw - 1)), max(max(y0 - yl, yl - (y0 + th - 1)), 0));
    if (W && (y < 0 || y >= ny)) dist = 1 << 20;
    const bool lo = W && y == 0, hi = W && !open_top && y == ny - 1;
    float* const sphi = reinterpret_cast<float*>(smem + TileSmem<ST>::PHI) + i;
    char* const own = smem + 4 * i;
    Row R;
    if (dist <= mg) {
        const unsigned int rc = 4u * nx * y, rm = 4u * nx * (y == 0 ? ny - 1 : y - 1);
        const unsigned int rp = 4u * nx * (y == ny - 1 ? (open_top ? y : 0) : y + 1);
        const unsigned int xc = 4u * x, xm = 4u * (x == 0 ? nx - 1 : x - 1);
        const unsigned int xp = 4u * (x == nx - 1 ? 0 : x + 1);
        const PullOff o{rm + xm, rm + xc, rm + xp, rc + xm, rc + xc, rc + xp, rp + xm, rp + xc, rp + xp};
#if LBM_DEBUG_CHECKS
        if (x < 0 || x >= nx || y < 0 || y >= ny || i >= TILE_THREADS) {
            atomicOr(A.flag, 4u);
            R = Row{};
        } else
#endif
            R.template pull<W>(A, o, lo, hi);
    }
    // neighbours in shared memory, as byte offsets from the own slot: rows w1 apart;
    // at the open top the row above is the row itself, at an edge row the ghost
    // phi row is the row itself
    const int pb = 4 * w1, up = open_top && y == ny - 1 ? 0 : pb;
    const PullOff o{unsigned(-pb - 4), unsigned(-pb), unsigned(-pb + 4), unsigned(-4), 0u, 4u,
                    unsigned(up - 4), unsigned(up), unsigned(up + 4)};
    const int n_ = W && y == ny - 1 ? 0 : w1, s_ = W && y == 0 ? 0 : -w1;
    for (int s = 1; s <= S; ++s) {
        const int reach = 2 * (S - s);  // nodes beyond the tile that still collide
        if (dist <= reach + 1) {
            if (s > 1) R.template pull_ring<W, LP>(own, o, lo, hi);
            *sphi = R.phi();
        }
        __syncthreads();
        if (dist <= reach) {
            const float phi = *sphi;
            const Stencil st = stencil<true>(phi, sphi[1], sphi[-1], sphi[n_], sphi[s_], sphi[n_ + 1], sphi[n_ - 1],
                                             sphi[s_ - 1], sphi[s_ + 1]);
            float f[9], g[9];
            R.values(f, g);
            const Macro M = macro_from<true>(m, Pop<ST>::template gmom<true>(g), phi, st.gx, st.gy, st.lap);
            if constexpr (CHK)
                if (dist == 0 && !isfinite(add(add(phi, M.ux), add(M.uy, M.p)))) report_nonfinite(A.flag);
            const float2 pu = collide_st<ST, true>(m, f, g, phi, st, M, R.prev);
            const unsigned int seed = (nstep + s) * 0x9e3779b9u;
            if (s < S)
                Row::template put_ring<LP>(own, f, g, phi, pu, (unsigned)(y * nx + x), seed);
            else
                Row::put(A, 4u * (y * nx + x), f, g, phi, pu, seed);
        }
        __syncthreads();
    }
}

}  // namespace lbmpf
