// lbm_march.cuh -- two time steps in one pass over the grid.
//
// A single step reads and writes the whole state (160 B per node with FP32
// storage), which bounds it on large grids.  This kernel advances two steps per
// read and write: a block owns a strip of columns and a chunk of rows and
// marches along the rows; the state between the two steps lives only in a
// five-row ring in shared memory.  The march also forms each row's phi once (the
// tile kernels recompute it on a ring around every tile) and keeps one set of
// column offsets per thread.
//
// The block has two sets of TW threads, one thread per column in each: the
// first set takes step 1, the second step 2.  Iteration t handles logical row t
// and rows behind it, in two halves:
//
//        step-1 threads                          step-2 threads
//   P    phi at row t, from the values pulled    phi at row t-3, from the ring
//        one iteration earlier                   rows t-4 .. t-2
//        -- barrier of the set --                -- barrier of the set --
//   Q    collide row t-1 (phi rows t-2 .. t),    collide row t-4 (phi rows
//        write ring row t-1, pull row t+1        t-5 .. t-3, ring rows
//        from global memory                      t-5 .. t-3), store it
//        ---------------- barrier of the block ----------------
//
// Logical row t is grid row first + dir * t.  A strip's three outermost columns
// and a chunk's three outermost rows on each side are computed by both
// neighbours (two of the rows collide in step 1).
//
// Every value is formed by the functions of the one-step kernels in the same
// order, and the ring holds what they would have stored, so the result is
// theirs bit for bit.
//
// What bounds it: latency.  At 2048^2 with FP32 storage a launch (two steps)
// moves 620 MB of DRAM traffic in 139 us, 0.66 of the measured copy bandwidth, at
// an IPC of 2.1 of 4; with FP16 335 MB at an IPC of 2.6.
// Measured (us per step, one-step kernel of its time -> this one): FP32 2048^2
// 103.2 -> 69.6, 1501 x 1103 51.9 -> 29.4, walled 2400 x 600 39.6 -> 26.6; FP16 70.4
// (64.6 with packed arithmetic) -> 59.4, 32.2 -> 25.7, 26.5 (24.4) -> 22.8; BF16-SR
// 73.6 (68.6) -> 62.3, 33.6 -> 27.0, 27.4 (25.2) -> 23.8.  One set of threads taking
// both steps, with four blocks of 128 threads per SM, took 84.5 (FP32) and 59.0
// (FP16) at 2048^2: its 112 registers left 16 warps to cover the loads.  Three
// blocks of 2 x 128 threads at 80 registers beat two at 128 (82.3 / 69.8) and four
// at 64 (spills: 86.7 / 62.4); strips of 64 / 96 / 192 threads 71.9 / 72.7 / 75.5
// against 71.2 at 128 (FP32).  Separate barriers and one or two more ring rows, so
// that step 1 may run ahead of step 2, gave nothing (70.0 / 59.1 at five rows, 84.5
// at six, whose shared memory leaves L1 28 KB).  L2 prefetch of the rows ahead
// (bulk copies or tensor boxes) was slower at every distance above two rows and on
// grids that fit L2, and was left out.
#pragma once
#include <type_traits>

#include "lbm_store.cuh"

namespace lbmpf {

// packed arithmetic (F2), us per step without -> with: FP32 768^2 12.6 -> 11.8,
// 2048^2 70.9 -> 69.6, walled 2400 x 600 27.2 -> 26.6; FP16 2048^2 59.5 -> 59.4, 701 x
// 333 6.7 -> 6.4
#ifndef LBM_MARCH_PK
#define LBM_MARCH_PK 1
#endif
constexpr bool MARCH_PK = LBM_MARCH_PK;

// byte offsets of a node's nine pull sources inside a plane of 4-byte entries:
// rows y-1, y, y+1 (m, c, p) x columns x-1, x, x+1
struct PullOff {
    unsigned int mm, mc, mp, cm, cc, cp, pm, pc, pp;
};
template <class T>
__device__ __forceinline__ T ldp(const char* base, unsigned int off) {
    return __ldg(reinterpret_cast<const T*>(base + off));
}
template <class T>
__device__ __forceinline__ void stp(char* base, unsigned int off, T v) {
    *reinterpret_cast<T*>(base + off) = v;
}

// A node's pull from nine planes: ld(i, offset) reads direction i's plane.
// lo / hi: bounce-back at the wall below / above (uniform over the block, which
// works on one row); ZERO: with the rest direction.
template <bool WALLS, bool ZERO, class T, class LD>
__device__ __forceinline__ void pull_dirs(LD ld, const PullOff& o, bool lo, bool hi, T v[9]) {
    lo = WALLS && lo;
    hi = WALLS && hi;
    if (ZERO) v[0] = ld(0, o.cc);
    v[1] = ld(1, o.cm);
    v[3] = ld(3, o.cp);
    // (selects rather than branches: two paths through the loads cost registers)
    v[2] = ld(lo ? 4 : 2, lo ? o.cc : o.mc);
    v[5] = ld(lo ? 7 : 5, lo ? o.cc : o.mm);
    v[6] = ld(lo ? 8 : 6, lo ? o.cc : o.mp);
    v[4] = ld(hi ? 2 : 4, hi ? o.cc : o.pc);
    v[7] = ld(hi ? 5 : 7, hi ? o.cc : o.pp);
    v[8] = ld(hi ? 6 : 8, hi ? o.cc : o.pm);
}
template <class T>
__device__ __forceinline__ T& sh(char* p) {
    return *reinterpret_cast<T*>(p);
}
template <class T>
__device__ __forceinline__ const T& sh(const char* p) {
    return *reinterpret_cast<const T*>(p);
}

// The pulled values of one node in a storage format: from global memory (pull;
// A.src(i): the planes in the ring's order) or from the shared ring (pull_ring; planes
// LP bytes apart; pull_ring_phi: only what phi needs).
template <int ST>
struct MarchRow {  // 16-bit formats: the code words as stored
    using P = Pop<ST>;
    static constexpr int RING_PLANES = 12;  // f_0, 8 words, g_0, (phi u)
    unsigned int w[9];
    float f0;
    unsigned short g0;
    float2 prev;  // (phi u) of the previous step
    template <bool WALLS, class ARGS>
    __device__ __forceinline__ void pull(const ARGS& A, const PullOff& o, bool lo, bool hi) {
        prev = make_float2(ldp<float>(A.src(10), o.cc), ldp<float>(A.src(11), o.cc));
        f0 = ldp<float>(A.src(0), o.cc);
        g0 = ldp<unsigned short>(A.src(9), o.cc >> 1);
        w[0] = 0u;
        pull_dirs<WALLS, false>([&](int i, unsigned int off) { return ldp<unsigned int>(A.src(i), off); }, o, lo, hi,
                                w);
    }
    template <bool WALLS, int LP>
    __device__ __forceinline__ void pull_ring_phi(const char* ring, const PullOff& o, bool lo, bool hi) {
        f0 = sh<float>(ring + o.cc);
        w[0] = 0u;
        pull_dirs<WALLS, false>([&](int i, unsigned int off) { return sh<unsigned int>(ring + (int)off + i * LP); }, o,
                                lo, hi, w);
    }
    template <bool WALLS, int LP>
    __device__ __forceinline__ void pull_ring(const char* ring, const PullOff& o, bool lo, bool hi) {
        pull_ring_phi<WALLS, LP>(ring, o, lo, hi);
        g0 = sh<unsigned short>(ring + o.cc + 9 * LP);
        prev = make_float2(sh<float>(ring + o.cc + 10 * LP), sh<float>(ring + o.cc + 11 * LP));
    }
    __device__ __forceinline__ float phi() const {
        float h[9];
        codes_f<ST>(w, f0, h);
        return P::template phi_of<MARCH_PK>(h);
    }
    __device__ __forceinline__ void values(float h[9], float k[9]) const {
        codes_f<ST>(w, f0, h);
        codes_g<ST>(w, g0, k);
    }
    // the post-collision node in storage form: to the ring, or to the planes d
    template <int LP>
    __device__ static __forceinline__ void put_ring(char* at, const float h[9], const float k[9], float phi,
                                                    float2 pu, unsigned int node, unsigned int seed) {
        unsigned int w[9];
        float r0;
        unsigned short q0;
        P::template encode<MARCH_PK>(h, k, phi, node, seed, w, r0, q0);
        sh<float>(at) = r0;
#pragma unroll
        for (int i = 1; i < 9; ++i) sh<unsigned int>(at + i * LP) = w[i];
        sh<unsigned short>(at + 9 * LP) = q0;
        sh<float>(at + 10 * LP) = pu.x;
        sh<float>(at + 11 * LP) = pu.y;
    }
    template <class ARGS>
    __device__ static __forceinline__ void put(const ARGS& A, unsigned int off, const float h[9], const float k[9],
                                               float phi, float2 pu, unsigned int seed) {
        unsigned int w[9];
        float r0;
        unsigned short q0;
        P::template encode<MARCH_PK>(h, k, phi, off >> 2, seed, w, r0, q0);
#pragma unroll
        for (int i = 1; i < 9; ++i) stp(A.dst(i), off, w[i]);
        stp(A.dst(0), off, r0);
        stp(A.dst(9), off >> 1, q0);
        stp(A.dst(10), off, pu.x);
        stp(A.dst(11), off, pu.y);
    }
};
template <>
struct MarchRow<ST_FP32> {
    static constexpr int RING_PLANES = 20;  // f, g, (phi u)
    float f[9], g[9];
    float2 prev;
    template <bool WALLS, class ARGS>
    __device__ __forceinline__ void pull(const ARGS& A, const PullOff& o, bool lo, bool hi) {
        prev = make_float2(ldp<float>(A.src(18), o.cc), ldp<float>(A.src(19), o.cc));
        pull_dirs<WALLS, true>([&](int i, unsigned int off) { return ldp<float>(A.src(i), off); }, o, lo, hi, f);
        pull_dirs<WALLS, true>([&](int i, unsigned int off) { return ldp<float>(A.src(9 + i), off); }, o, lo, hi, g);
    }
    template <bool WALLS, int LP>
    __device__ __forceinline__ void pull_ring_phi(const char* ring, const PullOff& o, bool lo, bool hi) {
        pull_dirs<WALLS, true>([&](int i, unsigned int off) { return sh<float>(ring + (int)off + i * LP); }, o, lo, hi, f);
    }
    template <bool WALLS, int LP>
    __device__ __forceinline__ void pull_ring(const char* ring, const PullOff& o, bool lo, bool hi) {
        pull_ring_phi<WALLS, LP>(ring, o, lo, hi);
        pull_dirs<WALLS, true>([&](int i, unsigned int off) { return sh<float>(ring + (int)off + (9 + i) * LP); }, o, lo,
                               hi, g);
        prev = make_float2(sh<float>(ring + o.cc + 18 * LP), sh<float>(ring + o.cc + 19 * LP));
    }
    __device__ __forceinline__ float phi() const { return sum9<MARCH_PK>(f); }
    __device__ __forceinline__ void values(float h[9], float k[9]) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            h[i] = f[i];
            k[i] = g[i];
        }
    }
    template <int LP>
    __device__ static __forceinline__ void put_ring(char* at, const float h[9], const float k[9], float phi,
                                                    float2 pu, unsigned int, unsigned int) {
        sh<float>(at) = sub(phi, sum8<MARCH_PK>(h));
#pragma unroll
        for (int i = 1; i < 9; ++i) sh<float>(at + i * LP) = h[i];
#pragma unroll
        for (int i = 0; i < 9; ++i) sh<float>(at + (9 + i) * LP) = k[i];
        sh<float>(at + 18 * LP) = pu.x;
        sh<float>(at + 19 * LP) = pu.y;
    }
    template <class ARGS>
    __device__ static __forceinline__ void put(const ARGS& A, unsigned int off, const float h[9], const float k[9],
                                               float phi, float2 pu, unsigned int) {
        stp(A.dst(0), off, sub(phi, sum8<MARCH_PK>(h)));
        stp(A.dst(9), off, k[0]);
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            stp(A.dst(i), off, h[i]);
            stp(A.dst(9 + i), off, k[i]);
        }
        stp(A.dst(18), off, pu.x);
        stp(A.dst(19), off, pu.y);
    }
};

constexpr int MARCH_HALO = 3;  // columns and rows computed beyond a block's own on each side
constexpr int MARCH_PAD = 16;  // bytes before and after the shared rows: the outermost threads read one past them

template <int TW, int ST>
struct MarchSmem {
    static constexpr int LINE = 4 * TW;                            // bytes of one row of one plane
    static constexpr int SLOT = LINE * MarchRow<ST>::RING_PLANES;  // one ring row
    static constexpr int PHI = MARCH_PAD;                          // phi of step 1, 3 rows, then of step 2
    static constexpr int RING = PHI + 6 * LINE;
    // FP32: 54.3 KB, so that three blocks stay within a 164 KB share of the SM's
    // 256 KB and leave the L1 cache 92 KB
    static constexpr int BYTES = RING + 5 * SLOT + MARCH_PAD;
};

// The planes read and written, in the ring's order (the addresses come from the
// constant bank, so they take no registers).
struct MarchArgs {
    const char* s[20];
    char* d[20];
    unsigned int* flag;
    int nx, ny;
    __device__ __forceinline__ const char* src(int i) const { return s[i]; }
    __device__ __forceinline__ char* dst(int i) const { return d[i]; }
};
// The same of one case of a batch, from its buffers' bases.
template <int ST>
struct MarchCase {
    const char *fs, *gs, *pus;
    char *fd, *gd, *pud;
    size_t plane;  // bytes of a plane of 4-byte entries
    unsigned int* flag;
    int nx, ny;
    static constexpr int G = ST == ST_FP32 ? 9 : 1;  // planes of the g buffer
    __device__ __forceinline__ const char* src(int i) const {
        return i < 9 ? fs + i * plane : i < 9 + G ? gs + (i - 9) * plane : pus + (i - 9 - G) * plane;
    }
    __device__ __forceinline__ char* dst(int i) const {
        return i < 9 ? fd + i * plane : i < 9 + G ? gd + (i - 9) * plane : pud + (i - 9 - G) * plane;
    }
};

// One block's strip of columns [x0, x0 + wlen) and chunk of rows [y0, y1),
// marched in direction dir.  m.seed / seed2: the
// dithers' seeds of the two steps.
// STEP: which of the two steps the calling threads take.
template <int STEP, int TW, int WALLS, int ST, bool CHK, class ARGS>
__device__ __forceinline__ void march_block(char* smem, const ARGS& A, const Model& m, int x0, int wlen,
                                            int y0, int y1, int dir, unsigned int seed2) {
    using Row = MarchRow<ST>;
    using S = MarchSmem<TW, ST>;
    constexpr bool W = WALLS != 0;
    constexpr int LP = S::LINE;
    const int nx = A.nx, ny = A.ny;
    const int tx = threadIdx.x % TW;
    const int x = fold_x(x0 - MARCH_HALO + tx, nx);
    const unsigned int xc = 4u * x, xm = 4u * (x == 0 ? nx - 1 : x - 1), xp = 4u * (x == nx - 1 ? 0 : x + 1);
    const bool out = tx >= MARCH_HALO && tx < MARCH_HALO + wlen;
    const bool open_top = W && m.walls == 2;
    const unsigned int pitch = 4u * nx;
    // whether logical row t, grid row y, is one of those computed k rows beyond
    // the block's own (walls: no row beyond the grid)
    const int rows = y1 - y0;
    auto takes = [&](int k, int t, int y) {
        return t >= 3 - k && t <= rows + 2 + k && (!W || (unsigned)y < (unsigned)ny);
    };

    char* const sx = smem + 4 * tx;  // this thread's column of every row
#if LBM_DEBUG_CHECKS
    for (int k = threadIdx.x; k < S::BYTES / 4; k += 2 * TW)
        reinterpret_cast<float*>(smem)[k] = __int_as_float(0x7fc00000);
    __syncthreads();
#endif
    // (with walls no row needs it, but a row number that is not linear in t keeps
    // the compiler from carrying every plane's address through the loop, which
    // spilled 144 bytes)
    auto wrap = [&](int y) { return y < 0 ? y + ny : (y >= ny ? y - ny : y); };
    // a row's pull offsets.  fast (a compile-time flag): the row and its
    // neighbours lie inside the grid, away from any wall or open top
    auto row_off = [&](auto fast, int y) {
        constexpr bool WF = W && decltype(fast)::value;
        const int ym = !WF && y == 0 ? ny - 1 : y - 1;
        const int yp = !WF && y == ny - 1 ? (open_top ? y : 0) : y + 1;
        const unsigned int rc = pitch * y, rm = pitch * ym, rp = pitch * yp;
        return PullOff{rm + xm, rm + xc, rm + xp, rc + xm, rc + xc, rc + xp, rp + xm, rp + xc, rp + xp};
    };
#if LBM_DEBUG_CHECKS
    auto row_bad = [&](int y) {
        const bool bad = y < 0 || y >= ny || x < 0 || x >= nx;
        if (bad) atomicOr(A.flag, 4u);
        return bad;
    };
#else
    auto row_bad = [](int) { return false; };
#endif
    auto load = [&](auto fast, Row& R, int yl) {
        constexpr bool WB = W && !decltype(fast)::value;
        const int y = wrap(yl);
        if (row_bad(y)) return;
        R.template pull<WB>(A, row_off(fast, y), WB && y == 0, WB && !open_top && y == ny - 1);
    };
    // ring offsets of rows y-1, y, y+1 (slots given for the logical rows before
    // and after, which are y-1 and y+1 or the reverse)
    auto ring_off = [&](auto fast, int before, int own, int after, int y) {
        const int m_ = dir > 0 ? before : after;
        int p_ = dir > 0 ? after : before;
        if (!decltype(fast)::value && open_top && y == ny - 1) p_ = own;
        return PullOff{unsigned(m_ - 4), unsigned(m_), unsigned(m_ + 4), unsigned(own - 4), unsigned(own),
                       unsigned(own + 4), unsigned(p_ - 4), unsigned(p_), unsigned(p_ + 4)};
    };
    // The phi stencil over the rows before, own and after.  With "after" for
    // north and dir = -1 every term but grad_y has the same bits (its sums pair
    // the same values), and grad_y the opposite sign (sgn * g + 0 keeps a zero
    // positive).
    struct Row3 {
        float w, c, e;
    };
    const float sgn = dir > 0 ? 1.f : -1.f;
    auto stencil_rows = [&](auto fast, Row3 b, Row3 c, Row3 a, int y) {
        if (W && !decltype(fast)::value) {  // the ghost row repeats the edge row
            if (y == (dir > 0 ? 0 : ny - 1)) b = c;
            if (y == (dir > 0 ? ny - 1 : 0)) a = c;
        }
        Stencil st = stencil<MARCH_PK>(c.c, c.e, c.w, a.c, b.c, a.e, a.w, b.w, b.e);
        st.gy = fma_rn(sgn, st.gy, 0.f);
        return st;
    };

    const int first = dir > 0 ? y0 - 3 : y1 + 2;
    const int iters = rows + 7;
    int e0 = 0, e1 = 4 * S::SLOT, e2 = 3 * S::SLOT, e3 = 2 * S::SLOT, e4 = S::SLOT;  // ring rows t .. t-4 (mod 5)
    int a0 = 0, a1 = 2 * LP, a2 = LP;  // phi rows, newest first (mod 3)
    char* const phis = sx + S::PHI + (STEP == 1 ? 0 : 3) * LP;
    char* const ring = sx + S::RING;
    auto row3 = [](const char* q) { return Row3{sh<float>(q - 4), sh<float>(q), sh<float>(q + 4)}; };
    // the barriers of this step's threads and of the whole block (named, as the
    // two sets reach them in different code)
    auto sync_set = [] { asm volatile("bar.sync %0, %1;" ::"n"(STEP), "n"(TW) : "memory"); };
    auto sync_block = [] { asm volatile("bar.sync 3, %0;" ::"n"(2 * TW) : "memory"); };
    auto rotate = [&] {
        const int p = a2;
        a2 = a1;
        a1 = a0;
        a0 = p;
        const int s = e4;
        e4 = e3;
        e3 = e2;
        e2 = e1;
        e1 = e0;
        e0 = s;
    };
    // collides the pulled row R, grid row y, between phi rows b and a
    auto collide_row = [&](auto fast, const Row& R, Row3 b, Row3 c, Row3 a, int y, bool own, float f[9], float g[9],
                           float& phi) {
        R.values(f, g);
        phi = c.c;
        const Stencil st = stencil_rows(fast, b, c, a, y);
        const Macro M = macro_from<MARCH_PK>(m, Pop<ST>::template gmom<MARCH_PK>(g), phi, st.gx, st.gy, st.lap);
        if constexpr (CHK)
            if (own && m.check_nonfinite && !isfinite(add(add(phi, M.ux), add(M.uy, M.p)))) report_nonfinite(A.flag);
        return collide_st<ST, MARCH_PK>(m, f, g, phi, st, M, R.prev);
    };
    std::false_type edge;
    std::true_type inner;

    if constexpr (STEP == 1) {
        // cur: row t-1, which collides; nxt: row t.  fast: every part of the
        // iteration has its row
        auto body = [&](auto fast, Row& cur, Row& nxt, int t) {
            constexpr bool F = decltype(fast)::value;
            const int yt = first + dir * t, yb = yt - dir, yn = yt + dir;
            if (F || takes(3, t, yt)) sh<float>(phis + a0) = nxt.phi();
            sync_set();
            if (F || takes(2, t - 1, yb)) {
                float f[9], g[9], phi;
                const float2 pu = collide_row(fast, cur, row3(phis + a2), row3(phis + a1), row3(phis + a0), yb,
                                              out && yb >= y0 && yb < y1, f, g, phi);
                Row::template put_ring<LP>(ring + e1, f, g, phi, pu, (unsigned)(wrap(yb) * nx + x), m.seed);
            }
            if (F || takes(3, t + 1, yn)) load(fast, cur, yn);
            sync_block();
            rotate();
        };
        Row A0, A1;
        if (takes(3, 0, first)) load(edge, A1, first);
        // iterations whose rows t-1 .. t+1 all take part and touch no boundary
        const int f_hi = W ? (dir > 0 ? min(y1 + 2, ny - 2) - first : first - max(y0 - 3, 1)) - 1 : rows + 4;
        const int f_lo = W ? max(2, (dir > 0 ? 1 - first : first - (ny - 2)) + 1) : 2;
        for (int t = 0; t < iters; t += 2) {
            if (t >= f_lo && t + 1 <= f_hi) {
                body(inner, A0, A1, t);
                body(inner, A1, A0, t + 1);
            } else {
                body(edge, A0, A1, t);
                if (t + 1 < iters) body(edge, A1, A0, t + 1);
            }
        }
    } else {
        auto body = [&](auto fast, int t) {
            constexpr bool F = decltype(fast)::value, WB = W && !F;
            const int yt = first + dir * t, ya = yt - 3 * dir, yc = yt - 4 * dir;
            if (F || takes(1, t - 3, ya)) {
                Row R;
                R.template pull_ring_phi<WB, LP>(ring, ring_off(fast, e4, e3, e2, ya), WB && ya == 0,
                                                 WB && !open_top && ya == ny - 1);
                sh<float>(phis + a0) = R.phi();
            }
            sync_set();
            if (F || takes(0, t - 4, yc)) {
                Row R;
                R.template pull_ring<WB, LP>(ring, ring_off(fast, e0, e4, e3, yc), WB && yc == 0,
                                             WB && !open_top && yc == ny - 1);
                float f[9], g[9], phi;
                const float2 pu = collide_row(fast, R, row3(phis + a2), row3(phis + a1), row3(phis + a0), yc, out, f,
                                              g, phi);
                if (out) Row::put(A, pitch * yc + xc, f, g, phi, pu, seed2);
            }
            sync_block();
            rotate();
        };
        // iterations whose rows t-4, t-3 take part and touch no boundary
        const int f_hi = (W ? (dir > 0 ? min(y1 - 1, ny - 3) - first : first - max(y0, 2)) : rows + 2) + 4;
        const int f_lo = W ? max(7, (dir > 0 ? 1 - first : first - (ny - 2)) + 4) : 7;
        for (int t = 0; t < iters; ++t) {
            if (t >= f_lo && t <= f_hi)
                body(inner, t);
            else
                body(edge, t);
        }
    }
}

}  // namespace lbmpf
