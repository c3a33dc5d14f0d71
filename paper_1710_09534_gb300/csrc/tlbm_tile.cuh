// One launch per time step for lattices that leave the marching kernel and
// its near-wall companion bound by latency.
//
//   k_step_march  large lattices (below)
//   k_step_tile  every node of a 32 x TY tile, one thread each, near-wall and
//                lid nodes included: c_1, c_2 and the node classes of the tile
//                plus two nodes around it go to shared memory once, the column
//                sums and mu of the tile plus one node around it are formed
//                from them, and every node then takes the update its class
//                asks for.
//
// The marching kernel serialises the rows of a segment, and a thread of the
// former near-wall kernel summed the order parameters of its whole 5x5 window
// by itself (450 loads and, in FP64, 25 times the additions; an FP64
// instruction of a warp takes 64 cycles of its scheduler on GB300, however few
// lanes are active).  On a large lattice neither shows; on a small one a step
// lasted as long as one segment and one such window.  Here every c is summed
// once per tile, and the launches of successive steps overlap
// (programmatic dependent launch: a block classifies its sites while the
// previous step finishes, then waits for it; 128x64 FP32 6.2 -> 3.7 us per
// step).  GB300, us per step, the two kernels against this one: 128x64 FP64
// 45.2 -> 13.4, FP32 13.5 -> 3.7; 512x256 with a lid FP32 20.6 -> 9.3.
//
// The arithmetic of every node is that of the other two kernels, operation by
// operation: interior nodes use the column sums (ColRings), the others the
// window form with the ghost rules of Eqs. 42-43 (window_macros), whose mu is
// kept apart (wm) because it rounds differently from the column form.  Near-wall
// nodes of a lattice of uniform properties take the general update in FP32
// arithmetic and the uniform one in FP64.
#pragma once
#include "tlbm_kernels.cuh"

namespace tlb {

template <typename R, int TY>
struct TileShared {
    using V = typename Vec2T<R>::type;
    static constexpr int CW = 36, CH = TY + 4, MW = 34, MH = TY + 2;
    V c[CH][CW];           // (c_1, c_2) of nodes x0 - 2 .., y0 - 2 ..; zero unless plain fluid
    V A[MH][CW], D[MH][CW];  // column sums of rows y0 - 1 .. (see ColRings)
    V mu[MH][MW];          // mu of nodes x0 - 1 .., y0 - 1 .., column form
    V wm[MH][MW];          // the same in the window form, where a near-wall node may read it
    V M[TY][MW];           // column sums of mu (general update)
    uint8_t k[CH][CW];     // node class, or the site kind of a node outside the lattice
};

// c and (window form) mu of shared node (i, j); the lid row carries those of
// the row below it (Eqs. 51-53).
template <typename R, int TY>
__device__ __forceinline__ auto tile_c(const TileShared<R, TY>& sh, int i, int j)
{
    return sh.c[j - ((sh.k[j][i] & CLS_KIND_MASK) == ST_LID ? 1 : 0)][i];
}

// mu of mu-node (i, j) in the window form: Eq. 8 with the wetting ghosts of Eq.
// 42 (zero unless plain fluid).
template <typename R, int TY>
__device__ __forceinline__ typename TileShared<R, TY>::V tile_window_mu(const TileShared<R, TY>& sh, const Prm<R>& P,
                                                                       int i, int j)
{
    using V = typename TileShared<R, TY>::V;
    R mu1 = R(0), mu2 = R(0);
    if ((sh.k[j + 1][i + 1] & CLS_KIND_MASK) == ST_FLUID) {
        const V c = sh.c[j + 1][i + 1];
        R o1, o2;
        wet_offset(P, c.x, c.y, o1, o2);
        R v1[9], v2[9];
        v1[0] = c.x;
        v2[0] = c.y;
#pragma unroll
        for (int k = 1; k < 9; k++) {
            const int s = sh.k[j + 1 + ey(k)][i + 1 + ex(k)] & CLS_KIND_MASK;
            if (fluidlike(s)) {
                const V v = tile_c(sh, i + 1 + ex(k), j + 1 + ey(k));
                v1[k] = v.x;
                v2[k] = v.y;
            } else if (s == ST_WET) {
                v1[k] = c.x + o1;
                v2[k] = c.y + o2;
            } else {
                v1[k] = c.x;
                v2[k] = c.y;
            }
        }
        chem_pot(P, c.x, c.y, lap9s(v1), lap9s(v2), mu1, mu2);
    }
    return V{mu1, mu2};
}

// Macros of the near-wall or lid-adjacent node at shared position (i, j):
// window_macros with the window in shared memory.
template <bool UNI, typename R, int TY>
__device__ __forceinline__ void tile_macros(const TileShared<R, TY>& sh, const Prm<R>& P, int i, int j, Macro<R>& m)
{
    R v1[9], v2[9], w1[9], w2[9];
#pragma unroll
    for (int k = 0; k < 9; k++) {
        int ii = i + ex(k), jj = j + ey(k);
        const int s = k == 0 ? int(ST_FLUID) : sh.k[jj][ii] & CLS_KIND_MASK;
        if (!fluidlike(s)) {  // Eq. 43
            ii = i;
            jj = j;
        } else if (s == ST_LID) {
            jj--;
        }
        const auto c = sh.c[jj][ii];
        const auto w = sh.wm[jj - 1][ii - 1];
        v1[k] = c.x;
        v2[k] = c.y;
        w1[k] = w.x;
        w2[k] = w.y;
    }
    m.c1 = v1[0];
    m.c2 = v2[0];
    m.mu1 = w1[0];
    m.mu2 = w2[0];
    grad9s(v1, m.g1x, m.g1y);
    grad9s(v2, m.g2x, m.g2y);
    if constexpr (UNI) {
        m.lm1 = m.lm2 = R(0);
        m.rho = P.rho[2];
    } else {
        m.lm1 = lap9s(w1);
        m.lm2 = lap9s(w2);
        m.rho = density(P, m.c1, m.c2);
    }
}

// Class byte of site (x, y) (on an inside site with its wrapped offset), or
// the kind of an outside one; sites further than two nodes outside are never
// read.
__device__ __forceinline__ int tile_site(const Geo& g, const uint8_t* __restrict__ cls, int x, int y, long long& off)
{
    if (x > g.nx + 1 || y < -2 || y > g.ny + 1) return ST_VOID;
    const int s = site_of(g, cls, x, y, off);
    return s == ST_FLUID ? cls[off] : s;
}

// One tile with its first node at (x0, y0).  WALL: its near-wall and lid nodes
// only (interior nodes lend their c).
template <typename S, typename R, int TY, bool MRT, bool UNI, bool WALL>
__device__ __forceinline__ void tile_step(const S* fA, S* fB, CuT<S>* cu,
                                          const uint8_t* __restrict__ cls, const Geo& g, const Prm<R>& P, int x0,
                                          int y0, TileShared<R, TY>& sh)
{
    using T = TileShared<R, TY>;
    using V = typename T::V;
    constexpr int NT = 32 * TY;
    constexpr int SE = (Store<S>::k16 && !MRT) ? Store<S>::kScaleExp : 0;
    constexpr R unscale = R(1.0 / double(1 << SE));
    const long long PL = g.plane;
    const int t = threadIdx.x, tx = t & 31, ty = t >> 5;
    const int x = x0 + tx, y = y0 + ty;
    const bool own = x < g.nx && y >= 0 && y < g.ny;
    const long long o = own ? (long long)y * g.pitch + x : 0;

    // class and place of the frame of two nodes around the tile (2 x 2 rows of
    // 36, then TY rows of 4) and of the thread's own site
    constexpr int FRAME = 4 * T::CW + 4 * TY, ROUNDS = (FRAME + NT - 1) / NT;
    int fs[ROUNDS], fi[ROUNDS], fj[ROUNDS];
    long long fo[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        const int n = r * NT + t;
        int i, j;
        if (n < 4 * T::CW) {
            j = n / T::CW;
            i = n - j * T::CW;
            j += j >= 2 ? TY : 0;
        } else {
            j = (n - 4 * T::CW) >> 2;
            i = (n - 4 * T::CW) & 3;
            j += 2;
            i += i >= 2 ? 32 : 0;
        }
        fi[r] = i;
        fj[r] = j;
        fo[r] = 0;
        fs[r] = ST_VOID;
        if (n < FRAME) fs[r] = tile_site(g, cls, x0 - 2 + i, y0 - 2 + j, fo[r]);
    }
    long long oo = 0;
    const int mine = tile_site(g, cls, x, y, oo);
    // the state is that of the previous launch, which may still be running
    // (programmatic dependent launch); the next one may start its own prologue
    if constexpr (!WALL) after_previous_launch();

    // the thread's own node: everything its update reads, and its c
    R f[18], lo[2] = {R(0), R(0)}, gv[9], cp[4];
    if (own) {
        f[0] = ld_pop<R, false>(fA, 0, PL, o);
        f[9] = ld_pop<R, false>(fA, 9, PL, o);
#pragma unroll
        for (int k = 1; k < 9; k++) ld_pair<R, false, SE != 0>(fA, k, PL, o, f[k], f[9 + k]);
        lo[0] = ld_lo<R, false>(fA, 0, PL, o);
        lo[1] = ld_lo<R, false>(fA, 1, PL, o);
        if (!WALL || !(mine & CLS_INTERIOR)) {
#pragma unroll
            for (int k = 0; k < 9; k++) gv[k] = ld_pop<R, false, SE != 0>(fA, 18 + k, PL, o);
#pragma unroll
            for (int q = 0; q < 4; q++) cp[q] = R(cu[q * PL + o]);
        }
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        if (r * NT + t < FRAME) {
            V c{R(0), R(0)};
            if ((fs[r] & CLS_KIND_MASK) == ST_FLUID) {
                R a, b;
                order_params<R, false>(fA, PL, fo[r], a, b);
                c = V{a, b};
            }
            sh.c[fj[r]][fi[r]] = c;
            sh.k[fj[r]][fi[r]] = (uint8_t)fs[r];
        }
    }
    {
        V c{R(0), R(0)};
        if ((mine & CLS_KIND_MASK) == ST_FLUID) {
            if (own) {
                const R f10 = f[0], f20 = f[9];
                if constexpr (Store<S>::kLo) {
                    f[0] += lo[0];
                    f[9] += lo[1];
                }
                c = V{sum9s<SE>(f), sum9s<SE>(f + 9)};
                f[0] = f10;
                f[9] = f20;
            } else {
                R a, b;
                order_params<R, false>(fA, PL, oo, a, b);
                c = V{a, b};
            }
        }
        sh.c[ty + 2][tx + 2] = c;
        sh.k[ty + 2][tx + 2] = (uint8_t)mine;
    }
    __syncthreads();
    // column sums of rows y0 - 1 .. y0 + TY
    if constexpr (!WALL) {
        for (int n = t; n < T::MH * T::CW; n += NT) {
            const int j = n / T::CW, i = n - j * T::CW;
            const V b = sh.c[j][i], c = sh.c[j + 1][i], a = sh.c[j + 2][i];
            sh.A[j][i] = V{fma(R(4), c.x, b.x + a.x), fma(R(4), c.y, b.y + a.y)};
            sh.D[j][i] = V{a.x - b.x, a.y - b.y};
        }
        __syncthreads();
    }
    // mu of the tile plus one node (Eq. 8 with Eq. 20b)
    for (int n = t; n < T::MH * T::MW; n += NT) {
        const int j = n / T::MW, i = n - j * T::MW;
        if constexpr (!WALL) {
            const V c = sh.c[j + 1][i + 1];
            R mu1, mu2;
            const V cb = sh.c[j][i + 1], ca = sh.c[j + 2][i + 1];
            const V al = sh.A[j][i], ar = sh.A[j][i + 2];
            chem_pot(P, c.x, c.y, fma(R(4), fma(R(-5), c.x, cb.x + ca.x), al.x + ar.x),
                     fma(R(4), fma(R(-5), c.y, cb.y + ca.y), al.y + ar.y), mu1, mu2);
            sh.mu[j][i] = V{mu1, mu2};
        }
        // the window form where a near-wall node may read it
        int all = CLS_INTERIOR;
#pragma unroll
        for (int k = 0; k < 9; k++) all &= sh.k[j + 1 + ey(k)][i + 1 + ex(k)];
        if (!all) sh.wm[j][i] = tile_window_mu(sh, P, i, j);
    }
    __syncthreads();
    if constexpr (!UNI && !WALL) {
        for (int n = t; n < TY * T::MW; n += NT) {
            const int j = n / T::MW, i = n - j * T::MW;
            const V b = sh.mu[j][i], c = sh.mu[j + 1][i], a = sh.mu[j + 2][i];
            sh.M[j][i] = V{fma(R(4), c.x, b.x + a.x), fma(R(4), c.y, b.y + a.y)};
        }
        __syncthreads();
    }
    if (!own) return;
    const int kind = mine & CLS_KIND_MASK;
    const PushOffsets po(g, x, y);

    // Interior nodes with an update of their own (FP32 arithmetic: the uniform-
    // property form, and the units of 16-bit storage): near-wall nodes take the
    // general one below.
    constexpr bool kSplit = (UNI && !kLean<R>) || SE != 0 || WALL;
    constexpr bool kUniWall = UNI && kLean<R>;
    const bool inner = (mine & CLS_INTERIOR) != 0;
    if (WALL && inner) return;
    Macro<R> m;
    if (!WALL && inner) {
        // column sums: operation by operation as in the marching kernel
        const V c = sh.c[ty + 2][tx + 2], w = sh.mu[ty + 1][tx + 1];
        m.c1 = c.x;
        m.c2 = c.y;
        m.mu1 = w.x;
        m.mu2 = w.y;
        const V al = sh.A[ty + 1][tx + 1], ar = sh.A[ty + 1][tx + 3];
        const V dl = sh.D[ty + 1][tx + 1], dc = sh.D[ty + 1][tx + 2], dr = sh.D[ty + 1][tx + 3];
        m.g1x = ar.x - al.x;
        m.g2x = ar.y - al.y;
        m.g1y = fma(R(4), dc.x, dl.x + dr.x);
        m.g2y = fma(R(4), dc.y, dl.y + dr.y);
        if constexpr (UNI) {
            m.lm1 = m.lm2 = R(0);
        } else {
            const V wb = sh.mu[ty][tx + 1], wa = sh.mu[ty + 2][tx + 1], ml = sh.M[ty][tx], mr = sh.M[ty][tx + 2];
            m.lm1 = fma(R(4), fma(R(-5), w.x, wb.x + wa.x), ml.x + mr.x);
            m.lm2 = fma(R(4), fma(R(-5), w.y, wb.y + wa.y), ml.y + mr.y);
        }
        m.rho = UNI ? P.rho[2] : density(P, m.c1, m.c2);
    }
    if constexpr (kSplit && !WALL) {
        if (inner) {
            Hydro<R> h;
            hydro_from_g<UNI, SE>(P, m, gv, h);
            const R c1ux = m.c1 * h.ux, c1uy = m.c1 * h.uy, c2ux = m.c2 * h.ux, c2uy = m.c2 * h.uy;
            cu[0 * PL + o] = CuT<S>(c1ux);
            cu[1 * PL + o] = CuT<S>(c1uy);
            cu[2 * PL + o] = CuT<S>(c2ux);
            cu[3 * PL + o] = CuT<S>(c2uy);
            CollideOf<S, MRT, R, UNI> col;
            col.template build<SE>(P, m, h, cp[0], cp[1], cp[2], cp[3]);
            collide_all<S, R, SE>(col, gv,
                [&](auto kc, R& f1k, R& f2k) {
                    f1k = f[decltype(kc)::value];
                    f2k = f[9 + decltype(kc)::value];
                },
                [&](R& l1, R& l2) {
                    l1 = lo[0];
                    l2 = lo[1];
                },
                [&](auto kc, auto o1, auto o2, auto og) {
                    constexpr int K = decltype(kc)::value;
                    st_three(fB, K, PL, K == 0 ? o : po.template dest<K>(), o1, o2, og);
                },
                [&](R l1, R l2) {
                    st_lo(fB, 0, PL, o, l1);
                    st_lo(fB, 1, PL, o, l2);
                });
            return;
        }
    }
    if (!fluidlike(kind)) return;

    // near-wall and lid nodes (wall_node with its window in shared memory) and,
    // where the update is the same, interior ones: a warp that holds both kinds
    // runs it once.  A lid node takes the macros of the row below it.
    const bool lid = kind == ST_LID;
    if (kSplit || !inner) tile_macros<kUniWall>(sh, P, tx + 2, ty + 2 - lid, m);
    const long long of = lid ? o - g.pitch : o;
    if (lid) {
#pragma unroll
        for (int k = 0; k < 9; k++) gv[k] = ld_pop<R, false>(fA, 18 + k, PL, of);
    } else if constexpr (SE != 0) {
#pragma unroll
        for (int k = 0; k < 9; k++) gv[k] *= unscale;
#pragma unroll
        for (int k = 1; k < 9; k++) {
            f[k] *= unscale;
            f[9 + k] *= unscale;
        }
    }
    Hydro<R> h;
    hydro_from_g<kUniWall>(P, m, gv, h);
    if (lid) {
        // Eq. 51: f(x_u) = f^eq(x_u) + [f(x_f) - f^eq(x_f)], for f^1, f^2 and g
        const R fx = h.ux, fy = h.uy;
        h.ux = P.lid_u;
        h.uy = R(0);
        h.usq = P.lid_u * P.lid_u;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            R e1u, e2u, egu, e1f, e2f, egf;
            equilibria(k, P, m.c1, m.c2, m.mu1, m.mu2, m.rho, h.p, h.ux, h.uy, e1u, e2u, egu);
            equilibria(k, P, m.c1, m.c2, m.mu1, m.mu2, m.rho, h.p, fx, fy, e1f, e2f, egf);
            R ff1 = ld_pop<R, false>(fA, k, PL, of), ff2 = ld_pop<R, false>(fA, 9 + k, PL, of);
            if constexpr (Store<S>::kLo) {
                if (k == 0) {
                    ff1 += ld_lo<R, false>(fA, 0, PL, of);
                    ff2 += ld_lo<R, false>(fA, 1, PL, of);
                }
            }
            f[k] = e1u + (ff1 - e1f);
            f[9 + k] = e2u + (ff2 - e2f);
            gv[k] = egu + (gv[k] - egf);
        }
        lo[0] = lo[1] = R(0);
    }
    const R c1ux = m.c1 * h.ux, c1uy = m.c1 * h.uy, c2ux = m.c2 * h.ux, c2uy = m.c2 * h.uy;
    cu[0 * PL + o] = CuT<S>(c1ux);
    cu[1 * PL + o] = CuT<S>(c1uy);
    cu[2 * PL + o] = CuT<S>(c2ux);
    cu[3 * PL + o] = CuT<S>(c2uy);
    CollideOf<S, MRT, R, kUniWall> col;
    col.build(P, m, h, cp[0], cp[1], cp[2], cp[3]);
    collide_all<S, R>(col, gv,
        [&](auto kc, R& f1k, R& f2k) {
            f1k = f[decltype(kc)::value];
            f2k = f[9 + decltype(kc)::value];
        },
        [&](R& l1, R& l2) {
            l1 = lo[0];
            l2 = lo[1];
        },
        [&](auto kc, auto o1, auto o2, auto og) {
            constexpr int K = decltype(kc)::value;
            if constexpr (K == 0) {
                st_three(fB, 0, PL, o, o1, o2, og);
            } else {
                const int s = sh.k[ty + 2 + ey(K)][tx + 2 + ex(K)] & CLS_KIND_MASK;
                if (fluidlike(s)) st_three(fB, K, PL, po.template dest<K>(), o1, o2, og);
                else if (s != ST_VOID) st_three(fB, opp(K), PL, o, o1, o2, og);  // Eq. 44
                // slots fed from beyond the lid receive nothing: keep them zero
                if (ey(K) == -1 && lid && (sh.k[ty + 3][tx + 2 - ex(K)] & CLS_KIND_MASK) == ST_VOID) {
                    st_pop(fB, K, PL, o, R(0));
                    st_pop(fB, 9 + K, PL, o, R(0));
                    st_pop(fB, 18 + K, PL, o, R(0));
                }
            }
        },
        [&](R l1, R l2) {
            st_lo(fB, 0, PL, o, l1);
            st_lo(fB, 1, PL, o, l2);
        });
}


// ---------------------------------------------------------------------------
// Read-out of macroscopic fields as FP64 planes (order c1 c2 c3 rho ux uy p
// mu1 mu2 mu3, only the planes selected by `mask`), by tiles: every node in the
// window form (window_macros, operation by operation), with the order
// parameters and mu of the tile formed once in shared memory.  With a window
// per thread each order parameter was summed by 25 threads: GB300, 5 planes of
// 2048^2, FP64 2837 -> 1266 us, FP32 338 -> 158.
// ---------------------------------------------------------------------------
template <typename S, typename R, int TY>
__global__ void __launch_bounds__(32 * TY)
k_read_fields(const S* __restrict__ fA, const uint8_t* __restrict__ cls, double* __restrict__ out, uint32_t mask, Geo g,
              Prm<R> P, int yshift)
{
    using T = TileShared<R, TY>;
    using V = typename T::V;
    __shared__ T sh;
    constexpr int NT = 32 * TY;
    const long long PL = g.plane;
    const int t = threadIdx.x, tx = t & 31, ty = t >> 5;
    const int x0 = blockIdx.x * 32, y0 = (int)blockIdx.y * TY - yshift;
    for (int n = t; n < T::CH * T::CW; n += NT) {
        const int j = n / T::CW, i = n - j * T::CW;
        long long off = 0;
        const int s = tile_site(g, cls, x0 - 2 + i, y0 - 2 + j, off);
        V c{R(0), R(0)};
        if ((s & CLS_KIND_MASK) == ST_FLUID) {
            R a, b;
            order_params<R>(fA, PL, off, a, b);
            c = V{a, b};
        }
        sh.c[j][i] = c;
        sh.k[j][i] = (uint8_t)s;
    }
    __syncthreads();
    for (int n = t; n < T::MH * T::MW; n += NT) {
        const int j = n / T::MW, i = n - j * T::MW;
        sh.wm[j][i] = tile_window_mu(sh, P, i, j);
    }
    __syncthreads();
    const int x = x0 + tx, y = y0 + ty;
    if (x >= g.nx || y < 0 || y >= g.ny) return;
    const int kind = sh.k[ty + 2][tx + 2] & CLS_KIND_MASK;
    double v[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (fluidlike(kind)) {
        // the lid row reads the row below it with u = (U0, 0)
        const int lid = kind == ST_LID;
        const long long of = (long long)(y - lid) * g.pitch + x;
        Macro<R> m;
        tile_macros<false>(sh, P, tx + 2, ty + 2 - lid, m);
        R gv[9];
#pragma unroll
        for (int k = 0; k < 9; k++) gv[k] = ld_pop<R>(fA, 18 + k, PL, of);
        Hydro<R> h;
        hydro_from_g(P, m, gv, h);
        if (lid) {
            h.ux = P.lid_u;
            h.uy = R(0);
        }
        v[0] = m.c1;
        v[1] = m.c2;
        v[2] = R(1) - m.c1 - m.c2;
        v[3] = m.rho;
        v[4] = h.ux;
        v[5] = h.uy;
        v[6] = h.p;
        v[7] = m.mu1;
        v[8] = m.mu2;
        v[9] = -fma(P.l3_l1, m.mu1, P.l3_l2 * m.mu2);
    }
    const long long n = (long long)y * g.nx + x, N = (long long)g.nx * g.ny;
    int plane = 0;
#pragma unroll
    for (int q = 0; q < 10; q++) {
        if (mask & (1u << q)) {
            out[plane * N + n] = v[q];
            plane++;
        }
    }
}

template <typename S, typename R, int TY, int MINB, bool MRT, bool UNI>
__global__ void __launch_bounds__(32 * TY, MINB)
k_step_tile(const S* fA, S* fB, CuT<S>* cu, const uint8_t* __restrict__ cls, Geo g, Prm<R> P, int yshift, int first)
{
    __shared__ TileShared<R, TY> sh;
    int by = (int)blockIdx.y + first;  // rows of tiles from row `first` on, cyclically
    by -= by >= (int)gridDim.y ? (int)gridDim.y : 0;
    tile_step<S, R, TY, MRT, UNI, false>(fA, fB, cu, cls, g, P, blockIdx.x * 32, by * TY - yshift, sh);
}

// ---------------------------------------------------------------------------
// One near-wall tile: column bx, row by of the tiles of 32 x TY nodes from row
// -tile_shift on.  A call of its own, so that its registers are not those of
// the interior update that shares its kernel (inlined into the batch kernel,
// FP64 spilled 40 words and FP16 100).
// ---------------------------------------------------------------------------
template <typename S, typename R, int TY, bool MRT>
__device__ __noinline__ void wall_tile(const S* fA, S* fB, CuT<S>* cu, const uint8_t* cls, const Geo& g, const Prm<R>& P,
                                       int bx, int by, TileShared<R, TY>& sh)
{
    fA = global_ptr(fA);
    fB = global_ptr(fB);
    cu = global_ptr(cu);
    const int y0 = by * TY - tile_shift(g.edge[3] == EDGE_LID, g.ny, TY);
    if (kLean<R> && P.uni != R(0))
        tile_step<S, R, TY, MRT, kLean<R>, true>(fA, fB, cu, cls, g, P, bx * 32, y0, sh);
    else
        tile_step<S, R, TY, MRT, false, true>(fA, fB, cu, cls, g, P, bx * 32, y0, sh);
}

// Shared data of a block that takes either kind of work.
template <typename R, int BLOCK, bool STASH>
union __align__(16) MarchShared {
    struct {
        ColRings<R, BLOCK> rings;
        PopStash<R, STASH ? BLOCK : 1> stash;
    } m;
    TileShared<R, BLOCK / 32> tile;
    __device__ MarchShared() {}
};

// One step of a large lattice: block b < nwalls takes near-wall tile walls[b]
// ((row << 16) | column, tiles of 32 x kWallTY nodes: short, because the
// near-wall nodes of a straight wall are two rows), the others a strip segment
// of the interior (interior_tile).  One launch, which overlaps the end of the
// step before it; as two launches on two streams between events, GB300, us per
// step: 2048^2 FP32 209.0 -> 200.1, FP16 149.8 -> 142.4, 1024x2048
// impact FP32 113.1 -> 110.5.  With plain loads (see after_previous_launch) and
// the overlap, against loads through the read-only path without it: 2048^2 FP64
// 1804 -> 1791, FP32 205 -> 202, 1024x2048 impact FP32 115 -> 113; 16-bit storage
// see kPipeG16.
template <typename S, typename R, int BLOCK, bool PREFETCH, int MINB, bool MRT, bool UNI>
__global__ void __launch_bounds__(BLOCK, MINB)
k_step_march(const S* fA, S* fB, CuT<S>* cu, const uint8_t* __restrict__ cls,
             const uint32_t* __restrict__ walls, int nwalls, int strips, const __grid_constant__ Geo g,
             const __grid_constant__ Prm<R> P, int rows)
{
    constexpr bool kStash = kStashPops && std::is_same<R, float>::value && !kDenseMrt<S, MRT>;
    __shared__ MarchShared<R, BLOCK, kStash> sh;
    after_previous_launch();
    const int b = (int)blockIdx.x - nwalls;
    if (b < 0) {
        const uint32_t w = walls[blockIdx.x];
        wall_tile<S, R, BLOCK / 32, MRT>(fA, fB, cu, cls, g, P, (int)(w & 0xffffu), (int)(w >> 16), sh.tile);
        return;
    }
    auto* st = reinterpret_cast<PopStash<R, BLOCK>*>(&sh.m.stash);  // used only when kStash
    interior_tile<S, R, BLOCK, PREFETCH, MRT, UNI, kStash>(fA, fB, cu, cls, g, P, b % strips, b / strips, rows,
                                                           sh.m.rings, st);
}

}  // namespace tlb
