// Launchers of one precision; included by tlbm_f64.cu and tlbm_f32.cu.
#pragma once
#include "tlbm_batch.cuh"
#include "tlbm_inplace.cuh"
#include "tlbm_kernels.cuh"
#include "tlbm_ops.h"
#include "tlbm_tile.cuh"
#include <cmath>

namespace tlb {

template <typename R>
inline Prm<R> cast_prm(const Prm<double>& d)
{
    Prm<R> r;
    for (int i = 0; i < 3; i++) {
        r.lam[i] = R(d.lam[i]);
        r.rho[i] = R(d.rho[i]);
        r.nu[i] = R(d.nu[i]);
    }
    for (int i = 0; i < 2; i++) {
        r.k34Dlam[i] = R(d.k34Dlam[i]);
        r.eta[i] = R(d.eta[i]);
        r.inv_tau[i] = R(d.inv_tau[i]);
        r.omt[i] = R(d.omt[i]);
        r.e0[i] = R(d.e0[i]);
        r.rate[i] = R(d.rate[i]);
        r.kj[i] = R(d.kj[i]);
        r.drho[i] = R(d.drho[i]);
        r.dnu[i] = R(d.dnu[i]);
        r.aM[i] = R(d.aM[i]);
        for (int c = 0; c < 2; c++) {
            r.aw[i][c] = R(d.aw[i][c]);
        }
    }
    r.lamT = R(d.lamT);
    r.two_lamT = R(d.two_lamT);
    r.k12D = R(d.k12D);
    r.k34D = R(d.k34D);
    r.k4D = R(d.k4D);
    r.l3_l1 = R(d.l3_l1);
    r.l3_l2 = R(d.l3_l2);
    r.cos12 = R(d.cos12);
    r.cos13 = R(d.cos13);
    r.cos23 = R(d.cos23);
    r.gx = R(d.gx);
    r.gy = R(d.gy);
    r.lid_u = R(d.lid_u);
    r.mrt = R(d.mrt);
    r.mrt_s_f = R(d.mrt_s_f);
    r.mrt_s_g = R(d.mrt_s_g);
    r.uni = R(d.uni);
    r.inv_rho3 = R(d.inv_rho3);
    r.inv_taug3 = R(d.inv_taug3);
    r.omtg3 = R(d.omtg3);
    r.kG3 = R(d.kG3);
    for (int c = 0; c < 2; c++) {
        r.Rw3[c] = R(d.Rw3[c]);
        r.Kw3[c] = R(d.Kw3[c]);
    }
    r.p3tg3 = R(d.p3tg3);
    r.rg3x = R(d.rg3x);
    r.rg3y = R(d.rg3y);
    for (int i = 0; i < 2; i++) {
        r.Kl[i] = R(d.Kl[i]);
        r.K34l6[i] = R(d.K34l6[i]);
        r.drho12[i] = R(d.drho12[i]);
        r.aM6[i] = R(d.aM6[i]);
        r.kq[i] = R(d.kq[i]);
        r.ks[i] = R(d.ks[i]);
        r.K3w3[i] = R(d.K3w3[i]);
        r.kqs[i] = R(d.kqs[i]);
        r.Kl1[i] = R(d.Kl1[i]);
        r.Kl2[i] = R(d.Kl2[i]);
        r.Kl3[i] = R(d.Kl3[i]);
        r.qa[i][0] = R(d.qa[i][0]);
        r.qa[i][1] = R(d.qa[i][1]);
    }
    r.Kt = R(d.Kt);
    r.rho23 = R(d.rho23);
    r.kp3 = R(d.kp3);
    return r;
}

// Streaming multiprocessors of the current device (queried once per process).
inline int sm_count()
{
    static int n = 0;
    if (n <= 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 152;
    }
    return n;
}

// Row-segment length of a single-lattice interior launch: `rows`, halved (down
// to 4) while the grid would not fill every SM with `per_sm` resident blocks,
// so that a small lattice still spreads over the chip (the halo work per node
// grows, but idle SMs cost more).
#ifndef TLB_ADAPTIVE_ROWS
#define TLB_ADAPTIVE_ROWS 1
#endif
// one_wave (the FP64 interior kernels): a lattice large enough for
// more than one wave of blocks gets segments long enough that the whole grid
// is resident at once, so that the halo rows' c sums and chemical potentials
// (FP64 arithmetic, the kernel's bound) are repeated on fewer rows.  GB300:
// FP64 2048^2 interior kernel 1.929 -> 1.911 ms, 1024x2048 cylinder impact
// within +-3%.  FP32 and 16-bit storage (latency-bound) lose the dynamic
// balancing of several waves: the cylinder impact ran 12% (FP32) and 10%
// (FP16) slower, so they keep short segments.
#ifndef TLB_ONE_WAVE
#define TLB_ONE_WAVE 1
#endif
// Otherwise segments of 12 to 24 rows, of the length that wastes least: blocks
// come in waves of the resident ones, so w = blocks / resident of them last
// ceil(w) / w as long as full waves would, and the `halo` rows' loads are
// repeated per segment (16 rows unless another length saves 2%; halo = 0: no
// such choice).  GB300, us per step, 16 rows against this: FP32 2048^2 204.5,
// 201.9; 1800x1700 154.5, 149.5; 3000x2000 300, 292; FP16 1500x1300 88.0, 77.6;
// 1800x1700 119.6, 110.6; 1024x2048 impact 91.5, 87.4; in place FP32 2048x1024
// 168.5, 152.7; 1500x1300 165, 152.  In place with 16-bit storage it lost as
// often as it gained (2048x1024 123.6, 126.0; 2048^2 237.6, 231.5) and is off.
// In-place FP64 takes the one-wave rule, in which its halo is cheap (c comes
// from planes): 2048x1024 1016 -> 889.
// A lattice of less than one wave of 16-row segments takes shorter ones: of 4 to
// 15 rows (two buffers), the length with the fewest row iterations in all, waves
// times rows and halo; halving until the blocks exceed the resident ones could end
// just beyond a wave.  GB300, us per step, halving against this: FP32 777^2 44.9,
// 36.7; 500x1000 38.6, 30.4; 860^2 48.8, 42.5; FP16 860^2 33.2, 30.3; 1255x695 42.1, 36.5.
constexpr int kMarchHalo = 4;  // halo rows of a segment of k_step_march
inline int rows_for(const Geo& g, int tx, int rows, int per_sm, bool one_wave, int halo)
{
    if (!TLB_ADAPTIVE_ROWS) return rows;
    const int strips = (g.nx + tx - 1) / tx;
    if (TLB_ONE_WAVE && one_wave) {
        const long long segs = (long long)sm_count() * per_sm / strips;
        if (segs >= 1) {
            const int r = (int)((g.ny + segs - 1) / segs);
            if (r > rows) return r;
        }
    }
    const long long slots = (long long)sm_count() * per_sm;
    auto blocks = [&](int r) { return (long long)strips * ((g.ny + r - 1) / r); };
    if (halo > 0 && blocks(rows) >= slots) {
        auto cost = [&](int r) {
            const double w = (double)blocks(r) / slots;
            return std::ceil(w) / w * (r + halo) / r;
        };
        int best = rows;
        for (int r = 12; r <= 24; r++)
            if (cost(r) < 0.98 * cost(rows) && cost(r) < cost(best)) best = r;
        return best;
    }
    if (halo == kMarchHalo) {
        auto iterations = [&](int r) { return (blocks(r) + slots - 1) / slots * (r + halo); };
        int best = rows;
        for (int r = rows - 1; r >= 4; r--)
            if (iterations(r) < iterations(best)) best = r;
        return best;
    }
    while (rows > 4 && blocks(rows) < slots) rows /= 2;
    return rows;
}

// Resident blocks per SM of the FP64 BGK uniform-property interior kernel,
// which needs fewer registers than the general one: at 4 (128 registers, no
// spills) it measured slower than at 3 (GB300, 2048^2: 1.913 -> 1.947 ms).
#ifndef TLB_MINB64_UNI
#define TLB_MINB64_UNI 3
#endif

template <typename S, typename R, int BLOCK, int ROWS, bool PREFETCH, int MINB, bool MRT>
struct OpsImpl {
    static constexpr int kMinBUni = std::is_same<R, double>::value && !MRT ? TLB_MINB64_UNI : MINB;
    static cudaError_t march(const void* fA, void* fB, void* cu, const uint8_t* cls, const uint32_t* walls, int nwalls,
                             const Geo& g, const Prm<double>& Pd, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        constexpr int TX = BLOCK - 4;
        static_assert(BLOCK == 32 * kWallTY, "a block takes a strip segment or a near-wall tile");
        // equal densities and viscosities: the uniform-property update
        const bool uni = Pd.uni != 0.0;
        const int rows = rows_for(g, TX, ROWS, uni ? kMinBUni : MINB, std::is_same<R, double>::value, kMarchHalo);
        const int strips = (g.nx + TX - 1) / TX, segs = (g.ny + rows - 1) / rows;
        auto* k = uni ? &k_step_march<S, R, BLOCK, PREFETCH, kMinBUni, MRT, true>
                      : &k_step_march<S, R, BLOCK, PREFETCH, MINB, MRT, false>;
        return launch_dependent(k, dim3(nwalls + strips * segs), BLOCK, 0, s, (const S*)fA, (S*)fB, (CuT<S>*)cu, cls,
                                walls, nwalls, strips, g, P, rows);
    }
    template <int TY, int MB>
    static cudaError_t launch_tile(const void* fA, void* fB, void* cu, const uint8_t* cls, const Geo& g,
                                   const Prm<double>& Pd, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        const int shift = tile_shift(g.edge[3] == EDGE_LID, g.ny, TY);
        const dim3 grid((g.nx + 31) / 32, (g.ny + shift + TY - 1) / TY);
        // A row of tiles with a lid takes longest (its nodes run the lid's update
        // after that of the rows below).  Beyond one wave of blocks it goes first,
        // so that it is not what the step ends on: GB300, us per step, last against
        // first: sheared drop FP64 240x280 61.3, 53.3; 320x400 97.4, 86.5; FP32
        // 512x256 9.7, 9.3.  Within one wave it stays last (FP64 160x160 26.7, 35.6).
        const bool lid = g.edge[3] == EDGE_LID && (long long)grid.x * grid.y > (long long)sm_count() * MB;
        auto* k = Pd.uni != 0.0 ? &k_step_tile<S, R, TY, MB, MRT, true> : &k_step_tile<S, R, TY, MB, MRT, false>;
        return launch_dependent(k, grid, 32 * TY, 0, s, (const S*)fA, (S*)fB, (CuT<S>*)cu, cls, g, P, shift,
                                lid ? (int)grid.y - 1 : 0);
    }
    // Tile height and resident blocks, GB300, us per step (4 x 2: TY = 4 at 2
    // blocks per SM, and so on):
    //   FP64 (bound by the FP64 unit, so by the busiest SM): short tiles while
    //     they spread over more SMs: 200^2 35.2 (4 x 2), 42.0 (8 x 2); 160^2 20.7,
    //     19.8; 240x280 43.6, 42.5; from about 4 short tiles per SM on, the smaller
    //     frame: 400x300 73.0, 72.0; 512^2 141, 121; 1000^2 506, 454.
    //   FP32 and 16-bit storage: TY = 8; a third block per SM (80 registers)
    //     pays once the grid exceeds 4 tiles per SM: FP32 240x280 5.8 (8 x 2),
    //     7.4 (8 x 3); 512x256 9.7, 10.2; 512x512 16.2, 14.0; 1024x1024 69.5, 64.8.
    static cudaError_t tile(const void* fA, void* fB, void* cu, const uint8_t* cls, const Geo& g,
                            const Prm<double>& Pd, cudaStream_t s)
    {
        const long long few = 4LL * sm_count(), strips = (g.nx + 31) / 32;
        if constexpr (std::is_same<R, double>::value) {
            if (strips * ((g.ny + 3) / 4) <= few) return launch_tile<4, 2>(fA, fB, cu, cls, g, Pd, s);
            return launch_tile<8, 2>(fA, fB, cu, cls, g, Pd, s);
        } else {
            if (strips * ((g.ny + 7) / 8) <= few) return launch_tile<8, 2>(fA, fB, cu, cls, g, Pd, s);
            return launch_tile<8, 3>(fA, fB, cu, cls, g, Pd, s);
        }
    }
    // One launch per step by tiles up to these sizes; beyond them the marching
    // kernel's loads one row ahead cover more of the memory latency (FP32, 16-bit)
    // or its halo is the smaller one (FP64).  GB300, us per step, k_step_tile
    // against k_step_march, uniform and general update: FP64 1000^2 454, 473 and
    // 574, 618; 1400^2 853, 847 and 1081, 1110; 1600^2 1095, 1043 and 1385, 1369.
    // FP32 500^2 14.0, 15.9 and 15.9, 16.5; 600^2 20.9, 21.4 and 23.5, 21.5; 777^2
    // 40.1, 36.7 and 43.1, 36.7; 1180^2 81.6, 73.5 and 86.6, 75.1.  FP16 500^2 13.7,
    // 14.3 and 14.9, 15.9; 600^2 18.7, 17.0 and 20.2, 18.7; 860^2 40.2, 30.3 and 42.9,
    // 32.6.  MRT: FP64 1400^2 1247, 1281; 1600^2 1601, 1578; FP32 500^2 21.4, 25.3;
    // 600^2 31.7, 30.4; 16-bit storage, whose dense update leaves the marching kernel
    // no loads ahead, later: FP16 860^2 58.3, 57.5; 1300^2 123.8, 124.1; 1500^2 162,
    // 168; 1730^2 215, 208; BF16 1180^2 98, 99; 1500^2 154, 158; 1730^2 205, 196.
    // Batches (their members' nodes together; the persistent kernel against
    // k_batch_tile): FP64 1.9 million 1242, 862; FP32 0.98 83.6, 74.9; 1.43 95.4, 103;
    // FP16 0.72 68, 52; 1.43 76, 93.
    static bool use_tile(long long nodes, bool batch)
    {
        if (std::is_same<S, double>::value) return nodes <= (batch ? 3000000 : 2200000);
        if (std::is_same<S, float>::value) return nodes <= (batch ? 1200000 : 350000);
        if (batch) return nodes <= 750000;
        return nodes <= (kDenseMrt<S, MRT> ? 2200000 : 300000);
    }
    static cudaError_t init(void* fA, void* cu, const uint8_t* cls, const double* c1, const double* c2,
                            const double* ux, const double* uy, const double* p, const Geo& g,
                            const Prm<double>& Pd, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        dim3 grid((g.nx + 127) / 128, g.ny);
        k_init<S, R><<<grid, 128, 0, s>>>((S*)fA, (CuT<S>*)cu, cls, c1, c2, ux, uy, p, g, P, 0, 0, g.ny);
        return cudaGetLastError();
    }
    static cudaError_t read(const void* fA, const uint8_t* cls, double* out, uint32_t mask, const Geo& g,
                            const Prm<double>& Pd, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        constexpr int TY = 8;
        const int shift = tile_shift(g.edge[3] == EDGE_LID, g.ny, TY);
        dim3 grid((g.nx + 31) / 32, (g.ny + shift + TY - 1) / TY);
        k_read_fields<S, R, TY><<<grid, 32 * TY, 0, s>>>((const S*)fA, cls, out, mask, g, P, shift);
        return cudaGetLastError();
    }
    static cudaError_t mass(const void* fA, const uint8_t* cls, double* part, int nparts, double* out,
                            const Geo& g, cudaStream_t s)
    {
        k_mass_partials<S, R><<<nparts, 256, 0, s>>>((const S*)fA, cls, part, g);
        k_mass_final<<<1, 256, 0, s>>>(part, nparts, out);
        return cudaGetLastError();
    }
    static cudaError_t contact(const void* fA, const uint8_t* cls, int comp, double* wallc, double* colh,
                               double* out, int max_drops, int* count, const Geo& g, cudaStream_t s)
    {
        k_contact_columns<S><<<(g.nx + 127) / 128, 128, 0, s>>>((const S*)fA, cls, comp, wallc, colh, g);
        k_contact_scan<<<1, 32, 0, s>>>(wallc, colh, g.nx, out, max_drops, count);
        return cudaGetLastError();
    }
    static cudaError_t film(const void* fA, const uint8_t* cls, int x, int y_top, int comps, double* out,
                            const Geo& g, cudaStream_t s)
    {
        k_film<S><<<1, 32, 0, s>>>((const S*)fA, cls, x, y_top, comps, out, g);
        return cudaGetLastError();
    }
    // the two block shapes the batch tuner chooses between
    static constexpr int kMinB64 = std::is_same<R, float>::value ? 8 : 6;
    static cudaError_t batch_step(const void* descs, const void* tiles, const void* walls, void* ctr, int parity,
                                  int variant, int grid, cudaStream_t s)
    {
        const LatDesc<R>* d = (const LatDesc<R>*)descs;
        const TileItem* ti = (const TileItem*)tiles;
        const WallItem* wi = (const WallItem*)walls;
        BatchCounters* c = (BatchCounters*)ctr;
        if (variant == 2)
            return launch_dependent(&k_batch_tile<S, R, kMinBBatchTile, MRT>, dim3(grid), 32 * kBatchTY, 0, s, d, ti, parity);
        if (variant == 0)
            return launch_dependent(&k_batch_interior<S, R, 64, PREFETCH, kMinB64, MRT>, dim3(grid), 64, 0, s, d, ti, wi, c, parity);
        return launch_dependent(&k_batch_interior<S, R, 128, PREFETCH, MINB, MRT>, dim3(grid), 128, 0, s, d, ti, wi, c, parity);
    }
    static constexpr int kMinBBatchTile = std::is_same<R, double>::value ? 2 : 3;
    static int batch_blocks_per_sm(int variant)
    {
        int n = 0;
        if (variant == 0)
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_interior<S, R, 64, PREFETCH, kMinB64, MRT>, 64, 0);
        else
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_interior<S, R, 128, PREFETCH, MINB, MRT>, 128, 0);
        return n;
    }
    static void fill_desc(void* dst, const void* buf0, const void* buf1, void* cu, const uint8_t* cls, const Geo& g,
                          const Prm<double>& P, int rows)
    {
        LatDesc<R>* d = (LatDesc<R>*)dst;
        d->buf[0] = buf0;
        d->buf[1] = buf1;
        d->cu = cu;
        d->cls = cls;
        d->g = g;
        d->P = cast_prm<R>(P);
        d->rows = rows;
    }
    static cudaError_t init_rows(void* fA, void* cu, const uint8_t* cls, const double* c1, const double* c2,
                                 const double* ux, const double* uy, const double* p, const Geo& g,
                                 const Prm<double>& Pd, int y0, int y1, int y_b, int rows, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        if (y1 <= y0) return cudaSuccess;
        dim3 grid((g.nx + 127) / 128, y1 - y0);
        k_init<S, R><<<grid, 128, 0, s>>>((S*)fA, (CuT<S>*)cu, cls, c1, c2, ux, uy, p, g, P, y0, y_b, rows);
        return cudaGetLastError();
    }
    static cudaError_t csum_ip(const void* f, void* cpl, const uint8_t* cls, const Geo& g, int odd, cudaStream_t s)
    {
        dim3 grid((g.pitch + 127) / 128, g.ny);
        if (odd) k_csum<S, R, true><<<grid, 128, 0, s>>>((const S*)f, (R*)cpl, cls, g);
        else k_csum<S, R, false><<<grid, 128, 0, s>>>((const S*)f, (R*)cpl, cls, g);
        return cudaGetLastError();
    }
    // resident blocks of the in-place interior kernel per step parity: its
    // FP32 form holds all 18 order-parameter populations at once; at 5 blocks
    // (96 registers) the odd (gathering) form spills a few words, and is still
    // faster than at 4 blocks (GB300, 2048^2: FP32 13.0 -> 14.1, FP16 13.6 ->
    // 15.1 G node updates/s with both parities at 5)
#ifndef TLB_IP_MINB_EVEN
#define TLB_IP_MINB_EVEN 5
#endif
#ifndef TLB_IP_MINB_ODD
#define TLB_IP_MINB_ODD 5
#endif
    // 16-bit storage with the whole next read set loaded one iteration ahead
    // (TLB_PIPE_IP16) runs at 4 blocks (GB300, 2048^2: 16.3 -> 17.2 G node
    // updates/s; at 5 blocks it spills and gains 1%)
#ifndef TLB_IP_MINB16
#define TLB_IP_MINB16 4
#endif
    static constexpr int kMinBIpEven =
        Store<S>::k16 && kPipeIp16 ? TLB_IP_MINB16 : (std::is_same<R, float>::value ? TLB_IP_MINB_EVEN : MINB);
    static constexpr int kMinBIpOdd =
        Store<S>::k16 && kPipeIp16 ? TLB_IP_MINB16 : (std::is_same<R, float>::value ? TLB_IP_MINB_ODD : MINB);
    template <bool UNI, bool ODD>
    static void launch_interior_ip(void* f, void* cu, const void* cpl, const uint8_t* cls, const Geo& g,
                                   const Prm<R>& P, cudaStream_t s)
    {
        constexpr int TX = BLOCK - 4;
        constexpr int kMinB = ODD ? kMinBIpOdd : kMinBIpEven;
        const int rows = rows_for(g, TX, ROWS, kMinB, std::is_same<R, double>::value, Store<S>::k16 ? 0 : 1);
        dim3 grid((g.nx + TX - 1) / TX, (g.ny + rows - 1) / rows);
        k_step_interior_ip<S, R, BLOCK, ROWS, PREFETCH, kMinB, MRT, UNI, ODD><<<grid, BLOCK, 0, s>>>(
            (S*)f, (CuT<S>*)cu, (const R*)cpl, cls, g, P, rows);
    }
    static cudaError_t interior_ip(void* f, void* cu, const void* cpl, const uint8_t* cls, const Geo& g,
                                   const Prm<double>& Pd, int odd, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        if (Pd.uni != 0.0) {
            if (odd) launch_interior_ip<true, true>(f, cu, cpl, cls, g, P, s);
            else launch_interior_ip<true, false>(f, cu, cpl, cls, g, P, s);
        } else {
            if (odd) launch_interior_ip<false, true>(f, cu, cpl, cls, g, P, s);
            else launch_interior_ip<false, false>(f, cu, cpl, cls, g, P, s);
        }
        return cudaGetLastError();
    }
    static cudaError_t wall_ip(void* f, void* cu, const void* cpl, const uint8_t* cls, const uint32_t* list,
                               int nlist, const Geo& g, const Prm<double>& Pd, int odd, int lid, cudaStream_t s)
    {
        const Prm<R> P = cast_prm<R>(Pd);
        if (nlist <= 0) return cudaSuccess;
        const int blocks = (nlist + 127) / 128;
        if (odd)
            k_step_wall_ip<S, R, MRT, true><<<blocks, 128, 0, s>>>((S*)f, (CuT<S>*)cu, (const R*)cpl, cls, list, nlist,
                                                                  g, P, lid);
        else
            k_step_wall_ip<S, R, MRT, false><<<blocks, 128, 0, s>>>((S*)f, (CuT<S>*)cu, (const R*)cpl, cls, list,
                                                                   nlist, g, P, lid);
        return cudaGetLastError();
    }
    static cudaError_t swap_ip(void* f, const uint8_t* cls, const Geo& g, cudaStream_t s)
    {
        dim3 grid((g.nx + 127) / 128, g.ny);
        k_swap<S><<<grid, 128, 0, s>>>((S*)f, cls, g);
        return cudaGetLastError();
    }
    static const Ops& table()
    {
        static const Ops t{sizeof(S), Store<S>::kPlanes, sizeof(CuT<S>), &march, &tile, &use_tile, &init, &read, &contact, &film, &batch_step,
                          &batch_blocks_per_sm, sizeof(LatDesc<R>), &fill_desc, &mass, &init_rows, sizeof(R),
                          &csum_ip, &interior_ip, &wall_ip, &swap_ip};
        return t;
    }
};

}  // namespace tlb
