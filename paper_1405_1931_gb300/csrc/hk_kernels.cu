// hk_kernels.cu -- the labelling passes.
//
//   K0 occupancy      stream phi once (coalesced row loads) and write the
//                     occupancy mask phi > 0, one 32-bit word per tile row.
//   K1 tile_label     label each tile from its mask words (Sec. 2's rules
//                     become union-find over x-runs), register boundary
//                     pieces, and write one code per run, the face summaries
//                     and the per-row count of interior cluster roots.
//   K2 face_merge     join boundary pieces across tile faces and periodic
//                     edges: the intra-GPU counterpart of Sec. 3's halo
//                     equivalences, resolved directly on a global union-find
//                     instead of being gathered to a root process.
//   K3 piece_finalize compress the union-find, add piece sizes into cluster
//                     roots and count cluster roots per row segment.
//   S1-S2 scan        exclusive prefix of the root counts: the compactified
//                     cluster numbering 1..n of Sec. 2 in row-major order.
//   K4 flatten        persistent: decode the run codes, write the labels, the
//                     sizes in label order and the histogram.
#include <cstring>
#include <mutex>
#include <type_traits>

#include "hk_device.cuh"
#include "hk_launch.h"

namespace hk {

// A site near a membrane (Sec. 6, step 2) votes with the sign of its index value: bit q
// when it is negative, bit 16 + q when positive (not for 0, NaN and the far sites).
__device__ __forceinline__ uint32_t near_bits(float v, int q) {
    return (v >= -0.5f && v < 0.0f ? 1u << q : 0u) | (v > 0.0f ? 0x10000u << q : 0u);
}

// --------------------------------------------------------------------------------------
// K0: occupancy.  One warp per tile streams phi row by row (one coalesced 128-byte
// load per row, 16 rows in flight per warp) and keeps phi > 0 (Sec. 2) as one
// 32-bit word per tile row, written tile-major.  Sites outside the lattice count
// as medium.
// --------------------------------------------------------------------------------------
template <int TY, int TZ, int NL>
__global__ void __launch_bounds__(256, 4) k_occupancy(const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    constexpr int R = SH::R, U = 16;
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (blockIdx.x == 0 && threadIdx.x == 0) *W.novf = 0;   // the tile pass appends after this pass
    if (t >= ntiles) return;
    const LatDev &L = B.lat[(NL == 1) ? 0 : find_lattice(B.lat, B.n, t)];
    const TileGeo g = tile_geo<TY, TZ>(L, t);
    const int64_t sxy = (int64_t)L.nx * L.ny;
    const float *base = L.phi + (int64_t)g.z0 * sxy + (int64_t)g.y0 * L.nx + g.x0 + lane;
    const bool xin = lane <= g.lastX;
    uint32_t *out = W.mask + t * R;
    // Whole 128-byte rows at 16-byte aligned addresses: lane l loads 4 sites (x = 4 (l % 8)
    // .. + 3) of row l / 8 of each group of 4 rows, and the 8 lanes of a row OR their
    // nibbles into the row's word.
    const bool vec = g.lastX == TX - 1 && (L.nx & 3) == 0 && (reinterpret_cast<uintptr_t>(L.phi) & 15) == 0;
    const int x4 = (lane & 7) * 4;
    const float *base4 = L.phi + (int64_t)g.z0 * sxy + (int64_t)g.y0 * L.nx + g.x0 + x4;
    uint32_t any_near = 0;
    for (int r0 = 0; r0 < R; r0 += 32) {        // lane j keeps the words of row r0 + j
        uint32_t mine = 0, neg = 0, pos = 0;
        if (vec) {
            float4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int rr = r0 + 4 * q + (lane >> 3), ly = rr % TY, lz = rr / TY;
                v[q] = (ly <= g.lastY && lz <= g.lastZ)
                           ? __ldcs(reinterpret_cast<const float4 *>(base4 + (int64_t)lz * sxy + (int64_t)ly * L.nx))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                uint32_t w = ((uint32_t)occupied(v[q].x, L.occ_mode) | ((uint32_t)occupied(v[q].y, L.occ_mode) << 1) |
                              ((uint32_t)occupied(v[q].z, L.occ_mode) << 2) | ((uint32_t)occupied(v[q].w, L.occ_mode) << 3))
                             << x4;
                w |= __shfl_xor_sync(0xffffffffu, w, 1);
                w |= __shfl_xor_sync(0xffffffffu, w, 2);
                w |= __shfl_xor_sync(0xffffffffu, w, 4);
                const uint32_t wq = __shfl_sync(0xffffffffu, w, (lane & 3) * 8);   // row r0 + 4 q + (lane & 3)
                if ((lane >> 2) == q) mine = wq;
                if (W.neg) {                           // uniform: signs of the near sites
                    uint32_t n = (near_bits(v[q].x, 0) | near_bits(v[q].y, 1) | near_bits(v[q].z, 2) | near_bits(v[q].w, 3));
                    uint32_t ps = (n >> 16) << x4;
                    n = (n & 0xffffu) << x4;
#pragma unroll
                    for (int d = 1; d < 8; d <<= 1) {
                        n |= __shfl_xor_sync(0xffffffffu, n, d);
                        ps |= __shfl_xor_sync(0xffffffffu, ps, d);
                    }
                    const uint32_t nq = __shfl_sync(0xffffffffu, n, (lane & 3) * 8);
                    const uint32_t pq = __shfl_sync(0xffffffffu, ps, (lane & 3) * 8);
                    if ((lane >> 2) == q) { neg = nq; pos = pq; }
                }
            }
        } else {
#pragma unroll
            for (int u0 = 0; u0 < 32; u0 += U) {
                float v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int rr = r0 + u0 + u, ly = rr % TY, lz = rr / TY;
                    v[u] = (xin && ly <= g.lastY && lz <= g.lastZ)
                               ? __ldcs(base + (int64_t)lz * sxy + (int64_t)ly * L.nx) : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t w = __ballot_sync(0xffffffffu, occupied(v[u], L.occ_mode));
                    if (lane == u0 + u) mine = w;
                    if (W.neg) {
                        const uint32_t n = near_bits(v[u], 0);
                        const uint32_t wn = __ballot_sync(0xffffffffu, n & 1u), wp = __ballot_sync(0xffffffffu, n >> 16);
                        if (lane == u0 + u) { neg = wn; pos = wp; }
                    }
                }
            }
        }
        out[r0 + lane] = mine;
        if (W.neg) {
            W.neg[t * R + r0 + lane] = neg;
            W.pos[t * R + r0 + lane] = pos;
            any_near |= neg | pos;
        }
        // first and last column of the tile, one bit per row (faces along x)
        const uint32_t c0 = __ballot_sync(0xffffffffu, mine & 1u);
        const uint32_t cl = __ballot_sync(0xffffffffu, (mine >> g.lastX) & 1u);
        if (lane == 0) {
            W.xcol[(t * 2) * (R / 32) + (r0 >> 5)] = c0;
            W.xcol[(t * 2 + 1) * (R / 32) + (r0 >> 5)] = cl;
        }
    }
    if (W.neg) {
        any_near = __reduce_or_sync(0xffffffffu, any_near);
        if (lane == 0) W.near_tile[t] = any_near != 0u;
    }
}

// K0 with TMA (every lattice of the launch with 16-byte aligned rows): persistent, a
// ring of two tile buffers per CTA filled by cp.async.bulk.tensor loads completed on
// mbarriers; while one tile is converted the next is in flight.
template <int TY, int TZ>
struct OccSmem {
    using SH = TileShape<TY, TZ>;
    alignas(128) float buf[2][SH::SITES];
    uint64_t bar[2];
};

// INDEX: also the signs of the near sites (its own instance: three votes a row, and a
// batch of plain fields took 381 against 333 us with the choice made at run time).
template <int TY, int TZ, int NL, bool INDEX>
__global__ void __launch_bounds__(256) k_occupancy_tma(const __grid_constant__ TmapBatch<NL> TB,
                                                       const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    constexpr int R = SH::R;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    OccSmem<TY, TZ> &S = *reinterpret_cast<OccSmem<TY, TZ> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (blockIdx.x == 0 && tid == 0) *W.novf = 0;           // the tile pass appends after this pass
    if (tid == 0) {
        mbar_init(&S.bar[0], 1);
        mbar_init(&S.bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    auto issue = [&](int64_t t, int s) {
        const int lat = (NL == 1) ? 0 : find_lattice(B.lat, B.n, t);
        const TileGeo g = tile_geo<TY, TZ>(B.lat[lat], t);
        fence_proxy_async();
        mbar_arrive_expect_tx(&S.bar[s], SH::SITES * 4);
        tma_load_3d(S.buf[s], &TB.tm[lat].phi, &S.bar[s], g.x0, g.y0, g.z0);
    };
    const int64_t t0 = blockIdx.x, step = gridDim.x;
    if (tid == 0) {
        if (t0 < ntiles) issue(t0, 0);
        if (t0 + step < ntiles) issue(t0 + step, 1);
    }
    int k = 0;
    for (int64_t t = t0; t < ntiles; t += step, ++k) {
        const int s = k & 1;
        // the decision to give up is the CTA's, so that every thread leaves together
        if (__syncthreads_or(!mbar_wait_bounded(&S.bar[s], (uint32_t)((k >> 1) & 1)))) {
            if (tid == 0) atomicOr(W.status, STATUS_TMA_TIMEOUT);
            // a second bounded wait for the copies still in flight into this CTA's
            // buffers (this tile's and the next one's) before its shared memory goes
            mbar_wait_bounded(&S.bar[s], (uint32_t)((k >> 1) & 1));
            if (t + step < ntiles) mbar_wait_bounded(&S.bar[s ^ 1], (uint32_t)(((k + 1) >> 1) & 1));
            return;
        }
        const LatDev &L = B.lat[(NL == 1) ? 0 : find_lattice(B.lat, B.n, t)];
        const int lastX = tile_geo<TY, TZ>(L, t).lastX;
        // warp w converts rows [32 w', 32 w' + 32) in turns; lane j keeps row 32 w' + j
        [[maybe_unused]] uint32_t any_near = 0;
        for (int r0 = wid * 32; r0 < R; r0 += 32 * (256 / 32)) {
            uint32_t mine = 0;
            if constexpr (INDEX) {
                uint32_t neg = 0, pos = 0;
#pragma unroll 8
                for (int j = 0; j < 32; ++j) {
                    const float v = S.buf[s][(r0 + j) * 32 + lane];
                    const uint32_t w = __ballot_sync(0xffffffffu, occupied(v, 1));
                    const uint32_t wn = __ballot_sync(0xffffffffu, v < 0.0f), wp = __ballot_sync(0xffffffffu, v > 0.0f);
                    if (lane == j) {
                        mine = w;
                        neg = wn;
                        pos = wp;
                    }
                }
                neg &= ~mine;                          // near and negative; a positive site is never far
                W.neg[t * R + r0 + lane] = neg;
                W.pos[t * R + r0 + lane] = pos;
                any_near |= neg | pos;
            } else {
#pragma unroll 8
                for (int j = 0; j < 32; ++j) {
                    const uint32_t w = __ballot_sync(0xffffffffu, occupied(S.buf[s][(r0 + j) * 32 + lane], L.occ_mode));
                    if (lane == j) mine = w;
                }
            }
            W.mask[t * R + r0 + lane] = mine;
            const uint32_t c0 = __ballot_sync(0xffffffffu, mine & 1u);
            const uint32_t cl = __ballot_sync(0xffffffffu, (mine >> lastX) & 1u);
            if (lane == 0) {
                W.xcol[(t * 2) * (R / 32) + (r0 >> 5)] = c0;
                W.xcol[(t * 2 + 1) * (R / 32) + (r0 >> 5)] = cl;
            }
        }
        // every warp is done with buffer s
        if constexpr (INDEX) {
            const bool near_tile = __syncthreads_or(any_near != 0u);
            if (tid == 0) W.near_tile[t] = near_tile;
        } else {
            __syncthreads();
        }
        if (tid == 0 && t + 2 * step < ntiles) issue(t + 2 * step, s);
    }
}

// --------------------------------------------------------------------------------------
// K1: tile labelling from the occupancy words (one tile per CTA)
//
// Bound by instruction issue (90 % of its rate at 512^3): 2 warp instructions a site at p_c.  With
// most pairs linked or left out instead of united, and with boundary pieces listed by the
// run that first touches a face instead of in passes over all runs: 1.82 against 2.38 ms
// at 1024^3, p_c, 0.79 against 1.06 ms on blocks of 16^3, 0.125 against 0.148 ms on a
// 512^3 bijel.
// --------------------------------------------------------------------------------------
template <int TY, int TZ, int CAP, int BL, bool INDEX>
struct LabelSmem {
    using SH = TileShape<TY, TZ>;
    uint32_t m[SH::R];                     // occupancy word of each row
    uint16_t rbase[SH::R];                 // first run id of each row
    int par[CAP];                          // union-find over run ids; after compression: the root
    alignas(16) int aux[CAP];              // union pair lists; then per root: size + AUX_FACE *
                                           // (runs touching a face); then -1 - k for boundary root k
    uint16_t desc[CAP];                    // per run: DESC_TOUCH | (tile row << 5) | first x
    uint16_t blist[BL];                    // run id of each boundary root, by its number
    uint32_t nylo[TZ], nyhi[TZ];           // neighbour rows across the y faces, per plane
    uint32_t nzlo[TY], nzhi[TY];           // neighbour rows across the z faces, per row
    uint32_t nxlo[SH::R / 32], nxhi[SH::R / 32];   // neighbour columns across the x faces
    uint32_t xo0[SH::R / 32], xol[SH::R / 32];     // this tile's first and last column
    static_assert(TZ <= 16 && TY <= 32 && SH::R / 32 <= 16 && SH::NT >= 64, "face loads use threads 0..63");
    static_assert(SH::R <= 256 && CAP <= 4096, "desc holds an 8-bit row and run ids fit in 16 bits");
    static constexpr int RPW = INDEX ? 4 : 1;   // rows a word of rowcnt: a byte each (at most 16), or a word
    uint32_t rowcnt[SH::R / RPW];          // roots, then interior roots of each row
    int nbnd;                              // boundary roots of the tile
    int nroot;                             // roots (index fields)
    int warp_tmp[32];
    uint32_t neg[INDEX ? SH::R : 1], pos[INDEX ? SH::R : 1];   // signs of the near sites of each row
    int votes[INDEX ? CAP : 1];            // per root: the votes of its piece's sites
};

constexpr int AUX_FACE = 1 << 14;   // > any piece size (a tile has at most 8192 sites)
constexpr int DESC_TOUCH = 1 << 13;  // desc flag: the run has a site connected across a tile face

// Resident CTAs per SM of the fast tile pass (its shared memory and 32 registers a
// thread allow 2048 threads) and of the pass over the tiles it hands on.
// Index fields whose votes are wanted hold fewer runs a row (membranes and bulk fluid), for
// room for their votes: 4 on average.
template <int TY, int TZ, bool FAST, bool INDEX = false>
struct LabelCfg {
    static constexpr int CAP = !FAST ? TileShape<TY, TZ>::MAXRUNS
                             : INDEX ? 4 * TileShape<TY, TZ>::R : TileShape<TY, TZ>::MR_FAST;
    // boundary pieces the fast pass lists (more go to the second pass, which has room for all)
    static constexpr int BL = FAST && TileShape<TY, TZ>::MAX_BOUNDARY > 512 ? 512 : TileShape<TY, TZ>::MAX_BOUNDARY;
    // resident threads of an SM; index fields wait more than they issue (729 capsules at
    // 1024^3: 1.34 ms at 1280, 1.19 at 1536, 1.11 at 1792 and 2048)
    static constexpr int THREADS = !FAST ? 1280 : INDEX ? 1792 : 2048;
    static constexpr int BLOCKS = THREADS / (TY * TZ) < 32 ? THREADS / (TY * TZ) : 32;
};

// FAST: tiles t = blockIdx.x, blockIdx.x + gridDim.x, ... below ntiles; a tile with
// more than MR_FAST runs or union pairs of one kind is appended to W.ovf instead.
// !FAST: the tiles listed in W.ovf, with room for every tile.
// INDEX: an index field whose clusters' votes are wanted (Sec. 6, step 5; one lattice).
template <int TY, int TZ, int NL, bool FAST, bool INDEX>
__global__ void __launch_bounds__(TY * TZ, (LabelCfg<TY, TZ, FAST, INDEX>::BLOCKS))
k_tile_label(const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    constexpr int R = SH::R, NT = SH::NT, MR = SH::MAXRUNS, CAP = LabelCfg<TY, TZ, FAST, INDEX>::CAP;
    constexpr int BL = LabelCfg<TY, TZ, FAST, INDEX>::BL;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    LabelSmem<TY, TZ, CAP, BL, INDEX> &S = *reinterpret_cast<LabelSmem<TY, TZ, CAP, BL, INDEX> *>(smem_raw);
    const int tid = threadIdx.x;
    const int64_t nwork = FAST ? ntiles : (int64_t)*reinterpret_cast<volatile int32_t *>(W.novf);

    for (int64_t it = blockIdx.x; it < nwork; it += gridDim.x) {
        const int64_t t = FAST ? it : (int64_t)W.ovf[it];
        const int lat = (NL == 1) ? 0 : find_lattice(B.lat, B.n, t);
        const LatDev &L = B.lat[lat];
        const TileGeo g = tile_geo<TY, TZ>(L, t);

        const int r = tid, ly = r % TY, lz = r / TY;
        const uint32_t m = W.mask[t * R + r];
        S.m[r] = m;
        bool near_here = false;                   // CTA-uniform: the tile or one across a face has near sites
        if (INDEX) {
            const int64_t plane = (int64_t)L.nbx * L.nby;
            const int64_t nb[7] = {t, g.bx > 0 ? t - 1 : t + (L.nbx - 1), g.bx < L.nbx - 1 ? t + 1 : t - (L.nbx - 1),
                                   g.by > 0 ? t - L.nbx : t + (int64_t)(L.nby - 1) * L.nbx,
                                   g.by < L.nby - 1 ? t + L.nbx : t - (int64_t)(L.nby - 1) * L.nbx,
                                   g.bz > 0 ? t - plane : t + (int64_t)(L.nbz - 1) * plane,
                                   g.bz < L.nbz - 1 ? t + plane : t - (int64_t)(L.nbz - 1) * plane};
            uint32_t any = 0;
#pragma unroll
            for (int k = 0; k < 7; ++k) any |= W.near_tile[nb[k]];
            near_here = any != 0u;
            if (near_here) {
                S.neg[r] = W.neg[t * R + r];
                S.pos[r] = W.pos[t * R + r];
            }
        }
        const uint32_t rs = run_starts(m);
        {
            const uint32_t c0 = __ballot_sync(0xffffffffu, m & 1u);
            const uint32_t cl = __ballot_sync(0xffffffffu, (m >> g.lastX) & 1u);
            if ((tid & 31) == 0) {
                S.xo0[tid >> 5] = c0;
                S.xol[tid >> 5] = cl;
            }
        }

        // Occupancy across the six faces, from the neighbour tiles' masks (the
        // occupancy pass has written all of them).  A face site is connected when
        // it and its neighbour across the face are both occupied; only pieces with a
        // connected site take part in the merge between tiles.
        {
            const int64_t plane = (int64_t)L.nbx * L.nby;
            const int lastY_lo = g.by > 0 ? TY - 1 : L.ny - 1 - (L.nby - 1) * TY;   // neighbour's last row
            const int lastZ_lo = g.bz > 0 ? TZ - 1 : L.nz - 1 - (L.nbz - 1) * TZ;
            constexpr int RW = R / 32;
            if (tid < TZ) {
                const int64_t tylo = g.by > 0 ? t - L.nbx : t + (int64_t)(L.nby - 1) * L.nbx;
                const int64_t tyhi = g.by < L.nby - 1 ? t + L.nbx : t - (int64_t)(L.nby - 1) * L.nbx;
                S.nylo[tid] = g.extYlo ? W.mask[tylo * R + tid * TY + lastY_lo] : 0u;
                S.nyhi[tid] = g.extYhi ? W.mask[tyhi * R + tid * TY] : 0u;
            } else if (tid >= 16 && tid < 16 + TY) {     // TZ <= 16, TY <= 32, R/32 <= 8, NT >= 64
                const int q = tid - 16;
                const int64_t tzlo = g.bz > 0 ? t - plane : t + (int64_t)(L.nbz - 1) * plane;
                const int64_t tzhi = g.bz < L.nbz - 1 ? t + plane : t - (int64_t)(L.nbz - 1) * plane;
                S.nzlo[q] = g.extZlo ? W.mask[tzlo * R + lastZ_lo * TY + q] : 0u;
                S.nzhi[q] = g.extZhi ? W.mask[tzhi * R + q] : 0u;
            } else if (tid >= 48 && tid < 48 + RW) {
                const int q = tid - 48;
                const int64_t txlo = g.bx > 0 ? t - 1 : t + (L.nbx - 1);
                const int64_t txhi = g.bx < L.nbx - 1 ? t + 1 : t - (L.nbx - 1);
                S.nxlo[q] = g.extXlo ? W.xcol[(txlo * 2 + 1) * RW + q] : 0u;   // its last column
                S.nxhi[q] = g.extXhi ? W.xcol[(txhi * 2) * RW + q] : 0u;       // its first column
            }
        }

        // a2: run ids (row-major), union lists, unions
        int total;
        const int rb = block_exscan<NT>(__popc(rs), S.warp_tmp, total);   // ends with a barrier
        if (FAST && total > CAP) {               // block-uniform; nothing read from S after the scan
            if (tid == 0) W.ovf[atomicAdd(W.novf, 1)] = (int32_t)t;
            continue;
        }
        S.rbase[r] = (uint16_t)rb;
        // Each run's own union-find node and its descriptor: position and whether one of
        // its sites is connected across a tile face with a neighbour tile (the site and
        // its neighbour there both occupied).
        if (m) {
            uint32_t conn = 0;
            if (ly == 0) conn |= S.nylo[lz];
            if (ly == g.lastY) conn |= S.nyhi[lz];
            if (lz == 0) conn |= S.nzlo[ly];
            if (lz == g.lastZ) conn |= S.nzhi[ly];
            if ((S.nxlo[r >> 5] >> (r & 31)) & 1u) conn |= 1u;
            if ((S.nxhi[r >> 5] >> (r & 31)) & 1u) conn |= 1u << g.lastX;
            conn &= m;
            // the run starts whose run holds a connected site, for the whole row at once
            const uint32_t touched = fill_down(m, conn) & rs;
            int id = rb;
            for (uint32_t w = rs; w;) {
                const uint32_t low = w & (0u - w);
                w ^= low;
                S.par[id] = id;
                S.desc[id] = (uint16_t)(((touched & low) ? DESC_TOUCH : 0) | (r << 5) | top_bit(low));
                ++id;
            }
        }
        const int ucap = (W.local_cap > 0 && W.local_cap < total) ? W.local_cap : total;   // union retry bound

        // y- and z-neighbours: one union per overlapping run pair of rows (y-1, y) and
        // (z-1, z), that is per segment of their common sites.  Two kinds of pairs need
        // none.  A run's first pair -- with row y - 1, or with row z - 1 if it meets no run
        // of row y - 1 -- is written straight into its own node (link): a smaller id, and
        // the node has no other writer yet, so no find and no atomic.  And a z pair is left
        // out where it starts at a site x with (x, y-1, z) and (x, y-1, z-1) occupied too:
        // the two runs are joined through those, by their own y pairs and the z pair of row
        // y - 1 (or what that one is joined through, down to the tile's first row).
        // At p_c 0.2 unions a run are left of 0.8, in smooth fields hardly any.
        // Both lists of the others come from one scan of packed counts (each total is at
        // most 16 * R < 2^16) and normally share one pass of unions, the z pairs listed
        // first (measured faster than y first).
        const uint32_t my = ly > 0 ? S.m[r - 1] : 0u, mz = lz > 0 ? S.m[r - TY] : 0u;
        const uint32_t oy = m & my, oz = m & mz, uy = fill_up(m, oy);
        uint32_t osy = run_starts(oy), osz = run_starts(oz);
        uint32_t link = osy & ~(uy << 1);                      // first y pair of each run
        osy ^= link;
        {
            const uint32_t zlink = osz & ~(fill_up(m, oz) << 1) & ~(uy | fill_down(m, oy));
            link |= zlink;
            osz &= ~zlink;
            if (ly > 0 && lz > 0) osz &= ~(my & S.m[r - TY - 1]);
        }
        int tot_packed;
        const int packed = block_exscan<NT>(__popc(osy) | (__popc(osz) << 16), S.warp_tmp, tot_packed);
        const int ny_tot = tot_packed & 0xffff, nz_tot = tot_packed >> 16;
        if (FAST && (ny_tot > CAP || nz_tot > CAP)) {   // block-uniform, as above
            if (tid == 0) W.ovf[atomicAdd(W.novf, 1)] = (int32_t)t;
            continue;
        }
        // run ids at a site of rows r (rb), r - 1 (rby) and r - TY (rbz): the run starts up to it
        const uint32_t rsy = run_starts(my), rsz = run_starts(mz);
        const int rby = ly > 0 ? S.rbase[r - 1] : 0, rbz = lz > 0 ? S.rbase[r - TY] : 0;
        while (link) {
            const uint32_t low = link & (0u - link), le = low | (low - 1u);
            link ^= low;
            const bool y = (my & low) != 0u;                   // a z link's run meets no run of row y - 1
            S.par[rb + __popc(rs & le) - 1] = (y ? rby : rbz) + __popc((y ? rsy : rsz) & le) - 1;
        }
        auto write_pairs = [&](uint32_t os, uint32_t rsq, int rbq, int j) {
            while (os) {
                const uint32_t low = os & (0u - os), le = low | (low - 1u);
                os ^= low;
                S.aux[j++] = ((rb + __popc(rs & le) - 1) << 16) | (rbq + __popc(rsq & le) - 1);
            }
        };
        auto union_pairs = [&](int n) {
            for (int i = tid; i < n; i += NT) {
                const uint32_t p = (uint32_t)S.aux[i];
                s_union(S.par, (int)(p >> 16), (int)(p & 0xffffu), ucap, W.status);
            }
        };
        if (ny_tot + nz_tot <= CAP) {           // block-uniform
            write_pairs(osz, rsz, rbz, packed >> 16);
            write_pairs(osy, rsy, rby, nz_tot + (packed & 0xffff));
            __syncthreads();
            union_pairs(ny_tot + nz_tot);
            __syncthreads();
        } else {
            write_pairs(osy, rsy, rby, packed & 0xffff);
            __syncthreads();
            union_pairs(ny_tot);
            __syncthreads();
            write_pairs(osz, rsz, rbz, packed >> 16);
            __syncthreads();
            union_pairs(nz_tot);
            __syncthreads();
        }

        // periodic edges inside the tile (an axis that fits in one tile).  A find from the far
        // row climbs the links of the rows between, so along y and z the pairs of a row are
        // shared out by nibbles (stripes of one site at 512 x 16 x 512: 43 us, 68 with one thread a
        // row).
        if (g.wrapX || g.wrapY || g.wrapZ) {
            const int nw_y = g.wrapY && g.lastY > 0 ? TZ : 0, nw = nw_y + (g.wrapZ && g.lastZ > 0 ? TY : 0);
#pragma unroll 1
            for (int k = tid; k < 8 * nw; k += NT) {
                const int j = k >> 3, a = j < nw_y ? j * TY : j - nw_y, b = a + (j < nw_y ? g.lastY : g.lastZ * TY);
                const uint32_t ma = S.m[a], mb = S.m[b];
                join_rows(S.par, ma, S.rbase[a], mb, S.rbase[b], 0xfu << (4 * (k & 7)), ucap, W.status);
            }
            if (m) {
                if (g.wrapX && g.lastX > 0 && (m & 1u) && ((m >> g.lastX) & 1u))
                    s_union(S.par, rb, run_of(rb, rs, g.lastX), ucap, W.status);
            }
            __syncthreads();
        }

        // Sizes accumulate in aux, which held the pair lists until the unions above.
        constexpr int RPW = LabelSmem<TY, TZ, CAP, BL, INDEX>::RPW;
        if (tid < R / RPW) S.rowcnt[tid] = 0u;
        if (tid == 0) S.nbnd = S.nroot = 0;
        for (int i = 4 * tid; i < total; i += 4 * NT)
            *reinterpret_cast<int4 *>(&S.aux[i]) = make_int4(0, 0, 0, 0);
        if (INDEX)
            for (int i = tid; i < total; i += NT) S.votes[i] = 0;
        __syncthreads();

        // Compression and piece sizes, one run id per thread: par[i] = root (the piece's
        // first run), and the run's length -- plus AUX_FACE if it touches a face -- is
        // added to its root.  The finds are read-only, so storing final roots while
        // others still search is safe.  A piece is a boundary piece iff its sum reaches
        // AUX_FACE (sizes stay below it): the run that brings its root there lists it and
        // gives the piece its number (in any order: a number only names the piece).  The
        // roots of each row are counted, a word a row: with four rows a word, a byte each, a warp
        // of single sites meets in one word (1.90 against 1.83 ms at 1024^3, p_c, 68 against 45
        // us on a 16 x 1024 x 1024 checkerboard; index fields have few roots).
        for (int i = tid; i < total; i += NT) {
            int root = S.par[i];
            while (true) {                       // two levels a step
                const int up = S.par[root];
                root = S.par[up];
                if (root == up) break;
            }
            S.par[i] = root;
            const int d = S.desc[i], row = (d >> 5) & 0xff;
            const int len = run_len(S.m[row], d & 31);
            const int face = (d & DESC_TOUCH) ? AUX_FACE : 0;
            if (atomicAdd(&S.aux[root], len + face) + (AUX_FACE - face) < AUX_FACE) {
                const int k = atomicAdd(&S.nbnd, 1);
                if (k < BL) S.blist[k] = (uint16_t)root;
            }
            if (root == i) {
                atomicAdd(&S.rowcnt[row / RPW], 1u << (8 * (row % RPW)));
                if (INDEX) atomicAdd(&S.nroot, 1);
            }
        }
        __syncthreads();

        // Votes (Sec. 6, step 5): every face-neighbour pair of a cluster site and a near site
        // adds the near site's sign to the cluster.  Per row, the signs of the six neighbours
        // of its sites are words like its own (a row of the tile, of the tile across a face
        // or across a periodic edge, or its own word moved by one along x), so a run's votes
        // are counts of bits; rows away from every membrane have none.
        if (INDEX && near_here && m) {
            const int64_t plane = (int64_t)L.nbx * L.nby;
            auto row_of = [&](const uint32_t *sw, const uint32_t *gw, int axis, bool hi) -> uint32_t {
                const int c = axis == 1 ? ly : lz, last = axis == 1 ? g.lastY : g.lastZ, step = axis == 1 ? 1 : TY;
                if (hi ? c < last : c > 0) return sw[hi ? r + step : r - step];
                const bool ext = axis == 1 ? (hi ? g.extYhi : g.extYlo) : (hi ? g.extZhi : g.extZlo);
                if (!ext) return (axis == 1 ? g.wrapY : g.wrapZ) ? sw[hi ? r - c * step : r + last * step] : 0u;
                const int b = axis == 1 ? g.by : g.bz, nb = axis == 1 ? L.nby : L.nbz, len = axis == 1 ? L.ny : L.nz;
                const int span = axis == 1 ? TY : TZ;
                const int nb_tile = hi ? (b < nb - 1 ? b + 1 : 0) : (b > 0 ? b - 1 : nb - 1);
                const int nc = hi ? 0 : min(span, len - nb_tile * span) - 1;
                return gw[(t + (nb_tile - b) * (axis == 1 ? (int64_t)L.nbx : plane)) * R + r + (nc - c) * step];
            };
            auto along_x = [&](const uint32_t *sw, const uint32_t *gw, bool hi) -> uint32_t {
                const uint32_t w = sw[r];
                uint32_t edge = 0;                             // the neighbour of the tile's first / last column
                if (hi) {
                    if (g.extXhi) edge = gw[(g.bx < L.nbx - 1 ? t + 1 : t - (L.nbx - 1)) * R + r] & 1u;
                    else if (g.wrapX) edge = w & 1u;
                    return (w >> 1) | (edge << g.lastX);
                }
                if (g.extXlo) edge = gw[(g.bx > 0 ? t - 1 : t + (L.nbx - 1)) * R + r] >> (g.bx > 0 ? TX - 1 : (L.nx - 1) % TX);
                else if (g.wrapX) edge = w >> g.lastX;
                return (w << 1) | (edge & 1u);
            };
            uint32_t nw[6], pw[6], any = 0;
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                nw[d] = m & (d < 2 ? along_x(S.neg, W.neg, d & 1) : row_of(S.neg, W.neg, d >> 1, d & 1));
                pw[d] = m & (d < 2 ? along_x(S.pos, W.pos, d & 1) : row_of(S.pos, W.pos, d >> 1, d & 1));
                any |= nw[d] | pw[d];
            }
            int id = rb;
            for (uint32_t w = any ? rs : 0u; w; ++id) {
                const uint32_t low = w & (0u - w), run = fill_up(m, low);
                w ^= low;
                if (!(any & run)) continue;
                int v = 0;
#pragma unroll
                for (int d = 0; d < 6; ++d) v += __popc(pw[d] & run) - __popc(nw[d] & run);
                if (v) atomicAdd(&S.votes[S.par[id]], v);
            }
        }
        if (INDEX) __syncthreads();

        // the boundary pieces' records
        const int base = (int)t * W.piece_stride;       // fixed slice of the piece table (31-bit ids)
        const int nb_ = S.nbnd;
        if (FAST && nb_ > BL) {                 // block-uniform; nothing global written yet
            if (tid == 0) W.ovf[atomicAdd(W.novf, 1)] = (int32_t)t;
            continue;
        }
        for (int k = tid; k < nb_; k += NT) {
            const int i = S.blist[k];
            const int d = S.desc[i];
            const int row = (d >> 5) & 0xff;
            const int pid = base + k;
            W.parent[pid] = pid;
            W.key[pid] = ((g.z0 + row / TY) * L.ny + (g.y0 + row % TY)) * L.nx + g.x0 + (d & 31);
            W.psize[pid] = S.aux[i] & (AUX_FACE - 1);
            if (INDEX) W.pvotes[pid] = S.votes[i];
            S.aux[i] = -1 - k;                   // from here on: boundary root k
            atomicAdd(&S.rowcnt[row / RPW], 0u - (1u << (8 * (row % RPW))));   // not an interior root
        }
        if (tid == 0)
            W.tinfo[t] = make_int4(g.x0, g.y0, g.z0,
                                   nb_ | (total << 11) | (lat << 24) | (INDEX && nb_ == 1 && S.nroot == 1 ? TILE_ONE_PIECE : 0));
        __syncthreads();

        // interior roots per row segment
        if (ly <= g.lastY && lz <= g.lastZ)
            W.cnt[L.seg0 + ((int64_t)(g.z0 + lz) * L.ny + (g.y0 + ly)) * L.nbx + g.bx] =
                INDEX ? reinterpret_cast<const uint8_t *>(S.rowcnt)[r] : (uint8_t)S.rowcnt[r / RPW];

        // one code per run (CODE_* encoding): aux of the run's root is -1 - k for boundary
        // piece k, else the interior piece's size
        uint16_t *C = W.codes + t * MR;
        for (int i = tid; i < total; i += NT) {
            const int v = S.par[i];
            const int a = S.aux[v];
            uint16_t c;
            if (v == i)
                c = a < 0 ? (uint16_t)(CODE_BOUNDARY | CODE_ROOT | (-1 - a)) : (uint16_t)(CODE_ROOT | a);
            else
                c = a < 0 ? (uint16_t)(CODE_BOUNDARY | (-1 - a)) : (uint16_t)(S.desc[v] & (DESC_TOUCH - 1));
            C[i] = c;
        }

        if (INDEX && S.nroot > nb_) {             // the tag of each run's piece, as if it were interior
            const int lane = tid & 31;
            uint32_t *T = W.tag + t * (MR / 16);
            for (int i0 = tid - lane; i0 < total; i0 += NT) {
                const int v = i0 + lane < total ? S.votes[S.par[i0 + lane]] : 1;
                const uint32_t in = __ballot_sync(0xffffffffu, v < 0), tie = __ballot_sync(0xffffffffu, v == 0);
                if (lane == 0) {
                    T[i0 >> 4] = in;
                    T[(i0 >> 4) + 1] = tie;
                }
            }
        }

        // Face lists.  A face site is connected when it and its neighbour across the
        // face are occupied.  Adjacent connected sites of a face lie in one piece on
        // either side, so one union per component of connected face sites suffices: a
        // connected site is emitted unless its face neighbour at lower x (y and z
        // faces) or at lower y or z (x faces) is connected too, which keeps the
        // lowest site of every component.  Both tiles of a face compute the same
        // connected sites, so their lists pair up entry by entry.  Warps take the faces
        // in turn (lo-x, hi-x, lo-y, hi-y, lo-z, hi-z); lane j owns one 32-bit word.
        {
            const int lane = tid & 31;
            for (int f = tid >> 5; f < 6; f += NT / 32) {
                const int hi = f & 1, axis = f >> 1;
                const bool ext = axis == 0 ? (hi ? g.extXhi : g.extXlo)
                               : axis == 1 ? (hi ? g.extYhi : g.extYlo) : (hi ? g.extZhi : g.extZlo);
                uint32_t c = 0;
                int row0 = 0;   // y and z faces: the row of this lane's word
                if (ext) {
                    if (axis == 0) {
                        if (lane < R / 32) c = hi ? (S.xol[lane] & S.nxhi[lane]) : (S.xo0[lane] & S.nxlo[lane]);
                    } else if (axis == 1) {
                        row0 = lane * TY + (hi ? g.lastY : 0);
                        if (lane < TZ) c = S.m[row0] & (hi ? S.nyhi[lane] : S.nylo[lane]);
                    } else {
                        row0 = (hi ? g.lastZ : 0) * TY + lane;
                        if (lane < TY) c = S.m[row0] & (hi ? S.nzhi[lane] : S.nzlo[lane]);
                    }
                }
                uint32_t prev = __shfl_up_sync(0xffffffffu, c, 1);
                if (lane == 0) prev = 0;
                uint32_t e;
                if (axis == 0) {
                    // bit i of word j is row 32 j + i; rows r - 1 (same plane) and r - TY
                    const uint32_t ym = ((c << 1) | (prev >> 31)) & ~SH::LY0;
                    const uint32_t zm = TY == 32 ? prev : ((c << (TY & 31)) | (prev >> ((32 - TY) & 31)));
                    e = c & ~ym & ~zm;
                } else {
                    e = c & ~(c << 1) & ~prev;
                }
                const int cnt = __popc(e);
                int inc = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, inc, d);
                    if (lane >= d) inc += u;
                }
                const int n = __shfl_sync(0xffffffffu, inc, 31);
                uint16_t *F = W.face + t * SH::FACE_STRIDE;
                const int off = f == 0 ? SH::OFF_LX : f == 1 ? SH::OFF_HX : f == 2 ? SH::OFF_LY
                              : f == 3 ? SH::OFF_HY : f == 4 ? SH::OFF_LZ : SH::OFF_HZ;
                int j = off + inc - cnt;
                while (e) {
                    const int b = __ffs(e) - 1;
                    e &= e - 1;
                    const int row = axis == 0 ? lane * 32 + b : row0;
                    const int x = axis == 0 ? (hi ? g.lastX : 0) : b;
                    F[j++] = (uint16_t)(-1 - S.aux[S.par[run_of(S.rbase[row], run_starts(S.m[row]), x)]]);
                }
                if (lane == 0) F[SH::OFF_CNT + f] = (uint16_t)n;
            }
        }
        __syncthreads();
    }
}

// --------------------------------------------------------------------------------------
// K2: face merge.  One warp per tile: its low face lists along x, y and z are joined
// entry by entry with the high face lists of its lower neighbours (for tile 0 of a
// periodic axis: the last tile, the wrap).  Each lane takes U entries at a time (a
// merge-schedule parameter: 1, 2 or 4) and
// walks the finds of all their endpoints in lockstep, so their loads are in flight
// together; the roots are then linked by CAS, and a lost CAS falls back to g_union.
// CTAs of FM_WARPS warps: a CTA's resources return only when its slowest warp (longest
// parent chain) is done, so small CTAs keep more warps waiting on loads in flight
// (32 CTAs of 2 warps still fill an SM).
// --------------------------------------------------------------------------------------
constexpr int FM_WARPS = 2;
constexpr int PF_WARPS = 4;
template <int TY, int TZ, int NL, int U>
__global__ void __launch_bounds__(32 * FM_WARPS)
k_face_merge(const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    constexpr int C = 2 * U;   // U unions, 2 U find chains per lane and step
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * FM_WARPS + (threadIdx.x >> 5);
    if (t >= ntiles) return;
    const LatDev &L = B.lat[(NL == 1) ? 0 : find_lattice(B.lat, B.n, t)];
    const TileGeo g = tile_geo<TY, TZ>(L, t);
    const int64_t plane = (int64_t)L.nbx * L.nby;
    const int64_t nbr[3] = {g.bx > 0 ? t - 1 : t + (L.nbx - 1),
                            g.by > 0 ? t - L.nbx : t + (int64_t)(L.nby - 1) * L.nbx,
                            g.bz > 0 ? t - plane : t + (int64_t)(L.nbz - 1) * plane};
    const uint16_t *F = W.face + t * SH::FACE_STRIDE;
    const int n0 = g.extXlo ? F[SH::OFF_CNT + 0] : 0;
    const int n1 = g.extYlo ? F[SH::OFF_CNT + 2] : 0;
    const int n2 = g.extZlo ? F[SH::OFF_CNT + 4] : 0;
    const int total = n0 + n1 + n2;
    const int base = (int)t * W.piece_stride;    // each tile owns a fixed slice of the piece table (31-bit ids)
    for (int i0 = 0; i0 < total; i0 += 32 * U) {
        int x[C], p[C];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * 32 + lane;
            if (i < total) {
                const int axis = i < n0 ? 0 : (i < n0 + n1 ? 1 : 2);
                const int j = i - (axis == 0 ? 0 : (axis == 1 ? n0 : n0 + n1));
                const int lo = axis == 0 ? SH::OFF_LX : axis == 1 ? SH::OFF_LY : SH::OFF_LZ;
                const int hi = axis == 0 ? SH::OFF_HX : axis == 1 ? SH::OFF_HY : SH::OFF_HZ;
                const int64_t nb = nbr[axis];
                x[2 * u] = base + F[lo + j];
                x[2 * u + 1] = (int)nb * W.piece_stride + W.face[nb * SH::FACE_STRIDE + hi + j];
            } else {
                x[2 * u] = x[2 * u + 1] = -1;   // no entry
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) p[c] = x[c] >= 0 ? __ldcg(W.parent + x[c]) : x[c];
        // finds with path halving, all chains one step per round
        for (int64_t it = 0;; ++it) {
            bool moving = false;
#pragma unroll
            for (int c = 0; c < C; ++c) moving |= p[c] != x[c];
            if (!moving) break;
            if (it > W.piece_cap) { atomicOr(W.status, STATUS_GLOBAL_LOOP); break; }
            int gp[C];
#pragma unroll
            for (int c = 0; c < C; ++c) gp[c] = p[c] != x[c] ? __ldcg(W.parent + p[c]) : x[c];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (p[c] == x[c]) continue;
                if (gp[c] == p[c]) {
                    x[c] = p[c];                      // p is a root
                } else {
                    __stcg(W.parent + x[c], gp[c]);   // path halving: gp is an ancestor of x
                    x[c] = gp[c];
                    p[c] = -2;                        // to reload
                }
            }
#pragma unroll
            for (int c = 0; c < C; ++c) p[c] = p[c] == -2 ? __ldcg(W.parent + x[c]) : (p[c] == x[c] || x[c] < 0 ? x[c] : p[c]);
        }
        // link the roots: the root with the larger key under the one with the smaller key
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int a = x[2 * u], b = x[2 * u + 1];
            if (a < 0 || a == b) continue;
            if (__ldg(W.key + b) < __ldg(W.key + a)) { const int tmp = a; a = b; b = tmp; }
            if (atomicCAS(W.parent + b, b, a) != b) g_union(W.parent, W.key, a, b, W.piece_cap, W.status);
        }
    }
}

// --------------------------------------------------------------------------------------
// K3: piece finalize (one warp per tile, one piece per lane).  Size additions into
// the same cluster root are combined per group of lanes; with HOT (a merge-schedule
// parameter) the root that collects most of them -- the percolating cluster's -- is
// further combined per warp and per CTA of PF_WARPS warps, because it collects pieces
// from most tiles.
// --------------------------------------------------------------------------------------
template <int NL, bool HOT>
__global__ void __launch_bounds__(32 * PF_WARPS)
k_piece_finalize(const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles) {
    grid_dep_wait();
    __shared__ int hot_target[PF_WARPS];   // per warp: the cluster root its pieces fed most, and the sum
    __shared__ int hot_sum[PF_WARPS], hot_votes[PF_WARPS];
    const int64_t t = (int64_t)blockIdx.x * PF_WARPS + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // The root that collects most sizes (the percolating cluster's, above all) is added
    // once per warp and then once per CTA; other roots once per group of lanes.
    int hot = -1, hot_acc = 0, hot_vacc = 0;
    const int nbnd = t < ntiles ? W.tinfo[t].w & 0x7ff : 0;
    if (nbnd > 0) {
        const LatDev &L = B.lat[(NL == 1) ? 0 : find_lattice(B.lat, B.n, t)];
        for (int j0 = 0; j0 < nbnd; j0 += 32) {
            const int j = j0 + lane;
            const bool valid = j < nbnd;
            const int pid = (int)t * W.piece_stride + j;
            int root = -1, add = 0, vadd = 0;
            if (valid) {
                root = g_find_ro(W.parent, pid, W.piece_cap, W.status);
                if (root != pid) {
                    __stcg(W.parent + pid, root);
                    add = W.psize[pid];
                    if (W.pvotes) vadd = W.pvotes[pid];     // votes of an index field add up like sizes
                    // from here on key[pid] is the cluster's label and psize[pid] < 0 marks a
                    // non-root; only roots' keys are read by other threads, and a root's key
                    // never changes
                    W.key[pid] = __ldcg(W.key + root);
                    W.psize[pid] = -1;
                } else {
                    const int k = W.key[pid];
                    const int q = k / L.nx, x = k - q * L.nx;          // q = z * ny + y
                    const int64_t seg = L.seg0 + (int64_t)q * L.nbx + (x >> 5);
                    // one byte per segment (at most 16 roots): add to it inside its aligned word
                    atomicAdd(reinterpret_cast<unsigned int *>(W.cnt + (seg & ~(int64_t)3)),
                              1u << (8 * (int)(seg & 3)));
                }
            }
            const int target = (valid && root != pid) ? root : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, target);
            const int sum = (int)__reduce_add_sync(peers, (unsigned)add);
            const int vsum = W.pvotes ? (int)__reduce_add_sync(peers, (unsigned)vadd) : 0;
            const bool leader = target >= 0 && lane == __ffs(peers) - 1;
            if (HOT && hot < 0) {   // warp-uniform: the first chunk names the warp's hot root (its largest group)
                const unsigned key = leader ? ((unsigned)__popc(peers) << 5) | (unsigned)lane : 0u;
                const unsigned best = __reduce_max_sync(0xffffffffu, key);
                if (best) hot = __shfl_sync(0xffffffffu, target, (int)(best & 31u));
            }
            if (leader) {
                if (target == hot) {
                    hot_acc += sum;
                    hot_vacc += vsum;
                } else {
                    atomicAdd(W.psize + target, sum);
                    if (vsum) atomicAdd(W.pvotes + target, vsum);
                }
            }
        }
    }
    if (!HOT) return;
    hot_acc = (int)__reduce_add_sync(0xffffffffu, (unsigned)hot_acc);
    if (W.pvotes) hot_vacc = (int)__reduce_add_sync(0xffffffffu, (unsigned)hot_vacc);
    if (lane == 0) {
        hot_target[wid] = hot;
        hot_sum[wid] = hot_acc;
        hot_votes[wid] = hot_vacc;
    }
    __syncthreads();
    if (threadIdx.x < PF_WARPS) {   // one add per distinct hot root of the CTA
        const int h = hot_target[threadIdx.x];
        if (h >= 0) {
            bool first = true;
            int s = 0, v = 0;
            for (int w = 0; w < PF_WARPS; ++w)
                if (hot_target[w] == h) {
                    if (w < (int)threadIdx.x) first = false;
                    s += hot_sum[w];
                    v += hot_votes[w];
                }
            if (first) atomicAdd(W.psize + h, s);
            if (first && v) atomicAdd(W.pvotes + h, v);
        }
    }
}

// --------------------------------------------------------------------------------------
// S1-S2: exclusive scan of the cluster roots per lattice row (the sum of the row's
// segment counts); ranks inside a row are completed by flatten from the segment
// counts before its own.  Launches and round trips bound it, not bytes: two launches
// (block sums, then the rows) where four were (block sums, their scan, the rows, and
// the counts and histograms), and blocks of 1024 rows where 4096 were, took a 256^3
// call from 94.3 to 74.2 us.
// --------------------------------------------------------------------------------------
constexpr int SCAN_NT = 256;
constexpr int SCAN_PER = 4;
constexpr int SCAN_CH = SCAN_NT * SCAN_PER;

template <int NL>
__device__ __forceinline__ uint32_t row_roots(const LatBatch<NL> &B, const uint8_t *cnt, int64_t q) {
    const LatDev &L = B.lat[(NL == 1) ? 0 : find_lattice_row(B.lat, B.n, q)];
    return bytes_sum(cnt, L.seg0 + (q - L.row0) * L.nbx, L.nbx);
}

template <int NL>
__global__ void __launch_bounds__(SCAN_NT) k_scan_reduce(const __grid_constant__ LatBatch<NL> B,
                                                         const uint8_t *cnt, int64_t n, uint32_t *bsum) {
    grid_dep_wait();
    __shared__ uint32_t red[SCAN_NT / 32];
    const int64_t b0 = (int64_t)blockIdx.x * SCAN_CH;
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_PER; ++j) {
        const int64_t i = b0 + (int64_t)j * SCAN_NT + threadIdx.x;
        if (i < n) s += row_roots(B, cnt, i);
    }
    for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (int w = 0; w < SCAN_NT / 32; ++w) tot += red[w];
        bsum[blockIdx.x] = tot;
    }
    // flatten adds to the histograms: cleared here, two passes before it
    for (int i = blockIdx.x * SCAN_NT + threadIdx.x; i < 32 * B.n; i += gridDim.x * SCAN_NT)
        if (B.lat[i >> 5].hist) B.lat[i >> 5].hist[i & 31] = 0;
}

// single block: exclusive scan of the block sums in place
__global__ void __launch_bounds__(1024) k_scan_blocks(uint32_t *bsum, int64_t nb) {
    grid_dep_wait();
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t carry;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t c0 = 0; c0 < nb; c0 += 1024) {
        const int64_t i = c0 + threadIdx.x;
        const uint32_t v = i < nb ? bsum[i] : 0u;
        uint32_t inc = v;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += u;
        }
        if (lane == 31) wsum[wid] = inc;
        __syncthreads();
        if (wid == 0) {
            uint32_t w = wsum[lane], wi = w;
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, wi, d);
                if (lane >= d) wi += u;
            }
            wsum[lane] = wi - w;
        }
        __syncthreads();
        const uint32_t ex = carry + wsum[wid] + inc - v;
        if (i < nb) bsum[i] = ex;
        __syncthreads();
        if (threadIdx.x == 1023) carry = ex + v;
        __syncthreads();
    }
}

// scanned: bsum holds the exclusive scan of the block sums; else the sums themselves, and
// every block adds up those before it (at most SCAN_DIRECT: a few loads a thread, for
// one launch less).
constexpr int64_t SCAN_DIRECT = 2048;
template <int NL>
__global__ void __launch_bounds__(SCAN_NT) k_scan_apply(const __grid_constant__ LatBatch<NL> B, const uint8_t *cnt,
                                                        int64_t n, const uint32_t *bsum, uint32_t *pre, bool scanned) {
    grid_dep_wait();
    __shared__ uint32_t wsum[SCAN_NT / 32], wbase[SCAN_NT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t before = 0;
    if (!scanned)
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += SCAN_NT) before += bsum[i];
    else if (threadIdx.x == 0)
        before = bsum[blockIdx.x];
    const int64_t b0 = (int64_t)blockIdx.x * SCAN_CH + (int64_t)threadIdx.x * SCAN_PER;
    uint32_t v[SCAN_PER];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_PER; ++j) {
        const int64_t i = b0 + j;
        v[j] = i < n ? row_roots(B, cnt, i) : 0u;
        s += v[j];
    }
    uint32_t inc = s;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += u;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31) {
        wsum[wid] = inc;
        wbase[wid] = before;
    }
    __syncthreads();
    uint32_t run = inc - s;
#pragma unroll
    for (int w = 0; w < SCAN_NT / 32; ++w) {
        run += wbase[w];
        if (w < wid) run += wsum[w];
    }
#pragma unroll
    for (int j = 0; j < SCAN_PER; ++j) {
        const int64_t i = b0 + j;
        if (i <= n) pre[i] = run;   // pre[n] = total
        run += v[j];
    }
}

// --------------------------------------------------------------------------------------
// K4: flatten (decode run codes; no union-find)
//
// Per tile: one thread per row numbers the row's runs (a block scan) and gives each run
// its own first site as label; one thread per run then replaces that label unless the
// run is the first of an interior piece (balanced over the threads whatever the rows
// hold) and notes the cluster roots in a bitmap; one thread per row ranks its row's
// roots and collects their sizes; and the labels leave, four sites a lane, straight to
// global memory.  The next tile's record, words, codes and boundary pieces come by bulk
// copy while the labels are written.
//
// Bound by instruction issue at p_c (1.2 warp instructions a site, 72 % of the issue
// rate at 512^3); on fields of long runs the label stores are two thirds of it.  Against
// a loop over each row's runs that decoded, ranked and filled them into a staged tile for a
// TMA store: 1.35 against 1.57 ms at 1024^3, p_c, 0.109 against 0.126 ms on a 512^3 bijel, 53
// against 65 us at 387 x 283 x 221 (unaligned rows), and no faster on blocks of 16^3 (0.91
// against 0.92 ms).  Slower on sixteen runs a row (stripes of one site at 512^3: 0.31 against
// 0.19 ms, of a call of 1.14 against 1.46), whose codes do not fit the staged ones, and on
// rows of four sites (0.13 against 0.09 ms at 4 x 2048 x 2048, p_c), where an eighth of the
// lanes store.
// --------------------------------------------------------------------------------------
// Resident threads of an SM (40 registers each).  2048 (32 registers, spills): 1.63 ms at
// 1024^3, p_c, against 1.50 for 1536 and 1.59 for 1280, in the form of that time.
constexpr int FLAT_THREADS = 1536;
// Items a CTA takes, each a stretch of consecutive tiles, so that a row's ranks and half
// full size sectors carry over along x: 4 or 1 longer ones, 1.39 and 1.38 against 1.41 ms
// at 1024^3, p_c, but 0.92 against 0.89 ms on blocks of 16^3, and a field whose parts
// differ needs several to even out.
constexpr int FLAT_ITEMS = 8;
template <int TY, int TZ>
struct FlatSmem {
    using SH = TileShape<TY, TZ>;
    // staged boundary pieces (a tile at p_c has about 124), few enough that six CTAs share an SM
    // (256 of them and five CTAs: 1.39 against 1.35 ms at 1024^3, p_c)
    static constexpr int GL = SH::MAX_BOUNDARY < 192 ? SH::MAX_BOUNDARY : 192;
    static constexpr int CC = SH::MR_FAST;                                       // staged run codes
    static_assert(GL % 4 == 0 && CC % 8 == 0 && SH::MAX_BOUNDARY % 4 == 0 && (SH::MAXRUNS * 2) % 16 == 0,
                  "bulk copies of whole 16-byte blocks from 16-byte aligned slices");
    // the staged tile (bulk copies)
    alignas(16) uint32_t words[SH::R];         // occupancy word of each row
    alignas(16) uint16_t codes[CC];            // run codes
    // tab[0, GL): label of each boundary piece's cluster (copied); tab[GL, GL + R): first site of
    // each row (computed)
    // (an interior root's code holds a size, whose row is read but not used: one entry more)
    alignas(16) int tab[GL + SH::R + 4];
    alignas(16) int gsize[GL + 4];             // cluster size if the piece is the cluster root, else -1;
                                               // [GL] = 1 stands for every interior piece
    alignas(16) int4 tinfo;
    uint64_t bar;                              // completion of the copies
    uint4 row[SH::R];                          // occupancy word, run starts, first run id of each row
    int lab[SH::MAXRUNS];                      // label of each run
    uint32_t rootbal[SH::MAXRUNS / 32 + 1];    // cluster-root bits of each 32 run ids
    alignas(16) int pend[SH::R][8];            // each row's sizes not yet written, by place in their sector
                                               // (mod 8: two sectors)
    int warp_tmp[SH::NT / 32];
    int hist[32];
};

// SLAB: one slab of a lattice split along z (W.site_off added to every label, each
// cluster's label written to W.roots); a separate instance, so that the common path
// carries neither.
template <int TY, int TZ, int NL, bool SLAB>
__global__ void __launch_bounds__(TY * TZ, FLAT_THREADS / (TY * TZ))
k_flatten(const __grid_constant__ LatBatch<NL> B, Work W, int64_t ntiles, uint32_t span) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    using FS = FlatSmem<TY, TZ>;
    constexpr int R = SH::R, NT = SH::NT, NW = NT / 32, MR = SH::MAXRUNS;
    constexpr int GL = FS::GL, CC = FS::CC;
    const uint32_t MB = (uint32_t)W.piece_stride;      // t * MB is a piece id: 31 bits
    extern __shared__ __align__(128) unsigned char smem_raw[];
    FS &S = *reinterpret_cast<FS *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

    if (tid < 32) S.hist[tid] = 0;
    if (tid == 0) S.gsize[GL] = 1;
    // Thread 0 issues the copies of a tile (its record ti says how much there is).  If they
    // do not complete within their bound the CTA records STATUS_TMA_TIMEOUT and stages
    // its tiles by plain loads from then on (prefetch becomes false, uniformly).
    auto issue = [&](uint32_t t, int4 ti) {
        const int nb = ti.w & 0x7ff, total = (ti.w >> 11) & 0x1fff;
        const int nc = min((total + 7) & ~7, CC), ng = min((nb + 3) & ~3, GL);
        fence_proxy_async();
        mbar_arrive_expect_tx(&S.bar, (uint32_t)(4 * R + 16 + 2 * nc + 8 * ng));
        bulk_load(&S.tinfo, W.tinfo + t, 16u, &S.bar);
        bulk_load(S.words, W.mask + (size_t)t * R, 4u * R, &S.bar);
        if (nc) bulk_load(S.codes, W.codes + (size_t)t * MR, 2u * nc, &S.bar);
        if (ng) {
            bulk_load(S.tab, W.key + t * MB, 4u * ng, &S.bar);
            bulk_load(S.gsize, W.psize + t * MB, 4u * ng, &S.bar);
        }
    };
    // CTA b takes the tiles [i span, (i + 1) span) of every item i = b, b + gridDim.x, ...
    const uint32_t nt = (uint32_t)ntiles, skip = (gridDim.x - 1u) * span;
    auto next_tile = [&](uint32_t &t, uint32_t &end) {
        if (++t >= end) {
            t = end + skip;
            end = t < nt ? min(t + span, nt) : t;
        }
    };
    uint32_t t = blockIdx.x * span, end = min(t + span, nt);
    bool fresh = true;                                 // uniform: the first tile of an item
    int4 ti_next = make_int4(0, 0, 0, 0);              // thread 0: the record of the next tile
    if (tid == 0) {
        mbar_init(&S.bar, 1);
        fence_mbar_init();
        // the first tile's counts are not waited for: all that can be staged is copied
        if (t < nt) issue(t, make_int4(0, 0, 0, min(GL, (int)MB) | (CC << 11)));
        uint32_t t1 = t, e1 = end;
        next_tile(t1, e1);
        if (t1 < nt) ti_next = W.tinfo[t1];
    }
    __syncthreads();
    bool prefetch = true;
    uint32_t parity = 0;
    int cur_lat = -1;
    constexpr uint32_t NO_RANK = ~0u;                  // ranks stay below 2^30
    uint32_t rank = NO_RANK, lo = NO_RANK;             // of this row: next rank, first one not written
    while (t < nt) {
        uint32_t m, rs;
        int inc;
        for (;;) {
            bool done = true;
            if (prefetch) {
                done = mbar_wait_bounded(&S.bar, parity);
            } else {
                const int4 ti = W.tinfo[t];
                const int nb = ti.w & 0x7ff, total = (ti.w >> 11) & 0x1fff;
                if (tid == 0) S.tinfo = ti;
                S.words[tid] = W.mask[(size_t)t * R + tid];
                for (int k = tid; k < total && k < CC; k += NT) S.codes[k] = W.codes[(size_t)t * MR + k];
                for (int k = tid; k < nb && k < GL; k += NT) {
                    S.tab[k] = W.key[t * MB + k];
                    S.gsize[k] = W.psize[t * MB + k];
                }
            }
            m = S.words[tid];
            rs = run_starts(m);
            inc = __popc(rs);                          // run ids: inclusive scan over the warp's rows
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += u;
            }
            if (lane == 31) S.warp_tmp[wid] = inc;
            if (!__syncthreads_or(!done)) break;       // ... and every thread is done with S.row, S.lab
            if (tid == 0) atomicOr(W.status, STATUS_TMA_TIMEOUT);
            mbar_wait_bounded(&S.bar, parity);         // the copies still in flight
            prefetch = false;
        }
        parity ^= 1;
        const int4 ti = S.tinfo;
        const int nb = ti.w & 0x7ff, total = (ti.w >> 11) & 0x1fff, lat = NL == 1 ? 0 : ti.w >> 24;
        const LatDev &L = B.lat[lat];
        const int r = tid, ly = r % TY, lz = r / TY;
        // a lattice's count, with its first tile (a uint32 difference: the prefix may wrap over
        // a launch, a lattice's count does not)
        if (tid == 0 && L.ncl && (ti.x | ti.y | ti.z) == 0)
            L.ncl[0] = (int64_t)(uint32_t)(W.pre[L.row0 + (int64_t)L.nz * L.ny] - W.pre[L.row0]);
        // Rank base of this row: the roots of the lattice's earlier rows, then of this row's
        // earlier segments; carried on while the tiles follow each other along x.  Looked up
        // in the first tile where one of the warp's rows has a run (looked up whether there is one
        // or not, an empty 65536 x 64 x 4 took 589 us against 282).
        const int q = (ti.z + lz) * L.ny + (ti.y + ly);
        const bool valid_row = ti.y + ly < L.ny && ti.z + lz < L.nz;
        if (fresh || ti.x == 0) rank = lo = NO_RANK;
        if (__any_sync(0xffffffffu, rs != 0u) && rank == NO_RANK && valid_row) {
            rank = W.pre[L.row0 + q] - W.pre[L.row0];
            if (ti.x) rank += bytes_sum(W.cnt, L.seg0 + (int64_t)q * L.nbx, ti.x / TX);
            lo = rank;
        }
        if (lat != cur_lat) {                          // uniform: flush the histogram per lattice
            if (cur_lat >= 0 && tid < 32 && S.hist[tid] && B.lat[cur_lat].hist)
                atomicAdd(reinterpret_cast<unsigned long long *>(B.lat[cur_lat].hist) + tid,
                          (unsigned long long)S.hist[tid]);
            if (tid < 32) S.hist[tid] = 0;
            cur_lat = lat;
        }
        int rb = inc - __popc(rs);
#pragma unroll
        for (int w = 0; w < NW; ++w)
            if (w < wid) rb += S.warp_tmp[w];
        S.row[r] = make_uint4(m, rs, (uint32_t)rb, 0u);

        // every run starts with its own first site as label
        const int soff = SLAB ? (int)W.site_off : 0;   // labels of a slab are sites of the whole lattice
        const int site_row = q * L.nx + ti.x + soff;
        S.tab[GL + r] = site_row;
        {
            int *lp = S.lab + rb;
            for (uint32_t w = rs; w;) {
                const uint32_t low = w & (0u - w);
                w ^= low;
                *lp++ = site_row + top_bit(low);
            }
        }
        __syncthreads();

        // The next two steps are compiled for tiles that are staged whole and for others.
        const uint16_t *C = W.codes + (size_t)t * MR;
        auto decode_runs = [&](auto BIG) {
            constexpr bool big = decltype(BIG)::value;
            // one run per thread: the label of its boundary piece's cluster, or of the first
            // run of its interior piece; and whether it is its cluster's first run.  The
            // pieces' labels and the rows' first sites are one table (tab), and gsize ends
            // with a positive entry for the interior pieces, so that nothing branches; the
            // lanes past the last run repeat it.
            for (int i0 = wid * 32; i0 < total; i0 += NT) {
                const int i = i0 + lane, ic = min(i, total - 1);
                const int c = (!big || ic < CC) ? (int)S.codes[ic] : (int)__ldg(C + ic);
                const int k = c & CODE_LOW;
                const bool isb = (c & CODE_BOUNDARY) != 0;
                int lab, gs;
                if (big && isb && k >= GL) {
                    lab = __ldg(W.key + (t * MB + k));
                    gs = __ldg(W.psize + (t * MB + k));
                } else {
                    lab = S.tab[isb ? k : GL + (k >> 5)];
                    gs = S.gsize[isb ? k : GL];
                }
                lab += isb ? soff : (k & 31);          // piece labels are sites of the slab
                if ((c & (CODE_BOUNDARY | CODE_ROOT)) != CODE_ROOT) S.lab[i] = lab;
                const uint32_t bal = __ballot_sync(0xffffffffu, gs > 0 && (c & CODE_ROOT));
                if (lane == 0) S.rootbal[i0 >> 5] = bal;
            }
        };
        const bool big = total > CC || nb > GL;        // uniform
        if (big) decode_runs(std::true_type{});
        else decode_runs(std::false_type{});
        __syncthreads();

        // a4, a6, a7: the roots of each row in x order get their ranks, sizes and
        // histogram entries
        const int n = __popc(rs);
        uint32_t bits = 0;                             // the row's runs are bits 0 .. n - 1 (n <= 16)
        if (n) bits = __funnelshift_r(S.rootbal[rb >> 5], S.rootbal[(rb >> 5) + 1], (uint32_t)rb & 31u) &
                      ((1u << n) - 1u);
        // Sizes wait in shared memory until their 32-byte sector is full (a row has fewer roots
        // in a tile than that; the next tile along x brings the rest): stores of single
        // sizes left part-written sectors that cost flatten 0.3 to 0.45 ms at 1024^3, p_c.
        const uint32_t cap = (uint32_t)min(L.sizes_cap, (int64_t)INT32_MAX);   // ranks stay below 2^30
        const uint32_t place = (uint32_t)(reinterpret_cast<uintptr_t>(L.sizes) >> 3);
        if (L.inside) {                                // index fields: the tags, in rank order like the sizes
            uint32_t k = rank;
            for (uint32_t w = bits; w && k < cap; w &= w - 1u, ++k) {
                const int id = rb + __ffs(w) - 1;
                const int c = id < CC ? (int)S.codes[id] : (int)__ldg(C + id);
                const uint32_t *T = W.tag + (size_t)t * (MR / 16) + 2 * (id >> 5);
                const int v = (c & CODE_BOUNDARY) ? W.pvotes[t * MB + (c & CODE_LOW)]
                            : (T[0] >> (id & 31)) & 1u ? -1 : (T[1] >> (id & 31)) & 1u ? 0 : 1;
                L.inside[k] = (int8_t)(v < 0 ? 1 : (v > 0 ? 0 : -1));
            }
        }
        auto flush = [&](bool all) {                   // the full sectors among ranks lo .. rank - 1, or all
            while (lo < rank) {
                const uint32_t e = lo + 4u - ((lo + place) & 3u);   // the first rank of the next sector
                if (e > rank && !all) break;
                if (e - lo == 4u && e <= rank && e <= cap) {
                    const int4 p = *reinterpret_cast<const int4 *>(&S.pend[r][(lo + place) & 7u]);
                    longlong2 *to = reinterpret_cast<longlong2 *>(L.sizes + lo);
                    to[0] = make_longlong2(p.x, p.y);
                    to[1] = make_longlong2(p.z, p.w);
                    lo = e;
                } else {
                    const uint32_t last = min(e, rank);
                    for (; lo < last; ++lo)
                        if (lo < cap) L.sizes[lo] = S.pend[r][(lo + place) & 7u];
                }
            }
        };
        auto write_roots = [&](auto BIG) {
            constexpr bool bigt = decltype(BIG)::value;
            while (bits) {
                do {
                    const uint32_t low = bits & (0u - bits);
                    bits ^= low;
                    const int id = rb + top_bit(low);
                    const int c = (!bigt || id < CC) ? (int)S.codes[id] : (int)__ldg(C + id);
                    const int k = c & CODE_LOW;
                    const bool isb = (c & CODE_BOUNDARY) != 0;
                    const int gs = (bigt && isb && k >= GL) ? __ldg(W.psize + (t * MB + k)) : S.gsize[isb ? k : GL];
                    const int size = isb ? gs : k;
                    if (SLAB && rank < cap) W.roots[rank] = S.lab[id];   // a root's label is its own first site
                    S.pend[r][(rank + place) & 7u] = size;
                    atomicAdd(&S.hist[top_bit((uint32_t)size)], 1);
                    ++rank;
                } while (bits && rank - lo < 8u);
                flush(false);
            }
        };
        if (big) write_roots(std::true_type{});
        else write_roots(std::false_type{});
        const uint32_t t_done = t;
        next_tile(t, end);
        fresh = t != t_done + 1u;
        if (fresh || ti.x + TX >= L.nx) flush(true);
        __syncthreads();                               // every thread is done with the staged tile
        if (tid == 0 && prefetch && t < nt) {
            issue(t, ti_next);
            uint32_t t1 = t, e1 = end;
            next_tile(t1, e1);
            if (t1 < nt) ti_next = W.tinfo[t1];
        }

        // a5: the labels.  Rows of whole 16-byte blocks: lane l writes sites x4 = 4 (l % 8) .. + 3
        // of row l / 8 of each group of 4 rows.  The warps step through the rows by whole
        // planes, so that y stays and z grows.  Other rows: one site a lane.
        constexpr int ZS = NW * 4 / TY;
        static_assert(ZS >= 1 && ZS * TY == NW * 4, "the warps' rows fill whole planes");
        const int64_t sxy = (int64_t)L.nx * L.ny;
        const int nrow = min(TZ, L.nz - ti.z) * TY;    // rows of the tile's planes inside the lattice
        if ((L.nx & 3) == 0 && (reinterpret_cast<uintptr_t>(L.labels) & 15) == 0) {
            const int x4 = (lane & 7) * 4;
            const int row0 = wid * 4 + (lane >> 3), y = ti.y + row0 % TY;
            const uint32_t below = (1u << x4) - 1u;
            int32_t *out = L.labels + (int64_t)(ti.z + row0 / TY) * sxy + (int64_t)y * L.nx + ti.x + x4;
            if (y < L.ny && ti.x + x4 < L.nx)
#pragma unroll 2
                for (int row = row0; row < nrow; row += NW * 4, out += ZS * sxy) {
                    const uint4 w = S.row[row];
                    const uint32_t mm = w.x >> x4, ss = w.y >> x4;
                    const int *lp = S.lab + (int)w.z - 1 + __popc(w.y & below);   // the last run that starts below x4
                    int4 v = make_int4(-1, -1, -1, -1);
                    if (ss & 1u) ++lp;
                    if (mm & 1u) v.x = *lp;
                    if (ss & 2u) ++lp;
                    if (mm & 2u) v.y = *lp;
                    if (ss & 4u) ++lp;
                    if (mm & 4u) v.z = *lp;
                    if (ss & 8u) ++lp;
                    if (mm & 8u) v.w = *lp;
                    __stcs(reinterpret_cast<int4 *>(out), v);
                }
        } else if (ti.x + lane < L.nx) {
            const uint32_t le = le_mask(lane);
            for (int yy = wid; yy < TY && ti.y + yy < L.ny; yy += NW) {
                int32_t *out = L.labels + (int64_t)ti.z * sxy + (int64_t)(ti.y + yy) * L.nx + ti.x + lane;
#pragma unroll 2
                for (int row = yy; row < nrow; row += TY, out += sxy) {
                    const uint4 w = S.row[row];
                    __stcs(out, site_label(w.x, w.y, (int)w.z, le, S.lab));
                }
            }
        }
    }
    __syncthreads();
    if (cur_lat >= 0 && tid < 32 && S.hist[tid] && B.lat[cur_lat].hist)
        atomicAdd(reinterpret_cast<unsigned long long *>(B.lat[cur_lat].hist) + tid, (unsigned long long)S.hist[tid]);
}

// --------------------------------------------------------------------------------------
// Interior state of every site of an index field (Sec. 6: 1 far inside, 0 far outside): a
// far site (I < -0.5) takes the tag that its cluster's votes give (-1 for a tie), a near
// site the side its value names (step 2: -d inside, +d outside), 1 for I < 0 and 0
// otherwise.  Like flatten it decodes the runs of each tile, but it needs neither ranks
// nor labels: it reads the words and codes and writes a byte a site.  One tile per CTA,
// one row per thread; a tile of one piece, as most are, needs no codes.  729 capsules at
// 1024^3 take 0.30 ms, two thirds of the copy rate for its 1.3 GB (0.51 with codes read in
// every tile and half sectors stored); the rest is the chain of dependent loads at a CTA's
// start (record, root, votes), which a 64-bit product in the root's address made 7 % longer.
// --------------------------------------------------------------------------------------
template <int TY, int TZ>
__global__ void __launch_bounds__(TY * TZ) k_state(const LatDev L, Work W, int8_t *state, bool vec) {
    grid_dep_wait();
    using SH = TileShape<TY, TZ>;
    constexpr int R = SH::R, NT = SH::NT, NW = NT / 32, MR = SH::MAXRUNS;
    __shared__ int8_t ptag[SH::MAX_BOUNDARY];          // tag of each boundary piece's cluster
    __shared__ uint2 row[R];                           // bits of the states 1 and -1 of each row
    __shared__ int warp_tmp[NW];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t t = blockIdx.x;
    const int32_t *parent = W.parent + blockIdx.x * (uint32_t)W.piece_stride;   // a piece id: 31 bits
    const int4 ti = W.tinfo[t];
    const int nb = ti.w & 0x7ff;
    const uint32_t m = W.mask[t * R + tid], near_in = W.neg[t * R + tid];
    const int root0 = parent[0];                       // of piece 0, if there is one
    const uint32_t rs = run_starts(m);
    uint32_t ones = near_in, ties = 0;
    if (ti.w & TILE_ONE_PIECE) {                       // uniform: the tile's far sites are one piece
        const int v = W.pvotes[root0];
        if (v < 0) ones |= m;
        if (v == 0) ties = m;
    } else {
        int inc = __popc(rs);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += u;
        }
        if (lane == 31) warp_tmp[wid] = inc;
        for (int k = tid; k < nb; k += NT) {
            const int v = W.pvotes[parent[k]];             // piece_finalize left every piece at its root
            ptag[k] = (int8_t)(v < 0 ? 1 : (v > 0 ? 0 : -1));
        }
        __syncthreads();
        int id = inc - __popc(rs);
#pragma unroll
        for (int w = 0; w < NW; ++w)
            if (w < wid) id += warp_tmp[w];
        for (uint32_t w = rs; w; ++id) {
            const uint32_t low = w & (0u - w), run = fill_up(m, low);
            w ^= low;
            const int c = __ldg(W.codes + t * MR + id);
            int tag;
            if (c & CODE_BOUNDARY) {
                tag = ptag[c & CODE_LOW];
            } else {
                const uint32_t *T = W.tag + t * (MR / 16) + 2 * (id >> 5);
                tag = (__ldg(T) >> (id & 31)) & 1u ? 1 : ((__ldg(T + 1) >> (id & 31)) & 1u ? -1 : 0);
            }
            if (tag > 0) ones |= run;
            if (tag < 0) ties |= run;
        }
    }
    const int64_t sxy = (int64_t)L.nx * L.ny;
    // bits 0-3 of n as the low bits of four bytes
    auto spread = [](uint32_t n) { return ((n & 15u) * 0x00204081u) & 0x01010101u; };
    if (vec) {      // rows of whole 16-byte blocks: two lanes a row, so that a store fills sectors
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = wid * 32 + h * 16 + (lane >> 1), x = 16 * (lane & 1);
            const uint32_t o = __shfl_sync(0xffffffffu, ones, h * 16 + (lane >> 1)) >> x;
            const uint32_t e = __shfl_sync(0xffffffffu, ties, h * 16 + (lane >> 1)) >> x;
            uint32_t b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = spread(o >> (4 * j)) | spread(e >> (4 * j)) * 255u;
            const int y = ti.y + r % TY, z = ti.z + r / TY;
            if (y < L.ny && z < L.nz && ti.x + x < L.nx)
                __stcs(reinterpret_cast<int4 *>(state + (int64_t)z * sxy + (int64_t)y * L.nx + ti.x + x),
                       make_int4((int)b[0], (int)b[1], (int)b[2], (int)b[3]));
        }
        return;
    }
    row[tid] = make_uint2(ones, ties);
    __syncthreads();
    const int nrow = min(TZ, L.nz - ti.z) * TY;
    for (int r = wid; r < nrow; r += NW) {
        const int y = ti.y + r % TY, z = ti.z + r / TY;
        if (y >= L.ny || ti.x + lane >= L.nx) continue;
        const uint2 w = row[r];
        state[(int64_t)z * sxy + (int64_t)y * L.nx + ti.x + lane] =
            (int8_t)((w.x >> lane) & 1u ? 1 : ((w.y >> lane) & 1u ? -1 : 0));
    }
}

// --------------------------------------------------------------------------------------
// Interior state of slowly moving membranes (Sec. 6, last paragraph): only the sites
// near a membrane now change, to the side their value names; every other site keeps
// its state.
// --------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t update_byte(uint32_t w, int b, float v) {
    const uint32_t side = v < 0.0f ? 1u : 0u;
    return (v < -0.5f) ? w : ((w & ~(0xffu << (8 * b))) | (side << (8 * b)));
}

// Dense form.  vec: all three arrays 16-byte aligned; then 16 sites per step, one
// 16-byte state load and store and four 16-byte index loads.
__global__ void __launch_bounds__(256) k_interior_update(const int8_t *prev, const float *index, int64_t n,
                                                          int8_t *out, bool vec) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (vec) {
        const int64_t nv = n / 16;
        for (int64_t i = t0; i < nv; i += stride) {
            const int4 sp = __ldcs(reinterpret_cast<const int4 *>(prev) + i);
            uint32_t w[4] = {(uint32_t)sp.x, (uint32_t)sp.y, (uint32_t)sp.z, (uint32_t)sp.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 v = __ldcs(reinterpret_cast<const float4 *>(index) + 4 * i + q);
                w[q] = update_byte(w[q], 0, v.x);
                w[q] = update_byte(w[q], 1, v.y);
                w[q] = update_byte(w[q], 2, v.z);
                w[q] = update_byte(w[q], 3, v.w);
            }
            __stcs(reinterpret_cast<int4 *>(out) + i, make_int4((int)w[0], (int)w[1], (int)w[2], (int)w[3]));
        }
        done = nv * 16;
    }
    for (int64_t s = done + t0; s < n; s += stride) {
        const float v = index[s];
        out[s] = (v < -0.5f) ? prev[s] : (int8_t)(v < 0.0f ? 1 : 0);
    }
}

// Dense form in place: a far site's state stays where it is, so only the 32-byte sectors of
// states (32 sites, two lanes) that hold a near one are read and written, and away from
// membranes the pass is the read of the index field.  A warp half of whose sectors held one
// loads its next states along with the index values.  Bound by memory; four CTAs an SM draw
// more from it than eight, above all on fields full of near sites, where eight lost to the
// form that moves every state.  In us, with none / a twentieth / all of the sites near:
//   2^30 sites   587 / 871 / 927 with four, 668 / 925 / 1013 with eight, 965 with every state moved
//   343 M sites  191 / 284 / 294 with four, 214 / 295 / 323 with eight, 309 with every state moved
// Groups of four sites, read and written one by one, were slower on fuller fields.
// vec: both arrays 16-byte aligned.
constexpr int UPDATE_IN_PLACE_CTAS = 4;   // of 256 threads, per SM
__global__ void __launch_bounds__(256, UPDATE_IN_PLACE_CTAS)
k_interior_update_in_place(int8_t *state, const float *index, int64_t n, bool vec) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (vec) {
        const int64_t nv = n / 16, lane = threadIdx.x & 31;
        bool many = false;                             // warp-uniform
        for (int64_t i0 = t0 - lane; i0 < nv; i0 += stride) {
            const int64_t i = i0 + lane;
            const bool in = i < nv;
            int4 sp = make_int4(0, 0, 0, 0);
            if (many && in) sp = __ldcs(reinterpret_cast<const int4 *>(state) + i);
            float4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = in ? __ldcs(reinterpret_cast<const float4 *>(index) + 4 * i + q) : make_float4(-1.f, -1.f, -1.f, -1.f);
            bool near = false;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                near |= !(v[q].x < -0.5f && v[q].y < -0.5f && v[q].z < -0.5f && v[q].w < -0.5f);
            const uint32_t nb = __ballot_sync(0xffffffffu, near);
            if (in && ((nb >> (lane & ~1)) & 3u)) {    // this lane's sector holds a near site
                if (!many) sp = __ldcs(reinterpret_cast<const int4 *>(state) + i);
                uint32_t w[4] = {(uint32_t)sp.x, (uint32_t)sp.y, (uint32_t)sp.z, (uint32_t)sp.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    w[q] = update_byte(w[q], 0, v[q].x);
                    w[q] = update_byte(w[q], 1, v[q].y);
                    w[q] = update_byte(w[q], 2, v[q].z);
                    w[q] = update_byte(w[q], 3, v[q].w);
                }
                __stcs(reinterpret_cast<int4 *>(state) + i, make_int4((int)w[0], (int)w[1], (int)w[2], (int)w[3]));
            }
            many = __popc((nb | (nb >> 1)) & 0x55555555u) >= 8;
        }
        done = nv * 16;
    }
    for (int64_t s = done + t0; s < n; s += stride) {
        const float v = index[s];
        if (!(v < -0.5f)) state[s] = (int8_t)(v < 0.0f ? 1 : 0);
    }
}

// Sparse form: the caller lists the near sites with their values.
__global__ void __launch_bounds__(256) k_interior_update_sites(int8_t *state, int64_t n, const int32_t *sites,
                                                                const float *values, int64_t m) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s = sites[i];
        const float v = values[i];
        if (s >= 0 && s < n && !(v < -0.5f)) state[s] = (int8_t)(v < 0.0f ? 1 : 0);
    }
}

static unsigned stream_grid(int64_t units, int per_sm = 8) {
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int64_t g = (units + 255) / 256;
    const int64_t cap = (int64_t)(nsm > 0 ? nsm : 1) * per_sm;
    if (g > cap) g = cap;
    return (unsigned)(g > 0 ? g : 1);
}

// In place, only the states near a membrane are moved where the two arrays (5 bytes a site)
// take more than four fifths of L2.  Below, both stay in L2 between steps and reading the
// states along with the index is as fast or faster (84 MB: 12.3 us, against 12.3 to 14.3 from
// none to all near; 105 MB: 17.6 against 14.4 to 17.9); above, it is not (115 MB: 19.5 against
// 16.3 to 18.6; 168 MB: 26.7 against 22.5 to 25.5; L2 holds 135 MB).
static bool update_in_place(int64_t n) {
    int dev = 0, l2 = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev);
    return 5 * n > (int64_t)l2 / 5 * 4;
}

cudaError_t launch_interior_update(const int8_t *prev, const float *index, int64_t n, int8_t *out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (prev == out && update_in_place(n)) {
        const bool vec = ((reinterpret_cast<uintptr_t>(index) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
        k_interior_update_in_place<<<stream_grid(vec ? n / 16 + 1 : n, UPDATE_IN_PLACE_CTAS), 256, 0, st>>>(out, index, n, vec);
        return cudaGetLastError();
    }
    const bool vec = ((reinterpret_cast<uintptr_t>(prev) | reinterpret_cast<uintptr_t>(index) |
                       reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    k_interior_update<<<stream_grid(vec ? n / 16 + 1 : n), 256, 0, st>>>(prev, index, n, out, vec);
    return cudaGetLastError();
}

cudaError_t launch_interior_update_sites(int8_t *state, int64_t n, const int32_t *sites, const float *values,
                                         int64_t m, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    k_interior_update_sites<<<stream_grid(m), 256, 0, st>>>(state, n, sites, values, m);
    return cudaGetLastError();
}

// Copy sized on the device: the host does not know the cluster count when it enqueues
// the copy of the sizes, so a grid-stride kernel reads it and copies that many (dst
// may be page-locked host memory, written across the host link).
__global__ void __launch_bounds__(256) k_copy_counted(const int64_t *src, const int64_t *count, int64_t cap,
                                                       int64_t *dst) {
    const int64_t n = min(*count, cap);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = __ldcs(src + i);
}

cudaError_t launch_copy_counted(const int64_t *src, const int64_t *count, int64_t cap, int64_t *dst,
                                cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int64_t g = (cap + 255) / 256;
    if (g > (int64_t)nsm * 8) g = (int64_t)nsm * 8;
    k_copy_counted<<<(unsigned)(g > 0 ? g : 1), 256, 0, st>>>(src, count, cap, dst);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------------------
// launch sequence
// --------------------------------------------------------------------------------------
// A kernel of the sequence, launched so that it may be set up while the previous kernel of
// the stream finishes (programmatic dependent launch; the kernel's grid_dep_wait()
// orders it after that kernel).  The first launch error of a sequence is kept in
// launch_error for launch_all to return.
static thread_local cudaError_t launch_error = cudaSuccess;
template <typename... KArgs, typename... Args>
static void launch_dep(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess && launch_error == cudaSuccess) launch_error = e;
}

template <typename K>
static int persistent_grid(K kernel, int threads, size_t smem, int64_t ntiles) {
    int dev = 0, nsm = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
    int64_t g = (int64_t)nsm * (per > 0 ? per : 1);
    if (g > ntiles) g = ntiles;
    return (int)(g > 0 ? g : 1);
}

template <int TY, int TZ, int NL>
static cudaError_t launch_all(const LatDev *lats, int n, const Plan &P, const Work &W, const PhiTmap *tms,
                              cudaStream_t st, cudaEvent_t *ev, MergeSchedule ms, int8_t *state) {
    using SH = TileShape<TY, TZ>;
    LatBatch<NL> B;
    B.n = n;
    B.pad_ = 0;
    for (int i = 0; i < n; ++i) B.lat[i] = lats[i];
    // tensor maps: the TMA occupancy pass needs every lattice's
    TmapBatch<NL> TB;
    std::memset(&TB, 0, sizeof(TB));
    bool all_tma = n > 0 && tms != nullptr;
    for (int i = 0; i < n; ++i) {
        if (tms) TB.tm[i] = tms[i];
        all_tma = all_tma && TB.tm[i].valid;
    }
    constexpr int CAP1 = LabelCfg<TY, TZ, true>::CAP, CAP1B = LabelCfg<TY, TZ, false>::CAP;
    constexpr int BL1 = LabelCfg<TY, TZ, true>::BL, BL1B = LabelCfg<TY, TZ, false>::BL;
    constexpr bool IX = NL == 1;   // the index-field passes take one lattice
    const bool index = IX && W.neg;
    const size_t smem1 = sizeof(LabelSmem<TY, TZ, CAP1, BL1, false>);
    const size_t smem1b = sizeof(LabelSmem<TY, TZ, CAP1B, BL1B, false>);
    const size_t smem1x = sizeof(LabelSmem<TY, TZ, LabelCfg<TY, TZ, true, IX>::CAP, BL1, IX>), smem1bx = sizeof(LabelSmem<TY, TZ, CAP1B, BL1B, IX>);
    const size_t smem4 = sizeof(FlatSmem<TY, TZ>);
    cudaError_t e;
    // Once per device a process uses: the shared-memory opt-ins (a device attribute of
    // each kernel) and the resident-CTA counts of the persistent passes.
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    static std::mutex init_mu;
    static int grid_cache[MAX_DEVICES][3];          // tile pass over dense tiles, flatten, TMA occupancy
    const size_t smem0 = sizeof(OccSmem<TY, TZ>);
    int grid1b, grid4, grid0;
    {
        std::lock_guard<std::mutex> init_lock(init_mu);
        int *c = grid_cache[dev];
        if (!c[1]) {
            e = cudaFuncSetAttribute(k_tile_label<TY, TZ, NL, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem1);
            if (e != cudaSuccess) return e;
            e = cudaFuncSetAttribute(k_tile_label<TY, TZ, NL, false, false>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1b);
            if (e != cudaSuccess) return e;
            if constexpr (IX) {
                e = cudaFuncSetAttribute(k_tile_label<TY, TZ, 1, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem1x);
                if (e != cudaSuccess) return e;
                e = cudaFuncSetAttribute(k_tile_label<TY, TZ, 1, false, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1bx);
                if (e != cudaSuccess) return e;
            }
            e = cudaFuncSetAttribute(k_flatten<TY, TZ, NL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem4);
            if (e != cudaSuccess) return e;
            if constexpr (NL == 1) {
                e = cudaFuncSetAttribute(k_flatten<TY, TZ, NL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem4);
                if (e != cudaSuccess) return e;
            }
            e = cudaFuncSetAttribute(k_occupancy_tma<TY, TZ, NL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem0);
            if (e != cudaSuccess) return e;
            if constexpr (IX) {
                e = cudaFuncSetAttribute(k_occupancy_tma<TY, TZ, NL, IX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem0);
                if (e != cudaSuccess) return e;
            }
            c[0] = persistent_grid(k_tile_label<TY, TZ, NL, false, IX>, SH::NT, smem1bx, INT32_MAX);
            c[2] = persistent_grid(k_occupancy_tma<TY, TZ, NL, IX>, 256, smem0, INT32_MAX);
            c[1] = persistent_grid(k_flatten<TY, TZ, NL, false>, SH::NT, smem4, INT32_MAX);
        }
        grid1b = c[0];
        grid4 = c[1];
        grid0 = c[2];
    }
    const unsigned g4 = (unsigned)(P.ntiles < grid4 ? P.ntiles : grid4);
    const uint32_t span4 = (uint32_t)((P.ntiles + (int64_t)grid4 * FLAT_ITEMS - 1) / ((int64_t)grid4 * FLAT_ITEMS));
    auto mark = [&](int i) { if (ev) cudaEventRecord(ev[i], st); };
    launch_error = cudaSuccess;
    mark(0);
    if (all_tma) {
        const unsigned g0 = (unsigned)(P.ntiles < grid0 ? P.ntiles : grid0);
        if (index) launch_dep(k_occupancy_tma<TY, TZ, NL, IX>, g0, 256, smem0, st, TB, B, W, P.ntiles);
        else launch_dep(k_occupancy_tma<TY, TZ, NL, false>, g0, 256, smem0, st, TB, B, W, P.ntiles);
    } else {
        launch_dep(k_occupancy<TY, TZ, NL>, (unsigned)((P.ntiles + 7) / 8), 256, 0, st, B, W, P.ntiles);
    }
    mark(1);
    // then the tiles handed on (none for fields with at most MR_FAST / R runs a row on average)
    const unsigned g1b = (unsigned)(P.ntiles < grid1b ? P.ntiles : grid1b);
    if (index) {
        launch_dep(k_tile_label<TY, TZ, NL, true, IX>, (unsigned)P.ntiles, SH::NT, smem1x, st, B, W, P.ntiles);
        launch_dep(k_tile_label<TY, TZ, NL, false, IX>, g1b, SH::NT, smem1bx, st, B, W, P.ntiles);
    } else {
        launch_dep(k_tile_label<TY, TZ, NL, true, false>, (unsigned)P.ntiles, SH::NT, smem1, st, B, W, P.ntiles);
        launch_dep(k_tile_label<TY, TZ, NL, false, false>, g1b, SH::NT, smem1b, st, B, W, P.ntiles);
    }
    mark(2);
    const unsigned gfm = (unsigned)((P.ntiles + FM_WARPS - 1) / FM_WARPS);
    if (ms.unions == 1) launch_dep(k_face_merge<TY, TZ, NL, 1>, gfm, 32 * FM_WARPS, 0, st, B, W, P.ntiles);
    else if (ms.unions == 4) launch_dep(k_face_merge<TY, TZ, NL, 4>, gfm, 32 * FM_WARPS, 0, st, B, W, P.ntiles);
    else launch_dep(k_face_merge<TY, TZ, NL, 2>, gfm, 32 * FM_WARPS, 0, st, B, W, P.ntiles);
    mark(3);
    const unsigned gpf = (unsigned)((P.ntiles + PF_WARPS - 1) / PF_WARPS);
    if (ms.hot) launch_dep(k_piece_finalize<NL, true>, gpf, 32 * PF_WARPS, 0, st, B, W, P.ntiles);
    else launch_dep(k_piece_finalize<NL, false>, gpf, 32 * PF_WARPS, 0, st, B, W, P.ntiles);
    mark(4);
    if constexpr (IX) {
        if (state) {                               // index fields: the state is all that is wanted
            mark(5);
            mark(6);
            const bool vec = (lats[0].nx & 15) == 0 && (reinterpret_cast<uintptr_t>(state) & 15) == 0;
            launch_dep(k_state<TY, TZ>, (unsigned)P.ntiles, SH::NT, 0, st, lats[0], W, state, vec);
            mark(7);
            return launch_error != cudaSuccess ? launch_error : cudaGetLastError();
        }
    }
    const int64_t nb = (P.nrows + SCAN_CH) / SCAN_CH;   // covers index nrows (the total)
    const bool scanned = nb > SCAN_DIRECT;
    launch_dep(k_scan_reduce<NL>, (unsigned)nb, SCAN_NT, 0, st, B, (const uint8_t *)W.cnt, P.nrows, W.bsum);
    if (scanned) launch_dep(k_scan_blocks, 1u, 1024u, 0, st, W.bsum, nb);
    launch_dep(k_scan_apply<NL>, (unsigned)nb, SCAN_NT, 0, st, B, (const uint8_t *)W.cnt, P.nrows,
               (const uint32_t *)W.bsum, W.pre, scanned);
    mark(5);
    mark(6);
    if constexpr (NL == 1) {
        if (W.roots || W.site_off) launch_dep(k_flatten<TY, TZ, NL, true>, g4, SH::NT, smem4, st, B, W, P.ntiles, span4);
        else launch_dep(k_flatten<TY, TZ, NL, false>, g4, SH::NT, smem4, st, B, W, P.ntiles, span4);
    } else {
        launch_dep(k_flatten<TY, TZ, NL, false>, g4, SH::NT, smem4, st, B, W, P.ntiles, span4);
    }
    mark(7);
    if (launch_error != cudaSuccess) return launch_error;
    return cudaGetLastError();
}

template <int TY, int TZ>
static cudaError_t launch_shape(const LatDev *lats, int n, const Plan &P, const Work &W, const PhiTmap *tms,
                                cudaStream_t st, cudaEvent_t *ev, MergeSchedule ms, int8_t *state) {
    if (n == 1) return launch_all<TY, TZ, 1>(lats, n, P, W, tms, st, ev, ms, state);
    return launch_all<TY, TZ, MAX_LAT_PER_LAUNCH>(lats, n, P, W, tms, st, ev, ms, nullptr);
}

template <int TY, int TZ>
static void shape_info(TileInfo &ti) {
    using SH = TileShape<TY, TZ>;
    ti.ty = TY;
    ti.tz = TZ;
    ti.rows = SH::R;
    ti.maxruns = SH::MAXRUNS;
    ti.face_stride = SH::FACE_STRIDE;
    ti.max_boundary = SH::MAX_BOUNDARY;
}

bool tile_info(int ty, int tz, TileInfo &ti) {
    if (ty == 8 && tz == 8) { shape_info<8, 8>(ti); return true; }
    if (ty == 16 && tz == 8) { shape_info<16, 8>(ti); return true; }
    if (ty == 16 && tz == 16) { shape_info<16, 16>(ti); return true; }
    if (ty == 32 && tz == 8) { shape_info<32, 8>(ti); return true; }
    return false;
}

cudaError_t launch_label(int ty, int tz, const LatDev *lats, int n, const Plan &P, const Work &W, const PhiTmap *tms,
                         cudaStream_t st, cudaEvent_t *ev, MergeSchedule ms, int8_t *state) {
    if (ty == 8 && tz == 8) return launch_shape<8, 8>(lats, n, P, W, tms, st, ev, ms, state);
    if (ty == 16 && tz == 8) return launch_shape<16, 8>(lats, n, P, W, tms, st, ev, ms, state);
    if (ty == 16 && tz == 16) return launch_shape<16, 16>(lats, n, P, W, tms, st, ev, ms, state);
    if (ty == 32 && tz == 8) return launch_shape<32, 8>(lats, n, P, W, tms, st, ev, ms, state);
    return cudaErrorInvalidValue;
}

}  // namespace hk
