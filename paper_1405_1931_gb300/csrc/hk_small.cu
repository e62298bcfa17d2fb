// hk_small.cu -- one launch for small lattices: one CTA labels a whole lattice of at
// most SMALL_MAX_SITES sites in shared memory (a batch of such lattices: one CTA each).
//
// The tiled passes of hk_kernels.cu need eight launches per call, whose gaps are
// the whole cost of a 32^3 lattice.  Here every step runs in one kernel, separated by
// barriers instead of launches:
//   a1  occupancy phi > 0 (Sec. 2) as one 32-bit word per row segment (32 sites along x);
//   a2  x-runs numbered in row-major order, union-find over them in shared memory with
//       union by minimum run id (Sec. 2's rules 1-3 applied to runs);
//   a3  the unions along x between segments, along y and z, and across every periodic
//       edge (Sec. 3, halo paragraph and Fig. 2 caption);
//   a4  the clusters' ranks: a scan of the root flags in run order, which is label order
//       (Sec. 2, final paragraph);
//   a5  labels: the smallest site of the cluster, -1 for the medium;
//   a6  sizes in label order (Sec. 5), a7 the floor(log2 size) histogram.
// Runs are numbered in row-major order of their first sites, so each cluster's root
// (its smallest run id) holds its smallest site, and ranking roots by run id ranks the
// clusters by label.  No workspace is used: the results go straight to the outputs.
//
// Latency bounds a call (barriers, chains of dependent shared loads, and the code fetched).
// With links for the first pairs, ranks from root bits and one scan for two segments a
// thread, one CTA takes 24.1 us for 32^3 at p = 0.3 (36.9 with every pair united by its
// segment's thread and ranks by blocks of run ids), a batch of 32 such lattices 25 us (89).
#include <cooperative_groups.h>

#include <cstddef>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "hk_device.cuh"
#include "hk_launch.h"

namespace hk {

namespace {

constexpr int SNT = 1024;   // threads of the one CTA per lattice

struct SmallSmem {
    uint32_t m[SMALL_MAX_SEG];         // occupancy word of each row segment (row-major)
    uint16_t sb[SMALL_MAX_SEG];        // first run id of each segment
    int par[SMALL_MAX_RUNS];           // union-find over run ids; after compression: the root
    int sz[SMALL_MAX_RUNS];            // piece size, summed at each root
    uint16_t desc[SMALL_MAX_RUNS];     // per run: (segment << 5) | first x
    uint32_t rootbal[SMALL_MAX_RUNS / 32];   // cluster-root bits of each 32 run ids
    uint16_t rootpre[SMALL_MAX_RUNS / 32];   // roots before them
    int warp_tmp[32];
    int scan_total;
    int hist[32];
};
static_assert(SMALL_MAX_RUNS % 32 == 0 && SMALL_MAX_RUNS / 32 <= SNT, "one thread scans one word of root bits");
static_assert(SMALL_MAX_SEG <= 2 * SNT, "two segments a thread");
static_assert(SMALL_MAX_SEG <= 2048 && SMALL_MAX_RUNS <= 65535, "desc holds an 11-bit segment, sb a 16-bit run id");
static_assert(sizeof(SmallSmem) <= 227 * 1024, "one CTA's shared memory");

// Division by a lattice constant d >= 1 by one multiply: floor(x / d) =
// (x * ceil(2^32 / d)) >> 32, exact while x * d < 2^32 (here x < 2^16 and d <= 2^15).
struct FastDiv {
    uint64_t m;
    __device__ explicit FastDiv(uint32_t d) : m(((1ull << 32) + d - 1) / d) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const { return (uint32_t)((x * m) >> 32); }
};

// Links make chains: of stripes across x a run hangs on the row below it, that one on the
// next, as many as there are rows.  From CHAIN links on each run is first pointed at what its
// parent points at, once a halving of the longest possible chain (an ancestor, so it does not
// matter which of two such stores a read meets).
constexpr int CHAIN = 24;
template <int NT>
__device__ __forceinline__ void shorten_chains(int *par, int total, int longest) {
    for (; longest > CHAIN; longest >>= 1) {
        for (int i = threadIdx.x; i < total; i += NT) par[i] = par[par[i]];
        __syncthreads();
    }
}

// the run of segment s (first run id b, occupancy word w) holding bit x
__device__ __forceinline__ int srun(int b, uint32_t w, int x) { return b + __popc(run_starts(w) & le_mask(x)) - 1; }

// Exclusive scan of one int per thread over the CTA's NT threads (NT a multiple of 32,
// at most 1024); *total gets the sum.  Ends with a barrier, after which warp_tmp and
// scan_total may be reused.
template <int NT, class SM>
__device__ __forceinline__ int cta_exscan(int v, SM &S, int &total) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += u;
    }
    if (lane == 31) S.warp_tmp[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const int w = lane < NW ? S.warp_tmp[lane] : 0;
        int wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += u;
        }
        if (lane < NW) S.warp_tmp[lane] = wi - w;
        if (lane == 31) S.scan_total = wi;
    }
    __syncthreads();
    const int r = S.warp_tmp[wid] + inc - v;
    total = S.scan_total;
    __syncthreads();
    return r;
}

template <int NL>
__global__ void __launch_bounds__(SNT, 1) k_small_label(const __grid_constant__ LatBatch<NL> B, int32_t *status,
                                                         int32_t local_cap) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem &S = *reinterpret_cast<SmallSmem *>(smem_raw);
    const LatDev &L = B.lat[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NW = SNT / 32;
    const int nx = L.nx, ny = L.ny, nz = L.nz, nbx = L.nbx;
    const int nseg = nbx * ny * nz;
    const bool flat = (nx & 31) == 0;   // segment s is sites 32 s .. 32 s + 31 of the lattice
    const FastDiv div_nbx((uint32_t)nbx), div_ny((uint32_t)ny);
    if (tid < 32) S.hist[tid] = 0;

    // a1: occupancy words; each warp keeps up to 32 segments' loads in flight (a 32^3
    // lattice in one round trip)
    constexpr int INF = 32;
    auto read_words = [&](auto FLAT) {
        for (int s0 = wid; s0 < nseg; s0 += NW * INF) {
            float v[INF];
#pragma unroll
            for (int j = 0; j < INF; ++j) {
                const int s = s0 + NW * j;
                if (decltype(FLAT)::value) {
                    v[j] = s < nseg ? __ldg(L.phi + 32 * s + lane) : 0.0f;
                } else {
                    const int q = (int)div_nbx((uint32_t)s), x = (s - q * nbx) * 32 + lane;
                    v[j] = (s < nseg && x < nx) ? __ldg(L.phi + (int64_t)q * nx + x) : 0.0f;
                }
            }
#pragma unroll
            for (int j = 0; j < INF; ++j) {
                const uint32_t w = __ballot_sync(0xffffffffu, occupied(v[j], L.occ_mode));
                if (lane == 0 && s0 + NW * j < nseg) S.m[s0 + NW * j] = w;
            }
        }
    };
    if (flat) read_words(std::true_type{});
    else read_words(std::false_type{});
    __syncthreads();

    // a2: run ids: one scan of the run counts of segments t (low half) and t + SNT
    const uint32_t w_a = tid < nseg ? S.m[tid] : 0u, w_b = tid + SNT < nseg ? S.m[tid + SNT] : 0u;
    const int n_a = __popc(run_starts(w_a)), n_b = __popc(run_starts(w_b));
    int packed_total;
    const int packed = cta_exscan<SNT>(n_a | (n_b << 16), S, packed_total);
    const int total = (packed_total & 0xffff) + (packed_total >> 16);
    auto first_run = [&](int h) { return h ? (packed_total & 0xffff) + (packed >> 16) : packed & 0xffff; };
    for (int h = 0; h < 2; ++h) {   // own node and descriptor of every run
        const int s = tid + h * SNT;
        if (s >= nseg) break;
        int id = first_run(h);
        S.sb[s] = (uint16_t)id;
        for (uint32_t w = run_starts(h ? w_b : w_a); w; ++id) {
            const uint32_t low = w & (0u - w);
            w ^= low;
            S.par[id] = id;
            S.sz[id] = 0;
            S.desc[id] = (uint16_t)((s << 5) | top_bit(low));
        }
    }
    __syncthreads();

    // a3: unions with the lower neighbours along x (previous segment), y and z, and
    // across the periodic edges (the wrap of an axis of length 1 is a self-edge; one of
    // length 2 repeats an interior edge).  As in the tile pass, a run's first pair with a
    // lower row is a store into its own node, and a z pair whose site is joined through
    // its y neighbours is left out; the others are united after a barrier.
    uint32_t rest_y[2] = {0u, 0u}, rest_z[2] = {0u, 0u};
    for (int h = 0; h < 2; ++h) {
        const int s = tid + h * SNT;
        const uint32_t w = h ? w_b : w_a;
        if (s >= nseg || !w) continue;
        const int q = (int)div_nbx((uint32_t)s), z = (int)div_ny((uint32_t)q), y = q - z * ny;
        const int sy = s - nbx, sz = s - nbx * ny;
        const uint32_t my = y > 0 ? S.m[sy] : 0u, mz = z > 0 ? S.m[sz] : 0u;
        const uint32_t oy = w & my, oz = w & mz, uy = fill_up(w, oy);
        const uint32_t osy = run_starts(oy), osz = run_starts(oz), rs = run_starts(w);
        const uint32_t ylink = osy & ~(uy << 1);
        const uint32_t zlink = osz & ~(fill_up(w, oz) << 1) & ~(uy | fill_down(w, oy));
        rest_y[h] = osy ^ ylink;
        rest_z[h] = osz & ~zlink;
        if (y > 0 && z > 0) rest_z[h] &= ~(my & S.m[sz - nbx]);
        const int b = first_run(h), by = y > 0 ? S.sb[sy] : 0, bz = z > 0 ? S.sb[sz] : 0;
        const uint32_t rsy = run_starts(my), rsz = run_starts(mz);
        for (uint32_t link = ylink | zlink; link;) {
            const uint32_t low = link & (0u - link), le = low | (low - 1u);
            link ^= low;
            const bool iy = (my & low) != 0u;
            S.par[b + __popc(rs & le) - 1] = (iy ? by : bz) + __popc((iy ? rsy : rsz) & le) - 1;
        }
    }
    __syncthreads();
    shorten_chains<SNT>(S.par, total, min(ny + nz, total));
    const int cap = (local_cap > 0 && local_cap < total) ? local_cap : total;
    // (each kind of pair has one loop around one union: the kernel runs once through its code,
    // and fetching that counts: 17.4 us for 8 lattices of 16^3, 18.0 with two loops for each)
    const int lastbit = (nx - 1) & 31;   // bit of x = nx - 1 in the last segment of a row
    for (int h = 0; h < 2; ++h) {
        const int s = tid + h * SNT;
        const uint32_t w = h ? w_b : w_a;
        if (s >= nseg || !w) continue;
        const int b = first_run(h);
#pragma unroll 1
        for (int d = 0; d < 2; ++d) {                // the pairs with the lower rows along z and y
            uint32_t os = d ? rest_y[h] : rest_z[h];
            if (!os) continue;
            const int t = d ? s - nbx : s - nbx * ny, bt = S.sb[t];
            const uint32_t wt = S.m[t];
            for (; os; os &= os - 1u) {
                const int x = top_bit(os & (0u - os));
                s_union(S.par, srun(b, w, x), srun(bt, wt, x), cap, status);
            }
        }
        if (w & 1u) {                                // along x: the segment before, or the periodic edge
            const int bx = s - (int)div_nbx((uint32_t)s) * nbx, t = bx > 0 ? s - 1 : s + nbx - 1, x = bx > 0 ? 31 : lastbit;
            if ((bx > 0 || (L.per[0] && nx >= 2)) && ((S.m[t] >> x) & 1u))
                s_union(S.par, b, srun(S.sb[t], S.m[t], x), cap, status);
        }
    }
    // The periodic edges along y and z.  A find from the far side climbs a row's links, one
    // for every row of stripes across x, so the pairs of a segment are shared out by nibbles
    // over the warps.
    {
        const int wrap_y = L.per[1] && ny >= 2 ? nbx * nz : 0, wraps = wrap_y + (L.per[2] && nz >= 2 ? nbx * ny : 0);
        const int shares = nx > 16 ? 3 : nx > 8 ? 2 : nx > 4 ? 1 : 0;   // log2; a word has pairs at its first nx bits only
        const uint32_t part = shares ? 0xfu << (4 * (wid & ((1 << shares) - 1))) : ~0u;
        for (int j = (wid >> shares) * 32 + lane; j < wraps; j += (NW >> shares) * 32) {
            const int z = (int)div_nbx((uint32_t)j), s = j < wrap_y ? z * ny * nbx + j - z * nbx : j - wrap_y;
            const int t = s + (j < wrap_y ? (ny - 1) * nbx : (nz - 1) * nbx * ny), b = S.sb[s], bt = S.sb[t];
            const uint32_t w = S.m[s], wt = S.m[t];
            for (uint32_t os = run_starts(w & wt) & part; os; os &= os - 1u) {
                const int x = top_bit(os & (0u - os));
                s_union(S.par, srun(b, w, x), srun(bt, wt, x), cap, status);
            }
        }
    }
    __syncthreads();

    // compression (two levels a step), piece sizes, and the root bits of the run ids
    for (int i0 = wid * 32; i0 < total; i0 += SNT) {
        const int i = i0 + lane;
        bool is_root = false;
        if (i < total) {
            int root = S.par[i];
            for (int up = S.par[root]; up != root; up = S.par[root]) root = S.par[up];
            S.par[i] = root;
            const int d = S.desc[i];
            atomicAdd(&S.sz[root], run_len(S.m[d >> 5], d & 31));
            is_root = root == i;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, is_root);
        if (lane == 0) S.rootbal[i0 >> 5] = bal;
    }
    __syncthreads();

    // a4, a6, a7: the roots in run order get consecutive ranks (a scan of the words of
    // root bits), and sizes leave in that order
    const int nchunks = (total + 31) >> 5;
    int nclus;
    const int before = cta_exscan<SNT>(tid < nchunks ? __popc(S.rootbal[tid]) : 0, S, nclus);
    if (tid < nchunks) S.rootpre[tid] = (uint16_t)before;
    __syncthreads();
    const int64_t capr = L.sizes_cap;
    for (int i0 = wid * 32; i0 < total; i0 += SNT) {
        const uint32_t bal = S.rootbal[i0 >> 5];
        if (!((bal >> lane) & 1u)) continue;
        const int i = i0 + lane, rank = S.rootpre[i0 >> 5] + __popc(bal & ((1u << lane) - 1u));
        const int size = S.sz[i];
        if (rank < capr) L.sizes[rank] = size;
        atomicAdd(&S.hist[top_bit((uint32_t)size)], 1);
        const int d = S.desc[i], rs_ = d >> 5, rq = (int)div_nbx((uint32_t)rs_);
        S.sz[i] = rq * nx + (rs_ - rq * nbx) * 32 + (d & 31);   // from here on: the root's site (its label)
    }
    __syncthreads();

    // a5: labels, one warp per segment, one lane per site
    auto write_labels = [&](auto FLAT) {
#pragma unroll 4
        for (int s = wid; s < nseg; s += NW) {
            const uint32_t w = S.m[s];
            const int lab = ((w >> lane) & 1u) ? S.sz[S.par[srun(S.sb[s], w, lane)]] : -1;
            if (decltype(FLAT)::value) {
                L.labels[32 * s + lane] = lab;
            } else {
                const int q = (int)div_nbx((uint32_t)s), x = (s - q * nbx) * 32 + lane;
                if (x < nx) L.labels[(int64_t)q * nx + x] = lab;
            }
        }
    };
    if (flat) write_labels(std::true_type{});
    else write_labels(std::false_type{});
    __syncthreads();
    if (tid < 32 && L.hist) L.hist[tid] = S.hist[tid];
    if (tid == 0 && L.ncl) L.ncl[0] = nclus;
}

// ---------------------------------------------------------------------------------------
// The same steps on a thread-block cluster: CS CTAs on CS SMs label one lattice, each
// holding the rows [c RP, (c + 1) RP) of the lattice (RP = ceil(ny nz / CS)) in its own
// shared memory, so that the loads, unions, ranks and label stores are spread over CS
// SMs.  A run of CTA c is numbered (c << CRUN_BITS) | its local id: numbers grow with
// the runs' first sites in row-major order, so union by minimum number still makes each
// cluster's root its first run.  Each CTA first joins the edges inside it on local ids;
// the edges to other CTAs are then joined between local roots, through distributed
// shared memory (the other CTAs' parents, occupancy words and run bases); every local
// root then learns its cluster root, so each run reaches its root in two steps, and
// each run's label is resolved once per run, not per site.  The phases that reach other
// CTAs are separated by cluster barriers.
//
// Latency bounds a call here too.  A 32^3 lattice gives a CTA 64 segments, so the pairs
// inside a CTA that links do not take are shared out by nibbles of a segment: 20.5 us at
// p = 0.3 and 0.45 (24.5 and 24.6 with all pairs counted, listed and united; 22.9 and 26.7
// with one thread a segment).
// ---------------------------------------------------------------------------------------
// CTAs per lattice: 16 where the device co-schedules that many (a non-portable cluster
// size), else 8 (the portable size); a template parameter of the kernel (CSB = log2).
constexpr int CNT = 1024;          // threads per CTA
constexpr int CSEG = 1024;         // row segments per CTA
constexpr int CRUN_BITS = 14;
constexpr int CRUN = 1 << CRUN_BITS;   // runs per CTA: at most 16 per segment
constexpr int DESC_LROOT = 0x8000;     // desc flag: the run is the root of its CTA-local tree
static_assert(16 * CSEG <= CRUN && CSEG <= CNT, "run ids of a CTA; one segment per thread in the union rounds");

struct ClusterSmem {
    uint32_t m[CSEG];        // occupancy word of each of this CTA's row segments
    uint16_t sb[CSEG];       // first local run id of each segment
    int par[CRUN];           // union-find over cluster run numbers; after compression: the root
    int sz[CRUN];            // piece size, summed at each root; after ranking: the root's site
    uint16_t desc[CRUN];     // per run: (local segment << 5) | first x, and DESC_LROOT
    int roots;               // cluster roots among this CTA's runs
    uint64_t bar;            // completion of the bulk copy of this CTA's rows of phi
    int warp_tmp[32];
    int scan_total;
    int hist[32];
};
static_assert(sizeof(ClusterSmem) <= 227 * 1024, "one CTA's shared memory");
static_assert(offsetof(ClusterSmem, sz) == offsetof(ClusterSmem, par) + sizeof(int) * CRUN &&
                  sizeof(int) * 2 * CRUN >= sizeof(float) * TX * CSEG,
              "par and sz together hold a CTA's rows of phi");

namespace cg = cooperative_groups;

struct ClusterView {
    ClusterSmem &S;
    cg::cluster_group cl;
    int c;
    // parent of run number g, wherever it lives
    __device__ __forceinline__ int *par(int g) const {
        int *p = &S.par[g & (CRUN - 1)];
        const int o = g >> CRUN_BITS;
        return o == c ? p : cl.map_shared_rank(p, o);
    }
    __device__ __forceinline__ int *sz(int g) const {
        int *p = &S.sz[g & (CRUN - 1)];
        const int o = g >> CRUN_BITS;
        return o == c ? p : cl.map_shared_rank(p, o);
    }
    // find with path halving (every store lowers a parent to an ancestor)
    __device__ int find(int x) const {
        int p = *par(x);
        while (p != x) {
            const int gp = *par(p);
            if (gp == p) return p;
            *par(x) = gp;
            x = gp;
            p = *par(x);
        }
        return x;
    }
    __device__ int find_ro(int x) const {
        int p = *par(x);
        while (p != x) {
            x = p;
            p = *par(x);
        }
        return x;
    }
    // each retry strictly lowers max(a, b): at most `cap` rounds
    __device__ void unite(int a, int b, int cap, int32_t *status) const {
        for (int it = 0; it <= cap; ++it) {
            a = find(a);
            b = find(b);
            if (a == b) return;
            const int hi = a > b ? a : b, lo = a > b ? b : a;
            const int old = atomicMin(par(hi), lo);
            if (old == hi) return;
            a = lo;
            b = old;
        }
        atomicOr(status, STATUS_LOCAL_LOOP);
    }
};

template <int CSB, int NL>
__global__ void __cluster_dims__(1 << CSB, 1, 1) __launch_bounds__(CNT, 1)
    k_small_cluster(const __grid_constant__ LatBatch<NL> B, int32_t *status, int32_t local_cap) {
    constexpr int CS_BITS = CSB, CS = 1 << CSB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ClusterSmem &S = *reinterpret_cast<ClusterSmem *>(smem_raw);
    cg::cluster_group cl = cg::this_cluster();
    const int c = (int)cl.block_rank();
    const ClusterView V{S, cl, c};
    const LatDev &L = B.lat[blockIdx.x / CS];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr int NW = CNT / 32;
    const int nx = L.nx, ny = L.ny, nz = L.nz, nbx = L.nbx;
    const int nrows = ny * nz, rp = (nrows + CS - 1) / CS;       // rows per CTA
    const int q0 = min(c * rp, nrows), q1 = min(q0 + rp, nrows);
    const int seg0 = q0 * nbx, nseg = (q1 - q0) * nbx;           // this CTA's segments
    const FastDiv div_nbx((uint32_t)nbx), div_ny((uint32_t)ny), div_rp((uint32_t)rp);
    const int cbase = c << CRUN_BITS;
    if (tid < 32) S.hist[tid] = 0;

    // a1: occupancy words of this CTA's segments.  Its rows of phi are one contiguous
    // range: one bulk copy lands it in par and sz (not in use yet) when it is 16-byte
    // aligned, and each warp turns landed segments into words by ballots; otherwise (or
    // if the copy does not complete within its bound) 32 loads in flight per warp.
    bool landed = false;
    {
        const float *src = L.phi + (int64_t)q0 * nx;
        const int nfl = (q1 - q0) * nx;
        if (nfl > 0 && (nfl & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {   // uniform
            const float *land = reinterpret_cast<const float *>(S.par);
            if (tid == 0) {
                mbar_init(&S.bar, 1);
                fence_mbar_init();
            }
            __syncthreads();
            if (tid == 0) {
                mbar_arrive_expect_tx(&S.bar, (uint32_t)nfl * 4u);
                bulk_load(S.par, src, (uint32_t)nfl * 4u, &S.bar);
            }
            landed = mbar_wait_bounded(&S.bar, 0);
            if (__syncthreads_or(!landed)) {
                if (tid == 0) atomicOr(status, STATUS_TMA_TIMEOUT);
                mbar_wait_bounded(&S.bar, 0);   // the copy still in flight
                landed = false;
            } else {
                landed = true;
                for (int ls = wid; ls < nseg; ls += NW) {
                    const int r = (int)div_nbx((uint32_t)ls), x = (ls - r * nbx) * 32 + lane;
                    const float v = x < nx ? land[r * nx + x] : 0.0f;
                    const uint32_t w = __ballot_sync(0xffffffffu, occupied(v, L.occ_mode));
                    if (lane == 0) S.m[ls] = w;
                }
            }
        }
    }
    constexpr int INF = 32;
    for (int l0 = landed ? nseg : wid; l0 < nseg; l0 += NW * INF) {
        float v[INF];
#pragma unroll
        for (int j = 0; j < INF; ++j) {
            const int ls = l0 + NW * j, sg = seg0 + ls;
            const int q = (int)div_nbx((uint32_t)sg), x = (sg - q * nbx) * 32 + lane;
            v[j] = (ls < nseg && x < nx) ? __ldg(L.phi + (int64_t)q * nx + x) : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < INF; ++j) {
            const uint32_t w = __ballot_sync(0xffffffffu, occupied(v[j], L.occ_mode));
            if (lane == 0 && l0 + NW * j < nseg) S.m[l0 + NW * j] = w;
        }
    }
    __syncthreads();

    // a2: local run ids (segments 2t and 2t + 1 of thread t), nodes and descriptors
    const int s_a = 2 * tid, s_b = 2 * tid + 1;
    const int n_a = s_a < nseg ? __popc(run_starts(S.m[s_a])) : 0;
    const int n_b = s_b < nseg ? __popc(run_starts(S.m[s_b])) : 0;
    int total;
    const int base = cta_exscan<CNT>(n_a + n_b, S, total);
    if (s_a < nseg) S.sb[s_a] = (uint16_t)base;
    if (s_b < nseg) S.sb[s_b] = (uint16_t)(base + n_a);
    for (int h = 0; h < 2; ++h) {
        const int ls = 2 * tid + h;
        if (ls >= nseg) break;
        uint32_t w = run_starts(S.m[ls]);
        int id = base + (h ? n_a : 0);
        while (w) {
            const int x0 = __ffs(w) - 1;
            w &= w - 1;
            S.par[id] = id;   // local ids until the edges inside this CTA are joined
            S.desc[id] = (uint16_t)((ls << 5) | x0);
            ++id;
        }
    }
    __syncthreads();

    // a3: unions with the lower neighbours along x, y and z and across the periodic
    // edges, in two rounds.  First the edges inside this CTA, on local run ids in its own
    // shared memory; then, once every CTA has compressed its runs onto their local roots,
    // the edges to runs of other CTAs, joined between local roots through distributed
    // shared memory.  The second round lists its run pairs first (a scan of per-segment
    // counts; sz serves as the list), so that the unions spread over all threads; where
    // the list would not fit each segment's pairs are joined as they are found.
    const int lastbit = (nx - 1) & 31;
    auto neighbours = [&](int ls, auto &&edge) {   // edge(global segment t) for every lower neighbour
        const int sg = seg0 + ls;
        const int q = (int)div_nbx((uint32_t)sg), z = (int)div_ny((uint32_t)q), y = q - z * ny;
        if (y > 0) edge(sg - nbx);
        else if (L.per[1] && ny >= 2) edge(sg + (ny - 1) * nbx);
        if (z > 0) edge(sg - nbx * ny);
        else if (L.per[2] && nz >= 2) edge(sg + (nz - 1) * nbx * ny);
    };
    auto owner = [&](int t, int &lt) {   // the CTA holding global segment t, and its local index there
        const int tq = (int)div_nbx((uint32_t)t), o = (int)div_rp((uint32_t)tq);
        lt = t - o * rp * nbx;
        return o;
    };
    // every pair of runs joined by an edge of segment ls to another CTA: pair(own local run,
    // CTA, its run)
    auto pairs = [&](int ls, auto &&pair) {
        const uint32_t w = S.m[ls];
        if (!w) return;
        const int b = S.sb[ls];
        neighbours(ls, [&](int t) {
            int lt;
            const int o = owner(t, lt);
            if (o == c) return;
            const uint32_t wt = *cl.map_shared_rank(&S.m[lt], o);
            uint32_t os = run_starts(w & wt);
            if (!os) return;
            const int bt = *cl.map_shared_rank(&S.sb[lt], o);
            while (os) {
                const int x = __ffs(os) - 1;
                os &= os - 1;
                pair(srun(b, w, x), o, srun(bt, wt, x));
            }
        });
    };
    // count, list and join them, one segment a thread
    auto join_cross = [&](auto &&join) {
        int np = 0;
        if (tid < nseg) pairs(tid, [&](int, int, int) { ++np; });
        int npairs;
        int j = cta_exscan<CNT>(np, S, npairs);
        if (npairs <= CRUN) {
            if (tid < nseg)
                pairs(tid, [&](int a, int o, int bb) {
                    S.sz[j++] = (int)(((uint32_t)a << (CRUN_BITS + CS_BITS)) | ((uint32_t)o << CRUN_BITS) |
                                      (uint32_t)bb);
                });
            __syncthreads();
            for (int k = tid; k < npairs; k += CNT) {
                const uint32_t u = (uint32_t)S.sz[k];
                join((int)(u >> (CRUN_BITS + CS_BITS)), (int)((u >> CRUN_BITS) & (CS - 1)), (int)(u & (CRUN - 1)));
            }
        } else if (tid < nseg) {
            pairs(tid, join);
        }
    };
    static_assert(2 * CRUN_BITS + CS_BITS <= 32 && CS <= 32, "a listed pair packs into 32 bits");
    if (total > 0) {                                 // CTA-uniform
        const int lcap = (local_cap > 0 && local_cap < total) ? local_cap : total;
        // the edges inside the CTA, one segment a thread: as in the tile pass a run's first
        // pair with a lower row is a store into its own node and a z pair whose site is
        // joined through its y neighbours is left out; the others follow after a
        // barrier, and with them those of the periodic edges along y and z (a segment has
        // those in place of its pairs with a lower row): 16 shares a segment (a nibble of its
        // z or y pairs) over as many threads as there are, since a find may climb a chain of
        // links as long as the lattice is wide (stripes across x)
        // (from half as many segments as threads on: all listed by a scan and taken in turn,
        // 51 against 54 us at 64 x 96 x 80, p_c)
        const int row = nbx * ny;
        uint32_t osy = 0, osz = 0;
        auto below = [&](int ls, bool z_) {          // the segment of ls's y or z pairs
            const int q = (int)div_nbx((uint32_t)(seg0 + ls)), z = (int)div_ny((uint32_t)q);
            if (z_) return z > 0 ? ls - row : ls + (nz - 1) * row;
            return q > z * ny ? ls - nbx : ls + (ny - 1) * nbx;
        };
        if (tid < nseg) {
            const int ls = tid, q = (int)div_nbx((uint32_t)(seg0 + ls)), z = (int)div_ny((uint32_t)q), y = q - z * ny;
            const int wy = ls + (ny - 1) * nbx, wz = ls + (nz - 1) * row;
            const uint32_t w = S.m[ls];
            const uint32_t my = y > 0 && ls >= nbx ? S.m[ls - nbx] : 0u, mz = z > 0 && ls >= row ? S.m[ls - row] : 0u;
            const uint32_t oy = w & my, oz = w & mz, uy = fill_up(w, oy), rs = run_starts(w);
            osy = run_starts(oy);
            osz = run_starts(oz);
            const uint32_t ylink = osy & ~(uy << 1);
            const uint32_t zlink = osz & ~(fill_up(w, oz) << 1) & ~(uy | fill_down(w, oy));
            osy ^= ylink;
            osz &= ~zlink;
            if (my && mz && ls >= row + nbx) osz &= ~(my & S.m[ls - row - nbx]);
            const uint32_t rsy = run_starts(my), rsz = run_starts(mz);
            const int b = S.sb[ls], by = my ? S.sb[ls - nbx] : 0, bz = mz ? S.sb[ls - row] : 0;
            for (uint32_t link = ylink | zlink; link;) {
                const uint32_t low = link & (0u - link), le = low | (low - 1u);
                link ^= low;
                const bool iy = (my & low) != 0u;
                S.par[b + __popc(rs & le) - 1] = (iy ? by : bz) + __popc((iy ? rsy : rsz) & le) - 1;
            }
            if (y == 0 && L.per[1] && ny >= 2 && wy < nseg) osy = run_starts(w & S.m[wy]);
            if (z == 0 && L.per[2] && nz >= 2 && wz < nseg) osz = run_starts(w & S.m[wz]);
        }
        const int longest = min(ny, rp) + rp / ny;   // links of a chain: y goes down, then z
        if (longest > CHAIN) {
            __syncthreads();
            shorten_chains<CNT>(S.par, total, min(longest, total));
        }
        bool listed = false;                         // CTA-uniform
        if (2 * nseg >= CNT) {
            int npairs;
            int j = cta_exscan<CNT>(__popc(osz) + __popc(osy), S, npairs);   // ends with a barrier: links are done
            listed = npairs <= CRUN;
            if (listed) {
                auto list = [&](int t, uint32_t os) {
                    const uint32_t w = S.m[tid], wt = S.m[t];
                    const int b = S.sb[tid], bt = S.sb[t];
                    for (; os; os &= os - 1u) {
                        const int x = top_bit(os & (0u - os));
                        S.sz[j++] = (srun(b, w, x) << CRUN_BITS) | srun(bt, wt, x);
                    }
                };
                if (osz) list(below(tid, true), osz);
                if (osy) list(below(tid, false), osy);
                __syncthreads();
                for (int k = tid; k < npairs; k += CNT)
                    s_union(S.par, S.sz[k] >> CRUN_BITS, S.sz[k] & (CRUN - 1), lcap, status);
            }
        }
        if (!listed) {
            if (tid < nseg) {
                S.sz[tid] = (int)osz;
                S.sz[CSEG + tid] = (int)osy;
            }
            __syncthreads();
        }
        const int groups = nseg > 0 ? CNT / nseg : 1, group = nseg > 0 ? tid / nseg : CNT;
        for (int share = (listed ? 16 : 0) + group; group < groups && share < 17; share += groups) {
            const int ls = tid - group * nseg;
            const uint32_t w = S.m[ls];
            if (share < 16) {
                uint32_t os = (uint32_t)S.sz[share < 8 ? ls : CSEG + ls] & (0xfu << (4 * (share & 7)));
                if (!os) continue;
                const int t = below(ls, share < 8), b = S.sb[ls], bt = S.sb[t];
                const uint32_t wt = S.m[t];
                for (; os; os &= os - 1u) {
                    const int x = top_bit(os & (0u - os));
                    s_union(S.par, srun(b, w, x), srun(bt, wt, x), lcap, status);
                }
            } else if (w & 1u) {                     // along x: rows of several segments, the periodic edge
                const int bx = seg0 + ls - (int)div_nbx((uint32_t)(seg0 + ls)) * nbx;
                const int t = bx > 0 ? ls - 1 : ls + nbx - 1, x = bx > 0 ? 31 : lastbit;
                if ((bx > 0 || (L.per[0] && nx >= 2)) && ((S.m[t] >> x) & 1u))
                    s_union(S.par, S.sb[ls], srun(S.sb[t], S.m[t], x), lcap, status);
            }
        }
        __syncthreads();
        // local roots, then cluster numbers: every run points at its local root
        for (int i = tid; i < total; i += CNT) {
            int root = S.par[i];
            for (int up = S.par[root]; up != root; up = S.par[root]) root = S.par[up];   // two levels a step
            S.sz[i] = root;
        }
        __syncthreads();
        for (int i = tid; i < total; i += CNT) {
            const int r = S.sz[i];
            S.par[i] = cbase | r;
            if (r == i) S.desc[i] |= DESC_LROOT;
        }
    }
    cl.sync();
    {   // the edges to other CTAs, joined between the two runs' local roots
        const int cap = (local_cap > 0 && local_cap < CS * CRUN) ? local_cap : CS * CRUN;
        join_cross([&](int a, int o, int bb) {
            V.unite(S.par[a], *cl.map_shared_rank(&S.par[bb], o), cap, status);
        });
    }
    __syncthreads();                                  // the pair list is read
    for (int i = tid; i < total; i += CNT) S.sz[i] = 0;
    cl.sync();                                        // ... and every size slot cleared
    // every local root learns its cluster's root (the finds that cross CTAs walk only
    // local roots); the other runs still point at their local roots
    for (int i = tid; i < total; i += CNT)
        if (S.desc[i] & DESC_LROOT) S.par[i] = V.find_ro(cbase | i);
    __syncthreads();

    // piece sizes: every run's length goes to its local root, in this CTA's shared
    // memory; a local root that is not its cluster's root then passes its sum on to the
    // cluster root, once per group of lanes with the same cluster root
    for (int i = tid; i < total; i += CNT) {
        const int d = S.desc[i];
        const int lr = (d & DESC_LROOT) ? i : (S.par[i] & (CRUN - 1));
        atomicAdd(&S.sz[lr], run_len(S.m[(d & ~DESC_LROOT) >> 5], d & 31));
    }
    __syncthreads();
    for (int i0 = 0; i0 < total; i0 += CNT) {   // warp-uniform trips
        const int i = i0 + tid;
        int root = -1, sum = 0;
        if (i < total && (S.desc[i] & DESC_LROOT) && S.par[i] != (cbase | i)) {
            root = S.par[i];
            sum = S.sz[i];
        }
        const unsigned peers = __match_any_sync(0xffffffffu, root);
        const int tot = (int)__reduce_add_sync(peers, (unsigned)sum);
        if (root >= 0 && lane == __ffs(peers) - 1) atomicAdd(V.sz(root), tot);
    }
    __syncthreads();
    for (int i = tid; i < total; i += CNT)   // every run now points at its cluster root
        if (!(S.desc[i] & DESC_LROOT)) S.par[i] = S.par[S.par[i] & (CRUN - 1)];

    // a4, a6, a7: the roots in run order get consecutive ranks; the roots of the CTAs
    // before this one come first.  The cluster roots (local roots pointing at
    // themselves) are counted before the barrier that completes the sizes, which then
    // publishes the counts too.
    const int per = (total + CNT - 1) / CNT;
    const int i0 = tid * per, i1 = min(i0 + per, total);
    int nr = 0;
    for (int i = i0; i < i1; ++i) nr += S.par[i] == (cbase | i);
    int nroots;
    int rank = cta_exscan<CNT>(nr, S, nroots);
    if (tid == 0) S.roots = nroots;
    cl.sync();
    int all = 0;
    if (wid == 0) {
        const int r = lane < CS ? (lane == c ? nroots : *cl.map_shared_rank(&S.roots, lane)) : 0;
        const int before = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < c ? r : 0));
        all = (int)__reduce_add_sync(0xffffffffu, (unsigned)r);
        if (lane == 0) S.scan_total = before;
    }
    __syncthreads();
    rank += S.scan_total;
    const int64_t capr = L.sizes_cap;
    for (int i = i0; i < i1; ++i) {
        if (S.par[i] != (cbase | i)) continue;
        const int size = S.sz[i];
        if (rank < capr) L.sizes[rank] = size;
        ++rank;
        atomicAdd(&S.hist[31 - __clz(size)], 1);
    }
    __syncthreads();   // this CTA's sizes are out: sz now takes each run's label

    // each run's label, the first site of its cluster's root run (the root's descriptor,
    // read once per group of lanes with the same root)
    for (int i0 = 0; i0 < total; i0 += CNT) {
        const int i = i0 + tid;
        const int root = i < total ? S.par[i] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, root);
        const int leader = __ffs(peers) - 1;
        int d = 0;
        if (root >= 0 && lane == leader) {
            const int o = root >> CRUN_BITS;
            const uint16_t *dp = &S.desc[root & (CRUN - 1)];
            d = o == c ? *dp : *cl.map_shared_rank(dp, o);
        }
        d = __shfl_sync(0xffffffffu, d, leader) & ~DESC_LROOT;
        if (i < total) {
            const int sg = (root >> CRUN_BITS) * rp * nbx + (d >> 5), rq = (int)div_nbx((uint32_t)sg);
            S.sz[i] = rq * nx + (sg - rq * nbx) * 32 + (d & 31);
        }
    }
    __syncthreads();

    // a5: labels, one warp per segment, one lane per site, four segments a step
    for (int l0 = wid; l0 < nseg; l0 += 4 * NW) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int ls = l0 + u * NW;
            if (ls >= nseg) break;
            const int sg = seg0 + ls;
            const int q = (int)div_nbx((uint32_t)sg), x = (sg - q * nbx) * 32 + lane;
            const uint32_t w = S.m[ls];
            const int lab = ((w >> lane) & 1u) ? S.sz[srun(S.sb[ls], w, lane)] : -1;
            if (x < nx) L.labels[(int64_t)q * nx + x] = lab;
        }
    }
    // the histogram of the whole lattice gathers in CTA 0
    if (c != 0 && tid < 32 && S.hist[tid]) atomicAdd(cl.map_shared_rank(&S.hist[tid], 0), S.hist[tid]);
    cl.sync();   // no CTA's shared memory is reached after this
    if (c == 0) {
        if (tid < 32 && L.hist) L.hist[tid] = S.hist[tid];
        if (tid == 0 && L.ncl) L.ncl[0] = all;
    }
}

}  // namespace

bool small_fits(int nx, int ny, int nz) {
    const int64_t N = (int64_t)nx * ny * nz;
    const int64_t nseg = (int64_t)((nx + TX - 1) / TX) * ny * nz;
    return N <= SMALL_MAX_SITES && nseg <= SMALL_MAX_SEG;
}

// log2 of the cluster size this device runs the cluster kernel with (4 or 3), or 0 if
// it cannot run it, and how many such clusters it holds at once; checked once per device
static int cluster_bits(int *slots_out = nullptr) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
        cudaGetLastError();
        return 0;
    }
    static int state[MAX_DEVICES];   // -1 unknown, else the cluster bits (0: none)
    static int slots[MAX_DEVICES];   // clusters resident at once
    static bool init = false;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (!init) {
        for (int &v : state) v = -1;
        init = true;
    }
    if (state[dev] < 0) {
        // the kernels take the attributes, and a cluster fits the device
        auto fits = [](auto k1, auto kn, int cs, int &nclusters) {
            if (cs > 8 && (cudaFuncSetAttribute(k1, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                           cudaFuncSetAttribute(kn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess))
                return false;
            if (cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClusterSmem)) !=
                    cudaSuccess ||
                cudaFuncSetAttribute(kn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ClusterSmem)) !=
                    cudaSuccess)
                return false;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(cs, 1, 1);
            cfg.blockDim = dim3(CNT, 1, 1);
            cfg.dynamicSmemBytes = sizeof(ClusterSmem);
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = cs;
            attr.val.clusterDim.y = 1;
            attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            nclusters = 0;
            return cudaOccupancyMaxActiveClusters(&nclusters, k1, &cfg) == cudaSuccess && nclusters > 0;
        };
        int bits = 0, n = 0;
        if (fits(k_small_cluster<4, 1>, k_small_cluster<4, MAX_LAT_PER_LAUNCH>, 16, n)) bits = 4;
        else if (fits(k_small_cluster<3, 1>, k_small_cluster<3, MAX_LAT_PER_LAUNCH>, 8, n)) bits = 3;
        cudaGetLastError();
        state[dev] = bits;
        slots[dev] = bits ? n : 0;
    }
    if (slots_out) *slots_out = slots[dev];
    return state[dev];
}

int cluster_slots() {
    int n = 0;
    cluster_bits(&n);
    return n;
}

bool cluster_ok() { return cluster_bits() > 0; }

bool cluster_fits(int nx, int ny, int nz) {
    const int cs = 1 << cluster_bits();
    const int64_t nbx = (nx + TX - 1) / TX, rows = (int64_t)ny * nz;
    return cluster_bits() > 0 && nx >= 1 && ny >= 1 && nz >= 1 && ((rows + cs - 1) / cs) * nbx <= CSEG;
}

template <int CSB>
static void launch_cluster(const LatDev *lats, int n, int32_t *status, int32_t local_cap, cudaStream_t st) {
    constexpr int CS = 1 << CSB;
    if (n == 1) {
        LatBatch<1> B;
        std::memset(&B, 0, sizeof(B));
        B.n = 1;
        B.lat[0] = lats[0];
        k_small_cluster<CSB, 1><<<CS, CNT, sizeof(ClusterSmem), st>>>(B, status, local_cap);
    } else {
        LatBatch<MAX_LAT_PER_LAUNCH> B;
        std::memset(&B, 0, sizeof(B));
        B.n = n;
        for (int i = 0; i < n; ++i) B.lat[i] = lats[i];
        k_small_cluster<CSB, MAX_LAT_PER_LAUNCH><<<(unsigned)(CS * n), CNT, sizeof(ClusterSmem), st>>>(B, status,
                                                                                                    local_cap);
    }
}

cudaError_t launch_small(const LatDev *lats, int n, int32_t *status, int32_t local_cap, cudaStream_t st,
                         bool cluster) {
    if (n <= 0) return cudaSuccess;
    if (n > MAX_LAT_PER_LAUNCH) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    if (cluster) {   // cluster_bits() has set the kernels' attributes
        const int bits = cluster_bits();
        if (bits == 4) launch_cluster<4>(lats, n, status, local_cap, st);
        else if (bits == 3) launch_cluster<3>(lats, n, status, local_cap, st);
        else return cudaErrorNotSupported;
        return cudaGetLastError();
    }
    static bool attr_set[MAX_DEVICES][2];
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (n == 1) {
        if (!attr_set[dev][0]) {
            e = cudaFuncSetAttribute(k_small_label<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(SmallSmem));
            if (e != cudaSuccess) return e;
            attr_set[dev][0] = true;
        }
        LatBatch<1> B;
        std::memset(&B, 0, sizeof(B));
        B.n = 1;
        B.lat[0] = lats[0];
        k_small_label<1><<<1, SNT, sizeof(SmallSmem), st>>>(B, status, local_cap);
    } else {
        if (!attr_set[dev][1]) {
            e = cudaFuncSetAttribute(k_small_label<MAX_LAT_PER_LAUNCH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(SmallSmem));
            if (e != cudaSuccess) return e;
            attr_set[dev][1] = true;
        }
        LatBatch<MAX_LAT_PER_LAUNCH> B;
        std::memset(&B, 0, sizeof(B));
        B.n = n;
        for (int i = 0; i < n; ++i) B.lat[i] = lats[i];
        k_small_label<MAX_LAT_PER_LAUNCH><<<(unsigned)n, SNT, sizeof(SmallSmem), st>>>(B, status, local_cap);
    }
    return cudaGetLastError();
}

}  // namespace hk
