// DSMC kernels: initialisation, the move with diffuse isothermal walls and binning by cell,
// and the per-cell stable ordering, no-time-counter hard-sphere collisions and
// Hermite-moment sampling.
//
// Particles live in per-cell bins of `bin` slots (cell c owns slots [c bin, (c+1) bin) of
// each state array, count[c] in use) and ping-pong between two halves. A DSMC step (the NTC
// order of Bird that the paper uses in Sec. 5: move, index, collide, sample) from the sorted
// particles of half p takes two passes:
//   k_move     one warp per source cell: body-force kick, free flight, diffuse wall
//              re-emission (Sec. 3.1), periodic wrap, new cell; the moved particle and its
//              order key (its displacement's neighbour offset, then its rank in the old cell;
//              see order_key) are appended to the bin of its new cell in half p^1 by a
//              warp-aggregated atomic.
//   k_collide  four consecutive cells per warp, a group of 8 lanes per cell: each arrival's
//              rank by key comes from a bitmap of the cell's keys with prefix counts, each
//              arrival is placed at its rank in the warp's shared-memory pool, the NTC candidates
//              of a cell are drawn and settled eight at a time by its lanes
//              (Eq. collisionnumber), the sums 1, v, vv, vvv are added to the FP64 cumulative
//              sums of the cell (Sec. 2.1, Fig. 1) and the sorted cell is written back in place.
//   k_step_end one thread after a context's collide pass: publishes the particle count and
//              advances the step and sample counters (in a batch the LB step does).
// Several steps in one call fuse the collide of step s with the move of step s + 1: the
// fused pass collides and samples a cell as above and then moves its particles straight from
// the pool into the bins of the other half, so a particle's state is read and written once
// per step. Cells that the step's LB2DSMC regenerates are written back in place instead.
// This file is compiled without FMA contraction so that positions, cell keys, pair choices
// and post-collision velocities are the IEEE float (or double) results of the written
// expressions.
#include <cmath>
#include <cstring>

#include "dsmc_move.cuh"

namespace hyb {

namespace {

// Isotropic unit vector (Marsaglia 1972) from the NTC scattering stream of candidate k.
template <typename Real>
__device__ __forceinline__ int unit_vector(uint64_t seed, uint32_t c, uint32_t s, uint32_t k, Real& nx,
                                           Real& ny, Real& nz) {
    for (int blk = 0; blk < kMaxScatterBlocks; ++blk) {
        const uint4 r = draw(seed, c, s, TAG_NTC_SCAT, k, (uint32_t)blk);
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            // u = 2 U - 1 with U of 24 bits is m 2^-23, m an integer
            const int m1 = (int)(w[2 * h] >> 8) - (1 << 23), m2 = (int)(w[2 * h + 1] >> 8) - (1 << 23);
            Real u1 = 0, u2 = 0, ss = 0;
            bool in;
            if constexpr (sizeof(Real) == 8) {
                // u1^2 + u2^2 and its comparison with one are exact in integers, and so is the
                // double sum: no operation of the FP64 pipe (19 cycles a warp instruction and SM)
                // for a rejected draw (20 steps of 64 x 64 cells 3.28 -> 3.12 ms)
                const long long mm = (long long)m1 * m1 + (long long)m2 * m2;
                in = mm < (1ll << 46);
                if (in) {
                    ss = (Real)mm * (Real)0x1p-46;
                    u1 = (Real)m1 * (Real)0x1p-23;
                    u2 = (Real)m2 * (Real)0x1p-23;
                }
            } else {
                u1 = (Real)m1 * (Real)0x1p-23;
                u2 = (Real)m2 * (Real)0x1p-23;
                ss = u1 * u1 + u2 * u2;
                in = ss < (Real)1;
            }
            if (in) {
                const Real a = (Real)2 * sqrt((Real)1 - ss);
                nx = u1 * a;
                ny = u2 * a;
                nz = (Real)1 - (Real)2 * ss;
                return 1;
            }
        }
    }
    nx = ny = nz = (Real)0;
    return 0;
}

// ---------------------------------------------------------------------------------------
template <typename Real>
__global__ void k_init_particles(DsmcArgs<Real> a) {
    const int64_t n = (int64_t)a.ncells * a.ppc;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t cl = (uint32_t)(s / a.ppc), k = (uint32_t)(s % a.ppc);
        const int ix = (int)(cl % (uint32_t)a.ncx);
        const int iy = a.y0 + (int)((cl / (uint32_t)a.ncx) % (uint32_t)a.ncy);  // the channel's row
        const int64_t slot = (int64_t)cl * a.bin + k;
        const uint32_t c = global_cell(cl, a.ncx, a.ncy, a.y0, a.ncy_g);  // key of the draws
        const uint4 rp = draw(a.seed, c, 0, TAG_INIT_POS, k, 0);
        const Real px = (Real)ix + (Real)u01f(rp.x);
        const Real py = (Real)iy + (Real)u01f(rp.y);
        const Real pz = a.ncz ? (Real)(cl / ((uint32_t)a.ncx * (uint32_t)a.ncy)) + (Real)u01f(rp.z)
                              : (Real)0;
        const uint4 rv = draw(a.seed, c, 0, TAG_INIT_VEL, k, 0);
        Real n0, n1, n2, n3;
        gauss_pair<Real>(rv.x, rv.y, n0, n1);
        gauss_pair<Real>(rv.z, rv.w, n2, n3);
        rec_put(a.drec, slot, px, py, pz, n0, n1, n2, 0u);
    }
}

template <typename Real>
__global__ void k_init_cells(DsmcArgs<Real> a) {
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < a.ncells;
         c += (int64_t)gridDim.x * blockDim.x) {
        a.count_d[c] = (uint32_t)a.ppc;
        a.count_s[c] = 0;
        a.crmax[c] = (Real)a.crmax_init;
        a.rem[c] = (Real)0;
        a.nbar_sum[c] = 0u;
        for (int m = 0; m < kMoments; ++m) a.acc[c * kMoments + m] = 0.0;
        if (c == 0) {
            for (int w = 0; w < CTRL_WORDS; ++w) a.ctrl[w] = 0;
            a.ctrl[CTRL_NTOT] = (uint32_t)((int64_t)a.ncells * a.ppc);
            for (int w = 0; w < HYB_NCOUNTERS; ++w) a.counters[w] = 0;
        }
    }
}

// ---------------------------------------------------------------------------------------
// Move (kick, drift, walls, wrap) of the sorted particles of half p into the bins of p^1.

template <typename Real>
__device__ __forceinline__ MoveCtx<Real> move_ctx(const DsmcArgs<Real>& a) {
    MoveCtx<Real> m;
    m.H = (Real)a.ncx;
    m.L = (Real)a.ncy_g;
    m.Lz = (Real)(a.ncz ? a.ncz : 1);
    m.dt = a.dt_r;
    m.g = a.g_r;
    m.ncx = a.ncx;
    m.ncy = a.ncy_g;
    m.ncz = a.ncz;
    m.y0 = a.y0;
    m.nly = a.ncy;
    m.bin = (uint32_t)a.bin;
    m.seed = a.seed;
    return m;
}

template <typename Real>
__device__ __forceinline__ Half<Real> half_s(const DsmcArgs<Real>& a) {
    return Half<Real>{a.srec, a.count_s};
}
template <typename Real>
__device__ __forceinline__ Half<Real> half_d(const DsmcArgs<Real>& a) {
    return Half<Real>{a.drec, a.count_d};
}

// One source cell, by one warp; 64 particles of the cell at a time, two per lane, with the
// loads, flights and binning atomics of both in flight together. In FP64 a particle that hits a
// wall takes some hundreds of instructions of 66 cycles' latency more (the re-emission's logarithm,
// square root, sine and cosine), and a warp would spend them again for every 32 particles of
// which one hits: such particles are listed in `later` and taken together, packed, when the others
// are done (20 steps of the FP64 64-cell channel 3.03 -> 2.80 ms, of 64 x 64 cells
// 3.52 -> 3.32 ms). A cell of at most 32 particles takes them all in one trip, wall or not: with a
// second trip for the walls' the move of 16k cells of 8 particles took 43.2 us, in 3D 60.4, against
// 38.3 and 53.6 in one. In FP32 the list cost what it saved (64 batched channels, 10
// steps: 1.11 against 1.04 ms).
template <typename Real, bool Z3>
__device__ __forceinline__ void move_cell(const DsmcArgs<Real>& a, int c, unsigned lane, uint8_t* later) {
    const uint32_t s = a.ctrl[CTRL_STEP];
    const MoveCtx<Real> m = move_ctx(a);
    const uint32_t bin = (uint32_t)a.bin;
    // the halves do not overlap: loads of the next records need not wait for earlier stores
    const Real* __restrict__ src = a.srec;
    const Half<Real> dst = half_d(a);
    uint32_t hits = 0, caps = 0, lost = 0;
    uint32_t n = a.count_s[c];
    __syncwarp();
    if (lane == 0) a.count_s[c] = 0;  // half p is consumed; its counts start the next arrivals
    if (n > bin) n = bin;
    const int64_t base = (int64_t)c * bin;
    // the channel's cell: the key of the wall draws and of the order keys
    const Origin org = origin_of(m, global_cell((uint32_t)c, a.ncx, a.ncy, a.y0, a.ncy_g));
    constexpr bool PACK = sizeof(Real) == 8;
    const unsigned below = (1u << lane) - 1u;
    uint32_t nlater = 0;
    auto put_away = [&](bool act, int dir, uint32_t key, uint32_t arr, uint32_t ok, const Real (&p)[6]) {
        if (act && dir < 0) {
            if (arr < bin)
                put_particle<Real, Z3>(dst, (int64_t)key * bin + arr, ok, p[0], p[1], p[2], p[3], p[4], p[5]);
            else
                lost += 1;
        } else if (act) {
            send_particle<Real, Z3>(a.xrec, a.xkey, a.xcount, a.xcap, dir, key, ok, p[0], p[1], p[2], p[3], p[4],
                                    p[5], lost);
        }
    };
    // all of a cell's particles in one trip of the warp: nothing to pack
    const bool few = PACK && n <= 32;
    Real p0[6] = {0, 0, 0, 0, 0, 0};
    for (uint32_t k0 = 0; k0 == 0 || k0 < n; k0 += 64) {
        const uint32_t k1 = k0 + lane, k2 = k1 + 32;
        Real p1[6] = {0, 0, 0, 0, 0, 0}, p2[6] = {0, 0, 0, 0, 0, 0};  // x y z vx vy vz
        uint32_t t1, t2;
        // the loads need only the bin size, not the count, so they travel with it
        if (k1 < bin) rec_get(src, base + k1, p1[0], p1[1], p1[2], p1[3], p1[4], p1[5], t1);
        if (k2 < bin) rec_get(src, base + k2, p2[0], p2[1], p2[2], p2[3], p2[4], p2[5], t2);
        if (few) {
#pragma unroll
            for (int i = 0; i < 6; ++i) p0[i] = p1[i];
            break;
        }
        const bool act1 = k1 < n && (!PACK || flies_straight(m, p1[0], p1[3]));
        const bool act2 = k2 < n && (!PACK || flies_straight(m, p2[0], p2[3]));
        if constexpr (PACK) {
            const unsigned w1 = __ballot_sync(kFull, k1 < n && !act1), w2 = __ballot_sync(kFull, k2 < n && !act2);
            if (k1 < n && !act1) later[nlater + __popc(w1 & below)] = (uint8_t)k1;
            nlater += __popc(w1);
            if (k2 < n && !act2) later[nlater + __popc(w2 & below)] = (uint8_t)k2;
            nlater += __popc(w2);
        }
        uint32_t key1 = 0, key2 = 0, ok1 = 0, ok2 = 0;
        int dir1 = -1, dir2 = -1;
        if (act1)
            key1 = move_particle<Real, Z3, !PACK>(m, org, k1, s, p1[0], p1[1], p1[2], p1[3], p1[4], p1[5], hits,
                                                  caps, dir1, ok1);
        if (act2)
            key2 = move_particle<Real, Z3, !PACK>(m, org, k2, s, p2[0], p2[1], p2[2], p2[3], p2[4], p2[5], hits,
                                                  caps, dir2, ok2);
        uint32_t arr1, arr2;
        bin_arrival2(dst.count, key1, act1 && dir1 < 0, key2, act2 && dir2 < 0, lane, arr1, arr2);
        put_away(act1, dir1, key1, arr1, ok1, p1);
        put_away(act2, dir2, key2, arr2, ok2, p2);
    }
    if (few) nlater = n;
    if (PACK && nlater > 0) {
        __syncwarp();
        for (uint32_t i0 = 0; i0 < nlater; i0 += 32) {
            const bool act = i0 + lane < nlater;
            Real p[6] = {p0[0], p0[1], p0[2], p0[3], p0[4], p0[5]};
            uint32_t key = 0, ok = 0, t;
            int dir = -1;
            if (act) {
                const uint32_t k = few ? lane : later[i0 + lane];
                if (!few) rec_get(src, base + k, p[0], p[1], p[2], p[3], p[4], p[5], t);
                key = move_particle<Real, Z3>(m, org, k, s, p[0], p[1], p[2], p[3], p[4], p[5], hits, caps, dir, ok);
            }
            const uint32_t arr = bin_arrival1(dst.count, key, act && dir < 0, lane);
            put_away(act, dir, key, arr, ok, p);
        }
    }
    move_events(a.counters, a.ctrl, hits, caps, lost, lane);
}

// One warp per source cell (the cells of all replicas in the batch form).
template <typename Real, bool BATCH, bool Z3 = false>
__global__ void __launch_bounds__(256, sizeof(Real) == 4 ? 4 : (BATCH ? 2 : 3)) k_move(Launch<DsmcArgs<Real>> L) {
    __shared__ uint8_t s_later[sizeof(Real) == 8 ? 8 : 1][256];  // a bin has at most 256 slots
    uint8_t* later = s_later[sizeof(Real) == 8 ? threadIdx.x >> 5 : 0];
    pdl_begin();
    const unsigned lane = lane_id();
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = gw; u < L.total; u += nw) {
        if constexpr (BATCH) {
            const int r = replica_of(L.pre, L.nrep, u);
            move_cell<Real, Z3>(L.tab[r], (int)(u - L.pre[r]), lane, later);
        } else {
            move_cell<Real, Z3>(L.one, (int)u, lane, later);
        }
    }
}

// ---------------------------------------------------------------------------------------
// Collide: a warp takes four consecutive cells, eight lanes per cell, from the arrivals to the
// written or moved particles, without waiting for any other warp. All loops that contain
// shuffles have warp-uniform trip counts (groups whose cell has less work are masked), so
// every shuffle is executed by the full warp.
//
// Bound by latency and issue, not by bandwidth (ncu, 6.55M particles with Kn along the channel:
// issue 52%, DRAM a third of its peak, 15.9 warp instructions per particle). No block barrier:
// while one warp of a block ran the block's NTC chains and the others waited, barriers were a
// fifth of the stalls (105M particles, 20 steps: 78.0 ms; warps on their own: 70.3 ms). The
// arrivals are copied to shared memory by asynchronous copies and stay where they land, a byte
// per rank pointing at them, and a cell's particles bound for one neighbour share one
// reservation of slots there, all nine in flight together, instead of one dependent global
// atomic per eight particles (61.7 ms; 819k particles 2.17 -> 1.35 ms, 3D 6.55M
// 13.6 -> 9.0 ms, 64 batched channels, 10 steps, 1.50 -> 1.04 ms).
constexpr int kGroup = 8;
constexpr int kWarpCells = 32 / kGroup;

// Blocks of 8 warps (32 cells) or 4 (16 cells) only group warps for a launch: a block keeps its
// shared memory until its slowest warp is done, so 4 are faster where the grid runs many waves
// (105M particles, 20 steps: 61.7 against 63.7 ms) and 8 by 2% where it does not. 24 resident warps
// per SM in FP32 (80 registers; the 3D fused pass spills 32 bytes at them): 28 took 67.2 ms (spills, and
// little L1 left beside the pools).
constexpr int kCollideWarps = 8;
template <typename Real, int W>
struct CollideCfg {
    static constexpr int MINB = (sizeof(Real) == 4 ? 24 : 16) / W;  // resident blocks per SM
};
enum CollideMode : int { MODE_COLLIDE = 0, MODE_FUSED = 1 };
constexpr int kCollideStatic = 64;  // bytes, at least the block's event sums beside the warps' memory

// Words of a cell's order-key bitmap: one bit per key below W bin, W = 9 neighbour offsets in
// 2D and 27 in 3D (bin is a multiple of 32).
template <bool Z3>
__host__ __device__ constexpr int neighbours() {
    return Z3 ? 27 : 9;
}
template <bool Z3>
__host__ __device__ constexpr int bitmap_words(uint32_t bin) {
    return neighbours<Z3>() * (int)(bin / 32u);
}
// Keys of farther-displaced particles a cell lists for their ranks (more are counted in full).
constexpr int kFarList = 8;

// Shared memory of one warp, byte offsets: per slot of its pool (x, y, vx, vy), then vz (, z), the
// order key (after the collide: the slot's place in its new cell) and the slot of each rank; then
// the cells' key bitmaps (words, listed far keys, prefix bytes), in whose place come, once the
// ranks are taken, the cells' FP64 sums and the slots reserved in each neighbour's bin.
struct WarpMem {
    uint32_t b, key, perm, scratch, total;
};
template <typename Real, bool Z3>
__host__ __device__ constexpr WarpMem warp_mem(uint32_t pool, uint32_t bin) {
    WarpMem m{};
    m.b = pool * 4u * (uint32_t)sizeof(Real);  // pool is a multiple of 8
    m.key = m.b + pool * (Z3 ? 2u : 1u) * (uint32_t)sizeof(Real);
    m.perm = m.key + pool * 4u;
    m.scratch = (m.perm + pool + 15u) / 16u * 16u;
    const uint32_t bits = (uint32_t)kWarpCells * ((uint32_t)bitmap_words<Z3>(bin) * 5u + (kFarList + 1u) * 4u);
    const uint32_t after = (uint32_t)kWarpCells * (kMoments * 8u + (uint32_t)neighbours<Z3>() * 8u);
    m.total = m.scratch + ((bits > after ? bits : after) + 15u) / 16u * 16u;
    return m;
}

// Four Reals of shared memory, 16-byte aligned (32 in FP64), as vector accesses.
__device__ __forceinline__ void get4(const float* p, float& a, float& b, float& c, float& d) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x, b = v.y, c = v.z, d = v.w;
}
__device__ __forceinline__ void get4(const double* p, double& a, double& b, double& c, double& d) {
    const double2 u = *reinterpret_cast<const double2*>(p), v = *reinterpret_cast<const double2*>(p + 2);
    a = u.x, b = u.y, c = v.x, d = v.y;
}
__device__ __forceinline__ void put4(float* p, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void put4(double* p, double a, double b, double c, double d) {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
    *reinterpret_cast<double2*>(p + 2) = make_double2(c, d);
}

// Adds a particle's velocity moments to a lane's partial sums: u, the six distinct products
// u_i u_j and the ten distinct u_i u_j u_k, in the order of the sampled sums (mo[0], the count,
// is set after the reduction). The sums are compared with a tolerance, so they use fused
// multiply-adds (this file is otherwise compiled without contraction).
template <typename Real>
__device__ __forceinline__ void add_moments(Real (&mo)[kMoments], Real ux, Real uy, Real uz) {
    const Real xx = ux * ux, yy = uy * uy, zz = uz * uz, xy = ux * uy;
    mo[1] += ux; mo[2] += uy; mo[3] += uz;
    mo[4] += xx; mo[5] = fma(ux, uy, mo[5]); mo[6] = fma(ux, uz, mo[6]);
    mo[7] += yy; mo[8] = fma(uy, uz, mo[8]); mo[9] += zz;
    mo[10] = fma(xx, ux, mo[10]); mo[11] = fma(xx, uy, mo[11]);
    mo[12] = fma(xx, uz, mo[12]); mo[13] = fma(yy, ux, mo[13]);
    mo[14] = fma(xy, uz, mo[14]); mo[15] = fma(zz, ux, mo[15]);
    mo[16] = fma(yy, uy, mo[16]); mo[17] = fma(yy, uz, mo[17]);
    mo[18] = fma(zz, uy, mo[18]); mo[19] = fma(zz, uz, mo[19]);
}

// t > v for values that are not negative (or equal): in FP64 on the integer pipe, where the bits of
// non-negative doubles order like the values.
__device__ __forceinline__ bool above(float t, float v) { return t > v; }
__device__ __forceinline__ bool above(double t, double v) {
    return __double_as_longlong(t) > __double_as_longlong(v);
}

// One NTC candidate: the pair (ranks in the cell), the acceptance uniform and the direction of
// the relative velocity after the collision (ok = 0 if its draws ran out).
template <typename Real>
struct Candidate {
    uint32_t i, j;
    Real R, nx, ny, nz;
    int ok;
};
template <typename Real>
__device__ __forceinline__ void draw_candidate(Candidate<Real>& q, uint64_t seed, uint32_t gc, uint32_t s,
                                               uint32_t n, uint32_t k) {
    const uint4 r = draw(seed, gc, s, TAG_NTC_PAIR, k, 0);
    q.i = uindex(r.x, n);
    q.j = uindex(r.y, n - 1u);
    if (q.j >= q.i) q.j += 1u;
    q.R = (Real)u01f(r.z);
    q.ok = unit_vector(seed, gc, s, k, q.nx, q.ny, q.nz);
}

// The NTC candidates of a cell group's cell (nsel of them, n particles; `va` and `vb` point at
// (vx, vy) and vz of slot 0, 4 and NB Reals a slot, perm gives the slot of each rank), applied in
// their order; q holds the lane's candidate of the first eight. The cell's lanes take eight
// consecutive candidates at a time and settle them together: every pending lane forms its
// relative speed from the current velocities, the running (sigma c_r)_max up to its candidate by
// a prefix maximum and its decision; a candidate that shares a particle with an earlier one of
// the window that collides must see that collision, so the candidates before the first such one
// are final and the others are taken again from the updated velocities. The results are those of
// applying the candidates one after another, bit for bit. Shared particles are found with 64-bit
// sets of the particles (index modulo 64; an alias only takes a candidate again). The first
// pending candidate is always final, so every pass settles at least one.
template <typename Real, int NB>
__device__ __forceinline__ void ntc_collisions(Candidate<Real>& q, uint64_t seed, uint32_t gc, uint32_t s, uint32_t n,
                                               uint32_t nsel, Real* va, Real* vb, const uint8_t* perm, int grp,
                                               int gl, Real& cm, uint32_t& ncoll, uint32_t& flags) {
    constexpr int G = kGroup;
    const uint32_t maxsel = __reduce_max_sync(kFull, nsel);
    for (uint32_t k0 = 0; k0 < maxsel; k0 += G) {
        const uint32_t k = k0 + (uint32_t)gl;
        bool pend = k < nsel;
        if (k0 > 0 && pend) draw_candidate(q, seed, gc, s, n, k);
        uint32_t pi = 0, pj = 0;
        if (pend) pi = perm[q.i], pj = perm[q.j];
        Real* ai = va + 4 * pi;
        Real* aj = va + 4 * pj;
        Real* bi = vb + NB * pi;
        Real* bj = vb + NB * pj;
        const uint32_t si = 1u << (q.i & 31u), sj = 1u << (q.j & 31u);
        const uint32_t mlo = ((q.i & 32u) ? 0u : si) | ((q.j & 32u) ? 0u : sj);
        const uint32_t mhi = ((q.i & 32u) ? si : 0u) | ((q.j & 32u) ? sj : 0u);
        while (__any_sync(kFull, pend)) {
            Real ax = 0, ay = 0, az = 0, bx = 0, by = 0, bz = 0, cr = 0;
            Real v = cm;
            if (pend) {
                ax = ai[0], ay = ai[1], az = bi[0];
                bx = aj[0], by = aj[1], bz = bj[0];
                const Real ddx = ax - bx, ddy = ay - by, ddz = az - bz;
                cr = sqrt(ddx * ddx + ddy * ddy + ddz * ddz);
                if (cr > cm) v = cr;
            }
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const Real t = __shfl_up_sync(kFull, v, o, G);
                if (gl >= o && above(t, v)) v = t;
            }
            const bool acc = pend && cr > q.R * v;
            const bool coll = acc && q.ok;
            uint32_t elo = coll ? mlo : 0u, ehi = coll ? mhi : 0u;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const uint32_t tl = __shfl_up_sync(kFull, elo, o, G), th = __shfl_up_sync(kFull, ehi, o, G);
                if (gl >= o) elo |= tl, ehi |= th;
            }
            // exclusive: the particles of the earlier lanes' collisions
            elo = __shfl_up_sync(kFull, elo, 1, G);
            ehi = __shfl_up_sync(kFull, ehi, 1, G);
            const bool conf = pend && gl > 0 && ((elo & mlo) | (ehi & mhi)) != 0u;
            const unsigned cb = (__ballot_sync(kFull, conf) >> (G * grp)) & ((1u << G) - 1u);
            const int cut = cb ? __ffs((int)cb) - 1 : G;
            if (pend && gl < cut) {
                pend = false;
                if (coll) {
                    const Real cx = (ax + bx) * (Real)0.5;
                    const Real cy = (ay + by) * (Real)0.5;
                    const Real cz = (az + bz) * (Real)0.5;
                    const Real h = cr * (Real)0.5;
                    const Real hx = h * q.nx, hy = h * q.ny, hz = h * q.nz;
                    ai[0] = cx + hx;
                    ai[1] = cy + hy;
                    bi[0] = cz + hz;
                    aj[0] = cx - hx;
                    aj[1] = cy - hy;
                    bj[0] = cz - hz;
                    ncoll += 1;
                } else if (acc) {
                    flags |= HYB_ST_SCATTER_CAP;
                }
            }
            cm = __shfl_sync(kFull, v, cut - 1, G);
            __syncwarp();
        }
    }
}

// The same with a window that moves on by the settled candidates after every pass, so that a pass
// takes eight as long as there are any. It saves passes of dense cells (20 steps of 64 x 64 cells in
// FP64 3.08 -> 2.93 ms, 10 of 64 batched channels 0.949 -> 0.919 ms) and costs shuffles where most
// cells have few candidates: FP32 fused passes keep the other (105M particles, 20 steps: 61.3
// against 61.6 ms; one function for both forms, 61.7 ms with its registers).
template <typename Real, int NB>
__device__ __forceinline__ void ntc_sliding(Candidate<Real>& q, uint64_t seed, uint32_t gc, uint32_t s, uint32_t n,
                                               uint32_t nsel, Real* va, Real* vb, const uint8_t* perm, int grp,
                                               int gl, Real& cm, uint32_t& ncoll, uint32_t& flags) {
    constexpr int G = kGroup;
    uint32_t kb = 0;  // the candidate of the group's first lane
    while (__any_sync(kFull, kb < nsel)) {
        const bool pend = kb + (uint32_t)gl < nsel;
        uint32_t pi = 0, pj = 0;
        if (pend) pi = perm[q.i], pj = perm[q.j];
        Real* ai = va + 4 * pi;
        Real* aj = va + 4 * pj;
        Real* bi = vb + NB * pi;
        Real* bj = vb + NB * pj;
        const uint32_t si = 1u << (q.i & 31u), sj = 1u << (q.j & 31u);
        const uint32_t mlo = ((q.i & 32u) ? 0u : si) | ((q.j & 32u) ? 0u : sj);
        const uint32_t mhi = ((q.i & 32u) ? si : 0u) | ((q.j & 32u) ? sj : 0u);
        Real ax = 0, ay = 0, az = 0, bx = 0, by = 0, bz = 0, cr = 0;
        Real v = cm;
        if (pend) {
            ax = ai[0], ay = ai[1], az = bi[0];
            bx = aj[0], by = aj[1], bz = bj[0];
            const Real ddx = ax - bx, ddy = ay - by, ddz = az - bz;
            cr = sqrt(ddx * ddx + ddy * ddy + ddz * ddz);
            if (cr > cm) v = cr;
        }
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const Real t = __shfl_up_sync(kFull, v, o, G);
            if (gl >= o && above(t, v)) v = t;
        }
        const bool acc = pend && cr > q.R * v;
        const bool coll = acc && q.ok;
        uint32_t elo = coll ? mlo : 0u, ehi = coll ? mhi : 0u;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const uint32_t tl = __shfl_up_sync(kFull, elo, o, G), th = __shfl_up_sync(kFull, ehi, o, G);
            if (gl >= o) elo |= tl, ehi |= th;
        }
        // exclusive: the particles of the earlier lanes' collisions
        elo = __shfl_up_sync(kFull, elo, 1, G);
        ehi = __shfl_up_sync(kFull, ehi, 1, G);
        const bool conf = pend && gl > 0 && ((elo & mlo) | (ehi & mhi)) != 0u;
        const unsigned cb = (__ballot_sync(kFull, conf) >> (G * grp)) & ((1u << G) - 1u);
        const int cut = cb ? __ffs((int)cb) - 1 : G;
        if (pend && gl < cut) {
            if (coll) {
                const Real cx = (ax + bx) * (Real)0.5;
                const Real cy = (ay + by) * (Real)0.5;
                const Real cz = (az + bz) * (Real)0.5;
                const Real h = cr * (Real)0.5;
                const Real hx = h * q.nx, hy = h * q.ny, hz = h * q.nz;
                ai[0] = cx + hx;
                ai[1] = cy + hy;
                bi[0] = cz + hz;
                aj[0] = cx - hx;
                aj[1] = cy - hy;
                bj[0] = cz - hz;
                ncoll += 1;
            } else if (acc) {
                flags |= HYB_ST_SCATTER_CAP;
            }
        }
        cm = __shfl_sync(kFull, v, cut - 1, G);
        __syncwarp();
        // the window moves on: the unsettled candidates to the first lanes, new ones behind them
        kb += (uint32_t)cut;
        if (__any_sync(kFull, cut < G)) {
            const int from = (gl + cut) & (G - 1);
            uint32_t w = q.i | q.j << 8 | (uint32_t)q.ok << 16;  // (a bin has at most 256 slots)
            w = __shfl_sync(kFull, w, from, G);
            q.i = w & 0xFFu, q.j = (w >> 8) & 0xFFu, q.ok = (int)(w >> 16);
            q.R = __shfl_sync(kFull, q.R, from, G);
            q.nx = __shfl_sync(kFull, q.nx, from, G);
            q.ny = __shfl_sync(kFull, q.ny, from, G);
            q.nz = __shfl_sync(kFull, q.nz, from, G);
        }
        if (gl + cut >= G && kb + (uint32_t)gl < nsel) draw_candidate(q, seed, gc, s, n, kb + (uint32_t)gl);
    }
}

// The four consecutive cells from cell0 of one context, by one warp: the arrivals of half p^1
// (d*) are put in stable order, collided and sampled; MODE_COLLIDE writes them back in
// place, MODE_FUSED moves them on (step s + 1) into the bins of half p (s*), except cells
// marked in a.coupled, which are written back in place for LB2DSMC. Returns the warp's
// candidates, collisions, particles and status bits.
template <typename Real, bool Z3, int MODE>
__device__ __forceinline__ void collide_warp(const DsmcArgs<Real>& a, uint32_t pool, int cell0, unsigned char* smem,
                                             uint32_t& ncand, uint32_t& ncoll, uint32_t& nlive,
                                             uint32_t& flags) {
    constexpr int G = kGroup;
    constexpr int NB = Z3 ? 2 : 1;
    constexpr int NOFF = neighbours<Z3>();
    constexpr int RB = (int)sizeof(Real);
    const unsigned lane = lane_id();
    const int grp = (int)lane / G, gl = (int)lane % G;
    const uint32_t bin = (uint32_t)a.bin;
    const WarpMem wm = warp_mem<Real, Z3>(pool, bin);
    unsigned char* scratch = smem + wm.scratch;
    const int BW = bitmap_words<Z3>(bin);
    const int CW = (BW + G - 1) / G;
    const uint32_t lim = (uint32_t)BW * 32u;
    uint32_t* bm = reinterpret_cast<uint32_t*>(scratch) + grp * BW;
    uint32_t* fl = reinterpret_cast<uint32_t*>(scratch) + kWarpCells * BW + grp * (kFarList + 1);
    uint8_t* pf = scratch + (size_t)kWarpCells * (BW + kFarList + 1) * 4 + grp * BW;
    // after the ranks: the cell's sums, and per neighbour the particles bound for it, then the
    // first of their slots and how many of them fit
    double* sums = reinterpret_cast<double*>(scratch) + grp * kMoments;
    uint2* dest = reinterpret_cast<uint2*>(scratch + kWarpCells * kMoments * 8) + grp * NOFF;
    const uint32_t s = a.ctrl[CTRL_STEP];
    const bool do_sample = a.sample_every == 1 || (s % (uint32_t)a.sample_every) == 0u;
    uint32_t hits = 0, caps = 0, lost = 0;

    const int c = cell0 + grp;
    const bool has = c < a.ncells;
    const int64_t base = (int64_t)c * bin;
    // the channel's cell: the key of the random streams and of the stable order
    const uint32_t gc = global_cell((uint32_t)c, a.ncx, a.ncy, a.y0, a.ncy_g);
    const Real* __restrict__ drec = a.drec;
    uint32_t n_all = has ? a.count_d[c] : 0u;
    uint32_t nb0 = 0;
    Real cm0 = (Real)0, rem0 = (Real)0;
    if (has) {
        nb0 = a.nbar_sum[c];
        cm0 = a.crmax[c];
        rem0 = a.rem[c];
    }
    const bool moving = MODE == MODE_FUSED && has && !(a.coupled && a.coupled[c]);
    if (n_all > bin) n_all = bin;
    // the cells' regions of the warp's pool (exclusive sums of the counts); if they do not
    // fit, the cells take the whole pool one after another
    uint32_t off = 0, tot = 0;
#pragma unroll
    for (int q = 0; q < kWarpCells; ++q) {
        const uint32_t t = __shfl_sync(kFull, n_all, q * G);
        if (q < grp) off += t;
        tot += t;
    }
    const bool fits = tot <= pool;
    if (!fits) off = 0;
    const int rounds = fits ? 1 : kWarpCells;
    Real* va = reinterpret_cast<Real*>(smem) + 4 * off;
    Real* vb = reinterpret_cast<Real*>(smem + wm.b) + NB * off;
    uint32_t* key = reinterpret_cast<uint32_t*>(smem + wm.key) + off;
    uint8_t* perm = smem + wm.perm + off;

    for (int round = 0; round < rounds; ++round) {
        const bool act = fits || grp == round;
        const bool has_r = has && act;
        const uint32_t n = act ? n_all : 0u;
        // every loop over a cell's particles runs as often as the fullest cell of the warp needs,
        // its lanes masked: trip counts of their own would have the warp run a loop's unrolled
        // body and its remainder one after the other
        const uint32_t nmax = __reduce_max_sync(kFull, n);
        // the cell's arrivals, copied to shared memory (no registers hold them, so all of a
        // warp's loads are in flight together)
#pragma unroll 2
        for (uint32_t k0 = 0; k0 < nmax; k0 += G) {
            const uint32_t k = k0 + (uint32_t)gl;
            if (k < n) {
                const Real* r = drec + (base + k) * kRec;
                cp_async_part<16>(va + 4 * k, r);
                if constexpr (RB == 8) cp_async_part<16>(va + 4 * k + 2, r + 2);
                cp_async_part<NB * RB>(vb + NB * k, r + RS_VZ);
                cp_async_part<4>(key + k, r + RS_TAG);
            }
        }
        cp_async_commit();
        // N_cand = 1/2 N Nbar F_N (sigma c_r)_max dt / V_c + remainder, and the first eight
        // candidates, while the arrivals come in
        uint32_t nsel = 0;
        Real cm = cm0;
        if (has_r) {
            const uint32_t nb = nb0 + n;
            if (gl == 0) a.nbar_sum[c] = nb;
            if (n >= 2) {
                const Real nbar = (Real)nb / (Real)(s + 1u);
                const Real cdt = a.coll_cell ? a.coll_cell[c] : a.coll_r;
                const Real want = (Real)0.5 * (Real)n * nbar * cm0 * cdt + rem0;
                const Real fw = floor(want);
                if (gl == 0) a.rem[c] = want - fw;
                if (fw > (Real)16777215) {
                    nsel = 16777215u;
                    flags |= HYB_ST_CELL_OVERFLOW;
                } else {
                    nsel = (uint32_t)fw;
                }
            }
            if (gl == 0) {
                nlive += n;
                ncand += nsel;
            }
        }
        Candidate<Real> cand{};
        if ((uint32_t)gl < nsel) draw_candidate(cand, a.seed, gc, s, n, (uint32_t)gl);
        // A. stable order: every arrival's rank among the cell's arrivals by order key. A key
        // below W bin (a particle from a neighbouring cell) sets bit `key` of the cell's
        // bitmap, and its rank is the number of set bits below it: the count before its word
        // (a prefix over the words, kept modulo 256: a queried word holds its own bit, so
        // the count is below bin) plus those below it within the word. Larger keys follow
        // all of these, each ranked by counting the larger keys below it (from a list of the
        // cell's larger keys while they are few, else from all keys).
        for (int q0 = 0; q0 < BW; q0 += G)
            if (q0 + gl < BW) bm[q0 + gl] = 0u;
        if (gl == 0) fl[0] = 0u;
        cp_async_wait_all();
        __syncwarp();
#pragma unroll 2
        for (uint32_t k0 = 0; k0 < nmax; k0 += G) {
            const uint32_t k = k0 + (uint32_t)gl;
            if (k >= n) continue;
            const uint32_t t = key[k];
            if (t < lim) {
                atomicOr(&bm[t >> 5], 1u << (t & 31u));
            } else {
                const uint32_t j = atomicAdd(&fl[0], 1u);
                if (j < (uint32_t)kFarList) fl[1 + j] = t;
            }
        }
        __syncwarp();
        {  // the prefix counts: lane gl owns words [gl CW, gl CW + CW)
            const int q0 = gl * CW;
            uint32_t mine = 0;
            for (int i = 0; i < CW; ++i)
                if (q0 + i < BW) mine += (uint32_t)__popc(bm[q0 + i]);
            uint32_t inc = mine;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, inc, o, G);
                if (gl >= o) inc += t;
            }
            uint32_t run = inc - mine;
            for (int i = 0; i < CW; ++i)
                if (q0 + i < BW) {
                    pf[q0 + i] = (uint8_t)run;
                    run += (uint32_t)__popc(bm[q0 + i]);
                }
        }
        __syncwarp();
#pragma unroll 2
        for (uint32_t k0 = 0; k0 < nmax; k0 += G) {
            const uint32_t k = k0 + (uint32_t)gl;
            if (k >= n) continue;
            const uint32_t t = key[k];
            uint32_t rk;
            if (t < lim) {
                const uint32_t q = t >> 5;
                rk = (uint32_t)pf[q] + (uint32_t)__popc(bm[q] & ((1u << (t & 31u)) - 1u));
            } else {
                const uint32_t nfar = fl[0];
                rk = n - nfar;
                if (nfar <= (uint32_t)kFarList) {
                    for (uint32_t m2 = 0; m2 < nfar; ++m2) rk += fl[1 + m2] < t ? 1u : 0u;
                } else {
                    for (uint32_t m2 = 0; m2 < n; ++m2) rk += (key[m2] >= lim && key[m2] < t) ? 1u : 0u;
                }
            }
            perm[rk] = (uint8_t)k;
        }
        __syncwarp();
        // the ranks are taken: the cell's FP64 sums are copied over the bitmaps while the cell
        // is collided (10 x 16 bytes), and the neighbours' counts start at zero
        if (has_r && do_sample)
#pragma unroll
            for (int i = 0; i < (kMoments / 2 + G - 1) / G; ++i) {
                const int j = gl + G * i;
                if (j < kMoments / 2) cp_async16(&sums[2 * j], &a.acc[(size_t)c * kMoments + 2 * j]);
            }
        cp_async_commit();
        if constexpr (MODE == MODE_FUSED)
#pragma unroll
            for (int i = 0; i < (NOFF + G - 1) / G; ++i)
                if (gl + G * i < NOFF) dest[gl + G * i] = make_uint2(0u, 0u);
        // B. the collisions
        if constexpr (RB == 8 || MODE == MODE_COLLIDE)
            ntc_sliding<Real, NB>(cand, a.seed, gc, s, n, nsel, va + 2, vb, perm, grp, gl, cm, ncoll, flags);
        else
            ntc_collisions<Real, NB>(cand, a.seed, gc, s, n, nsel, va + 2, vb, perm, grp, gl, cm, ncoll, flags);
        if (has_r && gl == 0) a.crmax[c] = cm;
        __syncwarp();
        // C. moment sums of the collided particles; the cell is written back in place in
        // stable order (the collide, and cells the step's LB2DSMC regenerates), or moved on.
        // Every lane sums its particles gl, gl + G, gl + 2 G, ... in this order, whether in
        // the loop below (cells written back) or in the move (cells moved on), so that the
        // sums of a fused pass equal those of single steps bit for bit.
        Real mo[kMoments];
#pragma unroll
        for (int q = 0; q < kMoments; ++q) mo[q] = (Real)0;
        const uint32_t nback = has_r && !moving ? n : 0u;
        const uint32_t backmax = MODE == MODE_FUSED ? __reduce_max_sync(kFull, nback) : nmax;
#pragma unroll 1
        for (uint32_t k0 = 0; k0 < backmax; k0 += G) {
            const uint32_t k = k0 + (uint32_t)gl;
            if (k >= nback) continue;
            const uint32_t p = perm[k];
            Real px, py, ux, uy;
            get4(va + 4 * p, px, py, ux, uy);
            const Real uz = vb[NB * p];
            rec_put(a.drec, base + k, px, py, Z3 ? vb[NB * p + NB - 1] : (Real)0, ux, uy, uz, 0u);
            if (do_sample) add_moments(mo, ux, uy, uz);
        }
        // the move of step s + 1 in place in the pool: every particle takes its place among those
        // of its cell bound for the same neighbour from a shared count
        const uint32_t nm = moving && act ? n : 0u;
        constexpr int NO = (NOFF + G - 1) / G;
        uint32_t to[NO], at[NO], many[NO];
        if constexpr (MODE == MODE_FUSED) {
            const MoveCtx<Real> m = move_ctx(a);
            const Origin org = origin_of(m, gc);
            const Half<Real> dst = half_s(a);
#pragma unroll 1
            for (uint32_t k0 = 0; k0 < nmax; k0 += G) {
                const uint32_t k = k0 + (uint32_t)gl;
                if (k >= nm) continue;
                const uint32_t p = perm[k];
                Real px, py, pz = 0, ux, uy, uz = vb[NB * p];
                get4(va + 4 * p, px, py, ux, uy);
                if constexpr (Z3) pz = vb[NB * p + NB - 1];
                if (do_sample) add_moments(mo, ux, uy, uz);
                int ix, iy, iz;
                fly<Real, Z3>(m, org, k, s + 1u, px, py, pz, ux, uy, uz, hits, caps, ix, iy, iz);
                const uint32_t o = neighbour_offset<Real, Z3>(m, org, ix, iy, iz);
                if (o != kFarOffset) {
                    key[p] = (o << 16) | atomicAdd(&dest[o].x, 1u);
                    put4(va + 4 * p, px, py, ux, uy);
                    vb[NB * p] = uz;
                    if constexpr (Z3) vb[NB * p + NB - 1] = pz;
                } else {  // farther than a neighbour: put away at once
                    key[p] = 0xFFFFFFFFu;
                    const uint32_t cell = (uint32_t)((iz * a.ncy + iy) * a.ncx + ix);
                    const uint32_t arr = atomicAdd(&dst.count[cell], 1u);
                    if (arr < bin)
                        put_particle<Real, Z3>(dst, (int64_t)cell * bin + arr, order_key(m, org, k, o), px, py, pz,
                                               ux, uy, uz);
                    else
                        lost += 1;
                }
            }
            __syncwarp();
            // one reservation of slots per neighbour, all of a cell's in flight together
#pragma unroll
            for (int i = 0; i < NO; ++i) {
                const int o = gl + G * i;
                many[i] = o < NOFF && moving && act ? dest[o].x : 0u;
                to[i] = at[i] = 0u;
                if (many[i] > 0u) {
                    int x = org.x + o % 3 - 1, y = org.y + (o / 3) % 3 - 1, z = 0;
                    if (y < 0) y += m.ncy;
                    if (y >= m.ncy) y -= m.ncy;
                    if constexpr (Z3) {
                        z = org.z + o / 9 - 1;
                        if (z < 0) z += m.ncz;
                        if (z >= m.ncz) z -= m.ncz;
                    }
                    to[i] = (uint32_t)((z * m.ncy + y) * m.ncx + x);
                    at[i] = atomicAdd(&dst.count[to[i]], many[i]);
                }
            }
            // the arrivals of half p^1 are consumed: their count starts the next step's
            // arrivals (a regenerated cell's count is consumed by LB2DSMC)
            if (moving && act && gl == 0) a.count_d[c] = 0;
        }
        if (do_sample) {
            // halving exchange over the group: lane gl ends with the totals of moments
            // 3 gl, 3 gl + 1, 3 gl + 2
            Real t[24];
#pragma unroll
            for (int q = 0; q < 24; ++q) t[q] = q < kMoments ? mo[q] : (Real)0;
#pragma unroll
            for (int o = G / 2, len = 12; o >= 1; o >>= 1, len >>= 1) {
                const bool hi = (gl & o) != 0;
#pragma unroll
                for (int q = 0; q < len; ++q) {
                    const Real send = hi ? t[q] : t[q + len];
                    const Real keep = hi ? t[q + len] : t[q];
                    t[q] = keep + __shfl_xor_sync(kFull, send, o);
                }
            }
            if (gl == 0) t[0] = (Real)n;  // the particle count, moment 0
            cp_async_wait_all();
            __syncwarp();
            if (has_r) {
                // one FP64 addition per sum to the cell's sums copied in above (each sum has
                // one writer per step)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int mq = 3 * gl + q;
                    if (mq < kMoments) a.acc[(size_t)c * kMoments + mq] = sums[mq] + (double)t[q];
                }
            }
        }
        if constexpr (MODE == MODE_FUSED) {
            const Half<Real> dst = half_s(a);
#pragma unroll
            for (int i = 0; i < NO; ++i)
                if (gl + G * i < NOFF)
                    dest[gl + G * i] = make_uint2(to[i] * bin + at[i], at[i] < bin ? bin - at[i] : 0u);
            __syncwarp();
#pragma unroll 1
            for (uint32_t k0 = 0; k0 < nmax; k0 += G) {
                const uint32_t k = k0 + (uint32_t)gl;
                if (k >= nm) continue;
                const uint32_t p = perm[k], w = key[p];
                if (w != 0xFFFFFFFFu) {
                    const uint32_t o = w >> 16, r = w & 0xFFFFu;
                    const uint2 d = dest[o];
                    Real px, py, ux, uy;
                    get4(va + 4 * p, px, py, ux, uy);
                    if (r < d.y)
                        put_particle<Real, Z3>(dst, (int64_t)(d.x + r), o * bin + k, px, py,
                                               Z3 ? vb[NB * p + NB - 1] : (Real)0, ux, uy, vb[NB * p]);
                    else
                        lost += 1;
                }
            }
        }
        __syncwarp();  // the pool and the sums are reused by the next round
    }
    if constexpr (MODE == MODE_FUSED) move_events(a.counters, a.ctrl, hits, caps, lost, lane);
}

template <typename Real, bool BATCH, bool Z3 = false, int MODE = MODE_COLLIDE, int W = kCollideWarps>
__global__ void __launch_bounds__(W * 32, (CollideCfg<Real, W>::MINB))
    k_collide(Launch<DsmcArgs<Real>> L, uint32_t pool, uint32_t warp_smem) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_tot[4], s_done;
    static_assert(sizeof(s_tot) + sizeof(s_done) <= kCollideStatic, "fitting_pool counts them");
    if (threadIdx.x < 4) s_tot[threadIdx.x] = 0u;
    if (threadIdx.x == 4) s_done = 0u;
    __syncthreads();
    pdl_begin();
    const DsmcArgs<Real>* ap = &L.one;
    int blk = (int)blockIdx.x;
    if constexpr (BATCH) {
        const int r = replica_of(L.pre, L.nrep, (int64_t)blockIdx.x);
        ap = &L.tab[r];
        blk = (int)(blockIdx.x - L.pre[r]);
    }
    const DsmcArgs<Real>& a = *ap;
    const int w = threadIdx.x >> 5;
    uint32_t ncand = 0, ncoll = 0, nlive = 0, flags = 0;
    const int cell0 = (blk * W + w) * kWarpCells;
    if (cell0 < a.ncells)
        collide_warp<Real, Z3, MODE>(a, pool, cell0, smem_raw + (size_t)w * warp_smem, ncand, ncoll, nlive, flags);
    // event counters: summed over the block in shared memory; the last warp to arrive adds the
    // block's sums, one atomic per counter (no warp waits for another)
    ncand = __reduce_add_sync(kFull, ncand);
    ncoll = __reduce_add_sync(kFull, ncoll);
    nlive = __reduce_add_sync(kFull, nlive);
    flags = __reduce_or_sync(kFull, flags);
    if (lane_id() == 0) {
        atomicAdd(&s_tot[0], ncand);
        atomicAdd(&s_tot[1], ncoll);
        atomicAdd(&s_tot[2], nlive);
        atomicOr(&s_tot[3], flags);
        __threadfence_block();
        if (atomicAdd(&s_done, 1u) == (uint32_t)W - 1u) {
            __threadfence_block();
            volatile uint32_t* t = s_tot;
            if (t[0]) atomicAdd(&a.counters[HYB_C_CANDIDATES], (unsigned long long)t[0]);
            if (t[1]) atomicAdd(&a.counters[HYB_C_COLLISIONS], (unsigned long long)t[1]);
            if (t[2]) atomicAdd(&a.ctrl[CTRL_NACC], t[2]);
            if (t[3]) atomicOr(&a.ctrl[CTRL_STATUS], t[3]);
            // (the end of the step, after the pass, publishes the count and advances the step)
        }
    }
}

// The end of a DSMC step (end_of_step) after a context's collide pass. (A batch's LB step does it in a
// block of its own, which saves a launch of 4.7 us; on single contexts that gained 2% at 819k
// particles and lost 2% in 3D and on the FP64 proof of concept.)
template <typename Real>
__global__ void k_step_end(DsmcArgs<Real> a) {
    pdl_begin();
    if (threadIdx.x == 0) end_of_step(a.ctrl, (uint32_t)a.sample_every);
}

// Appends the particles a streamwise slab received from its neighbours (records and channel
// cells from the slab below, then above) to the bins of their cells in half p^1, after the
// slab's move, with their order keys; then clears the slab's own send counts for its
// next move (the caller has copied its send buffers out by then). A received cell outside the
// slab is skipped and raises HYB_ST_BAD_INPUT.
template <typename Real, bool Z3>
__global__ void __launch_bounds__(256) k_merge(DsmcArgs<Real> a) {
    pdl_begin();
    const unsigned lane = lane_id();
    const uint32_t bin = (uint32_t)a.bin;
    const Half<Real> dst = half_d(a);
    const uint32_t cap = (uint32_t)a.xcap;
    const uint32_t n0 = min(*a.rcount[0], cap), n1 = min(*a.rcount[1], cap);
    const uint32_t total = n0 + n1;
    const uint32_t nz = a.ncz ? (uint32_t)a.ncz : 1u;
    uint32_t lost = 0, bad = 0;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32 * 32;
    const int64_t wstride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = w0; i0 < (int64_t)total; i0 += wstride) {  // warp-uniform trip count
        const int64_t i = i0 + lane;
        bool loc = false;
        uint32_t key = 0, tag = 0;
        Real px = 0, py = 0, pz = 0, ux = 0, uy = 0, uz = 0;
        if (i < (int64_t)total) {
            const int d = i < (int64_t)n0 ? 0 : 1;
            const int64_t j = d ? i - n0 : i;
            rec_get(a.rrec[d], j, px, py, pz, ux, uy, uz, tag);
            const uint32_t gk = a.rkey[d][j];
            const uint32_t plane = (uint32_t)a.ncx * (uint32_t)a.ncy_g;
            const uint32_t iz = gk / plane, r = gk - iz * plane;
            const uint32_t iy = r / (uint32_t)a.ncx, ix = r - iy * (uint32_t)a.ncx;
            const int iyl = (int)iy - a.y0;
            if (iyl >= 0 && iyl < a.ncy && iz < nz) {
                key = (iz * (uint32_t)a.ncy + (uint32_t)iyl) * (uint32_t)a.ncx + ix;
                loc = true;
            } else {
                bad += 1;
            }
        }
        const uint32_t arr = bin_arrival1(dst.count, key, loc, lane);
        if (loc) {
            if (arr < bin)
                put_particle<Real, Z3>(dst, (int64_t)key * bin + arr, tag, px, py, pz, ux, uy, uz);
            else
                lost += 1;
        }
    }
    lost = __reduce_add_sync(kFull, lost);
    bad = __reduce_add_sync(kFull, bad);
    if (lane == 0 && (lost | bad))
        atomicOr(&a.ctrl[CTRL_STATUS], (lost ? HYB_ST_CAPACITY : 0u) | (bad ? HYB_ST_BAD_INPUT : 0u));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.xcount[0] = 0u;
        *a.xcount[1] = 0u;
    }
}

// Sets coupled[cells[i]] = v for the listed cells (indices out of range are skipped).
__global__ void k_mark_cells(uint8_t* coupled, const int32_t* cells, int32_t n, int64_t ncells,
                             uint8_t v) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        const int32_t c = cells[i];
        if (c >= 0 && (int64_t)c < ncells) coupled[c] = v;
    }
}

template <typename Real>
DsmcArgs<Real> make_args(Ctx& c) {
    DsmcArgs<Real> a{};
    const int h = c.cur_p, o = c.cur_p ^ 1;
    a.srec = (Real*)c.st.part[h];
    a.drec = (Real*)c.st.part[o];
    a.count_s = c.st.count[h];
    a.count_d = c.st.count[o];
    a.crmax = (Real*)c.st.crmax;
    a.rem = (Real*)c.st.rem;
    a.nbar_sum = c.st.nbar_sum;
    a.acc = c.st.acc;
    a.ctrl = c.st.ctrl;
    a.counters = c.st.counters;
    a.coupled = c.st.coupled;
    a.ncx = c.p.ncx;
    a.ncy = c.p.ncy;
    a.ncells = (int32_t)c.d.ncells;
    a.bin = c.d.bin;
    a.sample_every = c.p.sample_every;
    a.ppc = c.p.ppc;
    a.dt = c.d.dt;
    a.g_step = c.d.g_step;
    a.coll_dt = c.d.coll_dt;
    a.dt_r = (Real)c.d.dt;
    a.g_r = (Real)c.d.g_step;
    a.coll_r = (Real)c.d.coll_dt;
    a.coll_cell = (const Real*)c.st.coll_cell;
    a.ncz = c.p.ncz >= 2 ? c.p.ncz : 0;
    a.crmax_init = c.p.crmax_init;
    a.seed = c.p.seed;
    a.y0 = c.p.ncy_global > 0 ? c.p.y0 : 0;
    a.ncy_g = c.p.ncy_global > 0 ? c.p.ncy_global : c.p.ncy;
    a.xcap = (int32_t)c.d.xcap;
    for (int d = 0; d < 2; ++d) {
        char* xs = c.st.xsend[d];
        char* xr = c.st.xrecv[d];
        const size_t keys = 256 + (size_t)c.d.xcap * kRec * sizeof(Real);
        a.xcount[d] = c.d.xcap ? (uint32_t*)xs : nullptr;
        a.xrec[d] = c.d.xcap ? (Real*)(xs + 256) : nullptr;
        a.xkey[d] = c.d.xcap ? (uint32_t*)(xs + keys) : nullptr;
        a.rcount[d] = c.d.xcap ? (const uint32_t*)xr : nullptr;
        a.rrec[d] = c.d.xcap ? (const Real*)(xr + 256) : nullptr;
        a.rkey[d] = c.d.xcap ? (const uint32_t*)(xr + keys) : nullptr;
    }
    return a;
}

int grid_for(const Ctx& c, int64_t work, int threads, int per_sm) {
    int64_t g = (work + threads - 1) / threads;
    const int64_t cap = (int64_t)c.num_sms * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

template <typename Real>
cudaError_t init_impl(Ctx& c) {
    // the initial particles go to half 0: arguments built with half 1 as the source
    c.cur_p = 1;
    DsmcArgs<Real> a = make_args<Real>(c);
    c.cur_p = 0;
    const int64_t n = c.d.ncells * c.p.ppc;
    k_init_particles<Real><<<grid_for(c, n, 256, 16), 256, 0, c.stream>>>(a);
    k_init_cells<Real><<<grid_for(c, c.d.ncells, 256, 16), 256, 0, c.stream>>>(a);
    if (c.st.coupled) cudaMemsetAsync(c.st.coupled, 0, (size_t)c.d.ncells, c.stream);
    for (int d = 0; d < 2 && c.d.xcap; ++d) {  // the exchange counts start at zero
        cudaMemsetAsync(c.st.xsend[d], 0, 4, c.stream);
        cudaMemsetAsync(c.st.xrecv[d], 0, 4, c.stream);
    }
    return cudaGetLastError();
}

template <typename Real, bool Z3>
cudaError_t move_impl(Ctx& c, int p) {
    const int save = c.cur_p;
    c.cur_p = p;
    Launch<DsmcArgs<Real>> L{};
    L.one = make_args<Real>(c);
    c.cur_p = save;
    L.total = c.d.ncells;
    prof_begin(c, K_MOVE);
    // one source cell per warp (the hardware schedules the blocks as resources free up)
    const cudaError_t e = launch_pdl(k_move<Real, false, Z3>, dim3(grid_for(c, c.d.ncells * 32, 256, 64)),
                                     dim3(256), 0, c.stream, L);
    prof_end(c, K_MOVE);
    return e;
}

// Pool slots of a collide warp in a block of `warps`: as many of the wanted `pool` (collide_pool) as
// leave the block within the shared memory a block may have (limit), and at least one bin, which the
// largest bins leave room for in either shape. A smaller pool only has more warps take their cells one
// at a time. Bins of 128 to 256 slots need it: in blocks of 8 warps from 95 particles per cell on in
// FP64 3D (at a capacity factor of 2.5), 130 in FP64 2D and 183 in FP32 3D, in blocks of 4 from 223 in
// FP64 3D.
template <typename Real, bool Z3>
uint32_t fitting_pool(uint32_t pool, uint32_t bin, int warps, int limit) {
    const uint32_t per_warp = (uint32_t)((limit - kCollideStatic) / warps);
    while (pool > bin && warp_mem<Real, Z3>(pool, bin).total > per_warp) pool -= 8u;
    return pool;
}

template <typename Real, bool Z3, int MODE, int W>
cudaError_t collide_impl_w(Ctx& c, int p) {
    const int save = c.cur_p;
    c.cur_p = p;
    Launch<DsmcArgs<Real>> L{};
    L.one = make_args<Real>(c);
    c.cur_p = save;
    constexpr int NC = W * kWarpCells;
    const uint32_t pool = fitting_pool<Real, Z3>(collide_pool(c), (uint32_t)c.d.bin, W, c.smem_block);
    const uint32_t warp_smem = warp_mem<Real, Z3>(pool, (uint32_t)c.d.bin).total;
    const size_t smem = (size_t)W * warp_smem;
    // (dynamic and static shared memory together may exceed the default 48 KB)
    cudaError_t e = cudaFuncSetAttribute(k_collide<Real, false, Z3, MODE, W>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((c.d.ncells + NC - 1) / NC);
    L.total = grid;
    constexpr int kid = MODE == MODE_FUSED ? K_FUSED : K_COLLIDE;
    prof_begin(c, kid);
    e = launch_pdl(k_collide<Real, false, Z3, MODE, W>, dim3(grid), dim3(W * 32), smem, c.stream, L, pool,
                   warp_smem);
    prof_end(c, kid);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_step_end<Real>, dim3(1), dim3(32), 0, c.stream, L.one);
}

// The context's collide block shape: 8 warps (32 cells) or 4 (16 cells).
template <typename Real, bool Z3, int MODE>
cudaError_t collide_impl(Ctx& c, int p) {
    return c.collide_warps == 4 ? collide_impl_w<Real, Z3, MODE, 4>(c, p) : collide_impl_w<Real, Z3, MODE, 8>(c, p);
}

__global__ void k_debug_philox(const uint32_t* ctr, uint64_t seed, uint32_t* out, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint4 r = philox(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]),
                               (uint32_t)seed, (uint32_t)(seed >> 32));
        out[4 * i] = r.x;
        out[4 * i + 1] = r.y;
        out[4 * i + 2] = r.z;
        out[4 * i + 3] = r.w;
    }
}

}  // namespace

cudaError_t launch_lbm_init(Ctx& c);

cudaError_t launch_init(Ctx& c) {
    cudaError_t e = (c.p.real_bytes == 4) ? init_impl<float>(c) : init_impl<double>(c);
    if (e != cudaSuccess) return e;
    return launch_lbm_init(c);
}

cudaError_t launch_dsmc_move(Ctx& c, int p) {
    if (c.p.ncz >= 2) return c.p.real_bytes == 4 ? move_impl<float, true>(c, p) : move_impl<double, true>(c, p);
    return c.p.real_bytes == 4 ? move_impl<float, false>(c, p) : move_impl<double, false>(c, p);
}

cudaError_t launch_dsmc_collide(Ctx& c, int p) {
    if (c.p.ncz >= 2)
        return c.p.real_bytes == 4 ? collide_impl<float, true, MODE_COLLIDE>(c, p)
                                   : collide_impl<double, true, MODE_COLLIDE>(c, p);
    return c.p.real_bytes == 4 ? collide_impl<float, false, MODE_COLLIDE>(c, p)
                               : collide_impl<double, false, MODE_COLLIDE>(c, p);
}

cudaError_t launch_dsmc_fused(Ctx& c, int p) {
    if (c.p.ncz >= 2)
        return c.p.real_bytes == 4 ? collide_impl<float, true, MODE_FUSED>(c, p)
                                   : collide_impl<double, true, MODE_FUSED>(c, p);
    return c.p.real_bytes == 4 ? collide_impl<float, false, MODE_FUSED>(c, p)
                               : collide_impl<double, false, MODE_FUSED>(c, p);
}

cudaError_t launch_dsmc_step(Ctx& c) {
    cudaError_t e = launch_dsmc_move(c, c.cur_p);
    if (e != cudaSuccess) return e;
    return launch_dsmc_collide(c, c.cur_p);
}

namespace {
template <typename Real, bool Z3>
cudaError_t merge_impl(Ctx& c, int p) {
    const int save = c.cur_p;
    c.cur_p = p;
    const DsmcArgs<Real> a = make_args<Real>(c);
    c.cur_p = save;
    return launch_pdl(k_merge<Real, Z3>, dim3(grid_for(c, c.d.xcap * 2, 256, 4)), dim3(256), 0,
                      c.stream, a);
}
}  // namespace

cudaError_t launch_dsmc_merge(Ctx& c, int p) {
    if (!c.d.xcap) return cudaSuccess;
    if (c.p.ncz >= 2) return c.p.real_bytes == 4 ? merge_impl<float, true>(c, p) : merge_impl<double, true>(c, p);
    return c.p.real_bytes == 4 ? merge_impl<float, false>(c, p) : merge_impl<double, false>(c, p);
}

cudaError_t launch_mark_cells(Ctx& c, const int32_t* cells, int32_t n, uint8_t v) {
    if (n <= 0) return cudaSuccess;
    k_mark_cells<<<(unsigned)((n + 255) / 256), 256, 0, c.stream>>>(c.st.coupled, cells, n,
                                                                    c.d.ncells, v);
    return cudaGetLastError();
}

size_t dsmc_args_bytes(int real_bytes) {
    return real_bytes == 4 ? sizeof(DsmcArgs<float>) : sizeof(DsmcArgs<double>);
}

void dsmc_args_fill(Ctx& c, int cur_p, void* out) {
    const int save = c.cur_p;
    c.cur_p = cur_p;
    if (c.p.real_bytes == 4) {
        const DsmcArgs<float> a = make_args<float>(c);
        std::memcpy(out, &a, sizeof(a));
    } else {
        const DsmcArgs<double> a = make_args<double>(c);
        std::memcpy(out, &a, sizeof(a));
    }
    c.cur_p = save;
}

namespace {
// Blocks of a collide kernel resident per SM at `smem` bytes of dynamic shared memory (the
// kernel's limit is raised to it first, as for a launch); 0 if the query fails.
template <typename Kern>
int collide_per_sm(Kern kernel, int threads, size_t smem) {
    int per_sm = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess)
        return 0;
    return per_sm;
}
}  // namespace

// Whether the fused pass's grid fills the GPU: at least as many blocks of the context's shape as fit
// on it at once. Below that a launch is one partial wave whose time is the latency of its slowest
// block, which the fused pass lengthens (a collide and a move in one block). us a step of ten-step calls,
// two passes / fused: hybrid steps 64 x 64 cells 40.6 / 42.6, 64 x 256 (just above) 53.4 / 55.7, 128 x 512
// 153 / 128; DSMC alone 40 x 40 cells at Kn 0.02 42.8 / 34.8, 64 x 64 26.4 / 24.3, 64 x 256 35.8 / 37.9,
// 128 x 512 124 / 97. FP64 passes are faster apart at every size measured (64 x 64 hybrid 229 / 271,
// 64 x 256 376 / 433): the one line for both calls and precisions lies where FP32 hybrid steps change
// over; hyb_set_fuse and the tuner choose otherwise.
namespace {
template <typename Real, bool Z3, int W>
int fused_per_sm(const Ctx& c) {
    const uint32_t bin = (uint32_t)c.d.bin;
    const uint32_t pool = fitting_pool<Real, Z3>(collide_pool(c), bin, W, c.smem_block);
    return collide_per_sm(k_collide<Real, false, Z3, MODE_FUSED, W>, W * 32,
                          (size_t)W * warp_mem<Real, Z3>(pool, bin).total);
}
template <int W>
bool fused_fills_gpu_w(const Ctx& c) {
    constexpr int NC = W * kWarpCells;
    const bool z3 = c.p.ncz >= 2;
    const int per_sm = c.p.real_bytes == 4 ? (z3 ? fused_per_sm<float, true, W>(c) : fused_per_sm<float, false, W>(c))
                                           : (z3 ? fused_per_sm<double, true, W>(c) : fused_per_sm<double, false, W>(c));
    if (per_sm < 1) return true;
    const int64_t blocks = (c.d.ncells + NC - 1) / NC;
    return blocks >= (int64_t)per_sm * c.num_sms;
}
}  // namespace

bool dsmc_fused_fills_gpu(const Ctx& c) {
    return c.collide_warps == 4 ? fused_fills_gpu_w<4>(c) : fused_fills_gpu_w<8>(c);
}

// Pool slots a collide warp should have: its four cells' counts add up to about 4 ppc with a spread of
// sqrt(4 ppc); room for four such spreads (a warp whose cells do not fit takes the pool one
// cell at a time), and at least one full bin (what a block has room for: fitting_pool).
uint32_t collide_pool(const Ctx& c) {
    const double mean = (double)kWarpCells * c.p.ppc;
    uint32_t pool = ((uint32_t)std::ceil(mean + 4.0 * std::sqrt(mean)) + 7u) / 8u * 8u;
    if (pool > (uint32_t)(kWarpCells * c.d.bin)) pool = (uint32_t)(kWarpCells * c.d.bin);
    if (pool < (uint32_t)c.d.bin) pool = (uint32_t)c.d.bin;
    return pool;
}

namespace {

template <typename Real>
cudaError_t batch_move_impl(BatchDev& b, int cur_p) {
    Launch<DsmcArgs<Real>> L{};
    L.tab = (const DsmcArgs<Real>*)b.dsmc[cur_p];
    L.pre = b.pre_cells;
    L.nrep = b.nrep;
    L.total = b.tot_cells;
    const int64_t blocks = (b.tot_cells * 32 + b.move_block - 1) / b.move_block;
    return launch_pdl(k_move<Real, true>, dim3((unsigned)blocks), dim3(b.move_block), 0, b.stream, L);
}

template <typename Real>
cudaError_t batch_collide_impl(BatchDev& b, int cur_p) {
    Launch<DsmcArgs<Real>> L{};
    L.tab = (const DsmcArgs<Real>*)b.dsmc[cur_p];
    L.nrep = b.nrep;
    cudaError_t e;
    const int warps = b.collide_block / 32;
    const uint32_t pool = fitting_pool<Real, false>(b.pool, b.maxbin, warps, b.smem_block);
    const uint32_t warp_smem = warp_mem<Real, false>(pool, b.maxbin).total;
    const size_t smem = (size_t)warps * warp_smem;
    if (b.collide_block == 128) {  // blocks of 16 cells
        L.pre = b.pre_blocks4;
        L.total = b.tot_blocks4;
        auto k = k_collide<Real, true, false, MODE_COLLIDE, 4>;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = launch_pdl(k, dim3((unsigned)L.total), dim3(128), smem, b.stream, L, pool, warp_smem);
    } else {  // blocks of 32 cells
        L.pre = b.pre_blocks;
        L.total = b.tot_blocks;
        auto k = k_collide<Real, true, false, MODE_COLLIDE, 8>;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = launch_pdl(k, dim3((unsigned)L.total), dim3(256), smem, b.stream, L, pool, warp_smem);
    }
    return e;  // (the batch's LB step ends the DSMC step)
}

}  // namespace

cudaError_t launch_batch_move(BatchDev& b, int cur_p) {
    return b.real_bytes == 4 ? batch_move_impl<float>(b, cur_p) : batch_move_impl<double>(b, cur_p);
}

cudaError_t launch_batch_collide(BatchDev& b, int cur_p) {
    return b.real_bytes == 4 ? batch_collide_impl<float>(b, cur_p) : batch_collide_impl<double>(b, cur_p);
}

cudaError_t launch_debug_philox(const uint32_t* ctr, uint64_t seed, uint32_t* out, int64_t n,
                                cudaStream_t s) {
    int64_t g = (n + 255) / 256;
    if (g > 4096) g = 4096;
    k_debug_philox<<<(int)g, 256, 0, s>>>(ctr, seed, out, n);
    return cudaGetLastError();
}

}  // namespace hyb
