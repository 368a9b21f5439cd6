// sph_kernels.cu -- plain path: one launch per substep phase on the handle's stream
// (captured once into a CUDA graph).  The arithmetic lives in sph_device.cuh.
#include "sph_device.cuh"

// Block shape and resident blocks per SM each pass is built for (its register budget).
// Measured (us, search + sums): search in 256-thread blocks at 5 blocks per SM, 48 registers
// (6 blocks, 40 registers: coupled 1.16 M 437 against 409; 4: the same); density sums at 4
// blocks, 64 registers, with the next quad's neighbours in flight (their instances spill 12 to
// 68 bytes; 5 blocks spill more: 476 against 414; 3 blocks: 422); force in 128-thread blocks, 6
// per SM, 80 registers (spilling 16 bytes, the volume variant 100): the pass waits for its
// gathers (4 bytes of list and 40 of state a partner), which more warps hide better than loads
// issued ahead (coupled 1.16 M: 224; 5 blocks of 96 registers 233, the next two partners
// fetched ahead at 5 / 4 blocks 297 / 264, 7 blocks 227), and blocks of 256 leave a longer last
// wave (234 at 3 per SM, 252 at 4 with the spills of 64 registers).
#define SPH_DENSITY_THREADS 256
#define SPH_DENSITY_MINB 4
#define SPH_FORCE_MINB 6
#define SPH_FORCE_COOP_MINB 3
// Low-latency density pass (SPH_FLAG_LOW_LATENCY): up to kLowLatency32Max particles 32 lanes each
// that walk over the candidates, above 16 lanes that sum over the search's list.  Walking (us)
// on the dam break (12k particles) / a compact stirring tank (4.8k) / the coupled scene with 60k
// fluid (83k): G = 8: 67 / 37 / 109; G = 16: 34 / 22 / 94; G = 32: 25 / 16 / 111 (4 resident
// blocks; 3 and 2 the same).  Search and list sums: dam break 28 (32 lanes), coupled 75 (16).
#ifndef SPH_LOW_LATENCY_MINB
#define SPH_LOW_LATENCY_MINB 4
#endif
constexpr int kLowLatency32Max = 20000;

namespace sphgb {

__global__ void __launch_bounds__(kTile) k_hash(SimConst c)
{
    chain_enter();
    hash_item(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_scan_tiles(SimConst c)
{
    chain_enter();
    scan_tiles_item(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_scan_apply(SimConst c)
{
    chain_enter();
    scan_apply_item(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_scan_lookback(SimConst c)
{
    chain_enter();
    scan_lookback_item(c);
}
// the substep's scan: single-pass (one launch; timed as the tile pass, the apply pass reads
// ~0) unless built with SPH_SCAN_LOOKBACK=0
#ifndef SPH_SCAN_LOOKBACK
#define SPH_SCAN_LOOKBACK 1
#endif
__global__ void __launch_bounds__(kTile) k_scatter(SimConst c)
{
    chain_enter();
    scatter_item(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_rank_gather(SimConst c)
{
    chain_enter();
    rank_gather_item(c, blockIdx.x);
}
template <int COOP, int MODE>
__global__ void __launch_bounds__(SPH_DENSITY_THREADS, SPH_DENSITY_MINB) k_density(SimConst c)
{
    chain_enter();
    density_item<SPH_DENSITY_THREADS, COOP, MODE, true, ReadOnly>(c, blockIdx.x);
}
#define SPH_SEARCH_THREADS 256
#define SPH_SEARCH_MINB 5
template <int COOP>
__global__ void __launch_bounds__(SPH_SEARCH_THREADS, SPH_SEARCH_MINB) k_search(SimConst c)
{
    chain_enter();
    search_item<SPH_SEARCH_THREADS, COOP, ReadOnly>(c, blockIdx.x);
}
template <int G>
__global__ void __launch_bounds__(kTile, SPH_LOW_LATENCY_MINB) k_density_walk(SimConst c)
{
    chain_enter();
    density_walk_item<G>(c, blockIdx.x);
}
template <int G>
__global__ void __launch_bounds__(kTile, SPH_LOW_LATENCY_MINB) k_density_lanes(SimConst c)
{
    chain_enter();
    density_lanes_item<G>(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_boundary_volume(SimConst c)
{
    chain_enter();
    boundary_volume_item<ReadOnly>(c, blockIdx.x);
}
template <bool VOL>
__global__ void __launch_bounds__(kForceThreads, SPH_FORCE_MINB) k_force(SimConst c)
{
    chain_enter();
    force_item_v<kForceThreads, VOL, ReadOnly>(c, blockIdx.x);
}
template <int G>
__global__ void __launch_bounds__(kTile, SPH_FORCE_COOP_MINB) k_force_coop(SimConst c)
{
    chain_enter();
    force_coop_item<G>(c, blockIdx.x);
}
template <int G>
__global__ void __launch_bounds__(kTile, SPH_FORCE_COOP_MINB) k_force_shares(SimConst c)
{
    chain_enter();
    force_shares_item<G>(c, blockIdx.x);
}
template <int G>
__global__ void __launch_bounds__(kTile, SPH_FORCE_COOP_MINB) k_force_ordered(SimConst c)
{
    chain_enter();
    force_ordered_item<G>(c, blockIdx.x);
}
__global__ void __launch_bounds__(kTile) k_wrench(SimConst c)
{
    chain_enter();
    wrench_item(c, blockIdx.x);
}
// the last substep of an update cycle: the cycle's end (the rolling-average log) in the
// block that finished the wrench, after its sums (the same values k_cycle_end would read)
__global__ void __launch_bounds__(kTile) k_wrench_cycle(SimConst c)
{
    chain_enter();
    if (wrench_item(c, blockIdx.x) && threadIdx.x == 0) cycle_end_item(c);
}
__global__ void k_cycle_end(SimConst c) { cycle_end_item(c); }

__device__ __forceinline__ void set_grab(const SimConst &c, int body, int grab, const float (&pv)[13],
                                         const float (&gl)[3], int set_pose, int path_n)
{
    for (int b = 0; b < c.nb; ++b) {
        DevBody &B = c.body[b];
        if (b != body) {
            if (grab) B.grabbed = 0;        // one grabbed body at a time
            continue;
        }
        B.grabbed = grab;
        if (!grab) { B.path_n = 0; continue; }
        for (int a = 0; a < 3; ++a) B.grab_local[a] = gl[a];
        if (set_pose) {
            for (int a = 0; a < 3; ++a) { B.t[a] = pv[a]; B.v[a] = pv[7 + a]; B.w[a] = pv[10 + a]; }
            for (int a = 0; a < 4; ++a) B.q[a] = pv[3 + a];
        }
        B.path_n = path_n;
        B.path_step0 = (int)c.ctr[0];
    }
}

__global__ void k_set_grab(SimConst c, int body, int grab, float pv0, float pv1, float pv2,
                           float pv3, float pv4, float pv5, float pv6, float pv7, float pv8,
                           float pv9, float pv10, float pv11, float pv12, float g0, float g1,
                           float g2, int set_pose, int path_n)
{
    const float pv[13] = {pv0, pv1, pv2, pv3, pv4, pv5, pv6, pv7, pv8, pv9, pv10, pv11, pv12};
    const float gl[3] = {g0, g1, g2};
    set_grab(c, body, grab, pv, gl, set_pose, path_n);
}

// A haptic cycle's two ends, in its graph: the pose comes from the slot in pinned memory, and the
// block that finishes the wrench writes it there with the status words.  As launches and copies
// of their own around the substep's graph the three took some 14 us of a cycle's ~100.
__global__ void k_haptic_pose(SimConst c, const HapticSlot *slot)
{
    chain_enter();
    float pv[13];
    for (int a = 0; a < 13; ++a) pv[a] = slot->pose_vel[a];
    const float gl[3] = {0.0f, 0.0f, 0.0f};
    set_grab(c, slot->body, 1, pv, gl, 1, 0);
}
__global__ void __launch_bounds__(kTile) k_wrench_haptic(SimConst c, HapticSlot *slot)
{
    chain_enter();
    if (!wrench_item(c, blockIdx.x)) return;
    if (threadIdx.x == 0) cycle_end_item(c);
    if (threadIdx.x < 6) slot->wrench[threadIdx.x] = c.wrench[6 * slot->body + threadIdx.x];
    else if (threadIdx.x < 9) slot->status[threadIdx.x - 6] = c.status[threadIdx.x - 6];
}

// Cell key and id of each sorted slot (test hook): recomputed from the sorted positions.
__global__ void k_sorted_keys(SimConst c, uint32_t *keys, int *ids)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= c.n) return;
    uint32_t bad = 0;
    int cx, cy, cz;
    cell_of(c, c.xA[p], cx, cy, cz, bad);
    keys[p] = (uint32_t)((cz * c.ny + cy) * c.nx + cx);
    ids[p] = __float_as_int(c.vA[p].w);
}

// The state in id order for the caller (one thread per slot; the scattered stores stay in L2).
// A host loop over the slots, after copies of 40 bytes a particle into buffers of its own, took
// most of a read.  With this kernel and the pages of the caller's arrays populated ahead of the
// copies (sph_get_state), together: 32 substeps of the 365k stirring tank and a read 11.2 ms, now
// 9.4; 100 of the 1.16 M coupled scene 72.3 ms, now 66.0.
__global__ void __launch_bounds__(kTile) k_state(SimConst c, StateOut o)
{
    const int p = blockIdx.x * kTile + threadIdx.x;
    if (p < 3) o.bad[1 + p] = c.status[p];
    if (p >= c.n) return;
    const float4 v = c.vB[p];
    const int id = __float_as_int(v.w);
    if ((unsigned)id >= (unsigned)c.n) {
        atomicOr(o.bad, 1u);
        return;
    }
    auto put3 = [&](float *d, float4 q) {
        d[3 * (size_t)id] = q.x;
        d[3 * (size_t)id + 1] = q.y;
        d[3 * (size_t)id + 2] = q.z;
    };
    if (o.x) put3(o.x, c.xB[p]);
    if (o.v) put3(o.v, v);
    if (o.rho) o.rho[id] = c.prho[p].x;
    if (o.nnbr) o.nnbr[id] = c.nnbr[p];
    if (o.acc) put3(o.acc, c.acc_dbg[p]);
}

// ----------------------------------------------------------------------- launchers

// Who walks with cooperating lanes (same results either way; us).  Lanes shorten the chain of a
// particle alone in its lane, a rigid one's ~226 neighbours above all, and cost work: a scene alone
// gains while it leaves the GPU room, scenes stepped side by side on their own streams pay.
//   3: every particle, 16 lanes, in scenes of up to 30,000.  Search and density sum of the dam break
//     (12k particles) 31 (8 lanes 41, 32 lanes 38) against 112 with one thread each.
//   2: rigid particles, 8 lanes, up to 60,000.  Whole substep with 3 / 2, alone and per substep of
//     8 scenes side by side: 22k coupled 92 / 103 and 321 / 206, 27k stirring 95 / 101 and 384 /
//     227, 30k coupled 99 / 103 and 398 / 216, 33k stirring 104 / 97 and 463 / 256; alone 42k coupled
//     108 / 102, 40k, 52k and 58k stirring 109 / 99, 128 / 114 and 135 / 117.  One thread each: 30k
//     coupled 214 and 301, 33k stirring 180 and 285 (that walk from before the search and the sums
//     were split).  Below 30,000 a scene alone counts; 64 scenes or more of a few thousand particles
//     take longer side by side than one thread each did (256 of 6.5k to 17k: 5.2 ms for 2.7 a
//     substep), and 2.2 in a batch, which walks with one thread each.
//   1: rigid particles, 4 lanes, up to 900,000: 307k of the coupled scene 103 against 159 (search and
//     sum), the 365k stirring tank (18.7k of them rigid) 156 against 184; 2 lanes 161 / 160, 8 lanes
//     108 / 166.
//   0: nobody else.
// Around 1's two lines (whole substep, 4 lanes / one thread).  Coupled scene from its fill,
// 30k / 7k rigid particles: 0.5 M particles 359 / 387 and 274 / 333, 0.8 M 487 / 495 and 401 /
// 440, 0.98 M 544 / 551 and 465 / 488, 1.15 M 619 / 621 and 544 / 559; from its stirred state the
// 1.16 M scene's search and sums took 389 / 385.  So 900,000 lies where the gain runs out for a
// large body, early for a small one.  Share of rigid particles: 12 % 155 / 225 (130k), 16 % 349 /
// 390, 24 % 440 / 464 and 224 / 259, 38 % 646 / 687, 55 % 1090 / 1058 (656k): the lanes pay well
// beyond an eighth, which is on the safe side of where they cross.
constexpr int kCoopAllMax = 30000, kCoopEightMax = 60000, kCoopRigidMax = 900000;
int walk_coop(const SimConst &c)
{
    if (c.Rc >= 2.5f) return 0;                 // the cooperative search's row table
    if (c.n <= kCoopEightMax) return c.n <= kCoopAllMax ? 3 : 2;
    return c.n <= kCoopRigidMax && c.n_rigid <= c.n / 8 ? 1 : 0;
}

static bool force_low_latency(const SimConst &c) { return (c.flags & FLAG_LOW_LATENCY) && !(c.flags & FLAG_VOLUME); }
static bool force_ordered(const SimConst &c)
{
    return c.coop == 3 && c.n <= kForceOrderedMax && !(c.flags & (FLAG_VOLUME | FLAG_LOW_LATENCY));
}
int force_blocks(const SimConst &c)
{
    const int per = force_low_latency(c) ? (c.n <= kLowLatency32Max ? 1 : 2) * kTile / kLowLatencyForceG
                    : force_ordered(c) ? kTile / kForceOrderedG : kForceThreads;
    return (c.n + per - 1) / per;
}

static inline int blocks_for(int n, int t) { return (n + t - 1) / t; }

cudaError_t launch_substep(const SimConst &c, cudaStream_t s, cudaEvent_t *ev, bool external,
                           bool cycle_end, unsigned ev_mask, HapticSlot *slot)
{
    const int nb = blocks_for(c.n, 256);
    // The short passes are put on the GPU while the pass before them ends; the long ones start
    // afterwards: early, their first blocks, the longest, would fill whichever SMs came free first.
    bool early = s != nullptr;            // (a kernel behind an event waits for the event)
    cudaError_t err = cudaSuccess;
    auto go = [&](void (*kernel)(SimConst), unsigned grid, unsigned threads, bool is_short) {
        if (err == cudaSuccess) err = launch_after(early && is_short, kernel, grid, threads, 0, s, c);
        early = s != nullptr;
    };
    int k = 0;
    auto mark = [&]() {
        if (ev && (ev_mask >> k & 1u)) {
            cudaEventRecordWithFlags(ev[k], s, external ? cudaEventRecordExternal : 0);
            early = false;
        }
        ++k;
    };
    if (slot) err = launch_after(false, k_haptic_pose, 1, 1, 0, s, c, slot);
    mark();
    go(k_hash, nb, kTile, true);
    mark();
    if (SPH_SCAN_LOOKBACK) {
        go(k_scan_lookback, c.n_scan_tiles, kTile, true);
        mark();
    } else {
        go(k_scan_tiles, c.n_scan_tiles, kTile, true);
        mark();
        go(k_scan_apply, c.n_scan_tiles, kTile, true);
    }
    mark();
    go(k_scatter, nb, kTile, true);
    mark();
    go(k_rank_gather, nb, kTile, true);
    mark();
    // the neighbour search and the sums over its lists (timed together); the volume variant's
    // boundary weights between them.  The low-latency pass's walk has rows for Rc < 2.5 (cells >= h
    // give Rc ~ 2)
    const bool lanes = force_low_latency(c) && c.Rc < 2.5f, walk = lanes && c.n <= kLowLatency32Max;
    const auto search = c.coop == 0 ? k_search<0> : c.coop == 1 ? k_search<1> : c.coop == 2 ? k_search<2> : k_search<3>;
    if (!walk) go(search, search_tiles(c, SPH_SEARCH_THREADS), SPH_SEARCH_THREADS, false);
    if (walk) {
        go(k_density_walk<32>, (unsigned)tiles_of(c.n, 32, kTile), kTile, false);
    } else if (lanes) {
        go(k_density_lanes<16>, (unsigned)tiles_of(c.n, 16, kTile), kTile, false);
    } else {
        const bool vol = (c.flags & FLAG_VOLUME) != 0;
        if (vol && c.n > c.nf) go(k_boundary_volume, blocks_for(c.n - c.nf, kTile), kTile, false);
        const auto of_mass = c.coop == 0 ? k_density<0, DENSITY_MASS> : c.coop == 1 ? k_density<1, DENSITY_MASS>
                             : c.coop == 2 ? k_density<2, DENSITY_MASS> : k_density<3, DENSITY_MASS>;
        const auto of_volume = c.coop == 0 ? k_density<0, DENSITY_VOLUME> : c.coop == 1 ? k_density<1, DENSITY_VOLUME>
                               : c.coop == 2 ? k_density<2, DENSITY_VOLUME> : k_density<3, DENSITY_VOLUME>;
        const auto density = vol ? of_volume : of_mass;
        go(density, density_tiles(c, SPH_DENSITY_THREADS), SPH_DENSITY_THREADS, false);
    }
    mark();
    if (force_low_latency(c))
        go(c.n <= kLowLatency32Max ? k_force_coop<kLowLatencyForceG> : k_force_shares<kLowLatencyForceG>,
           c.n_force_blocks, kTile, false);
    else if (force_ordered(c))
        go(k_force_ordered<kForceOrderedG>, c.n_force_blocks, kTile, false);
    else if (c.flags & FLAG_VOLUME)
        go(k_force<true>, c.n_force_blocks, kForceThreads, false);
    else
        go(k_force<false>, c.n_force_blocks, kForceThreads, false);
    mark();
    if (slot && err == cudaSuccess) err = launch_after(early, k_wrench_haptic, c.n_wgrid, kTile, 0, s, c, slot);
    else if (cycle_end) go(k_wrench_cycle, c.n_wgrid, kTile, true);
    else go(k_wrench, c.n_wgrid, kTile, true);
    mark();
    const cudaError_t last = cudaGetLastError();
    return err != cudaSuccess ? err : last;
}

__global__ void __launch_bounds__(kTile) k_cut(SimConst c, Blade t, unsigned *count)
{
    cut_item(c, blockIdx.x, t, count);
}

cudaError_t launch_cut(const SimConst &c, cudaStream_t s, const float tri[9], unsigned *count)
{
    Blade t;
    for (int i = 0; i < 9; ++i) t.v[i] = tri[i];
    const int nbody = c.n - c.nf;
    if (nbody <= 0) return cudaSuccess;
    const cudaError_t e = launch_sort(c, s);          // sorted current state + slot_of_id
    if (e != cudaSuccess) return e;
    k_cut<<<blocks_for(nbody, 256), kTile, 0, s>>>(c, t, count);
    return cudaGetLastError();
}

cudaError_t launch_sort(const SimConst &c, cudaStream_t s)
{
    const int nb = blocks_for(c.n, 256);
    k_hash<<<nb, kTile, 0, s>>>(c);
    k_scan_tiles<<<c.n_scan_tiles, kTile, 0, s>>>(c);
    k_scan_apply<<<c.n_scan_tiles, kTile, 0, s>>>(c);
    k_scatter<<<nb, kTile, 0, s>>>(c);
    k_rank_gather<<<nb, kTile, 0, s>>>(c);
    return cudaGetLastError();
}

cudaError_t launch_state(const SimConst &c, cudaStream_t s, const StateOut &o)
{
    k_state<<<blocks_for(c.n, kTile), kTile, 0, s>>>(c, o);
    return cudaGetLastError();
}

cudaError_t launch_cycle_end(const SimConst &c, cudaStream_t s)
{
    k_cycle_end<<<1, 1, 0, s>>>(c);
    return cudaGetLastError();
}

cudaError_t launch_set_grab(const SimConst &c, cudaStream_t s, int body, int grab,
                            const float *pv, const float *gl, int set_pose, int path_n)
{
    k_set_grab<<<1, 1, 0, s>>>(c, body, grab, pv[0], pv[1], pv[2], pv[3], pv[4], pv[5], pv[6],
                               pv[7], pv[8], pv[9], pv[10], pv[11], pv[12], gl[0], gl[1], gl[2],
                               set_pose, path_n);
    return cudaGetLastError();
}

cudaError_t launch_sorted_keys(const SimConst &c, cudaStream_t s, uint32_t *keys, int *ids)
{
    k_sorted_keys<<<blocks_for(c.n, 256), 256, 0, s>>>(c, keys, ids);
    return cudaGetLastError();
}

}  // namespace sphgb
