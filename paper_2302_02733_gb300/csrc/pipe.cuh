// The batched form: geodesics and transfers of many images in one persistent launch.
//
// Some warps integrate backward geodesics and save the states, the others walk completed paths toward
// the camera and do the transfer, FP64 or FP32 (the paper's Section 2.1).
//
// In the FP64 form each 8-warp block holds both roles, geo_warps of them the first: the transfer
// lives on the FP64 pipe, the geodesic on the integer pipes, and they share the SM.
//
// In the mixed form both live on the same pipes, and their loops together do not fit in the instruction
// cache: a step took 85,000 clocks where the geodesic alone takes 13,900. There the roles go to pairs
// of SMs (which share that cache), geo_warps of every 8 pairs the geodesic, handed out in the order in
// which the pairs' first blocks start, the first two one each. Geodesic warps that find no more rays
// transfer what is left, and one warp of each such pair is kept for the transfer should the pool run
// dry, so that the launch needs no other SM to end. Six mixed images of 128^2 to 512^2 take 163 ms at
// their best shape, 96 images 2.9 s (297 ms and 5.4 s with both roles in each block, 230 ms with a role to
// each SM, 167 ms and 3.7 s with a warp kept in every block; 197 ms and 3.4 s when the geodesic was
// FP64), and 86 ms and 1.5 s as one ray space in two kernels (mode 1).
//
// Flow control, all in global memory:
//  - rays come from a queue (geo_next) over all images of the batch;
//  - path blocks come from a free ring, so memory is bounded by the pool, not by the batch. A
//    lane that needs a block takes a ticket (a ring position) and polls only that slot, so
//    blocks are handed out first come, first served and waiting lanes touch no shared counter;
//  - a completed ray is published in a ready list (ready_tail) that the transfer warps
//    consume in order (xfer_next).
// Every wait is bounded, by the global nanosecond timer (sleeps are only hints) or by a poll
// count. A geodesic lane whose block has not come for kPoolStallNs gives its ray up as an
// arena overflow and frees the ray's blocks, so in-flight paths cannot deadlock the pool; it
// keeps its ticket and returns that block when it comes. A transfer lane that waits
// kReadyWaitNs for its ray, a ticket still open after kReadyWaitNs, or a ring slot that stays
// unchanged for kRingSpin polls sets an error bit that the host reports.
#pragma once
#include "geodesic.cuh"
#include "transfer_kernel.cuh"

namespace prt {

constexpr int kRingSpin = 1 << 22;
constexpr unsigned long long kPoolStallNs = 1000000000ull;   // 1 s without a free block
constexpr unsigned long long kReadyWaitNs = 30000000000ull;  // 30 s without the awaited ray

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Return a block to the ring at the next tail position. The slot is written only once the
// ticket of the previous lap has taken its value (that ticket exists: the ring never holds
// more than nblocks free blocks), and only after this lane's accesses to the block.
__device__ __forceinline__ int pool_free(const Pool &P, PipeCounters *c, int b) {
    unsigned long long pos = atomicAdd(&c->pool_tail, 1ull);
    volatile int *slot = P.ring + (pos % (unsigned long long)P.nblocks);
    int spin = 0;
    while (*slot >= 0) {
        if (++spin > kRingSpin) {
            atomicOr(&c->err, kPipeErrRing);
            return spin;
        }
    }
    __threadfence();
    *slot = b;
    return spin;
}

// Free every block of a ray from its current block back to the first (own writes only).
__device__ __forceinline__ int pool_free_chain(const Pool &P, PipeCounters *c, int blk) {
    int spins = 0;
    while (blk >= 0) {
        int pb = P.prev[blk];
        spins += pool_free(P, c, blk);
        blk = pb;
    }
    return spins;
}

__device__ __forceinline__ void save_state(const Pool &P, int blk, int slot, const double y[7], double h) {
    double4_32a *d = reinterpret_cast<double4_32a *>(P.states + (long long)blk * kBlockStates + slot);
    d[0] = make_double4_32a(y[0], y[1], y[2], y[3] - y[4]);  // K^t = W - K^r
    d[1] = make_double4_32a(y[4], y[5], y[6], h);
}

// Loads of data written by other SMs during this launch bypass L1 (a reused block may still
// sit in this SM's L1 from its previous ray).
__device__ __forceinline__ double4_32a load_cg(const double4_32a *p) {
    const double2 *q = reinterpret_cast<const double2 *>(p);
    double2 a = __ldcg(q), b = __ldcg(q + 1);
    return make_double4_32a(a.x, a.y, b.x, b.y);
}

// Publish a finished ray (record and path written before) to the transfer warps.
__device__ __forceinline__ void publish(const PipeArgs &p, long long ray, const RayRecord &rec) {
    p.rec[ray] = rec;
    __threadfence();
    unsigned long long pos = atomicAdd(&p.ctr->ready_tail, 1ull);
    atomicExch(p.ready + pos, (int)ray);
}

__device__ __forceinline__ void pipe_geodesic(const PipeArgs &p, const GeoTabs &tabs) {
    const unsigned long long nb = (unsigned long long)p.pool.nblocks;
    double y[7];
    StepCam sc{};  // the current ray's camera constants
    long long ray = -1, tk = -1;  // tk: pool ticket whose block has not come yet
    int job = 0, n = 0, blk = -1, slot = 0;
    bool live = false, drained = false, cancel = false;
    unsigned long long my_steps = 0, t0 = 0;
    unsigned long long n_iter = 0, n_sleep = 0, n_tpoll = 0, n_spin = 0, n_tick = 0;
    unsigned backoff = 256;
    for (;;) {
        n_iter++;
        bool want = !live && !drained && tk < 0;
        unsigned long long t = warp_pop(&p.ctr->geo_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ray = (long long)t;
                job = find_job(p.jobs, p.njobs, ray);
                const Camera &c = p.jobs[job].cam;
                int ix, iy;
                ray_pixel(ray - p.jobs[job].ray_begin, c.nx, c.ny, ix, iy);
                ray_start(c, ix, iy, y);
                sc = step_cam(c);
                n = 0;
                blk = -1;
                slot = kBlockStates;
                live = true;
            } else {
                drained = true;
            }
        }
        if (__all_sync(0xffffffffu, !live && drained && tk < 0)) break;
        // a ticket for a block when the current one cannot take the two states of a step
        bool ask = live && tk < 0 && slot > kBlockStates - 2;
        unsigned long long pos = warp_pop(&p.ctr->pool_head, ask);
        if (ask) {
            tk = (long long)pos;
            t0 = global_ns();
            n_tick++;
        }
        bool go = live && tk < 0;
        if (tk >= 0) {
            volatile int *sl = p.pool.ring + ((unsigned long long)tk % nb);
            int b = *sl;
            if (b >= 0) {
                *sl = -1;
                tk = -1;
                if (cancel) {  // the ray was given up: return the late block
                    n_spin += pool_free(p.pool, p.ctr, b);
                    cancel = false;
                } else {
                    if (blk >= 0) p.pool.fill[blk] = slot;
                    p.pool.prev[b] = blk;
                    blk = b;
                    slot = 0;
                    go = true;
                }
            } else if (!cancel && global_ns() - t0 > kPoolStallNs) {
                // no block for too long: give the ray up as an overflow, keep the ticket
                n_spin += pool_free_chain(p.pool, p.ctr, blk);
                RayRecord rec = {-1, 0, kOverflow, 0};
                publish(p, ray, rec);
                atomicAdd(&p.ctr->n_status[kOverflow], 1u);
                my_steps += (unsigned long long)n;
                live = false;
                cancel = true;
                t0 = global_ns();
            } else if (cancel && global_ns() - t0 > kReadyWaitNs) {
                atomicOr(&p.ctr->err, kPipeErrRing);
                tk = -1;
                cancel = false;
            }
            if (tk >= 0) n_tpoll++;
        }
        if (__all_sync(0xffffffffu, !go)) {  // nothing to step in this warp: wait a little
            if (__any_sync(0xffffffffu, live || tk >= 0)) {
                n_sleep++;
                __nanosleep(backoff);
                backoff = min(2u * backoff, 8192u);
            }
            continue;
        }
        backoff = 256;
        if (!go) continue;
        uint8_t status = 0;
        for (int k = 0; k < p.step_tile; k++) {
            double h, yn[7];
            bool refl = geo_step(tabs, sc, y, yn, h);
            save_state(p.pool, blk, slot, y, refl ? -h : h);
            slot++;
            n++;
#pragma unroll
            for (int i = 0; i < 7; i++) y[i] = yn[i];
            status = geo_stop(sc, y, n);
            if (status || slot > kBlockStates - 2) break;
        }
        if (status) {
            save_state(p.pool, blk, slot, y, 0.0);
            slot++;
            my_steps += (unsigned long long)n;
            RayRecord rec;
            if (status == kNan) {
                n_spin += pool_free_chain(p.pool, p.ctr, blk);
                rec = RayRecord{-1, 0, kNan, 0};
            } else {
                p.pool.fill[blk] = slot;
                rec = RayRecord{blk, n + 1, status, slot};
            }
            publish(p, ray, rec);
            atomicAdd(&p.ctr->n_status[status], 1u);
            live = false;
        }
    }
    if (my_steps) atomicAdd(&p.ctr->steps, my_steps);
    atomicAdd(&p.ctr->geo_iters, n_iter);
    if (n_sleep) atomicAdd(&p.ctr->geo_sleeps, n_sleep);
    if (n_tpoll) atomicAdd(&p.ctr->ticket_polls, n_tpoll);
    if (n_spin) atomicAdd(&p.ctr->free_spins, n_spin);
    if (n_tick) atomicAdd(&p.ctr->tickets, n_tick);
}

template <typename R, typename OutT>
__device__ __forceinline__ void pipe_transfer(const PipeArgs &p, const R *sgw) {
    long long ray = -1;
    int job = 0, blk = -1, slot = 0, n = 0, rstat = 0;
    unsigned long long ticket = 0, wait_t0 = 0;
    bool live = false, pending = false, drained = false;
    XLane<R> Ln;
    unsigned long long my_pts = 0, my_emit = 0;
    unsigned long long n_iter = 0, n_sleep = 0, n_rpoll = 0, n_spin = 0;
    unsigned backoff = 256;
    for (;;) {
        n_iter++;
        bool want = !live && !pending && !drained;
        unsigned long long t = warp_pop(&p.ctr->xfer_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ticket = t;
                pending = true;
                wait_t0 = global_ns();
            } else {
                drained = true;
            }
        }
        if (pending) {
            int v = *reinterpret_cast<volatile int *>(p.ready + ticket);
            if (v >= 0) {
                __threadfence();
                pending = false;
                ray = v;
                job = find_job(p.jobs, p.njobs, ray);
                int4 rr = __ldcg(reinterpret_cast<const int4 *>(p.rec + ray));
                rstat = rr.z;
                if (rr.y >= 2) {
                    blk = rr.x;
                    slot = rr.w - 1;
                    n = rr.y - 1;
                    Ln.reset();
                    live = true;
                } else {
                    const JobDev &J = p.jobs[job];
                    int ix, iy;
                    ray_pixel(ray - J.ray_begin, J.cam.nx, J.cam.ny, ix, iy);
                    long long pix = (long long)iy * J.cam.nx + ix;
                    xfer_zero<OutT>(pix, J.out, J.depth);
                    if (J.status) J.status[pix] = (uint8_t)rstat;
                }
            } else if (global_ns() - wait_t0 > kReadyWaitNs) {
                atomicOr(&p.ctr->err, kPipeErrReady);
                pending = false;
                drained = true;
            } else {
                n_rpoll++;
            }
        }
        if (__all_sync(0xffffffffu, !live && !pending && drained)) break;
        if (!__any_sync(0xffffffffu, live)) {  // the whole warp waits for rays: back off
            n_sleep++;
            __nanosleep(backoff);
            backoff = min(2u * backoff, 32768u);
            continue;
        }
        backoff = 256;
        if (!live) continue;

        // move from state n to state n-1, returning each block once it is passed
        if (--slot < 0) {
            int pb = __ldcg(p.pool.prev + blk);
            n_spin += pool_free(p.pool, p.ctr, blk);
            blk = pb;
            slot = __ldcg(p.pool.fill + blk) - 1;
        }
        n--;
        const JobDev &J = p.jobs[job];
        const double4_32a *src = reinterpret_cast<const double4_32a *>(p.pool.states + (long long)blk * kBlockStates + slot);
        double4_32a q0 = load_cg(src), q1 = load_cg(src + 1);
        KS<R> m;
        if (xfer_point(J.cam, J.model, q0, q1, sgw, Ln, m)) my_emit++;
        my_pts++;
        if (n == 0) {
            int ix, iy;
            ray_pixel(ray - J.ray_begin, J.cam.nx, J.cam.ny, ix, iy);
            xfer_finish<R, OutT>(J.cam, m, ix, iy, Ln, J.out, J.depth);
            if (J.status) J.status[(long long)iy * J.cam.nx + ix] = (uint8_t)rstat;
            n_spin += pool_free(p.pool, p.ctr, blk);
            live = false;
        }
    }
    if (my_pts) atomicAdd(&p.ctr->points, my_pts);
    if (my_emit) atomicAdd(&p.ctr->emitting, my_emit);
    atomicAdd(&p.ctr->xfer_iters, n_iter);
    if (n_sleep) atomicAdd(&p.ctr->xfer_sleeps, n_sleep);
    if (n_rpoll) atomicAdd(&p.ctr->ready_polls, n_rpoll);
    if (n_spin) atomicAdd(&p.ctr->free_spins, n_spin);
}

// Mixed form: how many of this block's warps integrate geodesics: none where its SM's pair transfers, else
// all, but one in the block that the pair's role was chosen for (one thread of the block asks).
__device__ __forceinline__ int pair_role(const PipeArgs &p) {
    unsigned sm;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
    unsigned *slot = p.ctr->role + (sm >> 1) % kRolePairs;
    unsigned v = atomicCAS(slot, 0u, 1u);
    const int geo = kPipeThreads / 32 - (v == 0u);
    if (v == 0u) {  // of 16 pairs in turn: the first, and g of the 14 after the second
        const unsigned k = atomicAdd(&p.ctr->role_next, 1u) & 15u, g = (unsigned)(p.geo_warps + p.geo_warps_odd) - 1u;
        v = k == 0u || (k > 1u && (k - 1u) * g / 14u != (k - 2u) * g / 14u) ? 2u : 3u;
        atomicExch(slot, v);
    }
    // the block that chooses is between two instructions; a wait that runs out leaves the transfer
    for (int spin = 0; v == 1u && spin < kRingSpin; spin++) v = atomicAdd(slot, 0u);
    return v == 2u ? geo : 0;
}

// Mixed form, the warp left over in a geodesic pair: asleep until every ray is taken, or a lane waits for a path
// block (more tickets than returns), or for kReadyWaitNs.
__device__ __forceinline__ void pipe_reserve(const PipeArgs &p) {
    const unsigned long long t0 = global_ns();
    volatile unsigned long long *next = &p.ctr->geo_next, *head = &p.ctr->pool_head, *tail = &p.ctr->pool_tail;
    for (;;) {
        int go = 0;
        if ((threadIdx.x & 31) == 0) go = *next >= (unsigned long long)p.nrays || *head > *tail || global_ns() - t0 > kReadyWaitNs;
        if (__shfl_sync(0xffffffffu, go, 0)) break;
        __nanosleep(20000);
    }
}

template <typename R, typename OutT>
__global__ void __launch_bounds__(kPipeThreads, sizeof(R) == 4 ? 2 : 1) pipe_kernel(PipeArgs p) {
    __shared__ R wsh[sizeof(R) == 4 ? 32 : 1];
    __shared__ __align__(16) fx64 fxtab[2 * kFxTab];  // the geodesic's sin/cos table
    const R *sgw = thermal_weights(wsh, p.therm);
    load_fx_table(p.sctab, fxtab);
    if constexpr (sizeof(R) == 4) {
        __shared__ int geo;
        if (threadIdx.x == 0) geo = pair_role(p);
        __syncthreads();
        if ((int)(threadIdx.x >> 5) < geo)
            pipe_geodesic(p, GeoTabs{fxtab, p.sctab});
        else if (geo > 0)
            pipe_reserve(p);
        pipe_transfer<R, OutT>(p, sgw);
        return;
    }
    __syncthreads();
    if ((int)(threadIdx.x >> 5) < ((blockIdx.x & 1) ? p.geo_warps_odd : p.geo_warps))
        pipe_geodesic(p, GeoTabs{fxtab, p.sctab});
    else
        pipe_transfer<R, OutT>(p, sgw);
}

}  // namespace prt
