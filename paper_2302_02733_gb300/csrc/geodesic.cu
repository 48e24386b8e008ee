// Backward null-geodesic integration from the camera (the paper's Section 2.1: one photon
// per pixel, integrated away from the observer and saved).
//
// Persistent kernel, one ray per lane. A lane whose ray stops takes the next ray from a
// global queue (warp-aggregated atomics), so long photon-ring rays do not hold a warp's
// other lanes idle. Every state is written to a block arena, 64 B per state: each lane
// writes two full 32 B sectors.
//
// The step runs in fixed point on the integer pipes (geofix.cuh): 4,800 instructions a warp and
// step, 19 of them on the FP64 pipe (346 in the FP64 form, 80 clocks each). The pipe of the integer
// multiply-adds bounds it (71% busy, 55% of the issue slots): 79 ms for the 3.68e8 steps of a
// 1024^2 image at 3 blocks per SM, against 228 ms in FP64. At 1 and 2 blocks per SM it takes 138 and
// 91 ms, at 4 (128 registers, 220 bytes of spills) 78. (Times before the transverse momentum's own
// scale, which costs 3%: 82 ms.)
#include <algorithm>
#include <cmath>
#include <vector>

#include "geodesic.cuh"

namespace prt {

static_assert(kGeoTabBytes == 3 * kSinTab * sizeof(double) + kFxTabBytes, "sin/cos table sizes");

// JOBS: the rays run over a table of images (p.jobs), each with its own camera; otherwise over
// the one image of p.cam. BLOCKS: the blocks per SM that its registers leave room for. At 3 (168
// registers) the integer pipes are busy, 82 ms for 1024^2 rays against 90 at 2; a launch that does not
// fill 2 blocks per SM is bound by the latency of a step instead, which is shorter where the step's
// values have more registers to be scheduled in (216): 5.6 against 6.0 ms for an ADAF at 64^2, 11.6
// against 12.3 for a torus at 128^2, 15.1 to 16.9 against 14.7 at 300^2.
template <bool JOBS, int BLOCKS>
__global__ void __launch_bounds__(kGeoThreads, BLOCKS) geodesic_kernel(GeoArgs p) {
    // the sin/cos table in shared memory: the RK4 stages read it at data-dependent indices, and
    // through the texture path those reads queued behind the transfer's gathers
    __shared__ __align__(16) fx64 fxtab[2 * kFxTab];
    const GeoTabs tabs{fxtab, p.sctab};
    load_fx_table(p.sctab, fxtab);
    __syncthreads();
    const Camera &c = p.cam;
    StepCam sc{};  // JOBS: the current ray's camera constants
    double y[7];
    long long ray = -1;
    int n = 0, blk = -1, slot = kBlockStates, pix = 0;
    bool live = false, drained = false;
    unsigned long long my_steps = 0;
    for (;;) {
        bool want = !live && !drained;
        unsigned long long t = warp_pop(&p.ctr->geo_next, want);
        if (want) {
            if (t < (unsigned long long)p.nrays) {
                ray = (long long)t;
                int ix, iy;
                if (JOBS) {  // the ray's global id (through the order list, if any) and image
                    const long long gid = p.pix_list ? p.pix_list[ray + p.ray_offset] : ray + p.ray_offset;
                    const JobDev &J = p.jobs[find_job(p.jobs, p.njobs, gid)];
                    ray_pixel(gid - J.ray_begin, J.cam.nx, J.cam.ny, ix, iy);
                    ray_start(J.cam, ix, iy, y);
                    sc = step_cam(J.cam);
                    pix = (int)gid;
                } else {
                    map_pixel(p.pix_list, ray + p.ray_offset, c.nx, c.ny, ix, iy);
                    pix = iy * c.nx + ix;
                    ray_start(c, ix, iy, y);
                }
                n = 0;
                blk = -1;
                slot = kBlockStates;
                live = true;
            } else {
                drained = true;
            }
        }
        if (__all_sync(0xffffffffu, !live && drained)) break;
        if (!live) continue;

        double h, yn[7];
        bool refl = JOBS ? geo_step(tabs, sc, y, yn, h) : geo_step(tabs, c, y, yn, h);
        // save state n with the step taken from it; then n+1 becomes current
        uint8_t status = 0;
        for (int pass = 0; pass < 2; pass++) {
            const double *z = pass ? yn : y;
            double hz = pass ? 0.0 : (refl ? -h : h);
            if (pass == 1 && status == 0) break;
            if (slot == kBlockStates) {
                unsigned long long b = atomicAdd(&p.ctr->arena_next, 1ull);
                if (b >= (unsigned long long)p.arena.nblocks) {
                    status = kOverflow;
                    break;
                }
                p.arena.prev[b] = blk;
                blk = (int)b;
                slot = 0;
            }
            PathState ps = {z[0], z[1], z[2], z[3] - z[4], z[4], z[5], z[6], hz};  // K^t = W - K^r
            reinterpret_cast<double4_32a *>(p.arena.states + (long long)blk * kBlockStates + slot)[0] =
                make_double4_32a(ps.r, ps.th, ps.ph, ps.kt);
            reinterpret_cast<double4_32a *>(p.arena.states + (long long)blk * kBlockStates + slot)[1] =
                make_double4_32a(ps.kr, ps.kth, ps.kph, ps.h);
            slot++;
            if (pass == 0) {
                n++;
#pragma unroll
                for (int k = 0; k < 7; k++) y[k] = yn[k];
                status = JOBS ? geo_stop(sc, y, n) : geo_stop(c, y, n);
            }
        }
        if (status) {
            RayRecord rec;
            bool ok = (status != kOverflow && status != kNan);
            rec.last_block = ok ? blk : -1;
            rec.nstates = ok ? n + 1 : 0;
            rec.status = status;
            p.rec[ray] = rec;
            if (p.steps_out) p.steps_out[pix] = (uint16_t)min(n, 65535);  // by pixel, or (JOBS) by global id
            my_steps += (unsigned long long)n;
            atomicAdd(&p.ctr->n_status[status], 1u);
            if (p.chunk_done) {
                // release this ray's states and record to the chunk's transfer: the fence orders
                // them before the count; the lane whose count completes the chunk fences again
                // (acquiring the others' and releasing to the host) and raises the flag
                __threadfence();
                const int k = p.layout.chunk_of(ray);
                if (atomicAdd(&p.chunk_done[k], 1u) + 1u == (unsigned)p.layout.size(k)) {
                    __threadfence_system();
                    *(volatile unsigned *)&p.chunk_flag[k] = 1u;
                }
            }
            live = false;
        }
    }
    // one counter update per lane
    if (my_steps) atomicAdd(&p.ctr->steps, my_steps);
}

__global__ void sincos_table_kernel(double *tab) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kSinTab) return;
    double th = kSinLo + k * kSinH;
    double s, c;
    sincos(th, &s, &c);
    tab[3 * k] = th;
    tab[3 * k + 1] = s;
    tab[3 * k + 2] = c;
}

// sin and cos of k 2^-8 to 2^-62: Taylor sums in double-double (Dekker's exact products, Knuth's
// exact sums), with the same result on every host. Built once per process.
static const fx64 *fx_table_host() {
    struct DD {
        double h, l;
    };
    auto add = [](DD a, DD b) {
        const double s = a.h + b.h, t = s - a.h;
        const double e = ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l), r = s + e;
        return DD{r, e - (r - s)};
    };
    auto mul = [](DD a, DD b) {
        const double p = a.h * b.h, e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h), r = p + e;
        return DD{r, e - (r - p)};
    };
    auto div = [](DD a, double d) {  // by a small integer
        const double q = a.h / d, e = (std::fma(-q, d, a.h) + a.l) / d, r = q + e;
        return DD{r, e - (r - q)};
    };
    static const std::vector<fx64> tab = [&] {
        std::vector<fx64> t(2 * kFxTab);
        for (int k = 0; k < kFxTab; k++) {
            const DD x{k / 256.0, 0.0}, m = mul(x, DD{-x.h, 0.0});
            DD s = x, c{1.0, 0.0}, ts = x, tc{1.0, 0.0};
            for (int n = 1; n < 30; n++) {
                tc = div(mul(tc, m), (2.0 * n - 1.0) * (2.0 * n));
                ts = div(mul(ts, m), (2.0 * n) * (2.0 * n + 1.0));
                c = add(c, tc);
                s = add(s, ts);
            }
            const DD v[2] = {s, c};
            for (int j = 0; j < 2; j++) {
                const double big = v[j].h * 4611686018427387904.0, whole = std::rint(big);  // 2^62
                t[2 * k + j] = (fx64)whole + (fx64)std::llrint((big - whole) + v[j].l * 4611686018427387904.0);
            }
        }
        return t;
    }();
    return tab.data();
}

// tab: the FP64 table (kSinTabBytes), then the fixed-point one (kFxTabBytes).
int launch_geo_tables(double *tab, cudaStream_t s) {
    sincos_table_kernel<<<(kSinTab + 255) / 256, 256, 0, s>>>(tab);
    if (cudaGetLastError() != cudaSuccess) return -1;
    return cudaMemcpyAsync(tab + 3 * kSinTab, fx_table_host(), kFxTabBytes, cudaMemcpyHostToDevice, s) == cudaSuccess
               ? 0
               : -1;
}

// The rays of 2 blocks on each SM: up to there every ray is resident in either variant (2 blocks of the
// larger one always fit: that is what it is compiled for).
static bool few_rays(long long nrays, int nsm) { return nrays <= 2ll * nsm * kGeoThreads; }

void launch_geodesic(const GeoArgs &a, int nsm, int blocks_per_sm, cudaStream_t s) {
    const int grid = ray_grid(nsm * blocks_per_sm, a.nrays, kGeoThreads);
    if (few_rays(a.nrays, nsm)) {
        if (a.jobs)
            geodesic_kernel<true, 2><<<grid, kGeoThreads, 0, s>>>(a);
        else
            geodesic_kernel<false, 2><<<grid, kGeoThreads, 0, s>>>(a);
    } else if (a.jobs) {
        geodesic_kernel<true, 3><<<grid, kGeoThreads, 0, s>>>(a);
    } else {
        geodesic_kernel<false, 3><<<grid, kGeoThreads, 0, s>>>(a);
    }
}

static int func_regs(const void *f) {
    cudaFuncAttributes a{};
    if (cudaFuncGetAttributes(&a, f) != cudaSuccess) {
        cudaGetLastError();
        return 255;
    }
    return a.numRegs;
}

int geodesic_regs(long long nrays, int nsm) {
    return few_rays(nrays, nsm)
               ? std::max(func_regs((const void *)geodesic_kernel<false, 2>), func_regs((const void *)geodesic_kernel<true, 2>))
               : std::max(func_regs((const void *)geodesic_kernel<false, 3>), func_regs((const void *)geodesic_kernel<true, 3>));
}

int geodesic_blocks_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, geodesic_kernel<false, 3>, kGeoThreads, 0) != cudaSuccess) n = 1;
    return n > 0 ? n : 1;
}

}  // namespace prt
