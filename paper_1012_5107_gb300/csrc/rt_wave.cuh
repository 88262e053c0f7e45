// rt_wave.cuh -- the wavefront form of the render loop.
//
// The persistent loop of rt_trace.cuh keeps one pixel per lane, so a warp
// integrates only while enough of its own lanes are inside the cloak and the
// others wait.  Here a block keeps a pool of pixels in flight in shared memory
// (each with its ray state in the cloak and everything else a lane would own)
// and two queues of pool entries: rays inside the cloak, ready to step, and
// rays that need service (an event located, a sample finished, a new pixel).
// Each warp repeatedly takes one task:
//   * integrate: up to 32 rays from the cloak queue, stepped together until
//     none is inside any more, or, in a task that is cut, until fewer than
//     min_active (scaled to the rays taken) are or a step cap is reached;
//     the rays still inside go back to the cloak queue, the others to the
//     service queue (see kWaveTaskSteps);
//   * serve: up to 32 entries of the service queue, filled up with free pool
//     entries that take new samples; each lane runs the service steps of
//     rt_trace.cuh until its ray is inside the cloak again (back to the cloak
//     queue) or the work list is exhausted (back to the free list).
// The work items are samples, not pixels: the samples of a pixel are traced
// at the same time, so the longest unit of work is one ray (a pixel of 4
// samples in a row would be up to four times longer and set the end of the
// launch).  Each finished sample leaves its colour in a scratch slot and
// counts itself in its pixel's counter; the last one adds the pixel's colours
// in sample order, the order of the per-lane loop, so the images are the same
// and only the grouping of rays into warps changes.
//
// The queues are rings of 16-bit pool indices guarded by a block-level lock
// (an atomic flag in shared memory) that one lane per warp takes for a few
// dozen cycles per task; every wait on it is bounded (WaveWait) and a timeout
// is counted in counters[kTimeouts] (reported as an error by the host).
#pragma once

#include "rt_trace.cuh"

namespace grt {

// An integration task runs to its end while the work list lasts: until none of
// its rays is inside any more.  Its rays came from neighbouring samples and
// stay together, so their steps take the same branches and end at about the
// same time; a task cut short hands its stragglers on one by one, and they
// break up the tasks after it (from 1 to 2 rays left behind the 1920 x 1080 x 16
// render goes from 85.6 to 114.8 ms; a queue of their own for the stragglers
// does not help: their tasks break up one another, and the step took 7.0 ms
// instead of 6.6).  Once the list has run dry, what is left
// are the longest rays, and a ray that needs service must not wait for the
// others of its task: the rays still inside go back to the cloak queue every
// kWaveTaskSteps steps, or when fewer than need are inside.
//
// Where neighbouring rays leave far apart -- a camera that looks across the
// grooves or at grazing elevation -- a task that waits for its last ray idles its
// lanes: at 900 x 900 x 4, E = 32, azimuth 90 and elevation 10 degrees 49.1 ms
// against 30.3 with tasks cut at min_active and every kWaveTaskSteps steps.  The
// FP32 loop of one scene measures it (wave_ragged) and cuts its tasks from then
// on: 30.4 ms.  In a launch of many scenes tasks of different scenes follow one
// another in the queues, where cut ones break up the uncut ones (the 64 uneven
// scenes: 682 ms uncut, 737 cut, 749 with the tally by scene, 790 with those cut
// that look across the grooves): all are cut if at least half of the samples
// look so (DevScene::ragged; 8 scenes of the view above at 512 x 512 x 4: 70.8 ms
// cut, 128 uncut), and none if not.  A served request's are cut if it and all in
// flight with it look so through a long box (rt_server.cu; 8 requests of that view
// 72.5 ms, uncut 129).
// Below 85 % of the lanes inside an uncut RK4 render is the slower one, above
// 89 % the faster (Dormand-Prince, with a third of the steps between services:
// 75 and 80 %).  The options build keeps its tasks uncut (Fresnel renders at
// kA = 0.6 are faster so at 63 %).
//
// Measured, cut throughout and so: the step's launch 7.05 / 6.41 ms, E = 8 / 32
// Dormand-Prince at 1920 x 1080 x 16 115.5 / 79.5 and 206.2 / 159.9, the Gaussian
// render 5.63 / 5.06 (384 x 384 x 4), the time form 8.70 / 8.49, Fresnel renders
// 7.90 / 6.02, the split FP64 render 39.1 / 37.8; uncut to the very end 64 x 64 x 1
// takes 1.52 ms instead of 1.25.  Over 128 scenes (elevations 10 to 55, azimuths
// 0 to 90 degrees, E = 8 and 32, kA = 0.1 and 0.25, RK4 and Dormand-Prince) it is
// within 5 % of the better of the two at 900 x 900 x 4, and within 16 % at
// 320 x 320 x 4, where half of the render is over before the tally tells.
// The general FP64 builds, bound by the FP64 pipe, whose instructions cost the
// same for few lanes as for all, are cut throughout.
constexpr int kWaveTaskSteps = 128;
constexpr int kWaveSpin = kDefaultWaitSpin;  // attempts (with a short sleep) before a wait gives up

// The block shape of the loop for a precision and integrator: threads per
// block, blocks per SM (which sets the registers a thread may use: 65536 /
// (threads x blocks)) and P, the samples in flight per block -- more than the
// block's lanes, so that a warp always finds work while the other warps hold
// theirs.  FP32: two blocks of 256 threads, 128 registers.  FP32
// Dormand-Prince keeps the running sums of its stages and two states live
// through a step and spills at 128 registers; with the step's start left in
// the pool (kInPool: it is read at the step's ends only) it spills 388 bytes (300
// before the loop in stretches) and 16 warps an SM beat the 12 that 168 registers allow (1920 x
// 1080 x 16, E = 2 / 8 / 32: 18.4 / 113.7 / 202.0 ms against 20.2 / 115.7 /
// 204.0 with one block of 384; with the start in registers 19.4 / 125.2 /
// 230.6).  FP32 RK4 in the pool is slower (7.07 -> 8.57 ms the step's launch:
// its steps are a quarter as long).  Its pool holds 320 samples a block: two
// blocks then fit the 196 KB split of the SM's memory, which leaves 60 KB of L1
// to the spills; with 384 they need the 228 KB one and the spills miss 28 KB
// (E = 8: 85.2 -> 80.8 ms, the same from 256 to 336 samples).  The Gaussian
// Dormand-Prince keeps the block of 384.  FP64: one block of 256 threads; the split RK4 step two.
template <class R, int INTEG>
struct WaveShape {
    static constexpr bool kDp = sizeof(R) == 4 && integ_of(INTEG) == RT_DP45;
    static constexpr bool kWide = kDp && gauss_of(INTEG);
    static constexpr bool kInPool = kDp && !gauss_of(INTEG);
    static constexpr bool kUncut = sizeof(R) == 4 || (INTEG & kModeSplit) != 0;   // see kWaveTaskSteps
    static constexpr int kEven = integ_of(INTEG) == RT_DP45 ? 72 : 82;            // see wave_ragged
    static constexpr int kBlock = kWide ? 384 : 256;
    static constexpr int kMinBlocks = ((sizeof(R) == 4 && !kWide) || split_of(INTEG)) ? 2 : 1;
    static constexpr int P = kWide ? 576 : kInPool ? 320 : (sizeof(R) == 4 ? 384 : (split_of(INTEG) ? 280 : 320));
};

static_assert((sizeof(Cold<double>) + sizeof(SplitBox) + 6) * 280 <= 115712, "two blocks of the split loop per SM");

template <class R, int INTEG>
constexpr size_t wave_smem_bytes()
{
    constexpr int P = WaveShape<R, INTEG>::P;
    return (sizeof(Cold<R>) + sizeof(LoopBox<R, INTEG>)) * P + 3 * sizeof(short) * P;
}

// Bytes of the Fresnel branch queues of a launch of `grid` blocks.
template <class R, int INTEG>
constexpr size_t wave_branch_bytes(int grid)
{
    return (size_t)grid * WaveShape<R, INTEG>::P * kMaxBranches * sizeof(Branch<R>);
}

struct WaveCtl {
    int lock;
    int in_head, in_cnt;     // cloak queue
    int sv_head, sv_cnt;     // service queue
    int fr_cnt;              // free list (stack)
    int exhausted;           // the work list has no pixels left
    int ragged;              // rays of a task leave too far apart: tasks are cut (kWaveTaskSteps)
    int error;
};

enum : int { WT_WAIT = 0, WT_INT = 1, WT_SRV = 2, WT_DONE = 3, WT_ERR = 4 };
// Where an integration task ends: WI_OPEN when none of its rays is inside,
// WI_CUT when fewer than min_active are or after kWaveTaskSteps, WI_LAST (the
// list has run dry) as the build does best.
enum : int { WI_LAST = 0, WI_CUT = 1, WI_OPEN = 2 };
enum : int { WD_NONE = 0, WD_IN = 1, WD_SRV = 2, WD_FREE = 3 };

// How the waits of a launch are bounded: `spin` attempts per wait (kWaveSpin
// unless the scene asks for fewer) and, with `hold` set, every block starts
// with its queue lock taken, so that every wait runs out and the launch ends
// with the timeouts counted (a test of failure detection; nothing faults).
struct WaveWait {
    int spin;
    int hold;
};

__device__ __forceinline__ bool wave_acquire(int* lock, int spin)
{
    for (int it = 0; it < spin; ++it) {
        if (atomicCAS(lock, 0, 1) == 0) {
            __threadfence_block();
            return true;
        }
        __nanosleep(32);
    }
    return false;
}

__device__ __forceinline__ void wave_release(int* lock)
{
    __threadfence_block();
    atomicExch(lock, 0);
}

// Publish the pool entries of the calling warp's lanes to the queue each
// names (dest); lanes with WD_NONE take part without publishing.  Returns
// false if the lock could not be taken.
template <int P>
__device__ __forceinline__ bool wave_push(WaveCtl& Q, short* inq, short* svq, short* frq, unsigned lane, int p,
                                          int dest, int spin)
{
    __threadfence_block();      // this lane's pool writes before its index is published
    const unsigned mi = __ballot_sync(0xffffffffu, dest == WD_IN);
    const unsigned ms = __ballot_sync(0xffffffffu, dest == WD_SRV);
    const unsigned mf = __ballot_sync(0xffffffffu, dest == WD_FREE);
    if ((mi | ms | mf) == 0u) return true;
    int ok = 1, ti = 0, ts = 0, tf = 0;
    if (lane == 0) {
        ok = wave_acquire(&Q.lock, spin) ? 1 : 0;
        if (ok) {
            ti = Q.in_head + Q.in_cnt;
            ts = Q.sv_head + Q.sv_cnt;
            tf = Q.fr_cnt;
            Q.in_cnt += __popc(mi);
            Q.sv_cnt += __popc(ms);
            Q.fr_cnt += __popc(mf);
            if (mf) Q.exhausted = 1;
        }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) return false;
    ti = __shfl_sync(0xffffffffu, ti, 0);
    ts = __shfl_sync(0xffffffffu, ts, 0);
    tf = __shfl_sync(0xffffffffu, tf, 0);
    const unsigned lt = (1u << lane) - 1u;
    if (dest == WD_IN) inq[(ti + __popc(mi & lt)) % P] = (short)p;
    else if (dest == WD_SRV) svq[(ts + __popc(ms & lt)) % P] = (short)p;
    else if (dest == WD_FREE) frq[tf + __popc(mf & lt)] = (short)p;
    __threadfence_block();
    __syncwarp();
    if (lane == 0) wave_release(&Q.lock);
    return true;
}

// A finished sample (its colour in C.acc): with one sample per pixel the pixel
// is written at once; otherwise the colour goes to the sample's scratch slot
// and the last sample of the pixel to finish writes the pixel.
template <class R, class Src>
__device__ __forceinline__ void wave_finish_sample(const Src& src, const DevScene& sc, const Cold<R>& C)
{
    float acc[3] = {C.acc[0], C.acc[1], C.acc[2]};
    const int spp = sc.spp;
    if (spp > 1) {
        float* col = src.sample_col(C.scene, C.work, C.sample);
        __stcg(reinterpret_cast<float4*>(col), make_float4(acc[0], acc[1], acc[2], 0.0f));
        __threadfence();                                     // the colour before the count
        if (atomicAdd(src.pixel_count(C.scene, C.work), 1) != spp - 1) return;
        __threadfence();                                     // the count before the other colours
        const float4* base = reinterpret_cast<const float4*>(col) - C.sample;
        acc[0] = acc[1] = acc[2] = 0.0f;
        for (int q = 0; q < spp; ++q) {
            const float4 v = __ldcg(base + q);
            acc[0] += v.x;
            acc[1] += v.y;
            acc[2] += v.z;
        }
        src.release_count(C.scene, C.work);
        // the block is dead: drop its lines from L2 without a write-back
        const char* blk = reinterpret_cast<const char*>(base);
        for (int64_t b = 0; b < col_block_bytes(spp); b += 128)
            asm volatile("discard.global.L2 [%0], 128;" ::"l"(blk + b) : "memory");
    }
    const float inv = 1.0f / (float)spp;
    float c[3];
    for (int a = 0; a < 3; ++a) c[a] = acc[a] * inv;
    float* o = src.rgb_of(C.scene) + 3 * C.work;
    o[0] = c[0]; o[1] = c[1]; o[2] = c[2];
    uint8_t* q8 = src.rgb8_of(C.scene);
    if (q8) {
        uint8_t* q = q8 + 3 * C.work;
        q[0] = quantize8(c[0]); q[1] = quantize8(c[1]); q[2] = quantize8(c[2]);
    }
    src.pixel_done(C.scene);
}

// Whether the work list has run dry (warp-uniform).
__device__ __forceinline__ bool wave_exhausted(const WaveCtl& Q)
{
    return __any_sync(0xffffffffu, *(volatile const int*)&Q.exhausted);
}

// Counts `its` steps of an uncut FP32 task of 32 rays, `lanes` of them by lanes
// still inside, and says whether such tasks kept fewer than kEven percent of
// their lanes inside of late, over all blocks of the launch.  The tally (steps,
// and lanes / 32, in halves of a word) is halved when it reaches kTallySteps,
// about a hundred steps of every warp of the GPU, so it follows the work; a
// launch's first tasks, whose early steps have all lanes inside, do not weigh on
// it for long.  (Told over the whole launch it came late in small renders and, at
// thresholds of 85 to 88 %, cut even ones: E = 8 at 55 degrees 17.8 -> 19.4 ms.)
constexpr unsigned kTallySteps = 1u << 19;
__device__ __forceinline__ bool wave_ragged(unsigned long long* counters, unsigned its, unsigned lanes, int even)
{
    unsigned long long now = 0;
    if ((threadIdx.x & 31u) == 0) {
        const unsigned long long add = ((unsigned long long)its << 32) + ((lanes + 16u) >> 5);
        const unsigned long long old = atomicAdd(&counters[kTally], add);
        now = old + add;
        if ((unsigned)(old >> 32) < kTallySteps && (unsigned)(now >> 32) >= kTallySteps)
            atomicAdd(&counters[kTally], 0ull - (((now >> 33) << 32) + ((now & 0xffffffffull) >> 1)));
    }
    now = __shfl_sync(0xffffffffu, now, 0);
    const unsigned long long n = now >> 32;
    return n > kTallySteps / 4 && (now & 0xffffffffull) * 100ull < n * (unsigned)even;
}

// The integration task of the split double precision step: the rays' states
// are SplitBoxes, stepped as in the general task of wave_loop.
__device__ __forceinline__ void wave_split_task(const DevScene& sc, Cold<double>& C, int p, SplitBox* boxes, int need,
                                                const WaveCtl& Q, bool open, int& dest, LaneStats& st,
                                                unsigned long long* iters)
{
    SplitBox& e = boxes[p >= 0 ? p : 0];
    int phase = PH_IDLE, surf = EV_NONE, steps = 0;
    if (p >= 0) {
        phase = PH_BOX;
        surf = C.surf;
        steps = C.steps;
    }
    const F2 kappa = sc.sp.kappa;
    const int64_t max_steps = sc.max_steps;
    int safe = 0;
    for (int it = 1;; ++it) {
#if RT_PROFILE
        ++*iters;
#endif
        if (phase == PH_BOX) split_box_step(sc, kappa, max_steps, C, e, phase, surf, steps, st, safe);
        if (__popc(__ballot_sync(0xffffffffu, phase == PH_BOX)) < need) break;
        if (it % kWaveTaskSteps == 0 && (!open || wave_exhausted(Q))) break;
    }
    if (p >= 0) {
        C.surf = surf;
        C.steps = steps;
        C.phase = phase;
        dest = (phase == PH_BOX) ? WD_IN : WD_SRV;
    }
}

template <class R, int INTEG, bool OPT, class Src>
__device__ __forceinline__ void wave_loop(const Src& src, unsigned long long* counters, int min_active, WaveWait ww)
{
    constexpr int P = WaveShape<R, INTEG>::P;
    extern __shared__ __align__(16) unsigned char wave_smem[];
    Cold<R>* cold = reinterpret_cast<Cold<R>*>(wave_smem);
    using LBox = LoopBox<R, INTEG>;
    LBox* boxes = reinterpret_cast<LBox*>(wave_smem + sizeof(Cold<R>) * P);
    short* inq = reinterpret_cast<short*>(wave_smem + (sizeof(Cold<R>) + sizeof(LBox)) * P);
    short* svq = inq + P;
    short* frq = svq + P;
    __shared__ WaveCtl Q;

    Branch<R>* branches = reinterpret_cast<Branch<R>*>(src.branches);
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        Cold<R>& C = cold[p];
        C.rays = 0;
        C.nevents = 0;
        C.scene = 0;
        for (int q = 0; q < 5; ++q) C.stat[q] = 0;
        C.br = branches ? branches + ((int64_t)blockIdx.x * P + p) * kMaxBranches : nullptr;
        frq[p] = (short)p;
    }
    if (threadIdx.x == 0) {
        Q.lock = ww.hold ? 1 : 0;
        Q.in_head = Q.in_cnt = Q.sv_head = Q.sv_cnt = 0;
        Q.fr_cnt = P;
        Q.exhausted = 0;
        Q.ragged = 0;
        Q.error = 0;
    }
    __syncthreads();

    const unsigned lane = threadIdx.x & 31u;
    LaneStats st = {0u, 0u, 0u, 0u};
#if RT_PROFILE
    // per warp (lane 0): cycles in integration tasks, cycles in service
    // tasks, integration iterations, cycles from the start to the exit
    unsigned long long prof[4] = {0, 0, 0, 0};
    const long long t_start = clock64();
#endif
    int idle = 0;
    bool failed = false;
    for (;;) {
        // ---- take a task (the leader decides under the lock) ----
        int task = WT_WAIT, m1 = 0, m2 = 0, b1 = 0, b2 = 0, locked = 0;
        int how = WI_LAST;             // integrate: where the task ends
        if (lane == 0) {
            if (!wave_acquire(&Q.lock, ww.spin)) {
                task = WT_ERR;
            } else {
                locked = 1;
                const int nin = Q.in_cnt, nsv = Q.sv_cnt, nfr = Q.fr_cnt;
                const bool fresh = !Q.exhausted && nfr > 0;
                if (Q.error) {
                    task = WT_ERR;
                } else if (nsv >= 32 || (nin < 32 && (nsv > 0 || fresh))) {
                    task = WT_SRV;
                    m1 = min(32, nsv);
                    b1 = Q.sv_head;
                    Q.sv_head = (Q.sv_head + m1) % P;
                    Q.sv_cnt -= m1;
                    m2 = fresh ? min(32 - m1, nfr) : 0;
                    Q.fr_cnt -= m2;
                    b2 = Q.fr_cnt;
                } else if (nin > 0) {
                    task = WT_INT;
                    if constexpr (WaveShape<R, INTEG>::kUncut)
                        how = Q.exhausted ? WI_LAST : Q.ragged ? WI_CUT : WI_OPEN;
                    m1 = min(32, nin);
                    b1 = Q.in_head;
                    Q.in_head = (Q.in_head + m1) % P;
                    Q.in_cnt -= m1;
                } else if (Q.exhausted) {
                    // nothing queued and no new pixels: whatever other warps
                    // hold, they finish themselves
                    task = WT_DONE;
                }
            }
        }
        task = __shfl_sync(0xffffffffu, task, 0);
        m1 = __shfl_sync(0xffffffffu, m1, 0);
        m2 = __shfl_sync(0xffffffffu, m2, 0);
        b1 = __shfl_sync(0xffffffffu, b1, 0);
        b2 = __shfl_sync(0xffffffffu, b2, 0);
        if constexpr (WaveShape<R, INTEG>::kUncut) how = __shfl_sync(0xffffffffu, how, 0);
        int p = -1;
        bool fresh = false;
        if (task == WT_INT && (int)lane < m1) p = inq[(b1 + (int)lane) % P];
        if (task == WT_SRV) {
            if ((int)lane < m1) {
                p = svq[(b1 + (int)lane) % P];
            } else if ((int)lane < m1 + m2) {
                p = frq[b2 + (int)lane - m1];
                fresh = true;
            }
        }
        __syncwarp();
        if (lane == 0 && locked) wave_release(&Q.lock);
        if (task == WT_ERR) { failed = true; break; }
        if (task == WT_DONE) break;
        if (task == WT_WAIT) {
            if (++idle > ww.spin) { failed = true; break; }
            __nanosleep(256);
            continue;
        }
        idle = 0;
#if RT_PROFILE
        const long long t_task = clock64();
#endif

        Cold<R>& C = cold[p >= 0 ? p : 0];
        const DevScene& sc = src.scene(C.scene);
        Box<R> b;
        int phase = PH_IDLE, surf = EV_NONE, steps = 0;
        int dest = WD_NONE;
        if (split_of(INTEG) && task == WT_INT) {
            unsigned long long* iters = nullptr;
#if RT_PROFILE
            iters = &prof[2];
#endif
            if constexpr (split_of(INTEG))
                wave_split_task(sc, C, p, boxes, how == WI_OPEN ? 1 : max(1, m1 - (32 - kMinActiveSplit)), Q, how == WI_OPEN,
                                dest, st, iters);
        } else if (task == WT_INT) {
            // ---- integrate ----
            if constexpr (!split_of(INTEG)) {
            // (kInPool steps the pool's entry in place)
            if (p >= 0) {
                if constexpr (!WaveShape<R, INTEG>::kInPool) b = boxes[p];
                phase = PH_BOX;
                surf = C.surf;
                steps = C.steps;
            }
            // one scene: the tally tells (wave_ragged); many: the host said (DevScene::ragged)
            constexpr bool kTallied = sizeof(R) == 4 && !OPT && Src::kParamScene;
            if constexpr (sizeof(R) == 4 && !OPT && !Src::kParamScene) {
                if (how == WI_OPEN && __any_sync(0xffffffffu, p >= 0 && sc.ragged)) how = WI_CUT;
            }
            int need = 1;
            if (!WaveShape<R, INTEG>::kUncut || how == WI_CUT) need = max(1, m1 - (32 - min_active));
            else if (sizeof(R) == 8 && how == WI_LAST) need = max(1, m1 - (32 - kMinActiveSplit));
            // step constants: read in place from the kernel parameters, or
            // copied once per task from a scene table in device memory
            const StepConst<R>* kp = &step_const<R>(sc);
            StepConst<R> kc;
            if constexpr (!Src::kParamScene) {
                kc = *kp;
                kp = &kc;
            }
            const int64_t max_steps = sc.max_steps;
            int safe = 0;                          // steps without the faces' tests (box_step_into)
            // stretches of kWaveTaskSteps steps (the loop within has no more
            // tests than a cut task needs: with the stretch's end tested in it
            // the step took 2 to 3 % longer)
            for (;;) {
                const int before = steps;
                int it = 0, inside = 0;
                for (; it < kWaveTaskSteps; ++it) {
#if RT_PROFILE
                    prof[2] += 1;
#endif
                    if (phase == PH_BOX) {
                        if constexpr (WaveShape<R, INTEG>::kInPool)
                            box_step<R, INTEG>(*kp, max_steps, C, boxes[p], phase, surf, steps, st, safe);
                        else
                            box_step<R, INTEG>(*kp, max_steps, C, b, phase, surf, steps, st, safe);
                    }
                    inside = __popc(__ballot_sync(0xffffffffu, phase == PH_BOX));
                    if (inside < need) { ++it; break; }
                }
                if (!WaveShape<R, INTEG>::kUncut || how != WI_OPEN) break;
                bool ragged = false;
                if constexpr (kTallied) {
                    if (m1 == 32) {
                        const unsigned lanes = __reduce_add_sync(0xffffffffu, (unsigned)(steps - before));
                        ragged = wave_ragged(counters, (unsigned)it, lanes, WaveShape<R, INTEG>::kEven);
                        if (ragged && lane == 0) *(volatile int*)&Q.ragged = 1;
                    }
                }
                if (inside < need || ragged || wave_exhausted(Q)) break;
            }
            if (p >= 0) {
                if constexpr (!WaveShape<R, INTEG>::kInPool) boxes[p] = b;
                C.surf = surf;
                C.steps = steps;
                C.phase = phase;
                dest = (phase == PH_BOX) ? WD_IN : WD_SRV;
            }
            }
        } else {
            // ---- serve ----
            if (p >= 0) {
                if (!fresh) {
                    phase = C.phase;
                    surf = C.surf;
                    steps = C.steps;
                    // (a step that crossed a surface is counted, but its start is kept)
                    if constexpr (split_of(INTEG))
                        from_split(sc, boxes[p], steps - boxes[p].steps0 - (phase == PH_EVENT ? 1 : 0), b);
                    else
                        b = boxes[p];
                }
                while (phase != PH_BOX && phase != PH_EXIT) {
                    if (phase == PH_EVENT || phase == PH_GUARD)
                        service_event<R, INTEG, OPT>(src.scene(C.scene), C, b, phase, surf, steps, src.rec_of(C.scene), st);
                    if (phase == PH_IDLE) {
                        const int64_t ws = src.grab(counters, lane);
                        if (ws < 0) { phase = PH_EXIT; break; }
                        int s, sample;
                        int64_t pix, out;
                        src.map_sample(ws, s, pix, out, sample);
                        C.scene = s;
                        C.work = out;
                        C.pix = pix;
                        C.sample = sample;
                        C.acc[0] = C.acc[1] = C.acc[2] = 0.0f;
                        start_sample<R, OPT>(src.scene(s), C, phase, surf, steps);
                    }
                    const DevScene& scs = src.scene(C.scene);
                    if (phase == PH_AIR) air_segment<R, INTEG, OPT>(scs, C, b, phase, surf, steps, src.rec_of(C.scene), st);
                    if (phase == PH_DONE) {
                        if (OPT && C.ibr < C.nbr) {
                            start_branch<R, INTEG>(scs, C, b, phase, surf, steps, st);   // next Fresnel branch
                        } else {
                            rt_ray_record* rec = src.rec_of(C.scene);
                            if (rec && (opt_flags<OPT>(scs) & RT_FLAG_FRESNEL)) {
                                // the record's colour: the sample's, summed over its paths
                                rt_ray_record* o = rec + C.work * scs.spp + C.sample;
                                o->rgb[0] = C.acc[0]; o->rgb[1] = C.acc[1]; o->rgb[2] = C.acc[2];
                            }
                            wave_finish_sample(src, scs, C);
                            phase = PH_IDLE;
                        }
                    }
                }
                if (phase == PH_BOX) {
                    if constexpr (split_of(INTEG)) to_split(src.scene(C.scene), b, steps, boxes[p]);
                    else boxes[p] = b;
                    C.surf = surf;
                    C.steps = steps;
                    C.phase = PH_BOX;
                    dest = WD_IN;
                } else {
                    dest = WD_FREE;
                }
            }
        }
        __syncwarp();
#if RT_PROFILE
        prof[task == WT_INT ? 0 : 1] += (unsigned long long)(clock64() - t_task);
#endif
        if (!wave_push<P>(Q, inq, svq, frq, lane, p, dest, ww.spin)) { failed = true; break; }
    }
#if RT_PROFILE
    prof[3] = (unsigned long long)(clock64() - t_start);
#endif
    if (failed && lane == 0) {
        atomicExch(&Q.error, 1);
        atomicAdd(&counters[kTimeouts], 1ull);
    }
    __syncthreads();

    // the split step evaluates four times and solves or continues W0 four times
    if constexpr (split_of(INTEG)) {
        st.evals += 4 * st.steps;
        st.newton += 4 * st.steps;
    }
    // counters: per-thread integration counters and the pool's per-pixel ones
    uint32_t v[11] = {0u, st.steps, st.evals, st.newton, 0u, st.refine, 0u, 0u, 0u, 0u, 0u};
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        const Cold<R>& C = cold[p];
        v[0] += C.rays;
        v[4] += C.nevents;
        for (int q = 0; q < 5; ++q) v[6 + q] += C.stat[q];
    }
#pragma unroll
    for (int q = 0; q < 11; ++q) {
        unsigned long long x = v[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0 && x) atomicAdd(&counters[1 + q], x);
    }
#if RT_PROFILE
    for (int q = 0; q < 4; ++q) {
        unsigned long long x = prof[q];
        if (lane == 0 && x) atomicAdd(&counters[12 + q], x);
    }
#endif
}

template <class R, int INTEG, bool OPT>
__global__ void __launch_bounds__(WaveShape<R, INTEG>::kBlock, WaveShape<R, INTEG>::kMinBlocks) wave_kernel(const __grid_constant__ DevScene sc,
                                                            float* __restrict__ rgb, uint8_t* __restrict__ rgb8,
                                                            rt_ray_record* rec, unsigned long long* counters,
                                                            int min_active, float* samp_col, int* pix_cnt,
                                                            void* branches, WaveWait ww)
{
    const OneScene src{sc, rgb, rgb8, rec, samp_col, pix_cnt, branches};
    wave_loop<R, INTEG, OPT>(src, counters, min_active, ww);
}

template <class R, int INTEG, bool OPT>
__global__ void __launch_bounds__(WaveShape<R, INTEG>::kBlock, WaveShape<R, INTEG>::kMinBlocks) wave_batch_kernel(
    const DevScene* __restrict__ scenes, const int64_t* __restrict__ offsets, const int64_t* __restrict__ soffsets,
    float* const* __restrict__ rgbs, int n, int64_t total, int64_t total_samples, float* samp_col, int* pix_cnt,
    void* branches, unsigned long long* counters, int min_active)
{
    // (double precision: a launch holds the samples that its table says)
    if constexpr (sizeof(R) == 8) {
        total_samples = __ldg(soffsets + n);
        if (total_samples == 0) return;
    }
    const ManyScenes src{scenes, offsets, soffsets, rgbs, n, total, total_samples, samp_col, pix_cnt, branches};
    wave_loop<R, INTEG, OPT>(src, counters, min_active, WaveWait{kWaveSpin, 0});
}

}  // namespace grt
