// trace.cu -- persistent path-tracing kernel (sm_103a).
//
// One GPU thread carries one path at a time.  What a traversal step needs
// lives in registers (the ray, its leaf, the optical depth left); the rest of
// the path (weights, vertex, directions, ids, sums) in a shared-memory slot
// of its own, touched only when a ray starts or ends.  A warp alternates
// between two loops:
//   steps  every lane on a ray crosses one leaf or handles one tentative
//          collision per iteration, whatever ray it is on (the path's free
//          flight or a sun ray), until enough lanes wait for something else;
//   rare   one pass over all waiting lanes: rays and paths that ended, chunk
//          sums, new chunks (one atomic per warp), the one Philox block,
//          path starts, vertices, ray starts.
//
// Physics (Villefranque et al. 2019):
//   free flight: null-collision sampling over leaves of uniform majorant M
//     (Sec. 2.3 steps 4a-4g, Eq. 2; Sec. 2.4 piecewise-uniform majorant):
//     optical depth -ln u is spent leaf by leaf; at a tentative collision the
//     true k is read and the collision is real with probability k / M.
//   local estimate (Sec. 4.1): at each real collision or ground hit the path
//     scores w * phase-or-BRDF toward the sun * T_sun, T_sun by ratio tracking
//     (t *= 1 - k/M, Russian roulette below 0.1) or delta tracking.
//   events: HG scattering with weight omega, Lambertian ground with weight
//     albedo, Russian roulette below w = 0.01; escape at the top.
// Random numbers: path id p, event e: stream (e, 0) for the flight (block 0
// word 0 its first optical depth -- the camera's first flight takes word 2
// of the path-start block instead -- and block j its j-th tentative
// collision); (e, 1) for the vertex ending that flight and its sun ray
// (block 0: two direction draws, roulette and, in word 3, the sun ray's
// first optical depth; block j the sun ray's j-th tentative collision);
// (0, 2) for the camera jitter / ground point; (0, 3) for the direct sun ray
// of a flux path.  A learned vertex draws from blocks kBlockVertex and
// kBlockVertex - 1 of stream (e, 0) (word 1 of the latter: its sun ray's
// first optical depth), a Rayleigh vertex its species from word 0 of block
// kBlockVertex.
//
// What bounds it: instruction issue.  The split keeps the step loop short (no
// sums, claims or path state in it, and of the random blocks only that of a
// tentative collision in a leaf of several voxels) and its registers few
// enough for 8 blocks of 128 threads an SM without spills; a single loop
// with everything in it, at 72 registers and one Philox block per iteration,
// took 95.1 ms for 16.8 M paths of the 512 x 512 x 160 cumulus image, this
// one 48.7 ms (octree image of 11.8 M paths 46.3 -> 29.8 ms, 16.8 M flux
// paths 81.8 -> 39.5 ms, 4 M over a relief 45.6 -> 19.3 ms).  7, 9 and 10
// resident blocks: 49.1, 48.9 and 49.1 ms (flux 40.8, 40.5, 39.3, relief
// 19.4, 19.9, 21.6).
// A step draws its Philox block only when its result depends on it: a
// voxel leaf's majorant is the voxel itself, so a tentative collision there
// is real (a sun ray's ratio 1 - k/M is 0) whatever the draw.
#include <cuda_bf16.h>

#include "mcrt_internal.h"

#ifndef MCRT_TRACE_MIN_BLOCKS
#define MCRT_TRACE_MIN_BLOCKS 8   // resident blocks of 128 threads the register budget must allow (64 registers)
#endif

namespace mcrt {

namespace {

constexpr unsigned kFull = 0xffffffffu;

enum Kind { kMain = 0, kSunLocal = 1, kSunDirect = 2, kSunHelp = 3 };   // kSunHelp: another lane's kSunLocal

// Counter slots (see mcrt_tally_counters).
enum {
    C_PATHS = 0, C_TENT = 1, C_REAL = 2, C_GROUND = 3, C_LEAF = 4,
    C_SUN_TENT = 5, C_SUN_LEAF = 6, C_SUN_RAYS = 7, C_ABORT = 8, C_FLIGHTS = 9
};
constexpr int kCounters = 10;
// Extra slots filled with atomicMax in counting mode: [10] most loop
// iterations spent on one path, [11] longest time (ns) a warp ran before the
// work queue ran dry, [12] longest time (ns) a warp ran in total.
enum { C_MAX_ITERS = 10, C_T_DRY = 11, C_T_END = 12 };
// Counting mode also records, per warp, the SM clock cycles spent in each
// section of the loop (slots 13..21): sums and claims, Philox, path start,
// ray start, steps, vertex, (two unused,) ended rays and paths.
constexpr int C_SEC = 13;
constexpr int kSections = 9;
// ... and, per step iteration, lane occupancy (slots 22..29): iterations,
// lanes holding a path, stepping, at a tentative collision, running in a rare
// pass, waiting for one, rare passes, lanes without a path.
constexpr int C_OCC = 22;
constexpr int kOcc = 8;

// What a lane is doing.  PH_STEP lanes take traversal steps; phases from
// PH_CLAIM on wait for the warp's next rare pass.
enum Phase {
    PH_STEP = 0,
    PH_IDLE,        // no chunk, nothing left to claim: free to help
    PH_HELPED,      // a helper whose sun ray has ended, until its owner takes the result
    PH_STALL,       // an owner waiting for a helper (its phase in K_WANT)
    PH_CLAIM,       // no chunk
    PH_FLUSH,       // chunk finished: its sums go to the tally, then a new chunk
    PH_START,       // a path starts
    PH_BEGIN,       // a ray starts: the flight from the vertex, or a flux path's direct sun ray
    PH_VERTEX,      // a volume vertex
    PH_GROUND,      // a ground vertex
    PH_RESUME,      // a path stopped at a learned vertex goes on
    PH_SUSPEND,     // a path stops at a learned vertex
    PH_WALK,        // the ray's hit on the heightfield is to be found
    PH_HIT,         // a tentative collision in a voxel leaf, at distance R.t
    PH_ROULETTE,    // ... that left a sun ray a residual Ts: its draw
    PH_REAL,        // a real collision at distance R.t of extinction K_VK
    PH_LAND,        // a flight met the heightfield at distance R.t
    PH_FLOOR,       // a flight met the plane z = 0 at distance R.t
    PH_SUN_END,     // a sun ray ended with transmissivity Ts
    PH_END          // the path ends
};

// Per-thread slots of a path's state outside its registers, [field][thread]
// (conflict-free); fields past kCold depend on the kernel variant.
enum Cold {
    K_PID_LO = 0, K_PID_HI, K_LEFT,          // path id, paths left in the chunk (this one included)
    K_CELL,                                  // tally cell (pixel; batch item)
    K_EV,                                    // event index | kTermAfter
    K_W, K_SCORE, K_CF,                      // weight, score so far, factor of the sun ray's estimate
    K_VX, K_VY, K_VZ, K_VK,                  // vertex and its extinction
    K_NX, K_NY, K_NZ,                        // direction of the next flight
    K_Q, K_WANT,                             // owner: its helpers in order, the phase it waits in
    kCold,
    // a helper's slots: its ray's end (0 tracking, 1 ended, 2 taken), its
    // first optical depth's word, its transmissivity
    K_DONE = K_LEFT, K_WORD = K_NX, K_TS = K_SCORE
};
constexpr uint32_t kTermAfter = 0x80000000u;   // the path ends with this event's estimate
// Heightfield walkers of a warp that go together.  A path walks about three
// times, so a pass rarely has two walkers, and each walk alone held the warp
// for some twenty dependent loads: 4 M flux paths over a 4096^2 relief 23.7
// ms with each walk at once, 20.9 ms in eights (21.6 in fours, 21.4 in
// twelves), 20.0 ms with a cell's corners in one record.
constexpr int kWalkBatch = 8;
// K_Q: the number of helpers at work (low 3 bits), then their lanes, first
// handed off first, 5 bits each.
constexpr uint32_t kMaxHelpers = 5;

// Helpers.  A path is a serial chain: flight, sun ray, flight, sun ray, ...,
// and a launch lasts as long as its longest one.  But the next flight does
// not need the sun ray's result, so a lane without a path (the work queue is
// dry, or the launch has fewer paths than lanes) takes a vertex's sun ray
// over from a lane of its warp, which goes on with its flight in the same
// pass.  The owner adds the results in the order of its vertices, so a
// path's score is the same sum, bit for bit.  A lone path takes about 5,500
// cycles per vertex with a helper, 8,000 without; 64 x 64 x 16 paths of the
// blob field 2.5 -> 2.05 ms, a 500 x 301 x 16 image 10.5 -> 9.3 ms.

// The ground: flat, or a heightfield in either of its forms (DevScene::hf).
enum Ground { kFlat = 0, kRecords, kHeights };

// A batch's kernel holds its lane's scene pointer and derivative sums besides:
// 12 fields 89.6 ms with spills at 8 blocks of 128, 88.0 without at 7.
constexpr int kBatchBlocks = 7;

// EXTRA: the variants that also handle decomposition tracking of sun rays
// and Rayleigh clear air (chosen at run time); the others carry neither, so
// the paper's estimator keeps its registers.  In batches, EXTRA instead
// adds the dT/dalpha estimate.  TERRAIN: the ground (Ground).
template <int SENSOR, bool BF16, bool COUNT, bool LEARNED, bool BATCH = false, int TERRAIN = kFlat, bool EXTRA = false>
__global__ void __launch_bounds__(128, BATCH ? kBatchBlocks : MCRT_TRACE_MIN_BLOCKS) trace_kernel(const __grid_constant__ TraceParams P)
{
    // Steps between looks at who waits.  Two spare half of the votes and the
    // loop: cumulus image of 16.8 M paths 49.5 -> 48.8 ms, 16.8 M flux paths 40.2
    // -> 39.4, a 64 x 64 x 16 image 2.0 -> 1.75; three do not fit the instruction
    // cache (52.9 ms), nor do two of the longer variants (4 M paths over a relief
    // 19.2 -> 20.7, Rayleigh image 8.8 -> 9.3, batch 86.8 -> 87.7; with dT/dalpha,
    // whose registers differ, 10.7 -> 10.4).
    constexpr int kSteps = COUNT || TERRAIN || EXTRA != BATCH ? 1 : 2;
    // quantities per path: camera radiance; flux T_dir, T_dif, T_tot (+ dT/dg, dT/dalpha in batches)
    constexpr int NQ = (SENSOR == kCamera) ? 1 : (BATCH ? 5 : 3);
    // decomposition tracking needs the leaf minorants
    constexpr bool DECOMP = EXTRA && !BATCH;
    // chunk sums of x and x^2 in FP32 (a chunk is at most 8 paths: relative
    // error below 7 * 2^-24 of the sum of |x| before the FP64 atomic add)
    constexpr int K_ACC = kCold;
    constexpr int K_TDIR = K_ACC + 2 * NQ;                     // flux: direct transmissivity
    constexpr int K_FZ = K_TDIR + (SENSOR == kFlux ? 1 : 0);   // heightfield flux: n_z of the surface at the path start
    constexpr int K_SG = K_FZ + (TERRAIN ? 1 : 0);             // batches: d/dg ...
    constexpr int K_SVP = K_SG + 1, K_CFS = K_SG + 2, K_DSC = K_SG + 3;
    constexpr int K_SA = K_SG + 4, K_DAL = K_SG + 5;           // ... and d/dalpha, the droplets' absorptivity
    constexpr int K_LV = K_SG + (BATCH ? 6 : 0);               // learned mode: volume vertices so far,
    constexpr int K_REC = K_LV + 1;                            // training record awaiting its own estimate
    constexpr int kFields = K_LV + (LEARNED ? 2 : 0);
    __shared__ float cold[kFields][128];

    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int tid = threadIdx.x;
    auto F = [&](int f) -> float& { return cold[f][tid]; };
    auto geti = [&](int f) -> uint32_t { return __float_as_uint(cold[f][tid]); };
    auto seti = [&](int f, uint32_t v) { cold[f][tid] = __uint_as_float(v); };
    auto get_pid = [&]() -> unsigned long long {
        return (unsigned long long)geti(K_PID_LO) | ((unsigned long long)geti(K_PID_HI) << 32);
    };
    auto set_pid = [&](unsigned long long pid) {
        seti(K_PID_LO, (uint32_t)pid);
        seti(K_PID_HI, (uint32_t)(pid >> 32));
    };

    // score + cf T: one operation, or two (a batch's other sums use the
    // product); each variant keeps the rounding it has always had
    auto add_estimate = [](float score, float cf, float T) -> float {
        return BATCH ? __fadd_rn(score, __fmul_rn(cf, T)) : __fmaf_rn(cf, T, score);
    };
    auto block = [&](unsigned long long pid, uint32_t c2, uint32_t b) -> uint4 {
        if constexpr (BATCH) return draw_block(pid, c2, b, P.items[geti(K_CELL)].key);
        else return philox4x32_10(make_uint4((uint32_t)pid, (uint32_t)(pid >> 32), c2, b), P.ks);
    };

    // the warp's FP64 sums for tally cell wcell (flux): lane q owns entry q
    __shared__ double wsum[SENSOR == kCamera ? 1 : 4][SENSOR == kCamera ? 1 : 2 * NQ];
    uint32_t wcell = 0u;
    auto spill_sums = [&]() {
        if (SENSOR == kFlux && lane < 2 * NQ) {
            double& a = wsum[tid >> 5][lane];
            if (a != 0.0) atomicAdd(((lane & 1) ? P.s2 : P.s1) + (size_t)wcell * NQ + (lane >> 1), a);
            a = 0.0;
        }
    };
    if (SENSOR == kFlux && lane < 2 * NQ) wsum[tid >> 5][lane] = 0.0;

    // ---- per-lane state ------------------------------------------------------
    const float kInf = __int_as_float(0x7f800000);
    bool exhausted = false;                 // warp-uniform: nothing left to claim
    int phase = lane < P.claim_lanes ? PH_CLAIM : PH_IDLE;
    Ray R;
    int kind = kMain;
    uint32_t blk = 1;                       // Philox block of the ray's next tentative collision
    float tau = 0.0f, Ts = 1.0f;
    float tg = kInf;                        // heightfield: distance of the flight's ground hit from R.o
    float tpend = kInf;                     // heightfield: where the flight enters the relief layer (walk pending)
#pragma unroll
    for (int q = 0; q < 2 * NQ; ++q) F(K_ACC + q) = 0.0f;
    seti(K_CELL, 0u);
    seti(K_LEFT, 0u);
    seti(K_Q, 0u);
    __shared__ uint8_t pairs[4][2][32];     // hand-offs of a pass: owners' and helpers' lanes by rank
    bool helping = false;                   // warp-uniform: a helper is at work
    if (LEARNED) seti(K_REC, 0xFFFFFFFFu);
    unsigned long long cnt[kCounters];
#pragma unroll
    for (int q = 0; q < kCounters; ++q) cnt[q] = 0;
    uint32_t path_iters = 0, max_iters = 0, tents = 0;
    unsigned long long sec[kSections];
#pragma unroll
    for (int q = 0; q < kSections; ++q) sec[q] = 0;
    unsigned long long occ[kOcc];
#pragma unroll
    for (int q = 0; q < kOcc; ++q) occ[q] = 0;
    long long tclk = COUNT ? clock64() : 0;
    auto mark = [&](int q) {
        if (COUNT) {
            __syncwarp();
            const long long now = clock64();
            sec[q] += (unsigned long long)(now - tclk);
            tclk = now;
        }
    };
    uint64_t t_start = 0, t_dry = 0;
    if (P.deadline_ns || COUNT) t_start = globaltimer_ns();
    int budget = 1024;                      // steps until the next deadline / cancel check

    for (;;) {
        // ==== rare pass: every lane that is not stepping ======================
        // ---- what ended the lane's ray ------------------------------------------
        // (the step loop only leaves the distance; points are the same fused
        // operation there and here.  Three lanes of a warp have a tentative
        // collision in an iteration, seven in a pass: handled in the loop, the
        // cumulus image of 16.8 M paths took 55.8 ms instead of 50.0, 16.8 M flux
        // paths 44.6 instead of 40.9.)
        if (phase == PH_HIT) {
            // the leaf's majorant is the voxel's own extinction: a flight's
            // collision is real, a sun ray keeps 1 - k/M, 0 but for rounding
            if (kind == kMain) {
                F(K_VK) = R.M;
                phase = PH_REAL;
                if (LEARNED) { seti(K_NX, (uint32_t)R.lo[0]); seti(K_NY, (uint32_t)R.lo[1]); seti(K_NZ, (uint32_t)R.lo[2]); }
            } else {
                phase = PH_SUN_END;
                if (P.sun_mode == MCRT_SUN_DELTA) {
                    Ts = 0.0f;
                } else {
                    Ts *= null_share<!EXTRA>(R.M, R.M);
                    if (Ts > 0.0f) phase = PH_ROULETTE;
                    else Ts = 0.0f;
                }
            }
        }
        if (phase == PH_REAL || phase == PH_FLOOR || (TERRAIN && phase == PH_LAND)) {
            float p[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) p[a] = __fmaf_rn(R.t, R.d[a], R.o[a]);
            if (phase != PH_REAL) {
                const DevScene& S = BATCH ? P.items[geti(K_CELL)].S : P.S;
                if (TERRAIN && phase == PH_LAND) {
                    // the surface hit (x, y wrapped into the domain)
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        if (p[a] < 0.0f) p[a] += S.Lper[a];
                        if (!(p[a] < S.Lper[a])) p[a] -= S.Lper[a];
                        if (!(p[a] >= 0.0f && p[a] < S.Lper[a])) p[a] = 0.0f;
                    }
                    p[2] = fmaxf(p[2], 0.0f);
                } else {
                    p[2] = 0.0f;
                    p[0] = fminf(fmaxf(p[0], 0.0f), S.Lper[0]);
                    p[1] = fminf(fmaxf(p[1], 0.0f), S.Lper[1]);
                    if (!(p[0] < S.Lper[0])) p[0] = 0.0f;
                    if (!(p[1] < S.Lper[1])) p[1] = 0.0f;
                }
                phase = PH_GROUND;
            } else {
                phase = PH_VERTEX;
                if (LEARNED && geti(K_LV) < (uint32_t)P.n_learned) phase = PH_SUSPEND;
            }
            F(K_VX) = p[0]; F(K_VY) = p[1]; F(K_VZ) = p[2];
        }
        if (phase == PH_ROULETTE) {
            // the block this tentative collision would have drawn: test (the
            // ratio's roulette below 0.1) and next optical depth
            const uint4 x = block(get_pid(),
                                  SENSOR == kFlux && kind == kSunDirect ? 3u : ((geti(K_EV) & ~kTermAfter) << 2) | 1u,
                                  blk);
            ++blk;
            phase = PH_STEP;
            if (Ts < 0.1f) {
                if (u01(x.x) * 0.1f <= Ts) Ts = 0.1f;
                else { Ts = 0.0f; phase = PH_SUN_END; }
            }
            tau = -__logf(u01(x.y));
        }
        if (helping) {
            if (phase == PH_SUN_END && kind == kSunHelp) {
                F(K_TS) = Ts;
                seti(K_DONE, 1u);
                phase = PH_HELPED;
            }
            __syncwarp();
            uint32_t q = geti(K_Q);
            while (q & 7u) {
                const int h = (tid & ~31) + (int)((q >> 3) & 31u);
                if (__float_as_uint(cold[K_DONE][h]) != 1u) break;
                const float cf = cold[K_CF][h], hT = cold[K_TS][h];
                F(K_SCORE) = add_estimate(F(K_SCORE), cf, hT);
                if constexpr (BATCH) {
                    const float e = __fmul_rn(cf, hT);
                    F(K_DSC) = __fmaf_rn(e, cold[K_CFS][h], F(K_DSC));
                    if (EXTRA) F(K_DAL) = __fmaf_rn(e, cold[K_SA][h], F(K_DAL));
                }
                cold[K_DONE][h] = __uint_as_float(2u);
                q = ((q >> 8) << 3) | ((q & 7u) - 1u);
            }
            seti(K_Q, q);
            __syncwarp();
            if (phase == PH_HELPED && geti(K_DONE) == 2u) phase = PH_IDLE;
            if (phase == PH_STALL) phase = (int)geti(K_WANT);
            helping = __any_sync(kFull, (q & 7u) != 0u);
            if ((q & 7u) && (phase == PH_END || (LEARNED && phase == PH_SUSPEND))) {
                seti(K_WANT, (uint32_t)phase);
                phase = PH_STALL;
            }
        }
        if (phase == PH_SUN_END) {
            if (SENSOR == kFlux && kind == kSunDirect) {
                if constexpr (SENSOR == kFlux) F(K_TDIR) = TERRAIN ? F(K_TDIR) * Ts : Ts;
                seti(K_EV, 0u);
                kind = kMain;
                phase = PH_BEGIN;
            } else {
                const float cf = F(K_CF);
                F(K_SCORE) = add_estimate(F(K_SCORE), cf, Ts);
                if constexpr (BATCH) {
                    const float e = __fmul_rn(cf, Ts);
                    F(K_DSC) = __fmaf_rn(e, F(K_SG) + F(K_CFS), F(K_DSC));
                    if (EXTRA) F(K_DAL) = __fmaf_rn(e, F(K_SA), F(K_DAL));
                    F(K_SG) += F(K_SVP);
                }
                if constexpr (LEARNED) {
                    const uint32_t rec = geti(K_REC);
                    if (rec != 0xFFFFFFFFu) {
                        P.rec_val[4 * (size_t)rec + 2] = cf * Ts;
                        seti(K_REC, 0xFFFFFFFFu);
                    }
                }
                const uint32_t e = geti(K_EV);
                if (e & kTermAfter) {
                    phase = PH_END;
                } else {
                    seti(K_EV, e + 1u);
                    kind = kMain;
                    phase = PH_BEGIN;
                }
            }
        }
        if (phase == PH_END) {
            const float score = F(K_SCORE);
            if constexpr (SENSOR == kCamera) {
                F(K_ACC) += score;
                F(K_ACC + 1) += score * score;
            } else {
                const float tdir = F(K_TDIR);
                const DevScene& S = BATCH ? P.items[geti(K_CELL)].S : P.S;
                const float pi_over_mu0 = __fdividef(kPi, TERRAIN ? F(K_FZ) * S.sun[2] : S.sun[2]);
                const float tf = pi_over_mu0 * score;
                const float tt = tdir + tf;
                F(K_ACC + 0) += tdir; F(K_ACC + 1) += tdir * tdir;
                F(K_ACC + 2) += tf; F(K_ACC + 3) += tf * tf;
                F(K_ACC + 4) += tt; F(K_ACC + 5) += tt * tt;
                if constexpr (BATCH) {
                    const float dt = pi_over_mu0 * F(K_DSC);
                    F(K_ACC + 6) += dt; F(K_ACC + 7) += dt * dt;
                    if (EXTRA) {
                        const float da = pi_over_mu0 * F(K_DAL);
                        F(K_ACC + 8) += da; F(K_ACC + 9) += da * da;
                    }
                }
            }
            if (COUNT) {
                cnt[C_PATHS]++;
                max_iters = max(max_iters, path_iters);
            }
            const unsigned long long pid = get_pid();
            if (LEARNED && P.final_score) P.final_score[pid - P.path_base] = score;
            const uint32_t left = geti(K_LEFT) - 1u;
            seti(K_LEFT, left);
            set_pid(pid + 1u);
            phase = left ? PH_START : PH_FLUSH;
        }
        mark(8);
        // ---- stop paths at a learned vertex: state and features to the queue
        if constexpr (LEARNED) {
            const unsigned smask = __ballot_sync(kFull, phase == PH_SUSPEND);
            if (smask) {
                const int leader = __ffs(smask) - 1;
                unsigned base = 0;
                if (lane == leader) base = atomicAdd(P.qout_count, (unsigned)__popc(smask));
                base = __shfl_sync(kFull, base, leader);
                if (phase == PH_SUSPEND) {
                    const DevScene& S = P.S;
                    const unsigned slot = base + (unsigned)__popc(smask & lt_mask);
                    const unsigned long long pid = get_pid();
                    if (slot < P.qout_cap) {
                        // features: position in [-1, 1], incoming direction, ln(k), ln(M1), ln(M2)
                        const float vx[3] = {F(K_VX), F(K_VY), F(K_VZ)}, vk = F(K_VK);
                        const int nv[3] = {(int)geti(K_NX), (int)geti(K_NY), (int)geti(K_NZ)};   // the collision's voxel
                        const float Lz = (float)S.n[2] * S.h[2];
                        float f[9];
                        f[0] = 2.0f * vx[0] / S.Lper[0] - 1.0f;
                        f[1] = 2.0f * vx[1] / S.Lper[1] - 1.0f;
                        f[2] = 2.0f * vx[2] / Lz - 1.0f;
                        f[3] = R.d[0]; f[4] = R.d[1]; f[5] = R.d[2];
                        f[6] = logf(vk + 1e-6f);
                        const float M1 = __ldg(P.pyr1 + ((size_t)(nv[2] >> 3) * P.d1[1] + (nv[1] >> 3)) * P.d1[0] +
                                               (nv[0] >> 3));
                        const int s2 = 3 * P.lev2;
                        const float M2 = __ldg(P.pyr2 + ((size_t)(nv[2] >> s2) * P.d2[1] + (nv[1] >> s2)) * P.d2[0] +
                                               (nv[0] >> s2));
                        f[7] = logf(M1 + S.k_gas + 1e-6f);
                        f[8] = logf(M2 + S.k_gas + 1e-6f);
                        uint32_t pk[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const __nv_bfloat162 v = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
                            pk[i] = *reinterpret_cast<const uint32_t*>(&v);
                        }
                        pk[4] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(f[8]));
                        pk[5] = pk[6] = pk[7] = 0u;
                        P.qout_feat[2 * (size_t)slot] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        P.qout_feat[2 * (size_t)slot + 1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                        P.qout[4 * (size_t)slot] = make_uint4((uint32_t)pid, (uint32_t)(pid >> 32), geti(K_EV), geti(K_LV));
                        P.qout[4 * (size_t)slot + 1] = make_uint4(__float_as_uint(vx[0]), __float_as_uint(vx[1]),
                                                                  __float_as_uint(vx[2]), __float_as_uint(vk));
                        P.qout[4 * (size_t)slot + 2] = make_uint4(__float_as_uint(R.d[0]), __float_as_uint(R.d[1]),
                                                                  __float_as_uint(R.d[2]), geti(K_W));
                        P.qout[4 * (size_t)slot + 3] =
                            make_uint4(geti(K_SCORE), SENSOR == kFlux ? geti(K_TDIR) : 0u, 0u, 0u);
                    }
                    const uint32_t left = geti(K_LEFT) - 1u;
                    seti(K_LEFT, left);
                    set_pid(pid + 1u);
                    phase = left ? PH_START : PH_FLUSH;
                }
            }
        }
        // ---- finished chunks: their sums go to the tally -----------------------
        unsigned fmask = __ballot_sync(kFull, phase == PH_FLUSH);
        if (fmask) {
            if constexpr (SENSOR == kCamera) {
                // (chunks that end together rarely share a pixel)
                if (phase == PH_FLUSH) {
                    const uint32_t c = geti(K_CELL);
                    MCRT_CHECK(c < (unsigned)(P.width * P.height), 3);
                    atomicAdd(P.s1 + c, (double)F(K_ACC));
                    atomicAdd(P.s2 + c, (double)F(K_ACC + 1));
                }
            } else {
                // lane q < 2 NQ adds quantity q of the finished chunks, one after
                // another, to the warp's FP64 sums of the tally cell it works on;
                // they reach the tally when the warp turns to another cell, and
                // at its end.  (A shuffle reduction of every quantity over the
                // warp and an atomic per finished chunk took 10-12 % of a
                // trace with claims of one path: 16.8 M flux paths 49.8 -> 44.5
                // ms, 4 M over a relief 25.3 -> 23.2, a learned image's passes
                // 22.3 -> 19.9.)
                __syncwarp();
                for (unsigned left = fmask; left; left &= left - 1u) {
                    const int src = (tid & ~31) + __ffs(left) - 1;
                    const uint32_t c = __float_as_uint(cold[K_CELL][src]);
                    MCRT_CHECK(c < (BATCH ? (unsigned)P.n_items : 1u), 3);
                    if (BATCH && c != wcell) {
                        spill_sums();
                        wcell = c;
                    }
                    if (lane < 2 * NQ) wsum[tid >> 5][lane] += (double)cold[K_ACC + lane][src];
                }
                __syncwarp();
            }
            if (phase == PH_FLUSH) {
                phase = PH_CLAIM;
#pragma unroll
                for (int q = 0; q < 2 * NQ; ++q) F(K_ACC + q) = 0.0f;
            }
        }
        // ---- claim chunks for idle lanes (one atomic per warp) -------------
        const unsigned idle = __ballot_sync(kFull, phase == PH_CLAIM);
        if (idle) {
            unsigned long long base = P.total;
            if (!exhausted) {
                const int nidle = __popc(idle);
                const int leader = __ffs(idle) - 1;
                if (lane == leader) base = atomicAdd(&P.work->next, (unsigned long long)nidle * P.chunk);
                base = __shfl_sync(kFull, base, leader);
                if (base + (unsigned long long)nidle * P.chunk >= P.total) {
                    exhausted = true;
                    if (COUNT) t_dry = globaltimer_ns();
                }
            }
            if (phase == PH_CLAIM) {
                phase = PH_IDLE;
                unsigned long long pid = base + (unsigned long long)__popc(idle & lt_mask) * P.chunk;
                if (pid < P.total) {
                    uint32_t left = (uint32_t)min((unsigned long long)P.chunk, P.total - pid);
                    phase = (LEARNED && P.resume) ? PH_RESUME : PH_START;
                    // the batch (learned mode) or shard (flux) this launch traces
                    if (!BATCH && !(LEARNED && P.resume)) pid += P.path_base;
                    if constexpr (BATCH) {
                        // items own chunk-aligned id ranges: find the item, use its local ids
                        int lo = 0, hi = P.n_items - 1;
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (P.items[mid].begin <= pid) lo = mid;
                            else hi = mid - 1;
                        }
                        const unsigned long long b = P.items[lo].begin, np = P.items[lo].npaths;
                        pid -= b;
                        if (pid >= np) phase = PH_CLAIM;      // padding ids of the item's last chunk
                        else left = (uint32_t)min((unsigned long long)left, np - pid);
                        seti(K_CELL, (uint32_t)lo);
                    }
                    if constexpr (SENSOR == kCamera) {
                        unsigned long long pix = pid / P.spp;
                        if (!LEARNED && P.pix_order) {
                            // claims walk the pixels in the given order (costly
                            // ones first); a path keeps its id, so its draws and
                            // its result do not depend on the order
                            const unsigned long long off = pid - pix * P.spp;
                            pix = __ldg(P.pix_order + pix);
                            pid = pix * P.spp + off;          // a chunk never straddles two pixels
                        }
                        seti(K_CELL, (uint32_t)pix);
                    }
                    set_pid(pid);
                    seti(K_LEFT, left);
                }
            }
        }
        if (!__any_sync(kFull, phase != PH_IDLE)) break;
        // ---- deadline / cancel, every 1024 steps ------------------------------
        if (budget <= 0) {
            budget = 1024;
            if (P.deadline_ns || P.cancel) {
                int stop = 0;
                if (lane == 0) {
                    if (P.cancel && *P.cancel) stop = 2;
                    else if (P.deadline_ns && globaltimer_ns() - t_start > P.deadline_ns) stop = 1;
                    const int others = *reinterpret_cast<volatile int*>(&P.work->status);
                    if (others) stop = others;
                }
                stop = __shfl_sync(kFull, stop, 0);
                if (stop) {
                    if (lane == 0) atomicMax(&P.work->status, stop);
                    break;
                }
            }
        }
        bool ran = phase >= PH_CLAIM && !(TERRAIN && phase == PH_WALK);
        if (COUNT) {
            if (ran) ++path_iters;
            const unsigned rr = __ballot_sync(kFull, ran);
            occ[4] += __popc(rr);
            occ[6] += rr ? 1 : 0;
            __syncwarp();
        }
        mark(0);

        // ---- the one Philox block of this pass ---------------------------------
        const DevScene& S = BATCH ? P.items[geti(K_CELL)].S : P.S;
        bool vert = phase == PH_VERTEX || phase == PH_GROUND;
        // ---- idle lanes take over the sun rays of this pass's vertices ----------
        const unsigned imask = __ballot_sync(kFull, phase == PH_IDLE), vmask = __ballot_sync(kFull, vert);
        bool handoff = false;             // this vertex's sun ray goes to a helper ...
        bool take = false;                // ... and this idle lane is one
        int mate = 0;                     // the helper's thread
        const bool pairing = vmask && (imask || helping);
        if (pairing) {
            const uint32_t q = geti(K_Q) & 7u;
            // (an owner whose helpers are all busy keeps the order of its sum)
            const unsigned wmask = __ballot_sync(kFull, vert && q < kMaxHelpers);
            const int rank = __popc((vert ? wmask : imask) & lt_mask);
            const int n = min(__popc(wmask), __popc(imask));
            handoff = vert && q < kMaxHelpers && rank < n;
            take = phase == PH_IDLE && rank < n;
            if (handoff) pairs[tid >> 5][0][rank] = (uint8_t)lane;
            if (take) {
                pairs[tid >> 5][1][rank] = (uint8_t)lane;
                seti(K_DONE, 2u);
            }
            __syncwarp();
            if (handoff) mate = (tid & ~31) + pairs[tid >> 5][1][rank];
            if (vert && !handoff && q) {
                seti(K_WANT, (uint32_t)phase);
                phase = PH_STALL;
                vert = false;
                ran = false;
            }
        }
        const uint32_t ev = geti(K_EV);
        const unsigned long long pid = get_pid();
        bool begin = phase == PH_BEGIN;   // start a ray now ...
        uint32_t tw = 0u;                 // ... whose first optical depth comes from this word
        float vx[3] = {0.0f, 0.0f, 0.0f}, nd[3] = {0.0f, 0.0f, 0.0f};
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (ran) {
            uint32_t xc2 = kind == kSunDirect ? 3u : ev << 2;     // PH_BEGIN: the ray's own block 0
            if (phase == PH_START) xc2 = 2u;
            else if (vert) xc2 = (ev << 2) | 1u;                   // the sun ray's block 0
            x = block(pid, xc2, 0u);
            tw = x.x;
            vx[0] = F(K_VX); vx[1] = F(K_VY); vx[2] = F(K_VZ);
            nd[0] = F(K_NX); nd[1] = F(K_NY); nd[2] = F(K_NZ);
        }
        mark(1);
        if (phase == PH_START) {
            seti(K_EV, 0u);
            F(K_W) = 1.0f;
            F(K_SCORE) = 0.0f;
            if constexpr (BATCH) {
                F(K_SG) = 0.0f; F(K_SVP) = 0.0f; F(K_CFS) = 0.0f; F(K_DSC) = 0.0f; F(K_SA) = 0.0f; F(K_DAL) = 0.0f;
            }
            if (LEARNED) seti(K_LV, 0u);
            if (COUNT) path_iters = 1;
            if constexpr (SENSOR == kCamera) {
                const uint32_t cell = geti(K_CELL);
                const int px = (int)(cell % (uint32_t)P.width), py = (int)(cell / (uint32_t)P.width);
                const float jx = 1.0f - u01(x.x), jy = 1.0f - u01(x.y);
                const float sx = (2.0f * ((float)px + jx) * P.inv_width - 1.0f) * P.tan_half;
                const float sy = (2.0f * ((float)py + jy) * P.inv_height - 1.0f) * P.tan_half * P.aspect;
                float d[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] = P.cam_f[a] + sx * P.cam_r[a] + sy * P.cam_u[a];
                const float inv = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
                float q[3] = {P.cam_pos[0], P.cam_pos[1], P.cam_pos[2]};
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] *= inv;
                bool enters = true;
                if (q[2] > P.Lz) {
                    if (d[2] < 0.0f) {
                        const float t = __fdividef(P.Lz - q[2], d[2]);
                        q[0] += t * d[0];
                        q[1] += t * d[1];
                        q[2] = P.Lz;
                    } else {
                        enters = false;
                    }
                } else if (q[2] < 0.0f) {
                    enters = false;
                }
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    q[a] -= floorf(__fdividef(q[a], S.Lper[a])) * S.Lper[a];
                    if (!(q[a] < S.Lper[a]) || q[a] < 0.0f) q[a] = 0.0f;
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) { vx[a] = q[a]; nd[a] = d[a]; }
                kind = kMain;
                if (enters) { begin = true; tw = x.z; }
                else phase = PH_END;           // a path that misses the field scores 0
            } else {
                vx[0] = (1.0f - u01(x.x)) * S.Lper[0];
                vx[1] = (1.0f - u01(x.y)) * S.Lper[1];
                vx[2] = 0.0f;
                if (!(vx[0] < S.Lper[0])) vx[0] = 0.0f;
                if (!(vx[1] < S.Lper[1])) vx[1] = 0.0f;
                kind = kSunDirect;
                phase = PH_BEGIN;      // (its four words used up: the ray starts in the next pass)
                F(K_TDIR) = 0.0f;
                if constexpr (TERRAIN) {
                    // the surface point above (x, y), lifted along its normal;
                    // directions cosine-weighted about the normal; the direct
                    // irradiance of the tilted element per horizontal area is
                    // max(n.s, 0) / (n_z mu0) T_sun, kept in tdir until T_sun
                    float n[3];
                    vx[2] = hf_height<TERRAIN == kRecords>(S, vx[0], vx[1], n);
#pragma unroll
                    for (int a = 0; a < 3; ++a) vx[a] += kTerrainOffset * n[a];
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        if (vx[a] < 0.0f) vx[a] += S.Lper[a];
                        if (!(vx[a] < S.Lper[a])) vx[a] -= S.Lper[a];
                        if (!(vx[a] >= 0.0f && vx[a] < S.Lper[a])) vx[a] = 0.0f;
                    }
                    cosine_about(n, u01(x.z), u01(x.w), nd);
                    F(K_FZ) = n[2];
                    const float ns = n[0] * S.sun[0] + n[1] * S.sun[1] + n[2] * S.sun[2];
                    F(K_TDIR) = __fdividef(fmaxf(ns, 0.0f), n[2] * S.sun[2]);
                    if (!(ns > 0.0f)) kind = kMain;      // self-shadowed: no direct sun ray
                } else {
                    cosine_up(u01(x.z), u01(x.w), nd);
                }
            }
            F(K_VX) = vx[0]; F(K_VY) = vx[1]; F(K_VZ) = vx[2];
            F(K_NX) = nd[0]; F(K_NY) = nd[1]; F(K_NZ) = nd[2];
            Ts = 1.0f;
        }
        mark(2);
        if (vert) {
            // weight, estimate factor toward the sun, new direction, roulette
            const float xi1 = u01(x.x), xi2 = u01(x.y), xr = u01(x.z);
            const int order = (int)ev + 1;
            const bool score_it = (P.max_order == 0) || (order <= P.max_order);
            float w = F(K_W), cf;
            if (phase == PH_VERTEX) {
                const float vk = F(K_VK);
                const float om = omega_at(S, vk);
                const float mu = R.d[0] * S.sun[0] + R.d[1] * S.sun[1] + R.d[2] * S.sun[2];
                float ph = hg_pdf(S.g, mu);
                float mu_new;
                if (DECOMP && S.rayleigh) {
                    // Rayleigh clear air: the mixture phase function in the estimate;
                    // the species sampled with word 0 of the flight's vertex block
                    const float pc = cloud_scatter_share(S, vk);
                    ph = pc * ph + (1.0f - pc) * rayleigh_pdf(mu);
                    const uint4 xs = block(pid, ev << 2, kBlockVertex);
                    mu_new = u01(xs.x) > pc ? rayleigh_sample_mu(xi1) : hg_sample_mu(S.g, xi1);
                } else {
                    mu_new = hg_sample_mu(S.g, xi1);
                }
                cf = score_it ? w * om * ph : 0.0f;
                w *= om;
                rotate_dir(R.d, mu_new, xi2, nd);
                if constexpr (BATCH) {
                    F(K_CFS) = hg_dlog_dg(S.g, mu);
                    F(K_SVP) = hg_dlog_dg(S.g, mu_new);
                    // d ln omega / d alpha = -k_cloud / (k omega) at this vertex
                    if (EXTRA && om > 0.0f) F(K_SA) -= __fdividef(fmaxf(vk - S.k_gas - S.k_clear, 0.0f), vk * om);
                }
                if (COUNT) cnt[C_REAL]++;
            } else if constexpr (TERRAIN) {
                // tilted ground: leave the surface along its normal, estimate
                // with n.s, scatter cosine-weighted about n
                float n[3];
                hf_height<TERRAIN == kRecords>(S, vx[0], vx[1], n);
#pragma unroll
                for (int a = 0; a < 3; ++a) vx[a] += kTerrainOffset * n[a];
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    if (vx[a] < 0.0f) vx[a] += S.Lper[a];
                    if (!(vx[a] < S.Lper[a])) vx[a] -= S.Lper[a];
                    if (!(vx[a] >= 0.0f && vx[a] < S.Lper[a])) vx[a] = 0.0f;
                }
                F(K_VX) = vx[0]; F(K_VY) = vx[1]; F(K_VZ) = vx[2];
                const float ns = n[0] * S.sun[0] + n[1] * S.sun[1] + n[2] * S.sun[2];
                cf = (score_it && ns > 0.0f) ? w * (S.albedo * (1.0f / kPi)) * ns : 0.0f;
                w *= S.albedo;
                cosine_about(n, xi1, xi2, nd);
                if (COUNT) cnt[C_GROUND]++;
            } else {
                cf = score_it ? w * (S.albedo * (1.0f / kPi)) * fmaxf(S.sun[2], 0.0f) : 0.0f;
                w *= S.albedo;
                cosine_up(xi1, xi2, nd);
                if constexpr (BATCH) { F(K_CFS) = 0.0f; F(K_SVP) = 0.0f; }
                if (COUNT) cnt[C_GROUND]++;
            }
            bool term_after = (P.max_order > 0) && (order >= P.max_order);
            if (!term_after && w < 0.01f) {
                if (xr * 0.01f <= w) w = 0.01f;
                else term_after = true;
            }
            if (term_after) seti(K_EV, ev | kTermAfter);
            F(K_W) = w;
            F(K_CF) = cf;
            F(K_NX) = nd[0]; F(K_NY) = nd[1]; F(K_NZ) = nd[2];
            // (a ground facet turned away from the sun sends no sun ray)
            kind = kSunLocal;
            const bool ray = score_it && (!TERRAIN || phase == PH_VERTEX || cf > 0.0f);
            if (handoff) {
                if (ray) {
                    cold[K_VX][mate] = vx[0]; cold[K_VY][mate] = vx[1]; cold[K_VZ][mate] = vx[2];
                    cold[K_PID_LO][mate] = F(K_PID_LO); cold[K_PID_HI][mate] = F(K_PID_HI);
                    cold[K_EV][mate] = __uint_as_float(ev);
                    cold[K_CELL][mate] = F(K_CELL);
                    cold[K_CF][mate] = cf;
                    cold[K_WORD][mate] = __uint_as_float(x.w);
                    cold[K_DONE][mate] = __uint_as_float(0u);
                    if constexpr (BATCH) {
                        cold[K_CFS][mate] = F(K_SG) + F(K_CFS);
                        if (EXTRA) cold[K_SA][mate] = F(K_SA);
                    }
                    const uint32_t q = geti(K_Q);
                    seti(K_Q, (q + 1u) | ((uint32_t)(mate & 31) << (3u + 5u * (q & 7u))));
                }
                if constexpr (BATCH) F(K_SG) += F(K_SVP);
                if (term_after) {
                    phase = PH_END;
                } else {
                    // the flight's own block 0
                    seti(K_EV, ev + 1u);
                    kind = kMain;
                    tw = block(pid, (ev + 1u) << 2, 0u).x;
                    begin = true;
                }
            } else if (ray) {
                Ts = 1.0f;
                begin = true;
                tw = x.w;        // word 3 of the vertex block
            } else {
                Ts = 0.0f;
                phase = PH_SUN_END;
            }
        }

        if constexpr (LEARNED) {
            if (phase == PH_RESUME) {
                // resume a path stopped at a learned vertex: state, network output,
                // one-sample MIS direction, weight p_HG / q
                const uint32_t slot = (uint32_t)pid;
                const uint4 q0 = P.qin[4 * (size_t)slot], q1 = P.qin[4 * (size_t)slot + 1];
                const uint4 q2 = P.qin[4 * (size_t)slot + 2], q3 = P.qin[4 * (size_t)slot + 3];
                const unsigned long long rpid = (unsigned long long)q0.x | ((unsigned long long)q0.y << 32);
                set_pid(rpid);
                const uint32_t rev = q0.z;
                vx[0] = __uint_as_float(q1.x); vx[1] = __uint_as_float(q1.y); vx[2] = __uint_as_float(q1.z);
                const float vk = __uint_as_float(q1.w);
                float rd[3] = {__uint_as_float(q2.x), __uint_as_float(q2.y), __uint_as_float(q2.z)};
                float w = __uint_as_float(q2.w);
                const float score = __uint_as_float(q3.x);
                F(K_SCORE) = score;
                if (SENSOR == kFlux) F(K_TDIR) = __uint_as_float(q3.y);
                if (SENSOR == kCamera) seti(K_CELL, (uint32_t)(rpid / P.spp));
                const uint4 xv = block(rpid, rev << 2, kBlockVertex);
                const uint4 xl = block(rpid, rev << 2, kBlockVertex - 1u);
                const float xi1 = u01(xv.x), xi2 = u01(xv.y), xr = u01(xv.z), xc = u01(xv.w), xlobe = u01(xl.x);
                const int order = (int)rev + 1;
                const bool score_it = (P.max_order == 0) || (order <= P.max_order);
                const float om = omega_at(S, vk);
                const float mu_s = rd[0] * S.sun[0] + rd[1] * S.sun[1] + rd[2] * S.sun[2];
                F(K_CF) = score_it ? w * om * hg_pdf(S.g, mu_s) : 0.0f;
                const float* mix = P.qin_mix + 48 * (size_t)slot;
                if (xc <= P.mis_alpha) {
                    rotate_dir(rd, hg_sample_mu(S.g, xi1), xi2, nd);
                } else {
                    int j = 7;
#pragma unroll
                    for (int i = 0; i < 7; ++i)
                        if (j == 7 && xlobe <= __ldg(mix + 6 * i + 4)) j = i;
                    const float mu_l[3] = {__ldg(mix + 6 * j), __ldg(mix + 6 * j + 1), __ldg(mix + 6 * j + 2)};
                    const float kap = __ldg(mix + 6 * j + 3);
                    float cw = 1.0f + __logf(xi1 + (1.0f - xi1) * __expf(-2.0f * kap)) / kap;
                    cw = fminf(fmaxf(cw, -1.0f), 1.0f);
                    rotate_dir(mu_l, cw, xi2, nd);
                }
                const float phg = hg_pdf(S.g, rd[0] * nd[0] + rd[1] * nd[1] + rd[2] * nd[2]);
                // mixture density: sum of pi_j C(kappa_j) exp(kappa_j (mu_j . w - 1))
                float qv = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float c = __ldg(mix + 6 * i) * nd[0] + __ldg(mix + 6 * i + 1) * nd[1] + __ldg(mix + 6 * i + 2) * nd[2];
                    qv += __ldg(mix + 6 * i + 5) * __expf(__ldg(mix + 6 * i + 3) * (c - 1.0f));
                }
                const float qmix = P.mis_alpha * phg + (1.0f - P.mis_alpha) * qv;
                // training record: features, direction, score so far, w * omega
                if (P.rec_count && slot < P.rec_slots) {
                    const unsigned idx = atomicAdd(P.rec_count, 1u);
                    if (idx < P.rec_cap) {
                        P.rec_feat[2 * (size_t)idx] = P.qin_feat[2 * (size_t)slot];
                        P.rec_feat[2 * (size_t)idx + 1] = P.qin_feat[2 * (size_t)slot + 1];
                        P.rec_dir[3 * (size_t)idx] = nd[0];
                        P.rec_dir[3 * (size_t)idx + 1] = nd[1];
                        P.rec_dir[3 * (size_t)idx + 2] = nd[2];
                        P.rec_val[4 * (size_t)idx] = score;
                        P.rec_val[4 * (size_t)idx + 1] = w * om;
                        P.rec_val[4 * (size_t)idx + 2] = 0.0f;
                        P.rec_val[4 * (size_t)idx + 3] = __uint_as_float((uint32_t)(rpid - P.path_base));
                        seti(K_REC, idx);
                    }
                }
                w *= om * __fdividef(phg, fmaxf(qmix, 1e-30f));
                seti(K_LV, q0.w + 1u);
                if (COUNT) cnt[C_REAL]++;
                bool term_after = (P.max_order > 0) && (order >= P.max_order);
                if (!term_after && w < 0.01f) {
                    if (xr * 0.01f <= w) w = 0.01f;
                    else term_after = true;
                }
                seti(K_EV, term_after ? rev | kTermAfter : rev);
                F(K_W) = w;
                F(K_VX) = vx[0]; F(K_VY) = vx[1]; F(K_VZ) = vx[2];
                F(K_NX) = nd[0]; F(K_NY) = nd[1]; F(K_NZ) = nd[2];
                kind = kSunLocal;
                if (score_it) {
                    Ts = 1.0f;
                    begin = true;
                    tw = xl.y;       // word 1 of the lobe block
                } else {
                    Ts = 0.0f;
                    phase = PH_SUN_END;
                }
            }
        }
        if (pairing) {
            __syncwarp();
            if (take && geti(K_DONE) == 0u) {
                vx[0] = F(K_VX); vx[1] = F(K_VY); vx[2] = F(K_VZ);
                tw = geti(K_WORD);
                kind = kSunHelp;
                Ts = 1.0f;
                begin = true;
            }
            helping = __any_sync(kFull, (geti(K_Q) & 7u) != 0u);
        }
        mark(5);
        // (a helper works on its owner's batch item)
        const DevScene& Z = BATCH ? P.items[geti(K_CELL)].S : P.S;
        // ---- ray starts: a camera path start or a vertex goes on into the
        //      ray it set up (its first optical depth a word of the block
        //      already drawn); a flight that follows a sun ray, and a flux
        //      path's direct sun ray, draw their own block ---------------------
        if (begin) {
            // the flight from vx along nd, or the sun ray from vx
            int v[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float d = (kind == kMain) ? nd[a] : Z.sun[a];
                R.o[a] = vx[a];
                R.d[a] = d;
                v[a] = locate(vx[a], d, Z.h[a], Z.inv_h[a], 0, Z.nm1[a]);
            }
            const uint2 e = __ldg(leaf_entry(Z, v));
#pragma unroll
            for (int a = 0; a < 3; ++a) R.inv_d[a] = (kind == kMain) ? dir_rcp(nd[a]) : Z.inv_sun[a];
            R.t = 0.0f;
            R.steps = 0;
            tau = -__logf(u01(tw));
            blk = 1;
            phase = PH_STEP;
            if constexpr (TERRAIN) {
                // a sun ray that meets the surface is shadowed (only one that starts
                // inside the relief layer can); a flight ends at the surface, found
                // first when it starts inside the relief layer, else once its
                // traversal reaches z = hmax
                tg = kInf;
                tpend = kInf;
                if (!(R.o[2] > Z.hmax)) phase = PH_WALK;
                else if (kind == kMain && R.d[2] < 0.0f) tpend = __fdiv_rn(Z.hmax - R.o[2], R.d[2]);
            }
            finish_leaf<BF16>(Z, R, v, e);
            if (COUNT) {
                if (kind == kMain) cnt[C_FLIGHTS]++;
                else cnt[C_SUN_RAYS]++;
            }
        }
        if constexpr (TERRAIN) {
            // ---- walks over the heightfield wait until kWalkBatch lanes walk
            //      together or too few lanes step to wait any longer -----------------
            const unsigned walkers = __ballot_sync(kFull, phase == PH_WALK);
            const int steppers = __popc(__ballot_sync(kFull, phase == PH_STEP));
            if (__popc(walkers) >= kWalkBatch || (walkers && steppers < P.min_steppers)) {
                if (phase == PH_WALK) {
                    const float th = terrain_hit<TERRAIN == kRecords>(Z, R.o, R.d);
                    phase = PH_STEP;
                    if (kind == kMain) {
                        tg = th;
                    } else if (th < kInf) {
                        Ts = 0.0f;
                        phase = PH_SUN_END;
                    }
                }
            }
        }
        __syncwarp();
        mark(3);

        // ==== steps: until enough lanes wait for a rare pass ====================
        unsigned stepping;
        do {
#pragma unroll
            for (int half = 0; half < kSteps; ++half) {
                // (heightfield: a flight whose current leaf reaches down into the relief
                //  layer first finds its ground hit, in a rare pass)
                if (TERRAIN && phase == PH_STEP && R.texit >= tpend) {
                    phase = PH_WALK;
                    tpend = kInf;
                }
                if (COUNT) {
                    const unsigned st = __ballot_sync(kFull, phase == PH_STEP), lv = __ballot_sync(kFull, phase != PH_IDLE);
                    occ[0] += 1; occ[1] += __popc(lv); occ[2] += __popc(st); occ[5] += __popc(lv) - __popc(st);
                    occ[7] += 32 - __popc(lv);
                    if (phase == PH_STEP) ++path_iters;
                }
                if (phase == PH_STEP) {
                    // one step: to the tentative collision inside the leaf, or across
                    // the leaf's exit face; both share the point and voxel arithmetic.
                    // Tracking majorant: the leaf's M, or M - m for a sun ray in
                    // decomposition tracking (the minorant m is applied exactly)
                    const bool decomp = DECOMP && kind != kMain && P.sun_mode == MCRT_SUN_DECOMP;
                    const float Mt = decomp ? R.M - R.mn : R.M;
                    const float te = TERRAIN ? fminf(R.texit, tg) : R.texit;
                    const float Mseg = Mt * (te - R.t);
                    const bool tent = Mt > 0.0f && tau < Mseg;
                    const bool at_ground = TERRAIN && !tent && tg <= R.texit;   // the surface cuts this leaf
                    const float tn = tent ? fminf(R.t + __fdividef(tau, Mt), te) : (at_ground ? tg : R.texit);
                    if (decomp) Ts *= __expf(-R.mn * (tn - R.t));   // the control over this piece of the leaf
                    float p[3];
                    int nv[3];
                    advance(Z, R, tn, !tent && !at_ground, p, nv);
                    const bool face = !tent && !at_ground;
                    int st = kInside;
                    uint2 e = make_uint2(0u, 0u);
                    if (face) {
                        tau -= Mseg;
                        float wdt;
                        st = cross_face(Z, R, p, nv, &wdt);
                        if (TERRAIN) { tg -= wdt; tpend -= wdt; }   // a periodic wrap restarts the segment
                        if (st == kInside) e = __ldg(leaf_entry(Z, nv));
                    }
                    if (tent) R.t = tn;
                    // the block of a tentative collision, or of the roulette at a leaf
                    // crossing of decomposition tracking (word 3, which uses it up)
                    const bool roulette = DECOMP && decomp && face && st == kInside && Ts < 0.1f;
                    const bool loads = tent && R.msk != 0;
                    if (COUNT && tent) {
                        ++tents;
                        if (kind == kMain) cnt[C_TENT]++;
                        else cnt[C_SUN_TENT]++;
                    }
                    uint4 x = make_uint4(0u, 0u, 0u, 0u);
                    if (loads || roulette) {
                        float k = 0.0f;
                        if (!DECOMP || loads) k = __fadd_rn(kfetch<BF16>(Z, nv[0], nv[1], nv[2]), Z.k_gas);
                        const uint32_t ev = geti(K_EV) & ~kTermAfter;
                        x = block(get_pid(), kind == kMain ? ev << 2 : (kind == kSunDirect ? 3u : (ev << 2) | 1u), blk);
                        ++blk;
                        if (!DECOMP || loads) {
                            const float u0 = u01(x.x);
                            if (kind == kMain) {
                                if (u0 * R.M <= k) {
                                    F(K_VK) = k;
                                    phase = PH_REAL;
                                    if (LEARNED) { seti(K_NX, (uint32_t)nv[0]); seti(K_NY, (uint32_t)nv[1]); seti(K_NZ, (uint32_t)nv[2]); }
                                }
                            } else if (P.sun_mode == MCRT_SUN_DELTA) {
                                if (u0 * R.M <= k) { Ts = 0.0f; phase = PH_SUN_END; }
                            } else {
                                Ts *= decomp ? null_share<!EXTRA>(k - R.mn, R.M - R.mn) : null_share<!EXTRA>(k, R.M);
                                if (!(Ts > 0.0f)) {
                                    Ts = 0.0f;
                                    phase = PH_SUN_END;
                                } else if (Ts < 0.1f) {
                                    if (u0 * 0.1f <= Ts) Ts = 0.1f;
                                    else { Ts = 0.0f; phase = PH_SUN_END; }
                                }
                            }
                            tau = -__logf(u01(x.y));
                        }
                    }
                    if (tent) {
                        if (!loads) phase = PH_HIT;
                    } else if (at_ground) {
                        R.t = tg;
                        phase = PH_LAND;
                    } else if (st == kInside) {
                        if (roulette) {
                            if (u01(x.w) * 0.1f <= Ts) Ts = 0.1f;
                            else { Ts = 0.0f; phase = PH_SUN_END; }
                        }
                        if (!roulette || phase == PH_STEP) {
                            if (COUNT) {
                                if (kind == kMain) cnt[C_LEAF]++;
                                else cnt[C_SUN_LEAF]++;
                            }
                            finish_leaf<BF16>(Z, R, nv, e);
                            if (R.steps > P.max_steps) {
                                if (COUNT) cnt[C_ABORT]++;
                                Ts = 0.0f;
                                phase = kind == kMain ? PH_END : PH_SUN_END;
                            }
                        }
                    } else if (kind != kMain) {
                        if (st == kGround) Ts = 0.0f;
                        phase = PH_SUN_END;
                    } else if (st == kTop) {
                        phase = PH_END;
                    } else {
                        phase = PH_FLOOR;
                    }
                }
            }
            stepping = __ballot_sync(kFull, phase == PH_STEP);
            budget -= kSteps;
        } while (stepping && budget > 0 &&
                 (__popc(stepping) >= P.min_steppers || !__any_sync(kFull, phase >= PH_CLAIM)));
        mark(4);
    }

    // ---- the warp's sums, and partial ones left by a deadline / cancel exit ----
    spill_sums();
    {
#pragma unroll
        for (int q = 0; q < 2 * NQ; ++q)
            if (F(K_ACC + q) != 0.0f)
                atomicAdd(((q & 1) ? P.s2 : P.s1) + (size_t)geti(K_CELL) * NQ + (q >> 1), (double)F(K_ACC + q));
    }
    if (COUNT) {
#pragma unroll
        for (int q = 0; q < kCounters; ++q) {
            unsigned long long a = cnt[q];
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
            if (lane == 0 && a) atomicAdd(P.counters + q, a);
        }
        unsigned long long nt = tents;
        for (int o = 16; o > 0; o >>= 1) nt += __shfl_xor_sync(kFull, nt, o);
        if (lane == 0) atomicAdd(P.counters + C_OCC + 3, nt);
        unsigned mi = max_iters;
        for (int o = 16; o > 0; o >>= 1) mi = max(mi, __shfl_xor_sync(kFull, mi, o));
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < kSections; ++q) atomicAdd(P.counters + C_SEC + q, sec[q]);
#pragma unroll
            for (int q = 0; q < kOcc; ++q)
                if (q != 3) atomicAdd(P.counters + C_OCC + q, occ[q]);
            const uint64_t t_end = globaltimer_ns();
            atomicMax(P.counters + C_MAX_ITERS, (unsigned long long)mi);
            if (t_dry) atomicMax(P.counters + C_T_DRY, (unsigned long long)(t_dry - t_start));
            atomicMax(P.counters + C_T_END, (unsigned long long)(t_end - t_start));
        }
    }
}

// Mean and standard error of each tally entry from its FP64 sums, all means
// first, so that each array goes to the caller's in one copy; a batch passes
// each cell's own path count (cell_n, nq entries per cell).
__global__ void finalize_kernel(const double* __restrict__ s1, const double* __restrict__ s2, double n_all, int count,
                                const unsigned long long* __restrict__ cell_n, int nq, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double n = cell_n ? (double)cell_n[i / nq] : n_all;
    const double m = s1[i] / n;
    double var = s2[i] / n - m * m;
    if (var < 0.0) var = 0.0;
    out[i] = m;
    out[(size_t)count + i] = n > 1.0 ? sqrt(var / (n - 1.0)) : 0.0;
}

// One thread walks one ray and records its leaves (traversal check), with
// the same device functions as the tracer.
template <bool BF16>
__global__ void debug_dda_kernel(DevScene S, float ox, float oy, float oz, float dx, float dy, float dz, int cap,
                                 int* cells, float* tio, int* count_status)
{
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    Ray R;
    const float p0[3] = {ox, oy, oz}, d[3] = {dx, dy, dz};
    ray_begin<BF16>(S, R, p0, d);
    float tbase = 0.0f;
    int n = 0, status = 0;
    for (;;) {
        if (n >= cap) { status = 3; break; }
        const int lev = __popc((unsigned)R.msk);
        cells[4 * n + 0] = lev / S.lb;        // level of the tracked grid
        cells[4 * n + 1] = R.lo[0] >> lev;
        cells[4 * n + 2] = R.lo[1] >> lev;
        cells[4 * n + 3] = R.lo[2] >> lev;
        tio[2 * n + 0] = __fadd_rn(tbase, R.t);
        tio[2 * n + 1] = __fadd_rn(tbase, R.texit);
        ++n;
        float wdt, p[3];
        int v[3];
        const int st = step_face(S, R, p, v, &wdt);
        if (wdt != 0.0f) tbase = __fadd_rn(tbase, wdt);
        if (st == kTop) { status = 1; break; }
        if (st == kGround) { status = 2; break; }
        finish_leaf<BF16>(S, R, v, __ldg(leaf_entry(S, v)));
        if (R.steps > (1u << 22)) { status = 4; break; }
    }
    count_status[0] = n;
    count_status[1] = status;
}

// Claim order of a camera trace: the cost of each tile of kOrderTile^2
// pixels is estimated by the majorant optical depth along the view ray
// through the tile's centre (the sum of M times the length over the leaves
// it crosses, capped): paths that enter thick cloud scatter many times and
// run longest.  Tracing the costly tiles first leaves cheap paths for the
// end of the launch, where a long path would otherwise run alone.
constexpr int kOrderTile = 8;

template <bool BF16>
__global__ void view_cost_kernel(TraceParams P, int tiles_x, int tiles_y, float* __restrict__ cost)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= tiles_x * tiles_y) return;
    const DevScene& S = P.S;
    const float cx = fminf((float)((i % tiles_x) * kOrderTile) + 0.5f * kOrderTile, (float)P.width - 0.5f);
    const float cy = fminf((float)((i / tiles_x) * kOrderTile) + 0.5f * kOrderTile, (float)P.height - 0.5f);
    const float sx = (2.0f * cx * P.inv_width - 1.0f) * P.tan_half;
    const float sy = (2.0f * cy * P.inv_height - 1.0f) * P.tan_half * P.aspect;
    float d[3], q[3] = {P.cam_pos[0], P.cam_pos[1], P.cam_pos[2]};
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = P.cam_f[a] + sx * P.cam_r[a] + sy * P.cam_u[a];
    const float inv = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] *= inv;
    float c = 0.0f;
    bool enters = true;
    if (q[2] > P.Lz) {
        if (d[2] < 0.0f) {
            const float t = (P.Lz - q[2]) / d[2];
            q[0] += t * d[0];
            q[1] += t * d[1];
            q[2] = P.Lz;
        } else {
            enters = false;
        }
    } else if (q[2] < 0.0f) {
        enters = false;
    }
    if (enters) {
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            q[a] -= floorf(q[a] / S.Lper[a]) * S.Lper[a];
            if (!(q[a] < S.Lper[a]) || q[a] < 0.0f) q[a] = 0.0f;
        }
        Ray R;
        ray_begin<BF16>(S, R, q, d);
        for (int n = 0; n < 4096 && c < 1e4f; ++n) {
            c += R.M * (R.texit - R.t);
            float wdt, p[3];
            int v[3];
            const int st = step_face(S, R, p, v, &wdt);
            if (st != kInside) break;
            finish_leaf<BF16>(S, R, v, __ldg(leaf_entry(S, v)));
        }
    }
    cost[i] = c;
}

// Tiles by cost, largest first, ties in raster order (a NaN cost counts as the
// largest), and the pixels before each: one block sorts up to kSortTiles keys
// in shared memory by a bitonic network, ~cost bits above the tile's index.
// One block, so bound by its 105 barriers at 16,384 tiles (a 1024 x 1024
// image), which is what 128 KB of keys hold; larger images sort on the host,
// where the copies and two waits cost more the smaller the trace is: a
// 1023 x 767 x 15 octree image took 30.44 ms that way and 30.02 ms this way,
// a 500 x 301 x 16 one 10.36 and 10.29.
constexpr int kSortTiles = 16384;

__global__ void __launch_bounds__(1024) sort_tiles_kernel(const float* __restrict__ cost, int n, int n2, int tiles_x,
                                                          int width, int height, uint32_t* __restrict__ tiles,
                                                          uint32_t* __restrict__ prefix)
{
    extern __shared__ unsigned long long key[];
    __shared__ uint32_t warp_sum[32];
    const int tid = threadIdx.x;
    for (int i = tid; i < n2; i += 1024) {
        unsigned long long k = ~0ull;                      // padding: last
        if (i < n) {
            const float c = cost[i];
            const float v = c > 0.0f ? c : c == 0.0f ? 0.0f : 3.0e38f;      // (-0 sorts as 0)
            k = ((unsigned long long)~__float_as_uint(v) << 32) | (uint32_t)i;
        }
        key[i] = k;
    }
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1)
        for (int d = size >> 1; d > 0; d >>= 1) {
            for (int q = tid; q < n2 / 2; q += 1024) {
                const int a = 2 * q - (q & (d - 1)), b = a + d;
                const unsigned long long x = key[a], y = key[b];
                if ((x > y) == ((a & size) == 0)) {
                    key[a] = y;
                    key[b] = x;
                }
            }
            __syncthreads();
        }
    // pixels before each tile: an exclusive scan, 1024 tiles at a time
    uint32_t base = 0;
    for (int i0 = 0; i0 < n; i0 += 1024) {
        const int i = i0 + tid;
        uint32_t tile = 0, px = 0;
        if (i < n) {
            tile = (uint32_t)key[i];
            const int x0 = (int)(tile % (uint32_t)tiles_x) * kOrderTile, y0 = (int)(tile / (uint32_t)tiles_x) * kOrderTile;
            px = (uint32_t)(min(kOrderTile, width - x0) * min(kOrderTile, height - y0));
        }
        uint32_t incl = px;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, o);
            if ((tid & 31) >= o) incl += v;
        }
        if ((tid & 31) == 31) warp_sum[tid >> 5] = incl;
        __syncthreads();
        uint32_t before = base, all = base;
        for (int w = 0; w < 32; ++w) {
            if (w < (tid >> 5)) before += warp_sum[w];
            all += warp_sum[w];
        }
        if (i < n) {
            tiles[i] = tile;
            prefix[i] = before + incl - px;
        }
        base = all;
        __syncthreads();
    }
}

// order[prefix[b] + j] = the j-th pixel (row-major inside the tile) of the
// b-th tile in claim order.
// One shard of a claim order: out[i] = order[i * stride + offset] (the
// identity order when order is NULL).
__global__ void shard_order_kernel(const uint32_t* __restrict__ order, uint32_t n_out, uint32_t stride,
                                   uint32_t offset, uint32_t* __restrict__ out)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_out) return;
    const uint32_t j = i * stride + offset;
    out[i] = order ? order[j] : j;
}

__global__ void expand_order_kernel(const uint32_t* __restrict__ tiles, const uint32_t* __restrict__ prefix, int n,
                                    int tiles_x, int width, int height, uint32_t* __restrict__ order)
{
    const int b = blockIdx.x;
    if (b >= n) return;
    const uint32_t tile = tiles[b];
    const int x0 = (int)(tile % (uint32_t)tiles_x) * kOrderTile, y0 = (int)(tile / (uint32_t)tiles_x) * kOrderTile;
    const int tw = min(kOrderTile, width - x0), th = min(kOrderTile, height - y0);
    const int t = threadIdx.x;
    if (t >= tw * th) return;
    const int tx = t % tw, ty = t / tw;
    order[prefix[b] + t] = (uint32_t)((y0 + ty) * width + x0 + tx);
}

// One thread per ray: the heightfield hit distance (terrain check).
__global__ void debug_terrain_kernel(DevScene S, const float* __restrict__ o, const float* __restrict__ d, int n,
                                     float* __restrict__ t)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float oo[3] = {o[3 * i], o[3 * i + 1], o[3 * i + 2]};
    const float dd[3] = {d[3 * i], d[3 * i + 1], d[3 * i + 2]};
    t[i] = S.hrec ? terrain_hit<true>(S, oo, dd) : terrain_hit<false>(S, oo, dd);
}

// One thread per point: surface height and normal (z, nx, ny, nz).
__global__ void debug_terrain_height_kernel(DevScene S, const float* __restrict__ xy, int n, float* __restrict__ zn)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float nn[3];
    zn[4 * i] = S.hrec ? hf_height<true>(S, xy[2 * i], xy[2 * i + 1], nn) : hf_height<false>(S, xy[2 * i], xy[2 * i + 1], nn);
    zn[4 * i + 1] = nn[0]; zn[4 * i + 2] = nn[1]; zn[4 * i + 3] = nn[2];
}

__global__ void debug_philox_kernel(const uint32_t* __restrict__ ctr, const uint32_t* __restrict__ key,
                                    uint32_t* __restrict__ out, size_t n)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 r = philox4x32_10(c, make_uint2(key[2 * i], key[2 * i + 1]));
    out[4 * i] = r.x; out[4 * i + 1] = r.y; out[4 * i + 2] = r.z; out[4 * i + 3] = r.w;
}

template <int SENSOR, bool BF16, bool COUNT, bool LEARNED, int TERRAIN = kFlat, bool EXTRA = false>
const void* kernel_ptr()
{
    return reinterpret_cast<const void*>(&trace_kernel<SENSOR, BF16, COUNT, LEARNED, false, TERRAIN, EXTRA>);
}

template <int TERRAIN, bool DECOMP>
const void* pick_t(int sensor, bool bf16, bool count)
{
    if (sensor == kCamera) {
        if (bf16) return count ? kernel_ptr<kCamera, true, true, false, TERRAIN, DECOMP>()
                               : kernel_ptr<kCamera, true, false, false, TERRAIN, DECOMP>();
        return count ? kernel_ptr<kCamera, false, true, false, TERRAIN, DECOMP>()
                     : kernel_ptr<kCamera, false, false, false, TERRAIN, DECOMP>();
    }
    if (bf16) return count ? kernel_ptr<kFlux, true, true, false, TERRAIN, DECOMP>()
                           : kernel_ptr<kFlux, true, false, false, TERRAIN, DECOMP>();
    return count ? kernel_ptr<kFlux, false, true, false, TERRAIN, DECOMP>()
                 : kernel_ptr<kFlux, false, false, false, TERRAIN, DECOMP>();
}

// Kernel of a plain trace: sensor, storage, counting, heightfield ground and
// whether decomposition tracking or Rayleigh clear air is in use (those have
// variants of their own, so the others keep their registers).
template <bool EXTRA>
const void* pick_g(int sensor, bool bf16, bool count, const DevScene& S)
{
    if (!S.hf) return pick_t<kFlat, EXTRA>(sensor, bf16, count);
    return S.hrec ? pick_t<kRecords, EXTRA>(sensor, bf16, count) : pick_t<kHeights, EXTRA>(sensor, bf16, count);
}

const void* pick(int sensor, bool bf16, bool count, const DevScene& S, bool extra)
{
    return extra ? pick_g<true>(sensor, bf16, count, S) : pick_g<false>(sensor, bf16, count, S);
}

template <bool DALPHA>
const void* pick_batch_t(bool bf16, bool count)
{
    if (count)
        return bf16 ? reinterpret_cast<const void*>(&trace_kernel<kFlux, true, true, false, true, kFlat, DALPHA>)
                    : reinterpret_cast<const void*>(&trace_kernel<kFlux, false, true, false, true, kFlat, DALPHA>);
    return bf16 ? reinterpret_cast<const void*>(&trace_kernel<kFlux, true, false, false, true, kFlat, DALPHA>)
                : reinterpret_cast<const void*>(&trace_kernel<kFlux, false, false, false, true, kFlat, DALPHA>);
}

const void* pick_batch(bool bf16, bool count, bool dalpha)
{
    return dalpha ? pick_batch_t<true>(bf16, count) : pick_batch_t<false>(bf16, count);
}

const void* pick_learned(int sensor, bool bf16)
{
    if (sensor == kCamera) return bf16 ? kernel_ptr<kCamera, true, false, true>() : kernel_ptr<kCamera, false, false, true>();
    return bf16 ? kernel_ptr<kFlux, true, false, true>() : kernel_ptr<kFlux, false, false, true>();
}

// Target weight of each training record: the radiance its sampled direction
// brought back, (final score - score before the vertex - the vertex's own
// local estimate) / (w * omega).
__global__ void targets_kernel(const float* __restrict__ rec_val, const float* __restrict__ final_score, unsigned n,
                               float* __restrict__ tgt)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 v = reinterpret_cast<const float4*>(rec_val)[i];
    const float fin = final_score[__float_as_uint(v.w)];
    const float t = v.y > 0.0f ? (fin - v.x - v.z) / v.y : 0.0f;
    tgt[i] = fmaxf(t, 0.0f);
}

}  // namespace

cudaError_t launch_trace(const TraceParams& P, int sensor, bool bf16, bool count, int grid, int block,
                         cudaStream_t st)
{
    void* args[] = {const_cast<TraceParams*>(&P)};
    const bool extra = P.sun_mode == MCRT_SUN_DECOMP || P.S.rayleigh;
    return cudaLaunchKernel(pick(sensor, bf16, count, P.S, extra), dim3(grid), dim3(block), args, 0, st);
}

cudaError_t launch_trace_learned(const TraceParams& P, int sensor, bool bf16, int grid, int block, cudaStream_t st)
{
    void* args[] = {const_cast<TraceParams*>(&P)};
    return cudaLaunchKernel(pick_learned(sensor, bf16), dim3(grid), dim3(block), args, 0, st);
}

int trace_learned_blocks_per_sm(int sensor, bool bf16, int block)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick_learned(sensor, bf16), block, 0) != cudaSuccess) return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_trace_batch(const TraceParams& P, bool bf16, bool count, bool dalpha, int grid, int block,
                               cudaStream_t st)
{
    void* args[] = {const_cast<TraceParams*>(&P)};
    return cudaLaunchKernel(pick_batch(bf16, count, dalpha), dim3(grid), dim3(block), args, 0, st);
}

int trace_batch_blocks_per_sm(bool bf16, bool count, bool dalpha, int block)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick_batch(bf16, count, dalpha), block, 0) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_targets(const float* rec_val, const float* final_score, unsigned n, float* tgt, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    targets_kernel<<<(n + 255) / 256, 256, 0, st>>>(rec_val, final_score, n, tgt);
    return cudaGetLastError();
}

int trace_blocks_per_sm(int sensor, bool bf16, bool count, const DevScene& S, bool extra, int block)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick(sensor, bf16, count, S, extra), block, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

cudaError_t launch_finalize(const double* s1, const double* s2, double n, int count, const unsigned long long* cell_n,
                            int nq, double* out, cudaStream_t st)
{
    finalize_kernel<<<(count + 255) / 256, 256, 0, st>>>(s1, s2, n, count, cell_n, nq, out);
    return cudaGetLastError();
}

cudaError_t launch_debug_dda(const DevScene& S, const float* o, const float* d, int cap, int* cells, float* tio,
                             int* count_status, bool bf16, cudaStream_t st)
{
    if (bf16)
        debug_dda_kernel<true><<<1, 32, 0, st>>>(S, o[0], o[1], o[2], d[0], d[1], d[2], cap, cells, tio,
                                                  count_status);
    else
        debug_dda_kernel<false><<<1, 32, 0, st>>>(S, o[0], o[1], o[2], d[0], d[1], d[2], cap, cells, tio,
                                                   count_status);
    return cudaGetLastError();
}

// Bounds-checked build: read (and clear) this unit's violation word.
bool bounds_checked_build()
{
#ifdef MCRT_CHECKED
    return true;
#else
    return false;
#endif
}

cudaError_t read_bounds_violations(unsigned* count, unsigned* first_code)
{
    *count = 0;
    *first_code = 0;
#ifdef MCRT_CHECKED
    unsigned h[2] = {0, 0};
    cudaError_t e = cudaMemcpyFromSymbol(h, g_mcrt_bounds, sizeof(h));
    if (e != cudaSuccess) return e;
    const unsigned zero[2] = {0, 0};
    e = cudaMemcpyToSymbol(g_mcrt_bounds, zero, sizeof(zero));
    *count = h[0];
    *first_code = h[1];
    return e;
#else
    return cudaSuccess;
#endif
}

int order_tiles(int width, int height, int* tiles_x)
{
    *tiles_x = (width + kOrderTile - 1) / kOrderTile;
    return *tiles_x * ((height + kOrderTile - 1) / kOrderTile);
}

cudaError_t launch_view_cost(const TraceParams& P, bool bf16, float* cost, cudaStream_t st)
{
    int tx = 0;
    const int n = order_tiles(P.width, P.height, &tx);
    const int ty = n / tx;
    if (bf16) view_cost_kernel<true><<<(n + 127) / 128, 128, 0, st>>>(P, tx, ty, cost);
    else view_cost_kernel<false><<<(n + 127) / 128, 128, 0, st>>>(P, tx, ty, cost);
    return cudaGetLastError();
}

bool sorts_on_device(int n) { return n <= kSortTiles; }

cudaError_t launch_sort_tiles(const float* cost, int n, int width, int height, uint32_t* tiles, uint32_t* prefix,
                              cudaStream_t st)
{
    int tx = 0, n2 = 2;
    order_tiles(width, height, &tx);
    while (n2 < n) n2 <<= 1;
    const size_t smem = (size_t)n2 * sizeof(unsigned long long);
    cudaError_t e = cudaFuncSetAttribute(sort_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSortTiles * (int)sizeof(unsigned long long));
    if (e != cudaSuccess) return e;
    sort_tiles_kernel<<<1, 1024, smem, st>>>(cost, n, n2, tx, width, height, tiles, prefix);
    return cudaGetLastError();
}

cudaError_t launch_shard_order(const uint32_t* order, uint32_t n_out, uint32_t stride, uint32_t offset,
                               uint32_t* out, cudaStream_t st)
{
    if (n_out == 0) return cudaSuccess;
    shard_order_kernel<<<(n_out + 255) / 256, 256, 0, st>>>(order, n_out, stride, offset, out);
    return cudaGetLastError();
}

cudaError_t launch_expand_order(const uint32_t* tiles, const uint32_t* prefix, int n, int width, int height,
                                uint32_t* order, cudaStream_t st)
{
    int tx = 0;
    order_tiles(width, height, &tx);
    expand_order_kernel<<<n, kOrderTile * kOrderTile, 0, st>>>(tiles, prefix, n, tx, width, height, order);
    return cudaGetLastError();
}

cudaError_t launch_debug_terrain(const DevScene& S, const float* o, const float* d, int n, float* t, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    debug_terrain_kernel<<<(n + 127) / 128, 128, 0, st>>>(S, o, d, n, t);
    return cudaGetLastError();
}

cudaError_t launch_debug_terrain_height(const DevScene& S, const float* xy, int n, float* zn, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    debug_terrain_height_kernel<<<(n + 127) / 128, 128, 0, st>>>(S, xy, n, zn);
    return cudaGetLastError();
}

cudaError_t launch_debug_philox(const uint32_t* ctr, const uint32_t* key, uint32_t* out, size_t n, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    debug_philox_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(ctr, key, out, n);
    return cudaGetLastError();
}

}  // namespace mcrt
