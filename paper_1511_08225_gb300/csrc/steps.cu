// steps.cu -- many timesteps of a 1D simulation in one launch, up to some 7 million slots.
//
// A step of the three kernels of kernels.cu takes 28 us however few particles there are:
// launches, the ramp of a one-CTA-per-SM grid, a cluster launch for the field, and global
// round trips between them.  Here one cooperative launch runs the steps.  Every CTA (one
// per SM, leaving one SM free for overlapped read-backs) pushes its share of the slots as
// k_particles does, walks the pushes that need iteration from a list of its own in shared
// memory, and adds its charge to a global accumulator; then comes the step's grid barrier;
// then every CTA makes the field for itself: it reads the summed deposit, adds the source
// particles' (made from their counters by every CTA, and stored by the one that pushes them
// next; a large source is made in shares and has a barrier of its own) and solves for E as
// k_field does, with the same integers and the same FP64 operations.  Nothing else of a step
// crosses CTAs, so 256 cells and 51,200 particles step in 12 us, 100 cells and 1.4e5 in 13.
//
// Particles, deposits, fields and counters are those of the three kernels bit for bit.
// The accumulators, the absorbed counts and a compacting step's output counts go by three
// turns: a turn's are added to before the barrier, read after it, and cleared before the
// barrier of the step after (when every CTA has passed the barrier that follows the
// reads), one step before they are added to again.
#include <algorithm>

#include "kernels.h"
#include "particle_step.cuh"
#include "push_math.cuh"
#include "slpic_internal.cuh"

namespace slpic {

constexpr int kST = kStepsThreads;
constexpr int kSW = kST / 32;
constexpr int kSList = 512;  // listed iterative pushes of a CTA and step (more are pushed in place)
// Source particles of a step that every CTA makes for itself; more are made in shares, which
// costs another barrier (4 us) and saves 1.6 us per 1,000 particles.  us a step, every CTA all of
// them / in shares / the three kernels, two species of 1,000, 2,000, 10,000 and 100,000 each:
// 256 cells 27 / 27 / 39, 33 / 28 / 44, 83 / 45 / 93, 575 / 172 / 749; 4,096 cells 30 / 30 / 38,
// 35 / 30 / 39, 77 / 40 / 55, 510 / 109 / 329; a wall source of 300 14 / 17 / 33.
constexpr int kStepsOwnSource = 2048;

struct StepsScratch {
    unsigned bar;  // arrivals at the grid barrier
    unsigned pad;
    unsigned long long out[3][kMaxSpecies];          // survivors of a compacting step
    unsigned long long absorbed[3][kMaxSpecies][2];  // this step's, per wall
    // followed by the accumulators [3][ns][nn]
};

struct ListedPush {
    int s, slot, c;
    float ax;
    float4 q;
};

size_t steps_scratch_bytes(int nn, int ns)
{
    return sizeof(StepsScratch) + sizeof(unsigned long long) * 3 * ns * nn;
}

size_t steps_smem_bytes(int nn, int ns, bool profile)
{
    return (size_t)ns * nn * 8 + 8 + sizeof(ListedPush) * kSList + (size_t)nn * 4 * (profile ? 2 : 1);
}

__device__ __forceinline__ void steps_fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// All CTAs (co-resident: a cooperative launch), once `target` have arrived in the launch.  A wait
// longer than `limit` SM cycles ends the launch (SLPIC_ERR_TIMEOUT): the CTA that gives up marks
// the counter, which it can only while one has not arrived, and nobody passes a marked
// counter.  So the barrier has one outcome for all: true everywhere, or false everywhere.
constexpr unsigned kStepsGivenUp = 0x80000000u;

__device__ __forceinline__ bool steps_barrier(StepsScratch *sc, unsigned target, long long limit, int *error)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        steps_fence();  // the CTA's writes, seen by this thread through the barrier above
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(&sc->bar) : "memory");
        const long long t0 = clock64();
        unsigned v;
        int ok = 1;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&sc->bar) : "memory");
            if (v & kStepsGivenUp) {
                ok = 0;
                break;
            }
            if (v >= target)
                break;
            if (clock64() - t0 > limit && atomicCAS(&sc->bar, v, v | kStepsGivenUp) == v) {
                atomicExch(error, SLPIC_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// x to the nearest double (ties to even), on the integer pipe: the value of the FP64
// conversion, whose pipe has 2 lanes an SM
__device__ __forceinline__ double u64_double_int(unsigned long long x)
{
    if (x == 0ULL)
        return 0.0;
    const int lz = __clzll((long long)x);
    const unsigned long long m = x << lz, r = m & 0x7FFULL;
    unsigned long long f = m >> 11;
    f += (r > 0x400ULL || (r == 0x400ULL && (f & 1ULL))) ? 1ULL : 0ULL;
    return __longlong_as_double((long long)(((unsigned long long)(1023 + 63 - lz - 1) << 52) + f));
}

// 2^64 hi + lo as k_field converts its 128-bit sums
__device__ __forceinline__ double u128_double_int(unsigned long long hi, unsigned long long lo)
{
    const double d = u64_double_int(lo);
    return hi ? fma(u64_double_int(hi), 18446744073709551616.0, d) : d;
}

// x to the nearest float on the integer pipe (outside FP32's normal range by the
// conversion instruction)
__device__ __forceinline__ float double_float_int(double x)
{
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const int e = (int)((h >> 20) & 0x7FFu) - 896;
    if (e < 1 || e > 254)
        return (float)x;
    const unsigned f = ((h & 0xFFFFFu) << 3) | (l >> 29), r = l & 0x1FFFFFFFu;
    const unsigned up = (r > 0x10000000u || (r == 0x10000000u && (f & 1u))) ? 1u : 0u;
    return __uint_as_float((h & 0x80000000u) | ((((unsigned)e << 23) | f) + up));
}

// sum over the warp modulo 2^64, as three 32-bit reductions of 27-bit pieces
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v)
{
    const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x7FFFFFFu);
    const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 27) & 0x7FFFFFFu);
    const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 54));
    return a + ((unsigned long long)b << 27) + ((unsigned long long)c << 54);
}

__device__ __forceinline__ unsigned long long warp_scan_u64(unsigned long long v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o)
            v += y;
    }
    return v;
}

struct StepsShared {
    long long count[kMaxSpecies], holes[kMaxSpecies];  // slots in use, holes among them
    long long injected[kMaxSpecies], absorbed[kMaxSpecies][2];  // of this launch
    double frac[kMaxSpecies];
    long long base[kMaxSpecies], make[kMaxSpecies];  // this step's source: first slot, particles
    int cut;                                         // a source was truncated
    struct Counts {  // before this step, and what it has absorbed and walked
        long long count, holes, lo, hi;
        double frac;
        unsigned walked;
    } before[kMaxSpecies];
    unsigned lost[kMaxSpecies][2];                   // absorbed by this CTA in this step
    unsigned listed;
    unsigned walked[kMaxSpecies];                    // by this CTA in this step
    unsigned long long iterative[kMaxSpecies];       // ... in the launch's steps before
    unsigned long long part[kMaxSpecies][kSW][4];    // per warp: sums of R, W (two words), T
    unsigned long long tot[kMaxSpecies][4];
    double K[kMaxSpecies];                           // k_field's K_s
    double c[4];                                     // a, B, and E at nodes 0 and N
};

// The slots are dealt to the CTAs in tiles of a warp's 32, round and round, so that the
// source's latest particles, which sit in consecutive slots and mostly need the iterative
// push, spread over all of them (with contiguous shares the slowest CTA kept the others at
// the barrier for 5 us of a step's 15 on the paper's sheath).  Species s starts at its own
// CTA, so that the tiles left over fall on different ones.
__device__ __forceinline__ int steps_first_tile(int s)
{
    const int b = (int)blockIdx.x + s * (int)gridDim.x / kMaxSpecies;
    return b < (int)gridDim.x ? b : b - (int)gridDim.x;
}

// E at the nodes from the total deposit s_acc [ns][nn]: k_field's solve by one CTA, with
// the same sums (a prefix sum fits 64 bits: fewer than 2^24 particles of 2^40 at most) and the
// same FP64 operations, of which each thread is left the one multiply-add per species and
// node: an FP64 operation costs 110 cycles in a chain and 16 cycles of the SM's pipe per
// warp, so the constants are made once, the step's by one thread, and integers turn into
// doubles, and E into floats, on the integer pipe (256 nodes: 11,900 -> 4,700 cycles).
// last: also the global copies.
__device__ __forceinline__ void steps_field(const StepParams &p, StepsShared &sh,
                                            const unsigned long long *s_acc, float *s_E, bool last)
{
    const int N = p.n_cells, nn = p.nn, ns = p.ns;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int chunk = (nn + kST - 1) / kST;
    const int j0 = min(nn, (int)threadIdx.x * chunk), j1 = min(nn, j0 + chunk);
    const int nw = (nn + 32 * chunk - 1) / (32 * chunk);  // warps with nodes
    // sums over this thread's nodes: R = rows 1..N-1, W = sum (N - j) acc in two words, T =
    // nodes j < N (periodic grids only); R's prefix over the warp's threads
    unsigned long long before[kMaxSpecies] = {};
    if (warp < nw) {
#pragma unroll
        for (int s = 0; s < kMaxSpecies; ++s) {
            if (s >= ns)
                break;
            unsigned long long R = 0, Wl = 0, Wh = 0, T = 0;
            for (int j = j0; j < j1; ++j) {
                const unsigned long long v = s_acc[s * nn + j];
                if (j < N)
                    T += v;
                if (j >= 1 && j < N) {
                    R += v;
                    Wl += (v & 0xFFFFFFFFULL) * (unsigned)(N - j);
                    Wh += (v >> 32) * (unsigned)(N - j);
                }
            }
            const unsigned long long incl = warp_scan_u64(R, lane);
            before[s] = incl - R;
            Wl = warp_sum_u64(Wl);
            Wh = warp_sum_u64(Wh);
            if (p.periodic)
                T = warp_sum_u64(T);
            if (lane == 31) {
                sh.part[s][warp][0] = incl;
                sh.part[s][warp][1] = Wl;
                sh.part[s][warp][2] = Wh;
                sh.part[s][warp][3] = T;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < 4 * ns) {  // quantity q of species s
        const int s = threadIdx.x >> 2, q = threadIdx.x & 3;
        unsigned long long t = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w)
            t += sh.part[s][w][q];
        sh.tot[s][q] = t;
    }
    if (warp == 0) {
        __syncwarp();
        if (lane == 0) {
            double sumW = 0.0, sumR = 0.0, sumT = 0.0;
            for (int s = 0; s < ns; ++s) {
                const double cs = p.sp[s].rho_unit;
                const unsigned long long wl = sh.tot[s][1], wh = sh.tot[s][2], lo = wl + (wh << 32);
                const unsigned long long hi = (wh >> 32) + (lo < wl ? 1ULL : 0ULL);
                sumR = fma(cs, u64_double_int(sh.tot[s][0]), sumR);
                sumW = fma(cs, u128_double_int(hi, lo), sumW);
                if (p.periodic)
                    sumT = fma(cs, u64_double_int(sh.tot[s][3]), sumT);
            }
            const double k2 = p.k2, inv2dx = 0.5 * p.inv_dx;
            if (p.periodic) {
                const double mean = sumT * p.inv_n;
                const double sumP = k2 * (sumW - mean * 0.5 * (double)N * (double)(N - 1));
                const double D0 = sumP * p.inv_n, P_last = k2 * (sumR - mean * (double)(N - 1));
                sh.c[0] = 2.0 * k2 * mean * inv2dx;
                sh.c[1] = (k2 * mean - 2.0 * D0) * inv2dx;
                sh.c[2] = ((P_last + 0.0) - 2.0 * D0) * inv2dx;
            } else {  // mean = 0: its terms, exact zeros, left out
                const double D0 = (p.phi_hi - p.phi_lo + k2 * sumW) * p.inv_n, P_last = k2 * sumR;
                sh.c[1] = (0.0 - 2.0 * D0) * inv2dx;
                sh.c[2] = -D0 * p.inv_dx;
                sh.c[3] = (P_last - D0) * p.inv_dx;
            }
        }
    } else if (warp < nw) {
        // the warps before this one (the first warp's prefix is complete)
#pragma unroll
        for (int s = 0; s < kMaxSpecies; ++s) {
            if (s >= ns)
                break;
#pragma unroll 4
            for (int w = 0; w < warp; ++w)
                before[s] += sh.part[s][w][0];
        }
    }
    __syncthreads();
    const int o0 = (int)((long long)nn * blockIdx.x / gridDim.x);
    const int o1 = (int)((long long)nn * (blockIdx.x + 1) / gridDim.x);  // nodes this CTA stores
    for (int j = j0; j < j1; ++j) {
        double e;
        if (j == 0) {
            e = sh.c[2];
        } else if (!p.periodic && j == N) {
            e = sh.c[3];
        } else {
            e = p.periodic ? fma(-sh.c[0], (double)j, sh.c[1]) : sh.c[1];
#pragma unroll
            for (int s = 0; s < kMaxSpecies; ++s) {
                if (s >= ns)
                    break;
                const unsigned long long prev = before[s];
                before[s] += s_acc[s * nn + j];  // row j (1 <= j <= N-1)
                const unsigned long long x = prev + before[s];
                e = fma(sh.K[s], u128_double_int(x < prev ? 1ULL : 0ULL, x), e);
            }
        }
        const float f = double_float_int(e);
        s_E[j] = f;
        if (last && j >= o0 && j < o1) {
            p.E64[j] = e;
            p.E[j] = f;
        }
    }
}

template <bool kProf, bool kSheath>
__global__ void __launch_bounds__(kST, 1)
    k_steps(const __grid_constant__ StepParams p, int nsteps, int every, StepsScratch *sc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kKind = kSheath ? SLPIC_BETA_HEAVISIDE : kAny;
    constexpr int kPer = kSheath ? 0 : kAny;
    const int nn = p.nn, ns = p.ns, tot = ns * nn;
    unsigned long long *s_acc = reinterpret_cast<unsigned long long *>(smem);  // [ns][nn], or
    unsigned *s_lo = reinterpret_cast<unsigned *>(smem), *s_hi = s_lo + tot;   // its two words
    ListedPush *s_list = reinterpret_cast<ListedPush *>(smem + (size_t)tot * 8 + ((tot & 1) ? 8 : 0));
    float *s_E = reinterpret_cast<float *>(s_list + kSList);
    float *s_lam = s_E + nn;
    __shared__ StepsShared sh;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long *acc3 = reinterpret_cast<unsigned long long *>(sc + 1);
    DevState *st = p.st;
    const long long step0 = *(volatile long long *)&st->step;
    if (*(volatile int *)&st->error == SLPIC_ERR_TIMEOUT)
        return;  // the launch before was cut short: no step until that has been reported

    for (int j = t; j < tot; j += kST) {
        s_lo[j] = 0u;
        s_hi[j] = 0u;
    }
    for (int j = t; j < nn; j += kST) {
        s_E[j] = p.E[j];
        if (kProf)
            s_lam[j] = j < p.n_cells ? __ldg(p.lam + j) : 0.0f;
    }
    if (t < kMaxSpecies) {
        const int P = (int)(step0 & 1);
        sh.count[t] = t < ns ? (long long)*(volatile unsigned long long *)&st->count[t][P] : 0;
        sh.holes[t] = t < ns ? (long long)*(volatile unsigned long long *)&st->holes[t][P] : 0;
        sh.frac[t] = t < ns ? *(volatile double *)&st->src_frac[t] : 0.0;
        sh.injected[t] = sh.absorbed[t][0] = sh.absorbed[t][1] = 0;
        sh.iterative[t] = sh.walked[t] = 0;
        sh.K[t] = t < ns ? p.k2 * p.sp[t].rho_unit * (0.5 * p.inv_dx) : 0.0;
        sh.lost[t][0] = sh.lost[t][1] = 0u;
    }
    if (t == 0) {
        sh.listed = 0u;
        sh.cut = 0;
    }
    __syncthreads();
    unsigned long long span[3] = {0, 0, 0}, tick = t == 0 && blockIdx.x == 0 ? gtimer() : 0ULL;
    auto lap = [&](int k) {
        if (t == 0 && blockIdx.x == 0) {
            const unsigned long long now = gtimer();
            span[k] += now - tick;
            tick = now;
        }
    };
    int turn = 0, e = 0;      // e: whole steps made
    unsigned arrivals = 0u;  // of all CTAs at the barriers so far
    for (; e < nsteps; ++e) {
        const long long step = step0 + e;
        const int P = (int)(step & 1), Q = P ^ 1;
        const bool compact = step % every == every - 1, last = e + 1 == nsteps;

        // ---- the particles of this CTA's slots, a warp to 32 slots at a time
        int f0[kMaxSpecies], w1[kMaxSpecies];  // first tile; this CTA's tiles up to and with species s
#pragma unroll
        for (int s = 0; s < kMaxSpecies; ++s) {
            f0[s] = steps_first_tile(s);
            const int tiles = s < ns ? (int)((sh.count[s] + 31) >> 5) : 0;
            w1[s] = (s ? w1[s - 1] : 0) + (tiles > f0[s] ? (tiles - f0[s] + (int)gridDim.x - 1) / (int)gridDim.x : 0);
        }
        // tile w of this CTA: species and slot (a warp's 32 in one species); its particle, read
        // through L2 (another SM may have written it), a tile ahead of its use
        auto slot_of = [&](int w, int &s) {
            s = 0;
            int k = w, f = f0[0];
#pragma unroll
            for (int r = 1; r < kMaxSpecies; ++r)
                if (w >= w1[r - 1]) {
                    s = r;
                    k = w - w1[r - 1];
                    f = f0[r];
                }
            return 32 * (f + k * (int)gridDim.x) + lane;
        };
        int s = 0, i = 0, c = -1;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        auto fetch = [&](int w, int &s, int &i, int &c, float4 &q) {
            c = -1;
            i = slot_of(w, s);
            if (i < sh.count[s]) {
                c = __ldcg(p.sp[s].cell[P] + i);
                q = __ldcg(p.sp[s].pv[P] + i);
            }
        };
        if (warp < w1[kMaxSpecies - 1])
            fetch(warp, s, i, c, q);
        for (int w = warp; w < w1[kMaxSpecies - 1]; w += kSW) {
            int s2 = 0, i2 = 0, c2 = -1;
            float4 q2 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (w + kSW < w1[kMaxSpecies - 1])
                fetch(w + kSW, s2, i2, c2, q2);
            const SpeciesDev &sp = p.sp[s];
            DepositSplit32 dep{s_lo + s * nn, s_hi + s * nn};
            const bool in = i < sh.count[s];
            bool live = c >= 0, hard = false;
            float ax = 0.0f, v0n = 0.0f;
            if (live) {
                ax = gather_ax<kPer>(p, sp, s_E, c, q.x);
                v0n = v0_at<kProf>(p, sp, c, s_lam);
                float vx;
                if (push_vx_easy(kSheath ? kKind : sp.kind, q.y, q.z, q.w, ax, p.dt, v0n, vx)) {
                    int wall = 0;
                    live = move_and_deposit<kProf, kKind, kPer>(p, sp, dep, c, q, vx, wall, v0n, s_lam);
                    if (!live)
                        atomicAdd(&sh.lost[s][wall], 1u);
                } else {
                    hard = true;
                }
            }
            const unsigned hm = __ballot_sync(0xffffffffu, hard);
            if (hm) {
                unsigned b = 0;
                if (lane == 0) {
                    b = atomicAdd(&sh.listed, (unsigned)__popc(hm));
                    atomicAdd(&sh.walked[s], (unsigned)__popc(hm));
                }
                b = __shfl_sync(0xffffffffu, b, 0) + __popc(hm & ((1u << lane) - 1u));
                if (hard) {
                    if (b < (unsigned)kSList) {
                        s_list[b] = ListedPush{s, i, c, ax, q};
                        live = false;  // stored after its walk
                    } else {
                        const float vx = push_vx_walk(sp.kind, q.y, q.z, q.w, ax, p.dt, v0n);
                        int wall = 0;
                        live = move_and_deposit<kProf, kKind, kPer>(p, sp, dep, c, q, vx, wall, v0n, s_lam);
                        if (!live)
                            atomicAdd(&sh.lost[s][wall], 1u);
                        hard = false;
                    }
                }
            }
            if (compact) {
                const unsigned m = __ballot_sync(0xffffffffu, live);
                unsigned long long o = 0;
                if (lane == 0 && m)
                    o = atomicAdd(&sc->out[turn][s], (unsigned long long)__popc(m));
                o = __shfl_sync(0xffffffffu, o, 0) + __popc(m & ((1u << lane) - 1u));
                if (live) {
                    sp.cell[Q][o] = c;
                    sp.pv[Q][o] = q;
                }
            } else if (in && !hard) {
                sp.cell[Q][i] = live ? c : -1;
                if (live)
                    sp.pv[Q][i] = q;
            }
            s = s2;
            i = i2;
            c = c2;
            q = q2;
        }
        lap(0);
        __syncthreads();
        // ---- the listed pushes: one lane each, spread over the warps
        {
            const unsigned n = min(sh.listed, (unsigned)kSList);
            const unsigned k = (unsigned)(lane * kSW + warp);
            if (k < n) {
                const ListedPush r = s_list[k];
                const SpeciesDev &sp = p.sp[r.s];
                DepositSplit32 dep{s_lo + r.s * nn, s_hi + r.s * nn};
                int c = r.c, wall = 0;
                float4 q = r.q;
                const float v0n = v0_at<kProf>(p, sp, c, s_lam);
                const float vx = push_vx_walk(sp.kind, q.y, q.z, q.w, r.ax, p.dt, v0n);
                const bool live = move_and_deposit<kProf, kKind, kPer>(p, sp, dep, c, q, vx, wall, v0n, s_lam);
                if (!live)
                    atomicAdd(&sh.lost[r.s][wall], 1u);
                if (!compact) {
                    sp.cell[Q][r.slot] = live ? c : -1;
                    if (live)
                        sp.pv[Q][r.slot] = q;
                } else if (live) {
                    const unsigned long long o = atomicAdd(&sc->out[turn][r.s], 1ULL);
                    sp.cell[Q][o] = c;
                    sp.pv[Q][o] = q;
                }
            }
        }
        __syncthreads();
        // ---- this CTA's charge and losses to the turn's accumulators; those of the next
        // turn cleared
        const int next = turn == 2 ? 0 : turn + 1;
        for (int j = t; j < tot; j += kST) {
            const unsigned long long v = ((unsigned long long)s_hi[j] << 32) + s_lo[j];
            if (v)
                atomicAdd(acc3 + (size_t)turn * tot + j, v);
        }
        if (t < 2 * ns) {
            unsigned &n = sh.lost[t >> 1][t & 1];
            if (n)
                atomicAdd(&sc->absorbed[turn][t >> 1][t & 1], (unsigned long long)n);
            n = 0u;
        }
        if (t == 0)
            sh.listed = 0u;
        for (int j = (int)((long long)tot * blockIdx.x / gridDim.x) + t,
                 j1 = (int)((long long)tot * (blockIdx.x + 1) / gridDim.x);
             j < j1; j += kST)
            acc3[(size_t)next * tot + j] = 0ULL;
        if (blockIdx.x == 0 && t < kMaxSpecies)
            sc->out[next][t] = sc->absorbed[next][t][0] = sc->absorbed[next][t][1] = 0ULL;
        lap(1);
        arrivals += gridDim.x;
        if (!steps_barrier(sc, arrivals, p.wait_cycles, &st->error))
            break;

        // ---- the step's totals and the source's counts (thread s for species s; every CTA the
        // same)
        if (t < ns) {
            const unsigned long long a0 = __ldcg(&sc->absorbed[turn][t][0]), a1 = __ldcg(&sc->absorbed[turn][t][1]);
            const unsigned long long ref =
                __ldcg(&sc->absorbed[turn][p.src_ref][0]) + __ldcg(&sc->absorbed[turn][p.src_ref][1]);
            const long long have = compact ? (long long)__ldcg(&sc->out[turn][t]) : sh.count[t];
            double f = sh.frac[t];
            long long k = source_count(p, p.sp[t], ref, f);
            const long long room = p.sp[t].capacity - have;
            sh.before[t] = StepsShared::Counts{sh.count[t], sh.holes[t], (long long)a0, (long long)a1, sh.frac[t],
                                               sh.walked[t]};
            if (k > room) {
                k = room;
                sh.cut = 1;
            }
            sh.frac[t] = f;
            sh.base[t] = have;
            sh.make[t] = k;
            sh.count[t] = have + k;
            sh.holes[t] = compact ? 0 : sh.holes[t] + (long long)(a0 + a1);
            sh.iterative[t] += sh.walked[t];
            sh.walked[t] = 0u;
            sh.injected[t] += k;
            sh.absorbed[t][0] += (long long)a0;
            sh.absorbed[t][1] += (long long)a1;
        }
        for (int j = t; j < tot; j += kST)
            s_acc[j] = __ldcg(acc3 + (size_t)turn * tot + j);
        __syncthreads();
        // ---- the source's particles: few are made by every CTA, more in shares, with their
        // charge through the accumulator and a barrier of its own
        {
            long long pre[kMaxSpecies + 1];
            pre[0] = 0;
#pragma unroll
            for (int s = 0; s < kMaxSpecies; ++s)
                pre[s + 1] = pre[s] + (s < ns ? sh.make[s] : 0);
            const bool shares = pre[kMaxSpecies] > kStepsOwnSource;
            long long k = t, k1 = pre[kMaxSpecies];
            if (shares) {
                k = t + k1 * blockIdx.x / gridDim.x;
                k1 = k1 * (blockIdx.x + 1) / gridDim.x;
                for (int j = t; j < tot; j += kST)
                    s_acc[j] = 0ULL;
                __syncthreads();
            }
            for (; k < k1; k += kST) {
                int s = 0;
                long long i = k;
#pragma unroll
                for (int r = 1; r < kMaxSpecies; ++r)
                    if (k >= pre[r]) {
                        s = r;
                        i = k - pre[r];
                    }
                const SpeciesDev &sp = p.sp[s];
                int c;
                float4 q;
                source_particle(p, sp, sm64_stream(p.seed, (unsigned long long)step, (unsigned)s), i, c, q);
                int c1 = c + 1;
                if (p.periodic && c1 == p.n_cells)
                    c1 = 0;
                // the accumulators' two words (little-endian), by native 32-bit atomics: 64-bit
                // ones in shared memory are compare-and-swap loops, and a wall source's
                // particles share a cell or two (250 of them took 15 us)
                unsigned *acc = reinterpret_cast<unsigned *>(s_acc + s * nn);
                unsigned llo, lhi, rlo, rhi;
                quantise_split(beta_q(sp.kind, q.y, q.z, q.w, v0_cell(p, sp, c)), q.x, llo, lhi, rlo, rhi);
                unsigned old = atomicAdd(acc + 2 * c, llo);
                lhi += (old + llo < old) ? 1u : 0u;
                if (lhi)
                    atomicAdd(acc + 2 * c + 1, lhi);
                old = atomicAdd(acc + 2 * c1, rlo);
                rhi += (old + rlo < old) ? 1u : 0u;
                if (rhi)
                    atomicAdd(acc + 2 * c1 + 1, rhi);
                const int o = (int)(sh.base[s] + i);  // stored by the CTA that pushes it next
                if (shares || (o >> 5) % (int)gridDim.x == steps_first_tile(s)) {
                    sp.cell[Q][o] = c;
                    sp.pv[Q][o] = q;
                }
            }
            if (shares) {
                __syncthreads();
                for (int j = t; j < tot; j += kST)
                    if (s_acc[j])
                        atomicAdd(acc3 + (size_t)turn * tot + j, s_acc[j]);
                arrivals += gridDim.x;
                if (!steps_barrier(sc, arrivals, p.wait_cycles, &st->error)) {
                    if (t < ns) {  // the step is not whole: its counts taken back
                        const StepsShared::Counts &c = sh.before[t];
                        sh.count[t] = c.count;
                        sh.holes[t] = c.holes;
                        sh.frac[t] = c.frac;
                        sh.iterative[t] -= c.walked;
                        sh.injected[t] -= sh.make[t];
                        sh.absorbed[t][0] -= c.lo;
                        sh.absorbed[t][1] -= c.hi;
                    }
                    break;
                }
                for (int j = t; j < tot; j += kST)
                    s_acc[j] = __ldcg(acc3 + (size_t)turn * tot + j);
            }
        }
        __syncthreads();
        steps_field(p, sh, s_acc, s_E, last);
        if (last) {
            const int a = (int)((long long)tot * blockIdx.x / gridDim.x);
            const int b = (int)((long long)tot * (blockIdx.x + 1) / gridDim.x);
            for (int j = a + t; j < b; j += kST) {
                p.acc[(size_t)Q * tot + j] = s_acc[j];
                p.acc[(size_t)P * tot + j] = 0ULL;
            }
        } else {
            __syncthreads();
            for (int j = t; j < tot; j += kST) {
                s_lo[j] = 0u;
                s_hi[j] = 0u;
            }
            __syncthreads();
        }
        lap(2);
        turn = next;
    }
    // ---- the launch's bookkeeping: of the whole steps (a step that was cut short has written
    // only the other buffers; deposit and field are then made again on the host's demand)
    if (t < ns && sh.iterative[t])
        atomicAdd((unsigned long long *)&st->iterative_total[t], sh.iterative[t]);
    if (blockIdx.x == 0 && t < ns) {
        const int Pf = (int)((step0 + e) & 1);
        st->count[t][Pf] = (unsigned long long)sh.count[t];
        st->holes[t][Pf] = (unsigned long long)sh.holes[t];
        st->count[t][Pf ^ 1] = 0ULL;
        st->holes[t][Pf ^ 1] = 0ULL;
        st->src_frac[t] = sh.frac[t];
        st->injected_total[t] += sh.injected[t];
        st->absorbed_total[t][0] += sh.absorbed[t][0];
        st->absorbed_total[t][1] += sh.absorbed[t][1];
    }
    if (blockIdx.x == 0 && t == 0) {
        if (sh.cut)
            atomicCAS(&st->error, 0, SLPIC_ERR_CAPACITY);
        for (int k = 0; k < 3; ++k) {
            st->span_ns[k] += span[k];
            st->span_launches[k] += (unsigned long long)e;
        }
        st->step = step0 + e;
    }
}

typedef void (*StepsKernel)(StepParams, int, int, StepsScratch *);

static StepsKernel steps_kernel(const StepParams &p)
{
    bool sheath = !p.periodic;
    for (int s = 0; s < p.ns; ++s)
        sheath = sheath && p.sp[s].kind == SLPIC_BETA_HEAVISIDE;
    return p.lam ? (sheath ? k_steps<true, true> : k_steps<true, false>)
                 : (sheath ? k_steps<false, true> : k_steps<false, false>);
}

cudaError_t configure_steps(int *max_smem)
{
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    *max_smem = optin - (int)sizeof(StepsShared) - 1024;
    for (auto f : {k_steps<false, false>, k_steps<false, true>, k_steps<true, false>, k_steps<true, true>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, *max_smem);
    return e;
}

cudaError_t launch_steps(const StepParams &p, int nsteps, int every, int ctas, void *scratch, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(scratch, 0, steps_scratch_bytes(p.nn, p.ns), st);
    if (e != cudaSuccess)
        return e;
    StepParams q = p;
    StepsScratch *sc = static_cast<StepsScratch *>(scratch);
    void *args[] = {&q, &nsteps, &every, &sc};
    return cudaLaunchCooperativeKernel((const void *)steps_kernel(p), dim3(ctas), dim3(kST), args,
                                       steps_smem_bytes(p.nn, p.ns, p.lam != nullptr), st);
}

}  // namespace slpic
