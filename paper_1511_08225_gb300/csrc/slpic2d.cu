// slpic2d.cu -- the 2D3V speed-limited PIC path behind include/slpic2d.h.
//
// Per step (Appendix A, Eq. slpicIntegration, on an nx x ny grid, periodic in x,
// absorbing plates in y):
//   k_particles2d_tiles (+ k_hard2d), or k_particles2d where its windows do not fit
//                  gather E (bilinear) -> push v (the same speed-limited solve as
//                  1D, along the direction of a) -> move -> plates/wrap -> deposit
//                  rho^{n+1} (quantised int64, bilinear) into the nodal arrays: the
//                  tile kernel through windows of the grid in shared memory, listing
//                  the pushes that need the piece walk for k_hard2d; the other by
//                  global atomics.  Absorbed particles leave holes (cell = -1) in
//                  place; every kCompact2d-th step the counting sort by cell drops
//                  them (k_particles2d packs the survivors itself on that step).
//   k_inject2d     source particles appended and deposited; k_book2d the bookkeeping.
//   k_cg2d         cooperative kernel: b from the deposits, Jacobi-PCG on the
//                  5-point system (FP64 vectors, FP64 dot products in a fixed
//                  order), then E^{n+1}; the deposits are cleared for the next step.
//
// Particle store per species, ping-pong buffers b = step & 1:
//   cell[b][i] int32 (cy*nx + cx, -1 = hole), pv[b][i] float4 {ox, oy, vx, vy},
//   vz[b][i] float  -- 24 bytes per macroparticle.
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "push_math.cuh"
#include "slpic2d.h"
#include "smem_limit.h"
#include "unet_internal.h"

namespace slpic {
void set_create_error(const std::string &msg);  // api.cu
}

namespace slpic2d {

using namespace slpic;

constexpr int kMaxS = SLPIC_MAX_SPECIES;
constexpr int kThreads = 256;
constexpr int kItems = 4;                       // particles per thread per tile
constexpr int kTile = kThreads * kItems;
constexpr int kWarps = kThreads / 32;
constexpr int kCompact2d = 16;                  // compacting step interval
constexpr int kCgVirtual = 256;  // threads of a virtual CTA of the CG: a unit of its sums
constexpr int kCgThreads = 2 * kCgVirtual;
constexpr int kCgMaxVirtual = 512;             // virtual CTAs (two per SM)
constexpr long long kCgWaitCycles = 2000000000LL;  // bounded wait for the other CTAs (~1 s)
constexpr long long kMaxTimedSteps2d = 4096;    // steps recorded by the kernel timing

struct Species2D {
    int32_t *cell[2];
    float4 *pv[2];
    float *vz[2];
    int32_t *hard;       // slots of this step's particles whose push needs the walk [capacity]
    long long capacity;
    float qm, v0, vth_src;
    int kind;
    double w, inv_w;
    double rho_unit;  // q w / dx^2 * 2^-40
};

struct State2D {
    long long step;
    unsigned long long count[kMaxS][2];   // slots in use (live + holes) per buffer
    unsigned long long holes[kMaxS][2];
    unsigned long long absorbed_step[kMaxS][2];
    long long absorbed_total[kMaxS][2];
    long long injected_total[kMaxS];
    double src_frac[kMaxS];
    unsigned long long hard_n[kMaxS];  // particles listed for k_hard2d this step
    unsigned long long iter_last;      // walked pushes of the last step, all species
    long long cg_total;
    double cg_res;
    int cg_iters;
    int error;
};

struct Params2D {
    int nx, ny, nn, ns;
    unsigned nx_m;  // c / nx = div_nx(c): the multiplier and shift of the round-up method
    int nx_s;
    float dt, dt_dx;
    double dx, dt64, k2;          // k2 = dx^2 / eps0
    double half_dx;               // 0.5 / dx
    double phi_lo, phi_hi, rtol2;  // rtol^2
    int cg_maxit;
    int src_mode, src_ref;
    float src_lo, src_len;
    double src_rate;
    unsigned long long seed;
    Species2D sp[kMaxS];
    unsigned long long *acc;  // [ns][nn] int64 deposits (two's complement)
    float2 *E;                // [nn] (Ex, Ey)
    double *phi, *r, *q;            // [nn] FP64: solution, standalone solve's rho, b
    float *fr, *fpA, *fpB, *fq, *fd;  // [nn] FP32 CG iterates, zero on the plate rows
    double *part;             // [3][cg_v] the CG's partial sums, by turn (kCgEmpty: not there yet)
    int cg_v;                 // virtual CTAs of the CG's sums
    State2D *st;
    // direct solver (SLPIC2D_SOLVER_FFT)
    int solver, log2nx;
    double2 *tw;              // [nx/2] (cos, sin)(2 pi m / nx)
    double2 *spec;            // [nn] Fourier coefficients along x, row by row
    double *inv_m;            // [nn] Thomas multipliers 1/m_j per (row j, mode k)
    double *seg_f, *seg_b;    // [nn] their products within a segment, up to / from row j
    double *rpart;            // [2 (ny+1)] per-row sums of r^2 and b^2
    unsigned *finished;       // CTAs of k_fft_finish that have written theirs
    int *hist, *cursor, *bsum;  // cell sort: counts per cell, then slots; block sums
};

// c / nx for 0 <= c < 2^32 and nx >= 2 without a division: Granlund and Montgomery's
// method for an invariant divisor (PLDI 1994, Fig. 4.1): with l = ceil(log2 nx) and
// m = floor(2^32 (2^l - nx) / nx) + 1 (host, make_div_nx), t = mulhi(m, c) and
// q = (t + ((c - t) >> 1)) >> (l - 1).
__device__ __forceinline__ int div_nx(const Params2D &p, int c)
{
    const unsigned n = (unsigned)c;
    const unsigned t = __umulhi(p.nx_m, n);
    return (int)((t + ((n - t) >> 1)) >> p.nx_s);
}

void make_div_nx(int nx, unsigned &m, int &s)
{
    int l = 0;
    while ((1LL << l) < nx)
        ++l;
    m = (unsigned)((((unsigned long long)1 << 32) * (unsigned long long)((1LL << l) - nx)) /
                       (unsigned long long)nx + 1ULL);
    s = l - 1;
}

// ---------------------------------------------------------------------------------
// Velocity push with a = (ax, ay, 0): the speed-limited solve of Appendix A,
// Eq. slpicIntegrationV, depends only on the component w of v along a and on
// |v_perp|, so the 1D solve (push_vx with a along +x) gives w at the end of the
// step and v changes by (w_end - w) in the direction of a.
// ---------------------------------------------------------------------------------
// kEasy: only the cases push_vx_easy solves; returns false (v untouched) for the
// rest, which need the piece walk.  Otherwise every case; returns true.
template <bool kEasy>
__device__ __forceinline__ bool push_v2_impl(int kind, float ux, float uy, float uz, float ax,
                                             float ay, float dt, float v0, float &vx, float &vy)
{
    if (kind == SLPIC_BETA_ONE) {
        vx = __fadd_rn(ux, __fmul_rn(ax, dt));
        vy = __fadd_rn(uy, __fmul_rn(ay, dt));
        return true;
    }
    // |a|, the direction of a and |v_perp| from reciprocal square roots (within a few
    // ulp; the push's bar is 1e-5 of |v|): one approximation instead of a correctly
    // rounded square root and two divisions
    const float a2 = __fadd_rn(__fmul_rn(ax, ax), __fmul_rn(ay, ay));
    if (a2 == 0.0f) {
        vx = ux;
        vy = uy;
        return true;
    }
    const float ra = rsqrtf(a2);
    const float A = __fmul_rn(a2, ra);
    const float hx = __fmul_rn(ax, ra), hy = __fmul_rn(ay, ra);
    const float wa = __fadd_rn(__fmul_rn(ux, hx), __fmul_rn(uy, hy));
    const float cr = __fsub_rn(__fmul_rn(ux, hy), __fmul_rn(uy, hx));
    const float vp2 = __fadd_rn(__fmul_rn(cr, cr), __fmul_rn(uz, uz));
    const float vp = vp2 > 0.0f ? __fmul_rn(vp2, rsqrtf(vp2)) : 0.0f;
    float we;
    if (kEasy) {
        if (!push_vx_easy(kind, wa, vp, 0.0f, A, dt, v0, we))
            return false;
    } else {
        we = push_vx(kind, wa, vp, 0.0f, A, dt, v0);
    }
    const float dw = __fsub_rn(we, wa);
    vx = __fadd_rn(ux, __fmul_rn(dw, hx));
    vy = __fadd_rn(uy, __fmul_rn(dw, hy));
    return true;
}

__device__ __forceinline__ void push_v2(int kind, float ux, float uy, float uz, float ax, float ay,
                                        float dt, float v0, float &vx, float &vy)
{
    push_v2_impl<false>(kind, ux, uy, uz, ax, ay, dt, v0, vx, vy);
}

__device__ __forceinline__ bool push_v2_easy(int kind, float ux, float uy, float uz, float ax,
                                             float ay, float dt, float v0, float &vx, float &vy)
{
    return push_v2_impl<true>(kind, ux, uy, uz, ax, ay, dt, v0, vx, vy);
}

// (q/m) E at a particle from its cell's four nodes, bilinear, in a fixed operation order
__device__ __forceinline__ void accel2d(float qm, float2 e00, float2 e10, float2 e01, float2 e11,
                                        float ox, float oy, float &ax, float &ay)
{
    const float wx0 = __fsub_rn(1.0f, ox), wy0 = __fsub_rn(1.0f, oy);
    const float ex = __fadd_rn(__fmul_rn(wy0, __fadd_rn(__fmul_rn(wx0, e00.x), __fmul_rn(ox, e10.x))),
                               __fmul_rn(oy, __fadd_rn(__fmul_rn(wx0, e01.x), __fmul_rn(ox, e11.x))));
    const float ey = __fadd_rn(__fmul_rn(wy0, __fadd_rn(__fmul_rn(wx0, e00.y), __fmul_rn(ox, e10.y))),
                               __fmul_rn(oy, __fadd_rn(__fmul_rn(wx0, e01.y), __fmul_rn(ox, e11.y))));
    ax = __fmul_rn(qm, ex);
    ay = __fmul_rn(qm, ey);
}

// the 2D quantised deposit rule stated in slpic2d.h: the charges of the cell's nodes
// (x, y), (x+1, y), (x, y+1), (x+1, y+1)
__device__ __forceinline__ void quantise2d(float b, float ox, float oy, unsigned long long &q00,
                                           unsigned long long &q10, unsigned long long &q01,
                                           unsigned long long &q11)
{
    const float two40 = 1099511627776.0f;
    const float bx = __fmul_rn(b, ox), by = __fmul_rn(b, oy), bxy = __fmul_rn(bx, oy);
    const unsigned long long qT = rint_u64(__fmul_rn(b, two40));
    const unsigned long long qX = rint_u64(__fmul_rn(bx, two40));
    const unsigned long long qY = rint_u64(__fmul_rn(by, two40));
    const unsigned long long qXY = rint_u64(__fmul_rn(bxy, two40));
    q00 = qT - qX - qY + qXY;
    q10 = qX - qXY;
    q01 = qY - qXY;
    q11 = qXY;
}

__device__ __forceinline__ void deposit2d(unsigned long long *acc, int k00, int k10, int k01,
                                          int k11, float b, float ox, float oy)
{
    unsigned long long q00, q10, q01, q11;
    quantise2d(b, ox, oy, q00, q10, q01, q11);
    atomicAdd(acc + k00, q00);
    atomicAdd(acc + k10, q10);
    atomicAdd(acc + k01, q01);
    atomicAdd(acc + k11, q11);
}

// ---------------------------------------------------------------------------------
// Particle step.  COMPACT = false: slot i of the input goes to slot i of the
// output (a hole where a particle is absorbed); true: the survivors are packed
// (one global atomic per CTA tile).
// ---------------------------------------------------------------------------------
template <bool COMPACT>
__global__ void __launch_bounds__(kThreads) k_particles2d(Params2D p)
{
    __shared__ int s_cnt[kItems * kWarps];
    __shared__ unsigned long long s_base;
    __shared__ unsigned s_abs[2];
    const int s = blockIdx.y;
    const Species2D &sp = p.sp[s];
    const long long step = *(volatile long long *)&p.st->step;
    const int P = (int)(step & 1);
    const long long n = (long long)p.st->count[s][P];
    const int32_t *__restrict__ cin = sp.cell[P];
    const float4 *__restrict__ vin = sp.pv[P];
    const float *__restrict__ zin = sp.vz[P];
    int32_t *__restrict__ cout = sp.cell[P ^ 1];
    float4 *__restrict__ vout = sp.pv[P ^ 1];
    float *__restrict__ zout = sp.vz[P ^ 1];
    unsigned long long *acc = p.acc + (size_t)s * p.nn;
    const int nx = p.nx, ny = p.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 2)
        s_abs[threadIdx.x] = 0u;
    __syncthreads();
    unsigned na0 = 0, na1 = 0;

    const long long ntiles = (n + kTile - 1) / kTile;
    for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long long base = t * kTile;
        int c[kItems];
        float4 q[kItems];
        float z[kItems];
        bool live[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const long long i = base + k * kThreads + threadIdx.x;
            live[k] = i < n;
            c[k] = -1;
            if (live[k]) {
                c[k] = __ldcs(cin + i);
                q[k] = __ldcs(vin + i);
                z[k] = __ldcs(zin + i);
            }
        }
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            const bool was = live[k];
            live[k] = live[k] && c[k] >= 0;
            if (live[k]) {
                const int cy = div_nx(p, c[k]), cx = c[k] - cy * nx;
                const int cx1 = (cx + 1 == nx) ? 0 : cx + 1;
                const int k00 = cy * nx + cx, k10 = cy * nx + cx1;
                const float2 e00 = __ldg(p.E + k00), e10 = __ldg(p.E + k10);
                const float2 e01 = __ldg(p.E + k00 + nx), e11 = __ldg(p.E + k10 + nx);
                const float ox = q[k].x, oy = q[k].y;
                float axp, ayp;
                accel2d(sp.qm, e00, e10, e01, e11, ox, oy, axp, ayp);
                float vx, vy;
                if (!push_v2_easy(sp.kind, q[k].z, q[k].w, z[k], axp, ayp, p.dt, sp.v0, vx, vy)) {
                    // the piece walk, here inline; counted for the diagnostics
                    namespace cg = cooperative_groups;
                    cg::coalesced_group g = cg::coalesced_threads();
                    if (g.thread_rank() == 0)
                        atomicAdd(&p.st->hard_n[s], (unsigned long long)g.size());
                    push_v2(sp.kind, q[k].z, q[k].w, z[k], axp, ayp, p.dt, sp.v0, vx, vy);
                }
                // x^{n+1} = x^n + beta(|v^{n+1/2}|) v^{n+1/2} dt, in cell units
                const float b = beta_q(sp.kind, vx, vy, z[k], sp.v0);
                const float xn = __fadd_rn(ox, __fmul_rn(__fmul_rn(b, vx), p.dt_dx));
                const float yn = __fadd_rn(oy, __fmul_rn(__fmul_rn(b, vy), p.dt_dx));
                const float fx = floorf(xn), fy = floorf(yn);
                int ncx = cx + (int)fx, ncy = cy + (int)fy;
                float dxn = __fsub_rn(xn, fx), dyn = __fsub_rn(yn, fy);
                if (dxn >= 1.0f) {
                    dxn = 0.0f;
                    ++ncx;
                }
                if (dyn >= 1.0f) {
                    dyn = 0.0f;
                    ++ncy;
                }
                if ((unsigned)ncx >= (unsigned)nx) {  // the x wrap
                    ncx %= nx;
                    if (ncx < 0)
                        ncx += nx;
                }
                if (ncy < 0) {
                    ++na0;
                    live[k] = false;
                } else if (ncy >= ny) {
                    ++na1;
                    live[k] = false;
                } else {
                    const int ncx1 = (ncx + 1 == nx) ? 0 : ncx + 1;
                    const int m00 = ncy * nx + ncx, m10 = ncy * nx + ncx1;
                    deposit2d(acc, m00, m10, m00 + nx, m10 + nx, b, dxn, dyn);
                    c[k] = m00;
                    q[k] = make_float4(dxn, dyn, vx, vy);
                }
            }
            if (!COMPACT && was) {
                const long long i = base + k * kThreads + threadIdx.x;
                if (live[k]) {
                    __stcs(cout + i, c[k]);
                    __stcs(vout + i, q[k]);
                    __stcs(zout + i, z[k]);
                } else {
                    __stcs(cout + i, -1);
                }
            }
        }
        if (COMPACT) {
            unsigned mask[kItems];
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                mask[k] = __ballot_sync(0xffffffffu, live[k]);
                if (lane == 0)
                    s_cnt[k * kWarps + warp] = __popc(mask[k]);
            }
            __syncthreads();
            if (warp == 0) {
                const int v = s_cnt[lane];
                int incl = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o)
                        incl += y;
                }
                s_cnt[lane] = incl - v;
                const int tot = __shfl_sync(0xffffffffu, incl, 31);
                if (lane == 0)
                    s_base = tot ? atomicAdd(&p.st->count[s][P ^ 1], (unsigned long long)tot) : 0ULL;
            }
            __syncthreads();
            const unsigned long long ob = s_base;
#pragma unroll
            for (int k = 0; k < kItems; ++k) {
                if (live[k]) {
                    const unsigned long long o = ob + (unsigned long long)s_cnt[k * kWarps + warp] +
                                                 __popc(mask[k] & ((1u << lane) - 1u));
                    __stcs(cout + o, c[k]);
                    __stcs(vout + o, q[k]);
                    __stcs(zout + o, z[k]);
                }
            }
            __syncthreads();  // s_cnt / s_base reused by the next tile
        }
    }
    na0 = __reduce_add_sync(0xffffffffu, na0);
    na1 = __reduce_add_sync(0xffffffffu, na1);
    if (lane == 0) {
        if (na0)
            atomicAdd(&s_abs[0], na0);
        if (na1)
            atomicAdd(&s_abs[1], na1);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_abs[threadIdx.x])
        atomicAdd(&p.st->absorbed_step[s][threadIdx.x], (unsigned long long)s_abs[threadIdx.x]);
}

// The move after the push: x^{n+1} = x^n + beta v^{n+1/2} dt in cell units from
// cell (cx, cy) and offset (ox, oy), the x wrap and the plates.  Returns 0 or 1 if
// the particle crossed the plate at y = 0 or y = Ly, else -1 with its new cell and
// offset.
__device__ __forceinline__ int move2d(const Params2D &p, int cx, int cy, float ox, float oy,
                                      float vx, float vy, float b, int &ncx, int &ncy,
                                      float &dxn, float &dyn)
{
    const int nx = p.nx;
    const float xn = __fadd_rn(ox, __fmul_rn(__fmul_rn(b, vx), p.dt_dx));
    const float yn = __fadd_rn(oy, __fmul_rn(__fmul_rn(b, vy), p.dt_dx));
    const float fx = floorf(xn), fy = floorf(yn);
    ncx = cx + (int)fx;
    ncy = cy + (int)fy;
    dxn = __fsub_rn(xn, fx);
    dyn = __fsub_rn(yn, fy);
    if (dxn >= 1.0f) {
        dxn = 0.0f;
        ++ncx;
    }
    if (dyn >= 1.0f) {
        dyn = 0.0f;
        ++ncy;
    }
    if ((unsigned)ncx >= (unsigned)nx) {  // the x wrap (at most a cell, but for beta = 1)
        ncx %= nx;
        if (ncx < 0)
            ncx += nx;
    }
    if (ncy < 0)
        return 0;
    if (ncy >= p.ny)
        return 1;
    return -1;
}

// ---------------------------------------------------------------------------------
// The in-place particle step with grid tiles in shared memory (the steps between
// cell sorts).  After the sort (every kCompact2d steps) consecutive slots hold
// particles of neighbouring cells, and each particle moves at most one cell per
// step, so a chunk of kChunk2d consecutive slots touches a small box of the grid.
// One CTA per chunk at a time:
//   1. the chunk is copied into shared memory by cp.async, 16 bytes each; a thread
//      fills the entries that it read out for the chunk before, so no barrier lies
//      between the two and the copies run while the window before is flushed;
//   2. the box of its cells, relative to the cell of a live particle near its
//      middle (x differences taken modulo nx, so a chunk that runs over the end of a
//      row is one box), widened by the gather's node and one cell of motion;
//   3. the window of nodes covering the box (at most kWin2d nodes) gets E copied in;
//   4. each particle is gathered, pushed, moved and deposited as k_particles2d does,
//      from and into the window where its four nodes are inside it, else from E and
//      into acc in global memory.  Lane l of a warp takes particles of slots kSeg2d l
//      on, so the lanes sit about a cell apart and their shared-memory atomics rarely
//      meet on a node.  A push that needs the piece walk is left to k_hard2d: its slot
//      goes to the step's list;
//   5. the chunk back to its slots, the window's deposits to acc (one atomic per
//      nonzero node) and cleared.
// The arithmetic per particle is that of k_particles2d (the same gathered values,
// push, move and quantised deposit), so the integer deposits and every particle are
// the same bit for bit; only where the charge is summed first differs.
//
// It is bound by instruction issue (about 450 instructions a particle; its 48 bytes of HBM
// traffic would take 475 us of the 960 at 1024^2 cells and 67 million particles), so what
// counts is few instructions and warps that are ready to issue: seven CTAs of 128 threads
// an SM, in different phases, rather than two of 512, which waited for each other at the
// barriers and for their copies (issue slots used 56% -> 66% with four of 256).  Measured
// there, with k_hard2d, a step: two CTAs of 512 threads and chunks of 2,048 1,640 us; four of
// 256 1,440; with cp.async, the two-word window sums and the slot list 1,190; the
// beta fixed 1,172; seven or eight of 128 and chunks of 512 1,070 (14 of 64: 1,170, the
// windows then cost more than the waiting).  At 256^2 and 2 million 124 -> 71 us.
// ---------------------------------------------------------------------------------
constexpr int kT2d = 128;                        // threads per CTA
constexpr int kTileCtas2d = 7;                   // CTAs per SM (227 KB of shared memory would hold 8)
constexpr int kPer2d = 4;                        // particles per thread per chunk
constexpr int kChunk2d = kT2d * kPer2d;          // 512 slots
constexpr int kSeg2d = kChunk2d / 32;            // slots of a lane's segment
constexpr int kWin2d = 768;                      // window nodes
static_assert(kSeg2d == 16 && kChunk2d <= 1024, "vslot2d, cslot2d; the limbs' range");

// Entries of slot j in shared memory, padded by 16 bytes a segment: a warp's 16-byte
// reads (a segment apart) meet no bank twice; its 4-byte reads neither, as the lanes of
// each group of eight take another of the four slots of a turn (phase 4).
__device__ __forceinline__ int vslot2d(int j) { return j + (j >> 4); }
__device__ __forceinline__ int cslot2d(int j) { return j + 4 * (j >> 4); }
constexpr int kVSlots2d = kChunk2d + 32, kCSlots2d = kChunk2d + 4 * 32;

size_t tile2d_smem_bytes()
{
    return (size_t)kVSlots2d * 16 + (size_t)kCSlots2d * (4 + 4) + (size_t)kWin2d * (8 + 4 + 4);
}

// The deposit rule of quantise2d in two signed words per node, value = hi 2^19 + lo: the
// window adds them by plain 32-bit atomics, without a carry.  For 0 <= x <= 1 and
// t = x 2^40 (exact):
//   x 2^21 + 1.5 2^23 rounds x 2^21 to the nearest integer (the float spacing there is
//        1), so hf, the sum less 1.5 2^23, is that integer and the sum's bits less those
//        of 1.5 2^23 are it as an int;
//   t - hf 2^19 is exact (|.| <= 2^18; both are multiples of the ulp of t, and at most 24
//        bits are left), and the same addition rounds it to an integer, ties to even:
//        rint(t), because hf 2^19 is an even integer.
// In the differences the bits of 1.5 2^23 cancel but for node (x+1, y+1).  |lo| of a
// deposit is at most 2^20 and a chunk adds at most 1,024 to a node: 2^30.  hi lies in
// [-2, 2^21 + 2], so its sum lies in [-2^16, 2^32 - 2^16): win_value.
__device__ __forceinline__ void quantise2d_limbs(float b, float ox, float oy, unsigned (&lo)[4],
                                                 unsigned (&hi)[4])
{
    const float bx = __fmul_rn(b, ox), by = __fmul_rn(b, oy), bxy = __fmul_rn(bx, oy);
    const float x[4] = {b, bx, by, bxy};
    unsigned l[4], h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float m = __fmaf_rn(x[k], 2097152.0f, 12582912.0f);
        const float hf = __fadd_rn(m, -12582912.0f);
        const float t = __fmul_rn(x[k], 1099511627776.0f);
        h[k] = __float_as_uint(m);
        l[k] = __float_as_uint(__fadd_rn(__fmaf_rn(hf, -524288.0f, t), 12582912.0f));
    }
    lo[0] = l[0] - l[1] - l[2] + l[3];
    hi[0] = h[0] - h[1] - h[2] + h[3];
    lo[1] = l[1] - l[3];
    hi[1] = h[1] - h[3];
    lo[2] = l[2] - l[3];
    hi[2] = h[2] - h[3];
    lo[3] = l[3] - 0x4B400000u;
    hi[3] = h[3] - 0x4B400000u;
}

// the value of a node's summed words
__device__ __forceinline__ unsigned long long win_value(unsigned lo, unsigned hi)
{
    const long long h = (long long)(hi + 65536u) - 65536;
    return (unsigned long long)(h * 524288 + (long long)(int)lo);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes)
                 : "memory");
}

template <int kKind>
__global__ void __launch_bounds__(kT2d, kTileCtas2d) k_particles2d_tiles(const __grid_constant__ Params2D p)
{
    extern __shared__ __align__(16) unsigned char smem2d[];
    float4 *s_v = reinterpret_cast<float4 *>(smem2d);                  // [kVSlots2d]
    float2 *s_E = reinterpret_cast<float2 *>(s_v + kVSlots2d);         // [kWin2d]
    int32_t *s_c = reinterpret_cast<int32_t *>(s_E + kWin2d);          // [kCSlots2d]
    float *s_z = reinterpret_cast<float *>(s_c + kCSlots2d);           // [kCSlots2d]
    unsigned *s_lo = reinterpret_cast<unsigned *>(s_z + kCSlots2d);    // [kWin2d]
    unsigned *s_hi = s_lo + kWin2d;                                    // [kWin2d]
    __shared__ int s_ref, s_box[2][4];  // reference cell; min dx, -max dx, min dy, -max dy
    __shared__ unsigned s_abs[2];
    __shared__ int s_nh;                         // the chunk's walked pushes: their number
    __shared__ unsigned short s_list[kChunk2d];  // and places

    const int s = blockIdx.y, tid = threadIdx.x;
    const Species2D &sp = p.sp[s];
    const long long step = *(volatile long long *)&p.st->step;
    const int P = (int)(step & 1);
    const long long n = (long long)p.st->count[s][P];
    const int32_t *__restrict__ cin = sp.cell[P];
    const float4 *__restrict__ vin = sp.pv[P];
    const float *__restrict__ zin = sp.vz[P];
    int32_t *__restrict__ cout = sp.cell[P ^ 1];
    float4 *__restrict__ vout = sp.pv[P ^ 1];
    float *__restrict__ zout = sp.vz[P ^ 1];
    unsigned long long *acc = p.acc + (size_t)s * p.nn;
    const int nx = p.nx, ny = p.ny;
    const int lane = tid & 31, warp = tid >> 5;
    const float qm = sp.qm, v0 = sp.v0, dt = p.dt;
    const int kind = kKind < 0 ? sp.kind : kKind;
    for (int k = tid; k < kWin2d; k += kT2d) {
        s_lo[k] = 0u;
        s_hi[k] = 0u;
    }
    if (tid < 8)
        s_box[tid >> 2][tid & 3] = INT_MAX;
    if (tid < 2)
        s_abs[tid] = 0u;
    if (tid == 0)
        s_nh = 0;
    __syncthreads();
    unsigned na0 = 0, na1 = 0;

    // ---- 1. a chunk into shared memory: this thread's four cells and vz (slots 4 tid on)
    // and its four of every kT2d (ox, oy, vx, vy); returns the cell of the middle slot
    auto load = [&](long long base, int cnt) -> int {
        const int left = cnt - 4 * tid;
        if (left > 0) {
            const int bytes = 4 * min(left, 4);
            cp_async16(s_c + cslot2d(4 * tid), cin + base + 4 * tid, bytes);
            cp_async16(s_z + cslot2d(4 * tid), zin + base + 4 * tid, bytes);
        }
#pragma unroll
        for (int i = 0; i < kPer2d; ++i) {
            const int j = tid + i * kT2d;
            if (j < cnt)
                cp_async16(s_v + vslot2d(j), vin + base + j, 16);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        return __ldcs(cin + base + cnt / 2);
    };

    const long long nchunks = (n + kChunk2d - 1) / kChunk2d;
    int ref_next = -1, turn = 0;
    if (blockIdx.x < nchunks)
        ref_next = load((long long)blockIdx.x * kChunk2d,
                        (int)min((long long)kChunk2d, n - (long long)blockIdx.x * kChunk2d));
    for (long long ch = blockIdx.x; ch < nchunks; ch += gridDim.x, turn ^= 1) {
        const long long base = ch * kChunk2d;
        const int cnt = (int)min((long long)kChunk2d, n - base);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // ---- 2. the reference cell (the middle slot's; if that is a hole, a live particle
        // after it, else before it) and the box of the chunk's cells relative to it
        int ref = ref_next;
        if (ref < 0) {
            __syncthreads();
            if (tid == 0) {
                int r = -1;
                for (int j = cnt / 2; j < cnt && r < 0; ++j)
                    r = s_c[cslot2d(j)];
                for (int j = cnt / 2 - 1; j >= 0 && r < 0; --j)
                    r = s_c[cslot2d(j)];
                s_ref = r;
            }
            __syncthreads();
            ref = s_ref;  // < 0: nothing live; the box is empty and phase 4 finds no particle
        }
        const int ry = ref < 0 ? 0 : div_nx(p, ref), rx = ref < 0 ? 0 : ref - ry * nx;
        {
            int mnx = INT_MAX, mxx = INT_MAX, mny = INT_MAX, mxy = INT_MAX;  // max as -min
            const int4 c4 = *reinterpret_cast<const int4 *>(s_c + cslot2d(4 * tid));
            const int cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int c = 4 * tid + k < cnt ? cc[k] : -1;
                if (c >= 0) {
                    const int cy = div_nx(p, c);
                    int dx = c - cy * nx - rx;  // to [-nx/2, nx/2)
                    if (dx >= nx - nx / 2)
                        dx -= nx;
                    else if (dx < -(nx / 2))
                        dx += nx;
                    const int dy = cy - ry;
                    mnx = min(mnx, dx);
                    mxx = min(mxx, -dx);
                    mny = min(mny, dy);
                    mxy = min(mxy, -dy);
                }
            }
            mnx = __reduce_min_sync(0xffffffffu, mnx);
            mxx = __reduce_min_sync(0xffffffffu, mxx);
            mny = __reduce_min_sync(0xffffffffu, mny);
            mxy = __reduce_min_sync(0xffffffffu, mxy);
            if (lane == 0) {
                atomicMin(&s_box[turn][0], mnx);
                atomicMin(&s_box[turn][1], mxx);
                atomicMin(&s_box[turn][2], mny);
                atomicMin(&s_box[turn][3], mxy);
            }
        }
        __syncthreads();  // the box, and the whole chunk in place
        // ---- 3. the window: node columns wx0 .. wx0+ww-1 (modulo nx), rows wy0 ..
        // wy0+wh-1, covering the box widened by the gather's node and one cell of
        // motion each way (cut to kWin2d nodes; particles outside it go to global memory)
        int ww = 0, wx0 = 0, wy0 = 0, wh = 0;
        if (ref >= 0) {
            const int *box = s_box[turn];
            ww = (-box[1]) - box[0] + 4;
            wx0 = rx + box[0] - 1;
            wy0 = max(0, ry + box[2] - 1);
            wh = min(ny, ry - box[3] + 2) - wy0 + 1;
            if (ww >= nx) {
                ww = nx;
                wx0 = 0;
            }
            wx0 %= nx;
            if (wx0 < 0)
                wx0 += nx;
            if (ww > kWin2d / 2)
                ww = kWin2d / 2;
            if (ww * wh > kWin2d)
                wh = kWin2d / ww;
        }
        if (tid < 4)
            s_box[turn ^ 1][tid] = INT_MAX;
        // a warp per window row, a lane per column
        for (int iy = warp; iy < wh; iy += kT2d / 32) {
            const float2 *Er = p.E + (size_t)(wy0 + iy) * nx;
            for (int ix = lane; ix < ww; ix += 32)
                s_E[iy * ww + ix] = __ldg(Er + (wx0 + ix < nx ? wx0 + ix : wx0 + ix - nx));
        }
        __syncthreads();
        // ---- 4. the particles, lanes of a warp a segment apart
#pragma unroll 1
        for (int k = 0; k < kPer2d; ++k) {
            const int j = lane * kSeg2d + warp * kPer2d + ((k + (lane >> 3)) & 3);
            const int qc = cslot2d(j), qv = vslot2d(j);
            const int c = j < cnt ? s_c[qc] : -1;
            if (c < 0)
                continue;
            const float4 pv = s_v[qv];
            const float z = s_z[qc];
            const int cy = div_nx(p, c), cx = c - cy * nx;
            int ix = cx - wx0;
            if (ix < 0)
                ix += nx;
            const int iy = cy - wy0;
            float2 e00, e10, e01, e11;
            if (ix <= ww - 2 && iy >= 0 && iy <= wh - 2) {
                const int k00 = iy * ww + ix;
                e00 = s_E[k00];
                e10 = s_E[k00 + 1];
                e01 = s_E[k00 + ww];
                e11 = s_E[k00 + ww + 1];
            } else {
                const int k10 = (cx + 1 == nx) ? c + 1 - nx : c + 1;
                e00 = __ldg(p.E + c);
                e10 = __ldg(p.E + k10);
                e01 = __ldg(p.E + c + nx);
                e11 = __ldg(p.E + k10 + nx);
            }
            float axp, ayp;
            accel2d(qm, e00, e10, e01, e11, pv.x, pv.y, axp, ayp);
            float vx, vy;
            if (!push_v2_easy(kind, pv.z, pv.w, z, axp, ayp, dt, v0, vx, vy)) {
                // the piece walk: k_hard2d pushes it and writes its slot
                s_list[atomicAdd(&s_nh, 1)] = (unsigned short)j;
                continue;
            }
            // x^{n+1} = x^n + beta(|v^{n+1/2}|) v^{n+1/2} dt, in cell units
            const float b = beta_q(kind, vx, vy, z, v0);
            int ncx, ncy;
            float dxn, dyn;
            const int wall = move2d(p, cx, cy, pv.x, pv.y, vx, vy, b, ncx, ncy, dxn, dyn);
            if (wall >= 0) {
                if (wall == 0)
                    ++na0;
                else
                    ++na1;
                s_c[qc] = -1;
                continue;
            }
            s_c[qc] = ncy * nx + ncx;
            s_v[qv] = make_float4(dxn, dyn, vx, vy);
            int nix = ncx - wx0;
            if (nix < 0)
                nix += nx;
            const int niy = ncy - wy0;
            if (nix <= ww - 2 && niy >= 0 && niy <= wh - 2) {
                unsigned lo[4], hi[4];
                quantise2d_limbs(b, dxn, dyn, lo, hi);
                unsigned *w0 = s_lo + niy * ww + nix, *w1 = w0 + ww;
                atomicAdd(w0, lo[0]);
                atomicAdd(w0 + kWin2d, hi[0]);
                atomicAdd(w0 + 1, lo[1]);
                atomicAdd(w0 + kWin2d + 1, hi[1]);
                atomicAdd(w1, lo[2]);
                atomicAdd(w1 + kWin2d, hi[2]);
                atomicAdd(w1 + 1, lo[3]);
                atomicAdd(w1 + kWin2d + 1, hi[3]);
            } else {
                const int m00 = ncy * nx + ncx, m10 = (ncx + 1 == nx) ? m00 + 1 - nx : m00 + 1;
                deposit2d(acc, m00, m10, m00 + nx, m10 + nx, b, dxn, dyn);
            }
        }
        __syncthreads();
        // ---- 5. the walked pushes to the list (their slots' contents here are overwritten
        // by k_hard2d), the chunk to its slots, the next chunk's copies, the window
        if (warp == 0) {
            const int nh = s_nh;
            if (nh) {
                unsigned long long hb = 0;
                if (lane == 0)
                    hb = atomicAdd(&p.st->hard_n[s], (unsigned long long)nh);
                hb = __shfl_sync(0xffffffffu, hb, 0);
                for (int i = lane; i < nh; i += 32)
                    sp.hard[hb + i] = (int32_t)(base + s_list[i]);
                if (lane == 0)
                    s_nh = 0;
            }
        }
        {
            const int4 c4 = *reinterpret_cast<const int4 *>(s_c + cslot2d(4 * tid));
            const float4 z4 = *reinterpret_cast<const float4 *>(s_z + cslot2d(4 * tid));
            const long long o = base + 4 * tid;
            const int left = cnt - 4 * tid;
            if (left >= 4) {
                __stcs(reinterpret_cast<int4 *>(cout + o), c4);
                __stcs(reinterpret_cast<float4 *>(zout + o), z4);
            } else if (left > 0) {
                __stcs(cout + o, c4.x);
                __stcs(zout + o, z4.x);
                if (left > 1) {
                    __stcs(cout + o + 1, c4.y);
                    __stcs(zout + o + 1, z4.y);
                }
                if (left > 2) {
                    __stcs(cout + o + 2, c4.z);
                    __stcs(zout + o + 2, z4.z);
                }
            }
#pragma unroll
            for (int i = 0; i < kPer2d; ++i) {
                const int j = tid + i * kT2d;
                if (j < cnt)
                    __stcs(vout + base + j, s_v[vslot2d(j)]);
            }
        }
        if (ch + gridDim.x < nchunks) {
            const long long nb = (ch + gridDim.x) * kChunk2d;
            ref_next = load(nb, (int)min((long long)kChunk2d, n - nb));
        }
        for (int iy = warp; iy < wh; iy += kT2d / 32) {
            unsigned long long *ar = acc + (size_t)(wy0 + iy) * nx;
            for (int ix = lane; ix < ww; ix += 32) {
                const int k = iy * ww + ix;
                const unsigned long long v = win_value(s_lo[k], s_hi[k]);
                s_lo[k] = 0u;
                s_hi[k] = 0u;
                if (v)
                    atomicAdd(ar + (wx0 + ix < nx ? wx0 + ix : wx0 + ix - nx), v);
            }
        }
    }
    na0 = __reduce_add_sync(0xffffffffu, na0);
    na1 = __reduce_add_sync(0xffffffffu, na1);
    if (lane == 0) {
        if (na0)
            atomicAdd(&s_abs[0], na0);
        if (na1)
            atomicAdd(&s_abs[1], na1);
    }
    __syncthreads();
    if (tid < 2 && s_abs[tid])
        atomicAdd(&p.st->absorbed_step[s][tid], (unsigned long long)s_abs[tid]);
}

// The instantiation for a simulation's species: the Heaviside beta fixed at compile time
// where all have it, else read per species (the same arithmetic).
typedef void (*TileKernel)(Params2D);

TileKernel tile_kernel(const Params2D &p)
{
    for (int s = 0; s < p.ns; ++s)
        if (p.sp[s].kind != SLPIC_BETA_HEAVISIDE)
            return k_particles2d_tiles<-1>;
    return k_particles2d_tiles<SLPIC_BETA_HEAVISIDE>;
}

// The particles the tile kernel listed: gathered again, the full push (series or piece walk, the
// arithmetic of the inline push), the move, the plates and the deposit by global
// atomics; each writes its own slot.  The species' lists are one index space.
__global__ void __launch_bounds__(256) k_hard2d(Params2D p)
{
    __shared__ unsigned s_abs[kMaxS][2];
    if (threadIdx.x < 2 * kMaxS)
        s_abs[threadIdx.x >> 1][threadIdx.x & 1] = 0u;
    __syncthreads();
    const long long step = *(volatile long long *)&p.st->step;
    const int P = (int)(step & 1);
    long long pre[kMaxS + 1];  // registers: constant indices only
    pre[0] = 0;
#pragma unroll
    for (int s = 0; s < kMaxS; ++s) {
        const long long n = s < p.ns ? (long long)*(volatile unsigned long long *)&p.st->hard_n[s] : 0;
        pre[s + 1] = pre[s] + n;
    }
    const long long total = pre[kMaxS];
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        int s = 0;
        long long i0 = 0;
#pragma unroll
        for (int r = 1; r < kMaxS; ++r)
            if (t >= pre[r]) {
                s = r;
                i0 = pre[r];
            }
        const Species2D &sp = p.sp[s];
        const int slot = __ldcs(sp.hard + (t - i0));
        const int c = sp.cell[P][slot];
        const float4 q = sp.pv[P][slot];
        const float z = sp.vz[P][slot];
        const int cy = div_nx(p, c), cx = c - cy * p.nx;
        const int k10 = (cx + 1 == p.nx) ? c + 1 - p.nx : c + 1;
        float ax, ay;
        accel2d(sp.qm, __ldg(p.E + c), __ldg(p.E + k10), __ldg(p.E + c + p.nx),
                __ldg(p.E + k10 + p.nx), q.x, q.y, ax, ay);
        float vx, vy;
        push_v2(sp.kind, q.z, q.w, z, ax, ay, p.dt, sp.v0, vx, vy);
        const float b = beta_q(sp.kind, vx, vy, z, sp.v0);
        int ncx, ncy;
        float dxn, dyn;
        const int wall = move2d(p, cx, cy, q.x, q.y, vx, vy, b, ncx, ncy, dxn, dyn);
        if (wall >= 0) {
            atomicAdd(&s_abs[s][wall], 1u);
            sp.cell[P ^ 1][slot] = -1;
        } else {
            const int nx = p.nx;
            const int ncx1 = (ncx + 1 == nx) ? 0 : ncx + 1;
            const int m00 = ncy * nx + ncx, m10 = ncy * nx + ncx1;
            deposit2d(p.acc + (size_t)s * p.nn, m00, m10, m00 + nx, m10 + nx, b, dxn, dyn);
            sp.cell[P ^ 1][slot] = m00;
            sp.pv[P ^ 1][slot] = make_float4(dxn, dyn, vx, vy);
            sp.vz[P ^ 1][slot] = z;
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * kMaxS) {
        const int s = threadIdx.x >> 1, w = threadIdx.x & 1;
        if (s < p.ns && s_abs[s][w])
            atomicAdd(&p.st->absorbed_step[s][w], (unsigned long long)s_abs[s][w]);
    }
}

// rho^0 from the particles of the current buffer (after a load)
__global__ void __launch_bounds__(kThreads) k_deposit2d(Params2D p)
{
    const int s = blockIdx.y;
    const Species2D &sp = p.sp[s];
    const int P = (int)(p.st->step & 1);
    const long long n = (long long)p.st->count[s][P];
    unsigned long long *acc = p.acc + (size_t)s * p.nn;
    const int nx = p.nx;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const int c = sp.cell[P][i];
        if (c < 0)
            continue;
        const float4 q = sp.pv[P][i];
        const int cy = c / nx, cx = c - cy * nx;
        const int cx1 = (cx + 1 == nx) ? 0 : cx + 1;
        const int k00 = cy * nx + cx, k10 = cy * nx + cx1;
        deposit2d(acc, k00, k10, k00 + nx, k10 + nx, beta_q(sp.kind, q.z, q.w, sp.vz[P][i], sp.v0),
                  q.x, q.y);
    }
}

// ---------------------------------------------------------------------------------
// Source (the 1D volume source with its band across y, x uniform over the period)
// and the step's bookkeeping.  Particle i of species s draws
// u_j = u24(SplitMix64(key(seed, step, s), 8i + j)): y = lo + u_0 len, x = u_5 nx (cells,
// FP32), a physical Maxwellian velocity from u_1..u_4 (Box-Muller).
// ---------------------------------------------------------------------------------
// The step's source count of species s (thread s): macroparticles k to make (cut to
// the room left; cut = true if it was), the first slot and the carried fraction.
__device__ __forceinline__ void source_count2d(const Params2D &p, const State2D *st, int s, int P,
                                               int compact, long long &k, long long &base,
                                               double &frac, bool &cut)
{
    double S = 0.0;
    if (p.src_mode == SLPIC_SRC_LOSS_MATCHED) {
        const int r = p.src_ref;
        S = (double)(st->absorbed_step[r][0] + st->absorbed_step[r][1]) * p.sp[r].w;
    } else if (p.src_mode == SLPIC_SRC_RATE) {
        S = p.src_rate * p.dt64;
    }
    k = 0;
    double f = st->src_frac[s];
    if (p.src_mode != SLPIC_SRC_NONE && p.sp[s].vth_src > 0.0f) {
        f = fma(S, p.sp[s].inv_w, f);
        k = (long long)floor(f);
        f -= (double)k;
    }
    // in place: the output uses the input's slots; compacted: counted by atomics
    base = (long long)(compact ? st->count[s][P ^ 1] : st->count[s][P]);
    const long long room = p.sp[s].capacity - base;
    cut = k > room;
    if (cut)
        k = room;
    frac = f;
}

// Every CTA derives the step's counts from the same state and makes its share of the
// species' particles, taken as one index space; k_book2d then updates the state.
__global__ void __launch_bounds__(256) k_inject2d(Params2D p, int compact)
{
    __shared__ long long s_k[kMaxS], s_base[kMaxS];
    const State2D *st = p.st;
    const long long step = st->step;
    const int P = (int)(step & 1);
    const int ns = p.ns;
    if ((int)threadIdx.x < kMaxS) {
        const int s = threadIdx.x;
        long long k = 0, base = 0;
        double f;
        bool cut;
        if (s < ns)
            source_count2d(p, st, s, P, compact, k, base, f, cut);
        s_k[s] = k;
        s_base[s] = base;
    }
    __syncthreads();
    long long pre[kMaxS + 1];  // registers: constant indices only
    pre[0] = 0;
#pragma unroll
    for (int s = 0; s < kMaxS; ++s)
        pre[s + 1] = pre[s] + s_k[s];
    const long long total = pre[kMaxS];
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        int s = 0;
        long long i0 = 0;
#pragma unroll
        for (int r = 1; r < kMaxS; ++r)
            if (t >= pre[r]) {
                s = r;
                i0 = pre[r];
            }
        const long long i = t - i0;
        const Species2D &sp = p.sp[s];
        const unsigned long long key = sm64_stream(p.seed, (unsigned long long)step, (unsigned)s);
        unsigned long long *acc = p.acc + (size_t)s * p.nn;
        const unsigned long long b8 = 8ULL * (unsigned long long)i;
        const float u0 = u24(sm64_at(key, b8 + 0)), u1 = u24(sm64_at(key, b8 + 1));
        const float u2 = u24(sm64_at(key, b8 + 2)), u3 = u24(sm64_at(key, b8 + 3));
        const float u4 = u24(sm64_at(key, b8 + 4)), u5 = u24(sm64_at(key, b8 + 5));
        const float yc = __fadd_rn(p.src_lo, __fmul_rn(u0, p.src_len));
        float xc = __fmul_rn(u5, (float)p.nx);
        if (xc >= (float)p.nx)
            xc = 0.0f;
        const float fx = floorf(xc), fy = floorf(yc);
        const int cx = (int)fx, cy = min(max((int)fy, 0), p.ny - 1);
        const float ox = __fsub_rn(xc, fx), oy = __fsub_rn(yc, fy);
        const float r1 = sqrtf(-2.0f * logf(u1)), r2 = sqrtf(-2.0f * logf(u3));
        float s2, c2;
        sincospif(2.0f * u2, &s2, &c2);
        const float vx = sp.vth_src * r1 * c2, vy = sp.vth_src * r1 * s2;
        const float vz = sp.vth_src * r2 * cospif(2.0f * u4);
        const long long o = s_base[s] + i;
        const int c = cy * p.nx + cx;
        sp.cell[P ^ 1][o] = c;
        sp.pv[P ^ 1][o] = make_float4(ox, oy, vx, vy);
        sp.vz[P ^ 1][o] = vz;
        const int cx1 = (cx + 1 == p.nx) ? 0 : cx + 1;
        deposit2d(acc, c, cy * p.nx + cx1, c + p.nx, cy * p.nx + cx1 + p.nx,
                  beta_q(sp.kind, vx, vy, vz, sp.v0), ox, oy);
    }
}

// The step's bookkeeping, after the source (one warp; thread s for species s, from
// the same counts as k_inject2d); the step index last.
__global__ void k_book2d(Params2D p, int compact)
{
    State2D *st = p.st;
    const long long step = st->step;
    const int P = (int)(step & 1);
    if ((int)threadIdx.x < p.ns) {
        const int s = threadIdx.x;
        long long k, base;
        double f;
        bool cut;
        source_count2d(p, st, s, P, compact, k, base, f, cut);
        if (cut)
            atomicCAS(&st->error, 0, SLPIC_ERR_CAPACITY);
        const unsigned long long a0 = st->absorbed_step[s][0], a1 = st->absorbed_step[s][1];
        st->src_frac[s] = f;
        st->holes[s][P ^ 1] = compact ? 0ULL : st->holes[s][P] + a0 + a1;
        st->count[s][P ^ 1] = (unsigned long long)(base + k);
        st->injected_total[s] += k;
        st->absorbed_total[s][0] += (long long)a0;
        st->absorbed_total[s][1] += (long long)a1;
        st->absorbed_step[s][0] = 0ULL;
        st->absorbed_step[s][1] = 0ULL;
        st->count[s][P] = 0ULL;
        st->holes[s][P] = 0ULL;
    }
    __syncwarp();
    if (threadIdx.x == 0) {
        unsigned long long it = 0;
        for (int s = 0; s < p.ns; ++s)
            it += st->hard_n[s];
        st->iter_last = it;
    }
    __syncwarp();
    if ((int)threadIdx.x < p.ns)
        st->hard_n[threadIdx.x] = 0ULL;
    if (threadIdx.x == 0)
        st->step = step + 1;
}

// ---------------------------------------------------------------------------------
// Field solve.  The unknowns are phi on rows j = 1..ny-1; with A the 5-point
// stencil times dx^2 (diagonal 4) and the plates moved to the right-hand side,
// A phi = b = (dx^2/eps0) rho + [j = 1] phi_lo + [j = ny-1] phi_hi.  Jacobi-
// preconditioned CG (M = 4 I) from the previous phi:
//   r = b - A phi, p = r/4, rz = r.r/4
//   loop: q = A p; alpha = rz / p.q; phi += alpha p; r -= alpha q;
//         stop if r.r <= rtol^2 b.b; p = r/4 + (r.r/4 / rz) p
// Each iteration is two grid-wide phases: (p, q = A p, p.q) and (phi, r, r.r), the
// new p formed on the fly from r and the previous p (two p buffers).  Dot products
// are FP64 per-CTA partial sums, added in CTA order by every CTA: the same value
// everywhere and in every run.
// ---------------------------------------------------------------------------------

// The CG's sums and barriers are one: a virtual CTA of kCgVirtual threads writes its
// partial sum to its slot, and every CTA polls all slots and adds them itself, in one
// fixed order (the same value everywhere and in every run).  That costs a write and a
// read of L2; a barrier of counters (atomics by groups, a generation word, sleeps) and
// then a read of the sums took 11 us a sum on 304 CTAs (now 6 at 250 x 241, 4 at 64 x 48).
// Slots go by three turns: a CTA empties its slots of the next turn before it writes this
// one's, when every CTA has passed the turn before and so read the one that used them.
//
// The order of the additions is that of cg_v CTAs of kCgVirtual threads, whatever is
// launched (a tree over each warp's lanes, the warps in order, the same over the CTAs'
// sums): CTAs of two virtual ones, and none for virtual CTAs without nodes, whose sums
// are zero.  What a sum costs is FP64 latency (an addition is 110 cycles on an idle pipe
// of 2 lanes an SM): the trees' levels are packed into as few warps as have pairs left,
// and the scalar work that follows is thread 0's alone (then, below).
constexpr unsigned long long kCgEmpty = ~0ULL;  // a NaN that no sum is stored as

struct CgShared {
    double v[kCgThreads], g[kCgVirtual];
};

struct CgSync {
    CgShared *sh;
    double *part;
    int v;     // virtual CTAs
    int turn;  // of the next sum
    int *error;
};

// float -> double on the integer pipe (the conversion instruction takes the FP64 pipe);
// zeros, subnormals, infinities and NaN by the instruction
__device__ __forceinline__ double cg_double(float x)
{
    const unsigned u = __float_as_uint(x), e = u & 0x7F800000u;
    if (e == 0u || e == 0x7F800000u)
        return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// (float)(a / b), the FP64 quotient rounded to FP32, without the FP64 division's chain of
// some 15 dependent instructions: the significands as pairs of floats and Dekker's quotient of
// such pairs (Numer. Math. 18, 1971: a first quotient, corrected by its remainder, which a
// fused multiply-add leaves exact), good to 2^-43, rounded; the FP64 division where that lies
// within 2^-38 of the middle between two floats (one quotient in 2^13), or where the operands
// or the quotient leave the normal range.
__device__ __forceinline__ float cg_quotient(double a, double b)
{
    const unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
    const unsigned bh = (unsigned)__double2hiint(b), bl = (unsigned)__double2loint(b);
    const int ea = (int)(ah >> 20), eb = (int)(bh >> 20);  // sign included: negative is out of range
    const int e = ea - eb;
    if (ea >= 1 && ea < 2047 && eb >= 1 && eb < 2047 && e > -120 && e < 120) {
        // 1.m = hi + lo: 24 bits and the 29 below them
        const float xh = __uint_as_float(0x3F800000u | ((ah & 0xFFFFFu) << 3) | (al >> 29));
        const float yh = __uint_as_float(0x3F800000u | ((bh & 0xFFFFFu) << 3) | (bl >> 29));
        const float xl = __fmul_rn((float)(al & 0x1FFFFFFFu), 0x1p-52f);
        const float yl = __fmul_rn((float)(bl & 0x1FFFFFFFu), 0x1p-52f);
        const float inv = __frcp_rn(yh);
        const float q0 = __fmul_rn(xh, inv);
        const float r = __fmaf_rn(-q0, yh, xh);  // exact
        const float q1 = __fmul_rn(__fmaf_rn(-q0, yl, __fadd_rn(r, xl)), inv);
        const float q = __fadd_rn(q0, q1);
        const float d = __fsub_rn(q1, __fsub_rn(q, q0));  // the quotient is q + d
        // the middles to q's neighbours lie half an ulp off (a quarter below a power of two)
        const float ulp = q >= 1.0f ? 0x1p-23f : 0x1p-24f;
        const float m = fabsf(d);
        if (fabsf(__fsub_rn(m, 0.5f * ulp)) > 0x1p-38f && fabsf(__fsub_rn(m, 0.25f * ulp)) > 0x1p-38f && q > 0.5f)
            return __fmul_rn(q, __uint_as_float((unsigned)(e + 127) << 23));
    }
    return (float)(a / b);
}

__device__ __forceinline__ void cg_release()
{
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
}
__device__ __forceinline__ unsigned long long cg_acquire(const unsigned long long *a)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cg_store(unsigned long long *a, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}

// The sum of v over all threads, given to then(sum) in every CTA's thread 0; also a
// barrier of all CTAs, after which their writes before it are visible (read them through
// L2) and what then() left in shared memory is.  False if a wait gave up.
template <typename Then>
__device__ __forceinline__ bool cg_sum(CgSync &sy, double v, Then then)
{
    // the second tree has its own array: another warp may be there while the first still
    // reads the last level of its own
    double *s_v = sy.sh->v, *s_g = sy.sh->g;
    constexpr int kW = kCgThreads / 32, kVW = kCgVirtual / 32;  // warps, of them a virtual CTA's
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long *slots = reinterpret_cast<unsigned long long *>(sy.part);
    // tree over the lanes of every warp: lane l of warp w at l kW + w, so that a level's
    // pairs are threads next to one another
    s_v[lane * kW + warp] = v;
    __syncthreads();
    double g = 0.0;
#pragma unroll
    for (int n = kCgThreads / 2; n >= 32; n >>= 1) {  // lanes l and l + n / kW
        if (t < n) {
            g = (n == kCgThreads / 2 ? s_v[t] : g) + s_v[t + n];
            if (t >= n / 2 && n > 32)
                s_v[t] = g;
        }
        if (n > 32)
            __syncthreads();
    }
    if (warp == 0) {
        static_assert(kW == 16, "the last level's pairs are half a warp apart");
        g += __shfl_down_sync(0xffffffffu, g, 16);  // lane w: the sum of warp w
        double c = 0.0;
#pragma unroll
        for (int k = 0; k < kVW; ++k)
            c += __shfl_sync(0xffffffffu, g, (lane & kVW) + k);
        if (lane == 0 || lane == kVW) {
            const int vcta = blockIdx.x * 2 + (lane ? 1 : 0), next = sy.turn == 2 ? 0 : sy.turn + 1;
            cg_store(slots + next * sy.v + vcta, kCgEmpty);
            cg_release();  // the CTA's writes (seen through the barriers) and the emptied slot
            cg_store(slots + sy.turn * sy.v + vcta,
                     isnan(c) ? 0x7FF8000000000000ULL : (unsigned long long)__double_as_longlong(c));
        }
    }
    bool ok = true;
    g = 0.0;
    if (t < kCgVirtual) {
        const long long t0 = clock64();
        for (int b = t; b < (int)gridDim.x * 2; b += kCgVirtual) {
            unsigned long long u;
            while ((u = cg_acquire(slots + sy.turn * sy.v + b)) == kCgEmpty)
                if (clock64() - t0 > kCgWaitCycles) {
                    atomicCAS(sy.error, 0, SLPIC_ERR_TIMEOUT);
                    ok = false;
                    break;
                }
            const double x = __longlong_as_double((long long)u);
            g = b < kCgVirtual ? x : g + x;
        }
        s_g[lane * kVW + warp] = g;  // the same tree over the virtual CTAs' sums
    }
    sy.turn = sy.turn == 2 ? 0 : sy.turn + 1;
    if (!__syncthreads_and(ok))
        return false;
#pragma unroll
    for (int n = kCgVirtual / 2; n >= 32; n >>= 1) {
        if (t < n) {
            g = (n == kCgVirtual / 2 ? s_g[t] : g) + s_g[t + n];
            if (t >= n / 2 && n > 32)
                s_g[t] = g;
        }
        if (n > 32)
            __syncthreads();
    }
    if (warp == 0) {
        g += __shfl_down_sync(0xffffffffu, g, 16);
        g += __shfl_down_sync(0xffffffffu, g, 8);
        double c = 0.0;
#pragma unroll
        for (int k = 0; k < kVW; ++k)
            c += __shfl_sync(0xffffffffu, g, k);
        if (lane == 0)
            then(c);
    }
    __syncthreads();
    return true;
}

// Arrays written by other CTAs of the cooperative grid are read with __ldcg
// (L2, not the CTA's own L1).
__device__ __forceinline__ double stencil(const double *u, int idx, int i, int nx)
{
    const int ip = (i + 1 == nx) ? idx + 1 - nx : idx + 1;
    const int im = (i == 0) ? idx - 1 + nx : idx - 1;
    return 4.0 * __ldcg(u + idx) -
           (__ldcg(u + ip) + __ldcg(u + im) + __ldcg(u + idx - nx) + __ldcg(u + idx + nx));
}

// E = -grad phi at node idx: centred differences, one-sided on the plates, periodic
// in x.  phi is read through L2 (written by other CTAs of the same grid).
__device__ __forceinline__ void store_E(const Params2D &p, int idx)
{
    const int nx = p.nx, ny = p.ny;
    const int j = idx / nx, i = idx - j * nx;
    const int ip = (i + 1 == nx) ? idx + 1 - nx : idx + 1;
    const int im = (i == 0) ? idx - 1 + nx : idx - 1;
    const double *f = p.phi;
    const double ex = -(__ldcg(f + ip) - __ldcg(f + im)) * p.half_dx;
    double ey;
    if (j == 0)
        ey = -(__ldcg(f + idx + nx) - __ldcg(f + idx)) / p.dx;
    else if (j == ny)
        ey = -(__ldcg(f + idx) - __ldcg(f + idx - nx)) / p.dx;
    else
        ey = -(__ldcg(f + idx + nx) - __ldcg(f + idx - nx)) * p.half_dx;
    p.E[idx] = make_float2((float)ex, (float)ey);
}

// mode 0: the simulation's solve (b from the deposits, which are then cleared;
// E written).  mode 1: b from p.r's initial content as rho (slpic2d_solve_poisson).
//
// Mixed precision with reliable updates: b and the solution phi are FP64; the CG
// iterates (search direction p, correction d, residual r) are FP32, with dot
// products summed in FP64.  Whenever the FP32 recursive residual has fallen by
// kUpdateDrop since the last update (or below the target), d is added to phi in
// FP64 and r is replaced by the true residual b - A phi formed in FP64; the search
// direction carries on, so the iteration keeps the convergence of one unbroken CG
// run, unless the true residual came out more than twice the recursive one (the
// FP32 recursion had drifted), when the search direction starts afresh.  At
// 1024 x 1024 with a plasma's smooth charge the correction is as large as phi
// itself early on, which limits how far an FP32 recursion can be trusted: hence
// an update at every tenfold drop.  The solve ends when that true residual meets ||b - A phi|| <= rtol ||b||,
// the figure reported.  FP64 arithmetic, narrow on this GPU, is left to the few
// updates.
//
// Node t of the interior belongs to thread t modulo the virtual grid's threads, at most K
// per thread, whose r, d, q and p stay in its registers: only the p and r that neighbours
// read go to memory.  K = 0: any number, all in memory (fd, fq).
constexpr double kUpdateDrop = 1e-1;

template <int K>
__global__ void __launch_bounds__(kCgThreads, 1) k_cg2d(const __grid_constant__ Params2D p, int mode)
{
    State2D *st = p.st;
    const int nx = p.nx, ny = p.ny, nn = p.nn;
    const int first = nx, last = ny * nx;  // interior nodes [first, last)
    const long long gtid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long gstride = (long long)p.cg_v * kCgVirtual;
    double *b64 = p.q;  // right-hand side, kept for the true residuals
    __shared__ CgShared s_sums;
    CgSync sy{&s_sums, p.part, p.cg_v, 0, &st->error};

    // ---- b (FP64, interior rows; 0 on the plates) and ||b||^2; FP32 iterates zeroed
    double bb = 0.0;
    for (long long t = gtid; t < nn; t += gstride) {
        const int idx = (int)t;
        const int j = idx / nx;
        double rho = 0.0;
        if (mode == 0) {
            for (int s = 0; s < p.ns; ++s) {
                unsigned long long *a = p.acc + (size_t)s * nn + idx;
                rho = fma(p.sp[s].rho_unit, (double)(long long)*a, rho);
                *a = 0ULL;
            }
        } else {
            rho = p.r[idx];
        }
        double b = 0.0;
        if (idx >= first && idx < last) {
            b = p.k2 * rho;
            if (j == 1)
                b += p.phi_lo;
            if (j == ny - 1)
                b += p.phi_hi;
        }
        b64[idx] = b;
        bb = fma(b, b, bb);
        p.fr[idx] = 0.0f;
        p.fpA[idx] = 0.0f;
        p.fpB[idx] = 0.0f;
        if (K == 0)
            p.fd[idx] = 0.0f;
    }
    // thread 0's scalars (no other thread has them), and what it tells the others
    double BB = 0.0, rz = 0.0, rlast = 0.0, rin = 0.0, RR = 0.0;
    __shared__ float s_f;   // alpha or beta
    __shared__ int s_what;  // 0 go on, 1 a reliable update is due, 2 solved
    if (!cg_sum(sy, bb, [&](double v) { BB = v == 0.0 ? 1.0 : v; }))
        return;

    // this thread's nodes: their place at the period's ends (bits: i == 0, i == nx - 1),
    // and the iterates
    int edge[K > 0 ? K : 1];  // (the plates' p and r are zero: no case of their own)
    float rk[K > 0 ? K : 1], dk[K > 0 ? K : 1], qk[K > 0 ? K : 1], pk[K > 0 ? K : 1];
    const int t0 = (int)gtid + first, stride = (int)gstride;
    auto edge_of = [&](int idx) {
        const int j = idx / nx, i = idx - j * nx;
        return (i == 0 ? 1 : 0) | (i == nx - 1 ? 2 : 0);
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int idx = t0 + k * stride;
        edge[k] = idx < last ? edge_of(idx) : 0;
        dk[k] = qk[k] = pk[k] = rk[k] = 0.0f;
    }

    int it = 0;
    // true residual in FP64: r = b - A phi (A phi on the unknowns = the full stencil
    // on phi, plate rows included, plus the plate terms held in b), stored in FP32
    auto true_residual = [&]() -> bool {
        double rr = 0.0;
        auto one = [&](int idx) {
            const int j = idx / nx, i = idx - j * nx;
            double ap = stencil(p.phi, idx, i, nx);
            if (j == 1)
                ap += p.phi_lo;
            if (j == ny - 1)
                ap += p.phi_hi;
            const double r = __ldcg(b64 + idx) - ap;
            rr = fma(r, r, rr);
            const float f = (float)r;
            p.fr[idx] = f;
            return f;
        };
        if (K > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (t0 + k * stride < last)
                    rk[k] = one(t0 + k * stride);
        } else {
            for (long long t = gtid + first; t < last; t += gstride)
                one((int)t);
        }
        return cg_sum(sy, rr, [&](double v) {
            RR = v;
            // the FP32 recursion had drifted from the truth (true residual more than twice
            // the recursive one): its search direction is stale, start afresh
            const bool restart = it == 0 || RR > 4.0 * rin;
            const double rz1 = 0.25 * RR;
            s_f = restart ? 0.0f : cg_quotient(rz1, rz);
            s_what = RR <= p.rtol2 * BB ? 2 : 0;
            rz = rz1;
            rlast = RR;
        });
    };
    if (!true_residual())
        return;
    bool done = s_what == 2;
    float bf = s_f;
    float *pold = p.fpA, *pnew = p.fpB;
    while (!done && it < p.cg_maxit) {
        // phase 1: p = r/4 + beta p_old at the node and its neighbours, q = A p
        double pq = 0.0;
        struct Nb {
            float pe, re, pw, rw, pn, rn, ps, rs;
        };
        auto load = [&](int idx, int e) {
            const int ip = (e & 2) ? idx + 1 - nx : idx + 1;
            const int im = (e & 1) ? idx - 1 + nx : idx - 1;
            return Nb{__ldcg(pold + ip),       __ldcg(p.fr + ip),       __ldcg(pold + im),
                      __ldcg(p.fr + im),       __ldcg(pold + idx + nx), __ldcg(p.fr + idx + nx),
                      __ldcg(pold + idx - nx), __ldcg(p.fr + idx - nx)};
        };
        auto direction = [&](const Nb &n, float po, float ro, float &pc) {
            pc = fmaf(bf, po, 0.25f * ro);
            const float pe = fmaf(bf, n.pe, 0.25f * n.re);
            const float pw = fmaf(bf, n.pw, 0.25f * n.rw);
            const float pn = fmaf(bf, n.pn, 0.25f * n.rn);
            const float ps = fmaf(bf, n.ps, 0.25f * n.rs);
            return 4.0f * pc - (pe + pw + pn + ps);
        };
        if (K > 0) {
            constexpr int kB = K > 0 && K < 4 ? K : 4;  // nodes whose loads are in flight together
#pragma unroll
            for (int k0 = 0; k0 < K; k0 += kB) {
                Nb nb[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k)
                    nb[k] = load(min(t0 + (k0 + k) * stride, last - 1), edge[k0 + k]);
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int idx = t0 + (k0 + k) * stride;
                    if (idx < last) {
                        float pc;
                        const float qv = direction(nb[k], pk[k0 + k], rk[k0 + k], pc);
                        qk[k0 + k] = qv;
                        pk[k0 + k] = pc;
                        pnew[idx] = pc;
                        pq = fma(cg_double(pc), cg_double(qv), pq);
                    }
                }
            }
        } else {
            for (long long t = gtid + first; t < last; t += gstride) {
                const int idx = (int)t;
                float pc;
                const float qv =
                    direction(load(idx, edge_of(idx)), __ldcg(pold + idx), __ldcg(p.fr + idx), pc);
                pnew[idx] = pc;
                p.fq[idx] = qv;
                pq = fma(cg_double(pc), cg_double(qv), pq);
            }
        }
        if (!cg_sum(sy, pq, [&](double v) { s_f = cg_quotient(rz, v); }))  // alpha
            return;
        const float af = s_f;
        // phase 2: d += alpha p, r -= alpha q
        double r2 = 0.0;
        if (K > 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int idx = t0 + k * stride;
                if (idx < last) {
                    dk[k] = fmaf(af, pk[k], dk[k]);
                    rk[k] = fmaf(-af, qk[k], rk[k]);
                    p.fr[idx] = rk[k];
                    r2 = fma(cg_double(rk[k]), cg_double(rk[k]), r2);
                }
            }
        } else {
            for (long long t = gtid + first; t < last; t += gstride) {
                const int idx = (int)t;
                p.fd[idx] = fmaf(af, pnew[idx], p.fd[idx]);
                const float r = fmaf(-af, p.fq[idx], p.fr[idx]);
                p.fr[idx] = r;
                r2 = fma(cg_double(r), cg_double(r), r2);
            }
        }
        ++it;
        if (!cg_sum(sy, r2, [&](double v) {
                rin = v;
                const bool update = rin <= kUpdateDrop * kUpdateDrop * rlast || rin <= 0.25 * p.rtol2 * BB ||
                                    it >= p.cg_maxit;
                s_what = update ? 1 : 0;
                if (!update) {
                    const double rz1 = 0.25 * rin;
                    s_f = cg_quotient(rz1, rz);  // beta
                    rz = rz1;
                }
            }))
            return;
        if (s_what == 1) {
            // reliable update: phi += d in FP64, r replaced by the true residual
            if (K > 0) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (t0 + k * stride < last) {
                        p.phi[t0 + k * stride] += (double)dk[k];
                        dk[k] = 0.0f;
                    }
            } else {
                for (long long t = gtid + first; t < last; t += gstride) {
                    const int idx = (int)t;
                    p.phi[idx] += (double)p.fd[idx];
                    p.fd[idx] = 0.0f;
                }
            }
            if (!cg_sum(sy, 0.0, [](double) {}))
                return;
            if (!true_residual())
                return;
            done = s_what == 2;
        }
        bf = s_f;
        float *tmp = pold;
        pold = pnew;
        pnew = tmp;
    }
    // E on every node from the final phi (complete after the last barrier)
    if (mode == 0)
        for (long long t = gtid; t < nn; t += gstride)
            store_E(p, (int)t);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->cg_iters = it;
        st->cg_total += it;
        st->cg_res = sqrt(RR / BB);
        if (!done)
            atomicCAS(&st->error, 0, SLPIC_ERR_NOCONVERGE);
    }
}

// the instantiation for a grid: the fewest registers that hold its nodes per thread
typedef void (*CgKernel)(Params2D, int);

CgKernel cg_kernel(const Params2D &p)
{
    const long long threads = (long long)p.cg_v * kCgVirtual, nodes = (long long)(p.ny - 1) * p.nx;
    const long long k = (nodes + threads - 1) / threads;
    return k <= 1 ? k_cg2d<1> : k <= 2 ? k_cg2d<2> : k <= 4 ? k_cg2d<4> : k <= 8 ? k_cg2d<8>
         : k <= 16 ? k_cg2d<16> : k_cg2d<0>;
}

// CTAs that have nodes
int cg_grid(const Params2D &p)
{
    return (int)std::min<long long>(p.cg_v / 2, ((long long)p.nn + kCgThreads - 1) / kCgThreads);
}

// ---- the direct solver (SLPIC2D_SOLVER_FFT) -----------------------------------------
// The 5-point system A phi = b on the interior rows j = 1..ny-1 is periodic in x,
// so the discrete Fourier transform along x diagonalises its x part: mode k of row
// j obeys (4 - 2 cos(2 pi k/nx)) u_j - u_{j-1} - u_{j+1} = b^_j with u_0 = u_ny = 0
// (the plate potentials are in b).  Three passes, in FP64: a forward FFT per row, the
// Thomas algorithm per mode (the multipliers tabulated at creation), the inverse FFT per
// row.  Then E and the true residual as for the CG.
//
// The arithmetic is that of a complex radix-2 transform (decimation in time) with unfused
// butterflies, of Thomas in 32 segments, to the last bit: what a wall absorbs turns on E's
// last bits, so a transform that rounds otherwise (of half the length, with fused
// multiply-adds: 166 us at 1,024^2) would change every run.  The FP64 pipe (2 lanes an SM)
// bounds the large grids: some 40 thousand instructions a row of 1,024 each way.  Small
// grids are bound by latency, so a thread keeps its points in registers over several levels
// of butterflies and the row's threads meet in shared memory only between those, twiddles and
// coefficients straight from L2 to registers.  The solve of a step (with the residual's report, a
// launch of its own before): 1,024^2 445 -> 299 us (the rows 117 us, 77% of the FP64 pipe),
// 256^2 73 -> 52.
constexpr int kFftMaxThreads = 512;
constexpr int kFinishThreads = 128;

// Levels of butterflies that a thread does between two meetings, on 2^levels points: 3, or
// 1 where that leaves fewer than 512 warps (3 an SM), too few to hide the FP64 latency.  The
// solve of a step with 1 and with 3: 64 x 64 37.2 and 45.4 us, 64 x 1,000 (250 warps with 3)
// 59.6 and 65.3, 256^2 52.4 and 57.8, 512^2 (1,022) 104.5 and 93.9, 1,024^2 316 and 299.
// Rows of fewer than 8 points always 1: they do not fill a thread's 8.
int fft_levels(int nx, int ny)
{
    return nx < 8 || ((long long)(ny - 1) * nx >> 8) < 512 ? 1 : 3;
}
// threads of a row's transform, and rows of a CTA (a warp at least)
__host__ __device__ __forceinline__ int fft_row_threads(int nx, int levels)
{
    const int T = nx >> levels ? nx >> levels : 1;
    return T < kFftMaxThreads ? T : kFftMaxThreads;
}
__host__ __device__ __forceinline__ int fft_cta_rows(int nx, int levels)
{
    const int T = fft_row_threads(nx, levels);
    return T < 32 ? 32 / T : 1;
}

// Place of point i of a row in shared memory: the low three bits of the place are mixed
// with the bits above, so that eight threads meet eight different 16-byte banks whichever
// three bits of i tell them apart.  Linear: the place of a sum of numbers without a bit in
// common is the exclusive or of theirs.
__device__ __forceinline__ int fft_place(int i) { return i ^ (((i >> 3) ^ (i >> 6) ^ (i >> 9)) & 7); }

// (u, v) -> (u + w v, u - w v), w = (wr, wi)
__device__ __forceinline__ void butterfly(double2 &u, double2 &v, double wr, double wi)
{
    const double tr = wr * v.x - wi * v.y, ti = wr * v.y + wi * v.x;
    const double2 a = u;
    u = make_double2(a.x + tr, a.y + ti);
    v = make_double2(a.x - tr, a.y - ti);
}
// w = 1
__device__ __forceinline__ void butterfly1(double2 &u, double2 &v)
{
    const double2 a = u, b = v;
    u = make_double2(a.x + b.x, a.y + b.y);
    v = make_double2(a.x - b.x, a.y - b.y);
}

// R levels from the first (points a unit apart; w: the tabulated eighths of a turn)
template <int R, bool INV>
__device__ __forceinline__ void first_levels(double2 *z, const double2 (&w)[4])
{
#pragma unroll
    for (int d = 0; d < R; ++d)
#pragma unroll
        for (int r = 0; r < (1 << R); ++r)
            if (!(r >> d & 1)) {
                const int e = (r & ((1 << d) - 1)) << (2 - d);
                if (e == 0)
                    butterfly1(z[r], z[r + (1 << d)]);
                else if (INV || d == 2)
                    butterfly(z[r], z[r + (1 << d)], w[e].x, INV ? w[e].y : -w[e].y);
                else {  // forward, the second level: both points are real
                    const double u = z[r].x, v = z[r + 2].x, tr = w[e].x * v, ti = -w[e].y * v;
                    z[r] = make_double2(u + tr, ti);
                    z[r + 2] = make_double2(u - tr, -ti);
                }
            }
}

// LV levels from points h apart; lo the first point's place among the h
template <int LV, bool INV>
__device__ __forceinline__ void more_levels(double2 *z, const double2 *__restrict__ tw, int nx, int lo,
                                            int lh)
{
#pragma unroll
    for (int d = 0; d < LV; ++d) {
        const int st = nx >> lh >> (d + 1);  // tw entries between the points of this level's turn
#pragma unroll
        for (int q = 0; q < (1 << d); ++q) {
            const double2 w = __ldg(tw + (lo + (q << lh)) * st);
#pragma unroll
            for (int r = q; r < (1 << LV); r += 2 << d)
                butterfly(z[r], z[r + (1 << d)], w.x, INV ? w.y : -w.y);
        }
    }
}

// The transform of a row's nx = 2^lm points by T threads: R0 levels first, then LV at a time
// (LV divides lm - R0; R0 >= 1), x the row's shared memory.  load(point, q) gives a point (the
// one q T after the thread's first of a turn); the last pass's go to store(point, value).
template <int LV, int R0, bool INV, typename Load, typename Store>
__device__ __forceinline__ void fft_row(double2 *x, const double2 *__restrict__ tw, int nx, int t, int T,
                                        int lm, Load load, Store store)
{
    constexpr int P = 1 << R0, N = 1 << LV, G = N / P;  // points a group, a thread; groups a thread
    double2 w[4] = {};
    if (R0 >= 2)
        w[2] = __ldg(tw + (nx >> 2));
    if (R0 >= 3) {
        w[1] = __ldg(tw + (nx >> 3));
        w[3] = __ldg(tw + 3 * (nx >> 3));
    }
    // a group: P points that end up next to each other in bit-reversed order, nx / P apart
    const int groups = nx >> R0;
    for (int g0 = t; g0 < groups; g0 += T * G) {
        double2 z[N];
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const int g = g0 + (q >> R0) * T, r = q & (P - 1);
            const int rev = R0 == 3 ? ((r & 1) << 2 | (r & 2) | r >> 2) : R0 == 2 ? ((r & 1) << 1 | r >> 1) : r;
            if (g < groups)
                z[q] = load(g + rev * groups, (q >> R0) + rev * G);
        }
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const int g = g0 + k * T;
            if (g < groups) {
                first_levels<R0, INV>(z + k * P, w);
                const int at = lm > R0 ? (int)(__brev((unsigned)g) >> (32 - (lm - R0))) << R0 : 0;
                const int pl = fft_place(at);
#pragma unroll
                for (int r = 0; r < P; ++r) {
                    if (lm == R0)
                        store(at + r, z[k * P + r]);
                    else
                        x[pl ^ r] = z[k * P + r];
                }
            }
        }
    }
    if (lm == R0)
        return;
    auto pass = [&](int lh, auto put) {
        __syncthreads();
        for (int g = t; g < nx >> LV; g += T) {
            const int lo = g & ((1 << lh) - 1), at = ((g >> lh) << (lh + LV)) + lo, pl = fft_place(at);
            double2 z[N];
#pragma unroll
            for (int r = 0; r < N; ++r)
                z[r] = x[pl ^ fft_place(r << lh)];
            more_levels<LV, INV>(z, tw, nx, lo, lh);
#pragma unroll
            for (int r = 0; r < N; ++r)
                put(at + (r << lh), pl ^ fft_place(r << lh), z[r]);
        }
    };
#pragma unroll 1
    for (int lh = R0; lh < lm - LV; lh += LV)
        pass(lh, [&](int, int place, double2 v) { x[place] = v; });
    pass(lm - LV, [&](int i, int, double2 v) { store(i, v); });
}

__device__ __forceinline__ double block_sum_fft(double v, double *s_red)
{
    for (int off = 16; off; off >>= 1)
        v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0)
        s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)blockDim.x / 32; ++w)
            t += s_red[w];
    __syncthreads();
    return t;
}

// forward: b of row j (from the deposits, then cleared, in mode 0; from rho in p.r
// in mode 1) into p.q, its transform into p.spec; ||b_j||^2 into rpart
template <int LV, int R0>
__global__ void __launch_bounds__(kFftMaxThreads) k_fft_rows(const __grid_constant__ Params2D p, int mode)
{
    constexpr int N = 1 << LV;  // nodes a thread at a time
    extern __shared__ double2 sx[];
    __shared__ double s_red[kFftMaxThreads / 32];
    const int nx = p.nx, ny = p.ny;
    const int T = fft_row_threads(nx, LV), rows = fft_cta_rows(nx, LV);
    const int t = threadIdx.x % T, rl = threadIdx.x / T;
    const int j = 1 + blockIdx.x * rows + rl;
    const bool act = j < ny;
    double2 *x = sx + (size_t)rl * nx;
    const size_t row = (size_t)j * nx;
    double bb = 0.0;
    double b[N] = {};  // of N nodes T apart (all of a species' loads in flight at once)
    if (act)
        for (int i0 = t; i0 < nx; i0 += T * N) {
#pragma unroll
            for (int q = 0; q < N; ++q)
                b[q] = 0.0;
            if (mode == 0) {
                for (int s = 0; s < p.ns; ++s) {
                    unsigned long long *a = p.acc + (size_t)s * p.nn + row + i0;
                    const double unit = p.sp[s].rho_unit;
                    unsigned long long v[N];
#pragma unroll
                    for (int q = 0; q < N; ++q)
                        if (i0 + q * T < nx)
                            v[q] = a[q * T];
#pragma unroll
                    for (int q = 0; q < N; ++q)
                        if (i0 + q * T < nx) {
                            b[q] = fma(unit, (double)(long long)v[q], b[q]);
                            a[q * T] = 0ULL;
                            // the plate rows' deposits are consumed here too
                            if (j == 1)
                                a[q * T - nx] = 0ULL;
                            if (j == ny - 1)
                                a[q * T + nx] = 0ULL;
                        }
                }
            } else {
#pragma unroll
                for (int q = 0; q < N; ++q)
                    if (i0 + q * T < nx)
                        b[q] = p.r[row + i0 + q * T];
            }
#pragma unroll
            for (int q = 0; q < N; ++q)
                if (i0 + q * T < nx) {
                    b[q] = p.k2 * b[q];
                    if (j == 1)
                        b[q] += p.phi_lo;
                    if (j == ny - 1)
                        b[q] += p.phi_hi;
                    p.q[row + i0 + q * T] = b[q];
                    bb = fma(b[q], b[q], bb);
                }
        }
    for (int off = min(T, 32) / 2; off; off >>= 1)
        bb += __shfl_down_sync(0xffffffffu, bb, off, min(T, 32));
    if (T > 32 && (threadIdx.x & 31) == 0)
        s_red[threadIdx.x >> 5] = bb;
    __syncthreads();
    const double *bq = p.q + row;
    double2 *out = p.spec + row;
    const bool one = T * N == nx;  // the row is in registers, a thread's point q T after its first in b[q]
    fft_row<LV, R0, false>(
        x, p.tw, nx, t, T, p.log2nx,
        [&](int i, int q) { return make_double2(one ? b[q] : act ? bq[i] : 0.0, 0.0); },
        [&](int i, double2 v) {
            if (act)
                out[i] = v;
        });
    if (t == 0 && act) {
        if (T > 32)
            for (int w = 1; w < T / 32; ++w)
                bb += s_red[w];
        p.rpart[2 * j + 1] = bb;
    }
}

// inverse: phi of row j from its coefficients
template <int LV, int R0>
__global__ void __launch_bounds__(kFftMaxThreads) k_ifft_rows(const __grid_constant__ Params2D p)
{
    extern __shared__ double2 sx[];
    const int nx = p.nx;
    const int T = fft_row_threads(nx, LV), rows = fft_cta_rows(nx, LV);
    const int t = threadIdx.x % T, rl = threadIdx.x / T;
    const int j = 1 + blockIdx.x * rows + rl;
    const bool act = j < p.ny;
    const double inv = 1.0 / nx;
    const double2 *in = p.spec + (size_t)j * nx;
    double *phi = p.phi + (size_t)j * nx;
    fft_row<LV, R0, true>(
        sx + (size_t)rl * nx, p.tw, nx, t, T, p.log2nx,
        [&](int i, int) { return act ? in[i] : make_double2(0.0, 0.0); },
        [&](int i, double2 v) {
            if (act)
                phi[i] = v.x * inv;
        });
}

// Thomas per mode k: forward u'_j = (b^_j + u'_{j-1}) / m_j, back u_j = u'_j + u_{j+1} / m_j
// (rows 1..ny-1), the multipliers 1/m_j tabulated.  Both are first-order linear
// recurrences, so each is solved in segments of L rows side by side: every segment
// from a zero start (x~), then the value entering each segment by a short sequential
// pass over the segments' ends, then x = x~ + P x_in with P the product of the
// segment's multipliers up to the row (tabulated: seg_f forward, seg_b backward).
// A CTA takes kTriModes modes (consecutive: 64 bytes a row) times kTriSegs segments.  What a
// step of a chain costs is FP64 latency (110 cycles on an idle pipe), if its operands are
// there: a batch of rows is loaded at once, the segments' ends and products are gathered
// before the sequential pass, and between the passes the values stay in shared memory
// where they fit (kShared; ny up to some 3,500), else in the coefficients' place.
constexpr int kTriModes = 4;
constexpr int kTriSegs = 32;
constexpr int kTriBatch = 8;

__host__ __device__ __forceinline__ int tri_seg_len(int ny)
{
    return (ny - 1 + kTriSegs - 1) / kTriSegs;
}

// shared memory of kShared: an odd number of rows a segment, so that the segments that a
// warp's threads work on lie in different banks
size_t tri_smem_bytes(int ny)
{
    return sizeof(double2) * kTriModes * kTriSegs * (size_t)(tri_seg_len(ny) | 1);
}

struct TriEnds {
    double2 end[kTriSegs][kTriModes], in[kTriSegs][kTriModes];  // values leaving (from zero), entering
    double prod[kTriSegs][kTriModes];                           // the product of a segment's multipliers
};

// the value entering each segment, in order (or from the last): a thread per mode
__device__ __forceinline__ void tri_chain(TriEnds &e, int kk, int used, bool back)
{
    double2 c = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int i = 0; i < used; ++i) {
        const int t = back ? used - 1 - i : i;
        e.in[t][kk] = c;
        const double f = e.prod[t][kk];
        const double2 v = e.end[t][kk];
        c = make_double2(fma(f, c.x, v.x), fma(f, c.y, v.y));
    }
}

template <bool kShared>
__global__ void __launch_bounds__(kTriModes * kTriSegs) k_tridiag_modes(const __grid_constant__ Params2D p)
{
    extern __shared__ double2 s_x[];
    __shared__ TriEnds e;
    const int nx = p.nx, ny = p.ny;
    const int kk = threadIdx.x % kTriModes, sg = threadIdx.x / kTriModes;
    const int k = blockIdx.x * kTriModes + kk;
    const int L = tri_seg_len(ny), used = (ny - 1 + L - 1) / L;  // segments with rows
    // this segment's rows [j0, j1) (64 bits: the last segments may start far past ny)
    const int j0 = (int)min((long long)ny, 1 + (long long)sg * L);
    const int j1 = k < nx ? (int)min((long long)ny, (long long)j0 + L) : j0;
    const size_t first = (size_t)j0 * nx + k;
    double2 *__restrict__ spec = p.spec + first;
    const double *__restrict__ invm = p.inv_m + first;
    const double *__restrict__ pf = p.seg_f + first;
    const double *__restrict__ pb = p.seg_b + first;
    double2 *xv = kShared ? s_x + (size_t)sg * (L | 1) * kTriModes + kk : spec;
    const size_t xs = kShared ? kTriModes : nx;  // from row to row
    const int rows = j1 - j0;
    // 1. forward, from zero
    double2 x = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int b = 0; b < rows; b += kTriBatch) {
        double2 v[kTriBatch];
        double m[kTriBatch];
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b + i < rows) {
                v[i] = spec[(size_t)(b + i) * nx];
                m[i] = __ldg(invm + (size_t)(b + i) * nx);
            }
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b + i < rows) {
                x = make_double2((v[i].x + x.x) * m[i], (v[i].y + x.y) * m[i]);
                xv[(b + i) * xs] = x;
            }
    }
    e.end[sg][kk] = x;
    e.prod[sg][kk] = rows > 0 ? __ldg(pf + (size_t)(rows - 1) * nx) : 0.0;
    __syncthreads();
    // 2. the forward value entering each segment
    if (sg == 0)
        tri_chain(e, kk, used, false);
    __syncthreads();
    // 3. the forward values completed, then the backward recurrence from zero, top down
    const double2 cf = e.in[sg][kk];
    double2 u = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int b = rows - 1; b >= 0; b -= kTriBatch) {
        double2 v[kTriBatch];
        double m[kTriBatch], f[kTriBatch];
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b - i >= 0) {
                v[i] = xv[(b - i) * xs];
                m[i] = __ldg(invm + (size_t)(b - i) * nx);
                f[i] = __ldg(pf + (size_t)(b - i) * nx);
            }
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b - i >= 0) {
                u = make_double2(fma(u.x, m[i], fma(f[i], cf.x, v[i].x)),
                                 fma(u.y, m[i], fma(f[i], cf.y, v[i].y)));
                xv[(b - i) * xs] = u;
            }
    }
    __syncthreads();  // every thread has read its value of pass 2
    e.end[sg][kk] = u;
    e.prod[sg][kk] = rows > 0 ? __ldg(pb) : 0.0;
    __syncthreads();
    // 4. the backward value entering each segment from above
    if (sg == 0)
        tri_chain(e, kk, used, true);
    __syncthreads();
    // 5. the backward values completed
    const double2 cb = e.in[sg][kk];
#pragma unroll 1
    for (int b = 0; b < rows; b += kTriBatch) {
        double2 v[kTriBatch];
        double g[kTriBatch];
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b + i < rows) {
                v[i] = xv[(b + i) * xs];
                g[i] = __ldg(pb + (size_t)(b + i) * nx);
            }
#pragma unroll
        for (int i = 0; i < kTriBatch; ++i)
            if (b + i < rows)
                spec[(size_t)(b + i) * nx] =
                    make_double2(fma(g[i], cb.x, v[i].x), fma(g[i], cb.y, v[i].y));
    }
}

// E on every node (mode 0) and the true residual r = b - A phi per row, a row per CTA, two
// nodes a thread; the last CTA adds the rows' sums in a fixed order (contiguous runs of
// rows per thread, then a fixed tree: the same result every run) and keeps the books.
__global__ void __launch_bounds__(kFinishThreads) k_fft_finish(const __grid_constant__ Params2D p, int mode)
{
    __shared__ double s_red[kFinishThreads / 32];
    __shared__ bool s_last;
    const int nx = p.nx, ny = p.ny, j = blockIdx.x;  // rows 0..ny
    const double h = p.half_dx;
    double rr = 0.0;
    const double *__restrict__ f = p.phi + (size_t)j * nx;
    for (int i = 2 * threadIdx.x; i < nx; i += 2 * kFinishThreads) {
        const double2 c = *reinterpret_cast<const double2 *>(f + i);
        const double l = f[i == 0 ? nx - 1 : i - 1], r = f[i + 2 == nx ? 0 : i + 2];
        double2 up = make_double2(0.0, 0.0), dn = up;
        if (j < ny)
            up = *reinterpret_cast<const double2 *>(f + nx + i);
        if (j > 0)
            dn = *reinterpret_cast<const double2 *>(f - nx + i);
        if (mode == 0) {
            double2 ey;
            if (j == 0)
                ey = make_double2(-(up.x - c.x) / p.dx, -(up.y - c.y) / p.dx);
            else if (j == ny)
                ey = make_double2(-(c.x - dn.x) / p.dx, -(c.y - dn.y) / p.dx);
            else
                ey = make_double2(-(up.x - dn.x) * h, -(up.y - dn.y) * h);
            *reinterpret_cast<float4 *>(p.E + (size_t)j * nx + i) =
                make_float4((float)(-(c.y - l) * h), (float)ey.x, (float)(-(r - c.x) * h), (float)ey.y);
        }
        if (j >= 1 && j < ny) {
            const double2 q = *reinterpret_cast<const double2 *>(p.q + (size_t)j * nx + i);
            double a0 = 4.0 * c.x - (c.y + l), a1 = 4.0 * c.y - (r + c.x);
            if (j > 1) {
                a0 -= dn.x;
                a1 -= dn.y;
            }
            if (j < ny - 1) {
                a0 -= up.x;
                a1 -= up.y;
            }
            const double r0 = q.x - a0, r1 = q.y - a1;
            rr = fma(r0, r0, rr);
            rr = fma(r1, r1, rr);
        }
    }
    const double rrs = block_sum_fft(rr, s_red);
    if (threadIdx.x == 0) {
        p.rpart[2 * j] = (j >= 1 && j < ny) ? rrs : 0.0;
        __threadfence();
        const unsigned n = atomicAdd(p.finished, 1u);
        s_last = n == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    const int rows = ny - 1, per = (rows + kFinishThreads - 1) / kFinishThreads;
    double r = 0.0, b = 0.0;
    for (int q = 0; q < per; ++q) {
        const int m = 1 + threadIdx.x * per + q;
        if (m < ny) {
            r += __ldcg(p.rpart + 2 * m);
            b += __ldcg(p.rpart + 2 * m + 1);
        }
    }
    const double R = block_sum_fft(r, s_red);
    const double B = block_sum_fft(b, s_red);
    if (threadIdx.x != 0)
        return;
    *p.finished = 0u;
    State2D *st = p.st;
    st->cg_iters = 0;
    st->cg_res = B > 0.0 ? sqrt(R / B) : 0.0;
    if (B > 0.0 && R > p.rtol2 * B)
        atomicCAS(&st->error, 0, SLPIC_ERR_NOCONVERGE);
}

// the instantiation for a grid
typedef void (*FftKernel)(Params2D, int);
typedef void (*IfftKernel)(Params2D);

FftKernel fft_kernel(const Params2D &p)
{
    if (fft_levels(p.nx, p.ny) == 1)
        return k_fft_rows<1, 1>;
    const int r = p.log2nx % 3;
    return r == 1 ? k_fft_rows<3, 1> : r == 2 ? k_fft_rows<3, 2> : k_fft_rows<3, 3>;
}

IfftKernel ifft_kernel(const Params2D &p)
{
    if (fft_levels(p.nx, p.ny) == 1)
        return k_ifft_rows<1, 1>;
    const int r = p.log2nx % 3;
    return r == 1 ? k_ifft_rows<3, 1> : r == 2 ? k_ifft_rows<3, 2> : k_ifft_rows<3, 3>;
}

// ---- counting sort of the particles by cell ------------------------------------------
// Particles in cell order make the gather of E and the deposit atomics of
// neighbouring threads land on neighbouring nodes.  Three passes over the live
// particles of buffer `src`: a histogram per cell (lanes of a warp in the same cell
// add once, __match_any_sync), an exclusive scan of the histogram into each cell's
// first slot, and a scatter into buffer `dst` (a slot per particle by an atomic on
// its cell's cursor, again once per warp group).  The order within a cell is
// whatever the atomics give; nothing computed depends on it.
constexpr int kScanThreads = 1024, kScanPer = 4, kScanBlock = kScanThreads * kScanPer;

__global__ void __launch_bounds__(kThreads) k_sort_count2d(Params2D p, int s, int src)
{
    const Species2D &sp = p.sp[s];
    const long long n = (long long)p.st->count[s][src];
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * kThreads;
    for (long long base = ((long long)blockIdx.x * kThreads + threadIdx.x) & ~31LL; base < n;
         base += stride) {
        const long long i = base + lane;
        const int c = i < n ? sp.cell[src][i] : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, c);
        if (c >= 0 && lane == __ffs(grp) - 1)
            atomicAdd(&p.hist[c], __popc(grp));
    }
}

// exclusive scan of hist[0..nn) into cursor: per block of kScanBlock entries, then
// the block totals, then their offsets added
__global__ void __launch_bounds__(kScanThreads) k_scan_blocks(Params2D p)
{
    __shared__ int s_w[kScanThreads / 32];
    const long long b0 = (long long)blockIdx.x * kScanBlock + threadIdx.x * kScanPer;
    int v[kScanPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = b0 + k < p.nn ? p.hist[b0 + k] : 0;
        sum += v[k];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += y;
    }
    if (lane == 31)
        s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = s_w[lane];
        int wi = w;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o)
                wi += y;
        }
        s_w[lane] = wi - w;  // exclusive over warps
        if (lane == 31)
            p.bsum[blockIdx.x] = wi;
    }
    __syncthreads();
    int run = s_w[warp] + incl - sum;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (b0 + k < p.nn)
            p.cursor[b0 + k] = run;
        run += v[k];
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_top(Params2D p, int nb)
{
    __shared__ int s_carry;
    __shared__ int s_w[kScanThreads / 32];
    if (threadIdx.x == 0)
        s_carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b0 = 0; b0 < nb; b0 += kScanThreads) {
        const int i = b0 + threadIdx.x;
        const int v = i < nb ? p.bsum[i] : 0;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o)
                incl += y;
        }
        if (lane == 31)
            s_w[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int w = s_w[lane];
            int wi = w;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o)
                    wi += y;
            }
            s_w[lane] = wi - w;
        }
        __syncthreads();
        const int carry = s_carry;
        if (i < nb)
            p.bsum[i] = carry + s_w[warp] + incl - v;
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1)
            s_carry = carry + s_w[warp] + incl;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(Params2D p)
{
    const long long i0 = (long long)blockIdx.x * kScanBlock;
    const int add = p.bsum[blockIdx.x];
    for (int k = threadIdx.x; k < kScanBlock; k += kScanThreads)
        if (i0 + k < p.nn)
            p.cursor[i0 + k] += add;
}

// the sorted buffer's slots: the end of the last cell's run; no holes
__global__ void k_sort_count_set(Params2D p, int s, int b)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        p.st->count[s][b] = (unsigned long long)p.cursor[p.nn - 1];
        p.st->holes[s][b] = 0ULL;
    }
}

__global__ void __launch_bounds__(kThreads) k_sort_scatter2d(Params2D p, int s, int src, int dst)
{
    const Species2D &sp = p.sp[s];
    const long long n = (long long)p.st->count[s][src];
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * kThreads;
    for (long long base = ((long long)blockIdx.x * kThreads + threadIdx.x) & ~31LL; base < n;
         base += stride) {
        const long long i = base + lane;
        const int c = i < n ? sp.cell[src][i] : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, c);
        const int leader = __ffs(grp) - 1;
        int slot = 0;
        if (c >= 0 && lane == leader)
            slot = atomicAdd(&p.cursor[c], __popc(grp));
        slot = __shfl_sync(0xffffffffu, slot, leader);
        if (c >= 0) {
            const int o = slot + __popc(grp & ((1u << lane) - 1u));
            sp.cell[dst][o] = c;
            sp.pv[dst][o] = sp.pv[src][i];
            sp.vz[dst][o] = sp.vz[src][i];
        }
    }
}

// ---- read-back (slpic2d_fields): rho from the deposits, which are cleared, with the
// operations of the solves; E's components apart
__global__ void __launch_bounds__(kThreads) k_rho2d(Params2D p, double *__restrict__ out)
{
    for (long long t = (long long)blockIdx.x * kThreads + threadIdx.x; t < p.nn;
         t += (long long)gridDim.x * kThreads) {
        double v = 0.0;
        for (int s = 0; s < p.ns; ++s) {
            unsigned long long *a = p.acc + (size_t)s * p.nn + t;
            v = fma(p.sp[s].rho_unit, (double)(long long)*a, v);
            *a = 0ULL;
        }
        out[t] = v;
    }
}

__global__ void __launch_bounds__(kThreads) k_split2d(Params2D p, float *__restrict__ ex, float *__restrict__ ey)
{
    for (long long t = (long long)blockIdx.x * kThreads + threadIdx.x; t < p.nn;
         t += (long long)gridDim.x * kThreads) {
        const float2 e = p.E[t];
        ex[t] = e.x;
        ey[t] = e.y;
    }
}

// ---- initial guess of the CG (slpic2d_set_warm_start) ------------------------------
// rho of rows 0..ny-1 as FP32 from the deposits (left in place for the CG kernel);
// row 0, a plate, is zero.  The layout is the nodal one, so the array is the
// U-Net's (H, W) = (ny, nx) input.
__global__ void __launch_bounds__(kThreads) k_rho32(Params2D p, float *__restrict__ out)
{
    const long long n = (long long)p.ny * p.nx;
    for (long long t = (long long)blockIdx.x * kThreads + threadIdx.x; t < n;
         t += (long long)gridDim.x * kThreads) {
        double rho = 0.0;
        if (t >= p.nx)
            for (int s = 0; s < p.ns; ++s)
                rho = fma(p.sp[s].rho_unit, (double)(long long)p.acc[(size_t)s * p.nn + t], rho);
        out[t] = (float)rho;
    }
}

// x = a - b (the change of the charge image since the previous step)
__global__ void __launch_bounds__(kThreads) k_sub32(const float *__restrict__ a,
                                                  const float *__restrict__ b,
                                                  float *__restrict__ x, long long n)
{
    for (long long t = (long long)blockIdx.x * kThreads + threadIdx.x; t < n;
         t += (long long)gridDim.x * kThreads)
        x[t] = a[t] - b[t];
}

// phi += y on the interior rows (the previous potential plus the predicted change)
__global__ void __launch_bounds__(kThreads) k_guess_add(Params2D p, const float *__restrict__ y)
{
    const long long first = p.nx, last = (long long)p.ny * p.nx;
    for (long long t = first + (long long)blockIdx.x * kThreads + threadIdx.x; t < last;
         t += (long long)gridDim.x * kThreads)
        p.phi[t] += (double)y[t];
}

// phi on the interior rows = the straight line between the plate potentials plus
// y (the network's guess for the zero-plate problem), or the line alone when y is
// null (the zero guess).
__global__ void __launch_bounds__(kThreads) k_guess(Params2D p, const float *__restrict__ y)
{
    const long long first = p.nx, last = (long long)p.ny * p.nx;
    for (long long t = first + (long long)blockIdx.x * kThreads + threadIdx.x; t < last;
         t += (long long)gridDim.x * kThreads) {
        const int j = (int)(t / p.nx);
        double v = p.phi_lo + (p.phi_hi - p.phi_lo) * ((double)j / p.ny);
        if (y)
            v += (double)y[t];
        p.phi[t] = v;
    }
}

}  // namespace slpic2d

// =================================================================================
// C ABI
// =================================================================================
using namespace slpic2d;

struct slpic2d_sim {
    slpic2d_config cfg{};
    cudaStream_t stream = nullptr, own_stream = nullptr;
    Params2D p{};
    int ctas = 1;     // particle-kernel CTAs per species
    int tile_ctas = 0;  // k_particles2d_tiles CTAs per species (0: not resident)
    int hard_ctas = 1;  // k_hard2d: all resident
    size_t tri_smem = 0;  // k_tridiag_modes' shared memory (0: the values do not fit)
    int small_ctas = 1; // k_inject2d: 2 CTAs of 256 threads per SM
    bool prepared = false;
    bool timing = false;               // record events around the kernels of each step
    std::vector<cudaEvent_t> events;   // 4 per recorded step
    long long t_steps = 0;             // steps recorded since the last read
    State2D *d_state = nullptr;
    int warm_mode = SLPIC2D_WARM_PREV;  // initial guess of each step's CG
    slpic_unet_t *net = nullptr;        // SLPIC2D_WARM_UNET: borrowed network
    float *rho32 = nullptr, *guess32 = nullptr;  // its input and output (ny * nx)
    float *rho32_prev = nullptr, *drho32 = nullptr;  // SLPIC2D_WARM_UNET_DELTA
    bool have_prev_rho = false;
    std::vector<void *> allocs;
    std::string err;
};

#define CK2(h, call)                                                                       \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            (h)->err = std::string(#call) + ": " + cudaGetErrorString(e_);                 \
            return SLPIC_ERR_CUDA;                                                         \
        }                                                                                  \
    } while (0)

static int fail2(slpic2d_t *h, int code, const std::string &msg)
{
    h->err = msg;
    return code;
}

static int device_status(slpic2d_t *h)
{
    CK2(h, cudaStreamSynchronize(h->stream));
    int e = 0;
    CK2(h, cudaMemcpy(&e, &h->d_state->error, sizeof(int), cudaMemcpyDeviceToHost));
    if (e) {
        const char *m = e == SLPIC_ERR_CAPACITY ? "particle store full: injection truncated"
                        : e == SLPIC_ERR_NOCONVERGE ? "CG did not reach cg_rtol within cg_maxit"
                        : e == SLPIC_ERR_TIMEOUT ? "grid barrier of the CG kernel timed out"
                                                 : "device error";
        return fail2(h, e, m);
    }
    return SLPIC_OK;
}

static int launch_cg(slpic2d_t *h, int mode)
{
    Params2D p = h->p;
    void *args[] = {&p, &mode};
    CK2(h, cudaMemsetAsync(p.part, 0xFF, sizeof(double) * 3 * p.cg_v, h->stream));  // kCgEmpty
    CK2(h, cudaLaunchCooperativeKernel((const void *)cg_kernel(p), dim3(cg_grid(p)), dim3(kCgThreads),
                                       args, 0, h->stream));
    return SLPIC_OK;
}

// The initial guess of the step's CG, on the handle's stream (SLPIC2D_WARM_PREV:
// phi as the previous step left it).
static int warm_start(slpic2d_t *h)
{
    const unsigned grid = (unsigned)std::min<long long>(
        ((long long)h->p.ny * h->p.nx + kThreads - 1) / kThreads, 152LL * 8);
    if (h->warm_mode == SLPIC2D_WARM_ZERO) {
        k_guess<<<grid, kThreads, 0, h->stream>>>(h->p, nullptr);
    } else if (h->warm_mode == SLPIC2D_WARM_UNET) {
        k_rho32<<<grid, kThreads, 0, h->stream>>>(h->p, h->rho32);
        CK2(h, cudaGetLastError());
        const int rc = slpic_unet_forward_on(h->net, 1, h->rho32, h->guess32, h->stream);
        if (rc)
            return fail2(h, rc, std::string("U-Net forward: ") + slpic_unet_last_error(h->net));
        k_guess<<<grid, kThreads, 0, h->stream>>>(h->p, h->guess32);
    } else if (h->warm_mode == SLPIC2D_WARM_UNET_DELTA) {
        // phi (still the previous step's) + net(rho - rho_prev); the first step
        // after a reset has no rho_prev and starts from the previous phi alone
        k_rho32<<<grid, kThreads, 0, h->stream>>>(h->p, h->rho32);
        CK2(h, cudaGetLastError());
        if (h->have_prev_rho) {
            const long long n = (long long)h->p.ny * h->p.nx;
            k_sub32<<<grid, kThreads, 0, h->stream>>>(h->rho32, h->rho32_prev, h->drho32, n);
            const int rc = slpic_unet_forward_on(h->net, 1, h->drho32, h->guess32, h->stream);
            if (rc)
                return fail2(h, rc, std::string("U-Net forward: ") + slpic_unet_last_error(h->net));
            k_guess_add<<<grid, kThreads, 0, h->stream>>>(h->p, h->guess32);
        }
        std::swap(h->rho32, h->rho32_prev);
        h->have_prev_rho = true;
    }
    CK2(h, cudaGetLastError());
    return SLPIC_OK;
}

extern "C" int slpic2d_set_warm_start(slpic2d_t *h, int32_t mode, slpic_unet_t *net)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    if (mode != SLPIC2D_WARM_PREV && mode != SLPIC2D_WARM_ZERO && mode != SLPIC2D_WARM_UNET &&
        mode != SLPIC2D_WARM_UNET_DELTA)
        return fail2(h, SLPIC_ERR_INVALID, "unknown warm-start mode");
    const bool uses_net = mode == SLPIC2D_WARM_UNET || mode == SLPIC2D_WARM_UNET_DELTA;
    if (uses_net) {
        if (!net)
            return fail2(h, SLPIC_ERR_INVALID, "this warm-start mode needs a network");
        int H, W, nb;
        slpic_unet_shape(net, &H, &W, &nb);
        if (H != h->p.ny || W != h->p.nx)
            return fail2(h, SLPIC_ERR_INVALID, "the network's grid must be (ny, nx)");
        if (!h->rho32) {
            const size_t n = (size_t)h->p.ny * h->p.nx;
            CK2(h, cudaMalloc(&h->rho32, sizeof(float) * n));
            h->allocs.push_back(h->rho32);
            CK2(h, cudaMalloc(&h->guess32, sizeof(float) * n));
            h->allocs.push_back(h->guess32);
            CK2(h, cudaMalloc(&h->rho32_prev, sizeof(float) * n));
            h->allocs.push_back(h->rho32_prev);
            CK2(h, cudaMalloc(&h->drho32, sizeof(float) * n));
            h->allocs.push_back(h->drho32);
        }
    }
    h->warm_mode = mode;
    h->net = uses_net ? net : nullptr;
    h->have_prev_rho = false;
    return SLPIC_OK;
}

// Sort every species' particles of buffer `src` by cell into buffer `dst` (holes
// dropped, the count set to the live particles), then swap the two buffers' roles,
// so that buffer index `src` names the sorted particles.
static int sort_particles(slpic2d_t *h, int src)
{
    Params2D &p = h->p;
    const int dst = src ^ 1;
    const unsigned nblk = (unsigned)((p.nn + kScanBlock - 1) / kScanBlock);
    for (int s = 0; s < p.ns; ++s) {
        CK2(h, cudaMemsetAsync(p.hist, 0, sizeof(int) * p.nn, h->stream));
        k_sort_count2d<<<h->ctas, kThreads, 0, h->stream>>>(p, s, src);
        k_scan_blocks<<<nblk, kScanThreads, 0, h->stream>>>(p);
        k_scan_top<<<1, kScanThreads, 0, h->stream>>>(p, (int)nblk);
        k_scan_add<<<nblk, kScanThreads, 0, h->stream>>>(p);
        k_sort_scatter2d<<<h->ctas, kThreads, 0, h->stream>>>(p, s, src, dst);
        k_sort_count_set<<<1, 32, 0, h->stream>>>(p, s, src);
        CK2(h, cudaGetLastError());
        std::swap(p.sp[s].cell[src], p.sp[s].cell[dst]);
        std::swap(p.sp[s].pv[src], p.sp[s].pv[dst]);
        std::swap(p.sp[s].vz[src], p.sp[s].vz[dst]);
    }
    return SLPIC_OK;
}

// The field solve of the configured solver (mode as for k_cg2d).
static int launch_solve(slpic2d_t *h, int mode)
{
    if (h->p.solver != SLPIC2D_SOLVER_FFT)
        return launch_cg(h, mode);
    const Params2D &p = h->p;
    const int lv = fft_levels(p.nx, p.ny), rows = fft_cta_rows(p.nx, lv), threads = rows * fft_row_threads(p.nx, lv);
    const int ctas = (p.ny - 1 + rows - 1) / rows, tri = (p.nx + kTriModes - 1) / kTriModes;
    const size_t smem = (size_t)16 * rows * p.nx;
    fft_kernel(p)<<<ctas, threads, smem, h->stream>>>(p, mode);
    if (h->tri_smem)
        k_tridiag_modes<true><<<tri, kTriModes * kTriSegs, h->tri_smem, h->stream>>>(p);
    else
        k_tridiag_modes<false><<<tri, kTriModes * kTriSegs, 0, h->stream>>>(p);
    ifft_kernel(p)<<<ctas, threads, smem, h->stream>>>(p);
    k_fft_finish<<<p.ny + 1, kFinishThreads, 0, h->stream>>>(p, mode);
    CK2(h, cudaGetLastError());
    return SLPIC_OK;
}

extern "C" int slpic2d_create(const slpic2d_config *c, slpic2d_t **out)
{
    if (!c || !out) {
        slpic::set_create_error("null argument");
        return SLPIC_ERR_INVALID;
    }
    std::string why;
    if (c->nx < 2 || c->ny < 2 || !(c->dx > 0) || !(c->dt > 0) || !(c->eps0 > 0))
        why = "need nx >= 2, ny >= 2, dx > 0, dt > 0, eps0 > 0";
    else if ((long long)c->nx * (c->ny + 1) > (1LL << 30))
        why = "grid too large";
    else if (c->n_species < 1 || c->n_species > SLPIC_MAX_SPECIES)
        why = "n_species out of range";
    else if (!(c->cg_rtol > 0 && c->cg_rtol < 1) || c->cg_maxit <= 0)
        why = "need 0 < cg_rtol < 1 and cg_maxit > 0";
    else if (c->solver != SLPIC2D_SOLVER_CG && c->solver != SLPIC2D_SOLVER_FFT)
        why = "unknown solver";
    else if (c->solver == SLPIC2D_SOLVER_FFT && (c->nx & (c->nx - 1) || c->nx > 8192))
        why = "the FFT solver needs nx a power of two, at most 8192";
    else if (c->src_mode < SLPIC_SRC_NONE || c->src_mode > SLPIC_SRC_RATE ||
             (c->src_mode == SLPIC_SRC_LOSS_MATCHED &&
              (c->src_ref_species < 0 || c->src_ref_species >= c->n_species)))
        why = "bad source mode or reference species";
    else if (c->src_mode != SLPIC_SRC_NONE &&
             !(c->src_lo_cells >= 0 && c->src_len_cells >= 0 &&
               c->src_lo_cells + c->src_len_cells <= c->ny))
        why = "source band outside the grid";
    for (int s = 0; why.empty() && s < c->n_species; ++s) {
        const slpic_species &sp = c->species[s];
        if (!(sp.m > 0) || !(sp.w > 0) || sp.capacity <= 0 || sp.capacity > (1LL << 31) - 1 ||
            !std::isfinite(sp.q) || sp.beta_kind < 0 || sp.beta_kind > 2 || !(sp.T_src >= 0))
            why = "species " + std::to_string(s) + ": bad parameters";
        else if (sp.beta_kind != SLPIC_BETA_ONE && !(sp.v0 > 0))
            why = "species " + std::to_string(s) + ": v0 must be > 0";
        else if (sp.beta_kind != SLPIC_BETA_ONE && c->dt * sp.v0 > c->dx) {
            slpic::set_create_error("species " + std::to_string(s) + ": dt * v0 > dx");
            return SLPIC_ERR_CFL;
        } else if (sp.beta_kind == SLPIC_BETA_ONE && c->max_speed > 0 &&
                   c->dt * c->max_speed > c->dx) {
            slpic::set_create_error("species " + std::to_string(s) + ": dt * max_speed > dx");
            return SLPIC_ERR_CFL;
        }
    }
    if (!why.empty()) {
        slpic::set_create_error(why);
        return SLPIC_ERR_INVALID;
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        slpic::set_create_error("no CUDA device");
        return SLPIC_ERR_CUDA;
    }
    slpic2d_t *h = new slpic2d_t();
    h->cfg = *c;
    auto bail = [&](int code, const std::string &m) {
        slpic::set_create_error(m);
        slpic2d_destroy(h);
        return code;
    };
    auto alloc = [&](void **ptr, size_t bytes) -> bool {
        if (cudaMalloc(ptr, bytes) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        h->allocs.push_back(*ptr);
        return true;
    };
    if (cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking) != cudaSuccess)
        return bail(SLPIC_ERR_CUDA, "stream creation failed");
    h->stream = h->own_stream;
    Params2D &p = h->p;
    p.nx = c->nx;
    make_div_nx(p.nx, p.nx_m, p.nx_s);
    p.ny = c->ny;
    p.nn = c->nx * (c->ny + 1);
    p.ns = c->n_species;
    p.dt = (float)c->dt;
    p.dt_dx = (float)(c->dt / c->dx);
    p.dx = c->dx;
    p.dt64 = c->dt;
    p.k2 = c->dx * c->dx / c->eps0;
    p.half_dx = 0.5 / c->dx;
    p.phi_lo = c->phi_lo;
    p.phi_hi = c->phi_hi;
    p.rtol2 = c->cg_rtol * c->cg_rtol;
    p.cg_maxit = c->cg_maxit;
    p.src_mode = c->src_mode;
    p.src_ref = c->src_ref_species;
    p.src_lo = (float)c->src_lo_cells;
    p.src_len = (float)c->src_len_cells;
    p.src_rate = c->src_rate;
    p.seed = c->seed;
    const size_t nn = (size_t)p.nn;
    bool ok = alloc((void **)&h->d_state, sizeof(State2D)) &&
              alloc((void **)&p.acc, sizeof(unsigned long long) * nn * p.ns) &&
              alloc((void **)&p.E, sizeof(float2) * nn) && alloc((void **)&p.phi, sizeof(double) * nn) &&
              alloc((void **)&p.r, sizeof(double) * nn) && alloc((void **)&p.q, sizeof(double) * nn) &&
              alloc((void **)&p.fr, sizeof(float) * nn) && alloc((void **)&p.fpA, sizeof(float) * nn) &&
              alloc((void **)&p.fpB, sizeof(float) * nn) && alloc((void **)&p.fq, sizeof(float) * nn) &&
              alloc((void **)&p.fd, sizeof(float) * nn);
    for (int s = 0; ok && s < p.ns; ++s) {
        const slpic_species &sp = c->species[s];
        Species2D &d = p.sp[s];
        for (int b = 0; ok && b < 2; ++b)
            ok = alloc((void **)&d.cell[b], sizeof(int32_t) * sp.capacity) &&
                 alloc((void **)&d.pv[b], sizeof(float4) * sp.capacity) &&
                 alloc((void **)&d.vz[b], sizeof(float) * sp.capacity);
        // the slots of a step's walked pushes (all of them, at most)
        if (ok)
            ok = alloc((void **)&d.hard, sizeof(int32_t) * sp.capacity);
        d.capacity = sp.capacity;
        d.qm = (float)(sp.q / sp.m);
        d.v0 = (float)sp.v0;
        d.vth_src = (float)std::sqrt(sp.T_src / sp.m);
        d.kind = sp.beta_kind;
        d.w = sp.w;
        d.inv_w = 1.0 / sp.w;
        d.rho_unit = sp.q * sp.w / (c->dx * c->dx) * std::ldexp(1.0, -40);
    }
    if (!ok)
        return bail(SLPIC_ERR_OOM, "device allocation failed");
    p.st = h->d_state;
    int dev = 0, sms = 1, occ = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    p.cg_v = std::min(2 * sms, kCgMaxVirtual);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, cg_kernel(p), kCgThreads, 0) != cudaSuccess ||
        occ < 1)
        return bail(SLPIC_ERR_CUDA, "CG kernel occupancy query failed");
    h->ctas = sms * 4;
    h->small_ctas = sms * 2;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hard2d, 256, 0) != cudaSuccess || occ < 1)
        return bail(SLPIC_ERR_CUDA, "kernel occupancy query failed");
    h->hard_ctas = sms * occ;
    {
        // the tile kernel: every CTA of both species resident at once
        int occ_t = 0;
        if (cudaFuncSetAttribute(tile_kernel(p), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)tile2d_smem_bytes()) == cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_t, tile_kernel(p), kT2d,
                                                          tile2d_smem_bytes()) == cudaSuccess &&
            occ_t > 0)
            h->tile_ctas = std::max(1, sms * std::min(occ_t, kTileCtas2d) / p.ns);
        cudaGetLastError();
    }
    if (!alloc((void **)&p.part, sizeof(double) * 3 * p.cg_v))
        return bail(SLPIC_ERR_OOM, "device allocation failed");
    if (!alloc((void **)&p.hist, sizeof(int) * nn) || !alloc((void **)&p.cursor, sizeof(int) * nn) ||
        !alloc((void **)&p.bsum, sizeof(int) * ((nn + kScanBlock - 1) / kScanBlock + 1)))
        return bail(SLPIC_ERR_OOM, "device allocation failed");
    p.solver = c->solver;
    if (p.solver == SLPIC2D_SOLVER_FFT) {
        // twiddles and the Thomas multipliers of every (row, mode), in FP64 on the host
        p.log2nx = 0;
        while ((1 << p.log2nx) < p.nx)
            ++p.log2nx;
        if (!alloc((void **)&p.tw, sizeof(double2) * (p.nx / 2)) ||
            !alloc((void **)&p.spec, sizeof(double2) * nn) ||
            !alloc((void **)&p.inv_m, sizeof(double) * nn) ||
            !alloc((void **)&p.seg_f, sizeof(double) * nn) ||
            !alloc((void **)&p.seg_b, sizeof(double) * nn) ||
            !alloc((void **)&p.rpart, sizeof(double) * 2 * (p.ny + 1)) ||
            !alloc((void **)&p.finished, sizeof(unsigned)))
            return bail(SLPIC_ERR_OOM, "device allocation failed");
        const double two_pi = 6.283185307179586;
        std::vector<double2> tw((size_t)p.nx / 2);
        for (int m = 0; m < p.nx / 2; ++m)
            tw[m] = make_double2(std::cos(two_pi * m / p.nx), std::sin(two_pi * m / p.nx));
        // the multipliers and their products within each segment of rows (k_tridiag_modes)
        std::vector<double> tables(3 * nn, 0.0);
        double *inv_m = tables.data(), *seg_f = inv_m + nn, *seg_b = seg_f + nn;
        const int L = tri_seg_len(p.ny);
        for (int k = 0; k < p.nx; ++k) {
            const auto at = [&](int j) { return (size_t)j * p.nx + k; };
            const double a = 4.0 - 2.0 * std::cos(two_pi * k / p.nx);
            double prev = 0.0;  // 1/m_{j-1}
            for (int j = 1; j < p.ny; ++j) {
                prev = 1.0 / (a - prev);
                inv_m[at(j)] = prev;
            }
            for (int j0 = 1; j0 < p.ny; j0 += L) {
                const int j1 = std::min(p.ny, j0 + L);
                double f = 1.0, g = 1.0;
                for (int j = j0; j < j1; ++j) {
                    f *= inv_m[at(j)];
                    seg_f[at(j)] = f;
                }
                for (int j = j1 - 1; j >= j0; --j) {
                    g *= inv_m[at(j)];
                    seg_b[at(j)] = g;
                }
            }
        }
        cudaError_t e2 = cudaMemcpy(p.tw, tw.data(), sizeof(double2) * tw.size(), cudaMemcpyHostToDevice);
        if (e2 == cudaSuccess)
            e2 = cudaMemcpy(p.inv_m, inv_m, sizeof(double) * nn, cudaMemcpyHostToDevice);
        if (e2 == cudaSuccess)
            e2 = cudaMemcpy(p.seg_f, seg_f, sizeof(double) * nn, cudaMemcpyHostToDevice);
        if (e2 == cudaSuccess)
            e2 = cudaMemcpy(p.seg_b, seg_b, sizeof(double) * nn, cudaMemcpyHostToDevice);
        if (e2 == cudaSuccess)
            e2 = cudaMemset(p.finished, 0, sizeof(unsigned));
        const size_t tri = tri_smem_bytes(p.ny);
        if (e2 == cudaSuccess && allow_dynamic_smem(k_tridiag_modes<true>, tri) == cudaSuccess)
            h->tri_smem = tri;
        cudaGetLastError();
        const size_t smem = (size_t)16 * p.nx * fft_cta_rows(p.nx, fft_levels(p.nx, p.ny));
        if (e2 == cudaSuccess)
            e2 = allow_dynamic_smem(fft_kernel(p), smem);
        if (e2 == cudaSuccess)
            e2 = allow_dynamic_smem(ifft_kernel(p), smem);
        if (e2 != cudaSuccess)
            return bail(SLPIC_ERR_CUDA, cudaGetErrorString(e2));
    }
    cudaError_t e = cudaMemset(h->d_state, 0, sizeof(State2D));
    if (e == cudaSuccess)
        e = cudaMemset(p.acc, 0, sizeof(unsigned long long) * nn * p.ns);
    if (e == cudaSuccess)
        e = cudaMemset(p.E, 0, sizeof(float2) * nn);
    if (e == cudaSuccess)
        e = cudaMemset(p.phi, 0, sizeof(double) * nn);
    if (e != cudaSuccess)
        return bail(SLPIC_ERR_CUDA, cudaGetErrorString(e));
    // plate rows of phi
    std::vector<double> row((size_t)p.nx, c->phi_lo);
    cudaMemcpy(p.phi, row.data(), sizeof(double) * p.nx, cudaMemcpyHostToDevice);
    std::fill(row.begin(), row.end(), c->phi_hi);
    cudaMemcpy(p.phi + (size_t)p.ny * p.nx, row.data(), sizeof(double) * p.nx,
               cudaMemcpyHostToDevice);
    if (cudaDeviceSynchronize() != cudaSuccess)
        return bail(SLPIC_ERR_CUDA, "initialisation failed");
    *out = h;
    return SLPIC_OK;
}

extern "C" int slpic2d_destroy(slpic2d_t *h)
{
    if (!h)
        return SLPIC_OK;
    if (h->own_stream)
        cudaStreamSynchronize(h->own_stream);
    if (h->stream)
        cudaStreamSynchronize(h->stream);
    for (cudaEvent_t e : h->events)
        cudaEventDestroy(e);
    for (void *a : h->allocs)
        cudaFree(a);
    if (h->own_stream)
        cudaStreamDestroy(h->own_stream);
    delete h;
    return SLPIC_OK;
}

extern "C" const char *slpic2d_last_error(const slpic2d_t *h) { return h ? h->err.c_str() : ""; }

extern "C" int slpic2d_set_stream(slpic2d_t *h, void *stream)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    h->stream = (cudaStream_t)stream;
    return SLPIC_OK;
}

static int read_state(slpic2d_t *h, State2D &st)
{
    CK2(h, cudaStreamSynchronize(h->stream));
    CK2(h, cudaMemcpy(&st, h->d_state, sizeof(State2D), cudaMemcpyDeviceToHost));
    return SLPIC_OK;
}

extern "C" int slpic2d_load_particles(slpic2d_t *h, int s, int64_t n, const int32_t *cell,
                                      const float *offset, const float *v)
{
    if (!h || s < 0 || s >= h->p.ns || n < 0 || (n > 0 && (!cell || !offset || !v)))
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    if (n == 0)
        return SLPIC_OK;
    const int nx = h->p.nx, ny = h->p.ny;
    for (int64_t i = 0; i < n; ++i) {
        const float ox = offset[2 * i], oy = offset[2 * i + 1];
        if (cell[i] < 0 || cell[i] >= nx * ny || !(ox >= 0.0f && ox < 1.0f) ||
            !(oy >= 0.0f && oy < 1.0f) || !std::isfinite(v[3 * i]) ||
            !std::isfinite(v[3 * i + 1]) || !std::isfinite(v[3 * i + 2]))
            return fail2(h, SLPIC_ERR_INVALID,
                         "particle " + std::to_string(i) + ": cell or offset out of range");
    }
    State2D st;
    int rc = read_state(h, st);
    if (rc)
        return rc;
    const int P = (int)(st.step & 1);
    const long long have = (long long)st.count[s][P];
    if (have + n > h->p.sp[s].capacity)
        return fail2(h, SLPIC_ERR_CAPACITY, "load exceeds the species capacity");
    std::vector<float4> pv((size_t)n);
    std::vector<float> vz((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        pv[i] = make_float4(offset[2 * i], offset[2 * i + 1], v[3 * i], v[3 * i + 1]);
        vz[i] = v[3 * i + 2];
    }
    const Species2D &d = h->p.sp[s];
    CK2(h, cudaMemcpy(d.cell[P] + have, cell, sizeof(int32_t) * n, cudaMemcpyHostToDevice));
    CK2(h, cudaMemcpy(d.pv[P] + have, pv.data(), sizeof(float4) * n, cudaMemcpyHostToDevice));
    CK2(h, cudaMemcpy(d.vz[P] + have, vz.data(), sizeof(float) * n, cudaMemcpyHostToDevice));
    const unsigned long long cnt = (unsigned long long)(have + n);
    CK2(h, cudaMemcpy(&h->d_state->count[s][P], &cnt, sizeof(cnt), cudaMemcpyHostToDevice));
    h->prepared = false;
    return SLPIC_OK;
}

extern "C" int slpic2d_prepare(slpic2d_t *h)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    Params2D &p = h->p;
    State2D st;
    int rc = read_state(h, st);
    if (rc)
        return rc;
    if ((rc = sort_particles(h, (int)(st.step & 1))))  // the load in cell order
        return rc;
    CK2(h, cudaMemsetAsync(p.acc, 0, sizeof(unsigned long long) * p.nn * p.ns, h->stream));
    k_deposit2d<<<dim3(h->ctas, p.ns), kThreads, 0, h->stream>>>(p);
    CK2(h, cudaGetLastError());
    rc = launch_solve(h, 0);
    if (rc)
        return rc;
    h->prepared = true;
    h->have_prev_rho = false;
    return device_status(h);
}

extern "C" int slpic2d_step(slpic2d_t *h, int64_t nsteps)
{
    if (!h || nsteps < 0)
        return h ? fail2(h, SLPIC_ERR_INVALID, "nsteps < 0") : SLPIC_ERR_INVALID;
    if (!h->prepared)
        return fail2(h, SLPIC_ERR_INVALID, "slpic2d_prepare must follow a load");
    State2D st;
    int rc = read_state(h, st);
    if (rc)
        return rc;
    if (st.error)
        return device_status(h);
    long long step = st.step;
    Params2D &p = h->p;
    for (int64_t k = 0; k < nsteps; ++k, ++step) {
        // every kCompact2d-th step the particles are sorted by cell again; with the tile
        // kernel that step is in place too (the sort drops the holes), else the global
        // kernel packs the survivors first
        const bool sort = (step % kCompact2d) == kCompact2d - 1;
        const bool compact = sort && !h->tile_ctas;
        cudaEvent_t *ev = nullptr;
        if (h->timing && h->t_steps < kMaxTimedSteps2d) {
            while ((long long)h->events.size() < 4 * (h->t_steps + 1)) {
                cudaEvent_t e;
                CK2(h, cudaEventCreate(&e));
                h->events.push_back(e);
            }
            ev = &h->events[4 * h->t_steps++];
        }
        if (ev)
            CK2(h, cudaEventRecord(ev[0], h->stream));
        if (compact)
            k_particles2d<true><<<dim3(h->ctas, p.ns), kThreads, 0, h->stream>>>(p);
        else if (h->tile_ctas) {
            tile_kernel(p)<<<dim3(h->tile_ctas, p.ns), kT2d, tile2d_smem_bytes(), h->stream>>>(p);
            k_hard2d<<<h->hard_ctas, 256, 0, h->stream>>>(p);
        } else {
            k_particles2d<false><<<dim3(h->ctas, p.ns), kThreads, 0, h->stream>>>(p);
        }
        if (ev)
            CK2(h, cudaEventRecord(ev[1], h->stream));
        k_inject2d<<<h->small_ctas, 256, 0, h->stream>>>(p, compact ? 1 : 0);
        k_book2d<<<1, 32, 0, h->stream>>>(p, compact ? 1 : 0);
        CK2(h, cudaGetLastError());
        // particles by cell (sources appended; holes dropped)
        if (sort && (rc = sort_particles(h, (int)((step + 1) & 1))))
            return rc;
        if (ev)
            CK2(h, cudaEventRecord(ev[2], h->stream));
        if (h->p.solver == SLPIC2D_SOLVER_CG && (rc = warm_start(h)))
            return rc;
        rc = launch_solve(h, 0);
        if (rc)
            return rc;
        if (ev)
            CK2(h, cudaEventRecord(ev[3], h->stream));
    }
    return SLPIC_OK;
}

extern "C" int slpic2d_enable_kernel_timing(slpic2d_t *h, int on)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    h->timing = on != 0;
    h->t_steps = 0;
    return SLPIC_OK;
}

extern "C" int slpic2d_kernel_times(slpic2d_t *h, double *particle_ms, double *inject_ms,
                                    double *field_ms, int64_t *steps)
{
    if (!h || !particle_ms || !inject_ms || !field_ms || !steps)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    CK2(h, cudaStreamSynchronize(h->stream));
    double a = 0.0, b = 0.0, c = 0.0;
    for (long long t = 0; t < h->t_steps; ++t) {
        float x = 0.f, y = 0.f, z = 0.f;
        CK2(h, cudaEventElapsedTime(&x, h->events[4 * t], h->events[4 * t + 1]));
        CK2(h, cudaEventElapsedTime(&y, h->events[4 * t + 1], h->events[4 * t + 2]));
        CK2(h, cudaEventElapsedTime(&z, h->events[4 * t + 2], h->events[4 * t + 3]));
        a += x;
        b += y;
        c += z;
    }
    *steps = h->t_steps;
    const double n = h->t_steps ? (double)h->t_steps : 1.0;
    *particle_ms = a / n;
    *inject_ms = b / n;
    *field_ms = c / n;
    h->t_steps = 0;
    return SLPIC_OK;
}

extern "C" int slpic2d_synchronize(slpic2d_t *h)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    return device_status(h);
}

// Every page of a host buffer that a copy will fill, written once (with what it holds) by the
// CPU: a fresh buffer's pages otherwise come into being one by one under the copy, which
// took 20 ms for the 25 MB of a 1,024^2 grid (2.4 with the pages there).
static void touch_pages(void *buf, size_t bytes)
{
    volatile char *c = static_cast<volatile char *>(buf);
    for (size_t i = 0; c && i < bytes; i += 4096)
        c[i] = c[i];
}

extern "C" int slpic2d_fields(slpic2d_t *h, double *rho, double *phi, float *Ex, float *Ey)
{
    if (!h)
        return SLPIC_ERR_INVALID;
    // while the steps in flight run
    touch_pages(rho, sizeof(double) * h->p.nn);
    touch_pages(phi, sizeof(double) * h->p.nn);
    touch_pages(Ex, sizeof(float) * h->p.nn);
    touch_pages(Ey, sizeof(float) * h->p.nn);
    int rc = device_status(h);
    if (rc)
        return rc;
    const Params2D &p = h->p;
    const size_t nn = (size_t)p.nn;
    const unsigned grid = (unsigned)std::min<size_t>((nn + kThreads - 1) / kThreads, 152 * 8);
    if (phi)
        CK2(h, cudaMemcpyAsync(phi, p.phi, sizeof(double) * nn, cudaMemcpyDeviceToHost, h->stream));
    if (Ex || Ey) {
        // the components apart, in two of the CG's vectors (free between solves)
        k_split2d<<<grid, kThreads, 0, h->stream>>>(p, p.fr, p.fq);
        CK2(h, cudaGetLastError());
        if (Ex)
            CK2(h, cudaMemcpyAsync(Ex, p.fr, sizeof(float) * nn, cudaMemcpyDeviceToHost, h->stream));
        if (Ey)
            CK2(h, cudaMemcpyAsync(Ey, p.fq, sizeof(float) * nn, cudaMemcpyDeviceToHost, h->stream));
    }
    if (rho) {
        // rho of the current level from the deposits of the particles now stored (the consumed
        // deposit was cleared by the solve): made again here, in the vector of a standalone
        // solve's charge, and the deposits cleared
        CK2(h, cudaMemsetAsync(p.acc, 0, sizeof(unsigned long long) * nn * p.ns, h->stream));
        k_deposit2d<<<dim3(h->ctas, p.ns), kThreads, 0, h->stream>>>(p);
        k_rho2d<<<grid, kThreads, 0, h->stream>>>(p, p.r);
        CK2(h, cudaGetLastError());
        CK2(h, cudaMemcpyAsync(rho, p.r, sizeof(double) * nn, cudaMemcpyDeviceToHost, h->stream));
    }
    CK2(h, cudaStreamSynchronize(h->stream));
    return SLPIC_OK;
}

extern "C" int slpic2d_charge_raw(slpic2d_t *h, int s, int64_t *acc)
{
    if (!h || s < 0 || s >= h->p.ns || !acc)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    int rc = device_status(h);
    if (rc)
        return rc;
    const Params2D &p = h->p;
    const size_t nn = (size_t)p.nn;
    CK2(h, cudaMemsetAsync(p.acc, 0, sizeof(unsigned long long) * nn * p.ns, h->stream));
    k_deposit2d<<<dim3(h->ctas, p.ns), kThreads, 0, h->stream>>>(p);
    CK2(h, cudaGetLastError());
    CK2(h, cudaStreamSynchronize(h->stream));
    CK2(h, cudaMemcpy(acc, p.acc + (size_t)s * nn, sizeof(int64_t) * nn, cudaMemcpyDeviceToHost));
    CK2(h, cudaMemsetAsync(p.acc, 0, sizeof(unsigned long long) * nn * p.ns, h->stream));
    return device_status(h);
}

extern "C" int slpic2d_particle_count(slpic2d_t *h, int s, int64_t *n)
{
    if (!h || s < 0 || s >= h->p.ns || !n)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    State2D st;
    int rc = read_state(h, st);
    if (rc)
        return rc;
    const int P = (int)(st.step & 1);
    *n = (int64_t)(st.count[s][P] - st.holes[s][P]);
    return SLPIC_OK;
}

extern "C" int slpic2d_get_particles(slpic2d_t *h, int s, int32_t *cell, float *offset, float *v,
                                     int64_t *n)
{
    if (!h || s < 0 || s >= h->p.ns || !n || !cell || !offset || !v)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    State2D st;
    int rc = read_state(h, st);
    if (rc)
        return rc;
    const int P = (int)(st.step & 1);
    const long long slots = (long long)st.count[s][P];
    const long long live = slots - (long long)st.holes[s][P];
    if (*n < live)
        return fail2(h, SLPIC_ERR_CAPACITY, "output arrays too small");
    std::vector<int32_t> c((size_t)slots);
    std::vector<float4> pv((size_t)slots);
    std::vector<float> vz((size_t)slots);
    const Species2D &d = h->p.sp[s];
    if (slots) {
        CK2(h, cudaMemcpy(c.data(), d.cell[P], sizeof(int32_t) * slots, cudaMemcpyDeviceToHost));
        CK2(h, cudaMemcpy(pv.data(), d.pv[P], sizeof(float4) * slots, cudaMemcpyDeviceToHost));
        CK2(h, cudaMemcpy(vz.data(), d.vz[P], sizeof(float) * slots, cudaMemcpyDeviceToHost));
    }
    long long k = 0;
    for (long long i = 0; i < slots; ++i) {
        if (c[i] < 0)
            continue;
        cell[k] = c[i];
        offset[2 * k] = pv[i].x;
        offset[2 * k + 1] = pv[i].y;
        v[3 * k] = pv[i].z;
        v[3 * k + 1] = pv[i].w;
        v[3 * k + 2] = vz[i];
        ++k;
    }
    *n = k;
    return SLPIC_OK;
}

extern "C" int slpic2d_diagnostics(slpic2d_t *h, slpic2d_diag *out)
{
    if (!h || !out)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    int rc = device_status(h);
    if (rc)
        return rc;
    State2D st;
    rc = read_state(h, st);
    if (rc)
        return rc;
    std::memset(out, 0, sizeof(*out));
    out->step = st.step;
    out->time = (double)st.step * h->cfg.dt;
    const int P = (int)(st.step & 1);
    for (int s = 0; s < h->p.ns; ++s) {
        out->count[s] = (int64_t)(st.count[s][P] - st.holes[s][P]);
        out->absorbed[s][0] = st.absorbed_total[s][0];
        out->absorbed[s][1] = st.absorbed_total[s][1];
        out->injected[s] = st.injected_total[s];
    }
    out->cg_iterations = st.cg_iters;
    out->iterative_last = (int32_t)std::min<unsigned long long>(st.iter_last, 0x7fffffffULL);
    out->cg_iterations_total = st.cg_total;
    out->cg_rel_residual = st.cg_res;
    return SLPIC_OK;
}

extern "C" int slpic2d_solve_poisson(slpic2d_t *h, const double *rho, double *phi,
                                     int32_t *iterations, double *rel_residual)
{
    if (!h || !rho || !phi)
        return h ? fail2(h, SLPIC_ERR_INVALID, "bad arguments") : SLPIC_ERR_INVALID;
    int rc = device_status(h);
    if (rc)
        return rc;
    Params2D saved = h->p;
    Params2D &p = h->p;
    const size_t nn = (size_t)p.nn;
    // private phi and rho buffers so the simulation's fields stay as they are
    double *d_phi = nullptr;
    CK2(h, cudaMalloc(&d_phi, sizeof(double) * nn));
    std::vector<double> guess(phi, phi + nn);
    for (int i = 0; i < p.nx; ++i) {
        guess[i] = p.phi_lo;
        guess[(size_t)p.ny * p.nx + i] = p.phi_hi;
    }
    cudaError_t e = cudaMemcpy(d_phi, guess.data(), sizeof(double) * nn, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(p.r, rho, sizeof(double) * nn, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(d_phi);
        return fail2(h, SLPIC_ERR_CUDA, cudaGetErrorString(e));
    }
    p.phi = d_phi;
    rc = launch_solve(h, 1);
    h->p = saved;
    if (rc == SLPIC_OK)
        rc = device_status(h);
    if (rc == SLPIC_ERR_NOCONVERGE) {
        // a standalone solve's non-convergence is reported, not kept as the
        // simulation's error
        const int zero = 0;
        cudaMemcpy(&h->d_state->error, &zero, sizeof(int), cudaMemcpyHostToDevice);
    }
    State2D st;
    if (rc == SLPIC_OK || rc == SLPIC_ERR_NOCONVERGE) {
        if (read_state(h, st) == SLPIC_OK) {
            if (iterations)
                *iterations = st.cg_iters;
            if (rel_residual)
                *rel_residual = st.cg_res;
        }
        cudaMemcpy(phi, d_phi, sizeof(double) * nn, cudaMemcpyDeviceToHost);
    }
    cudaFree(d_phi);
    return rc;
}
