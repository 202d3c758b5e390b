// particle_step.cuh -- advance one macroparticle by one SLPIC step (device code),
// shared by every particle kernel of the library.
#pragma once

#include "push_math.cuh"
#include "slpic_internal.cuh"

namespace slpic {

__device__ __forceinline__ void deposit_node(unsigned long long *hist, int c, int c1, float b,
                                             float off)
{
    unsigned long long qL, qR;
    quantise(b, off, qL, qR);
    atomicAdd(hist + c, qL);
    atomicAdd(hist + c1, qR);
}

// Compile-time shape of a particle loop: kKind the species' beta kind (SLPIC_BETA_*)
// and kPer whether the grid is periodic (0/1), or kAny for "read at run time".  The
// fixed forms drop the run-time tests from the hot loop; the arithmetic, and so every
// result bit, is the same.
constexpr int kAny = -1;

// Gather (Sec. II): linear interpolation of the nodal field at the particle.
template <int kPer = kAny>
__device__ __forceinline__ float gather_ax(const StepParams &p, const SpeciesDev &sp,
                                           const float *sE, int c, float d)
{
    const bool periodic = kPer == kAny ? (p.periodic != 0) : (kPer != 0);
    int c1 = c + 1;
    if (periodic && c1 == p.n_cells)
        c1 = 0;
    // explicit roundings: every kernel that inlines this gets the same bits
    float Ep = __fmaf_rn(d, sE[c1], __fmul_rn(1.0f - d, sE[c]));
    return __fmul_rn(sp.qm, Ep);
}

// The speed limit of species sp in cell c (Sec. II: v0 may vary with position).
// kProf: a per-cell profile is set (p.lam), and the limit is the FP32 product
// v0 * lam[c] rounded to nearest; otherwise the species' uniform v0.  lam: a copy of
// the profile (in shared memory) to read instead of p.lam, or null.
template <bool kProf>
__device__ __forceinline__ float v0_at(const StepParams &p, const SpeciesDev &sp, int c,
                                       const float *lam = nullptr)
{
    if (!kProf)
        return sp.v0;
    return __fmul_rn(sp.v0, lam ? lam[c] : __ldg(p.lam + c));
}

// The same where a kernel serves both cases at run time (p.lam may be null).
__device__ __forceinline__ float v0_cell(const StepParams &p, const SpeciesDev &sp, int c)
{
    return p.lam ? __fmul_rn(sp.v0, __ldg(p.lam + c)) : sp.v0;
}

// After the velocity push (new vx): x^{n+1} = x^n + beta(|v^{n+1/2}|) v^{n+1/2} dt in
// cell units, walls or wrap, and rho^{n+1} += q w beta S(x - x^{n+1}) through
// dep(c, c+1, beta, offset).  Returns false if absorbed (wall = 0 at x=0, 1 at x=L).
// v0n is the limit of the start cell (that of the push); with kProf the deposit
// takes beta with the limit of the cell the particle ends in (the same beta if it
// stayed in its cell: a warp whose particles all stay skips the second division).
template <bool kProf = false, int kKind = kAny, int kPer = kAny, typename Dep>
__device__ __forceinline__ bool move_and_deposit(const StepParams &p, const SpeciesDev &sp,
                                                 Dep &dep, int &c, float4 &q, float vx, int &wall,
                                                 float v0n, const float *lam = nullptr)
{
    const int N = p.n_cells;
    const int kind = kKind == kAny ? sp.kind : kKind;
    const bool periodic = kPer == kAny ? (p.periodic != 0) : (kPer != 0);
    float b = beta_q(kind, vx, q.z, q.w, v0n);
    float xn = __fmaf_rn(__fmul_rn(b, vx), p.dt_dx, q.x);
    float fl = floorf(xn);
    int cn = c + (int)fl;
    float dn = xn - fl;
    if (dn >= 1.0f) {  // x just below a cell edge rounded up to it
        dn = 0.0f;
        cn += 1;
    }
    if (periodic) {
        cn %= N;
        if (cn < 0)
            cn += N;
    } else if (cn < 0) {
        wall = 0;
        return false;
    } else if (cn >= N) {
        wall = 1;
        return false;
    }
    int cn1 = cn + 1;
    if (periodic && cn1 == N)
        cn1 = 0;
    if (kProf && cn != c)
        b = beta_q(kind, vx, q.z, q.w, v0_at<true>(p, sp, cn, lam));
    dep(cn, cn1, b, dn);
    c = cn;
    q.x = dn;
    q.y = vx;
    return true;
}

// int64 shared-memory histogram
struct DepositU64 {
    unsigned long long *hist;
    __device__ __forceinline__ void operator()(int c, int c1, float b, float off)
    {
        deposit_node(hist, c, c1, b, off);
    }
};

// The same integers kept as two 32-bit words per node (value = hi 2^32 + lo):
// 32-bit shared-memory atomics are native; the carry out of lo is detected from
// the old value the atomic returns and added to hi, so the sum stays exact.
struct DepositSplit32 {
    unsigned *lo, *hi;
    __device__ __forceinline__ void add(int c, unsigned vl, unsigned vh)
    {
        unsigned old = atomicAdd(lo + c, vl);
        vh += (old + vl < old) ? 1u : 0u;
        if (vh)
            atomicAdd(hi + c, vh);
    }
    __device__ __forceinline__ void operator()(int c, int c1, float b, float off)
    {
        unsigned llo, lhi, rlo, rhi;
        quantise_split(b, off, llo, lhi, rlo, rhi);
        add(c, llo, lhi);
        add(c1, rlo, rhi);
    }
};

// Push one particle (Appendix A): returns false if absorbed (wall = 0 at x=0,
// 1 at x=L).  c, q updated in place.
__device__ __forceinline__ bool advance(const StepParams &p, const SpeciesDev &sp,
                                        const float *sE, unsigned long long *hist, int &c,
                                        float4 &q, int &wall)
{
    float ax = gather_ax(p, sp, sE, c, q.x);
    // v^{n+1/2} = v^{n-1/2} + a int beta dt
    float vx = push_vx(sp.kind, q.y, q.z, q.w, ax, p.dt, sp.v0);
    DepositU64 dep{hist};
    return move_and_deposit(p, sp, dep, c, q, vx, wall, sp.v0);
}

// Source particle i of species s for the step (Sec. IV source, the readings of
// LOSS_MATCHED / RATE): it takes uniforms u_j = u24(SplitMix64(key, 8i+j)), key the
// species' stream of the step, for its position in the band (FP32, pinned
// operations) and a physical Maxwellian velocity (Box-Muller): the g-source equals
// the f-source.
__device__ __forceinline__ void source_particle(const StepParams &p, const SpeciesDev &sp,
                                                unsigned long long key, long long i, int &c, float4 &q)
{
    const int N = p.n_cells;
    const unsigned long long b8 = 8ULL * (unsigned long long)i;
    const float u0 = u24(sm64_at(key, b8 + 0)), u1 = u24(sm64_at(key, b8 + 1));
    const float u2 = u24(sm64_at(key, b8 + 2)), u3 = u24(sm64_at(key, b8 + 3));
    const float u4 = u24(sm64_at(key, b8 + 4));
    if (p.src_mode == SLPIC_SRC_WALL) {
        // through the plate at x = L: the flux-weighted half-Maxwellian (|vx|
        // Rayleigh, towards -x), placed where it has moved since a uniformly
        // random entry time in the step; a position that rounds to the plate is
        // put at the largest cell coordinate below it
        const float vxm = sp.vth_src * sqrtf(-2.0f * logf(u1));
        const float rw = sp.vth_src * sqrtf(-2.0f * logf(u2));
        float sw, cw;
        sincospif(2.0f * u3, &sw, &cw);
        const float vy = rw * cw, vz = rw * sw;
        const float b = beta_q(sp.kind, -vxm, vy, vz, v0_cell(p, sp, N - 1));
        float xc = __fsub_rn((float)N, __fmul_rn(u0, __fmul_rn(__fmul_rn(b, vxm), p.dt_dx)));
        if (!(xc < (float)N))
            xc = __int_as_float(__float_as_int((float)N) - 1);
        xc = fmaxf(xc, 0.0f);
        const float fc = floorf(xc);
        c = (int)fc;
        q = make_float4(xc - fc, -vxm, vy, vz);
    } else {
        const float xc = __fadd_rn(p.src_lo_cells, __fmul_rn(u0, p.src_len_cells));
        const float fc = floorf(xc);
        c = (int)fc;
        // physical Maxwellian (Box-Muller); the g-source equals the f-source
        const float r1 = sqrtf(-2.0f * logf(u1)), r2 = sqrtf(-2.0f * logf(u3));
        float s2, c2;
        sincospif(2.0f * u2, &s2, &c2);
        q = make_float4(xc - fc, sp.vth_src * r1 * c2, sp.vth_src * r1 * s2,
                        sp.vth_src * r2 * cospif(2.0f * u4));
    }
}

// The step's source count of a species: macroparticles k to make, given the ref species'
// absorbed macroparticles of the step and the fraction carried (updated).
__device__ __forceinline__ long long source_count(const StepParams &p, const SpeciesDev &sp,
                                                  unsigned long long ref_absorbed, double &frac)
{
    double S = 0.0;
    if (p.src_mode == SLPIC_SRC_LOSS_MATCHED)
        S = (double)ref_absorbed * p.sp[p.src_ref].w;
    else if (p.src_mode == SLPIC_SRC_RATE)
        S = p.src_rate * p.dt64;
    long long k = 0;
    if (p.src_mode == SLPIC_SRC_WALL) {
        if (sp.wall_rate > 0.0) {
            frac += sp.wall_rate;
            k = (long long)floor(frac);
            frac -= (double)k;
        }
    } else if (p.src_mode != SLPIC_SRC_NONE && sp.vth_src > 0.0f) {
        frac = fma(S, sp.inv_w, frac);
        k = (long long)floor(frac);
        frac -= (double)k;
    }
    return k;
}

// the GPU's global timer, ns
__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

}  // namespace slpic
