// unet_blocked.cuh -- the U-Net's tensor-core convolutions on BF16 operands that lie in
// memory the way the tensor cores read them (included by unet.cu).
//
// What bounds a U-Net pass is moving activations, not the multiplies: at 1024 x 1024
// with 32 base channels the forward's 204 GFLOP take 0.11 ms at the measured BF16 rate.
// The implicit-GEMM kernels that gather their A operand from FP32 planes
// (k_conv_fwd_tc, k_conv_wgrad_tc in unet.cu) spend the time on that gather: nine
// taps x 2 loads, conversions and bounds tests per pixel and channel, on 66 % of the
// issue slots with the tensor pipe 9 % busy.  Here the producer of a tensor rounds it
// to BF16 once, at the same place in the arithmetic, and stores it in channel blocks
//
//     value (n, c, y, x)  at  p[((n * groups + c / 8) * ps + (y + 1) * P + x + 1) * 8 + c % 8],
//     P = W + 2, one zero column left and right, a zero row above and below
//
// so that a pixel's 8 channels are 16 contiguous bytes: one row of an 8 x 16-byte core
// matrix.  A run of pixels of one channel block is then a contiguous piece of memory
// (one bulk copy), already in the shared-memory image the MMA descriptors want, and a
// tap's shift by one pixel is a shift of the descriptor's start address by 16 bytes:
// the nine taps read one copy of the rows.  The zero frame is the convolution's padding,
// so no tap needs a bounds test.  The layout serves both operand orders: K-major for the
// convolutions (K = channels) and M/N-major for the weight gradient (K = pixels).
//
// The sums keep the K order of the gather kernels (tap-major, 16 channels per MMA), so
// activations and input gradients are theirs bit for bit (the weight gradient's partial
// sums split the pixels elsewhere).  Pooling, upsampling, the ReLU masks and the bias
// gradient, which were passes over memory of their own, happen in the epilogues, on the
// FP32 accumulators.
//
// A ReLU output of zero is stored as -0 (0x8000): +0 is then a positive value too small
// for BF16, and the backward mask a > 0 of the FP32 activation is "bits != 0x8000".  To
// the MMAs both are zero.
#pragma once

namespace {

struct Blk {  // a blocked BF16 tensor; positions include the frame
    __nv_bfloat16 *p;
    int groups;  // channel blocks per sample
    int off;     // first block of the view
    size_t ps;   // positions per block: plane and slack
};

constexpr int kBX = 128;               // pixels per MMA tile (M), along a row
constexpr int kBSlab = (kBX + 2) * 16; // bytes of one channel block of a tile's row
constexpr int kBRing = 32;             // most stages of the weight ring
constexpr int kBRows = 8;              // most row buffers
constexpr int kBPiece = kBX * 16;      // one channel block of one tap (streamed A)
constexpr int kBEpi = 16;              // epilogue warps
constexpr int kBThreads = 32 * (kBEpi + 3);  // and the row, weight and MMA warps
constexpr uint16_t kZeroAct = 0x8000;  // stored for a ReLU output of zero

enum BlkMode {
    kBmOut = 0,     // out: FP32 image of channel 0, bias added, no ReLU
    kBmAct = 1,     // bias, ReLU, to dst; with MT == 2 and pool.p also the 2x2 mean to pool
    kBmActUp = 2,   // bias, ReLU, nearest-upsampled into dst (the finer level)
    kBmGradUp = 3,  // channels < cup: 2x2 sums, masked, to dst (the coarser level); the
                    // rest as FP32 to f32
    kBmGradPool = 4,  // 4 finer pixels f32 + v/4 each, masked, to dst (the finer level)
    kBmGradMask = 5,  // masked, to dst
};

struct ConvBlk {
    Blk x;            // input operand
    int G;            // its channel blocks that take part (even)
    int H, W;         // the grid the conv runs on
    const __nv_bfloat16 *wp;  // packed weights of this launch's output channels
    size_t bstride;   // elements between their chunks
    int Np, nout;     // output channels: padded, stored
    int o0;           // first output channel of this launch
    const float *bias;
    int nb;           // samples
    int slabs;        // row buffers (MT + 2 .. kBRows)
    int bst;          // stages of the weight ring (all chunks where they fit)
    int mode;
    Blk dst, pool, mask;
    float *f32;
    int cup;          // kBmGradUp: channels of the upsampled half
    double *bpart;    // the CTAs' bias-gradient sums [CTA][bchan] (gradient modes)
    int bchan;
    int *flag;
};

__device__ __forceinline__ uint64_t blk_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) |
           ((uint64_t)(sbo >> 4) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ void blk_copy(uint32_t dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(tc_smem(bar))
        : "memory");
}

__device__ __forceinline__ void blk_expect(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void blk_mma(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %4, 0; "
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d),
        "l"(da), "l"(db), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void blk_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     tc_smem(bar))
                 : "memory");
}

__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t p;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(p));
    return p;
}

// tc_wait for a barrier that has mostly completed by now: no clock is read before the
// first test has failed
__device__ __forceinline__ bool blk_wait(uint64_t *bar, unsigned parity, int *flag)
{
    unsigned ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(tc_smem(bar)), "r"(parity)
        : "memory");
    return ok || tc_wait(bar, parity, flag);
}

__device__ __forceinline__ uint32_t blk_cols(int n) { return n <= 32 ? 32u : n <= 64 ? 64u : n <= 128 ? 128u : n <= 256 ? 256u : 512u; }

// 8 columns of one or two accumulators for this thread's lane.  The loads and their wait
// are one statement, so that no use of a register can be placed between them.
__device__ __forceinline__ void blk_ld(uint32_t addr, float (&v)[1][8], int)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(v[0][0]), "=f"(v[0][1]), "=f"(v[0][2]), "=f"(v[0][3]), "=f"(v[0][4]),
                   "=f"(v[0][5]), "=f"(v[0][6]), "=f"(v[0][7])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void blk_ld(uint32_t addr, float (&v)[2][8], int next)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
                 "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(v[0][0]), "=f"(v[0][1]), "=f"(v[0][2]), "=f"(v[0][3]), "=f"(v[0][4]),
                   "=f"(v[0][5]), "=f"(v[0][6]), "=f"(v[0][7]), "=f"(v[1][0]), "=f"(v[1][1]),
                   "=f"(v[1][2]), "=f"(v[1][3]), "=f"(v[1][4]), "=f"(v[1][5]), "=f"(v[1][6]),
                   "=f"(v[1][7])
                 : "r"(addr), "r"(addr + (uint32_t)next)
                 : "memory");
}

__device__ __forceinline__ uint32_t bf16_bits(float a)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a));
}
__device__ __forceinline__ uint4 pack8(const float (&v)[8])
{
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        w[q] = bf16_bits(v[2 * q]) | (bf16_bits(v[2 * q + 1]) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// ReLU outputs: a zero (a not > 0) as -0
__device__ __forceinline__ uint4 pack8_act(const float (&v)[8])
{
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
        w[q] = v[q] > 0.0f ? bf16_bits(v[q]) : (uint32_t)kZeroAct;
    return make_uint4(w[0] | (w[1] << 16), w[2] | (w[3] << 16), w[4] | (w[5] << 16), w[6] | (w[7] << 16));
}
// g where the activation whose code is stored was > 0, else 0
__device__ __forceinline__ void mask8(float (&g)[8], uint4 code)
{
    const uint32_t c[4] = {code.x, code.y, code.z, code.w};
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if (((c[q >> 1] >> ((q & 1) * 16)) & 0xFFFFu) == kZeroAct)
            g[q] = 0.0f;
}

__device__ __forceinline__ uint4 *blk_at(const Blk &b, int n, int g, size_t pos)
{
    return reinterpret_cast<uint4 *>(b.p) + (((size_t)n * b.groups + b.off + g) * b.ps + pos);
}

// The bias gradients' sums: over a warp's tile on the FP32 pipe, from there on in FP64, whose
// pipe (2 lanes per SM here) could not take one addition per value.  A tile's sum is three
// numbers, a the FP32 sum, b the sum of its additions' exact errors (Knuth's two-sum), c that
// of b's: Ogita, Rump and Oishi's cascaded summation (SIAM J. Sci. Comput. 26, 2005) with
// three terms, good to some 70 bits of the sum of the magnitudes, more than FP64 keeps.  FP32's
// range does not hold partial sums of large values: those go to FP64 (bias_large).  Over pairs
// (48 bits) the third term costs 30 us of the 1,640 of loss and gradients of 512^2, batch 2.
struct Sum3 {
    float a, b, c;
};
__device__ __forceinline__ float two_sum(float x, float y, float &e)
{
    const float s = __fadd_rn(x, y), t = __fsub_rn(s, x);
    e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, t)), __fsub_rn(y, t));
    return s;
}
__device__ __forceinline__ void sum3_add(Sum3 &s, float v)
{
    float e, f;
    s.a = two_sum(s.a, v, e);
    s.b = two_sum(s.b, e, f);
    s.c = __fadd_rn(s.c, f);
}
// x and y of T terms, the rest zero (the sum has a term more)
template <int T>
__device__ __forceinline__ Sum3 sum3_add(const Sum3 &x, const Sum3 &y)
{
    float e, f, g;
    Sum3 r{0.0f, 0.0f, 0.0f};
    r.a = two_sum(x.a, y.a, e);
    if (T == 1) {
        r.b = e;
        return r;
    }
    r.b = two_sum(x.b, y.b, f);
    r.b = two_sum(r.b, e, g);
    r.c = __fadd_rn(f, g);
    if (T == 3)
        r.c = __fadd_rn(__fadd_rn(x.c, y.c), r.c);
    return r;
}
template <int T>
__device__ __forceinline__ Sum3 sum3_shfl(const Sum3 &s, int o)
{
    return Sum3{__shfl_xor_sync(0xffffffffu, s.a, o), T > 1 ? __shfl_xor_sync(0xffffffffu, s.b, o) : 0.0f,
                T > 2 ? __shfl_xor_sync(0xffffffffu, s.c, o) : 0.0f};
}
// one exchange: of 2 K channels a lane keeps K
template <int T, int K>
__device__ __forceinline__ void sum3_exchange(Sum3 (&v)[8])
{
    const bool up = threadIdx.x & (4 * K);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const Sum3 keep = up ? v[k + K] : v[k], send = up ? v[k] : v[k + K];
        v[k] = sum3_add<T>(keep, sum3_shfl<T>(send, 4 * K));
    }
}
// The sums of 8 channels over the warp's lanes (sums of T terms), added to bp[8]; channel
// (l>>4 & 1)*4 + (l>>3 & 1)*2 + (l>>2 & 1) ends in lane l.
template <int T>
__device__ __forceinline__ void bias_warp(Sum3 (&v)[8], double *bp)
{
    constexpr int T1 = T < 3 ? T + 1 : 3, T2 = T1 < 3 ? T1 + 1 : 3;
    sum3_exchange<T, 4>(v);
    sum3_exchange<T1, 2>(v);
    sum3_exchange<T2, 1>(v);
    v[0] = sum3_add<3>(v[0], sum3_shfl<3>(v[0], 2));
    v[0] = sum3_add<3>(v[0], sum3_shfl<3>(v[0], 1));
    const int lane = threadIdx.x & 31;
    if (!(lane & 3))  // this warp's own entry
        bp[(lane >> 4) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] +=
            (double)v[0].a + ((double)v[0].b + (double)v[0].c);
}
// Where a lane's eight values reach 2^100 in sum (large values, infinities, NaN: rare), the
// warp's are added to bp[8] in FP64 and taken out of v.  The whole warp.
__device__ __forceinline__ void bias_large(float (&v)[8], double *bp)
{
    float m = fabsf(v[0]);
#pragma unroll
    for (int q = 1; q < 8; ++q)
        m = __fadd_rn(m, fabsf(v[q]));
    if (__all_sync(0xffffffffu, m < 0x1p100f))
        return;
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
        double d = 0.0;
#pragma unroll
        for (int r = 0; r < 8; ++r)  // (constant indices: v stays in registers)
            if (r == q) {
                d = (double)v[r];
                v[r] = 0.0f;
            }
        for (int o = 16; o; o >>= 1)
            d += __shfl_xor_sync(0xffffffffu, d, o);
        if ((threadIdx.x & 31) == 0)
            bp[q] += d;
    }
    __syncwarp();
}

// ---- convolution (and, on mirrored weights, its input gradient) ---------------------
// A persistent CTA per SM takes units of MT vertically adjacent rows x kBX pixels (MT
// accumulators in TMEM, twice, so that a unit's epilogue runs beside the next unit's
// MMAs), going down a column of the image: MT of a unit's MT + 2 input rows are new, the
// other two are still in the ring of row buffers.  A producer warp copies the rows,
// another the weight chunks (once, where all of them fit beside the rows; else a ring),
// one warp issues the MMAs as they land; 16 warps run the epilogues.  The MMAs are the
// bound at many channels (operands from shared memory at 128 B a cycle: 40 cycles for M
// 128 N 32 K 16, measured), the epilogue's stores at few.  With a CTA per unit instead
// (one resident, of 122 KB, at 96 channels) the latencies of copies, MMAs and epilogue
// added up to 13 us a unit: 355 us for the 96 -> 32 conv at 1024 x 1024.
// Every wait is bounded (tc_wait); a wait that gives up sets the flag, the roles stop, and
// the copies already issued are waited for before the CTA leaves.
//
// kStream: where the rows do not fit (many channels), the A operand is copied chunk by
// chunk beside the weights (128 pixels of the chunk's four 16-channel slices at their
// taps): every row is then read nine times, from L2.
template <int MT, bool kStream, bool kGrad>
__global__ void __launch_bounds__(kBThreads, 1) k_conv_blk(const __grid_constant__ ConvBlk a)
{
    extern __shared__ __align__(1024) unsigned char bsm[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_row[kBRows], s_rfree[kBRows], s_wfull[kBRing], s_wfree[kBRing];
    __shared__ __align__(8) uint64_t s_done[2], s_tfree[2];
    __shared__ volatile int s_fail;
    __shared__ double s_bp[kGrad ? 4 : 1][kGrad ? 256 : 1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int P = a.W + 2, G = a.G;
    const int HP = (a.H + MT - 1) / MT, xt = (a.W + kBX - 1) / kBX;
    const int units = a.nb * xt * HP;
    const int u0 = (int)((long long)units * blockIdx.x / gridDim.x);
    const int u1 = (int)((long long)units * (blockIdx.x + 1) / gridDim.x);
    const int wbytes = a.Np * kTcKC * 2;
    const int abytes = kStream ? MT * 8 * kBPiece : 0;  // of a stage
    const int chunkB = wbytes + abytes;                 // a stage: weights, then A
    const int nkb = 9 * (G / 2), nkc = (nkb + 3) / 4;
    const int slab = G * kBSlab;
    unsigned char *s_w = bsm + (kStream ? (size_t)0 : (size_t)a.slabs * slab);
    const uint32_t ncols = blk_cols(2 * MT * a.Np);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc_smem(&s_tmem)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 32) {
        auto init = [](uint64_t *b, int n, unsigned count) {
            for (int r = 0; r < n; ++r)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(b + r)), "r"(count));
        };
        init(s_row, kBRows, 1);
        init(s_rfree, kBRows, 1);
        init(s_wfull, kBRing, 1);
        init(s_wfree, kBRing, 1);
        init(s_done, 2, 1);
        init(s_tfree, 2, kBEpi);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    if (kGrad)
        for (int k = tid; k < 4 * 256; k += kBThreads)
            s_bp[k >> 8][k & 255] = 0.0;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp == kBEpi && !kStream) {
        // ---- the input rows, a bulk copy per channel block: of a column's first unit all
        // MT + 2, of the next ones the MT new ones
        int load = 0, st = 0;
        unsigned ph = 1u;  // parity of the buffer's previous use
        bool ok = true;
        for (int u = u0; u < u1 && ok; ++u) {
            const int pr = u % HP, c = u / HP, x0 = (c % xt) * kBX, n = c / xt;
            for (int r = (u == u0 || pr == 0) ? 0 : 2; r < MT + 2; ++r, ++load) {
                if (load >= a.slabs && lane == 0)
                    ok = tc_wait(&s_rfree[st], ph, a.flag);
                ok = __all_sync(0xffffffffu, ok && !s_fail);
                if (!ok)
                    break;
                if (lane == 0)
                    blk_expect(&s_row[st], (unsigned)slab);
                __syncwarp();
                const uint32_t dst = tc_smem(bsm + (size_t)st * slab);
                const uint4 *src = blk_at(a.x, n, 0, (size_t)(pr * MT + r) * P + x0);
                for (int g = lane; g < G; g += 32)
                    blk_copy(dst + g * kBSlab, src + (size_t)g * a.x.ps, kBSlab, &s_row[st]);
                if (++st == a.slabs) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
        if (lane == 0) {
            if (!ok)
                s_fail = 1;
            for (int k = load > a.slabs ? load - a.slabs : 0; k < load; ++k)  // landed before the CTA may leave
                tc_wait(&s_row[k % a.slabs], (unsigned)((k / a.slabs) & 1), a.flag);
        }
    } else if (warp == kBEpi + 1) {
        // ---- the weights (and a streamed A), chunk by chunk (64 k): once each where every
        // chunk has a stage of its own, else round the ring for every unit
        const bool once = !kStream && a.bst >= nkc;
        int g = 0, st = 0;
        unsigned ph = 1u;
        bool ok = true;
        for (int u = u0; u < (once ? min(u0 + 1, u1) : u1) && ok; ++u) {
            const int pr = u % HP, c = u / HP, x0 = (c % xt) * kBX, n = c / xt;
            for (int kc = 0; kc < nkc; ++kc, ++g) {
                if (g >= a.bst && lane == 0)
                    ok = tc_wait(&s_wfree[st], ph, a.flag);
                ok = __all_sync(0xffffffffu, ok && !s_fail);
                if (!ok)
                    break;
                const uint32_t dst = tc_smem(s_w + (size_t)st * chunkB);
                const int kbs = min(4, nkb - 4 * kc);  // k slices of this chunk
                if (lane == 0) {
                    blk_expect(&s_wfull[st], (unsigned)(wbytes + (kStream ? MT * kbs * 2 * kBPiece : 0)));
                    blk_copy(dst, a.wp + (size_t)kc * a.bstride, (unsigned)wbytes, &s_wfull[st]);
                }
                if (kStream) {
                    __syncwarp();
                    if (lane < MT * kbs * 2) {
                        const int mt = lane / (kbs * 2), e = lane - mt * kbs * 2;  // slice e/2, block e%2
                        const int kb = 4 * kc + (e >> 1), t = kb / (G / 2), gg = 2 * (kb - t * (G / 2)) + (e & 1);
                        const int di = t / 3, dj = t - di * 3;
                        blk_copy(dst + wbytes + (mt * 8 + e) * kBPiece,
                                 blk_at(a.x, n, gg, (size_t)(pr * MT + mt + di) * P + x0 + dj), kBPiece,
                                 &s_wfull[st]);
                    }
                }
                if (++st == a.bst) {
                    st = 0;
                    ph ^= 1u;
                }
            }
        }
        if (lane == 0) {
            if (!ok)
                s_fail = 1;
            for (int k = g > a.bst ? g - a.bst : 0; k < g; ++k)  // landed before the CTA may leave
                tc_wait(&s_wfull[k % a.bst], (unsigned)((k / a.bst) & 1), a.flag);
        }
    } else if (warp == kBEpi + 2) {
        // ---- MMAs in the K order tap-major, 16 channels each.  The warp's instructions pace
        // the tensor pipe, so the descriptors advance by additions on their low word (start
        // address in 16-byte units), stages and phases are counted, and the whole warp runs
        // the loops with one elected lane issuing: no branch of them depends on a wait's
        // result, and the descriptors stay in uniform registers.  (A single lane's loop took
        // 188 cycles per MMA, 470 with the descriptors formed from scratch.)
        const uint32_t lead = elect_one();
        const uint32_t idesc = tc_idesc(a.Np);
        const uint32_t sa = tc_smem(bsm) >> 4, sw = tc_smem(s_w) >> 4;
        const uint32_t alo = (uint32_t)((kStream ? kBPiece : kBSlab) >> 4) << 16, ahi = (128u >> 4) | (1u << 14);
        const uint32_t blo = (128u >> 4) << 16, bhi = (1024u >> 4) | (1u << 14);
        const uint32_t slab16 = (uint32_t)slab >> 4, chunk16 = (uint32_t)chunkB >> 4;
        constexpr uint32_t kStep = 2 * (kStream ? kBPiece : kBSlab) / 16;  // 16 channels of A
        const bool once = !kStream && a.bst >= nkc;
        int st = 0, slot = 0;        // weight stage; row buffer of the unit's first row
        unsigned ph = 0u, rph = 0u;  // their phases
        bool ok = true;
        for (int u = u0, k = 0; u < u1; ++u, ++k) {
            const uint32_t acc = tmem + (uint32_t)((k & 1) * MT * a.Np);
            if (k >= 2)
                ok = ok && blk_wait(&s_tfree[k & 1], (unsigned)(((k >> 1) - 1) & 1), a.flag);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // the unit's rows: buffer and phase; those shared with the unit before have landed
            const bool first = k == 0 || u % HP == 0;
            int rs[MT + 2];
            unsigned rp[MT + 2];
            {
                int s = slot;
                unsigned f = rph;
#pragma unroll
                for (int r = 0; r < MT + 2; ++r) {
                    rs[r] = s;
                    rp[r] = f;
                    if (++s == a.slabs) {
                        s = 0;
                        f ^= 1u;
                    }
                }
            }
            int kk = 0;
            uint32_t accum = 0u, bd = 0u, ad[MT];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                ad[mt] = 0u;
            if (once)
                st = 0;
#pragma unroll
            for (int di = 0; di < 3; ++di) {
                if (!kStream)
#pragma unroll
                    for (int r = 0; r < MT + 2; ++r)
                        if ((di == 0 ? r < MT : r == di + MT - 1) && (first || r >= 2))
                            ok = ok && blk_wait(&s_row[rs[r]], rp[r], a.flag);
#pragma unroll 1
                for (int dj = 0; dj < 3; ++dj) {
                    if (!kStream)
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt)
                            ad[mt] = (sa + (uint32_t)rs[di + mt] * slab16 + (uint32_t)dj) | alo;
#pragma unroll 1
                    for (int cb = 0; cb < G / 2; ++cb) {
                        if (kk == 0) {
                            if (!once || k == 0) {
                                ok = ok && blk_wait(&s_wfull[st], ph, a.flag);
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            }
                            bd = (sw + (uint32_t)st * chunk16) | blo;
                            if (kStream)
#pragma unroll
                                for (int mt = 0; mt < MT; ++mt)
                                    ad[mt] = (sw + (uint32_t)st * chunk16 +
                                              (uint32_t)((wbytes + mt * 8 * kBPiece) >> 4)) | alo;
                        }
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            if (lead)
                                blk_mma(acc + (uint32_t)(mt * a.Np), ((uint64_t)ahi << 32) | ad[mt],
                                        ((uint64_t)bhi << 32) | bd, idesc, accum);
                            ad[mt] += kStep;
                        }
                        accum = 1u;
                        bd += 256 / 16;
                        if (++kk == 4) {
                            if (!once && lead)
                                blk_commit(&s_wfree[st]);
                            kk = 0;
                            if (++st == a.bst) {
                                st = 0;
                                ph ^= 1u;
                            }
                        }
                    }
                }
            }
            if (kk) {  // a last chunk of fewer slices
                if (!once && lead)
                    blk_commit(&s_wfree[st]);
                if (++st == a.bst) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            if (once) {
                st = 0;
                ph = 0u;
            }
            // the rows that no later unit reads (a commit covers every MMA before it)
            if (!kStream) {
                const bool last = (u + 1) % HP == 0 || u + 1 == u1;
#pragma unroll
                for (int r = 0; r < MT + 2; ++r)
                    if (r < MT || last) {
                        if (lead)
                            blk_commit(&s_rfree[rs[r]]);
                        if (++slot == a.slabs) {
                            slot = 0;
                            rph ^= 1u;
                        }
                    }
            }
            // after a wait that gave up the sums are void: the epilogues stop at s_fail
            if (!ok)
                s_fail = 1;
            __threadfence_block();
            if (lead)
                blk_commit(&s_done[k & 1]);
        }
    } else if (warp < kBEpi) {
        // ---- epilogues: thread = pixel x0 + 32 (warp mod 4) + lane; the groups of four
        // warps take the blocks of 8 channels in turn
        bool ok = true;
        for (int u = u0, k = 0; u < u1; ++u, ++k) {
            const int y0 = (u % HP) * MT, cc = u / HP, x0 = (cc % xt) * kBX, n = cc / xt;
            ok = tc_wait(&s_done[k & 1], (unsigned)((k >> 1) & 1), a.flag);
            ok = __all_sync(0xffffffffu, ok && !s_fail);
            if (!ok)
                break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int m = (warp & 3) * 32 + lane, x = x0 + m;
            const uint32_t tl = tmem + (uint32_t)((k & 1) * MT * a.Np) + ((uint32_t)((warp & 3) * 32) << 16);
            const bool inx = x < a.W;
            for (int og = warp >> 2; og * 8 < a.nout; og += kBEpi / 4) {
                float v[MT][8];
                blk_ld(tl + (uint32_t)(og * 8), v, a.Np);
                Sum3 bs[8];
                double *bp = s_bp[kGrad ? warp & 3 : 0] + (kGrad ? og * 8 : 0);
                if (!kGrad && a.mode == kBmOut) {
                    if (og == 0)
#pragma unroll
                        for (int t = 0; t < MT; ++t)
                            if (inx && y0 + t < a.H)
                                a.f32[((size_t)n * a.H + y0 + t) * a.W + x] = v[t][0] + a.bias[0];
                } else if (!kGrad) {
#pragma unroll
                    for (int t = 0; t < MT; ++t) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            v[t][q] = fmaxf(v[t][q] + __ldg(a.bias + og * 8 + q), 0.0f);
                        const int y = y0 + t;
                        if (inx && y < a.H) {
                            const uint4 w = pack8_act(v[t]);
                            if (a.mode == kBmAct) {
                                *blk_at(a.dst, n, a.o0 / 8 + og, (size_t)(y + 1) * P + x + 1) = w;
                            } else {
                                const int Pf = 2 * a.W + 2;
                                uint4 *d = blk_at(a.dst, n, a.o0 / 8 + og,
                                                  (size_t)(2 * y + 1) * Pf + 2 * x + 1);
                                d[0] = w;
                                d[1] = w;
                                d[Pf] = w;
                                d[Pf + 1] = w;
                            }
                        }
                    }
                    if (MT == 2 && a.pool.p) {
                        float s[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float t0 = v[0][q] + __shfl_xor_sync(0xffffffffu, v[0][q], 1);
                            const float t1 = v[MT - 1][q] + __shfl_xor_sync(0xffffffffu, v[MT - 1][q], 1);
                            s[q] = 0.25f * (t0 + t1);
                        }
                        if (inx && !(lane & 1))
                            *blk_at(a.pool, n, a.o0 / 8 + og,
                                    (size_t)(y0 / 2 + 1) * (a.W / 2 + 2) + x / 2 + 1) = pack8(s);
                    }
                } else if (a.mode == kBmGradUp) {
                    if (a.o0 + og * 8 < a.cup) {
                        // gradient of the upsampled activation: the cell's four, masked
                        float s[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float t0 = v[0][q] + __shfl_xor_sync(0xffffffffu, v[0][q], 1);
                            const float t1 = v[MT - 1][q] + __shfl_xor_sync(0xffffffffu, v[MT - 1][q], 1);
                            s[q] = t0 + t1;
                        }
                        const bool mine = inx && !(lane & 1);
                        if (mine) {
                            const int cg = a.o0 / 8 + og;
                            mask8(s, *blk_at(a.mask, n, cg, (size_t)(y0 + 1) * P + x + 1));
                            *blk_at(a.dst, n, cg, (size_t)(y0 / 2 + 1) * (a.W / 2 + 2) + x / 2 + 1) = pack8(s);
                        } else {
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                s[q] = 0.0f;
                        }
                        bias_large(s, bp);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            bs[q] = Sum3{s[q], 0.0f, 0.0f};
                        bias_warp<1>(bs, bp);
                    } else {
                        const int cg = (a.o0 - a.cup) / 8 + og, gs = (a.bchan - a.cup) / 8;
#pragma unroll
                        for (int t = 0; t < MT; ++t)
                            if (inx) {
                                float4 *d = reinterpret_cast<float4 *>(a.f32) +
                                            ((((size_t)n * gs + cg) * a.H + y0 + t) * a.W + x) * 2;
                                d[0] = make_float4(v[t][0], v[t][1], v[t][2], v[t][3]);
                                d[1] = make_float4(v[t][4], v[t][5], v[t][6], v[t][7]);
                            }
                    }
                } else if (a.mode == kBmGradPool) {
                    const int Wf = 2 * a.W, Pf = Wf + 2, cg = a.o0 / 8 + og, gs = a.bchan / 8;
#pragma unroll
                    for (int t = 0; t < MT; ++t) {
                        const int y = y0 + t;
                        if (y < a.H) {
#pragma unroll
                            for (int f = 0; f < 4; ++f) {
                                float s[8] = {};
                                if (inx) {
                                    const int yf = 2 * y + (f >> 1), xf = 2 * x + (f & 1);
                                    const float4 *d = reinterpret_cast<const float4 *>(a.f32) +
                                                      ((((size_t)n * gs + cg) * (2 * a.H) + yf) * Wf + xf) * 2;
                                    const float4 d0 = d[0], d1 = d[1];
                                    const float e[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
                                    for (int q = 0; q < 8; ++q)
                                        s[q] = e[q] + 0.25f * v[t][q];
                                    const size_t pos = (size_t)(yf + 1) * Pf + xf + 1;
                                    mask8(s, *blk_at(a.mask, n, cg, pos));
                                    *blk_at(a.dst, n, cg, pos) = pack8(s);
                                }
                                bias_large(s, bp);
#pragma unroll
                                for (int q = 0; q < 8; ++q)
                                    if (t == 0 && f == 0)
                                        bs[q] = Sum3{s[q], 0.0f, 0.0f};
                                    else if (t == 0 && f == 1)
                                        bs[q] = sum3_add<1>(bs[q], Sum3{s[q], 0.0f, 0.0f});
                                    else
                                        sum3_add(bs[q], s[q]);
                            }
                        }
                    }
                    bias_warp<3>(bs, bp);
                } else {  // kBmGradMask
#pragma unroll
                    for (int t = 0; t < MT; ++t) {
                        const int y = y0 + t, cg = a.o0 / 8 + og;
                        if (y < a.H) {
                            if (inx) {
                                const size_t pos = (size_t)(y + 1) * P + x + 1;
                                mask8(v[t], *blk_at(a.mask, n, cg, pos));
                                *blk_at(a.dst, n, cg, pos) = pack8(v[t]);
                            } else {
#pragma unroll
                                for (int q = 0; q < 8; ++q)
                                    v[t][q] = 0.0f;
                            }
                            bias_large(v[t], bp);
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                bs[q] = t == 0 ? Sum3{v[t][q], 0.0f, 0.0f}
                                               : sum3_add<1>(bs[q], Sum3{v[t][q], 0.0f, 0.0f});
                        }
                    }
                    bias_warp<MT>(bs, bp);
                }
            }
            // the accumulators may be overwritten
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc_smem(&s_tfree[k & 1])) : "memory");
        }
        if (kGrad) {
            // the CTA's bias-gradient sums, the four warps of pixels in order
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kBEpi) : "memory");
            for (int o = tid; o < a.nout; o += 32 * kBEpi)
                a.bpart[(size_t)blockIdx.x * a.bchan + a.o0 + o] =
                    ((s_bp[0][o] + s_bp[1][o]) + s_bp[2][o]) + s_bp[3][o];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// db[o] = the CTAs' sums in a fixed order (FP64; a CTA per channel)
__global__ void __launch_bounds__(kT) k_bias_tiles(const double *__restrict__ part, int tiles, int bchan,
                                                 float *__restrict__ db)
{
    __shared__ double s_red[kT / 32];
    const int o = blockIdx.x;
    double acc = 0.0;
    for (int t = threadIdx.x; t < tiles; t += kT)
        acc += part[(size_t)t * bchan + o];
    for (int off = 16; off; off >>= 1)
        acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0)
        s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int k = 0; k < kT / 32; ++k)
            v += s_red[k];
        db[o] = (float)v;
    }
}

// ---- weight gradient --------------------------------------------------------------
// dW[o][c][(di, dj)] = sum over pixels p of dz[o][p] x[c][p + (di - 1) P + dj - 1], a GEMM
// with K = pixels: both operands lie M/N-major in the blocked layout (a pixel's 8
// channels contiguous, pixels 16 B apart), so bulk copies of runs of positions are the
// operands and no thread touches them.  K runs over the positions of rows 1..H, frame
// columns included: dz is zero there, so they add nothing and rows of any width need no
// remainder.  The M rows of a tile are 16 channel blocks of the list (di, c / 8): three
// shifted rows of x side by side in shared memory, one copy serving the three dj by a
// shift of the descriptor start.  A CTA holds up to 512 TMEM columns of tiles and a range
// of the pixel chunks; the ranges' sums are added afterwards in a fixed order.
constexpr int kWKP = 64;              // positions per chunk
constexpr int kWThreads = 320;        // 8 warps for the results, a copy warp, an MMA warp
constexpr int kWRun = (kWKP + 2) * 16;

struct WgradBlk {
    Blk x, dz;
    int G;         // channel blocks of x that take part
    int Np;        // output channels, padded to 16
    int H, W, nb;
    int mper;      // tiles of 16 blocks per CTA and dj
    int djs;       // dj per CTA: 3, or 1 (blockIdx.y then walks dj)
    int mtiles;    // ceil(3 G / 16)
    int stages;
    float *part;   // [split][dj][mtiles * 128][Np]
    int *flag;
};

__global__ void __launch_bounds__(kWThreads) k_wgrad_blk(const __grid_constant__ WgradBlk a)
{
    extern __shared__ __align__(1024) unsigned char bsm[];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_full[4], s_free[4], s_done;
    __shared__ volatile int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int P = a.W + 2;
    const int m0 = blockIdx.x * a.mper, nm = min(a.mper, a.mtiles - m0);
    const int dj0 = a.djs == 3 ? 0 : blockIdx.y;
    const int g0 = m0 * 16, ng = min(3 * a.G - g0, nm * 16);  // (di, block) entries loaded
    const int ngz = a.Np / 8;
    const uint32_t ncols = blk_cols(a.djs * a.mper * a.Np);
    const int xbytes = a.mper * 16 * kWRun, stage = xbytes + ngz * kWKP * 16;
    const long long per = (a.H * (long long)P + kWKP - 1) / kWKP, total = per * a.nb;
    const int c0 = (int)(total * blockIdx.z / gridDim.z), c1 = (int)(total * (blockIdx.z + 1) / gridDim.z);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc_smem(&s_tmem)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 32) {
        for (int r = 0; r < 4; ++r) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&s_full[r])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&s_free[r])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&s_done)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    const int n = c1 - c0;
    if (warp == 8) {
        // ---- copies: the CTA's rows of x for all its taps, and dz
        bool ok = true;
        int k = 0;
        for (; k < n; ++k) {
            const int st = k % a.stages;
            if (k >= a.stages && lane == 0)
                ok = tc_wait(&s_free[st], (unsigned)((k / a.stages - 1) & 1), a.flag);
            ok = __all_sync(0xffffffffu, ok && !s_fail);
            if (!ok)
                break;
            const int smp = (int)((c0 + k) / per);
            const size_t pos = (size_t)P + (size_t)((c0 + k) - smp * per) * kWKP;  // first position
            if (lane == 0)
                blk_expect(&s_full[st], (unsigned)(ng * kWRun + ngz * kWKP * 16));
            __syncwarp();
            const uint32_t dst = tc_smem(bsm + (size_t)st * stage);
            for (int e = lane; e < ng; e += 32) {
                const int di = (g0 + e) / a.G, g = (g0 + e) - di * a.G;
                // from position pos - 1 + (di - 1) P: the tensors have slack in front
                const uint4 *src = blk_at(a.x, smp, g, pos) + ((long long)(di - 1) * P - 1);
                blk_copy(dst + e * kWRun, src, kWRun, &s_full[st]);
            }
            for (int e = lane; e < ngz; e += 32)
                blk_copy(dst + xbytes + e * kWKP * 16, blk_at(a.dz, smp, e, pos), kWKP * 16, &s_full[st]);
        }
        if (lane == 0) {
            if (!ok)
                s_fail = 1;
            for (int j = k > a.stages ? k - a.stages : 0; j < k; ++j)  // landed before the CTA may leave
                tc_wait(&s_full[j % a.stages], (unsigned)((j / a.stages) & 1), a.flag);
        }
    } else if (warp == 9) {
        // the MMAs (the whole warp in the loops, as in k_conv_blk)
        const uint32_t lead = elect_one();
        const uint32_t idesc = tc_idesc(a.Np) | (1u << 15) | (1u << 16);  // both operands M/N-major
        const uint32_t lo = (128u >> 4) << 16;
        const uint32_t ahi = (uint32_t)(kWRun >> 4) | (1u << 14), bhi = (uint32_t)(kWKP * 16 >> 4) | (1u << 14);
        int st = 0;
        unsigned ph = 0u;
        uint32_t accum = 0u;
        bool ok = true;
        for (int j = 0; j < n; ++j) {
            ok = ok && blk_wait(&s_full[st], ph, a.flag);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t sx = tc_smem(bsm + (size_t)st * stage);
            uint32_t ak = ((sx >> 4) + (uint32_t)dj0) | lo, bd = ((sx + (uint32_t)xbytes) >> 4) | lo;
#pragma unroll 1
            for (int kk = 0; kk < kWKP / 16; ++kk) {  // 16 positions each
#pragma unroll 1
                for (int d = 0; d < a.djs; ++d) {  // a tap's shift: one position
                    uint32_t ad = ak + (uint32_t)d, col = tmem + (uint32_t)(d * a.mper * a.Np);
#pragma unroll 1
                    for (int m = 0; m < nm; ++m) {
                        if (lead)
                            blk_mma(col, ((uint64_t)ahi << 32) | ad, ((uint64_t)bhi << 32) | bd, idesc, accum);
                        ad += 16 * kWRun / 16;
                        col += (uint32_t)a.Np;
                    }
                }
                accum = 1u;
                ak += 256 / 16;
                bd += 256 / 16;
            }
            if (lead)
                blk_commit(&s_free[st]);
            if (++st == a.stages) {
                st = 0;
                ph ^= 1u;
            }
        }
        if (!ok)
            s_fail = 1;
        __threadfence_block();
        if (lead)
            blk_commit(&s_done);
    } else {
        // ---- the sums of this range
        bool ok = tc_wait(&s_done, 0u, a.flag);
        ok = ok && !s_fail && n > 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncwarp();
        const bool all_ok = __all_sync(0xffffffffu, ok);
        const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int row = (warp & 3) * 32 + lane;
        for (int d = 0; d < a.djs; ++d)
            for (int m = 0; m < nm; ++m) {
                float *dst = a.part + ((((size_t)blockIdx.z * 3 + dj0 + d) * a.mtiles + m0 + m) * 128 + row) * a.Np;
                for (int og = warp >> 2; og * 8 < a.Np; og += 2) {
                    float v[1][8] = {{0, 0, 0, 0, 0, 0, 0, 0}};
                    if (all_ok)
                        blk_ld(tl + (uint32_t)((d * a.mper + m) * a.Np + og * 8), v, 0);
                    float4 *q = reinterpret_cast<float4 *>(dst + og * 8);
                    q[0] = make_float4(v[0][0], v[0][1], v[0][2], v[0][3]);
                    q[1] = make_float4(v[0][4], v[0][5], v[0][6], v[0][7]);
                }
            }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
}

// dW[o][c][t] = the pixel ranges' sums in their order (FP64).  A CTA takes one row (t, c)
// and 32 output channels; its 8 warps each add an eighth of the ranges, so that the loads
// of a few ranges, not of all, follow one another.
__global__ void __launch_bounds__(kT) k_wgrad_blk_reduce(const float *__restrict__ part, int splits, int mtiles,
                                                       int G, int Np, int cin, int cout,
                                                       float *__restrict__ dw)
{
    __shared__ double s_sum[kT / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int o = blockIdx.x * 32 + lane, t = blockIdx.y / cin, c = blockIdx.y - t * cin;
    const int di = t / 3, dj = t - di * 3;
    const size_t stride = (size_t)3 * mtiles * 128 * Np;
    double acc = 0.0;
    if (o < cout) {
        const float *src = part + (((size_t)dj * mtiles * 16 + di * G + c / 8) * 8 + c % 8) * Np + o;
        const int s1 = splits * (warp + 1) / (kT / 32);
#pragma unroll 4
        for (int s = splits * warp / (kT / 32); s < s1; ++s)
            acc += (double)__ldg(src + s * stride);
    }
    s_sum[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && o < cout) {
        double v = 0.0;
        for (int k = 0; k < kT / 32; ++k)
            v += s_sum[k][lane];
        dw[((size_t)o * cin + c) * 9 + t] = (float)v;
    }
}

// An FP32 image per sample into channel 0 of a blocked tensor (block 0; the other
// channels stay zero), times inv[n] if given; part: per-CTA FP64 sums of the values
// (the bias gradient of a one-channel conv), or null.  Grid (CTAs, samples).
__global__ void __launch_bounds__(kT) k_image_blk(const float *__restrict__ img, const float *__restrict__ scale,
                                                Blk dst, int H, int W, double *__restrict__ part)
{
    __shared__ double s_red[kT / 32];
    const int n = blockIdx.y, HW = H * W;
    const float inv = scale ? 1.0f / scale[n] : 1.0f;
    double acc = 0.0;
    for (int q = blockIdx.x * kT + threadIdx.x; q < HW; q += gridDim.x * kT) {
        const int y = q / W, x = q - y * W;
        const float v = img[(size_t)n * HW + q];
        *blk_at(dst, n, 0, (size_t)(y + 1) * (W + 2) + x + 1) =
            make_uint4(bf16_bits(scale ? v * inv : v), 0u, 0u, 0u);
        if (part)
            acc += v;
    }
    if (!part)
        return;
    for (int off = 16; off; off >>= 1)
        acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0)
        s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int k = 0; k < kT / 32; ++k)
            v += s_red[k];
        part[(size_t)n * gridDim.x + blockIdx.x] = v;
    }
}

}  // namespace
