// nn_tc.cu -- the 3x3 convolutions and weight gradients of nn_conv.cu on the
// fifth-generation tensor cores (tcgen05), for rows of a multiple of 64
// points: BF16 operands from shared memory, FP32 accumulator in tensor memory
// (TMEM), one thread issuing the MMAs.
//
// Tile: 128 (or 64) consecutive output points of one latitude row (M) x the
// output channels (N = COUT).  Operands use the no-swizzle K-major layout:
// 16-byte rows (8 channels) of consecutive points (or output channels), one
// plane per 8 input channels.  In this layout a longitude tap shift is a
// start-address offset of 16 bytes per point, so the nine taps read the
// staged halo rows directly: for tap (ky, kx) and input channels 16 ks ..
// 16 ks + 15, A starts at row ky, plane 2 ks, point kx, and one
// tcgen05.mma of K = 16 accumulates it.
//
// A block works down strips of up to 8 rows of one tile's column.  Input
// rows sit in a ring of shared-memory slots (the shifted pole rows of the
// input gradient among them), so every input row of a strip is staged once.
// Every mbarrier wait is bounded.
#include <cuda_bf16.h>
#include <cstdint>

#include "nn_internal.h"

namespace nn {

namespace {

constexpr unsigned long long TC_WAIT_NS = 200000000ull;   // longest wait: 0.2 s

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp16(void *s, const void *g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}

__device__ __forceinline__ unsigned long long gtime()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// shared-memory matrix descriptor: start, leading (K) and stride (M/N)
// byte offsets in 16-byte units, descriptor version 1, no swizzle.  In both
// the K-major and the MN-major no-swizzle layouts the leading offset is the
// step between core matrices along K and the stride offset the step along
// M or N.
__device__ __forceinline__ unsigned long long sdesc(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (unsigned long long)((addr & 0x3FFFF) >> 4) | ((unsigned long long)((lbo >> 4) & 0x3FFF) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N and M
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

// one MMA, issued by the lane with one != 0 of a warp that runs together: the
// descriptors are then warp-uniform values
__device__ __forceinline__ void mma_bf16_one(unsigned dtmem, unsigned long long a, unsigned long long b, unsigned id,
                                             unsigned accumulate, unsigned one)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %4, 0;\n setp.ne.u32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate), "r"(one)
        : "memory");
}

__device__ __forceinline__ void mma_commit_one(unsigned mbar, unsigned one)
{
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.u32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar),
        "r"(one)
        : "memory");
}

// one lane of a converged warp: 1 in that lane, 0 in the others
__device__ __forceinline__ unsigned elect_one()
{
    unsigned one;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(one));
    return one;
}

// wait for the mbarrier phase of the given parity; false after TC_WAIT_NS
// (the clock is read every 64 polls)
__device__ __forceinline__ bool mbar_wait(unsigned mbar, unsigned parity)
{
    unsigned long long t0 = 0;
    for (unsigned n = 0;; ++n) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((n & 63) == 0) {
            const unsigned long long t = gtime();
            if (n == 0) t0 = t;
            else if (t - t0 > TC_WAIT_NS) return false;
        }
    }
}

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float (&v)[8])
{
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void tmem_ld16(unsigned taddr, float *v)
{
    unsigned r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned long long *b)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

// 16 of a thread's 32 (8 of 16) values as BF16: the upper half if hi; zero
// where mask (if any) is not positive
template <int N>
__device__ __forceinline__ void store_half(const float (&v)[N], int hi, const __nv_bfloat16 *mask, __nv_bfloat16 *out)
{
#pragma unroll
    for (int k = 0; k < N / 16; ++k) {
        float x[8];
#pragma unroll
        for (int z = 0; z < 8; ++z) x[z] = hi ? v[N / 2 + 8 * k + z] : v[8 * k + z];
        if (mask) {
            const uint4 mq = __ldg((const uint4 *)mask + k);
            const __nv_bfloat16 *mv = (const __nv_bfloat16 *)&mq;
#pragma unroll
            for (int z = 0; z < 8; ++z)
                if (!(__bfloat162float(mv[z]) > 0.f)) x[z] = 0.f;
        }
        __nv_bfloat162 o2[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) o2[z] = __floats2bfloat162_rn(x[2 * z], x[2 * z + 1]);
        ((uint4 *)out)[k] = *(const uint4 *)o2;
    }
}

__host__ __device__ constexpr int tmem_cols(int n) { return n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : (n <= 256 ? 256 : 512))); }

} // namespace

// ---------------------------------------------------------------------------
// forward and input-gradient convolution
// ---------------------------------------------------------------------------
// what the epilogue makes of an output row
enum Epi : int {
    EP_ACT,       // bias, ReLU, BF16
    EP_ACT_POOL,  // the same, and the 2x2 mean of two rows for the next level
    EP_Y,         // the network's output: channel 0 plus bias, FP32
    EP_MASK,      // zero where mask <= 0 (ReLU derivative), BF16
    EP_F32,       // FP32
    EP_UP         // input gradient of [up(coarse), skip]: the first UP_C channels
                  // summed over 2x2 points, zero where the coarse activation is
                  // <= 0, BF16; the others FP32
};
constexpr int UP_C = 64;                    // channels of the coarse level in both concatenations

// ring slots of input rows, as many as fit beside the weights, at most 8
template <int TW, int CIN, int COUT>
struct ConvShape {
    static constexpr int TC_P = TW + 2;                           // staged points of a row (halo)
    static constexpr int KC = CIN / 8;                            // 16-byte channel chunks of a point
    static constexpr size_t WB = (size_t)9 * KC * COUT * 16;      // weights
    static constexpr size_t SLOT = (size_t)KC * TC_P * 16;        // one staged row
    static constexpr int FIT = (int)((215 * 1024 - WB) / SLOT);
    static constexpr int RING = FIT > 8 ? 8 : FIT;
    static constexpr size_t BYTES = WB + RING * SLOT;
    // rows whose copies stay in flight behind the newest one's
    static constexpr int DEPTH = RING >= 6 ? 4 : RING - 2;
    static constexpr unsigned TCOLS = tmem_cols(COUT);            // columns of one accumulator
    // groups of four epilogue warps: with 64 or more channels a row's stores
    // and sums are more than four warps do beside the MMAs
    static constexpr int EG = COUT >= 64 ? 2 : 1;
    static constexpr int THREADS = 128 * EG + 160;                // epilogue, 4 producer warps, 1 MMA warp
    // two blocks per SM where shared memory (with the static part and what the
    // system keeps) and the epilogue's registers allow
    static constexpr int MINB = 2 * (BYTES + 3072) <= 227 * 1024 && COUT <= 32 ? 2 : 1;
};
constexpr int ACCS = 4;                     // accumulators: three rows in progress, one read out

// What bounds it: with one set of 128 threads that staged, issued and read out
// in turn, a 128-point row of c5 (96 -> 32) took 4 us, of which the MMAs need
// 0.9 (each reads a 4 KB A operand from shared memory) and the row's bytes
// 0.6; the rest was one row's copies, MMAs and stores waiting for each other.
// So the three jobs run in warps of their own, handing rows on through
// mbarriers.  Producers copy input rows into a ring (cp.async), several rows
// in flight.  One thread takes an input row as soon as it is there and issues
// everything that reads it: kernel row ky of the weights adds it to output row
// r + 1 - ky, so three output rows are in progress in TMEM, an input row's slot
// is free after its own 9 CIN / 16 MMAs, and the whole ring but one slot holds
// rows to come (which is what 128 input channels need: beside their weights
// only four rows fit).  The epilogue warps read a finished accumulator while
// the next rows run.  A block takes the COUT output channels of blockIdx.y;
// with CS > 0 the first CS input channels come from the coarser level (nearest
// neighbour) and the others from a second field, so the concatenation is never
// stored.  us at 32 samples of 256 x 128, before (with the pooling, the
// concatenation or its adjoint that is now part of the kernel) and now: c1 96,
// 42; c2 59, 31; c4 354, 86; c5 298, 111; c6 84, 38; d6 96, 47; d5 481, 96; d4
// 285, 85; d2 87, 35.  An N = 32 MMA takes 38 ns in c5, about twice its operands'
// shared-memory time: the MMAs bound c4, c5 and d4, the bytes c1, c6 and d6.
template <int TW, int CIN, int CS, int COUT, bool DGRAD, int EPI>
__global__ void __launch_bounds__(ConvShape<TW, CIN, COUT>::THREADS, ConvShape<TW, CIN, COUT>::MINB) k_conv_tc(ConvArgs a, int strip, int *err)
{
    typedef ConvShape<TW, CIN, COUT> S;
    constexpr int KC = S::KC, RING = S::RING, DEPTH = S::DEPTH, SLOT = (int)S::SLOT, TC_P = S::TC_P;
    static_assert(RING >= DEPTH + 2, "a slot is freed once its row, handed over, is done");
    static_assert(COUT % 16 == 0 && ACCS * S::TCOLS <= 512, "");
    constexpr unsigned TCOLS = S::TCOLS;
    constexpr unsigned ID = idesc_bf16(TW, COUT);
    constexpr int EG = S::EG;
    constexpr int CHUNK = EG > 1 || COUT < 32 ? 16 : 32;    // columns read out at once
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *Ws = smem;                       // [9][KC][COUT] x 16 B
    unsigned char *Xs = Ws + S::WB;                 // [slot][KC][TC_P] x 16 B
    __shared__ __align__(8) unsigned long long s_full[RING], s_empty[RING], s_accf[ACCS], s_acce[ACCS], s_done;
    __shared__ unsigned s_tmem;
    __shared__ int s_bad;
    __shared__ float s_bias[COUT];
    const int H = a.H, W = a.W;
    const int nseg = W / TW;
    const int nstrip = (H + strip - 1) / strip;
    const long nunits = (long)a.B * nseg * nstrip;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int n0 = blockIdx.y * COUT, ntot = gridDim.y * COUT;

    if (threadIdx.x == 0) {
        s_bad = 0;
        for (int q = 0; q < RING; ++q) {
            mbar_init(&s_full[q], 128);
            mbar_init(&s_empty[q], 1);
        }
        for (int q = 0; q < ACCS; ++q) {
            mbar_init(&s_accf[q], 1);
            mbar_init(&s_acce[q], 128 * EG);
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(ACCS * TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int q = threadIdx.x; q < 9 * COUT * KC; q += blockDim.x) {
        const int c = q % KC, o = (q / KC) % COUT, tap = q / KC / COUT;
        cp16(Ws + ((size_t)(tap * KC + c) * COUT + o) * 16, a.w + ((size_t)tap * ntot + n0 + o) * CIN + c * 8);
    }
    for (int q = threadIdx.x; q < COUT; q += blockDim.x) s_bias[q] = a.bias ? a.bias[n0 + q] : 0.f;
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    volatile int *bad = &s_bad;
    // a unit is `strip` output rows of one 128-point column of one sample.  Its
    // ring entries, in order: forward, the input rows h0 - 1 .. h1 (beyond a
    // pole, the pole row shifted by half a circle); gradient, the rows among
    // them that exist, after the shifted pole row of the first strip and before
    // that of the last.  Entry numbers run on over the block's units.
    struct Unit { int b, w0, h0, h1, r0, south, north, nent; };
    auto unit_of = [&](long u) {
        Unit q;
        q.w0 = (int)(u % nseg) * TW;
        q.h0 = (int)((u / nseg) % nstrip) * strip;
        q.b = (int)(u / nseg / nstrip);
        q.h1 = min(q.h0 + strip, H);
        q.south = (DGRAD && q.h0 == 0) ? 1 : 0;
        q.north = (DGRAD && q.h1 == H) ? 1 : 0;
        q.r0 = q.h0 - 1 + q.south;                               // first row entry
        q.nent = q.south + (q.h1 - q.north - q.r0 + 1) + q.north;
        return q;
    };

    if (warp >= 4 * EG && warp < 4 * EG + 4) {
        // ---- producers ----
        // a thread's pieces (16 bytes, channel chunk c of point pt) are the same
        // in every row: their places in the slot and in a row are kept
        const int p = threadIdx.x - 128 * EG;
        constexpr int NP = (TC_P * KC + 127) / 128;
        int src[NP], cur_w0 = -1, cur_shift = 0;
        auto place = [&](int w0, int shift) {    // offsets of the pieces in their source rows
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                const int z = p + 128 * k, c = z % KC;
                int ws = w0 - 1 + z / KC + shift;
                if (ws < 0) ws += W;
                else if (ws >= W) ws -= W;
                src[k] = CS > 0 && c < CS / 8 ? (ws >> 1) * CS + c * 8 : ws * (CIN - CS) + (c - CS / 8) * 8;
            }
            cur_w0 = w0;
            cur_shift = shift;
        };
        int e = 0, told = 0;
        auto hand_over = [&](int upto) {         // entries [told, upto) are complete
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (; told < upto; ++told) mbar_arrive(&s_full[told % RING]);
        };
        for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
            const Unit q = unit_of(u);
            for (int k = 0; k < q.nent; ++k, ++e) {
                const int slot = e % RING;
                if (e >= RING && !mbar_wait(smem_u32(&s_empty[slot]), (e / RING - 1) & 1)) { *bad = 1; break; }
                int hr = q.r0 + k - q.south, shift = 0;
                if (DGRAD && (k < q.south || k - q.south > q.h1 - q.north - q.r0)) {
                    hr = k < q.south ? 0 : H - 1;
                    shift = W / 2;
                } else if (hr < 0 || hr >= H) {
                    hr = hr < 0 ? 0 : H - 1;
                    shift = W / 2;
                }
                unsigned char *base = Xs + (size_t)slot * SLOT;
                const __nv_bfloat16 *row = a.x + ((size_t)q.b * H + hr) * W * (CIN - CS);
                const __nv_bfloat16 *crow =
                    CS > 0 ? a.xc + ((size_t)q.b * (H / 2) + hr / 2) * (W / 2) * CS : nullptr;
                if (q.w0 != cur_w0 || shift != cur_shift) place(q.w0, shift);
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const int z = p + 128 * k, c = z % KC;
                    unsigned char *dst = base + (c * TC_P + z / KC) * 16;
                    if (TC_P * KC % 128 != 0 && k == NP - 1 && z >= TC_P * KC) break;
                    cp16(dst, (CS > 0 && c < CS / 8 ? crow : row) + src[k]);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH) : "memory");
                if (e >= DEPTH) hand_over(e + 1 - DEPTH);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        hand_over(e);
    } else if (warp == 4 * EG + 4) {
        // ---- MMAs ----
        // the whole warp runs the role and one lane issues, so that everything
        // but the issue is warp-uniform (a row of c5 took 3.1 us with one
        // thread in a branch of its own)
        {
            const unsigned one = elect_one();
            const unsigned long long A0 = sdesc(smem_u32(Xs), TC_P * 16, 128), B0 = sdesc(smem_u32(Ws), COUT * 16, 128);
            int e = 0, t0 = 0;                      // ring entry; number of the unit's first output row
            for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
                const Unit q = unit_of(u);
                unsigned begun = 0;                 // output rows (bit t % ACCS) that have been added to
                // three taps of kernel row ky: slot's row into output row h
                auto add = [&](int slot, int ky, int h) {
                    const int t = t0 + h - q.h0, buf = t % ACCS;
                    if (!(begun >> buf & 1) && t >= ACCS && !mbar_wait(smem_u32(&s_acce[buf]), (t / ACCS - 1) & 1))
                        return false;
                    if (!(begun >> buf & 1)) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned d = tmem + (unsigned)buf * TCOLS;
                    unsigned acc = begun >> buf & 1;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const unsigned long long ad = A0 + (unsigned)(slot * (SLOT / 16) + kx);
                        const unsigned long long bd = B0 + (unsigned)((ky * 3 + kx) * KC * COUT);
#pragma unroll
                        for (int ks = 0; ks < CIN / 16; ++ks) {
                            mma_bf16_one(d, ad + 2 * ks * TC_P, bd + 2 * ks * COUT, ID, acc, one);
                            acc = 1;
                        }
                    }
                    begun |= 1u << buf;
                    return true;
                };
                auto finish = [&](int h) {          // output row h is complete
                    const int buf = (t0 + h - q.h0) % ACCS;
                    begun &= ~(1u << buf);
                    mma_commit_one(smem_u32(&s_accf[buf]), one);
                };
                for (int k = 0; k < q.nent; ++k, ++e) {
                    const int slot = e % RING;
                    bool ok = mbar_wait(smem_u32(&s_full[slot]), (e / RING) & 1);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // the adjoint of the ghost rows: the pole row collects what
                    // the row beyond it had copied (kernel row 2 at the first
                    // row, 0 at the last)
                    if (DGRAD && k < q.south) {
                        ok = ok && add(slot, 2, 0);
                    } else if (DGRAD && q.north && k == q.nent - 1) {
                        ok = ok && add(slot, 0, H - 1);
                        finish(H - 1);
                    } else {
                        const int r = q.r0 + k - q.south;
                        for (int ky = 2; ky >= 0; --ky) {
                            const int h = r + 1 - ky;
                            if (h >= q.h0 && h < q.h1) ok = ok && add(slot, ky, h);
                        }
                        if (r - 1 >= q.h0) finish(r - 1);
                    }
                    mma_commit_one(smem_u32(&s_empty[slot]), one);
                    if (!ok) { *bad = 1; break; }
                }
                t0 += q.h1 - q.h0;
            }
            // everything issued has completed before TMEM and the barriers go
            mma_commit_one(smem_u32(&s_done), one);
            if (!mbar_wait(smem_u32(&s_done), 0)) *bad = 1;
        }
        __syncwarp();
    } else {
        // ---- epilogue: thread = output point, warp w reads TMEM lanes 32 (w % 4)
        // .. + 31, group w / 4 every EG-th chunk of columns ----
        // (M = 64: output point 16 w + l in lane 32 w + l, l < 16)
        const int eg = warp / 4;
        const bool on = lane < TW / 4;
        int t = 0;
        // pair sums of the even row
        float hold[EPI == EP_ACT_POOL || EPI == EP_UP ? (EPI == EP_UP && COUT > UP_C ? UP_C : COUT) / EG : 1];
        for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
            const Unit q = unit_of(u);
            const int w = q.w0 + (warp & 3) * (TW / 4) + lane % (TW / 4);
            for (int h = q.h0; h < q.h1; ++h, ++t) {
                const int buf = t % ACCS;
                if (!mbar_wait(smem_u32(&s_accf[buf]), (t / ACCS) & 1)) *bad = 1;
                if (__any_sync(0xffffffffu, *bad)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned trow = tmem + (unsigned)buf * TCOLS + ((unsigned)((warp & 3) * 32) << 16);
                const size_t pix = ((size_t)q.b * H + h) * W + w;
                const size_t cpix = ((size_t)q.b * (H / 2) + h / 2) * (W / 2) + w / 2;
#pragma unroll
                for (int ci = 0; ci < COUT / CHUNK; ci += EG) {
                    const int c0 = (ci + eg) * CHUNK, hc = ci / EG * CHUNK;
                    float v[CHUNK];
#pragma unroll
                    for (int k = 0; k < CHUNK; k += 16) {
                        if (EPI == EP_Y) { tmem_ld8(trow, *(float (*)[8])v); break; }
                        tmem_ld16(trow + c0 + k, v + k);
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (ci + EG >= COUT / CHUNK) {
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        mbar_arrive(&s_acce[buf]);
                    }
                    if constexpr (EPI == EP_Y) {
                        if (on) a.yf[pix] = v[0] + s_bias[0];
                    } else if constexpr (EPI == EP_F32) {
                        float4 *o = (float4 *)(a.yf + pix * ntot + n0 + c0);
#pragma unroll
                        for (int k = 0; k < CHUNK / 4; ++k)
                            if (on) o[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                    } else if constexpr (EPI == EP_UP) {
                        const int col = n0 + c0;
                        if (ci * CHUNK >= UP_C || col >= UP_C) {
                            float4 *o = (float4 *)(a.yf + pix * (ntot - UP_C) + col - UP_C);
#pragma unroll
                            for (int k = 0; k < CHUNK / 4; ++k)
                                if (on) o[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                        } else {
#pragma unroll
                            for (int k = 0; k < CHUNK; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1);
                            if ((h & 1) == 0) {
#pragma unroll
                                for (int k = 0; k < CHUNK; ++k) hold[hc + k] = v[k];
                            } else {
                                // each point of the pair writes half of the channels
#pragma unroll
                                for (int k = 0; k < CHUNK; ++k) v[k] = hold[hc + k] + v[k];
                                const size_t at = cpix * UP_C + col + (lane & 1) * (CHUNK / 2);
                                if (on) store_half(v, lane & 1, a.mask + at, a.y + at);
                            }
                        }
                    } else {
                        if constexpr (EPI == EP_MASK) {
                            const uint4 *m = (const uint4 *)(a.mask + pix * ntot + n0 + c0);
#pragma unroll
                            for (int k = 0; k < CHUNK / 8; ++k) {
                                const uint4 mq = on ? __ldg(m + k) : make_uint4(0, 0, 0, 0);
                                const __nv_bfloat16 *mv = (const __nv_bfloat16 *)&mq;
#pragma unroll
                                for (int z = 0; z < 8; ++z)
                                    if (!(__bfloat162float(mv[z]) > 0.f)) v[8 * k + z] = 0.f;
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < CHUNK; ++k) v[k] = fmaxf(v[k] + s_bias[c0 + k], 0.f);
                        }
                        uint4 *o = (uint4 *)(a.y + pix * ntot + n0 + c0);
#pragma unroll
                        for (int k = 0; k < CHUNK / 8; ++k) {
                            __nv_bfloat162 o2[4];
#pragma unroll
                            for (int z = 0; z < 4; ++z) o2[z] = __floats2bfloat162_rn(v[8 * k + 2 * z], v[8 * k + 2 * z + 1]);
                            if (on) o[k] = *(const uint4 *)o2;
                        }
                        if constexpr (EPI == EP_ACT_POOL) {
                            // the mean is of the activations as stored
#pragma unroll
                            for (int k = 0; k < CHUNK; ++k) {
                                v[k] = __bfloat162float(__float2bfloat16_rn(v[k]));
                                v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1);
                            }
                            if ((h & 1) == 0) {
#pragma unroll
                                for (int k = 0; k < CHUNK; ++k) hold[hc + k] = v[k];
                            } else {
#pragma unroll
                                for (int k = 0; k < CHUNK; ++k) v[k] = 0.25f * (hold[hc + k] + v[k]);
                                const size_t at = cpix * ntot + n0 + c0 + (lane & 1) * (CHUNK / 2);
                                if (on) store_half(v, lane & 1, nullptr, a.yp + at);
                            }
                        }
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (s_bad && threadIdx.x == 0) atomicExch(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ACCS * TCOLS)
                     : "memory");
}

template <int TW, int CIN, int CS, int COUT, bool DGRAD, int EPI>
static cudaError_t conv_tw_t(const ConvArgs &a, int nsplit, int sms, int *err, cudaStream_t s)
{
    typedef ConvShape<TW, CIN, COUT> S;
    const size_t smem = S::BYTES;
    int bps = 0;
    cudaError_t e = occupancy_once<k_conv_tc<TW, CIN, CS, COUT, DGRAD, EPI>>(S::THREADS, smem, &bps);
    if (e != cudaSuccess) return e;
    if (bps < 1) return cudaErrorInvalidConfiguration;
    // (the occupancy query answers 1 for every kernel that allocates TMEM)
    bps = S::MINB;
    static_assert(S::MINB * ACCS * S::TCOLS <= 512, "");
    // strips of 8 rows (10 input rows each), shorter while blocks would be idle
    const long cap = (long)bps * sms / nsplit > 0 ? (long)bps * sms / nsplit : 1;
    int strip = 8;
    auto units = [&](int st) { return (long)a.B * (a.W / TW) * ((a.H + st - 1) / st); };
    while (strip > 2 && units(strip) < cap) strip /= 2;
    const long n = units(strip);
    k_conv_tc<TW, CIN, CS, COUT, DGRAD, EPI><<<dim3((unsigned)(n < cap ? n : cap), nsplit), S::THREADS, smem, s>>>(a, strip, err);
    return cudaGetLastError();
}

template <int CIN, int CS, int COUT, bool DGRAD, int EPI>
static cudaError_t conv_tc_t(const ConvArgs &a, int nsplit, int sms, int *err, cudaStream_t s)
{
    return a.W % 128 == 0 ? conv_tw_t<128, CIN, CS, COUT, DGRAD, EPI>(a, nsplit, sms, err, s)
                          : conv_tw_t<64, CIN, CS, COUT, DGRAD, EPI>(a, nsplit, sms, err, s);
}

cudaError_t launch_conv_tc(ConvStep step, const ConvArgs &a, int sms, int *err, cudaStream_t s)
{
    switch (step) {
    case CONV_C1: return conv_tc_t<16, 0, 32, false, EP_ACT_POOL>(a, 1, sms, err, s);
    case CONV_C2: return conv_tc_t<32, 0, 64, false, EP_ACT_POOL>(a, 1, sms, err, s);
    case CONV_C3: return conv_tc_t<64, 0, 64, false, EP_ACT>(a, 1, sms, err, s);
    // 128 input channels: 147 KB of weights for 64 outputs, so 32 a block
    case CONV_C4: return conv_tc_t<128, 64, 32, false, EP_ACT>(a, 2, sms, err, s);
    case CONV_C5: return conv_tc_t<96, 64, 32, false, EP_ACT>(a, 1, sms, err, s);
    case CONV_C6: return conv_tc_t<32, 0, 16, false, EP_Y>(a, 1, sms, err, s);
    case CONV_D6: return conv_tc_t<16, 0, 32, true, EP_MASK>(a, 1, sms, err, s);
    case CONV_D5: return conv_tc_t<32, 0, 96, true, EP_UP>(a, 1, sms, err, s);
    case CONV_D4: return conv_tc_t<64, 0, 64, true, EP_UP>(a, 2, sms, err, s);
    case CONV_D3: return conv_tc_t<64, 0, 64, true, EP_F32>(a, 1, sms, err, s);
    case CONV_D2: return conv_tc_t<64, 0, 32, true, EP_F32>(a, 1, sms, err, s);
    }
    return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// weight gradient
// ---------------------------------------------------------------------------
// dW[ky][kx][co][ci] = sum over points p of x[row h + ky - 1][p] g[row h][p - kx + 1][co]
// with the forward convolution's sphere halo on x (beyond a pole the pole row
// shifted by half a circle; periodic in longitude).  As a GEMM D[m][n] = sum_k
// A[m][k] B[n][k]: m = input channels of one or more consecutive input rows
// (M = 128), n = co (N = COUT) for each kx, k = points.  Both operands sit in
// shared memory one plane per 8 channels, a 16-byte row per point: the MN-major
// no-swizzle layout (8 consecutive MN elements per 16-byte row, 8 rows per K
// core matrix), read with the transpose bits of the instruction descriptor.
// The longitude shift of a tap is a 16-byte start offset, and it is on g, the
// smaller operand: an A read that does not start on a core matrix costs twice.
//
// Input rows sit in a ring of slots that follow one another in memory, so that
// with fewer than 128 input channels one A operand spans the rows of several
// ky: all three with 16 or 32 channels, two with 64 (the rows of D beyond the
// third are never read out).  The first slots are kept twice, behind the last
// one, for rows that wrap.
//
// What bounds it: one set of 128 threads that staged, issued and waited in turn
// took 4.8 us per 128-point row of c5 (its 72 MMAs need about 2), and mma.sync
// with nothing in flight 180 us for the padded c6.  The jobs run in warps of
// their own, as in k_conv_tc: producers stage a step (an input row and a
// gradient row) at a time, several in flight; one warp issues a step's MMAs into
// the 3 COUT columns of each group of rows, accumulated over all of the block's
// steps; the four warps that read the result out at the end add up the bias
// gradient meanwhile.  us at 32 samples of 256 x 128, before and now:
// c1 143, 59; c2 56, 29; c4 178, 112; c5 260, 123; c6 180, 50.
template <int TW, int CIN, int COUT>
struct WgShape {
    static constexpr int TC_TW = TW, TC_P = TW + 2;                // points of an input row, of a gradient row (halo)
    static constexpr int KC = CIN / 8, GC = COUT / 8;
    static constexpr int RPG = 128 / CIN > 3 ? 3 : 128 / CIN;      // kernel rows of one A operand
    static constexpr int NG = (3 + RPG - 1) / RPG;                 // A operands per step
    static constexpr int MIR = RPG - 1;                            // slots kept twice
    static constexpr size_t XSLOT = (size_t)KC * TC_TW * 16;
    static constexpr size_t GSLOT = (size_t)GC * TC_P * 16;
    static constexpr int GR = 5;                                   // gradient-row slots
    // the last slot's A operand reads 16 planes
    static constexpr size_t PAD = (size_t)(16 - KC) * TC_TW * 16;
    static constexpr int FIT = (int)((222 * 1024 - GR * GSLOT - PAD) / XSLOT) - MIR;
    static constexpr int XR = FIT > 8 ? 8 : FIT;                   // input-row slots
    static constexpr size_t XBYTES = (XR + MIR) * XSLOT + PAD;
    static constexpr size_t BYTES = XBYTES + GR * GSLOT;
    static constexpr int DEPTH = 2;                                // steps in flight behind the newest one
    static constexpr int NCOL = NG * 3 * COUT;
};

template <int TW, int CIN, int CS, int COUT>
__global__ void __launch_bounds__(288) k_wgrad_tc(WgradArgs a, int strip, int *err)
{
    typedef WgShape<TW, CIN, COUT> S;
    constexpr int KC = S::KC, GC = S::GC, XR = S::XR, GR = S::GR, DEPTH = S::DEPTH, TC_TW = TW, TC_P = S::TC_P;
    static_assert(XR >= 4 && S::NCOL <= 512 && DEPTH < GR, "");
    constexpr unsigned TCOLS = tmem_cols(S::NCOL);
    // BF16 A and B, both MN-major (transpose bits 15 and 16), FP32 accumulator
    constexpr unsigned ID = idesc_bf16(128, COUT) | (1u << 15) | (1u << 16);
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *Xs = smem, *Gs = smem + S::XBYTES;
    __shared__ __align__(8) unsigned long long s_full[GR], s_empty[GR], s_done;
    __shared__ unsigned s_tmem;
    __shared__ int s_bad;
    const int H = a.H, W = a.W;
    const int nseg = W / TC_TW, nstrip = (H + strip - 1) / strip;
    const long nunits = (long)a.B * nseg * nstrip;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int n0 = blockIdx.y * COUT, ntot = gridDim.y * COUT;

    if (threadIdx.x == 0) {
        s_bad = 0;
        for (int q = 0; q < GR; ++q) {
            mbar_init(&s_full[q], 128);
            mbar_init(&s_empty[q], 5);      // the step's MMAs, and the four bias warps
        }
        mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TCOLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    volatile int *bad = &s_bad;
    struct Unit { int b, w0, h0, h1; };
    auto unit_of = [&](long u) {
        Unit q;
        q.w0 = (int)(u % nseg) * TW;
        q.h0 = (int)((u / nseg) % nstrip) * strip;
        q.b = (int)(u / nseg / nstrip);
        q.h1 = min(q.h0 + strip, H);
        return q;
    };
    // step n of the block is one gradient row; input rows h0 - 1 .. h1 of a unit
    // are entries of their ring, numbered on over the units, entry i of a unit
    // last read by its step min(i, h1 - h0 - 1)

    if (warp >= 4 && warp < 8) {
        // ---- producers ----
        const int p = threadIdx.x - 128;
        constexpr int NX = TW * KC / 128, NGP = (TC_P * GC + 127) / 128;      // pieces per thread of a row
        int n = 0, told = 0, done = 0;           // steps staged, handed over, known to be complete
        auto hand_over = [&](int upto) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            for (; told < upto; ++told) mbar_arrive(&s_full[told % GR]);
        };
        auto wait_step = [&](int step) {         // step `step` is complete
            if (step >= told) {                  // it may wait for copies in flight
                asm volatile("cp.async.wait_all;" ::: "memory");
                hand_over(n);
            }
            for (; done <= step; ++done)
                if (!mbar_wait(smem_u32(&s_empty[done % GR]), (done / GR) & 1)) return false;
            return true;
        };
        // a thread's pieces (16 bytes, channel chunk c of point pt) are the same
        // in every row: their offsets in a row are kept
        int src[NX], gsrc[NGP], cur_w0 = -1, cur_shift = -1;
        int e = 0, last[XR];                     // next entry; last step that reads each slot's row
#pragma unroll
        for (int q = 0; q < XR; ++q) last[q] = -1;
        for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
            const Unit q = unit_of(u);
            const int rows = q.h1 - q.h0, n_first = n;
            bool ok = true;
            for (int i = 0; i < rows && ok; ++i) {
                if (n >= GR) ok = ok && wait_step(n - GR);
                for (int r = i == 0 ? 0 : i + 2; r <= i + 2; ++r, ++e) {
                    const int slot = e % XR;
                    int before = -1;
#pragma unroll
                    for (int k = 0; k < XR; ++k)
                        if (k == slot) {
                            before = last[k];
                            last[k] = n_first + min(r, rows - 1);
                        }
                    ok = ok && (before < 0 || wait_step(before));
                    int hr = q.h0 - 1 + r, shift = 0;
                    if (hr < 0 || hr >= H) {
                        hr = hr < 0 ? 0 : H - 1;
                        shift = W / 2;
                    }
                    const __nv_bfloat16 *row = a.x + ((size_t)q.b * H + hr) * W * (CIN - CS);
                    const __nv_bfloat16 *crow =
                        CS > 0 ? a.xc + ((size_t)q.b * (H / 2) + hr / 2) * (W / 2) * CS : nullptr;
                    unsigned char *base = Xs + (size_t)slot * S::XSLOT;
                    if (q.w0 != cur_w0 || shift != cur_shift) {
#pragma unroll
                        for (int k = 0; k < NX; ++k) {
                            const int z = p + 128 * k, c = z % KC;
                            int ws = q.w0 + z / KC + shift;
                            if (ws >= W) ws -= W;
                            src[k] = CS > 0 && c < CS / 8 ? (ws >> 1) * CS + c * 8 : ws * (CIN - CS) + (c - CS / 8) * 8;
                        }
#pragma unroll
                        for (int k = 0; k < NGP; ++k) {
                            const int z = p + 128 * k;
                            int ws = q.w0 - 1 + z / GC;
                            if (ws < 0) ws += W;
                            else if (ws >= W) ws -= W;
                            gsrc[k] = ws * ntot + z % GC * 8;
                        }
                        cur_w0 = q.w0;
                        cur_shift = shift;
                    }
#pragma unroll
                    for (int k = 0; k < NX; ++k) {
                        const int z = p + 128 * k, c = z % KC;
                        const __nv_bfloat16 *sp = (CS > 0 && c < CS / 8 ? crow : row) + src[k];
                        unsigned char *dst = base + (c * TC_TW + z / KC) * 16;
                        cp16(dst, sp);
                        if (slot < S::MIR) cp16(dst + XR * S::XSLOT, sp);
                    }
                }
                const __nv_bfloat16 *grow = a.g + ((size_t)q.b * H + q.h0 + i) * W * ntot + n0;
                unsigned char *gb = Gs + (size_t)(n % GR) * S::GSLOT;
#pragma unroll
                for (int k = 0; k < NGP; ++k) {
                    const int z = p + 128 * k;
                    if (z >= TC_P * GC) break;
                    cp16(gb + (z % GC * TC_P + z / GC) * 16, grow + gsrc[k]);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                ++n;
                asm volatile("cp.async.wait_group %0;" ::"n"(DEPTH) : "memory");
                if (n - DEPTH > told) hand_over(n - DEPTH);
            }
            if (!ok) *bad = 1;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        hand_over(n);
    } else if (warp == 8) {
        // ---- MMAs: the whole warp runs the role, one lane issues ----
        const unsigned one = elect_one();
        // the leading offset steps along K (8 points, 128 bytes), the stride
        // offset along MN (one plane)
        const unsigned long long A0 = sdesc(smem_u32(Xs), 128, TC_TW * 16), B0 = sdesc(smem_u32(Gs), 128, TC_P * 16);
        int n = 0, e0 = 0;
        unsigned acc = 0;
        for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
            const Unit q = unit_of(u);
            for (int i = 0; i < q.h1 - q.h0; ++i, ++n) {
                if (!mbar_wait(smem_u32(&s_full[n % GR]), (n / GR) & 1)) { *bad = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned long long gd = B0 + (unsigned)(n % GR) * (unsigned)(S::GSLOT / 16);
#pragma unroll
                for (int gq = 0; gq < S::NG; ++gq) {
                    const int slot = (e0 + i + gq * S::RPG) % XR;
                    const unsigned long long xd = A0 + (unsigned)slot * (unsigned)(S::XSLOT / 16);
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                        for (int ks = 0; ks < TC_TW / 16; ++ks)
                            mma_bf16_one(tmem + (unsigned)((gq * 3 + kx) * COUT), xd + ks * 16, gd + (ks * 16 + 2 - kx),
                                         ID, acc | (unsigned)ks, one);
                }
                mma_commit_one(smem_u32(&s_empty[n % GR]), one);
                acc = 1;
            }
            e0 += q.h1 - q.h0 + 2;
        }
        mma_commit_one(smem_u32(&s_done), one);
        if (!mbar_wait(smem_u32(&s_done), 0)) *bad = 1;
    } else {
        // ---- bias gradient: thread t adds channel t % COUT over every
        // (128 / COUT)-th point of the step's row ----
        constexpr int NPART = 128 / COUT;
        const int co = threadIdx.x % COUT, p0 = threadIdx.x / COUT;
        float bsum = 0.f;
        int n = 0;
        for (long u = blockIdx.x; u < nunits && !*bad; u += gridDim.x) {
            const Unit q = unit_of(u);
            for (int i = 0; i < q.h1 - q.h0; ++i, ++n) {
                if (!mbar_wait(smem_u32(&s_full[n % GR]), (n / GR) & 1)) *bad = 1;
                if (__any_sync(0xffffffffu, *bad)) break;
                const __nv_bfloat16 *gs =
                    (const __nv_bfloat16 *)(Gs + (size_t)(n % GR) * S::GSLOT + (size_t)(co / 8 * TC_P + 1) * 16) + co % 8;
#pragma unroll 8
                for (int k = p0; k < TC_TW; k += NPART) bsum += __bfloat162float(gs[k * 8]);
                __syncwarp();
                if (lane == 0) mbar_arrive(&s_empty[n % GR]);
            }
        }
        if (a.db && !*bad) atomicAdd(a.db + n0 + co, bsum);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!s_bad && warp < 4) {
        // lanes = (kernel row of the group, input channel), columns = (group, kx, co)
        const int m = warp * 32 + lane, kr = m / CIN, ci = m % CIN;
        const unsigned trow = tmem + ((unsigned)(warp * 32) << 16);
#pragma unroll 2
        for (int c0 = 0; c0 < S::NCOL; c0 += 16) {
            float v[16];
            tmem_ld16(trow + c0, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int grp = c0 / (3 * COUT), kx = c0 / COUT % 3, co = n0 + c0 % COUT;
            const int ky = grp * S::RPG + kr;
            if (kr < S::RPG && ky < 3) {
                float *dw = a.dw + ((size_t)(ky * 3 + kx) * ntot + co) * CIN + ci;
#pragma unroll
                for (int k = 0; k < 16; ++k) atomicAdd(dw + (size_t)k * CIN, v[k]);
            }
        }
    }
    if (s_bad && threadIdx.x == 0) atomicExch(err, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
}

template <int TW, int CIN, int CS, int COUT>
static cudaError_t wgrad_tw_t(const WgradArgs &a, int nsplit, int sms, int *err, cudaStream_t s)
{
    const size_t smem = WgShape<TW, CIN, COUT>::BYTES;
    int bps = 0;
    cudaError_t e = occupancy_once<k_wgrad_tc<TW, CIN, CS, COUT>>(288, smem, &bps);
    if (e != cudaSuccess) return e;
    if (bps < 1) return cudaErrorInvalidConfiguration;
    // one block per SM; strips of 8 rows, shorter while blocks would be idle
    const long cap = sms / nsplit > 0 ? sms / nsplit : 1;
    int strip = 8;
    auto units = [&](int st) { return (long)a.B * (a.W / TW) * ((a.H + st - 1) / st); };
    while (strip > 2 && units(strip) < cap) strip /= 2;
    const long n = units(strip);
    k_wgrad_tc<TW, CIN, CS, COUT><<<dim3((unsigned)(n < cap ? n : cap), nsplit), 288, smem, s>>>(a, strip, err);
    return cudaGetLastError();
}

template <int CIN, int CS, int COUT>
static cudaError_t wgrad_tc_t(const WgradArgs &a, int nsplit, int sms, int *err, cudaStream_t s)
{
    return a.W % 128 == 0 ? wgrad_tw_t<128, CIN, CS, COUT>(a, nsplit, sms, err, s)
                          : wgrad_tw_t<64, CIN, CS, COUT>(a, nsplit, sms, err, s);
}

cudaError_t launch_wgrad_tc(int cin, int cout, const WgradArgs &a, int sms, int *err, cudaStream_t s)
{
    if (cin == 16 && cout == 32) return wgrad_tc_t<16, 0, 32>(a, 1, sms, err, s);
    if (cin == 32 && cout == 64) return wgrad_tc_t<32, 0, 64>(a, 1, sms, err, s);
    if (cin == 64 && cout == 64) return wgrad_tc_t<64, 0, 64>(a, 1, sms, err, s);
    // 9 x 64 accumulator columns are more than TMEM has: 32 outputs a block
    if (cin == 128 && cout == 64) return wgrad_tc_t<128, 64, 32>(a, 2, sms, err, s);
    if (cin == 96 && cout == 32) return wgrad_tc_t<96, 64, 32>(a, 1, sms, err, s);
    if (cin == 32 && cout == 16) return wgrad_tc_t<32, 0, 16>(a, 1, sms, err, s);
    return cudaErrorInvalidValue;
}

} // namespace nn
