// 8-bit weights as integers on the 5th-generation tensor cores: the sparse FC on signed 8-bit codes with tcgen05.mma kind::i8.
//
// The codes are integers, so they go into the tensor core as they lie in memory: the 128 columns of a tile are the M rows of the
// MMA, and a TMA box of 128 channels with 128-byte swizzle is its operand (MN-major).  The activations become integers too: the
// pruned and scaled values of a batch row are written as 45-bit fixed point under a common exponent, that of the largest one
// among the rank's channels - three limbs of 15 bits, each of them two signed 8-bit digits - and the six digits are the N columns of the
// MMA (digit x BR + row).  Products and sums are exact 32-bit integers in one accumulator, read once at the end.  So a weight costs no
// instruction at all, where the mma.sync kernel (scap_fc_qm.cu) spends 1.5 on its conversion to bf16, and an activation is prepared
// once per CTA instead of once per warp.
//
//   grid = (128-column tiles, S), cluster (1, S, 1), 384 threads, two CTAs per SM; a rank takes a contiguous range of blocks of
//   128 channels; one or two blocks are a stage of the ring
//   warp 0      boxes and MMAs (the whole warp runs the loop, one lane issues)
//   warps 1-11  activations: a unit is a block's 128 channels of four batch rows, a lane has four channels of each row.  First the
//               largest value of every row (the warp keeps the values of its first units in registers), then the digits
//   warps 4-7   at the end: a thread per column reads the accumulator
//
// Precision: no bit of a value is rounded away.  The 24 bits of a value down to 2^-20 of its row's largest one in the rank all lie in its
// digits.  A kept value below that, or one that is not finite, has no digits: its row is marked, and value x code of those channels is
// added by itself at the end, in binary64.  (Four digits under the same exponent cut every value below 2^-6 of the largest: with one
// activation 10^4 times the others the columns that do not use it were 5e-6 off.)  The sum of a rank is put together from its digits
// in binary32, a rounding per limb and one between two limbs.
//
// What bounds it: K = 11008, N = 4096, half pruned, weights from DRAM, us per call, mma.sync kernel -> this one: 3 rows
// 18.1 -> 12.3, 8 rows 23.8 -> 14.6, 16 rows 41.0 -> 19.4 (the 45 MB of codes take 6.9 at copy speed).  The first MMA starts 3 - 4 us
// into the call: activations through L2 (1 us under the weight stream), the pass for the exponents, the digits - code that all 24
// warps of an SM run at once, bound by instruction issue - while the ring has been full for two of them.  So a limb comes off a value by
// additions and multiply-adds, where a conversion to an integer takes four issue slots, and whether a value lies below the digits' window is
// asked only where the threshold and the scales do not rule it out (16 rows 20.1 -> 19.4).  Six digits then cost what four by
// conversion did in a long layer (3 / 8 / 11 / 16 rows 12.5 / 14.9 / 17.7 / 20.3 -> 12.3 / 14.6 / 15.7 / 19.4) and more in a short one (K = 4096, four
// blocks per rank, 7.0 / 8.0 / 9.3 / 10.1 -> 7.2 / 8.2 / 9.7 / 10.7).  Values below the window cost time at the end (dense, 8 rows: none 14.6, one
// in 10^5 17.5, a tenth 74, nearly all 330).
// Tried and slower: an exponent per block and an accumulator per block or two, so that the first MMA does not
// wait for a pass over all activations (8 rows 15.4 - 16.3, 16 rows 21.5 - 30.6: reading 11 accumulators costs more than the pass);
// 256 threads (15.4); 4-bit codes the same way, the nibbles separated in shared memory (11008 x 4096, one row 15.4 - 27 against 13.0:
// half the bytes per stage, and an accumulator read per scale group).
// Every wait is bounded (as in scap_fc_tc.cu): one that runs out sets the status word, the CTA stops issuing work, still passes
// its barriers, waits for the copies and MMAs under way and frees its TMEM.
#include <string.h>

#include <type_traits>

#include "scap_qm.cuh"
#include "scap_tc.cuh"

namespace scap {

constexpr int I8_TN = 128;        // columns per CTA
constexpr int I8_KB = 128;        // channels per block (a box, a unit of activations)
constexpr int I8_THREADS = 384;
constexpr int I8_WARPS = I8_THREADS / 32;
constexpr int I8_PREP = I8_WARPS - 1;         // warps that prepare activations
constexpr int I8_KEEP = 2;        // units whose values a warp keeps between the two passes
static_assert(I8_KEEP == 2, "the first pass asks for two units at once");
constexpr int I8_BOX = I8_KB * I8_TN;         // 16 KB
constexpr int I8_ND = 6;          // digits of an activation
// BR = batch rows of the instantiation (4, 8 or 16).  Two blocks are a stage: eight MMAs of 32 channels per round of waits.  (One with
// sixteen rows, whose activations take half of the shared memory otherwise.)
__host__ __device__ constexpr int i8_bps(int BR) { return BR == 16 ? 1 : 2; }
// 16 channels of the activation operand: 6 BR rows of 16 bytes, and 16 bytes more, so that the chunks of a warp's stores start in different banks
__host__ __device__ constexpr int i8_chunk(int BR) { return I8_ND * BR * 16 + 16; }
__host__ __device__ constexpr int i8_xbytes(int BR) { return i8_bps(BR) * I8_KB / 16 * i8_chunk(BR); }
__host__ __device__ constexpr int i8_ncols(int BR) { return (I8_ND * BR + 15) / 16 * 16; }  // N of the MMA (four rows: eight more, whose sums nobody reads)
__host__ __device__ constexpr int i8_tcols(int BR) { return i8_ncols(BR) <= 32 ? 32 : i8_ncols(BR) <= 64 ? 64 : 128; }
__host__ __device__ constexpr int i8_nw(int BR) { return BR == 16 ? 4 : 5; }  // blocks of weights in the ring
__host__ __device__ constexpr int i8_nx(int BR) { return BR == 4 ? 4 : BR == 8 ? 2 : 3; }  // stages of activations
// Barriers that say that a stage has been multiplied.  At least as many as there are slots, and as lie between two units of a warp (11
// units go round; one, two, or three and four per block): a warp that waits for a stage then knows that the one before on the same
// barrier is done, and the one after cannot be (it needs this warp's own unit) - a parity only tells neighbours apart.
__host__ __device__ constexpr int i8_ne(int BR) { return BR == 4 ? 6 : BR == 8 ? 3 : 4; }
constexpr int i8_apart(int ups, int bps) { return ((I8_PREP + ups - 1) / ups + bps - 1) / bps; }  // stages between two units of a warp, at most
static_assert(i8_apart(1, i8_bps(4)) <= i8_ne(4) && i8_apart(2, i8_bps(8)) <= i8_ne(8) && i8_apart(3, i8_bps(16)) <= i8_ne(16) && i8_apart(4, i8_bps(16)) <= i8_ne(16) &&
                  i8_nx(4) <= i8_ne(4) && i8_nx(8) <= i8_ne(8) && i8_nx(16) <= i8_ne(16), "barriers of the stages of activations");
// What the host works out once instead of every warp of every CTA: the code before the first MMA runs on all warps of an SM at the same
// moment and is bound by instruction issue (a division costs a warp as much as the activations of a row).
struct I8Args {
    FcArgs f;
    int blocks, extra;  // blocks per rank; the first `extra` ranks have one more
    int per;            // columns a rank finishes (the last rank may own fewer)
    uint32_t per_inv;   // ceil(2^20 / per): (i * per_inv) >> 20 = i / per for i < 2048
};
struct I8Misc {
    unsigned long long wfull[5], wempty[5];  // a block of weights has landed / has been multiplied
    unsigned long long xfull[4], xempty[6];  // activations of a stage are written (per slot) / have been multiplied (stage modulo i8_ne)
    unsigned long long done, recv;
    uint32_t tmem_base;
    int abort;
    uint32_t top[16], fin[16];  // pattern of a row's largest magnitude; of the largest finite one
    uint32_t apart;             // rows with a value too small for the digits
    uint32_t scale;             // pattern of the rank's smallest scale magnitude
};
struct I8Entry {
    float v;
    int k;
};
struct I8Apart {  // in the ring, when the stream is done
    float sum[16][I8_TN];             // per row and column: the channels without digits
    double part[I8_THREADS / I8_TN][I8_TN];
    int count[I8_WARPS];
    I8Entry entry[I8_WARPS][I8_KB];   // a warp's list
};
static_assert(sizeof(I8Apart) <= i8_nw(16) * I8_BOX, "it must fit in the ring");
__host__ __device__ constexpr int i8_off_x(int BR) { return i8_nw(BR) * I8_BOX; }
__host__ __device__ constexpr int i8_off_gather(int BR) { return i8_off_x(BR) + i8_nx(BR) * i8_xbytes(BR); }
__host__ __device__ constexpr int i8_off_misc(int BR) { return i8_off_gather(BR) + BR * (I8_TN + 16) * 4; }
__host__ __device__ constexpr int i8_smem(int BR) { return i8_off_misc(BR) + (int)sizeof(I8Misc) + 1024; }
static_assert(2 * (i8_smem(4) + 1024) <= 233472 && 2 * (i8_smem(8) + 1024) <= 233472 && 2 * (i8_smem(16) + 1024) <= 233472,
              "two CTAs must fit in the shared memory of an SM");

__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(0u)
        : "memory");
}
// Predicated 8-byte activation load through L2 (zeros where off).
__device__ __forceinline__ uint2 ld_act8_if(const void *p, bool on) {
    uint2 v;
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %3, 0; mov.u32 %0, 0; mov.u32 %1, 0; @q ld.global.cg.v2.u32 {%0,%1}, [%2]; }"
                 : "=r"(v.x), "=r"(v.y) : "l"(p), "r"((unsigned)on) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_act8(const void *p) {
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_act16u(const void *p) {
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
// A bounded wait that sleeps in the barrier instead of polling (after a first look); `limit` in tries.
__device__ __forceinline__ bool i8_wait(unsigned long long *bar, uint32_t parity, int code, volatile int *abort_flag, uint32_t limit, int *status) {
    for (uint32_t i = 0; i < limit; ++i) {
        if (i == 0 ? mbar_test(bar, parity) : mbarrier_try_wait(smem_u32(bar), parity)) return true;
        if (*abort_flag) return false;
    }
    if (status) atomicCAS(status, 0, code);
    *abort_flag = 1;
    return false;
}

__device__ __forceinline__ uint32_t i8_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t i8_top(const float (&v)[4]) { return max(max(i8_bits(v[0]), i8_bits(v[1])), max(i8_bits(v[2]), i8_bits(v[3]))); }
// Fixed point under the exponent e of `top`: |v| < 2^(e - 126), so times 2^(140 - e) it is below 2^14, the most that the first limb
// takes.  Three limbs then hold multiples of 2^(e - 170): all bits of a value from 2^(e - 147) on.
__device__ __forceinline__ int i8_shift(uint32_t top) { return min(140 - (int)(top >> 23), 126); }
__device__ __forceinline__ float i8_pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }
__device__ __forceinline__ float i8_least(int shift) { return i8_pow2(max(-7 - shift, -126)); }
// A value that gets no digits (`least` of its row; dropped channels are zeros and have digits).
__device__ __forceinline__ bool i8_is_apart(float v, float least) { return (fabsf(v) < least && v != 0.0f) || i8_bits(v) >= 0x7f800000u; }

// Sums of value x code over the channels without digits, for the rows that have some, to `out`.  The whole CTA, when the ring is free.  A
// warp lists the channels of 128 in their order, a third of the threads each takes a third of the lists, a thread per column.
template <int MODE, typename XT>
__device__ __noinline__ void i8_apart_sums(const FcArgs *a, I8Apart *out, const uint32_t *top, uint32_t rows, int k_lo, int k_hi, int tile) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = tid % I8_TN, third = tid / I8_TN, col = tile * I8_TN + c;
    const float tau = MODE == MODE_GATHER ? ld_act(a->tau) : 0.0f;
    const signed char *W = static_cast<const signed char *>(a->W) + col;
    for (; rows; rows &= rows - 1) {
        const int b = __ffs(rows) - 1;
        const float least = i8_least(i8_shift(top[b]));
        const XT *x = static_cast<const XT *>(a->x) + (size_t)b * a->x_ld;
        double sum = 0.0;
        for (int k0 = k_lo; k0 < k_hi; k0 += I8_WARPS * I8_KB) {
            int n = 0;
            for (int e = 0; e < I8_KB; e += 32) {
                const int k = k0 + warp * I8_KB + e + lane;
                float v = 0.0f;
                if (k < k_hi) {
                    v = widen1(ld_act(x + k));
                    if (MODE == MODE_GATHER && a->m) v = __fsub_rn(v, ld_act(a->m + k));
                    v = MODE == MODE_DENSE || fabsf(v) >= tau ? __fmul_rn(v, ld_act(a->wscale + k)) : 0.0f;
                }
                const bool on = i8_is_apart(v, least);
                const uint32_t vote = __ballot_sync(0xffffffffu, on);
                if (on) out->entry[warp][n + __popc(vote & ((1u << lane) - 1u))] = I8Entry{v, k};
                n += __popc(vote);
            }
            if (lane == 0) out->count[warp] = n;
            __syncthreads();
            if (col < a->Nh) {
                for (int w = third; w < I8_WARPS; w += I8_THREADS / I8_TN)
                    for (int i = 0; i < out->count[w]; ++i) {
                        const I8Entry q = out->entry[w][i];
                        sum += (double)q.v * (double)W[(size_t)q.k * a->ldw];
                    }
            }
            __syncthreads();
        }
        out->part[third][c] = sum;
        __syncthreads();
        if (third == 0) out->sum[b][c] = (float)(out->part[0][c] + out->part[1][c] + out->part[2][c]);
    }
    __syncthreads();
}

template <int BR, int MODE, typename XT>
__global__ void __launch_bounds__(I8_THREADS, 2) fc_i8_kernel(const __grid_constant__ I8Args ia, const __grid_constant__ CUtensorMap tmap) {
    const FcArgs &a = ia.f;
    constexpr int NC = i8_ncols(BR), NW = i8_nw(BR), NX = i8_nx(BR), NE = i8_ne(BR), BPS = i8_bps(BR);
    constexpr uint32_t XB = i8_xbytes(BR), LBO = i8_chunk(BR), TCOLS = i8_tcols(BR);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *s_w = smem, *s_x = smem + i8_off_x(BR);
    float *s_gather = reinterpret_cast<float *>(smem + i8_off_gather(BR));
    I8Misc *misc = reinterpret_cast<I8Misc *>(smem + i8_off_misc(BR));
    volatile int *abort_flag = &misc->abort;
    const uint32_t spin = a.spin ? (uint32_t)a.spin : TRIES;
    int *const status = a.status;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x, s = blockIdx.y;
    const int B = a.B, S = a.S, K = a.K;
    const int per = ia.per;
    const uint32_t recv_bar = smem_addr(&misc->recv);
    const int b_lo = s * ia.blocks + min(s, ia.extra), n = ia.blocks + (s < ia.extra ? 1 : 0);  // this rank's blocks
    const int k_lo = b_lo * I8_KB, k_hi = min(K, k_lo + n * I8_KB), nst = (n + BPS - 1) / BPS;   // its channels and stages
    const int ups = (B + 3) >> 2;  // units of a block: four batch rows each
    if (tid == 0) {
        for (int i = 0; i < NW; ++i) {
            mbar_init(&misc->wfull[i], 1);
            mbar_init(&misc->wempty[i], 1);
        }
        for (int i = 0; i < NX; ++i) mbar_init(&misc->xfull[i], BPS * ups);
        for (int i = 0; i < NE; ++i) mbar_init(&misc->xempty[i], 1);
        mbar_init(&misc->done, 1);
        misc->abort = 0;
        misc->apart = 0;
        misc->scale = 0x7fffffffu;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (S > 1) {
            const int owned = max(0, min(per, I8_TN - s * per));
            mbarrier_init(recv_bar, 1);
            mbarrier_arrive_expect(recv_bar, (uint32_t)(S * B * owned * 4));
        }
    }
    if (tid < 16) misc->top[tid] = misc->fin[tid] = 0;
    if (S > 1) cluster_arrive_relaxed();
    // m, x and the scales are asked into L2 ahead of the weight stream (hints, as in the dense-stream kernel)
    if (warp == 1 && MODE == MODE_GATHER && a.m)
        for (int k = k_lo + lane * 32; k < k_hi; k += 1024) prefetch_l2_keep(a.m + k);
    if (warp == 2)
        for (int k = k_lo + lane * 32; k < k_hi; k += 1024) prefetch_l2_keep(a.wscale + k);
    if (warp >= 4)
        for (int b = warp - 4; b < B; b += 8)
            for (int k = k_lo + lane * 64; k < k_hi; k += 2048) prefetch_l2_keep(static_cast<const XT *>(a.x) + (size_t)b * a.x_ld + k);
    // The codes are constants of the layer: the first ring is asked for before the wait for earlier work on the stream.
    auto box = [&](int blk, uint32_t slot) {
        mbar_arrive_expect_tx(&misc->wfull[slot], I8_BOX);
        tma_box_2d(smem_u32(s_w) + slot * I8_BOX, &tmap, tile * I8_TN, (b_lo + blk) * I8_KB, &misc->wfull[slot]);
    };
    const int first = min(n, NW);
    if (tid == 0) {
        for (int i = 0; i < first; ++i) box(i, i);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&misc->tmem_base)), "r"(TCOLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();  // barriers and TMEM address
    tc_fence_after();
    griddep_wait();
    griddep_launch_dependents();

    struct Raw {
        uint4 m, c;
        uint2 x[4];
    } raw, raw1;
    // Units go round the preparing warps, (ub, uq) = block and quarter of the rows.
    const uint32_t ups_inv = ups == 3 ? 86u : 256u >> (ups >> 1);  // ceil(256 / ups)
    const int di = (I8_PREP * ups_inv) >> 8, dq = I8_PREP - di * ups;
    int ub = ((warp - 1) * ups_inv) >> 8, uq = (warp - 1) - ub * ups;
    auto step = [&](int &blk, int &rq) {
        blk += di;
        rq += dq;
        if (rq >= ups) {
            rq -= ups;
            ++blk;
        }
    };
    auto load = [&](Raw &raw, int blk, int rq) {
        const int kb = k_lo + blk * I8_KB, k = kb + lane * 4, b0 = rq * 4;
        const XT *xp = static_cast<const XT *>(a.x) + (size_t)b0 * a.x_ld + k;
        if (kb + I8_KB <= k_hi && (MODE == MODE_DENSE || a.m)) {
            // (a row that the batch does not have repeats the last one; its values are not used)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                raw.x[r] = ld_act8(xp);
                if (b0 + r + 1 < B) xp += a.x_ld;
            }
            if constexpr (MODE == MODE_GATHER) raw.m = ld_act16u(a.m + k);
            raw.c = ld_act16u(a.wscale + k);
        } else {
            const bool in = k < k_hi;  // (K is a multiple of eight: four channels are inside the matrix or outside together)
#pragma unroll
            for (int r = 0; r < 4; ++r) raw.x[r] = ld_act8_if(xp + (size_t)r * a.x_ld, in && b0 + r < B);
            if constexpr (MODE == MODE_GATHER) raw.m = ld_act16_if(a.m + k, in && a.m != nullptr);
            raw.c = ld_act16_if(a.wscale + k, in);
        }
    };
    float tau = 0.0f;
    // Pruned and scaled values of row r of the unit: zeros for dropped channels.  Beyond the matrix everything is zero, kept or not.
    auto value = [&](const Raw &raw, int r, float (&v)[4]) {
        const XT *xe = reinterpret_cast<const XT *>(&raw.x[r]);
        const float *me = reinterpret_cast<const float *>(&raw.m), *ce = reinterpret_cast<const float *>(&raw.c);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float d = widen1(xe[e]);
            if constexpr (MODE == MODE_GATHER) d = __fsub_rn(d, me[e]);  // (m == NULL: zeros)
            const bool on = MODE == MODE_DENSE || fabsf(d) >= tau;
            v[e] = on ? __fmul_rn(d, ce[e]) : 0.0f;  // (the scale of a dropped channel has no part in y, whatever it is)
        }
    };
    float keep[I8_KEEP][4][4];
    if (warp >= 1) {
        if (ub < n) load(raw, ub, uq);
        if constexpr (MODE == MODE_GATHER) tau = ld_act(a.tau);
        int b1 = ub, q1 = uq;
        step(b1, q1);
        if (b1 < n) load(raw1, b1, q1);
        // ---- first pass: the largest value of every row
        int blk = ub, rq = uq;
        auto largest = [&](const Raw &raw, float (&v)[4][4]) {
            const int b0 = rq * 4;
            uint32_t top[4];
            if (MODE == MODE_GATHER && rq == 0) {  // the smallest scale (beyond the matrix there is none)
                const float *ce = reinterpret_cast<const float *>(&raw.c);
                const uint32_t t = min(min(i8_bits(ce[0]), i8_bits(ce[1])), min(i8_bits(ce[2]), i8_bits(ce[3])));
                const uint32_t least = __reduce_min_sync(0xffffffffu, k_lo + blk * I8_KB + lane * 4 < k_hi ? t : 0x7fffffffu);
                if (lane == 0) atomicMin(&misc->scale, least);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (b0 + r < B) {
                    value(raw, r, v[r]);
                    top[r] = i8_top(v[r]);
                }
            }
            if (MODE == MODE_GATHER && BR == 4 && a.bits && tile == 0) {  // union mask (up to two rows), a word per 32 channels = eight lanes
                const int k = k_lo + blk * I8_KB + lane * 4;
                const float *me = reinterpret_cast<const float *>(&raw.m);
                uint32_t w = 0;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool k0 = fabsf(__fsub_rn(widen1(reinterpret_cast<const XT *>(&raw.x[0])[e]), me[e])) >= tau;
                    const bool k1 = B > 1 && fabsf(__fsub_rn(widen1(reinterpret_cast<const XT *>(&raw.x[1])[e]), me[e])) >= tau;
                    w |= k0 || k1 ? 1u << e : 0u;
                }
                w = k < k_hi ? w << (4 * (lane & 7)) : 0u;
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
                if ((lane & 7) == 0 && k < k_hi) a.bits[k >> 5] = w;
            }
            step(blk, rq);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (b0 + r < B) {
                    const uint32_t t = __reduce_max_sync(0xffffffffu, top[r]);
                    if (lane == 0) atomicMax(&misc->top[b0 + r], t);
                }
            }
        };
        if (blk < n) largest(raw, keep[0]);
        int b2 = b1, q2 = q1;
        step(b2, q2);
        if (b2 < n) load(raw, b2, q2);  // asked for two units ahead
        if (blk < n) largest(raw1, keep[1]);
#pragma unroll 1
        while (blk < n) {
            float v[4][4];
            raw1 = raw;
            step(b2, q2);
            if (b2 < n) load(raw, b2, q2);
            largest(raw1, v);
        }
    }
    __syncthreads();
    uint32_t odd = 0;  // rows with a value that is not finite
#pragma unroll
    for (int b = 0; b < BR; ++b) odd |= misc->top[b] >= 0x7f800000u ? 1u << b : 0u;
    if (odd) {  // the largest of the others (rare; the same for the whole CTA)
        if (warp >= 1) {
            for (int blk = ub, rq = uq; blk < n; step(blk, rq)) {
                load(raw, blk, rq);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float v[4];
                    uint32_t t = 0;
                    value(raw, r, v);
#pragma unroll
                    for (int e = 0; e < 4; ++e) t = max(t, i8_bits(v[e]) < 0x7f800000u ? i8_bits(v[e]) : 0u);
                    atomicMax(&misc->fin[rq * 4 + r], t);
                }
            }
        }
        __syncthreads();
        if (tid < BR && (odd >> tid & 1)) misc->top[tid] = misc->fin[tid];
        __syncthreads();
    }
    const uint32_t tmem = misc->tmem_base;
    // A wait by a whole warp; all lanes agree on the outcome.
    auto warp_wait = [&](unsigned long long *bar, uint32_t parity, int code) -> bool {
        const bool go = i8_wait(bar, parity, code, abort_flag, spin, status);
        return __all_sync(0xffffffffu, go) != 0;
    };

    if (warp == 0) {
        // ---- MMAs.  D: 32-bit integers; codes signed, MN-major; digits signed, K-major.  The whole warp runs the loop and one
        // lane issues: descriptors and addresses then stay in uniform registers (with the loop inside `if (lane == 0)` 128 channels
        // took 1600 cycles instead of 430).
        uint32_t leader;
        asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(leader));
        constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | ((uint32_t)(NC >> 3) << 17) | ((uint32_t)(I8_TN >> 4) << 24);
        constexpr uint32_t WK = 32 * I8_TN >> 4, XK = (2 * LBO) >> 4;  // 32 channels further, in units of 16 bytes
        const uint64_t dw0 = tc_desc(smem_u32(s_w), I8_BOX, 1024, 2), dx0 = tc_desc(smem_u32(s_x), LBO, 128, 0);
        uint32_t ws = 0, wpar = 0, xs = 0, xpar = 0, xe = 0, rs = 0, rpar = 0;  // slots: weights, activations and their barrier, weights to ask for
        auto next = [&](uint32_t &slot, uint32_t &par) {
            if (++slot == NW) { slot = 0; par ^= 1u; }
        };
        int asked = first;
#pragma unroll 1
        for (int i = 0; i < nst; ++i) {
            // both operands, and the slots of the stage before, which take the next boxes: each is waited for by a lane of its own
            const bool two = BPS == 2 && 2 * i + 1 < n;
            const int refill = i >= 1 ? min(BPS, n - asked) : 0;
            uint32_t ws1 = ws, wpar1 = wpar, rs1 = rs, rpar1 = rpar;
            next(ws1, wpar1);
            next(rs1, rpar1);
            unsigned long long *bar = &misc->wfull[ws];
            uint32_t bpar = wpar;
            if (lane == 1) { bar = &misc->xfull[xs]; bpar = xpar; }
            if (lane == 2 && two) { bar = &misc->wfull[ws1]; bpar = wpar1; }
            if (lane == 3 && refill > 0) { bar = &misc->wempty[rs]; bpar = rpar; }
            if (lane == 4 && refill > 1) { bar = &misc->wempty[rs1]; bpar = rpar1; }
            if (!warp_wait(bar, bpar, 2)) break;
            tc_fence_after();
            const uint64_t da = dw0 + ws * (I8_BOX >> 4), db = dw0 + ws1 * (I8_BOX >> 4), dx = dx0 + xs * (XB >> 4);
            const int left = (k_hi - k_lo - i * BPS * I8_KB + 31) >> 5;  // steps of 32 channels
            if (leader) {
                if (left >= 4 * BPS) {
#pragma unroll
                    for (uint32_t ks = 0; ks < 4; ++ks) tc_mma_i8(tmem, da + ks * WK, dx + ks * XK, idesc, (ks > 0 || i > 0) ? 1u : 0u);
                    if constexpr (BPS == 2) {
#pragma unroll
                        for (uint32_t ks = 0; ks < 4; ++ks) tc_mma_i8(tmem, db + ks * WK, dx + (4 + ks) * XK, idesc, 1u);
                    }
                } else {
#pragma unroll 1
                    for (int ks = 0; ks < left; ++ks) tc_mma_i8(tmem, (ks < 4 ? da : db) + (ks & 3) * WK, dx + ks * XK, idesc, (ks > 0 || i > 0) ? 1u : 0u);
                }
                tc_commit(&misc->wempty[ws]);
                if (two) tc_commit(&misc->wempty[ws1]);
                tc_commit(&misc->xempty[xe]);
                if (refill > 0) box(asked, rs);
                if (refill > 1) box(asked + 1, rs1);
            }
            if (refill > 0) next(rs, rpar);
            if (refill > 1) next(rs, rpar);
            asked += max(0, refill);
            next(ws, wpar);
            if constexpr (BPS == 2) next(ws, wpar);
            if (++xs == NX) { xs = 0; xpar ^= 1u; }
            if (++xe == NE) xe = 0;
        }
        // all MMAs have finished, and no copy is under way, before anyone leaves
        int own_abort = 0;
        if (leader) tc_commit(&misc->done);
        i8_wait(&misc->done, 0, 4, &own_abort, TRIES, status);
        if (*abort_flag)
            for (int q = max(0, asked - NW); q < asked; ++q) i8_wait(&misc->wfull[q % NW], (uint32_t)(q / NW) & 1u, 5, &own_abort, TRIES, status);
    } else {
        // ---- second pass: the digits
        int blk = ub, rq = uq;
        const int shifts = lane < BR ? i8_shift(misc->top[lane]) : 0;  // lane b: of row b
        // Rows that can have a value without digits: a kept one is no smaller than the threshold times the smallest scale (products are
        // rounded alike), which mostly settles it for the whole rank.
        const bool can = lane < B && (MODE == MODE_DENSE || odd || !(__fmul_rn(tau, __uint_as_float(misc->scale)) >= i8_least(shifts)));
        const uint32_t check = __ballot_sync(0xffffffffu, can);
        auto digits = [&](float (&v)[4][4]) -> bool {
            const int i = blk / BPS;
            const uint32_t xs = (uint32_t)i % NX;
            if (i >= NX && !warp_wait(&misc->xempty[(uint32_t)(i - NX) % NE], ((uint32_t)(i - NX) / NE) & 1u, 1)) return false;
            unsigned char *dst = s_x + xs * XB + ((blk % BPS) * (I8_KB / 16) + (lane >> 2)) * LBO + (lane & 3) * 4 + rq * 64;  // (rows of 16 bytes follow one another)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (rq * 4 + r < B) {
                    const int shift = __shfl_sync(0xffffffffu, shifts, rq * 4 + r);
                    const float up = i8_pow2(shift);
                    if (check >> (rq * 4 + r) & 1u) {
                        const float least = i8_least(shift);
                        bool some = odd != 0;
#pragma unroll
                        for (int e = 0; e < 4; ++e) some |= fabsf(v[r][e]) < least && v[r][e] != 0.0f;
                        if (some) {  // (rare)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                if (i8_is_apart(v[r][e], least)) {
                                    v[r][e] = 0.0f;
                                    atomicOr(&misc->apart, 1u << (rq * 4 + r));
                                }
                            }
                        }
                    }
                    // Limbs from the top, rounded to the nearest integer by adding 1.5 x 2^23; 128 more, and the second byte of the sum is the upper
                    // digit, the first one the lower digit with its sign turned round.  What is left of a value is exact at every step.
                    constexpr float M = 12582912.0f + 128.0f;
                    uint32_t t[3][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float t2 = __fmaf_rn(v[r][e], up, M), d1 = __fmaf_rn(v[r][e], up, -__fsub_rn(t2, M));
                        const float t1 = __fmaf_rn(d1, 32768.0f, M), d0 = __fmaf_rn(d1, 32768.0f, -__fsub_rn(t1, M));
                        t[0][e] = __float_as_uint(__fmaf_rn(d0, 32768.0f, M));
                        t[1][e] = __float_as_uint(t1);
                        t[2][e] = __float_as_uint(t2);
                    }
#pragma unroll
                    for (int l = 0; l < 3; ++l) {  // digit x BR + row: the lowest first
                        const uint32_t t01 = __byte_perm(t[l][0], t[l][1], 0x5140), t23 = __byte_perm(t[l][2], t[l][3], 0x5140);
                        *reinterpret_cast<uint32_t *>(dst + (2 * l * BR + r) * 16) = __byte_perm(t01, t23, 0x5410) ^ 0x80808080u;
                        *reinterpret_cast<uint32_t *>(dst + ((2 * l + 1) * BR + r) * 16) = __byte_perm(t01, t23, 0x7632);
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the tensor core
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&misc->xfull[xs]);
                if (BPS == 2 && blk + 1 == n && blk % 2 == 0) mbar_arrive(&misc->xfull[xs]);  // the last stage has no second block
            }
            step(blk, rq);
            return true;
        };
        bool ok = true;
#pragma unroll
        for (int j = 0; j < I8_KEEP; ++j) {
            if (j + 1 == I8_KEEP) {  // the first unit that was not kept, asked for a unit ahead
                int nb = blk, nq = rq;
                step(nb, nq);
                if (nb < n) load(raw, nb, nq);
            }
            if (ok && blk < n) ok = digits(keep[j]);
        }
        while (ok && blk < n) {
            float v[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r) value(raw, r, v[r]);
            int nb = blk, nq = rq;
            step(nb, nq);
            if (nb < n) load(raw, nb, nq);
            ok = digits(v);
        }
    }
    // ---- cluster exchange, push form: a column of the tile is a TMEM lane; every sum of the rank goes to the rank that finishes its
    // column as a store that counts down its barrier
    __syncthreads();  // (all MMAs have finished, and every row with a value without digits is marked)
    const uint32_t apart = misc->apart | odd;
    I8Apart *const s_apart = reinterpret_cast<I8Apart *>(s_w);
    if (apart) i8_apart_sums<MODE, XT>(&a, s_apart, misc->top, apart, k_lo, k_hi, tile);
    if (S > 1) cluster_wait();  // every rank's barrier is initialised (all ranks arrived before their streams)
    if (warp >= 4 && warp < 8) {
        const bool ok = warp_wait(&misc->done, 0, 4) && __all_sync(0xffffffffu, *abort_flag == 0);
        tc_fence_after();
        const int dc = (warp & 3) * 32 + lane;
        const int r = (int)((uint32_t)dc * ia.per_inv >> 20), slot0 = s * BR * per + (dc - r * per);
        const uint32_t dst0 = S > 1 ? cluster_addr(smem_addr(s_gather) + 4u * (uint32_t)slot0, (uint32_t)r) : 0u;
        const uint32_t dbar = S > 1 ? cluster_addr(recv_bar, (uint32_t)r) : 0u;
        const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        constexpr int RL = 4;  // rows at a time
#pragma unroll
        for (int b0 = 0; b0 < BR; b0 += RL) {
            if (b0 >= B) break;  // (the same for the whole warp)
            uint32_t v[I8_ND][RL];
            if (ok) {
#pragma unroll
                for (int d = 0; d < I8_ND; ++d) tc_ldn(v[d], lanes + (uint32_t)(d * BR + b0));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            }
#pragma unroll
            for (int e = 0; e < RL; ++e) {
                const int b = b0 + e;
                if (b < B) {
                    float y = 0.0f;
                    if (ok) {
                        float limb[3];
#pragma unroll
                        for (int l = 0; l < 3; ++l) limb[l] = fmaf((float)(int)v[2 * l + 1][e], 256.0f, (float)(int)v[2 * l][e]);
                        y = fmaf(fmaf(limb[0], 0x1p-15f, limb[1]), 0x1p-15f, limb[2]) * i8_pow2(-i8_shift(misc->top[b]));
                        if (apart >> b & 1) y += s_apart->sum[b][dc];
                    }
                    if (S > 1) st_async_f32(dst0 + 4u * (uint32_t)(b * per), y, dbar);
                    else s_gather[slot0 + b * per] = y;
                }
            }
        }
    }
    // the bias of this thread's first result, asked for ahead of the last wait
    const int c0 = (int)((uint32_t)tid * ia.per_inv >> 20);  // batch row of result tid
    const int mine = s * per + tid - c0 * per;               // its column in the tile
    float bias = 0.0f;
    if (tid < per * B && mine < I8_TN && tile * I8_TN + mine < a.Nh && a.bias) bias = __ldcg(a.bias + tile * I8_TN + mine);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
    if (warp * 32 >= per * B) return;
    if (S > 1) {
        bool landed = false;
#pragma unroll 1
        for (uint32_t it = 0; it < TRIES && !landed; ++it) landed = mbarrier_try_wait(recv_bar, 0);
        if (!landed && status) atomicCAS(status, 0, 6);  // never in a correct run; the result is then incomplete
    }
    // the S partials of a result in rank order, and the bias
    for (int i = tid; i < per * B; i += I8_THREADS) {
        const int b = (int)((uint32_t)i * ia.per_inv >> 20), c = s * per + i - b * per, col = tile * I8_TN + c;
        if (c < I8_TN && col < a.Nh) {
            float v = i == tid ? bias : a.bias ? __ldcg(a.bias + col) : 0.0f;
#pragma unroll
            for (int q = 0; q < MAX_CLUSTER; ++q)
                if (q < S) v += s_gather[q * BR * per + i];
            a.y[(size_t)b * a.y_ld + col] = v;
        }
    }
}

// ---- host side ------------------------------------------------------------------------------------------------

// The codes as a 2-D tensor of bytes: boxes of 128 columns x 128 channels, 128-byte swizzle; rows and columns beyond the matrix read as
// zeros.  The map covers this GPU's own W only, and every box goes to the one CTA that asked for it.
static bool i8_tensor_map(CUtensorMap *map, const void *W, int K, int N) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)K};
    const cuuint64_t strides[1] = {(cuuint64_t)N};
    const cuuint32_t box[2] = {I8_TN, I8_KB};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(W), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BR, int MODE, typename XT>
static cudaError_t launch_i8_b(const FcArgs &a, const CUtensorMap &map, cudaStream_t st) {
    static SmemOptIn opt_in;
    auto kern = fc_i8_kernel<BR, MODE, XT>;
    cudaError_t e0 = ensure_dynamic_smem(kern, i8_smem(BR), opt_in);
    if (e0 != cudaSuccess) return e0;
    I8Args ia;
    ia.f = a;
    const int blocks = (a.K + I8_KB - 1) / I8_KB;
    ia.blocks = blocks / a.S;
    ia.extra = blocks % a.S;
    ia.per = (I8_TN + a.S - 1) / a.S;
    ia.per_inv = ((1u << 20) + ia.per - 1) / ia.per;
    return launch_cluster(kern, dim3((a.ldw + I8_TN - 1) / I8_TN, a.S), dim3(I8_THREADS), i8_smem(BR), a.S, st, g_tune.pdl != 0, ia, map);
}
template <int MODE, typename XT>
static cudaError_t launch_i8_x(const FcArgs &a, const CUtensorMap &map, cudaStream_t st) {
    if (a.B <= 4) return launch_i8_b<4, MODE, XT>(a, map, st);
    if (a.B <= 8) return launch_i8_b<8, MODE, XT>(a, map, st);
    return launch_i8_b<16, MODE, XT>(a, map, st);
}

// Split-K factor: the most CTAs that are all resident (two per SM), at least one block per rank.
int i8_split(const FcArgs &a) {
    const int tiles = (a.ldw + I8_TN - 1) / I8_TN, blocks = (a.K + I8_KB - 1) / I8_KB;
    int best_S = 1;
    long long best = -1;
    for (int S = 1; S <= MAX_CLUSTER; ++S) {
        if (g_tune.split_k > 0 && S > g_tune.split_k) continue;
        const long long ctas = (long long)tiles * S;
        if (S > blocks || (S > 1 && ctas > resident_ctas(S))) continue;
        if (ctas >= best) { best = ctas; best_S = S; }
    }
    return best_S;
}

int i8_blocks_per_rank(const FcArgs &a, int S) { return ((a.K + I8_KB - 1) / I8_KB + S - 1) / S; }

// Rows of x and of the codes must lie on 16-byte boundaries (vector loads, stride of the tensor map), and the 32-bit sums must hold a
// rank's channels (2^14 per product).
bool i8_applicable(const FcArgs &a, int blocks_per_rank) {
    return a.K % 8 == 0 && a.ldw % 16 == 0 && a.B >= 1 && a.B <= 16 && !a.hold_dependents && aligned16(a.wscale) && blocks_per_rank <= 512;
}

cudaError_t launch_fc_i8(int mode, int xkind, FcArgs a, cudaStream_t st) {
    CUtensorMap map;
    if (!i8_tensor_map(&map, a.W, a.K, a.ldw)) return cudaErrorNotSupported;
    a.status = tc_status_ptr();
    a.spin = g_tune.tc_spin;
    if (mode == MODE_DENSE) return xkind == 1 ? launch_i8_x<MODE_DENSE, __nv_bfloat16>(a, map, st) : launch_i8_x<MODE_DENSE, __half>(a, map, st);
    return xkind == 1 ? launch_i8_x<MODE_GATHER, __nv_bfloat16>(a, map, st) : launch_i8_x<MODE_GATHER, __half>(a, map, st);
}

}  // namespace scap
