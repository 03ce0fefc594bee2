// Quantised weights on the tensor cores: the sparse FC on 8-bit or group-wise 4-bit codes, every row of the weight streamed
// once for up to eight batch rows (more rows: two halves side by side in the grid, the second one meets the codes in L2).
//
// The codes are exact in bf16, the pruned activation (binary32) is split exactly into three bf16 parts, and the products
// run through mma.sync.m16n8k16 with the weights as the M operand (16 columns) and the activations as the N operand
// (batch rows x parts).  Everything stays in registers: a lane loads the codes of four consecutive channels for its
// columns, pairs the channels with byte permutes, and turns them into operand fragments with 1.5 (8-bit) or 1.25 (4-bit)
// instructions per weight; the same lane loads, thresholds and splits the activations of those four channels.  The k order
// inside an MMA is free as long as both operands agree, which is what makes 16-byte loads of one row usable directly.
// All warps run the same short loop and share nothing until the end: no staging, no barrier, no kept list.
//   (The same decomposition on tcgen05 - codes through shared memory into a swizzled operand, warps specialised into
//   copy, convert, threshold, issue and promote - took 43 us for 8-bit 11008 x 4096 at one row: six different
//   instruction streams on every scheduler and a dozen hand-overs per stage cost more than the tensor core saves.)
//
// (8-bit calls of three and more rows of a long layer take the integer kernel of scap_fc_i8.cu.)
//
// Why it is here: beyond two rows the fp32-FMA kernels run two rows per launch, so the codes cross the chip B / 2 times.
// K = 11008, N = 4096, half of the entries pruned, weights from DRAM, FMA kernel -> this one, device us per call:
//   8-bit            4 rows 24.6 -> 18.3   8 rows 48.0 -> 23.9   16 rows  94.6 -> 41.2
//   4-bit, group 128 4 rows 36.1 -> 16.8   8 rows 71.6 -> 21.3   16 rows 142   -> 37.0
// The codes are 45 (22.5) MB, 7 (3.5) us at copy speed.  What is left, by counters at eight rows: 9.3 M (10.7 M) warp instructions,
// 421 (485) per 16 channels x 128 columns with everything included, 56 % (48 %) of them on the half-rate integer pipe, at 0.38
// (0.48) a cycle and scheduler; a warp waits for its loads more than half (a quarter) of the time, since with 128 registers a
// thread there are 16 warps on an SM with two blocks each in flight.
//
// Precision: codes, parts and products (16 bits at most) are exact; the sum of a chain is truncated by the tensor core where the
// exponents of its terms lie too far apart.  The two smaller parts never share an accumulator with the leading one.  Error against
// 64 bits 8e-8 (8-bit FMA kernel 1.3e-7).
// A rank's channels are spread over 4 or 8 warps and S ranks, added at the end in fixed order in binary32.
//
//   grid = (128-column tiles, S, 1 or 2), cluster (1, S, 1), 256 threads, two CTAs per SM
//   warps: up to four rows 128 columns x 8 ranges of channels; up to eight rows 64 columns x 4 ranges (accumulators)
#include <string.h>

#include <type_traits>

#include "scap_qm.cuh"

namespace scap {

constexpr int QM_TN = 128;
constexpr int QM_SCALE_MAX = 60 * 1024;  // shared memory for the scales and zero points of a rank's groups
constexpr int QM_GROUP_BYTES = QM_TN * 5;  // 128 scales and 128 zero points
__host__ __device__ constexpr int qm_cw(int BT) { return BT <= 4 ? 128 : 64; }     // columns per warp
__host__ __device__ constexpr int qm_nkg(int BT) { return FC_WARPS * qm_cw(BT) / QM_TN; }  // ranges of channels per rank
__host__ __device__ constexpr int qm_red_bytes(int BT) { return qm_nkg(BT) * BT * QM_TN * 4; }
// 8-bit weights: the leading sums leave the tensor core's accumulators every 16 QM_CHAIN channels, for slots of the thread in shared
// memory.  A truncating accumulator that holds a large value (one activation a thousand times the others) loses up to 2^-23 of it with
// every product: a chain of 224 (14336 x 11008, 16 rows, one rank) was off by 6.3e-6 of the result, the FMA kernel by 2.4e-7; in chains of eight it is
// 3.1e-7, and 7e-8 (FMA 1.9e-7) where the large ones are thirty times the others.  11008 x 4096, us: four rows 17.8 -> 18.3, eight rows
// 23.8 -> 23.9, sixteen 41.0 -> 41.2.  (The 4-bit sums are closed once per group.)
constexpr int QM_CHAIN = 8;
__host__ __device__ constexpr int qm_slot_quads(int BT) { return qm_cw(BT) / 16; }  // float4 per thread
__host__ __device__ constexpr int qm_slot_bytes(int WB, int BT) { return WB == 8 ? FC_THREADS * qm_slot_quads(BT) * 16 : 0; }
__host__ __device__ constexpr int qm_smem(int BT) { return qm_red_bytes(BT) + BT * GATHER_LD * 4 + 16; }  // partials | gather | barrier
static_assert(2 * (qm_smem(4) + QM_SCALE_MAX + 1024) <= 233472 && 2 * (qm_smem(8) + QM_SCALE_MAX + 1024) <= 233472, "two CTAs must fit in the shared memory of an SM");

template <int BYTES>
struct QmRow;  // one row's codes of a lane
template <>
struct alignas(16) QmRow<16> { uint32_t w[4]; };
template <>
struct alignas(8) QmRow<8> { uint32_t w[2]; };
template <>
struct QmRow<4> { uint32_t w[1]; };

__device__ __forceinline__ void qm_ld(QmRow<16> &r, const void *p) {
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]) : "l"(p));
}
__device__ __forceinline__ void qm_ld(QmRow<8> &r, const void *p) {
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(r.w[0]), "=r"(r.w[1]) : "l"(p));
}
__device__ __forceinline__ void qm_ld(QmRow<4> &r, const void *p) {
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(r.w[0]) : "l"(p));
}
__device__ __forceinline__ uint2 ld_act8(const void *p) {
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_act16(const void *p) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t bf16x2_fma(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// An integer 0..255 in the low bits of a bf16 is that integer times 2^-133 (the subnormals and the first binade are one
// straight line), so one fma per pair turns codes into bf16 values: times 2^127, minus the offset - exact, and 1/64 of the
// code, which the epilogue puts right.  Signed bytes 0 and 2 of t:
__device__ __forceinline__ uint32_t qm_pair8(uint32_t t) { return bf16x2_fma((t ^ 0x00800080u) & 0x00ff00ffu, 0x7f007f00u, 0xc000c000u); }
// Low (high) nibbles of bytes 0 and 2 of t, minus 8 (the zero points are put right once per group):
__device__ __forceinline__ uint32_t qm_pair4_lo(uint32_t t) { return bf16x2_fma(t & 0x000f000fu, 0x7f007f00u, 0xbe00be00u); }
__device__ __forceinline__ uint32_t qm_pair4_hi(uint32_t t) { return bf16x2_fma(t & 0x00f000f0u, 0x7d007d00u, 0xbe00be00u); }

template <int WB, int BT, int MODE, typename XT>
__global__ void __launch_bounds__(FC_THREADS, 2) fc_qm_kernel(const QmArgs qa) {
    constexpr int CW = qm_cw(BT), NKG = qm_nkg(BT), CPT = CW / 8, RB = CPT * WB / 8, NP = CPT / 2;
    constexpr int NS = BT == 8 ? 2 : 1;  // accumulator sets: eight rows: leading part | the other two; fewer rows: parts are N columns
    extern __shared__ __align__(16) unsigned char smem[];
    float *s_red = reinterpret_cast<float *>(smem);
    float *s_gather = reinterpret_cast<float *>(smem + qm_red_bytes(BT));
    const uint32_t bar = smem_addr(smem + qm_red_bytes(BT) + BT * GATHER_LD * 4);
    unsigned char *s_scale = smem + qm_smem(BT);                 // [group of the rank][128] scales
    unsigned char *s_zero = s_scale + (size_t)qa.sg * QM_TN * 4;  // [group of the rank][128] zero points

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int tile = blockIdx.x, s = blockIdx.y;
    FcArgs a = qa.f;
    if (gridDim.z == 2) {  // more than eight rows: the halves of the batch
        const int h = (a.B + 1) >> 1, b0 = blockIdx.z ? h : 0;
        a.x = static_cast<const XT *>(a.x) + (size_t)b0 * a.x_ld;
        a.y += (size_t)b0 * a.y_ld;
        a.B = blockIdx.z ? a.B - h : h;
    }
    const int B = a.B, S = a.S, K = a.K, N = a.ldw;
    const int per = (QM_TN + S - 1) / S;  // columns this rank finishes (the last rank may own fewer)
    if (S > 1) {
        if (tid == 0) {
            const int owned = max(0, min(per, QM_TN - s * per));
            mbarrier_init(bar, 1);
            mbarrier_arrive_expect(bar, (uint32_t)(S * B * owned * 4));
        }
        cluster_arrive_relaxed();
    }
    // this rank's blocks of 16 channels; a warp takes a contiguous stretch of them
    const int nblk = (K + 15) >> 4;
    const int r_lo = (int)((long long)nblk * s / S), r_n = (int)((long long)nblk * (s + 1) / S) - r_lo;
    const int ch = CW == 64 ? warp & 1 : 0, kg = CW == 64 ? warp >> 1 : warp;
    const int b_lo = r_lo + r_n * kg / NKG, b_hi = r_lo + r_n * (kg + 1) / NKG;
    const int lcol = ch * 64 + g * CPT;  // this lane's first column in the tile
    // Columns, rows and parts that do not exist are computed from existing ones (their results have no reader); channels
    // beyond K have zero activations.
    const int wcol = tile * QM_TN + lcol < N ? tile * QM_TN + lcol : 0;
    const size_t row_bytes = (size_t)N * WB / 8;
    const unsigned char *w0 = static_cast<const unsigned char *>(a.W) + (size_t)wcol * WB / 8;
    const int bx = g % BT, part = g / BT;  // batch row and part of this lane's N column
    const XT *xp = static_cast<const XT *>(a.x) + (size_t)(bx < B ? bx : 0) * a.x_ld;
    struct Codes {
        QmRow<RB> w[4];
    };
    struct Acts {
        uint2 x;
        float4 m, c;
    };
    // K is a multiple of four: a lane's channels are inside the matrix or outside together
    auto load_w = [&](Codes &c, int blk) {
        const int k = blk * 16 + 4 * t;
        const unsigned char *p = w0 + (size_t)(k < K ? k : 0) * row_bytes;
#pragma unroll
        for (int i = 0; i < 4; ++i) qm_ld(c.w[i], p + i * row_bytes);
    };
    auto load_x = [&](Acts &v, int blk) {
        const int k = blk * 16 + 4 * t, kk = k < K ? k : 0;
        v.x = ld_act8(xp + kk);
        if constexpr (MODE == MODE_GATHER) v.m = a.m ? ld_act16(a.m + kk) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if constexpr (WB == 8) v.c = ld_act16(a.wscale + kk);
    };
    // The codes are constants of the layer, so the first ones are asked for before the wait for earlier work on the stream;
    // everything else may be an output of that work.
    constexpr int PW = 2, PX = 2;  // blocks of codes and of activations in flight (four of the latter: no faster, 5 - 20 % slower at 8 bits)
    Codes cw[PW];
    Acts ax[PX];
#pragma unroll
    for (int i = 0; i < PW; ++i)
        if (b_lo + i < b_hi) load_w(cw[i], b_lo + i);
    griddep_wait();
    griddep_launch_dependents();
    // (tau by every warp: handing it on from one thread through shared memory costs a barrier, 0.4 us of a 3 us call)
    const float tau = MODE == MODE_GATHER ? ld_act(a.tau) : 0.0f;
#pragma unroll
    for (int i = 0; i < PX; ++i)
        if (b_lo + i < b_hi) load_x(ax[i], b_lo + i);
    float bias0[2], bias1[2];
    prefetch_bias<true, EPI_BIAS, QM_TN>(a, tile, s, per, bias0, bias1);
    const int gb = WB == 4 ? qa.group >> 4 : 1;  // blocks per scale group
    const int g_lo = r_lo / gb;                  // first group of the rank
    bool careful = false;                        // a scale of the rank is not finite
    if constexpr (WB == 4) {
        bool odd = false;
        const int ng = r_n > 0 ? (r_lo + r_n - 1) / gb - g_lo + 1 : 0;
        for (int i = tid; i < ng * 40; i += FC_THREADS) {
            const int gi = i / 40, p = i - gi * 40;
            const int c = p < 32 ? p * 4 : (p - 32) * 16;
            const bool on = tile * QM_TN + c < N;
            const size_t at = (size_t)(g_lo + gi) * N + tile * QM_TN + c;
            const uint4 v = ld_act16_if(p < 32 ? (const void *)(qa.scale + at) : (const void *)(qa.zero + at), on);
            *reinterpret_cast<uint4 *>(p < 32 ? s_scale + (size_t)(gi * QM_TN + c) * 4 : s_zero + (size_t)(gi * QM_TN + c)) = v;
            const uint32_t top = max(max(v.x << 1, v.y << 1), max(v.z << 1, v.w << 1));
            odd |= p < 32 && top >= 0xff000000u;
        }
        careful = __syncthreads_or(odd) != 0;
    }

    float acc[NS][NP][4], ds[NS][4], y[WB == 4 ? NS : 1][WB == 4 ? NP : 1][4];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
#pragma unroll
        for (int i = 0; i < 4; ++i) ds[q][i] = 0.0f;
#pragma unroll
        for (int j = 0; j < NP; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[q][j][i] = 0.0f;
                if constexpr (WB == 4) y[q][j][i] = 0.0f;
            }
    }

    auto process = [&](const Codes &c, const Acts &v4, int blk) {
        // ---- activations: threshold and exact split; f[0..2] are the N operands of up to three MMAs
        const bool k_ok = blk * 16 + 4 * t < K;
        const XT *xe = reinterpret_cast<const XT *>(&v4.x);
        const float mv[4] = {v4.m.x, v4.m.y, v4.m.z, v4.m.w}, cv[4] = {v4.c.x, v4.c.y, v4.c.z, v4.c.w};
        uint32_t hi[4], mid[4], lo[4], kept = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float v = widen1(xe[i]);
            if constexpr (MODE == MODE_GATHER) v = __fsub_rn(v, mv[i]);  // (m == NULL: zeros)
            const bool on = k_ok && (MODE == MODE_DENSE || fabsf(v) >= tau);
            kept |= on ? 1u << i : 0u;
            if constexpr (WB == 8) v = __fmul_rn(v, cv[i]);
            v = on ? v : 0.0f;  // (after the scale: that of a dropped channel has no part in y, whatever it is)
            // three consecutive 8-bit fields of the significand; an infinity stays one part (its rest would be NaN)
            hi[i] = __float_as_uint(v) & 0xffff0000u;
            float rest = v - __uint_as_float(hi[i]);
            rest = rest == rest ? rest : 0.0f;
            mid[i] = __float_as_uint(rest) & 0xffff0000u;
            lo[i] = __float_as_uint(rest - __uint_as_float(mid[i]));
        }
        if (MODE == MODE_GATHER && BT <= 2 && a.bits && tile == 0) {  // one half-word of the union mask per block
            const uint32_t w = __reduce_or_sync(0xffffffffu, part == 0 && bx < B ? kept << (4 * t) : 0u);
            if (lane == 0) {
                unsigned short *half = reinterpret_cast<unsigned short *>(a.bits);
                half[blk] = (unsigned short)w;
                if (blk == nblk - 1 && (blk & 1) == 0) half[blk + 1] = 0;
            }
        }
        // Up to two rows: lane column g = part * BT + row; four rows: leading and middle part side by side, then the last part
        // under the middle one; eight rows: one part each.
        uint2 f[3];
        if constexpr (BT <= 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i) hi[i] = part == 0 ? hi[i] : part == 1 ? mid[i] : lo[i];
        } else if constexpr (BT == 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                hi[i] = part == 0 ? hi[i] : mid[i];
                mid[i] = part == 0 ? 0u : lo[i];
            }
        }
        f[0] = make_uint2(__byte_perm(hi[0], hi[1], 0x7632), __byte_perm(hi[2], hi[3], 0x7632));
        f[1] = make_uint2(__byte_perm(mid[0], mid[1], 0x7632), __byte_perm(mid[2], mid[3], 0x7632));
        f[2] = make_uint2(__byte_perm(lo[0], lo[1], 0x7632), __byte_perm(lo[2], lo[3], 0x7632));
        auto mma_all = [&](float (&c0)[4], float (&c1)[4], const uint32_t (&w)[4]) {
            mma_k16<true>(c0, w, f[0].x, f[0].y);
            if constexpr (BT == 4) mma_k16<true>(c0, w, f[1].x, f[1].y);
            if constexpr (BT == 8) {
                mma_k16<true>(c1, w, f[2].x, f[2].y);
                mma_k16<true>(c1, w, f[1].x, f[1].y);
            }
        };
        // ---- weights: channel pairs (0, 1) and (2, 3) of columns 2 j and 2 j + 1
#pragma unroll
        for (int h = 0; h < CPT * WB / 16; ++h) {  // half-words of the row pieces: 2 columns (8-bit) or 4 columns (4-bit) each
            const uint32_t sel = (h & 1) ? 0x7632u : 0x5410u;
            const uint32_t t0 = __byte_perm(c.w[0].w[h >> 1], c.w[1].w[h >> 1], sel), t1 = __byte_perm(c.w[2].w[h >> 1], c.w[3].w[h >> 1], sel);
            const uint32_t u0 = t0 >> 8, u1 = t1 >> 8;
            if constexpr (WB == 8) {
                const uint32_t wa[4] = {qm_pair8(t0), qm_pair8(u0), qm_pair8(t1), qm_pair8(u1)};
                mma_all(acc[0][h], acc[NS - 1][h], wa);
            } else {
                const uint32_t wa[4] = {qm_pair4_lo(t0), qm_pair4_hi(t0), qm_pair4_lo(t1), qm_pair4_hi(t1)};
                mma_all(acc[0][2 * h], acc[NS - 1][2 * h], wa);
                const uint32_t wb[4] = {qm_pair4_lo(u0), qm_pair4_hi(u0), qm_pair4_lo(u1), qm_pair4_hi(u1)};
                mma_all(acc[0][2 * h + 1], acc[NS - 1][2 * h + 1], wb);
            }
        }
        if constexpr (WB == 4) {  // sum of the activations, like the codes times 1/64
            const uint32_t ones[4] = {0x3c803c80u, 0x3c803c80u, 0x3c803c80u, 0x3c803c80u};
            mma_all(ds[0], ds[NS - 1], ones);
        }
    };
    // 4-bit: y += scale (sum d (q - 8) - (zero - 8) sum d), once per group (and warp).  The scale of a group that a row has dropped
    // has no part in y, whatever it is: where a scale is not finite, sums of zero are left out (checking always: 2 % at groups of 32).
    auto flush_as = [&](int blk, auto careful_tag) {
        const int gi = blk / gb - g_lo;
        const float *sc = reinterpret_cast<const float *>(s_scale) + gi * QM_TN + lcol;
        const unsigned char *zp = s_zero + gi * QM_TN + lcol;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const float2 sv = *reinterpret_cast<const float2 *>(sc + 2 * j);
            const uint32_t zv = *reinterpret_cast<const unsigned short *>(zp + 2 * j);
            const float z0 = 8.0f - (float)(zv & 0xffu), z1 = 8.0f - (float)(zv >> 8);
#pragma unroll
            for (int q = 0; q < NS; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float sum = fmaf(i < 2 ? z0 : z1, ds[q][i & 1], acc[q][j][i]);
                    if (!decltype(careful_tag)::value || sum != 0.0f) y[q][j][i] = fmaf(i < 2 ? sv.x : sv.y, sum, y[q][j][i]);
                    acc[q][j][i] = 0.0f;
                }
        }
#pragma unroll
        for (int q = 0; q < NS; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) ds[q][i] = 0.0f;
    };
    auto flush = [&](int blk) {
        if (careful) flush_as(blk, std::true_type{});
        else flush_as(blk, std::false_type{});
    };
    bool promoted = false;
    auto add_slots = [&]() {
        const float4 *s_slot = reinterpret_cast<const float4 *>(smem + qm_smem(BT)) + threadIdx.x;  // [quad][thread]
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const float4 p = s_slot[j * FC_THREADS];
            acc[0][j][0] += p.x; acc[0][j][1] += p.y; acc[0][j][2] += p.z; acc[0][j][3] += p.w;
        }
    };
    auto promote = [&]() {
        if (promoted) add_slots();
        promoted = true;
        float4 *s_slot = reinterpret_cast<float4 *>(smem + qm_smem(BT)) + threadIdx.x;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            s_slot[j * FC_THREADS] = make_float4(acc[0][j][0], acc[0][j][1], acc[0][j][2], acc[0][j][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[0][j][i] = 0.0f;
        }
    };
    int left = WB == 4 ? gb - b_lo % gb : 0;  // blocks until the group ends
#pragma unroll 1
    for (int blk = b_lo; blk < b_hi; blk += PX) {
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            if (blk + i < b_hi) {
                process(cw[i % PW], ax[i], blk + i);
                if (blk + i + PW < b_hi) load_w(cw[i % PW], blk + i + PW);
                if (blk + i + PX < b_hi) load_x(ax[i], blk + i + PX);
                if (WB == 4 && (--left == 0 || blk + i + 1 == b_hi)) { flush(blk + i); left = gb; }
            }
        }
        if (WB == 8 && (blk + PX - b_lo) % QM_CHAIN == 0 && blk + PX < b_hi) promote();
    }
    if (WB == 8 && promoted) add_slots();

    // ---- parts of a batch row added smallest first, and the factor 64; this warp's partial tile -> shared memory
#pragma unroll
    for (int j = 0; j < NP; ++j) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float v;
            if constexpr (WB == 4) v = BT == 8 ? y[NS - 1][j][i] + y[0][j][i] : y[0][j][i];
            else v = BT == 8 ? acc[NS - 1][j][i] + acc[0][j][i] : acc[0][j][i];
            const int c = lcol + 2 * j + (i >> 1);
            float *dst = s_red + (size_t)(kg * BT) * QM_TN + c;
            if constexpr (BT == 1) {  // N columns 0, 1 (lane t = 0) and 2 (t = 1): the parts
                // element i & 1 of lane t is part 2 t + (i & 1)
                const float third = __shfl_xor_sync(0xffffffffu, v, 1);
                float second = 0.0f;
                if ((i & 1) == 0) second = WB == 4 ? y[0][j][i | 1] : acc[0][j][i | 1];
                if ((i & 1) == 0 && t == 0) dst[0] = 64.0f * ((third + second) + v);
            } else if constexpr (BT == 2) {  // lane t: part t of rows 0 and 1
                const float second = __shfl_xor_sync(0xffffffffu, v, 1), third = __shfl_xor_sync(0xffffffffu, v, 2);
                if (t == 0) dst[(i & 1) * QM_TN] = 64.0f * ((third + second) + v);
            } else if constexpr (BT == 4) {  // lanes 0, 1: leading part; lanes 2, 3: the rest
                const float rest = __shfl_xor_sync(0xffffffffu, v, 2);
                if (t < 2) dst[(2 * t + (i & 1)) * QM_TN] = 64.0f * (rest + v);
            } else {
                dst[(2 * t + (i & 1)) * QM_TN] = 64.0f * v;
            }
        }
    }
    if (S > 1) cluster_wait();  // every rank's barrier is initialised (all ranks arrived at kernel start)
    __syncthreads();
    if (S > 1) {
        reduce_send_round<BT, EPI_BIAS, QM_TN, NKG, BT>(s_red, 0, B, s, per, smem_addr(s_gather), bar);
        bool landed = false;
#pragma unroll 1
        for (uint32_t it = 0; it < TRIES && !landed; ++it) landed = mbarrier_try_wait(bar, 0);
        if (!landed && a.status) atomicCAS(a.status, 0, 2);  // never in a correct run; the result is then incomplete
    } else {
        float *owner[MAX_CLUSTER];
#pragma unroll
        for (int q = 0; q < MAX_CLUSTER; ++q) owner[q] = s_gather;
        reduce_push_round<BT, EPI_BIAS, QM_TN, NKG, BT>(s_red, 0, B, s, per, owner);
        __syncthreads();
    }
    finish_columns<true, BT, EPI_BIAS, QM_TN>(a, tile, s, per, s_gather, bias0, bias1);
}

// ---- host side ------------------------------------------------------------------------------------------------

template <int WB, int BT, int MODE, typename XT>
static cudaError_t launch_qm_b(const QmArgs &qa, cudaStream_t st) {
    static SmemOptIn opt_in;
    auto kern = fc_qm_kernel<WB, BT, MODE, XT>;
    cudaError_t e0 = ensure_dynamic_smem(kern, qm_smem(BT) + (WB == 4 ? QM_SCALE_MAX : qm_slot_bytes(WB, BT)), opt_in);
    if (e0 != cudaSuccess) return e0;
    // (the slots are there where a warp has more than one chain)
    const int blocks = (qa.f.K + 15) / 16, warps = qm_nkg(BT) * qa.f.S;
    const int extra = WB == 4 ? qa.sg * QM_GROUP_BYTES : (blocks + warps - 1) / warps > QM_CHAIN ? qm_slot_bytes(WB, BT) : 0;
    return launch_cluster(kern, dim3((qa.f.ldw + QM_TN - 1) / QM_TN, qa.f.S, qa.f.B > 8 ? 2 : 1), dim3(FC_THREADS), qm_smem(BT) + extra,
                          qa.f.S, st, g_tune.pdl != 0, qa);
}
template <int WB, int MODE, typename XT>
static cudaError_t launch_qm_x(const QmArgs &qa, cudaStream_t st) {
    const int B = qa.f.B;
    if (B == 1) return launch_qm_b<WB, 1, MODE, XT>(qa, st);
    if (B == 2) return launch_qm_b<WB, 2, MODE, XT>(qa, st);
    if (B <= 4) return launch_qm_b<WB, 4, MODE, XT>(qa, st);
    return launch_qm_b<WB, 8, MODE, XT>(qa, st);
}
template <int WB>
static cudaError_t launch_qm_w(int mode, int xkind, const QmArgs &qa, cudaStream_t st) {
    if (mode == MODE_DENSE) return xkind == 1 ? launch_qm_x<WB, MODE_DENSE, __nv_bfloat16>(qa, st) : launch_qm_x<WB, MODE_DENSE, __half>(qa, st);
    return xkind == 1 ? launch_qm_x<WB, MODE_GATHER, __nv_bfloat16>(qa, st) : launch_qm_x<WB, MODE_GATHER, __half>(qa, st);
}

// Split-K factor: the most CTAs that are all resident (two per SM), at least one block per rank.
static int qm_split(const QmArgs &a) {
    const int tiles = (a.f.ldw + QM_TN - 1) / QM_TN * (a.f.B > 8 ? 2 : 1), blocks = (a.f.K + 15) / 16;
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
// Groups that a rank can meet: its channels over the group size, one more where its range begins inside a group.
static int qm_groups(const QmArgs &a, int S) { return (((a.f.K + 15) / 16 + S - 1) / S * 16 + a.group - 1) / a.group + 1; }

bool qm_applicable(int wbits, const QmArgs &a) {
    if (a.f.K % 4 != 0 || a.f.ldw % 16 != 0 || a.f.B < 1 || a.f.B > 16 || a.f.hold_dependents) return false;
    if (wbits == 8) return aligned16(a.f.wscale);
    return qm_groups(a, qm_split(a)) * QM_GROUP_BYTES <= QM_SCALE_MAX;
}

int qm_blocks_per_warp(const QmArgs &a) {
    const int per = qm_nkg(1) * qm_split(a);
    return ((a.f.K + 15) / 16 + per - 1) / per;
}

cudaError_t launch_fc_qm(int wbits, int mode, int xkind, QmArgs a, cudaStream_t st) {
    a.f.S = qm_split(a);
    if (wbits == 4) a.sg = qm_groups(a, a.f.S);
    a.f.status = tc_status_ptr();
    return wbits == 8 ? launch_qm_w<8>(mode, xkind, a, st) : launch_qm_w<4>(mode, xkind, a, st);
}

}  // namespace scap
