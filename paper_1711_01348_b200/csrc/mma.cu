// Tensor-core kernel for contraction programs (contract.h), fp32 in and fp32 out.
//
// Every fp32 operand element is multiplied by 2^24 and split exactly into three bf16 values, 2^24 x = x1 + x2 + x3 (8 + 8 + 8
// significant bits, each part the rounded remainder of the ones before it), and a product is the sum of six bf16 products,
//     a b = a1 b1 + (a1 b2 + a2 b1) + (a1 b3 + a2 b2 + a3 b1).
// The factor keeps the parts of the smallest operands out of the subnormal numbers: bf16 ends where fp32 ends, so the third
// part of an |x| below 2^-109 would lose bits, then the second (relative error 2e-6 at 2^-115, 5e-4 at 1e-37); with it every
// fp32 value below 2^104 is split exactly, and the sums are multiplied by 2^-48, which is exact.
// What is left out, a2 b3 + a3 b2 + a3 b3, is at most 2^-23 |a b| and about 2^-26 |a b| in the mean square, below
// the rounding of the additions.  bf16 products are exact in the fp32 accumulator; the accumulator itself
// truncates, so a sum stays in it for one stage of 64 summation indices only (small products first, then four
// steps of a1 b1) and the stages are added up in fp32 registers with round-to-nearest.  Measured against float64
// (2-norm, normal operands): 0.8e-7 at 64 terms, 1.2e-7 at 1100, 1.3e-7 at 2048; chains of fp32 multiply-adds
// gave 4.2e-7 at 1100.  Where sums come out non-finite (an infinity times a zero part, an operand of 2^104 or more, a sum of
// 2^80 or more) the tile is evaluated again with fp32 multiply-adds from the operands themselves, so infinities and NaNs are
// those of the definition.
//
// One block per SM.  Warps 0-15 gather the operands of a stage through the offset tables (global -> registers, a
// whole stage ahead), split them and write them to shared memory in the 128-byte swizzled layout of the MMA
// (K-major when the lanes run along the rows, MN-major when they run along the summation index) or, for a row
// operand with its lanes along the rows, to tensor memory (the MMA then reads half as much shared memory); warp 16
// prepares the offset tables and issues the MMAs.  While stage s is multiplied, stage s + 1 is gathered and stage
// s - 1 is added to the registers.
//
// What bounds it: the six bf16 products of a 128 x 128 x 64 stage take 1536 clocks of the tensor core, gathering,
// splitting and adding up about 2900 clocks of the sixteen warps where both operands are gathered (4096 x 4096 x 4096: 775 us,
// 712 us without the MMAs, 543 us without the loads; 705 with the column operand split ahead by tad_mma_image_kernel).
// Measured against the fp32 multiply-add tiles of contract.cu: strided convolution 64 x 256 x 2048 with 1280 terms 1930 -> 455 us
// (190 TFLOP/s), 4096 x 2048 x 4096 product 1490 -> 346 us, 37 x 4907 x 159 convolution 26.6 -> 9.3 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "launch.h"
#include "contract.cuh"

namespace {

using namespace tadc;

constexpr int KS = TADC_KS;               // summation indices per stage
constexpr int NCW = 16;                   // warps that gather, split and add up
constexpr int NT = (NCW + 4) * 32;        // ... and the warpgroup of the MMA warp
// registers: 640 threads start with 96 each; the last warpgroup goes down to 32, the gathering ones up to 112
constexpr int REG_CONV = 112, REG_MMA = 32;
constexpr int BM = 128;
constexpr int KT = 3;                     // stages of the ring of k tables
constexpr int WAIT_LIMIT = 200000;        // polls after which a wait gives up

// ---- PTX ----
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
__device__ __forceinline__ void mbar_arrive(unsigned bar) { asm volatile("{ .reg .b64 t; mbarrier.arrive.shared::cta.b64 t, [%0]; }" ::"r"(bar) : "memory"); }
// false: this wait ran out, or another one of the block did (`failed`)
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int *failed)
{
    for (int i = 0; i < WAIT_LIMIT; ++i) {
        unsigned ok;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (__all_sync(0xffffffffu, ok)) return true;
        if (__any_sync(0xffffffffu, *failed != 0)) return false;
    }
    *failed = 1;
    return false;
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The whole warp runs these with warp-uniform operands and one elected lane issues: the descriptors then stay in
// uniform registers (issued from inside an if (lane == 0) every operand is moved there first: 154 clocks per MMA
// instead of the 68 the tensor core takes).
__device__ __forceinline__ void mma_ss(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, unsigned acc)
{
    asm volatile("{ .reg .pred p, q; elect.sync _|q, 0xffffffff; setp.ne.u32 p, %4, 0; @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_ts(unsigned d, unsigned a, unsigned long long b, unsigned idesc, unsigned acc)
{
    asm volatile("{ .reg .pred p, q; elect.sync _|q, 0xffffffff; setp.ne.u32 p, %4, 0; @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p; }" ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned bar)
{
    asm volatile("{ .reg .pred q; elect.sync _|q, 0xffffffff; @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0]; }" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(unsigned addr, unsigned (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st4(unsigned addr, const unsigned (&r)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// named barrier of some warps of a block (THREADS threads): the answer, the same for all, is whether x holds in any of them
template <int THREADS>
__device__ __forceinline__ bool any_of_warps(bool x)
{
    unsigned r;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; barrier.cta.red.or.pred q, 1, %2, p; selp.u32 %0, 1, 0, q; }" : "=r"(r) : "r"((unsigned)x), "n"(THREADS) : "memory");
    return r != 0;
}

// shared-memory matrix descriptor, 128-byte swizzle: leading / stride byte offsets in units of 16 bytes
__device__ __forceinline__ unsigned long long make_desc(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (unsigned long long)((addr & 0x3ffffu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) | ((unsigned long long)(sbo >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

// ---- gather ----
// An operand's stage is made of units of eight values along one direction (t), at one position of the other
// direction, the one the lanes run along (l):  offset = base(l) + tab(t0 + j), all tables in bytes.
//   TM_ROW   l = row, t = summation index    8 scalar loads, coalesced along the rows            -> K-major
//   TM_KVEC  t = summation index, contiguous and aligned: two 128-bit loads                      -> K-major
//   TM_K     l = summation index, t = row    8 scalar loads, coalesced along the summation index -> MN-major
//   TM_RVEC  t = row, contiguous and aligned: two 128-bit loads                                  -> MN-major
// (the row operand of the TM_ROW mode goes to tensor memory: a thread then takes the row of its own lane and the
// sixteen summation indices of MMA step warp / 4)
template <int MODE, int R, bool TMEM>
struct Unit {
    static constexpr bool KMAJOR = MODE == TM_ROW || MODE == TM_KVEC, VEC = MODE == TM_KVEC || MODE == TM_RVEC;
    int l, t0, dst;
    __device__ __forceinline__ Unit(int tid, int i)
    {
        if (TMEM) place(tid % BM, (tid / BM) * 2 + i);
        else at(tid + i * NCW * 32, KS / 8);
    }
    // the u-th unit of a stage of n_o octets of summation indices
    struct Among { int n_o; };
    __device__ __forceinline__ Unit(int u, Among a) { at(u, a.n_o); }
    __device__ __forceinline__ void at(int u, int n_o)
    {
        if (MODE == TM_ROW) place(u % R, u / R);
        else if (MODE == TM_KVEC) { const int q = n_o == KS / 8 ? u / (KS / 8) : (u * (65536 / n_o + 1)) >> 16; place(q, u - q * n_o); }   // (u < 1024)
        else if (MODE == TM_K) place(u % KS, u / KS);
        else place((u / 8) % KS, (u / (8 * KS)) * 8 + u % 8);
    }
    __device__ __forceinline__ void place(int lane_at, int o)
    {
        l = lane_at; t0 = o * 8;
        dst = (KMAJOR ? 0 : (o >> 3) * (KS * 128)) + l * 128 + (((o & 7) ^ (l & 7)) << 4);
    }
};

__device__ __forceinline__ float ldf(const float *__restrict__ src, unsigned byte_off)
{
    return __ldg(reinterpret_cast<const float *>(reinterpret_cast<const char *>(src) + byte_off));
}

// rows: offsets and guards of the tile's rows; kt: offsets and guards of the stage's summation indices (KS each)
template <bool CHECK, class U>
__device__ __forceinline__ void load_unit(float (&v)[8], const float *__restrict__ src, const U &u, const unsigned *row, const int *rowg,
                                          const unsigned *kt, const int *ktg, const unsigned gext)
{
    const unsigned base = U::KMAJOR ? row[u.l] : kt[u.l];
    const unsigned *tab = (U::KMAJOR ? kt : row) + u.t0;
    const int gbase = CHECK ? (U::KMAJOR ? rowg[u.l] : ktg[u.l]) : 0;
    const int *gtab = (U::KMAJOR ? ktg : rowg) + u.t0;
    if (U::VEC) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (!CHECK || (unsigned)(gbase + gtab[0]) < gext) {
            const float4 *p = reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(src) + (base + tab[0]));
            a = __ldg(p); b = __ldg(p + 1);
        }
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        return;
    }
    const uint4 t0 = *reinterpret_cast<const uint4 *>(tab), t1 = *reinterpret_cast<const uint4 *>(tab + 4);
    const unsigned t[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
    if (!CHECK) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = ldf(src, base + t[j]);
    } else {
        const int4 g0 = *reinterpret_cast<const int4 *>(gtab), g1 = *reinterpret_cast<const int4 *>(gtab + 4);
        const int g[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] = 0.f;
            if ((unsigned)(gbase + g[j]) < gext) v[j] = ldf(src, base + t[j]);
        }
    }
}

// Summation indices past the end of the range (left of them remain from the stage's first on) count as zeros.  They are
// loaded like all others - their table entries repeat the first index, rows past the edge of the matrix repeat the first
// row, whose offset has the alignment that vector loads need - and masked when they are used: a test at the load would
// wait for every unit's data in turn.
template <class U>
__device__ __forceinline__ void mask_unit(float (&v)[8], const U &u, const int left)
{
#pragma unroll
    for (int j = 0; j < 8; ++j) if ((U::KMAJOR ? u.t0 + j : u.l) >= left) v[j] = 0.f;
}

constexpr float SPLIT_SCALE = 0x1p24f, SUM_SCALE = 0x1p-48f;      // of an operand, of a sum of products

// two fp32 operations per instruction
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mul.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{ .reg .b64 x, y, w, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 w, {%6, %7}; fma.rn.f32x2 z, x, y, w; mov.b64 {%0, %1}, z; }"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}

// eight values times 2^24 -> three times eight bf16 (packed in pairs).  PAIRS: with two operations per instruction, which takes
// the scaling out of the tile kernel's time (4096 x 2048 x 4096 353 -> 346 us); the one-stage kernel, whose few gathering warps
// have no registers to spare for aligned pairs, is slower with it (8192 x 64 x 8192 153 -> 166 us).
template <bool PAIRS>
__device__ __forceinline__ void split_unit(const float (&v)[8], unsigned (&p1)[4], unsigned (&p2)[4], unsigned (&p3)[4])
{
    const float2 up = make_float2(SPLIT_SCALE, SPLIT_SCALE), minus = make_float2(-1.f, -1.f);
    auto less = [&](float2 x, unsigned h) {                    // what two rounded parts leave
        const float2 q = make_float2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u));
        return PAIRS ? fma2(q, minus, x) : make_float2(x.x - q.x, x.y - q.y);
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 w = make_float2(v[2 * j], v[2 * j + 1]), x = PAIRS ? mul2(w, up) : make_float2(w.x * SPLIT_SCALE, w.y * SPLIT_SCALE);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p1[j]) : "f"(x.y), "f"(x.x));
        const float2 r = less(x, p1[j]);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2[j]) : "f"(r.y), "f"(r.x));
        const float2 t = less(r, p2[j]);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p3[j]) : "f"(t.y), "f"(t.x));
    }
}

template <int BN, int MA, int MB>
struct MmaCfg {
    static constexpr bool TS = MA == TM_ROW, IMAGE = MB == TM_IMAGE;
    static constexpr int PART_A = BM * KS * 2, PART_B = BN * KS * 2;                 // bytes of one bf16 part of a stage
    static constexpr int STAGE = (TS ? 0 : 3 * PART_A) + 3 * PART_B;
    static constexpr int UA = BM * KS / 8 / (NCW * 32), UB = IMAGE ? 0 : BN * KS / 8 / (NCW * 32);   // units per thread
    static constexpr int COLS = BN * 32 / (NCW * 8);                                  // accumulator columns per thread
    static constexpr int TABLES = (BM + BN) * 12 + KT * KS * 16;                      // row offsets, guards, output offsets; k tables
    static constexpr size_t SMEM = 1024 + 2 * size_t(STAGE) + TABLES;
};

template <int BN, int MA, int MB>
__global__ void __launch_bounds__(NT, 1)
tad_mma_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs, const unsigned tiles_n)
{
    using C = MmaCfg<BN, MA, MB>;
    constexpr bool TS = C::TS;
    constexpr int COLS = C::COLS;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned long long bars[6 + KT];
    __shared__ unsigned tmem_base_s;
    __shared__ volatile int failed;
    const unsigned smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *stages = smem_raw + (smem0 - smem_u32(smem_raw));
    unsigned *rowA = reinterpret_cast<unsigned *>(stages + 2 * C::STAGE), *rowB = rowA + BM;          // bytes
    int *rowgA = reinterpret_cast<int *>(rowB + BN), *rowgB = rowgA + BM, *outM = rowgB + BN, *outN = outM + BM;
    int *ktab = outN + BN;                                   // per ring slot: offsets A, guards A, offsets B, guards B (KS each)
    const unsigned bar_full = smem_u32(&bars[0]), bar_done = smem_u32(&bars[2]), bar_tab = smem_u32(&bars[6]), bar_copy = smem_u32(&bars[4]);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const unsigned tile_n = blockIdx.x % tiles_n, tile_m = blockIdx.x / tiles_n;
    const unsigned ks = blockIdx.y, zb = blockIdx.z;
    const unsigned Mext = (unsigned)P.M.extent, Next = (unsigned)P.N.extent;
    const unsigned kbeg = ks * (unsigned)P.kchunk, kend = min((unsigned)P.K.extent, kbeg + (unsigned)P.kchunk);
    const int n_stages = (int)((kend - kbeg + KS - 1) / KS);
    const Parts z = decode(P.Z, zb);

    auto fill_ktab = [&](int s, int first) {                 // 32 threads, two entries each
        int *t = ktab + (s % KT) * 4 * KS;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = first + 32 * h;
            const unsigned k = kbeg + (unsigned)s * KS + e;
            Parts p{0, 0, 0, DEAD, DEAD};
            if (k < kend) p = decode(P.K, k);
            t[e] = p.a * 4; t[KS + e] = p.ga; t[2 * KS + e] = p.b * 4; t[3 * KS + e] = p.gb;
        }
    };
    if (warp == NCW) {
        if (lane == 0) {
            failed = 0;
            mbar_init(bar_full, NCW); mbar_init(bar_full + 8, NCW);
            mbar_init(bar_done, 1); mbar_init(bar_done + 8, 1);
            mbar_init(bar_copy, 1); mbar_init(bar_copy + 8, 1);
            for (int i = 0; i < KT; ++i) mbar_init(bar_tab + 8 * i, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp < NCW) {
        if (warp < KT) fill_ktab(warp, lane);
        for (int r = tid; r < BM; r += NCW * 32) {
            const unsigned m = tile_m * BM + r;
            const Parts p = decode(P.M, m < Mext ? m : 0u);
            rowA[r] = (unsigned)(P.baseA + z.a + p.a) * 4u; rowgA[r] = m < Mext ? P.guardA_c0 + z.ga + p.ga : DEAD; outM[r] = p.o;
        }
        for (int r = tid - BM; r < BN; r += NCW * 32) {
            if (r < 0) continue;
            const unsigned n = tile_n * BN + r;
            const Parts p = decode(P.N, n < Next ? n : 0u);
            rowB[r] = (unsigned)(P.baseB + z.b + p.b) * 4u; rowgB[r] = n < Next ? P.guardB_c0 + z.gb + p.gb : DEAD; outN[r] = p.o;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    tad_wait_previous();                                     // (nothing above reads memory)
    const unsigned tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    constexpr unsigned TMEM_A = 2 * BN;                      // columns of the row operand's stages (TS): 3 x 32 each
    bool ok = true;

    if (warp >= NCW) {
        // ---- MMA warp ----
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_MMA));
        const int n_stages_mma = warp == NCW ? n_stages : 0;
        constexpr bool a_k = MA == TM_ROW || MA == TM_KVEC, b_k = MB == TM_ROW || MB == TM_KVEC || MB == TM_IMAGE;
        const unsigned n_pad = min((unsigned)BN, (Next - tile_n * BN + 15u) / 16u * 16u);
        const unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | (a_k ? 0u : 1u << 15) | (b_k ? 0u : 1u << 16) | ((n_pad >> 3) << 17) | ((BM >> 4) << 24);
        // K-major: eight rows of 128 bytes per repeat; MN-major: blocks of 64 rows, eight summation indices per repeat
        constexpr unsigned stepA = a_k ? 32u : 16u * 128u, stepB = b_k ? 32u : 16u * 128u;
        constexpr unsigned lboA = a_k ? 16u : KS * 128u, lboB = b_k ? 16u : KS * 128u;
        int issued = 0;
        for (int s = 0; s < n_stages_mma && ok; ++s) {
            ok = mbar_wait(bar_full + 8 * (s & 1), (s >> 1) & 1, &failed);
            if (C::IMAGE) ok = ok && mbar_wait(bar_copy + 8 * (s & 1), (s >> 1) & 1, &failed);
            fence_after();
            if (!ok) break;
            const unsigned sm = smem0 + (s & 1) * C::STAGE;
            const unsigned d = tmem + (s & 1) * BN;
            const unsigned ta = tmem + TMEM_A + (s & 1) * 96;
            const int steps = (int)min((unsigned)KS / 16u, (kend - kbeg - (unsigned)s * KS + 15u) / 16u);
            const unsigned long long db = make_desc(sm + (TS ? 0 : 3 * C::PART_A), lboB, 1024u), da = make_desc(sm, lboA, 1024u);
            // (a3 b1) (a2 b2) (a1 b3) (a2 b1) (a1 b2) (a1 b1)
            constexpr int PA[6] = {2, 1, 0, 1, 0, 0}, PB[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
            for (int pr = 0; pr < 6; ++pr)
#pragma unroll
                for (int kk = 0; kk < KS / 16; ++kk) {
                    if (kk >= steps) continue;
                    const unsigned long long bd = db + ((PB[pr] * C::PART_B + kk * stepB) >> 4);
                    if (TS) mma_ts(d, ta + PA[pr] * 32 + kk * 8, bd, idesc, pr + kk > 0);
                    else mma_ss(d, da + ((PA[pr] * C::PART_A + kk * stepA) >> 4), bd, idesc, pr + kk > 0);
                }
            mma_commit(bar_done + 8 * (s & 1));
            ++issued;
            // every warp has read the tables up to stage s + 1: the slot of stage s takes stage s + KT
            if (s + KT < n_stages) {
                fill_ktab(s + KT, lane);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tab + 8 * (s % KT));
            }
        }
        // MMAs of a block that gave up still read its shared memory: wait for them (again with a limit)
        if (!ok)
            for (int s = max(0, issued - 2); s < issued; ++s)
                for (int i = 0; i < WAIT_LIMIT; ++i) {
                    unsigned done;
                    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }" : "=r"(done) : "r"(bar_done + 8 * (s & 1)), "r"((s >> 1) & 1) : "memory");
                    if (__all_sync(0xffffffffu, done)) break;
                }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REG_CONV));
        float acc[COLS];
#pragma unroll
        for (int j = 0; j < COLS; ++j) acc[j] = 0.f;
        const int quad = warp & 3, col0 = (warp >> 2) * COLS;
        const float *__restrict__ A = ptrs.in[P.ptrA];
        const float *__restrict__ B = ptrs.in[P.ptrB];
        const unsigned gextA = (unsigned)P.guardA_ext, gextB = (unsigned)P.guardB_ext;
        float va[C::UA][8], vb[C::UB > 0 ? C::UB : 1][8];
        auto load = [&](float (&v)[8], int i, int s, bool second, bool check) {
            const unsigned *t = reinterpret_cast<const unsigned *>(ktab + (s % KT) * 4 * KS) + (second ? 2 * KS : 0);
            const int *tg = reinterpret_cast<const int *>(t + KS);
            if constexpr (C::IMAGE) second = false;
            if (!second) {
                const Unit<MA, BM, TS> u(tid, i);
                if (check) load_unit<true>(v, A, u, rowA, rowgA, t, tg, gextA);
                else load_unit<false>(v, A, u, rowA, rowgA, t, tg, gextA);
            } else {
                const Unit<C::IMAGE ? (int)TM_ROW : MB, BN, false> u(tid, i);
                if (check) load_unit<true>(v, B, u, rowB, rowgB, t, tg, gextB);
                else load_unit<false>(v, B, u, rowB, rowgB, t, tg, gextB);
            }
        };
        // the column operand's image of stage s, as one bulk copy behind the row operand's buffer (its MMAs of stage s - 2 are done)
        int copies = 0;
        auto copy_image = [&](int s) {
            if (!C::IMAGE || warp != 0 || s >= n_stages) return;
            ++copies;
            if (lane == 0) {
                const size_t total = ((size_t)P.K.extent + KS - 1) / KS;
                const unsigned char *from = ptrs.image +
                                   (((size_t)zb * tiles_n + tile_n) * total + kbeg / KS + s) * (3 * C::PART_B);
                const unsigned to = smem0 + (s & 1) * C::STAGE + (TS ? 0 : 3 * C::PART_A), bar = bar_copy + 8 * (s & 1);
                asm volatile("fence.proxy.async.global;" ::: "memory");   // (the image is another kernel's plain stores)
                asm volatile("{ .reg .b64 t; mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1; }" ::"r"(bar), "r"(3 * C::PART_B) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to), "l"(from), "r"(3 * C::PART_B), "r"(bar) : "memory");
            }
            __syncwarp();
        };
        copy_image(0);
        copy_image(1);
        // adds the finished stage s to the registers
        auto collect = [&](int s) {
            ok = ok && mbar_wait(bar_done + 8 * (s & 1), (s >> 1) & 1, &failed);
            fence_after();
            if (!ok) return;
            copy_image(s + 2);
            const unsigned at = tmem + ((unsigned)(quad * 32) << 16) + (s & 1) * BN + col0;
#pragma unroll
            for (int c = 0; c < COLS; c += 16) {
                unsigned r[16];
                tmem_ld16(at + c, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[c + j] += __uint_as_float(r[j]);
            }
            fence_before();
        };
#pragma unroll
        for (int i = 0; i < C::UA; ++i) load(va[i], i, 0, false, P.guardA != 0);
#pragma unroll
        for (int i = 0; i < C::UB; ++i) load(vb[i], i, 0, true, P.guardB != 0);
        for (int s = 0; s < n_stages && ok; ++s) {
            unsigned char *st = stages + (s & 1) * C::STAGE;
            const bool more = s + 1 < n_stages;
            const int left = (int)min((unsigned)KS, kend - kbeg - (unsigned)s * KS);
            if (more && s + 1 >= KT) ok = mbar_wait(bar_tab + 8 * ((s + 1) % KT), ((s + 1) / KT - 1) & 1, &failed);
            if (!ok) break;
            if (left < KS) {
#pragma unroll
                for (int i = 0; i < C::UA; ++i) mask_unit(va[i], Unit<MA, BM, TS>(tid, i), left);
#pragma unroll
                for (int i = 0; i < C::UB; ++i) mask_unit(vb[i], Unit<C::IMAGE ? (int)TM_ROW : MB, BN, false>(tid, i), left);
            }
            unsigned p1[4], p2[4], p3[4];
#pragma unroll
            for (int i = 0; i < C::UA; ++i) {
                split_unit<true>(va[i], p1, p2, p3);
                if (more) load(va[i], i, s + 1, false, P.guardA != 0);
                const Unit<MA, BM, TS> u(tid, i);
                if (TS) {
                    const unsigned at = tmem + ((unsigned)(quad * 32) << 16) + TMEM_A + (s & 1) * 96 + u.t0 / 2;
                    tmem_st4(at, p1); tmem_st4(at + 32, p2); tmem_st4(at + 64, p3);
                } else {
                    *reinterpret_cast<uint4 *>(st + u.dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
                    *reinterpret_cast<uint4 *>(st + C::PART_A + u.dst) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
                    *reinterpret_cast<uint4 *>(st + 2 * C::PART_A + u.dst) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
                }
            }
            st += TS ? 0 : 3 * C::PART_A;
#pragma unroll
            for (int i = 0; i < C::UB; ++i) {
                split_unit<true>(vb[i], p1, p2, p3);
                if (more) load(vb[i], i, s + 1, true, P.guardB != 0);
                const Unit<C::IMAGE ? (int)TM_ROW : MB, BN, false> u(tid, i);
                *reinterpret_cast<uint4 *>(st + u.dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
                *reinterpret_cast<uint4 *>(st + C::PART_B + u.dst) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
                *reinterpret_cast<uint4 *>(st + 2 * C::PART_B + u.dst) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
            }
            if (TS) { tmem_wait_st(); fence_before(); }
            fence_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full + 8 * (s & 1));
            if (s > 0) collect(s - 1);
        }
        if (n_stages > 0) collect(n_stages - 1);
        // copies of a block that gave up still write its shared memory: wait for them (again with a limit)
        if (!ok)
            for (int s = max(0, copies - 2); s < copies; ++s)
                for (int i = 0; i < WAIT_LIMIT; ++i) {
                    unsigned there;
                    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }" : "=r"(there) : "r"(bar_copy + 8 * (s & 1)), "r"((s >> 1) & 1) : "memory");
                    if (__all_sync(0xffffffffu, there)) break;
                }
        // ---- outputs: a thread holds COLS columns of its row; consecutive lanes are consecutive rows ----
        const unsigned rl = (unsigned)(quad * 32 + lane), m = tile_m * BM + rl, n0 = tile_n * BN + col0;
        const int live = m < Mext && n0 < Next ? (int)min((unsigned)COLS, Next - n0) : 0;
        bool odd = !ok;
#pragma unroll
        for (int j = 0; j < COLS; ++j) odd = odd || (j < live && !(fabsf(acc[j]) <= 3.0e38f));
        odd = __any_sync(0xffffffffu, odd);
        if (!odd && live) {
#pragma unroll
            for (int j = 0; j < COLS; ++j) acc[j] *= SUM_SCALE;
            if (P.ksplit > 1) {
                // plane of this share: columns outermost, so that the lanes write consecutive elements
                float *dst = ptrs.part + ((size_t)zb * (unsigned)P.ksplit + ks) * Next * Mext + (size_t)n0 * Mext + m;
#pragma unroll
                for (int j = 0; j < COLS; ++j) if (j < live) dst[(size_t)j * Mext] = acc[j];
            } else {
                const int ob = P.baseO + z.o + outM[rl];
                const float scale = P.scale;
                unsigned off[COLS];
#pragma unroll
                for (int j = 0; j < COLS; ++j) { acc[j] *= scale; off[j] = (unsigned)(ob + outN[col0 + (j < live ? j : 0)]); }
#define TAD_EPI_ALL(expr) _Pragma("unroll") for (int j = 0; j < COLS; ++j) { expr; }
                for (int e = 0; e < P.n_epi; ++e) {
                    const int op = P.epi_op[e];
                    const float imm = P.epi_imm[e];
                    const float *__restrict__ src = (op == TE_MUL_LOAD || op == TE_ADD_LOAD) ? ptrs.in[P.epi_ptr[e]] : nullptr;
                    const int sb = P.epi_base[e];
                    switch (op) {
                    case TE_NEG: TAD_EPI_ALL(acc[j] = -acc[j]) break;
                    case TE_EXP: TAD_EPI_ALL(acc[j] = __expf(acc[j])) break;
                    case TE_MULC: TAD_EPI_ALL(acc[j] *= imm) break;
                    case TE_ADDC: TAD_EPI_ALL(acc[j] += imm) break;
                    case TE_SQR: TAD_EPI_ALL(acc[j] *= acc[j]) break;
                    case TE_TANH: TAD_EPI_ALL(acc[j] = own_tanh(acc[j])) break;
                    case TE_MUL_LOAD: TAD_EPI_ALL(acc[j] *= __ldg(src + (unsigned)(sb + (int)off[j]))) break;
                    case TE_ADD_LOAD: TAD_EPI_ALL(acc[j] += __ldg(src + (unsigned)(sb + (int)off[j]))) break;
                    default: break;
                    }
                }
#undef TAD_EPI_ALL
                float *__restrict__ out = ptrs.out;
                if (P.accumulate) {
#pragma unroll
                    for (int j = 0; j < COLS; ++j) if (j < live) out[off[j]] += acc[j];
                } else {
#pragma unroll
                    for (int j = 0; j < COLS; ++j) if (j < live) out[off[j]] = acc[j];
                }
            }
        }
        // Warps with an infinite or NaN sum: their outputs once more, by the whole block, with fp32 multiply-adds from the operands
        // themselves, 32 summation indices at a time through shared memory (the stages' place: every MMA and copy into it has been
        // waited for).  Outputs with a NaN among their operands are NaN, and where that is all of them no sum is formed.
        // Strided convolution 64 x 256 x 2048 with 1280 terms, NaN operands / one infinity / infinities: 1.6 / 0.5 / 6.6 ms; every output from its
        // own terms 103 / 7.4 / 103 ms, the multiply-add tiles of contract.cu 1.93 ms whatever the values.
        if (any_of_warps<NCW * 32>(odd)) {
            constexpr int RK = 32, LA = BM + 4, LB = BN + 4, PER = BM * RK / (NCW * 32), PART = 16;
            static_assert((LA + LB) * RK * 4 + 4 * RK * 4 + (BM + BN) * 4 <= 2 * C::STAGE, "room for the operands");
            float *ta = reinterpret_cast<float *>(stages), *tb = ta + RK * LA;
            int *rt = reinterpret_cast<int *>(tb + RK * LB);                        // offsets A, guards A, offsets B, guards B
            int *nans = rt + 4 * RK;                                                // rows of A, columns of B that hold a NaN
            constexpr bool a_rows = MA == TM_ROW;
            const bool b_rows = P.modeB == TM_ROW || P.modeB == TM_RVEC;
            for (int r = tid; r < BM + BN; r += NCW * 32) nans[r] = 0;
            // indices k0 .. k0 + 31 of one operand (rows, its first guard part, its tables), zero where there is none; returns which are NaN
            auto stage = [&](const float *src, bool rows, auto size, int ld, float *dst, int *flags, const unsigned *row, const int *rowg, const int *t, unsigned gext) {
                constexpr int n = decltype(size)::value;
                float x[PER];                                  // (all loads are under way before the first is stored)
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const int e = tid + i * NCW * 32, r = (rows ? e % n : e / RK) % n, k = (rows ? e / n : e) % RK;
                    x[i] = 0.f;
                    if (e < n * RK && (unsigned)(rowg[r] + t[RK + k]) < gext) x[i] = ldf(src, row[r] + (unsigned)t[k]);
                }
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    const int e = tid + i * NCW * 32, r = rows ? e % n : e / RK, k = rows ? e / n : e % RK;
                    if (e >= n * RK) continue;
                    dst[k * ld + r] = x[i];
                    if (x[i] != x[i]) flags[r] = 1;
                }
            };
            // pass -1 looks for NaNs, pass q forms the sums of the q-th sixteen columns of every warp
#pragma unroll 1
            for (int pass = -1; pass < COLS / PART; ++pass) {
                float sum[PART];
#pragma unroll
                for (int j = 0; j < PART; ++j) sum[j] = 0.f;
#pragma unroll 1
                for (unsigned k0 = kbeg; k0 < kend; k0 += RK) {
                    any_of_warps<NCW * 32>(false);             // (the block is done with the indices before)
                    if (tid < RK) {
                        Parts p{0, 0, 0, DEAD, DEAD};
                        if (k0 + tid < kend) p = decode(P.K, k0 + tid);
                        rt[tid] = p.a * 4; rt[RK + tid] = p.ga; rt[2 * RK + tid] = p.b * 4; rt[3 * RK + tid] = p.gb;
                    }
                    any_of_warps<NCW * 32>(false);
                    stage(ptrs.in[P.ptrA], a_rows, std::integral_constant<int, BM>{}, LA, ta, nans, rowA, rowgA, rt, (unsigned)P.guardA_ext);     // (extent 1 without a guard)
                    stage(ptrs.in[P.ptrB], b_rows, std::integral_constant<int, BN>{}, LB, tb, nans + BM, rowB, rowgB, rt + 2 * RK, (unsigned)P.guardB_ext);
                    if (pass < 0) continue;
                    any_of_warps<NCW * 32>(false);
                    const int kn = (int)min((unsigned)RK, kend - k0);
                    if (!odd) continue;
#pragma unroll 4
                    for (int k = 0; k < kn; ++k) {
                        const float x = ta[k * LA + rl];
                        const float4 *y = reinterpret_cast<const float4 *>(tb + k * LB + col0 + pass * PART);
#pragma unroll
                        for (int c = 0; c < PART / 4; ++c) {
                            const float4 q = y[c];
                            sum[4 * c] = fmaf(x, q.x, sum[4 * c]); sum[4 * c + 1] = fmaf(x, q.y, sum[4 * c + 1]);
                            sum[4 * c + 2] = fmaf(x, q.z, sum[4 * c + 2]); sum[4 * c + 3] = fmaf(x, q.w, sum[4 * c + 3]);
                        }
                    }
                }
                bool left = false;                             // some output to be summed
                if (pass < 0) {
                    any_of_warps<NCW * 32>(false);
                    if (odd && !nans[rl]) for (int j = 0; j < live; ++j) left = left || !nans[BM + col0 + j];
                    left = any_of_warps<NCW * 32>(left);
                    if (left) continue;
                }
                // (no output to be summed: one turn stores the NaNs of all columns)
#pragma unroll 1
                for (int c = pass < 0 ? 0 : pass * PART; odd && c < (pass < 0 ? COLS : (pass + 1) * PART); c += PART) {
#pragma unroll
                    for (int j = 0; j < PART; ++j) {
                        if (c + j >= live) continue;
                        const float v = nans[rl] || nans[BM + col0 + c + j] ? __int_as_float(0x7fffffff) : sum[j];
                        if (P.ksplit > 1) ptrs.part[((size_t)zb * (unsigned)P.ksplit + ks) * Next * Mext + (size_t)(n0 + c + j) * Mext + m] = v;
                        else {
                            const unsigned off = (unsigned)(P.baseO + z.o + outM[rl] + outN[col0 + c + j]);
                            const float r = epilogue(P, ptrs, v * P.scale, off);
                            ptrs.out[off] = P.accumulate ? ptrs.out[off] + r : r;
                        }
                    }
                }
                if (pass < 0) break;
            }
        }
        fence_before();
    }
    __syncthreads();
    if (warp == NCW) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------------------
// Contractions of one stage (up to 64 summation indices): forward passes and staged adjoints of expressions whose sum
// was pushed inside, where the work is the epilogue and the traffic of the outputs.  With a block per tile, gather,
// split, MMA and epilogue of a tile ran one after another (8192 x 8192 x 34: 220 us for 268 MB of output).  Here a block
// walks a run of tiles with the row tile fastest and its warps work on different tiles at a time:
//   warps 16-22  gather and split the row operand of the next tile (and the column operand where the column tile changes)
//   warp 23      issues the MMAs of the current one into one of two accumulators
//   warps 0-15   read the accumulator of the tile before (32 rows x 32 columns each), apply the epilogue and store; the
//                values of a tensor that the epilogue reads are loaded while the MMAs still run
// ---------------------------------------------------------------------------------------------------------
constexpr int SE = 16, SC = 7, SNT = (SE + SC + 1) * 32;    // epilogue and gather warps; six warps per scheduler leave 80 registers each

struct ShortCfg {
    static constexpr int PART = BM * KS * 2, OPERAND = 3 * PART;
    static constexpr int MAX_TILES = 1024;      // of a block: the marks of its pieces must fit
    static constexpr int TABLES = 2 * BM * 8 + 2 * BM * 8 + 4 * KS * 4 + SE * 64 * 4 + SE * MAX_TILES / 4;    // row tables of both operands (twice), k tables, output columns, marks
    static constexpr size_t SMEM = 1024 + 4 * size_t(OPERAND) + TABLES;
};

template <int MA, int MB>
__global__ void __launch_bounds__(SNT, 1)
tad_mma_short_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs, const unsigned tiles_m, const unsigned tiles_n, const unsigned n_items)
{
    tad_wait_previous();
    using C = ShortCfg;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned long long bars[6];
    __shared__ unsigned tmem_base_s;
    __shared__ volatile int failed;
    const unsigned smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *bufs = smem_raw + (smem0 - smem_u32(smem_raw));                     // A0, A1, B0, B1
    unsigned *rowoff = reinterpret_cast<unsigned *>(bufs + 4 * C::OPERAND);            // [operand][buffer][row], then the guards likewise
    int *rowgrd = reinterpret_cast<int *>(rowoff + 4 * BM);
    int *ktab = rowgrd + 4 * BM;                                                       // offsets A, guards A, offsets B, guards B
    int *outN = ktab + 4 * KS;                                                         // per epilogue warp: output offsets of its 32 columns, twice
    unsigned *marks = reinterpret_cast<unsigned *>(outN + SE * 64) + (threadIdx.x >> 5) * (ShortCfg::MAX_TILES / 16);   // per epilogue warp: two pieces of every tile
    const unsigned bar_full = smem_u32(&bars[0]), bar_done = smem_u32(&bars[2]), bar_free = smem_u32(&bars[4]);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const unsigned Mext = (unsigned)P.M.extent, Next = (unsigned)P.N.extent, K = (unsigned)P.K.extent;
    const unsigned per = n_items / gridDim.x, extra = n_items % gridDim.x;
    const unsigned first = blockIdx.x * per + min(blockIdx.x, extra);
    const unsigned strip0 = first / tiles_m, row0 = first - strip0 * tiles_m;          // strip: column tile and batch index
    const int n_tiles = (int)(per + (blockIdx.x < extra ? 1u : 0u));
    const int kpad = (int)((K + 15u) & ~15u);
    if (warp == SE + SC) {
        if (lane == 0) {
            failed = 0;
            for (int i = 0; i < 2; ++i) { mbar_init(bar_full + 8 * i, SC); mbar_init(bar_done + 8 * i, 1); mbar_init(bar_free + 8 * i, SE); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_base_s)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (tid < KS) {
        Parts p{0, 0, 0, DEAD, DEAD};
        if ((unsigned)tid < K) p = decode(P.K, tid);
        ktab[tid] = p.a * 4; ktab[KS + tid] = p.ga; ktab[2 * KS + tid] = p.b * 4; ktab[3 * KS + tid] = p.gb;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    bool ok = true;
    if (warp == SE + SC) {
        // ---- MMA warp ----
        constexpr bool a_k = MA == TM_ROW || MA == TM_KVEC, b_k = MB == TM_ROW || MB == TM_KVEC;
        constexpr unsigned stepA = a_k ? 32u : 16u * 128u, stepB = b_k ? 32u : 16u * 128u;
        constexpr unsigned lboA = a_k ? 16u : KS * 128u, lboB = b_k ? 16u : KS * 128u;
        constexpr int PA[6] = {2, 1, 0, 1, 0, 0}, PB[6] = {0, 1, 2, 0, 1, 0};      // small products first
        unsigned strip = strip0, tile_m = row0;
        int q = 0, t = 0;
        for (; t < n_tiles && ok; ++t) {
            if (t > 0 && ++tile_m == tiles_m) { tile_m = 0; ++strip; ++q; }
            ok = mbar_wait(bar_full + 8 * (t & 1), (t >> 1) & 1, &failed);
            if (ok && t >= 2) ok = mbar_wait(bar_free + 8 * (t & 1), ((t - 2) >> 1) & 1, &failed);
            fence_after();
            if (!ok) break;
            const unsigned n_pad = min((unsigned)BM, (Next - (strip % tiles_n) * BM + 15u) / 16u * 16u);
            const unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | (a_k ? 0u : 1u << 15) | (b_k ? 0u : 1u << 16) | ((n_pad >> 3) << 17) | ((BM >> 4) << 24);
            const unsigned long long da = make_desc(smem0 + (t & 1) * C::OPERAND, lboA, 1024u), db = make_desc(smem0 + (2 + (q & 1)) * C::OPERAND, lboB, 1024u);
            const int steps = kpad / 16;
#pragma unroll
            for (int pr = 0; pr < 6; ++pr)
#pragma unroll
                for (int kk = 0; kk < KS / 16; ++kk) {
                    if (kk >= steps) continue;
                    mma_ss(tmem + (t & 1) * BM, da + ((PA[pr] * C::PART + kk * stepA) >> 4), db + ((PB[pr] * C::PART + kk * stepB) >> 4), idesc, pr + kk > 0);
                }
            mma_commit(bar_done + 8 * (t & 1));
        }
        // MMAs of a block that gave up still read its shared memory: wait for them (again with a limit)
        if (!ok)
            for (int s = max(0, t - 2); s < t; ++s)
                for (int i = 0; i < WAIT_LIMIT; ++i) {
                    unsigned done;
                    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }" : "=r"(done) : "r"(bar_done + 8 * (s & 1)), "r"((s >> 1) & 1) : "memory");
                    if (__all_sync(0xffffffffu, done)) break;
                }
    } else if (warp >= SE) {
        // ---- gathering warps ----
        const int ct = tid - SE * 32;
        constexpr int CT = SC * 32, UNITS = BM * KS / 8, UN = (UNITS + CT - 1) / CT;
        unsigned tile_m = row0, strip = strip0, tile_n = 0;
        int q = -1;
        Parts z{0, 0, 0, 0, 0};
        auto gather = [&](auto mode, const float *__restrict__ src, const unsigned *row, const int *rowg, const int *kt, bool check, unsigned gext, unsigned char *dst) {
            constexpr int MODE = decltype(mode)::value;
            using U = Unit<MODE, BM, false>;
            const unsigned *kto = reinterpret_cast<const unsigned *>(kt);
            // vectors along the summation index: the octets past its end are no units (34 indices: four rounds of units instead of five)
            const int n_o = MODE == TM_KVEC ? kpad / 8 : KS / 8, units = MODE == TM_KVEC ? BM * n_o : UNITS;
            float v[UN][8];
#pragma unroll
            for (int i = 0; i < UN; ++i) {
                const U u(ct + i * CT, typename U::Among{n_o});
                if (ct + i * CT >= units || (U::KMAJOR ? u.t0 : u.l) >= kpad) continue;
                if (check) load_unit<true>(v[i], src, u, row, rowg, kto, kt + KS, gext);
                else load_unit<false>(v[i], src, u, row, rowg, kto, kt + KS, gext);
            }
#pragma unroll
            for (int i = 0; i < UN; ++i) {
                const U u(ct + i * CT, typename U::Among{n_o});
                if (ct + i * CT >= units || (U::KMAJOR ? u.t0 : u.l) >= kpad) continue;
                unsigned p1[4], p2[4], p3[4];
                if (kpad != (int)K) mask_unit(v[i], u, (int)K);
                split_unit<false>(v[i], p1, p2, p3);
                *reinterpret_cast<uint4 *>(dst + u.dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
                *reinterpret_cast<uint4 *>(dst + C::PART + u.dst) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
                *reinterpret_cast<uint4 *>(dst + 2 * C::PART + u.dst) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
            }
        };
        for (int t = 0; t < n_tiles && ok; ++t) {
            // the MMAs of tile t - 2 are done: its row buffer, and every column buffer but the last two, are free
            if (t >= 2) ok = mbar_wait(bar_done + 8 * (t & 1), ((t - 2) >> 1) & 1, &failed);
            const bool fresh = t == 0 || ++tile_m == tiles_m;
            if (fresh) {
                if (t > 0) { tile_m = 0; ++strip; }
                ++q;
                tile_n = strip % tiles_n;
                z = decode(P.Z, strip / tiles_n);
            }
            for (int r = ct; r < (fresh ? 2 : 1) * BM; r += CT) {
                if (r < BM) {
                    const unsigned m = tile_m * BM + r;
                    const Parts p = decode(P.M, m < Mext ? m : 0u);
                    rowoff[(t & 1) * BM + r] = (unsigned)(P.baseA + z.a + p.a) * 4u;
                    rowgrd[(t & 1) * BM + r] = m < Mext ? P.guardA_c0 + z.ga + p.ga : DEAD;
                } else {
                    const unsigned n = tile_n * BM + (r - BM);
                    const Parts p = decode(P.N, n < Next ? n : 0u);
                    rowoff[(2 + (q & 1)) * BM + r - BM] = (unsigned)(P.baseB + z.b + p.b) * 4u;
                    rowgrd[(2 + (q & 1)) * BM + r - BM] = n < Next ? P.guardB_c0 + z.gb + p.gb : DEAD;
                }
            }
            // (a warp that is here has read the tables of the tile before: the tables alternate, one barrier per tile is enough.)
            // Every warp comes here whatever its wait said, and all leave together if one ran out: a warp that left on its own
            // would leave the others in this barrier for ever, and a wait can end either way when the MMAs finish at its limit.
            if (any_of_warps<CT>(!ok)) { ok = false; break; }
            if (fresh)
                gather(std::integral_constant<int, MB>{}, ptrs.in[P.ptrB], rowoff + (2 + (q & 1)) * BM, rowgrd + (2 + (q & 1)) * BM, ktab + 2 * KS,
                       P.guardB != 0, (unsigned)P.guardB_ext, bufs + (2 + (q & 1)) * C::OPERAND);
            gather(std::integral_constant<int, MA>{}, ptrs.in[P.ptrA], rowoff + (t & 1) * BM, rowgrd + (t & 1) * BM, ktab,
                   P.guardA || (tile_m + 1) * BM > Mext, (unsigned)P.guardA_ext, bufs + (t & 1) * C::OPERAND);
            fence_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full + 8 * (t & 1));
        }
    } else {
        // ---- epilogue warps: 32 rows x 32 columns of a tile each ----
        const int quad = warp & 3, col0 = (warp >> 2) * 32;
        int *cols = outN + warp * 64;                          // output offsets of this warp's columns, of an even and an odd column tile
        for (int i = lane; i < (n_tiles + 15) / 16; i += 32) marks[i] = 0;
        __syncwarp();
        int pre = -1;                                          // the epilogue step whose tensor is loaded ahead
        for (int e = P.n_epi - 1; e >= 0; --e) if (P.epi_op[e] == TE_MUL_LOAD || P.epi_op[e] == TE_ADD_LOAD) pre = e;
        // A tile is two pieces of 16 columns.  The values that the epilogue reads for a piece are loaded a piece ahead (the
        // ones of a tile's first piece while its MMAs still run); one copy of the code serves both pieces.
        unsigned tile_m = row0, strip = strip0, n0 = 0;
        int ncol = 0, ob = 0;                                  // columns of this warp, the same for all its lanes; the row's output offset
        bool row = false;
        int zo = 0;
        float w[16], wn[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) { w[j] = 0.f; wn[j] = 0.f; }
        const float *__restrict__ src0 = pre >= 0 ? ptrs.in[P.epi_ptr[pre]] + (ptrdiff_t)P.epi_base[pre] : nullptr;
        const bool pre_mul = pre >= 0 && P.epi_op[pre] == TE_MUL_LOAD;
        const float scale = P.scale * SUM_SCALE;               // (exact: the host keeps smaller constants away from this kernel)
        auto begin_tile = [&](int t) {
            if (t == 0 || ++tile_m == tiles_m) {
                if (t > 0) { tile_m = 0; ++strip; }
                n0 = (strip % tiles_n) * BM + col0;
                zo = P.baseO + decode(P.Z, strip / tiles_n).o;
                ncol = n0 < Next ? (int)min(32u, Next - n0) : 0;
                __syncwarp();
                cols[(strip & 1u) * 32 + lane] = n0 + lane < Next ? decode(P.N, n0 + lane).o : 0;
                __syncwarp();
            }
            const unsigned m = tile_m * BM + quad * 32 + lane;
            row = m < Mext;
            ob = zo + decode(P.M, row ? m : 0u).o;
        };
        auto load_ahead = [&](int h) {
            if (pre < 0 || !row) return;
            const int *cs = cols + (strip & 1u) * 32;
            if (ncol >= h + 16) {
#pragma unroll
                for (int j = 0; j < 16; ++j) wn[j] = __ldg(src0 + (ob + cs[h + j]));
            } else if (ncol > h) {
#pragma unroll
                for (int j = 0; j < 16; ++j) wn[j] = __ldg(src0 + (ob + cs[h + j < ncol ? h + j : h]));
            }
        };
        if (n_tiles > 0) { begin_tile(0); load_ahead(0); }
#pragma unroll 1
        for (int it = 0; it < 2 * n_tiles; ++it) {
            const int t = it >> 1, h = (it & 1) * 16, live = ncol - h;
            if (h == 0) {
                ok = ok && mbar_wait(bar_done + 8 * (t & 1), (t >> 1) & 1, &failed);
                fence_after();
            }
            float v[16];
            if (ok) {
                unsigned r[16];
                tmem_ld16(tmem + ((unsigned)(quad * 32) << 16) + (t & 1) * BM + col0 + h, r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
            }
            if (h != 0) {
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_free + 8 * (t & 1));
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) w[j] = wn[j];
            // one multiply-add per value finds the non-finite ones (columns past the end hold leftovers of another kernel)
            float test = 0.f;
            if (live < 16) {
#pragma unroll
                for (int j = 0; j < 16; ++j) if (j >= live) v[j] = 0.f;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) test = fmaf(v[j], 0.f, test);
            const bool redo = __any_sync(0xffffffffu, (row && test != 0.f) || !ok);
            const int off0 = ob;
            const bool row_now = row;
            const unsigned m_tile = tile_m, s_now = strip;
            const int *co = cols + (s_now & 1u) * 32 + h;
            if (h == 0) load_ahead(16);
            else if (t + 1 < n_tiles) { __syncwarp(); begin_tile(t + 1); load_ahead(0); }
            if (!redo) {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] *= scale;
#define TAD_EPI_ALL(expr) _Pragma("unroll") for (int j = 0; j < 16; ++j) { float &x = v[j]; expr; }
                for (int e = 0; e < P.n_epi; ++e) {
                    const float imm = P.epi_imm[e];
                    switch (P.epi_op[e]) {
                    case TE_NEG: TAD_EPI_ALL(x = -x) break;
                    case TE_EXP: TAD_EPI_ALL(x = __expf(x)) break;
                    case TE_MULC: TAD_EPI_ALL(x *= imm) break;
                    case TE_ADDC: TAD_EPI_ALL(x += imm) break;
                    case TE_SQR: TAD_EPI_ALL(x *= x) break;
                    case TE_TANH: TAD_EPI_ALL(x = own_tanh(x)) break;
                    case TE_MUL_LOAD: case TE_ADD_LOAD: {
                        const bool mul = P.epi_op[e] == TE_MUL_LOAD;
                        if (e == pre) { if (pre_mul) { TAD_EPI_ALL(x *= w[j]) } else { TAD_EPI_ALL(x += w[j]) } }
                        else if (row_now) {
                            const float *__restrict__ src = ptrs.in[P.epi_ptr[e]];
                            const int sb = P.epi_base[e];
                            TAD_EPI_ALL(if (j < live) { const float y = __ldg(src + (unsigned)(sb + off0 + co[j])); x = mul ? x * y : x + y; })
                        }
                        break;
                    }
                    default: break;
                    }
                }
#undef TAD_EPI_ALL
                float *__restrict__ out = ptrs.out;
                if (row_now && P.accumulate) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) if (j < live) out[(unsigned)(off0 + co[j])] += v[j];
                } else if (row_now && live >= 16) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) out[(unsigned)(off0 + co[j])] = v[j];
                } else if (row_now) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) if (j < live) out[(unsigned)(off0 + co[j])] = v[j];
                }
            } else if (lane == 0) marks[t >> 4] |= 1u << ((t & 15) * 2 + (it & 1));
        }
        // Pieces with non-finite sums, once more behind the loop (inside it the code costs the loop its registers: 225 -> 255 us at
        // 8192 x 8192 x 34 with a tensor in the epilogue): fp32 multiply-adds from the operands themselves, sixteen columns at a
        // time.  Outputs with a NaN among their operands are NaN, and where that is all of them no sum is formed.
        // 8192 x 64 x 8192 with NaN operands / one infinity / infinities: 0.8 / 0.8 / 2.3 ms; with a decoded index and dependent loads for
        // every term 18.8 / 8.0 / 18.8 ms, the multiply-add tiles of contract.cu 0.25 ms whatever the values.
        __syncwarp();
        const char *pa = reinterpret_cast<const char *>(ptrs.in[P.ptrA]), *pb = reinterpret_cast<const char *>(ptrs.in[P.ptrB]);
        const unsigned gextA = (unsigned)P.guardA_ext, gextB = (unsigned)P.guardB_ext;         // (1 without a guard: the sum of the parts is then 0)
        // which of 32 rows (columns; one per lane) hold a NaN: the lanes run along the summation index
        auto holds_nan = [&](const char *src, unsigned off, int grd, const int *kt, unsigned gext) {
            unsigned mask = 0;
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
                const unsigned ro = __shfl_sync(0xffffffffu, off, r);
                const int rg = __shfl_sync(0xffffffffu, grd, r);
                bool nan = false;
#pragma unroll
                for (int k = 0; k < KS; k += 32) {
                    float x = 0.f;
                    if ((unsigned)(rg + kt[KS + k + lane]) < gext) x = __ldg(reinterpret_cast<const float *>(src + (ro + (unsigned)kt[k + lane])));
                    nan = nan || x != x;
                }
                if (__any_sync(0xffffffffu, nan)) mask |= 1u << r;
            }
            return mask;
        };
        unsigned strip_of = 0xffffffffu, rb = 0, nan_col = 0, z_of = 0;
        int gb = 0, on = 0;
        Parts zp{0, 0, 0, 0, 0};
#pragma unroll 1
        for (int t = 0; t < n_tiles; ++t) {
            const unsigned pieces = (marks[t >> 4] >> ((t & 15) * 2)) & 3u;
            if (!pieces) continue;
            const unsigned at = first + (unsigned)t, s_at = at / tiles_m, c0 = (s_at % tiles_n) * BM + col0;
            if (s_at != strip_of) {
                strip_of = s_at;
                z_of = s_at / tiles_n;
                zp = decode(P.Z, z_of);
                const Parts pn = decode(P.N, c0 + lane < Next ? c0 + lane : 0u);
                rb = (unsigned)(P.baseB + zp.b + pn.b) * 4u;
                gb = c0 + lane < Next ? P.guardB_c0 + zp.gb + pn.gb : DEAD;
                on = pn.o;
                nan_col = holds_nan(pb, rb, gb, ktab + 2 * KS, gextB);
            }
            const unsigned m = (at - s_at * tiles_m) * BM + quad * 32 + lane;
            const bool live_row = m < Mext;
            const Parts pm = decode(P.M, live_row ? m : 0u);
            const unsigned ra = (unsigned)(P.baseA + zp.a + pm.a) * 4u;
            const int ga = live_row ? P.guardA_c0 + zp.ga + pm.ga : DEAD, o_row = P.baseO + zp.o + pm.o;
            const bool nan_row = (holds_nan(pa, ra, ga, ktab, gextA) >> lane) & 1u;
            const bool some = __any_sync(0xffffffffu, live_row && !nan_row);
#pragma unroll 1
            for (int h = 0; h < 32; h += 16) {
                const int n = min(16, (int)min(32u, Next > c0 ? Next - c0 : 0u) - h);
                if (!((pieces >> (h / 16)) & 1u) || n <= 0) continue;
                float sum[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) sum[j] = 0.f;
                if (some && ((~nan_col >> h) & ((1u << n) - 1u))) {
#pragma unroll 2
                    for (unsigned k = 0; k < K; ++k) {
                        const float x = (unsigned)(ga + ktab[KS + k]) < gextA ? __ldg(reinterpret_cast<const float *>(pa + (ra + (unsigned)ktab[k]))) : 0.f;
                        // (lane j loads the value of column j)
                        const float y = (unsigned)(gb + ktab[3 * KS + k]) < gextB ? __ldg(reinterpret_cast<const float *>(pb + (rb + (unsigned)ktab[2 * KS + k]))) : 0.f;
#pragma unroll
                        for (int j = 0; j < 16; ++j) sum[j] = fmaf(x, __shfl_sync(0xffffffffu, y, h + j), sum[j]);
                    }
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const unsigned off = (unsigned)(o_row + __shfl_sync(0xffffffffu, on, h + j));
                    if (!live_row || j >= n) continue;
                    const float v0 = nan_row || ((nan_col >> (h + j)) & 1u) ? __int_as_float(0x7fffffff) : sum[j];
                    const float v1 = epilogue(P, ptrs, v0 * P.scale, off);
                    ptrs.out[off] = P.accumulate ? ptrs.out[off] + v1 : v1;
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == SE + SC) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
    }
}

// Adds the planes of a split summation, plane 0 first: planes are [column][row], a thread per output, consecutive
// threads on consecutive rows.
__global__ void __launch_bounds__(256)
tad_mma_reduce(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    const unsigned Mext = (unsigned)P.M.extent, Next = (unsigned)P.N.extent;
    const unsigned per_z = Mext * Next;
    const unsigned planes = (unsigned)P.ksplit;
    for (unsigned zb = 0; zb < (unsigned)P.Z.extent; ++zb) {
        const int oz = P.baseO + decode(P.Z, zb).o;
        for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < per_z; c += gridDim.x * blockDim.x) {
            const unsigned n = c / Mext, m = c - n * Mext;
            const float *src = ptrs.part + (size_t)zb * planes * per_z + c;
            float sum = 0.f;
#pragma unroll 4
            for (unsigned s = 0; s < planes; ++s) sum += src[(size_t)s * per_z];
            const unsigned off = (unsigned)(oz + decode(P.M, m).o + decode(P.N, n).o);
            float v = epilogue(P, ptrs, sum * P.scale, off);
            if (P.accumulate) v += ptrs.out[off];
            ptrs.out[off] = v;
        }
    }
}

// Splits the column operand into the images of its tiles: a block per stage, 32 columns and batch index reads 32 x 64
// elements (lanes along the index that is consecutive; eight loads a thread, all in flight), and writes the three bf16 parts
// of every column in the K-major, 128-byte swizzled order of the MMA's shared memory.  A block per whole tile and stage took
// 21 us at any size (a serial chain of table, loads and stores in 20 to 40 blocks); pieces of 32 columns take about 5.
constexpr int IC = 32, IMAGE_BN = TADC_IMAGE_COLS;     // columns of a block, of a tile

__global__ void __launch_bounds__(256)
tad_mma_image_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs)
{
    constexpr int BN = IMAGE_BN, LD = KS + 1, PART = BN * KS * 2;
    __shared__ float tile[IC * LD];
    __shared__ unsigned rows[IC], kt[KS];
    __shared__ int rowg[IC], ktg[KS];
    const int tid = threadIdx.x;
    const unsigned stage = blockIdx.x, n0 = blockIdx.y * IC, zb = blockIdx.z, Next = (unsigned)P.N.extent, K = (unsigned)P.K.extent;
    if (tid < IC + KS) {
        if (tid < IC) {
            const Parts z = decode(P.Z, zb);
            const unsigned n = n0 + tid;
            const Parts p = decode(P.N, n < Next ? n : 0u);
            rows[tid] = (unsigned)(P.baseB + z.b + p.b); rowg[tid] = n < Next ? P.guardB_c0 + z.gb + p.gb : DEAD;
        } else {
            const unsigned k = stage * KS + (tid - IC);
            const Parts p = decode(P.K, k < K ? k : 0u);
            kt[tid - IC] = (unsigned)p.b; ktg[tid - IC] = k < K ? p.gb : DEAD;
        }
    }
    __syncthreads();
    tad_wait_previous();
    const float *__restrict__ B = ptrs.in[P.ptrB];
    const bool along_rows = P.modeB == TM_ROW || P.modeB == TM_RVEC;
    constexpr int UNITS = IC * KS / 256;
    float v[UNITS];
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
        const int e = tid + i * 256, r = along_rows ? e % IC : e / KS, k = along_rows ? e / IC : e % KS;
        // (columns past the edge, indices past the end and guarded elements are zeros; a program without a guard has extent 1)
        v[i] = (unsigned)(rowg[r] + ktg[k]) < (unsigned)P.guardB_ext ? __ldg(B + (rows[r] + kt[k])) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
        const int e = tid + i * 256, r = along_rows ? e % IC : e / KS, k = along_rows ? e / IC : e % KS;
        tile[r * LD + k] = v[i];
    }
    __syncthreads();
    const unsigned tiles = (Next + BN - 1) / BN, stages = (K + KS - 1) / KS, tile_n = n0 / BN;
    unsigned char *dst = ptrs.image + (((size_t)zb * tiles + tile_n) * stages + stage) * (3 * PART);
    const int lc = tid / (KS / 8), l = n0 % BN + lc, o = tid % (KS / 8);
    unsigned p1[4], p2[4], p3[4];
    float u[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) u[j] = tile[lc * LD + o * 8 + j];
    split_unit<false>(u, p1, p2, p3);
    unsigned char *at = dst + l * 128 + ((o ^ (l & 7)) << 4);
    *reinterpret_cast<uint4 *>(at) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
    *reinterpret_cast<uint4 *>(at + PART) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
    *reinterpret_cast<uint4 *>(at + 2 * PART) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
}
static_assert(IC * KS / 8 == 256, "one unit a thread");

template <int BN, int MA, int MB>
cudaError_t launch_mma(const TadcProgram &P, const TadpPointers &ptrs, cudaStream_t stream)
{
    using C = MmaCfg<BN, MA, MB>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    auto kern = tad_mma_kernel<BN, MA, MB>;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
        if (e != cudaSuccess) return e;
        // the warpgroups' register shares must fit into what the block is launched with
        cudaFuncAttributes at;
        e = cudaFuncGetAttributes(&at, kern);
        if (e != cudaSuccess) return e;
        if (at.numRegs * NT < NCW * 32 * REG_CONV + 128 * REG_MMA) return cudaErrorInvalidConfiguration;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const unsigned tiles_m = ((unsigned)P.M.extent + BM - 1) / BM, tiles_n = ((unsigned)P.N.extent + BN - 1) / BN;
    dim3 grid(tiles_m * tiles_n, (unsigned)std::max(1, P.ksplit), (unsigned)P.Z.extent);
    tad_launch(kern, grid, NT, C::SMEM, stream, P, ptrs, tiles_n);
    return cudaGetLastError();
}

template <int MA, int MB>
cudaError_t launch_short(const TadcProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream)
{
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    auto kern = tad_mma_short_kernel<MA, MB>;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ShortCfg::SMEM);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const unsigned tiles_m = ((unsigned)P.M.extent + BM - 1) / BM, tiles_n = ((unsigned)P.N.extent + BM - 1) / BM;
    const unsigned long long items = (unsigned long long)tiles_m * tiles_n * (unsigned)P.Z.extent;
    if (items >= (1ull << 31)) return cudaErrorInvalidValue;
    return tad_launch(kern, (unsigned)std::min<unsigned long long>(items, sms), SNT, ShortCfg::SMEM, stream, P, ptrs, tiles_m, tiles_n, (unsigned)items);
}

}  // namespace

cudaError_t tad_launch_mma(const TadcProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream)
{
    cudaError_t e = cudaErrorInvalidValue;
    // the pipelined kernel from four tiles per SM on (8192 x 8192 x 34 forward 220 -> 148 us, staged adjoint 280 -> 181 us);
    // with one or two tiles a block has nothing to overlap (1301 x 2477 x 23: 18 us as blocks of one tile, 23 us here)
    const unsigned long long tiles = (unsigned long long)((P.M.extent + BM - 1) / BM) * (unsigned)((P.N.extent + BM - 1) / BM) * (unsigned)P.Z.extent;
    const bool short_pays = P.K.extent <= KS && P.ksplit <= 1 && P.N.extent > 64 && tiles >= 4ull * sms && tiles <= (unsigned long long)ShortCfg::MAX_TILES * sms;
#define TAD_MMA_CASE(MA, MB)                                                                                              \
    case MA * 4 + MB: e = short_pays ? launch_short<MA, MB>(P, ptrs, sms, stream) : P.N.extent <= 64 ? launch_mma<64, MA, MB>(P, ptrs, stream) : launch_mma<128, MA, MB>(P, ptrs, stream); break;
    if (P.image && !short_pays) {
        const dim3 grid((unsigned)(P.K.extent + KS - 1) / KS, (unsigned)(P.N.extent + IMAGE_BN - 1) / IMAGE_BN * (IMAGE_BN / IC), (unsigned)P.Z.extent);
        e = tad_launch(tad_mma_image_kernel, grid, 256, 0, stream, P, ptrs);
        if (e != cudaSuccess) return e;
        switch (P.modeA) {
        case TM_ROW: e = launch_mma<IMAGE_BN, TM_ROW, TM_IMAGE>(P, ptrs, stream); break;
        case TM_KVEC: e = launch_mma<IMAGE_BN, TM_KVEC, TM_IMAGE>(P, ptrs, stream); break;
        default: e = launch_mma<IMAGE_BN, TM_K, TM_IMAGE>(P, ptrs, stream); break;
        }
    } else
#define TAD_MMA_ROW(MA) TAD_MMA_CASE(MA, TM_ROW) TAD_MMA_CASE(MA, TM_KVEC) TAD_MMA_CASE(MA, TM_K) TAD_MMA_CASE(MA, TM_RVEC)
    switch (P.modeA * 4 + P.modeB) { TAD_MMA_ROW(TM_ROW) TAD_MMA_ROW(TM_KVEC) TAD_MMA_ROW(TM_K) default: break; }
#undef TAD_MMA_ROW
#undef TAD_MMA_CASE
    if (e == cudaSuccess && P.ksplit > 1) {
        const unsigned long long cells = (unsigned long long)P.M.extent * P.N.extent;
        const unsigned blocks = (unsigned)std::min<unsigned long long>((cells + 255) / 256, (unsigned long long)sms * 8);
        tad_launch(tad_mma_reduce, blocks, 256, 0, stream, P, ptrs);
        e = cudaGetLastError();
    }
    return e;
}
