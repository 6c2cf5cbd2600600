// Tensor-core kernel for contraction programs (contract.h), fp32 in and fp32 out.
//
// Every fp32 operand element is split exactly into three bf16 values, x = x1 + x2 + x3 (8 + 8 + 8 significant
// bits, each part the rounded remainder of the ones before it), and a product is the sum of six bf16 products,
//     a b = a1 b1 + (a1 b2 + a2 b1) + (a1 b3 + a2 b2 + a3 b1).
// What is left out, a2 b3 + a3 b2 + a3 b3, is at most 2^-23 |a b| and about 2^-26 |a b| in the mean square, below
// the rounding of the additions.  bf16 products are exact in the fp32 accumulator; the accumulator itself
// truncates, so a sum stays in it for one stage of 64 summation indices only (small products first, then four
// steps of a1 b1) and the stages are added up in fp32 registers with round-to-nearest.  Measured against float64
// (2-norm, normal operands): 0.8e-7 at 64 terms, 1.2e-7 at 1100, 1.3e-7 at 2048; chains of fp32 multiply-adds
// gave 4.2e-7 at 1100.  Outputs of a warp whose sums come out non-finite or huge (an operand beyond the bf16
// range, an infinity times a zero part) are evaluated again with fp32 multiply-adds from the operands
// themselves, so infinities and NaNs are those of the definition.
//
// One block per SM.  Warps 0-15 gather the operands of a stage through the offset tables (global -> registers, a
// whole stage ahead), split them and write them to shared memory in the 128-byte swizzled layout of the MMA
// (K-major when the lanes run along the rows, MN-major when they run along the summation index) or, for a row
// operand with its lanes along the rows, to tensor memory (the MMA then reads half as much shared memory); warp 16
// prepares the offset tables and issues the MMAs.  While stage s is multiplied, stage s + 1 is gathered and stage
// s - 1 is added to the registers.
//
// What bounds it: the six bf16 products of a 128 x 128 x 64 stage take 1536 clocks of the tensor core, gathering,
// splitting and adding up about 2900 clocks of the sixteen warps (4096 x 4096 x 4096: 775 us, 712 us without the
// MMAs, 543 us without the loads).  Measured against the fp32 multiply-add tiles of contract.cu: strided
// convolution 64 x 256 x 2048 with 1280 terms 1930 -> 535 us (160 TFLOP/s), its gradients 2110 -> 755 and
// 1984 -> 534 us; 1500 x 1100 x 1333 product 153 -> 48 us; 37 x 4907 x 159 convolution 26.6 -> 10.2 us.
#include <cuda_runtime.h>

#include <algorithm>

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
        const int u = tid + i * NCW * 32;
        int o;
        if (TMEM) { l = tid % BM; o = (tid / BM) * 2 + i; }
        else if (MODE == TM_ROW) { l = u % R; o = u / R; }
        else if (MODE == TM_KVEC) { o = u % (KS / 8); l = u / (KS / 8); }
        else if (MODE == TM_K) { l = u % KS; o = u / KS; }
        else { l = (u / 8) % KS; o = (u / (8 * KS)) * 8 + u % 8; }
        t0 = o * 8;
        dst = (KMAJOR ? 0 : (o >> 3) * (KS * 128)) + l * 128 + (((o & 7) ^ (l & 7)) << 4);
    }
};

__device__ __forceinline__ float ldf(const float *__restrict__ src, unsigned byte_off)
{
    return __ldg(reinterpret_cast<const float *>(reinterpret_cast<const char *>(src) + byte_off));
}

// rows: offsets and guards of the tile's rows; kt: offsets and guards of the stage's summation indices (KS each)
template <int MODE, int R, bool TMEM, bool CHECK>
__device__ __forceinline__ void load_unit(float (&v)[8], const float *__restrict__ src, const int tid, const int i, const unsigned *row, const int *rowg,
                                          const unsigned *kt, const int *ktg, const unsigned gext)
{
    using U = Unit<MODE, R, TMEM>;
    const U u(tid, i);
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

// eight values -> three times eight bf16 (packed in pairs)
__device__ __forceinline__ void split_unit(const float (&v)[8], unsigned (&p1)[4], unsigned (&p2)[4], unsigned (&p3)[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float x = v[2 * j], y = v[2 * j + 1];
        unsigned h, m, l;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(y), "f"(x));
        const float rx = x - __uint_as_float(h << 16), ry = y - __uint_as_float(h & 0xffff0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(ry), "f"(rx));
        const float sx = rx - __uint_as_float(m << 16), sy = ry - __uint_as_float(m & 0xffff0000u);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(sy), "f"(sx));
        p1[j] = h; p2[j] = m; p3[j] = l;
    }
}

template <int BN, int MA, int MB>
struct MmaCfg {
    static constexpr bool TS = MA == TM_ROW;
    static constexpr int PART_A = BM * KS * 2, PART_B = BN * KS * 2;                 // bytes of one bf16 part of a stage
    static constexpr int STAGE = (TS ? 0 : 3 * PART_A) + 3 * PART_B;
    static constexpr int UA = BM * KS / 8 / (NCW * 32), UB = BN * KS / 8 / (NCW * 32);   // units per thread
    static constexpr int COLS = BN * 32 / (NCW * 8);                                  // accumulator columns per thread
    static constexpr int TABLES = (BM + BN) * 12 + KT * KS * 16;                      // row offsets, guards, output offsets; k tables
    static constexpr size_t SMEM = 1024 + 2 * size_t(STAGE) + TABLES;
};

template <int BN, int MA, int MB>
__global__ void __launch_bounds__(NT, 1)
tad_mma_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs, const unsigned tiles_n)
{
    tad_wait_previous();
    using C = MmaCfg<BN, MA, MB>;
    constexpr bool TS = C::TS;
    constexpr int COLS = C::COLS;
    extern __shared__ unsigned char smem_raw[];
    __shared__ unsigned long long bars[4 + KT];
    __shared__ unsigned tmem_base_s;
    __shared__ volatile int failed;
    const unsigned smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *stages = smem_raw + (smem0 - smem_u32(smem_raw));
    unsigned *rowA = reinterpret_cast<unsigned *>(stages + 2 * C::STAGE), *rowB = rowA + BM;          // bytes
    int *rowgA = reinterpret_cast<int *>(rowB + BN), *rowgB = rowgA + BM, *outM = rowgB + BN, *outN = outM + BM;
    int *ktab = outN + BN;                                   // per ring slot: offsets A, guards A, offsets B, guards B (KS each)
    const unsigned bar_full = smem_u32(&bars[0]), bar_done = smem_u32(&bars[2]), bar_tab = smem_u32(&bars[4]);

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
            Parts p{0, 0, 0, 0, 0};
            if (m < Mext) p = decode(P.M, m);
            rowA[r] = m < Mext ? (unsigned)(P.baseA + z.a + p.a) * 4u : 0u; rowgA[r] = m < Mext ? P.guardA_c0 + z.ga + p.ga : DEAD; outM[r] = p.o;
        }
        for (int r = tid - BM; r < BN; r += NCW * 32) {
            if (r < 0) continue;
            const unsigned n = tile_n * BN + r;
            Parts p{0, 0, 0, 0, 0};
            if (n < Next) p = decode(P.N, n);
            rowB[r] = n < Next ? (unsigned)(P.baseB + z.b + p.b) * 4u : 0u; rowgB[r] = n < Next ? P.guardB_c0 + z.gb + p.gb : DEAD; outN[r] = p.o;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = __shfl_sync(0xffffffffu, tmem_base_s, 0);
    constexpr unsigned TMEM_A = 2 * BN;                      // columns of the row operand's stages (TS): 3 x 32 each
    bool ok = true;

    if (warp >= NCW) {
        // ---- MMA warp ----
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REG_MMA));
        const int n_stages_mma = warp == NCW ? n_stages : 0;
        constexpr bool a_k = MA == TM_ROW || MA == TM_KVEC, b_k = MB == TM_ROW || MB == TM_KVEC;
        const unsigned n_pad = min((unsigned)BN, (Next - tile_n * BN + 15u) / 16u * 16u);
        const unsigned idesc = (1u << 4) | (1u << 7) | (1u << 10) | (a_k ? 0u : 1u << 15) | (b_k ? 0u : 1u << 16) | ((n_pad >> 3) << 17) | ((BM >> 4) << 24);
        // K-major: eight rows of 128 bytes per repeat; MN-major: blocks of 64 rows, eight summation indices per repeat
        constexpr unsigned stepA = a_k ? 32u : 16u * 128u, stepB = b_k ? 32u : 16u * 128u;
        constexpr unsigned lboA = a_k ? 16u : KS * 128u, lboB = b_k ? 16u : KS * 128u;
        int issued = 0;
        for (int s = 0; s < n_stages_mma && ok; ++s) {
            ok = mbar_wait(bar_full + 8 * (s & 1), (s >> 1) & 1, &failed);
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
        const bool edgeA = P.guardA || (tile_m + 1) * BM > Mext, edgeB = P.guardB || (tile_n + 1) * BN > Next;
        const unsigned gextA = (unsigned)P.guardA_ext, gextB = (unsigned)P.guardB_ext;
        float va[C::UA][8], vb[C::UB][8];
        auto load = [&](float (&v)[8], int i, int s, bool second, bool check) {
            const unsigned *t = reinterpret_cast<const unsigned *>(ktab + (s % KT) * 4 * KS) + (second ? 2 * KS : 0);
            const int *tg = reinterpret_cast<const int *>(t + KS);
            if (!second) {
                if (check) load_unit<MA, BM, TS, true>(v, A, tid, i, rowA, rowgA, t, tg, gextA);
                else load_unit<MA, BM, TS, false>(v, A, tid, i, rowA, rowgA, t, tg, gextA);
            } else {
                if (check) load_unit<MB, BN, false, true>(v, B, tid, i, rowB, rowgB, t, tg, gextB);
                else load_unit<MB, BN, false, false>(v, B, tid, i, rowB, rowgB, t, tg, gextB);
            }
        };
        // adds the finished stage s to the registers
        auto collect = [&](int s) {
            ok = ok && mbar_wait(bar_done + 8 * (s & 1), (s >> 1) & 1, &failed);
            fence_after();
            if (!ok) return;
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
        for (int i = 0; i < C::UA; ++i) load(va[i], i, 0, false, edgeA || kend - kbeg < KS);
#pragma unroll
        for (int i = 0; i < C::UB; ++i) load(vb[i], i, 0, true, edgeB || kend - kbeg < KS);
        for (int s = 0; s < n_stages && ok; ++s) {
            unsigned char *st = stages + (s & 1) * C::STAGE;
            const bool more = s + 1 < n_stages, tail = kend - kbeg - (unsigned)s * KS < 2 * KS;      // the next stage is a partial one
            if (more && s + 1 >= KT) ok = mbar_wait(bar_tab + 8 * ((s + 1) % KT), ((s + 1) / KT - 1) & 1, &failed);
            if (!ok) break;
            unsigned p1[4], p2[4], p3[4];
#pragma unroll
            for (int i = 0; i < C::UA; ++i) {
                split_unit(va[i], p1, p2, p3);
                if (more) load(va[i], i, s + 1, false, edgeA || tail);
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
                split_unit(vb[i], p1, p2, p3);
                if (more) load(vb[i], i, s + 1, true, edgeB || tail);
                const Unit<MB, BN, false> u(tid, i);
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
        // ---- outputs: a thread holds COLS columns of its row; consecutive lanes are consecutive rows ----
        const unsigned rl = (unsigned)(quad * 32 + lane), m = tile_m * BM + rl, n0 = tile_n * BN + col0;
        const int live = m < Mext && n0 < Next ? (int)min((unsigned)COLS, Next - n0) : 0;
        bool odd = !ok;
#pragma unroll
        for (int j = 0; j < COLS; ++j) odd = odd || (j < live && !(fabsf(acc[j]) <= 3.0e38f));
        if (__any_sync(0xffffffffu, odd)) {
            // the warp's outputs once more, with fp32 multiply-adds from the operands themselves
            const float *__restrict__ A = ptrs.in[P.ptrA];
            const float *__restrict__ B = ptrs.in[P.ptrB];
#pragma unroll 1
            for (int j = 0; j < live; ++j) {
                const char *pa = reinterpret_cast<const char *>(A), *pb = reinterpret_cast<const char *>(B);
                const unsigned ra = rowA[rl], rb = rowB[col0 + j];
                const int ga = rowgA[rl], gb = rowgB[col0 + j];
                float sum = 0.f;
#pragma unroll 1
                for (unsigned k = kbeg; k < kend; ++k) {
                    const Parts p = decode(P.K, k);
                    const bool la = !P.guardA || (unsigned)(ga + p.ga) < (unsigned)P.guardA_ext, lb = !P.guardB || (unsigned)(gb + p.gb) < (unsigned)P.guardB_ext;
                    const float x = la ? __ldg(reinterpret_cast<const float *>(pa + (ra + (unsigned)p.a * 4u))) : 0.f;
                    const float y = lb ? __ldg(reinterpret_cast<const float *>(pb + (rb + (unsigned)p.b * 4u))) : 0.f;
                    sum = fmaf(x, y, sum);
                }
                if (P.ksplit > 1) ptrs.part[((size_t)zb * (unsigned)P.ksplit + ks) * Next * Mext + (size_t)(n0 + j) * Mext + m] = sum;
                else {
                    const unsigned off = (unsigned)(P.baseO + z.o + outM[rl] + outN[col0 + j]);
                    const float v = epilogue(P, ptrs, sum * P.scale, off);
                    ptrs.out[off] = P.accumulate ? ptrs.out[off] + v : v;
                }
            }
        } else if (live) {
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
        fence_before();
    }
    __syncthreads();
    if (warp == NCW) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
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
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    const unsigned tiles_m = ((unsigned)P.M.extent + BM - 1) / BM, tiles_n = ((unsigned)P.N.extent + BN - 1) / BN;
    dim3 grid(tiles_m * tiles_n, (unsigned)std::max(1, P.ksplit), (unsigned)P.Z.extent);
    tad_launch(kern, grid, NT, C::SMEM, stream, P, ptrs, tiles_n);
    return cudaGetLastError();
}

}  // namespace

cudaError_t tad_launch_mma(const TadcProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream)
{
    cudaError_t e = cudaErrorInvalidValue;
#define TAD_MMA_CASE(MA, MB)                                                                                              \
    case MA * 4 + MB: e = P.N.extent <= 64 ? launch_mma<64, MA, MB>(P, ptrs, stream) : launch_mma<128, MA, MB>(P, ptrs, stream); break;
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
