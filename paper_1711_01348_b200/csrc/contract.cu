// Tile kernel for contraction programs (contract.h): a thread block owns a BM x BN tile of
// outputs, gathers BK summation indices of both operands at a time into shared memory with
// asynchronous copies (two stages), and every thread keeps a TM x TN tile of sums in
// registers that it feeds from shared memory with 128-bit loads.  Operand elements outside a
// guard, past the end of the summation range or in the ragged edge of a tile arrive as zeros
// (zero-fill copies), so the multiply-add loop has no tests.  No atomics: a summation split over
// several blocks writes planes of partial sums that tad_contract_reduce adds in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>

#include "launch.h"
#include "contract.cuh"

namespace {

constexpr int BK = TADC_BK;
constexpr int KK_UNROLL = 8;          // summation indices per unrolled body of the multiply-add loop
constexpr int STAGES = 2;
using namespace tadc;

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool live)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = live ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(bytes));
}
__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool live)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = live ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// One stage of one operand: BK x BR values into smem[kl * (BR + 4) + rl].  rows[rl] = (offset part, guard
// part) of tile row rl, ktab[kl] the same for the stage's summation index kl.  CHECK = false is the path
// of a stage whose every element exists and is read (no guard on the operand, tile and stage inside
// the ranges): offset add, copy.  pre = rows[row of this thread] for the modes whose threads keep one row.
template <int BR, int NT, bool CHECK>
__device__ __forceinline__ void gather(float *smem, const float *__restrict__ src, const int2 *rows, const int2 *ktab,
                                       const int2 pre, const int mode, const unsigned gext, const unsigned tid, const unsigned klimit)
{
    // The copies carry no memory clobber (the group commit and wait do), and the table entries of a batch of
    // copies are read before the first of them is issued, so that the table reads overlap instead of each
    // waiting its turn.  klimit: summation indices of this stage that the multiply-add loop will read.
    constexpr int LD = BR + 4;
    constexpr bool REGULAR = NT % BR == 0 && (BR * BK) % NT == 0 && NT % (BR / 4) == 0 && NT % (4 * BK) == 0;
    if constexpr (!REGULAR) {
        // any number of threads: element e of the stage -> (row, summation index) by the mode's own order
        const unsigned total = mode == TG_ROW16 ? (BR / 4) * BK : BR * BK;
        for (unsigned e0 = tid; e0 < total; e0 += 4 * NT) {
            unsigned off[4], dst[4]; bool live[4], use[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned e = e0 + j * NT;
                unsigned rl, kl;
                if (mode == TG_ROW16) { rl = (e % (BR / 4)) * 4; kl = e / (BR / 4); }
                else if (mode == TG_ROW) { rl = e % BR; kl = e / BR; }
                else { kl = e % BK; rl = e / BK; }
                use[j] = e < total && kl < klimit;
                const int2 r = rows[use[j] ? rl : 0], kt = ktab[use[j] ? kl : 0];
                live[j] = !CHECK || (unsigned)(r.y + kt.y) < gext;
                off[j] = live[j] ? (unsigned)(r.x + kt.x) : 0u;
                dst[j] = kl * LD + rl;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (use[j]) { if (mode == TG_ROW16) cp_async16(smem + dst[j], src + off[j], live[j]); else cp_async4(smem + dst[j], src + off[j], live[j]); }
        }
        return;
    } else {
    if (mode == TG_ROW16) {
        constexpr unsigned CH = BR / 4, TOTAL = CH * BK, PER = (TOTAL + NT - 1) / NT, KSTEP = NT / CH;
        const unsigned rl = (tid % CH) * 4, kl0 = tid / CH;
        if (TOTAL % NT != 0 && kl0 >= BK) return;
        unsigned off[PER]; bool live[PER];
#pragma unroll
        for (unsigned j = 0; j < PER; ++j) {
            const int2 kt = ktab[kl0 + KSTEP * j];
            live[j] = !CHECK || (unsigned)(pre.y + kt.y) < gext;
            off[j] = live[j] ? (unsigned)(pre.x + kt.x) : 0u;
        }
#pragma unroll
        for (unsigned j = 0; j < PER; ++j)
            if (kl0 + KSTEP * j < klimit) cp_async16(smem + (kl0 + KSTEP * j) * LD + rl, src + off[j], live[j]);
    } else if (mode == TG_ROW) {
        constexpr unsigned TOTAL = BR * BK, PER = TOTAL / NT, KSTEP = NT / BR;
        const unsigned rl = tid % BR, kl0 = tid / BR;
        unsigned off[PER]; bool live[PER];
#pragma unroll
        for (unsigned j = 0; j < PER; ++j) {
            const int2 kt = ktab[kl0 + KSTEP * j];
            live[j] = !CHECK || (unsigned)(pre.y + kt.y) < gext;
            off[j] = live[j] ? (unsigned)(pre.x + kt.x) : 0u;
        }
#pragma unroll
        for (unsigned j = 0; j < PER; ++j)
            if (kl0 + KSTEP * j < klimit) cp_async4(smem + (kl0 + KSTEP * j) * LD + rl, src + off[j], live[j]);
    } else {
        // a warp copies 8 summation indices x 4 rows: full 32-byte sectors of a row-major operand, and the
        // 32 shared-memory words it writes (row stride BR + 4) fall into 32 different banks
        constexpr unsigned TOTAL = BR * BK, PER = TOTAL / NT, RSTEP = NT / BK;
        const unsigned kl = (tid % 8) + 8 * ((tid / 32) % (BK / 8)), rl0 = (tid / 8) % 4 + 4 * (tid / (4 * BK));
        if (kl >= klimit) return;
        const int2 kt = ktab[kl];
        unsigned off[PER]; bool live[PER];
#pragma unroll
        for (unsigned j = 0; j < PER; ++j) {
            const int2 r = rows[rl0 + RSTEP * j];
            live[j] = !CHECK || (unsigned)(r.y + kt.y) < gext;
            off[j] = live[j] ? (unsigned)(r.x + kt.x) : 0u;
        }
#pragma unroll
        for (unsigned j = 0; j < PER; ++j) cp_async4(smem + kl * LD + rl0 + RSTEP * j, src + off[j], live[j]);
    }
    }
}

template <int BM, int BN, int TM, int TN>
struct Cfg {
    static constexpr int NT = (BM / TM) * (BN / TN);
    static constexpr int LDA = BM + 4, LDB = BN + 4;
    static constexpr int STAGE_FLOATS = BK * (LDA + LDB);
    static constexpr size_t SMEM = size_t(STAGES) * STAGE_FLOATS * 4 + size_t(BM + BN) * 8 + size_t(BM + BN) * 4 +
                                   size_t(STAGES + 1) * BK * 16;      // stages, row tables, output offsets, two k tables
};

template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(Cfg<BM, BN, TM, TN>::NT, (TM * TN >= 64 ? 2 : Cfg<BM, BN, TM, TN>::NT <= 160 ? 4 : 3))
tad_contract_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs, const unsigned tiles_m, const unsigned tiles_n)
{
    tad_wait_previous();
    using C = Cfg<BM, BN, TM, TN>;
    constexpr int NT = C::NT, LDA = C::LDA, LDB = C::LDB;
    constexpr int GM = TM / 4, GN = TN / 4;           // groups of four rows / columns per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *stage_mem = reinterpret_cast<float *>(smem_raw);
    int2 *ktabA = reinterpret_cast<int2 *>(stage_mem + STAGES * C::STAGE_FLOATS);
    int2 *ktabB = ktabA + (STAGES + 1) * BK;
    int2 *rowA = ktabB + (STAGES + 1) * BK;
    int2 *rowB = rowA + BM;
    int *outM = reinterpret_cast<int *>(rowB + BN);
    int *outN = outM + BM;

    const unsigned tid = threadIdx.x;
    const unsigned tile = blockIdx.x;
    const unsigned tile_m = tile % tiles_m, tile_n = tile / tiles_m;
    const unsigned ks = blockIdx.y, zb = blockIdx.z;
    const Parts z = decode(P.Z, zb);
    // Offsets are sums of signed 32-bit parts that may be negative one by one (a band that starts below
    // zero, a negative stride); only the complete sum of a live element is a valid element offset, so the
    // constant parts go into the row tables and the pointer stays the tensor's own.
    const bool onesB = P.ptrB < 0;                // B is a tensor of ones: a plain summation of A
    const float *__restrict__ A = ptrs.in[P.ptrA];
    const float *__restrict__ B = onesB ? A : ptrs.in[P.ptrB];
    const int constA = P.baseA + z.a, constB = P.baseB + z.b;
    const unsigned Mext = (unsigned)P.M.extent, Next = (unsigned)P.N.extent;
    const unsigned kbeg = ks * (unsigned)P.kchunk;
    const unsigned kend = min((unsigned)P.K.extent, kbeg + (unsigned)P.kchunk);
    const int n_stages = (int)((kend - kbeg + BK - 1) / BK);

    // per-row parts of the operand offsets, guards and output offsets of this tile
    for (unsigned r = tid; r < BM; r += NT) {
        const unsigned m = tile_m * BM + r;
        if (m < Mext) { const Parts p = decode(P.M, m); rowA[r] = make_int2(constA + p.a, P.guardA_c0 + z.ga + p.ga); outM[r] = p.o; }
        else { rowA[r] = make_int2(0, DEAD); outM[r] = 0; }
    }
    for (unsigned r = tid; r < BN; r += NT) {
        const unsigned n = tile_n * BN + r;
        if (n < Next) { const Parts p = decode(P.N, n); rowB[r] = make_int2(constB + p.b, P.guardB_c0 + z.gb + p.gb); outN[r] = p.o; }
        else { rowB[r] = make_int2(0, DEAD); outN[r] = 0; }
    }
    auto fill_ktab = [&](int kstage) {
        if (tid < BK) {
            const unsigned k = kbeg + (unsigned)kstage * BK + tid;
            int2 ea = make_int2(0, DEAD), eb = make_int2(0, DEAD);
            if (k < kend) { const Parts p = decode(P.K, k); ea = make_int2(p.a, p.ga); eb = make_int2(p.b, p.gb); }
            ktabA[(kstage % (STAGES + 1)) * BK + tid] = ea;
            ktabB[(kstage % (STAGES + 1)) * BK + tid] = eb;
        }
    };
    for (int s = 0; s < STAGES; ++s) fill_ktab(s);
    if (onesB)
        for (unsigned e = tid; e < (unsigned)(STAGES * BK * LDB); e += NT) {
            const unsigned s = e / (BK * LDB), r = e - s * (BK * LDB);
            stage_mem[s * C::STAGE_FLOATS + BK * LDA + r] = 1.f;
        }
    __syncthreads();
    const unsigned gextA = (unsigned)P.guardA_ext, gextB = (unsigned)P.guardB_ext;
    const int modeA = P.modeA, modeB = P.modeB;
    // the row a thread keeps through all stages (modes with the lanes along the row index)
    const int2 preA = rowA[modeA == TG_ROW16 ? (tid % (BM / 4)) * 4 : tid % BM];
    const int2 preB = rowB[modeB == TG_ROW16 ? (tid % (BN / 4)) * 4 : tid % BN];      // (unused by tiles with irregular thread counts)
    // tiles inside the ranges and operands without a guard take the copy path without tests
    const bool plainA = !P.guardA && (tile_m + 1) * BM <= Mext, plainB = !P.guardB && (tile_n + 1) * BN <= Next;
    auto issue = [&](int kstage) {
        if (kstage < n_stages) {
            float *as = stage_mem + (kstage % STAGES) * C::STAGE_FLOATS;
            float *bs = as + BK * LDA;
            const int slot = (kstage % (STAGES + 1)) * BK;
            const unsigned left = kend - kbeg - (unsigned)kstage * BK;
            const bool full = left >= BK;
            const unsigned klimit = full ? BK : (left + KK_UNROLL - 1) / KK_UNROLL * KK_UNROLL;
            if (plainA && full) gather<BM, NT, false>(as, A, rowA, ktabA + slot, preA, modeA, gextA, tid, klimit);
            else gather<BM, NT, true>(as, A, rowA, ktabA + slot, preA, modeA, gextA, tid, klimit);
            if (onesB) {}
            else if (plainB && full) gather<BN, NT, false>(bs, B, rowB, ktabB + slot, preB, modeB, gextB, tid, klimit);
            else gather<BN, NT, true>(bs, B, rowB, ktabB + slot, preB, modeB, gextB, tid, klimit);
        }
        cp_async_commit();
    };
    for (int s = 0; s < STAGES - 1; ++s) issue(s);

    // a warp covers 8 thread columns x 4 thread rows: its 128-bit reads of a stage touch 128 consecutive bytes
    // of the B tile and 64 of the A tile, one shared-memory wavefront each (tiles whose thread columns do not
    // come in eights number their threads row by row)
    constexpr unsigned TCOLS = BN / TN;
    const unsigned warp = tid / 32, lane = tid % 32;
    const int tx = TCOLS % 8 == 0 ? (int)((warp % (TCOLS / 8 ? TCOLS / 8 : 1)) * 8 + lane % 8) : (int)(tid % TCOLS);
    const int ty = TCOLS % 8 == 0 ? (int)((warp / (TCOLS / 8 ? TCOLS / 8 : 1)) * 4 + lane / 8) : (int)(tid / TCOLS);
    float acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

    for (int it = 0; it < n_stages; ++it) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();
        fill_ktab(it + STAGES);
        issue(it + STAGES - 1);
        const float *as = stage_mem + (it % STAGES) * C::STAGE_FLOATS;
        const float *bs = as + BK * LDA;
        // operands of summation index kk + 1 are fetched from shared memory while those of kk are multiplied
        float a[2][TM], b[2][TN];
        auto fetch = [&](int kk, float *av, float *bv) {
#pragma unroll
            for (int g = 0; g < GM; ++g) {
                const float4 v = *reinterpret_cast<const float4 *>(as + kk * LDA + g * (BM / GM) + ty * 4);
                av[4 * g] = v.x; av[4 * g + 1] = v.y; av[4 * g + 2] = v.z; av[4 * g + 3] = v.w;
            }
#pragma unroll
            for (int g = 0; g < GN; ++g) {
                const float4 v = *reinterpret_cast<const float4 *>(bs + kk * LDB + g * (BN / GN) + tx * 4);
                bv[4 * g] = v.x; bv[4 * g + 1] = v.y; bv[4 * g + 2] = v.z; bv[4 * g + 3] = v.w;
            }
        };
        fetch(0, a[0], b[0]);
        // bodies of KK_UNROLL summation indices; a last stage with few indices left runs only the bodies that hold some
        const int n_bodies = min(BK / KK_UNROLL, (int)(((kend - kbeg) - (unsigned)it * BK + KK_UNROLL - 1) / KK_UNROLL));
        for (int body = 0; body < n_bodies; ++body) {
            const float *as_b = as + body * KK_UNROLL * LDA, *bs_b = bs + body * KK_UNROLL * LDB;
#pragma unroll
            for (int u = 0; u < KK_UNROLL; ++u) {
                if (u + 1 < KK_UNROLL || body + 1 < n_bodies) {
#pragma unroll
                    for (int q = 0; q < GM; ++q) {
                        const float4 v = *reinterpret_cast<const float4 *>(as_b + (u + 1) * LDA + q * (BM / GM) + ty * 4);
                        a[(u + 1) & 1][4 * q] = v.x; a[(u + 1) & 1][4 * q + 1] = v.y; a[(u + 1) & 1][4 * q + 2] = v.z; a[(u + 1) & 1][4 * q + 3] = v.w;
                    }
#pragma unroll
                    for (int q = 0; q < GN; ++q) {
                        const float4 v = *reinterpret_cast<const float4 *>(bs_b + (u + 1) * LDB + q * (BN / GN) + tx * 4);
                        b[(u + 1) & 1][4 * q] = v.x; b[(u + 1) & 1][4 * q + 1] = v.y; b[(u + 1) & 1][4 * q + 2] = v.z; b[(u + 1) & 1][4 * q + 3] = v.w;
                    }
                }
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[u & 1][i], b[u & 1][j], acc[i][j]);
            }
        }
    }
    cp_async_wait<0>();

    // ---- store ----
    // The sums go through shared memory (the stage buffers are free now): a compact loop then applies the epilogue
    // to four columns at a time and writes whole rows of the tile, consecutive threads to consecutive columns.
    // (Storing straight from the 64 registers would unroll the epilogue 64 times: code that no longer fits the
    // instruction cache and is run once per tile.)
    constexpr int LDC = BN + 4;
    static_assert(BM * LDC <= STAGES * C::STAGE_FLOATS, "the tile of sums must fit into the stage buffers");
    float *cs = stage_mem;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int rl = (i / 4) * (BM / GM) + ty * 4 + (i % 4);
#pragma unroll
        for (int q = 0; q < GN; ++q)
            *reinterpret_cast<float4 *>(cs + rl * LDC + q * (BN / GN) + tx * 4) =
                make_float4(acc[i][4 * q], acc[i][4 * q + 1], acc[i][4 * q + 2], acc[i][4 * q + 3]);
    }
    __syncthreads();
    const bool partial = P.ksplit > 1;
    float *__restrict__ out = partial ? ptrs.part : ptrs.out;
    const float scale = P.scale;
    const int n_epi = partial ? 0 : P.n_epi;
    const int obase = P.baseO + z.o;
    const bool vec_ok = partial ? (Next & 3u) == 0 : P.out_vec4 != 0;
    // four pieces of four columns per pass: every epilogue step is dispatched once for 16 values and the loads of a
    // step (a tensor laid out like the output) are issued together
    constexpr int EU = 4;
    for (unsigned e0 = tid; e0 < (unsigned)(BM * BN / 4); e0 += NT * EU) {
        float v[EU][4];
        unsigned off[EU][4];
        int live[EU];
#pragma unroll
        for (int u = 0; u < EU; ++u) {
            const unsigned e = e0 + (unsigned)u * NT;
            const unsigned rl = e / (BN / 4), cl = (e % (BN / 4)) * 4;
            const unsigned m = tile_m * BM + rl, n = tile_n * BN + cl;
            const bool in = e < (unsigned)(BM * BN / 4) && m < Mext && n < Next;
            live[u] = in ? (int)min(4u, Next - n) : 0;
            const float4 s4 = in ? *reinterpret_cast<const float4 *>(cs + rl * LDC + cl) : make_float4(0.f, 0.f, 0.f, 0.f);
            v[u][0] = s4.x; v[u][1] = s4.y; v[u][2] = s4.z; v[u][3] = s4.w;
            if (partial) {
                const unsigned o0 = (unsigned)(((zb * (unsigned)P.ksplit + ks) * Mext + m) * Next + n);     // < 2^25 cells per plane set
#pragma unroll
                for (int j = 0; j < 4; ++j) off[u][j] = in ? o0 + j : 0u;
            } else {
                const int ob = obase + outM[in ? rl : 0];
                if (vec_ok) {
                    const unsigned o0 = (unsigned)(ob + outN[in ? cl : 0]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) { off[u][j] = o0 + j; v[u][j] *= scale; }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) { off[u][j] = (unsigned)(ob + outN[in && j < live[u] ? cl + j : 0]); v[u][j] *= scale; }
                }
            }
        }
#define TAD_EPI_ALL(expr)                                               \
    _Pragma("unroll") for (int u = 0; u < EU; ++u)                       \
        _Pragma("unroll") for (int j = 0; j < 4; ++j) { expr; }
        for (int s = 0; s < n_epi; ++s) {
            const int op = P.epi_op[s];
            const float imm = P.epi_imm[s];
            const float *src = (op == TE_MUL_LOAD || op == TE_ADD_LOAD) ? ptrs.in[P.epi_ptr[s]] : nullptr;
            const int sb = P.epi_base[s];
            switch (op) {
            case TE_NEG: TAD_EPI_ALL(v[u][j] = -v[u][j]) break;
            case TE_EXP: TAD_EPI_ALL(v[u][j] = __expf(v[u][j])) break;
            case TE_MULC: TAD_EPI_ALL(v[u][j] *= imm) break;
            case TE_ADDC: TAD_EPI_ALL(v[u][j] += imm) break;
            case TE_SQR: TAD_EPI_ALL(v[u][j] *= v[u][j]) break;
            case TE_TANH: TAD_EPI_ALL(v[u][j] = own_tanh(v[u][j])) break;
            case TE_MUL_LOAD: case TE_ADD_LOAD: {
                float w[EU][4];
                if (vec_ok && ((sb & 3) == 0) && ((reinterpret_cast<uintptr_t>(src) & 15u) == 0)) {
#pragma unroll
                    for (int u = 0; u < EU; ++u) {
                        const float4 w4 = live[u] ? __ldg(reinterpret_cast<const float4 *>(src + (unsigned)(sb + (int)off[u][0]))) : make_float4(0.f, 0.f, 0.f, 0.f);
                        w[u][0] = w4.x; w[u][1] = w4.y; w[u][2] = w4.z; w[u][3] = w4.w;
                    }
                } else {
                    TAD_EPI_ALL(w[u][j] = j < live[u] ? __ldg(src + (unsigned)(sb + (int)off[u][j])) : 0.f)
                }
                if (op == TE_MUL_LOAD) { TAD_EPI_ALL(v[u][j] *= w[u][j]) } else { TAD_EPI_ALL(v[u][j] += w[u][j]) }
                break;
            }
            default: break;
            }
        }
#undef TAD_EPI_ALL
#pragma unroll
        for (int u = 0; u < EU; ++u) {
            if (!live[u]) continue;
            if (vec_ok) {
                float4 *dst = reinterpret_cast<float4 *>(out + off[u][0]);
                float4 r = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
                if (!partial && P.accumulate) { const float4 o = *dst; r.x += o.x; r.y += o.y; r.z += o.z; r.w += o.w; }
                *dst = r;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < live[u]) out[off[u][j]] = (!partial && P.accumulate) ? v[u][j] + out[off[u][j]] : v[u][j];
            }
        }
    }
}

// Adds the planes of partial sums of a split summation, plane 0 first, and stores the outputs.
__global__ void __launch_bounds__(256)
tad_contract_reduce(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    const unsigned Mext = (unsigned)P.M.extent, Next = (unsigned)P.N.extent;
    const unsigned per_z = Mext * Next;
    const unsigned cells = per_z * (unsigned)P.Z.extent;
    const unsigned planes = (unsigned)P.ksplit;
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += gridDim.x * blockDim.x) {
        const unsigned zb = c / per_z, rem = c - zb * per_z;
        const unsigned m = rem / Next, n = rem - m * Next;
        const float *src = ptrs.part + (size_t)zb * planes * per_z + rem;
        float sum = 0.f;
        for (unsigned s = 0; s < planes; ++s) sum += src[(size_t)s * per_z];
        const unsigned off = (unsigned)(P.baseO + decode(P.Z, zb).o + decode(P.M, m).o + decode(P.N, n).o);
        float v = epilogue(P, ptrs, sum * P.scale, off);
        if (P.accumulate) v += ptrs.out[off];
        ptrs.out[off] = v;
    }
}

// Plain or weighted sums of the rows of one operand (a contraction with a single output column):
//     out[m] (+)= scale * sum_k A[row(m) + k * stride] (* B[k])
// Bound by HBM: every element of A is read once, in pieces of 16 bytes from the first aligned one on where the row is consecutive
// (and its weights lie alike), four in flight per lane.  A warp per output, or, where that would leave the GPU idle, a block of
// eight (WARPS): 264 rows of 6523 elements.  Sums are added in a fixed order.  Four blocks to an SM (BLOCKS): short rows wait for one load
// after another and live on the warps beside them (with two, weighted 500000 x 64 197 us, 30000 x 100 13.4, strided 500000 x 9 184; with
// four 113, 7.9, 74).  Two where weighted rows are no more than that many: eight pieces in flight per lane take the registers of four blocks
// (1500 x 60000 77 and 122 us, 200 x 500000 90 and 140).
template <int WARPS, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS)
tad_rowsum_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    constexpr unsigned N = 32 * WARPS;                    // threads of a row
    __shared__ float parts[8];
    const unsigned lane = threadIdx.x % N;
    const unsigned first = WARPS == 1 ? (blockIdx.x * blockDim.x + threadIdx.x) >> 5 : blockIdx.x, step = WARPS == 1 ? (gridDim.x * blockDim.x) >> 5 : gridDim.x;
    const float *__restrict__ A = ptrs.in[P.ptrA];
    const bool weighted = P.ptrB >= 0;                   // B[k]: one weight per summation index
    const float *__restrict__ B = (weighted ? ptrs.in[P.ptrB] : A) + (weighted ? P.baseB : 0);
    const int kb = P.K.n_digits ? P.K.sB[0] : 0;
    const unsigned K = (unsigned)P.K.extent;
    const int ks = P.K.n_digits ? P.K.sA[0] : 0;
    const bool pieces = ks == 1 && (!weighted || kb == 1) && K > 32u;      // (an element a lane is not worth the alignment)
    for (unsigned m = first; m < (unsigned)P.M.extent; m += step) {
        const Parts p = decode(P.M, m);
        const int base = P.baseA + p.a;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        if (pieces) {
            const float *row = A + base;
            const unsigned off_a = (unsigned)(reinterpret_cast<uintptr_t>(row) >> 2) & 3u, off_b = (unsigned)(reinterpret_cast<uintptr_t>(B) >> 2) & 3u;
            const unsigned head = min((4u - off_a) & 3u, K), K4 = (K - head) / 4u, tail = head + 4u * K4;
            const float4 *row4 = reinterpret_cast<const float4 *>(row + head), *wts4 = reinterpret_cast<const float4 *>(B + head);
            unsigned k = lane;
            if (weighted && off_a != off_b) {
                // (the weights are the same for every row: their lines are in the L1 cache)
                const float *w = B + head;
                auto four = [&](unsigned i) { const float4 a = __ldg(row4 + i); const float *q = w + 4 * i; return (a.x * __ldg(q) + a.y * __ldg(q + 1)) + (a.z * __ldg(q + 2) + a.w * __ldg(q + 3)); };
                for (; k + N < K4; k += 2 * N) { const float a = four(k), b = four(k + N); s0 += a; s1 += b; }
                for (; k < K4; k += N) s0 += four(k);
            } else if (weighted) {
                for (; k + 3 * N < K4; k += 4 * N) {
                    const float4 a = __ldg(row4 + k), b = __ldg(row4 + k + N), c = __ldg(row4 + k + 2 * N), d = __ldg(row4 + k + 3 * N);
                    const float4 wa = __ldg(wts4 + k), wb = __ldg(wts4 + k + N), wc = __ldg(wts4 + k + 2 * N), wd = __ldg(wts4 + k + 3 * N);
                    s0 += (a.x * wa.x + a.y * wa.y) + (a.z * wa.z + a.w * wa.w); s1 += (b.x * wb.x + b.y * wb.y) + (b.z * wb.z + b.w * wb.w);
                    s2 += (c.x * wc.x + c.y * wc.y) + (c.z * wc.z + c.w * wc.w); s3 += (d.x * wd.x + d.y * wd.y) + (d.z * wd.z + d.w * wd.w);
                }
                for (; k < K4; k += N) { const float4 a = __ldg(row4 + k), wa = __ldg(wts4 + k); s0 += (a.x * wa.x + a.y * wa.y) + (a.z * wa.z + a.w * wa.w); }
            } else {
                for (; k + 3 * N < K4; k += 4 * N) {
                    const float4 a = __ldg(row4 + k), b = __ldg(row4 + k + N), c = __ldg(row4 + k + 2 * N), d = __ldg(row4 + k + 3 * N);
                    s0 += (a.x + a.y) + (a.z + a.w); s1 += (b.x + b.y) + (b.z + b.w);
                    s2 += (c.x + c.y) + (c.z + c.w); s3 += (d.x + d.y) + (d.z + d.w);
                }
                for (; k < K4; k += N) { const float4 a = __ldg(row4 + k); s0 += (a.x + a.y) + (a.z + a.w); }
            }
            if (lane < head) s1 = weighted ? fmaf(__ldg(row + lane), __ldg(B + lane), s1) : s1 + __ldg(row + lane);
            if (tail + lane < K) s2 = weighted ? fmaf(__ldg(row + tail + lane), __ldg(B + tail + lane), s2) : s2 + __ldg(row + tail + lane);
        } else {
            unsigned k = lane;
            auto at = [&](unsigned i) { return __ldg(A + (unsigned)(base + (int)i * ks)); };
            auto wt = [&](unsigned i) { return __ldg(ptrs.in[P.ptrB] + (unsigned)(P.baseB + (int)i * kb)); };
            if (weighted) {
                for (; k + 3 * N < K; k += 4 * N) { s0 = fmaf(at(k), wt(k), s0); s1 = fmaf(at(k + N), wt(k + N), s1); s2 = fmaf(at(k + 2 * N), wt(k + 2 * N), s2); s3 = fmaf(at(k + 3 * N), wt(k + 3 * N), s3); }
                for (; k < K; k += N) s0 = fmaf(at(k), wt(k), s0);
            } else {
                for (; k + 3 * N < K; k += 4 * N) { const float a = at(k), b = at(k + N), c = at(k + 2 * N), d = at(k + 3 * N); s0 += a; s1 += b; s2 += c; s3 += d; }
                for (; k < K; k += N) s0 += at(k);
            }
        }
        float s = (s0 + s1) + (s2 + s3);
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if constexpr (WARPS > 1) {
            if ((threadIdx.x & 31u) == 0) parts[threadIdx.x >> 5] = s;
            __syncthreads();
            s = ((parts[0] + parts[1]) + (parts[2] + parts[3])) + ((parts[4] + parts[5]) + (parts[6] + parts[7]));
            __syncthreads();
        }
        if (lane == 0) {
            const unsigned off = (unsigned)(P.baseO + p.o);
            float v = s * P.scale;
            if (P.accumulate) v += ptrs.out[off];
            ptrs.out[off] = v;
        }
    }
}

// Plain or weighted sums of an operand that is consecutive along its row index:
//     out[m] = sum_k A[m + k * stride] (* B[k]),   a thread per m, a slice of k per block row (grid.y);
// consecutive threads read consecutive elements, four loads in flight per thread.  Slices write planes of
// partial sums that tad_contract_reduce adds in order.
__global__ void __launch_bounds__(256)
tad_colsum_kernel(const __grid_constant__ TadcProgram P, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    const unsigned m = blockIdx.x * 256u + threadIdx.x;
    const unsigned Mext = (unsigned)P.M.extent, K = (unsigned)P.K.extent;
    if (m >= Mext) return;
    const float *__restrict__ A = ptrs.in[P.ptrA];
    const bool weighted = P.ptrB >= 0;
    const float *__restrict__ B = weighted ? ptrs.in[P.ptrB] : A;
    const int ks = P.K.sA[0], kb = P.K.sB[0];
    const unsigned kbeg = blockIdx.y * (unsigned)P.kchunk, kend = min(K, kbeg + (unsigned)P.kchunk);
    const int base = P.baseA + (int)m * P.M.sA[0];
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    unsigned k = kbeg;
    for (; k + 7 < kend; k += 8) {
        float a[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] = __ldg(A + (unsigned)(base + (int)(k + u) * ks));
        if (weighted) {
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] *= __ldg(B + (unsigned)(P.baseB + (int)(k + u) * kb));
        }
        s0 += a[0] + a[4]; s1 += a[1] + a[5]; s2 += a[2] + a[6]; s3 += a[3] + a[7];
    }
    for (; k < kend; ++k) {
        const float a0 = __ldg(A + (unsigned)(base + (int)k * ks));
        s0 = weighted ? fmaf(a0, __ldg(B + (unsigned)(P.baseB + (int)k * kb)), s0) : s0 + a0;
    }
    const float s = (s0 + s1) + (s2 + s3);
    if (P.ksplit > 1) ptrs.part[(size_t)blockIdx.y * Mext + m] = s;
    else {
        const unsigned off = (unsigned)(P.baseO + (int)m * P.M.sO[0]);
        float v = s * P.scale;
        if (P.accumulate) v += ptrs.out[off];
        ptrs.out[off] = v;
    }
}

template <int BM, int BN, int TM, int TN>
cudaError_t launch_shape(const TadcProgram &P, const TadpPointers &ptrs, cudaStream_t stream)
{
    using C = Cfg<BM, BN, TM, TN>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    auto kern = tad_contract_kernel<BM, BN, TM, TN>;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    const unsigned tiles_m = ((unsigned)P.M.extent + BM - 1) / BM, tiles_n = ((unsigned)P.N.extent + BN - 1) / BN;
    dim3 grid(tiles_m * tiles_n, (unsigned)std::max(1, P.ksplit), (unsigned)P.Z.extent);
    tad_launch(kern, grid, C::NT, C::SMEM, stream, P, ptrs, tiles_m, tiles_n);
    return cudaGetLastError();
}

}  // namespace

cudaError_t tad_launch_mma(const TadcProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream);

cudaError_t tad_launch_contract(const TadcProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream)
{
    if (P.M.extent <= 0 || P.N.extent <= 0 || P.Z.extent <= 0) return cudaSuccess;
    if (P.shape == 7) return tad_launch_mma(P, ptrs, sms, stream);
    if (P.shape == 6) {
        dim3 grid(((unsigned)P.M.extent + 255u) / 256u, (unsigned)std::max(1, P.ksplit), 1u);
        tad_launch(tad_colsum_kernel, grid, 256, 0, stream, P, ptrs);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess && P.ksplit > 1) {
            const unsigned blocks = (unsigned)std::min<unsigned long long>(((unsigned long long)P.M.extent + 255) / 256, (unsigned long long)sms * 8);
            tad_launch(tad_contract_reduce, blocks, 256, 0, stream, P, ptrs);
            e = cudaGetLastError();
        }
        return e;
    }
    if (P.shape == 4) {
        // (weighted rows, warp / block a row, us: 264 of 512 2.1 / 2.3, of 1024 2.5 / 2.4, of 8192 7.5 / 3.0; 592 of 1024 2.5 / 2.8, of 4096
        // 4.7 / 3.0; 1100 of 1024 2.6 / 4.0, of 4096 4.9 / 4.5; 1200 rows are eight warps to an SM)
        const unsigned rows = (unsigned)P.M.extent;
        const bool by_block = rows < sms * 8u && (unsigned)P.K.extent >= std::max(512u, 4u * rows);
        const unsigned blocks = by_block ? rows : (rows + 7u) / 8u;
        const bool few = P.ptrB >= 0 && blocks <= sms * 2u;
        auto kernel = by_block ? (few ? tad_rowsum_kernel<8, 2> : tad_rowsum_kernel<8, 4>) : (few ? tad_rowsum_kernel<1, 2> : tad_rowsum_kernel<1, 4>);
        tad_launch(kernel, std::min(blocks, by_block ? blocks : sms * 16u), 256, 0, stream, P, ptrs);
        return cudaGetLastError();
    }
    cudaError_t e = P.shape == 1 ? launch_shape<128, 32, 8, 4>(P, ptrs, stream)
                  : P.shape == 3 ? launch_shape<128, 36, 8, 4>(P, ptrs, stream)
                  : P.shape == 2 ? launch_shape<128, 64, 8, 4>(P, ptrs, stream) : launch_shape<128, 128, 8, 8>(P, ptrs, stream);
    if (e != cudaSuccess) return e;
    if (P.ksplit > 1) {
        const unsigned long long cells = (unsigned long long)P.M.extent * P.N.extent * P.Z.extent;
        const unsigned blocks = (unsigned)std::min<unsigned long long>((cells + 255) / 256, (unsigned long long)sms * 8);
        tad_launch(tad_contract_reduce, blocks, 256, 0, stream, P, ptrs);
        e = cudaGetLastError();
    }
    return e;
}
