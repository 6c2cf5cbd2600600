// Element-wise kernel: programs without loops (forward passes of expressions without sums, function
// tables, operand matrices of contractions, the element-wise remainder of a factored kernel).
//
// The program is a short accumulator program over two value registers X and Y (ew.h), every step
// dispatched once for the four consecutive outputs a thread owns along the output's contiguous
// variable; a thread block covers a tile of rows x 4-element columns chosen so that short rows still
// fill the block.  Index arithmetic: the row number is split into the outer variables with
// multiply-shift divisions prepared by the host, every load's offset is its affine form in those
// variables.  Loads whose offset steps by +1 along the row and are 16-byte aligned are 128-bit loads,
// loads that do not move along the row are read once; the store is one 128-bit store.
#include <cuda_runtime.h>

#include <algorithm>

#include "launch.h"
#include "ew.h"
#include "vm.cuh"

namespace {

using tadvm::apply_fn;
using tadvm::fast_sincos;
using tadvm::fast_tanh;

constexpr int EG = 4;          // groups of four consecutive outputs per thread, one block-wide row segment apart

__global__ void __launch_bounds__(256)
tad_ew_kernel(const __grid_constant__ TadeProgram P, const __grid_constant__ TadpPointers ptrs, const unsigned n_items,
              const unsigned cols, const unsigned lane_blocks, const unsigned n_rows)
{
    tad_wait_previous();
    const unsigned tid = threadIdx.x;
    const unsigned rows_per_block = 256u / cols;
    const unsigned tc = tid % cols, tr = tid / cols;
    const int lane_var = P.lane_var;
    const unsigned lane_ext = (unsigned)P.outer_ext[lane_var];
    const unsigned gstride = cols * 4u;                       // elements between two groups of a thread
    const bool few_vars = P.n_outer <= 4;
    for (unsigned item = blockIdx.x; item < n_items; item += gridDim.x) {
        const unsigned lb = item % lane_blocks, rb = item / lane_blocks;
        const unsigned row = rb * rows_per_block + tr, lane0 = lb * gstride * EG + tc * 4u;
        if (row >= n_rows || lane0 >= lane_ext) continue;
        int live[EG];
#pragma unroll
        for (int g = 0; g < EG; ++g) { const unsigned l = lane0 + g * gstride; live[g] = l >= lane_ext ? 0 : (int)min(4u, lane_ext - l); }
        // outer variables of this row (the lane variable holds the first of the thread's elements)
        int var[TADP_MAX_VARS];
        unsigned rem = row;
#pragma unroll
        for (int v = TADP_MAX_VARS - 1; v >= 0; --v) {
            var[v] = 0;
            if (v < P.n_outer) {
                if (v == lane_var) var[v] = P.outer_lo[v] + (int)lane0;
                else {
                    const unsigned q = (unsigned)(((unsigned long long)rem * (unsigned)P.div_mul[v]) >> P.div_shift[v]);
                    var[v] = P.outer_lo[v] + (int)(rem - q * (unsigned)P.outer_ext[v]);
                    rem = q;
                }
            }
        }
        // offset = base + coef . var (the variables stay in registers: every index below is a compile-time constant)
#define TAD_EW_AFFINE(off, coef, base)                                                                   \
    unsigned off = (unsigned)(base);                                                                       \
    if (few_vars) { _Pragma("unroll") for (int v = 0; v < 4; ++v) off += (unsigned)(coef)[v] * (unsigned)var[v]; } \
    else { _Pragma("unroll") for (int v = 0; v < TADP_MAX_VARS; ++v) off += (unsigned)(coef)[v] * (unsigned)var[v]; }
        float X[EG][4], Y[EG][4];
#pragma unroll
        for (int g = 0; g < EG; ++g)
#pragma unroll
            for (int j = 0; j < 4; ++j) { X[g][j] = 0.f; Y[g][j] = 0.f; }
#define TAD_EW_ALL(expr)                                                \
    _Pragma("unroll") for (int g = 0; g < EG; ++g)                       \
        _Pragma("unroll") for (int j = 0; j < 4; ++j) { expr; }
        for (int s = 0; s < P.n_steps; ++s) {
            const TadeStep st = P.steps[s];
            switch (st.op) {
            case E_LD: {
                const TadpLoad &L = P.loads[st.a];
                TAD_EW_AFFINE(off0, L.coef, L.base)
                const int step = L.coef[lane_var];
                const float *__restrict__ src = ptrs.in[L.ptr];
                const bool wide = step == 1 && ((off0 & 3u) == 0) && ((reinterpret_cast<uintptr_t>(src) & 15u) == 0);
                const float first = step == 0 ? __ldg(src + off0) : 0.f;
#pragma unroll
                for (int g = 0; g < EG; ++g) {
                    float v4[4];
                    const unsigned off = (unsigned)((int)off0 + g * (int)gstride * step);
                    if (step == 0) { v4[0] = v4[1] = v4[2] = v4[3] = first; }
                    else if (wide && live[g] == 4) {
                        const float4 q = __ldg(reinterpret_cast<const float4 *>(src + off));
                        v4[0] = q.x; v4[1] = q.y; v4[2] = q.z; v4[3] = q.w;
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v4[j] = j < live[g] ? __ldg(src + (unsigned)((int)off + j * step)) : 0.f;
                    }
                    if (st.b == 0) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) X[g][j] = v4[j];
                    } else if (st.b == 1) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) X[g][j] += v4[j];
                    } else if (st.b == 2) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) X[g][j] *= v4[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) { const float t = X[g][j] + v4[j]; X[g][j] = t * t; }
                    }
                }
                break;
            }
            case E_PUSH: TAD_EW_ALL(Y[g][j] = X[g][j]) break;
            case E_CONST: TAD_EW_ALL(X[g][j] = st.imm) break;
            case E_NEG: TAD_EW_ALL(X[g][j] = -X[g][j]) break;
            case E_SQR: TAD_EW_ALL(X[g][j] *= X[g][j]) break;
            case E_CUBE: TAD_EW_ALL(X[g][j] = X[g][j] * X[g][j] * X[g][j]) break;
            case E_MULC: TAD_EW_ALL(X[g][j] *= st.imm) break;
            case E_ADDC: TAD_EW_ALL(X[g][j] += st.imm) break;
            case E_ADDY: TAD_EW_ALL(X[g][j] = Y[g][j] + X[g][j]) break;
            case E_SUBY: TAD_EW_ALL(X[g][j] = Y[g][j] - X[g][j]) break;
            case E_MULY: TAD_EW_ALL(X[g][j] = Y[g][j] * X[g][j]) break;
            case E_DIVY: TAD_EW_ALL(X[g][j] = Y[g][j] / X[g][j]) break;
            case E_FN:
                // (every loop over the values is fully unrolled: X and Y must stay in registers)
                switch (st.b) {
                case F_EXP: TAD_EW_ALL(X[g][j] = __expf(X[g][j])) break;
                case F_TANH: TAD_EW_ALL(X[g][j] = fast_tanh(X[g][j])) break;
                case F_SIN: TAD_EW_ALL(X[g][j] = fabsf(X[g][j]) < 8192.f ? fast_sincos(X[g][j], 0) : apply_fn(F_SIN, X[g][j], 0)) break;
                case F_COS: TAD_EW_ALL(X[g][j] = fabsf(X[g][j]) < 8192.f ? fast_sincos(X[g][j], 1) : apply_fn(F_COS, X[g][j], 0)) break;
                default: TAD_EW_ALL(X[g][j] = apply_fn(st.b, X[g][j], st.a)) break;
                }
                break;
            default: break;
            }
        }
#undef TAD_EW_ALL
        float *__restrict__ out = ptrs.out;
        const int ostep = P.out_coef[lane_var];
        TAD_EW_AFFINE(out0, P.out_coef, P.out_base)
        const bool wide_out = ostep == 1 && ((out0 & 3u) == 0) && ((reinterpret_cast<uintptr_t>(out) & 15u) == 0);
#pragma unroll
        for (int g = 0; g < EG; ++g) {
            const unsigned out_off = (unsigned)((int)out0 + g * (int)gstride * ostep);
            if (wide_out && live[g] == 4) {
                float4 *dst = reinterpret_cast<float4 *>(out + out_off);
                float4 r = make_float4(X[g][0], X[g][1], X[g][2], X[g][3]);
                if (P.accumulate) { const float4 o = *dst; r.x += o.x; r.y += o.y; r.z += o.z; r.w += o.w; }
                *dst = r;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < live[g]) { const unsigned o = (unsigned)((int)out_off + j * ostep); out[o] = P.accumulate ? out[o] + X[g][j] : X[g][j]; }
            }
        }
#undef TAD_EW_AFFINE
    }
}


// ---------------------------------------------------------------------------------------------------------
// Products of loads.  Most element-wise kernels that remain after the function tables are
//     out = c * L_1^e1 * L_2^e2 * ...        (e in 1..3),
// and at one multiplication per load the index arithmetic of the general program dominates.  Here a thread
// owns four outputs of a row and walks a run of consecutive rows along another outer variable, so the
// variables are decoded once per run and every offset advances by a constant per row.  Two layouts:
//   vector:      the four outputs are consecutive; every load that moves along the row is a 128-bit load
//                (forward, or reversed for offsets that step by -1), which the host has proven aligned in every row;
//   interleaved: output j of a thread lies j * (threads per row) further, so that plain loads of neighbouring
//                threads fall into the same lines whatever the load's step.
// Loads that do not change from row to row are read once per run, loads that do not move along the row once per row.  What bounds
// it is the latency of the reads (the tables live in L1 and L2): every load of the rows in flight is issued before the first is
// used, without a branch between them (sin x[2i + j, j - k] y^2 over 512^3 outputs 132 -> 104 us, 300^3 46 -> 31, a table read along
// steps of three, 4096 x 4096 outputs, 37 -> 27 us).  Where a thread has one piece only there is nothing to keep in flight, and the
// registers for it cost warps (x y w over 10^6 outputs 7.8 us with them, 5.5 without; x y over 2 10^6 9.3, 7.8): builds of their own.
// ---------------------------------------------------------------------------------------------------------
enum ProdKind : int { PK_HOIST = 0, PK_BCAST, PK_FWD, PK_REV, PK_GEN };

struct ProdLoad { int32_t load, kind, exp; };
struct ProdPlan {
    int32_t n_loads, n_moving, n_single, row_var, run, vec;      // moving loads first, n_single of them read once a row (behind the others);
    float c;                                                     // run: rows per thread along row_var, or pieces of a single row (row_var < 0)
    ProdLoad ld[4];
};

__device__ __forceinline__ float powe(float v, int e) { return e == 1 ? v : e == 2 ? v * v : v * v * v; }

// where a run stands: offsets of its loads and of its output, and what they advance by from row to row
struct ProdRun { const float *src[3]; int off[3], step[3], adv[3], exp[3]; bool rev[3]; int out, ostep, oadv; };

// U rows: MG loads with a value for each of the four outputs, in pieces of W, and MB with one.  Outputs from `live` on lie outside
// the row (interleaved layout): their values are read where the first one's are and not stored.
template <bool VEC, int W, int MG, int MB, int U>
__device__ __forceinline__ void prod_rows(ProdRun &R, const int live, const float (&held)[4], const bool powers, const bool accumulate, float *__restrict__ out)
{
    float v[U][MG > 0 ? MG : 1][4], b[U][MB > 0 ? MB : 1];
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int l = 0; l < MG; ++l) {
            const float *__restrict__ s = R.src[l];
            const int o = R.off[l];
            if constexpr (W == 4) {
                const float4 q = __ldg(reinterpret_cast<const float4 *>(s + (unsigned)(R.rev[l] ? o - 3 : o)));
                v[u][l][0] = R.rev[l] ? q.w : q.x; v[u][l][1] = R.rev[l] ? q.z : q.y; v[u][l][2] = R.rev[l] ? q.y : q.z; v[u][l][3] = R.rev[l] ? q.x : q.w;
            } else if constexpr (W == 2) {
                const float2 q0 = __ldg(reinterpret_cast<const float2 *>(s + (unsigned)(R.rev[l] ? o - 1 : o)));
                const float2 q1 = __ldg(reinterpret_cast<const float2 *>(s + (unsigned)(R.rev[l] ? o - 3 : o + 2)));
                v[u][l][0] = R.rev[l] ? q0.y : q0.x; v[u][l][1] = R.rev[l] ? q0.x : q0.y; v[u][l][2] = R.rev[l] ? q1.y : q1.x; v[u][l][3] = R.rev[l] ? q1.x : q1.y;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) v[u][l][j] = __ldg(s + (unsigned)(VEC || j < live ? o + j * R.step[l] : o));
            }
            R.off[l] += R.adv[l];
        }
#pragma unroll
        for (int l = 0; l < MB; ++l) { b[u][l] = __ldg(R.src[MG + l] + (unsigned)R.off[MG + l]); R.off[MG + l] += R.adv[MG + l]; }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        float q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = held[j];
#pragma unroll
        for (int l = 0; l < MG; ++l)
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] *= powers ? powe(v[u][l][j], R.exp[l]) : v[u][l][j];
#pragma unroll
        for (int l = 0; l < MB; ++l) {
            const float f = powers ? powe(b[u][l], R.exp[MG + l]) : b[u][l];
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] *= f;
        }
        if constexpr (VEC) {
            float4 *dst = reinterpret_cast<float4 *>(out + (unsigned)R.out);
            float4 r = make_float4(q[0], q[1], q[2], q[3]);
            if (accumulate) { const float4 o = *dst; r.x += o.x; r.y += o.y; r.z += o.z; r.w += o.w; }
            *dst = r;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (j < live) { const unsigned o = (unsigned)(R.out + j * R.ostep); out[o] = accumulate ? out[o] + q[j] : q[j]; }
        }
        R.out += R.oadv;
    }
}

template <bool VEC, int W, int MG, int MB, int U>
__device__ __forceinline__ void prod_run(ProdRun &R, const int n_rows, const int live, const float (&held)[4], const bool powers, const bool accumulate, float *__restrict__ out)
{
    int r = 0;
    for (; r + U <= n_rows; r += U) prod_rows<VEC, W, MG, MB, U>(R, live, held, powers, accumulate, out);
#pragma unroll 1
    for (; r < n_rows; ++r) prod_rows<VEC, W, MG, MB, 1>(R, live, held, powers, accumulate, out);
}

// SINGLE: one long row, its runs along it, a block's width from one piece to the next; ONE: runs of one piece
template <bool VEC, int MG, int MB, bool SINGLE, bool ONE>
__global__ void __launch_bounds__(256, ONE ? 6 - (MG + 1) / 2 : VEC && MG + MB <= 1 ? 6 : VEC && MG + MB == 2 ? 4 : !VEC && MG + MB == 3 ? 4 : 3)
tad_prod_kernel(const __grid_constant__ TadeProgram P, const __grid_constant__ ProdPlan Q, const __grid_constant__ TadpPointers ptrs,
                const unsigned n_items, const unsigned cols, const unsigned lane_blocks, const unsigned n_runs, const unsigned runs_per_line)
{
    tad_wait_previous();
    constexpr int M = MG + MB, U = ONE ? 1 : VEC && MG + MB <= 2 ? 4 : !VEC && MG + MB == 3 ? 1 : 2;      // (as many as their registers allow)
    const unsigned tid = threadIdx.x;
    const unsigned rows_per_block = 256u / cols;
    const unsigned tc = tid % cols, tr = tid / cols;
    const int lane_var = P.lane_var, row_var = Q.row_var;
    const unsigned lane_ext = (unsigned)P.outer_ext[lane_var];
    const unsigned es = VEC ? 1u : cols;                       // distance between two outputs of a thread
    const bool accumulate = P.accumulate != 0;
    float *__restrict__ out = ptrs.out;
    for (unsigned item = blockIdx.x; item < n_items; item += gridDim.x) {
        const unsigned lb = item % lane_blocks, rb = item / lane_blocks;
        const unsigned run = rb * rows_per_block + tr;
        const unsigned lane0 = lb * cols * 4u * (SINGLE ? (unsigned)Q.run : 1u) + (VEC ? tc * 4u : tc);
        if (run >= n_runs || lane0 >= lane_ext) continue;
        auto inside = [&](unsigned lane) {                     // outputs of this thread inside the row
            return lane >= lane_ext ? 0 : VEC ? (int)min(4u, lane_ext - lane) : (int)min(4u, (lane_ext - lane + cols - 1u) / cols);
        };
        int live = inside(lane0);
        // the run: its position along row_var, then the other outer variables
        const unsigned piece = run % runs_per_line;
        unsigned rem = run / runs_per_line;
        int var[TADP_MAX_VARS];
#pragma unroll
        for (int v = TADP_MAX_VARS - 1; v >= 0; --v) {
            var[v] = 0;
            if (v < P.n_outer) {
                if (v == lane_var) var[v] = P.outer_lo[v] + (int)lane0;
                else if (v == row_var) var[v] = P.outer_lo[v] + (int)(piece * (unsigned)Q.run);
                else {
                    const unsigned q = (unsigned)(((unsigned long long)rem * (unsigned)P.div_mul[v]) >> P.div_shift[v]);
                    var[v] = P.outer_lo[v] + (int)(rem - q * (unsigned)P.outer_ext[v]);
                    rem = q;
                }
            }
        }
        const unsigned whole = SINGLE && live == 4 ? (lane_ext - 1u - 3u * es - lane0) / (4u * cols) + 1u : 1u;      // pieces of four
        const int n_rows = SINGLE ? (int)min((unsigned)Q.run, whole) : min(Q.run, P.outer_ext[row_var] - (int)(piece * (unsigned)Q.run));
        // loads that stay put from row to row are multiplied into one factor per output (with the constant); the
        // others ("moving", first in Q.ld) keep an offset that advances by a constant per row
        float held[4] = {Q.c, Q.c, Q.c, Q.c};
        ProdRun R;
        bool powers = false;
        int width = 4;                                         // values per vector load in this run
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            if (l >= Q.n_loads) continue;
            const TadpLoad &L = P.loads[Q.ld[l].load];
            int o = L.base;
#pragma unroll
            for (int v = 0; v < TADP_MAX_VARS; ++v) o += L.coef[v] * var[v];
            const int st = L.coef[lane_var] * (int)es;
            if (l >= M) {
                const float *__restrict__ src = ptrs.in[L.ptr];
#pragma unroll
                for (int j = 0; j < 4; ++j) if (j < live) held[j] *= powe(__ldg(src + (unsigned)(o + j * st)), Q.ld[l].exp);
            } else if (l < 3) {
                R.src[l] = ptrs.in[L.ptr]; R.off[l] = o; R.step[l] = st; R.exp[l] = Q.ld[l].exp;
                R.adv[l] = SINGLE ? L.coef[lane_var] * (int)(4u * cols) : L.coef[row_var];
                R.rev[l] = Q.ld[l].kind == PK_REV;
                powers = powers || R.exp[l] != 1;
                if (l < MG) {
                    const unsigned first = (unsigned)(R.rev[l] ? o - 3 : o);
                    width = min(width, (first & 3u) == 0 ? 4 : (first & 1u) == 0 ? 2 : 1);
                }
            }
        }
        R.out = P.out_base;
#pragma unroll
        for (int v = 0; v < TADP_MAX_VARS; ++v) R.out += P.out_coef[v] * var[v];
        R.ostep = P.out_coef[lane_var] * (int)es; R.oadv = SINGLE ? P.out_coef[lane_var] * (int)(4u * cols) : P.out_coef[row_var];
        if constexpr (M == 0 && ONE) {
            if (VEC && live == 4) {
                float4 *dst = reinterpret_cast<float4 *>(out + (unsigned)R.out);
                float4 q = make_float4(held[0], held[1], held[2], held[3]);
                if (accumulate) { const float4 o = *dst; q.x += o.x; q.y += o.y; q.z += o.z; q.w += o.w; }
                *dst = q;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) if (j < live) { const unsigned o = (unsigned)(R.out + j * R.ostep); out[o] = accumulate ? out[o] + held[j] : held[j]; }
            }
            continue;
        }
        if (ONE && live == 4) {
            if constexpr (ONE && M > 0) {                      // (one piece: no loop, no remainder behind it)
                if (width == 4) prod_rows<VEC, 4, MG, MB, 1>(R, live, held, powers, accumulate, out);
                else if (width == 2) prod_rows<VEC, 2, MG, MB, 1>(R, live, held, powers, accumulate, out);
                else prod_rows<VEC, 1, MG, MB, 1>(R, live, held, powers, accumulate, out);
            }
            continue;
        }
        if (!ONE && (!VEC || live == 4)) {
            if constexpr (ONE) {}
            else if constexpr (!VEC || MG == 0) prod_run<VEC, 1, MG, MB, U>(R, n_rows, live, held, powers, accumulate, out);
            else if (width == 4) prod_run<VEC, 4, MG, MB, U>(R, n_rows, live, held, powers, accumulate, out);
            else if (width == 2) prod_run<VEC, 2, MG, MB, U>(R, n_rows, live, held, powers, accumulate, out);
            else prod_run<VEC, 1, MG, MB, U>(R, n_rows, live, held, powers, accumulate, out);
            live = SINGLE && live == 4 && n_rows < Q.run ? inside(lane0 + (unsigned)n_rows * 4u * cols) : 0;
            if (live == 0) continue;
        }
        // the last outputs of a row that is no multiple of four
#pragma unroll 1
        for (int r = 0; r < (SINGLE ? 1 : n_rows); ++r) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if (j >= live) continue;
                float q = held[j];
#pragma unroll
                for (int l = 0; l < M; ++l) q *= powe(__ldg(R.src[l] + (unsigned)(R.off[l] + (l < MG ? j * R.step[l] : 0))), R.exp[l]);
                const unsigned o = (unsigned)(R.out + j * R.ostep);
                out[o] = accumulate ? out[o] + q : q;
            }
#pragma unroll
            for (int l = 0; l < M; ++l) R.off[l] += R.adv[l];
            R.out += R.oadv;
        }
    }
}

// c * product of powers of loads, read off the accumulator program; false when the program is anything else
bool product_form(const TadeProgram &P, ProdPlan &Q)
{
    struct Group { float c; int exp[TADE_MAX_LOADS]; bool any; };
    Group x{}, y{};
    bool have_x = false, have_y = false;
    auto raise = [](Group &g, int k) {
        for (int l = 0; l < TADE_MAX_LOADS; ++l) { g.exp[l] *= k; if (g.exp[l] > 3) return false; }
        g.c = k == 2 ? g.c * g.c : g.c * g.c * g.c;
        return true;
    };
    for (int s = 0; s < P.n_steps; ++s) {
        const TadeStep &st = P.steps[s];
        switch (st.op) {
        case E_LD:
            if (st.a < 0 || st.a >= TADE_MAX_LOADS) return false;
            if (st.b == 0) { x = Group{}; x.c = 1.f; x.exp[st.a] = 1; have_x = true; }
            else if (st.b == 2 && have_x) { if (++x.exp[st.a] > 3) return false; }
            else return false;
            break;
        case E_PUSH: if (!have_x || have_y) return false; y = x; have_y = true; have_x = false; break;
        case E_NEG: if (!have_x) return false; x.c = -x.c; break;
        case E_MULC: if (!have_x) return false; x.c *= st.imm; break;
        case E_SQR: if (!have_x || !raise(x, 2)) return false; break;
        case E_CUBE: if (!have_x || !raise(x, 3)) return false; break;
        case E_MULY:
            if (!have_x || !have_y) return false;
            x.c *= y.c;
            for (int l = 0; l < TADE_MAX_LOADS; ++l) { x.exp[l] += y.exp[l]; if (x.exp[l] > 3) return false; }
            have_y = false;
            break;
        default: return false;
        }
    }
    if (!have_x || have_y) return false;
    Q = ProdPlan{};
    Q.c = x.c;
    for (int l = 0; l < TADE_MAX_LOADS; ++l)
        if (x.exp[l] > 0) {
            if (Q.n_loads == 4 || l >= P.n_loads) return false;
            Q.ld[Q.n_loads].load = l; Q.ld[Q.n_loads].exp = x.exp[l]; ++Q.n_loads;
        }
    return Q.n_loads > 0;
}

// layout and load kinds of a product program; the row variable is the innermost outer variable besides the lane variable
bool plan_product(const TadeProgram &P, const TadpPointers &ptrs, unsigned sms, ProdPlan &Q)
{
    const int lane = P.lane_var;
    Q.row_var = -1;
    for (int v = P.n_outer - 1; v >= 0; --v) if (v != lane && P.outer_ext[v] > 1) { Q.row_var = v; break; }
    double elems = 1;
    for (int v = 0; v < P.n_outer; ++v) elems *= (double)P.outer_ext[v];
    // rows per thread: as many as leave every SM a few thousand threads
    int run = 1;
    while (run < 32 && elems / (4.0 * run * 2) >= (double)sms * 2048.0) run *= 2;
    Q.run = Q.row_var < 0 ? run : std::min(run, P.outer_ext[Q.row_var]);
    // the output is stored in 128-bit pieces when its first element of every row is a multiple of four; a load needs
    // only a row step that is one (the width of its vector loads is settled per run)
    auto aligned = [&](const int32_t *coef, int64_t base) {
        int64_t o = base;
        for (int v = 0; v < P.n_outer; ++v) { o += (int64_t)coef[v] * P.outer_lo[v]; if (v != lane && P.outer_ext[v] > 1 && coef[v] % 4 != 0) return false; }
        return o % 4 == 0;
    };
    bool vec = P.out_coef[lane] == 1 && aligned(P.out_coef, P.out_base) && (reinterpret_cast<uintptr_t>(ptrs.out) & 15u) == 0;
    for (int i = 0; i < Q.n_loads; ++i) {
        const TadpLoad &L = P.loads[Q.ld[i].load];
        const int step = L.coef[lane], adv = Q.row_var < 0 ? 4 * step : L.coef[Q.row_var];
        const bool base16 = (reinterpret_cast<uintptr_t>(ptrs.in[L.ptr]) & 15u) == 0;
        int kind = PK_GEN;
        // (a run of a single row: loads move only in so far as that lets them be read in pieces)
        if (Q.run == 1 ? !(base16 && std::abs(step) == 1) : adv == 0) kind = PK_HOIST;
        else if (step == 0) kind = PK_BCAST;
        else if (step == 1 && base16 && (adv % 4 == 0 || Q.run == 1)) kind = PK_FWD;
        else if (step == -1 && base16 && (adv % 4 == 0 || Q.run == 1)) kind = PK_REV;
        if (kind == PK_GEN) vec = false;
        Q.ld[i].kind = kind;
    }
    if (Q.run == 1 && (!vec || Q.row_var >= 0)) for (int i = 0; i < Q.n_loads; ++i) Q.ld[i].kind = PK_HOIST;
    // moving loads first, those read once a row behind the others
    auto rank = [](const ProdLoad &a) { return a.kind == PK_HOIST ? 2 : a.kind == PK_BCAST ? 1 : 0; };
    std::stable_sort(Q.ld, Q.ld + Q.n_loads, [&](const ProdLoad &a, const ProdLoad &b) { return rank(a) < rank(b); });
    Q.n_moving = Q.n_single = 0;
    for (int i = 0; i < Q.n_loads; ++i) { Q.n_moving += Q.ld[i].kind != PK_HOIST; Q.n_single += Q.ld[i].kind == PK_BCAST; }
    Q.vec = vec ? 1 : 0;
    return Q.n_moving <= 3;
}

}  // namespace

cudaError_t tad_launch_ew(const TadeProgram &P, const TadpPointers &ptrs, unsigned sms, cudaStream_t stream)
{
    const unsigned lane_ext = (unsigned)P.outer_ext[P.lane_var];
    unsigned long long rows = 1;
    for (int v = 0; v < P.n_outer; ++v) if (v != P.lane_var) rows *= (unsigned long long)P.outer_ext[v];
    if (lane_ext == 0 || rows == 0) return cudaSuccess;
    ProdPlan Q;
    if (product_form(P, Q) && plan_product(P, ptrs, sms, Q)) {
        unsigned pc = 1;
        while (pc < 256u && pc * 4u < lane_ext) pc *= 2u;
        if (!Q.vec && pc < 32u) pc = 32u;                      // interleaved outputs: a warp covers a run of 32 columns
        const unsigned per_block = 256u / pc;
        const unsigned per_run = pc * 4u * (Q.row_var < 0 ? (unsigned)Q.run : 1u), lblocks = (lane_ext + per_run - 1u) / per_run;
        const unsigned long long row_ext = Q.row_var < 0 ? 1ull : (unsigned long long)P.outer_ext[Q.row_var];
        const unsigned long long per_line = Q.row_var < 0 ? 1ull : (row_ext + Q.run - 1) / Q.run;
        const unsigned long long runs = rows / row_ext * per_line;
        const unsigned long long its = ((runs + per_block - 1) / per_block) * lblocks;
        if (its >= (1ull << 32) || runs >= (1ull << 31)) return cudaErrorInvalidValue;
        const unsigned g = (unsigned)std::min<unsigned long long>(its, (unsigned long long)sms * 32ull);
#define TAD_PROD_ARGS g, 256, 0, stream, P, Q, ptrs, (unsigned)its, pc, lblocks, (unsigned)runs, (unsigned)per_line
#define TAD_PROD_LAUNCH(G, B)                                                                                                           \
    case 4 * G + B:                                                                                                                     \
        if (Q.row_var < 0) { if (Q.vec) tad_launch(tad_prod_kernel<true, G, B, true, false>, TAD_PROD_ARGS); else tad_launch(tad_prod_kernel<false, G, B, true, false>, TAD_PROD_ARGS); } \
        else { if (Q.vec) tad_launch(tad_prod_kernel<true, G, B, false, false>, TAD_PROD_ARGS); else tad_launch(tad_prod_kernel<false, G, B, false, false>, TAD_PROD_ARGS); } \
        break;
#define TAD_PROD_LAUNCH_ONE(G) case G: tad_launch(tad_prod_kernel<true, G, 0, true, true>, TAD_PROD_ARGS); break;
        if (Q.run == 1) {                                      // (nothing moves but in a single row that is read in pieces)
            if (Q.row_var >= 0 && Q.vec) tad_launch(tad_prod_kernel<true, 0, 0, false, true>, TAD_PROD_ARGS);
            else if (Q.row_var >= 0) tad_launch(tad_prod_kernel<false, 0, 0, false, true>, TAD_PROD_ARGS);
            else if (!Q.vec) tad_launch(tad_prod_kernel<false, 0, 0, true, true>, TAD_PROD_ARGS);
            else switch (Q.n_moving) {
            TAD_PROD_LAUNCH_ONE(0) TAD_PROD_LAUNCH_ONE(1) TAD_PROD_LAUNCH_ONE(2) TAD_PROD_LAUNCH_ONE(3)
            default: return cudaErrorInvalidValue;
            }
        } else switch (4 * (Q.n_moving - Q.n_single) + Q.n_single) {
        TAD_PROD_LAUNCH(0, 0) TAD_PROD_LAUNCH(0, 1) TAD_PROD_LAUNCH(0, 2) TAD_PROD_LAUNCH(0, 3) TAD_PROD_LAUNCH(1, 0) TAD_PROD_LAUNCH(1, 1)
        TAD_PROD_LAUNCH(1, 2) TAD_PROD_LAUNCH(2, 0) TAD_PROD_LAUNCH(2, 1) TAD_PROD_LAUNCH(3, 0)
        default: return cudaErrorInvalidValue;
        }
#undef TAD_PROD_LAUNCH_ONE
#undef TAD_PROD_LAUNCH
#undef TAD_PROD_ARGS
        return cudaGetLastError();
    }
    unsigned cols = 1;
    while (cols < 256u && cols * 4u * EG < lane_ext) cols *= 2u;
    const unsigned rows_per_block = 256u / cols;
    const unsigned lane_blocks = (lane_ext + cols * 4u * EG - 1u) / (cols * 4u * EG);
    const unsigned long long row_blocks = (rows + rows_per_block - 1) / rows_per_block;
    const unsigned long long items = row_blocks * lane_blocks;
    if (items >= (1ull << 32) || rows >= (1ull << 31)) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)std::min<unsigned long long>(items, (unsigned long long)sms * 16ull);
    tad_launch(tad_ew_kernel, grid, 256, 0, stream, P, ptrs, (unsigned)items, cols, lane_blocks, (unsigned)rows);
    return cudaGetLastError();
}
