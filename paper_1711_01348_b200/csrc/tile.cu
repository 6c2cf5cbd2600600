// Kernel for tile programs (tile.h).
//
// A term as written costs a few multiply-adds per point; what bounded the interpreter on it was fetching: a load and a dispatch
// per value and operation.  Here every operand of a tile is fetched (and evaluated, where it is more than a load) once into
// shared memory, with copies of the next piece of l in flight behind the arithmetic, and the 16 or 32 sums of a thread share two to
// five 128-bit reads per value of l.  Few outputs with long sums are spread over groups of threads that share l (lg) and
// over the eight blocks of a cluster, whose sums meet in shared memory: no planes of partial sums, no second launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "launch.h"
#include "tile.h"
#include "vm.cuh"

namespace {

using tadvm::apply_fn;
using tadvm::fast_sincos;
using tadvm::fast_tanh;

constexpr int NT = TADT_NT, S = TADT_SHARES;

struct Where { int p0, q0, z[TADT_Z]; };         // first values of the tile

__device__ __forceinline__ unsigned line_of(const TadtLoad &L, const Where &w)
{
    unsigned o = (unsigned)L.base;
#pragma unroll
    for (int d = 0; d < TADT_Z; ++d) o += (unsigned)L.cz[d] * (unsigned)w.z[d];
    return o;
}

__device__ __forceinline__ float eval_fn(int fn, float x, int n)
{
    switch (fn) {
    case F_EXP: return __expf(x);
    case F_TANH: return fast_tanh(x);
    case F_SIN: case F_COS: return fabsf(x) < 8192.f ? fast_sincos(x, fn == F_COS) : apply_fn(fn, x, 0);
    default: return apply_fn(fn, x, n);
    }
}

// steps [s0, s0 + n) on R rows from p and C columns from q (values past the edge repeat the last one); sum: the finished sums
template <int R, int C>
__device__ __forceinline__ void run_steps(const TadtProgram &P, const TadpPointers &ptrs, const Where &w, const int s0, const int n,
                                          const int p, const int q, const int l, const float (&sum)[R][C], float (&X)[R][C])
{
    float Y[R][C];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < C; ++j) { X[i][j] = 0.f; Y[i][j] = 0.f; }
#define TAD_T_ALL(expr)                             \
    _Pragma("unroll") for (int i = 0; i < R; ++i)    \
        _Pragma("unroll") for (int j = 0; j < C; ++j) { float &x = X[i][j]; expr; }
    for (int s = s0; s < s0 + n; ++s) {
        const TadeStep st = P.steps[s];
        switch (st.op) {
        case E_LD: {
            float v[R][C];
            if (st.a == TADT_SUM) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int j = 0; j < C; ++j) v[i][j] = sum[i][j];
            } else {
                const TadtLoad &L = P.loads[st.a];
                const float *__restrict__ src = ptrs.in[L.ptr];
                const unsigned o = line_of(L, w) + (unsigned)(L.cl * l);
                const bool wide = C == 4 && L.cq == 1 && q + C <= P.q_ext && ((o + (unsigned)q) & 3u) == 0 && (L.cp & 3) == 0 &&
                                  (reinterpret_cast<uintptr_t>(src) & 15u) == 0;
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const unsigned oi = o + (unsigned)(L.cp * min(p + i, P.p_ext - 1));
                    if (wide) {
                        const float4 f = __ldg(reinterpret_cast<const float4 *>(src + (oi + (unsigned)q)));
                        v[i][0] = f.x; v[i][1 % C] = f.y; v[i][2 % C] = f.z; v[i][3 % C] = f.w;
                    } else {
#pragma unroll
                        for (int j = 0; j < C; ++j) v[i][j] = __ldg(src + (oi + (unsigned)(L.cq * min(q + j, P.q_ext - 1))));
                    }
                }
            }
            if (st.b == 0) TAD_T_ALL(x = v[i][j])
            else if (st.b == 1) TAD_T_ALL(x += v[i][j])
            else if (st.b == 2) TAD_T_ALL(x *= v[i][j])
            else TAD_T_ALL(x += v[i][j]; x *= x)
            break;
        }
        case E_PUSH: TAD_T_ALL(Y[i][j] = x) break;
        case E_CONST: TAD_T_ALL(x = st.imm) break;
        case E_NEG: TAD_T_ALL(x = -x) break;
        case E_SQR: TAD_T_ALL(x *= x) break;
        case E_CUBE: TAD_T_ALL(x = x * x * x) break;
        case E_MULC: TAD_T_ALL(x *= st.imm) break;
        case E_ADDC: TAD_T_ALL(x += st.imm) break;
        case E_ADDY: TAD_T_ALL(x = Y[i][j] + x) break;
        case E_SUBY: TAD_T_ALL(x = Y[i][j] - x) break;
        case E_MULY: TAD_T_ALL(x = Y[i][j] * x) break;
        case E_DIVY: TAD_T_ALL(x = Y[i][j] / x) break;
        case E_FN:
            if (st.b == F_EXP) TAD_T_ALL(x = __expf(x))
            else TAD_T_ALL(x = eval_fn(st.b, x, st.a))
            break;
        default: break;
        }
    }
#undef TAD_T_ALL
}

template <int V>
__device__ __forceinline__ void copy_async(unsigned dst, const float *src)
{
    if constexpr (V == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst), "l"(src) : "memory");
}

// operand o for values [l0, l0 + nl) of l and `width` values from `first` of p (rows) or q into dst[l * pitch + value]
__device__ __forceinline__ void stage(const TadtProgram &P, const TadpPointers &ptrs, const Where &w, const TadtOperand &o, const bool row,
                                      const int width, const int pitch, const int first, const int l0, const int nl, float *dst)
{
    const int last = (row ? P.p_ext : P.q_ext) - 1, tid = (int)threadIdx.x;
    const TadtLoad &L = P.loads[o.load0];
    const int cv = row ? L.cp : L.cq, cl = L.cl;
    const float *__restrict__ src = ptrs.in[L.ptr] + line_of(L, w);
    src += (long long)cl * l0;
    const bool plain = !o.n_steps && o.load1 < 0 && o.e == 1 && o.c == 1.f;
    const unsigned to0 = (unsigned)__cvta_generic_to_shared(dst);
    if (plain && o.along_l) {
        // eight values of l by 32 of p or q at a time: 32-byte pieces of memory, no two threads of a warp in one bank
        const int l = tid & 7, v = tid >> 3;
        for (int u = v; u < width; u += NT / 8) {
            const float *from = src + (cv * min(first + u, last) + cl * l);
            unsigned to = to0 + 4u * (unsigned)(l * pitch + u);
#pragma unroll 4
            for (int m = l; m < nl; m += 8) { copy_async<1>(to, from); from += 8 * cl; to += 32u * (unsigned)pitch; }
        }
        return;
    }
    // neighbouring threads take neighbouring values, whole pieces of 16 bytes where they are aligned
    const bool wide = plain && cv == 1 && (cl & 3) == 0 && first + width - 1 <= last && (reinterpret_cast<uintptr_t>(src + first) & 15u) == 0;
    const int units = wide ? width / 4 : width, vw = units <= 8 ? 3 : units <= 16 ? 4 : units <= 32 ? 5 : units <= 64 ? 6 : 7;
    const int v = tid & ((1 << vw) - 1), dl = NT >> vw;
    if (v >= units) return;
    if (plain) {
        int l = tid >> vw;
        const float *from = src + ((wide ? first + 4 * v : cv * min(first + v, last)) + cl * l);
        unsigned to = to0 + 4u * (unsigned)(l * pitch + (wide ? 4 * v : v));
        if (wide) { for (; l < nl; l += dl) { copy_async<4>(to, from); from += dl * cl; to += 4u * (unsigned)(dl * pitch); } }
        else { for (; l < nl; l += dl) { copy_async<1>(to, from); from += dl * cl; to += 4u * (unsigned)(dl * pitch); } }
        return;
    }
    const int at = min(first + v, last);
    if (o.n_steps) {
        for (int l = tid >> vw; l < nl; l += dl) {
            const float none[1][1] = {{0.f}};
            float x[1][1];
            run_steps<1, 1>(P, ptrs, w, o.step0, o.n_steps, row ? at : 0, row ? 0 : at, l0 + l, none, x);
            dst[l * pitch + v] = x[0][0];
        }
        return;
    }
    const bool pair = o.load1 >= 0;
    const TadtLoad &M = P.loads[pair ? o.load1 : o.load0];
    const float *from1 = ptrs.in[M.ptr] + line_of(M, w) + (long long)M.cl * l0 + (row ? M.cp : M.cq) * at, *from = src + cv * at;
    const int e = o.e, ml = M.cl;
    const float c = o.c;
#pragma unroll 4
    for (int l = tid >> vw; l < nl; l += dl) {
        const float x = __ldg(from + cl * l), y = pair ? __ldg(from1 + ml * l) : 1.f;
        dst[l * pitch + v] = (e == 1 ? x : e == 2 ? x * x : x * x * x) * c * y;
    }
}

// the core read step by step, for one value of l
__device__ __forceinline__ void run_core(const TadtProgram &P, const float *const (&at)[TADT_OPS], const int (&step)[TADT_OPS], const int l, const float (&mat)[4][4], float (&sum)[4][4])
{
    float X[4][4], Y[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { X[i][j] = 0.f; Y[i][j] = 0.f; }
    auto fetch = [&](int o, float (&v)[4][4]) {
        const int kind = P.op[o].kind;
        if (kind == TK_MAT) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[i][j] = mat[i][j];
            return;
        }
        const float *b = nullptr;
#pragma unroll
        for (int k = 0; k < TADT_OPS; ++k) if (k == o) b = at[k] + l * step[k];
        const float4 f = *reinterpret_cast<const float4 *>(b);
        const float e[4] = {f.x, f.y, f.z, f.w};
        const bool row = kind == TK_ROW || kind == TK_ROWC;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[i][j] = row ? e[i] : e[j];
    };
#define TAD_T_ALL(expr)                             \
    _Pragma("unroll") for (int i = 0; i < 4; ++i)    \
        _Pragma("unroll") for (int j = 0; j < 4; ++j) { float &x = X[i][j]; expr; }
    for (uint64_t code = P.core; code; code >>= 8) {
        const int op = (int)code & 15, o = ((int)code >> 4) & 3, o2 = ((int)code >> 6) & 3;
        switch (op) {
        case T_LD: case T_ADD: case T_SUB: case T_RSUB: case T_MUL: case T_FMA: {
            float v[4][4];
            fetch(o, v);
            if (op == T_LD) TAD_T_ALL(x = v[i][j])
            else if (op == T_ADD) TAD_T_ALL(x += v[i][j])
            else if (op == T_SUB) TAD_T_ALL(x -= v[i][j])
            else if (op == T_RSUB) TAD_T_ALL(x = v[i][j] - x)
            else if (op == T_MUL) TAD_T_ALL(x *= v[i][j])
            else {
                float u[4][4];
                fetch(o2, u);
                TAD_T_ALL(x = fmaf(x, v[i][j], u[i][j]))
            }
            break;
        }
        case T_SQR: TAD_T_ALL(x *= x) break;
        case T_CUBE: TAD_T_ALL(x = x * x * x) break;
        case T_NEG: TAD_T_ALL(x = -x) break;
        case T_MULC: { const float c = P.imm[o]; TAD_T_ALL(x *= c) } break;
        case T_ADDC: { const float c = P.imm[o]; TAD_T_ALL(x += c) } break;
        case T_PUSH: TAD_T_ALL(Y[i][j] = x) break;
        case T_BINY:
            if (o == 0) TAD_T_ALL(x = Y[i][j] + x)
            else if (o == 1) TAD_T_ALL(x = Y[i][j] - x)
            else if (o == 2) TAD_T_ALL(x = Y[i][j] * x)
            else TAD_T_ALL(x = Y[i][j] / x)
            break;
        case T_FN: TAD_T_ALL(x = eval_fn(o | o2 << 2, x, 0)) break;
        case T_ACC:
            if (o2 == 0) TAD_T_ALL(sum[i][j] += x)
            else {
                float v[4][4];
                fetch(o, v);
                TAD_T_ALL(sum[i][j] = fmaf(x, v[i][j], sum[i][j]))
            }
            break;
        default: break;
        }
    }
#undef TAD_T_ALL
}

template <int N>
__device__ __forceinline__ void values_of(const float *p, float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4) { const float4 f = *reinterpret_cast<const float4 *>(p + i); v[i] = f.x; v[i + 1] = f.y; v[i + 2] = f.z; v[i + 3] = f.w; }
}

// values l = lg, lg + groups, ... < nl of the staged piece
template <int TM, int PATH>
__device__ __forceinline__ void run_piece(const TadtProgram &P, const float *const (&at)[TADT_OPS], const int (&step)[TADT_OPS], const int lg,
                                          const int groups, const int nl, const float (&mat)[TM][4], float (&sum)[TM][4])
{
#define TAD_T_ALL(expr)                             \
    _Pragma("unroll") for (int i = 0; i < TM; ++i)   \
        _Pragma("unroll") for (int j = 0; j < 4; ++j) { expr; }
    if constexpr (PATH == 0) {
        for (int l = lg; l < nl; l += groups) run_core(P, at, step, l, mat, sum);
    } else {
        const int rstep = step[PATH == 3 ? 2 : 0], cstep = step[1];
        const float *rp = at[PATH == 3 ? 2 : 0] + lg * rstep, *cp = at[1] + lg * cstep, *dp = at[3] + lg * rstep;
        float k[TM];
        if constexpr (PATH == 2) values_of<TM>(at[2], k);
#pragma unroll 2
        for (int l = lg; l < nl; l += groups) {
            float r[TM], c[4];
            values_of<TM>(rp, r); values_of<4>(cp, c);
            rp += groups * rstep; cp += groups * cstep;
            if constexpr (PATH == 1) {
                TAD_T_ALL(const float s = r[i] + c[j]; sum[i][j] = fmaf(s, s, sum[i][j]))
            } else if constexpr (PATH == 2) {
                float d[TM];
                values_of<TM>(dp, d);
                dp += groups * rstep;
                TAD_T_ALL(const float s = r[i] + c[j]; sum[i][j] += fmaf(s * s, k[i], d[i]))
            } else {
                TAD_T_ALL(sum[i][j] = fmaf(mat[i][j] + c[j], r[i], sum[i][j]))
            }
        }
    }
#undef TAD_T_ALL
}

// steps [s0, s0 + n) on a thread's TM rows, four at a time
template <int TM>
__device__ __forceinline__ void matrix_of(const TadtProgram &P, const TadpPointers &ptrs, const Where &w, const int s0, const int n, const int p, const int q,
                                          float (&X)[TM][4])
{
#pragma unroll
    for (int h = 0; h < TM; h += 4) {
        const float none[4][4] = {};
        float x[4][4];
        run_steps<4, 4>(P, ptrs, w, s0, n, p + h, q, 0, none, x);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) X[h + i][j] = x[i][j];
    }
}

// from the sums of four rows from p and four columns from q (one where q is summed) to the outputs
__device__ __forceinline__ void finish(const TadtProgram &P, const TadpPointers &ptrs, const Where &w, float *__restrict__ out, const int p, const int q,
                                       const float (&sum)[4][4])
{
    if (p >= P.p_ext || q >= P.q_ext) return;
    float X[4][4];
    run_steps<4, 4>(P, ptrs, w, P.epi0, P.n_epi, p, q, 0, sum, X);
    unsigned o = (unsigned)P.out_base + (unsigned)(P.out_cq * q);
#pragma unroll
    for (int d = 0; d < TADT_Z; ++d) o += (unsigned)P.out_cz[d] * (unsigned)w.z[d];
    const int cols = P.q_sum ? 1 : min(4, P.q_ext - q);
    const bool wide = cols == 4 && P.out_cq == 1 && !P.accumulate && (o & 3u) == 0 && (P.out_cp & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (p + i >= P.p_ext) break;
        float *at = out + (o + (unsigned)(P.out_cp * (p + i)));
        if (wide) *reinterpret_cast<float4 *>(at) = make_float4(X[i][0], X[i][1], X[i][2], X[i][3]);
        else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (j < cols) { float *e = at + P.out_cq * j; *e = P.accumulate ? *e + X[i][j] : X[i][j]; }
        }
    }
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ float peer_value(const float *p, unsigned rank)
{
    unsigned a;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

template <int TM, int PATH, bool QS>
__device__ __forceinline__ void run_block(const TadtProgram &P, const TadpPointers &ptrs, float *out, float *sm, const unsigned bx)
{
    const unsigned rank = P.shares > 1 ? bx % (unsigned)S : 0u, t = P.shares > 1 ? bx / (unsigned)S : bx;
    if (t >= (unsigned)P.n_blocks) return;
    const int ct_n = P.ct, rt_n = P.rt, tid = (int)threadIdx.x;
    const int row = (int)(((unsigned)tid * P.ct_mul) >> 16), ct = tid - row * ct_n, lg = (int)(((unsigned)row * P.rt_mul) >> 16), rt = row - lg * rt_n;
    const bool idle = lg >= P.lg;
    const int bm = TM * rt_n, bn = 4 * ct_n;
    Where w;
    {
        unsigned rest = t, tq = 0;
        if (!QS) { rest = t / (unsigned)P.tiles_q; tq = t - rest * (unsigned)P.tiles_q; }
        unsigned next = rest / (unsigned)P.tiles_p;
        w.p0 = (int)(rest - next * (unsigned)P.tiles_p) * bm;
        w.q0 = (QS ? (int)rank : (int)tq) * bn;
        w.z[0] = (int)next; w.z[1] = 0;
        if (P.z_ext[1] > 1) { w.z[0] = (int)(next / (unsigned)P.z_ext[1]); w.z[1] = (int)next - w.z[0] * P.z_ext[1]; }
    }
    // the block's share of l, or (q summed) of the tiles of q
    int l_begin = 0, l_end = P.l_ext;
    if (P.shares > 1 && !QS) {
        const int per = (P.l_ext + S - 1) / S;
        l_begin = min(P.l_ext, (int)rank * per); l_end = min(P.l_ext, l_begin + per);
    }
    // shared memory: pieces of the rows' and columns' operands, then the operands that do not vary along l
    const int chunk = P.chunk, pm = bm + 4, pn = bn + 4, piece = chunk * (P.n_rows * pm + P.n_cols * pn);
    const bool rows_stay = QS && chunk >= l_end - l_begin;                // the rows of a tile are the rows of the next
    const float *at[TADT_OPS];
    int step[TADT_OPS], off[TADT_OPS];
    {
        int next_row = 0, next_col = chunk * P.n_rows * pm, held = P.buffers * piece;
#pragma unroll
        for (int o = 0; o < TADT_OPS; ++o) {
            off[o] = 0; step[o] = 0; at[o] = sm;
            if (o >= P.n_ops) continue;
            switch (P.op[o].kind) {
            case TK_ROW: off[o] = next_row; next_row += chunk * pm; step[o] = pm; at[o] = sm + off[o] + TM * rt; break;
            case TK_COL: off[o] = next_col; next_col += chunk * pn; step[o] = pn; at[o] = sm + off[o] + 4 * ct; break;
            case TK_ROWC: off[o] = held; held += bm; at[o] = sm + off[o] + TM * rt; break;
            case TK_COLC: off[o] = held; held += bn; at[o] = sm + off[o] + 4 * ct; break;
            default: break;
            }
        }
    }
    float sum[TM][4], mat[TM][4], total[QS ? TM : 1];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        if constexpr (QS) total[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) { sum[i][j] = 0.f; mat[i][j] = 0.f; }
    }
    const int p = w.p0 + TM * rt;
    // pieces of l, and (q summed) tiles of q; the next piece is on its way while one is worked on (the first turn only stages)
    int l_next = l_begin, l_now = l_begin, buf = 0;
    bool more = l_begin < l_end && (!QS || w.q0 < P.q_ext);
    for (bool first = true, now = false; more || now; first = false) {
        const int q0 = w.q0;
        if (!first) {
            l_now = l_next;
            l_next += chunk;
            if (l_next >= l_end) { l_next = l_begin; more = false; if (QS) { w.q0 += (int)P.shares * bn; more = w.q0 < P.q_ext; } }
        }
        if (more) {
            const int nl = min(chunk, l_end - l_next), to = first ? 0 : buf ^ 1;
#pragma unroll 1
            for (int o = 0; o < P.n_ops; ++o) {
                const int kind = P.op[o].kind;
                const bool held = kind == TK_ROWC || kind == TK_COLC, rows = kind == TK_ROW || kind == TK_ROWC;
                if (kind == TK_MAT || (!first && (held || (rows && rows_stay)))) continue;
                int a = 0;
#pragma unroll
                for (int k = 0; k < TADT_OPS; ++k) if (k == o) a = off[k];
                stage(P, ptrs, w, P.op[o], rows, rows ? bm : bn, rows ? pm : pn, rows ? w.p0 : w.q0, held ? 0 : l_next, held ? 1 : nl,
                      sm + a + (held ? 0 : to * piece));
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        now = true;
        if (first) continue;
        const int q = q0 + 4 * ct;
        if constexpr (PATH == 0 || PATH == 3) {
            if (l_now == l_begin)
#pragma unroll 1
                for (int o = 0; o < P.n_ops; ++o)
                    if (P.op[o].kind == TK_MAT) matrix_of<TM>(P, ptrs, w, P.op[o].step0, P.op[o].n_steps, p, q, mat);
        }
        if (more) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (!idle) run_piece<TM, PATH>(P, at, step, lg, P.lg, min(chunk, l_end - l_now), mat, sum);
        if constexpr (QS) {
            if (l_next == l_begin) {
                if (P.n_post) {
                    float f[TM][4];
                    matrix_of<TM>(P, ptrs, w, P.post0, P.n_post, p, q, f);
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) sum[i][j] *= f[i][j];
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    float v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) { v[j] = q + j < P.q_ext ? sum[i][j] : 0.f; sum[i][j] = 0.f; }
                    total[i] += (v[0] + v[1]) + (v[2] + v[3]);
                }
            }
        }
        __syncthreads();
        if (more) {
            const int turn = buf ? -piece : piece;
#pragma unroll
            for (int k = 0; k < TADT_OPS; ++k)
                if (k < P.n_ops && (P.op[k].kind == TK_COL || (P.op[k].kind == TK_ROW && !rows_stay))) at[k] += turn;
            buf ^= 1;
        }
        now = more;
    }
    // sums of the groups, then of the blocks, in a fixed order; shared memory is free: the last piece has been read
    const int width = QS ? 1 : bn, groups = QS ? P.lg * ct_n : P.lg, cells = bm * width, group = QS ? lg * ct_n + ct : lg;
    if (!idle) {
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            float *cell = sm + group * cells + (TM * rt + i) * width;
            if constexpr (QS) *cell = total[i];
            else *reinterpret_cast<float4 *>(cell + 4 * ct) = make_float4(sum[i][0], sum[i][1], sum[i][2], sum[i][3]);
        }
    }
    __syncthreads();
    if (groups > 1) {
        for (int c = tid; c < cells; c += NT) {
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            int g = 0;
            for (; g + 4 <= groups; g += 4)
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] += sm[(g + u) * cells + c];
            for (; g < groups; ++g) v[0] += sm[g * cells + c];
            sm[c] = (v[0] + v[1]) + (v[2] + v[3]);
        }
        if (P.shares == 1) __syncthreads();
    }
    if (P.shares > 1) cluster_sync();
    const int per_row = QS ? 1 : ct_n, items = bm / 4 * per_row;
#pragma unroll 1
    for (int it = tid + (int)rank * NT; it < items; it += NT * P.shares) {
        const int r = QS ? it : it / ct_n, c = it - r * per_row;
        float v[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float *cell = sm + (4 * r + i) * width + (QS ? 0 : 4 * c);
            if (P.shares > 1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[i][j] = 0.f;
                    if (QS && j > 0) continue;
                    float u[S];
#pragma unroll
                    for (int b = 0; b < S; ++b) u[b] = peer_value(cell + j, (unsigned)b);
                    v[i][j] = ((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + (u[6] + u[7]));
                }
            } else if (QS) { v[i][0] = *cell; v[i][1] = v[i][2] = v[i][3] = 0.f; }
            else { const float4 f = *reinterpret_cast<const float4 *>(cell); v[i][0] = f.x; v[i][1] = f.y; v[i][2] = f.z; v[i][3] = f.w; }
        }
        finish(P, ptrs, w, out, w.p0 + 4 * r, QS ? 0 : w.q0 + 4 * c, v);
    }
    if (P.shares > 1) cluster_sync();             // (a block's sums stay until every other one has read them)
}

// KIND: the core's build and whether q is summed (2 path + q_sum), or -1: any (several programs in a launch)
template <int N, int KIND, int TM>
__global__ void __launch_bounds__(NT, 2)
tad_tile_kernel(const __grid_constant__ TadtBatch<N> B, const __grid_constant__ TadpPointers ptrs)
{
    extern __shared__ __align__(16) float sm[];
    if constexpr (KIND >= 0) {
        tad_wait_previous();
        run_block<TM, KIND / 2, KIND % 2 != 0>(B.p[0], ptrs, B.out[0], sm, blockIdx.x);
    } else {
        int i = 0;
        while (i + 1 < B.n && blockIdx.x >= B.first[i + 1]) ++i;
        const TadtProgram &P = B.p[i];
        tad_wait_previous();
        const unsigned bx = blockIdx.x - B.first[i];
        switch (2 * P.path + P.q_sum) {
        case 2: run_block<TM, 1, false>(P, ptrs, B.out[i], sm, bx); break;
        case 3: run_block<TM, 1, true>(P, ptrs, B.out[i], sm, bx); break;
        case 4: run_block<TM, 2, false>(P, ptrs, B.out[i], sm, bx); break;
        case 6: run_block<TM, 3, false>(P, ptrs, B.out[i], sm, bx); break;
        case 1: if constexpr (TM == 4) run_block<4, 0, true>(P, ptrs, B.out[i], sm, bx); break;
        default: if constexpr (TM == 4) run_block<4, 0, false>(P, ptrs, B.out[i], sm, bx); break;
        }
    }
}

template <int N, int KIND, int TM>
cudaError_t launch(const TadtProgram *const *progs, float *const *out, int n, const TadpPointers &ptrs, cudaStream_t stream)
{
    TadtBatch<N> B;
    B.n = n;
    size_t smem = 0;
    bool shared = false;
    for (int i = 0; i < n; ++i) shared = shared || progs[i]->shares > 1;
    B.first[0] = 0;
    for (int i = 0; i < N; ++i) {
        const TadtProgram &P = *progs[std::min(i, n - 1)];
        B.p[i] = P; B.out[i] = out[std::min(i, n - 1)];
        unsigned blocks = i < n ? (unsigned)P.n_blocks * (unsigned)P.shares : 0u;
        if (shared) blocks = (blocks + S - 1) / S * S;
        B.first[i + 1] = B.first[i] + blocks;
        smem = std::max(smem, (size_t)P.smem);
    }
    auto kernel = tad_tile_kernel<N, KIND, TM>;
    if (smem > 48 * 1024) {
        static std::atomic<bool> allowed[64];
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        std::atomic<bool> *known = dev >= 0 && dev < 64 ? &allowed[dev] : nullptr;
        if (!known || !known->load(std::memory_order_relaxed)) {
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TADT_SMEM);
            if (e != cudaSuccess) return e;
            if (known) known->store(true, std::memory_order_relaxed);
        }
    }
    return tad_launch_cluster(kernel, B.first[n], NT, smem, stream, shared ? S : 1, B, ptrs);
}

}  // namespace

// programs of one launch: not more than TADT_BATCH, all of one tm, none reads what another writes
cudaError_t tad_launch_tiles(const TadtProgram *const *progs, float *const *out, int n, const TadpPointers &ptrs, cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    if (n > 1) return progs[0]->tm == 8 ? launch<TADT_BATCH, -1, 8>(progs, out, n, ptrs, stream) : launch<TADT_BATCH, -1, 4>(progs, out, n, ptrs, stream);
    const bool tall = progs[0]->tm == 8;
    switch (2 * progs[0]->path + progs[0]->q_sum) {
    case 2: return tall ? launch<1, 2, 8>(progs, out, n, ptrs, stream) : launch<1, 2, 4>(progs, out, n, ptrs, stream);
    case 3: return tall ? launch<1, 3, 8>(progs, out, n, ptrs, stream) : launch<1, 3, 4>(progs, out, n, ptrs, stream);
    case 4: return tall ? launch<1, 4, 8>(progs, out, n, ptrs, stream) : launch<1, 4, 4>(progs, out, n, ptrs, stream);
    case 6: return tall ? launch<1, 6, 8>(progs, out, n, ptrs, stream) : launch<1, 6, 4>(progs, out, n, ptrs, stream);
    case 1: return launch<1, 1, 4>(progs, out, n, ptrs, stream);
    default: return launch<1, 0, 4>(progs, out, n, ptrs, stream);
    }
}
