// Kernel for point programs (point.h).
//
// What bounds small kernels on the interpreter (vm.cuh) is its code: handlers are built per stack depth and vector
// shape, and a launch of a few blocks waits for instruction fetches most of the time (ncu: 5 to 15 of 11 to 22 stall
// cycles per issued instruction are "no instruction"), on one value per thread and one serial load after another.
// Here there is one handler per operation (the stack lives in shared memory), one or four points per thread, and the
// terms of an output are spread over as many lanes of a block as it takes to fill the GPU.
#include <cuda_runtime.h>

#include <algorithm>

#include "launch.h"
#include "point.h"
#include "vm.cuh"

namespace {

using tadvm::apply_fn;
using tadvm::fast_sincos;
using tadvm::fast_tanh;

constexpr int NT = 256, MV = TADQ_MAX_VARS, MS = TADQ_MAX_SUMS;

template <int U>
struct Vals { float v[U]; };

template <int U>
__device__ __forceinline__ Vals<U> slot_get(const float *sm, int s)
{
    Vals<U> r;
    const float *p = sm + (s * NT + (int)threadIdx.x) * U;
    if constexpr (U == 4) { const float4 q = *reinterpret_cast<const float4 *>(p); r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w; }
    else r.v[0] = *p;
    return r;
}
template <int U>
__device__ __forceinline__ void slot_put(float *sm, int s, const Vals<U> &x)
{
    float *p = sm + (s * NT + (int)threadIdx.x) * U;
    if constexpr (U == 4) *reinterpret_cast<float4 *>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
    else *p = x.v[0];
}

// steps [pc, end) for the points in var; every index is inside its tensor for every value the variables can take
template <int U>
__device__ __forceinline__ void run_steps(const TadqProgram &P, const TadpPointers &ptrs, float *sm, int pc, const int end,
                                          const int (&var)[MV][U], const unsigned live, Vals<U> &X, Vals<U> &acc)
{
    int k[MS] = {0, 0, 0, 0};
#define TAD_Q_ALL(expr) _Pragma("unroll") for (int u = 0; u < U; ++u) { float &x = X.v[u]; expr; }
    while (pc < end) {
        const TadqStep st = P.steps[pc];
        ++pc;
        switch (st.op) {
        case Q_CONST: case Q_SLOT: case Q_LOAD: case Q_LDADD: case Q_LDMUL: case Q_LDADDSQ: {
            Vals<U> v;
            if (st.op == Q_CONST) { const float c = __int_as_float(st.imm); _Pragma("unroll") for (int u = 0; u < U; ++u) v.v[u] = c; }
            else if (st.op == Q_SLOT) v = slot_get<U>(sm, st.a);
            else {
                const TadqLoad &L = P.loads[st.a];
                int base = L.base;
#pragma unroll
                for (int s = 0; s < MS; ++s) if (s < P.n_sums) base += L.scoef[s] * k[s];
                const float *__restrict__ src = ptrs.in[L.ptr];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    int o = base;
#pragma unroll
                    for (int d = 0; d < MV; ++d) o += L.coef[d] * var[d][u];
                    v.v[u] = __ldg(src + (unsigned)o);
                }
            }
            if (st.op == Q_LDADD) { TAD_Q_ALL(x += v.v[u]) }
            else if (st.op == Q_LDMUL) { TAD_Q_ALL(x *= v.v[u]) }
            else if (st.op == Q_LDADDSQ) { TAD_Q_ALL(x += v.v[u]; x *= x) }
            else { if (st.s != TADQ_NONE) slot_put<U>(sm, st.s, X); X = v; }
            break;
        }
        case Q_NEG: TAD_Q_ALL(x = -x) break;
        case Q_SQR: TAD_Q_ALL(x *= x) break;
        case Q_CUBE: TAD_Q_ALL(x = x * x * x) break;
        case Q_MULC: { const float c = __int_as_float(st.imm); TAD_Q_ALL(x *= c) } break;
        case Q_ADDC: { const float c = __int_as_float(st.imm); TAD_Q_ALL(x += c) } break;
        case Q_FN:
            switch (st.b) {
            case F_EXP: TAD_Q_ALL(x = __expf(x)) break;
            case F_TANH: TAD_Q_ALL(x = fast_tanh(x)) break;
            case F_SIN: case F_COS: TAD_Q_ALL(x = fabsf(x) < 8192.f ? fast_sincos(x, st.b == F_COS) : apply_fn(st.b, x, 0)) break;
            default: TAD_Q_ALL(x = apply_fn(st.b, x, st.imm)) break;
            }
            break;
        case Q_ADD: { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(x = y.v[u] + x) } break;
        case Q_SUB: { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(x = y.v[u] - x) } break;
        case Q_MUL: { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(x = y.v[u] * x) } break;
        case Q_DIV: { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(x = y.v[u] / x) } break;
        case Q_FMA: { const Vals<U> y = slot_get<U>(sm, st.s), z = slot_get<U>(sm, st.a); TAD_Q_ALL(x = fmaf(y.v[u], z.v[u], x)) } break;
        case Q_STORE: slot_put<U>(sm, st.a, X); if (st.s != TADQ_NONE) X = slot_get<U>(sm, st.s); break;
        case Q_ACC: TAD_Q_ALL(if (live & (1u << u)) acc.v[u] += x) break;
        case Q_MACC: { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(if (live & (1u << u)) acc.v[u] = fmaf(y.v[u], x, acc.v[u])) } break;
        case Q_SCALE: TAD_Q_ALL(acc.v[u] *= x) break;
        case Q_LOOP: {
            const int lo = P.s_lo[st.a];
#pragma unroll
            for (int s = 0; s < MS; ++s) if (s == st.a) k[s] = lo;
            if (lo > P.s_hi[st.a]) pc = st.imm;
            break;
        }
        case Q_SUMNEXT: case Q_NEXT: {
            if (st.op == Q_SUMNEXT) { const Vals<U> y = slot_get<U>(sm, st.s); TAD_Q_ALL(x = y.v[u] + x) }
            int n = 0;
#pragma unroll
            for (int s = 0; s < MS; ++s) if (s == st.a) n = ++k[s];
            if (n <= P.s_hi[st.a]) pc = st.imm;
            break;
        }
        default: break;
        }
    }
#undef TAD_Q_ALL
}

// variables [first, first + n) of point u from a flattened index, last one fastest
template <int U>
__device__ __forceinline__ void decode(const TadqProgram &P, const int first, const int n, unsigned idx, int (&var)[MV][U], const int u)
{
#pragma unroll
    for (int d = MV - 1; d >= 0; --d) {
        if (d < first || d >= first + n) continue;
        const unsigned q = (unsigned)(((unsigned long long)idx * P.div_mul[d]) >> P.div_shift[d]);
        var[d][u] = P.lo[d] + (int)(idx - q * (unsigned)P.ext[d]);
        idx = q;
    }
}

// block bx of the program; its share number by of n_shares
template <int U>
__device__ __forceinline__ void run_block(const TadqProgram &P, const TadpPointers &ptrs, float *out, float *sm, const unsigned bx, const unsigned by, const unsigned n_shares)
{
    const int tid = (int)threadIdx.x;
    int var[MV][U];
#pragma unroll
    for (int d = 0; d < MV; ++d)
#pragma unroll
        for (int u = 0; u < U; ++u) var[d][u] = 0;
    Vals<U> X, acc;
#pragma unroll
    for (int u = 0; u < U; ++u) { X.v[u] = 0.f; acc.v[u] = 0.f; }
    const unsigned points = (unsigned)P.points, terms = (unsigned)P.terms;
    // Without terms a thread owns U outputs, a block's width apart.  With terms a block owns 256 / lt outputs, lt threads
    // each, and a thread walks every (lt)-th term of its block's share, U at a time.
    const bool sums = terms > 1 || P.lt > 1;
    const unsigned lt = (unsigned)P.lt, lo_n = NT / lt;
    const unsigned tl = P.along_terms ? tid % lt : tid / lo_n, ol = P.along_terms ? tid / lt : tid % lo_n;
    const unsigned per = (terms + n_shares - 1u) / n_shares, t0 = by * per, t1 = min(terms, t0 + per);
    // fixed-order tree over the term lanes of an output
    float *red = sm + P.n_slots * NT * U;
    auto total = [&]() {
        float sum = acc.v[0];
#pragma unroll
        for (int u = 1; u < U; ++u) sum += acc.v[u];
        red[ol * lt + tl] = sum;
        __syncthreads();
        for (unsigned h = lt / 2; h >= 1; h /= 2) {
            if (tl < h) red[ol * lt + tl] += red[ol * lt + tl + h];
            __syncthreads();
        }
    };
    unsigned live = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const unsigned q = sums ? bx * lo_n + ol : (bx * U + u) * NT + tid;
        if (q < points) live |= 1u << u;
        decode<U>(P, 0, P.n_out, min(q, points - 1u), var, u);
        decode<U>(P, P.n_out, P.n_z, 0u, var, u);
    }
    // steps once per output, steps per batch of terms, steps on the sum (the factor outside it: it scales every partial
    // sum); one call site, so that the handlers exist once
    for (unsigned t = t0, phase = 0; phase < 3u;) {
        int pc = 0, end = P.n_steps;
        unsigned mask = live;
        if (!sums) phase = 3u;
        else if (phase == 0u) { end = P.body; phase = 1u; }
        else if (t < t1) {
            mask = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned q = t + u * lt + tl;
                if (q < t1) mask |= 1u << u;
                decode<U>(P, P.n_out, P.n_z, min(q, terms - 1u), var, u);
            }
            pc = P.body; end = P.tail;
            t += lt * U;
        } else {
            pc = P.tail; phase = 3u;
            if (P.value_slot >= 0) {
                // the sum of the output, known to all of its lanes, is a value of the tail
                total();
                Vals<U> s;
#pragma unroll
                for (int u = 0; u < U; ++u) { s.v[u] = red[ol * lt]; acc.v[u] = 0.f; }
                slot_put<U>(sm, P.value_slot, s);
                mask = live;
            }
        }
        run_steps<U>(P, ptrs, sm, pc, end, var, mask, X, acc);
    }
    if (!sums) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            int o = P.out_base;
#pragma unroll
            for (int d = 0; d < MV; ++d) o += P.out_coef[d] * var[d][u];
            if (live & (1u << u)) out[(unsigned)o] = P.accumulate ? out[(unsigned)o] + acc.v[u] : acc.v[u];
        }
        return;
    }
    if (P.value_slot < 0) total();
    if (tl != 0 || !live) return;
    const float sum = P.value_slot < 0 ? red[ol * lt] : acc.v[0];
    int o = P.out_base; unsigned cell = 0;
#pragma unroll
    for (int d = 0; d < MV; ++d) { o += P.out_coef[d] * var[d][0]; if (d < P.n_out) cell += (unsigned)(P.part_coef[d] * (var[d][0] - P.lo[d])); }
    if (P.zsplit > 1) ptrs.part[(size_t)by * (unsigned)P.part_limit + cell] = sum;
    else out[(unsigned)o] = P.accumulate ? out[(unsigned)o] + sum : sum;
}

template <int U>
__global__ void __launch_bounds__(NT)
tad_point_kernel(const __grid_constant__ TadqProgram P, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    extern __shared__ __align__(16) float sm[];
    run_block<U>(P, ptrs, ptrs.out, sm, blockIdx.x, blockIdx.y, gridDim.y);
}

template <int U>
__global__ void __launch_bounds__(NT)
tad_point_batch_kernel(const __grid_constant__ TadqBatch B, const __grid_constant__ TadpPointers ptrs)
{
    tad_wait_previous();
    extern __shared__ __align__(16) float sm[];
    int i = 0;
    while (i + 1 < B.n && blockIdx.x >= B.first[i + 1]) ++i;
    run_block<U>(B.p[i], ptrs, B.out[i], sm, blockIdx.x - B.first[i], 0u, 1u);
}

template <int U>
unsigned blocks_of(const TadqProgram &P)
{
    const unsigned per = P.terms > 1 || P.lt > 1 ? (unsigned)(NT / P.lt) : (unsigned)NT * U;
    return ((unsigned)P.points + per - 1u) / per;
}

template <int U>
size_t smem_of(const TadqProgram &P) { return ((size_t)P.n_slots * U + 1) * NT * 4; }

template <int U, class K>
cudaError_t allow_smem(K kernel, size_t smem)
{
    if (smem <= 48 * 1024) return cudaSuccess;
    static bool attr_set[64] = {};                             // (one per kernel type: the batch and the single kernel differ in K)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (TADQ_MAX_SLOTS * U + 1) * NT * 4);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    return cudaSuccess;
}

template <int U>
cudaError_t launch_batch(TadqBatch &B, const TadpPointers &ptrs, cudaStream_t stream)
{
    size_t smem = 0;
    B.first[0] = 0;
    for (int i = 0; i < B.n; ++i) { B.first[i + 1] = B.first[i] + blocks_of<U>(B.p[i]); smem = std::max(smem, smem_of<U>(B.p[i])); }
    const cudaError_t e = allow_smem<U>(tad_point_batch_kernel<U>, smem);
    return e != cudaSuccess ? e : tad_launch(tad_point_batch_kernel<U>, B.first[B.n], NT, smem, stream, B, ptrs);
}

template <int U>
cudaError_t launch_points(const TadqProgram &P, const TadpPointers &ptrs, cudaStream_t stream)
{
    const size_t smem = smem_of<U>(P);
    const cudaError_t e = allow_smem<U>(tad_point_kernel<U>, smem);
    return e != cudaSuccess ? e : tad_launch(tad_point_kernel<U>, dim3(blocks_of<U>(P), (unsigned)std::max(1, P.zsplit)), NT, smem, stream, P, ptrs);
}

}  // namespace

cudaError_t tad_launch_points(const TadqProgram &P, const TadpPointers &ptrs, cudaStream_t stream)
{
    if (P.points <= 0) return cudaSuccess;
    return P.unroll == 4 ? launch_points<4>(P, ptrs, stream) : launch_points<1>(P, ptrs, stream);
}

// n programs (at most TADQ_BATCH, none split into shares) that write out[i]
cudaError_t tad_launch_point_batch(const TadqProgram *const *progs, float *const *out, int n, const TadpPointers &ptrs, cudaStream_t stream)
{
    TadqBatch B;
    B.n = n;
    bool four = false;
    for (int i = 0; i < n; ++i) { B.p[i] = *progs[i]; B.out[i] = out[i]; four = four || progs[i]->unroll == 4; }
    for (int i = n; i < TADQ_BATCH; ++i) { B.p[i] = *progs[0]; B.out[i] = nullptr; B.first[i + 1] = 0; }
    return four ? launch_batch<4>(B, ptrs, stream) : launch_batch<1>(B, ptrs, stream);
}
