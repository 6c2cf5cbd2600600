// Device helpers shared by the contraction kernels (contract.cu, mma.cu).
#pragma once
#include <climits>

#include "contract.h"
#include "program.h"

namespace tadc {

constexpr int DEAD = INT_MIN / 2;      // guard part of a row or summation index that does not exist

struct Parts { int a, b, o, ga, gb; };

// digits of a flattened index, last digit fastest, folded into the offset parts of the group
__device__ __forceinline__ Parts decode(const TadcGroup &G, unsigned idx)
{
    Parts p{0, 0, 0, 0, 0};
#pragma unroll
    for (int d = TADC_MAX_DIGITS - 1; d >= 0; --d) {
        if (d < G.n_digits) {
            const unsigned e = (unsigned)G.ext[d];
            const unsigned q = (unsigned)(((unsigned long long)idx * G.div_mul[d]) >> G.div_shift[d]);
            const int r = (int)(idx - q * e);
            idx = q;
            p.a += r * G.sA[d]; p.b += r * G.sB[d]; p.o += r * G.sO[d];
            p.ga += r * G.gA[d]; p.gb += r * G.gB[d];
        }
    }
    return p;
}

__device__ __forceinline__ float own_tanh(float x)
{
    const float ax = fabsf(x);
    const float e = __expf(2.f * ax);
    const float t = 1.f - __fdividef(2.f, e + 1.f);
    const float x2 = x * x;
    const float small = x * (1.f + x2 * (-0.33333334f + x2 * (0.13333334f + x2 * -0.05396825f)));
    return ax < 0.25f ? small : copysignf(t, x);
}

// the steps every finished sum goes through before it is stored
__device__ __forceinline__ float epilogue(const TadcProgram &P, const TadpPointers &ptrs, float v, unsigned off)
{
    for (int s = 0; s < P.n_epi; ++s) {
        switch (P.epi_op[s]) {
        case TE_NEG: v = -v; break;
        case TE_EXP: v = __expf(v); break;
        case TE_MULC: v *= P.epi_imm[s]; break;
        case TE_ADDC: v += P.epi_imm[s]; break;
        case TE_SQR: v *= v; break;
        case TE_TANH: v = own_tanh(v); break;
        case TE_MUL_LOAD: v *= __ldg(ptrs.in[P.epi_ptr[s]] + (unsigned)(P.epi_base[s] + (int)off)); break;
        case TE_ADD_LOAD: v += __ldg(ptrs.in[P.epi_ptr[s]] + (unsigned)(P.epi_base[s] + (int)off)); break;
        default: break;
        }
    }
    return v;
}

}  // namespace tadc
