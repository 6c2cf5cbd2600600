// Tile programs: sums whose term couples two variables as written, such as (a[p, l] + b[q, l])^2 c[p] + d[p, l] or
// g[p, l] (a[p, q] + b[q, l]), run by tad_tile_kernel (tile.cu).
//
// A block owns a tile of values of p and q and walks l.  What depends on (p, l) or (q, l) alone (an operand) is evaluated
// once per tile into shared memory, what depends on (p, q) alone once into registers; the term itself, the core, runs on the four
// by four (or eight by four) values of a thread as a short accumulator program over a value X, a value Y and the sums.
#pragma once
#include <stdint.h>

#include "ew.h"
#include "program.h"

#define TADT_NT 256            // threads of a block
#define TADT_OPS 4             // operands of a core
#define TADT_LOADS 10
#define TADT_STEPS 40          // steps of all operands, the factor of a tile's sums and the epilogue
#define TADT_Z 2               // further output variables, one value each per block
#define TADT_SHARES 8          // blocks of a cluster that share a summation
#define TADT_BATCH 4
#define TADT_SMEM (72 * 1024)
#define TADT_SUM (-1)          // E_LD of this load: the finished sum

// One byte per step, the first in the lowest byte: operation | operand << 4 | second operand << 6.
enum TadtOp : int {
    T_END = 0,
    T_LD, T_ADD, T_SUB, T_RSUB, T_MUL,       // X <- o, X + o, X - o, o - X, X * o
    T_FMA,                                   // X <- X * o + o2
    T_SQR, T_CUBE, T_NEG,
    T_MULC, T_ADDC,                          // constant imm[o]
    T_PUSH,                                  // Y <- X
    T_BINY,                                  // X <- Y op X; o: 0 add, 1 sub, 2 mul, 3 div
    T_FN,                                    // function o | o2 << 2 (TadpFn, no powers)
    T_ACC                                    // sum += X (o2 = 0), X * o (1)
};
enum TadtKind : int { TK_ROW = 0, TK_COL, TK_ROWC, TK_COLC, TK_MAT };      // (p, l), (q, l), (p), (q), (p, q)

struct TadtLoad { int32_t ptr, base, cp, cq, cl, cz[TADT_Z]; };
struct TadtOperand {
    int16_t kind, along_l;     // along_l: neighbours along l are neighbours in memory
    int16_t step0, n_steps;    // its program; n_steps = 0: c * load0^e * load1
    int16_t load0, load1, e;   // load1 < 0: none
    float c;
};

struct alignas(16) TadtProgram {
    uint64_t core;
    float imm[4];
    int32_t p_ext, q_ext, l_ext, z_ext[TADT_Z];
    int32_t tm;                // values of p of a thread, 4 or 8; four of q
    int32_t rt, ct, lg;        // threads along p and q, and groups of threads that share l: rt * ct * lg <= TADT_NT
    uint32_t ct_mul, rt_mul;   // n / ct = n * ct_mul >> 16 for n < TADT_NT
    int32_t chunk;             // values of l staged at a time
    int32_t buffers;           // 2 where another piece follows, 1 where one is all
    int32_t smem;              // bytes of shared memory
    int32_t q_sum;             // 1: q is summed too; the blocks of a cluster share its tiles, else they share l
    int32_t shares;            // 1 or TADT_SHARES
    int32_t tiles_p, tiles_q, n_blocks;
    int32_t n_loads, n_ops, n_rows, n_cols;      // loads; operands; those in shared memory of either kind
    int32_t post0, n_post;     // q_sum: factor of a value's sum over l
    int32_t epi0, n_epi;       // from the sum to the output
    int32_t out_base, out_cp, out_cq, out_cz[TADT_Z], accumulate;
    int32_t path;              // which build of the core (0: read step by step)
    TadtOperand op[TADT_OPS];
    TadtLoad loads[TADT_LOADS];
    TadeStep steps[TADT_STEPS];
};

template <int N>
struct TadtBatch {
    int32_t n;
    uint32_t first[N + 1];     // first block of every program, a multiple of the cluster
    float *out[N];
    TadtProgram p[N];
};

// cores with a build of their own: the square of a sum of two operands, alone and as c X + d, and a sum of two operands, one of
// which stays, times a third
constexpr uint64_t tadt_step(int op, int o = 0, int o2 = 0) { return (uint64_t)(op | o << 4 | o2 << 6); }
constexpr uint64_t TADT_SQUARES = tadt_step(T_LD, 0) | tadt_step(T_ADD, 1) << 8 | tadt_step(T_SQR) << 16 | tadt_step(T_ACC) << 24;
constexpr uint64_t TADT_SQUARES_FMA = tadt_step(T_LD, 0) | tadt_step(T_ADD, 1) << 8 | tadt_step(T_SQR) << 16 | tadt_step(T_FMA, 2, 3) << 24 |
                                      tadt_step(T_ACC) << 32;
constexpr uint64_t TADT_WEIGHTED = tadt_step(T_LD, 0) | tadt_step(T_ADD, 1) << 8 | tadt_step(T_ACC, 2, 1) << 16;
