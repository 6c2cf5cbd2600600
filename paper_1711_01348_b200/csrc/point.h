// Point programs: general expressions over small index spaces, run by tad_point_kernel (point.cu).
//
// A point is an output (kernels without summation loops) or a term of an output (loops with fixed ranges, flattened
// into one term index).  The program is the stack program of the interpreter with the top of the stack in registers
// and everything below it, and the temporaries, in numbered slots of shared memory, so that one handler serves every
// stack depth.
#pragma once
#include <stdint.h>

#include "program.h"

#define TADQ_MAX_STEPS 96
#define TADQ_MAX_LOADS 12
#define TADQ_MAX_VARS 4        // output variables and flattened loop variables
#define TADQ_MAX_SUMS 4        // bound sums inside the term
#define TADQ_MAX_SLOTS 24
#define TADQ_NONE 255

enum TadqOp : int {
    Q_CONST = 0,  // push imm                      (a push stores the old top in slot s, TADQ_NONE: there is none)
    Q_LOAD,       // push load a
    Q_SLOT,       // push slot a
    Q_NEG, Q_SQR, Q_CUBE, Q_MULC, Q_ADDC,
    Q_LDADD, Q_LDMUL, Q_LDADDSQ,
    Q_FN,         // function b, exponent imm
    Q_ADD, Q_SUB, Q_MUL, Q_DIV,      // top <- slot s op top
    Q_FMA,        // top <- slot s * slot a + top
    Q_STORE,      // slot a <- top, top <- slot s
    Q_ACC,        // sum += top
    Q_MACC,       // sum += slot s * top
    Q_SCALE,      // sum *= top
    Q_LOOP,       // bound sum a begins; jumps to imm when empty
    Q_NEXT,       // bound sum a: next index, jumps to imm while in range
    Q_SUMNEXT     // Q_ADD followed by Q_NEXT
};

struct TadqStep { uint8_t op, s, a, b; int32_t imm; };
struct TadqLoad { int32_t ptr, base, coef[TADQ_MAX_VARS], scoef[TADQ_MAX_SUMS]; };     // over (var), (bound sum index)

struct alignas(16) TadqProgram {
    int32_t n_out, n_z;                    // variables 0 .. n_out-1 index the outputs, the next n_z the terms; last one of a group fastest
    int32_t points, terms;                 // products of their extents
    int32_t lo[TADQ_MAX_VARS], ext[TADQ_MAX_VARS];
    uint32_t div_mul[TADQ_MAX_VARS]; int32_t div_shift[TADQ_MAX_VARS];     // multiply-shift division by ext
    int32_t s_lo[TADQ_MAX_SUMS], s_hi[TADQ_MAX_SUMS];
    int32_t body, tail, n_steps;           // steps [0, body) once per output, [body, tail) per term, [tail, n_steps) on the sum
    int32_t n_slots, n_sums;
    int32_t value_slot;                    // >= 0: the finished sum goes to this slot and the tail computes the output from it
    int32_t out_base, out_coef[TADQ_MAX_VARS], accumulate;
    int32_t unroll;                        // points of a thread in flight: 1 or 4
    int32_t lt, along_terms;               // term lanes per output in a block of 256 threads; lanes run along the terms
    int32_t zsplit, part_limit, part_coef[TADQ_MAX_VARS];      // > 1: grid.y shares of the terms, a plane of partial sums each
    TadqLoad loads[TADQ_MAX_LOADS];
    TadqStep steps[TADQ_MAX_STEPS];
};

// Programs that do not read each other's results run as one launch, each on a range of its blocks.
#define TADQ_BATCH 6
struct alignas(16) TadqBatch {
    int32_t n;
    uint32_t first[TADQ_BATCH + 1];        // first block of every program
    float *out[TADQ_BATCH];
    TadqProgram p[TADQ_BATCH];
};
