// Compact records: scalar and data-axis streams' (32 bytes, run by scalar.cu) and, of twice the
// size, those of streams with matrices and no data axis (matrix.cu).
//
// A Plan's stream (DInst, 48 bytes, operands as kind and index) describes every tape.  A
// stream made of scalar instructions only is translated once, on the host, into records
// the interpreter can execute with few instructions of its own: operands are byte offsets
// into the thread's slot column (one shift-add per operand), constants are part of the
// record, and the cheap rules share one record kind whose unused operands are not loaded.
// A scalar record executes 36 instructions where the general interpreter executes 102, a
// matrix record 118 for 172 (a logistic recurrence and a 4-state Kalman filter).
#pragma once
#include <cstdint>
#include <vector>

#include "plan.h"

namespace ndvm {

// Record kinds.  Fields w[1..7] by kind; slots are kCSlotUnit * slot index, kCNone = none.
enum COp : uint32_t {
  C_ARITH = 0,  // w1 = fma(+-w2, w3, w4) (kCNeg); an absent w3 names the slot of 1, an absent w4 that
                // of -0 (kCHasB, kCHasC: present); kCGate: a zero w2 leaves w4; kCSave: result to
                // workspace w7
  C_FETCH,      // asynchronous copies into slots w1, w3, w5 of workspace w2, w4, w6; kCCommit, kCWait
  C_OBS,        // the point's observations: slots w1, w3, w5 from columns w2, w4, w6 (count in kCCount)
  // forward: w1 result, w2 and w3 operands, w5 auxiliary slot, w6 auxiliary save or power, w7 save
  C_DIV,        // w2 / w3; w4: the slot of 1 / w3 if a C_RCP made it; w5 keeps 1 / w3
  C_RCP,        // w1 = 1 / w2, as C_DIV computes it, for the divisions by w2
  C_POW, C_EXP, C_LOG, C_TANH, C_SQRT, C_ABS, C_SIN, C_COS, C_POWI,
  C_CMP,        // comparison in kCCount
  C_SELECT,     // w2 predicate, w3, w4
  // reverse: w1 the result's adjoint, w2 and w3 targets (kCFirstA, kCFirstB), w4 a, w5 b, w6 result,
  // w7 auxiliary (1/b, or the power)
  R_DIV, R_POW, R_TANH, R_LOG, R_ABS, R_SQRT, R_POWI,
  R_SELECT,     // w4 predicate
  R_DSUM,       // target w2 += adjoint w1 * partial w4
  // the interpreter's inner loop ends at these
  C_END,        // end of the stream
  C_CHUNK,      // end of a chunk (the last of each kCChunk records of a long stream)
  C_LOOP,       // w1 points, w2 stride, w3 base, w4 pc of the matching C_ENDLOOP, w5 validity slot;
                // kCExt: the points' values are in the extended observations
  C_ENDLOOP,
  C_LOADC,      // w1 = constant: w2, w3 its binary64 bits (low, high), w4 its binary32 bits
  C_LOADP,      // w1 = parameter w2
  C_LOADO,      // w1 = observation w2
  C_LOADS,      // w1 = workspace element w2
  C_ZERO,       // w2 slots from w1 on
  C_SEED,       // w1 = 1
  C_GREDUCE,    // w2 slots from w1 on: sums over the thread's points and the lane's threads
  C_LOSS,       // loss = w1
  C_GRAD,       // gradient w2 = w1 (kCNone: 0)
  // matrices (matrix records, 16 words; matrix.cu).  A matrix operand is a slot or, by the flags,
  // an index into the stream's constants; w7 workspace of the result as above
  // products: w1 (rows x cols) = X Y over K terms, element (i, j) = sum over q of X[i xi + q xq]
  // Y[q yq + j yj]; w2 X, w3 Y, w4 = rows | cols << 8 | K << 16, w5 = xi | xq << 16, w6 = yq | yj << 16,
  // w9 2^20 / cols rounded up.  Forward (M_F + K, K = 0 for more than 8): w7 save; kMPost: w11 = w12
  // +- the product too, its save w13 (kMPostNeg, kMPostConst).  Reverse (M_R + K): w10 elements of the
  // gating operand; kMAcc: added to w1, kCNeg: subtracted; kMGateX, kMGateY: an all-zero X (Y)
  // contributes nothing
  M_F, M_F1, M_F2, M_F3, M_F4, M_F5, M_F6, M_F7, M_F8,
  M_R, M_R1, M_R2, M_R3, M_R4, M_R5, M_R6, M_R7, M_R8,
  M_FSPARSE,    // the same with one operand constant, by the list at w8: NZ (w4 >> 24) words per element
  M_RSPARSE,    // of the result, constant's index | other operand's element << 16, kMSplit, kCNone for none
  M_SELECT,     // elements of a slot run w2 by the list at w8 (kCNone: 0); otherwise as M_F
  M_RSELECT,    // the same as M_R without kMAcc
  M_ADD,        // w1 = w2 + w3 (kCNeg: -), w4 elements; slots
  M_COPY,       // w1 = w2 (kCNeg: -), w4 elements
  M_ADDC,       // w1 = w2 + w3 (kCNeg: -), w4 elements; slots or constants
  M_SCALE,      // w1 = w2 (scalar) * w3, w4 elements
  M_INV,        // w1 = inverse of w2, w3 scratch, w4 n | (2^20 / n rounded up) << 8
  M_DET, M_LOGDET,  // w1 of w2, w3 and w4 as above, w5 inverse to slots, w6 inverse to workspace
  M_TRACE,      // w1 of w2, w4 n, w7 save
  M_GATHER,     // w1 = elements named by args[w2 ...], w3 of them
  M_FETCH,      // asynchronous copies of w3 elements from workspace (kMFromObs: observations) w2 on into w1
  M_RSCALE,     // w2 target scalar, w3 target matrix, w5 scalar, w6 matrix, w4 elements
  M_RDET,       // w2 target, w4 as above, w5 determinant (kCNone: log-determinant), w6 inverse
  M_RTRACE,     // w2 target, w4 n
  M_RGATHER,    // args[w2 ...]: w3 pairs (target, first)
  M_RSCATTER,   // w2 target of w5 elements, args[w3 ...]: w4 elements
  C_NOPS
};
// matrix record flags (bits the scalar records' flags leave free); bits 24 to 26 of w0: 1 + the
// groups of copies that may stay pending before the next record (0: no wait)
constexpr uint32_t kMConstX = 1u << 8, kMConstY = 1u << 9, kMAcc = 1u << 10, kMGateX = 1u << 16, kMGateY = 1u << 17,
                   kMPost = 1u << 18, kMPostNeg = 1u << 19, kMPostConst = 1u << 20, kMFromObs = 1u << 21,
                   kMOtherY = 1u << 22;  // products with a list: Y is the operand that varies
constexpr uint32_t kMChains = 1u << 23;  // products with a list: two chains, by kMSplit
constexpr uint32_t kMSplit = 0xfffffffeu;  // in a list: the terms of the second chain follow
constexpr int kMWaitShift = 24;
constexpr size_t kMChunk = 32;         // records of a chunk
constexpr size_t kMMaxConsts = 8192;   // constants a stream may hold in shared memory
constexpr int kMAhead = 3;             // records between a matrix operand's fetch and its use
constexpr uint32_t kCHasB = 1u << 8, kCHasC = 1u << 9, kCGate = 1u << 10, kCSave = 1u << 11, kCFirstA = 1u << 12,
                   kCFirstB = 1u << 13, kCCommit = 1u << 14, kCWait = 1u << 15, kCExt = 1u << 15, kCNeg = 1u << 31;
constexpr int kCCountShift = 16;      // 3 bits: copies of a record, a comparison
constexpr int kCPendingShift = 20;    // 3 bits: groups that may stay pending after a wait
constexpr uint32_t kCNone = 0xffffffffu;
constexpr uint32_t kCSlotUnit = 128;  // a slot row of 32 threads in binary32
constexpr size_t kCChunk = 128;       // records of a chunk
constexpr size_t kCResident = 1024;   // longer loop-free streams are read in chunks
constexpr int kCMaxReciprocals = 8;   // shared reciprocals of a stream (a slot each)
constexpr int kCCopies = 3;           // copies per C_OBS or C_FETCH record

struct alignas(16) CRec {
  uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
};
static_assert(sizeof(CRec) == 4 * kCompactWords, "CRec layout");
struct alignas(16) MRec {
  uint32_t w[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
};
static_assert(sizeof(MRec) == 4 * kMatrixWords, "MRec layout");

// Slots after the plan's own: the validity of a thread's points, and the constants 1 and -0.
constexpr int kCSlotValid = 0, kCSlotOne = 1, kCSlotMinusZero = 2, kCExtraSlots = 3;

// Sets p.compact, p.compact_slots and p.compact_points (and its derive plans') from p.code and
// the constant pool (the tape's `consts`, then p.extra_consts); p.compact stays empty when the
// stream has an instruction without a compact form.  Sets the records' work.
// For a tape with matrices and no data axis, the same for p.matrix*.
void compact_plan(Plan& p, const std::vector<double>& consts);

}  // namespace ndvm
