// Compact records of scalar and data-axis streams, run by the kernels of scalar.cu.
//
// A Plan's stream (DInst, 48 bytes, operands as kind and index) describes every tape.  A
// stream made of scalar instructions only is translated once, on the host, into records
// the interpreter can execute with few instructions of its own: operands are byte offsets
// into the thread's slot column (one shift-add per operand), constants are part of the
// record, and the cheap rules share one record kind whose unused operands are not loaded.
// A record spends about 25 instructions around its arithmetic where the general
// interpreter spends about 100.
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
  C_LOOP,       // w1 points, w2 stride, w3 base, w4 pc of the matching C_ENDLOOP, w5 validity slot
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
  C_NOPS
};
constexpr uint32_t kCHasB = 1u << 8, kCHasC = 1u << 9, kCGate = 1u << 10, kCSave = 1u << 11, kCFirstA = 1u << 12,
                   kCFirstB = 1u << 13, kCCommit = 1u << 14, kCWait = 1u << 15, kCNeg = 1u << 31;
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

// Slots after the plan's own: the validity of a thread's points, and the constants 1 and -0.
constexpr int kCSlotValid = 0, kCSlotOne = 1, kCSlotMinusZero = 2, kCExtraSlots = 3;

// Sets p.compact, p.compact_slots and p.compact_points (and its derive plans') from p.code and
// the constant pool (the tape's `consts`, then p.extra_consts); p.compact stays empty when the
// stream has an instruction without a compact form.
void compact_plan(Plan& p, const std::vector<double>& consts);

}  // namespace ndvm
