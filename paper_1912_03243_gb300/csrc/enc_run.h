// Runs of gates on the two-byte code (k_enc.cu): one pass applies a run of
// consecutive gates whose targets are in-block qubits or a few chosen block
// bits, and sign flips on any qubits, in circuit order with the per-gate
// re-encoding of the code.
#pragma once

#include <cstdint>

#include "sv_internal.h"

namespace sv {

constexpr int kEncRunMaxOps = 64;  // ops of one run (one pass)
constexpr int kEncRunMaxBits = 4;  // block bits of a run's tiles

// Shape of a gate's matrix, from its exact zeros.
enum EncShape { ENC_GENERAL = 0, ENC_REAL = 1, ENC_DIAG = 2, ENC_DIAG1 = 3 };  // (DIAG1: u00 = 1)

enum EncOpKind : int {
    ENC_OP_IN = 0,    // 2x2 update on in-block target t
    ENC_OP_FLIP = 1,  // sign flip of the codes
    ENC_OP_PAIR = 2,  // 2x2 update across blocks, target tile bit t
    ENC_OP_SWAP = 3,  // X across blocks: exchange of blocks, target tile bit t
};

struct EncRunOp {
    int kind;
    int t, c;                  // target, in-block control (-1: none)
    int shape;                 // EncShape, as the single-gate kernels use it
    uint32_t lo_mask, lo_val;  // flip: in-block index bits of the condition
    uint32_t amps;             // flip: which of a lane's 8 amplitudes meet bits 0..2 of the condition
    uint32_t pad;
    uint64_t hi_mask, hi_val;  // block-index bits of the condition (block-level control / flip bits)
    float u[8];
};

// The run op of a gate on an n-qubit two-byte state (t of a gate across
// blocks: the target's block-index bit), or false if n < 8.
bool enc_run_op(int n, const Gate1 &g, EncRunOp *op);
// One pass of nops <= kEncRunMaxOps ops (device array) over tiles of 2^nbits
// blocks that differ in the block-index bits pos[0..nbits) (ascending).
cudaError_t launch_enc_run(sv_state *h, const EncRunOp *d_ops, int nops, int nbits, const int *pos);

}  // namespace sv
