// The program of a resident run (k_resident): the passes of a recorded
// circuit as blocks of 32-bit words in the integer pool, written by the
// runtime and read by the kernel.
#pragma once
#include <cstdint>

#include "sv_internal.h"

namespace sv {

constexpr int RES_MAX_BATCH = 8;              // blocks prepared side by side
constexpr int RES_FINAL_BLOCKS = 8;           // of 256 amplitudes in a chunk of the final sample
constexpr int RES_MAX_ROWS = 8192;            // Pauli ops of a resident run (one byte each)
constexpr size_t RES_MAX_SMEM = 224 * 1024;   // dynamic shared memory of a CTA

// A recorded pass is one folded block, or stage blocks whose dense stages act
// on at most two qubits (group bits 0 and 1).  A block is a header, the
// stages, tables and matrices, and (when the pass ends in a reduction, in
// its last block) the decide that follows it.  Offsets inside a block
// are in words from its start.
enum : int32_t {
    RB_NSTAGES = 0,
    RB_RED = 1,      // kind | qubits << 4 | terms or outcomes << 8
    RB_COEF = 2,     // RED_DIAG: float64 weights [term][bin]; RED_FORMS: forms, then residuals
    RB_DECIDE = 3,
    RB_SO = 4,       // swizzled offsets of the four group bits
    RB_SF = 8,       // swizzled offsets of the other address bits, 16 bits each, in lane order
    RB_FOLD = 14,    // the stages are composed into one 16 x 16 matrix
    RB_RUN = 15,     // RED_DIAG: amplitudes per bin that a register pass's group adds up first
    RB_STAGES = 16,
    RS_WORDS = 8
};
// stage words: 0: kind | k << 4 | reset << 8 | pre-drawn << 9 |
// conditional << 10 | value << 11 | classical bit << 12 | parameter set << 20;
// 1: group bits; 2: choice column or pre-drawn row; 3: matrix entries (for a
// parameter set: constant-pool offset) or Pauli table; 4: distance between
// terms (words; reals for a parameter set); 5: structure of every term
// (integer-pool offset for a parameter set); 6: byte offset of the scaled
// matrix of a per-branch stage

// decide words
enum : int32_t {
    RD_KIND = 0, RD_R, RD_PEND, RD_OP, RD_R2, RD_OP2, RD_PEND2, RD_M, RD_CLBITS, RD_WORDS
};

constexpr int RES_MONO_REAL = 1 << 16;  // a monomial matrix's phases are real (with its mono_info)

struct ResDesc {
    int32_t np;           // address bits of the state in shared memory (at least 4)
    int32_t n_states;     // set at launch
    int32_t n_batches;
    int32_t index_off;    // integer-pool offset of (offset, words) per block
    int32_t batch_off;    // integer-pool offset of (first block, blocks) per batch
    int32_t mb;           // most blocks of a batch
    int32_t folds;        // a block is folded
    int32_t max_stages;   // of a block
    int32_t block_words;  // largest block, rounded up
    int32_t br_bytes;     // largest per-branch matrix area of a block
    int32_t n_rows;       // pre-drawn Pauli ops
    int32_t row_table;    // integer-pool offset of their descriptors
    int32_t has_final;
    uint32_t fin_op;
    unsigned long long* hist;  // per shot: its history word, nullable
};

inline int res_swz(int a) { return a ^ ((a >> 4) & 15) ^ ((a >> 8) & 15) ^ ((a >> 12) & 15); }

int resident_threads(int prec, int np);
inline bool resident_one_cta(int prec, int np) { return np >= (prec ? 13 : 14); }  // per SM
int resident_batch(int prec, int np);  // most blocks of a batch
size_t resident_smem_bytes(int prec, const ResDesc& p);
// counts the different words of hist[0..n): words 1 and 0 of the table take
// their number and the sum of number x runs; history_slots words follow
constexpr int HIST_COUNTS = 2;
inline size_t history_slots(uint64_t n) {
    size_t s = 64;
    while (s < 2 * n) s *= 2;
    return s;
}
cudaError_t launch_history_count(const unsigned long long* hist, uint64_t n, unsigned long long* tab,
                                 unsigned long long runs, cudaStream_t s);
cudaError_t init_resident();
cudaError_t launch_resident(const DevBatch& d, int prec, const ResDesc& p, int n_states, int n_sm, cudaStream_t s);

}  // namespace sv
