// batch.cuh -- launch interface of the relation-mode batch checker.
#pragma once

#include "amc_internal.cuh"

namespace amc {

struct BatchParams {
    const uint8_t* tok;
    const int32_t* payload;
    const int64_t* prog_tok_off;
    const int32_t* prog_nvars;
    const int64_t* prog_var_off;
    int64_t n_progs;
    int64_t n_tokens;
    const uint8_t* init_mask;      // nullable: every variable starts as {(V,I)}
    uint8_t* step_mask;
    uint8_t* final_mask;
    int64_t* prog_first_fault;
    uint8_t* save;                 // [n_tokens][save_rows]: a unit of tokens [a, b) has the bytes from
    uint8_t* alt;                  //   save_rows a to save_rows b, rows of b - a in them
    const int32_t* order;          // nullable: program queue order
    uint64_t* queue_head;
    int* err;
    int64_t split;                 // segment length of split programs
    int save_rows;                 // construct levels the save / alt rows hold (deeper: AMC_E_INVALID)
    SetTables tab;
};

struct BatchLaunch {
    const uint8_t* tok = nullptr;
    const int32_t* payload = nullptr;
    const int64_t* prog_tok_off = nullptr;
    const int32_t* prog_nvars = nullptr;
    const int64_t* prog_var_off = nullptr;
    int64_t n_progs = 0;
    int64_t n_tokens = 0;
    const uint8_t* init_mask = nullptr;
    uint8_t* step_mask = nullptr;
    uint8_t* final_mask = nullptr;
    int64_t* prog_first_fault = nullptr;
    int* err = nullptr;
    void* workspace = nullptr;
    int longest_first = 1;
    int max_ctas = 0;
    int no_split = 0;              // never split a program (no reduce-pass scratch)
    int save_rows = AMC_MAX_DEPTH; // construct levels with save / alt rows (0: straight-line only)
    int profile = 0;
};

// Programs evaluated variable by variable (batch_vars.cu): positions fit 16
// bits and the variables' last ops a warp's share of shared memory.
constexpr int32_t VARS_MAX_NV = 4096;
constexpr int64_t VARS_MAX_LEN = 65535;
__device__ __forceinline__ bool program_fits_vars(int64_t len, int32_t nv, int64_t split)
{
    return len <= VARS_MAX_LEN && len <= split && nv <= VARS_MAX_NV;
}
// Whether that is done for program `prog`: reported and left out when its
// extents are malformed.
__device__ __forceinline__ bool program_by_vars(const BatchParams& p, int64_t prog)
{
    const int64_t a = p.prog_tok_off[prog], b = p.prog_tok_off[prog + 1];
    const int32_t nv = p.prog_nvars[prog];
    if (a < 0 || b < a || b > p.n_tokens || nv < 0 || p.prog_var_off[prog] < 0 ||
        p.prog_var_off[prog + 1] - p.prog_var_off[prog] != nv) {
        if ((threadIdx.x & 31) == 0) raise_error(p.err, AMC_E_INVALID);
        return false;
    }
    return program_fits_vars(b - a, nv, p.split);
}
// Those programs of the batch (p.save / p.alt with AMC_MAX_DEPTH rows: 8 bytes
// a token each); *queue is zero.  None when *off (device) is set.  Starts beside the
// kernel launched before it, from all before which it takes its input.
int launch_batch_vars(const BatchParams& p, int64_t max_ctas, unsigned long long* queue, const int* off, cudaStream_t s);

size_t batch_workspace_bytes(int64_t n_tokens, int64_t n_progs);
size_t batch_workspace_bytes(int64_t n_tokens, int64_t n_progs, bool no_split, int save_rows);
int launch_batch(const BatchLaunch& B, cudaStream_t s);

}  // namespace amc
