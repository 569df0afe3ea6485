// scan_owner.cuh -- launch interface of the owner-sorted reduce / carry / apply
// check (scan_owner.cu).
#pragma once

#include "scan_trace.cuh"

namespace amc {

// Variables whose statuses fit a CTA's shared memory beside a tile.
constexpr int32_t OWN_MAX_VARS = 1 << 16;
// ... with 128 owners.
constexpr int32_t OWN_NARROW_VARS = 8192;

// Scratch after the single-pass workspace (chunk rows); the sorted tiles take
// the single-pass workspace itself.
size_t owner_workspace_bytes(int64_t n_ops, int32_t n_vars);
// A plain trace: 128 threads a CTA and a three-kernel carry (five kernels), or,
// wide, 256 threads and a one-kernel carry (three kernels).
int launch_scan_owner(const ScanLaunch& L, bool wide, uint8_t* ws, cudaStream_t s);
// A guarded trace in one go (L: the whole check, without guard): the guards
// resolved from the statuses with GT read as Noop.
int launch_guarded_owner(const ScanLaunch& L, bool wide, uint8_t* ws, cudaStream_t s);

}  // namespace amc
