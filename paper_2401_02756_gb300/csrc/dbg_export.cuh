// The sorted export by bins (dbg_export_bins.cu), for tables of at most
// 2^32 - 1 slots, k up to 64.
#pragma once

#include "dbg_internal.cuh"

namespace dbg {

// Device bytes of scratch export_bins needs for outputs of `rows` rows of a table.
int export_bins_scratch(int k, uint64_t rows, uint64_t n_slots, uint64_t &bytes);

// Sorted keys and counter rows into 16-byte aligned device outputs of
// `max_rows` rows; *D receives the number of vertices (more than max_rows:
// nothing is written).  `scratch`: caller's device memory (256-byte aligned),
// or null to take it from the library's pool.  *too_dense: more of the
// keys crowd into a few bins than this sort takes (or has scratch for), and the
// outputs hold nothing of use.  Waits for `s`.
// `no_records` (if not null): the outputs are to be written once, in order --
// pinned host memory --, so the records must have a place of their own; set,
// with nothing else done, when there is none.  Returns the graph's sticky
// status (or NEEDS_GROW) when it has one.
int export_bins(dbg_handle h, uint64_t *keys_out, uint32_t *counts_out, uint64_t max_rows,
                uint64_t *D, cudaStream_t s, void *scratch, uint64_t scratch_bytes,
                bool *too_dense, bool *no_records = nullptr);

// Bytes of the handle's second event buffer (dbg_binned.cu).
uint64_t bin_ev2_bytes(dbg_handle h);

}  // namespace dbg
