// search_fixed.h -- registry of the compile-time-planned kernels (search_fixed.cuh).
#pragma once
#include <vector>

#include "internal.h"

namespace prnu {

// Rows per TMA box of an H-row strip of NC columns (float2): a divisor of H of
// at most 256 rows whose box size is a multiple of 128 bytes, so that every
// box lands 128-byte aligned in shared memory.
__host__ __device__ constexpr int tma_box_rows(int H, int NC, int esize = 8) {
  for (int br = 256; br >= 1; --br)
    if (H % br == 0 && (br * NC * esize) % 128 == 0) return br;
  return 0;
}

// one instantiated column-pass variant: columns per block, threads, shared
// memory; with tma the kernel moves its strip by TMA tile copies of br rows
// and takes a CUtensorMap of the workspace spectra as a second argument,
// otherwise each thread loads and stores its own elements
struct FixedCol {
  int nc;
  int threads;
  size_t smem;
  void* fn;
  bool tma;
  int br;
  int mode;   // 0 plain loads, 1 strip by TMA, 2 fingerprint by bulk copies into the strip buffer, 3/4 into its own region
};

// one instantiated pair of row kernels: row pairs per block, threads per pair
struct FixedRow {
  int ppb;
  int threads;               // per row pair, forward kernel
  int threads_inv;           // per row pair, inverse kernel
  size_t smem;
  void* fwd[kNumStoreLayouts];   // by residual storage type (kF32, kF16, kBF16, kF16P, kBF16P, kF32I)
  void* inv;
  void* fin;                 // per-candidate PCE: one block per candidate, or per window pair (fin_split)
  bool fin_split;
  int fin_threads;
  size_t fin_smem;
};

// the persistent kernel of a shape: row pairs per task, columns per task,
// block size, shared memory, resident blocks per SM, by residual type
struct FixedPersist {
  int ppb, nc, threads;
  size_t smem;
  void* fn[3];
  int blocks_per_sm[3];
};

// Device state of one persistent launch: the ticket, the error flag, and the
// per-candidate completion counts of the four phases ([G] each), all zeroed
// before the launch.  S = workspace slots (spectra, row statistics).
struct PersistArgs {
  int* ticket;
  int* error;
  int* rf_done;
  int* col_done;
  int* ri_done;
  int* fin_done;
  int G;
  int S;
};

struct FixedShape {
  int W, H;
  std::vector<FixedRow> rows;
  std::vector<FixedCol> cols;  // the first is the default tuning's
  int f32_col;               // the one that takes a mode-4 variant's place for FP32 fingerprints
  FixedCol col_fwd, col_inv; // the column pass split for forward units (k_col_fwd_fx, k_col_inv_fx)
  FixedCol col_inv_h;        // k_col_inv_fx with a fingerprint region for FP16 bins (mode 4), taken instead when
                             // every fingerprint of the wave is FP16; fn null where none is instantiated
  FixedPersist persist;
  // the row kernels with `ppb` pairs per block, else the first variant (what
  // the default tuning asks row_for(1) for)
  const FixedRow& row_for(int ppb) const {
    for (auto& r : rows)
      if (r.ppb == ppb) return r;
    return rows.front();
  }
};

// one frame size's instantiated kernels each
FixedShape fixed_shape_256();
FixedShape fixed_shape_720();
FixedShape fixed_shape_1080();
FixedShape fixed_shape_2160();

// The instantiated kernels for frames of H x W, or nullptr.
const FixedShape* find_fixed(int H, int W);

// whether the row kernels chosen for `ppb` pairs per block tile H/2 row pairs exactly
bool fixed_supports(const FixedShape& fs, int H, int ppb);

// row forward, column pass, row inverse and finalisation of one wave (a.nitems candidates)
void launch_fixed_wave(const PassArgs& a, const FixedShape& fs, int col_variant, cudaStream_t s, LaunchCounter& lc);

// every phase of p.G candidates (items 0..G-1 of a) in one persistent launch;
// a.spec / a.stats hold p.S workspace slots
void launch_persistent(const PassArgs& a, const PersistArgs& p, const FixedShape& fs, int sm_count, cudaStream_t s,
                       LaunchCounter& lc);

constexpr int kPersistSlots = 8;

}  // namespace prnu
