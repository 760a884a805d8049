// What the batch's kernels share: one circuit of a batch on the device.
#pragma once

#include "qs_internal.cuh"

namespace qs {

// largest circuit of the one-block-per-circuit kernel (its tableau and two
// layers of gate records in 227 KB of shared memory)
constexpr uint32_t kResidentMaxQubits = 640;

struct BCirc {
  uint32_t n, k, cs, rs, ncols, nrows;
  uint32_t lpr;      // lanes per row in the persistent kernel's update phase (power of two <= 32)
  uint32_t nrounds;
  uint64_t *X, *Z, *S, *RX, *RZ;
  uint32_t *colx;
  int64_t *mst;
  uint64_t *det_x, *det_z;  // k chunks x rs words
  int32_t *det_scal;        // k
  const uint32_t *gates;    // packed records of this circuit
  const int64_t *lptr;      // n_layers + 1 offsets into gates
  const uint32_t *rl, *rm;  // per round: first layer, first measurement (nrounds + 1 each)
  const uint32_t *qubits;   // measured qubits in program order
  uint8_t *record;
  uint64_t seed, shot;
};

// the circuits ids[0..count) (n <= kResidentMaxQubits), one block each, with
// smem >= batch_resident_smem of the largest
size_t batch_resident_smem(uint32_t n);
cudaError_t launch_batch_resident(const BCirc *circs, const uint32_t *ids, uint32_t count, uint32_t threads,
                                  size_t smem, uint32_t round_limit, uint32_t *err, cudaStream_t s);

}  // namespace qs
