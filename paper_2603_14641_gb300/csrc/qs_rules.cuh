// Per-word Clifford update rules shared by the fused and batched kernels.
//
// Sec. 2.4 Eq. 4 gives H, P and CX; the rest of the paper's 11-gate set
// (Sec. 6) is the composition of those rules evaluated in registers:
// S^dag = S^3, CZ = H_t CX H_t, CY = S_t CX S_t^dag (circuit order S_t^dag,
// CX, S_t), SWAP, ISWAP = CZ, SWAP, S_a, S_b (circuit order). Each call updates
// one word (32 or 64 rows) of the columns of qubits a (and b) and XORs the
// sign contribution into s. With SIGNS = false (Pauli frames) X/Y/Z change
// nothing and S^dag acts like S.
#pragma once

#include <stdint.h>

#include "../../include/qs.h"

namespace qs {

template <bool SIGNS, typename W>
__device__ __forceinline__ void rule(uint32_t type, W &xa, W &za, W &xb, W &zb, W &s) {
  switch (type) {
    case QS_X: if (SIGNS) s ^= za; break;
    case QS_Z: if (SIGNS) s ^= xa; break;
    case QS_Y: if (SIGNS) s ^= xa ^ za; break;
    case QS_H: { if (SIGNS) s ^= xa & za; W t = xa; xa = za; za = t; } break;
    case QS_S: if (SIGNS) s ^= xa & za; za ^= xa; break;
    case QS_SDG: if (SIGNS) s ^= xa & ~za; za ^= xa; break;
    case QS_CX:
      if (SIGNS) s ^= xa & zb & ~(xb ^ za);
      xb ^= xa; za ^= zb; break;
    case QS_CZ:
      if (SIGNS) s ^= xa & xb & (za ^ zb);
      za ^= xb; zb ^= xa; break;
    case QS_CY:  // S_b^dag, CX(a, b), S_b
      if (SIGNS) s ^= xb & ~zb;
      zb ^= xb;
      if (SIGNS) s ^= xa & zb & ~(xb ^ za);
      xb ^= xa; za ^= zb;
      if (SIGNS) s ^= xb & zb;
      zb ^= xb; break;
    case QS_SWAP: { W t = xa; xa = xb; xb = t; t = za; za = zb; zb = t; } break;
    case QS_ISWAP: {  // CZ, SWAP, S_a, S_b
      if (SIGNS) s ^= xa & xb & (za ^ zb);
      W nza = za ^ xb, nzb = zb ^ xa;
      W t = xa; xa = xb; xb = t;
      za = nzb; zb = nza;
      if (SIGNS) s ^= xa & za;
      za ^= xa;
      if (SIGNS) s ^= xb & zb;
      zb ^= xb;
    } break;
    default: break;
  }
}

// which words a rule changes: bit t of each mask for gate type t
constexpr uint32_t kWritesXa = 1u << QS_H | 1u << QS_SWAP | 1u << QS_ISWAP;
constexpr uint32_t kWritesZa = 1u << QS_H | 1u << QS_S | 1u << QS_SDG | 1u << QS_CX | 1u << QS_CY | 1u << QS_CZ |
                               1u << QS_SWAP | 1u << QS_ISWAP;
constexpr uint32_t kWritesXb = 1u << QS_CX | 1u << QS_CY | 1u << QS_SWAP | 1u << QS_ISWAP;
constexpr uint32_t kWritesZb = 1u << QS_CY | 1u << QS_CZ | 1u << QS_SWAP | 1u << QS_ISWAP;

}  // namespace qs
