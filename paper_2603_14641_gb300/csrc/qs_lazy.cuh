// Deferred one-qubit gates.
//
// A one-qubit gate reads and writes its two columns for nothing if a two-qubit
// gate reads them again soon after. Within a run of layers, every one-qubit
// gate is therefore only composed into a pending operation of its qubit (7
// bits), and a two-qubit gate takes the pending operations of both qubits along
// and applies them to the words it loads anyway; what is pending after the last
// layer is applied then. Nothing else touches a qubit's columns in between, so
// the words and the sign terms are those of applying each gate in its layer.
//
// A one-qubit Clifford acts on the words (x, z) of a column pair and the signs s as
//   x' = m0 x + m1 z,  z' = m2 x + m3 z,  s += a x + b z + c x z   (over GF(2));
// the operation is kept as those 7 bits with m0 and m3 inverted, so that 0 is
// the identity. With m invertible the product x' z' is m0 m2 x + m1 m3 z + x z,
// which gives the composition rules below (Sec. 2.4 Eq. 4 and the 11-gate set).
#pragma once

#include <stdint.h>

#include "../../include/qs.h"

namespace qs {

// bits of an operation
constexpr uint32_t kOpM0 = 1, kOpM1 = 2, kOpM2 = 4, kOpM3 = 8, kOpA = 16, kOpB = 32, kOpC = 64;

// operation `op` followed by the one-qubit gate `type`
__host__ __device__ __forceinline__ uint32_t op_then(uint32_t op, uint32_t type) {
  uint32_t m0 = (op & 1) ^ 1, m1 = (op >> 1) & 1, m2 = (op >> 2) & 1, m3 = ((op >> 3) & 1) ^ 1;
  uint32_t a = (op >> 4) & 1, b = (op >> 5) & 1, c = (op >> 6) & 1;
  const bool h = type == QS_H, s = type == QS_S, sdg = type == QS_SDG;
  if (h || s || sdg) {  // s += x' z', for S^dag + x'
    a ^= (m0 & m2) ^ (sdg ? m0 : 0);
    b ^= (m1 & m3) ^ (sdg ? m1 : 0);
    c ^= 1;
  }
  if (type == QS_X || type == QS_Y) { a ^= m2; b ^= m3; }  // s += z'
  if (type == QS_Z || type == QS_Y) { a ^= m0; b ^= m1; }  // s += x'
  if (h) {
    uint32_t t = m0; m0 = m2; m2 = t;
    t = m1; m1 = m3; m3 = t;
  }
  if (s || sdg) { m2 ^= m0; m3 ^= m1; }  // z' += x'
  return (m0 ^ 1) | m1 << 1 | m2 << 2 | (m3 ^ 1) << 3 | a << 4 | b << 5 | c << 6;
}

// the one-qubit gate `type` followed by operation `op`
__host__ __device__ __forceinline__ uint32_t op_after(uint32_t type, uint32_t op) {
  uint32_t m0 = (op & 1) ^ 1, m1 = (op >> 1) & 1, m2 = (op >> 2) & 1, m3 = ((op >> 3) & 1) ^ 1;
  uint32_t a = (op >> 4) & 1, b = (op >> 5) & 1, c = (op >> 6) & 1;
  if (type == QS_H) {  // (x, z) -> (z, x), s += x z
    uint32_t t = m0; m0 = m1; m1 = t;
    t = m2; m2 = m3; m3 = t;
    t = a; a = b; b = t;
    c ^= 1;
  } else if (type == QS_S || type == QS_SDG) {  // z -> x + z, s += x z, for S^dag + x; x (x + z) = x + x z
    m0 ^= m1;
    m2 ^= m3;
    a ^= b ^ c ^ (type == QS_SDG);
    c ^= 1;
  } else {
    a ^= type == QS_Z || type == QS_Y;  // s += x
    b ^= type == QS_X || type == QS_Y;  // s += z
  }
  return (m0 ^ 1) | m1 << 1 | m2 << 2 | (m3 ^ 1) << 3 | a << 4 | b << 5 | c << 6;
}

// whether the operation changes the x (z) word
__device__ __forceinline__ bool op_changes_x(uint32_t op) { return op & (kOpM0 | kOpM1); }
__device__ __forceinline__ bool op_changes_z(uint32_t op) { return op & (kOpM2 | kOpM3); }

// the operation's seven bits as word masks
struct OpMasks {
  uint32_t m0, m1, m2, m3, a, b, c;
  __device__ __forceinline__ explicit OpMasks(uint32_t op) {
    auto mask = [op](int bit) { return (uint32_t)((int32_t)(op << (31 - bit)) >> 31); };
    m0 = ~mask(0); m1 = mask(1); m2 = mask(2); m3 = ~mask(3);
    a = mask(4); b = mask(5); c = mask(6);
  }
};

__device__ __forceinline__ uint32_t widen(uint32_t m, uint32_t) { return m; }
__device__ __forceinline__ uint64_t widen(uint32_t m, uint64_t) { return ((uint64_t)m << 32) | m; }

template <bool SIGNS, typename W>
__device__ __forceinline__ void op_apply(const OpMasks &o, W &x, W &z, W &s) {
  if (SIGNS) s ^= (x & ((z & widen(o.c, x)) ^ widen(o.a, x))) ^ (z & widen(o.b, x));
  const W nx = (x & widen(o.m0, x)) ^ (z & widen(o.m1, x));
  z = (x & widen(o.m2, x)) ^ (z & widen(o.m3, x));
  x = nx;
}

// Record of a two-qubit gate with the pending operations of its qubits:
// type << 20 | qa, with opA from bit 24; qb, with opB from bit 24 (n <= 2^20).
__device__ __forceinline__ uint2 pair_record(uint32_t type, uint32_t qa, uint32_t qb, uint32_t opa, uint32_t opb) {
  return make_uint2(opa << 24 | type << 20 | qa, opb << 24 | qb);
}
// Record of an operation left pending (type QS_I)
__device__ __forceinline__ uint2 single_record(uint32_t q, uint32_t op) { return make_uint2(op << 24 | q, 0); }

}  // namespace qs
