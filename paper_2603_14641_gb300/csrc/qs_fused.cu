// Fused gate segments: many consecutive layers per tableau pass.
//
// Every generator row evolves independently under the update rules (Sec. 2.4,
// Eq. 4: the rules apply to each row index i), so the rows held by one column
// word can run through a whole segment of layers -- up to the next measurement --
// without any other row. A block loads a slice of a few words of every column
// (X[q][w], Z[q][w] for all n qubits) into shared memory, applies every gate of
// every layer of the segment there (gates of one layer touch disjoint qubits, so
// threads of one layer never collide; a barrier separates layers), accumulates
// its sign contributions in registers and writes the slice back once. Global
// traffic per segment drops from (layers x touched columns) to one read and one
// write of the tableau plus the gate records. The paper launches one kernel per
// window (Sec. 4.1, Alg. 2); this is the fused alternative for tableaus whose
// one-word slice fits in the shared memory of an SM (n up to 14,080 qubits).
//
// Three launches per segment of up to kFusedLayers layers:
//   fused_scatter  act[l][q] = what layer l does to qubit q (all gates at once);
//   fused_records  one record per two-qubit gate with the one-qubit gates since
//                  the previous two-qubit gate of either qubit, composed walking
//                  back through act (qs_lazy.cuh), and one per qubit with
//                  something left over after the last layer;
//   fused_segment  the slices. What bounds it is shared-memory bank conflicts
//                  (random columns, 16 lanes a wavefront of 64-bit words: 3.1
//                  wavefronts each on average) and per-word instructions, so
//                  one-qubit gates cost nothing of their own, only changed words
//                  are written, and where a block holds several words of a
//                  column, neighbouring lanes take them (8 words: 1.5).
#include <algorithm>
#include <cmath>

#include "qs_internal.cuh"
#include "qs_lazy.cuh"
#include "qs_rules.cuh"

namespace qs {

constexpr size_t kFusedSmemMax = 220 * 1024;
constexpr uint8_t kActTwo = 0xFF;  // act: a two-qubit gate (else the one-qubit gate's type, 0 for none)

bool fused_fits(uint32_t n) { return (size_t)16 * n <= kFusedSmemMax; }

// records per layer: its two-qubit gates; one more layer of up to n records at the end
static uint32_t rec_stride(uint32_t n) { return std::max(1u, n / 2); }

struct FusedScratch {
  uint32_t *count;  // records per layer, kFusedLayers + 1
  uint8_t *act;     // [layer][qubit]
  uint2 *rec;       // [layer][rec_stride], then n
};

static size_t act_offset() { return ((kFusedLayers + 1) * 4 + 255) / 256 * 256; }
static size_t rec_offset(uint32_t n) { return act_offset() + ((size_t)kFusedLayers * n + 255) / 256 * 256; }

size_t fused_scratch_bytes(uint32_t n) {
  return fused_fits(n) ? rec_offset(n) + ((size_t)kFusedLayers * rec_stride(n) + n) * 8 : 0;
}

// Gate offsets of the segment's layers. They go with the launch: copied to the
// device first, they cost an event and a transfer the kernels wait for.
struct LayerOffsets {
  int64_t base;
  uint32_t off[kFusedLayers + 1];
};

__device__ __forceinline__ bool valid_gate(uint2 q, uint32_t n) {
  const uint32_t type = q.x >> 24, qa = q.x & 0xFFFFFFu;
  const bool two = type >= QS_CX && type <= QS_ISWAP;
  return qa < n && type < QS_NUM_GATE_TYPES && !(two && (q.y >= n || q.y == qa));
}

__global__ void __launch_bounds__(256)
fused_scatter_kernel(const uint2 *__restrict__ packed, const __grid_constant__ LayerOffsets o, uint32_t n,
                     uint8_t *__restrict__ act, uint32_t *__restrict__ err) {
  const uint32_t l = blockIdx.y, g = o.off[l] + blockIdx.x * 256 + threadIdx.x;
  if (g >= o.off[l + 1]) return;
  const uint2 q = __ldg(packed + o.base + g);
  if (!valid_gate(q, n)) {
    atomicOr(err, kErrBadGate);
    return;
  }
  const uint32_t type = q.x >> 24;
  uint8_t *row = act + (size_t)l * n;
  if (type >= QS_CX) {
    row[q.x & 0xFFFFFFu] = kActTwo;
    row[q.y] = kActTwo;
  } else {
    row[q.x & 0xFFFFFFu] = (uint8_t)type;
  }
}

// the one-qubit gates on qubit q between its last two-qubit gate and layer l
__device__ __forceinline__ uint32_t pending_before(const uint8_t *__restrict__ act, uint32_t n, uint32_t l, uint32_t q) {
  uint32_t op = 0;
  while (l > 0) {
    const uint32_t t = __ldg(act + (size_t)(--l) * n + q);
    if (t == kActTwo) break;
    if (t) op = op_after(t, op);
  }
  return op;
}

// grid.y = layers + 1: the last row lists what is pending after the last layer
__global__ void __launch_bounds__(256)
fused_records_kernel(const uint2 *__restrict__ packed, const __grid_constant__ LayerOffsets o, uint32_t n, uint32_t layers,
                     const uint8_t *__restrict__ act, uint2 *__restrict__ rec, uint32_t stride,
                     uint32_t *__restrict__ count) {
  __shared__ uint32_t s_warp[8], s_base;
  const uint32_t l = blockIdx.y, t = threadIdx.x, lane = t & 31, warp = t >> 5, i = blockIdx.x * 256 + t;
  bool emit = false;
  uint2 out = make_uint2(0, 0);
  if (l < layers) {
    const uint32_t a = o.off[l], end = o.off[l + 1], g = a + i;
    if (a + blockIdx.x * 256 >= end) return;  // uniform over the block
    if (g < end) {
      const uint2 q = __ldg(packed + o.base + g);
      const uint32_t type = q.x >> 24, qa = q.x & 0xFFFFFFu;
      if (type >= QS_CX && valid_gate(q, n)) {
        out = pair_record(type, qa, q.y, pending_before(act, n, l, qa), pending_before(act, n, l, q.y));
        emit = true;
      }
    }
  } else if (i < n) {
    const uint32_t op = pending_before(act, n, l, i);
    out = single_record(i, op);
    emit = op != 0;
  }
  const uint32_t ball = __ballot_sync(0xffffffffu, emit);
  if (lane == 0) s_warp[warp] = __popc(ball);
  __syncthreads();
  if (t == 0) {
    uint32_t sum = 0;
    for (int w = 0; w < 8; ++w) sum += s_warp[w];
    s_base = sum ? atomicAdd(count + l, sum) : 0;
  }
  __syncthreads();
  uint32_t at = s_base + __popc(ball & ((1u << lane) - 1));
  for (uint32_t w = 0; w < warp; ++w) at += s_warp[w];
  if (emit) rec[(size_t)l * stride + at] = out;
}

struct FusedArgs {
  void *X, *Z, *S;             // in words of the kernel's type
  uint32_t n, stride, nwords;  // column stride and the words that matter, same type
  const uint2 *rec;
  const uint32_t *count;
  uint32_t rec_stride, layers;  // with the final list: layers + 1 record lists
};

constexpr int kSliceAhead = 8;  // columns per thread in flight while a slice is read

// W: word type (32-bit words halve a slice where 64-bit ones would leave SMs
// idle); J: words per block and lanes per gate; R: records per thread loaded one
// layer ahead (further ones are loaded when they are due; two layers ahead with
// the counts in shared memory measured no faster)
template <typename W, bool SIGNS, int J, int R>
__global__ void __launch_bounds__(1024) fused_segment_kernel(const FusedArgs a) {
  extern __shared__ __align__(16) uint8_t fsm[];
  __shared__ uint32_t s_sign[J * sizeof(W) / 4];
  W *sx = reinterpret_cast<W *>(fsm), *sz = sx + (size_t)a.n * J;
  W *X = static_cast<W *>(a.X), *Z = static_cast<W *>(a.Z);
  const uint32_t t = threadIdx.x, T = blockDim.x, w0 = blockIdx.x * J, n = a.n;
  const uint32_t j = t % J, gl = t / J, gs = T / J;
  if (SIGNS && t < J * sizeof(W) / 4) s_sign[t] = 0;
  uint32_t cnt = __ldg(a.count), cnt1 = __ldg(a.count + 1);
  const bool in = w0 + j < a.nwords;
  for (uint32_t q0 = gl; q0 < n; q0 += kSliceAhead * gs) {
    W vx[kSliceAhead], vz[kSliceAhead];
#pragma unroll
    for (int i = 0; i < kSliceAhead; ++i) {
      const uint32_t q = q0 + i * gs;
      const bool ld = in && q < n;
      vx[i] = ld ? X[(size_t)q * a.stride + w0 + j] : W(0);
      vz[i] = ld ? Z[(size_t)q * a.stride + w0 + j] : W(0);
    }
#pragma unroll
    for (int i = 0; i < kSliceAhead; ++i) {
      const uint32_t q = q0 + i * gs;
      if (q < n) { sx[q * J + j] = vx[i]; sz[q * J + j] = vz[i]; }
    }
  }
  uint2 pre[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const uint32_t g = gl + i * gs;
    pre[i] = g < cnt ? __ldg(a.rec + g) : make_uint2(0, 0);
  }
  W sacc = 0;
  auto gate = [&](uint2 r) {
    const uint32_t type = (r.x >> 20) & 15, opa = r.x >> 24, opb = r.y >> 24;
    W *xa = sx + (r.x & 0xFFFFFu) * J + j, *za = sz + (r.x & 0xFFFFFu) * J + j;
    W va = *xa, ua = *za;
    if (type) {
      W *xb = sx + (r.y & 0xFFFFFu) * J + j, *zb = sz + (r.y & 0xFFFFFu) * J + j;
      W vb = *xb, ub = *zb;
      op_apply<SIGNS>(OpMasks(opa), va, ua, sacc);
      op_apply<SIGNS>(OpMasks(opb), vb, ub, sacc);
      if (type == QS_CX) {
        rule<SIGNS>(QS_CX, va, ua, vb, ub, sacc);
        if (op_changes_x(opa)) *xa = va;
        *za = ua;
        *xb = vb;
        if (op_changes_z(opb)) *zb = ub;
      } else {
        rule<SIGNS>(type, va, ua, vb, ub, sacc);
        *xa = va;
        *za = ua;
        *xb = vb;
        *zb = ub;
      }
    } else {
      op_apply<SIGNS>(OpMasks(opa), va, ua, sacc);
      if (op_changes_x(opa)) *xa = va;
      if (op_changes_z(opa)) *za = ua;
    }
  };
  __syncthreads();
  for (uint32_t l = 0; l <= a.layers; ++l) {
    const uint32_t cnt2 = l + 2 <= a.layers ? __ldg(a.count + l + 2) : 0;
    const uint2 *rec = a.rec + (size_t)l * a.rec_stride;
    uint2 cur[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      cur[i] = pre[i];
      const uint32_t g = gl + i * gs;
      pre[i] = l < a.layers && g < cnt1 ? __ldg(rec + a.rec_stride + g) : make_uint2(0, 0);
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (gl + i * gs < cnt) gate(cur[i]);
    for (uint32_t g = gl + R * gs; g < cnt; g += gs) gate(__ldg(rec + g));
    __syncthreads();
    cnt = cnt1;
    cnt1 = cnt2;
  }
  for (uint32_t q = gl; q < n; q += gs)
    if (in) {
      X[(size_t)q * a.stride + w0 + j] = sx[q * J + j];
      Z[(size_t)q * a.stride + w0 + j] = sz[q * J + j];
    }
  if (SIGNS) {
    const uint64_t v = sacc;
    if ((uint32_t)v) atomicXor(s_sign + j * (sizeof(W) / 4), (uint32_t)v);
    if (sizeof(W) == 8 && (uint32_t)(v >> 32)) atomicXor(s_sign + 2 * j + 1, (uint32_t)(v >> 32));
    __syncthreads();
    constexpr uint32_t per = sizeof(W) / 4;
    if (t < J * per && w0 + t / per < a.nwords) static_cast<uint32_t *>(a.S)[w0 * per + t] ^= s_sign[t];
  }
}

template <typename W, bool SIGNS, int J, int R>
static cudaError_t launch_fused_t(const FusedArgs &a, uint32_t threads, cudaStream_t s) {
  static std::atomic<uint64_t> attr_set{0};  // one bit per device ordinal
  cudaError_t e = once_per_device(attr_set, []() {
    return cudaFuncSetAttribute(fused_segment_kernel<W, SIGNS, J, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kFusedSmemMax);
  });
  if (e != cudaSuccess) return e;
  fused_segment_kernel<W, SIGNS, J, R>
      <<<(a.nwords + J - 1) / J, threads, 2 * (size_t)a.n * J * sizeof(W), s>>>(a);
  return cudaGetLastError();
}

template <typename W, bool SIGNS, int J>
static cudaError_t launch_fused_r(const FusedArgs &a, uint32_t threads, uint32_t records, cudaStream_t s) {
  const uint32_t r = (records * J + threads - 1) / threads;
  if (r <= 1) return launch_fused_t<W, SIGNS, J, 1>(a, threads, s);
  if (r <= 2) return launch_fused_t<W, SIGNS, J, 2>(a, threads, s);
  return launch_fused_t<W, SIGNS, J, 4>(a, threads, s);
}

// Short segments of small programs, where three more launches cost more than
// deferring saves: one launch that applies every gate in its layer, one 64-bit
// word per block. With few gates a thread what bounds it is the latency of a
// layer, so each thread copies its R records of the layers ahead to its own slots
// of a ring of D stages, D - 1 layers ahead (R = 0: no ring, plain loads). 100
// layers of 256 qubits: 69 us with the next layer's records in registers and the
// offsets copied to the device first, 48 now; 1,500 qubits, 10 layers 26 and 23.
// (The rules without a branch on the gate type measured the same here.)
template <bool SIGNS, int R, int D>
__global__ void __launch_bounds__(1024)
fused_direct_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ S, uint32_t n,
                    uint32_t stride, const uint2 *packed, const __grid_constant__ LayerOffsets o,
                    uint32_t layers, uint32_t *__restrict__ err) {
  chain_start();
  extern __shared__ __align__(16) uint8_t fsm[];
  __shared__ uint32_t s_sign[2];
  uint64_t *sx = reinterpret_cast<uint64_t *>(fsm), *sz = sx + n;
  uint2 *ring = reinterpret_cast<uint2 *>(sz + n);
  const uint32_t t = threadIdx.x, T = blockDim.x, w = blockIdx.x;
  if (SIGNS && t < 2) s_sign[t] = 0;
  packed += o.base;
  auto fetch = [&](uint32_t l) {
    if (l < layers) {
      const uint32_t a = o.off[l], b = o.off[l + 1];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const uint32_t g = a + t + i * T;
        if (g < b) {
          const uint32_t slot = (uint32_t)__cvta_generic_to_shared(ring + ((l % D) * R + i) * T + t);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(slot), "l"(packed + g) : "memory");
        }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int l = 0; l < D - 1; ++l) fetch(l);
  for (uint32_t q = t; q < n; q += T) {
    sx[q] = X[(size_t)q * stride + w];
    sz[q] = Z[(size_t)q * stride + w];
  }
  uint64_t sacc = 0;
  bool bad = false;
  auto gate = [&](uint2 r) {
    if (!valid_gate(r, n)) {
      bad = true;
      return;
    }
    const uint32_t type = r.x >> 24, qa = r.x & 0xFFFFFFu, qb = type >= QS_CX ? r.y : qa;
    uint64_t xa = sx[qa], za = sz[qa], xb = sx[qb], zb = sz[qb];
    rule<SIGNS>(type, xa, za, xb, zb, sacc);
    if ((kWritesXa >> type) & 1) sx[qa] = xa;
    if ((kWritesZa >> type) & 1) sz[qa] = za;
    if ((kWritesXb >> type) & 1) sx[qb] = xb;
    if ((kWritesZb >> type) & 1) sz[qb] = zb;
  };
  __syncthreads();
  for (uint32_t l = 0; l < layers; ++l) {
    fetch(l + D - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
    const uint32_t a = o.off[l], b = o.off[l + 1];
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (a + t + i * T < b) gate(ring[((l % D) * R + i) * T + t]);
    for (uint32_t g = a + t + R * T; g < b; g += T) gate(packed[g]);
    __syncthreads();
  }
  if (bad && blockIdx.x == 0) atomicOr(err, kErrBadGate);
  for (uint32_t q = t; q < n; q += T) {
    X[(size_t)q * stride + w] = sx[q];
    Z[(size_t)q * stride + w] = sz[q];
  }
  if (SIGNS) {
    if ((uint32_t)sacc) atomicXor(s_sign, (uint32_t)sacc);
    if ((uint32_t)(sacc >> 32)) atomicXor(s_sign + 1, (uint32_t)(sacc >> 32));
    __syncthreads();
    if (t == 0) S[w] ^= ((uint64_t)s_sign[1] << 32) | s_sign[0];
  }
}

static size_t direct_smem(uint32_t n, uint32_t threads, uint32_t R, uint32_t D) {
  return (size_t)16 * n + (size_t)8 * R * D * threads;
}

template <bool SIGNS, int R, int D>
static cudaError_t launch_direct_t(uint64_t *X, uint64_t *Z, uint64_t *S, uint32_t n, uint32_t stride, uint32_t nwords,
                                   const uint2 *gates, const LayerOffsets &o, uint32_t L, uint32_t threads,
                                   uint32_t *err, cudaStream_t s) {
  static std::atomic<uint64_t> attr_set{0};
  cudaError_t e = once_per_device(attr_set, []() {
    return cudaFuncSetAttribute(fused_direct_kernel<SIGNS, R, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kFusedSmemMax);
  });
  if (e != cudaSuccess) return e;
  return launch_chained(fused_direct_kernel<SIGNS, R, D>, nwords, threads, direct_smem(n, threads, R, D), s, X, Z, S, n,
                        stride, gates, o, L, err);
}

template <bool SIGNS>
static cudaError_t launch_direct(uint64_t *X, uint64_t *Z, uint64_t *S, uint32_t n, uint32_t stride, uint32_t nwords,
                                 const uint2 *gates, const LayerOffsets &o, uint32_t L, uint32_t max_gates,
                                 uint32_t *err, cudaStream_t s) {
  const uint32_t threads = std::min(1024u, std::max(128u, (max_gates + 31) / 32 * 32));
  const bool one = max_gates <= threads;
  if (one && direct_smem(n, threads, 1, 8) <= kFusedSmemMax)
    return launch_direct_t<SIGNS, 1, 8>(X, Z, S, n, stride, nwords, gates, o, L, threads, err, s);
  if (!one && direct_smem(n, threads, 4, 4) <= kFusedSmemMax)
    return launch_direct_t<SIGNS, 4, 4>(X, Z, S, n, stride, nwords, gates, o, L, threads, err, s);
  // columns that leave no room (from 5,900 qubits at 1,024 threads): a handful of layers
  return launch_direct_t<SIGNS, 0, 1>(X, Z, S, n, stride, nwords, gates, o, L, threads, err, s);
}

struct FusedShape { int words; bool half; uint32_t threads; };

// Shape of the slices: words per block (64-bit, or one 32-bit word) and threads,
// by the estimated cycles of a layer. With `items` (two-qubit gates x words, about
// half of `records`) a block's layer takes max(c items / 32 * w, rounds (l + r
// warps)): w cycles per 32 items of each of the c blocks an SM holds (bank
// conflicts and instructions), and a latency per round of its threads; times the
// waves of blocks. The constants are fitted to 15 sizes; the choice is within 4 %
// of the best measured shape on average, e.g. per layer 10,000 qubits 8.7 us (one
// 64-bit word, 1,024 threads; 9.5 with 32-bit words), 5,000 qubits 3.05 (two
// words; 3.4 with one), frames of 1,000 qubits and 200,000 shots 4.5 (two words,
// 256 threads; 4.9 with one), of 10,000 qubits and 1,024 shots 2.3 (32-bit words;
// 2.9 with 64-bit ones). Applying each one-qubit gate in its layer, one word per
// lane: 14.1, 5.1, 17.1 and 4.7 us.
static FusedShape fused_shape(uint32_t n, uint32_t nwords, uint32_t records, bool signs, int sms) {
  FusedShape best{1, false, 1024};
  double least = 1e30;
  const double gates = std::max(1.0, 0.5 * records);
  const struct { int words; bool half; } kinds[5] = {{8, false}, {4, false}, {2, false}, {1, false}, {1, true}};
  for (const auto &k : kinds) {
    const uint32_t total = k.half ? 2 * nwords : nwords;
    const size_t smem = (size_t)n * k.words * (k.half ? 8 : 16);
    if (smem > kFusedSmemMax || (k.words > 1 && (uint32_t)k.words > nwords)) continue;
    const double items = gates * k.words;
    for (uint32_t threads : {1024u, 512u, 256u, 128u}) {
      const uint32_t ahead = (records * k.words + threads - 1) / threads;  // records a thread holds
      const uint32_t regs = k.half && ahead <= 2 ? 32 : signs ? 64 : 56;
      const uint32_t per_sm = std::max<uint32_t>(
          1, std::min<uint32_t>(64000 / (regs * threads), (uint32_t)((227 * 1024) / (smem + 1024))));
      const uint32_t blocks = (total + k.words - 1) / k.words, slots = per_sm * sms;
      const uint32_t waves = (blocks + slots - 1) / slots, here = std::min(per_sm, (blocks + sms - 1) / sms);
      const double rounds = std::ceil(items / threads), warps = std::min(items, (double)threads) / 32;
      const double cost = waves * std::max(here * items / 32 * (k.half ? 38 : 52),
                                           rounds * (1150 + warps * (k.half ? 20 : 32) + 0.05 * threads));
      if (cost < least) { least = cost; best = {k.words, k.half, threads}; }
    }
  }
  return best;
}

template <bool SIGNS>
static cudaError_t launch_slices(FusedArgs a, const FusedShape &f, uint32_t records, cudaStream_t s) {
  if (f.half) {
    a.stride *= 2;
    a.nwords *= 2;
    return launch_fused_r<uint32_t, SIGNS, 1>(a, f.threads, records, s);
  }
  if (f.words == 8) return launch_fused_r<uint64_t, SIGNS, 8>(a, f.threads, records, s);
  if (f.words == 4) return launch_fused_r<uint64_t, SIGNS, 4>(a, f.threads, records, s);
  if (f.words == 2) return launch_fused_r<uint64_t, SIGNS, 2>(a, f.threads, records, s);
  return launch_fused_r<uint64_t, SIGNS, 1>(a, f.threads, records, s);
}

cudaError_t launch_fused_segment(uint64_t *X, uint64_t *Z, uint64_t *S, uint32_t n, uint32_t stride, uint32_t nwords,
                                 const uint32_t *packed, const int64_t *ptr, uint32_t L, int sms, void *scratch,
                                 uint32_t *err, cudaStream_t s, int *launches) {
  if (L == 0 || L > kFusedLayers) return cudaErrorInvalidValue;
  LayerOffsets o;
  uint32_t max_gates = 0;  // layers hold at most n gates (checked when they were added)
  o.base = ptr[0];
  for (uint32_t l = 0; l <= L; ++l) o.off[l] = (uint32_t)(ptr[l] - ptr[0]);
  for (uint32_t l = 0; l < L; ++l) max_gates = std::max(max_gates, o.off[l + 1] - o.off[l]);
  const uint2 *gates = reinterpret_cast<const uint2 *>(packed);
  // Deferring halves what the blocks of an SM spend on a layer beyond its latency,
  // about 52 cycles per 32 two-qubit gates of a word; three more launches and a
  // memset cost about 8 us. Measured, deferred / direct: 256 qubits 10 layers
  // 28 / 16 us (1,040 by this count), 1,500 qubits 50 layers 54 / 54 (30,468), 2,500
  // qubits 25 layers 52 / 51 (25,390) and 100 layers 104 / 152 (101,562), 1,000
  // qubits and 20,000 shots 25 layers 56 / 61 (30,468)
  const double cycles = 0.25 * n / 32 * 52 * ((nwords + sms - 1) / sms);
  if (cycles * L < 28000) {
    *launches += 1;
    return S ? launch_direct<true>(X, Z, S, n, stride, nwords, gates, o, L, max_gates, err, s)
             : launch_direct<false>(X, Z, S, n, stride, nwords, gates, o, L, max_gates, err, s);
  }
  *launches += max_gates ? 3 : 2;
  uint8_t *p = static_cast<uint8_t *>(scratch);
  uint32_t *count = reinterpret_cast<uint32_t *>(p);
  uint8_t *act = p + act_offset();
  uint2 *rec = reinterpret_cast<uint2 *>(p + rec_offset(n));
  cudaError_t e = cudaMemsetAsync(p, 0, act_offset() + (size_t)L * n, s);
  if (e != cudaSuccess) return e;
  if (max_gates)
    fused_scatter_kernel<<<dim3((max_gates + 255) / 256, L), 256, 0, s>>>(gates, o, n, act, err);
  fused_records_kernel<<<dim3((std::max(max_gates, n) + 255) / 256, L + 1), 256, 0, s>>>(gates, o, n, L, act, rec,
                                                                                        rec_stride(n), count);
  FusedArgs a{X, Z, S, n, stride, nwords, rec, count, rec_stride(n), L};
  const uint32_t records = std::min(max_gates, rec_stride(n));
  const FusedShape f = fused_shape(n, nwords, records, S != nullptr, sms);
  return S ? launch_slices<true>(a, f, records, s) : launch_slices<false>(a, f, records, s);
}

}  // namespace qs
