// Pauli-frame many-shot sampling, Sec. 5 (Alg. 9).
//
// Frames are two bit matrices X~, Z~ stored per qubit as fw 64-bit shot words
// (bit s of word j = shot 64 j + s), the layout of Alg. 9 with one word
// holding 64 shots of one qubit. Gate layers reuse the column-major gate
// kernel with signs compiled out (qs_gates.cu).
//   Randomize (Alg. 9 init):  X~ = 0; Z~[q][j] = word (j & 3) of
//                             Philox(ctr = (0, q, j >> 2, 1), key = (seed, 0xF4A3E)).
//   MeasureSample (Alg. 9):   out[m][j] = X~[q][j] XOR (ref[m] ? ~0 : 0),
//                             Z~[q][j] = word (j & 3) of Philox(ctr = (m + 1, q, j >> 2, 1), ...).
// The XOR with the reference record is the reading of Alg. 9 that makes the
// output a sample (the frames carry flips relative to one valid record).
//   Noise (frames carry error events, Sec. 3): target i of noise op e fires
//                             in shot s iff u < floor(p 2^32); bit 31 - k of u
//                             is bit (s & 63) of word (k & 3) of
//                             Philox(ctr = (e, i, 8 (s >> 6) + (k >> 2), 3),
//                             key = (seed, 0xE5505));
//                             the Pauli of a depolarising channel comes from
//                             word 0 of Philox(ctr = (e, i, s, 4), same key).
#include <algorithm>

#include "qs_internal.cuh"

namespace qs {

// fw is a multiple of 4: one Philox block fills 4 consecutive shot words
__global__ void frame_init_kernel(uint64_t *__restrict__ FZ, uint32_t n, uint32_t fw, uint64_t seed) {
  chain_start();
  const uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t quads = fw >> 2;
  const uint64_t total = (uint64_t)n * quads;
  if (idx >= total) return;
  const uint32_t q = (uint32_t)(idx / quads), j4 = (uint32_t)(idx % quads);
  P4 r = philox4x64_10(0, q, j4, 1, seed, kFrameKey);
  ulonglong2 *p = reinterpret_cast<ulonglong2 *>(FZ + (uint64_t)q * fw + 4ull * j4);
  p[0] = make_ulonglong2(r.v[0], r.v[1]);
  p[1] = make_ulonglong2(r.v[2], r.v[3]);
}

cudaError_t launch_frame_init(uint64_t *FX, uint64_t *FZ, uint32_t n, uint32_t fw, uint64_t seed,
                              cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(FX, 0, (size_t)n * fw * sizeof(uint64_t), s);
  if (e != cudaSuccess) return e;
  const uint64_t total = (uint64_t)n * (fw >> 2);
  return launch_chained(frame_init_kernel, (unsigned)((total + 255) / 256), 256, 0, s, FZ, n, fw, seed);
}

// grid.x over shot-word quads, grid.y over the measurements of the window
// (the qubits of one launch are distinct)
// The measured qubits: a device list, or MAX of them in the launch's parameters.
struct DeviceQubits {
  const uint32_t *q;
  __device__ __forceinline__ uint32_t operator[](uint32_t i) const { return q[i]; }
};
constexpr uint32_t kParamQubits = 1024;
template <int MAX>
struct ParamQubits {
  uint32_t q[MAX];
  __device__ __forceinline__ uint32_t operator[](uint32_t i) const { return q[i]; }
};

template <class Qubits>
__global__ void frame_measure_kernel(const uint64_t *FX, uint64_t *__restrict__ FZ,
                                     uint32_t n, uint32_t fw, const __grid_constant__ Qubits qubits,
                                     uint64_t m0, const uint8_t *ref,
                                     uint64_t *__restrict__ out, uint64_t shots, uint64_t seed,
                                     uint32_t *__restrict__ err) {
  chain_start();
  const uint32_t i = blockIdx.y;
  const uint32_t j4 = blockIdx.x * blockDim.x + threadIdx.x;
  if (j4 >= (fw >> 2)) return;
  const uint32_t q = qubits[i];
  if (q >= n) {
    if (j4 == 0) atomicOr(err, kErrBadQubit);
    return;
  }
  const uint64_t m = m0 + i;
  const uint64_t ow = (shots + 63) / 64;  // output words per measurement
  const uint64_t flip = ref[m] ? ~0ull : 0ull;
  const uint64_t *fx = FX + (uint64_t)q * fw + 4ull * j4;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const uint64_t j = 4ull * j4 + t;
    if (j < ow) {
      uint64_t v = fx[t] ^ flip;
      if (j == ow - 1 && (shots & 63)) v &= (1ull << (shots & 63)) - 1;
      out[m * ow + j] = v;
    }
  }
  P4 r = philox4x64_10(m + 1, q, j4, 1, seed, kFrameKey);
  ulonglong2 *pz = reinterpret_cast<ulonglong2 *>(FZ + (uint64_t)q * fw + 4ull * j4);
  pz[0] = make_ulonglong2(r.v[0], r.v[1]);
  pz[1] = make_ulonglong2(r.v[2], r.v[3]);
}

template <class Qubits>
static cudaError_t frame_measure(uint64_t *FX, uint64_t *FZ, uint32_t n, uint32_t fw, const Qubits &qubits, uint32_t count,
                                 uint64_t m0, const uint8_t *ref, uint64_t *out, uint64_t shots, uint64_t seed,
                                 uint32_t *err, cudaStream_t s) {
  const uint32_t quads = fw >> 2;
  const uint32_t threads = quads < 128 ? ((quads + 31) / 32) * 32 : 128;
  const dim3 grid((quads + threads - 1) / threads, count);
  return launch_chained(frame_measure_kernel<Qubits>, grid, threads, 0, s, FX, FZ, n, fw, qubits, m0, ref, out, shots, seed,
                        err);
}

cudaError_t launch_frame_measure(uint64_t *FX, uint64_t *FZ, uint32_t n, uint32_t fw,
                                 const uint32_t *qubits, uint32_t count, uint64_t m0,
                                 const uint8_t *ref, uint64_t *out, uint64_t shots, uint64_t seed,
                                 uint32_t *err, cudaStream_t s) {
  // grid.y is limited to 65535: split long windows
  cudaError_t e = cudaSuccess;
  for (uint32_t off = 0; off < count && e == cudaSuccess; off += 65535)
    e = frame_measure(FX, FZ, n, fw, DeviceQubits{qubits + off}, std::min(65535u, count - off), m0 + off, ref, out, shots,
                      seed, err, s);
  return e;
}

// Staged, a list is a copy and an event besides the launch, and the kernel waits
// for the copy engine; up to 2,048 qubits they go with one or two launches.
bool param_qubits_fit(uint32_t count) { return count <= 2 * kParamQubits; }

cudaError_t launch_frame_measure_host(uint64_t *FX, uint64_t *FZ, uint32_t n, uint32_t fw, const uint32_t *qubits,
                                      uint32_t count, uint64_t m0, const uint8_t *ref, uint64_t *out, uint64_t shots,
                                      uint64_t seed, uint32_t *err, cudaStream_t s, int *launches) {
  cudaError_t e = cudaSuccess;
  for (uint32_t off = 0; off < count && e == cudaSuccess; off += kParamQubits) {
    const uint32_t c = std::min(kParamQubits, count - off);
    if (c <= 128) {
      ParamQubits<128> list;
      std::copy(qubits + off, qubits + off + c, list.q);
      e = frame_measure(FX, FZ, n, fw, list, c, m0 + off, ref, out, shots, seed, err, s);
    } else {
      ParamQubits<kParamQubits> list;
      std::copy(qubits + off, qubits + off + c, list.q);
      e = frame_measure(FX, FZ, n, fw, list, c, m0 + off, ref, out, shots, seed, err, s);
    }
    ++*launches;
  }
  return e;
}

// Pauli noise channels on the frames (X_ERROR, Y_ERROR, Z_ERROR, DEPOLARIZE1,
// DEPOLARIZE2; frames carry error events, Sec. 3). An item is a (target, shot
// word j). The 64 shots' 32-bit draws u are bit-sliced: bit 31 - k of every
// shot's u sits in random word W_k, so u < thr is decided for all 64 shots at
// once from the most significant bit down, four words (one Philox block) at a
// time, and stops as soon as no shot is undecided. The fire mask applies X/Y/Z
// directly; only the shots that fired draw the Pauli of a depolarising channel.
// Targets of one op are distinct, so every frame word has one writer.
//
// What bounds it is Philox, and what it wastes is lanes: after two blocks (8
// bits) 22 % of the items are undecided and at p = 1e-3 6 % have a shot that
// fired, but nearly every warp has such an item, so warps ran 4.4 blocks per
// item where 2.3 are needed. A block therefore takes 256 items through the first
// two Philox blocks and then deals the undecided ones, and the shots that fired (up
// to kNoiseDense), densely over its threads. (Passing in the first two rounds'
// uniform products and the round keys from the host measured slower, as did a
// four-product 64 x 64 multiply in place of __umul64hi and the low product.) One launch takes up to
// kNoiseGroupMax consecutive ops on distinct qubits (the depolarising ops after
// one layer), so that their latencies overlap. 1,667 + 1,250 targets and 16,384
// shots at p = 1e-3: 49 -> 35 us.

// words of Philox(ctr = (e, i, ctr, tag), key)
__device__ __forceinline__ P4 noise_philox(uint64_t e, uint64_t seed, uint32_t i, uint32_t ctr, int tag) {
  return philox4x64_10(e, i, ctr, tag, seed, kNoiseKey);
}

constexpr int kNoiseThreads = 128, kNoiseItems = 2 * kNoiseThreads;  // items per block
// Fired shots of a block beyond which a thread draws those of its own two items, side
// by side, instead of having all dealt out: dealing costs a search, a selection and
// shared atomics a draw, which pay where lanes would wait for a few busy ones. 1,000
// qubits x 20,000 shots, ten layers, dealt / own: p = 0.02 320 / 388 us, 0.1 575 / 642, 0.2
// 881 / 807, 0.5 1,610 / 1,423, 1 3,273 / 1,905 (dealt with the bits of a shot word counted
// off one by one 5,090, a thread per item throughout 1,885).
constexpr uint32_t kNoiseDense = 16 * kNoiseItems;

// one more Philox block of an item's draws: 4 bits of u from bit 31 - 4 t down
__device__ __forceinline__ void noise_bits(uint64_t e, uint64_t seed, uint32_t thr, uint32_t i, uint32_t j, int t,
                                           uint64_t &fire, uint64_t &undecided) {
  const P4 r = noise_philox(e, seed, i, 8 * j + t, 3);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint64_t w = r.v[q];
    if ((thr >> (31 - (4 * t + q))) & 1u) {
      fire |= undecided & ~w;  // u has 0 where thr has 1: u < thr
      undecided &= w;
    } else {
      undecided &= ~w;  // u has 1 where thr has 0: u > thr
    }
  }
}

// index of bit r (from 0) among the bits of m
__device__ __forceinline__ uint32_t nth_bit(uint64_t m, uint32_t r) {
  uint32_t w = (uint32_t)m, at = 0, c = __popc(w);
  if (r >= c) { r -= c; w = (uint32_t)(m >> 32); at = 32; }
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) {
    c = __popc(w & ((1u << h) - 1));
    if (r >= c) { r -= c; w >>= h; at += h; }
  }
  return at;
}

// the Pauli of a shot that fired: 0 I, 1 X, 2 Y, 3 Z on the first and second target
__device__ __forceinline__ void noise_pauli(int kind, uint64_t v, uint32_t &pa, uint32_t &pb) {
  pb = 0;
  if (kind == QS_NOISE_DEPOLARIZE1) {
    pa = 1 + (uint32_t)__umul64hi(v, 3);
  } else {
    const uint32_t idx = 1 + (uint32_t)__umul64hi(v, 15);
    pa = idx >> 2;
    pb = idx & 3;
  }
}

// one op of a launch; its blocks follow those of the ops before it
struct NoiseLaunch {
  const uint32_t *targets;
  uint64_t items, thr, e;
  uint32_t i0, first_block;
  int kind;
};
struct NoiseGroup {
  NoiseLaunch op[kNoiseGroupMax];
  uint64_t seed;
  int ops;
};

// DENSE: some op's probability (above 0.2: 12.8 fired shots an item) may let blocks have
// more than kNoiseDense of them. Without that part the kernel needs 62 registers
// instead of 72: 4,999 qubits x 16,384 shots at p = 1e-3 2,079 -> 2,029 us.
template <bool DENSE>
__global__ void __launch_bounds__(kNoiseThreads)
frame_noise_kernel(uint64_t *__restrict__ FX, uint64_t *__restrict__ FZ, uint32_t fw, uint32_t ow,
                   const __grid_constant__ NoiseGroup G) {
  chain_start();
  int o = 0;
  while (o + 1 < G.ops && blockIdx.x >= G.op[o + 1].first_block) ++o;
  const uint32_t *targets = G.op[o].targets;
  const uint64_t items = G.op[o].items, thr = G.op[o].thr;
  const uint32_t i0 = G.op[o].i0, blk = blockIdx.x - G.op[o].first_block;
  const int kind = G.op[o].kind;
  const uint64_t e = G.op[o].e, seed = G.seed;
  __shared__ uint64_t s_fire[kNoiseItems], s_und[kNoiseItems];
  __shared__ __align__(16) uint32_t s_pauli[kNoiseItems][8];  // x, z of the first and second target, as halves
  __shared__ uint32_t s_first[kNoiseItems];     // draws before an item
  __shared__ uint16_t s_queue[kNoiseItems];
  __shared__ uint32_t s_n, s_warp[kNoiseThreads / 32];
  const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint64_t base = (uint64_t)blk * kNoiseItems;
  const uint32_t n = (uint32_t)(items - base < kNoiseItems ? items - base : kNoiseItems);
  const uint32_t b_i = (uint32_t)(base / ow), b_j = (uint32_t)(base % ow);  // uniform
  // item x of the block: target index and shot word (x < 256: one 32-bit division)
  auto place = [&](uint32_t x, uint32_t &i, uint32_t &j) {
    const uint32_t d = (b_j + x) / ow;
    i = b_i + d;
    j = b_j + x - d * ow;
  };
  const bool draws = kind == QS_NOISE_DEPOLARIZE1 || kind == QS_NOISE_DEPOLARIZE2;
  bool dense = false;
  if (t == 0) s_n = 0;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kNoiseItems / kNoiseThreads; ++u) {
    const uint32_t x = u * kNoiseThreads + t;
    uint64_t fire = 0, und = 0;
    if (x < n) {
      if (thr >> 32) {
        fire = ~0ull;  // p >= 1
      } else {
        uint32_t i, j;
        place(x, i, j);
        und = ~0ull;
        noise_bits(e, seed, (uint32_t)thr, i0 + i, j, 0, fire, und);
        noise_bits(e, seed, (uint32_t)thr, i0 + i, j, 1, fire, und);
      }
    }
    s_fire[x] = fire;
    s_und[x] = und;
    const uint32_t ball = __ballot_sync(0xffffffffu, und != 0);
    uint32_t at = 0;
    if (lane == 0 && ball) at = atomicAdd(&s_n, (uint32_t)__popc(ball));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (und) s_queue[at + __popc(ball & ((1u << lane) - 1))] = (uint16_t)x;
  }
  __syncthreads();
  for (uint32_t k = t; k < s_n; k += kNoiseThreads) {
    const uint32_t x = s_queue[k];
    uint32_t i, j;
    place(x, i, j);
    uint64_t fire = s_fire[x], und = s_und[x];
    for (int b = 2; b < 8 && und; ++b) noise_bits(e, seed, (uint32_t)thr, i0 + i, j, b, fire, und);
    s_fire[x] = fire;  // shots still undecided after 32 bits have u == thr: no fire
  }
  __syncthreads();
  if (draws) {
    // the shots that fired, numbered through the block's items
    const uint32_t f0 = __popcll(s_fire[2 * t]), f1 = __popcll(s_fire[2 * t + 1]);
    uint32_t inc = f0 + f1;
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= (uint32_t)d) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    uint32_t before = inc - f0 - f1, total = 0;
    for (uint32_t w = 0; w < kNoiseThreads / 32; ++w) {
      if (w < warp) before += s_warp[w];
      total += s_warp[w];
    }
    s_first[2 * t] = before;
    s_first[2 * t + 1] = before + f0;
    dense = DENSE && total > kNoiseDense;
    for (uint32_t k = t; k < kNoiseItems * 8 && !dense; k += kNoiseThreads) s_pauli[k >> 3][k & 7] = 0;
    __syncthreads();
    for (uint32_t k = t; k < total && !dense; k += kNoiseThreads) {
      uint32_t lo = 0, hi = kNoiseItems;  // last item with first <= k
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (s_first[mid] <= k) lo = mid; else hi = mid;
      }
      const uint32_t b = nth_bit(s_fire[lo], k - s_first[lo]);
      uint32_t i, j, pa, pb;
      place(lo, i, j);
      noise_pauli(kind, noise_philox(e, seed, i0 + i, 64 * j + b, 4).v[0], pa, pb);
      uint32_t *acc = s_pauli[lo] + (b >> 5);
      const uint32_t bit = 1u << (b & 31);
      if (pa == 1 || pa == 2) atomicOr(acc, bit);
      if (pa >= 2) atomicOr(acc + 2, bit);
      if (pb == 1 || pb == 2) atomicOr(acc + 4, bit);
      if (pb >= 2) atomicOr(acc + 6, bit);
    }
    __syncthreads();
  }
  if (DENSE && dense) {
    // a thread's two items side by side: two Philox chains in flight
    uint64_t m[2], acc[2][4] = {};
    uint32_t i[2], j[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t x = u * kNoiseThreads + t;
      m[u] = x < n ? s_fire[x] : 0;
      place(x, i[u], j[u]);
    }
    while (m[0] | m[1]) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t b = (uint32_t)__ffsll((long long)m[u]) - 1;
        const uint64_t bit = m[u] & (0 - m[u]);  // 0 for an item that is done
        uint32_t pa, pb;
        noise_pauli(kind, noise_philox(e, seed, i0 + i[u], 64 * j[u] + b, 4).v[0], pa, pb);
        if (pa == 1 || pa == 2) acc[u][0] |= bit;
        if (pa >= 2) acc[u][1] |= bit;
        if (pb == 1 || pb == 2) acc[u][2] |= bit;
        if (pb >= 2) acc[u][3] |= bit;
        m[u] ^= bit;
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint64_t *pauli = reinterpret_cast<uint64_t *>(s_pauli[u * kNoiseThreads + t]);
#pragma unroll
      for (int v = 0; v < 4; ++v) pauli[v] = acc[u][v];
    }
  }
  for (uint32_t x = t; x < n; x += kNoiseThreads) {
    const uint64_t fire = s_fire[x];
    if (!fire) continue;
    uint32_t i, j;
    place(x, i, j);
    uint64_t ax = 0, az = 0, bx = 0, bz = 0;
    if (draws) {
      const uint64_t *acc = reinterpret_cast<const uint64_t *>(s_pauli[x]);
      ax = acc[0]; az = acc[1]; bx = acc[2]; bz = acc[3];
    } else {
      if (kind != QS_NOISE_Z) ax = fire;
      if (kind != QS_NOISE_X) az = fire;
    }
    const uint64_t qa = kind == QS_NOISE_DEPOLARIZE2 ? targets[2 * (uint64_t)i] : targets[i];
    if (ax) FX[qa * fw + j] ^= ax;
    if (az) FZ[qa * fw + j] ^= az;
    if (kind == QS_NOISE_DEPOLARIZE2) {
      const uint64_t qb = targets[2 * (uint64_t)i + 1];
      if (bx) FX[qb * fw + j] ^= bx;
      if (bz) FZ[qb * fw + j] ^= bz;
    }
  }
}

cudaError_t launch_frame_noise(uint64_t *FX, uint64_t *FZ, uint32_t fw, uint32_t ow, const NoiseOp *ops, int n,
                               uint64_t seed, cudaStream_t s, int *launches) {
  NoiseGroup G;
  G.ops = 0;
  G.seed = seed;
  uint64_t blocks = 0;
  bool dense = false;
  for (int i = 0; i < n; ++i) {
    const NoiseOp &x = ops[i];
    dense |= x.thr > (1ull << 32) / 5;
    if (x.count == 0 || ow == 0 || x.thr == 0) continue;  // never fires
    if (G.ops == kNoiseGroupMax) return cudaErrorInvalidValue;
    NoiseLaunch &l = G.op[G.ops++];
    l.targets = x.targets;
    l.items = (uint64_t)x.count * ow;
    l.thr = x.thr;
    l.i0 = x.i0;
    l.kind = x.kind;
    l.first_block = (uint32_t)blocks;
    l.e = x.e;
    blocks += (l.items + kNoiseItems - 1) / kNoiseItems;
    if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
  }
  if (G.ops == 0) return cudaSuccess;
  if (launches) *launches += 1;
  return launch_chained(dense ? frame_noise_kernel<true> : frame_noise_kernel<false>, (unsigned)blocks, kNoiseThreads, 0,
                        s, FX, FZ, fw, ow, G);
}

}  // namespace qs
