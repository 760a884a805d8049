// Tableau initialisation and Clifford gate layers on the column-major tableau.
//
// Sec. 4.4 (Alg. 3) applies a window of gates on disjoint qubits to every
// generator row, words of a column in parallel; the update rules are those of
// Sec. 2.4 Eq. 4 (H, P, CX) and, for the rest of the 11-gate set of Sec. 6,
// their compositions (S^dag = S^3, CZ = H_t CX H_t, CY = S_t CX S_t^dag,
// SWAP, ISWAP = CZ, SWAP, S_a, S_b), evaluated in registers so that each gate
// still reads and writes every touched column word once.
//
// GB300 mapping: a thread owns one 128-bit pair of column words (128 rows)
// for a run of gates; its sign contributions stay in registers and leave the
// block as one 64-bit XOR atomic per word per gate group (the paper's
// CollapseSigns tree of Alg. 3 becomes a register XOR). The same kernel, with
// signs compiled out, evolves the Pauli frames of Sec. 5 (Alg. 9 reuses the
// gate kernel on frames).
#include <algorithm>
#include <climits>
#include <vector>

#include "qs_internal.cuh"
#include "qs_lazy.cuh"
#include "qs_rules.cuh"

namespace qs {

__device__ __forceinline__ ulonglong2 ld2(const uint64_t *p) {
  return *reinterpret_cast<const ulonglong2 *>(p);
}
__device__ __forceinline__ void st2(uint64_t *p, ulonglong2 v) {
  *reinterpret_cast<ulonglong2 *>(p) = v;
}

__device__ __forceinline__ bool is_two_qubit(uint32_t t) { return t >= QS_CX && t <= QS_ISWAP; }

// ---------------------------------------------------------------------
// init: D_i = X_i, S_i = Z_i, signs of both rows of qubit i = initstate[i]
// (Sec. 4.1 Alg. 2 InitializeTableau; pattern of Sec. 2.5 Eq. 8).
// X and Z are zeroed beforehand by cudaMemsetAsync.
// ---------------------------------------------------------------------
__global__ void init_diag_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint32_t n,
                                 uint32_t k, uint32_t cs) {
  uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  uint64_t bit = 1ull << (q & 63);
  X[(size_t)q * cs + (q >> 6)] = bit;        // destabilizer row q
  Z[(size_t)q * cs + k + (q >> 6)] = bit;    // stabilizer row 64 k + q
}

// word w of the signs
__device__ __forceinline__ uint64_t init_sign_word(const uint8_t *init, uint32_t n, uint32_t k, uint32_t w) {
  uint64_t v = 0;
  if (init != nullptr && w < 2 * k) {
    uint32_t base = (w < k ? w : w - k) * 64;
    for (uint32_t b = 0; b < 64; ++b) {
      uint32_t i = base + b;
      if (i < n && init[i]) v |= 1ull << b;
    }
  }
  return v;
}

__global__ void init_signs_kernel(uint64_t *__restrict__ S, const uint8_t *__restrict__ init,
                                  uint32_t n, uint32_t k, uint32_t cs) {
  uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w < cs) S[w] = init_sign_word(init, n, k, w);
}

// Small tableaus: everything a reset writes in one launch, where three memsets and
// three kernels are six launches: job of 256 qubits 311 -> 298 us (the call 14 -> 6).
__global__ void __launch_bounds__(256)
init_all_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ S,
                const uint8_t *init, uint32_t n, uint32_t k, uint32_t cs, uint32_t words,
                int64_t *__restrict__ mst, uint32_t *__restrict__ err) {
  chain_start();
  const uint32_t t = blockIdx.x * 256 + threadIdx.x;
  for (uint32_t i = t; i < words; i += gridDim.x * 256) {
    const uint32_t q = i / cs, w = i - q * cs;
    const uint64_t bit = q < n ? 1ull << (q & 63) : 0;
    X[i] = w == (q >> 6) ? bit : 0;
    Z[i] = w == k + (q >> 6) ? bit : 0;
  }
  if (t < cs) S[t] = init_sign_word(init, n, k, t);
  if (t < kMeasStateWords) mst[t] = t == kMsPivot ? LLONG_MAX : 0;
  if (t == 0) *err = 0;
}

bool init_all_fits(const Layout &L) { return (uint64_t)L.ncols * L.cs <= kInitAllWords; }

cudaError_t launch_init_all(const Dev &d, const uint8_t *initstate_dev, cudaStream_t s) {
  const Layout &L = d.L;
  const uint32_t words = L.ncols * L.cs;  // at least cs and kMeasStateWords
  const uint32_t blocks = std::min<uint32_t>((words + 255) / 256, 16u * (uint32_t)d.sms);
  return launch_chained(init_all_kernel, blocks, 256, 0, s, d.X, d.Z, d.S, initstate_dev, L.n, L.k, L.cs, words, d.mst,
                        d.err);
}

cudaError_t launch_init(const Dev &d, const uint8_t *initstate_dev, cudaStream_t s) {
  const Layout &L = d.L;
  size_t colbytes = (size_t)L.ncols * L.cs * sizeof(uint64_t);
  cudaError_t e;
  if ((e = cudaMemsetAsync(d.X, 0, colbytes, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(d.Z, 0, colbytes, s)) != cudaSuccess) return e;
  init_diag_kernel<<<(L.n + 255) / 256, 256, 0, s>>>(d.X, d.Z, L.n, L.k, L.cs);
  init_signs_kernel<<<(L.cs + 255) / 256, 256, 0, s>>>(d.S, initstate_dev, L.n, L.k, L.cs);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------
// gate layer
//   packed[2 g] = type << 24 | q0, packed[2 g + 1] = q1
//   block: P pair-threads x `lanes` gate lanes (P * lanes <= 256);
//   grid.x: gate groups of `lanes * gpl` gates; grid.y: chunks of P pairs.
// On the tableau a thread walks its gates two at a time: both gates' column
// words are loaded before either is stored (the gates of a layer touch
// disjoint columns), which doubles the bytes each thread keeps in flight -- at
// one gate per thread the kernel is bound by memory latency x bytes in flight
// (0.87 of the HBM peak at 180k qubits; 0.97 with two). Frames with short
// columns (many gate lanes per block) keep one gate per thread.
// ---------------------------------------------------------------------
struct GateIn {
  uint32_t type, qa, qb;
  ulonglong2 x1, z1, x2, z2;
};

// Reads the column words the gate of record (w0, qb) needs; false for an
// invalid record (flagged, skipped).
template <bool SIGNS>
__device__ __forceinline__ bool gate_load(GateIn &in, uint32_t w0, uint32_t qb, uint64_t *X, uint64_t *Z, uint32_t n,
                                          uint32_t cs, size_t off, bool flag, uint32_t *err) {
  const uint32_t type = w0 >> 24, qa = w0 & 0xFFFFFFu;
  const bool two = is_two_qubit(type);
  if (qa >= n || type >= QS_NUM_GATE_TYPES || (two && (qb >= n || qb == qa))) {
    if (flag) atomicOr(err, kErrBadGate);
    return false;
  }
  in.type = type;
  in.qa = qa;
  in.qb = qb;
  const uint64_t *xa = X + (size_t)qa * cs + off, *za = Z + (size_t)qa * cs + off;
  const uint64_t *xb = X + (size_t)qb * cs + off, *zb = Z + (size_t)qb * cs + off;
  const ulonglong2 zero = make_ulonglong2(0, 0);
  in.x1 = in.z1 = in.x2 = in.z2 = zero;
  switch (type) {
    case QS_X: if (SIGNS) in.z1 = ld2(za); break;
    case QS_Z: if (SIGNS) in.x1 = ld2(xa); break;
    case QS_Y: if (SIGNS) { in.x1 = ld2(xa); in.z1 = ld2(za); } break;
    case QS_H: case QS_S: case QS_SDG: in.x1 = ld2(xa); in.z1 = ld2(za); break;
    case QS_CX: case QS_CZ: case QS_CY: case QS_SWAP: case QS_ISWAP:
      in.x1 = ld2(xa); in.z1 = ld2(za); in.x2 = ld2(xb); in.z2 = ld2(zb); break;
    default: break;  // QS_I
  }
  return true;
}

// Applies the rules of qs_rules.cuh to both words and stores the columns the
// gate changes.
template <bool SIGNS>
__device__ __forceinline__ void gate_apply(GateIn &in, ulonglong2 &sacc, uint64_t *X, uint64_t *Z,
                                           uint32_t cs, size_t off) {
  uint64_t *xa = X + (size_t)in.qa * cs + off, *za = Z + (size_t)in.qa * cs + off;
  uint64_t *xb = X + (size_t)in.qb * cs + off, *zb = Z + (size_t)in.qb * cs + off;
  uint64_t s0 = 0, s1 = 0;
  uint64_t a0 = in.x1.x, b0 = in.z1.x, c0 = in.x2.x, d0 = in.z2.x;
  uint64_t a1 = in.x1.y, b1 = in.z1.y, c1 = in.x2.y, d1 = in.z2.y;
  rule<SIGNS>(in.type, a0, b0, c0, d0, s0);
  rule<SIGNS>(in.type, a1, b1, c1, d1, s1);
  in.x1 = make_ulonglong2(a0, a1);
  in.z1 = make_ulonglong2(b0, b1);
  in.x2 = make_ulonglong2(c0, c1);
  in.z2 = make_ulonglong2(d0, d1);
  if (SIGNS) { sacc.x ^= s0; sacc.y ^= s1; }
  switch (in.type) {
    case QS_H: st2(xa, in.x1); st2(za, in.z1); break;
    case QS_S: case QS_SDG: st2(za, in.z1); break;
    case QS_CX: st2(xb, in.x2); st2(za, in.z1); break;
    case QS_CZ: st2(za, in.z1); st2(zb, in.z2); break;
    case QS_CY: st2(za, in.z1); st2(xb, in.x2); st2(zb, in.z2); break;
    case QS_SWAP: case QS_ISWAP:
      st2(xa, in.x1); st2(za, in.z1); st2(xb, in.x2); st2(zb, in.z2); break;
    default: break;  // I, X, Y, Z change signs only
  }
}

// One thread block's gates [g0, g1) of a layer; record(g) gives gate g's two words.
template <bool SIGNS, int INFLIGHT, class Record>
__device__ __forceinline__ void gate_block(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ S,
                                           uint32_t n, uint32_t cs, Record record, uint32_t g0, uint32_t g1, uint32_t P,
                                           uint32_t lanes, uint32_t *__restrict__ err) {
  const uint32_t npairs = cs >> 1;
  const uint32_t t = threadIdx.x;
  const uint32_t lane = t / P;
  const uint32_t pair = blockIdx.y * P + (t - lane * P);
  const bool active = pair < npairs;
  ulonglong2 sacc = make_ulonglong2(0, 0);

  if (active) {
    const size_t off = 2 * (size_t)pair;
    const bool flag = pair == 0;
    for (uint32_t g = g0 + lane; g < g1; g += INFLIGHT * lanes) {
      GateIn in[INFLIGHT];
      bool ok[INFLIGHT];
#pragma unroll
      for (int u = 0; u < INFLIGHT; ++u) {
        ok[u] = g + u * lanes < g1;
        if (ok[u]) {
          const uint2 r = record(g + u * lanes);
          ok[u] = gate_load<SIGNS>(in[u], r.x, r.y, X, Z, n, cs, off, flag, err);
        }
      }
#pragma unroll
      for (int u = 0; u < INFLIGHT; ++u)
        if (ok[u]) gate_apply<SIGNS>(in[u], sacc, X, Z, cs, off);
    }
  }
  if (SIGNS) {
    if (lanes > 1) {
      __shared__ ulonglong2 red[256];
      red[t] = sacc;
      __syncthreads();
      if (t < P) {
        for (uint32_t l = 1; l < lanes; ++l) {
          ulonglong2 v = red[l * P + t];
          sacc.x ^= v.x; sacc.y ^= v.y;
        }
      }
    }
    if (active && lane == 0) {
      if (sacc.x) atomicXor(reinterpret_cast<unsigned long long *>(S + 2 * (size_t)pair), sacc.x);
      if (sacc.y) atomicXor(reinterpret_cast<unsigned long long *>(S + 2 * (size_t)pair + 1), sacc.y);
    }
  }
}

template <bool SIGNS, int INFLIGHT>
__global__ void __launch_bounds__(256, INFLIGHT == 2 ? 4 : 6)
gate_layer_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ S,
                  uint32_t n, uint32_t cs, const uint32_t *packed, uint32_t n_gates,
                  uint32_t P, uint32_t lanes, uint32_t gpl, uint32_t *__restrict__ err) {
  chain_start();
  const uint32_t group = lanes * gpl, g0 = blockIdx.x * group;
  gate_block<SIGNS, INFLIGHT>(
      X, Z, S, n, cs, [&](uint32_t g) { return make_uint2(packed[2 * g], packed[2 * g + 1]); }, g0,
      min(g0 + group, n_gates), P, lanes, err);
}

// A host layer whose records ride in the launch itself: one word a gate (type
// << 28 | q0 << 14 | q1, up to 16,384 qubits), MAX of them in the kernel's
// parameters. Staged, a layer is a copy and an event besides the launch, and
// the kernel waits for the copy engine: 8.9 us a layer at 127 qubits from
// back-to-back calls of the Python API, 5.9 with the records in the launch (host
// time, both); 1,000 qubits 10.0 and 6.7. Limits: qubit numbers of 14 bits, and
// beyond 2,048 gates (8 KB) the copy costs no more (4,000 qubits: 14.6 and 14.2).
constexpr uint32_t kParamGroup = 512;  // gates of a block
template <int MAX>
struct ParamLayer {
  uint32_t rec[MAX];
};

template <int MAX>
__global__ void __launch_bounds__(256, 4)
param_layer_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ S, uint32_t n, uint32_t cs,
                   uint32_t n_gates, uint32_t P, uint32_t lanes, uint32_t gpl, uint32_t *__restrict__ err,
                   const __grid_constant__ ParamLayer<MAX> layer) {
  chain_start();
  __shared__ uint32_t rec[kParamGroup];
  const uint32_t group = lanes * gpl, g0 = blockIdx.x * group, g1 = min(g0 + group, n_gates);
  for (uint32_t i = threadIdx.x; g0 + i < g1; i += blockDim.x) rec[i] = layer.rec[g0 + i];
  __syncthreads();
  gate_block<true, 2>(
      X, Z, S, n, cs,
      [&](uint32_t g) {
        const uint32_t r = rec[g - g0];
        return make_uint2(r >> 28 << 24 | (r >> 14 & 0x3FFF), r & 0x3FFF);
      },
      g0, g1, P, lanes, err);
}

struct GateGrid {
  dim3 grid, block;
  uint32_t P, lanes, gpl;
};

// Launch shape: P pair-threads per gate lane (a column chunk of up to 256
// pairs = 32 KB), as many gate lanes as fit 256 threads, and enough gates per
// lane that the grid covers the 152 SMs several times over while each block
// still amortises its sign atomics over several gates.
static GateGrid gate_grid(uint32_t npairs, uint32_t n_gates) {
  GateGrid g;
  g.P = std::min<uint32_t>(npairs, 256);
  g.lanes = std::max<uint32_t>(1, 256 / g.P);
  uint32_t chunks = (npairs + g.P - 1) / g.P;
  uint64_t slots = (n_gates + g.lanes - 1) / g.lanes;
  uint64_t want_blocks = 8ull * 152;
  uint64_t gpl = (slots * chunks + want_blocks - 1) / want_blocks;
  g.gpl = (uint32_t)std::min<uint64_t>(64, std::max<uint64_t>(4, gpl));
  uint64_t group = (uint64_t)g.lanes * g.gpl;
  g.grid = dim3((uint32_t)((n_gates + group - 1) / group), chunks, 1);
  g.block = dim3(g.P * g.lanes, 1, 1);
  return g;
}

cudaError_t launch_gate_layer(const Dev &d, const uint32_t *packed, uint32_t n_gates,
                              cudaStream_t s) {
  if (n_gates == 0) return cudaSuccess;
  GateGrid g = gate_grid(d.L.cs / 2, n_gates);
  return launch_chained(gate_layer_kernel<true, 2>, g.grid, g.block, 0, s, d.X, d.Z, d.S, d.L.n, d.L.cs, packed, n_gates,
                        g.P, g.lanes, g.gpl, d.err);
}

template <int MAX>
static cudaError_t launch_param(const Dev &d, const uint32_t *packed, uint32_t n_gates, cudaStream_t s) {
  ParamLayer<MAX> layer;
  for (uint32_t g = 0; g < n_gates; ++g)
    layer.rec[g] = packed[2 * g] >> 24 << 28 | (packed[2 * g] & 0x3FFF) << 14 | packed[2 * g + 1];
  GateGrid g = gate_grid(d.L.cs / 2, n_gates);
  g.gpl = std::max(1u, std::min(g.gpl, kParamGroup / g.lanes));
  g.grid.x = (n_gates + g.lanes * g.gpl - 1) / (g.lanes * g.gpl);
  return launch_chained(param_layer_kernel<MAX>, g.grid, g.block, 0, s, d.X, d.Z, d.S, d.L.n, d.L.cs, n_gates, g.P,
                        g.lanes, g.gpl, d.err, layer);
}

bool param_layer_fits(uint32_t n, uint32_t n_gates) { return n <= 16384 && n_gates <= 2048; }

cudaError_t launch_param_layer(const Dev &d, const uint32_t *packed, uint32_t n_gates, cudaStream_t s) {
  if (n_gates <= 128) return launch_param<128>(d, packed, n_gates, s);
  if (n_gates <= 512) return launch_param<512>(d, packed, n_gates, s);
  return launch_param<2048>(d, packed, n_gates, s);
}

cudaError_t launch_frame_layer(uint64_t *FX, uint64_t *FZ, uint32_t n, uint32_t fw,
                               const uint32_t *packed, uint32_t n_gates, uint32_t *err,
                               cudaStream_t s) {
  if (n_gates == 0) return cudaSuccess;
  GateGrid g = gate_grid(fw / 2, n_gates);
  if (g.lanes == 1)  // long frame columns (>= 512 shot words): as the tableau, two gates in flight
    return launch_chained(gate_layer_kernel<false, 2>, g.grid, g.block, 0, s, FX, FZ, nullptr, n, fw, packed, n_gates,
                          g.P, g.lanes, g.gpl, err);
  return launch_chained(gate_layer_kernel<false, 1>, g.grid, g.block, 0, s, FX, FZ, nullptr, n, fw, packed, n_gates,
                        g.P, g.lanes, g.gpl, err);
}

// ---------------------------------------------------------------------
// Layers with deferred one-qubit gates (qs_lazy.cuh), one launch per layer:
// launch l applies layer l's two-qubit gates with the pending operations of
// their qubits, and its first blocks turn layer l + 1 into such records (a
// separate launch for that took as long as the layer itself at 15,000 qubits). After the last layer the operations still pending are listed and
// applied the same way.
// At 180,000 qubits (p_cx 0.4) the one-qubit gates are half of a layer's 468,000
// column accesses; deferred, about 245,000 remain: 3.13 -> 1.71 ms a layer; 30,001 qubits 99 -> 58 us.
// ---------------------------------------------------------------------
struct LazyScratch {
  uint2 *rec0, *rec1;  // records of the layers of even and odd launches
  uint32_t *count;     // their number: three counters take turns (read, filled, cleared)
  uint8_t *pend;       // pending operation per qubit
};

struct LazyArgs {
  uint64_t *X, *Z, *S;
  uint32_t cs, n, P, lanes, gx;  // gx: blocks over the layer's gates
  uint32_t prep_blocks;          // first blocks of the grid: the next layer's records
  const uint32_t *next;          // its gates (4-byte aligned), or nullptr: list what is pending
  uint32_t next_gates;
  uint32_t step;
  LazyScratch L;
  uint32_t *err;
};

constexpr uint32_t kLazyPrepBlocks = 256;
constexpr int kPrepGates = 2;  // gates per thread and pass, loaded together

// The next layer's records: one-qubit gates compose into their qubit's pending
// operation, two-qubit gates take both along. One atomic per block and pass.
__device__ __forceinline__ void lazy_prepare(const LazyArgs &a) {
  __shared__ uint32_t s_warp[8], s_base;
  uint2 *rec = a.step & 1 ? a.L.rec0 : a.L.rec1;
  uint32_t *count = a.L.count + (a.step + 1) % 3;
  const uint32_t t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5, warps = (T + 31) >> 5;
  // the warp's last lane and its lanes: the last warp of a block need not be whole
  const uint32_t last = min(31u, T - 1 - 32 * warp), members = 0xffffffffu >> (31 - last);
  const uint32_t items = a.next ? a.next_gates : a.n, pass = T * kPrepGates;
  for (uint32_t b0 = blockIdx.x * pass; b0 < items; b0 += a.prep_blocks * pass) {
    // records, then pending operations, then updates: the qubits of a layer are
    // distinct, but the compiler cannot move a load past a store to pend
    uint2 in[kPrepGates], out[kPrepGates];
    uint32_t pa[kPrepGates], pb[kPrepGates], emit = 0;
    bool ok[kPrepGates];
#pragma unroll
    for (int i = 0; i < kPrepGates; ++i) {
      const uint32_t g = b0 + i * T + t;
      in[i] = make_uint2(QS_I << 24, 0);
      if (g < items) in[i] = a.next ? make_uint2(__ldcg(a.next + 2 * (size_t)g), __ldcg(a.next + 2 * (size_t)g + 1))
                                        : make_uint2(QS_I << 24 | g, 0);
    }
#pragma unroll
    for (int i = 0; i < kPrepGates; ++i) {
      const uint32_t type = in[i].x >> 24, qa = in[i].x & 0xFFFFFFu, qb = in[i].y;
      const bool two = is_two_qubit(type);
      ok[i] = b0 + i * T + t < items;
      if (ok[i] && (qa >= a.n || type >= QS_NUM_GATE_TYPES || (two && (qb >= a.n || qb == qa)))) {
        atomicOr(a.err, kErrBadGate);
        ok[i] = false;
      }
      pa[i] = ok[i] ? a.L.pend[qa] : 0;
      pb[i] = ok[i] && two ? a.L.pend[qb] : 0;
    }
#pragma unroll
    for (int i = 0; i < kPrepGates; ++i) {
      const uint32_t type = in[i].x >> 24, qa = in[i].x & 0xFFFFFFu, qb = in[i].y;
      if (!ok[i]) continue;
      if (is_two_qubit(type)) {
        out[i] = pair_record(type, qa, qb, pa[i], pb[i]);
        if (pa[i]) a.L.pend[qa] = 0;
        if (pb[i]) a.L.pend[qb] = 0;
        emit |= 1u << i;
      } else if (!a.next) {  // after the last layer: what is still pending
        out[i] = single_record(qa, pa[i]);
        emit |= (uint32_t)(pa[i] != 0) << i;
      } else if (type != QS_I) {
        a.L.pend[qa] = (uint8_t)op_then(pa[i], type);
      }
    }
    // inclusive prefix over the warp; its lanes are named, so that they meet here
    // whichever way they went through the branches above
    uint32_t inc = __popc(emit);
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(members, inc, d);
      if (lane >= (uint32_t)d) inc += y;
    }
    if (lane == last) s_warp[warp] = inc;
    __syncthreads();
    if (t == 0) {
      uint32_t sum = 0;
      for (uint32_t w = 0; w < warps; ++w) sum += s_warp[w];
      s_base = sum ? atomicAdd(count, sum) : 0;
    }
    __syncthreads();
    uint32_t at = s_base + inc - __popc(emit);
    for (uint32_t w = 0; w < warp; ++w) at += s_warp[w];
#pragma unroll
    for (int i = 0; i < kPrepGates; ++i)
      if ((emit >> i) & 1) rec[at++] = out[i];
    __syncthreads();  // s_warp is rewritten
  }
}

// one word of a gate: both qubits' pending operations, then the gate
__device__ __forceinline__ void lazy_word(uint32_t type, uint32_t opa, uint32_t opb, unsigned long long &xa_,
                                          unsigned long long &za_, unsigned long long &xb_, unsigned long long &zb_,
                                          unsigned long long &s_) {
  uint64_t xa = xa_, za = za_, xb = xb_, zb = zb_, s = s_;
  if (opa) op_apply<true>(OpMasks(opa), xa, za, s);
  if (opb) op_apply<true>(OpMasks(opb), xb, zb, s);
  if (type) rule<true>(type, xa, za, xb, zb, s);
  xa_ = xa; za_ = za; xb_ = xb; zb_ = zb; s_ = s;
}

// As gate_layer_kernel, two gates in flight a thread; the layer's gates are
// split evenly over gx blocks (their number is known on the device only).
__global__ void __launch_bounds__(256, 4) lazy_layer_kernel(const LazyArgs a) {
  chain_start();
  if (blockIdx.x < a.prep_blocks) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.L.count[(a.step + 2) % 3] = 0;
    lazy_prepare(a);
    return;
  }
  const uint32_t n_gates = a.L.count[a.step % 3];
  const uint2 *recs = a.step & 1 ? a.L.rec1 : a.L.rec0;
  const uint32_t blk = blockIdx.x - a.prep_blocks, bx = blk % a.gx, by = blk / a.gx;
  const uint32_t t = threadIdx.x, lanes = a.lanes, lane = t / a.P, pair = by * a.P + (t - lane * a.P), cs = a.cs;
  uint64_t *X = a.X, *Z = a.Z;
  const bool active = pair < cs >> 1;
  const uint32_t slots = (n_gates + lanes - 1) / lanes, per = (slots + a.gx - 1) / a.gx * lanes;
  const uint32_t g0 = min(n_gates, bx * per), g1 = min(n_gates, g0 + per);
  ulonglong2 sacc = make_ulonglong2(0, 0);
  if (active) {
    const size_t off = 2 * (size_t)pair;
    for (uint32_t g = g0 + lane; g < g1; g += 2 * lanes) {
      uint2 rec[2];
      ulonglong2 xa[2], za[2], xb[2], zb[2];
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (g + u * lanes < g1) {
          rec[u] = recs[g + u * lanes];
          const size_t oa = (size_t)(rec[u].x & 0xFFFFFu) * cs + off;
          xa[u] = ld2(X + oa);
          za[u] = ld2(Z + oa);
          if ((rec[u].x >> 20) & 15) {
            const size_t ob = (size_t)(rec[u].y & 0xFFFFFu) * cs + off;
            xb[u] = ld2(X + ob);
            zb[u] = ld2(Z + ob);
          }
        }
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (g + u * lanes < g1) {
          const uint32_t type = (rec[u].x >> 20) & 15, opa = rec[u].x >> 24, opb = rec[u].y >> 24;
          lazy_word(type, opa, opb, xa[u].x, za[u].x, xb[u].x, zb[u].x, sacc.x);
          lazy_word(type, opa, opb, xa[u].y, za[u].y, xb[u].y, zb[u].y, sacc.y);
          const size_t oa = (size_t)(rec[u].x & 0xFFFFFu) * cs + off;
          if (((kWritesXa >> type) & 1) || op_changes_x(opa)) st2(X + oa, xa[u]);
          if (((kWritesZa >> type) & 1) || op_changes_z(opa)) st2(Z + oa, za[u]);
          if (type) {
            const size_t ob = (size_t)(rec[u].y & 0xFFFFFu) * cs + off;
            if (((kWritesXb >> type) & 1) || op_changes_x(opb)) st2(X + ob, xb[u]);
            if (((kWritesZb >> type) & 1) || op_changes_z(opb)) st2(Z + ob, zb[u]);
          }
        }
    }
  }
  if (lanes > 1) {
    __shared__ ulonglong2 red[256];
    red[t] = sacc;
    __syncthreads();
    if (t < a.P)
      for (uint32_t l = 1; l < lanes; ++l) {
        const ulonglong2 v = red[l * a.P + t];
        sacc.x ^= v.x; sacc.y ^= v.y;
      }
  }
  if (active && lane == 0) {
    if (sacc.x) atomicXor(reinterpret_cast<unsigned long long *>(a.S + 2 * (size_t)pair), sacc.x);
    if (sacc.y) atomicXor(reinterpret_cast<unsigned long long *>(a.S + 2 * (size_t)pair + 1), sacc.y);
  }
}

// n records each: the list of pending operations may hold every qubit
size_t lazy_scratch_bytes(uint32_t n) { return 256 + 2 * (size_t)n * 8 + n; }

cudaError_t launch_lazy_layers(const Dev &d, void *scratch, const uint32_t *packed, const int64_t *ptr, size_t nlayers,
                               cudaStream_t s, int *launches) {
  const uint32_t n = d.L.n, npairs = d.L.cs / 2;
  uint8_t *p = static_cast<uint8_t *>(scratch);
  LazyArgs a{};
  a.X = d.X; a.Z = d.Z; a.S = d.S; a.cs = d.L.cs; a.n = n; a.err = d.err;
  a.L.count = reinterpret_cast<uint32_t *>(p);
  a.L.rec0 = reinterpret_cast<uint2 *>(p + 256);
  a.L.rec1 = a.L.rec0 + n;
  a.L.pend = p + 256 + 2 * (size_t)n * 8;
  cudaError_t e = cudaMemsetAsync(a.L.count, 0, 12, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.L.pend, 0, n, s);
  if (e != cudaSuccess) return e;
  std::vector<size_t> todo;  // nonempty layers
  for (size_t l = 0; l < nlayers; ++l)
    if (ptr[l + 1] > ptr[l]) todo.push_back(l);
  uint64_t gates = 0;  // at most so many records in the launch's layer
  // launch i: layer i - 1 applied (the list of pending operations at the end), layer i prepared
  for (size_t i = 0; i <= todo.size() + 1; ++i) {
    a.step = (uint32_t)i;
    uint64_t next = 0;
    a.next = nullptr;
    if (i < todo.size()) {
      next = (uint64_t)(ptr[todo[i] + 1] - ptr[todo[i]]);
      a.next = packed + 2 * ptr[todo[i]];
    } else if (i == todo.size()) {
      next = n;
    }
    a.next_gates = (uint32_t)next;
    const GateGrid g = gate_grid(npairs, (uint32_t)std::max<uint64_t>(gates, 1));
    const uint32_t threads = g.block.x;
    a.P = g.P;
    a.lanes = g.lanes;
    // one wave of the four resident blocks per SM, eight at the largest sizes:
    // 20,000 qubits 31.4 us a layer (two waves 35.1), 60,000 210 (212), 180,000
    // 1,732 (eight waves 1,710)
    const uint32_t chunks = g.grid.y;
    const uint64_t wave = 4ull * d.sms, blocks_x = (gates * chunks > 1024 * wave ? 8 : 1) * wave / chunks;
    a.gx = i ? (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(blocks_x, (gates + g.lanes - 1) / g.lanes)) : 0;
    a.prep_blocks = (uint32_t)std::min<uint64_t>(kLazyPrepBlocks, (next + threads * kPrepGates - 1) / (threads * kPrepGates));
    const uint32_t blocks = a.prep_blocks + a.gx * chunks;
    if (blocks && (e = launch_chained(lazy_layer_kernel, blocks, threads, 0, s, a)) != cudaSuccess) return e;
    gates = i < todo.size() ? std::min<uint64_t>(next, std::max(1u, n / 2)) : n;
  }
  if (launches) *launches += (int)todo.size() + 2;
  return cudaSuccess;
}

}  // namespace qs
