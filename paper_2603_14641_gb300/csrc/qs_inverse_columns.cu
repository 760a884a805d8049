// Inverse-tableau measurement by columns: a block of up to 64 measurements in
// two launches, on the column-major tableau the gate layers work on.
//
// One measurement of Alg. 1 (qs_inverse.cu) maps every column -- an image's x
// bits s (stabilizer half) and z bits d (destabilizer half) over the n input
// positions -- by CX gates from the pivot p to the targets T (the later
// stabilizers with XS[t][q] = 1), H or H_YZ on p, and X on p if the coin asks
// for it. With the image written i^e X^s Z^d instead of with a sign per Y (e =
// 2 sign + |s & d| mod 4), CX gates change no phase, so the sums over targets
// of Eqs. 9-11 drop out and a step is
//   a = s[p], b = d[p] ^ parity(T & d), s ^= a T, then on (a, b) alone
//   H:    e += 2ab,    (a, b) <- (b, a);
//   H_YZ: e += 2a + b, a ^= b;
//   X:    e += 2b.
// X columns carry S_S, Z columns S_D. Only the measured X columns decide p, T,
// the Y case and the flip, so
//   1. inv_lead_kernel, one block of threads: the measured columns in registers,
//      one measurement after the other. Record, kinds, and the steps as a
//      log; no column is written.
//   2. inv_apply_kernel: the log on every column, a warp per qubit. Rows that
//      are a pivot of the block are kept aside, 64 bits of s and of d per
//      column (log: masks without them, and each mask's bits at them). On
//      the other rows d is constant, so all parities come first (a lane per
//      step, columns broadcast), then the steps on the pivot bits alone (a
//      lane per column), then s with the masks of the steps that had a = 1.
// Measured at 2,000 qubits, 64 measurements: 60 us (55 in a chain of blocks), of which the leading kernel
// 40 (0.6 us a step: shuffle, first target, two ballots, one barrier, three
// redux, all dependent) and the apply kernel 18. Alg. 1 row by row (qs_inverse.cu)
// took 1,720: four dependent launches of 26 us together for each measurement,
// whatever the size. At 16,384 qubits it is 8.7 us a measurement against 46. A
// leading kernel with a warp per column and a redux per column and step took
// 51 us; there the warps of the later columns took the issue slots of the one
// warp that every other waited for.
#include <algorithm>
#include <atomic>

#include "qs_internal.cuh"

namespace qs {

namespace {

constexpr uint32_t kNone = 0xFFFFFFFFu;

// Step log of a block; the masks (kBlock of 32 W words) follow it.
struct InvLog {
  uint64_t at[64];    // targets of step j among the pivot rows: bit i for row p_i
  uint64_t own[64];   // slots i with p_i = p_j
  uint64_t first;     // slots that are the first of their row
  uint64_t yz, flip;  // Y case, X injection
  uint32_t steps, pad;
  uint32_t p[64];
};
static_assert(sizeof(InvLog) % 16 == 0, "masks are read as vectors");

// Words (32 bits) of a column's half in the apply kernel's lanes: 32 W >= 2 k.
template <int W>
constexpr uint32_t kBlock = W <= 8 ? 64 : 32;  // measurements per block

}  // namespace

// lane = measured column (C of them: lane and 32 + lane), warp = V words of
// every column, so that what a step decides per column costs one instruction
// for 32 columns and the targets' words are a broadcast from one lane. With the
// pivot row left in the targets, b is the parity of T & d over all rows: each
// warp publishes its first target row, that row's bits of s and its parities
// before it is known which warp has the pivot, and a step takes one barrier.
template <int V, int C>
__global__ void __launch_bounds__(1024)
inv_lead_kernel(const uint64_t *X, const uint64_t *qsig, uint32_t n, uint32_t k,
                uint32_t cs, uint32_t stride, const uint32_t *qubits, uint32_t count, uint64_t m0,
                uint64_t seed, uint64_t shot, uint8_t *__restrict__ record, uint8_t *__restrict__ kinds,
                InvLog *__restrict__ log, uint32_t *__restrict__ err) {
  extern __shared__ __align__(16) uint32_t masks[];  // stride words per step; at most 64 KB
  __shared__ uint32_t s_q[64], s_coin[64], s_e[64], s_p[64], s_step[64], s_clear[512];
  __shared__ uint4 s_cand[2][32];  // per warp: first target row, the columns' parities
  __shared__ uint2 s_row[2][32];   // the columns' s at that row
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
  chain_start();
  for (uint32_t i = tid; i < 64; i += blockDim.x) {
    s_q[i] = i < count ? qubits[i] : kNone;
    s_p[i] = kNone;
    s_e[i] = s_step[i] = s_coin[i] = 0;
    s_cand[i / 32][i & 31] = make_uint4(kNone, 0, 0, 0);
    if (i < count) {
      s_coin[i] = (uint32_t)(philox4x64_10(m0 + i, shot, 0, 0, seed, kCoinKey).v[0] & 1u);
      if (s_q[i] >= n)
        atomicOr(err, kErrBadQubit);
      else
        s_e[i] = (uint32_t)(qsig[s_q[i] >> 6] >> (s_q[i] & 63) & 1u) << 1;
    }
  }
  for (uint32_t i = tid; i < 512; i += blockDim.x) s_clear[i] = 0;
  __syncthreads();
  uint32_t s[C][V], d[C][V];
  bool valid[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const uint32_t q = s_q[32 * c + lane];
    valid[c] = q < n;
    const uint64_t *col = X + (size_t)(valid[c] ? q : 0) * cs;
    uint32_t y = 0;
#pragma unroll
    for (int i = 0; i < V; i += 2) {
      const uint32_t w = (V * warp + i) / 2;
      const bool in = valid[c] && w < k;
      const uint64_t dv = in ? __ldcg(col + w) : 0, sv = in ? __ldcg(col + k + w) : 0;
      d[c][i] = (uint32_t)dv; d[c][i + 1] = (uint32_t)(dv >> 32);
      s[c][i] = (uint32_t)sv; s[c][i + 1] = (uint32_t)(sv >> 32);
      y += __popcll(sv & dv);
    }
    if (y) atomicAdd(&s_e[32 * c + lane], y);
  }
  __syncthreads();
  // bit lane of a word per column: e mod 4 in two planes, coin, outcome, kind
  uint32_t e0[C], e1[C], coin[C], out[C], kind[C];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const uint32_t e = s_e[32 * c + lane];
    e0[c] = __ballot_sync(0xffffffffu, e & 1);
    e1[c] = __ballot_sync(0xffffffffu, e >> 1 & 1);
    coin[c] = __ballot_sync(0xffffffffu, s_coin[32 * c + lane]);
    out[c] = kind[c] = 0;
  }
  uint32_t steps = 0;
#pragma unroll
  for (int sl = 0; sl < C; ++sl) {
    for (uint32_t l = 0; l < 32 && 32 * sl + l < count; ++l) {
      const uint32_t buf = l & 1;
      // The warp's lanes hold the same t, row, D, ...: all lanes store them, which
      // costs no branch. Registers have no index: select chains.
      uint32_t t[V], row[C], par[C] = {}, tw = 0, iw = 0;
#pragma unroll
      for (int i = 0; i < V; ++i) t[i] = __shfl_sync(0xffffffffu, s[sl][i], l);
#pragma unroll
      for (int c = 0; c < C; ++c) row[c] = 0;
#pragma unroll
      for (int i = V - 1; i >= 0; --i) {
        const bool any = t[i] != 0;
        tw = any ? t[i] : tw;
        iw = any ? i : iw;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          row[c] = any ? s[c][i] : row[c];
          par[c] ^= t[i] & d[c][i];
        }
      }
#pragma unroll
      for (int i = 0; i < V; i += 4)
        *reinterpret_cast<uint4 *>(masks + (size_t)steps * stride + V * warp + i) =
            make_uint4(t[i], t[i + 1], t[i + 2], t[i + 3]);
      const uint32_t bit = tw & (0u - tw);
      uint32_t A[C], D[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        A[c] = __ballot_sync(0xffffffffu, row[c] & bit);
        D[c] = __ballot_sync(0xffffffffu, __popc(par[c]) & 1);
      }
      s_cand[buf][warp] = make_uint4(tw ? (V * warp + iw) * 32 + __ffs(tw) - 1 : kNone, D[0], D[C - 1], 0);
      s_row[buf][warp] = make_uint2(A[0], A[C - 1]);
      __syncthreads();
      const uint4 cand = s_cand[buf][lane];
      const uint32_t p = __reduce_min_sync(0xffffffffu, cand.x);
      D[0] = __reduce_xor_sync(0xffffffffu, cand.y);
      if (C > 1) D[C - 1] = __reduce_xor_sync(0xffffffffu, cand.z);
      if (p == kNone) {  // no x bit in the column: its sign is e / 2
        out[sl] |= e1[sl] & 1u << l;
        continue;
      }
      const uint32_t wp = p / (32 * V);
      const uint2 pr = s_row[buf][wp];
      A[0] = pr.x;
      if (C > 1) A[C - 1] = pr.y;
      // the measured column has a = 1 and no x bit left after H (b = 0, e stays) or
      // H_YZ (b = 1, e = 1 or 3 takes 3 more): its sign is e / 2 from before
      const uint32_t yz = 0u - (D[sl] >> l & 1), flip = 0u - ((e1[sl] ^ coin[sl]) >> l & 1);
      out[sl] |= coin[sl] & 1u << l;
      kind[sl] |= 1u << l;
      s_step[steps] = p | (yz & 1) << 30 | (flip & 1) << 31;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const uint32_t na = D[c] ^ (A[c] & yz), nb = yz ? D[c] : A[c];
        // H: e += 2ab; H_YZ: e += 2a + b; X: e += 2b
        const uint32_t carry = yz ? A[c] ^ (e0[c] & D[c]) : A[c] & D[c];
        e0[c] ^= D[c] & yz;
        e1[c] ^= carry ^ (nb & flip);
        const uint32_t am = 0u - (A[c] >> lane & 1);
#pragma unroll
        for (int i = 0; i < V; ++i) s[c][i] ^= t[i] & am;
        A[c] = na;
        D[c] = nb;
      }
      if (warp == wp) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const uint32_t va = 0u - (A[c] >> lane & 1), vb = 0u - (D[c] >> lane & 1);
#pragma unroll
          for (int i = 0; i < V; ++i) {
            const uint32_t at = iw == (uint32_t)i ? bit : 0;
            s[c][i] = (s[c][i] & ~at) | (va & at);
            d[c][i] = (d[c][i] & ~at) | (vb & at);
          }
        }
      }
      ++steps;
    }
  }
  if (warp == 0)
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (valid[c]) {
        record[m0 + 32 * c + lane] = (uint8_t)(out[c] >> lane & 1);
        kinds[m0 + 32 * c + lane] = (uint8_t)(kind[c] >> lane & 1);
      }
  __syncthreads();
  for (uint32_t j = tid; j < steps; j += blockDim.x) {
    const uint32_t v = s_step[j];
    s_p[j] = v & 0x3FFFFFFFu;
    s_step[j] = v >> 30;
  }
  __syncthreads();
  // each mask's bits at the pivot rows, and the masks without those rows
  for (uint32_t j = tid; j < steps; j += blockDim.x) atomicOr(&s_clear[s_p[j] >> 5], 1u << (s_p[j] & 31));
  const uint32_t p0 = s_p[lane], p1 = s_p[32 + lane];
  for (uint32_t j = warp; j < steps; j += warps) {
    const uint32_t *mask = masks + (size_t)j * stride, pj = s_p[j];
    const uint32_t b0 = p0 != kNone ? mask[p0 >> 5] >> (p0 & 31) & 1 : 0;
    const uint32_t b1 = p1 != kNone ? mask[p1 >> 5] >> (p1 & 31) & 1 : 0;
    const uint64_t at = __ballot_sync(0xffffffffu, b0) | (uint64_t)__ballot_sync(0xffffffffu, b1) << 32;
    const uint64_t own = __ballot_sync(0xffffffffu, p0 == pj) | (uint64_t)__ballot_sync(0xffffffffu, p1 == pj) << 32;
    if (lane == 0) {
      log->at[j] = at & ~own;
      log->own[j] = own;
      log->p[j] = pj;
      if ((own & ((1ull << j) - 1)) == 0) s_step[j] |= 4;
    }
  }
  __syncthreads();
  if (warp == 0) {
    uint64_t bits[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      bits[i] = __ballot_sync(0xffffffffu, s_step[lane] >> i & 1) |
                (uint64_t)__ballot_sync(0xffffffffu, s_step[32 + lane] >> i & 1) << 32;
    if (lane == 0) {
      log->yz = bits[0];
      log->flip = bits[1];
      log->first = bits[2];
      log->steps = steps;
    }
  }
  uint32_t *gm = reinterpret_cast<uint32_t *>(log + 1);
  for (uint32_t i = tid; i < steps * stride; i += blockDim.x) {
    const uint32_t w = i & (stride - 1);  // a power of two
    gm[i] = w < V * warps ? masks[i] & ~s_clear[w] : 0;
  }
}

template <int W>
constexpr uint32_t kApplyWarps = W <= 8 ? 32 : 16;

template <int W>
__global__ void __launch_bounds__(32 * kApplyWarps<W>)
inv_apply_kernel(uint64_t *__restrict__ X, uint64_t *__restrict__ Z, uint64_t *__restrict__ qsig, uint32_t n,
                 uint32_t k, uint32_t cs, uint32_t rs, const InvLog *log) {
  constexpr uint32_t B = kBlock<W>, S = B + 1;  // odd stride: lanes over steps and over words both conflict-free
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ InvLog lg;
  __shared__ uint64_t s_r[2 * kApplyWarps<W>], s_a[2 * kApplyWarps<W>], s_b[2 * kApplyWarps<W>];
  __shared__ uint64_t s_c[2 * kApplyWarps<W>];
  __shared__ uint32_t s_e[2 * kApplyWarps<W>];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
  chain_start();
  const uint32_t steps = log->steps;
  if (steps == 0) return;
  uint32_t *m = sm;                                                 // word w of mask j at w S + j
  uint32_t *colbase = sm + (((size_t)32 * W * S + 3) & ~(size_t)3) + (size_t)warp * 4 * 32 * W;
  const uint32_t *gm = reinterpret_cast<const uint32_t *>(log + 1);
  for (uint32_t i = tid; i < sizeof(InvLog) / 4; i += blockDim.x)
    reinterpret_cast<uint32_t *>(&lg)[i] = __ldcg(reinterpret_cast<const uint32_t *>(log) + i);
#pragma unroll 4
  for (uint32_t i = tid; i < steps * 32 * W; i += blockDim.x) m[(size_t)(i % (32 * W)) * S + i / (32 * W)] = __ldcg(gm + i);
  for (uint32_t i = steps * 32 * W + tid; i < B * 32 * W; i += blockDim.x)
    m[(size_t)(i % (32 * W)) * S + i / (32 * W)] = 0;
  const uint32_t rounds = (n + gridDim.x * warps - 1) / (gridDim.x * warps);
  for (uint32_t round = 0; round < rounds; ++round) {
    const uint32_t q = blockIdx.x + gridDim.x * (warp + warps * round);
    const bool live = q < n;
    uint32_t *g[2] = {reinterpret_cast<uint32_t *>(X + (size_t)(live ? q : 0) * cs),
                      reinterpret_cast<uint32_t *>(Z + (size_t)(live ? q : 0) * cs)};
    // s at colbase + 64 W c, d at 32 W behind it
    uint32_t e0[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t y = 0;
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const uint32_t x = 32 * i + lane;
        const bool in = live && x < 2 * k;
        const uint32_t dv = in ? g[c][x] : 0, sv = in ? g[c][2 * k + x] : 0;
        colbase[64 * W * c + x] = sv;
        colbase[64 * W * c + 32 * W + x] = dv;
        y += __popc(sv & dv);
      }
      e0[c] = __reduce_add_sync(0xffffffffu, y);
    }
    __syncthreads();  // the log and the masks; the columns
    if (live) {
      // parities of the masks with d: lane = step
      uint32_t r[2][2] = {};
      const uint4 *d0 = reinterpret_cast<const uint4 *>(colbase + 32 * W);
      const uint4 *d1 = reinterpret_cast<const uint4 *>(colbase + 96 * W);
#pragma unroll 2
      for (uint32_t w = 0; w < 2 * k; w += 4) {
        const uint4 x0 = d0[w / 4], x1 = d1[w / 4];
        const uint32_t xa[4] = {x0.x, x0.y, x0.z, x0.w}, xb[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t t = m[(size_t)(w + i) * S + lane];
          r[0][0] ^= t & xa[i];
          r[1][0] ^= t & xb[i];
          if (B == 64) {
            const uint32_t u = m[(size_t)(w + i) * S + 32 + lane];
            r[0][1] ^= u & xa[i];
            r[1][1] ^= u & xb[i];
          }
        }
      }
      const uint32_t p0 = lane < steps ? lg.p[lane] : 0, p1 = lane + 32 < steps ? lg.p[lane + 32] : 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const uint32_t *s = colbase + 64 * W * c, *d = s + 32 * W;
        const uint64_t R = __ballot_sync(0xffffffffu, __popc(r[c][0]) & 1) |
                           (uint64_t)__ballot_sync(0xffffffffu, __popc(r[c][1]) & 1) << 32;
        const uint64_t A = __ballot_sync(0xffffffffu, s[p0 >> 5] >> (p0 & 31) & 1) |
                           (uint64_t)__ballot_sync(0xffffffffu, s[p1 >> 5] >> (p1 & 31) & 1) << 32;
        const uint64_t D = __ballot_sync(0xffffffffu, d[p0 >> 5] >> (p0 & 31) & 1) |
                           (uint64_t)__ballot_sync(0xffffffffu, d[p1 >> 5] >> (p1 & 31) & 1) << 32;
        if (lane == 0) {
          s_r[2 * warp + c] = R;
          s_a[2 * warp + c] = A;
          s_b[2 * warp + c] = D;
          s_e[2 * warp + c] = e0[c];
        }
      }
    }
    __syncthreads();
    // the steps on the pivot bits: lane = column; every slot of a row holds its
    // bit, parities count its first slot
    if (tid < 2 * warps) {
      uint64_t A = s_a[tid], D = s_b[tid], used = 0;
      const uint64_t R = s_r[tid], first = lg.first, yzs = lg.yz, flips = lg.flip;
      uint32_t e = s_e[tid];
#pragma unroll 4
      for (uint32_t j = 0; j < steps; ++j) {
        const uint64_t at = lg.at[j], own = lg.own[j], v = at & first & D;
        const uint32_t a = (uint32_t)(A >> j) & 1, b0 = (uint32_t)(D >> j) & 1;
        const uint32_t b = (b0 ^ (uint32_t)(R >> j) ^ __popc((uint32_t)v ^ (uint32_t)(v >> 32))) & 1;
        const bool yz = yzs >> j & 1;
        const uint32_t na = yz ? a ^ b : b, nb = yz ? b : a;
        e += (yz ? 2 * a + b : 2 * (a & b)) + 2 * ((uint32_t)(flips >> j) & nb);
        A ^= (at & (0ull - a)) ^ (own & (0ull - (uint64_t)(a ^ na)));
        D ^= own & (0ull - (uint64_t)(b0 ^ nb));
        used |= (uint64_t)a << j;
      }
      s_a[tid] ^= A;  // what changed
      s_b[tid] ^= D;
      s_c[tid] = used;
      s_e[tid] = e;
    }
    __syncthreads();
    if (live) {
      uint32_t acc[2][W] = {};
      const uint64_t c0 = s_c[2 * warp], c1 = s_c[2 * warp + 1];
#pragma unroll
      for (int h = 0; h < (B == 64 ? 2 : 1); ++h) {
        const uint32_t u0 = (uint32_t)(c0 >> 32 * h), u1 = (uint32_t)(c1 >> 32 * h);
        if (32 * h >= steps) break;
#pragma unroll 8
        for (uint32_t j = 0; j < 32; ++j) {
          const uint32_t m0 = (uint32_t)((int)(u0 << (31 - j)) >> 31), m1 = (uint32_t)((int)(u1 << (31 - j)) >> 31);
#pragma unroll
          for (int i = 0; i < W; ++i) {
            const uint32_t t = m[(size_t)(32 * i + lane) * S + 32 * h + j];
            acc[0][i] ^= t & m0;
            acc[1][i] ^= t & m1;
          }
        }
      }
      const uint64_t first = lg.first;
      const uint32_t f0 = (uint32_t)first >> lane & 1, f1 = (uint32_t)(first >> 32) >> lane & 1;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t *s = colbase + 64 * W * c, *d = s + 32 * W;
#pragma unroll
        for (int i = 0; i < W; ++i) s[32 * i + lane] ^= acc[c][i];
        __syncwarp();
        const uint64_t da = s_a[2 * warp + c], db = s_b[2 * warp + c];
        if (f0) {
          const uint32_t p = lg.p[lane], bit = 1u << (p & 31);
          if ((uint32_t)da >> lane & 1) atomicXor(s + (p >> 5), bit);
          if ((uint32_t)db >> lane & 1) atomicXor(d + (p >> 5), bit);
        }
        if (f1) {
          const uint32_t p = lg.p[32 + lane], bit = 1u << (p & 31);
          if ((uint32_t)(da >> 32) >> lane & 1) atomicXor(s + (p >> 5), bit);
          if ((uint32_t)(db >> 32) >> lane & 1) atomicXor(d + (p >> 5), bit);
        }
        __syncwarp();
        uint32_t y = 0;
#pragma unroll
        for (int i = 0; i < W; ++i) {
          const uint32_t x = 32 * i + lane;
          const uint32_t sv = s[x], dv = d[x];
          y += __popc(sv & dv);
          if (x < 2 * k) {
            g[c][x] = dv;
            g[c][2 * k + x] = sv;
          }
        }
        y = __reduce_add_sync(0xffffffffu, y);
        if (lane == 0 && ((s_e[2 * warp + c] - y) >> 1 & 1))
          atomicXor(reinterpret_cast<unsigned long long *>(qsig + (c ? rs : 0) + (q >> 6)), 1ull << (q & 63));
      }
    }
  }
}

namespace {

template <int W>
cudaError_t measure_columns(const Dev &d, const uint32_t *qubits, uint32_t count, uint64_t m0, qs_key key,
                            cudaStream_t s, int *launches) {
  static std::atomic<uint64_t> attr_set{0};
  const Layout &L = d.L;
  constexpr uint32_t B = kBlock<W>;
  // 64 measurements at 1,000 / 2,000 / 4,000 qubits: 40, 60, 91 us with 4 words a
  // warp, 43, 58, 85 with 8
  constexpr int V = W == 1 ? 4 : W <= 8 ? 8 : 16;
  constexpr auto lead = inv_lead_kernel<V, B / 32>;
  constexpr size_t lead_smem = (size_t)B * 32 * W * 4;
  auto apply_smem = [](uint32_t warps) {
    return ((((size_t)32 * W * (B + 1) + 3) & ~(size_t)3) + (size_t)warps * 4 * 32 * W) * 4;
  };
  cudaError_t e = once_per_device(attr_set, [&]() {
    cudaError_t x = cudaFuncSetAttribute(lead, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    return x != cudaSuccess ? x
                            : cudaFuncSetAttribute(inv_apply_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)apply_smem(kApplyWarps<W>));
  });
  if (e != cudaSuccess) return e;
  InvLog *log = reinterpret_cast<InvLog *>(d.inv_part);
  // a warp per qubit, on all multiprocessors before a second one joins the first
  const uint32_t sms = (uint32_t)d.sms, grid = std::min(L.n, sms), lead_warps = (2 * L.k + V - 1) / V;
  const uint32_t warps = std::max(4u, std::min(kApplyWarps<W>, (L.n + sms - 1) / sms));
  for (uint32_t off = 0; off < count; off += B) {
    const uint32_t c = std::min(B, count - off);
    e = launch_chained(lead, 1, 32 * lead_warps, lead_smem, s, d.X, d.qsig, L.n, L.k, L.cs, 32 * W, qubits + off, c,
                       m0 + off, key.seed, key.shot, d.record, d.kinds, log, d.err);
    if (e == cudaSuccess)
      e = launch_chained(inv_apply_kernel<W>, grid, 32 * warps, apply_smem(warps), s, d.X, d.Z, d.qsig, L.n, L.k, L.cs,
                         L.rs, log);
    if (e != cudaSuccess) return e;
    if (launches) *launches += 2;
  }
  return cudaSuccess;
}

}  // namespace

size_t inv_log_words(const Layout &L) {  // 64-bit words of a block's log
  const uint32_t W = L.n <= 1024 ? 1 : L.n <= 2048 ? 2 : L.n <= 4096 ? 4 : L.n <= 8192 ? 8 : 16;
  return sizeof(InvLog) / 8 + (size_t)(W <= 8 ? 64 : 32) * 16 * W;
}

cudaError_t launch_inv_measure_columns(const Dev &d, const uint32_t *qubits, uint32_t count, uint64_t m0, qs_key key,
                                       cudaStream_t s, int *launches) {
  const uint32_t n = d.L.n;
  if (n <= 1024) return measure_columns<1>(d, qubits, count, m0, key, s, launches);
  if (n <= 2048) return measure_columns<2>(d, qubits, count, m0, key, s, launches);
  if (n <= 4096) return measure_columns<4>(d, qubits, count, m0, key, s, launches);
  if (n <= 8192) return measure_columns<8>(d, qubits, count, m0, key, s, launches);
  return measure_columns<16>(d, qubits, count, m0, key, s, launches);
}

}  // namespace qs
