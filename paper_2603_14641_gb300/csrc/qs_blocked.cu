// Blocked CHP measurement: up to 64 consecutive Z-measurements per pass over
// the row-major tableau, with exactly the result of measuring them one by one.
//
// Sequential CHP (Sec. 2.5) only ever (a) left-multiplies target rows by the
// current pivot row, (b) copies the pivot row into its destabilizer partner and
// (c) replaces the pivot row by (-1)^b Z_q. Which rows are pivots and targets
// depends only on the x bits of the measured columns, so the block is run in
// three parts:
//  1. symbolic pass: every packed row r carries C_r = its x bits at the block's
//     qubits q_0..q_{B-1} (one 64-bit word). Step j picks the pivot (smallest
//     stabilizer with bit j set), XORs the pivot's C into the targets and records
//     in M_r which steps targeted r; the destabilizer partner gets the pivot's C
//     (base = step j, M reset), the pivot row is marked. A step without a pivot
//     has a deterministic outcome and changes nothing.
//  2. pivot rows: V_j = (V_{j'} ... over the steps j' that targeted row p_j, in
//     order) * original row p_j, built word-parallel; their signs follow from
//     the phase of a product of Paulis,
//       i^(2 sum r + sum |x_a & z_a| + 2 sum_{a<b} z_a . x_b - |X & Z|),
//     whose cross term is GF(2)-bilinear, so per-word popcounts summed over the
//     row (|x & z| of each V, of each original pivot row, parities
//     G[s][t] = z_{V_s} . x_{V_t}) are enough.
//  3. one streaming pass: row r becomes (prod over s in M_r of V_s) * base_r,
//     base_r = its original value or V_j if it was replaced at step j; the XOR
//     accumulation reads the V words of a column chunk from shared memory, the
//     phase uses the same product formula with cross term
//     z_acc . x_base + sum_{s>t in M_r} G[s][t]. Pivot rows become +-Z_q.
// Per block the tableau is read and written once instead of once per
// measurement (the paper measures one qubit at a time, Alg. 2).
//
// Deterministic outcomes of a window are evaluated together after its last
// block: measurements of one window commute, so (-1)^m Z_q stays in the
// stabilizer group, and with it its value, until the window ends.
//
// Launches: a window is a memset, blk_front, then per block blk_middle,
// blk_apply and blk_front (which signs block b's rows and starts block b + 1),
// then blk_det. The serial parts run in the block of a grid that arrives last,
// so the host neither waits nor reads anything back: 3 launches per block where
// a launch per part took 9 and a wait per round. 64 measurements of a dense
// 10,000-qubit state: 172 -> 103 us; 3,000 measurements of a shallow 1,500-qubit
// state, 2,456 of them deterministic (measured one by one before): 30.3 -> 2.4 ms.
#include <algorithm>
#include <climits>

#include "qs_internal.cuh"

namespace qs {

constexpr int32_t kBaseOrig = -1;
constexpr int32_t kBasePivot = 1000;  // base = kBasePivot + j: pivot row of step j
constexpr int kCW = 32;               // column words per phase-3 chunk
constexpr int64_t kBlkNone = LLONG_MAX;

// state of one block (two of them alternate: blk_front signs block b's rows
// with one while its symbolic pass fills the other for block b + 1)
struct BlkState {
  int64_t slot[3];     // pivot search results, rotating (step-by-step symbolic pass)
  uint32_t ntouched;   // rows the block changes (entries of the apply pass's row list)
  uint32_t pad;
  int64_t piv[64];     // pivot row of each step, or kBlkNone (deterministic)
  uint64_t mpiv[64];   // steps that targeted the pivot row before it became pivot
  uint64_t cpiv[64];   // C of the pivot row at its step (0: deterministic)
  uint64_t E[64];      // V_j = product of the original pivot rows of the steps in E_j
  uint64_t lin[64];    // M_r = XOR of lin[t] over the bits t of C_r (rows never replaced)
  int32_t A[64];       // |x_V & z_V| mod 4 (summed over words)
  int32_t B0[64];      // |x & z| of the original pivot row
  int32_t Cp[64];      // parity of (z_V ^ z_orig) . x_orig
  int32_t rV[64];      // sign bit of V_j
  uint64_t G[64];      // G[s] bit t = parity(z_{V_s} . x_{V_t})
};

constexpr uint32_t kDetChunks = 512;  // 32-word column chunks of the largest row (n = 2^20)

// state of one window; zeroed before its first block together with the
// accumulators behind it
struct BlkWindow {
  uint32_t front_arrived, middle_arrived, ndet, pad;
  uint32_t det_chunk[kDetChunks];  // row ranges of blk_det that have arrived, per column chunk
  BlkState st[2];
};

__device__ __forceinline__ int m4(int v) { return ((v % 4) + 4) % 4; }

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// The x bits of one row at a run of measured qubits. Measured qubits are cut
// into runs of consecutive ones inside a word, so that an ascending list takes
// one load, shift and mask per 64 qubits.
struct ColRuns {
  uint32_t n;
  uint32_t word[64];
  uint64_t mask[64];
  uint8_t shift[64], pos[64];
};

// fills R from qubits[0..B); called by the first 64 threads of a block, which
// then synchronises. Out-of-range qubits belong to no run (their bits are 0).
__device__ __forceinline__ void build_runs(ColRuns &R, const uint32_t *qubits, int B, uint32_t n) {
  __shared__ uint32_t s_start[2], s_ok[2];
  const int t = threadIdx.x;
  const uint32_t q = t < B ? qubits[t] : 0xFFFFFFFFu;
  const uint32_t before = (t > 0 && t - 1 < B) ? qubits[t - 1] : 0xFFFFFFFFu;
  const bool ok = q < n;
  const bool start = ok && !(before < n && q == before + 1 && (q & 63) != 0);
  const uint32_t bs = __ballot_sync(0xffffffffu, start), bo = __ballot_sync(0xffffffffu, ok);
  if ((t & 31) == 0) { s_start[t >> 5] = bs; s_ok[t >> 5] = bo; }
  asm volatile("bar.sync 1, 64;" ::: "memory");
  const uint64_t st = ((uint64_t)s_start[1] << 32) | s_start[0], okm = ((uint64_t)s_ok[1] << 32) | s_ok[0];
  if (start) {
    const int i = __popcll(st & ((1ull << t) - 1));
    const uint64_t stop = (st | ~okm) & ~((2ull << t) - 1);  // the next start or invalid entry ends the run
    const int len = (stop ? __ffsll((long long)stop) - 1 : 64) - t;
    R.word[i] = q >> 6;
    R.shift[i] = (uint8_t)(q & 63);
    R.pos[i] = (uint8_t)t;
    R.mask[i] = len >= 64 ? ~0ull : (1ull << len) - 1;
  }
  if (t == 0) R.n = (uint32_t)__popcll(st);
}

// the runs' bits of row r, four words in flight
__device__ __forceinline__ uint64_t gather_runs(const ColRuns &R, const uint64_t *row) {
  uint64_t c = 0;
  for (uint32_t i = 0; i < R.n; i += 4) {
    uint64_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = i + u < R.n ? row[R.word[i + u]] : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u < R.n) c |= ((w[u] >> R.shift[i + u]) & R.mask[i + u]) << R.pos[i + u];
  }
  return c;
}

// E_j = {j} xor (xor of E_s over the steps s that targeted p_j): thread t of
// the first 64 keeps column t of E (bit s = whether t is in E_s), so a step is
// one parity per thread and no exchange; the ballots are the rows.
__device__ __forceinline__ void build_products(const uint64_t *mpiv, const int64_t *piv, int B, uint64_t *E) {
  const int t = threadIdx.x;
  uint64_t col = 0;
  for (int j = 0; j < 64; ++j) {
    uint32_t bit = 0;
    if (j < B && piv[j] != kBlkNone) bit = (uint32_t)(__popcll(col & mpiv[j]) & 1) ^ (t == j ? 1u : 0u);
    const uint32_t row = __ballot_sync(0xffffffffu, bit);
    col |= (uint64_t)bit << j;
    if ((t & 31) == 0) reinterpret_cast<uint32_t *>(&E[j])[t >> 5] = row;
  }
}

// ---------------------------------------------------------------------------
// blk_front: signs of the previous block's rows, C of the next block's, and in
// the last block to arrive the next block's symbolic pass
// ---------------------------------------------------------------------------
struct FrontArgs {
  const uint64_t *RX;
  uint64_t *S;
  uint64_t nrows;
  uint32_t rs, n, k, chunks;
  const uint32_t *window;       // measured qubits of the window
  uint32_t i0, B;               // next block: first measurement and count (0: none)
  uint32_t prev_i0, prev_B;     // previous block (0: none)
  int cur;                      // state of the next block; the previous block's is the other
  int lazy;                     // run the symbolic pass here (else step by step)
  uint64_t *C, *listC;          // C of every row; nonzero stabilizer rows of each 256-row range: C,
  uint32_t *listRow;            // their rows,
  uint32_t *cnt, *done;         // their number, the steps replayed on them
  uint64_t *orC;                // and the OR of their C
  uint64_t *M;
  int32_t *base;
  const int32_t *Tp;
  BlkWindow *win;
  uint32_t *det;                // window positions of deterministic outcomes
  uint64_t m0, seed, shot;
  uint8_t *record, *kinds;
  uint32_t *err;
};

// per row: new sign from the accumulated terms; pivot rows get their coin; record
__device__ __forceinline__ void sign_rows(const FrontArgs &a, uint64_t r) {
  __shared__ int sw[64];          // 2 rV_s + A_s of each step
  __shared__ uint64_t sG[64];     // G rows
  __shared__ uint32_t s_det[2];
  const BlkState &st = a.win->st[a.cur ^ 1];
  const uint64_t m0 = a.m0 + a.prev_i0;  // record index of the block's first measurement
  const int t = threadIdx.x, B = (int)a.prev_B;
  if (t < 64) {
    sw[t] = 2 * st.rV[t] + st.A[t];
    sG[t] = st.G[t];
  }
  __syncthreads();
  if (blockIdx.x == 0 && t < 64) {
    const bool in = t < B, prob = in && st.piv[t] != kBlkNone;
    if (in) {
      a.record[m0 + t] = prob ? (uint8_t)(philox4x64_10(m0 + t, a.shot, 0, 0, a.seed, kCoinKey).v[0] & 1u) : 0;
      a.kinds[m0 + t] = prob;
    }
    const bool det = in && !prob && a.window[a.prev_i0 + t] < a.n;
    const uint32_t ball = __ballot_sync(0xffffffffu, det);
    if ((t & 31) == 0) s_det[t >> 5] = ball;
    const uint32_t first = a.win->ndet;
    asm volatile("bar.sync 1, 64;" ::: "memory");
    if (det) a.det[first + (t >= 32 ? __popc(s_det[0]) : 0) + __popc(ball & ((1u << (t & 31)) - 1))] = a.prev_i0 + t;
    if (t == 0) a.win->ndet = first + __popc(s_det[0]) + __popc(s_det[1]);
  }
  uint64_t delta = 0;
  if (r < a.nrows) {
    const int32_t b = a.base[r];
    const uint64_t sr = a.M[r];
    const uint64_t old = (a.S[r >> 6] >> (r & 63)) & 1u;
    uint64_t nb = old;
    if (b >= kBasePivot) {
      nb = philox4x64_10(m0 + (b - kBasePivot), a.shot, 0, 0, a.seed, kCoinKey).v[0] & 1u;
    } else if (b != kBaseOrig || sr != 0) {
      const int rb = (b == kBaseOrig) ? (int)old : st.rV[b];
      int e = 2 * rb, csum = 0;
#pragma unroll 4
      for (uint32_t ch = 0; ch < a.chunks; ++ch) {
        const int32_t v = a.Tp[(uint64_t)ch * a.nrows + r];
        e += v >> 1;  // arithmetic shift: t
        csum ^= v & 1;
      }
      e += 2 * csum;
      // + sum over s in M_r of (2 rV_s + A_s) + 2 sum over s > t in M_r of G[s] bit t
      uint64_t mm = sr;
      while (mm) {
        const int s = __ffsll((long long)mm) - 1;
        mm &= mm - 1;
        e += sw[s] + 2 * (__popcll(sG[s] & sr & ((1ull << s) - 1)) & 1);
      }
      e = m4(e);
      if (e & 1) atomicOr(a.err, kErrOddPhase);
      nb = (uint64_t)(e >> 1);
    }
    delta = (nb ^ old) << (r & 63);
  }
  // fold the sign changes of the 32 rows of this warp into one atomic
  for (int o = 16; o > 0; o >>= 1) delta |= __shfl_xor_sync(0xffffffffu, delta, o);
  if ((threadIdx.x & 31) == 0 && r < a.nrows && delta)
    atomicXor(reinterpret_cast<unsigned long long *>(&a.S[r >> 6]), delta);
}

// Symbolic pass. Only the pivot sequence (p_j, v_j = C_{p_j} at step j) has to
// be found in order, and the pivot of step j is the first stabilizer row whose
// current C has bit j. Rows with C = 0 never take part, and in any state the
// pivots come from the first nonzero rows, so the first 1,024 of those are held
// by the block's 8 warps, 128 rows each, transposed: lane t of a warp holds the
// warp's rows' bits at steps t and t + 32 as four words each. A step is then a
// broadcast of column j, a search for its first bit and one masked XOR into the
// columns v_j has; the pivot row clears itself (its C is v_j). Warp 0 runs alone
// while its rows hold a pivot (no barriers: 64 steps of a dense state take about
// 5 us); at its first miss the other warps replay the steps so far on their
// rows and all eight go on in step. Nonzero rows beyond the first 1,024 are only
// looked at when those have no pivot for a step: range by range of 256 rows,
// skipping a range when an upper bound on the OR of its C rules the step's bit
// out (exact when the range was last replayed, then grown by v_s for every step
// s whose bit the bound has).
constexpr int kGroup = 1024;

struct Tile {  // one warp's 128 rows: columns lane and lane + 32
  uint32_t lo[4], hi[4];
};

// 32 x 32 bit transpose over the warp: out[lane t] bit r = in[lane r] bit t
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const uint32_t low = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & ~low) | ((y & ~low) >> j)) : ((x & low) | ((y & low) << j));
  }
  return x;
}

__device__ __forceinline__ void tile_column(const Tile &T, int j, uint32_t (&w)[4]) {
#pragma unroll
  for (int m = 0; m < 4; ++m) w[m] = __shfl_sync(0xffffffffu, j < 32 ? T.lo[m] : T.hi[m], j & 31);
}

// first row with a bit in column w (-1: none)
__device__ __forceinline__ int tile_first(const uint32_t (&w)[4]) {
  int p = -1;
#pragma unroll
  for (int m = 3; m >= 0; --m)
    if (w[m]) p = 32 * m + __ffs(w[m]) - 1;
  return p;
}

// C of row p of the tile (warp-uniform p)
__device__ __forceinline__ uint64_t tile_row(const Tile &T, int p) {
  const int m = p >> 5, b = p & 31;
  uint32_t l = T.lo[0], h = T.hi[0];
#pragma unroll
  for (int i = 1; i < 4; ++i)
    if (m == i) { l = T.lo[i]; h = T.hi[i]; }
  const uint32_t vl = __ballot_sync(0xffffffffu, (l >> b) & 1u), vh = __ballot_sync(0xffffffffu, (h >> b) & 1u);
  return ((uint64_t)vh << 32) | vl;
}

// rows with bit j (w) take v
__device__ __forceinline__ void tile_apply(Tile &T, const uint32_t (&w)[4], uint64_t v, int lane) {
  const uint32_t ml = 0u - (uint32_t)((v >> lane) & 1u), mh = 0u - (uint32_t)((v >> (lane + 32)) & 1u);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    T.lo[m] ^= w[m] & ml;
    T.hi[m] ^= w[m] & mh;
  }
}

__device__ __forceinline__ uint64_t lazy_bound(uint64_t u, int a, int j, const uint64_t *v) {
  for (int s = a; s < j; ++s)
    if ((u >> s) & 1ull) u |= v[s];
  return u;
}

struct SymbolicShared {
  uint64_t c[kGroup];          // C of the first nonzero rows
  uint32_t row[kGroup];
  uint64_t v[64];              // C of each step's pivot (0: none)
  int64_t piv[64];
  uint64_t mpiv[64], E[64];
  uint64_t cand_v[2][8], wor[8];
  int cand[2][8];
  uint32_t sum[8], flags[8];
  int j0;
  int found;
  uint64_t found_v;
  int64_t found_row;
};

// pivot of step j among the nonzero rows past the first kGroup (all 256
// threads; off[w] = nonzero rows before range w); leaves found_* in sh
__device__ void search_rest(const FrontArgs &a, SymbolicShared &sh, const uint32_t *off, uint32_t nwin, int j) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  __syncthreads();
  if (t == 0) sh.found = 0;
  for (uint32_t w0 = 0; w0 < nwin; w0 += 256) {
    const uint32_t w = w0 + t;
    bool may = false;
    if (w < nwin) {
      const uint32_t c = __ldcg(a.cnt + w);
      may = c && off[w] + c > (uint32_t)kGroup &&
            ((lazy_bound(__ldcg(a.orC + w), (int)__ldcg(a.done + w), j, sh.v) >> j) & 1ull);
    }
    const uint32_t ball = __ballot_sync(0xffffffffu, may);
    if (lane == 0) sh.flags[warp] = ball;
    __syncthreads();
    for (int f = 0; f < 8; ++f) {
      uint32_t bits = sh.flags[f];  // uniform
      while (bits) {
        const uint32_t ww = w0 + 32 * f + __ffs(bits) - 1;
        bits &= bits - 1;
        const uint32_t cnt = __ldcg(a.cnt + ww);
        const int from = (int)__ldcg(a.done + ww);
        const bool in = (uint32_t)t < cnt && off[ww] + t >= (uint32_t)kGroup;
        uint64_t c = 0;
        if (in) {
          c = __ldcg(a.listC + (size_t)ww * 256 + t);
          for (int s = from; s < j; ++s)
            if ((c >> s) & 1ull) c ^= sh.v[s];
          __stcg(a.listC + (size_t)ww * 256 + t, c);
        }
        const uint32_t has = __ballot_sync(0xffffffffu, (c >> j) & 1ull);
        uint64_t o = c;
        for (int d = 16; d > 0; d >>= 1) o |= __shfl_xor_sync(0xffffffffu, o, d);
        const int first = has ? __ffs(has) - 1 : 0;
        const uint64_t fv = shfl64(c, first);
        if (lane == 0) {
          sh.cand[0][warp] = has ? 32 * warp + first : -1;
          sh.cand_v[0][warp] = fv;
          sh.wor[warp] = o;
        }
        __syncthreads();
        int win = -1;
        uint64_t all = 0;
#pragma unroll
        for (int i = 7; i >= 0; --i) {
          if (sh.cand[0][i] >= 0) win = i;
          all |= sh.wor[i];
        }
        if (t == 0) {
          __stcg(a.orC + ww, all);
          __stcg(a.done + ww, (uint32_t)j);
          if (win >= 0) {
            sh.found = 1;
            sh.found_v = sh.cand_v[0][win];
            sh.found_row = (int64_t)__ldcg(a.listRow + (size_t)ww * 256 + sh.cand[0][win]);
          }
        }
        __syncthreads();
        if (win >= 0) return;
      }
    }
    __syncthreads();  // flags are rewritten
  }
}

__device__ void symbolic_pass(const FrontArgs &a, SymbolicShared &sh, uint32_t *off, uint32_t nwin) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, B = (int)a.B;
  BlkState &st = a.win->st[a.cur];
  // off[w] = nonzero rows before range w
  const uint32_t per = (nwin + 255) / 256, w0 = min(nwin, t * per), w1 = min(nwin, w0 + per);
  uint32_t sum = 0;
  for (uint32_t w = w0; w < w1; ++w) sum += __ldcg(a.cnt + w);
  uint32_t inc = sum;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += y;
  }
  if (lane == 31) sh.sum[warp] = inc;
  if (t < 64) { sh.v[t] = 0; sh.piv[t] = kBlkNone; }
  __syncthreads();
  uint32_t before = inc - sum, total = 0;
  for (int i = 0; i < 8; ++i) {
    if (i < warp) before += sh.sum[i];
    total += sh.sum[i];
  }
  for (uint32_t w = w0; w < w1; ++w) {
    off[w] = before;
    before += __ldcg(a.cnt + w);
  }
  __syncthreads();
  const uint32_t group = min(total, (uint32_t)kGroup);
#pragma unroll
  for (int i = 0; i < kGroup / 256; ++i) {
    const uint32_t g = t + 256 * i;
    uint64_t c = 0;
    uint32_t row = 0;
    if (g < group) {
      uint32_t lo = 0, hi = nwin;  // last range with off <= g
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (off[mid] <= g) lo = mid; else hi = mid;
      }
      const size_t e = (size_t)lo * 256 + (g - off[lo]);
      c = __ldcg(a.listC + e);
      row = __ldcg(a.listRow + e);
    }
    sh.c[g] = c;
    sh.row[g] = row;
  }
  __syncthreads();
  Tile T;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const uint64_t c = sh.c[128 * warp + 32 * m + lane];
    T.lo[m] = transpose32((uint32_t)c, lane);
    T.hi[m] = transpose32((uint32_t)(c >> 32), lane);
  }
  uint32_t w[4];
  if (warp == 0) {
    int j = 0;
    for (; j < B; ++j) {
      tile_column(T, j, w);
      const int p = tile_first(w);
      if (p < 0) {
        if (group > 128) break;  // the other warps' rows may have one
        continue;
      }
      const uint64_t v = tile_row(T, p);
      tile_apply(T, w, v, lane);
      if (lane == 0) { sh.v[j] = v; sh.piv[j] = sh.row[p]; }
    }
    if (lane == 0) sh.j0 = j;
  }
  __syncthreads();
  const int j0 = sh.j0;
  if (j0 < B) {
    if (warp > 0)
      for (int s = 0; s < j0; ++s) {
        const uint64_t v = sh.v[s];
        if (!v) continue;
        tile_column(T, s, w);
        tile_apply(T, w, v, lane);
      }
    for (int j = j0, par = 0; j < B; ++j, par ^= 1) {
      tile_column(T, j, w);
      const int p = tile_first(w);
      const uint64_t v = p >= 0 ? tile_row(T, p) : 0;
      if (lane == 0) {
        sh.cand[par][warp] = p >= 0 ? 128 * warp + p : -1;
        sh.cand_v[par][warp] = v;
      }
      __syncthreads();
      int win = -1;
#pragma unroll
      for (int i = 7; i >= 0; --i)
        if (sh.cand[par][i] >= 0) win = i;
      uint64_t pv = 0;
      int64_t prow = kBlkNone;
      if (win >= 0) {
        pv = sh.cand_v[par][win];
        prow = sh.row[sh.cand[par][win]];
      } else if (total > (uint32_t)kGroup) {
        search_rest(a, sh, off, nwin, j);
        if (sh.found) { pv = sh.found_v; prow = sh.found_row; }
        __syncthreads();
      }
      if (pv) tile_apply(T, w, pv, lane);
      if (t == 0) { sh.v[j] = pv; sh.piv[j] = prow; }
    }
    __syncthreads();
  }
  // M is linear in C: lin[t] = the steps that reduce unit vector t; mpiv from it
  if (t < 64) {
    uint64_t c = 1ull << t, m = 0;
    for (int s = t; s < B; ++s) {
      const uint64_t v = sh.v[s];
      if (v && ((c >> s) & 1ull)) { c ^= v; m |= 1ull << s; }
    }
    st.lin[t] = m;
  } else if (t < 128) {
    const int j = t - 64;
    uint64_t m = 0;
    if (j < B && sh.v[j]) {
      uint64_t c = __ldcg(a.C + sh.piv[j]);
      for (int s = 0; s < j; ++s) {
        const uint64_t v = sh.v[s];
        if (v && ((c >> s) & 1ull)) { c ^= v; m |= 1ull << s; }
      }
    }
    sh.mpiv[j] = m;
  }
  __syncthreads();
  if (t < 64) build_products(sh.mpiv, sh.piv, B, sh.E);
  __syncthreads();
  if (t < 64) {
    st.piv[t] = sh.piv[t];
    st.cpiv[t] = sh.v[t];
    st.mpiv[t] = sh.mpiv[t];
    st.E[t] = sh.E[t];
    st.A[t] = 0; st.B0[t] = 0; st.Cp[t] = 0; st.rV[t] = 0; st.G[t] = 0;
  }
  if (t == 0) st.ntouched = 0;
}

__global__ void __launch_bounds__(256) blk_front_kernel(const FrontArgs a) {
  extern __shared__ uint32_t s_off[];  // gridDim.x words (lazy symbolic pass)
  __shared__ ColRuns s_runs;
  __shared__ SymbolicShared s_sym;
  __shared__ uint32_t s_cnt[8];
  __shared__ uint64_t s_or[8];
  __shared__ bool s_last;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint64_t r = (uint64_t)blockIdx.x * 256 + t;
  if (a.prev_B) sign_rows(a, r);
  if (!a.B) return;
  if (t < 64) {
    build_runs(s_runs, a.window + a.i0, (int)a.B, a.n);
    if (blockIdx.x == 0 && t < (int)a.B && a.window[a.i0 + t] >= a.n) atomicOr(a.err, kErrBadQubit);
  }
  __syncthreads();
  uint64_t c = 0;
  if (r < a.nrows) {
    c = gather_runs(s_runs, a.RX + r * a.rs);
    a.C[r] = c;
  }
  const bool stab = r >= 64ull * a.k && r < 64ull * a.k + a.n;
  if (!a.lazy) {
    if (r < a.nrows) { a.M[r] = 0; a.base[r] = kBaseOrig; }
    const uint32_t ball = __ballot_sync(0xffffffffu, stab && (c & 1ull));
    if (lane == 0 && ball)
      atomicMin(reinterpret_cast<long long *>(&a.win->st[a.cur].slot[0]), (long long)(r + __ffs(ball) - 1));
    return;
  }
  // nonzero stabilizer rows of this range, in order, and the OR of their C
  const bool keep = stab && c != 0;
  const uint32_t ball = __ballot_sync(0xffffffffu, keep);
  uint64_t o = keep ? c : 0;
  for (int d = 16; d > 0; d >>= 1) o |= __shfl_xor_sync(0xffffffffu, o, d);
  if (lane == 0) { s_cnt[warp] = __popc(ball); s_or[warp] = o; }
  __syncthreads();
  uint32_t at = __popc(ball & ((1u << lane) - 1));
  for (int i = 0; i < warp; ++i) at += s_cnt[i];
  if (keep) {
    a.listC[(size_t)blockIdx.x * 256 + at] = c;
    a.listRow[(size_t)blockIdx.x * 256 + at] = (uint32_t)r;
  }
  if (t == 0) {
    uint32_t cnt = 0;
    uint64_t all = 0;
    for (int i = 0; i < 8; ++i) { cnt += s_cnt[i]; all |= s_or[i]; }
    a.cnt[blockIdx.x] = cnt;
    a.orC[blockIdx.x] = all;
    a.done[blockIdx.x] = 0;
  }
  __threadfence();
  __syncthreads();
  if (t == 0) {
    s_last = atomicAdd(&a.win->front_arrived, 1u) == gridDim.x - 1;
    if (s_last) a.win->front_arrived = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  symbolic_pass(a, s_sym, s_off, gridDim.x);
}

// ---------------------------------------------------------------------------
// step-by-step symbolic pass (QS_FLAG_STEP_SYMBOLIC): reset, one launch per
// step over every row, then the products E
// ---------------------------------------------------------------------------
__global__ void blk_step_reset_kernel(BlkState *st) {
  const int t = threadIdx.x;
  if (t < 3) st->slot[t] = kBlkNone;
  if (t == 0) st->ntouched = 0;
  st->piv[t] = kBlkNone; st->mpiv[t] = 0; st->cpiv[t] = 0;
  st->A[t] = 0; st->B0[t] = 0; st->Cp[t] = 0; st->rV[t] = 0; st->G[t] = 0;
}

// symbolic step j: Cin -> Cout
__global__ void __launch_bounds__(256)
blk_step_kernel(uint64_t nrows, uint32_t n, uint32_t k, int j, int B, const uint64_t *__restrict__ Cin,
                uint64_t *__restrict__ Cout, uint64_t *__restrict__ M, int32_t *__restrict__ base,
                BlkState *st) {
  const int64_t p = st->slot[j % 3];
  const bool prob = p != kBlkNone;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->slot[(j + 2) % 3] = kBlkNone;
    st->piv[j] = p;
  }
  const int64_t pd = p - 64ll * k;
  const uint64_t cp = prob ? Cin[p] : 0;
  const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint64_t c = 0;
  if (r < nrows) {
    c = Cin[r];
    if (prob) {
      if ((int64_t)r == p) {
        st->mpiv[j] = M[r];
        st->cpiv[j] = cp;
        M[r] = 0;
        base[r] = kBasePivot + j;
        c = 0;
      } else if ((int64_t)r == pd) {
        c = cp;
        M[r] = 0;
        base[r] = j;
      } else if ((c >> j) & 1ull) {
        c ^= cp;
        M[r] |= 1ull << j;
      }
    }
    Cout[r] = c;
  }
  if (j + 1 < B) {
    const bool stab = r >= 64ull * k && r < 64ull * k + n;
    const uint32_t ball = __ballot_sync(0xffffffffu, stab && ((c >> (j + 1)) & 1ull));
    if ((threadIdx.x & 31) == 0 && ball)
      atomicMin(reinterpret_cast<long long *>(&st->slot[(j + 1) % 3]), (long long)(r + __ffs(ball) - 1));
  }
}

__global__ void __launch_bounds__(64) blk_step_finish_kernel(BlkState *st, int B) {
  build_products(st->mpiv, st->piv, B, st->E);
}

// ---------------------------------------------------------------------------
// blk_middle: the pivot rows V_j with their phase sums (and in the last of
// those blocks their signs), next to the blocks that turn C into M, the bases
// and the list of rows the block changes
// ---------------------------------------------------------------------------
constexpr int kMidThreads = 1024;
constexpr int kVrowSplit = 4;  // blocks per chunk; block y computes G rows 16 y .. 16 y + 15
constexpr size_t kVrowSmem = 4ull * 64 * 32 * sizeof(uint64_t);  // original and V rows, x and z

struct MiddleArgs {
  const uint64_t *RX, *RZ, *S, *C;
  uint64_t nrows;
  uint32_t rs, k, chunks, B;
  int lazy;
  uint64_t *VX, *VZ, *M;
  int32_t *base;
  uint4 *list;
  BlkWindow *win;
  BlkState *st;
  uint32_t *err;
};

// signs of V_j (first 64 x 16 threads of the block). The phase exponent of step j is
//   e_j = 2 r(p_j) + B0_j - A_j + 2 Cp_j + sum_{s in m_j} (2 rV_s + A_s) + 2 cross(m_j)
// (mod 4), cross(m) = sum over s > t in m of G[s] bit t; everything but the
// 2 rV_s terms is independent of the other steps. With b_j = e'_j / 2 the signs
// solve rV = b + m rV (m strictly lower triangular), so rV_j = parity(E_j & b).
__device__ __forceinline__ void pivot_signs(const MiddleArgs &a) {
  __shared__ int sA[64];
  __shared__ uint64_t sm[64], sG[64];
  __shared__ uint32_t s_b[64];
  BlkState *st = a.st;
  const int t = threadIdx.x;
  if (t < 64) {
    sm[t] = t < (int)a.B ? __ldcg(&st->mpiv[t]) : 0;
    sA[t] = __ldcg(&st->A[t]);
    sG[t] = __ldcg(&st->G[t]);
  }
  __syncthreads();
  const int j = t >> 4, part = t & 15;  // 16 threads per step, 4 bits of m each
  const uint64_t m = sm[j];
  int e = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = 4 * part + i;
    if ((m >> s) & 1ull) e += sA[s] + 2 * (__popcll(sG[s] & m & ((1ull << s) - 1)) & 1);
  }
  for (int o = 8; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (part == 0) {
    uint32_t b = 0;
    const int64_t p = j < (int)a.B ? st->piv[j] : kBlkNone;
    if (p != kBlkNone) {
      e += 2 * (int)((a.S[p >> 6] >> (p & 63)) & 1u) + __ldcg(&st->B0[j]) - sA[j] + 2 * __ldcg(&st->Cp[j]);
      e = m4(e);
      if (e & 1) atomicOr(a.err, kErrOddPhase);
      b = (uint32_t)(e >> 1);
    }
    s_b[j] = b;
  }
  __syncthreads();
  if (t < 64) {
    const uint64_t E = st->E[t];
    int rv = 0;
    for (int s = 0; s < 64; ++s) rv ^= (int)((E >> s) & s_b[s] & 1u);
    st->rV[t] = rv;
  }
}

__device__ __forceinline__ void pivot_rows(const MiddleArgs &a, uint32_t chunk, int y) {
  extern __shared__ uint64_t vsm[];
  uint64_t(*ox)[32] = reinterpret_cast<uint64_t(*)[32]>(vsm);
  uint64_t(*oz)[32] = reinterpret_cast<uint64_t(*)[32]>(vsm + 64 * 32);
  uint64_t(*vx)[32] = reinterpret_cast<uint64_t(*)[32]>(vsm + 2 * 64 * 32);
  uint64_t(*vz)[32] = reinterpret_cast<uint64_t(*)[32]>(vsm + 3 * 64 * 32);
  __shared__ uint64_t sE[64];
  __shared__ bool s_last;
  BlkState *st = a.st;
  const uint32_t rs = a.rs;
  const int L = (int)a.B;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kMidThreads >> 5;
  const bool lead = y == 0;  // writes the V rows and the per-step sums
  // every word of the padded row (u < rs): padding qubit words are zero in the
  // tableau and come out zero in the V rows too
  const uint32_t u = chunk * 32 + lane;
  const bool in = u < rs;
  for (int j = w; j < L; j += nw) {
    const int64_t p = st->piv[j];
    const bool ld = in && p != kBlkNone;
    ox[j][lane] = ld ? a.RX[(uint64_t)p * rs + u] : 0;
    oz[j][lane] = ld ? a.RZ[(uint64_t)p * rs + u] : 0;
  }
  if (threadIdx.x < 64) sE[threadIdx.x] = st->E[threadIdx.x];
  __syncthreads();
  // every block builds all V rows of its chunk (G needs them); the lead block
  // also stores them and adds the per-step popcount sums. Deterministic steps
  // have an empty E: their V row is zero.
  for (int j = w; j < L; j += nw) {
    const uint64_t x0 = ox[j][lane], z0 = oz[j][lane];
    uint64_t ax = 0, az = 0, e = sE[j];
    while (e) {
      const int s2 = __ffsll((long long)e) - 1;
      e &= e - 1;
      ax ^= ox[s2][lane];
      az ^= oz[s2][lane];
    }
    vx[j][lane] = ax;
    vz[j][lane] = az;
    if (!lead) continue;
    if (in) {
      a.VX[(uint64_t)j * rs + u] = ax;
      a.VZ[(uint64_t)j * rs + u] = az;
    }
    const int av = __reduce_add_sync(0xffffffffu, __popcll(ax & az));
    const int b = __reduce_add_sync(0xffffffffu, __popcll(x0 & z0));
    const uint32_t c = __ballot_sync(0xffffffffu, __popcll((az ^ z0) & x0) & 1);
    if (lane == 0) {
      if (av) atomicAdd(&st->A[j], av);
      if (b) atomicAdd(&st->B0[j], b);
      if (__popc(c) & 1) atomicXor(&st->Cp[j], 1);
    }
  }
  __syncthreads();
  // G[s] bit t = parity of z_{V_s} . x_{V_t} over the chunk: block y takes
  // s = 16 y + w / 2, each warp half of the t range
  const int sg = 16 * y + (w >> 1), t0 = 32 * (w & 1);
  if (sg < L) {
    const uint64_t zs = vz[sg][lane];
    uint64_t row = 0;
    for (int t = t0; t < t0 + 32 && t < L; ++t) {
      const uint32_t bal = __ballot_sync(0xffffffffu, __popcll(zs & vx[t][lane]) & 1);
      row |= (uint64_t)(__popc(bal) & 1) << t;
    }
    if (lane == 0 && row) atomicXor(reinterpret_cast<unsigned long long *>(&st->G[sg]), row);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(&a.win->middle_arrived, 1u) == a.chunks * kVrowSplit - 1;
    if (s_last) a.win->middle_arrived = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  pivot_signs(a);
}

// M, base and the row list of 1,024 rows. A row that is neither a pivot nor a
// replaced destabilizer has M_r = XOR of lin[t] over the bits of C_r: 16
// lookups in tables of 4 bits each instead of replaying 64 steps. The partner
// of step j starts from C = v_j with only the later steps left. The list holds
// every row the block changes with its pattern and base (one atomic per warp);
// rows left alone (M_r = 0, original base: e.g. the +-Z_q pivot rows of earlier
// blocks) are neither listed, read nor written by the apply pass.
__device__ __forceinline__ void list_rows(const MiddleArgs &a, uint32_t blk) {
  __shared__ uint64_t tab[16 * 16];
  __shared__ int16_t special[kMidThreads];
  const int t = threadIdx.x, lane = t & 31;
  const uint64_t r0 = (uint64_t)blk * kMidThreads, r = r0 + t;
  uint64_t m = 0;
  int32_t b = kBaseOrig;
  if (a.lazy) {
    special[t] = -1;
    if (t < 256) {
      const int g = t >> 4, pat = t & 15;
      uint64_t x = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if ((pat >> i) & 1) x ^= a.st->lin[4 * g + i];
      tab[t] = x;
    }
    __syncthreads();
    if (t < (int)a.B) {
      const int64_t p = a.st->piv[t];
      if (p != kBlkNone) {
        const int64_t dp = p - (int64_t)r0, dd = dp - 64ll * a.k;
        if (dp >= 0 && dp < kMidThreads) special[dp] = (int16_t)(kBasePivot + t);
        if (dd >= 0 && dd < kMidThreads) special[dd] = (int16_t)t;
      }
    }
    __syncthreads();
    if (r < a.nrows) {
      b = special[t];
      uint64_t c = 0;
      if (b == kBaseOrig) c = a.C[r];
      else if (b < kBasePivot) c = a.st->cpiv[b] & ~((2ull << b) - 1);
#pragma unroll
      for (int g = 0; g < 16; ++g) m ^= tab[16 * g + ((c >> (4 * g)) & 15)];
      a.M[r] = m;
      a.base[r] = b;
    }
  } else if (r < a.nrows) {
    m = a.M[r];
    b = a.base[r];
  }
  const bool touched = r < a.nrows && (b != kBaseOrig || m != 0);
  const uint32_t ball = __ballot_sync(0xffffffffu, touched);
  uint32_t at = 0;
  if (lane == 0 && ball) at = atomicAdd(&a.st->ntouched, (uint32_t)__popc(ball));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (touched)
    a.list[at + __popc(ball & ((1u << lane) - 1))] =
        make_uint4((uint32_t)r, (uint32_t)b, (uint32_t)m, (uint32_t)(m >> 32));
}

__global__ void __launch_bounds__(kMidThreads) blk_middle_kernel(const MiddleArgs a) {
  const uint32_t nv = a.chunks * kVrowSplit;
  if (blockIdx.x < nv) pivot_rows(a, blockIdx.x / kVrowSplit, (int)(blockIdx.x % kVrowSplit));
  else list_rows(a, blockIdx.x - nv);
}

// phase 3: block = one chunk of kCW (32) column words x a range of rows.
// The XOR of any subset of the 64 V rows is assembled from tables of XOR
// combinations of consecutive steps (the "Four Russians" method), built once
// per block: T[g][c] = XOR of V[first step of g + b] over the bits b of c. A
// warp handles one row (lane = column word, x and z side by side in one
// 16-byte entry, 512 bytes per entry over the warp); a row segment is 256
// contiguous bytes of each matrix, the shortest that keeps HBM fully
// efficient. Each warp keeps the next two rows' loads in flight while it
// works on the current one; the row loop is unrolled by three so the
// in-flight rows rotate through registers without copies.
//
// The tables live in two memories of the SM. Steps 0..43 use shared memory:
// seven groups of 6 steps and one of 2 (452 entries, 226 KB). Steps 44..63
// use tensor memory (TMEM, 512 columns x 128 lanes of 32 bits): four groups
// of 5 steps. TMEM lane l of each 32-lane quarter holds column word l of the
// chunk and every quarter holds the same four tables (a warp reads only the
// lanes of its quarter, warp mod 4), so an entry is 4 columns (x lo, x hi,
// z lo, z hi) and group t, pattern p sits at columns 128 t + 4 p. A row costs
// 8 shared-memory lookups (32 wavefronts; 13 lookups and 52 wavefronts with
// 5-step groups in shared memory alone, which bounded the pass on the
// shared-memory pipe) and 4 TMEM loads on the tensor-memory read path.
constexpr int kEntryBytes = kCW * 16;   // 512

struct ApplyRow {
  uint32_t r;
  int32_t b;
  uint32_t lo, hi;  // M_r
  uint2 x, z;       // this lane's word of x and z, as 32-bit halves
};

// row, pattern M_r and base_r of a row the block changes (one stage ahead of
// its words): entry j of the row list, or row = nrows past its end
struct ApplyMeta {
  uint32_t r;
  int32_t b;
  uint32_t lo, hi;
};

__device__ __forceinline__ void apply_meta(ApplyMeta &m, uint32_t j, uint32_t cnt, uint32_t nrows,
                                           const uint4 *list) {
  m.r = nrows;
  m.b = kBaseOrig;
  m.lo = m.hi = 0;
  if (j < cnt) {
    const uint4 e = __ldg(list + j);
    m.r = e.x;
    m.b = (int32_t)e.y;
    m.lo = e.z;
    m.hi = e.w;
  }
}

// the row's words, fetched only when the row changes: a row that no step
// targeted and that kept its original base (M_r = 0, base_r original; e.g.
// the +-Z_q pivot rows of earlier blocks) is neither read nor written
template <typename Idx>
__device__ __forceinline__ void apply_fetch(ApplyRow &a, const ApplyMeta &m, const uint64_t *RX,
                                            const uint64_t *RZ, uint32_t rs, uint32_t word, uint32_t nrows,
                                            bool ok) {
  a.r = m.r;
  a.b = m.b;
  a.lo = m.lo;
  a.hi = m.hi;
  a.x = a.z = make_uint2(0, 0);
  if (ok && m.r < nrows) {
    const Idx off = (Idx)m.r * rs + word;
    a.x = reinterpret_cast<const uint2 *>(RX)[off];
    a.z = reinterpret_cast<const uint2 *>(RZ)[off];
  }
}

// a ^ b ^ c in one three-input logic operation
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ void acc3(uint4 &a, const uint4 &p, const uint4 &q) {
  a.x = xor3(a.x, p.x, q.x);
  a.y = xor3(a.y, p.y, q.y);
  a.z = xor3(a.z, p.z, q.z);
  a.w = xor3(a.w, p.w, q.w);
}

constexpr int kSmemGroups = 8;            // shared-memory groups (steps 0..43)
constexpr int kSmemEntries = 7 * 64 + 4;  // 452 entries of 512 bytes
constexpr int kTmemStep0 = 44;            // first step held in TMEM
constexpr uint32_t kTmemCols = 512;       // all of the SM's tensor memory
__host__ __device__ constexpr int smem_group_bits(int g) { return g < 7 ? 6 : 2; }
__host__ __device__ constexpr int smem_group_base(int g) { return 64 * g; }

// byte offset (pattern * 512) of shared group g (6 steps from 6 g; group 7: steps 42, 43)
template <int g>
__device__ __forceinline__ uint32_t pat_off(uint32_t lo, uint32_t hi) {
  constexpr int sh = 6 * g, nb = smem_group_bits(g);
  constexpr uint32_t mask = (uint32_t)((1 << nb) - 1) * kEntryBytes;
  if constexpr (sh + nb <= 32) {
    if constexpr (sh >= 9) return (lo >> (sh - 9)) & mask;
    else return (lo << (9 - sh)) & mask;
  } else if constexpr (sh >= 32) {
    if constexpr (sh - 32 >= 9) return (hi >> (sh - 32 - 9)) & mask;
    else return (hi << (9 - (sh - 32))) & mask;
  } else {
    return __funnelshift_r(lo, hi, sh - 9) & mask;  // bits straddle the halves
  }
}

// shared table entry of group g for this lane: (x lo, x hi, z lo, z hi); the
// pattern's byte offset is a multiple of 512 and the lane's (16 lane) is
// below 512, so one OR joins them
template <int g>
__device__ __forceinline__ uint4 tab(const char *tb, uint32_t lane16, uint32_t lo, uint32_t hi) {
  return *reinterpret_cast<const uint4 *>(tb + smem_group_base(g) * kEntryBytes + (pat_off<g>(lo, hi) | lane16));
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint4 &v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(taddr));
}

// waits for this thread's TMEM loads; the operands tie the loaded registers
// to the wait so that no use is scheduled before it
__device__ __forceinline__ void tmem_wait_ld(uint4 &a, uint4 &b, uint4 &c, uint4 &d) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a.x), "+r"(a.y), "+r"(a.z), "+r"(a.w), "+r"(b.x), "+r"(b.y), "+r"(b.z), "+r"(b.w),
                 "+r"(c.x), "+r"(c.y), "+r"(c.z), "+r"(c.w), "+r"(d.x), "+r"(d.y), "+r"(d.z), "+r"(d.w)
               :
               : "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint4 v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

template <typename Idx>
__device__ __forceinline__ void apply_row(const ApplyRow &a, uint32_t nrows, uint64_t *RX, uint64_t *RZ,
                                          bool ok, uint32_t word, const uint32_t *qubits,
                                          const uint64_t *VX, const uint64_t *VZ, uint32_t rs,
                                          uint32_t lane, const char *tb, uint32_t tq, int32_t *Tp,
                                          uint64_t tp0) {
  const uint32_t r = a.r;
  if (r >= nrows) return;  // uniform over the warp
  const Idx off = (Idx)r * rs + word;
  uint2 *px = reinterpret_cast<uint2 *>(RX), *pz = reinterpret_cast<uint2 *>(RZ);
  if (a.b >= kBasePivot) {  // pivot row of step j: +-Z_q (sign set by blk_front_kernel)
    const uint32_t q = qubits[a.b - kBasePivot];
    if (ok) {
      px[off] = make_uint2(0, 0);
      const uint32_t bit = ((q >> 6) == word) ? 1u << (q & 31) : 0u;
      pz[off] = (q & 32) ? make_uint2(0, bit) : make_uint2(bit, 0);
    }
    return;
  }
  if (a.b == kBaseOrig && (a.lo | a.hi) == 0) return;
  uint2 xb = a.x, zb = a.z;
  if (a.b != kBaseOrig && ok) {  // destabilizer replaced by V_b at step b
    xb = reinterpret_cast<const uint2 *>(VX)[(uint64_t)a.b * rs + word];
    zb = reinterpret_cast<const uint2 *>(VZ)[(uint64_t)a.b * rs + word];
  }
  const uint32_t lo = a.lo, hi = a.hi;
  // steps 44..63 = bits 12..31 of hi: TMEM group t holds bits 12 + 5 t ..
  uint4 m0, m1, m2, m3;
  tmem_ld4(tq + 4 * ((hi >> 12) & 31), m0);
  tmem_ld4(tq + 128 + 4 * ((hi >> 17) & 31), m1);
  tmem_ld4(tq + 256 + 4 * ((hi >> 22) & 31), m2);
  tmem_ld4(tq + 384 + 4 * (hi >> 27), m3);
  const uint32_t l16 = lane * 16;
  uint4 acc = tab<0>(tb, l16, lo, hi);
  acc3(acc, tab<1>(tb, l16, lo, hi), tab<2>(tb, l16, lo, hi));
  acc3(acc, tab<3>(tb, l16, lo, hi), tab<4>(tb, l16, lo, hi));
  acc3(acc, tab<5>(tb, l16, lo, hi), tab<6>(tb, l16, lo, hi));
  const uint4 s7 = tab<7>(tb, l16, lo, hi);
  tmem_wait_ld(m0, m1, m2, m3);
  acc3(acc, s7, m0);
  acc3(acc, m1, m2);
  acc.x ^= m3.x;
  acc.y ^= m3.y;
  acc.z ^= m3.z;
  acc.w ^= m3.w;
  const uint2 xf = make_uint2(xb.x ^ acc.x, xb.y ^ acc.y), zf = make_uint2(zb.x ^ acc.z, zb.y ^ acc.w);
  if (ok) {
    px[off] = xf;
    pz[off] = zf;
  }
  const int t = __popc(xb.x & zb.x) + __popc(xb.y & zb.y) - __popc(xf.x & zf.x) - __popc(xf.y & zf.y);
  const int c = __popc((acc.z & xb.x) ^ (acc.w & xb.y)) & 1;  // parity of z_acc . x_b
  const int v = __reduce_add_sync(0xffffffffu, 64 * t + c);
  if (lane == 0) Tp[tp0 + r] = (v >> 6) * 2 + (v & 1);
}

// 1,024 threads at 64 registers: 6.80 ms per dense block at 180k, against
// 7.46 ms with 768 threads (80 registers) and 9.55 ms with 512 (100)
constexpr int kApplyThreads = 1024;
// blocks per SM over the grid: 6.41 ms per dense 180k block with 32 waves of
// one block per SM, 6.43 with 24, 6.49 with 16, 6.79 with 8, 7.46 with 4 (the
// tails of the last wave shrink; a block's table build stays small)
constexpr int kApplyWaves = 32;

template <typename Idx>
__global__ void __launch_bounds__(kApplyThreads, 1)
blk_apply_kernel(uint64_t *__restrict__ RX, uint64_t *__restrict__ RZ, uint32_t rs, uint32_t nrows,
                 const uint32_t *__restrict__ qubits, int L, const uint64_t *__restrict__ VX,
                 const uint64_t *__restrict__ VZ, const uint4 *__restrict__ list,
                 int32_t *__restrict__ Tp, const BlkState *st) {
  extern __shared__ ulonglong2 T[];  // [kSmemEntries][kCW] of (x word, z word)
  __shared__ uint32_t s_tmem;
  const uint32_t cnt = st->ntouched;
  if (cnt == 0) return;  // every outcome of the block is deterministic
  const uint32_t u0 = blockIdx.x * kCW;  // first column word of the chunk
  const uint32_t nw = min((uint32_t)kCW, rs - u0);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {  // the whole TMEM of the SM: one block per SM (the tables fill shared memory)
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(&s_tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // shared tables, one item per (group, quarter of its entries, word): the
  // quarter's two top steps give its first entry, then its entries follow in
  // Gray-code order, each one V row away from the previous
  for (int it = threadIdx.x; it < kSmemGroups * 4 * 32; it += blockDim.x) {
    const int w = it & 31, sr = (it >> 5) & 3, g = it >> 7;
    const int nb = smem_group_bits(g), e0 = smem_group_base(g) + (sr << (nb - 2));
    ulonglong2 vv[6];
#pragma unroll
    for (int b = 0; b < 6; ++b) {
      const int st = 6 * g + b;
      vv[b] = make_ulonglong2(0, 0);
      if (b < nb && st < L && (uint32_t)w < nw)
        vv[b] = make_ulonglong2(VX[(uint64_t)st * rs + u0 + w], VZ[(uint64_t)st * rs + u0 + w]);
    }
    const ulonglong2 t0 = nb == 6 ? vv[4] : vv[0], t1 = nb == 6 ? vv[5] : vv[1];
    ulonglong2 e = make_ulonglong2(((sr & 1) ? t0.x : 0) ^ ((sr & 2) ? t1.x : 0),
                                   ((sr & 1) ? t0.y : 0) ^ ((sr & 2) ? t1.y : 0));
    T[e0 * kCW + w] = e;
    if (nb == 6) {
#pragma unroll
      for (int k = 1; k < 16; ++k) {
        const int lb = (k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : 3;
        e.x ^= vv[lb].x;
        e.y ^= vv[lb].y;
        T[(e0 + (k ^ (k >> 1))) * kCW + w] = e;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tq = s_tmem + ((32u * (warp & 3)) << 16);  // lane quarter of this warp
  if (warp < 16) {
    // TMEM table t = warp / 4 of this warp's quarter, entries in Gray-code order
    const int t = warp >> 2;
    uint4 v[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
      const int st = kTmemStep0 + 5 * t + b;
      v[b] = make_uint4(0, 0, 0, 0);
      if (st < L && lane < nw) {
        const uint2 x = reinterpret_cast<const uint2 *>(VX)[(uint64_t)st * rs + u0 + lane];
        const uint2 z = reinterpret_cast<const uint2 *>(VZ)[(uint64_t)st * rs + u0 + lane];
        v[b] = make_uint4(x.x, x.y, z.x, z.y);
      }
    }
    uint4 e = make_uint4(0, 0, 0, 0);
    tmem_st4(tq + 128 * t, e);
#pragma unroll
    for (int k = 1; k < 32; ++k) {
      const int b = (k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4;
      e.x ^= v[b].x;
      e.y ^= v[b].y;
      e.z ^= v[b].z;
      e.w ^= v[b].w;
      tmem_st4(tq + 128 * t + 4 * (k ^ (k >> 1)), e);
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  {
    const bool ok = lane < nw;
    const uint32_t word = u0 + lane;
    const char *tb = reinterpret_cast<const char *>(T);
    const uint32_t units = gridDim.y * (blockDim.x >> 5);
    const uint64_t tp0 = (uint64_t)blockIdx.x * nrows;
    // the warp's entries of the row list: j, j + units, ...
    uint32_t j = blockIdx.y * (blockDim.x >> 5) + warp;
    ApplyRow a0, a1, a2;
    ApplyMeta mn;
    apply_meta(mn, j, cnt, nrows, list);
    apply_fetch<Idx>(a0, mn, RX, RZ, rs, word, nrows, ok);
    apply_meta(mn, j + units, cnt, nrows, list);
    apply_fetch<Idx>(a1, mn, RX, RZ, rs, word, nrows, ok);
    apply_meta(mn, j + 2 * units, cnt, nrows, list);
    for (; j < cnt; j += 3 * units) {
      apply_fetch<Idx>(a2, mn, RX, RZ, rs, word, nrows, ok);
      apply_meta(mn, j + 3 * units, cnt, nrows, list);
      apply_row<Idx>(a0, nrows, RX, RZ, ok, word, qubits, VX, VZ, rs, lane, tb, tq, Tp, tp0);
      apply_fetch<Idx>(a0, mn, RX, RZ, rs, word, nrows, ok);
      apply_meta(mn, j + 4 * units, cnt, nrows, list);
      apply_row<Idx>(a1, nrows, RX, RZ, ok, word, qubits, VX, VZ, rs, lane, tb, tq, Tp, tp0);
      apply_fetch<Idx>(a1, mn, RX, RZ, rs, word, nrows, ok);
      apply_meta(mn, j + 5 * units, cnt, nrows, list);
      apply_row<Idx>(a2, nrows, RX, RZ, ok, word, qubits, VX, VZ, rs, lane, tb, tq, Tp, tp0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kTmemCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// blk_det: the deterministic outcomes of a window, after its last block.
// (-1)^m Z_q = prod of S_i over the destabilizers D_i with x_iq = 1 (Sec. 2.5);
// the phase of the product P_1 ... P_t is 2 sum r + sum |x_a & z_a| +
// 2 sum_{a<b} z_a . x_b (mod 4), in any order of the rows since they commute.
// An item is (up to 32 outcomes) x (32 column words) x (a range of rows): a
// block gathers the outcomes' column bits of 128 destabilizer rows at a time,
// keeps the rows that belong to any of them, and each of its four warps folds
// those rows into 8 outcomes (lane = word; XOR totals X, Z and the cross term
// in registers). With one group of outcomes the rows are split over blocks
// (about 152 (range, outcome) pairs, as one outcome per launch had), whose
// totals the last block of a column chunk merges: cross ^= X_range . Z_before.
// The last block of a group of outcomes writes their record entries.
// ---------------------------------------------------------------------------
constexpr int kDetThreads = 128;
constexpr int kDetGroup = 32;

struct DetArgs {
  const uint64_t *RX, *RZ, *S;
  uint32_t rs, n, k, chunks;
  const uint32_t *window, *det;
  BlkWindow *win;
  int32_t *acc;         // phase exponent per outcome
  uint32_t *arrived;    // items of a group that are done
  uint64_t *det_x, *det_z;
  uint64_t m0;
  uint8_t *record;
  uint32_t *err;
};

__global__ void __launch_bounds__(kDetThreads) blk_det_kernel(const DetArgs a) {
  __shared__ uint32_t s_q[kDetGroup];
  __shared__ uint32_t s_row[kDetThreads], s_d[kDetThreads];
  __shared__ uint32_t s_cnt[4];
  __shared__ int s_flag;
  const uint32_t nd = a.win->ndet;
  if (nd == 0) return;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t groups = (nd + kDetGroup - 1) / kDetGroup;
  const uint32_t R = groups > 1 ? 1u : max(1u, min((uint32_t)kDetBlocks / nd, (a.n + kDetThreads - 1) / kDetThreads));
  const uint32_t per = ((a.n + R - 1) / R + kDetThreads - 1) / kDetThreads * kDetThreads;
  const uint64_t items = (uint64_t)groups * a.chunks * R;
  for (uint64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const uint32_t range = (uint32_t)(it % R), ch = (uint32_t)(it / R % a.chunks), g = (uint32_t)(it / R / a.chunks);
    const uint32_t d = min((uint32_t)kDetGroup, nd - g * kDetGroup);
    __syncthreads();
    if (t < kDetGroup) s_q[t] = (uint32_t)t < d ? a.window[a.det[g * kDetGroup + t]] : 0;
    __syncthreads();
    const uint32_t u = ch * 32 + lane;
    const bool in = u < a.k;
    uint64_t X[8], Z[8], cross[8];
    int cnt[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { X[j] = Z[j] = cross[j] = 0; cnt[j] = 0; }
    const uint32_t i1 = min(a.n, (range + 1) * per);
    for (uint32_t i0 = range * per; i0 < i1; i0 += kDetThreads) {
      const uint32_t i = i0 + t;
      uint32_t D = 0;
      if (i < i1) {
        const uint64_t *row = a.RX + (uint64_t)i * a.rs;
        uint32_t lastw = 0xFFFFFFFFu;
        uint64_t word = 0;
        for (uint32_t j = 0; j < d; ++j) {
          const uint32_t q = s_q[j];
          if ((q >> 6) != lastw) { lastw = q >> 6; word = row[lastw]; }
          D |= (uint32_t)((word >> (q & 63)) & 1u) << j;
        }
      }
      const uint32_t ball = __ballot_sync(0xffffffffu, D != 0);
      if (lane == 0) s_cnt[warp] = __popc(ball);
      __syncthreads();
      uint32_t at = __popc(ball & ((1u << lane) - 1)), rows = 0;
      for (int w = 0; w < 4; ++w) {
        if (w < warp) at += s_cnt[w];
        rows += s_cnt[w];
      }
      if (D) { s_row[at] = i; s_d[at] = D; }
      __syncthreads();
      for (uint32_t e0 = 0; e0 < rows; e0 += 4) {
        uint64_t x[4], z[4];
        uint32_t m[4], rb[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const uint32_t e = e0 + v;
          m[v] = e < rows ? (s_d[e] >> (8 * warp)) & 0xFFu : 0u;
          x[v] = z[v] = 0;
          rb[v] = 0;
          if (m[v]) {
            const uint64_t row = 64ull * a.k + s_row[e];
            if (in) { x[v] = a.RX[row * a.rs + u]; z[v] = a.RZ[row * a.rs + u]; }
            if (ch == 0 && lane == 0) rb[v] = (uint32_t)(a.S[row >> 6] >> (row & 63)) & 1u;
          }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          if (!m[v]) continue;
          const int pc = __popcll(x[v] & z[v]) + 2 * (int)rb[v];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if ((m[v] >> j) & 1u) {  // uniform over the warp
              cross[j] ^= x[v] & Z[j];
              X[j] ^= x[v];
              Z[j] ^= z[v];
              cnt[j] += pc;
            }
        }
      }
      __syncthreads();  // the row list is rewritten
    }
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t o = 8 * warp + j;
      if (o >= d) break;
      const int v = __reduce_add_sync(0xffffffffu, cnt[j] + 2 * (__popcll(cross[j]) & 1));
      if (lane == 0 && v) atomicAdd(a.acc + g * kDetGroup + o, v);
      if (R == 1) {
        const uint32_t q = s_q[o];
        bad |= in && (X[j] != 0 || Z[j] != (u == (q >> 6) ? 1ull << (q & 63) : 0ull));
      } else if (in) {
        a.det_x[((uint64_t)range * d + o) * a.rs + u] = X[j];
        a.det_z[((uint64_t)range * d + o) * a.rs + u] = Z[j];
      }
    }
    __threadfence();
    __syncthreads();
    if (R > 1) {
      if (t == 0) s_flag = atomicAdd(&a.win->det_chunk[ch], 1u) == R - 1;
      __syncthreads();
      if (!s_flag) continue;
      __threadfence();
      for (uint32_t o = warp; o < d; o += 4) {  // last range of this chunk: merge the ranges
        uint64_t c = 0, xb = 0, zb = 0;
        if (in)
#pragma unroll 4
          for (uint32_t q = 0; q < R; ++q) {
            const uint64_t x = __ldcg(a.det_x + ((uint64_t)q * d + o) * a.rs + u),
                           z = __ldcg(a.det_z + ((uint64_t)q * d + o) * a.rs + u);
            c ^= x & zb;
            xb ^= x;
            zb ^= z;
          }
        const int v = __reduce_add_sync(0xffffffffu, 2 * (__popcll(c) & 1));
        if (lane == 0 && v) atomicAdd(a.acc + o, v);
        const uint32_t q = s_q[o];
        bad |= in && (xb != 0 || zb != (u == (q >> 6) ? 1ull << (q & 63) : 0ull));
      }
      __threadfence();
    }
    if (bad) atomicOr(a.err, kErrDetProduct);
    __syncthreads();
    if (t == 0) s_flag = atomicAdd(a.arrived + g, 1u) == a.chunks - 1;
    __syncthreads();
    if (!s_flag) continue;
    __threadfence();
    if ((uint32_t)t < d) {
      const int e = m4(__ldcg(a.acc + g * kDetGroup + t));
      if (e & 1) atomicOr(a.err, kErrOddPhase);
      a.record[a.m0 + a.det[g * kDetGroup + t]] = (uint8_t)(e >> 1);
    }
  }
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
static uint32_t blk_chunks(const Layout &L) { return (L.rs + kCW - 1) / kCW; }

// device scratch of the blocked measurement
struct BlkScratch {
  uint8_t *zero;       // start of the part zeroed per window: win, acc, arrived
  size_t zero_bytes;
  BlkWindow *win;
  int32_t *acc;
  uint32_t *arrived;
  uint64_t *C0, *C1, *M, *orC, *VX, *VZ;
  uint32_t *listRow, *cnt, *done, *det;
  int32_t *base, *Tp;
  uint4 *list;
  size_t total;
};

// measurements per window (the capacity of det and acc)
static uint32_t blk_window_cap(const Layout &L) { return (uint32_t)L.nrows; }

static BlkScratch blk_scratch(const Layout &L, void *scratch) {
  BlkScratch b;
  size_t off = 0;
  uint8_t *p = static_cast<uint8_t *>(scratch);
  auto take = [&](size_t bytes) {
    uint8_t *q = p + off;
    off += (bytes + 255) & ~size_t(255);
    return q;
  };
  const size_t cap = blk_window_cap(L), ranges = (L.nrows + 255) / 256;
  b.zero = p;
  b.win = reinterpret_cast<BlkWindow *>(take(sizeof(BlkWindow)));
  b.acc = reinterpret_cast<int32_t *>(take(cap * 4));
  b.arrived = reinterpret_cast<uint32_t *>(take((cap / kDetGroup + 1) * 4));
  b.zero_bytes = off;
  b.C0 = reinterpret_cast<uint64_t *>(take(L.nrows * 8));
  b.C1 = reinterpret_cast<uint64_t *>(take(ranges * 256 * 8));
  b.M = reinterpret_cast<uint64_t *>(take(L.nrows * 8));
  b.base = reinterpret_cast<int32_t *>(take(L.nrows * 4));
  b.Tp = reinterpret_cast<int32_t *>(take((size_t)blk_chunks(L) * L.nrows * 4));
  b.VX = reinterpret_cast<uint64_t *>(take(64ull * L.rs * 8));
  b.VZ = reinterpret_cast<uint64_t *>(take(64ull * L.rs * 8));
  b.list = reinterpret_cast<uint4 *>(take(L.nrows * 16));
  b.listRow = reinterpret_cast<uint32_t *>(take(ranges * 256 * 4));
  b.cnt = reinterpret_cast<uint32_t *>(take(ranges * 4));
  b.done = reinterpret_cast<uint32_t *>(take(ranges * 4));
  b.orC = reinterpret_cast<uint64_t *>(take(ranges * 8));
  b.det = reinterpret_cast<uint32_t *>(take(cap * 4));
  b.total = off;
  return b;
}

size_t blocked_scratch_bytes(const Layout &L) { return blk_scratch(L, nullptr).total; }

static std::atomic<uint64_t> g_blk_attr_set{0};

// about kApplyWaves waves of one block per SM (the tables take 226 KB of
// shared memory and all of TMEM), but at least 512 rows per block so that
// building the tables stays small next to the rows they serve
static uint32_t apply_rows_y(const Dev &d, uint32_t chunks) {
  return std::max<uint32_t>(1, (uint32_t)std::min<uint64_t>(((uint64_t)d.sms * kApplyWaves + chunks - 1) / chunks,
                                                            d.L.nrows / 512));
}

static cudaError_t measure_window_cap(const Dev &d, void *scratch, const uint32_t *window, uint32_t count,
                                      uint64_t m0, qs_key key, cudaStream_t s, int *launches) {
  const Layout &L = d.L;
  const BlkScratch b = blk_scratch(L, scratch);
  const uint32_t chunks = blk_chunks(L), ranges = (uint32_t)((L.nrows + 255) / 256);
  const size_t smem = (size_t)kSmemEntries * kEntryBytes;
  cudaError_t e = once_per_device(g_blk_attr_set, [&]() {
    cudaError_t x = cudaFuncSetAttribute(blk_apply_kernel<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (x == cudaSuccess)
      x = cudaFuncSetAttribute(blk_apply_kernel<uint64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (x == cudaSuccess)
      x = cudaFuncSetAttribute(blk_middle_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVrowSmem);
    if (x == cudaSuccess)  // 4 bytes per range of 256 rows: 32 KB at n = 2^20, next to 17 KB of static arrays
      x = cudaFuncSetAttribute(blk_front_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
    return x;
  });
  if (e == cudaSuccess) e = cudaMemsetAsync(b.zero, 0, b.zero_bytes, s);
  if (e != cudaSuccess) return e;
  FrontArgs f{};
  f.RX = d.RX; f.S = d.S; f.nrows = L.nrows; f.rs = L.rs; f.n = L.n; f.k = L.k; f.chunks = chunks;
  f.window = window;
  f.lazy = !d.step_symbolic;
  f.C = b.C0; f.listC = b.C1; f.listRow = b.listRow; f.cnt = b.cnt; f.done = b.done; f.orC = b.orC;
  f.M = b.M; f.base = b.base; f.Tp = b.Tp; f.win = b.win; f.det = b.det;
  f.m0 = m0; f.seed = key.seed; f.shot = key.shot;
  f.record = d.record; f.kinds = d.kinds; f.err = d.err;
  MiddleArgs m{};
  m.RX = d.RX; m.RZ = d.RZ; m.S = d.S; m.C = b.C0; m.nrows = L.nrows; m.rs = L.rs; m.k = L.k; m.chunks = chunks;
  m.lazy = f.lazy;
  m.VX = b.VX; m.VZ = b.VZ; m.M = b.M; m.base = b.base; m.list = b.list; m.win = b.win; m.err = d.err;
  const uint32_t mid_blocks = chunks * kVrowSplit + (uint32_t)((L.nrows + kMidThreads - 1) / kMidThreads);
  const uint32_t rows_y = apply_rows_y(d, chunks);
  const bool narrow = !d.wide_offsets && (uint64_t)L.nrows * L.rs < (1ull << 32);
  int nl = 0;
  for (uint32_t i0 = 0, cur = 0;; i0 += 64, cur ^= 1) {
    // signs of the block before i0, symbolic pass of the block at i0
    f.prev_i0 = f.i0; f.prev_B = f.B;
    f.i0 = i0;
    f.B = i0 < count ? std::min<uint32_t>(64, count - i0) : 0;
    f.cur = (int)cur;
    BlkState *st = &b.win->st[cur];
    const int kind = f.B ? QS_TIME_BLK_SYMBOLIC : QS_TIME_BLK_SIGNS;
    tbegin(d.timer, kind, s);
    if (!f.lazy && f.B) {
      blk_step_reset_kernel<<<1, 64, 0, s>>>(st);
      ++nl;
    }
    blk_front_kernel<<<ranges, 256, f.lazy ? ranges * 4 : 0, s>>>(f);
    ++nl;
    if (!f.lazy && f.B) {
      // C0 -> C1 -> C0 ...; nothing reads C after the last step
      for (int j = 0; j < (int)f.B; ++j)
        blk_step_kernel<<<ranges, 256, 0, s>>>(L.nrows, L.n, L.k, j, (int)f.B, (j & 1) ? b.C1 : b.C0,
                                               (j & 1) ? b.C0 : b.C1, b.M, b.base, st);
      blk_step_finish_kernel<<<1, 64, 0, s>>>(st, (int)f.B);
      nl += (int)f.B + 1;
    }
    tend(d.timer, kind, s);
    if (!f.B) break;
    m.B = f.B;
    m.st = st;
    tbegin(d.timer, QS_TIME_BLK_PIVOT_ROWS, s);
    blk_middle_kernel<<<mid_blocks, kMidThreads, kVrowSmem, s>>>(m);
    tend(d.timer, QS_TIME_BLK_PIVOT_ROWS, s);
    tbegin(d.timer, QS_TIME_BLK_APPLY, s);
    if (narrow)
      blk_apply_kernel<uint32_t><<<dim3(chunks, rows_y), kApplyThreads, smem, s>>>(
          d.RX, d.RZ, L.rs, (uint32_t)L.nrows, window + i0, (int)f.B, b.VX, b.VZ, b.list, b.Tp, st);
    else
      blk_apply_kernel<uint64_t><<<dim3(chunks, rows_y), kApplyThreads, smem, s>>>(
          d.RX, d.RZ, L.rs, (uint32_t)L.nrows, window + i0, (int)f.B, b.VX, b.VZ, b.list, b.Tp, st);
    tend(d.timer, QS_TIME_BLK_APPLY, s);
    nl += 2;
    if (d.timer && (i0 & 4095) == 4032) d.timer->resolve();  // completed event pairs go back to the pool
  }
  DetArgs t{};
  t.RX = d.RX; t.RZ = d.RZ; t.S = d.S; t.rs = L.rs; t.n = L.n; t.k = L.k; t.chunks = (L.k + 31) / 32;
  t.window = window; t.det = b.det; t.win = b.win; t.acc = b.acc; t.arrived = b.arrived;
  t.det_x = d.det_x; t.det_z = d.det_z; t.m0 = m0; t.record = d.record; t.err = d.err;
  // enough blocks for one outcome's ranges and for every group; blocks without an item leave at once
  const uint64_t most = std::max<uint64_t>(kDetBlocks, (count + kDetGroup - 1) / kDetGroup) * t.chunks;
  blk_det_kernel<<<(unsigned)std::min<uint64_t>(most, 12ull * d.sms), kDetThreads, 0, s>>>(t);
  if (launches) *launches += nl + 2;
  return cudaGetLastError();
}

cudaError_t launch_measure_blocks(const Dev &d, void *scratch, const uint32_t *window, uint32_t count, uint64_t m0,
                                  qs_key key, cudaStream_t s, int *launches) {
  const uint32_t cap = blk_window_cap(d.L);
  for (uint32_t off = 0; off < count; off += cap) {
    const cudaError_t e = measure_window_cap(d, scratch, window + off, std::min(cap, count - off), m0 + off, key, s,
                                             launches);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace qs
