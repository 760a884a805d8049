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
// a launch per part took 9 and a wait per round, and each kernel is resident
// before the one ahead of it ends (launch_chained). 64 measurements of a dense
// 10,000-qubit state: 172 -> 62 us; 3,000 measurements of a shallow 1,500-qubit
// state, 2,456 of them deterministic (measured one by one before): 30.3 -> 1.2 ms.
// The chain alone: 256 qubits, all measured, 10 % of the job; 10,000 qubits 6 %.
#include <algorithm>
#include <climits>

#include "qs_internal.cuh"

namespace qs {

constexpr int32_t kBaseOrig = -1;    // all bits set
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
  uint32_t AD[64];     // sums over 4-word chunks of two values mod 4: |x_V & z_V| (low half) and
                       // |x_o & z_o| - |x_V & z_V| + 2 parity((z_V ^ z_o) . x_o), o = the original pivot row
  int32_t rV[64];      // sign bit of V_j
  uint64_t G[64];      // G[s] bit t = parity(z_{V_s} . x_{V_t})
};

// state of one window; zeroed before its first block together with the
// accumulators behind it
struct BlkWindow {
  uint32_t front_arrived, middle_arrived, ndet, pad;
  BlkState st[2];
};

__device__ __forceinline__ int m4(int v) { return ((v % 4) + 4) % 4; }

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

// part `part` of `parts` of the runs' bits of a row, four words in flight
__device__ __forceinline__ uint64_t gather_runs(const ColRuns &R, const uint64_t *row, uint32_t part, uint32_t parts) {
  uint64_t c = 0;
  for (uint32_t i = part; i < R.n; i += 4 * parts) {
    uint64_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = i + u * parts < R.n ? row[R.word[i + u * parts]] : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t x = i + u * parts;
      if (x < R.n) c |= ((w[u] >> R.shift[x]) & R.mask[x]) << R.pos[x];
    }
  }
  return c;
}

// E_j = {j} xor (xor of E_s over the steps s that targeted p_j), for the steps
// of half h (32 h .. 32 h + 31) among themselves; one warp. Lane t keeps column
// t (bit s = whether t is in E_s), so a step is one parity per lane and no
// exchange; the ballots are the rows. prob: bit j set where step j has a pivot.
__device__ __forceinline__ void half_products(const uint64_t *mpiv, uint64_t prob, int h, uint32_t *E) {
  const int lane = threadIdx.x & 31;
  const uint32_t m = (uint32_t)(mpiv[32 * h + lane] >> (32 * h)), pm = (uint32_t)(prob >> (32 * h));
  uint32_t col = 0, mine = 0;
#pragma unroll 8
  for (int j = 0; j < 32; ++j) {
    const uint32_t mj = __shfl_sync(0xffffffffu, m, j);
    const uint32_t bit = ((__popc(col & mj) & 1u) ^ (lane == j)) & (pm >> j);
    col |= bit << j;
    const uint32_t row = __ballot_sync(0xffffffffu, bit);
    if (lane == j) mine = row;
  }
  E[lane] = mine;
}

// the two halves joined by one warp: with the steps' targets m split into
// halves, E_low = E1, E_high = E2 and below the diagonal E2 (m E1); tmp: 32 words
__device__ __forceinline__ void join_products(const uint64_t *mpiv, const uint32_t *E1, const uint32_t *E2,
                                              uint32_t *tmp, uint64_t *E) {
  const int lane = threadIdx.x & 31;
  const uint32_t m = (uint32_t)mpiv[32 + lane], e2 = E2[lane];
  uint32_t x = 0;
#pragma unroll 8
  for (int s = 0; s < 32; ++s) x ^= E1[s] & (0u - ((m >> s) & 1u));
  tmp[lane] = x;
  __syncwarp();
  uint32_t y = 0;
#pragma unroll 8
  for (int s = 0; s < 32; ++s) y ^= tmp[s] & (0u - ((e2 >> s) & 1u));
  E[lane] = E1[lane];
  E[32 + lane] = ((uint64_t)e2 << 32) | y;
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
  uint64_t *C, *listC;          // C of every row; nonzero stabilizer rows of each range (the rows of one
  uint32_t *listRow;            // block): C, row,
  uint32_t *cnt, *done;         // number, steps replayed on them
  uint64_t *orC;                // and OR of their C
  uint64_t *M;
  int32_t *base;
  const uint8_t *Tp;            // phase sums mod 4 of the apply pass, per column chunk and row
  BlkWindow *win;
  uint32_t *det;                // window positions of deterministic outcomes
  uint64_t m0, seed, shot;
  uint8_t *record, *kinds;
  uint32_t *err;
};

// Threads per row: 8 where blocks of 256 rows would leave SMs idle (up to 32,768
// rows), which then share a row's column words, chunk sums and table lookups;
// else 1. At 4,000 qubits with 64 scattered measured qubits the gather alone
// took 21,000 cycles with one thread per row.
constexpr uint64_t kFrontSplitRows = 32768;

template <int P>
__device__ __forceinline__ uint64_t or_parts(uint64_t v) {
#pragma unroll
  for (int d = 1; d < P; d <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// what signing a row reads of it
struct SignIn {
  int32_t b;
  uint64_t m, word;
  int e;  // this part's chunk sums
};

template <int P>
__device__ __forceinline__ SignIn sign_load(const FrontArgs &a, uint64_t r, int part) {
  SignIn in;
  in.b = a.base[r];
  in.m = a.M[r];
  in.word = a.S[r >> 6];
  in.e = 0;
  // with several threads per row the sums are few and are loaded
  // beside the rest; rows the block left alone have stale ones, which nothing uses
  if (P == 1 && (in.b >= kBasePivot || (in.b == kBaseOrig && in.m == 0))) return in;
#pragma unroll 4
  for (uint32_t ch = part; ch < a.chunks; ch += P) in.e += a.Tp[(uint64_t)ch * a.nrows + r];
  return in;
}

struct SignShared {
  uint64_t x[256];
  int sum[256];
  int rV[64];
  uint32_t det[2];
};

// Over the steps s of M_r: the sum of 2 rV_s + A_s, and the XOR X of G[s]
// restricted to earlier steps, whose parity with M_r is the sum over s > t in
// M_r of G[s] bit t. Both come from tables over 4 steps each, 16 lookups a row
// (a loop over the steps of M_r took most of the 7 us this part needed on its own).
__device__ __forceinline__ void sign_tables(const FrontArgs &a, SignShared &sh) {
  const BlkState &st = a.win->st[a.cur ^ 1];
  const int t = threadIdx.x, g = t >> 4, pat = t & 15;
  uint64_t x = 0;
  int sum = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int s = 4 * g + i;
    const uint64_t gs = st.G[s] & ((1ull << s) - 1);
    const int ws = 2 * st.rV[s] + (int)(st.AD[s] & 3u);
    if ((pat >> i) & 1) { x ^= gs; sum += ws; }
  }
  sh.x[t] = x;
  sh.sum[t] = sum;
  if (t < 64) sh.rV[t] = st.rV[t];
}

// the block's record entries; its deterministic outcomes are listed for blk_det
__device__ __forceinline__ void sign_record(const FrontArgs &a, SignShared &sh) {
  const BlkState &st = a.win->st[a.cur ^ 1];
  const uint64_t m0 = a.m0 + a.prev_i0;  // record index of the block's first measurement
  const int t = threadIdx.x, B = (int)a.prev_B;
  const bool in = t < B, prob = in && st.piv[t] != kBlkNone;
  if (in) {
    a.record[m0 + t] = prob ? (uint8_t)(philox4x64_10(m0 + t, a.shot, 0, 0, a.seed, kCoinKey).v[0] & 1u) : 0;
    a.kinds[m0 + t] = prob;
  }
  const bool det = in && !prob && a.window[a.prev_i0 + t] < a.n;
  const uint32_t ball = __ballot_sync(0xffffffffu, det);
  if ((t & 31) == 0) sh.det[t >> 5] = ball;
  const uint32_t first = a.win->ndet;
  asm volatile("bar.sync 1, 64;" ::: "memory");
  if (det) a.det[first + (t >= 32 ? __popc(sh.det[0]) : 0) + __popc(ball & ((1u << (t & 31)) - 1))] = a.prev_i0 + t;
  if (t == 0) a.win->ndet = first + __popc(sh.det[0]) + __popc(sh.det[1]);
}

// new sign of a row from the accumulated terms; pivot rows get their coin
template <int P>
__device__ __forceinline__ void sign_row(const FrontArgs &a, const SignShared &sh, const SignIn &in, uint64_t r,
                                         int part) {
  const int32_t b = in.b;
  const uint64_t sr = in.m, old = (in.word >> (r & 63)) & 1u;
  uint64_t nb = old;
  const bool product = b < kBasePivot && (b != kBaseOrig || sr != 0);
  int e = 0;
  if (product) {
    uint64_t x = 0;
#pragma unroll
    for (int q = 0; q < 16 / P; ++q) {
      const int g = part + P * q, i = 16 * g + (int)((sr >> (4 * g)) & 15);
      x ^= sh.x[i];
      e += sh.sum[i];
    }
    // the parity of an XOR: the parts may be counted apart
    e += in.e + 2 * (__popcll(x & sr) & 1);
  }
#pragma unroll
  for (int d = 1; d < P; d <<= 1) e += __shfl_xor_sync(0xffffffffu, e, d);
  if (b >= kBasePivot) {
    nb = philox4x64_10(a.m0 + a.prev_i0 + (b - kBasePivot), a.shot, 0, 0, a.seed, kCoinKey).v[0] & 1u;
  } else if (product) {
    e = m4(e + 2 * ((b == kBaseOrig) ? (int)old : sh.rV[b]));
    if (e & 1) atomicOr(a.err, kErrOddPhase);
    nb = (uint64_t)(e >> 1);
  }
  uint64_t delta = (nb ^ old) << (r & 63);
  // fold the sign changes of this warp's rows (at most 32, in one word) into one atomic
  for (int o = 16; o >= P; o >>= 1) delta |= __shfl_xor_sync(0xffffffffu, delta, o);
  if ((threadIdx.x & 31) == 0 && delta) atomicXor(reinterpret_cast<unsigned long long *>(&a.S[r >> 6]), delta);
}

// Symbolic pass. Only the pivot sequence (p_j, v_j = C_{p_j} at step j) has to
// be found in order, and the pivot of step j is the first stabilizer row whose
// current C has bit j. Rows with C = 0 never take part, and in any state the
// pivots come from the first nonzero rows, so the first 768 of those are held in
// registers by the block's 8 warps, 96 rows each, three a lane (64 steps of a
// random state miss a pivot among 96 rows once in 2^32). A step is a
// ballot, a shuffle of the pivot's C and one XOR per row that has the bit. The
// registers rotate right by one per step, so that step j always looks at bit 0;
// a row is done with that bit and keeps it as it was, so the bits that went
// round are the row's M, and the pivot brings the steps that targeted it along.
// Warp 0 first runs all steps alone, without branches (312 cycles a step with
// them and four rows a lane); if its rows lack a pivot for a step and there are more rows, all eight
// warps replay the steps before it and go on in step. Nonzero rows beyond the first 768 are only looked at when those have
// no pivot for a step: 256 rows at a time, skipping those that an upper bound on
// the OR of their C rules out (exact when they were last replayed, then grown by
// v_s for every step s whose bit the bound has).
constexpr int kLaneRows = 3, kTileRows = 32 * kLaneRows, kGroup = 8 * kTileRows;

// 0 or all ones by bit b
__device__ __forceinline__ uint64_t spread(uint64_t x, int b) { return 0ull - ((x >> b) & 1ull); }

// one warp's rows, lane l holding rows 3 l .. 3 l + 2, rotated right by the
// step; above: bits of the rotated word past bit 0 that have not gone round yet
struct Tile {
  uint32_t lo[kLaneRows], hi[kLaneRows];
  uint32_t above_lo, above_hi;
};

// the warp's first row with bit 0: raw_* (without bit 0 if there is none) and
// its index, without branches, in every lane
__device__ __forceinline__ void tile_first(const Tile &T, uint32_t &raw_lo, uint32_t &raw_hi, int &index) {
  const bool p0 = T.lo[0] & 1u, p1 = T.lo[1] & 1u, p2 = T.lo[2] & 1u;
  const uint32_t b = __ballot_sync(0xffffffffu, p0 | p1 | p2);
  const uint32_t sl = p0 ? T.lo[0] : p1 ? T.lo[1] : T.lo[2];
  const uint32_t sh = p0 ? T.hi[0] : p1 ? T.hi[1] : T.hi[2];
  const int m = p0 ? 0 : p1 ? 1 : 2;
  const int l = __ffs(b) - 1;  // -1 reads lane 31, whose row 2 has no bit 0 then
  raw_lo = __shfl_sync(0xffffffffu, sl, l);
  raw_hi = __shfl_sync(0xffffffffu, sh, l);
  index = kLaneRows * l + __shfl_sync(0xffffffffu, m, l);
}

// rows with bit 0 take the pivot's bits above (raw 0: no pivot); on to the next step
__device__ __forceinline__ void tile_step(Tile &T, uint32_t raw_lo, uint32_t raw_hi) {
  const uint32_t vl = raw_lo & T.above_lo & ~1u, vh = raw_hi & T.above_hi;
#pragma unroll
  for (int m = 0; m < kLaneRows; ++m) {
    uint32_t l = T.lo[m], h = T.hi[m];
    if (l & 1u) { l ^= vl; h ^= vh; }
    T.lo[m] = __funnelshift_r(l, h, 1);
    T.hi[m] = __funnelshift_r(h, l, 1);
  }
  T.above_lo = __funnelshift_r(T.above_lo, T.above_hi, 1);
  T.above_hi >>= 1;
}

__device__ __forceinline__ uint64_t rotl64(uint64_t x, int b) { return (x << b) | (x >> ((64 - b) & 63)); }

__device__ __forceinline__ uint64_t lazy_bound(uint64_t u, int a, int j, const uint64_t *v) {
  for (int s = a; s < j; ++s)
    if ((u >> s) & 1ull) u |= v[s];
  return u;
}

struct SymbolicShared {
  uint32_t row[kGroup];        // rows of the group
  uint64_t raw[64];            // each step's pivot: its bits rotated right by the step (0: none),
  int index[64];               // index in warp 0's rows (first run),
  int64_t piv[64];             // row,
  uint64_t v[64], mpiv[64];    // C, and steps that targeted it
  uint64_t cand_v[2][8], wor[8];
  int cand[2][8];
  uint32_t sum[8], flags[8];
  uint32_t E1[32], E2[32], tmp[32];
  int found;
  uint64_t found_v;
  int64_t found_row;
};

// pivot of step j among the nonzero rows past the first kGroup (all 256
// threads; off[w] = nonzero rows before range w, P ranges per 256 rows); leaves
// found_* in sh
template <int P>
__device__ __forceinline__ void search_rest(const FrontArgs &a, SymbolicShared &sh, const uint32_t *off, uint32_t ranges, int j) {
  constexpr int kRange = 256 / P;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t chunks = ranges / P;
  __syncthreads();
  if (t == 0) sh.found = 0;
  for (uint32_t w0 = 0; w0 < chunks; w0 += 256) {
    const uint32_t w = w0 + t;
    bool may = false;
    if (w < chunks) {
      uint64_t o = 0;
      uint32_t end = 0;
      for (int i = 0; i < P; ++i) {
        const uint32_t c = __ldcg(a.cnt + w * P + i);
        if (c) { o |= __ldcg(a.orC + w * P + i); end = off[w * P + i] + c; }
      }
      may = end > (uint32_t)kGroup && ((lazy_bound(o, (int)__ldcg(a.done + w * P), j, sh.v) >> j) & 1ull);
    }
    const uint32_t ball = __ballot_sync(0xffffffffu, may);
    if (lane == 0) sh.flags[warp] = ball;
    __syncthreads();
    for (int f = 0; f < 8; ++f) {
      uint32_t bits = sh.flags[f];  // uniform
      while (bits) {
        const uint32_t ww = w0 + 32 * f + __ffs(bits) - 1;
        bits &= bits - 1;
        const uint32_t range = ww * P + t / kRange, e = t % kRange;
        const int from = (int)__ldcg(a.done + ww * P);
        const bool in = e < __ldcg(a.cnt + range) && off[range] + e >= (uint32_t)kGroup;
        uint64_t c = 0;
        if (in) {
          c = __ldcg(a.listC + (size_t)ww * 256 + t);
          for (int s = from; s < j; ++s)
            if ((c >> s) & 1ull) c ^= sh.v[s] & ~(1ull << s);
          __stcg(a.listC + (size_t)ww * 256 + t, c);
        }
        const uint32_t has = __ballot_sync(0xffffffffu, (c >> j) & 1ull);
        uint64_t o = c;
        for (int d = 16; d > 0; d >>= 1) o |= __shfl_xor_sync(0xffffffffu, o, d);
        const int first = has ? __ffs(has) - 1 : 0;
        const uint64_t fv = __shfl_sync(0xffffffffu, c, first);
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
        if (t < P) __stcg(a.orC + ww * P + t, all);
        if (t == 0) {
          __stcg(a.done + ww * P, (uint32_t)j);
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

template <int P>
__device__ __forceinline__ void symbolic_pass(const FrontArgs &a, SymbolicShared &sh, uint32_t *off, uint32_t nwin) {
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
  if (t < 64) { sh.raw[t] = 0; sh.v[t] = 0; sh.mpiv[t] = 0; sh.piv[t] = kBlkNone; }
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
  Tile T;
  T.above_lo = T.above_hi = ~0u;
  uint64_t c0[kLaneRows];
  {
    // last range with off <= g, for the lane's rows side by side
    uint32_t lo[kLaneRows], hi[kLaneRows];
    const uint32_t g0 = kTileRows * warp + kLaneRows * lane;
#pragma unroll
    for (int m = 0; m < kLaneRows; ++m) { lo[m] = 0; hi[m] = nwin; }
    for (uint32_t left = nwin; left > 1; left = (left + 1) >> 1)
#pragma unroll
      for (int m = 0; m < kLaneRows; ++m) {
        const uint32_t mid = (lo[m] + hi[m]) >> 1;
        const bool up = mid > lo[m] && off[mid] <= g0 + m;
        lo[m] = up ? mid : lo[m];
        hi[m] = up ? hi[m] : mid;
      }
    uint32_t row[kLaneRows];
#pragma unroll
    for (int m = 0; m < kLaneRows; ++m) {
      const bool in = g0 + m < group;
      const size_t e = in ? (size_t)lo[m] * (256 / P) + (g0 + m - off[lo[m]]) : 0;
      c0[m] = in ? __ldcg(a.listC + e) : 0;
      row[m] = in ? __ldcg(a.listRow + e) : 0;
    }
#pragma unroll
    for (int m = 0; m < kLaneRows; ++m) {
      sh.row[g0 + m] = row[m];
      T.lo[m] = (uint32_t)c0[m];
      T.hi[m] = (uint32_t)(c0[m] >> 32);
    }
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll 8
    for (int j = 0; j < 64; ++j) {
      uint32_t rl, rh;
      int index;
      tile_first(T, rl, rh, index);
      tile_step(T, rl, rh);
      sh.raw[j] = ((uint64_t)rh << 32) | rl;  // every lane, the same value; no bit 0: no pivot
      sh.index[j] = index;
    }
  }
  __syncthreads();
  // the first step warp 0 has no pivot for, if other rows may have one
  int j0 = B;
  {
    const uint32_t lo = __ballot_sync(0xffffffffu, !(sh.raw[lane] & 1u)),
                   hi = __ballot_sync(0xffffffffu, !(sh.raw[lane + 32] & 1u));
    const uint64_t none = ((uint64_t)hi << 32) | lo;
    if (group > (uint32_t)kTileRows && none) j0 = min(B, __ffsll((long long)none) - 1);
  }
  // from the rotated frame: C and the steps that targeted the pivot
  auto unrotate = [&](int j) {
    const uint64_t raw = rotl64(sh.raw[j], j), low = (1ull << j) - 1;
    sh.v[j] = raw & ~low;
    sh.mpiv[j] = raw & low;
  };
  if (t < j0 && (sh.raw[t] & 1u)) {
    unrotate(t);
    sh.piv[t] = sh.row[sh.index[t]];
  }
  if (j0 < B) {
    __syncthreads();
    if (warp == 0) {
      T.above_lo = T.above_hi = ~0u;
#pragma unroll
      for (int m = 0; m < kLaneRows; ++m) { T.lo[m] = (uint32_t)c0[m]; T.hi[m] = (uint32_t)(c0[m] >> 32); }
    }
    for (int s = 0; s < j0; ++s) tile_step(T, (uint32_t)sh.raw[s], (uint32_t)(sh.raw[s] >> 32));
    for (int j = j0, par = 0; j < B; ++j, par ^= 1) {
      uint32_t rl, rh;
      int index;
      tile_first(T, rl, rh, index);
      if (lane == 0) {
        sh.cand[par][warp] = (rl & 1u) ? kTileRows * warp + index : -1;
        sh.cand_v[par][warp] = ((uint64_t)rh << 32) | rl;
      }
      __syncthreads();
      int win = -1;
#pragma unroll
      for (int i = 7; i >= 0; --i)
        if (sh.cand[par][i] >= 0) win = i;
      uint64_t raw = 0;
      int64_t prow = kBlkNone;
      if (win >= 0) {
        raw = sh.cand_v[par][win];
        prow = sh.row[sh.cand[par][win]];
      } else if (total > (uint32_t)kGroup) {
        search_rest<P>(a, sh, off, nwin, j);
        if (sh.found) { raw = rotl64(sh.found_v, (64 - j) & 63); prow = sh.found_row; }
        __syncthreads();
      }
      tile_step(T, (uint32_t)raw, (uint32_t)(raw >> 32));
      if (t == 0) {
        sh.raw[j] = raw;
        sh.piv[j] = prow;
        unrotate(j);
      }
    }
  }
  __syncthreads();
  uint64_t prob = 0;  // steps with a pivot
  {
    const uint32_t lo = __ballot_sync(0xffffffffu, sh.v[lane] != 0), hi = __ballot_sync(0xffffffffu, sh.v[lane + 32] != 0);
    prob = ((uint64_t)hi << 32) | lo;
  }
  // M is linear in C: lin[t] = the steps that reduce unit vector t (bits stay
  // behind as above); next to it the products, the two halves of steps apart
  if (t < 64) {
    uint32_t lo = t < 32 ? 1u << t : 0, hi = t < 32 ? 0 : 1u << (t - 32);
#pragma unroll 8
    for (int s = 0; s < 32; ++s) {
      const uint64_t v = sh.v[s];
      const uint32_t on = 0u - ((lo >> s) & 1u);
      lo ^= (uint32_t)v & ~(1u << s) & on;
      hi ^= (uint32_t)(v >> 32) & on;
    }
#pragma unroll 8
    for (int s = 0; s < 32; ++s) hi ^= (uint32_t)(sh.v[s + 32] >> 32) & ~(1u << s) & (0u - ((hi >> s) & 1u));
    st.lin[t] = (((uint64_t)hi << 32) | lo) & prob;
  } else if (warp == 2) {
    half_products(sh.mpiv, prob, 0, sh.E1);
  } else if (warp == 3) {
    half_products(sh.mpiv, prob, 1, sh.E2);
  } else if (warp >= 6) {
    const int i = t - 192;
    st.piv[i] = sh.piv[i];
    st.cpiv[i] = sh.v[i];
    st.mpiv[i] = sh.mpiv[i];
    st.AD[i] = 0;
    st.G[i] = 0;
    if (i == 0) st.ntouched = 0;
  }
  __syncthreads();
  if (warp == 0) join_products(sh.mpiv, sh.E1, sh.E2, sh.tmp, st.E);
}

template <int P>
__global__ void __launch_bounds__(256, 4) blk_front_kernel(const FrontArgs a) {
  extern __shared__ uint32_t s_off[];  // a word per range (lazy symbolic pass)
  __shared__ ColRuns s_runs;
  __shared__ SymbolicShared s_sym;
  __shared__ SignShared s_sign;
  __shared__ uint32_t s_cnt[8];
  __shared__ uint64_t s_or[8];
  __shared__ bool s_last;
  chain_start();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, part = t % P;
  // the first blocks gather the next block's columns, the others sign the rows
  // of the previous one (nothing of which the symbolic pass needs)
  const uint32_t ranges = (uint32_t)(a.nrows / (256 / P));  // nrows is a multiple of 256
  const bool signs = blockIdx.x >= (a.B ? ranges : 0);
  const uint32_t range = signs && a.B ? blockIdx.x - ranges : blockIdx.x;
  const uint64_t r = (uint64_t)range * (256 / P) + t / P;
  if (signs) {
    const SignIn in = sign_load<P>(a, r, part);
    sign_tables(a, s_sign);
    __syncthreads();
    if (range == 0 && t < 64) sign_record(a, s_sign);
    sign_row<P>(a, s_sign, in, r, part);
    return;
  }
  if (t < 64) {
    build_runs(s_runs, a.window + a.i0, (int)a.B, a.n);
    if (range == 0 && t < (int)a.B && a.window[a.i0 + t] >= a.n) atomicOr(a.err, kErrBadQubit);
  }
  __syncthreads();
  const uint64_t c = or_parts<P>(gather_runs(s_runs, a.RX + r * a.rs, part, P));
  const bool stab = part == 0 && r >= 64ull * a.k && r < 64ull * a.k + a.n;
  if (part == 0) a.C[r] = c;
  if (!a.lazy) {
    const uint32_t ball = __ballot_sync(0xffffffffu, stab && (c & 1ull));
    if (lane == 0 && ball)
      atomicMin(reinterpret_cast<long long *>(&a.win->st[a.cur].slot[0]), (long long)(r + (__ffs(ball) - 1) / P));
    return;
  }
  // nonzero stabilizer rows of this range, in order, and the OR of their C
  const bool keep = stab && c != 0;
  const uint32_t ball = __ballot_sync(0xffffffffu, keep);
  uint64_t o = keep ? c : 0;
  for (int d = 16; d >= P; d >>= 1) o |= __shfl_xor_sync(0xffffffffu, o, d);
  if (lane == 0) { s_cnt[warp] = __popc(ball); s_or[warp] = o; }
  __syncthreads();
  uint32_t at = __popc(ball & ((1u << lane) - 1));
  for (int i = 0; i < warp; ++i) at += s_cnt[i];
  if (keep) {
    a.listC[(size_t)blockIdx.x * (256 / P) + at] = c;
    a.listRow[(size_t)blockIdx.x * (256 / P) + at] = (uint32_t)r;
  }
  if (t == 0) {
    uint32_t cnt = 0;
    uint64_t all = 0;
    for (int i = 0; i < 8; ++i) { cnt += s_cnt[i]; all |= s_or[i]; }
    a.cnt[blockIdx.x] = cnt;
    a.orC[blockIdx.x] = all;
    a.done[blockIdx.x] = 0;
  }
  __syncthreads();
  if (t == 0) {
    __threadfence();
    s_last = atomicAdd(&a.win->front_arrived, 1u) == ranges - 1;
    if (s_last) a.win->front_arrived = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  symbolic_pass<P>(a, s_sym, s_off, ranges);
}

// ---------------------------------------------------------------------------
// step-by-step symbolic pass (QS_FLAG_STEP_SYMBOLIC): reset, one launch per
// step over every row, then the products E
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(64) blk_step_reset_kernel(BlkState *st) {
  const int t = threadIdx.x;
  if (t < 3) st->slot[t] = kBlkNone;
  if (t == 0) st->ntouched = 0;
  st->piv[t] = kBlkNone; st->mpiv[t] = 0; st->cpiv[t] = 0;
  st->AD[t] = 0; st->G[t] = 0;
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

__global__ void __launch_bounds__(64) blk_step_finish_kernel(BlkState *st) {
  __shared__ uint64_t s_m[64];
  __shared__ uint32_t s_prob[2], E1[32], E2[32], tmp[32];
  const int t = threadIdx.x;
  s_m[t] = st->mpiv[t];
  const uint32_t ball = __ballot_sync(0xffffffffu, st->piv[t] != kBlkNone);
  if ((t & 31) == 0) s_prob[t >> 5] = ball;
  __syncthreads();
  half_products(s_m, ((uint64_t)s_prob[1] << 32) | s_prob[0], t >> 5, t < 32 ? E1 : E2);
  __syncthreads();
  if (t < 32) join_products(s_m, E1, E2, tmp, st->E);
}

// ---------------------------------------------------------------------------
// blk_middle: the pivot rows V_j with their phase sums (and in the last of
// those blocks their signs), next to the blocks that turn C into M, the bases
// and the list of rows the block changes
// ---------------------------------------------------------------------------
constexpr int kMidThreads = 256;
constexpr int kVW = 4;  // column words per chunk of pivot rows: a thread per (step, word)

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

// signs of V_j, four threads per step. The phase exponent of step j is
//   e_j = 2 r(p_j) + D_j + sum_{s in m_j} (2 rV_s + A_s) + 2 cross(m_j)   (mod 4),
// A and D the halves of AD, cross(m) = sum over s > t in m of G[s] bit t;
// everything but the 2 rV_s terms is independent of the other steps. With
// b_j = e'_j / 2 the signs solve rV = b + m rV (m strictly lower triangular), so
// rV_j = parity(E_j & b).
__device__ __forceinline__ void pivot_signs(const MiddleArgs &a) {
  __shared__ uint32_t sAD[64];
  __shared__ uint64_t sG[64];
  __shared__ uint32_t s_b[8];
  BlkState *st = a.st;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int j = t >> 2, part = t & 3;  // 16 bits of m each
  const int64_t p = j < (int)a.B ? st->piv[j] : kBlkNone;
  const uint64_t m = p != kBlkNone ? st->mpiv[j] : 0;
  const int rp = p != kBlkNone ? (int)((a.S[p >> 6] >> (p & 63)) & 1u) : 0;
  if (t < 64) {
    sAD[t] = __ldcg(&st->AD[t]);
    sG[t] = __ldcg(&st->G[t]) & ((1ull << t) - 1);
  }
  __syncthreads();
  int e = 0;
  uint64_t x = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int sidx = 16 * part + i;
    if ((m >> sidx) & 1ull) { e += (int)(sAD[sidx] & 3u); x ^= sG[sidx]; }
  }
  e += 2 * (__popcll(x & m) & 1);
  e += __shfl_xor_sync(0xffffffffu, e, 1);
  e += __shfl_xor_sync(0xffffffffu, e, 2);
  e = p != kBlkNone ? m4(e + 2 * rp + (int)(sAD[j] >> 16)) : 0;
  if (e & 1) atomicOr(a.err, kErrOddPhase);
  const uint32_t ball = __ballot_sync(0xffffffffu, part == 0 && (e >> 1));  // steps 8 warp .. + 7 at lanes 0, 4, ..
  if (lane == 0) {
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) b |= ((ball >> (4 * i)) & 1u) << i;
    s_b[warp] = b;
  }
  __syncthreads();
  if (t < 64) {
    uint64_t b = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) b |= (uint64_t)s_b[i] << (8 * i);
    st->rV[t] = __popcll(st->E[t] & b) & 1;
  }
}

// Pivot rows of one chunk of 4 column words: thread = (step j, word). The V rows
// are products over E_j of the original rows in shared memory (64 predicated
// XORs), and G[s][t] = z_{V_s} . x_{V_t} is one bit per word, thread (s, word)
// walking the 64 steps t; the four words of a step meet by shuffles. With 32-word
// chunks, lane = word and loops over the bits of E, the kernel took 21 us at 256
// qubits (4 of 32 lanes busy) and 22 us at 10,000 (5 chunks); now 4-word chunks
// fill the lanes at any size.
__device__ __forceinline__ void pivot_rows(const MiddleArgs &a, uint32_t chunk) {
  __shared__ ulonglong2 so[64][kVW], sv[64][kVW];  // (x, z) of the original and the V rows
  __shared__ bool s_last;
  BlkState *st = a.st;
  const uint32_t rs = a.rs;
  const int t = threadIdx.x, j = t >> 2, w = t & 3;
  const uint32_t u = chunk * kVW + w;  // rs is a multiple of 4
  // deterministic steps have no row and an empty E: their V row is zero
  const int64_t p = j < (int)a.B ? st->piv[j] : kBlkNone;
  const uint64_t E = st->E[j];
  ulonglong2 o = make_ulonglong2(0, 0);
  if (p != kBlkNone) o = make_ulonglong2(a.RX[(uint64_t)p * rs + u], a.RZ[(uint64_t)p * rs + u]);
  so[j][w] = o;
  __syncthreads();
  uint64_t x = 0, z = 0;
#pragma unroll 16
  for (int s = 0; s < 64; ++s) {
    const ulonglong2 q = so[s][w];
    const uint64_t on = spread(E, s);
    x ^= q.x & on;
    z ^= q.y & on;
  }
  sv[j][w] = make_ulonglong2(x, z);
  if (j < (int)a.B) {
    a.VX[(uint64_t)j * rs + u] = x;
    a.VZ[(uint64_t)j * rs + u] = z;
  }
  int av = __popcll(x & z), dv = __popcll(o.x & o.y) - av + 2 * (__popcll((z ^ o.y) & o.x) & 1);
#pragma unroll
  for (int d = 1; d < 4; d <<= 1) {
    av += __shfl_xor_sync(0xffffffffu, av, d);
    dv += __shfl_xor_sync(0xffffffffu, dv, d);
  }
  const uint32_t ad = (uint32_t)m4(av) | ((uint32_t)m4(dv) << 16);
  if (w == 0 && ad) atomicAdd(&st->AD[j], ad);
  __syncthreads();
  // bits t = 0..31 enter glo at the top and move down, then 32..63 ghi
  const uint32_t zl = (uint32_t)z, zh = (uint32_t)(z >> 32);
  uint32_t glo = 0, ghi = 0;
#pragma unroll 16
  for (int q = 0; q < 32; ++q) {
    const uint64_t x0 = sv[q][w].x, x1 = sv[q + 32][w].x;
    glo = __funnelshift_r(glo, __popc((zl & (uint32_t)x0) ^ (zh & (uint32_t)(x0 >> 32))), 1);
    ghi = __funnelshift_r(ghi, __popc((zl & (uint32_t)x1) ^ (zh & (uint32_t)(x1 >> 32))), 1);
  }
#pragma unroll
  for (int d = 1; d < 4; d <<= 1) {
    glo ^= __shfl_xor_sync(0xffffffffu, glo, d);
    ghi ^= __shfl_xor_sync(0xffffffffu, ghi, d);
  }
  const uint64_t g = ((uint64_t)ghi << 32) | glo;
  if (w == 0 && g) atomicXor(reinterpret_cast<unsigned long long *>(&st->G[j]), g);
  __syncthreads();
  if (t == 0) {
    __threadfence();
    s_last = atomicAdd(&a.win->middle_arrived, 1u) == a.chunks - 1;
    if (s_last) a.win->middle_arrived = 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  pivot_signs(a);
}

// M, base and the row list of 256 rows. A row that is neither a pivot nor a
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
  chain_start();
  if (blockIdx.x < a.chunks) pivot_rows(a, blockIdx.x);
  else list_rows(a, blockIdx.x - a.chunks);
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
    const uint4 e = __ldcg(list + j);
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

// Phase terms of one word (mod 4, summed over the row's words): with base row
// (xb, zb) and result (xf, zf) = V product * base,
//   |xb & zb| - |xf & zf| + 2 parity((zf ^ zb) & xb).
// -|b| = |~b| - 32 makes it a sum of four popcounts, which a full adder and a
// half adder fold into a ones and a twos word: two popcounts instead of five
// (a quarter-rate instruction).
__device__ __forceinline__ int phase_word(uint2 xb, uint2 zb, uint2 xf, uint2 zf) {
  const uint32_t a0 = xb.x & zb.x, a1 = xb.y & zb.y, n0 = ~(xf.x & zf.x), n1 = ~(xf.y & zf.y);
  const uint32_t d0 = xb.x & (zf.x ^ zb.x), d1 = xb.y & (zf.y ^ zb.y);
  const uint32_t s = a0 ^ a1 ^ n0, cy = (a0 & a1) | (a0 & n0) | (a1 & n0);
  const uint32_t t = ((s & n1) ^ cy) ^ d0 ^ d1;
  return __popc(s ^ n1) + 2 * __popc(t);
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
                                          uint32_t lane, const char *tb, uint32_t tq, uint8_t *Tp,
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
    xb = __ldcg(reinterpret_cast<const uint2 *>(VX) + (uint64_t)a.b * rs + word);
    zb = __ldcg(reinterpret_cast<const uint2 *>(VZ) + (uint64_t)a.b * rs + word);
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
  if (lane == 0) Tp[tp0 + r] = (uint8_t)(((v >> 6) + 2 * (v & 1)) & 3);
}

// 1,024 threads at 64 registers: 6.80 ms per dense block at 180k, against
// 7.46 ms with 768 threads (80 registers) and 9.55 ms with 512 (100). Fewer
// instructions per row do not help (measured: 64-bit multiply-adds for the row
// addresses, two popcounts instead of five): the pass waits on memory.
constexpr int kApplyThreads = 1024;

template <typename Idx>
__global__ void __launch_bounds__(kApplyThreads, 1)
blk_apply_kernel(uint64_t *__restrict__ RX, uint64_t *__restrict__ RZ, uint32_t rs, uint32_t nrows,
                 const uint32_t *qubits, int L, const uint64_t *VX, const uint64_t *VZ, const uint4 *list,
                 uint8_t *__restrict__ Tp, const BlkState *st) {
  extern __shared__ ulonglong2 T[];  // [kSmemEntries][kCW] of (x word, z word)
  __shared__ uint32_t s_tmem;
  chain_start();
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
        vv[b] = make_ulonglong2(__ldcg(VX + (uint64_t)st * rs + u0 + w), __ldcg(VZ + (uint64_t)st * rs + u0 + w));
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
        const uint2 x = __ldcg(reinterpret_cast<const uint2 *>(VX) + (uint64_t)st * rs + u0 + lane);
        const uint2 z = __ldcg(reinterpret_cast<const uint2 *>(VZ) + (uint64_t)st * rs + u0 + lane);
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

// The same pass for small tableaus, where building 226 KB of tables for a few
// hundred rows a block is most of the work and few blocks would run: 16 groups
// of 4 steps (256 entries) over chunks of CW = 4 or 8 column words, 16 or 32 KB
// of shared memory, 256 threads. CW lanes share a row, a warp has 32 / CW rows.
// Twice the lookups per word of the large variant, an eighth of its table build.
// Up to 6,144 qubits: 5,000 qubits take 14.7 us (large variant 16.2), 10,000 take
// 38.7 (28.5); 256 qubits 19 -> 6.1 us, 1,500 qubits 22.7 -> 7.2 us.
constexpr uint32_t kSmallApplyQubits = 6144;
constexpr int kSmallThreads = 256;

// the words of a listed row. bx, bz: this lane's word of row 0; a row is one
// 32 x 32 -> 64-bit multiply-add away from it
__device__ __forceinline__ void apply_fetch_small(ApplyRow &a, const ApplyMeta &m, const uint64_t *bx, const uint64_t *bz,
                                            uint32_t row_bytes, uint32_t nrows, bool ok) {
  a.r = m.r;
  a.b = m.b;
  a.lo = m.lo;
  a.hi = m.hi;
  a.x = a.z = make_uint2(0, 0);
  if (ok && m.r < nrows) {
    const uint64_t off = (uint64_t)m.r * row_bytes;
    a.x = *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(bx) + off);
    a.z = *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(bz) + off);
  }
}

template <int CW>
__global__ void __launch_bounds__(kSmallThreads)
blk_apply_small_kernel(uint64_t *__restrict__ RX, uint64_t *__restrict__ RZ, uint32_t rs, uint32_t nrows,
                       const uint32_t *qubits, int L, const uint64_t *VX, const uint64_t *VZ, const uint4 *list,
                       uint8_t *__restrict__ Tp,
                       const BlkState *st) {
  __shared__ ulonglong2 T[16 * 16][CW];
  chain_start();
  const uint32_t cnt = st->ntouched;
  const uint32_t t = threadIdx.x, w = t % CW, word = blockIdx.x * CW + w;
  const uint32_t group = t / CW, units = gridDim.y * (kSmallThreads / CW);
  if (cnt == 0) return;  // every outcome of the block is deterministic
  const bool ok = word < rs;
  // entry p of step group g = XOR of the V rows of p's bits; a thread builds its
  // word's entries of one group, each one row away from an earlier one
  for (uint32_t g = group; g < 16; g += kSmallThreads / CW) {
    ulonglong2 v[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int s = 4 * (int)g + b;
      v[b] = make_ulonglong2(0, 0);
      if (ok && s < L)
        v[b] = make_ulonglong2(__ldcg(VX + (uint64_t)s * rs + word), __ldcg(VZ + (uint64_t)s * rs + word));
    }
    ulonglong2 e[16];
    e[0] = make_ulonglong2(0, 0);
#pragma unroll
    for (int p = 1; p < 16; ++p) {
      const int b = p & 8 ? 3 : p & 4 ? 2 : p & 2 ? 1 : 0;
      e[p] = make_ulonglong2(e[p ^ (1 << b)].x ^ v[b].x, e[p ^ (1 << b)].y ^ v[b].y);
    }
#pragma unroll
    for (int p = 0; p < 16; ++p) T[16 * g + p][w] = e[p];
  }
  __syncthreads();
  const uint32_t row_bytes = rs * 8;
  uint64_t *bx = RX + word, *bz = RZ + word;
  uint8_t *tp = Tp + (uint64_t)blockIdx.x * nrows;
  const char *tw = reinterpret_cast<const char *>(&T[0][w]);
  ApplyRow a, nx;
  ApplyMeta m;
  // rows of a warp in step (the shuffles below), so the loop runs to the warp's last
  const uint32_t first = blockIdx.y * (kSmallThreads / CW), lane0 = first + (t & ~31u) / CW;
  uint32_t j = first + group;
  apply_meta(m, j, cnt, nrows, list);
  apply_fetch_small(a, m, bx, bz, row_bytes, nrows, ok);
  for (uint32_t j0 = lane0; j0 < cnt; j0 += units, j += units) {
    apply_meta(m, j + units, cnt, nrows, list);
    apply_fetch_small(nx, m, bx, bz, row_bytes, nrows, ok);
    uint2 xb = a.x, zb = a.z;
    if (a.b != kBaseOrig && a.b < kBasePivot && ok) {  // destabilizer replaced by V_b at step b
      xb = __ldcg(reinterpret_cast<const uint2 *>(VX) + (uint64_t)a.b * rs + word);
      zb = __ldcg(reinterpret_cast<const uint2 *>(VZ) + (uint64_t)a.b * rs + word);
    }
    uint4 f = make_uint4(xb.x, xb.y, zb.x, zb.y);
#pragma unroll
    for (int g = 0; g < 16; g += 2) {
      const uint32_t mw = g < 8 ? a.lo : a.hi;
      const int sh = 4 * (g & 7);
      const uint4 e0 = *reinterpret_cast<const uint4 *>(tw + (16 * g + ((mw >> sh) & 15)) * (16 * CW));
      const uint4 e1 = *reinterpret_cast<const uint4 *>(tw + (16 * (g + 1) + ((mw >> (sh + 4)) & 15)) * (16 * CW));
      acc3(f, e0, e1);
    }
    uint2 xf = make_uint2(f.x, f.y), zf = make_uint2(f.z, f.w);
    int v = phase_word(xb, zb, xf, zf);
    if (!ok) v = 0;
    if (a.b >= kBasePivot) {  // pivot row of step b: +-Z_q (sign set by blk_front_kernel)
      const uint32_t q = qubits[a.b - kBasePivot];
      const uint32_t bit = ((q >> 6) == word) ? 1u << (q & 31) : 0u;
      xf = make_uint2(0, 0);
      zf = (q & 32) ? make_uint2(0, bit) : make_uint2(bit, 0);
    }
    if (ok && a.r < nrows) {
      const uint64_t off = (uint64_t)a.r * row_bytes;
      *reinterpret_cast<uint2 *>(reinterpret_cast<char *>(bx) + off) = xf;
      *reinterpret_cast<uint2 *>(reinterpret_cast<char *>(bz) + off) = zf;
    }
#pragma unroll
    for (int d = 1; d < CW; d <<= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    if (w == 0 && a.r < nrows) tp[a.r] = (uint8_t)(v & 3);
    a = nx;
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
// in registers). With few outcomes the rows are split over blocks (about 152
// (range, outcome) pairs, as one outcome per launch had: up to 76 outcomes), whose
// totals the last block of a column chunk merges: cross ^= X_range . Z_before. What
// bounds an item is its walk over the rows, so 33 scattered outcomes without the
// split take longer (8.3 ms at 60,000 qubits) than one by one (3.6 ms).
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
  uint32_t *ranges;     // row ranges that are done, per group (three at most) and column chunk
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
  chain_start();
  const uint32_t nd = a.win->ndet;
  if (nd == 0) return;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const uint32_t groups = (nd + kDetGroup - 1) / kDetGroup;
  const uint32_t R = max(1u, min((uint32_t)kDetBlocks / nd, (a.n + kDetThreads - 1) / kDetThreads));
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
        a.det_x[((uint64_t)range * nd + g * kDetGroup + o) * a.rs + u] = X[j];
        a.det_z[((uint64_t)range * nd + g * kDetGroup + o) * a.rs + u] = Z[j];
      }
    }
    __threadfence();
    __syncthreads();
    if (R > 1) {
      if (t == 0) s_flag = atomicAdd(a.ranges + g * a.chunks + ch, 1u) == R - 1;
      __syncthreads();
      if (!s_flag) continue;
      __threadfence();
      for (uint32_t o = warp; o < d; o += 4) {  // last range of this chunk: merge the ranges
        uint64_t c = 0, xb = 0, zb = 0;
        if (in)
#pragma unroll 4
          for (uint32_t q = 0; q < R; ++q) {
            const uint64_t x = __ldcg(a.det_x + ((uint64_t)q * nd + g * kDetGroup + o) * a.rs + u),
                           z = __ldcg(a.det_z + ((uint64_t)q * nd + g * kDetGroup + o) * a.rs + u);
            c ^= x & zb;
            xb ^= x;
            zb ^= z;
          }
        const int v = __reduce_add_sync(0xffffffffu, 2 * (__popcll(c) & 1));
        if (lane == 0 && v) atomicAdd(a.acc + g * kDetGroup + o, v);
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
// column words per chunk of the apply pass: 4 or 8 (small variant) or 32
static uint32_t apply_words(const Layout &L) {
  if (L.n > kSmallApplyQubits) return kCW;
  return L.rs <= 4 ? 4 : 8;
}
static uint32_t apply_chunks(const Layout &L) { return (L.rs + apply_words(L) - 1) / apply_words(L); }

// device scratch of the blocked measurement
struct BlkScratch {
  uint8_t *zero;       // start of the part zeroed per window: win, acc, arrived, det_ranges
  size_t zero_bytes;
  BlkWindow *win;
  int32_t *acc;
  uint32_t *arrived, *det_ranges;
  uint64_t *C0, *C1, *M, *orC, *VX, *VZ;
  uint32_t *listRow, *cnt, *done, *det;
  int32_t *base;
  uint8_t *Tp;
  uint4 *list;
  size_t total;
};

// column chunks of blk_det
static uint32_t det_chunks(const Layout &L) { return (L.k + 31) / 32; }

// measurements per window (the capacity of det and acc)
static uint32_t blk_window_cap(const Layout &L) { return (uint32_t)L.nrows; }

// rows per block of blk_front
static uint32_t front_range(const Layout &L) { return L.nrows <= kFrontSplitRows ? 32 : 256; }

static BlkScratch blk_scratch(const Layout &L, void *scratch) {
  BlkScratch b;
  size_t off = 0;
  uint8_t *p = static_cast<uint8_t *>(scratch);
  auto take = [&](size_t bytes) {
    uint8_t *q = p + off;
    off += (bytes + 255) & ~size_t(255);
    return q;
  };
  const size_t cap = blk_window_cap(L), ranges = L.nrows / front_range(L);
  b.zero = p;
  b.win = reinterpret_cast<BlkWindow *>(take(sizeof(BlkWindow)));
  b.acc = reinterpret_cast<int32_t *>(take(cap * 4));
  b.arrived = reinterpret_cast<uint32_t *>(take((cap / kDetGroup + 1) * 4));
  b.det_ranges = reinterpret_cast<uint32_t *>(take(3 * (size_t)det_chunks(L) * 4));
  b.zero_bytes = off;
  b.C0 = reinterpret_cast<uint64_t *>(take(L.nrows * 8));
  b.C1 = reinterpret_cast<uint64_t *>(take(L.nrows * 8));
  b.M = reinterpret_cast<uint64_t *>(take(L.nrows * 8));
  b.base = reinterpret_cast<int32_t *>(take(L.nrows * 4));
  b.Tp = take((size_t)apply_chunks(L) * L.nrows);
  b.VX = reinterpret_cast<uint64_t *>(take(64ull * L.rs * 8));
  b.VZ = reinterpret_cast<uint64_t *>(take(64ull * L.rs * 8));
  b.list = reinterpret_cast<uint4 *>(take(L.nrows * 16));
  b.listRow = reinterpret_cast<uint32_t *>(take(L.nrows * 4));
  b.cnt = reinterpret_cast<uint32_t *>(take(ranges * 4));
  b.done = reinterpret_cast<uint32_t *>(take(ranges * 4));
  b.orC = reinterpret_cast<uint64_t *>(take(ranges * 8));
  b.det = reinterpret_cast<uint32_t *>(take(cap * 4));
  b.total = off;
  return b;
}

size_t blocked_scratch_bytes(const Layout &L) { return blk_scratch(L, nullptr).total; }

static std::atomic<uint64_t> g_blk_attr_set{0};

// Row ranges of the apply pass's grid. The large variant runs one block per SM
// (its tables fill shared memory and TMEM), so a grid just past a whole number
// of waves leaves SMs idle for one: at 10,000 qubits 195 blocks of 518 rows took
// 42 us and one wave of 150 takes 28.5. A wave costs a table build (about 4 us)
// and more waves even out the SMs (about 1.3 % at one, 0.4 % at three): with
// u_k the filled share of k waves, k minimises (1 + 0.013 / k) / u_k + 4 us k / T,
// T = 31 ns per row and chunk over the SMs. Dense blocks of 64, before (at least
// 512 rows per block, at most 32 waves) and after: 20,000 qubits 127 -> 97 us,
// 60,000 918 -> 845, 90,000 1,729 -> 1,570, 180,000 6,310 -> 6,180.
// The small variant holds several blocks per SM: three measured best at 3,000
// and 5,000 qubits (10.0 and 14.7 us; 24 us with the large variant's old grid).
static uint32_t apply_rows_y(const Dev &d, uint32_t chunks, uint32_t words) {
  const uint64_t nrows = d.L.nrows, sms = d.sms;
  if (words < kCW)
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(3 * sms / chunks, nrows / (kSmallThreads / words)));
  const double total_us = 0.031 * (double)nrows * chunks / (double)sms;
  uint32_t best = 1;
  double least = 1e30;
  for (uint32_t k = 1; k <= 12; ++k) {
    const uint64_t ry = k * sms / chunks;
    if (ry == 0) continue;
    const double cost = (1 + 0.013 / k) * (double)(k * sms) / (double)(ry * chunks) + 4.0 * k / total_us;
    if (cost < least) { least = cost; best = (uint32_t)ry; }
  }
  return best;
}

static cudaError_t measure_window_cap(const Dev &d, void *scratch, const uint32_t *window, uint32_t count,
                                      uint64_t m0, qs_key key, cudaStream_t s, int *launches) {
  const Layout &L = d.L;
  const BlkScratch b = blk_scratch(L, scratch);
  const uint32_t words = apply_words(L), chunks = apply_chunks(L), ranges = (uint32_t)(L.nrows / front_range(L)),
                 row_blocks = (uint32_t)(L.nrows / 256);  // nrows is a multiple of 256
  const size_t smem = (size_t)kSmemEntries * kEntryBytes;
  cudaError_t e = once_per_device(g_blk_attr_set, [&]() {
    cudaError_t x = cudaFuncSetAttribute(blk_apply_kernel<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (x == cudaSuccess)
      x = cudaFuncSetAttribute(blk_apply_kernel<uint64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (x == cudaSuccess)  // 4 bytes per range of 256 rows: 32 KB at n = 2^20, next to the static arrays
      x = cudaFuncSetAttribute(blk_front_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024);
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
  m.RX = d.RX; m.RZ = d.RZ; m.S = d.S; m.C = b.C0; m.nrows = L.nrows; m.rs = L.rs; m.k = L.k;
  m.chunks = L.rs / kVW;
  m.lazy = f.lazy;
  m.VX = b.VX; m.VZ = b.VZ; m.M = b.M; m.base = b.base; m.list = b.list; m.win = b.win; m.err = d.err;
  const uint32_t mid_blocks = m.chunks + row_blocks;  // kMidThreads rows each
  const uint32_t rows_y = apply_rows_y(d, chunks, words);
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
    const uint32_t blocks = (f.B ? ranges : 0) + (f.prev_B ? ranges : 0);
    const size_t off_bytes = f.lazy ? ranges * 4 : 0;
    if ((e = launch_chained(L.nrows <= kFrontSplitRows ? blk_front_kernel<8> : blk_front_kernel<1>, blocks, 256, off_bytes,
                            s, f)) != cudaSuccess)
      return e;
    ++nl;
    if (!f.lazy && f.B) {
      // the previous block's M and base are signed; C0 -> C1 -> C0 ...
      if ((e = cudaMemsetAsync(b.M, 0, L.nrows * 8, s)) != cudaSuccess) return e;
      if ((e = cudaMemsetAsync(b.base, 0xFF, L.nrows * 4, s)) != cudaSuccess) return e;  // kBaseOrig
      for (int j = 0; j < (int)f.B; ++j)
        blk_step_kernel<<<row_blocks, 256, 0, s>>>(L.nrows, L.n, L.k, j, (int)f.B, (j & 1) ? b.C1 : b.C0,
                                               (j & 1) ? b.C0 : b.C1, b.M, b.base, st);
      blk_step_finish_kernel<<<1, 64, 0, s>>>(st);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      nl += (int)f.B + 1;
    }
    tend(d.timer, kind, s);
    if (!f.B) break;
    m.B = f.B;
    m.st = st;
    tbegin(d.timer, QS_TIME_BLK_PIVOT_ROWS, s);
    if ((e = launch_chained(blk_middle_kernel, mid_blocks, kMidThreads, 0, s, m)) != cudaSuccess) return e;
    tend(d.timer, QS_TIME_BLK_PIVOT_ROWS, s);
    tbegin(d.timer, QS_TIME_BLK_APPLY, s);
    auto apply = [&](auto kernel, int threads, size_t bytes) {
      return launch_chained(kernel, dim3(chunks, rows_y), threads, bytes, s, d.RX, d.RZ, L.rs, (uint32_t)L.nrows,
                            window + i0, (int)f.B, b.VX, b.VZ, b.list, b.Tp, st);
    };
    if (words == 4)
      e = apply(blk_apply_small_kernel<4>, kSmallThreads, 0);
    else if (words == 8)
      e = apply(blk_apply_small_kernel<8>, kSmallThreads, 0);
    else if (!d.wide_offsets && (uint64_t)L.nrows * L.rs < (1ull << 32))
      e = apply(blk_apply_kernel<uint32_t>, kApplyThreads, smem);
    else
      e = apply(blk_apply_kernel<uint64_t>, kApplyThreads, smem);
    if (e != cudaSuccess) return e;
    tend(d.timer, QS_TIME_BLK_APPLY, s);
    nl += 2;
    if (d.timer && (i0 & 4095) == 4032) d.timer->resolve();  // completed event pairs go back to the pool
  }
  DetArgs t{};
  t.RX = d.RX; t.RZ = d.RZ; t.S = d.S; t.rs = L.rs; t.n = L.n; t.k = L.k; t.chunks = det_chunks(L);
  t.window = window; t.det = b.det; t.win = b.win; t.acc = b.acc; t.arrived = b.arrived; t.ranges = b.det_ranges;
  t.det_x = d.det_x; t.det_z = d.det_z; t.m0 = m0; t.record = d.record; t.err = d.err;
  // enough blocks for one outcome's ranges and for every group; blocks without an item leave at once
  const uint64_t most = std::max<uint64_t>(kDetBlocks, (count + kDetGroup - 1) / kDetGroup) * t.chunks;
  if (launches) *launches += nl + 1;
  return launch_chained(blk_det_kernel, (unsigned)std::min<uint64_t>(most, 12ull * d.sms), kDetThreads, 0, s, t);
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
