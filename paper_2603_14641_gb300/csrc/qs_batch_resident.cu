// Batched small circuits, one block per circuit with its tableau in shared
// memory for the whole program (n <= 640).
//
// The persistent batch kernel (qs_batch.cu) walks all circuits in lock-step with
// three grid barriers per measurement: 56 circuits of 50..1,000 qubits with
// 1,000 measurements each at most took 19 ms, nearly all of it barriers. A
// circuit of n <= 640 qubits fits one SM (2,080 ceil(n/64)^2 bytes, 208 KB at
// 640), and there everything is a block barrier away.
//
// Layout: the tableau is kept as 64 x 64-bit blocks (u, w), u = qubit / 64, w =
// packed row / 64, 65 words apart so that neighbouring blocks start one bank
// later. In gate phases word i of block (u, w) is word w of the column of qubit
// 64 u + i; in measurement phases it is word u of packed row 64 w + i. The
// layout switch transposes every block in place.
//   gates:   thread = (column word w, gate lane): a warp's lanes walk the words
//            of a gate's columns (conflict-free), signs stay in a register for
//            the whole run of layers, the next layer's records arrive by cp.async.
//   measure: thread = packed row (two at most), eight measurements per pass over
//            the rows, as in the blocked measurement of large tableaus: steps on
//            the rows' x bits at the eight qubits, in registers, one barrier each;
//            the pivot rows V_j, and tables of their products by four; then
//            each row takes two products. Rows are held as i^e X^x Z^z meanwhile:
//            a product adds the phases and twice one parity, z of the left
//            row with x of the right. What bounds it is shared memory: a row
//            word moves 20 eight-byte words per eight measurements where
//            a pass per measurement moved 6 for each: six circuits of 585 to 638
//            qubits, 1,270 measurements each at most, 3,313 -> 1,502 us.
//            Deterministic outcomes of a round are evaluated after it, one warp
//            each (measurements of a round commute).
#include <climits>

#include "qs_batch.cuh"
#include "qs_rules.cuh"

namespace qs {

constexpr uint32_t kListed = 1024;  // measurements whose qubits and coins are staged at a time
constexpr uint32_t kSteps = 8;      // measurements per pass over the rows
constexpr uint32_t kRows = 2;       // rows per thread at most: 128 ceil(n / 64) <= 2 threads
constexpr uint32_t kOwn = 0xFF, kBecomesZ = 0x10;  // a row's base: itself, V_j (j), or +-Z_q of step j (kBecomesZ + j)

__host__ __device__ constexpr size_t resident_blocks_words(uint32_t k) { return (size_t)k * 2 * k * 65; }

size_t batch_resident_smem(uint32_t n) {
  const uint32_t k = (n + 63) / 64;
  // tableau; V rows and two tables of 16 products; signs and phases; gate records; staged measurements
  return 2 * resident_blocks_words(k) * 8 + (size_t)(2 * kSteps + 64) * k * 8 + 4 * k * 8 + 2 * (size_t)n * 8 +
         kListed * (2 + 1 + 2) + 64;
}

// rows lane (lo) and lane + 32 (hi) of a 64 x 64 bit block -> its transpose
__device__ __forceinline__ void transpose_block(uint64_t &lo, uint64_t &hi, int lane) {
  {
    const uint64_t t = ((lo >> 32) ^ hi) & 0x00000000FFFFFFFFull;
    lo ^= t << 32;
    hi ^= t;
  }
  const uint64_t masks[5] = {0x0000FFFF0000FFFFull, 0x00FF00FF00FF00FFull, 0x0F0F0F0F0F0F0F0Full,
                             0x3333333333333333ull, 0x5555555555555555ull};
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int j = 16 >> s;
    const uint64_t m = masks[s];
    const uint64_t pl = __shfl_xor_sync(0xffffffffu, lo, j), ph = __shfl_xor_sync(0xffffffffu, hi, j);
    if ((lane & j) == 0) {
      lo ^= (((lo >> j) ^ pl) & m) << j;
      hi ^= (((hi >> j) ^ ph) & m) << j;
    } else {
      lo ^= ((pl >> j) ^ lo) & m;
      hi ^= ((ph >> j) ^ hi) & m;
    }
  }
}

__global__ void __launch_bounds__(1024)
batch_resident_kernel(const BCirc *__restrict__ circs, const uint32_t *__restrict__ ids, uint32_t round_limit,
                      uint32_t *__restrict__ err) {
  extern __shared__ uint64_t sm[];
  __shared__ uint32_t s_cand[2][32], s_p[kSteps], s_mp[kSteps], s_ndet;
  __shared__ uint8_t s_ve[kSteps], s_te[32];
  const BCirc &C = circs[ids[blockIdx.x]];
  const uint32_t n = C.n, k = C.k, KB = 2 * k, T = blockDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const size_t words = resident_blocks_words(k);
  uint64_t *X = sm, *Z = X + words;
  uint64_t *VX = Z + words, *VZ = VX + kSteps * k;        // V_j word u at j k + u
  uint64_t *TX = VZ + kSteps * k, *TZ = TX + 32 * k;      // product m of nibble h, word u at (h k + u) 16 + m
  uint32_t *S = reinterpret_cast<uint32_t *>(TZ + 32 * k);  // 2 KB words of 32 rows
  uint32_t *E = S + 2 * KB;                               // measurement phases: low bits of the phases
  uint2 *gbuf = reinterpret_cast<uint2 *>(E + 2 * KB);    // two layers of gate records
  uint16_t *s_q = reinterpret_cast<uint16_t *>(gbuf + 2 * (size_t)n);
  uint16_t *s_det = s_q + kListed;
  uint8_t *s_coin = reinterpret_cast<uint8_t *>(s_det + kListed);
  auto at = [KB](uint32_t u, uint32_t w, uint32_t i) { return (u * KB + w) * 65 + i; };

  // D_i = X_i, S_i = Z_i, no signs (Alg. 2 init)
  for (size_t i = t; i < 2 * words; i += T) sm[i] = 0;
  for (uint32_t i = t; i < 4 * KB; i += T) S[i] = 0;  // E with it
  for (uint32_t i = t; i < 64; i += T) s_cand[i >> 5][i & 31] = UINT_MAX;
  uint32_t buf = 0;
  __syncthreads();
  for (uint32_t q = t; q < n; q += T) {
    X[at(q >> 6, q >> 6, q & 63)] = 1ull << (q & 63);
    Z[at(q >> 6, k + (q >> 6), q & 63)] = 1ull << (q & 63);
  }
  __syncthreads();

  auto transpose_all = [&]() {
    for (uint32_t b = warp; b < 2 * k * KB; b += T >> 5) {
      uint64_t *p = sm + (size_t)b * 65;  // X and Z blocks lie one after the other
      uint64_t lo = p[lane], hi = p[lane + 32];
      transpose_block(lo, hi, (int)lane);
      p[lane] = lo;
      p[lane + 32] = hi;
    }
    __syncthreads();
  };

  // Between sign and phase of the rows: a row is (-1)^s prod i^(xz) X^x Z^z in gate
  // phases and i^(2 S + E) X^x Z^z in measurement phases.
  auto convert = [&](bool back) {
    for (uint32_t r0 = 0; r0 < 64 * KB; r0 += T) {
      const uint32_t row = r0 + t, w = row >> 6, i = row & 63;
      if (row - lane >= 64 * KB) break;
      uint32_t y = 0;
      for (uint32_t u = 0; u < k; ++u) y += __popcll(X[at(u, w, i)] & Z[at(u, w, i)]);
      const uint32_t one = __ballot_sync(0xffffffffu, y & 1), two = __ballot_sync(0xffffffffu, y >> 1 & 1);
      if (lane == 0) {
        // 2 S + y, and back 2 S + E - y, where E is y mod 2 for a Hermitian row
        S[row >> 5] ^= two;
        if (back && E[row >> 5] != one) atomicOr(err, kErrOddPhase);
        E[row >> 5] = back ? 0 : one;
      }
    }
    __syncthreads();
  };

  const uint32_t gate_lanes = T / KB, gw = t % KB, gl = t / KB;
  const uint32_t rounds = min(C.nrounds, round_limit);
  for (uint32_t r = 0; r < rounds; ++r) {
    const uint32_t l0 = C.rl[r], l1 = C.rl[r + 1];
    if (l1 > l0) {
      // records of a layer: g[a .. b) -> buffer, one 8-byte copy per thread and record
      auto fetch = [&](int64_t a, int64_t b, uint2 *dst) {
        for (int64_t g = a + t; g < b; g += T) {
          const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + (g - a));
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(C.gates + 2 * g) : "memory");
        }
      };
      int64_t a = C.lptr[l0], b = C.lptr[l0 + 1], c = l0 + 2 <= l1 ? C.lptr[l0 + 2] : b;
      fetch(a, b, gbuf);
      uint64_t sacc = 0;
      for (uint32_t l = l0; l < l1; ++l) {
        const int64_t after = l + 3 <= l1 ? __ldg(C.lptr + l + 3) : c;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();  // this layer's records are here; the previous layer is done with its buffer
        if (l + 1 < l1) fetch(b, c, gbuf + ((l + 1 - l0) & 1) * (size_t)n);
        const uint2 *rec = gbuf + ((l - l0) & 1) * (size_t)n;
        const uint32_t cnt = (uint32_t)(b - a);
        if (gl < gate_lanes)
          for (uint32_t g = gl; g < cnt; g += gate_lanes) {
            const uint2 q = rec[g];
            const uint32_t type = q.x >> 24, qa = q.x & 0xFFFFFFu, qb = q.y;
            const bool two = type >= QS_CX && type <= QS_ISWAP;
            if (qa >= n || type >= QS_NUM_GATE_TYPES || (two && (qb >= n || qb == qa))) {
              atomicOr(err, kErrBadGate);
              continue;
            }
            const uint32_t ia = at(qa >> 6, gw, qa & 63), ib = two ? at(qb >> 6, gw, qb & 63) : ia;
            uint64_t xa = X[ia], za = Z[ia], xb = 0, zb = 0;
            if (two) { xb = X[ib]; zb = Z[ib]; }
            rule<true>(type, xa, za, xb, zb, sacc);
            if ((kWritesXa >> type) & 1) X[ia] = xa;
            if ((kWritesZa >> type) & 1) Z[ia] = za;
            if ((kWritesXb >> type) & 1) X[ib] = xb;
            if ((kWritesZb >> type) & 1) Z[ib] = zb;
          }
        a = b; b = c; c = after;
      }
      if (gl < gate_lanes) {
        if ((uint32_t)sacc) atomicXor(S + 2 * gw, (uint32_t)sacc);
        if ((uint32_t)(sacc >> 32)) atomicXor(S + 2 * gw + 1, (uint32_t)(sacc >> 32));
      }
      __syncthreads();
    }
    const uint32_t m0 = C.rm[r], m1 = C.rm[r + 1];
    if (m1 == m0) continue;
    transpose_all();
    convert(false);
    for (uint32_t base = m0; base < m1; base += kListed) {
      const uint32_t cnt = min(kListed, m1 - base);
      for (uint32_t j = t; j < cnt; j += T) {
        s_q[j] = (uint16_t)C.qubits[base + j];
        s_coin[j] = (uint8_t)(philox4x64_10(base + j, C.shot, 0, 0, C.seed, kCoinKey).v[0] & 1u);
      }
      if (t == 0) s_ndet = 0;
      __syncthreads();
      for (uint32_t j0 = 0; j0 < cnt; j0 += kSteps) {
        const uint32_t nb = min(kSteps, cnt - j0);
        // own rows: x bits at the block's qubits, steps that multiply into the row, base
        uint32_t cx[kRows], hit[kRows], base_of[kRows];
#pragma unroll
        for (uint32_t m = 0; m < kRows; ++m) {
          const uint32_t row = t + m * T, w = row >> 6, i = row & 63;
          cx[m] = hit[m] = 0;
          base_of[m] = kOwn;
          if (row < 64 * KB)
            for (uint32_t j = 0; j < nb; ++j) {
              const uint32_t q = s_q[j0 + j];
              cx[m] |= (uint32_t)((X[at(q >> 6, w, i)] >> (q & 63)) & 1ull) << j;
            }
        }
        for (uint32_t j = 0; j < nb; ++j) {
          uint32_t cand = UINT_MAX;  // smallest stabilizer row with bit j, with its words
#pragma unroll
          for (uint32_t m = 0; m < kRows; ++m) {
            const uint32_t row = t + m * T;
            if (row >= 64 * k && (cx[m] >> j & 1)) cand = min(cand, row << 16 | hit[m] << 8 | cx[m]);
          }
          s_cand[buf][warp] = __reduce_min_sync(0xffffffffu, cand);
          __syncthreads();
          const uint32_t piv = __reduce_min_sync(0xffffffffu, s_cand[buf][lane]);
          buf ^= 1;
          if (t == 0) {
            s_p[j] = piv == UINT_MAX ? UINT_MAX : piv >> 16;
            s_mp[j] = piv >> 8 & 0xFF;
            if (piv == UINT_MAX)
              s_det[s_ndet++] = (uint16_t)(j0 + j);  // nothing changes; evaluated after the list
            else
              C.record[base + j0 + j] = s_coin[j0 + j];
          }
          if (piv == UINT_MAX) continue;
          const uint32_t p = piv >> 16, pd = p - 64 * k;
#pragma unroll
          for (uint32_t m = 0; m < kRows; ++m) {
            const uint32_t row = t + m * T;
            if (row == pd) {  // D_{p-n} <- S_p
              cx[m] = piv & 0xFF;
              hit[m] = 0;
              base_of[m] = j;
            } else if (row == p) {
              cx[m] = hit[m] = 0;
              base_of[m] = kBecomesZ + j;
            } else if (cx[m] >> j & 1) {
              cx[m] ^= piv & 0xFF;
              hit[m] |= 1u << j;
            }
          }
        }
        __syncthreads();
        // V_j = the pivot row as step j finds it (left products; V rows commute), lane = word
        if (warp == 0) {
          uint64_t vx[kSteps], vz[kSteps];
          uint32_t ve[kSteps];
#pragma unroll
          for (uint32_t j = 0; j < kSteps; ++j) {
            vx[j] = vz[j] = 0;
            ve[j] = 0;
            const uint32_t p = j < nb ? s_p[j] : UINT_MAX;
            if (p != UINT_MAX) {
              const uint32_t mp = s_mp[j];
              uint64_t x = 0, z = 0, cross = 0;
              if (lane < k) {
                x = X[at(lane, p >> 6, p & 63)];
                z = Z[at(lane, p >> 6, p & 63)];
              }
              uint32_t e = 2 * (S[p >> 5] >> (p & 31) & 1) + (E[p >> 5] >> (p & 31) & 1);
#pragma unroll
              for (uint32_t i = 0; i < kSteps; ++i)
                if (i < j && (mp >> i & 1)) {
                  cross ^= vz[i] & x;
                  x ^= vx[i];
                  z ^= vz[i];
                  e += ve[i];
                }
              vx[j] = x;
              vz[j] = z;
              ve[j] = e + 2 * (__popc(__ballot_sync(0xffffffffu, __popcll(cross) & 1)) & 1);
            }
            if (lane < k) {
              VX[j * k + lane] = vx[j];
              VZ[j * k + lane] = vz[j];
            }
            if (lane == 0) s_ve[j] = ve[j] & 3;
          }
        }
        __syncthreads();
        for (uint32_t m = warp; m < 32; m += T >> 5) {  // a warp per product of up to four V, lane = word
          uint64_t x = 0, z = 0, cross = 0;
          uint32_t e = 0;
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i)
            if (m >> i & 1) {
              const uint32_t j = (m >> 4) * 4 + i;
              const uint64_t ax = lane < k ? VX[j * k + lane] : 0, az = lane < k ? VZ[j * k + lane] : 0;
              cross ^= az & x;
              x ^= ax;
              z ^= az;
              e += s_ve[j];
            }
          e += 2 * (__popc(__ballot_sync(0xffffffffu, __popcll(cross) & 1)) & 1);
          if (lane < k) {
            TX[((m >> 4) * k + lane) * 16 + (m & 15)] = x;
            TZ[((m >> 4) * k + lane) * 16 + (m & 15)] = z;
          }
          if (lane == 0) s_te[m] = e & 3;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t m = 0; m < kRows; ++m) {
          const uint32_t row = t + m * T, w = row >> 6, i = row & 63;
          if (row - lane >= 64 * KB) break;  // uniform over the warp
          uint32_t e = 2 * (S[row >> 5] >> lane & 1) + (E[row >> 5] >> lane & 1);
          if (base_of[m] != kOwn && base_of[m] >= kBecomesZ) {
            const uint32_t j = j0 + base_of[m] - kBecomesZ, q = s_q[j];
            for (uint32_t u = 0; u < k; ++u) {
              X[at(u, w, i)] = 0;
              Z[at(u, w, i)] = u == (q >> 6) ? 1ull << (q & 63) : 0ull;
            }
            e = 2 * s_coin[j];
          } else if (hit[m] || base_of[m] != kOwn) {
            const bool own = base_of[m] == kOwn;
            const uint64_t *lx = TX + (hit[m] & 15), *hx = TX + 16 * k + (hit[m] >> 4);
            const uint64_t *lz = TZ + (hit[m] & 15), *hz = TZ + 16 * k + (hit[m] >> 4);
            uint64_t cross = 0;
#pragma unroll 2
            for (uint32_t u = 0; u < k; ++u) {
              uint64_t x = own ? X[at(u, w, i)] : VX[base_of[m] * k + u], z = own ? Z[at(u, w, i)] : VZ[base_of[m] * k + u];
              cross ^= lz[16 * u] & x;
              x ^= lx[16 * u];
              z ^= lz[16 * u];
              cross ^= hz[16 * u] & x;
              X[at(u, w, i)] = x ^ hx[16 * u];
              Z[at(u, w, i)] = z ^ hz[16 * u];
            }
            e = (own ? e : s_ve[base_of[m]]) + s_te[hit[m] & 15] + s_te[16 + (hit[m] >> 4)] +
                2 * (__popcll(cross) & 1);
          }
          const uint32_t lo = __ballot_sync(0xffffffffu, e & 1), hi = __ballot_sync(0xffffffffu, e >> 1 & 1);
          __syncwarp();
          if (lane == 0) {
            S[row >> 5] = hi;
            E[row >> 5] = lo;
          }
        }
      }
      __syncthreads();
      // deterministic outcomes: (-1)^m Z_q = prod of S_i over D_i with x_iq = 1, a warp each, lane = word
      for (uint32_t d = warp; d < s_ndet; d += T >> 5) {
        const uint32_t j = s_det[d], q = s_q[j];
        uint64_t px = 0, pz = 0, cross = 0;
        int cnt4 = 0;
        for (uint32_t w = 0; w < k; ++w) {
          const uint64_t *col = X + at(q >> 6, w, 0);
          const uint32_t lo = __ballot_sync(0xffffffffu, (col[lane] >> (q & 63)) & 1ull);
          const uint32_t hi = __ballot_sync(0xffffffffu, (col[lane + 32] >> (q & 63)) & 1ull);
          uint64_t m = ((uint64_t)hi << 32) | lo;
          if (lane == 0)
            cnt4 += 2 * (__popc(lo & S[2 * (k + w)]) + __popc(hi & S[2 * (k + w) + 1])) +
                    __popc(lo & E[2 * (k + w)]) + __popc(hi & E[2 * (k + w) + 1]);
          while (m) {
            const uint32_t i = (uint32_t)__ffsll((long long)m) - 1;
            m &= m - 1;
            if (lane < k) {
              const uint64_t x = X[at(lane, k + w, i)], z = Z[at(lane, k + w, i)];
              cross ^= x & pz;
              px ^= x;
              pz ^= z;
            }
          }
        }
        const int e = __reduce_add_sync(0xffffffffu, cnt4 + 2 * (__popcll(cross) & 1)) & 3;
        const uint64_t want = lane == (q >> 6) ? 1ull << (q & 63) : 0ull;
        if (lane < k && (px != 0 || pz != want)) atomicOr(err, kErrDetProduct);
        if (lane == 0) {
          if (e & 1) atomicOr(err, kErrOddPhase);
          C.record[base + j] = (uint8_t)(e >> 1);
        }
      }
      __syncthreads();
    }
    convert(true);
    transpose_all();
  }
  // the column-major tableau with its zero padding
  for (size_t i = t; i < (size_t)C.ncols * C.cs; i += T) {
    const uint32_t q = (uint32_t)(i / C.cs), w = (uint32_t)(i % C.cs);
    const bool in = q < 64 * k && w < KB;
    C.X[i] = in ? X[at(q >> 6, w, q & 63)] : 0;
    C.Z[i] = in ? Z[at(q >> 6, w, q & 63)] : 0;
  }
  for (uint32_t w = t; w < C.cs; w += T) C.S[w] = w < KB ? ((uint64_t)S[2 * w + 1] << 32) | S[2 * w] : 0;
}

cudaError_t launch_batch_resident(const BCirc *circs, const uint32_t *ids, uint32_t count, uint32_t threads,
                                  size_t smem, uint32_t round_limit, uint32_t *err, cudaStream_t s) {
  static std::atomic<uint64_t> attr_set{0};
  cudaError_t e = once_per_device(attr_set, []() {
    return cudaFuncSetAttribute(batch_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)batch_resident_smem(kResidentMaxQubits));
  });
  if (e != cudaSuccess) return e;
  batch_resident_kernel<<<count, threads, smem, s>>>(circs, ids, round_limit, err);
  return cudaGetLastError();
}

}  // namespace qs
