// k_potts.cu -- q = 4 Potts glass, H = -sum_<ij> J_ij delta(s_i, s_j),
// heat-bath update (IANUS_LAYOUT_U8X4).
//
// A 32-bit word holds one site of 4 samples (byte b = sample 4q+b, state
// 0..3), the counterpart of the paper's 2-bit Potts spins (Sec. 3.2); one
// Philox block supplies the 4 random words of the word.  The local counts
// n_k = sum_j J_ij [s_j == k] select a row of cumulative heat-bath thresholds
// (the look-up table of Sec. 3.2); the new state is the smallest k with
// r < T_k, else 3.  Words of one colour are contiguous (checkerboard-split
// order, Sec. 3.1).
//
// The row is linear in the counts (kPottsCoef, lattice.h), so each neighbour
// adds a term fixed by its state and coupling sign.  The terms of the 4
// samples are looked up together: state and sign make a nibble, two
// neighbours' nibbles fill the word, and a byte permute of an 8-entry table
// maps four nibbles at a time to the low (5 bits) or high digit of the term.
// Six terms of 5 bits fit a byte, so the digits are added as bytes.
//
// Bound: integer issue and, with few words a thread, the latency of a site's
// loads.  L=32, 128 x 2: 12 us per colour pass (19 us with the counts of each
// sample extracted one by one and the rows, 16 bytes in a 1 MB table, read
// through L1): 238 warp instructions per word against 408.
#include <algorithm>

#include "potts_words.cuh"

namespace ianus {

namespace {

constexpr int kBlock = 256;

// Low or high 5-bit digit of the term of (state, sign): byte state + 4 sign.
constexpr uint32_t potts_digit(int state, bool neg, int hi) {
  const uint32_t c = neg ? (kPottsRows - kPottsCoef[state]) & (kPottsRows - 1u) : kPottsCoef[state];
  return hi ? c >> 5 : c & 31u;
}
constexpr uint32_t potts_digits(bool neg, int hi) {
  return potts_digit(0, neg, hi) | potts_digit(1, neg, hi) << 8 | potts_digit(2, neg, hi) << 16 |
         potts_digit(3, neg, hi) << 24;
}

template <int D>
struct JModel {
  static constexpr uint32_t kRows = kPottsRows;
  uint32_t nf[D], nb[D];  // bit 2 of a byte: the coupling is -1

  __device__ __forceinline__ void prepare(const uint32_t* J, uint32_t N, const potts::Nbr<D>& n) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      nf[d] = __ldg(J + (size_t)d * N + n.self);
      nb[d] = __ldg(J + (size_t)d * N + n.bw[d]);
    }
  }

  __device__ __forceinline__ void rows(const uint32_t* sf, const uint32_t* sb, uint32_t* row) const {
    constexpr uint32_t lp = potts_digits(false, 0), ln = potts_digits(true, 0);
    constexpr uint32_t hp = potts_digits(false, 1), hn = potts_digits(true, 1);
    uint32_t l01 = 0, l23 = 0, h01 = 0, h23 = 0;  // samples 0 and 1, 2 and 3: two bytes each
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const uint32_t y = (sf[d] | (nf[d] & 0x04040404u)) + 16u * (sb[d] | (nb[d] & 0x04040404u));
      const uint32_t z = y >> 16;
      l01 += potts::prmt(lp, ln, y);
      h01 += potts::prmt(hp, hn, y);
      l23 += potts::prmt(lp, ln, z);
      h23 += potts::prmt(hp, hn, z);
    }
    // both neighbours of every direction, then low + 32 high, two samples per word
    auto fold = [](uint32_t x) { return (x & 0x00ff00ffu) + ((x >> 8) & 0x00ff00ffu); };
    const uint32_t r01 = (fold(l01) + 32u * fold(h01)) & 0x03ff03ffu;
    const uint32_t r23 = (fold(l23) + 32u * fold(h23)) & 0x03ff03ffu;
    row[0] = r01 & 0xffffu;
    row[1] = r01 >> 16;
    row[2] = r23 & 0xffffu;
    row[3] = r23 >> 16;
  }

  // a satisfied bond (equal states) counts -J
  static __device__ __forceinline__ void count_bond(uint32_t s, uint32_t sn, uint32_t J, uint32_t& good,
                                                    uint32_t& bad) {
    const uint32_t eq = potts::zero2(s ^ sn);
    good += eq & ~(J >> 1);
    bad += eq & (J >> 1);
  }
};

template <int D, int RT, bool KONE>
__global__ void __launch_bounds__(kBlock, RT == 2 ? 4 : 5) k_sweep_potts(const potts::Params p) {
  __shared__ uint4 tab[KONE ? kPottsRows : 1];
  potts::sweep_words<JModel<D>, D, RT, KONE>(p, tab);
}

__global__ void k_init_potts(uint32_t* spins, uint32_t* J, Geom geom, int Q4, int slots, int ferro,
                             PhiloxKeys keys) {
  const uint64_t total = (uint64_t)Q4 * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t q = (uint32_t)(idx / geom.N), i = (uint32_t)(idx - (uint64_t)q * geom.N);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint32_t j = split_index(geom, x, y, z);
    const uint32_t g = q >> 4, l0 = 4u * (q & 15u);
    for (int d = 0; d < geom.D; ++d) {
      const uint4 r = philox10(i, (uint32_t)d, (TAG_J << 28) | g, 0u, keys);
      const uint64_t wbits = (uint64_t)r.x | ((uint64_t)r.y << 32);
      uint32_t w = 0;
      for (int b = 0; b < 4; ++b) {
        const uint32_t neg = ferro ? 0u : (uint32_t)((wbits >> (l0 + b)) & 1ull);
        w |= (neg ? 0xFFu : 0x01u) << (8 * b);
      }
      J[((size_t)q * geom.D + d) * geom.N + j] = w;
    }
    for (int sg = 0; sg < slots; ++sg) {
      const uint4 r = philox10(i, 0u, (TAG_PINIT << 28) | ((uint32_t)sg << 16) | q, 0u, keys);
      spins[((size_t)sg * Q4 + q) * geom.N + j] =
          (r.x >> 30) | ((r.y >> 30) << 8) | ((r.z >> 30) << 16) | ((r.w >> 30) << 24);
    }
  }
}

constexpr int kPottsMeasIters = 32;

// Q = sum_i delta(s_i^0, s_i^1) between the replica-0 and replica-1
// configurations holding temperature k; stored in acc[s][k*R][6].
__global__ void __launch_bounds__(kBlock) k_overlap_potts(const uint32_t* __restrict__ spins,
                                                          const int32_t* __restrict__ slot_at, int64_t* acc,
                                                          uint32_t N, int S, int R, int K, int Q4, int slots) {
  const int qk = blockIdx.y;  // q * K + k
  const int q = qk / K, k = qk - q * K;
  const uint32_t* w0[4];
  const uint32_t* w1[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int s = 4 * q + b;
    const int t0 = s < S ? slot_at[((size_t)s * R + 0) * K + k] : k;
    const int t1 = s < S ? slot_at[((size_t)s * R + 1) * K + k] : k;
    w0[b] = spins + ((size_t)(t0 * R + 0) * Q4 + q) * N;
    w1[b] = spins + ((size_t)(t1 * R + 1) * Q4 + q) * N;
  }
  const uint32_t base = blockIdx.x * (uint32_t)(kBlock * kPottsMeasIters);
  long long v[4] = {0, 0, 0, 0};
  for (int it = 0; it < kPottsMeasIters; ++it) {
    const uint32_t j = base + (uint32_t)it * kBlock + threadIdx.x;
    if (j >= N) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) v[b] += (((w0[b][j] ^ w1[b][j]) >> (8 * b)) & 3u) == 0u ? 1 : 0;
  }
#pragma unroll
  for (int b = 0; b < 4; ++b)
    for (int off = 16; off > 0; off >>= 1) v[b] += __shfl_down_sync(0xffffffffu, v[b], off);
  if ((threadIdx.x & 31) == 0) {
    for (int b = 0; b < 4; ++b) {
      const int s = 4 * q + b;
      if (s < S)
        atomicAdd((unsigned long long*)&acc[((size_t)s * slots + (size_t)k * R) * kAccStride + 6],
                  (unsigned long long)v[b]);
    }
  }
}

__global__ void k_get_spins_potts(const uint32_t* spins, int8_t* out, Geom geom, int S, int Q4, int slots) {
  const uint64_t total = (uint64_t)S * slots * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int sg = (int)(rest % slots), s = (int)(rest / slots);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint32_t w = spins[((size_t)sg * Q4 + (s >> 2)) * geom.N + split_index(geom, x, y, z)];
    out[idx] = (int8_t)((w >> (8 * (s & 3))) & 3u);
  }
}

__global__ void k_set_spins_potts(uint32_t* spins, const int8_t* in, Geom geom, int S, int Q4, int slots) {
  const uint64_t total = (uint64_t)S * slots * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  // one thread per (slot, quad, site) so that bytes of one word are written together
  const uint64_t words = (uint64_t)slots * Q4 * geom.N;
  (void)total;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < words;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int q = (int)(rest % Q4), sg = (int)(rest / Q4);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    uint32_t* wp = &spins[((size_t)sg * Q4 + q) * geom.N + split_index(geom, x, y, z)];
    uint32_t w = *wp;
    for (int b = 0; b < 4; ++b) {
      const int s = 4 * q + b;
      if (s >= S) break;
      const uint32_t v = (uint32_t)in[((size_t)s * slots + sg) * geom.N + i] & 3u;
      w = (w & ~(0xFFu << (8 * b))) | (v << (8 * b));
    }
    *wp = w;
  }
}

__global__ void k_get_couplings_potts(const uint32_t* J, int8_t* out, Geom geom, int S) {
  const uint64_t total = (uint64_t)S * geom.D * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int d = (int)(rest % geom.D), s = (int)(rest / geom.D);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    const uint32_t w = J[((size_t)(s >> 2) * geom.D + d) * geom.N + split_index(geom, x, y, z)];
    out[idx] = (int8_t)(uint8_t)(w >> (8 * (s & 3)));
  }
}

__global__ void k_set_couplings_potts(uint32_t* J, const int8_t* in, Geom geom, int S, int Q4) {
  const uint64_t words = (uint64_t)Q4 * geom.D * geom.N;
  const uint32_t L = (uint32_t)geom.L;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < words;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int d = (int)(rest % geom.D), q = (int)(rest / geom.D);
    const int x = (int)(i % L), y = (int)((i / L) % L), z = geom.D == 3 ? (int)(i / (L * L)) : 0;
    uint32_t* wp = &J[((size_t)q * geom.D + d) * geom.N + split_index(geom, x, y, z)];
    uint32_t w = *wp;
    for (int b = 0; b < 4; ++b) {
      const int s = 4 * q + b;
      if (s >= S) break;
      const uint32_t v = (uint32_t)(uint8_t)in[((size_t)s * geom.D + d) * geom.N + i];
      w = (w & ~(0xFFu << (8 * b))) | (v << (8 * b));
    }
    *wp = w;
  }
}

inline unsigned grid_for(uint64_t total, unsigned block = 256, unsigned cap = 152u * 16u) {
  uint64_t g = (total + block - 1) / block;
  if (g > cap) g = cap;
  if (g == 0) g = 1;
  return (unsigned)g;
}

}  // namespace

cudaError_t launch_init_potts(Lattice& lat, int jmode) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_init_perm(lat, jmode);
  const int ferro = jmode == 1;  // Potts lattices take the J stream or J = +1
  k_init_potts<<<grid_for((uint64_t)lat.Q4 * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.spins, (uint32_t*)lat.J, lat.geom, lat.Q4, lat.slots, ferro, lat.keys);
  return cudaGetLastError();
}

cudaError_t launch_sweep_potts(Lattice& lat, int colour, uint64_t t) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_sweep_perm(lat, colour, t);
  const void* k[2][2][2] = {{{(const void*)k_sweep_potts<2, 1, false>, (const void*)k_sweep_potts<2, 1, true>},
                             {(const void*)k_sweep_potts<2, 2, false>, (const void*)k_sweep_potts<2, 2, true>}},
                            {{(const void*)k_sweep_potts<3, 1, false>, (const void*)k_sweep_potts<3, 1, true>},
                             {(const void*)k_sweep_potts<3, 2, false>, (const void*)k_sweep_potts<3, 2, true>}}};
  const int rt = lat.R % 2 == 0 ? 2 : 1;
  return potts::launch_sweep(lat, colour, t, k[lat.D - 2][rt - 1][lat.K == 1], rt, rt == 2 ? 4 : 5);
}

int sweep_chains_potts(const Lattice& lat) {
  const uint64_t pieces = (uint64_t)(lat.R % 2 == 0 ? lat.R / 2 : lat.R) * (uint64_t)lat.Q4;
  if (pieces < 4 || pieces * lat.geom.half * (uint64_t)lat.K < kChainSites) return 1;
  return 4;
}

cudaError_t launch_measure_potts(Lattice& lat, int want_q) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_measure_perm(lat, want_q);
  if (lat.D == 3)
    return potts::launch_measure(lat, want_q, potts::k_measure<JModel<3>, 3, 1>, potts::k_measure<JModel<3>, 3, 2>);
  return potts::launch_measure(lat, want_q, potts::k_measure<JModel<2>, 2, 1>, potts::k_measure<JModel<2>, 2, 2>);
}

cudaError_t launch_overlap_potts(Lattice& lat) {
  const uint32_t per_block = kBlock * kPottsMeasIters;
  dim3 gq((lat.N + per_block - 1) / per_block, (unsigned)(lat.Q4 * lat.K));
  k_overlap_potts<<<gq, kBlock, 0, lat.stream>>>((const uint32_t*)lat.spins, lat.slot_at, lat.acc, lat.N, lat.S,
                                                 lat.R, lat.K, lat.Q4, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_get_spins_potts(Lattice& lat, int8_t* dev_out) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_get_spins_perm(lat, dev_out);
  k_get_spins_potts<<<grid_for((uint64_t)lat.S * lat.slots * lat.N), 256, 0, lat.stream>>>(
      (const uint32_t*)lat.spins, dev_out, lat.geom, lat.S, lat.Q4, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_set_spins_potts(Lattice& lat, const int8_t* dev_in) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_set_spins_perm(lat, dev_in);
  k_set_spins_potts<<<grid_for((uint64_t)lat.slots * lat.Q4 * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.spins, dev_in, lat.geom, lat.S, lat.Q4, lat.slots);
  return cudaGetLastError();
}

cudaError_t launch_get_couplings_potts(Lattice& lat, int8_t* dev_out) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_get_couplings_perm(lat, dev_out);
  k_get_couplings_potts<<<grid_for((uint64_t)lat.S * lat.D * lat.N), 256, 0, lat.stream>>>(
      (const uint32_t*)lat.J, dev_out, lat.geom, lat.S);
  return cudaGetLastError();
}

cudaError_t launch_set_couplings_potts(Lattice& lat, const int8_t* dev_in) {
  if (lat.model == IANUS_POTTS4_PERM) return launch_set_couplings_perm(lat, dev_in);
  k_set_couplings_potts<<<grid_for((uint64_t)lat.Q4 * lat.D * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.J, dev_in, lat.geom, lat.S, lat.Q4);
  return cudaGetLastError();
}

}  // namespace ianus
