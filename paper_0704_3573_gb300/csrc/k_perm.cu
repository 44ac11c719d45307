// k_perm.cu -- the glassy Potts model of Eq. (3),
// H = -sum_<ij> delta(s_i, pi_ij(s_j)), with quenched permutation couplings
// pi_ij of (0,1,2,3), heat bath, in 2, 3 or 4 dimensions (Sec. 4.2 runs it in
// 3D and 4D).
//
// Storage follows IANUS_LAYOUT_U8X4: a 32-bit word holds one site of 4
// samples (byte b = sample 4q+b, state 0..3); a coupling word holds the 8-bit
// permutation codes pi(0) | pi(1) << 2 | pi(2) << 4 | pi(3) << 6 of the 4
// samples (the paper's 8-bit Potts couplings, Sec. 3.2).  Sites are in the
// checkerboard-split order of Sec. 3.1 generalised to D dimensions: word
// (2 row + c) h + x / 2, where row = i / L collects the coordinates after x
// and c is the colour, so every neighbour of a colour-c word is a colour-(1-c)
// word with the same x / 2 (or x / 2 +- 1 along x).
//
// Update: each of the 2D bonds is satisfied by exactly one state k of s_i,
// k = pi(s_j) for a forward bond (i, j = i + e_d) and k = pi^-1(s_j) for a
// backward bond (j = i - e_d, i); the counts (n0, n1, n2) give a row of
// cumulative heat-bath thresholds (perm_row, lattice.h).  The row is linear
// in the counts, so it is summed over the bonds for the 4 samples of a word at
// once, one byte each (4D: two bytes, then 16 bits):
//   forward: pi(s_j) by two byte-wise selects of the code's fields on the bits
//     of s_j; the sums of its bits t0, t1 and t0 t1 give the three counts;
//   backward: code XOR s_j in every field is zero in field pi^-1(s_j) only;
//     those one-hot fields are added as 2-bit numbers.
//
// Bound: integer issue.  3D L=32, 256 x 2: 21.6 us per colour pass (44 us with
// each sample's bonds done one by one, pi^-1 by a shared 256-byte table); 4D
// L=16, 256 x 2: 51 us (102 us).
#include <algorithm>

#include "potts_words.cuh"

namespace ianus {

namespace {

constexpr int kBlock = 256;
constexpr uint32_t kIdentityCode = 0xE4u;  // (0, 1, 2, 3)

// Natural index -> split index, any D.
__device__ __forceinline__ uint32_t perm_split(const Geom& g, uint32_t i) {
  const uint32_t L = (uint32_t)g.L;
  const uint32_t x = i % L, row = i / L;
  uint32_t r = row, psum = x;
  for (int d = 1; d < g.D; ++d) {
    psum += r % L;
    r /= L;
  }
  return (2u * row + (psum & 1u)) * (uint32_t)g.h + x / 2u;
}

// Code of permutation number p (lexicographic): digit p / 6 picks the first
// value among the four, then p / 2 mod 3 among the remaining three, etc.
__device__ __forceinline__ uint32_t perm_code_of(uint32_t p) {
  uint32_t pool = kIdentityCode;  // remaining values, increasing, 2 bits each
  uint32_t code = 0;
  const uint32_t wgt[3] = {6u, 2u, 1u};
#pragma unroll
  for (int pos = 0; pos < 3; ++pos) {
    const uint32_t pick = p / wgt[pos];
    p -= pick * wgt[pos];
    code |= ((pool >> (2u * pick)) & 3u) << (2 * pos);
    const uint32_t low = pool & ((1u << (2u * pick)) - 1u);
    pool = low | ((pool >> (2u * pick + 2u)) << (2u * pick));
  }
  return code | ((pool & 3u) << 6);
}

// pi(s) in the low two bits of each byte (the rest is not defined), from the
// codes c of 4 samples.
__device__ __forceinline__ uint32_t perm_apply(uint32_t c, uint32_t s) {
  // a byte of ones where bit 1 (bit 0) of the state is set: sign replication of the shifted byte
  const uint32_t m1 = potts::prmt(s << 6, 0u, 0xBA98u), m0 = potts::prmt(s << 7, 0u, 0xBA98u);
  const uint32_t c1 = (m1 & (c >> 4)) | (~m1 & c);
  return (m0 & (c1 >> 2)) | (~m0 & c1);
}

template <int D>
struct PermModel {
  static constexpr uint32_t kRows = D == 4 ? 592u : 256u;
  uint32_t cf[D], cb[D];

  __device__ __forceinline__ void prepare(const uint32_t* J, uint32_t N, const potts::Nbr<D>& n) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      cf[d] = __ldg(J + (size_t)d * N + n.self);
      cb[d] = __ldg(J + (size_t)d * N + n.bw[d]);
    }
  }

  __device__ __forceinline__ void rows(const uint32_t* sf, const uint32_t* sb, uint32_t* row) const {
    using potts::kOnes;
    uint32_t t0 = 0, t1 = 0, t01 = 0;  // forward: sums of the bits of pi(s_j)
    uint32_t z[D];                     // backward: bit 2k set where pi^-1(s_j) = k
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const uint32_t t = perm_apply(cf[d], sf[d]), h = t >> 1;
      t0 += t & kOnes;
      t1 += h & kOnes;
      t01 += t & h & kOnes;
      const uint32_t x = cb[d] ^ (sb[d] * 0x55u);
      z[d] = ~(x | (x >> 1)) & 0x55555555u;
    }
    uint32_t zs = z[0] + z[1];  // 2-bit fields: up to three of them add without overflow
    if (D >= 3) zs += z[2 % D];
    if constexpr (D < 4) {
      // n0 + 37 n1 + 16 n2 per byte: a forward bond adds 1 + 36 t0 + 15 t1 - 52 t0 t1
      const uint32_t idx = (zs & 0x33333333u) + 37u * ((zs >> 2) & 0x03030303u) + (uint32_t)D * kOnes + 36u * t0 +
                           15u * t1 - 52u * t01;
      row[0] = idx & 0xffu;
      row[1] = (idx >> 8) & 0xffu;
      row[2] = (idx >> 16) & 0xffu;
      row[3] = idx >> 24;
    } else {
      const uint32_t e = (zs & 0x33333333u) + (z[3 % D] & 0x33333333u);                  // n0, n2 as nibbles
      const uint32_t o = ((zs >> 2) & 0x33333333u) + ((z[3 % D] >> 2) & 0x33333333u);    // n1, n3
      // n0 + 9 n1 and n2 per byte; a forward bond adds 1 + 8 t0 - t1 - 8 t0 t1 and t1 - t0 t1
      const uint32_t a = (e & 0x0f0f0f0fu) + 9u * (o & 0x0f0f0f0fu) + 4u * kOnes + 8u * (t0 - t01) - t1;
      const uint32_t b = ((e >> 4) & 0x0f0f0f0fu) + t1 - t01;
      const uint32_t r02 = (a & 0x00ff00ffu) + 73u * (b & 0x00ff00ffu);
      const uint32_t r13 = ((a >> 8) & 0x00ff00ffu) + 73u * ((b >> 8) & 0x00ff00ffu);
      // permutation codes keep rows below kRows; the bound holds for any bytes
      row[0] = min(r02 & 0xffffu, kRows - 1u);
      row[1] = min(r13 & 0xffffu, kRows - 1u);
      row[2] = min(r02 >> 16, kRows - 1u);
      row[3] = min(r13 >> 16, kRows - 1u);
    }
  }

  static __device__ __forceinline__ void count_bond(uint32_t s, uint32_t sn, uint32_t J, uint32_t& good, uint32_t&) {
    good += potts::zero2(perm_apply(J, sn) ^ s);
  }
};

template <int D, int RT, bool KONE>
__global__ void __launch_bounds__(kBlock, RT == 2 ? 4 : 5) k_sweep_perm(const potts::Params p) {
  __shared__ uint4 tab[KONE ? PermModel<D>::kRows : 1];
  potts::sweep_words<PermModel<D>, D, RT, KONE>(p, tab);
}

// Couplings from the PERM stream (jmode 0) or identity permutations (jmode
// 1); initial states from the PINIT stream, as for the J-weighted Potts glass.
__global__ void k_init_perm(uint32_t* spins, uint32_t* J, Geom geom, int Q4, int slots, int jmode, PhiloxKeys keys) {
  const uint64_t total = (uint64_t)Q4 * geom.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t q = (uint32_t)(idx / geom.N), i = (uint32_t)(idx - (uint64_t)q * geom.N);
    const uint32_t j = perm_split(geom, i);
    for (int d = 0; d < geom.D; ++d) {
      uint32_t w = 0;
      if (jmode == 1) {
        w = kIdentityCode * 0x01010101u;
      } else {
        const uint4 r = philox10(i, (uint32_t)d, (TAG_PERM << 28) | q, 0u, keys);
        const uint32_t xs[4] = {r.x, r.y, r.z, r.w};
        for (int b = 0; b < 4; ++b) w |= perm_code_of((uint32_t)(((uint64_t)xs[b] * 24u) >> 32)) << (8 * b);
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

// natural order [S][per][N] <-> packed split words, any D.  Spins: words
// [per = slots][Q4][N]; couplings (by_quad): words [Q4][per = D][N].
__device__ __forceinline__ size_t perm_word_row(bool by_quad, int m, int q, int Q4, int per, uint32_t N) {
  return by_quad ? ((size_t)q * per + m) * N : ((size_t)m * Q4 + q) * N;
}

__global__ void k_get_bytes_perm(const uint32_t* words, int8_t* out, Geom geom, int S, int Q4, int per,
                                 bool by_quad) {
  const uint64_t total = (uint64_t)S * per * geom.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int m = (int)(rest % per), s = (int)(rest / per);
    const uint32_t w = words[perm_word_row(by_quad, m, s >> 2, Q4, per, geom.N) + perm_split(geom, i)];
    out[idx] = (int8_t)(uint8_t)(w >> (8 * (s & 3)));
  }
}

__global__ void k_set_bytes_perm(uint32_t* words, const int8_t* in, Geom geom, int S, int Q4, int per, bool by_quad,
                                 uint32_t mask) {
  const uint64_t total = (uint64_t)Q4 * per * geom.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)(idx % geom.N);
    const uint64_t rest = idx / geom.N;
    const int m = (int)(rest % per), q = (int)(rest / per);
    uint32_t* wp = &words[perm_word_row(by_quad, m, q, Q4, per, geom.N) + perm_split(geom, i)];
    uint32_t w = *wp;
    for (int b = 0; b < 4; ++b) {
      const int s = 4 * q + b;
      if (s >= S) break;
      const uint32_t v = (uint32_t)(uint8_t)in[((size_t)s * per + m) * geom.N + i] & mask;
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

cudaError_t launch_init_perm(Lattice& lat, int jmode) {
  k_init_perm<<<grid_for((uint64_t)lat.Q4 * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.spins, (uint32_t*)lat.J, lat.geom, lat.Q4, lat.slots, jmode, lat.keys);
  return cudaGetLastError();
}

cudaError_t launch_sweep_perm(Lattice& lat, int colour, uint64_t t) {
  const void* k[3][2][2] = {{{(const void*)k_sweep_perm<2, 1, false>, (const void*)k_sweep_perm<2, 1, true>},
                             {(const void*)k_sweep_perm<2, 2, false>, (const void*)k_sweep_perm<2, 2, true>}},
                            {{(const void*)k_sweep_perm<3, 1, false>, (const void*)k_sweep_perm<3, 1, true>},
                             {(const void*)k_sweep_perm<3, 2, false>, (const void*)k_sweep_perm<3, 2, true>}},
                            {{(const void*)k_sweep_perm<4, 1, false>, (const void*)k_sweep_perm<4, 1, true>},
                             {(const void*)k_sweep_perm<4, 2, false>, (const void*)k_sweep_perm<4, 2, true>}}};
  const int rt = lat.R % 2 == 0 ? 2 : 1;
  return potts::launch_sweep(lat, colour, t, k[lat.D - 2][rt - 1][lat.K == 1], rt, rt == 2 ? 4 : 5);
}


cudaError_t launch_measure_perm(Lattice& lat, int want_q) {
  if (lat.D == 4)
    return potts::launch_measure(lat, want_q, potts::k_measure<PermModel<4>, 4, 1>,
                                 potts::k_measure<PermModel<4>, 4, 2>);
  if (lat.D == 3)
    return potts::launch_measure(lat, want_q, potts::k_measure<PermModel<3>, 3, 1>,
                                 potts::k_measure<PermModel<3>, 3, 2>);
  return potts::launch_measure(lat, want_q, potts::k_measure<PermModel<2>, 2, 1>, potts::k_measure<PermModel<2>, 2, 2>);
}

cudaError_t launch_get_spins_perm(Lattice& lat, int8_t* dev_out) {
  k_get_bytes_perm<<<grid_for((uint64_t)lat.S * lat.slots * lat.N), 256, 0, lat.stream>>>(
      (const uint32_t*)lat.spins, dev_out, lat.geom, lat.S, lat.Q4, lat.slots, false);
  return cudaGetLastError();
}

cudaError_t launch_set_spins_perm(Lattice& lat, const int8_t* dev_in) {
  k_set_bytes_perm<<<grid_for((uint64_t)lat.slots * lat.Q4 * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.spins, dev_in, lat.geom, lat.S, lat.Q4, lat.slots, false, 3u);
  return cudaGetLastError();
}

cudaError_t launch_get_couplings_perm(Lattice& lat, int8_t* dev_out) {
  k_get_bytes_perm<<<grid_for((uint64_t)lat.S * lat.D * lat.N), 256, 0, lat.stream>>>(
      (const uint32_t*)lat.J, dev_out, lat.geom, lat.S, lat.Q4, lat.D, true);
  return cudaGetLastError();
}

cudaError_t launch_set_couplings_perm(Lattice& lat, const int8_t* dev_in) {
  k_set_bytes_perm<<<grid_for((uint64_t)lat.Q4 * lat.D * lat.N), 256, 0, lat.stream>>>(
      (uint32_t*)lat.J, dev_in, lat.geom, lat.S, lat.Q4, lat.D, true, 0xFFu);
  return cudaGetLastError();
}

}  // namespace ianus
